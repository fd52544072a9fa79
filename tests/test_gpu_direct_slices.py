"""Direct sums at the number of targets from which the sources are cut into
more slices, with fewer tiles than slices and with many."""
import pytest

from tests import test_gpu_direct

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,ns", [([70001], 1792), ([70001], 1793), ([300], 2048), ([3000, 500], 2500)])
def test_direct_more_slices(sizes, ns):
    test_gpu_direct.test_direct_edges(sizes, ns)
