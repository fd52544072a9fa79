"""The training pass on one cluster, where a block has no tile, a round is not
full, a mini-batch takes several rounds, and at the largest mini-batch it
serves and the next: one step is the library's own gradient (another kernel)
and Adam, a pass repeats bit for bit."""
import pytest

from tests import test_gpu_train_edges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(100, 112), (128, 128), (129, 4096), (1040, 4096), (4000, 4096), (4096, 4096),
                                     (4097, 4097), (9000, 4096), (300, 120)])
def test_cluster_steps(n, batch):
    test_gpu_train_edges.test_one_step_is_gradient_and_adam(n, batch)
