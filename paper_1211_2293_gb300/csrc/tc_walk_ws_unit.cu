// tc_walk_ws_unit.cu -- the walk on producer and consumer warps for list
// tiles of TC_WALK_TILE entries, every mode.  The build compiles this file
// once per tile in {64, 128, 256}, defining the macro, and once with 32, the
// quadrupole walk.
#include <algorithm>

#include "tc_walk.cuh"
#include "tc_walk_ws.cuh"

#if !defined(TC_WALK_TILE)
#error "compile with -DTC_WALK_TILE=<32|64|128|256>"
#endif

#define TC_PASTE2(a, b) a##b
#define TC_UNIT_NAME(stem, t) TC_PASTE2(stem, t)

namespace tc {

#if TC_WALK_TILE == 32
// by shared memory (and 1 KB a block of 228 on an SM) and by registers: 128 a
// thread, the launch bounds' cap, so eight teams of two warps
int walk_ws_teams(const WalkConfig& c)
{
    const WsShape w = ws_shape(c, c.quadw ? 32 : c.tile, c.learned && !c.record);
    const int teams = w.threads / 64, by_smem = (int)(228 * 1024 / (w.smem + 1024));
    return std::min(by_smem, 8 / teams) * teams;
}

cudaError_t prepare_walk_ws_t32(const WalkConfig& c, int num_sms, int* grid, size_t* smem)
{
    if (!c.quadw || c.learned || !c.precise || c.gmax > 64) return cudaErrorInvalidValue;
    if (c.want_pot) return prepare_ws_t<32, true, true, 0>(c, num_sms, grid, smem);
    return prepare_ws_t<32, true, false, 0>(c, num_sms, grid, smem);
}

cudaError_t launch_walk_ws_t32(const WalkArgs& a, const WalkConfig& c, int grid, size_t smem, cudaStream_t s)
{
    if (!c.quadw || c.learned || !c.precise || c.gmax > 64) return cudaErrorInvalidValue;
    if (c.want_pot) return launch_ws_t<32, true, true, 0>(a, c, grid, smem, s);
    return launch_ws_t<32, true, false, 0>(a, c, grid, smem, s);
}
#else
// precise or plain, with or without the potential; the learned walk (precise,
// no potential) evaluates its band cells or
// records them for k_band_eval
cudaError_t TC_UNIT_NAME(prepare_walk_ws_t, TC_WALK_TILE)(const WalkConfig& c, int num_sms, int* grid, size_t* smem)
{
    const bool p = c.precise != 0, pot = c.want_pot != 0;
    if (c.quadw || (c.learned && (!p || pot))) return cudaErrorInvalidValue;
    if (c.learned && c.record) return prepare_ws_t<TC_WALK_TILE, true, false, 1>(c, num_sms, grid, smem);
    if (c.learned) return prepare_ws_t<TC_WALK_TILE, true, false, 2>(c, num_sms, grid, smem);
    if (p && pot) return prepare_ws_t<TC_WALK_TILE, true, true, 0>(c, num_sms, grid, smem);
    if (p) return prepare_ws_t<TC_WALK_TILE, true, false, 0>(c, num_sms, grid, smem);
    if (pot) return prepare_ws_t<TC_WALK_TILE, false, true, 0>(c, num_sms, grid, smem);
    return prepare_ws_t<TC_WALK_TILE, false, false, 0>(c, num_sms, grid, smem);
}

cudaError_t TC_UNIT_NAME(launch_walk_ws_t, TC_WALK_TILE)(const WalkArgs& a, const WalkConfig& c, int grid, size_t smem,
                                                         cudaStream_t s)
{
    const bool p = c.precise != 0, pot = c.want_pot != 0;
    if (c.quadw || (c.learned && (!p || pot))) return cudaErrorInvalidValue;
    if (c.learned && c.record) return launch_ws_t<TC_WALK_TILE, true, false, 1>(a, c, grid, smem, s);
    if (c.learned) return launch_ws_t<TC_WALK_TILE, true, false, 2>(a, c, grid, smem, s);
    if (p && pot) return launch_ws_t<TC_WALK_TILE, true, true, 0>(a, c, grid, smem, s);
    if (p) return launch_ws_t<TC_WALK_TILE, true, false, 0>(a, c, grid, smem, s);
    if (pot) return launch_ws_t<TC_WALK_TILE, false, true, 0>(a, c, grid, smem, s);
    return launch_ws_t<TC_WALK_TILE, false, false, 0>(a, c, grid, smem, s);
}

#endif

}  // namespace tc
