// tc_build.cu -- oct-tree construction on the GPU (Sec. 3.1 of the paper:
// the space is divided recursively into 8 sub-cubes until a cube holds no
// more than a threshold of bodies; every cell carries its total mass and
// centre of mass).
//
// The bodies of a batch of independent systems are processed together: each
// system gets its own root cube and tree, and a system boundary acts like a
// difference in the first digit of two keys.
//
// Pipeline (all on one stream):
//   1. k_build_init, k_bbox  scratch zeroed; per-system bounding box ->
//                  power-of-two root cube on a 2^21 grid (FP64)
//   2. k_keys      63-bit Morton keys (exact quantisation) and the sort's
//                  digit counts
//   3. radix sort  stable sort by (system, key, index)    [tc_sort.cu]
//   4. the bodies in Morton order as float4 (x, y, z, m): k_gather, or with
//                  the sort's completion
//   5. k_window, k_window_max, k_node_levels (or k_node_levels_tiled), k_scan_levels
//                  which cubes of the recursive subdivision start at each
//                  sorted body (a sliding-window test, below), how many of
//                  each level per block of bodies, and their scan: the
//                  nodes' places in breadth-first order
//   6. k_emit_nodes  the node records: first body, first child, parent,
//                  integer centre
//   7. k_leaf_nodes  children and counts; mass / centre of mass (float-pair
//                  sums, FP64-class, stored in FP64) / second moments (FP32)
//                  of the leaves; the internal cells bottom-up in the same
//                  launch (small trees) or by k_level_moments level by level
//                  from the deepest
//   8. k_group_marks + k_group_table   body groups for the walk
//
// Which cubes exist.  Let cd(a, b) be the number of leading octal digits two
// keys share.  The level-l run of equal l-digit prefixes that contains sorted
// body s holds more than leaf_max bodies iff some window of leaf_max + 1
// consecutive bodies containing s lies inside it, i.e. iff
//     W_s = max_{j in [s - leaf_max, s]} cd(key_j, key_{j + leaf_max}) >= l.
// A cube at level l is created by the subdivision iff its parent cube holds
// more than leaf_max bodies (and the parent is above level 21).  So the cubes
// whose first body is s are the levels l with
//     delta_s < l <= min(W_s + 1, 21),   delta_s = cd(key_{s-1}, key_s)
// (delta_0 = -1), and the deepest of them is a leaf.  Breadth-first order of
// the tree is the order of (level, first body).
#include "tc_internal.cuh"
#include "tc_lookback.cuh"
#include "tc_pdl.cuh"

// With several systems, cd() of two bodies of different systems is taken as
// -1 (no common cube), so delta_s = -1 at the first body of every system and
// each system's root is a node of level 0.  The node table is sized by the
// host from an earlier build; a device-side check stops the build (error word
// kErrCapacity) if a later tree needs more, so no kernel writes past it.

namespace tc {

namespace {

__device__ __forceinline__ int common_digits(uint64_t a, uint64_t b)
{
    uint64_t x = a ^ b;
    if (x == 0) return kMaxLevel;
    return (__clzll((long long)x) - 1) / 3;  // keys use bits 0..62
}

__device__ __forceinline__ uint64_t spread3(uint64_t v)
{
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x1f00000000ffffull;
    v = (v | (v << 16)) & 0x1f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__device__ __forceinline__ uint32_t compact3(uint64_t v)
{
    v &= 0x1249249249249249ull;
    v = (v ^ (v >> 2)) & 0x10c30c30c30c30c3ull;
    v = (v ^ (v >> 4)) & 0x100f00f00f00f00full;
    v = (v ^ (v >> 8)) & 0x1f0000ff0000ffull;
    v = (v ^ (v >> 16)) & 0x1f00000000ffffull;
    v = (v ^ (v >> 32)) & 0x1fffffull;
    return (uint32_t)v;
}

__device__ __forceinline__ bool capacity_failed(const Info* info)
{
    return (*(volatile const int32_t*)&info->err & kErrCapacity) != 0;
}

// ------------------------------------------------------------------ systems
__global__ void k_sys_ids(const int64_t* off, int nsys, int64_t n, uint32_t* sys_of,
                          SysParams* sysp)
{
    pdl_begin();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nsys) {
        sysp[i].first = (int32_t)off[i];
        sysp[i].end = (int32_t)off[i + 1];
    }
    if (i >= n) return;
    int lo = 0, hi = nsys - 1;  // last system whose offset is <= i
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    sys_of[i] = (uint32_t)lo;
}

// ------------------------------------------------------------------ bbox
constexpr int kBboxThreads = 256;

// floats as ints with the same order (no NaN): min/max by integer atomics
__device__ __forceinline__ int f2o(float x)
{
    const int i = __float_as_int(x);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float o2f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

__device__ __forceinline__ float warp_min(float x)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
__device__ __forceinline__ float warp_max(float x)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

__global__ void k_build_init(uint4* zero, int64_t nzero, SysParams* sysp, int nsys, Info* info,
                             int reset_err)
{
    pdl_begin();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = t; i < nzero; i += stride) zero[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t s = t; s < nsys; s += stride) {
        for (int a = 0; a < 3; a++) {
            sysp[s].bb[a] = f2o(INFINITY);
            sysp[s].bb[3 + a] = f2o(-INFINITY);
        }
        sysp[s].done = 0;
    }
    if (t == 0) {
        info->depth = 0;
        if (reset_err) info->err = 0;
    }
}

// Root cube of each system: side L = smallest power of two with
// L >= extent * (1 + 2^-20), grid step h = L / 2^21, corner c0 = floor(min/h) h.
__device__ void sys_cube(SysParams& P)
{
    double dlo[3], dhi[3];
    for (int a = 0; a < 3; a++) {
        dlo[a] = (double)o2f(__ldcg(&P.bb[a]));
        dhi[a] = (double)o2f(__ldcg(&P.bb[3 + a]));
    }
    double extent = 0.0;
    for (int a = 0; a < 3; a++) {
        const double e = dhi[a] - dlo[a];
        if (e > extent) extent = e;
    }
    const double target = extent * (1.0 + 0x1p-20);
    double L = 1.0;  // all bodies coincide (or a non-finite input): unit cube
    if (target > 0.0 && target < INFINITY) {
        int e;
        const double m = frexp(target, &e);
        L = (m == 0.5) ? target : ldexp(1.0, e);
    }
    const double h = L / 2097152.0;
    int eh;
    frexp(h, &eh);        // h = 2^(eh - 1)
    P.qexp = 1 - eh;      // 1/h = 2^qexp
    for (int a = 0; a < 3; a++) {
        double K0 = floor(dlo[a] / h);
        if (!(K0 == K0) || K0 > 9e15 || K0 < -9e15) K0 = 0.0;  // non-finite input: keys are reported, not used
        P.c0[a] = K0 * h;
        P.qoff[a] = (long long)K0;
    }
    P.L = L;
    P.h = h;
    P.Lf = (float)L;
    P.uf = (float)(h * 0.5);
}

// one block per chunk (system, start, end, chunks of the system); CUBES: the
// block that completes a system's last chunk forms its root cube
template <bool CUBES>
__global__ void __launch_bounds__(kBboxThreads) k_bbox(const float* pos, const int4* chunks,
                                                       SysParams* sysp, int32_t* err)
{
    pdl_begin();
    __shared__ float sm[6][kBboxThreads / 32];
    const int4 ch = chunks[blockIdx.x];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    bool bad = false;
    for (int64_t i = ch.y + threadIdx.x; i < ch.z; i += kBboxThreads) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const float x = pos[3 * i + a];
            bad |= !isfinite(x);
            lo[a] = fminf(lo[a], x);
            hi[a] = fmaxf(hi[a], x);
        }
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(err, kErrNonFinite);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float l = warp_min(lo[a]), h = warp_max(hi[a]);
        if (lane == 0) {
            sm[a][w] = l;
            sm[3 + a][w] = h;
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int a = threadIdx.x;
        float r = a < 3 ? INFINITY : -INFINITY;
        for (int k = 0; k < kBboxThreads / 32; k++) r = a < 3 ? fminf(r, sm[a][k]) : fmaxf(r, sm[a][k]);
        if (a < 3) atomicMin(&sysp[ch.x].bb[a], f2o(r));
        else atomicMax(&sysp[ch.x].bb[a], f2o(r));
        if (!CUBES) return;
        __threadfence();  // before this chunk counts as done
        __syncwarp(0x3fu);
        if (a == 0 && atomicAdd(&sysp[ch.x].done, 1) == ch.w - 1) {
            __threadfence();
            sys_cube(sysp[ch.x]);
        }
    }
}

__global__ void k_cubes(SysParams* sysp, int nsys)
{
    pdl_begin();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nsys) sys_cube(sysp[s]);
}

// ------------------------------------------------------------------ keys
// q = floor((x - c0) / h) clamped to [0, 2^21 - 1], evaluated exactly: h is
// a power of two and c0 = K0 h with K0 an integer, so q = floor(x * 2^k) - K0
// with 2^k = 1/h -- an exact float scaling, an exact floor and an integer
// subtraction.  Key digit l holds the level-l bits of (qx, qy, qz), x highest.
__device__ __forceinline__ uint64_t quantise(float x, int k, long long K0)
{
    float t = floorf(scalbnf(x, k));
    if (x < 0.0f && t == 0.0f) t = -1.0f;  // a negative value scaled below the float range
    long long q = __float2ll_rz(t) - K0;    // the conversion saturates out-of-range values
    q = q < 0 ? 0 : (q > 2097151 ? 2097151 : q);
    return (uint64_t)q;
}

constexpr int kKeyRounds = 4;  // bodies of a thread whose loads are in flight together

// also (ghist not null) the digit counts of the sort's passes, per block in
// shared memory
__global__ void __launch_bounds__(256) k_keys(const float* pos, const float* mass, int64_t n,
                                              const uint32_t* sys_of, const SysParams* sysp,
                                              uint64_t* keys, uint32_t* idx, SortPlan plan,
                                              uint32_t* ghist, int32_t* err)
{
    pdl_begin();
    __shared__ uint32_t h[kSortMaxPasses][256];
    const int npass = ghist ? plan.npass : 0;
    for (int p = 0; p < npass; p++) h[p][threadIdx.x] = 0u;
    __syncthreads();
    bool bad = false;
    for (int64_t i0 = (int64_t)blockIdx.x * (256 * kKeyRounds); i0 < n; i0 += (int64_t)gridDim.x * (256 * kKeyRounds)) {
        float x[kKeyRounds][3], m[kKeyRounds];
        uint32_t sy[kKeyRounds];
#pragma unroll
        for (int r = 0; r < kKeyRounds; r++) {
            const int64_t i = min(i0 + r * 256 + threadIdx.x, n - 1);
            sy[r] = sys_of[i];
            x[r][0] = pos[3 * i];
            x[r][1] = pos[3 * i + 1];
            x[r][2] = pos[3 * i + 2];
            m[r] = mass[i];
        }
#pragma unroll
        for (int r = 0; r < kKeyRounds; r++) {
            const int64_t i = i0 + r * 256 + threadIdx.x;
            const int64_t left = n - (i - (threadIdx.x & 31));  // bodies from the warp's first on
            const unsigned act = left >= 32 ? 0xffffffffu : (left > 0 ? (1u << left) - 1u : 0u);
            if (i >= n) continue;
            const SysParams& P = sysp[sy[r]];
            const int k = P.qexp;
            const uint64_t qx = quantise(x[r][0], k, P.qoff[0]);
            const uint64_t qy = quantise(x[r][1], k, P.qoff[1]);
            const uint64_t qz = quantise(x[r][2], k, P.qoff[2]);
            const uint64_t key = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
            keys[i] = key;
            idx[i] = (uint32_t)i;
            bad |= !(isfinite(m[r]) && m[r] > 0.0f);
            for (int p = 0; p < npass; p++) {
                const SortDigit dg = plan.digit(p);
                const uint32_t d = dg.of(key, sy[r]);
                if (dg.sys) {  // shared by most of a warp: one add for its equal digits
                    const unsigned same = __match_any_sync(act, d);
                    if ((same & ((1u << (threadIdx.x & 31)) - 1u)) == 0u) atomicAdd(&h[p][d], (uint32_t)__popc(same));
                } else {
                    atomicAdd(&h[p][d], 1u);
                }
            }
        }
    }
    if (bad) atomicOr(err, kErrNonFinite);
    __syncthreads();
    for (int p = 0; p < npass; p++) {
        const uint32_t c = h[p][threadIdx.x];
        if (c) atomicAdd(&ghist[p * 256 + threadIdx.x], c);
    }
}

__global__ void k_gather(const float* pos, const float* mass,
                         const uint32_t* perm, int64_t n, float4* body)
{
    pdl_begin();
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int64_t i = perm[k];
    body[k] = make_float4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], mass[i]);
}

// ------------------------------------------------------------------ nodes
// Blocks of kNodeBlock sorted bodies count and place the nodes that start at
// their bodies.  Breadth-first order is (level, first body), so the exclusive
// scan of the blocks' counts, laid out level by level, is the place of each
// block's first node of each level: no pre-order table and no sort by level
// lie between the counts and the node table.
// A thread takes kNodeRounds bodies, so that a block's chain of barriers and
// loads is shared by four times as many bodies as with one each (59 -> 40 and
// 94 -> 47 us for the two kernels at 2^22).
constexpr int kNodeThreads = 256, kNodeRounds = 4;
constexpr int kNodeBlock = kNodeThreads * kNodeRounds;
constexpr int kNodeSets = kNodeBlock / 32;  // runs of 32 consecutive bodies, set r * 8 + warp
constexpr int kLevels = kMaxLevel + 1;
constexpr int kTileWindow = 256;

__device__ __forceinline__ uint32_t warp_incl(uint32_t x)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// the starts per level of a set of 32 bodies (levels d < l <= t of each): lane l
// holds level l's
__device__ __forceinline__ uint32_t set_levels(int d, int t)
{
    uint32_t mine = 0;
    const int hi = __reduce_max_sync(0xffffffffu, t);  // the set's levels
    for (int l = __reduce_min_sync(0xffffffffu, t > d ? d : kMaxLevel) + 1; l <= hi; l++) {
        const unsigned m = __ballot_sync(0xffffffffu, d < l && l <= t);
        if ((int)(threadIdx.x & 31) == l) mine = __popc(m);
    }
    return mine;
}

// per level, the block's nodes -> cnt[l][block]; the deepest level of the
// forest (a block maximum, then one atomic a block)
__device__ __forceinline__ void count_levels(const int (&d)[kNodeRounds], const int (&t)[kNodeRounds],
                                             uint32_t* cnt, int32_t* depth)
{
    __shared__ uint32_t wc[kNodeThreads / 32][kLevels];
    __shared__ int wmax[kNodeThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t mine = 0;
    int hi = -1;
#pragma unroll
    for (int r = 0; r < kNodeRounds; r++) {
        mine += set_levels(d[r], t[r]);
        hi = max(hi, t[r]);
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane < kLevels) wc[w][lane] = mine;
    if (lane == 31) wmax[w] = hi;
    __syncthreads();
    if (threadIdx.x < kLevels) {
        uint32_t c = 0;
#pragma unroll
        for (int k = 0; k < kNodeThreads / 32; k++) c += wc[k][threadIdx.x];
        cnt[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = c;
    } else if (threadIdx.x == 32) {
        for (int k = 0; k < kNodeThreads / 32; k++) hi = max(hi, wmax[k]);
        atomicMax(depth, hi);
    }
}

__global__ void k_window(const uint64_t* keys, const uint32_t* sys_of, int64_t n,
                         int leaf_max, int8_t* w)
{
    pdl_begin();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    w[j] = (j + leaf_max < n && sys_of[j] == sys_of[j + leaf_max])
               ? (int8_t)common_digits(keys[j], keys[j + leaf_max])
               : (int8_t)-1;
}

// leaf_max > kTileWindow: the window digits come from k_window, a body's
// deepest level into top[] by a thread each (four long windows one after
// another in the threads of k_node_levels left few warps to wait for their
// loads: 4096 bodies of leaf_max 4096 49 us with a thread each, 200 with four
// bodies a thread)
__global__ void __launch_bounds__(256) k_window_max(const int8_t* w, int64_t n, int leaf_max, int8_t* top)
{
    pdl_begin();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    int W = -1;
    const int64_t j0 = s - leaf_max < 0 ? 0 : s - leaf_max;
    for (int64_t j = j0; j <= s; j++) W = max(W, (int)w[j]);
    top[s] = (int8_t)min(W + 1, kMaxLevel);
}

__global__ void __launch_bounds__(kNodeThreads) k_node_levels(const uint64_t* keys,
                                                              const uint32_t* sys_of, int64_t n,
                                                              int8_t* delta, const int8_t* top,
                                                              int32_t* gref_at, uint32_t* cnt,
                                                              int32_t* depth)
{
    pdl_begin();
    int d[kNodeRounds], t[kNodeRounds];
#pragma unroll
    for (int r = 0; r < kNodeRounds; r++) {
        const int64_t s = (int64_t)blockIdx.x * kNodeBlock + r * kNodeThreads + threadIdx.x;
        t[r] = -1;
        d[r] = 0;
        if (s < n) {
            d[r] = (s == 0 || sys_of[s] != sys_of[s - 1]) ? -1 : common_digits(keys[s - 1], keys[s]);
            t[r] = top[s];
            delta[s] = (int8_t)d[r];
            gref_at[s] = 0;
        }
    }
    count_levels(d, t, cnt, depth);
}

// The same in one kernel for leaf_max <= kTileWindow: a block stages the keys
// and systems of [b0 - leaf_max, b0 + kNodeBlock + leaf_max) in shared memory,
// forms the window digits cd(key_j, key_j+leaf_max) there, and takes each
// body's window maximum from them.
__global__ void __launch_bounds__(kNodeThreads) k_node_levels_tiled(const uint64_t* keys,
                                                                    const uint32_t* sys_of, int64_t n,
                                                                    int leaf_max, int8_t* delta,
                                                                    int8_t* top,
                                                                    int32_t* gref_at,
                                                                    uint32_t* cnt,
                                                                    int32_t* depth)
{
    pdl_begin();
    __shared__ uint64_t sk[kNodeBlock + 2 * kTileWindow];
    __shared__ uint32_t ss[kNodeBlock + 2 * kTileWindow];
    __shared__ int8_t sw[kNodeBlock + kTileWindow];
    const int64_t b0 = (int64_t)blockIdx.x * kNodeBlock;
    const int64_t base = b0 - leaf_max;  // smem index 0 holds body base
    const int nk = kNodeBlock + 2 * leaf_max;
#pragma unroll 6
    for (int i = threadIdx.x; i < nk; i += kNodeThreads) {
        const int64_t j = base + i;
        const bool in = j >= 0 && j < n;
        sk[i] = in ? keys[j] : 0ull;
        ss[i] = in ? sys_of[j] : 0xffffffffu;
    }
    __syncthreads();
    // window digits of bodies base .. b0 + kNodeBlock - 1
    const int nw = kNodeBlock + leaf_max;
    for (int i = threadIdx.x; i < nw; i += kNodeThreads) {
        const int64_t j = base + i;
        int8_t v = -1;
        if (j >= 0 && j + leaf_max < n && ss[i] == ss[i + leaf_max]) v = (int8_t)common_digits(sk[i], sk[i + leaf_max]);
        sw[i] = v;
    }
    __syncthreads();
    int d[kNodeRounds], t[kNodeRounds];
#pragma unroll
    for (int r = 0; r < kNodeRounds; r++) {
        const int at = r * kNodeThreads + threadIdx.x;
        const int64_t s = b0 + at;
        t[r] = -1;
        d[r] = 0;
        if (s < n) {
            const int i = at + leaf_max;  // smem index of body s
            d[r] = (s == 0 || ss[i] != ss[i - 1]) ? -1 : common_digits(sk[i - 1], sk[i]);
            int W = -1;
            const int i0 = s - leaf_max < 0 ? (int)(leaf_max - s) : 0;  // window clipped at body 0
            for (int k = i0; k <= leaf_max; k++) W = max(W, (int)sw[at + k]);
            t[r] = min(W + 1, kMaxLevel);
            delta[s] = (int8_t)d[r];
            top[s] = (int8_t)t[r];
            gref_at[s] = 0;
        }
    }
    count_levels(d, t, cnt, depth);
}

// Exclusive scan of the counts in place, one pass; the total is the number of
// nodes (info->M follows with the records).  A look-back that gave up raises
// kErrCapacity too, so nothing is placed by offsets that are not known.
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

// the block's exclusive scan of one value per thread (kScanThreads of them),
// plus the sum of the tiles before this one; *total: this prefix + the tile
__device__ __forceinline__ uint32_t scan_tile(uint32_t x, int64_t tile, unsigned long long* st, uint32_t* total,
                                              bool* ok)
{
    __shared__ uint32_t wsum[kScanThreads / 32];
    __shared__ uint32_t pre_sh;
    __shared__ bool ok_sh;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t incl = warp_incl(x);
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int k = 0; k < kScanThreads / 32; k++) {
        if (k < w) before += wsum[k];
        all += wsum[k];
    }
    if (w == 0) {
        bool good;
        const uint32_t pre = tile_prefix(st, tile, all, &good);
        if (lane == 0) {
            pre_sh = pre;
            ok_sh = good;
        }
    }
    __syncthreads();
    *total = pre_sh + all;
    *ok = ok_sh;
    return pre_sh + before + incl - x;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_levels(uint32_t* cnt, int64_t ncnt,
                                                              unsigned long long* st, uint32_t* counter, int64_t cap_m,
                                                              Info* info)
{
    pdl_begin();
    __shared__ int tile_sh;
    if (threadIdx.x == 0) tile_sh = (int)atomicAdd(counter, 1u);
    __syncthreads();
    const int64_t tile = tile_sh, t0 = tile * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems], sum = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        v[i] = t0 + i < ncnt ? cnt[t0 + i] : 0u;
        sum += v[i];
    }
    uint32_t total;
    bool ok;
    uint32_t e = scan_tile(sum, tile, st, &total, &ok);
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        if (t0 + i < ncnt) cnt[t0 + i] = e;
        e += v[i];
    }
    if (threadIdx.x == 0) {
        if (!ok) atomicOr(&info->err, kErrWorkLoop | kErrCapacity);
        if (tile == gridDim.x - 1) {
            info->count = total;
            if (cap_m >= 0 && (int64_t)total > cap_m) atomicOr(&info->err, kErrCapacity);
        }
    }
}

// The node records of every body of a block: (s, l) for delta < l <= top, at
// place offs[l][block] + its rank among the block's starts of level l.  Its
// first child is (s, l + 1); its parent the last node of level l - 1 that
// starts at or before s.  fam = 1 marks a node that follows a sibling (the
// topmost one starting at its body), so the children of a cell are its first
// child and the marked nodes right after it.  Counts follow bottom-up.
__global__ void __launch_bounds__(kNodeThreads) k_emit_nodes(const uint64_t* keys,
                                                             const int8_t* delta,
                                                             const int8_t* top,
                                                             const uint32_t* sys_of, int64_t n,
                                                             const uint32_t* offs, Info* info,
                                                             uint32_t* lstart, NodeTables nt)
{
    pdl_begin();
    if (capacity_failed(info)) return;
    __shared__ uint32_t wc[kNodeSets][kLevels];
    __shared__ uint4 list[kNodeThreads / 32][64];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
    const int64_t b0 = (int64_t)blockIdx.x * kNodeBlock;
    int d[kNodeRounds], t[kNodeRounds];
    uint64_t key[kNodeRounds];
    uint32_t sy[kNodeRounds];
#pragma unroll
    for (int r = 0; r < kNodeRounds; r++) {
        const int64_t s = b0 + r * kNodeThreads + threadIdx.x;
        d[r] = s < n ? delta[s] : 0;
        t[r] = s < n ? top[s] : -1;
        key[r] = s < n ? keys[s] : 0ull;
        sy[r] = s < n ? sys_of[s] : 0u;
    }
    if (blockIdx.x == 0 && threadIdx.x <= kLevels)  // the first node of each level
        lstart[threadIdx.x] = threadIdx.x < kLevels ? offs[(int64_t)threadIdx.x * gridDim.x] : (uint32_t)info->count;
    if (blockIdx.x == 0 && threadIdx.x == 0) info->M = info->count;
#pragma unroll
    for (int r = 0; r < kNodeRounds; r++) {
        const uint32_t mine = set_levels(d[r], t[r]);
        if (lane < kLevels) wc[r * (kNodeThreads / 32) + w][lane] = mine;
    }
    __syncthreads();
    // a warp per level: the sets' counts -> the place of each set's first node
    for (int l = w; l < kLevels; l += kNodeThreads / 32) {
        static_assert(kNodeSets == 32, "a lane per set");
        const uint32_t c = wc[lane][l];
        wc[lane][l] = offs[(int64_t)l * gridDim.x + blockIdx.x] + warp_incl(c) - c;
    }
    __syncthreads();
    // the warp's nodes pass through a list, so that 32 lanes write 32 records
    // (a set has about a dozen, spread over its levels)
    int cnt = 0;
    auto flush = [&](int m) {  // the last m <= 32 nodes of the list
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        if (lane < m) q = list[w][cnt - m + lane];
        cnt -= m;
        const int from = q.x & 31, lv = (q.x >> 5) & 31, r = (q.x >> 11) & (kNodeRounds - 1);
        uint64_t k = 0ull;
        uint32_t ky = 0u;
#pragma unroll
        for (int u = 0; u < kNodeRounds; u++) {
            const uint64_t ku = __shfl_sync(0xffffffffu, key[u], from);
            const uint32_t su = __shfl_sync(0xffffffffu, sy[u], from);
            if (u == r) {
                k = ku;
                ky = su;
            }
        }
        __syncwarp();
        if (lane < m) {
            const uint32_t at = q.y;
            const uint64_t pfx = lv == 0 ? 0ull : (k >> (3 * (kMaxLevel - lv)));
            const int c1 = 1 << (kMaxLevel - lv);
            nt.b[at] = make_int4((int)b0 + r * kNodeThreads + w * 32 + from, 0, (int32_t)q.z, lv);
            nt.c[at] = make_int4((int)(2 * compact3(pfx >> 2) + 1) * c1, (int)(2 * compact3(pfx >> 1) + 1) * c1,
                                 (int)(2 * compact3(pfx) + 1) * c1, (int)ky);
            nt.fam[at] = (uint8_t)((q.x >> 10) & 1u);
            nt.parent[at] = (int32_t)q.w;
            nt.pend[at] = 0u;
        }
    };
#pragma unroll
    for (int r = 0; r < kNodeRounds; r++) {
        const uint32_t* place = wc[r * (kNodeThreads / 32) + w];
        const int lhi = __reduce_max_sync(0xffffffffu, t[r]);  // the set's levels
        const int llo = __reduce_min_sync(0xffffffffu, t[r] > d[r] ? d[r] : kMaxLevel) + 1;
        if (lhi < llo) continue;
        uint32_t before = llo > 0 ? place[llo - 1] : 0u;  // nodes of the level above up to body s
        bool had = false;
        uint32_t pos = 0;
        int32_t par = -1;
        for (int l = llo; l <= lhi + 1; l++) {
            const bool here = l < kLevels && d[r] < l && l <= t[r];
            const unsigned m = __ballot_sync(0xffffffffu, here), hm = __ballot_sync(0xffffffffu, had);
            const uint32_t base = l < kLevels ? place[l] : 0u;
            const uint32_t p = base + __popc(m & lt);
            if (had)  // node (s, l - 1), whose first child is (s, l) if that exists
                list[w][cnt + __popc(hm & lt)] =
                    make_uint4((unsigned)lane | ((unsigned)(l - 1) << 5) | (l == d[r] + 2 ? 1024u : 0u) | ((unsigned)r << 11),
                               pos, here ? p : 0xffffffffu, (uint32_t)par);
            cnt += __popc(hm);
            __syncwarp();
            if (cnt >= 32) flush(32);
            par = l > 0 ? (int32_t)before - 1 : -1;
            before = base + __popc(m & le);
            pos = p;
            had = here;
        }
    }
    if (cnt > 0) flush(cnt);
}

// children of the cell whose first child is cf: cf and the marked nodes after it
__device__ __forceinline__ int family(const uint8_t* fam, int64_t cf, int64_t M)
{
    unsigned marks = 0;
#pragma unroll
    for (int k = 1; k < 8; k++) marks |= (cf + k < M && fam[cf + k]) ? 1u << (k - 1) : 0u;
    return __ffs(~marks);  // 1 + the run of marks
}

// ------------------------------------------------------------------ moments
// Mass, centre of mass and second moments about the centre of mass.  The
// sums of m and m x are kept as unevaluated pairs of floats (hi + lo, about
// 48 significant bits) on the FP32 pipe and stored in FP64 as well; GB300's
// FP64 pipe, a small fraction of its FP32 rate, bound these kernels when
// they summed in FP64.  Leaves sum their bodies;
// an internal cell combines its children: M = sum M_c,
// com = sum M_c com_c / M, Q = sum Q_c + M_c dc dc^T with dc = com_c - com.
// Leaves are done in one launch.  Internal cells follow level by level from
// the deepest, one thread per cell of the level (cells of a level are
// contiguous in breadth-first order), so every lane of a warp has a cell to
// do; in small trees, where each of those launches is a few microseconds of
// latency, the thread that completes a cell's last child computes the cell
// in the leaves' launch (k_leaf_nodes): a build of 4096 / 100003 / 300000
// bodies takes 174 / 204 / 238 us so, 187 / 220 / 247 with a launch per
// level, but 370 against 366 us at 10^6 and 990 against 852 at 2^22, where
// the fences of every climb cost more.
__device__ __forceinline__ void cube_centre(const SysParams& P, int4 c, double* C)
{
    const double u = 0.5 * P.h;
    C[0] = P.c0[0] + (double)c.x * u;
    C[1] = P.c0[1] + (double)c.y * u;
    C[2] = P.c0[2] + (double)c.z * u;
}

// The exact FP64 value of a float, formed on the integer pipe from the
// IEEE-754 fields (sign, exponent rebased from 127 to 1023, the 23 mantissa
// bits moved to the top of the 52): GB300's FP64 pipe, which the leaf
// moments saturate, then only adds and multiplies.  Zero, subnormal and
// non-finite values take the conversion instruction.
__device__ __forceinline__ double widen(float f)
{
    const uint32_t u = __float_as_uint(f);
    const uint32_t e = (u >> 23) & 0xffu;
    if (e == 0u || e == 0xffu) return (double)f;
    const uint64_t d = ((uint64_t)(u >> 31) << 63) | ((uint64_t)(e + 896u) << 52) | ((uint64_t)(u & 0x7fffffu) << 29);
    return __longlong_as_double((long long)d);
}

// (hi, lo) += p + e for a normalised pair (|lo| <= ulp(hi) / 2): hi + p by
// Knuth's TwoSum (s + t = hi + p exactly), the error t, lo and e added in
// FP32, then renormalised by Dekker's FastTwoSum (exact: |t| is a few ulps
// of s at most, or s = 0).  One call errs by at most about 2^-46 |s|.
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float p, float e)
{
    const float s = hi + p;
    const float bp = s - hi;
    const float t = ((hi - (s - bp)) + (p - bp)) + (lo + e);
    hi = s + t;
    lo = t - (hi - s);
}

// the centre of mass S / m of float pairs as a pair of floats: q1 = Sh / mh,
// the remainder S - q1 m (Sh - q1 mh exact by one FMA: the residual of a
// correctly rounded quotient is a float), q2 = remainder / mh; q1 + q2 is
// S / m within about 2^-44 of it, taken exactly into FP64 (com) and rounded
// once to float (comf); the FP64 pipe is spared the division
__device__ __forceinline__ void pair_quotient(const float (&Sh)[3], const float (&Sl)[3], float mh, float ml,
                                              double (&com)[3], float (&comf)[3])
{
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float q1 = Sh[a] / mh;
        const float r = fmaf(-q1, mh, Sh[a]) + fmaf(-q1, ml, Sl[a]);
        const float q2 = r / mh;
        com[a] = widen(q1) + widen(q2);
        comf[a] = q1 + q2;
    }
}

// comf / Mf: the float roundings of com and M when the caller has
// them (the same values, without the FP64 pipe's conversions)
template <bool QUAD>
__device__ void store_node(const NodeTables& nt, int64_t v, double M, const double* com, const float* Q, const double* C,
                           const float* comf = nullptr, float Mf = 0.f)
{
    nt.mass64[v] = M;
    for (int a = 0; a < 3; a++) nt.com64[3 * v + a] = com[a];
    const float mf = comf ? Mf : (float)M;
    nt.a[v] = make_float4((float)(com[0] - C[0]), (float)(com[1] - C[1]), (float)(com[2] - C[2]), mf);
    if (comf) nt.d[v] = make_float4(comf[0], comf[1], comf[2], mf);
    else nt.d[v] = make_float4((float)com[0], (float)com[1], (float)com[2], mf);
    if (QUAD) {
        for (int a = 0; a < 6; a++) nt.quad[6 * v + a] = Q[a];
    }
}

// Mass and centre of mass as float pairs (FP64-class); second moments in
// FP32.  The second moments only feed the learned correction's BF16
// features and the quadrupole terms, small corrections to the monopole, so
// FP32 serves them (their error stays a few hundred FP32 ulps of M s^2).
// Per leaf: Q about the cube centre C from the bodies'
// offsets x - C, then moved to the centre of mass by the parallel-axis rule
// Q_com = Q_C - M (com - C)(com - C)^T.  The offsets are formed in FP32
// against C split into C_hi = fl(C) and C_lo = fl(C - C_hi): (x - C_hi) -
// C_lo, within 2 FP32 roundings of x - C (the first subtraction is exact
// unless |C| < 2 s, where its rounding is one of a number below 2 s).
// loads of what another thread of the same launch may have written (CG): past
// the first-level cache, which other SMs' writes do not reach
template <bool CG, typename T>
__device__ __forceinline__ T ld(const T* p)
{
    return CG ? __ldcg(p) : *p;
}

// one internal cell v from its nch children: mass and
// the sum of m x as float pairs, the children's pairs added by two_sum_acc
// (each addition errs by at most about 2^-47 of the magnitudes added, so a
// body's term collects at most depth x 2^-47 of relative error on its way
// to the root: 1.5e-13 at depth 21), the centre of mass as their float-pair
// quotient, both stored in FP64 too; second moments in FP32 by the parallel-axis rule
// from the children's, Q_v = sum_c Q_c + m_c d_c d_c^T, d_c = com_c - com_v
// formed in FP32 from the stored offsets of the centres of mass from their
// cube centres, d_c = (a_c - a_v) + (k_c - k_v) u (k the integer cube
// centres in units u = h/2, their difference exact).  The loads of all
// children are issued before the first sum: in turn they were most of a
// level's time.
template <bool QUAD, bool CG>
__device__ __forceinline__ void level_node(int64_t v, int4 pb, int nch, SysParams* sysp,
                                           const NodeTables& nt)
{
    float4 h[8], lo[8];
#pragma unroll
    for (int k = 0; k < 8; k++)
        if (k < nch) {
            h[k] = ld<CG>(&nt.dsum[2 * ((int64_t)pb.z + k)]);
            lo[k] = ld<CG>(&nt.dsum[2 * ((int64_t)pb.z + k) + 1]);
        }
    const int4 last = ld<CG>(&nt.b[pb.z + nch - 1]);
    const int4 cc = nt.c[v];
    SysParams& P = sysp[cc.w];
    float mh = 0.f, ml = 0.f, Sh[3] = {0.f, 0.f, 0.f}, Sl[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 8; k++)
        if (k < nch) {
            two_sum_acc(mh, ml, h[k].x, lo[k].x);
            two_sum_acc(Sh[0], Sl[0], h[k].y, lo[k].y);
            two_sum_acc(Sh[1], Sl[1], h[k].z, lo[k].z);
            two_sum_acc(Sh[2], Sl[2], h[k].w, lo[k].w);
        }
    const double m = widen(mh) + widen(ml);
    double com[3];
    float comf[3];
    pair_quotient(Sh, Sl, mh, ml, com, comf);
    nt.b[v] = make_int4(pb.x, last.x + last.y - pb.x, pb.z, (pb.w & 255) | (nch << 8));
    nt.dsum[2 * v] = make_float4(mh, Sh[0], Sh[1], Sh[2]);
    nt.dsum[2 * v + 1] = make_float4(ml, Sl[0], Sl[1], Sl[2]);
    double C[3];
    cube_centre(P, cc, C);
    float Q[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float av[3] = {(float)(com[0] - C[0]), (float)(com[1] - C[1]), (float)(com[2] - C[2])};
    const float uf = P.uf;
    for (int k = 0; QUAD && k < nch; k++) {
        const int64_t c = pb.z + k;
        const float4 ac = ld<CG>(&nt.a[c]);
        const int4 kc = nt.c[c];
        const float mc = ac.w;
        const float d[3] = {fmaf((float)(kc.x - cc.x), uf, ac.x - av[0]), fmaf((float)(kc.y - cc.y), uf, ac.y - av[1]),
                            fmaf((float)(kc.z - cc.z), uf, ac.z - av[2])};
        const float* qc = nt.quad + 6 * c;
        Q[0] += fmaf(mc * d[0], d[0], ld<CG>(qc));
        Q[1] += fmaf(mc * d[0], d[1], ld<CG>(qc + 1));
        Q[2] += fmaf(mc * d[0], d[2], ld<CG>(qc + 2));
        Q[3] += fmaf(mc * d[1], d[1], ld<CG>(qc + 3));
        Q[4] += fmaf(mc * d[1], d[2], ld<CG>(qc + 4));
        Q[5] += fmaf(mc * d[2], d[2], ld<CG>(qc + 5));
    }
    store_node<QUAD>(nt, v, m, com, Q, C, comf, mh + ml);
    if ((pb.w & 255) == 0) P.msys = (float)m;  // a system's root
}

constexpr int kRunSteps = 32;

// Per node: a leaf's body count (its run of bodies) and moments; an internal
// cell's number of children.  CLIMB: the thread that completes a cell's last
// child computes the cell and goes on to its parent, so no launch per level
// follows.
template <bool QUAD, bool CLIMB>
__global__ void k_leaf_nodes(const float4* body, const uint64_t* keys, const int8_t* delta, int64_t n,
                             SysParams* sysp, const Info* info, NodeTables nt)
{
    pdl_begin();
    if (capacity_failed(info)) return;
    const int64_t M = info->M;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < M; v += (int64_t)gridDim.x * blockDim.x) {
        int4 b = nt.b[v];
        const int l = b.w & 255;
        if (b.z >= 0) {  // internal
            if (!CLIMB) nt.b[v].w = l | (family(nt.fam, b.z, M) << 8);
            continue;
        }
        // the leaf's run: bodies sharing l digits with their predecessor, past
        // kRunSteps of them by bisection on the keys (a build of 2^20 bodies at
        // two points 86 ms one by one, 60 so)
        const int4 c = nt.c[v];
        int64_t e = (int64_t)b.x + 1;
        const int64_t near = min(n, e + kRunSteps);
        while (e < near && delta[e] >= l) e++;
        if (e == near && e < n && delta[e] >= l) {
            const int sh = 3 * (kMaxLevel - l);
            const uint64_t pfx = l == 0 ? 0ull : keys[b.x] >> sh;
            int64_t hi = sysp[c.w].end;
            e++;
            while (e < hi) {
                const int64_t mid = (e + hi) >> 1;
                if (l > 0 && (keys[mid] >> sh) != pfx) hi = mid;
                else e = mid + 1;
            }
        }
        b.y = (int)(e - b.x);
        b.w = l;
        nt.b[v] = b;
        double C[3];
        cube_centre(sysp[c.w], c, C);
        float Chi[3] = {0.f, 0.f, 0.f}, Clo[3] = {0.f, 0.f, 0.f};
        if (QUAD)
            for (int a = 0; a < 3; a++) {
                Chi[a] = (float)C[a];
                Clo[a] = (float)(C[a] - (double)Chi[a]);
            }
        // m and sum m x in absolute coordinates as unevaluated sums of two
        // floats (hi + lo): each product m x split exactly into p + e by
        // one FMA and added by two_sum_acc.  Over a leaf's c bodies the error
        // stays below about c 2^-46 of the largest partial sum of |terms|
        // (2.3e-13 of it for c = 16): FP64-class accuracy on the FP32 pipe,
        // which GB300 runs 64 times faster than its FP64 pipe; the pair goes
        // to the levels above, and hi + lo exactly into FP64.  Q about C in
        // FP32 alongside.
        float mh = 0.f, ml = 0.f, Sh[3] = {0.f, 0.f, 0.f}, Sl[3] = {0.f, 0.f, 0.f};
        float QC[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int j = b.x; j < b.x + b.y; j++) {
            const float4 q = body[j];
            two_sum_acc(mh, ml, q.w, 0.f);
            const float xs[3] = {q.x, q.y, q.z};
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const float p = q.w * xs[a];
                const float err = fmaf(q.w, xs[a], -p);  // q.w x = p + err exactly
                two_sum_acc(Sh[a], Sl[a], p, err);
            }
            if (QUAD) {
                const float dx = (q.x - Chi[0]) - Clo[0], dy = (q.y - Chi[1]) - Clo[1], dz = (q.z - Chi[2]) - Clo[2];
                const float wx = q.w * dx, wy = q.w * dy, wz = q.w * dz;
                QC[0] = fmaf(wx, dx, QC[0]);
                QC[1] = fmaf(wx, dy, QC[1]);
                QC[2] = fmaf(wx, dz, QC[2]);
                QC[3] = fmaf(wy, dy, QC[3]);
                QC[4] = fmaf(wy, dz, QC[4]);
                QC[5] = fmaf(wz, dz, QC[5]);
            }
        }
        const double m = widen(mh) + widen(ml);
        double com[3];
        float comf[3];
        pair_quotient(Sh, Sl, mh, ml, com, comf);
        float Q[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (QUAD) {
            const float ex = (float)(com[0] - C[0]), ey = (float)(com[1] - C[1]), ez = (float)(com[2] - C[2]);
            const float mf = (float)m;
            Q[0] = fmaf(-mf * ex, ex, QC[0]);
            Q[1] = fmaf(-mf * ex, ey, QC[1]);
            Q[2] = fmaf(-mf * ex, ez, QC[2]);
            Q[3] = fmaf(-mf * ey, ey, QC[3]);
            Q[4] = fmaf(-mf * ey, ez, QC[4]);
            Q[5] = fmaf(-mf * ez, ez, QC[5]);
        }
        store_node<QUAD>(nt, v, m, com, Q, C, comf, mh + ml);
        if (l == 0) sysp[c.w].msys = (float)m;  // a system's root
        nt.dsum[2 * v] = make_float4(mh, Sh[0], Sh[1], Sh[2]);
        nt.dsum[2 * v + 1] = make_float4(ml, Sl[0], Sl[1], Sl[2]);
        if (CLIMB) {
            for (int32_t p = nt.parent[v];;) {
                if (p < 0) break;
                const int4 pb = nt.b[p];  // (x, z and the level: written before this launch)
                const int32_t up = nt.parent[p];
                const int nch = family(nt.fam, pb.z, M);
                // the arrival releases this child's record and, the last one,
                // acquires the others'
                uint32_t old;
                asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(&nt.pend[p]) : "memory");
                if (old + 1u < (uint32_t)nch) break;
                level_node<QUAD, true>(p, pb, nch, sysp, nt);
                p = up;
            }
        }
    }
}

// internal cells of level `lev`: [level_start[lev], level_start[lev + 1])
template <bool QUAD>
__global__ void k_level_moments(int lev, const uint32_t* level_start, SysParams* sysp,
                                const Info* info, NodeTables nt)
{
    pdl_begin();
    if (capacity_failed(info)) return;
    const int64_t start = level_start[lev];
    const int64_t end = level_start[lev + 1];
    for (int64_t v = start + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < end;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int4 pb = nt.b[v];
        if (pb.z >= 0) level_node<QUAD, false>(v, pb, pb.w >> 8, sysp, nt);
    }
}

// levels lev_hi - 1 down to lev_lo in one block: those past the depth a
// captured step expects (normally none), and the topmost, which hold few
// cells
template <bool QUAD>
__global__ void __launch_bounds__(512) k_level_moments_block(int lev_hi, int lev_lo,
                                                             const uint32_t* level_start,
                                                             SysParams* sysp, const Info* info,
                                                             NodeTables nt)
{
    pdl_begin();
    if (capacity_failed(info)) return;
    for (int lev = lev_hi - 1; lev >= lev_lo; lev--) {
        const int64_t start = level_start[lev];
        const int64_t end = level_start[lev + 1];
        for (int64_t v = start + threadIdx.x; v < end; v += blockDim.x) {
            const int4 pb = nt.b[v];
            if (pb.z >= 0) level_node<QUAD, true>(v, pb, pb.w >> 8, sysp, nt);
        }
        __threadfence_block();
        __syncthreads();
    }
}

// ------------------------------------------------------------------ groups
// Bodies are walked in groups of at most gmax consecutive Morton-ordered
// bodies of one system.  A cube holding more than gmax bodies is split into
// groups: a leaf into consecutive chunks of gmax; an internal cube by packing
// runs of its consecutive children that hold at most gmax each, greedily left
// to right (children holding more than gmax are split in turn by their own
// thread).  A root holding at most gmax is one group.  Each group records a
// reference cube (itself, the leaf it was cut from, or the common parent of
// the packed children); the walk measures positions from that cube's centre.
// gref_at[s] = the reference cube + 1 of the group that starts at body s (0: none)
__global__ void k_group_marks(const Info* info, const NodeTables nt, int gmax, int32_t* gref_at)
{
    pdl_begin();
    if (capacity_failed(info)) return;
    const int64_t M = info->M;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < M; v += (int64_t)gridDim.x * blockDim.x) {
        const int4 b = nt.b[v];
        const int nch = b.w >> 8;
        if (b.y <= gmax) {
            if ((b.w & 255) == 0) gref_at[b.x] = (int32_t)v + 1;  // a root
            continue;
        }
        if (nch == 0) {
            for (int s = 0; s < b.y; s += gmax) gref_at[b.x + s] = (int32_t)v + 1;
            continue;
        }
        int2 kid[8];  // first body and bodies of each child, loaded together
#pragma unroll
        for (int k = 0; k < 8; k++)
            if (k < nch) kid[k] = *reinterpret_cast<const int2*>(&nt.b[b.z + k]);
        int run_first = -1, run_count = 0, run_len = 0, run_only = -1;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            if (k >= nch) break;
            if (kid[k].y > gmax || run_count + kid[k].y > gmax) {
                if (run_len > 0) gref_at[run_first] = (run_len == 1 ? run_only : (int32_t)v) + 1;
                run_len = 0;
                run_count = 0;
            }
            if (kid[k].y > gmax) continue;
            if (run_len == 0) {
                run_first = kid[k].x;
                run_only = b.z + k;
            }
            run_count += kid[k].y;
            run_len++;
        }
        if (run_len > 0) gref_at[run_first] = (run_len == 1 ? run_only : (int32_t)v) + 1;
    }
}

// the marked bodies in order -> the group table, one pass (which stays as it is
// where the build stopped)
__global__ void __launch_bounds__(kScanThreads) k_group_table(const int32_t* gref_at, int64_t n,
                                                              unsigned long long* st, uint32_t* counter,
                                                              int32_t* gfirst, int32_t* gref,
                                                              int32_t* part_done, Info* info)
{
    pdl_begin();
    __shared__ int tile_sh;
    __shared__ int32_t mark[kScanTile];
    if (threadIdx.x == 0) tile_sh = capacity_failed(info) ? -1 : (int)atomicAdd(counter, 1u);
    __syncthreads();
    if (tile_sh < 0) return;
    const int64_t tile = tile_sh, t0 = tile * kScanTile;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        const int p = i * kScanThreads + threadIdx.x;
        mark[p] = t0 + p < n ? gref_at[t0 + p] : 0;
    }
    __syncthreads();
    uint32_t has = 0;  // which of the thread's kScanItems consecutive bodies start a group
#pragma unroll
    for (int i = 0; i < kScanItems; i++) has |= mark[threadIdx.x * kScanItems + i] ? 1u << i : 0u;
    uint32_t total;
    bool ok;
    uint32_t g = scan_tile(__popc(has), tile, st, &total, &ok);
    if (!ok) {
        if (threadIdx.x == 0) atomicOr(&info->err, kErrWorkLoop | kErrCapacity);
        return;
    }
    for (; has; has &= has - 1, g++) {
        const int i = threadIdx.x * kScanItems + __ffs(has) - 1;
        gfirst[g] = (int32_t)(t0 + i);
        gref[g] = mark[i] - 1;
        part_done[g] = 0;
    }
    if (tile == gridDim.x - 1 && threadIdx.x == 0) {
        gfirst[total] = (int32_t)n;
        info->G = total;
    }
}

// The groups ordered by the layout the walk gives them (group_class), the
// largest first and in tree order within a class: the warps of an SM then
// sum with the same loop at the same time (the loops of all layouts together
// do not fit its instruction cache: the 2^20 cube's walk waited 2.6 cycles
// per issued instruction for fetches with the groups in tree order), and a
// walk that launches one kernel per class finds its groups in one range.
// Block b of kSplitBlocks takes the b-th contiguous range of the group
// table; a first pass counts each range's groups per class, a second gives
// every group its place (the classes before its own, the ranges before its
// own, then warp ballots within the range).
constexpr int kSplitBlocks = 256;
constexpr int kSplitThreads = 256;

__device__ __forceinline__ int group_class(const int32_t* gfirst, int64_t g)
{
    const int n = gfirst[g + 1] - gfirst[g];
    if (n > 64) return n > 96 ? 0 : 1;
    if (n > 32) return n > 48 ? 2 : (n > 40 ? 3 : 4);
    return n > 16 ? 5 : 6;
}

__device__ __forceinline__ void split_range(const Info* info, int64_t& lo, int64_t& hi)
{
    const int64_t G = capacity_failed(info) ? 0 : info->G;
    const int64_t per = (G + gridDim.x - 1) / gridDim.x;
    lo = min(G, (int64_t)blockIdx.x * per);
    hi = min(G, lo + per);
}

__device__ __forceinline__ int warp_sum_i(int v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(kSplitThreads) k_order_count(const int32_t* gfirst, const Info* info,
                                                               int32_t* bcount)
{
    pdl_begin();
    __shared__ int cnt[kGroupClasses];
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < kGroupClasses) cnt[tid] = 0;
    __syncthreads();
    int64_t lo, hi;
    split_range(info, lo, hi);
    for (int64_t c0 = lo; c0 < hi; c0 += kSplitThreads) {
        const int cls = c0 + tid < hi ? group_class(gfirst, c0 + tid) : -1;
#pragma unroll
        for (int k = 0; k < kGroupClasses; k++) {
            const unsigned m = __ballot_sync(0xffffffffu, cls == k);
            if (lane == 0 && m) atomicAdd(&cnt[k], __popc(m));
        }
    }
    __syncthreads();
    if (tid < kGroupClasses) bcount[kGroupClasses * blockIdx.x + tid] = cnt[tid];
}

__global__ void __launch_bounds__(kSplitThreads) k_order_scatter(const int32_t* gfirst, const Info* info,
                                                                 const int32_t* bcount,
                                                                 int32_t* order, int32_t* seg)
{
    pdl_begin();
    constexpr int W = kSplitThreads / 32, NC = kGroupClasses;
    __shared__ int red[W][2 * NC];
    __shared__ int wcnt[W][NC];
    __shared__ int base[NC];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // groups of each class in the ranges before this one, and in all
    int v[2 * NC];
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) v[k] = 0;
    for (int j = tid; j < (int)gridDim.x; j += blockDim.x) {
#pragma unroll
        for (int k = 0; k < NC; k++) {
            const int x = bcount[NC * j + k];
            if (j < (int)blockIdx.x) v[k] += x;
            v[NC + k] += x;
        }
    }
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) {
        const int s = warp_sum_i(v[k]);
        if (lane == 0) red[w][k] = s;
    }
    __syncthreads();
    if (tid < NC) {
        int mine = 0;
        for (int ww = 0; ww < W; ww++) mine += red[ww][tid];
        int start = 0;
        for (int k = 0; k < tid; k++)
            for (int ww = 0; ww < W; ww++) start += red[ww][NC + k];
        base[tid] = start + mine;
        if (blockIdx.x == 0) {
            // the ranges of groups of more than 64 (classes 0, 1), 33 to 64
            // (2 to 4) and up to 32 bodies
            if (tid == 0) seg[0] = 0;
            if (tid == 2) seg[1] = start;
            if (tid == 5) seg[2] = start;
            if (tid == NC - 1) {
                int all = start;
                for (int ww = 0; ww < W; ww++) all += red[ww][NC + tid];
                seg[3] = all;
            }
        }
    }
    int64_t lo, hi;
    split_range(info, lo, hi);
    const unsigned lt = (1u << lane) - 1u;
    for (int64_t c0 = lo; c0 < hi; c0 += kSplitThreads) {
        const int64_t g = c0 + tid;
        const int cls = g < hi ? group_class(gfirst, g) : -1;
        int rank = 0;
        unsigned m[NC];
#pragma unroll
        for (int k = 0; k < NC; k++) {
            m[k] = __ballot_sync(0xffffffffu, cls == k);
            if (cls == k) rank = __popc(m[k] & lt);
        }
        __syncthreads();  // base is set; the previous chunk's readers of wcnt and base are done
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < NC; k++) wcnt[w][k] = __popc(m[k]);
        __syncthreads();
        if (cls >= 0) {
            int off = base[cls] + rank;
            for (int ww = 0; ww < w; ww++) off += wcnt[ww][cls];
            order[off] = (int32_t)g;
        }
        __syncthreads();
        if (tid < NC) {
            int t = 0;
            for (int ww = 0; ww < W; ww++) t += wcnt[ww][tid];
            base[tid] += t;
        }
    }
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }
// grid of a grid-stride kernel over a device-side count bounded by cap
inline unsigned gsgrid(int64_t cap, int t)
{
    int64_t g = (cap + t - 1) / t;
    const int64_t gmax = 16 * (int64_t)sm_count();
    if (g > gmax) g = gmax;
    return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

void launch_sys_ids(const int64_t* offsets, int nsys, int64_t n, uint32_t* sys_of, SysParams* sysp, ChainStream s)
{
    const int64_t m = n > nsys ? n : nsys;
    pdl_launch(k_sys_ids, nblk(m, 256), 256, 0, s, offsets, nsys, n, sys_of, sysp);
    count_launches(1);
}

void launch_build_init(uint4* zero, int64_t nzero, SysParams* sysp, int nsys, Info* info, bool reset_err,
                       ChainStream s)
{
    const int64_t m = nzero > nsys ? nzero : nsys;
    pdl_launch(k_build_init, gsgrid(m, 256), 256, 0, s, zero, nzero, sysp, nsys, info, reset_err);
    count_launches(1);
}

void launch_bbox(const float* pos, const int4* chunks, int nchunks, SysParams* sysp, int nsys, int32_t* err,
                 ChainStream s)
{
    if (nsys <= kCubeSystems) {
        pdl_launch(k_bbox<true>, nchunks, kBboxThreads, 0, s, pos, chunks, sysp, err);
        count_launches(1);
        return;
    }
    pdl_launch(k_bbox<false>, nchunks, kBboxThreads, 0, s, pos, chunks, sysp, err);
    pdl_launch(k_cubes, nblk(nsys, 128), 128, 0, s, sysp, nsys);
    count_launches(2);
}

void launch_keys(const float* pos, const float* mass, int64_t n, const uint32_t* sys_of, const SysParams* sysp,
                 uint64_t* keys, uint32_t* idx, const SortPlan& plan, uint32_t* ghist, int32_t* err, ChainStream s)
{
    int64_t g = (n + 1023) / 1024;
    if (g > 6 * sm_count()) g = 6 * sm_count();
    pdl_launch(k_keys, g, 256, 0, s, pos, mass, n, sys_of, sysp, keys, idx, plan, ghist, err);
    count_launches(1);
}

void launch_gather(const float* pos, const float* mass, const uint32_t* perm, int64_t n, float4* body,
                   ChainStream s)
{
    pdl_launch(k_gather, nblk(n, 256), 256, 0, s, pos, mass, perm, n, body);
    count_launches(1);
}

int64_t level_counts_size(int64_t n) { return (int64_t)kLevels * ((n + kNodeBlock - 1) / kNodeBlock); }

// words of the two single-pass scans' look-back: the levels' counts, then the
// groups' marks, then two tile counters (all zeroed by the caller)
namespace {
int64_t scan_tiles(int64_t n) { return (n + kScanTile - 1) / kScanTile; }
}  // namespace
int64_t build_scan_words(int64_t n) { return scan_tiles(level_counts_size(n)) + scan_tiles(n) + 1; }

void launch_node_levels(const uint64_t* keys, const uint32_t* sys_of, int64_t n, int leaf_max, int8_t* w,
                        int8_t* delta, int8_t* top, int32_t* gref_at, uint32_t* cnt, unsigned long long* scan,
                        int64_t cap_m, Info* info, ChainStream s)
{
    const unsigned nb = nblk(n, kNodeBlock);
    if (leaf_max <= kTileWindow) {
        pdl_launch(k_node_levels_tiled, nb, kNodeThreads, 0, s, keys, sys_of, n, leaf_max, delta, top, gref_at, cnt,
                   &info->depth);
        count_launches(1);
    } else {
        pdl_launch(k_window, nblk(n, 256), 256, 0, s, keys, sys_of, n, leaf_max, w);
        pdl_launch(k_window_max, nblk(n, 256), 256, 0, s, w, n, leaf_max, top);
        pdl_launch(k_node_levels, nb, kNodeThreads, 0, s, keys, sys_of, n, delta, top, gref_at, cnt, &info->depth);
        count_launches(3);
    }
    const int64_t nc = level_counts_size(n);
    uint32_t* counters = reinterpret_cast<uint32_t*>(scan + build_scan_words(n) - 1);
    pdl_launch(k_scan_levels, scan_tiles(nc), kScanThreads, 0, s, cnt, nc, scan, counters, cap_m, info);
    count_launches(1);
}

void launch_emit_nodes(const uint64_t* keys, const int8_t* delta, const int8_t* top, const uint32_t* sys_of, int64_t n,
                       const uint32_t* offs, Info* info, uint32_t* lstart, NodeTables nt, ChainStream s)
{
    pdl_launch(k_emit_nodes, nblk(n, kNodeBlock), kNodeThreads, 0, s, keys, delta, top, sys_of, n, offs, info, lstart,
               nt);
    count_launches(1);
}

void launch_moments(const float4* body, const uint64_t* keys, const int8_t* delta, int64_t n, int nsys,
                    int64_t cap_m, int depth, int depth_hint, const uint32_t* level_start, SysParams* sysp,
                    const Info* info, NodeTables nt, bool quad, ChainStream s)
{
    const unsigned g = gsgrid(cap_m, 128);
    const bool climb = n <= kClimbBodies;
    if (climb) {
        if (quad) pdl_launch(k_leaf_nodes<true, true>, g, 128, 0, s, body, keys, delta, n, sysp, info, nt);
        else pdl_launch(k_leaf_nodes<false, true>, g, 128, 0, s, body, keys, delta, n, sysp, info, nt);
        count_launches(1);
        return;
    }
    if (quad) pdl_launch(k_leaf_nodes<true, false>, g, 128, 0, s, body, keys, delta, n, sysp, info, nt);
    else pdl_launch(k_leaf_nodes<false, false>, g, 128, 0, s, body, keys, delta, n, sysp, info, nt);
    count_launches(1);
    // the level launches take a small grid (4 blocks per SM): most levels
    // hold few internal cells, the launches past the tree's depth none, and a
    // large grid costs more to start than they work
    const unsigned glim = 4u * (unsigned)sm_count();
    const unsigned gl = g < glim ? g : glim;
    auto block = [&](int hi, int lo) {
        if (quad) pdl_launch(k_level_moments_block<true>, 1, 512, 0, s, hi, lo, level_start, sysp, info, nt);
        else pdl_launch(k_level_moments_block<false>, 1, 512, 0, s, hi, lo, level_start, sysp, info, nt);
        count_launches(1);
    };
    int top = depth < 0 ? kMaxLevel : depth;
    if (depth < 0 && depth_hint >= 0 && depth_hint + 3 < kMaxLevel) {
        // depth unknown on the host (a captured step): the levels from the
        // expected depth + 3 down get a launch each, any deeper ones one block
        top = depth_hint + 3;
        block(kMaxLevel, top);
    }
    // the topmost levels, of at most 2048 cells each, share a block too
    int few = 0;
    while (few < top && ((int64_t)nsys << (3 * few)) <= 2048) few++;
    if (few < 2) few = 0;
    for (int lev = top - 1; lev >= few; lev--) {
        if (quad) pdl_launch(k_level_moments<true>, gl, 128, 0, s, lev, level_start, sysp, info, nt);
        else pdl_launch(k_level_moments<false>, gl, 128, 0, s, lev, level_start, sysp, info, nt);
        count_launches(1);
    }
    if (few) block(few, 0);
}

void launch_groups(int64_t cap_m, Info* info, const NodeTables nt, int gmax, int64_t n, int32_t* gref_at,
                   unsigned long long* scan, int32_t* gfirst, int32_t* gref, int32_t* part_done, ChainStream s)
{
    pdl_launch(k_group_marks, gsgrid(cap_m, 128), 128, 0, s, info, nt, gmax, gref_at);
    uint32_t* counters = reinterpret_cast<uint32_t*>(scan + build_scan_words(n) - 1);
    pdl_launch(k_group_table, scan_tiles(n), kScanThreads, 0, s, gref_at, n, scan + scan_tiles(level_counts_size(n)),
               counters + 1, gfirst, gref, part_done, info);
    count_launches(2);
}

size_t group_order_scratch() { return (size_t)kGroupClasses * kSplitBlocks; }

void launch_group_order(const int32_t* gfirst, const Info* info, int32_t* order, int32_t* seg, int32_t* scratch,
                        ChainStream s)
{
    pdl_launch(k_order_count, kSplitBlocks, kSplitThreads, 0, s, gfirst, info, scratch);
    pdl_launch(k_order_scatter, kSplitBlocks, kSplitThreads, 0, s, gfirst, info, scratch, order, seg);
    count_launches(2);
}

}  // namespace tc
