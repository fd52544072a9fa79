// tc_fmm.cu -- the fast multipole method on the treecode's tree (Sec. 5
// names it as the treecode's O(N) successor and gives no formulation; the
// reading built here is stated in full in include/tc.h beside tc_ctx_fmm).
//
// Every cell carries a monopole at its centre of mass (the build's FP64
// reduction) and gets a third-order local expansion about it: the field L0,
// its Jacobian L1 (symmetric, 6 numbers), its second and third derivatives
// L2 and L3 (symmetric, 10 and 15 numbers).  The dual traversal decides which ordered pairs of
// cells interact through expansions (M2L) and which pairs of leaves
// directly (P2P): from (root, root), a pair of a cell with itself splits into
// all pairs of its children; a pair of distinct cells is accepted when
// r_A + r_B < theta |c_A - c_B| (r_X: the cell's radius about its centre of
// mass), else summed directly when both are leaves, else the target B is
// split when it is internal and (A is a leaf or r_B >= r_A), else the source
// A.  Per target cell B that is a walk: B's candidate sources are its
// parent's unresolved sources and its parent's children (B itself among
// them); B refines every candidate wider than itself, applies M2L to the
// accepted ones, and keeps the rest for its own children.  So the traversal runs level by level, top down, one warp per
// cell, and no pair list is ever written: a cell's unresolved candidates go
// to a pool its children read, and its local expansion is its parent's moved
// to its own centre (L2L) plus its own M2L terms.  A leaf walks its
// candidates to the end: accepted cells feed its expansion, leaves it meets
// send their bodies to a shared-memory tile (P2P), and its expansion and its
// parent's are evaluated at its bodies (L2P).  A leaf holds fewer bodies
// than a warp has lanes, so its P2P splits the tile: lane t + c k (c the
// leaf's bodies) sums the tile's pairs k, k + S, k + 2S, ... for body t
// (S = 32 / c slices), with the compensated summation of the treecode's
// force loop, and the slices are added at the end.
//
// One launch walks all levels: warps take the cells in breadth-first order
// and a cell waits (bounded) for its parent's record, which an earlier ticket
// holds.  With a launch per level the top levels ran alone, a few long walks
// at a time: an outlying body is a leaf of the first level whose walk meets
// the whole tree (139 us; levels 1 to 4 of a Plummer sphere 0.31 ms of 1.47
// at 250000 bodies).
//
// Bound: instructions.  A cell meets 295 accepted cells and 29 leaves on
// average (10^6 bodies, theta 0.55).  So lanes are kept filled: a round tests
// 32 candidates, the children of up to four split cells and further
// candidates in the lanes left over; accepted cells wait in shared memory
// until some 300 of them are added together, and met leaves until 32 of them
// are listed together (8.4 thousand instructions a cell with both done by the
// lanes that met them, round by round; 5.5 now).  The M2L sums live only while
// the queue is added, so the walk itself has registers to spare.  10^6 bodies:
// 3.9 ms with a launch per level, 1.91 now; 20000: 1.5 ms for a whole call,
// now 0.55, which an outlying leaf's walk of the whole tree takes.
//
// Radii are FP64 (leaves from their bodies, cells from their children's
// spheres, in one launch that climbs: the last of a cell's children to finish
// goes on with the cell), rounded to FP32 for the test; the same pass gathers
// each cell's walk record (centre of mass, cube centre, radius, body and
// child ranges) into one 48-byte run, one gather per candidate.  The
// acceptance test runs in FP32 on cell-relative values (integer cube centres
// in units of h/2 plus the float offset of each centre of mass from its cube
// centre), as the treecode walk does.
#include "tc_walk.cuh"

namespace tc {

namespace {

constexpr int kFmmWarps = 8;
constexpr unsigned kFmmChunk = 8;  // cells a block takes at a time
// split cells per warp (shared memory), each standing for up to eight sources;
// a round takes four and adds 32 at most, the newest first
constexpr int kFmmStack = 320;
constexpr int kFmmTile = 128;
constexpr int kFmmQueue = 320;   // accepted cells that wait
constexpr int kFmmBlocksPerSm = 2;
constexpr long long kFmmWaitCycles = 1ll << 31;  // about 1 s of SM clock
constexpr int kLocW = 36;         // floats per local expansion: L0 3, L1 6, L2 10, L3 15, two spare

// Symmetric storage of the expansion's coefficients: a sorted index tuple
// is stored once, in lexicographic order -- L1 (00 01 02 11 12 22), L2
// (000 001 ... 222, 10 entries), L3 (0000 ... 2222, 15 entries).  The
// positions are pure arithmetic on the indices, so in the unrolled loops
// below every one folds to a constant (the coefficients stay in registers).
__host__ __device__ constexpr int mn(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int mx(int a, int b) { return a < b ? b : a; }
// sorted pair x <= y over the alphabet 0..n-1
__host__ __device__ constexpr int si2n(int x, int y, int n) { return x * n - x * (x - 1) / 2 + (y - x); }
// sorted triples over 0..n-1 whose first element is below x
__host__ __device__ constexpr int off3n(int x, int n)
{
    return x == 0 ? 0 : (x == 1 ? n * (n + 1) / 2 : n * (n + 1) / 2 + (n - 1) * n / 2);
}
__host__ __device__ constexpr int si3s(int a, int b, int c, int n) { return off3n(a, n) + si2n(b - a, c - a, n - a); }
__host__ __device__ constexpr int si2(int i, int j) { return si2n(mn(i, j), mx(i, j), 3); }
__host__ __device__ constexpr int si3(int i, int j, int k)
{
    return si3s(mn(mn(i, j), k), i + j + k - mn(mn(i, j), k) - mx(mx(i, j), k), mx(mx(i, j), k), 3);
}
__host__ __device__ constexpr int si4(int i, int j, int k, int l)
{
    // a four-element sorting network: the extremes, then the middle pair
    return (mn(mn(i, j), mn(k, l)) == 0 ? 0 : (mn(mn(i, j), mn(k, l)) == 1 ? 10 : 14)) +
           si3s(mn(mx(mn(i, j), mn(k, l)), mn(mx(i, j), mx(k, l))) - mn(mn(i, j), mn(k, l)),
                mx(mx(mn(i, j), mn(k, l)), mn(mx(i, j), mx(k, l))) - mn(mn(i, j), mn(k, l)),
                mx(mx(i, j), mx(k, l)) - mn(mn(i, j), mn(k, l)), 3 - mn(mn(i, j), mn(k, l)));
}
static_assert(si2(2, 1) == 4 && si3(2, 0, 1) == 4 && si3(2, 1, 1) == 7 && si4(0, 1, 1, 2) == 7 &&
                  si4(2, 1, 2, 1) == 12 && si4(2, 2, 1, 2) == 13 && si4(2, 2, 2, 2) == 14 && si4(1, 0, 0, 0) == 1,
              "symmetric storage positions");

// the monomials of an offset t over the sorted pairs and triples
__device__ __forceinline__ void monomials(const float (&t)[3], float (&t2)[6], float (&t3)[10])
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++) t2[si2(i, j)] = t[i] * t[j];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++)
#pragma unroll
            for (int k = j; k < 3; k++) t3[si3(i, j, k)] = t2[si2(i, j)] * t[k];
}

// M2L: the softened field of mass gm (G M) seen from d = c_A - c_B and its
// first three derivatives with respect to the evaluation point are
//   L0_i    += gm d_i / rho^3
//   L1_ij   += gm (3 d_i d_j / rho^5 - delta_ij / rho^3)
//   L2_ijk  += gm (15 d_i d_j d_k / rho^7 - 3 (delta_ij d_k + delta_ik d_j + delta_jk d_i) / rho^5)
//   L3_ijkl += gm (105 d_i d_j d_k d_l / rho^9 - 15 (6 terms delta d d) / rho^7
//                  + 3 (3 terms delta delta) / rho^5)
// so a cell's sums are those of g_k = gm / rho^k times the monomials of d, an
// FMA each; the deltas are put in once per cell (Loc::from).
constexpr int kMoments = 45;
constexpr int kG3D = 0, kG3 = 3, kG5D = 4, kG5 = 7, kG5DD = 8, kG7DD = 14, kG7DDD = 20, kG9DDDD = 30;
struct Moments {
    float v[kMoments];
    __device__ void zero()
    {
#pragma unroll
        for (int k = 0; k < kMoments; k++) v[k] = 0.f;
    }
    __device__ void add(float gm, const float (&d)[3], float eps2)
    {
        const float r2 = fmaf(d[2], d[2], fmaf(d[1], d[1], fmaf(d[0], d[0], eps2)));
        const float ri = rsqrtf(r2);
        const float ri2 = ri * ri;
        const float g3 = gm * ri * ri2;
        const float g5 = g3 * ri2;
        const float g7 = g5 * ri2;
        const float g9 = g7 * ri2;
        float dd[6], b7[6], b9[6];
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = i; j < 3; j++) dd[si2(i, j)] = d[i] * d[j];
#pragma unroll
        for (int k = 0; k < 6; k++) {
            b7[k] = g7 * dd[k];
            b9[k] = g9 * dd[k];
        }
        v[kG3] += g3;
        v[kG5] += g5;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            v[kG3D + i] = fmaf(g3, d[i], v[kG3D + i]);
            v[kG5D + i] = fmaf(g5, d[i], v[kG5D + i]);
        }
#pragma unroll
        for (int k = 0; k < 6; k++) {
            v[kG5DD + k] = fmaf(g5, dd[k], v[kG5DD + k]);
            v[kG7DD + k] += b7[k];
        }
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = i; j < 3; j++)
#pragma unroll
                for (int k = j; k < 3; k++) {
                    v[kG7DDD + si3(i, j, k)] = fmaf(b7[si2(i, j)], d[k], v[kG7DDD + si3(i, j, k)]);
#pragma unroll
                    for (int l = k; l < 3; l++)
                        v[kG9DDDD + si4(i, j, k, l)] = fmaf(b9[si2(i, j)], dd[si2(k, l)], v[kG9DDDD + si4(i, j, k, l)]);
                }
    }
    // one step of a halving sum over the warp: of N values the lanes with bit
    // O set keep the upper half's, the others the lower half's
    template <int N, int O>
    __device__ __forceinline__ void halve()
    {
        constexpr int h = (N + 1) / 2;
        const bool up = (threadIdx.x & O) != 0;
#pragma unroll
        for (int i = 0; i < h; i++) {
            const float lo = v[i], hi = h + i < N ? v[h + i < N ? h + i : 0] : 0.f;
            v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, O);
        }
    }
    // the warp's sums, added to out[kMoments] in shared memory; at, len: sum_range()
    __device__ __forceinline__ void sum(float* out, int at, int len)
    {
        halve<45, 16>();
        halve<23, 8>();
        halve<12, 4>();
        halve<6, 2>();
        halve<3, 1>();
        if (len > 0) out[at] += v[0];
        if (len > 1) out[at + 1] += v[1];
        __syncwarp();
    }
    // the sums that this lane ends with
    __device__ static void sum_range(int* at, int* len)
    {
        int a = 0, n = kMoments;
        const int h[5] = {23, 12, 6, 3, 2};
#pragma unroll
        for (int k = 0; k < 5; k++) {
            if (threadIdx.x & (16 >> k)) {
                a += h[k];
                n -= h[k];
            } else {
                n = min(n, h[k]);
            }
        }
        *at = a;
        *len = max(n, 0);
    }
};

// The Taylor series of the field about a cell's centre to third order:
// a(c + t) = L0 + L1 t + (1/2) L2 t t + (1/6) L3 t t t (L1 the Jacobian,
// L2, L3 the second and third derivatives).
struct Loc {
    float l0[3];
    float l1[6];
    float l2[10];
    float l3[15];
    __device__ void from(const float* m)  // (shared memory)
    {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            l0[i] = m[kG3D + i];
#pragma unroll
            for (int j = i; j < 3; j++) {
                l1[si2(i, j)] = fmaf(3.f, m[kG5DD + si2(i, j)], i == j ? -m[kG3] : 0.f);
#pragma unroll
                for (int k = j; k < 3; k++) {
                    float s = 0.f;
                    if (i == j) s += m[kG5D + k];
                    if (i == k) s += m[kG5D + j];
                    if (j == k) s += m[kG5D + i];
                    l2[si3(i, j, k)] = fmaf(15.f, m[kG7DDD + si3(i, j, k)], -3.f * s);
#pragma unroll
                    for (int l = k; l < 3; l++) {
                        float s6 = 0.f;
                        if (i == j) s6 += m[kG7DD + si2(k, l)];
                        if (i == k) s6 += m[kG7DD + si2(j, l)];
                        if (i == l) s6 += m[kG7DD + si2(j, k)];
                        if (j == k) s6 += m[kG7DD + si2(i, l)];
                        if (j == l) s6 += m[kG7DD + si2(i, k)];
                        if (k == l) s6 += m[kG7DD + si2(i, j)];
                        const int s3 = (i == j && k == l) + (i == k && j == l) + (i == l && j == k);
                        l3[si4(i, j, k, l)] =
                            fmaf(105.f, m[kG9DDDD + si4(i, j, k, l)], fmaf(-15.f, s6, (float)(3 * s3) * m[kG5]));
                    }
                }
            }
        }
    }
    // the field of the series at offset t from its centre (L2P, and the L0
    // part of L2L): L0 + L1 t + (1/2) L2 t t + (1/6) L3 t t t, each sum over
    // the sorted index tuples with their multiplicities
    __device__ void eval(const float (&t)[3], const float (&t2)[6], const float (&t3)[10], float (&o)[3]) const
    {
        eval_series(l0, l1, l2, l3, t, t2, t3, o);
    }
    // the same for any storage of the 34 coefficients
    template <typename A0, typename A1, typename A2, typename A3>
    __device__ static void eval_series(const A0& l0, const A1& l1, const A2& l2, const A3& l3, const float (&t)[3],
                                       const float (&t2)[6], const float (&t3)[10], float (&o)[3])
    {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            float s = l0[i];
#pragma unroll
            for (int j = 0; j < 3; j++) s = fmaf(l1[si2(i, j)], t[j], s);
            float s2 = 0.f;
#pragma unroll
            for (int j = 0; j < 3; j++)
#pragma unroll
                for (int k = j; k < 3; k++) s2 = fmaf((float)(j == k ? 1 : 2) * l2[si3(i, j, k)], t2[si2(j, k)], s2);
            float s3 = 0.f;
#pragma unroll
            for (int j = 0; j < 3; j++)
#pragma unroll
                for (int k = j; k < 3; k++)
#pragma unroll
                    for (int m = k; m < 3; m++) {
                        const int mult = (j == k && k == m) ? 1 : ((j == k || k == m) ? 3 : 6);
                        s3 = fmaf((float)mult * l3[si4(i, j, k, m)], t3[si3(j, k, m)], s3);
                    }
            o[i] = s + 0.5f * s2 + (1.f / 6.f) * s3;
        }
    }
    // this += parent's series moved to offset t (L2L):
    //   L0 += L0p + L1p t + (1/2) L2p t t + (1/6) L3p t t t
    //   L1 += L1p + L2p t + (1/2) L3p t t,  L2 += L2p + L3p t,  L3 += L3p
    // (the parent's record q: L0 at q[0..3), L1 at q[3..9), L2 at q[9..19),
    // L3 at q[19..34))
    __device__ void add_shifted(const float* q, const float (&t)[3])
    {
        const float *p0 = q, *p1 = q + 3, *p2 = q + 9, *p3 = q + 19;
        float t2[6], t3[10];
        monomials(t, t2, t3);
        float s[3];
        eval_series(p0, p1, p2, p3, t, t2, t3, s);
#pragma unroll
        for (int i = 0; i < 3; i++) l0[i] += s[i];
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = i; j < 3; j++) {
                float u = p1[si2(i, j)];
#pragma unroll
                for (int m = 0; m < 3; m++) u = fmaf(p2[si3(i, j, m)], t[m], u);
                float w = 0.f;
#pragma unroll
                for (int m = 0; m < 3; m++)
#pragma unroll
                    for (int n = m; n < 3; n++) w = fmaf((float)(m == n ? 1 : 2) * p3[si4(i, j, m, n)], t2[si2(m, n)], w);
                l1[si2(i, j)] += fmaf(0.5f, w, u);
            }
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = i; j < 3; j++)
#pragma unroll
                for (int m = j; m < 3; m++) {
                    float u = p2[si3(i, j, m)];
#pragma unroll
                    for (int n = 0; n < 3; n++) u = fmaf(p3[si4(i, j, m, n)], t[n], u);
                    l2[si3(i, j, m)] += u;
                }
#pragma unroll
        for (int k = 0; k < 15; k++) l3[k] += p3[k];
    }
};

struct FmmArgs {
    const float4* body;      // Morton order, absolute positions, mass
    const uint32_t* perm;    // Morton position -> original index
    const SysParams* sysp;
    NodeTables nt;
    const Info* info;
    int32_t* err;
    float* loc;              // cap_m x kLocW
    int32_t* near;           // the cells' unresolved candidates
    unsigned long long* ctr; // [0] pool fill, [1] tickets, [2] pool need, [3] slab need, [4..7] statistics
    int64_t pool_cap;
    int32_t* slab;           // one list of slab_cap entries per resident warp
    int64_t slab_cap;
    int64_t* near_off;       // per node: its list in the pool
    int32_t* near_cnt;       // and its entries + 1, 0 until the node's records are in memory
    float* acc;              // n x 3, original order
    unsigned long long* rec; // per node: M2L pairs, P2P pairs, their hashes (target = the node)
    const int4* fnode;       // per node, 3 entries: {com offset, mass}, {cube centre, r_X (FP32 bits)}, b
    int records;             // keep the pair-set hashes and the per-node records
    float theta2, eps2, G;
};

// P2P of one lane: body (X, Y, Z) against the pairs k, k + S, ... of a
// pair-interleaved tile, compensated across flushes
struct P2PSum {
    float sx, sy, sz, cx, cy, cz;
    __device__ void init() { sx = sy = sz = cx = cy = cz = 0.f; }
    __device__ void flush(float* tile, int n, f2 X, f2 Y, f2 Z, f2 E2, int k, int S)
    {
        if (n <= 0) return;
        if ((n & 1) && (threadIdx.x & 31) == 0) put_entry(tile, n, make_float4(0.f, 0.f, 0.f, 0.f));
        __syncwarp();
        const int np = (n + 1) >> 1;
        const ulonglong2* t2 = reinterpret_cast<const ulonglong2*>(tile);
        f2 ax = 0ull, ay = 0ull, az = 0ull;
#pragma unroll 4
        for (int p = k; p < np; p += S) {
            const ulonglong2 xy = t2[2 * p];
            const ulonglong2 zm = t2[2 * p + 1];
            const f2 dx = f2sub(xy.x, X);
            const f2 dy = f2sub(xy.y, Y);
            const f2 dz = f2sub(zm.x, Z);
            const f2 r2 = f2fma(dz, dz, f2fma(dy, dy, f2fma(dx, dx, E2)));
            float r2a, r2b;
            f2unpack(r2, r2a, r2b);
            const f2 ri = f2pack(rsqrt_sfu(r2a), rsqrt_sfu(r2b));
            const f2 mri3 = f2mul(f2mul(zm.y, ri), f2mul(ri, ri));
            ax = f2fma(dx, mri3, ax);
            ay = f2fma(dy, mri3, ay);
            az = f2fma(dz, mri3, az);
        }
        two_sum_acc(sx, cx, f2sum(ax));
        two_sum_acc(sy, cy, f2sum(ay));
        two_sum_acc(sz, cz, f2sum(az));
        __syncwarp();
    }
};

// r_X (FP64): a leaf's farthest body from its centre of mass, above, the
// farthest child sphere.  A thread per cell starts at the leaves and climbs
// (pend: children done, zero before the launch), in one launch instead of one
// per level.  FP64 is slow (two lanes a cycle on an SM), so the farthest body
// or child is found in FP32 and only that one is computed in FP64; where the
// second comes within the FP32 values' error of the first, all are.  10^6
// bodies: 92 us, 295 with a launch per level and FP64 throughout.
constexpr float kRadiusTiny = 1e-24f;  // squares whose FP32 rounding is relative
__global__ void __launch_bounds__(128) k_fmm_radius(const float4* __restrict__ body, const SysParams* __restrict__ sysp,
                                                    NodeTables nt, double* __restrict__ rad, int4* __restrict__ fnode,
                                                    uint32_t* __restrict__ pend, const Info* info)
{
    if ((*(volatile const int32_t*)&info->err & kErrCapacity) != 0) return;  // no tree
    const int64_t M = info->M;
    const auto record = [&](int64_t v, const int4 b, const float4 na, const int4 nc, double r) {
        __stcg(&rad[v], r);
        // the walk's record of the cell, gathered into one place
        fnode[3 * v] = make_int4(__float_as_int(na.x), __float_as_int(na.y), __float_as_int(na.z), __float_as_int(na.w));
        fnode[3 * v + 1] = make_int4(nc.x, nc.y, nc.z, __float_as_int((float)r));
        fnode[3 * v + 2] = b;
    };
    for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v0 < M; v0 += (int64_t)gridDim.x * blockDim.x) {
        int64_t v = v0;
        int4 b = nt.b[v];
        if ((b.w >> 8) != 0) continue;
        double c[3] = {nt.com64[3 * v], nt.com64[3 * v + 1], nt.com64[3 * v + 2]};
        const auto body2 = [&](int i) {
            const float4 q = body[i];
            const double e0 = (double)q.x - c[0], e1 = (double)q.y - c[1], e2 = (double)q.z - c[2];
            return e0 * e0 + e1 * e1 + e2 * e2;
        };
        float hi[3], lo[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            hi[k] = (float)c[k];
            lo[k] = (float)(c[k] - (double)hi[k]);
        }
        float first = -1.f, second = -1.f;  // the largest squares
        int far = b.x;
        for (int i = b.x; i < b.x + b.y; i++) {
            const float4 q = body[i];
            const float e0 = (q.x - hi[0]) - lo[0], e1 = (q.y - hi[1]) - lo[1], e2 = (q.z - hi[2]) - lo[2];
            const float r2 = fmaf(e2, e2, fmaf(e1, e1, e0 * e0));
            if (r2 > first) {
                second = first;
                first = r2;
                far = i;
            } else {
                second = fmaxf(second, r2);
            }
        }
        double r2max = body2(far);
        if (!(second < first * (1.f - 1e-5f) && first > kRadiusTiny))  // (also infinities, NaN and underflows)
            for (int i = b.x; i < b.x + b.y; i++) r2max = fmax(r2max, body2(i));
        record(v, b, nt.a[v], nt.c[v], sqrt(r2max));
        for (;;) {
            const int32_t p = nt.parent[v];
            if (p < 0) break;
            b = nt.b[p];
            const int nch = b.w >> 8;
            // the arrival releases this child's radius and, the last one,
            // acquires the others'
            uint32_t old;
            asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(&pend[p]) : "memory");
            if (old + 1u < (uint32_t)nch) break;
            v = p;
#pragma unroll
            for (int k = 0; k < 3; k++) c[k] = nt.com64[3 * v + k];
            const float4 na = nt.a[v];
            const int4 nc = nt.c[v];
            const float uf = sysp[nc.w].uf;
            const auto sphere = [&](int64_t k) {
                const double e0 = nt.com64[3 * k] - c[0], e1 = nt.com64[3 * k + 1] - c[1], e2 = nt.com64[3 * k + 2] - c[2];
                return sqrt(e0 * e0 + e1 * e1 + e2 * e2) + __ldcg(&rad[k]);
            };
            first = second = -1.f;
            far = b.z;
#pragma unroll 4
            for (int k = b.z; k < b.z + nch; k++) {
                const float4 ka = nt.a[k];
                const int4 kc = nt.c[k];
                const float e0 = fmaf((float)(kc.x - nc.x), uf, ka.x - na.x), e1 = fmaf((float)(kc.y - nc.y), uf, ka.y - na.y),
                            e2 = fmaf((float)(kc.z - nc.z), uf, ka.z - na.z);
                const float r = sqrtf(fmaf(e2, e2, fmaf(e1, e1, e0 * e0))) + (float)__ldcg(&rad[k]);
                if (r > first) {
                    second = first;
                    first = r;
                    far = k;
                } else {
                    second = fmaxf(second, r);
                }
            }
            double r = sphere(far);
            const float side = ldexpf(uf, kMaxLevel + 1 - (b.w & 255));  // the cell's: what the offsets are rounded to
            if (!(second < first * (1.f - 1e-5f) - 1e-6f * side && side * side > kRadiusTiny))
                for (int k = b.z; k < b.z + nch; k++) r = fmax(r, sphere(k));
            record(v, b, na, nc, r);
        }
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

struct FmmWarp {  // a warp's shared memory
    float4 mq[kFmmQueue];  // accepted cells not added yet: d, G M
    float red[48];     // the sums of a cell's M2L terms
    float par[kLocW + 12];  // the parent's expansion
    float tile[4 * tile_cap(kFmmTile)];
    int2 leaves[64];   // met leaves whose bodies are not listed yet: first body, bodies
    int32_t row[32];
    uint32_t stk[kFmmStack];  // split cells: first child, children
    uint8_t stn[kFmmStack];
};
static_assert(sizeof(FmmWarp) % 16 == 0 && kFmmQueue >= 64, "a warp's shared memory");

// One lane: the warp's next cell.  A block takes kFmmChunk cells in a row from
// the device's counter, so that its warps walk siblings, whose candidates are
// much the same, at the same time (250000 bodies: L2 sends 32 million sectors,
// 112 million when the warps of small blocks took single cells).
// state: the next chunk's first cell << 8 | its cells taken, kFmmChunk + 1
// while a warp fetches the next chunk.
__device__ __forceinline__ int64_t next_cell(unsigned long long* state, unsigned long long* counter, int64_t M,
                                             int32_t* err)
{
    const long long t0 = clock64();
    for (;;) {
        const unsigned long long s = *(volatile unsigned long long*)state;
        const unsigned used = (unsigned)s & 255u;
        if (used <= kFmmChunk) {
            if (atomicCAS(state, s, s + 1) == s) {
                if (used < kFmmChunk) return (int64_t)(s >> 8) + used;
                const unsigned long long b = atomicAdd(counter, (unsigned long long)kFmmChunk);
                atomicExch(state, (b << 8) | 1ull);
                return (int64_t)b;
            }
        } else if (clock64() - t0 > kFmmWaitCycles) {
            atomicOr(err, kErrWorkLoop);
            return M;
        }
    }
}

// one warp per cell, in breadth-first order: the target walk described above
__global__ void __launch_bounds__(kFmmWarps * 32, kFmmBlocksPerSm) k_fmm_walk(FmmArgs a)
{
    extern __shared__ __align__(16) unsigned char fmm_smem[];
    __shared__ unsigned long long cells;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    FmmWarp& W = reinterpret_cast<FmmWarp*>(fmm_smem)[w];
    uint32_t* stk = W.stk;
    uint8_t* stn = W.stn;
    float* btile = W.tile;
    int32_t* slab = a.slab + ((int64_t)blockIdx.x * kFmmWarps + w) * a.slab_cap;
    const uint32_t lt = (1u << lane) - 1u, le = lt | (1u << lane);
    if ((*(volatile const int32_t*)&a.info->err & kErrCapacity) != 0) return;  // no tree
    const int64_t M = a.info->M;
    const NodeTables nt = a.nt;
    const f2 E2 = f2pack(a.eps2, a.eps2);
    int at, len;
    Moments::sum_range(&at, &len);
    unsigned long long t_m2l = 0, t_p2p = 0, th_m2l = 0, th_p2p = 0;  // the warp's totals
    if (threadIdx.x == 0) cells = kFmmChunk;
    __syncthreads();
    for (;;) {
        long long next = 0;
        if (lane == 0) next = next_cell(&cells, &a.ctr[1], M, a.err);
        const int64_t B = __shfl_sync(0xffffffffu, next, 0);
        if (B >= M) break;
        const int4 b0 = __ldg(a.fnode + 3 * B), bc = __ldg(a.fnode + 3 * B + 1), bb = __ldg(a.fnode + 3 * B + 2);
        const float bx = __int_as_float(b0.x), by = __int_as_float(b0.y), bz = __int_as_float(b0.z);
        const SysParams& SP = a.sysp[__ldg(&nt.c[B].w)];
        const float uf = SP.uf;
        const bool leafB = (bb.w >> 8) == 0;
        const float rB = __int_as_float(bc.w);
        const int P = nt.parent[B];
        // candidates: the parent's unresolved sources, then its children; a
        // root has none, or itself when it is a leaf
        int np = 0, nch = 0, pz = 0;
        int64_t poff = 0;
        if (P >= 0) {
            const int4 pb = __ldg(a.fnode + 3 * (int64_t)P + 2);
            nch = pb.w >> 8;
            pz = pb.z;
            // the parent's records.  Its ticket is an earlier one, though it
            // may still be untaken among the eight that another block holds.
            // The wait ends: of the unfinished cells the first waits for
            // nobody, and if it is untaken, the warps of the block that holds
            // it are at cells of earlier tickets (a block takes its cells in
            // order), which are finished, so one of them takes it
            if (lane == 0) {
                volatile const int32_t* done = &a.near_cnt[P];
                const long long t0 = clock64();
                while ((np = *done) == 0) {
                    if (clock64() - t0 > kFmmWaitCycles) break;
                    __nanosleep(100);
                }
                __threadfence();
            }
            np = __shfl_sync(0xffffffffu, np, 0) - 1;
            if (np < 0) {
                if (lane == 0) atomicOr(a.err, kErrWorkLoop);
                break;
            }
            __syncwarp();  // (the last cell's reads of W.par)
            poff = __ldcg(&a.near_off[P]);
            // its expansion, needed after the walk
            if (lane < kLocW / 4) cp_async16(W.par + 4 * lane, a.loc + (int64_t)P * kLocW + 4 * lane);
        } else if (leafB) {
            nch = 1;
            pz = (int)B;
        }
        const int ntot = np + nch;
        const int32_t* near = a.near + poff;
        // a leaf's bodies, 32 per round (one per lane)
        const int rounds = leafB ? max(1, (bb.y + 31) >> 5) : 1;
        for (int r = 0; r < rounds; r++) {
            // lane = t + c k: body t of this round, tile slice k of S
            const int c = leafB ? min(32, bb.y - 32 * r) : 32;
            const int S = 32 / c;
            const int t = lane % c, ks = lane / c;
            const bool slice = leafB && ks < S;
            const int ib = 32 * r + t;
            float4 me = make_float4(0.f, 0.f, 0.f, 0.f);
            if (slice) me = a.body[bb.x + ib];
            const f2 XA = f2pack(me.x, me.x), YA = f2pack(me.y, me.y), ZA = f2pack(me.z, me.z);
            P2PSum fsum;
            fsum.init();
            const int k0 = slice ? ks : (1 << 30);  // lanes past the slices sum nothing
            if (lane < 24) W.red[lane] = W.red[24 + lane] = 0.f;
            int sp = 0, ip = 0, bn = 0, mn = 0, ln = 0;
            int64_t nn = 0;
            bool bad = false, more = true;
            unsigned n_m2l = 0, n_p2p = 0;                 // this cell's pairs
            unsigned long long h_m2l = 0, h_p2p = 0;       // their hashes (per lane)
            while (more) {
                more = sp > 0 || ip < ntot;
                if (more) {
                    // the children of up to four split cells, then candidates
                    const int ne = min(sp, 4);
                    sp -= ne;
                    int A = -1;
                    if (lane < 8 * ne) {
                        const int e = sp + (lane >> 3);
                        if ((lane & 7) < (int)stn[e]) A = (int)stk[e] + (lane & 7);
                    } else {
                        const int k = ip + lane - 8 * ne;
                        if (k < ntot) A = k < np ? __ldcg(near + k) : pz + (k - np);
                    }
                    ip += 32 - 8 * ne;
                    bool m2l = false, p2p = false, keep = false, split = false;
                    int4 ab = make_int4(0, 0, 0, 0);
                    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (A >= 0) {
                        // the candidate's record: one 48-byte run
                        const int4* fr = a.fnode + 3 * (int64_t)A;
                        const int4 a0 = __ldg(fr), ac = __ldg(fr + 1);
                        ab = __ldg(fr + 2);
                        const bool leafA = (ab.w >> 8) == 0;
                        q.x = fmaf((float)(ac.x - bc.x), uf, __int_as_float(a0.x) - bx);
                        q.y = fmaf((float)(ac.y - bc.y), uf, __int_as_float(a0.y) - by);
                        q.z = fmaf((float)(ac.z - bc.z), uf, __int_as_float(a0.z) - bz);
                        q.w = a.G * __int_as_float(a0.w);
                        const float rA = __int_as_float(ac.w);
                        const float d2 = fmaf(q.z, q.z, fmaf(q.y, q.y, q.x * q.x));
                        const float rr = rA + rB;
                        const bool self = A == (int)B;  // an internal cell's self pair is its children's pairs
                        m2l = !self && rr * rr < a.theta2 * d2;
                        p2p = !m2l && leafB && (leafA || self);
                        keep = !m2l && !self && !leafB && (leafA || rB >= rA);
                        split = !m2l && !self && !p2p && !keep;
                        if (a.records && r == 0 && (m2l || p2p)) {
                            const unsigned long long hh = mix64(((unsigned long long)(unsigned)A << 32) ^ (unsigned long long)B);
                            if (m2l) h_m2l += hh;
                            else h_p2p += hh;
                        }
                    }
                    const unsigned mm = __ballot_sync(0xffffffffu, m2l), pm = __ballot_sync(0xffffffffu, p2p);
                    const unsigned sm = __ballot_sync(0xffffffffu, split);
                    // refined sources: their children are tested next
                    if (sp + __popc(sm) > kFmmStack) {
                        bad = true;
                        break;
                    }
                    if (split) {
                        stk[sp + __popc(sm & lt)] = (uint32_t)ab.z;
                        stn[sp + __popc(sm & lt)] = (uint8_t)(ab.w >> 8);
                    }
                    sp += __popc(sm);
                    if (m2l) W.mq[mn + __popc(mm & lt)] = q;
                    mn += __popc(mm);
                    n_m2l += __popc(mm);
                    if (p2p) W.leaves[ln + __popc(pm & lt)] = make_int2(ab.x, ab.y);
                    ln += __popc(pm);
                    n_p2p += __popc(pm);
                    if (!leafB) {
                        // unresolved sources go to the warp's slab (counted past its end)
                        const unsigned km = __ballot_sync(0xffffffffu, keep);
                        if (keep) {
                            const int64_t to = nn + __popc(km & lt);
                            if (to < a.slab_cap) slab[to] = A;
                        }
                        nn += __popc(km);
                    }
                }
                __syncwarp();
                if (mn > kFmmQueue - 32 || (!more && mn > 0)) {
                    Moments mom;
                    mom.zero();
#pragma unroll 1
                    for (int i = lane; i < mn; i += 32) {
                        const float4 q = W.mq[i];
                        const float d[3] = {q.x, q.y, q.z};
                        mom.add(q.w, d, a.eps2);
                    }
                    mom.sum(W.red, at, len);
                    mn = 0;
                }
                if (ln >= 32 || (!more && ln > 0)) {
                    // the bodies of the last m leaves to the tile, 32 at a
                    // time: row[r] turns a body's offset among them into its
                    // index, r found by counting the leaves that start at or
                    // before it
                    const int m = min(ln, 32);
                    ln -= m;
                    int2 lf = make_int2(0, 0);
                    if (lane < m) lf = W.leaves[ln + lane];
                    const int incl = warp_incl_scan_i(lf.y);
                    const int excl = incl - lf.y;
                    const int T = __shfl_sync(0xffffffffu, incl, 31);
                    W.row[lane] = lf.x - excl;
                    __syncwarp();
                    int rb = -1;
                    for (int o = 0; o < T; o += 32) {
                        const unsigned st = (unsigned)(excl - o);
                        const unsigned starts = __reduce_or_sync(0xffffffffu, lane < m && st < 32u ? 1u << st : 0u);
                        if (o + lane < T)
                            put_entry(btile, bn + lane, __ldg(&a.body[W.row[rb + __popc(starts & le)] + o + lane]));
                        rb += __popc(starts);
                        bn += min(32, T - o);
                        if (bn >= kFmmTile) {
                            __syncwarp();
                            fsum.flush(btile, bn, XA, YA, ZA, E2, k0, S);
                            bn = 0;
                        }
                    }
                }
                __syncwarp();
            }
            if (bad) {
                cp_async_wait_all();
                if (lane == 0) {
                    atomicOr(a.err, kErrFmmStack);
                    if (!leafB) {
                        a.near_off[B] = 0;
                        __threadfence();
                        *(volatile int32_t*)&a.near_cnt[B] = 1;
                    }
                }
                __syncwarp();
                break;
            }
            if (r == 0) {
                // this cell's pair records
                t_m2l += n_m2l;
                t_p2p += n_p2p;
                if (a.records) {
#pragma unroll
                    for (int o = 16; o; o >>= 1) {
                        h_m2l += __shfl_xor_sync(0xffffffffu, h_m2l, o);
                        h_p2p += __shfl_xor_sync(0xffffffffu, h_p2p, o);
                    }
                    th_m2l += h_m2l;
                    th_p2p += h_p2p;
                    if (lane == 0)
                        reinterpret_cast<ulonglong4_32a*>(a.rec)[B] = make_ulonglong4_32a(n_m2l, n_p2p, h_m2l, h_p2p);
                }
            }
            float4 pa = make_float4(0.f, 0.f, 0.f, 0.f);
            int4 pc = bc;
            if (P >= 0) {
                const int4 p0 = __ldg(a.fnode + 3 * (int64_t)P);
                pa = make_float4(__int_as_float(p0.x), __int_as_float(p0.y), __int_as_float(p0.z), 0.f);
                pc = __ldg(a.fnode + 3 * (int64_t)P + 1);
                cp_async_wait_all();
                __syncwarp();
            }
            // this cell's centre of mass seen from its parent's
            const float sh3[3] = {fmaf((float)(bc.x - pc.x), uf, bx - pa.x), fmaf((float)(bc.y - pc.y), uf, by - pa.y),
                                  fmaf((float)(bc.z - pc.z), uf, bz - pa.z)};
            Loc L;
            if (leafB) {
                // the cube's centre (absolute, FP64) as two floats, an axis a lane
                const int ax = lane % 3;
                const double cd = SP.c0[ax] + (double)(ax == 0 ? bc.x : (ax == 1 ? bc.y : bc.z)) * (0.5 * SP.h);
                const float ch = (float)cd, cl = (float)(cd - (double)ch);
                float hi[3], lo[3];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    hi[k] = __shfl_sync(0xffffffffu, ch, k);
                    lo[k] = __shfl_sync(0xffffffffu, cl, k);
                }
                fsum.flush(btile, bn, XA, YA, ZA, E2, k0, S);
                // the slices' sums, added by the lanes of slice 0 (through the tile)
                float fx = 0.f, fy = 0.f, fz = 0.f;
                btile[3 * lane + 0] = fsum.sx + fsum.cx;
                btile[3 * lane + 1] = fsum.sy + fsum.cy;
                btile[3 * lane + 2] = fsum.sz + fsum.cz;
                __syncwarp();
                if (ks == 0) {
                    for (int k = 0; k < S; k++) {
                        fx += btile[3 * (t + c * k) + 0];
                        fy += btile[3 * (t + c * k) + 1];
                        fz += btile[3 * (t + c * k) + 2];
                    }
                    // L2P at the lane's body: the cell's own terms at its
                    // offset from the cell's centre of mass, the parent's
                    // expansion at that from the parent's
                    const float ot[3] = {((me.x - hi[0]) - lo[0]) - bx, ((me.y - hi[1]) - lo[1]) - by,
                                         ((me.z - hi[2]) - lo[2]) - bz};
                    float o2[6], o3[10], lc[3], lp[3] = {0.f, 0.f, 0.f};
                    if (P >= 0) {
                        const float pt[3] = {ot[0] + sh3[0], ot[1] + sh3[1], ot[2] + sh3[2]};
                        monomials(pt, o2, o3);
                        Loc::eval_series(W.par, W.par + 3, W.par + 9, W.par + 19, pt, o2, o3, lp);
                    }
                    monomials(ot, o2, o3);
                    L.from(W.red);
                    L.eval(ot, o2, o3, lc);
                    const int64_t o = a.perm[bb.x + ib];
                    a.acc[3 * o + 0] = fmaf(a.G, fx, lc[0] + lp[0]);
                    a.acc[3 * o + 1] = fmaf(a.G, fy, lc[1] + lp[1]);
                    a.acc[3 * o + 2] = fmaf(a.G, fz, lc[2] + lp[2]);
                }
                __syncwarp();
                continue;
            }
            // plus the parent's expansion moved to this centre (L2L)
            L.from(W.red);
            if (P >= 0) L.add_shifted(W.par, sh3);
            long long off = -1;
            if (lane == 0) {
                float o[kLocW];
#pragma unroll
                for (int k = 0; k < 3; k++) o[k] = L.l0[k];
#pragma unroll
                for (int k = 0; k < 6; k++) o[3 + k] = L.l1[k];
#pragma unroll
                for (int k = 0; k < 10; k++) o[9 + k] = L.l2[k];
#pragma unroll
                for (int k = 0; k < 15; k++) o[19 + k] = L.l3[k];
                o[34] = o[35] = 0.f;
                float4* to = reinterpret_cast<float4*>(a.loc + B * kLocW);
#pragma unroll
                for (int k = 0; k < kLocW / 4; k++)
                    __stcg(to + k, make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]));
                // the unresolved candidates, from the slab to the pool
                if (nn > a.slab_cap) {
                    atomicMax(&a.ctr[3], (unsigned long long)nn);
                    atomicOr(a.err, kErrFmmSlab);
                } else {
                    const unsigned long long o0 = atomicAdd(&a.ctr[0], (unsigned long long)nn);
                    if ((int64_t)(o0 + nn) > a.pool_cap) {
                        atomicMax(&a.ctr[2], o0 + nn);
                        atomicOr(a.err, kErrFmmPool);
                    } else {
                        off = (long long)o0;
                    }
                }
            }
            off = __shfl_sync(0xffffffffu, off, 0);
            if (off >= 0)
                for (int64_t k = lane; k < nn; k += 32) __stcg(&a.near[off + k], slab[k]);
            __threadfence();  // the records, before the count that says so
            __syncwarp();
            if (lane == 0) {
                __stcg(&a.near_off[B], off < 0 ? (int64_t)0 : (int64_t)off);
                __threadfence();
                *(volatile int32_t*)&a.near_cnt[B] = off < 0 ? 1 : (int32_t)nn + 1;
            }
            __syncwarp();
        }
    }
    if (lane == 0 && (t_m2l | t_p2p)) {
        atomicAdd(&a.ctr[4], t_m2l);
        atomicAdd(&a.ctr[5], t_p2p);
        atomicAdd(&a.ctr[6], th_m2l);
        atomicAdd(&a.ctr[7], th_p2p);
    }
}

int fmm_grid_max() { return kFmmBlocksPerSm * sm_count(); }

}  // namespace

int64_t fmm_slab_warps() { return (int64_t)fmm_grid_max() * kFmmWarps; }
int fmm_loc_width() { return kLocW; }

cudaError_t launch_fmm(const FmmLaunch& p, cudaStream_t s)
{
    int64_t g = (p.cap_m + 127) / 128;
    if (g > 16 * sm_count()) g = 16 * sm_count();
    k_fmm_radius<<<(unsigned)(g < 1 ? 1 : g), 128, 0, s>>>(p.body, p.sysp, p.nt, p.rad, p.fnode, p.pend, p.info);
    FmmArgs a;
    a.body = p.body;
    a.perm = p.perm;
    a.sysp = p.sysp;
    a.nt = p.nt;
    a.info = p.info;
    a.err = p.err;
    a.loc = p.loc;
    a.near = p.pool;
    a.ctr = p.ctr;
    a.pool_cap = p.pool_cap;
    a.slab = p.slab;
    a.slab_cap = p.slab_cap;
    a.near_off = p.near_off;
    a.near_cnt = p.near_cnt;
    a.acc = p.acc;
    a.rec = p.rec;
    a.fnode = p.fnode;
    a.records = p.records;
    a.theta2 = p.theta * p.theta;
    a.eps2 = p.eps * p.eps;
    a.G = p.G;
    int64_t blocks = (p.cap_m + kFmmWarps - 1) / kFmmWarps;
    if (blocks > fmm_grid_max()) blocks = fmm_grid_max();
    const int smem = kFmmWarps * (int)sizeof(FmmWarp);
    const cudaError_t e = cudaFuncSetAttribute(k_fmm_walk, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_fmm_walk<<<(unsigned)(blocks < 1 ? 1 : blocks), kFmmWarps * 32, smem, s>>>(a);
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace tc
