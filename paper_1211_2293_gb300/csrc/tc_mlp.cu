// tc_mlp.cu -- the learned far-field correction's network on the GPU:
// batch inference, training (forward, backward, Adam) and the exact labels
// of training pairs.
//
// Network: 13 -> 64 -> 64 -> 3, ReLU after the hidden layers, BF16 operands
// on the tensor cores (warp-level mma.sync m16n8k16), FP32 accumulation,
// FP32 master weights.  Every kernel works on 16-row tiles, one warp each.
//
// Training loss: L = (1/B) sum_i w_i |y_i - t_i|^2 over a mini-batch of B
// pairs (targets pre-divided by the output scale; w_i = 1 without weights).
// Backward, per 16-row tile:
//   dY = 2 w (Y - T) / B,  dW3 = H2^T dY,  dH2 = (dY W3^T) * [H2 > 0],
//   dW2 = H1^T dH2,      dH1 = (dH2 W2^T) * [H1 > 0],   dW1 = X^T dH1,
// biases by column sums; the transposed operands are staged in shared
// memory and read with ldmatrix.  Every warp sums its tiles' gradient into a
// partial of its own; the partials are added in warp order.
#include <cuda_bf16.h>

#include "tc_internal.cuh"
#include "tc_mma.cuh"

namespace tc {

namespace {

constexpr int kTrainWarps = 4;

// padded gradient layout in shared memory
constexpr int kGW1 = 0;                                   // [16][64]
constexpr int kGB1 = kGW1 + kMlpInPad * kMlpHid;          // [64]
constexpr int kGW2 = kGB1 + kMlpHid;                      // [64][64]
constexpr int kGB2 = kGW2 + kMlpHid * kMlpHid;            // [64]
constexpr int kGW3 = kGB2 + kMlpHid;                      // [64][8]
constexpr int kGB3 = kGW3 + kMlpHid * kMlpOutPad;         // [8]
constexpr int kGPad = kGB3 + kMlpOutPad;

// per-warp staging (BF16): X, H1, H2, dY, dH2, dH1 of a 16-row tile, row-major;
// rows of 48, 144 and 16 bytes, so that the eight rows an ldmatrix reads lie
// in distinct banks
constexpr int kLdX = 24, kLdH = 72, kLdY = 8;
constexpr int kStX = 0;
constexpr int kStH1 = kStX + 16 * kLdX;
constexpr int kStH2 = kStH1 + 16 * kLdH;
constexpr int kStDY = kStH2 + 16 * kLdH;
constexpr int kStDH2 = kStDY + 16 * kLdY;
constexpr int kStDH1 = kStDH2 + 16 * kLdH;
constexpr int kStSize = kStDH1 + 16 * kLdH;

// store a C tile (16 x 8, column block nb) into a row-major BF16 matrix
__device__ __forceinline__ void store_c(__nv_bfloat16* M, int ld, int nb, const float (&c)[4], int lane)
{
    const int g = lane >> 2, q = lane & 3;
    *reinterpret_cast<uint32_t*>(&M[g * ld + nb * 8 + 2 * q]) = pack_bf16(c[0], c[1]);
    *reinterpret_cast<uint32_t*>(&M[(g + 8) * ld + nb * 8 + 2 * q]) = pack_bf16(c[2], c[3]);
}

// A fragment of the transpose of a row-major BF16 matrix S (S is k x m:
// A[m][k] = S[k][m]), m-tile mt, one 16-deep k-step at k = 0
__device__ __forceinline__ void load_at(uint32_t (&a)[4], const __nv_bfloat16* S, int ld, int mt, int lane)
{
    // matrices: (k 0-7, m 0-7), (k 0-7, m 8-15), (k 8-15, m 0-7), (k 8-15, m 8-15)
    const int i = lane >> 3, r = lane & 7;
    const uint32_t p = (uint32_t)__cvta_generic_to_shared(&S[(r + 8 * (i >> 1)) * ld + mt * 16 + 8 * (i & 1)]);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(p)
                 : "memory");
}

// B fragment of a row-major BF16 matrix S (B[k][n] = S[k][n]), k-step 0,
// column block nb
__device__ __forceinline__ void load_bs(uint32_t (&b)[2], const __nv_bfloat16* S, int ld, int nb, int lane)
{
    const uint32_t p = (uint32_t)__cvta_generic_to_shared(&S[(lane & 15) * ld + nb * 8]);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(b[0]), "=r"(b[1])
                 : "r"(p)
                 : "memory");
}

// B fragment of the transpose of a k-major weight W[n][k] (B[k][n] = W[n][k]
// with W stored [n][ldk]), k-step ks, column block nb
__device__ __forceinline__ void load_bt(uint32_t (&b)[2], const __nv_bfloat16* W, int ldk, int ks, int nb, int lane)
{
    const int g = lane >> 2, q = lane & 3;
    const uint32_t* w = reinterpret_cast<const uint32_t*>(&W[(nb * 8 + g) * ldk + ks * 16 + 2 * q]);
    b[0] = w[0];
    b[1] = w[4];
}

// a C tile into the warp's own partial gradient G: each element belongs to
// the same lane for every tile, so the sums are plain additions in the warp's
// order of tiles (the first tile's are stored)
__device__ __forceinline__ void add_c(float* G, int ld, int mt, int nb, const float (&c)[4], int lane, bool first)
{
    const int g = lane >> 2, q = lane & 3;
    float2* p0 = reinterpret_cast<float2*>(&G[(mt * 16 + g) * ld + nb * 8 + 2 * q]);
    float2* p1 = reinterpret_cast<float2*>(&G[(mt * 16 + g + 8) * ld + nb * 8 + 2 * q]);
    float2 a = make_float2(c[0], c[1]), b = make_float2(c[2], c[3]);
    if (!first) {
        const float2 x = *p0, y = *p1;
        a.x += x.x;
        a.y += x.y;
        b.x += y.x;
        b.y += y.y;
    }
    *p0 = a;
    *p1 = b;
}

// column sums of a C tile over its 16 rows into G[col]
__device__ __forceinline__ void colsum_c(float* G, int nb, const float (&c)[4], int lane, bool first)
{
    float s0 = c[0] + c[2], s1 = c[1] + c[3];
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if (lane < 4) {
        float2* p = reinterpret_cast<float2*>(&G[nb * 8 + 2 * lane]);
        float2 v = make_float2(s0, s1);
        if (!first) {
            const float2 x = *p;
            v.x += x.x;
            v.y += x.y;
        }
        *p = v;
    }
}

// the same of all eight column blocks: each exchange halves the values a lane
// still sums (the same pairs are added as above, 14 shuffles instead of 48)
__device__ __forceinline__ void colsum_c8(float* G, const float (&c)[8][4], int lane, bool first)
{
    float v[16];
#pragma unroll
    for (int nb = 0; nb < 8; nb++) {
        v[2 * nb] = c[nb][0] + c[nb][2];
        v[2 * nb + 1] = c[nb][1] + c[nb][3];
    }
#pragma unroll
    for (int h = 8, o = 4; h > 1; h >>= 1, o <<= 1)
#pragma unroll
        for (int i = 0; i < h; i++) {
            const bool up = (lane & o) != 0;
            const float got = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[h + i], o);
            v[i] = (up ? v[h + i] : v[i]) + got;
        }
    const int nb = (lane & 4) | ((lane >> 2) & 2) | (lane >> 4);
    float2* p = reinterpret_cast<float2*>(&G[nb * 8 + 2 * (lane & 3)]);
    float2 x = make_float2(v[0], v[1]);
    if (!first) {
        const float2 y = *p;
        x.x += y.x;
        x.y += y.y;
    }
    *p = x;
}

// what a lane holds of a tile's rows before the network runs: row r0 = tile x
// 16 + g and r0 + 8, features 2q, 2q + 1, 2q + 8, 2q + 9 of each, the targets
// of its output columns 2q, 2q + 1 and the loss weights (rows past B: zero)
struct TrainRows {
    float a[8];
    float t[4];
    float w[2];
    bool v[2];
};

// a lane's two row indices of a tile (-1 past B)
__device__ __forceinline__ int2 train_index(const int32_t* __restrict__ idx, int B, int tile, int lane)
{
    const int row = tile * 16 + (lane >> 2);
    return make_int2(row < B ? idx[row] : -1, row + 8 < B ? idx[row + 8] : -1);
}

__device__ __forceinline__ TrainRows train_rows(const float* __restrict__ X, const float* __restrict__ T,
                                                const float* __restrict__ W, int2 index, int lane)
{
    TrainRows r;
    const int q = lane & 3;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int at = h ? index.y : index.x;
        r.v[h] = at >= 0;
        const int64_t i = r.v[h] ? at : 0;
        const float2 z = make_float2(0.f, 0.f);
        const float2 lo = r.v[h] ? *reinterpret_cast<const float2*>(&X[i * kMlpInPad + 2 * q]) : z;
        const float2 hi = r.v[h] ? *reinterpret_cast<const float2*>(&X[i * kMlpInPad + 2 * q + 8]) : z;
        r.a[2 * h] = lo.x;
        r.a[2 * h + 1] = lo.y;
        r.a[4 + 2 * h] = hi.x;
        r.a[4 + 2 * h + 1] = hi.y;
        r.t[2 * h] = r.v[h] && 2 * q < kMlpOut ? T[i * kMlpOut + 2 * q] : 0.f;
        r.t[2 * h + 1] = r.v[h] && 2 * q + 1 < kMlpOut ? T[i * kMlpOut + 2 * q + 1] : 0.f;
        r.w[h] = W && r.v[h] ? W[i] : 1.f;
    }
    return r;
}

__device__ __forceinline__ TrainRows train_rows(const float* __restrict__ X, const float* __restrict__ T,
                                                const float* __restrict__ W, const int32_t* __restrict__ idx, int B,
                                                int tile, int lane)
{
    return train_rows(X, T, W, train_index(idx, B, tile, lane), lane);
}

// Forward and backward of one 16-row tile on one warp: the matrices of the
// gradient's products into st, the gradients of the biases into b1, b2, b3,
// the weighted squared errors onto lsum.
__device__ __forceinline__ void tile_backward(const MlpDev& m, const TrainRows& r, __nv_bfloat16* st, float* b1, float* b2,
                                              float* b3, bool first, float inv_b, float& lsum, int lane)
{
    const int g = lane >> 2, q = lane & 3;
    uint32_t x[4];
#pragma unroll
    for (int k = 0; k < 4; k++) x[k] = pack_bf16(r.a[2 * k], r.a[2 * k + 1]);
    // X tile, row-major, for dW1 = X^T dH1
    *reinterpret_cast<uint32_t*>(&st[kStX + g * kLdX + 2 * q]) = x[0];
    *reinterpret_cast<uint32_t*>(&st[kStX + (g + 8) * kLdX + 2 * q]) = x[1];
    *reinterpret_cast<uint32_t*>(&st[kStX + g * kLdX + 2 * q + 8]) = x[2];
    *reinterpret_cast<uint32_t*>(&st[kStX + (g + 8) * kLdX + 2 * q + 8]) = x[3];
    float h1[8][4], h2[8][4], y[4];
    mlp16(m.frag, x, h1, h2, y, lane);
    // dY = 2 w (Y - T) / B on the 3 used columns of valid rows
    float dy[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int h = k >> 1;
        if (r.v[h] && 2 * q + (k & 1) < kMlpOut) {
            const float e = y[k] - r.t[k];
            lsum += r.w[h] * e * e;
            dy[k] = 2.f * r.w[h] * e * inv_b;
        }
    }
#pragma unroll
    for (int nb = 0; nb < 8; nb++) {
        store_c(st + kStH1, kLdH, nb, h1[nb], lane);
        store_c(st + kStH2, kLdH, nb, h2[nb], lane);
    }
    store_c(st + kStDY, kLdY, 0, dy, lane);
    colsum_c(b3, 0, dy, lane, first);
    // dH2 = dY W3^T * [H2 > 0]; dY padded to a 16-deep k-step with zeros
    float dh2[8][4];
    {
        const uint32_t a[4] = {pack_bf16(dy[0], dy[1]), pack_bf16(dy[2], dy[3]), 0u, 0u};
#pragma unroll
        for (int nb = 0; nb < 8; nb++) {
            const uint32_t b[2] = {*reinterpret_cast<const uint32_t*>(&m.w3[(nb * 8 + g) * kMlpOutPad + 2 * q]), 0u};
            dh2[nb][0] = dh2[nb][1] = dh2[nb][2] = dh2[nb][3] = 0.f;
            mma_bf16(dh2[nb], a, b);
#pragma unroll
            for (int e = 0; e < 4; e++) dh2[nb][e] = h2[nb][e] > 0.f ? dh2[nb][e] : 0.f;
            store_c(st + kStDH2, kLdH, nb, dh2[nb], lane);
        }
    }
    // dH1 = dH2 W2^T * [H1 > 0]
    float dh1[8][4];
#pragma unroll
    for (int nb = 0; nb < 8; nb++) dh1[nb][0] = dh1[nb][1] = dh1[nb][2] = dh1[nb][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 4; ks++) {
        uint32_t a[4];
        c_to_a(a, dh2[2 * ks], dh2[2 * ks + 1]);
#pragma unroll
        for (int nb = 0; nb < 8; nb++) {
            uint32_t b[2];
            load_bt(b, m.w2, kMlpHid, ks, nb, lane);
            mma_bf16(dh1[nb], a, b);
        }
    }
#pragma unroll
    for (int nb = 0; nb < 8; nb++) {
#pragma unroll
        for (int e = 0; e < 4; e++) dh1[nb][e] = h1[nb][e] > 0.f ? dh1[nb][e] : 0.f;
        store_c(st + kStDH1, kLdH, nb, dh1[nb], lane);
    }
    colsum_c8(b2, dh2, lane, first);
    colsum_c8(b1, dh1, lane, first);
    __syncwarp();
}

// The same with the whole gradient into gs (the warp's partial, kGPad floats).
__device__ __forceinline__ void train_tile(const MlpDev& m, const TrainRows& r, __nv_bfloat16* st, float* gs, bool first,
                                           float inv_b, float& lsum, int lane)
{
    tile_backward(m, r, st, gs + kGB1, gs + kGB2, gs + kGB3, first, inv_b, lsum, lane);
    // dW3 = H2^T dY
    uint32_t by[2];
    load_bs(by, st + kStDY, kLdY, 0, lane);
#pragma unroll
    for (int mt = 0; mt < 4; mt++) {
        uint32_t a[4];
        load_at(a, st + kStH2, kLdH, mt, lane);
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(c, a, by);
        add_c(gs + kGW3, kMlpOutPad, mt, 0, c, lane, first);
    }
    // dW2 = H1^T dH2
#pragma unroll
    for (int nb = 0; nb < 8; nb++) {
        uint32_t b[2];
        load_bs(b, st + kStDH2, kLdH, nb, lane);
#pragma unroll
        for (int mt = 0; mt < 4; mt++) {
            uint32_t a[4];
            load_at(a, st + kStH1, kLdH, mt, lane);
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(c, a, b);
            add_c(gs + kGW2, kMlpHid, mt, nb, c, lane, first);
        }
    }
    __syncwarp();
    // dW1 = X^T dH1
    {
        uint32_t a[4];
        load_at(a, st + kStX, kLdX, 0, lane);
#pragma unroll
        for (int nb = 0; nb < 8; nb++) {
            uint32_t b[2];
            load_bs(b, st + kStDH1, kLdH, nb, lane);
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(c, a, b);
            add_c(gs + kGW1, kMlpHid, 0, nb, c, lane, first);
        }
    }
    __syncwarp();
}

// blocks of a mini-batch of B rows (one warp per 16 rows, at most max_blocks),
// and the warps of them that have a tile
__host__ __device__ __forceinline__ int train_blocks(int B, int max_blocks)
{
    const int b = (B + 16 * kTrainWarps - 1) / (16 * kTrainWarps);
    return b < max_blocks ? b : max_blocks;
}
__device__ __forceinline__ int train_warps(int B, int blocks)
{
    const int t = (B + 15) / 16;
    return t < blocks * kTrainWarps ? t : blocks * kTrainWarps;
}

// the tiles of a mini-batch on this warp; r: its first tile's rows
__device__ __forceinline__ void train_warp(const MlpDev& m, TrainRows r, const float* __restrict__ X,
                                           const float* __restrict__ T, const float* __restrict__ W,
                                           const int32_t* __restrict__ idx, int B, int blocks, __nv_bfloat16* st,
                                           float* __restrict__ part, float* __restrict__ lpart, int lane)
{
    const int gw = blockIdx.x * kTrainWarps + (threadIdx.x >> 5);
    const int ntiles = (B + 15) / 16;
    if (gw >= ntiles) return;
    const float inv_b = 1.0f / (float)B;
    float* gs = part + (int64_t)gw * kGPad;
    float lsum = 0.f;
    for (int tile = gw; tile < ntiles; tile += blocks * kTrainWarps) {
        if (tile != gw) r = train_rows(X, T, W, idx, B, tile, lane);
        train_tile(m, r, st, gs, tile == gw, inv_b, lsum, lane);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) lpart[gw] = lsum * inv_b;
}

__device__ __forceinline__ void load_model(MlpDev& m, const MlpDev* __restrict__ model)
{
    static_assert(sizeof(MlpDev) % 16 == 0, "the model is copied in 16-byte chunks");
    for (int i = threadIdx.x; i < (int)(sizeof(MlpDev) / 16); i += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(reinterpret_cast<uint4*>(&m) + i)),
                     "l"(reinterpret_cast<const uint4*>(model) + i)
                     : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// X: n x 16 normalised features (FP32, padding zero); T: n x 3 scaled
// targets; W: n weights (nullable); idx: the batch's row indices (B of
// them).  Every warp sums its tiles' gradient into its own partial (part,
// kGPad floats per warp) and its loss into lpart; the partials are added in
// warp order, so a training run repeats bit for bit.
__global__ void __launch_bounds__(kTrainWarps * 32) k_mlp_train(const float* __restrict__ X,
                                                                 const float* __restrict__ T,
                                                                 const float* __restrict__ W,
                                                                 const int32_t* __restrict__ idx, int B,
                                                                 const MlpDev* __restrict__ model,
                                                                 float* __restrict__ part, float* __restrict__ lpart)
{
    extern __shared__ __align__(16) unsigned char smem[];
    MlpDev& m = *reinterpret_cast<MlpDev*>(smem);
    __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(smem + sizeof(MlpDev)) + (threadIdx.x >> 5) * kStSize;
    const int lane = threadIdx.x & 31;
    const TrainRows r = train_rows(X, T, W, idx, B, blockIdx.x * kTrainWarps + (threadIdx.x >> 5), lane);
    load_model(m, model);
    __syncthreads();
    train_warp(m, r, X, T, W, idx, B, gridDim.x, st, part, lpart, lane);
}

// Element e of the packed gradient (W1[13][64], b1, W2, b2, W3[64][3], b3;
// e = kMlpNParam: the loss) from the nw partials: eight sums, of the warps
// k = j, j + 8, ..., then the eight in turn -- one fixed order.
constexpr int kReduceSlices = 8;
constexpr int kPB1 = kMlpIn * kMlpHid, kPW2 = kPB1 + kMlpHid, kPB2 = kPW2 + kMlpHid * kMlpHid;
constexpr int kPW3 = kPB2 + kMlpHid, kPB3 = kPW3 + kMlpHid * kMlpOut;
static_assert(kPB3 + kMlpOut == kMlpNParam, "packed gradient layout");

// packed index -> the padded index of a warp's partial (stride kGPad), or the
// loss partials (stride 1)
__device__ __forceinline__ const float* element_partials(const float* part, const float* lpart, int e, int64_t* stride)
{
    *stride = e < kMlpNParam ? kGPad : 1;
    if (e < kPB1) return part + kGW1 + e;
    if (e < kPW2) return part + kGB1 + (e - kPB1);
    if (e < kPB2) return part + kGW2 + (e - kPW2);
    if (e < kPW3) return part + kGB2 + (e - kPB2);
    if (e < kPB3) return part + kGW3 + ((e - kPW3) / kMlpOut) * kMlpOutPad + ((e - kPW3) % kMlpOut);
    return e < kMlpNParam ? part + kGB3 + (e - kPB3) : lpart;
}

// NT = 1, 2, 4 or 8 neighbouring lanes share an element; lane sub of them
// takes the sums j = sub NT' .. and all return the element's sum
template <int NT>
__device__ __forceinline__ float reduce_element(const float* part, const float* lpart, int nw, int e, int sub)
{
    constexpr int NS = kReduceSlices / NT;
    int64_t stride;
    const float* src = element_partials(part, lpart, e, &stride);
    float s[NS];
#pragma unroll
    for (int j = 0; j < NS; j++) s[j] = 0.f;
#pragma unroll 8
    for (int k = sub * NS; k < nw; k += kReduceSlices) {
#pragma unroll
        for (int j = 0; j < NS; j++)
            if (k + j < nw) s[j] += __ldcg(src + (int64_t)(k + j) * stride);
    }
    float t = 0.f;
#pragma unroll
    for (int j = 0; j < kReduceSlices; j++) {
        const float x = NT == 1 ? s[j % NS] : __shfl_sync(0xffffffffu, s[j % NS], j / NS, NT);
        t = j == 0 ? x : t + x;
    }
    return t;
}

// a block takes 32 elements, its warps a sum each of the eight: a gradient of
// 20000 rows (1216 partials) takes 72 us, 171 with a thread an element
__global__ void __launch_bounds__(32 * kReduceSlices) k_grad_reduce(const float* __restrict__ part,
                                                                    const float* __restrict__ lpart, int nw,
                                                                    float* __restrict__ grad, float* __restrict__ loss)
{
    __shared__ float sums[kReduceSlices][32];
    const int x = threadIdx.x & 31, j = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + x;
    if (e <= kMlpNParam) {
        int64_t stride;
        const float* src = element_partials(part, lpart, e, &stride);
        float s = 0.f;
#pragma unroll 8
        for (int k = j; k < nw; k += kReduceSlices) s += src[(int64_t)k * stride];
        sums[j][x] = s;
    }
    __syncthreads();
    if (j > 0 || e > kMlpNParam) return;
    float t = sums[0][x];
#pragma unroll
    for (int k = 1; k < kReduceSlices; k++) t += sums[k][x];
    if (e < kMlpNParam) grad[e] = t;
    else *loss += t;
}

// Adam on one FP32 master parameter (the contractions written out, so that
// the rounding does not depend on what is compiled around it)
__device__ __forceinline__ void adam_update(float& p, float& mom, float& vel, float gi, float lr, float b1, float b2,
                                            float eps, float c1, float c2)
{
    const float mi = fmaf(1.f - b1, gi, b1 * mom);
    const float vi = fmaf((1.f - b2) * gi, gi, b2 * vel);
    mom = mi;
    vel = vi;
    p -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// the parts of the device model that a training step reads, for parameter e:
// its place in the forward fragments, and for W2 and W3 the k-major copy the
// backward pass takes its transposes from
__device__ __forceinline__ void put_parameter(MlpDev* m, int e, float p)
{
    const __nv_bfloat16 v = __float2bfloat16_rn(p);
    auto frag = [](uint2* f, int k, int n) {  // 16-bit slot of W[k][n] in a 16 x 8 block's fragment, k < 16, n < 8
        return reinterpret_cast<__nv_bfloat16*>(f + n * 4 + ((k & 7) >> 1)) + 2 * (k >> 3) + (k & 1);
    };
    if (e < kPB1) {
        const int k = e / kMlpHid, n = e % kMlpHid;
        *frag(m->frag.f1[n >> 3], k, n & 7) = v;
    } else if (e < kPW2) {
        const int n = e - kPB1;
        reinterpret_cast<float*>(m->frag.b1)[n] = p;  // [column block][q] pairs: plain column order
    } else if (e < kPB2) {
        const int k = (e - kPW2) / kMlpHid, n = (e - kPW2) % kMlpHid;
        *frag(m->frag.f2[k >> 4][n >> 3], k & 15, n & 7) = v;
        m->w2[e - kPW2] = v;
    } else if (e < kPW3) {
        reinterpret_cast<float*>(m->frag.b2)[e - kPB2] = p;
    } else if (e < kPB3) {
        const int k = (e - kPW3) / kMlpOut, n = (e - kPW3) % kMlpOut;
        *frag(m->frag.f3[k >> 4], k & 15, n) = v;
        m->w3[k * kMlpOutPad + n] = v;
    } else {
        reinterpret_cast<float*>(m->frag.b3)[e - kPB3] = p;
    }
}

// all blocks of a cooperative launch; a wait that runs out (about a second)
// raises kErrWorkLoop and returns false in every thread of the block
__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t target, int32_t* err)
{
    __shared__ bool ok_sh;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();  // (the block's writes, ordered before this thread by the barrier above)
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        bool ok = true;
        const long long t0 = clock64();
        for (;;) {
            uint32_t v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (v >= target) break;
            if (clock64() - t0 > (1ll << 31)) {
                ok = false;
                atomicOr(err, kErrWorkLoop);
                break;
            }
        }
        ok_sh = ok;
    }
    __syncthreads();
    const bool ok = ok_sh;
    __syncthreads();
    return ok;
}

constexpr int kUpdateLanes = 2;

// One pass over the pairs in mini-batches, one cooperative launch.  A step
// used to be four dependent launches (gradient, reduction, Adam, packing) of
// a few blocks each, 43 us of latency for 1024 rows, 15 us now; the blocks
// meet at two grid barriers a step: after the gradient (a warp per 16 rows),
// and after the update, where two lanes per parameter (1 / 2 / 4 lanes: 21 /
// 15 / 17 us a step) add the partials in their order and one of them keeps
// the master parameter and its Adam moments in registers through the pass
// and writes the BF16 copies the next step reads.  The next step's rows are
// loaded before the barriers.  (Mini-batches above kClusterRows.)  Same operations in the same order as the
// single kernels: the same network bit for bit.
__global__ void __launch_bounds__(kTrainWarps * 32) k_mlp_epoch(const float* __restrict__ X, const float* __restrict__ T,
                                                                 const float* __restrict__ W,
                                                                 const int32_t* __restrict__ idx, int n, int batch,
                                                                 int max_blocks, MlpDev* model, float* params,
                                                                 float* mom, float* vel,
                                                                 const float* __restrict__ sched, float b1, float b2,
                                                                 float eps, float* part, float* lpart, float* loss,
                                                                 uint32_t* bar, int32_t* err)
{
    extern __shared__ __align__(16) unsigned char smem[];
    MlpDev& m = *reinterpret_cast<MlpDev*>(smem);
    __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(smem + sizeof(MlpDev)) + (threadIdx.x >> 5) * kStSize;
    const int lane = threadIdx.x & 31;
    const int gw = blockIdx.x * kTrainWarps + (threadIdx.x >> 5);
    // kUpdateLanes neighbouring lanes to a parameter; the last parameter's
    // follow is the loss, and lanes past it repeat it
    const int t = blockIdx.x * blockDim.x + threadIdx.x, sub = t % kUpdateLanes;
    const int e = min(t / kUpdateLanes, kMlpNParam);
    const bool own = sub == 0 && t / kUpdateLanes <= kMlpNParam;
    const bool any = (t & ~31) / kUpdateLanes <= kMlpNParam;  // the warp holds an element
    float pe = 0.f, me = 0.f, ve = 0.f;
    if (e < kMlpNParam) {
        pe = params[e];
        me = mom[e];
        ve = vel[e];
    } else if (e == kMlpNParam) {
        pe = *loss;
    }
    uint32_t target = 0;
    TrainRows r = train_rows(X, T, W, idx, min(batch, n), gw, lane);
    for (int b0 = 0, step = 0; b0 < n; b0 += batch, step++) {
        const int B = min(batch, n - b0), blocks = train_blocks(B, max_blocks);
        if (blockIdx.x < blocks) {
            load_model(m, model);
            __syncthreads();
            train_warp(m, r, X, T, W, idx + b0, B, blocks, st, part, lpart, lane);
        }
        if (b0 + batch < n) r = train_rows(X, T, W, idx + b0 + batch, min(batch, n - b0 - batch), gw, lane);
        target += gridDim.x;
        if (!grid_barrier(bar, target, err)) return;
        if (any) {
            const float g = reduce_element<kUpdateLanes>(part, lpart, train_warps(B, blocks), e, sub);
            if (!own) {
            } else if (e < kMlpNParam) {
                adam_update(pe, me, ve, g, sched[3 * step], b1, b2, eps, sched[3 * step + 1], sched[3 * step + 2]);
                put_parameter(model, e, pe);
            } else {
                pe += g;
            }
        }
        target += gridDim.x;
        if (!grid_barrier(bar, target, err)) return;
    }
    if (own && e < kMlpNParam) {
        params[e] = pe;
        mom[e] = me;
        vel[e] = ve;
    } else if (own) {
        *loss = pe;
    }
}

// The same pass on one cluster of eight blocks, for mini-batches whose tiles
// its 64 warps do in a few rounds.  A step at two grid barriers is mostly
// their latency and the partials' way through L2; here everything stays in
// the cluster's shared memory.  Block j takes the tiles k = j mod 8 (the
// order of reduce_element's eight sums): its warps do a tile each, then each
// takes a column block of the weights' gradients over the tiles in turn, so
// the block's sum comes out in registers.  Every block then owns an eighth of
// the parameters: it adds the eight blocks' sums (distributed shared memory),
// updates, and stores the parameter in all eight blocks, which turn them into
// the BF16 copies the next step reads.  Same operations, same order, same
// network.  Bound by latency at two warps a scheduler: of six cycles an
// instruction waits, 1.9 are for shared memory, 1.4 fixed latencies, 0.7 loads
// and 0.7 barriers, while the tensor unit is busy 11 % (8 cycles a mma.sync).
// 7.3 of a step's 17 thousand cycles are forward and backward, two tiles a
// scheduler, 2.6 the gradient's products, 2.2 the two cluster barriers.  The
// sums' and parameters' exchange was 3.9 when each of a thread's three
// elements was read, updated and stored in turn, and the row indices of the
// next tile cost their latency when they were not loaded a tile ahead.
// Training on 2^18 pairs, us a step in all, grid barriers / cluster: 256 rows
// 9.5 / 6.7, 1024 14.0 / 10.1, 4096 28.7 / 28.2, 8192 47 / 52.
constexpr int kClusterRows = 4096;
constexpr int kClusterBlocks = kReduceSlices, kClusterWarps = 8;
constexpr int kOwn = (kMlpNParam + 1 + kClusterBlocks - 1) / kClusterBlocks;  // elements a block updates
constexpr int kOwnThread = (kOwn + kClusterWarps * 32 - 1) / (kClusterWarps * 32);
constexpr int kSideB2 = kMlpHid, kSideB3 = 2 * kMlpHid, kSideLoss = kSideB3 + kMlpOut;  // per tile: biases' gradients, loss
// packed order with the rows of W2 ld apart (72 and 68: the accesses below
// meet no bank conflicts)
constexpr int kLdSum = 72, kLdP = 68;
__device__ __forceinline__ int padded(int e, int ld)
{
    return e < kPW2 ? e : (e < kPB2 ? e + ((e - kPW2) / kMlpHid) * (ld - kMlpHid) : e + kMlpHid * (ld - kMlpHid));
}
struct ClusterShared {
    MlpDev m;
    float sum[(kMlpNParam + 1 + kMlpHid * (kLdSum - kMlpHid) + 3) & ~3];  // the block's sums
    float p[(kMlpNParam + kMlpHid * (kLdP - kMlpHid) + 3) & ~3];          // the new parameters
    float side[kClusterWarps][2 * kMlpHid + kMlpOutPad];
    __nv_bfloat16 st[kClusterWarps][kStSize];
};
static_assert(kSideLoss < 2 * kMlpHid + kMlpOutPad && kStSize % 8 == 0 && sizeof(ClusterShared) <= 227 * 1024,
              "the cluster kernel's shared memory");

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// the address of this block's shared p in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank)
{
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(d)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return d;
}

// all parameters (padded order, shared memory) into the model's parts that a
// step reads, as put_parameter does one by one
__device__ __forceinline__ void put_parameters(MlpDev& m, const float* p)
{
    for (int i = threadIdx.x; i < 8 * 32; i += blockDim.x) {
        const int l = i & 31, n = (i >> 5) * 8 + (l >> 2), k = 2 * (l & 3);
        const auto w = [&](int r) { return r < kMlpIn ? p[r * kMlpHid + n] : 0.f; };
        m.frag.f1[i >> 5][l] = make_uint2(pack_bf16(w(k), w(k + 1)), pack_bf16(w(k + 8), w(k + 9)));
    }
    for (int i = threadIdx.x; i < 4 * 8 * 32; i += blockDim.x) {
        const int l = i & 31, n = ((i >> 5) & 7) * 8 + (l >> 2), k = (i >> 8) * 16 + 2 * (l & 3);
        const auto w = [&](int r) { return p[kPW2 + r * kLdP + n]; };
        m.frag.f2[i >> 8][(i >> 5) & 7][l] = make_uint2(pack_bf16(w(k), w(k + 1)), pack_bf16(w(k + 8), w(k + 9)));
    }
    for (int i = threadIdx.x; i < kMlpHid * kMlpHid / 4; i += blockDim.x) {
        const float4 v = *reinterpret_cast<const float4*>(&p[kPW2 + (i >> 4) * kLdP + 4 * (i & 15)]);
        reinterpret_cast<uint2*>(m.w2)[i] = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
    }
    constexpr int kAfter = kMlpHid * (kLdP - kMlpHid);  // the padding before what follows W2
    for (int i = threadIdx.x; i < kMlpHid * kMlpOut; i += blockDim.x) {
        const int k = i / kMlpOut, n = i % kMlpOut;
        const __nv_bfloat16 v = __float2bfloat16_rn(p[kPW3 + kAfter + i]);
        reinterpret_cast<__nv_bfloat16*>(&m.frag.f3[k >> 4][n * 4 + ((k & 7) >> 1)])[2 * ((k >> 3) & 1) + (k & 1)] = v;
        m.w3[k * kMlpOutPad + n] = v;
    }
    for (int i = threadIdx.x; i < kMlpHid; i += blockDim.x) {
        reinterpret_cast<float*>(m.frag.b1)[i] = p[kPB1 + i];
        reinterpret_cast<float*>(m.frag.b2)[i] = p[kPB2 + kAfter + i];
    }
    if (threadIdx.x < kMlpOut) reinterpret_cast<float*>(m.frag.b3)[threadIdx.x] = p[kPB3 + kAfter + threadIdx.x];
}

__global__ void __cluster_dims__(kClusterBlocks, 1, 1) __launch_bounds__(kClusterWarps * 32)
    k_mlp_cluster(const float* __restrict__ X, const float* __restrict__ T, const float* __restrict__ W,
                  const int32_t* __restrict__ idx, int n, int batch, MlpDev* model, float* params, float* mom, float* vel,
                  const float* __restrict__ sched, float b1, float b2, float eps, float* loss)
{
    extern __shared__ __align__(16) unsigned char smem[];
    ClusterShared& S = *reinterpret_cast<ClusterShared*>(smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
    const int cta = blockIdx.x;  // (one cluster: its rank)
    // the elements this thread updates; the one past the parameters is the loss
    float pe[kOwnThread], me[kOwnThread], ve[kOwnThread];
    const auto own = [&](int i) {
        const int o = threadIdx.x + i * kClusterWarps * 32;
        const int e = cta * kOwn + o;
        return o < kOwn && e <= kMlpNParam ? e : -1;
    };
#pragma unroll
    for (int i = 0; i < kOwnThread; i++) {
        const int e = own(i);
        pe[i] = me[i] = ve[i] = 0.f;
        if (e >= 0 && e < kMlpNParam) pe[i] = params[e], me[i] = mom[e], ve[i] = vel[e];
        else if (e >= 0) pe[i] = *loss;
    }
    load_model(S.m, model);
    __syncthreads();
    // a warp's tiles follow each other through the rounds of all steps: the
    // rows of the next one are loaded while this one's products run, the
    // indices of the one after it before that
    int fb = 0, ft = 0;  // the tile whose indices are loaded next: its step's first row, its round's first tile
    const auto next_index = [&]() {
        if (fb >= n) return make_int2(-1, -1);
        const int B = min(batch, n - fb);
        const int2 x = train_index(idx + fb, B, cta + kClusterBlocks * (ft + w), lane);
        ft += kClusterWarps;
        if (kClusterBlocks * ft + cta >= (B + 15) / 16) {
            ft = 0;
            fb += batch;
        }
        return x;
    };
    TrainRows r = train_rows(X, T, W, next_index(), lane);
    int2 index = next_index();
    for (int b0 = 0, step = 0; b0 < n; b0 += batch, step++) {
        const int B = min(batch, n - b0), ntiles = (B + 15) / 16;
        const float inv_b = 1.0f / (float)B;
        const int mine = ntiles > cta ? (ntiles - cta - 1) / kClusterBlocks + 1 : 0;  // this block's tiles
        const float lr = sched[3 * step], c1 = sched[3 * step + 1], c2 = sched[3 * step + 2];  // (needed after the sums)
        float acc1[4], acc2[4][4], acc3[4], side = 0.f;
#pragma unroll
        for (int k = 0; k < 4; k++) acc1[k] = acc3[k] = acc2[0][k] = acc2[1][k] = acc2[2][k] = acc2[3][k] = 0.f;
        for (int t0 = 0; t0 < mine; t0 += kClusterWarps) {
            if (t0 > 0) __syncthreads();  // the last round's matrices are read
            if (t0 + w < mine) {
                float lsum = 0.f;
                tile_backward(S.m, r, S.st[w], S.side[w], S.side[w] + kSideB2, S.side[w] + kSideB3, true, inv_b, lsum, lane);
#pragma unroll
                for (int o = 16; o; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
                if (lane == 0) S.side[w][kSideLoss] = lsum * inv_b;
            }
            r = train_rows(X, T, W, index, lane);
            index = next_index();
            __syncthreads();
            const int nt = min(mine - t0, kClusterWarps);
            for (int i = 0; i < nt; i++) {
                const __nv_bfloat16* st = S.st[i];
                uint32_t a[4], b[2];
                load_bs(b, st + kStDH2, kLdH, w, lane);  // dW2 = H1^T dH2, columns 8 w ..
#pragma unroll
                for (int mt = 0; mt < 4; mt++) {
                    load_at(a, st + kStH1, kLdH, mt, lane);
                    float c[4] = {0.f, 0.f, 0.f, 0.f};
                    mma_bf16(c, a, b);
#pragma unroll
                    for (int k = 0; k < 4; k++) acc2[mt][k] += c[k];
                }
                load_bs(b, st + kStDH1, kLdH, w, lane);  // dW1 = X^T dH1
                load_at(a, st + kStX, kLdX, 0, lane);
                {
                    float c[4] = {0.f, 0.f, 0.f, 0.f};
                    mma_bf16(c, a, b);
#pragma unroll
                    for (int k = 0; k < 4; k++) acc1[k] += c[k];
                }
                if (w < 4) {  // dW3 = H2^T dY, rows 16 w ..
                    load_bs(b, st + kStDY, kLdY, 0, lane);
                    load_at(a, st + kStH2, kLdH, w, lane);
                    float c[4] = {0.f, 0.f, 0.f, 0.f};
                    mma_bf16(c, a, b);
#pragma unroll
                    for (int k = 0; k < 4; k++) acc3[k] += c[k];
                }
                if (threadIdx.x <= kSideLoss) side += S.side[i][threadIdx.x];
            }
        }
        // the block's sums
        constexpr int kAfter = kMlpHid * (kLdSum - kMlpHid);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int row = g + 8 * h, col = w * 8 + 2 * q;
            if (row < kMlpIn) *reinterpret_cast<float2*>(&S.sum[row * kMlpHid + col]) = make_float2(acc1[2 * h], acc1[2 * h + 1]);
#pragma unroll
            for (int mt = 0; mt < 4; mt++)
                *reinterpret_cast<float2*>(&S.sum[kPW2 + (mt * 16 + row) * kLdSum + col]) =
                    make_float2(acc2[mt][2 * h], acc2[mt][2 * h + 1]);
#pragma unroll
            for (int k = 0; k < 2; k++)
                if (w < 4 && 2 * q + k < kMlpOut) S.sum[kPW3 + kAfter + (w * 16 + row) * kMlpOut + 2 * q + k] = acc3[2 * h + k];
        }
        if (threadIdx.x < kSideB2) S.sum[kPB1 + threadIdx.x] = side;
        else if (threadIdx.x < kSideB3) S.sum[kPB2 + kAfter + threadIdx.x - kSideB2] = side;
        else if (threadIdx.x < kSideLoss) S.sum[kPB3 + kAfter + threadIdx.x - kSideB3] = side;
        else if (threadIdx.x == kSideLoss) S.sum[kMlpNParam + kAfter] = side;
        cluster_sync();
        float s[kOwnThread][kClusterBlocks];
#pragma unroll
        for (int i = 0; i < kOwnThread; i++) {
            const int e = own(i);
            const float* from = &S.sum[padded(e < 0 ? 0 : e, kLdSum)];
#pragma unroll
            for (int j = 0; j < kClusterBlocks; j++)
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(s[i][j]) : "r"(cluster_addr(from, j)) : "memory");
        }
#pragma unroll
        for (int i = 0; i < kOwnThread; i++) {
            const int e = own(i);
            float t = s[i][0];
#pragma unroll
            for (int j = 1; j < kClusterBlocks; j++) t += s[i][j];
            if (e == kMlpNParam) pe[i] += t;
            else if (e >= 0) adam_update(pe[i], me[i], ve[i], t, lr, b1, b2, eps, c1, c2);
        }
#pragma unroll
        for (int i = 0; i < kOwnThread; i++) {
            const int e = own(i);
            if (e < 0 || e == kMlpNParam) continue;
            const float* to = &S.p[padded(e, kLdP)];
#pragma unroll
            for (int j = 0; j < kClusterBlocks; j++)
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr(to, j)), "f"(pe[i]) : "memory");
        }
        cluster_sync();
        put_parameters(S.m, S.p);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < kOwnThread; i++) {
        const int e = own(i);
        if (e >= 0 && e < kMlpNParam) params[e] = pe[i], mom[e] = me[i], vel[e] = ve[i];
        else if (e >= 0) *loss = pe[i];
    }
    if (cta == 0)
        for (int i = threadIdx.x; i < (int)(sizeof(MlpDev) / 16); i += blockDim.x)
            reinterpret_cast<uint4*>(model)[i] = reinterpret_cast<const uint4*>(&S.m)[i];
}

// packed FP32 parameters + feature/output maps -> device BF16 model: the
// k-major weights for training and the fragment-arranged inference copy
__global__ void k_mlp_pack(const float* __restrict__ p, const float* __restrict__ maps, MlpDev* __restrict__ m)
{
    const float* W1 = p;
    const float* b1 = W1 + kMlpIn * kMlpHid;
    const float* W2 = b1 + kMlpHid;
    const float* b2 = W2 + kMlpHid * kMlpHid;
    const float* W3 = b2 + kMlpHid;
    const float* b3 = W3 + kMlpHid * kMlpOut;
    // padded weights: input rows past 13 and output columns past 3 are zero
    auto w1 = [&](int k, int n) { return k < kMlpIn ? W1[k * kMlpHid + n] : 0.f; };
    auto w3 = [&](int k, int n) { return n < kMlpOut ? W3[k * kMlpOut + n] : 0.f; };
    auto bf = [](float lo, float hi) {
        __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t*>(&v);
    };
    for (int i = threadIdx.x; i < kMlpInPad * kMlpHid; i += blockDim.x)
        m->w1[i] = __float2bfloat16_rn(w1(i / kMlpHid, i % kMlpHid));
    for (int i = threadIdx.x; i < kMlpHid * kMlpHid; i += blockDim.x) m->w2[i] = __float2bfloat16_rn(W2[i]);
    for (int i = threadIdx.x; i < kMlpHid * kMlpOutPad; i += blockDim.x)
        m->w3[i] = __float2bfloat16_rn(w3(i / kMlpOutPad, i % kMlpOutPad));
    // B fragments: lane (g, q) of column block nb, k-step ks holds
    // {W[16 ks + 2q][n], W[16 ks + 2q + 1][n]}, {W[16 ks + 2q + 8][n], W[16 ks + 2q + 9][n]}, n = 8 nb + g
    MlpFrag& f = m->frag;
    for (int i = threadIdx.x; i < 8 * 32; i += blockDim.x) {
        const int nb = i / 32, lane = i % 32, g = lane >> 2, q = lane & 3, n = nb * 8 + g, k = 2 * q;
        f.f1[nb][lane] = make_uint2(bf(w1(k, n), w1(k + 1, n)), bf(w1(k + 8, n), w1(k + 9, n)));
    }
    for (int i = threadIdx.x; i < 4 * 8 * 32; i += blockDim.x) {
        const int ks = i / 256, nb = (i / 32) % 8, lane = i % 32, g = lane >> 2, q = lane & 3;
        const int n = nb * 8 + g, k = ks * 16 + 2 * q;
        f.f2[ks][nb][lane] = make_uint2(bf(W2[k * kMlpHid + n], W2[(k + 1) * kMlpHid + n]),
                                        bf(W2[(k + 8) * kMlpHid + n], W2[(k + 9) * kMlpHid + n]));
    }
    for (int i = threadIdx.x; i < 4 * 32; i += blockDim.x) {
        const int ks = i / 32, lane = i % 32, g = lane >> 2, q = lane & 3, k = ks * 16 + 2 * q;
        f.f3[ks][lane] = make_uint2(bf(w3(k, g), w3(k + 1, g)), bf(w3(k + 8, g), w3(k + 9, g)));
    }
    for (int i = threadIdx.x; i < kMlpHid; i += blockDim.x) {
        m->b1[i] = b1[i];
        m->b2[i] = b2[i];
    }
    for (int i = threadIdx.x; i < 32; i += blockDim.x) {
        const int nb = i / 4, q = i % 4;
        f.b1[nb][q] = make_float2(b1[nb * 8 + 2 * q], b1[nb * 8 + 2 * q + 1]);
        f.b2[nb][q] = make_float2(b2[nb * 8 + 2 * q], b2[nb * 8 + 2 * q + 1]);
    }
    for (int i = threadIdx.x; i < kMlpOutPad; i += blockDim.x) {
        m->b3[i] = i < kMlpOut ? b3[i] : 0.f;
        f.yscale[i] = i < kMlpOut ? maps[2 * kMlpIn + i] : 0.f;
    }
    for (int i = threadIdx.x; i < 4; i += blockDim.x)
        f.b3[i] = make_float2(2 * i < kMlpOut ? b3[2 * i] : 0.f, 2 * i + 1 < kMlpOut ? b3[2 * i + 1] : 0.f);
    for (int i = threadIdx.x; i < kMlpInPad; i += blockDim.x) {
        f.xscale[i] = i < kMlpIn ? maps[kMlpIn + i] : 0.f;
        f.xoff[i] = i < kMlpIn ? -maps[i] * maps[kMlpIn + i] : 0.f;
    }
}

// batch inference: Y (n x 3) = network(X) * yscale, X normalised n x 16 --
// the same fragment path the walk evaluates its corrections with
__global__ void __launch_bounds__(128) k_mlp_infer(const float* __restrict__ X, int64_t n,
                                                   const MlpDev* __restrict__ model, float* __restrict__ Y)
{
    __shared__ MlpFrag m;
    for (int i = threadIdx.x; i < (int)(sizeof(MlpFrag) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t*>(&m)[i] = reinterpret_cast<const uint32_t*>(&model->frag)[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int g = lane >> 2, q = lane & 3;
    const int64_t ntiles = (n + 15) / 16;
    for (int64_t tile = (int64_t)blockIdx.x * 4 + w; tile < ntiles; tile += (int64_t)gridDim.x * 4) {
        const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
        const bool v0 = r0 < n, v1 = r1 < n;
        auto xv = [&](int64_t r, bool v, int c) { return v ? X[r * kMlpInPad + c] : 0.f; };
        uint32_t x[4];
        x[0] = pack_bf16(xv(r0, v0, 2 * q), xv(r0, v0, 2 * q + 1));
        x[1] = pack_bf16(xv(r1, v1, 2 * q), xv(r1, v1, 2 * q + 1));
        x[2] = pack_bf16(xv(r0, v0, 2 * q + 8), xv(r0, v0, 2 * q + 9));
        x[3] = pack_bf16(xv(r1, v1, 2 * q + 8), xv(r1, v1, 2 * q + 9));
        float y[4];
        mlp16_infer(m, x, y, lane);
        const int c0 = 2 * q, c1 = 2 * q + 1;
        if (v0 && c0 < 3) Y[r0 * 3 + c0] = y[0] * m.yscale[c0];
        if (v0 && c1 < 3) Y[r0 * 3 + c1] = y[1] * m.yscale[c1];
        if (v1 && c0 < 3) Y[r1 * 3 + c0] = y[2] * m.yscale[c0];
        if (v1 && c1 < 3) Y[r1 * 3 + c1] = y[3] * m.yscale[c1];
    }
}

// Features, exact label and label factor of (body, cell) pairs, one thread
// per pair: features at the body's position; factor F = G M s^2 / r^4 (the
// scale of the quadrupole term); label = (a_exact - a_mono) / F with a_exact
// the softened sum over the cell's bodies (FP64 accumulation).
__global__ void k_pair_labels(const int32_t* __restrict__ pb, const int32_t* __restrict__ pv, int64_t np,
                              const float4* __restrict__ body, const uint32_t* __restrict__ sys_of,
                              const SysParams* __restrict__ sysp, NodeTables nt, float eps, float G,
                              float* __restrict__ feat, float* __restrict__ lab, float* __restrict__ fac)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= np) return;
    const int64_t ib = pb[k], v = pv[k];
    const float4 xb = body[ib];
    const double x[3] = {xb.x, xb.y, xb.z};
    const int4 b = nt.b[v];
    const int4 cc = nt.c[v];
    const SysParams& P = sysp[cc.w];
    const double s = ldexp(P.L, -(b.w & 255));
    const double M = nt.mass64[v];
    const double* com = &nt.com64[3 * v];
    double d[3], r2 = 0.0;
    for (int a = 0; a < 3; a++) {
        d[a] = com[a] - x[a];
        r2 += d[a] * d[a];
    }
    const double r = sqrt(r2);
    float* f = feat + k * kMlpIn;
    for (int a = 0; a < 3; a++) f[a] = (float)(d[a] / s);
    f[3] = (float)(s / r);
    f[4] = (float)(eps / s);
    f[5] = (float)log2((double)b.y);
    f[6] = (float)(M / nt.mass64[cc.w]);  // the system's root is node cc.w
    for (int q = 0; q < 6; q++) f[7 + q] = (float)((double)nt.quad[6 * v + q] / (M * s * s));
    const double e2 = (double)eps * (double)eps;
    double ae[3] = {0, 0, 0};
    for (int j = b.x; j < b.x + b.y; j++) {
        const float4 y = body[j];
        const double dx = (double)y.x - x[0], dy = (double)y.y - x[1], dz = (double)y.z - x[2];
        const double q2 = dx * dx + dy * dy + dz * dz + e2;
        const double ri = 1.0 / sqrt(q2);
        const double fm = (double)y.w * ri * ri * ri;
        ae[0] += fm * dx;
        ae[1] += fm * dy;
        ae[2] += fm * dz;
    }
    const double rm = 1.0 / sqrt(r2 + e2);
    const double fmo = M * rm * rm * rm;
    const double F = (double)G * M * s * s / (r2 * r2);
    for (int a = 0; a < 3; a++) lab[k * 3 + a] = (float)((double)G * (ae[a] - fmo * d[a]) / F);
    if (fac) fac[k] = (float)F;
}

// ---------------------------------------------------------------- node features
// The nine features of a cell that do not depend on the point it is
// evaluated at -- eps/s, log2(count), M / M_sys and the six moment ratios
// Q_ab / (M s^2) -- normalised with the model's maps and packed as BF16
// pairs in the order of a network row (words 2..7: features 4..12, then the
// zero padding), once per node and force phase, so a walk that evaluates a
// cell forms only d/s and s/r itself.
__global__ void k_node_features(const Info* info, const SysParams* __restrict__ sysp, NodeTables nt, float eps,
                                const MlpDev* __restrict__ model)
{
    if ((*(volatile const int32_t*)&info->err & kErrCapacity) != 0) return;
    const int64_t M = info->M;
    const MlpFrag& m = model->frag;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < M; v += (int64_t)gridDim.x * blockDim.x) {
        const int4 nb = nt.b[v];
        const float4 na = nt.a[v];
        const int4 cc = nt.c[v];
        const SysParams& P = sysp[cc.w];
        const int level = nb.w & 255;
        const float inv_s = scalbnf(1.0f / P.Lf, level);  // exact: sides are powers of two
        const float Mc = na.w;
        const float iq = __fdividef(inv_s * inv_s, Mc);
        const float* qd = nt.quad + 6 * v;
        float f[kMlpInPad];
#pragma unroll
        for (int k = 0; k < kMlpInPad; k++) f[k] = 0.f;
        f[4] = eps * inv_s;
        f[5] = __log2f((float)nb.y);
        f[6] = Mc * (1.0f / P.msys);
#pragma unroll
        for (int k = 0; k < 6; k++) f[7 + k] = qd[k] * iq;
#pragma unroll
        for (int k = 4; k < kMlpIn; k++) f[k] = fmaf(f[k], m.xscale[k], m.xoff[k]);
        nt.feat[2 * v] = make_uint4(pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]), pack_bf16(f[8], f[9]),
                                    pack_bf16(f[10], f[11]));
        nt.feat[2 * v + 1] = make_uint4(pack_bf16(f[12], 0.f), 0u, 0u, 0u);
    }
}

// ---------------------------------------------------------------- training data
// Sums over the n training pairs, in FP64: x_c (13), x_c^2 (13), t_c^2 (3)
// and F^2 of the label factors (F null: skipped).  Every block takes every
// gridDim-th run of rows and leaves its sums in part[block]; k_mlp_maps adds
// the blocks in order, so the maps (and the training that follows) repeat
// bit for bit.  (One block per column read each row thirty times over: 373 us
// for 2^18 pairs, a quarter of the pass.)
constexpr int kSumThreads = 128;
__global__ void __launch_bounds__(kSumThreads) k_mlp_sums(const float* __restrict__ X, const float* __restrict__ T,
                                                          const float* __restrict__ F, int64_t n,
                                                          double* __restrict__ part)
{
    double s[kMlpSums];
#pragma unroll
    for (int c = 0; c < kMlpSums; c++) s[c] = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kSumThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kSumThreads) {
        float x[kMlpIn], t[kMlpOut];
#pragma unroll
        for (int c = 0; c < kMlpIn; c++) x[c] = X[i * kMlpIn + c];
#pragma unroll
        for (int c = 0; c < kMlpOut; c++) t[c] = T[i * kMlpOut + c];
        const double f = F ? (double)F[i] : 0.0;
#pragma unroll
        for (int c = 0; c < kMlpIn; c++) {
            const double v = x[c];
            s[c] += v;
            s[kMlpIn + c] += v * v;
        }
#pragma unroll
        for (int c = 0; c < kMlpOut; c++) s[2 * kMlpIn + c] += (double)t[c] * (double)t[c];
        s[kMlpSums - 1] += f * f;
    }
    __shared__ double red[kSumThreads / 32][kMlpSums];
#pragma unroll
    for (int c = 0; c < kMlpSums; c++) {
#pragma unroll
        for (int o = 16; o; o >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][c] = s[c];
    }
    __syncthreads();
    if (threadIdx.x < kMlpSums) {
        double v = red[0][threadIdx.x];
        for (int w = 1; w < kSumThreads / 32; w++) v += red[w][threadIdx.x];
        part[(int64_t)blockIdx.x * kMlpSums + threadIdx.x] = v;
    }
}

// the model's maps from the sums: feature means and inverse standard
// deviations (0 for a constant feature), output RMS (1 for an all-zero
// output); and the factor-weight scale n / sum F^2
// (one warp per j = 0..7 adds the blocks b = j mod 8, then the eight sums in
// turn: one chain of FP64 additions per column took 56 us of 2^18 pairs' 2.6 ms,
// 15)
constexpr int kMapWarps = 8;
__global__ void __launch_bounds__(32 * kMapWarps) k_mlp_maps(const double* __restrict__ part, int nblocks, int64_t n,
                                                             float* __restrict__ maps, float* __restrict__ wscale)
{
    __shared__ double red[kMapWarps][kMlpSums], sums[kMlpSums];
    const int k = threadIdx.x & 31, j = threadIdx.x >> 5;
    if (k < kMlpSums) {
        double v = 0.0;
#pragma unroll 8
        for (int b = j; b < nblocks; b += kMapWarps) v += part[(int64_t)b * kMlpSums + k];
        red[j][k] = v;
    }
    __syncthreads();
    if (j > 0) return;
    if (k < kMlpSums) {
        double v = red[0][k];
#pragma unroll
        for (int w = 1; w < kMapWarps; w++) v += red[w][k];
        sums[k] = v;
    }
    __syncwarp();
    const double inv_n = 1.0 / (double)n;
    if (k < kMlpIn) {
        const double mean = sums[k] * inv_n;
        const double var = fmax(0.0, sums[kMlpIn + k] * inv_n - mean * mean);
        maps[k] = (float)mean;
        maps[kMlpIn + k] = var > 1e-30 ? (float)(1.0 / sqrt(var)) : 0.f;
    } else if (k < kMlpIn + kMlpOut) {
        const double rms = sqrt(sums[2 * kMlpIn + k - kMlpIn] * inv_n);
        maps[2 * kMlpIn + k - kMlpIn] = rms > 1e-30 ? (float)rms : 1.f;
    } else if (k == kMlpIn + kMlpOut) {
        const double s2 = sums[kMlpSums - 1];
        *wscale = s2 > 0.0 ? (float)((double)n / s2) : 0.f;
    }
}

// normalised padded rows (x - mean) * scale, each operation rounded on its
// own (no contraction), zero padding; targets t / yscale
__global__ void k_mlp_rows(const float* __restrict__ X, const float* __restrict__ T, int64_t n,
                           const float* __restrict__ maps, float* __restrict__ rows, float* __restrict__ tout)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * kMlpInPad;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / kMlpInPad;
        const int k = (int)(e % kMlpInPad);
        rows[e] = k < kMlpIn ? __fmul_rn(__fsub_rn(X[i * kMlpIn + k], maps[k]), maps[kMlpIn + k]) : 0.f;
        if (T && k < kMlpOut) tout[i * kMlpOut + k] = __fdiv_rn(T[i * kMlpOut + k], maps[2 * kMlpIn + k]);
    }
}

// loss weights in place: mode 0 checks the given weights (finite, >= 0;
// *bad = 1 otherwise), mode 1 turns label factors F into F^2 n / sum F^2
__global__ void k_mlp_weights(float* __restrict__ w, int64_t n, int mode, const float* __restrict__ wscale,
                              int32_t* __restrict__ bad)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float v = w[i];
        if (!isfinite(v) || (mode == 0 && v < 0.f)) {
            *bad = 1;
            continue;
        }
        if (mode == 1) w[i] = __fmul_rn(__fmul_rn(v, v), *wscale);
    }
}

// Fresh parameters: weights and biases of layer l uniform in +-1/sqrt(fan-in)
// from a counter-based generator (SplitMix64 of seed and index)
__device__ __forceinline__ uint64_t splitmix(uint64_t z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_mlp_init(float* __restrict__ p, uint64_t seed)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kMlpNParam) return;
    const int l1 = kMlpIn * kMlpHid + kMlpHid;
    const double fan = i < l1 ? (double)kMlpIn : (double)kMlpHid;
    const double u = (double)(splitmix(seed * 0x100000001B3ull + (uint64_t)i) >> 11) * (1.0 / 9007199254740992.0);
    p[i] = (float)((2.0 * u - 1.0) / sqrt(fan));
}

// A random permutation of [0, n) without sorting: a 4-round Feistel network
// is a bijection on [0, 4^h) (4^h >= n, h the half width in bits); walking
// its cycle from i until the value falls below n gives a bijection on
// [0, n) (the walk ends: the cycle through i < n returns to i).  Key 0
// gives the identity.
__device__ __forceinline__ uint32_t feistel(uint32_t x, int h, uint64_t key)
{
    const uint32_t mask = (1u << h) - 1u;
    uint32_t L = x >> h, R = x & mask;
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const uint32_t f = (uint32_t)splitmix(key + 0x632BE59BD9B4E019ull * (uint64_t)r + R) & mask;
        const uint32_t t = L ^ f;
        L = R;
        R = t;
    }
    return (L << h) | R;
}

__global__ void k_mlp_shuffle(int64_t n, int h, uint64_t key, int32_t* __restrict__ idx)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t x = (uint32_t)i;
        if (key != 0) {
            do {
                x = feistel(x, h, key);
            } while ((int64_t)x >= n);
        }
        idx[i] = (int32_t)x;
    }
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

size_t mlp_train_smem() { return sizeof(MlpDev) + (size_t)kTrainWarps * kStSize * 2; }
int mlp_train_blocks(int B, int max_blocks) { return train_blocks(B, max_blocks); }
int64_t mlp_train_part_floats(int blocks) { return (int64_t)blocks * kTrainWarps * (kGPad + 1); }

cudaError_t launch_mlp_train(const float* X, const float* T, const float* W, const int32_t* idx, int B,
                             const void* model, float* grad, float* loss, float* part, int max_blocks, cudaStream_t s)
{
    const size_t smem = mlp_train_smem();
    cudaError_t e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int blocks = train_blocks(B, max_blocks);
    const int ntiles = (B + 15) / 16, nw = ntiles < blocks * kTrainWarps ? ntiles : blocks * kTrainWarps;
    float* lpart = part + (int64_t)blocks * kTrainWarps * kGPad;
    k_mlp_train<<<blocks, kTrainWarps * 32, smem, s>>>(X, T, W, idx, B, (const MlpDev*)model, part, lpart);
    k_grad_reduce<<<(kMlpNParam + 1 + 31) / 32, 32 * kReduceSlices, 0, s>>>(part, lpart, nw, grad, loss);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_mlp_epoch(const float* X, const float* T, const float* W, const int32_t* idx, int n, int batch,
                             int max_blocks, void* model, float* params, float* mom, float* vel, const float* sched,
                             float* part, float* loss, uint32_t* bar, int32_t* err, cudaStream_t s)
{
    const size_t smem = mlp_train_smem();
    float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    if (batch <= kClusterRows) {
        const cudaError_t e = cudaFuncSetAttribute(k_mlp_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)sizeof(ClusterShared));
        if (e != cudaSuccess) return e;
        k_mlp_cluster<<<kClusterBlocks, kClusterWarps * 32, sizeof(ClusterShared), s>>>(
            X, T, W, idx, n, batch, (MlpDev*)model, params, mom, vel, sched, b1, b2, eps, loss);
        count_launches(1);
        return cudaGetLastError();
    }
    cudaError_t e = cudaFuncSetAttribute(k_mlp_epoch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(bar, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    // a thread per parameter (and one for the loss), a warp per tile
    const int threads = kTrainWarps * 32;
    int grid = ((kMlpNParam + 1) * kUpdateLanes + threads - 1) / threads;
    const int blocks = train_blocks(batch < n ? batch : n, max_blocks);
    if (blocks > grid) grid = blocks;
    float* lpart = part + (int64_t)max_blocks * kTrainWarps * kGPad;
    MlpDev* mdl = (MlpDev*)model;
    void* args[] = {&X, &T, &W, &idx, &n, &batch, &max_blocks, &mdl, &params, &mom, &vel, &sched,
                    &b1, &b2, &eps, &part, &lpart, &loss, &bar, &err};
    e = cudaLaunchCooperativeKernel((const void*)k_mlp_epoch, dim3(grid), dim3(threads), args, smem, s);
    count_launches(1);
    return e;
}

void mlp_adam_corrections(int t, float* c1, float* c2)
{
    const float b1 = 0.9f, b2 = 0.999f;
    *c1 = 1.f - powf(b1, (float)t);
    *c2 = 1.f - powf(b2, (float)t);
}

void launch_mlp_pack(const float* params, const float* maps, void* model, cudaStream_t s)
{
    k_mlp_pack<<<1, 256, 0, s>>>(params, maps, (MlpDev*)model);
    count_launches(1);
}

void launch_mlp_infer(const float* X, int64_t n, const void* model, float* Y, cudaStream_t s)
{
    int64_t g = (n + 63) / 64;
    if (g > 4096) g = 4096;
    k_mlp_infer<<<(unsigned)(g < 1 ? 1 : g), 128, 0, s>>>(X, n, (const MlpDev*)model, Y);
    count_launches(1);
}

namespace {
// (body, node) pairs as sort keys (body position in the high half) and back
__global__ void k_pair_keys(const int32_t* __restrict__ pb, const int32_t* __restrict__ pv, int64_t np,
                            uint64_t* __restrict__ keys, uint32_t* __restrict__ vals)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < np; k += (int64_t)gridDim.x * blockDim.x) {
        keys[k] = ((uint64_t)(uint32_t)pb[k] << 32) | (uint32_t)pv[k];
        vals[k] = (uint32_t)k;
    }
}

__global__ void k_pair_unkey(const uint64_t* __restrict__ keys, int64_t np, int32_t* __restrict__ pb,
                             int32_t* __restrict__ pv)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < np; k += (int64_t)gridDim.x * blockDim.x) {
        pb[k] = (int32_t)(keys[k] >> 32);
        pv[k] = (int32_t)(keys[k] & 0xffffffffu);
    }
}
}  // namespace

void launch_pair_order(int32_t* pb, int32_t* pv, int64_t np, uint64_t* keys, uint32_t* vals, SortBufs& b,
                       cudaStream_t s)
{
    int64_t g = nblk(np, 256);
    if (g > 8 * sm_count()) g = 8 * sm_count();
    k_pair_keys<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(pb, pv, np, keys, vals);
    count_launches(1);
    radix_sort_u64(keys, vals, np, 63, b, s);
    k_pair_unkey<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(keys, np, pb, pv);
    count_launches(1);
}

void launch_pair_labels(const int32_t* pb, const int32_t* pv, int64_t np, const float4* body, const uint32_t* sys_of,
                        const SysParams* sysp, NodeTables nt, float eps, float G, float* feat, float* lab,
                        float* fac, cudaStream_t s)
{
    k_pair_labels<<<nblk(np, 128), 128, 0, s>>>(pb, pv, np, body, sys_of, sysp, nt, eps, G, feat, lab, fac);
    count_launches(1);
}

int mlp_sum_blocks(int64_t n)
{
    const int64_t b = (n + kSumThreads - 1) / kSumThreads;
    return (int)(b < kMlpSumBlocks ? b : kMlpSumBlocks);
}

void launch_mlp_maps(const float* X, const float* T, const float* F, int64_t n, double* part, float* maps,
                     float* wscale, cudaStream_t s)
{
    const int nb = mlp_sum_blocks(n);
    k_mlp_sums<<<nb, kSumThreads, 0, s>>>(X, T, F, n, part);
    k_mlp_maps<<<1, 32 * kMapWarps, 0, s>>>(part, nb, n, maps, wscale);
    count_launches(2);
}

void launch_mlp_rows(const float* X, const float* T, int64_t n, const float* maps, float* rows, float* tout,
                     cudaStream_t s)
{
    int64_t g = (n * kMlpInPad + 255) / 256;
    if (g > 16 * sm_count()) g = 16 * sm_count();
    k_mlp_rows<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(X, T, n, maps, rows, tout);
    count_launches(1);
}

void launch_mlp_weights(float* w, int64_t n, int mode, const float* wscale, int32_t* bad, cudaStream_t s)
{
    int64_t g = (n + 255) / 256;
    if (g > 16 * sm_count()) g = 16 * sm_count();
    k_mlp_weights<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(w, n, mode, wscale, bad);
    count_launches(1);
}

void launch_mlp_init(float* params, uint64_t seed, cudaStream_t s)
{
    k_mlp_init<<<nblk(kMlpNParam, 256), 256, 0, s>>>(params, seed);
    count_launches(1);
}

void launch_mlp_shuffle(int64_t n, uint64_t key, int32_t* idx, cudaStream_t s)
{
    int h = 1;
    while (((int64_t)1 << (2 * h)) < n) h++;
    int64_t g = (n + 255) / 256;
    if (g > 16 * sm_count()) g = 16 * sm_count();
    k_mlp_shuffle<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(n, h, key, idx);
    count_launches(1);
}

void launch_node_features(const Info* info, int64_t cap_m, const SysParams* sysp, NodeTables nt, float eps,
                          const void* model, cudaStream_t s)
{
    int64_t g = (cap_m + 255) / 256;
    if (g > 16 * sm_count()) g = 16 * sm_count();
    k_node_features<<<(unsigned)(g < 1 ? 1 : g), 256, 0, s>>>(info, sysp, nt, eps, (const MlpDev*)model);
    count_launches(1);
}

size_t mlp_dev_size() { return sizeof(MlpDev); }
size_t mlp_frag_size() { return sizeof(MlpFrag); }

}  // namespace tc
