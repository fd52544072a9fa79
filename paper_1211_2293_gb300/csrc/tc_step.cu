// tc_step.cu -- moving the bodies (kick-drift-kick leapfrog), FP64
// diagnostics and the direct-summation reference.
//
// Paper, Sec. 3.1: after the force summation each body updates its position
// and velocity.  The integrator is not named; the kick-drift-kick leapfrog
// (velocity Verlet) is used: v += a dt/2; x += v dt; forces; v += a dt/2.
#include <cfloat>

#include "tc_f32x2.cuh"
#include "tc_internal.cuh"

namespace tc {

namespace {

// v' = v + a*hk, x' = x + v'*dt, each a separately rounded float32 op.  A
// step whose build or walk raised the error word leaves the state as it is
// (the error is reported at the next synchronisation).
__device__ __forceinline__ bool failed(const Info* info) { return *(volatile const int32_t*)&info->err != 0; }

// The update is elementwise over the 3 n floats of the state: x += (v +=
// a hk) dt.  Each thread takes float4 runs (grid-stride) when the arrays are
// 16-byte aligned, else single floats; the error word is read once per warp.
__device__ __forceinline__ bool warp_failed(const Info* info)
{
    bool f = false;
    if ((threadIdx.x & 31) == 0) f = failed(info);
    return __shfl_sync(0xffffffffu, f, 0);
}

__device__ __forceinline__ float kick1(float v, float a, float hk) { return __fadd_rn(v, __fmul_rn(a, hk)); }
__device__ __forceinline__ float drift1(float x, float v, float dt) { return __fadd_rn(x, __fmul_rn(v, dt)); }

template <bool DRIFT, bool VEC>
__global__ void k_kick_drift(float* __restrict__ pos, float* __restrict__ vel, const float* __restrict__ acc,
                             int64_t n3, float hk, float dt, const Info* info)
{
    if (warp_failed(info)) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t done = 0;
    if (VEC) {
        const int64_t n4 = n3 >> 2;
        float4* v4 = reinterpret_cast<float4*>(vel);
        float4* p4 = reinterpret_cast<float4*>(pos);
        const float4* a4 = reinterpret_cast<const float4*>(acc);
        for (int64_t i = i0; i < n4; i += stride) {
            const float4 a = a4[i];
            float4 v = v4[i];
            v.x = kick1(v.x, a.x, hk);
            v.y = kick1(v.y, a.y, hk);
            v.z = kick1(v.z, a.z, hk);
            v.w = kick1(v.w, a.w, hk);
            v4[i] = v;
            if (DRIFT) {
                float4 x = p4[i];
                x.x = drift1(x.x, v.x, dt);
                x.y = drift1(x.y, v.y, dt);
                x.z = drift1(x.z, v.z, dt);
                x.w = drift1(x.w, v.w, dt);
                p4[i] = x;
            }
        }
        done = n4 << 2;
    }
    for (int64_t i = done + i0; i < n3; i += stride) {
        const float v = kick1(vel[i], acc[i], hk);
        vel[i] = v;
        if (DRIFT) pos[i] = drift1(pos[i], v, dt);
    }
}

// Results for the caller, who keeps what was there where the force phase
// failed.  The kernel looks at the error word itself, so one wait serves the
// copy and the word, and takes both arrays in one launch (a call with the
// potential over 2079 bodies 31 us, its wait included, 34 as two copies): the
// first `blocks` blocks the accelerations.  A thread copies kCopy elements, all loads first; an array's
// first block the up to three floats behind them.
constexpr int kCopy = 4;
template <typename T>
struct CopyJob {
    T* dst;
    const T* src;
    int64_t n;
    int rest;
};

template <typename T>
__global__ void __launch_bounds__(256) k_copy_good(CopyJob<T> acc, CopyJob<T> pot, unsigned blocks, const Info* info)
{
    const bool first = blockIdx.x < blocks;
    const CopyJob<T> j = first ? acc : pot;
    const int64_t i0 = (int64_t)(first ? blockIdx.x : blockIdx.x - blocks) * (256 * kCopy) + threadIdx.x;
    T x[kCopy];
#pragma unroll
    for (int k = 0; k < kCopy; k++)
        if (i0 + k * 256 < j.n) x[k] = j.src[i0 + k * 256];
    if (warp_failed(info)) return;
#pragma unroll
    for (int k = 0; k < kCopy; k++)
        if (i0 + k * 256 < j.n) j.dst[i0 + k * 256] = x[k];
    if (i0 < j.rest)
        reinterpret_cast<float*>(j.dst + j.n)[i0] = reinterpret_cast<const float*>(j.src + j.n)[i0];
}

// KE, PE = 1/2 sum m pot, P, L in FP64; block sums, then FP64 atomics
__global__ void k_diag(const float* __restrict__ pos, const float* __restrict__ vel, const float* __restrict__ mass,
                       const float* __restrict__ pot, int64_t n, double* __restrict__ out)
{
    __shared__ double sm[8][8];
    double q[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double m = mass[i];
        double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
        double vx = vel[3 * i], vy = vel[3 * i + 1], vz = vel[3 * i + 2];
        q[0] += 0.5 * m * (vx * vx + vy * vy + vz * vz);
        if (pot) q[1] += 0.5 * m * (double)pot[i];
        q[2] += m * vx;
        q[3] += m * vy;
        q[4] += m * vz;
        q[5] += m * (y * vz - z * vy);
        q[6] += m * (z * vx - x * vz);
        q[7] += m * (x * vy - y * vx);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 8; k++) {
#pragma unroll
        for (int o = 16; o; o >>= 1) q[k] += __shfl_xor_sync(0xffffffffu, q[k], o);
        if (lane == 0) sm[k][w] = q[k];
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        double s = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); k++) s += sm[threadIdx.x][k];
        atomicAdd(&out[threadIdx.x], s);
    }
}

// Direct summation for ns targets over the bodies of each target's system
// (original order).  FP32 terms; each 256-source tile is summed in FP32 and
// added in FP64.
//
// Block (bx, s) takes the 256 targets from 256 bx on and slice s of the
// source tiles of their systems (the union of the systems' ranges, tiles
// counted from its start); k_direct_reduce adds the slices in order (a single
// one writes the results itself).  With
// one block per 256 targets and no slices, the 4096 sampled targets of an
// accuracy check kept 16 of 152 SMs busy: 44.6 ms over 2^20 bodies, 1.9 of
// 80 TFLOP/s; sliced and packed 1.9 ms, 45 TFLOP/s.  A thread holds four
// targets as two packed pairs, so each paired FP32 instruction serves two of
// them and the broadcast loads of a source (stored twice, {x, x}) serve four; per target the operations and
// their order inside a tile are those of the scalar loop, bit for bit.  The
// bound is the FP32 pipe (13 operations a pair of bodies).
constexpr int kDirTile = 256;                       // sources per tile
constexpr int kDirTargets = 256;                    // targets per block
constexpr int kDirPack = 2;                         // packed target pairs per thread
constexpr int kDirThreads = kDirTargets / (2 * kDirPack);
constexpr int kDirBlocksPerSm = 8;

// FTZ: eps2 is a normal float, so r2 >= eps2 is never subnormal and the SFU
// approximation needs no range fix-up (same bits); else rsqrtf
template <bool FTZ>
__device__ __forceinline__ float dir_rsqrt(float x)
{
    return FTZ ? rsqrt_sfu(x) : rsqrtf(x);
}

// ONE: a single slice, which writes the results (a branch instead cost the
// sliced sums 1.3 %)
template <bool FTZ, bool ONE>
__global__ void __launch_bounds__(kDirThreads, kDirBlocksPerSm)
    k_direct(const float* __restrict__ pos, const float* __restrict__ mass, const uint32_t* __restrict__ sys_of,
             const SysParams* __restrict__ sysp, const int64_t* __restrict__ idx, int64_t ns, float eps2, float G,
             double* __restrict__ part, double* __restrict__ acc, double* __restrict__ pot)
{
    __shared__ __align__(16) f2 tile[kDirTile * 4];  // {x, x}, {y, y}, {z, z}, {m, m} per source
    __shared__ long long lo_sh, hi_sh;
    constexpr int NT = 2 * kDirPack;
    const int64_t t0 = (int64_t)blockIdx.x * kDirTargets;
    int64_t j0[NT], j1[NT];
    float xi[NT], yi[NT], zi[NT];
    if (threadIdx.x == 0) {
        const SysParams& P = sysp[sys_of[idx[t0]]];
        lo_sh = P.first;
        hi_sh = P.end;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NT; q++) {
        const int64_t t = t0 + q * kDirThreads + threadIdx.x;
        const int64_t i = idx[t < ns ? t : t0];
        const SysParams& P = sysp[sys_of[i]];
        j0[q] = P.first;
        j1[q] = P.end;
        xi[q] = pos[3 * i];
        yi[q] = pos[3 * i + 1];
        zi[q] = pos[3 * i + 2];
        if (j0[q] < lo_sh) atomicMin(&lo_sh, (long long)j0[q]);
        if (j1[q] > hi_sh) atomicMax(&hi_sh, (long long)j1[q]);
    }
    __syncthreads();
    const int64_t blo = lo_sh, bhi = hi_sh;
    bool one = true;
#pragma unroll
    for (int q = 0; q < NT; q++) one &= j0[q] == blo && j1[q] == bhi;
    one = __syncthreads_and(one) != 0;  // every target's system is the block's range
    f2 X[kDirPack], Y[kDirPack], Z[kDirPack];
#pragma unroll
    for (int p = 0; p < kDirPack; p++) {
        X[p] = f2pack(xi[2 * p], xi[2 * p + 1]);
        Y[p] = f2pack(yi[2 * p], yi[2 * p + 1]);
        Z[p] = f2pack(zi[2 * p], zi[2 * p + 1]);
    }
    const f2 E2 = f2pack(eps2, eps2);
    double ax[NT], ay[NT], az[NT], ph[NT];
#pragma unroll
    for (int q = 0; q < NT; q++) ax[q] = ay[q] = az[q] = ph[q] = 0.0;

    const int64_t ntiles = (bhi - blo + kDirTile - 1) / kDirTile;
    const int64_t per = (ntiles + gridDim.y - 1) / gridDim.y;
    const int64_t tl0 = (int64_t)blockIdx.y * per, tl1 = min(ntiles, tl0 + per);
    for (int64_t tl = tl0; tl < tl1; tl++) {
        const int64_t base = blo + tl * kDirTile;
        const int cnt = (int)min((int64_t)kDirTile, bhi - base);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += kDirThreads) {
            const int64_t j = base + k;
            const float x = pos[3 * j], y = pos[3 * j + 1], z = pos[3 * j + 2], m = mass[j];
            tile[4 * k] = f2pack(x, x);
            tile[4 * k + 1] = f2pack(y, y);
            tile[4 * k + 2] = f2pack(z, z);
            tile[4 * k + 3] = f2pack(m, m);
        }
        __syncthreads();
        if (one) {
            f2 tx[kDirPack], ty[kDirPack], tz[kDirPack], tp[kDirPack];
#pragma unroll
            for (int p = 0; p < kDirPack; p++) tx[p] = ty[p] = tz[p] = tp[p] = 0ull;
            const ulonglong2* t2 = reinterpret_cast<const ulonglong2*>(tile);
#pragma unroll 4
            for (int k = 0; k < cnt; k++) {
                const ulonglong2 xy = t2[2 * k], zm = t2[2 * k + 1];
#pragma unroll
                for (int p = 0; p < kDirPack; p++) {
                    const f2 dx = f2sub(xy.x, X[p]), dy = f2sub(xy.y, Y[p]), dz = f2sub(zm.x, Z[p]);
                    const f2 r2 = f2fma(dz, dz, f2fma(dy, dy, f2fma(dx, dx, E2)));
                    float ra, rb;
                    f2unpack(r2, ra, rb);
                    const f2 ri = f2pack(dir_rsqrt<FTZ>(ra), dir_rsqrt<FTZ>(rb));
                    const f2 mri = f2mul(zm.y, ri);
                    const f2 mri3 = f2mul(f2mul(mri, ri), ri);
                    tx[p] = f2fma(dx, mri3, tx[p]);
                    ty[p] = f2fma(dy, mri3, ty[p]);
                    tz[p] = f2fma(dz, mri3, tz[p]);
                    tp[p] = f2sub(tp[p], mri);
                }
            }
#pragma unroll
            for (int p = 0; p < kDirPack; p++) {
                float a, b;
                f2unpack(tx[p], a, b);
                ax[2 * p] += a;
                ax[2 * p + 1] += b;
                f2unpack(ty[p], a, b);
                ay[2 * p] += a;
                ay[2 * p + 1] += b;
                f2unpack(tz[p], a, b);
                az[2 * p] += a;
                az[2 * p + 1] += b;
                f2unpack(tp[p], a, b);
                ph[2 * p] += a;
                ph[2 * p + 1] += b;
            }
        } else {
            // targets of several systems: each sums its own part of the tile
#pragma unroll 1
            for (int q = 0; q < NT; q++) {
                float x = xi[0], y = yi[0], z = zi[0];
                int64_t a0 = j0[0], a1 = j1[0];
#pragma unroll
                for (int u = 1; u < NT; u++)
                    if (q == u) {
                        x = xi[u];
                        y = yi[u];
                        z = zi[u];
                        a0 = j0[u];
                        a1 = j1[u];
                    }
                const int k0 = (int)max((int64_t)0, min((int64_t)cnt, a0 - base));
                const int k1 = (int)max((int64_t)0, min((int64_t)cnt, a1 - base));
                float tx = 0.f, ty = 0.f, tz = 0.f, tp = 0.f;
                for (int k = k0; k < k1; k++) {
                    float sx, sy, sz, sm;
                    f2unpack(tile[4 * k], sx, sx);
                    f2unpack(tile[4 * k + 1], sy, sy);
                    f2unpack(tile[4 * k + 2], sz, sz);
                    f2unpack(tile[4 * k + 3], sm, sm);
                    const float dx = sx - x, dy = sy - y, dz = sz - z;
                    const float r2 = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, eps2)));
                    const float ri = dir_rsqrt<FTZ>(r2);
                    const float mri = __fmul_rn(sm, ri);
                    const float mri3 = __fmul_rn(__fmul_rn(mri, ri), ri);
                    tx = fmaf(dx, mri3, tx);
                    ty = fmaf(dy, mri3, ty);
                    tz = fmaf(dz, mri3, tz);
                    tp = __fsub_rn(tp, mri);
                }
#pragma unroll
                for (int u = 0; u < NT; u++)
                    if (q == u) {
                        ax[u] += tx;
                        ay[u] += ty;
                        az[u] += tz;
                        ph[u] += tp;
                    }
            }
        }
    }
    double* o = part + (int64_t)blockIdx.y * 4 * ns;
#pragma unroll
    for (int q = 0; q < NT; q++) {
        const int64_t t = t0 + q * kDirThreads + threadIdx.x;
        if (t >= ns) continue;
        if (ONE) {
            acc[3 * t] = (double)G * ax[q];
            acc[3 * t + 1] = (double)G * ay[q];
            acc[3 * t + 2] = (double)G * az[q];
            if (pot) pot[t] = (double)G * (ph[q] + (double)(mass[idx[t]] * rsqrtf(eps2)));
            continue;
        }
        o[t] = ax[q];
        o[ns + t] = ay[q];
        o[2 * ns + t] = az[q];
        o[3 * ns + t] = ph[q];
    }
}

// the slices' sums in order, scaled; the potential drops the target's own
// -m_i / eps term
__global__ void __launch_bounds__(256) k_direct_reduce(const double* __restrict__ part, int S, int64_t ns,
                                                       const float* __restrict__ mass,
                                                       const int64_t* __restrict__ idx, float eps2, float G,
                                                       double* __restrict__ acc, double* __restrict__ pot)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 4 * ns) return;
    double s = 0.0;
#pragma unroll 8
    for (int k = 0; k < S; k++) s += part[(int64_t)k * 4 * ns + e];
    const int64_t c = e / ns, t = e - c * ns;
    if (c < 3) acc[3 * t + c] = (double)G * s;
    else if (pot) pot[t] = (double)G * (s + (double)(mass[idx[t]] * rsqrtf(eps2)));
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

namespace {
template <bool DRIFT>
void launch_update(float* pos, float* vel, const float* acc, int64_t n, float hkick, float dt, const Info* info,
                   cudaStream_t s)
{
    const bool vec = ((reinterpret_cast<uintptr_t>(vel) | reinterpret_cast<uintptr_t>(acc) |
                       (DRIFT ? reinterpret_cast<uintptr_t>(pos) : 0)) & 15u) == 0;
    int64_t g = nblk(vec ? (3 * n + 3) / 4 : 3 * n, 256);
    if (g > 8 * sm_count()) g = 8 * sm_count();
    if (g < 1) g = 1;
    if (vec) k_kick_drift<DRIFT, true><<<(unsigned)g, 256, 0, s>>>(pos, vel, acc, 3 * n, hkick, dt, info);
    else k_kick_drift<DRIFT, false><<<(unsigned)g, 256, 0, s>>>(pos, vel, acc, 3 * n, hkick, dt, info);
    count_launches(1);
}
}  // namespace

void launch_kick_drift(float* pos, float* vel, const float* acc, int64_t n, float hkick, float dt, const Info* info,
                       cudaStream_t s)
{
    launch_update<true>(pos, vel, acc, n, hkick, dt, info, s);
}

// acc or pot may be null
void launch_copy_good(float* acc, const float* from_acc, float* pot, const float* from_pot, int64_t n,
                      const Info* info, cudaStream_t s)
{
    const auto go = [&](auto zero) {
        using T = decltype(zero);
        constexpr int64_t w = sizeof(T) / sizeof(float);
        const auto job = [&](float* to, const float* from, int64_t k) {
            if (!to) k = 0;
            return CopyJob<T>{reinterpret_cast<T*>(to), reinterpret_cast<const T*>(from), k / w, (int)(k % w)};
        };
        const auto blocks = [&](const CopyJob<T>& j) { return nblk(j.n + (j.rest > 0), 256 * kCopy); };
        const CopyJob<T> a = job(acc, from_acc, 3 * n), p = job(pot, from_pot, n);
        const unsigned ga = blocks(a), gp = blocks(p);
        if (ga + gp == 0) return;
        k_copy_good<T><<<ga + gp, 256, 0, s>>>(a, p, ga, info);
        count_launches(1);
    };
    const uintptr_t all = reinterpret_cast<uintptr_t>(acc) | reinterpret_cast<uintptr_t>(from_acc) |
                          reinterpret_cast<uintptr_t>(pot) | reinterpret_cast<uintptr_t>(from_pot);
    if ((all & 15u) == 0) go(float4{});
    else go(0.f);
}

void launch_kick(float* vel, const float* acc, int64_t n, float hkick, const Info* info, cudaStream_t s)
{
    launch_update<false>(nullptr, vel, acc, n, hkick, 0.f, info, s);
}

// FP32 throughput probe: every thread runs 8 independent chains of `iters`
// fused multiply-adds (scalar, or paired f32x2 instructions), 2 flops each;
// the chains' ends are folded into one store so nothing is dead code.
template <bool PAIRED>
__global__ void __launch_bounds__(256) k_fp32_probe(int iters, float seed, float* out)
{
    if (PAIRED) {
        unsigned long long a[4], m, c;
        const float x = seed + threadIdx.x * 1e-7f;
        asm("mov.b64 %0, {%1, %1};" : "=l"(m) : "f"(0.999999f));
        asm("mov.b64 %0, {%1, %1};" : "=l"(c) : "f"(1e-7f));
#pragma unroll
        for (int k = 0; k < 4; k++) asm("mov.b64 %0, {%1, %2};" : "=l"(a[k]) : "f"(x + k), "f"(x - k));
        for (int i = 0; i < iters; i++) {
#pragma unroll
            for (int k = 0; k < 4; k++) asm volatile("fma.rn.f32x2 %0, %0, %1, %2;" : "+l"(a[k]) : "l"(m), "l"(c));
        }
        float sum = 0.f;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            float lo, hi;
            asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a[k]));
            sum += lo + hi;
        }
        if (sum == 12345.f) out[0] = sum;
    } else {
        float a[8];
        const float x = seed + threadIdx.x * 1e-7f;
#pragma unroll
        for (int k = 0; k < 8; k++) a[k] = x + k;
        for (int i = 0; i < iters; i++) {
#pragma unroll
            for (int k = 0; k < 8; k++) asm volatile("fma.rn.f32 %0, %0, %1, %2;" : "+f"(a[k]) : "f"(0.999999f), "f"(1e-7f));
        }
        float sum = 0.f;
#pragma unroll
        for (int k = 0; k < 8; k++) sum += a[k];
        if (sum == 12345.f) out[0] = sum;
    }
}

void launch_fp32_probe(bool paired, int blocks, int iters, float* out, cudaStream_t s)
{
    if (paired) k_fp32_probe<true><<<blocks, 256, 0, s>>>(iters, 1.0f, out);
    else k_fp32_probe<false><<<blocks, 256, 0, s>>>(iters, 1.0f, out);
    count_launches(1);
}

void launch_diag(const float* pos, const float* vel, const float* mass, const float* pot, int64_t n, Info* info,
                 cudaStream_t s)
{
    cudaMemsetAsync(info->diag, 0, 8 * sizeof(double), s);
    unsigned nb = nblk(n, 256);
    if (nb > 1024) nb = 1024;
    k_diag<<<nb, 256, 0, s>>>(pos, vel, mass, pot, n, info->diag);
    count_launches(1);
}

// Source slices of a direct sum: with few target blocks as many as fill the SMs
// once (kDirBlocksPerSm resident blocks each); from eight target blocks on
// three times as many, so that blocks that end early (a scheduler favours its
// oldest warps) are replaced: 4096 targets of 2^20 / 2^18 bodies take 1910 /
// 563 us, 1999 / 586 when filled once, 1962 / 577 with four times; 512 targets
// of 2^20 464, 378 when filled once (the slices' sums to add).  Never more
// than there are tiles.
int direct_slices(int64_t n, int64_t ns)
{
    const int64_t nbx = nblk(ns, kDirTargets), room = (int64_t)kDirBlocksPerSm * sm_count();
    int64_t S = (nbx >= 8 ? 3 * room : room) / nbx;
    const int64_t tiles = (n + kDirTile - 1) / kDirTile;
    if (S > tiles) S = tiles;
    return (int)(S < 1 ? 1 : S);
}

// part: slices x 4 x ns doubles of scratch, none for one slice
void launch_direct(const float* pos, const float* mass, const uint32_t* sys_of, const SysParams* sysp,
                   const int64_t* idx, int64_t ns, int slices, float eps2, float G, double* part, double* acc,
                   double* pot, cudaStream_t s)
{
    const dim3 grid(nblk(ns, kDirTargets), (unsigned)slices);
    const auto go = [&](auto* kernel) {
        kernel<<<grid, kDirThreads, 0, s>>>(pos, mass, sys_of, sysp, idx, ns, eps2, G, part, acc, pot);
        count_launches(1);
    };
    if (slices == 1) eps2 >= FLT_MIN ? go(k_direct<true, true>) : go(k_direct<false, true>);
    else eps2 >= FLT_MIN ? go(k_direct<true, false>) : go(k_direct<false, false>);
    if (slices == 1) return;
    k_direct_reduce<<<nblk(4 * ns, 256), 256, 0, s>>>(part, slices, ns, mass, idx, eps2, G, acc, pot);
    count_launches(1);
}

}  // namespace tc
