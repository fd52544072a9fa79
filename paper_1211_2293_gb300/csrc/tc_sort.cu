// tc_sort.cu -- stable LSD radix sort of 64-bit keys with 32-bit values.
//
// The Morton keys are sorted with ties kept in original-index order (a
// stable sort), so bodies sharing a leaf are ordered by key, then by index.
// Written here (no CUB).
//
// Onesweep (8-bit digits): the digit histograms of every pass are counted
// beforehand (the kernel that forms the keys counts them), then each pass is
// a single kernel whose tiles find their place by decoupled look-back
// (tc_lookback.cuh): a tile publishes its per-digit counts, then adds up its
// predecessors' counts walking back until it meets an inclusive prefix, and
// publishes its own inclusive prefix.  A tile that gives up waiting sets the
// error word and writes nothing.
//
// Bound: the latency of a tile, not memory.  With __match_any_sync in 16
// dependent rounds and one predecessor per look-back round trip a pass over
// 2^22 items took 69 us, 10.7 of 23 stall cycles per instruction in the
// rounds; with peers from eight ballots, counters raised by shared atomics
// whose results are collected after eight rounds, and the digits' offsets
// formed by each tile itself it takes 58: 3 us of a tile's 20 are its loads,
// 5 its ranks, 5 to 14 its look-back (4 predecessors a round trip; 8 and 16
// were slower), 3 the exchange.
#include <mutex>

#include "tc_internal.cuh"
#include "tc_lookback.cuh"
#include "tc_pdl.cuh"

namespace tc {

namespace {

constexpr int kMaxDevices = 64;
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
// items per thread: tiles of 4096 items; of 1024 for up to kSortSmall items,
// where few large tiles leave most SMs without one
constexpr int kItemsLarge = 16, kItemsSmall = 4;
constexpr int64_t kSortSmall = 1 << 19;
constexpr int kLookAhead = 4;
__host__ __device__ constexpr int sort_tile(int items) { return kSortThreads * items; }
int sort_items(int64_t n) { return n <= kSortSmall ? kItemsSmall : kItemsLarge; }

// digit histograms of npass passes from bit shift0 up
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const uint64_t* keys, int64_t n, int npass,
                                                            uint32_t* ghist)
{
    pdl_begin();
    __shared__ uint32_t h[8][256];
    for (int i = threadIdx.x; i < 8 * 256; i += kSortThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = keys[k];
        for (int p = 0; p < npass; p++) atomicAdd(&h[p][(uint32_t)(key >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int p = 0; p < npass; p++) {
        const uint32_t c = h[p][threadIdx.x];
        if (c) atomicAdd(&ghist[p * 256 + threadIdx.x], c);
    }
}

__device__ __forceinline__ void sort_cp16(void* smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void sort_cp_wait() { asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory"); }

// Dynamic shared memory of one onesweep tile: the tile's items (keys, then
// values) in input order, then in their locally sorted order, so that the
// write to the output is one contiguous run per digit.
constexpr size_t onesweep_smem(int items) { return (size_t)sort_tile(items) * (sizeof(uint64_t) + sizeof(uint32_t)); }

// the lanes of `in` whose low eight bits of d equal this lane's
__device__ __forceinline__ unsigned digit_peers(unsigned in, uint32_t d)
{
    unsigned m = in;
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const unsigned bal = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        m &= (d >> b) & 1u ? bal : ~bal;
    }
    return m;
}

// SYS: the digit holds bits of the system of the value's body (SortPlan)
template <bool SYS, int ITEMS>
__global__ void __launch_bounds__(kSortThreads, 3)
    k_onesweep(const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
               uint32_t* vout, int64_t n, SortDigit dg, const uint32_t* ghist,
               unsigned long long* status, uint32_t* tile_counter, int32_t* err, const uint32_t* sys_of)
{
    pdl_begin();
    constexpr int TILE = sort_tile(ITEMS), WARP = 32 * ITEMS, H = ITEMS < 8 ? ITEMS : 8;
    extern __shared__ __align__(16) unsigned char dsm[];
    uint64_t* skey = reinterpret_cast<uint64_t*>(dsm);
    uint32_t* sval = reinterpret_cast<uint32_t*>(dsm + (size_t)TILE * sizeof(uint64_t));
    __shared__ uint32_t wh[kSortWarps][256];
    __shared__ uint32_t base[256];
    __shared__ uint32_t tstart[256];
    __shared__ uint32_t wsum[kSortWarps], gsum[kSortWarps];
    __shared__ int tile_sh;
    __shared__ int fail_sh;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t hist = ghist[threadIdx.x];  // items of this thread's digit in all tiles
    for (int i = threadIdx.x; i < kSortWarps * 256; i += kSortThreads) (&wh[0][0])[i] = 0;
    if (threadIdx.x == 0) {
        tile_sh = (int)atomicAdd(tile_counter, 1u);
        fail_sh = 0;
    }
    __syncthreads();
    const int tile = tile_sh;
    const int64_t tbase = (int64_t)tile * TILE;
    const int tile_n = (int)min((int64_t)TILE, n - tbase);

    // the tile's items into the staging buffer in their input order: a full
    // tile by cp.async, every 16-byte chunk in flight at once
    if (tile_n == TILE && ((reinterpret_cast<uintptr_t>(kin + tbase) | reinterpret_cast<uintptr_t>(vin + tbase)) & 15u) == 0) {
        const unsigned char* gk = reinterpret_cast<const unsigned char*>(kin + tbase);
        const unsigned char* gv = reinterpret_cast<const unsigned char*>(vin + tbase);
        unsigned char* sk = reinterpret_cast<unsigned char*>(skey);
        unsigned char* sv = reinterpret_cast<unsigned char*>(sval);
        for (int i = threadIdx.x; i < TILE / 2; i += kSortThreads) sort_cp16(sk + 16 * i, gk + 16 * i);
        for (int i = threadIdx.x; i < TILE / 4; i += kSortThreads) sort_cp16(sv + 16 * i, gv + 16 * i);
        sort_cp_wait();
    } else {
        for (int i = threadIdx.x; i < tile_n; i += kSortThreads) {
            skey[i] = kin[tbase + i];
            sval[i] = vin[tbase + i];
        }
    }
    __syncthreads();

    // stable ranks within the tile: warp w owns items [w * WARP, +WARP), 32 a
    // round; the lanes of a round with equal digits find each other by
    // ballots and the lowest reserves their places from the warp's counters
    const uint32_t lt = (1u << lane) - 1u;
    uint64_t key[ITEMS];
    uint32_t rank[(ITEMS + 1) / 2];   // two 16-bit ranks a word
    uint32_t dsys[(ITEMS + 3) / 4] = {};  // SYS: four digits a word
    if (SYS) {
        uint32_t sy[ITEMS];
#pragma unroll
        for (int r = 0; r < ITEMS; r++) {
            const int li = w * WARP + r * 32 + lane;
            sy[r] = li < tile_n ? sys_of[sval[li]] : 0u;
        }
#pragma unroll
        for (int r = 0; r < ITEMS; r++) {
            const int li = w * WARP + r * 32 + lane;
            const uint32_t d = dg.of(li < tile_n ? skey[li] : 0ull, sy[r]);
            dsys[r / 4] |= d << (8 * (r % 4));
        }
    }
    auto digit = [&](int r, uint64_t k) { return SYS ? (dsys[r / 4] >> (8 * (r % 4))) & 255u : (uint32_t)(k >> dg.kshift) & 255u; };
#pragma unroll
    for (int h = 0; h < ITEMS; h += H) {
        unsigned peers[H], old[H];
#pragma unroll
        for (int r = 0; r < H; r++) {
            const int li = w * WARP + (h + r) * 32 + lane;
            const bool ok = li < tile_n;
            key[h + r] = ok ? skey[li] : 0ull;
            const unsigned in = __ballot_sync(0xffffffffu, ok);
            peers[r] = digit_peers(in, digit(h + r, key[h + r]));
            if (!ok) peers[r] = 0u;
        }
#pragma unroll
        for (int r = 0; r < H; r++) {
            old[r] = 0u;
            if (peers[r] && (peers[r] & lt) == 0u) old[r] = atomicAdd(&wh[w][digit(h + r, key[h + r])], (uint32_t)__popc(peers[r]));
            __syncwarp();
        }
#pragma unroll
        for (int r = 0; r < H; r++) {
            const uint32_t o = __shfl_sync(0xffffffffu, old[r], peers[r] ? __ffs(peers[r]) - 1 : lane);
            const uint32_t k = o + __popc(peers[r] & lt);
            if ((h + r) % 2 == 0) rank[(h + r) / 2] = k;
            else rank[(h + r) / 2] |= k << 16;
        }
    }
    __syncthreads();

    // per digit: offsets of the warps inside the tile and the tile's count;
    // the digits' starts inside the tile and in the output (block scans);
    // then the decoupled look-back over the preceding tiles
    const int d = threadIdx.x;
    uint32_t run = 0;
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ww++) {
        const uint32_t c = wh[ww][d];
        wh[ww][d] = run;
        run += c;
    }
    volatile unsigned long long* st = status;
    st[(int64_t)tile * 256 + d] = (tile == 0 ? kFlagPrefix : kFlagAgg) | run;
    uint32_t goff;
    {
        uint32_t x = run, y = hist;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x2 = __shfl_up_sync(0xffffffffu, x, o), y2 = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) {
                x += x2;
                y += y2;
            }
        }
        if (lane == 31) {
            wsum[w] = x;
            gsum[w] = y;
        }
        __syncthreads();
        uint32_t before = 0, gbefore = 0;
        for (int ww = 0; ww < w; ww++) {
            before += wsum[ww];
            gbefore += gsum[ww];
        }
        tstart[d] = before + x - run;
        goff = gbefore + y - hist;
    }
    {
        uint32_t excl = 0;
        if (tile > 0) {
            // kLookAhead predecessors a round trip, taken in order up to the
            // first that has published nothing yet
            int64_t k = tile - 1;
            unsigned polls = 0;
            bool fail = false;
            while (k >= 0) {
                unsigned long long v[kLookAhead];
#pragma unroll
                for (int j = 0; j < kLookAhead; j++) {
                    v[j] = kFlagPrefix;  // before tile 0: a prefix of zero
                    if (k - j >= 0) v[j] = st[(k - j) * 256 + d];
                }
                int took = 0;
                bool done = false;
#pragma unroll
                for (int j = 0; j < kLookAhead; j++) {
                    const unsigned f = (unsigned)(v[j] >> 62);
                    if (!done && took == j && f != 0u) {
                        excl += (uint32_t)v[j];
                        took++;
                        done = f == 2u;
                    }
                }
                if (done) break;
                k -= took;
                if (took == 0) {
                    if (++polls > kLookbackMaxPolls) {
                        fail = true;
                        break;
                    }
                    if (polls > 64) __nanosleep(32);
                }
            }
            st[(int64_t)tile * 256 + d] = kFlagPrefix | (uint32_t)(excl + run);
            if (fail) {
                fail_sh = 1;
                atomicOr(err, kErrWorkLoop);
            }
        }
        base[d] = goff + excl;
    }
    __syncthreads();
    // the tile in its sorted order (positions are inside [0, tile_n)): the
    // keys are in registers, the values follow them
    uint32_t val[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int li = w * WARP + r * 32 + lane;
        if (li < tile_n) {
            const uint32_t dd = digit(r, key[r]);
            const uint32_t lp = tstart[dd] + wh[w][dd] + ((rank[r / 2] >> (16 * (r % 2))) & 0xffffu);
            val[r] = sval[li];
            skey[lp] = key[r];
            if (r % 2 == 0) rank[r / 2] = (rank[r / 2] & 0xffff0000u) | lp;
            else rank[r / 2] = (rank[r / 2] & 0xffffu) | (lp << 16);
        }
    }
    __syncthreads();  // every value has been read
#pragma unroll
    for (int r = 0; r < ITEMS; r++)
        if (w * WARP + r * 32 + lane < tile_n) sval[(rank[r / 2] >> (16 * (r % 2))) & 0xffffu] = val[r];
    __syncthreads();
    if (fail_sh) return;  // positions unknown: write nothing
    // write out: consecutive items of one digit go to consecutive places
#pragma unroll 4
    for (int i = threadIdx.x; i < tile_n; i += kSortThreads) {
        const uint64_t kk = skey[i];
        const uint32_t vv = sval[i];
        const uint32_t dd = SYS ? dg.of(kk, sys_of[vv]) : (uint32_t)(kk >> dg.kshift) & 255u;
        const uint32_t q = base[dd] + (uint32_t)i - tstart[dd];
        kout[q] = kk;
        vout[q] = vv;
    }
}

void sort_attributes();  // (below, after every kernel that it prepares)

}  // namespace

int64_t radix_status_words(int64_t n)
{
    const int64_t small = n < kSortSmall ? n : kSortSmall;  // a shorter sort in the same buffers may have more tiles
    const int64_t ts = (small + sort_tile(kItemsSmall) - 1) / sort_tile(kItemsSmall);
    const int64_t tl = (n + sort_tile(kItemsLarge) - 1) / sort_tile(kItemsLarge);
    return 256 * (int64_t)kSortMaxPasses * (ts > tl ? ts : tl);
}

int64_t radix_status_words(int64_t n, int npass)
{
    const int64_t tile = sort_tile(sort_items(n));
    return 256 * (int64_t)npass * ((n + tile - 1) / tile);
}

void launch_sort_passes(uint64_t* ka, uint32_t* va, uint64_t* kb, uint32_t* vb, int64_t n, const SortPlan& plan,
                        const uint32_t* sys_of, const SortBufs& b, ChainStream s)
{
    sort_attributes();
    const int items = sort_items(n);
    const int64_t nt = (n + sort_tile(items) - 1) / sort_tile(items);
    const size_t dsm = onesweep_smem(items);
    for (int p = 0; p < plan.npass; p++) {
        const SortDigit dg = plan.digit(p);
        unsigned long long* st = b.status + (size_t)p * nt * 256;
        auto go = [&](auto* kernel) {
            pdl_launch(kernel, nt, kSortThreads, dsm, s, ka, va, kb, vb, n, dg, b.ghist + 256 * p, st, b.tiles + p,
                       b.err, sys_of);
        };
        if (items == kItemsLarge) dg.sys ? go(k_onesweep<true, kItemsLarge>) : go(k_onesweep<false, kItemsLarge>);
        else dg.sys ? go(k_onesweep<true, kItemsSmall>) : go(k_onesweep<false, kItemsSmall>);
        count_launches(1);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
}

// ---------------------------------------------------- per-run completion
// After passes over bits [low_bit, 63) only, items with equal top bits (and
// equal system) sit together in value order; each such run is put in
// (key, val) order -- which, the values being distinct, is the order of
// the full sort.  A run of at most kShortRun items is ranked by its own
// threads (one item each, rank = the items of the run that precede it), a
// longer one by the block its first item lies in.
namespace {

constexpr int kShortRun = 32;

__device__ __forceinline__ bool same_run(const uint64_t* k, const uint32_t* v,
                                         const uint32_t* sys_of, int low_bit, int64_t i, int64_t j)
{
    if ((k[i] >> low_bit) != (k[j] >> low_bit)) return false;
    return !sys_of || sys_of[v[i]] == sys_of[v[j]];
}

__device__ __forceinline__ bool before(uint64_t ka, uint32_t va, uint64_t kb, uint32_t vb)
{
    return ka < kb || (ka == kb && va < vb);
}

// Also the bodies in that order: body[k] = (x, y, z, m) of the k-th item.
__global__ void __launch_bounds__(256) k_sort_runs(const uint64_t* kin, const uint32_t* vin,
                                                   uint64_t* kout, uint32_t* vout, int64_t n,
                                                   int low_bit, const uint32_t* sys_of,
                                                   const float* pos, const float* mass,
                                                   float4* body, int64_t run_max, int32_t* err)
{
    pdl_begin();
    __shared__ int nlong;
    __shared__ int64_t longs[256 / kShortRun + 1];
    __shared__ long long en_sh;
    auto put = [&](int64_t at, uint64_t k, uint32_t v) {
        kout[at] = k;
        vout[at] = v;
        body[at] = make_float4(pos[3 * (int64_t)v], pos[3 * (int64_t)v + 1], pos[3 * (int64_t)v + 2], mass[v]);
    };
    for (int64_t i0 = (int64_t)blockIdx.x * 256; i0 < n; i0 += (int64_t)gridDim.x * 256) {
        if (threadIdx.x == 0) nlong = 0;
        __syncthreads();
        const int64_t i = i0 + threadIdx.x;
        if (i < n) {
            int64_t st = i;
            while (st > 0 && i - st < kShortRun && same_run(kin, vin, sys_of, low_bit, st - 1, i)) st--;
            int64_t en = i + 1;
            while (en < n && en - st <= kShortRun && same_run(kin, vin, sys_of, low_bit, en, i)) en++;
            if (en - st > kShortRun || (st > 0 && i - st >= kShortRun && same_run(kin, vin, sys_of, low_bit, st - 1, i))) {
                // part of a long run: its first item lists it for the block
                if (i == 0 || !same_run(kin, vin, sys_of, low_bit, i - 1, i)) longs[atomicAdd(&nlong, 1)] = i;
            } else {
                const uint64_t k = kin[i];
                const uint32_t v = vin[i];
                int64_t r = 0;
                for (int64_t j = st; j < en; j++) r += before(kin[j], vin[j], k, v) ? 1 : 0;
                put(st + r, k, v);
            }
        }
        __syncthreads();
        for (int q = 0; q < nlong; q++) {
            const int64_t st = longs[q];
            // the run's end: the first item past st of another run (or n), or
            // past run_max items
            const int64_t lim = min(n, st + run_max + 1);
            if (threadIdx.x == 0) en_sh = lim;
            __syncthreads();
            for (int64_t j = st + 1 + threadIdx.x; j < lim; j += blockDim.x) {
                if (j >= *(volatile long long*)&en_sh) break;
                if (!same_run(kin, vin, sys_of, low_bit, j, st)) atomicMin(&en_sh, (long long)j);
            }
            __syncthreads();
            const int64_t en = en_sh;
            if (en - st > run_max) {
                if (threadIdx.x == 0) atomicOr(err, kErrSortRun | kErrCapacity);
            } else {
                for (int64_t j0 = st + threadIdx.x; j0 < en; j0 += blockDim.x) {
                    const uint64_t k = kin[j0];
                    const uint32_t v = vin[j0];
                    int64_t r = 0;
                    for (int64_t j = st; j < en; j++) r += before(kin[j], vin[j], k, v) ? 1 : 0;
                    put(st + r, k, v);
                }
            }
            __syncthreads();
        }
    }
}

}  // namespace

// ---------------------------------------------------- small sorts
// Up to kBlockSortMax items: every pass, the completion of the runs and the
// bodies in one block, the items staying in shared memory.  Each of the four
// or five passes of 4096 items took 10 us as a launch of its own (tile
// counter, loads, look-back, stores); here all of them and the completion
// take 26.  With 12 items a thread (10007 items) one block took 72 us, more
// than the launches.  Runs of more than kBlockRun items (a tree far deeper
// than the last one, or leaves of many bodies) are not ranked, in quadratic
// time: the block goes on to sort every digit (builds of 4000 bodies in runs of
// 64 / 100 / 200 / 400 / 1000: 158 / 196 / 272 / 448 / 933 us ranked, 153 / 157
// / 163 / 193 / 254 so).
namespace {

constexpr int kBlockThreads = 1024, kBlockWarps = kBlockThreads / 32;
constexpr int kBlockRun = 64;
constexpr size_t block_sort_smem(int items)
{
    return (size_t)kBlockThreads * items * (sizeof(uint64_t) + sizeof(uint32_t)) + kBlockWarps * 256 * sizeof(uint32_t);
}

template <int ITEMS>
__global__ void __launch_bounds__(kBlockThreads, 1)
    k_sort_block(const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
                 uint32_t* vout, int n, SortPlan plan, const uint32_t* sys_of,
                 const float* pos, const float* mass, float4* body)
{
    pdl_begin();
    constexpr int WARP = 32 * ITEMS;
    extern __shared__ __align__(16) unsigned char dsm[];
    uint64_t* skey = reinterpret_cast<uint64_t*>(dsm);
    uint32_t* sval = reinterpret_cast<uint32_t*>(skey + kBlockThreads * ITEMS);
    uint32_t* wh = sval + kBlockThreads * ITEMS;  // [warp][256]
    __shared__ uint32_t wsum[kBlockWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint64_t key[ITEMS];
    uint32_t val[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int li = w * WARP + r * 32 + lane;
        key[r] = li < n ? kin[li] : 0ull;
        val[r] = li < n ? vin[li] : 0u;
    }
    int st[ITEMS], en[ITEMS];  // the items' runs of equal top bits (and system)
    for (;;) {
        for (int p = 0; p < plan.npass; p++) {
            const SortDigit dg = plan.digit(p);
            for (int i = threadIdx.x; i < kBlockWarps * 256; i += kBlockThreads) wh[i] = 0u;
            __syncthreads();
            uint32_t rank[ITEMS];  // the digit above a 16-bit rank
#pragma unroll
            for (int r = 0; r < ITEMS; r++) {
                const bool ok = w * WARP + r * 32 + lane < n;
                const uint32_t dd = dg.of(key[r], dg.sys && ok ? sys_of[val[r]] : 0u);
                unsigned peers = digit_peers(__ballot_sync(0xffffffffu, ok), dd);
                if (!ok) peers = 0u;
                uint32_t old = 0u;
                if (peers && (peers & lt) == 0u) old = atomicAdd(&wh[w * 256 + dd], (uint32_t)__popc(peers));
                __syncwarp();
                rank[r] = (dd << 16) | (__shfl_sync(0xffffffffu, old, peers ? __ffs(peers) - 1 : lane) + __popc(peers & lt));
            }
            __syncthreads();
            // where each (digit, warp) starts: thread (d, part) of four adds up
            // eight warps of digit d, then the digits are scanned
            {
                const int d = threadIdx.x >> 2, part = threadIdx.x & 3;
                uint32_t c[8], sum = 0;
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    c[k] = wh[(part * 8 + k) * 256 + d];
                    sum += c[k];
                }
                uint32_t incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (lane == 31) wsum[w] = incl;
                __syncthreads();
                uint32_t run = incl - sum;
                for (int k = 0; k < w; k++) run += wsum[k];
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    wh[(part * 8 + k) * 256 + d] = run;
                    run += c[k];
                }
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < ITEMS; r++) {
                if (w * WARP + r * 32 + lane < n) {
                    const uint32_t lp = wh[w * 256 + (rank[r] >> 16)] + (rank[r] & 0xffffu);
                    skey[lp] = key[r];
                    sval[lp] = val[r];
                }
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < ITEMS; r++) {
                const int li = w * WARP + r * 32 + lane;
                if (li < n) {
                    key[r] = skey[li];
                    val[r] = sval[li];
                }
            }
        }
        if (plan.npass == 0) {
#pragma unroll
            for (int r = 0; r < ITEMS; r++) {
                const int li = w * WARP + r * 32 + lane;
                if (li < n) {
                    skey[li] = key[r];
                    sval[li] = val[r];
                }
            }
            __syncthreads();
        }
        if (plan.low_bit == 0) break;
        bool lng = false;
#pragma unroll
        for (int r = 0; r < ITEMS; r++) {
            const int i = w * WARP + r * 32 + lane;
            st[r] = i;
            en[r] = i + 1;
            if (i >= n) continue;
            const uint32_t* so = plan.sys_bits > 0 ? sys_of : nullptr;
            while (st[r] > 0 && i - st[r] < kBlockRun && same_run(skey, sval, so, plan.low_bit, st[r] - 1, i)) st[r]--;
            while (en[r] < n && en[r] - i < kBlockRun && same_run(skey, sval, so, plan.low_bit, en[r], i)) en[r]++;
            lng |= en[r] - st[r] > kBlockRun;
        }
        if (!__syncthreads_or(lng)) break;
        // (the items lie in value order within equal keys, so do the passes leave them)
        plan = SortPlan::make(plan.low_bit + plan.kb, 0, plan.sys_bits);
    }
    // the items' places: within its run each item goes to the rank of its
    // (key, val)
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int i = w * WARP + r * 32 + lane;
        if (i >= n) continue;
        int at = i;
        if (plan.low_bit > 0) {
            at = st[r];
            for (int j = st[r]; j < en[r]; j++) at += before(skey[j], sval[j], key[r], val[r]) ? 1 : 0;
        }
        const int64_t v = val[r];
        kout[at] = key[r];
        vout[at] = val[r];
        body[at] = make_float4(pos[3 * v], pos[3 * v + 1], pos[3 * v + 2], mass[v]);
    }
}

constexpr int kBlockItems = 4;

}  // namespace

namespace {

// the kernels need more than the default 48 KB of shared memory: a
// per-device function attribute, set once per device (before any stream
// capture: every context builds eagerly once before it captures a step)
void sort_attributes()
{
    static std::mutex mu;
    static bool done[kMaxDevices] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= kMaxDevices || done[dev]) return;
    const auto set = [](auto* kernel, size_t bytes) {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    set(k_onesweep<false, kItemsLarge>, onesweep_smem(kItemsLarge));
    set(k_onesweep<true, kItemsLarge>, onesweep_smem(kItemsLarge));
    set(k_onesweep<false, kItemsSmall>, onesweep_smem(kItemsSmall));
    set(k_onesweep<true, kItemsSmall>, onesweep_smem(kItemsSmall));
    set(k_sort_block<kBlockItems>, block_sort_smem(kBlockItems));
    done[dev] = true;
}

}  // namespace

static_assert(kBlockSortMax == kBlockThreads * kBlockItems, "one block's items");

void launch_sort_block(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout, int64_t n,
                       const SortPlan& plan, const uint32_t* sys_of, const float* pos, const float* mass, float4* body,
                       ChainStream s)
{
    sort_attributes();
    pdl_launch(k_sort_block<kBlockItems>, 1, kBlockThreads, block_sort_smem(kBlockItems), s, kin, vin, kout, vout,
               (int)n, plan, sys_of, pos, mass, body);
    count_launches(1);
}

void launch_sort_runs(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout, int64_t n,
                      int low_bit, const uint32_t* sys_of, const float* pos, const float* mass, float4* body,
                      int64_t run_max, int32_t* err, ChainStream s)
{
    if (run_max < 1 || run_max > kSortRunMax) run_max = kSortRunMax;
    int64_t g = (n + 255) / 256;
    if (g > 16 * sm_count()) g = 16 * sm_count();
    pdl_launch(k_sort_runs, g < 1 ? 1 : g, 256, 0, s, kin, vin, kout, vout, n, low_bit, sys_of, pos, mass, body,
               run_max, err);
    count_launches(1);
}

void radix_sort_u64(uint64_t* keys, uint32_t* vals, int64_t n, int nbits, SortBufs& b, cudaStream_t s)
{
    if (n <= 1) return;
    const SortPlan plan = SortPlan::make(nbits, 0, 0);
    cudaMemsetAsync(b.ghist, 0, kSortMaxPasses * 256 * sizeof(uint32_t), s);
    cudaMemsetAsync(b.tiles, 0, kSortMaxPasses * sizeof(uint32_t), s);
    cudaMemsetAsync(b.status, 0, radix_status_words(n, plan.npass) * sizeof(unsigned long long), s);
    int64_t hb = (n + kSortThreads * 16 - 1) / (kSortThreads * 16);
    if (hb > 4 * sm_count()) hb = 4 * sm_count();
    pdl_launch(k_sort_hist, hb, kSortThreads, 0, s, keys, n, plan.npass, b.ghist);
    count_launches(1);
    launch_sort_passes(keys, vals, b.keys_alt, b.vals_alt, n, plan, nullptr, b, s);
    if (plan.npass % 2) {
        cudaMemcpyAsync(keys, b.keys_alt, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(vals, b.vals_alt, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
    }
}

// Self-test of the look-back's wait limit: one block is handed tile 1 of a
// two-tile pass whose tile 0 never runs, so its look-back finds no
// predecessor, gives up after kLookbackMaxPolls polls, sets kErrWorkLoop in
// *err and writes nothing.  All buffers are the caller's device memory:
// keys/vals/kout/vout two large tiles of items, status 2 * 256 words (zeroed
// here), counter 1 word, hist 256 words.
cudaError_t sort_wait_selftest(uint64_t* keys, uint32_t* vals, uint64_t* kout, uint32_t* vout,
                               unsigned long long* status, uint32_t* counter, uint32_t* hist, int32_t* err,
                               cudaStream_t s)
{
    const int64_t n = sort_selftest_items();
    cudaMemsetAsync(status, 0, 2 * 256 * sizeof(unsigned long long), s);
    cudaMemsetAsync(hist, 0, 256 * sizeof(uint32_t), s);
    const uint32_t one = 1;  // the only block launched takes tile 1
    cudaMemcpyAsync(counter, &one, sizeof(one), cudaMemcpyHostToDevice, s);
    sort_attributes();
    pdl_launch(k_onesweep<false, kItemsLarge>, 1, kSortThreads, onesweep_smem(kItemsLarge), s, keys, vals, kout, vout,
               n, SortPlan::make(63, 0, 0).digit(0), hist, status, counter, err, nullptr);
    count_launches(1);
    return cudaGetLastError();
}
int64_t sort_selftest_items() { return 2 * (int64_t)sort_tile(kItemsLarge); }

}  // namespace tc
