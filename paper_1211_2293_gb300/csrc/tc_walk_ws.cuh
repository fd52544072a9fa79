// tc_walk_ws.cuh -- the force phase with the tree walk and the force loop on
// different warps (included by tc_walk_ws_unit.cu).
//
// k_walk gives each warp a whole group: it walks a step, sums a full list
// tile, walks on, and the walk of one warp hardly overlaps the sums of the
// others.  Here a block holds teams of one producer warp and C consumer
// warps.  The producer walks a group as k_walk does (opening test, ballots,
// list compaction) but never sums: it fills list tiles in a ring of slots in
// shared memory -- at any time one open tile of cells and one of bodies --
// and hands a tile over when it is full or the group ends.  The consumers
// hold the group's bodies and sum every tile they are handed (the
// compensated paired-FP32 loop), then write the group's accelerations.
//
// Bound.  Both kinds of warp share an SM partition's issue slots and
// register-file ports; with two of each per partition the measured time is
// the sum of the loop's cycles (29 per pair of sources and body, its rate
// alone) and about 1.3 per producer instruction -- hiding latency (the next
// step's nodes loaded ahead, three consumers for two producers, 24 warps of
// 80 registers) changed nothing, fewer instructions and fewer empty lanes
// did.  Walk of a 2^20 cube at theta 0.5 1.38 -> 1.22 ms, of a 2^22 Plummer
// sphere at theta 0.62 5.64 -> 5.21 ms with the layouts, the ordering of the
// groups by layout (launch_group_order) and the step below.
//
// The walk's step.  The stack holds opened cells.  A step tests the children
// of eight of them, eight lanes to a cell, two cells to a lane; opened leaves
// wait until 32 of them list their bodies together.  With single nodes on the
// stack, scans that packed children and bodies were most of a step: 14.3
// thousand instructions per group of the cube, now 10.2.
//
// Bodies over lanes.  A group holds 1 to gmax bodies, 45 of 64 on average.
// With one or two bodies per lane a quarter of the loop's work went to lanes
// without a body.  Instead a warp's lanes are cut into S slices of 32 / S
// lanes; every slice holds all of the group's bodies, K per lane, and sums
// every S-th quad of the list, so the work grows in steps of 32 K / S body
// slots: (K, S) = (1, 2), (1, 1), (5, 4), (3, 2), (2, 1) take groups of up
// to 16, 32, 40, 48, 64 bodies (three and four per lane up to 128).  Lanes
// holding a body, over the groups of a 2^20 cube / Plummer sphere: 0.76 /
// 0.78 -> 0.86 / 0.89.  The slices' compensated sums are added at the end of
// the group by TwoSum.
//
// Parts of a group.  With few groups the longest list is what a walk waits
// for (a group of packed siblings whose box spans a dense octant lists most
// of a small system: 16000 bodies, 357 us on a team while the chip idles).
// Then every group is walked in P parts, a task each.  All parts walk the
// cells that hold more than a 64th of the system, and of what is below those
// each takes every P-th cell, by its place (sharing out the stack after
// some steps instead left one part the dense core that most of a Plummer
// sphere's lists lie in: 317 us).  A part leaves its compensated
// sums in memory; the one that ends last adds them in the parts' order, so
// the sums don't depend on which it is.  Walk of Plummer spheres at theta
// 0.5, us, with the consumers of a team sharing its list as before / with
// parts: 4096 bodies 81 / 38, 10000 171 / 55, 16000 205 / 100, 50000 130 /
// 128.  walk_parts (tc_api.cu) states the rule.
//
// Tiles.  The four planes x, y, z, m of a tile are contiguous: 32 lanes
// store 32 entries without bank conflicts (pair-interleaved entries of four
// words met four-way conflicts) and a 16-byte load yields four sources as
// two packed pairs.
//
// Order.  Tiles are handed over at positions 0, 1, 2, ...; position k uses
// mbarriers full[k % kWsSlots] and empty[k % kWsSlots] and names its slot in
// seq[k % kWsSlots].  The producer holds two slots, so at most kWsSlots - 2
// positions are in flight; it takes slots in the order in which they were
// handed over, after waiting for that position's empty barrier, so a
// position's words are never rewritten before its consumers left it, and the
// two sides never wait on each other in a cycle.
//
// Every wait is bounded (about a second of SM clock): a wait that runs out
// raises kErrWorkLoop in the error word and its warp returns, so a fault in
// the protocol ends the kernel with an error instead of a hang.
#pragma once

namespace tc {

namespace {

// The quadrupole walk (precise, gmax up to 64) is the walk with list tiles of
// 32 cells: ten planes hold a cell with its second moments, fetched by
// cp.async as the bodies are (the trace is summed in the loop), and a slot of
// that size 64 to 95 bodies.  Bound by the loop: 97 cycles per pair of cells
// and body, where its 32 packed operations take 80 with the register reads of
// the FMAs.  Plummer spheres at theta 0.68, us, one-warp walk / this: 10^4
// bodies 365 / 59, 10^5 251 / 231, 10^6 1941 / 1865, 4 10^6 7909 / 7710.
// (Cell loop unrolled twice: 1971 at 10^6, it no longer fits the instruction
// cache with the others.)
constexpr int kWsQuadTile = 32;
__host__ __device__ constexpr bool ws_quad(int tile) { return tile == kWsQuadTile; }

// tiles per team: two open, the others in flight
__host__ __device__ constexpr int ws_slots(int tile) { return tile > 128 || ws_quad(tile) ? 5 : 6; }
constexpr int kWsMaxPairs = 4;                   // pairs per block (block = 2 x pairs warps)
constexpr long long kWsWaitCycles = 1ll << 31;   // about 1 s of SM clock

// entries of a plane: a step adds at most 64 to a tile that was not full,
// and the count is padded to a multiple of 16 (four slices of quads)
__host__ __device__ constexpr int ws_cap(int tile) { return tile + 64; }
__host__ __device__ constexpr int ws_planes(int tile) { return ws_quad(tile) ? 10 : 4; }
// of a body tile: entries at which it is handed over, entries of a plane
__host__ __device__ constexpr int ws_body_tile(int tile) { return ws_quad(tile) ? 64 : tile; }
__host__ __device__ constexpr int ws_body_cap(int tile) { return ws_quad(tile) ? 128 : ws_cap(tile); }

// slot header (64 bytes at the front of a slot)
struct WsHdr {
    int32_t flags;  // kWs*
    int32_t n;      // entries, padded to a multiple of 16 with massless ones
    int32_t gfirst, gend;
    int32_t group, part;
    float corr[3];  // the learned correction (at the group's last position)
    int32_t pad;
    double ref[3];  // centre of the group's reference cube (absolute, FP64)
};
static_assert(sizeof(WsHdr) == 64, "slot header");
enum : int32_t { kWsFirst = 1, kWsLast = 2, kWsDone = 4, kWsAbort = 8, kWsBodies = 16 };

// One team's shared memory: barriers and slot numbers (128 bytes), the ring,
// the walk stack (first child and number of children of each opened cell),
// the opened leaves, the consumer's body positions (absolute and
// reference-relative), and where the producer runs the network its pending
// cells and rows (the block's copy of the network lies in front of the teams).
// nb: body slots of a group (64, or 128 for gmax 128).
__host__ __device__ constexpr size_t ws_slot_bytes(int tile) { return sizeof(WsHdr) + (size_t)ws_planes(tile) * ws_cap(tile) * 4; }
__host__ __device__ constexpr size_t ws_pos_bytes(int nb) { return (size_t)6 * nb * 4; }
constexpr int kWsShared = 128;     // of a stack entry's number of children: all parts walk it
constexpr int kWsSharedFrac = 64;  // cells of more than this fraction of a system (16 to 128 measure alike)
constexpr int kWsLeaves = 96;  // opened leaves: up to 31 left over + 64 of a step
__host__ __device__ constexpr size_t ws_team_bytes(int tile, int stack, int nb, bool rows)
{
    return 128 + ws_slots(tile) * ws_slot_bytes(tile) + (size_t)stack * 4 + ((stack + 15) & ~15) + kWsLeaves * 8 +
           32 * 4 + ws_pos_bytes(nb) + (rows ? (kPend + 32 * kRowW) * 4 : 0);
}
static_assert(2 * 8 * ws_slots(64) + 4 * ws_slots(64) <= 128 && 2 * 8 * ws_slots(256) + 4 * ws_slots(256) <= 128,
              "a team's barriers and slot numbers");
__host__ __device__ constexpr int ws_body_slots(int gmax) { return gmax > 64 ? 128 : 64; }

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}

// one lane of a warp arrives, after a __syncwarp that orders the other
// lanes' accesses before it
__device__ __forceinline__ void mbar_arrive(uint64_t* b)
{
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}" ::"r"(smem_addr(b)) : "memory");
}

// the opened leaves' bodies reach a slot by cp.async; before the producer's
// arrival on the full barrier every lane makes the barrier track its copies
// (cp.async.mbarrier.arrive without .noinc: the pending count rises now and
// falls when the lane's copies have landed), so the phase completes only
// once the bodies are in the tile
__device__ __forceinline__ void mbar_track_copies(uint64_t* b)
{
    asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];" ::"r"(smem_addr(b)) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(b)), "r"(parity)
        : "memory");
    return ok != 0;
}

// wait for the phase of the given parity to complete, at most
// kWsWaitCycles; warp-uniform result (false if any lane ran out)
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity)
{
    bool ok = mbar_try(b, parity);
    if (!ok) {
        const long long t0 = clock64();
        while (!(ok = mbar_try(b, parity)))
            if (clock64() - t0 > kWsWaitCycles) break;
    }
    return __all_sync(0xffffffffu, ok);
}

// what the warps of a team share
struct WsTeam {
    uint64_t *full, *empty;
    int32_t* seq;
    unsigned char* slots;
    int slot_bytes;
    __device__ __forceinline__ WsHdr* hdr(int slot) const { return reinterpret_cast<WsHdr*>(slots + slot * slot_bytes); }
    __device__ __forceinline__ float* tile(int slot) const
    {
        return reinterpret_cast<float*>(slots + slot * slot_bytes + sizeof(WsHdr));
    }
};

// One group, or part `part` of one (part < 0: whole), on one consumer warp:
// positions from the warp's shared-memory copy, K bodies per lane, S slices.  Starts at position k
// (whose full barrier has been waited for) and returns the position after
// the group's last tile, or -1 when a wait ran out.
template <int K, int S, int TILE, bool PRECISE, bool POT, int LEARNED>
__device__ __forceinline__ int consume_group(const WsTeam& t, int k, const float* __restrict__ pos, int nb, int part,
                                             int gfirst, int ng, const WalkArgs& a)
{
    constexpr int L = 32 / S;                      // lanes of a slice
    constexpr bool QUADW = ws_quad(TILE);
    constexpr int CAP = ws_body_cap(TILE);  // (of all tiles but the quadrupole walk's cells)
    constexpr int kWsSlots = ws_slots(TILE);
    constexpr int kUnroll = K >= 3 ? 1 : (K == 2 ? 2 : 4);  // about eight pairs of sources and bodies in flight
    // pairs summed between two compensations (the quadrupole walk: as the
    // one-warp walk's smallest tiles)
    constexpr int kFold = QUADW ? 48 : (TILE + 32) / 2;
    const int lane = threadIdx.x & 31;
    const int sl = lane / L, j = lane % L;
    const f2 E2 = f2pack(a.eps2, a.eps2);
    f2 ax[K], ay[K], az[K], ph[K];
    float sx[K], sy[K], sz[K], sp[K], cx[K], cy[K], cz[K], cp[K];
#pragma unroll
    for (int b = 0; b < K; b++) {
        ax[b] = ay[b] = az[b] = ph[b] = 0ull;
        sx[b] = sy[b] = sz[b] = sp[b] = cx[b] = cy[b] = cz[b] = cp[b] = 0.f;
    }
    auto fold = [&]() {
#pragma unroll
        for (int b = 0; b < K; b++) {
            two_sum_acc(sx[b], cx[b], f2sum(ax[b]));
            two_sum_acc(sy[b], cy[b], f2sum(ay[b]));
            two_sum_acc(sz[b], cz[b], f2sum(az[b]));
            if (POT) two_sum_acc(sp[b], cp[b], f2sum(ph[b]));
            ax[b] = ay[b] = az[b] = ph[b] = 0ull;
        }
    };
    int pairs = 0;
    int flags;
    float corr[3] = {0.f, 0.f, 0.f};
    for (;;) {
        const int slot = t.seq[k % kWsSlots];
        const WsHdr* h = t.hdr(slot);
        flags = h->flags;
        if (LEARNED == 2 && (flags & kWsLast)) {
#pragma unroll
            for (int v = 0; v < 3; v++) corr[v] = h->corr[v];
        }
        const int rounds = (h->n >> 2) / S;        // n is a multiple of 4 S
        if (rounds > 0) {
            if (PRECISE) {
                if (pairs + 2 * rounds > kFold && pairs > 0) {
                    fold();
                    pairs = 0;
                }
                pairs += 2 * rounds;
            }
            // cells are relative to the group's reference cube in the
            // precise mode, bodies absolute
            const float* q = pos + ((PRECISE && !(flags & kWsBodies)) ? 3 * nb : 0) + j;
            f2 X[K], Y[K], Z[K];
#pragma unroll
            for (int b = 0; b < K; b++) {
                const float x = q[b * L], y = q[nb + b * L], z = q[2 * nb + b * L];
                X[b] = f2pack(x, x);
                Y[b] = f2pack(y, y);
                Z[b] = f2pack(z, z);
            }
            const float* p = t.tile(slot) + 4 * sl;
            if (QUADW && !(flags & kWsBodies)) {
                constexpr int QC = ws_cap(TILE);
#pragma unroll 1
                for (int r = 0; r < rounds; r++, p += 4 * S) {
#pragma unroll
                    for (int hh = 0; hh < 2; hh++) {
                        const auto plane = [&](int k) { return *reinterpret_cast<const f2*>(p + k * QC + 2 * hh); };
                        const f2 Q[6] = {plane(4), plane(5), plane(6), plane(7), plane(8), plane(9)};
                        const f2 tr = f2mul(f2pack(-1.5f, -1.5f), f2add(f2add(Q[0], Q[3]), Q[5]));
                        const f2 x2 = plane(0), y2 = plane(1), z2 = plane(2), m2 = plane(3);
#pragma unroll
                        for (int b = 0; b < K; b++)
                            quad_term<POT>(x2, y2, z2, m2, Q, tr, X[b], Y[b], Z[b], E2, ax[b], ay[b], az[b], ph[b]);
                    }
                }
            } else
#pragma unroll(kUnroll)
            for (int r = 0; r < rounds; r++, p += 4 * S) {
                const ulonglong2 xx = *reinterpret_cast<const ulonglong2*>(p);
                const ulonglong2 yy = *reinterpret_cast<const ulonglong2*>(p + CAP);
                const ulonglong2 zz = *reinterpret_cast<const ulonglong2*>(p + 2 * CAP);
                const ulonglong2 mm = *reinterpret_cast<const ulonglong2*>(p + 3 * CAP);
#pragma unroll
                for (int hh = 0; hh < 2; hh++) {
                    const f2 x2 = hh ? xx.y : xx.x, y2 = hh ? yy.y : yy.x, z2 = hh ? zz.y : zz.x, m2 = hh ? mm.y : mm.x;
#pragma unroll
                    for (int b = 0; b < K; b++) {
                        const f2 dx = f2sub(x2, X[b]);
                        const f2 dy = f2sub(y2, Y[b]);
                        const f2 dz = f2sub(z2, Z[b]);
                        const f2 r2 = f2fma(dz, dz, f2fma(dy, dy, f2fma(dx, dx, E2)));
                        float r2a, r2b;
                        f2unpack(r2, r2a, r2b);
                        const f2 ri = f2pack(rsqrt_sfu(r2a), rsqrt_sfu(r2b));
                        const f2 mri = f2mul(m2, ri);
                        const f2 mri3 = f2mul(mri, f2mul(ri, ri));
                        ax[b] = f2fma(dx, mri3, ax[b]);
                        ay[b] = f2fma(dy, mri3, ay[b]);
                        az[b] = f2fma(dz, mri3, az[b]);
                        if (POT) ph[b] = f2sub(ph[b], mri);
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&t.empty[k % kWsSlots]);
        k++;
        if (flags & kWsLast) break;
        if (!mbar_wait(&t.full[k % kWsSlots], (k / kWsSlots) & 1)) return -1;
    }
    fold();  // (plain mode: the plain sums, uncompensated so far)
    // the slices' sums: both lanes of an exchange form the same sum
#pragma unroll
    for (int o = L; o < 32; o <<= 1) {
#pragma unroll
        for (int b = 0; b < K; b++) {
            auto join = [&](float& s, float& comp) {
                const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, comp, o);
                comp = __fadd_rn(comp, c2);
                two_sum_acc(s, comp, s2);
            };
            join(sx[b], cx[b]);
            join(sy[b], cy[b]);
            join(sz[b], cz[b]);
            if (POT) join(sp[b], cp[b]);
        }
    }
    if (part >= 0) {
        float* o = a.part_sum + (int64_t)part * kPartPlanes * a.part_stride + gfirst;
#pragma unroll
        for (int b = 0; b < K; b++) {
            const int i = j + b * L;
            if (b % S != sl || i >= ng) continue;
            o[0 * a.part_stride + i] = sx[b];
            o[1 * a.part_stride + i] = cx[b];
            o[2 * a.part_stride + i] = sy[b];
            o[3 * a.part_stride + i] = cy[b];
            o[4 * a.part_stride + i] = sz[b];
            o[5 * a.part_stride + i] = cz[b];
            if (POT) {
                o[6 * a.part_stride + i] = sp[b];
                o[7 * a.part_stride + i] = cp[b];
            }
            if (LEARNED == 2) {
#pragma unroll
                for (int v = 0; v < 3; v++) o[(6 + v) * a.part_stride + i] = corr[v];
            }
        }
        return k;
    }
    const auto with = [&](float f, int v) { return LEARNED == 2 ? f + corr[v] : f; };
    if (flags & kWsAbort) return k;
#pragma unroll
    for (int b = 0; b < K; b++) {
        const int i = j + b * L;
        if (b % S != sl || i >= ng) continue;
        const int64_t o = a.perm[gfirst + i];
        a.acc[3 * o + 0] = with(a.G * (sx[b] + cx[b]), 0);
        a.acc[3 * o + 1] = with(a.G * (sy[b] + cy[b]), 1);
        a.acc[3 * o + 2] = with(a.G * (sz[b] + cz[b]), 2);
        // (the potential drops the body's own term, -m_i / eps, summed with the list)
        if (POT) a.pot[o] = a.G * ((sp[b] + cp[b]) + a.body[gfirst + i].w * rsqrtf(a.eps2));
    }
    return k;
}

// A part of group g has been summed (the sums are in memory): the warp of
// the group's last part adds the parts' sums in their order.
template <bool POT, int LEARNED>
__device__ __forceinline__ void add_parts(int g, int gfirst, int ng, const WalkArgs& a)
{
    const int lane = threadIdx.x & 31;
    const int parts = 1 << a.part_log2;
    __threadfence();  // each lane's sums before the count
    __syncwarp();
    int32_t done = 0;
    if (lane == 0) done = atomicAdd(&a.part_done[g], 1);
    done = __shfl_sync(0xffffffffu, done, 0);
    if (done != parts - 1) return;
    __threadfence();
    if (lane == 0) a.part_done[g] = 0;  // for the next force phase on this tree
    for (int i = lane; i < ng; i += 32) {
        float s[POT ? 4 : 3], c[POT ? 4 : 3];
#pragma unroll
        for (int v = 0; v < (POT ? 4 : 3); v++) s[v] = c[v] = 0.f;
        float corr[3] = {0.f, 0.f, 0.f};
        const float* o = a.part_sum + gfirst + i;
        for (int p = 0; p < parts; p++, o += kPartPlanes * a.part_stride) {
            if (LEARNED == 2) {
#pragma unroll
                for (int v = 0; v < 3; v++) corr[v] += __ldcg(o + (6 + v) * a.part_stride);
            }
#pragma unroll
            for (int v = 0; v < (POT ? 4 : 3); v++) {
                c[v] = __fadd_rn(c[v], __ldcg(o + (2 * v + 1) * a.part_stride));
                two_sum_acc(s[v], c[v], __ldcg(o + 2 * v * a.part_stride));
            }
        }
        const auto with = [&](float f, int v) { return LEARNED == 2 ? f + corr[v] : f; };
        const int64_t b = a.perm[gfirst + i];
        a.acc[3 * b + 0] = with(a.G * (s[0] + c[0]), 0);
        a.acc[3 * b + 1] = with(a.G * (s[1] + c[1]), 1);
        a.acc[3 * b + 2] = with(a.G * (s[2] + c[2]), 2);
        if (POT) a.pot[b] = a.G * ((s[POT ? 3 : 0] + c[POT ? 3 : 0]) + a.body[gfirst + i].w * rsqrtf(a.eps2));
    }
    __syncwarp();
}

// inclusive warp prefix sum, two instructions a step
__device__ __forceinline__ unsigned ws_incl_scan(unsigned x)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        asm volatile(
            "{\n .reg .pred p;\n .reg .b32 t;\n shfl.sync.up.b32 t|p, %0, %1, 0, -1;\n @p add.u32 %0, %0, t;\n}"
            : "+r"(x)
            : "r"(o));
    return x;
}

// LEARNED: band cells (accepted, two bodies or more, s >= band d) go through
// the correction's network.  1: the producer records them, and the group's
// record (box centre and frame), for k_band_eval after the walk; 2: the
// producer runs the network on 32 of them at a time, as k_walk does, and hands
// the group's correction over with its last tile.  What that costs is
// instructions and their fetch, not the tensor unit (2^20 bodies at theta
// 0.667, band 0.55: 1.31 ms against 1.00 without a band cell; 13 % more
// instructions, fetch stalls 0.47 -> 0.79 per issue, issue 60 -> 55 %, the
// tensor unit busy 6 % of the cycles, 8 a mma.sync).  Plummer spheres at
// theta 0.67, band 0.55, us, one-warp walk / recorded / in the producers: 5000
// bodies 154 / 79 / 48, 20000 182 / 100 / 77, 300000 446 / 424 / 414, 2^22
// 5326 / 5273 / 5205.
template <int TILE, bool PRECISE, bool POT, int LEARNED>
__global__ void __launch_bounds__(2 * 32 * kWsMaxPairs, 2) k_walk_ws(WalkArgs a, int stack_cap, int nb)
{
    constexpr bool QUADW = ws_quad(TILE);
    constexpr int kTile = TILE, kBodyTile = ws_body_tile(TILE);
    constexpr int CAP = ws_cap(TILE), BCAP = ws_body_cap(TILE);
    constexpr int kWsSlots = ws_slots(TILE);
    static_assert(4 * BCAP <= ws_planes(TILE) * CAP && kBodyTile + 32 <= BCAP && (!QUADW || PRECISE), "tile layout");
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int teams = (int)(blockDim.x >> 6);
    const bool producer = warp < teams;
    const int team = producer ? warp : warp - teams;
    const size_t team_bytes = ws_team_bytes(TILE, stack_cap, nb, LEARNED == 2);
    unsigned char* base = smem + (LEARNED == 2 ? mlp_frag_bytes() : 0) + (size_t)team * team_bytes;
    WsTeam t;
    t.full = reinterpret_cast<uint64_t*>(base);
    t.empty = t.full + kWsSlots;
    t.seq = reinterpret_cast<int32_t*>(t.empty + kWsSlots);
    t.slots = base + 128;
    t.slot_bytes = (int)ws_slot_bytes(TILE);
    uint32_t* stk = reinterpret_cast<uint32_t*>(base + 128 + kWsSlots * ws_slot_bytes(TILE));
    int2* leaves = reinterpret_cast<int2*>(stk + stack_cap);  // first body, bodies
    int32_t* row = reinterpret_cast<int32_t*>(leaves + kWsLeaves);
    uint8_t* stn = reinterpret_cast<uint8_t*>(row + 32);
    float* pos = reinterpret_cast<float*>(stn + ((stack_cap + 15) & ~15));
    uint32_t* pend = reinterpret_cast<uint32_t*>(pos + 6 * nb);  // LEARNED 2
    uint32_t* rows = pend + kPend;
    MlpFrag* mlp = reinterpret_cast<MlpFrag*>(smem);

    const Info* info = a.info;
    if (info->err & kErrCapacity) return;  // the build stopped: no tree to walk (uniform: no barrier used yet)
    if (LEARNED == 2)  // the inference part at the front of the device model
        for (int i = threadIdx.x; i < (int)(sizeof(MlpFrag) / 4); i += blockDim.x)
            reinterpret_cast<uint32_t*>(mlp)[i] = reinterpret_cast<const uint32_t*>(a.mlp)[i];
    if (producer && lane == 0) {
        for (int s = 0; s < kWsSlots; s++) {
            mbar_init(&t.full[s], 1);
            mbar_init(&t.empty[s], 1);
        }
    }
    __syncthreads();

    if (producer) {
        // ------------------------------------------------------------ producer
        const uint32_t lt = (1u << lane) - 1u, le = lt | (1u << lane);
        const bool list_stats = a.hash != nullptr;
        const int64_t G = info->G;
        const NodeTables nt = a.nt;
        int k = 0;              // positions handed over so far
        int taken = 2;          // slots taken so far: two open ones
        uint32_t handed = 0;    // slots of the last kWsSlots positions, the latest in the low nibble
        int cs = 0, bs = 1;     // the open cell tile's and body tile's slots
        float *ctile = t.tile(0), *btile = t.tile(1);
        int cn = 0, bn = 0;     // their entries
        int first = kWsFirst;   // the group's next position is its first
        int gfirst = 0, gend = 0, g = 0;
        const int parts = 1 << a.part_log2;
        int part = 0;
        double gx = 0, gy = 0, gz = 0;
        float corr[3] = {0.f, 0.f, 0.f};  // LEARNED 2: this group's (or part's)
        bool alive = true;
        // hands a slot's tile of n entries over (flags: kind, last, ...) and
        // takes the next free slot in its place (-1: a wait ran out)
        auto hand_over = [&](int slot, int n, int flags) -> int {
            float* tile = t.tile(slot);
            const int n16 = (n + 15) & ~15;
            if (n + lane < n16) {  // massless padding
                const int cap = flags & kWsBodies ? BCAP : CAP;
                tile[n + lane] = 0.f;
                tile[cap + n + lane] = 0.f;
                tile[2 * cap + n + lane] = 0.f;
                tile[3 * cap + n + lane] = 0.f;
                if (QUADW && !(flags & kWsBodies))
#pragma unroll
                    for (int i = 4; i < 10; i++) tile[i * CAP + n + lane] = 0.f;
            }
            if (lane == 0) {
                WsHdr* h = t.hdr(slot);
                h->flags = flags | first;
                h->n = n16;
                if (LEARNED == 2) h->corr[0] = corr[0], h->corr[1] = corr[1], h->corr[2] = corr[2];
                if (first) {
                    h->gfirst = gfirst;
                    h->gend = gend;
                    h->group = g;
                    h->part = part;
                    h->ref[0] = gx;
                    h->ref[1] = gy;
                    h->ref[2] = gz;
                }
                t.seq[k % kWsSlots] = slot;
            }
            first = 0;
            if (QUADW || (flags & kWsBodies)) mbar_track_copies(&t.full[k % kWsSlots]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&t.full[k % kWsSlots]);
            handed = (handed << 4) | (uint32_t)slot;
            k++;
            const int take = taken++;
            if (take < kWsSlots) return take;  // never used yet
            const int pos = take - kWsSlots;   // the position whose slot is taken; k - 1 is the latest
            if (!mbar_wait(&t.empty[pos % kWsSlots], (pos / kWsSlots) & 1)) {
                if (lane == 0) atomicOr(&a.info->err, kErrWorkLoop);
                alive = false;
                return 0;
            }
            return (int)((handed >> (4 * (k - 1 - pos))) & 15u);
        };
        auto close_cells = [&](int flags) {
            cs = hand_over(cs, cn, flags);
            ctile = t.tile(cs);
            cn = 0;
        };
        auto close_bodies = [&](int flags) {
            bs = hand_over(bs, bn, flags | kWsBodies);
            btile = t.tile(bs);
            bn = 0;
        };
        // band cells: this warp's chunk of the record (cbase < 0: none yet)
        int64_t cbase = -1;
        int cused = kBandChunk;
        const int64_t band_lim = (a.band_cap / kBandChunk) * kBandChunk;
        auto band_append = [&](bool band, int v, int g) {
            const unsigned bm = __ballot_sync(0xffffffffu, band);
            const int c = __popc(bm);
            if (c == 0) return;
            const int rank = __popc(bm & lt);
            const int room = kBandChunk - cused;
            int64_t nbase = -1;
            if (c > room) {  // a new chunk for the cells that do not fit
                long long x = -1;
                if (lane == 0) {
                    x = (long long)atomicAdd(a.band_n, (unsigned long long)kBandChunk);
                    if (x + kBandChunk > band_lim) {
                        atomicOr(&a.info->err, kErrBand);
                        x = -1;
                    }
                }
                nbase = __shfl_sync(0xffffffffu, x, 0);
            }
            if (band) {
                int64_t pos = -1;
                if (rank < room) pos = cbase + cused + rank;
                else if (nbase >= 0) pos = nbase + (rank - room);
                if (pos >= 0) a.band[pos] = make_int2(v, g);
            }
            if (c > room) {
                cbase = nbase;
                cused = nbase >= 0 ? c - room : kBandChunk;
            } else {
                cused += c;
            }
        };
        while (alive) {
            unsigned task = 0;
            if (lane == 0) task = atomicAdd(&a.info->work[a.work_slot], 1u);
            task = __shfl_sync(0xffffffffu, task, 0);
            g = (int)(task >> a.part_log2);
            part = (int)(task & (unsigned)(parts - 1));
            if (g >= G) {
                first = 0;
                close_cells(kWsDone);
                // the unused tail of the chunk: no cell
                if (LEARNED == 1 && cbase >= 0)
                    for (int i = cused + lane; i < kBandChunk; i += 32) a.band[cbase + i] = make_int2(-1, 0);
                break;
            }
            if (a.glist) g = __ldg(a.glist + g);
            gfirst = a.gfirst[g];
            gend = a.gfirst[g + 1];
            first = kWsFirst;
            const uint32_t sysid = a.sys_of[gfirst];
            const SysParams& SP = a.sysp[sysid];
            const double ud = 0.5 * SP.h;
            const float uf = SP.uf;
            const float Lf = SP.Lf;
            const int4 rc = nt.c[a.gref[g]];
            gx = SP.c0[0] + (double)rc.x * ud;
            gy = SP.c0[1] + (double)rc.y * ud;
            gz = SP.c0[2] + (double)rc.z * ud;
            // the group's bounding box
            float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
            for (int i = gfirst + lane; i < gend; i += 32) {
                const float4 qb = a.body[i];
                lo[0] = fminf(lo[0], qb.x); hi[0] = fmaxf(hi[0], qb.x);
                lo[1] = fminf(lo[1], qb.y); hi[1] = fmaxf(hi[1], qb.y);
                lo[2] = fminf(lo[2], qb.z); hi[2] = fmaxf(hi[2], qb.z);
            }
#pragma unroll
            for (int kk = 0; kk < 3; kk++) {
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    lo[kk] = fminf(lo[kk], __shfl_xor_sync(0xffffffffu, lo[kk], o));
                    hi[kk] = fmaxf(hi[kk], __shfl_xor_sync(0xffffffffu, hi[kk], o));
                }
            }
            // box relative to the reference centre: integer part (units of
            // u) + float remainder; lane k < 6 splits one bound
            int kb = 0;
            float fb = 0.f;
            if (lane < 6) {
                const int ax = lane % 3;
                const double gref = ax == 0 ? gx : (ax == 1 ? gy : gz);
                const double tt = (double)(lane < 3 ? lo[ax] : hi[ax]) - gref;
                const double kf = floor(tt / ud);
                kb = (int)kf;
                fb = (float)(tt - kf * ud);
            }
            float klof[3], khif[3], flo[3], fhi[3];
            const float rcf[3] = {(float)rc.x, (float)rc.y, (float)rc.z};
#pragma unroll
            for (int kk = 0; kk < 3; kk++) {
                klof[kk] = (float)__shfl_sync(0xffffffffu, kb, kk);
                khif[kk] = (float)__shfl_sync(0xffffffffu, kb, kk + 3);
                flo[kk] = __shfl_sync(0xffffffffu, fb, kk);
                fhi[kk] = __shfl_sync(0xffffffffu, fb, kk + 3);
            }
            // the group's box centre, reference-relative (as k_walk forms it)
            float xc[3];
#pragma unroll
            for (int kk = 0; kk < 3; kk++) xc[kk] = 0.5f * (fmaf(klof[kk], uf, flo[kk]) + fmaf(khif[kk], uf, fhi[kk]));
            int qn = 0, nevals = 0;  // LEARNED 2: pending band cells, cells evaluated
            corr[0] = corr[1] = corr[2] = 0.f;
            if (LEARNED == 1 && lane == 0 && part == 0) {
                // the group's record: the centre and the frame the network's
                // rows need
                a.grec[2 * (int64_t)g] = make_float4(xc[0], xc[1], xc[2], uf);
                a.grec[2 * (int64_t)g + 1] =
                    make_float4(__int_as_float(rc.x), __int_as_float(rc.y), __int_as_float(rc.z), Lf);
            }
            int Lc = 0, Lb = 0;
            unsigned long long hsh = 0;
            const bool fast_side = ((__float_as_int(Lf) >> 23) & 255) > kMaxLevel + 1;
            bool overflow = false;
            int sp = 0;  // opened cells whose children are to be tested
            int shared_min;  // all parts of a group walk cells of more bodies
            int ln = 0;  // opened leaves whose bodies are not listed yet
            {
                // the system's root: holds every body, always opened
                const int4 rb = nt.b[sysid];
                shared_min = rb.y / kWsSharedFrac;
                if ((rb.w >> 8) != 0) {
                    if (lane == 0) {
                        stk[0] = (uint32_t)rb.z;
                        stn[0] = (uint8_t)((rb.w >> 8) | (parts > 1 ? kWsShared : 0));
                    }
                    sp = 1;
                } else if (part == 0) {
                    if (lane == 0) {
                        leaves[0] = make_int2(rb.x, rb.y);
                        if (list_stats) hsh = mix64(2ull * sysid + 2ull);
                    }
                    ln = 1;
                }
            }
            __syncwarp();
            // the bodies of the last m <= 32 opened leaves -> the body tile,
            // 32 at a time: row[r] turns a body's offset among them into its
            // index, r found by counting the leaves that start at or before it
            auto list_leaves = [&](int m) {
                int2 lf = make_int2(0, 0);
                if (lane < m) lf = leaves[ln - m + lane];
                ln -= m;
                const int incl = (int)ws_incl_scan((unsigned)lf.y);
                const int excl = incl - lf.y;
                const int T = __shfl_sync(0xffffffffu, incl, 31);
                Lb += T;
                row[lane] = lf.x - excl;
                __syncwarp();
                const int32_t* r = row - 1;
                for (int o = 0; o < T; o += 32) {
                    const unsigned st = (unsigned)(excl - o);
                    const unsigned starts = __reduce_or_sync(0xffffffffu, lane < m && st < 32u ? 1u << st : 0u);
                    if (o + lane < T) {
                        const float* src4 = reinterpret_cast<const float*>(&a.body[r[__popc(starts & le)] + o + lane]);
                        float* q = btile + bn + lane;
                        cp_async4(q, src4);
                        cp_async4(q + BCAP, src4 + 1);
                        cp_async4(q + 2 * BCAP, src4 + 2);
                        cp_async4(q + 3 * BCAP, src4 + 3);
                    }
                    r += __popc(starts);
                    bn += min(32, T - o);
                    if (bn >= kBodyTile) {
                        close_bodies(0);
                        if (!alive) break;
                    }
                }
                __syncwarp();
            };
            const int slot8 = lane >> 3, child8 = lane & 7;
            while (sp > 0) {
                // A step tests the children of the up to eight topmost
                // opened cells, eight lanes to a cell and two cells to a
                // lane: cells have 7 to 8 children on average, so a fixed
                // place for each beats scans that pack them, a cell's
                // records are read as whole lines, and the two tests of a
                // lane are independent.
                const int np = min(sp, 8);
                sp -= np;
                int v[2], stn8[2], push[2];
                int4 nbd[2];
                float4 src[2];
                float band_e2[2];
                bool acc[2], oleaf[2], oint[2];
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const int e = slot8 + 4 * u;
                    stn8[u] = (int)stn[sp + min(e, np - 1)];
                    const bool have = e < np && child8 < (stn8[u] & 15);
                    v[u] = have ? (int)stk[sp + e] + child8 : (int)sysid;  // (the other lanes read a root's records)
                    nbd[u] = __ldg(&nt.b[v[u]]);
                    const float4 na = __ldg(&nt.a[v[u]]);
                    const int4 cc = __ldg(&nt.c[v[u]]);
                    const bool overlap = (nbd[u].x < gend) && (gfirst < nbd[u].x + nbd[u].y);
                    const float D[3] = {(float)cc.x - rcf[0], (float)cc.y - rcf[1], (float)cc.z - rcf[2]};
                    const float off[3] = {na.x, na.y, na.z};
                    float e2 = 0.f;
#pragma unroll
                    for (int kk = 0; kk < 3; kk++) {
                        const float lo_c = fmaf(klof[kk] - D[kk], uf, flo[kk]);
                        const float hi_c = fmaf(khif[kk] - D[kk], uf, fhi[kk]);
                        const float ee = fmaxf(fmaxf(lo_c - off[kk], off[kk] - hi_c), 0.f);
                        e2 = fmaf(ee, ee, e2);
                    }
                    const float sz = pow2_down(Lf, nbd[u].w & 255, fast_side);
                    acc[u] = have && !overlap && (sz * sz) < a.theta2 * e2;
                    band_e2[u] = e2;
                    if (PRECISE) {
                        src[u] = make_float4(fmaf(D[0], uf, off[0]), fmaf(D[1], uf, off[1]), fmaf(D[2], uf, off[2]), na.w);
                    } else {
                        src[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (acc[u]) src[u] = nt.d[v[u]];
                    }
                    const bool open = have && !acc[u];
                    oint[u] = open && (nbd[u].w >> 8) != 0;
                    oleaf[u] = open && (nbd[u].w >> 8) == 0;
                    push[u] = nbd[u].w >> 8;
                    if (stn8[u] & kWsShared) {  // below a cell that all parts walk
                        // (the cell's coordinates on its level's grid: siblings
                        // differ, and a system's place in a batch is no matter)
                        const int sh = kMaxLevel + 1 - (nbd[u].w & 255);
                        const int own = (cc.x >> sh) + 2 * (cc.y >> sh) + 4 * (cc.z >> sh);
                        const bool mine = (own & (parts - 1)) == part;
                        acc[u] = acc[u] && mine;
                        oleaf[u] = oleaf[u] && mine;
                        if (nbd[u].y > shared_min) push[u] |= kWsShared;
                        else oint[u] = oint[u] && mine;
                    }
                }
                const unsigned om0 = __ballot_sync(0xffffffffu, oint[0]), om1 = __ballot_sync(0xffffffffu, oint[1]);
                const unsigned lm0 = __ballot_sync(0xffffffffu, oleaf[0]), lm1 = __ballot_sync(0xffffffffu, oleaf[1]);
                const unsigned am0 = __ballot_sync(0xffffffffu, acc[0]), am1 = __ballot_sync(0xffffffffu, acc[1]);
                // (the ballots also order the lanes' reads of the stack before the pushes)
                const int no0 = __popc(om0), no1 = __popc(om1);
                if (sp + no0 + no1 > stack_cap) {
                    overflow = true;
                    break;
                }
                const int nl0 = __popc(lm0), na0 = __popc(am0);
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    if (oint[u]) {
                        const int q = sp + (u ? no0 + __popc(om1 & lt) : __popc(om0 & lt));
                        stk[q] = (uint32_t)nbd[u].z;
                        stn[q] = (uint8_t)push[u];
                    }
                    if (oleaf[u]) {
                        leaves[ln + (u ? nl0 + __popc(lm1 & lt) : __popc(lm0 & lt))] = make_int2(nbd[u].x, nbd[u].y);
                        if (list_stats) hsh += mix64(2ull * (unsigned)v[u] + 2ull);
                    }
                    if (acc[u]) {
                        float* q = ctile + cn + (u ? na0 + __popc(am1 & lt) : __popc(am0 & lt));
                        q[0] = src[u].x;
                        q[CAP] = src[u].y;
                        q[2 * CAP] = src[u].z;
                        q[3 * CAP] = src[u].w;
                        if (QUADW) {
                            const float* q6 = nt.quad + 6 * (int64_t)v[u];
#pragma unroll
                            for (int i = 0; i < 6; i++) cp_async4(q + (4 + i) * CAP, q6 + i);
                        }
                        if (list_stats) hsh += mix64(2ull * (unsigned)v[u] + 1ull);
                    }
                }
                sp += no0 + no1;
                ln += nl0 + __popc(lm1);
                const int nacc = na0 + __popc(am1);
                cn += nacc;
                Lc += nacc;
                if (LEARNED) {
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        bool band = false;
                        if (acc[u] && nbd[u].y >= 2) {
                            const float sz = pow2_down(Lf, nbd[u].w & 255, fast_side);
                            band = sz * sz >= a.band2 * band_e2[u];
                        }
                        if (LEARNED == 1) {
                            band_append(band, v[u], g);
                            continue;
                        }
                        const unsigned bm = __ballot_sync(0xffffffffu, band);
                        if (!bm) continue;
                        if (band) pend[qn + __popc(bm & lt)] = (uint32_t)v[u];
                        qn += __popc(bm);
                        __syncwarp();
                        if (qn >= 32) {
                            learned_rows(*mlp, pend, 32, rows, nt, rc, uf, Lf, 1.0f / Lf, xc, a.eps, 0.f, a.G, corr, lane);
                            nevals += 32;
                            // the cells past the first 32 to the front (read all, then write)
                            const uint32_t t32 = lane < qn - 32 ? pend[32 + lane] : 0u;
                            __syncwarp();
                            if (lane < qn - 32) pend[lane] = t32;
                            qn -= 32;
                            __syncwarp();
                        }
                    }
                }
                __syncwarp();
                if (cn >= kTile) {
                    close_cells(0);
                    if (!alive) break;
                }
                while (ln >= 32 && alive) list_leaves(32);
                if (!alive) break;
            }
            if (alive && !overflow && ln > 0) list_leaves(ln);
            if (!alive) break;
            if (overflow) {
                if (lane == 0) atomicOr(&a.info->err, kErrStack);
                cp_async_wait_all();  // copies into the dropped tile
                __syncwarp();
                cn = bn = 0;
                close_bodies(kWsLast | kWsAbort);
                continue;
            }
            if (cn > 0) close_cells(0);
            if (!alive) break;
            if (LEARNED == 2) {
                if (qn > 0) {
                    learned_rows(*mlp, pend, qn, rows, nt, rc, uf, Lf, 1.0f / Lf, xc, a.eps, 0.f, a.G, corr, lane);
                    nevals += qn;
                }
#pragma unroll
                for (int kk = 0; kk < 3; kk++)
#pragma unroll
                    for (int o = 16; o; o >>= 1) corr[kk] += __shfl_xor_sync(0xffffffffu, corr[kk], o);
                if (lane == 0 && a.mlp_evals) atomicAdd(a.mlp_evals, (unsigned long long)nevals);
            }
            close_bodies(kWsLast);
            if (list_stats) {
#pragma unroll
                for (int o = 16; o; o >>= 1) hsh += __shfl_xor_sync(0xffffffffu, hsh, o);
            }
            if (lane == 0) {
                const int gc = gend - gfirst;
                atomicAdd(&a.info->interactions, (unsigned long long)gc * (unsigned long long)(Lc + Lb));
                atomicAdd(&a.info->cells, (unsigned long long)gc * (unsigned long long)Lc);
                atomicAdd(&a.info->bodies, (unsigned long long)gc * (unsigned long long)Lb);
                if (parts > 1) {  // (zeroed before the launch)
                    if (a.ncell) atomicAdd(&a.ncell[g], Lc);
                    if (a.nbody) atomicAdd(&a.nbody[g], Lb);
                    if (a.hash) atomicAdd(&a.hash[g], hsh);
                } else {
                    if (a.ncell) a.ncell[g] = Lc;
                    if (a.nbody) a.nbody[g] = Lb;
                    if (a.hash) a.hash[g] = hsh;
                }
            }
            __syncwarp();
        }
        cp_async_wait_all();  // (a warp that gave up may still have copies in flight)
        return;
    }

    // ---------------------------------------------------------------- consumer
    for (int k = 0;;) {
        bool ok = mbar_wait(&t.full[k % kWsSlots], (k / kWsSlots) & 1);
        if (ok) {
            const WsHdr* h = t.hdr(t.seq[k % kWsSlots]);
            if (h->flags & kWsDone) return;
            const int gfirst = h->gfirst, ng = h->gend - h->gfirst;
            const double gx = h->ref[0], gy = h->ref[1], gz = h->ref[2];
            const int g = h->group, part = a.part_log2 ? h->part : -1;
            // positions of every body slot (slots past the group repeat its
            // first body; their sums are dropped)
            const int slots = ng <= 32 ? 32 : (ng <= 64 ? 64 : nb);
            __syncwarp();
            for (int i = lane; i < slots; i += 32) {
                const float4 q = a.body[gfirst + (i < ng ? i : 0)];
                pos[i] = q.x;
                pos[nb + i] = q.y;
                pos[2 * nb + i] = q.z;
                pos[3 * nb + i] = (float)((double)q.x - gx);
                pos[4 * nb + i] = (float)((double)q.y - gy);
                pos[5 * nb + i] = (float)((double)q.z - gz);
            }
            __syncwarp();
#define TC_WS_GROUP(K, S) consume_group<K, S, TILE, PRECISE, POT, LEARNED>(t, k, pos, nb, part, gfirst, ng, a)
            if (ng <= 16) k = TC_WS_GROUP(1, 2);
            else if (ng <= 32) k = TC_WS_GROUP(1, 1);
            else if (!ws_quad(TILE) && ng <= 40) k = TC_WS_GROUP(5, 4);
            else if (ng <= 48) k = TC_WS_GROUP(3, 2);
            else if (ws_quad(TILE) || ng <= 64) k = TC_WS_GROUP(2, 1);
            else if (ng <= 96) k = TC_WS_GROUP(3, 1);
            else k = TC_WS_GROUP(4, 1);
#undef TC_WS_GROUP
            ok = k >= 0;
            if (ok && part >= 0) add_parts<POT, LEARNED>(g, gfirst, ng, a);
        }
        if (!ok) {
            if (lane == 0) atomicOr(&a.info->err, kErrWorkLoop);
            return;
        }
    }
}

// a launch's block and shared memory
struct WsShape {
    int threads, nb, stack;
    size_t smem;
};
constexpr size_t kWsSmemMax = 227 * 1024;

__host__ __forceinline__ WsShape ws_shape(const WalkConfig& c, int tile, bool rows)
{
    WsShape w;
    const int teams = c.warps < 1 ? 1 : (c.warps > kWsMaxPairs ? kWsMaxPairs : c.warps);
    w.threads = teams * 64;
    w.nb = ws_body_slots(c.gmax);
    // a stack that leaves no room for the ring is cut (an entry stands for
    // all the children of a cell, so it holds several times as many nodes
    // as one entry per node)
    w.stack = (c.stack + 3) & ~3;
    const auto bytes = [&](int stack) {
        return ws_team_bytes(tile, stack, w.nb, rows) * teams + (rows ? mlp_frag_bytes() : 0);
    };
    while (w.stack > 64 && bytes(w.stack) > kWsSmemMax) w.stack -= 16;
    // the network and its rows take the room of a second block on the SM; a
    // stack no larger than the default gives way down to 512 opened cells,
    // which hold more than that many nodes did (a step takes 8 of them where
    // it took 32 nodes, and adds as many children to each).  A stack that was
    // asked for is given, if need be with one block on the SM
    if (rows && c.stack <= kDefaultStack && bytes(512) <= kWsSmemMax / 2 - 1024)
        while (w.stack > 512 && bytes(w.stack) > kWsSmemMax / 2 - 1024) w.stack -= 16;
    w.smem = bytes(w.stack);
    return w;
}

template <int TILE, bool PRECISE, bool POT, int LEARNED>
cudaError_t prepare_ws_t(const WalkConfig& c, int num_sms, int* grid, size_t* smem_out)
{
    const WsShape w = ws_shape(c, TILE, LEARNED == 2);
    const int threads = w.threads;
    const size_t smem = w.smem;
    auto kern = k_walk_ws<TILE, PRECISE, POT, LEARNED>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (c.blocks_per_sm > 0 && c.blocks_per_sm < per_sm) per_sm = c.blocks_per_sm;
    *grid = num_sms * per_sm;
    *smem_out = smem;
    return cudaSuccess;
}

template <int TILE, bool PRECISE, bool POT, int LEARNED>
cudaError_t launch_ws_t(const WalkArgs& a, const WalkConfig& c, int grid, size_t smem, cudaStream_t s)
{
    // the split walk has no list export, training pairs, size classes or
    // quadrupole terms of large groups (those run on k_walk)
    if (a.list_cells || a.pair_body || a.gseg) return cudaErrorInvalidValue;
    if (LEARNED == 1 && (!a.band || !a.band_n || !a.grec)) return cudaErrorInvalidValue;
    if (LEARNED == 2 && !a.mlp) return cudaErrorInvalidValue;
    if (a.part_log2 && (!a.part_sum || !a.part_done)) return cudaErrorInvalidValue;
    const WsShape w = ws_shape(c, TILE, LEARNED == 2);
    k_walk_ws<TILE, PRECISE, POT, LEARNED><<<grid, w.threads, smem, s>>>(a, w.stack, w.nb);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

}  // namespace tc
