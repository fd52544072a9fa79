// tc_internal.cuh -- device-side data layout and launchers of the treecode
// library (CUDA, sm_103a).  Internal to libtc.so; the public C ABI is
// include/tc.h.
//
// A context holds a batch of S >= 1 independent systems whose bodies are
// concatenated (system s owns bodies [off_s, off_s+1) in the caller's order
// and the same positions in Morton order).  Every system has its own root
// cube and its own tree; the trees form one forest in one node table, and
// one walk launch serves the groups of every system.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace tc {

constexpr int kMaxLevel = 21;      // 21 bits per axis, 63-bit Morton keys
constexpr int kLeafMaxLimit = 4096;
constexpr int kBboxChunk = 4096;   // bodies per bounding-box block (never across systems) ...
constexpr int kBboxChunkSmall = 1024;  // ... of up to 2^19 bodies

// error bits of the device error word
enum : int32_t {
    kErrNonFinite = 1,    // NaN/Inf position or mass
    kErrStack = 2,        // walk stack overflow
    kErrCapacity = 4,     // the node table outgrew its allocation
    kErrWorkLoop = 8,     // a bounded wait gave up
    kErrBand = 16,        // the learned walk's band-cell record outgrew its buffer
    kErrFmmPool = 32,     // the FMM's unresolved-source pool outgrew its allocation (regrown, rerun)
    kErrFmmSlab = 64,     // one cell's unresolved-source list outgrew its slab (regrown, rerun)
    kErrFmmStack = 128,   // the FMM's refinement stack overflowed
    kErrSortRun = 256,    // a rebuild inside a step met a run of equal top key bits too long to complete
};

// Per-system root cube (written by the bounding-box kernels).
struct SysParams {
    double c0[3];      // root cube corner
    double L;          // root cube side (power of two)
    double h;          // grid step L / 2^21
    long long qoff[3]; // c0 / h (integers): q = floor(x / h) - qoff
    int32_t qexp;      // 1 / h = 2^qexp
    float Lf;          // L as float (exact)
    float uf;          // h / 2 as float (exact): unit of the integer centres
    int32_t first;     // bodies [first, end)
    int32_t end;
    int32_t bb[6];     // bounding box as order-preserving ints: lo xyz, hi xyz
    float msys;        // total mass (for the learned correction's features)
    int32_t done;      // bounding-box chunks of the system that are done
};

// Per-context scalars kept in device memory (written by kernels, read by
// kernels and, at synchronisation points, by the host).
// a stream, and whether a kernel launched on it may come while the kernel
// before it still runs (tc_pdl.cuh)
struct ChainStream {
    cudaStream_t s;
    bool chain;
    ChainStream(cudaStream_t stream, bool c = false) : s(stream), chain(c) {}
};

struct Info {
    int32_t err;       // error bits
    int32_t depth;     // deepest level of the forest
    int64_t M;         // nodes in the node table
    int64_t G;         // groups in the group table
    int64_t count;     // nodes that the last build counted (M once they are in the table)
    uint32_t work[4];  // walk work-queue counters, one per launch of a force phase
    unsigned long long interactions;  // body-source interactions of the last walk
    unsigned long long cells;         // body-cell interactions (group size x accepted cells)
    unsigned long long bodies;        // body-body interactions (group size x direct-list bodies)
    double diag[8];    // KE, PE, P[3], L[3]
};

// Node record as the walk reads it (breadth-first order, index v; the roots
// of systems 0..S-1 are nodes 0..S-1).
//   a: centre of mass minus cube centre (float), mass (float)
//   b: first body, body count, first child, level | nchild << 8
//   c: cube centre in units of u = h/2 of its system (exact integers), system
//   d: centre of mass in absolute coordinates (float), mass (plain mode)
struct NodeTables {
    float4* a;
    int4* b;
    int4* c;
    float4* d;
    float* quad;     // 6 per node, second moments about the COM (FP32)
    uint4* feat;     // 2 per node: the learned correction's cell-only features (eps/s, log2 count,
                     // M / M_sys, 6 moment ratios), normalised, as BF16 pairs (words 2..7 of a row)
    double* mass64;  // the bottom-up reduction's results in FP64
    double* com64;   // 3 per node
    float4* dsum;    // 2 per node: the bottom-up sums {m, m x} as float pairs, hi parts then lo parts
    int32_t* parent; // -1 for a root
    uint8_t* fam;    // 1: the node follows a sibling (its predecessor in the table)
    uint32_t* pend;  // children of an internal cell that are done (bottom-up in one launch)
};

// scratch of the radix sort
struct SortBufs {
    uint64_t* keys_alt;
    uint32_t* vals_alt;
    uint32_t* ghist;                 // passes x 256 digit counts
    unsigned long long* status;      // look-back words, passes x tiles x 256
    uint32_t* tiles;                 // tile counters, one per pass
    int32_t* err;                    // device error word (bounded look-back)
};
constexpr int kSortMaxPasses = 10;   // 63 key bits + up to 16 system bits

// ---------------------------------------------------------------- launchers
// all launches go on `s`; none synchronises.  Every launcher adds the number
// of kernels it launched to a process-wide counter (count_launches).
void count_launches(int k);
long long launches_total();
// streaming multiprocessors of the current device (cached per device; a
// host query, allowed while a stream is being captured)
int sm_count();
// records the reason of a failure outside any context (tc_last_error(NULL))
void set_thread_error(const char* msg);

// One 8-bit digit of the sort's order: the bits of (system, key >> low_bit)
// taken as one number, the system above the kb key bits.
struct SortDigit {
    int kshift;   // right shift of the key (past its bits for the topmost digits)
    int sys;      // 1: the digit holds bits of the system
    int sleft;    // left shift of the system (where key bits share the digit), else
    int sright;   // right shift
    __host__ __device__ uint32_t of(uint64_t key, uint32_t system) const
    {
        const uint32_t k = kshift < 64 ? (uint32_t)(key >> kshift) : 0u;
        return (sys ? (k | ((system << sleft) >> sright)) : k) & 255u;
    }
};
// The passes of a sort by the key bits [low_bit, nbits) and then sys_bits
// bits of the system: as few digits as hold them together.
struct SortPlan {
    int npass, low_bit, kb, sys_bits;
    __host__ __device__ static SortPlan make(int nbits, int low_bit, int sys_bits)
    {
        const int kb = nbits - low_bit;
        return SortPlan{(kb + sys_bits + 7) / 8, low_bit, kb, sys_bits};
    }
    __host__ __device__ SortDigit digit(int p) const
    {
        SortDigit d;
        d.kshift = 8 * p < kb ? low_bit + 8 * p : 64;
        d.sys = sys_bits > 0 && 8 * p + 8 > kb;
        d.sleft = d.sys && 8 * p < kb ? kb - 8 * p : 0;
        d.sright = d.sys && 8 * p > kb ? 8 * p - kb : 0;
        return d;
    }
};

// The passes of a plan from (ka, va) to (kb, vb) and back, n >= 2 items; the
// result lies in (ka, va) after an even number of passes.  b.ghist holds the
// digit counts of every pass; b.tiles and radix_status_words(n, npass) words
// of b.status are zero.
void launch_sort_passes(uint64_t* ka, uint32_t* va, uint64_t* kb, uint32_t* vb, int64_t n, const SortPlan& plan,
                        const uint32_t* sys_of, const SortBufs& b, ChainStream s);
int64_t radix_status_words(int64_t n, int npass);
int64_t radix_status_words(int64_t n);  // enough for any sort of up to n items
// After passes over bits [low_bit, 63): every run of items with equal top
// bits (and system; sys_of null: one system) in (key, val) order, which is
// the full sort's order as the values are distinct (the bodies' indices),
// and body[] in it.  A run longer than run_max (at most kSortRunMax) raises
// kErrSortRun and kErrCapacity instead.
constexpr int64_t kSortRunMax = 16384;
constexpr int64_t kSortRunMaxSynced = 1024;  // a synchronised build re-sorts every digit past this
constexpr int kSortMarginLevels = 2;  // levels below the last synchronised depth a step's sort orders
void launch_sort_runs(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout, int64_t n,
                      int low_bit, const uint32_t* sys_of, const float* pos, const float* mass, float4* body,
                      int64_t run_max, int32_t* err, ChainStream s);
// Up to kBlockSortMax items: the passes, the completion (low_bit > 0) and the
// bodies in one launch of one block; no digit counts or scratch needed.
constexpr int64_t kBlockSortMax = 4096;
void launch_sort_block(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout, int64_t n,
                       const SortPlan& plan, const uint32_t* sys_of, const float* pos, const float* mass, float4* body,
                       ChainStream s);
// A whole sort of (key, val) by bits [0, nbits) of key, in place.
void radix_sort_u64(uint64_t* keys, uint32_t* vals, int64_t n, int nbits, SortBufs& b, cudaStream_t s);
// self-test of the radix pass's bounded look-back (see tc_sort.cu)
cudaError_t sort_wait_selftest(uint64_t* keys, uint32_t* vals, uint64_t* kout, uint32_t* vout,
                               unsigned long long* status, uint32_t* counter, uint32_t* hist, int32_t* err,
                               cudaStream_t s);
int64_t sort_selftest_items();

// build pieces
void launch_sys_ids(const int64_t* offsets, int nsys, int64_t n, uint32_t* sys_of, SysParams* sysp,
                    ChainStream s);
// start of a build: nzero 16-byte words of scratch zeroed, info->depth (and,
// reset_err, info->err) too, the bounding boxes emptied
void launch_build_init(uint4* zero, int64_t nzero, SysParams* sysp, int nsys, Info* info, bool reset_err,
                       ChainStream s);
// bounding boxes, and each system's root cube once its last chunk is done;
// chunks: (system, start, end, chunks of the system).  Batches of more than
// kCubeSystems systems form the cubes in a launch of their own, a thread each:
// by one thread of each block they are microseconds of FP64 latency that tens
// of thousands of blocks queue for (builds of 512 x 1000 / 2048 x 16 / 8192 x
// 16 / 65536 x 16 bodies: 258 / 124 / 189 / 643 us so, 260 / 113 / 159 / 455
// with the launch)
constexpr int kCubeSystems = 512;
void launch_bbox(const float* pos, const int4* chunks, int nchunks, SysParams* sysp, int nsys, int32_t* err,
                 ChainStream s);
// Morton keys, indices and (ghist not null) the digit counts of the plan's passes
void launch_keys(const float* pos, const float* mass, int64_t n, const uint32_t* sys_of, const SysParams* sysp,
                 uint64_t* keys, uint32_t* idx, const SortPlan& plan, uint32_t* ghist, int32_t* err, ChainStream s);
void launch_gather(const float* pos, const float* mass, const uint32_t* perm, int64_t n,
                   float4* body, ChainStream s);
// The levels of the cubes that start at each sorted body (delta < l <= top),
// their number per level and block of bodies, and the exclusive scan of those
// (level by level, so the nodes' breadth-first places); zeroes gref_at;
// info->count = nodes, kErrCapacity where cap_m >= 0 and it exceeds that.  cnt:
// level_counts_size(n) words; scan: build_scan_words(n) words, zeroed.
int64_t level_counts_size(int64_t n);
int64_t build_scan_words(int64_t n);
void launch_node_levels(const uint64_t* keys, const uint32_t* sys_of, int64_t n, int leaf_max, int8_t* w,
                        int8_t* delta, int8_t* top, int32_t* gref_at, uint32_t* cnt, unsigned long long* scan,
                        int64_t cap_m, Info* info, ChainStream s);
// the node records at those places (counts and children follow with the
// moments), lstart[0..22], the first node of each level, and info->M; nothing
// (so M stays that of the table) after kErrCapacity
void launch_emit_nodes(const uint64_t* keys, const int8_t* delta, const int8_t* top, const uint32_t* sys_of, int64_t n,
                       const uint32_t* offs, Info* info, uint32_t* lstart, NodeTables nt, ChainStream s);
// counts, children and moments: the leaves, then the internal cells, in the
// same launch for up to kClimbBodies bodies, else level by level from
// depth - 1 (depth < 0: the depth is known on the device only; with
// depth_hint >= 0, the depth of an earlier build, levels depth_hint + 2 .. 0
// get a launch each and any deeper ones one block, else all 21 levels get a
// launch); each level reads its range on the device.  Also each system's mass.
constexpr int64_t kClimbBodies = 1 << 19;  // (both ways timed: tc_build.cu, "moments")
void launch_moments(const float4* body, const uint64_t* keys, const int8_t* delta, int64_t n, int nsys,
                    int64_t cap_m, int depth, int depth_hint, const uint32_t* level_start, SysParams* sysp, const Info* info, NodeTables nt,
                    bool quad, ChainStream s);
// the body groups: gfirst[0..G], gref[0..G), info->G
void launch_groups(int64_t cap_m, Info* info, const NodeTables nt, int gmax, int64_t n, int32_t* gref_at,
                   unsigned long long* scan, int32_t* gfirst, int32_t* gref, int32_t* part_done, ChainStream s);
// the groups by the walk's layout of their bodies (kGroupClasses of them),
// the largest first, stable: order[0, G); seg[0..3] = the ranges of groups of
// more than 64, 33 to 64 and up to 32 bodies in it; scratch holds
// group_order_scratch() ints
constexpr int kGroupClasses = 7;
size_t group_order_scratch();
void launch_group_order(const int32_t* gfirst, const Info* info, int32_t* order, int32_t* seg, int32_t* scratch,
                        ChainStream s);
// walk + force
struct WalkArgs {
    const float4* body;        // Morton order (x, y, z, m)
    const uint32_t* perm;      // Morton position -> original index
    const uint32_t* sys_of;    // body position -> system
    const SysParams* sysp;     // per-system root cube
    NodeTables nt;
    const int32_t* gfirst;     // G + 1 entries
    const int32_t* gref;       // G
    Info* info;
    float* acc;                // n x 3, original order
    float* pot;                // n, original order (nullable)
    int32_t* ncell;            // per group (nullable)
    int32_t* nbody;
    unsigned long long* hash;
    float theta2, eps2, G;
    float inv_eps;             // 1/eps for the potential self term
    // learned correction (null model: off)
    const void* mlp;           // device MlpDev
    float band2;               // accepted cells with s^2 >= band2 d^2 get a correction
    float eps;
    // training pairs (null: off): accepted cells with count >= 2 in the band
    // are emitted with probability pair_prob as (a body of the group, cell)
    int32_t* pair_body;
    int32_t* pair_node;
    unsigned long long* pair_count;
    int64_t pair_cap;
    float pair_prob;
    unsigned long long pair_seed;
    unsigned long long* mlp_evals;   // corrections evaluated (nullable)
    // list export (null: off): walk group list_group only, write its accepted
    // cells and opened leaves (walk order, at most list_cap each) and their
    // counts to list_n[0..1]; no forces or totals are written
    int32_t* list_cells;
    int32_t* list_leaves;
    int64_t list_cap;
    int64_t* list_n;
    int32_t list_group;
    // the order in which groups are walked (null: 0..G-1); gseg (null: all of
    // it): walk glist[gseg[0], gseg[1]) only
    const int32_t* glist;
    const int32_t* gseg;
    int work_slot;  // this launch's work-queue counter, info->work[work_slot]
    // split walk: 2^part_log2 parts per group; a part's compensated sums in
    // part_sum[(kPartPlanes part + 2 component (+ 1: compensation)) part_stride + body]
    // (the learned correction in planes 6 to 8),
    // the parts done so far in part_done[group] (zero before and after)
    int part_log2;
    float* part_sum;
    int32_t* part_done;
    int64_t part_stride;
    // learned correction evaluated after the walk (split walk): the band
    // cells of every group recorded as (node, group) pairs in chunks of
    // kBandChunk entries taken from *band_n (unused tails hold node -1), at
    // most band_cap entries; grec[2 g], grec[2 g + 1] the group's record for
    // the rows: {box centre in its reference cube's frame, h/2} and
    // {reference cube centre (integer units of h/2, as int bits), root side}
    int2* band;
    unsigned long long* band_n;
    int64_t band_cap;
    float4* grec;
};
constexpr int kDefaultStack = 1024;  // tc_config.stack of a new context
constexpr int kBandChunk = 256;
constexpr int kPartPlanes = 9;
struct WalkConfig {
    int gmax;         // 32, 64 or 128
    int warps;        // warps per block
    int precise;      // cell-relative sources + compensated accumulation
    int want_pot;
    int verify;
    int blocks_per_sm;
    int stack;        // walk stack entries per warp
    int tile;         // list tile entries: 64, 128 or 256
    int learned;      // 1: learned far-field correction (precise mode, no potential)
    int quadw;        // 1: accepted cells add their quadrupole term (precise mode)
    int classes;      // 1: one launch per group size class (the smaller beside the largest); 0: one launch
    int split;        // 1: monopole walks on producer/consumer warps (k_walk_ws)
    int part_log2;    // split: each group is walked in 2^part_log2 parts
    int record;       // split, learned: the band cells are recorded for a launch after the walk
};
// host-side preparation of the walk kernel's launch (attributes, occupancy);
// call before a stream capture
cudaError_t prepare_walk(const WalkConfig& c, int num_sms, int* grid, size_t* smem);
// teams of the split walk that fit an SM
int walk_ws_teams(const WalkConfig& c);
// reset_totals: zero the work-queue counters and (outside list export) the
// interaction totals first -- the first launch of a force phase; the later
// launches of a phase split over size classes count on counters of their own
// (a.work_slot) zeroed with the first
cudaError_t launch_walk(const WalkArgs& a, const WalkConfig& c, int grid, size_t smem, cudaStream_t s,
                        bool reset_totals = true);

// the walk's force loop alone (tc_force_probe.cu); returns the interactions
// the launch sums
double launch_force_probe(int blocks, int reps, float* out, cudaStream_t s);

// learned far-field correction (tc_mlp.cu)
size_t mlp_dev_size();
size_t mlp_frag_size();  // the inference part at the front of a device model
size_t mlp_train_smem();
// loss and gradient on B rows: per-warp partial gradients in part (at least
// mlp_train_part_floats(max_blocks) floats), added in warp order into grad
// (the packed gradient, overwritten) and the loss added to *loss
int64_t mlp_train_part_floats(int blocks);
int mlp_train_blocks(int B, int max_blocks);  // blocks of a mini-batch of B rows
cudaError_t launch_mlp_train(const float* X, const float* T, const float* W, const int32_t* idx, int B,
                             const void* model, float* grad, float* loss, float* part, int max_blocks, cudaStream_t s);
// one pass over n rows in mini-batches of `batch`, a cooperative launch; sched
// holds three floats per step: the learning rate and Adam's bias corrections
// (mlp_adam_corrections).  The model's copies for inference and W1's k-major
// one are not kept up (launch_mlp_pack does).
cudaError_t launch_mlp_epoch(const float* X, const float* T, const float* W, const int32_t* idx, int n, int batch,
                             int max_blocks, void* model, float* params, float* mom, float* vel, const float* sched,
                             float* part, float* loss, uint32_t* bar, int32_t* err, cudaStream_t s);
void mlp_adam_corrections(int t, float* c1, float* c2);
void launch_mlp_pack(const float* params, const float* maps, void* model, cudaStream_t s);
void launch_mlp_infer(const float* X, int64_t n, const void* model, float* Y, cudaStream_t s);
// the learned correction evaluated after a split walk: every recorded band
// cell's row at its group's centre through the network on the tensor cores,
// F label summed per group into gcorr (G x 3, zeroed by the caller); then
// each body's acceleration gains its group's sum
void launch_band_eval(const WalkArgs& a, const void* model, float* gcorr, unsigned long long* evals,
                      cudaStream_t s);
void launch_band_apply(const Info* info, int64_t cap_g, const int32_t* gfirst, const uint32_t* perm,
                       const float* gcorr, float* acc, cudaStream_t s);
// the learned correction's per-cell features of every node for softening
// eps under the model (run before a learned walk)
void launch_node_features(const Info* info, int64_t cap_m, const SysParams* sysp, NodeTables nt, float eps,
                          const void* model, cudaStream_t s);
// the emitted (body, node) pairs sorted by (body, node): the walk emits them
// in whatever order its warps finish, the training wants one order
void launch_pair_order(int32_t* pb, int32_t* pv, int64_t np, uint64_t* keys, uint32_t* vals, SortBufs& b,
                       cudaStream_t s);
void launch_pair_labels(const int32_t* pb, const int32_t* pv, int64_t np, const float4* body, const uint32_t* sys_of,
                        const SysParams* sysp, NodeTables nt, float eps, float G, float* feat, float* lab,
                        float* fac, cudaStream_t s);
// training data on the device: the model's maps (and the factor-weight scale
// n / sum F^2) from FP64 sums of x, x^2, t^2 (and F^2) over the pairs (part:
// kMlpSumBlocks x kMlpSums doubles), normalised rows and scaled targets, loss
// weights (mode 0: check the given ones, mode 1: F^2 n / sum F^2; *bad = 1
// for a non-finite or negative weight), fresh parameters, and a seeded
// permutation of [0, n)
constexpr int kMlpSums = 13 + 13 + 3 + 1;
constexpr int kMlpSumBlocks = 608;
void launch_mlp_maps(const float* X, const float* T, const float* F, int64_t n, double* part, float* maps,
                     float* wscale, cudaStream_t s);
void launch_mlp_rows(const float* X, const float* T, int64_t n, const float* maps, float* rows, float* tout,
                     cudaStream_t s);
void launch_mlp_weights(float* w, int64_t n, int mode, const float* wscale, int32_t* bad, cudaStream_t s);
void launch_mlp_init(float* params, uint64_t seed, cudaStream_t s);
void launch_mlp_shuffle(int64_t n, uint64_t key, int32_t* idx, cudaStream_t s);

// FP32 throughput probe (8 independent FMA chains per thread, scalar or
// paired f32x2 instructions)
void launch_fp32_probe(bool paired, int blocks, int iters, float* out, cudaStream_t s);

// dynamics and diagnostics
void launch_kick_drift(float* pos, float* vel, const float* acc, int64_t n, float hkick, float dt,
                       const Info* info, cudaStream_t s);
void launch_kick(float* vel, const float* acc, int64_t n, float hkick, const Info* info, cudaStream_t s);
// n bodies' accelerations and potentials (either may be null) to memory of this
// device, unless the error word is set
void launch_copy_good(float* acc, const float* from_acc, float* pot, const float* from_pot, int64_t n,
                      const Info* info, cudaStream_t s);
void launch_diag(const float* pos, const float* vel, const float* mass, const float* pot,
                 int64_t n, Info* info, cudaStream_t s);
// source slices of a direct sum that fill the device; launch_direct's scratch
// holds 4 ns doubles for each of two or more, one needs none
int direct_slices(int64_t n, int64_t ns);
void launch_direct(const float* pos, const float* mass, const uint32_t* sys_of, const SysParams* sysp,
                   const int64_t* idx, int64_t ns, int slices, float eps2, float G, double* part, double* acc,
                   double* pot, cudaStream_t s);

// fast multipole method (tc_fmm.cu): the radii, then the walk of every cell.
// Scratch: loc (cap_m x fmm_loc_width() floats), near_off, near_cnt and pend
// (cap_m; the last two zero before the launch), a pool of pool_cap entries, a
// slab of slab_cap entries for each of fmm_slab_warps() warps, ctr (8
// counters: pool fill, tickets, pool need, slab need, M2L pairs, P2P pairs
// and their two hashes; zero before the launch); rec: per node its M2L and
// P2P pairs as target and their hashes.
struct FmmLaunch {
    const float4* body;
    const uint32_t* perm;
    const SysParams* sysp;
    NodeTables nt;
    const Info* info;
    int32_t* err;
    int64_t cap_m;
    uint32_t* pend;
    float* loc;
    int32_t* pool;
    int64_t pool_cap;
    int32_t* slab;
    int64_t slab_cap;
    int64_t* near_off;
    int32_t* near_cnt;
    unsigned long long* ctr;
    unsigned long long* rec;  // 4 per node (M2L pairs, P2P pairs, their hashes), 32-byte aligned
    double* rad;              // per node: r_X (FP64)
    int4* fnode;              // per node, 3 entries: the walk's record with r_X in FP32
    int records;              // pair-set hashes and per-node records (else counts only)
    float* acc;
    float theta, eps, G;
};
int64_t fmm_slab_warps();
int fmm_loc_width();
cudaError_t launch_fmm(const FmmLaunch& p, cudaStream_t s);

}  // namespace tc
