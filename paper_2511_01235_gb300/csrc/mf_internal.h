// Internal structures of the GB300 max-flow library (not part of the ABI).
//
// Device layout of one residual graph (Sec. 5.1 Bi-CSR), structure of arrays:
//   off[n+1]   reserved start of each row (rows are never moved in place)
//   deg[n]     used slots of the row: base slots (sorted by dst) then inserted slots
//   bdeg[n]    number of sorted base slots (binary search range)
//   dst[S]     head v of slot (u, v)
//   cf[S]      residual capacity c_f(u, v)
//   cap[S]     capacity c(u, v) (0 for a reverse-only slot)
//   rev[S]     index of the slot (v, u)
//   pcap[S]    c(u, v) + c(v, u): with the pair-sum invariant (Sec. 3.1
//              Theorem 3.3) c_f(v, u) = pcap - c_f(u, v), so the backward BFS
//              reads the reverse residual without a gather through rev.
//   h[n]       heights (int32), e[n] excesses (int64)
#pragma once
#include <stddef.h>
#include <stdint.h>
#include <cuda_runtime.h>

#define MF_BLOCK 512          // threads per CTA of the persistent kernel
#define MF_WARPS (MF_BLOCK / 32)
#define MF_SMALL_DEG 8        // discharge: rows up to this many slots get one thread
#define MF_SMALL_DEG_SPARSE 4 // ... on a graph of at most MF_SPARSE_DEG merged directed edges per vertex
#define MF_SPARSE_DEG 8
#define MF_HUB_DEG 512        // discharge: rows above this many slots get a 4-warp group (or a whole CTA)
#define MF_NBIN 4             // discharge row kinds: thread, warp, 4-warp group, CTA
#define MF_GROUP_WARPS 4      // warps of a group; a group keeps rows up to a quarter of the snapshot
#define MF_BFS_HUB 128        // BFS: rows above this many slots enter the frontier as work items
#define MF_BFS_CHUNK 128      // BFS: slots per work item
#define MF_DEFAULT_ROUNDS 2   // adaptive discharge rounds: the minimum per iteration
#define MF_MAX_ROUNDS 1024    // adaptive rounds: upper bound per iteration
#define MF_TRACE 256          // hook timeline entries kept per launch
#define MF_BU_ALPHA 14        // BFS default: go bottom-up when the frontier's slots exceed the unexplored slots / alpha
#define MF_BU_BETA 24         // BFS default: back to top-down when the frontier holds fewer than n / beta vertices
#define MF_WARP_STAGE 512     // discharge: largest row a warp keeps on chip (per-warp slice of the snapshot)
#define MF_ROW_ALIGN 4        // rows start on multiples of this many slots (16-byte loads of slot fields)
#define MF_BU_SCAN 256        // bottom-up BFS: slots of a row its warp scans before deferring the rest
#define MF_BU_CHUNK 256       // bottom-up BFS: slots per deferred work item (one warp, 8 per lane)
#define MF_NEAR_SINK 8        // near iterations: the sink's row holds at most 1/8 of the vertices
#define MF_LARGE_SLOTS 65536  // near iterations and short rounds: graphs of at least this many reserved slots
#define MF_NEAR_STEP 2        // near iterations: a cut that settled less than half asks for 2^2 times the excess next
#define MF_NEAR_SUB 8192      // walks: residuals up to this are taken with one atomic subtraction
#define MF_Q_BFS 8192         // on-chip queue of a CTA: labelled vertices of one BFS phase,
#define MF_Q_LONG 2048        // ... those with long rows,
#define MF_Q_WL 4096          // ... worklist entries of one phase (vertex; bin and place)
#define MF_Q_INTS (MF_Q_BFS + MF_Q_LONG + 2 * MF_Q_WL)
#define MF_CLUSTER 8          // CTAs per thread-block cluster; the first cluster is the squad
#define MF_SQUAD_CAP 4096     // queue entries of a squad CTA
#define MF_SQUAD_LONG 1024    // long-row vertices a squad CTA keeps on chip
#define MF_SQUAD_INTS (6 * MF_SQUAD_CAP + MF_SQUAD_LONG)   // two queues of vertex, row start, row length; long rows
#define MF_SQUAD_LEVEL 256    // BFS levels of at most this many vertices per squad CTA ...
#define MF_SQUAD_SLOTS 2048   // ... and slots run in the squad
#define MF_SQUAD_ACTIVE 256   // so do discharge rounds of at most this many vertices per squad CTA
#define MF_HANDOVER 2         // copies of the state that the first CTA hands over at a barrier (MfCtrl)
#define MF_DEEP 16            // a BFS of this many levels is deep: no level turns bottom-up, and a small graph runs short rounds
#define MF_SHORT_ROW 512      // rounds of one cycle per vertex: the longest row

// Solve-kernel status (ctrl->status)
#define MF_ST_RUNNING 0
#define MF_ST_CONVERGED 1
#define MF_ST_CAP 2           // iteration or time cap
#define MF_ST_ERROR 3         // MfReport.err holds the error

// MfReport.err values
#define MF_E_NONE 0
#define MF_E_INVALID 1        // batch entry out of range / negative capacity
#define MF_E_OVERFLOW 2       // insertion needs more slack than a row has
#define MF_E_WAIT 3           // a grid barrier wait gave up
#define MF_E_INTERNAL 4
#define MF_E_TOO_LARGE 5      // a batch would leave a pair with c(u,v) + c(v,u) > INT32_MAX

// Kernel modes (bit mask)
#define MF_M_STATIC_INIT 1    // c_f = cap, e = 0, h = 0, saturate the source (Alg. 1)
#define MF_M_APPLY 2          // the batch part of Alg. 5
#define MF_M_SOLVE 4          // the push-relabel loop
#define MF_M_BFS_ONLY 8       // one backward BFS, then stop
#define MF_M_NO_DEFICIT_ROOTS 16  // BFS roots: the sink only (flow extraction runs)
#define MF_M_SKIP_SOURCE_SAT 32   // apply without saturating the source again
#define MF_M_SAT_SINK 64          // static init also saturates every edge into the sink (Sec. 5.2.2 static push-pull)
#define MF_M_NO_SRC_SAT 128       // static init leaves the source edges alone (the pull-only static solve)
#define MF_M_CUT 256              // after the batch: record the sides of the last cut, saturate the edges S -> T
#define MF_M_SCHED 1024            // after the batch: the network picks the schedule (MfParams.net)
#define MF_M_NO_VALUE 512         // skip the value phase (the side-limited push / pull parts)

struct alignas(128) MfLine {
    unsigned int w[32];
};

// Every word that many CTAs update with atomics during a phase sits on a line
// of its own in a counter set.  Phase k (the stretch up to grid barrier k of a
// launch) uses set k mod 3; behind the barrier every CTA reads the whole set
// and works out by itself what comes next, so no CTA has to decide for the
// others and publish the decision.  Set (k + 2) mod 3 was last read behind
// barrier k - 1, before any CTA arrived at barrier k, so the first CTA can
// clear it during phase k + 1, and nobody touches it before phase k + 2.
enum MfLineId {
    L_BFS = 0,            // regular frontier entries appended in this phase
    L_HUB,                // frontier work items
    L_DEFER,              // bottom-up chunks deferred to the level's second pass
    L_HEAD0,              // dynamic work heads
    L_HEAD1,
    L_HEAD2,
    L_HEAD3,
    L_WL,                 // [MF_NBIN] worklist entries per bin (built by the BFS)
    L_AUX = L_WL + MF_NBIN,       // [MF_NBIN] next-round worklist entries per bin
    L_FIX = L_AUX + MF_NBIN,      // [2] remove-invalid lists (warp / CTA)
    L_ACT = L_FIX + 2,    // active vertices (only when the worklist is a pass of its own)
    L_FEAT,               // learned schedule: updates touching s, touching t, deleting
    L_FCAP,               // learned schedule: 64-bit sum of the batch's capacities; w[2]: 1 + the action it picked
    L_MISC,               // w[0] new pairs, w[1] a row without room, w[2] dedup entries, w[3] error (MF_E_*)
    L_LAB,                // 64-bit: labelled vertices << 32 | their slots
    L_TOTAL,              // 64-bit: used slots of the whole graph (summed by the BFS roots pass)
    L_EXC,                // 64-bit: excess of the vertices labelled in this phase (near iterations)
    L_DEM,                // 64-bit: what the roots can take (BFS roots pass, near iterations)
    L_TIME,               // 64-bit: the first CTA's clock when it arrived at the barrier
    MF_LINES
};

struct MfSet {
    MfLine l[MF_LINES];
};

#define MF_PACK 16384     // host batches of up to this many updates are packed into pinned memory
#define MF_MAX_CTAS 1024  // CTAs whose finish times and slots are traced (a grid is far smaller)

// What the phases read, the same in every CTA (kept in shared memory).
struct MfDesc {
    int status;
    int level;
    int lvl_lo, lvl_hi;           // this level's regular frontier in border[]
    int hub_lo, hub_hi;           // ... work items in bitem[]
    int app_bfs, app_hub;         // where this phase's entries of the two lists start
    int wl_app[MF_NBIN];          // where this phase's worklist entries start
    int bfs_done;
    int bu_mode;                  // the coming BFS level runs bottom-up
    int bu_split;                 // the bottom-up level just scanned deferred long rows: their pass follows
    int defer_n;                  // work items of that pass
    int bfs_squad;                // the coming top-down level is small: the squad runs it, and the next small ones, alone
    int dis_short;                // the coming discharge round has short rows only: one cycle per vertex
    int dis_squad;                // ... and few of them: the squad runs it, and the next small ones, alone
    int dis_stamp;                // a short round queues behind stamps (mf_round_stamps)
    int need_total;               // the coming BFS roots pass sums the used slots (first BFS of a launch)
    int wl_sel;                   // which worklist buffer the current round reads
    int wl_n[MF_NBIN];
    int ins_n, hused_n;           // batch: new pairs, dedup table entries
    int round;                    // discharge round within the iteration
    int dis_more;                 // another discharge round follows
    int resolve;                  // the picked action re-solves from zero flow
    int near;                     // this launch may cut its global relabels short and walk the excess down
    int cut;                      // ... and this iteration's was cut short
    int fix_n[2];                 // vertices for remove-invalid-edges (warp list, CTA list); grows over the rounds
    int qstamp, fstamp;           // dedupe stamps (never reset: they only grow across launches)
};

// The rest of what every CTA carries from barrier to barrier.  Decisions take
// the first CTA's clock, read from the counter set, so all CTAs decide alike.
struct MfState {
    unsigned long long t_phase;   // this CTA's clock behind the last barrier (statistics only)
    unsigned long long t_now;     // the first CTA's clock when it arrived at the last barrier
    unsigned long long t_start, t_bfs0, t_dis0;   // t_now at the first barrier, at this iteration's BFS and discharge
    unsigned long long ns_bfs, ns_dis, ns_fix, ns_wl, ns_apply;
    long long vis_slots;          // slots of the vertices labelled so far in this BFS
    long long lvl_slots, lvl_cnt; // slots and number of the vertices labelled by the level that is running
    long long used_slots;         // used slots of the graph (0: not summed yet)
    long long sup, dem, dem_prev; // this BFS: excess labelled, what the roots can take (and the BFS before)
    int cut_prev, cut_shift;      // the iteration before was cut short; how much more excess a cut asks for
    int full_run, pad0;           // complete relabels in a row that left excess to move (near)
    long long iters, bfs_levels, rounds_total, barriers, active_first, active_total;
    int err;                      // MF_E_*
    int trace_n;
};

// Whether round `round` of an iteration's discharge, if it is a short one, has to
// queue behind stamps, by the round before.  Without stamps a short round needs a
// list whose vertices all have excess.  A BFS and an unstamped short round leave
// such a list.  A round of several cycles does not: u sends its excess, a
// neighbour pushes to u and queues it, and a later cycle of u's sends that too;
// nor do the walks, where u may take along what another walk has left there.  In
// an unstamped round such a vertex, listed with e = 0, could be queued by a
// receiver and then by itself, and the round after would hold it twice: two
// owners that both take the same residual, below zero.
#ifdef __CUDACC__
__host__ __device__
#endif
inline int mf_round_stamps(int round, int last_short, int last_stamped)
{
    return round > 0 && (last_stamped || !last_short) ? 1 : 0;
}

// Work counters.  Each CTA keeps its own in shared memory and adds them to the
// control block once, at the end of the launch.
enum MfStat {
    ST_PUSHES = 0, ST_RELABELS, ST_STEEP,
    ST_SLOTS_BFS, ST_VERTS_BFS,
    ST_HSCAN_BFS,         // heights read by the passes over all vertices of bottom-up levels
    ST_LAB_BFS,           // vertices labelled by all BFS levels
    ST_SLOTS_DIS, ST_CYCLES_DIS,
    ST_SLOTS_FIX, ST_VERTS_FIX,
    ST_N_APPLY,
    ST_SLOTS_APPLY,       // slots read by the batch phases (slot search, source row)
    ST_CLAMPS_APPLY,      // slots whose residual went negative and was sent back
    ST_NS_CTA, ST_NS_WARP, ST_NS_THREAD,  // discharge time by row kind, summed over workers
    MF_STATS
};

// What the host reads of a launch.  The kernel's first CTA writes it straight to
// the context's pinned memory (MfParams.rep), so nothing has to be copied back.
struct MfReport {
    int err;              // MF_E_*
    int status;           // MF_ST_*
    int action, pad;      // the action the network picked (MF_M_SCHED)
    long long iters, value;
    long long bfs_levels, active_total, active_first;
    long long cut_slots, used_slots;      // slots of the vertices the last BFS labelled; of all
    long long stat[MF_STATS];     // MfStat, summed over the CTAs at the end of a launch
    unsigned long long ns_bfs, ns_dis, ns_fix, ns_wl, ns_apply;
    long long rounds_total;
    unsigned long long t_entry;   // kernel entry (first CTA), last barrier
    unsigned long long t_exit;
    long long barriers;
    int trace_n;
    int trace_hook[MF_TRACE];
    unsigned long long trace_t[MF_TRACE];
    // work per traced phase: slots scanned so far (BFS + discharge + remove-invalid, cumulative), and
    // BFS: bit 30 = the level ran bottom-up, bits 20..29 = work items, bits 0..19 = vertices labelled;
    // discharge round: bits 20..29 = CTA-bin (hub) vertices, bits 0..19 = vertices in the round's lists
    long long trace_slots[MF_TRACE];
    int trace_info[MF_TRACE];
    // when the CTAs finished the phase that a barrier closes (ns after the previous barrier):
    // the last one and the mean, per traced barrier
    unsigned trace_fin_max[MF_TRACE], trace_fin_mean[MF_TRACE];
};

struct MfCtrl {
    MfReport rep;         // of launches without pinned memory to report to
    int qstamp, fstamp;   // carried over from launch to launch
    long long value;
    long long stat[MF_STATS];
    MfLine bar;           // w[0]: arrivals in this launch (the first CTA leaves it at zero);
                          // w[1]: a CTA of the first cluster gave up at a barrier
    MfSet set[3];
    // the first CTA's state for the others, after its squad ran phases alone.
    // Barrier k uses copy k mod MF_HANDOVER: a CTA may still be reading copy k
    // when the first one, which only needs its own cluster to get there, writes
    // the copy of barrier k + 1; it writes copy k again only for barrier k + 2,
    // after every CTA has arrived at k + 1 and so has read it.
    MfDesc jd[MF_HANDOVER];
    MfState js[MF_HANDOVER];
    // per phase (mod 3) and CTA: finish time, slots scanned
    unsigned fin[3][MF_MAX_CTAS], scanned[3][MF_MAX_CTAS];
};
// The part the host clears after a launch that ended in a barrier that gave up.
#define MF_CTRL_SYNC_BYTES (sizeof(MfLine) + sizeof(MfSet) * 3)

// A schedule (action) of the learned scheduler; the table is fixed.
struct MfAction {
    int32_t mode;      // 0: incremental (Alg. 5), 1: apply the batch, then re-solve from zero flow (Alg. 1)
    int32_t rounds;    // discharge rounds per global relabel (0: adaptive)
    int32_t cycles;    // KERNEL_CYCLES (0: the average-degree heuristic of Sec. 6.1)
    int32_t cycle_div; // > 0: rows of d slots get max(cycles, d / cycle_div) cycles
    int32_t fix;       // 1: remove-invalid-edges (Alg. 3) after each iteration's discharge
};
// Index 0 is the library's default schedule, 5 the paper's fixed one (one
// round, KERNEL_CYCLES = average degree, Alg. 3 after every discharge) and 18
// the paper's static re-solve.
#define MF_ACTIONS                                                                                      \
    {0, 0, 0, 0, 0},   {0, 0, 0, 256, 0}, {0, 0, 4, 0, 0},   {0, 0, 64, 0, 0},  {0, 0, 64, 256, 0},     \
    {0, 1, 0, 0, 1},   {0, 1, 16, 0, 0},  {0, 1, 64, 0, 0},  {0, 4, 4, 0, 0},   {0, 4, 16, 0, 0},       \
    {0, 4, 64, 0, 0},  {0, 16, 4, 0, 0},  {0, 16, 16, 0, 0}, {0, 16, 64, 0, 0}, {0, 64, 16, 0, 0},      \
    {0, 64, 64, 0, 0}, {1, 0, 0, 0, 0},   {1, 0, 64, 0, 0},  {1, 1, 0, 0, 1},   {1, 16, 16, 0, 0},

// The network that picks one, and what it looks at besides the batch.
#define MF_FEATURES 16
#define MF_NET_HIDDEN 256
struct MfNet {
    const float *p;           // its parameters (mlp.cu's layout); nullptr: none
    int32_t hidden, n_out;
    long long m;              // merged directed edges
    float mean_cap;
    float host[6];            // features 9..14
};

struct MfGraph {
    int32_t n;
    int64_t slot_cap;
    int32_t *off, *deg, *bdeg;
    int32_t *dst, *cf, *cap, *rev, *pcap;
    int32_t *h;
    long long *e;
};

struct MfScratch {
    int32_t *border;          // [n] BFS order (level segments)
    int2 *bitem;              // [n + slot_cap / MF_BFS_CHUNK + 64] frontier work items (first slot, length)
    int2 *bdefer;             // [n + slot_cap / MF_BFS_CHUNK + 64] bottom-up deferred chunks (vertex, first slot);
                              // nullptr: bottom-up threads scan whole rows themselves
    int32_t *wl[2][MF_NBIN];  // [n] worklists (two buffers for discharge rounds) per row kind: thread, warp,
                              // 4-warp group, CTA
    int32_t *vmark;           // [n] round stamp of the last time a vertex was queued
    int32_t *fixmark;         // [n] iteration stamp of the last time a vertex was listed for Alg. 3
    int32_t *par;             // [n] slot (v, parent) of the vertices labelled by a near BFS (nullptr: never near)
    long long *dem;           // [n] what a root can still take in a near iteration
    int32_t *fixl[2];         // [n] vertices relabelled this iteration: rows <= MF_HUB_DEG, rows above
    // batch apply
    int64_t batch_cap;
    int32_t hash_bits;
    unsigned long long *hkey; // [1 << hash_bits] directed-pair dedup
    int32_t *hval;
    unsigned long long *pkey; // [1 << hash_bits] new-pair dedup
    int32_t *bslot;           // [batch_cap] slot of each update (-2: superseded or ignored)
    int32_t *ins_list;        // [batch_cap] new-pair table positions
    int32_t *hused;           // [batch_cap] dedup table positions in use
    int32_t *ins_need;        // [n]
    int32_t *bu;              // [3 * batch_cap] a host batch: tails, heads, capacities one after the other
};

struct MfParams {
    MfGraph g;
    MfScratch sc;
    MfCtrl *ctrl;
    MfReport *rep;            // where the launch reports (pinned host memory, or ctrl->rep)
    int32_t *cf;              // residual array of this run (g.cf, or a copy for extraction)
    int32_t *h;
    long long *e;
    int32_t sink, source;
    int32_t mode;
    int32_t kernel_cycles;
    int32_t rounds;           // discharge rounds between two global relabels (1 = the paper's O1 worklist);
                              // 0: adaptive (at least MF_DEFAULT_ROUNDS, more while discharging has taken
                              // less than half the time of this iteration's BFS)
    int32_t small_deg;        // discharge: rows up to this many slots get one thread
    int32_t hub_deg;          // discharge / remove-invalid: rows above this many slots get a group (or a CTA)
    int32_t group_deg;        // discharge: rows above this many slots get a whole CTA (<= hub_deg: no groups)
    int32_t bfs_hub;          // BFS: rows above this many slots enter the frontier as work items
    int32_t bu_alpha;         // BFS direction switch (0: top-down only), see MF_BU_ALPHA
    int32_t bu_beta;
    int32_t fix_steep;
    int32_t data_driven;
    int32_t pull;             // 0: push excess toward t and deficits;
                              // 1: pull for deficits from s and excess (Sec. 5.2.2)
    int32_t side_root;        // -1: every deficient (push) / overflowing (pull) vertex is a root;
                              // else only side[v] == side_root
    uint8_t *side;            // [n] sides of the last cut (1: reaches t or a deficit, 0: not); written by MF_M_CUT
    int32_t test_skip_cta;    // >= 0: that CTA never arrives at the first barrier (tests the bounded waits)
    int32_t requeue;          // discharge rounds: a vertex still active after its cycles joins the next round
    int32_t cycle_div;        // > 0: a row of d slots gets max(kernel_cycles, d / cycle_div) cycles
    int32_t tail_slots;       // BFS: a top-down level whose frontier holds at most this many slots (and
                              // vertices) runs in the squad, without grid barriers; 0: none does; -1: MF_SQUAD_SLOTS per CTA
    int32_t stage_slots;      // dynamic shared memory of the launch in ints: the discharge's on-chip row snapshot
                              // (a CTA keeps rows up to this many slots; 0: none)
    int32_t allow_near;       // 0: no near iterations (the caller has set a cap on iterations, which counts complete relabels)
    long long max_iters;
    unsigned long long time_limit_ns;
    unsigned long long wait_limit_ns;
    int32_t avg_cycles;       // KERNEL_CYCLES by the average degree
    MfNet net;                // MF_M_SCHED
    // batch
    int64_t bcount;
    const int32_t *bu, *bv, *bc;
};

// Host-built Bi-CSR (graph_build.cpp)
struct MfHostGraph {
    int32_t n = 0;
    int64_t m_merged = 0;     // directed edges with capacity > 0 or explicitly given (merged)
    int64_t slot_cap = 0, slots = 0;
    int32_t *off = nullptr, *deg = nullptr, *bdeg = nullptr;
    int32_t *dst = nullptr, *cap = nullptr, *rev = nullptr, *pcap = nullptr, *cf = nullptr;
    void release();
};

// Build from COO.  Returns MAXFLOW_* status.
int mf_build_host(int32_t n, int64_t m, const int32_t *src, const int32_t *dst, const int32_t *cap,
                  float slack_factor, int32_t slack_min, MfHostGraph &out);

// Reserved slots of a row with d used ones: slack of max(smin, ceil(d * factor)), rounded up
// so that the next row starts on a 16-byte boundary.
#ifdef __CUDACC__
__host__ __device__
#endif
inline long long mf_row_size(long long d, float factor, int smin)
{
    const double want = (double)d * (double)factor;
    long long sl = (long long)want;
    if ((double)sl < want) ++sl;
    if (sl < smin) sl = smin;
    if (sl > (1 << 24)) sl = 1 << 24;
    return (d + sl + MF_ROW_ALIGN - 1) / MF_ROW_ALIGN * MF_ROW_ALIGN;
}

// build.cu: the same layout, made on the device.  mf_build_sizes uploads, checks and
// sorts the edges and sizes the rows; the caller then allocates the slot arrays
// (slots entries each) and mf_build_fill writes them.  Both wait for the stream.
#define MF_BUILD_MIN 16384            // edge lists shorter than this are built on the host
#define MF_BUILD_SCRATCH (4ll << 30)  // ... and those that would need more scratch memory than this
struct MfBuild {
    void *scratch = nullptr;          // device, mf_build_scratch(n, m) bytes
    int32_t *deg = nullptr, *bdeg = nullptr;   // device, [n]
    long long pairs = 0;              // used slots
    long long slots = 0;              // reserved slots
    long long merged = 0;             // directed edges with a capacity
    double cap_sum = 0;
    int bits = 0, launches = 0;
};
size_t mf_build_scratch(int n, long long m);
int mf_build_sizes(MfBuild &b, int n, long long m, const int32_t *src, const int32_t *dst, const int32_t *cap,
                   float slack_factor, int slack_min, void *stream);
int mf_build_fill(MfBuild &b, int n, long long m, const MfGraph &g, void *stream);

// solver.cu
// Exclusive scan of a[0 .. n) in place, its total into a[n]; mf_rebuild_scratch(n) values.  Three kernels.
int mf_scan64(long long *a, long long n, void *stream);
// cluster: 1, or MF_CLUSTER (then grid, and gsize, are multiples of it)
int mf_launch(const MfParams &p, int grid, int cluster, void *stream);
int mf_launch_multi(const MfParams *plist_dev, int count, int gsize, int grid, unsigned *gstate, unsigned *head,
                    unsigned long long wait_ns, int *abort, int cluster, void *stream, int stage_bytes);
int mf_stage_bytes(int device, int *bytes);
int mf_max_coresident_blocks(int device, int *per_sm, int *num_sms, int dyn_bytes);
int mf_max_clustered_blocks(int dyn_bytes, int *blocks);   // with clusters of MF_CLUSTER; 0 where there are none
int mf_launch_aux(int which, const MfParams &p, void *stream, long long *dev_out, const void *extra);

#define MF_AUX_SET_CF_RESET 1     // cf = cap on all used slots
#define MF_AUX_SET_FLOW 2         // extra = {count, u, v, f} device arrays; validate into dev_out[0] or apply
#define MF_AUX_EXCESS 3           // e = sum(cf - cap) per row
#define MF_AUX_CHECK 4            // dev_out[0..5]
#define MF_AUX_ANSWER 5           // extra = MfAnswer: the source side and the capacity of the cut
#define MF_AUX_REVERSE_CF 7       // extra = int32_t* out: out[x] = cf[rev[x]]
#define MF_AUX_CLEAR_SCRATCH 8    // reset hash tables and ins_need
#define MF_AUX_DUMP 9             // extra = int32_t* rowid per slot (u of each slot index)
#define MF_AUX_NEGATE_E 10        // e = -e
#define MF_AUX_PCAP 11            // pcap = cap + cap[rev] on every used slot (after a restore)

struct MfAnswer {
    uint8_t *side;        // [n] 1: source side (device-accessible; nullptr: not wanted)
    long long *cut;       // capacity of the cut (device-accessible; nullptr: not wanted)
    long long *acc;       // device, [2], zero before and after
    int from_sink;        // sum over the sink side's rows instead of the source side's
};

// device-side rebuild (rows grow, flows and excesses stay in place); noff holds
// n + 1 row starts followed by the scan's tile totals: mf_rebuild_scratch(n) int64
#define MF_SCAN_TILE 4096
inline long long mf_scan_tiles(long long n) { return n / MF_SCAN_TILE + 1; }
inline long long mf_rebuild_scratch(long long n) { return n + 1 + mf_scan_tiles(n) + 1; }
int mf_rebuild_capacity(const MfParams &p, void *stream, float slack_factor, int slack_min, long long *noff);
// the copy: rows of more than MF_MOVE_PIECE new slots are moved in pieces of that
// size, listed in items[] (mf_move_items(slot_cap) entries) with their count in *nitems
#define MF_MOVE_PIECE 1024
inline long long mf_move_items(long long slot_cap) { return 2 * (slot_cap / MF_MOVE_PIECE) + 64; }
int mf_rebuild_move(const MfParams &p, void *stream, const long long *noff, int32_t *off, int32_t *dst, int32_t *cf,
                    int32_t *cap, int32_t *rev, int32_t *pcap, long long slot_cap, int2 *items, unsigned *nitems);

// scheduler features of a batch (16 floats)
struct MfFeatIn {
    const int32_t *bu, *bv, *bc;
    long long count;
    int32_t n, s, t;
    long long m;
    float mean_cap;
    float host[6];            // features 9..14, known on the host
};
int mf_features(const MfFeatIn &f, float *out_dev, void *stream);

int mf_set_flow_items(const MfParams &p, void *stream, long long *dev_bad, long long count, const int32_t *du,
                      const int32_t *dv, const int32_t *df, int apply);
