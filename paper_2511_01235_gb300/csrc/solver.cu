// Device code of the GB300 dynamic max-flow library (sm_103a).
//
// One cooperative, persistent kernel runs a whole solve: the optional static
// initialisation (Alg. 1) or batch repair (Alg. 5),
// then the loop { backward BFS (Alg. 4 / Alg. 6), direction-optimising, which
// also builds the active-vertex worklist (Sec. 5.2.1 O1) ; stop if empty ;
// push-relabel discharge (Alg. 2) in one or more rounds ; remove-invalid-edges
// (Alg. 3, when enabled: off by default) }, then the value formula of Alg. 5.
// Phases are separated by a grid barrier instead of kernel launches, so the
// termination test never leaves the device and a small update costs one
// launch.  Every wait at a barrier in memory (grid, group) is bounded in time: on
// expiry the CTA records MF_E_WAIT and returns, and the host reports
// MAXFLOW_ERR_INTERNAL.  A cluster's barrier is the hardware's and has no limit
// of its own; it ends because each CTA of the cluster reaches it after bounded
// work and bounded waits, or has left the kernel, which counts as having arrived.
//
// A solve is bound by its chain of phases, each a few dependent trips to L2
// (302 clocks; DRAM 824) and a barrier, and not by bytes: most of what follows
// shortens that chain.  Every CTA takes the decisions between phases itself
// from the phase's counters (advance); a phase's results are queued on chip and
// appended with one reservation per CTA (flush_queue); small levels and rounds
// stay in one cluster (squad); rounds on short rows are one cycle per vertex;
// and on graphs with a short sink row a relabel ends early and the excess walks
// down its tree (near iterations).
//
// Readings of the paper used here (the same as the CPU oracle's):
//   - BFS roots are the sink and every vertex other than s, t with e < 0
//     (Alg. 6), in the static solve too, and h(s) = n always;
//   - termination is tested right after a complete BFS;
//   - a relabel with no residual neighbour, or above n, sets h = n;
//   - ties between equal-height neighbours go to the lowest slot index;
//   - the value is the sum of e(v) over v != s with h(v) < n.
// Excess of the sink and the source is accumulated per CTA in shared memory
// and added once per phase (every vertex may push into the sink, and one
// global atomic per push would serialise on that word).
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/maxflow.h"
#include "mf_internal.h"

namespace {

constexpr unsigned long long kEmpty = ~0ull;

// The CTAs that run one solve: the whole grid for mf_solve_kernel, one group
// of the grid for mf_multi_kernel.  Every phase distributes its work over
// vb() in [0, vn()), and the grid barrier waits for vn() CTAs.
__shared__ int g_vb, g_vn;

// The parameters of the running solve, in shared memory: the phases read them
// often.  P and sh (below) are variables of the file and not arguments, so that
// the compiler knows that they are shared memory: through a pointer every
// access is a generic one and every addition to a counter a choice between two
// kinds of atomics, which had made a single phase 20 to 80 KB of code, more than
// the instruction cache holds beside the rest of an iteration.
__shared__ MfParams P;

// Dynamic shared memory of the persistent kernels: the on-chip snapshot of a
// row during its discharge (P.stage_slots ints).
extern __shared__ __align__(16) int mf_stage[];
__device__ __forceinline__ int vb() { return g_vb; }
__device__ __forceinline__ int vn() { return g_vn; }

// Row kind of a vertex with d used slots: 0 thread, 1 warp, 2 four-warp group, 3 CTA.
__device__ __forceinline__ int row_bin(int d)
{
    return d <= P.small_deg ? 0 : (d <= P.hub_deg ? 1 : (d <= P.group_deg ? 2 : 3));
}

// First work index of this thread in a grid-stride loop (stride vn() *
// blockDim.x) that spreads a short list over the whole grid: consecutive
// indices go to different CTAs, so a batch of a few thousand updates keeps
// every SM's memory pipeline busy instead of crowding onto the first CTAs.
// spread_warp keeps 32 consecutive indices in one warp (warp-uniform loops).
__device__ __forceinline__ long long spread_thread() { return (long long)threadIdx.x * vn() + vb(); }
__device__ __forceinline__ long long spread_warp(int nctas)
{
    return ((long long)(threadIdx.x >> 5) * nctas + vb()) * 32 + (threadIdx.x & 31);
}

__device__ __forceinline__ int ldg_cg(const int *p) { return __ldcg(p); }
__device__ __forceinline__ long long ldg_cg(const long long *p) { return __ldcg(p); }

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ long long atomic_add_ll(long long *p, long long v)
{
    return (long long)atomicAdd((unsigned long long *)p, (unsigned long long)v);
}

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w < v ? w : v;
    }
    return v;
}

__device__ __forceinline__ long long warp_sum_ll(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ unsigned hash_slot(unsigned long long key, int bits)
{
    return (unsigned)((key * 0x9E3779B97F4A7C15ull) >> (64 - bits));
}

// Claim k work items from a shared head; returns the first index (>= cnt when
// the work is exhausted).  The head is read first so that idle warps do not
// queue atomics on it once the work is gone.  Call with the whole warp.
__device__ __forceinline__ int warp_grab(unsigned *head, int cnt, unsigned k)
{
    int b = 0;
    if ((threadIdx.x & 31) == 0) {
        unsigned cur = *(volatile unsigned *)head;
        b = (int)(cur >= (unsigned)cnt ? cur : atomicAdd(head, k));
    }
    return __shfl_sync(0xffffffffu, b, 0);
}

// Items [0, cnt) dealt out to nw workers without a rush on one counter: the
// worker of rank w takes chunk [w*k, w*k + k) first, with no atomic; the
// chunks past nw*k are grabbed k at a time from the head (which starts at 0).
// A grab-only scheme sends, when every warp of the grid starts a short phase at
// once, one atomic per warp to the same word; the L2 serialises them, and a
// warp that comes back for more work waits behind all of them.  `first` is the
// caller's flag, true before the first call.  Called by the whole warp.
__device__ __forceinline__ int warp_deal(unsigned *head, int cnt, unsigned k, int w, int nw, bool &first)
{
    if (first) {
        first = false;
        const long long b = (long long)w * k;
        if (b < cnt) return (int)b;
    }
    const long long base = (long long)nw * k;
    if (base >= cnt) return cnt;
    long long b = 0;
    if ((threadIdx.x & 31) == 0) {
        const unsigned cur = *(volatile unsigned *)head;
        b = base + (base + cur >= cnt ? cur : atomicAdd(head, k));
    }
    b = __shfl_sync(0xffffffffu, b, 0);
    return b < cnt ? (int)b : cnt;
}

// Rank of this warp for warp_deal among the warps of nctas CTAs (all of the
// grid, or CTA 0 alone): consecutive ranks sit in different CTAs, so a few
// items spread over many SMs, and the ranks are rotated by `skip`, so that the
// warps that took the first `skip` items of an earlier list come last in this
// one.
__device__ __forceinline__ int warp_rank(int nctas, int skip)
{
    const int nw = nctas * (int)(blockDim.x >> 5);
    const int r = (int)(threadIdx.x >> 5) * nctas + vb();
    const int s = skip < nw ? skip : skip % nw;
    return r >= s ? r - s : r - s + nw;
}

// What one CTA of the squad tells the others after a phase.
struct alignas(16) SquadSum {
    int cnt;              // entries of its next queue
    unsigned slots;       // BFS: their slots (with those of long rows)
    int labelled;         // BFS: vertices labelled
    int flag;             // SQ_*
    long long exc;        // near BFS: excess labelled
    long long pad;
};
enum { SQ_SPILL = 1,      // something went onto the grid's lists: long rows, a full queue
       SQ_STOP = 2,       // (first CTA) the grid should take over: out of time
       SQ_OVER = 4 };     // (first CTA) the discharge has had its share of the time

// What a CTA keeps in shared memory: its accumulators, its copy of the launch's
// state (the same in every CTA between two barriers), and work space of phases.
struct Sh {
    long long sink_e, src_e;          // excess of the sink and the source, added to memory before every barrier
    long long value;                  // this CTA's share of the value
    unsigned ft_s, ft_t, ft_del;      // learned schedule: this CTA's updates touching s, touching t, deleting
    long long ft_cap;                 // ... and their capacities' sum
    float x[MF_FEATURES], h1[MF_NET_HIDDEN], h2[MF_NET_HIDDEN], y[64];   // the network's layers
    int action;                       // what it picked (-1: nothing yet)
    long long stat[MF_STATS];         // work counters, added to memory at the end of the launch
    unsigned long long lab;           // BFS: vertices labelled this phase << 32 | their slots
    unsigned long long exc, dem;      // near BFS: excess labelled, what the roots can take, this phase
    unsigned long long red[MF_WARPS];
    long long wsum[MF_WARPS];
    int wcnt[MF_WARPS];
    int bcast_i;
    long long tb_e[MF_BLOCK / (32 * MF_GROUP_WARPS)];   // per team (CTA: [0]; 4-warp groups: [g]) broadcasts
    int tb_h[MF_BLOCK / (32 * MF_GROUP_WARPS)];
    int tb_i[MF_BLOCK / (32 * MF_GROUP_WARPS)];
    int ok;
    unsigned phase;                   // barriers passed in this launch
    MfSet *cs;                        // the counter set of the running phase
    int tr_hook, tr_info;             // of the last barrier, for the trace
    // of the parameters, for advance(): BFS direction switch, worklist wanted, longest level of the squad (slots; 0: none)
    int k_alpha, k_beta, k_wl, k_squad;
    // the squad: its CTAs, this one's rank, whether it is the whole solve; what
    // each of its CTAs found in a phase (two sets, written by their owners into
    // every CTA); this CTA's entries of the next queue
    int csize, crank, one_cluster;
    unsigned arrivals;                // arrivals at the grid barrier so far
    SquadSum sq[2][MF_CLUSTER];
    int so_cnt, so_long, so_flag, so_go, so_par;
    // on-chip queue of a phase (place_labelled, place_active): entries taken, per kind
    int q_bfs, q_long, q_wn, q_wl[MF_NBIN];
    int q_base[MF_NBIN + 1];
    int4 cnt[MF_LINES];               // the counters of the phase that just ended
    MfDesc d;
    MfState hs;
};

__shared__ Sh sh;

enum Hook {
    H_START = 0,          // unused (a launch starts without a barrier); keeps the trace ids
    H_NONE,
    H_APPLY_VALID,
    H_APPLY_LOCATED,
    H_APPLY_CHECKED,      // unused (the room check runs inside the locate phase); keeps the trace ids
    H_APPLY_DELTA,
    H_ITER,
    H_BFS_START,
    H_BFS_NEXT,
    H_WL,
    H_DIS,
    H_FINAL,
    H_BU_SPLIT,
    H_JOIN,               // unused (a squad's run ends like the phase it ended with); keeps the trace ids
    H_EXPANDED,           // unused (long rows are split into work items as they are queued); keeps the trace ids
};

// x += v, x in shared memory, as two 32-bit additions with the carry between
// them.  A 64-bit atomic on shared memory is a loop of compare and swap, which
// the threads of a CTA that add to one word run one after another, dozens of
// clocks each; 32-bit additions to one word are combined in hardware (512
// threads: 42 clocks).
template <class T>
__device__ __forceinline__ void add_shared(T &x, long long v)
{
    static_assert(sizeof(T) == 8, "a 64-bit word");
    unsigned *w = reinterpret_cast<unsigned *>(&x);
    const unsigned lo = (unsigned)v;
    const unsigned old = atomicAdd(w, lo);
    const unsigned hi = (unsigned)((unsigned long long)v >> 32) + (old + lo < old ? 1u : 0u);
    if (hi) atomicAdd(w + 1, hi);
}

__device__ __forceinline__ void add_stat(MfStat i, long long v)
{
    if (v) add_shared(sh.stat[i], v);
}

__device__ __forceinline__ int cnt32(int line) { return sh.cnt[line].x; }
__device__ __forceinline__ unsigned long long cnt64(int line)
{
    return (unsigned long long)(unsigned)sh.cnt[line].x | ((unsigned long long)(unsigned)sh.cnt[line].y << 32);
}

// A top-down level of cnt vertices with fr slots, none of them long, that the
// squad runs alone (squad_bfs).
__device__ __forceinline__ bool squad_level(long long cnt, long long fr)
{
    return sh.k_squad > 0 && cnt <= MF_SQUAD_LEVEL * sh.csize && fr <= sh.k_squad;
}

// Direction of a BFS level that follows a top-down one (Beamer's test): bottom-up
// once the frontier's slots (fr) exceed 1/alpha of the unexplored ones.  Not in a
// deep BFS, whose frontiers are short: near its end the unexplored slots get few
// too, and a bottom-up level still visits every vertex (256 x 256 grid, window
// updates 4.9 -> 4.7 ms; 64 batched instances 12.0 -> 11.3).  The squad asks the
// same: what it leaves for a bottom-up level has to become one.
__device__ __forceinline__ bool turns_bottom_up(int alpha, int level, long long fr, long long unexplored)
{
    return alpha > 0 && level < MF_DEEP && fr * alpha > unexplored;
}

// Adaptive rounds: whether this iteration's discharge may still take time beside
// its BFS: half of it with rounds of KERNEL_CYCLES cycles, all of it with short
// ones (grid 1024 window 15.5 -> 13.6 ms, 64 batched instances 14.6 -> 11.6 ms;
// twice the BFS's time 13.5 and 11.0, but a 512 grid's static solve 33 -> 36).
__device__ __forceinline__ bool rounds_left(const MfDesc &d, const MfState &st, unsigned long long t)
{
    return (d.dis_short ? 1 : 2) * (t - st.t_dis0) < st.t_dis0 - st.t_bfs0;
}

// How the coming discharge round (number d.round of its iteration) over the
// worklists in d runs.  Short: a push with the default schedule over rows of at
// most MF_SHORT_ROW slots gets one cycle per vertex (phase_discharge_short), and
// few vertices are left to the squad (squad_discharge).  On a small graph that
// takes a BFS of many levels: short rounds pay where many rounds follow; where
// two or three do, the whole KERNEL_CYCLES in each settle more.  Behind a round
// of another kind it queues behind stamps, unless the squad runs it, which drops
// the entries without excess first (64 batched instances: 11.9 ms, and 17.5
// without short rounds there).
__device__ __forceinline__ void pick_round(MfDesc &d, int csize)
{
    d.dis_stamp = mf_round_stamps(d.round, d.dis_short, d.dis_stamp);
    d.dis_short = P.rounds == 0 && !P.pull && !P.fix_steep && P.data_driven && P.requeue &&
                          P.stage_slots >= MF_SQUAD_INTS && P.hub_deg <= MF_SHORT_ROW &&
                          (P.g.slot_cap >= MF_LARGE_SLOTS || d.level >= MF_DEEP) &&
                          d.wl_n[2] + d.wl_n[3] == 0
                      ? 1 : 0;
    d.dis_squad = d.dis_short && d.wl_n[0] + d.wl_n[1] <= MF_SQUAD_ACTIVE * csize ? 1 : 0;
}

// The termination test of the loop (Alg. 1 / Alg. 5: stop when no active
// vertex remains), taken right after a complete backward BFS.
__device__ __forceinline__ void decide_iteration(int active)
{
    MfDesc &d = sh.d;
    MfState &st = sh.hs;
    d.round = 0;
    d.fix_n[0] = d.fix_n[1] = 0;
    ++d.qstamp;
    ++d.fstamp;
    st.t_dis0 = st.t_now;
    for (int b = 0; b < MF_NBIN; ++b) d.wl_n[b] = d.wl_app[b];
    pick_round(d, sh.csize);
    if (d.near) d.dis_short = d.dis_squad = 0;        // a near iteration starts with the walks
    if (st.iters == 0) st.active_first = active;
    st.active_total += active;
    if (active == 0) {
        d.status = MF_ST_CONVERGED;
    } else if (st.iters >= P.max_iters || st.t_now - st.t_start > P.time_limit_ns) {
        d.status = MF_ST_CAP;
    } else {
        ++st.iters;
    }
}

// Whether the launch may run near iterations: a push solve with the default
// schedule, and a sink that can be reached from few vertices directly.  With a
// longer sink row (grids: every pixel has an edge to t) what the sink can take
// exceeds any excess, no relabel would be cut, and the bookkeeping would only
// cost.  Nor under the caller's own cap on iterations: those behind a cut relabel
// settle less, so a cap that sufficed would not.
__device__ __forceinline__ int near_allowed()
{
    if (!P.allow_near || P.sc.par == nullptr || !(P.mode & MF_M_SOLVE) || (P.mode & MF_M_NO_DEFICIT_ROOTS) || P.pull ||
        P.side_root >= 0 || P.rounds != 0 || P.fix_steep || !P.data_driven || P.g.slot_cap < MF_LARGE_SLOTS)
        return 0;
    return (long long)ldg_cg(P.g.deg + P.sink) * MF_NEAR_SINK <= (long long)P.g.n ? 1 : 0;
}

// ---- learned schedule ----
//
// The network is asked inside the launch that applies the batch: the phase that
// validates the batch sums what the features need, the last CTA runs the 16 ->
// H -> H -> n_out network beside the phase that locates the slots (which takes
// longer), and behind that phase's barrier every CTA sets its parameters to the
// picked action's.  As kernels of their own, features, network and the host's
// read of the choice cost 28 held-out updates of ER, R-MAT and grid graphs 35.7
// ms against 26.5 with the default schedule; here both take 21 ms.

__constant__ MfAction kActionTable[] = {MF_ACTIONS};

// The features of a batch (with updates touching s, touching t and deleting, and
// the sum of its capacities) on a graph of n vertices and m edges.
__device__ __forceinline__ void make_features(float *x, long long count, long long edges, int vertices, unsigned at_s,
                                              unsigned at_t, unsigned deleting, long long cap_sum, float mean_cap,
                                              const float *host)
{
    const float B = (float)count, m = (float)(edges > 0 ? edges : 1), n = (float)vertices;
    const float inv = count > 0 ? 1.f / B : 0.f;
    x[0] = log2f(1.f + B) / 20.f;
    x[1] = fminf(B / m, 1.f);
    x[2] = log2f(n) / 24.f;
    x[3] = log2f(1.f + m) / 28.f;
    x[4] = (m / n) / 16.f;
    x[5] = (float)at_s * inv;
    x[6] = (float)at_t * inv;
    x[7] = (float)deleting * inv;
    x[8] = count > 0 && mean_cap > 0.f ? fminf((float)cap_sum * inv / mean_cap, 4.f) / 4.f : 0.f;
    for (int k = 0; k < 6; ++k) x[9 + k] = host[k];
    x[15] = 1.f;
}

// One thread: the features of the launch's batch.
__device__ __noinline__ void batch_features()
{
    make_features(sh.x, P.bcount, P.net.m, P.g.n, (unsigned)sh.cnt[L_FEAT].x, (unsigned)sh.cnt[L_FEAT].y,
                  (unsigned)sh.cnt[L_FEAT].z, (long long)cnt64(L_FCAP), P.net.mean_cap, P.net.host);
}

// y = w x + b by one CTA (relu: not below zero), a warp per output with its lanes
// over the inputs, so that the weights come in whole lines.
__device__ __forceinline__ void net_layer(const float *__restrict__ w, const float *__restrict__ b, const float *x,
                                          int n_in, int n_out, float *y, bool relu)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int j = (int)(threadIdx.x >> 5); j < n_out; j += MF_WARPS) {
        float a = 0.f;
        for (int k = lane; k < n_in; k += 32) a += __ldg(w + j * n_in + k) * x[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        a += __ldg(b + j);
        if (lane == 0) y[j] = !relu || a > 0.f ? a : 0.f;
    }
    __syncthreads();
}

// Forward pass and choice, by one CTA; 1 + the action goes to the counter set.
__device__ __noinline__ void pick_action()
{
    const int H = P.net.hidden, no = P.net.n_out;
    const float *w1 = P.net.p, *b1 = w1 + H * MF_FEATURES, *w2 = b1 + H, *b2 = w2 + H * H, *w3 = b2 + H,
                *b3 = w3 + no * H;
    net_layer(w1, b1, sh.x, MF_FEATURES, H, sh.h1, true);
    net_layer(w2, b2, sh.h1, H, H, sh.h2, true);
    net_layer(w3, b3, sh.h2, H, no, sh.y, false);
    if (threadIdx.x == 0) {
        int best = 0;
        for (int i = 1; i < no; ++i)
            if (sh.y[i] < sh.y[best]) best = i;
        sh.cs->l[L_FCAP].w[2] = (unsigned)(1 + best);
    }
}

// One thread of every CTA: the launch goes on with this action.
__device__ __noinline__ void take_action(int action)
{
    const int k = min(max(action, 0), (int)(sizeof(kActionTable) / sizeof(MfAction)) - 1);
    const MfAction A = kActionTable[k];
    sh.action = k;
    P.kernel_cycles = A.cycles > 0 ? A.cycles : P.avg_cycles;
    P.rounds = A.rounds;
    P.cycle_div = A.cycle_div;
    P.fix_steep = A.fix;
    sh.d.resolve = A.mode;
    // near_allowed() for these rounds; the sink's row, which the next phase may
    // already be changing, was read at the launch's start
    if (A.rounds != 0 || A.fix != 0) sh.d.near = 0;
}

// Opens an iteration of the loop (its BFS comes next).
__device__ __forceinline__ void begin_iteration()
{
    MfDesc &d = sh.d;
    sh.hs.t_bfs0 = sh.hs.t_now;
    sh.hs.vis_slots = sh.hs.lvl_slots = sh.hs.lvl_cnt = sh.hs.sup = 0;
    d.lvl_lo = d.lvl_hi = d.hub_lo = d.hub_hi = 0;
    d.app_bfs = d.app_hub = 0;
    for (int b = 0; b < MF_NBIN; ++b) d.wl_app[b] = 0;
    // the used-slot total only changes with insertions, which come before the
    // first BFS: later iterations keep it
    d.need_total = sh.hs.used_slots == 0;
    d.bu_mode = 0;
}

// After a phase of the BFS.  On the critical path of every level: all it needs
// is read before anything is written, so its shared-memory accesses overlap
// instead of following one another.  Returns what the trace shows.
__device__ __forceinline__ int advance_bfs(int &hook)
{
    MfDesc &d = sh.d;
    MfState &st = sh.hs;
    const int c_bfs = cnt32(L_BFS), c_hub = cnt32(L_HUB), c_defer = cnt32(L_DEFER);
    const int c_w0 = cnt32(L_WL), c_w1 = cnt32(L_WL + 1), c_w2 = cnt32(L_WL + 2), c_w3 = cnt32(L_WL + 3);
    const unsigned long long lab = cnt64(L_LAB), exc = cnt64(L_EXC);
    const int alpha = sh.k_alpha, beta = sh.k_beta, want_wl = sh.k_wl, n = P.g.n, near = d.near;
    const int app_bfs = d.app_bfs + c_bfs, app_hub = d.app_hub + c_hub;
    const int w0 = d.wl_app[0] + c_w0, w1 = d.wl_app[1] + c_w1, w2 = d.wl_app[2] + c_w2, w3 = d.wl_app[3] + c_w3;
    const int lvl_hi = d.lvl_hi, hub_hi = d.hub_hi, hub_lo = d.hub_lo, level = d.level, bu_was = d.bu_mode;
    const long long fr = st.lvl_slots + (long long)(lab & 0xffffffffull), cnt = st.lvl_cnt + (long long)(lab >> 32);
    const long long sup = st.sup + (long long)exc, levels = st.bfs_levels;
    long long used = st.used_slots, dem = st.dem;
    const long long vis = st.vis_slots + fr;
    int shift = st.cut_shift;
    // the lists grew by what the phase appended
    d.app_bfs = app_bfs;
    d.app_hub = app_hub;
    d.wl_app[0] = w0;
    d.wl_app[1] = w1;
    d.wl_app[2] = w2;
    d.wl_app[3] = w3;
    st.sup = sup;
    if (hook == H_BU_SPLIT) {
        // after the first pass of a bottom-up level: a second pass over the
        // deferred long rows, or (none deferred) the level is complete
        d.defer_n = c_defer;
        d.bu_split = c_defer > 0 ? 1 : 0;
        if (c_defer > 0) {
            st.lvl_slots = fr;
            st.lvl_cnt = cnt;
            return (1 << 30) | min(c_defer, (1 << 20) - 1);
        }
        hook = H_BFS_NEXT;
    }
    const bool first = hook == H_BFS_START;
    if (first) {
        if (d.need_total) st.used_slots = used = (long long)cnt64(L_TOTAL);
        if (near) {
            // a cut-short relabel whose walks settled less than half of what was
            // open looks for more excess this time, so that after a few of them
            // the relabel is a complete one
            dem = (long long)cnt64(L_DEM);
            if (st.cut_prev && 2 * dem > st.dem_prev) shift = min(shift + MF_NEAR_STEP, 60);
            st.cut_shift = shift;
            st.dem = st.dem_prev = dem;
        }
    }
    const bool done = lvl_hi == app_bfs && hub_hi == app_hub;
    if (!first && !done) st.bfs_levels = levels + 1;
    d.lvl_lo = lvl_hi;
    d.hub_lo = hub_hi;
    d.lvl_hi = app_bfs;
    d.hub_hi = app_hub;
    d.level = first ? 0 : level + 1;
    st.vis_slots = vis;
    st.lvl_slots = st.lvl_cnt = 0;
    // direction of the coming level: back to top-down once the frontier holds
    // fewer than n/beta vertices
    int bu = bu_was;
    if (alpha <= 0) bu = 0;
    else if (!bu) bu = turns_bottom_up(alpha, d.level, fr, used - vis) ? 1 : 0;
    else if (cnt * beta < (long long)n) bu = 0;
    d.bu_mode = bu;
    d.bu_split = 0;
    d.bfs_squad = !done && !bu && app_hub == hub_hi && squad_level(cnt, fr) ? 1 : 0;
    // near iterations: the levels so far hold as much excess as the roots can
    // take.  Not when the solve is to end at a cap behind this BFS: it leaves a
    // complete labelling then, and the value is summed over it
    const int cut = near && !done && sup > 0 && (sup >> shift) >= dem && st.iters < P.max_iters &&
                            st.t_now - st.t_start <= P.time_limit_ns
                        ? 1 : 0;
    d.cut = cut;
    st.cut_prev = cut;
    d.bfs_done = done || cut ? 1 : 0;
    if ((done || cut) && want_wl) decide_iteration(w0 + w1 + w2 + w3);
    return ((first ? 0 : bu_was) << 30) | ((first ? 0 : min(hub_hi - hub_lo, 1023)) << 20) |
           (int)min(cnt, (long long)((1 << 20) - 1));
}

// What comes after a grid barrier: thread 0 of every CTA works it out from the
// counters of the phase that ended (sh.cnt) and the state all CTAs share, in
// shared memory only, so all of them arrive at the same answer.  t: the first
// CTA's clock.
__device__ __noinline__ void advance(int hook, unsigned long long t)
{
    MfDesc &d = sh.d;
    MfState &st = sh.hs;
    const int trace_n = st.trace_n, perr = sh.cnt[L_MISC].w;
    const int err = st.err == 0 ? perr : st.err;
    const long long barriers = st.barriers;
    const unsigned long long now = gtimer(), dt = now - st.t_phase;
    st.t_phase = now;
    st.t_now = t;
    if (barriers == 0) st.t_start = t;
    st.barriers = barriers + 1;
    st.trace_n = trace_n + 1;
    st.err = err;
    int tinfo = 0;
    if (hook == H_BU_SPLIT || hook == H_BFS_START || hook == H_BFS_NEXT) {
        st.ns_bfs += dt;
        sh.tr_info = advance_bfs(hook);
        sh.tr_hook = hook;
        if (err != 0) d.status = MF_ST_ERROR;
        return;
    }
    switch (hook) {
    case H_APPLY_VALID:
        st.ns_apply += dt;
        d.hused_n = sh.cnt[L_MISC].z;
        if (P.mode & MF_M_SCHED) batch_features();
        break;
    case H_APPLY_LOCATED:
        st.ns_apply += dt;
        d.ins_n = sh.cnt[L_MISC].x;
        if (sh.cnt[L_MISC].y != 0 && st.err == 0) st.err = MF_E_OVERFLOW;   // a row has no room for its new pairs
        if (P.mode & MF_M_SCHED) take_action(sh.cnt[L_FCAP].z - 1);
        break;
    case H_APPLY_DELTA:
    case H_NONE:
        st.ns_apply += dt;
        break;
    case H_ITER:
        if (P.mode & (MF_M_STATIC_INIT | MF_M_APPLY) && st.iters == 0) st.ns_apply += dt;
        else st.ns_fix += dt;
        begin_iteration();
        break;
    case H_WL:
        st.ns_wl += dt;
        for (int b = 0; b < MF_NBIN; ++b) d.wl_app[b] = cnt32(L_WL + b);
        decide_iteration(cnt32(L_ACT));
        break;
    case H_DIS: {
        // after a discharge round: run another one over the vertices that
        // became active during it, or end the discharge of this iteration
        st.ns_dis += dt;
        tinfo = (min(d.wl_n[2] + d.wl_n[3], 1023) << 20) |
                min(d.wl_n[0] + d.wl_n[1] + d.wl_n[2] + d.wl_n[3], (1 << 20) - 1);
        ++st.rounds_total;
        d.fix_n[0] += cnt32(L_FIX);
        d.fix_n[1] += cnt32(L_FIX + 1);
        int nxt = 0;
        for (int b = 0; b < MF_NBIN; ++b) nxt += cnt32(L_AUX + b);
        // fixed: P.rounds rounds; adaptive (P.rounds == 0): at least
        // MF_DEFAULT_ROUNDS, then more while this iteration's discharge has
        // taken less than half of its BFS -- a global relabel that costs much
        // (deep BFS, e.g. grids) is amortised over more rounds
        bool more = nxt > 0 && st.err == 0 && d.round + 1 < MF_MAX_ROUNDS;
        if (d.near && d.round == 0) {
            // the walks: rounds, which scan hub rows whole, follow only when a
            // second complete relabel in a row has left something to do, and
            // only while they are cheap beside it
            more = more && !d.cut && st.full_run > 0 && rounds_left(d, st, t);
            st.full_run = d.cut ? 0 : st.full_run + 1;
        } else if (more && d.round + 1 >= (P.rounds > 0 ? P.rounds : MF_DEFAULT_ROUNDS))
            more = P.rounds > 0 ? false : rounds_left(d, st, t);
        d.dis_more = more ? 1 : 0;
        if (more) {
            d.wl_sel ^= 1;
            for (int b = 0; b < MF_NBIN; ++b) d.wl_n[b] = cnt32(L_AUX + b);
            ++d.round;
            ++d.qstamp;
            pick_round(d, sh.csize);
        } else if (!P.fix_steep) {
            // without Alg. 3 the next iteration's BFS follows at once: this
            // barrier opens it
            begin_iteration();
        }
        break;
    }
    default:
        break;
    }
    sh.tr_hook = hook;
    sh.tr_info = tinfo;
    if (st.err != 0) d.status = MF_ST_ERROR;
}

// One entry of the hook timeline, written by the last warp of the first CTA
// beside the phase that follows: the barrier, when it was reached, and from
// what every CTA left before arriving when they finished and the slots scanned.
__device__ __noinline__ void write_trace(unsigned phase)
{
    MfCtrl *c = P.ctrl;
    const int lane = threadIdx.x & 31;
    const int i = sh.hs.trace_n - 1;
    if (i >= MF_TRACE) return;
    const unsigned *fin = c->fin[phase % 3], *scn = c->scanned[phase % 3];
    // hardware reductions of 32-bit words: times in units of 16 ns, the slot counts in halves
    unsigned fmax = 0, fsum = 0, lo = 0, hi = 0;
    const int n = min(vn(), MF_MAX_CTAS);
    for (int q = lane; q < n; q += 32) {
        const unsigned f = __ldcg(fin + q), c2 = __ldcg(scn + q);
        fmax = max(fmax, f);
        fsum += min(f, 1u << 25) >> 4;
        lo += c2 & 0xffffu;
        hi += c2 >> 16;
    }
    fmax = __reduce_max_sync(0xffffffffu, fmax);
    fsum = __reduce_add_sync(0xffffffffu, fsum);
    lo = __reduce_add_sync(0xffffffffu, lo);
    hi = __reduce_add_sync(0xffffffffu, hi);
    const unsigned long long slots = (unsigned long long)lo + ((unsigned long long)hi << 16);
    if (lane == 0) {
        MfReport *r = P.rep;
        r->trace_hook[i] = sh.tr_hook;
        r->trace_t[i] = sh.hs.t_phase;
        r->trace_slots[i] = (long long)slots;
        r->trace_info[i] = sh.tr_info;
        r->trace_fin_max[i] = fmax;
        r->trace_fin_mean[i] = (unsigned)((unsigned long long)fsum * 16u / (unsigned)n);
    }
}

// A warp copies a structure between shared memory and device memory.
__device__ __forceinline__ void words_out(int *dst, const int *sh_src, int words)
{
    for (int i = threadIdx.x & 31; i < words; i += 32) __stcg(dst + i, sh_src[i]);
}
__device__ __forceinline__ void words_in(int *sh_dst, const int *src, int words)
{
    for (int i = threadIdx.x & 31; i < words; i += 32) sh_dst[i] = __ldcg(src + i);
}

// Excess of sink and source and the BFS label counters go to memory, the
// finish time and the slots scanned into this CTA's place.  Called by warp 0
// after a __syncthreads.
__device__ __forceinline__ void arrive()
{
    MfCtrl *c = P.ctrl;
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        const unsigned long long now = gtimer();
        const int s3 = (int)(sh.phase % 3u);
        if (vb() < MF_MAX_CTAS) {
            c->fin[s3][vb()] = (unsigned)(now > sh.hs.t_phase ? now - sh.hs.t_phase : 0);
            c->scanned[s3][vb()] = (unsigned)(sh.stat[ST_SLOTS_BFS] + sh.stat[ST_SLOTS_DIS] + sh.stat[ST_SLOTS_FIX]);
        }
        if (vb() == 0) *(unsigned long long *)sh.cs->l[L_TIME].w = now;
    } else if (lane == 1) {
        if (sh.sink_e) atomic_add_ll(P.e + P.sink, sh.sink_e);
        sh.sink_e = 0;
    } else if (lane == 2) {
        if (sh.src_e) atomic_add_ll(P.e + P.source, sh.src_e);
        sh.src_e = 0;
    } else if (lane == 3) {
        if (sh.lab) atomicAdd((unsigned long long *)sh.cs->l[L_LAB].w, sh.lab);
        sh.stat[ST_LAB_BFS] += (long long)(sh.lab >> 32);
        sh.lab = 0;
    } else if (lane == 4) {
        if (sh.exc) atomicAdd((unsigned long long *)sh.cs->l[L_EXC].w, sh.exc);
        sh.exc = 0;
    } else if (lane == 7) {
        if (sh.ft_s) atomicAdd(&sh.cs->l[L_FEAT].w[0], sh.ft_s);
        if (sh.ft_t) atomicAdd(&sh.cs->l[L_FEAT].w[1], sh.ft_t);
        if (sh.ft_del) atomicAdd(&sh.cs->l[L_FEAT].w[2], sh.ft_del);
        if (sh.ft_cap) atomicAdd((unsigned long long *)sh.cs->l[L_FCAP].w, (unsigned long long)sh.ft_cap);
        sh.ft_s = sh.ft_t = sh.ft_del = 0;
        sh.ft_cap = 0;
    } else if (lane == 6) {
        sh.q_bfs = sh.q_long = sh.q_wn = 0;
        for (int b = 0; b < MF_NBIN; ++b) sh.q_wl[b] = 0;
    } else if (lane == 5) {
        if (sh.dem) atomicAdd((unsigned long long *)sh.cs->l[L_DEM].w, sh.dem);
        sh.dem = 0;
    }
    __syncwarp();
}

// One thread: this CTA is at the grid barrier.
__device__ __forceinline__ void signal_all()
{
    ++sh.arrivals;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&P.ctrl->bar.w[0]) : "memory");
}

// Wait until every CTA has arrived at the current barrier; false after the
// wait limit (MF_E_WAIT is recorded).  One thread.
__device__ __forceinline__ bool wait_all()
{
    MfCtrl *c = P.ctrl;
    const unsigned target = sh.arrivals * (unsigned)vn();
    unsigned long long t0 = 0;
    unsigned spins = 0;
    while ((int)(ld_acquire(&c->bar.w[0]) - target) < 0) {
        if ((++spins & 255u) == 0) {
            const unsigned long long now = gtimer();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > P.wait_limit_ns) {
                if (vb() < sh.csize) atomicExch(&c->bar.w[1], 1u);      // squad_entered
                *(volatile int *)&P.rep->err = MF_E_WAIT;
                return false;
            }
            if (spins > 4096) __nanosleep(100);
        }
    }
    return true;
}

// ---- thread-block clusters ----

__device__ __forceinline__ unsigned cluster_size()
{
    unsigned v;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(v));
    return v;
}

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned v;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
    return v;
}

// All threads of all CTAs of the cluster (threads that have left the kernel do
// not count).  538 clocks, against 2250 for the barrier of as many CTAs
// through memory.
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The squad's own barrier; called by all its threads.
__device__ __forceinline__ void squad_sync()
{
    if (sh.csize > 1) cluster_sync();
    else __syncthreads();
}

// Before the squad runs phases alone, all its CTAs make sure that none has given
// up at the barrier before (it may have, and left the kernel, just as the others
// saw that barrier complete): they write into one another's shared memory, which
// has to be there.  A CTA of the first cluster that gives up leaves a mark in
// memory and passes the cluster's barrier once more before it leaves
// (grid_sync); the others read the mark behind that barrier, which they pass
// here, and then all of them leave.  Only CTAs of this cluster set the mark, so
// nobody can set it between two reads.  squad_enter and squad_entered are the
// barrier's two halves; what the squad reads first is loaded between them.
__device__ __forceinline__ void squad_enter()
{
    if (sh.csize > 1 && !sh.one_cluster) {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
}
__device__ __forceinline__ bool squad_entered()
{
    if (sh.csize > 1 && !sh.one_cluster) {
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (threadIdx.x == 0) sh.ok = __ldcg(&P.ctrl->bar.w[1]) == 0 ? 1 : 0;
        __syncthreads();
    }
    return sh.ok != 0;
}

// sq[par][my rank] in every CTA of the squad = mine, by one warp; visible behind squad_sync.
__device__ __forceinline__ void squad_tell(int par, const SquadSum &mine)
{
    const int lane = threadIdx.x & 31;
    constexpr int kW = (int)(sizeof(SquadSum) / 4);
    if (lane < sh.csize) {
        const unsigned own = (unsigned)__cvta_generic_to_shared(&sh.sq[par][sh.crank]);
        unsigned there = own;
        if (sh.csize > 1) asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(own), "r"(lane));
        const int *w = reinterpret_cast<const int *>(&mine);
#pragma unroll
        for (int i = 0; i < kW; ++i)
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(there + 4u * i), "r"(w[i]) : "memory");
    }
}

// Grid-wide barrier with a hook.  Returns false if this CTA gave up waiting
// (the caller must return from the kernel at once).  One counter, which every
// CTA raises and then watches: the arrival that completes it releases all of
// them at once (304 CTAs: 1.4 us, against 2.5 us when the last one resets the
// counter and publishes a generation word), and each works out the next step
// from the counter set by itself (advance), where one thread running that
// behind the barrier for all held them up for another 3 us.  A solve that is
// one cluster uses the cluster's barrier.  With take_state, every CTA takes the
// first one's state (its squad ran phases alone) before working out the next;
// two such barriers may follow one another, so the state has two copies (MfCtrl).
__device__ __noinline__ bool grid_sync(int hook, bool take_state = false)
{
    MfCtrl *c = P.ctrl;
    __syncthreads();
    const unsigned k = sh.phase;
    const bool one = sh.one_cluster != 0;
    if (threadIdx.x < 32) {
        if (take_state && vb() == 0) {
            words_out((int *)&c->jd[k % MF_HANDOVER], (const int *)&sh.d, (int)(sizeof(MfDesc) / 4));
            words_out((int *)&c->js[k % MF_HANDOVER], (const int *)&sh.hs, (int)(sizeof(MfState) / 4));
        }
        arrive();
    }
    if (one) cluster_sync();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int ok = 1;
        if (lane == 0 && !one) {
            signal_all();
            ok = wait_all() ? 1 : 0;
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
        if (ok) {
            if (lane < MF_LINES) {
                sh.cnt[lane] = __ldcg(reinterpret_cast<const int4 *>(&sh.cs->l[lane]));
                if (vb() == 0) __stcg(reinterpret_cast<int4 *>(&c->set[(k + 2u) % 3u].l[lane]), make_int4(0, 0, 0, 0));
            }
            if (take_state && vb() != 0) {
                words_in((int *)&sh.d, (const int *)&c->jd[k % MF_HANDOVER], (int)(sizeof(MfDesc) / 4));
                words_in((int *)&sh.hs, (const int *)&c->js[k % MF_HANDOVER], (int)(sizeof(MfState) / 4));
            }
            __syncwarp();
            if (lane == 0) advance(hook, cnt64(L_TIME));
        }
        if (lane == 0) {
            sh.ok = ok;
            sh.phase = k + 1u;
            sh.cs = &c->set[(k + 1u) % 3u];
        }
    }
    __syncthreads();
    if (vb() == 0 && (threadIdx.x >> 5) == (blockDim.x >> 5) - 1 && sh.ok) write_trace(k);
    if (sh.ok == 0 && sh.csize > 1 && !one && vb() < sh.csize) cluster_sync();    // squad_entered
    return sh.ok != 0;
}

// The end of a launch: the counters go to the control block, every CTA arrives
// once more, and the first one alone waits for the others, writes the results
// down and leaves barrier and counter sets at zero for the next launch.
__device__ __noinline__ bool finish()
{
    MfCtrl *c = P.ctrl;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        if (lane < MF_STATS && sh.stat[lane]) atomic_add_ll(&c->stat[lane], sh.stat[lane]);
        if (lane == 31 && sh.value) atomic_add_ll(&c->value, sh.value);
        __syncwarp();
        arrive();
        if (lane == 0) signal_all();
        if (vb() == 0) {
            int ok = 0;
            if (lane == 0) ok = wait_all() ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            __syncwarp();
            if (lane == 0) {
                sh.ok = ok;
                MfState &st = sh.hs;
                st.t_phase = gtimer();
                ++st.barriers;
                ++st.trace_n;
                sh.tr_hook = H_FINAL;
                sh.tr_info = 0;
            }
            __syncwarp();
            if (ok) {
                write_trace(sh.phase);
                const int4 zero = make_int4(0, 0, 0, 0);
                if (lane < MF_LINES)
                    for (int q = 0; q < 3; ++q) __stcg(reinterpret_cast<int4 *>(&c->set[q].l[lane]), zero);
                MfReport *r = P.rep;
                if (lane < MF_STATS) r->stat[lane] = __ldcg(&c->stat[lane]);
                if (lane == 0) {
                    const MfState &st = sh.hs;
                    c->bar.w[0] = 0;
                    c->qstamp = sh.d.qstamp;
                    c->fstamp = sh.d.fstamp;
                    r->err = st.err;
                    r->status = sh.d.status;
                    r->action = sh.action;
                    r->value = __ldcg(&c->value);
                    r->iters = st.iters;
                    r->bfs_levels = st.bfs_levels;
                    r->active_total = st.active_total;
                    r->active_first = st.active_first;
                    r->cut_slots = st.vis_slots;
                    r->used_slots = st.used_slots;
                    r->ns_bfs = st.ns_bfs;
                    r->ns_dis = st.ns_dis;
                    r->ns_fix = st.ns_fix;
                    r->ns_wl = st.ns_wl;
                    r->ns_apply = st.ns_apply;
                    r->rounds_total = st.rounds_total;
                    r->barriers = st.barriers;
                    r->trace_n = st.trace_n;
                    r->t_exit = st.t_phase;
                }
            }
        }
    }
    __syncthreads();
    return vb() != 0 || sh.ok != 0;
}

// Add d to the excess of z (sink and source go to the CTA accumulators).
__device__ __forceinline__ void add_excess(int z, long long d)
{
    if (z == P.sink)
        add_shared(sh.sink_e, d);
    else if (z == P.source)
        add_shared(sh.src_e, d);
    else
        atomic_add_ll(P.e + z, d);
}

// ---------------------------------------------------------------------------
// Static initialisation (Alg. 1)
// ---------------------------------------------------------------------------

// c_f = c on every slot, e = h = 0: a streaming copy, 16-byte vectors with four
// in flight per thread (the slot arrays start on 256-byte boundaries).
__device__ __noinline__ void phase_static_reset()
{
    const long long gt = (long long)vb() * blockDim.x + threadIdx.x;
    const long long gs = (long long)vn() * blockDim.x;
    const long long n4 = P.g.slot_cap >> 2;
    const int4 *src = reinterpret_cast<const int4 *>(P.g.cap);
    int4 *dst = reinterpret_cast<int4 *>(P.cf);
    long long x = gt;
    for (; x + 3 * gs < n4; x += 4 * gs) {
        const int4 a = __ldcs(src + x), b = __ldcs(src + x + gs), c = __ldcs(src + x + 2 * gs),
                   d = __ldcs(src + x + 3 * gs);
        __stcg(dst + x, a);
        __stcg(dst + x + gs, b);
        __stcg(dst + x + 2 * gs, c);
        __stcg(dst + x + 3 * gs, d);
    }
    for (; x < n4; x += gs) __stcg(dst + x, __ldcs(src + x));
    for (long long y = (n4 << 2) + gt; y < P.g.slot_cap; y += gs) P.cf[y] = __ldcg(P.g.cap + y);
    for (long long v = gt; v < P.g.n; v += gs) {
        P.e[v] = 0;
        P.h[v] = 0;
    }
}

__device__ __noinline__ void phase_saturate_source()
{
    const int s = P.source;
    const int r0 = P.g.off[s];
    const int d = ldg_cg(P.g.deg + s);
    long long acc = 0;
    for (int j = vb() * blockDim.x + threadIdx.x; j < d; j += vn() * blockDim.x) {
        int x = r0 + j;
        int c = ldg_cg(P.g.cap + x);
        int y = ldg_cg(P.g.rev + x);
        P.cf[x] = 0;
        P.cf[y] = ldg_cg(P.g.pcap + x);
        int z = ldg_cg(P.g.dst + x);
        if (z == P.sink)
            add_shared(sh.sink_e, c);
        else
            P.e[z] = c;
        acc -= c;
    }
    if (acc) add_shared(sh.src_e, acc);
}

// Static push-pull (Sec. 5.2.2): every edge into t is saturated as well; its
// tail keeps the deficit, and the deficient vertices then act as sinks.
__device__ __noinline__ void phase_saturate_sink()
{
    const int t = P.sink;
    const int r0 = P.g.off[t];
    const int d = ldg_cg(P.g.deg + t);
    long long acc = 0;
    for (int j = vb() * blockDim.x + threadIdx.x; j < d; j += vn() * blockDim.x) {
        const int x = r0 + j;                  // slot (t, z)
        const int y = ldg_cg(P.g.rev + x);     // slot (z, t)
        const int c = ldg_cg(P.cf + y);
        if (c > 0) {
            P.cf[y] = 0;
            P.cf[x] = ldg_cg(P.cf + x) + c;
            add_excess(ldg_cg(P.g.dst + x), -(long long)c);
            acc += c;
        }
    }
    if (acc) add_shared(sh.sink_e, acc);
}

// Dynamic push-pull (Sec. 5.2.2): the sides of the last cut, read from the
// heights the previous solve ended with (1: the vertex reached t or a
// deficit, 0: it did not) ...
__device__ __noinline__ void phase_cut_side()
{
    const int n = P.g.n;
    const long long gs = (long long)vn() * blockDim.x;
    for (long long v = (long long)vb() * blockDim.x + threadIdx.x; v < n; v += gs) {
        uint8_t sd = ldg_cg(P.h + v) < n ? 1 : 0;
        if (v == P.source) sd = 0;
        if (v == P.sink) sd = 1;
        P.side[v] = sd;
    }
}

// ... then every residual edge from side 0 to side 1 sends all it can, so
// that no residual path leads from side 0 to side 1.  Slots j0, j0 + step, ... of
// a row; returns what its vertex sent.
__device__ __forceinline__ long long saturate_row(int r0, int d, int j0, int step)
{
    long long out = 0;
    for (int j = j0; j < d; j += step) {
        const int x = r0 + j;
        const int c = ldg_cg(P.cf + x);
        if (c <= 0) continue;
        const int z = ldg_cg(P.g.dst + x);
        if (P.side[z] != 1) continue;
        P.cf[x] = 0;
        atomicAdd(P.cf + ldg_cg(P.g.rev + x), c);
        add_excess(z, (long long)c);
        out += c;
    }
    return out;
}

// One warp per row, consecutive rows in different CTAs; rows of more than
// MF_HUB_DEG slots wait in a list for their whole CTA.  The longest chain of a
// warp's rows bounds it: with hub rows walked by one warp each, the longest on
// R-MAT 20 was 6578 steps of 32 slots when 4864 warps shared the rows and 9402
// when 4608 did (whose count has more factors of two, as the hubs' numbers do),
// 7.7 and 9.3 ms of an update by push-pull; the whole update now takes 3.4 ms.
__device__ __noinline__ void phase_saturate_cut()
{
    const int n = P.g.n;
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)vn() * blockDim.x) >> 5;
    if (threadIdx.x == 0) sh.bcast_i = 0;
    __syncthreads();
    for (long long u = warp_rank(vn(), 0); u < n; u += nw) {
        if (P.side[u] != 0) continue;
        const int r0 = P.g.off[u], d = ldg_cg(P.g.deg + u);
        if (d > MF_HUB_DEG) {
            int at = 0;
            if (lane == 0) {
                at = atomicAdd(&sh.bcast_i, 1);
                if (at < P.stage_slots) mf_stage[at] = (int)u;
            }
            if (__shfl_sync(0xffffffffu, at, 0) < P.stage_slots) continue;
        }
        const long long out = warp_sum_ll(saturate_row(r0, d, lane, 32));
        if (lane == 0 && out) add_excess((int)u, -out);
    }
    __syncthreads();
    const int nl = min(sh.bcast_i, P.stage_slots);
    for (int i = 0; i < nl; ++i) {
        const int u = mf_stage[i];
        const long long out = warp_sum_ll(saturate_row(P.g.off[u], ldg_cg(P.g.deg + u), threadIdx.x, blockDim.x));
        if (lane == 0 && out) add_excess(u, -out);
    }
}

// Append val to arr for the lanes with take, one atomic per warp.  Called by
// the whole warp.
__device__ __forceinline__ void warp_append(unsigned *tail, int *arr, bool take, int val)
{
    const unsigned m = __ballot_sync(0xffffffffu, take);
    if (m == 0) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(tail, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (take) arr[base + __popc(m & ((1u << lane) - 1u))] = val;
}

// ---------------------------------------------------------------------------
// Batch apply and repair (Alg. 5)
// ---------------------------------------------------------------------------

__device__ __forceinline__ bool batch_entry(long long i, int &u, int &v, int &c)
{
    u = __ldcg(P.bu + i);
    v = __ldcg(P.bv + i);
    c = __ldcg(P.bc + i);
    return u >= 0 && u < P.g.n && v >= 0 && v < P.g.n && c >= 0;
}

// Validate every entry; insert the directed key into the dedup table, where
// the largest batch index (the last update of the pair) wins.
__device__ __noinline__ void phase_apply_validate()
{
    MfSet *cs = sh.cs;
    const int bits = P.sc.hash_bits;
    const unsigned mask = (1u << bits) - 1u;
    const int lane = threadIdx.x & 31;
    const bool sched = (P.mode & MF_M_SCHED) != 0;
    unsigned fs = 0, ft = 0, fz = 0;
    long long fcap = 0;
    // warp-uniform loop: the positions taken in the table are appended with one atomic per warp
    for (long long base = spread_warp(vn()) - lane; base < P.bcount; base += (long long)vn() * blockDim.x) {
        const long long i = base + lane;
        bool fresh = false;
        unsigned pos = 0;
        int u, v, c;
        if (i < P.bcount) {
            const bool fine = batch_entry(i, u, v, c);
            if (sched) {
                fs += u == P.source || v == P.source;
                ft += u == P.sink || v == P.sink;
                fz += c == 0;
                fcap += c;
            }
            if (!fine) {
                atomicCAS(&cs->l[L_MISC].w[3], 0u, (unsigned)MF_E_INVALID);
            } else if (u != v) {
                unsigned long long key = ((unsigned long long)(unsigned)u << 32) | (unsigned)v;
                pos = hash_slot(key, bits);
                for (unsigned probe = 0; probe <= mask; ++probe) {
                    unsigned long long prev = atomicCAS(P.sc.hkey + pos, kEmpty, key);
                    if (prev == kEmpty || prev == key) {
                        fresh = prev == kEmpty;
                        atomicMax(P.sc.hval + pos, (int)i);
                        break;
                    }
                    pos = (pos + 1u) & mask;
                }
            }
        }
        warp_append(&cs->l[L_MISC].w[2], P.sc.hused, fresh, (int)pos);   // positions to clear afterwards
    }
    if (sched) {
        fs = __reduce_add_sync(0xffffffffu, fs);
        ft = __reduce_add_sync(0xffffffffu, ft);
        fz = __reduce_add_sync(0xffffffffu, fz);
        fcap = warp_sum_ll(fcap);
        if (lane == 0) {
            if (fs) atomicAdd(&sh.ft_s, fs);
            if (ft) atomicAdd(&sh.ft_t, ft);
            if (fz) atomicAdd(&sh.ft_del, fz);
            if (fcap) add_shared(sh.ft_cap, fcap);
        }
    }
}

// Slot of (u, v) in u's row, or -1: an 8-way search of the sorted base slots
// (seven pivots loaded together per round, so a row of 2^15 slots takes five
// dependent rounds instead of fifteen), then a scan of the inserted slots.
// *probes counts the dst entries read.
__device__ __noinline__ int find_slot(const MfParams &P, int u, int v, int *probes = nullptr)
{
    const int r0 = P.g.off[u];
    const int bd = ldg_cg(P.g.bdeg + u);
    int lo = r0, hi = r0 + bd;      // the first base slot with dst >= v lies in [lo, hi]
    int k = 0;
    while (hi - lo > 8) {
        const int step = (hi - lo) >> 3;
        int below = 0;
#pragma unroll
        for (int q = 1; q < 8; ++q) below += ldg_cg(P.g.dst + lo + q * step) < v ? 1 : 0;
        k += 7;
        const int nlo = below > 0 ? lo + below * step + 1 : lo;
        if (below < 7) hi = lo + (below + 1) * step;
        lo = nlo;
    }
    int below = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) below += (lo + q < hi && ldg_cg(P.g.dst + lo + q) < v) ? 1 : 0;
    k += hi - lo;
    int found = -1;
    const int lb = lo + below;
    if (lb < r0 + bd && ldg_cg(P.g.dst + lb) == v) found = lb;
    ++k;
    if (found < 0) {
        const int end = r0 + ldg_cg(P.g.deg + u);
        for (int x = r0 + bd; x < end; ++x) {
            ++k;
            if (ldg_cg(P.g.dst + x) == v) {
                found = x;
                break;
            }
        }
    }
    if (probes) *probes += k;
    return found;
}

// Slot of (u, v), or -1, looked for in the shorter of the two rows: the pair has a
// slot in both, and on power-law graphs one end of most edges is a hub.  A row's
// base slots are searched, its inserted ones read one by one, so the other row
// is only taken if it has no more of those.
__device__ __forceinline__ int find_pair(int u, int v, int *probes)
{
    const int bu = ldg_cg(P.g.bdeg + u), bv = ldg_cg(P.g.bdeg + v);
    const int iu = ldg_cg(P.g.deg + u) - bu, iv = ldg_cg(P.g.deg + v) - bv;
    if (2ll * bv < bu && iv <= iu) {
        const int y = find_slot(P, v, u, probes);
        return y < 0 ? -1 : ldg_cg(P.g.rev + y);
    }
    return find_slot(P, u, v, probes);
}

__device__ __forceinline__ unsigned hash_find(const unsigned long long *keys, int bits, unsigned long long key)
{
    const unsigned mask = (1u << bits) - 1u;
    unsigned pos = hash_slot(key, bits);
    for (unsigned probe = 0; probe <= mask; ++probe) {
        unsigned long long k = __ldcg(keys + pos);
        if (k == key) return pos;
        if (k == kEmpty) return 0xffffffffu;
        pos = (pos + 1u) & mask;
    }
    return 0xffffffffu;
}

// Locate the slot of every surviving update; a missing pair is entered once
// into the new-pair table and counted against both rows' spare slots.  The
// pair sum the batch leaves behind is checked here, before anything changes:
// c' plus the final capacity of the reverse direction -- the batch's own
// update of (v, u) if it has one, else the current c(v, u), else 0 for a new
// pair -- must fit int32 (residual capacities are int32 and c_f(u,v) +
// c_f(v,u) equals that sum).  A batch that breaks it sets MF_E_TOO_LARGE and
// is refused whole.  Done by the first nctas CTAs.
__device__ __noinline__ void phase_apply_locate(int nctas)
{
    MfSet *cs = sh.cs;
    const int bits = P.sc.hash_bits;
    const unsigned mask = (1u << bits) - 1u;
    const int lane = threadIdx.x & 31;
    int probes = 0;
    for (long long base = spread_warp(nctas) - lane; base < P.bcount; base += (long long)nctas * blockDim.x) {
        const long long i = base + lane;
        bool fresh = false;
        unsigned pp = 0;
        int u = 0, v = 0, c = 0;
        if (i < P.bcount) batch_entry(i, u, v, c);
        unsigned long long key = ((unsigned long long)(unsigned)u << 32) | (unsigned)v;
        const unsigned pos = (i < P.bcount && u != v) ? hash_find(P.sc.hkey, bits, key) : 0xffffffffu;
        if (i >= P.bcount) {
            // past the batch
        } else if (pos == 0xffffffffu || __ldcg(P.sc.hval + pos) != (int)i) {
            P.sc.bslot[i] = -2;     // a self-loop, or a later update of the same pair wins
        } else {
            const int x = find_pair(u, v, &probes);
            P.sc.bslot[i] = x;
            {
                const unsigned long long rkey = ((unsigned long long)(unsigned)v << 32) | (unsigned)u;
                const unsigned rp = hash_find(P.sc.hkey, bits, rkey);
                long long crev = 0;
                if (rp != 0xffffffffu) crev = __ldcg(P.bc + __ldcg(P.sc.hval + rp));
                else if (x >= 0) crev = ldg_cg(P.g.cap + ldg_cg(P.g.rev + x));
                if ((long long)c + crev > (long long)INT32_MAX)
                    atomicCAS(&cs->l[L_MISC].w[3], 0u, (unsigned)MF_E_TOO_LARGE);
            }
            if (x < 0) {
                const int a = min(u, v), b = max(u, v);
                const unsigned long long pk = ((unsigned long long)(unsigned)a << 32) | (unsigned)b;
                pp = hash_slot(pk, bits);
                for (unsigned probe = 0; probe <= mask; ++probe) {
                    unsigned long long prev = atomicCAS(P.sc.pkey + pp, kEmpty, pk);
                    if (prev == kEmpty) {
                        // the room check: the increment that reaches a row's final
                        // demand sees it, so a row short of spare slots is flagged
                        fresh = true;
                        const int na = atomicAdd(P.sc.ins_need + a, 1) + 1;
                        const int nb = atomicAdd(P.sc.ins_need + b, 1) + 1;
                        if (na > P.g.off[a + 1] - P.g.off[a] - ldg_cg(P.g.deg + a) ||
                            nb > P.g.off[b + 1] - P.g.off[b] - ldg_cg(P.g.deg + b))
                            atomicExch(&cs->l[L_MISC].w[1], 1u);
                        break;
                    }
                    if (prev == pk) break;
                    pp = (pp + 1u) & mask;
                }
            }
        }
        warp_append(&cs->l[L_MISC].w[0], P.sc.ins_list, fresh, (int)pp);   // each new pair once
    }
    add_stat(ST_SLOTS_APPLY, probes);
}

// Winning new capacity of the directed pair (a, b) in the batch, or -1 if the
// batch does not set it.
__device__ __forceinline__ int batch_cap_of(int a, int b)
{
    const unsigned long long key = ((unsigned long long)(unsigned)a << 32) | (unsigned)b;
    const unsigned pos = hash_find(P.sc.hkey, P.sc.hash_bits, key);
    return pos == 0xffffffffu ? -1 : __ldcg(P.bc + __ldcg(P.sc.hval + pos));
}

// Alg. 5, capacity step, in one phase: (1) every new pair gets its two slots,
// with the batch's capacities set directly (no flow runs on a new pair, so
// c_f = c); (2) every located update sets c(u,v) = c', adds c' - c to c_f(u,v)
// and to both pair sums, and when c_f(u,v) drops below zero sends the
// difference back (the clamp step: c_f(v,u) -= d, e(u) += d, e(v) -= d).
// The dedup table gives every directed pair one owner; the only other writer
// of c_f(u,v) is the owner of (v,u), and the two clamps cannot both fire (the
// pair's residuals sum to the new c(u,v) + c(v,u) >= 0), so the order of the
// atomics does not matter.
__device__ __noinline__ void phase_apply_change()
{
    const int nins = sh.d.ins_n;
    long long applied = 0, clamped = 0;
    for (long long k = spread_thread(); k < nins; k += (long long)vn() * blockDim.x) {
        int pp = __ldcg(P.sc.ins_list + k);
        unsigned long long pk = __ldcg(P.sc.pkey + pp);
        int a = (int)(pk >> 32), b = (int)(pk & 0xffffffffu);
        const int ca = batch_cap_of(a, b), cb = batch_cap_of(b, a);
        const int xa = P.g.off[a] + atomicAdd(P.g.deg + a, 1);
        const int xb = P.g.off[b] + atomicAdd(P.g.deg + b, 1);
        const int va = ca > 0 ? ca : 0, vb2 = cb > 0 ? cb : 0;
        P.g.dst[xa] = b;
        P.g.dst[xb] = a;
        P.g.rev[xa] = xb;
        P.g.rev[xb] = xa;
        P.g.cap[xa] = va;
        P.g.cap[xb] = vb2;
        P.g.pcap[xa] = P.g.pcap[xb] = va + vb2;
        P.cf[xa] = va;
        P.cf[xb] = vb2;
        P.sc.ins_need[a] = 0;
        P.sc.ins_need[b] = 0;
        applied += (ca >= 0 ? 1 : 0) + (cb >= 0 ? 1 : 0);
    }
    for (long long i = spread_thread(); i < P.bcount; i += (long long)vn() * blockDim.x) {
        const int x = __ldcg(P.sc.bslot + i);
        if (x < 0) continue;                 // superseded, ignored, or a new pair (set above)
        int u, v, c;
        batch_entry(i, u, v, c);
        const int old = ldg_cg(P.g.cap + x);
        const int delta = c - old;
        ++applied;
        if (delta == 0) continue;
        const int y = ldg_cg(P.g.rev + x);
        P.g.cap[x] = c;
        const int cf_new = atomicAdd(P.cf + x, delta) + delta;
        atomicAdd(P.g.pcap + x, delta);
        atomicAdd(P.g.pcap + y, delta);
        if (cf_new < 0) {
            const int d = -cf_new;
            atomicAdd(P.cf + x, d);
            atomicAdd(P.cf + y, -d);
            add_excess(u, (long long)d);
            add_excess(v, -(long long)d);
            ++clamped;
        }
    }
    add_stat(ST_N_APPLY, applied);
    add_stat(ST_CLAMPS_APPLY, clamped);
}

// keep_need: leave ins_need[] as it is (the rows' demand of spare slots after
// an overflow; the rebuild that follows reads and clears it).
__device__ __noinline__ void phase_apply_cleanup(bool keep_need)
{
    const int nused = sh.d.hused_n;
    const int nins = sh.d.ins_n;
    for (int k = vb() * blockDim.x + threadIdx.x; k < nused; k += vn() * blockDim.x) {
        int pos = __ldcg(P.sc.hused + k);
        P.sc.hkey[pos] = kEmpty;
        P.sc.hval[pos] = -1;
    }
    for (int k = vb() * blockDim.x + threadIdx.x; k < nins; k += vn() * blockDim.x) {
        int pp = __ldcg(P.sc.ins_list + k);
        unsigned long long pk = __ldcg(P.sc.pkey + pp);
        if (pk != kEmpty && !keep_need) {
            int a = (int)(pk >> 32), b = (int)(pk & 0xffffffffu);
            P.sc.ins_need[a] = 0;
            P.sc.ins_need[b] = 0;
        }
        P.sc.pkey[pp] = kEmpty;
    }
}

// The source step of Alg. 5 (reading: push the remaining residual of every edge out
// of the source and add it to the head's excess).
__device__ __noinline__ void phase_resaturate()
{
    const int s = P.source;
    const int r0 = P.g.off[s];
    const int d = ldg_cg(P.g.deg + s);
    long long acc = 0;
    if (vb() == 0 && threadIdx.x == 0) add_stat(ST_SLOTS_APPLY, d);
    for (int j = vb() * blockDim.x + threadIdx.x; j < d; j += vn() * blockDim.x) {
        int x = r0 + j;
        int c = ldg_cg(P.cf + x);
        if (c > 0) {
            P.cf[x] = 0;
            atomicAdd(P.cf + ldg_cg(P.g.rev + x), c);
            add_excess(ldg_cg(P.g.dst + x), (long long)c);
            acc -= c;
        }
    }
    if (acc) add_shared(sh.src_e, acc);
}

// ---------------------------------------------------------------------------
// Backward BFS (Alg. 4 / Alg. 6)
// ---------------------------------------------------------------------------

// The work items of vertex z (d slots from r0), by one thread: where a queue has no room.
__device__ __forceinline__ void put_items(int r0, int d, unsigned at)
{
    for (int j = 0; j < d; j += MF_BFS_CHUNK)
        P.sc.bitem[at++] = make_int2(r0 + j, d - j < MF_BFS_CHUNK ? d - j : MF_BFS_CHUNK);
}

__device__ __forceinline__ int chunks_of(int d) { return (d + MF_BFS_CHUNK - 1) / MF_BFS_CHUNK; }

// z (a row of d slots) joins a worklist: the BFS's own (line L_WL, the lists
// wl[sel]) or the next round's (L_AUX, wl[sel ^ 1]).  The entry waits in the
// CTA's queue until the phase ends, so that each CTA, not each warp, takes its
// room in the shared lists with one atomic per list: returning atomics on one
// word are served one after another, about 2.4 clocks each, and a level whose
// 4864 warps append alone spends some 5 us on that.
__device__ __forceinline__ void place_active(int z, int d, int line, int sel,
                                             const int *app)
{
    const int bin = row_bin(d);
    if (P.stage_slots >= MF_Q_INTS) {
        const int j = atomicAdd(&sh.q_wn, 1);
        if (j < MF_Q_WL) {
            int *q = mf_stage + MF_Q_BFS + MF_Q_LONG;
            q[j] = z;
            q[MF_Q_WL + j] = (bin << 28) | atomicAdd(&sh.q_wl[bin], 1);
            return;
        }
    }
    P.sc.wl[sel][bin][(app ? app[bin] : 0) + atomicAdd(&sh.cs->l[line + bin].w[0], 1u)] = z;
}

// A labelled vertex enters the next frontier either as one entry of the regular
// list (rows of at most bfs_hub slots, expanded warp-cooperatively) or, for
// longer rows, as ceil(deg / MF_BFS_CHUNK) work items (first slot, length) that
// any warp can take: no row is ever walked by one warp alone.  One that has
// excess (ev > 0; never the sink or the source) also joins the worklist of the
// coming discharge (Sec. 5.2.1 O1): it is active exactly when this BFS labels
// it, so no separate pass over all vertices is needed.  The entries wait in the
// CTA's queue (flush_labelled).
__device__ __forceinline__ void place_labelled(int z, int d, long long ev)
{
    const bool room = P.stage_slots >= MF_Q_INTS;
    if (d > P.bfs_hub) {
        const int i = room ? atomicAdd(&sh.q_long, 1) : MF_Q_LONG;
        if (i < MF_Q_LONG)
            mf_stage[MF_Q_BFS + i] = z;
        else
            put_items(P.g.off[z], d, sh.d.app_hub + atomicAdd(&sh.cs->l[L_HUB].w[0], (unsigned)chunks_of(d)));
    } else {
        const int i = room ? atomicAdd(&sh.q_bfs, 1) : MF_Q_BFS;
        if (i < MF_Q_BFS)
            mf_stage[i] = z;
        else
            P.sc.border[sh.d.app_bfs + atomicAdd(&sh.cs->l[L_BFS].w[0], 1u)] = z;
    }
    if (ev > 0) {
        place_active(z, d, L_WL, sh.d.wl_sel, sh.d.wl_app);
        if (sh.d.near) add_shared(sh.exc, ev);
    }
}

// The work items of nl long-row vertices (in shared memory), by the whole CTA: a
// warp takes 32 vertices, makes room for all their items at once and writes
// them together, each lane finding the vertex that owns its item.  (A warp per
// vertex took 5 us where three CTAs had labelled 270 hubs between them.)
__device__ __forceinline__ void write_long(const int *list, int nl)
{
    const int lane = threadIdx.x & 31;
    for (int b = (int)(threadIdx.x & ~31u); b < nl; b += blockDim.x) {
        const int z = b + lane < nl ? list[b + lane] : -1;
        const int d = z >= 0 ? ldg_cg(P.g.deg + z) : 0, r0 = z >= 0 ? P.g.off[z] : 0, nc = chunks_of(d);
        int incl = nc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int excl = incl - nc, tot = __shfl_sync(0xffffffffu, incl, 31);
        unsigned at = 0;
        if (lane == 0) at = sh.d.app_hub + atomicAdd(&sh.cs->l[L_HUB].w[0], (unsigned)tot);
        at = __shfl_sync(0xffffffffu, at, 0);
        for (int i0 = 0; i0 < tot; i0 += 32) {
            const int i = i0 + lane;
            int owner = 0;
#pragma unroll
            for (int st = 16; st >= 1; st >>= 1) {
                const int cand = owner + st;
                const int ec = __shfl_sync(0xffffffffu, excl, cand & 31);
                if (cand < 32 && ec <= i) owner = cand;
            }
            const int rb = __shfl_sync(0xffffffffu, r0, owner), rd_ = __shfl_sync(0xffffffffu, d, owner);
            const int j = (i - __shfl_sync(0xffffffffu, excl, owner)) * MF_BFS_CHUNK;
            if (i < tot) P.sc.bitem[at + i] = make_int2(rb + j, rd_ - j < MF_BFS_CHUNK ? rd_ - j : MF_BFS_CHUNK);
        }
    }
}

// The end of a phase: the CTA's queue goes onto the shared lists, and what its
// threads labelled (vertices, slots) to the counters.  Long rows' work items
// are written here.
__device__ __forceinline__ void flush_queue(int line, int sel, const int *app, int lab,
                                            unsigned lab_slots)
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    __syncwarp();
    lab = __reduce_add_sync(0xffffffffu, lab);
    lab_slots = __reduce_add_sync(0xffffffffu, lab_slots);
    if (lane == 0 && lab) add_shared(sh.lab, ((long long)lab << 32) | lab_slots);
    __syncthreads();
    const int nb = min(sh.q_bfs, MF_Q_BFS), nl = min(sh.q_long, MF_Q_LONG), nw = min(sh.q_wn, MF_Q_WL);
    if (nb + nw > 0) {
        // a lane per list, so the reservations are in flight together
        if (tid < MF_NBIN) {
            if (sh.q_wl[tid])
                sh.q_base[tid] = (app ? app[tid] : 0) + (int)atomicAdd(&sh.cs->l[line + tid].w[0], (unsigned)sh.q_wl[tid]);
        } else if (tid == MF_NBIN) {
            if (nb) sh.q_base[MF_NBIN] = sh.d.app_bfs + (int)atomicAdd(&sh.cs->l[L_BFS].w[0], (unsigned)nb);
        }
        __syncthreads();
        for (int i = tid; i < nb; i += nt) P.sc.border[sh.q_base[MF_NBIN] + i] = mf_stage[i];
        const int *q = mf_stage + MF_Q_BFS + MF_Q_LONG;
        for (int i = tid; i < nw; i += nt) {
            const int b = q[MF_Q_WL + i];
            P.sc.wl[sel][b >> 28][sh.q_base[b >> 28] + (b & 0x0fffffff)] = q[i];
        }
    }
    write_long(mf_stage + MF_Q_BFS, nl);
}

__device__ __forceinline__ void flush_labelled(int lab, unsigned lab_slots)
{
    flush_queue(L_WL, sh.d.wl_sel, sh.d.wl_app, lab, lab_slots);
}

__device__ __noinline__ void phase_bfs_init()
{
    const int n = P.g.n;
    const bool deficit_roots = (P.mode & MF_M_NO_DEFICIT_ROOTS) == 0;
    const bool pull = P.pull != 0;
    const bool need_total = sh.d.need_total != 0;
    const bool near = sh.d.near != 0;
    long long total = 0, take = 0;        // near: what the roots can take
    int lab = 0;
    unsigned lab_slots = 0;
    const int lane = threadIdx.x & 31;
    const long long gs = (long long)vn() * blockDim.x;
    if (near) {
        const int r0 = P.g.off[P.sink], d = ldg_cg(P.g.deg + P.sink);
        for (long long j = (long long)vb() * blockDim.x + threadIdx.x; j < d; j += gs)
            take += ldg_cg(P.g.pcap + r0 + j) - ldg_cg(P.cf + r0 + j);
    }
    if (vb() == 0 && threadIdx.x == 0) add_stat(ST_VERTS_BFS, n);     // every vertex: e read, h written
    for (long long base = (long long)vb() * blockDim.x + threadIdx.x - lane; base < n; base += gs) {
        const int v = (int)base + lane;
        bool root = false;
        int dall = 0;
        if (v < n) {
            if (need_total) dall = ldg_cg(P.g.deg + v);
            // push: t and the deficient vertices; pull (Sec. 5.2.2): s and the
            // overflowing vertices; with a side given, only that side's
            const bool side_ok = P.side_root < 0 || P.side[v] == P.side_root;
            if (pull)
                root = (v == P.source) || (v != P.sink && side_ok && ldg_cg(P.e + v) > 0);
            else {
                const long long e = (deficit_roots && v != P.source && v != P.sink && side_ok) ? ldg_cg(P.e + v) : 0;
                root = v == P.sink || e < 0;
                if (near && e < 0) {
                    P.sc.dem[v] = -e;
                    take -= e;
                }
            }
            P.h[v] = root ? 0 : n;
            if (root) {
                const int d = need_total ? dall : ldg_cg(P.g.deg + v);
                ++lab;
                lab_slots += (unsigned)d;
                place_labelled(v, d, 0);
            }
        }
        total += dall;
    }
    if (take) add_shared(sh.dem, take);
    flush_labelled(lab, lab_slots);
    if (need_total) {
        // one atomic per CTA for the used-slot total
        total = warp_sum_ll(total);
        if (lane == 0) sh.wsum[threadIdx.x >> 5] = total;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long t = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh.wsum[w];
            if (t) atomicAdd((unsigned long long *)sh.cs->l[L_TOTAL].w, (unsigned long long)t);
        }
        __syncthreads();
    }
}

// Visit BR slots per lane at level L.  Slot x = (u, z): z gets height L+1 if
// it is unlabelled, is not the source, and has a residual edge (z, u), i.e.
// c_f(z, u) = pcap - c_f(u, z) > 0.  Each stage (slot loads, height gathers,
// claims, degree/excess loads) is issued for all BR slots together, so each
// lane keeps BR independent requests in flight.
template <int BR>
__device__ __forceinline__ void bfs_visit(const int (&x)[BR], const bool (&valid)[BR], int L,
                                          int &lab, unsigned &lab_slots)
{
    const bool with_wl = P.data_driven && !(P.mode & MF_M_BFS_ONLY);
    const bool pull = P.pull != 0;
    const int skip = pull ? P.sink : P.source;     // the terminal a BFS never labels
    const bool near = sh.d.near != 0;
    const int t0 = near && L == 0 ? P.g.off[P.sink] : 0, t1 = near && L == 0 ? t0 + ldg_cg(P.g.deg + P.sink) : 0;
    const int n = P.g.n;
    int z[BR], rc[BR], hz[BR], d[BR];
    bool claim[BR];
    long long ev[BR];
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        z[r] = valid[r] ? ldg_cg(P.g.dst + x[r]) : skip;
        // push heights follow c_f(z, u) (backward); pull heights c_f(u, z) (forward)
        rc[r] = valid[r] ? (pull ? ldg_cg(P.cf + x[r]) : ldg_cg(P.g.pcap + x[r]) - ldg_cg(P.cf + x[r])) : 0;
    }
#pragma unroll
    for (int r = 0; r < BR; ++r) hz[r] = (rc[r] > 0 && z[r] != skip) ? ldg_cg(P.h + z[r]) : 0;
#pragma unroll
    for (int r = 0; r < BR; ++r) claim[r] = hz[r] == n && atomicCAS(P.h + z[r], n, L + 1) == n;
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        d[r] = claim[r] ? ldg_cg(P.g.deg + z[r]) : 0;
        const bool term = z[r] == P.sink || z[r] == P.source;
        ev[r] = (with_wl && claim[r] && !term) ? (pull ? -ldg_cg(P.e + z[r]) : ldg_cg(P.e + z[r])) : 0;
        if (near && claim[r]) {
            P.sc.par[z[r]] = ldg_cg(P.g.rev + x[r]);
            if (x[r] >= t0 && x[r] < t1) P.sc.dem[z[r]] = rc[r];     // z's own edge into the sink
        }
    }
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        if (!claim[r]) continue;
        ++lab;
        lab_slots += (unsigned)d[r];
        place_labelled(z[r], d[r], ev[r]);
    }
}

constexpr int kBR = 4;

__device__ __noinline__ void phase_bfs_level()
{
    MfSet *cs = sh.cs;
    const int L = sh.d.level;
    const int lane = threadIdx.x & 31;
    long long slots = 0;
    const int nctas = vn();
    int lab = 0;
    unsigned lab_slots = 0;
    const int nwarps = nctas * (int)(blockDim.x >> 5);
    // first the chunks of long rows, one per warp, then the regular frontier:
    // warps take up to 32 vertices at a time and expand their rows together
    // (each lane finds the entry that owns its slot).  A frontier of fewer is
    // dealt out evenly and at once, so that its rows spread over all warps and
    // nobody comes back for more (a level of 5116 vertices, one for each of 4864
    // warps and a rush of all of them on the head for the rest, took 19 us, one
    // of 4438 took 11).  One copy of the expansion serves both: the code of a
    // level has to come through the instruction cache before its few warps can
    // run it.
    const int ilo = sh.d.hub_lo, icnt = sh.d.hub_hi - ilo;
    const int lo = sh.d.lvl_lo, cnt = sh.d.lvl_hi - lo;
    const int take = max(1, min(32, (cnt + nwarps - 1) / nwarps));
    for (int kind = icnt > 0 ? 0 : 1; kind < 2; ++kind) {
        bool first = true;
        const int rank = warp_rank(nctas, kind ? icnt : 0);
        for (;;) {
            int d = 0, r0 = 0;
            if (kind == 0) {
                const int i = warp_deal(&cs->l[L_HEAD1].w[0], icnt, 1u, rank, nwarps, first);
                if (i >= icnt) break;
                if (lane == 0) {
                    const int2 it = __ldcg(P.sc.bitem + ilo + i);
                    r0 = it.x;
                    d = it.y;
                }
            } else {
                const int b = warp_deal(&cs->l[L_HEAD0].w[0], cnt, (unsigned)take, rank, nwarps, first);
                if (b >= cnt) break;
                const int idx = b + lane;
                const int u = (lane < take && idx < cnt) ? __ldcg(P.sc.border + lo + idx) : -1;
                d = u >= 0 ? ldg_cg(P.g.deg + u) : 0;
                r0 = u >= 0 ? P.g.off[u] : 0;
            }
            int incl = d;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int excl = incl - d;
            const int T = __shfl_sync(0xffffffffu, incl, 31);
            if (lane == 0) slots += T;
            for (int kb = 0; kb < T; kb += 32 * kBR) {
                int xs[kBR];
                bool vs[kBR];
#pragma unroll
                for (int r = 0; r < kBR; ++r) {
                    const int k = kb + r * 32 + lane;
                    int owner = 0;
#pragma unroll
                    for (int step = 16; step >= 1; step >>= 1) {
                        int cand = owner + step;
                        int ec = __shfl_sync(0xffffffffu, excl, cand & 31);
                        if (cand < 32 && ec <= k) owner = cand;
                    }
                    int rb = __shfl_sync(0xffffffffu, r0, owner);
                    int eb = __shfl_sync(0xffffffffu, excl, owner);
                    vs[r] = k < T;
                    xs[r] = rb + (k - eb);
                }
                bfs_visit<kBR>(xs, vs, L, lab, lab_slots);
            }
        }
    }
    add_stat(ST_SLOTS_BFS, slots);
    flush_labelled(lab, lab_slots);
}

// Near BFS, bottom-up: slot x = (v, z) with residual c leads v down to z at
// level L.  Several lanes may find a slot for the same v; any of them will do
// (there is one slot (v, sink) at most, so dem[v] fits par[v] either way).
__device__ __forceinline__ void note_parent(int v, int x, int z, int c, int L)
{
    P.sc.par[v] = x;
    if (L == 0 && z == P.sink) P.sc.dem[v] = c;
}

// A BFS level bottom-up (direction-optimising BFS): every unlabelled vertex v
// looks through its own row for a neighbour u of the current level with a
// residual edge towards it -- c_f(v, u) > 0, v's own slot, for the push
// heights; c_f(u, v) = pcap - c_f(v, u) for the pull heights -- and stops at
// the first one.  The labels equal the top-down level's (each vertex is
// labelled L + 1 exactly when it has such a neighbour); the work follows the
// unlabelled vertices' rows up to the first hit instead of the frontier's
// rows, which pays off once the frontier holds most of the graph.
__device__ __noinline__ void phase_bfs_bottom_up()
{
    MfSet *cs = sh.cs;
    const int n = P.g.n;
    const int L = sh.d.level;
    const bool pull = P.pull != 0;
    const int skip = pull ? P.sink : P.source;
    const bool with_wl = P.data_driven && !(P.mode & MF_M_BFS_ONLY);
    const int lane = threadIdx.x & 31;
    const long long gs = (long long)vn() * blockDim.x;
    // A warp takes 32 vertices.  Each unlabelled one first looks at kA slots of
    // its row alone; the rows still open after that are scanned by the whole
    // warp together, 128 slots per step over their concatenation (each lane
    // finds the row that owns its slot), and a row drops out of the scan as
    // soon as one of its slots finds a neighbour of level L.  Slots past
    // MF_BU_SCAN of a row go to the level's second pass as work items, so no
    // warp walks a very long row alone.
    constexpr int kA = 4;
    const int cap = P.sc.bdefer != nullptr ? MF_BU_SCAN : 0x7fffffff;
    const bool near = sh.d.near != 0;
    long long slots = 0, unl = 0;
    int lab = 0;
    unsigned lab_slots = 0;
    if (vb() == 0 && threadIdx.x == 0) add_stat(ST_HSCAN_BFS, n);    // every vertex's height is read
    for (long long base = (long long)vb() * blockDim.x + threadIdx.x - lane; base < n; base += gs) {
        const int v = (int)base + lane;
        const bool ok = v < n && v != skip;
        const int hv = ok ? ldg_cg(P.h + v) : 0;
        const int r0 = ok ? P.g.off[v] : 0;
        const int d = ok ? ldg_cg(P.g.deg + v) : 0;
        const bool open = ok && hv == n;
        bool take = false;
        if (open) {
            ++unl;
            int c[kA], z[kA];
#pragma unroll
            for (int r = 0; r < kA; ++r) {
                const int x = r0 + r;
                const bool in = r < d;
                c[r] = in ? (pull ? ldg_cg(P.g.pcap + x) - ldg_cg(P.cf + x) : ldg_cg(P.cf + x)) : 0;
                z[r] = in ? ldg_cg(P.g.dst + x) : 0;
            }
#pragma unroll
            for (int r = 0; r < kA; ++r) {
                const bool hitr = c[r] > 0 && ldg_cg(P.h + z[r]) == L;
                take |= hitr;
                if (near && hitr) note_parent(v, r0 + r, z[r], c[r], L);
            }
            slots += d < kA ? d : kA;
        }
        // the warp-cooperative scan of the rows still open
        const int lim = d < cap ? d : cap;
        const int rem = (open && !take && lim > kA) ? lim - kA : 0;
        int incl = rem;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int excl = incl - rem;
        const int T = __shfl_sync(0xffffffffu, incl, 31);
        const unsigned pend = __ballot_sync(0xffffffffu, rem > 0);
        unsigned hit = 0;
        for (int kb = 0; kb < T && (pend & ~hit) != 0; kb += 32 * kA) {
            int c[kA], z[kA], ow[kA], xs[kA];
#pragma unroll
            for (int r = 0; r < kA; ++r) {
                const int k = kb + r * 32 + lane;
                int owner = 0;
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1) {
                    const int cand = owner + step;
                    const int ec = __shfl_sync(0xffffffffu, excl, cand & 31);
                    if (cand < 32 && ec <= k) owner = cand;
                }
                const int rb = __shfl_sync(0xffffffffu, r0, owner);
                const int eb = __shfl_sync(0xffffffffu, excl, owner);
                const bool live = k < T && !((hit >> owner) & 1u);
                const int x = rb + kA + (k - eb);
                xs[r] = x;
                ow[r] = owner;
                c[r] = live ? (pull ? ldg_cg(P.g.pcap + x) - ldg_cg(P.cf + x) : ldg_cg(P.cf + x)) : 0;
                z[r] = live ? ldg_cg(P.g.dst + x) : 0;
                slots += live ? 1 : 0;
            }
            unsigned mine = 0;
#pragma unroll
            for (int r = 0; r < kA; ++r)
                if (c[r] > 0 && ldg_cg(P.h + z[r]) == L) {
                    mine |= 1u << ow[r];
                    if (near) note_parent((int)base + ow[r], xs[r], z[r], c[r], L);
                }
            hit |= __reduce_or_sync(0xffffffffu, mine);
        }
        if ((hit >> lane) & 1u) take = true;
        int nitem = 0, x0 = 0;
        if (take) {
            P.h[v] = L + 1;
            const long long ev = with_wl && v != P.sink && v != P.source ? (pull ? -ldg_cg(P.e + v) : ldg_cg(P.e + v)) : 0;
            ++lab;
            lab_slots += (unsigned)d;
            place_labelled(v, d, ev);
        } else if (open && d > lim) {
            nitem = (d - lim + MF_BU_CHUNK - 1) / MF_BU_CHUNK;
            x0 = r0 + lim;
        }
        if (__any_sync(0xffffffffu, nitem > 0)) {
            int ic = nitem;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, ic, o);
                if (lane >= o) ic += y;
            }
            const int tot = __shfl_sync(0xffffffffu, ic, 31);
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&cs->l[L_DEFER].w[0], (unsigned)tot);
            at = __shfl_sync(0xffffffffu, at, 0) + (unsigned)(ic - nitem);
            for (int cc = 0; cc < nitem; ++cc) P.sc.bdefer[at + cc] = make_int2(v, x0 + cc * MF_BU_CHUNK);
        }
    }
    add_stat(ST_SLOTS_BFS, slots);
    flush_labelled(lab, lab_slots);
    add_stat(ST_VERTS_BFS, unl);
}

// Second pass of a bottom-up level: the deferred chunks of long rows whose
// first MF_BU_SCAN slots held no neighbour of level L with a residual edge
// towards it.  One warp per chunk of MF_BU_CHUNK slots, 8 per lane; the first
// chunk of a row that finds one labels the vertex (a claim by CAS, as other
// chunks of the same row may find one too).
__device__ __noinline__ void phase_bfs_bottom_up_long()
{
    MfSet *cs = sh.cs;
    const int n = P.g.n;
    const int L = sh.d.level;
    const bool pull = P.pull != 0;
    const bool with_wl = P.data_driven && !(P.mode & MF_M_BFS_ONLY);
    const int lane = threadIdx.x & 31;
    const int cnt = sh.d.defer_n;
    const bool near = sh.d.near != 0;
    constexpr int kR = MF_BU_CHUNK / 32;
    long long slots = 0;
    int lab = 0;
    unsigned lab_slots = 0;
    const int nwarps = vn() * (int)(blockDim.x >> 5);
    const int rank = warp_rank(vn(), 0);
    bool first = true;
    for (;;) {
        const int i = warp_deal(&cs->l[L_HEAD1].w[0], cnt, 1u, rank, nwarps, first);
        if (i >= cnt) break;
        const int2 it = __ldcg(P.sc.bdefer + i);
        const int v = it.x;
        if (ldg_cg(P.h + v) != n) continue;       // another chunk of the row labelled it (same value in every lane)
        const int d = ldg_cg(P.g.deg + v);
        const int end = P.g.off[v] + d;
        const int len = end - it.y < MF_BU_CHUNK ? end - it.y : MF_BU_CHUNK;
        int c[kR], z[kR];
        bool hit = false;
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            const int j = r * 32 + lane;
            const int x = it.y + j;
            const bool ok = j < len;
            c[r] = ok ? (pull ? ldg_cg(P.g.pcap + x) - ldg_cg(P.cf + x) : ldg_cg(P.cf + x)) : 0;
            z[r] = ok ? ldg_cg(P.g.dst + x) : 0;
        }
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            const bool hitr = c[r] > 0 && ldg_cg(P.h + z[r]) == L;
            hit |= hitr;
            if (near && hitr) note_parent(v, it.y + r * 32 + lane, z[r], c[r], L);
        }
        if (lane == 0) slots += len;
        if (__any_sync(0xffffffffu, hit) && lane == 0 && atomicCAS(P.h + v, n, L + 1) == n) {
            const long long ev = with_wl && v != P.sink && v != P.source ? (pull ? -ldg_cg(P.e + v) : ldg_cg(P.e + v)) : 0;
            ++lab;
            lab_slots += (unsigned)d;
            place_labelled(v, d, ev);
        }
        __syncwarp();
    }
    add_stat(ST_SLOTS_BFS, slots);
    flush_labelled(lab, lab_slots);
}

// ---------------------------------------------------------------------------
// Worklist of active vertices (Sec. 5.2.1 O1) with the termination count
// ---------------------------------------------------------------------------

__device__ __noinline__ void phase_worklist()
{
    MfSet *cs = sh.cs;
    const int sel = sh.d.wl_sel;
    const int n = P.g.n;
    const int lane = threadIdx.x & 31;
    const long long gs = (long long)vn() * blockDim.x;
    for (long long base = (long long)vb() * blockDim.x + threadIdx.x - lane; base < n; base += gs) {
        int v = (int)base + lane;
        bool cand = v < n && v != P.sink && v != P.source;
        const long long ev = cand ? ldg_cg(P.e + v) : 0;
        bool act = cand && ldg_cg(P.h + v) < n && (P.pull ? ev < 0 : ev > 0);
        bool listed = P.data_driven ? act : cand;
        int bin = 0;
        if (listed) bin = row_bin(ldg_cg(P.g.deg + v));
        unsigned am = __ballot_sync(0xffffffffu, act);
        if (lane == 0 && am) atomicAdd(&cs->l[L_ACT].w[0], (unsigned)__popc(am));
#pragma unroll
        for (int b = 0; b < MF_NBIN; ++b) warp_append(&cs->l[L_WL + b].w[0], P.sc.wl[sel][b], listed && bin == b, v);
    }
}

// ---------------------------------------------------------------------------
// Discharge (Alg. 2)
// ---------------------------------------------------------------------------

// What a discharge round needs besides the graph: where vertices that become
// active are queued for the next round, and the stamps that keep each vertex
// at most once per round in that queue and once per iteration in the lists
// of remove-invalid-edges.
struct DisCtx {
    int nsel;        // worklist buffer of the next round
    int qstamp;      // stamp of this round's queue
    int fstamp;      // stamp of this iteration's remove-invalid lists
    bool queue;      // a next round follows, so queue newly active vertices
    MfSet *cs;       // this phase's counter set
    int fix0, fix1;  // where this round's entries of the remove-invalid lists start
};

// z just became active (its excess went from <= 0 to > 0 during this round):
// give it to the next round (Alg. 2's kernel checks e(u) > 0 on every cycle,
// so a vertex that receives flow while the kernel runs is discharged too).
__device__ __forceinline__ void enqueue_active(int z, const DisCtx &dc)
{
    const int dz = ldg_cg(P.g.deg + z);      // in flight together with the stamp exchange
    if (atomicExch(P.sc.vmark + z, dc.qstamp) == dc.qstamp) return;
    const int bin = row_bin(dz);
    const unsigned pos = atomicAdd(&dc.cs->l[L_AUX + bin].w[0], 1u);
    P.sc.wl[dc.nsel][bin][pos] = z;
}

// u still has something to move after its KERNEL_CYCLES cycles (excess for a
// push, a deficit for a pull) and a height below n: with P.requeue it joins the
// next round's queue too, instead of waiting for the next global relabel.
template <bool PULL>
__device__ __forceinline__ void requeue_if_active(int u, const DisCtx &dc)
{
    if (!P.requeue || !dc.queue) return;
    const long long eu = ldg_cg(P.e + u);
    if ((PULL ? eu < 0 : eu > 0) && ldg_cg(P.h + u) < P.g.n) enqueue_active(u, dc);
}

// u was relabelled: list it (once per iteration) for remove-invalid-edges;
// only relabelled vertices can have steep residual edges.
__device__ __forceinline__ void note_relabel(int u, const DisCtx &dc)
{
    if (atomicExch(P.sc.fixmark + u, dc.fstamp) == dc.fstamp) return;
    const int d = ldg_cg(P.g.deg + u);
    const int li = d > P.hub_deg ? 1 : 0;
    const unsigned pos = (li ? dc.fix1 : dc.fix0) + atomicAdd(&dc.cs->l[L_FIX + li].w[0], 1u);
    P.sc.fixl[li][pos] = u;
}

// Move amt > 0 along slot x = (u, z) of u, y = rev[x]: a push lowers c_f(u, z)
// (slot x), a pull (Sec. 5.2.2) lowers c_f(z, u) (slot y); e(z) changes by
// -/+ amt and z joins the next round's queue if that makes it active.  The
// caller updates e(u).  Only u's owner lowers the slot it moves through, so
// an amount read from that slot can always be moved.
template <bool PULL>
__device__ __forceinline__ void move_flow(int x, int y, int z, long long amt,
                                          const DisCtx &dc)
{
    if (PULL) {
        atomicSub(P.cf + y, (int)amt);
        atomicAdd(P.cf + x, (int)amt);
    } else {
        atomicSub(P.cf + x, (int)amt);
        atomicAdd(P.cf + y, (int)amt);
    }
    const long long dz = PULL ? -amt : amt;
    if (z == P.sink) {
        add_shared(sh.sink_e, dz);
    } else if (z == P.source) {
        add_shared(sh.src_e, dz);
    } else {
        const long long old = atomic_add_ll(P.e + z, dz);
        const bool became = PULL ? (old >= 0 && old + dz < 0) : (old <= 0 && old + dz > 0);
        if (dc.queue && became) enqueue_active(z, dc);
    }
}

// Residual of slot x in the direction of the move, from the slot's own row:
// c_f(u, z) for a push, c_f(z, u) = pcap - c_f(u, z) for a pull.
template <bool PULL>
__device__ __forceinline__ int residual_dir(int x)
{
    return PULL ? ldg_cg(P.g.pcap + x) - ldg_cg(P.cf + x) : ldg_cg(P.cf + x);
}

// The amount slot x of u can move now (exact): c_f(u, z) for a push, c_f(z, u) for a pull.
template <bool PULL>
__device__ __forceinline__ int movable(int x, int y)
{
    return PULL ? ldg_cg(P.cf + y) : ldg_cg(P.cf + x);
}

// Lowest residual neighbour over slots j = j0, j0 + step, ... (j < d) of the
// row at r0, as a key (h(v) << 32 | j) so the minimum also breaks ties by the
// lowest slot index.  Slots are read kU at a time with their loads issued
// together.
template <int kU, bool PULL>
__device__ __forceinline__ unsigned long long scan_lowest(int r0, int d, int j0, int step)
{
    unsigned long long best = kEmpty;
    for (int jb = j0; jb < d; jb += step * kU) {
        int c[kU], z[kU], hz[kU];
#pragma unroll
        for (int r = 0; r < kU; ++r) {
            int j = jb + r * step;
            // push: out-residual c_f(u, z); pull: in-residual c_f(z, u) = pcap - c_f(u, z)
            c[r] = j < d ? (PULL ? ldg_cg(P.g.pcap + r0 + j) - ldg_cg(P.cf + r0 + j) : ldg_cg(P.cf + r0 + j)) : 0;
            z[r] = j < d ? ldg_cg(P.g.dst + r0 + j) : 0;
        }
#pragma unroll
        for (int r = 0; r < kU; ++r) hz[r] = c[r] > 0 ? ldg_cg(P.h + z[r]) : 0;
#pragma unroll
        for (int r = 0; r < kU; ++r) {
            if (c[r] > 0) {
                unsigned long long key = ((unsigned long long)(unsigned)hz[r] << 32) | (unsigned)(jb + r * step);
                best = key < best ? key : best;
            }
        }
    }
    return best;
}

// Heights of a row's heads kept on chip for the cycles after the first scan:
// stg[j] = h(head of slot j) for a slot with residual capacity in the move's
// direction, kNoRes for the others.  A snapshot: heights only rise while the
// discharge runs and residuals of u's own slots only rise except through u's
// own moves (which update stg), so every candidate is checked against global
// memory before flow moves through it.  Slots that gain residual capacity
// meanwhile wait for the next discharge call.
constexpr int kNoRes = 0x7fffffff;

// KERNEL_CYCLES of Alg. 2 for a row of d slots: P.kernel_cycles, or with
// P.cycle_div > 0 at least d / P.cycle_div, so that a long row, whose first
// scan dominates its discharge, makes more of its pushes per scan.
__device__ __forceinline__ int cycles_for(int d)
{
    if (P.cycle_div <= 0) return P.kernel_cycles;
    const int k = d / P.cycle_div;
    return k > P.kernel_cycles ? k : P.kernel_cycles;
}
// push passes of one discharge call that may find only stale snapshot entries
// without using up a cycle (each such pass corrects at least one entry upward)
constexpr int kStaleMax = 8;

__device__ __forceinline__ int comp4(const int4 &a, int e)
{
    return e == 0 ? a.x : (e == 1 ? a.y : (e == 2 ? a.z : a.w));
}

// The first scan of a row: the lowest residual height as scan_lowest does, and the
// snapshot of every slot of the row in stg.  With 16-byte loads: rows start on
// multiples of four slots (MF_ROW_ALIGN), so slot group g (slots 4g .. 4g+3) is
// one int4 of each slot array.  Thread t of nt takes groups t, t + nt, ... two at
// a time (eight slots in flight).
template <bool PULL>
__device__ __forceinline__ unsigned long long scan_and_stage(int r0, int d, int t, int nt,
                                                                int *stg)
{
    unsigned long long best = kEmpty;
    const int ng = (d + 3) >> 2;
    const int4 *cf4 = reinterpret_cast<const int4 *>(P.cf + r0);
    const int4 *dst4 = reinterpret_cast<const int4 *>(P.g.dst + r0);
    const int4 *pc4 = reinterpret_cast<const int4 *>(P.g.pcap + r0);
    for (int g0 = t; g0 < ng; g0 += 2 * nt) {
        int4 c[2], z[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int g = g0 + q * nt;
            if (g < ng) {
                c[q] = __ldcg(cf4 + g);
                z[q] = __ldcg(dst4 + g);
                if (PULL) {
                    const int4 pc = __ldcg(pc4 + g);
                    c[q] = make_int4(pc.x - c[q].x, pc.y - c[q].y, pc.z - c[q].z, pc.w - c[q].w);
                }
            } else {
                c[q] = make_int4(0, 0, 0, 0);
                z[q] = make_int4(0, 0, 0, 0);
            }
        }
        int hz[8], res[8];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = 4 * (g0 + q * nt) + e;
                res[4 * q + e] = j < d ? comp4(c[q], e) : 0;
                hz[4 * q + e] = res[4 * q + e] > 0 ? ldg_cg(P.h + comp4(z[q], e)) : kNoRes;
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = 4 * (g0 + q * nt) + e;
                if (j < d) stg[j] = hz[4 * q + e];
                if (res[4 * q + e] > 0) {
                    const unsigned long long key = ((unsigned long long)(unsigned)hz[4 * q + e] << 32) | (unsigned)j;
                    best = key < best ? key : best;
                }
            }
        }
    }
    return best;
}

// Later scans: the lowest entry of the snapshot, from shared memory only.
__device__ __forceinline__ unsigned long long scan_staged(const int *stg, int d, int j0, int step)
{
    unsigned long long best = kEmpty;
    for (int j = j0; j < d; j += step) {
        const int hz = stg[j];
        if (hz != kNoRes) {
            const unsigned long long key = ((unsigned long long)(unsigned)hz << 32) | (unsigned)j;
            best = key < best ? key : best;
        }
    }
    return best;
}

// What slot x of u (row position j, snapshot entry *sj) can move now towards
// a head of height want: 0 unless the head still has that height and the slot
// still has residual capacity; the snapshot entry is corrected on the way.
template <bool PULL>
__device__ __forceinline__ int staged_amount(int x, int want, int &sj)
{
    const int hz = ldg_cg(P.h + ldg_cg(P.g.dst + x));
    if (hz != want) {
        sj = hz;
        return 0;
    }
    const int c = movable<PULL>(x, ldg_cg(P.g.rev + x));
    if (c <= 0) {
        sj = kNoRes;
        return 0;
    }
    return c;
}

// One thread per vertex (rows of at most small_deg slots).  Returns true
// if u was relabelled (only then can it have steep residual edges, Alg. 3).
// PULL: u is deficient and pulls (Sec. 5.2.2); its "excess" is -e(u).
// Rows of at most kTS slots keep the heads' heights in registers after the
// first scan.
template <bool PULL>
__device__ __noinline__ bool discharge_thread(int u, const DisCtx &dc)
{
    constexpr int kTS = 8;
    bool lifted = false;
    const int n = P.g.n;
    const int r0 = P.g.off[u];
    const int d = ldg_cg(P.g.deg + u);
    int hu = ldg_cg(P.h + u);
    long long scans = 0, moves = 0, fused = 0, gscan = 0;
    int cyc = 0;
    if (d <= kTS) {
        int hc[kTS];
        bool have = false;
        int stale = 0;
        while (cyc < P.kernel_cycles) {
            const long long eu = PULL ? -ldg_cg(P.e + u) : ldg_cg(P.e + u);
            if (!(hu < n && eu > 0)) break;
            ++scans;
            unsigned long long best = kEmpty;
            // the snapshot serves the pushes; a relabel is decided on fresh values
            // (a slot that gained residual capacity since the snapshot may be lower)
            for (int pass = 0; pass < 2; ++pass) {
                if (!have || pass == 1) {
                    int c[kTS], z[kTS];
#pragma unroll
                    for (int j = 0; j < kTS; ++j) {
                        c[j] = j < d ? residual_dir<PULL>(r0 + j) : 0;
                        z[j] = j < d ? ldg_cg(P.g.dst + r0 + j) : 0;
                    }
#pragma unroll
                    for (int j = 0; j < kTS; ++j) hc[j] = c[j] > 0 ? ldg_cg(P.h + z[j]) : kNoRes;
                    gscan += d;
                }
                const bool fresh = !have || pass == 1;
                have = true;
                best = kEmpty;
#pragma unroll
                for (int j = 0; j < kTS; ++j) {
                    if (hc[j] != kNoRes) {
                        const unsigned long long key = ((unsigned long long)(unsigned)hc[j] << 32) | (unsigned)j;
                        best = key < best ? key : best;
                    }
                }
                const int bh = best == kEmpty ? 0x7fffffff : (int)(best >> 32);
                if (fresh || !(best == kEmpty || hu <= bh)) break;
            }
            const int best_h = best == kEmpty ? 0x7fffffff : (int)(best >> 32);
            if (best == kEmpty || hu <= best_h) {
                // relabel (the relabel step of Alg. 2), then on to the pushes it makes admissible
                hu = (best == kEmpty || best_h >= n - 1) ? n : best_h + 1;
                P.h[u] = hu;
                lifted = true;
                add_stat(ST_RELABELS, 1);
                ++cyc;
                if (hu >= n || cyc >= P.kernel_cycles) continue;
            }
            // the cycles Alg. 2 would run next: the slots of height best_h in slot
            // order, each taking min(residual, what is left)
            long long rem = eu, sent = 0;
            int k = 0;
            const int jstart = (int)(best & 0xffffffffu);
#pragma unroll
            for (int j = 0; j < kTS; ++j) {
                if (j < jstart || j >= d || rem <= 0 || cyc + k >= P.kernel_cycles || hc[j] != best_h) continue;
                const int x = r0 + j;
                int sj = hc[j];
                const int c = staged_amount<PULL>(x, best_h, sj);
                hc[j] = sj;
                ++fused;
                if (c <= 0) continue;
                const long long a = rem < (long long)c ? rem : (long long)c;
                move_flow<PULL>(x, ldg_cg(P.g.rev + x), ldg_cg(P.g.dst + x), a, dc);
                if (a == c) hc[j] = kNoRes;
                rem -= a;
                sent += a;
                ++k;
            }
            if (sent) atomic_add_ll(P.e + u, PULL ? sent : -sent);
            moves += k;
            // a pass that found only stale entries corrected them and costs no cycle (bounded)
            if (k > 0) cyc += k;
            else if (++stale > kStaleMax) cyc += 1;
        }
    } else {
        while (cyc < P.kernel_cycles) {
            const long long eu = PULL ? -ldg_cg(P.e + u) : ldg_cg(P.e + u);
            if (!(hu < n && eu > 0)) break;
            ++scans;
            gscan += d;
            unsigned long long best = scan_lowest<4, PULL>(r0, d, 0, 1);
            int best_h = best == kEmpty ? 0x7fffffff : (int)(best >> 32);
            if (best == kEmpty || hu <= best_h) {
                hu = (best == kEmpty || best_h >= n - 1) ? n : best_h + 1;
                P.h[u] = hu;
                lifted = true;
                add_stat(ST_RELABELS, 1);
                ++cyc;
                if (hu >= n || cyc >= P.kernel_cycles) continue;
            }
            long long rem = eu, sent = 0;
            int k = 0;
            int j = (int)(best & 0xffffffffu);
            const int jstart = j;
            for (; j < d && rem > 0 && cyc + k < P.kernel_cycles; ++j) {
                const int x = r0 + j;
                if (residual_dir<PULL>(x) <= 0) continue;
                const int z = ldg_cg(P.g.dst + x);
                if (ldg_cg(P.h + z) != best_h) continue;
                const int y = ldg_cg(P.g.rev + x);
                const int c = movable<PULL>(x, y);
                if (c <= 0) continue;
                const long long a = rem < (long long)c ? rem : (long long)c;
                move_flow<PULL>(x, y, z, a, dc);
                rem -= a;
                sent += a;
                ++k;
            }
            if (sent) atomic_add_ll(P.e + u, PULL ? sent : -sent);
            moves += k;
            fused += j - jstart;
            cyc += k > 0 ? k : 1;
        }
    }
    if (scans) {
        add_stat(ST_CYCLES_DIS, scans);
        add_stat(ST_SLOTS_DIS, gscan + fused);
    }
    add_stat(ST_PUSHES, moves);
    return lifted;
}

// One warp per vertex; ST: the row's heads are kept in stg (this warp's slice
// of the on-chip snapshot) after the first scan.
template <bool PULL, bool ST>
__device__ __noinline__ bool discharge_warp_rows(int u, int d, const DisCtx &dc, int *stg)
{
    bool lifted = false;
    const int n = P.g.n;
    const int lane = threadIdx.x & 31;
    const int r0 = P.g.off[u];
    const int kcyc = cycles_for(d);
    constexpr bool st = ST;
    bool have = false;
    int stale = 0;
    int hu = ldg_cg(P.h + u);
    long long scans = 0, moves = 0, fused = 0, gscan = 0;
    int cyc = 0;
    while (cyc < kcyc) {
        const long long eu = PULL ? -ldg_cg(P.e + u) : ldg_cg(P.e + u);
        if (!(hu < n && eu > 0)) break;
        ++scans;
        unsigned long long best;
        if (!st) {
            best = warp_min_u64(scan_lowest<8, PULL>(r0, d, lane, 32));
            gscan += d;
        } else if (!have) {
            best = warp_min_u64(scan_and_stage<PULL>(r0, d, lane, 32, stg));
            have = true;
            gscan += d;
            __syncwarp();
        } else {
            best = warp_min_u64(scan_staged(stg, d, lane, 32));
            const int bh = best == kEmpty ? 0x7fffffff : (int)(best >> 32);
            if (best == kEmpty || hu <= bh) {
                // a relabel is decided on fresh values: refresh the snapshot first
                __syncwarp();
                best = warp_min_u64(scan_and_stage<PULL>(r0, d, lane, 32, stg));
                gscan += d;
                __syncwarp();
            }
        }
        int best_h = best == kEmpty ? 0x7fffffff : (int)(best >> 32);
        if (best == kEmpty || hu <= best_h) {
            // relabel, then straight on to the pushes it makes admissible
            hu = (best == kEmpty || best_h >= n - 1) ? n : best_h + 1;
            lifted = true;
            if (lane == 0) {
                P.h[u] = hu;
                add_stat(ST_RELABELS, 1);
            }
            ++cyc;
            if (hu >= n || cyc >= kcyc) {
                __syncwarp();
                continue;
            }
        }
        {
            // Alg. 2's next cycles, fused: the slots of height best_h in slot
            // order take min(residual, what is left); each step covers 8 * 32
            // slots, every lane 8 contiguous ones, with a warp prefix sum over
            // the lanes' totals.
            constexpr int kSeg = 8;
            const int j0 = (int)(best & 0xffffffffu);
            long long rem = eu, sent = 0;
            int k = 0;
            int seg = 1;    // one slot per lane first, kSeg after
            for (int jb = j0; jb < d && rem > 0 && cyc + k < kcyc; jb += seg * 32, seg = kSeg) {
                const int js = jb + lane * seg;
                int a[kSeg];
                long long tsum = 0;
                int tcnt = 0;
                if (st) {
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        const int j = js + r;
                        a[r] = (r < seg && j < d && stg[j] == best_h) ? 1 : 0;
                    }
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r]) {
                            int sj = stg[js + r];
                            a[r] = staged_amount<PULL>(r0 + js + r, best_h, sj);
                            stg[js + r] = sj;
                            ++fused;
                            tsum += a[r];
                            tcnt += a[r] > 0 ? 1 : 0;
                        }
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        a[r] = 0;
                        const int j = js + r;
                        if (r < seg && j < d && residual_dir<PULL>(r0 + j) > 0) a[r] = 1;
                    }
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r]) {
                            const int x = r0 + js + r;
                            a[r] = ldg_cg(P.h + ldg_cg(P.g.dst + x)) == best_h ? 1 : 0;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r]) {
                            const int x = r0 + js + r;
                            const int c = movable<PULL>(x, ldg_cg(P.g.rev + x));
                            a[r] = c > 0 ? c : 0;
                            tsum += a[r];
                            tcnt += a[r] > 0 ? 1 : 0;
                        }
                    }
                    fused += seg;
                }
                long long incl = tsum;
                int cincl = tcnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const long long t = __shfl_up_sync(0xffffffffu, incl, o);
                    const int tc = __shfl_up_sync(0xffffffffu, cincl, o);
                    if (lane >= o) {
                        incl += t;
                        cincl += tc;
                    }
                }
                long long off = incl - tsum;
                int coff = cincl - tcnt;
                long long mine = 0;
                int mk = 0;
                if (tcnt > 0 && off < rem && cyc + k + coff < kcyc) {
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r] <= 0) continue;
                        if (off < rem && cyc + k + coff < kcyc) {
                            const long long g = a[r] < rem - off ? a[r] : rem - off;
                            const int x = r0 + js + r;
                            move_flow<PULL>(x, ldg_cg(P.g.rev + x), ldg_cg(P.g.dst + x), g, dc);
                            if (st && g == a[r]) stg[js + r] = kNoRes;
                            mine += g;
                            ++mk;
                        }
                        off += a[r];
                        ++coff;
                    }
                }
                const long long tot = warp_sum_ll(mine);
                const int kk = (int)warp_sum_ll((long long)mk);
                rem -= tot;
                sent += tot;
                k += kk;
                __syncwarp();              // snapshot entries written above are read by other lanes next
            }
            if (lane == 0 && sent) atomic_add_ll(P.e + u, PULL ? sent : -sent);
            moves += k;
            // staged: a pass that found only stale entries corrected them and costs no cycle (bounded)
            if (k > 0) cyc += k;
            else if (!st || ++stale > kStaleMax) cyc += 1;
        }
        __syncwarp();
    }
    fused = warp_sum_ll(fused);
    if (lane == 0) {
        if (scans) {
            add_stat(ST_CYCLES_DIS, scans);
            add_stat(ST_SLOTS_DIS, gscan + fused);
        }
        add_stat(ST_PUSHES, moves);
    }
    return lifted;
}

// One warp per vertex (returns the same value in every lane).  stg: this
// warp's slice of the on-chip snapshot (wcap entries), used when the row fits.
template <bool PULL>
__device__ __forceinline__ bool discharge_warp(int u, const DisCtx &dc, int *stg, int wcap)
{
    const int d = ldg_cg(P.g.deg + u);
    if (stg != nullptr && d <= wcap) return discharge_warp_rows<PULL, true>(u, d, dc, stg);
    return discharge_warp_rows<PULL, false>(u, d, dc, nullptr);
}

// The threads that discharge one long row together: the whole CTA, or a group
// of MF_GROUP_WARPS warps (a quarter of the CTA, with its own named barrier and
// its own quarter of the snapshot), so that four rows of moderate length are
// discharged side by side.  tid: thread index in the team, n: its threads,
// w0 / nw: its first warp and warp count in the CTA, g: its broadcast slot.
struct CtaTeam {
    int tid, n, w0, nw, g;
    __device__ CtaTeam() : tid((int)threadIdx.x), n((int)blockDim.x), w0(0), nw((int)(blockDim.x >> 5)), g(0) {}
    __device__ void sync() const { __syncthreads(); }
};

struct GroupTeam {
    int tid, n, w0, nw, g;
    __device__ GroupTeam()
        : tid((int)threadIdx.x & (32 * MF_GROUP_WARPS - 1)), n(32 * MF_GROUP_WARPS),
          w0((int)(threadIdx.x >> 5) & ~(MF_GROUP_WARPS - 1)), nw(MF_GROUP_WARPS),
          g((int)threadIdx.x / (32 * MF_GROUP_WARPS))
    {
    }
    __device__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(n) : "memory"); }
};

// One team per vertex; ST: the row's heads are kept in stg (the team's share of
// the on-chip snapshot) after the first scan.
template <bool PULL, bool ST, class Team>
__device__ __noinline__ bool discharge_team_rows(int u, int d, const DisCtx &dc, int *stg)
{
    const Team T;
    bool lifted = false;
    const int n = P.g.n;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int r0 = P.g.off[u];
    const int kcyc = cycles_for(d);
    constexpr bool st = ST;
    bool have = false;
    int stale = 0;
    long long cand = 0;
    int cyc = 0;
    while (cyc < kcyc) {
        if (T.tid == 0) {
            sh.tb_e[T.g] = PULL ? -ldg_cg(P.e + u) : ldg_cg(P.e + u);
            sh.tb_h[T.g] = ldg_cg(P.h + u);
        }
        T.sync();
        const long long eu = sh.tb_e[T.g];
        const int hu = sh.tb_h[T.g];
        if (!(hu < n && eu > 0)) {
            T.sync();
            break;
        }
        unsigned long long best;
        bool global_scan = !st || !have;
        if (!st) best = scan_lowest<8, PULL>(r0, d, T.tid, T.n);
        else if (!have) best = scan_and_stage<PULL>(r0, d, T.tid, T.n, stg);
        else best = scan_staged(stg, d, T.tid, T.n);
        have = true;
        best = warp_min_u64(best);
        if (lane == 0) sh.red[wid] = best;
        T.sync();
        unsigned long long b = kEmpty;
        for (int w = T.w0; w < T.w0 + T.nw; ++w) b = sh.red[w] < b ? sh.red[w] : b;
        if (!global_scan && (b == kEmpty || hu <= (int)(b >> 32))) {
            // a relabel is decided on fresh values: refresh the snapshot first
            T.sync();               // every warp has read sh.red
            best = warp_min_u64(scan_and_stage<PULL>(r0, d, T.tid, T.n, stg));
            if (lane == 0) sh.red[wid] = best;
            T.sync();
            b = kEmpty;
            for (int w = T.w0; w < T.w0 + T.nw; ++w) b = sh.red[w] < b ? sh.red[w] : b;
            global_scan = true;
        }
        const int best_h = b == kEmpty ? 0x7fffffff : (int)(b >> 32);
        if (T.tid == 0) {
            add_stat(ST_CYCLES_DIS, 1);
            if (global_scan) add_stat(ST_SLOTS_DIS, d);
        }
        bool go = b != kEmpty && hu > best_h;
        if (!go) {
            // relabel, then straight on to the pushes it makes admissible
            const int nh = (b == kEmpty || best_h >= n - 1) ? n : best_h + 1;
            if (T.tid == 0) {
                P.h[u] = nh;
                add_stat(ST_RELABELS, 1);
            }
            lifted = true;
            ++cyc;
            go = nh < n && cyc < kcyc;
        }
        if (go) {
            // Alg. 2's next cycles, fused (as in discharge_warp): a step covers
            // seg * T.n slots, every thread seg contiguous ones, so slot
            // order is thread order and one team prefix sum over the threads'
            // totals orders all the amounts of the step.  The first step takes
            // one slot per thread (the excess often runs out there), later
            // ones kSeg.
            constexpr int kSeg = 8;
            const int j0 = (int)(b & 0xffffffffu);
            long long rem = eu;
            int k = 0;
            long long sent = 0;
            int seg = 1;
            for (int jb = j0; jb < d && rem > 0 && cyc + k < kcyc; jb += seg * T.n, seg = kSeg) {
                const int js = jb + T.tid * seg;
                int a[kSeg];
                long long tsum = 0;
                int tcnt = 0;
                if (st) {
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        const int j = js + r;
                        a[r] = (r < seg && j < d && stg[j] == best_h) ? 1 : 0;
                    }
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r]) {
                            int sj = stg[js + r];
                            a[r] = staged_amount<PULL>(r0 + js + r, best_h, sj);
                            stg[js + r] = sj;
                            ++cand;
                            tsum += a[r];
                            tcnt += a[r] > 0 ? 1 : 0;
                        }
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        a[r] = 0;
                        const int j = js + r;
                        if (r < seg && j < d && residual_dir<PULL>(r0 + j) > 0) a[r] = 1;   // candidate
                    }
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r]) {
                            const int x = r0 + js + r;
                            const int z = ldg_cg(P.g.dst + x);
                            a[r] = ldg_cg(P.h + z) == best_h ? 1 : 0;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r]) {
                            const int x = r0 + js + r;
                            const int c = movable<PULL>(x, ldg_cg(P.g.rev + x));
                            a[r] = c > 0 ? c : 0;
                            tsum += a[r];
                            tcnt += a[r] > 0 ? 1 : 0;
                        }
                    }
                    if (T.tid == 0)
                        add_stat(ST_SLOTS_DIS, seg * T.n);
                }
                long long incl = tsum;
                int cincl = tcnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const long long t = __shfl_up_sync(0xffffffffu, incl, o);
                    const int tc = __shfl_up_sync(0xffffffffu, cincl, o);
                    if (lane >= o) {
                        incl += t;
                        cincl += tc;
                    }
                }
                if (lane == 31) {
                    sh.wsum[wid] = incl;
                    sh.wcnt[wid] = cincl;
                }
                T.sync();
                long long off = incl - tsum;
                int coff = cincl - tcnt;
                for (int w = T.w0; w < wid; ++w) {
                    off += sh.wsum[w];
                    coff += sh.wcnt[w];
                }
                long long mine = 0;
                int mk = 0;
                if (tcnt > 0 && off < rem && cyc + k + coff < kcyc) {
#pragma unroll
                    for (int r = 0; r < kSeg; ++r) {
                        if (a[r] <= 0) continue;
                        if (off < rem && cyc + k + coff < kcyc) {
                            const long long g = a[r] < rem - off ? a[r] : rem - off;
                            const int x = r0 + js + r;
                            move_flow<PULL>(x, ldg_cg(P.g.rev + x), ldg_cg(P.g.dst + x), g, dc);
                            if (st && g == a[r]) stg[js + r] = kNoRes;
                            mine += g;
                            ++mk;
                        }
                        off += a[r];
                        ++coff;
                    }
                }
                const long long wt = warp_sum_ll(mine);
                const int wk = (int)warp_sum_ll((long long)mk);
                T.sync();               // every warp has read the prefix words
                if (lane == 0) {
                    sh.wsum[wid] = wt;
                    sh.wcnt[wid] = wk;
                }
                T.sync();
                long long tot = 0;
                int kk = 0;
                for (int w = T.w0; w < T.w0 + T.nw; ++w) {
                    tot += sh.wsum[w];
                    kk += sh.wcnt[w];
                }
                rem -= tot;
                sent += tot;
                k += kk;
                T.sync();               // before the words are reused
            }
            if (T.tid == 0) {
                if (sent) atomic_add_ll(P.e + u, PULL ? sent : -sent);
                add_stat(ST_PUSHES, k);
            }
            // staged: a pass that found only stale entries corrected them and costs no cycle (bounded)
            if (k > 0) cyc += k;
            else if (!st || ++stale > kStaleMax) cyc += 1;
        }
        T.sync();
    }
    if (cand) add_stat(ST_SLOTS_DIS, cand);
    return lifted;
}

// One CTA per vertex (hubs).  All threads of the CTA call this together;
// the return value is meaningful in thread 0.  stg: the CTA's on-chip
// snapshot (ccap entries), used when the row fits.
template <bool PULL>
__device__ __forceinline__ bool discharge_cta(int u, const DisCtx &dc, int *stg, int ccap)
{
    const int d = ldg_cg(P.g.deg + u);
    if (stg != nullptr && d <= ccap) return discharge_team_rows<PULL, true, CtaTeam>(u, d, dc, stg);
    return discharge_team_rows<PULL, false, CtaTeam>(u, d, dc, nullptr);
}

// One 4-warp group per vertex (rows up to group_deg slots, which fit the
// group's share of the snapshot).  All threads of the group call this
// together; the return value is meaningful in the group's thread 0.
template <bool PULL>
__device__ __forceinline__ bool discharge_group(int u, const DisCtx &dc, int *stg, int gcap)
{
    const int d = ldg_cg(P.g.deg + u);
    if (stg != nullptr && d <= gcap) return discharge_team_rows<PULL, true, GroupTeam>(u, d, dc, stg);
    return discharge_team_rows<PULL, false, GroupTeam>(u, d, dc, nullptr);
}

template <bool PULL>
__device__ __noinline__ void phase_discharge()
{
    MfSet *cs = sh.cs;
    const int lane = threadIdx.x & 31;
    const int sel = sh.d.wl_sel;
    DisCtx dc;
    dc.nsel = sel ^ 1;
    dc.qstamp = sh.d.qstamp;
    dc.fstamp = sh.d.fstamp;
    dc.cs = cs;
    dc.fix0 = sh.d.fix_n[0];
    dc.fix1 = sh.d.fix_n[1];
    // queue the vertices that become active for a next round if one may follow
    // (adaptive rounds: the hook decides after this round)
    dc.queue = sh.d.round + 1 < (P.rounds > 0 ? P.rounds : MF_MAX_ROUNDS);
    const int *wl0 = P.sc.wl[sel][0], *wl1 = P.sc.wl[sel][1], *wl2 = P.sc.wl[sel][2], *wl3 = P.sc.wl[sel][3];
    int *stage = P.stage_slots > 0 ? mf_stage : nullptr;
    const unsigned long long t_a = gtimer();
    // the longest rows: one CTA each
    const int nh = sh.d.wl_n[3];
    for (;;) {
        if (threadIdx.x == 0) {
            unsigned cur = *(volatile unsigned *)&cs->l[L_HEAD2].w[0];
            sh.bcast_i = (int)(cur >= (unsigned)nh ? cur : atomicAdd(&cs->l[L_HEAD2].w[0], 1u));
        }
        __syncthreads();
        int i = sh.bcast_i;
        __syncthreads();
        if (i >= nh) break;
        const int u = __ldcg(wl3 + i);
        const bool lifted = discharge_cta<PULL>(u, dc, stage, P.stage_slots);
        if (threadIdx.x == 0) {
            if (lifted) note_relabel(u, dc);
            requeue_if_active<PULL>(u, dc);
        }
    }
    // long rows up to group_deg: one 4-warp group each, four side by side per
    // CTA, each group on its own quarter of the snapshot buffer
    {
        const GroupTeam T;
        const int gcap = P.stage_slots / (MF_BLOCK / (32 * MF_GROUP_WARPS));
        int *gstage = stage != nullptr ? stage + T.g * gcap : nullptr;
        const int ng = sh.d.wl_n[2];
        for (;;) {
            if (T.tid == 0) {
                unsigned cur = *(volatile unsigned *)&cs->l[L_HEAD3].w[0];
                sh.tb_i[T.g] = (int)(cur >= (unsigned)ng ? cur : atomicAdd(&cs->l[L_HEAD3].w[0], 1u));
            }
            T.sync();
            const int i = sh.tb_i[T.g];
            T.sync();
            if (i >= ng) break;
            const int u = __ldcg(wl2 + i);
            const bool lifted = discharge_group<PULL>(u, dc, gstage, gcap);
            if (T.tid == 0) {
                if (lifted) note_relabel(u, dc);
                requeue_if_active<PULL>(u, dc);
            }
        }
    }
    const unsigned long long t_b = gtimer();
    if (lane == 0) add_stat(ST_NS_CTA, (long long)(t_b - t_a));
    // mid-degree rows: one warp each, on a slice of its own group's quarter of
    // the snapshot buffer (free once the group has left the loop above, while
    // the other groups may still be on their rows)
    const int nm = sh.d.wl_n[1];
    const int gq = P.stage_slots / (MF_BLOCK / (32 * MF_GROUP_WARPS));
    const int wcap = min(MF_WARP_STAGE, gq / MF_GROUP_WARPS);
    const int wid = (int)(threadIdx.x >> 5);
    int *wstage = stage != nullptr && wcap > 0
                      ? stage + (wid / MF_GROUP_WARPS) * gq + (wid % MF_GROUP_WARPS) * wcap : nullptr;
    for (;;) {
        const int i = warp_grab(&cs->l[L_HEAD1].w[0], nm, 1u);
        if (i >= nm) break;
        const int u = __ldcg(wl1 + i);
        const bool lifted = discharge_warp<PULL>(u, dc, wstage, wcap);
        if (lane == 0) {
            if (lifted) note_relabel(u, dc);
            requeue_if_active<PULL>(u, dc);
        }
    }
    const unsigned long long t_c = gtimer();
    // small rows: one thread each, 32 per grab
    const int ns = sh.d.wl_n[0];
    for (;;) {
        const int b = warp_grab(&cs->l[L_HEAD0].w[0], ns, 32u);
        if (b >= ns) break;
        if (b + lane < ns) {
            const int u = __ldcg(wl0 + b + lane);
            if (discharge_thread<PULL>(u, dc)) note_relabel(u, dc);
            requeue_if_active<PULL>(u, dc);
        }
    }
    __syncwarp();
    const unsigned long long t_d = gtimer();
    if (lane == 0) {
        // per warp, into the CTA's counters
        add_stat(ST_NS_WARP, (long long)(t_c - t_b));
        add_stat(ST_NS_THREAD, (long long)(t_d - t_c));
    }
}

// ---------------------------------------------------------------------------
// Short rounds and small phases
// ---------------------------------------------------------------------------
//
// On grids, geometric and layered graphs most BFS levels hold a few hundred
// vertices and most discharge rounds a few dozen, all with short rows.
//
// A short round (phase_discharge_short) gives each of its vertices one cycle of
// Alg. 2, on values read in that round: a chain of four dependent accesses
// (the vertex's state beside its row, the heads' heights, the receivers'
// excess), against KERNEL_CYCLES such chains in phase_discharge.  The flow
// moves one step per round either way, so the number of rounds hardly changes
// (grid 1024: 1172 rounds of one cycle, 1066 of two).
//
// What a smaller phase still costs across the grid is the barrier, the room
// taken in the shared lists and the counters behind it, about 9 us, not its
// work.  The squad -- the CTAs of the first thread-block cluster, or the first
// CTA of a launch without clusters -- runs consecutive small ones alone: each
// of its CTAs keeps the vertices it labelled or activated in a queue in its
// shared memory and takes them up in the next phase, the CTAs tell one another
// how many they have through distributed shared memory, and the cluster's
// barrier stands between the phases.  The other CTAs wait at one grid barrier,
// where they take the squad's state.  What bounds a phase there is a chain of
// three (level) or four (round) dependent accesses, and then the one scattered
// access per clock of each SM, some 14 per vertex.

// Whether the squad should go back to the grid: it has held up the others for a
// quarter of the longest wait at a barrier.
__device__ __forceinline__ bool squad_timeout(unsigned long long t0)
{
    return gtimer() - t0 > P.wait_limit_ns / 4;
}

// A squad CTA's queues: vertex, row start and row length of its entries.
struct SquadQ {
    int *v, *r, *d;
};
__device__ __forceinline__ SquadQ squad_q(int which)
{
    SquadQ q;
    q.v = mf_stage + which * MF_SQUAD_CAP;
    q.r = q.v + 2 * MF_SQUAD_CAP;
    q.d = q.r + 2 * MF_SQUAD_CAP;
    return q;
}
__device__ __forceinline__ void squad_put(const SquadQ &q, int i, int v, int r0, int d)
{
    q.v[i] = v;
    q.r[i] = r0;
    q.d[i] = d;
}

// bfs_visit for a level of the squad: labelled vertices go straight into this
// CTA's next queue.
template <int BR>
__device__ __forceinline__ void squad_visit(const int (&x)[BR], const bool (&valid)[BR],
                                            int L, const SquadQ &nq, int &lab, unsigned &lab_slots)
{
    const bool want_wl = sh.k_wl != 0, near = sh.d.near != 0;
    const int n = P.g.n;
    int z[BR], rc[BR], d[BR], r0[BR];
    bool claim[BR];
    long long ev[BR];
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        z[r] = valid[r] ? ldg_cg(P.g.dst + x[r]) : P.source;
        rc[r] = valid[r] ? ldg_cg(P.g.pcap + x[r]) - ldg_cg(P.cf + x[r]) : 0;
    }
#pragma unroll
    for (int r = 0; r < BR; ++r) claim[r] = rc[r] > 0 && z[r] != P.source && ldg_cg(P.h + z[r]) == n;
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        // in flight together with the claims
        d[r] = claim[r] ? ldg_cg(P.g.deg + z[r]) : 0;
        r0[r] = claim[r] ? P.g.off[z[r]] : 0;
        ev[r] = claim[r] && want_wl ? ldg_cg(P.e + z[r]) : 0;
        if (claim[r]) claim[r] = atomicCAS(P.h + z[r], n, L + 1) == n;
    }
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        if (!claim[r]) continue;
        ++lab;
        lab_slots += (unsigned)d[r];
        if (near) {
            const int y = ldg_cg(P.g.rev + x[r]);
            P.sc.par[z[r]] = y;
            if (L == 0 && ldg_cg(P.g.dst + y) == P.sink) P.sc.dem[z[r]] = rc[r];
        }
        if (d[r] > P.bfs_hub) {
            const int i = atomicAdd(&sh.so_long, 1);
            if (i < MF_SQUAD_LONG)
                mf_stage[6 * MF_SQUAD_CAP + i] = z[r];
            else
                put_items(r0[r], d[r], sh.d.app_hub + atomicAdd(&sh.cs->l[L_HUB].w[0], (unsigned)chunks_of(d[r])));
            sh.so_flag = SQ_SPILL;
        } else {
            const int i = atomicAdd(&sh.so_cnt, 1);
            if (i < MF_SQUAD_CAP) {
                squad_put(nq, i, z[r], r0[r], d[r]);
            } else {
                P.sc.border[sh.d.app_bfs + atomicAdd(&sh.cs->l[L_BFS].w[0], 1u)] = z[r];
                sh.so_flag = SQ_SPILL;
            }
        }
        if (ev[r] > 0 && z[r] != P.sink) {
            const int bin = row_bin(d[r]);
            P.sc.wl[sh.d.wl_sel][bin][sh.d.wl_app[bin] + atomicAdd(&sh.cs->l[L_WL + bin].w[0], 1u)] = z[r];
            if (near) add_shared(sh.exc, ev[r]);
        }
    }
}

// Top-down BFS levels, one after another, while they stay small.  The last one
// leaves its results where a level of the grid would, and the grid barrier that
// follows takes them up as that level's (with the squad's state).  False: a CTA of
// the squad is gone, and the caller leaves the kernel too.
__device__ __noinline__ bool squad_bfs()
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nwarps = nt >> 5;
    const int csize = sh.csize, rank = sh.crank;
    const unsigned long long t0 = gtimer();
    int cur = 0, cnt;
    squad_enter();
    {
        // entry i of the frontier belongs to squad CTA i mod csize
        const int lo = sh.d.lvl_lo, all = sh.d.lvl_hi - lo;
        cnt = all > rank ? (all - rank + csize - 1) / csize : 0;
        const SquadQ q = squad_q(0);
        for (int i = tid; i < cnt; i += nt) {
            const int v = __ldcg(P.sc.border + lo + i * csize + rank);
            squad_put(q, i, v, P.g.off[v], ldg_cg(P.g.deg + v));
        }
    }
    if (tid == 0) sh.so_cnt = sh.so_long = sh.so_flag = 0;
    __syncthreads();
    if (!squad_entered()) return false;
    for (;;) {
        const int L = sh.d.level, par = sh.so_par;
        const SquadQ cq = squad_q(cur), nq = squad_q(cur ^ 1);
        int lab = 0;
        unsigned lab_slots = 0;
        long long scanned = 0;
        const int take = max(1, min(32, (cnt + nwarps - 1) / nwarps));
        for (int b = wid * take; b < cnt; b += nwarps * take) {
            const bool in = lane < take && b + lane < cnt;
            const int d = in ? cq.d[b + lane] : 0, r0 = in ? cq.r[b + lane] : 0;
            int incl = d;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int excl = incl - d;
            const int T = __shfl_sync(0xffffffffu, incl, 31);
            scanned += T;
            for (int kb = 0; kb < T; kb += 32 * kBR) {
                int xs[kBR];
                bool vs[kBR];
#pragma unroll
                for (int r = 0; r < kBR; ++r) {
                    const int k = kb + r * 32 + lane;
                    int owner = 0;
#pragma unroll
                    for (int st = 16; st >= 1; st >>= 1) {
                        const int cand = owner + st;
                        const int ec = __shfl_sync(0xffffffffu, excl, cand & 31);
                        if (cand < 32 && ec <= k) owner = cand;
                    }
                    const int rb = __shfl_sync(0xffffffffu, r0, owner), eb = __shfl_sync(0xffffffffu, excl, owner);
                    vs[r] = k < T;
                    xs[r] = rb + (k - eb);
                }
                squad_visit<kBR>(xs, vs, L, nq, lab, lab_slots);
            }
        }
        __syncwarp();
        lab = __reduce_add_sync(0xffffffffu, lab);
        lab_slots = __reduce_add_sync(0xffffffffu, lab_slots);
        if (lane == 0) {
            if (lab) add_shared(sh.lab, ((long long)lab << 32) | lab_slots);
            add_stat(ST_SLOTS_BFS, scanned);
        }
        __syncthreads();
        if (wid == 0) {
            SquadSum mine{};
            mine.cnt = min(sh.so_cnt, MF_SQUAD_CAP);
            mine.slots = (unsigned)(sh.lab & 0xffffffffull);
            mine.labelled = (int)(sh.lab >> 32);
            mine.flag = sh.so_flag | (rank == 0 && squad_timeout(t0) ? SQ_STOP : 0);
            mine.exc = (long long)sh.exc;
            squad_tell(par, mine);
        }
        squad_sync();
        if (tid == 0) {
            // the same in every CTA of the squad
            MfDesc &d = sh.d;
            MfState &st = sh.hs;
            int c = 0, flag = 0;
            long long fr = 0, lab_n = 0, exc = 0;
            for (int q = 0; q < csize; ++q) {
                const SquadSum s = sh.sq[par][q];
                c += s.cnt;
                flag |= s.flag;
                fr += s.slots;
                lab_n += s.labelled;
                exc += s.exc;
            }
            const long long vis = st.vis_slots + fr, sup = st.sup + exc;
            const bool go = c > 0 && flag == 0 && squad_level(c, fr) &&
                            !turns_bottom_up(sh.k_alpha, sh.d.level + 1, fr, st.used_slots - vis) &&
                            !(d.near && sup > 0 && (sup >> st.cut_shift) >= st.dem);
            if (go) {
                // what advance() does for a level that is followed by another small one
                ++d.level;
                ++st.bfs_levels;
                st.vis_slots = vis;
                st.sup = sup;
                sh.stat[ST_LAB_BFS] += (long long)(sh.lab >> 32);
                sh.lab = sh.exc = 0;
            }
            sh.so_go = go ? 1 : 0;
            sh.so_par = par ^ 1;
        }
        __syncthreads();
        const int mine = min(sh.so_cnt, MF_SQUAD_CAP);
        cur ^= 1;
        if (!sh.so_go) {
            // the frontier goes onto the shared list
            int at = 0;
            if (tid == 0 && mine) sh.bcast_i = at = (int)atomicAdd(&sh.cs->l[L_BFS].w[0], (unsigned)mine);
            __syncthreads();
            at = sh.d.app_bfs + sh.bcast_i;
            for (int i = tid; i < mine; i += nt) P.sc.border[at + i] = squad_q(cur).v[i];
            write_long(mf_stage + 6 * MF_SQUAD_CAP, min(sh.so_long, MF_SQUAD_LONG));
            return true;
        }
        __syncthreads();
        if (tid == 0) sh.so_cnt = sh.so_flag = 0;
        cnt = mine;
        __syncthreads();
    }
}

// z received flow and became active, or stays active after its cycle: into the
// next round, once (by the stamp or for the reasons at short_push).  In the squad:
// into this CTA's queue, or, when that is full or z's row is long, onto the grid's
// lists; else into the CTA's queue of worklist entries.
template <bool SQUAD>
__device__ __forceinline__ void short_enqueue(int z, int r0, int d, const SquadQ &nq)
{
    if (!SQUAD) {
        if (sh.d.dis_stamp && atomicExch(P.sc.vmark + z, sh.d.qstamp) == sh.d.qstamp) return;
        place_active(z, d, L_AUX, sh.d.wl_sel ^ 1, nullptr);
        return;
    }
    if (d <= MF_SHORT_ROW) {
        const int i = atomicAdd(&sh.so_cnt, 1);
        if (i < MF_SQUAD_CAP) {
            squad_put(nq, i, z, r0, d);
            return;
        }
    }
    const int bin = row_bin(d);
    P.sc.wl[sh.d.wl_sel ^ 1][bin][atomicAdd(&sh.cs->l[L_AUX + bin].w[0], 1u)] = z;
    sh.so_flag = SQ_SPILL;
}

// g units along slot x = (u, z), y its reverse.  A round straight behind the BFS,
// or behind other such short rounds, needs no stamp to queue a receiver: its list
// holds every vertex once, and each with e > 0.  A listed vertex lowers its own
// excess once, by what it read at first, and queues itself if some is left; until
// then its excess is above zero and no receiver queues it, and after that it
// rises from zero at most once.  A vertex that is not listed never lowers its
// excess.  So everyone is queued once, with e > 0.
template <bool SQUAD>
__device__ __forceinline__ void short_push(int x, int z, int y, int g, const SquadQ &nq)
{
    atomicSub(P.cf + x, g);
    atomicAdd(P.cf + y, g);
    if (z == P.sink) {
        add_shared(sh.sink_e, g);
    } else if (z == P.source) {
        add_shared(sh.src_e, g);
    } else {
        const int d = ldg_cg(P.g.deg + z), r0 = SQUAD ? P.g.off[z] : 0;     // in flight together with the excess
        const long long old = atomic_add_ll(P.e + z, (long long)g);
        if (old <= 0 && old + g > 0) short_enqueue<SQUAD>(z, r0, d, nq);
    }
}

// u's new height when its lowest residual neighbour has height best (INT_MAX:
// none): Alg. 2's relabel if u is not above it.
__device__ __forceinline__ int short_lift(int u, int hu, int best, bool write)
{
    const int n = P.g.n;
    if (best < hu) return hu;
    const int nh = best >= n - 1 ? n : best + 1;
    if (write) {
        P.h[u] = nh;
        add_stat(ST_RELABELS, 1);
    }
    return nh;
}

// One cycle of Alg. 2 for u by one thread (rows of at most 8 slots): relabel if
// needed, then push to the lowest neighbours in slot order.
template <bool SQUAD>
__device__ __forceinline__ int short_thread(int u, int r0, int d, const SquadQ &nq)
{
    const int4 none = make_int4(0, 0, 0, 0);
    const long long eu = ldg_cg(P.e + u);
    int hu = ldg_cg(P.h + u);
    int z[8], c[8], hz[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const bool in = 4 * q < d;
        const int4 cf = in ? __ldcg(reinterpret_cast<const int4 *>(P.cf + r0) + q) : none;
        const int4 dz = in ? __ldcg(reinterpret_cast<const int4 *>(P.g.dst + r0) + q) : none;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            c[4 * q + k] = 4 * q + k < d ? comp4(cf, k) : 0;
            z[4 * q + k] = comp4(dz, k);
        }
    }
    if (eu <= 0 || hu >= P.g.n) return 0;
    int best = 0x7fffffff;
#pragma unroll
    for (int k = 0; k < 8; ++k) hz[k] = c[k] > 0 ? ldg_cg(P.h + z[k]) : 0x7fffffff;
#pragma unroll
    for (int k = 0; k < 8; ++k) best = min(best, hz[k]);
    hu = short_lift(u, hu, best, true);
    if (hu >= P.g.n) return 0;
    long long rem = eu;
    int pushes = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (hz[k] != best || rem <= 0) continue;
        const int g = rem < (long long)c[k] ? (int)rem : c[k];
        short_push<SQUAD>(r0 + k, z[k], ldg_cg(P.g.rev + r0 + k), g, nq);
        rem -= g;
        ++pushes;
    }
    const long long old = atomic_add_ll(P.e + u, rem - eu);
    if (old + rem - eu > 0) short_enqueue<SQUAD>(u, r0, d, nq);
    return pushes;
}

// The same by one warp (rows of up to MF_SHORT_ROW slots): every lane holds four
// slots of each 128, and a prefix sum over the lanes deals out the excess.
template <bool SQUAD>
__device__ __forceinline__ int short_warp(int u, int r0, int d, const SquadQ &nq)
{
    constexpr int kQ = MF_SHORT_ROW / 128;
    const int lane = threadIdx.x & 31;
    const int4 none = make_int4(0, 0, 0, 0);
    const long long eu = ldg_cg(P.e + u);
    int hu = ldg_cg(P.h + u);
    if (eu <= 0 || hu >= P.g.n) return 0;                 // the same in every lane
    int c[4 * kQ], hz[4 * kQ];
    int best = 0x7fffffff;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const int j = q * 128 + lane * 4;
        const bool in = j < d;
        const int4 cf = in ? __ldcg(reinterpret_cast<const int4 *>(P.cf + r0 + j)) : none;
        const int4 dz = in ? __ldcg(reinterpret_cast<const int4 *>(P.g.dst + r0 + j)) : none;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            c[4 * q + k] = j + k < d ? comp4(cf, k) : 0;
            hz[4 * q + k] = c[4 * q + k] > 0 ? ldg_cg(P.h + comp4(dz, k)) : 0x7fffffff;
        }
    }
#pragma unroll
    for (int k = 0; k < 4 * kQ; ++k) best = min(best, hz[k]);
    best = __reduce_min_sync(0xffffffffu, best);
    hu = short_lift(u, hu, best, lane == 0);
    if (hu >= P.g.n) return 0;
    long long mine = 0;
#pragma unroll
    for (int k = 0; k < 4 * kQ; ++k) mine += hz[k] == best ? c[k] : 0;
    long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const long long total = __shfl_sync(0xffffffffu, incl, 31);
    long long rem = eu - (incl - mine);                   // what is left when this lane's turn comes
    int pushes = 0;
#pragma unroll
    for (int k = 0; k < 4 * kQ; ++k) {
        if (hz[k] != best || rem <= 0) continue;
        const int g = rem < (long long)c[k] ? (int)rem : c[k];
        const int x = r0 + (k >> 2) * 128 + lane * 4 + (k & 3);
        short_push<SQUAD>(x, ldg_cg(P.g.dst + x), ldg_cg(P.g.rev + x), g, nq);
        rem -= g;
        ++pushes;
    }
    __syncwarp();
    pushes = __reduce_add_sync(0xffffffffu, pushes);
    if (lane == 0) {
        const long long sent = total < eu ? total : eu;
        const long long old = atomic_add_ll(P.e + u, -sent);
        if (old - sent > 0) short_enqueue<SQUAD>(u, r0, d, nq);
    }
    __syncwarp();
    return pushes;
}

// A discharge round of one cycle per vertex across the grid: a thread for a row
// of at most 8 slots, a warp for a longer one.
__device__ __noinline__ void phase_discharge_short()
{
    const int lane = threadIdx.x & 31;
    const int sel = sh.d.wl_sel, n0 = sh.d.wl_n[0], n1 = sh.d.wl_n[1], cnt = n0 + n1;
    const SquadQ none{};
    long long pushes = 0, slots = 0, scans = 0;
    for (long long k = spread_thread(); k < cnt; k += (long long)vn() * blockDim.x) {
        const int i = (int)k;
        const int u = __ldcg(i < n0 ? P.sc.wl[sel][0] + i : P.sc.wl[sel][1] + (i - n0));
        const int d = ldg_cg(P.g.deg + u), r0 = P.g.off[u];
        if (d > 8) continue;
        pushes += short_thread<false>(u, r0, d, none);
        slots += d;
        ++scans;
    }
    __syncwarp();
    const int lo = P.small_deg <= 8 ? n0 : 0;          // the first list holds rows of at most small_deg slots
    for (int i = lo + warp_rank(vn(), 0); i < cnt; i += vn() * (int)(blockDim.x >> 5)) {
        const int u = __ldcg(i < n0 ? P.sc.wl[sel][0] + i : P.sc.wl[sel][1] + (i - n0));
        const int d = ldg_cg(P.g.deg + u), r0 = P.g.off[u];
        if (d <= 8) continue;
        const int p = short_warp<false>(u, r0, d, none);
        if (lane == 0) {
            pushes += p;
            slots += d;
            ++scans;
        }
    }
    add_stat(ST_PUSHES, pushes);
    add_stat(ST_SLOTS_DIS, slots);
    add_stat(ST_CYCLES_DIS, scans);
    flush_queue(L_AUX, sel ^ 1, nullptr, 0, 0u);
}

// Discharge rounds, one after another, while few vertices are active.  The last
// one leaves its results where a round of the grid would.  False as squad_bfs.
__device__ __noinline__ bool squad_discharge()
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
    const int csize = sh.csize, rank = sh.crank;
    const unsigned long long t0 = gtimer();
    int cur = 0, cnt;
    squad_enter();
    {
        const int sel = sh.d.wl_sel, n0 = sh.d.wl_n[0], all = n0 + sh.d.wl_n[1];
        const bool stamped = sh.d.dis_stamp != 0;
        if (tid == 0) sh.so_cnt = 0;
        __syncthreads();
        cnt = all > rank ? (all - rank + csize - 1) / csize : 0;
        const SquadQ q = squad_q(0);
        for (int i = tid; i < cnt; i += nt) {
            const int k = i * csize + rank;
            const int v = __ldcg(k < n0 ? P.sc.wl[sel][0] + k : P.sc.wl[sel][1] + (k - n0));
            const int r0 = P.g.off[v], d = ldg_cg(P.g.deg + v);
            if (!stamped) squad_put(q, i, v, r0, d);
            else if (ldg_cg(P.e + v) > 0) squad_put(q, atomicAdd(&sh.so_cnt, 1), v, r0, d);
        }
        __syncthreads();
        if (stamped) cnt = sh.so_cnt;
        __syncthreads();
        if (tid == 0) sh.so_cnt = sh.so_flag = sh.d.dis_stamp = 0;
        __syncthreads();
        if (!squad_entered()) return false;
        // without the vertices that have no excess the list is as a short round
        // wants it, and no stamps are needed; nobody pushes before every CTA of
        // the squad has looked
        if (stamped) squad_sync();
    }
    for (;;) {
        const int par = sh.so_par;
        const SquadQ cq = squad_q(cur), nq = squad_q(cur ^ 1);
        long long slots = 0, pushes = 0, scans = 0;
        for (int i = tid; i < cnt; i += nt) {
            const int d = cq.d[i];
            if (d > 8) continue;
            pushes += short_thread<true>(cq.v[i], cq.r[i], d, nq);
            slots += d;
            ++scans;
        }
        __syncwarp();
        for (int i = wid; i < cnt; i += nt >> 5) {
            const int d = cq.d[i];
            if (d <= 8) continue;
            const int p = short_warp<true>(cq.v[i], cq.r[i], d, nq);
            if (lane == 0) {
                pushes += p;
                slots += d;
                ++scans;
            }
        }
        add_stat(ST_PUSHES, pushes);
        add_stat(ST_SLOTS_DIS, slots);
        add_stat(ST_CYCLES_DIS, scans);
        __syncthreads();
        if (wid == 0) {
            SquadSum mine{};
            mine.cnt = min(sh.so_cnt, MF_SQUAD_CAP);
            mine.flag = sh.so_flag;
            if (rank == 0) {
                const unsigned long long now = gtimer();
                if (sh.d.round + 1 >= MF_DEFAULT_ROUNDS && !rounds_left(sh.d, sh.hs, now)) mine.flag |= SQ_OVER;
                if (squad_timeout(t0)) mine.flag |= SQ_STOP;
            }
            squad_tell(par, mine);
        }
        squad_sync();
        if (tid == 0) {
            // the same in every CTA of the squad
            int c = 0, flag = 0;
            for (int q = 0; q < csize; ++q) {
                c += sh.sq[par][q].cnt;
                flag |= sh.sq[par][q].flag;
            }
            const bool over = c == 0 || (flag & SQ_OVER) || sh.d.round + 1 >= MF_MAX_ROUNDS;
            sh.so_go = over ? 0 : (flag != 0 || c > MF_SQUAD_ACTIVE * csize ? 2 : 1);
            if (sh.so_go == 1) {
                ++sh.d.round;
                ++sh.hs.rounds_total;
            }
            sh.so_par = par ^ 1;
        }
        __syncthreads();
        const int go = sh.so_go, mine = min(sh.so_cnt, MF_SQUAD_CAP);
        cur ^= 1;
        if (go != 1) {
            // more rounds, but not here: the queue goes onto the grid's lists
            // (what is left when the discharge is over waits for the next BFS)
            if (go == 2) {
                for (int i = tid; i < mine; i += nt) {
                    const int bin = row_bin(nq.d[i]);
                    P.sc.wl[sh.d.wl_sel ^ 1][bin][atomicAdd(&sh.cs->l[L_AUX + bin].w[0], 1u)] = nq.v[i];
                }
            }
            return true;
        }
        __syncthreads();
        if (tid == 0) sh.so_cnt = sh.so_flag = 0;
        cnt = mine;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Near iterations: the excess walks down the BFS forest
// ---------------------------------------------------------------------------

// Take up to a from the residual of slot y; returns what was there to take.
// One subtraction, and what was not there is given back: other walkers see less
// than there is meanwhile, never more.  Large residuals go by compare and swap,
// because the overdraft of all walkers at once has to stay within int32 (at
// most 2^18 threads times MF_NEAR_SUB = 2^13).
__device__ __forceinline__ int draw(int *cf, long long a)
{
    int c = ldg_cg(cf);
    if (c <= 0) return 0;
    if (c <= MF_NEAR_SUB) {
        const int g = a < c ? (int)a : c;
        const int old = atomicSub(cf, g);
        const int got = old >= g ? g : (old > 0 ? old : 0);
        if (got < g) atomicAdd(cf, g - got);
        return got;
    }
    for (;;) {
        const int g = a < c ? (int)a : c;
        const int old = atomicCAS(cf, c, c - g);
        if (old == c) return g;
        c = old;
        if (c <= 0) return 0;
    }
}

// One thread per active vertex.  It climbs the BFS forest to its root -- a
// deficient vertex, or the neighbour through which its tree enters the sink --
// reserves there what the root can still take, and carries that much down,
// parent by parent; where an edge holds less, the rest stays as that vertex's
// excess.  Heights do not change meanwhile, every step goes from height k to
// k - 1 along residual capacity, so these are pushes Alg. 2 could make.
//
// What bounds it is one chain of dependent accesses per step (parent slot, its
// head and reverse, the residual's atomic), a few steps long, with every
// active vertex under way at once.  A discharge round over the same vertices
// scans their whole rows: on R-MAT 20 with 10 K updates two rounds read some
// 5 M slots of hub rows and took 120-190 us, the walks take about 10 us.
__device__ __noinline__ void phase_walk()
{
    const int sel = sh.d.wl_sel;
    DisCtx dc;
    dc.nsel = sel ^ 1;
    dc.qstamp = sh.d.qstamp;
    dc.fstamp = sh.d.fstamp;
    dc.cs = sh.cs;
    dc.fix0 = dc.fix1 = 0;
    dc.queue = !sh.d.cut;      // discharge rounds may follow a complete relabel
    int n0 = sh.d.wl_n[0], n1 = n0 + sh.d.wl_n[1], n2 = n1 + sh.d.wl_n[2], total = n2 + sh.d.wl_n[3];
    long long pushes = 0;
    for (long long i = spread_thread(); i < total; i += (long long)vn() * blockDim.x) {
        const int k = (int)i;
        const int u = __ldcg(k < n0 ? P.sc.wl[sel][0] + k
                                    : (k < n1 ? P.sc.wl[sel][1] + (k - n0)
                                              : (k < n2 ? P.sc.wl[sel][2] + (k - n1) : P.sc.wl[sel][3] + (k - n2))));
        const long long eu = ldg_cg(P.e + u);
        if (eu <= 0) continue;
        int root = u;
        for (;;) {
            const int w = ldg_cg(P.g.dst + ldg_cg(P.sc.par + root));
            if (w == P.sink) break;
            const bool top = ldg_cg(P.h + w) == 0;
            root = w;
            if (top) break;
        }
        long long a = ldg_cg(P.sc.dem + root);
        a = a < eu ? a : eu;
        if (a > 0) {
            const long long old = atomic_add_ll(P.sc.dem + root, -a);
            const long long got = old >= a ? a : (old > 0 ? old : 0);
            if (got < a) atomic_add_ll(P.sc.dem + root, a - got);
            a = got;
        }
        if (a <= 0) {
            if (dc.queue) enqueue_active(u, dc);
            continue;
        }
        atomic_add_ll(P.e + u, -a);
        if (dc.queue && eu > a) enqueue_active(u, dc);
        int v = u;
        do {
            const int y = ldg_cg(P.sc.par + v);
            const int w = ldg_cg(P.g.dst + y), r = ldg_cg(P.g.rev + y);
            const int g = draw(P.cf + y, a);
            if (g > 0) {
                atomicAdd(P.cf + r, g);
                ++pushes;
            }
            if (g < a) {
                atomic_add_ll(P.e + v, a - g);
                if (dc.queue) enqueue_active(v, dc);
            }
            a = g;
            v = w;
        } while (a > 0 && v != P.sink && ldg_cg(P.h + v) > 0);
        if (a > 0) add_excess(v, a);
    }
    add_stat(ST_PUSHES, pushes);
}

// ---------------------------------------------------------------------------
// Remove invalid edges (Alg. 3)
// ---------------------------------------------------------------------------

// Alg. 3 on slots j = j0, j0 + step, ... of u's row: push the whole residual
// of every steep slot (h(u) > h(v) + 1).  Returns the flow sent out of u.
// Only vertices relabelled in the discharge can have steep slots (heights are
// exact after the BFS and neighbours only rise), so only those are scanned.
// PULL (Sec. 5.2.2): a steep in-residual c_f(v, u) is pulled whole, and the
// return value is minus the flow received.
template <bool PULL>
__device__ __forceinline__ long long fix_scan(int hu, int r0, int d, int j0, int step)
{
    constexpr int kF = 4;
    long long out = 0;
    for (int jb = j0; jb < d; jb += step * kF) {
        int c[kF], z[kF], hz[kF];
#pragma unroll
        for (int r = 0; r < kF; ++r) {
            const int j = jb + r * step;
            c[r] = j < d ? (PULL ? ldg_cg(P.g.pcap + r0 + j) - ldg_cg(P.cf + r0 + j) : ldg_cg(P.cf + r0 + j)) : 0;
            z[r] = j < d ? ldg_cg(P.g.dst + r0 + j) : 0;
        }
#pragma unroll
        for (int r = 0; r < kF; ++r) hz[r] = c[r] > 0 ? ldg_cg(P.h + z[r]) : 0x7fffffff;
#pragma unroll
        for (int r = 0; r < kF; ++r) {
            if (c[r] > 0 && hu > hz[r] + 1) {
                const int x = r0 + jb + r * step;
                if (PULL) {
                    const int y = ldg_cg(P.g.rev + x);
                    const int old = atomicExch(P.cf + y, 0);
                    if (old > 0) {
                        atomicAdd(P.cf + x, old);
                        add_excess(z[r], -(long long)old);
                        add_stat(ST_STEEP, 1);
                        out -= old;
                    }
                } else {
                    const int old = atomicExch(P.cf + x, 0);
                    if (old > 0) {
                        atomicAdd(P.cf + ldg_cg(P.g.rev + x), old);
                        add_excess(z[r], (long long)old);
                        add_stat(ST_STEEP, 1);
                        out += old;
                    }
                }
            }
        }
    }
    return out;
}

template <bool PULL>
__device__ __noinline__ void phase_fix()
{
    MfSet *cs = sh.cs;
    const int lane = threadIdx.x & 31;
    long long slots = 0, verts = 0;
    // rows above hub_deg: one CTA each
    const int nh = sh.d.fix_n[1];
    for (;;) {
        if (threadIdx.x == 0) {
            unsigned cur = *(volatile unsigned *)&cs->l[L_HEAD2].w[0];
            sh.bcast_i = (int)(cur >= (unsigned)nh ? cur : atomicAdd(&cs->l[L_HEAD2].w[0], 1u));
        }
        __syncthreads();
        int i = sh.bcast_i;
        __syncthreads();
        if (i >= nh) break;
        const int u = __ldcg(P.sc.fixl[1] + i);
        const int hu = ldg_cg(P.h + u);
        const int r0 = P.g.off[u], d = ldg_cg(P.g.deg + u);
        long long out = fix_scan<PULL>(hu, r0, d, threadIdx.x, blockDim.x);
        if (out) atomic_add_ll(P.e + u, -out);
        if (threadIdx.x == 0) { slots += d; ++verts; }
    }
    // the others: one warp each
    const int nw = sh.d.fix_n[0];
    for (;;) {
        const int i = warp_grab(&cs->l[L_HEAD1].w[0], nw, 1u);
        if (i >= nw) break;
        const int u = __ldcg(P.sc.fixl[0] + i);
        const int hu = ldg_cg(P.h + u);
        const int r0 = P.g.off[u], d = ldg_cg(P.g.deg + u);
        long long out = warp_sum_ll(fix_scan<PULL>(hu, r0, d, lane, 32));
        if (lane == 0) {
            if (out) atomic_add_ll(P.e + u, -out);
            slots += d;
            ++verts;
        }
    }
    add_stat(ST_SLOTS_FIX, slots);
    add_stat(ST_VERTS_FIX, verts);
}

// ---------------------------------------------------------------------------
// Value (Alg. 5 last lines, reading R3)
// ---------------------------------------------------------------------------

__device__ __noinline__ void phase_value()
{
    // push (R3): sum of e(v) over v != s with h(v) < n; pull (Sec. 5.2.2, the
    // mirror): sum of -e(v) over v != t with h(v) < n
    const int n = P.g.n;
    const bool pull = P.pull != 0;
    const int skip = pull ? P.sink : P.source;
    long long acc = 0;
    for (long long v = (long long)vb() * blockDim.x + threadIdx.x; v < n; v += (long long)vn() * blockDim.x)
        if ((int)v != skip && ldg_cg(P.h + v) < n) acc += pull ? -ldg_cg(P.e + v) : ldg_cg(P.e + v);
    acc = warp_sum_ll(acc);
    if ((threadIdx.x & 31) == 0 && acc) add_shared(sh.value, acc);
}

// One whole solve of one instance by the vn() CTAs of the caller: the
// optional static initialisation or batch repair, the push-relabel loop and
// the value.  Returns false only if this CTA gave up waiting at a barrier
// (the caller must then leave the kernel); every other exit is taken by all
// CTAs together.
__device__ __noinline__ bool solve_instance()
{
    __syncthreads();          // the parameters are in shared memory
    if (threadIdx.x < MF_STATS) sh.stat[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        MfCtrl *c = P.ctrl;
        sh.sink_e = sh.src_e = sh.value = sh.ft_cap = 0;
        sh.ft_s = sh.ft_t = sh.ft_del = 0;
        sh.action = -1;
        sh.lab = sh.exc = sh.dem = 0;
        sh.q_bfs = sh.q_long = sh.q_wn = 0;
        for (int b = 0; b < MF_NBIN; ++b) sh.q_wl[b] = 0;
        sh.phase = 0;
        sh.arrivals = 0;
        const int cs = (int)cluster_size();
        sh.csize = cs > 1 && cs <= MF_CLUSTER && vn() % cs == 0 ? cs : 1;
        sh.crank = sh.csize > 1 ? (int)cluster_rank() : 0;
        sh.one_cluster = sh.csize > 1 && vn() == sh.csize && P.test_skip_cta < 0 ? 1 : 0;
        sh.so_par = 0;
        sh.cs = &c->set[0];
        sh.d = MfDesc{};
        sh.hs = MfState{};
        sh.d.qstamp = __ldcg(&c->qstamp);
        sh.d.fstamp = __ldcg(&c->fstamp);
        sh.d.near = near_allowed();
        sh.k_alpha = P.bu_alpha;
        sh.k_beta = P.bu_beta;
        sh.k_wl = P.data_driven && !(P.mode & MF_M_BFS_ONLY) ? 1 : 0;
        sh.k_squad = P.pull || P.stage_slots < MF_SQUAD_INTS ? 0 : (P.tail_slots >= 0 ? P.tail_slots : MF_SQUAD_SLOTS * sh.csize);
        sh.hs.t_phase = gtimer();
    }
    if (vb() == 0) {
        // results start at zero; the other CTAs add to them at the end of the launch
        MfCtrl *c = P.ctrl;
        if (threadIdx.x < MF_STATS) c->stat[threadIdx.x] = 0;
        if (threadIdx.x == 0) {
            c->value = 0;
            P.rep->t_entry = gtimer();
        }
    }
    __syncthreads();
    // a CTA that never arrives (tests only): the others give up after
    // wait_limit_ns, record MF_E_WAIT and leave the kernel
    if (P.test_skip_cta == vb()) return true;

    const bool loops = (P.mode & (MF_M_SOLVE | MF_M_BFS_ONLY)) != 0;
    bool opened = false;      // the last barrier opened the first iteration
    if (P.mode & MF_M_STATIC_INIT) {
        const bool sat = !(P.mode & MF_M_NO_SRC_SAT), sink = (P.mode & MF_M_SAT_SINK) != 0;
        phase_static_reset();
        if (!grid_sync(sat || sink || !loops ? H_NONE : H_ITER)) return false;
        if (sat) {
            phase_saturate_source();
            if (!grid_sync(sink || !loops ? H_NONE : H_ITER)) return false;
        }
        if (sink) {
            phase_saturate_sink();
            if (!grid_sync(loops ? H_ITER : H_NONE)) return false;
        }
        opened = loops;
    }
    if (P.mode & MF_M_APPLY) {
        phase_apply_validate();
        if (!grid_sync(H_APPLY_VALID)) return false;
        if (sh.d.status != MF_ST_RUNNING) {
            phase_apply_cleanup(false);
            return finish();
        }
        // the last CTA asks the network while the others locate the slots
        const int finders = (P.mode & MF_M_SCHED) && vn() > 1 ? vn() - 1 : vn();
        if ((P.mode & MF_M_SCHED) && vb() == vn() - 1) pick_action();
        if (vb() < finders) phase_apply_locate(finders);
        if (!grid_sync(H_APPLY_LOCATED)) return false;
        if (sh.d.status != MF_ST_RUNNING) {
            // a row overflow keeps the rows' demand for the rebuild that follows;
            // a refused batch (pair sum) leaves nothing behind
            phase_apply_cleanup(sh.hs.err == MF_E_OVERFLOW);
            return finish();
        }
        phase_apply_change();
        if (!grid_sync(H_APPLY_DELTA)) return false;
        // the source step reads the final residuals; the tables are cleared beside it
        phase_apply_cleanup(false);
        if (!(P.mode & MF_M_SKIP_SOURCE_SAT) && !sh.d.resolve) phase_resaturate();
        if (sh.d.resolve) {
            // the picked action re-solves the changed graph from zero flow
            if (!grid_sync(H_NONE)) return false;
            phase_static_reset();
            if (!grid_sync(H_NONE)) return false;
            phase_saturate_source();
        }
        // straight on to the loop: this barrier opens its first iteration
        opened = loops && !(P.mode & MF_M_CUT);
        if (!opened && !(P.mode & MF_M_CUT) && !loops) return finish();
        if (!grid_sync(opened ? H_ITER : H_NONE)) return false;
        if (P.mode & MF_M_CUT) {
            phase_cut_side();
            if (!grid_sync(H_NONE)) return false;
            phase_saturate_cut();
            if (!grid_sync(H_NONE)) return false;
        }
        if (sh.d.status != MF_ST_RUNNING) return finish();
    }
    if (!loops) return finish();

    if (!opened && !grid_sync(H_ITER)) return false;
    for (;;) {
        // backward BFS
        phase_bfs_init();
        if (!grid_sync(H_BFS_START)) return false;
        while (!sh.d.bfs_done) {
            if (sh.d.bfs_squad) {
                // the others wait at the grid barrier and take the squad's state there
                if (vb() < sh.csize && !squad_bfs()) return false;
                if (!grid_sync(H_BFS_NEXT, true)) return false;
                continue;
            }
            if (sh.d.bu_mode) {
                phase_bfs_bottom_up();
                if (!grid_sync(H_BU_SPLIT)) return false;     // ends the level if nothing was deferred
                if (sh.d.bu_split) {
                    phase_bfs_bottom_up_long();
                    if (!grid_sync(H_BFS_NEXT)) return false;
                }
            } else {
                phase_bfs_level();
                if (!grid_sync(H_BFS_NEXT)) return false;
            }
        }
        if (P.mode & MF_M_BFS_ONLY) return finish();
        // worklist and termination test (built during the BFS when data-driven)
        if (!P.data_driven) {
            phase_worklist();
            if (!grid_sync(H_WL)) return false;
        }
        if (sh.d.status != MF_ST_RUNNING) break;
        // discharge rounds, then remove-invalid-edges
        do {
            if (sh.d.dis_squad) {
                if (vb() < sh.csize && !squad_discharge()) return false;
                if (!grid_sync(H_DIS, true)) return false;
                continue;
            }
            if (sh.d.near && sh.d.round == 0) phase_walk();
            else if (sh.d.dis_short) phase_discharge_short();
            else if (P.pull) phase_discharge<true>();
            else phase_discharge<false>();
            if (!grid_sync(H_DIS)) return false;
        } while (sh.d.dis_more);
        if (P.fix_steep) {
            if (P.pull) phase_fix<true>();
            else phase_fix<false>();
            if (!grid_sync(H_ITER)) return false;
        }
    }
    if (sh.d.status != MF_ST_ERROR && !(P.mode & MF_M_NO_VALUE)) phase_value();
    return finish();
}

__global__ void __launch_bounds__(MF_BLOCK, 2) mf_solve_kernel(const __grid_constant__ MfParams params)
{
    for (int i = threadIdx.x; i < (int)(sizeof(MfParams) / 4); i += blockDim.x)
        reinterpret_cast<int *>(&P)[i] = reinterpret_cast<const int *>(&params)[i];
    if (threadIdx.x == 0) {
        g_vb = blockIdx.x;
        g_vn = gridDim.x;
    }
    __syncthreads();
    solve_instance();
}

// Barrier of one group of CTAs (no hook): w[0] arrivals, w[1] generation.  In
// clusters, a CTA that gives up sets its cluster's bit (w[3], w[4]) and the whole
// cluster leaves: the squads of the instance that follows write into one
// another's shared memory.  Only a cluster's own CTAs set its bit, before the
// cluster's barrier behind which all of them read it.
__device__ bool group_sync(unsigned *w, unsigned &gen_local, unsigned long long wait_ns, int *abort)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int good = 1;
        const unsigned gen = gen_local;
        __threadfence();
        if (atomicAdd(w, 1u) + 1u == (unsigned)vn()) {
            atomicExch(w, 0u);
            __threadfence();
            st_release(w + 1, gen + 1u);
        } else {
            unsigned long long t0 = 0;
            unsigned spins = 0;
            while (ld_acquire(w + 1) == gen) {
                ++spins;
                if (spins > 64) __nanosleep(spins > 4096 ? 200 : 32);
                if ((spins & 31u) == 0) {
                    unsigned long long now = gtimer();
                    if (t0 == 0) {
                        t0 = now;
                    } else if (now - t0 > wait_ns) {
                        const unsigned q = (unsigned)vb() / cluster_size();
                        if (cluster_size() > 1) atomicOr(w + 3 + (q >> 5), 1u << (q & 31u));
                        atomicExch(abort, 1);
                        good = 0;
                        break;
                    }
                }
            }
        }
        __threadfence();
        gen_local = gen + 1u;
        ok = good;
    }
    __syncthreads();
    if (cluster_size() > 1) {
        const unsigned q = (unsigned)vb() / cluster_size();
        cluster_sync();
        if (threadIdx.x == 0 && (__ldcg(w + 3 + (q >> 5)) >> (q & 31u) & 1u)) ok = 0;
        __syncthreads();
    }
    return ok != 0;
}

// Many instances in one persistent launch: the grid is cut into groups of
// gsize CTAs; each group takes the next instance from a shared queue (the host
// orders it largest first) and runs its whole solve, then takes another.
// gstate holds, per group, 32 words: w[0] arrivals, w[1] generation, w[2] the
// instance the group's first CTA took, w[3] and w[4] the clusters that left.
__global__ void __launch_bounds__(MF_BLOCK, 2) mf_multi_kernel(const MfParams *__restrict__ plist, int count,
                                                               int gsize, unsigned *gstate, unsigned *head,
                                                               unsigned long long wait_ns, int *abort)
{
    __shared__ unsigned ggen;
    const int grp = blockIdx.x / gsize;
    unsigned *gw = gstate + 32 * grp;
    if (threadIdx.x == 0) {
        g_vb = blockIdx.x % gsize;
        g_vn = gsize;
        ggen = ld_acquire(gw + 1);
    }
    __syncthreads();
    for (;;) {
        if (vb() == 0 && threadIdx.x == 0) gw[2] = atomicAdd(head, 1u);
        if (!group_sync(gw, ggen, wait_ns, abort)) return;
        const int i = (int)__ldcg(gw + 2);
        if (i >= count) return;
        for (int w = threadIdx.x; w < (int)(sizeof(MfParams) / 4); w += blockDim.x)
            reinterpret_cast<int *>(&P)[w] = __ldcg(reinterpret_cast<const int *>(plist + i) + w);
        if (!solve_instance()) {
            atomicExch(abort, 1);
            return;
        }
    }
}

// ---------------------------------------------------------------------------
// Auxiliary kernels (state load/readback, checks, queries)
// ---------------------------------------------------------------------------

__global__ void k_cf_reset(MfParams P)
{
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < P.g.slot_cap;
         x += (long long)gridDim.x * blockDim.x)
        P.cf[x] = P.g.cap[x];
}

struct FlowItems {
    long long count;
    const int32_t *u, *v, *f;
    int apply;
};

__global__ void k_set_flow(MfParams P, FlowItems F, long long *bad)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < F.count;
         i += (long long)gridDim.x * blockDim.x) {
        int u = F.u[i], v = F.v[i], f = F.f[i];
        if (u < 0 || u >= P.g.n || v < 0 || v >= P.g.n || u == v) {
            atomicAdd((unsigned long long *)bad, 1ull);
            continue;
        }
        int x = find_slot(P, u, v);
        if (x < 0 || f < 0 || f > P.g.cap[x]) {
            atomicAdd((unsigned long long *)bad, 1ull);
            continue;
        }
        if (F.apply && f > 0) {
            atomicSub(P.cf + x, f);
            atomicAdd(P.cf + P.g.rev[x], f);
        }
    }
}

// K8: e(v) = sum over v's slots of c_f - c.
__global__ void k_excess(MfParams P, long long *mismatch)
{
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < P.g.n;
         v += (long long)gridDim.x * blockDim.x) {
        int r0 = P.g.off[v], d = P.g.deg[v];
        long long s = 0;
        for (int j = 0; j < d; ++j) s += (long long)P.cf[r0 + j] - (long long)P.g.cap[r0 + j];
        if (mismatch) {
            if (s != P.e[v]) atomicAdd((unsigned long long *)mismatch, 1ull);
        } else {
            P.e[v] = s;
        }
    }
}

__global__ void k_check(MfParams P, long long *out)
{
    const int n = P.g.n;
    long long pair_bad = 0, cross = 0, act = 0, cut = 0, val = 0;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (long long)gridDim.x * blockDim.x) {
        int r0 = P.g.off[v], d = P.g.deg[v];
        int hv = P.h[v];
        for (int j = 0; j < d; ++j) {
            int x = r0 + j, y = P.g.rev[x];
            long long lhs = (long long)P.cf[x] + P.cf[y];
            long long rhs = (long long)P.g.cap[x] + P.g.cap[y];
            if (P.cf[x] < 0 || lhs != rhs || P.g.pcap[x] != rhs || P.g.dst[y] != (int)v || P.g.rev[y] != x) ++pair_bad;
            if (hv == n && P.h[P.g.dst[x]] < n) {
                cut += P.g.cap[x];
                if (P.cf[x] > 0) ++cross;
            }
        }
        if ((int)v != P.sink && (int)v != P.source && P.e[v] > 0 && hv < n) ++act;
        if ((int)v != P.source && hv < n) val += P.e[v];
    }
    atomicAdd((unsigned long long *)&out[0], (unsigned long long)pair_bad);
    atomicAdd((unsigned long long *)&out[2], (unsigned long long)cross);
    atomicAdd((unsigned long long *)&out[3], (unsigned long long)act);
    atomicAdd((unsigned long long *)&out[4], (unsigned long long)cut);
    atomicAdd((unsigned long long *)&out[5], (unsigned long long)val);
}

// The answer of a solve: the source side A = {h = n} and the capacity of the
// cut.  Both come from one pass over the heights, four vertices per lane; the
// side goes straight to the caller's (pinned) memory in 128-byte pieces.  The
// cut is summed over the rows of whichever side has fewer slots: from A the
// capacities c(u, v) of its slots into the other side, from the other side
// c(u, v) = pcap - c(v, u) of its slots (v, u) into A, without a gather through
// rev.  Warps take the rows of 32 vertices as one concatenated range; a row of
// more than kAnswerLong slots goes to its whole CTA, and the terminal's row,
// which on grids holds an edge to every pixel, to all CTAs (one warp per row
// took 1.5 ms for the 262 K slots of a 512 x 512 grid's source).  The last CTA
// to finish writes the sum and leaves the accumulators at zero.
constexpr int kAnswerThreads = 256, kAnswerLong = 1024, kAnswerList = 128;

__device__ __forceinline__ long long answer_slot(const MfParams &P, int x, bool from_sink)
{
    const int hz = ldg_cg(P.h + ldg_cg(P.g.dst + x));
    if (from_sink) return hz == P.g.n ? (long long)ldg_cg(P.g.pcap + x) - ldg_cg(P.g.cap + x) : 0;
    return hz < P.g.n ? ldg_cg(P.g.cap + x) : 0;
}

__global__ void __launch_bounds__(kAnswerThreads) k_answer(MfParams P, MfAnswer A)
{
    __shared__ int longs[kAnswerList];
    __shared__ int nlong;
    __shared__ long long part[kAnswerThreads / 32];
    const int n = P.g.n, tid = threadIdx.x, lane = tid & 31;
    const bool want = A.cut != nullptr, fs = A.from_sink != 0;
    const int term = fs ? P.sink : P.source;
    if (tid == 0) nlong = 0;
    __syncthreads();
    long long sum = 0;
    const long long nw = (long long)gridDim.x * (kAnswerThreads / 32);
    for (long long w = (long long)blockIdx.x * (kAnswerThreads / 32) + (tid >> 5); w * 128 < n; w += nw) {
        const int v0 = (int)(w * 128) + 4 * lane;
        int h[4];
        if (v0 + 4 <= n) {
            const int4 q = __ldcg(reinterpret_cast<const int4 *>(P.h + v0));
            h[0] = q.x, h[1] = q.y, h[2] = q.z, h[3] = q.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) h[k] = v0 + k < n ? ldg_cg(P.h + v0 + k) : -1;
        }
        if (A.side) {
            if (v0 + 4 <= n) {
                *reinterpret_cast<uchar4 *>(A.side + v0) = make_uchar4(h[0] == n, h[1] == n, h[2] == n, h[3] == n);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (v0 + k < n) A.side[v0 + k] = h[k] == n;
            }
        }
        if (!want) continue;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int v = v0 + k;
            const bool mine = h[k] >= 0 && (h[k] == n) != fs && v != term;
            if (!__any_sync(0xffffffffu, mine)) continue;
            const int r0 = mine ? P.g.off[v] : 0;
            int d = mine ? ldg_cg(P.g.deg + v) : 0;
            if (d > kAnswerLong) {
                const int i = atomicAdd(&nlong, 1);
                if (i < kAnswerList) {
                    longs[i] = v;
                    d = 0;
                }
            }
            int incl = d;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int excl = incl - d, T = __shfl_sync(0xffffffffu, incl, 31);
            for (int kb = 0; kb < T; kb += 128) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int j = kb + r * 32 + lane;
                    int owner = 0;
#pragma unroll
                    for (int st = 16; st >= 1; st >>= 1) {
                        const int cand = owner + st;
                        const int ec = __shfl_sync(0xffffffffu, excl, cand & 31);
                        if (cand < 32 && ec <= j) owner = cand;
                    }
                    const int rb = __shfl_sync(0xffffffffu, r0, owner), eb = __shfl_sync(0xffffffffu, excl, owner);
                    if (j < T) sum += answer_slot(P, rb + (j - eb), fs);
                }
            }
        }
    }
    if (!want) return;
    const int t0 = P.g.off[term], td = ldg_cg(P.g.deg + term);
    for (long long j = (long long)blockIdx.x * kAnswerThreads + tid; j < td; j += (long long)gridDim.x * kAnswerThreads)
        sum += answer_slot(P, t0 + (int)j, fs);
    __syncthreads();
    for (int i = 0; i < min(nlong, kAnswerList); ++i) {
        const int r0 = P.g.off[longs[i]], d = ldg_cg(P.g.deg + longs[i]);
        for (int j = tid; j < d; j += kAnswerThreads) sum += answer_slot(P, r0 + j, fs);
    }
    sum = warp_sum_ll(sum);
    if (lane == 0) part[tid >> 5] = sum;
    __syncthreads();
    if (tid == 0) {
        long long t = 0;
        for (int i = 0; i < kAnswerThreads / 32; ++i) t += part[i];
        if (t) atomic_add_ll(A.acc, t);
        __threadfence();
        if (atomic_add_ll(A.acc + 1, 1) + 1 == (long long)gridDim.x) {
            __threadfence();
            *A.cut = __ldcg(A.acc);
            A.acc[0] = A.acc[1] = 0;
        }
    }
}

__global__ void k_reverse_cf(MfParams P, const int32_t *in, int32_t *out)
{
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < P.g.slot_cap;
         x += (long long)gridDim.x * blockDim.x)
        out[x] = in[P.g.rev[x]];
}

// pcap = c(u, v) + c(v, u) on every used slot, from cap and rev (the pair sum
// a parked state does not keep).  One warp per row.
__global__ void k_pcap(MfParams P)
{
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < P.g.n; u += nw) {
        const int r0 = P.g.off[u], d = P.g.deg[u];
        for (int j = lane; j < d; j += 32) {
            const int x = r0 + j;
            P.g.pcap[x] = P.g.cap[x] + P.g.cap[P.g.rev[x]];
        }
    }
}

__global__ void k_rowid(MfParams P, int32_t *rowid)
{
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < P.g.n;
         v += (long long)gridDim.x * blockDim.x) {
        int r0 = P.g.off[v], d = P.g.deg[v], end = P.g.off[v + 1];
        for (int x = r0; x < end; ++x) rowid[x] = x < r0 + d ? (int)v : -1;
    }
}

__global__ void k_negate(long long *e, int n)
{
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x)
        e[v] = -e[v];
}

// ---- device-side rebuild of the layout (rows grow; nothing moves to the host) ----

// New reserved size of every row: used slots + pending insertions + slack.
__global__ void k_row_capacity(MfParams P, float slack_factor, int slack_min, long long *cap_out)
{
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < P.g.n;
         u += (long long)gridDim.x * blockDim.x) {
        cap_out[u] = mf_row_size((long long)P.g.deg[u] + P.sc.ins_need[u], slack_factor, slack_min);
    }
}

// Exclusive scan of n int64 values in place, in three passes: every CTA scans
// its tile of MF_SCAN_TILE values and leaves the tile's total in part[]; one CTA
// scans the totals; every CTA adds its tile's offset.  a[n] gets the total.
constexpr int kScanThreads = 1024, kScanPer = MF_SCAN_TILE / kScanThreads;

__device__ __forceinline__ long long block_exclusive_scan(long long x, long long *warp_sums, long long &total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[w] = incl;
    __syncthreads();
    if (w == 0) {
        const long long ws = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
        long long wi = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        warp_sums[lane] = wi - ws;              // exclusive offset of each warp
        if (lane == 31) warp_sums[32] = wi;     // the CTA's total
    }
    __syncthreads();
    total = warp_sums[32];
    const long long r = warp_sums[w] + incl - x;
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(long long *a, long long n, long long *part)
{
    __shared__ long long ws[33];
    const long long base = (long long)blockIdx.x * MF_SCAN_TILE + (long long)threadIdx.x * kScanPer;
    long long v[kScanPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        v[k] = base + k < n ? a[base + k] : 0;
        sum += v[k];
    }
    long long total;
    long long run = block_exclusive_scan(sum, ws, total);
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (base + k < n) a[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == 0) part[blockIdx.x] = total;
}

// One CTA: exclusive scan of the tile totals (any count), total into part[nt].
__global__ void __launch_bounds__(kScanThreads) k_scan_parts(long long *part, long long nt)
{
    __shared__ long long ws[33];
    long long carry = 0;
    for (long long b0 = 0; b0 < nt; b0 += blockDim.x) {
        const long long i = b0 + threadIdx.x;
        const long long x = i < nt ? part[i] : 0;
        long long total;
        const long long r = block_exclusive_scan(x, ws, total);
        if (i < nt) part[i] = carry + r;
        carry += total;
    }
    if (threadIdx.x == 0) part[nt] = carry;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_add(long long *a, long long n, const long long *part,
                                                            long long nt)
{
    const long long off = part[blockIdx.x];
    const long long base = (long long)blockIdx.x * MF_SCAN_TILE;
    for (int k = threadIdx.x; k < MF_SCAN_TILE; k += blockDim.x)
        if (base + k < n) a[base + k] += off;
    if (blockIdx.x == 0 && threadIdx.x == 0) a[n] = part[nt];
}

struct MoveOut {
    const long long *noff;   // new row starts (int64, n + 1)
    int32_t *off, *dst, *cf, *cap, *rev, *pcap;   // new arrays
    long long slot_cap;
    int2 *items;             // pieces of the long rows: (row, first slot of the piece)
    unsigned *nitems;        // their number
};

// New slot y of row u at position j: the old slot's values when j < d (the
// reverse index of slot (u, v) moves with row v: new_rev = new_off[v] + (rev -
// old_off[v])), else an empty slot (dst = u, no capacity, rev = itself).
__device__ __forceinline__ void move_slot(const MfParams &P, const MoveOut &M, int u, int o0, int d, int j,
                                          long long y)
{
    if (j < d) {
        const int x = o0 + j;
        const int v = __ldcs(P.g.dst + x);
        const int cf = __ldcs(P.g.cf + x), cap = __ldcs(P.g.cap + x), pc = __ldcs(P.g.pcap + x);
        const int rv = __ldcs(P.g.rev + x);
        const int rn = (int)__ldg(M.noff + v) + (rv - __ldg(P.g.off + v));
        M.dst[y] = v;
        M.cf[y] = cf;
        M.cap[y] = cap;
        M.pcap[y] = pc;
        M.rev[y] = rn;
    } else {
        M.dst[y] = u;
        M.cf[y] = 0;
        M.cap[y] = 0;
        M.pcap[y] = 0;
        M.rev[y] = (int)y;
    }
}

// Rows longer than MF_MOVE_PIECE slots (new size) become pieces of that many
// slots, listed once the new sizes are known.
__global__ void k_move_items(MfParams P, MoveOut M)
{
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < P.g.n;
         u += (long long)gridDim.x * blockDim.x) {
        const long long S = M.noff[u + 1] - M.noff[u];
        if (S <= MF_MOVE_PIECE) continue;
        const int np = (int)((S + MF_MOVE_PIECE - 1) / MF_MOVE_PIECE);
        const unsigned at = atomicAdd(M.nitems, (unsigned)np);
        for (int k = 0; k < np; ++k) M.items[at + k] = make_int2((int)u, k * MF_MOVE_PIECE);
    }
}

// Copy every row to its new place.  Warps take either 32 consecutive rows, of
// which they copy the rows of at most MF_MOVE_PIECE slots as one concatenated
// range (each lane finds the row that owns its slot), or one piece of a long
// row; each lane moves kMv slots per step, so a step keeps kMv independent
// load chains in flight per lane.
constexpr int kMv = 4;
__global__ void k_move_rows(MfParams P, MoveOut M)
{
    const int lane = threadIdx.x & 31;
    const long long nblk = ((long long)P.g.n + 31) >> 5;
    const long long nw = nblk + *(volatile unsigned *)M.nitems;
    for (long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw;
         w += ((long long)gridDim.x * blockDim.x) >> 5) {
        if (w >= nblk) {
            const int2 it = M.items[w - nblk];
            const int u = it.x;
            const long long n0 = M.noff[u];
            const int S = (int)(M.noff[u + 1] - n0);
            const int o0 = P.g.off[u], d = P.g.deg[u];
            const int end = it.y + MF_MOVE_PIECE < S ? it.y + MF_MOVE_PIECE : S;
            for (int jb = it.y; jb < end; jb += 32 * kMv) {
#pragma unroll
                for (int r = 0; r < kMv; ++r) {
                    const int j = jb + r * 32 + lane;
                    if (j < end) move_slot(P, M, u, o0, d, j, n0 + j);
                }
            }
            continue;
        }
        const int u0 = (int)(w << 5);
        const int u = u0 + lane;
        const bool ok = u < P.g.n;
        const long long n0 = ok ? M.noff[u] : 0;
        const int S = ok ? (int)(M.noff[u + 1] - n0) : 0;
        const int Ss = S <= MF_MOVE_PIECE ? S : 0;      // long rows go by pieces
        const int o0 = ok ? P.g.off[u] : 0, d = ok ? P.g.deg[u] : 0;
        if (ok) M.off[u] = (int)n0;
        int incl = Ss;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int excl = incl - Ss;
        const int T = __shfl_sync(0xffffffffu, incl, 31);
        for (int kb = 0; kb < T; kb += 32 * kMv) {        // the same trip count in every lane
#pragma unroll
            for (int r = 0; r < kMv; ++r) {
                const int k = kb + r * 32 + lane;
                int owner = 0;
#pragma unroll
                for (int st = 16; st >= 1; st >>= 1) {
                    const int cand = owner + st;
                    const int ec = __shfl_sync(0xffffffffu, excl, cand & 31);
                    if (cand < 32 && ec <= k) owner = cand;
                }
                const long long rn0 = __shfl_sync(0xffffffffu, n0, owner);
                const int ro = __shfl_sync(0xffffffffu, o0, owner);
                const int rd_ = __shfl_sync(0xffffffffu, d, owner);
                const int re = __shfl_sync(0xffffffffu, excl, owner);
                if (k < T) move_slot(P, M, u0 + owner, ro, rd_, k - re, rn0 + (k - re));
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) M.off[P.g.n] = (int)M.noff[P.g.n];
}

__global__ void k_clear_need(MfParams P)
{
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < P.g.n;
         u += (long long)gridDim.x * blockDim.x)
        P.sc.ins_need[u] = 0;
}

inline int cuda_rc(cudaError_t e) { return e == cudaSuccess ? MAXFLOW_OK : MAXFLOW_ERR_CUDA; }

}  // namespace

// Dynamic shared memory per CTA of the persistent kernels: as much as still
// lets two CTAs share an SM (the register budget allows two).  Computed once per
// device, with that device current; the kernels' attributes are set to allow it.
int mf_stage_bytes(int device, int *bytes)
{
    static std::mutex mu;
    static int cache[64];
    static bool init = false;
    std::lock_guard<std::mutex> lock(mu);
    if (!init) {
        for (int &x : cache) x = -1;
        init = true;
    }
    if (device < 0 || device >= 64) return MAXFLOW_ERR_INVALID;
    if (cache[device] < 0) {
        cudaFuncAttributes a1{}, a2{};
        int smem_sm = 0, reserved = 0, optin = 0;
        if (cudaFuncGetAttributes(&a1, mf_solve_kernel) != cudaSuccess ||
            cudaFuncGetAttributes(&a2, mf_multi_kernel) != cudaSuccess ||
            cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device) != cudaSuccess ||
            cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess)
            return MAXFLOW_ERR_CUDA;
        const long long stat = (long long)(a1.sharedSizeBytes > a2.sharedSizeBytes ? a1.sharedSizeBytes
                                                                                   : a2.sharedSizeBytes);
        long long b = (long long)smem_sm / 2 - reserved - stat;
        if (b > (long long)optin - stat) b = (long long)optin - stat;
        b &= ~255ll;
        if (b < 0) b = 0;
        if (cudaFuncSetAttribute(mf_solve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b) != cudaSuccess ||
            cudaFuncSetAttribute(mf_multi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b) != cudaSuccess)
            return MAXFLOW_ERR_CUDA;
        cudaFuncSetAttribute(mf_solve_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
        cudaFuncSetAttribute(mf_multi_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
        cudaGetLastError();
        cache[device] = (int)b;
    }
    *bytes = cache[device];
    return MAXFLOW_OK;
}

int mf_max_coresident_blocks(int device, int *per_sm, int *num_sms, int dyn_bytes)
{
    int k = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, mf_solve_kernel, MF_BLOCK, (size_t)dyn_bytes) != cudaSuccess)
        return MAXFLOW_ERR_CUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return MAXFLOW_ERR_CUDA;
    *per_sm = k;
    *num_sms = sms;
    return k > 0 ? MAXFLOW_OK : MAXFLOW_ERR_CUDA;
}

namespace {

// A cooperative launch, in thread-block clusters of `cluster` CTAs where that is more than one.
cudaError_t launch_kernel(const void *kernel, int grid, int cluster, size_t dyn, cudaStream_t st, void **args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(MF_BLOCK);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = st;
    cudaLaunchAttribute at[2]{};
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelExC(&cfg, kernel, args);
}

}  // namespace

// CTAs of the solve kernels that fit the GPU at once in clusters of MF_CLUSTER
// (a cluster's CTAs sit in one GPC, so a few SMs may be left over), with the
// device current; 0 where there are none.
int mf_max_clustered_blocks(int dyn_bytes, int *blocks)
{
    *blocks = 0;
    int least = 0;
    for (const void *k : {(const void *)mf_solve_kernel, (const void *)mf_multi_kernel}) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(MF_CLUSTER);
        cfg.blockDim = dim3(MF_BLOCK);
        cfg.dynamicSmemBytes = (size_t)dyn_bytes;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = MF_CLUSTER;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, k, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return MAXFLOW_OK;
        }
        least = k == (const void *)mf_solve_kernel || nc < least ? nc : least;
    }
    *blocks = least * MF_CLUSTER;
    return MAXFLOW_OK;
}

int mf_launch_multi(const MfParams *plist_dev, int count, int gsize, int grid, unsigned *gstate, unsigned *head,
                    unsigned long long wait_ns, int *abort, int cluster, void *stream, int stage_bytes)
{
    void *args[] = {(void *)&plist_dev, &count, &gsize, &gstate, &head, &wait_ns, &abort};
    return cuda_rc(launch_kernel((const void *)mf_multi_kernel, grid, cluster, (size_t)stage_bytes,
                                 (cudaStream_t)stream, args));
}

int mf_launch(const MfParams &p, int grid, int cluster, void *stream)
{
    MfParams q = p;
    void *args[] = {&q};
    return cuda_rc(launch_kernel((const void *)mf_solve_kernel, grid, cluster, (size_t)p.stage_slots * sizeof(int),
                                 (cudaStream_t)stream, args));
}

int mf_launch_aux(int which, const MfParams &p, void *stream, long long *dev_out, const void *extra)
{
    cudaStream_t st = (cudaStream_t)stream;
    const int B = 256;
    long long nv = p.g.n, ns = p.g.slot_cap;
    int gv = (int)((nv + B - 1) / B);
    int gs = (int)((ns + B - 1) / B);
    if (gv > 65535) gv = 65535;
    if (gs > 65535) gs = 65535;
    if (gv < 1) gv = 1;
    if (gs < 1) gs = 1;
    switch (which) {
    case MF_AUX_SET_CF_RESET:
        k_cf_reset<<<gs, B, 0, st>>>(p);
        break;
    case MF_AUX_SET_FLOW: {
        const FlowItems *f = (const FlowItems *)extra;
        int g = (int)((f->count + B - 1) / B);
        if (g < 1) g = 1;
        if (g > 65535) g = 65535;
        k_set_flow<<<g, B, 0, st>>>(p, *f, dev_out);
        break;
    }
    case MF_AUX_EXCESS:
        k_excess<<<gv, B, 0, st>>>(p, dev_out);
        break;
    case MF_AUX_CHECK:
        k_check<<<gv, B, 0, st>>>(p, dev_out);
        if (cudaGetLastError() != cudaSuccess) return MAXFLOW_ERR_CUDA;
        k_excess<<<gv, B, 0, st>>>(p, dev_out + 1);
        break;
    case MF_AUX_ANSWER: {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return MAXFLOW_ERR_CUDA;
        const long long blocks = (nv + 4 * kAnswerThreads - 1) / (4 * kAnswerThreads);
        k_answer<<<(int)(blocks < 8ll * sms ? blocks : 8ll * sms), kAnswerThreads, 0, st>>>(p, *(const MfAnswer *)extra);
        break;
    }
    case MF_AUX_REVERSE_CF: {
        const int32_t *const *io = (const int32_t *const *)extra;
        k_reverse_cf<<<gs, B, 0, st>>>(p, io[0], (int32_t *)io[1]);
        break;
    }
    case MF_AUX_DUMP:
        k_rowid<<<gv, B, 0, st>>>(p, (int32_t *)extra);
        break;
    case MF_AUX_NEGATE_E:
        k_negate<<<gv, B, 0, st>>>(p.e, p.g.n);
        break;
    case MF_AUX_PCAP: {
        long long g = (nv * 32 + B - 1) / B;
        k_pcap<<<(int)(g > 65535 ? 65535 : (g < 1 ? 1 : g)), B, 0, st>>>(p);
        break;
    }
    default:
        return MAXFLOW_ERR_INVALID;
    }
    return cuda_rc(cudaGetLastError());
}

int mf_set_flow_items(const MfParams &p, void *stream, long long *dev_bad, long long count,
                                  const int32_t *du, const int32_t *dv, const int32_t *df, int apply)
{
    FlowItems f{count, du, dv, df, apply};
    return mf_launch_aux(MF_AUX_SET_FLOW, p, stream, dev_bad, &f);
}

int mf_rebuild_capacity(const MfParams &p, void *stream, float slack_factor, int slack_min, long long *noff)
{
    cudaStream_t st = (cudaStream_t)stream;
    int g = (int)((p.g.n + 255) / 256);
    if (g > 65535) g = 65535;
    if (g < 1) g = 1;
    k_row_capacity<<<g, 256, 0, st>>>(p, slack_factor, slack_min, noff);
    if (cudaGetLastError() != cudaSuccess) return MAXFLOW_ERR_CUDA;
    return mf_scan64(noff, p.g.n, stream);
}

// The tile totals sit behind the n + 1 values (mf_rebuild_scratch).
int mf_scan64(long long *a, long long n, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    const long long nt = mf_scan_tiles(n);
    long long *part = a + n + 1;
    k_scan_tiles<<<(int)nt, kScanThreads, 0, st>>>(a, n, part);
    if (cudaGetLastError() != cudaSuccess) return MAXFLOW_ERR_CUDA;
    k_scan_parts<<<1, kScanThreads, 0, st>>>(part, nt);
    if (cudaGetLastError() != cudaSuccess) return MAXFLOW_ERR_CUDA;
    k_scan_add<<<(int)nt, kScanThreads, 0, st>>>(a, n, part, nt);
    return cuda_rc(cudaGetLastError());
}

int mf_rebuild_move(const MfParams &p, void *stream, const long long *noff, int32_t *off, int32_t *dst, int32_t *cf,
                    int32_t *cap, int32_t *rev, int32_t *pcap, long long slot_cap, int2 *items, unsigned *nitems)
{
    cudaStream_t st = (cudaStream_t)stream;
    MoveOut M{noff, off, dst, cf, cap, rev, pcap, slot_cap, items, nitems};
    if (cudaMemsetAsync(nitems, 0, sizeof(unsigned), st) != cudaSuccess) return MAXFLOW_ERR_CUDA;
    int gi = (int)((p.g.n + 255) / 256);
    if (gi > 65535) gi = 65535;
    if (gi < 1) gi = 1;
    k_move_items<<<gi, 256, 0, st>>>(p, M);
    if (cudaGetLastError() != cudaSuccess) return MAXFLOW_ERR_CUDA;
    // a persistent grid: warps stride over the blocks of 32 rows, then the pieces
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return MAXFLOW_ERR_CUDA;
    k_move_rows<<<sms * 8, 256, 0, st>>>(p, M);
    if (cudaGetLastError() != cudaSuccess) return MAXFLOW_ERR_CUDA;
    int gv = (int)((p.g.n + 255) / 256);
    if (gv > 65535) gv = 65535;
    if (gv < 1) gv = 1;
    k_clear_need<<<gv, 256, 0, st>>>(p);
    return cuda_rc(cudaGetLastError());
}

// ---- scheduler features of a batch (one CTA) ----
__global__ void __launch_bounds__(256) k_features(MfFeatIn F, float *out)
{
    __shared__ long long red[4][8];
    long long vals[4] = {0, 0, 0, 0};              // touching s, touching t, deleting, capacities
    for (long long i = threadIdx.x; i < F.count; i += blockDim.x) {
        const int u = F.bu[i], v = F.bv[i], c = F.bc[i];
        vals[0] += u == F.s || v == F.s;
        vals[1] += u == F.t || v == F.t;
        vals[2] += c == 0;
        vals[3] += c;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const long long x = warp_sum_ll(vals[k]);
        if (lane == 0) red[k][w] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long tot[4] = {0, 0, 0, 0};
        for (int k = 0; k < 4; ++k)
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tot[k] += red[k][q];
        make_features(out, F.count, F.m, F.n, (unsigned)tot[0], (unsigned)tot[1], (unsigned)tot[2], tot[3], F.mean_cap,
                      F.host);
    }
}

int mf_features(const MfFeatIn &f, float *out_dev, void *stream)
{
    k_features<<<1, 256, 0, (cudaStream_t)stream>>>(f, out_dev);
    return cuda_rc(cudaGetLastError());
}
