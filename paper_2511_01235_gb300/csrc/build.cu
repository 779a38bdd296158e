// Device construction of the residual Bi-CSR (Sec. 5.1), slot for slot the one
// that graph_build.cpp makes on the host.
//
// Every edge (u, v, c) becomes two records, (u, v) with its capacity and (v, u)
// as a placeholder for the reverse slot.  The records are sorted by (tail, head)
// with a least-significant-digit radix sort, runs of equal pairs are merged
// (capacities of parallel edges add up, a placeholder adds nothing), the rows
// get their slack and their 16-byte aligned places, and each slot finds its
// reverse by binary search in its head's row.
//
// The host needed 57 ms for the 1 M edges of an R-MAT 16 graph (two counting
// sorts, a sort per row and a binary search per slot, over arrays that do not
// fit its caches).  Here the passes over memory bound it: per record and
// digit 32 bytes (the key for the counts, then key and value read and written),
// and the upload of the edge list itself.  With 2^bits the first power of two
// above n there are ceil(2 bits / 8) digits: 5 for R-MAT 16, 6 for R-MAT 20.
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/maxflow.h"
#include "mf_internal.h"

namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kTile = 4096;                   // records per CTA of a sort pass
constexpr int kChunk = kTile / kWarps;        // ... and per warp, taken in order
constexpr int kRadix = 256;

// What the passes tell the host.
struct BuildOut {
    int err;                                  // 1: an entry out of range, 2: a capacity sum above INT32_MAX
    int pad;
    long long loops;                          // self-loops (dropped)
    unsigned long long cap_sum;
    long long merged;                         // directed edges with a capacity after merging
};

__device__ __forceinline__ long long warp_sum(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(kThreads) k_records(const int32_t *src, const int32_t *dst, const int32_t *cap,
                                                      long long m, int n, int bits, unsigned long long *key,
                                                      int32_t *val, BuildOut *out)
{
    long long loops = 0, sum = 0;
    bool bad = false;
    const unsigned long long none = (unsigned long long)n << bits;      // sorts behind every pair
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < m; i += (long long)gridDim.x * kThreads) {
        const int u = src[i], v = dst[i], c = cap[i];
        const bool ok = (unsigned)u < (unsigned)n && (unsigned)v < (unsigned)n && c >= 0;
        const bool keep = ok && u != v;
        bad |= !ok;
        loops += ok && u == v;
        sum += c;
        key[2 * i] = keep ? ((unsigned long long)u << bits) | (unsigned)v : none;
        key[2 * i + 1] = keep ? ((unsigned long long)v << bits) | (unsigned)u : none;
        val[2 * i] = c;
        val[2 * i + 1] = -1;
    }
    loops = warp_sum(loops);
    sum = warp_sum(sum);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) out->err = 1;
    if ((threadIdx.x & 31) == 0) {
        if (loops) atomicAdd((unsigned long long *)&out->loops, (unsigned long long)loops);
        if (sum) atomicAdd(&out->cap_sum, (unsigned long long)sum);
    }
}

// Digit counts of each warp's chunk in cnt[warp][digit].
__device__ __forceinline__ void count_chunk(const unsigned long long *key, long long K, int shift,
                                            unsigned (*cnt)[kRadix])
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kWarps * kRadix; i += kThreads) (&cnt[0][0])[i] = 0;
    __syncthreads();
    const long long base = (long long)blockIdx.x * kTile + w * kChunk;
    for (int j = lane; j < kChunk; j += 32)
        if (base + j < K) atomicAdd(&cnt[w][(unsigned)(key[base + j] >> shift) & (kRadix - 1)], 1u);
    __syncthreads();
}

// table[digit * tiles + tile] = records of the tile with that digit.
__global__ void __launch_bounds__(kThreads) k_digits(const unsigned long long *key, long long K, int shift,
                                                     long long *table)
{
    __shared__ unsigned cnt[kWarps][kRadix];
    count_chunk(key, K, shift, cnt);
    unsigned t = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += cnt[w][threadIdx.x];
    table[(long long)threadIdx.x * gridDim.x + blockIdx.x] = t;
}

// Stable scatter by one digit: the table, scanned, holds where each tile's
// records of a digit start; inside the tile the warps' chunks follow one
// another, and inside a chunk the lanes of a step (match mask).
__global__ void __launch_bounds__(kThreads) k_scatter(const unsigned long long *key, const int32_t *val, long long K,
                                                      int shift, const long long *table, unsigned long long *key_out,
                                                      int32_t *val_out)
{
    __shared__ unsigned cnt[kWarps][kRadix];
    __shared__ long long start[kRadix];
    count_chunk(key, K, shift, cnt);
    {
        const int dgt = threadIdx.x;
        start[dgt] = table[(long long)dgt * gridDim.x + blockIdx.x];
        unsigned run = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const unsigned c = cnt[w][dgt];
            cnt[w][dgt] = run;                // the chunk's place among the tile's records of this digit
            run += c;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long base = (long long)blockIdx.x * kTile + w * kChunk;
    for (int j = 0; j < kChunk; j += 32) {
        const long long i = base + j + lane;
        const bool in = i < K;
        const unsigned long long k = in ? key[i] : 0;
        const int v = in ? val[i] : 0;
        const unsigned dgt = in ? (unsigned)(k >> shift) & (kRadix - 1) : kRadix;
        const unsigned same = __match_any_sync(0xffffffffu, dgt);
        const int leader = __ffs(same) - 1;
        unsigned at = 0;
        if (in && lane == leader) {
            at = cnt[w][dgt];
            cnt[w][dgt] = at + __popc(same);
        }
        at = __shfl_sync(0xffffffffu, at, leader);
        if (in) {
            const long long to = start[dgt] + at + __popc(same & ((1u << lane) - 1u));
            key_out[to] = k;
            val_out[to] = v;
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kThreads) k_heads(const unsigned long long *key, long long K, long long *head)
{
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < K; i += (long long)gridDim.x * kThreads)
        head[i] = i == 0 || key[i] != key[i - 1] ? 1 : 0;
}

// idx: the heads' exclusive scan (K + 1 values).  Record i belongs to pair idx[i + 1] - 1.
__global__ void __launch_bounds__(kThreads) k_merge(const unsigned long long *key, const int32_t *val, long long K,
                                                    const long long *idx, unsigned long long *pair,
                                                    unsigned long long *sum)
{
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < K; i += (long long)gridDim.x * kThreads) {
        const long long j = idx[i + 1] - 1;
        if (idx[i] == j) pair[j] = key[i];    // its first record
        if (val[i] > 0) atomicAdd(sum + j, (unsigned long long)val[i]);
    }
}

__device__ __forceinline__ long long lower(const unsigned long long *pair, long long lo, long long hi,
                                           unsigned long long k)
{
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        if (pair[mid] < k) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Row u holds the pairs [row[u], row[u + 1]).
__global__ void __launch_bounds__(kThreads) k_rows(const unsigned long long *pair, long long U, int n, int bits,
                                                   int32_t *row)
{
    for (long long u = (long long)blockIdx.x * kThreads + threadIdx.x; u <= n; u += (long long)gridDim.x * kThreads)
        row[u] = (int32_t)lower(pair, 0, U, (unsigned long long)u << bits);
}

__global__ void __launch_bounds__(kThreads) k_sizes(const int32_t *row, int n, float factor, int smin, int32_t *deg,
                                                    int32_t *bdeg, long long *size)
{
    for (long long u = (long long)blockIdx.x * kThreads + threadIdx.x; u < n; u += (long long)gridDim.x * kThreads) {
        const int d = row[u + 1] - row[u];
        deg[u] = bdeg[u] = d;
        size[u] = mf_row_size(d, factor, smin);
    }
}

struct Slots {
    int32_t *off, *dst, *cf, *cap, *rev, *pcap;
};

__global__ void __launch_bounds__(kThreads) k_place(const unsigned long long *pair, const unsigned long long *sum,
                                                    long long U, int bits, const int32_t *row, const long long *start,
                                                    Slots s, BuildOut *out)
{
    const unsigned long long mask = (1ull << bits) - 1ull;
    long long real = 0;
    bool over = false;
    for (long long j = (long long)blockIdx.x * kThreads + threadIdx.x; j < U; j += (long long)gridDim.x * kThreads) {
        const unsigned long long k = pair[j];
        const int u = (int)(k >> bits), v = (int)(k & mask);
        const long long r = lower(pair, row[v], row[v + 1], ((unsigned long long)v << bits) | (unsigned)u);
        const unsigned long long c = sum[j], cr = sum[r];
        over |= c > INT32_MAX || cr > INT32_MAX || c + cr > INT32_MAX;
        const long long x = start[u] + (j - row[u]);
        s.dst[x] = v;
        s.cap[x] = s.cf[x] = (int32_t)c;
        s.pcap[x] = (int32_t)(c + cr);
        s.rev[x] = (int32_t)(start[v] + (r - row[v]));
        real += c > 0;
    }
    real = warp_sum(real);
    if (__any_sync(0xffffffffu, over) && (threadIdx.x & 31) == 0) out->err = 2;
    if ((threadIdx.x & 31) == 0 && real) atomicAdd((unsigned long long *)&out->merged, (unsigned long long)real);
}

// Row starts, and the spare slots (a slot to itself without capacity).  One warp per row.
__global__ void __launch_bounds__(kThreads) k_spare(const long long *start, const int32_t *deg, int n, Slots s)
{
    const int lane = threadIdx.x & 31;
    for (long long u = ((long long)blockIdx.x * kThreads + threadIdx.x) >> 5; u < n;
         u += (long long)gridDim.x * kWarps) {
        const long long b = start[u], e = start[u + 1];
        if (lane == 0) s.off[u] = (int32_t)b;
        if (lane == 0 && u == n - 1) s.off[n] = (int32_t)e;
        for (long long x = b + deg[u] + lane; x < e; x += 32) {
            s.dst[x] = (int32_t)u;
            s.rev[x] = (int32_t)x;
            s.cap[x] = s.cf[x] = s.pcap[x] = 0;
        }
    }
}

inline size_t pad(size_t b) { return (b + 255) & ~(size_t)255; }
inline int blocks(long long items) { return (int)(items < 1 ? 1 : (items + kThreads - 1) / kThreads > 65535 ? 65535 : (items + kThreads - 1) / kThreads); }

// Where the parts of the scratch block lie.
struct Parts {
    size_t key_a, key_b, val_a, val_b, pair, sum, table, row, start, out, total;
    long long K, tiles;
    Parts(int n, long long m)
    {
        K = 2 * m;
        tiles = (K + kTile - 1) / kTile;
        if (tiles < 1) tiles = 1;
        size_t o = 0;
        auto take = [&](size_t b) {
            const size_t at = o;
            o += pad(b);
            return at;
        };
        const size_t k = (size_t)K;
        key_a = take(8 * k);
        key_b = take(8 * (size_t)mf_rebuild_scratch(K));        // also the heads' scan
        val_a = take(4 * k);
        val_b = take(4 * k);
        pair = take(8 * k);
        sum = take(8 * k);                                      // first the edge list itself (12 bytes an edge)
        table = take(8 * (size_t)mf_rebuild_scratch(kRadix * tiles));
        row = take(4 * ((size_t)n + 1));
        start = take(8 * (size_t)mf_rebuild_scratch(n));
        out = take(sizeof(BuildOut));
        total = o;
    }
};

inline int ok(cudaError_t e) { return e == cudaSuccess ? MAXFLOW_OK : MAXFLOW_ERR_CUDA; }
#define B_TRY(expr)                          \
    do {                                     \
        int _rc = (expr);                    \
        if (_rc != MAXFLOW_OK) return _rc;   \
    } while (0)

}  // namespace

size_t mf_build_scratch(int n, long long m) { return Parts(n, m).total; }

int mf_build_sizes(MfBuild &b, int n, long long m, const int32_t *src, const int32_t *dst, const int32_t *cap,
                   float slack_factor, int slack_min, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    const Parts p(n, m);
    char *s = (char *)b.scratch;
    int32_t *in = (int32_t *)(s + p.sum);
    const size_t mb = sizeof(int32_t) * (size_t)m;
    B_TRY(ok(cudaMemcpyAsync(in, src, mb, cudaMemcpyHostToDevice, st)));
    B_TRY(ok(cudaMemcpyAsync(in + m, dst, mb, cudaMemcpyHostToDevice, st)));
    B_TRY(ok(cudaMemcpyAsync(in + 2 * m, cap, mb, cudaMemcpyHostToDevice, st)));
    BuildOut *out = (BuildOut *)(s + p.out);
    B_TRY(ok(cudaMemsetAsync(out, 0, sizeof(BuildOut), st)));
    int bits = 1;
    while ((1ll << bits) < (long long)n + 1) ++bits;            // row n: the dropped records
    unsigned long long *key[2] = {(unsigned long long *)(s + p.key_a), (unsigned long long *)(s + p.key_b)};
    int32_t *val[2] = {(int32_t *)(s + p.val_a), (int32_t *)(s + p.val_b)};
    long long *table = (long long *)(s + p.table);
    k_records<<<blocks(m), kThreads, 0, st>>>(in, in + m, in + 2 * m, m, n, bits, key[0], val[0], out);
    int cur = 0, launches = 1;
    for (int shift = 0; shift < 2 * bits; shift += 8) {
        k_digits<<<(int)p.tiles, kThreads, 0, st>>>(key[cur], p.K, shift, table);
        B_TRY(mf_scan64(table, kRadix * p.tiles, st));
        k_scatter<<<(int)p.tiles, kThreads, 0, st>>>(key[cur], val[cur], p.K, shift, table, key[cur ^ 1], val[cur ^ 1]);
        cur ^= 1;
        launches += 5;
    }
    // the heads' scan needs room behind K values, which only the second key buffer has
    if (cur == 1) {
        B_TRY(ok(cudaMemcpyAsync(key[0], key[1], 8 * (size_t)p.K, cudaMemcpyDeviceToDevice, st)));
    }
    BuildOut h{};
    B_TRY(ok(cudaMemcpyAsync(&h, out, sizeof(h), cudaMemcpyDeviceToHost, st)));
    B_TRY(ok(cudaStreamSynchronize(st)));
    b.launches = launches;
    if (h.err) return MAXFLOW_ERR_INVALID;
    b.cap_sum = (double)h.cap_sum;
    const long long K = p.K - 2 * h.loops;                      // the dropped records are the last ones
    long long *idx = (long long *)key[1];
    unsigned long long *pair = (unsigned long long *)(s + p.pair), *sum = (unsigned long long *)(s + p.sum);
    B_TRY(ok(cudaMemsetAsync(sum, 0, 8 * (size_t)p.K, st)));
    if (K > 0) {
        k_heads<<<blocks(K), kThreads, 0, st>>>(key[0], K, idx);
        B_TRY(mf_scan64(idx, K, st));
        k_merge<<<blocks(K), kThreads, 0, st>>>(key[0], val[cur], K, idx, pair, sum);
        B_TRY(ok(cudaMemcpyAsync(&b.pairs, idx + K, sizeof(long long), cudaMemcpyDeviceToHost, st)));
        B_TRY(ok(cudaStreamSynchronize(st)));
        b.launches += 5;
    } else {
        b.pairs = 0;
    }
    if (b.pairs >= (long long)INT32_MAX - 1) return MAXFLOW_ERR_TOO_LARGE;
    int32_t *row = (int32_t *)(s + p.row);
    long long *start = (long long *)(s + p.start);
    k_rows<<<blocks((long long)n + 1), kThreads, 0, st>>>(pair, b.pairs, n, bits, row);
    k_sizes<<<blocks(n), kThreads, 0, st>>>(row, n, slack_factor, slack_min, b.deg, b.bdeg, start);
    B_TRY(mf_scan64(start, n, st));
    B_TRY(ok(cudaMemcpyAsync(&b.slots, start + n, sizeof(long long), cudaMemcpyDeviceToHost, st)));
    B_TRY(ok(cudaStreamSynchronize(st)));
    b.launches += 5;
    b.bits = bits;
    return b.slots >= (long long)INT32_MAX - 1 ? MAXFLOW_ERR_TOO_LARGE : ok(cudaGetLastError());
}

int mf_build_fill(MfBuild &b, int n, long long m, const MfGraph &g, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    const Parts p(n, m);
    char *s = (char *)b.scratch;
    BuildOut *out = (BuildOut *)(s + p.out);
    const Slots sl{g.off, g.dst, g.cf, g.cap, g.rev, g.pcap};
    const long long *start = (const long long *)(s + p.start);
    k_place<<<blocks(b.pairs), kThreads, 0, st>>>((const unsigned long long *)(s + p.pair),
                                                  (const unsigned long long *)(s + p.sum), b.pairs, b.bits,
                                                  (const int32_t *)(s + p.row), start, sl, out);
    k_spare<<<blocks(32ll * n), kThreads, 0, st>>>(start, b.deg, n, sl);
    BuildOut h{};
    B_TRY(ok(cudaMemcpyAsync(&h, out, sizeof(h), cudaMemcpyDeviceToHost, st)));
    B_TRY(ok(cudaStreamSynchronize(st)));
    b.launches += 2;
    b.merged = h.merged;
    return h.err ? MAXFLOW_ERR_TOO_LARGE : MAXFLOW_OK;
}
