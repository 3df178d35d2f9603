// rs_topk.cu -- top-K nodes by (score descending, node id ascending)
// (Alg. 1 Step 4).
//
// Each node is a unique 96-bit key (bits(score) << 32 | ~id): for scores >= 0
// the IEEE bit pattern orders like the value, and ~id makes smaller ids rank
// higher among equal scores.  One cooperative launch (at most one 1024-thread
// CTA per SM, grid-wide barriers from cooperative groups) runs a
// most-significant-digit radix select with 12-bit digits:
//   per level (two grid-wide barriers): privatised shared-memory histograms of
//   the digit over the current candidates, merged into a global histogram; every
//   CTA finds the bucket that holds the K-th key in it for itself; keys of higher
//   buckets are final ("sure"), keys of that bucket stay candidates, both appended
//   with one atomic per warp.  The levels take turns with two global histograms:
//   one is cleared while the other is read.
// As soon as the sure keys and the candidates fit the final ranking (16,384 keys
// at most) the grid ranks them: runs of 256 keys are sorted, a run per CTA, and
// every key's rank is its place in its own run plus the number of greater keys in
// each other run (binary searches, the runs spread over the lanes), which is where
// it is written.
//
// Latency bounds it: the passes over the scores are a few microseconds, the rest are
// barriers and the launch.  Against the form before this one (three barriers a level, a
// bitonic sort of all the keys by one CTA): 31 -> 22 us for n = 2,000, k = 50 (two plain
// launches), 52 -> 38 us for n = 1,000,000, k = 1,000, 260 -> 54 us for n = 1,000,000,
// k = 10,000 and 112 -> 74 us for n = 8,000,000, k = 1,000.
#include <algorithm>
#include <cooperative_groups.h>

#include "rs.h"
#include "rs_internal.cuh"

namespace cg = cooperative_groups;
using namespace rs;

namespace {

constexpr int kTkThreads = 1024;
constexpr int kBits = 12;
constexpr int kBins = 1 << kBits;
constexpr int kLevels = 96 / kBits;
constexpr int kSortMax = 16384;   // largest K, and the most keys the final ranking takes
constexpr int kRun = 256;         // keys per sorted run of the final ranking

enum { C_SURE = 0, C_NEXT = 1 /* and 2: candidate counters of even / odd levels */ };

// keys left when the selection stops and ranks: ranking 8,192 keys costs less than
// another radix level does, and 2 K keys are met for every K up to kSortMax / 2
__host__ __device__ __forceinline__ int rank_target(int k) { return 2 * k > 8192 ? kSortMax : 8192; }

// digit `level` (0 = most significant) of the 96-bit key (key64 : ~id)
__device__ __forceinline__ uint32_t digit_of(unsigned long long key, uint32_t nid, int level) {
    int hi = 95 - kBits * level;                 // top bit of the digit
    int lo = hi - kBits + 1;
    if (lo >= 32) return (uint32_t)(key >> (lo - 32)) & (kBins - 1);
    if (hi < 32) return (nid >> lo) & (kBins - 1);
    // straddles the two words: bits [hi-32 .. 0] of key, then bits [31 .. lo] of nid
    uint32_t top = (uint32_t)(key & ((1ull << (hi - 31)) - 1));
    return ((top << (32 - lo)) | (nid >> lo)) & (kBins - 1);
}

struct TkArgs {
    const double *scores;
    int64_t n;
    int32_t k;
    int32_t *ids_out;
    double *scores_out;
    uint32_t *hist;                 // 2 x kBins
    int *ctrl;
    unsigned long long *key[2];     // candidate buffers (n each)
    uint32_t *nid[2];
    unsigned long long *skey;       // sure keys (kSortMax)
    uint32_t *snid;
};

__device__ __forceinline__ void load_item(const TkArgs &A, int level, int src, int64_t i,
                                          unsigned long long &key, uint32_t &nid) {
    if (level == 0) {
        key = (unsigned long long)__double_as_longlong(A.scores[i]);
        nid = ~(uint32_t)i;
    } else {
        key = A.key[src][i];
        nid = A.nid[src][i];
    }
}

// append the flagged items of a warp to buf at a position drawn with one atomic
// per warp (every lane of the warp calls; order inside the buffer is free)
__device__ __forceinline__ void warp_append(bool flag, unsigned long long key, uint32_t nid, int *counter,
                                            unsigned long long *kbuf, uint32_t *ibuf) {
    unsigned m = __ballot_sync(0xFFFFFFFFu, flag);
    if (!m) return;
    int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(counter, __popc(m));
    base = __shfl_sync(0xFFFFFFFFu, base, leader);
    if (flag) {
        int p = base + __popc(m & ((1u << lane) - 1u));
        kbuf[p] = key; ibuf[p] = nid;
    }
}

// keys of the sorted (descending) run key/nid[0, len) that rank above (k, id)
__device__ __forceinline__ int greater_in_run(const unsigned long long *key, const uint32_t *nid, int len,
                                              unsigned long long k, uint32_t id) {
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const unsigned long long x = key[mid];
        if (x > k || (x == k && nid[mid] > id)) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The final ranking, step 1: the ns sure keys and total - ns items of buffer src (level 0:
// of the scores), as runs of kRun keys, each sorted by one CTA into the candidate buffer not
// in use; a key's place is the number of greater keys in its run, counted by four threads.
// sh: 4 kRun words.
__device__ __forceinline__ void sort_runs(const TkArgs &A, int level, int src, int ns, int total, uint32_t *sh) {
    const int tid = threadIdx.x;
    const int runs = (total + kRun - 1) / kRun;
    unsigned long long *wkey = (unsigned long long *)sh;
    uint32_t *wnid = sh + 2 * kRun, *wplace = wnid + kRun;
    for (int r = blockIdx.x; r < runs; r += gridDim.x) {
        const int len = min(kRun, total - r * kRun);
        __syncthreads();
        if (tid < len) {
            const int i = r * kRun + tid;
            unsigned long long key; uint32_t nid;
            if (i < ns) { key = A.skey[i]; nid = A.snid[i]; }
            else load_item(A, level, src, i - ns, key, nid);
            wkey[tid] = key; wnid[tid] = nid; wplace[tid] = 0;
        }
        __syncthreads();
        constexpr int kParts = kTkThreads / kRun;
        const int i = tid & (kRun - 1), share = tid / kRun;
        if (i < len) {
            const unsigned long long key = wkey[i]; const uint32_t nid = wnid[i];
            uint32_t above = 0;
            const int hi = min(len, (share + 1) * (kRun / kParts));
            for (int j = share * (kRun / kParts); j < hi; ++j)
                above += wkey[j] > key || (wkey[j] == key && wnid[j] > nid);
            if (above) atomicAdd(&wplace[i], above);
        }
        __syncthreads();
        if (tid < len) {
            const int p = r * kRun + (int)wplace[tid];
            A.key[src ^ 1][p] = wkey[tid]; A.nid[src ^ 1][p] = wnid[tid];
        }
    }
}

// step 2: every key's rank, by `lanes` lanes per key, each over every lanes-th run; the keys of
// rank below K are written at their rank
__device__ __forceinline__ void rank_runs(const TkArgs &A, int src, int total) {
    const unsigned long long *rkey = A.key[src ^ 1];
    const uint32_t *rnid = A.nid[src ^ 1];
    const int runs = (total + kRun - 1) / kRun, lane = threadIdx.x & 31;
    int lanes = 1;
    while (lanes < runs && lanes < 32) lanes <<= 1;
    const int sub = lane & (lanes - 1);
    const int64_t gsize = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll; t0 < (int64_t)total * lanes; t0 += gsize) {
        const int i = (int)((t0 + lane) / lanes);
        const bool in = i < total;
        unsigned long long key = 0; uint32_t nid = 0;
        int rank = 0;
        if (in) {
            const int own = i / kRun;
            key = rkey[i]; nid = rnid[i];
            for (int r = sub; r < runs; r += lanes)
                rank += r == own ? i - own * kRun
                                 : greater_in_run(rkey + r * kRun, rnid + r * kRun, min(kRun, total - r * kRun), key, nid);
        }
        for (int o = lanes >> 1; o; o >>= 1) rank += __shfl_xor_sync(0xFFFFFFFFu, rank, o);
        if (in && sub == 0 && rank < A.k) {
            A.ids_out[rank] = (int32_t)~nid;
            if (A.scores_out) A.scores_out[rank] = __longlong_as_double((long long)key);
        }
    }
}

__global__ void __launch_bounds__(kTkThreads) tk_select_kernel(TkArgs A) {
    cg::grid_group grid = cg::this_grid();
    __shared__ __align__(16) uint32_t sh_hist[kBins];
    __shared__ uint32_t part[32];
    __shared__ int sh_sel;
    __shared__ int sh_above;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + tid;
    const int64_t gsize = (int64_t)gridDim.x * blockDim.x;
    // every warp walks the same trip count, so warp-wide ballots see whole warps
    const int64_t wbase = gtid & ~31ll;
    int *ctrl = A.ctrl;
    // the state every thread derives alike: candidates m in buffer src, rank need among them
    int src = 0;
    int64_t m = A.n;
    int64_t need = A.k;
    bool done = false;                                          // n > rank_target(k)
    if (gtid == 0) { ctrl[C_SURE] = 0; ctrl[C_NEXT] = 0; ctrl[C_NEXT + 1] = 0; }
    for (int64_t b = gtid; b < 2 * kBins; b += gsize) A.hist[b] = 0;
    grid.sync();
    int level = 0;
    for (; level < kLevels && !done; ++level) {
        uint32_t *hist = A.hist + (level & 1) * kBins, *other = A.hist + ((level + 1) & 1) * kBins;
        // histogram of this level's digit (the global one was cleared before)
        for (int b = tid; b < kBins; b += blockDim.x) sh_hist[b] = 0;
        __syncthreads();
        // four items per lane and trip, loaded together; lanes with the same digit add
        // once (the top digits of real scores crowd a few bins, where per-lane shared
        // atomics would serialise)
        for (int64_t i0 = wbase; i0 < m; i0 += 4 * gsize) {
            uint32_t dg[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t i = i0 + j * gsize + lane;
                unsigned long long key = 0; uint32_t nid = 0;
                dg[j] = kBins;                                  // no bin: lanes past the end
                if (i < m) { load_item(A, level, src, i, key, nid); dg[j] = digit_of(key, nid, level); }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned same = __match_any_sync(0xFFFFFFFFu, dg[j]);
                if (dg[j] < kBins && lane == __ffs(same) - 1) atomicAdd(&sh_hist[dg[j]], (uint32_t)__popc(same));
            }
        }
        __syncthreads();
        for (int b = tid; b < kBins; b += blockDim.x)
            if (sh_hist[b]) atomicAdd(&hist[b], sh_hist[b]);
        grid.sync();
        // every CTA: the bucket holding the need-th largest key
        {
            constexpr int per = kBins / kTkThreads;             // 4 bins per thread, from the top
            const int top = kBins - per * tid;
            uint32_t f[per], sacc = 0;
            for (int j = 0; j < per; ++j) { f[j] = __ldcg(&hist[top - 1 - j]); sacc += f[j]; }
            // inclusive scan over the threads: within warps by shuffles, then over the warp sums
            uint32_t incl = sacc;
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane == 31) part[wid] = incl;
            __syncthreads();
            if (wid == 0) {
                uint32_t w = part[lane];
                for (int o = 1; o < 32; o <<= 1) {
                    uint32_t v = __shfl_up_sync(0xFFFFFFFFu, w, o);
                    if (lane >= o) w += v;
                }
                part[lane] = w;                                 // inclusive sums of the warp sums
            }
            __syncthreads();
            const int64_t mine = (int64_t)incl + (wid ? part[wid - 1] : 0u);
            const int64_t before = mine - sacc;
            if (before < need && need <= mine) {
                int64_t acc = before;
                for (int j = 0; j < per; ++j) {
                    if (acc + f[j] >= need) { sh_sel = top - 1 - j; sh_above = (int)acc; break; }
                    acc += f[j];
                }
            }
            __syncthreads();
        }
        // compact: higher buckets are sure, the selected bucket stays; the other global
        // histogram is cleared for the next level (last read before this level's barrier),
        // and the candidate counter of the next level reset (likewise)
        const uint32_t sel = (uint32_t)sh_sel;
        need -= sh_above;
        const int dst = src ^ 1;
        int *next = &ctrl[C_NEXT + (level & 1)];
        for (int64_t b = gtid; b < kBins; b += gsize) other[b] = 0;
        if (gtid == 0) ctrl[C_NEXT + ((level + 1) & 1)] = 0;
        for (int64_t i0 = wbase; i0 < m; i0 += 4 * gsize) {
            unsigned long long key[4]; uint32_t nid[4], dg[4];
            bool in[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t i = i0 + j * gsize + lane;
                key[j] = 0; nid[j] = 0; dg[j] = 0;
                in[j] = i < m;
                if (in[j]) { load_item(A, level, src, i, key[j], nid[j]); dg[j] = digit_of(key[j], nid[j], level); }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                warp_append(in[j] && dg[j] > sel, key[j], nid[j], &ctrl[C_SURE], A.skey, A.snid);
                warp_append(in[j] && dg[j] == sel, key[j], nid[j], next, A.key[dst], A.nid[dst]);
            }
        }
        grid.sync();
        m = __ldcg(next);
        src = dst;
        done = m <= need || __ldcg(&ctrl[C_SURE]) + m <= rank_target(A.k);
    }
    // the sure keys and the candidates left
    const int ns = __ldcg(&ctrl[C_SURE]);
    sort_runs(A, level, src, ns, ns + (int)m, sh_hist);
    grid.sync();
    rank_runs(A, src, ns + (int)m);
}

// n <= rank_target(k): every score goes to the final ranking, as two plain launches (the
// barrier between them costs less than a cooperative launch does)
__global__ void __launch_bounds__(kTkThreads) tk_runs_kernel(TkArgs A) {
    __shared__ __align__(16) uint32_t sh[4 * kRun];
    chain_wait();
    sort_runs(A, 0, 0, 0, (int)A.n, sh);
}
__global__ void __launch_bounds__(kTkThreads) tk_rank_kernel(TkArgs A) {
    chain_wait();
    rank_runs(A, 0, (int)A.n);
}

}  // namespace

static int ensure_topk_workspace(rs_graph *g, int64_t n) {
    if (g->tk_cap >= n && g->tk_hist) return 0;
    void *old[] = {g->tk_hist, g->tk_ctrl, g->tk_keys, g->tk_ids};
    RS_CUDA_TRY(pool_free_many(old, 4));
    g->tk_hist = nullptr; g->tk_ctrl = nullptr; g->tk_keys = nullptr; g->tk_ids = nullptr;
    int64_t cap = n > 1 ? n : 1;
    RS_CUDA_TRY(pool_malloc((void **)&g->tk_hist, 2 * kBins * sizeof(uint32_t)));
    RS_CUDA_TRY(pool_malloc((void **)&g->tk_ctrl, 8 * sizeof(int)));
    RS_CUDA_TRY(pool_malloc((void **)&g->tk_keys, (2 * cap + kSortMax) * sizeof(unsigned long long)));
    RS_CUDA_TRY(pool_malloc((void **)&g->tk_ids, (2 * cap + kSortMax) * sizeof(uint32_t)));
    g->tk_cap = cap;
    g->version++;                     // captured steps hold the old buffers
    return 0;
}

static int tk_grid = 0;   // one CTA per SM, found once per process

// workspace for n scores and the selection kernel's launch shape
int rs::topk_prepare(rs_graph *g, int64_t n) {
    if (int rc = ensure_topk_workspace(g, n)) return rc;
    if (!tk_grid) {
        int dev = 0, sms = 0, per_sm = 0;
        RS_CUDA_TRY(cudaGetDevice(&dev));
        RS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        RS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tk_select_kernel, kTkThreads, 0));
        if (per_sm < 1) return fail(RS_ECUDA, "rs_topk: selection kernel does not fit an SM");
        tk_grid = sms;
    }
    return 0;
}

int rs::topk_scores(rs_graph *g, const double *scores, int64_t n, int32_t k, int32_t *ids, double *out_scores,
                    cudaStream_t s) {
    if (k > kSortMax) return fail(RS_EINVAL, "rs_topk: k above 16384 is not supported");
    if (n > 2147483647LL) return fail(RS_EINVAL, "rs_topk: n too large");
    if (int rc = topk_prepare(g, n)) return rc;
    int64_t cap = g->tk_cap;
    TkArgs A;
    A.scores = scores; A.n = n; A.k = k; A.ids_out = ids; A.scores_out = out_scores;
    A.hist = g->tk_hist; A.ctrl = g->tk_ctrl;
    unsigned long long *kb = g->tk_keys;
    uint32_t *ib = (uint32_t *)g->tk_ids;
    A.key[0] = kb; A.key[1] = kb + cap; A.skey = kb + 2 * cap;
    A.nid[0] = ib; A.nid[1] = ib + cap; A.snid = ib + 2 * cap;
    prof_begin(g, s);
    if (n <= rank_target(k)) {
        const int runs = (int)((n + kRun - 1) / kRun);
        RS_CUDA_TRY(launch(true, tk_runs_kernel, runs, kTkThreads, 0, s, A));
        RS_LAUNCHED(g, s, "tk_runs");
        RS_CUDA_TRY(launch(true, tk_rank_kernel,
                           std::min(tk_grid, (int)((n * std::min(runs, 32) + kTkThreads - 1) / kTkThreads) + 1),
                           kTkThreads, 0, s, A));
        RS_LAUNCHED(g, s, "tk_rank");
        return 0;
    }
    // a CTA for every 2,048 scores of the levels' passes, or every run of the ranking
    const int grid = (int)std::min<int64_t>(tk_grid, std::max<int64_t>((n + 2047) / 2048, rank_target(k) / kRun));
    void *args[] = {&A};
    RS_CUDA_TRY(cudaLaunchCooperativeKernel((void *)tk_select_kernel, dim3(grid), dim3(kTkThreads), args, 0, s));
    RS_LAUNCHED(g, s, "tk_select");
    return 0;
}
