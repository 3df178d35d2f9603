// rs_score.cu -- the Robust Spanning Index of every node on the GPU.
//
// The score (Sec. III-B, Eq. RSI) sums, for each node u, the geometric means
// (w_v(u) w_w(v) w_w(u))^(1/3) over ordered pairs (w, v) with w in N(u),
// C(w) != C(u), v in N(w), v != u, C(v) != C(w) and (v in N(u) or
// C(v) = C(u)).  By Lemma 1 a weight depends on the target only through its
// community, w_v(u) = w_v(C(u)), so with sigma_v(c) = w_v(c)^(1/3) the sum
// splits exactly into two kinds of triads:
//
//  * Type-II (Sec. III-A), every v with C(v) = C(u), adjacent to u or not:
//      sum_w sigma_w(C(u))^2 (Q_w(C(u)) - s_u),
//    with s_x = sigma_x(C(x)) (Lemma 2) and Q_w(c) = sum of s_x over the
//    neighbours x of w in community c;
//  * Type-I, v adjacent to u with three distinct communities: the triangles of
//    the cross-community subgraph G_x (every edge of which joins two
//    communities, so each of its triangles spans three); the two ordered
//    triads at apex a of triangle {a, b, c} add
//      S(b->a) S(c->a) (S(b->c) + S(c->b)),   S(x->y) = sigma_x(C(y)).
//
// Passes (Alg. 1 Steps 1-3 and the kernels of Sec. V-B, re-planned):
//   P1  per row v: neighbour-community counts f_v(c) (the interaction_matrix
//       row), aggregates T, L, X, the row's largest weight (-> w_max, Alg. 1
//       Step 2 / normalize_weights), s_v, the cross degree dx(v) (border
//       vertex iff dx > 0, Alg. 1 Step 1);
//   GX  offsets of the cross subgraph rows (nodes with dx >= 2);
//   P2  per row w: counts and Q_w again, sigma_w per column, the Type-II
//       terms pushed to the neighbours, and the G_x rows of w (out-neighbours
//       of higher (dx, id) rank first, in-neighbours from the back);
//   P3  per node a: oriented triangle listing on G_x (pairs of out-neighbours,
//       closing edge by binary search), the Type-I terms of the three apexes;
//   FIN R(u) = acc(u) / (w_max d(u)(d(u)-1)), 0 when d(u) < 2 or w_max = 0.
// All terms are added into 192-bit fixed-point accumulators, and Type-I terms are
// exact products, so the scores depend neither on the order in which threads run
// nor on how terms are grouped before they are added.
#include <initializer_list>
#include <type_traits>
#include <utility>

#include "rs.h"
#include "rs_internal.cuh"
#include "rs_device.cuh"

using namespace rs;

#define FULL 0xFFFFFFFFu

namespace {

// ---- block reductions (every thread of the CTA must call) ----------------------
template <int NT>
__device__ __forceinline__ uint32_t block_sum_u32(uint32_t v, uint32_t *sh) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    uint32_t s = 0;
    for (int i = 0; i < NT / 32; ++i) s += sh[i];
    return s;
}
template <int NT>
__device__ __forceinline__ u128 block_sum_u128(u128 v, u128 *sh) {
    v = warp_sum_u128(v);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    u128 s = 0;
    for (int i = 0; i < NT / 32; ++i) s += sh[i];
    return s;
}
template <int NT>
__device__ __forceinline__ df block_max_df(df v, df *sh) {
    v = warp_max_df(v);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    df m = sh[0];
    for (int i = 1; i < NT / 32; ++i) m = df_max(m, sh[i]);
    return m;
}

// sum of the staged values over the lanes of `grp` (exact, fixed order)
__device__ __forceinline__ u128 group_sum_all(const uint64_t *stage, unsigned grp) {
    u128 q = 0;
    while (grp) {
        int j = __ffs(grp) - 1;
        q += stage[j];
        grp &= grp - 1;
    }
    return q;
}

// Every weight of a row with L distinct neighbour communities is at most
// L log2 L (an entropy over at most L categories is at most log2 L); a row
// whose bound cannot exceed the w_max found so far needs no column maximum.
__device__ __forceinline__ bool row_may_raise_max(uint32_t L, float wcur) {
    if (L < 2) return false;
    float fl = (float)L;
    return fl * __log2f(fl) * 1.001f + 1e-6f > wcur;
}
// w_max found so far, rounded down to a float (read once per warp)
__device__ __forceinline__ float current_wmax(const unsigned long long *wmax_bits) {
    unsigned long long b = *(volatile const unsigned long long *)wmax_bits;
    return __double2float_rd(__longlong_as_double((long long)b));
}

// publish a row's largest weight when it may raise its graph's w_max (wcur is
// the w_max read earlier, rounded down: any m above w_max has m.hi >= wcur)
__device__ __forceinline__ void publish_max(const Batch &B, int32_t gi, df m, float wcur) {
    if (m.hi > 0.0f && m.hi >= wcur) atomicMax(&B.wmax[gi], double_bits(m));
}

// ======================================================================================
// P1
// ======================================================================================

// Row kernels take their next row from a per-launch counter (zeroed at the start of
// every scoring pass), so warps or CTAs that drew short rows take more and no long
// tail is left on a few of them.
__device__ __forceinline__ int64_t warp_next(unsigned long long *ctr) {
    unsigned long long t = 0;
    if ((threadIdx.x & 31) == 0) t = atomicAdd(ctr, 1ull);
    return (int64_t)__shfl_sync(FULL, t, 0);
}
__device__ __forceinline__ int64_t cta_next(unsigned long long *ctr, long long *sh) {
    __syncthreads();
    if (threadIdx.x == 0) *sh = (long long)atomicAdd(ctr, 1ull);
    __syncthreads();
    return *sh;
}

constexpr int kSlots = kSmallMax;

constexpr int kFewRows = 8;             // rows per tile of the small-row kernels on small graphs

__device__ __forceinline__ void store_rowsum(RowSum *rsum, int32_t v, const RowAgg &a) {
    RowSum r;
    r.xlo = (uint64_t)a.X;
    r.xhi = (uint64_t)(a.X >> 64);
    r.L = a.L;
    r.pad = 0;
    rsum[v] = r;
}

// Small rows, tiles of 32 consecutive rows (id order) per warp: the union of
// their CSR segments is streamed with one neighbour per lane (coalesced
// columns, one label gather per lane), (row, community) groups come from warp
// matching, and lane l then finishes row l of the tile.  A row of degree
// <= 32 spans at most two chunks, so its foreign list holds at most 32
// entries (a community seen in two chunks appears twice and is merged).
struct SmallTile {
    int32_t flab[kSlots][32];       // foreign (community, count) entries, entry-major
    uint8_t fcnt[kSlots][32];
    uint8_t row[32];                // the tile's rows with entries, in order
    int32_t pre[33];                // prefix sums of the tile's degrees
    int64_t rb[32];                 // row starts
    int32_t cv[32];                 // row labels
    uint32_t own[32], nf[32];
    int32_t nx[32];                 // cross list fill
};

// one chunk of up to 32 tile entries, entry e0 + lane in this lane (act): its row r, the
// lanes of that row, its neighbour x and x's label c; the own-community counts, the cross
// lists and the (row, community) groups are updated.  Issue slots bound it: a row's lanes are
// consecutive, so they come from the rows' start bits and only the communities take a warp
// match (three matches and a binary search per entry for its row: p1_small and p2_small 1,023
// and 892 us on a 256-graph batch, 1,013 and 829 us this way; 315 and 242, 308 and 240 us on
// 1M nodes)
__device__ __forceinline__ void p1_small_chunk(SmallTile &T, bool act, int32_t r, unsigned lanes, int32_t x, int32_t c,
                                               int32_t *__restrict__ cl_col, int32_t *__restrict__ cl_lab, int lane) {
    const bool own = act && c == T.cv[r];
    const bool foreign = act && !own;
    const unsigned gown = __ballot_sync(FULL, own) & lanes, fm = __ballot_sync(FULL, foreign), grow = fm & lanes;
    const int32_t xbase = foreign ? T.nx[r] : 0;
    const uint32_t fbase = foreign ? T.nf[r] : 0;
    unsigned gc = 0;
    if (foreign) gc = __match_any_sync(fm, c) & lanes;
    const bool lead = foreign && lane == __ffs(gc) - 1;
    const unsigned gl = __ballot_sync(FULL, lead) & lanes;
    __syncwarp();                                       // the row's fill counts are read
    if (own && lane == __ffs(gown) - 1) T.own[r] += __popc(gown);
    if (foreign) {
        const int64_t p = T.rb[r] + xbase + __popc(grow & lanemask_lt());
        cl_col[p] = x;
        cl_lab[p] = c;
        if (lead) {
            const uint32_t slot = fbase + __popc(gl & lanemask_lt());
            T.flab[slot][r] = c;
            T.fcnt[slot][r] = (uint8_t)__popc(gc);
        }
        if (lane == __ffs(grow) - 1) {
            T.nx[r] = xbase + __popc(grow);
            T.nf[r] = fbase + __popc(gl);
        }
    }
    __syncwarp();
}

// lane `lane` finishes row v (degree d, label cv) of the tile: aggregates, weights, s_v
__device__ __forceinline__ void p1_small_finish(SmallTile &T, int32_t v, int32_t d, int32_t cv, const Batch &B,
                                                const uint64_t *__restrict__ LG, NodeRec *__restrict__ rec,
                                                int32_t *__restrict__ Lall, RowSum *__restrict__ rsum, int lane) {
    int32_t gi = graph_of(B, v);
    float wcur = current_wmax(&B.wmax[gi]);
    uint32_t own = T.own[lane];
    int nf = (int)T.nf[lane];
    // merge a community listed from two chunks
    for (int j = 1; j < nf; ++j)
        for (int j2 = 0; j2 < j; ++j2)
            if (T.fcnt[j2][lane] && T.flab[j2][lane] == T.flab[j][lane]) {
                T.fcnt[j2][lane] += T.fcnt[j][lane];
                T.fcnt[j][lane] = 0;
                break;
            }
    u128 X = (u128)own * LG[own];
    uint64_t seen = own ? (1ull << own) : 0ull;
    uint32_t L = own > 0 ? 1u : 0u;
    for (int j = 0; j < nf; ++j) {
        uint32_t f = T.fcnt[j][lane];
        if (!f) continue;
        X += (u128)f * LG[f];
        seen |= 1ull << f;
        ++L;
    }
    RowAgg a{(uint32_t)d, L, X};
    store_rowsum(rsum, v, a);
    bool want_max = row_may_raise_max(a.L, wcur);
    df cm{0.0f, 0.0f}, wown{0.0f, 0.0f};
    if (want_max) {
        while (seen) {
            uint32_t f = (uint32_t)(__ffsll((long long)seen) - 1);
            df w = column_weight(a, f, LG);
            if (f == own) wown = w;
            cm = df_max(cm, w);
            seen &= seen - 1;
        }
    } else if (own > 0) {
        wown = column_weight(a, own, LG);
    }
    NodeRec rr;
    df m = p1_row_result(a, own, cm, k_of(B, gi), LG, rr, cv, wown, want_max);
    publish_max(B, gi, m, wcur);
    rec[v] = rr;
    Lall[v] = (int32_t)a.L;
}

// the tile's R rows: lane l takes row rows[t0 + l]; prefix sums of the degrees, row starts
// and labels into T; returns the tile's entry count D
template <int R>
__device__ __forceinline__ int32_t p1_small_setup(SmallTile &T, const int64_t *__restrict__ off,
                                                  const int32_t *__restrict__ lab, const int32_t *__restrict__ rows,
                                                  int64_t nrows, int64_t t0, int lane, bool &have, int32_t &v,
                                                  int32_t &d, int32_t &cv) {
    int64_t i = t0 + lane;
    have = lane < R && i < nrows;
    v = have ? rows[i] : 0;
    int64_t b = have ? off[v] : 0;
    d = have ? (int32_t)(off[v + 1] - b) : 0;
    cv = have ? lab[v] : -1;
    int32_t incl = d;
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    T.pre[lane + 1] = incl;
    if (lane == 0) T.pre[0] = 0;
    const unsigned some = __ballot_sync(FULL, d > 0);
    if (d > 0) T.row[__popc(some & lanemask_lt())] = (uint8_t)lane;
    T.rb[lane] = b;
    T.cv[lane] = cv;
    T.own[lane] = 0;
    T.nf[lane] = 0;
    T.nx[lane] = 0;
    __syncwarp();
    return __shfl_sync(FULL, incl, 31);
}

// R rows per tile: 32, or kFewRows where that leaves too few warps to fill the GPU, whose time
// is then one tile's chain of chunks (2,000 rows: 17 -> 12 us)
template <int R>
__global__ void __launch_bounds__(kThreads) p1_small_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ col, const int32_t *__restrict__ lab,
    const int32_t *__restrict__ rows, int64_t nrows, Batch B, const uint64_t *__restrict__ LG,
    NodeRec *__restrict__ rec, int32_t *__restrict__ Lall,
    RowSum *__restrict__ rsum, int32_t *__restrict__ cl_col, int32_t *__restrict__ cl_lab) {
    chain_wait();
    __shared__ SmallTile tiles[kThreads / 32];
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    SmallTile &T = tiles[wid];
    int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t0 = warp * R; t0 < nrows; t0 += nwarps * R) {
        bool have;
        int32_t v, d, cv;
        const int32_t D = p1_small_setup<R>(T, off, lab, rows, nrows, t0, lane, have, v, d, cv);
        // chunk e0 of the tile: the lanes where a row starts, and entry e0 + lane's row and
        // column (`started`: the rows that start before the chunk)
        const int32_t first = T.pre[lane];
        auto locate = [&](int32_t e0, int &started, unsigned &starts, int32_t &r, int32_t &x) {
            const int32_t q = first - e0;
            starts = __reduce_or_sync(FULL, d > 0 && q >= 0 && q < 32 ? 1u << q : 0u);
            if (e0 + lane < D) {
                r = T.row[started + rows_started(starts) - 1];
                x = col[T.rb[r] + (e0 + lane - T.pre[r])];
            }
            started += __popc(starts);
        };
        // software pipeline: the label of the next chunk and the column of the one
        // after it are loaded while the current chunk is matched
        int32_t rA = 0, xA = -1, cA = -1, rB = 0, xB = -1;
        int started = 0;
        unsigned sA, sB;
        locate(0, started, sA, rA, xA);
        if (lane < D) cA = lab[xA];
        locate(32, started, sB, rB, xB);
        for (int32_t e0 = 0; e0 < D; e0 += 32) {
            const int32_t r = rA, x = xA, c = cA;
            const unsigned starts = sA;
            const bool act = e0 + lane < D;
            int32_t cB = -1, rC = 0, xC = -1;
            unsigned sC;
            if (e0 + 32 + lane < D) cB = lab[xB];
            locate(e0 + 64, started, sC, rC, xC);
            rA = rB; xA = xB; cA = cB; sA = sB; rB = rC; xB = xC; sB = sC;
            p1_small_chunk(T, act, r, row_lanes(starts), x, c, cl_col, cl_lab, lane);
        }
        // lane `lane` finishes row `lane` of the tile
        if (have) p1_small_finish(T, v, d, cv, B, LG, rec, Lall, rsum, lane);
        __syncwarp();
    }
}

// The same tiles with the loads staged in shared memory by asynchronous copies
// (p1_stage = 1): lane l copies its row's columns (cp.async, 4 bytes each) to the tile's
// entry range [pre[l], pre[l+1]) and writes the entries' row number; after the wait the
// lanes copy the labels of those neighbours in the same way (a gather by cp.async);
// the chunks then read row, column and label from shared memory.  A warp keeps its
// tile's entries (at most 32 x 32) and their labels in flight at once instead of two
// chunks ahead.  Dynamic shared memory: kStageWarps x (SmallTile + SmallStage).
constexpr int kStageWarps = 4;
struct SmallStage {
    int32_t col[kSmallMax * 32];
    int32_t lab[kSmallMax * 32];
    uint8_t row[kSmallMax * 32];
};

__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

__global__ void __launch_bounds__(kStageWarps * 32) p1_small_staged_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ col, const int32_t *__restrict__ lab,
    const int32_t *__restrict__ rows, int64_t nrows, Batch B, const uint64_t *__restrict__ LG,
    NodeRec *__restrict__ rec, int32_t *__restrict__ Lall,
    RowSum *__restrict__ rsum, int32_t *__restrict__ cl_col, int32_t *__restrict__ cl_lab) {
    extern __shared__ __align__(16) unsigned char st_smem[];
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    SmallTile &T = reinterpret_cast<SmallTile *>(st_smem)[wid];
    SmallStage &S = reinterpret_cast<SmallStage *>(st_smem + kStageWarps * sizeof(SmallTile))[wid];
    int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t0 = warp * 32; t0 < nrows; t0 += nwarps * 32) {
        bool have;
        int32_t v, d, cv;
        const int32_t D = p1_small_setup<32>(T, off, lab, rows, nrows, t0, lane, have, v, d, cv);
        {
            const int32_t p0 = T.pre[lane];
            const int32_t *src = col + T.rb[lane];
            for (int32_t j = 0; j < d; ++j) {
                cp_async4(&S.col[p0 + j], src + j);
                S.row[p0 + j] = (uint8_t)lane;
            }
            cp_async_wait_all();
            __syncwarp();
            for (int32_t e = lane; e < D; e += 32) cp_async4(&S.lab[e], lab + S.col[e]);
            cp_async_wait_all();
            __syncwarp();
        }
        for (int32_t e0 = 0; e0 < D; e0 += 32) {
            const int32_t e = e0 + lane;
            const bool act = e < D;
            const int32_t r = act ? S.row[e] : 0, x = act ? S.col[e] : -1, c = act ? S.lab[e] : -1;
            p1_small_chunk(T, act, r, __match_any_sync(FULL, act ? r : -1), x, c, cl_col, cl_lab, lane);
        }
        if (have) p1_small_finish(T, v, d, cv, B, LG, rec, Lall, rsum, lane);
        __syncwarp();
    }
}

// Mid rows, one warp per row, a per-warp shared-memory table of kWarpCap slots.
constexpr int kMidWarps = kThreads / 32;

__global__ void __launch_bounds__(kThreads) p1_mid_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ col, const int32_t *__restrict__ lab,
    const int32_t *__restrict__ rows, int64_t nrows, Batch B, const uint64_t *__restrict__ LG,
    NodeRec *__restrict__ rec, int32_t *__restrict__ Lall, int *err,
    RowSum *__restrict__ rsum, int32_t *__restrict__ cl_col, int32_t *__restrict__ cl_lab,
    unsigned long long *wq) {
    __shared__ int32_t skey[kMidWarps][kWarpCap];
    __shared__ uint32_t scnt[kMidWarps][kWarpCap];
    __shared__ int16_t sused[kMidWarps][kWarpCap];    // slots taken by the current row
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (uint32_t j = lane; j < kWarpCap; j += 32) { skey[wid][j] = kEmpty; scnt[wid][j] = 0; }
    __syncwarp();
    for (int64_t i = warp_next(wq); i < nrows; i = warp_next(wq)) {
        int32_t v = rows[i];
        int64_t b = off[v];
        int d = (int)(off[v + 1] - b);
        int32_t cv = lab[v];
        int32_t gi = graph_of(B, v);
        uint32_t cap = dev_pow2_at_least(2u * (uint32_t)min(d, k_of(B, gi)));
        Tab t{skey[wid], scnt[wid], nullptr, nullptr, cap - 1};
        uint32_t own = 0, nused = 0;
        int32_t nx = 0;
        u128 X = 0;                       // foreign part, from count deltas at insert time
        // software pipeline: the next chunk's labels and the columns of the one after
        // it are loaded while the current chunk is inserted
        int32_t xA = lane < d ? col[b + lane] : -1;
        int32_t cA = lane < d ? lab[xA] : -1;
        int32_t xB = 32 + lane < d ? col[b + 32 + lane] : -1;
        for (int base = 0; base < d; base += 32) {
            int e = base + lane;
            bool act = e < d;
            const int32_t x = xA, c = cA;
            const int32_t cB = e + 32 < d ? lab[xB] : -1;
            const int32_t xC = e + 64 < d ? col[b + e + 64] : -1;
            xA = xB; cA = cB; xB = xC;
            own += (act && c == cv);
            bool foreign = act && c != cv;
            unsigned fm = __ballot_sync(FULL, foreign);
            bool lead = false, fresh = false;
            int sl = -1;
            if (foreign) {
                int64_t p = b + nx + __popc(fm & lanemask_lt());
                cl_col[p] = x;
                cl_lab[p] = c;
                unsigned grp = __match_any_sync(fm, c);
                lead = lane == __ffs(grp) - 1;
                if (lead) {
                    uint32_t old, g = __popc(grp);
                    sl = tab_insert_old(t, c, g, old, fresh, err);
                    X += (u128)(old + g) * LG[old + g] - (u128)old * LG[old];
                }
            }
            unsigned nm = __ballot_sync(FULL, fresh);
            if (fresh) sused[wid][nused + __popc(nm & lanemask_lt())] = (int16_t)sl;
            nused += __popc(nm);
            nx += __popc(fm);
        }
        __syncwarp();
        for (int o = 16; o; o >>= 1) own += __shfl_xor_sync(FULL, own, o);
        RowAgg a{(uint32_t)d, nused + (own > 0 ? 1u : 0u), warp_sum_u128(X) + (u128)own * LG[own]};
        float wcur = 0.0f;
        if (lane == 0) wcur = current_wmax(&B.wmax[gi]);
        wcur = __shfl_sync(FULL, wcur, 0);
        bool want_max = row_may_raise_max(a.L, wcur);
        df cm{0.0f, 0.0f}, wown{0.0f, 0.0f};
        if (want_max)
            for (uint32_t j = lane; j < nused; j += 32) cm = df_max(cm, column_weight(a, t.cnt[sused[wid][j]], LG));
        if (own > 0 && lane == 0) { wown = column_weight(a, own, LG); cm = df_max(cm, wown); }
        cm = warp_max_df(cm);
        if (lane == 0) {
            NodeRec r;
            df m = p1_row_result(a, own, cm, k_of(B, gi), LG, r, cv, wown, want_max);
            publish_max(B, gi, m, wcur);
            rec[v] = r;
            Lall[v] = (int32_t)a.L;
            store_rowsum(rsum, v, a);
        }
        __syncwarp();
        for (uint32_t j = lane; j < nused; j += 32) { int sl = sused[wid][j]; t.key[sl] = kEmpty; t.cnt[sl] = 0; }
        __syncwarp();
    }
}

// Large rows, one CTA per row, a per-CTA table of up to kMidCap slots
// CTA-ordered position of the flagged threads of one round; every thread calls
template <int NT>
__device__ __forceinline__ int32_t cta_rank(bool flag, int32_t &base, int32_t *sh_cnt) {
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned m = __ballot_sync(FULL, flag);
    if (lane == 0) sh_cnt[wid] = __popc(m);
    __syncthreads();
    int32_t p = base, tot = 0;
    for (int j = 0; j < NT / 32; ++j) {
        if (j < wid) p += sh_cnt[j];
        tot += sh_cnt[j];
    }
    p += __popc(m & lanemask_lt());
    base += tot;
    __syncthreads();
    return p;
}

template <int NT>
__global__ void __launch_bounds__(NT) p1_large_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ col, const int32_t *__restrict__ lab,
    const int32_t *__restrict__ rows, int64_t nrows, Batch B, const uint64_t *__restrict__ LG,
    NodeRec *__restrict__ rec, int32_t *__restrict__ Lall, int *err,
    RowSum *__restrict__ rsum, int32_t *__restrict__ cl_col, int32_t *__restrict__ cl_lab,
    unsigned long long *wq) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t sh_u32[NT / 32];
    __shared__ u128 sh_u128[NT / 32];
    __shared__ df sh_df[NT / 32];
    __shared__ int32_t sh_cnt[NT / 32];
    int tid = threadIdx.x, lane = tid & 31;
    __shared__ long long sh_next;
    for (int64_t i = cta_next(wq, &sh_next); i < nrows; i = cta_next(wq, &sh_next)) {
        int32_t v = rows[i];
        int64_t b = off[v];
        int d = (int)(off[v + 1] - b);
        int32_t cv = lab[v];
        int32_t gi = graph_of(B, v);
        uint32_t cap = dev_pow2_at_least(2u * (uint32_t)min(d, k_of(B, gi)));
        Tab t{(int32_t *)smem, (uint32_t *)(smem + 4 * cap), nullptr, nullptr, cap - 1};
        for (uint32_t j = tid; j < cap; j += NT) { t.key[j] = kEmpty; t.cnt[j] = 0; }
        __syncthreads();
        uint32_t own = 0;
        int32_t nx = 0;
        int32_t xA = tid < d ? col[b + tid] : -1;
        int32_t cA = tid < d ? lab[xA] : -1;
        int32_t xB = NT + tid < d ? col[b + NT + tid] : -1;
        for (int base = 0; base < d; base += NT) {
            int e = base + tid;
            bool act = e < d;
            const int32_t x = xA, c = cA;
            const int32_t cB = e + NT < d ? lab[xB] : -1;
            const int32_t xC = e + 2 * NT < d ? col[b + e + 2 * NT] : -1;
            xA = xB; cA = cB; xB = xC;
            own += (act && c == cv);
            bool foreign = act && c != cv;
            unsigned fm = __ballot_sync(FULL, foreign);
            if (foreign) {
                unsigned grp = __match_any_sync(fm, c);
                if (lane == __ffs(grp) - 1) tab_insert(t, c, __popc(grp), err);
            }
            int32_t p = cta_rank<NT>(foreign, nx, sh_cnt);
            if (foreign) { cl_col[b + p] = x; cl_lab[b + p] = c; }
        }
        own = block_sum_u32<NT>(own, sh_u32);      // syncs: the table is complete
        uint32_t Lf = 0;
        u128 X = 0;
        for (uint32_t j = tid; j < cap; j += NT)
            if (t.key[j] != kEmpty) { Lf++; X += (u128)t.cnt[j] * LG[t.cnt[j]]; }
        Lf = block_sum_u32<NT>(Lf, sh_u32);
        X = block_sum_u128<NT>(X, sh_u128);
        RowAgg a{(uint32_t)d, Lf + (own > 0 ? 1u : 0u), X + (u128)own * LG[own]};
        float wcur = current_wmax(&B.wmax[gi]);
        bool want_max = __syncthreads_or(row_may_raise_max(a.L, wcur));
        df cm{0.0f, 0.0f}, wown{0.0f, 0.0f};
        if (want_max)
            for (uint32_t j = tid; j < cap; j += NT)
                if (t.key[j] != kEmpty) cm = df_max(cm, column_weight(a, t.cnt[j], LG));
        if (own > 0) { wown = column_weight(a, own, LG); cm = df_max(cm, wown); }
        cm = block_max_df<NT>(cm, sh_df);
        if (tid == 0) {
            NodeRec r;
            df m = p1_row_result(a, own, cm, k_of(B, gi), LG, r, cv, wown, want_max);
            publish_max(B, gi, m, wcur);
            rec[v] = r;
            Lall[v] = (int32_t)a.L;
            store_rowsum(rsum, v, a);
        }
        __syncthreads();                              // table reuse
    }
}

// hub rows: chunks insert foreign communities into the row's global table
template <int NT>
__global__ void __launch_bounds__(NT) hub_p1_insert_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ col, const int32_t *__restrict__ lab,
    const HubInfo *__restrict__ hubs, const int32_t *__restrict__ items, const int32_t *__restrict__ chunks,
    int64_t nitems, int32_t chunk_len, int32_t *hkey, uint32_t *hcnt, HubAgg *hagg, int *err) {
    __shared__ uint32_t sh_u32[NT / 32];
    int tid = threadIdx.x, lane = tid & 31;
    for (int64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
        HubInfo h = hubs[items[it]];
        int64_t b = off[h.row];
        int64_t d = off[h.row + 1] - b;
        int64_t lo = (int64_t)chunks[it] * chunk_len;
        int64_t hi = min(d, lo + chunk_len);
        int32_t cv = lab[h.row];
        Tab t{hkey + h.tab, hcnt + h.tab, nullptr, nullptr, (uint32_t)h.cap - 1};
        uint32_t own = 0;
        for (int64_t base = lo; base < hi; base += NT) {
            int64_t e = base + tid;
            bool act = e < hi;
            int32_t c = act ? lab[col[b + e]] : -1;
            own += (act && c == cv);
            bool foreign = act && c != cv;
            unsigned fm = __ballot_sync(FULL, foreign);
            if (foreign) {
                unsigned grp = __match_any_sync(fm, c);
                if (lane == __ffs(grp) - 1) tab_insert(t, c, __popc(grp), err);
            }
        }
        own = block_sum_u32<NT>(own, sh_u32);
        if (tid == 0 && own) atomicAdd(&hagg[items[it]].own, own);
        __syncthreads();
    }
}

// hub rows, P1 step 2: each slot range of a hub's table adds its foreign groups and
// their sum f LG[f] to the hub's aggregates (exact integer sums, so any order gives the
// same bits)
template <int NT>
__global__ void __launch_bounds__(NT) hub_p1_sums_kernel(
    const HubInfo *__restrict__ hubs, const int32_t *__restrict__ sitem, const int32_t *__restrict__ srange,
    int64_t nsitems, const uint64_t *__restrict__ LG, const int32_t *hkey, const uint32_t *hcnt, HubAgg *hagg) {
    __shared__ uint32_t sh_u32[NT / 32];
    __shared__ u128 sh_u128[NT / 32];
    for (int64_t it = blockIdx.x; it < nsitems; it += gridDim.x) {
        const int32_t hi = sitem[it];
        const HubInfo h = hubs[hi];
        const int64_t j0 = (int64_t)srange[it] * kHubSlotRange, j1 = min((int64_t)h.cap, j0 + (int64_t)kHubSlotRange);
        uint32_t Lf = 0;
        u128 X = 0;
        for (int64_t j = j0 + threadIdx.x; j < j1; j += NT) {
            const int64_t s = h.tab + j;
            if (hkey[s] != kEmpty) {
                const uint32_t c = hcnt[s];
                Lf++;
                X += (u128)c * LG[c];
            }
        }
        Lf = block_sum_u32<NT>(Lf, sh_u32);
        X = block_sum_u128<NT>(X, sh_u128);
        if (threadIdx.x == 0) {
            if (Lf) atomicAdd(&hagg[hi].L, Lf);
            if (X) atomic_add_u128(reinterpret_cast<unsigned long long *>(&hagg[hi].X), X);
        }
        __syncthreads();                               // the reductions' words are reused
    }
}

// hub rows, P1 step 3, a thread per hub: the row aggregates with the own community, the
// own and absent columns' weights (published to w_max), the node record
template <int NT>
__global__ void __launch_bounds__(NT) hub_p1_finish_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ lab, const HubInfo *__restrict__ hubs,
    int64_t nhubs, Batch B, const uint64_t *__restrict__ LG, HubAgg *hagg, NodeRec *__restrict__ rec,
    int32_t *__restrict__ Lall) {
    for (int64_t hi = (int64_t)blockIdx.x * NT + threadIdx.x; hi < nhubs; hi += (int64_t)gridDim.x * NT) {
        const HubInfo h = hubs[hi];
        const int32_t gi = graph_of(B, h.row);
        const int64_t d = off[h.row + 1] - off[h.row];
        HubAgg g = hagg[hi];
        const uint32_t own = g.own;
        const RowAgg a{(uint32_t)d, g.L + (own > 0 ? 1u : 0u), g.X + (u128)own * LG[own]};
        df wown{0.0f, 0.0f};
        if (own > 0) wown = column_weight(a, own, LG);
        NodeRec r;
        const df m = p1_row_result(a, own, wown, k_of(B, gi), LG, r, lab[h.row], wown, true);
        publish_max(B, gi, m, current_wmax(&B.wmax[gi]));
        rec[h.row] = r;
        Lall[h.row] = (int32_t)a.L;
        g.X = a.X;
        g.L = a.L;
        hagg[hi] = g;
    }
}

// hub rows, P1 step 4: the weight of every foreign column of each slot range, its cube root
// sigma kept for P2 (a column's weight depends only on the row's aggregates and its count,
// both final here), and the range's largest weight to w_max (a maximum, so the order of
// the ranges does not matter).  A positive sigma is stored negated when the column has a
// single member (no Type-II push to make), so that P2 reads one word instead of two; the
// sign change is exact, and a zero sigma (no push either) stays +0.
template <int NT>
__global__ void __launch_bounds__(NT) hub_p1_colmax_kernel(
    const int64_t *__restrict__ off, const HubInfo *__restrict__ hubs, const int32_t *__restrict__ sitem,
    const int32_t *__restrict__ srange, int64_t nsitems, Batch B, const uint64_t *__restrict__ LG,
    const int32_t *hkey, const uint32_t *hcnt, const HubAgg *__restrict__ hagg, df *hsig) {
    __shared__ df sh_df[NT / 32];
    for (int64_t it = blockIdx.x; it < nsitems; it += gridDim.x) {
        const int32_t hi = sitem[it];
        const HubInfo h = hubs[hi];
        const HubAgg g = hagg[hi];
        const RowAgg a{(uint32_t)(off[h.row + 1] - off[h.row]), g.L, g.X};
        const int64_t j0 = (int64_t)srange[it] * kHubSlotRange, j1 = min((int64_t)h.cap, j0 + (int64_t)kHubSlotRange);
        df cm{0.0f, 0.0f};
        for (int64_t j = j0 + threadIdx.x; j < j1; j += NT) {
            const int64_t s = h.tab + j;
            if (hkey[s] != kEmpty) {
                const df w = column_weight(a, hcnt[s], LG);
                cm = df_max(cm, w);
                const df sg = df_cbrt(w);
                hsig[s] = (hcnt[s] > 1 || !(sg.hi > 0.0f)) ? sg : df{-sg.hi, -sg.lo};
            }
        }
        cm = block_max_df<NT>(cm, sh_df);
        if (threadIdx.x == 0) {
            const int32_t gi = graph_of(B, h.row);
            publish_max(B, gi, cm, current_wmax(&B.wmax[gi]));
        }
        __syncthreads();                               // the reduction's words are reused
    }
}

// ======================================================================================
// P2 row lists by cross degree (known after P1): each P2 kernel then walks only its rows
//   0 mid and large rows, dx <= 32 (tiles)
//   1 mid rows, and large rows with dx <= dx_cta, 32 < dx <= 128 (p2_mid: a warp per row)
//   2 the same with dx > 128 (p2_large of kP2SmallCta threads)
//   3 large rows, dx > dx_cta (p2_large)
// ======================================================================================
constexpr int kP2Lists = 4;
constexpr int32_t kP2WarpDx = 128;            // a warp keeps a row of this cross degree in registers
constexpr int kP2SmallCta = 256;

__device__ __forceinline__ void append_row(int32_t *list, int32_t *cnt, bool take, int32_t v) {
    unsigned m = __ballot_sync(FULL, take);
    int lane = threadIdx.x & 31;
    int32_t base = 0;
    if (m && lane == __ffs(m) - 1) base = atomicAdd(cnt, __popc(m));
    base = __shfl_sync(FULL, base, __ffs(m ? m : 1u) - 1);
    if (take) list[base + __popc(m & lanemask_lt())] = v;
}

// every list has room for all mid and large rows
struct P2Split {
    const int32_t *rows_mid, *rows_large;
    int64_t n_mid, n_large;
    int32_t dx_cta;
    int32_t *lists, *cnt;
};
__host__ __device__ __forceinline__ int64_t p2_list_start(int c, int64_t n_mid, int64_t n_large) {
    return c * (n_mid + n_large);
}
__device__ __forceinline__ void p2_split(const P2Split &A, const NodeRec *rec, int block, int blocks) {
    const int64_t total = A.n_mid + A.n_large;
    for (int64_t i0 = (int64_t)block * blockDim.x; i0 < total; i0 += (int64_t)blocks * blockDim.x) {
        const int64_t i = i0 + threadIdx.x;
        const bool act = i < total, mid = i < A.n_mid;
        const int32_t v = act ? (mid ? A.rows_mid[i] : A.rows_large[i - A.n_mid]) : 0;
        const int32_t dx = act ? rec[v].dx : 0;
        const int cls = !act ? -1 : dx <= 32 ? 0 : !mid && dx > A.dx_cta ? 3 : dx <= kP2WarpDx ? 1 : 2;
        for (int c = 0; c < kP2Lists; ++c)
            append_row(A.lists + p2_list_start(c, A.n_mid, A.n_large), A.cnt + c, cls == c, v);
    }
}

// ======================================================================================
// G_x row offsets: nodes with dx >= 2 keep dx slots; xoff is the exclusive scan of
// those capacities, in one pass (decoupled look-back).  Tiles of kGxTile nodes are
// taken in ticket order; a tile publishes its own total at once and its inclusive
// prefix as soon as the tiles before it have, and its first warp sums the published
// words of its predecessors back to the nearest inclusive one, 32 tiles per step.  A predecessor has
// always started (its ticket is smaller), so every wait ends; the wait is bounded
// all the same (spin_limit reads of a word).  If the bound is ever reached, the tile
// flags err (bit 32, reported by rs_score as RS_ETIMEOUT) and takes its prefix from a
// direct sum of the capacities of every node before it instead, so the offsets stay
// exact.  withhold_tile >= 0 (a test hook, -1 otherwise) keeps that tile from
// publishing its words, so that the waits of the tiles after it run out.
// ======================================================================================
constexpr int kGxThreads = 256;
constexpr int kGxPer = kGxTile / kGxThreads;
constexpr unsigned long long kGxAgg = 1ull << 62, kGxIncl = 2ull << 62, kGxMask = (1ull << 62) - 1;

// status: one word per tile (flag in the top two bits), zeroed before the launch;
// ticket: zeroed before the launch.  Warp w of a tile scans its kGxPer runs of 32
// consecutive nodes (coalesced loads and stores), carrying its running total.
__global__ void __launch_bounds__(kGxThreads) gx_offsets_kernel(
    const NodeRec *__restrict__ rec, int64_t n, int64_t *__restrict__ xoff, unsigned long long *status,
    unsigned long long *ticket, int *err, long spin_limit, int64_t withhold_tile, int32_t *__restrict__ cover,
    int32_t *last, P2Split split, int split_blocks) {
    chain_wait();
    if ((int)blockIdx.x < split_blocks) {              // the P2 row lists, by blocks of their own
        p2_split(split, rec, blockIdx.x, split_blocks);
        return;
    }
    __shared__ int64_t warp_tot[kGxThreads / 32];
    __shared__ unsigned long long sh_tile;
    __shared__ int64_t sh_prefix;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) sh_tile = atomicAdd(ticket, 1ull);
    __syncthreads();
    const int64_t t = (int64_t)sh_tile;
    const int64_t base = t * kGxTile + (int64_t)wid * (32 * kGxPer);
    int32_t cap[kGxPer];
#pragma unroll
    for (int k = 0; k < kGxPer; ++k) {
        int64_t v = base + k * 32 + lane;
        int32_t dx = v < n ? rec[v].dx : 0;
        cap[k] = dx >= 2 ? dx : 0;
    }
    int64_t val[kGxPer];
    int64_t carry = 0;
#pragma unroll
    for (int k = 0; k < kGxPer; ++k) {
        int64_t x = cap[k];
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        val[k] = carry + x;                           // inclusive within the warp's nodes
        carry += __shfl_sync(FULL, x, 31);
    }
    if (lane == 0) warp_tot[wid] = carry;
    __syncthreads();
    if (wid == 0) {
        // exclusive prefixes of the warps inside the tile, and the tile's total
        int64_t c = lane < kGxThreads / 32 ? warp_tot[lane] : 0, x = c;
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        const int64_t total = __shfl_sync(FULL, x, 31);
        if (lane < kGxThreads / 32) warp_tot[lane] = x - c;
        int64_t excl = 0;
        const bool publish = t != withhold_tile;
        if (t == 0) {
            if (lane == 0 && publish) *(volatile unsigned long long *)&status[0] = kGxIncl | (unsigned long long)total;
        } else {
            if (lane == 0 && publish) *(volatile unsigned long long *)&status[t] = kGxAgg | (unsigned long long)total;
            // look back 32 tiles at a time: lane l reads tile hi - l; the nearest
            // inclusive word ends the walk, the aggregates after it are added
            bool gave_up = false;
            for (int64_t hi = t - 1;; hi -= 32) {
                const int64_t j = hi - lane;
                unsigned long long w = kGxIncl;          // before tile 0: an inclusive zero
                if (j >= 0) {
                    long spins = 0;
                    do {
                        w = *(volatile unsigned long long *)&status[j];
                    } while (!(w >> 62) && ++spins < spin_limit);
                }
                if (__any_sync(FULL, !(w >> 62))) {     // a wait ran out
                    gave_up = true;
                    break;
                }
                const unsigned inc = __ballot_sync(FULL, (w >> 62) == 2);
                const int stop = inc ? __ffs(inc) - 1 : 31;
                int64_t add = lane <= stop ? (int64_t)(w & kGxMask) : 0;
                for (int o = 16; o; o >>= 1) add += __shfl_xor_sync(FULL, add, o);
                excl += add;
                if (inc) break;
            }
            if (gave_up) {
                // the exact prefix from the node records themselves
                if (lane == 0) atomicOr(err, 32);
                int64_t sum = 0;
                for (int64_t v = lane; v < t * kGxTile; v += 32) {
                    const int32_t dx = rec[v].dx;
                    sum += dx >= 2 ? dx : 0;
                }
                for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
                excl = sum;
            }
            if (lane == 0 && publish)
                *(volatile unsigned long long *)&status[t] = kGxIncl | (unsigned long long)(excl + total);
        }
        if (lane == 0) sh_prefix = excl;
    }
    __syncthreads();
    const int64_t before = sh_prefix + warp_tot[wid];
    int32_t own_last = -1;                            // the warp's last node with slots
    if (t == 0 && threadIdx.x == 0) xoff[0] = 0;
#pragma unroll
    for (int k = 0; k < kGxPer; ++k) {
        int64_t v = base + k * 32 + lane;
        const int64_t hi = before + val[k], lo = hi - cap[k];
        if (v < n) xoff[v + 1] = hi;
        // the mirror's tiles that start in v's slots (every slot lies in exactly one row)
        if (cover && cap[k] > 0)
            for (int64_t m = (lo + kMirTile - 1) / kMirTile; m * kMirTile < hi; ++m) cover[m] = (int32_t)v;
        const unsigned some = __ballot_sync(FULL, cap[k] > 0);
        if (some) own_last = (int32_t)(base + k * 32 + 31 - __clz(some));
    }
    if (cover && lane == 0 && own_last >= 0) atomicMax(last, own_last);
}

// ======================================================================================
// P2
// ======================================================================================
// P2 for small and mid rows walks the cross list P1 wrote (the neighbours of
// another community, in id order) and the row aggregates; own-community
// neighbours are never touched again.

constexpr int kNarrowRows = 8;                 // rows per tile of the narrow mid and large rows

// Rows with at most 32 cross neighbours, tiles of R <= 32 consecutive rows of a list
// per warp (the small rows, R = 32, and the mid and large rows with dx <= 32, whose
// longer cross lists take smaller tiles so that more warps share them).  The
// union of the tile's cross lists is processed in chunks of whole rows, one
// entry per lane (a chunk ends before the first row that would not fit its 32
// lanes); lane l prepares and closes row l.  As no row spans two chunks, a
// community's count f and Type-II sum come from one warp match on
// (row, community).
// one G_x slot p of a row: its id and value, and for the first slot of an 8-slot sector of
// the slot space also the packed index entry xsk[p / 8] (searches of long out-lists read it;
// every slot inside a row is written once here, so the entries of sectors starting inside
// rows are complete when P2 ends)
// (the P2 kernels are compiled for both kinds of slots: a stride in bytes, known to the launch only,
// took 0.6% of a batch of 256 graphs)
__device__ __forceinline__ void put_sig(SigPair *xS, int64_t p, uint64_t sig) { xS[p].f = sig; }
__device__ __forceinline__ void put_sig(uint64_t *xS, int64_t p, uint64_t sig) { xS[p] = sig; }
template <class Slot>
__device__ __forceinline__ void gx_put(int32_t *xcol, Slot *xS, int32_t *xsk, int64_t p, int32_t u, uint64_t sig) {
    xcol[p] = u;
    put_sig(xS, p, sig);
    if ((p & 7) == 0) xsk[p >> 3] = u;
}

// what P3 needs of a G_x node at once: one 16-byte load instead of three random ones
__device__ __forceinline__ GxNode load_node(const GxNode *xnode, int32_t v) {
    const longlong2 x = __ldg(reinterpret_cast<const longlong2 *>(xnode + v));
    return GxNode{x.x, (int32_t)(uint32_t)(unsigned long long)x.y, (int32_t)(uint32_t)((unsigned long long)x.y >> 32)};
}

struct P2Tile {
    int32_t pre[33];            // prefix sums of dx over the tile
    uint8_t row[32];            // the tile's rows with entries, in order
    int64_t rb[32], xb[32];     // cross list start (= CSR start), G_x row start
    int32_t dx[32], w[32];
    uint32_t d[32], L[32];
    uint64_t xlo[32], xhi[32];
    uint64_t sig1[32];          // sigma of a column with one member, fixed point
    int32_t no[32], ni[32];
    uint64_t st[32];
};

template <int R, class Slot>
__global__ void __launch_bounds__(kThreads) p2_small_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ rows, int64_t nrows_host,
    const int32_t *__restrict__ nrows_dev, const uint64_t *__restrict__ LG, const NodeRec *__restrict__ rec, const RowSum *__restrict__ rsum,
    const int32_t *__restrict__ cl_col, const int32_t *__restrict__ cl_lab, unsigned long long *acc,
    const int64_t *__restrict__ xoff, int32_t *__restrict__ xcol, Slot *__restrict__ xS, int32_t *__restrict__ xsk,
    int32_t *__restrict__ xout, int32_t *__restrict__ xin, GxNode *__restrict__ xnode, Strict SX) {
    chain_wait();
    __shared__ P2Tile tiles[kThreads / 32];
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    P2Tile &T = tiles[wid];
    int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t nrows = nrows_dev ? *nrows_dev : nrows_host;   // a list counted by p2_split, or the small rows
    for (int64_t t0 = warp * R; t0 < nrows; t0 += nwarps * R) {
        int64_t i = t0 + lane;
        bool have = lane < R && i < nrows;
        int32_t w = have ? rows[i] : 0;
        int32_t dx = 0;
        if (have) {
            int64_t b = off[w];
            NodeRec rw = rec[w];
            dx = rw.dx;
            T.rb[lane] = b;
            T.d[lane] = (uint32_t)(off[w + 1] - b);
            T.w[lane] = w;
            if (dx > 0) {
                RowSum rs = rsum[w];
                T.xlo[lane] = rs.xlo; T.xhi[lane] = rs.xhi; T.L[lane] = rs.L;
                RowAgg a{T.d[lane], rs.L, ((u128)rs.xhi << 64) | rs.xlo};
                T.sig1[lane] = sig_fixed(df_cbrt(column_weight(a, 1, LG)));
                T.xb[lane] = xoff[w];
            }
        }
        T.dx[lane] = dx;
        T.no[lane] = 0;
        T.ni[lane] = 0;
        int32_t incl = dx;
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        int32_t DX = __shfl_sync(FULL, incl, 31);
        T.pre[lane + 1] = incl;
        if (lane == 0) T.pre[0] = 0;
        const unsigned some = __ballot_sync(FULL, dx > 0);
        if (dx > 0) T.row[__popc(some & lanemask_lt())] = (uint8_t)lane;
        int started = 0;                               // rows that start before the chunk
        __syncwarp();
        for (int32_t e0 = 0; e0 < DX;) {
            // rows [.., rb) end within e0 + 32: the chunk is [e0, pre[rb])
            unsigned fit = __ballot_sync(FULL, incl <= e0 + 32);
            int32_t rb = 32 - __clz(fit);
            int32_t E = __shfl_sync(FULL, incl, rb - 1);
            int32_t e = e0 + lane;
            bool act = e < E;
            int32_t r = 0, u = -1, c = -1, j = 0;
            NodeRec ru{0, -1, 0};
            const int32_t q = incl - dx - e0;
            const unsigned starts = __reduce_or_sync(FULL, dx > 0 && q >= 0 && e0 + q < E ? 1u << q : 0u);
            const unsigned lanes = row_lanes(starts);
            if (act) {
                r = T.row[started + rows_started(starts) - 1];
                j = e - T.pre[r];
                u = cl_col[T.rb[r] + j];
                c = cl_lab[T.rb[r] + j];
                ru = rec[u];
            }
            T.st[lane] = ru.s_fix;
            __syncwarp();
            started += __popc(starts);
            unsigned am = __ballot_sync(FULL, act);
            unsigned gc = 0;
            if (act) gc = __match_any_sync(am, c) & lanes;
            uint64_t sf = 0;
            if (act) {
                uint32_t f = __popc(gc);
                u128 rest = 0;
                if (f > 1) {
                    unsigned m = gc & ~(1u << lane);
                    while (m) { rest += T.st[__ffs(m) - 1]; m &= m - 1; }
                }
                if (f == 1) sf = T.sig1[r];
                else {
                    RowAgg a{T.d[r], T.L[r], ((u128)T.xhi[r] << 64) | T.xlo[r]};
                    const df sig = df_cbrt(column_weight(a, f, LG));
                    sf = sig_fixed(sig);
                    push_type2(acc, u, sig, strict_rest(SX, off, T.w[r], u, rest));
                }
            }
            // G_x entries of this chunk, in id order within each row
            bool gx = act && T.dx[r] >= 2 && ru.dx >= 2;
            bool o = gx && rank_after(ru.dx, u, T.dx[r], T.w[r]);
            bool in = gx && !o;
            const unsigned go = __ballot_sync(FULL, o) & lanes, gi = __ballot_sync(FULL, in) & lanes;
            int32_t bo = o ? T.no[r] : 0, bi = in ? T.ni[r] : 0;
            __syncwarp();
            if (o) {
                int64_t p = T.xb[r] + bo + __popc(go & lanemask_lt());
                gx_put(xcol, xS, xsk, p, u, sf);
                if (lane == __ffs(go) - 1) T.no[r] = bo + __popc(go);
            }
            if (in) {
                int64_t p = T.xb[r] + T.dx[r] - 1 - (bi + __popc(gi & lanemask_lt()));
                gx_put(xcol, xS, xsk, p, u, sf);
                if (lane == __ffs(gi) - 1) T.ni[r] = bi + __popc(gi);
            }
            __syncwarp();
            e0 = E;
        }
        if (have) { xout[w] = T.no[lane]; xin[w] = T.ni[lane]; xnode[w] = GxNode{T.xb[lane], T.no[lane], dx}; }
        __syncwarp();
    }
}

// Mid rows, one warp per row: a per-warp table (community -> count, Type-II
// sum) over the cross list, then the terms and the G_x entries in id order.
//
// A row has at most kP2WarpDx cross neighbours, so its list and their records are loaded at
// once into registers (kP2Per entries per lane), and an entry's table slot is kept from the
// insertion for the terms: the loads of a row are two dependent steps.  With the list read
// chunk by chunk, twice, and the table searched again, a row of 129-256 neighbours took up to
// 50 us of one warp, the end of the whole phase on small graphs; those rows now take a CTA.
constexpr int kP2Per = kP2WarpDx / 32;
constexpr int kP2MidSlots = 2 * kP2WarpDx, kMidSlotBytes = 4 + 4 + 16;   // key, count, 2-word sum
constexpr size_t kP2MidSmem = (size_t)kMidWarps * kP2MidSlots * kMidSlotBytes;

template <class Slot>
__global__ void __launch_bounds__(kThreads) p2_mid_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ rows, const int32_t *__restrict__ nrows_dev, Batch B,
    const uint64_t *__restrict__ LG, const NodeRec *__restrict__ rec, const RowSum *__restrict__ rsum,
    const int32_t *__restrict__ cl_col, const int32_t *__restrict__ cl_lab, unsigned long long *acc,
    const int64_t *__restrict__ xoff, int32_t *__restrict__ xcol, Slot *__restrict__ xS, int32_t *__restrict__ xsk,
    int32_t *__restrict__ xout, int32_t *__restrict__ xin, GxNode *__restrict__ xnode, int *err, Strict SX, unsigned long long *wq) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t stage[kThreads];
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t *st = stage + (threadIdx.x & ~31);
    unsigned char *base_w = smem + (size_t)wid * kP2MidSlots * kMidSlotBytes;
    const int64_t nrows = *nrows_dev;               // rows of this kernel, counted by p2_split
    for (int64_t i = warp_next(wq); i < nrows; i = warp_next(wq)) {
        const int32_t w = rows[i];
        const int64_t b = off[w];
        const int d = (int)(off[w + 1] - b);
        const int dx = rec[w].dx;
        const int64_t xb = xoff[w];
        const RowSum rs = rsum[w];
        int32_t u[kP2Per], c[kP2Per], sl[kP2Per], udx[kP2Per];
        uint64_t s[kP2Per];
#pragma unroll
        for (int j = 0; j < kP2Per; ++j) {
            const int e = 32 * j + lane;
            u[j] = e < dx ? cl_col[b + e] : -1;
            c[j] = e < dx ? cl_lab[b + e] : -1;
        }
        const uint32_t cap = dev_pow2_at_least(2u * (uint32_t)min(dx, k_of(B, graph_of(B, w))));
        Tab t;
        t.q = (unsigned long long *)base_w;
        t.key = (int32_t *)(base_w + 16 * kP2MidSlots);
        t.cnt = (uint32_t *)(base_w + 20 * kP2MidSlots);
        t.sig = nullptr;
        t.mask = cap - 1;
        for (uint32_t j = lane; j < cap; j += 32) { t.key[j] = kEmpty; t.cnt[j] = 0; t.q[2 * j] = 0; t.q[2 * j + 1] = 0; }
#pragma unroll
        for (int j = 0; j < kP2Per; ++j) {
            NodeRec r{0, -1, 0};
            if (u[j] >= 0) r = rec[u[j]];
            s[j] = r.s_fix;
            udx[j] = r.dx;
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kP2Per; ++j) {
            sl[j] = -1;
            if (32 * j < dx) {
                const bool act = u[j] >= 0;
                st[lane] = s[j];
                __syncwarp();
                const unsigned am = __ballot_sync(FULL, act);
                if (act) {
                    const unsigned grp = __match_any_sync(am, c[j]);
                    const int leader = __ffs(grp) - 1;
                    int q = -1;
                    if (lane == leader) {
                        q = tab_insert(t, c[j], __popc(grp), err);
                        if (q >= 0) atomic_add_u128(t.q + 2 * q, group_sum_all(st, grp));
                    }
                    sl[j] = __shfl_sync(grp, q, leader);
                }
                __syncwarp();
            }
        }
        const RowAgg a{(uint32_t)d, rs.L, ((u128)rs.xhi << 64) | rs.xlo};
        const uint64_t sig1 = sig_fixed(df_cbrt(column_weight(a, 1, LG)));   // the usual count of a foreign community
        int32_t bo = 0, bi = 0;
#pragma unroll
        for (int j = 0; j < kP2Per; ++j) {
            if (32 * j < dx) {
                uint64_t sf = sig1;
                const bool ok = sl[j] >= 0;
                if (ok) {
                    const uint32_t f = t.cnt[sl[j]];
                    if (f > 1) {
                        const df sig = df_cbrt(column_weight(a, f, LG));
                        sf = sig_fixed(sig);
                        const u128 q = ((u128)t.q[2 * sl[j] + 1] << 64) | t.q[2 * sl[j]];
                        push_type2(acc, u[j], sig, strict_rest(SX, off, w, u[j], q - s[j]));
                    }
                }
                const bool inx = ok && udx[j] >= 2;
                const bool o = inx && rank_after(udx[j], u[j], dx, w);
                const bool in = inx && !o;
                const unsigned mo = __ballot_sync(FULL, o), mi = __ballot_sync(FULL, in);
                if (o) gx_put(xcol, xS, xsk, xb + bo + __popc(mo & lanemask_lt()), u[j], sf);
                if (in) gx_put(xcol, xS, xsk, xb + dx - 1 - (bi + __popc(mi & lanemask_lt())), u[j], sf);
                bo += __popc(mo); bi += __popc(mi);
            }
        }
        if (lane == 0) { xout[w] = bo; xin[w] = bi; xnode[w] = GxNode{xb, bo, dx}; }
        __syncwarp();
    }
}

// slot layout of the P2 tables: key[cap] | cnt[cap] | q[2 cap] | sig[cap]  (32 B per slot)
__device__ __forceinline__ Tab p2_table(unsigned char *base, uint32_t cap) {
    Tab t;
    t.q = (unsigned long long *)base;
    t.sig = (df *)(base + 16 * (size_t)cap);
    t.key = (int32_t *)(base + 24 * (size_t)cap);
    t.cnt = (uint32_t *)(base + 28 * (size_t)cap);
    t.mask = cap - 1;
    return t;
}

// CTA-ordered compaction of the G_x entries of one round; returns this thread's position
template <int NT, class Slot>
__device__ __forceinline__ void gx_round(bool out, bool in, int64_t xb, int32_t dxw, int32_t u, uint64_t sig,
                                         int32_t &base_out, int32_t &base_in, int32_t *xcol, Slot *xS,
                                         int32_t *xsk, int32_t *sh_cnt /* 2 * NT/32 */) {
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned mo = __ballot_sync(FULL, out), mi = __ballot_sync(FULL, in);
    if (lane == 0) { sh_cnt[wid] = __popc(mo); sh_cnt[NT / 32 + wid] = __popc(mi); }
    __syncthreads();
    int32_t po = base_out, pi = base_in, to = 0, ti = 0;
    for (int j = 0; j < NT / 32; ++j) {
        if (j < wid) { po += sh_cnt[j]; pi += sh_cnt[NT / 32 + j]; }
        to += sh_cnt[j]; ti += sh_cnt[NT / 32 + j];
    }
    if (out) gx_put(xcol, xS, xsk, xb + po + __popc(mo & lanemask_lt()), u, sig);
    if (in) gx_put(xcol, xS, xsk, xb + dxw - 1 - (pi + __popc(mi & lanemask_lt())), u, sig);
    base_out += to; base_in += ti;
    __syncthreads();
}

template <int NT, class Slot>
__global__ void __launch_bounds__(NT) p2_large_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ rows, const int32_t *__restrict__ nrows_dev, Batch B,
    const uint64_t *__restrict__ LG, const NodeRec *__restrict__ rec, const RowSum *__restrict__ rsum,
    const int32_t *__restrict__ cl_col, const int32_t *__restrict__ cl_lab, unsigned long long *acc,
    const int64_t *__restrict__ xoff, int32_t *__restrict__ xcol, Slot *__restrict__ xS, int32_t *__restrict__ xsk,
    int32_t *__restrict__ xout, int32_t *__restrict__ xin, GxNode *__restrict__ xnode, int *err, Strict SX, unsigned long long *wq) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int32_t sh_cnt[2 * NT / 32];
    __shared__ uint64_t stage[NT];
    int tid = threadIdx.x, lane = tid & 31;
    uint64_t *st = stage + (tid & ~31);
    const int64_t nrows = *nrows_dev;               // rows of this kernel, counted by p2_split
    __shared__ long long sh_next;
    for (int64_t i = cta_next(wq, &sh_next); i < nrows; i = cta_next(wq, &sh_next)) {
        int32_t w = rows[i];
        int64_t b = off[w];
        int d = (int)(off[w + 1] - b);
        NodeRec rw = rec[w];
        int dx = rw.dx;
        uint32_t cap = dev_pow2_at_least(2u * (uint32_t)min(dx, k_of(B, graph_of(B, w))));
        Tab t = p2_table(smem, cap);
        for (uint32_t j = tid; j < cap; j += NT) {
            t.key[j] = kEmpty; t.cnt[j] = 0; t.q[2 * j] = 0; t.q[2 * j + 1] = 0;
        }
        __syncthreads();
        for (int base = 0; base < dx; base += NT) {
            int e = base + tid;
            bool act = e < dx;
            int32_t c = act ? cl_lab[b + e] : -1;
            st[lane] = act ? rec[cl_col[b + e]].s_fix : 0;
            __syncwarp();
            unsigned am = __ballot_sync(FULL, act);
            if (act) {
                unsigned grp = __match_any_sync(am, c);
                if (lane == __ffs(grp) - 1) {
                    int sl = tab_insert(t, c, __popc(grp), err);
                    if (sl >= 0) atomic_add_u128(t.q + 2 * sl, group_sum_all(st, grp));
                }
            }
            __syncwarp();
        }
        __syncthreads();
        RowSum rs = rsum[w];
        RowAgg a{(uint32_t)d, rs.L, ((u128)rs.xhi << 64) | rs.xlo};
        for (uint32_t j = tid; j < cap; j += NT)
            if (t.key[j] != kEmpty) t.sig[j] = df_cbrt(column_weight(a, t.cnt[j], LG));
        __syncthreads();
        int64_t xb = xoff[w];
        int32_t bo = 0, bi = 0;
        for (int base = 0; base < dx; base += NT) {
            int e = base + tid;
            bool act = e < dx;
            int32_t u = act ? cl_col[b + e] : -1;
            NodeRec ru{0, -1, 0};
            if (act) ru = rec[u];
            bool ok = act;
            df sig{0.0f, 0.0f};
            if (act) {
                int sl = tab_find(t, cl_lab[b + e]);
                if (sl < 0) { atomicOr(err, 2); ok = false; }
                else {
                    sig = t.sig[sl];
                    if (t.cnt[sl] > 1) {
                        u128 q = ((u128)t.q[2 * sl + 1] << 64) | t.q[2 * sl];
                        push_type2(acc, u, sig, strict_rest(SX, off, w, u, q - ru.s_fix));
                    }
                }
            }
            if (dx >= 2) {
                bool inx = ok && ru.dx >= 2;
                bool o = inx && rank_after(ru.dx, u, dx, w);
                gx_round<NT>(o, inx && !o, xb, dx, u, inx ? sig_fixed(sig) : 0, bo, bi, xcol, xS, xsk, sh_cnt);
            }
        }
        if (tid == 0) { xout[w] = bo; xin[w] = bi; xnode[w] = GxNode{xb, bo, dx}; }
        __syncthreads();
    }
}

// hub rows, P2 step 1: Type-II group sums and per-chunk G_x counts; every entry's table slot
// (found once per group of lanes with the same community) is kept for step 3
template <int NT>
__global__ void __launch_bounds__(NT) hub_p2_insert_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ col, const HubInfo *__restrict__ hubs,
    const int32_t *__restrict__ items, const int32_t *__restrict__ chunks, int64_t nitems, int32_t chunk_len,
    const NodeRec *__restrict__ rec, const int32_t *hkey, unsigned long long *hq,
    int32_t *hitem_out, int32_t *hitem_in, int32_t *__restrict__ hslot, int *err) {
    __shared__ uint32_t sh_u32[NT / 32];
    __shared__ uint64_t stage[NT];
    int tid = threadIdx.x, lane = tid & 31;
    uint64_t *st = stage + (tid & ~31);
    for (int64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
        HubInfo h = hubs[items[it]];
        int64_t b = off[h.row];
        int64_t d = off[h.row + 1] - b;
        int64_t lo = (int64_t)chunks[it] * chunk_len;
        int64_t hi = min(d, lo + chunk_len);
        NodeRec rw = rec[h.row];
        Tab t{(int32_t *)hkey + h.tab, nullptr, hq + 2 * h.tab, nullptr, (uint32_t)h.cap - 1};
        uint32_t no = 0, ni = 0;
        for (int64_t base = lo; base < hi; base += NT) {
            int64_t e = base + tid;
            bool act = e < hi;
            int32_t u = act ? col[b + e] : -1;
            NodeRec ru{0, -1, 0};
            if (act) ru = rec[u];
            bool foreign = act && ru.label != rw.label;
            st[lane] = ru.s_fix;
            __syncwarp();
            unsigned fm = __ballot_sync(FULL, foreign);
            if (foreign) {
                unsigned grp = __match_any_sync(fm, ru.label);
                const int leader = __ffs(grp) - 1;
                int s = -1;
                if (lane == leader) {
                    s = tab_find(t, ru.label);
                    if (s < 0) atomicOr(err, 4);
                    else atomic_add_u128(t.q + 2 * s, group_sum_all(st, grp));
                }
                hslot[h.ent + e] = __shfl_sync(grp, s, leader);
            } else if (act) {
                hslot[h.ent + e] = -1;
            }
            __syncwarp();
            if (rw.dx >= 2 && foreign && ru.dx >= 2) {
                if (rank_after(ru.dx, u, rw.dx, h.row)) no++; else ni++;
            }
        }
        no = block_sum_u32<NT>(no, sh_u32);
        ni = block_sum_u32<NT>(ni, sh_u32);
        if (tid == 0) { hitem_out[it] = (int32_t)no; hitem_in[it] = (int32_t)ni; }
        __syncthreads();
    }
}

// hub rows, P2 step 2, a thread per hub: the row's G_x out and in counts, summed over its chunks
template <int NT>
__global__ void __launch_bounds__(NT) hub_p2_counts_kernel(
    const HubInfo *__restrict__ hubs, int64_t nhubs, const int32_t *hitem_out, const int32_t *hitem_in,
    const int64_t *__restrict__ xoff, const NodeRec *__restrict__ rec, int32_t *xout, int32_t *xin, GxNode *xnode) {
    for (int64_t hi = (int64_t)blockIdx.x * NT + threadIdx.x; hi < nhubs; hi += (int64_t)gridDim.x * NT) {
        const HubInfo h = hubs[hi];
        int32_t so = 0, si = 0;
        for (int j = 0; j < h.n_items; ++j) {
            so += hitem_out[h.first_item + j];
            si += hitem_in[h.first_item + j];
        }
        xout[h.row] = so;
        xin[h.row] = si;
        xnode[h.row] = GxNode{xoff[h.row], so, rec[h.row].dx};
    }
}

// hub rows, P2 step 3: Type-II terms and the G_x entries of each chunk
template <int NT, class Slot>
__global__ void __launch_bounds__(NT) hub_p2_emit_kernel(
    const int64_t *__restrict__ off, const int32_t *__restrict__ col, const HubInfo *__restrict__ hubs,
    const int32_t *__restrict__ items, const int32_t *__restrict__ chunks, int64_t nitems, int32_t chunk_len,
    const NodeRec *__restrict__ rec, const int32_t *__restrict__ hslot,
    const unsigned long long *hq, const df *hsig, const int32_t *hitem_out, const int32_t *hitem_in,
    unsigned long long *acc, const int64_t *__restrict__ xoff, int32_t *__restrict__ xcol,
    Slot *__restrict__ xS, int32_t *__restrict__ xsk, int *err, Strict SX) {
    __shared__ int32_t sh_cnt[2 * NT / 32];
    int tid = threadIdx.x;
    for (int64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
        int32_t hidx = items[it];
        HubInfo h = hubs[hidx];
        int64_t b = off[h.row];
        int64_t d = off[h.row + 1] - b;
        int32_t ch = chunks[it];
        int64_t lo = (int64_t)ch * chunk_len;
        int64_t hi = min(d, lo + chunk_len);
        NodeRec rw = rec[h.row];
        int32_t bo = 0, bi = 0;
        for (int j = 0; j < ch; ++j) { bo += hitem_out[h.first_item + j]; bi += hitem_in[h.first_item + j]; }
        int64_t xb = xoff[h.row];
        for (int64_t base = lo; base < hi; base += NT) {
            int64_t e = base + tid;
            bool act = e < hi;
            int32_t u = act ? col[b + e] : -1;
            NodeRec ru{0, -1, 0};
            if (act) ru = rec[u];
            // the slot step 1 found (-1: own community, or a miss step 1 flagged)
            const int s = act ? hslot[h.ent + e] : -1;
            bool cross = s >= 0;
            df sig{0.0f, 0.0f};
            if (cross) {
                int64_t gs = h.tab + s;
                const df st = hsig[gs];                // negative: a single member, no push
                sig = st.hi < 0.0f ? df{-st.hi, -st.lo} : st;
                if (st.hi > 0.0f) {
                    u128 q = ((u128)hq[2 * gs + 1] << 64) | hq[2 * gs];
                    push_type2(acc, u, sig, strict_rest(SX, off, h.row, u, q - ru.s_fix, b + e));
                }
            }
            if (rw.dx >= 2) {
                bool inx = cross && ru.dx >= 2;
                bool o = inx && rank_after(ru.dx, u, rw.dx, h.row);
                gx_round<NT>(o, inx && !o, xb, rw.dx, u, inx ? sig_fixed(sig) : 0, bo, bi, xcol, xS, xsk, sh_cnt);
            }
        }
    }
}

// ======================================================================================
// P3: Type-I triads from G_x triangles
// ======================================================================================
// The reverse value of a G_x edge.  Row x writes its in-neighbours (the G_x
// neighbours of lower rank) from the back of its G_x row in increasing id
// order, so its in-list read backwards from the row's last slot is sorted and
// S(x -> y) for an in-neighbour y is found by binary search there.  P3 needs
// the reverse values only of the edges of triangles.  It either looks them up
// per triangle (three searches in in-lists), or reads them beside the forward
// values, where the mirror pass below puts them for every G_x edge beforehand (one
// search per edge, in a short out-list).  The first wins when triangles are few per G_x edge
// (0.11 on the 1M-node DC-SBM graph), the second when they are many; the
// choice is a launch parameter (p3_mirror).
__device__ __forceinline__ uint64_t in_value(int32_t x, int32_t y, const int64_t *xoff, const int32_t *xcol,
                                             const uint64_t *xf, const int32_t *xin, int *err) {
    const int64_t last = xoff[x + 1] - 1;
    const int32_t len = xin[x];
    int32_t l = 0, h = len;
    while (l < h) {
        int32_t mid = (l + h) >> 1;
        if (xcol[last - mid] < y) l = mid + 1; else h = mid;
    }
    if (l < len && xcol[last - l] == y) return xf[last - l];
    atomicOr(err, 16);
    return 0;
}

// where P3 takes an edge's values: both at the out-slot (mirror pass), or the reverse one
// in the in-list of the higher-ranked end
struct Rev {
    const void *xS;                  // SigPair per slot, or (not mirrored) f alone
    const int64_t *xoff;
    const int32_t *xcol;
    const int32_t *xin;
    int *err;
    bool mirrored;
    // S(lo -> hi) and S(hi -> lo) for the G_x edge whose out-slot (lo -> hi) is `slot`
    __device__ __forceinline__ SigPair get(int64_t slot, int32_t hi, int32_t lo) const {
        if (mirrored) {
            const ulonglong2 v = __ldg(static_cast<const ulonglong2 *>(xS) + slot);
            return SigPair{v.x, v.y};
        }
        const uint64_t *xf = static_cast<const uint64_t *>(xS);
        return SigPair{xf[slot], in_value(hi, lo, xoff, xcol, xf, xin, err)};
    }
};

// position of key in the sorted list xcol[lo, lo + len), or -1
__device__ __forceinline__ int64_t find_in_list(const int32_t *xcol, int64_t lo, int32_t len, int32_t key) {
    int32_t l = 0, h = len;
    while (l < h) {
        int32_t mid = (l + h) >> 1;
        if (xcol[lo + mid] < key) l = mid + 1; else h = mid;
    }
    return (l < len && xcol[lo + l] == key) ? lo + l : -1;
}

// lists of at most this many ids are binary-searched directly (they span at most 9 sectors)
constexpr int32_t kSkipMin = 64;

// position of key in the sorted list xcol[lo, lo + len), or -1.  A list of more than
// kSkipMin ids is searched first in xsk (xsk[t] = xcol[8 t], the first id of every 8-slot
// sector of the slot space, written by P2 with the slots), over the sectors that start
// inside the list, for the one sector that can hold key (the last whose first id is <= key;
// before them, the sector holding the list's head, when the list does not start a sector);
// that sector is then read with two 16-byte loads and its slots inside the list compared
// with key.  The chain of dependent loads of a long list thus runs over the packed index (8
// times denser than the list) and ends with one sector.  xcol is padded to whole sectors,
// so the last sector is readable.
__device__ __forceinline__ int64_t find_in_list_sk(const int32_t *xcol, const int32_t *xsk, int64_t lo, int32_t len,
                                                   int32_t key) {
    if (len <= kSkipMin) return find_in_list(xcol, lo, len, key);
    const int64_t end = lo + len;
    const int64_t t0 = (lo + 7) >> 3;                // first sector starting inside the list
    const int32_t ns = (int32_t)(((end - 1) >> 3) - t0 + 1);
    int32_t l = 0, h = ns;                           // first of them whose first id exceeds key
    while (l < h) {
        const int32_t mid = (l + h) >> 1;
        if (__ldg(xsk + t0 + mid) <= key) l = mid + 1; else h = mid;
    }
    const int64_t t = t0 + l - 1;
    if (t < (lo >> 3)) return -1;                    // key is below the first id, which starts a sector
    const int4 *v = reinterpret_cast<const int4 *>(xcol + 8 * t);
    const int4 x = __ldg(v), y = __ldg(v + 1);
    const int32_t e[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    const int64_t b = 8 * t;
    int64_t pos = -1;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (e[j] == key && b + j >= lo && b + j < end) pos = b + j;
    return pos;
}

// P3m (mirror, when p3_mirror is set): every G_x out-slot (w -> u) receives the reverse value
// S(u -> w), which row u wrote at its in-slot for w.  Node u's slots are
// [xoff[u], xoff[u] + dx(u)), its in-slots the last xin(u) of them.  The slot
// space [0, xoff[n]) is cut into tiles of kMirTile consecutive slots, one
// tile per CTA trip, so the work per CTA does not depend on the in-degrees.
// The nodes a tile spans run from the node holding its first slot to the one
// holding the next tile's first slot (a table filled with the offsets, so no tile
// searches them; `last` is the last node with slots).  A tile stages their offsets in shared memory, counts
// their in-slots inside the tile and spreads only those over the threads; a
// slot's out-slot twin is found in w's out-list (w has the lower rank), by
// find_in_list_sk: a binary search, or for a list of more than kSkipMin ids one
// through the packed sector index.  A tile spanning more than kMirNodes nodes
// (long runs of nodes outside G_x) searches the offsets in global memory.
constexpr int kMirNodes = 1024;

__device__ __forceinline__ int64_t last_leq(const int64_t *xoff, int64_t lo, int64_t hi, int64_t key) {
    // last index i in [lo, hi) with xoff[i] <= key (xoff[lo] <= key)
    while (hi - lo > 1) {
        int64_t mid = lo + ((hi - lo) >> 1);
        if (xoff[mid] <= key) lo = mid; else hi = mid;
    }
    return lo;
}

// copy S(u -> w) from u's in-slot sl to w's out-slot for u (found in w's out-list, through
// the packed index when the list is long)
__device__ __forceinline__ void mirror_one(int64_t sl, int32_t u, const int32_t *xcol,
                                           const int32_t *xsk, SigPair *xS, const GxNode *xnode, int *err) {
    const int32_t w = xcol[sl];
    const GxNode nw = load_node(xnode, w);
    const int64_t pos = find_in_list_sk(xcol, xsk, nw.off, nw.out, u);
    if (pos >= 0) xS[pos].r = xS[sl].f;
    else atomicOr(err, 16);
}

__global__ void __launch_bounds__(kThreads) gx_mirror_kernel(
    int64_t n, const int64_t *__restrict__ xoff, const int32_t *__restrict__ xcol, SigPair *__restrict__ xS,
    const GxNode *__restrict__ xnode, const int32_t *__restrict__ xin, const int32_t *__restrict__ cover,
    const int32_t *__restrict__ last, const int32_t *__restrict__ xsk, int *err) {
    chain_wait();
    __shared__ int64_t s_lo[kMirNodes];          // first in-slot of each staged node inside the tile
    __shared__ int32_t s_pre[kMirNodes + 1];     // prefix sums of the staged nodes' in-slots in the tile
    __shared__ int32_t s_wsum[kThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t S = xoff[n];
    const int64_t tiles = (S + kMirTile - 1) / kMirTile;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        int64_t s0 = t * kMirTile, s1 = min(S, s0 + kMirTile);
        // nodes [ulo, uhi): from the one holding s0 to the one holding s1 (or the last slot)
        int64_t ulo = cover[t], uhi = (int64_t)(t + 1 < tiles ? cover[t + 1] : *last) + 1;
        __syncthreads();                             // the previous tile's stage is free
        int32_t nn = (int32_t)(uhi - ulo);
        if (nn > kMirNodes) {
            for (int64_t sl = s0 + tid; sl < s1; sl += blockDim.x) {
                int64_t u = last_leq(xoff, ulo, uhi, sl);
                if (sl >= xoff[u + 1] - xin[u]) mirror_one(sl, (int32_t)u, xcol, xsk, xS, xnode, err);
            }
            continue;
        }
        // in-slots of each staged node inside [s0, s1): four consecutive nodes per thread
        constexpr int kPer = kMirNodes / kThreads;
        int32_t cnt[kPer];
        int32_t mine = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            int32_t i = tid * kPer + j;
            cnt[j] = 0;
            if (i < nn) {
                int64_t end = xoff[ulo + i + 1];
                int64_t lo = max(end - (int64_t)xin[ulo + i], s0);
                int64_t hi = min(end, s1);
                s_lo[i] = lo;
                cnt[j] = hi > lo ? (int32_t)(hi - lo) : 0;
            }
            mine += cnt[j];
        }
        int32_t incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_wsum[wid] = incl;
        __syncthreads();
        int32_t before = 0, total = 0;
        for (int j = 0; j < kThreads / 32; ++j) {
            if (j < wid) before += s_wsum[j];
            total += s_wsum[j];
        }
        int32_t run = before + incl - mine;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            int32_t i = tid * kPer + j;
            if (i < nn) s_pre[i] = run;
            run += cnt[j];
        }
        if (tid == 0) s_pre[nn] = total;
        __syncthreads();
        for (int32_t q = tid; q < total; q += blockDim.x) {
            int32_t lo = 0, hi = nn;                    // last staged node with s_pre <= q
            while (hi - lo > 1) {
                int32_t mid = (lo + hi) >> 1;
                if (s_pre[mid] <= q) lo = mid; else hi = mid;
            }
            mirror_one(s_lo[lo] + (q - s_pre[lo]), (int32_t)(ulo + lo), xcol, xsk, xS, xnode, err);
        }
    }
}

// P3 lists the triangles of G_x once each, from their lowest-ranked node a
// (rank = (dx, id); a node's out-list holds its higher-ranked G_x neighbours,
// sorted by id).  Every pair {b, c} of a's out-neighbours is a candidate, and
// it closes a triangle iff the higher-ranked of the two is in the out-list of
// the lower-ranked one.  There are sum_a d+(a)(d+(a)-1)/2 candidates, several
// times fewer than the wedges a -> b -> c on these graphs.
//
// A CTA of four warps takes a group of up to 32 consecutive nodes and stages their
// out-lists (with each entry's G_x offset, out-degree and rank) in shared memory, window
// by window of at most kWinCap entries.  All candidate pairs of a window form one flat
// index space that the threads share evenly: entry e owns the pairs (e, f > e) of its
// node.  The closing edge is looked up in the lower-ranked node's out-list in global
// memory by find_in_list_sk (a binary search, or for a long list one through the packed
// sector index).  Found triangles are queued per warp and finished 32 at a time, one per
// lane: a triangle's terms all have the form S S (S + S) with one factor on an edge
// a - x of the window, so their pair products are summed per window entry in shared
// memory, and the entries' sums are scaled and added to the accumulators once per window
// (a's over its entries first).  Nodes with more than kWinCap out-neighbours (heavy
// nodes) are walked by wedges instead (p3_heavy_kernel).
//
// What bounds it is the chain of dependent loads per window (and, where most pairs close, the
// data path of the loads), so a window is shared by four warps and the groups shrink on small
// graphs.  A warp per window, with three double-float terms and three 128-bit global adds per
// triangle, took, against this form: 174 -> 40 us on 33,333 nodes, 283 -> 98 us on 200,001,
// 142 -> 135 us on 1M nodes (10.3M edges, 262K triangles), 3.83 -> 2.33 ms on a batch of 256
// graphs (81M edges), 9.11 -> 5.34 ms on the 8M-node hub-skewed graph.
constexpr int kP3Threads = 128, kP3Warps = kP3Threads / 32, kP3CtasPerSm = 12;
static_assert(kP3Threads == kWinCap, "a thread per window entry");

struct P3Stage {
    int64_t boff[kWinCap];          // xoff[b]
    int64_t aoff[32];               // xoff[a]
    int64_t qpos[kP3Warps][64];     // triangles found and not yet finished: the closing slot
    uint8_t qlo[kP3Warps][64];      //   and the window entries of the lower- and higher-ranked
    uint8_t qhi[kP3Warps][64];      //   neighbours
    int32_t nb[kWinCap];            // b
    int32_t bdeg[kWinCap];          // d+(b)
    int32_t bdx[kWinCap];           // dx(b): rank(b) = (dx(b), b)
    // sums of pair products per entry x, 0 between windows: `to` those that S(a->x) scales
    // (they belong to x), `from` those that S(x->a) scales (they belong to a).  An entry
    // closes fewer than kWinCap triangles, so the words do not overflow
    uint32_t to[kLimbs][kWinCap], from[kLimbs][kWinCap];
    int32_t seg[33];                // first entry of each lane's node in the window
    int32_t anode[32];              // a
    uint32_t wsum[kP3Warps];
    uint16_t ppre[kWinCap + 1];     // prefix sums of the pairs (e, f > e) owned by the entries
    uint8_t owner[kWinCap];         // lane (node) of the entry
    int32_t found;                  // whether the window has a triangle
    long long ticket;
};

__device__ __forceinline__ void limbs_add(uint32_t (*l)[kWinCap], int e, Product p) {
#pragma unroll
    for (int j = 0; j < kLimbs; ++j) {
        const uint32_t v = pair_limb(p, j);
        if (v) atomicAdd(&l[j][e], v);
    }
}
__device__ __forceinline__ u96 limbs_take(uint32_t (*l)[kWinCap], int e) {
    const u96 p = from_limbs(l[0][e], l[1][e], l[2][e], l[3][e]);
#pragma unroll
    for (int j = 0; j < kLimbs; ++j) l[j][e] = 0;
    return p;
}

// the out-slot of window entry e, in its node's out-list
__device__ __forceinline__ int64_t p3_slot(const P3Stage &S, int e) {
    const int o = S.owner[e];
    return S.aoff[o] + (e - S.seg[o]);
}

// finish the first m (<= 32) triangles queued by the warp, one per lane
__device__ __forceinline__ void p3_flush(P3Stage &S, int wid, int m, const Rev &R, int lane) {
    if (lane < m) {
        const int el = S.qlo[wid][lane], eh = S.qhi[wid][lane];
        const int32_t a = S.anode[S.owner[el]], b = S.nb[el], c = S.nb[eh];
        const SigPair bc = R.get(S.qpos[wid][lane], c, b), ab = R.get(p3_slot(S, el), b, a),
                      ac = R.get(p3_slot(S, eh), c, a);
        limbs_add(S.from, el, product(ac.r, bc.f + bc.r));      // a: scaled by S(b->a)
        limbs_add(S.to, el, product(bc.r, ac.f + ac.r));        // b: scaled by S(a->b)
        limbs_add(S.to, eh, product(bc.f, ab.f + ab.r));        // c: scaled by S(a->c)
    }
}

__device__ __forceinline__ bool rank_less(int32_t dx1, int32_t id1, int32_t dx2, int32_t id2) {
    return dx1 < dx2 || (dx1 == dx2 && id1 < id2);
}

// groups of `group` (<= 32) nodes are handed out by an atomic counter (next_group, zeroed
// before the launch), so CTAs that drew light groups take more and no tail is left waiting.
// kScr (graphs built with RS_REORDER): lane j of group g takes node
// (group g + j) * stride mod n (stride coprime to n), because consecutive ids then hold a
// community's heaviest nodes together and one group of them would be a long tail for
// its CTA; otherwise lane j takes node group g + j and stride is unused.
template <bool kScr>
__global__ void __launch_bounds__(kP3Threads, kP3CtasPerSm) p3_list_kernel(
    int64_t n, const int64_t *__restrict__ xoff, const int32_t *__restrict__ xcol, const int32_t *__restrict__ xsk,
    Rev R, const int32_t *__restrict__ xout, const GxNode *__restrict__ xnode, unsigned long long *acc,
    unsigned long long *next_group, int32_t group, int64_t stride, unsigned long long *hvl, int64_t hvcap,
    unsigned long long *hv_count) {
    chain_wait();
    __shared__ P3Stage S;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int j = 0; j < kLimbs; ++j) { S.to[j][tid] = 0; S.from[j][tid] = 0; }
    if (tid == 0) { S.found = 0; S.ticket = (long long)atomicAdd(next_group, 1ull); }
    __syncthreads();
    while (true) {
        const int64_t base = S.ticket * group;
        if (base >= n) break;
        __syncthreads();                               // everyone has read the ticket
        if (tid == 0) S.ticket = (long long)atomicAdd(next_group, 1ull);   // read after the windows' barriers
        // every warp works out the windows alike: lane j holds node j of the group
        int64_t av = base + lane;
        const bool have = lane < group && av < n;
        if (kScr && have) av = (int64_t)(((unsigned __int128)av * (uint64_t)stride) % (uint64_t)n);
        const int32_t da = have ? xout[av] : 0;
        const bool grp = da >= 2 && da <= kWinCap;
        const int32_t mine = grp ? da : 0;
        int32_t incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        const int64_t ba = grp ? xoff[av] : 0;
        // windows of consecutive nodes whose entries fit kWinCap
        int32_t start = 0;
        while (true) {
            const int32_t excl0 = start > 0 ? __shfl_sync(FULL, incl, start - 1) : 0;
            const unsigned fitm = __ballot_sync(FULL, lane >= start && incl - excl0 <= kWinCap);
            if (start >= 32 || fitm == 0) break;
            const int32_t end = 32 - __clz(fitm);             // lanes [start, end) fit
            const int32_t Ew = __shfl_sync(FULL, incl, end - 1) - excl0;
            if (Ew > 0) {
                if (wid == 0) {
                    // seg is nondecreasing over all 32 lanes: the entry j belongs to the
                    // last lane o with seg[o] <= j (lanes without entries share the next seg)
                    const bool inwin = lane >= start && lane < end;
                    S.seg[lane] = lane < start ? 0 : (inwin ? incl - mine - excl0 : Ew);
                    if (lane == 0) S.seg[32] = Ew;
                    S.aoff[lane] = ba;
                    S.anode[lane] = (int32_t)av;
                }
                __syncthreads();
                // a thread per entry: its data and the pair prefix sums
                uint32_t x = 0;
                if (tid < Ew) {
                    int32_t lo = 0, hi = 32;
                    while (hi - lo > 1) {
                        const int32_t mid = (lo + hi) >> 1;
                        if (S.seg[mid] <= tid) lo = mid; else hi = mid;
                    }
                    const int32_t loc = tid - S.seg[lo];
                    const int32_t b = xcol[S.aoff[lo] + loc];
                    S.nb[tid] = b;
                    S.owner[tid] = (uint8_t)lo;
                    const GxNode nb = load_node(xnode, b);
                    S.boff[tid] = nb.off;
                    S.bdeg[tid] = nb.out;
                    S.bdx[tid] = nb.dx;
                    x = (uint32_t)(S.seg[lo + 1] - S.seg[lo] - 1 - loc);   // pairs (e, f > e) of the node
                }
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(FULL, x, o);
                    if (lane >= o) x += y;
                }
                if (lane == 31) S.wsum[wid] = x;
                __syncthreads();
                for (int j = 0; j < wid; ++j) x += S.wsum[j];
                if (tid < Ew) S.ppre[tid + 1] = (uint16_t)x;
                if (tid == 0) S.ppre[0] = 0;
                __syncthreads();
                const int32_t P = S.ppre[Ew];
                int qn = 0;                                // triangles queued by the warp (uniform)
                for (int32_t p0 = 32 * wid; p0 < P; p0 += kP3Threads) {
                    const int32_t pv = p0 + lane;
                    int32_t el = 0, eh = 0;
                    int64_t pos = -1;
                    if (pv < P) {
                        int32_t lo = 0, hi = Ew;            // last entry with ppre[e] <= pv
                        while (hi - lo > 1) {
                            const int32_t mid = (lo + hi) >> 1;
                            if (S.ppre[mid] <= pv) lo = mid; else hi = mid;
                        }
                        const int32_t f = lo + 1 + (pv - S.ppre[lo]);
                        const bool e_low = rank_less(S.bdx[lo], S.nb[lo], S.bdx[f], S.nb[f]);
                        el = e_low ? lo : f;
                        eh = e_low ? f : lo;
                        pos = find_in_list_sk(xcol, xsk, S.boff[el], S.bdeg[el], S.nb[eh]);
                    }
                    const bool hit = pos >= 0;
                    const unsigned hm = __ballot_sync(FULL, hit);
                    if (hit) {
                        const int slot = qn + __popc(hm & lanemask_lt());
                        S.qpos[wid][slot] = pos;
                        S.qlo[wid][slot] = (uint8_t)el;
                        S.qhi[wid][slot] = (uint8_t)eh;
                        S.found = 1;
                    }
                    qn += __popc(hm);
                    // a full warp of triangles, or (in the warp's last trip) what is left
                    const bool last = p0 + kP3Threads >= P;
                    while (qn >= 32 || (last && qn > 0)) {
                        const int m = min(qn, 32);
                        __syncwarp();
                        p3_flush(S, wid, m, R, lane);
                        __syncwarp();
                        if (lane < qn - m) {
                            S.qpos[wid][lane] = S.qpos[wid][32 + lane];
                            S.qlo[wid][lane] = S.qlo[wid][32 + lane];
                            S.qhi[wid][lane] = S.qhi[wid][32 + lane];
                        }
                        qn -= m;
                        __syncwarp();
                    }
                }
                __syncthreads();
                // the window's sums to the accumulators, a thread per entry
                if (S.found) {
                    u192 ta{0, 0, 0};
                    int own = -1;
                    if (tid < Ew) {
                        own = S.owner[tid];
                        const u96 to = limbs_take(S.to, tid), from = limbs_take(S.from, tid);
                        if (to.lo | to.hi | from.lo | from.hi) {
                            const SigPair ax = R.get(p3_slot(S, tid), S.nb[tid], S.anode[own]);
                            if (to.lo | to.hi) atomic_add_u192(acc + 3 * (int64_t)S.nb[tid], scale(ax.f, to));
                            ta = scale(ax.r, from);
                        }
                    }
                    // a's terms, summed over the lanes of each node (consecutive) to its first lane
                    if (__any_sync(FULL, (ta.w0 | ta.w1 | ta.w2) != 0)) {
                        for (int o = 1; o < 32; o <<= 1) {
                            const int oo = __shfl_down_sync(FULL, own, o);
                            const u192 y{__shfl_down_sync(FULL, ta.w0, o), __shfl_down_sync(FULL, ta.w1, o),
                                         __shfl_down_sync(FULL, ta.w2, o)};
                            if (lane + o < 32 && oo == own) ta = u192_add(ta, y);
                        }
                        const int before = __shfl_up_sync(FULL, own, 1);
                        if (own >= 0 && (lane == 0 || before != own) && (ta.w0 | ta.w1 | ta.w2))
                            atomic_add_u192(acc + 3 * (int64_t)S.anode[own], ta);
                    }
                    __syncthreads();
                    if (tid == 0) S.found = 0;
                }
                __syncthreads();                           // the stage is reused next
            }
            start = end;
        }
        // heavy nodes' tasks go to the list (its capacity bounds their number, so the
        // error branch is not taken)
        if (wid == 0 && da > kWinCap) {
            const int32_t nt = (da + kHvBlock - 1) / kHvBlock;
            const unsigned long long h = atomicAdd(hv_count, (unsigned long long)nt);
            if (h + nt <= (unsigned long long)hvcap) {
                for (int32_t i = 0; i < nt; ++i) hvl[h + i] = (unsigned long long)av << 32 | (unsigned)i;
            } else {
                atomicOr(R.err, 64);
            }
        }
        __syncthreads();                                   // the next ticket is there
    }
}

// Heavy nodes: a wedge walk, one CTA per task.  A task is a heavy node a with a block
// of kHvBlock of its out-neighbours b.  The CTA stages a's out-list A (sorted by id),
// kHvIds ids at a time, as a shared-memory hash table (id -> position in the chunk) beside
// the value S(c->a) and the sum S(a->c) + S(c->a) for every c of the chunk.  Its warps then
// take the task's out-neighbours b one at a time: a warp streams b's out-list (the nodes c
// ranked above b), coalesced, and looks every c up in the table; a hit closes the triangle
// {a, b, c}, which is met once, at its middle-ranked node b.  When A takes several chunks,
// b's out-list is first cut to the chunk's id range.  There are several times more wedges
// than pairs on such nodes, but a wedge costs a coalesced load and one 4-byte load from
// shared memory where a pair costs a binary search in global memory.
//
// A third of the heavy wedges close on the 8M-node graph, so finishing the triangles
// dominates.  Hits are queued (one word each) and finished a warp at a time, one triangle
// per lane, by three pair products, whose outer factors come out of the sums: a's and b's
// pairs are summed in registers over the warp's walk of b (S(b->a) and S(a->b) scale them
// once at its end), c's pairs in four 32-bit words per staged position in shared memory
// (S(a->c) scales them once per chunk).  The products are exact, so the bits do not depend
// on the grouping.
//
// Issue slots and the latency of the loads bound it.  Before this form
// (4-slot buckets read 16 bytes at a time, three double-float products and three fixed-point
// conversions per triangle, c's sums by 64-bit shared atomics, which take five times as long
// as 32-bit ones) it ran the shared-memory pipe at 74% and issue at 66%: 43.8 -> 36.2 ms on the
// 8M-node graph (6.4e9 wedges, 2.1e9 triangles), 5.87 -> 4.52 ms on 2M nodes, where the pipe is
// now at 41% and issue at 58%.
//
// The warp whose group holds a heavy node does not walk it: it appends the node's
// tasks to the task list (slots taken with an atomic counter), and p3_heavy_kernel,
// launched next on the same stream, runs them, a CTA per task.
constexpr int kHvIds = 1024;                  // ids of A staged per chunk
constexpr int kHvBits = 13, kHvSlots = 1 << kHvBits;   // hash slots: at most an eighth used
constexpr int kHvUnroll = 4;                  // 32-entry rows of b's out-list per trip
constexpr int kHvQ = 32 * kHvUnroll + 32;     // queued triangles per warp: < 32 left + one trip
constexpr int kHvWarps = kThreads / 32;

// The hash of an id is a product by an odd constant modulo 2^32, a bijection: its top
// kHvBits bits are the home slot, the 19 bits below identify the id there.  A slot word
// holds bit 31 (taken), kMore (an id whose home is this slot is elsewhere), kMoved (its own
// id is not at home), the id's position and its 19 bits; an id at home is thus recognised
// exactly by one 4-byte load.  Moved ids are in the slots after their home; their bits
// alone do not identify them, so they are checked against A itself.
constexpr uint32_t kHvTaken = 1u << 31, kHvMore = 1u << 30, kHvMoved = 1u << 29;
constexpr int kHvRest = 32 - kHvBits;
constexpr uint32_t kHvRestMask = (1u << kHvRest) - 1, kHvPosMask = kHvIds - 1;
static_assert(kHvRest + 10 + 3 == 32 && kHvIds == 1 << 10, "a slot word's fields");
__device__ __forceinline__ uint32_t hv_hash(int32_t c) { return (uint32_t)c * 0x9E3779B1u; }

struct P3Heavy {
    SigPair sp[kHvIds];                       // S(c->a), S(a->c) + S(c->a)
    uint32_t tab[kHvSlots];
    uint32_t sum[kLimbs][kHvIds];             // c's pairs of the chunk; at most kHvBlock each
    uint32_t q[kHvWarps][kHvQ];               // hits: c's entry in b's out-list << 10 | position
    int64_t a, bA;
    int32_t dA, eb0, nb, next_b, stop;
};
static_assert(kHvBlock <= 128, "the words of a pair sum take 128 pairs");

// first position of the sorted p[0, cnt) (cnt >= 1) holding an id >= key, or cnt;
// the trip count depends on cnt alone
__device__ __forceinline__ int32_t lower_pos(const int32_t *p, int32_t cnt, int32_t key) {
    int32_t base = 0, len = cnt;
    while (len > 1) {
        const int32_t half = len >> 1;
        base = p[base + half] < key ? base + half : base;
        len -= half;
    }
    return base + (p[base] < key ? 1 : 0);
}

// position of an id that is not at home, or -1: the slots after its home (hash h), up to
// the first empty one.  A: the chunk's ids
__device__ __forceinline__ int32_t hv_find_moved(const P3Heavy &H, int32_t c, uint32_t h, const int32_t *A) {
    uint32_t s = h >> kHvRest;
    for (int it = 0; it < kHvSlots; ++it) {
        s = (s + 1) & (kHvSlots - 1);
        const uint32_t w = H.tab[s];
        if (!w) break;
        const int32_t p = (int32_t)(w >> kHvRest & kHvPosMask);
        if ((w & kHvMoved) && (w & kHvRestMask) == (h & kHvRestMask) && A[p] == c) return p;
    }
    return -1;
}

// an out-neighbour b of the task (entry eb of A): its out-list [ob + s, ob + e) cut to
// the chunk's id range [lo_id, hi_id] when A takes several chunks, and the values of
// the edge a -> b
struct HvB {
    int32_t b, s, e;
    int64_t ob;
    SigPair ab;
};
__device__ __forceinline__ HvB hv_load_b(int32_t a, int64_t eb, bool cut, int32_t lo_id, int32_t hi_id,
                                         const int32_t *xcol, const Rev &R, const GxNode *xnode) {
    HvB B;
    B.b = xcol[eb];
    const GxNode nb = load_node(xnode, B.b);
    B.ob = nb.off;
    const int32_t db = nb.out;
    B.s = 0;
    B.e = db;
    if (cut && db > 0) {
        B.s = lower_pos(xcol + B.ob, db, lo_id);
        B.e = lower_pos(xcol + B.ob, db, hi_id + 1);
    }
    B.ab = R.get(eb, B.b, a);
    return B;
}

// the sum of v over the warp's lanes (below 2^96), by hardware sums of 27-bit pieces
__device__ __forceinline__ u96 warp_sum_u96(u96 v) {
    constexpr uint32_t M = (1u << 27) - 1;
    const u128 x = ((u128)v.hi << 64) | v.lo;
    const uint32_t r0 = __reduce_add_sync(FULL, (uint32_t)x & M);
    const uint32_t r1 = __reduce_add_sync(FULL, (uint32_t)(x >> 27) & M);
    const uint32_t r2 = __reduce_add_sync(FULL, (uint32_t)(x >> 54) & M);
    const uint32_t r3 = __reduce_add_sync(FULL, (uint32_t)(x >> 81));
    const u128 s = (u128)r0 + ((u128)r1 << 27) + ((u128)r2 << 54) + ((u128)r3 << 81);
    return u96{(uint64_t)s, (uint32_t)(s >> 64)};
}

// one warp's walk of out-neighbour b over the staged chunk (ids A): each trip loads and
// looks up kHvUnroll rows of 32 entries of b's out-list, queues the hits, and finishes the
// queued triangles 32 at a time (at the end of the list, the rest too); the finishing code
// is inlined once.  A list has at most 2^20 ids (each of them has a cross degree at least
// as large, and nnz < 2^40), so a hit fits one word; a walk closes at most kHvIds
// triangles, so its pair sums stay below 2^96
__device__ __forceinline__ void hv_walk_b(P3Heavy &H, uint32_t *Q, const HvB &B, const int32_t *A,
                                          const int32_t *xcol, const Rev &R, unsigned long long *acc, int lane,
                                          u192 &acc_a) {
    if (B.s >= B.e) return;
    const uint64_t Pab = B.ab.f + B.ab.r;
    int qn = 0;                                        // queued triangles (warp-uniform)
    bool any = false;
    u96 sum_a{0, 0}, sum_b{0, 0};
    for (int32_t j0 = B.s; j0 < B.e; j0 += 32 * kHvUnroll) {
        int32_t c[kHvUnroll], pos[kHvUnroll];
#pragma unroll
        for (int u = 0; u < kHvUnroll; ++u) {
            const int32_t k = j0 + u * 32 + lane;
            c[u] = k < B.e ? xcol[B.ob + k] : -1;      // -1 is nobody's id, and the hash is a bijection
        }
        bool more = false;
#pragma unroll
        for (int u = 0; u < kHvUnroll; ++u) {
            const uint32_t h = hv_hash(c[u]);
            const uint32_t w = H.tab[h >> kHvRest];
            const bool hit = ((w ^ (kHvTaken | (h & kHvRestMask))) & (kHvTaken | kHvMoved | kHvRestMask)) == 0;
            pos[u] = hit ? (int32_t)(w >> kHvRest & kHvPosMask) : -1;
            more |= !hit && (w & kHvMore);
        }
        if (__any_sync(FULL, more)) {
#pragma unroll 1
            for (int u = 0; u < kHvUnroll; ++u)
#pragma unroll
                for (int v = 0; v < kHvUnroll; ++v)    // (registers are not indexed)
                    if (u == v && pos[v] < 0 && c[v] >= 0 && (H.tab[hv_hash(c[v]) >> kHvRest] & kHvMore))
                        pos[v] = hv_find_moved(H, c[v], hv_hash(c[v]), A);
        }
#pragma unroll
        for (int u = 0; u < kHvUnroll; ++u) {
            const bool hit = pos[u] >= 0;
            const unsigned hm = __ballot_sync(FULL, hit);
            if (hit) Q[qn + __popc(hm & lanemask_lt())] = (uint32_t)(j0 + u * 32 + lane) << 10 | (uint32_t)pos[u];
            qn += __popc(hm);
        }
        const bool last = j0 + 32 * kHvUnroll >= B.e;
        int f = 0;
        while (qn - f >= 32 || (last && qn > f)) {
            const int m = min(32, qn - f);
            any = true;
            __syncwarp();
            if (lane < m) {
                const uint32_t q = Q[f + lane];
                const int32_t p = (int32_t)(q & kHvPosMask);
                const int64_t pc = B.ob + (q >> 10);
                const SigPair bc = R.get(pc, R.mirrored ? 0 : xcol[pc], B.b), sp = H.sp[p];
                u96_add(sum_a, pair_term(sp.f, bc.f + bc.r));
                u96_add(sum_b, pair_term(bc.r, sp.r));
                const Product t = product(bc.f, Pab);
#pragma unroll
                for (int j = 0; j < kLimbs; ++j) {
                    const uint32_t v = pair_limb(t, j);
                    if (j < kLimbs - 1 || v) atomicAdd(&H.sum[j][p], v);
                }
            }
            f += m;
        }
        if (f > 0) {                                   // the rest (< 32) to the front
            __syncwarp();
            uint32_t q = 0;
            if (lane < qn - f) q = Q[f + lane];
            __syncwarp();
            if (lane < qn - f) Q[lane] = q;
            qn -= f;
        }
        __syncwarp();
    }
    if (any) {
        acc_a = u192_add(acc_a, scale(B.ab.r, sum_a));
        sum_b = warp_sum_u96(sum_b);
        if (lane == 0) atomic_add_u192(acc + 3 * (int64_t)B.b, scale(B.ab.f, sum_b));
    }
}

// the heavy-node tasks listed by p3_list_kernel, a CTA per task, claimed with an atomic
// counter; the CTA's warps claim the task's out-neighbours b from a counter in shared
// memory (dynamic shared memory: sizeof(P3Heavy))
__global__ void __launch_bounds__(kThreads, 3) p3_heavy_kernel(
    int64_t n, const int64_t *__restrict__ xoff, const int32_t *__restrict__ xcol, Rev R,
    const int32_t *__restrict__ xout, const GxNode *__restrict__ xnode, unsigned long long *acc,
    const unsigned long long *__restrict__ hvl, int64_t hvcap, const unsigned long long *hv_count,
    unsigned long long *hv_next) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char hv_smem[];
    P3Heavy &H = *reinterpret_cast<P3Heavy *>(hv_smem);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tid = threadIdx.x;
    uint32_t *Q = H.q[wid];
    unsigned long long lim = *hv_count;
    if (lim > (unsigned long long)hvcap) lim = (unsigned long long)hvcap;
    if (lim == 0) return;
    for (int i = tid; i < kHvIds; i += kThreads)
#pragma unroll
        for (int j = 0; j < kLimbs; ++j) H.sum[j][i] = 0;
    while (true) {
        __syncthreads();                               // the previous task is flushed
        if (tid == 0) {
            const unsigned long long t = atomicAdd(hv_next, 1ull);
            H.stop = t >= lim;
            H.a = -1;
            if (!H.stop) {
                const unsigned long long w = hvl[t];
                const int64_t a = (int64_t)(w >> 32), blk = (int64_t)(w & 0xffffffffull);
                if (a >= n || xout[a] <= kWinCap || blk * kHvBlock >= xout[a]) {
                    atomicOr(R.err, 64);
                } else {
                    H.a = a;
                    H.bA = xoff[a];
                    H.dA = xout[a];
                    H.eb0 = (int32_t)(blk * kHvBlock);
                    H.nb = min(kHvBlock, H.dA - H.eb0);
                }
            }
        }
        __syncthreads();
        if (H.stop) break;
        if (H.a < 0) continue;
        const int32_t a = (int32_t)H.a, dA = H.dA, eb0 = H.eb0, nb = H.nb;
        const int64_t bA = H.bA;
        u192 acc_a{0, 0, 0};
        for (int32_t k0 = 0; k0 < dA; k0 += kHvIds) {
            const int32_t cnt = min(kHvIds, dA - k0);
            const int32_t *A = xcol + bA + k0;
            for (int i = tid; i < kHvSlots / 4; i += kThreads) reinterpret_cast<uint4 *>(H.tab)[i] = make_uint4(0, 0, 0, 0);
            if (tid == 0) H.next_b = 0;
            __syncthreads();
            for (int32_t i = tid; i < cnt; i += kThreads) {
                const int32_t c = A[i];
                const uint32_t h = hv_hash(c), home = h >> kHvRest;
                const uint32_t word = kHvTaken | (uint32_t)i << kHvRest | (h & kHvRestMask);
                // home, or the next free slot after it (an eighth of the slots at most are used)
                if ((atomicCAS(&H.tab[home], 0u, word)) != 0) {
                    atomicOr(&H.tab[home], kHvMore);
                    uint32_t s = home;
                    int it = 0;
                    do s = (s + 1) & (kHvSlots - 1);
                    while (atomicCAS(&H.tab[s], 0u, word | kHvMoved) != 0 && ++it < kHvSlots);
                    if (it >= kHvSlots) atomicOr(R.err, 64);
                }
                const SigPair v = R.get(bA + k0 + i, c, a);
                H.sp[i] = SigPair{v.r, v.f + v.r};
            }
            __syncthreads();
            const int32_t lo_id = A[0], hi_id = A[cnt - 1];
            const bool cut = dA > kHvIds;
            // the warp claims out-neighbours one at a time; the next one's data is loaded
            // while the current one is walked
            auto claim = [&]() {
                int32_t j = 0;
                if (lane == 0) j = atomicAdd(&H.next_b, 1);
                return __shfl_sync(FULL, j, 0);
            };
            int32_t j = claim();
            HvB cur{};
            if (j < nb) cur = hv_load_b(a, bA + eb0 + j, cut, lo_id, hi_id, xcol, R, xnode);
            while (j < nb) {
                const int32_t jn = claim();
                HvB nxt{};
                if (jn < nb) nxt = hv_load_b(a, bA + eb0 + jn, cut, lo_id, hi_id, xcol, R, xnode);
                hv_walk_b(H, Q, cur, A, xcol, R, acc, lane, acc_a);
                j = jn;
                cur = nxt;
            }
            __syncthreads();
            // c's sums of the chunk to the accumulators, zeroed for the next chunk
            for (int32_t i = tid; i < cnt; i += kThreads) {
                const u96 t = from_limbs(H.sum[0][i], H.sum[1][i], H.sum[2][i], H.sum[3][i]);
                if (t.lo | t.hi) {
                    atomic_add_u192(acc + 3 * (int64_t)A[i], scale(H.sp[i].r - H.sp[i].f, t));
#pragma unroll
                    for (int l = 0; l < kLimbs; ++l) H.sum[l][i] = 0;
                }
            }
            __syncthreads();
        }
        for (int m = 16; m; m >>= 1)
            acc_a = u192_add(acc_a, u192{__shfl_xor_sync(FULL, acc_a.w0, m), __shfl_xor_sync(FULL, acc_a.w1, m),
                                         __shfl_xor_sync(FULL, acc_a.w2, m)});
        if (lane == 0 && (acc_a.w0 | acc_a.w1 | acc_a.w2)) atomic_add_u192(acc + 3 * (int64_t)a, acc_a);
    }
}

// ======================================================================================
// Strict reading: X(w, u) for every pushed pair, from the closed triads (u, w, v)
// with C(v) = C(u) != C(w): for every intra-community edge {u, v} (u < v) and
// every common neighbour w of another community, s_v is added at u's entry in
// w's row and s_u at v's.  w is a cross neighbour of both u and v, so only their
// cross lists (P1's, sorted by id) are walked and searched, not their rows: the
// shorter one is walked, w is looked up in the other, and the entries in w's row
// are found by binary search.  A hub row has no cross list; its whole row stands
// in for it (walked, its own community is skipped; searched, it holds w just the same).
//
// A warp takes 32 consecutive CSR entries, so a hub's row is spread over many
// warps, and shares the candidates (edge, walked w) of its edges evenly among its
// lanes.  What bounds it is the chain of dependent loads of a candidate's search.
// The form before this one gave a warp a whole row and a lane an edge, and walked
// whole rows with a label gather per entry: 4.12 ms on a 100,003-node graph (0.81M
// edges, degrees to 1,000), most of it the tail of a few warps, against 0.13 ms.
// ======================================================================================
__device__ __forceinline__ int64_t csr_find(const int64_t *off, const int32_t *col, int32_t row, int32_t key) {
    int64_t lo = off[row], hi = off[row + 1], end = hi;
    while (lo < hi) {
        int64_t mid = lo + ((hi - lo) >> 1);
        if (col[mid] < key) lo = mid + 1; else hi = mid;
    }
    return (lo < end && col[lo] == key) ? lo : -1;
}

struct StrictWarp {
    const int32_t *walk[32], *look[32];                // the walked and the searched list of each edge
    int64_t ends[32];                                  // row ends, while the entries' rows are found
    uint64_t su[32], sv[32];
    int32_t look_len[32], u[32], v[32];
    int32_t skip[32];                                  // a walked hub row: its own label, else -1
    int32_t pre[33];                                   // prefix sums of the walked lists' lengths
};

__global__ void __launch_bounds__(kThreads) strict_pairs_kernel(
    int64_t n, const int64_t *__restrict__ off, const int32_t *__restrict__ col, const int32_t *__restrict__ lab,
    const NodeRec *__restrict__ rec, const int32_t *__restrict__ cl_col, Batch B, int32_t small_max, int32_t cta_cap,
    unsigned long long *sx) {
    __shared__ StrictWarp warps[kThreads / 32];
    const int lane = threadIdx.x & 31;
    StrictWarp &S = warps[threadIdx.x >> 5];
    const int64_t E = off[n];
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t e0 = 32 * w0; e0 < E; e0 += 32 * nw) {
        const int64_t e = e0 + lane;
        const bool act = e < E;
        // the rows of the warp's entries: the ends of 32 rows from that of the first entry
        // without one (once, unless many empty rows lie between)
        int64_t u = -1;
        while (true) {
            const unsigned open = __ballot_sync(FULL, act && u < 0);
            if (!open) break;
            const int64_t r = warp_row_of(off, n, e0 + __ffs(open) - 1, lane);
            S.ends[lane] = r + lane < n ? off[r + lane + 1] : INT64_MAX;
            __syncwarp();
            int32_t lo = 0, hi = 32;                   // first row that ends after e
            while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                if (S.ends[mid] <= e) lo = mid + 1; else hi = mid;
            }
            if (u < 0 && lo < 32) u = r + lo;
            __syncwarp();
        }
        int32_t cnt = 0;
        if (act) {
            const int32_t v = col[e];
            if (v > u && lab[v] == lab[u]) {
                const NodeRec ru = rec[u], rv = rec[v];
                if (ru.dx > 0 && rv.dx > 0) {
                    const int32_t k = k_of(B, graph_of(B, v));
                    const int64_t bu = off[u], bv = off[v];
                    const int32_t du = (int32_t)(off[u + 1] - bu), dv = (int32_t)(off[v + 1] - bv);
                    auto hub = [&](int32_t d) {        // a row of the hub class
                        return d > small_max && (d > kLargeDeg || dev_pow2_at_least(2u * (uint32_t)min(d, k)) > (uint32_t)cta_cap);
                    };
                    const bool hu = hub(du), hv = hub(dv);
                    const int32_t lu = hu ? du : ru.dx, lv = hv ? dv : rv.dx;
                    const int32_t *pu = hu ? col + bu : cl_col + bu, *pv = hv ? col + bv : cl_col + bv;
                    const bool walk_u = lu <= lv;
                    S.walk[lane] = walk_u ? pu : pv;
                    S.look[lane] = walk_u ? pv : pu;
                    S.look_len[lane] = walk_u ? lv : lu;
                    S.skip[lane] = (walk_u ? hu : hv) ? ru.label : -1;
                    S.u[lane] = (int32_t)u;
                    S.v[lane] = v;
                    S.su[lane] = ru.s_fix;
                    S.sv[lane] = rv.s_fix;
                    cnt = min(lu, lv);
                }
            }
        }
        // candidates of the 32 edges: degrees are below 2^24, so the sum is below 2^29
        int32_t incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        S.pre[lane + 1] = incl;
        if (lane == 0) S.pre[0] = 0;
        __syncwarp();
        const int32_t total = S.pre[32];
        for (int32_t f = lane; f < total; f += 32) {
            int32_t lo = 0, hi = 32;                   // last edge with pre <= f
            while (hi - lo > 1) {
                const int32_t mid = (lo + hi) >> 1;
                if (S.pre[mid] <= f) lo = mid; else hi = mid;
            }
            const int32_t w = S.walk[lo][f - S.pre[lo]];
            if (S.skip[lo] >= 0 && lab[w] == S.skip[lo]) continue;
            const int32_t *p = S.look[lo];
            int32_t l = 0, h = S.look_len[lo];
            const int32_t len = h;
            while (l < h) {
                const int32_t mid = (l + h) >> 1;
                if (p[mid] < w) l = mid + 1; else h = mid;
            }
            if (l >= len || p[l] != w) continue;
            const int64_t pu = csr_find(off, col, w, S.u[lo]), pv = csr_find(off, col, w, S.v[lo]);
            if (S.sv[lo] && pu >= 0) atomic_add_u128(sx + 2 * pu, (u128)S.sv[lo]);
            if (S.su[lo] && pv >= 0) atomic_add_u128(sx + 2 * pv, (u128)S.su[lo]);
        }
        __syncwarp();
    }
}

// ======================================================================================
// finalize: R(u) = acc(u) / (w_max d (d - 1))
// ======================================================================================
__global__ void graph_scale_kernel(const unsigned long long *__restrict__ wmax_bits, int32_t ng, double *winv) {
    int32_t gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= ng) return;
    double wm = __longlong_as_double((long long)wmax_bits[gi]);
    winv[gi] = wm > 0.0 ? 1.0 / wm : 0.0;
}

// one graph (gid null): every CTA takes 1 / w_max itself; a batch reads the
// per-graph reciprocals graph_scale_kernel wrote.  A reordered graph (perm) writes
// each score at the caller's id of its node.
__global__ void __launch_bounds__(kThreads) finalize_kernel(
    int64_t n, const int64_t *__restrict__ off, const unsigned long long *__restrict__ acc,
    const int32_t *__restrict__ gid, const double *__restrict__ winv, const unsigned long long *__restrict__ wmax_bits,
    const double *__restrict__ RD, const int32_t *__restrict__ perm, double *scores) {
    chain_wait();
    __shared__ double sh_w;
    if (!gid) {
        if (threadIdx.x == 0) {
            double wm = __longlong_as_double((long long)wmax_bits[0]);
            sh_w = wm > 0.0 ? 1.0 / wm : 0.0;
        }
        __syncthreads();
    }
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        int64_t d = off[u + 1] - off[u];
        double r = 0.0;
        if (d >= 2) {
            double W = gid ? winv[gid[u]] : sh_w;
            const u192 s{acc[3 * u], acc[3 * u + 1], acc[3 * u + 2]};
            if ((s.w0 | s.w1 | s.w2) && W > 0.0) r = u192_to_double(s) * W * RD[d];
        }
        scores[perm ? (int64_t)perm[u] : u] = r;
    }
}

// everything a scoring pass starts from, set by one launch (a memset each took about 2 us
// of the chain: 13 us of a 97 us step on 2,000 nodes)
struct InitRange {
    unsigned long long *p;
    int64_t words;
    unsigned long long fill;
};
struct InitArgs {
    InitRange r[10];
    int n;
};
__global__ void __launch_bounds__(kThreads) init_kernel(InitArgs A) {
    chain_wait();
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int j = 0; j < A.n; ++j) {
        const InitRange &r = A.r[j];
        ulonglong2 *p2 = reinterpret_cast<ulonglong2 *>(r.p);
        for (int64_t i = t0; i < r.words / 2; i += step) p2[i] = make_ulonglong2(r.fill, r.fill);
        if (t0 == 0 && (r.words & 1)) r.p[r.words - 1] = r.fill;
    }
}

}  // namespace

// ======================================================================================
// host orchestration
// ======================================================================================
// dynamic shared memory limits of the table kernels, set once per process
template <class Slot>
static int prepare_p2_kernels() {
    RS_CUDA_TRY(cudaFuncSetAttribute(p2_large_kernel<256, Slot>, cudaFuncAttributeMaxDynamicSharedMemorySize, 32 * kMidCap));
    RS_CUDA_TRY(cudaFuncSetAttribute(p2_large_kernel<512, Slot>, cudaFuncAttributeMaxDynamicSharedMemorySize, 32 * kMidCap));
    RS_CUDA_TRY(cudaFuncSetAttribute(p2_large_kernel<1024, Slot>, cudaFuncAttributeMaxDynamicSharedMemorySize, 32 * kMidCap));
    RS_CUDA_TRY(cudaFuncSetAttribute(p2_mid_kernel<Slot>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kP2MidSmem));
    return 0;
}
int rs::prepare_score_kernels() {
    static int done = 0;
    if (done) return 0;
    RS_CUDA_TRY(cudaFuncSetAttribute(p1_large_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * kMidCap));
    RS_CUDA_TRY(cudaFuncSetAttribute(p1_large_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * kMidCap));
    RS_CUDA_TRY(cudaFuncSetAttribute(p1_large_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * kMidCap));
    if (int rc = prepare_p2_kernels<SigPair>()) return rc;
    if (int rc = prepare_p2_kernels<uint64_t>()) return rc;
    RS_CUDA_TRY(cudaFuncSetAttribute(p3_heavy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(P3Heavy)));
    RS_CUDA_TRY(cudaFuncSetAttribute(p1_small_staged_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(kStageWarps * (sizeof(SmallTile) + sizeof(SmallStage)))));
    done = 1;
    return 0;
}

// the CTA-per-row kernels at the tuned CTA size
template <int NT>
static void launch_p1_large(rs_graph *g, const Batch &B, int *err, size_t smem, cudaStream_t st) {
    p1_large_kernel<NT><<<grid_for(g->n_large, 1, 4), NT, smem, st>>>(
        g->off, g->col, g->lab, g->rows_large, g->n_large, B, g->LG, g->rec, g->Lall, err,
        g->rsum, g->cl_col, g->cl_lab, g->wq + 1);
}
// p2_large over P2 list `list`, at most per_sm CTAs per SM
template <int NT, class Slot>
static void launch_p2_large(rs_graph *g, Slot *xS, const Batch &B, int *err, size_t smem, int list, int per_sm,
                            unsigned long long *wq, cudaStream_t st) {
    p2_large_kernel<NT, Slot><<<grid_for(list == 3 ? g->n_large : g->n_mid + g->n_large, 1, per_sm), NT, smem, st>>>(
        g->off, g->p2rows + p2_list_start(list, g->n_mid, g->n_large), g->p2cnt + list, B, g->LG, g->rec, g->rsum,
        g->cl_col, g->cl_lab, g->acc, g->xoff, g->xcol, xS, g->xsk, g->xout, g->xin, g->xnode, err,
        Strict{g->col, g->sx}, wq);
}

// a stride near n / golden ratio, coprime to n (a bijection of [0, n) by multiplication)
static int64_t p3_stride(int64_t n) {
    if (n < 3) return 1;
    auto gcd = [](int64_t a, int64_t b) { while (b) { int64_t t = a % b; a = b; b = t; } return a; };
    int64_t st = (int64_t)((double)n * 0.6180339887) | 1;
    while (st < n && gcd(st, n) != 1) st += 2;
    return st < n ? st : 1;
}

int rs::score_graph(rs_graph *g, double *scores, cudaStream_t s) {
    int64_t n = g->n;
    if (!g->classified || g->dmax > g->tab_dmax)     // row lists or constant tables that are not there
        return fail(RS_EINVAL, "rs_score: the last change of the graph failed half way; repeat it (or rs_set_tuning) first");
    if (!g->xS || g->xS_bytes != (g->tune.p3_mirror ? sizeof(SigPair) : sizeof(uint64_t)))
        return fail(RS_EINVAL, "rs_score: the buffers of p3_mirror are missing (rs_set_tuning failed); set it again");
    g->scored_version = g->version;
    if (n == 0) return 0;
    constexpr int NT = kThreads;
    int *err = g->d_flag + 4;
    const int cps = g->tune.ctas_per_sm;
    if (int rc = prepare_score_kernels()) return rc;
    prof_begin(g, s);
    Batch B{g->gid, g->gk, g->k, g->wmax_bits};
    InitArgs I{};
    int64_t init_words = 0;
    auto init = [&](void *p, int64_t words, unsigned long long fill) {
        I.r[I.n++] = InitRange{(unsigned long long *)p, words, fill};
        init_words += words;
    };
    init(g->wmax_bits, g->n_graphs, 0);
    init(g->acc, 3 * n, 0);
    init(err, 1, 0);                                 // (and the unused flag word after it)
    init(g->wq, wq_hv_word(n), 0);                   // row counters and the G_x scan's ticket and tile words
    init(g->p2cnt, 8, 0);                            // P2 list counts; word 8: the last node with slots
    if (g->n_hubs) {
        init(g->hkey, g->hub_slots / 2, ~0ull);      // tables are powers of two of at least 2 slots
        init(g->hcnt, g->hub_slots / 2, 0);
        init(g->hq, 2 * g->hub_slots, 0);
        init(g->hagg, g->n_hubs * (int64_t)(sizeof(HubAgg) / sizeof(unsigned long long)), 0);
    }
    if (g->strict) init(g->sx, 2 * g->nnz, 0);
    static_assert(sizeof(HubAgg) % sizeof(unsigned long long) == 0, "HubAgg is cleared by words");
    RS_CUDA_TRY(launch(false, init_kernel, grid_for(init_words / 2 + 1, NT, 8), NT, 0, s, I));
    RS_LAUNCHED(g, s, "init");
    size_t p1_smem = 8 * (size_t)g->large_cap, p2_smem = 32 * (size_t)g->large_cap;
    // streams of the row kernels (rows_streams): every class on its own stream (0); the hub
    // chain on stream 3 and every other class in turn on stream 0 (1); every kernel in turn
    // on the step's stream (2).  On large graphs with hub rows each class fills the GPU alone,
    // and the classes spread over six streams held the hub chain back (8M-node hub-skewed
    // graph: step 65.7 ms against 63.9 with two streams; a batch of 1,024 graphs: 46.5 against
    // 42.1 ms); on smaller graphs the classes' long per-row chains overlap best on separate
    // streams (1M-node graph without hubs: 0.901 against 1.039 ms; a 1.2M-node graph with 489
    // hubs: 1.095 against 1.189 ms).  The automatic choice (-1) takes two streams for graphs
    // with hub rows and at least kRowsTwoStreamNnz CSR entries.
    constexpr int64_t kRowsTwoStreamNnz = 32000000;
    const int rmode = g->tune.rows_streams >= 0 ? g->tune.rows_streams
                                                : (g->n_hubs && g->nnz >= kRowsTwoStreamNnz ? 1 : 0);
    // (a phase with one class of rows takes the step's stream, and only the streams in use are
    // forked and joined)
    const bool mid_large = g->n_mid + g->n_large > 0;
    // at most two 32-row tiles per SM: smaller ones
    // (and where launches are most of the time, chained ones)
    const bool few_rows = g->n_small <= 32 * 2 * (int64_t)grid_for(INT64_MAX / 2, 1, 1);
    unsigned used = 0;
    auto plan = [&](std::initializer_list<std::pair<int, bool>> classes) {
        used = 0;
        int k = 0;
        if (rmode != 2)
            for (auto &c : classes)
                if (c.second) { used |= 1u << (rmode == 1 ? (c.first == 3 ? 3 : 0) : c.first); ++k; }
        if (k < 2) used = 0;
    };
    auto AX = [&](int i) -> cudaStream_t {
        const int j = rmode == 1 ? (i == 3 ? 3 : 0) : i;
        return used >> j & 1 ? g->aux[j] : s;
    };
    const bool chain = few_rows && !mid_large && !g->n_hubs && !g->strict;
    plan({{3, g->n_hubs > 0}, {2, g->n_large > 0}, {4, g->n_mid > 0}, {0, g->n_small > 0}});
    // ---- P1: the larger classes are launched first (with per-class streams, on
    //      high-priority ones), so their maxima seed w_max early and most small rows skip
    //      theirs (the small rows fill in at the lowest priority)
    if (int rc = fork_aux(g, s, used)) return rc;
    if (g->n_hubs) {
        hub_p1_insert_kernel<NT><<<grid_for(g->n_hub_items, 1, 8), NT, 0, AX(3)>>>(
            g->off, g->col, g->lab, g->hubs, g->hub_items, g->hub_item_chunk, g->n_hub_items,
            g->tune.hub_chunk, g->hkey, g->hcnt, g->hagg, err);
        RS_LAUNCHED(g, AX(3), "hub_p1_insert");
        hub_p1_sums_kernel<NT><<<grid_for(g->n_hub_sitems, 1, 8), NT, 0, AX(3)>>>(
            g->hubs, g->hub_sitem, g->hub_srange, g->n_hub_sitems, g->LG, g->hkey, g->hcnt, g->hagg);
        RS_LAUNCHED(g, AX(3), "hub_p1_sums");
        hub_p1_finish_kernel<NT><<<(unsigned)((g->n_hubs + NT - 1) / NT), NT, 0, AX(3)>>>(
            g->off, g->lab, g->hubs, g->n_hubs, B, g->LG, g->hagg, g->rec, g->Lall);
        RS_LAUNCHED(g, AX(3), "hub_p1_finish");
        hub_p1_colmax_kernel<NT><<<grid_for(g->n_hub_sitems, 1, 8), NT, 0, AX(3)>>>(
            g->off, g->hubs, g->hub_sitem, g->hub_srange, g->n_hub_sitems, B, g->LG, g->hkey, g->hcnt, g->hagg,
            g->hsig);
        RS_LAUNCHED(g, AX(3), "hub_p1_colmax");
    }
    if (g->n_large) {
        switch (g->tune.p1_cta_threads) {
        case 128: launch_p1_large<128>(g, B, err, p1_smem, AX(2)); break;
        case 512: launch_p1_large<512>(g, B, err, p1_smem, AX(2)); break;
        default: launch_p1_large<256>(g, B, err, p1_smem, AX(2)); break;
        }
        RS_LAUNCHED(g, AX(2), "p1_large");
    }
    if (g->n_mid) {
        p1_mid_kernel<<<grid_for(g->n_mid * 32, NT, cps), NT, 0, AX(4)>>>(
            g->off, g->col, g->lab, g->rows_mid, g->n_mid, B, g->LG, g->rec, g->Lall, err,
            g->rsum, g->cl_col, g->cl_lab, g->wq + 0);
        RS_LAUNCHED(g, AX(4), "p1_mid");
    }
    if (g->n_small) {
        if (g->tune.p1_stage)
            p1_small_staged_kernel<<<grid_for(g->n_small, kStageWarps * 32, cps), kStageWarps * 32,
                                     kStageWarps * (sizeof(SmallTile) + sizeof(SmallStage)), AX(0)>>>(
                g->off, g->col, g->lab, g->rows_small, g->n_small, B, g->LG, g->rec, g->Lall,
                g->rsum, g->cl_col, g->cl_lab);
        else if (few_rows)
            RS_CUDA_TRY(launch(chain, p1_small_kernel<kFewRows>, grid_for(g->n_small * (32 / kFewRows), NT, cps), NT, 0, AX(0),
                g->off, g->col, g->lab, g->rows_small, g->n_small, B, g->LG, g->rec, g->Lall,
                g->rsum, g->cl_col, g->cl_lab));
        else
            p1_small_kernel<32><<<grid_for(g->n_small, NT, cps), NT, 0, AX(0)>>>(
                g->off, g->col, g->lab, g->rows_small, g->n_small, B, g->LG, g->rec, g->Lall,
                g->rsum, g->cl_col, g->cl_lab);
        RS_LAUNCHED(g, AX(0), "p1_small");
    }
    if (int rc = join_aux(g, s, used)) return rc;
    // ---- the G_x offsets (and the mirror's tiles) and the P2 row lists, in one launch
    const int64_t nm = g->n_mid, nl = g->n_large;
    auto Lst = [&](int c) { return g->p2rows + p2_list_start(c, nm, nl); };
    int32_t *last_node = g->p2cnt + 8;
    const int64_t gx_tiles = (n + kGxTile - 1) / kGxTile;
    const int split_blocks = mid_large ? grid_for(nm + nl, kGxThreads, 8) : 0;
    RS_CUDA_TRY(launch(chain, gx_offsets_kernel, (unsigned)(split_blocks + gx_tiles), kGxThreads, 0, s,
        g->rec, n, g->xoff, g->wq + kWqGxStatus, g->wq + kWqGxTicket, err, g->gx_spin, g->gx_withhold,
        g->tune.p3_mirror ? g->xtile : nullptr, last_node,
        P2Split{g->rows_mid, g->rows_large, nm, nl, g->tune.p2_cta_dx, g->p2rows, g->p2cnt}, split_blocks));
    RS_LAUNCHED(g, s, "gx_offsets");
    const Strict SX{g->col, g->strict ? g->sx : nullptr};
    if (g->strict) {
        strict_pairs_kernel<<<grid_for(g->nnz, NT, cps), NT, 0, s>>>(n, g->off, g->col, g->lab, g->rec, g->cl_col, B,
                                                                     g->tune.small_max, g->tune.cta_cap, g->sx);
        RS_LAUNCHED(g, s, "strict_pairs");
    }
    // ---- P2: with per-class streams, the many-short-rows kernels on the low-priority
    //      streams 0 and 1, the rows with long chains on the others.  The hub
    //      chain (three dependent kernels, the longest of the phase on hub-skewed graphs)
    //      is issued first, so that its blocks are dispatched ahead of the other classes'
    plan({{3, g->n_hubs > 0}, {0, g->n_small > 0}, {1, mid_large}, {5, mid_large}, {2, mid_large}, {4, g->n_large > 0}});
    if (int rc = fork_aux(g, s, used)) return rc;
    auto p2 = [&](auto *xS) -> int {
        using Slot = std::remove_pointer_t<decltype(xS)>;
        if (g->n_hubs) {
            hub_p2_insert_kernel<NT><<<grid_for(g->n_hub_items, 1, 8), NT, 0, AX(3)>>>(
                g->off, g->col, g->hubs, g->hub_items, g->hub_item_chunk, g->n_hub_items, g->tune.hub_chunk, g->rec,
                g->hkey, g->hq,
                g->hitem_out, g->hitem_in, g->hslot, err);
            RS_LAUNCHED(g, AX(3), "hub_p2_insert");
            hub_p2_counts_kernel<NT><<<(unsigned)((g->n_hubs + NT - 1) / NT), NT, 0, AX(3)>>>(
                g->hubs, g->n_hubs, g->hitem_out, g->hitem_in, g->xoff, g->rec, g->xout, g->xin, g->xnode);
            RS_LAUNCHED(g, AX(3), "hub_p2_counts");
            hub_p2_emit_kernel<NT, Slot><<<grid_for(g->n_hub_items, 1, 8), NT, 0, AX(3)>>>(
                g->off, g->col, g->hubs, g->hub_items, g->hub_item_chunk, g->n_hub_items, g->tune.hub_chunk, g->rec,
                g->hslot,
                g->hq, g->hsig, g->hitem_out, g->hitem_in, g->acc, g->xoff, g->xcol, xS, g->xsk, err, SX);
            RS_LAUNCHED(g, AX(3), "hub_p2_emit");
        }
        if (g->n_small) {
            if (few_rows)
                RS_CUDA_TRY(launch(chain, p2_small_kernel<kNarrowRows, Slot>, grid_for(g->n_small * (32 / kNarrowRows), NT, cps), NT, 0, AX(0),
                g->off, g->rows_small, g->n_small, nullptr, g->LG, g->rec, g->rsum, g->cl_col, g->cl_lab, g->acc,
                g->xoff, g->xcol, xS, g->xsk, g->xout, g->xin, g->xnode, SX));
            else
                p2_small_kernel<32, Slot><<<grid_for(g->n_small, NT, cps), NT, 0, AX(0)>>>(
                g->off, g->rows_small, g->n_small, nullptr, g->LG, g->rec, g->rsum, g->cl_col, g->cl_lab, g->acc,
                g->xoff, g->xcol, xS, g->xsk, g->xout, g->xin, g->xnode, SX);
            RS_LAUNCHED(g, AX(0), "p2_small");
        }
        if (mid_large) {
            // the mid and large rows with at most 32 cross neighbours, in the tile kernel
            p2_small_kernel<kNarrowRows, Slot><<<grid_for((nm + nl) * (32 / kNarrowRows), NT, cps), NT, 0, AX(1)>>>(
                g->off, Lst(0), 0, g->p2cnt + 0, g->LG, g->rec, g->rsum, g->cl_col, g->cl_lab, g->acc, g->xoff,
                g->xcol, xS, g->xsk, g->xout, g->xin, g->xnode, SX);
            RS_LAUNCHED(g, AX(1), "p2_narrow");
            p2_mid_kernel<Slot><<<grid_for((nm + nl) * 32, NT, 4), NT, kP2MidSmem, AX(5)>>>(
                g->off, Lst(1), g->p2cnt + 1, B, g->LG, g->rec, g->rsum, g->cl_col, g->cl_lab, g->acc, g->xoff, g->xcol,
                xS, g->xsk, g->xout, g->xin, g->xnode, err, SX, g->wq + 2);
            RS_LAUNCHED(g, AX(5), "p2_mid");
            launch_p2_large<kP2SmallCta>(g, xS, B, err, 32 * (size_t)kWarpCap, 2, 8, g->wq + 3, AX(2));
            RS_LAUNCHED(g, AX(2), "p2_cta");
        }
        if (g->n_large) {
            switch (g->tune.p2_cta_threads) {
            case 256: launch_p2_large<256>(g, xS, B, err, p2_smem, 3, 2, g->wq + 6, AX(4)); break;
            case 512: launch_p2_large<512>(g, xS, B, err, p2_smem, 3, 2, g->wq + 6, AX(4)); break;
            default: launch_p2_large<1024>(g, xS, B, err, p2_smem, 3, 2, g->wq + 6, AX(4)); break;
            }
            RS_LAUNCHED(g, AX(4), "p2_large");
        }
        return 0;
    };
    if (int rc = g->tune.p3_mirror ? p2(static_cast<SigPair *>(g->xS)) : p2(static_cast<uint64_t *>(g->xS))) return rc;
    if (int rc = join_aux(g, s, used)) return rc;
    // ---- P3: reverse values (mirror mode), then triangles
    if (g->tune.p3_mirror) {
        RS_CUDA_TRY(launch(chain, gx_mirror_kernel, grid_for(g->nnz, kMirTile, cps), NT, 0, s, n, g->xoff, g->xcol, static_cast<SigPair *>(g->xS), g->xnode,
                                                                       g->xin, g->xtile, last_node, g->xsk, err));
        RS_LAUNCHED(g, s, "gx_mirror");
    }
    const Rev R{g->xS, g->xoff, g->xcol, g->xin, err, g->tune.p3_mirror != 0};
    unsigned long long *next_group = g->wq + 7;
    unsigned long long *hvl = g->wq + wq_hv_word(n);
    const int64_t hvcap = hv_cap(g->nnz);
    // nodes per group: 32, or fewer on graphs with too few groups of 32 to go around
    int32_t group = 32;
    while (group > 4 && n / group < 16 * (int64_t)grid_for(INT64_MAX / 2, 1, 1)) group >>= 1;
    const int list_grid = grid_for(n, group, kP3CtasPerSm);
    if (g->perm)                                     // a graph numbered by community: scrambled groups
        RS_CUDA_TRY(launch(chain, p3_list_kernel<true>, list_grid, kP3Threads, 0, s, n, g->xoff, g->xcol, g->xsk, R, g->xout, g->xnode, g->acc,
                                                              next_group, group, p3_stride(n), hvl, hvcap,
                                                              g->wq + kWqHvCount));
    else
        RS_CUDA_TRY(launch(chain, p3_list_kernel<false>, list_grid, kP3Threads, 0, s, n, g->xoff, g->xcol, g->xsk, R, g->xout, g->xnode, g->acc,
                                                               next_group, group, 1, hvl, hvcap, g->wq + kWqHvCount));
    RS_LAUNCHED(g, s, "p3_list");
    if (g->dmax > kWinCap) {                         // else no node has that many out-neighbours
        RS_CUDA_TRY(launch(chain, p3_heavy_kernel, grid_for(hvcap, 1, 3), NT, sizeof(P3Heavy), s,
            n, g->xoff, g->xcol, R, g->xout, g->xnode, g->acc, hvl, hvcap, g->wq + kWqHvCount, g->wq + kWqHvNext));
        RS_LAUNCHED(g, s, "p3_heavy");
    }
    // ---- finalize
    if (g->gid) {
        graph_scale_kernel<<<(g->n_graphs + 255) / 256, 256, 0, s>>>(g->wmax_bits, g->n_graphs, g->winv);
        RS_LAUNCHED(g, s, "graph_scale");
    }
    RS_CUDA_TRY(launch(chain && !g->gid, finalize_kernel, grid_for(n, NT, cps), NT, 0, s, n, g->off, g->acc, g->gid, g->winv, g->wmax_bits, g->RD,
                                                         g->perm, scores));
    RS_LAUNCHED(g, s, "finalize");
    return 0;
}
