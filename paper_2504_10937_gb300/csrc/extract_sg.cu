// ExtractSG (Alg. 2): stable groups and compact-number bounds from the exact
// feasible solution of the last Frank-Wolfe run on a handle.
//
// 1. Vertices are sorted by exact load R = D r descending, ties by id
//    ascending (one radix sort of (Rmax - R, id) keys).
// 2. e_j, the number of patterns (edges or triangles) inside the first j
//    vertices, is a histogram over each pattern's largest position plus a scan.
// 3. Position j is a cut point when e_j / j is strictly larger than e_j' / j'
//    for every j' > j (argmax over j' >= j with ties to the larger j').  A tile
//    reduction, a suffix pass over tiles and a per-tile suffix scan compare the
//    fractions exactly with 128-bit cross products.
// 4. Candidates (segments between cut points) are checked against Def. 5
//    (Def. 12 for triangles) on a modified feasible solution: every pattern that
//    touches the segment S and has a vertex after S (in Z) gives its weight to
//    its lowest-load Z vertex; otherwise, if it has a vertex before S (in X),
//    to its lowest-load S vertex; for an edge that is "all weight to the other
//    endpoint".  S is accepted when every X vertex stays above max_S r' and
//    every Z vertex below min_S r'; a failed candidate merges with the next one
//    (Alg. 2's loop).  For a fixed start, growing the segment only lowers the X
//    vertices' modified loads and only raises max_S r': once the X-side test
//    fails it fails for every longer merge, so the rest is the unaccepted
//    remainder.  The whole walk runs in one cooperative launch
//    (sg_walk_kernel), up to 32 candidates per step.
// 5. Accepted groups give lo = min_S R', hi = max_S R' (over the denominator D);
//    by Lemma 4 / Lemma 8 lo <= D phi(u) <= hi for u in the group.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <climits>
#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "extract_sg.cuh"
#include "prims.cuh"

namespace lds {

namespace {

typedef __int128 i128;

// a/b > c/d for b, d > 0 (the numerator -1 stands for minus infinity)
__device__ __forceinline__ bool frac_gt(int64_t a, int64_t b, int64_t c, int64_t d) {
    return (i128)a * (i128)d > (i128)c * (i128)b;
}

__global__ void rmax_kernel(const int64_t* R, int32_t n, unsigned long long* out) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long m = 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride)
        m = max(m, (unsigned long long)R[x]);
    if (m) atomicMax(out, m);
}

// ties are broken by the original id (internal ids put isolated vertices last)
__global__ void sg_keys_kernel(const int64_t* R, const int32_t* to_orig, int32_t n, uint64_t rmax, int bits,
                               uint64_t* key) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride)
        key[x] = ((rmax - (uint64_t)R[x]) << bits) | (uint64_t)to_orig[x];
}

__global__ void sg_order_kernel(const uint64_t* key, const int32_t* to_int, int32_t n, uint64_t mask, int32_t* order,
                                int32_t* pos) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
        int32_t x = to_int[(int32_t)(key[p] & mask)];
        order[p] = x;
        pos[x] = (int32_t)p;
    }
}

__global__ void sg_hist_edges_kernel(const int32_t* eu, const int32_t* ev, int64_t m, const int32_t* pos, int32_t* h) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride)
        atomicAdd(h + max(pos[eu[e]], pos[ev[e]]), 1);
}

__global__ void sg_hist_tris_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t nt,
                                    const int32_t* pos, int32_t* h) {
    // neighbouring triangles share vertices, and on a skewed graph most maxima are a few
    // positions: one addition per position and warp (R-MAT 18: 3.5 ms to 1.4)
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < nt; t0 += stride) {
        const int64_t t = t0 + lane;
        const int32_t p = t < nt ? max(pos[ta[t]], max(pos[tb[t]], pos[tc[t]])) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, p);
        if (p >= 0 && lane == __ffs(peers) - 1) atomicAdd(h + p, __popc(peers));
    }
}

constexpr int CUT_THREADS = 256;
constexpr int CUT_ITEMS = 4;
constexpr int CUT_TILE = CUT_THREADS * CUT_ITEMS;

// excl_prefix[p] = patterns inside positions < p; e_{p+1} = excl_prefix[p] + h[p].
__device__ __forceinline__ void frac_max(int64_t& a, int64_t& b, int64_t c, int64_t d) {
    if (frac_gt(c, d, a, b)) { a = c; b = d; }
}

__global__ void cut_tilemax_kernel(const int64_t* incl, int32_t n, int64_t* tnum, int64_t* tden) {
    __shared__ int64_t sn[CUT_THREADS], sd[CUT_THREADS];
    int64_t base = (int64_t)blockIdx.x * CUT_TILE + threadIdx.x * CUT_ITEMS;
    int64_t bn = -1, bd = 1;
    for (int k = 0; k < CUT_ITEMS; ++k) {
        int64_t p = base + k;
        if (p < n) frac_max(bn, bd, incl[p], p + 1);
    }
    sn[threadIdx.x] = bn;
    sd[threadIdx.x] = bd;
    __syncthreads();
    for (int o = CUT_THREADS / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            int64_t a = sn[threadIdx.x], b = sd[threadIdx.x];
            frac_max(a, b, sn[threadIdx.x + o], sd[threadIdx.x + o]);
            sn[threadIdx.x] = a;
            sd[threadIdx.x] = b;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        tnum[blockIdx.x] = sn[0];
        tden[blockIdx.x] = sd[0];
    }
}

// suffix max over tiles, exclusive: sfx[b] = max over tiles > b.  One block: thread
// t takes a contiguous share of the tiles, the shares' maxima are combined by a
// suffix scan in shared memory, then every thread walks its share once more.
constexpr int SUF_THREADS = 1024;
__global__ void __launch_bounds__(SUF_THREADS) cut_tile_suffix_kernel(const int64_t* tnum, const int64_t* tden,
                                                                      int64_t ntiles, int64_t* snum, int64_t* sden) {
    __shared__ int64_t sn[SUF_THREADS], sd[SUF_THREADS];
    const int t = threadIdx.x;
    const int64_t lo = ntiles * t / SUF_THREADS, hi = ntiles * (t + 1) / SUF_THREADS;
    int64_t a = -1, b = 1;
    for (int64_t i = lo; i < hi; ++i) frac_max(a, b, tnum[i], tden[i]);
    sn[t] = a;
    sd[t] = b;
    __syncthreads();
    for (int o = 1; o < SUF_THREADS; o <<= 1) {
        int64_t cn = -1, cd = 1;
        if (t + o < SUF_THREADS) { cn = sn[t + o]; cd = sd[t + o]; }
        __syncthreads();
        frac_max(a, b, cn, cd);
        sn[t] = a;
        sd[t] = b;
        __syncthreads();
    }
    a = -1;
    b = 1;
    if (t + 1 < SUF_THREADS) { a = sn[t + 1]; b = sd[t + 1]; }
    for (int64_t i = hi - 1; i >= lo; --i) {
        snum[i] = a;
        sden[i] = b;
        frac_max(a, b, tnum[i], tden[i]);
    }
}

__global__ void cut_flags_kernel(const int64_t* incl, int32_t n, const int64_t* snum, const int64_t* sden,
                                 int32_t* flag) {
    __shared__ int64_t sn[CUT_THREADS], sd[CUT_THREADS];
    const int t = threadIdx.x;
    int64_t base = (int64_t)blockIdx.x * CUT_TILE + t * CUT_ITEMS;
    // max of this thread's items
    int64_t mn = -1, md = 1;
    for (int k = 0; k < CUT_ITEMS; ++k) {
        int64_t p = base + k;
        if (p < n) frac_max(mn, md, incl[p], p + 1);
    }
    sn[t] = mn;
    sd[t] = md;
    __syncthreads();
    // exclusive suffix max over threads t+1.. (Hillis-Steele on a reversed scan)
    int64_t an = mn, ad = md;       // inclusive suffix value
    for (int o = 1; o < CUT_THREADS; o <<= 1) {
        int64_t cn = -1, cd = 1;
        if (t + o < CUT_THREADS) { cn = sn[t + o]; cd = sd[t + o]; }
        __syncthreads();
        frac_max(an, ad, cn, cd);
        sn[t] = an;
        sd[t] = ad;
        __syncthreads();
    }
    int64_t rn = snum[blockIdx.x], rd = sden[blockIdx.x];
    if (t + 1 < CUT_THREADS) frac_max(rn, rd, sn[t + 1], sd[t + 1]);
    for (int k = CUT_ITEMS - 1; k >= 0; --k) {
        int64_t p = base + k;
        if (p >= n) continue;
        int64_t en = incl[p], ed = p + 1;
        flag[p] = frac_gt(en, ed, rn, rd) ? 1 : 0;
        frac_max(rn, rd, en, ed);
    }
}

__global__ void cut_list_kernel(const int32_t* flag, const int64_t* excl, int32_t n, int64_t* cuts) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride)
        if (flag[p]) cuts[excl[p]] = p + 1;
}


constexpr int SW_COLS = 32;
constexpr int SW_THREADS = 1024;
constexpr int SW_ACC = 4 * SW_COLS + 2;      // min X, max S, min S, max Z per column; untouched S min, Z max

// ---- candidate i is the positions (cuts[i-1], cuts[i]]; pattern incidences of a
// position: the edges (triangles) of its vertex.

// *rows: 1 + the last position whose vertex has a pattern
__global__ void sg_positions_kernel(const int64_t* R, const int32_t* order, int32_t n, const int64_t* ptr, int32_t nact,
                                    int64_t* Rp, int64_t* icnt, unsigned long long* acc, int32_t* rows) {
    if (blockIdx.x == 0 && threadIdx.x < SW_ACC) {
        const int i = threadIdx.x, kind = i < 4 * SW_COLS ? i / SW_COLS : i - 4 * SW_COLS + 2;
        acc[i] = (kind & 1) ? 0ull : ~0ull;      // the first window's extremes
    }
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int32_t last = 0;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p <= n; p += stride) {
        if (p == n) {
            icnt[p] = 0;
            continue;
        }
        const int32_t x = order[p];
        const int64_t c = (ptr && x < nact) ? ptr[x + 1] - ptr[x] : 0;
        Rp[p] = R[x];
        icnt[p] = c;
        if (c) last = (int32_t)p + 1;
    }
    last = __reduce_max_sync(0xffffffffu, last);
    if ((threadIdx.x & 31) == 0 && last > *rows) atomicMax(rows, last);
}

// A pattern's change of the loads for a segment S, from where each member lies
// (0: before S, in X; 1: in S; 2: after S, in Z):
//   * no member in S: none;
//   * a member in Z: every member outside Z gives its weight to the Z member of
//     largest position (the lowest load in Z);
//   * else a member in X: every X member gives its weight to the S member of
//     largest position;
//   * else (all in S): none.
template <int K>
__device__ __forceinline__ void pattern_delta(const int (&side)[3], const int32_t (&pp)[3], const int64_t (&w)[3],
                                              int64_t (&d)[3]) {
    int tgt = -1, anys = 0, anyx = 0, anyz = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        anyx |= side[j] == 0;
        anys |= side[j] == 1;
        anyz |= side[j] == 2;
        d[j] = 0;
    }
    if (!anys || (!anyz && !anyx)) return;
    const int to = anyz ? 2 : 1;
#pragma unroll
    for (int j = 0; j < K; ++j)
        if (side[j] == to && (tgt < 0 || pp[j] > pp[tgt])) tgt = j;
    int64_t moved = 0;
#pragma unroll
    for (int j = 0; j < K; ++j)
        if (anyz ? side[j] != 2 : side[j] == 0) {
            d[j] = -w[j];
            moved += w[j];
        }
#pragma unroll
    for (int j = 0; j < K; ++j)
        if (j == tgt) d[j] += moved;
}

// ---- the walk of Alg. 2's merge loop, grid-wide, many candidates at a time.
//
// A window takes the next w <= 32 candidates.  In a chain (fixed start a, S = [a,
// b] growing by one candidate per step) column j of the window is the step that
// adds candidate k0 + j; in a run of single candidates column j is that candidate
// alone.  Phase 1: every incidence of the window's positions, one thread each,
// adds its pattern's change of the loads to a table of one row of 32 columns per
// position, at the columns where the change happens (the columns of the pattern's
// members in the window; each pattern once, by its member of largest position).
// Phase 2: one warp per touched row; a chain's row is summed along its columns
// (warp prefix sum), which gives the vertex's load after every step, and lane j
// keeps the extremes of X, S and Z for column j.  Rows that no pattern of the
// window touched hold one load throughout, so the rows touched earlier in the
// chain (list M) add one minimum (S) and one maximum (Z), and the unmodified rest
// of Z is at most its first position's load.  Positions past the last one with a
// pattern (isolated vertices, for triangles those in none) never change and have no
// row: their extremes are the sorted loads at the ends of their range.  (With a row for
// each, 50,000 vertices of 2^23 took a table of 268 MB, and windows of 4 because of it:
// over 50 s after binary64 iterations, 1.6 s so.)  Then every block takes the same
// decision from the 4 x 32 extremes: the first column that accepts or fails on
// the X side ends the chain there, else the next window continues it.
//
// A step of the walk is latency: a candidate's few incidences cannot fill the
// chip, so the bound is the two grid barriers of a window, shared by up to 32
// candidates.  ExtractSG per query, sort included, against one candidate at a time
// in one block (GB300): Barabasi-Albert n = 40,000, 6 rounds 337 -> 3.8 ms; R-MAT
// scale 18 triangles, 2,930 steps 360 -> 24 ms; G(n, p) n = 2,000, 1,207 steps 5.4
// -> 0.9 ms; the 1M-vertex power-law graph, 6 steps 15.1 -> 2.8 ms (there the host
// candidate lists and the slot -> edge sort were most of it).
struct SgWalkArgs {
    const int32_t *order, *pos;
    const int64_t *Rp, *cuts, *cand, *ioff;   // cand: cuts before a position; ioff: incidences before it (n + 1)
    const int64_t* rowptr;
    const int32_t* col;
    const int64_t* eshift;
    const int64_t* vt_ptr;
    const int32_t *vt_idx, *ta, *tb, *tc;
    const int64_t* W;
    int64_t Dn;
    int32_t n, ncand, cols, maxrows;
    const int32_t* rows;                      // 1 + the last position with a pattern
    int64_t cap0, max_windows;
    long long* table;                         // [maxrows][cols], zero between windows
    int64_t* delta;                           // [maxrows] change of a position's load, valid when dstamp is the chain's
    int32_t *stamp, *dstamp;                  // [maxrows] window (chain) that last touched the position
    int32_t *list, *mlist;                    // rows touched in this window; positions touched in this chain
    unsigned long long* acc;                  // [3][SW_ACC]
    int32_t* cnt;                             // [0..2] list counts, [3] mlist count
    int64_t* gend;                            // accepted groups: exclusive end positions and bounds
    int64_t *glo, *ghi;
    int32_t* out;                             // groups, error, windows, steps
};

struct SgTouch {
    const SgWalkArgs& A;
    int32_t win;
    int32_t* cnt;
    __device__ __forceinline__ void mark(int32_t p) const {
        if (__ldcg(A.stamp + p) != win && atomicExch(A.stamp + p, win) != win) A.list[atomicAdd(cnt, 1)] = p;
    }
    __device__ __forceinline__ void add(int c, int32_t p, int64_t v) const {
        mark(p);
        atomicAdd(reinterpret_cast<unsigned long long*>(A.table + (int64_t)p * A.cols + c), (unsigned long long)v);
    }
};

// one incidence: the pattern's changes at every window column of its members
template <int K>
__device__ __forceinline__ void sw_pattern(const SgTouch& T, bool chain, const int32_t (&pp)[3], const int64_t (&w)[3],
                                           int32_t a, int32_t b0, int32_t bw, int32_t k0, int ncol) {
    int col[3];
#pragma unroll
    for (int j = 0; j < K; ++j)
        col[j] = pp[j] < a ? -2 : pp[j] <= b0 ? -1 : pp[j] > bw ? ncol : (int)T.A.cand[pp[j]] - k0;
    int64_t prev[3], d[3];
    int side[3];
    auto sides = [&](int c) {
#pragma unroll
        for (int j = 0; j < K; ++j) {
            if (chain) side[j] = col[j] == -2 ? 0 : col[j] <= c ? 1 : 2;
            else side[j] = col[j] < c ? 0 : col[j] == c ? 1 : 2;
        }
    };
    sides(-1);
    if (chain) {
        pattern_delta<K>(side, pp, w, prev);
    } else {
#pragma unroll
        for (int j = 0; j < K; ++j) prev[j] = 0;
    }
    int done = -1;
#pragma unroll
    for (int r = 0; r < K; ++r) {
        int c = ncol;                        // next column after `done` among the members'
#pragma unroll
        for (int j = 0; j < K; ++j)
            if (col[j] > done && col[j] < c) c = col[j];
        if (c >= ncol) break;
        sides(c);
        pattern_delta<K>(side, pp, w, d);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            if (d[j] != prev[j]) T.add(c, pp[j], d[j] - prev[j]);
            if (chain) prev[j] = d[j];
        }
        done = c;
    }
}

// canonical edge of slot q = (x, y): the slot of the row of the smaller endpoint
// plus that row's shift
__device__ __forceinline__ int64_t edge_of_slot(int32_t x, int32_t y, int64_t q, const int64_t* rowptr,
                                                const int32_t* col, const int64_t* eshift) {
    if (x < y) return q + eshift[x];
    int64_t lo = rowptr[y], hi = rowptr[y + 1];
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (col[mid] < x) lo = mid + 1; else hi = mid;
    }
    return lo + eshift[y];
}

template <bool TRI>
__global__ void __launch_bounds__(SW_THREADS, 1) sg_walk_kernel(const SgWalkArgs A) {
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    __shared__ unsigned long long s_acc[SW_ACC];
    __shared__ int32_t s_B[SW_COLS];                     // end position of each column
    __shared__ int32_t s_w, s_start, s_b0, s_k0, s_chainmode, s_fresh, s_chain, s_ng, s_stop, s_m;
    __shared__ int64_t s_cap, s_steps;
    __shared__ unsigned long long s_rX, s_rS;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + tid, nthreads = (int64_t)gridDim.x * blockDim.x;
    const int32_t n = A.n, P = *A.rows;
    if (P > A.maxrows) {                                 // (vertices with patterns have loads: they sort first)
        if (gtid == 0) A.out[1] = 2;
        return;
    }
    if (tid == 0) {
        s_start = 0;
        s_b0 = -1;
        s_k0 = 0;
        s_chainmode = 1;
        s_fresh = 1;
        s_chain = 1;
        s_ng = 0;
        s_stop = 0;
        s_m = 0;
        s_cap = A.cap0;
        s_steps = 0;
        s_rX = ~0ull;
        s_rS = 0;
    }
    __syncthreads();
    int32_t win = 0;
    for (;; ++win) {
        if (s_stop || s_k0 >= A.ncand) break;
        if (win >= A.max_windows) {
            if (gtid == 0) A.out[1] = 1;
            break;
        }
        unsigned long long* acc = A.acc + (win % 3) * SW_ACC;
        if (wid == 0) {
            // as many candidates as fit the incidence budget, at least one
            const int64_t k = (int64_t)s_k0 + lane;
            const bool in = k < A.ncand && lane < A.cols;
            const int32_t e = in ? (int32_t)A.cuts[k] - 1 : 0;
            const bool ok = in && (lane == 0 || A.ioff[e + 1] - A.ioff[s_b0 + 1] <= s_cap);
            const unsigned bal = __ballot_sync(0xffffffffu, ok);
            s_B[lane] = e;
            if (lane == 0) s_w = bal == 0xffffffffu ? 32 : __ffs(~bal) - 1;
        }
        for (int i = tid; i < SW_ACC; i += blockDim.x) {
            const int kind = i < 4 * SW_COLS ? i / SW_COLS : i - 4 * SW_COLS + 2;     // 0, 2: minima; 1, 3: maxima
            const unsigned long long id = (kind & 1) ? 0ull : ~0ull;
            s_acc[i] = id;
            if (blockIdx.x == 0) A.acc[((win + 1) % 3) * SW_ACC + i] = id;
        }
        if (gtid == 0) {
            A.cnt[(win + 1) % 3] = 0;
            if (s_fresh) A.cnt[3] = 0;
        }
        __syncthreads();
        const int w = s_w;
        const int32_t a = s_start, b0 = s_b0, bw = s_B[w - 1], k0 = s_k0, chain = s_chain;
        const bool cmode = s_chainmode != 0;
        const SgTouch T{A, win + 1, A.cnt + win % 3};
        // phase 1
        const int32_t bm = min(bw, P - 1);
        for (int64_t p = (int64_t)b0 + 1 + gtid; p <= bm; p += nthreads) T.mark((int32_t)p);
        const int64_t i1 = A.ioff[bw + 1];
        for (int64_t i = A.ioff[b0 + 1] + gtid; i < i1; i += nthreads) {
            int32_t lo = b0 + 1, hi = bw + 1;            // the last position with ioff <= i
            while (hi - lo > 1) {
                const int32_t mid = lo + ((hi - lo) >> 1);
                if (A.ioff[mid] <= i) lo = mid; else hi = mid;
            }
            const int32_t x = A.order[lo];
            const int64_t r = i - A.ioff[lo];
            int32_t pp[3];
            int64_t wt[3];
            if (TRI) {
                const int32_t t = A.vt_idx[A.vt_ptr[x] + r];
                const int32_t v0 = A.ta[t], v1 = A.tb[t], v2 = A.tc[t];
                pp[0] = A.pos[v0];
                pp[1] = A.pos[v1];
                pp[2] = A.pos[v2];
                // the pattern's owner: its member of largest position in the window
                if ((pp[0] > lo && pp[0] <= bw) || (pp[1] > lo && pp[1] <= bw) || (pp[2] > lo && pp[2] <= bw)) continue;
                wt[0] = A.W[3 * (int64_t)t];
                wt[1] = A.W[3 * (int64_t)t + 1];
                wt[2] = A.W[3 * (int64_t)t + 2];
                sw_pattern<3>(T, cmode, pp, wt, a, b0, bw, k0, w);
            } else {
                const int64_t q = A.rowptr[x] + r;
                const int32_t y = A.col[q];
                pp[0] = lo;
                pp[1] = A.pos[y];
                if (pp[1] > lo && pp[1] <= bw) continue;
                const int64_t we = A.W[edge_of_slot(x, y, q, A.rowptr, A.col, A.eshift)];
                wt[0] = x < y ? we : A.Dn - we;
                wt[1] = A.Dn - wt[0];
                sw_pattern<2>(T, cmode, pp, wt, a, b0, bw, k0, w);
            }
        }
        grid.sync();
        // phase 2
        {
            unsigned long long mX = ~0ull, xS = 0, mS = ~0ull, xZ = 0;
            const int32_t nl = __ldcg(A.cnt + win % 3);
            const int64_t gw = gtid >> 5, nw = nthreads >> 5;
            const int32_t la = lane == 0 ? b0 + 1 : s_B[lane - 1] + 1, lb = s_B[lane];
            for (int64_t r = gw; r < nl; r += nw) {
                const int32_t p = __ldcg(A.list + r);
                long long d = 0;
                if (lane < w) {
                    long long* cell = A.table + (int64_t)p * A.cols + lane;
                    d = __ldcg(cell);
                    if (d) *cell = 0;
                }
                unsigned long long base = (unsigned long long)A.Rp[p];
                if (cmode) {
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const long long t = __shfl_up_sync(0xffffffffu, d, o);
                        if (lane >= o) d += t;
                    }
                    const bool seen = __ldcg(A.dstamp + p) == chain;
                    const long long old = seen ? (long long)__ldcg(A.delta + p) : 0;
                    if (lane == 31) {
                        A.delta[p] = old + d;
                        if (!seen) {
                            A.dstamp[p] = chain;
                            A.mlist[atomicAdd(A.cnt + 3, 1)] = p;
                        }
                    }
                    base += (unsigned long long)old;
                }
                const unsigned long long v = base + (unsigned long long)d;
                if (lane < w) {
                    if (p < (cmode ? a : la)) mX = min(mX, v);
                    else if (p <= lb) { mS = min(mS, v); xS = max(xS, v); }
                    else xZ = max(xZ, v);
                }
            }
            if (gw < nl && lane < w) {
                atomicMin(s_acc + lane, mX);
                atomicMax(s_acc + SW_COLS + lane, xS);
                atomicMin(s_acc + 2 * SW_COLS + lane, mS);
                atomicMax(s_acc + 3 * SW_COLS + lane, xZ);
            }
            // positions of this chain that the window left alone
            unsigned long long cS = ~0ull, cZ = 0;
            const int32_t m = s_m;
            for (int64_t i = gtid; i < m; i += nthreads) {
                const int32_t p = __ldcg(A.mlist + i);
                if (p < a || __ldcg(A.stamp + p) == win + 1) continue;
                const unsigned long long v = (unsigned long long)A.Rp[p] + (unsigned long long)__ldcg(A.delta + p);
                if (p <= b0) cS = min(cS, v);
                else cZ = max(cZ, v);
            }
            if (m) {
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    cS = min(cS, __shfl_xor_sync(0xffffffffu, cS, o));
                    cZ = max(cZ, __shfl_xor_sync(0xffffffffu, cZ, o));
                }
                if (lane == 0) {
                    atomicMin(s_acc + 4 * SW_COLS, cS);
                    atomicMax(s_acc + 4 * SW_COLS + 1, cZ);
                }
            }
            __syncthreads();
            for (int i = tid; i < SW_ACC; i += blockDim.x) {
                const int kind = i < 4 * SW_COLS ? i / SW_COLS : i - 4 * SW_COLS + 2;
                const unsigned long long v = s_acc[i];
                if (kind & 1) {
                    if (v) atomicMax(acc + i, v);
                } else if (v != ~0ull) {
                    atomicMin(acc + i, v);
                }
            }
        }
        grid.sync();
        // decision, the same in every block
        if (wid == 0) {
            const bool act = lane < w;
            const int32_t la = lane == 0 ? b0 + 1 : s_B[lane - 1] + 1, lb = s_B[lane];
            unsigned long long mx = __ldcg(acc + lane), hi = __ldcg(acc + SW_COLS + lane);
            unsigned long long lo = __ldcg(acc + 2 * SW_COLS + lane), mz = __ldcg(acc + 3 * SW_COLS + lane);
            const int32_t sa = cmode ? a : la;
            const bool past = bw >= P;                   // the window reaches past the rows
            if (past && act && lb >= P) {
                hi = max(hi, (unsigned long long)A.Rp[max(sa, P)]);
                lo = min(lo, (unsigned long long)A.Rp[lb]);
            }
            if (cmode) {
                mx = min(mx, s_rX);
                hi = max(hi, s_rS);
                lo = min(lo, __ldcg(acc + 4 * SW_COLS));
                mz = max(mz, __ldcg(acc + 4 * SW_COLS + 1));
                // the first position of Z that no row stands for
                const int32_t q = past ? max(lb + 1, P) : bw + 1;
                if (q < n) mz = max(mz, (unsigned long long)A.Rp[q]);
            } else if (act) {
                if (la > 0) mx = min(mx, (unsigned long long)A.Rp[la - 1]);
                if (lb + 1 < n) mz = max(mz, (unsigned long long)A.Rp[lb + 1]);
            }
            const bool xok = sa == 0 || mx > hi;
            const bool zok = lb == n - 1 || mz < lo;
            const unsigned accept = __ballot_sync(0xffffffffu, act && xok && zok);
            const unsigned stopx = __ballot_sync(0xffffffffu, act && !xok);
            const unsigned all = w == 32 ? 0xffffffffu : (1u << w) - 1u;
            // the column the window ends at, and whether a group is recorded by this lane
            const unsigned ends = cmode ? (accept | stopx) : (all & ~accept);
            const int f = ends ? __ffs(ends) - 1 : w;
            const bool rec = cmode ? (lane == f && ((accept >> lane) & 1u)) : lane < f;
            if (rec && blockIdx.x == 0) {
                const int32_t at = s_ng + (cmode ? 0 : lane);
                A.gend[at] = (int64_t)lb + 1;
                A.glo[at] = (int64_t)lo;
                A.ghi[at] = (int64_t)hi;
            }
            __syncwarp();
            const unsigned long long lastX = __shfl_sync(0xffffffffu, mx, w - 1), lastS = __shfl_sync(0xffffffffu, hi, w - 1);
            if (lane == 0) {
                int32_t start = a;
                bool again = false;                      // a new chain starts
                s_steps += f < w ? f + 1 : w;
                if (cmode) {
                    if (f == w) {                        // the chain goes on
                        s_b0 = bw;
                        s_k0 = k0 + w;
                        s_cap = min(s_cap * 4, A.cap0 * 256);
                        s_rX = lastX;
                        s_rS = lastS;
                        s_fresh = 0;
                        s_m = __ldcg(A.cnt + 3);
                    } else if ((accept >> f) & 1u) {
                        ++s_ng;
                        start = s_B[f] + 1;
                        s_k0 = k0 + f + 1;
                        s_chainmode = f > 0;             // after a single candidate, try a run of them
                        s_cap = A.cap0;
                        again = true;
                    } else {
                        s_stop = 1;
                    }
                } else {
                    s_ng += f;
                    if (f == w) {
                        start = bw + 1;
                        s_k0 = k0 + w;
                        s_cap = min(s_cap * 4, A.cap0 * 256);
                    } else if ((stopx >> f) & 1u) {
                        s_stop = 1;
                    } else {                             // fails on the Z side: a chain from that candidate
                        start = f == 0 ? b0 + 1 : s_B[f - 1] + 1;
                        s_k0 = k0 + f;
                        s_chainmode = 1;
                        s_cap = A.cap0;
                    }
                    again = true;
                }
                if (again) {
                    s_start = start;
                    s_b0 = start - 1;
                    s_fresh = 1;
                    ++s_chain;
                    if (s_chainmode) s_cap = A.cap0;
                    s_m = 0;
                    s_rX = start > 0 ? (unsigned long long)A.Rp[start - 1] : ~0ull;
                    s_rS = 0;
                }
            }
        }
        __syncthreads();
    }
    if (gtid == 0) {
        A.out[0] = s_ng;
        A.out[2] = win;
        A.out[3] = (int32_t)min(s_steps, (int64_t)INT32_MAX);
    }
}

__global__ void vt_key_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t nt, uint32_t* key,
                              uint32_t* tid) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 3 * nt; i += stride) {
        int64_t t = i / 3;
        int k = (int)(i % 3);
        key[i] = (uint32_t)(k == 0 ? ta[t] : (k == 1 ? tb[t] : tc[t]));
        tid[i] = (uint32_t)t;
    }
}

__global__ void vt_ptr_kernel(const uint32_t* key, int64_t k3, int32_t nact, int64_t* ptr) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k3; i += stride) {
        int64_t x = (int64_t)key[i];
        int64_t prev = i == 0 ? -1 : (int64_t)key[i - 1];
        for (int64_t r = prev + 1; r <= x; ++r) ptr[r] = i;
        if (i == k3 - 1)
            for (int64_t r = x + 1; r <= nact; ++r) ptr[r] = k3;
    }
}

}  // namespace

void build_vertex_triangles(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t nt, int32_t nact,
                            DevBuf<int64_t>& vt_ptr, DevBuf<int32_t>& vt_idx, cudaStream_t s) {
    const int blk = 256;
    vt_idx.alloc(std::max<int64_t>(3 * nt, 1), s);
    if (nt == 0) {
        vt_ptr.alloc(nact + 1, s);
        LDS_CUDA(cudaMemsetAsync(vt_ptr.get(), 0, (nact + 1) * sizeof(int64_t), s));
        LDS_CUDA(cudaStreamSynchronize(s));
        return;
    }
    DevBuf<uint32_t> key(3 * nt, s);
    uint32_t* tid = reinterpret_cast<uint32_t*>(vt_idx.get());
    LDS_LAUNCH(vt_key_kernel, grid_for(3 * nt, blk), blk, 0, s, ta, tb, tc, nt, key.get(), tid);
    radix_sort_u32(key.get(), tid, 3 * nt, bit_length_u64((uint64_t)nact - 1), s);
    vt_ptr.alloc(nact + 1, s);       // last: its presence says that the index is whole
    LDS_LAUNCH(vt_ptr_kernel, grid_for(3 * nt, blk), blk, 0, s, key.get(), 3 * nt, nact, vt_ptr.get());
    LDS_CUDA(cudaStreamSynchronize(s));
}

void ensure_vertex_triangles(lds_graph* g) {
    if (g->vt_ptr.p) return;
    ensure_triangles(g);
    build_vertex_triangles(g->ta.get(), g->tb.get(), g->tc.get(), g->ntri, g->nact, g->vt_ptr, g->vt_idx, g->stream);
}

// 0: windows of up to 32 candidates; 1: windows of one
std::atomic<int> g_sg_variant{0};

// Alg. 2's walk over the candidates (dcuts[0 .. ncut), cand: cuts before each
// position) in one cooperative launch.
static void sg_walk(lds_graph* g, SgState& st, const int64_t* cand) {
    cudaStream_t s = g->stream;
    const int32_t n = g->n;
    const bool tri = g->fw_density == LDS_TRIANGLE;
    const int64_t ncut = st.ncut;
    if (tri) ensure_vertex_triangles(g);
    else ensure_edge_shift(g);
    const int64_t* ptr = tri ? (g->ntri > 0 ? g->vt_ptr.get() : nullptr) : (g->m > 0 ? g->rowptr.get() : nullptr);
    const int64_t incid = tri ? 3 * std::max<int64_t>(g->ntri, 0) : 2 * g->m;
    // Rows: vertices with a pattern have loads above zero, so they sort before the others.
    // Table columns: 32, fewer where that is more than 64 B per vertex and edge (two thirds
    // of the 96 a query is admitted with; fewer than 3 edges a vertex) or than 8 GB, never
    // under 4, so that a long chain still moves in windows.  The other arrays take 64 B per
    // vertex and 32 per row.  Keeping the sum within the 96 would leave 15 columns at 2^20
    // vertices with 200k edges, 300 ms against 164 with 30 (249 with a row for every vertex).
    const int32_t rows = std::max(1, std::min(n, g->nact));
    const int64_t bytes = std::min<int64_t>(64 * (g->m + n) + (1 << 20), (int64_t)1 << 33);
    int32_t cols = (int32_t)std::max<int64_t>(4, std::min<int64_t>(SW_COLS, bytes / 8 / rows));
    if (g_sg_variant.load(std::memory_order_relaxed) == 1) cols = 1;
    DevBuf<int64_t> Rp(n, s), icnt(n + 1, s), delta(rows, s);
    DevBuf<long long> table((size_t)rows * cols, s);
    DevBuf<int32_t> stamps(2 * (size_t)rows, s), lists(2 * (size_t)rows, s), ctl(9, s);
    DevBuf<unsigned long long> acc(3 * SW_ACC, s);
    LDS_CUDA(cudaMemsetAsync(table.get(), 0, (size_t)rows * cols * sizeof(long long), s));
    LDS_CUDA(cudaMemsetAsync(stamps.get(), 0, 2 * (size_t)rows * sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(ctl.get(), 0, 9 * sizeof(int32_t), s));
    LDS_LAUNCH(sg_positions_kernel, grid_for(n + 1, 256), 256, 0, s, g->fw_R.get(), st.order.get(), n, ptr, g->nact,
               Rp.get(), icnt.get(), acc.get(), ctl.get() + 8);
    exclusive_scan_i64_dev(icnt.get(), icnt.get(), (int64_t)n + 1, nullptr, s);
    st.gend.alloc(ncut, s);
    st.lo.alloc(ncut, s);
    st.hi.alloc(ncut, s);
    const void* fn = tri ? (const void*)sg_walk_kernel<true> : (const void*)sg_walk_kernel<false>;
    // few blocks for a small graph: a grid barrier of one block per SM costs more than its
    // share of the work.  The walk's call with 1,024, 4,096 and 16,384 incidences and
    // positions a block: G(n, p) of 2,000 vertices 0.26, 0.29, 0.36 ms; Barabasi-Albert
    // 40,000 0.63, 0.63, 0.78; power law 60,000 3.52, 3.49, 3.56; R-MAT 14 triangles 0.54,
    // 0.53, 0.54
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms(), (incid + n + 4095) / 4096));
    SgWalkArgs A{};
    A.order = st.order.get();
    A.pos = st.pos.get();
    A.Rp = Rp.get();
    A.cuts = st.cuts.get();
    A.cand = cand;
    A.ioff = icnt.get();
    A.rowptr = g->rowptr.get();
    A.col = g->col.get();
    A.eshift = g->edge_shift.get();
    A.vt_ptr = g->vt_ptr.get();
    A.vt_idx = g->vt_idx.get();
    A.ta = g->ta.get();
    A.tb = g->tb.get();
    A.tc = g->tc.get();
    A.W = g->fw_W.get();
    A.Dn = g->fw_D;
    A.n = n;
    A.ncand = (int32_t)ncut;
    A.cols = cols;
    A.maxrows = rows;
    A.rows = ctl.get() + 8;
    A.cap0 = 2 * (int64_t)grid * SW_THREADS;
    A.max_windows = 2 * ncut + 64;           // every second window at least decides a candidate
    A.table = table.get();
    A.delta = delta.get();
    A.stamp = stamps.get();
    A.dstamp = stamps.get() + rows;
    A.list = lists.get();
    A.mlist = lists.get() + rows;
    A.acc = acc.get();
    A.cnt = ctl.get();
    A.gend = st.gend.get();
    A.glo = st.lo.get();
    A.ghi = st.hi.get();
    A.out = ctl.get() + 4;
    void* args[] = {(void*)&A};
    LDS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(SW_THREADS), args, 0, s));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    int32_t h[4];
    LDS_CUDA(cudaMemcpyAsync(h, ctl.get() + 4, sizeof(h), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    LDS_REQUIRE(h[1] != 2, LDS_ECUDA, "extract_sg: a vertex with patterns has no load (internal error)");
    LDS_REQUIRE(h[1] == 0, LDS_ETIMEOUT, "extract_sg: the walk hit its window bound");
    st.ng = h[0];
    st.windows = h[2];
    st.steps = h[3];
}

void extract_sg(lds_graph* g, SgState& st) {
    LDS_REQUIRE(g->fw_valid, LDS_EINVAL, "extract_sg: run lds_fw on this graph first");
    const auto t_start = std::chrono::steady_clock::now();
    cudaStream_t s = g->stream;
    const int blk = 256;
    const int32_t n = g->n;
    const bool tri = g->fw_density == LDS_TRIANGLE;
    st.D = g->fw_D;
    st.order.alloc(std::max(n, 1), s);
    st.pos.alloc(std::max(n, 1), s);
    st.ncut = 0;
    st.ng = 0;
    if (n == 0) return;
    // 1. order by (R desc, id asc)
    DevBuf<unsigned long long> rmax(1, s);
    LDS_CUDA(cudaMemsetAsync(rmax.get(), 0, sizeof(unsigned long long), s));
    LDS_LAUNCH(rmax_kernel, grid_for(n, blk), blk, 0, s, g->fw_R.get(), n, rmax.get());
    unsigned long long hrmax = 0;
    LDS_CUDA(cudaMemcpyAsync(&hrmax, rmax.get(), sizeof(hrmax), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    const int idbits = std::max(1, bit_length_u64((uint64_t)std::max(n - 1, 1)));
    const int rbits = bit_length_u64(hrmax);
    LDS_REQUIRE(rbits + idbits <= 64, LDS_EOVERFLOW, "extract_sg: loads too large for the sort key");
    {
        DevBuf<uint64_t> key(n, s);
        LDS_LAUNCH(sg_keys_kernel, grid_for(n, blk), blk, 0, s, g->fw_R.get(), g->to_orig.get(), n, (uint64_t)hrmax,
                   idbits, key.get());
        radix_sort_u64(key.get(), nullptr, n, rbits + idbits, s);
        LDS_LAUNCH(sg_order_kernel, grid_for(n, blk), blk, 0, s, key.get(), g->to_int.get(), n, (1ull << idbits) - 1ull,
                   st.order.get(), st.pos.get());
    }
    // 2. e_j
    DevBuf<int32_t> h(n, s);
    LDS_CUDA(cudaMemsetAsync(h.get(), 0, n * sizeof(int32_t), s));
    if (!tri && g->m)
        LDS_LAUNCH(sg_hist_edges_kernel, grid_for(g->m, blk), blk, 0, s, g->eu.get(), g->ev.get(), g->m, st.pos.get(), h.get());
    if (tri && g->ntri)
        LDS_LAUNCH(sg_hist_tris_kernel, grid_for(g->ntri, blk), blk, 0, s, g->ta.get(), g->tb.get(), g->tc.get(), g->ntri,
                   st.pos.get(), h.get());
    DevBuf<int64_t> incl(n + 1, s);
    {
        DevBuf<int32_t> h1(n + 1, s);
        LDS_CUDA(cudaMemsetAsync(h1.get(), 0, (n + 1) * sizeof(int32_t), s));
        LDS_CUDA(cudaMemcpyAsync(h1.get(), h.get(), n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
        // exclusive scan of [h0, h1, ..., 0]: entry p + 1 is the inclusive prefix up to p
        exclusive_scan_i32_dev(h1.get(), incl.get(), n + 1, s);
    }
    const int64_t* inclp = incl.get() + 1;     // inclp[p] = e_{p+1}
    // 3. cut points
    const int64_t ntiles = (n + CUT_TILE - 1) / CUT_TILE;
    DevBuf<int64_t> tn(ntiles, s), td(ntiles, s), sn(ntiles, s), sd(ntiles, s);
    LDS_LAUNCH(cut_tilemax_kernel, (unsigned)ntiles, CUT_THREADS, 0, s, inclp, n, tn.get(), td.get());
    LDS_LAUNCH(cut_tile_suffix_kernel, 1, SUF_THREADS, 0, s, tn.get(), td.get(), ntiles, sn.get(), sd.get());
    DevBuf<int32_t> flag(n, s);
    LDS_LAUNCH(cut_flags_kernel, (unsigned)ntiles, CUT_THREADS, 0, s, inclp, n, sn.get(), sd.get(), flag.get());
    DevBuf<int64_t> fex(n, s);
    st.ncut = exclusive_scan_i32_to_i64(flag.get(), fex.get(), n, s);
    st.cuts.alloc(std::max<int64_t>(st.ncut, 1), s);
    LDS_LAUNCH(cut_list_kernel, grid_for(n, blk), blk, 0, s, flag.get(), fex.get(), n, st.cuts.get());
    h.release();
    incl.release();
    flag.release();
    // 4. the candidate walk (the last position is always a cut, so ncut >= 1)
    const double ms_cuts = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
    sg_walk(g, st, fex.get());
    const char* vb = getenv("LDS_VERBOSE");
    if (vb && vb[0] == '1')
        fprintf(stderr, "[extract_sg] n=%d candidates=%lld groups=%d steps=%d windows=%d; sort+cuts %.2f ms, walk %.2f ms\n",
                n, (long long)st.ncut, st.ng, st.steps, st.windows, ms_cuts,
                std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count() - ms_cuts);
}

}  // namespace lds

using namespace lds;

extern "C" lds_status lds_set_extract_variant(int32_t variant) {
    return guard([&] {
        LDS_REQUIRE(variant == 0 || variant == 1, LDS_EINVAL, "lds_set_extract_variant: %d is not 0 or 1", variant);
        g_sg_variant.store(variant, std::memory_order_relaxed);
    });
}

extern "C" lds_status lds_extract_sg(lds_graph* g, int32_t* order, int32_t* ngroups, int64_t* group_end,
                                     int64_t* lo_num, int64_t* hi_num, int64_t* D, int32_t* ncuts, int64_t* cuts) {
    return guard([&] {
        LDS_REQUIRE(g && ngroups, LDS_EINVAL, "lds_extract_sg: NULL argument");
        SgState st;
        extract_sg(g, st);
        const int32_t n = g->n;
        cudaStream_t s = g->stream;
        *ngroups = st.ng;
        if (D) *D = st.D;
        if (ncuts) *ncuts = (int32_t)st.ncut;
        if (n == 0) return;
        DevBuf<int32_t> o;
        if (order) {
            o.alloc(n, s);
            map_ids(st.order.get(), g->to_orig.get(), n, o.get(), s);
        }
        copy_out(order, LDS_MEM_HOST, o.get(), n * sizeof(int32_t), s);
        copy_out(group_end, LDS_MEM_HOST, st.gend.get(), st.ng * sizeof(int64_t), s);
        copy_out(lo_num, LDS_MEM_HOST, st.lo.get(), st.ng * sizeof(int64_t), s);
        copy_out(hi_num, LDS_MEM_HOST, st.hi.get(), st.ng * sizeof(int64_t), s);
        copy_out(cuts, LDS_MEM_HOST, st.cuts.get(), st.ncut * sizeof(int64_t), s);
        LDS_CUDA(cudaStreamSynchronize(s));
    });
}
