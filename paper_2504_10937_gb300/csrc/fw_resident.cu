// Frank-Wolfe (Alg. 1, edge density) of one small or mid-size graph with every CSR
// slot resident in registers for all iterations.
//
// Each CTA owns a contiguous range of rows of the symmetric CSR (whole rows, ranges
// balanced by slots) and keeps its slots in registers: the two endpoints of a slot
// packed in one word, and the weight W = D_i alpha of the row endpoint, which grows
// by 2(i+1) whenever that endpoint takes the edge.  Per iteration a CTA copies the
// load words of all vertices into shared memory, decides its slots (32 at a time by
// ballot; a row segment's receipts are the popcount of its lanes, one shared atomic
// per segment), updates its own rows' words and publishes them; one barrier over the
// CTAs ends the iteration.  Both endpoints of an edge decide it, so no count crosses
// CTAs and no choice plane is written or folded.  Same iterates, ties and rounding
// as the other forms: an edge goes to the endpoint of smaller load, ties to the
// larger id; exact R <- R + 2(i+1) c, or binary32 r <- (1 - gamma) r + gamma c with
// gamma = 2 / (i + 2) and each operation rounded on its own.
//
// An iteration here is latency: the grid-wide pass (fw_quad_kernel and before it one slot a lane) pays two grid
// barriers, a flush of shared counts and gathers from L2 whatever the size, and its
// working set would fit the chip's registers many times over.  What is left is the
// barrier, the copy of the load words (4 B per vertex and CTA, from L2) and about 25
// instructions per 32 slots.  The CTAs are one (no barrier beyond the block's), one
// cluster of 8, or up to one per SM, by the number of slots.  Per iteration against
// the grid-wide pass (GB300): 1,500 vertices with 348k edges 10.4 -> 3.2 us, 40,000
// with 240k edges 10.3 -> 4.2 us, 6,000 with 24k edges 8.1 -> 2.4 us, 300 with 1,500
// edges 4.9 -> 0.85 us (the 8-CTA form that counted both endpoints in shared memory
// took 2.6 us at 2k edges and 5 at 32k).  With 16 slots a thread the registers spill
// (96 to 128 B); 2M slots on 20,000 vertices still take 7.4 us against 9.0 by the pass
// over quads, 1.6M on 8,000 5.6 against 9.0.
#include <cooperative_groups.h>

#include <algorithm>

#include "fw_internal.cuh"

namespace lds {

namespace {

namespace cg = cooperative_groups;

constexpr unsigned FULL = 0xffffffffu;
constexpr int RES_THREADS = 1024;
constexpr int RES_CLUSTER = 8;
constexpr int RES_UMAX = 16;                         // slots per thread at most
constexpr size_t RES_SMEM = 224 * 1024;

enum ResSync { RES_BLOCK, RES_CLUSTER_SYNC, RES_GRID };

struct ResArgs {
    const int64_t* rowptr;
    const int32_t* col;
    const int64_t* eshift;      // canonical edge of slot q = (x, y), x < y: q + eshift[x]
    int32_t nact, N;
    uint32_t* words;            // [2][nact padded to 4] published load words
    int64_t* W;                 // [m] out
    int64_t* R;                 // [nact] out (zero on entry)
    double* r;                  // [nact] out
    uint8_t* last;              // [m] or null
};

// lanes of this chunk that belong to the lane's row segment, from the lanes that
// start one (f)
__device__ __forceinline__ unsigned segment(unsigned f, int lane) {
    const unsigned le = lane == 31 ? FULL : (2u << lane) - 1u;
    const unsigned above = f & ~le;
    const unsigned ge = FULL << (31 - __clz((f & le) | 1u));
    return ge & (above ? (above & (0u - above)) - 1u : FULL);
}

template <int U, bool FP32, ResSync SYNC>
__global__ void __launch_bounds__(RES_THREADS, 1) fw_resident_kernel(const ResArgs A) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ int32_t s_row[2];
    const int32_t nv = A.nact;
    const int32_t nv4 = (nv + 3) & ~3;
    uint32_t* L = sm;                                // load words of every vertex
    uint32_t* C = sm + nv4;                          // receipts of this CTA's rows
    const int tid = threadIdx.x, lane = tid & 31;
    const int b = blockIdx.x, G = gridDim.x;
    if (tid < 2) {
        // first row whose first slot is at or past this CTA's (the next CTA's) share
        const int64_t want = A.rowptr[nv] * (b + tid) / G;
        int32_t lo = 0, hi = nv;
        while (lo < hi) {
            const int32_t mid = (lo + hi) >> 1;
            if (A.rowptr[mid] < want) lo = mid + 1; else hi = mid;
        }
        s_row[tid] = b + tid == G ? nv : lo;
    }
    __syncthreads();
    const int32_t r0 = s_row[0], r1 = s_row[1];
    const int64_t s0 = A.rowptr[r0], s1 = A.rowptr[r1];
    uint32_t xy[U], W[U];
    uint32_t starts = 0, valid = 0;                  // bit u: the slot starts a row segment; exists
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t s = s0 + (int64_t)u * RES_THREADS + tid;
        xy[u] = 0;
        W[u] = 1;                                    // W0 = D_0 / 2
        int32_t x = -1;
        if (s < s1) {
            int32_t lo = r0, hi = r1;                // last row with rowptr <= s
            while (hi - lo > 1) {
                const int32_t mid = (lo + hi) >> 1;
                if (A.rowptr[mid] <= s) lo = mid; else hi = mid;
            }
            x = lo;
            xy[u] = ((uint32_t)x << 16) | (uint32_t)A.col[s];
            valid |= 1u << u;
        }
        const int32_t px = __shfl_up_sync(FULL, x, 1);
        if (lane == 0 || px != x) starts |= 1u << u;
    }
    for (int32_t x = tid; x < nv; x += RES_THREADS) {
        const uint32_t d = (uint32_t)(A.rowptr[x + 1] - A.rowptr[x]);
        L[x] = FP32 ? __float_as_uint(__fmul_rn((float)d, 0.5f)) : d;     // r0 = deg / 2, R0 = D_0 r0 = deg
    }
    for (int32_t x = r0 + tid; x < r1; x += RES_THREADS) C[x - r0] = 0;
    __syncthreads();
    uint32_t took = 0;                               // bit u: the row endpoint took the edge last
    for (int32_t i = 1; i <= A.N; ++i) {
        const uint32_t inc = 2u * (uint32_t)(i + 1);
        took = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned any = __ballot_sync(FULL, (valid >> u) & 1u);
            if (any == 0) break;                     // whole chunks run out together
            const uint32_t x = xy[u] >> 16, y = xy[u] & 0xffffu;
            const uint32_t lx = L[x], ly = L[y];
            bool recv = FP32 ? (__uint_as_float(lx) < __uint_as_float(ly)) : (lx < ly);
            recv |= lx == ly && x > y;               // (equal words are equal loads: no load is -0)
            recv &= (valid >> u) & 1u;
            const unsigned bal = __ballot_sync(FULL, recv);
            const bool start = (starts >> u) & 1u;
            const unsigned f = __ballot_sync(FULL, start);
            if (start && ((valid >> u) & 1u)) {
                const int c = __popc(bal & segment(f, lane));
                if (c) atomicAdd(C + (x - r0), (uint32_t)c);
            }
            if (recv) {
                W[u] += inc;
                took |= 1u << u;
            }
        }
        __syncthreads();
        uint32_t* out = A.words + (int64_t)(i & 1) * nv4;
        const float gam = __fdiv_rn(2.0f, (float)(i + 2));
        const float om = __fsub_rn(1.0f, gam);
        for (int32_t x = r0 + tid; x < r1; x += RES_THREADS) {
            const uint32_t c = C[x - r0];
            C[x - r0] = 0;
            const uint32_t w =
                FP32 ? __float_as_uint(__fadd_rn(__fmul_rn(om, __uint_as_float(L[x])), __fmul_rn(gam, (float)c)))
                     : L[x] + inc * c;
            if (SYNC == RES_BLOCK) L[x] = w;
            else __stcg(out + x, w);
        }
        if (SYNC == RES_BLOCK) {
            __syncthreads();
        } else {
            if (SYNC == RES_CLUSTER_SYNC) cg::this_cluster().sync();
            else cg::this_grid().sync();
            const uint4* in = reinterpret_cast<const uint4*>(out);
            uint4* l4 = reinterpret_cast<uint4*>(L);
#pragma unroll 8
            for (int32_t j = tid; j < nv4 >> 2; j += RES_THREADS) l4[j] = __ldcg(in + j);
            __syncthreads();
        }
    }
    // outputs: W of the lower endpoint's slot, R = the sum of a row's W, r
    const double D = (double)((int64_t)(A.N + 1) * (A.N + 2));
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const bool ok = (valid >> u) & 1u;
        if (__ballot_sync(FULL, ok) == 0) break;
        const uint32_t x = xy[u] >> 16, y = xy[u] & 0xffffu;
        if (ok && x < y) {
            const int64_t e = s0 + (int64_t)u * RES_THREADS + tid + A.eshift[x];
            A.W[e] = (int64_t)W[u];
            if (A.last) A.last[e] = (uint8_t)((took >> u) & 1u);
        }
        if (FP32) {
            // sum of the segment's W: prefix sums at its ends
            const bool start = (starts >> u) & 1u;
            const unsigned seg = segment(__ballot_sync(FULL, start), lane);
            long long p = ok ? (long long)W[u] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long t = __shfl_up_sync(FULL, p, o);
                if (lane >= o) p += t;
            }
            const long long e = __shfl_sync(FULL, p, 31 - __clz(seg));
            if (start && ok)
                atomicAdd(reinterpret_cast<unsigned long long*>(A.R + x), (unsigned long long)(e - p + (long long)W[u]));
        }
    }
    for (int32_t x = r0 + tid; x < r1; x += RES_THREADS) {
        if (!FP32) A.R[x] = (int64_t)L[x];
        A.r[x] = FP32 ? (double)__uint_as_float(L[x]) : (double)L[x] / D;
    }
}

template <ResSync SYNC>
const void* res_kernel(int U, bool fp32) {
    switch (U) {
        case 2: return fp32 ? (const void*)fw_resident_kernel<2, true, SYNC> : (const void*)fw_resident_kernel<2, false, SYNC>;
        case 4: return fp32 ? (const void*)fw_resident_kernel<4, true, SYNC> : (const void*)fw_resident_kernel<4, false, SYNC>;
        case 8: return fp32 ? (const void*)fw_resident_kernel<8, true, SYNC> : (const void*)fw_resident_kernel<8, false, SYNC>;
        default:
            return fp32 ? (const void*)fw_resident_kernel<16, true, SYNC> : (const void*)fw_resident_kernel<16, false, SYNC>;
    }
}

// ---- Alg. 1 literally in binary64 on the same layout: one alpha per slot in a
// register pair, alpha <- (1 - gamma) alpha + gamma alpha_hat, every operation rounded
// on its own (with alpha_hat 0 or 1 that is one product, plus gamma where the row
// endpoint receives), then r_x summed left to right over row x from shared memory by
// one thread.  The binary64 pipe issues two instructions a clock and SM, so a CTA
// takes few slots; two launches an iteration, slot pass and row sums, took 12.3 us on
// 567 vertices with 844 edges, 4.6 us so, most of it a row's 54 additions in turn.
constexpr int R64_UMAX = 4;

struct Res64Args {
    const int64_t* rowptr;
    const int32_t* col;
    const int64_t* eshift;
    int32_t nact, N;
    double* words;              // [2][nact padded to 2] published loads
    int64_t *W, *R;             // [m], [nact] out
    double* r;                  // [nact] out
    uint8_t* last;              // [m] or null
};

template <int U, ResSync SYNC>
__global__ void __launch_bounds__(RES_THREADS, 1) fw_resident64_kernel(const Res64Args A) {
    extern __shared__ __align__(16) double smd[];
    __shared__ int32_t s_row[2];
    const int32_t nv = A.nact, nv2 = (nv + 1) & ~1;
    double* L = smd;                                 // loads of every vertex
    double* S = smd + nv2;                           // this CTA's alphas, in slot order
    const int tid = threadIdx.x;
    const int b = blockIdx.x, G = gridDim.x;
    if (tid < 2) {
        const int64_t want = A.rowptr[nv] * (b + tid) / G;
        int32_t lo = 0, hi = nv;
        while (lo < hi) {
            const int32_t mid = (lo + hi) >> 1;
            if (A.rowptr[mid] < want) lo = mid + 1; else hi = mid;
        }
        s_row[tid] = b + tid == G ? nv : lo;
    }
    __syncthreads();
    const int32_t r0 = s_row[0], r1 = s_row[1];
    const int64_t s0 = A.rowptr[r0], s1 = A.rowptr[r1];
    uint32_t xy[U];
    double alpha[U];
    uint32_t valid = 0, took = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t s = s0 + (int64_t)u * RES_THREADS + tid;
        xy[u] = 0;
        alpha[u] = 0.5;
        if (s < s1) {
            int32_t lo = r0, hi = r1;                // last row with rowptr <= s
            while (hi - lo > 1) {
                const int32_t mid = (lo + hi) >> 1;
                if (A.rowptr[mid] <= s) lo = mid; else hi = mid;
            }
            xy[u] = ((uint32_t)lo << 16) | (uint32_t)A.col[s];
            valid |= 1u << u;
        }
    }
    for (int32_t x = tid; x < nv; x += RES_THREADS) L[x] = 0.5 * (double)(A.rowptr[x + 1] - A.rowptr[x]);
    __syncthreads();
    for (int32_t i = 1; i <= A.N; ++i) {
        const double gam = 2.0 / (double)(i + 2);
        const double om = 1.0 - gam;
        took = 0;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if ((valid >> u) & 1u) {
                const uint32_t x = xy[u] >> 16, y = xy[u] & 0xffffu;
                const double rx = L[x], ry = L[y];
                const bool recv = rx < ry || (rx == ry && x > y);
                double a = __dmul_rn(om, alpha[u]);
                if (recv) {
                    a = __dadd_rn(a, gam);
                    took |= 1u << u;
                }
                alpha[u] = a;
                S[u * RES_THREADS + tid] = a;
            }
        __syncthreads();
        double* out = A.words + (int64_t)(i & 1) * nv2;
        for (int32_t x = r0 + tid; x < r1; x += RES_THREADS) {
            int32_t q = (int32_t)(A.rowptr[x] - s0);
            const int32_t e = (int32_t)(A.rowptr[x + 1] - s0);
            double acc = 0.0;
            // eight loads ahead of the chain of additions
            for (; q + 8 <= e; q += 8) {
                double v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = S[q + j];
#pragma unroll
                for (int j = 0; j < 8; ++j) acc = __dadd_rn(acc, v[j]);
            }
            for (; q < e; ++q) acc = __dadd_rn(acc, S[q]);
            if (SYNC == RES_BLOCK) L[x] = acc;
            else __stcg(out + x, acc);
        }
        if (SYNC == RES_BLOCK) {
            __syncthreads();
        } else {
            if (SYNC == RES_CLUSTER_SYNC) cg::this_cluster().sync();
            else cg::this_grid().sync();
            const double2* in = reinterpret_cast<const double2*>(out);
            double2* l2 = reinterpret_cast<double2*>(L);
#pragma unroll 4
            for (int32_t j = tid; j < nv2 >> 1; j += RES_THREADS) l2[j] = __ldcg(in + j);
            __syncthreads();
        }
    }
    // outputs: every alpha D rounded, R = the sum of a row's, r
    const double D = (double)((int64_t)(A.N + 1) * (A.N + 2));
    int64_t* SI = reinterpret_cast<int64_t*>(S);
#pragma unroll
    for (int u = 0; u < U; ++u)
        if ((valid >> u) & 1u) {
            const uint32_t x = xy[u] >> 16, y = xy[u] & 0xffffu;
            const int64_t w = (int64_t)(uint32_t)llrint(alpha[u] * D);
            SI[u * RES_THREADS + tid] = w;
            if (x < y) {
                const int64_t e = s0 + (int64_t)u * RES_THREADS + tid + A.eshift[x];
                A.W[e] = w;
                if (A.last) A.last[e] = (uint8_t)((took >> u) & 1u);
            }
        }
    __syncthreads();
    for (int32_t x = r0 + tid; x < r1; x += RES_THREADS) {
        int64_t sum = 0;
        for (int64_t q = A.rowptr[x] - s0; q < A.rowptr[x + 1] - s0; ++q) sum += SI[q];
        A.R[x] = sum;
        A.r[x] = L[x];
    }
}

template <ResSync SYNC>
const void* res64_kernel(int U) {
    return U == 1 ? (const void*)fw_resident64_kernel<1, SYNC>
           : U == 2 ? (const void*)fw_resident64_kernel<2, SYNC> : (const void*)fw_resident64_kernel<4, SYNC>;
}

// launch of either form over G CTAs
void res_launch(const void* fn, int G, ResSync sync, size_t smem, void** args, int N, PassTimer& timer, cudaStream_t s) {
    LDS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RES_SMEM));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(RES_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (sync == RES_CLUSTER_SYNC) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = RES_CLUSTER;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = sync == RES_GRID ? 1 : 0;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    timer.start(s);
    LDS_CUDA(cudaLaunchKernelExC(&cfg, fn, args));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    timer.stop(s, N);
}

}  // namespace

// The binary64 form; false when the graph does not fit.
static bool fw_resident64_run(lds_graph* g, int32_t N, uint8_t* last, PassTimer& timer) {
    const int64_t maxdeg = std::max(g->info.max_degree, 1), slots = 2 * g->m;
    // CTAs: one up to 1,024 slots, a cluster of 8 up to 8,192, then one per 1,024 slots, by
    // microseconds an iteration (300 iterations, GB300) of one CTA, a cluster and the grid:
    // 480 slots 3.5, 3.1; 1,800 9.2, 4.5, 7.9; 7,300 14.4, 8.5, 9.2; 10,000 15.5, 11.1, 11.2;
    // 16,700 16.5, 15.0, 12.2; 29,000 20.6, 21.8, 14.0
    constexpr int64_t kShare = 1024;
    int G = slots <= kShare ? 1
            : slots <= RES_CLUSTER * kShare ? RES_CLUSTER : (int)std::min<int64_t>(num_sms(), (slots + kShare - 1) / kShare);
    const int64_t most = G == 1 ? slots : slots / G + maxdeg + 1;
    if (most > (int64_t)R64_UMAX * RES_THREADS) return false;
    int U = 1;
    while ((int64_t)U * RES_THREADS < most) U *= 2;
    const size_t nv2 = ((size_t)g->nact + 1) & ~(size_t)1;
    const size_t smem = (nv2 + (size_t)U * RES_THREADS) * sizeof(double);
    if (smem > RES_SMEM) return false;
    cudaStream_t s = g->stream;
    const ResSync sync = G == 1 ? RES_BLOCK : slots <= RES_CLUSTER * kShare ? RES_CLUSTER_SYNC : RES_GRID;
    const void* fn = sync == RES_BLOCK          ? res64_kernel<RES_BLOCK>(U)
                     : sync == RES_CLUSTER_SYNC ? res64_kernel<RES_CLUSTER_SYNC>(U) : res64_kernel<RES_GRID>(U);
    ensure_edge_shift(g);
    g->fw_W.alloc(g->m, s);
    DevBuf<double> words(2 * nv2, s);
    LDS_CUDA(cudaMemsetAsync(g->fw_R.get(), 0, g->n * sizeof(int64_t), s));
    LDS_CUDA(cudaMemsetAsync(g->fw_r.get(), 0, g->n * sizeof(double), s));
    Res64Args A{g->rowptr.get(), g->col.get(),  g->edge_shift.get(), g->nact, N, words.get(),
                g->fw_W.get(),   g->fw_R.get(), g->fw_r.get(),       last};
    void* args[] = {(void*)&A};
    res_launch(fn, G, sync, smem, args, N, timer, s);
    return true;
}

bool fw_resident_run(lds_graph* g, int32_t N, lds_precision p, uint8_t* last, PassTimer& timer) {
    if (N < 1 || g->m < 1 || g->nact > 65536) return false;
    if (p == LDS_FP64) return fw_resident64_run(g, N, last, timer);
    const bool fp32 = p == LDS_FP32;
    const int64_t maxdeg = std::max(g->info.max_degree, 1), slots = 2 * g->m;
    const unsigned __int128 D = (unsigned __int128)(N + 1) * (unsigned __int128)(N + 2);
    // weights, and exact loads, fit 32 bits
    if ((fp32 ? D : D * (unsigned __int128)maxdeg) >> 32) return false;
    // CTAs, by microseconds an iteration (400 iterations, exact, GB300): one up to 4,096
    // slots (3,000 slots: 0.85 us against 1.28 on a cluster), a cluster of 8 up to
    // 20,480 (16,000: 1.7 against 2.1 grid-wide, 2.6 on four CTAs), then one per 1,024
    // slots up to one per SM (48,000: 2.4 against 3.4 with 4,096 a CTA)
    constexpr int64_t kBlock = 4096, kCluster = 20480, kShare = 1024;
    int G = slots <= kBlock ? 1
            : slots <= kCluster ? RES_CLUSTER
                                : (int)std::min<int64_t>(num_sms(), (slots + kShare - 1) / kShare);
    // slots of a CTA: its share plus what whole rows add
    auto cta_slots = [&](int n) { return n == 1 ? slots : slots / n + maxdeg + 1; };
    const int64_t cap = (int64_t)RES_UMAX * RES_THREADS;
    if (cta_slots(G) > cap) G = num_sms();
    if (cta_slots(G) > cap) return false;
    const int64_t most = cta_slots(G);
    int U = 2;
    while ((int64_t)U * RES_THREADS < most) U *= 2;
    const size_t smem = (((size_t)g->nact + 3) & ~(size_t)3) * 4 + (size_t)std::min<int64_t>(g->nact, most) * 4;
    if (smem > RES_SMEM) return false;
    cudaStream_t s = g->stream;
    const ResSync sync = G == 1 ? RES_BLOCK : G == RES_CLUSTER && slots <= kCluster ? RES_CLUSTER_SYNC : RES_GRID;
    const void* fn = sync == RES_BLOCK          ? res_kernel<RES_BLOCK>(U, fp32)
                     : sync == RES_CLUSTER_SYNC ? res_kernel<RES_CLUSTER_SYNC>(U, fp32)
                                                : res_kernel<RES_GRID>(U, fp32);
    ensure_edge_shift(g);
    g->fw_W.alloc(g->m, s);
    const size_t nv4 = ((size_t)g->nact + 3) & ~(size_t)3;
    DevBuf<uint32_t> words(2 * nv4, s);
    // isolated vertices hold no load; binary32 sums its R into zeros
    LDS_CUDA(cudaMemsetAsync(g->fw_R.get(), 0, g->n * sizeof(int64_t), s));
    LDS_CUDA(cudaMemsetAsync(g->fw_r.get(), 0, g->n * sizeof(double), s));
    ResArgs A{g->rowptr.get(), g->col.get(),   g->edge_shift.get(), g->nact, N, words.get(),
              g->fw_W.get(),   g->fw_R.get(),  g->fw_r.get(),       last};
    void* args[] = {(void*)&A};
    res_launch(fn, G, sync, smem, args, N, timer, s);
    return true;
}

}  // namespace lds
