// Frank-Wolfe for the triangle program (Eq. 4, Alg. 6), exact and binary32.
//
// Layout (the "triangle view", built once per graph).  Vertices are relabelled by
// triangle count, descending.  T is sorted by (a, b, c), so the triangles of one pair
// (a, b) are consecutive: a group.  Only c is stored per triangle, four to a quad,
// every group padded to whole quads; bit 31 of a quad's first c marks the first quad
// of a group, and tv_grp holds the group's (a, b).  tv_chunk_g0 is the group of the
// first quad of each 32-quad chunk.
//
// Pass.  A warp takes a chunk, a lane a quad.  The group's candidate among a and b
// (the smaller load, ties to b) is decided once for the quad; a triangle goes to c
// when its load is not larger, else to that candidate: the lowest-load member, ties
// to the larger id.  The loads of the highest-count vertices are staged in shared
// memory with counters beside them; the receipts of a and b are added once per group
// segment (bit-sliced popcounts over the segment's lanes), those of c one by one.
// Two choice bits per triangle are four ballot words each per chunk: plane 0, b took
// it; plane 1, c took it.  Many iterations (pass, grid barrier, vertex update, grid
// barrier) run in one cooperative launch.  The update also keeps the exact loads
// R = D r of the weights that the choices make: R += 6(i+1) receipts, whatever the
// arithmetic of r.
//
// What bounds it: 4 B of c per triangle from HBM when they exceed L2, about 80 warp
// instructions per 128 triangles, and the shared atomics of the c receipts.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "fw_internal.cuh"
#include "prims.cuh"

namespace lds {

namespace {

namespace cg = cooperative_groups;

constexpr unsigned FULL = 0xffffffffu;
constexpr int TQ_THREADS = 1024;
constexpr int TQ_CHUNK = 32;                     // quads of a warp step
constexpr int32_t TQ_NONE = 0x7fffffff;          // padding (no vertex has this id)
constexpr size_t TQ_SMEM = 224 * 1024;

__device__ __forceinline__ unsigned lanes_le(int lane) { return lane == 31 ? FULL : (2u << lane) - 1u; }

// ---------------------------------------------------------------- view

// receipts of runs are added once: consecutive triangles share a, often b
__global__ void tv_count_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t nt, int32_t* cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < nt; t0 += stride) {
        const int64_t t = t0 + lane;
        const bool ok = t < nt;
        const int32_t a = ok ? ta[t] : -1, b = ok ? tb[t] : -1;
        const unsigned pa = __match_any_sync(FULL, a), pb = __match_any_sync(FULL, b);
        if (!ok) continue;
        if (lane == __ffs(pa) - 1) atomicAdd(cnt + a, __popc(pa));
        if (lane == __ffs(pb) - 1) atomicAdd(cnt + b, __popc(pb));
        atomicAdd(cnt + tc[t], 1);
    }
}

__global__ void tv_rank_keys_kernel(const int32_t* cnt, const int64_t* vt_ptr, int32_t nact, uint64_t* key) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nact; x += stride) {
        const uint32_t c = vt_ptr ? (uint32_t)(vt_ptr[x + 1] - vt_ptr[x]) : (uint32_t)cnt[x];
        key[x] = ((uint64_t)(0xffffffffu - c) << 32) | (uint64_t)x;
    }
}

__global__ void tv_rank_kernel(const uint64_t* key, int32_t nact, int32_t* perm, int32_t* rank, uint32_t* count) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += stride) {
        const int32_t x = (int32_t)(key[p] & 0xffffffffu);
        perm[p] = x;
        rank[x] = (int32_t)p;
        count[p] = 0xffffffffu - (uint32_t)(key[p] >> 32);
    }
}

// bit t of start: triangle t begins a group
__global__ void tv_start_kernel(const int32_t* ta, const int32_t* tb, int64_t nt, uint32_t* start, int32_t* cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5, nw = (nt + 31) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw; w += nwarps) {
        const int64_t t = (w << 5) + lane;
        const bool st = t < nt && (t == 0 || ta[t] != ta[t - 1] || tb[t] != tb[t - 1]);
        const unsigned b = __ballot_sync(FULL, st);
        if (lane == 0) {
            start[w] = b;
            cnt[w] = __popc(b);
        }
    }
}

__global__ void tv_group_kernel(const int32_t* ta, const int32_t* tb, int64_t nt, const uint32_t* start,
                                const int64_t* base, const int32_t* rank, int64_t* gstart, int2* grp, int64_t ng) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride) {
        const uint32_t b = start[t >> 5];
        if (!((b >> (t & 31)) & 1u)) continue;
        const int64_t g = base[t >> 5] + __popc(b & ((1u << (t & 31)) - 1u));
        gstart[g] = t;
        grp[g] = make_int2(rank[ta[t]], rank[tb[t]]);
        if (g == 0) gstart[ng] = nt;
    }
}

__global__ void tv_quads_kernel(const int64_t* gstart, int64_t ng, int32_t* nq) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g <= ng; g += stride)
        nq[g] = g < ng ? (int32_t)((gstart[g + 1] - gstart[g] + 3) >> 2) : 0;
}

__global__ void tv_fill_none_kernel(int32_t* c, int64_t k) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += stride) c[i] = TQ_NONE;
}

__global__ void tv_fill_kernel(const int32_t* tc, int64_t nt, const uint32_t* start, const int64_t* base,
                               const int64_t* gstart, const int64_t* qstart, const int32_t* rank, int32_t* c,
                               uint32_t* qt, int32_t* chunk_g0) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride) {
        const uint32_t b = start[t >> 5];
        const int64_t g = base[t >> 5] + __popc(b & lanes_le((int)(t & 31))) - 1;
        const int64_t off = t - gstart[g], q = qstart[g] + (off >> 2);
        c[4 * q + (off & 3)] = rank[tc[t]] | (off == 0 ? (int32_t)0x80000000 : 0);
        if ((off & 3) == 0) {
            qt[q] = (uint32_t)t;
            if ((q & (TQ_CHUNK - 1)) == 0) chunk_g0[q / TQ_CHUNK] = (int32_t)g;
        }
    }
}

// ---------------------------------------------------------------- iterations

struct TqArgs {
    const int4* c;               // [nq padded to whole chunks]
    const int32_t* chunk_g0;
    const int2* grp;
    int64_t nchunks;
    int32_t nact, nhot;
    void* load;                  // [nact] loads by rank: float, or R as int64 (exact)
    int64_t* R;                  // [nact] exact loads of the weights (binary32 only; exact has them in load)
    uint32_t* cnt;               // [nact] receipts, zero between iterations
    uint4* planes;               // per iteration: [nchunks] words of plane 0, then of plane 1
    int32_t i_first, K;
};

template <class L>
__global__ void __launch_bounds__(TQ_THREADS, 1) fw_tri_quad_kernel(const TqArgs A) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(16) unsigned char smem[];
    L* hl = reinterpret_cast<L*>(smem);
    uint32_t* hc = reinterpret_cast<uint32_t*>(smem + (((size_t)A.nhot * sizeof(L) + 15) & ~(size_t)15));
    L* const load = reinterpret_cast<L*>(A.load);
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + tid, nthreads = (int64_t)gridDim.x * blockDim.x;
    const int64_t warp = gtid >> 5, nwarps = nthreads >> 5;
    const int32_t nhot = A.nhot, nact = A.nact;
    const unsigned le = lanes_le(lane);
    for (int32_t it = 0; it < A.K; ++it) {
        const int32_t i = A.i_first + it;
        for (int32_t j = tid; j < nhot; j += TQ_THREADS) {
            hl[j] = __ldcg(load + j);
            hc[j] = 0;
        }
        __syncthreads();
        uint4* p0 = A.planes + 2 * (int64_t)it * A.nchunks;
        uint4* p1 = p0 + A.nchunks;
        int4 cn = make_int4(TQ_NONE, TQ_NONE, TQ_NONE, TQ_NONE);
        int32_t gn = 0;
        if (warp < A.nchunks) {
            cn = __ldg(A.c + warp * TQ_CHUNK + lane);
            gn = __ldg(A.chunk_g0 + warp);
        }
        for (int64_t ch = warp; ch < A.nchunks; ch += nwarps) {
            const int4 c4 = cn;
            const int32_t g0 = gn;
            if (ch + nwarps < A.nchunks) {
                cn = __ldg(A.c + (ch + nwarps) * TQ_CHUNK + lane);
                gn = __ldg(A.chunk_g0 + ch + nwarps);
            }
            const unsigned f = __ballot_sync(FULL, c4.x < 0);
            const int2 ab = __ldg(A.grp + (g0 + __popc(f & le) - (int)(f & 1u)));
            const int32_t c[4] = {c4.x & 0x7fffffff, c4.y, c4.z, c4.w};
            L rc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int32_t cj = c[j] < nact ? c[j] : 0;
                rc[j] = cj < nhot ? hl[cj] : __ldcg(load + cj);
            }
            const L ra = ab.x < nhot ? hl[ab.x] : __ldcg(load + ab.x);
            const L rb = ab.y < nhot ? hl[ab.y] : __ldcg(load + ab.y);
            const bool to_a = ra < rb;
            const L val = to_a ? ra : rb;
            const int32_t win = to_a ? ab.x : ab.y;
            const unsigned bb = __ballot_sync(FULL, !to_a);
            unsigned w0[4], w1[4];
            int k = 0;                           // triangles of the quad that a or b takes
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool ok = c[j] < nact;
                const bool cw = ok && !(val < rc[j]);
                const unsigned okm = __ballot_sync(FULL, ok);
                w1[j] = __ballot_sync(FULL, cw);
                w0[j] = okm & bb & ~w1[j];
                k += ok && !cw;
                if (cw) {
                    if (c[j] < nhot) atomicAdd(hc + c[j], 1u);
                    else atomicAdd(A.cnt + c[j], 1u);
                }
            }
            if (lane == 0) {
                __stcs(p0 + ch, make_uint4(w0[0], w0[1], w0[2], w0[3]));
                __stcs(p1 + ch, make_uint4(w1[0], w1[1], w1[2], w1[3]));
            }
            // receipts of the group segment: k summed over its lanes by bits
            const unsigned k0 = __ballot_sync(FULL, k & 1), k1 = __ballot_sync(FULL, k & 2), k2 = __ballot_sync(FULL, k & 4);
            if (lane == 0 || ((f >> lane) & 1u)) {
                const unsigned above = f & ~le;
                const unsigned seg = (FULL << lane) & (above ? (above & (0u - above)) - 1u : FULL);
                const unsigned n = __popc(k0 & seg) + 2 * __popc(k1 & seg) + 4 * __popc(k2 & seg);
                if (n) {
                    if (win < nhot) atomicAdd(hc + win, n);
                    else atomicAdd(A.cnt + win, n);
                }
            }
        }
        __syncthreads();
        for (int32_t j = tid; j < nhot; j += TQ_THREADS) {
            const uint32_t v = hc[j];
            if (v) atomicAdd(A.cnt + j, v);
        }
        grid.sync();
        const float gam = __fdiv_rn(2.0f, (float)(i + 2));
        const float om = __fsub_rn(1.0f, gam);
        for (int64_t p = gtid; p < nact; p += nthreads) {
            const uint32_t n = __ldcg(A.cnt + p);
            if (n) A.cnt[p] = 0;
            const int64_t grow = 6 * (int64_t)(i + 1) * (int64_t)n;
            if constexpr (std::is_same<L, float>::value) {
                __stcg(load + p, __fadd_rn(__fmul_rn(om, __ldcg(load + p)), __fmul_rn(gam, (float)n)));
                if (n) A.R[p] += grow;
            } else {
                if (n) __stcg(load + p, __ldcg(load + p) + grow);
            }
        }
        grid.sync();
    }
}

__global__ void tq_init_kernel(const uint32_t* count, int32_t nact, float* r32, int64_t* R) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += stride) {
        R[p] = 2 * (int64_t)count[p];            // R0 = D_0 t / 3, D_0 = 6
        if (r32) r32[p] = __fdiv_rn((float)count[p], 3.0f);
    }
}

// ---------------------------------------------------------------- fold

// 32 x 32 bit transpose over a warp: lane l gives row l and receives column l
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
    uint32_t m = 0x0000ffffu;
#pragma unroll
    for (int s = 16; s; s >>= 1) {
        const uint32_t y = __shfl_xor_sync(FULL, x, s);
        x = (lane & s) ? ((x & ~m) | ((y >> s) & m)) : ((x & m) | ((y << s) & ~m));
        m ^= m << (s >> 1);
    }
    return x;
}

// sum over set bits j of (first + j), by bits of j
__device__ __forceinline__ uint32_t weighted(uint32_t w, uint32_t first) {
    return first * __popc(w) + __popc(w & 0xaaaaaaaau) + 2 * __popc(w & 0xccccccccu) + 4 * __popc(w & 0xf0f0f0f0u) +
           8 * __popc(w & 0xff00ff00u) + 16 * __popc(w & 0xffff0000u);
}

// W of b and of c grow by 6(i+1) per set bit of their plane.  A block takes 8 chunks
// (32 words of each plane), 32 iterations at a time: the words of 32 iterations are
// transposed in the warp, so a lane holds one triangle's 32 choices and adds their
// weights by popcounts.  Word j, bit l of a chunk is item 4 l + j.
constexpr int TF_CHUNKS = 8;
__global__ void __launch_bounds__(1024) fw_tri_fold_kernel(const uint32_t* __restrict__ planes, int nplanes,
                                                           int64_t nchunks, int64_t i_first, uint32_t* Wb, uint32_t* Wc) {
    __shared__ uint32_t tile[2][32][33];
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const int64_t words = 4 * nchunks;
    for (int64_t c0 = (int64_t)blockIdx.x * TF_CHUNKS; c0 < nchunks; c0 += (int64_t)gridDim.x * TF_CHUNKS) {
        uint32_t ab = 0, ac = 0;
        for (int k0 = 0; k0 < nplanes; k0 += 32) {
            const int k = k0 + w;
            const int64_t at = 4 * c0 + lane;
            const bool in = k < nplanes && at < words;
            tile[0][w][lane] = in ? __ldcs(planes + 2 * (int64_t)k * words + at) : 0u;
            tile[1][w][lane] = in ? __ldcs(planes + (2 * (int64_t)k + 1) * words + at) : 0u;
            __syncthreads();
            // warp w takes word w: row l of the matrix is iteration l
            const uint32_t hb = transpose32(tile[0][lane][w], lane), hcc = transpose32(tile[1][lane][w], lane);
            const uint32_t first = (uint32_t)(i_first + k0 + 1);
            ab += 6u * weighted(hb, first);
            ac += 6u * weighted(hcc, first);
            __syncthreads();
        }
        // word w is word (w & 3) of chunk c0 + (w >> 2)
        const int64_t ch = c0 + (w >> 2);
        if (ch < nchunks) {
            const int64_t item = ch * 128 + 4 * lane + (w & 3);
            Wb[item] += ab;
            Wc[item] += ac;
        }
    }
}

// weights and last choices in triangle order
__global__ void tq_output_kernel(const int32_t* c, const uint32_t* qt, int64_t nq, int32_t nact, const uint32_t* Wb,
                                 const uint32_t* Wc, uint32_t D3, int64_t* W, const uint32_t* plane0,
                                 const uint32_t* plane1, uint8_t* last) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += stride) {
        const int64_t t0 = qt[q];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t item = 4 * q + j;
            if ((c[item] & 0x7fffffff) >= nact) break;
            const uint32_t b = Wb[item] + 2u, cc = Wc[item] + 2u;      // W0 = D_0 / 3
            W[3 * (t0 + j)] = (int64_t)(D3 - b - cc);
            W[3 * (t0 + j) + 1] = (int64_t)b;
            W[3 * (t0 + j) + 2] = (int64_t)cc;
            if (last) {
                uint32_t col = 2;
                if (plane0) {
                    const int64_t word = 4 * (q >> 5) + j;
                    col = ((plane0[word] >> (q & 31)) & 1u) | (((plane1[word] >> (q & 31)) & 1u) << 1);
                }
                last[t0 + j] = (uint8_t)col;
            }
        }
    }
}

__global__ void tq_loads_out_kernel(const int32_t* perm, int32_t nact, const int64_t* R, const float* r32, double D3,
                                    int64_t* R_int, double* r_int) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += stride) {
        const int32_t x = perm[p];
        R_int[x] = R[p];
        r_int[x] = r32 ? (double)r32[p] : (double)R[p] / D3;
    }
}

}  // namespace

// Builds the triangle view of the handle if not present (T is listed and not empty).
static void ensure_tri_view(lds_graph* g) {
    if (g->tv_c.p) return;
    cudaStream_t s = g->stream;
    const int blk = 256;
    const int32_t nact = g->nact;
    const int64_t nt = g->ntri;
    DevBuf<int32_t> rank(nact, s), cnt(g->vt_ptr.p ? 0 : nact, s);
    DevBuf<uint64_t> key(nact, s);
    if (!g->vt_ptr.p) {
        LDS_CUDA(cudaMemsetAsync(cnt.get(), 0, nact * sizeof(int32_t), s));
        LDS_LAUNCH(tv_count_kernel, grid_for(nt, blk), blk, 0, s, g->ta.get(), g->tb.get(), g->tc.get(), nt, cnt.get());
    }
    LDS_LAUNCH(tv_rank_keys_kernel, grid_for(nact, blk), blk, 0, s, cnt.get(), g->vt_ptr.get(), nact, key.get());
    radix_sort_u64(key.get(), nullptr, nact, 64, s);
    g->tv_perm.alloc(nact, s);
    g->tv_count.alloc(nact, s);
    LDS_LAUNCH(tv_rank_kernel, grid_for(nact, blk), blk, 0, s, key.get(), nact, g->tv_perm.get(), rank.get(),
               g->tv_count.get());
    const int64_t nw = (nt + 31) / 32;
    DevBuf<uint32_t> start(nw, s);
    DevBuf<int32_t> wc(nw, s);
    DevBuf<int64_t> base(nw, s);
    LDS_LAUNCH(tv_start_kernel, grid_for(nt, blk), blk, 0, s, g->ta.get(), g->tb.get(), nt, start.get(), wc.get());
    const int64_t ng = exclusive_scan_i32_to_i64(wc.get(), base.get(), nw, s);
    DevBuf<int64_t> gstart(ng + 1, s), qstart(ng + 1, s);
    DevBuf<int32_t> nqs(ng + 1, s);
    g->tv_grp.alloc(ng, s);
    LDS_LAUNCH(tv_group_kernel, grid_for(nt, blk), blk, 0, s, g->ta.get(), g->tb.get(), nt, start.get(), base.get(),
               rank.get(), gstart.get(), g->tv_grp.get(), ng);
    LDS_LAUNCH(tv_quads_kernel, grid_for(ng + 1, blk), blk, 0, s, gstart.get(), ng, nqs.get());
    g->tv_nq = exclusive_scan_i32_to_i64(nqs.get(), qstart.get(), ng + 1, s);
    const int64_t chunks = (g->tv_nq + TQ_CHUNK - 1) / TQ_CHUNK;
    DevBuf<int32_t> c(4 * TQ_CHUNK * chunks, s);
    g->tv_qt.alloc(g->tv_nq, s);
    g->tv_chunk_g0.alloc(chunks, s);
    LDS_LAUNCH(tv_fill_none_kernel, grid_for(4 * TQ_CHUNK * chunks, blk), blk, 0, s, c.get(), 4 * TQ_CHUNK * chunks);
    LDS_LAUNCH(tv_fill_kernel, grid_for(nt, blk), blk, 0, s, g->tc.get(), nt, start.get(), base.get(), gstart.get(),
               qstart.get(), rank.get(), c.get(), g->tv_qt.get(), g->tv_chunk_g0.get());
    g->tv_c = std::move(c);
}

void run_tri_fw(lds_graph* g, int N, lds_precision p, bool want_last, PassTimer& timer) {
    cudaStream_t s = g->stream;
    const int blk = 256;
    const int32_t n = g->n, nact = g->nact;
    const int64_t nt = g->ntri;
    const bool fp32 = p == LDS_FP32;
    LDS_CUDA(cudaMemsetAsync(g->fw_R.get(), 0, std::max(n, 1) * sizeof(int64_t), s));
    LDS_CUDA(cudaMemsetAsync(g->fw_r.get(), 0, std::max(n, 1) * sizeof(double), s));
    g->fw_W.alloc(std::max<int64_t>(3 * nt, 1), s);
    if (want_last) g->fw_last.alloc(std::max<int64_t>(nt, 1), s);
    if (nt == 0) return;
    ensure_tri_view(g);
    const int64_t nq = g->tv_nq, nchunks = (nq + TQ_CHUNK - 1) / TQ_CHUNK;
    DevBuf<int64_t> R(nact, s);
    DevBuf<float> r32(fp32 ? nact : 0, s);
    DevBuf<uint32_t> cnt(nact, s);
    LDS_CUDA(cudaMemsetAsync(cnt.get(), 0, nact * sizeof(uint32_t), s));
    LDS_LAUNCH(tq_init_kernel, grid_for(nact, blk), blk, 0, s, g->tv_count.get(), nact, r32.get(), R.get());
    const int K = planes_capacity(8 * nchunks, N);
    DevBuf<uint4> planes(std::max<int64_t>(1, 2 * (int64_t)K * nchunks), s);
    DevBuf<uint32_t> Wb(128 * nchunks, s), Wc(128 * nchunks, s);
    LDS_CUDA(cudaMemsetAsync(Wb.get(), 0, 128 * nchunks * sizeof(uint32_t), s));
    LDS_CUDA(cudaMemsetAsync(Wc.get(), 0, 128 * nchunks * sizeof(uint32_t), s));
    const void* fn = fp32 ? (const void*)fw_tri_quad_kernel<float> : (const void*)fw_tri_quad_kernel<int64_t>;
    LDS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TQ_SMEM));
    const size_t lsize = fp32 ? sizeof(float) : sizeof(int64_t);
    const int32_t nhot = (int32_t)std::min<int64_t>(nact, (int64_t)((TQ_SMEM - 32) / (lsize + 4)));
    const size_t smem = (((size_t)nhot * lsize + 15) & ~(size_t)15) + (size_t)nhot * 4;
    // two chunks a warp at least: a block's staging and flush of the hot vertices is
    // shared by its passes over them
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms(), (nchunks + 63) / 64));
    int stored = 0;
    for (int i = 1; i <= N; i += stored) {
        stored = std::min(K, N - i + 1);
        TqArgs A{reinterpret_cast<const int4*>(g->tv_c.get()), g->tv_chunk_g0.get(), g->tv_grp.get(), nchunks, nact, nhot,
                 fp32 ? (void*)r32.get() : (void*)R.get(), R.get(), cnt.get(), planes.get(), i, stored};
        void* args[] = {(void*)&A};
        timer.start(s);
        LDS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(TQ_THREADS), args, smem, s));
        g_launches.fetch_add(1, std::memory_order_relaxed);
        timer.stop(s, stored);
        const int64_t fblocks = (nchunks + TF_CHUNKS - 1) / TF_CHUNKS;
        LDS_LAUNCH(fw_tri_fold_kernel, (unsigned)std::min<int64_t>(fblocks, (int64_t)num_sms() * 16), 1024, 0, s,
                   reinterpret_cast<const uint32_t*>(planes.get()), stored, nchunks, (int64_t)i, Wb.get(), Wc.get());
    }
    const int64_t D3 = 3 * (int64_t)(N + 1) * (N + 2);
    const uint32_t* last0 = N ? reinterpret_cast<const uint32_t*>(planes.get() + 2 * (int64_t)(stored - 1) * nchunks) : nullptr;
    LDS_LAUNCH(tq_output_kernel, grid_for(nq, blk), blk, 0, s, g->tv_c.get(), g->tv_qt.get(), nq, nact, Wb.get(), Wc.get(),
               (uint32_t)D3, g->fw_W.get(), last0, last0 ? last0 + 4 * nchunks : nullptr,
               want_last ? g->fw_last.get() : nullptr);
    LDS_LAUNCH(tq_loads_out_kernel, grid_for(nact, blk), blk, 0, s, g->tv_perm.get(), nact, R.get(), r32.get(), (double)D3,
               g->fw_R.get(), g->fw_r.get());
}

}  // namespace lds
