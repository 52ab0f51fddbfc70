// Frank-Wolfe for the triangle program (Eq. 4, Alg. 6), exact and binary32.
//
// Layout (the "triangle view", built once per graph).  Vertices are relabelled by
// triangle count, descending.  T is sorted by (a, b, c), so the triangles of one pair
// (a, b) are consecutive: a group.  Only c is stored per triangle, four to a quad;
// bit 31 of a quad's first c marks the first quad of a group, and a list holds the
// groups' (a, b).  Triangles whose three vertices are all among the hot ones (those
// whose loads and counters fit shared memory) come first, the others after them, each
// part with its own groups, padded to whole quads: the hot part, most of a skewed
// graph's triangles, then needs no test of where a vertex lives.
//
// Pass.  A warp takes 32 quads, a lane one.  The group's candidate among a and b
// (the smaller load, ties to b) is decided once for the quad; a triangle goes to c
// when its load is not larger, else to that candidate: the lowest-load member, ties
// to the larger id.  The receipts of a and b are added once per group segment (its
// places that c did not win), those of c one by one.  Two choice bits per triangle
// are four ballot words each per chunk: plane 0, b took it; plane 1, c took it.  Many
// iterations (pass, grid barrier, vertex update, grid barrier) run in one cooperative
// launch.  The update also keeps the exact loads R = D r of the weights that the
// choices make: R += 6(i+1) receipts, whatever the arithmetic of r.
//
// What bounds it: 4 B of c per triangle from HBM when they exceed L2, the warp
// instructions of a chunk, and the shared-memory gathers and atomics of c.  Per
// iteration on R-MAT scale 18 (84.6M triangles, binary32, GB300): 0.38 ms with one
// thread per triangle and global atomics, 0.20 ms with quads whose every access
// chose between shared and global memory (210 instructions a chunk), 0.17 ms with the
// two parts (a chunk then waited 2,000 cycles for its groups' (a, b)), 0.134 ms with
// the fetches a chunk and two ahead.
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
constexpr size_t TQ_SMEM = 224 * 1024;
constexpr int32_t TQ_HOT = (int32_t)(TQ_SMEM / 8) - 8;     // hot ids with 4-byte loads: 4 B and a 4 B counter
constexpr int64_t TQ_HOT_LEAST = 4096;

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

__global__ void tv_rank_keys_kernel(const int32_t* cnt, const int64_t* vt_ptr, int32_t nact, uint32_t* key,
                                    uint32_t* id) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nact; x += stride) {
        const uint32_t c = vt_ptr ? (uint32_t)(vt_ptr[x + 1] - vt_ptr[x]) : (uint32_t)cnt[x];
        key[x] = 0xffffffffu - c;
        id[x] = (uint32_t)x;
    }
}

__global__ void tv_rank_kernel(const uint32_t* key, const uint32_t* id, int32_t nact, int32_t* perm, int32_t* rank,
                               uint32_t* count) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += stride) {
        const int32_t x = (int32_t)id[p];
        perm[p] = x;
        rank[x] = (int32_t)p + 1;                // id 0 is padding
        count[p] = 0xffffffffu - key[p];
    }
}

// bit t of start: triangle t begins a group; of hot: its vertices all have ids below nhot
__global__ void tv_start_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t nt, const int32_t* rank,
                                int32_t nhot, uint32_t* start, uint32_t* hot, int32_t* scnt, int32_t* hcnt) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5, nw = (nt + 31) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw; w += nwarps) {
        const int64_t t = (w << 5) + lane;
        bool st = false, h = false;
        if (t < nt) {
            const int32_t a = ta[t], b = tb[t];
            st = t == 0 || a != ta[t - 1] || b != tb[t - 1];
            h = rank[a] < nhot && rank[b] < nhot && rank[tc[t]] < nhot;
        }
        const unsigned sb = __ballot_sync(FULL, st), hb = __ballot_sync(FULL, h);
        if (lane == 0) {
            start[w] = sb;
            hot[w] = hb;
            scnt[w] = __popc(sb);
            hcnt[w] = __popc(hb);
        }
    }
}

__global__ void tv_group_kernel(int64_t nt, const uint32_t* start, const int64_t* sbase, int64_t* gstart, int64_t ng) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride) {
        const uint32_t b = start[t >> 5];
        if (!((b >> (t & 31)) & 1u)) continue;
        const int64_t g = sbase[t >> 5] + __popc(b & ((1u << (t & 31)) - 1u));
        gstart[g] = t;
        if (g == 0) gstart[ng] = nt;
    }
}

// hot triangles before t
__device__ __forceinline__ int64_t hot_before(int64_t t, int64_t nt, const uint32_t* hot, const int64_t* hbase) {
    if (t >= nt) t = nt;
    const int64_t w = t >> 5;
    return (t & 31) ? hbase[w] + __popc(hot[w] & ((1u << (t & 31)) - 1u)) : hbase[w];
}

// quads of each group in the hot part and in the other, and whether it has any
__global__ void tv_quads_kernel(const int64_t* gstart, int64_t ng, int64_t nt, const uint32_t* hot, const int64_t* hbase,
                                int32_t* qh, int32_t* qx, int32_t* anyh, int32_t* anyx) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g <= ng; g += stride) {
        int64_t h = 0, x = 0;
        if (g < ng) {
            h = hot_before(gstart[g + 1], nt, hot, hbase) - hot_before(gstart[g], nt, hot, hbase);
            x = gstart[g + 1] - gstart[g] - h;
        }
        qh[g] = (int32_t)((h + 3) >> 2);
        qx[g] = (int32_t)((x + 3) >> 2);
        anyh[g] = h > 0;
        anyx[g] = x > 0;
    }
}

struct TvFill {
    const uint32_t *start, *hot;
    const int64_t *sbase, *hbase, *gstart;
    const int64_t *qh, *qx, *gh, *gx;     // per group: first quad and index among the part's groups
    int64_t xquad, xgrp;                  // first quad and group of the second part
    const int32_t* rank;
    int32_t* c;
    uint32_t* it;
    int32_t* chunk_g0;
    int2* grp;
};

__global__ void tv_fill_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t nt, TvFill F) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride) {
        const int64_t w = t >> 5;
        const int l = (int)(t & 31);
        const int64_t g = F.sbase[w] + __popc(F.start[w] & lanes_le(l)) - 1;
        const int64_t gs = F.gstart[g];
        const int64_t hb = hot_before(t, nt, F.hot, F.hbase) - hot_before(gs, nt, F.hot, F.hbase);
        const bool h = (F.hot[w] >> l) & 1u;
        const int64_t off = h ? hb : (t - gs) - hb;
        const int64_t q = (h ? F.qh[g] : F.xquad + F.qx[g]) + (off >> 2);
        const int64_t gi = h ? F.gh[g] : F.xgrp + F.gx[g];
        F.c[4 * q + (off & 3)] = F.rank[tc[t]] | (off == 0 ? (int32_t)0x80000000 : 0);
        F.it[4 * q + (off & 3)] = (uint32_t)t;
        if (off == 0) F.grp[gi] = make_int2(F.rank[ta[t]], F.rank[tb[t]]);
        if ((off & 3) == 0 && (q & (TQ_CHUNK - 1)) == 0) F.chunk_g0[q / TQ_CHUNK] = (int32_t)gi;
    }
}

// ---------------------------------------------------------------- iterations

struct TqArgs {
    const int4* c;               // [nq padded to whole chunks]
    const int32_t* chunk_g0;
    const int2* grp;
    int64_t nchunks, hchunks;    // chunks in all; of the hot part (its ids all below nhot), which comes first
    int32_t nact, nhot;          // vertices 1 .. nact by rank; the first nhot ids are staged
    void* load;                  // [nact + 1] loads by rank: float, or R as int64 (exact)
    int64_t* R;                  // [nact + 1] exact loads of the weights (binary32 only; exact has them in load)
    uint32_t* cnt;               // [nact + 1] receipts, zero between iterations
    uint4* planes;               // per iteration: [nchunks] words of plane 0, then of plane 1
    int32_t i_first, K;
};

// Id 0 is the padding of a quad: its load -1 lies below every load, so it always
// "wins" its place, receives nothing, and needs no test of its own.
template <class L>
__global__ void __launch_bounds__(TQ_THREADS, 1) fw_tri_quad_kernel(const TqArgs A) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(16) unsigned char smem[];
    L* const hl = reinterpret_cast<L*>(smem);
    uint32_t* const hc = reinterpret_cast<uint32_t*>(smem + (((size_t)A.nhot * sizeof(L) + 15) & ~(size_t)15));
    L* const load = reinterpret_cast<L*>(A.load);
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + tid, nthreads = (int64_t)gridDim.x * blockDim.x;
    const uint32_t warp = (uint32_t)(gtid >> 5), nwarps = (uint32_t)(nthreads >> 5), nch = (uint32_t)A.nchunks;
    const uint32_t nhot = (uint32_t)A.nhot, hch = (uint32_t)A.hchunks;
    const unsigned le = lanes_le(lane);
    for (int32_t it = 0; it < A.K; ++it) {
        const int32_t i = A.i_first + it;
        for (uint32_t j = tid; j < nhot; j += TQ_THREADS) {
            hl[j] = __ldcg(load + j);
            hc[j] = 0;
        }
        __syncthreads();
        uint4* const p0 = A.planes + 2 * (int64_t)it * A.nchunks;
        uint4* const p1 = p0 + A.nchunks;
        // three chunks in flight: the groups' (a, b) of this one have arrived, the next one's
        // are fetched (its c have arrived), the c of the one after are fetched
        auto fetch_c = [&](uint32_t ch) { return ch < nch ? __ldg(A.c + (int64_t)ch * TQ_CHUNK + lane) : make_int4(0, 0, 0, 0); };
        auto fetch_g = [&](uint32_t ch) { return ch < nch ? __ldg(A.chunk_g0 + ch) : 0; };
        auto fetch_ab = [&](const int4& c, int32_t g0) {
            const unsigned f = __ballot_sync(FULL, c.x < 0);
            return __ldg(A.grp + (g0 + __popc(f & le) - (int)(f & 1u)));
        };
        int4 ca = fetch_c(warp), cb = fetch_c(warp + nwarps);
        int32_t gb = fetch_g(warp + nwarps);
        int2 aba = fetch_ab(ca, fetch_g(warp));
        // one chunk; ld and add reach a vertex's load and counter
        auto chunk = [&](uint32_t ch, auto&& ld, auto&& add) {
            const int4 c4 = ca, cc = fetch_c(ch + 2 * nwarps);
            const int32_t gc = fetch_g(ch + 2 * nwarps);
            const int2 ab = aba, abb = fetch_ab(cb, gb);
            const unsigned f = __ballot_sync(FULL, c4.x < 0);
            const uint32_t c[4] = {(uint32_t)c4.x & 0x7fffffffu, (uint32_t)c4.y, (uint32_t)c4.z, (uint32_t)c4.w};
            L rc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) rc[j] = ld(c[j]);
            const L ra = ld((uint32_t)ab.x), rb = ld((uint32_t)ab.y);
            const bool to_a = ra < rb;
            const L val = to_a ? ra : rb;
            const unsigned bb = __ballot_sync(FULL, !to_a);
            unsigned w1[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool cw = !(val < rc[j]);
                w1[j] = __ballot_sync(FULL, cw);
                if (cw && c[j] != 0) add(c[j], 1u);
            }
            if (lane == 0) {
                __stcs(p0 + ch, make_uint4(bb & ~w1[0], bb & ~w1[1], bb & ~w1[2], bb & ~w1[3]));
                __stcs(p1 + ch, make_uint4(w1[0], w1[1], w1[2], w1[3]));
            }
            // receipts of a or b in the group segment: its places that c did not win
            if (lane == 0 || c4.x < 0) {
                const unsigned above = f & ~le;
                const unsigned seg = (FULL << lane) & (above ? (above & (0u - above)) - 1u : FULL);
                const unsigned n = 4 * __popc(seg) - (__popc(w1[0] & seg) + __popc(w1[1] & seg) + __popc(w1[2] & seg) +
                                                      __popc(w1[3] & seg));
                if (n) add((uint32_t)(to_a ? ab.x : ab.y), n);
            }
            ca = cb;
            cb = cc;
            gb = gc;
            aba = abb;
        };
        uint32_t ch = warp;
        for (; ch < hch; ch += nwarps)
            chunk(ch, [&](uint32_t x) { return hl[x]; }, [&](uint32_t x, uint32_t v) { atomicAdd(hc + x, v); });
        for (; ch < nch; ch += nwarps)
            chunk(
                ch, [&](uint32_t x) { return *((x < nhot ? hl : load) + x); },
                [&](uint32_t x, uint32_t v) {
                    if (x < nhot) atomicAdd(hc + x, v);
                    else atomicAdd(A.cnt + x, v);
                });
        __syncthreads();
        for (uint32_t j = tid; j < nhot; j += TQ_THREADS) {
            const uint32_t v = hc[j];
            if (v) atomicAdd(A.cnt + j, v);
        }
        grid.sync();
        const float gam = __fdiv_rn(2.0f, (float)(i + 2));
        const float om = __fsub_rn(1.0f, gam);
        for (int64_t p = 1 + gtid; p <= A.nact; p += nthreads) {
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
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p <= nact; p += stride) {
        R[p] = p ? 2 * (int64_t)count[p - 1] : -1;           // R0 = D_0 t / 3, D_0 = 6
        if (r32) r32[p] = p ? __fdiv_rn((float)count[p - 1], 3.0f) : -1.0f;
    }
}

// ---------------------------------------------------------------- outputs

// weights and last choices in triangle order
__global__ void tq_output_kernel(const int32_t* c, const uint32_t* it, int64_t items, const uint32_t* Wb,
                                 const uint32_t* Wc, uint32_t D3, int64_t* W, const uint32_t* plane0,
                                 const uint32_t* plane1, uint8_t* last) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += stride) {
        if ((c[i] & 0x7fffffff) == 0) continue;
        const int64_t t = it[i];
        const uint32_t b = Wb[i] + 2u, cc = Wc[i] + 2u;      // W0 = D_0 / 3
        W[3 * t] = (int64_t)(D3 - b - cc);
        W[3 * t + 1] = (int64_t)b;
        W[3 * t + 2] = (int64_t)cc;
        if (last) {
            uint32_t col = 2;
            if (plane0) {
                const int64_t q = i >> 2, word = 4 * (q >> 5) + (i & 3);
                col = ((plane0[word] >> (q & 31)) & 1u) | (((plane1[word] >> (q & 31)) & 1u) << 1);
            }
            last[t] = (uint8_t)col;
        }
    }
}

__global__ void tq_loads_out_kernel(const int32_t* perm, int32_t nact, const int64_t* R, const float* r32, double D3,
                                    int64_t* R_int, double* r_int) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += stride) {
        const int32_t x = perm[p];
        R_int[x] = R[p + 1];
        r_int[x] = r32 ? (double)r32[p + 1] : (double)R[p + 1] / D3;
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
    DevBuf<uint32_t> key(nact, s), id(nact, s);
    if (!g->vt_ptr.p) {
        LDS_CUDA(cudaMemsetAsync(cnt.get(), 0, nact * sizeof(int32_t), s));
        LDS_LAUNCH(tv_count_kernel, grid_for(nt, blk), blk, 0, s, g->ta.get(), g->tb.get(), g->tc.get(), nt, cnt.get());
    }
    LDS_LAUNCH(tv_rank_keys_kernel, grid_for(nact, blk), blk, 0, s, cnt.get(), g->vt_ptr.get(), nact, key.get(),
               id.get());
    radix_sort_u32(key.get(), id.get(), nact, 32, s);
    g->tv_perm.alloc(nact, s);
    g->tv_count.alloc(nact, s);
    LDS_LAUNCH(tv_rank_kernel, grid_for(nact, blk), blk, 0, s, key.get(), id.get(), nact, g->tv_perm.get(), rank.get(),
               g->tv_count.get());
    const int64_t nw = (nt + 31) / 32;
    DevBuf<uint32_t> start(nw, s), hot(nw, s);
    DevBuf<int32_t> sc(nw, s), hc(nw + 1, s);
    DevBuf<int64_t> sbase(nw, s), hbase(nw + 1, s);
    LDS_CUDA(cudaMemsetAsync(hc.get() + nw, 0, sizeof(int32_t), s));
    LDS_LAUNCH(tv_start_kernel, grid_for(nt, blk), blk, 0, s, g->ta.get(), g->tb.get(), g->tc.get(), nt, rank.get(),
               TQ_HOT, start.get(), hot.get(), sc.get(), hc.get());
    exclusive_scan_i32_dev(hc.get(), hbase.get(), nw + 1, s);
    const int64_t ng = exclusive_scan_i32_to_i64(sc.get(), sbase.get(), nw, s);
    DevBuf<int64_t> gstart(ng + 1, s), qh(ng + 1, s), qx(ng + 1, s), gh(ng + 1, s), gx(ng + 1, s);
    LDS_LAUNCH(tv_group_kernel, grid_for(nt, blk), blk, 0, s, nt, start.get(), sbase.get(), gstart.get(), ng);
    int64_t nqh, nqx, ngh, ngx;
    {
        DevBuf<int32_t> a(ng + 1, s), b(ng + 1, s), c(ng + 1, s), d(ng + 1, s);
        LDS_LAUNCH(tv_quads_kernel, grid_for(ng + 1, blk), blk, 0, s, gstart.get(), ng, nt, hot.get(), hbase.get(), a.get(),
                   b.get(), c.get(), d.get());
        nqh = exclusive_scan_i32_to_i64(a.get(), qh.get(), ng + 1, s);
        nqx = exclusive_scan_i32_to_i64(b.get(), qx.get(), ng + 1, s);
        ngh = exclusive_scan_i32_to_i64(c.get(), gh.get(), ng + 1, s);
        ngx = exclusive_scan_i32_to_i64(d.get(), gx.get(), ng + 1, s);
    }
    g->tv_hchunks = (nqh + TQ_CHUNK - 1) / TQ_CHUNK;
    g->tv_chunks = g->tv_hchunks + (nqx + TQ_CHUNK - 1) / TQ_CHUNK;
    const int64_t items = 4 * TQ_CHUNK * g->tv_chunks;
    DevBuf<int32_t> c(items, s);
    g->tv_it.alloc(items, s);
    g->tv_chunk_g0.alloc(g->tv_chunks, s);
    g->tv_grp.alloc(ngh + ngx, s);
    LDS_CUDA(cudaMemsetAsync(c.get(), 0, items * sizeof(int32_t), s));
    TvFill F{start.get(),  hot.get(), sbase.get(), hbase.get(), gstart.get(), qh.get(), qx.get(),  gh.get(),
             gx.get(),     g->tv_hchunks * TQ_CHUNK, ngh,       rank.get(),   c.get(),  g->tv_it.get(),
             g->tv_chunk_g0.get(), g->tv_grp.get()};
    LDS_LAUNCH(tv_fill_kernel, grid_for(nt, blk), blk, 0, s, g->ta.get(), g->tb.get(), g->tc.get(), nt, F);
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
    const int64_t nchunks = g->tv_chunks, items = 4 * TQ_CHUNK * nchunks;
    DevBuf<int64_t> R((size_t)nact + 1, s);
    DevBuf<float> r32(fp32 ? (size_t)nact + 1 : 0, s);
    DevBuf<uint32_t> cnt((size_t)nact + 1, s);
    LDS_CUDA(cudaMemsetAsync(cnt.get(), 0, ((size_t)nact + 1) * sizeof(uint32_t), s));
    LDS_LAUNCH(tq_init_kernel, grid_for(nact, blk), blk, 0, s, g->tv_count.get(), nact, r32.get(), R.get());
    const int K = planes_capacity(8 * nchunks, N, quad_plane_bytes(nt, 2));
    DevBuf<uint4> planes(std::max<int64_t>(1, 2 * (int64_t)K * nchunks), s);
    DevBuf<uint32_t> Wb(items, s), Wc(items, s);
    LDS_CUDA(cudaMemsetAsync(Wb.get(), 0, items * sizeof(uint32_t), s));
    LDS_CUDA(cudaMemsetAsync(Wc.get(), 0, items * sizeof(uint32_t), s));
    const void* fn = fp32 ? (const void*)fw_tri_quad_kernel<float> : (const void*)fw_tri_quad_kernel<int64_t>;
    LDS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TQ_SMEM));
    const size_t lsize = fp32 ? sizeof(float) : sizeof(int64_t);
    // Two chunks a warp at least: a block's staging and flush of the hot vertices is shared by
    // its passes over them.  And a vertex a thread where there are blocks for it: few
    // triangles on many vertices left the update to a few blocks (10,000 triangles on 30,000
    // vertices: five).
    const int grid = (int)std::max<int64_t>(
        1, std::min<int64_t>(num_sms(), std::max<int64_t>((nchunks + 63) / 64, (nact + TQ_THREADS - 1) / TQ_THREADS)));
    // Hot ids: twice the entries of a block's share, as in the edge pass; binary32 stages
    // all of them when that is within an eighth of all, for the hot part's own form (144k
    // triangles on 17,000 vertices: 8.1 us an iteration so, 8.6 without).  Microseconds an
    // iteration, exact / binary32, of every id that fits in every block on the smaller grid,
    // and so: 216k triangles on 100,000 vertices 15.4 / 16.4, 9.3 / 9.3; 10,000 on 30,000
    // 13.6 / 13.7, 6.6 / 6.8; 246k on 167,000 12.4 / 11.7, 7.8 / 7.0.  From 270,000 quads or
    // so every id that fits is staged.
    const int64_t fit = fp32 ? (int64_t)TQ_HOT : (int64_t)((TQ_SMEM - 32) / (lsize + 4));
    const int64_t every = std::min<int64_t>((int64_t)nact + 1, TQ_HOT);          // ids of the hot part
    int64_t hot = std::max<int64_t>(TQ_HOT_LEAST, 2 * (4 * TQ_CHUNK * nchunks / grid));
    if (fp32 && hot + hot / 8 >= every) hot = std::max(hot, every);
    const int32_t nhot = (int32_t)std::min(std::min<int64_t>((int64_t)nact + 1, fit), hot);
    const size_t smem = (((size_t)nhot * lsize + 15) & ~(size_t)15) + (size_t)nhot * 4;
    // the hot part's own form needs all of its ids staged; else every chunk takes the general one
    const int64_t hchunks = nhot >= every ? g->tv_hchunks : 0;
    int stored = 0;
    for (int i = 1; i <= N; i += stored) {
        stored = std::min(K, N - i + 1);
        TqArgs A{reinterpret_cast<const int4*>(g->tv_c.get()), g->tv_chunk_g0.get(), g->tv_grp.get(), nchunks, hchunks, nact, nhot,
                 fp32 ? (void*)r32.get() : (void*)R.get(), R.get(), cnt.get(), planes.get(), i, stored};
        void* args[] = {(void*)&A};
        timer.start(s);
        LDS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(TQ_THREADS), args, smem, s));
        g_launches.fetch_add(1, std::memory_order_relaxed);
        timer.stop(s, stored);
        fold_quads(reinterpret_cast<const uint32_t*>(planes.get()), stored, nchunks, i, 6, Wb.get(), Wc.get(), s);
    }
    const int64_t D3 = 3 * (int64_t)(N + 1) * (N + 2);
    const uint32_t* last0 = N ? reinterpret_cast<const uint32_t*>(planes.get() + 2 * (int64_t)(stored - 1) * nchunks) : nullptr;
    LDS_LAUNCH(tq_output_kernel, grid_for(items, blk), blk, 0, s, g->tv_c.get(), g->tv_it.get(), items, Wb.get(), Wc.get(),
               (uint32_t)D3, g->fw_W.get(), last0, last0 ? last0 + 4 * nchunks : nullptr,
               want_last ? g->fw_last.get() : nullptr);
    LDS_LAUNCH(tq_loads_out_kernel, grid_for(nact, blk), blk, 0, s, g->tv_perm.get(), nact, R.get(), r32.get(), (double)D3,
               g->fw_R.get(), g->fw_r.get());
}

}  // namespace lds
