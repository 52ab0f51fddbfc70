// Frank-Wolfe (Alg. 1, edge density) on graphs past the register-resident form: the
// degree-oriented pass over quads, exact and binary32 with 32-bit load words.
//
// Layout (the "quad view", built once per graph).  Vertices are relabelled by
// (degree descending, id ascending).  Every edge is stored once, in the row of its
// lower-ranked endpoint, as 1 + the rank of its higher-ranked one, four to a quad,
// every row padded to whole quads with 0; fwq_src holds 1 + the rank of each quad's
// row.
//
// Pass.  A warp takes a chunk, a lane a quad: the row's load is read once for four
// targets.  The row endpoint receives an edge when its load is smaller, ties to the
// larger id.  The loads of the highest-degree vertices (the targets of most edges)
// are staged in shared memory, with 16-bit counters packed two to a word beside them
// (a vertex receives at most its degree < 2^16 in an iteration).  The 128 decisions
// of a chunk are four words of the iteration's choice plane: bit l of word j is entry
// j of quad l.  A target's receipts go to the shared counter of a hot target or to
// its global one; a row endpoint's are the popcount of its row's bits, taken by the
// vertex update.  Pass, grid barrier, update, grid barrier: many iterations in one
// cooperative launch.  The update also keeps the exact loads R = D r of the weights
// that the choices make, whatever the arithmetic of r.
//
// What bounds it: the chains of L2 accesses.  A warp has 19 chunks an iteration on the
// 1M-vertex power-law graph, and with the list of rows behind the targets and the loads
// behind both a chunk took 2,800 cycles.  So a quad names its row, the targets of the
// chunk after next and the loads of the next one are fetched while a chunk is decided,
// and the update works on two vertices at a time.  Per iteration there (10.6M edges,
// exact, GB300): 52.3 us before quads, 52 with quads and the dependent loads,
// 41 us so.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "fw_internal.cuh"
#include "prims.cuh"

namespace lds {

namespace {

namespace cg = cooperative_groups;

constexpr unsigned FULL = 0xffffffffu;
constexpr int EQ_THREADS = 1024;
constexpr int EQ_CHUNK = 32;                     // quads of a warp step
constexpr int32_t EQ_HOT = 38144;                // hot ids: 4 B of load and 2 B of count each
constexpr size_t EQ_SMEM = (size_t)EQ_HOT * 6;
constexpr int32_t EQ_HOT_LEAST = 4096;

__device__ __forceinline__ unsigned lanes_le(int lane) { return lane == 31 ? FULL : (2u << lane) - 1u; }

// ---------------------------------------------------------------- view

__global__ void eq_slot_keys_kernel(const int32_t* eu, const int32_t* ev, int64_t m, const int32_t* pos, int bits,
                                    uint64_t* key, uint32_t* eid) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
        const uint32_t a = (uint32_t)pos[eu[e]], b = (uint32_t)pos[ev[e]];
        const bool u_src = a > b;
        key[e] = ((uint64_t)(u_src ? a : b) << bits) | (u_src ? b : a);
        eid[e] = ((uint32_t)e << 1) | (u_src ? 1u : 0u);
    }
}

// first slot of every row, from the sorted keys
__global__ void eq_rowptr_kernel(const uint64_t* key, int64_t m, int bits, int32_t nact, int32_t* rowptr) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < m; s += stride) {
        const int64_t x = (int64_t)(key[s] >> bits), prev = s == 0 ? -1 : (int64_t)(key[s - 1] >> bits);
        for (int64_t r = prev + 1; r <= x; ++r) rowptr[r] = (int32_t)s;
        if (s == m - 1)
            for (int64_t r = x + 1; r <= nact; ++r) rowptr[r] = (int32_t)m;
    }
}

__global__ void eq_row_quads_kernel(const int32_t* rowptr, int32_t nact, int32_t* nq) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= nact; r += stride)
        nq[r] = r < nact ? (rowptr[r + 1] - rowptr[r] + 3) >> 2 : 0;
}

__global__ void eq_qptr_kernel(const int64_t* qp64, int32_t nact, int32_t* qptr) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= nact; r += stride) qptr[r] = (int32_t)qp64[r];
}

__global__ void eq_fill_kernel(const uint64_t* key, int64_t m, int bits, const int32_t* rowptr, const int32_t* qptr,
                               int32_t* c, int32_t* src, int32_t* qs) {
    const uint64_t mask = (1ull << bits) - 1ull;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < m; s += stride) {
        const uint64_t k = key[s];
        const int64_t x = (int64_t)(k >> bits);
        const int32_t off = (int32_t)(s - rowptr[x]);
        const int64_t q = qptr[x] + (off >> 2);
        c[4 * q + (off & 3)] = (int32_t)(k & mask) + 1;
        if ((off & 3) == 0) {
            qs[q] = (int32_t)s;
            src[q] = (int32_t)x + 1;
        }
    }
}

// ---------------------------------------------------------------- iterations

struct EqArgs {
    const int4* c;               // [chunks * 32]
    const int32_t* src;          // [chunks * 32] id of each quad's row (padding: 0)
    const int32_t* qptr;         // [nact + 1] quads of the row of each rank
    const int32_t* perm;         // [nact] rank -> internal id
    int64_t nchunks;
    int32_t nact, nhot;          // ids 1 .. nact by rank; ids below nhot are staged
    void* word;                  // [nact + 1] load words by id: R, or r in binary32; id 0: below every load
    int64_t* R;                  // [nact + 1] exact loads of the weights (binary32)
    uint32_t* cnt;               // [nact + 1] receipts as targets, zero between iterations
    uint4* planes;               // [K][nchunks]
    int32_t i_first, K;
};

template <class Word>
__global__ void __launch_bounds__(EQ_THREADS, 1) fw_quad_kernel(const EqArgs A) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(16) unsigned char smem[];
    Word* const hw = reinterpret_cast<Word*>(smem);
    uint32_t* const hc = reinterpret_cast<uint32_t*>(smem + (size_t)EQ_HOT * 4);     // two 16-bit counts a word
    Word* const word = reinterpret_cast<Word*>(A.word);
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t gtid = blockIdx.x * blockDim.x + tid, nthreads = gridDim.x * blockDim.x;
    const uint32_t warp = gtid >> 5, nwarps = nthreads >> 5, nch = (uint32_t)A.nchunks, nhot = (uint32_t)A.nhot;
    const uint32_t nact = (uint32_t)A.nact;
    for (int32_t it = 0; it < A.K; ++it) {
        const int32_t i = A.i_first + it;
        uint4* const plane = A.planes + (int64_t)it * A.nchunks;
        {
            const uint4* w4 = reinterpret_cast<const uint4*>(word);
            uint4* h4 = reinterpret_cast<uint4*>(hw);
#pragma unroll 4
            for (uint32_t j = tid; j < nhot >> 2; j += EQ_THREADS) h4[j] = __ldcg(w4 + j);
            for (uint32_t j = (nhot & ~3u) + tid; j < nhot; j += EQ_THREADS) hw[j] = __ldcg(word + j);
            for (uint32_t j = tid; j < (nhot + 1) >> 1; j += EQ_THREADS) hc[j] = 0;
        }
        __syncthreads();
        // three chunks in flight: a's loads have arrived, b's targets have, c's are fetched
        struct Quad {
            int4 c;
            uint32_t s;
        };
        auto targets = [&](uint32_t ch) -> Quad {
            if (ch >= nch) return Quad{make_int4(0, 0, 0, 0), 0u};
            return Quad{__ldg(A.c + (int64_t)ch * EQ_CHUNK + lane), (uint32_t)__ldg(A.src + (int64_t)ch * EQ_CHUNK + lane)};
        };
        auto at = [&](uint32_t x) -> Word { return *((x < nhot ? hw : word) + x); };
        Quad qa = targets(warp), qb = targets(warp + nwarps);
        Word wa[5] = {at((uint32_t)qa.c.x), at((uint32_t)qa.c.y), at((uint32_t)qa.c.z), at((uint32_t)qa.c.w), at(qa.s)};
        for (uint32_t ch = warp; ch < nch; ch += nwarps) {
            const Quad qc = targets(ch + 2 * nwarps);
            const Word wb[5] = {at((uint32_t)qb.c.x), at((uint32_t)qb.c.y), at((uint32_t)qb.c.z), at((uint32_t)qb.c.w),
                                at(qb.s)};
            const uint32_t c[4] = {(uint32_t)qa.c.x, (uint32_t)qa.c.y, (uint32_t)qa.c.z, (uint32_t)qa.c.w};
            const Word ws = wa[4];
            unsigned w[4];
            bool tie = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) tie |= ws == wa[j] && c[j] != 0;
            // equal loads are rare; then the ids decide
            int32_t id = 0;
            if (tie) id = __ldg(A.perm + qa.s - 1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                bool recv = ws < wa[j];
                if (tie && ws == wa[j] && c[j] != 0) recv = id > __ldg(A.perm + c[j] - 1);
                recv &= c[j] != 0;
                w[j] = __ballot_sync(FULL, recv);
                if (!recv && c[j] != 0) {
                    if (c[j] < nhot) atomicAdd(hc + (c[j] >> 1), 1u << ((c[j] & 1) << 4));
                    else atomicAdd(A.cnt + c[j], 1u);
                }
            }
            if (lane == 0) __stcg(plane + ch, make_uint4(w[0], w[1], w[2], w[3]));
            qa = qb;
            qb = qc;
#pragma unroll
            for (int j = 0; j < 5; ++j) wa[j] = wb[j];
        }
        __syncthreads();
        for (uint32_t j = tid; j < (nhot + 1) >> 1; j += EQ_THREADS) {
            const uint32_t v = hc[j];
            if (v & 0xffffu) atomicAdd(A.cnt + 2 * j, v & 0xffffu);
            if (v >> 16) atomicAdd(A.cnt + 2 * j + 1, v >> 16);
        }
        grid.sync();
        const float gam = __fdiv_rn(2.0f, (float)(i + 2));
        const float om = __fsub_rn(1.0f, gam);
        const uint32_t inc = 2u * (uint32_t)(i + 1);
        // two vertices at a time: count, row and the row's first plane words in flight together
        for (uint32_t p0 = gtid; p0 < nact; p0 += 2 * nthreads) {
            uint32_t n[2], q0[2], q1[2];
            Word wv[2];
            uint4 b[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t p = p0 + h * nthreads;
                const bool ok = p < nact;
                n[h] = ok ? __ldcg(A.cnt + p + 1) : 0u;
                q0[h] = ok ? (uint32_t)__ldg(A.qptr + p) : 0u;
                q1[h] = ok ? (uint32_t)__ldg(A.qptr + p + 1) : 0u;
                wv[h] = ok ? __ldcg(word + p + 1) : Word(0);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) b[h] = q0[h] < q1[h] ? __ldcg(plane + (q0[h] >> 5)) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t p = p0 + h * nthreads;
                if (p >= nact) break;
                if (n[h]) A.cnt[p + 1] = 0;
                // receipts as a row endpoint: the bits of quads [q0, q1) in the four words of each chunk
                if (q0[h] < q1[h]) {
                    const uint32_t ca = q0[h] >> 5, cb = (q1[h] - 1) >> 5;
                    for (uint32_t q = ca; q <= cb; ++q) {
                        unsigned mask = FULL;
                        if (q == ca) mask &= FULL << (q0[h] & 31);
                        if (q == cb) mask &= lanes_le((int)((q1[h] - 1) & 31));
                        const uint4 v = q == ca ? b[h] : __ldcg(plane + q);
                        n[h] += __popc(v.x & mask) + __popc(v.y & mask) + __popc(v.z & mask) + __popc(v.w & mask);
                    }
                }
                if constexpr (std::is_same<Word, float>::value) {
                    __stcg(word + p + 1, __fadd_rn(__fmul_rn(om, wv[h]), __fmul_rn(gam, (float)n[h])));
                    // not waited for: reading R first put one more L2 access behind every vertex
                    // (a ring of 300,000: 9.6 us an iteration, 8.7 so)
                    if (n[h]) atomicAdd(reinterpret_cast<unsigned long long*>(A.R + p + 1), (unsigned long long)inc * n[h]);
                } else {
                    if (n[h]) __stcg(word + p + 1, wv[h] + inc * n[h]);
                }
            }
        }
        grid.sync();
    }
}

__global__ void eq_init_kernel(const int64_t* rowptr, const int32_t* perm, int32_t nact, uint32_t* w32, float* r32,
                               int64_t* R) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p <= nact; p += stride) {
        const int64_t d = p ? rowptr[perm[p - 1] + 1] - rowptr[perm[p - 1]] : 0;
        if (r32) {
            r32[p] = p ? __fmul_rn((float)d, 0.5f) : -1.0f;
            R[p] = d;
        } else {
            w32[p] = (uint32_t)d;
        }
    }
}

// W per entry and last choices, in canonical edge order
__global__ void eq_output_kernel(const int32_t* c, const int32_t* qs, const uint32_t* eid, int64_t nq,
                                 const uint32_t* W, uint32_t Dn, int64_t* Wout, const uint32_t* plane, uint8_t* last) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += stride) {
        const int64_t s0 = qs[q];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (c[4 * q + j] == 0) break;
            const uint32_t id = eid[s0 + j];
            const int64_t e = id >> 1;
            const bool u_src = id & 1u;
            const uint32_t w = W[4 * q + j] + 1u;            // W0 = D_0 / 2
            Wout[e] = (int64_t)(u_src ? w : Dn - w);
            if (last) {
                const uint32_t b = (plane[4 * (q >> 5) + j] >> (q & 31)) & 1u;
                last[e] = (uint8_t)(u_src ? b : 1u - b);
            }
        }
    }
}

__global__ void eq_loads_out_kernel(const int32_t* perm, int32_t nact, const uint32_t* w32, const float* r32,
                                    const int64_t* R, double Dn, int64_t* R_int, double* r_int) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += stride) {
        const int32_t x = perm[p];
        R_int[x] = r32 ? R[p + 1] : (int64_t)w32[p + 1];
        r_int[x] = r32 ? (double)r32[p + 1] : (double)w32[p + 1] / Dn;
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

// A warp takes two chunks (one 32-byte sector of each plane) and a lane one of 32
// iterations, the next 32 on their way: each word is transposed in the warp, so a lane
// holds one entry's 32 choices and adds their weights by six popcounts, and a chunk's
// entries are written whole.  No barrier and no shared memory: a block of 32 warps that
// exchanged the words through it waited for memory and for itself in turn (84.6 million
// triangles, planes of 2 GB: 1.63 ms, 1.31 so; the popcounts and shuffles bound it now,
// the planes' bytes would take 0.3 ms).
constexpr int FQ_THREADS = 256;
template <int P>
__global__ void __launch_bounds__(FQ_THREADS) fold_quads_kernel(const uint4* __restrict__ planes, int nplanes,
                                                                int64_t nchunks, int64_t i_first, uint32_t mult,
                                                                uint32_t* W0, uint32_t* W1) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c0 = 2 * (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); c0 < nchunks; c0 += 2 * nwarps) {
        const bool two = c0 + 1 < nchunks;
        uint32_t acc[P][8];
        uint4 cur[P][2], nxt[P][2];
        auto fetch = [&](int k0, uint4 (&to)[P][2]) {
            const int64_t k = k0 + lane;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const uint4* at = planes + (P * k + p) * nchunks + c0;
                to[p][0] = k < nplanes ? __ldcs(at) : make_uint4(0, 0, 0, 0);
                to[p][1] = k < nplanes && two ? __ldcs(at + 1) : make_uint4(0, 0, 0, 0);
            }
        };
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[p][j] = 0;
        fetch(0, cur);
        for (int k0 = 0; k0 < nplanes; k0 += 32) {
            fetch(k0 + 32, nxt);
            const uint32_t first = (uint32_t)(i_first + k0 + 1);
#pragma unroll
            for (int p = 0; p < P; ++p)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    acc[p][4 * h] += weighted(transpose32(cur[p][h].x, lane), first);
                    acc[p][4 * h + 1] += weighted(transpose32(cur[p][h].y, lane), first);
                    acc[p][4 * h + 2] += weighted(transpose32(cur[p][h].z, lane), first);
                    acc[p][4 * h + 3] += weighted(transpose32(cur[p][h].w, lane), first);
                    cur[p][h] = nxt[p][h];
                }
        }
        // entry 4 * lane + j of a chunk is bit `lane` of its word j
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h && !two) continue;
                uint4* at = reinterpret_cast<uint4*>((p ? W1 : W0) + (c0 + h) * 128) + lane;
                uint4 v = *at;
                v.x += mult * acc[p][4 * h];
                v.y += mult * acc[p][4 * h + 1];
                v.z += mult * acc[p][4 * h + 2];
                v.w += mult * acc[p][4 * h + 3];
                *at = v;
            }
    }
}

}  // namespace

void fold_quads(const uint32_t* planes, int nplanes, int64_t nchunks, int64_t i_first, uint32_t mult, uint32_t* W0,
                uint32_t* W1, cudaStream_t s) {
    if (nplanes <= 0 || nchunks <= 0) return;
    const uint4* p4 = reinterpret_cast<const uint4*>(planes);
    const unsigned grid = grid_for((nchunks + 1) / 2 * 32, FQ_THREADS);
    if (W1) LDS_LAUNCH(fold_quads_kernel<2>, grid, FQ_THREADS, 0, s, p4, nplanes, nchunks, i_first, mult, W0, W1);
    else LDS_LAUNCH(fold_quads_kernel<1>, grid, FQ_THREADS, 0, s, p4, nplanes, nchunks, i_first, mult, W0, W1);
}

static void ensure_quad_view(lds_graph* g) {
    if (g->fwq_c.p) return;
    cudaStream_t s = g->stream;
    const int blk = 256;
    const int32_t nact = g->nact;
    const int64_t m = g->m;
    ensure_fw_ranks(g);
    const int bits = std::max(1, bit_length_u64((uint64_t)nact));
    DevBuf<uint64_t> key(m, s);
    g->fwq_eid.alloc(m, s);
    LDS_LAUNCH(eq_slot_keys_kernel, grid_for(m, blk), blk, 0, s, g->eu.get(), g->ev.get(), m, g->fwv_pos.get(), bits,
               key.get(), g->fwq_eid.get());
    radix_sort_u64(key.get(), g->fwq_eid.get(), m, 2 * bits, s);
    DevBuf<int32_t> rowptr((size_t)nact + 1, s), nq((size_t)nact + 1, s);
    DevBuf<int64_t> qp64((size_t)nact + 1, s);
    LDS_LAUNCH(eq_rowptr_kernel, grid_for(m, blk), blk, 0, s, key.get(), m, bits, nact, rowptr.get());
    LDS_LAUNCH(eq_row_quads_kernel, grid_for(nact + 1, blk), blk, 0, s, rowptr.get(), nact, nq.get());
    g->fwq_nq = exclusive_scan_i32_to_i64(nq.get(), qp64.get(), (int64_t)nact + 1, s);
    const int64_t chunks = (g->fwq_nq + EQ_CHUNK - 1) / EQ_CHUNK;
    g->fwq_qptr.alloc((size_t)nact + 1, s);
    LDS_LAUNCH(eq_qptr_kernel, grid_for(nact + 1, blk), blk, 0, s, qp64.get(), nact, g->fwq_qptr.get());
    DevBuf<int32_t> c(4 * EQ_CHUNK * chunks, s);
    g->fwq_qs.alloc(g->fwq_nq, s);
    g->fwq_src.alloc(EQ_CHUNK * chunks, s);
    LDS_CUDA(cudaMemsetAsync(c.get(), 0, 4 * EQ_CHUNK * chunks * sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(g->fwq_src.get(), 0, EQ_CHUNK * chunks * sizeof(int32_t), s));
    LDS_LAUNCH(eq_fill_kernel, grid_for(m, blk), blk, 0, s, key.get(), m, bits, rowptr.get(), g->fwq_qptr.get(), c.get(),
               g->fwq_src.get(), g->fwq_qs.get());
    g->fwq_c = std::move(c);
}

bool run_edge_fw_quads(lds_graph* g, int N, lds_precision p, bool want_last, PassTimer& timer) {
    if (p != LDS_EXACT && p != LDS_FP32) return false;
    const int32_t n = g->n, nact = g->nact;
    const int64_t m = g->m;
    const int64_t maxdeg = std::max(g->info.max_degree, 1);
    const int64_t Dn = (int64_t)(N + 1) * (N + 2);
    const bool fp32 = p == LDS_FP32;
    // 32-bit words: every scaled load below 2^32 and per-block hot counts below 2^16
    if (m == 0 || maxdeg >= 65536) return false;
    if (!fp32 && (unsigned __int128)maxdeg * (unsigned __int128)Dn >= ((unsigned __int128)1 << 32)) return false;
    ensure_quad_view(g);
    cudaStream_t s = g->stream;
    const int blk = 256;
    const int64_t nq = g->fwq_nq, nchunks = (nq + EQ_CHUNK - 1) / EQ_CHUNK;
    LDS_CUDA(cudaMemsetAsync(g->fw_R.get(), 0, n * sizeof(int64_t), s));
    LDS_CUDA(cudaMemsetAsync(g->fw_r.get(), 0, n * sizeof(double), s));
    g->fw_W.alloc(m, s);
    if (want_last) g->fw_last.alloc(m, s);
    DevBuf<uint32_t> w32(fp32 ? 0 : (size_t)nact + 1, s), cnt((size_t)nact + 1, s);
    DevBuf<float> r32(fp32 ? (size_t)nact + 1 : 0, s);
    DevBuf<int64_t> R(fp32 ? (size_t)nact + 1 : 0, s);
    LDS_CUDA(cudaMemsetAsync(cnt.get(), 0, ((size_t)nact + 1) * sizeof(uint32_t), s));
    LDS_LAUNCH(eq_init_kernel, grid_for(nact + 1, blk), blk, 0, s, g->rowptr.get(), g->fwv_perm.get(), nact, w32.get(),
               r32.get(), R.get());
    const int K = planes_capacity(4 * nchunks, N, quad_plane_bytes(m, 1));
    DevBuf<uint4> planes(std::max<int64_t>(1, (int64_t)K * nchunks), s);
    DevBuf<uint32_t> W(128 * nchunks, s);
    LDS_CUDA(cudaMemsetAsync(W.get(), 0, 128 * nchunks * sizeof(uint32_t), s));
    const void* fn = fp32 ? (const void*)fw_quad_kernel<float> : (const void*)fw_quad_kernel<uint32_t>;
    LDS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EQ_SMEM));
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms(), (nchunks + 31) / 32));
    // Hot ids: twice the entries of a block's share, so that staging and flushing them stays
    // in proportion to the pass (both take every block of every iteration).  Staged whole,
    // graphs of 55,000 to 200,000 vertices spent more on it than on their edges: 58,000
    // vertices with 291k edges, exact, 11.3 us an iteration with 38,144 ids, 8.9 with 8,192,
    // 8.6 with 4,096, 9.0 with none (9.1 by this rule); 400,000 with 817k edges 14.8, 13.2,
    // 12.8, 14.8, and 12.5 with 16,384 (13.1 by this rule).  Past 2.9M entries or so every
    // id that fits is staged.
    const int64_t share = 4 * EQ_CHUNK * nchunks / grid;
    const int32_t nhot =
        (int32_t)std::min<int64_t>((int64_t)nact + 1, std::min<int64_t>(EQ_HOT, std::max<int64_t>(EQ_HOT_LEAST, 2 * share)));
    int stored = 0;
    for (int i = 1; i <= N; i += stored) {
        stored = std::min(K, N - i + 1);
        EqArgs A{reinterpret_cast<const int4*>(g->fwq_c.get()), g->fwq_src.get(), g->fwq_qptr.get(),
                 g->fwv_perm.get(), nchunks, nact, nhot, fp32 ? (void*)r32.get() : (void*)w32.get(), R.get(), cnt.get(),
                 planes.get(), i, stored};
        void* args[] = {(void*)&A};
        timer.start(s);
        LDS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(EQ_THREADS), args, EQ_SMEM, s));
        g_launches.fetch_add(1, std::memory_order_relaxed);
        timer.stop(s, stored);
        fold_quads(reinterpret_cast<const uint32_t*>(planes.get()), stored, nchunks, i, 2, W.get(), nullptr, s);
    }
    const uint32_t* last = N ? reinterpret_cast<const uint32_t*>(planes.get() + (int64_t)(stored - 1) * nchunks) : nullptr;
    LDS_LAUNCH(eq_output_kernel, grid_for(nq, blk), blk, 0, s, g->fwq_c.get(), g->fwq_qs.get(), g->fwq_eid.get(), nq,
               W.get(), (uint32_t)Dn, g->fw_W.get(), last, want_last && N ? g->fw_last.get() : nullptr);
    if (want_last && N == 0) LDS_CUDA(cudaMemsetAsync(g->fw_last.get(), 0, m, s));
    LDS_LAUNCH(eq_loads_out_kernel, grid_for(nact, blk), blk, 0, s, g->fwv_perm.get(), nact, w32.get(), r32.get(), R.get(),
               (double)Dn, g->fw_R.get(), g->fw_r.get());
    return true;
}

}  // namespace lds
