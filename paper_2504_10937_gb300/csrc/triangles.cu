// Triangle listing (the set T of Eq. 3 / Eq. 4) and core / tr-core numbers
// (Def. 6, Def. 11).
//
// Listing: every edge is oriented from the endpoint of lower (degree, id) rank
// to the higher one, which bounds out-degrees by O(sqrt(m)); each oriented edge
// x -> y meets out(x) and out(y) (both ascending) by a merge walk, and each
// common out-neighbour w closes the triangle {x, y, w} exactly once.  A count
// pass sizes the output, a write pass fills it, and a radix sort puts the rows in
// (a, b, c) order: one of the packed triangles up to 2^21 vertices, two stable ones
// with payload past them.
//
// Core numbers: level-synchronous peeling.  At level k every live vertex whose
// remaining degree (number of live triangles for tr-core) is <= k gets core k
// and is removed, its neighbours' degrees drop, and the step repeats until no
// vertex is removed; then k moves to the smallest remaining degree.
#include <algorithm>
#include <climits>

#include <cooperative_groups.h>
#include <cstdio>
#include <cstdlib>

#include "graph.cuh"
#include "prims.cuh"

namespace cg = cooperative_groups;

namespace lds {

namespace {

__device__ __forceinline__ bool precedes(int32_t dx, int32_t x, int32_t dy, int32_t y) {
    return dx < dy || (dx == dy && x < y);
}

// One warp per row, ballots keeping the row's order: a thread per row left the hubs' rows
// (10^4 neighbours, each with two dependent loads) to one lane; 7.1 ms for the two passes
// on an R-MAT 18 graph, 0.77 ms so.
__global__ void orient_count_kernel(const int64_t* rowptr, const int32_t* col, int32_t nact, int32_t* outdeg) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < nact; x += nwarps) {
        const int64_t b = rowptr[x], e = rowptr[x + 1];
        const int32_t dx = (int32_t)(e - b);
        int32_t c = 0;
        for (int64_t s = b + lane; s < e; s += 32) {
            const int32_t y = col[s];
            c += precedes(dx, (int32_t)x, (int32_t)(rowptr[y + 1] - rowptr[y]), y);
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) outdeg[x] = c;
    }
}

// oriented neighbours and the source vertex of every oriented slot
__global__ void orient_fill_kernel(const int64_t* rowptr, const int32_t* col, int32_t nact, const int64_t* optr,
                                   int32_t* ocol, int32_t* osrc) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < nact; x += nwarps) {
        const int64_t b = rowptr[x], e = rowptr[x + 1];
        const int32_t dx = (int32_t)(e - b);
        int64_t o = optr[x];
        for (int64_t s0 = b; s0 < e; s0 += 32) {
            const int64_t s = s0 + lane;
            int32_t y = 0;
            bool take = false;
            if (s < e) {
                y = col[s];
                take = precedes(dx, (int32_t)x, (int32_t)(rowptr[y + 1] - rowptr[y]), y);
            }
            const unsigned m = __ballot_sync(0xffffffffu, take);
            if (take) {
                const int64_t at = o + __popc(m & ((1u << lane) - 1u));
                ocol[at] = y;
                osrc[at] = (int32_t)x;
            }
            o += __popc(m);
        }
    }
}

template <bool WRITE>
__global__ void tri_intersect_kernel(const int64_t* optr, const int32_t* ocol, const int32_t* osrc, int64_t nos,
                                     int64_t* count, const int64_t* offset, int32_t* ta, int32_t* tb, int32_t* tc) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < nos; s += stride) {
        int32_t x = osrc[s], y = ocol[s];
        int64_t i = optr[x], ie = optr[x + 1];
        int64_t j = optr[y], je = optr[y + 1];
        int64_t c = 0;
        int64_t o = WRITE ? offset[s] : 0;
        while (i < ie && j < je) {
            int32_t a = ocol[i], b = ocol[j];
            if (a < b) ++i;
            else if (b < a) ++j;
            else {
                if (WRITE) {
                    int32_t p = x, q = y, r = a;
                    if (p > q) { int32_t t = p; p = q; q = t; }
                    if (q > r) { int32_t t = q; q = r; r = t; }
                    if (p > q) { int32_t t = p; p = q; q = t; }
                    ta[o] = p; tb[o] = q; tc[o] = r;
                    ++o;
                }
                ++c; ++i; ++j;
            }
        }
        if (!WRITE) count[s] = c;
    }
}

__global__ void tri_key_bc_kernel(const int32_t* tb, const int32_t* tc, int64_t ntri, int64_t nn, uint64_t* key,
                                  uint32_t* idx) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ntri; t += stride) {
        key[t] = (uint64_t)tb[t] * (uint64_t)nn + (uint64_t)tc[t];
        idx[t] = (uint32_t)t;
    }
}

__global__ void tri_key_a_kernel(const int32_t* ta, const uint32_t* idx, int64_t ntri, uint64_t* key) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ntri; t += stride) key[t] = (uint64_t)ta[idx[t]];
}

__global__ void tri_pack_kernel(const int32_t* a, const int32_t* b, const int32_t* c, int64_t k, int bits, uint64_t* key) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < k; t += stride)
        key[t] = ((((uint64_t)a[t] << bits) | (uint64_t)b[t]) << bits) | (uint64_t)c[t];
}

__global__ void tri_unpack_kernel(const uint64_t* key, int64_t k, int bits, int32_t* a, int32_t* b, int32_t* c) {
    const uint64_t mask = (1ull << bits) - 1ull;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < k; t += stride) {
        const uint64_t x = key[t];
        a[t] = (int32_t)(x >> (2 * bits));
        b[t] = (int32_t)((x >> bits) & mask);
        c[t] = (int32_t)(x & mask);
    }
}

__global__ void permute3_kernel(const int32_t* a, const int32_t* b, const int32_t* c, const uint32_t* idx, int64_t k,
                                int32_t* oa, int32_t* ob, int32_t* oc) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < k; t += stride) {
        uint32_t j = idx[t];
        oa[t] = a[j]; ob[t] = b[j]; oc[t] = c[j];
    }
}

__global__ void tri_rows_orig_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, const int32_t* to_orig,
                                     int64_t ntri, int32_t* out) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ntri; t += stride) {
        out[3 * t] = to_orig[ta[t]];
        out[3 * t + 1] = to_orig[tb[t]];
        out[3 * t + 2] = to_orig[tc[t]];
    }
}

// ---- peeling

constexpr int32_t PEEL_DEAD = -(1 << 30);   // count of a vertex that is peeled or outside the mask

__global__ void alive_init_kernel(const uint8_t* init, int32_t nact, uint8_t* alive, int64_t* core, int32_t* nalive) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int32_t c = 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nact; x += stride) {
        uint8_t a = init ? (init[x] ? 1 : 0) : 1;
        alive[x] = a;
        core[x] = -1;
        c += a;
    }
    if (c) atomicAdd(nalive, c);
}

// one warp per vertex: live neighbours
__global__ void alive_degree_kernel(const int64_t* rowptr, const int32_t* col, const uint8_t* alive, int32_t nact,
                                    int32_t* deg) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < nact; x += nwarps) {
        if (!alive[x]) {
            // stays negative when every neighbour takes one off it
            if (lane == 0) deg[x] = INT_MIN + (int32_t)(rowptr[x + 1] - rowptr[x]);
            continue;
        }
        int32_t d = 0;
        for (int64_t q = rowptr[x] + lane, e = rowptr[x + 1]; q < e; q += 32) d += alive[col[q]];
        d = __reduce_add_sync(0xffffffffu, d);
        if (lane == 0) deg[x] = d;
    }
}

// every listed pattern of a live vertex is live: its count is its list's length
__global__ void full_count_kernel(const int64_t* ptr, const uint8_t* alive, int32_t nact, int32_t* deg) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nact; x += stride)
        deg[x] = alive[x] ? (int32_t)(ptr[x + 1] - ptr[x]) : PEEL_DEAD;
}

// triangle counts of G[alive]; triangles with a dead vertex are marked dead
__global__ void tri_all_alive_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t ntri,
                                     const uint8_t* alive, int32_t* flag) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ntri; t += stride)
        flag[t] = alive[ta[t]] && alive[tb[t]] && alive[tc[t]];
}

__global__ void tri_compact_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t ntri,
                                   const int32_t* flag, const int64_t* tpos, int32_t* oa, int32_t* ob, int32_t* oc) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ntri; t += stride)
        if (flag[t]) {
            const int64_t o = tpos[t];
            oa[o] = ta[t];
            ob[o] = tb[t];
            oc[o] = tc[t];
        }
}

// the other two members of every incidence's triangle, in vertex-triangle order; a warp
// takes 128 incidences and looks their rows up between the rows of the first and the last
__global__ void incidence_pairs_kernel(const int64_t* ptr, const int32_t* idx, const int32_t* ta, const int32_t* tb,
                                       const int32_t* tc, int32_t nact, int64_t n3, int2* pairs) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // the row r in [lo, hi] with ptr[r] <= i < ptr[r + 1]
    auto row_of = [&](int64_t i, int32_t lo, int32_t hi) {
        while (lo < hi) {
            const int32_t mid = (int32_t)(((int64_t)lo + hi) >> 1);
            if (ptr[mid + 1] > i) hi = mid;
            else lo = mid + 1;
        }
        return lo;
    };
    for (int64_t i0 = 128 * (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); i0 < n3; i0 += 128 * nwarps) {
        const int64_t i1 = min(n3, i0 + 128);
        int32_t r = lane < 2 ? row_of(lane ? i1 - 1 : i0, 0, nact - 1) : 0;
        const int32_t lo = __shfl_sync(0xffffffffu, r, 0), hi = __shfl_sync(0xffffffffu, r, 1);
        for (int64_t i = i0 + lane; i < i1; i += 32) {
            const int32_t x = row_of(i, lo, hi), t = idx[i];
            const int32_t a = ta[t], b = tb[t], c = tc[t];
            pairs[i] = make_int2(a == x ? b : a, c == x ? b : c);
        }
    }
}

__global__ void alive_tri_count_kernel(const int32_t* ta, const int32_t* tb, const int32_t* tc, int64_t ntri,
                                       const uint8_t* alive, int32_t* deg, uint8_t* tdead) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ntri; t += stride) {
        int32_t a = ta[t], b = tb[t], c = tc[t];
        if (alive[a] && alive[b] && alive[c]) {
            atomicAdd(deg + a, 1);
            atomicAdd(deg + b, 1);
            atomicAdd(deg + c, 1);
        } else {
            unsigned int* word = (unsigned int*)(tdead + (t & ~3ll));
            atomicOr(word, 1u << (8 * (t & 3)));
        }
    }
}

// one atomic per group of converged threads that append together
__device__ __forceinline__ unsigned long long agg_slot(unsigned long long* ctr) {
    cg::coalesced_group grp = cg::coalesced_threads();
    unsigned long long base = 0;
    if (grp.thread_rank() == 0) base = atomicAdd(ctr, (unsigned long long)grp.size());
    return grp.shfl(base, 0) + grp.thread_rank();
}

__global__ void mark_dead_kernel(const uint8_t* alive, int32_t nact, int32_t* deg) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nact; x += stride)
        if (!alive[x]) deg[x] = PEEL_DEAD;
}

// A frontier is a queue of chunks: up to PEEL_CHUNK incidences of one peeled
// vertex, taken by one warp, so a hub is shared by the whole grid.
constexpr int PEEL_CHUNK = 64;
struct __align__(16) PeelChunk {
    int64_t start;
    int32_t len, x;
};

// The lanes with `want` append the chunks of their vertex y (whole warp calls).
__device__ __forceinline__ void peel_push(bool want, int32_t y, const int64_t* ptr, PeelChunk* Q,
                                          unsigned long long* cnt, int lane) {
    unsigned mask = __ballot_sync(0xffffffffu, want);
    if (!mask) return;
    int64_t b = 0;
    int32_t len = 0;
    if (want) {
        b = ptr[y];
        len = (int32_t)(ptr[y + 1] - b);
    }
    const int32_t nch = (len + PEEL_CHUNK - 1) / PEEL_CHUNK;
    int32_t incl = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    unsigned long long base = 0;
    if (lane == 31 && incl) base = atomicAdd(cnt, (unsigned long long)incl);
    base = __shfl_sync(0xffffffffu, base, 31);
    for (; mask; mask &= mask - 1) {
        const int l = __ffs(mask) - 1;
        const int32_t vy = __shfl_sync(0xffffffffu, y, l), vlen = __shfl_sync(0xffffffffu, len, l);
        const int64_t vb = __shfl_sync(0xffffffffu, b, l);
        const int32_t vn = __shfl_sync(0xffffffffu, nch, l), ve = __shfl_sync(0xffffffffu, incl, l);
        for (int32_t c = lane; c < vn; c += 32) {
            PeelChunk e{vb + (int64_t)c * PEEL_CHUNK, min(PEEL_CHUNK, vlen - c * PEEL_CHUNK), vy};
            Q[base + (unsigned long long)(ve - vn + c)] = e;
        }
    }
}

constexpr int PEEL_SOLO = 8192;      // live vertices the one-block kernel finishes with, in shared memory
constexpr int PEEL_SOLO_T = 1024;    // its threads
constexpr int SOLO_CHUNK = 128;      // neighbours a warp takes at a time (4 per lane)
constexpr size_t PEEL_SOLO_SMEM = (size_t)PEEL_SOLO * (4 + 4 + 2 * 2 + 2 * 4) + 16;

// ctrl words of a peel
constexpr int PC_Q = 0;        // [3] chunk counts of the queues
constexpr int PC_ERR = 3;      // step bound hit
constexpr int PC_LIST = 4;     // [3] live-list counts
constexpr int PC_MIN = 7;      // [3] lower bound of the live counts
constexpr int PC_STEPS = 10;   // steps and last level (reported)
constexpr int PC_LEVEL = 11;
constexpr int PC_SOLO = 12;    // hand-over: flag, list, live count, level, steps
constexpr int PC_WORDS = 17;

// A peel in one block: the dense tail of an edge peel once at most PEEL_SOLO
// vertices are live (SOLO_TAIL, handed over by the grid-wide kernel), or a whole
// small graph (SOLO_EDGES, SOLO_TRIS).  For the tail the live subgraph was
// compacted to 16-bit local ids (cadj, rows at coff, padded to whole 4-entry
// groups with 0xffff), so a round reads live neighbours only; a whole graph's rows
// are used as they are, vertex x being slot x.  Counts, frontiers and the dead
// bits of triangles sit in shared memory.  A frontier entry is a vertex and the
// number of 128-incidence chunks before it, both handed out by one 64-bit shared
// atomic; warps find their chunk's vertex by a 32-way search.  One block barrier
// per round.  Same levels and rules as the grid-wide kernel.
//
// Bounded by the chain of one round (row entry from L2, shared count, frontier) in
// one SM: 1.0-1.5 us a step where grid barriers make it 4 or more.  The one-block
// tail over uncompacted rows took 8.7 us a step on the 1M-vertex power-law graph.
enum SoloKind { SOLO_TAIL, SOLO_EDGES, SOLO_TRIS };
constexpr int64_t PEEL_SOLO_TRIS = 1 << 19;     // most triangles of SOLO_TRIS (their dead bits: 64 KB)
constexpr size_t PEEL_SOLO_TRIS_SMEM = PEEL_SOLO_SMEM + PEEL_SOLO_TRIS / 8;

template <SoloKind KIND>
__global__ void __launch_bounds__(PEEL_SOLO_T, 1) peel_solo_kernel(
    const int32_t* A0, const int32_t* A1, const int32_t* deg, const int32_t* coff, const uint16_t* cadj, int32_t n,
    const int64_t* ptr, const int32_t* __restrict__ adj, const int32_t* __restrict__ ta,
    const int32_t* __restrict__ tb, const int32_t* __restrict__ tc, const uint8_t* __restrict__ tdead, int64_t nt,
    int64_t* core, unsigned long long* ctrl, int64_t max_steps) {
    extern __shared__ __align__(16) unsigned char psm[];
    __shared__ unsigned long long q[3];
    __shared__ int32_t smin[3];
    if (KIND == SOLO_TAIL && ctrl[PC_SOLO] == 0) return;   // the grid-wide kernel finished the peel
    const int32_t* list = KIND == SOLO_TAIL ? (ctrl[PC_SOLO + 1] ? A1 : A0) : nullptr;
    const int32_t nl = KIND == SOLO_TAIL ? (int32_t)ctrl[PC_SOLO + 2] : n;
    int32_t k = KIND == SOLO_TAIL ? (int32_t)ctrl[PC_SOLO + 3] : 0;
    int64_t steps = KIND == SOLO_TAIL ? (int64_t)ctrl[PC_SOLO + 4] : 0;
    int32_t* sd = reinterpret_cast<int32_t*>(psm);                // live count (negative once peeled)
    int32_t* off = sd + PEEL_SOLO;                                // [nl + 1] row starts
    int32_t* fo = off + PEEL_SOLO + 4;                            // [2][PEEL_SOLO] chunks before a frontier entry
    uint16_t* fv = reinterpret_cast<uint16_t*>(fo + 2 * PEEL_SOLO);   // [2][PEEL_SOLO] its vertex
    uint32_t* dead = reinterpret_cast<uint32_t*>(fv + 2 * PEEL_SOLO); // SOLO_TRIS: one bit per triangle
    const int tid = threadIdx.x, bd = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = bd >> 5;
    for (int i = tid; i < nl; i += bd) {
        const int32_t d = deg[KIND == SOLO_TAIL ? list[i] : i];
        sd[i] = KIND == SOLO_TAIL && d < 0 ? PEEL_DEAD : d;
    }
    for (int i = tid; i <= nl; i += bd) off[i] = KIND == SOLO_TAIL ? coff[i] : (int32_t)ptr[i];
    if (KIND == SOLO_TRIS)
        // triangles with a vertex outside the mask are dead from the start
        for (int64_t t = tid; t < ((nt + 31) & ~31ll); t += bd) {
            const unsigned m = __ballot_sync(0xffffffffu, t < nt && tdead[t]);
            if (lane == 0) dead[t >> 5] = m;
        }
    if (tid < 3) {
        q[tid] = 0;
        smin[tid] = INT_MAX;
    }
    __syncthreads();
    int ph = 0, lv = 0;                          // queue phase and level, modulo 3 for the counters
    // vertex i is peeled at level k: core number, and its row joins the next frontier
    auto peel = [&](int i) {
        core[KIND == SOLO_TAIL ? list[i] : i] = k;
        const unsigned nch = (unsigned)(off[i + 1] - off[i] + SOLO_CHUNK - 1) / SOLO_CHUNK;
        if (nch == 0) return;
        const unsigned long long o = atomicAdd(&q[(ph + 1) % 3], ((unsigned long long)nch << 32) | 1ull);
        const int at = ((ph + 1) & 1) * PEEL_SOLO + (int)(unsigned)o;
        fv[at] = (uint16_t)i;
        fo[at] = (int32_t)(o >> 32);
    };
    int32_t mn = INT_MAX;
    // a vertex whose count falls from k + 1 to k is peeled at k
    auto drop = [&](int y) {
        const int32_t old = atomicSub(sd + y, 1);
        if (old == k + 1) {
            sd[y] = PEEL_DEAD;
            peel(y);
        } else if (old > k) {
            mn = min(mn, old - 1);
        }
    };
    for (;;) {
        if (++steps > max_steps) {
            if (tid == 0) ctrl[PC_ERR] = 1;
            return;
        }
        if (tid == 0) {
            q[(ph + 2) % 3] = 0;
            smin[(lv + 1) % 3] = INT_MAX;
        }
        // level scan
        bool kept = false;
        mn = INT_MAX;
        for (int i = tid; i < nl; i += bd) {
            const int32_t d = sd[i];
            if (d < 0) continue;
            if (d <= k) {
                sd[i] = PEEL_DEAD;
                peel(i);
            } else {
                kept = true;
                mn = min(mn, d);
            }
        }
        mn = __reduce_min_sync(0xffffffffu, mn);
        if (lane == 0 && mn != INT_MAX) atomicMin(&smin[lv % 3], mn);
        const bool more = __syncthreads_or(kept) != 0;
        ++ph;
        unsigned long long cur = q[ph % 3];
        while (cur) {
            if (++steps > max_steps) {
                if (tid == 0) ctrl[PC_ERR] = 1;
                return;
            }
            if (tid == 0) q[(ph + 2) % 3] = 0;
            const int nf = (int)(unsigned)cur, nc = (int)(cur >> 32);
            const int32_t* cfo = fo + (ph & 1) * PEEL_SOLO;
            const uint16_t* cfv = fv + (ph & 1) * PEEL_SOLO;
            mn = INT_MAX;
            for (int c = wid; c < nc; c += nw) {
                int lo = 0, cnt = nf;                  // last entry with fo <= c
                while (cnt > 1) {
                    const int st = (cnt + 31) >> 5, at = lane * st;
                    const unsigned m = __ballot_sync(0xffffffffu, at < cnt && cfo[lo + at] <= c);
                    const int j = 31 - __clz(m);
                    lo += j * st;
                    cnt = min(st, cnt - j * st);
                }
                const int i = cfv[lo];
                const int32_t e = off[i + 1], b = off[i] + (c - cfo[lo]) * SOLO_CHUNK;
                if (KIND == SOLO_TAIL) {
                    if (b + lane * 4 < e) {
                        const ushort4 v = *reinterpret_cast<const ushort4*>(cadj + b + lane * 4);
                        const int y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (y[j] != 0xffff) drop(y[j]);
                    }
                } else {
                    int32_t y[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[j] = b + 32 * j + lane < e ? adj[b + 32 * j + lane] : -1;
                    if (KIND == SOLO_EDGES) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (y[j] >= 0) drop(y[j]);
                    } else {
                        int32_t v[4][3];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t bit = 1u << (y[j] & 31);
                            // else it died with another vertex
                            if (y[j] >= 0 && (atomicOr(dead + (y[j] >> 5), bit) & bit)) y[j] = -1;
                            if (y[j] >= 0) {
                                v[j][0] = ta[y[j]];
                                v[j][1] = tb[y[j]];
                                v[j][2] = tc[y[j]];
                            }
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (y[j] >= 0) {
#pragma unroll
                                for (int r = 0; r < 3; ++r)
                                    if (v[j][r] != i) drop(v[j][r]);
                            }
                    }
                }
            }
            mn = __reduce_min_sync(0xffffffffu, mn);
            if (lane == 0 && mn != INT_MAX) atomicMin(&smin[lv % 3], mn);
            __syncthreads();
            ++ph;
            cur = q[ph % 3];
        }
        if (!more) {
            if (tid == 0) {
                ctrl[PC_STEPS] = (unsigned long long)steps;
                ctrl[PC_LEVEL] = (unsigned long long)k;
            }
            return;
        }
        k = max(k + 1, smin[lv % 3]);
        ++lv;
    }
}

// Whole peeling loop in one cooperative launch (peeling by levels).  A level k
// starts with a scan of the live-vertex list: vertices with count <= k are peeled
// (core k) and their chunks queued, the others go to the other list.  Rounds then
// take the queued chunks, one warp each; removing a peeled vertex lowers the count
// of each neighbour (of each other vertex of each live triangle), and a vertex
// whose count falls to k is peeled at level k too and queued for the next round.
// The scan and every drop also keep a lower bound of the live counts, the next
// level when it is above k + 1.  Peeled vertices hold PEEL_DEAD: their counts stay
// negative whatever is taken off them.
//
// A level of the dense part has little work, so what bounds it is the chain of
// dependent L2 accesses of a round and its grid barrier.  Every counter is kept
// three times and used in turn, so one barrier ends a round or a scan, and a queue
// entry carries its chunk's start and length, so a round is entry -> neighbours ->
// counts.  (Four barriers a round and a separate pass that queued the chunks of
// heavy vertices took 16.7 us a step on the R-MAT scale-18 triangles.)
//
// An edge peel hands over to peel_solo_kernel once `solo` or fewer vertices are
// live, after compacting the live subgraph to local ids.
//
// Triangles: PEEL_TRIS marks a dead triangle in tdead and looks its members up.
// PEEL_PAIRS has each incidence's other two members beside it and keeps the round in
// which a vertex is taken (stamp): a triangle died earlier if another member was taken in
// an earlier round, and of members taken together the smallest id counts it.  That is two
// dependent accesses a round less, and the pairs are read in order.  R-MAT 18 (84.6 million
// triangles, 6,700 steps): 58.1 ms with the counts' atomics one after the other, 51.2 with
// them together, 45.5 with pairs, their making included.
enum PeelKind { PEEL_EDGES, PEEL_TRIS, PEEL_PAIRS };
template <PeelKind KIND>
__global__ void __launch_bounds__(1024, 1) peel_coop_kernel(const int64_t* __restrict__ ptr,
                                                            const int32_t* __restrict__ adj,
                                                            const int32_t* __restrict__ ta,
                                                            const int32_t* __restrict__ tb,
                                                            const int32_t* __restrict__ tc, uint8_t* tdead,
                                                            int32_t* deg, int64_t* core, PeelChunk* Q0, PeelChunk* Q1,
                                                            int32_t* A0, int32_t* A1, unsigned long long* ctrl,
                                                            int64_t max_steps, int32_t solo, int32_t* slot,
                                                            int32_t* coff, uint16_t* cadj,
                                                            const int2* __restrict__ pairs, int32_t* stamp) {
    constexpr bool TRI = KIND != PEEL_EDGES;
    cg::grid_group grid = cg::this_grid();
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const int64_t warp = tid >> 5, nwarps = nthreads >> 5;
    int ph = 0, lv = 0;
    int32_t k = 0;
    int64_t steps = 0, na = (int64_t)__ldcg(ctrl + PC_LIST);
    for (;;) {
        const int32_t* cl = lv & 1 ? A1 : A0;
        int32_t* nlst = lv & 1 ? A0 : A1;
        if constexpr (!TRI) if (na <= solo) {
            __shared__ int32_t wsum[32];
            for (int64_t i = tid; i < na; i += nthreads) {
                const int32_t x = __ldcg(cl + i);
                if (__ldcg(deg + x) >= 0) slot[x] = (int32_t)i;
            }
            if (blockIdx.x == 0) {
                // row starts: a live vertex has deg live neighbours, padded to groups of 4
                int32_t run = 0;
                for (int64_t base = 0; base < na; base += blockDim.x) {
                    const int64_t i = base + threadIdx.x;
                    int32_t l = 0;
                    if (i < na) l = (max(__ldcg(deg + __ldcg(cl + i)), 0) + 3) & ~3;
                    int32_t incl = l;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int32_t v = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += v;
                    }
                    if (lane == 31) wsum[threadIdx.x >> 5] = incl;
                    __syncthreads();
                    int32_t before = 0, tot = 0;
                    for (int j = 0; j < (int)(blockDim.x >> 5); ++j) {
                        if (j < (int)(threadIdx.x >> 5)) before += wsum[j];
                        tot += wsum[j];
                    }
                    if (i < na) coff[i] = run + before + incl - l;
                    run += tot;
                    __syncthreads();
                }
                if (threadIdx.x == 0) coff[na] = run;
            }
            grid.sync();
            for (int64_t i = warp; i < na; i += nwarps) {
                const int32_t x = __ldcg(cl + i);
                if (__ldcg(deg + x) < 0) continue;
                int32_t o = __ldcg(coff + i);
                const int32_t end = __ldcg(coff + i + 1);
                const int64_t e = ptr[x + 1];
                for (int64_t q0 = ptr[x]; q0 < e; q0 += 128) {
                    int32_t y[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int64_t q = q0 + 32 * j + lane;
                        y[j] = q < e ? adj[q] : -1;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[j] = y[j] >= 0 ? __ldcg(slot + y[j]) : -1;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const unsigned bal = __ballot_sync(0xffffffffu, y[j] >= 0);
                        if (y[j] >= 0) cadj[o + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)y[j];
                        o += __popc(bal);
                    }
                }
                if (o + lane < end) cadj[o + lane] = 0xffff;
            }
            if (tid == 0) {
                ctrl[PC_SOLO + 1] = lv & 1;
                ctrl[PC_SOLO + 2] = (unsigned long long)na;
                ctrl[PC_SOLO + 3] = (unsigned long long)k;
                ctrl[PC_SOLO + 4] = (unsigned long long)steps;
                ctrl[PC_SOLO] = 1;
            }
            return;
        }
        if (++steps > max_steps) {
            if (tid == 0) ctrl[PC_ERR] = 1;
            return;
        }
        if (tid == 0) {
            ctrl[PC_Q + (ph + 2) % 3] = 0;
            ctrl[PC_LIST + (lv + 2) % 3] = 0;
            ctrl[PC_MIN + (lv + 1) % 3] = ~0ull;
        }
        unsigned long long* mnp = ctrl + PC_MIN + lv % 3;
        // level scan, warp by warp: one atomic per warp for the list and for the minimum
        for (int64_t base = tid - lane; base < na; base += nthreads) {
            const int64_t i = base + lane;
            int32_t x = 0, d = -1;
            if (i < na) {
                x = __ldcg(cl + i);
                d = __ldcg(deg + x);
            }
            const bool keep = d > k, peel = d >= 0 && d <= k;
            const unsigned km = __ballot_sync(0xffffffffu, keep);
            const unsigned dmin = __reduce_min_sync(0xffffffffu, keep ? (unsigned)d : 0xffffffffu);
            unsigned long long kb = 0;
            if (lane == 0 && km) {
                kb = atomicAdd(ctrl + PC_LIST + (lv + 1) % 3, (unsigned long long)__popc(km));
                if (dmin < __ldcg(mnp)) atomicMin(mnp, (unsigned long long)dmin);
            }
            kb = __shfl_sync(0xffffffffu, kb, 0);
            if (keep) nlst[kb + __popc(km & ((1u << lane) - 1u))] = x;
            if (peel) {
                deg[x] = PEEL_DEAD;
                core[x] = k;
                if (KIND == PEEL_PAIRS) stamp[x] = ph + 1;
            }
            peel_push(peel, x, ptr, (ph + 1) & 1 ? Q1 : Q0, ctrl + PC_Q + (ph + 1) % 3, lane);
        }
        grid.sync();
        ++ph;
        int64_t nq = (int64_t)__ldcg(ctrl + PC_Q + ph % 3);
        na = (int64_t)__ldcg(ctrl + PC_LIST + (lv + 1) % 3);
        // frontier rounds at level k
        while (nq > 0) {
            if (++steps > max_steps) {
                if (tid == 0) ctrl[PC_ERR] = 1;
                return;
            }
            if (tid == 0) ctrl[PC_Q + (ph + 2) % 3] = 0;
            const PeelChunk* cq = ph & 1 ? Q1 : Q0;
            PeelChunk* nx = (ph + 1) & 1 ? Q1 : Q0;
            unsigned long long* ncnt = ctrl + PC_Q + (ph + 1) % 3;
            unsigned mn = 0xffffffffu;
            for (int64_t c = warp; c < nq; c += nwarps) {
                const int4 raw = __ldcg(reinterpret_cast<const int4*>(cq + c));
                const int64_t q0 = (int64_t)(((unsigned long long)(unsigned)raw.y << 32) | (unsigned)raw.x);
                const int32_t len = raw.z, x = raw.w;
                int32_t it[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) it[j] = KIND != PEEL_PAIRS && lane + 32 * j < len ? adj[q0 + lane + 32 * j] : -1;
                if (!TRI) {
                    bool hit[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        hit[j] = false;
                        if (it[j] >= 0) {
                            const int32_t old = atomicSub(deg + it[j], 1);
                            hit[j] = old == k + 1;
                            if (hit[j]) {
                                deg[it[j]] = PEEL_DEAD;
                                core[it[j]] = k;
                            } else if (old > k) {
                                mn = min(mn, (unsigned)(old - 1));
                            }
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j) peel_push(hit[j], it[j], ptr, nx, ncnt, lane);
                } else {
                    int32_t y[4];
                    if (KIND == PEEL_PAIRS) {
                        int2 p[2];
                        int32_t st[2][2];
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            p[j] = lane + 32 * j < len ? pairs[q0 + lane + 32 * j] : make_int2(-1, -1);
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            st[j][0] = p[j].x >= 0 ? __ldcg(stamp + p[j].x) : -1;
                            st[j][1] = p[j].x >= 0 ? __ldcg(stamp + p[j].y) : -1;
                        }
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            // a stamp of ph + 1 may be of this very round: alive for it
                            const bool mine = st[j][0] >= ph && st[j][1] >= ph && !(st[j][0] == ph && p[j].x < x) &&
                                              !(st[j][1] == ph && p[j].y < x);
                            y[2 * j] = mine && st[j][0] > ph ? p[j].x : -1;
                            y[2 * j + 1] = mine && st[j][1] > ph ? p[j].y : -1;
                        }
                    } else {
                        bool first[2];
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            first[j] = false;
                            if (it[j] >= 0) {
                                unsigned int* word = (unsigned int*)(tdead + (it[j] & ~3));
                                const unsigned int bit = 1u << (8 * (it[j] & 3));
                                first[j] = !(atomicOr(word, bit) & bit);      // else it died with another vertex
                            }
                        }
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            y[2 * j] = y[2 * j + 1] = -1;
                            if (first[j]) {
                                const int32_t a = ta[it[j]], b = tb[it[j]], cc = tc[it[j]];
                                y[2 * j] = a == x ? b : a;
                                y[2 * j + 1] = cc == x ? b : cc;
                            }
                        }
                    }
                    // consecutive triangles of x share a member: one atomic per distinct vertex,
                    // all four under way before the first is needed
                    int32_t n[4], old[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const unsigned peers = __match_any_sync(0xffffffffu, y[j]);
                        n[j] = y[j] >= 0 && (peers & ((1u << lane) - 1u)) == 0 ? __popc(peers) : 0;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) old[j] = n[j] ? atomicSub(deg + y[j], n[j]) : PEEL_DEAD;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool hit = old[j] > k && old[j] - n[j] <= k;
                        if (hit) {
                            deg[y[j]] = PEEL_DEAD;
                            core[y[j]] = k;
                            if (KIND == PEEL_PAIRS) stamp[y[j]] = ph + 1;
                        } else if (old[j] > k) {
                            mn = min(mn, (unsigned)(old[j] - n[j]));
                        }
                        peel_push(hit, y[j], ptr, nx, ncnt, lane);
                    }
                }
            }
            if (warp < nq) {
                mn = __reduce_min_sync(0xffffffffu, mn);
                if (lane == 0 && mn < __ldcg(mnp)) atomicMin(mnp, (unsigned long long)mn);
            }
            grid.sync();
            ++ph;
            nq = (int64_t)__ldcg(ctrl + PC_Q + ph % 3);
        }
        const unsigned long long mb = __ldcg(mnp);
        if (na == 0) {
            if (tid == 0) {
                ctrl[PC_STEPS] = (unsigned long long)steps;
                ctrl[PC_LEVEL] = (unsigned long long)k;
            }
            return;
        }
        k = (int32_t)max((unsigned long long)k + 1, mb);
        ++lv;
    }
}

// list of the live vertices
__global__ void alive_list_kernel(const uint8_t* alive, int32_t nact, int32_t* list, unsigned long long* cnt) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nact; x += stride)
        if (alive[x]) list[agg_slot(cnt)] = (int32_t)x;
}

}  // namespace

void ensure_triangles(lds_graph* g) {
    if (g->ntri >= 0) return;
    cudaStream_t s = g->stream;
    const int32_t nact = g->nact;
    const int blk = 256;
    if (g->m == 0 || nact == 0) {
        g->ntri = 0;
        return;
    }
    DevBuf<int32_t> outdeg(nact + 1, s);
    LDS_CUDA(cudaMemsetAsync(outdeg.get(), 0, (nact + 1) * sizeof(int32_t), s));
    LDS_LAUNCH(orient_count_kernel, grid_for((int64_t)nact * 32, blk), blk, 0, s, g->rowptr.get(), g->col.get(), nact, outdeg.get());
    LDS_CHECK_LAUNCH();
    DevBuf<int64_t> optr(nact + 1, s);
    int64_t nos = exclusive_scan_i32_to_i64(outdeg.get(), optr.get(), nact + 1, s);
    LDS_REQUIRE(nos == g->m, LDS_ECUDA, "triangle listing: orientation lost edges (internal error)");
    DevBuf<int32_t> ocol(nos, s), osrc(nos, s);
    LDS_LAUNCH(orient_fill_kernel, grid_for((int64_t)nact * 32, blk), blk, 0, s, g->rowptr.get(), g->col.get(), nact,
               optr.get(), ocol.get(), osrc.get());
    LDS_CHECK_LAUNCH();
    DevBuf<int64_t> cnt(nos, s), off(nos, s);
    LDS_LAUNCH(tri_intersect_kernel<false>, grid_for(nos, blk), blk, 0, s, optr.get(), ocol.get(), osrc.get(), nos, cnt.get(),
                                                                   nullptr, nullptr, nullptr, nullptr);
    LDS_CHECK_LAUNCH();
    int64_t ntri = exclusive_scan_i64(cnt.get(), off.get(), nos, s);
    LDS_REQUIRE(ntri < ((int64_t)1 << 32), LDS_EOVERFLOW, "triangle listing: |T| = %lld exceeds 2^32",
                (long long)ntri);
    DevBuf<int32_t> a(ntri, s), b(ntri, s), c(ntri, s);
    if (ntri) {
        LDS_LAUNCH(tri_intersect_kernel<true>, grid_for(nos, blk), blk, 0, s, optr.get(), ocol.get(), osrc.get(), nos, nullptr,
                                                                      off.get(), a.get(), b.get(), c.get());
        LDS_CHECK_LAUNCH();
    }
    cnt.release(); off.release(); ocol.release(); osrc.release(); optr.release(); outdeg.release();
    g->ta.alloc(ntri, s);
    g->tb.alloc(ntri, s);
    g->tc.alloc(ntri, s);
    if (ntri) {
        DevBuf<uint64_t> key(ntri, s);
        const uint64_t nn = (uint64_t)nact;
        const int bits = bit_length_u64(nn - 1);
        if (3 * bits <= 64) {
            // the whole triangle is the key: no payload, one sort, no gathers
            LDS_LAUNCH(tri_pack_kernel, grid_for(ntri, blk), blk, 0, s, a.get(), b.get(), c.get(), ntri, bits, key.get());
            radix_sort_u64(key.get(), nullptr, ntri, 3 * bits, s);
            LDS_LAUNCH(tri_unpack_kernel, grid_for(ntri, blk), blk, 0, s, key.get(), ntri, bits, g->ta.get(), g->tb.get(),
                       g->tc.get());
        } else {
            DevBuf<uint32_t> idx(ntri, s);
            LDS_LAUNCH(tri_key_bc_kernel, grid_for(ntri, blk), blk, 0, s, b.get(), c.get(), ntri, (int64_t)nn, key.get(),
                       idx.get());
            radix_sort_u64(key.get(), idx.get(), ntri, bit_length_u64(nn * nn), s);
            LDS_LAUNCH(tri_key_a_kernel, grid_for(ntri, blk), blk, 0, s, a.get(), idx.get(), ntri, key.get());
            radix_sort_u64(key.get(), idx.get(), ntri, bit_length_u64(nn), s);
            LDS_LAUNCH(permute3_kernel, grid_for(ntri, blk), blk, 0, s, a.get(), b.get(), c.get(), idx.get(), ntri,
                       g->ta.get(), g->tb.get(), g->tc.get());
        }
    }
    LDS_CUDA(cudaStreamSynchronize(s));
    g->ntri = ntri;
    g->info.triangles = ntri;
}

// Core (tr-core) numbers of G[alive] in internal ids: core_int[nact]; vertices
// outside `init_alive` (device mask, NULL = every vertex) get -1.
static void core_numbers_internal(lds_graph* g, bool tri, int64_t* core_int, const uint8_t* init_alive) {
    cudaStream_t s = g->stream;
    const int32_t nact = g->nact;
    const int blk = 256;
    if (nact == 0) return;
    DevBuf<uint8_t> alive(nact, s);
    DevBuf<int32_t> nalive(1, s);
    LDS_CUDA(cudaMemsetAsync(nalive.get(), 0, sizeof(int32_t), s));
    LDS_LAUNCH(alive_init_kernel, grid_for(nact, blk), blk, 0, s, init_alive, nact, alive.get(), core_int, nalive.get());
    if (tri) ensure_triangles(g);
    int32_t remaining = nact;
    if (init_alive) {
        LDS_CUDA(cudaMemcpyAsync(&remaining, nalive.get(), sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        LDS_CUDA(cudaStreamSynchronize(s));
    }
    if (remaining == 0) return;
    // every vertex alive: the whole graph's core numbers, peeled once per handle
    DevBuf<int64_t>& whole = g->core_all[tri ? 1 : 0];
    const bool all_alive = remaining == nact;
    if (all_alive && whole.p) {
        LDS_CUDA(cudaMemcpyAsync(core_int, whole.get(), (size_t)nact * sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
        return;
    }
    DevBuf<int32_t> deg(nact, s);
    DevBuf<uint8_t> tdead;
    // the triangle list the peeling walks: all of T, or, when few vertices are alive,
    // only the triangles whose three members are alive (the others never count)
    DevBuf<int32_t> cta, ctb, ctc, cvi;
    DevBuf<int64_t> cvp;
    const int64_t* ptr = g->rowptr.get();
    const int32_t *adj = g->col.get(), *tta = nullptr, *ttb = nullptr, *ttc = nullptr;
    int64_t tnt = 0;
    if (!tri) {
        if (all_alive)
            LDS_LAUNCH(full_count_kernel, grid_for(nact, blk), blk, 0, s, ptr, alive.get(), nact, deg.get());
        else
            LDS_LAUNCH(alive_degree_kernel, grid_for((int64_t)nact * 32, blk), blk, 0, s, ptr, adj, alive.get(), nact,
                       deg.get());
    } else {
        if ((int64_t)remaining * 4 < (int64_t)nact && g->ntri) {
            const int64_t ntri = g->ntri;
            DevBuf<int32_t> flag(ntri + 1, s);
            DevBuf<int64_t> tpos(ntri + 1, s);
            LDS_CUDA(cudaMemsetAsync(flag.get() + ntri, 0, sizeof(int32_t), s));
            LDS_LAUNCH(tri_all_alive_kernel, grid_for(ntri, blk), blk, 0, s, g->ta.get(), g->tb.get(), g->tc.get(), ntri,
                       alive.get(), flag.get());
            tnt = exclusive_scan_i32_to_i64(flag.get(), tpos.get(), ntri + 1, s);
            cta.alloc(std::max<int64_t>(tnt, 1), s);
            ctb.alloc(std::max<int64_t>(tnt, 1), s);
            ctc.alloc(std::max<int64_t>(tnt, 1), s);
            if (tnt)
                LDS_LAUNCH(tri_compact_kernel, grid_for(ntri, blk), blk, 0, s, g->ta.get(), g->tb.get(), g->tc.get(), ntri,
                           flag.get(), tpos.get(), cta.get(), ctb.get(), ctc.get());
            build_vertex_triangles(cta.get(), ctb.get(), ctc.get(), tnt, nact, cvp, cvi, s);
            ptr = cvp.get();
            adj = cvi.get();
            tta = cta.get();
            ttb = ctb.get();
            ttc = ctc.get();
        } else {
            ensure_vertex_triangles(g);
            tnt = g->ntri;
            ptr = g->vt_ptr.get();
            adj = g->vt_idx.get();
            tta = g->ta.get();
            ttb = g->tb.get();
            ttc = g->tc.get();
        }
        tdead.alloc(((tnt + 3) & ~3ll) + 4, s);
        LDS_CUDA(cudaMemsetAsync(tdead.get(), 0, ((tnt + 3) & ~3ll) + 4, s));
        if (all_alive || tta == cta.get()) {
            // every triangle listed is live
            LDS_LAUNCH(full_count_kernel, grid_for(nact, blk), blk, 0, s, ptr, alive.get(), nact, deg.get());
        } else {
            LDS_CUDA(cudaMemsetAsync(deg.get(), 0, nact * sizeof(int32_t), s));
            if (tnt)
                LDS_LAUNCH(alive_tri_count_kernel, grid_for(tnt, blk), blk, 0, s, tta, ttb, ttc, tnt, alive.get(),
                           deg.get(), tdead.get());
            LDS_LAUNCH(mark_dead_kernel, grid_for(nact, blk), blk, 0, s, alive.get(), nact, deg.get());
        }
    }
    DevBuf<unsigned long long> ctrl(PC_WORDS, s);
    unsigned long long hctrl[PC_WORDS] = {};
    for (int j = 0; j < 3; ++j) hctrl[PC_MIN + j] = ~0ull;
    LDS_CUDA(cudaMemcpyAsync(ctrl.get(), hctrl, sizeof(hctrl), cudaMemcpyHostToDevice, s));
    const int64_t max_steps = 4 * (int64_t)nact + 64;
    // a small graph peels in one block from the start; a triangle peel only while its
    // dead bits fit and its incidences do not need more than one SM
    const bool small = nact <= PEEL_SOLO && (!tri || tnt <= PEEL_SOLO_TRIS);
    const int64_t incid = tri ? 3 * tnt : 2 * g->m;
    // a vertex is queued once: at most one chunk per vertex plus one per PEEL_CHUNK incidences
    const int64_t qcap = small ? 0 : (int64_t)nact + incid / PEEL_CHUNK + 1;
    const bool tail = !small && !tri;
    DevBuf<PeelChunk> Q0(qcap, s), Q1(qcap, s);
    DevBuf<int32_t> A0(small ? 0 : nact, s), A1(small ? 0 : nact, s);
    // the one-block tail only for edges: a triangle tail's incidences (hub triangles)
    // keep the whole grid busy
    const int32_t solo = tri ? -1 : PEEL_SOLO;
    DevBuf<int32_t> slotb(tail ? nact : 0, s), coff(tail ? PEEL_SOLO + 1 : 0, s);
    // live neighbours of at most PEEL_SOLO vertices, rows padded to groups of 4
    const int64_t ccap = std::min<int64_t>(2 * g->m, (int64_t)PEEL_SOLO * (PEEL_SOLO - 1)) + 4 * PEEL_SOLO;
    DevBuf<uint16_t> cadj(tail ? ccap : 0, s);
    uint8_t* td = tri ? tdead.get() : nullptr;
    int32_t* dg = deg.get();
    PeelChunk *q0 = Q0.get(), *q1 = Q1.get();
    int32_t *a0 = A0.get(), *a1 = A1.get();
    unsigned long long* ct = ctrl.get();
    int32_t *slp = slotb.get(), *cop = coff.get();
    uint16_t* cap = cadj.get();
    const char* vb = getenv("LDS_VERBOSE");
    const bool verbose = vb && vb[0] == '1';
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (verbose) {
        LDS_CUDA(cudaEventCreate(&e0));
        LDS_CUDA(cudaEventCreate(&e1));
        LDS_CUDA(cudaEventRecord(e0, s));
    }
    int grid = 1;
    if (small && tri) {
        LDS_CUDA(cudaFuncSetAttribute(peel_solo_kernel<SOLO_TRIS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)PEEL_SOLO_TRIS_SMEM));
        LDS_LAUNCH(peel_solo_kernel<SOLO_TRIS>, 1, PEEL_SOLO_T, PEEL_SOLO_TRIS_SMEM, s, a0, a1, dg, cop, cap, nact, ptr,
                   adj, tta, ttb, ttc, td, tnt, core_int, ct, max_steps);
    } else if (small) {
        LDS_CUDA(cudaFuncSetAttribute(peel_solo_kernel<SOLO_EDGES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)PEEL_SOLO_SMEM));
        LDS_LAUNCH(peel_solo_kernel<SOLO_EDGES>, 1, PEEL_SOLO_T, PEEL_SOLO_SMEM, s, a0, a1, dg, cop, cap, nact, ptr, adj,
                   tta, ttb, ttc, td, tnt, core_int, ct, max_steps);
    } else {
        LDS_LAUNCH(alive_list_kernel, grid_for(nact, blk), blk, 0, s, alive.get(), nact, a0, ct + PC_LIST);
        // one block of 1024 threads per SM: grid barriers get cheaper with fewer blocks
        const int pblk = 1024;
        // A peel of the whole triangle list takes thousands of short rounds: worth the pairs
        // (24 B a triangle, less than the index's sort had in use).  Pruning rounds peel a
        // compacted list in tens of rounds and would spend more on building them.
        const bool paired = tri && all_alive && tta != cta.get() && tnt > 0 && nact < (1 << 28);
        DevBuf<int2> pairs(paired ? 3 * tnt : 0, s);
        DevBuf<int32_t> stamp(paired ? nact : 0, s);
        if (paired) {
            LDS_CUDA(cudaMemsetAsync(stamp.get(), 0x7f, (size_t)nact * sizeof(int32_t), s));      // not taken
            LDS_LAUNCH(incidence_pairs_kernel, grid_for(3 * tnt, 4 * blk), blk, 0, s, ptr, adj, tta, ttb, ttc, nact, 3 * tnt,
                       pairs.get());
        }
        const int2* prs = pairs.get();
        int32_t* stp = stamp.get();
        const void* fn = paired ? (const void*)peel_coop_kernel<PEEL_PAIRS>
                                : tri ? (const void*)peel_coop_kernel<PEEL_TRIS> : (const void*)peel_coop_kernel<PEEL_EDGES>;
        grid = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms(), ((int64_t)nact + incid / 8 + pblk - 1) / pblk));
        if (tail) LDS_CUDA(cudaMemsetAsync(slotb.get(), 0xff, (size_t)nact * sizeof(int32_t), s));
        void* args[] = {(void*)&ptr, (void*)&adj, (void*)&tta, (void*)&ttb, (void*)&ttc, (void*)&td, (void*)&dg,
                        (void*)&core_int, (void*)&q0, (void*)&q1, (void*)&a0, (void*)&a1, (void*)&ct,
                        (void*)&max_steps, (void*)&solo, (void*)&slp, (void*)&cop, (void*)&cap,
                        (void*)&prs, (void*)&stp};
        LDS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(pblk), args, 0, s));
        g_launches.fetch_add(1, std::memory_order_relaxed);
        if (tail) {
            LDS_CUDA(cudaFuncSetAttribute(peel_solo_kernel<SOLO_TAIL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)PEEL_SOLO_SMEM));
            LDS_LAUNCH(peel_solo_kernel<SOLO_TAIL>, 1, PEEL_SOLO_T, PEEL_SOLO_SMEM, s, a0, a1, dg, cop, cap, nact, ptr,
                       adj, tta, ttb, ttc, td, tnt, core_int, ct, max_steps);
        }
    }
    if (verbose) LDS_CUDA(cudaEventRecord(e1, s));
    LDS_CUDA(cudaMemcpyAsync(hctrl, ctrl.get(), sizeof(hctrl), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    if (verbose) {
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        fprintf(stderr, "[core] nact=%d live=%d peel %.2f ms, %llu steps, last level %llu, grid %d\n", nact, remaining,
                ms, hctrl[PC_STEPS], hctrl[PC_LEVEL], grid);
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    }
    LDS_REQUIRE(hctrl[PC_ERR] == 0, LDS_ETIMEOUT, "core numbers: peeling hit its iteration bound");
    if (all_alive) {
        whole.alloc(nact, s);
        LDS_CUDA(cudaMemcpyAsync(whole.get(), core_int, (size_t)nact * sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
    }
}

void core_numbers(lds_graph* g, bool tri, int64_t* core_int_out, const uint8_t* init_alive) {
    core_numbers_internal(g, tri, core_int_out, init_alive);
}

}  // namespace lds

using namespace lds;

extern "C" {

lds_status lds_list_triangles(lds_graph* g, int64_t* count) {
    return guard([&] {
        LDS_REQUIRE(g, LDS_EINVAL, "lds_list_triangles: NULL graph");
        ensure_triangles(g);
        if (count) *count = g->ntri;
    });
}

lds_status lds_get_triangles(lds_graph* g, int32_t* tri, lds_mem where) {
    return guard([&] {
        LDS_REQUIRE(g && tri, LDS_EINVAL, "lds_get_triangles: NULL argument");
        LDS_REQUIRE(g->ntri >= 0, LDS_EINVAL, "lds_get_triangles: call lds_list_triangles first");
        if (g->ntri == 0) return;
        cudaStream_t s = g->stream;
        DevBuf<int32_t> rows(3 * g->ntri, s);
        LDS_LAUNCH(tri_rows_orig_kernel, grid_for(g->ntri, 256), 256, 0, s, g->ta.get(), g->tb.get(), g->tc.get(),
                                                                    g->to_orig.get(), g->ntri, rows.get());
        LDS_CHECK_LAUNCH();
        copy_out(tri, where, rows.get(), 3 * g->ntri * sizeof(int32_t), s);
        LDS_CUDA(cudaStreamSynchronize(s));
    });
}

lds_status lds_core_numbers(lds_graph* g, lds_density d, int64_t* core, lds_mem where) {
    return guard([&] {
        LDS_REQUIRE(g && core, LDS_EINVAL, "lds_core_numbers: NULL argument");
        LDS_REQUIRE(d == LDS_EDGE || d == LDS_TRIANGLE, LDS_EINVAL, "lds_core_numbers: bad density");
        cudaStream_t s = g->stream;
        const int32_t n = g->n;
        if (n == 0) return;
        DevBuf<int64_t> ci(n, s), co(n, s);
        LDS_CUDA(cudaMemsetAsync(ci.get(), 0, n * sizeof(int64_t), s));
        core_numbers_internal(g, d == LDS_TRIANGLE, ci.get(), nullptr);
        to_original_order_i64(g, ci.get(), co.get());
        copy_out(core, where, co.get(), n * sizeof(int64_t), s);
        LDS_CUDA(cudaStreamSynchronize(s));
    });
}

}  // extern "C"
