// Maximum flow and maximal minimum cut of the pattern network (Alg. 8) on the
// GPU, by push-relabel from a warm-started preflow.
//
// Network.  Alg. 8's network has a source s, a sink t, a node per pattern (a
// set of 1-3 vertices: an edge, a loop, a triangle or the part of one) and a
// node per vertex; arcs s -> pattern and pattern -> member have capacity q,
// vertex -> t has capacity p (rho = p / q).  Every capacity is multiplied by a
// power of two K (the cut structure is unchanged) so that a fractional split
// of each pattern's unit among its members can be written in integers.
//
// The preflow saturates every s -> pattern arc and splits each pattern's qK
// units among its members (in proportion to `share`, e.g. the Frank-Wolfe
// weights alpha, so that a near-optimal split leaves little excess); each
// vertex sends what it receives to t up to pK and keeps the rest as excess.
// Pattern nodes then hold no excess, and they are contracted where that is
// exact:
//   * a one-member pattern (a loop) only feeds its member: no node, no arc;
//   * a two-member pattern {a, b} with split (f_a, f_b) becomes the arc pair
//     a -> b (residual f_a) and b -> a (residual f_b): moving d units of the
//     pattern from a to b is a push along a -> b.  For a vertex set A on the
//     source side this pair adds f_a + f_b = qK to the cut exactly when one
//     member is in A and the other is not, which is what the pattern node's
//     arcs cost in Alg. 8's network, so every cut, the maximum flow and the
//     maximal minimum cut are unchanged;
//   * a pattern with three or more members keeps its node, with arcs
//     pattern -> member (residual qK - f) and member -> pattern (residual f).
// Excess that would return to s is never moved: it stays on nodes that cannot
// reach t, which is all the maximum flow and the largest source side need.
//
// Algorithm.  The preflow phase of push-relabel (Goldberg and Tarjan 1988) in
// the lock-free form for many threads (Hong 2008): an active node (positive
// excess, label below DEAD) pushes to its lowest residual neighbour when its
// label is higher, else relabels itself to that label plus one; capacities
// and excesses change by atomic adds only.  One warp serves one active node
// and scans its arcs 32 at a time (vertex nodes have hundreds of arcs).  Only
// active nodes are visited: a push that activates a node appends it to the
// next round's work list.  A global relabel (breadth-first search from t over
// residual arcs) runs first and whenever the relabels since the last one
// exceed the node count; nodes it does not reach are DEAD.  When no active
// node is left after a global relabel, the flow into t is the maximum flow and
// the DEAD vertices are the largest source side of a minimum cut (the cut that
// Lemma 9 uses).  Excess on a DEAD node can never reach t: a push into a DEAD
// node needs a label above DEAD, and valid labels of nodes that reach t stay
// below the node count.  Every loop is bounded; running out of the bound
// returns LDS_ETIMEOUT.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <utility>

#include "flow.cuh"
#include "prims.cuh"

namespace lds {

namespace {

constexpr int FB = 256;
constexpr int32_t DEAD = 0x3fffffff;       // label of nodes that cannot reach t
constexpr unsigned FULL = 0xffffffffu;

typedef unsigned long long ull;
typedef __int128 i128;

struct Net {
    int32_t nv;            // vertex nodes 0..nv-1 (they alone have sink arcs)
    int32_t nn;            // all nodes (vertex nodes, then pattern nodes)
    const int64_t* ptr;    // [nn + 1] arcs of node x at ptr[x] .. ptr[x+1]
    const int32_t* head;   // [A]
    int64_t* cap;          // [A] residual capacities
    const int64_t* rev;    // [A] twin arc
    int64_t* tcap;         // [nv] residual capacity to t
    int64_t* excess;       // [nn]
    int32_t* height;       // [nn]
};

// split of every pattern's qK units among its members; big[j] = pattern j keeps a node
__global__ void split_kernel(const int64_t* pptr, int32_t np, const int64_t* share, int64_t qK, int64_t* f,
                             int32_t* big) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const int64_t b = pptr[j], e = pptr[j + 1], len = e - b;
        big[j] = len >= 3;
        if (len == 0) continue;
        i128 tot = 0;
        if (share)
            for (int64_t k = b; k < e; ++k) tot += (i128)(share[k] > 0 ? share[k] : (int64_t)0);
        int64_t given = 0;
        for (int64_t k = b; k < e; ++k) {
            int64_t v;
            if (k == e - 1) v = qK - given;
            else if (tot > 0) v = (int64_t)((i128)qK * (i128)(share[k] > 0 ? share[k] : (int64_t)0) / tot);
            else v = qK / len;
            f[k] = v;
            given += v;
        }
    }
}

// node degrees and the flow each vertex receives
__global__ void degree_kernel(const int64_t* pptr, const int32_t* pidx, int32_t np, const int64_t* f,
                              const int64_t* bigpos, int32_t nv, int32_t* deg, ull* in) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const int64_t b = pptr[j], e = pptr[j + 1], len = e - b;
        for (int64_t k = b; k < e; ++k) {
            atomicAdd(in + pidx[k], (ull)f[k]);
            if (len >= 2) atomicAdd(deg + pidx[k], 1);
        }
        if (len >= 3) deg[nv + bigpos[j]] = (int32_t)len;
    }
}

__global__ void fill_kernel(const int64_t* pptr, const int32_t* pidx, int32_t np, const int64_t* f,
                            const int64_t* bigpos, int32_t nv, int64_t qK, const int64_t* ptr, int32_t* cursor,
                            int32_t* head, int64_t* cap, int64_t* rev) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const int64_t b = pptr[j], e = pptr[j + 1], len = e - b;
        if (len == 2) {
            const int32_t x = pidx[b], y = pidx[b + 1];
            const int64_t ax = ptr[x] + atomicAdd(cursor + x, 1);
            const int64_t ay = ptr[y] + atomicAdd(cursor + y, 1);
            head[ax] = y;
            cap[ax] = f[b];
            rev[ax] = ay;
            head[ay] = x;
            cap[ay] = f[b + 1];
            rev[ay] = ax;
        } else if (len >= 3) {
            const int32_t node = nv + (int32_t)bigpos[j];
            for (int64_t k = b; k < e; ++k) {
                const int32_t v = pidx[k];
                const int64_t ap = ptr[node] + (k - b);
                const int64_t av = ptr[v] + atomicAdd(cursor + v, 1);
                head[ap] = v;
                cap[ap] = qK - f[k];
                rev[ap] = av;
                head[av] = node;
                cap[av] = f[k];
                rev[av] = ap;
            }
        }
    }
}

__global__ void init_kernel(Net net, const ull* in, int64_t pK, ull* flow_t) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    ull acc = 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < net.nn; x += stride) {
        if (x < net.nv) {
            const int64_t r = (int64_t)in[x];
            const int64_t toT = min(r, pK);
            net.tcap[x] = pK - toT;
            net.excess[x] = r - toT;
            acc += (ull)toT;
        } else {
            net.excess[x] = 0;
        }
    }
    if (acc) atomicAdd(flow_t, acc);
}

// ---- global relabel

__global__ void gr_init_kernel(Net net, int32_t* frontier, int32_t* fcnt) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < net.nn; x += stride) {
        const bool hit = x < net.nv && net.tcap[x] > 0;
        net.height[x] = hit ? 1 : DEAD;
        if (hit) frontier[atomicAdd(fcnt, 1)] = (int32_t)x;
    }
}

// one level: x joins at level + 1 when it has a residual arc to a frontier node y
__global__ void gr_level_kernel(Net net, const int32_t* frontier, const int32_t* fcnt, int32_t level, int32_t* next,
                                int32_t* ncnt) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int32_t nf = *fcnt;
    for (int64_t i = warp; i < nf; i += nwarps) {
        const int32_t y = frontier[i];
        for (int64_t a = net.ptr[y] + lane; a < net.ptr[y + 1]; a += 32) {
            const int32_t x = net.head[a];
            if (__ldcg(net.height + x) == DEAD && net.cap[net.rev[a]] > 0)
                if (atomicCAS(net.height + x, DEAD, level + 1) == DEAD) next[atomicAdd(ncnt, 1)] = x;
        }
    }
}

// after a global relabel: work list of the active nodes, count of stuck excess
__global__ void gr_finish_kernel(Net net, int32_t* list, int32_t* lcnt, int32_t* inq, int32_t tag, int32_t* stuck) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int32_t st = 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < net.nn; x += stride) {
        if (net.excess[x] <= 0) continue;
        if (net.height[x] < DEAD) {
            inq[x] = tag;
            list[atomicAdd(lcnt, 1)] = (int32_t)x;
        } else {
            ++st;
        }
    }
    if (st) atomicAdd(stuck, st);
}

// ---- push-relabel round: one warp per node of the current work list.  The
// lists and counts were written by earlier launches; values that other warps
// change during the round are read through L2 (__ldcg) or by atomics.
__global__ void __launch_bounds__(FB) pr_round_kernel(Net net, const int32_t* cur, const int32_t* cur_cnt, int32_t* nxt,
                                                     int32_t* nxt_cnt, int32_t* clear_cnt, int32_t* inq, int32_t tag,
                                                     int pulses, ull* flow_t, int32_t* relabels) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *clear_cnt = 0;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int32_t ncur = *cur_cnt;
    int32_t nrel = 0;
    for (int64_t i = warp; i < ncur; i += nwarps) {
        const int32_t x = cur[i];
        const int64_t a0 = net.ptr[x], a1 = net.ptr[x + 1];
        for (int it = 0; it < pulses; ++it) {
            const int64_t e = __ldcg(net.excess + x);
            const int32_t hx = __ldcg(net.height + x);
            if (e <= 0 || hx >= DEAD) break;
            if (x < net.nv) {
                const int64_t tc = __ldcg(net.tcap + x);
                if (tc > 0) {          // t (label 0) is the lowest neighbour
                    if (lane == 0) {
                        const int64_t d = min(e, tc);
                        atomicAdd((ull*)(net.tcap + x), (ull)(-d));
                        atomicAdd((ull*)(net.excess + x), (ull)(-d));
                        atomicAdd(flow_t, (ull)d);
                    }
                    __syncwarp();
                    continue;
                }
            }
            int32_t hmin = INT32_MAX;
            int64_t best = -1, capb = 0;
            for (int64_t a = a0 + lane; a < a1; a += 32) {
                const int64_t c = __ldcg(net.cap + a);
                if (c > 0) {
                    const int32_t hy = __ldcg(net.height + net.head[a]);
                    if (hy < hmin) {
                        hmin = hy;
                        best = a;
                        capb = c;
                    }
                }
            }
            const int32_t gmin = (int32_t)__reduce_min_sync(FULL, (unsigned)hmin);
            if (gmin == INT32_MAX) {           // no residual arc left
                if (lane == 0) net.height[x] = DEAD;
                __syncwarp();
                break;
            }
            const int src = __ffs(__ballot_sync(FULL, hmin == gmin)) - 1;
            best = __shfl_sync(FULL, best, src);
            capb = __shfl_sync(FULL, capb, src);
            if (hx > gmin) {
                if (lane == 0) {
                    // only x lowers its own arcs' capacities and its own excess, so d stays available
                    const int64_t d = min(e, capb);
                    const int32_t y = net.head[best];
                    atomicAdd((ull*)(net.cap + best), (ull)(-d));
                    atomicAdd((ull*)(net.cap + net.rev[best]), (ull)d);
                    atomicAdd((ull*)(net.excess + x), (ull)(-d));
                    const long long old = (long long)atomicAdd((ull*)(net.excess + y), (ull)d);
                    if (old <= 0 && atomicExch(inq + y, tag) != tag) nxt[atomicAdd(nxt_cnt, 1)] = y;
                }
            } else {
                if (lane == 0) net.height[x] = min(gmin + 1, DEAD);
                ++nrel;
            }
            __syncwarp();
        }
        if (lane == 0 && (long long)atomicAdd((ull*)(net.excess + x), 0ull) > 0 && __ldcg(net.height + x) < DEAD &&
            atomicExch(inq + x, tag) != tag)
            nxt[atomicAdd(nxt_cnt, 1)] = x;
    }
    if (lane == 0 && nrel) atomicAdd(relabels, nrel);
}

__global__ void side_kernel(const int32_t* height, int32_t nv, uint8_t* side) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += stride) side[v] = height[v] >= DEAD;
}

// blocks for a warp-per-item launch, at most 8 blocks per SM
int warps_grid(int64_t items) {
    const int64_t cap = (int64_t)num_sms() * 8;
    const int64_t b = (items * 32 + FB - 1) / FB;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, cap));
}

// ---- vertex-node form (no pattern nodes)
//
// After the preflow every pattern P holds its qK units split among its members
// (f_{P,x}).  In Alg. 8's network the residual path x -> P -> y exists exactly
// when f_{P,x} > 0, and pushing d units along it is f_{P,x} -= d, f_{P,y} += d.
// So the network needs no pattern nodes: x has a hyper-arc to every other
// member y of P, all of them drawing on the same capacity f_{P,x}.  Labels
// stay valid under such a push: if h(x) = h(y) + 1 and the push makes y -> z
// through P residual for a third member z, then x -> z through P was residual,
// so h(x) <= h(z) + 1 and h(y) <= h(z).  The vertices that cannot reach t in
// this residual structure are exactly those that cannot reach t in Alg. 8's
// network, so the DEAD vertices at the end are the largest source side.
//
// Layout: the incidences of every vertex are contiguous (vptr); incidence i
// holds f (its vertex's share of the pattern) and the incidences / vertices of
// the pattern's other members (at most two; -1 where absent).  Loops (one
// member) only feed their vertex and have no incidence.
struct HNet {
    int32_t nv;
    const int64_t* vptr;   // [nv + 1]
    int64_t* f;            // [ninc]
    const int32_t* o1;     // [ninc] incidence of another member, -1 if none
    const int32_t* o2;
    const int32_t* w1;     // [ninc] vertex of that member, -1 if none
    const int32_t* w2;
    int64_t* tcap;         // [nv] residual capacity to t
    int64_t* excess;       // [nv]
    int32_t* h;            // [nv] exact distance to t (DEAD: cannot reach it)
    int64_t* claim;        // [nv] admissible capacity claimed in this sweep
    const int2* chunk;     // vertex and first incidence of every chunk of HY_CHUNK incidences
    const int64_t* nchunk; // their number
};

constexpr int HY_GROUP = 8;                    // lanes that take a chunk together
constexpr int HY_ITEMS = 4;                    // incidences per lane
constexpr int HY_CHUNK = HY_GROUP * HY_ITEMS;
constexpr int HY_THREADS = 1024;

__global__ void hyper_chunk_count_kernel(const int64_t* vptr, int32_t nv, int32_t* cnt) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= nv; v += stride)
        cnt[v] = v < nv ? (int32_t)((vptr[v + 1] - vptr[v] + HY_CHUNK - 1) / HY_CHUNK) : 0;
}

// one warp per vertex
__global__ void hyper_chunk_fill_kernel(const int64_t* vptr, int32_t nv, const int64_t* coff, int2* chunk) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < nv; v += nwarps)
        for (int64_t c = coff[v] + lane; c < coff[v + 1]; c += 32)
            chunk[c] = make_int2((int32_t)v, (int32_t)(vptr[v] + (c - coff[v]) * HY_CHUNK));
}

// widths above 3 are refused (wide bit 0; bit 1: some pattern has three members); count[v] = incidences of v; in[v] = flow v receives
__global__ void hyper_degree_kernel(const int64_t* pptr, const int32_t* pidx, int32_t np, const int64_t* f,
                                    int32_t* deg, ull* in, int32_t* wide) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const int64_t b = pptr[j], e = pptr[j + 1], len = e - b;
        if (len > 3) {
            atomicOr(wide, 1);
            continue;
        }
        if (len == 3 && !(__ldcg(wide) & 2)) atomicOr(wide, 2);
        for (int64_t k = b; k < e; ++k) {
            atomicAdd(in + pidx[k], (ull)f[k]);
            if (len >= 2) atomicAdd(deg + pidx[k], 1);
        }
    }
}

// position of every slot (of a pattern with >= 2 members) in its vertex's incidence list
__global__ void hyper_pos_kernel(const int64_t* pptr, const int32_t* pidx, int32_t np, const int64_t* vptr,
                                 int32_t* cursor, int32_t* pos) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const int64_t b = pptr[j], e = pptr[j + 1];
        if (e - b < 2 || e - b > 3) continue;
        for (int64_t k = b; k < e; ++k) pos[k] = (int32_t)(vptr[pidx[k]] + atomicAdd(cursor + pidx[k], 1));
    }
}

// The same counts and positions where few vertices take many patterns: a block counts
// its range of patterns in shared memory, takes one run of every vertex's list from the
// cursor, and numbers its slots within the runs, one shared addition per vertex and warp.
// With global counters 22 million triangles over 988 vertices took 6.1 ms to count and
// 6.4 ms to place, all on the same few addresses; 0.21 ms, 0.26 ms, and 0.25 ms for the
// flow that each vertex receives, so.  Positions in runs also help the fill (3.0 to 1.8
// ms) and the flow itself (16.2 to 11.0 ms).
constexpr int HP_THREADS = 512;
constexpr int HP_MAX_NV = 8192;                // 32 KB of counters a block
__global__ void __launch_bounds__(HP_THREADS) hyper_count_runs_kernel(const int64_t* pptr, const int32_t* pidx, int32_t np,
                                                                      const int64_t* f, int32_t nv, int64_t per,
                                                                      int32_t* deg, ull* in, int32_t* wide, int32_t* runs) {
    extern __shared__ int32_t hcount[];
    for (int32_t v = threadIdx.x; v < nv; v += HP_THREADS) hcount[v] = 0;
    __syncthreads();
    const int64_t j0 = blockIdx.x * per, j1 = min((int64_t)np, j0 + per);
    for (int64_t j = j0 + threadIdx.x; j < j1; j += HP_THREADS) {
        const int64_t b = pptr[j], e = pptr[j + 1], len = e - b;
        if (len > 3) {
            atomicOr(wide, 1);
            continue;
        }
        if (len == 3 && !(__ldcg(wide) & 2)) atomicOr(wide, 2);
        if (len == 1) atomicAdd(in + pidx[b], (ull)f[b]);
        else
            for (int64_t k = b; k < e; ++k) atomicAdd(hcount + pidx[k], 1);
    }
    __syncthreads();
    for (int32_t v = threadIdx.x; v < nv; v += HP_THREADS) {
        const int32_t c = hcount[v];
        runs[(int64_t)blockIdx.x * nv + v] = c;
        if (c) atomicAdd(deg + v, c);
    }
}

__global__ void __launch_bounds__(HP_THREADS) hyper_place_runs_kernel(const int64_t* pptr, const int32_t* pidx, int32_t np,
                                                                      int32_t nv, int64_t per, const int64_t* vptr,
                                                                      int32_t* cursor, const int32_t* runs, int32_t* pos) {
    extern __shared__ int32_t hcount[];
    const int lane = threadIdx.x & 31;
    for (int32_t v = threadIdx.x; v < nv; v += HP_THREADS) {
        const int32_t c = runs[(int64_t)blockIdx.x * nv + v];
        hcount[v] = c ? (int32_t)vptr[v] + atomicAdd(cursor + v, c) : 0;
    }
    __syncthreads();
    const int64_t j0 = blockIdx.x * per, j1 = min((int64_t)np, j0 + per);
    for (int64_t jw = j0 + threadIdx.x - lane; jw < j1; jw += HP_THREADS) {
        const int64_t j = jw + lane;
        int64_t b = 0;
        int len = 0;
        if (j < j1) {
            b = pptr[j];
            len = (int)(pptr[j + 1] - b);
        }
        if (len < 2 || len > 3) len = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int32_t x = k < len ? pidx[b + k] : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, x);
            const int lead = __ffs(peers) - 1;
            int32_t at = 0;
            if (x >= 0 && lane == lead) at = atomicAdd(hcount + x, __popc(peers));
            at = __shfl_sync(0xffffffffu, at, lead);
            if (x >= 0) pos[b + k] = at + __popc(peers & ((1u << lane) - 1u));
        }
    }
}

// in[v] += flow over v's incidences; `parts` warps a vertex
__global__ void hyper_in_kernel(HNet net, int32_t parts, ull* in) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < (int64_t)net.nv * parts; w += nwarps) {
        const int32_t v = (int32_t)(w / parts), part = (int32_t)(w % parts);
        const int64_t e = net.vptr[v + 1];
        ull sum = 0;
        for (int64_t i = net.vptr[v] + part * 32 + lane; i < e; i += 32 * (int64_t)parts) sum += (ull)net.f[i];
        for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0 && sum) atomicAdd(in + v, sum);
    }
}

__global__ void hyper_fill_kernel(const int64_t* pptr, const int32_t* pidx, int32_t np, const int64_t* fslot,
                                  const int32_t* pos, HNet net) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const int64_t b = pptr[j], e = pptr[j + 1], len = e - b;
        if (len < 2 || len > 3) continue;
        for (int64_t k = b; k < e; ++k) {
            const int64_t a = k == b ? b + 1 : b;                  // the other members, in slot order
            const int64_t c = len == 3 ? (k == e - 1 ? e - 2 : e - 1) : -1;
            const int32_t i = pos[k];
            net.f[i] = fslot[k];
            ((int32_t*)net.o1)[i] = pos[a];
            ((int32_t*)net.w1)[i] = pidx[a];
            ((int32_t*)net.o2)[i] = c >= 0 ? pos[c] : -1;
            ((int32_t*)net.w2)[i] = c >= 0 ? pidx[c] : -1;
        }
    }
}

__global__ void hyper_init_kernel(HNet net, const ull* in, int64_t pK, ull* flow_t) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    ull acc = 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < net.nv; x += stride) {
        const int64_t r = (int64_t)in[x];
        const int64_t toT = min(r, pK);
        net.tcap[x] = pK - toT;
        net.excess[x] = r - toT;
        acc += (ull)toT;
    }
    if (acc) atomicAdd(flow_t, acc);
}

// hyper_flow_kernel control words
enum : int {
    HC_EXCESS = 0,     // [3] vertices holding excess (by phase, three rotating counters)
    HC_ACTIVE = 3,     // [3] of them, those that label 1 takes
    HC_ADDED = 6,      // [3] a breadth-first level: vertices it labelled, << 32 those holding excess
    HC_FLOW = 9,       // flow into t
    HC_STATUS = 10,    // 0 finished, 1 phase bound hit, 2 stopped: some excess cannot reach t
    HC_PHASES = 11,
    HC_LEVELS = 12,    // breadth-first levels run in all
    HC_WORDS = 13
};

// One cooperative launch runs the whole preflow phase.  Each phase settles the
// vertices (what the last sweep pushed leaves their excess; label 1 pushes into t),
// computes exact distance labels by a breadth-first search from t over the residual
// hyper-arcs (a global relabel), stopping once every vertex that holds excess has a
// label, then sweeps the labels from the highest down to 2: every vertex at label L
// with excess pushes it along its admissible hyper-arcs (to members at label L - 1)
// until the excess or those arcs run out.  Within a label no two vertices touch the
// same share from below (a share is lowered only by its own vertex, and vertices at
// label L receive nothing while label L is swept), so a push needs atomics only on
// the target's share and excess.  The chunks of one vertex share its excess through
// `claim`: a chunk adds its admissible capacity there and may push what of the
// excess lies past the capacity claimed before it, so exactly min(excess, admissible
// capacity) leaves the vertex.  Every vertex that still holds excess then has no
// admissible hyper-arc, and since no push shortens a distance, its label rises in
// the next phase; labels are at most nv, so there are at most nv^2 + 1 phases.
// `max_phases` bounds the loop (status 1).
//
// The phases are short and many (100 on the 1,511-vertex core of the 1M-vertex
// power-law graph), so what bounds a step is its chain of L2 accesses and the grid
// barrier.  Incidences are cut into chunks of 32, eight lanes take one with four
// loads in flight each, and a lane looks at one chunk's vertex to find the chunks
// that have work, so low and high degrees spread alike; one block of 1,024 threads
// per SM keeps the barrier cheap.  IsDensest, building the network included, against
// one warp per vertex and four blocks per SM (GB300): that core 7.3 -> 3.0 ms; 37,622
// vertices of degree 11 (Barabasi-Albert) 9.4 -> 1.4 ms; 66.6M incidences of 988
// vertices (R-MAT scale 18 triangles) 90 -> 55 ms.
template <bool PAIRS>
__global__ void __launch_bounds__(HY_THREADS, 1) hyper_flow_kernel(const HNet net, ull* ctrl, int64_t max_phases,
                                                                   int stop_if_short, int want_side) {
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31, gl = lane & (HY_GROUP - 1), gbase = lane & ~(HY_GROUP - 1);
    const int64_t warp = tid >> 5, ngroups = nthreads / HY_GROUP;
    const int32_t nv = net.nv;
    const int64_t nc = *net.nchunk;
    // calls body(active, v, start, e) warp-wide for every chunk that pick(v, e) takes,
    // one per group of lanes at a time; e is what pick stored
    auto for_chunks = [&](auto&& pick, auto&& body) {
        for (int64_t base = warp * (32 / HY_GROUP); base < nc; base += HY_GROUP * ngroups) {
            const int64_t c = base + gbase / HY_GROUP + (int64_t)gl * ngroups;
            int2 ch = make_int2(0, 0);
            int64_t e = 0;
            bool take = false;
            if (c < nc) {
                ch = net.chunk[c];
                take = pick(ch.x, e);
            }
            unsigned mask = (__ballot_sync(FULL, take) >> gbase) & ((1u << HY_GROUP) - 1u);
            while (__any_sync(FULL, mask != 0)) {
                const bool on = mask != 0;
                const int from = gbase + (on ? __ffs(mask) - 1 : 0);
                mask &= mask - 1;
                const int32_t v = __shfl_sync(FULL, ch.x, from), st = __shfl_sync(FULL, ch.y, from);
                body(on, v, st, __shfl_sync(FULL, e, from));
            }
        }
    };
    int lc = 0;                                   // breadth-first levels so far
    for (int64_t phase = 0;; ++phase) {
        if (phase >= max_phases) {
            if (tid == 0) ctrl[HC_STATUS] = 1;
            return;
        }
        const int ps = (int)(phase % 3), pn = (int)((phase + 1) % 3);
        if (tid == 0) {
            ctrl[HC_EXCESS + pn] = ctrl[HC_ACTIVE + pn] = 0;
            ctrl[HC_ADDED + lc % 3] = 0;
            ctrl[HC_PHASES] = (ull)phase + 1;
        }
        // settle: excess after the last sweep, label 1 for what can still push into t
        {
            unsigned ne = 0, na = 0;
            ull fl = 0;
            for (int64_t v = tid; v < nv; v += nthreads) {
                int64_t e = __ldcg(net.excess + v), tc = __ldcg(net.tcap + v);
                if (phase > 0 && e > 0) {
                    if (__ldcg(net.h + v) == 1) {
                        const int64_t d = min(e, tc);
                        tc -= d;
                        e -= d;
                        fl += (ull)d;
                        net.tcap[v] = tc;
                        net.excess[v] = e;
                    } else {
                        const int64_t d = min(e, __ldcg(net.claim + v));
                        if (d) {
                            e -= d;
                            net.excess[v] = e;
                            net.claim[v] = 0;
                        }
                    }
                }
                net.h[v] = tc > 0 ? 1 : DEAD;
                ne += e > 0;
                na += e > 0 && tc > 0;
            }
            ne = __reduce_add_sync(FULL, ne);
            na = __reduce_add_sync(FULL, na);
            for (int o = 16; o; o >>= 1) fl += __shfl_xor_sync(FULL, fl, o);
            if (lane == 0) {
                if (ne) atomicAdd(ctrl + HC_EXCESS + ps, (ull)ne);
                if (na) atomicAdd(ctrl + HC_ACTIVE + ps, (ull)na);
                if (fl) atomicAdd(ctrl + HC_FLOW, fl);
            }
        }
        grid.sync();
        const ull ne = __ldcg(ctrl + HC_EXCESS + ps);
        ull act = __ldcg(ctrl + HC_ACTIVE + ps);
        if (ne == 0 && !want_side) return;               // the flow is complete (status 0)
        // breadth-first levels: an unlabelled vertex joins level L + 1 when one of its
        // hyper-arcs (share > 0) leads to a member at level L
        int32_t top = 1;
        while (ne == 0 || act < ne) {
            const int32_t L = top;
            if (tid == 0) {
                ctrl[HC_ADDED + (lc + 1) % 3] = 0;
                ctrl[HC_LEVELS] += 1;
            }
            unsigned won = 0, wone = 0;                  // vertices this thread labelled, those holding excess
            for_chunks([&](int32_t v, int64_t&) { return __ldcg(net.h + v) == DEAD; },
                       [&](bool on, int32_t v, int32_t st, int64_t) {
                           bool hit = false;
                           if (on) {
                               const int32_t end = (int32_t)min(net.vptr[v + 1], (int64_t)st + HY_CHUNK);
                               int32_t w[HY_ITEMS][2];
#pragma unroll
                               for (int j = 0; j < HY_ITEMS; ++j) {
                                   const int32_t i = st + gl + j * HY_GROUP;
                                   w[j][0] = w[j][1] = -1;
                                   if (i < end && __ldcg(net.f + i) > 0) {
                                       w[j][0] = net.w1[i];
                                       if (!PAIRS) w[j][1] = net.w2[i];
                                   }
                               }
#pragma unroll
                               for (int j = 0; j < HY_ITEMS; ++j) {
                                   if (w[j][0] >= 0) hit |= __ldcg(net.h + w[j][0]) == L;
                                   if (!PAIRS && w[j][1] >= 0) hit |= __ldcg(net.h + w[j][1]) == L;
                               }
                           }
                           const unsigned any = (__ballot_sync(FULL, hit) >> gbase) & ((1u << HY_GROUP) - 1u);
                           // the group's first lane labels the vertex, once
                           if (any && gl == 0 && atomicCAS(net.h + v, DEAD, L + 1) == DEAD) {
                               ++won;
                               wone += __ldcg(net.excess + v) > 0;
                           }
                       });
            won = __reduce_add_sync(FULL, won);
            wone = __reduce_add_sync(FULL, wone);
            if (lane == 0 && won) atomicAdd(ctrl + HC_ADDED + lc % 3, ((ull)wone << 32) | won);
            grid.sync();
            // this level's own counter: blocks that run ahead write the next one
            const ull added = __ldcg(ctrl + HC_ADDED + lc % 3);
            act += added >> 32;
            ++lc;
            if (!added) break;
            top = L + 1;
        }
        if (ne == 0) return;
        if (stop_if_short && act < ne) {
            if (tid == 0) ctrl[HC_STATUS] = 2;
            return;
        }
        if (act == 0) return;
        // downhill sweep
        for (int32_t L = top; L >= 2; --L) {
            for_chunks(
                [&](int32_t v, int64_t& e) {
                    if (__ldcg(net.h + v) != L) return false;
                    e = __ldcg(net.excess + v);
                    return e > 0;
                },
                [&](bool on, int32_t v, int32_t st, int64_t e) {
                    int64_t cap[HY_ITEMS], mine = 0;
                    int32_t to[HY_ITEMS];
                    bool second[HY_ITEMS];
#pragma unroll
                    for (int j = 0; j < HY_ITEMS; ++j) {
                        cap[j] = 0;
                        to[j] = -1;
                        second[j] = false;
                    }
                    if (on) {
                        const int32_t end = (int32_t)min(net.vptr[v + 1], (int64_t)st + HY_CHUNK);
                        int32_t w[HY_ITEMS][2];
#pragma unroll
                        for (int j = 0; j < HY_ITEMS; ++j) {
                            const int32_t i = st + gl + j * HY_GROUP;
                            w[j][0] = w[j][1] = -1;
                            if (i < end) {
                                cap[j] = __ldcg(net.f + i);
                                w[j][0] = net.w1[i];
                                if (!PAIRS) w[j][1] = net.w2[i];
                            }
                        }
#pragma unroll
                        for (int j = 0; j < HY_ITEMS; ++j) {
                            if (cap[j] > 0) {
                                if (w[j][0] >= 0 && __ldcg(net.h + w[j][0]) == L - 1) {
                                    to[j] = w[j][0];
                                } else if (!PAIRS && w[j][1] >= 0 && __ldcg(net.h + w[j][1]) == L - 1) {
                                    to[j] = w[j][1];
                                    second[j] = true;
                                }
                            }
                            if (to[j] < 0) cap[j] = 0;
                            mine += cap[j];
                        }
                    }
                    // shares of all incidences sum to at most np q K <= 2^61: no overflow
                    int64_t incl = mine;
#pragma unroll
                    for (int o = 1; o < HY_GROUP; o <<= 1) {
                        const int64_t t = __shfl_up_sync(FULL, incl, o, HY_GROUP);
                        if (gl >= o) incl += t;
                    }
                    const int64_t all = __shfl_sync(FULL, incl, HY_GROUP - 1, HY_GROUP);
                    int64_t before = 0;
                    if (gl == 0 && all > 0) before = (int64_t)atomicAdd((ull*)(net.claim + v), (ull)all);
                    before = __shfl_sync(FULL, before, 0, HY_GROUP);
                    if (all > 0) {
                        int64_t rem = e - before - (incl - mine);       // excess left for this lane's arcs
#pragma unroll
                        for (int j = 0; j < HY_ITEMS; ++j) {
                            const int64_t d = min(cap[j], rem);
                            if (d > 0) {
                                const int32_t i = st + gl + j * HY_GROUP;
                                __stcg(net.f + i, cap[j] - d);
                                atomicAdd((ull*)(net.f + (second[j] ? net.o2[i] : net.o1[i])), (ull)d);
                                atomicAdd((ull*)(net.excess + to[j]), (ull)d);
                            }
                            rem -= cap[j];
                        }
                    }
                });
            grid.sync();
        }
    }
}

}  // namespace

std::atomic<int> g_flow_variant{0};

// The vertex-node form of the maximum flow, from the split f of every slot.
static int64_t hyper_max_flow(const int64_t* pptr, const int32_t* pidx, int32_t np, int32_t nv, int64_t nidx,
                              const int64_t* fslot, int64_t pK, int64_t K, uint8_t* side, bool stop_if_short,
                              cudaStream_t s) {
    const int32_t nvp = std::max(nv, 1);
    DevBuf<int32_t> deg(nvp + 1, s), cursor(nvp, s), wide(1, s);
    DevBuf<ull> in(nvp, s), ctrl(HC_WORDS, s);
    LDS_CUDA(cudaMemsetAsync(deg.get(), 0, (nvp + 1) * sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(cursor.get(), 0, nvp * sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(wide.get(), 0, sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(in.get(), 0, nvp * sizeof(ull), s));
    LDS_CUDA(cudaMemsetAsync(ctrl.get(), 0, HC_WORDS * sizeof(ull), s));
    // counters per block: at least as many patterns a block as it has counters to flush.
    // Verification of a query with them and without: 2,000 vertices with 1M edges 0.92 and
    // 1.3 ms; triangles of R-MAT 14 5.1 and 7.5, of R-MAT 16 4.7 and 9.0
    const int64_t blocks = std::min<int64_t>(2 * num_sms(), np / std::max(nv, 1024));
    const bool by_runs = nv > 0 && nv <= HP_MAX_NV && blocks >= 2;
    const int64_t per = by_runs ? (np + blocks - 1) / blocks : 0;
    const size_t hsmem = (size_t)nv * sizeof(int32_t);
    DevBuf<int32_t> runs(by_runs ? blocks * nv : 0, s);
    if (by_runs)
        LDS_LAUNCH(hyper_count_runs_kernel, (unsigned)blocks, HP_THREADS, hsmem, s, pptr, pidx, np, fslot, nv, per, deg.get(),
                   in.get(), wide.get(), runs.get());
    else if (np)
        LDS_LAUNCH(hyper_degree_kernel, grid_for(np, FB), FB, 0, s, pptr, pidx, np, fslot, deg.get(), in.get(),
                   wide.get());
    DevBuf<int64_t> vptr(nvp + 1, s);
    const int64_t ninc = exclusive_scan_i32_to_i64(deg.get(), vptr.get(), (int64_t)nv + 1, s);
    int32_t hwide = 0;
    LDS_CUDA(cudaMemcpyAsync(&hwide, wide.get(), sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    LDS_REQUIRE(!(hwide & 1), LDS_EINVAL, "max flow: a pattern has more than three members");
    LDS_REQUIRE(ninc < (int64_t)INT32_MAX, LDS_EOVERFLOW, "max flow: %lld incidences exceed the 32-bit index",
                (long long)ninc);
    DevBuf<int32_t> pos(std::max<int64_t>(nidx, 1), s);
    DevBuf<int64_t> f(std::max<int64_t>(ninc, 1), s), tcap(nvp, s), excess(nvp, s);
    DevBuf<int32_t> o1(std::max<int64_t>(ninc, 1), s), o2(std::max<int64_t>(ninc, 1), s);
    DevBuf<int32_t> w1(std::max<int64_t>(ninc, 1), s), w2(std::max<int64_t>(ninc, 1), s), h(nvp, s);
    DevBuf<int64_t> claim(nvp, s), coff(nvp + 1, s);
    DevBuf<int2> chunk((size_t)nvp + ninc / HY_CHUNK + 1, s);
    LDS_CUDA(cudaMemsetAsync(claim.get(), 0, nvp * sizeof(int64_t), s));
    HNet net{nv,         vptr.get(),   f.get(), o1.get(),    o2.get(),    w1.get(),       w2.get(),
             tcap.get(), excess.get(), h.get(), claim.get(), chunk.get(), coff.get() + nv};
    if (nv) {
        DevBuf<int32_t> ccnt(nvp + 1, s);
        LDS_LAUNCH(hyper_chunk_count_kernel, grid_for(nv + 1, FB), FB, 0, s, vptr.get(), nv, ccnt.get());
        exclusive_scan_i32_dev(ccnt.get(), coff.get(), (int64_t)nv + 1, s);
        LDS_LAUNCH(hyper_chunk_fill_kernel, grid_for((int64_t)nv * 32, FB), FB, 0, s, vptr.get(), nv, coff.get(),
                   chunk.get());
    }
    if (np) {
        if (by_runs)
            LDS_LAUNCH(hyper_place_runs_kernel, (unsigned)blocks, HP_THREADS, hsmem, s, pptr, pidx, np, nv, per, vptr.get(),
                       cursor.get(), runs.get(), pos.get());
        else
            LDS_LAUNCH(hyper_pos_kernel, grid_for(np, FB), FB, 0, s, pptr, pidx, np, vptr.get(), cursor.get(), pos.get());
        LDS_LAUNCH(hyper_fill_kernel, grid_for(np, FB), FB, 0, s, pptr, pidx, np, fslot, pos.get(), net);
        if (by_runs) {
            // 16,384 warps in all: R-MAT 16 triangles 4.7 ms, with one a vertex 5.6, with 2,048
            // warps 5.2, with 65,536 4.8
            const int32_t parts = (int32_t)std::max(1, 16384 / nv);
            LDS_LAUNCH(hyper_in_kernel, grid_for((int64_t)nv * parts * 32, FB), FB, 0, s, net, parts, in.get());
        }
    }
    if (nv) LDS_LAUNCH(hyper_init_kernel, grid_for(nv, FB), FB, 0, s, net, in.get(), pK, ctrl.get() + HC_FLOW);
    if (nv) {
        // a group of lanes per chunk; at most one block per SM, all resident at once
        const int64_t want = (((int64_t)nv + ninc / HY_CHUNK) * HY_GROUP + HY_THREADS - 1) / HY_THREADS;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, num_sms()));
        const int64_t max_phases = std::min<int64_t>((int64_t)nv * nv + 2, (int64_t)1 << 40);
        int stop = stop_if_short ? 1 : 0, ws = side ? 1 : 0;
        ull* cp = ctrl.get();
        void* args[] = {(void*)&net, (void*)&cp, (void*)&max_phases, (void*)&stop, (void*)&ws};
        const void* fn = hwide & 2 ? (const void*)hyper_flow_kernel<false> : (const void*)hyper_flow_kernel<true>;
        LDS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(HY_THREADS), args, 0, s));
        g_launches.fetch_add(1, std::memory_order_relaxed);
    }
    ull hc[HC_WORDS];
    LDS_CUDA(cudaMemcpyAsync(hc, ctrl.get(), sizeof(hc), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    LDS_REQUIRE(hc[HC_STATUS] != 1, LDS_ETIMEOUT, "max flow: phase bound hit");
    if (hc[HC_STATUS] == 2) return -1;
    if (side && nv) LDS_LAUNCH(side_kernel, grid_for(nv, FB), FB, 0, s, h.get(), nv, side);
    LDS_CUDA(cudaStreamSynchronize(s));
    const ull ft = hc[HC_FLOW];
    LDS_REQUIRE((int64_t)ft % K == 0, LDS_ECUDA, "max flow: flow value %llu is not a multiple of the scale", ft);
    return (int64_t)ft / K;
}

int64_t pattern_max_flow(const int64_t* pptr, const int32_t* pidx, int32_t np, int32_t nv, int64_t p, int64_t q,
                         const int64_t* share, uint8_t* side, bool stop_if_short, cudaStream_t s) {
    LDS_REQUIRE(q > 0 && p >= 0 && np >= 0 && nv >= 0, LDS_EINVAL, "max flow: bad network");
    // K: the largest power of two up to 2^20 with np q K <= 2^61, so every sum of flows fits
    int64_t K = 1;
    const i128 unit = (i128)std::max<int64_t>(np, 1) * q;
    while (K < (1 << 20) && unit * (K * 2) <= ((i128)1 << 61)) K *= 2;
    LDS_REQUIRE(unit * K <= ((i128)1 << 62) && (i128)p * K <= ((i128)1 << 62), LDS_EOVERFLOW,
                "max flow: capacities overflow");
    const int64_t qK = q * K, pK = p * K;
    int64_t nidx = 0;
    if (np) {
        LDS_CUDA(cudaMemcpyAsync(&nidx, pptr + np, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        LDS_CUDA(cudaStreamSynchronize(s));
    }
    DevBuf<int64_t> f(std::max<int64_t>(nidx, 1), s);
    DevBuf<int32_t> big(np + 1, s);
    DevBuf<int64_t> bigpos(np + 1, s);
    LDS_CUDA(cudaMemsetAsync(big.get(), 0, (np + 1) * sizeof(int32_t), s));
    int64_t n3 = 0;
    if (np) {
        LDS_LAUNCH(split_kernel, grid_for(np, FB), FB, 0, s, pptr, np, share, qK, f.get(), big.get());
        n3 = exclusive_scan_i32_to_i64(big.get(), bigpos.get(), np + 1, s);
    }
    // the vertex-node form is the default (variant 0)
    const int variant = g_flow_variant.load(std::memory_order_relaxed);
    if (variant != 1)
        return hyper_max_flow(pptr, pidx, np, nv, nidx, f.get(), pK, K, side, stop_if_short, s);
    LDS_REQUIRE((int64_t)nv + n3 < (int64_t)DEAD, LDS_EOVERFLOW, "max flow: too many nodes");
    const int32_t nn = nv + (int32_t)n3;
    const int32_t nnp = std::max(nn, 1);
    DevBuf<int32_t> deg(nnp + 1, s), cursor(nnp, s);
    DevBuf<ull> in(nnp, s);
    LDS_CUDA(cudaMemsetAsync(deg.get(), 0, (nnp + 1) * sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(cursor.get(), 0, nnp * sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(in.get(), 0, nnp * sizeof(ull), s));
    if (np) LDS_LAUNCH(degree_kernel, grid_for(np, FB), FB, 0, s, pptr, pidx, np, f.get(), bigpos.get(), nv, deg.get(), in.get());
    DevBuf<int64_t> ptr(nnp + 1, s);
    const int64_t A = exclusive_scan_i32_to_i64(deg.get(), ptr.get(), nn + 1, s);
    DevBuf<int32_t> head(std::max<int64_t>(A, 1), s);
    DevBuf<int64_t> cap(std::max<int64_t>(A, 1), s), rev(std::max<int64_t>(A, 1), s);
    if (np)
        LDS_LAUNCH(fill_kernel, grid_for(np, FB), FB, 0, s, pptr, pidx, np, f.get(), bigpos.get(), nv, qK, ptr.get(),
                   cursor.get(), head.get(), cap.get(), rev.get());
    DevBuf<int64_t> tcap(std::max(nv, 1), s), excess(nnp, s);
    DevBuf<int32_t> height(nnp, s), inq(nnp, s);
    DevBuf<int32_t> la(nnp, s), lb(nnp, s), cnt(4, s), gcnt(3, s);
    DevBuf<ull> flow_t(1, s);
    LDS_CUDA(cudaMemsetAsync(inq.get(), 0, nnp * sizeof(int32_t), s));
    LDS_CUDA(cudaMemsetAsync(flow_t.get(), 0, sizeof(ull), s));
    Net net{nv, nn, ptr.get(), head.get(), cap.get(), rev.get(), tcap.get(), excess.get(), height.get()};
    if (nn) LDS_LAUNCH(init_kernel, grid_for(nn, FB), FB, 0, s, net, in.get(), pK, flow_t.get());

    int32_t tag = 0;
    // cnt: [0..2] work-list counts (triple-buffered), [3] relabels;
    // gcnt: [0..1] breadth-first frontier counts, [2] nodes with stuck excess
    auto global_relabel = [&]() -> std::pair<int32_t, int32_t> {
        LDS_CUDA(cudaMemsetAsync(gcnt.get(), 0, 3 * sizeof(int32_t), s));
        if (nn) LDS_LAUNCH(gr_init_kernel, grid_for(nn, FB), FB, 0, s, net, la.get(), gcnt.get());
        int32_t fsize = 0;
        LDS_CUDA(cudaMemcpyAsync(&fsize, gcnt.get(), sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        LDS_CUDA(cudaStreamSynchronize(s));
        int32_t* cur = la.get();
        int32_t* nxt = lb.get();
        int32_t* ccur = gcnt.get();
        int32_t* cnxt = gcnt.get() + 1;
        for (int32_t level = 1; fsize > 0; ++level) {
            LDS_REQUIRE(level <= nn + 1, LDS_ETIMEOUT, "max flow: global relabel did not finish");
            LDS_CUDA(cudaMemsetAsync(cnxt, 0, sizeof(int32_t), s));
            LDS_LAUNCH(gr_level_kernel, warps_grid(fsize), FB, 0, s, net, cur, ccur, level, nxt, cnxt);
            LDS_CUDA(cudaMemcpyAsync(&fsize, cnxt, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            LDS_CUDA(cudaStreamSynchronize(s));
            std::swap(cur, nxt);
            std::swap(ccur, cnxt);
        }
        // the work list goes to la with its count in cnt[0]
        LDS_CUDA(cudaMemsetAsync(cnt.get(), 0, 4 * sizeof(int32_t), s));
        LDS_CUDA(cudaMemsetAsync(gcnt.get() + 2, 0, sizeof(int32_t), s));
        ++tag;
        if (nn) LDS_LAUNCH(gr_finish_kernel, grid_for(nn, FB), FB, 0, s, net, la.get(), cnt.get(), inq.get(), tag, gcnt.get() + 2);
        int32_t h[2] = {0, 0};
        LDS_CUDA(cudaMemcpyAsync(&h[0], cnt.get(), sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        LDS_CUDA(cudaMemcpyAsync(&h[1], gcnt.get() + 2, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        LDS_CUDA(cudaStreamSynchronize(s));
        return {h[0], h[1]};
    };

    const int pulses = 8;
    const int batch = 8;
    const int64_t max_rounds = 64 * (int64_t)nn + 100000;
    const int round_grid = warps_grid(nn);
    int64_t rounds = 0;
    while (true) {
        const std::pair<int32_t, int32_t> gr = global_relabel();
        if (stop_if_short && gr.second > 0) return -1;
        if (gr.first == 0) break;
        // rounds until the list empties or enough relabels pile up for a new global relabel
        int32_t* lists[2] = {la.get(), lb.get()};
        for (int r = 0;;) {
            for (int b = 0; b < batch; ++b, ++r) {
                ++tag;
                LDS_LAUNCH(pr_round_kernel, round_grid, FB, 0, s, net, lists[r & 1], cnt.get() + (r % 3),
                           lists[(r + 1) & 1], cnt.get() + ((r + 1) % 3), cnt.get() + ((r + 2) % 3), inq.get(), tag,
                           pulses, flow_t.get(), cnt.get() + 3);
            }
            int32_t h[2];
            LDS_CUDA(cudaMemcpyAsync(&h[0], cnt.get() + (r % 3), sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            LDS_CUDA(cudaMemcpyAsync(&h[1], cnt.get() + 3, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            LDS_CUDA(cudaStreamSynchronize(s));
            rounds += batch;
            LDS_REQUIRE(rounds < max_rounds, LDS_ETIMEOUT, "max flow: push-relabel did not finish");
            if (h[0] == 0 || h[1] > nn) break;
        }
    }
    ull ft = 0;
    LDS_CUDA(cudaMemcpyAsync(&ft, flow_t.get(), sizeof(ull), cudaMemcpyDeviceToHost, s));
    if (side && nv) LDS_LAUNCH(side_kernel, grid_for(nv, FB), FB, 0, s, height.get(), nv, side);
    LDS_CUDA(cudaStreamSynchronize(s));
    // every cut of the network is a multiple of K
    LDS_REQUIRE((int64_t)ft % K == 0, LDS_ECUDA, "max flow: flow value %llu is not a multiple of the scale", ft);
    return (int64_t)ft / K;
}

}  // namespace lds

using namespace lds;

extern "C" lds_status lds_set_flow_variant(int32_t variant) {
    return guard([&] {
        LDS_REQUIRE(variant >= 0 && variant <= 2, LDS_EINVAL, "lds_set_flow_variant: %d is not 0, 1 or 2", variant);
        g_flow_variant.store(variant, std::memory_order_relaxed);
    });
}

extern "C" lds_status lds_pattern_max_flow(int32_t nv, int32_t np, const int64_t* pat_ptr, const int32_t* pat_idx,
                                           int64_t p, int64_t q, int64_t* flow, uint8_t* source_side) {
    return guard([&] {
        LDS_REQUIRE(nv >= 0 && np >= 0 && p >= 0 && q > 0, LDS_EINVAL, "lds_pattern_max_flow: bad sizes or capacities");
        LDS_REQUIRE(flow && (np == 0 || (pat_ptr && pat_idx)), LDS_EINVAL, "lds_pattern_max_flow: NULL argument");
        LDS_REQUIRE(lds_device_count() > 0, LDS_ECUDA, "lds_pattern_max_flow: no CUDA device");
        LDS_REQUIRE(np == 0 || pat_ptr[0] == 0, LDS_EINVAL, "lds_pattern_max_flow: pat_ptr[0] must be 0");
        for (int32_t j = 0; j < np; ++j)
            LDS_REQUIRE(pat_ptr[j + 1] >= pat_ptr[j], LDS_EINVAL, "lds_pattern_max_flow: pat_ptr not ascending");
        const int64_t k = np ? pat_ptr[np] : 0;
        for (int64_t i = 0; i < k; ++i)
            LDS_REQUIRE(pat_idx[i] >= 0 && pat_idx[i] < nv, LDS_EINVAL, "lds_pattern_max_flow: vertex index out of range");
        for (int32_t j = 0; j < np; ++j)
            for (int64_t a = pat_ptr[j]; a < pat_ptr[j + 1]; ++a)
                for (int64_t b = a + 1; b < pat_ptr[j + 1]; ++b)
                    LDS_REQUIRE(pat_idx[a] != pat_idx[b], LDS_EINVAL, "lds_pattern_max_flow: pattern %d repeats a vertex", j);
        cudaStream_t s = nullptr;
        DevBuf<int64_t> dp(np + 1, s);
        DevBuf<int32_t> di(std::max<int64_t>(k, 1), s);
        DevBuf<uint8_t> side(std::max(nv, 1), s);
        if (np) copy_in(dp.get(), pat_ptr, LDS_MEM_HOST, (np + 1) * sizeof(int64_t), s);
        else LDS_CUDA(cudaMemsetAsync(dp.get(), 0, sizeof(int64_t), s));
        if (k) copy_in(di.get(), pat_idx, LDS_MEM_HOST, k * sizeof(int32_t), s);
        *flow = pattern_max_flow(dp.get(), di.get(), np, nv, p, q, nullptr, side.get(), false, s);
        if (source_side && nv) {
            copy_out(source_side, LDS_MEM_HOST, side.get(), nv, s);
            LDS_CUDA(cudaStreamSynchronize(s));
        }
    });
}
