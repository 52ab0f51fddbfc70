// Graph ingest: raw (src, dst) pairs -> canonical edge list and symmetric CSR
// on the device (the simple undirected G = (V, E) of Sec. 3).
//
// One stable radix sort of the 2m directed keys x << bits | y (self-loops mapped to a
// key above every real one) gives, after removing repeats, the symmetric CSR in
// row-major order; the slots with row < col, in order, are the canonical edges.  Flags
// are bit words and their scans run over words, row starts come from the key
// boundaries, and the host waits three times (distinct keys, vertices, the end).
#include "graph.cuh"
#include "prims.cuh"

namespace lds {

namespace {

// both directions of every pair as keys a << bits | b; self-loops and pairs with a bad id
// (counted apart) take the key above every real one
__global__ void directed_keys_kernel(const int32_t* src, const int32_t* dst, int64_t m, int32_t n, int bits,
                                     uint64_t loop_key, uint64_t* keys, unsigned long long* loops) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long local = 0, bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const int32_t a = src[i], b = dst[i];
        const bool ok = a >= 0 && a < n && b >= 0 && b < n;
        ulonglong2 k = make_ulonglong2(loop_key, loop_key);
        if (!ok) ++bad;
        else if (a == b) ++local;
        else k = make_ulonglong2(((uint64_t)a << bits) | (uint64_t)b, ((uint64_t)b << bits) | (uint64_t)a);
        reinterpret_cast<ulonglong2*>(keys)[i] = k;
    }
    if (local) atomicAdd(loops, local);
    if (bad) atomicAdd(loops + 1, bad);
}

// bit i of flag: key i is real and differs from the one before; cnt: set bits per word
__global__ void unique_flags_kernel(const uint64_t* keys, int64_t k, uint64_t loop_key, uint32_t* flag, int32_t* cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5, nw = (k + 31) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw; w += nwarps) {
        const int64_t i = (w << 5) + lane;
        const uint64_t x = i < k ? keys[i] : loop_key;
        uint64_t px = __shfl_up_sync(0xffffffffu, x, 1);
        if (lane == 0) px = i > 0 ? keys[i - 1] : loop_key;
        const unsigned b = __ballot_sync(0xffffffffu, x != loop_key && (i == 0 || px != x));
        if (lane == 0) {
            flag[w] = b;
            cnt[w] = __popc(b);
        }
    }
}

__global__ void compact_kernel(const uint64_t* keys, const uint32_t* flag, const int64_t* base, int64_t k, uint64_t* out) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += stride) {
        const uint32_t f = flag[i >> 5];
        const int l = (int)(i & 31);
        if ((f >> l) & 1u) out[base[i >> 5] + __popc(f & ((1u << l) - 1u))] = keys[i];
    }
}

// 1 + the first slot of every original vertex that has one (the rest stay 0)
__global__ void row_starts_kernel(const uint64_t* ukeys, int64_t k2, int bits, int64_t* start) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < k2; s += stride) {
        const int64_t x = (int64_t)(ukeys[s] >> bits);
        if (s == 0 || (int64_t)(ukeys[s - 1] >> bits) != x) start[x] = s + 1;
    }
}

__global__ void nonisolated_flag_kernel(const int64_t* start, int32_t n, int32_t* flag) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) flag[i] = start[i] > 0;
}

// id maps, and the row starts by internal id (isolated vertices have no slots)
__global__ void id_maps_kernel(const int64_t* start, const int64_t* nz_rank, int32_t n, int32_t nact, int64_t k2,
                               int32_t* to_int, int32_t* to_orig, int64_t* rowptr) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t b = start[i];
        const int32_t id = b > 0 ? (int32_t)nz_rank[i] : (int32_t)(nact + (i - nz_rank[i]));
        to_int[i] = id;
        to_orig[id] = (int32_t)i;
        if (b > 0) rowptr[id] = b - 1;
        if (i == 0) rowptr[nact] = k2;
    }
}

// columns; bit s of upper: slot s is its edge's canonical one (row < column); the last
// slot of each row gives the row's degree
__global__ void fill_csr_kernel(const uint64_t* ukeys, int64_t k2, int bits, const int32_t* to_int,
                                const int64_t* start, int32_t* col, uint32_t* upper, int32_t* cnt, int* maxdeg) {
    const uint64_t mask = (1ull << bits) - 1ull;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5, nw = (k2 + 31) >> 5;
    int dmax = 0;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw; w += nwarps) {
        const int64_t s = (w << 5) + lane;
        bool up = false;
        if (s < k2) {
            const uint64_t x = ukeys[s];
            if (s == k2 - 1 || (ukeys[s + 1] >> bits) != (x >> bits))
                dmax = max(dmax, (int)(s + 2 - start[(int64_t)(x >> bits)]));
            col[s] = to_int[(int64_t)(x & mask)];
            up = (x >> bits) < (x & mask);          // the map is monotone on these vertices
        }
        const unsigned b = __ballot_sync(0xffffffffu, up);
        if (lane == 0) {
            upper[w] = b;
            cnt[w] = __popc(b);
        }
    }
    dmax = __reduce_max_sync(0xffffffffu, dmax);
    if (lane == 0 && dmax > *maxdeg) atomicMax(maxdeg, dmax);
}

__global__ void canonical_edges_kernel(const uint64_t* ukeys, const int32_t* col, const uint32_t* upper,
                                       const int64_t* base, int64_t k2, int bits, const int32_t* to_int, int32_t* eu,
                                       int32_t* ev) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < k2; s += stride) {
        const uint32_t f = upper[s >> 5];
        const int l = (int)(s & 31);
        if (!((f >> l) & 1u)) continue;
        const int64_t e = base[s >> 5] + __popc(f & ((1u << l) - 1u));
        eu[e] = to_int[(int64_t)(ukeys[s] >> bits)];
        ev[e] = col[s];
    }
}

// symmetric FW view: columns with bit 31 on the first slot of each row, and the row of
// the first slot of each 32-slot chunk
__global__ void row_marks_kernel(const int64_t* rowptr, int32_t nact, int32_t* fwcol, int32_t* chunk_row0) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nact; r += stride) {
        int64_t b = rowptr[r], e = rowptr[r + 1];
        fwcol[b] |= (int32_t)0x80000000;
        // chunks whose first slot lies in [b, e)
        for (int64_t g = (b + 31) >> 5; (g << 5) < e; ++g) chunk_row0[g] = (int32_t)r;
    }
}

// upper neighbours of every row; the row lists its lower neighbours first, then its
// upper ones in canonical edge order
__global__ void upper_degree_kernel(const int64_t* rowptr, const int32_t* col, int32_t nact, int64_t* updeg) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nact; r += stride) {
        int64_t lo = rowptr[r], hi = rowptr[r + 1], e = hi;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (col[mid] <= r) lo = mid + 1; else hi = mid;
        }
        updeg[r] = e - lo;
    }
}

// the first upper slot of row x, rowptr[x + 1] - updeg[x], is canonical edge eptr[x]
__global__ void edge_shift_kernel(const int64_t* rowptr, const int64_t* updeg, const int64_t* eptr, int32_t nact,
                                  int64_t* shift) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nact; x += stride)
        shift[x] = eptr[x] - (rowptr[x + 1] - updeg[x]);
}

__global__ void map_ids_kernel(const int32_t* in, const int32_t* map, int64_t k, int32_t* out) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += stride) out[i] = map[in[i]];
}

template <class T>
__global__ void scatter_orig_kernel(const T* in, const int32_t* to_orig, int32_t n, T* out) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[to_orig[i]] = in[i];
}

}  // namespace

void map_ids(const int32_t* in, const int32_t* map, int64_t k, int32_t* out, cudaStream_t s) {
    if (k <= 0) return;
    LDS_LAUNCH(map_ids_kernel, grid_for(k, 256), 256, 0, s, in, map, k, out);
    LDS_CHECK_LAUNCH();
}

void ensure_symmetric_view(lds_graph* g) {
    if (g->fwcol.p || g->m == 0) return;
    cudaStream_t s = g->stream;
    const int64_t k2 = 2 * g->m;
    DevBuf<int32_t> c(k2, s);
    g->chunk_row0.alloc((k2 + 31) / 32, s);
    LDS_CUDA(cudaMemcpyAsync(c.get(), g->col.get(), k2 * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    LDS_LAUNCH(row_marks_kernel, grid_for(g->nact, 256), 256, 0, s, g->rowptr.get(), g->nact, c.get(), g->chunk_row0.get());
    g->fwcol = std::move(c);
}

void ensure_edge_shift(lds_graph* g) {
    if (g->edge_shift.p || g->m == 0) return;
    cudaStream_t s = g->stream;
    DevBuf<int64_t> updeg(g->nact, s), eptr(g->nact, s);
    LDS_LAUNCH(upper_degree_kernel, grid_for(g->nact, 256), 256, 0, s, g->rowptr.get(), g->col.get(), g->nact, updeg.get());
    exclusive_scan_i64_dev(updeg.get(), eptr.get(), g->nact, nullptr, s);
    g->edge_shift.alloc(g->nact, s);
    LDS_LAUNCH(edge_shift_kernel, grid_for(g->nact, 256), 256, 0, s, g->rowptr.get(), updeg.get(), eptr.get(), g->nact,
               g->edge_shift.get());
}

void to_original_order_i64(const lds_graph* g, const int64_t* in_int, int64_t* out_orig) {
    if (g->n <= 0) return;
    LDS_LAUNCH(scatter_orig_kernel<int64_t>, grid_for(g->n, 256), 256, 0, g->stream, in_int, g->to_orig.get(), g->n, out_orig);
    LDS_CHECK_LAUNCH();
}

void to_original_order_f64(const lds_graph* g, const double* in_int, double* out_orig) {
    if (g->n <= 0) return;
    LDS_LAUNCH(scatter_orig_kernel<double>, grid_for(g->n, 256), 256, 0, g->stream, in_int, g->to_orig.get(), g->n, out_orig);
    LDS_CHECK_LAUNCH();
}

static void build_graph(lds_graph* g, int32_t n, int64_t m_in, const int32_t* src, const int32_t* dst, lds_mem where) {
    cudaStream_t s = g->stream;
    g->n = n;
    g->info.n = n;
    g->info.input_pairs = m_in;
    g->info.triangles = -1;
    const int32_t* dsrc = src;
    const int32_t* ddst = dst;
    DevBuf<int32_t> hsrc, hdst;
    if (where == LDS_MEM_HOST && m_in > 0) {
        hsrc.alloc(m_in, s);
        hdst.alloc(m_in, s);
        copy_in(hsrc.get(), src, LDS_MEM_HOST, m_in * sizeof(int32_t), s);
        copy_in(hdst.get(), dst, LDS_MEM_HOST, m_in * sizeof(int32_t), s);
        dsrc = hsrc.get();
        ddst = hdst.get();
    }
    // ids fit in bits; the top key would be a self-loop, so it is no real key
    const int bits = n > 1 ? bit_length_u64((uint64_t)n - 1) : 1;
    const uint64_t loop_key = (1ull << (2 * bits)) - 1ull;
    const int64_t K = 2 * m_in, kw = (K + 31) / 32;

    DevBuf<uint64_t> keys(K, s);
    DevBuf<unsigned long long> loops(2, s);        // self-loops, pairs with a bad id
    LDS_CUDA(cudaMemsetAsync(loops.get(), 0, 2 * sizeof(unsigned long long), s));
    if (m_in > 0)
        LDS_LAUNCH(directed_keys_kernel, grid_for(m_in, 256), 256, 0, s, dsrc, ddst, m_in, n, bits, loop_key, keys.get(),
                   loops.get());
    hsrc.release();
    hdst.release();
    radix_sort_u64(keys.get(), nullptr, K, 2 * bits, s);

    DevBuf<uint32_t> flag(kw, s);
    DevBuf<int32_t> wcnt(kw, s);
    DevBuf<int64_t> base(kw, s);
    if (K > 0)
        LDS_LAUNCH(unique_flags_kernel, grid_for(K, 256), 256, 0, s, keys.get(), K, loop_key, flag.get(), wcnt.get());
    unsigned long long hloops[2] = {0, 0};
    LDS_CUDA(cudaMemcpyAsync(hloops, loops.get(), sizeof(hloops), cudaMemcpyDeviceToHost, s));
    const int64_t K2 = exclusive_scan_i32_to_i64(wcnt.get(), base.get(), kw, s);
    LDS_REQUIRE(hloops[1] == 0, LDS_EINVAL, "lds_create_graph: vertex id outside [0, %d)", n);
    LDS_REQUIRE(K2 % 2 == 0, LDS_ECUDA, "lds_create_graph: asymmetric key set (internal error)");
    g->m = K2 / 2;
    DevBuf<uint64_t> ukeys(K2, s);
    DevBuf<int64_t> start(n, s);
    LDS_CUDA(cudaMemsetAsync(start.get(), 0, (size_t)n * sizeof(int64_t), s));
    if (K2 > 0) {
        LDS_LAUNCH(compact_kernel, grid_for(K, 256), 256, 0, s, keys.get(), flag.get(), base.get(), K, ukeys.get());
        LDS_LAUNCH(row_starts_kernel, grid_for(K2, 256), 256, 0, s, ukeys.get(), K2, bits, start.get());
    }
    keys.release();

    // id maps
    DevBuf<int32_t> nzflag(n, s);
    DevBuf<int64_t> nzrank(n, s);
    if (n > 0) LDS_LAUNCH(nonisolated_flag_kernel, grid_for(n, 256), 256, 0, s, start.get(), n, nzflag.get());
    const int64_t nact = exclusive_scan_i32_to_i64(nzflag.get(), nzrank.get(), n, s);
    g->nact = (int32_t)nact;
    g->to_int.alloc(n, s);
    g->to_orig.alloc(n, s);
    g->rowptr.alloc(nact + 1, s);
    DevBuf<int> maxdeg(1, s);
    LDS_CUDA(cudaMemsetAsync(maxdeg.get(), 0, sizeof(int), s));
    if (n > 0)
        LDS_LAUNCH(id_maps_kernel, grid_for(n, 256), 256, 0, s, start.get(), nzrank.get(), n, g->nact, K2,
                   g->to_int.get(), g->to_orig.get(), g->rowptr.get());
    else
        LDS_CUDA(cudaMemsetAsync(g->rowptr.get(), 0, sizeof(int64_t), s));
    g->col.alloc(K2, s);
    g->eu.alloc(g->m, s);
    g->ev.alloc(g->m, s);
    if (K2 > 0) {
        LDS_LAUNCH(fill_csr_kernel, grid_for(K2, 256), 256, 0, s, ukeys.get(), K2, bits, g->to_int.get(), start.get(),
                   g->col.get(), flag.get(), wcnt.get(), maxdeg.get());
        exclusive_scan_i32_dev(wcnt.get(), base.get(), (K2 + 31) / 32, s);
        LDS_LAUNCH(canonical_edges_kernel, grid_for(K2, 256), 256, 0, s, ukeys.get(), g->col.get(), flag.get(), base.get(),
                   K2, bits, g->to_int.get(), g->eu.get(), g->ev.get());
    }
    int hmax = 0;
    LDS_CUDA(cudaMemcpyAsync(&hmax, maxdeg.get(), sizeof(int), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    g->info.m = g->m;
    g->info.self_loops = (int64_t)hloops[0];
    g->info.duplicates = m_in - (int64_t)hloops[0] - g->m;
    g->info.max_degree = hmax;
    g->info.isolated = n - g->nact;
}

void set_stream(lds_graph* g, cudaStream_t s) {
    g->stream = s;
    g->to_orig.s = s;
    g->to_int.s = s;
    g->eu.s = s;
    g->ev.s = s;
    g->rowptr.s = s;
    g->col.s = s;
    g->fwcol.s = s;
    g->chunk_row0.s = s;
    g->edge_shift.s = s;
    g->ta.s = s;
    g->tb.s = s;
    g->tc.s = s;
    g->vt_ptr.s = s;
    g->vt_idx.s = s;
    g->core_all[0].s = s;
    g->core_all[1].s = s;
    g->fwv_perm.s = s;
    g->fwv_pos.s = s;
    g->fwv_col.s = s;
    g->fwv_nzrow.s = s;
    g->fwv_chunk_nz0.s = s;
    g->fwv_edge.s = s;
    g->fwv_rowptr.s = s;
    g->tv_perm.s = s;
    g->tv_count.s = s;
    g->tv_c.s = s;
    g->tv_it.s = s;
    g->tv_chunk_g0.s = s;
    g->tv_grp.s = s;
    g->fwq_c.s = s;
    g->fwq_qs.s = s;
    g->fwq_src.s = s;
    g->fwq_qptr.s = s;
    g->fwq_eid.s = s;
    g->fw_R.s = s;
    g->fw_r.s = s;
    g->fw_W.s = s;
    g->fw_last.s = s;
}

}  // namespace lds

using namespace lds;

extern "C" {

lds_status lds_create_graph(int32_t n, int64_t m, const int32_t* src, const int32_t* dst, lds_mem where,
                            void* stream, lds_graph** out) {
    return guard([&] {
        LDS_REQUIRE(out != nullptr, LDS_EINVAL, "lds_create_graph: out is NULL");
        *out = nullptr;
        LDS_REQUIRE(n >= 0 && n <= 0x7ffffffe, LDS_EINVAL, "lds_create_graph: n = %d out of range", n);
        LDS_REQUIRE(m >= 0, LDS_EINVAL, "lds_create_graph: m = %lld < 0", (long long)m);
        LDS_REQUIRE(m == 0 || (src && dst), LDS_EINVAL, "lds_create_graph: src / dst is NULL");
        LDS_REQUIRE(where == LDS_MEM_HOST || where == LDS_MEM_DEVICE, LDS_EINVAL, "lds_create_graph: bad lds_mem");
        LDS_REQUIRE(lds_device_count() > 0, LDS_ECUDA, "lds_create_graph: no CUDA device");
        lds_graph* g = new lds_graph();
        g->stream = (cudaStream_t)stream;
        const int dev = g->device = handle_created();
        try {
            build_graph(g, n, m, src, dst, where);
        } catch (...) {
            delete g;
            handle_freed(dev);
            throw;
        }
        *out = g;
    });
}

void lds_free(lds_graph* g) {
    if (!g) return;
    const cudaStream_t s = g->stream;
    const int dev = g->device;
    cudaStreamSynchronize(s);
    delete g;
    cudaStreamSynchronize(s);          // its buffers are free now, and can be given back
    handle_freed(dev);
}

lds_status lds_graph_info(const lds_graph* g, lds_graph_info_t* info) {
    return guard([&] {
        LDS_REQUIRE(g && info, LDS_EINVAL, "lds_graph_info: NULL argument");
        *info = g->info;
        info->triangles = g->ntri;
    });
}

lds_status lds_get_edges(const lds_graph* g, int32_t* u, int32_t* v, lds_mem where) {
    return guard([&] {
        LDS_REQUIRE(g && u && v, LDS_EINVAL, "lds_get_edges: NULL argument");
        cudaStream_t s = g->stream;
        if (g->m == 0) return;
        DevBuf<int32_t> ou(g->m, s), ov(g->m, s);
        // internal -> original ids (monotone, so the order is kept)
        map_ids(g->eu.get(), g->to_orig.get(), g->m, ou.get(), s);
        map_ids(g->ev.get(), g->to_orig.get(), g->m, ov.get(), s);
        copy_out(u, where, ou.get(), g->m * sizeof(int32_t), s);
        copy_out(v, where, ov.get(), g->m * sizeof(int32_t), s);
        LDS_CUDA(cudaStreamSynchronize(s));
    });
}

}  // extern "C"

