// Exclusive scans and a stable LSD radix sort (see prims.cuh).
#include "prims.cuh"

namespace lds {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <class In>
__device__ __forceinline__ int64_t load_as_i64(const In* p, int64_t i, int64_t n) {
    return i < n ? (int64_t)p[i] : 0;
}

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ int64_t block_exclusive_scan(int64_t x, int64_t* excl) {
    constexpr int NW = SCAN_THREADS / 32;
    __shared__ int64_t warp_tot[NW];
    __shared__ int64_t block_total;
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < NW ? warp_tot[lane] : 0;
        int64_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < NW) warp_tot[lane] = wi - w;
        if (lane == NW - 1) block_total = wi;
    }
    __syncthreads();
    *excl = warp_tot[warp] + incl - x;
    int64_t t = block_total;
    __syncthreads();
    return t;
}

template <class In>
__global__ void scan_reduce_kernel(const In* in, int64_t n, int64_t* block_sums) {
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int64_t s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) s += load_as_i64(in, base + k, n);
    int64_t excl;
    int64_t tot = block_exclusive_scan(s, &excl);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = tot;
}

template <class In>
__global__ void scan_apply_kernel(const In* in, int64_t* out, int64_t n, const int64_t* block_offsets) {
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int64_t v[SCAN_ITEMS];
    int64_t s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        v[k] = load_as_i64(in, base + k, n);
        s += v[k];
    }
    int64_t excl;
    block_exclusive_scan(s, &excl);
    int64_t run = excl + (block_offsets ? block_offsets[blockIdx.x] : 0);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
}

// Short scans in one launch of one block, total included: a query makes hundreds of
// them, and the tiled form takes three launches each.  One block against tiles: 5.6 and
// 14.7 us for 100 items, 11.9 and 23.6 for 8,192, 18.0 and 25.0 for 16,384, 30.3 and
// 24.0 for 32,768.
constexpr int64_t SCAN_SHORT = 16384;
constexpr int SCAN_SHORT_T = 1024;
template <class In>
__global__ void __launch_bounds__(SCAN_SHORT_T) scan_short_kernel(const In* in, int64_t* out, int64_t n, int64_t* total) {
    __shared__ int64_t wtot[2][32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int64_t carry = 0;
    int round = 0;
    for (int64_t base = 0; base < n; base += SCAN_SHORT_T * SCAN_ITEMS, ++round) {
        const int64_t b = base + (int64_t)tid * SCAN_ITEMS;
        int64_t v[SCAN_ITEMS], s = 0;
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            v[k] = load_as_i64(in, b + k, n);
            s += v[k];
        }
        int64_t incl = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        int64_t* w = wtot[round & 1];
        if (lane == 31) w[wid] = incl;
        __syncthreads();
        // every warp sums the warp totals before it and in all
        int64_t t = w[lane], ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        int64_t run = carry + __shfl_sync(0xffffffffu, ti - t, wid) + incl - s;
        carry += __shfl_sync(0xffffffffu, ti, 31);
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            if (b + k < n) out[b + k] = run;
            run += v[k];
        }
    }
    if (total && tid == 0) *total = carry;
}

template <class In>
void scan_impl(const In* in, int64_t* out, int64_t n, int64_t* total_dev, cudaStream_t s) {
    if (n <= 0) {
        if (total_dev) LDS_CUDA(cudaMemsetAsync(total_dev, 0, sizeof(int64_t), s));
        return;
    }
    if (n <= SCAN_SHORT) {
        LDS_LAUNCH(scan_short_kernel<In>, 1, SCAN_SHORT_T, 0, s, in, out, n, total_dev);
        return;
    }
    int64_t nblocks = (n + SCAN_TILE - 1) / SCAN_TILE;
    DevBuf<int64_t> sums(nblocks, s);
    LDS_LAUNCH(scan_reduce_kernel<In>, (unsigned)nblocks, SCAN_THREADS, 0, s, in, n, sums.get());
    LDS_CHECK_LAUNCH();
    DevBuf<int64_t> offs(nblocks, s);
    scan_impl<int64_t>(sums.get(), offs.get(), nblocks, total_dev, s);
    LDS_LAUNCH(scan_apply_kernel<In>, (unsigned)nblocks, SCAN_THREADS, 0, s, in, out, n, offs.get());
    LDS_CHECK_LAUNCH();
}

}  // namespace

void exclusive_scan_i64_dev(const int64_t* in, int64_t* out, int64_t n, int64_t* total_dev,
                            cudaStream_t s) {
    scan_impl<int64_t>(in, out, n, total_dev, s);
}

int64_t exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s) {
    DevBuf<int64_t> tot(1, s);
    scan_impl<int64_t>(in, out, n, tot.get(), s);
    int64_t h = 0;
    LDS_CUDA(cudaMemcpyAsync(&h, tot.get(), sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    return h;
}

int64_t exclusive_scan_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, cudaStream_t s) {
    DevBuf<int64_t> tot(1, s);
    scan_impl<int32_t>(in, out, n, tot.get(), s);
    int64_t h = 0;
    LDS_CUDA(cudaMemcpyAsync(&h, tot.get(), sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    LDS_CUDA(cudaStreamSynchronize(s));
    return h;
}

void exclusive_scan_i32_dev(const int32_t* in, int64_t* out, int64_t n, cudaStream_t s) {
    scan_impl<int32_t>(in, out, n, nullptr, s);
}

// ------------------------------------------------------------------ radix sort

namespace {

// One pass: digit counts of every tile, their scan (digit-major), and the scatter.  The
// scatter is bound by its latencies and by the sectors it writes: a thread takes all its
// keys in one go, a warp ranks its share by itself, and the tile is put in digit order in
// shared memory first, so that a tile's keys of one digit (16 to 32 on average) go out as
// one run of neighbouring lanes.  Keys per thread: as many as fit 64 registers (two
// blocks a multiprocessor) without spills to speak of.  Measured with 8, 12 and 16:
//   60M 64-bit keys with payload, 18 bits: 1.87, 2.22, 2.11 ms (4.46 in rounds of 256
//   keys with three barriers each and no reordering); 32-bit keys: 1.64, 1.60, 1.48 ms;
//   36M 64-bit keys, 40 bits: 1.90, 1.78, 1.81 ms (2.76).
constexpr int RS_THREADS = 512;
constexpr int RS_WARPS = RS_THREADS / 32;
template <class Key, bool VALS>
constexpr int RS_ROUNDS = sizeof(Key) == 4 ? 16 : VALS ? 8 : 12;
template <class Key, bool VALS>
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS<Key, VALS>;

template <class Key, bool VALS>
__global__ void __launch_bounds__(RS_THREADS) rs_histogram_kernel(const Key* keys, int64_t n, int shift, int64_t ntiles,
                                                                  int32_t* counts) {
    __shared__ uint32_t h[256];
    if (threadIdx.x < 256) h[threadIdx.x] = 0;
    __syncthreads();
    constexpr int ROUNDS = RS_ROUNDS<Key, VALS>, TILE = RS_TILE<Key, VALS>;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    if (base + TILE <= n) {
        Key k[ROUNDS];
#pragma unroll
        for (int j = 0; j < ROUNDS; ++j) k[j] = keys[base + j * RS_THREADS + threadIdx.x];
#pragma unroll
        for (int j = 0; j < ROUNDS; ++j) atomicAdd(&h[(k[j] >> shift) & 0xFF], 1u);
    } else {
        for (int64_t i = base + threadIdx.x; i < n; i += RS_THREADS) atomicAdd(&h[(keys[i] >> shift) & 0xFF], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 256) counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = (int32_t)h[threadIdx.x];
}

template <class Key, bool VALS>
constexpr size_t rs_scatter_smem() {
    return (size_t)RS_TILE<Key, VALS> * (sizeof(Key) + (VALS ? sizeof(uint32_t) : 0)) + RS_WARPS * 256 * sizeof(uint16_t);
}

template <class Key, bool VALS>
__global__ void __launch_bounds__(RS_THREADS, 2) rs_scatter_kernel(const Key* __restrict__ keys_in,
                                                                   const uint32_t* __restrict__ vals_in, Key* keys_out,
                                                                   uint32_t* vals_out, int64_t n, int shift, int64_t ntiles,
                                                                   const int64_t* offsets) {
    constexpr int ROUNDS = RS_ROUNDS<Key, VALS>, TILE = RS_TILE<Key, VALS>;
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ int64_t goff[256];
    __shared__ uint32_t dstart[256], wsum[8];
    Key* sk = reinterpret_cast<Key*>(rsm);
    uint32_t* sv = reinterpret_cast<uint32_t*>(sk + TILE);
    uint16_t* wcnt = reinterpret_cast<uint16_t*>(sv + (VALS ? TILE : 0));      // [RS_WARPS][256]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    const int cnt = (int)min((int64_t)TILE, n - base);
    const int first = warp * (32 * ROUNDS) + lane;
    Key k[ROUNDS];
#pragma unroll
    for (int j = 0; j < ROUNDS; ++j) k[j] = first + 32 * j < cnt ? keys_in[base + first + 32 * j] : Key(0);
    int64_t off = 0;
    if (t < 256) off = offsets[(int64_t)t * ntiles + blockIdx.x];
    for (int i = t; i < RS_WARPS * 128; i += RS_THREADS) reinterpret_cast<uint32_t*>(wcnt)[i] = 0;
    __syncthreads();
    uint16_t* mine = wcnt + warp * 256;
    uint32_t rk[ROUNDS / 2];                      // two ranks a word
#pragma unroll
    for (int j = 0; j < ROUNDS; ++j) {
        const int d = first + 32 * j < cnt ? (int)((k[j] >> shift) & 0xFF) : 256;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = d < 256 ? mine[d] : 0;
        __syncwarp();
        if (d < 256 && (peers & lt) == 0) mine[d] = (uint16_t)(before + __popc(peers));
        __syncwarp();
        const uint32_t r = before + __popc(peers & lt);
        if (j & 1) rk[j / 2] |= r << 16;
        else rk[j / 2] = r;
    }
    __syncthreads();
    uint32_t run = 0, incl = 0;
    if (t < 256) {
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) {
            const uint32_t c = wcnt[w * 256 + t];
            wcnt[w * 256 + t] = (uint16_t)run;
            run += c;
        }
        incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
    }
    __syncthreads();
    if (t < 256) {
        uint32_t st = incl - run;
        for (int w = 0; w < warp; ++w) st += wsum[w];
        dstart[t] = st;
        goff[t] = off - st;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ROUNDS; ++j) {
        if (first + 32 * j < cnt) {
            const int d = (int)((k[j] >> shift) & 0xFF);
            const uint32_t pos = dstart[d] + mine[d] + ((rk[j / 2] >> (16 * (j & 1))) & 0xFFFFu);
            sk[pos] = k[j];
            if (VALS) sv[pos] = vals_in[base + first + 32 * j];
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = t; i < cnt; i += RS_THREADS) {
        const Key x = sk[i];
        const int64_t at = goff[(int)((x >> shift) & 0xFF)] + i;
        keys_out[at] = x;
        if (VALS) vals_out[at] = sv[i];
    }
}

// The whole sort of at most RS_SMALL keys in one block and one launch: keys (and
// payload) ping-pong in shared memory.  A warp owns a contiguous segment and ranks it
// 32 keys at a time (lanes of equal digit by match), counting per warp and digit; one
// scan over (digit, warp) then places every key, so each pass is stable and takes four
// block barriers.  The tiled form takes three to five launches a pass: 36-bit keys take
// 34 us here and 138 us there for 4,096 of them, 57 and 148 us for 8,192, which is what
// shared memory holds.
constexpr int RS_SMALL = 8192;
constexpr int RS_SMALL_T = 1024;
constexpr int RS_SMALL_ROUNDS = RS_SMALL / RS_SMALL_T;
template <class Key, bool VALS>
__global__ void __launch_bounds__(RS_SMALL_T, 1) rs_small_kernel(Key* keys, uint32_t* vals, int n, int passes) {
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ uint32_t dtot[256], wsum[8];
    Key* ka = reinterpret_cast<Key*>(rsm);
    Key* kb = ka + n;
    uint32_t* va = reinterpret_cast<uint32_t*>(kb + n);
    uint32_t* vb = va + (VALS ? n : 0);
    uint16_t* wcnt = reinterpret_cast<uint16_t*>(vb + (VALS ? n : 0));        // [32][256]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const int seg = ((n + RS_SMALL_T - 1) / RS_SMALL_T) * 32, first = wid * seg;
    for (int i = tid; i < n; i += RS_SMALL_T) {
        ka[i] = keys[i];
        if (VALS) va[i] = vals[i];
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        for (int i = tid; i < 32 * 128; i += RS_SMALL_T) reinterpret_cast<uint32_t*>(wcnt)[i] = 0;
        __syncthreads();
        uint16_t rk[RS_SMALL_ROUNDS];
        uint16_t* mine = wcnt + wid * 256;
#pragma unroll
        for (int r = 0; r < RS_SMALL_ROUNDS; ++r) {
            if (r * 32 >= seg) break;
            const int i = first + r * 32 + lane;
            const int d = i < n ? (int)((ka[i] >> shift) & 0xFF) : 256;
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            const uint32_t base = d < 256 ? mine[d] : 0;
            __syncwarp();
            if (d < 256 && (peers & lt) == 0) mine[d] = (uint16_t)(base + __popc(peers));
            __syncwarp();
            rk[r] = (uint16_t)(base + __popc(peers & lt));
        }
        __syncthreads();
        if (tid < 256) {
            uint32_t run = 0;
            for (int w = 0; w < 32; ++w) {
                const uint32_t t = wcnt[w * 256 + tid];
                wcnt[w * 256 + tid] = (uint16_t)run;
                run += t;
            }
            uint32_t incl = run;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) wsum[wid] = incl;
            dtot[tid] = incl - run;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RS_SMALL_ROUNDS; ++r) {
            if (r * 32 >= seg) break;
            const int i = first + r * 32 + lane;
            if (i < n) {
                const Key k = ka[i];
                const int d = (int)((k >> shift) & 0xFF);
                uint32_t pos = dtot[d] + mine[d] + rk[r];
                for (int w = 0; w < (d >> 5); ++w) pos += wsum[w];
                kb[pos] = k;
                if (VALS) vb[pos] = va[i];
            }
        }
        __syncthreads();
        Key* tk = ka;
        ka = kb;
        kb = tk;
        uint32_t* tv = va;
        va = vb;
        vb = tv;
    }
    for (int i = tid; i < n; i += RS_SMALL_T) {
        keys[i] = ka[i];
        if (VALS) vals[i] = va[i];
    }
}

}  // namespace

template <class Key, bool VALS>
static void radix_sort(Key* keys, uint32_t* vals, int64_t n, int bits, cudaStream_t s) {
    if (n <= 1 || bits <= 0) return;
    const int passes = (bits + 7) / 8;
    if (n <= RS_SMALL) {
        constexpr size_t per = 2 * (sizeof(Key) + (VALS ? sizeof(uint32_t) : 0)), fixed = 32 * 256 * sizeof(uint16_t);
        LDS_CUDA(cudaFuncSetAttribute(rs_small_kernel<Key, VALS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(RS_SMALL * per + fixed)));
        auto kernel = rs_small_kernel<Key, VALS>;
        LDS_LAUNCH(kernel, 1, RS_SMALL_T, (size_t)n * per + fixed, s, keys, vals, (int)n, passes);
        return;
    }
    const int64_t ntiles = (n + RS_TILE<Key, VALS> - 1) / RS_TILE<Key, VALS>;
    constexpr size_t smem = rs_scatter_smem<Key, VALS>();
    auto histogram = rs_histogram_kernel<Key, VALS>;
    auto scatter = rs_scatter_kernel<Key, VALS>;
    LDS_CUDA(cudaFuncSetAttribute(scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    DevBuf<Key> kbuf(n, s);
    DevBuf<uint32_t> vbuf;
    if (VALS) vbuf.alloc(n, s);
    DevBuf<int32_t> counts(256 * ntiles, s);
    DevBuf<int64_t> offs(256 * ntiles, s);
    Key* kin = keys;
    Key* kout = kbuf.get();
    uint32_t* vin = vals;
    uint32_t* vout = VALS ? vbuf.get() : nullptr;
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        LDS_LAUNCH(histogram, (unsigned)ntiles, RS_THREADS, 0, s, kin, n, shift, ntiles, counts.get());
        exclusive_scan_i32_dev(counts.get(), offs.get(), 256 * ntiles, s);
        LDS_LAUNCH(scatter, (unsigned)ntiles, RS_THREADS, smem, s, kin, vin, kout, vout, n, shift, ntiles, offs.get());
        std::swap(kin, kout);
        std::swap(vin, vout);
    }
    if (kin != keys) {
        LDS_CUDA(cudaMemcpyAsync(keys, kin, n * sizeof(Key), cudaMemcpyDeviceToDevice, s));
        if (VALS) LDS_CUDA(cudaMemcpyAsync(vals, vin, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    }
}

void radix_sort_u64(uint64_t* keys, uint32_t* vals, int64_t n, int bits, cudaStream_t s) {
    if (vals) radix_sort<uint64_t, true>(keys, vals, n, bits, s);
    else radix_sort<uint64_t, false>(keys, nullptr, n, bits, s);
}

void radix_sort_u32(uint32_t* keys, uint32_t* vals, int64_t n, int bits, cudaStream_t s) {
    radix_sort<uint32_t, true>(keys, vals, n, bits, s);
}

}  // namespace lds
