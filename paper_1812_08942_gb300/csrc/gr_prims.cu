// Device primitives: stream-ordered workspace, exclusive scan, stable LSD
// radix sort of (key, value) pairs.  Used by CSR construction, aggregation
// and Galerkin coarsening.
#include <atomic>

#include "gr_internal.cuh"

namespace gr {

static std::atomic<uint64_t> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
uint64_t launch_count() { return g_launches.load(std::memory_order_relaxed); }

// ---------------------------------------------------------------------------
// Workspace
// ---------------------------------------------------------------------------
cudaError_t Workspace::get(int slot, size_t bytes, void** out) {
    if ((int)slots.size() <= slot) slots.resize(slot + 1);
    Slot& s = slots[slot];
    if (bytes == 0) bytes = 16;
    if (s.bytes < bytes) {
        if (s.ptr) {
            cudaError_t e = cudaFreeAsync(s.ptr, stream);
            s.ptr = nullptr;
            s.bytes = 0;
            if (e != cudaSuccess) return e;
        }
        size_t want = bytes + bytes / 4;
        want = (want + 255) & ~size_t(255);
        cudaError_t e = cudaMallocAsync(&s.ptr, want, stream);
        if (e != cudaSuccess) {
            s.ptr = nullptr;
            return e;
        }
        s.bytes = want;
    }
    *out = s.ptr;
    return cudaSuccess;
}

void Workspace::release() {
    for (Slot& s : slots)
        if (s.ptr) cudaFreeAsync(s.ptr, stream);
    slots.clear();
}

int64_t* host_scratch() {
    static thread_local int64_t* buf = nullptr;
    if (!buf && cudaMallocHost(&buf, 64) != cudaSuccess) buf = nullptr;
    return buf;
}

void tune_mempool(int device) {
    static bool done[64] = {false};
    if (device < 0 || device >= 64 || done[device]) return;
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, device) == cudaSuccess) {
        uint64_t thr = ~0ull;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    done[device] = true;
}

int bits_for(uint64_t v) {
    int b = 1;
    while (b < 64 && (v >> b) != 0) ++b;
    return b;
}

// ---------------------------------------------------------------------------
// Exclusive scan.  Up to SCAN_ONE entries: one block, tile by tile with a
// carry.  More: tile sums, which the last block to finish scans, then the
// tiles with their offsets.  The level loop scans a few dozen times; tile
// sums, their scan and the tiles in three launches took 9 us even for a
// thousand entries (each waits for the one before), one block takes 3.6; over
// the reduction of the 128^3 mesh 148 us of scans became 83.
// ---------------------------------------------------------------------------
constexpr int SCAN_THREADS = 512;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
constexpr int64_t SCAN_ONE = 2 * SCAN_TILE;
// place of entry i of a tile in shared memory: a gap per thread's SCAN_ITEMS
// consecutive entries (without it 16 lanes' 8-byte entries shared a bank)
constexpr int SCAN_PAD_TILE = SCAN_TILE + SCAN_TILE / SCAN_ITEMS;
__device__ __forceinline__ int scan_at(int i) { return i + i / SCAN_ITEMS; }

template <typename T>
__device__ T block_exclusive_scan(T x, T* warp_tot, T* block_total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        T t = lane < nw ? warp_tot[lane] : T(0);
        T ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        if (lane < nw) warp_tot[lane] = ti - t;
        if (lane == 31) *block_total = ti;
    }
    __syncthreads();
    T r = warp_tot[warp] + inc - x;
    return r;
}

// exclusive scan of one tile of `in` plus `carry` into `out` (out may be in);
// returns the tile's total
template <typename T>
__device__ T scan_tile(const T* in, T* out, int64_t base, int64_t count, T carry, T* tile, T* warp_tot, T* total) {
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int64_t idx = base + (int64_t)i * SCAN_THREADS + threadIdx.x;
        tile[scan_at(i * SCAN_THREADS + threadIdx.x)] = idx < count ? in[idx] : T(0);
    }
    __syncthreads();
    T loc[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        loc[i] = s;
        s += tile[scan_at(threadIdx.x * SCAN_ITEMS + i)];
    }
    T ex = block_exclusive_scan<T>(s, warp_tot, total) + carry;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) tile[scan_at(threadIdx.x * SCAN_ITEMS + i)] = ex + loc[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int64_t idx = base + (int64_t)i * SCAN_THREADS + threadIdx.x;
        if (idx < count) out[idx] = tile[scan_at(i * SCAN_THREADS + threadIdx.x)];
    }
    return *total;
}

// one block, tile by tile
template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_one(const T* in, T* out, int64_t count) {
    __shared__ T tile[SCAN_PAD_TILE];
    __shared__ T warp_tot[SCAN_THREADS / 32];
    __shared__ T total;
    T carry = 0;
    for (int64_t base = 0; base < count; base += SCAN_TILE) {
        carry += scan_tile<T>(in, out, base, count, carry, tile, warp_tot, &total);
        __syncthreads();
    }
}

// tile sums; the last block turns them into the tiles' offsets (ticket: zero
// before and after)
template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(const T* in, int64_t count, T* bsum, unsigned* ticket) {
    __shared__ T red[SCAN_THREADS / 32];
    __shared__ T total;
    __shared__ bool last;
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    T s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int64_t idx = base + (int64_t)i * SCAN_THREADS + threadIdx.x;
        if (idx < count) s += in[idx];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        T t = 0;
        for (int w = 0; w < SCAN_THREADS / 32; ++w) t += red[w];
        bsum[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int64_t nb = gridDim.x;
    T carry = 0;
    for (int64_t b = 0; b < nb; b += SCAN_THREADS) {
        const int64_t idx = b + threadIdx.x;
        const T x = idx < nb ? __ldcg(bsum + idx) : T(0);
        const T ex = block_exclusive_scan<T>(x, red, &total);
        if (idx < nb) bsum[idx] = ex + carry;
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_apply(const T* in, T* out, int64_t count, const T* bsum) {
    __shared__ T tile[SCAN_PAD_TILE];
    __shared__ T warp_tot[SCAN_THREADS / 32];
    __shared__ T total;
    scan_tile<T>(in, out, (int64_t)blockIdx.x * SCAN_TILE, count, bsum[blockIdx.x], tile, warp_tot, &total);
}

template <typename T>
static cudaError_t scan_exclusive(const T* in, T* out, int64_t count, Workspace& ws,
                                  cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    if (count <= SCAN_ONE) {
        k_scan_one<T><<<1, SCAN_THREADS, 0, s>>>(in, out, count); count_launch();
        return cudaGetLastError();
    }
    int64_t nb = ceil_div(count, SCAN_TILE);
    void *p = nullptr, *pt = nullptr;
    GR_CUDA(ws.get(WS_SCAN, sizeof(T) * (size_t)nb, &p));
    const bool fresh = (int)ws.slots.size() <= WS_SCAN_TICKET || !ws.slots[WS_SCAN_TICKET].ptr;
    GR_CUDA(ws.get(WS_SCAN_TICKET, 16, &pt));
    if (fresh) GR_CUDA(cudaMemsetAsync(pt, 0, 16, s));
    T* bsum = (T*)p;
    k_scan_reduce<T><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, count, bsum, (unsigned*)pt); count_launch();
    k_scan_apply<T><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, out, count, bsum); count_launch();
    return cudaGetLastError();
}

cudaError_t scan_exclusive_i64(const int64_t* in, int64_t* out, int64_t count, Workspace& ws,
                               cudaStream_t s) {
    return scan_exclusive<int64_t>(in, out, count, ws, s);
}
cudaError_t scan_exclusive_i32(const int32_t* in, int32_t* out, int64_t count, Workspace& ws,
                               cudaStream_t s) {
    return scan_exclusive<int32_t>(in, out, count, ws, s);
}

// ---------------------------------------------------------------------------
// Stable LSD radix sort of (key, value) pairs.  Per pass: per-tile digit
// histogram, one exclusive scan over the digit-major histogram, then a stable
// scatter.  A pass moves every pair once whatever its digit's width, so the
// key is cut into the fewest digits of up to 10 bits (8 at least), and a block
// takes 8,192 pairs: a digit's run in the output is then 16 pairs at 9 bits.
// Every warp ranks its keys chunk by chunk (warp order = input order); keys
// equal in a digit find each other with one vote per bit.  The block places
// its keys, then their values, in shared memory in (digit, input) order and
// writes them out in whole runs.  Shared memory holds first the warps' 16-bit
// digit counts (two digits are added as one word), then the tile.
// Bound by the phases of a block (two blocks an SM), not by memory: 16 M pairs
// of 64-bit keys take 100 us a scatter where 384 MB would take 57.  Measured
// against tiles of 2,048 pairs and 8-bit digits with __match_any_sync:
// 16 M 64-bit keys of 34 bits 584 us (881 before), 32-bit keys of 19 bits
// 264 (465); 100,000 keys 95 (121) and 54 (66); 9,001 keys 84 (91) and 39 (48).
// ---------------------------------------------------------------------------
constexpr int SORT_THREADS = 512;
constexpr int SORT_WARPS = SORT_THREADS / 32;
constexpr int SORT_ITEMS = 16;
constexpr int SORT_TILE = SORT_THREADS * SORT_ITEMS;
static_assert(SORT_TILE < 65536, "positions in a tile are 16-bit");

template <typename KT>
__global__ void __launch_bounds__(SORT_THREADS) k_radix_hist(const KT* __restrict__ keys, int64_t count,
                                                             int shift, int bits, int32_t* __restrict__ hist,
                                                             int nb) {
    __shared__ int32_t cnt[1024];
    const int R = 1 << bits;
    for (int d = threadIdx.x; d < R; d += SORT_THREADS) cnt[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * SORT_TILE + threadIdx.x;
    const int left = count - base > SORT_TILE ? SORT_TILE : (int)(count - base);
    KT k[SORT_ITEMS];
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i) k[i] = i * SORT_THREADS < left ? __ldg(keys + base + i * SORT_THREADS) : 0;
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i)
        if (i * SORT_THREADS < left) atomicAdd(&cnt[(int)(k[i] >> shift) & (R - 1)], 1);
    __syncthreads();
    for (int d = threadIdx.x; d < R; d += SORT_THREADS) hist[(int64_t)d * nb + blockIdx.x] = cnt[d];
}

template <typename KT, int BITS>
constexpr size_t scatter_smem() {
    const size_t counts = (size_t)SORT_WARPS * (1u << BITS) * 2, tile = (size_t)SORT_TILE * sizeof(KT);
    return counts > tile ? counts : tile;
}

template <typename KT, int BITS>
__global__ void __launch_bounds__(SORT_THREADS, 2) k_radix_scatter(
    const KT* __restrict__ keys, const uint32_t* __restrict__ vals, int64_t count, int shift,
    const int32_t* __restrict__ offs, int nb, KT* __restrict__ keys_out, uint32_t* __restrict__ vals_out) {
    constexpr int R = 1 << BITS;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int32_t delta[R];  // a digit's output position minus its position in the tile
    __shared__ int32_t wsum[SORT_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t tbase = (int64_t)blockIdx.x * SORT_TILE;
    const int total = count - tbase > SORT_TILE ? SORT_TILE : (int)(count - tbase);
    const int w0 = warp * 32 * SORT_ITEMS + lane;
    uint16_t* whist = reinterpret_cast<uint16_t*>(smem) + warp * R;
    KT k[SORT_ITEMS];
    uint32_t rnk[SORT_ITEMS / 2];  // two 16-bit ranks, then positions, a word
    // past the end: the highest digit, after every key of that digit
#pragma unroll
    for (int c = 0; c < SORT_ITEMS; ++c) k[c] = w0 + c * 32 < total ? __ldg(keys + tbase + w0 + c * 32) : ~(KT)0;
    for (int d = lane; d < R / 2; d += 32) reinterpret_cast<uint32_t*>(whist)[d] = 0;
    __syncwarp();
#pragma unroll
    for (int c = 0; c < SORT_ITEMS; ++c) {
        const unsigned dg = (unsigned)(k[c] >> shift) & (R - 1);
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < BITS; ++b) {
            const unsigned bit = (dg >> b) & 1u;
            peers &= __ballot_sync(0xffffffffu, bit) ^ (bit - 1u);
        }
        const int before = whist[dg];
        const uint32_t r = (uint32_t)(before + __popc(peers & lt_mask));
        if (c & 1) rnk[c / 2] |= r << 16;
        else rnk[c / 2] = r;
        __syncwarp();
        if ((peers & lt_mask) == 0) whist[dg] = (uint16_t)(before + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    // two digits per thread: the warps' bases within each digit, its count
    uint32_t* W2 = reinterpret_cast<uint32_t*>(smem);
    uint32_t tot = 0;
    if (tid < R / 2) {
        for (int w = 0; w < SORT_WARPS; ++w) {
            const uint32_t x = W2[w * (R / 2) + tid];
            W2[w * (R / 2) + tid] = tot;
            tot += x;
        }
    }
    const int32_t t0 = (int32_t)(tot & 0xffffu), t1 = (int32_t)(tot >> 16);
    int32_t incl = t0 + t1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (tid < R / 2) {
        int32_t start = incl - t0 - t1;
        for (int w = 0; w < warp; ++w) start += wsum[w];
        const uint32_t pair = (uint32_t)start | ((uint32_t)(start + t0) << 16);
        for (int w = 0; w < SORT_WARPS; ++w) W2[w * (R / 2) + tid] += pair;
        delta[2 * tid] = offs[(int64_t)(2 * tid) * nb + blockIdx.x] - start;
        delta[2 * tid + 1] = offs[(int64_t)(2 * tid + 1) * nb + blockIdx.x] - (start + t0);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < SORT_ITEMS; ++c)
        rnk[c / 2] += (uint32_t)whist[(unsigned)(k[c] >> shift) & (R - 1)] << (c & 1 ? 16 : 0);
    __syncthreads();
    KT* skey = reinterpret_cast<KT*>(smem);
    uint32_t* sval = reinterpret_cast<uint32_t*>(smem);
#pragma unroll
    for (int c = 0; c < SORT_ITEMS; ++c) skey[(rnk[c / 2] >> (c & 1 ? 16 : 0)) & 0xffffu] = k[c];
    uint32_t v[SORT_ITEMS];
#pragma unroll
    for (int c = 0; c < SORT_ITEMS; ++c)
        v[c] = !vals ? (uint32_t)(tbase + w0 + c * 32)
                     : w0 + c * 32 < total ? __ldg(vals + tbase + w0 + c * 32) : 0u;
    __syncthreads();
    int32_t g[SORT_ITEMS];
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i) {
        const int j = tid + i * SORT_THREADS;
        const KT key = skey[j];
        g[i] = delta[(unsigned)(key >> shift) & (R - 1)] + j;
        if (j < total) keys_out[g[i]] = key;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < SORT_ITEMS; ++c) sval[(rnk[c / 2] >> (c & 1 ? 16 : 0)) & 0xffffu] = v[c];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i) {
        const int j = tid + i * SORT_THREADS;
        if (j < total) vals_out[g[i]] = sval[j];
    }
}

template <typename KT, int BITS>
static cudaError_t radix_scatter(const KT* keys, const uint32_t* vals, int64_t count, int shift,
                                 const int32_t* offs, int nb, KT* keys_out, uint32_t* vals_out, cudaStream_t s) {
    constexpr size_t smem = scatter_smem<KT, BITS>();
    GR_CUDA(cudaFuncSetAttribute(k_radix_scatter<KT, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    k_radix_scatter<KT, BITS><<<nb, SORT_THREADS, smem, s>>>(keys, vals, count, shift, offs, nb, keys_out,
                                                             vals_out);
    count_launch();
    return cudaGetLastError();
}

// in, vin: the input (keys and vals themselves, or other arrays, which stay as
// they are; vin null: the values are the positions)
template <typename KT>
static cudaError_t radix_sort(const KT* in, const uint32_t* vin, KT* keys, uint32_t* vals, KT* keys_alt,
                              uint32_t* vals_alt, int64_t count, int bits, Workspace& ws, cudaStream_t s, int* result_in_alt) {
    *result_in_alt = 0;
    if (count <= 0 || bits <= 0) return cudaSuccess;
    const int passes = (bits + 9) / 10;
    const int width = (bits + passes - 1) / passes < 8 ? 8 : (bits + passes - 1) / passes;
    const int nb = (int)ceil_div(count, SORT_TILE);
    void* p = nullptr;
    GR_CUDA(ws.get(WS_SORT_HIST, (sizeof(int32_t) << width) * (size_t)nb, &p));
    int32_t* hist = (int32_t*)p;
    const KT* ki = in;
    const uint32_t* vi = vin;
    KT* ko = keys_alt;
    uint32_t* vo = vals_alt;
    for (int i = 0; i < passes; ++i) {
        const int shift = i * width;
        k_radix_hist<KT><<<nb, SORT_THREADS, 0, s>>>(ki, count, shift, width, hist, nb); count_launch();
        GR_CUDA(scan_exclusive_i32(hist, hist, (int64_t)nb << width, ws, s));
        const cudaError_t e =
            width == 8 ? radix_scatter<KT, 8>(ki, vi, count, shift, hist, nb, ko, vo, s)
            : width == 9 ? radix_scatter<KT, 9>(ki, vi, count, shift, hist, nb, ko, vo, s)
                         : radix_scatter<KT, 10>(ki, vi, count, shift, hist, nb, ko, vo, s);
        if (e != cudaSuccess) return e;
        ki = ko;
        vi = vo;
        ko = ko == keys ? keys_alt : keys;
        vo = vo == vals ? vals_alt : vals;
    }
    *result_in_alt = passes & 1;
    return cudaSuccess;
}

cudaError_t radix_sort_u32(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt,
                           uint32_t* vals_alt, int64_t count, int bits, Workspace& ws,
                           cudaStream_t s, int* result_in_alt) {
    return radix_sort<uint32_t>(keys, vals, keys, vals, keys_alt, vals_alt, count, bits, ws, s, result_in_alt);
}
cudaError_t radix_sort_u64(uint64_t* keys, uint32_t* vals, uint64_t* keys_alt,
                           uint32_t* vals_alt, int64_t count, int bits, Workspace& ws,
                           cudaStream_t s, int* result_in_alt) {
    return radix_sort<uint64_t>(keys, vals, keys, vals, keys_alt, vals_alt, count, bits, ws, s, result_in_alt);
}
cudaError_t radix_order_u32(const uint32_t* in, uint32_t* keys, uint32_t* vals, uint32_t* keys_alt,
                            uint32_t* vals_alt, int64_t count, int bits, Workspace& ws,
                            cudaStream_t s, int* result_in_alt) {
    return radix_sort<uint32_t>(in, nullptr, keys, vals, keys_alt, vals_alt, count, bits, ws, s, result_in_alt);
}
cudaError_t radix_order_u64(const uint64_t* in, uint64_t* keys, uint32_t* vals, uint64_t* keys_alt,
                            uint32_t* vals_alt, int64_t count, int bits, Workspace& ws,
                            cudaStream_t s, int* result_in_alt) {
    return radix_sort<uint64_t>(in, nullptr, keys, vals, keys_alt, vals_alt, count, bits, ws, s, result_in_alt);
}

}  // namespace gr
