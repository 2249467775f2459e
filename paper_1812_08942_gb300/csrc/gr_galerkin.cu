// Galerkin reduced graph L_R = P^T L_G P (Sec. 3.2.2), assembled row by row.
//
// Coarse row A owns the CSR slots of its member nodes.  Each slot becomes the
// key (B << 32 | fine edge id) with B the aggregate of the slot's neighbour
// (slots of edges inside A become NOKEY), written into A's segment of a
// scratch array.  Sorting a segment groups equal B in ascending fine edge id,
// so summing each run in order gives w_R(A, B) exactly as the plain
// definition adds the crossing fine weights (ascending edge id), and the runs
// in order are A's coarse row with ascending neighbours -- the coarse CSR and
// the canonical coarse edge list come out directly, with no global sort.
//
// When no row has more than 32 slots (the first level of a mesh or grid), a
// row takes a thread: the block loads its rows' segments in whole lines into
// columns of shared memory, each thread sorts its column in registers by a
// merge network sized to the warp's longest row and adds up the runs in step
// with its warp (605k rows of 21 slots: 151 us; a warp per row 308, at 80 %
// issue).  Else segments are sorted by one warp each: up to 32 slots in
// registers, up to 128 in a small shared-memory buffer, up to 1,024 in a
// larger one (169k rows of 37 slots: 162 us; a thread each, with networks of
// up to 64 keys, 176).  A sorting network costs O(s log^2 s)
// per row, so graphs with longer rows use the global sort.
#include "gr_ieee.cuh"
#include "gr_internal.cuh"
#include "gr_vec.cuh"

namespace gr {

namespace {

constexpr int GT = 256;
constexpr int THREAD_P = 32;      // rows up to this many slots can take a thread each
constexpr int ROW_T = 128;        // rows and threads per block of that kernel
constexpr int SMALL_P = 128;      // rows up to this many slots: the small-row kernel, a warp each
constexpr int MEDIUM_P = 1024;    // up to this many: a warp with a 16 KB buffer
constexpr int MEDIUM_WARPS = 4;   // warps per block in the medium kernel
constexpr uint64_t NOKEY = ~0ull;

__device__ __forceinline__ int32_t key_col(uint64_t k) { return (int32_t)(k >> 32); }
__device__ __forceinline__ int32_t key_edge(uint64_t k) { return (int32_t)(uint32_t)k; }

// Coarse row as the row kernels leave it: entries [base, base + cnt) of the
// scratch, the last `up` of them with B > A
struct RowMeta {
    uint32_t base;
    int32_t cnt, up, pad;
};
__device__ __forceinline__ void store_row(int64_t A, int64_t base, int32_t U, int32_t up,
                                          RowMeta* __restrict__ meta, unsigned long long* __restrict__ packed) {
    RowMeta r;
    r.base = (uint32_t)base;
    r.cnt = U;
    r.up = up;
    r.pad = 0;
    meta[A] = r;
    packed[A] = ((unsigned long long)(uint32_t)U << 32) | (unsigned long long)(uint32_t)up;
}

// Slots per aggregate (2 m < 2^32), and each node's place in its aggregate's
// segment: the sum before its claim.  USED_BIT: a node without slots uses the
// label.
constexpr unsigned long long SLOT_MASK = 0xffffffffull, USED_BIT = 1ull << 32;
__global__ void k_gal_count(const int32_t* __restrict__ agg, const int64_t* __restrict__ rowptr, int64_t n,
                            int64_t nc, unsigned long long* __restrict__ cnt, uint32_t* __restrict__ place,
                            int32_t* __restrict__ bad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t a = agg[i];
    if (a < 0 || a >= nc) {
        *bad = 1;
        return;
    }
    const unsigned long long len = (unsigned long long)(rowptr[i + 1] - rowptr[i]);
    if (len) place[i] = (uint32_t)atomicAdd(&cnt[a], len);
    else atomicOr(&cnt[a], USED_BIT);
}

// slot counts for the scan; every label used; the longest row; rows past the
// small kernel listed.  flags: [0] bad label, [1] listed rows, [4..5] longest row
__global__ void __launch_bounds__(GT) k_gal_check(const unsigned long long* __restrict__ cnt, int64_t nc,
                                                  int64_t* __restrict__ scnt, int32_t* __restrict__ flags,
                                                  int32_t* __restrict__ med) {
    __shared__ unsigned long long smax;
    if (threadIdx.x == 0) smax = 0;
    __syncthreads();
    const int64_t A = (int64_t)blockIdx.x * GT + threadIdx.x;
    unsigned long long s = 0;
    if (A <= nc) {
        const unsigned long long c = A < nc ? cnt[A] : 0ull;
        s = c & SLOT_MASK;
        scnt[A] = (int64_t)s;
        if (A < nc && c == 0) flags[0] = 1;
    }
    const int32_t km = warp_slot(s > SMALL_P && s <= MEDIUM_P, flags + 1);
    if (km >= 0) med[km] = (int32_t)A;
    const uint32_t w = __reduce_max_sync(0xffffffffu, (uint32_t)s);
    if ((threadIdx.x & 31) == 0 && w) atomicMax(&smax, (unsigned long long)w);
    __syncthreads();
    if (threadIdx.x == 0 && smax) atomicMax((unsigned long long*)(flags + 4), smax);
}

// each fine node's slots into its aggregate's key segment; LPN lanes per node
template <int LPN>
__global__ void k_gal_scatter(const int32_t* __restrict__ agg, const int64_t* __restrict__ rowptr,
                              const int32_t* __restrict__ col, const int32_t* __restrict__ eid, int64_t n,
                              const int64_t* __restrict__ sptr, const uint32_t* __restrict__ place,
                              uint64_t* __restrict__ keys) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LPN;
    const int l = threadIdx.x % LPN;
    if (i >= n) return;
    const int32_t a = agg[i];
    const int64_t b0 = rowptr[i], len = rowptr[i + 1] - b0;
    if (len == 0) return;
    const int64_t off = sptr[a] + place[i];
    for (int64_t k = l; k < len; k += LPN) {
        const int64_t j = b0 + k;
        const int32_t B = __ldg(agg + col[j]);
        keys[off + k] = B == a ? NOKEY : (((uint64_t)(uint32_t)B << 32) | (uint64_t)(uint32_t)eid[j]);
    }
}

// Each fine node's slots into its aggregate's key segment, a warp per 32
// consecutive nodes: the warp runs over the nodes' slots -- one contiguous range -- a slot per
// lane, so the column and edge-id reads come in whole lines.  Ranges longer
// than SC_CAP slots are written by each node's own lane.
constexpr int SC_CAP = 1024;

__global__ void __launch_bounds__(GT) k_gal_scatter_warp(const int32_t* __restrict__ agg,
                                                         const int64_t* __restrict__ rowptr,
                                                         const int32_t* __restrict__ col,
                                                         const int32_t* __restrict__ eid, int64_t n,
                                                         const int64_t* __restrict__ sptr,
                                                         const uint32_t* __restrict__ place,
                                                         uint64_t* __restrict__ keys) {
    __shared__ uint8_t s_row[GT / 32][SC_CAP];
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t pw = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
    if (pw >= n) return;  // whole warp
    const int64_t p = pw + lane;
    const bool in = p < n;
    const int32_t a = in ? agg[p] : 0;
    const int64_t b0 = in ? rowptr[p] : 0;
    const int64_t len = in ? rowptr[p + 1] - b0 : 0;
    int64_t off = 0;
    if (len) off = sptr[a] + place[p];
    const int lv = (int)((n - pw < 32 ? n - pw : 32) - 1);
    const int64_t R0 = __shfl_sync(FULL, b0, 0);
    const int64_t R1 = __shfl_sync(FULL, b0 + len, lv);
    if (R1 - R0 > SC_CAP) {
        for (int64_t k = 0; k < len; ++k) {
            const int64_t j = b0 + k;
            const int32_t B = __ldg(agg + col[j]);
            keys[off + k] = B == a ? NOKEY : (((uint64_t)(uint32_t)B << 32) | (uint64_t)(uint32_t)eid[j]);
        }
        return;
    }
    uint8_t* S = s_row[wp];
    for (int64_t k = 0; k < len; ++k) S[b0 - R0 + k] = (uint8_t)lane;
    __syncwarp();
    const int ns = (int)(R1 - R0);
    for (int j0 = 0; j0 < ns; j0 += 32) {
        const int j = j0 + lane;
        const int r = j < ns ? S[j] : 0;
        const int32_t ar = __shfl_sync(FULL, a, r);
        const int64_t offr = __shfl_sync(FULL, off, r);
        const int64_t br = __shfl_sync(FULL, b0, r);
        if (j < ns) {
            const int64_t g = R0 + j;
            const int32_t B = __ldg(agg + col[g]);
            keys[offr + (g - br)] = B == ar ? NOKEY : (((uint64_t)(uint32_t)B << 32) | (uint64_t)(uint32_t)eid[g]);
        }
    }
}

// ascending bitonic sort of P (power of two, at least 64) keys in shared
// memory by one warp; the lanes take the stage's P / 2 compare-exchange
// pairs (t, t + j), t with bit j clear, so none idles
__device__ __forceinline__ void warp_bitonic(uint64_t* K, int P, int lane) {
    for (int k = 2; k <= P; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int p = lane; p < (P >> 1); p += 32) {
                const int t = ((p & ~(j - 1)) << 1) | (p & (j - 1));
                const int u = t | j;
                const uint64_t a = K[t], b = K[u];
                if ((a > b) == ((t & k) == 0)) {
                    K[t] = b;
                    K[u] = a;
                }
            }
            __syncwarp();
        }
}

__device__ __forceinline__ int next_pow2_dev(int x) { return x <= 1 ? 1 : 1 << (32 - __clz(x - 1)); }

// Runs of equal B in the sorted segment K[0, s) -> the coarse row of A, by one
// warp: weights gathered in parallel into Wt, each run summed in order by the
// lane holding its first slot.
__device__ __forceinline__ void warp_emit(const uint64_t* K, double* Wt, int s, int32_t A, int lane,
                                          const double* __restrict__ ew, int64_t base,
                                          int32_t* __restrict__ ucol, double* __restrict__ uw,
                                          RowMeta* __restrict__ meta, unsigned long long* __restrict__ packed) {
    int valid = 0;
    for (int b = 0; b < s; b += 32) {
        const int t = b + lane;
        const bool ok = t < s && K[t] != NOKEY;
        if (ok) Wt[t] = __ldg(ew + key_edge(K[t]));
        valid += __popc(__ballot_sync(0xffffffffu, ok));
    }
    __syncwarp();
    int run = 0, up = 0;
    for (int b = 0; b < valid; b += 32) {
        const int t = b + lane;
        const bool h = t < valid && (t == 0 || key_col(K[t]) != key_col(K[t - 1]));
        const unsigned bal = __ballot_sync(0xffffffffu, h);
        const bool hu = h && key_col(K[t]) > A;
        if (h) {
            const int32_t B = key_col(K[t]);
            double sum = Wt[t];
            for (int u = t + 1; u < valid && key_col(K[u]) == B; ++u) sum += Wt[u];
            const int64_t r = base + run + __popc(bal & ((1u << lane) - 1u));
            ucol[r] = B;
            uw[r] = sum;
        }
        run += __popc(bal);
        up += __popc(__ballot_sync(0xffffffffu, hu));
    }
    if (lane == 0) store_row(A, base, run, up, meta, packed);
}

// A row of at most 32 slots, one slot per lane, without shared memory: the
// lanes sort 32-bit keys (B << 5 | slot) -- runs of equal B come out
// contiguous -- then rank the slots of each run by fine edge id, and the
// run's first lane adds the run's weights in that order.  Needs B < 2^27.
__device__ __forceinline__ void row32(const uint64_t* __restrict__ keys, int64_t base, int s, int32_t A, int lane,
                                      const double* __restrict__ ew, int32_t* __restrict__ ucol,
                                      double* __restrict__ uw, RowMeta* __restrict__ meta,
                                      unsigned long long* __restrict__ packed) {
    constexpr unsigned FULL = 0xffffffffu;
    const uint64_t k = lane < s ? keys[base + lane] : NOKEY;
    const bool ok = k != NOKEY;
    const int32_t e = key_edge(k);
    const double w = ok ? __ldg(ew + e) : 0.0;
    uint32_t sk = ok ? (((uint32_t)key_col(k) << 5) | (uint32_t)lane) : 0xffffffffu;
#pragma unroll
    for (int kk = 2; kk <= 32; kk <<= 1)
#pragma unroll
        for (int j = kk >> 1; j > 0; j >>= 1) {
            const uint32_t o = __shfl_xor_sync(FULL, sk, j);
            const bool keep_min = ((lane & j) == 0) == ((lane & kk) == 0);
            sk = keep_min ? min(sk, o) : max(sk, o);
        }
    const bool v = sk != 0xffffffffu;
    const int src = (int)(sk & 31u);
    const int32_t B = (int32_t)(sk >> 5);
    const int32_t ee = __shfl_sync(FULL, e, src);
    const double ww = __shfl_sync(FULL, w, src);
    const int32_t Bp = __shfl_up_sync(FULL, B, 1);
    const bool head = v && (lane == 0 || Bp != B);
    const unsigned hb = __ballot_sync(FULL, head);
    const unsigned vb = __ballot_sync(FULL, v);
    // this lane's run [start, end): from the last head at or below it to the
    // next head or the first empty lane after it
    const int start = 31 - __clz(hb & (FULL >> (31 - lane)));
    const unsigned after = lane == 31 ? 0u : ((hb | ~vb) & (FULL << (lane + 1)));
    const int end = after ? __ffs(after) - 1 : 32;
    const int len = v ? end - start : 0;
    int R = len;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) R = max(R, __shfl_xor_sync(FULL, R, o));
    int rank = 0;
    for (int d = 1; d < R; ++d) {
        const int32_t eu_ = __shfl_up_sync(FULL, ee, d);
        const int32_t ed_ = __shfl_down_sync(FULL, ee, d);
        if (v && lane - d >= start && eu_ < ee) ++rank;
        if (v && lane + d < end && ed_ < ee) ++rank;
    }
    const unsigned runmask = v ? ((end == 32 ? FULL : ((1u << end) - 1u)) & ~((1u << start) - 1u)) : 0u;
    double sum = 0.0;
    for (int r = 0; r < R; ++r) {
        const unsigned pick = __ballot_sync(FULL, v && rank == r) & runmask;
        const double x = __shfl_sync(FULL, ww, pick ? __ffs(pick) - 1 : lane);
        if (head && r < len) sum = r == 0 ? x : sum + x;
    }
    const unsigned ub = __ballot_sync(FULL, head && B > A);
    if (head) {
        const int64_t r = base + __popc(hb & ((1u << lane) - 1u));
        ucol[r] = B;
        uw[r] = sum;
    }
    if (lane == 0) store_row(A, base, __popc(hb), __popc(ub), meta, packed);
}

// rows of at most SMALL_P slots, a warp each (all rows visited, longer ones skipped)
__global__ void __launch_bounds__(GT) k_gal_rows_small(int64_t nc, const int64_t* __restrict__ sptr,
                                                       const uint64_t* __restrict__ keys,
                                                       const double* __restrict__ ew, int32_t* __restrict__ ucol,
                                                       double* __restrict__ uw, RowMeta* __restrict__ meta,
                                                       unsigned long long* __restrict__ packed) {
    __shared__ uint64_t sk[GT / 32][SMALL_P];
    __shared__ double sw[GT / 32][SMALL_P];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t A = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (A >= nc) return;
    const int64_t base = sptr[A];
    const int s = (int)(sptr[A + 1] - base > SMALL_P ? SMALL_P + 1 : sptr[A + 1] - base);
    if (s > SMALL_P) return;
    if (s <= 32) {
        row32(keys, base, s, (int32_t)A, lane, ew, ucol, uw, meta, packed);
        return;
    }
    uint64_t* K = sk[w];
    const int P = next_pow2_dev(s);
    for (int t = lane; t < P; t += 32) K[t] = t < s ? keys[base + t] : NOKEY;
    __syncwarp();
    warp_bitonic(K, P, lane);
    warp_emit(K, sw[w], s, (int32_t)A, lane, ew, base, ucol, uw, meta, packed);
}

// Ascending sort of N numbers in a thread's registers: Batcher's odd-even
// merge network (Knuth, The Art of Computer Programming 3, 5.3.4), for N not a
// power of two the next one's without the comparators past N.
template <int N, int P = 1, int K = 1>
__device__ __forceinline__ void merge_network(uint64_t (&x)[N]) {
#pragma unroll
    for (int i = 0; i + K < N; ++i) {
        // comparators (i, i + K): i counted from K % P in groups of 2 K
        const int o = i - K % P;
        if (o >= 0 && o % (2 * K) < K && i / (2 * P) == (i + K) / (2 * P)) {
            const uint64_t a = x[i], b = x[i + K];
            const bool up = a <= b;
            x[i] = up ? a : b;
            x[i + K] = up ? b : a;
        }
    }
    // (stages by recursion: as nested loops they were not unrolled, and the
    // numbers went to local memory)
    if constexpr (K > 1) merge_network<N, P, K / 2>(x);
    else if constexpr (2 * P < N) merge_network<N, 2 * P, 2 * P>(x);
}

// Place of key i of row r: rows are columns, each line turned by its number,
// so that neither a row's consecutive keys nor a key number's consecutive
// rows share a bank (unturned, filling the columns took half of the kernel)
__device__ __forceinline__ int key_at(int i, int r) { return i * ROW_T + ((r + i) & (ROW_T - 1)); }

// Sort row r's first k <= N keys in registers
template <int N>
__device__ __forceinline__ void sort_column(uint64_t* K, int r, int k) {
    uint64_t x[N];
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = i < k ? K[key_at(i, r)] : NOKEY;
    merge_network<N>(x);
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < k) K[key_at(i, r)] = x[i];
}

// Rows of at most THREAD_P slots (all rows), a thread per row
__global__ void __launch_bounds__(ROW_T) k_gal_rows_thread(int64_t nc, const int64_t* __restrict__ sptr,
                                                           const uint64_t* __restrict__ keys,
                                                           const double* __restrict__ ew,
                                                           RowMeta* __restrict__ meta, int32_t* __restrict__ ucol,
                                                           double* __restrict__ uw,
                                                           unsigned long long* __restrict__ packed) {
    __shared__ uint64_t K[THREAD_P * ROW_T];
    __shared__ uint32_t off[ROW_T + 1];  // segment starts, from the block's first
    const int tid = threadIdx.x;
    const int64_t A0 = (int64_t)blockIdx.x * ROW_T, A = A0 + tid;
    const int64_t s0 = sptr[A0], b0 = sptr[A < nc ? A : nc], b1 = sptr[A + 1 < nc ? A + 1 : nc];
    const bool mine = A < nc;
    off[tid] = (uint32_t)(b0 - s0);
    if (tid == ROW_T - 1) off[ROW_T] = (uint32_t)(b1 - s0);
    __syncthreads();
    const uint32_t tot = off[ROW_T];
    for (uint32_t t0 = 0; t0 < tot; t0 += 4 * ROW_T) {
        uint64_t x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t t = t0 + u * ROW_T + tid;
            x[u] = t < tot ? __ldg(keys + s0 + t) : NOKEY;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t t = t0 + u * ROW_T + tid;
            int r = 0;  // the last row that starts at or before slot t
#pragma unroll
            for (int h = ROW_T / 2; h > 0; h >>= 1)
                if (off[r + h] <= t) r += h;
            if (t < tot) K[key_at((int)(t - off[r]), r)] = x[u];
        }
    }
    __syncthreads();
    // inner edges' slots (NOKEY) sort to the end, past which no run is opened
    const int k = mine ? (int)(b1 - b0) : 0;
    const int kmax = __reduce_max_sync(0xffffffffu, k);
    if (kmax <= 16) sort_column<16>(K, tid, k);
    else if (kmax <= 24) sort_column<24>(K, tid, k);
    else sort_column<THREAD_P>(K, tid, k);
    // the runs, kmax positions in step for the whole warp, four weights in flight
    int32_t B = -1, U = 0, up = 0;  // B: the open run's neighbour
    double sum = 0.0;
    auto emit = [&]() {
        ucol[b0 + U] = B;
        uw[b0 + U] = sum;
        up += B > (int32_t)A ? 1 : 0;
        ++U;
    };
#pragma unroll 1
    for (int t = 0; t < kmax; t += 4) {
        int32_t b[4];
        double w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            b[u] = -2;
            w[u] = 0.0;
            const uint64_t x = t + u < k ? K[key_at(t + u, tid)] : NOKEY;
            if (x != NOKEY) {
                b[u] = key_col(x);
                w[u] = __ldg(ew + key_edge(x));
            }
        }
        if (!__any_sync(0xffffffffu, b[0] >= 0)) break;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool same = b[u] == B;
            if (!same && B >= 0) emit();
            sum = same ? sum + w[u] : w[u];
            B = b[u];
        }
    }
    if (B >= 0) emit();
    if (mine) store_row(A, b0, U, up, meta, packed);
}

// listed rows of SMALL_P < s <= MEDIUM_P slots, a warp each, 16 KB of shared memory per warp
__global__ void __launch_bounds__(MEDIUM_WARPS * 32) k_gal_rows_medium(
    const int32_t* __restrict__ list, const int32_t* __restrict__ count, const int64_t* __restrict__ sptr,
    const uint64_t* __restrict__ keys, const double* __restrict__ ew, int32_t* __restrict__ ucol,
    double* __restrict__ uw, RowMeta* __restrict__ meta, unsigned long long* __restrict__ packed) {
    extern __shared__ uint64_t smem_med[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t* K = smem_med + (size_t)w * 2 * MEDIUM_P;
    double* Wt = reinterpret_cast<double*>(K + MEDIUM_P);
    const int total = *count;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < total;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t A = list[r];
        const int64_t base = sptr[A];
        const int s = (int)(sptr[A + 1] - base);
        const int P = next_pow2_dev(s);
        for (int t = lane; t < P; t += 32) K[t] = t < s ? keys[base + t] : NOKEY;
        __syncwarp();
        warp_bitonic(K, P, lane);
        warp_emit(K, Wt, s, A, lane, ew, base, ucol, uw, meta, packed);
        __syncwarp();
    }
}

// row pointers and edge-id bases from the scanned pairs; p[R] is raised by a
// row with more than ROW_PART_SHORT entries on a side of the diagonal
__global__ void k_gal_unpack(int64_t R, unsigned long long* p, int64_t* __restrict__ rowptr,
                             int64_t* __restrict__ eptr) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= R) return;
    const unsigned long long x = p[i];
    rowptr[i] = (int64_t)(x >> 32);
    eptr[i] = (int64_t)(x & 0xffffffffull);
    if (i + 1 == R) return;
    const unsigned long long d = p[i + 1] - x;  // (entries, entries past the row)
    const unsigned all = (unsigned)(d >> 32), up = (unsigned)d;
    if (up > ROW_PART_SHORT || all - up > ROW_PART_SHORT) p[R] = 1;
}

// D(A, A) of short rows, a thread per row: the weights in slot order
// (= ascending edge id), the plain definition's order.  Four loads in flight.
__global__ void __launch_bounds__(GT) k_gal_degree(int64_t nc, const RowMeta* __restrict__ meta,
                                                   const double* __restrict__ uw, double* __restrict__ deg) {
    const int64_t A = (int64_t)blockIdx.x * GT + threadIdx.x;
    if (A >= nc) return;
    const int4 m = __ldg(reinterpret_cast<const int4*>(meta) + A);
    const double* w = uw + (uint32_t)m.x;
    double s = 0.0;
    for (int32_t i = 0; i < m.y; i += 4) {
        double x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u < m.y) x[u] = __ldg(w + i + u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u < m.y) s += x[u];
    }
    deg[A] = s;
}

// Coarse CSR, row-scaled weights and canonical edge list from the rows; long
// rows (G = 32) also their degrees.
// Lower entries (B < A) take the id of edge (B, A): A's position among B's
// upper entries.
template <int G>
__global__ void k_gal_fill(int64_t nc, const RowMeta* __restrict__ meta, const int32_t* __restrict__ ucol,
                           const double* __restrict__ uw, double* __restrict__ deg, const int64_t* __restrict__ rowptr, const int64_t* __restrict__ eptr,
                           int32_t* __restrict__ col, int32_t* __restrict__ eid, double* __restrict__ wn64,
                           int2* __restrict__ cw32, int32_t* __restrict__ eu, int32_t* __restrict__ ev,
                           double* __restrict__ ew) {
    const int64_t A = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int l = threadIdx.x % G;
    if (A >= nc) return;
    const int4 mA = __ldg(reinterpret_cast<const int4*>(meta) + A);
    const uint32_t base = (uint32_t)mA.x;
    const int32_t U = mA.y, low = U - mA.z;
    const int64_t r0 = rowptr[A], e0 = eptr[A];
    double dA = 0.0;
    if constexpr (G == 32) {  // lane sums in slot order, combined by a fixed butterfly
        for (int32_t i = l; i < U; i += G) dA += uw[base + i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dA += __shfl_xor_sync(0xffffffffu, dA, o);
        if (l == 0) deg[A] = dA;
    } else {
        dA = deg[A];
    }
    const double inv = row_inverse(dA);
    for (int32_t i = l; i < U; i += G) {
        const int32_t B = ucol[base + i];
        const double w = uw[base + i];
        const double x = w * inv;
        col[r0 + i] = B;
        wn64[r0 + i] = x;
        cw32[r0 + i] = make_int2(B, __float_as_int(f64_to_f32(x)));
        int64_t e;
        if (i >= low) {
            e = e0 + (i - low);
            eu[e] = (int32_t)A;
            ev[e] = B;
            ew[e] = w;
        } else {
            const int4 mB = __ldg(reinterpret_cast<const int4*>(meta) + B);
            const int32_t* bc = ucol + (uint32_t)mB.x;
            const int32_t blow = mB.y - mB.z;
            int32_t lo = blow, hi = mB.y;  // A is among B's upper entries
            while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                if (bc[mid] < (int32_t)A) lo = mid + 1;
                else hi = mid;
            }
            e = eptr[B] + (lo - blow);
        }
        eid[r0 + i] = (int32_t)e;
    }
}

}  // namespace

gr_status galerkin_rows(gr_ctx* c, const int32_t* agg, int64_t nc, gr_ctx* cc, bool* too_long) {
    const int64_t n = c->n, m = c->m, slots = 2 * m;
    cudaStream_t s = c->stream;
    *too_long = false;
    int64_t* hs = host_scratch();
    if (!hs) return set_error(c, GR_ENOMEM, "coarsen: pinned scratch unavailable");

    // per-row arrays
    size_t need = 0;
    auto add = [&](size_t bytes) {
        size_t off = need;
        need += (bytes + 255) & ~size_t(255);
        return off;
    };
    const size_t R = (size_t)nc + 1;
    const size_t o_cnt = add(8 * R), o_flags = add(64), o_sptr = add(8 * R), o_place = add(4 * (size_t)n),
                 o_med = add(4 * R), o_meta = add(sizeof(RowMeta) * R), o_pack = add(8 * (R + 1));
    void* pr;
    GR_TRY_CUDA(c, c->ws.get(WS_GAL_ROWS, need, &pr), "coarsen scratch");
    char* Bp = (char*)pr;
    unsigned long long* cnt = (unsigned long long*)(Bp + o_cnt);
    int32_t* flags = (int32_t*)(Bp + o_flags);
    int64_t* sptr = (int64_t*)(Bp + o_sptr);
    uint32_t* place = (uint32_t*)(Bp + o_place);
    int32_t* med = (int32_t*)(Bp + o_med);
    RowMeta* meta = (RowMeta*)(Bp + o_meta);
    unsigned long long* packed = (unsigned long long*)(Bp + o_pack);
    // the counts and, right after them, the flags
    GR_TRY_CUDA(c, cudaMemsetAsync(cnt, 0, o_flags + 64 - o_cnt, s), "memset");
    if (n > 0) {
        k_gal_count<<<(unsigned)ceil_div(n, GT), GT, 0, s>>>(agg, c->rowptr, n, nc, cnt, place, flags);
        count_launch();
    }
    k_gal_check<<<(unsigned)ceil_div(nc + 1, GT), GT, 0, s>>>(cnt, nc, sptr, flags, med);
    count_launch();
    GR_TRY_CUDA(c, cudaMemcpyAsync(hs, flags, 32, cudaMemcpyDeviceToHost, s), "readback");
    GR_TRY_CUDA(c, scan_exclusive_i64(sptr, sptr, (int64_t)R, c->ws, s), "scan slots");
    GR_TRY_CUDA(c, cudaStreamSynchronize(s), "sync");
    const int32_t* hc = (const int32_t*)hs;
    if (hc[0]) return set_error(c, GR_EINVAL, "coarsen: labels must lie in [0, nc) and all be used");
    const int32_t nmed = hc[1];
    const unsigned long long smax = ((const unsigned long long*)hs)[2];
    // (the register path packs B into 27 bits)
    if (smax > (unsigned long long)MEDIUM_P || nc >= (int64_t(1) << 27)) {
        *too_long = true;
        return GR_OK;
    }

    void *pk, *pc, *pw;
    GR_TRY_CUDA(c, c->ws.get(WS_GAL_KEYS, sizeof(uint64_t) * (size_t)(slots > 0 ? slots : 1), &pk), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_GAL_UCOL, sizeof(int32_t) * (size_t)(slots > 0 ? slots : 1), &pc), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_GAL_UW, sizeof(double) * (size_t)(slots > 0 ? slots : 1), &pw), "ws");
    uint64_t* keys = (uint64_t*)pk;
    int32_t* ucol = (int32_t*)pc;
    double* uw = (double*)pw;

    if (slots > 0) {
        if (slots >= 32 * n) {
            k_gal_scatter<32><<<(unsigned)ceil_div(n * 32, GT), GT, 0, s>>>(agg, c->rowptr, c->col, c->eid, n, sptr,
                                                                           place, keys);
        } else {
            k_gal_scatter_warp<<<(unsigned)ceil_div(n, GT), GT, 0, s>>>(agg, c->rowptr, c->col, c->eid, n, sptr,
                                                                       place, keys);
        }
        count_launch();
    }
    if (smax <= THREAD_P)
        k_gal_rows_thread<<<(unsigned)ceil_div(nc, ROW_T), ROW_T, 0, s>>>(nc, sptr, keys, c->ew, meta, ucol, uw, packed);
    else
        k_gal_rows_small<<<(unsigned)ceil_div(nc * 32, GT), GT, 0, s>>>(nc, sptr, keys, c->ew, ucol, uw, meta, packed);
    count_launch();
    if (nmed > 0) {
        const size_t dyn = (size_t)MEDIUM_WARPS * 2 * MEDIUM_P * sizeof(uint64_t);
        GR_TRY_CUDA(c, cudaFuncSetAttribute(k_gal_rows_medium, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn),
                    "smem attribute");
        const int64_t want = ceil_div(nmed, MEDIUM_WARPS), cap = (int64_t)c->num_sms * 3;
        k_gal_rows_medium<<<(unsigned)(want < cap ? want : cap), MEDIUM_WARPS * 32, dyn, s>>>(
            med, flags + 1, sptr, keys, c->ew, ucol, uw, meta, packed);
        count_launch();
    }
    GR_TRY_CUDA(c, cudaGetLastError(), "galerkin rows");

    // coarse row pointers and edge-id bases: one scan of (entries, entries past the row)
    GR_TRY_CUDA(c, cudaMemsetAsync(packed + nc, 0, 16, s), "memset");
    GR_TRY_CUDA(c, scan_exclusive_i64((const int64_t*)packed, (int64_t*)packed, (int64_t)R, c->ws, s), "scan rows");
    SlabPlan rows;
    const size_t o_eptr = rows.add(sizeof(int64_t) * R), o_row = rows.add(sizeof(int64_t) * (R + CSR_PAD_ROWS)),
                 o_deg = rows.add(sizeof(double) * (size_t)(nc > 0 ? nc : 1));
    GR_TRY_CUDA(c, cudaMallocAsync(&cc->slab[0], rows.need, s), "alloc rows");
    char* b0 = (char*)cc->slab[0];
    cc->eptr = (int64_t*)(b0 + o_eptr);
    cc->rowptr = (int64_t*)(b0 + o_row);
    cc->deg = (double*)(b0 + o_deg);
    k_gal_unpack<<<(unsigned)ceil_div((int64_t)R, GT), GT, 0, s>>>((int64_t)R, packed, cc->rowptr, cc->eptr);
    count_launch();
    GR_TRY_CUDA(c, cudaMemcpyAsync(hs, packed + nc, 16, cudaMemcpyDeviceToHost, s), "readback");
    GR_TRY_CUDA(c, cudaStreamSynchronize(s), "sync");
    cc->parts = hs[1] ? 0 : 1;
    const int64_t mc = (int64_t)((uint64_t)hs[0] & 0xffffffffull);
    if ((int64_t)((uint64_t)hs[0] >> 32) != 2 * mc)
        return set_error(c, GR_ECUDA, "coarsen: coarse rows are not symmetric");
    cc->m = mc;
    const size_t cs = (size_t)(2 * mc > 0 ? 2 * mc : 1) + CSR_PAD_SLOTS, ce = (size_t)(mc > 0 ? mc : 1);
    SlabPlan ents;
    const size_t o_eu = ents.add(sizeof(int32_t) * ce), o_ev = ents.add(sizeof(int32_t) * ce),
                 o_ew = ents.add(sizeof(double) * ce), o_col = ents.add(sizeof(int32_t) * cs),
                 o_eid = ents.add(sizeof(int32_t) * cs), o_cw = ents.add(sizeof(int2) * cs),
                 o_wn = ents.add(sizeof(double) * cs);
    GR_TRY_CUDA(c, cudaMallocAsync(&cc->slab[1], ents.need, s), "alloc entries");
    char* b1 = (char*)cc->slab[1];
    cc->eu = (int32_t*)(b1 + o_eu);
    cc->ev = (int32_t*)(b1 + o_ev);
    cc->ew = (double*)(b1 + o_ew);
    cc->col = (int32_t*)(b1 + o_col);
    cc->eid = (int32_t*)(b1 + o_eid);
    cc->cw32 = (int2*)(b1 + o_cw);
    cc->wn64 = (double*)(b1 + o_wn);
    const int G = 2 * mc >= 32 * nc ? 32 : 4;
    const unsigned grid = (unsigned)ceil_div(nc * G, GT);
    if (G == 32) {
        k_gal_fill<32><<<grid, GT, 0, s>>>(nc, meta, ucol, uw, cc->deg, cc->rowptr, cc->eptr, cc->col, cc->eid,
                                           cc->wn64, cc->cw32, cc->eu, cc->ev, cc->ew);
    } else {
        k_gal_degree<<<(unsigned)ceil_div(nc, GT), GT, 0, s>>>(nc, meta, uw, cc->deg);
        count_launch();
        k_gal_fill<4><<<grid, GT, 0, s>>>(nc, meta, ucol, uw, cc->deg, cc->rowptr, cc->eptr, cc->col, cc->eid,
                                          cc->wn64, cc->cw32, cc->eu, cc->ev, cc->ew);
    }
    count_launch();
    GR_TRY_CUDA(c, cudaGetLastError(), "galerkin fill");
    return GR_OK;
}

}  // namespace gr
