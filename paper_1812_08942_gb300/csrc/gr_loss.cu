// Spectral-mismatch loss on a reduced graph with free edge weights w_c, and
// its hand-written adjoint (reverse sweeps).  Not in the paper: it turns the
// edge-weight sensitivity of Sec. 3.3.3 (d lambda / d w = -lambda (e^T u)^2)
// into the exact gradient of a smooth objective built from the weighted
// Jacobi filter of Alg. 3 on the reduced graph.
//
//   R_f[k]  = x_k^T L_G x_k / x_k^T x_k
//   y_0     = M^-1 P^T X                            (aggregate means)
//   y_{s+1} = (1-w) y_s + w D_c^-1 A_c y_s          (isolated node: unchanged)
//   R_c[k]  = y^T L_c y / sum_A M_A (y_A - mu_k)^2,  mu_k = sum M y / sum M
//   loss    = (1/K) sum_k (R_c[k]/R_f[k] - 1)^2
// Vectors are FP32.  A sum over all rows or edges runs in FP32 over some 64
// terms a lane, those blocks and a warp's lanes are added in FP32, the rest in
// FP64, in a fixed order: a lane's error stays that of a few dozen additions
// whatever the size of the graph and the length of its rows.
//
// Layout.  Every pass over vectors is a pass over rows in which G = K / 4
// lanes hold one row, a 16-byte chunk each (short rows: 32 / G rows a warp),
// or a warp holds one row, its sub-groups taking slots in turn (long rows).
// Sums over edges take the edges in blocks of 64 instead where a row may be
// long (parts_short): a row pass left a hub of 1,000,000 edges to one lane's
// chain (231 ms and a relative error of 5e-4 of R_f, K = 8; by edges 0.4 ms and 3e-8).
// A thread per entry or per edge, reading K scalars 4 bytes at a time, took
// 17 us for a sweep of the 32,768-node reduced mesh (K = 24) and 200 us for
// the fine quotients of the 128^3 mesh.  The weights are put in slot order
// once per call, so that a sweep reads them with the columns instead of
// through the edge ids.  Column sums end in the kernel that makes them (last
// block); one-block kernels adding 304 rows of partials took 49 us each,
// eight per loss and gradient.  Loss and gradient of the 128^3 mesh (K = 24,
// aggregates of about 64 nodes, 5 sweeps): 1,505 us before, 522 now, of which the fine
// pass takes 139.
#include "gr_loss.cuh"
#include "gr_sweep.cuh"
#include "gr_vec.cuh"

namespace gr {

namespace {

constexpr int LT = 256;
constexpr int LW = LT / 32;
// Blocks per SM of the row passes, which is also their grid: a larger grid
// would leave its later blocks to a second wave over rows that have left L2
// (the fine pass read 427 MB for 301 in 181 us).  Loss and gradient with four,
// five and six: 555, 540 and 527 us.
constexpr int ROW_BLOCKS = 6;

// lanes of a warp over rows and 16-byte chunks of a row
template <int K, bool LONG>
struct RowLanes {
    static constexpr int G = K / 4, GP = next_pow2_c(G);
    static constexpr int RPW = LONG ? 1 : 32 / G;   // rows per warp
    static constexpr int TS = LONG ? 32 / GP : 1;   // sub-groups sharing a row's slots
    int seg, q, t;
    bool ok;
    __device__ RowLanes() {
        const int lane = threadIdx.x & 31;
        seg = LONG ? 0 : lane / G;
        q = LONG ? lane % GP : lane % G;
        t = LONG ? lane / GP : 0;
        ok = LONG ? q < G : seg < RPW;
    }
    __device__ bool writes() const { return ok && t == 0; }
};

__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void st4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }

struct NoStep {
    __device__ void operator()() const {}
};
// f(w, x) for every slot of the lane's share of [b, e): x the chunk of the
// slot's column in src; eight slots in flight (a reduced mesh's row of 14 in
// two round trips), in slot order per lane; step() after each round of eight
template <int K, bool LONG, typename F, typename Step = NoStep>
__device__ __forceinline__ void for_slots(const RowLanes<K, LONG>& m, int64_t b, int64_t e,
                                          const int2* __restrict__ cw, const float* __restrict__ src, F f,
                                          Step step = Step()) {
    constexpr int U = 8, TS = RowLanes<K, LONG>::TS;
    if (!m.ok) return;
    for (int64_t j = b + m.t; j < e; j += U * TS) {
        int2 v[U];
        float4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j + u * TS < e) v[u] = __ldg(cw + j + u * TS);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j + u * TS < e) x[u] = ld4(src + (int64_t)v[u].x * K + m.q * 4);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j + u * TS < e) f(__int_as_float(v[u].y), x[u]);
        step();
    }
}

// sum over a long row's sub-groups (every lane of the warp calls it)
template <int K, bool LONG>
__device__ __forceinline__ void join_row(float4& a) {
    if constexpr (LONG) {
#pragma unroll
        for (int o = RowLanes<K, true>::GP; o < 32; o <<= 1) {
            a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
            a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
            a.z += __shfl_xor_sync(0xffffffffu, a.z, o);
            a.w += __shfl_xor_sync(0xffffffffu, a.w, o);
        }
    }
}

// Column sums of a lane, by blocks of SUM_BLOCK terms or a little more.  The
// closed blocks' sums are in shared memory, an entry per thread: in registers
// they cost the fine pass 68 bytes of spills, and loss and gradient of the
// 128^3 mesh 540 us against 522 (518 in one chain).
constexpr unsigned SUM_BLOCK = 64;
struct LaneSum {
    float4 open;
    float4* closed;
    __device__ explicit LaneSum(float4* shared) : open(make_float4(0.f, 0.f, 0.f, 0.f)), closed(shared + threadIdx.x) {
        if (shared) *closed = open;  // (none: not used)
    }
    __device__ __forceinline__ void close() {
        *closed = total();
        open = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ float4 total() const {
        const float4 c = *closed;
        return make_float4(c.x + open.x, c.y + open.y, c.z + open.z, c.w + open.w);
    }
};
struct LaneSums {
    LaneSum a, b;
    unsigned terms;
    __device__ explicit LaneSums(float4 (*shared)[LT]) : a(shared[0]), b(shared[1]), terms(0) {}
    __device__ __forceinline__ void close() {
        a.close();
        b.close();
        terms = 0;
    }
    // t more terms have been added
    __device__ __forceinline__ void count(unsigned t) {
        terms += t;
        if (terms >= SUM_BLOCK) close();
    }
};

// Two column sums per lane (chunks s1, s2) into the block's partial row:
// lanes of one chunk added in FP32, warps in FP64.  COUNT: the first sum of s2
// is the whole numbers `cnt` of the warp's lanes.  True in the last block,
// with the totals in red (K of s1, then K of s2).
template <int K, bool LONG, bool COUNT = false>
__device__ bool finish_cols(const RowLanes<K, LONG>& m, float4 s1, float4 s2, double* part, unsigned* counter,
                            double* red, unsigned cnt = 0) {
    using L = RowLanes<K, LONG>;
    __shared__ double ws[LW][2 * K];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float a[8] = {s1.x, s1.y, s1.z, s1.w, s2.x, s2.y, s2.z, s2.w};
    constexpr int STEP = LONG ? L::GP : L::G, CNT = LONG ? L::TS : L::RPW;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float t = m.ok ? a[i] : 0.f;
        float acc = t;
#pragma unroll
        for (int r = 1; r < CNT; ++r) acc += __shfl_sync(0xffffffffu, t, (lane + r * STEP) & 31);
        a[i] = acc;
    }
    if (lane < L::G) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ws[warp][lane * 4 + i] = (double)a[i];
            ws[warp][K + lane * 4 + i] = (double)a[4 + i];
        }
    }
    if constexpr (COUNT) {
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) ws[warp][K] = (double)cnt;
    }
    __syncthreads();
    if (threadIdx.x < 2 * K) {
        double t = 0.0;
        for (int w = 0; w < LW; ++w) t += ws[w][threadIdx.x];
        part[(int64_t)blockIdx.x * 2 * K + threadIdx.x] = t;
    }
    __threadfence();
    __syncthreads();
    return finish_partials<K, LT>(part, gridDim.x, counter, red);
}

__device__ __forceinline__ void add_squares(float4& s, const float4& x) {
    s.x = fmaf(x.x, x.x, s.x);
    s.y = fmaf(x.y, x.y, s.y);
    s.z = fmaf(x.z, x.z, s.z);
    s.w = fmaf(x.w, x.w, s.w);
}
// s += w (x - y)^2
__device__ __forceinline__ void add_edge(float4& s, float w, const float4& x, const float4& y) {
    float t = x.x - y.x;
    s.x = fmaf(w * t, t, s.x);
    t = x.y - y.y;
    s.y = fmaf(w * t, t, s.y);
    t = x.z - y.z;
    s.z = fmaf(w * t, t, s.z);
    t = x.w - y.w;
    s.w = fmaf(w * t, t, s.w);
}

// S.a += w(e) (x_u - x_v)^2 over the canonical list: a warp takes SUM_BLOCK R
// consecutive edges at a time, each of its R lane groups every R-th of them,
// EDGE_FLIGHT in flight (a block of consecutive edges per group, whose loads lie 64
// edges apart: forward pass without sweeps on 16 M edges of a power-law graph,
// 8 columns, 690 us; so 515).  The first end's chunk is loaded again only
// where the node changes.  Xq: the lane's chunk of row 0.
constexpr int EDGE_FLIGHT = 4;
template <int R, typename Wt>
__device__ __forceinline__ void edge_blocks(int64_t m, int64_t warp, int64_t warps, int group,
                                            const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                                            const float* __restrict__ Xq, int K, LaneSums& S, Wt weight) {
    constexpr unsigned U = EDGE_FLIGHT;
    static_assert(SUM_BLOCK % U == 0, "a block is whole rounds");
    // shorter blocks where there are too few edges for all warps (m < 2^31)
    unsigned per = (unsigned)((m + warps * R - 1) / (unsigned)(warps * R));
    per = (per + U - 1) / U * U;
    const int64_t STEP = (int64_t)(per < SUM_BLOCK ? per : SUM_BLOCK) * R;
    for (int64_t b = warp * STEP; b < m; b += warps * STEP) {
        const int64_t e = b + STEP < m ? b + STEP : m;
        int32_t cur = -1;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int64_t j = b + group; j < e; j += (int64_t)U * R) {
            int32_t p[U], q[U];
            float w[U];
            float4 y[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j + u * R < e) {
                    p[u] = __ldg(eu + j + u * R);
                    q[u] = __ldg(ev + j + u * R);
                    w[u] = weight(j + u * R);
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j + u * R < e) y[u] = ld4(Xq + (int64_t)q[u] * K);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j + u * R < e) {
                    if (p[u] != cur) x = ld4(Xq + (int64_t)(cur = p[u]) * K);
                    add_edge(S.a.open, w[u], x, y[u]);
                }
        }
        S.close();
    }
}

// R_f: per column sum_e w (x_u - x_v)^2 over the edges (p, v) of row p and
// sum_p x_p^2, in one pass over the rows.
template <int K, bool LONG>
__global__ void __launch_bounds__(LT, ROW_BLOCKS) k_fine_quotients(int64_t n, const int64_t* __restrict__ eptr,
                                                       const int32_t* __restrict__ ev, const double* __restrict__ ew,
                                                       const float* __restrict__ X, double* part, unsigned* counter,
                                                       float* __restrict__ Rf) {
    __shared__ double red[LT];
    const RowLanes<K, LONG> m;
    constexpr int U = 2, TS = RowLanes<K, LONG>::TS, RPW = RowLanes<K, LONG>::RPW;
    __shared__ float4 closed[2][LT];
    LaneSums S(closed);  // numerator, denominator
    // 32-bit row and edge numbers (n, m < 2^31) keep the kernel at 4 blocks per SM or more
    const unsigned rows = (unsigned)n, stride = ((gridDim.x * LT) >> 5) * RPW;
    unsigned p = ((blockIdx.x * LT + threadIdx.x) >> 5) * RPW + m.seg;
    if (!m.ok) p = rows;
    unsigned b1 = 0, e1 = 0;  // the next row's edges, read one row ahead
    if (p < rows) {
        b1 = (unsigned)__ldg(eptr + p);
        e1 = (unsigned)__ldg(eptr + p + 1);
    }
    const float* Xq = X + m.q * 4;
    while (p < rows) {
        const unsigned b = b1, e = e1;
        const float4 x = ld4(Xq + (size_t)p * K);
        p += stride;
        if (p < rows) {
            b1 = (unsigned)__ldg(eptr + p);
            e1 = (unsigned)__ldg(eptr + p + 1);
            if (m.q == 0 && m.t == 0 && b1 < e1) {
                // the next row's edges into L1: no register waits for them
                asm volatile("prefetch.global.L1 [%0];" ::"l"(ev + b1));
                asm volatile("prefetch.global.L1 [%0];" ::"l"(ew + b1));
            }
        }
        if (m.t == 0) add_squares(S.b.open, x);
        for (unsigned j = b + m.t; j < e; j += U * TS) {
            float w[U];
            float4 y[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j + u * TS < e) {
                    y[u] = ld4(Xq + (size_t)__ldg(ev + j + u * TS) * K);
                    w[u] = f64_to_f32(__ldg(ew + j + u * TS));
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j + u * TS < e) add_edge(S.a.open, w[u], x, y[u]);
        }
        S.count(e - b + 1);
    }
    if (finish_cols<K, LONG>(m, S.a.total(), S.b.total(), part, counter, red) && threadIdx.x < K)
        Rf[threadIdx.x] = (float)(red[threadIdx.x] / red[K + threadIdx.x]);
}

// The same with the edges in blocks for graphs that may have long rows
template <int K>
__global__ void __launch_bounds__(LT) k_fine_edges(int64_t n, int64_t m, const int32_t* __restrict__ eu,
                                                   const int32_t* __restrict__ ev, const double* __restrict__ ew,
                                                   const float* __restrict__ X, double* part, unsigned* counter,
                                                   float* __restrict__ Rf) {
    __shared__ double red[LT];
    const RowLanes<K, false> L;
    constexpr int RPW = RowLanes<K, false>::RPW;
    __shared__ float4 closed[2][LT];
    LaneSums S(closed);
    const int64_t warp = ((int64_t)blockIdx.x * LT + threadIdx.x) >> 5, warps = ((int64_t)gridDim.x * LT) >> 5;
    const float* Xq = X + L.q * 4;
    if (L.ok) {
        edge_blocks<RPW>(m, warp, warps, L.seg, eu, ev, Xq, K, S, [&](int64_t e) { return f64_to_f32(__ldg(ew + e)); });
        for (int64_t p = warp * RPW + L.seg; p < n; p += warps * RPW) {
            add_squares(S.b.open, ld4(Xq + p * K));
            S.count(1);
        }
    }
    if (finish_cols<K, false>(L, S.a.total(), S.b.total(), part, counter, red) && threadIdx.x < K)
        Rf[threadIdx.x] = (float)(red[threadIdx.x] / red[K + threadIdx.x]);
}

// y0[A] = mean of the member rows, M_A = size.  A warp per aggregate: its
// sub-groups take members in turn, four in flight each.
template <int K>
__global__ void __launch_bounds__(LT) k_aggregate_means(int64_t nc, const int32_t* __restrict__ start,
                                                        const uint32_t* __restrict__ members,
                                                        const float* __restrict__ X, float* __restrict__ y0,
                                                        float* __restrict__ mass) {
    const RowLanes<K, true> m;
    constexpr int U = 4, TS = RowLanes<K, true>::TS;
    const int64_t A = ((int64_t)blockIdx.x * LT + threadIdx.x) >> 5;
    if (A >= nc) return;
    const int32_t b = start[A], e = start[A + 1];
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m.ok)
        for (int32_t i = b + m.t; i < e; i += U * TS) {
            float4 x[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i + u * TS < e) x[u] = ld4(X + (int64_t)__ldg(members + i + u * TS) * K + m.q * 4);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i + u * TS < e) {
                    s.x += x[u].x;
                    s.y += x[u].y;
                    s.z += x[u].z;
                    s.w += x[u].w;
                }
        }
    join_row<K, true>(s);
    const float c = (float)(e - b);
    if (m.writes())
        st4(y0 + A * K + m.q * 4, e > b ? make_float4(s.x / c, s.y / c, s.z / c, s.w / c) : s);
    if ((threadIdx.x & 31) == 0) mass[A] = c;
}

// Weights in slot order beside their columns, and the row sums D; SCALE: also
// the FP64 row sums dP and the smallest dG / dP over rows with dP > 0 (positive
// doubles order like their bit patterns, so an integer minimum is exact).
// P lanes per row, lane sums in slot order, combined by a fixed butterfly.
template <int P, bool SCALE>
__global__ void __launch_bounds__(LT) k_param_slots(int64_t nc, const int64_t* __restrict__ rowptr,
                                                    const int32_t* __restrict__ col, const int32_t* __restrict__ eid,
                                                    const float* __restrict__ w, int2* __restrict__ cw,
                                                    float* __restrict__ D, double* __restrict__ dP,
                                                    const double* __restrict__ dG,
                                                    unsigned long long* __restrict__ lam) {
    const int l = threadIdx.x % P;
    const int64_t A = ((int64_t)blockIdx.x * LT + threadIdx.x) / P;
    float s = 0.f;
    double sd = 0.0;
    if (A < nc) {
        const int64_t e = rowptr[A + 1];
        for (int64_t j = rowptr[A] + l; j < e; j += P) {
            const float x = w[eid[j]];
            cw[j] = make_int2(col[j], __float_as_int(x));
            s += x;
            if (SCALE) sd += f32_to_f64(x);
        }
    }
#pragma unroll
    for (int o = P / 2; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        if (SCALE) sd += __shfl_xor_sync(0xffffffffu, sd, o);
    }
    if (A < nc && l == 0) {
        D[A] = s;
        if (SCALE) dP[A] = sd;
    }
    if constexpr (SCALE) {
        if (!lam) return;  // uniform
        unsigned long long v = ~0ull;
        if (A < nc && l == 0 && sd > 0.0) v = (unsigned long long)__double_as_longlong(dG[A] / sd);
#pragma unroll
        for (int o = 16; o >= P; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, v, o);
            v = x < v ? x : v;
        }
        if ((threadIdx.x & 31) == 0 && v != ~0ull) atomicMin(lam, v);
    }
}

// One forward sweep: z = D^-1 A y (or y where D is not positive),
// y1 = (1-w) y + w z.  SWEEP false: y1 = y, nothing written.  MEAN: the
// mass-weighted column means of y1 end in mu.
template <int K, bool LONG, bool SWEEP, bool MEAN>
__global__ void __launch_bounds__(LT, 3) k_param_sweep(int64_t n, const int64_t* __restrict__ rowptr,
                                                    const int2* __restrict__ cw, const float* __restrict__ D,
                                                    const float* __restrict__ y, float omega,
                                                    float* __restrict__ z_out, float* __restrict__ y1,
                                                    const float* __restrict__ mass, double* part, unsigned* counter,
                                                    double* __restrict__ mu) {
    __shared__ double red[LT];
    const RowLanes<K, LONG> m;
    constexpr int RPW = RowLanes<K, LONG>::RPW;
    const float zero = 0.f, one_m = 1.f - omega;
    __shared__ float4 closed[MEAN ? LT : 1];
    LaneSum S(MEAN ? closed : nullptr);
    unsigned terms = 0, total = 0;  // sizes are whole numbers, n of them in all
    const int64_t stride = (((int64_t)gridDim.x * LT) >> 5) * RPW;
    for (int64_t A = (((int64_t)blockIdx.x * LT + threadIdx.x) >> 5) * RPW + m.seg; A < n; A += stride) {
        float4 yi = make_float4(zero, zero, zero, zero);
        if (m.ok) yi = ld4(y + A * K + m.q * 4);
        if constexpr (SWEEP) {
            float4 s = make_float4(zero, zero, zero, zero);
            for_slots<K, LONG>(m, rowptr[A], rowptr[A + 1], cw, y, [&](float w, const float4& x) {
                s.x = fmaf(w, x.x, s.x);
                s.y = fmaf(w, x.y, s.y);
                s.z = fmaf(w, x.z, s.z);
                s.w = fmaf(w, x.w, s.w);
            });
            join_row<K, LONG>(s);
            if (m.writes()) {
                const float d = D[A];
                const float4 z = d > 0.f ? make_float4(s.x / d, s.y / d, s.z / d, s.w / d) : yi;
                if (z_out) st4(z_out + A * K + m.q * 4, z);
                yi.x = one_m * yi.x + omega * z.x;
                yi.y = one_m * yi.y + omega * z.y;
                yi.z = one_m * yi.z + omega * z.z;
                yi.w = one_m * yi.w + omega * z.w;
                st4(y1 + A * K + m.q * 4, yi);
            }
        }
        if constexpr (MEAN) {
            if (m.writes()) {
                const float M = mass[A];
                S.open.x = fmaf(M, yi.x, S.open.x);
                S.open.y = fmaf(M, yi.y, S.open.y);
                S.open.z = fmaf(M, yi.z, S.open.z);
                S.open.w = fmaf(M, yi.w, S.open.w);
                if (m.q == 0) total += (unsigned)M;
                if (++terms % SUM_BLOCK == 0) S.close();
            }
        }
    }
    if constexpr (MEAN) {
        const float4 none = make_float4(zero, zero, zero, zero);
        if (finish_cols<K, LONG, true>(m, S.total(), none, part, counter, red, total) && threadIdx.x < K)
            mu[threadIdx.x] = red[threadIdx.x] / red[K];
    }
}

// Loop control of the edge scaling, from this iteration's loss: convergence
// test, step size from the loss ratio, lambda_1 after the last update.
__device__ __forceinline__ void scale_control(const ScaleStep& st, float loss) {
    ScaleState& S = *st.state;
    if (S.stop) return;
    const double L = (double)loss;
    if (!st.lam_prev) {
        S.L0 = L;
        S.lam1 = 1.0;
        S.eta = st.eta_max;
    } else {
        if ((S.L_prev - L) / L < st.eps) {
            S.stop = 1;
            return;
        }
        if (*st.lam_prev != ~0ull) S.lam1 = __longlong_as_double((long long)*st.lam_prev);
        S.eta = (S.L_prev / S.L0) * st.eta_max;
    }
    S.inv_bound = 1.0 / (S.lam1 * st.bound_step);
    *st.lam_next = ~0ull;
    *st.loss_hist = loss;
    S.L_prev = L;
    S.it += 1;
}

// Quotients of the smoothed block: y^T L y from the squared differences over
// every row's slots (each edge twice), sum M (y - mu)^2; in the last block
// the loss and the adjoint's coefficients
//   coef[0..K) = 2 g / Q, [K..2K) = 2 g N / Q^2, [2K..3K) = g / Q, [3K..4K) = mu,
// g = d loss / d R_c.  LY: L y is stored.  Where rows may be long, blocks are
// closed within the rows (CLOSED_ROWS, with L y, which walks them anyway: a pass
// over the edges beside it cost the gradient on a reduced graph of 13,152 nodes
// and 14.6 M edges, 16 columns, 4,335 us for 3,620), or the squared differences
// come from the edge list and its weights w in blocks (EDGE_LIST: no row is one
// group's).
enum QuotientMode { SHORT_ROWS, CLOSED_ROWS, EDGE_LIST };
struct EdgeList {
    int64_t m = 0;
    const int32_t *eu = nullptr, *ev = nullptr;
    const float* w = nullptr;
};
template <int K, bool LONG, bool LY, QuotientMode MODE>
__global__ void __launch_bounds__(LT) k_quotients(int64_t n, const int64_t* __restrict__ rowptr,
                                                  const int2* __restrict__ cw, EdgeList E, const float* __restrict__ y,
                                                  const float* __restrict__ mass, const double* __restrict__ mu,
                                                  double* part, unsigned* counter, const float* __restrict__ Rf,
                                                  const float* __restrict__ grad_loss, float* __restrict__ loss_out,
                                                  float* __restrict__ ly_out, float* __restrict__ coef, ScaleStep st) {
    __shared__ double red[LT];
    const RowLanes<K, LONG> m;
    constexpr int RPW = RowLanes<K, LONG>::RPW;
    const float zero = 0.f;
    __shared__ float4 closed[2][LT];
    LaneSums S(closed);
    float4 mk = make_float4(zero, zero, zero, zero);
    if (m.ok) {
        const double* u = mu + m.q * 4;
        mk = make_float4((float)u[0], (float)u[1], (float)u[2], (float)u[3]);
    }
    const int64_t stride = (((int64_t)gridDim.x * LT) >> 5) * RPW;
    const int64_t first = (((int64_t)blockIdx.x * LT + threadIdx.x) >> 5) * RPW + m.seg;
    if constexpr (MODE == EDGE_LIST) {
        // (a long row's sub-groups are groups here)
        constexpr int R = RPW * RowLanes<K, LONG>::TS;
        if (m.ok)
            edge_blocks<R>(E.m, first / RPW, stride / RPW, m.seg + m.t, E.eu, E.ev, y + m.q * 4, K, S,
                           [&](int64_t e) { return __ldg(E.w + e); });
    }
    for (int64_t A = first; A < n; A += stride) {
        float4 ya = make_float4(zero, zero, zero, zero), l = ya;
        if (m.ok) ya = ld4(y + A * K + m.q * 4);
        if constexpr (LY || MODE != EDGE_LIST) {
            const int64_t b = rowptr[A], e = rowptr[A + 1];
            for_slots<K, LONG>(m, b, e, cw, y, [&](float w, const float4& x) {
                float d = ya.x - x.x, wd = w * d;
                if (MODE != EDGE_LIST) S.a.open.x = fmaf(wd, d, S.a.open.x);
                l.x += wd;
                d = ya.y - x.y, wd = w * d;
                if (MODE != EDGE_LIST) S.a.open.y = fmaf(wd, d, S.a.open.y);
                l.y += wd;
                d = ya.z - x.z, wd = w * d;
                if (MODE != EDGE_LIST) S.a.open.z = fmaf(wd, d, S.a.open.z);
                l.z += wd;
                d = ya.w - x.w, wd = w * d;
                if (MODE != EDGE_LIST) S.a.open.w = fmaf(wd, d, S.a.open.w);
                l.w += wd;
            }, [&] {
                if (MODE == CLOSED_ROWS) S.count(8);  // for_slots' round
            });
            if (MODE == SHORT_ROWS) S.terms += (unsigned)(e - b);
        }
        if constexpr (LY) {
            join_row<K, LONG>(l);
            if (m.writes()) st4(ly_out + A * K + m.q * 4, l);
        }
        if (m.writes()) {
            const float M = mass[A];
            float t = ya.x - mk.x;
            S.b.open.x = fmaf(M * t, t, S.b.open.x);
            t = ya.y - mk.y;
            S.b.open.y = fmaf(M * t, t, S.b.open.y);
            t = ya.z - mk.z;
            S.b.open.z = fmaf(M * t, t, S.b.open.z);
            t = ya.w - mk.w;
            S.b.open.w = fmaf(M * t, t, S.b.open.w);
        }
        S.count(1);
    }
    if (!finish_cols<K, LONG>(m, S.a.total(), S.b.total(), part, counter, red)) return;
    const int k = threadIdx.x;
    if (k >= 32) return;  // the first warp: a column per lane
    double s = 0.0;
    if (k < K) {
        const double Ns = MODE == EDGE_LIST ? red[k] : 0.5 * red[k], Qs = red[K + k], f = (double)Rf[k];
        const double Rc = Ns / Qs, r = Rc / f - 1.0;
        s = r * r;
        if (coef) {
            const double gq = (grad_loss ? (double)*grad_loss : 1.0) * (2.0 / K) * r / (f * Qs);
            coef[k] = (float)(2.0 * gq);
            coef[K + k] = (float)(2.0 * gq * Rc);
            coef[2 * K + k] = (float)gq;
            coef[3 * K + k] = (float)mu[k];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (k == 0) {
        const float loss = (float)(s * (1.0 / K));
        if (loss_out) *loss_out = loss;
        if (st.state) scale_control(st, loss);
    }
}

// Adjoint of the quotients: yb = 2 g / Q (L y) - 2 g N / Q^2 M (y - mu), and
// T = yb / D, which the reverse sweeps gather
template <int K>
__global__ void __launch_bounds__(LT) k_adj_start(int64_t n, const float* __restrict__ ly, const float* __restrict__ y,
                                                  const float* __restrict__ mass, const float* __restrict__ D,
                                                  const float* __restrict__ coef, float* __restrict__ yb,
                                                  float* __restrict__ T) {
    const int64_t idx = (int64_t)blockIdx.x * LT + threadIdx.x;  // 16-byte chunk
    if (idx >= n * (K / 4)) return;
    const int64_t A = idx / (K / 4);
    const int q = (int)(idx % (K / 4)) * 4;
    const float4 l = ld4(ly + idx * 4), v = ld4(y + idx * 4);
    const float M = mass[A], d = D[A];
    const float li[4] = {l.x, l.y, l.z, l.w}, vi[4] = {v.x, v.y, v.z, v.w};
    float o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        o[i] = coef[q + i] * li[i] - coef[K + q + i] * M * (vi[i] - coef[3 * K + q + i]);
    st4(yb + idx * 4, make_float4(o[0], o[1], o[2], o[3]));
    st4(T + idx * 4, make_float4(o[0] / d, o[1] / d, o[2] / d, o[3] / d));
}

// reverse sweep: yb_s = (1-w) yb + w A T (isolated: yb_s = yb), T_s = yb_s / D
template <int K, bool LONG>
__global__ void __launch_bounds__(LT) k_param_sweep_adj(int64_t n, const int64_t* __restrict__ rowptr,
                                                        const int2* __restrict__ cw, const float* __restrict__ D,
                                                        const float* __restrict__ yb, const float* __restrict__ T,
                                                        float omega, float* __restrict__ yb_out,
                                                        float* __restrict__ T_out) {
    const RowLanes<K, LONG> m;
    constexpr int RPW = RowLanes<K, LONG>::RPW;
    const float zero = 0.f, one_m = 1.f - omega;
    const int64_t stride = (((int64_t)gridDim.x * LT) >> 5) * RPW;
    for (int64_t A = (((int64_t)blockIdx.x * LT + threadIdx.x) >> 5) * RPW + m.seg; A < n; A += stride) {
        float4 s = make_float4(zero, zero, zero, zero);
        for_slots<K, LONG>(m, rowptr[A], rowptr[A + 1], cw, T, [&](float w, const float4& x) {
            s.x = fmaf(w, x.x, s.x);
            s.y = fmaf(w, x.y, s.y);
            s.z = fmaf(w, x.z, s.z);
            s.w = fmaf(w, x.w, s.w);
        });
        join_row<K, LONG>(s);
        if (!m.writes()) continue;
        const float d = D[A];
        float4 b = ld4(yb + A * K + m.q * 4);
        if (d > 0.f) {
            b.x = one_m * b.x + omega * s.x;
            b.y = one_m * b.y + omega * s.y;
            b.z = one_m * b.z + omega * s.z;
            b.w = one_m * b.w + omega * s.w;
        }
        st4(yb_out + A * K + m.q * 4, b);
        st4(T_out + A * K + m.q * 4, make_float4(b.x / d, b.y / d, b.z / d, b.w / d));
    }
}

// Alg. 1's update of edge e = (A, B) with gradient g: momentum, the lambda_1
// guard, never below zero
__device__ __forceinline__ void update_edge(int64_t e, int32_t A, int32_t B, float g, const ScaleStep& st) {
    const double inv = st.state->inv_bound, eta = st.state->eta;
    double d = st.alpha * (double)st.dw[e] - eta * (double)g;
    d = d > 0.0 ? d : 0.0;
    // min(dG / (dP + d)) <= bound at either end <=> d >= min(dG / bound - dP)
    const double cp = st.dG[A] * inv - st.dP[A], cq = st.dG[B] * inv - st.dP[B];
    const double cap = cp < cq ? cp : cq;
    if (d >= cap) d = cap > 0.0 ? cap : 0.0;
    st.dw[e] = (float)d;
    st.w[e] = (float)((double)st.w[e] + d);
}

// Per reduced edge (A, B): the direct term g / Q (y_A - y_B)^2 plus, over the
// sweeps, w [T_A (y_B - z_A) + T_B (y_A - z_B)]; G lanes per edge, a 16-byte
// chunk of the columns each.  SCALE: the edge's scaling update in place of
// its gradient; the sweeps read the slot-order copy of the weights, so w may
// change here.
template <int K, bool SCALE>
__global__ void __launch_bounds__(LT) k_edge_grad(int64_t m, const int32_t* __restrict__ eu,
                                                  const int32_t* __restrict__ ev, int S, int64_t nK,
                                                  const float* __restrict__ Y, const float* __restrict__ Z,
                                                  const float* __restrict__ T, float omega,
                                                  const float* __restrict__ coef, float* __restrict__ grad,
                                                  ScaleStep st) {
    constexpr int G = K / 4, EPW = 32 / G;  // edges per warp
    const int lane = threadIdx.x & 31, seg = lane / G, q = lane % G;
    const int64_t e = (((int64_t)blockIdx.x * LT + threadIdx.x) >> 5) * EPW + seg;
    const bool ok = seg < EPW && e < m;
    float g = 0.f, gs = 0.f;
    if (ok) {
        const int32_t A = eu[e], B = ev[e];
        const int64_t a = (int64_t)A * K + q * 4, b = (int64_t)B * K + q * 4;
        const float4 c = ld4(coef + 2 * K + q * 4);
        const float4 ya = ld4(Y + (int64_t)S * nK + a), yb = ld4(Y + (int64_t)S * nK + b);
        float t = ya.x - yb.x;
        g = c.x * t * t;
        t = ya.y - yb.y;
        g = fmaf(c.y * t, t, g);
        t = ya.z - yb.z;
        g = fmaf(c.z * t, t, g);
        t = ya.w - yb.w;
        g = fmaf(c.w * t, t, g);
#pragma unroll 2
        for (int s = 0; s < S; ++s) {
            const int64_t o = (int64_t)s * nK;
            const float4 ta = ld4(T + o + a), tb = ld4(T + o + b);  // T_{s+1}
            const float4 y0 = ld4(Y + o + a), y1 = ld4(Y + o + b);
            const float4 z0 = ld4(Z + o + a), z1 = ld4(Z + o + b);
            gs = fmaf(ta.x, y1.x - z0.x, gs);
            gs = fmaf(ta.y, y1.y - z0.y, gs);
            gs = fmaf(ta.z, y1.z - z0.z, gs);
            gs = fmaf(ta.w, y1.w - z0.w, gs);
            gs = fmaf(tb.x, y0.x - z1.x, gs);
            gs = fmaf(tb.y, y0.y - z1.y, gs);
            gs = fmaf(tb.z, y0.z - z1.z, gs);
            gs = fmaf(tb.w, y0.w - z1.w, gs);
        }
    }
    g = fmaf(omega, gs, g);
    float tot = g;
#pragma unroll
    for (int i = 1; i < G; ++i) tot += __shfl_down_sync(0xffffffffu, g, i);
    if constexpr (!SCALE) {
        if (ok && q == 0) grad[e] = tot;
    } else {
        // the update is FP64 work (four divisions an edge): the block's edges
        // are handed to full warps, one lane in G would pay the pipe for all
        constexpr int EPB = EPW * LW;
        __shared__ float s_g[EPB];
        if (seg < EPW && q == 0) s_g[(threadIdx.x >> 5) * EPW + seg] = tot;
        __syncthreads();
        const int64_t f = (int64_t)blockIdx.x * EPB + threadIdx.x;
        if (threadIdx.x >= EPB || f >= m || st.state->stop) return;
        update_edge(f, eu[f], ev[f], s_g[threadIdx.x], st);
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// A warp per row from a mean of 32 slots on; below, G lanes hold a row's
// slots in flight by themselves and the other rows of the warp hide them
// (a warp per row on 7,680 rows of 13 slots, K = 16: 9 us a sweep against 6).
bool long_rows(const gr_ctx* c, int64_t slots) { return slots >= 32 * c->n; }

// blocks of a row pass: one wave, and what the statistics tickets can count
template <int K, bool LONG>
unsigned row_grid(const gr_ctx* c, int64_t n) {
    const int64_t want = ceil_div(n > 0 ? n : 1, (int64_t)RowLanes<K, LONG>::RPW * LW);
    int64_t cap = (int64_t)c->num_sms * ROW_BLOCKS;
    if (cap > STATS_GROUP * STATS_MAX_GROUPS) cap = STATS_GROUP * STATS_MAX_GROUPS;
    return (unsigned)(want < cap ? want : cap);
}
constexpr size_t PART_ROWS = (size_t)STATS_GROUP * STATS_MAX_GROUPS;

template <int K, bool LONG>
gr_status fine_quotients(gr_ctx* f, const float* X, double* part, unsigned* counter, float* Rf) {
    k_fine_quotients<K, LONG><<<row_grid<K, LONG>(f, f->n), LT, 0, f->stream>>>(f->n, f->eptr, f->ev, f->ew, X, part,
                                                                               counter, Rf);
    count_launch();
    GR_TRY_CUDA(f, cudaGetLastError(), "fine quotients");
    return GR_OK;
}

template <int K>
gr_status fine_edges(gr_ctx* f, const float* X, double* part, unsigned* counter, float* Rf) {
    const int64_t rounds = ceil_div(f->m, EDGE_FLIGHT), work = rounds > f->n ? rounds : f->n;
    k_fine_edges<K><<<row_grid<K, false>(f, work), LT, 0, f->stream>>>(f->n, f->m, f->eu, f->ev, f->ew, X, part,
                                                                      counter, Rf);
    count_launch();
    GR_TRY_CUDA(f, cudaGetLastError(), "fine edges");
    return GR_OK;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

template <int K>
gr_status fine_k(gr_ctx* f, gr_ctx* cc, const int32_t* agg, const float* X, float* y0, float* Rf, float* mass,
                 bool* bad) {
    cudaStream_t s = f->stream;
    const int64_t n = f->n, nc = cc->n;
    bool short_parts;
    GR_TRY_CUDA(f, parts_short(f, &short_parts), "row lengths");
    // rows are moved in 16-byte chunks: a block or result that does not start
    // on such a boundary goes through an aligned copy
    const bool cx = !aligned16(X), cy = !aligned16(y0);
    const size_t b_part = sizeof(double) * 2 * K * PART_ROWS, b_y = cy ? sizeof(float) * (size_t)nc * K : 0;
    void* p;
    GR_TRY_CUDA(cc, cc->ws.get(WS_LOSS_A, b_part + STATS_COUNTER_BYTES + 256 + b_y +
                                              (cx ? sizeof(float) * (size_t)n * K : 0), &p), "ws");
    double* part = (double*)p;
    unsigned* counter = (unsigned*)((char*)p + b_part);
    float* ytmp = (float*)((char*)p + ((b_part + STATS_COUNTER_BYTES + 255) & ~size_t(255)));
    float* yout = cy ? ytmp : y0;
    if (cx) {
        float* t = (float*)((char*)ytmp + b_y);
        GR_TRY_CUDA(cc, cudaMemcpyAsync(t, X, sizeof(float) * (size_t)n * K, cudaMemcpyDeviceToDevice, s), "copy");
        X = t;
    }
    GR_TRY_CUDA(cc, cudaMemsetAsync(counter, 0, STATS_COUNTER_BYTES, s), "memset");
    MapChain ch;
    ch.map[0] = agg;
    ch.count = 1;
    GroupJob job;
    gr_status st = group_begin(cc, WS_LOSS_C, ch, n, nc, &job);
    if (st != GR_OK) return st;
    // upper edges per row: half the slots
    if (!short_parts) st = fine_edges<K>(f, X, part, counter, Rf);
    else st = long_rows(f, f->m) ? fine_quotients<K, true>(f, X, part, counter, Rf)
                                 : fine_quotients<K, false>(f, X, part, counter, Rf);
    if (st != GR_OK) return st;
    st = group_finish(cc, &job, bad);
    if (st != GR_OK || *bad) return st;
    k_aggregate_means<K><<<(unsigned)ceil_div(nc * 32, LT), LT, 0, s>>>(nc, job.start, job.members, X, yout, mass);
    count_launch();
    if (cy) GR_TRY_CUDA(cc, cudaMemcpyAsync(y0, yout, b_y, cudaMemcpyDeviceToDevice, s), "copy");
    GR_TRY_CUDA(cc, cudaGetLastError(), "aggregate means");
    return GR_OK;
}

template <int K, bool LONG>
gr_status coarse_k(gr_ctx* cc, int S, double omega, const float* y0, const float* Rf, const float* mass,
                   const LossWork& W, bool adjoint, const float* grad_loss, float* loss_out, const ScaleStep& st) {
    cudaStream_t s = cc->stream;
    const int64_t nc = cc->n, nK = nc * K;
    const unsigned grid = row_grid<K, LONG>(cc, nc);
    const float om = (float)omega;
    const float* y = y0;
    if (S == 0) {
        k_param_sweep<K, LONG, false, true><<<grid, LT, 0, s>>>(nc, cc->rowptr, W.cw, W.D, y, om, nullptr, nullptr,
                                                                 mass, W.part, W.counter, W.mu);
        count_launch();
    }
    for (int it = 0; it < S; ++it) {
        // without the adjoint two buffers take turns
        float* out = adjoint ? W.Y + (size_t)(it + 1) * nK : W.Y + (size_t)(it & 1) * nK;
        float* z = adjoint ? W.Z + (size_t)it * nK : nullptr;
        if (it + 1 < S)
            k_param_sweep<K, LONG, true, false><<<grid, LT, 0, s>>>(nc, cc->rowptr, W.cw, W.D, y, om, z, out, nullptr,
                                                                     nullptr, nullptr, nullptr);
        else
            k_param_sweep<K, LONG, true, true><<<grid, LT, 0, s>>>(nc, cc->rowptr, W.cw, W.D, y, om, z, out, mass,
                                                                    W.part, W.counter, W.mu);
        count_launch();
        y = out;
    }
    EdgeList E;
    E.m = cc->m;
    E.eu = cc->eu;
    E.ev = cc->ev;
    E.w = W.w;
    auto quotients = [&](auto kern, unsigned blocks) {
        kern<<<blocks, LT, 0, s>>>(nc, cc->rowptr, W.cw, E, y, mass, W.mu, W.part, W.counter, Rf,
                                   adjoint ? grad_loss : nullptr, loss_out, adjoint ? W.yb1 : nullptr,
                                   adjoint ? W.coef : nullptr, st);
        count_launch();
    };
    if (W.short_parts) {
        adjoint ? quotients(k_quotients<K, LONG, true, SHORT_ROWS>, grid)
                : quotients(k_quotients<K, LONG, false, SHORT_ROWS>, grid);
    } else if (adjoint) {
        quotients(k_quotients<K, LONG, true, CLOSED_ROWS>, grid);
    } else {  // a round of edges for every warp, if there are as many
        const int64_t rounds = ceil_div(cc->m, EDGE_FLIGHT * RowLanes<K, LONG>::TS);
        quotients(k_quotients<K, LONG, false, EDGE_LIST>, row_grid<K, LONG>(cc, rounds > nc ? rounds : nc));
    }
    GR_TRY_CUDA(cc, cudaGetLastError(), "loss");
    return GR_OK;
}

template <int K, bool LONG>
gr_status adjoint_k(gr_ctx* cc, int S, double omega, const float* mass, const LossWork& W, float* grad,
                    const ScaleStep& st) {
    cudaStream_t s = cc->stream;
    const int64_t nc = cc->n, nK = nc * K;
    const unsigned grid = row_grid<K, LONG>(cc, nc);
    const float om = (float)omega;
    if (S > 0) {
        float *yb = W.yb0, *yn = W.yb1;  // yb1 held L y
        k_adj_start<K><<<(unsigned)ceil_div(nc * (K / 4), LT), LT, 0, s>>>(nc, W.yb1, W.Y + (size_t)S * nK, mass, W.D,
                                                                          W.coef, yb, W.T + (size_t)(S - 1) * nK);
        count_launch();
        // T_S .. T_1; the adjoint of y_0 itself enters no gradient
        for (int it = S - 1; it >= 1; --it) {
            k_param_sweep_adj<K, LONG><<<grid, LT, 0, s>>>(nc, cc->rowptr, W.cw, W.D, yb, W.T + (size_t)it * nK, om, yn,
                                                            W.T + (size_t)(it - 1) * nK);
            count_launch();
            float* t = yb;
            yb = yn;
            yn = t;
        }
    }
    if (cc->m > 0) {
        constexpr int EPB = (32 / (K / 4)) * LW;
        const unsigned ge = (unsigned)ceil_div(cc->m, EPB);
        if (st.state)
            k_edge_grad<K, true><<<ge, LT, 0, s>>>(cc->m, cc->eu, cc->ev, S, nK, W.Y, W.Z, W.T, om, W.coef, nullptr, st);
        else
            k_edge_grad<K, false><<<ge, LT, 0, s>>>(cc->m, cc->eu, cc->ev, S, nK, W.Y, W.Z, W.T, om, W.coef, grad, st);
        count_launch();
    }
    GR_TRY_CUDA(cc, cudaGetLastError(), "loss adjoint");
    return GR_OK;
}

template <int K>
gr_status coarse_pick(gr_ctx* cc, int S, double omega, const float* y0, const float* Rf, const float* mass,
                      const LossWork& W, bool adjoint, const float* grad_loss, float* loss_out, const ScaleStep& st) {
    return long_rows(cc, 2 * cc->m) ? coarse_k<K, true>(cc, S, omega, y0, Rf, mass, W, adjoint, grad_loss, loss_out, st)
                                       : coarse_k<K, false>(cc, S, omega, y0, Rf, mass, W, adjoint, grad_loss, loss_out, st);
}

template <int K>
gr_status adjoint_pick(gr_ctx* cc, int S, double omega, const float* mass, const LossWork& W, float* grad,
                       const ScaleStep& st) {
    return long_rows(cc, 2 * cc->m) ? adjoint_k<K, true>(cc, S, omega, mass, W, grad, st)
                                       : adjoint_k<K, false>(cc, S, omega, mass, W, grad, st);
}

}  // namespace

gr_status loss_fine(gr_ctx* f, gr_ctx* cc, const int32_t* agg, const float* X, int K, float* y0, float* Rf,
                    float* mass, bool* bad) {
    auto run = [&]() {
        switch (K) {
            case 4: return fine_k<4>(f, cc, agg, X, y0, Rf, mass, bad);
            case 8: return fine_k<8>(f, cc, agg, X, y0, Rf, mass, bad);
            case 16: return fine_k<16>(f, cc, agg, X, y0, Rf, mass, bad);
            case 24: return fine_k<24>(f, cc, agg, X, y0, Rf, mass, bad);
            case 32: return fine_k<32>(f, cc, agg, X, y0, Rf, mass, bad);
        }
        return set_error(f, GR_EINVAL, "loss: K must be 4, 8, 16, 24 or 32");
    };
    const gr_status st = run();
    // a refused call leaves no kernel behind that reads X or writes R_f
    if (st != GR_OK || *bad) cudaStreamSynchronize(f->stream);
    return st;
}

gr_status loss_work(gr_ctx* cc, int K, int S, bool adjoint, LossWork* W) {
    const size_t nc = (size_t)cc->n, nK = nc * (size_t)K;
    size_t need = 0;
    auto add = [&](size_t bytes) {
        size_t off = need;
        need += (bytes + 255) & ~size_t(255);
        return off;
    };
    const size_t o_cw = add(sizeof(int2) * (size_t)(cc->m > 0 ? 2 * cc->m : 1)), o_D = add(4 * nc),
                 o_part = add(sizeof(double) * 2 * (size_t)K * PART_ROWS), o_ctr = add(STATS_COUNTER_BYTES),
                 o_coef = add(sizeof(float) * 4 * (size_t)K), o_mu = add(sizeof(double) * (size_t)K),
                 o_Y = add(4 * nK * (adjoint ? (size_t)S + 1 : 2)), o_Z = add(adjoint ? 4 * nK * (size_t)S : 0),
                 o_T = add(adjoint ? 4 * nK * (size_t)S : 0), o_b0 = add(adjoint ? 4 * nK : 0),
                 o_b1 = add(adjoint ? 4 * nK : 0);
    GR_TRY_CUDA(cc, parts_short(cc, &W->short_parts), "row lengths");
    void* base;
    GR_TRY_CUDA(cc, cc->ws.get(WS_LOSS_B, need, &base), "ws");
    char* B = (char*)base;
    W->cw = (int2*)(B + o_cw);
    W->D = (float*)(B + o_D);
    W->part = (double*)(B + o_part);
    W->counter = (unsigned*)(B + o_ctr);
    W->coef = (float*)(B + o_coef);
    W->mu = (double*)(B + o_mu);
    W->Y = (float*)(B + o_Y);
    W->Z = (float*)(B + o_Z);
    W->T = (float*)(B + o_T);
    W->yb0 = (float*)(B + o_b0);
    W->yb1 = (float*)(B + o_b1);
    GR_TRY_CUDA(cc, cudaMemsetAsync(W->counter, 0, STATS_COUNTER_BYTES, cc->stream), "memset");
    return GR_OK;
}

gr_status loss_weights(gr_ctx* cc, const float* w, LossWork& W, double* dP, const double* dG,
                       unsigned long long* lam) {
    cudaStream_t s = cc->stream;
    const int64_t nc = cc->n;
    W.w = w;
    auto run = [&](auto kern, int lanes) {
        kern<<<(unsigned)ceil_div(nc * lanes, LT), LT, 0, s>>>(nc, cc->rowptr, cc->col, cc->eid, w, W.cw, W.D, dP, dG,
                                                                lam);
        count_launch();
    };
    // a warp wherever a row may be long: its sum is FP32 (8 lanes on a hub of
    // 62,500 slots took 5 ms)
    const bool lng = long_rows(cc, 2 * cc->m) || !W.short_parts;
    if (dP) lng ? run(k_param_slots<32, true>, 32) : run(k_param_slots<8, true>, 8);
    else lng ? run(k_param_slots<32, false>, 32) : run(k_param_slots<8, false>, 8);
    GR_TRY_CUDA(cc, cudaGetLastError(), "parameter weights");
    return GR_OK;
}

gr_status loss_coarse(gr_ctx* cc, int K, int S, double omega, const float* y0, const float* Rf, const float* mass,
                      const LossWork& W, bool adjoint, const float* grad_loss, float* loss_out, const ScaleStep& st) {
    switch (K) {
        case 4: return coarse_pick<4>(cc, S, omega, y0, Rf, mass, W, adjoint, grad_loss, loss_out, st);
        case 8: return coarse_pick<8>(cc, S, omega, y0, Rf, mass, W, adjoint, grad_loss, loss_out, st);
        case 16: return coarse_pick<16>(cc, S, omega, y0, Rf, mass, W, adjoint, grad_loss, loss_out, st);
        case 24: return coarse_pick<24>(cc, S, omega, y0, Rf, mass, W, adjoint, grad_loss, loss_out, st);
        case 32: return coarse_pick<32>(cc, S, omega, y0, Rf, mass, W, adjoint, grad_loss, loss_out, st);
    }
    return set_error(cc, GR_EINVAL, "loss: K must be 4, 8, 16, 24 or 32");
}

gr_status loss_adjoint(gr_ctx* cc, int K, int S, double omega, const float* mass, const LossWork& W, float* grad,
                       const ScaleStep& st) {
    switch (K) {
        case 4: return adjoint_pick<4>(cc, S, omega, mass, W, grad, st);
        case 8: return adjoint_pick<8>(cc, S, omega, mass, W, grad, st);
        case 16: return adjoint_pick<16>(cc, S, omega, mass, W, grad, st);
        case 24: return adjoint_pick<24>(cc, S, omega, mass, W, grad, st);
        case 32: return adjoint_pick<32>(cc, S, omega, mass, W, grad, st);
    }
    return set_error(cc, GR_EINVAL, "loss: K must be 4, 8, 16, 24 or 32");
}

gr_status loss_fwd_impl(gr_ctx* fine, gr_ctx* coarse, const int32_t* agg, const float* X, int K,
                        const float* w_c, int sweeps, double omega, float* loss, float* saved) {
    const int64_t nK = coarse->n * K;
    float *y0 = saved, *Rf = saved + nK, *mass = Rf + K;
    bool bad = false;
    gr_status st = loss_fine(fine, coarse, agg, X, K, y0, Rf, mass, &bad);
    if (st != GR_OK) return st;
    if (bad) return set_error(fine, GR_EINVAL, "loss_fwd: agg labels must lie in [0, coarse n)");
    LossWork W;
    st = loss_work(coarse, K, sweeps, false, &W);
    if (st != GR_OK) return st;
    const float* y = y0;
    if (!aligned16(y0)) {  // the sweeps read 16-byte chunks
        GR_TRY_CUDA(coarse, cudaMemcpyAsync(W.Y + nK, y0, sizeof(float) * nK, cudaMemcpyDeviceToDevice, coarse->stream),
                    "copy");
        y = W.Y + nK;
    }
    st = loss_weights(coarse, w_c, W, nullptr, nullptr, nullptr);
    if (st != GR_OK) return st;
    return loss_coarse(coarse, K, sweeps, omega, y, Rf, mass, W, false, nullptr, loss, ScaleStep());
}

gr_status loss_bwd_impl(gr_ctx* coarse, const float* saved, int K, const float* w_c, int sweeps,
                        double omega, const float* grad_loss, float* grad_w) {
    const int64_t nK = coarse->n * K;
    const float *Rf = saved + nK, *mass = Rf + K;
    LossWork W;
    gr_status st = loss_work(coarse, K, sweeps, true, &W);
    if (st != GR_OK) return st;
    GR_TRY_CUDA(coarse, cudaMemcpyAsync(W.Y, saved, sizeof(float) * nK, cudaMemcpyDeviceToDevice, coarse->stream),
                "copy");
    st = loss_weights(coarse, w_c, W, nullptr, nullptr, nullptr);
    if (st != GR_OK) return st;
    st = loss_coarse(coarse, K, sweeps, omega, W.Y, Rf, mass, W, true, grad_loss, nullptr, ScaleStep());
    if (st != GR_OK) return st;
    return loss_adjoint(coarse, K, sweeps, omega, mass, W, grad_w, ScaleStep());
}

}  // namespace gr
