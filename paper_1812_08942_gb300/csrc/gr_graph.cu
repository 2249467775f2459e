// Graph construction: the symmetric CSR of A_G and the degrees D_G (Sec. 2.1),
// and Galerkin coarsening L_R = P^T L_G P (Sec. 3.2.2): row by row in shared
// memory (gr_galerkin.cu), or by a global sort + segmented sum when a coarse
// row is too long for that.
#include <utility>

#include "gr_ieee.cuh"
#include "gr_internal.cuh"
#include "gr_vec.cuh"

namespace gr {

constexpr int TB = 256;

// ---------------------------------------------------------------------------
// CSR construction from a canonical edge list
// ---------------------------------------------------------------------------
constexpr int PT = 4;  // list positions a thread of the per-edge kernels takes, their loads in flight together

// eptr[p] = first edge with u >= p (u is sorted), for p in [0, n]
__global__ void __launch_bounds__(TB) k_upper_ptr(const int32_t* __restrict__ eu, int64_t m, int64_t n,
                                                  int64_t* __restrict__ eptr) {
    const int64_t t0 = (int64_t)blockIdx.x * (TB * PT) + threadIdx.x;
    int64_t prev[PT], cur[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int64_t e = t0 + i * TB;
        prev[i] = e == 0 || e > m ? -1 : (int64_t)__ldg(eu + e - 1);
        cur[i] = e == m ? n : e > m ? -1 : (int64_t)__ldg(eu + e);
    }
#pragma unroll
    for (int i = 0; i < PT; ++i)
        for (int64_t p = prev[i] + 1; p <= cur[i]; ++p) eptr[p] = t0 + i * TB;
}

// The lower parts from the edges sorted by v: lstart[p] = first position with
// v >= p, for p in [0, n], and with the upper parts before it the row's start.
// long_low (may be null) is raised by a lower part past ROW_PART_SHORT edges.
__global__ void __launch_bounds__(TB) k_lower_ptr(const uint32_t* __restrict__ skey, int64_t m, int64_t n,
                                                  const int64_t* __restrict__ eptr, int64_t* __restrict__ lstart,
                                                  int64_t* __restrict__ rowptr, int32_t* __restrict__ long_low) {
    const int64_t t0 = (int64_t)blockIdx.x * (TB * PT) + threadIdx.x;
    int64_t prev[PT], cur[PT];
    bool far = false;
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int64_t t = t0 + i * TB;
        prev[i] = t == 0 || t > m ? -1 : (int64_t)__ldg(skey + t - 1);
        cur[i] = t == m ? n : t > m ? -1 : (int64_t)__ldg(skey + t);
        if (long_low && t >= ROW_PART_SHORT && t < m) far |= (int64_t)__ldg(skey + t - ROW_PART_SHORT) == cur[i];
    }
#pragma unroll
    for (int i = 0; i < PT; ++i)
        for (int64_t p = prev[i] + 1; p <= cur[i]; ++p) {
            lstart[p] = t0 + i * TB;
            rowptr[p] = t0 + i * TB + eptr[p];
        }
    if (far) *long_low = 1;
}

// lower part of row p: edges (q, p), q < p, in ascending q (= ascending id);
// position t of the stable sort by v holds the t-th such edge overall.
__global__ void k_fill_lower(const uint32_t* __restrict__ skey, const uint32_t* __restrict__ sval,
                             int64_t m, const int64_t* __restrict__ lstart,
                             const int64_t* __restrict__ rowptr, const int32_t* __restrict__ eu,
                             const double* __restrict__ ew, int32_t* __restrict__ col,
                             int32_t* __restrict__ eid, double* __restrict__ wslot) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    int64_t p = skey[t];
    int64_t e = sval[t];
    int64_t slot = rowptr[p] + (t - lstart[p]);
    col[slot] = eu[e];
    eid[slot] = (int32_t)e;
    wslot[slot] = ew[e];
}

// upper part of row p: edges (p, v), v > p, after the lower part
__global__ void k_fill_upper(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                             const double* __restrict__ ew, int64_t m,
                             const int64_t* __restrict__ eptr, const int64_t* __restrict__ rowptr,
                             int32_t* __restrict__ col, int32_t* __restrict__ eid,
                             double* __restrict__ wslot) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m) return;
    int64_t p = eu[e];
    int64_t slot = rowptr[p + 1] - (eptr[p + 1] - e);
    col[slot] = ev[e];
    eid[slot] = (int32_t)e;
    wslot[slot] = ew[e];
}

// Warp per row of a dense graph, from the lower edge ids sorted by v: the
// slots, D(p,p) = the lanes' sums in slot order combined by a fixed tree, and
// the row-scaled weights w / D(p,p) that D^-1 A uses, in one pass.  A row of
// up to 128 slots stays in registers; a longer one keeps its weights in the
// slot array between its two passes.  Four slots in flight a lane (eight leave
// four blocks an SM: 427 us against 373 below).
// Bound by the waits for the two dependent gathers and by the FP64 pipe, which
// takes an instruction of one lane as long as one of 32: the tree and the
// division of eight rows are one warp's, a lane per pair and per row (a
// shuffle tree and a division in every warp: 607 us).  434,000 rows, 32 M
// slots: 966 us with separate fills of the two parts and a scaling pass, 373
// now; 13,000 rows, 26 M slots: 446 and 315.
constexpr int FIN_ROWS = TB / 32;
constexpr int FIN_FLIGHT = 4;  // slots in flight a lane

struct FinRow {
    int64_t r0, l0, e0;
    int low, len;
};

struct FinArrays {
    const uint32_t* sval;
    const int32_t *eu, *ev;
    const double* ew;
    int32_t *col, *eid;
    double* wn64;
    int2* cw32;
};

// sum of a row's lane sums, for the block's rows: every thread calls it
__device__ __forceinline__ double fin_inverse(double s, double* __restrict__ deg, int64_t n) {
    __shared__ double part[FIN_ROWS][32];
    __shared__ double inv[FIN_ROWS];
    static_assert(FIN_ROWS == 8, "the tree's first step is four pairs a lane");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {  // lane l of a row takes l + o
            double x[4];
#pragma unroll
            for (int i = 0; i < (o + 3) / 4; ++i) {
                const int j = lane + 32 * i;
                if (j < FIN_ROWS * o) x[i] = part[j / o][j % o] + part[j / o][j % o + o];
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < (o + 3) / 4; ++i) {
                const int j = lane + 32 * i;
                if (j < FIN_ROWS * o) part[j / o][j % o] = x[i];
            }
            __syncwarp();
        }
        const int64_t p = (int64_t)blockIdx.x * FIN_ROWS + lane;
        if (lane < FIN_ROWS) {
            const double d = part[lane][0];
            if (p < n) deg[p] = d;
            inv[lane] = row_inverse(d);
        }
    }
    __syncthreads();
    return inv[warp];
}

template <int U, int N>
__device__ __forceinline__ double fin_load(const FinArrays& A, const FinRow& R, int b, int32_t (&e)[N],
                                           int32_t (&q)[N], double (&w)[N], double s) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int i = b + 32 * u;
        if (i < R.len) e[u] = i < R.low ? (int32_t)__ldg(A.sval + R.l0 + i) : (int32_t)(R.e0 + (i - R.low));
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (b + 32 * u < R.len) {
            q[u] = __ldg((b + 32 * u < R.low ? A.eu : A.ev) + e[u]);
            w[u] = __ldg(A.ew + e[u]);
        }
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (b + 32 * u < R.len) s += w[u];
    return s;
}

template <int U, int N>
__device__ __forceinline__ void fin_store(const FinArrays& A, const FinRow& R, int b, const int32_t (&e)[N],
                                          const int32_t (&q)[N], const double (&w)[N], double inv) {
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (b + 32 * u < R.len) {
            const int64_t j = R.r0 + b + 32 * u;
            const double x = w[u] * inv;
            A.col[j] = q[u];
            A.eid[j] = e[u];
            A.wn64[j] = x;
            A.cw32[j] = make_int2(q[u], __float_as_int(f64_to_f32(x)));
        }
}

__global__ void __launch_bounds__(TB, 5) k_row_finish_sorted(int64_t n, const int64_t* __restrict__ rowptr,
                                                          const int64_t* __restrict__ lstart,
                                                          const int64_t* __restrict__ eptr, FinArrays A,
                                                          double* __restrict__ deg) {
    const int lane = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * FIN_ROWS + (threadIdx.x >> 5);
    FinRow R{0, 0, 0, 0, 0};
    if (p < n) {
        R.r0 = rowptr[p];
        R.l0 = lstart[p];
        R.e0 = eptr[p];
        R.low = (int)(lstart[p + 1] - R.l0);
        R.len = (int)(rowptr[p + 1] - R.r0);
    }
    int32_t e[FIN_FLIGHT], q[FIN_FLIGHT];
    double w[FIN_FLIGHT], s = 0.0;
    const bool kept = R.len <= 32 * FIN_FLIGHT;
    // by length, for an FP64 instruction whose lanes are all past the end
    // takes the pipe like any other
    if (R.len <= 32) {
        s = fin_load<1>(A, R, lane, e, q, w, s);
    } else if (R.len <= 64) {
        s = fin_load<2>(A, R, lane, e, q, w, s);
    } else if (kept) {
        s = fin_load<4>(A, R, lane, e, q, w, s);
    } else {
        for (int b = lane; b < R.len; b += 32 * FIN_FLIGHT) {
            int32_t ee[FIN_FLIGHT], qq[FIN_FLIGHT];
            double ww[FIN_FLIGHT];
            s = fin_load<FIN_FLIGHT>(A, R, b, ee, qq, ww, s);
#pragma unroll
            for (int u = 0; u < FIN_FLIGHT; ++u)
                if (b + 32 * u < R.len) {
                    const int64_t j = R.r0 + b + 32 * u;
                    A.col[j] = qq[u];
                    A.eid[j] = ee[u];
                    A.wn64[j] = ww[u];
                }
        }
    }
    const double inv = fin_inverse(s, deg, n);
    if (kept) {
        if (R.len <= 32) fin_store<1>(A, R, lane, e, q, w, inv);
        else if (R.len <= 64) fin_store<2>(A, R, lane, e, q, w, inv);
        else fin_store<4>(A, R, lane, e, q, w, inv);
        return;
    }
    // a lane reads back what it wrote itself
    for (int b = lane; b < R.len; b += 32 * FIN_FLIGHT) {
        int32_t qq[FIN_FLIGHT];
        double ww[FIN_FLIGHT];
#pragma unroll
        for (int u = 0; u < FIN_FLIGHT; ++u)
            if (b + 32 * u < R.len) {
                ww[u] = A.wn64[R.r0 + b + 32 * u];
                qq[u] = A.col[R.r0 + b + 32 * u];
            }
#pragma unroll
        for (int u = 0; u < FIN_FLIGHT; ++u)
            if (b + 32 * u < R.len) {
                const double x = ww[u] * inv;
                A.wn64[R.r0 + b + 32 * u] = x;
                A.cw32[R.r0 + b + 32 * u] = make_int2(qq[u], __float_as_int(f64_to_f32(x)));
            }
    }
}

// thread per row (short rows): D(p,p) summed sequentially in slot order,
// which is ascending edge id -- the plain definition's order.  A warp's 32
// rows are consecutive: when their slots fit the warp's shared-memory buffer
// the warp reads the weights and columns in whole lines, each thread sums and
// scales its row there, and the warp writes both slot arrays in whole lines.
// A row past DS_LONG slots is added up by its warp, 32 weights at a time and in
// the same order, and scaled by all lanes (three hubs of 88,000 edges
// among 400,000 rows: a graph in 20.0 ms with a thread each, 5.3 with the warp).
constexpr int DS_CAP = 512;  // slots a warp stages
constexpr int DS_LONG = 256;

__global__ void __launch_bounds__(TB, 4) k_degree_scale_rows(const int64_t* __restrict__ rowptr,
                                                          const int32_t* __restrict__ col, int64_t n,
                                                          double* __restrict__ wn64, int2* __restrict__ cw32,
                                                          double* __restrict__ deg) {
    __shared__ double s_w[TB / 32][DS_CAP];
    __shared__ int32_t s_c[TB / 32][DS_CAP];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t pw = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
    if (pw >= n) return;  // whole warp
    const int64_t p = pw + lane;
    const int lv = (int)((n - pw < 32 ? n - pw : 32) - 1);
    const int64_t R0 = rowptr[pw], R1 = rowptr[pw + lv + 1];
    if (R1 - R0 <= DS_CAP) {
        double* W = s_w[wp];
        int32_t* C = s_c[wp];
        const int ns = (int)(R1 - R0);
        for (int j = lane; j < ns; j += 32) {
            W[j] = wn64[R0 + j];
            C[j] = col[R0 + j];
        }
        __syncwarp();
        if (p < n) {
            const int b = (int)(rowptr[p] - R0), e = (int)(rowptr[p + 1] - R0);
            double s = 0.0;
            for (int j = b; j < e; ++j) s += W[j];
            deg[p] = s;
            const double inv = row_inverse(s);
            for (int j = b; j < e; ++j) W[j] = W[j] * inv;
        }
        __syncwarp();
        for (int j = lane; j < ns; j += 32) {
            const double x = W[j];
            wn64[R0 + j] = x;
            cw32[R0 + j] = make_int2(C[j], __float_as_int(f64_to_f32(x)));
        }
        return;
    }
    const int64_t b = p < n ? rowptr[p] : 0, e = p < n ? rowptr[p + 1] : 0;
    const bool far = e - b > DS_LONG;
    if (p < n && !far) {
        double s = 0.0;
        for (int64_t j = b; j < e; ++j) s += wn64[j];
        deg[p] = s;
        const double inv = row_inverse(s);
        for (int64_t j = b; j < e; ++j) {
            const double x = wn64[j] * inv;
            wn64[j] = x;
            cw32[j] = make_int2(col[j], __float_as_int(f64_to_f32(x)));
        }
    }
    constexpr unsigned FULL = 0xffffffffu;
    for (unsigned todo = __ballot_sync(FULL, far); todo; todo &= todo - 1) {
        const int o = __ffs(todo) - 1;
        const int64_t ob = __shfl_sync(FULL, b, o), oe = __shfl_sync(FULL, e, o);
        double s = 0.0, w = wn64[ob + lane];  // (a long row has 32 slots and more)
        for (int64_t j = ob; j < oe; j += 32) {
            const double next = j + 32 + lane < oe ? wn64[j + 32 + lane] : 0.0;
#pragma unroll
            for (int i = 0; i < 32; ++i) s += __shfl_sync(FULL, w, i);  // past the end: + 0
            w = next;
        }
        if (lane == 0) deg[pw + o] = s;
        const double inv = row_inverse(s);
        for (int64_t j = ob + lane; j < oe; j += 32) {
            const double x = wn64[j] * inv;
            wn64[j] = x;
            cw32[j] = make_int2(col[j], __float_as_int(f64_to_f32(x)));
        }
    }
}

// ---------------------------------------------------------------------------
// CSR of a sparse graph by lower-part sorting.  The upper part of row p
// (edges (p, v), v > p) is a contiguous, sorted run of the canonical list; the
// lower part (edges (q, p), q < p) is gathered by atomic slot claims and then
// sorted per row by edge id, which for a fixed p is ascending q.  One pass per
// row then writes both parts, the degree and the row-scaled weights.
// ---------------------------------------------------------------------------
constexpr int LOWER_THREAD = 32;   // lower parts up to this long: sorted by the row's own thread
constexpr int LOWER_WARP = 2048;   // up to this long: by a warp in shared memory; longer: global sort
constexpr int FW = 4;              // warps per block of the warp kernel

// per edge: canonical-input check (when asked) and, unless lcnt is null, the
// lower count of v; the block maximum of the counts reached goes to lmax;
// long_up is raised by an upper part past ROW_PART_SHORT edges (u is sorted)
__global__ void __launch_bounds__(TB) k_csr_count(int64_t n, int64_t m, const int32_t* __restrict__ u,
                                                  const int32_t* __restrict__ v, const double* __restrict__ w,
                                                  int check, int32_t* __restrict__ lcnt, int32_t* __restrict__ bad,
                                                  int32_t* __restrict__ lmax, int32_t* __restrict__ long_up) {
    __shared__ int32_t bmax;
    if (threadIdx.x == 0) bmax = 0;
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * (TB * PT) + threadIdx.x;
    int32_t a[PT], b[PT], reached = 0;
    bool far = false, wrong = false;
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int64_t e = t0 + i * TB;
        a[i] = e < m ? __ldg(u + e) : -1;
        b[i] = e < m ? __ldg(v + e) : -1;
        if (e < m && e >= ROW_PART_SHORT) far |= __ldg(u + e - ROW_PART_SHORT) == a[i];
    }
    if (check) {
        // positive and finite, on the weight's bits: FP64 compares would take
        // the FP64 pipe longer than the loads take
        int64_t wb[PT];
        int32_t pa[PT], pb[PT];
#pragma unroll
        for (int i = 0; i < PT; ++i) {
            const int64_t e = t0 + i * TB;
            wb[i] = e < m ? __ldg(reinterpret_cast<const long long*>(w) + e) : 1;
            pa[i] = e > 0 && e < m ? __ldg(u + e - 1) : -1;
            pb[i] = e > 0 && e < m ? __ldg(v + e - 1) : -1;
        }
#pragma unroll
        for (int i = 0; i < PT; ++i) {
            const bool ok = a[i] >= 0 && b[i] < n && a[i] < b[i] && wb[i] > 0 && wb[i] < 0x7ff0000000000000ll &&
                            (t0 + i * TB == 0 || pa[i] < a[i] || (pa[i] == a[i] && pb[i] < b[i]));
            if (t0 + i * TB < m && !ok) wrong = true;
        }
    }
    if (lcnt) {
#pragma unroll
        for (int i = 0; i < PT; ++i)
            if (b[i] >= 0 && b[i] < n) reached = max(reached, atomicAdd(&lcnt[b[i]], 1) + 1);
        reached = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)reached);
        if ((threadIdx.x & 31) == 0 && reached) atomicMax(&bmax, reached);
    }
    if (far) *long_up = 1;
    if (wrong) atomicExch(bad, 1);
    __syncthreads();
    if (threadIdx.x == 0 && bmax) atomicMax(lmax, bmax);
}

__global__ void k_row_total(const int32_t* __restrict__ lcnt, const int64_t* __restrict__ eptr, int64_t n,
                            int64_t* __restrict__ rowcnt) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) rowcnt[p] = (int64_t)lcnt[p] + (eptr[p + 1] - eptr[p]);
    else if (p == n) rowcnt[p] = 0;
}

// lower part of row v: edge ids in claim order (sorted by the row pass)
__global__ void k_lower_claim(const int32_t* __restrict__ ev, int64_t m, const int64_t* __restrict__ rowptr,
                              int32_t* __restrict__ lfill, int32_t* __restrict__ eid) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m) return;
    const int32_t b = ev[e];
    eid[rowptr[b] + atomicAdd(&lfill[b], 1)] = (int32_t)e;
}

// thread per row (graphs of mean degree below 32): insertion-sort the lower ids, write
// the row, D(p,p) summed sequentially in slot order (= ascending edge id),
// then w / D(p,p).  Rows with longer lower parts go to the warp kernel's list.
//
// A warp's 32 rows are consecutive, so their slots and their upper edges are
// two contiguous ranges.  When both fit the warp's shared-memory buffers (and
// no row of the warp is listed), the warp reads the claimed lower ids and the
// upper edges' ends and weights in whole lines, each thread builds its row in
// the buffers, and the warp writes the four slot arrays in whole lines; only
// the lower edges' own ends and weights are gathered.  Other warps write each
// row from its thread (the same values in the same order).
constexpr int FIN_CAP = 256;   // slots a warp stages
constexpr int FIN_ECAP = 160;  // upper edges a warp stages

__global__ void __launch_bounds__(TB, 4) k_row_finish_thread(int64_t n, const int64_t* __restrict__ rowptr,
                                                          const int64_t* __restrict__ eptr,
                                                          const int32_t* __restrict__ lcnt,
                                                          const int32_t* __restrict__ eu,
                                                          const int32_t* __restrict__ ev,
                                                          const double* __restrict__ ew, int32_t* __restrict__ col,
                                                          int32_t* __restrict__ eid, double* __restrict__ wn64,
                                                          int2* __restrict__ cw32, double* __restrict__ deg,
                                                          int32_t* __restrict__ list, int32_t* __restrict__ nlist) {
    __shared__ int32_t s_col[TB / 32][FIN_CAP];
    __shared__ int32_t s_eid[TB / 32][FIN_CAP];
    __shared__ double s_w[TB / 32][FIN_CAP];
    __shared__ int32_t s_ev[TB / 32][FIN_ECAP];
    __shared__ double s_ew[TB / 32][FIN_ECAP];
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t pw = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);  // the warp's first row
    if (pw >= n) return;                                                       // whole warp
    const int64_t p = pw + lane;
    const bool in = p < n;
    const int L = in ? lcnt[p] : 0;
    const bool listed = L > LOWER_THREAD;
    const int32_t k = warp_slot(listed, nlist);
    if (k >= 0) list[k] = (int32_t)p;
    int64_t r0 = 0, e0 = 0, e1 = 0;
    if (in) {
        r0 = rowptr[p];
        e0 = eptr[p];
        e1 = eptr[p + 1];
    }
    const int lv = (int)((n - pw < 32 ? n - pw : 32) - 1);  // the warp's last row
    const int64_t R0 = __shfl_sync(FULL, r0, 0), E0 = __shfl_sync(FULL, e0, 0);
    const int64_t E1 = __shfl_sync(FULL, e1, lv);
    const int64_t R1 = __shfl_sync(FULL, r0 + L + (e1 - e0), lv);
    const bool staged = !__any_sync(FULL, listed) && R1 - R0 <= FIN_CAP && E1 - E0 <= FIN_ECAP;
    if (staged) {
        int32_t* S_col = s_col[wp];
        int32_t* S_eid = s_eid[wp];
        double* S_w = s_w[wp];
        int32_t* S_ev = s_ev[wp];
        double* S_ew = s_ew[wp];
        const int ns = (int)(R1 - R0), ne = (int)(E1 - E0);
        for (int j = lane; j < ns; j += 32) S_eid[j] = eid[R0 + j];  // lower parts: ids in claim order
        for (int j = lane; j < ne; j += 32) {
            S_ev[j] = ev[E0 + j];
            S_ew[j] = ew[E0 + j];
        }
        __syncwarp();
        if (in) {
            const int b = (int)(r0 - R0), u0 = (int)(e0 - E0), U = (int)(e1 - e0);
            for (int i = 1; i < L; ++i) {
                const int32_t x = S_eid[b + i];
                int j = i;
                while (j > 0 && S_eid[b + j - 1] > x) {
                    S_eid[b + j] = S_eid[b + j - 1];
                    --j;
                }
                S_eid[b + j] = x;
            }
            double sum = 0.0;
            for (int i0 = 0; i0 < L; i0 += 4) {  // four lower edges' ends and weights in flight
                int32_t e4[4], c4[4];
                double w4[4];
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (i0 + t < L) {
                        e4[t] = S_eid[b + i0 + t];
                        w4[t] = ew[e4[t]];
                        c4[t] = eu[e4[t]];
                    }
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (i0 + t < L) {
                        S_col[b + i0 + t] = c4[t];
                        S_w[b + i0 + t] = w4[t];
                        sum += w4[t];
                    }
            }
            for (int i = 0; i < U; ++i) {
                const double w = S_ew[u0 + i];
                S_col[b + L + i] = S_ev[u0 + i];
                S_eid[b + L + i] = (int32_t)(e0 + i);
                S_w[b + L + i] = w;
                sum += w;
            }
            deg[p] = sum;
            const double inv = row_inverse(sum);
            for (int i = 0; i < L + U; ++i) S_w[b + i] = S_w[b + i] * inv;
        }
        __syncwarp();
        for (int j = lane; j < ns; j += 32) {
            const int32_t cj = S_col[j];
            const double x = S_w[j];
            col[R0 + j] = cj;
            eid[R0 + j] = S_eid[j];
            wn64[R0 + j] = x;
            cw32[R0 + j] = make_int2(cj, __float_as_int(f64_to_f32(x)));
        }
        return;
    }
    if (!in || listed) return;
    int32_t le[LOWER_THREAD];
    for (int i = 0; i < L; ++i) {
        const int32_t x = eid[r0 + i];
        int j = i;
        while (j > 0 && le[j - 1] > x) {
            le[j] = le[j - 1];
            --j;
        }
        le[j] = x;
    }
    double sum = 0.0;
    for (int i = 0; i < L; ++i) {
        const int32_t e = le[i];
        const double w = ew[e];
        col[r0 + i] = eu[e];
        eid[r0 + i] = e;
        wn64[r0 + i] = w;
        sum += w;
    }
    for (int64_t e = e0; e < e1; ++e) {
        const int64_t j = r0 + L + (e - e0);
        const double w = ew[e];
        col[j] = ev[e];
        eid[j] = (int32_t)e;
        wn64[j] = w;
        sum += w;
    }
    deg[p] = sum;
    const double inv = row_inverse(sum);
    const int64_t r1 = r0 + L + (e1 - e0);
    for (int64_t j = r0; j < r1; ++j) {
        const double x = wn64[j] * inv;
        wn64[j] = x;
        cw32[j] = make_int2(col[j], __float_as_int(f64_to_f32(x)));
    }
}

// warp per listed row (lower part longer than a thread sorts): lower ids
// bitonic-sorted in shared memory; D(p,p) as lane-strided sums in slot order
// combined by a fixed shuffle tree
__global__ void __launch_bounds__(FW * 32) k_row_finish_warp(
    const int32_t* __restrict__ list, const int32_t* __restrict__ nlist,
    const int64_t* __restrict__ rowptr, const int64_t* __restrict__ eptr, const int32_t* __restrict__ lcnt,
    const int32_t* __restrict__ eu, const int32_t* __restrict__ ev, const double* __restrict__ ew,
    int32_t* __restrict__ col, int32_t* __restrict__ eid, double* __restrict__ wn64, int2* __restrict__ cw32,
    double* __restrict__ deg) {
    __shared__ int32_t sh[FW][LOWER_WARP];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t* S = sh[w];
    const int64_t count = *nlist;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < count;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t p = list[r];
        const int L = lcnt[p];
        const int64_t r0 = rowptr[p], e0 = eptr[p], e1 = eptr[p + 1];
        const int P = L <= 1 ? 1 : 1 << (32 - __clz(L - 1));
        for (int t = lane; t < P; t += 32) S[t] = t < L ? eid[r0 + t] : 0x7fffffff;
        __syncwarp();
        for (int kk = 2; kk <= P; kk <<= 1)
            for (int j = kk >> 1; j > 0; j >>= 1) {
                for (int t = lane; t < P; t += 32) {
                    const int u2 = t ^ j;
                    if (u2 > t) {
                        const int32_t x = S[t], y = S[u2];
                        if ((x > y) == ((t & kk) == 0)) {
                            S[t] = y;
                            S[u2] = x;
                        }
                    }
                }
                __syncwarp();
            }
        const int64_t len = L + (e1 - e0);
        double sum = 0.0;
        for (int64_t i = lane; i < len; i += 32) {
            int32_t e, q;
            if (i < L) {
                e = S[i];
                q = eu[e];
            } else {
                e = (int32_t)(e0 + (i - L));
                q = ev[e];
            }
            const double wv = ew[e];
            col[r0 + i] = q;
            eid[r0 + i] = e;
            wn64[r0 + i] = wv;
            sum += wv;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) deg[p] = sum;
        const double inv = row_inverse(sum);
        for (int64_t i = lane; i < len; i += 32) {
            const double x = wn64[r0 + i] * inv;
            wn64[r0 + i] = x;
            cw32[r0 + i] = make_int2(col[r0 + i], __float_as_int(f64_to_f32(x)));
        }
        __syncwarp();
    }
}

// the canonical edge list's arrays
cudaError_t alloc_edges(gr_ctx* c, int64_t m) {
    const size_t me = (size_t)(m > 0 ? m : 1);
    SlabPlan sl;
    const size_t o_u = sl.add(sizeof(int32_t) * me), o_v = sl.add(sizeof(int32_t) * me),
                 o_w = sl.add(sizeof(double) * me);
    const cudaError_t e = cudaMallocAsync(&c->slab[0], sl.need, c->stream);
    if (e != cudaSuccess) {
        c->slab[0] = nullptr;
        return e;
    }
    c->eu = (int32_t*)((char*)c->slab[0] + o_u);
    c->ev = (int32_t*)((char*)c->slab[0] + o_v);
    c->ew = (double*)((char*)c->slab[0] + o_w);
    return cudaSuccess;
}

gr_status build_csr(gr_ctx* c, bool check, bool* invalid) {
    const int64_t n = c->n, m = c->m;
    cudaStream_t s = c->stream;
    if (invalid) *invalid = false;
    int64_t* hs = host_scratch();
    if (!hs) return set_error(c, GR_ENOMEM, "csr: pinned scratch unavailable");
    const size_t slots = (size_t)(2 * m > 0 ? 2 * m : 1) + CSR_PAD_SLOTS;
    SlabPlan sl;
    const size_t o_eptr = sl.add(sizeof(int64_t) * (size_t)(n + 1)),
                 o_row = sl.add(sizeof(int64_t) * (size_t)(n + 1 + CSR_PAD_ROWS)),
                 o_deg = sl.add(sizeof(double) * (size_t)(n > 0 ? n : 1)), o_col = sl.add(sizeof(int32_t) * slots),
                 o_eid = sl.add(sizeof(int32_t) * slots), o_cw = sl.add(sizeof(int2) * slots),
                 o_wn = sl.add(sizeof(double) * slots);
    GR_TRY_CUDA(c, cudaMallocAsync(&c->slab[1], sl.need, s), "alloc csr");
    char* base = (char*)c->slab[1];
    c->eptr = (int64_t*)(base + o_eptr);
    c->rowptr = (int64_t*)(base + o_row);
    c->deg = (double*)(base + o_deg);
    c->col = (int32_t*)(base + o_col);
    c->eid = (int32_t*)(base + o_eid);
    c->cw32 = (int2*)(base + o_cw);
    c->wn64 = (double*)(base + o_wn);

    // lcnt (n+1), lfill (n+1), list (n+1), flags (16 B)
    void *p_i32, *p_i64;
    const size_t R = (size_t)(n + 1);
    GR_TRY_CUDA(c, c->ws.get(WS_COARSE_TMP, sizeof(int32_t) * (3 * R + 4), &p_i32), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_C, sizeof(int64_t) * R, &p_i64), "ws");
    int32_t* lcnt = (int32_t*)p_i32;
    int32_t* lfill = lcnt + R;
    int32_t* list = lfill + R;
    int32_t* flags = list + R;  // [0] not canonical, [1] longest lower part, [2] listed rows, [3] long part
    // dense graphs (mean degree 32 or more): the global sort of the lower
    // parts beats per-row sorting of long lower parts, and gives their counts:
    // counting by atomics took 200 to 280 us a level of 13 to 16 M edges
    const bool sparse = 2 * m < 32 * n;
    if (sparse) GR_TRY_CUDA(c, cudaMemsetAsync(lcnt, 0, sizeof(int32_t) * (2 * R), s), "memset");
    GR_TRY_CUDA(c, cudaMemsetAsync(flags, 0, 16, s), "memset");
    if (m > 0 && (check || sparse)) {
        k_csr_count<<<(unsigned)ceil_div(m, TB * PT), TB, 0, s>>>(n, m, c->eu, c->ev, c->ew, check ? 1 : 0,
                                                            sparse ? lcnt : nullptr, flags, flags + 1, flags + 3);
        count_launch();
    }
    int32_t lmax = 0;
    if (check || sparse) {
        GR_TRY_CUDA(c, cudaMemcpyAsync(hs, flags, 16, cudaMemcpyDeviceToHost, s), "readback");
        GR_TRY_CUDA(c, cudaStreamSynchronize(s), "sync");
        const int32_t* hf = (const int32_t*)hs;
        if (hf[0]) {
            if (invalid) *invalid = true;
            return set_error(c, GR_EINVAL, "csr: the edge list is not canonical");
        }
        lmax = hf[1];
        if (sparse) c->parts = lmax <= ROW_PART_SHORT && !hf[3] ? 1 : 0;
        c->short_rows = check && c->parts == 1;
    }
    k_upper_ptr<<<(unsigned)ceil_div(m + 1, TB * PT), TB, 0, s>>>(c->eu, m, n, c->eptr); count_launch();
    if (!sparse || lmax > LOWER_WARP) {
        const gr_status st = build_csr_sorted(c, check && !sparse ? flags + 3 : nullptr);
        if (st != GR_OK || sparse || !check) return st;
        GR_TRY_CUDA(c, cudaMemcpyAsync(hs, flags, 16, cudaMemcpyDeviceToHost, s), "readback");
        GR_TRY_CUDA(c, cudaStreamSynchronize(s), "sync");
        c->short_rows = !((const int32_t*)hs)[3];
        c->parts = c->short_rows ? 1 : 0;
        return GR_OK;
    }
    int64_t* rowcnt = (int64_t*)p_i64;
    k_row_total<<<(unsigned)ceil_div(n + 1, TB), TB, 0, s>>>(lcnt, c->eptr, n, rowcnt); count_launch();
    GR_TRY_CUDA(c, scan_exclusive_i64(rowcnt, c->rowptr, n + 1, c->ws, s), "scan rowptr");
    if (m > 0) {
        k_lower_claim<<<(unsigned)ceil_div(m, TB), TB, 0, s>>>(c->ev, m, c->rowptr, lfill, c->eid);
        count_launch();
    }
    if (n > 0) {
        k_row_finish_thread<<<(unsigned)ceil_div(n, TB), TB, 0, s>>>(n, c->rowptr, c->eptr, lcnt, c->eu, c->ev,
                                                                   c->ew, c->col, c->eid, c->wn64, c->cw32, c->deg,
                                                                   list, flags + 2);
        count_launch();
        if (lmax > LOWER_THREAD) {
            k_row_finish_warp<<<(unsigned)(c->num_sms * 16), FW * 32, 0, s>>>(list, flags + 2, c->rowptr, c->eptr,
                                                                              lcnt, c->eu, c->ev, c->ew, c->col,
                                                                              c->eid, c->wn64, c->cw32, c->deg);
            count_launch();
        }
    }
    GR_TRY_CUDA(c, cudaGetLastError(), "csr kernels");
    return GR_OK;
}

// *longer = 1 if a row has more than ROW_PART_SHORT slots on a side of the diagonal
__global__ void k_row_parts(int64_t n, const int64_t* __restrict__ rowptr, const int64_t* __restrict__ eptr,
                            int64_t* __restrict__ longer) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t up = eptr[p + 1] - eptr[p], low = rowptr[p + 1] - rowptr[p] - up;
    if (up > ROW_PART_SHORT || low > ROW_PART_SHORT) *longer = 1;
}

cudaError_t parts_short(gr_ctx* c, bool* yes) {
    *yes = c->parts == 1;
    if (c->parts >= 0) return cudaSuccess;
    cudaStreamCaptureStatus cap;
    GR_CUDA(cudaStreamIsCapturing(c->stream, &cap));
    if (cap != cudaStreamCaptureStatusNone) return cudaSuccess;
    int64_t* hs = host_scratch();
    if (!hs) return cudaErrorMemoryAllocation;
    hs[0] = 0;
    if (c->n > 0) {
        k_row_parts<<<(unsigned)ceil_div(c->n, TB), TB, 0, c->stream>>>(c->n, c->rowptr, c->eptr, hs);
        count_launch();
    }
    GR_CUDA(cudaGetLastError());
    GR_CUDA(cudaStreamSynchronize(c->stream));
    c->parts = hs[0] ? 0 : 1;
    *yes = c->parts == 1;
    return cudaSuccess;
}

// Dense graphs, and rows with a lower part too long for one warp's shared
// memory: a stable radix sort of the edge ids by v lists every row's lower
// part in order.
gr_status build_csr_sorted(gr_ctx* c, int32_t* long_low) {
    const int64_t n = c->n, m = c->m;
    cudaStream_t s = c->stream;
    void *p_start, *p_k0, *p_v0, *p_alt;
    const size_t M = (size_t)(m > 0 ? m : 1);
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_C, sizeof(int64_t) * (size_t)(n + 1), &p_start), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_A, sizeof(uint32_t) * M, &p_k0), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_B, sizeof(uint32_t) * M, &p_v0), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_D, sizeof(uint32_t) * M * 2, &p_alt), "ws");
    int64_t* lstart = (int64_t*)p_start;
    uint32_t *k0 = (uint32_t*)p_k0, *v0 = (uint32_t*)p_v0;
    uint32_t *k1 = (uint32_t*)p_alt, *v1 = k1 + M;
    int alt = 0;
    if (m > 0) {
        GR_TRY_CUDA(c, radix_order_u32((const uint32_t*)c->ev, k0, v0, k1, v1, m, bits_for((uint64_t)(n - 1)), c->ws,
                                       s, &alt),
                    "sort by v");
    }
    const uint32_t* sk = alt ? k1 : k0;
    const uint32_t* sv = alt ? v1 : v0;
    k_lower_ptr<<<(unsigned)ceil_div(m + 1, TB * PT), TB, 0, s>>>(sk, m, n, c->eptr, lstart, c->rowptr, long_low);
    count_launch();
    if (m > 0 && 2 * m >= 32 * n) {
        const FinArrays A{sv, c->eu, c->ev, c->ew, c->col, c->eid, c->wn64, c->cw32};
        k_row_finish_sorted<<<(unsigned)ceil_div(n, FIN_ROWS), TB, 0, s>>>(n, c->rowptr, lstart, c->eptr, A, c->deg);
        count_launch();
    } else if (n > 0) {  // a few long rows among short ones
        k_fill_lower<<<(unsigned)ceil_div(m, TB), TB, 0, s>>>(sk, sv, m, lstart, c->rowptr, c->eu,
                                                              c->ew, c->col, c->eid, c->wn64); count_launch();
        k_fill_upper<<<(unsigned)ceil_div(m, TB), TB, 0, s>>>(c->eu, c->ev, c->ew, m, c->eptr, c->rowptr,
                                                              c->col, c->eid, c->wn64); count_launch();
        k_degree_scale_rows<<<(unsigned)ceil_div(n, TB), TB, 0, s>>>(c->rowptr, c->col, n, c->wn64, c->cw32,
                                                                     c->deg);
        count_launch();
    }
    GR_TRY_CUDA(c, cudaGetLastError(), "csr kernels");
    return GR_OK;
}

// ---------------------------------------------------------------------------
// Galerkin coarsening
// ---------------------------------------------------------------------------
// key of fine edge e = (min(A,B), max(A,B)), kb bits each (nc <= 2^kb); an edge
// inside one aggregate gets the sentinel, 2 kb ones: no pair, and after all.
__global__ void __launch_bounds__(TB) k_galerkin_keys(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                                                      const int32_t* __restrict__ agg, int64_t m, int kb,
                                                      uint64_t sentinel, uint64_t* __restrict__ keys) {
    const int64_t t0 = (int64_t)blockIdx.x * (TB * PT) + threadIdx.x;
    int32_t a[PT], b[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int64_t e = t0 + i * TB;
        a[i] = e < m ? __ldg(eu + e) : 0;
        b[i] = e < m ? __ldg(ev + e) : 0;
    }
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        a[i] = __ldg(agg + a[i]);
        b[i] = __ldg(agg + b[i]);
    }
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int64_t e = t0 + i * TB;
        if (e >= m) continue;
        const uint64_t lo = (uint32_t)min(a[i], b[i]), hi = (uint32_t)max(a[i], b[i]);
        keys[e] = lo == hi ? sentinel : lo << kb | hi;
    }
}

// Segments of equal keys in tiles of TB * PT keys, PT rounds of 32 a warp: a
// count of each tile's first keys, a scan of the counts, and the sums, which
// find their rank again by votes (a flag and a position per key, scanned in
// full, took 110 us more on 16 M edges).
constexpr int SEG_TILE = TB * PT;

// bit i: this thread's key of round i heads a segment
__device__ __forceinline__ unsigned seg_heads(const uint64_t* __restrict__ keys, int64_t m, uint64_t sentinel,
                                              int64_t w0, uint64_t (&k)[PT]) {
    const int lane = threadIdx.x & 31;
    unsigned h = 0;
    uint64_t prev[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int64_t t = w0 + 32 * i + lane;
        k[i] = t < m ? __ldg(keys + t) : sentinel;
        prev[i] = t > 0 && t < m ? __ldg(keys + t - 1) : sentinel;
    }
#pragma unroll
    for (int i = 0; i < PT; ++i)
        if (k[i] != sentinel && k[i] != prev[i]) h |= 1u << i;
    return h;
}

__global__ void __launch_bounds__(TB) k_segment_count(const uint64_t* __restrict__ keys, int64_t m, uint64_t sentinel,
                                                      int32_t* __restrict__ count) {
    __shared__ int32_t total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    uint64_t k[PT];
    const int64_t w0 = (int64_t)blockIdx.x * SEG_TILE + (threadIdx.x >> 5) * (32 * PT);
    const unsigned c = __reduce_add_sync(0xffffffffu, (unsigned)__popc(seg_heads(keys, m, sentinel, w0, k)));
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&total, (int32_t)c);
    __syncthreads();
    if (threadIdx.x == 0) count[blockIdx.x] = total;
}

// one thread per segment head: sum the segment's fine weights in sorted order
// (ascending fine edge id, the sort being stable) into the reduced edge.
__global__ void __launch_bounds__(TB) k_segment_sum(const uint64_t* __restrict__ keys,
                                                    const uint32_t* __restrict__ vals,
                                                    const int32_t* __restrict__ start, int64_t m, int kb,
                                                    uint64_t sentinel, const double* __restrict__ ew,
                                                    int32_t* __restrict__ uc, int32_t* __restrict__ vc,
                                                    double* __restrict__ wc) {
    __shared__ int32_t wcount[TB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)blockIdx.x * SEG_TILE + warp * (32 * PT);
    uint64_t k[PT];
    const unsigned h = seg_heads(keys, m, sentinel, w0, k);
    double sum[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) sum[i] = h >> i & 1u ? __ldg(ew + __ldg(vals + w0 + 32 * i + lane)) : 0.0;
    int32_t before[PT], c = 0;
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const unsigned b = __ballot_sync(0xffffffffu, h >> i & 1u);
        before[i] = c + __popc(b & ((1u << lane) - 1u));
        c += __popc(b);
    }
    if (lane == 0) wcount[warp] = c;
    __syncthreads();
    int64_t r0 = start[blockIdx.x];
    for (int w = 0; w < warp; ++w) r0 += wcount[w];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        if (!(h >> i & 1u)) continue;
        for (int64_t j = w0 + 32 * i + lane + 1; j < m && keys[j] == k[i]; ++j) sum[i] += ew[vals[j]];
        const int64_t r = r0 + before[i];
        uc[r] = (int32_t)(k[i] >> kb);
        vc[r] = (int32_t)(k[i] & ((1ull << kb) - 1ull));
        wc[r] = sum[i];
    }
}

__global__ void k_total_i32(const int32_t* __restrict__ count, const int32_t* __restrict__ pos,
                            int64_t len, int64_t* __restrict__ out) {
    *out = len > 0 ? (int64_t)pos[len - 1] + count[len - 1] : 0;
}

gr_status coarsen_impl(gr_ctx* c, const int32_t* agg, int64_t nc, gr_ctx** out) {
    const int64_t n = c->n, m = c->m;
    cudaStream_t s = c->stream;
    int64_t* hs = host_scratch();
    if (!hs) return set_error(c, GR_ENOMEM, "coarsen: pinned scratch unavailable");
    if (nc < 1 || nc > n) return set_error(c, GR_EINVAL, "coarsen: nc must be in [1, n]");
    if ((uint64_t)nc > (1ull << 31)) return set_error(c, GR_EINVAL, "coarsen: nc too large");

    gr_ctx* cc = new gr_ctx();
    cc->stream = s;
    cc->device = c->device;
    cc->num_sms = c->num_sms;
    cc->ws.stream = s;
    cc->n = nc;
    auto fail = [&](gr_status st) {
        graph_reduce_destroy(cc);
        return st;
    };
    // row-by-row assembly unless a coarse row is too long for shared memory
    bool too_long = false;
    {
        gr_status st = galerkin_rows(c, agg, nc, cc, &too_long);
        if (st != GR_OK) return fail(st);
        if (!too_long) {
            if (cudaMallocAsync(&cc->parent_map, sizeof(int32_t) * (size_t)(n > 0 ? n : 1), s) != cudaSuccess) {
                set_error(c, GR_ENOMEM, "coarsen: allocation failed");
                return fail(GR_ENOMEM);
            }
            GR_TRY_CUDA(c, cudaMemcpyAsync(cc->parent_map, agg, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice,
                                           s), "copy map");
            cc->parent_n = n;
            *out = cc;
            return GR_OK;
        }
    }
    // global sort path (the labels have been checked above)
    int64_t mc = 0;
    if (m > 0) {
        void *p_k, *p_v, *p_head;
        const int64_t tiles = ceil_div(m, SEG_TILE);
        GR_TRY_CUDA(c, c->ws.get(WS_COARSE_KEYS, sizeof(uint64_t) * (size_t)m * 2, &p_k), "ws");
        GR_TRY_CUDA(c, c->ws.get(WS_COARSE_VALS, sizeof(uint32_t) * (size_t)m * 2, &p_v), "ws");
        GR_TRY_CUDA(c, c->ws.get(WS_SORT_A, sizeof(int32_t) * (size_t)tiles * 2, &p_head), "ws");
        uint64_t* k0 = (uint64_t*)p_k;
        uint64_t* k1 = k0 + m;
        uint32_t* v0 = (uint32_t*)p_v;
        uint32_t* v1 = v0 + m;
        int32_t* head = (int32_t*)p_head;
        int32_t* hpos = head + tiles;
        int kb = bits_for((uint64_t)(nc - 1));
        if (kb < 1) kb = 1;
        const uint64_t sentinel = (1ull << (2 * kb)) - 1ull;
        k_galerkin_keys<<<(unsigned)ceil_div(m, TB * PT), TB, 0, s>>>(c->eu, c->ev, agg, m, kb, sentinel, k0);
        count_launch();
        int alt = 0;
        GR_TRY_CUDA(c, radix_order_u64(k0, k0, v0, k1, v1, m, 2 * kb, c->ws, s, &alt), "sort keys");
        const uint64_t* sk = alt ? k1 : k0;
        const uint32_t* sv = alt ? v1 : v0;
        k_segment_count<<<(unsigned)tiles, TB, 0, s>>>(sk, m, sentinel, head); count_launch();
        GR_TRY_CUDA(c, scan_exclusive_i32(head, hpos, tiles, c->ws, s), "scan heads");
        k_total_i32<<<1, 1, 0, s>>>(head, hpos, tiles, hs); count_launch();
        GR_TRY_CUDA(c, cudaGetLastError(), "galerkin kernels");
        GR_TRY_CUDA(c, cudaStreamSynchronize(s), "sync");
        mc = hs[0];
        cc->m = mc;
        if (alloc_edges(cc, mc) != cudaSuccess) {
            set_error(c, GR_ENOMEM, "coarsen: allocation failed");
            return fail(GR_ENOMEM);
        }
        k_segment_sum<<<(unsigned)tiles, TB, 0, s>>>(sk, sv, hpos, m, kb, sentinel, c->ew, cc->eu, cc->ev, cc->ew);
        count_launch();
        GR_TRY_CUDA(c, cudaGetLastError(), "segment sum");
    } else {
        cc->m = 0;
        if (alloc_edges(cc, 0) != cudaSuccess) {
            set_error(c, GR_ENOMEM, "coarsen: allocation failed");
            return fail(GR_ENOMEM);
        }
    }
    // in this graph's scratch: the coarse graph is smaller
    std::swap(c->ws, cc->ws);
    gr_status st = build_csr(cc, false, nullptr);
    std::swap(c->ws, cc->ws);
    if (st != GR_OK) {
        set_error(c, st, "coarsen: " + cc->last_error);
        return fail(st);
    }
    if (cudaMallocAsync(&cc->parent_map, sizeof(int32_t) * (size_t)(n > 0 ? n : 1), s) != cudaSuccess) {
        set_error(c, GR_ENOMEM, "coarsen: allocation failed");
        return fail(GR_ENOMEM);
    }
    GR_TRY_CUDA(c, cudaMemcpyAsync(cc->parent_map, agg, sizeof(int32_t) * (size_t)n,
                                   cudaMemcpyDeviceToDevice, s), "copy map");
    cc->parent_n = n;
    *out = cc;
    return GR_OK;
}

// ---------------------------------------------------------------------------
// Map composition (fine -> coarsest)
// ---------------------------------------------------------------------------
__global__ void k_compose(MapChain chain, int64_t n, int32_t* __restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t x = (int32_t)i;
    for (int l = 0; l < chain.count; ++l) x = chain.map[l][x];
    out[i] = x;
}

gr_status map_chain(gr_ctx* const* levels, int nlevels, MapChain* out) {
    gr_ctx* c0 = levels[0];
    if (nlevels > 64) return set_error(c0, GR_EINVAL, "compose: at most 64 levels");
    MapChain& ch = *out;
    ch.count = nlevels;
    for (int l = 0; l < nlevels; ++l) {
        if (!levels[l] || !levels[l]->parent_map)
            return set_error(c0, GR_ESTATE, "compose: every level must come from coarsen");
        if (l > 0 && levels[l]->parent_n != levels[l - 1]->n)
            return set_error(c0, GR_EINVAL, "compose: levels do not chain");
        ch.map[l] = levels[l]->parent_map;
    }
    return GR_OK;
}

gr_status compose_impl(gr_ctx* const* levels, int nlevels, int32_t* out) {
    gr_ctx* c0 = levels[0];
    MapChain ch;
    const gr_status st = map_chain(levels, nlevels, &ch);
    if (st != GR_OK) return st;
    int64_t n = c0->parent_n;
    if (n > 0) {
        k_compose<<<(unsigned)ceil_div(n, TB), TB, 0, c0->stream>>>(ch, n, out);
        count_launch();
    }
    GR_TRY_CUDA(c0, cudaGetLastError(), "compose");
    return GR_OK;
}

}  // namespace gr
