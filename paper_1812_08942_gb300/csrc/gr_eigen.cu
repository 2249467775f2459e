// Multilevel Laplacian eigensolver (Alg. 5, Sec. 4.1; Eqs. equ:lgl, equ:lgs).
//
// Coarsest level: the first k eigenpairs of L u = lambda B u (B = I ratio
// cut, B = D normalised cut, each level's own; or the Galerkin-consistent
// mass B_l = P^T B_(l-1) P carried from the finest I or D) from a
// Chebyshev-filtered subspace iteration on the coarsest graph
// (gr_chfsi.cu).  Then, level by level toward the finest: U_fine = P U_coarse (the parent map), and `iters` weighted-Jacobi
// iterations on (L - lambda_k B) y = 0 for every column k, the shift being the
// coarsest eigenvalue.  Finally modified Gram-Schmidt over the columns.  Every
// reduction is FP64 with a fixed summation order (per-block partials, then a
// last-block finish), so results are reproducible.
#include <vector>

#include "gr_ieee.cuh"
#include "gr_internal.cuh"
#include "gr_sweep.cuh"

namespace gr {

namespace {

constexpr int ET = 256;

// U_fine[i, :] = U_coarse[map[i], :]  (H = P, Alg. 5 step 5)
__global__ void k_prolong(int64_t n, int k, const int32_t* __restrict__ map, const double* __restrict__ Uc,
                          double* __restrict__ Uf) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * k) return;
    const int64_t i = idx / k;
    const int c = (int)(idx % k);
    Uf[idx] = Uc[(int64_t)map[i] * k + c];
}

// Weighted-Jacobi iteration on (L - lambda_c B) y = 0 for every column c:
//   y <- (1 - w) y + w (A y)_r / (D_r - lambda_c B_r),
// with (A y)_r = D_r (D^-1 A y)_r from the row-scaled weights and B the
// diagonal mass b (NULL: B = I); a row whose shifted diagonal is not positive
// keeps its value.  The gain g_rc = w D_r / (D_r - lambda_c B_r) depends only
// on the level, so it is computed once per level (g = -1: the row keeps its
// value; otherwise g >= 0) and an iteration is
//   y <- (1 - w) y + g (D^-1 A y)_r:
// FP64 runs at a small fraction of the FP32 rate on this part, and the
// division, taken per entry and iteration, cost more than the row's
// products.  The division of the gains runs on the integer pipe, bit for bit
// the same; both tests of a sign are integer compares (a floating compare
// would take the FP64 pipe too).
__global__ void k_shift_gain(int64_t n, int k, const double* __restrict__ deg, const double* __restrict__ lam,
                             const double* __restrict__ b, double omega, double* __restrict__ g) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * k) return;
    const int64_t r = idx / k;
    const int c = (int)(idx % k);
    const double D = deg[r];
    const double diag = D - lam[c] * (b ? b[r] : 1.0);
    const bool positive = ieee_bits(diag) - 1 < 0x7ff0000000000000ull;  // and not NaN
    g[idx] = positive ? ieee_div(omega * D, diag) : -1.0;
}

// One iteration, thread per (row, column).
__global__ void k_shifted_jacobi(int64_t n, int k, const int64_t* __restrict__ rowptr,
                                 const int32_t* __restrict__ col, const double* __restrict__ wn64,
                                 const double* __restrict__ gain, double omega, const double* __restrict__ Yin,
                                 double* __restrict__ Yout) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * k) return;
    const int64_t r = idx / k;
    const int c = (int)(idx % k);
    const double y = Yin[idx];
    const double g = gain[idx];
    if (__double2hiint(g) < 0) {
        Yout[idx] = y;
        return;
    }
    double s = 0.0;
    for (int64_t j = rowptr[r]; j < rowptr[r + 1]; ++j) s += wn64[j] * Yin[(int64_t)col[j] * k + c];
    Yout[idx] = fma(g, s, (1.0 - omega) * y);
}

// The same iteration with G lanes per row, each holding one 16-byte chunk
// (two columns) of the row: the slot entries are read once per lane group and
// each neighbour row is gathered chunk-wise; rows in grid-stride order.
template <int K>
__global__ void __launch_bounds__(ET) k_shifted_jacobi_rows(int64_t n64, const int64_t* __restrict__ rowptr,
                                                           const int32_t* __restrict__ col,
                                                           const double* __restrict__ wn64,
                                                           const double* __restrict__ gain, double omega,
                                                           const double* __restrict__ Yin,
                                                           double* __restrict__ Yout) {
    constexpr int E = K >= 2 ? 2 : 1, G = K / E, RPW = 32 / G;
    const int64_t n = n64;
    const int lane = threadIdx.x & 31, seg = lane / G, q = lane % G;
    if (seg >= RPW) return;
    const int64_t stride = (((int64_t)gridDim.x * blockDim.x) >> 5) * RPW;
    for (int64_t r = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * RPW + seg; r < n; r += stride) {
        double acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = 0.0;
        const int64_t j1 = rowptr[r + 1];
        // two neighbour chunks in flight per step
        for (int64_t j = rowptr[r]; j < j1; j += 2) {
            const bool two = j + 1 < j1;
            const double w0 = wn64[j], w1 = two ? wn64[j + 1] : 0.0;
            const double* s0 = Yin + (int64_t)col[j] * K + q * E;
            const double* s1 = Yin + (int64_t)col[two ? j + 1 : j] * K + q * E;
            if constexpr (E == 2) {
                const double2 x0 = __ldg(reinterpret_cast<const double2*>(s0));
                const double2 x1 = __ldg(reinterpret_cast<const double2*>(s1));
                acc[0] = fma(w0, x0.x, acc[0]);
                acc[1] = fma(w0, x0.y, acc[1]);
                if (two) {
                    acc[0] = fma(w1, x1.x, acc[0]);
                    acc[1] = fma(w1, x1.y, acc[1]);
                }
            } else {
                const double x0 = __ldg(s0), x1 = __ldg(s1);
                acc[0] = fma(w0, x0, acc[0]);
                if (two) acc[0] = fma(w1, x1, acc[0]);
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int c = q * E + e;
            const double y = Yin[r * K + c];
            const double g = gain[r * K + c];
            Yout[r * K + c] = __double2hiint(g) >= 0 ? fma(g, acc[e], (1.0 - omega) * y) : y;
        }
    }
}

// finest-level mass: 1 (ratio cut) or the degree, 1 for a degree-0 node
__global__ void k_base_mass(int64_t n, const double* __restrict__ deg, int normalized, double* __restrict__ b) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = normalized ? (deg[i] > 0.0 ? deg[i] : 1.0) : 1.0;
}

// ---------------------------------------------------------------------------
// Modified Gram-Schmidt in column order, right-looking: step j finishes
// column j, whose products with the columns after it are then known, and step
// j + 1 subtracts its share from all of them in the same pass that makes the
// next products: k passes instead of k (k + 1) / 2 pairs of them.  Column-by-
// column MGS (each column loses its parts along 0, 1, ... in that order) with
// the normalisation put off: columns stay as they are, their products are
// divided by the squared norm, and the last pass scales; the results are equal
// up to rounding.  A thread holds a row, columns are
// stored one after the other (coalesced; the first pass reads the row-major
// block and the last writes it), and only the columns that are left are
// touched.  Bound by the FP64 pipe, k (k + 1) multiply-adds a row (2,097,152 x
// 8: 285 us at 530 G a second): dots, axpys, divisions and transposes apart
// took 1,450 us, the passes and the final scaling take 550.
// ---------------------------------------------------------------------------
constexpr int MG_BLOCKS = 4;  // per SM
constexpr int RQ_EDGES = 64;  // consecutive edges of a Rayleigh quotient a thread takes at a time

// Step with R columns left, of which `left` (<= R) exist: V points at the first
// of them, prev (NULL: step 0, the columns come from row-major Y) holds the
// products of the column before it, prev[0] its squared norm.  R is the
// register width: a column guarded at run time would still take its turn on
// the FP64 pipe.
template <int R>
__global__ void __launch_bounds__(ET, R <= 8 ? MG_BLOCKS : 1) k_mgs_step(int64_t n, int left,
                                                                        const double* __restrict__ Y, double* V,
                                                                        const double* __restrict__ prev,
                                                                        double* part, unsigned* counter,
                                                                        double* __restrict__ sums) {
    constexpr int NS = R <= 2 ? 2 : (R + 1) / 2 * 2;
    __shared__ double red[ET];
    __shared__ double ws[ET / 32][NS];
    double acc[R], f[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        acc[i] = 0.0;
        f[i] = prev && i < left ? prev[i + 1] / prev[0] : 0.0;
    }
    for (int64_t r = (int64_t)blockIdx.x * ET + threadIdx.x; r < n; r += (int64_t)gridDim.x * ET) {
        double v[R];
        if (!prev) {
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = i < left ? Y[r * left + i] : 0.0;
        } else {
            const double p = V[r - n];
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = i < left ? V[(int64_t)i * n + r] : 0.0;
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = fma(-f[i], p, v[i]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            if (i < left) V[(int64_t)i * n + r] = v[i];
            acc[i] = fma(v[0], v[i], acc[i]);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        double t = acc[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) ws[warp][i] = t;
    }
    __syncthreads();
    if (threadIdx.x < NS) {
        double t = 0.0;
        if (threadIdx.x < R)
            for (int w = 0; w < ET / 32; ++w) t += ws[w][threadIdx.x];
        part[(int64_t)blockIdx.x * NS + threadIdx.x] = t;
    }
    __threadfence();
    __syncthreads();
    if (finish_partials<NS / 2, ET>(part, gridDim.x, counter, red) && (int)threadIdx.x < left)
        sums[threadIdx.x] = red[threadIdx.x];
}

// U (row-major) = the finished columns over their norms: the first sum of a
// column's step is its squared norm.  One rounding an entry: the division runs
// on the integer pipe (times a reciprocal, rounded twice: the same time).
__global__ void __launch_bounds__(ET) k_mgs_take(int64_t n, int k, const double* __restrict__ V,
                                                 const double* __restrict__ sums, int ld, double* __restrict__ U) {
    __shared__ double norm[32];
    if ((int)threadIdx.x < k) norm[threadIdx.x] = sqrt(sums[threadIdx.x * ld]);
    __syncthreads();
    for (int64_t r = (int64_t)blockIdx.x * ET + threadIdx.x; r < n; r += (int64_t)gridDim.x * ET)
        for (int i = 0; i < k; ++i) U[r * k + i] = ieee_div(V[(int64_t)i * n + r], norm[i]);
}

// x' L x and x' B x of every column: thread per (row, column) over the row's
// upper edges, w (x_u - x_v)^2, and b x^2 (b NULL: 1).  Column-wise passes
// over the edge list gathered 8 bytes at a time.  Bound by the FP64 pipe
// (three operations per edge and column).  LISTED (graphs that may have long
// rows): the edges in blocks of 64 of the canonical list, the first end's
// entry loaded again where it changes; by rows, a hub of 1,000,000 edges took
// 344 ms.  out[2 c] and out[2 c + 1].
template <bool LISTED>
__global__ void __launch_bounds__(ET) k_rayleigh(int64_t n, int k, int64_t m, const int64_t* __restrict__ eptr,
                                                 const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                                                 const double* __restrict__ ew, const double* __restrict__ b,
                                                 const double* __restrict__ U, double* part, unsigned* counter,
                                                 double* __restrict__ out) {
    __shared__ double red[ET], s1[ET], s2[ET];
    const int rpb = ET / k, c = threadIdx.x % k, rt = threadIdx.x / k;
    double num = 0.0, den = 0.0;
    // edges [e0, e1), four in flight; `cur` is the node whose entry is x
    auto edges = [&](int64_t e0, int64_t e1, int32_t cur, double x) {
        constexpr int W = 4;
        for (int64_t e = e0; e < e1; e += W) {
            int32_t p[W];
            double y[W], w[W];
#pragma unroll
            for (int u = 0; u < W; ++u)
                if (e + u < e1) {
                    if (LISTED) p[u] = __ldg(eu + e + u);
                    y[u] = U[(int64_t)__ldg(ev + e + u) * k + c];
                    w[u] = __ldg(ew + e + u);
                }
#pragma unroll
            for (int u = 0; u < W; ++u)
                if (e + u < e1) {
                    if (LISTED && p[u] != cur) x = U[(int64_t)(cur = p[u]) * k + c];
                    const double d = x - y[u];
                    num = fma(w[u] * d, d, num);
                }
        }
    };
    if (rt < rpb) {
        const int64_t first = (int64_t)blockIdx.x * rpb + rt, stride = (int64_t)gridDim.x * rpb;
        if constexpr (LISTED)
            for (int64_t e = first * RQ_EDGES; e < m; e += stride * RQ_EDGES)
                edges(e, e + RQ_EDGES < m ? e + RQ_EDGES : m, -1, 0.0);
        for (int64_t r = first; r < n; r += stride) {
            const double x = U[r * k + c];
            if constexpr (!LISTED) edges(eptr[r], eptr[r + 1], (int32_t)r, x);
            den = fma(b ? b[r] * x : x, x, den);
        }
    }
    s1[threadIdx.x] = num;
    s2[threadIdx.x] = den;
    __syncthreads();
    if (threadIdx.x < 64) {  // sum 2 q + 0 / 1 of column q
        const int q = threadIdx.x >> 1;
        const double* s = (threadIdx.x & 1) ? s2 : s1;
        double t = 0.0;
        if (q < k)
            for (int i = 0; i < rpb; ++i) t += s[i * k + q];
        part[(int64_t)blockIdx.x * 64 + threadIdx.x] = t;
    }
    __threadfence();
    __syncthreads();
    if (finish_partials<32, ET>(part, gridDim.x, counter, red) && (int)threadIdx.x < 2 * k)
        out[threadIdx.x] = red[threadIdx.x];
}

}  // namespace

gr_status eigensolve_impl(gr_ctx* const* levels, int nlevels, int k, int normalized, int galerkin_mass,
                          double omega, int iters, double* U_out, double* lambda_out, double* rayleigh_out) {
    gr_ctx* f = levels[0];
    gr_ctx* c = levels[nlevels - 1];
    cudaStream_t s = f->stream;
    const int64_t n0 = f->n;
    auto blocks = [](int64_t work) { return (unsigned)ceil_div(work > 0 ? work : 1, ET); };

    // scratch: two n x k blocks at the finest size, column-major copy,
    // reduction partials, scalars
    int64_t nmax = 0;
    for (int l = 0; l < nlevels; ++l) nmax = levels[l]->n > nmax ? levels[l]->n : nmax;
    int RB = f->num_sms * MG_BLOCKS;  // blocks of the reductions
    if (RB > STATS_GROUP * STATS_MAX_GROUPS) RB = STATS_GROUP * STATS_MAX_GROUPS;
    size_t need = 0;
    auto add = [&](size_t bytes) {
        size_t off = need;
        need += (bytes + 255) & ~size_t(255);
        return off;
    };
    const size_t o_Y0 = add(sizeof(double) * (size_t)nmax * k), o_Y1 = add(sizeof(double) * (size_t)nmax * k),
                 o_G = add(sizeof(double) * (size_t)nmax * k),
                 o_V = add(sizeof(double) * (size_t)n0 * k), o_sums = add(sizeof(double) * 32 * (size_t)k),
                 o_part = add(sizeof(double) * 64 * (size_t)RB), o_sc = add(sizeof(double) * 64),
                 o_lam = add(sizeof(double) * 32), o_ctr = add(STATS_COUNTER_BYTES);
    // Galerkin masses of every level: b_0 = 1 or D (degree 0 -> 1), then the
    // member sums level by level
    std::vector<size_t> o_mass;
    if (galerkin_mass)
        for (int l = 0; l < nlevels; ++l) o_mass.push_back(add(sizeof(double) * (size_t)(levels[l]->n > 0 ? levels[l]->n : 1)));
    void* base;
    GR_TRY_CUDA(f, f->ws.get(WS_EIG, need, &base), "eigensolver scratch");
    char* Bp = (char*)base;
    double* Y[2] = {(double*)(Bp + o_Y0), (double*)(Bp + o_Y1)};
    double* gain = (double*)(Bp + o_G);
    double* V = (double*)(Bp + o_V);
    double* sums = (double*)(Bp + o_sums);  // per step: the products of its column with those from it on
    double* part = (double*)(Bp + o_part);
    double* sc = (double*)(Bp + o_sc);
    double* lam = (double*)(Bp + o_lam);
    unsigned* ctr = (unsigned*)(Bp + o_ctr);
    GR_TRY_CUDA(f, cudaMemsetAsync(ctr, 0, STATS_COUNTER_BYTES, s), "memset");
    // the diagonal mass of each level (NULL: B = I)
    std::vector<const double*> mass(nlevels, nullptr);
    if (galerkin_mass) {
        double* b0 = (double*)(Bp + o_mass[0]);
        k_base_mass<<<blocks(n0), ET, 0, s>>>(n0, f->deg, normalized, b0);
        count_launch();
        mass[0] = b0;
        for (int l = 1; l < nlevels; ++l) {
            double* bl = (double*)(Bp + o_mass[l]);
            gr_ctx* const one[1] = {levels[l]};
            const gr_status st = reduce_data_impl(one, 1, mass[l - 1], 1, 1, 0, bl);
            if (st != GR_OK) return set_error(f, st, "eigensolve: Galerkin mass: " + levels[l]->last_error);
            mass[l] = bl;
        }
    } else if (normalized) {
        for (int l = 0; l < nlevels; ++l) mass[l] = levels[l]->deg;
    }

    // 1) coarsest eigenpairs (Alg. 5 step 2, Eq. equ:lgs)
    int cur = 0;
    {
        const gr_status st = coarsest_eigenpairs(c, mass[nlevels - 1], k, f->ws, s, lam, lambda_out, Y[cur], nullptr);
        if (st != GR_OK) return set_error(f, st, c->last_error);
    }

    // 2) map and smooth, level by level (Alg. 5 steps 4-10)
    for (int l = nlevels - 2; l >= 0; --l) {
        gr_ctx* g = levels[l];
        const int64_t n = g->n;
        k_prolong<<<blocks(n * k), ET, 0, s>>>(n, k, levels[l + 1]->parent_map, Y[cur], Y[cur ^ 1]);
        count_launch();
        cur ^= 1;
        if (iters > 0) {
            k_shift_gain<<<blocks(n * k), ET, 0, s>>>(n, k, g->deg, lam, mass[l], omega, gain);
            count_launch();
        }
        for (int it = 0; it < iters; ++it) {
            const unsigned gr = (unsigned)(f->num_sms * 8);
#define GR_SJ_ROWS(KK)                                                                                    \
    k_shifted_jacobi_rows<KK><<<gr, ET, 0, s>>>(n, g->rowptr, g->col, g->wn64, gain, omega, Y[cur], Y[cur ^ 1])
            switch (k) {
                case 2: GR_SJ_ROWS(2); break;
                case 4: GR_SJ_ROWS(4); break;
                case 8: GR_SJ_ROWS(8); break;
                case 16: GR_SJ_ROWS(16); break;
                case 32: GR_SJ_ROWS(32); break;
                default:
                    k_shifted_jacobi<<<blocks(n * k), ET, 0, s>>>(n, k, g->rowptr, g->col, g->wn64, gain, omega,
                                                                Y[cur], Y[cur ^ 1]);
            }
#undef GR_SJ_ROWS
            count_launch();
            cur ^= 1;
        }
    }

    // 3) modified Gram-Schmidt over the columns (Alg. 5 step 11)
    const int64_t rbw = ceil_div(n0 > 0 ? n0 : 1, ET);
    const unsigned rb = (unsigned)(RB < rbw ? RB : rbw);
    for (int j = 0; j < k; ++j) {
        const double* prev = j > 0 ? sums + (size_t)(j - 1) * 32 : nullptr;
        double* Vj = V + (int64_t)j * n0;
        const int left = k - j;
#define GR_MGS(RR) k_mgs_step<RR><<<rb, ET, 0, s>>>(n0, left, Y[cur], Vj, prev, part, ctr, sums + (size_t)j * 32)
        switch (left) {
            case 1: GR_MGS(1); break;
            case 2: GR_MGS(2); break;
            case 3: GR_MGS(3); break;
            case 4: GR_MGS(4); break;
            case 5: GR_MGS(5); break;
            case 6: GR_MGS(6); break;
            case 7: GR_MGS(7); break;
            case 8: GR_MGS(8); break;
            default:
                if (left <= 12) GR_MGS(12);
                else if (left <= 16) GR_MGS(16);
                else if (left <= 24) GR_MGS(24);
                else GR_MGS(32);
        }
#undef GR_MGS
        count_launch();
    }
    k_mgs_take<<<rb, ET, 0, s>>>(n0, k, V, sums, 32, U_out);
    count_launch();

    // 4) Rayleigh quotients of the result, x' L x / x' B x
    if (rayleigh_out) {
        bool short_parts;
        GR_TRY_CUDA(f, parts_short(f, &short_parts), "row lengths");
        const int64_t items = !short_parts && ceil_div(f->m, RQ_EDGES) > n0 ? ceil_div(f->m, RQ_EDGES) : n0;
        const int64_t qbw = ceil_div(items > 0 ? items : 1, ET / k);
        auto rayleigh = [&](auto kern) {
            kern<<<(unsigned)(RB < qbw ? RB : qbw), ET, 0, s>>>(n0, k, f->m, f->eptr, f->eu, f->ev, f->ew,
                                                                normalized ? f->deg : nullptr, U_out, part, ctr, sc);
        };
        short_parts ? rayleigh(k_rayleigh<false>) : rayleigh(k_rayleigh<true>);
        count_launch();
        int64_t* hs = host_scratch();
        if (!hs) return set_error(f, GR_ENOMEM, "eigensolve: pinned scratch unavailable");
        double* hq = (double*)hs;  // 64 B: up to 4 pairs at a time
        for (int i0 = 0; i0 < k; i0 += 4) {
            const int cnt = k - i0 < 4 ? k - i0 : 4;
            GR_TRY_CUDA(f, cudaMemcpyAsync(hq, sc + 2 * i0, sizeof(double) * 2 * cnt, cudaMemcpyDeviceToHost, s),
                        "readback");
            GR_TRY_CUDA(f, cudaStreamSynchronize(s), "sync");
            for (int t = 0; t < cnt; ++t) rayleigh_out[i0 + t] = hq[2 * t] / hq[2 * t + 1];
        }
    }
    GR_TRY_CUDA(f, cudaGetLastError(), "eigensolve kernels");
    GR_TRY_CUDA(f, cudaStreamSynchronize(s), "sync");
    return GR_OK;
}

}  // namespace gr
