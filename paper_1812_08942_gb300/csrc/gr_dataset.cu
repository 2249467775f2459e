// Reduced data set F_R = H_G^R F (Alg. 6, step 4) with H_G^R = P^T composed
// over the levels: row A of F_R is the sum (or, on request, the mean) of the
// rows of the fine nodes that end in coarsest aggregate A.  The members of
// every aggregate are listed in ascending id (gr_group.cu) and added in that
// order (FP64 accumulation).
#include "gr_internal.cuh"
#include "gr_vec.cuh"

namespace gr {

namespace {

constexpr int DT = 256;

__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) { return f32_to_f64(x); }

// Thread per (aggregate, column): the members' entries added one by one, eight
// loads in flight.  Bound by the FP64 pipe: one addition per entry at 530 G a
// second (63 us for 2,097,152 rows of 16 columns, which takes 92); FP32
// entries are widened with integer operations, since conversions share that
// pipe and doubled its work (168 us, one load at a time 170).
template <typename T>
__global__ void __launch_bounds__(DT) k_segment_rows(int64_t nc, int d, const int32_t* __restrict__ start,
                                                     const uint32_t* __restrict__ mem, const T* __restrict__ F,
                                                     int mean, T* __restrict__ out) {
    constexpr int U = 8;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nc * d) return;
    const int64_t A = idx / d;
    const int j = (int)(idx - A * d);
    const int32_t b = start[A], e = start[A + 1];
    double s = 0.0;
    int32_t t = b;
    for (; t + U <= e; t += U) {
        T x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = __ldg(F + (int64_t)__ldg(mem + t + u) * d + j);
#pragma unroll
        for (int u = 0; u < U; ++u) s += widen(x[u]);
    }
    if (t < e) {
        T x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t + u < e) x[u] = __ldg(F + (int64_t)__ldg(mem + t + u) * d + j);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t + u < e) s += widen(x[u]);
    }
    if (mean && e > b) s = s / (double)(e - b);
    out[idx] = (T)s;
}

}  // namespace

gr_status reduce_data_impl(gr_ctx* const* levels, int nlevels, const void* F, int d, int f64, int mean,
                           void* F_out) {
    gr_ctx* c0 = levels[0];
    cudaStream_t s = c0->stream;
    const int64_t n = c0->parent_n, nc = levels[nlevels - 1]->n;
    MapChain ch;
    gr_status st = map_chain(levels, nlevels, &ch);
    if (st != GR_OK) return st;
    GroupJob job;
    bool bad = false;
    st = group_begin(c0, WS_DATASET, ch, n, nc, &job);
    if (st == GR_OK) st = group_finish(c0, &job, &bad);
    if (st != GR_OK) return st;
    if (bad) return set_error(c0, GR_ECUDA, "reduce_data: composed map out of range");
    if (nc > 0 && d > 0) {
        if (f64) {
            k_segment_rows<double><<<(unsigned)ceil_div(nc * d, DT), DT, 0, s>>>(
                nc, d, job.start, job.members, (const double*)F, mean, (double*)F_out);
        } else {
            k_segment_rows<float><<<(unsigned)ceil_div(nc * d, DT), DT, 0, s>>>(
                nc, d, job.start, job.members, (const float*)F, mean, (float*)F_out);
        }
        count_launch();
    }
    GR_TRY_CUDA(c0, cudaGetLastError(), "reduce_data kernels");
    return GR_OK;
}

}  // namespace gr
