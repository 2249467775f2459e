// Members of every label of a node map, in ascending node id: what the
// aggregate means of the loss and the reduced data set add up, in that order.
//
// One pass counts the labels and keeps each node's place among its label's
// claims (the counter's old value), a scan turns the counts into starts, the
// nodes are written to start + place, and a warp per label sorts its list.
// Atomic claims and short sorts replace a radix sort of all nodes by label
// (two passes of histogram, three scan kernels and scatter for 2^15 labels):
// 2,097,152 nodes into 32,768 labels in 58 us of kernels against 103, and 7
// launches against 16.
// Labels with more than GROUP_SORT_MAX members (a map onto few nodes) take
// that radix sort: one warp would sort such a list for too long.
#include "gr_internal.cuh"

namespace gr {

namespace {

constexpr int QT = 256;
constexpr int GROUP_SORT_MAX = 1024;

__device__ __forceinline__ int32_t chain_label(const MapChain& ch, int64_t i) {
    int32_t x = (int32_t)i;
    for (int l = 0; l < ch.count; ++l) x = ch.map[l][x];
    return x;
}

// per node (label, place among the label's claims); flags: [0] a label
// outside [0, nc), [1] the largest group
__global__ void __launch_bounds__(QT) k_group_count(MapChain ch, int64_t n, int64_t nc, int32_t* __restrict__ cnt,
                                                    int2* __restrict__ place, int32_t* __restrict__ flags) {
    __shared__ int32_t bmax;
    if (threadIdx.x == 0) bmax = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    int32_t a = -1;
    if (i < n) {
        a = chain_label(ch, i);
        if (a < 0 || a >= nc) {
            flags[0] = 1;
            a = -1;
        }
    }
    // one claim per run of equal labels in the warp (maps of meshes give
    // neighbours the same label): its first lane claims for all
    constexpr unsigned FULL = 0xffffffffu;
    const int32_t prev = __shfl_up_sync(FULL, a, 1);
    const unsigned heads = __ballot_sync(FULL, lane == 0 || prev != a);
    const int first = 31 - __clz(heads & (FULL >> (31 - lane)));
    const unsigned after = lane == 31 ? 0u : heads & (FULL << (lane + 1));
    const int len = (after ? __ffs(after) - 1 : 32) - lane;  // of the run, in its first lane
    int32_t base = 0;
    if (a >= 0 && first == lane) base = atomicAdd(&cnt[a], len);
    const int32_t r = __shfl_sync(FULL, base, first) + (lane - first);
    if (i < n) place[i] = make_int2(a, a >= 0 ? r : 0);
    const int32_t w = __reduce_max_sync(FULL, a >= 0 ? r + 1 : 0);
    if (lane == 0 && w) atomicMax(&bmax, w);
    __syncthreads();
    if (threadIdx.x == 0 && bmax) atomicMax(flags + 1, bmax);
}

__global__ void k_group_place(int64_t n, const int2* __restrict__ place, const int32_t* __restrict__ start,
                              uint32_t* __restrict__ members) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int2 p = place[i];
    members[start[p.x] + p.y] = (uint32_t)i;
}

// Ascending bitonic sort of 32 R numbers in a warp's registers, number
// r 32 + lane in register r: exchanges at a distance of 32 and more are
// between a lane's own registers, the others between lanes.
template <int R>
__device__ __forceinline__ void warp_sort(uint32_t (&x)[R], int lane) {
#pragma unroll
    for (int kk = 2; kk <= 32 * R; kk <<= 1)
#pragma unroll
        for (int j = kk >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int o = r ^ (j / 32);
                    if (o > r) {
                        const bool up = ((r * 32) & kk) == 0;
                        const uint32_t lo = min(x[r], x[o]), hi = max(x[r], x[o]);
                        x[r] = up ? lo : hi;
                        x[o] = up ? hi : lo;
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, x[r], j);
                    const bool keep_min = ((lane & j) == 0) == (((r * 32 + lane) & kk) == 0);
                    x[r] = keep_min ? min(x[r], o) : max(x[r], o);
                }
            }
        }
}

template <int R>
__device__ __forceinline__ void sort_list(uint32_t* __restrict__ m, int len, int lane) {
    uint32_t x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = r * 32 + lane < len ? m[r * 32 + lane] : 0xffffffffu;
    warp_sort<R>(x, lane);
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (r * 32 + lane < len) m[r * 32 + lane] = x[r];
}

// warp per label: up to 128 members sorted in registers (64 members: 43 us
// for 32,768 lists in shared memory), up to GROUP_SORT_MAX in shared memory
// (bitonic, a compare-exchange pair per lane)
__global__ void __launch_bounds__(QT) k_group_sort(int64_t nc, const int32_t* __restrict__ start,
                                                   uint32_t* __restrict__ members) {
    __shared__ uint32_t sh[QT / 32][GROUP_SORT_MAX];
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t A = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (A >= nc) return;
    const int32_t b = start[A], len = start[A + 1] - b;
    if (len <= 1) return;
    if (len <= 32) return sort_list<1>(members + b, len, lane);
    if (len <= 64) return sort_list<2>(members + b, len, lane);
    if (len <= 128) return sort_list<4>(members + b, len, lane);
    uint32_t* S = sh[threadIdx.x >> 5];
    const int P = 1 << (32 - __clz(len - 1));  // at most GROUP_SORT_MAX: the caller checked the largest group
    for (int t = lane; t < P; t += 32) S[t] = t < len ? members[b + t] : FULL;
    __syncwarp();
    for (int kk = 2; kk <= P; kk <<= 1)
        for (int j = kk >> 1; j > 0; j >>= 1) {
            for (int q = lane; q < (P >> 1); q += 32) {
                const int t = ((q & ~(j - 1)) << 1) | (q & (j - 1)), u = t | j;
                const uint32_t x = S[t], y = S[u];
                if ((x > y) == ((t & kk) == 0)) {
                    S[t] = y;
                    S[u] = x;
                }
            }
            __syncwarp();
        }
    for (int t = lane; t < len; t += 32) members[b + t] = S[t];
}

__global__ void k_group_keys(int64_t n, const int2* __restrict__ place, uint32_t* __restrict__ keys,
                             uint32_t* __restrict__ vals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    keys[i] = (uint32_t)place[i].x;
    vals[i] = (uint32_t)i;
}

}  // namespace

gr_status group_begin(gr_ctx* c, int slot, const MapChain& map, int64_t n, int64_t nc, GroupJob* job) {
    cudaStream_t s = c->stream;
    size_t need = 0;
    auto add = [&](size_t bytes) {
        size_t off = need;
        need += (bytes + 255) & ~size_t(255);
        return off;
    };
    const size_t o_cnt = add(4 * (size_t)(nc + 1) + 16), o_start = add(4 * (size_t)(nc + 1)),
                 o_place = add(8 * (size_t)n), o_mem = add(4 * (size_t)n);
    void* base;
    GR_TRY_CUDA(c, c->ws.get(slot, need, &base), "group scratch");
    char* B = (char*)base;
    int32_t* cnt = (int32_t*)(B + o_cnt);
    int32_t* flags = cnt + nc + 1;
    job->n = n;
    job->nc = nc;
    job->start = (int32_t*)(B + o_start);
    job->place = (int2*)(B + o_place);
    job->members = (uint32_t*)(B + o_mem);
    job->host = (int32_t*)host_scratch();
    if (!job->host) return set_error(c, GR_ENOMEM, "group: pinned scratch unavailable");
    if (!c->event) GR_TRY_CUDA(c, cudaEventCreateWithFlags(&c->event, cudaEventDisableTiming), "event");
    GR_TRY_CUDA(c, cudaMemsetAsync(cnt, 0, 4 * (size_t)(nc + 1) + 8, s), "memset");
    if (n > 0) {
        k_group_count<<<(unsigned)ceil_div(n, QT), QT, 0, s>>>(map, n, nc, cnt, job->place, flags);
        count_launch();
    }
    GR_TRY_CUDA(c, cudaMemcpyAsync(job->host, flags, 8, cudaMemcpyDeviceToHost, s), "readback");
    GR_TRY_CUDA(c, cudaEventRecord(c->event, s), "event");
    GR_TRY_CUDA(c, scan_exclusive_i32(cnt, job->start, nc + 1, c->ws, s), "scan");
    return GR_OK;
}

gr_status group_finish(gr_ctx* c, GroupJob* job, bool* bad) {
    cudaStream_t s = c->stream;
    const int64_t n = job->n;
    GR_TRY_CUDA(c, cudaEventSynchronize(c->event), "group sync");
    *bad = job->host[0] != 0;
    if (*bad || n == 0) return GR_OK;
    const unsigned gn = (unsigned)ceil_div(n, QT);
    if (job->host[1] <= GROUP_SORT_MAX) {
        k_group_place<<<gn, QT, 0, s>>>(n, job->place, job->start, job->members);
        count_launch();
        if (job->host[1] > 1) {
            k_group_sort<<<(unsigned)ceil_div(job->nc * 32, QT), QT, 0, s>>>(job->nc, job->start, job->members);
            count_launch();
        }
        GR_TRY_CUDA(c, cudaGetLastError(), "group kernels");
        return GR_OK;
    }
    void *pk, *pv, *pa;
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_A, 4 * (size_t)n, &pk), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_B, 4 * (size_t)n, &pv), "ws");
    GR_TRY_CUDA(c, c->ws.get(WS_SORT_D, 8 * (size_t)n, &pa), "ws");
    uint32_t *k0 = (uint32_t*)pk, *v0 = (uint32_t*)pv, *k1 = (uint32_t*)pa, *v1 = k1 + n;
    k_group_keys<<<gn, QT, 0, s>>>(n, job->place, k0, v0);
    count_launch();
    int alt = 0;
    GR_TRY_CUDA(c, radix_sort_u32(k0, v0, k1, v1, n, bits_for((uint64_t)(job->nc > 1 ? job->nc - 1 : 1)), c->ws, s,
                                  &alt), "sort by label");
    job->members = alt ? v1 : v0;
    return GR_OK;
}

}  // namespace gr
