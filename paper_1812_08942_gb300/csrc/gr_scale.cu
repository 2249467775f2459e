// Edge-weight scaling of a reduced graph by constrained SGD with momentum
// (Alg. 1), driven by the exact gradient of the spectral-mismatch loss.
//
// L_P is the reduced graph with the weights being scaled, L_G the same graph
// with its initial weights, so the lambda_1 estimate min_p d_G(p) / d_P(p)
// (Eq. courant-fischer-3) starts at 1.  The loss stands in for lambda_n:
// its gradient is the weight sensitivity, its ratio to the first loss scales
// the step size, its relative decrease is the convergence test.
// Every edge of an iteration updates from the degrees at the iteration's start
// (the paper gives no edge order, and this order parallelises); updates never
// go below zero, as the scheme only scales weights up.
#include <math.h>
#include <string.h>

#include "gr_loss.cuh"

namespace gr {

// iterations whose loss and lambda_1 the device keeps before the host reads
// them: scratch of a fixed size, since kmax may be any number ("until it
// converges")
constexpr int64_t SCALE_HIST = 1024;

gr_status scale_edges_impl(gr_ctx* fine, gr_ctx* coarse, const int32_t* agg, const float* X, int K, int sweeps,
                           double omega, double alpha, double eta_max, double delta_bar, double eps, int kmax,
                           float* w, int32_t* iters_out, double* loss_hist, double* lam1_hist) {
    cudaStream_t s = fine->stream;
    const int64_t nc = coarse->n, mc = coarse->m;
    const int64_t hist = kmax < SCALE_HIST ? kmax : SCALE_HIST;
    size_t need = 0;
    auto add = [&](size_t bytes) {
        size_t off = need;
        need += (bytes + 255) & ~size_t(255);
        return off;
    };
    const size_t o_dG = add(8 * (size_t)nc), o_dP = add(8 * (size_t)nc), o_dw = add(4 * (size_t)mc),
                 o_y0 = add(4 * (size_t)nc * K), o_Rf = add(4 * (size_t)K), o_mass = add(4 * (size_t)nc),
                 o_state = add(sizeof(ScaleState)), o_loss = add(4 * (size_t)hist), o_lam = add(8 * (size_t)hist);
    void* base;
    GR_TRY_CUDA(fine, fine->ws.get(WS_SCALE, need, &base), "scaling scratch");
    char* B = (char*)base;
    double* dG = (double*)(B + o_dG);
    double* dP = (double*)(B + o_dP);
    float* dw = (float*)(B + o_dw);
    float* y0 = (float*)(B + o_y0);
    float* Rf = (float*)(B + o_Rf);
    float* mass = (float*)(B + o_mass);
    ScaleState* state = (ScaleState*)(B + o_state);
    float* lossd = (float*)(B + o_loss);
    // per update (k - 1 modulo hist): bits of the smallest d_G / d_P after it
    unsigned long long* lam = (unsigned long long*)(B + o_lam);
    int64_t* hs = host_scratch();
    if (!hs) return set_error(fine, GR_ENOMEM, "scale_edges: pinned scratch unavailable");

    bool bad = false;
    gr_status st = loss_fine(fine, coarse, agg, X, K, y0, Rf, mass, &bad);
    if (st != GR_OK) return st;
    if (bad) return set_error(fine, GR_EINVAL, "scale_edges: agg labels must lie in [0, coarse n)");
    LossWork W;
    st = loss_work(coarse, K, sweeps, true, &W);
    if (st != GR_OK) return st;
    GR_TRY_CUDA(fine, cudaMemcpyAsync(W.Y, y0, 4 * (size_t)nc * K, cudaMemcpyDeviceToDevice, s), "copy");
    GR_TRY_CUDA(fine, cudaMemsetAsync(dw, 0, 4 * (size_t)mc, s), "memset");
    GR_TRY_CUDA(fine, cudaMemsetAsync(state, 0, sizeof(ScaleState), s), "memset");
    GR_TRY_CUDA(fine, cudaMemsetAsync(lam, 0xff, 8 * (size_t)hist, s), "memset");

    ScaleStep step;
    step.state = state;
    step.eta_max = eta_max;
    step.eps = eps;
    step.bound_step = pow(delta_bar, 1.0 / kmax);  // per-iteration share of the bound
    step.alpha = alpha;
    step.dG = dG;
    step.dP = dP;
    step.dw = dw;
    step.w = w;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    auto done = [&](gr_status r) {
        if (r != GR_OK) cudaStreamSynchronize(s);  // a failed call leaves no kernel that reads X
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        return r;
    };
    for (cudaEvent_t& e : ev)
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess)
            return done(set_error(fine, GR_ECUDA, "scale_edges: event"));
    auto cuda = [&](cudaError_t e) { return e == cudaSuccess ? GR_OK : cuda_error(fine, e, "scale_edges"); };
    // the histories of the updates done, from update `read` on, which begins the device's arrays
    ScaleState now;
    int64_t read = 0;
    double lam1 = 1.0;
    auto read_hist = [&](int64_t len) {
        float hl[SCALE_HIST];
        unsigned long long hm[SCALE_HIST];
        gr_status r = cuda(cudaMemcpyAsync(&now, state, sizeof(now), cudaMemcpyDeviceToHost, s));
        if (r == GR_OK) r = cuda(cudaMemcpyAsync(hl, lossd, 4 * (size_t)len, cudaMemcpyDeviceToHost, s));
        if (r == GR_OK) r = cuda(cudaMemcpyAsync(hm, lam, 8 * (size_t)len, cudaMemcpyDeviceToHost, s));
        const gr_status sync = cuda(cudaStreamSynchronize(s));
        if (r == GR_OK) r = sync;
        if (r != GR_OK) return r;
        for (int64_t i = read; i < now.it && i < read + len; ++i) {
            const unsigned long long b = hm[i - read];
            if (b != ~0ull) memcpy(&lam1, &b, 8);
            if (loss_hist) loss_hist[i] = (double)hl[i - read];
            if (lam1_hist) lam1_hist[i] = lam1;
        }
        read += len;
        return GR_OK;
    };
    bool stopped = false;
    for (int64_t k = 1; k <= kmax; ++k) {
        const int slot = (int)(k & 1);
        if (k > 2) {  // has iteration k - 2 ended the loop?
            if ((st = cuda(cudaEventSynchronize(ev[slot]))) != GR_OK) return done(st);
            if (((const int32_t*)hs)[slot]) {
                stopped = true;
                break;
            }
        }
        unsigned long long* prev = k > 1 ? lam + (k - 2) % hist : nullptr;
        if (k == 1) {
            st = loss_weights(coarse, w, W, dG, nullptr, nullptr);
            if (st == GR_OK) st = cuda(cudaMemcpyAsync(dP, dG, 8 * (size_t)nc, cudaMemcpyDeviceToDevice, s));
        } else {
            st = loss_weights(coarse, w, W, dP, dG, prev);
        }
        if (st == GR_OK && k > 1 && (k - 1) % hist == 0) st = read_hist(hist);
        if (st != GR_OK) return done(st);
        step.lam_prev = prev;
        step.lam_next = lam + (k - 1) % hist;
        step.loss_hist = lossd + (k - 1) % hist;
        st = loss_coarse(coarse, K, sweeps, omega, W.Y, Rf, mass, W, true, nullptr, nullptr, step);
        if (st == GR_OK) st = loss_adjoint(coarse, K, sweeps, omega, mass, W, nullptr, step);
        if (st == GR_OK) st = cuda(cudaMemcpyAsync((int32_t*)hs + slot, &state->stop, 4, cudaMemcpyDeviceToHost, s));
        if (st == GR_OK) st = cuda(cudaEventRecord(ev[slot], s));
        if (st != GR_OK) return done(st);
    }
    // lambda_1 after the last update
    if (!stopped) st = loss_weights(coarse, w, W, dP, dG, lam + (kmax - 1) % hist);
    if (st == GR_OK) st = read_hist(hist < kmax - read ? hist : kmax - read);
    if (st != GR_OK) return done(st);
    if (iters_out) *iters_out = now.it;
    return done(cuda(cudaGetLastError()));
}

}  // namespace gr
