// Pieces of the spectral-mismatch loss shared with the edge scaling, which
// runs its fine-graph part once and its reduced-graph part every iteration.
#pragma once

#include "gr_internal.cuh"

namespace gr {

// Control of the edge-scaling loop, kept on the device so that iterations are
// queued without a host wait between them (all zero before the first).
struct ScaleState {
    double L0, L_prev, lam1, eta;
    double inv_bound;  // 1 / (lam1 times the iteration's share of the bound)
    int it;    // iterations whose update ran or is running
    int stop;  // the convergence test has ended the loop
};

// What the loop control of one iteration needs (state NULL: a plain loss).
struct ScaleStep {
    ScaleState* state = nullptr;
    double eta_max = 0.0, eps = 0.0, bound_step = 0.0, alpha = 0.0;
    const unsigned long long* lam_prev = nullptr;  // bits of the last update's smallest ratio (NULL: first iteration)
    unsigned long long* lam_next = nullptr;        // where this one's will be taken: emptied by the loop control
    float* loss_hist = nullptr;                    // entry of this iteration
    const double* dG = nullptr;
    const double* dP = nullptr;
    float* dw = nullptr;
    float* w = nullptr;
};

// Device buffers of the reduced-graph part
struct LossWork {
    bool short_parts;   // of the reduced graph: see parts_short
    const float* w;     // m: the weights that loss_weights took
    int2* cw;           // 2m: (column, weight) in slot order
    float* D;           // nc: weighted degrees
    double* part;       // per-block partial sums
    unsigned* counter;  // tickets (zero between kernels)
    float* coef;        // 4K: adjoint coefficients
    double* mu;         // K: mass-weighted means of the smoothed block
    float *Y, *Z, *T;   // iterates y_0 .. y_S, z_0 .. z_{S-1}, T_1 .. T_S (T = adjoint / D)
    float *yb0, *yb1;   // adjoint iterate, in turn
};

// Fine part: R_f, the aggregate means y0 and the aggregate sizes, from the
// map `agg`.  cc's workspace holds the scratch.  *bad: a label out of range.
gr_status loss_fine(gr_ctx* f, gr_ctx* cc, const int32_t* agg, const float* X, int K, float* y0, float* Rf,
                    float* mass, bool* bad);
// scratch on cc for `sweeps` sweeps; adjoint: with room for the iterates and
// the adjoint, else two iterates
gr_status loss_work(gr_ctx* cc, int K, int sweeps, bool adjoint, LossWork* W);
// slot-order weights and degrees of w (and, for the edge scaling, FP64 row
// sums dP and the smallest dG / dP as bits)
gr_status loss_weights(gr_ctx* cc, const float* w, LossWork& W, double* dP, const double* dG,
                       unsigned long long* lam);
// sweeps from W.Y, the quotients and the loss; adjoint: keeps what loss_adjoint reads
gr_status loss_coarse(gr_ctx* cc, int K, int sweeps, double omega, const float* y0, const float* Rf, const float* mass,
                      const LossWork& W, bool adjoint, const float* grad_loss, float* loss_out, const ScaleStep& st);
// the reverse sweeps and the edge gradients (grad), or the scaling update (st.state)
gr_status loss_adjoint(gr_ctx* cc, int K, int sweeps, double omega, const float* mass, const LossWork& W, float* grad,
                       const ScaleStep& st);

}  // namespace gr
