// pd_adjoint.cuh -- shared by the adjoint's translation units: the arguments
// of a step's adjoint, the FP32 derivatives of the bond law and the
// compensated node sums (pd_adjoint.cu: FP64 states and mixed states off the
// stencil path; pd_adjoint_stencil.cu: mixed states on it).
#pragma once

#include "pd_device.cuh"

namespace pdi {

struct AdjArgs {
    int B;
    long long N, nb;
    int nx, ny;
    double dx, c, V, dt, rho, a, b;
    double dt_rb, a_b;  // dt / (rho b) and a / b (no FP64 division per DOF)
    int law;
    double s_ratio, k, alpha, gfA;
    const int32_t *row_ptr, *col;
    const uint8_t *codes;
    const float *s0, *kappa;
    int n_obs;
    const int32_t *obs;  // [n_obs] local step of each observation
    const double *w;     // [B][n_obs]
    const int32_t *coord;  // packed grid coordinates per node
    // FP32 constants of the mixed path, rounded on the host (the FP64 pipe is
    // narrow on this part): c V, dx, and |xi| = sqrt(q) dx and its reciprocal
    // for q = |k|^2 < 64
    float cVf, dxf, s_ratio_f, gfA_f, k_f, alpha_f;
    float L0q[64], iL0q[64];
};

// dD/ds and the total dD/ds0 of law_derivs (pd_adjoint.cu) in FP32.
__device__ __forceinline__ void law_derivs_f(const AdjArgs &a, float s, float s0, float &dDds, float &dDds0) {
    const float sc = a.gfA_f > 0.f ? s0 + a.gfA_f / s0 : a.s_ratio_f * s0;
    const float dsc = a.gfA_f > 0.f ? 1.0f - a.gfA_f / (s0 * s0) : a.s_ratio_f;
    dDds = 0.0f;
    dDds0 = 0.0f;
    if (s <= s0 || s >= sc) return;
    const float w = sc - s0;
    if (a.law == PD_LAW_BILINEAR) {
        dDds = s0 * sc / (s * s * w);
        dDds0 = -(sc / s - 1.0f) * sc / (w * w) + dsc * (-s0 * (1.0f - s0 / s) / (w * w));
        return;
    }
    const float k = a.k_f, al = a.alpha_f;
    const float t = (s - s0) / w;
    const float e = expf(-k * t), ek = 1.0f - expf(-k);
    const float beta = 1.0f - (1.0f - e) / ek + al * (1.0f - t);
    const float dbeta = -k * e / ek - al;
    const float dtds = 1.0f / w, dtds0 = (s - sc) / (w * w), dtdsc = -(s - s0) / (w * w);
    dDds = (s0 * beta / (s * s) - (s0 / s) * dbeta * dtds) / (1.0f + al);
    dDds0 = (-(beta / s + (s0 / s) * dbeta * dtds0) - dsc * (s0 / s) * dbeta * dtdsc) / (1.0f + al);
}

// s + x accumulated with the rounding error carried in c (Knuth's TwoSum).
__device__ __forceinline__ void fold(float &s, float &c, float x) {
    const float t = s + x;
    const float z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
}

// R_obs[b][o] = reaction[b][m] for the observations inside a segment of len
// steps from start.
int adjoint_gather_obs(int B, int len, int start, int n_obs, const int32_t *obs, const double *reaction, double *R_obs,
                       cudaStream_t s);

// The adjoint run of a mixed state on the stencil path with ascending CSR
// rows: forward run with checkpoints every k steps, recomputation and reverse
// sweep (pd_adjoint's contract; a.obs is on the device). steps: [B] the samples'
// current steps, on the host.
int adjoint_stencil(pd_state *st, const AdjArgs &a, int n_steps, int k, const int32_t *steps, double *grad_s0, double *grad_kappa,
                    double *R_obs, pd_stream stream);

}  // namespace pdi
