// What starts a step -- the predictor of Alg. 1, the drive anchors, the counters, the augmented
// Lagrangian warm start -- shared by their kernels (k_step.cu, k_sweep.cu), the fused per-body
// prelude of ground-only scenes (k_collision.cu) and the one-launch front of small scenes
// (k_front.cu).
#pragma once
#include "pabd_internal.h"

namespace pabd {

__device__ __forceinline__ void quat_to_mat(float4 q, float* R) {
    float x = q.x, y = q.y, z = q.z, w = q.w;
    R[0] = 1.f - 2.f * (y * y + z * z); R[1] = 2.f * (x * y - z * w);       R[2] = 2.f * (x * z + y * w);
    R[3] = 2.f * (x * y + z * w);       R[4] = 1.f - 2.f * (x * x + z * z); R[5] = 2.f * (y * z - x * w);
    R[6] = 2.f * (x * z - y * w);       R[7] = 2.f * (y * z + x * w);       R[8] = 1.f - 2.f * (x * x + y * y);
}

__device__ __forceinline__ void store_q(float4* q, int b, const float* c, const float* A) {
    q[3 * b] = make_float4(c[0], c[1], c[2], A[0]);
    q[3 * b + 1] = make_float4(A[1], A[2], A[3], A[4]);
    q[3 * b + 2] = make_float4(A[5], A[6], A[7], A[8]);
}

// Predictor (Alg. 1): v* = v + h g; c* = c + h v*; Q* = normalise(Q + h/2 [w, 0] Q);
// A* = R(Q*); s = q^0 = (c*, A*).  Pinned bodies, and those of a group held this step, keep q^n.
__device__ __forceinline__ void predict_body(const Dev& d, int b) {
    if ((d.bflags[b] & BF_PINNED) || held(d, b)) {
        float4 a0 = d.qn[3 * b], a1 = d.qn[3 * b + 1], a2 = d.qn[3 * b + 2];
        d.sq[3 * b] = a0; d.sq[3 * b + 1] = a1; d.sq[3 * b + 2] = a2;
        d.qa[3 * b] = a0; d.qa[3 * b + 1] = a1; d.qa[3 * b + 2] = a2;
        d.qb[3 * b] = a0; d.qb[3 * b + 1] = a1; d.qb[3 * b + 2] = a2;
        d.qstar[b] = d.quat[b];
        return;
    }
    const float h = d.p.h;
    float4 v = d.vel[b], w = d.omg[b], Q = d.quat[b], c4 = d.qn[3 * b];
    float vs[3] = {v.x + h * d.p.g[0], v.y + h * d.p.g[1], v.z + h * d.p.g[2]};
    float cs[3] = {c4.x + h * vs[0], c4.y + h * vs[1], c4.z + h * vs[2]};
    float4 wq = make_float4(w.x * Q.w + (w.y * Q.z - w.z * Q.y), w.y * Q.w + (w.z * Q.x - w.x * Q.z),
                            w.z * Q.w + (w.x * Q.y - w.y * Q.x), -(w.x * Q.x + w.y * Q.y + w.z * Q.z));
    const float hh = 0.5f * h;
    float4 Qn = make_float4(Q.x + hh * wq.x, Q.y + hh * wq.y, Q.z + hh * wq.z, Q.w + hh * wq.w);
    float inv = rsqrtf(Qn.x * Qn.x + Qn.y * Qn.y + Qn.z * Qn.z + Qn.w * Qn.w);
    Qn.x *= inv; Qn.y *= inv; Qn.z *= inv; Qn.w *= inv;
    float A[9];
    quat_to_mat(Qn, A);
    store_q(d.sq, b, cs, A);
    store_q(d.qa, b, cs, A);
    d.qstar[b] = Qn;
}

// Drive anchors at t = (step + 1) h: x_i = x_i0 + arm (cos th r + sin th (u x r)),
// th = amp sin(2 pi t / period + phase).
__device__ __forceinline__ void drive_update(const Dev& d, int k) {
    const double t = (double)(*d.step_index + 1) * d.p.h_d;
    float4 a = d.drv[3 * k], r = d.drv[3 * k + 1], ur = d.drv[3 * k + 2];
    float2 pp = d.drv_t[k];
    const float th = r.w * sinf((float)(6.283185307179586 * t / (double)pp.x) + pp.y);
    float cs, sn;
    sincosf(th, &sn, &cs);
    const int bi = d.drv_bond[k];
    float4 cur = d.bxi[bi];
    d.bxi[bi] = make_float4(a.x + a.w * (cs * r.x + sn * ur.x), a.y + a.w * (cs * r.y + sn * ur.y),
                            a.z + a.w * (cs * r.z + sn * ur.z), cur.w);
}

// the step's counters (C_NBONDS and the contact counts are set again later in the step)
__device__ __forceinline__ void reset_counters(const Dev& d) {
    d.ctr[C_NPAIRS] = 0;
    d.ctr[C_CELLBITS] = 0;
    d.ctr[C_NLARGE] = 0;
    d.ctr[C_NHEAVY] = 0;
    d.ctr[C_FP64DYN] = 0;
    for (int k = C_NPHEAVY; k < C_COUNT; ++k) d.ctr[k] = 0;
}

// augmented Lagrangian warm start of bond b at the start of a step (Eq. 29), from the values the
// previous step ended with (parity n_iter): kappa <- max(gamma kappa, kappa_start),
// lambda <- alpha gamma lambda, into the parity-0 buffer read by the first sweep
__device__ __forceinline__ void al_warm(const Dev& d, int b) {
    if (d.bmeta[b].z != K_AL) return;
    const float2 kl = (d.p.n_iter & 1) ? d.al_st1[b] : d.al_st0[b];
    const float4 pr = d.al_par[b];  // (kappa_start, beta, alpha, gamma)
    d.al_st0[b] = make_float2(fmaxf(pr.w * kl.x, pr.x), pr.z * pr.w * kl.y);
}

}  // namespace pabd
