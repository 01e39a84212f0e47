// Per-camera pieces shared by the optimiser-step kernels (the streaming path's camera step
// and the quadratic form's fused step): compensated sums, the chain rule from an image pair's
// sums to one of its cameras, and the FP64 Adam / exponential-map update of one camera.
#pragma once

#include <math.h>

#include "fm_walk.cuh"

namespace fm {

constexpr int STEP_CAMS = 8;   // cameras (warps) per block of the step kernels
constexpr int STEP_VALS = 8;   // per camera: 6 pose gradient components, loss, scale gradient

// (hi, lo) += (bhi, blo) with the rounding error of the high parts kept (Knuth's TwoSum)
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float bhi, float blo) {
    const float s = hi + bhi;
    const float bb = s - hi;
    const float err = (hi - (s - bb)) + (bhi - bb);
    const float l = lo + blo + err;
    hi = s + l;
    lo = l - (hi - s);
}

// ---- per camera: pose record --------------------------------------------------------------------
// R (9 floats), centre as hi + lo floats (3 + 3), keypoint scale s (focal refinement)
__device__ __forceinline__ void write_camrec(float *rec, const double *R, const double *c, float s) {
#pragma unroll
    for (int i = 0; i < 9; ++i) rec[i] = (float)R[i];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float hi = (float)c[q];
        rec[9 + q] = hi;
        rec[12 + q] = (float)__dsub_rn(c[q], (double)hi);
    }
    rec[15] = s;
}

// keypoint scale of camera k: exp(rho_k), 1 without focal state
__device__ __forceinline__ double camera_scale(const DevProblem &d, int k) {
    return d.rho ? exp(d.rho[k]) : 1.0;
}

__device__ __forceinline__ void vee(const float *M, float *v) {
    v[0] = M[7] - M[5];
    v[1] = M[2] - M[6];
    v[2] = M[3] - M[1];
}

// 1/sqrt(x) in FP64: an FP32 seed refined by two Newton steps (the relative error squares
// each step: ~2e-7 -> ~1e-13 -> below FP64 rounding)
__device__ __forceinline__ double rsqrt64(double x) {
    double y = (double)rsqrtf((float)x);
    const double hx = __dmul_rn(-0.5, x);
    y = __dmul_rn(y, __fma_rn(hx, __dmul_rn(y, y), 1.5));
    y = __dmul_rn(y, __fma_rn(hx, __dmul_rn(y, y), 1.5));
    return y;
}

// Row r of Exp(phi) - I = a K + b K^2 (K = [phi]_x) in FP32. A rotation increment is small, so its
// FP32 relative error (a few ulp) is an absolute error of a few 1e-7 |phi|, the same order as
// that of phi itself, which Adam computes in FP32. For |phi| < 0.1 the Taylor series of a and b
// through the t^6 terms (truncation below 1e-13); otherwise sin and b = 2 sin^2(t/2) / t^2.
__device__ __forceinline__ void so3_exp_minus_identity_row(const float *phi, int r, float *A) {
    const float th2 = rdot3(phi[0], phi[0], phi[1], phi[1], phi[2], phi[2]);
    float a, b;
    if (th2 < 0.01f) {
        a = rfma(-rmul(th2, 1.f / 6.f), rfma(-rmul(th2, 1.f / 20.f), radd(1.f, -rmul(th2, 1.f / 42.f)), 1.f), 1.f);
        b = rmul(0.5f, rfma(-rmul(th2, 1.f / 12.f), rfma(-rmul(th2, 1.f / 30.f), radd(1.f, -rmul(th2, 1.f / 56.f)), 1.f), 1.f));
    } else {
        const float th = __fsqrt_rn(th2);
        const float sh = sinf(rmul(0.5f, th));
        a = __fdiv_rn(sinf(th), th);
        b = __fdiv_rn(rmul(rmul(2.f, sh), sh), th2);
    }
    const float K[9] = {0.f, -phi[2], phi[1], phi[2], 0.f, -phi[0], -phi[1], phi[0], 0.f};
    float k[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) k[c] = r == 0 ? K[c] : (r == 1 ? K[3 + c] : K[6 + c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float k2 = rdot3(k[0], K[c], k[1], K[3 + c], k[2], K[6 + c]);
        A[c] = rfma(b, k2, rmul(a, k[c]));
    }
}

// Gram-Schmidt on the rows: r0 normalised, r1 orthogonalised and normalised, r2 = r0 x r1
__device__ __forceinline__ void orthonormalize_rows(double *R) {
    const double n0 = rsqrt64(rdot3(R[0], R[0], R[1], R[1], R[2], R[2]));
    for (int q = 0; q < 3; ++q) R[q] = __dmul_rn(R[q], n0);
    const double dp = rdot3(R[0], R[3], R[1], R[4], R[2], R[5]);
    for (int q = 0; q < 3; ++q) R[3 + q] = __fma_rn(-dp, R[q], R[3 + q]);
    const double n1 = rsqrt64(rdot3(R[3], R[3], R[4], R[4], R[5], R[5]));
    for (int q = 0; q < 3; ++q) R[3 + q] = __dmul_rn(R[3 + q], n1);
    R[6] = __fma_rn(R[1], R[5], -__dmul_rn(R[2], R[4]));
    R[7] = __fma_rn(R[2], R[3], -__dmul_rn(R[0], R[5]));
    R[8] = __fma_rn(R[0], R[4], -__dmul_rn(R[1], R[3]));
}

// Chain rule of one image pair (or one range partial of it) to one of its cameras.
// gr = the pair's geometry record, sum[0..8] = sum s * o2 o1^T over the point pairs,
// sum[9] = their loss terms. Writes the camera's 6 pose gradient components, (for the first
// camera only) the loss in contrib[6], and in contrib[7] the gradient with respect to the
// camera's keypoint scale s: with F = S_j E S_i, dL/dE = S_j G S_i (G = dL/dF) and
// dL/ds_i = sum_{a, b<2} G_ab E_ab (S_j)_a, dL/ds_j = sum_{a<2, b} G_ab E_ab (S_i)_b.
// FOCAL = false: the scale gradient is not formed (contrib[7] = 0); the pair matrix still
// carries the scales, so dL/dE = S_j G S_i either way.
template <bool FOCAL>
__device__ __forceinline__ void pair_chain_rule(const float *gr, int role, const float *sum,
                                                float gscale, float lscale, float *contrib) {
    float Gp[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) Gp[q] = rmul(sum[q], gscale);
    const float2 cen_i = make_float2(gr[22], gr[23]), cen_j = make_float2(gr[33], gr[34]);
    float M[9], G[9];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        M[3 * a] = rfma(Gp[3 * a + 2], cen_i.x, Gp[3 * a]);
        M[3 * a + 1] = rfma(Gp[3 * a + 2], cen_i.y, Gp[3 * a + 1]);
        M[3 * a + 2] = Gp[3 * a + 2];
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        G[b] = rfma(cen_j.x, M[6 + b], M[b]);
        G[3 + b] = rfma(cen_j.y, M[6 + b], M[3 + b]);
        G[6 + b] = M[6 + b];
    }
    const float *Rn = gr + 9;
    const float tn[3] = {gr[18], gr[19], gr[20]};
    const float inv = gr[21];
    const float *Rj = gr + 24;
    const float th[3] = {rmul(tn[0], inv), rmul(tn[1], inv), rmul(tn[2], inv)};
    // focal: E = [th]_x R_n, the scale gradient from G = dL/dF, then G <- dL/dE
    const float s_i = gr[35], s_j = gr[36];
    {
        const float si[3] = {s_i, s_i, 1.f}, sj[3] = {s_j, s_j, 1.f};
        float gs = 0.f;
        if (FOCAL) {
            float E[9];
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                E[b] = rfma(th[1], Rn[6 + b], rmul(-th[2], Rn[3 + b]));
                E[3 + b] = rfma(-th[0], Rn[6 + b], rmul(th[2], Rn[b]));
                E[6 + b] = rfma(th[0], Rn[3 + b], rmul(-th[1], Rn[b]));
            }
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const float ge = rmul(G[3 * a + b], E[3 * a + b]);
                    if (role == 0 ? b < 2 : a < 2) gs = rfma(ge, role == 0 ? sj[a] : si[b], gs);
                }
        }
        contrib[7] = gs;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) G[3 * a + b] = rmul(rmul(G[3 * a + b], sj[a]), si[b]);
    }
    float A[9];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        A[b] = -rfma(th[1], G[6 + b], rmul(-th[2], G[3 + b]));
        A[3 + b] = -rfma(-th[0], G[6 + b], rmul(th[2], G[b]));
        A[6 + b] = -rfma(th[0], G[3 + b], rmul(-th[1], G[b]));
    }
    float GRt[9];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            GRt[3 * a + b] = rdot3(G[3 * a], Rn[3 * b], G[3 * a + 1], Rn[3 * b + 1], G[3 * a + 2], Rn[3 * b + 2]);
    float gth[3], gt[3], gc[3], gp[3];
    vee(GRt, gth);
    const float dp = rdot3(th[0], gth[0], th[1], gth[1], th[2], gth[2]);
#pragma unroll
    for (int q = 0; q < 3; ++q) gt[q] = rmul(rfma(-dp, th[q], gth[q]), inv);
#pragma unroll
    for (int q = 0; q < 3; ++q) gc[q] = rdot3(Rj[q], gt[0], Rj[3 + q], gt[1], Rj[6 + q], gt[2]);
    if (role == 0) {
        float RtA[9];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) RtA[3 * a + b] = rdot3(Rn[a], A[b], Rn[3 + a], A[3 + b], Rn[6 + a], A[6 + b]);
        vee(RtA, gp);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            contrib[q] = -gp[q];
            contrib[3 + q] = gc[q];
        }
        contrib[6] = rmul(sum[9], lscale);
    } else {
        float ARt[9];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b)
                ARt[3 * a + b] = rdot3(A[3 * a], Rn[3 * b], A[3 * a + 1], Rn[3 * b + 1], A[3 * a + 2], Rn[3 * b + 2]);
        vee(ARt, gp);
        contrib[0] = radd(gp[0], rfma(tn[1], gt[2], rmul(-tn[2], gt[1])));
        contrib[1] = radd(gp[1], rfma(tn[2], gt[0], rmul(-tn[0], gt[2])));
        contrib[2] = radd(gp[2], rfma(tn[0], gt[1], rmul(-tn[1], gt[0])));
#pragma unroll
        for (int q = 0; q < 3; ++q) contrib[3 + q] = -gc[q];
        contrib[6] = 0.f;
    }
}


// Warp-wide TwoSum sums of N (hi, lo) pairs: value i ends in hi[0], lo[0] of lane spread_lane(N, i).
// TwoSum is symmetric in its operands, so this is the butterfly's result bit for bit, with 9 of
// these accumulations for N = 7 where the butterfly takes 35.
template <int N>
__device__ __forceinline__ void warp_two_sum_spread(float *hi, float *lo, int lane) {
    int cnt = N;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (cnt > 1) {
            const int h = (cnt + 1) / 2;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (i >= h) break;
                const float oh = h + i < cnt ? hi[h + i] : 0.f, ol = h + i < cnt ? lo[h + i] : 0.f;
                const float gh = up ? hi[i] : oh, gl = up ? lo[i] : ol;
                hi[i] = up ? oh : hi[i];
                lo[i] = up ? ol : lo[i];
                const float bh = __shfl_xor_sync(0xffffffffu, gh, o);
                const float bl = __shfl_xor_sync(0xffffffffu, gl, o);
                two_sum_acc(hi[i], lo[i], bh, bl);
            }
            cnt = h;
        } else {
            const float bh = __shfl_xor_sync(0xffffffffu, hi[0], o);
            const float bl = __shfl_xor_sync(0xffffffffu, lo[0], o);
            two_sum_acc(hi[0], lo[0], bh, bl);
        }
    }
}

// ---- the update of a block's C cameras ------------------------------------------------------------
// What a block of a step kernel holds of its cameras: the sums of phase 1 (6 pose gradient components,
// the loss, the keypoint-scale gradient, as hi + lo), Adam's m (6) and v (6), R (9) and c (3) in FP64,
// the current record's rotation (9) and keypoint scale, and the hyper-parameters lr_rot, lr_c, beta1,
// beta2, eps, lr_focal.
template <int C>
struct StepState {
    float hi[STEP_VALS][C], lo[STEP_VALS][C], mv[C][12], rec[C][10], hyper[6];
    double Rc[C][12];
    __device__ __forceinline__ void load(const DevProblem &d, const float *cam, int cam0) {
        for (int i = threadIdx.x; i < C * 12; i += blockDim.x) {
            const int cc = i / 12, q = i % 12;
            if (cam0 + cc < d.n_cams) {
                const size_t k = cam0 + cc;
                mv[cc][q] = q < 6 ? d.m[k * 6 + q] : d.v[k * 6 + q - 6];
                Rc[cc][q] = q < 9 ? d.R[k * 9 + q] : d.c[k * 3 + q - 9];
                if (q < 10) rec[cc][q] = cam[k * CAMREC + (q < 9 ? q : 15)];
            }
        }
        if (threadIdx.x < 6) hyper[threadIdx.x] = (float)d.hyper[threadIdx.x];
    }
};

// 1 - beta^t
__device__ __forceinline__ float bias_correction(float beta, long long t) { return radd(1.f, -powf(beta, (float)t)); }

// Adam's step of one component (gradient g; m and v are replaced)
__device__ __forceinline__ float adam_delta(float g, float lr, const float *hyper, float bc1, float bc2, float &m, float &v) {
    const float b1 = hyper[2], b2 = hyper[3], eps = hyper[4];
    m = rfma(b1, m, rmul(radd(1.f, -b1), g));
    v = rfma(b2, v, rmul(rmul(radd(1.f, -b2), g), g));
    return __fdiv_rn(rmul(-lr, __fdiv_rn(m, bc1)), radd(__fsqrt_rn(__fdiv_rn(v, bc2)), eps));
}

// Phase 2 of a step, by the warps that take the roles 0 .. ROT_ROLES(C) of their block (a role a warp,
// behind a block barrier after phase 1). One Adam step (FP32 moments) and the new pose:
// R <- R + (Exp(phi) - I) R and c <- c + delta_c in FP64, where the small increment (Exp(phi) - I) R is
// formed in FP32 from the camera's FP32 record rotation (its error, a few 1e-7 |phi|, is of the order of
// phi's own FP32 error), then Gram-Schmidt on the rows in FP64 on every eighth step (steps 1, 9, 17, ...)
// and the new camera record in `records`. apply = 0: the gradient (FP64 sum of its hi + lo parts) and the
// focal gradient are written, nothing else. With focal refinement rho = log s takes its own Adam step
// (gradient s dL/ds); without, the record keeps its scale. KEEP: the new state is left in `st` as well
// and goes to memory only with `store` (a kernel of several steps).
// The first roles take the rotations of three cameras each, lane 9 c + 3 r + q the entry (r, q); the
// last role the centres, keypoint scales and loss shares of all, lane 3 c + a a component.
// GB300 issues an FP64 instruction (conversions included) of a warp over 64 cycles, whatever its active
// lanes, and every block of a step reaches this phase at the same moment. So the update keeps its FP64
// work to the state itself and spreads it over lanes and over the SM's four sub-partitions, one role
// each: 3 such instructions in series for a rotation (re-orthonormalisation, about 40, only every eighth
// step) and 8 for a centre and its loss, where one warp with a lane per row of R took 26 with the
// conversions of the hyper-parameters (and a lane per camera 48): 1.2 us of an iteration on 119 k point
// pairs, 1.6 us on 3.1 M, 0.9 us of a form iteration. Between two re-orthonormalisations R leaves SO(3) by the
// FP32 rounding of the increments, a few 1e-7 |phi| per step, far below the FP32 camera record's resolution.
constexpr int rot_roles(int cams) { return (cams + 2) / 3; }

template <bool FOCAL, bool KEEP, int C>
__device__ __forceinline__ void step_update(const DevProblem &d, StepState<C> &st, int cam0, int role, int lane, float bc1,
                                            float bc2, long long t_step, int apply, bool store, float *records) {
    if (role < rot_roles(C)) {
        if (!apply) return;
        const int c9 = lane / 9, r = (lane % 9) / 3, q = lane % 3, base = 9 * c9;
        const int cc = 3 * role + c9, kc = cam0 + cc;
        const bool on = lane < 27 && cc < C && kc < d.n_cams;
        const int s = on ? cc : 0;
        // the FP32 gradient: hi is the rounded value of hi + lo (TwoSum keeps |lo| within half an
        // ulp of hi), so hi + lo in FP32 is the same number the FP64 sum would round to
        const float g = radd(st.hi[r][s], st.lo[r][s]);
        if (on && !isfinite(g)) atomicOr(d.err, ERR_NONFINITE);
        float m = st.mv[s][r], v = st.mv[s][6 + r], phi[3], A[3];
        const float dl = adam_delta(g, st.hyper[0], st.hyper, bc1, bc2, m, v);
#pragma unroll
        for (int a = 0; a < 3; ++a) phi[a] = __shfl_sync(0xffffffffu, dl, min(base + 3 * a, 31));
        so3_exp_minus_identity_row(phi, r, A);
        const float *R32 = st.rec[s];
        double Rn = __dadd_rn(st.Rc[s][3 * r + q], (double)rdot3(A[0], R32[q], A[1], R32[3 + q], A[2], R32[6 + q]));
        if ((t_step & 7) == 1) {
            double M[9];
#pragma unroll
            for (int i = 0; i < 6; ++i) M[i] = __shfl_sync(0xffffffffu, Rn, min(base + i, 31));
            orthonormalize_rows(M);
#pragma unroll
            for (int i = 0; i < 9; ++i) Rn = i == 3 * r + q ? M[i] : Rn;
        }
        if (KEEP) __syncwarp();   // every lane has read the rows that are replaced
        if (on) {
            records[(size_t)kc * CAMREC + 3 * r + q] = (float)Rn;
            if (!KEEP || store) d.R[(size_t)kc * 9 + 3 * r + q] = Rn;
            if (KEEP) {
                st.Rc[s][3 * r + q] = Rn;
                st.rec[s][3 * r + q] = (float)Rn;
            }
            if (q == 0) {
                if (!KEEP || store) {
                    d.m[(size_t)kc * 6 + r] = m;
                    d.v[(size_t)kc * 6 + r] = v;
                }
                if (KEEP) {
                    st.mv[s][r] = m;
                    st.mv[s][6 + r] = v;
                }
            }
        }
        return;
    }
    const int cc = lane / 3, a = lane % 3, kc = cam0 + cc;
    const bool on = cc < C && kc < d.n_cams;
    const int s = on ? cc : 0;
    const double bl = (double)st.hi[6][s] + (double)st.lo[6][s];
    const double s_cur = FOCAL && on ? camera_scale(d, kc) : 1.0;
    const double g_rho = FOCAL ? s_cur * ((double)st.hi[7][s] + (double)st.lo[7][s]) : 0.0;
    if (on && a == 0 && (!KEEP || store)) d.cam_loss[kc] = bl;
    if (!apply) {
        bool ok = isfinite(st.hi[6][s]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int q = 3 * h + a;
            const double g = (double)st.hi[q][s] + (double)st.lo[q][s];
            ok = ok && isfinite(g);
            if (on) d.grad[(size_t)kc * 6 + q] = g;
        }
        if (on && !ok) atomicOr(d.err, ERR_NONFINITE);
        if (on && a == 0 && d.grad_rho) d.grad_rho[kc] = g_rho;
        return;
    }
    const float g = radd(st.hi[3 + a][s], st.lo[3 + a][s]);
    if (on && !(isfinite(g) && isfinite(st.hi[6][s]))) atomicOr(d.err, ERR_NONFINITE);
    float s_new = st.rec[s][9];
    if (FOCAL && on && a == 0) {
        const float b1 = st.hyper[2], b2 = st.hyper[3], g1 = (float)g_rho;
        const float mo = rfma(b1, d.rho_m[kc], rmul(radd(1.f, -b1), g1));
        const float vo = rfma(b2, d.rho_v[kc], rmul(rmul(radd(1.f, -b2), g1), g1));
        d.rho_m[kc] = mo;
        d.rho_v[kc] = vo;
        const double r = d.rho[kc] - (double)__fdiv_rn(rmul(st.hyper[5], __fdiv_rn(mo, bc1)),
                                                       radd(__fsqrt_rn(__fdiv_rn(vo, bc2)), st.hyper[4]));
        d.rho[kc] = r;
        d.grad_rho[kc] = g_rho;
        s_new = (float)exp(r);
    }
    float m = st.mv[s][3 + a], v = st.mv[s][9 + a];
    const float dl = adam_delta(g, st.hyper[1], st.hyper, bc1, bc2, m, v);
    const double cn = __dadd_rn(st.Rc[s][9 + a], (double)dl);
    if (on) {
        float *rec_out = records + (size_t)kc * CAMREC;
        const float c_hi = (float)cn;
        rec_out[9 + a] = c_hi;
        rec_out[12 + a] = (float)__dsub_rn(cn, (double)c_hi);
        if (a == 0) rec_out[15] = s_new;
        if (!KEEP || store) {
            d.c[(size_t)kc * 3 + a] = cn;
            d.m[(size_t)kc * 6 + 3 + a] = m;
            d.v[(size_t)kc * 6 + 3 + a] = v;
        }
        if (KEEP) {
            st.Rc[s][9 + a] = cn;
            st.mv[s][3 + a] = m;
            st.mv[s][9 + a] = v;
            if (a == 0) st.rec[s][9] = s_new;
        }
    }
}

}  // namespace fm
