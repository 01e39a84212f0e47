// Per-iteration kernels of the epipolar adjustment (Sec. "Epipolar Adjustment").
//
//   stream_loss per range  : E'_n of the range's pairs from the camera records, epsilon = o2^T E'_n o1 for
//                            every point pair, the loss term and the adjoint G'_n += s * o2 o1^T, segmented
//                            per image pair (stream_reweight: with the round's IRLS weights)
//   camera_step per camera : chain rule of its pairs' partial sums, compensated sum, Adam, R_k <- Exp(phi_k) R_k,
//                            the new camera record
//   finalize    per chain  : loss total, step count, camera records back in their first buffer
// Once per round or call: cam_prep (camera records from the poses), pair_setup (geometry records of the
// pairs), irls_weights / residuals (the streaming walk writing one value per point pair). combine and gather: the
// chain rule per pair and its sums per camera, for the evaluation without allocation.
#include <math.h>

#include <algorithm>

#include "fm_step.cuh"

namespace fm {

template <int S>
constexpr int PASS_BYTES = S * STAGE_BYTES + CameraE::BYTES;   // shared memory of a warp

// A warp per block, a range each, staged in shared memory S chunks deep (walk_range_staged). The last block
// has no range: when the pass follows an optimiser camera step (prev_loss > 0), it finishes the
// step's loss total (over prev_loss per-camera shares) and step count.
// Bound by HBM on large scenes, by the latency of a range's loads and by the launches around the pass
// on small ones. Loading 4 groups per warp into registers after the wait for the launch before
// (8 warps a block) left the memory system idle while a pass filled up and drained. An iteration of
// fm_step (this pass, then the camera step; chains of 100), before -> now: 119 k point pairs FP32 18.7 ->
// 7.7 us, 3.1 M FP32 28.0 -> 11.4, 12 M FP16 39.6 -> 27.5, 49 M FP32 161 -> 142, 49 M FP16 92.3 -> 77.2, 141 M FP16
// 227.9 -> 214.5.
template <int STORE, int MODE, int S>
__global__ void __launch_bounds__(32, 32) k_stream_loss(DevProblem d, int prev_loss) {
    extern __shared__ __align__(16) unsigned char stage[];
    const int r = blockIdx.x;
    if (r >= d.n_ranges) {
        pdl_wait();
        pdl_trigger();
        if (prev_loss > 0 && blockIdx.x == gridDim.x - 1)
            finish_step<32>(d, prev_loss, 1, reinterpret_cast<double *>(stage));
        return;
    }
    LossBody<MODE> body(d);
    walk_range_staged<STORE, MODE == MODE_LOSS_IRLS, S, STAGE_GROUPS, CameraE>(d, r, threadIdx.x, body, stage, [] {
        pdl_wait();     // camera records of this pass
        pdl_trigger();  // the per-camera step may be scheduled once the last wave has started
    });
}

// The first pass of an IRLS round fused with the round's reweighting: the residual at the
// round's starting poses gives the weight (filtered by tau, floored by delta, quantised as the
// storage keeps it), which is written and at once used for the loss and adjoint sums. Same
// arithmetic as the weights kernel followed by the streaming pass, one read of the keypoints
// instead of two. tau comes from d.hyper[6] so one captured graph serves every round.
template <int STORE>
struct ReweightLossBody {
    LossBody<MODE_LOSS_IRLS> loss;
    const DevProblem &d;
    float tau, delta, scale;
    float out[2];
    unsigned kept;
    __device__ ReweightLossBody(const DevProblem &dd, float t)
        : loss(dd), d(dd), tau(t), delta((float)dd.delta), scale(dd.w_scale), kept(0) {
        out[0] = out[1] = 0.f;
    }
    __device__ __forceinline__ void point(int k, float e, float x1, float y1, float x2, float y2, float) {
        const float a = fabsf(e);
        const bool keep = a <= tau;  // NaN residuals are filtered
        const float wf = keep ? irls_weight(a, delta) : 0.f;
        const float w = STORE == FM_STORE_FP32 ? wf : __half2float(__float2half_rn(wf * scale));
        out[k] = w;
        kept += keep ? 1u : 0u;
        loss.point(k, e, x1, y1, x2, y2, w);
    }
    __device__ __forceinline__ void segment_begin(int seg) { loss.segment_begin(seg); }
    __device__ __forceinline__ void segment_end(int seg, int r, int lane, bool last) {
        loss.segment_end(seg, r, lane, last);
    }
    __device__ __forceinline__ void group_done(int gb, int p_end, int lane) {
        const int q = gb + lane * Fmt<STORE>::PPL;
        if (STORE == FM_STORE_FP32) {
            static_cast<float *>(d.w)[q] = q < p_end ? out[0] : 0.f;
        } else {
            // already on the FP16 grid: the conversion is exact
            const float a = q < p_end ? out[0] : 0.f;
            const float b = q + 1 < p_end ? out[1] : 0.f;
            reinterpret_cast<__half2 *>(d.w)[q >> 1] = __floats2half2_rn(a, b);
        }
        out[0] = out[1] = 0.f;
    }
};

template <int STORE, int S>
__global__ void __launch_bounds__(32, 32) k_stream_reweight(DevProblem d) {
    extern __shared__ __align__(16) unsigned char stage[];
    const int r = blockIdx.x;
    ReweightLossBody<STORE> body(d, 0.f);
    walk_range_staged<STORE, false, S, STAGE_GROUPS, CameraE>(d, r, threadIdx.x, body, stage, [&] {
        pdl_wait();     // camera records of this pass, the threshold
        pdl_trigger();
        body.tau = (float)d.hyper[6];
    });
    unsigned k = body.kept;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    if ((threadIdx.x & 31) == 0 && k) atomicAdd(d.counter, (unsigned long long)k);
}

// ---- per-point-pair maps (IRLS weights, residual export) ------------------------------------------
template <int STORE>
struct WeightBody {
    const DevProblem &d;
    float tau, delta, scale;
    float out[2];
    unsigned kept;
    __device__ WeightBody(const DevProblem &dd, float t) : d(dd), tau(t), delta((float)dd.delta),
                                                            scale(dd.w_scale), kept(0) {
        out[0] = out[1] = 0.f;
    }
    __device__ __forceinline__ void point(int k, float e, float, float, float, float, float) {
        const float a = fabsf(e);
        // filtered (w = 0) when |eps| > tau; NaN residuals are filtered too
        const bool keep = a <= tau;
        out[k] = keep ? irls_weight(a, delta) : 0.f;
        kept += keep ? 1u : 0u;
    }
    __device__ __forceinline__ void segment_begin(int) {}
    __device__ __forceinline__ void segment_end(int, int, int, bool) {}
    __device__ __forceinline__ void group_done(int gb, int p_end, int lane) {
        const int q = gb + lane * Fmt<STORE>::PPL;
        if (STORE == FM_STORE_FP32) {
            static_cast<float *>(d.w)[q] = q < p_end ? out[0] : 0.f;
        } else {
            const float a = q < p_end ? out[0] * scale : 0.f;
            const float b = q + 1 < p_end ? out[1] * scale : 0.f;
            reinterpret_cast<__half2 *>(d.w)[q >> 1] = __floats2half2_rn(a, b);
        }
        out[0] = out[1] = 0.f;
    }
};

template <int STORE, int S>
__global__ void __launch_bounds__(32) k_irls_weights(DevProblem d, float tau) {
    extern __shared__ __align__(16) unsigned char stage[];
    const int lane = threadIdx.x, r = blockIdx.x;
    WeightBody<STORE> body(d, tau);
    walk_range_staged<STORE, false, S>(d, r, lane, body, stage, [] {});
    unsigned k = body.kept;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    if (lane == 0 && k) atomicAdd(d.counter, (unsigned long long)k);
}

template <int STORE>
struct ResidualBody {
    const int *perm;
    float *out_input;   // input order
    float out[2];
    __device__ ResidualBody(const DevProblem &d, float *o) : perm(d.perm), out_input(o) { out[0] = out[1] = 0.f; }
    __device__ __forceinline__ void point(int k, float e, float, float, float, float, float) {
        out[k] = e;
    }
    __device__ __forceinline__ void segment_begin(int) {}
    __device__ __forceinline__ void segment_end(int, int, int, bool) {}
    __device__ __forceinline__ void group_done(int gb, int p_end, int lane) {
        const int q = gb + lane * Fmt<STORE>::PPL;
#pragma unroll
        for (int k = 0; k < Fmt<STORE>::PPL; ++k)
            if (q + k < p_end) out_input[perm ? perm[q + k] : q + k] = out[k];
    }
};

template <int STORE, int S>
__global__ void __launch_bounds__(32) k_residuals(DevProblem d, float *out) {
    extern __shared__ __align__(16) unsigned char stage[];
    const int r = blockIdx.x;
    ResidualBody<STORE> body(d, out);
    walk_range_staged<STORE, false, S>(d, r, threadIdx.x, body, stage, [] {});
}

__global__ void k_cam_prep(DevProblem d) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n_cams) return;
    write_camrec(d.cam + (size_t)k * CAMREC, d.R + 9 * (size_t)k, d.c + 3 * (size_t)k, (float)camera_scale(d, k));
}

struct Hyper {
    double v[6];
};
__global__ void k_set_hyper(DevProblem d, Hyper h) { d.hyper[threadIdx.x] = h.v[threadIdx.x]; }

// threshold and kept count of a round whose first pass is fused with the reweighting
__global__ void k_begin_round(DevProblem d, double tau) {
    d.hyper[6] = tau;
    *d.counter = 0;
}

// new parameters from the caller's device memory, and their camera records
__global__ void k_set_params(DevProblem d, const double *R, const double *c) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n_cams) return;
    double Rk[9], ck[3];
#pragma unroll
    for (int q = 0; q < 9; ++q) d.R[9 * (size_t)k + q] = Rk[q] = R[9 * (size_t)k + q];
#pragma unroll
    for (int q = 0; q < 3; ++q) d.c[3 * (size_t)k + q] = ck[q] = c[3 * (size_t)k + q];
    write_camrec(d.cam + (size_t)k * CAMREC, Rk, ck, (float)camera_scale(d, k));
}

// g_R = 0.5 s [g_phi]_x R and g_c = s g_c of every camera, a thread per row
__global__ void k_pose_gradient(int n_cams, const double *grad, const double *R, const double *scale, double *gR, double *gc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, k = i / 3, a = i % 3;
    if (k >= n_cams) return;
    const double s = *scale, *g = grad + 6 * (size_t)k, *Rk = R + 9 * (size_t)k;
    const int b = (a + 1) % 3, c = (a + 2) % 3;   // row a of [g]_x: -g_c at column b, g_b at column c
    const double hb = -0.5 * (g[c] * s), hc = 0.5 * (g[b] * s);
#pragma unroll
    for (int q = 0; q < 3; ++q) gR[9 * (size_t)k + 3 * a + q] = hb * Rk[3 * b + q] + hc * Rk[3 * c + q];
    gc[3 * (size_t)k + a] = g[3 + a] * s;
}

__global__ void __launch_bounds__(256) k_pair_setup(DevProblem d) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n < d.n_pairs) pair_geometry(d, n, d.cam_i[n], d.cam_j[n]);
}

// ---- per pair: combine partials and chain rule ----------------------------------------------------
__global__ void k_combine(DevProblem d, float gscale, float lscale) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= d.n_pairs) return;
    const int p0 = d.pair_off[n], p1 = d.pair_off[n + 1];
    const int r0 = p0 / WR, r1 = (p1 - 1) / WR;
    float sum[10], cmp[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) sum[k] = cmp[k] = 0.f;
    for (int r = r0; r <= r1; ++r) {
        const float4 *s = reinterpret_cast<const float4 *>(d.slots + (size_t)(n + r) * SLOT);
        const float4 a = s[0], b = s[1], c = s[2];
        const float v[10] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y};
#pragma unroll
        for (int k = 0; k < 10; ++k) {  // Kahan-compensated FP32 sum
            const float y = v[k] - cmp[k];
            const float t = sum[k] + y;
            cmp[k] = (t - sum[k]) - y;
            sum[k] = t;
        }
    }
    float Gp[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) Gp[k] = sum[k] * gscale;
    const float loss = sum[9] * lscale;
    const int i = d.cam_i[n], j = d.cam_j[n];
    // G = T_j G' T_i^T (gradient with respect to E from the one with respect to E')
    const float2 cen_i = d.cen[i], cen_j = d.cen[j];
    float M[9], G[9];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        M[3 * a] = Gp[3 * a] + Gp[3 * a + 2] * cen_i.x;
        M[3 * a + 1] = Gp[3 * a + 1] + Gp[3 * a + 2] * cen_i.y;
        M[3 * a + 2] = Gp[3 * a + 2];
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        G[b] = M[b] + cen_j.x * M[6 + b];
        G[3 + b] = M[3 + b] + cen_j.y * M[6 + b];
        G[6 + b] = M[6 + b];
    }
    const float *g = d.geo + (size_t)n * GEO;
    float Rn[9], tn[3];
#pragma unroll
    for (int k = 0; k < 9; ++k) Rn[k] = g[9 + k];
    tn[0] = g[18];
    tn[1] = g[19];
    tn[2] = g[20];
    const float inv = g[21];
    const float th[3] = {tn[0] * inv, tn[1] * inv, tn[2] * inv};
    // A = -[th]_x G
    float A[9];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        A[b] = -(-th[2] * G[3 + b] + th[1] * G[6 + b]);
        A[3 + b] = -(th[2] * G[b] - th[0] * G[6 + b]);
        A[6 + b] = -(-th[1] * G[b] + th[0] * G[3 + b]);
    }
    // g_th = vee(G R_n^T); g_t = (I - th th^T) g_th / |t|
    float GRt[9], ARt[9], RtA[9];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            GRt[3 * a + b] = G[3 * a] * Rn[3 * b] + G[3 * a + 1] * Rn[3 * b + 1] + G[3 * a + 2] * Rn[3 * b + 2];
            ARt[3 * a + b] = A[3 * a] * Rn[3 * b] + A[3 * a + 1] * Rn[3 * b + 1] + A[3 * a + 2] * Rn[3 * b + 2];
            RtA[3 * a + b] = Rn[a] * A[b] + Rn[3 + a] * A[3 + b] + Rn[6 + a] * A[6 + b];
        }
    float gth[3], gt[3], gpj[3], gpi[3];
    vee(GRt, gth);
    const float dp = th[0] * gth[0] + th[1] * gth[1] + th[2] * gth[2];
#pragma unroll
    for (int q = 0; q < 3; ++q) gt[q] = (gth[q] - dp * th[q]) * inv;
    vee(ARt, gpj);
    gpj[0] += tn[1] * gt[2] - tn[2] * gt[1];
    gpj[1] += tn[2] * gt[0] - tn[0] * gt[2];
    gpj[2] += tn[0] * gt[1] - tn[1] * gt[0];
    vee(RtA, gpi);
    const float *Rj = d.cam + (size_t)j * CAMREC;
    float gc[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) gc[q] = Rj[q] * gt[0] + Rj[3 + q] * gt[1] + Rj[6 + q] * gt[2];
    float4 *out = reinterpret_cast<float4 *>(d.pair_grad + (size_t)n * PG);
    out[0] = make_float4(-gpi[0], -gpi[1], -gpi[2], gc[0]);
    out[1] = make_float4(gc[1], gc[2], gpj[0], gpj[1]);
    out[2] = make_float4(gpj[2], -gc[0], -gc[1], -gc[2]);
    out[3] = make_float4(loss, 0.f, 0.f, 0.f);
    bool ok = isfinite(loss);
#pragma unroll
    for (int q = 0; q < 3; ++q) ok = ok && isfinite(gpi[q]) && isfinite(gpj[q]) && isfinite(gc[q]);
    if (!ok) atomicOr(d.err, ERR_NONFINITE);
}

// ---- per camera: gradient gather (FP64) and the loss sum ------------------------------------------
constexpr int GATHER_THREADS = 256;

__global__ void __launch_bounds__(GATHER_THREADS) k_gather(DevProblem d, int count_step) {
    if (blockIdx.x == gridDim.x - 1) {
        // loss = sum over pairs, FP64, fixed partition and fixed tree order
        __shared__ double red[GATHER_THREADS];
        double s = 0.0;
        for (int n = threadIdx.x; n < d.n_pairs; n += GATHER_THREADS)
            s += (double)d.pair_grad[(size_t)n * PG + 12];
        red[threadIdx.x] = s;
        __syncthreads();
        for (int w = GATHER_THREADS / 2; w > 0; w >>= 1) {
            if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            *d.loss_out = red[0];
            if (count_step) *d.step += 1;
        }
        return;
    }
    const int k = blockIdx.x * GATHER_THREADS + threadIdx.x;
    if (k >= d.n_cams) return;
    double g[6] = {0, 0, 0, 0, 0, 0};
    for (int e = d.cam_off[k]; e < d.cam_off[k + 1]; ++e) {
        const int ent = d.cam_ent[e];
        const float *pg = d.pair_grad + (size_t)(ent >> 1) * PG + (ent & 1) * 6;
#pragma unroll
        for (int q = 0; q < 6; ++q) g[q] += (double)pg[q];
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) d.grad[(size_t)k * 6 + q] = g[q];
}

// ---- per camera: Adam + exponential map (FP64) -----------------------------------------------------
// Fused per-camera step, C cameras a block and W warps a camera (all blocks resident at once for up to
// 4,864 cameras). Before waiting for the streaming pass (griddepcontrol.wait) the block fetches everything
// that is at least two kernels old: its cameras' Adam moments, poses and the step count, and for
// each camera the (pair, role) entries, their range-partial counts and the pairs' geometry (formed again
// from the camera records). After the wait only the partial sums remain to be read.
// Phase 1: the chain rule is linear in a pair's sums, so it is applied to every (pair, warp-range partial)
// item separately; the items are spread evenly over the lanes of the camera's warps, 32 a pass, W passes
// at once (a pair that spans many ranges does not hold up one lane). Each sum is carried as an unevaluated
// hi + lo pair (TwoSum); a lane's items are added in the order of their passes and the lanes by a
// butterfly, whatever W is, so every W gives the same bits; with W > 1 the warps share the values out.
// What bounds it is latency: a pass of loads and chain rule takes about 2,000 cycles, and a warp a camera
// makes three of them in series on 1,000 cameras and 49 M point pairs (8 cameras of one warp a block there
// cost an iteration 2.5 us more, and 0.9 us more on 16 cameras and 119 k).
// Phase 2: the update of the block's cameras, spread over warps (step_update). The two powers of its
// bias corrections are formed before the wait.
// The new records go to cam_dst, a second buffer (with apply): other blocks may still read this step's
// records. The loss of a pair is counted by its first camera only; each camera's FP64 loss share goes to
// cam_loss[camera], and the next kernel (the next pass or the finalize kernel) adds them up in a fixed
// order and advances the step count.
template <bool FOCAL, int C, int W>
__global__ void __launch_bounds__(32 * C * W, 1024 / (32 * C * W))
k_camera_step(DevProblem d, float gscale, float lscale, int apply, float *cam_dst) {
    constexpr int NV = FOCAL ? STEP_VALS : STEP_VALS - 1;      // sums carried per camera
    constexpr int NQ = W == 1 ? NV : (STEP_VALS + W - 1) / W;  // of which a warp adds up
    __shared__ StepState<C> st;
    __shared__ int4 s_item[C][32];
    constexpr int ROW = GEO - 8 + 4;   // a record from its float 8 on; 16-byte reads free of bank conflicts
    __shared__ __align__(16) float s_geo[8 + C * 32 * ROW];
    __shared__ float s_con[W > 1 ? C : 1][W][STEP_VALS][32];   // contributions of W passes over the items
    __shared__ float s_bc[2][2];
    __shared__ long long s_step;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cc = warp / W, sub = warp % W;
    const int cam0 = blockIdx.x * C, k = cam0 + cc;
    // the warps of a camera, barrier 1 + cc (literal ids: with an id in a register a block reserves all 16
    // barriers, and an SM then holds only three blocks beside a pass)
    static_assert(W == 1 || C <= 4, "a barrier per camera");
    auto camera_sync = [&] {
        if (W == 1) __syncwarp();
        else if (C < 2 || cc == 0) asm volatile("bar.sync 1, %0;" ::"n"(32 * W) : "memory");
        else if (C < 3 || cc == 1) asm volatile("bar.sync 2, %0;" ::"n"(32 * W) : "memory");
        else if (cc == 2) asm volatile("bar.sync 3, %0;" ::"n"(32 * W) : "memory");
        else asm volatile("bar.sync 4, %0;" ::"n"(32 * W) : "memory");
    };
    st.load(d, d.cam, cam0);
    // bias corrections before the wait: the pass that runs now may or may not have added the step before
    // this one to the count, so they are formed for both counts
    if (warp == C * W - 1 && lane < 4) {
        const long long t = *reinterpret_cast<volatile long long *>(d.step);
        s_bc[lane >> 1][lane & 1] = bias_correction((float)d.hyper[2 + (lane & 1)], t + 1 + (lane >> 1));
        if (lane == 0) s_step = t;
    }
    const int e_begin = k < d.n_cams ? d.cam_off[k] : 0;
    const int e_end = k < d.n_cams ? d.cam_off[k + 1] : 0;
    // this camera's entries, 32 at a time: pair, role, first range and number of ranges; the
    // pair's geometry at the records of the pass goes to shared memory
    auto load_chunk = [&](int base) -> int {
        const int e = base + lane;
        int n = 0, role = 0, r0 = 0, cnt = 0;
        if (e < e_end) {
            const int ent = d.cam_ent[e];
            n = ent >> 1;
            role = ent & 1;
            r0 = d.pair_off[n] / WR;
            cnt = (d.pair_off[n + 1] - 1) / WR - r0 + 1;
            if (sub == 0) {
                float g[GEO];
                pair_geometry_regs(d.cam, d.cen, d.cam_i[n], d.cam_j[n], g);   // (the pass has reported degenerate pairs)
                float4 *dst = reinterpret_cast<float4 *>(s_geo + (cc * 32 + lane) * ROW);
#pragma unroll
                for (int q = 2; q < GEO / 4; ++q) dst[q] = make_float4(g[4 * q], g[4 * q + 1], g[4 * q + 2], g[4 * q + 3]);
            }
        }
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (sub == 0) s_item[cc][lane] = make_int4(incl - cnt, n, role, r0);
        camera_sync();
        return __shfl_sync(0xffffffffu, incl, 31);
    };
    auto find = [&](int t) {   // the entry of item t
        int lo = 0, hi = 31;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_item[cc][mid].x <= t) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    int total = load_chunk(e_begin);
    const int first = find(32 * sub + lane);
    pdl_wait();     // partial sums of the streaming pass
    pdl_trigger();
    const long long t_step = *d.step + 1;
    if (k < d.n_cams) {
        float hi[NQ], lo[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) hi[q] = lo[q] = 0.f;
        for (int base = e_begin; base < e_end; base += 32) {
            if (base != e_begin) {
                camera_sync();
                total = load_chunk(base);
            }
            for (int t0 = 0; t0 < total; t0 += 32 * W) {
                const int t = t0 + 32 * sub + lane;
                float contrib[STEP_VALS];
                if (t < total) {
                    const int li = t0 == 0 && base == e_begin ? first : find(t);
                    const int4 it = s_item[cc][li];
                    const float4 *sl = reinterpret_cast<const float4 *>(d.slots + (size_t)(it.y + it.w + (t - it.x)) * SLOT);
                    const float4 sa = sl[0], sb = sl[1], sc = sl[2];
                    const float sum[10] = {sa.x, sa.y, sa.z, sa.w, sb.x, sb.y, sb.z, sb.w, sc.x, sc.y};
                    pair_chain_rule<FOCAL>(s_geo + (cc * 32 + li) * ROW, it.z, sum, gscale, lscale, contrib);
                }
                if (W == 1) {
                    if (t < total) {
#pragma unroll
                        for (int q = 0; q < NV; ++q) two_sum_acc(hi[q], lo[q], contrib[q], 0.f);
                    }
                    continue;
                }
                if (t < total) {
#pragma unroll
                    for (int q = 0; q < NV; ++q) s_con[cc][sub][q][lane] = contrib[q];
                }
                camera_sync();
#pragma unroll
                for (int w = 0; w < W; ++w)   // a lane's items in their order
                    if (t0 + 32 * w + lane < total) {
#pragma unroll
                        for (int j = 0; j < NQ; ++j)
                            if (sub + W * j < NV) two_sum_acc(hi[j], lo[j], s_con[cc][w][sub + W * j][lane], 0.f);
                    }
                if (t0 + 32 * W < total) camera_sync();
            }
        }
        warp_two_sum_spread<NQ>(hi, lo, lane);
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const int q = W == 1 ? j : sub + W * j;
            if (lane == spread_lane(NQ, j) && q < NV) {
                st.hi[q][cc] = hi[0];
                st.lo[q][cc] = lo[0];
            }
        }
    }
    __syncthreads();
    // blocks of one SM start their roles in different sub-partitions
    constexpr int ROLES = rot_roles(C) + 1, APART = ROLES == 2 ? 2 : 1;
    static_assert(ROLES * APART <= C * W, "a warp for each role");
    const int role = ((warp - (int)(blockIdx.x / 152)) & (C * W - 1)) / APART;
    if (role < ROLES && ((warp - (int)(blockIdx.x / 152)) & (APART - 1)) == 0) {
        const long long ahead = t_step - 1 - s_step;
        float bc1 = s_bc[ahead & 1][0], bc2 = s_bc[ahead & 1][1];
        if (ahead < 0 || ahead > 1) {   // the count moved by more than that step
            bc1 = bias_correction(st.hyper[2], t_step);
            bc2 = bias_correction(st.hyper[3], t_step);
        }
        step_update<FOCAL, false>(d, st, cam0, role, lane, bc1, bc2, t_step, apply, true, cam_dst);
    }
}

// Adam step with a given gradient (d.grad, FP64): the same update as the camera-step kernel (with the
// gradient split into FP32 hi + lo parts, whose FP32 sum is the gradient rounded to FP32, as there); the
// step count is advanced by k_bump_step.
__global__ void __launch_bounds__(128) k_apply_gradient(DevProblem d) {
    __shared__ StepState<STEP_CAMS> st;
    const int cam0 = blockIdx.x * STEP_CAMS;
    const long long t_step = *d.step + 1;
    st.load(d, d.cam, cam0);
    if (threadIdx.x < STEP_CAMS * STEP_VALS) {
        const int q = threadIdx.x % STEP_VALS, cc = threadIdx.x / STEP_VALS;
        const double g = q < 6 && cam0 + cc < d.n_cams ? d.grad[(size_t)(cam0 + cc) * 6 + q] : 0.0;
        st.hi[q][cc] = (float)g;
        st.lo[q][cc] = (float)__dsub_rn(g, (double)st.hi[q][cc]);
    }
    __syncthreads();
    step_update<false, false>(d, st, cam0, threadIdx.x >> 5, threadIdx.x & 31, bias_correction(st.hyper[2], t_step),
                              bias_correction(st.hyper[3], t_step), t_step, 1, true, d.cam);
}

__global__ void k_bump_step(DevProblem d) { *d.step += 1; }

// closes a chain of steps: loss of the last step and `count` steps added to the step count (loss_copy: the
// caller's loss, or null), by block 0; the others copy the camera records back from the alternate buffer
// (copy_src, or null: a float4 per thread) and (check) report image pairs that the last step left degenerate
__global__ void __launch_bounds__(FIN_THREADS) k_finalize(DevProblem d, int n_loss, int count, double *loss_copy,
                                                          const float *copy_src, int check) {
    const int i = ((int)blockIdx.x - 1) * FIN_THREADS + threadIdx.x;
    const bool pair = check && i >= 0 && i < d.n_pairs;
    const int ci = pair ? d.cam_i[i] : 0, cj = pair ? d.cam_j[i] : 0;
    pdl_wait();
    pdl_trigger();
    __shared__ double red[FIN_THREADS];
    if (blockIdx.x == 0) {
        finish_step(d, n_loss, count, red);
        if (loss_copy && threadIdx.x == 0) *loss_copy = red[0];
        return;
    }
    if (copy_src && i < d.n_cams * (CAMREC / 4))
        reinterpret_cast<float4 *>(d.cam)[i] = reinterpret_cast<const float4 *>(copy_src)[i];
    if (pair) {
        float g[GEO];
        if (!pair_geometry_regs(copy_src ? copy_src : d.cam, d.cen, ci, cj, g)) atomicOr(d.err, ERR_DEGENERATE);
    }
}

// ---- launchers -------------------------------------------------------------------------------------
static inline int blocks_for(int64_t n, int t) { return (int)((n + t - 1) / t); }

int camera_step_blocks(const DevProblem &d) { return blocks_for(d.n_cams, STEP_CAMS); }

void launch_cam_prep(const DevProblem &d, cudaStream_t s) {
    k_cam_prep<<<blocks_for(d.n_cams, 128), 128, 0, s>>>(d);
}

void launch_pair_setup(const DevProblem &d, cudaStream_t s) {
    k_pair_setup<<<blocks_for(d.n_pairs, 256), 256, 0, s>>>(d);
}

void launch_set_hyper(const DevProblem &d, const double *h, cudaStream_t s) {
    Hyper v;
    for (int q = 0; q < 6; ++q) v.v[q] = h[q];
    k_set_hyper<<<1, 6, 0, s>>>(d, v);
}

void launch_begin_round(const DevProblem &d, double tau, cudaStream_t s) { k_begin_round<<<1, 1, 0, s>>>(d, tau); }

void launch_set_params(const DevProblem &d, const double *R, const double *c, cudaStream_t s) {
    k_set_params<<<blocks_for(d.n_cams, 64), 64, 0, s>>>(d, R, c);
}

void launch_finalize(const DevProblem &d, int count, const float *copy_src, bool check, cudaStream_t s, bool pdl,
                     double *loss_copy) {
    const int work = std::max(copy_src ? d.n_cams * (CAMREC / 4) : 0, check ? d.n_pairs : 0);
    launch_k(k_finalize, dim3(1 + blocks_for(work, FIN_THREADS)), dim3(FIN_THREADS), s, pdl, d, d.n_cams, count, loss_copy,
             copy_src, check ? 1 : 0);
}

void launch_stream_loss(const DevProblem &d, cudaStream_t s, bool pdl, bool after_step) {
    const int prev = after_step ? d.n_cams : 0;
    with_stages(d, [&](auto store, auto depth) {
        constexpr int STORE = decltype(store)::value, S = decltype(depth)::value;
        static_assert(S * STAGE_BYTES >= FIN_THREADS * sizeof(double), "the last block finishes a step in its stage");
        const dim3 grid(d.n_ranges + 1), block(32);
        if (d.loss == FM_LOSS_IRLS)
            launch_smem(k_stream_loss<STORE, MODE_LOSS_IRLS, S>, grid, block, PASS_BYTES<S>, s, pdl, d, prev);
        else
            launch_smem(k_stream_loss<STORE, MODE_LOSS_L1, S>, grid, block, PASS_BYTES<S>, s, pdl, d, prev);
    });
}

void launch_stream_reweight(const DevProblem &d, cudaStream_t s, bool pdl) {
    with_stages(d, [&](auto store, auto depth) {
        constexpr int STORE = decltype(store)::value, S = decltype(depth)::value;
        launch_smem(k_stream_reweight<STORE, S>, dim3(d.n_ranges), dim3(32), PASS_BYTES<S>, s,
                    pdl, d);
    });
}

void launch_combine(const DevProblem &d, cudaStream_t s) {
    const double Z = d.z > 0.0 ? d.z : (double)d.n_pp;
    float gscale, lscale;
    if (d.loss == FM_LOSS_IRLS) {  // stored weights are w * s
        gscale = (float)(2.0 / (Z * d.w_scale));
        lscale = (float)(1.0 / (Z * d.w_scale));
    } else {
        gscale = (float)(1.0 / Z);
        lscale = (float)(1.0 / Z);
    }
    k_combine<<<blocks_for(d.n_pairs, 128), 128, 0, s>>>(d, gscale, lscale);
}

void launch_gather(const DevProblem &d, bool count_step, cudaStream_t s) {
    k_gather<<<blocks_for(d.n_cams, GATHER_THREADS) + 1, GATHER_THREADS, 0, s>>>(d, count_step ? 1 : 0);
}

void loss_scales(const DevProblem &d, float &gscale, float &lscale) {
    const double Z = d.z > 0.0 ? d.z : (double)d.n_pp;
    if (d.loss == FM_LOSS_IRLS) {  // stored weights are w * s
        gscale = (float)(2.0 / (Z * d.w_scale));
        lscale = (float)(1.0 / (Z * d.w_scale));
    } else {
        gscale = (float)(1.0 / Z);
        lscale = (float)(1.0 / Z);
    }
}

void launch_apply_gradient(const DevProblem &d, cudaStream_t s) {
    k_apply_gradient<<<blocks_for(d.n_cams, STEP_CAMS), 128, 0, s>>>(d);
    k_bump_step<<<1, 1, 0, s>>>(d);
}

void launch_camera_step(const DevProblem &d, bool apply, float *cam_dst, cudaStream_t s, bool pdl) {
    float gscale, lscale;
    loss_scales(d, gscale, lscale);
    auto go = [&](auto cams, auto warps) {
        constexpr int C = decltype(cams)::value, W = decltype(warps)::value;
        const dim3 grid(blocks_for(d.n_cams, C)), block(32 * C * W);
        if (d.refine_focal) launch_k(k_camera_step<true, C, W>, grid, block, s, pdl, d, gscale, lscale, apply ? 1 : 0, cam_dst);
        else launch_k(k_camera_step<false, C, W>, grid, block, s, pdl, d, gscale, lscale, apply ? 1 : 0, cam_dst);
    };
    using std::integral_constant;
    // Items (range partials of a camera's pairs) a camera: at most 2 (ranges + pairs) / cameras. us an
    // iteration with C x W = 8 x 1, 2 x 2, 1 x 4:
    //   many items (46 to 320): 16 cameras, 5 M point pairs 24.2, 19.1, 17.1; 100 cameras, 3.1 M 13.1, 11.6, 11.3;
    //     1,000 cameras, 49 M FP32 144.9, 141.9, 140.6
    //   fewer (13 to 40): 128 cameras, 1 M 11.4, 10.3, 10.9; 152 cameras, 3.1 M FP16 12.8, 11.7, 12.2; 1,000 cameras,
    //     3 M 20.6, 20.9, 30.8; 2,000 cameras, 80 M FP32 231.1, 228.9, 232.8
    //   more cameras than 2 x 2 has resident: 3,000 cameras, 60 M 103.6, 107.3, 111.8; 4,000, 140 M 215.8, 221.1, 227.2
    const int64_t items = 2 * ((int64_t)d.n_ranges + d.n_pairs);
    if (d.n_cams <= 8 * 152 && items > 44 * (int64_t)d.n_cams)
        go(integral_constant<int, 1>(), integral_constant<int, 4>());
    else if (d.n_cams <= 16 * 152)
        go(integral_constant<int, 2>(), integral_constant<int, 2>());
    else
        go(integral_constant<int, 8>(), integral_constant<int, 1>());
}

void launch_irls_weights(const DevProblem &d, float tau, cudaStream_t s) {
    with_stages<RECORD_STAGES>(d, [&](auto store, auto depth) {
        constexpr int STORE = decltype(store)::value, S = decltype(depth)::value;
        k_irls_weights<STORE, S><<<d.n_ranges, 32, S * STAGE_BYTES, s>>>(d, tau);
    });
}

void launch_residuals(const DevProblem &d, float *out_input_order, cudaStream_t s) {
    with_stages<RECORD_STAGES>(d, [&](auto store, auto depth) {
        constexpr int STORE = decltype(store)::value, S = decltype(depth)::value;
        k_residuals<STORE, S><<<d.n_ranges, 32, S * STAGE_BYTES, s>>>(d, out_input_order);
    });
}

cudaError_t launch_pose_gradient(int n_cams, const double *grad, const double *R, const double *scale, double *gR,
                                 double *gc, cudaStream_t s) {
    k_pose_gradient<<<blocks_for(3 * (int64_t)n_cams, 96), 96, 0, s>>>(n_cams, grad, R, scale, gR, gc);
    return cudaGetLastError();
}

}  // namespace fm
