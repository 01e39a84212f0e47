// Pre-aggregated quadratic form of the IRLS objective (Eq. epipolar-objective-l2 and the IRLS
// equation after it): with the weights fixed for a round, the objective of image pair n is a
// quadratic function of e_n = vec(E'_n), so one streaming pass per round collects, per pair,
//   c0 = sum w eps0^2,   g0 = sum w eps0 a,   W = sum w a a^T      (a = vec(o2 o1^T))
// at the anchor e0 (the essential matrices of the poses the pass ran at, eps0 = a^T e0), and
// every iteration of the round evaluates the pair in O(1) from e = e0 + d:
//   sum w eps^2      = c0 + d^T (2 g0 + W d)
//   sum w eps a      = g0 + W d       (the same sums the streaming pass produces)
// Anchoring matters for accuracy: e^T W e on its own cancels by a factor (|a| |e| / eps)^2
// (about 1e5 near the optimum), whereas the anchored form keeps the FP32 error structure of
// the streaming pass (the large W enters only through the step d).
//
// W has Kronecker structure: a a^T = (o2 o2^T) (x) (o1 o1^T), so its 81 entries take only
// 6 x 6 = 36 distinct values M[u][v] = sum w m2_u m1_v over the monomials
//   m2 = (x2^2, x2 y2, x2, y2^2, y2, 1),  m1 = (x1^2, x1 y1, x1, y1^2, y1, 1),
// with W[3p+q][3r+s] = M[sym(p,r)][sym(q,s)], sym the index of the unordered pair in
// (00, 01, 02, 11, 12, 22). Per point pair that is 36 multiply-adds instead of 45, issued as 18
// packed pairs.
#include "fm_grid.cuh"
#include "fm_step.cuh"

namespace fm {

// REWEIGHT: the IRLS weights are computed from the residual at the same poses (and written,
// quantised as the storage keeps them) before they enter the sums
template <int STORE, bool REWEIGHT>
struct QuadBody {
    const DevProblem &d;
    float tau, delta, scale;
    float acc[QSUMS];
    float out[2];
    unsigned kept;
    __device__ QuadBody(const DevProblem &dd, float t)
        : d(dd), tau(t), delta((float)dd.delta), scale(dd.w_scale), kept(0) {
#pragma unroll
        for (int i = 0; i < QSUMS; ++i) acc[i] = 0.f;
        out[0] = out[1] = 0.f;
    }
    __device__ __forceinline__ void segment_begin(int) {}
    __device__ __forceinline__ void point(int k, float e, float x1, float y1, float x2, float y2, float w) {
        if (REWEIGHT) {
            const float ae = fabsf(e);
            const bool keep = ae <= tau;  // NaN residuals are filtered
            const float wf = keep ? irls_weight(ae, delta) : 0.f;
            w = STORE == FM_STORE_FP32 ? wf : __half2float(__float2half_rn(wf * scale));
            out[k] = w;
            kept += keep ? 1u : 0u;
        }
        // c0 and g0 = sum (w eps o2) (x) o1
        const float we = w * e;
        acc[0] = fmaf(we, e, acc[0]);
        float tx, ty;                       // w eps o2 = (tx, ty, we)
        mul2(tx, ty, we, we, x2, y2);
        fma2(acc[1], acc[2], tx, tx, x1, y1);
        fma2(acc[4], acc[5], ty, ty, x1, y1);
        fma2(acc[7], acc[8], we, we, x1, y1);
        add2(acc[3], acc[6], tx, ty);
        acc[9] += we;
        // M[u][v] += (w m2_u) m1_v, two neighbouring entries of a row per packed instruction (the
        // pass is bound by instruction issue, not by the FP32 pipe)
        float wx2, wy2, u[6], v[6];
        mul2(wx2, wy2, w, w, x2, y2);
        mul2(u[0], u[1], wx2, wx2, x2, y2);
        u[2] = wx2;
        u[3] = wy2 * y2;
        u[4] = wy2;
        u[5] = w;
        mul2(v[0], v[1], x1, x1, x1, y1);
        v[2] = x1;
        v[3] = y1 * y1;
        v[4] = y1;
        v[5] = 1.f;
#pragma unroll
        for (int a = 0; a < 6; ++a)
#pragma unroll
            for (int b = 0; b < 6; b += 2) fma2(acc[10 + 6 * a + b], acc[10 + 6 * a + b + 1], u[a], u[a], v[b], v[b + 1]);
    }
    __device__ __forceinline__ void segment_end(int seg, int r, int lane, bool) {
#pragma unroll
        for (int i = 0; i < QSUMS; ++i) {
            float v = acc[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            acc[i] = v;
        }
        if (lane == 0) {
            float4 *s = reinterpret_cast<float4 *>(d.qslots + (size_t)(seg + r) * QSLOT);
#pragma unroll
            for (int q = 0; q < QSLOT / 4; ++q) {
                float v[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) v[c] = 4 * q + c < QSUMS ? acc[4 * q + c] : 0.f;
                s[q] = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
#pragma unroll
        for (int i = 0; i < QSUMS; ++i) acc[i] = 0.f;
    }
    __device__ __forceinline__ void group_done(int gb, int p_end, int lane) {
        if (!REWEIGHT) return;
        const int q = gb + lane * Fmt<STORE>::PPL;
        if (STORE == FM_STORE_FP32) {
            static_cast<float *>(d.w)[q] = q < p_end ? out[0] : 0.f;
        } else {
            // the values are already multiples of the FP16 grid: the conversion is exact
            const float a = q < p_end ? out[0] : 0.f;
            const float b = q + 1 < p_end ? out[1] : 0.f;
            reinterpret_cast<__half2 *>(d.w)[q >> 1] = __floats2half2_rn(a, b);
        }
        out[0] = out[1] = 0.f;
    }
};

// One warp per block and range, staged 3 chunks deep, two groups of a chunk in straight code: 94
// registers, 20 warps per SM. Bound by instruction issue and the FP32 pipe (66 operations a point pair).
// The 46 sums leave no registers for loads in flight, and four groups in straight code overran the
// instruction cache; with 4 groups loaded ahead and 16 warps per SM in blocks of 8 the pass took, on
// 48.9 M point pairs with / without reweighting, FP16 224 / 189 us and FP32 309 / 246 us; now 183 / 152
// and 184 / 159 (3.1 M: FP16 30 / 27 -> 25 / 21, FP32 35 / 29 -> 26 / 23).
constexpr int QUAD_STAGES = 3, QUAD_UNROLL = 2, QUAD_WARPS_PER_SM = 20;

template <int STORE, bool REWEIGHT>
__global__ void __launch_bounds__(32, QUAD_WARPS_PER_SM) k_quad_accumulate(DevProblem d, float tau) {
    __shared__ __align__(16) unsigned char stage[QUAD_STAGES * STAGE_BYTES];
    QuadBody<STORE, REWEIGHT> body(d, tau);
    walk_range_staged<STORE, !REWEIGHT, QUAD_STAGES, QUAD_UNROLL>(d, blockIdx.x, threadIdx.x, body, stage, [] {});
    if (REWEIGHT) {
        unsigned k = body.kept;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
        if (threadIdx.x == 0 && k) atomicAdd(d.counter, (unsigned long long)k);
    }
}

// per pair (one warp, a lane per sum): Kahan-sum the range partials into the pair's record
//   [0..35] M, [36] c0, [37..45] g0, [46..54] e0 = E'_n of the geometry record, [55] 0
// (M first, so that the fused step reads it as 16-byte aligned vectors)
__global__ void k_quad_combine(DevProblem d) {
    const int n = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (n >= d.n_pairs) return;
    const int r0 = d.pair_off[n] / WR, r1 = (d.pair_off[n + 1] - 1) / WR;
    float *rec = d.quad + (size_t)n * QREC;
    for (int q = lane; q < QSUMS; q += 32) {
        float sum = 0.f, c = 0.f;
        for (int r = r0; r <= r1; ++r) {
            const float y = d.qslots[(size_t)(n + r) * QSLOT + q] - c;
            const float t = sum + y;
            c = (t - sum) - y;
            sum = t;
        }
        rec[q < 10 ? 36 + q : q - 10] = sum;
    }
    if (lane < 9) rec[46 + lane] = d.geo[(size_t)n * GEO + lane];
    if (lane == 9) rec[55] = 0.f;
}

// The form's sums at a pair's current matrix (g[0..8] = E'_n): sum[0..8] = q = g0 + W d, sum[9] =
// c0 + d^T (g0 + q), d = E'_n - e0; rec = the pair's record
__device__ __forceinline__ void form_sums(const float4 *rec, const float *g, float *sum) {
    constexpr int SYM[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
    float t[20];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        const float4 x = rec[9 + v];
        t[4 * v] = x.x; t[4 * v + 1] = x.y; t[4 * v + 2] = x.z; t[4 * v + 3] = x.w;
    }
    // t[0] = c0, t[1..9] = g0, t[10..18] = e0
    float dv[9], q[9];
    float loss = t[0];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        dv[a] = g[a] - t[10 + a];
        q[a] = t[1 + a];
        loss = fmaf(dv[a], t[1 + a], loss);
    }
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const float4 x = rec[c];
        const float mc[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int u = (4 * c + h) / 6, v = (4 * c + h) % 6;
#pragma unroll
            for (int pp = 0; pp < 3; ++pp)
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    if (SYM[pp][r] != u) continue;
#pragma unroll
                    for (int qq = 0; qq < 3; ++qq)
#pragma unroll
                        for (int ss = 0; ss < 3; ++ss)
                            if (SYM[qq][ss] == v) q[3 * pp + qq] = fmaf(mc[h], dv[3 * r + ss], q[3 * pp + qq]);
                }
        }
    }
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        loss = fmaf(dv[a], q[a], loss);
        sum[a] = q[a];
    }
    sum[9] = loss;
}

// One optimiser iteration on the form, fused into one launch. Warp w owns camera
// k = 8 * block + w; its lanes take the camera's image pairs, each computing the pair's
// geometry from the two camera records (cam_src), the form's sums at the current E'_n,
//   q = g0 + W d,  loss = c0 + d^T (g0 + q),  d = E'_n - e0,
// and the chain rule to camera k. Both cameras of a pair evaluate it (O(1) each), which
// removes a per-pair launch and the wait on it. The warp reduces with compensated butterflies,
// then the block updates its cameras (step_update) and writes the new records to cam_dst: the
// records of this step's poses stay intact in cam_src for the other blocks. The Adam step count is *d.step + 1 + it; the launch that closes the chain adds
// the chain's length to *d.step.
template <bool FOCAL>
__global__ void __launch_bounds__(STEP_CAMS * 32, 4)
k_quad_step(DevProblem d, int it, const float *cam_src, float *cam_dst, float gscale, float lscale, int apply) {
    constexpr int NV = FOCAL ? STEP_VALS : STEP_VALS - 1;   // sums carried per camera
    __shared__ StepState<STEP_CAMS> st;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * STEP_CAMS + warp;
    const int e_begin = k < d.n_cams ? d.cam_off[k] : 0;
    const int e_end = k < d.n_cams ? d.cam_off[k + 1] : 0;
    // the camera's first 32 (pair, role) entries and the pairs' cameras are static: fetch them
    // while the previous step finishes
    int e = e_begin + lane;
    int n = 0, role = 0, ci = 0, cj = 0;
    if (e < e_end) {
        const int ent = d.cam_ent[e];
        n = ent >> 1;
        role = ent & 1;
        ci = d.cam_i[n];
        cj = d.cam_j[n];
    }
    pdl_wait();     // camera records, poses and moments of the previous step
    pdl_trigger();
    st.load(d, cam_src, blockIdx.x * STEP_CAMS);
    const long long t_step = *d.step + 1 + it;
    if (k < d.n_cams) {
        float hi[STEP_VALS], lo[STEP_VALS];
#pragma unroll
        for (int q = 0; q < STEP_VALS; ++q) hi[q] = lo[q] = 0.f;
        for (; e < e_end; e += 32) {
            if (e >= e_begin + 32) {
                const int ent = d.cam_ent[e];
                n = ent >> 1;
                role = ent & 1;
                ci = d.cam_i[n];
                cj = d.cam_j[n];
            }
            float g[GEO];
            if (!pair_geometry_regs(cam_src, d.cen, ci, cj, g)) atomicOr(d.err, ERR_DEGENERATE);
            float sum[10];
            form_sums(reinterpret_cast<const float4 *>(d.quad + (size_t)n * QREC), g, sum);
            float contrib[STEP_VALS];
            pair_chain_rule<FOCAL>(g, role, sum, gscale, lscale, contrib);
#pragma unroll
            for (int w = 0; w < NV; ++w) two_sum_acc(hi[w], lo[w], contrib[w], 0.f);
        }
        warp_two_sum_spread<NV>(hi, lo, lane);
#pragma unroll
        for (int q = 0; q < NV; ++q)
            if (lane == spread_lane(NV, q)) {
                st.hi[q][warp] = hi[0];
                st.lo[q][warp] = lo[0];
            }
    }
    __syncthreads();
    if (warp <= rot_roles(STEP_CAMS))
        step_update<FOCAL, false>(d, st, blockIdx.x * STEP_CAMS, warp, lane, bias_correction(st.hyper[2], t_step),
                                  bias_correction(st.hyper[3], t_step), t_step, apply, true, cam_dst);
}

// iters of these iterations in one cooperative launch, one grid barrier each, for as many cameras as
// resident warps: warp w of a block owns camera 8 block + w for the whole launch, and the records of the
// camera's first 32 image pairs, which do not change, stay in shared memory (a row of 60 floats a
// lane: 16-byte loads free of bank conflicts). The same arithmetic as k_quad_step, bit for bit. What bounds
// an iteration is its serial chain: other cameras' records from L2, geometry and chain rule,
// the compensated sums, the FP64 update and the barrier. 25 iterations on 1,000 cameras and 11,700
// pairs: 114 us, 4.5 us each with the launch, 4.2 in a chain of 1,000 (12.4 us as launches). More cameras than resident warps take k_quad_step, whose
// blocks then overlap each other's latencies (4,000 cameras: 500 blocks, 13 us an iteration).
constexpr int QROW = 60;
constexpr int QUAD_SMEM = STEP_CAMS * 32 * QROW * (int)sizeof(float);

template <bool FOCAL>
__global__ void __launch_bounds__(STEP_CAMS * 32, 2)
k_quad_steps(DevProblem d, int iters, float gscale, float lscale) {
    constexpr int NV = FOCAL ? STEP_VALS : STEP_VALS - 1;   // sums carried per camera
    extern __shared__ __align__(16) float s_rec[];          // [STEP_CAMS][32][QROW]
    __shared__ StepState<STEP_CAMS> st;                      // stays here from iteration to iteration
    __shared__ float s_bc[2][2];                             // bias corrections of this and the next iteration
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cam0 = blockIdx.x * STEP_CAMS, k = cam0 + warp;
    GridBarrier gb(d.grid_state, d.err);
    const int e_begin = k < d.n_cams ? d.cam_off[k] : 0;
    const int e_end = k < d.n_cams ? d.cam_off[k + 1] : 0;
    int n = 0, role = 0, ci = 0, cj = 0;
    auto load_entry = [&](int e) {
        const int ent = d.cam_ent[e];
        n = ent >> 1;
        role = ent & 1;
        ci = d.cam_i[n];
        cj = d.cam_j[n];
    };
    float4 *row = reinterpret_cast<float4 *>(s_rec + (warp * 32 + lane) * QROW);
    if (e_begin + lane < e_end) {
        load_entry(e_begin + lane);
        const float4 *rec = reinterpret_cast<const float4 *>(d.quad + (size_t)n * QREC);
#pragma unroll
        for (int q = 0; q < QREC / 4; ++q) row[q] = rec[q];
    }
    const long long t0 = *d.step;
    st.load(d, d.cam, cam0);
    if (threadIdx.x < 2) s_bc[0][threadIdx.x] = bias_correction((float)d.hyper[2 + threadIdx.x], t0 + 1);
    for (int it = 0; it < iters; ++it) {
        const float *src = (it & 1) ? d.cam_alt : d.cam;
        float *dst = (it & 1) ? d.cam : d.cam_alt;
        if (k < d.n_cams) {
            float hi[STEP_VALS], lo[STEP_VALS];
#pragma unroll
            for (int q = 0; q < STEP_VALS; ++q) hi[q] = lo[q] = 0.f;
            for (int e = e_begin + lane; e < e_end; e += 32) {
                const bool first = e < e_begin + 32;
                if (e_end - e_begin > 32) load_entry(e);
                float g[GEO], sum[10], contrib[STEP_VALS];
                if (!pair_geometry_regs(src, d.cen, ci, cj, g)) atomicOr(d.err, ERR_DEGENERATE);
                form_sums(first ? row : reinterpret_cast<const float4 *>(d.quad + (size_t)n * QREC), g, sum);
                pair_chain_rule<FOCAL>(g, role, sum, gscale, lscale, contrib);
#pragma unroll
                for (int w = 0; w < NV; ++w) two_sum_acc(hi[w], lo[w], contrib[w], 0.f);
            }
            warp_two_sum_spread<NV>(hi, lo, lane);
#pragma unroll
            for (int q = 0; q < NV; ++q)
                if (lane == spread_lane(NV, q)) {
                    st.hi[q][warp] = hi[0];
                    st.lo[q][warp] = lo[0];
                }
        }
        __syncthreads();
        if (warp <= rot_roles(STEP_CAMS))
            step_update<FOCAL, true>(d, st, cam0, warp, lane, s_bc[it & 1][0], s_bc[it & 1][1], t0 + 1 + it, 1,
                                     it + 1 == iters, dst);
        else if (warp == STEP_CAMS - 1 && lane < 2)
            s_bc[(it + 1) & 1][lane] = bias_correction(st.hyper[2 + lane], t0 + 2 + it);
        if (!gb.sync()) return;
    }
    gb.finish();
    if (iters & 1)     // the records end in d.cam
        for (int i = threadIdx.x; i < STEP_CAMS * CAMREC; i += STEP_CAMS * 32)
            if (cam0 + i / CAMREC < d.n_cams) d.cam[(size_t)cam0 * CAMREC + i] = __ldcg(d.cam_alt + (size_t)cam0 * CAMREC + i);
    if (blockIdx.x == 0) finish_step(d, d.n_cams, iters, reinterpret_cast<double *>(s_rec));
}

static inline int blocks_for(int64_t n, int t) { return (int)((n + t - 1) / t); }

// tau < 0: keep the current weights; otherwise reweight with threshold tau in the same pass
void launch_quad_accumulate(const DevProblem &d, float tau, cudaStream_t s) {
    const int grid = d.n_ranges, block = 32;
    if (tau < 0.f) {
        if (d.storage == FM_STORE_FP32) k_quad_accumulate<FM_STORE_FP32, false><<<grid, block, 0, s>>>(d, tau);
        else k_quad_accumulate<FM_STORE_FP16, false><<<grid, block, 0, s>>>(d, tau);
    } else {
        if (d.storage == FM_STORE_FP32) k_quad_accumulate<FM_STORE_FP32, true><<<grid, block, 0, s>>>(d, tau);
        else k_quad_accumulate<FM_STORE_FP16, true><<<grid, block, 0, s>>>(d, tau);
    }
}

void launch_quad_combine(const DevProblem &d, cudaStream_t s) {
    k_quad_combine<<<blocks_for(d.n_pairs, 8), 256, 0, s>>>(d);
}

void launch_quad_step(const DevProblem &d, int it, const float *cam_src, float *cam_dst, bool apply,
                      cudaStream_t s, bool pdl) {
    float gscale, lscale;
    loss_scales(d, gscale, lscale);
    if (d.refine_focal)
        launch_k(k_quad_step<true>, dim3(camera_step_blocks(d)), dim3(STEP_CAMS * 32), s, pdl, d, it, cam_src,
                 cam_dst, gscale, lscale, apply ? 1 : 0);
    else
        launch_k(k_quad_step<false>, dim3(camera_step_blocks(d)), dim3(STEP_CAMS * 32), s, pdl, d, it, cam_src,
                 cam_dst, gscale, lscale, apply ? 1 : 0);
}

cudaError_t quad_steps_capacity(bool focal, int *blocks) {
    auto kernel = focal ? k_quad_steps<true> : k_quad_steps<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, QUAD_SMEM);
    return e == cudaSuccess ? coop_blocks(kernel, STEP_CAMS * 32, blocks, QUAD_SMEM) : e;
}

cudaError_t launch_quad_steps(const DevProblem &d, int iters, cudaStream_t s) {
    float gscale, lscale;
    loss_scales(d, gscale, lscale);
    return launch_coop(d.refine_focal ? k_quad_steps<true> : k_quad_steps<false>, camera_step_blocks(d), STEP_CAMS * 32,
                       QUAD_SMEM, s, d, iters, gscale, lscale);
}

}  // namespace fm
