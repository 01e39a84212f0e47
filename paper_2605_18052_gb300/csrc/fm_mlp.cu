// Learned inlier weights: a small MLP (8 -> 32 -> 32 -> 1, ReLU, sigmoid) that predicts the
// probability p that a point pair is an inlier from its residual history, its match score and
// statistics of its image pair; the reweighting step of the IRLS loop (Sec. "Epipolar
// Adjustment") then uses w = p / max(|eps|, delta). The thesis has no learned component; the
// network, its features and its training follow the benchmark's description.
//
// Numerics (shared by inference and training): features, weights and hidden activations are
// rounded to BF16, every product is accumulated in FP32, biases are FP32.
//   * inference runs inside the streaming walk on the tensor cores (mma.sync BF16, FP32
//     accumulate): 16 point pairs per tile, 19 MMAs per tile; the FP32 accumulator fragments of
//     one layer are the BF16 A fragments of the next after packing;
//   * training runs tiles of samples as register-tiled FP32 products (forward and backward), sums
//     the gradient per block in a fixed order and applies FP32 Adam to FP32 master parameters.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "fm_walk.cuh"

namespace fm {

// ---- per-pair statistics of the current residuals ---------------------------------------------
struct StatsBody {
    const DevProblem &d;
    float tau;
    float acc[2];
    __device__ StatsBody(const DevProblem &dd, float t) : d(dd), tau(t) { acc[0] = acc[1] = 0.f; }
    __device__ __forceinline__ void segment_begin(int) {}
    __device__ __forceinline__ void point(int, float e, float, float, float, float, float) {
        const float a = fabsf(e);
        acc[0] += __logf(a + LOG_FLOOR);
        acc[1] += a <= tau ? 1.f : 0.f;
    }
    __device__ __forceinline__ void segment_end(int seg, int r, int lane, bool) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
        if (lane == 0) {
            d.slots[(size_t)(seg + r) * SLOT] = acc[0];
            d.slots[(size_t)(seg + r) * SLOT + 1] = acc[1];
        }
        acc[0] = acc[1] = 0.f;
    }
    __device__ __forceinline__ void group_done(int, int, int) {}
};

template <int STORE, int S>
__global__ void __launch_bounds__(32) k_pair_stats(DevProblem d, float tau) {
    extern __shared__ __align__(16) unsigned char stage[];
    const int r = blockIdx.x;
    StatsBody body(d, tau);
    walk_range_staged<STORE, false, S>(d, r, threadIdx.x, body, stage, [] {});
}

__global__ void k_pair_stats_combine(DevProblem d) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= d.n_pairs) return;
    const int p0 = d.pair_off[n], p1 = d.pair_off[n + 1];
    float s0 = 0.f, s1 = 0.f;
    for (int r = p0 / WR; r <= (p1 - 1) / WR; ++r) {
        s0 += d.slots[(size_t)(n + r) * SLOT];
        s1 += d.slots[(size_t)(n + r) * SLOT + 1];
    }
    const float cnt = (float)(p1 - p0);
    reinterpret_cast<float4 *>(d.pstat)[n] = make_float4(s0 / cnt, s1 / cnt, logf(cnt) * 0.1f, 0.f);
}

// ---- the network on the tensor cores ---------------------------------------------------------------
// c (16 x 8, FP32) += a (16 x 16, BF16) b (16 x 8), and the same with 8 columns of a
__device__ __forceinline__ void mma_k16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k16_first(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_k8(float (&c)[4], unsigned a0, unsigned a1, unsigned b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(b0));
}

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&v);
}

// max(lo, 0) and max(hi, 0) rounded to BF16 and packed (lo in the low half): one instruction,
// the same bits as pack_bf16(fmaxf(lo, 0), fmaxf(hi, 0))
__device__ __forceinline__ unsigned pack_relu_bf16(float lo, float hi) {
    unsigned d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// v = hi + mid + lo with three BF16 values (exact for FP32 v up to the last bit of lo)
__device__ __forceinline__ void bf16_split3(float v, float &hi, float &mid, float &lo) {
    hi = __bfloat162float(__float2bfloat16_rn(v));
    mid = __bfloat162float(__float2bfloat16_rn(v - hi));
    lo = v - hi - mid;
}

// The B operands of the three layers, in registers. For lane (g = lane / 4, t = lane % 4) and the n-tile
// j the register b0 holds W[k][8j + g] for k = 2t, 2t + 1, b1 for k = 2t + 8, 2t + 9. A layer's bias
// is three BF16 parts (hi + mid + lo = b) against three constant-1 columns of its A operand, so
// that it is added inside the FP32 accumulation: layer 1 in columns 8..10 beside the 8 features, layers
// 2 and 3 as a slice of 8 columns after their 32 inputs. The output layer has its vector in every column,
// so that every lane of a row's quad gets the row's value.
struct NetFrag {
    unsigned w1[4][2], w2[2][4][2], b2[4], w3[2][2], b3;
    unsigned ones;        // the lane's pair of the constant columns
    __device__ __forceinline__ void load(const float *master, const __nv_bfloat16 *wbf, int lane) {
        const int g = lane >> 2, t = lane & 3;
        const __nv_bfloat16 *W1 = wbf, *W2 = wbf + MLP_IN * MLP_H, *W3 = W2 + MLP_H * MLP_H;
        auto pk = [](__nv_bfloat16 lo, __nv_bfloat16 hi) {
            return (unsigned)__bfloat16_as_ushort(lo) | ((unsigned)__bfloat16_as_ushort(hi) << 16);
        };
        auto bias = [&](float v) {   // the lane's pair of (hi, mid, lo, 0, ...)
            float h, m, l;
            bf16_split3(v, h, m, l);
            return t == 0 ? pack_bf16(h, m) : (t == 1 ? pack_bf16(l, 0.f) : 0u);
        };
        ones = t == 0 ? pack_bf16(1.f, 1.f) : (t == 1 ? pack_bf16(1.f, 0.f) : 0u);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            w1[j][0] = pk(W1[(2 * t) * MLP_H + 8 * j + g], W1[(2 * t + 1) * MLP_H + 8 * j + g]);
            w1[j][1] = bias(master[MLP_OFF_B1 + 8 * j + g]);
            b2[j] = bias(master[MLP_OFF_B2 + 8 * j + g]);
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = 16 * s + 8 * h + 2 * t;
                    w2[s][j][h] = pk(W2[k * MLP_H + 8 * j + g], W2[(k + 1) * MLP_H + 8 * j + g]);
                }
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int h = 0; h < 2; ++h) w3[s][h] = pk(W3[16 * s + 8 * h + 2 * t], W3[16 * s + 8 * h + 2 * t + 1]);
        b3 = bias(master[MLP_OFF_B3]);
    }
    // the network's logit of a tile's 16 rows: z0 of row g, z1 of row g + 8; f0, f1: the lane's pair of
    // the features of those rows
    __device__ __forceinline__ void tile(unsigned f0, unsigned f1, float &z0, float &z1) const {
        const unsigned a1[4] = {f0, f1, ones, ones};
        float h[4][4];
        unsigned a[2][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_k16_first(h[j], a1, w1[j][0], w1[j][1]);
        auto pack = [&]() {   // an accumulator tile of one layer is an A operand of the next
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                a[s][0] = pack_relu_bf16(h[2 * s][0], h[2 * s][1]);
                a[s][1] = pack_relu_bf16(h[2 * s][2], h[2 * s][3]);
                a[s][2] = pack_relu_bf16(h[2 * s + 1][0], h[2 * s + 1][1]);
                a[s][3] = pack_relu_bf16(h[2 * s + 1][2], h[2 * s + 1][3]);
            }
        };
        pack();
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_k16_first(h[j], a[0], w2[0][j][0], w2[0][j][1]);
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_k16(h[j], a[1], w2[1][j][0], w2[1][j][1]);
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_k8(h[j], ones, ones, b2[j]);
        pack();
        float z[4];
        mma_k16_first(z, a[0], w3[0][0], w3[0][1]);
        mma_k16(z, a[1], w3[1][0], w3[1][1]);
        mma_k8(z, ones, ones, b3);
        z0 = z[0];
        z1 = z[2];
    }
};

// learned IRLS weight p / max(|eps|, delta) (fast quotient, within 2 ulp; every learned kernel
// uses this one expression, so the fused and separate passes agree bit for bit)
__device__ __forceinline__ float learned_weight(float p, float ae, float delta) {
    return __fdividef(p, fmaxf(ae, delta));
}

// ---- features of a point pair ---------------------------------------------------------------------
//  0 log(|e|+1e-6) - log(tau)      1 log(|e|+1e-6) - pair mean log    2 log(|e_prev|+1e-6) - log(|e|+1e-6)
//  3 match score                   4 pair fraction with |e| <= tau    5 log(pair count) / 10
//  6 round / 10                    7 log(|e_prev|+1e-6) - log(tau)
template <int STORE>
struct CollectBody {
    static constexpr int PPL = Fmt<STORE>::PPL;
    const DevProblem &d;
    float log_tau, round_f;
    int hist_valid;
    float st_mean, st_frac, st_cnt;
    float le[PPL], sm[PPL], sf[PPL], sc[PPL];
    __nv_bfloat16 *feat_out;
    __device__ CollectBody(const DevProblem &dd) : d(dd) {}
    __device__ __forceinline__ void segment_begin(int seg) {
        const float4 p = reinterpret_cast<const float4 *>(d.pstat)[seg];
        st_mean = p.x;
        st_frac = p.y;
        st_cnt = p.z;
    }
    __device__ __forceinline__ void point(int k, float e, float, float, float, float, float) {
        le[k] = __logf(fabsf(e) + LOG_FLOOR);
        sm[k] = st_mean;
        sf[k] = st_frac;
        sc[k] = st_cnt;
    }
    __device__ __forceinline__ void segment_end(int, int, int, bool) {}
    __device__ __forceinline__ void group_done(int gb, int p_end, int lane) {
        const int q = gb + lane * PPL;
        float lp[PPL], sco[PPL];
#pragma unroll
        for (int k = 0; k < PPL; ++k) {
            lp[k] = hist_valid ? __half2float(d.le_hist[q + k]) : le[k];
            sco[k] = __half2float(d.score[q + k]);
        }
#pragma unroll
        for (int k = 0; k < PPL; ++k) {
            if (q + k >= p_end) continue;
            const int64_t dst = d.perm ? d.perm[q + k] : q + k;
            *reinterpret_cast<uint4 *>(feat_out + dst * MLP_IN) =
                make_uint4(pack_bf16(le[k] - log_tau, le[k] - sm[k]), pack_bf16(lp[k] - le[k], sco[k]),
                           pack_bf16(sf[k], sc[k]), pack_bf16(round_f, lp[k] - log_tau));
            d.le_hist[q + k] = __float2half_rn(le[k]);
        }
#pragma unroll
        for (int k = 0; k < PPL; ++k) le[k] = 0.f;
    }
};

// Two chunks in flight in either storage: the history, the scores and the scattered rows are not staged, so
// their latency is hidden by warps alone, and 10 KB a block (4 chunks) leave 20 warps an SM. FP32, 20.0 M point
// pairs, 12,000 / 50,000 / 200,000 image pairs: 4 chunks, groups one by one 333 / 352 / 427 us, 2 chunks 281 / 293 / 356,
// 2 chunks and four groups in straight code 241 / 264 / 355 (FP16: 198 / 214 / 272 one by one, 195 / 208 / 269).
constexpr int COLLECT_STAGES = 2;

template <int STORE>
__global__ void __launch_bounds__(32)
k_collect_features(DevProblem d, float tau, int round, int hist_valid, __nv_bfloat16 *feat_out) {
    __shared__ __align__(16) unsigned char stage[COLLECT_STAGES * STAGE_BYTES];
    const int r = blockIdx.x;
    CollectBody<STORE> body(d);
    body.log_tau = __logf(tau);
    body.round_f = round * 0.1f;
    body.hist_valid = hist_valid;
    body.feat_out = feat_out;
    walk_range_staged<STORE, false, COLLECT_STAGES>(d, r, threadIdx.x, body, stage, [] {});
}

// ---- the learned reweighting -------------------------------------------------------------------------
// A warp streams its range in blocks of 64 point pairs, two per lane: features, the network's logit, the
// weight (written, and rounded as the storage keeps it), the residual history; FUSE: also the loss
// and adjoint sums with the new weights (the round's first pass), closing every image pair that ends in
// the block, in the streaming pass's order.
// The network runs on mma.sync tiles of 16 rows, four per block, wholly in registers: the accumulators
// of one layer, rounded by one instruction per two values, are the A operand of the next, the weights
// stay in 34 registers for the whole range, and there is no barrier. Row g of tile T is the first point
// pair of lane 4 g + T and row g + 8 its second, so that only the features change lanes (one 16-byte
// shared store per point pair, one ldmatrix per two tiles) and a lane finds its own logits in its
// accumulators. On fifth-generation tensor memory (tcgen05, M = 128 over a warpgroup) the same products
// are an eighth of the tensor work, but three MMA round trips through shared memory, an mbarrier and
// TMEM per 128 rows, and 296 instructions per point pair: 837 us on 48.9 M point pairs (FP16,
// fused), 127 us on 3.1 M (FP32, weights only). Both give the same bits (each product of 16 terms and
// its FP32 accumulation are rounded alike; compared on 3.3 M random outputs). Now 618 and 56 us, at 240
// instructions per point pair; the tensor pipe is 62% busy (8.3 cycles per mma.sync and
// sub-partition: 415 us on 48.9 M if it never waited), the rest is the latency of a block's phases with
// four warps per sub-partition. Two tiles interleaved by hand, with 4 or 3 blocks per SM, changed
// nothing (619, 637 us); 5 blocks an SM spill far more (818 us; at 4, 128 registers, the fused
// variants spill 28 bytes).
constexpr int LP_WARPS = 4;
constexpr int LP_BLOCK = 64;                // point pairs per warp and step
constexpr int LP_STAGES = 4;                // steps whose loads are in flight
constexpr int LP_STAGE_BYTES = LP_BLOCK * (16 + 2 + 2);   // keypoints (FP32 size), scores, history

template <int STORE, bool FUSE>
__global__ void __launch_bounds__(LP_WARPS * 32, 4)
k_learned_pass(DevProblem d, const float *master, const __nv_bfloat16 *wbf, float tau, float tau_cap, int round,
               int hist_valid) {
    using F = Fmt<STORE>;
    constexpr int PPL = F::PPL, SUBS = 2 / PPL, GROUP = 32 * PPL;   // SUBS groups of GROUP point pairs per step
    constexpr int KP_BYTES = LP_BLOCK * (STORE == FM_STORE_FP32 ? 16 : 8);
    __shared__ __align__(16) unsigned char s_stage[LP_WARPS][LP_STAGES][LP_STAGE_BYTES];
    __shared__ __align__(16) uint4 s_feat[LP_WARPS][2 * 36];        // [slot][tile][row], 9 rows a tile
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = lane & 3;
    NetFrag net;
    net.load(master, wbf, lane);
    pdl_trigger();   // the camera step behind the fused pass may be scheduled
    const int r = blockIdx.x * LP_WARPS + warp;
    if (r >= d.n_ranges) return;
    const float log_tau = __logf(tau), delta = (float)d.delta, wscale = d.w_scale, round_f = round * 0.1f;
    const int p_begin = r * WR, p_end = (int)min((int64_t)p_begin + WR, d.n_pp);
    const int steps = (p_end - p_begin + LP_BLOCK - 1) / LP_BLOCK;
    auto request = [&](int c) {
        if (c < steps) {
            unsigned char *dst = s_stage[warp][c % LP_STAGES];
            const size_t q = (size_t)p_begin + (size_t)c * LP_BLOCK;
            const unsigned char *kp = static_cast<const unsigned char *>(d.kp) + q * (KP_BYTES / LP_BLOCK);
#pragma unroll
            for (int u = 0; u < KP_BYTES / 512; ++u) cp_async16(dst + (u * 32 + lane) * 16, kp + (u * 32 + lane) * 16);
            if (lane < 16) {   // 64 scores (lanes 0..7) and 64 history values (8..15)
                const __half *src = lane < 8 ? d.score : d.le_hist;
                cp_async16(dst + KP_BYTES + lane * 16, src + q + (lane & 7) * 8);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int c = 0; c < LP_STAGES; ++c) request(c);
    int seg = d.range_pair[r], seg_end = d.pair_off[seg + 1];
    LossBody<MODE_LOSS_IRLS> loss(d);
    unsigned kept = 0;
    float E[9];
    load_E(d.geo, seg, E);
    float4 st = reinterpret_cast<const float4 *>(d.pstat)[seg];
    uint4 *feat = s_feat[warp];
    const int my_row = (lane & 3) * 9 + (lane >> 2);
    const uint32_t frag_row = (uint32_t)__cvta_generic_to_shared(feat + ((lane >> 3) & 1) * 36 + (lane >> 4) * 9 + (lane & 7));
    for (int c = 0; c < steps; ++c) {
        const int b0 = p_begin + c * LP_BLOCK;
        asm volatile("cp.async.wait_group %0;" ::"n"(LP_STAGES - 1) : "memory");
        __syncwarp();
        const unsigned char *src = s_stage[warp][c % LP_STAGES];
        uint4 kp[SUBS];
#pragma unroll
        for (int u = 0; u < SUBS; ++u) kp[u] = *reinterpret_cast<const uint4 *>(src + (u * 32 + lane) * 16);
        float sco[2], lp[2];
        {
            const __half *sc = reinterpret_cast<const __half *>(src + KP_BYTES), *hs = sc + LP_BLOCK;
            if (PPL == 2) {
                const float2 a = __half22float2(reinterpret_cast<const __half2 *>(sc)[lane]);
                const float2 b = __half22float2(reinterpret_cast<const __half2 *>(hs)[lane]);
                sco[0] = a.x;
                sco[1] = a.y;
                lp[0] = b.x;
                lp[1] = b.y;
            } else {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    sco[k] = __half2float(sc[32 * k + lane]);
                    lp[k] = __half2float(hs[32 * k + lane]);
                }
            }
        }
        // ---- features of the lane's two point pairs
        const int seg0 = seg, seg0_end = seg_end;
        float x1[2], y1[2], x2[2], y2[2], e[2], le[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            typename F::Raw raw;
            raw.kp = kp[k / PPL];
            raw.w = 0u;
            float unused;
            F::get(raw, k % PPL, x1[k], y1[k], x2[k], y2[k], unused);
            e[k] = le[k] = 0.f;
        }
        auto feature = [&](int k) {
            e[k] = epi(E, x1[k], y1[k], x2[k], y2[k]);
            le[k] = __logf(fabsf(e[k]) + LOG_FLOOR);
            const float lpk = hist_valid ? lp[k] : le[k];
            feat[k * 36 + my_row] = make_uint4(pack_bf16(le[k] - log_tau, le[k] - st.x), pack_bf16(lpk - le[k], sco[k]),
                                               pack_bf16(st.y, st.z), pack_bf16(round_f, lpk - log_tau));
        };
        const bool whole = b0 + LP_BLOCK <= seg_end;   // one image pair, no end of the range
        if (whole) {
            feature(0);
            feature(1);
        } else {
#pragma unroll
            for (int u = 0; u < SUBS; ++u) {
                const int gb = b0 + u * GROUP, g_end = min(gb + GROUP, p_end);
                int lo = gb;
                while (lo < g_end) {
                    const int hi = min(seg_end, g_end);
#pragma unroll
                    for (int k = 0; k < PPL; ++k) {
                        const int q = gb + lane * PPL + k;
                        if (q >= lo && q < hi) feature(u * PPL + k);
                    }
                    lo = hi;
                    if (seg_end >= g_end) break;
                    ++seg;
                    seg_end = d.pair_off[seg + 1];
                    load_E(d.geo, seg, E);
                    st = reinterpret_cast<const float4 *>(d.pstat)[seg];
                }
#pragma unroll
                for (int k = 0; k < PPL; ++k)   // rows past the end of the range: any finite input
                    if (gb + lane * PPL + k >= p_end) feat[(u * PPL + k) * 36 + my_row] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        __syncwarp();
        // ---- the network
        float z[2] = {0.f, 0.f};
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            unsigned f[4];
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3])
                         : "r"(frag_row + (uint32_t)(m * 2 * 9 * 16))
                         : "memory");
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float z0, z1;
                net.tile(f[2 * h], f[2 * h + 1], z0, z1);
                z[0] = t == 2 * m + h ? z0 : z[0];
                z[1] = t == 2 * m + h ? z1 : z[1];
            }
        }
        __syncwarp();   // the features and the stage have been read
        request(c + LP_STAGES);
        // ---- weights, history, kept count
        float w[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int q = b0 + (k / PPL) * GROUP + lane * PPL + k % PPL;
            const float pk = __frcp_rn(1.f + __expf(-z[k]));
            const float ae = fabsf(e[k]);
            const bool in = q < p_end && ae <= tau_cap;
            const float wf = in ? learned_weight(pk, ae, delta) : 0.f;
            w[k] = STORE == FM_STORE_FP32 ? wf : __half2float(__float2half_rn(wf * wscale));
            kept += in ? 1u : 0u;
        }
        if (PPL == 2) {
            const int q = b0 + 2 * lane;
            reinterpret_cast<__half2 *>(d.w)[q >> 1] = __floats2half2_rn(w[0], w[1]);
            const __half2 hv = __floats2half2_rn(le[0], le[1]);
            if (q + 1 < p_end) reinterpret_cast<__half2 *>(d.le_hist)[q >> 1] = hv;
            else if (q < p_end) d.le_hist[q] = __low2half(hv);
        } else {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int q = b0 + 32 * k + lane;
                static_cast<float *>(d.w)[q] = w[k];
                if (q < p_end) d.le_hist[q] = __float2half_rn(le[k]);
            }
        }
        if (!FUSE) continue;
        // ---- loss and adjoint sums with the new weights
        if (whole) {
#pragma unroll
            for (int k = 0; k < 2; ++k) loss.point(k, e[k], x1[k], y1[k], x2[k], y2[k], w[k]);
        } else {
            int sb = seg0, sb_end = seg0_end;
#pragma unroll
            for (int u = 0; u < SUBS; ++u) {
                const int gb = b0 + u * GROUP, g_end = min(gb + GROUP, p_end);
                int lo = gb;
                while (lo < g_end) {
                    const int hi = min(sb_end, g_end);
#pragma unroll
                    for (int k = 0; k < PPL; ++k) {
                        const int q = gb + lane * PPL + k, i = u * PPL + k;
                        if (q >= lo && q < hi) loss.point(i, e[i], x1[i], y1[i], x2[i], y2[i], w[i]);
                    }
                    lo = hi;
                    if (sb_end >= g_end) break;
                    loss.segment_end(sb, r, lane, false);
                    ++sb;
                    sb_end = d.pair_off[sb + 1];
                }
            }
        }
    }
    if (FUSE) loss.segment_end(seg, r, lane, true);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
    if (lane == 0 && kept) atomicAdd(d.counter, (unsigned long long)kept);
}

static inline int blocks_for(int64_t n, int t) { return (int)((n + t - 1) / t); }

void launch_learned_loss(const DevProblem &d, const float *master, const __nv_bfloat16 *wbf, float tau,
                         float tau_cap, int round, int hist_valid, cudaStream_t s) {
    const dim3 grid(blocks_for(d.n_ranges, LP_WARPS)), block(LP_WARPS * 32);
    if (d.storage == FM_STORE_FP32)
        k_learned_pass<FM_STORE_FP32, true><<<grid, block, 0, s>>>(d, master, wbf, tau, tau_cap, round, hist_valid);
    else
        k_learned_pass<FM_STORE_FP16, true><<<grid, block, 0, s>>>(d, master, wbf, tau, tau_cap, round, hist_valid);
}

void launch_pair_stats(const DevProblem &d, float tau, cudaStream_t s) {
    with_stages<RECORD_STAGES>(d, [&](auto store, auto depth) {
        constexpr int STORE = decltype(store)::value, S = decltype(depth)::value;
        k_pair_stats<STORE, S><<<d.n_ranges, 32, S * STAGE_BYTES, s>>>(d, tau);
    });
    k_pair_stats_combine<<<blocks_for(d.n_pairs, 128), 128, 0, s>>>(d);
}

void launch_learned_weights(const DevProblem &d, const float *master, const __nv_bfloat16 *wbf, float tau,
                            float tau_cap, int round, int hist_valid, cudaStream_t s) {
    const dim3 grid(blocks_for(d.n_ranges, LP_WARPS)), block(LP_WARPS * 32);
    if (d.storage == FM_STORE_FP32)
        k_learned_pass<FM_STORE_FP32, false><<<grid, block, 0, s>>>(d, master, wbf, tau, tau_cap, round, hist_valid);
    else
        k_learned_pass<FM_STORE_FP16, false><<<grid, block, 0, s>>>(d, master, wbf, tau, tau_cap, round, hist_valid);
}

void launch_collect_features(const DevProblem &d, float tau, int round, int hist_valid,
                             __nv_bfloat16 *feat, cudaStream_t s) {
    if (d.storage == FM_STORE_FP32)
        k_collect_features<FM_STORE_FP32><<<d.n_ranges, 32, 0, s>>>(d, tau, round, hist_valid, feat);
    else
        k_collect_features<FM_STORE_FP16><<<d.n_ranges, 32, 0, s>>>(d, tau, round, hist_valid, feat);
}

// ---- training: register-tiled forward and backward, block-level gradient sums, FP32 Adam --------
constexpr int TRAIN_THREADS = 128;

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// forward with BF16 weights (wf, from the BF16 copies) and FP32 biases; returns z3 and fills
// h1b, h2b (BF16-rounded activations) and the ReLU masks
__device__ __forceinline__ float mlp_forward_thread(const float *wf, const float *x, float *h1b, float *h2b,
                                                    unsigned &m1, unsigned &m2) {
    const float *W1 = wf + MLP_OFF_W1, *b1 = wf + MLP_OFF_B1, *W2 = wf + MLP_OFF_W2, *b2 = wf + MLP_OFF_B2,
                *W3 = wf + MLP_OFF_W3;
    m1 = m2 = 0u;
    for (int j = 0; j < MLP_H; ++j) {
        float z = b1[j];
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) z = fmaf(x[k], W1[k * MLP_H + j], z);
        if (z > 0.f) m1 |= 1u << j;
        h1b[j] = bf16r(fmaxf(z, 0.f));
    }
    for (int j = 0; j < MLP_H; ++j) {
        float z = b2[j];
        for (int k = 0; k < MLP_H; ++k) z = fmaf(h1b[k], W2[k * MLP_H + j], z);
        if (z > 0.f) m2 |= 1u << j;
        h2b[j] = bf16r(fmaxf(z, 0.f));
    }
    float z3 = wf[MLP_OFF_B3];
    for (int k = 0; k < MLP_H; ++k) z3 = fmaf(h2b[k], W3[k], z3);
    return z3;
}

__device__ __forceinline__ void load_weights_smem(float *wf, const float *master, const __nv_bfloat16 *wbf) {
    for (int q = threadIdx.x; q < MLP_NPARAM; q += blockDim.x) {
        float v;
        if (q < MLP_OFF_B1) v = __bfloat162float(wbf[q]);
        else if (q < MLP_OFF_W2) v = master[q];
        else if (q < MLP_OFF_B2) v = __bfloat162float(wbf[q - MLP_H]);
        else if (q < MLP_OFF_W3) v = master[q];
        else if (q < MLP_OFF_B3) v = __bfloat162float(wbf[q - 2 * MLP_H]);
        else v = master[q];
        wf[q] = v;
    }
}

// Gradient sums of tiles of TG_T samples. A tile goes through the network as small matrix products
// with the operands in shared memory, one value per (unit, sample), and a register tile of 4
// samples x 4 units per thread: units jg + 8c (c = 0..3) for jg = tid % 8, samples 4 sg .. 4 sg + 3
// for sg = tid / 8, so the eight threads that share a sample sit in one warp and the sums over the
// units of the output layer are three shuffles. Weights are stored permuted (the four units of a
// thread adjacent), activations with a row stride of TG_LD floats: every 16-byte shared load is
// free of bank conflicts and feeds 8 multiply-adds. (One sample per thread with rows of 32 floats
// put all 32 lanes of a warp on one bank: 46 us a launch at 16,384 samples; 10.3 us now.)
// FP32 throughout: weights and hidden activations are BF16 values held in FP32, as in inference.
// A block walks tiles blockIdx.x, blockIdx.x + gridDim.x, ... with its 1377 sums in registers and
// writes them once, in a fixed order: results are bit-reproducible.
constexpr int TG_T = 64;                 // samples per tile
constexpr int TG_LD = TG_T + 4;          // row stride: 8 consecutive rows cover the 32 banks
constexpr int TG_ROW = 1408;             // floats per block partial: 1377 sums, the loss, padding
constexpr int TG_BLOCKS = 304;           // most blocks: two per SM

struct TrainSmem {
    float4 w1[MLP_IN][8];                // w1[k][jg] = W1[k][jg + 8c]
    float4 w2[MLP_H][8];                 // w2[k][jg] = W2[k][jg + 8c]
    float4 w2t[MLP_H][8];                // w2t[j][kg] = W2[kg + 8c][j]
    float4 b1[8], b2[8], w3[8];
    float x[MLP_IN][TG_LD], h1[MLP_H][TG_LD], dz2[MLP_H][TG_LD], dz1[MLP_H][TG_LD];
    float y[TG_T];
    float red[TRAIN_THREADS / 32][MLP_H + 2];
};

__global__ void __launch_bounds__(TRAIN_THREADS)
k_mlp_grad(const float *master, const __nv_bfloat16 *wbf, const __nv_bfloat16 *feat, const float *labels, int n,
           float inv_n, float *gpart) {
    __shared__ TrainSmem sm;
    const int tid = threadIdx.x, jg = tid & 7, sg = tid >> 3, lane = tid & 31, warp = tid >> 5;
    pdl_wait();     // the parameters of the previous step, the caller's samples
    pdl_trigger();
    {
        const __nv_bfloat16 *W1 = wbf, *W2 = wbf + MLP_IN * MLP_H, *W3 = W2 + MLP_H * MLP_H;
        for (int q = tid; q < MLP_IN * MLP_H; q += TRAIN_THREADS) {
            const int k = q / MLP_H, j = q % MLP_H;
            reinterpret_cast<float *>(sm.w1[k])[4 * (j & 7) + (j >> 3)] = __bfloat162float(W1[q]);
        }
        for (int q = tid; q < MLP_H * MLP_H; q += TRAIN_THREADS) {
            const int k = q / MLP_H, j = q % MLP_H;
            const float v = __bfloat162float(W2[q]);
            reinterpret_cast<float *>(sm.w2[k])[4 * (j & 7) + (j >> 3)] = v;
            reinterpret_cast<float *>(sm.w2t[j])[4 * (k & 7) + (k >> 3)] = v;
        }
        if (tid < MLP_H) {
            const int o = 4 * (tid & 7) + (tid >> 3);
            reinterpret_cast<float *>(sm.b1)[o] = master[MLP_OFF_B1 + tid];
            reinterpret_cast<float *>(sm.b2)[o] = master[MLP_OFF_B2 + tid];
            reinterpret_cast<float *>(sm.w3)[o] = __bfloat162float(W3[tid]);
        }
    }
    const float b3 = master[MLP_OFF_B3];
    const bool wide = (reinterpret_cast<uintptr_t>(feat) & 15) == 0;
    // the block's sums: W2 rows 2 kp, 2 kp + 1 (kp = tid / 8) x columns jg + 8c; W1 row tid / 16 x
    // columns tid % 16 (+ 16); a bias unit per thread (b1: tid < 32, b2: 32 <= tid < 64)
    float g2[2][4] = {}, g1[2] = {}, gb = 0.f, g3[4] = {}, gb3 = 0.f, gl = 0.f;
    for (int64_t base = (int64_t)blockIdx.x * TG_T; base < n; base += (int64_t)gridDim.x * TG_T) {
        __syncthreads();   // the weights, and the last tile's readers
        if (tid < TG_T) {
            const int64_t s = base + tid;
            __align__(16) __nv_bfloat16 xv[MLP_IN];
            *reinterpret_cast<uint4 *>(xv) = make_uint4(0u, 0u, 0u, 0u);
            if (s < n) {
                if (wide) *reinterpret_cast<uint4 *>(xv) = *reinterpret_cast<const uint4 *>(feat + s * MLP_IN);
                else
#pragma unroll
                    for (int k = 0; k < MLP_IN; ++k) xv[k] = feat[s * MLP_IN + k];
            }
#pragma unroll
            for (int k = 0; k < MLP_IN; ++k) sm.x[k][tid] = __bfloat162float(xv[k]);
            sm.y[tid] = s < n ? labels[s] : 0.f;
        }
        __syncthreads();
        float acc[4][4];   // [unit c][sample]
        unsigned m1 = 0u, m2 = 0u;
        // layer 1
        {
            const float4 b = sm.b1[jg];
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[c][i] = bv[c];
#pragma unroll
            for (int k = 0; k < MLP_IN; ++k) {
                const float4 xv = *reinterpret_cast<const float4 *>(&sm.x[k][4 * sg]);
                const float4 wv = sm.w1[k][jg];
                const float xs[4] = {xv.x, xv.y, xv.z, xv.w}, ws[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[c][i] = fmaf(xs[i], ws[c], acc[c][i]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float h[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (acc[c][i] > 0.f) m1 |= 1u << (4 * c + i);
                    h[i] = bf16r(fmaxf(acc[c][i], 0.f));
                }
                *reinterpret_cast<float4 *>(&sm.h1[jg + 8 * c][4 * sg]) = make_float4(h[0], h[1], h[2], h[3]);
            }
        }
        __syncwarp();   // a sample's units belong to one warp
        // layer 2 and the output
        float z3[4], dz3[4];
        {
            const float4 b = sm.b2[jg];
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[c][i] = bv[c];
#pragma unroll 8
            for (int k = 0; k < MLP_H; ++k) {
                const float4 xv = *reinterpret_cast<const float4 *>(&sm.h1[k][4 * sg]);
                const float4 wv = sm.w2[k][jg];
                const float xs[4] = {xv.x, xv.y, xv.z, xv.w}, ws[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[c][i] = fmaf(xs[i], ws[c], acc[c][i]);
            }
            const float4 w3v = sm.w3[jg];
            const float w3[4] = {w3v.x, w3v.y, w3v.z, w3v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) z3[i] = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (acc[c][i] > 0.f) m2 |= 1u << (4 * c + i);
                    acc[c][i] = bf16r(fmaxf(acc[c][i], 0.f));
                    z3[i] = fmaf(acc[c][i], w3[c], z3[i]);
                }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) z3[i] += __shfl_xor_sync(0xffffffffu, z3[i], o);
                z3[i] += b3;
                const bool valid = base + 4 * sg + i < n;
                const float y = sm.y[4 * sg + i];
                const float p = 1.f / (1.f + expf(-z3[i]));
                dz3[i] = valid ? (p - y) * inv_n : 0.f;
                if (jg == 0) {
                    gb3 += dz3[i];
                    gl += valid ? fmaxf(z3[i], 0.f) - z3[i] * y + log1pf(expf(-fabsf(z3[i]))) : 0.f;
                }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    g3[c] = fmaf(acc[c][i], dz3[i], g3[c]);
                    d[i] = ((m2 >> (4 * c + i)) & 1u) ? w3[c] * dz3[i] : 0.f;
                }
                *reinterpret_cast<float4 *>(&sm.dz2[jg + 8 * c][4 * sg]) = make_float4(d[0], d[1], d[2], d[3]);
            }
        }
        __syncwarp();
        // dz1 = mask1 . (W2 dz2)
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[c][i] = 0.f;
#pragma unroll 8
        for (int j = 0; j < MLP_H; ++j) {
            const float4 xv = *reinterpret_cast<const float4 *>(&sm.dz2[j][4 * sg]);
            const float4 wv = sm.w2t[j][jg];
            const float xs[4] = {xv.x, xv.y, xv.z, xv.w}, ws[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[c][i] = fmaf(ws[c], xs[i], acc[c][i]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float d[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i] = ((m1 >> (4 * c + i)) & 1u) ? acc[c][i] : 0.f;
            *reinterpret_cast<float4 *>(&sm.dz1[jg + 8 * c][4 * sg]) = make_float4(d[0], d[1], d[2], d[3]);
        }
        __syncthreads();
        // weight gradients: sums over the tile's samples
        const int kp = tid >> 3, k1 = tid >> 4, j1 = tid & 15;
        const float *brow = tid < MLP_H ? sm.dz1[tid] : sm.dz2[tid & (MLP_H - 1)];
#pragma unroll 4
        for (int s = 0; s < TG_T; s += 4) {
            float4 a[2], d[4];
#pragma unroll
            for (int r = 0; r < 2; ++r) a[r] = *reinterpret_cast<const float4 *>(&sm.h1[2 * kp + r][s]);
#pragma unroll
            for (int c = 0; c < 4; ++c) d[c] = *reinterpret_cast<const float4 *>(&sm.dz2[jg + 8 * c][s]);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    g2[r][c] = fmaf(a[r].w, d[c].w, fmaf(a[r].z, d[c].z, fmaf(a[r].y, d[c].y, fmaf(a[r].x, d[c].x, g2[r][c]))));
            const float4 xv = *reinterpret_cast<const float4 *>(&sm.x[k1][s]);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float4 e = *reinterpret_cast<const float4 *>(&sm.dz1[j1 + 16 * r][s]);
                g1[r] = fmaf(xv.w, e.w, fmaf(xv.z, e.z, fmaf(xv.y, e.y, fmaf(xv.x, e.x, g1[r]))));
            }
            if (warp < 2) {
                const float4 e = *reinterpret_cast<const float4 *>(&brow[s]);
                gb += (e.x + e.y) + (e.z + e.w);
            }
        }
    }
    // the block's partial
    float *gout = gpart + (size_t)blockIdx.x * TG_ROW;
    const int kp = tid >> 3;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) gout[MLP_OFF_W2 + (2 * kp + r) * MLP_H + jg + 8 * c] = g2[r][c];
#pragma unroll
    for (int r = 0; r < 2; ++r) gout[MLP_OFF_W1 + (tid >> 4) * MLP_H + (tid & 15) + 16 * r] = g1[r];
    if (tid < MLP_H) gout[MLP_OFF_B1 + tid] = gb;
    else if (tid < 2 * MLP_H) gout[MLP_OFF_B2 + tid - MLP_H] = gb;
    // the output layer's sums over the samples: lanes with equal jg, then the four warps
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) g3[c] += __shfl_xor_sync(0xffffffffu, g3[c], o);
        gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
        gl += __shfl_xor_sync(0xffffffffu, gl, o);
    }
    if (lane < 8)
#pragma unroll
        for (int c = 0; c < 4; ++c) sm.red[warp][lane + 8 * c] = g3[c];
    if (lane == 0) {
        sm.red[warp][MLP_H] = gb3;
        sm.red[warp][MLP_H + 1] = gl;
    }
    __syncthreads();
    if (tid < MLP_H + 2) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < TRAIN_THREADS / 32; ++w) v += sm.red[w][tid];
        gout[MLP_OFF_W3 + tid] = v;   // W3, b3, and the loss behind them
    }
}

__global__ void k_mlp_refresh(const float *master, __nv_bfloat16 *wbf) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < MLP_NPARAM; q += gridDim.x * blockDim.x) {
        if (q < MLP_OFF_B1) wbf[q] = __float2bfloat16_rn(master[q]);
        else if (q >= MLP_OFF_W2 && q < MLP_OFF_B2) wbf[q - MLP_H] = __float2bfloat16_rn(master[q]);
        else if (q >= MLP_OFF_W3 && q < MLP_OFF_B3) wbf[q - 2 * MLP_H] = __float2bfloat16_rn(master[q]);
    }
}

// Adam on the sum of the block partials: 32 parameters per block, eight warps share the partials
// (coalesced rows, a fixed order), one warp takes the step and refreshes the BF16 copies. The
// column behind the parameters is the loss. (One block for all parameters, each thread adding the
// partials of its parameters one after the other, took 21 us at 128 partials; 3.5 us now at 256.)
constexpr int ADAM_ROWS = 8;
static_assert(TG_ROW % 32 == 0 && TG_ROW > MLP_NPARAM, "a block partial holds the parameters and the loss");

__global__ void __launch_bounds__(32 * ADAM_ROWS)
k_mlp_adam(float *master, __nv_bfloat16 *wbf, float *m, float *v, const float *gpart, int nblocks, float lr, float bc1,
           float bc2, float inv_n, float *loss_out) {
    __shared__ float red[ADAM_ROWS][32];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int q = blockIdx.x * 32 + lane;
    pdl_wait();     // the block partials
    pdl_trigger();
    float s = 0.f;
    if (q <= MLP_NPARAM)
#pragma unroll 4
        for (int b = row; b < nblocks; b += ADAM_ROWS) s += gpart[(size_t)b * TG_ROW + q];
    red[row][lane] = s;
    __syncthreads();
    if (row != 0 || q > MLP_NPARAM) return;
    float g = 0.f;
#pragma unroll
    for (int r = 0; r < ADAM_ROWS; ++r) g += red[r][lane];
    if (q == MLP_NPARAM) {
        *loss_out = g * inv_n;
        return;
    }
    const float mq = 0.9f * m[q] + 0.1f * g;
    const float vq = 0.999f * v[q] + 0.001f * g * g;
    m[q] = mq;
    v[q] = vq;
    const float p = master[q] - lr * (mq / bc1) / (sqrtf(vq / bc2) + 1e-8f);
    master[q] = p;
    if (q < MLP_OFF_B1) wbf[q] = __float2bfloat16_rn(p);
    else if (q >= MLP_OFF_W2 && q < MLP_OFF_B2) wbf[q - MLP_H] = __float2bfloat16_rn(p);
    else if (q >= MLP_OFF_W3 && q < MLP_OFF_B3) wbf[q - 2 * MLP_H] = __float2bfloat16_rn(p);
}

// Sums of the block partials in block order, a thread per column, left in the first partial. (On the host, which
// had to copy every partial, this was most of a gradient: 375 us at 16,384 samples, 50 now.)
__global__ void __launch_bounds__(32) k_mlp_sum(float *gpart, int nblocks) {
    const int q = blockIdx.x * 32 + threadIdx.x;
    if (q > MLP_NPARAM) return;
    float *col = gpart + q;
    float s = 0.f;
#pragma unroll 16
    for (int b = 0; b < nblocks; ++b) s += col[(size_t)b * TG_ROW];
    *col = s;
}

__global__ void __launch_bounds__(TRAIN_THREADS)
k_mlp_forward(const float *master, const __nv_bfloat16 *wbf, const __nv_bfloat16 *feat, int n, float *p_out) {
    extern __shared__ float sm[];
    float *wf = sm;
    float *h = wf + MLP_NPARAM;
    load_weights_smem(wf, master, wbf);
    __syncthreads();
    const int s = blockIdx.x * TRAIN_THREADS + threadIdx.x;
    if (s >= n) return;
    float x[MLP_IN];
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) x[k] = __bfloat162float(feat[(size_t)s * MLP_IN + k]);
    unsigned m1, m2;
    const float z3 = mlp_forward_thread(wf, x, h + threadIdx.x * 2 * MLP_H, h + threadIdx.x * 2 * MLP_H + MLP_H, m1, m2);
    p_out[s] = 1.f / (1.f + expf(-z3));
}

}  // namespace fm

// ====================================== C ABI ======================================================
using namespace fm;

void fm_internal_set_error(const char *msg);

struct fm_mlp {
    float *master = nullptr, *m = nullptr, *v = nullptr, *gpart = nullptr, *loss = nullptr;
    __nv_bfloat16 *wbf = nullptr;
    long long step = 0;
};

namespace {
fm_status mlp_fail(fm_status s, const std::string &m) {
    fm_internal_set_error(m.c_str());
    return s;
}
#define MLP_CUDA(call)                                                                         \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess) return mlp_fail(FM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

constexpr int MLP_MAX_BATCH = 1 << 16;

// blocks of the gradient kernel: one per tile while they fit two per SM, then a walk over tiles
int train_blocks(int count) { return std::min((count + TG_T - 1) / TG_T, TG_BLOCKS); }
}  // namespace

// device pointers of a network, for fm_learned_weights (fm_api.cu)
void fm_internal_mlp_params(const fm_mlp *net, const float **master, const __nv_bfloat16 **wbf) {
    *master = net->master;
    *wbf = net->wbf;
}

extern "C" {

FM_API fm_status fm_mlp_create(const float *params, fm_mlp **out) {
    if (!out || !params) return mlp_fail(FM_EINVAL, "fm_mlp_create: params and out must not be NULL");
    *out = nullptr;
    for (int q = 0; q < MLP_NPARAM; ++q)
        if (!std::isfinite(params[q])) return mlp_fail(FM_EINVAL, "fm_mlp_create: parameters must be finite");
    fm_mlp *n = new fm_mlp();
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = cudaMalloc(&n->master, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(&n->m, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(&n->v, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(&n->gpart, sizeof(float) * TG_ROW * TG_BLOCKS);
    if (e == cudaSuccess) e = cudaMalloc(&n->loss, sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->wbf, sizeof(__nv_bfloat16) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMemcpy(n->master, params, sizeof(float) * MLP_NPARAM, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) {
        k_mlp_refresh<<<2, 1024>>>(n->master, n->wbf);
        e = cudaDeviceSynchronize();
    }
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(sizeof(float) * (MLP_NPARAM + TRAIN_THREADS * 2 * MLP_H)));
    if (e != cudaSuccess) {
        fm_mlp_destroy(n);
        return mlp_fail(e == cudaErrorMemoryAllocation ? FM_ENOMEM : FM_ECUDA,
                        std::string("fm_mlp_create: ") + cudaGetErrorString(e));
    }
    *out = n;
    return FM_OK;
}

FM_API void fm_mlp_destroy(fm_mlp *n) {
    if (!n) return;
    cudaDeviceSynchronize();
    cudaFree(n->master);
    cudaFree(n->m);
    cudaFree(n->v);
    cudaFree(n->gpart);
    cudaFree(n->loss);
    cudaFree(n->wbf);
    delete n;
}

FM_API fm_status fm_mlp_get_params(fm_mlp *n, float *params) {
    if (!n || !params) return mlp_fail(FM_EINVAL, "fm_mlp_get_params: NULL argument");
    MLP_CUDA(cudaMemcpy(params, n->master, sizeof(float) * MLP_NPARAM, cudaMemcpyDeviceToHost));
    return FM_OK;
}

FM_API fm_status fm_mlp_set_params(fm_mlp *n, const float *params) {
    if (!n || !params) return mlp_fail(FM_EINVAL, "fm_mlp_set_params: NULL argument");
    for (int q = 0; q < MLP_NPARAM; ++q)
        if (!std::isfinite(params[q])) return mlp_fail(FM_EINVAL, "fm_mlp_set_params: parameters must be finite");
    MLP_CUDA(cudaMemcpy(n->master, params, sizeof(float) * MLP_NPARAM, cudaMemcpyHostToDevice));
    k_mlp_refresh<<<2, 1024>>>(n->master, n->wbf);
    MLP_CUDA(cudaDeviceSynchronize());
    return FM_OK;
}

FM_API fm_status fm_mlp_train_step(fm_mlp *n, const void *d_features, const float *d_labels, int32_t count,
                                   float lr, float *loss, void *stream) {
    if (!n || !d_features || !d_labels) return mlp_fail(FM_EINVAL, "fm_mlp_train_step: NULL argument");
    if (count < 1 || count > MLP_MAX_BATCH) return mlp_fail(FM_EINVAL, "fm_mlp_train_step: count must be in [1, 65536]");
    if (!(lr >= 0.f) || !std::isfinite(lr)) return mlp_fail(FM_EINVAL, "fm_mlp_train_step: lr must be finite and >= 0");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int nb = train_blocks(count);
    const float inv_n = 1.f / (float)count;
    MLP_CUDA(launch_k(k_mlp_grad, dim3(nb), dim3(TRAIN_THREADS), s, true, (const float *)n->master,
                      (const __nv_bfloat16 *)n->wbf, static_cast<const __nv_bfloat16 *>(d_features), d_labels, (int)count,
                      inv_n, n->gpart));
    n->step += 1;
    const float bc1 = 1.f - powf(0.9f, (float)n->step), bc2 = 1.f - powf(0.999f, (float)n->step);
    MLP_CUDA(launch_k(k_mlp_adam, dim3(TG_ROW / 32), dim3(32 * ADAM_ROWS), s, true, n->master, n->wbf, n->m, n->v,
                      (const float *)n->gpart, nb, lr, bc1, bc2, inv_n, n->loss));
    MLP_CUDA(cudaGetLastError());
    if (loss) {
        MLP_CUDA(cudaMemcpyAsync(loss, n->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
        MLP_CUDA(cudaStreamSynchronize(s));
    }
    return FM_OK;
}

FM_API fm_status fm_mlp_gradient(fm_mlp *n, const void *d_features, const float *d_labels, int32_t count,
                                 float *grad, float *loss) {
    if (!n || !d_features || !d_labels || !grad) return mlp_fail(FM_EINVAL, "fm_mlp_gradient: NULL argument");
    if (count < 1 || count > MLP_MAX_BATCH) return mlp_fail(FM_EINVAL, "fm_mlp_gradient: count must be in [1, 65536]");
    const int nb = train_blocks(count);
    MLP_CUDA(launch_k(k_mlp_grad, dim3(nb), dim3(TRAIN_THREADS), cudaStream_t(nullptr), false, (const float *)n->master,
                      (const __nv_bfloat16 *)n->wbf, static_cast<const __nv_bfloat16 *>(d_features), d_labels, (int)count,
                      1.f / (float)count, n->gpart));
    k_mlp_sum<<<TG_ROW / 32, 32>>>(n->gpart, nb);
    MLP_CUDA(cudaGetLastError());
    float sums[MLP_NPARAM + 1];
    MLP_CUDA(cudaMemcpy(sums, n->gpart, sizeof sums, cudaMemcpyDeviceToHost));
    std::memcpy(grad, sums, sizeof(float) * MLP_NPARAM);
    if (loss) *loss = sums[MLP_NPARAM] / (float)count;
    return FM_OK;
}

FM_API fm_status fm_mlp_forward(fm_mlp *n, const void *d_features, int32_t count, float *d_p, void *stream) {
    if (!n || !d_features || !d_p) return mlp_fail(FM_EINVAL, "fm_mlp_forward: NULL argument");
    if (count < 1) return mlp_fail(FM_EINVAL, "fm_mlp_forward: count must be >= 1");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    k_mlp_forward<<<(count + TRAIN_THREADS - 1) / TRAIN_THREADS, TRAIN_THREADS,
                    sizeof(float) * (MLP_NPARAM + TRAIN_THREADS * 2 * MLP_H), s>>>(
        n->master, n->wbf, static_cast<const __nv_bfloat16 *>(d_features), count, d_p);
    MLP_CUDA(cudaGetLastError());
    return FM_OK;
}

FM_API int32_t fm_mlp_num_params(void) { return MLP_NPARAM; }

}  // extern "C"
