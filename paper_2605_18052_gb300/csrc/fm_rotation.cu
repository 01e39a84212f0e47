// Global rotation stage (Sec. "Global Rotation", Eq. fastmap-rotation-objective):
// world-to-camera rotations from relative rotations R_{i->j} of the image pairs.
//
// Initialisation (paragraph "Initialization details", column-wise least squares): column 1 of
// every rotation minimises sum_p ||x_j - R_p x_i||^2, column 2 the same (scaled by 1/|P|) plus
// (1/N) sum_k (x_k^T y_k)^2; camera 0's column is held at e1 / e2 (the gauge, R_0 = I), which
// leaves a symmetric positive definite system in the other cameras' columns:
//   A v = w_pair (deg_k v_k - sum_{p: k=j} R_p v_i - sum_{p: k=i} R_p^T v_j) + D_k v_k = b,
// solved by preconditioned conjugate gradients with the operator applied per camera from the
// CSR of the pair table (no matrix stored) and the 3x3 diagonal blocks as preconditioner, one
// persistent kernel per column (k_cg_solve).
// Columns are then normalised, column 2 orthogonalised to column 1, column 3 = 1 x 2.
//
// Refinement: L_R = (1/|P|) sum_p d(R_j, R_p R_i), d = geodesic distance, with each R_k given
// by the 6D representation (a1, a2): b1 = a1/|a1|, b2 = (a2 - (b1.a2) b1)/|.|, b3 = b1 x b2.
// An evaluation is two launches: k_rot_pair computes every pair's distance and its gradient with
// respect to R_i and R_j, and k_rot_cam gathers a camera's gradient and maps it through the 6D
// representation. Optimiser steps run in one persistent kernel (k_rot_steps) that needs no
// distances and no per-pair memory. All in FP64.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "fm_grid.cuh"
#include "fm_walk.cuh"

void fm_internal_set_error(const char *msg);

using namespace fm;

namespace {

constexpr int RT_THREADS = 256;
constexpr int RT_CAMS = 8;    // cameras (warps) per block of the per-camera kernels
constexpr double C_MAX = 1.0 - 1e-12;

struct DevRot {
    int n_cams, n_pairs;
    const int *cam_i, *cam_j, *cam_off, *cam_ent;
    const double *Rrel;      // n_pairs x 9 (row-major)
    double *a;               // n_cams x 6: the 6D parameters
    double *R;               // n_cams x 9: rotations of the current parameters
    float *m, *v;            // Adam moments, n_cams x 6
    double *pgrad;           // n_pairs x 18: d d_p / d R_i (9), d d_p / d R_j (9)
    double *pdist;           // n_pairs: d_p
    double *blk;             // per-block partial sums (loss, CG dot products): two rows of camera blocks
    double *loss;
    double *hyper;           // lr, beta1, beta2, eps
    long long *step;
    // conjugate gradients: vectors n_cams x 3 (p twice), the preconditioner (n_cams x 3), r.z of
    // every camera, and per column the first and last r.z and the iteration count
    double *x, *r, *z, *p, *p2, *q, *pre, *col1, *col2, *cam_rz, *scal;
    unsigned *grid_state;    // grid barriers of the persistent kernels
    unsigned *err;
};

__host__ __device__ inline int cam_blocks(int n) { return (n + RT_CAMS - 1) / RT_CAMS; }

// warp-wide sum of n doubles (fixed butterfly order)
template <int N>
__device__ __forceinline__ void warp_sum(double *v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
}

// GB300 issues one FP64 instruction of a warp every 64 cycles per SM sub-partition, whatever its
// active lanes and whatever else the warp has in flight (measured: one warp of 8 independent FMA
// chains takes as long as one chain eight times as long), so what the camera kernels count is FP64
// instructions per warp: values that belong to different cameras or components go to different lanes
// of one warp, and a division or square root (9 such instructions each) is shared where it can be.

// Warp-wide sums of N doubles that leave value i with lane spread_lane(N, i): at each butterfly
// level a lane keeps half of its values and hands the other half over, so N = 9 takes 12 additions
// instead of 45. The order of every sum is the butterfly's.
template <int N>
__device__ __forceinline__ double warp_sum_spread(double (&v)[N], int lane) {
    int cnt = N;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (cnt > 1) {
            const int h = (cnt + 1) / 2;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (i >= h) break;
                const double other = h + i < cnt ? v[h + i < N ? h + i : 0] : 0.0;
                const double keep = up ? other : v[i], give = up ? v[i] : other;
                v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
            cnt = h;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
    return v[0];
}

// a / b from y = 1/b rounded to nearest: the residual corrections of a y (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990) round the quotient to nearest,
// so several quotients by one divisor cost one division and 5 instructions each. For operands whose
// residuals do not underflow (|a| and |b| above about 1e-290) and finite y.
__device__ __forceinline__ double quotient(double a, double b, double y) {
    double q = __dmul_rn(a, y);
    q = __fma_rn(__fma_rn(-q, b, a), y, q);
    return __fma_rn(__fma_rn(-q, b, a), y, q);
}

// The three components of a camera's vector, from the lanes base .. base + 2 that hold one each.
struct Vec3 {
    double v[3];
    __device__ __forceinline__ Vec3(double mine, int base) {
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = __shfl_sync(0xffffffffu, mine, base + a);
    }
    __device__ __forceinline__ double operator[](int a) const { return v[a]; }
};
// a0 b0 + a1 b1 + a2 b2. The roundings of this and of the other sums of products of the solves are spelled out: which
// product of a sum the compiler contracts depends on the code around it, and the refinement behind the
// initialisation amplifies a last bit.
__device__ __forceinline__ double sum3(double a0, double b0, double a1, double b1, double a2, double b2) {
    return __fma_rn(a2, b2, __fma_rn(a0, b0, __dmul_rn(a1, b1)));
}
__device__ __forceinline__ double dot(const Vec3 &u, const Vec3 &v) { return sum3(u[0], v[0], u[1], v[1], u[2], v[2]); }
// component a of u x v
__device__ __forceinline__ double cross(const Vec3 &u, const Vec3 &v, int a) {
    const double p = a == 0 ? u[1] : (a == 1 ? u[2] : u[0]), q = a == 0 ? v[2] : (a == 1 ? v[0] : v[1]);
    const double r = a == 0 ? u[2] : (a == 1 ? u[0] : u[1]), w = a == 0 ? v[1] : (a == 1 ? v[2] : v[0]);
    return p * q - r * w;
}

__device__ __forceinline__ void cross3(const double *u, const double *v, double *o) {
    o[0] = u[1] * v[2] - u[2] * v[1];
    o[1] = u[2] * v[0] - u[0] * v[2];
    o[2] = u[0] * v[1] - u[1] * v[0];
}

// ---- conjugate gradients on the anchored column system ----------------------------------------
// Sums over the grid that reproduce a 256-thread tree (thread t adds the values t, t + 256, ..., then
// halves from 128 down) with a warp, lane l standing for the threads l, l + 32, ..., l + 224. Levels
// that would only add zeros are left out. Every lane gets the total.
__device__ __forceinline__ double tree_256(const double (&v)[8], int n) {
    double s;
    if (n > 128) s = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
    else if (n > 64) s = (v[0] + v[2]) + (v[1] + v[3]);
    else if (n > 32) s = v[0] + v[1];
    else s = v[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (n > o) s += __shfl_xor_sync(0xffffffffu, s, o);
    return n > 16 ? s : __shfl_sync(0xffffffffu, s, 0);
}
// of n values in memory
__device__ __forceinline__ double sum_values(const double *val, int n, int lane) {
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        int b = lane + 32 * j;
        v[j] = b < n ? __ldcg(val + b) : 0.0;
        for (b += 256; b < n; b += 256) v[j] += __ldcg(val + b);
    }
    return tree_256(v, n);
}

// One anchored column system, solved and finished in one cooperative launch: camera 0's column is
// e_axis, the data term is weighted w_pair and the orthogonality penalty along t.col1 w_pen. Warp w
// of a block owns camera 8 block + w (then 8 (block + grid) + w, ... when the cameras exceed the
// resident warps). An iteration is two phases with a grid-wide sum behind each:
//   p = z + beta p (own camera, and recomputed for the neighbours, so no third phase), q = A p; p.q
//   x += alpha p, r -= alpha q, z = M^-1 r with M the 3x3 diagonal blocks;               r.z
// The first phase runs a warp per camera, with the relative rotations in registers from iteration
// to iteration; what is left per camera runs in one warp, a lane per component of each of the group's
// cameras. It stops at a multiple of CG_CHUNK iterations, as soon as the preconditioned residual norm has fallen by tol.
// Then the column is normalised; column 2 (axis 1) is orthogonalised to column 1 first and the
// rotations [c1 c2 c1 x c2], their parameters and a fresh Adam state are written, unless a column
// vanished. (As five launches an iteration this took 22 us an iteration on 1,000 cameras; 9 us now,
// of which the two barriers take 2.5 us and the serial FP64 instructions of the phases most of the rest.)
constexpr int CG_CHUNK = 32;

// SINGLE: a group of 8 cameras a block, whose state stays in registers; otherwise (more than 2,432 cameras) the
// state goes through memory and a block's warps take the per-camera work of its groups in turn. AHEAD: a
// warp's next pairs are on their way while 32 are used: always without SINGLE, and with it where a camera has
// more than 256 pairs (below, its registers cost what it gives). us a solve of both columns, one warp for all
// groups and no reading ahead -> now: 3,000 cameras, 24 pairs each 24.9 -> 23.8 ms, 20,000 with 60 183 -> 169, with 120
// 202 -> 176, 1,000 cameras, all pairs, 4.1 -> 3.4; 1,000 cameras with 24 4.4 -> 4.3 (z and p by plain loads,
// behind the barrier's acquire, instead of from L2).
template <bool SINGLE, bool AHEAD>
__global__ void __launch_bounds__(RT_CAMS * 32, 2)
k_cg_solve(DevRot t, int axis, double w_pair, double w_pen, int max_iters, double tol) {
    __shared__ double s_sum[2][RT_CAMS][3], s_rz[256], s_out, s_alpha;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int stride = gridDim.x * RT_CAMS, k0 = blockIdx.x * RT_CAMS;
    const int groups = cam_blocks(t.n_cams), trees = (t.n_cams + 255) / 256;
    if (axis == 1 && (*t.err & ERR_DEGENERATE)) return;   // column 1 vanished: leave the state as it is
    GridBarrier gb(t.grid_state, t.err);
    // The groups' sums lie in two rows of t.blk: r.z of the setup in one, p.q of the iterations in the other.
    // The setup has one barrier: a block may reach the first p.q while another still reads the setup's r.z.
    double *slot = t.blk, *slot_setup = t.blk + groups, *cam_rz = t.cam_rz;
    // warp 0: lane 3 c + a holds component a of the block's camera c
    const int cc = lane / 3, ca = lane % 3, base = 3 * cc;
    // (its state stays in registers when the block owns one group; it goes through memory otherwise)
    double xk = 0.0, rk = 0.0, zk = 0.0, pk = 0.0, qk = 0.0, ck = 0.0, al = 1.0, y = 1.0, f = 0.0, deg = 0.0;
    double M[9];          // the lane's first entry: R_p for the second camera of a pair, else R_p^T
    int other = 0;
    bool have = false;
    auto load_entry = [&](int e) {
        const int ent = t.cam_ent[e];
        const int n = ent >> 1, role = ent & 1;
        other = role ? t.cam_i[n] : t.cam_j[n];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) M[3 * a + b] = t.Rrel[(size_t)n * 9 + (role ? 3 * a + b : 3 * b + a)];
    };
    auto mat_v = [&](const double *v, double *o) {
#pragma unroll
        for (int a = 0; a < 3; ++a) o[a] = sum3(M[3 * a], v[0], M[3 * a + 1], v[1], M[3 * a + 2], v[2]);
    };
    // a warp's sums over the pairs of its camera to s_sum[half][warp]
    auto put_sums = [&](double (&s)[3], int half) {
        const double mine = warp_sum_spread<3>(s, lane);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (lane == spread_lane(3, a)) s_sum[half][warp][a] = mine;
    };
    // warp 0: a value per camera (in its first lane) summed over the group in camera order
    auto group_sum = [&](double mine) {
        double b = __shfl_sync(0xffffffffu, mine, 0);
#pragma unroll
        for (int w = 1; w < RT_CAMS; ++w) b += __shfl_sync(0xffffffffu, mine, 3 * w);
        return b;
    };
    // setup: x = 0 except the anchor, r = b - A x = the anchor's contribution, z = M^-1 r, p = 0
    for (int kb = k0; kb < t.n_cams; kb += stride) {
        const int k = kb + warp;
        if (k < t.n_cams) {
            const int e_begin = t.cam_off[k], e_end = t.cam_off[k + 1];
            double s[3] = {0.0, 0.0, 0.0}, ax[3], o[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) ax[a] = a == axis ? 1.0 : 0.0;
            for (int e = e_begin + lane; e < e_end; e += 32) {
                load_entry(e);
                if (k == 0 || other != 0) continue;
                mat_v(ax, o);
#pragma unroll
                for (int a = 0; a < 3; ++a) s[a] += o[a];
            }
            have = SINGLE && e_end - e_begin <= 32;
            put_sums(s, 0);
        }
        __syncthreads();
        if (warp == 0) {
            const int kc = kb + cc;
            const bool on = cc < RT_CAMS && kc < t.n_cams;
            deg = on ? (double)(t.cam_off[kc + 1] - t.cam_off[kc]) : 1.0;
            ck = on ? t.col1[(size_t)kc * 3 + ca] : 0.0;
            rk = on ? w_pair * s_sum[0][cc][ca] : 0.0;
            // M = w_pair deg I + w_pen c c^T: M^-1 = (I - beta/(alpha + beta |c|^2) c c^T) / alpha
            const Vec3 cv(ck, base), rv(rk, base);
            al = w_pair * deg;
            f = w_pen / __fma_rn(w_pen, dot(cv, cv), al);
            y = 1.0 / al;
            const double cr = dot(cv, rv);
            zk = quotient(__fma_rn(-__dmul_rn(f, ck), cr, rk), al, y);
            const Vec3 zv(zk, base);
            const double rz = on && kc != 0 ? dot(rv, zv) : 0.0;
            xk = kc == 0 && ca == axis ? 1.0 : 0.0;
            pk = 0.0;
            if (on) {
                const size_t o3 = (size_t)kc * 3 + ca;
                t.pre[o3] = ca == 0 ? al : (ca == 1 ? y : f);
                t.x[o3] = xk;
                t.r[o3] = rk;
                t.z[o3] = zk;
                t.p[o3] = 0.0;
                t.p2[o3] = 0.0;
                if (kc == 0 && ca == 0) cam_rz[0] = 0.0;
            }
            const double b = group_sum(rz);
            if (lane == 0) slot_setup[kb / RT_CAMS] = b;
        }
        if (!SINGLE) __syncthreads();
    }
    bool ok = true;
    if (warp == 0) {
        gb.arrive();
        ok = gb.wait();
        const double v = sum_values(slot_setup, groups, lane);
        if (lane == 0) s_out = v;
    }
    if (!__syncthreads_and(ok)) return;
    const double rz0 = s_out;
    double rz = rz0, beta = 0.0;
    int it = 0;
    while (it < max_iters && rz > tol * tol * rz0 && rz > 0.0) {
        for (int c = 0; c < CG_CHUNK; ++c) {
            const double *p_old = (c & 1) ? t.p2 : t.p;
            double *p_new = (c & 1) ? t.p : t.p2;
            int turn = 0;   // the block's groups one after the other
            for (int kb = k0; kb < t.n_cams; kb += stride, ++turn) {
                const int k = kb + warp, half = SINGLE ? 0 : turn & 1;
                if (k > 0 && k < t.n_cams) {
                    const int e_begin = t.cam_off[k], e_end = t.cam_off[k + 1];
                    double s[3] = {0.0, 0.0, 0.0}, o[3];
                    if (!AHEAD || have) {
                        for (int e = e_begin + lane; e < e_end; e += 32) {
                            if (!have) load_entry(e);
                            if (other == 0) continue;
                            double vo[3];
#pragma unroll
                            for (int a = 0; a < 3; ++a)
                                vo[a] = __fma_rn(beta, p_old[(size_t)other * 3 + a], t.z[(size_t)other * 3 + a]);
                            mat_v(vo, o);
                            if (have) {   // the warp's only chunk
#pragma unroll
                                for (int a = 0; a < 3; ++a) s[a] = o[a];
                            } else {
#pragma unroll
                                for (int a = 0; a < 3; ++a) s[a] += o[a];
                            }
                        }
                    } else {
                        if (e_begin + lane < e_end) load_entry(e_begin + lane);
                        for (int e = e_begin + lane; e < e_end; e += 32) {
                            double A[9], vo[3];
                            const int cam = other;
#pragma unroll
                            for (int q = 0; q < 9; ++q) A[q] = M[q];
                            if (e + 32 < e_end) load_entry(e + 32);
                            if (cam == 0) continue;
#pragma unroll
                            for (int a = 0; a < 3; ++a)
                                vo[a] = __fma_rn(beta, p_old[(size_t)cam * 3 + a], t.z[(size_t)cam * 3 + a]);
#pragma unroll
                            for (int a = 0; a < 3; ++a) o[a] = sum3(A[3 * a], vo[0], A[3 * a + 1], vo[1], A[3 * a + 2], vo[2]);
#pragma unroll
                            for (int a = 0; a < 3; ++a) s[a] += o[a];
                        }
                    }
                    put_sums(s, half);
                }
                __syncthreads();
                // the block's groups in turn by its warps, each while the others go on to the next group
                // (whose sums take the other half: this half is written again two barriers on)
                if (warp == (SINGLE ? 0 : turn % RT_CAMS)) {
                    const int kc = kb + cc;
                    const bool on = cc < RT_CAMS && kc > 0 && kc < t.n_cams;
                    const size_t o3 = (size_t)(on ? kc : 0) * 3 + ca;
                    if (!SINGLE) {
                        deg = on ? (double)(t.cam_off[kc + 1] - t.cam_off[kc]) : 0.0;
                        ck = on ? t.col1[o3] : 0.0;
                        zk = on ? __ldcg(t.z + o3) : 0.0;
                        pk = on ? __ldcg(p_old + o3) : 0.0;
                    }
                    pk = __fma_rn(beta, pk, zk);
                    const double sk = on ? s_sum[half][cc][ca] : 0.0;
                    const Vec3 pv(pk, base);
                    const double cp = dot(Vec3(ck, base), pv);
                    // w_pair (deg p - s) + w_pen c (c.p)
                    qk = __fma_rn(w_pair, __fma_rn(deg, pk, -sk), __dmul_rn(__dmul_rn(w_pen, ck), cp));
                    const double pq = dot(Vec3(qk, base), pv);
                    if (on) {
                        p_new[o3] = pk;
                        if (!SINGLE) t.q[o3] = qk;
                    }
                    const double b = group_sum(on ? pq : 0.0);
                    if (lane == 0) slot[kb / RT_CAMS] = b;
                }
            }
            if (!SINGLE) __syncthreads();   // every warp's groups are written
            double y_rz = 0.0;   // for the quotient behind the second sum, while warp 0 is at the first
            if (warp != 0) y_rz = 1.0 / rz;
            double alpha = 0.0;
            if (warp == 0) {
                gb.arrive();
                ok = gb.wait();
                const double pq = sum_values(slot, groups, lane);
                // (the shuffle keeps the division out of the divergent code below)
                alpha = __shfl_sync(0xffffffffu, pq > 0.0 ? rz / pq : 0.0, 0);
                if (!SINGLE && lane == 0) s_alpha = alpha;
            }
            if (!SINGLE) {
                __syncthreads();
                alpha = s_alpha;
            }
            turn = 0;
            for (int kb = k0; kb < t.n_cams; kb += stride, ++turn) {
                if (warp != (SINGLE ? 0 : turn % RT_CAMS)) continue;
                const int kc = kb + cc;
                const bool on = cc < RT_CAMS && kc > 0 && kc < t.n_cams;
                const size_t o3 = (size_t)(on ? kc : 0) * 3;
                if (!SINGLE) {
                    al = on ? t.pre[o3] : 1.0;
                    y = on ? t.pre[o3 + 1] : 1.0;
                    f = on ? t.pre[o3 + 2] : 0.0;
                    ck = on ? t.col1[o3 + ca] : 0.0;
                    xk = on ? t.x[o3 + ca] : 0.0;
                    rk = on ? t.r[o3 + ca] : 0.0;
                    pk = on ? p_new[o3 + ca] : 0.0;
                    qk = on ? t.q[o3 + ca] : 0.0;
                }
                xk = __fma_rn(alpha, pk, xk);
                rk = __fma_rn(-alpha, qk, rk);
                const Vec3 rv(rk, base);
                const double cr = dot(Vec3(ck, base), rv);
                zk = quotient(__fma_rn(-__dmul_rn(f, ck), cr, rk), al, y);
                const double rzk = dot(rv, Vec3(zk, base));
                if (on) {
                    t.z[o3 + ca] = zk;
                    if (ca == 0) cam_rz[kc] = rzk;
                    if (!SINGLE) {
                        t.x[o3 + ca] = xk;
                        t.r[o3 + ca] = rk;
                    }
                }
            }
            if (!SINGLE) __syncthreads();
            if (warp == 0) {
                gb.arrive();
                ok = gb.wait() && ok;
            }
            if (!__syncthreads_and(ok)) return;
            // r.z: a tree for every 256 cameras (a warp each), then one over their totals (every warp)
            if (warp == 1 && lane == 0) s_out = y_rz;
            for (int g = warp; g < trees; g += RT_CAMS) {
                const int n = min(256, t.n_cams - 256 * g);
                const double v = sum_values(cam_rz + 256 * g, n, lane);
                if (lane == 0) {
                    if (g < 256) s_rz[g] = v;
                    else s_rz[g & 255] += v;     // g and g + 256 belong to one warp
                }
            }
            __syncthreads();
            double v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = lane + 32 * j < trees ? s_rz[lane + 32 * j] : 0.0;
            const double rzn = tree_256(v, min(trees, 256));
            // (far past convergence the sums leave the range in which 1/rz and the residuals are exact)
            if (rz > 1e-280 && rzn > 1e-280) beta = quotient(rzn, rz, s_out);
            else beta = rz > 0.0 ? rzn / rz : 0.0;
            rz = rzn;
        }
        it += CG_CHUNK;
    }
    gb.finish();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        t.scal[4 * axis] = rz0;
        t.scal[4 * axis + 1] = rz;
        t.scal[4 * axis + 2] = (double)it;
    }
    if (warp != 0) return;
    if (SINGLE && cc < RT_CAMS && k0 + cc > 0 && k0 + cc < t.n_cams) t.x[(size_t)(k0 + cc) * 3 + ca] = xk;
    __syncwarp();
    if (lane >= RT_CAMS) return;
    for (int k = k0 + lane; k < t.n_cams; k += stride) {
        double v[3] = {t.x[(size_t)k * 3], t.x[(size_t)k * 3 + 1], t.x[(size_t)k * 3 + 2]};
        const double *c1 = t.col1 + (size_t)k * 3;
        double n = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        if (!(n > 0.0) || !isfinite(n)) {
            atomicOr(t.err, ERR_DEGENERATE);
            n = 1.0;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] /= n;
        if (axis == 1) {
            const double d = c1[0] * v[0] + c1[1] * v[1] + c1[2] * v[2];
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] -= d * c1[a];
            n = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
            if (!(n > 0.0) || !isfinite(n)) {
                atomicOr(t.err, ERR_DEGENERATE);
                n = 1.0;
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] /= n;
        }
        double *col = axis == 1 ? t.col2 : t.col1;
#pragma unroll
        for (int a = 0; a < 3; ++a) col[(size_t)k * 3 + a] = v[a];
        if (axis == 1) {
            double z[3];
            cross3(c1, v, z);
            double *R = t.R + (size_t)k * 9;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                R[3 * r] = c1[r];
                R[3 * r + 1] = v[r];
                R[3 * r + 2] = z[r];
                t.a[(size_t)k * 6 + r] = c1[r];
                t.a[(size_t)k * 6 + 3 + r] = v[r];
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) t.m[(size_t)k * 6 + q] = t.v[(size_t)k * 6 + q] = 0.f;
        }
    }
    if (axis == 1 && blockIdx.x == 0 && threadIdx.x == 0) *t.step = 0;
}

// ---- 6D representation and the geodesic objective ----------------------------------------------
// (quotients by a norm share its reciprocal: the FP64 divisions of the two maps were most of a
// camera's step)
// R (row-major) with columns b1, b2, b3 from a = (a1, a2)
__device__ void rot_from_6d(const double *a, double *R) {
    double b1[3], u[3], b2[3], b3[3];
    const double n1 = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]), y1 = 1.0 / n1;
#pragma unroll
    for (int q = 0; q < 3; ++q) b1[q] = quotient(a[q], n1, y1);
    const double d = b1[0] * a[3] + b1[1] * a[4] + b1[2] * a[5];
#pragma unroll
    for (int q = 0; q < 3; ++q) u[q] = a[3 + q] - d * b1[q];
    const double nu = sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), yu = 1.0 / nu;
#pragma unroll
    for (int q = 0; q < 3; ++q) b2[q] = quotient(u[q], nu, yu);
    cross3(b1, b2, b3);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        R[3 * r] = b1[r];
        R[3 * r + 1] = b2[r];
        R[3 * r + 2] = b3[r];
    }
}

// gradient with respect to a of a scalar whose gradient with respect to R is gR (row-major)
__device__ void rot_6d_backward(const double *a, const double *gR, double *ga) {
    double b1[3], u[3], b2[3], g1[3], g2[3], g3[3], gb1[3], gb2[3], gu[3], t1[3], t2[3];
    const double n1 = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]), y1 = 1.0 / n1;
#pragma unroll
    for (int q = 0; q < 3; ++q) b1[q] = quotient(a[q], n1, y1);
    const double d = b1[0] * a[3] + b1[1] * a[4] + b1[2] * a[5];
#pragma unroll
    for (int q = 0; q < 3; ++q) u[q] = a[3 + q] - d * b1[q];
    const double nu = sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), yu = 1.0 / nu;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        b2[q] = quotient(u[q], nu, yu);
        g1[q] = gR[3 * q];
        g2[q] = gR[3 * q + 1];
        g3[q] = gR[3 * q + 2];
    }
    cross3(b2, g3, t1);      // b3 = b1 x b2: gradient b2 x g3 on b1, g3 x b1 on b2
    cross3(g3, b1, t2);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        gb1[q] = g1[q] + t1[q];
        gb2[q] = g2[q] + t2[q];
    }
    const double b2g = b2[0] * gb2[0] + b2[1] * gb2[1] + b2[2] * gb2[2];
#pragma unroll
    for (int q = 0; q < 3; ++q) gu[q] = quotient(gb2[q] - b2[q] * b2g, nu, yu);
    const double b1gu = b1[0] * gu[0] + b1[1] * gu[1] + b1[2] * gu[2];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        ga[3 + q] = gu[q] - b1[q] * b1gu;
        gb1[q] = gb1[q] - gu[q] * d - a[3 + q] * b1gu;
    }
    const double b1g = b1[0] * gb1[0] + b1[1] * gb1[1] + b1[2] * gb1[2];
#pragma unroll
    for (int q = 0; q < 3; ++q) ga[q] = quotient(gb1[q] - b1[q] * b1g, n1, y1);
}

__global__ void k_rot_from_params(DevRot t) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= t.n_cams) return;
    double R[9];
    rot_from_6d(t.a + (size_t)k * 6, R);
#pragma unroll
    for (int q = 0; q < 9; ++q) t.R[(size_t)k * 9 + q] = R[q];
}

// per pair: X = R_p R_i, Y = R_p^T R_j, c = (tr(R_j^T X) - 1)/2, d = arccos(c);
// d d/d R_j = s X, d d/d R_i = s Y with s = -1/(2 sqrt(1 - c^2)) (c clamped below 1); returns s
__device__ __forceinline__ double pair_gradient(const double *Rp, const double *Ri, const double *Rj, double *X, double *Y,
                                                double *dist) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            X[3 * a + b] = Rp[3 * a] * Ri[b] + Rp[3 * a + 1] * Ri[3 + b] + Rp[3 * a + 2] * Ri[6 + b];
            Y[3 * a + b] = Rp[a] * Rj[b] + Rp[3 + a] * Rj[3 + b] + Rp[6 + a] * Rj[6 + b];
        }
    double tr = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) tr += Rj[q] * X[q];
    const double c = 0.5 * (tr - 1.0);
    const double cc = fmin(fmax(c, -1.0), C_MAX);
    if (dist) *dist = acos(fmin(fmax(c, -1.0), 1.0));
    return -0.5 / sqrt(1.0 - cc * cc);
}

__global__ void __launch_bounds__(RT_THREADS) k_rot_pair(DevRot t) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = n < t.n_pairs ? t.cam_i[n] : 0, j = n < t.n_pairs ? t.cam_j[n] : 0;
    pdl_wait();     // rotations of the previous step
    pdl_trigger();
    if (n >= t.n_pairs) return;
    double X[9], Y[9];
    const double s = pair_gradient(t.Rrel + (size_t)n * 9, t.R + (size_t)i * 9, t.R + (size_t)j * 9, X, Y, t.pdist + n);
    double *g = t.pgrad + (size_t)n * 18;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        g[q] = s * Y[q];
        g[9 + q] = s * X[q];
    }
}

// warp per camera: gather d L/d R_k from its pairs (scaled 1/|P|); then lanes 0..RT_CAMS-1 of
// warp 0 map the block's cameras through the 6D representation, one camera per lane: GB300's FP64
// pipe charges a whole warp instruction per operation, so the FP64 tail runs once per block
// instead of once per camera. Block partials of the loss.
__global__ void __launch_bounds__(RT_CAMS * 32) k_rot_cam(DevRot t, double *grad_out) {
    __shared__ double s_g[RT_CAMS][10];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * RT_CAMS + warp;
    pdl_wait();     // pair gradients of this evaluation
    pdl_trigger();
    {
        double g[10];
#pragma unroll
        for (int q = 0; q < 10; ++q) g[q] = 0.0;
        if (k < t.n_cams) {
            for (int e = t.cam_off[k] + lane; e < t.cam_off[k + 1]; e += 32) {
                const int ent = t.cam_ent[e];
                const int n = ent >> 1, role = ent & 1;
                const double *pg = t.pgrad + (size_t)n * 18 + (role ? 9 : 0);
#pragma unroll
                for (int q = 0; q < 9; ++q) g[q] += pg[q];
                if (role == 0) g[9] += t.pdist[n];     // each pair's distance counted once
            }
            warp_sum<10>(g);
        }
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < 10; ++q) s_g[warp][q] = g[q];
        }
    }
    __syncthreads();
    if (warp != 0 || lane >= RT_CAMS) return;
    const int kc = blockIdx.x * RT_CAMS + lane;
    if (kc < t.n_cams) {
        const double inv_b = 1.0 / (double)t.n_pairs;
        double g[9], ga[6];
#pragma unroll
        for (int q = 0; q < 9; ++q) g[q] = s_g[lane][q] * inv_b;
        rot_6d_backward(t.a + (size_t)kc * 6, g, ga);
#pragma unroll
        for (int q = 0; q < 6; ++q) grad_out[(size_t)kc * 6 + q] = ga[q];
    }
    if (lane == 0) {   // loss partial of the block, cameras in order
        double b = 0.0;
        for (int w = 0; w < RT_CAMS; ++w) b += s_g[w][9];
        t.blk[blockIdx.x] = b;
    }
}

// loss of an evaluation (one block, fixed order)
__global__ void __launch_bounds__(RT_THREADS) k_rot_finish(DevRot t) {
    __shared__ double red[RT_THREADS];
    pdl_wait();
    pdl_trigger();
    const int nb = cam_blocks(t.n_cams);
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += RT_THREADS) s += t.blk[b];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = RT_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *t.loss = red[0] / (double)t.n_pairs;
}

// iters Adam steps in one cooperative launch, two grid barriers per step. Phase 1: a thread per
// image pair (the pairs spread evenly over the blocks; relative rotations stay in registers from
// step to step) computes the pair's gradient with respect to R_i and R_j as k_rot_pair does,
// without the distance, which only the loss needs. Phase 2: warp w of a block gathers the gradient of
// camera 8 block + w (+ 8 grid, ...), then warp 0, a lane per component of each of the block's
// cameras, goes through the 6D backward pass, Adam and the new rotation. The norms and unit columns
// of the new rotation are those of the next step's backward pass and stay in registers. What bounds it
// is the serial chain of FP64 instructions: about 107 in phase 1, 42 and 90 in phase 2. 13 us a step
// on 1,000 cameras and 11,700 pairs, 33 us as three launches of 46, 125 and 4 blocks.
struct SixD {             // lane 3 c + a: component a of camera c's two unit columns, and the norms
    double b1, b2, d, n1, y1, nu, yu;
    __device__ __forceinline__ void from_params(double a1, double a2, int base) {
        const Vec3 a1v(a1, base);
        n1 = sqrt(dot(a1v, a1v));
        y1 = 1.0 / n1;
        b1 = quotient(a1, n1, y1);
        d = dot(Vec3(b1, base), Vec3(a2, base));
        const double u = a2 - d * b1;
        const Vec3 uv(u, base);
        nu = sqrt(dot(uv, uv));
        yu = 1.0 / nu;
        b2 = quotient(u, nu, yu);
    }
};

__global__ void __launch_bounds__(RT_CAMS * 32, 1) k_rot_steps(DevRot t, int iters) {
    __shared__ double s_g[RT_CAMS][9];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int stride = gridDim.x * RT_CAMS, k0 = blockIdx.x * RT_CAMS;
    const bool single = t.n_cams <= stride;
    const int per = (t.n_pairs + gridDim.x - 1) / gridDim.x;
    const int n_end = min(t.n_pairs, ((int)blockIdx.x + 1) * per);
    const int cc = lane / 3, ca = lane % 3, base = 3 * cc;
    GridBarrier gb(t.grid_state, t.err);
    const long long t0 = *t.step;
    const double inv_b = 1.0 / (double)t.n_pairs;
    const float lr = (float)t.hyper[0], b1 = (float)t.hyper[1], b2 = (float)t.hyper[2], eps = (float)t.hyper[3];
    double Rp[9];         // the thread's first pair
    int ci = 0, cj = 0;
    // the lane's first entry of the warp's camera, and the state of warp 0's cameras, stay in registers
    // when the block owns one group of cameras
    const int k_own = k0 + warp;
    int e_begin = 0, e_end = 0, first = -1;
    if (single && k_own < t.n_cams) {
        e_begin = t.cam_off[k_own];
        e_end = t.cam_off[k_own + 1];
        if (e_begin + lane < e_end) first = t.cam_ent[e_begin + lane];
    }
    SixD six;
    double a12[2] = {1.0, 1.0};
    float mv[4] = {0.f, 0.f, 0.f, 0.f};
    for (int it = 0; it < iters; ++it) {
        for (int n = blockIdx.x * per + threadIdx.x; n < n_end; n += RT_CAMS * 32) {
            if (it == 0 || per > RT_CAMS * 32) {
                ci = t.cam_i[n];
                cj = t.cam_j[n];
#pragma unroll
                for (int q = 0; q < 9; ++q) Rp[q] = t.Rrel[(size_t)n * 9 + q];
            }
            double Ri[9], Rj[9], X[9], Y[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                Ri[q] = __ldcg(t.R + (size_t)ci * 9 + q);
                Rj[q] = __ldcg(t.R + (size_t)cj * 9 + q);
            }
            const double s = pair_gradient(Rp, Ri, Rj, X, Y, nullptr);
            double *g = t.pgrad + (size_t)n * 18;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                g[q] = s * Y[q];
                g[9 + q] = s * X[q];
            }
        }
        if (!gb.sync()) return;
        for (int kb = k0; kb < t.n_cams; kb += stride) {
            const int k = kb + warp;
            if (k < t.n_cams) {
                double g[9];
#pragma unroll
                for (int q = 0; q < 9; ++q) g[q] = 0.0;
                if (!single) {
                    e_begin = t.cam_off[k];
                    e_end = t.cam_off[k + 1];
                    first = e_begin + lane < e_end ? t.cam_ent[e_begin + lane] : -1;
                }
                if (first >= 0) {
                    const double *pg = t.pgrad + (size_t)(first >> 1) * 18 + ((first & 1) ? 9 : 0);
#pragma unroll
                    for (int q = 0; q < 9; ++q) g[q] = __ldcg(pg + q);
                }
                for (int e = e_begin + 32 + lane; e < e_end; e += 32) {
                    const int ent = t.cam_ent[e];
                    const double *pg = t.pgrad + (size_t)(ent >> 1) * 18 + ((ent & 1) ? 9 : 0);
#pragma unroll
                    for (int q = 0; q < 9; ++q) g[q] += __ldcg(pg + q);
                }
                const double mine = warp_sum_spread<9>(g, lane);
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    if (lane == spread_lane(9, q)) s_g[warp][q] = mine;
            }
            __syncthreads();
            if (warp == 0) {
                const int kc = kb + cc;
                const bool on = cc < RT_CAMS && kc < t.n_cams;
                const size_t o = (size_t)(on ? kc : 0) * 6 + ca;
                if (!single || it == 0) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        a12[h] = t.a[o + 3 * h];
                        mv[h] = t.m[o + 3 * h];
                        mv[2 + h] = t.v[o + 3 * h];
                    }
                    six.from_params(a12[0], a12[1], base);
                }
                const double *gr = s_g[on ? cc : 0] + 3 * ca;
                const double g1 = gr[0] * inv_b, g2 = gr[1] * inv_b, g3 = gr[2] * inv_b;
                const Vec3 b1v(six.b1, base), b2v(six.b2, base), g3v(g3, base);
                double gb1 = g1 + cross(b2v, g3v, ca);
                const double gb2 = g2 + cross(g3v, b1v, ca);
                const double b2g = dot(b2v, Vec3(gb2, base));
                const double gu = quotient(gb2 - six.b2 * b2g, six.nu, six.yu);
                const double b1gu = dot(b1v, Vec3(gu, base));
                double ga[2];
                ga[1] = gu - six.b1 * b1gu;
                gb1 = gb1 - gu * six.d - a12[1] * b1gu;
                const double b1g = dot(b1v, Vec3(gb1, base));
                ga[0] = quotient(gb1 - six.b1 * b1g, six.n1, six.y1);
                const float ts = (float)(t0 + 1 + it);
                const float bc1 = 1.f - powf(b1, ts), bc2 = 1.f - powf(b2, ts);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float gq = (float)ga[h];
                    mv[h] = rfma(radd(1.f, -b1), gq, rmul(b1, mv[h]));
                    mv[2 + h] = rfma(rmul(radd(1.f, -b2), gq), gq, rmul(b2, mv[2 + h]));
                    a12[h] -= (double)(lr * (mv[h] / bc1) / (sqrtf(mv[2 + h] / bc2) + eps));
                    if (on && (!single || it + 1 == iters)) {
                        t.m[o + 3 * h] = mv[h];
                        t.v[o + 3 * h] = mv[2 + h];
                        t.a[o + 3 * h] = a12[h];
                    }
                }
                six.from_params(a12[0], a12[1], base);
                const double b3 = cross(Vec3(six.b1, base), Vec3(six.b2, base), ca);
                if (on) {
                    double *R = t.R + (size_t)kc * 9 + 3 * ca;
                    R[0] = six.b1;
                    R[1] = six.b2;
                    R[2] = b3;
                }
            }
            if (!single) __syncthreads();   // s_g is written again
        }
        if (!gb.sync()) return;
    }
    gb.finish();
    if (blockIdx.x == 0 && threadIdx.x == 0) *t.step = t0 + iters;
}

// 6D parameters from rotations (columns 1 and 2)
__global__ void k_params_from_rot(DevRot t) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= t.n_cams) return;
    const double *R = t.R + (size_t)k * 9;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        t.a[(size_t)k * 6 + q] = R[3 * q];
        t.a[(size_t)k * 6 + 3 + q] = R[3 * q + 1];
    }
}

}  // namespace

struct fm_rotation {
    DevRot d{};
    fm_rotation_options opt{};
    cudaStream_t user = nullptr;
    cudaStream_t s = nullptr;
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    double *grad6 = nullptr;
    int step_grid = 0, cg_grid = 0;       // blocks of the persistent kernels
    void (*cg_solve)(DevRot, int, double, double, int, double) = nullptr;   // the instantiation for the graph
    std::vector<void *> allocs;
    int cg_iters_last = 0;
    double cg_resid_last = 0.0;
};

namespace {

fm_status rfail(fm_status s, const std::string &msg) {
    fm_internal_set_error(msg.c_str());
    return s;
}

#define RT_CUDA(call)                                                                         \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return rfail(e_ == cudaErrorMemoryAllocation ? FM_ENOMEM : FM_ECUDA,              \
                         std::string(#call) + ": " + cudaGetErrorString(e_));                 \
    } while (0)

template <class T>
cudaError_t ralloc(fm_rotation *p, T **ptr, size_t count) {
    cudaError_t e = cudaMalloc(reinterpret_cast<void **>(ptr), sizeof(T) * (count ? count : 1));
    if (e == cudaSuccess) p->allocs.push_back(*ptr);
    return e;
}

cudaError_t rjoin_in(fm_rotation *p) {
    cudaError_t e = cudaEventRecord(p->ev_in, p->user);
    if (e != cudaSuccess) return e;
    return cudaStreamWaitEvent(p->s, p->ev_in, 0);
}

cudaError_t rjoin_out(fm_rotation *p) {
    cudaError_t e = cudaEventRecord(p->ev_out, p->s);
    if (e != cudaSuccess) return e;
    return cudaStreamWaitEvent(p->user, p->ev_out, 0);
}

fm_status rcheck_errors(fm_rotation *p) {
    unsigned err = 0;
    RT_CUDA(cudaMemcpyAsync(&err, p->d.err, sizeof err, cudaMemcpyDeviceToHost, p->s));
    RT_CUDA(cudaStreamSynchronize(p->s));
    if (err & ERR_GRID) {
        RT_CUDA(cudaMemsetAsync(p->d.err, 0, sizeof err, p->s));
        RT_CUDA(cudaMemsetAsync(p->d.grid_state, 0, sizeof(unsigned) * GRID_STATE_WORDS, p->s));
        RT_CUDA(cudaStreamSynchronize(p->s));
        return rfail(FM_ECUDA, "a grid barrier ran into its limit");
    }
    if (err & ERR_DEGENERATE) {
        const unsigned zero = 0;
        RT_CUDA(cudaMemcpyAsync(p->d.err, &zero, sizeof zero, cudaMemcpyHostToDevice, p->s));
        RT_CUDA(cudaStreamSynchronize(p->s));
        return rfail(FM_EDEGENERATE, "a solved rotation column vanished or is not finite (last solve: " +
                                         std::to_string(p->cg_iters_last) + " conjugate-gradient iterations, " +
                                         "relative residual " + std::to_string(p->cg_resid_last) + ")");
    }
    return FM_OK;
}

constexpr int ROT_CHAIN = 4096;

int cblocks(const fm_rotation *p) { return cam_blocks(p->d.n_cams); }
int tblocks(const fm_rotation *p) { return (p->d.n_cams + RT_THREADS - 1) / RT_THREADS; }

void free_rot(fm_rotation *p) {
    if (!p) return;
    if (p->s) cudaStreamSynchronize(p->s);
    for (void *a : p->allocs) cudaFree(a);
    if (p->ev_in) cudaEventDestroy(p->ev_in);
    if (p->ev_out) cudaEventDestroy(p->ev_out);
    if (p->s) cudaStreamDestroy(p->s);
    delete p;
}

bool rfinite(const double *a, size_t n) {
    for (size_t i = 0; i < n; ++i)
        if (!std::isfinite(a[i])) return false;
    return true;
}

fm_status upload_hyper(fm_rotation *p) {
    const double h[4] = {p->opt.lr, p->opt.beta1, p->opt.beta2, p->opt.adam_eps};
    RT_CUDA(cudaMemcpyAsync(p->d.hyper, h, sizeof h, cudaMemcpyHostToDevice, p->s));
    RT_CUDA(cudaStreamSynchronize(p->s));
    return FM_OK;
}

fm_status create_rot(fm_rotation *p, int32_t n_cams, int32_t n_pairs, const int32_t *cam_i, const int32_t *cam_j,
                     const double *R_rel) {
    DevRot &d = p->d;
    d.n_cams = n_cams;
    d.n_pairs = n_pairs;
    RT_CUDA(cudaStreamCreateWithFlags(&p->s, cudaStreamNonBlocking));
    RT_CUDA(cudaEventCreateWithFlags(&p->ev_in, cudaEventDisableTiming));
    RT_CUDA(cudaEventCreateWithFlags(&p->ev_out, cudaEventDisableTiming));
    RT_CUDA(rjoin_in(p));
    std::vector<int> cam_off(n_cams + 1, 0), cam_ent(2 * (size_t)n_pairs);
    for (int n = 0; n < n_pairs; ++n) {
        cam_off[cam_i[n] + 1]++;
        cam_off[cam_j[n] + 1]++;
    }
    for (int k = 0; k < n_cams; ++k) cam_off[k + 1] += cam_off[k];
    {
        std::vector<int> fill(cam_off.begin(), cam_off.end() - 1);
        for (int n = 0; n < n_pairs; ++n) {
            cam_ent[fill[cam_i[n]]++] = 2 * n;
            cam_ent[fill[cam_j[n]]++] = 2 * n + 1;
        }
    }
    int *ci = nullptr, *cj = nullptr, *co = nullptr, *ce = nullptr;
    double *rr = nullptr;
    RT_CUDA(ralloc(p, &ci, (size_t)n_pairs));
    RT_CUDA(ralloc(p, &cj, (size_t)n_pairs));
    RT_CUDA(ralloc(p, &co, (size_t)n_cams + 1));
    RT_CUDA(ralloc(p, &ce, 2 * (size_t)n_pairs));
    RT_CUDA(ralloc(p, &rr, 9 * (size_t)n_pairs));
    d.cam_i = ci;
    d.cam_j = cj;
    d.cam_off = co;
    d.cam_ent = ce;
    d.Rrel = rr;
    const size_t nc = (size_t)n_cams;
    RT_CUDA(ralloc(p, &d.a, 6 * nc));
    RT_CUDA(ralloc(p, &d.R, 9 * nc));
    RT_CUDA(ralloc(p, &d.m, 6 * nc));
    RT_CUDA(ralloc(p, &d.v, 6 * nc));
    RT_CUDA(ralloc(p, &d.pgrad, 18 * (size_t)n_pairs));
    RT_CUDA(ralloc(p, &d.pdist, (size_t)n_pairs));
    int most_pairs = 0, most_blocks = 0;
    for (int k = 0; k < n_cams; ++k) most_pairs = std::max(most_pairs, cam_off[k + 1] - cam_off[k]);
    p->cg_solve = most_pairs > 256 ? k_cg_solve<true, true> : k_cg_solve<true, false>;
    RT_CUDA(coop_blocks(p->cg_solve, RT_CAMS * 32, &most_blocks));
    if (cam_blocks(n_cams) > most_blocks) {
        p->cg_solve = k_cg_solve<false, true>;
        RT_CUDA(coop_blocks(p->cg_solve, RT_CAMS * 32, &most_blocks));
    }
    p->cg_grid = most_blocks;
    RT_CUDA(coop_blocks(k_rot_steps, RT_CAMS * 32, &p->step_grid));
    p->cg_grid = std::min(p->cg_grid, cam_blocks(n_cams));
    p->step_grid = std::min(p->step_grid, std::max(cam_blocks(n_cams), (n_pairs + 63) / 64));
    RT_CUDA(ralloc(p, &d.blk, 2 * (size_t)cam_blocks(n_cams)));
    RT_CUDA(ralloc(p, &d.grid_state, (size_t)GRID_STATE_WORDS));
    RT_CUDA(ralloc(p, &d.loss, 1));
    RT_CUDA(ralloc(p, &d.hyper, 4));
    RT_CUDA(ralloc(p, &d.step, 1));
    RT_CUDA(ralloc(p, &d.x, 22 * nc));   // the vectors of the solves in one allocation
    {
        double **part[] = {&d.r, &d.z, &d.p, &d.p2, &d.q, &d.pre, &d.cam_rz};
        double *at = d.x;
        for (double **v : part) *v = at += 3 * nc;
    }
    RT_CUDA(ralloc(p, &d.col1, 3 * nc));
    RT_CUDA(ralloc(p, &d.col2, 3 * nc));
    RT_CUDA(ralloc(p, &p->grad6, 6 * nc));
    RT_CUDA(ralloc(p, &d.scal, 8));
    RT_CUDA(ralloc(p, &d.err, 1));
    RT_CUDA(cudaMemcpyAsync(ci, cam_i, sizeof(int) * n_pairs, cudaMemcpyHostToDevice, p->s));
    RT_CUDA(cudaMemcpyAsync(cj, cam_j, sizeof(int) * n_pairs, cudaMemcpyHostToDevice, p->s));
    RT_CUDA(cudaMemcpyAsync(co, cam_off.data(), sizeof(int) * (n_cams + 1), cudaMemcpyHostToDevice, p->s));
    RT_CUDA(cudaMemcpyAsync(ce, cam_ent.data(), sizeof(int) * 2 * n_pairs, cudaMemcpyHostToDevice, p->s));
    RT_CUDA(cudaMemcpyAsync(rr, R_rel, sizeof(double) * 9 * n_pairs, cudaMemcpyHostToDevice, p->s));
    RT_CUDA(cudaMemsetAsync(d.m, 0, sizeof(float) * 6 * nc, p->s));
    RT_CUDA(cudaMemsetAsync(d.v, 0, sizeof(float) * 6 * nc, p->s));
    RT_CUDA(cudaMemsetAsync(d.step, 0, sizeof(long long), p->s));
    RT_CUDA(cudaMemsetAsync(d.err, 0, sizeof(unsigned), p->s));
    RT_CUDA(cudaMemsetAsync(d.col1, 0, sizeof(double) * 3 * nc, p->s));
    RT_CUDA(cudaMemsetAsync(d.scal, 0, sizeof(double) * 8, p->s));
    RT_CUDA(cudaMemsetAsync(d.grid_state, 0, sizeof(unsigned) * GRID_STATE_WORDS, p->s));
    if (fm_status st = upload_hyper(p)) return st;
    RT_CUDA(rjoin_out(p));
    return FM_OK;
}

fm_status rcheck(const fm_rotation *p) {
    if (!p) return rfail(FM_EINVAL, "rotation problem is NULL");
    return FM_OK;
}

}  // namespace

extern "C" {

FM_API void fm_rotation_default_options(fm_rotation_options *opt) {
    if (!opt) return;
    opt->lr = 1e-3;
    opt->beta1 = 0.9;
    opt->beta2 = 0.999;
    opt->adam_eps = 1e-12;
    opt->cg_tol = 1e-9;
    opt->cg_max_iters = 20000;
    opt->use_graph = 1;
}

FM_API fm_status fm_rotation_create(int32_t n_cams, int32_t n_pairs, const int32_t *cam_i, const int32_t *cam_j,
                                    const double *R_rel, const fm_rotation_options *opt, void *stream,
                                    fm_rotation **out) {
    if (!out) return rfail(FM_EINVAL, "out must not be NULL");
    *out = nullptr;
    if (n_cams < 2) return rfail(FM_EINVAL, "n_cams must be >= 2");
    if (n_pairs < 1) return rfail(FM_EINVAL, "n_pairs must be >= 1");
    if (!cam_i || !cam_j || !R_rel) return rfail(FM_EINVAL, "array arguments must not be NULL");
    for (int n = 0; n < n_pairs; ++n)
        if (cam_i[n] < 0 || cam_i[n] >= n_cams || cam_j[n] < 0 || cam_j[n] >= n_cams || cam_i[n] == cam_j[n])
            return rfail(FM_EINVAL, "camera indices must be in [0, n_cams) with cam_i != cam_j");
    if (!rfinite(R_rel, 9 * (size_t)n_pairs)) return rfail(FM_EINVAL, "relative rotations must be finite");
    for (int n = 0; n < n_pairs; ++n) {
        const double *M = R_rel + 9 * (size_t)n;
        double worst = 0.0;
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) {
                const double dot = M[a] * M[b] + M[3 + a] * M[3 + b] + M[6 + a] * M[6 + b];
                worst = std::max(worst, std::fabs(dot - (a == b ? 1.0 : 0.0)));
            }
        const double det = M[0] * (M[4] * M[8] - M[5] * M[7]) - M[1] * (M[3] * M[8] - M[5] * M[6]) +
                           M[2] * (M[3] * M[7] - M[4] * M[6]);
        if (worst > 1e-6 || std::fabs(det - 1.0) > 1e-6)
            return rfail(FM_EINVAL, "relative rotations must be rotation matrices (orthonormal, det +1)");
    }
    {
        // the image graph must be connected (the anchored systems are singular otherwise)
        std::vector<int> parent(n_cams);
        for (int k = 0; k < n_cams; ++k) parent[k] = k;
        auto find = [&](int k) {
            while (parent[k] != k) k = parent[k] = parent[parent[k]];
            return k;
        };
        int comps = n_cams;
        for (int n = 0; n < n_pairs; ++n) {
            const int a = find(cam_i[n]), b = find(cam_j[n]);
            if (a != b) {
                parent[a] = b;
                --comps;
            }
        }
        if (comps != 1) return rfail(FM_EINVAL, "the image graph must be connected");
    }
    fm_rotation_options o;
    fm_rotation_default_options(&o);
    if (opt) o = *opt;
    if (!(o.lr > 0.0) || !(o.beta1 >= 0.0 && o.beta1 < 1.0) || !(o.beta2 >= 0.0 && o.beta2 < 1.0) ||
        !(o.adam_eps > 0.0) || !(o.cg_tol > 0.0) || o.cg_max_iters < 1 || (o.use_graph != 0 && o.use_graph != 1))
        return rfail(FM_EINVAL, "invalid options");
    fm_rotation *p = new (std::nothrow) fm_rotation();
    if (!p) return rfail(FM_ENOMEM, "host allocation failed");
    p->opt = o;
    p->user = static_cast<cudaStream_t>(stream);
    fm_status st = create_rot(p, n_cams, n_pairs, cam_i, cam_j, R_rel);
    if (st != FM_OK) {
        free_rot(p);
        return st;
    }
    *out = p;
    return FM_OK;
}

FM_API void fm_rotation_destroy(fm_rotation *p) { free_rot(p); }

FM_API fm_status fm_rotation_initialize(fm_rotation *p, int32_t *cg_iters, double *cg_residual) {
    if (fm_status st = rcheck(p)) return st;
    RT_CUDA(rjoin_in(p));
    const double n_pairs = (double)p->d.n_pairs, n_cams = (double)p->d.n_cams;
    // column 1: sum ||x_j - R_p x_i||^2, anchored x_0 = e1; column 2: (1/|P|) sum ||y_j - R_p y_i||^2 +
    // (1/N) sum (x_k^T y_k)^2, anchored y_0 = e2
    RT_CUDA(cudaMemsetAsync(p->d.scal, 0, sizeof(double) * 8, p->s));
    RT_CUDA(launch_coop(p->cg_solve, p->cg_grid, RT_CAMS * 32, 0, p->s, p->d, 0, 1.0, 0.0, (int)p->opt.cg_max_iters,
                        p->opt.cg_tol));
    RT_CUDA(launch_coop(p->cg_solve, p->cg_grid, RT_CAMS * 32, 0, p->s, p->d, 1, 1.0 / n_pairs, 1.0 / n_cams,
                        (int)p->opt.cg_max_iters, p->opt.cg_tol));
    double sc[8] = {};
    RT_CUDA(cudaMemcpyAsync(sc, p->d.scal, sizeof sc, cudaMemcpyDeviceToHost, p->s));
    RT_CUDA(cudaStreamSynchronize(p->s));
    auto resid = [&](int c) { return sc[4 * c] > 0.0 ? std::sqrt(sc[4 * c + 1] / sc[4 * c]) : 0.0; };
    p->cg_iters_last = (int)(sc[6] > 0.0 ? sc[6] : sc[2]);
    p->cg_resid_last = sc[6] > 0.0 ? resid(1) : resid(0);
    if (fm_status st = rcheck_errors(p)) return st;
    if (cg_iters) *cg_iters = (int)(sc[2] + sc[6]);
    if (cg_residual) *cg_residual = std::max(resid(0), resid(1));
    return FM_OK;
}

FM_API fm_status fm_rotation_set_rotations(fm_rotation *p, const double *R) {
    if (fm_status st = rcheck(p)) return st;
    if (!R) return rfail(FM_EINVAL, "R must not be NULL");
    if (!rfinite(R, 9 * (size_t)p->d.n_cams)) return rfail(FM_EINVAL, "rotations must be finite");
    RT_CUDA(rjoin_in(p));
    RT_CUDA(cudaMemcpyAsync(p->d.R, R, sizeof(double) * 9 * p->d.n_cams, cudaMemcpyHostToDevice, p->s));
    k_params_from_rot<<<tblocks(p), RT_THREADS, 0, p->s>>>(p->d);
    k_rot_from_params<<<tblocks(p), RT_THREADS, 0, p->s>>>(p->d);
    RT_CUDA(cudaGetLastError());
    RT_CUDA(cudaMemsetAsync(p->d.m, 0, sizeof(float) * 6 * p->d.n_cams, p->s));
    RT_CUDA(cudaMemsetAsync(p->d.v, 0, sizeof(float) * 6 * p->d.n_cams, p->s));
    RT_CUDA(cudaMemsetAsync(p->d.step, 0, sizeof(long long), p->s));
    RT_CUDA(cudaStreamSynchronize(p->s));
    return FM_OK;
}

FM_API fm_status fm_rotation_set_params(fm_rotation *p, const double *a6) {
    if (fm_status st = rcheck(p)) return st;
    if (!a6) return rfail(FM_EINVAL, "a6 must not be NULL");
    if (!rfinite(a6, 6 * (size_t)p->d.n_cams)) return rfail(FM_EINVAL, "parameters must be finite");
    RT_CUDA(rjoin_in(p));
    RT_CUDA(cudaMemcpyAsync(p->d.a, a6, sizeof(double) * 6 * p->d.n_cams, cudaMemcpyHostToDevice, p->s));
    k_rot_from_params<<<tblocks(p), RT_THREADS, 0, p->s>>>(p->d);
    RT_CUDA(cudaGetLastError());
    RT_CUDA(cudaMemsetAsync(p->d.m, 0, sizeof(float) * 6 * p->d.n_cams, p->s));
    RT_CUDA(cudaMemsetAsync(p->d.v, 0, sizeof(float) * 6 * p->d.n_cams, p->s));
    RT_CUDA(cudaMemsetAsync(p->d.step, 0, sizeof(long long), p->s));
    RT_CUDA(cudaStreamSynchronize(p->s));
    return FM_OK;
}

FM_API fm_status fm_rotation_loss_grad(fm_rotation *p, double *loss, double *grad6) {
    if (fm_status st = rcheck(p)) return st;
    if (!loss) return rfail(FM_EINVAL, "loss must not be NULL");
    RT_CUDA(rjoin_in(p));
    const dim3 gp((p->d.n_pairs + RT_THREADS - 1) / RT_THREADS);
    launch_k(k_rot_pair, gp, dim3(RT_THREADS), p->s, false, p->d);
    launch_k(k_rot_cam, dim3(cblocks(p)), dim3(RT_CAMS * 32), p->s, true, p->d, p->grad6);
    launch_k(k_rot_finish, dim3(1), dim3(RT_THREADS), p->s, true, p->d);
    RT_CUDA(cudaGetLastError());
    RT_CUDA(cudaMemcpyAsync(loss, p->d.loss, sizeof(double), cudaMemcpyDeviceToHost, p->s));
    if (grad6)
        RT_CUDA(cudaMemcpyAsync(grad6, p->grad6, sizeof(double) * 6 * p->d.n_cams, cudaMemcpyDeviceToHost, p->s));
    return rcheck_errors(p);
}

FM_API fm_status fm_rotation_step(fm_rotation *p, int32_t n_iters) {
    if (fm_status st = rcheck(p)) return st;
    if (n_iters < 0) return rfail(FM_EINVAL, "n_iters must be >= 0");
    if (n_iters == 0) return FM_OK;
    RT_CUDA(rjoin_in(p));
    // launches of bounded length (a step takes microseconds); use_graph makes no difference
    for (int left = n_iters; left > 0; left -= ROT_CHAIN)
        RT_CUDA(launch_coop(k_rot_steps, p->step_grid, RT_CAMS * 32, 0, p->s, p->d, std::min(left, ROT_CHAIN)));
    RT_CUDA(rjoin_out(p));
    return FM_OK;
}

FM_API fm_status fm_rotation_set_learning_rate(fm_rotation *p, double lr) {
    if (fm_status st = rcheck(p)) return st;
    if (!(lr > 0.0) || std::isinf(lr)) return rfail(FM_EINVAL, "lr must be finite and > 0");
    RT_CUDA(rjoin_in(p));
    p->opt.lr = lr;
    return upload_hyper(p);
}

FM_API fm_status fm_rotation_get_rotations(fm_rotation *p, double *R) {
    if (fm_status st = rcheck(p)) return st;
    if (!R) return rfail(FM_EINVAL, "R must not be NULL");
    RT_CUDA(rjoin_in(p));
    RT_CUDA(cudaMemcpyAsync(R, p->d.R, sizeof(double) * 9 * p->d.n_cams, cudaMemcpyDeviceToHost, p->s));
    return rcheck_errors(p);
}

FM_API fm_status fm_rotation_get_params(fm_rotation *p, double *a6) {
    if (fm_status st = rcheck(p)) return st;
    if (!a6) return rfail(FM_EINVAL, "a6 must not be NULL");
    RT_CUDA(rjoin_in(p));
    RT_CUDA(cudaMemcpyAsync(a6, p->d.a, sizeof(double) * 6 * p->d.n_cams, cudaMemcpyDeviceToHost, p->s));
    return rcheck_errors(p);
}

}  // extern "C"
