// grad.cuh -- adjoint of (rational) Bezier curve evaluation.
//
// For curves C(t) = A(t) / W(t), A = sum_i B_i(t) w_i P_i, W = sum_i B_i(t) w_i
// (w = 1 for integral curves) and an upstream gradient g_j = dL/dC(t_j):
//   dL/dP_i = sum_j (w_i B_i(t_j) / W_j) g_j
//   dL/dw_i = sum_j B_i(t_j) (P_i - C_j) . g_j / W_j
//   dL/dt_j = g_j . (A'(t_j) - C_j W'(t_j)) / W_j      (0 where t was clamped)
// with A' = d sum_i B_i^(d-1) (w_(i+1) P_(i+1) - w_i P_i) and W' likewise.
// The Bernstein values come from the basis triangle B^(r)_i = (1-t) B^(r-1)_i
// + t B^(r-1)_(i-1), whose level d-1 gives the derivative basis.
//
// Fused squared error (target given): g_j = 2 s (C(t_j) - target_j) is formed
// in the kernel from the curve value it computes anyway, and the per-curve
// loss s sum_j ||C(t_j) - target_j||^2 is summed alongside, so a fitting step
// reads t and the targets once and writes dt (no point or gradient arrays).
//
// One warp per curve; lanes take samples j = lane + 32 m (coalesced reads of
// t and g), two at a time (j and j + 32: independent arithmetic to
// interleave), keep per-lane partial sums of the per-curve gradients in
// registers, and combine them at the end of the curve (one 16-value
// reduce-scatter for fixed degrees, butterflies otherwise).  Per-sample dt is
// written directly (per-curve t) or summed over curves (shared t) in shared
// memory and then with one global atomic per block and parameter.  The next
// pair's loads are issued before the current pair's arithmetic, and the
// output mode is decided once per launch, outside the sample loop.
//
// Integral curves of degree <= 4 (GradPoly): the curve and its derivative come
// from the power basis about t = 1/2 by one Horner scheme, and dL/dP_i sums
// t^i (1-t)^(d-i) g, the binomial applied once per curve (products of powers, so
// small basis values keep their relative accuracy): 47 arithmetic instructions a
// sample of a cubic in 3D instead of 79 for the basis triangle and its sums.
// 65,536 cubics x 512 with their own t and the fused loss: 139 -> 128 us (5.3
// TB/s; issue 66 %, waiting on the sample loads); 2D: 1034 -> 106 us with the
// runtime-degree kernel before; degree 4: 175 -> 144 us.
// Rational curves and higher degrees (GradCurve):
// per curve the homogeneous points q_i = w_i P_i and the scaled differences
// d (q_(i+1) - q_i), d (w_(i+1) - w_i) are formed once, so a sample costs the
// basis triangle plus one FMA per (point, coordinate) for each of A, A' and
// dL/dP.  Integral curves (RAT false) drop W, W', the division and the weight
// sums: C = A exactly as the Bernstein sum.
#pragma once

#include "curve_eval.cuh"

namespace bez {

constexpr int kGradMaxDim = 4;

// samples per loop iteration: two independent samples to interleave while
// the pair's registers fit, one for high degrees
__host__ __device__ constexpr int grad_pair(int D, bool RAT) { return (D >= 1 && D <= (RAT ? 3 : 4)) ? 2 : 1; }

// resident blocks per SM the register budget is sized for (48 to 128 registers
// a thread at 256 threads a block); measured with one more and one fewer (us at
// 65,536 x 512: degree 4 144 at 3, 179 at 2; 2D conics with weights 145 at 3,
// 174 at 2; 3D rational cubics 205 at 2, 239 at 3; cubics 128 at 4, 183 at 5)
__host__ __device__ constexpr int grad_min_blocks(int D, int DIM, bool RAT)
{
    return D == 0 ? 2
           : RAT ? (D * DIM <= 6 ? 3 : 2)
                 : D <= 1 ? 5 : D <= 3 ? 4 : (D + 1) * DIM <= 18 ? 3 : 2;
}

// dL/dt output: none, per-curve array, or shared t summed over curves with
// atomics into gt_sum (this block's shared-memory partial sums, or the global
// array when n_t is too large for shared memory)
enum { GT_NONE = 0, GT_PER_CURVE = 1, GT_SHARED = 2 };

// One curve's state in a lane: control data and the lane's partial sums.
template <int D, int DIM, bool RAT>
struct GradCurve {
    static constexpr int N = Deg<D>::N;
    static constexpr int M = DIM ? DIM : kGradMaxDim;
    int d, dim;
    float P[N][M], w[N], dq[N][M], dw[N];
    float acc_c[N][M], acc_w[N], loss;

    __device__ __forceinline__ void setup(const GradArgs& a, int64_t c)
    {
        d = Deg<D>::get(a.degree);
        dim = DIM ? DIM : a.dim;
        const int dd = D ? D : d;  // a constant bound unrolls; the runtime degree loops
        float q[N][M];
#pragma unroll
        for (int i = 0; i <= dd; ++i) {
            w[i] = RAT ? __ldg(a.weights + c * (d + 1) + i) : 1.f;
#pragma unroll
            for (int k = 0; k < M; ++k) {
                if (k >= dim) break;
                P[i][k] = __ldg(a.ctrl + (c * (d + 1) + i) * dim + k);
                q[i][k] = RAT ? w[i] * P[i][k] : P[i][k];
            }
        }
        const float fd = (float)d;
#pragma unroll
        for (int i = 0; i < dd; ++i) {
            if (RAT) dw[i] = fd * (w[i + 1] - w[i]);
#pragma unroll
            for (int k = 0; k < M; ++k) {
                if (k >= dim) break;
                dq[i][k] = fd * (q[i + 1][k] - q[i][k]);
            }
        }
#pragma unroll
        for (int i = 0; i <= dd; ++i) {
            acc_w[i] = 0.f;
#pragma unroll
            for (int k = 0; k < M; ++k) acc_c[i][k] = 0.f;
        }
        loss = 0.f;
    }

    // One sample: accumulate its dL/dP, dL/dw (and loss) terms; return dL/dt.
    // FUSED: v is the target and g = g2 (C - v) mask; else v is g.  A sample
    // past the end arrives with mask 0 (fused) or v = 0, and adds nothing.
    template <bool FUSED>
    __device__ __forceinline__ float sample(float traw, const float (&v)[M], float mask, float g2)
    {
        const int dd = D ? D : d;
        const float t = clamp01(traw);
        const float s = 1.0f - t;
        // basis triangle; keep level d-1 for the derivative
        float B[N], Bd[N];
        B[0] = 1.f;
#pragma unroll
        for (int r = 1; r <= dd; ++r) {
            if (r == dd) {
#pragma unroll
                for (int i = 0; i < dd; ++i) Bd[i] = B[i];
            }
            B[r] = t * B[r - 1];
#pragma unroll
            for (int i = r - 1; i >= 1; --i) B[i] = fmaf(t, B[i - 1], s * B[i]);
            B[0] = s * B[0];
        }
        float A[M], dA[M];
        float W = RAT ? 0.f : 1.f, dW = 0.f;
#pragma unroll
        for (int k = 0; k < M; ++k) A[k] = dA[k] = 0.f;
#pragma unroll
        for (int i = 0; i <= dd; ++i) {
            const float bw = RAT ? B[i] * w[i] : B[i];
            if (RAT) W += bw;
#pragma unroll
            for (int k = 0; k < M; ++k)
                if (k < dim) A[k] = fmaf(bw, P[i][k], A[k]);
        }
#pragma unroll
        for (int i = 0; i < dd; ++i) {
            if (RAT) dW = fmaf(Bd[i], dw[i], dW);
#pragma unroll
            for (int k = 0; k < M; ++k)
                if (k < dim) dA[k] = fmaf(Bd[i], dq[i][k], dA[k]);
        }
        const float invW = RAT ? __frcp_rn(W) : 1.f;
        float C[M], gj[M];
#pragma unroll
        for (int k = 0; k < M; ++k) {
            C[k] = RAT ? A[k] * invW : A[k];
            if (FUSED) {
                // fused squared error: g = 2 s (C - target), loss += ||C - target||^2
                const float r = (C[k] - v[k]) * mask;
                gj[k] = g2 * r;
                if (k < dim) loss = fmaf(r, r, loss);
            } else {
                gj[k] = v[k];
            }
        }
#pragma unroll
        for (int i = 0; i <= dd; ++i) {
            const float f = RAT ? B[i] * w[i] * invW : B[i];
#pragma unroll
            for (int k = 0; k < M; ++k)
                if (k < dim) acc_c[i][k] = fmaf(f, gj[k], acc_c[i][k]);
            if (RAT) {
                float dot = 0.f;
#pragma unroll
                for (int k = 0; k < M; ++k)
                    if (k < dim) dot = fmaf(P[i][k] - C[k], gj[k], dot);
                acc_w[i] = fmaf(B[i] * invW, dot, acc_w[i]);
            }
        }
        float gt = 0.f;
#pragma unroll
        for (int k = 0; k < M; ++k)
            if (k < dim) gt = fmaf(gj[k], RAT ? fmaf(-C[k], dW, dA[k]) : dA[k], gt);
        return (traw >= 0.f && traw <= 1.f) ? (RAT ? gt * invW : gt) : 0.f;  // clamped t: no dL/dt
    }

    // Per-curve sums over the warp.  Fixed degree and dim: the values
    // (dL/dP, dL/dw, loss) go through one 16-value reduce-scatter, lane 2e
    // writing value e, and any beyond 16 through butterflies; otherwise one
    // butterfly per value, lane e writing element e.
    __device__ __forceinline__ void finish(const GradArgs& a, int64_t c, int lane)
    {
        if constexpr (D > 0 && DIM > 0) {
            constexpr int NC = N * M;                      // dL/dP values
            constexpr int NV = NC + (RAT ? N : 0) + 1;     // + dL/dw + loss
            float v[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                float x = 0.f;
                if (e < NC) x = acc_c[e / M][e % M];
                else if (RAT && e < NC + N) x = acc_w[e - NC];
                else if (e == NV - 1) x = loss;
                v[e] = x;
            }
            const float tot = warp_sum16_scatter(v, lane);
            const int e = (lane >> 1) & 15;
            if ((lane & 1) == 0) {
                if (e < NC) {
                    if (a.grad_ctrl) a.grad_ctrl[c * NC + e] = tot;
                } else if (RAT && e < NC + N) {
                    if (a.grad_w) a.grad_w[c * N + (e - NC)] = tot;
                } else if (e == NV - 1 && a.loss) {
                    a.loss[c] = a.loss_scale * tot;
                }
            }
            if constexpr (NV > 16) {
                // values 16.. (at most 16 more here): one butterfly each
#pragma unroll
                for (int e2 = 16; e2 < NV; ++e2) {
                    float x = e2 < NC ? acc_c[e2 / M][e2 % M] : (RAT && e2 < NC + N) ? acc_w[e2 - NC] : loss;
                    x = warp_sum(x);
                    if (lane == 0) {
                        if (e2 < NC) {
                            if (a.grad_ctrl) a.grad_ctrl[c * NC + e2] = x;
                        } else if (RAT && e2 < NC + N) {
                            if (a.grad_w) a.grad_w[c * N + (e2 - NC)] = x;
                        } else if (a.loss) {
                            a.loss[c] = a.loss_scale * x;
                        }
                    }
                }
            }
            return;
        }
        const int nc = (d + 1) * dim;
        const int dd = D ? D : d;
#pragma unroll
        for (int i = 0; i <= dd; ++i) {
#pragma unroll
            for (int k = 0; k < M; ++k) {
                if (k >= dim) break;
                const float v = warp_sum(acc_c[i][k]);
                if (a.grad_ctrl && lane == (i * dim + k) % 32) a.grad_ctrl[c * nc + i * dim + k] = v;
            }
            if (RAT) {
                const float vw = warp_sum(acc_w[i]);
                if (a.grad_w && lane == i % 32) a.grad_w[c * (d + 1) + i] = vw;
            }
        }
        if (a.loss) {
            const float l = warp_sum(loss);
            if (lane == 0) a.loss[c] = a.loss_scale * l;
        }
    }
};

// binom(D, i) as immediate operands (binom_c, called with an unrolled loop's
// index, would recurse at run time)
template <int D>
struct BinomRow {
    float v[D + 1];
};
template <int D>
constexpr BinomRow<D> make_binom_row()
{
    BinomRow<D> r{};
    for (int i = 0; i <= D; ++i) r.v[i] = (float)binom_c(D, i);
    return r;
}

// Coefficients about t = 1/2 of one component b_0 .. b_D of a curve, D <= 4.
// Those of order >= 1 cancel the curve's distance from the origin.  From degree 3
// they are formed from differences of its points (mirrored pairs b_(D-i) - b_i,
// and distances from the middle): summed from the points themselves they keep the
// rounding of the distance, and C' of a unit cubic 1000 from the origin an error
// of 5.6e-5 instead of 6.9e-8 (at the origin 9.4e-8 and 9.2e-8, quartics 1.31e-7
// and 1.27e-7: RMS over uniform points and t).  In degrees 1 and 2 the sums of
// the points cancel without that.
template <int D>
__device__ __forceinline__ void centred_from_differences(const float (&b)[D + 1], float (&c)[D + 1])
{
    constexpr CentredMatrix<D> T = make_centred_matrix<D>();
#pragma unroll
    for (int m = 0; m <= (D >= 3 ? 0 : D); ++m) {
        float x = T.t[m][0] * b[0];
#pragma unroll
        for (int i = 1; i <= D; ++i) x = fmaf(T.t[m][i], b[i], x);
        c[m] = x;
    }
    if constexpr (D == 3) {
        const float p = b[3] - b[0], q = b[2] - b[1], r = b[0] - b[1], s = b[3] - b[2];
        c[1] = fmaf(0.75f, p, 0.75f * q);
        c[2] = fmaf(1.5f, r, 1.5f * s);
        c[3] = fmaf(-3.f, q, p);
    } else if constexpr (D == 4) {
        const float p = b[4] - b[0], q = b[3] - b[1];
        const float r = b[0] - b[2], s = b[4] - b[2], v = b[1] - b[2], w = b[3] - b[2];
        c[1] = fmaf(0.5f, p, q);
        c[2] = fmaf(1.5f, r, 1.5f * s);
        c[3] = fmaf(2.f, p, -4.f * q);
        c[4] = fmaf(-4.f, v, fmaf(-4.f, w, r + s));
    }
}

// One integral curve of fixed degree <= 4 in a lane: its coefficients about
// t = 1/2 and the lane's sums.
template <int D, int DIM>
struct GradPoly {
    static constexpr int M = DIM;
    float c[D + 1][DIM], acc[D + 1][DIM], loss;

    __device__ __forceinline__ void setup(const GradArgs& a, int64_t cv)
    {
        const float* ctrl = a.ctrl + cv * ((D + 1) * DIM);
        float b[DIM][D + 1];
#pragma unroll
        for (int i = 0; i <= D; ++i)
#pragma unroll
            for (int k = 0; k < DIM; ++k) b[k][i] = __ldg(ctrl + i * DIM + k);
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            float x[D + 1];
            centred_from_differences<D>(b[k], x);
#pragma unroll
            for (int m = 0; m <= D; ++m) {
                c[m][k] = x[m];
                acc[m][k] = 0.f;
            }
        }
        loss = 0.f;
    }

    // One sample, as GradCurve::sample.
    template <bool FUSED>
    __device__ __forceinline__ float sample(float traw, const float (&v)[DIM], float mask, float g2)
    {
        const float t = clamp01(traw);
        const float u = t - 0.5f, s = 1.0f - t;
        float g[DIM], gt = 0.f;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            float p = c[D][k], d = 0.f;
#pragma unroll
            for (int i = D - 1; i >= 0; --i) {
                d = i == D - 1 ? p : fmaf(d, u, p);
                p = fmaf(p, u, c[i][k]);
            }
            if (FUSED) {
                // fused squared error: g = 2 s (C - target), loss += ||C - target||^2
                const float r = (p - v[k]) * mask;
                g[k] = g2 * r;
                loss = fmaf(r, r, loss);
            } else {
                g[k] = v[k];
            }
            gt = fmaf(g[k], d, gt);
        }
        float tp[D + 1], sp[D + 1];
        tp[0] = sp[0] = 1.f;
        tp[1] = t;
        sp[1] = s;
#pragma unroll
        for (int i = 2; i <= D; ++i) {
            tp[i] = tp[i - 1] * t;
            sp[i] = sp[i - 1] * s;
        }
#pragma unroll
        for (int i = 0; i <= D; ++i) {
            const float B = i == 0 ? sp[D] : i == D ? tp[D] : tp[i] * sp[D - i];  // Bernstein value / binom(D, i)
#pragma unroll
            for (int k = 0; k < DIM; ++k) acc[i][k] = fmaf(B, g[k], acc[i][k]);
        }
        return (traw >= 0.f && traw <= 1.f) ? gt : 0.f;  // clamped t: no dL/dt
    }

    // Sums over the warp, 16 values at a time by reduce-scatter: lane 2e writes
    // value e.
    __device__ __forceinline__ void finish(const GradArgs& a, int64_t cv, int lane)
    {
        constexpr int NC = (D + 1) * DIM, NV = NC + 1;
        constexpr BinomRow<D> bin = make_binom_row<D>();
#pragma unroll
        for (int r = 0; r < (NV + 15) / 16; ++r) {
            float v[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int x = 16 * r + e;
                v[e] = x < NC ? bin.v[x / DIM] * acc[x / DIM][x % DIM] : x == NC ? loss : 0.f;
            }
            const float tot = warp_sum16_scatter(v, lane);
            const int e = 16 * r + (lane >> 1);
            if ((lane & 1) == 0) {
                if (e < NC) {
                    if (a.grad_ctrl) a.grad_ctrl[cv * NC + e] = tot;
                } else if (e == NC && a.loss) {
                    a.loss[cv] = a.loss_scale * tot;
                }
            }
        }
    }
};

template <int D, int DIM, bool RAT>
struct GradPick {
    using type = GradCurve<D, DIM, RAT>;
};
template <int DIM>
struct GradPick<1, DIM, false> {
    using type = GradPoly<1, DIM>;
};
template <int DIM>
struct GradPick<2, DIM, false> {
    using type = GradPoly<2, DIM>;
};
template <int DIM>
struct GradPick<3, DIM, false> {
    using type = GradPoly<3, DIM>;
};
template <int DIM>
struct GradPick<4, DIM, false> {
    using type = GradPoly<4, DIM>;
};

// read-only load asking L2 to fetch the whole 256-byte block around the
// address, so that a warp's streaming reads of t and the targets bring the
// next rows into L2 with the current ones
__device__ __forceinline__ float ld_stream(const float* p)
{
    float v;
    asm("ld.global.nc.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

template <int M>
__device__ __forceinline__ void load_sample(const float* tc, const float* vc, int dim, int n_t, int j, float& t,
                                            float (&v)[M])
{
    t = 0.f;
#pragma unroll
    for (int k = 0; k < M; ++k) v[k] = 0.f;
    if (j < n_t) {
        t = ld_stream(tc + j);
#pragma unroll
        for (int k = 0; k < M; ++k)
            if (k < dim) v[k] = ld_stream(vc + j * dim + k);
    }
}

template <int GTM>
__device__ __forceinline__ void put_gt(float* gtc, float* gt_sum, int j, float gt)
{
    if (GTM == GT_PER_CURVE) gtc[j] = gt;
    else if (GTM == GT_SHARED) atomicAdd(gt_sum + j, gt);
}

template <int D, int DIM, bool RAT, bool FUSED, int GTM>
__device__ __forceinline__ void grad_curves(const GradArgs& a, float* gt_sum)
{
    using G = typename GradPick<D, DIM, RAT>::type;
    constexpr int M = G::M;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int n_t = a.n_t;
    const int dim = DIM ? DIM : a.dim;
    const float* vsrc = FUSED ? a.target : a.g;
    const float g2 = 2.0f * a.loss_scale;
    const int64_t n_warps = (int64_t)gridDim.x * kWarps;
    for (int64_t c = (int64_t)blockIdx.x * kWarps + wib; c < a.n_curves; c += n_warps) {
        G e;
        const float* tc = a.t + c * a.t_stride;
        const float* vc = vsrc + c * (int64_t)n_t * dim;
        float* gtc = GTM == GT_PER_CURVE ? a.grad_t + c * (int64_t)n_t : nullptr;
        if constexpr (grad_pair(D, RAT) == 2) {
            float tA, tB, vA[M], vB[M];
            load_sample<M>(tc, vc, dim, n_t, lane, tA, vA);
            load_sample<M>(tc, vc, dim, n_t, lane + 32, tB, vB);
            e.setup(a, c);  // its loads go out beside the first pair's
            for (int j = lane; j < n_t; j += 64) {
                const float t0 = tA, t1 = tB;
                float v0[M], v1[M];
#pragma unroll
                for (int k = 0; k < M; ++k) {
                    v0[k] = vA[k];
                    v1[k] = vB[k];
                }
                load_sample<M>(tc, vc, dim, n_t, j + 64, tA, vA);
                load_sample<M>(tc, vc, dim, n_t, j + 96, tB, vB);
                const bool has1 = j + 32 < n_t;
                const float gt0 = e.template sample<FUSED>(t0, v0, 1.f, g2);
                const float gt1 = e.template sample<FUSED>(t1, v1, has1 ? 1.f : 0.f, g2);
                put_gt<GTM>(gtc, gt_sum, j, gt0);
                if (has1) put_gt<GTM>(gtc, gt_sum, j + 32, gt1);
            }
        } else {
            float tA, vA[M];
            load_sample<M>(tc, vc, dim, n_t, lane, tA, vA);
            e.setup(a, c);
            for (int j = lane; j < n_t; j += 32) {
                const float t0 = tA;
                float v0[M];
#pragma unroll
                for (int k = 0; k < M; ++k) v0[k] = vA[k];
                load_sample<M>(tc, vc, dim, n_t, j + 32, tA, vA);
                put_gt<GTM>(gtc, gt_sum, j, e.template sample<FUSED>(t0, v0, 1.f, g2));
            }
        }
        e.finish(a, c, lane);
    }
}

template <int D, int DIM, bool RAT>
__global__ void __launch_bounds__(kWarps * 32, grad_min_blocks(D, DIM, RAT)) k_grad(const GradArgs a)
{
    extern __shared__ float s_gt[];  // shared-t dL/dt partial sums of this block
    const int gtm = !a.grad_t ? GT_NONE : a.t_stride ? GT_PER_CURVE : GT_SHARED;
    const bool smem_sum = gtm == GT_SHARED && a.shared_gt;
    float* gt_sum = smem_sum ? s_gt : a.grad_t;
    if (smem_sum) {
        for (int j = threadIdx.x; j < a.n_t; j += blockDim.x) s_gt[j] = 0.f;
        __syncthreads();
    }
    if (a.target) {
        if (gtm == GT_NONE) grad_curves<D, DIM, RAT, true, GT_NONE>(a, gt_sum);
        else if (gtm == GT_PER_CURVE) grad_curves<D, DIM, RAT, true, GT_PER_CURVE>(a, gt_sum);
        else grad_curves<D, DIM, RAT, true, GT_SHARED>(a, gt_sum);
    } else {
        if (gtm == GT_NONE) grad_curves<D, DIM, RAT, false, GT_NONE>(a, gt_sum);
        else if (gtm == GT_PER_CURVE) grad_curves<D, DIM, RAT, false, GT_PER_CURVE>(a, gt_sum);
        else grad_curves<D, DIM, RAT, false, GT_SHARED>(a, gt_sum);
    }
    if (smem_sum) {
        __syncthreads();
        for (int j = threadIdx.x; j < a.n_t; j += blockDim.x) atomicAdd(a.grad_t + j, s_gt[j]);
    }
}

// The kernels of points of dimension DIM (degrees 1..7 in 3D, 1..5 otherwise),
// or NULL for the runtime-degree kernel.
template <int DIM, bool RAT>
static const void* grad_kernel_dim(int degree)
{
    switch (degree) {
    case 1: return (const void*)k_grad<1, DIM, RAT>;
    case 2: return (const void*)k_grad<2, DIM, RAT>;
    case 3: return (const void*)k_grad<3, DIM, RAT>;
    case 4: return (const void*)k_grad<4, DIM, RAT>;
    case 5: return (const void*)k_grad<5, DIM, RAT>;
    default: break;
    }
    if constexpr (DIM == 3) {
        if (degree == 6) return (const void*)k_grad<6, DIM, RAT>;
        if (degree == 7) return (const void*)k_grad<7, DIM, RAT>;
    }
    return nullptr;
}
// dimensions 1, 2 and 4 (grad_dims.cu)
const void* grad_kernel_dims(int degree, int dim, bool rat);

}  // namespace bez
