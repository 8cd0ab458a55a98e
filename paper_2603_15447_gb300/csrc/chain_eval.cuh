// chain_eval.cuh -- C0 piecewise Bezier chains evaluated in registers.
//
// A chain of n_seg segments of degree p shares end points: segment k uses
// control points k*p .. k*p+p.  Global t in [0, n_seg] selects segment
// k = min(floor(t), n_seg-1) and local parameter tau = t - k (the reading
// used for ties: an integer t starts the later segment).  One warp owns a
// chain, stages its control points in shared memory, and evaluates each
// sample with the per-curve evaluators of curve_eval.cuh (setup per sample,
// since consecutive samples may fall in different segments).  Centred Horner
// on quadratic and cubic 3D chains stages the segments' power coefficients
// about tau = 1/2 instead (one conversion per segment, not per sample), one
// float4 per coefficient, so a sample reads d + 1 vectors and runs d FMA per
// coordinate.
#pragma once

#include "curve_tile.cuh"

namespace bez {

// global chain parameter of sample j, clamped to [0, n_seg] (NaN kept)
template <int TM>
__device__ __forceinline__ float chain_param(const CurveArgs& a, int64_t c, int j, uint32_t kc)
{
    const float ns = (float)a.n_seg;
    if (TM == TM_ARRAY) {
        const float t = __ldg(a.t + c * a.t_stride + j);
        return t < 0.f ? 0.f : (t > ns ? ns : t);
    }
    if (TM == TM_UNIFORM) return ns * (a.n_t > 1 ? __fdiv_rn((float)j, (float)(a.n_t - 1)) : 0.f);
    return ns * hash_unit(lowbias32(kc ^ (uint32_t)j));
}

__device__ __forceinline__ int chain_segment(float t, int n_seg)
{
    int k = (int)floorf(t);  // NaN converts to 0; the NaN then flows through tau
    k = k < 0 ? 0 : k;
    return k > n_seg - 1 ? n_seg - 1 : k;
}

// segments staged as centred power coefficients (float4 each)
template <int VAR, int D, int DIM>
__host__ __device__ constexpr bool chain_coef() { return VAR == VAR_HORNER_CENTRED && (D == 2 || D == 3) && DIM == 3; }

// shared floats per warp for the staged chain (control points or coefficients)
template <int VAR, int D, int DIM>
__host__ __device__ inline int chain_stage_floats(int n_seg, int degree)
{
    return chain_coef<VAR, D, DIM>() ? n_seg * (D + 1) * 4 : (n_seg * degree + 1) * DIM;
}

template <int VAR, int D, int DIM, int TM, int OM>
__global__ void __launch_bounds__(kWarps * 32) k_chain(const CurveArgs a)
{
    using E = typename Pick<VAR, D, DIM>::type;
    constexpr int N = E::N;
    constexpr bool COEF = chain_coef<VAR, D, DIM>();
    extern __shared__ float s_dyn[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int deg = Deg<D>::get(a.degree);
    const int n_pts = a.n_seg * deg + 1;
    const int per = n_pts * DIM;
    const int held = chain_stage_floats<VAR, D, DIM>(a.n_seg, deg);
    float* my = s_dyn + wib * held;
    float* stage = s_dyn + kWarps * held + wib * 32 * DIM;
    const int64_t n_warps = (int64_t)gridDim.x * kWarps;

    for (int64_t c = (int64_t)blockIdx.x * kWarps + wib; c < a.n_curves; c += n_warps) {
        if constexpr (COEF) {
            // lane per segment: its centred power coefficients a_m, m = 0..D
            float4* my4 = reinterpret_cast<float4*>(my);
            for (int sg = lane; sg < a.n_seg; sg += 32) {
                float b[N][DIM];
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int q = 0; q < DIM; ++q) b[i][q] = load_elem(a.ctrl, a.dtype, c * per + (sg * D + i) * DIM + q);
                E e;
                e.setup(b, D);
#pragma unroll
                for (int m = 0; m < N; ++m) my4[sg * N + m] = make_float4(e.a[m][0], e.a[m][1], e.a[m][2], 0.f);
            }
        } else {
            for (int i = lane; i < per; i += 32) my[i] = load_elem(a.ctrl, a.dtype, c * per + i);
        }
        __syncwarp();
        const uint32_t kc = (TM == TM_HASH) ? lowbias32(a.key ^ (uint32_t)c) : 0u;
        const int n_t = a.n_t;
        auto point = [&](int j, float (&P)[DIM]) {
            const float t = chain_param<TM>(a, c, j, kc);
            const int k = chain_segment(t, a.n_seg);
            const float tau = t - (float)k;
            if constexpr (COEF) {
                const float4* sa = reinterpret_cast<const float4*>(my) + k * N;
                const float u = tau - 0.5f;
                float4 acc = sa[N - 1];
#pragma unroll
                for (int m = N - 2; m >= 0; --m) {
                    const float4 am = sa[m];
                    acc = make_float4(fmaf(acc.x, u, am.x), fmaf(acc.y, u, am.y), fmaf(acc.z, u, am.z), 0.f);
                }
                P[0] = acc.x;
                P[1] = acc.y;
                P[2] = acc.z;
            } else {
                float b[N][DIM];
                const float* src = my + k * deg * DIM;
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int q = 0; q < DIM; ++q) b[i][q] = (i <= deg) ? src[i * DIM + q] : 0.f;
                E e;
                e.setup(b, deg);
                e.eval(tau, P);
            }
        };
        if (OM == OM_POINTS) {
            for (int j0 = 0; j0 < n_t; j0 += 32) {
                const int j = j0 + lane;
                float P[DIM];
#pragma unroll
                for (int q = 0; q < DIM; ++q) P[q] = 0.f;
                if (j < n_t) point(j, P);
#pragma unroll
                for (int q = 0; q < DIM; ++q) stage[lane * DIM + q] = P[q];
                __syncwarp();
                const int valid = min(32, n_t - j0) * DIM;
                float* o = a.out + (c * n_t + j0) * DIM;
#pragma unroll
                for (int m = 0; m < DIM; ++m) {
                    const int idx = lane + 32 * m;
                    if (idx < valid) o[idx] = stage[idx];
                }
                __syncwarp();
            }
        } else {
            const int chunk = (n_t + 31) / 32;
            const int jb = lane * chunk;
            const int je = min(jb + chunk, n_t);
            float acc = 0.f;
            float first[DIM], prev[DIM];
#pragma unroll
            for (int q = 0; q < DIM; ++q) first[q] = prev[q] = 0.f;
            if (jb < je) {
                point(jb, first);
#pragma unroll
                for (int q = 0; q < DIM; ++q) prev[q] = first[q];
                for (int j = jb + 1; j < je; ++j) {
                    float P[DIM];
                    point(j, P);
                    acc += seg_len<DIM>(P, prev);
#pragma unroll
                    for (int q = 0; q < DIM; ++q) prev[q] = P[q];
                }
            }
            float pl[DIM];
#pragma unroll
            for (int q = 0; q < DIM; ++q) pl[q] = __shfl_up_sync(kFull, prev[q], 1);
            if (lane > 0 && jb < je) acc += seg_len<DIM>(first, pl);
            acc = warp_sum(acc);
            if (lane == 0) a.out[c] = acc;
        }
        __syncwarp();  // every lane is done with `my` before the next chain overwrites it
    }
}

// ---------------------------------------------------------------- replicated table

// At in-kernel draws the lanes of a warp read unrelated segments, and the staged
// chain's banks collide: 64 quadratic segments cost 31 shared-memory cycles per
// 32 points (l1tex 98 % busy).  Here a block holds 32 copies of the chain, word w
// of lane l's copy at w 32 + l, so that every lane reads a bank of its own: one
// cycle per word, whatever the segments.  One block takes a chain; its lanes walk
// runs of a multiple of 4 samples (lengths) or write tiles of 128 points a warp.
constexpr int kRepThreads = 512;
constexpr int kRepWarps = kRepThreads / 32;
constexpr int kRepTile = 128;
constexpr size_t kRepMaxSmem = 100 * 1024;  // two blocks per SM at least
// Draws per chain from which the copies pay: 64 segments break even at about 2800
// and 8 segments at 7300 (20,000 chains x 1024: 72 us with a warp per chain, 138
// with the copies; 2000 x 10,000 points 110 and 65).
constexpr int kRepMinSamples = 8192;

template <int VAR, int D, int DIM>
__host__ __device__ inline size_t chain_rep_smem(int n_seg, int om)
{
    const int held = chain_coef<VAR, D, DIM>() ? n_seg * (D + 1) * DIM : (n_seg * D + 1) * DIM;
    return ((size_t)held * 33 + 3 + (om == OM_POINTS ? kRepWarps * kRepTile * DIM : 0)) * sizeof(float);
}

template <int VAR, int D, int DIM, int TM, int OM>
__global__ void __launch_bounds__(kRepThreads, 2) k_chain_rep(const CurveArgs a)
{
    using E = Eval<VAR, D, DIM>;
    constexpr bool COEF = chain_coef<VAR, D, DIM>();
    extern __shared__ float4 s_rep4[];
    __shared__ float s_last[kRepWarps][DIM], s_sum[kRepWarps];
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int n_seg = a.n_seg;
    const int per = (n_seg * D + 1) * DIM;
    const int held = COEF ? n_seg * (D + 1) * DIM : per;
    float* stage = reinterpret_cast<float*>(s_rep4) + (OM == OM_POINTS ? wib * kRepTile * DIM : 0);
    float* rep = reinterpret_cast<float*>(s_rep4) + (OM == OM_POINTS ? kRepWarps * kRepTile * DIM : 0);
    float* plain = rep + held * 32;
    const float* mine = rep + lane;
    const uint32_t n_t = (uint32_t)a.n_t;
    for (int64_t c = blockIdx.x; c < a.n_curves; c += gridDim.x) {
        if constexpr (COEF) {
            for (int sg = tid; sg < n_seg; sg += kRepThreads) {
                float b[D + 1][DIM];
#pragma unroll
                for (int i = 0; i <= D; ++i)
#pragma unroll
                    for (int q = 0; q < DIM; ++q) b[i][q] = load_elem(a.ctrl, a.dtype, c * per + (sg * D + i) * DIM + q);
                E e;
                e.setup(b, D);
#pragma unroll
                for (int i = 0; i <= D; ++i)
#pragma unroll
                    for (int q = 0; q < DIM; ++q) plain[(sg * (D + 1) + i) * DIM + q] = e.a[i][q];
            }
        } else {
            for (int i = tid; i < per; i += kRepThreads) plain[i] = load_elem(a.ctrl, a.dtype, c * per + i);
        }
        __syncthreads();
        for (int w = wib; w < held; w += kRepWarps) rep[w * 32 + lane] = plain[w];
        __syncthreads();
        const uint32_t kc = curve_key<TM>(a, c);
        const float ns = (float)n_seg;
        auto point = [&](uint32_t j, float (&P)[DIM]) {
            float t;
            if (TM == TM_ARRAY || TM == TM_UNIFORM) t = chain_param<TM>(a, c, (int)j, kc);
            else t = ns * hash_unit(TM == TM_HASH16 ? lowbias32_premixed(kc, j) : lowbias32(kc ^ j));
            const int k = chain_segment(t, n_seg);
            const float tau = t - (float)k;
            const float* src = mine + k * ((COEF ? D + 1 : D) * DIM * 32);
            E e;
            if constexpr (COEF) {
                e.d = D;
#pragma unroll
                for (int i = 0; i <= D; ++i)
#pragma unroll
                    for (int q = 0; q < DIM; ++q) e.a[i][q] = src[(i * DIM + q) * 32];
            } else {
                float b[D + 1][DIM];
#pragma unroll
                for (int i = 0; i <= D; ++i)
#pragma unroll
                    for (int q = 0; q < DIM; ++q) b[i][q] = src[(i * DIM + q) * 32];
                e.setup(b, D);
            }
            e.eval(tau, P);
        };
        // two samples at once (lengths)
        auto point2 = [&](uint32_t ja, uint32_t jb, f32x2 (&P)[DIM]) {
            float tau[2];
            const float* src[2];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const uint32_t j = x == 0 ? ja : jb;
                const float t = ns * hash_unit(TM == TM_HASH16 ? lowbias32_premixed(kc, j) : lowbias32(kc ^ j));
                const int k = chain_segment(t, n_seg);
                tau[x] = t - (float)k;
                src[x] = mine + k * ((COEF ? D + 1 : D) * DIM * 32);
            }
            const f32x2 u = COEF ? pack2(tau[0] - 0.5f, tau[1] - 0.5f) : pack2(tau[0], tau[1]);
            const f32x2 minus = pack2(-tau[0], -tau[1]);
#pragma unroll
            for (int q = 0; q < DIM; ++q) {
                f32x2 w[D + 1];
#pragma unroll
                for (int i = 0; i <= D; ++i) w[i] = pack2(src[0][(i * DIM + q) * 32], src[1][(i * DIM + q) * 32]);
                if constexpr (COEF) {
                    P[q] = w[D];
#pragma unroll
                    for (int i = D - 1; i >= 0; --i) P[q] = fma2(P[q], u, w[i]);
                } else {
#pragma unroll
                    for (int r = 1; r <= D; ++r)
#pragma unroll
                        for (int i = 0; i <= D - r; ++i) w[i] = fma2(u, w[i + 1], fma2(minus, w[i], w[i]));
                    P[q] = w[0];
                }
            }
        };
        if (OM == OM_POINTS) {
            for (uint32_t j0 = wib * kRepTile; j0 < n_t; j0 += kRepThreads * (kRepTile / 32)) {
                const int cnt = (int)min((uint32_t)kRepTile, n_t - j0);
#pragma unroll
                for (int m = 0; m < kRepTile / 32; ++m) {
                    if (lane + 32 * m < cnt) {
                        float P[DIM];
                        point(j0 + lane + 32 * m, P);
#pragma unroll
                        for (int q = 0; q < DIM; ++q) stage[(lane + 32 * m) * DIM + q] = P[q];
                    }
                }
                __syncwarp();
                tile_copy(a.out + (c * (int64_t)n_t + j0) * DIM, stage, cnt * DIM, lane, 32);
                __syncwarp();
            }
        } else {
            // two half runs a lane, side by side in packed pairs (as packed_run)
            const uint32_t run = ((n_t + kRepThreads - 1) / kRepThreads + 7) & ~7u;
            const uint32_t jb = min(tid * run, n_t), jm = min(jb + run / 2, n_t), je = min(jb + run, n_t);
            const uint32_t both = min(jm - jb, je - jm);
            float acc = 0.f, first[DIM], mid[DIM], pa[DIM], prev[DIM];
#pragma unroll
            for (int q = 0; q < DIM; ++q) first[q] = mid[q] = pa[q] = prev[q] = 0.f;
            if (both > 0) {
                f32x2 acc2 = 0ull, prev2[DIM];
                point2(jb, jm, prev2);
#pragma unroll
                for (int q = 0; q < DIM; ++q) unpack2(prev2[q], first[q], mid[q]);
#pragma unroll 4
                for (uint32_t i = 1; i < both; ++i) {
                    f32x2 P[DIM], d2 = 0ull;
                    point2(jb + i, jm + i, P);
#pragma unroll
                    for (int q = 0; q < DIM; ++q) {
                        const f32x2 d = sub2(P[q], prev2[q]);
                        d2 = q == 0 ? mul2(d, d) : fma2(d, d, d2);
                        prev2[q] = P[q];
                    }
                    float qa, qb;
                    unpack2(d2, qa, qb);
                    acc2 = add2(acc2, pack2(sqrt_approx(qa), sqrt_approx(qb)));
                }
                float aa, ab;
                unpack2(acc2, aa, ab);
                acc = aa + ab;
#pragma unroll
                for (int q = 0; q < DIM; ++q) unpack2(prev2[q], pa[q], prev[q]);
            }
            // the first half is the longer one in the last run only
#pragma unroll 1
            for (uint32_t j = jb + both; j < jm; ++j) {
                float P[DIM];
                point(j, P);
                if (j == jb) {
#pragma unroll
                    for (int q = 0; q < DIM; ++q) first[q] = P[q];
                } else {
                    acc += seg_len<DIM>(P, pa);
                }
#pragma unroll
                for (int q = 0; q < DIM; ++q) pa[q] = P[q];
            }
            if (both > 0) {
                acc += seg_len<DIM>(mid, pa);
            } else {
#pragma unroll
                for (int q = 0; q < DIM; ++q) prev[q] = pa[q];
            }
            // the segments joining two runs: within the warp, then across warps
            if (lane == 31) {
#pragma unroll
                for (int q = 0; q < DIM; ++q) s_last[wib][q] = prev[q];
            }
            float pl[DIM];
#pragma unroll
            for (int q = 0; q < DIM; ++q) pl[q] = __shfl_up_sync(kFull, prev[q], 1);
            __syncthreads();
            if (lane == 0 && wib > 0) {
#pragma unroll
                for (int q = 0; q < DIM; ++q) pl[q] = s_last[wib - 1][q];
            }
            if (tid > 0 && jb < je) acc += seg_len<DIM>(first, pl);
            acc = warp_sum(acc);
            if (lane == 0) s_sum[wib] = acc;
            __syncthreads();
            if (wib == 0) {
                const float v = warp_sum(lane < kRepWarps ? s_sum[lane] : 0.f);
                if (lane == 0) a.out[c] = v;
            }
        }
        // the next chain's first barrier comes before its copies overwrite
        // these and after warp 0 has read s_sum
    }
}

template <int VAR, int D, int DIM, int TM, int OM>
LaunchResult launch_chain_rep(const CurveArgs& a, cudaStream_t s, const LaunchHooks& h)
{
    auto kern = k_chain_rep<VAR, D, DIM, TM, OM>;
    const size_t smem = chain_rep_smem<VAR, D, DIM>(a.n_seg, OM);
    // one limit for every launch of the kernel (calls on several threads)
    const cudaError_t e =
        cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRepMaxSmem);
    if (e != cudaSuccess) return {0, e};
    const int grid = persistent_grid((const void*)kern, kRepThreads, smem, h.sm_count, a.n_curves);
    h.count(h.self);
    h.begin(h.self, s);
    kern<<<grid, kRepThreads, smem, s>>>(a);
    const cudaError_t err = cudaGetLastError();
    h.end(h.self, s);
    return {1, err};
}

template <int VAR, int D, int DIM, int TM, int OM>
LaunchResult launch_chain_one(const CurveArgs& a, cudaStream_t s, const LaunchHooks& h)
{
    auto kern = k_chain<VAR, D, DIM, TM, OM>;
    const int held = chain_stage_floats<VAR, D, DIM>(a.n_seg, a.degree);
    const size_t smem = (size_t)kWarps * (held + 32 * DIM) * sizeof(float);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return {0, e};
    }
    const int grid = persistent_grid((const void*)kern, kWarps * 32, smem, h.sm_count, (a.n_curves + kWarps - 1) / kWarps);
    h.count(h.self);
    h.begin(h.self, s);
    kern<<<grid, kWarps * 32, smem, s>>>(a);
    cudaError_t err = cudaGetLastError();
    h.end(h.self, s);
    return {1, err};
}

template <int VAR, int D, int DIM>
LaunchResult launch_chain_modes(const CurveArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    // in-kernel draws, enough of them to pay for the copies, and a table that
    // leaves two blocks to an SM
    if constexpr (D > 0 && (VAR == VAR_DECASTELJAU || chain_coef<VAR, D, DIM>())) {
        // (lengths over at most 4 segments collide too little to gain: 75 us, 73 before)
        if (tm == TM_HASH && a.n_t >= kRepMinSamples && (a.n_seg > 4 || om == OM_POINTS) && chain_rep_smem<VAR, D, DIM>(a.n_seg, om) <= kRepMaxSmem) {
            if (om == OM_POINTS) return launch_chain_rep<VAR, D, DIM, TM_HASH, OM_POINTS>(a, s, h);
            if (a.n_t <= 65536) return launch_chain_rep<VAR, D, DIM, TM_HASH16, OM_LENGTH>(a, s, h);
            return launch_chain_rep<VAR, D, DIM, TM_HASH, OM_LENGTH>(a, s, h);
        }
    }
    if (om == OM_POINTS) {
        if (tm == TM_ARRAY) return launch_chain_one<VAR, D, DIM, TM_ARRAY, OM_POINTS>(a, s, h);
        if (tm == TM_UNIFORM) return launch_chain_one<VAR, D, DIM, TM_UNIFORM, OM_POINTS>(a, s, h);
        return launch_chain_one<VAR, D, DIM, TM_HASH, OM_POINTS>(a, s, h);
    }
    if (tm == TM_ARRAY) return launch_chain_one<VAR, D, DIM, TM_ARRAY, OM_LENGTH>(a, s, h);
    if (tm == TM_UNIFORM) return launch_chain_one<VAR, D, DIM, TM_UNIFORM, OM_LENGTH>(a, s, h);
    return launch_chain_one<VAR, D, DIM, TM_HASH, OM_LENGTH>(a, s, h);
}

// quadratic and cubic 2D and 3D chains get fixed-degree kernels, the rest the
// runtime-degree evaluator
template <int VAR>
LaunchResult launch_chain_variant(const CurveArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    if (a.dim == 3 && a.degree == 2) return launch_chain_modes<VAR, 2, 3>(a, tm, om, s, h);
    if (a.dim == 3 && a.degree == 3) return launch_chain_modes<VAR, 3, 3>(a, tm, om, s, h);
    if (a.dim == 2 && a.degree == 2) return launch_chain_modes<VAR, 2, 2>(a, tm, om, s, h);
    if (a.dim == 2 && a.degree == 3) return launch_chain_modes<VAR, 3, 2>(a, tm, om, s, h);
    switch (a.dim) {
    case 1: return launch_chain_modes<VAR, 0, 1>(a, tm, om, s, h);
    case 2: return launch_chain_modes<VAR, 0, 2>(a, tm, om, s, h);
    case 3: return launch_chain_modes<VAR, 0, 3>(a, tm, om, s, h);
    default: return launch_chain_modes<VAR, 0, 4>(a, tm, om, s, h);
    }
}

}  // namespace bez
