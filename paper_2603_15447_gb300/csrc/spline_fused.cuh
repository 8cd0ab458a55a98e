// spline_fused.cuh -- B-spline / NURBS evaluation in one kernel for degrees 1..5
// whose spans fit in shared memory: a block extracts the Bezier spans of a few
// curves into shared memory and evaluates their samples from there.
//
// GB300 runs FP64 at 1/64 of its FP32 rate, and the FP64 knot insertion of
// spline.cuh took 110 us for the 278,494 spans of 8191 cubic splines (FP64 pipe
// 87 % busy).  Here a span of a clamped uniform spline applies its operator,
// known to the compiler, as compensated FP32 dot products, and other spans run
// the same knot insertion in float-float arithmetic: unevaluated sums hi + lo of
// two floats, differences and products exact (Knuth's TwoSum, fma; Dekker 1971),
// about 46 significant bits.  Both round once to FP32 at the end, like the FP64
// form (errors against 64 bits unchanged: 4.7e-8, NURBS 7.2e-8).  A span that
// comes out infinite or NaN (values near the end of the FP32 range) is extracted
// again in FP64.
//
// Fusing the phases also drops the span buffer's trip through memory and one
// launch.  Blocks are small (128 threads, about as many spans), so that one
// block's extraction overlaps another's evaluation on an SM; the kernel is bound
// by instruction issue (74 %).  GB300, a call: 8191 cubic splines of 37 points x
// 256 133 -> 21 us, 4099 quadratic NURBS with their own knots x 200 56 -> 20 us,
// 65,536 quintics x 100 2178 -> 161 us, 30 cubics x 4096 114 -> 18 us.  Degrees
// 6, 7 and longer splines keep the two kernels of spline.cu.
#pragma once

#include "curve_eval.cuh"
#include "spline.cuh"

namespace bez {

constexpr int kFusedThreads = 128;
constexpr int kFusedWarps = kFusedThreads / 32;
constexpr int kFusedRun = 4;                     // samples of a lane per tile
constexpr int kFusedTile = 32 * kFusedRun;       // samples of a warp per tile
constexpr int kFusedMaxDegree = 5;
constexpr size_t kFusedMaxSmem = 40 * 1024;      // of a block: 5 resident blocks at worst

// ---------------------------------------------------------------- float-float

struct F2 {
    float h, l;
};

__device__ __forceinline__ F2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v))};
}

__device__ __forceinline__ F2 quick_sum(float a, float b)  // |a| >= |b| or a == 0
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// (x - y) / (z - w) for FP32 knots: exact differences, quotient and its
// residual divided once more
__device__ __forceinline__ F2 knot_ratio(float x, float y, float z, float w)
{
    const F2 n = two_sum(x, -y), d = two_sum(z, -w);
    const float q = __fdiv_rn(n.h, d.h);
    const float r = __fadd_rn(fmaf(-q, d.h, n.h), fmaf(-q, d.l, n.l));
    return quick_sum(q, __fdiv_rn(r, d.h));
}

// a + t (b - a)
__device__ __forceinline__ F2 lerp2(F2 a, F2 b, F2 t)
{
    F2 d = two_sum(b.h, -a.h);
    d.l = __fadd_rn(d.l, __fsub_rn(b.l, a.l));
    const float p = __fmul_rn(t.h, d.h);
    const float pe = fmaf(t.h, d.l, fmaf(t.l, d.h, fmaf(t.h, d.h, -p)));
    F2 s = two_sum(a.h, p);
    s.l = __fadd_rn(s.l, __fadd_rn(a.l, pe));
    return quick_sum(s.h, s.l);
}

// ---------------------------------------------------------------- extraction

// Bezier points of one span from its P + 1 de Boor points (rows of `ctrl`,
// weights `w` or NULL) and local knots s[1..2P]; false when a result is not
// finite.  The weights of the insertion steps are formed once and serve every
// component.
template <int P>
__device__ __forceinline__ bool extract_span_f2(const float* ctrl, const float* w, int dim, const float (&s)[2 * P + 1],
                                                float* out)
{
    const int comps = w ? dim + 1 : dim;
    constexpr int STEPS = P > 1 ? P * (P + 1) / 2 - 1 : 1;  // of either pass
    F2 al[STEPS], be[STEPS];
    // steps of weight 1 (b is already an argument: clamped ends, repeated knots)
    // keep their point as the FP64 form does: they carry the weight 2.  a + 1 (b - a)
    // would lose a homogeneous or inserted point beside one 2^20 times its size.
    // (Weight 0 returns a as it is.)
    {
        const float a = s[P], b = s[P + 1];
        int k = 0;
#pragma unroll
        for (int l = 1; l <= P - 1; ++l)
#pragma unroll
            for (int i = 0; i <= P - l; ++i) al[k++] = knot_ratio(a, s[i + l], s[P + i + 1], s[i + l]);
        k = 0;
#pragma unroll
        for (int l = 1; l <= P - 1; ++l)
#pragma unroll
            for (int i = P; i >= l; --i, ++k) {
                be[k] = knot_ratio(b, a, s[P + i - l + 1], a);
                if (s[P + i - l + 1] == b) be[k].h = 2.f;
            }
    }
    bool fine = true;
#pragma unroll 1
    for (int q = 0; q < comps; ++q) {
        F2 Q[P + 1];
#pragma unroll
        for (int i = 0; i <= P; ++i) {
            const float x = q < dim ? ctrl[i * dim + q] : 1.f;
            Q[i] = {x, 0.f};
            if (w) {
                Q[i].h = __fmul_rn(w[i], x);
                Q[i].l = fmaf(w[i], x, -Q[i].h);
            }
        }
        int k = 0;
#pragma unroll
        for (int l = 1; l <= P - 1; ++l)
#pragma unroll
            for (int i = 0; i <= P - l; ++i, ++k) Q[i] = lerp2(Q[i], Q[i + 1], al[k]);
        k = 0;
#pragma unroll
        for (int l = 1; l <= P - 1; ++l)
#pragma unroll
            for (int i = P; i >= l; --i, ++k) {
                const F2 v = lerp2(Q[i - 1], Q[i], be[k]);
                Q[i] = be[k].h > 1.5f ? Q[i] : v;
            }
#pragma unroll
        for (int i = 0; i <= P; ++i) {
            const float v = __fadd_rn(Q[i].h, Q[i].l);
            fine = fine && isfinite(v);
            out[i * comps + q] = v;
        }
    }
    return fine;
}

// Extraction operator of span e = 0 .. P - 1 of a clamped uniform spline of at
// least 2P - 1 spans: its local knots in units of the knot distance are
// s_j = max(0, e - P + j), whole numbers that do not depend on the spline's
// length; e = P - 1 is every interior span, and the last P - 1 spans are the
// first ones mirrored.  Knot insertion on unit vectors, by the compiler.
template <int P>
struct UniformOp {
    float h[P + 1][P + 1], l[P + 1][P + 1];
};
template <int P>
constexpr UniformOp<P> make_uniform_op(int e)
{
    double Q[P + 1][P + 1] = {};
    for (int i = 0; i <= P; ++i) Q[i][i] = 1.0;
    double s[2 * P + 1] = {};
    for (int j = 1; j <= 2 * P; ++j) s[j] = e - P + j > 0 ? e - P + j : 0;
    const double a = s[P], b = s[P + 1];
    for (int l = 1; l <= P - 1; ++l)
        for (int i = 0; i <= P - l; ++i) {
            const double t = (a - s[i + l]) / (s[P + i + 1] - s[i + l]);
            for (int j = 0; j <= P; ++j) Q[i][j] += t * (Q[i + 1][j] - Q[i][j]);
        }
    for (int l = 1; l <= P - 1; ++l)
        for (int i = P; i >= l; --i) {
            const double t = (b - a) / (s[P + i - l + 1] - a);
            for (int j = 0; j <= P; ++j) Q[i][j] = Q[i - 1][j] + t * (Q[i][j] - Q[i - 1][j]);
        }
    UniformOp<P> r{};
    for (int i = 0; i <= P; ++i)
        for (int j = 0; j <= P; ++j) {
            r.h[i][j] = (float)Q[i][j];
            r.l[i][j] = (float)(Q[i][j] - (double)r.h[i][j]);
        }
    return r;
}
template <int P>
struct EdgeOps {
    UniformOp<P> e[P > 1 ? P - 1 : 1];
};
template <int P>
constexpr EdgeOps<P> make_edge_ops()
{
    EdgeOps<P> r{};
    for (int e = 0; e < P - 1; ++e) r.e[e] = make_uniform_op<P>(e);
    return r;
}
template <int P>
static __device__ const EdgeOps<P> kEdgeOps = make_edge_ops<P>();

// The span points of such a span: each a compensated dot product (Dot2: Ogita,
// Rump & Oishi 2005) of an operator row hi + lo with the de Boor points -- for
// an interior cubic span 10 products of 11 instructions a component, operands
// immediate, instead of 10 insertion steps of 23 and their weights.  Edge
// spans read their operator (edge e, points and rows in reverse order at the
// curve's end).
template <int P, int C, bool RAT, bool INNER>
__device__ __forceinline__ bool extract_uniform(const float* ctrl, const float* w, int e, bool reverse, float* out)
{
    constexpr UniformOp<P> inner = make_uniform_op<P>(P - 1);
    constexpr int DIM = RAT ? C - 1 : C;
    const UniformOp<P>& edge = kEdgeOps<P>.e[INNER ? 0 : e];
    float pts[kSpanStride(P, C)];
    bool fine = true;
#pragma unroll
    for (int i = (P + 1) * C; i < kSpanStride(P, C); ++i) pts[i] = 0.f;
#pragma unroll
    for (int q = 0; q < C; ++q) {
        F2 x[P + 1];
#pragma unroll
        for (int j = 0; j <= P; ++j) {
            const int r = !INNER && reverse ? P - j : j;
            x[j] = {q < DIM ? ctrl[r * DIM + q] : 1.f, 0.f};
            if (RAT) {
                const float v = x[j].h;
                x[j].h = __fmul_rn(w[r], v);
                x[j].l = q < DIM ? fmaf(w[r], v, -x[j].h) : 0.f;
            }
        }
#pragma unroll
        for (int i = 0; i <= P; ++i) {
            float sh = 0.f, corr = 0.f;
            bool first = true;
#pragma unroll
            for (int j = 0; j <= P; ++j) {
                if (INNER && inner.h[i][j] == 0.f) continue;
                const float mh = INNER ? inner.h[i][j] : __ldg(&edge.h[i][j]);
                const float ml = INNER ? inner.l[i][j] : __ldg(&edge.l[i][j]);
                const float pr = __fmul_rn(mh, x[j].h);
                float er = fmaf(mh, x[j].h, -pr);
                if (RAT && q < DIM) er = fmaf(mh, x[j].l, er);
                if (!INNER || inner.l[i][j] != 0.f) er = fmaf(ml, x[j].h, er);
                if (first) {
                    sh = pr;
                    corr = er;
                } else {
                    const F2 t = two_sum(sh, pr);
                    sh = t.h;
                    corr = __fadd_rn(corr, __fadd_rn(t.l, er));
                }
                first = false;
            }
            const float v = __fadd_rn(sh, corr);
            fine = fine && isfinite(v);
            pts[i * C + q] = v;
        }
    }
    if (!INNER && reverse) {
#pragma unroll
        for (int i = 0; i < (P + 1) / 2; ++i)
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const float v = pts[i * C + q];
                pts[i * C + q] = pts[(P - i) * C + q];
                pts[(P - i) * C + q] = v;
            }
    }
#pragma unroll
    for (int k = 0; k < kSpanStride(P, C) / 4; ++k)
        reinterpret_cast<float4*>(out)[k] = make_float4(pts[4 * k], pts[4 * k + 1], pts[4 * k + 2], pts[4 * k + 3]);
    return fine;
}

// out of line: taken by spans with infinite or NaN values only
static __device__ __noinline__ void extract_span_again(const float* ctrl, const float* w, const float* knots, int n, int p,
                                                int dim, int k, float* out)
{
    extract_span(ctrl, w, knots, n, p, dim, k, out);
}

// ---------------------------------------------------------------- kernel

// Shared memory of a block of CB curves, in floats: control points and weights
// (FP32, as given), knots, spans, and one staging tile per warp.
struct FusedLayout {
    int ctrl, weights, knots, spans, total;
};
__host__ __device__ inline FusedLayout fused_layout(int cb, int n_ctrl, int p, int dim, bool rat, bool knots)
{
    FusedLayout f;
    const int comps = rat ? dim + 1 : dim;
    f.ctrl = kFusedWarps * kFusedTile * dim;  // after the tiles, which are float4-aligned
    f.weights = f.ctrl + cb * n_ctrl * dim;
    f.knots = f.weights + (rat ? cb * n_ctrl : 0);
    f.spans = f.knots + (knots ? cb * (n_ctrl + p + 1) : 0);
    f.spans = (f.spans + 3) & ~3;  // spans are read as float4s
    f.total = f.spans + cb * (n_ctrl - p) * kSpanStride(p, comps);
    return f;
}

// One curve of the block as the evaluation sees it.
struct FusedCurve {
    const float* spans;
    const float* breaks;  // U_p .. U_n in shared memory, or NULL (clamped uniform)
    int ns;
    float lo, hi;
};

// parameters of samples j + i step (i < N), of which those below je exist
template <int N>
__device__ __forceinline__ void fused_params(const FusedCurve& c, const GridDiv& grid, int tm, const float* t,
                                             uint32_t key, uint32_t j, uint32_t step, uint32_t je, float (&v)[N])
{
    if (tm == TM_ARRAY) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = j + i * step < je ? __ldg(t + (j + i * step)) : 0.f;
#pragma unroll
        for (int i = 0; i < N; ++i)
            v[i] = !c.breaks ? clamp01(v[i]) : v[i] < c.lo ? c.lo : (v[i] > c.hi ? c.hi : v[i]);
        return;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t ji = j + i * step;
        const float u = tm == TM_UNIFORM ? grid((int)ji) : hash_unit(lowbias32(key ^ ji));
        v[i] = c.breaks ? fmaf(c.hi - c.lo, u, c.lo) : u;
    }
}

template <int P, int DIM, bool RAT>
__device__ __forceinline__ void fused_point(const SplineArgs& a, const FusedCurve& c, float t, float (&out)[DIM])
{
    constexpr int C = RAT ? DIM + 1 : DIM;
    float tau;
    int s;
    if (!c.breaks) {
        s = uniform_span(t, c.ns, tau);
    } else {
        int lo = 0, hi = c.ns;  // count of breaks[i] <= t over i < ns, by bisection
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (c.breaks[mid] <= t) lo = mid + 1;
            else hi = mid;
        }
        s = lo > 0 ? lo - 1 : 0;
        const float b0 = c.breaks[s], b1 = c.breaks[s + 1];
        tau = (t - b0) / (b1 - b0);
    }
    constexpr int S4 = kSpanStride(P, C) / 4;
    const float4* src = reinterpret_cast<const float4*>(c.spans + s * 4 * S4);
    float q[4 * S4], v[C];
#pragma unroll
    for (int m = 0; m < S4; ++m) {
        const float4 x = src[m];
        q[4 * m] = x.x;
        q[4 * m + 1] = x.y;
        q[4 * m + 2] = x.z;
        q[4 * m + 3] = x.w;
    }
    span_point_fixed<P, C, RAT>(q, tau, v);
    if (RAT && v[C - 1] == 0.f && a.err_word) atomicAdd(a.err_word, 1);
#pragma unroll
    for (int k = 0; k < DIM; ++k) out[k] = v[k];
}

// cb curves per block; for points, the samples of a block's curves may be cut
// into `parts` ranges of part_len samples, one block each (cb is 1 then).
template <int P, int DIM, bool RAT>
__global__ void __launch_bounds__(kFusedThreads) k_spline_fused(const SplineArgs a, int tm, int om, int cb, int parts,
                                                                uint32_t part_len)
{
    constexpr int C = RAT ? DIM + 1 : DIM;
    extern __shared__ float4 s_fused[];
    float* sm = reinterpret_cast<float*>(s_fused);
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int n = a.n_ctrl, ns = a.n_spans;
    const FusedLayout f = fused_layout(cb, n, P, DIM, RAT, a.knots != nullptr);
    const int64_t blk = parts > 1 ? blockIdx.x / parts : blockIdx.x;
    const int64_t c0 = blk * cb;
    const int nc = (int)min((int64_t)cb, a.n_curves - c0);
    for (int i = tid; i < nc * n * DIM; i += kFusedThreads) sm[f.ctrl + i] = __ldg(a.ctrl + c0 * n * DIM + i);
    if (RAT)
        for (int i = tid; i < nc * n; i += kFusedThreads) sm[f.weights + i] = __ldg(a.weights + c0 * n + i);
    if (a.knots)
        for (int i = tid; i < nc * (n + P + 1); i += kFusedThreads)
            sm[f.knots + i] = __ldg(a.knots + c0 * (n + P + 1) + i);
    __syncthreads();
    // interior spans of clamped uniform curves first, then the others, so that
    // few warps run both kinds
    const bool tabled = !a.knots && ns >= 2 * P - 1;
    const int ni = tabled ? ns - 2 * (P - 1) : 0, no = ns - ni;
    for (int item = tid; item < nc * ns; item += kFusedThreads) {
        const bool inner = item < nc * ni;
        const int r = inner ? item : item - nc * ni;
        const int cc = r / (inner ? ni : no);
        int s0 = r - cc * (inner ? ni : no);  // span [U_k, U_(k+1)), k = s0 + P
        if (inner) s0 += P - 1;
        else if (tabled && s0 >= P - 1) s0 += ni;
        const int k = s0 + P;
        const float* ctrl = sm + f.ctrl + (cc * n + s0) * DIM;
        const float* w = RAT ? sm + f.weights + cc * n + s0 : nullptr;
        const float* U = a.knots ? sm + f.knots + cc * (n + P + 1) : nullptr;
        float* out = sm + f.spans + (cc * ns + s0) * kSpanStride(P, C);
        bool fine;
        if (inner) {
            fine = extract_uniform<P, C, RAT, true>(ctrl, w, 0, false, out);
        } else if (tabled) {
            const bool end = s0 >= P - 1;
            fine = extract_uniform<P, C, RAT, false>(ctrl, w, end ? ns - 1 - s0 : s0, end, out);
        } else {
            float s[2 * P + 1];
            s[0] = 0.f;
#pragma unroll
            for (int j = 1; j <= 2 * P; ++j)
                // clamped uniform knots times the span count: whole numbers, same ratios
                s[j] = U ? U[k - P + j] : (float)min(max(k - 2 * P + j, 0), ns);
            if (s[P] < s[P + 1]) {
                fine = extract_span_f2<P>(ctrl, w, DIM, s, out);
            } else {
                fine = true;
#pragma unroll 1
                for (int i = 0; i < (P + 1) * C; ++i) out[i] = 0.f;
            }
        }
        if (!fine)
            extract_span_again(sm + f.ctrl + cc * n * DIM, RAT ? sm + f.weights + cc * n : nullptr, U, n, P, DIM, k,
                               out);
    }
    __syncthreads();

    GridDiv grid;
    grid.init(a.n_t);
    const uint32_t n_t = (uint32_t)a.n_t;
    auto curve = [&](int cc) {
        FusedCurve c;
        c.spans = sm + f.spans + cc * ns * kSpanStride(P, C);
        c.ns = ns;
        c.breaks = a.knots ? sm + f.knots + cc * (n + P + 1) + P : nullptr;
        c.lo = a.knots ? c.breaks[0] : 0.f;
        c.hi = a.knots ? c.breaks[ns] : 1.f;
        return c;
    };
    if (om == OM_POINTS) {
        // units of one warp: a tile of one curve's samples
        const uint32_t j_lo = parts > 1 ? (uint32_t)(blockIdx.x - blk * parts) * part_len : 0u;
        const uint32_t j_hi = parts > 1 ? min(n_t, j_lo + part_len) : n_t;
        const uint32_t tiles = (j_hi - j_lo + kFusedTile - 1) / kFusedTile;
        float* stage = sm + wib * kFusedTile * DIM;
        int cc = 0;
        uint32_t tile = wib;
        for (;;) {
            while (tile >= tiles && cc < nc) {
                tile -= tiles;
                ++cc;
            }
            if (cc >= nc) break;
            const FusedCurve c = curve(cc);
            const uint32_t j0 = j_lo + tile * kFusedTile;
            const int cnt = (int)min((uint32_t)kFusedTile, j_hi - j0);
            float t[kFusedRun];
            fused_params(c, grid, tm, a.t + (c0 + cc) * a.t_stride, lowbias32(a.key ^ (uint32_t)(c0 + cc)), j0 + lane,
                         32u, j_hi, t);
#pragma unroll
            for (int m = 0; m < kFusedRun; ++m) {
                if (32 * m >= cnt) break;
                if (lane + 32 * m < cnt) {
                    float P_[DIM];
                    fused_point<P, DIM, RAT>(a, c, t[m], P_);
#pragma unroll
                    for (int k = 0; k < DIM; ++k) stage[(lane + 32 * m) * DIM + k] = P_[k];
                }
            }
            __syncwarp();
            float* o = a.out + ((c0 + cc) * (int64_t)n_t + j0) * DIM;
            const int valid = cnt * DIM;
            int e = lane;
            if ((reinterpret_cast<uintptr_t>(o) & 15) == 0) {
                for (int q = lane; q < valid / 4; q += 32)
                    reinterpret_cast<float4*>(o)[q] = reinterpret_cast<const float4*>(stage)[q];
                e = (valid & ~3) + lane;
            }
            for (; e < valid; e += 32) o[e] = stage[e];
            __syncwarp();
            tile += kFusedWarps;
        }
    } else {
        // a warp per curve, each lane a contiguous run; one shuffle joins runs
        for (int cc = wib; cc < nc; cc += kFusedWarps) {
            const FusedCurve c = curve(cc);
            const uint32_t run = (n_t + 31) / 32;
            const uint32_t jb = min(lane * run, n_t), je = min(jb + run, n_t);
            float acc = 0.f, first[DIM], prev[DIM];
#pragma unroll
            for (int k = 0; k < DIM; ++k) first[k] = prev[k] = 0.f;
            const float* tc = a.t + (c0 + cc) * a.t_stride;
            const uint32_t key = lowbias32(a.key ^ (uint32_t)(c0 + cc));
            for (uint32_t j = jb; j < je; ++j) {
                float P_[DIM], t[1];
                fused_params(c, grid, tm, tc, key, j, 1u, je, t);
                fused_point<P, DIM, RAT>(a, c, t[0], P_);
                if (j == jb) {
#pragma unroll
                    for (int k = 0; k < DIM; ++k) first[k] = P_[k];
                } else {
                    acc += seg_len<DIM>(P_, prev);
                }
#pragma unroll
                for (int k = 0; k < DIM; ++k) prev[k] = P_[k];
            }
            float pl[DIM];
#pragma unroll
            for (int k = 0; k < DIM; ++k) pl[k] = __shfl_up_sync(kFull, prev[k], 1);
            if (lane > 0 && jb < je) acc += seg_len<DIM>(first, pl);
            acc = warp_sum(acc);
            if (lane == 0) a.out[c0 + cc] = acc;
        }
    }
}

// the kernels of degrees 4 and 5 (spline_fused_high.cu)
const void* fused_kernel_high(int degree, int dim, bool rat);

template <int P>
static const void* fused_kernel(int dim, bool rat)
{
    switch (dim) {
    case 1: return rat ? (const void*)k_spline_fused<P, 1, true> : (const void*)k_spline_fused<P, 1, false>;
    case 2: return rat ? (const void*)k_spline_fused<P, 2, true> : (const void*)k_spline_fused<P, 2, false>;
    case 3: return rat ? (const void*)k_spline_fused<P, 3, true> : (const void*)k_spline_fused<P, 3, false>;
    default: return rat ? (const void*)k_spline_fused<P, 4, true> : (const void*)k_spline_fused<P, 4, false>;
    }
}

}  // namespace bez
