// curve_tile.cuh -- the general register kernels for single curves of fixed
// degree (1..7) and any dimension: points (k_points; k_points_few for small
// calls) and polyline lengths (k_length), several curves per warp, and the fused
// draw-and-measure form of centred Horner in packed FP32 pairs.
//
// The parameter kind (array, uniform grid, draw) is a launch argument: a lane
// fetches the parameters of four samples behind one uniform branch, so one
// kernel per (evaluator, degree, dimension) serves all of them.
#pragma once

#include "curve_eval.cuh"

namespace bez {

constexpr int kTileSamples = 256;  // samples a warp evaluates between two write-outs
constexpr int kTileMaxRun = 8;     // of one lane: kTileSamples / 32

// T_d of make_centred_tables in FP32 (exact: small integers over powers of
// two), rows of 8 read by lanes that each form one coefficient.
struct CentredRows {
    float t[8][8][8];
};
constexpr CentredRows make_centred_rows()
{
    CentredRows r{};
    const CentredTables d = make_centred_tables();
    for (int p = 0; p < 8; ++p)
        for (int m = 0; m < 8; ++m)
            for (int i = 0; i < 8; ++i) r.t[p][m][i] = (float)d.t[p][m][i];
    return r;
}
static __device__ const CentredRows kCentredRows = make_centred_rows();

// Coefficient m about t = 1/2 of one component of a degree-D curve (b strided
// by `stride`).  Plain FP32 up to degree 4; from degree 5 the compensated dot
// product of Ogita, Rump & Oishi (Dot2, 2005: products split exactly by fma,
// partial sums by Knuth's TwoSum), which is as accurate as summing in twice
// the precision and rounding once, at FP32 rate (FP64 runs at 1/64 of it).  A sum
// comes out infinite or NaN where a term leaves the FP32 range.
template <int D>
__device__ __forceinline__ float centred_entry(const float* b, int stride, int m)
{
    const float* T = kCentredRows.t[D][m];
    if constexpr (D < kFp64SetupCentred) {
        float acc = 0.f;
#pragma unroll
        for (int i = 0; i <= D; ++i) acc = fmaf(__ldg(T + i), b[i * stride], acc);
        return acc;
    } else {
        float sh = 0.f, corr = 0.f;
#pragma unroll
        for (int i = 0; i <= D; ++i) {
            const float w = __ldg(T + i), x = b[i * stride];
            const float pr = __fmul_rn(w, x);
            const float e = fmaf(w, x, -pr);
            const float s = __fadd_rn(sh, pr);
            const float bv = __fsub_rn(s, sh);
            const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bv)), __fsub_rn(pr, bv));
            sh = s;
            corr = __fadd_rn(corr, __fadd_rn(err, e));
        }
        return __fadd_rn(sh, corr);
    }
}

// Shared memory of one warp: the tile's points in output order (the control
// points before them), and the power coefficients of the warp's curves.
template <int D, int DIM, int FLOATS>
struct TileSmem {
    static constexpr int PER = (D + 1) * DIM;
    static constexpr int kMaxCurves = 8;
    alignas(16) float stage[FLOATS];
    alignas(16) float coef[kMaxCurves * PER];
    static_assert(FLOATS >= kMaxCurves * PER, "the stage holds the control points of the warp's curves");
};

// The evaluator of this lane's curve (group `grp` of the nc curves from c0
// on).  Control points load coalesced; the centred power basis is formed
// cooperatively, one coefficient per lane, and read back by every lane.
template <int VAR, int D, int DIM, int FLOATS>
__device__ __forceinline__ void tile_setup(const CurveArgs& a, TileSmem<D, DIM, FLOATS>& sm, int64_t c0, int nc,
                                           int grp, int lane, Eval<VAR, D, DIM>& e)
{
    constexpr int PER = (D + 1) * DIM;
    if (a.dtype == 0) {
        const float* src = static_cast<const float*>(a.ctrl) + c0 * PER;
        for (int i = lane; i < nc * PER; i += 32) sm.stage[i] = __ldg(src + i);
    } else {
        for (int i = lane; i < nc * PER; i += 32) sm.stage[i] = load_elem(a.ctrl, a.dtype, c0 * PER + i);
    }
    __syncwarp();
    const int g = grp < nc ? grp : nc - 1;  // lanes without a curve follow the last one
    if constexpr (VAR == VAR_HORNER_CENTRED) {
        bool fine = true;
        for (int i = lane; i < nc * PER; i += 32) {
            const int cc = i / PER, r = i - cc * PER, m = r / DIM, k = r - m * DIM;
            const float v = centred_entry<D>(sm.stage + cc * PER + k, DIM, m);
            if (D >= kFp64SetupCentred) fine = fine && isfinite(v);
            sm.coef[i] = v;
        }
        if (D >= kFp64SetupCentred && __any_sync(kFull, !fine)) {
            // terms are up to 35 times a point and cancel: such a coefficient again in FP64
#pragma unroll 1
            for (int i = lane; i < nc * PER; i += 32) {
                const int cc = i / PER, r = i - cc * PER, m = r / DIM, k = r - m * DIM;
                double acc = 0.0;
#pragma unroll 1
                for (int j = 0; j <= D; ++j)
                    acc = fma((double)__ldg(&kCentredRows.t[D][m][j]), (double)sm.stage[cc * PER + j * DIM + k], acc);
                if (!isfinite(sm.coef[i])) sm.coef[i] = (float)acc;
            }
        }
        __syncwarp();
        e.d = D;
        if constexpr (PER % 4 == 0) {  // whole float4s, on 16-byte boundaries
#pragma unroll
            for (int q = 0; q < PER / 4; ++q) {
                const float4 v = reinterpret_cast<const float4*>(sm.coef + g * PER)[q];
                const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) e.a[(4 * q + r) / DIM][(4 * q + r) % DIM] = x[r];
            }
        } else {
#pragma unroll
            for (int i = 0; i <= D; ++i)
#pragma unroll
                for (int k = 0; k < DIM; ++k) e.a[i][k] = sm.coef[g * PER + i * DIM + k];
        }
    } else {
        float b[D + 1][DIM];
#pragma unroll
        for (int i = 0; i <= D; ++i)
#pragma unroll
            for (int k = 0; k < DIM; ++k) b[i][k] = sm.stage[g * PER + i * DIM + k];
        e.setup(b, D);
    }
    __syncwarp();
}

// How a launch's parameters are made: the kernel kind, the grid's division
// and the curve's draw key.
struct TileParams {
    GridDiv grid;
    uint32_t key;
    const float* t;
    __device__ __forceinline__ void curve(const CurveArgs& a, int tm, int64_t c)
    {
        key = tm == TM_HASH ? curve_key<TM_HASH>(a, c) : tm == TM_HASH16 ? curve_key<TM_HASH16>(a, c) : 0u;
        t = a.t + c * a.t_stride;
    }
    // t[i] = parameter of sample j0 + i step for i < N; array elements from
    // index je on are not read (ALL: every index is below je)
    template <int N, bool ALL = false>
    __device__ __forceinline__ void get(int tm, uint32_t j0, uint32_t step, uint32_t je, float (&v)[N]) const
    {
        if (tm == TM_ARRAY) {
#pragma unroll
            for (int i = 0; i < N; ++i)
                v[i] = ALL || j0 + i * step < je ? clamp01(__ldg(t + (j0 + i * step))) : 0.f;
        } else if (tm == TM_UNIFORM) {
#pragma unroll
            for (int i = 0; i < N; ++i) v[i] = grid((int)(j0 + i * step));
        } else if (tm == TM_HASH16) {
#pragma unroll
            for (int i = 0; i < N; ++i) v[i] = hash_unit(lowbias32_premixed(key, j0 + i * step));
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) v[i] = hash_unit(lowbias32(key ^ (j0 + i * step)));
        }
    }
};

// `n` staged floats to consecutive addresses by `lanes` lanes (this one is
// `lane` of them), as float4s where the destination starts on a 16-byte
// boundary (the stage's parts do where it does: both advance alike).
__device__ __forceinline__ void tile_copy(float* o, const float* src, int n, int lane, int lanes)
{
    int f = lane;
    if (((reinterpret_cast<uintptr_t>(o) | reinterpret_cast<uintptr_t>(src)) & 15) == 0) {
#pragma unroll 2
        for (int q = lane; q < n / 4; q += lanes)
            reinterpret_cast<float4*>(o)[q] = reinterpret_cast<const float4*>(src)[q];
        f = (n & ~3) + lane;
    }
    for (; f < n; f += lanes) o[f] = src[f];
}

// The samples of one lane in a tile, G apart, into their staged positions:
// sample m exists while m G < left.  All parameter loads go out together.
template <int VAR, int D, int DIM, bool ALL>
__device__ __forceinline__ void tile_points(const Eval<VAR, D, DIM>& e, const TileParams& tp, int tm, uint32_t j,
                                            int G, uint32_t jend, float* mine, int left)
{
    float t[kTileMaxRun];
    tp.get<kTileMaxRun, ALL>(tm, j, G, jend, t);
#pragma unroll
    for (int m = 0; m < kTileMaxRun; ++m) {
        if (ALL || m * G < left) {
            float P[DIM];
            e.eval(t[m], P);
#pragma unroll
            for (int k = 0; k < DIM; ++k) mine[m * G * DIM + k] = P[k];
        }
    }
}

// Points.  2^lg lanes take a curve, so a warp takes 32 >> lg consecutive
// curves, and a lane eight samples of its curve per tile.  Where the curves
// are few, one warp takes a curve (lg = 5) and it may be cut into `parts`
// ranges of part_len samples (a multiple of the tile), one unit of work each.
// A tile is staged in output order: one contiguous stretch of the output when
// it holds whole curves, one per curve otherwise.
template <int VAR, int D, int DIM>
__global__ void __launch_bounds__(kWarps * 32, (D + 1) * DIM > 20 ? 3 : (D + 1) * DIM > 12 ? 4 : 5)
    k_points(const CurveArgs a, int tm, int lg, int parts, int part_len)
{
    using Smem = TileSmem<D, DIM, (kTileSamples + 32) * DIM>;
    __shared__ Smem s_tile[kWarps];
    const int lane = threadIdx.x & 31;
    Smem& sm = s_tile[threadIdx.x >> 5];
    const int G = 1 << lg, cpw = 32 >> lg, grp = lane >> lg, li = lane & (G - 1);
    const uint32_t n_t = (uint32_t)a.n_t;  // unsigned: an index may step past 2^31 - 1
    const int64_t n_units = parts > 1 ? a.n_curves * parts : (a.n_curves + cpw - 1) / cpw;
    const int64_t n_warps = (int64_t)gridDim.x * kWarps;
    TileParams tp;
    tp.grid.init(a.n_t);
    for (int64_t u = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5); u < n_units; u += n_warps) {
        const int64_t c0 = parts > 1 ? u / parts : u * cpw;
        const uint32_t jb = parts > 1 ? (uint32_t)(u - c0 * parts) * (uint32_t)part_len : 0u;
        const uint32_t jend = parts > 1 ? min(n_t, jb + (uint32_t)part_len) : n_t;
        const int nc = (int)min((int64_t)cpw, a.n_curves - c0);
        Eval<VAR, D, DIM> e;
        tile_setup<VAR>(a, sm, c0, nc, grp, lane, e);
        const bool live = grp < nc;
        tp.curve(a, tm, c0 + (live ? grp : 0));
        for (uint32_t j0 = jb; j0 < jend; j0 += kTileMaxRun * G) {
            const int ns = (int)min((uint32_t)(kTileMaxRun * G), jend - j0);  // samples of each curve in this tile
            // curves end to end, or on strides that keep the groups' stores in
            // different banks (row lengths that are a multiple of 32 floats
            // would put them all in the same ones)
            const bool apart = lg < 5 && ((uint32_t)ns != n_t || (ns * DIM & 31) == 0);
            float* seg = sm.stage + grp * (ns + (apart ? G : 0)) * DIM;
            float* mine = seg + li * DIM;
            // a whole tile tests no sample (lanes without a curve stage values that are not copied)
            if (ns == kTileMaxRun * G) tile_points<VAR, D, DIM, true>(e, tp, tm, j0 + li, G, jend, mine, 0);
            else tile_points<VAR, D, DIM, false>(e, tp, tm, j0 + li, G, jend, mine, live ? ns - li : 0);
            __syncwarp();
            float* o = a.out + (c0 * (int64_t)n_t + j0) * DIM;
            if (!apart) tile_copy(o, sm.stage, nc * ns * DIM, lane, 32);
            else if (live) tile_copy(o + grp * (int64_t)n_t * DIM, seg, ns * DIM, li, G);
            __syncwarp();
        }
    }
}

// The evaluator of one curve from its control points in registers, with
// tile_setup's arithmetic (centred Horner: below degree 5).
template <int VAR, int D, int DIM>
__device__ __forceinline__ void register_setup(const float (&b)[D + 1][DIM], Eval<VAR, D, DIM>& e)
{
    if constexpr (VAR == VAR_HORNER_CENTRED) {
        static_assert(D < kFp64SetupCentred, "plain FP32 sums");
        constexpr CentredMatrix<D> T = make_centred_matrix<D>();
        e.d = D;
#pragma unroll
        for (int m = 0; m <= D; ++m)
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                float acc = 0.f;
#pragma unroll
                for (int i = 0; i <= D; ++i) acc = fmaf(T.t[m][i], b[i][k], acc);
                e.a[m][k] = acc;
            }
    } else {
        e.setup(b, D);
    }
}

// The points of curve c in registers.
template <int D, int DIM>
__device__ __forceinline__ void load_curve(const CurveArgs& a, int64_t c, float (&b)[D + 1][DIM])
{
    const int64_t at = c * ((D + 1) * DIM);
    if (a.dtype == 0) {
#pragma unroll
        for (int m = 0; m <= D; ++m)
#pragma unroll
            for (int k = 0; k < DIM; ++k) b[m][k] = __ldg(static_cast<const float*>(a.ctrl) + at + m * DIM + k);
    } else {
#pragma unroll
        for (int m = 0; m <= D; ++m)
#pragma unroll
            for (int k = 0; k < DIM; ++k) b[m][k] = load_elem(a.ctrl, a.dtype, at + m * DIM + k);
    }
}

constexpr int kFewThreads = 128;

// Points of a small call, one thread per sample or few: the curve's points come
// straight into registers, beside the parameter, and nothing is staged, so that
// a call is one load latency long instead of three.  Thread (c, q) takes samples
// q, q + per, q + 2 per, ... of curve c, `per` threads a curve.
template <int VAR, int D, int DIM>
__global__ void __launch_bounds__(kFewThreads) k_points_few(const CurveArgs a, int tm, uint32_t per, uint32_t total)
{
    const uint32_t i = blockIdx.x * kFewThreads + threadIdx.x;
    if (i >= total) return;
    const uint32_t n_t = (uint32_t)a.n_t, c = i / per;
    uint32_t j = i - c * per;
    float t = 0.f, b[D + 1][DIM], P[DIM];
    const float* tc = a.t + c * a.t_stride;
    if (tm == TM_ARRAY) t = __ldg(tc + j);
    load_curve<D, DIM>(a, c, b);
    Eval<VAR, D, DIM> e;
    register_setup<VAR, D, DIM>(b, e);
    const uint32_t key = curve_key<TM_HASH>(a, c);
    const float den = (float)(n_t - 1);
    float* o = a.out + (int64_t)c * n_t * DIM;
    for (;;) {
        float x = clamp01(t);
        const uint32_t next = j + per;
        if (tm == TM_ARRAY) t = next < n_t ? __ldg(tc + next) : 0.f;
        else if (tm == TM_UNIFORM) x = n_t > 1 ? __fdiv_rn((float)j, den) : 0.f;
        else x = hash_unit(lowbias32(key ^ j));
        e.eval(x, P);
#pragma unroll
        for (int k = 0; k < DIM; ++k) o[j * DIM + k] = P[k];
        if (next >= n_t) break;
        j = next;
    }
}

// ---------------------------------------------------------------- packed lengths

// Two FP32 values per register pair.  sm_103a runs add, multiply and fma on both
// halves with one instruction of two cycles: as many operations per cycle as the
// scalar forms, for half of the issue slots, and the fused draw-and-measure loop
// is bound by instruction issue: 28 -> 21.5 lane instructions per point of a 3D
// cubic.  1,048,576 cubics x 1024 draws: 868 -> 799 us (the FMA pipe that also
// takes the integer multiplies then 76 % busy, issue 70 %; scalar subtractions,
// additions or square-root sums, 2 or 4 samples side by side and 80 registers
// all measured slower or the same); 65,536 x 400 of degree 5 68 -> 38 us, 2D
// cubics 217 -> 25 us.
using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Centred Horner at two parameters at once, u = t - 1/2.
template <int D, int DIM>
struct PackedHorner {
    f32x2 c[D + 1][DIM];
    __device__ __forceinline__ void setup(const Eval<VAR_HORNER_CENTRED, D, DIM>& e)
    {
#pragma unroll
        for (int i = 0; i <= D; ++i)
#pragma unroll
            for (int k = 0; k < DIM; ++k) c[i][k] = pack2(e.a[i][k], e.a[i][k]);
    }
    __device__ __forceinline__ void eval(f32x2 u, f32x2 (&P)[DIM]) const
    {
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            f32x2 acc = c[D][k];
#pragma unroll
            for (int i = D - 1; i >= 0; --i) acc = fma2(acc, u, c[i][k]);
            P[k] = acc;
        }
    }
};

// u = t - 1/2 at the pre-mixed draws of samples ja + i and jb + i, i < 4 (ja, jb
// multiples of 4, so a draw's input is one xor from the group's).  1.m - 3/2
// equals (1.m - 1) - 1/2, both subtractions of the scalar form being exact.
__device__ __forceinline__ void packed_draws(uint32_t key, uint32_t ja, uint32_t jb, f32x2 (&u)[4])
{
    const uint32_t ka = key ^ ja, kb = key ^ jb;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        u[i] = add2(pack2(hash_one_plus(lowbias32_tail((ka ^ (uint32_t)i) * kLowbiasMul1)),
                          hash_one_plus(lowbias32_tail((kb ^ (uint32_t)i) * kLowbiasMul1))),
                    pack2(-1.5f, -1.5f));
}

// The order of a length's sum depends on n_t (and on whether the parameters are an
// array) alone, so that a curve's length to the last bit does not depend on the
// other curves of the call: a curve's samples are cut into 2^lg runs, a run is
// summed over its groups of 4 segments in order, and the runs pairwise.  A lane
// takes a run.  In a call of few curves (FEW) 2^lk lanes share a run's groups, put
// the group sums into shared memory, and the last of them adds these in order.

constexpr uint32_t kSharedRunSamples = 4096;  // most samples of a curve whose runs are shared

// the groups [g0, g1) of lane `sub` of a run of `groups`
__device__ __forceinline__ void shared_groups(uint32_t groups, int sub, int lk, uint32_t& g0, uint32_t& g1)
{
    const uint32_t each = (groups + (1u << lk) - 1) >> lk;
    g0 = min(each * sub, groups);
    g1 = min(g0 + each, groups);
}

// u = t - 1/2 at the draws of samples ja and jb
__device__ __forceinline__ f32x2 packed_draw(uint32_t key, uint32_t ja, uint32_t jb)
{
    return add2(pack2(hash_one_plus(lowbias32_premixed(key, ja)), hash_one_plus(lowbias32_premixed(key, jb))),
                pack2(-1.5f, -1.5f));
}

// Length over a run's samples [s, end): the half runs [s, m) and [m, end) side by
// side in the halves of the packed registers, their ends joined.  s and m are
// multiples of 4 and the halves' groups of 4 differ by at most one, so at most
// 7 samples of the first and 3 of the second half are left for scalar steps.
// `first`, `last`: the run's end points; FEW: these and the length come back in
// the last of the run's lanes (`sub` of 2^lk), `sums` holds the run's group sums.
template <int D, int DIM, bool FEW>
__device__ __forceinline__ float packed_run(const Eval<VAR_HORNER_CENTRED, D, DIM>& e, const TileParams& tp,
                                            uint32_t s, uint32_t m, uint32_t end, f32x2* sums, int sub, int lk,
                                            float (&first)[DIM], float (&last)[DIM])
{
    PackedHorner<D, DIM> h;
    h.setup(e);
    const uint32_t both = min(m - s, end - m) & ~3u;
    const bool shared = FEW && lk > 0;
    uint32_t i0 = 0, i1 = both;
    if (shared) {
        shared_groups(both / 4, sub, lk, i0, i1);
        i0 *= 4;
        i1 *= 4;
    }
    f32x2 acc2 = 0ull, prev[DIM];
    float acc = 0.f, fb[DIM], pa[DIM], pb[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) fb[k] = pa[k] = pb[k] = 0.f;
    if (both > 0) {
        f32x2 u[4];
        packed_draws(tp.key, s + i0, m + i0, u);
        // the run's first segment ends where it starts: length 0
        h.eval(FEW && i0 > 0 ? packed_draw(tp.key, s + i0 - 1, m + i0 - 1) : u[0], prev);
#pragma unroll
        for (int k = 0; k < DIM; ++k) unpack2(prev[k], first[k], fb[k]);
        for (uint32_t i = i0; i < i1; i += 4) {
            if (i > i0) packed_draws(tp.key, s + i, m + i, u);
            f32x2 gs = 0ull;  // a group's 4 segments are summed first
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                f32x2 P[DIM], q = 0ull;
                h.eval(u[g], P);
#pragma unroll
                for (int k = 0; k < DIM; ++k) {
                    const f32x2 d = sub2(P[k], prev[k]);
                    q = k == 0 ? mul2(d, d) : fma2(d, d, q);
                    prev[k] = P[k];
                }
                float qa, qb;
                unpack2(q, qa, qb);
                const f32x2 sl = pack2(sqrt_approx(qa), sqrt_approx(qb));
                gs = g == 0 ? sl : add2(gs, sl);
            }
            if (shared) sums[i / 4] = gs;
            else acc2 = add2(acc2, gs);
        }
#pragma unroll
        for (int k = 0; k < DIM; ++k) unpack2(prev[k], pa[k], pb[k]);
    }
    if (shared) {
        const int base = (threadIdx.x & 31) - sub;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            first[k] = __shfl_sync(kFull, first[k], base);
            fb[k] = __shfl_sync(kFull, fb[k], base);
        }
        __syncwarp();
        if (sub != (1 << lk) - 1) return 0.f;
        for (uint32_t g = 0; g < both / 4; ++g) acc2 = add2(acc2, sums[g]);
    }
    if (both > 0) {
        float aa, ab;
        unpack2(acc2, aa, ab);
        acc = aa + ab;
    }
    // what is left of either half
    auto step = [&](uint32_t j, bool start, float (&f)[DIM], float (&p)[DIM]) {
        float t[1], P[DIM];
        tp.get<1, true>(TM_HASH16, j, 1, 0, t);
        e.eval(t[0], P);
        if (start) {
#pragma unroll
            for (int k = 0; k < DIM; ++k) f[k] = P[k];
        } else {
            acc += seg_len<DIM>(P, p);
        }
#pragma unroll
        for (int k = 0; k < DIM; ++k) p[k] = P[k];
    };
#pragma unroll 1
    for (uint32_t j = s + both; j < m; ++j) step(j, j == s, first, pa);
#pragma unroll 1
    for (uint32_t j = m + both; j < end; ++j) step(j, j == m, fb, pb);
    if (end > m) {
        acc += seg_len<DIM>(fb, pa);
#pragma unroll
        for (int k = 0; k < DIM; ++k) last[k] = pb[k];
    } else {
#pragma unroll
        for (int k = 0; k < DIM; ++k) last[k] = pa[k];
    }
    return acc;
}

// Samples of a run of the scalar form, 2^lg runs a curve.  An odd count where the
// lanes read arrays: with a multiple of 32 they would all read the same bank of the
// L1 (65,536 x 256 with their own t: 63 us, 24 with 33; x 1024 at shared t 233 and 79).
__host__ __device__ __forceinline__ uint32_t length_run(uint32_t n_t, int lg, int tm)
{
    const uint32_t run = (n_t + (1u << lg) - 1) >> lg;
    return tm == TM_ARRAY ? run | 1u : run;
}

// The same over samples [s, end) at any parameters, one sample after the other.
template <int VAR, int D, int DIM, bool FEW>
__device__ __forceinline__ float scalar_run(const Eval<VAR, D, DIM>& e, const TileParams& tp, int tm, uint32_t s,
                                            uint32_t end, float* sums, int sub, int lk, float (&first)[DIM],
                                            float (&prev)[DIM])
{
    const uint32_t groups = s < end ? (end - s - 1) / 4 : 0;  // of 4 segments; up to 3 segments are left
    const bool shared = FEW && lk > 0;
    uint32_t g0 = 0, g1 = groups;
    if (shared) shared_groups(groups, sub, lk, g0, g1);
    float acc = 0.f;
    if (s < end) {
        float t[1];
        tp.get<1, true>(tm, s + 4 * g0, 1, end, t);
        e.eval(t[0], first);
#pragma unroll
        for (int k = 0; k < DIM; ++k) prev[k] = first[k];
    }
    uint32_t j = s + 1 + 4 * g0;
    for (uint32_t g = g0; g < g1; ++g, j += 4) {
        // the group's 4 segments are summed first and then added to the run
        float t[4], gs = 0.f;
        tp.get<4, true>(tm, j, 1, end, t);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            float P[DIM];
            e.eval(t[m], P);
            gs += seg_len<DIM>(P, prev);
#pragma unroll
            for (int k = 0; k < DIM; ++k) prev[k] = P[k];
        }
        if (shared) sums[g] = gs;
        else acc += gs;
    }
    if (shared) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) first[k] = __shfl_sync(kFull, first[k], (threadIdx.x & 31) - sub);
        __syncwarp();
        if (sub != (1 << lk) - 1) return 0.f;
        for (uint32_t g = 0; g < groups; ++g) acc += sums[g];
    }
    if (j < end) {
        float t[4];
        tp.get(tm, j, 1, end, t);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            if (j + m < end) {
                float P[DIM];
                e.eval(t[m], P);
                acc += seg_len<DIM>(P, prev);
#pragma unroll
                for (int k = 0; k < DIM; ++k) prev[k] = P[k];
            }
        }
    }
    return acc;
}

// Polyline lengths, 2^lg runs a curve, one lane each (65,536 cubics x 400
// samples: shared t 33 us, uniform 35, own t 38, against 42, 48 and 52 with a warp
// per curve): each lane walks a contiguous run of samples (PACKED: centred Horner at
// pre-mixed draws, two half runs at a time), the segments joining two runs are closed
// with one shuffle, and the run sums are added over the curve's lanes.  FEW: 2^lk lanes
// share a run, and where the set-up needs no other lane, every lane loads its curve
// itself.  A call's time (us, GB300) before and after: 1000 cubics x 256 shared t 4.6 ->
// 3.1, 1000 quintics x 1024 draws 13.8 -> 4.7, 100 cubics x 65,536 draws 541 -> 70.
template <int VAR, int D, int DIM, bool PACKED, bool FEW>
__global__ void __launch_bounds__(kWarps * 32, (D + 1) * DIM > 20 ? 3 : 4)
    k_length(const CurveArgs a, int tm, int lg, int lk)
{
    using Smem = TileSmem<D, DIM, 8 * (D + 1) * DIM>;
    __shared__ Smem s_tile[kWarps];
    __shared__ f32x2 s_sums[FEW ? kWarps : 1][FEW ? kSharedRunSamples / 8 : 1];  // group sums of a warp's curves
    const int lane = threadIdx.x & 31;
    Smem& sm = s_tile[threadIdx.x >> 5];
    const int lanes = FEW ? 1 << lk : 1, ll = FEW ? lg + lk : lg;  // lanes of a run, log2 of a curve's
    const int B = 1 << lg, cpw = 32 >> ll, grp = lane >> ll, li = lane & ((1 << ll) - 1);
    const int br = FEW ? li >> lk : li, sub = FEW ? li & (lanes - 1) : 0;
    const uint32_t n_t = (uint32_t)a.n_t;  // unsigned: an index may step past 2^31 - 1
    const uint32_t run = length_run(n_t, lg, tm);
    const int64_t n_units = (a.n_curves + cpw - 1) / cpw;
    const int64_t n_warps = (int64_t)gridDim.x * kWarps;
    TileParams tp;
    tp.grid.init(a.n_t);
    for (int64_t u = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5); u < n_units; u += n_warps) {
        const int64_t c0 = u * cpw;
        const int nc = (int)min((int64_t)cpw, a.n_curves - c0);
        Eval<VAR, D, DIM> e;
        const bool live = grp < nc;
        if constexpr (FEW && (VAR != VAR_HORNER_CENTRED || D < kFp64SetupCentred)) {
            float b[D + 1][DIM];
            load_curve<D, DIM>(a, c0 + (live ? grp : 0), b);
            register_setup<VAR, D, DIM>(b, e);
        } else {
            tile_setup<VAR>(a, sm, c0, nc, grp, lane, e);
        }
        tp.curve(a, tm, c0 + (live ? grp : 0));
        float acc = 0.f, first[DIM], prev[DIM];
#pragma unroll
        for (int k = 0; k < DIM; ++k) first[k] = prev[k] = 0.f;
        uint32_t jb, je;
        if constexpr (PACKED) {
            // two half runs a lane, in whole groups of 4 samples shared out evenly
            const uint32_t ng = (n_t + 3) / 4, q = ng >> (lg + 1), r = ng & (2 * B - 1);
            const uint32_t h0 = 2 * br, h1 = h0 + 1, h2 = h0 + 2;
            jb = min(n_t, 4 * (h0 * q + min(h0, r)));
            je = live ? min(n_t, 4 * (h2 * q + min(h2, r))) : jb;
            const uint32_t jm = min(je, 4 * (h1 * q + min(h1, r)));
            f32x2* sums = FEW ? s_sums[threadIdx.x >> 5] + (grp * B + br) * (q + (r > 0)) : nullptr;
            if (FEW || jb < je) acc = packed_run<D, DIM, FEW>(e, tp, jb, jm, je, sums, sub, lk, first, prev);
        } else {
            jb = min(br * run, n_t);
            je = live ? min(jb + run, n_t) : jb;
            float* sums = FEW ? reinterpret_cast<float*>(s_sums[threadIdx.x >> 5]) + (grp * B + br) * (run / 4) : nullptr;
            if (FEW || jb < je) acc = scalar_run<VAR, D, DIM, FEW>(e, tp, tm, jb, je, sums, sub, lk, first, prev);
        }
        float pl[DIM];
#pragma unroll
        for (int k = 0; k < DIM; ++k) pl[k] = __shfl_up_sync(kFull, prev[k], lanes);
        if (br > 0 && jb < je && sub == lanes - 1) acc += seg_len<DIM>(first, pl);
        for (int o = B >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o * lanes);  // over the curve's runs
        if (li == lanes - 1 && live) a.out[c0 + grp] = acc;
        if (FEW) __syncwarp();  // the next unit's group sums come after this one's are read
    }
}

// ---------------------------------------------------------------- launch shape

// units of work a launch should have at least before lanes are taken from a
// curve's samples: two for each of the 32 warps an SM holds of these kernels
inline int64_t tile_target_units(int sm_count) { return (int64_t)sm_count * 64; }

inline int tile_grid(const void* kern, int64_t units, int sm_count)
{
    // one unit per warp while they all fit the SMs twice over, otherwise
    // blocks of four units per warp, refilled by the block scheduler
    const int64_t work = (units + kWarps - 1) / kWarps;
    const int full = persistent_grid(kern, kWarps * 32, 0, sm_count, work);
    if (work <= 2 * (int64_t)full) return (int)work;
    const int64_t g = (work + 3) / 4;
    return (int)(g > 2 * (int64_t)full ? (g < 2147483647 ? g : 2147483647) : 2 * (int64_t)full);
}

template <int VAR, int D, int DIM>
LaunchResult launch_points(const CurveArgs& a, int tm, cudaStream_t s, const LaunchHooks& h)
{
    // Small calls (centred Horner from degree 5 on shares its compensated set-up
    // over a curve's lanes, and keeps k_points).  us on GB300, k_points against
    // k_points_few with 1, 2 and 4 samples a thread, FP32, shared t: cubics 100 x 64
    // 2.9: 1.4; 1953 x 64 3.3: 2.1, 2.2, 2.4; 7812 x 64 5.5: 4.2, 3.3, 3.1; 15,625 x
    // 64 8.7: 6.6, 4.8, 4.3; 3906 x 256 5.2: 6.6, 4.8, 4.2; 62,500 x 64 12.8: 22.4,
    // 14.9, 11.5; 15,625 x 256 11.7: 22.2, 14.7, 11.0, with 8 samples 9.5; 125,000 x 8
    // 9.5: 6.7, 5.4, 9.8; 166,666 x 24 14.6: 22.7, 15.3, 18.3.  4D quartics 10,000 x
    // 100 7.9: 8.5, 6.7; 40,000 x 100 17.1: 29.7, 20.5, 19.4; 4D Bernstein of degree 7
    // 62,500 x 8 10.5: 9.4; 125,000 x 8 13.2: 16.9.
    const int64_t samples = a.n_curves * (int64_t)a.n_t;
    constexpr int64_t kMost = DIM == 4 ? 1000000 : 4000000, kMostShort = DIM == 4 ? 500000 : 1000000;
    if constexpr (VAR != VAR_HORNER_CENTRED || D < kFp64SetupCentred) {
        if (samples <= (a.n_t >= 64 ? kMost : kMostShort)) {
            const bool long_curves = a.n_t >= 256;
            const uint32_t run = samples <= 200000                           ? 1
                                 : samples <= (long_curves ? 600000 : 1000000)  ? 2
                                 : samples <= 2000000 || !long_curves           ? 4
                                                                               : 8;
            const uint32_t per = ((uint32_t)a.n_t + run - 1) / run, total = (uint32_t)a.n_curves * per;
            h.count(h.self);
            h.begin(h.self, s);
            k_points_few<VAR, D, DIM><<<(total + kFewThreads - 1) / kFewThreads, kFewThreads, 0, s>>>(a, tm, per, total);
            const cudaError_t err = cudaGetLastError();
            h.end(h.self, s);
            return {1, err};
        }
    }
    auto kern = k_points<VAR, D, DIM>;
    // As few lanes per curve as hold its samples in one tile (8 a lane), 16 at
    // most, so that a lane's setup serves 8 samples and more; more lanes when
    // that leaves the SMs short of warps.  Cubic 3D points, FP32, shared t,
    // against one warp per curve (us, GB300): 1,000,000 x 24 82 / 232, 500,000
    // x 64 98 / 125, 65,536 x 256 40 / 41 (32 lanes: 47); 60,013 2D cubics x
    // 40 on a grid 20 / 122 with the runtime-degree kernel.
    int lg = a.n_t <= 32 ? 2 : a.n_t <= 64 ? 3 : 4;
    const int64_t target = tile_target_units(h.sm_count);
    while (lg < 5 && ((a.n_curves << lg) >> 5) < target) ++lg;
    int parts = 1, part_len = 0;
    if (lg == 5 && a.n_curves < target) {
        const int64_t tiles = ((int64_t)a.n_t + kTileSamples - 1) / kTileSamples;
        const int64_t want = (target + a.n_curves - 1) / a.n_curves;
        const int64_t per = want >= tiles ? 1 : tiles / want;
        parts = (int)((tiles + per - 1) / per);
        part_len = parts > 1 ? (int)per * kTileSamples : 0;
    }
    const int64_t units = parts > 1 ? a.n_curves * parts : (a.n_curves + (32 >> lg) - 1) / (32 >> lg);
    const int grid = tile_grid((const void*)kern, units, h.sm_count);
    h.count(h.self);
    h.begin(h.self, s);
    kern<<<grid, kWarps * 32, 0, s>>>(a, tm, lg, parts, part_len);
    const cudaError_t err = cudaGetLastError();
    h.end(h.self, s);
    return {1, err};
}

template <int VAR, int D, int DIM>
LaunchResult launch_length(const CurveArgs& a, int tm, cudaStream_t s, const LaunchHooks& h)
{
    constexpr bool PACKED = VAR == VAR_HORNER_CENTRED;  // the packed form serves the pre-mixed draw
    const bool packed = PACKED && tm == TM_HASH16;
    // Runs of 16 to 32 samples until a curve has 32; of in-kernel draws, where nothing
    // is read per sample and a lane's set-up and joins serve the longest runs, of up
    // to 256 samples.
    int lg = 2;
    const uint32_t n_t = (uint32_t)a.n_t;
    while (lg < 5 && n_t > ((packed ? 256u : 32u) << lg)) ++lg;
    // Lanes that share a run, while their warps fit the SMs at once and (two lanes,
    // whose second start and joins cost the most) leave the SMs short of warps.  us on
    // GB300, a lane / 2^lk lanes a run; draws, cubics 32 x 1024 7.7 / 3.8 and 4000 x 1024
    // 11.2 / 7.9 (8 lanes), 8000 x 1024 11.4 / 13.5 (2); quintics 1000 x 256 5.8 / 3.3,
    // 1000 x 1024 13.0 / 4.7, 4000 x 4096 21.3 / 28.0 (2); shared t, cubics 1000 x 128
    // 4.4 / 2.8, 4000 x 256 4.9 / 4.3 (2), 8000 x 256 5.5 / 5.8; Seiler on a grid 1000 x
    // 256 3.8 / 3.1, 4000 x 256 3.9 / 4.2 (2).
    const uint32_t groups = packed ? (n_t + 4) >> (lg + 3) : (length_run(n_t, lg, tm) - 1) / 4;
    auto warps = [&](int k) { return (a.n_curves << (lg + k)) >> 5; };
    int lk = 0;
    if (n_t <= kSharedRunSamples)
        while (lk < 5 - lg && groups >> (lk + 1) >= 1 && warps(lk + 1) <= (int64_t)h.sm_count * 18) ++lk;
    if (lk == 1 && tm != TM_ARRAY && warps(1) > (int64_t)h.sm_count * 7) lk = 0;
    // (up to 64 samples, lanes that load their curve themselves are faster throughout:
    // 65,536 cubics x 64 draws 8.3 -> 7.8)
    const bool few = lk > 0 || (n_t <= 64 && (VAR != VAR_HORNER_CENTRED || D < kFp64SetupCentred));
    auto kern = packed ? (few ? k_length<VAR, D, DIM, PACKED, true> : k_length<VAR, D, DIM, PACKED, false>)
                       : (few ? k_length<VAR, D, DIM, false, true> : k_length<VAR, D, DIM, false, false>);
    const int cpw = 32 >> (few ? lg + lk : lg);
    const int64_t units = (a.n_curves + cpw - 1) / cpw;
    const int grid = tile_grid((const void*)kern, units, h.sm_count);
    h.count(h.self);
    h.begin(h.self, s);
    kern<<<grid, kWarps * 32, 0, s>>>(a, tm, lg, lk);
    const cudaError_t err = cudaGetLastError();
    h.end(h.self, s);
    return {1, err};
}

// ---------------------------------------------------------------- dispatch

// Runtime-degree kernels (degree 8..15): one warp per curve.
template <int VAR, int DIM>
LaunchResult launch_dynamic(const CurveArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    if (om == OM_POINTS) {
        if (tm == TM_ARRAY) return launch_one<VAR, 0, DIM, TM_ARRAY, OM_POINTS>(a, s, h);
        if (tm == TM_UNIFORM) return launch_one<VAR, 0, DIM, TM_UNIFORM, OM_POINTS>(a, s, h);
        return launch_one<VAR, 0, DIM, TM_HASH, OM_POINTS>(a, s, h);
    }
    if (tm == TM_ARRAY) return launch_one<VAR, 0, DIM, TM_ARRAY, OM_LENGTH>(a, s, h);
    if (tm == TM_UNIFORM) return launch_one<VAR, 0, DIM, TM_UNIFORM, OM_LENGTH>(a, s, h);
    return launch_one<VAR, 0, DIM, TM_HASH, OM_LENGTH>(a, s, h);
}

// Fixed degrees: k_points and k_length (the pre-mixed draw needs every sample
// index below 2^16).
template <int VAR, int D, int DIM>
LaunchResult launch_fixed(const CurveArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    if (om == OM_POINTS) return launch_points<VAR, D, DIM>(a, tm, s, h);
    const bool draw16 = tm == TM_HASH && a.n_t <= 65536;
    // (the other evaluators' fused draw-and-measure form keeps a warp per curve)
    if constexpr (DIM == 3 && VAR != VAR_HORNER_CENTRED) {
        if (draw16) return launch_one<VAR, D, DIM, TM_HASH16, OM_LENGTH>(a, s, h);
    }
    return launch_length<VAR, D, DIM>(a, draw16 ? TM_HASH16 : tm, s, h);
}

template <int VAR, int DIM>
LaunchResult launch_degree(const CurveArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    switch (a.degree) {
    case 1: return launch_fixed<VAR, 1, DIM>(a, tm, om, s, h);
    case 2: return launch_fixed<VAR, 2, DIM>(a, tm, om, s, h);
    case 3: return launch_fixed<VAR, 3, DIM>(a, tm, om, s, h);
    case 4: return launch_fixed<VAR, 4, DIM>(a, tm, om, s, h);
    case 5: return launch_fixed<VAR, 5, DIM>(a, tm, om, s, h);
    case 6: return launch_fixed<VAR, 6, DIM>(a, tm, om, s, h);
    case 7: return launch_fixed<VAR, 7, DIM>(a, tm, om, s, h);
    default: return launch_dynamic<VAR, DIM>(a, tm, om, s, h);
    }
}

template <int VAR>
LaunchResult launch_curve_variant(const CurveArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    switch (a.dim) {
    case 1: return launch_degree<VAR, 1>(a, tm, om, s, h);
    case 2: return launch_degree<VAR, 2>(a, tm, om, s, h);
    case 3: return launch_degree<VAR, 3>(a, tm, om, s, h);
    default: return launch_degree<VAR, 4>(a, tm, om, s, h);
    }
}

}  // namespace bez
