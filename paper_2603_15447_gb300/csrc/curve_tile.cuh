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
    const int64_t at = (int64_t)c * ((D + 1) * DIM);
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
// cubic.  1,048,576 cubics x 1024 draws: 868 -> 823 us (the FMA pipe that also
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

// Length over one lane's samples [s, e): the half runs [s, m) and [m, e) side by
// side in the halves of the packed registers, their ends joined.  s and m are
// multiples of 4 and the halves' groups of 4 differ by at most one, so at most
// 7 samples of the first and 3 of the second half are left for scalar steps.
// `first`, `last`: the run's end points.
template <int D, int DIM>
__device__ __forceinline__ float packed_run(const Eval<VAR_HORNER_CENTRED, D, DIM>& e, const TileParams& tp,
                                            uint32_t s, uint32_t m, uint32_t end, float (&first)[DIM],
                                            float (&last)[DIM])
{
    PackedHorner<D, DIM> h;
    h.setup(e);
    const uint32_t both = min(m - s, end - m) & ~3u;
    f32x2 acc2 = 0ull, prev[DIM];
    float acc = 0.f, fb[DIM], pa[DIM], pb[DIM];
    if (both > 0) {
        f32x2 u[4];
        packed_draws(tp.key, s, m, u);
        h.eval(u[0], prev);  // the run's first segment ends where it starts: length 0
#pragma unroll
        for (int k = 0; k < DIM; ++k) unpack2(prev[k], first[k], fb[k]);
        for (uint32_t i = 0; i < both; i += 4) {
            if (i > 0) packed_draws(tp.key, s + i, m + i, u);
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
            acc2 = add2(acc2, gs);
        }
#pragma unroll
        for (int k = 0; k < DIM; ++k) unpack2(prev[k], pa[k], pb[k]);
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

// resident blocks per SM that k_length's registers are sized for (the packed
// form holds its coefficients twice)
__host__ __device__ constexpr int length_blocks(bool packed, int D, int DIM)
{
    const int per = (D + 1) * DIM;
    return packed ? (per <= 6 ? 5 : per <= 12 ? 4 : per <= 16 ? 3 : 2) : per > 20 ? 3 : 4;
}

// Polyline lengths, 2^lg lanes a curve (65,536 cubics x 400 samples: shared t
// 36 us, uniform 35, own t 43, against 42, 48 and 52 with a warp per curve): each
// lane walks a contiguous run of samples (PACKED: centred Horner at pre-mixed
// draws, two half runs at a time), the segments joining two runs are closed with one shuffle, and the
// run sums are added over the curve's lanes.
template <int VAR, int D, int DIM, bool PACKED>
__global__ void __launch_bounds__(kWarps * 32, (D + 1) * DIM > 20 ? 3 : (D + 1) * DIM > 12 ? 4 : 4)
    k_length(const CurveArgs a, int tm, int lg)
{
    using Smem = TileSmem<D, DIM, 8 * (D + 1) * DIM>;
    __shared__ Smem s_tile[kWarps];
    const int lane = threadIdx.x & 31;
    Smem& sm = s_tile[threadIdx.x >> 5];
    const int G = 1 << lg, cpw = 32 >> lg, grp = lane >> lg, li = lane & (G - 1);
    const uint32_t n_t = (uint32_t)a.n_t;  // unsigned: an index may step past 2^31 - 1
    const uint32_t run = (n_t + G - 1) >> lg;
    const int64_t n_units = (a.n_curves + cpw - 1) / cpw;
    const int64_t n_warps = (int64_t)gridDim.x * kWarps;
    TileParams tp;
    tp.grid.init(a.n_t);
    for (int64_t u = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5); u < n_units; u += n_warps) {
        const int64_t c0 = u * cpw;
        const int nc = (int)min((int64_t)cpw, a.n_curves - c0);
        Eval<VAR, D, DIM> e;
        tile_setup<VAR>(a, sm, c0, nc, grp, lane, e);
        const bool live = grp < nc;
        tp.curve(a, tm, c0 + (live ? grp : 0));
        float acc = 0.f, first[DIM], prev[DIM];
#pragma unroll
        for (int k = 0; k < DIM; ++k) first[k] = prev[k] = 0.f;
        uint32_t jb, je;
        if constexpr (PACKED) {
            // two half runs a lane, in whole groups of 4 samples shared out evenly
            const uint32_t ng = (n_t + 3) / 4, q = ng >> (lg + 1), r = ng & (2 * G - 1);
            const uint32_t h0 = 2 * li, h1 = h0 + 1, h2 = h0 + 2;
            jb = min(n_t, 4 * (h0 * q + min(h0, r)));
            je = live ? min(n_t, 4 * (h2 * q + min(h2, r))) : jb;
            const uint32_t jm = min(je, 4 * (h1 * q + min(h1, r)));
            if (jb < je) acc = packed_run<D, DIM>(e, tp, jb, jm, je, first, prev);
        } else {
            jb = min(li * run, n_t);
            je = live ? min(jb + run, n_t) : jb;
            if (jb < je) {
                float t1[1];
                tp.get<1, true>(tm, jb, 1, je, t1);
                e.eval(t1[0], first);
#pragma unroll
                for (int k = 0; k < DIM; ++k) prev[k] = first[k];
            }
            uint32_t j = jb + 1;
            for (; j + 4 <= je; j += 4) {
                // the group's 4 segments are summed first and then added to the run
                float t[4], gs = 0.f;
                tp.get<4, true>(tm, j, 1, je, t);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    float P[DIM];
                    e.eval(t[m], P);
                    gs += seg_len<DIM>(P, prev);
#pragma unroll
                    for (int k = 0; k < DIM; ++k) prev[k] = P[k];
                }
                acc += gs;
            }
            if (j < je) {
                float t[4];
                tp.get(tm, j, 1, je, t);
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    if (j + m < je) {
                        float P[DIM];
                        e.eval(t[m], P);
                        acc += seg_len<DIM>(P, prev);
#pragma unroll
                        for (int k = 0; k < DIM; ++k) prev[k] = P[k];
                    }
                }
            }
        }
        float pl[DIM];
#pragma unroll
        for (int k = 0; k < DIM; ++k) pl[k] = __shfl_up_sync(kFull, prev[k], 1);
        if (li > 0 && jb < je) acc += seg_len<DIM>(first, pl);
        for (int o = G >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);  // over the curve's lanes
        if (li == 0 && live) a.out[c0 + grp] = acc;
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
        const int64_t tiles = (a.n_t + kTileSamples - 1) / kTileSamples;
        const int64_t want = (target + a.n_curves - 1) / a.n_curves;
        const int64_t per = want >= tiles ? 1 : tiles / want;
        part_len = (int)per * kTileSamples;
        parts = (a.n_t + part_len - 1) / part_len;
        if (parts == 1) part_len = 0;
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
    auto kern = packed ? k_length<VAR, D, DIM, PACKED> : k_length<VAR, D, DIM, false>;
    // runs of 16 to 32 samples a lane until a curve has a warp.  By n_t alone:
    // the order of the sum, and so a curve's length to the last bit, does not
    // depend on the other curves of the call.
    // In-kernel draws of 64 samples and more take 4 lanes a curve: nothing is
    // read per sample, and a lane's set-up and joins serve the longest runs.
    int lg = 2;
    if (!packed)
        while (lg < 5 && a.n_t > (32 << lg)) ++lg;
    const int64_t units = (a.n_curves + (32 >> lg) - 1) / (32 >> lg);
    const int grid = tile_grid((const void*)kern, units, h.sm_count);
    h.count(h.self);
    h.begin(h.self, s);
    kern<<<grid, kWarps * 32, 0, s>>>(a, tm, lg);
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
