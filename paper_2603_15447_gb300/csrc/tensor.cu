// tensor.cu -- tensor-product Bezier surfaces and volumes on uniform grids
// (paper Sec. 2.2: a surface splits its order between u and v, a volume
// between u, v and w; the bicubic case evaluates the four column curves at u
// and then the isoline cubic in v).
//
// Separable contraction (bicubic 3D patches on grids of up to 64 rows take one
// warp per patch, larger ones a block; tricubic scalar volumes one warp per
// volume: k_volume_tricubic1_warp in tensor_common.cuh, shared with the texture
// volumes; every other grid k_grid, one warp per block of rows):
//   surface  X[a][j] = sum_i Bu[a][i] C[i][j]          (isoline control points)
//            P[a][b] = sum_j X[a][j] Bv[b][j]
//   volume   Y[a][j][l] = sum_i Bu[a][i] C[i][j][l]
//            Z[a][b][l] = sum_j Bv[b][j] Y[a][j][l]
//            V[a][b][c] = sum_l Bw[c][l] Z[a][b][l]
// with Bernstein tables of the grid values t_a = fl32(a) / fl32(n-1) built
// once per block.  The output is write-bound; every thread writes runs of
// consecutive floats (float4 when the layout allows), so stores are fully
// coalesced.  The contraction has a reduction depth of 4 for bicubic
// patches, far too small to keep tensor cores busy on a store-bound kernel,
// so it runs on the FP32 pipes.
#include "curve_tile.cuh"
#include "tensor_common.cuh"

namespace bez {

// Fast path: bicubic 3D patches, nv a multiple of 4.  Each thread owns four
// consecutive points of one grid row and writes them as three float4.
__global__ void __launch_bounds__(kTensorThreads) k_surface_bicubic3(const TensorArgs a)
{
    __shared__ float4 s_bv[kTensorMaxGrid];        // Bv[b][0..3]
    __shared__ float s_bu[kTensorMaxGrid * 4];     // Bu[a][0..3]
    __shared__ float s_c[48];                      // C[i][j][k]
    __shared__ float s_x[kTensorMaxGrid * 12];     // X[a][j][k]
    const int tid = threadIdx.x;
    bernstein_table(s_bu, a.nu, 3, tid, kTensorThreads);
    {
        float* bv = reinterpret_cast<float*>(s_bv);
        bernstein_table(bv, a.nv, 3, tid, kTensorThreads);
    }
    const int nu = a.nu, nv = a.nv;
    const int quads_per_row = nv / 4;
    const int n_quads = nu * quads_per_row;
    const int64_t pts = (int64_t)nu * nv;
    // the next patch's control points are loaded while the current one is
    // evaluated and stored
    float nxt = (tid < 48 && (int64_t)blockIdx.x < a.n) ? load_elem(a.ctrl, a.dtype, (int64_t)blockIdx.x * 48 + tid) : 0.f;
    for (int64_t p = blockIdx.x; p < a.n; p += gridDim.x) {
        __syncthreads();  // tables ready / previous patch done with s_c, s_x
        if (tid < 48) s_c[tid] = nxt;
        __syncthreads();
        const int64_t pn = p + gridDim.x;
        if (tid < 48 && pn < a.n) nxt = load_elem(a.ctrl, a.dtype, pn * 48 + tid);
        for (int e = tid; e < nu * 12; e += kTensorThreads) {
            const int row = e / 12, jk = e - row * 12;
            const float* bu = s_bu + row * 4;
            float x = bu[0] * s_c[jk];
            x = fmaf(bu[1], s_c[12 + jk], x);
            x = fmaf(bu[2], s_c[24 + jk], x);
            x = fmaf(bu[3], s_c[36 + jk], x);
            s_x[e] = x;
        }
        __syncthreads();
        float4* out = reinterpret_cast<float4*>(a.out + p * pts * 3);
        for (int q = tid; q < n_quads; q += kTensorThreads) {
            const int row = q / quads_per_row;
            const int b0 = (q - row * quads_per_row) * 4;
            const float* X = s_x + row * 12;
            float r[12];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float4 bv = s_bv[b0 + m];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    float v = bv.x * X[k];
                    v = fmaf(bv.y, X[3 + k], v);
                    v = fmaf(bv.z, X[6 + k], v);
                    v = fmaf(bv.w, X[9 + k], v);
                    r[m * 3 + k] = v;
                }
            }
            float4* o = out + ((int64_t)row * nv + b0) * 3 / 4;
            o[0] = make_float4(r[0], r[1], r[2], r[3]);
            o[1] = make_float4(r[4], r[5], r[6], r[7]);
            o[2] = make_float4(r[8], r[9], r[10], r[11]);
        }
    }
}

// Fast path for small grids (nu <= 64, nv a multiple of 4): one warp per
// patch, no block barrier after the tables.  Lane l builds the isoline
// control points X[a] of rows a = l, l + 32 (12 floats each), then the warp
// sweeps the grid one row of up to 32 points at a time: lane l evaluates
// point (a, b0 + l) with Bv[b0 + l] held in registers, stages its 3 floats in
// a warp-private buffer and 24 lanes write the 384-byte row segment as float4.
__global__ void __launch_bounds__(kSurfWarps * 32, 5) k_surface_bicubic3_warp(const TensorArgs a)
{
    __shared__ float4 s_bv[kTensorMaxGrid];                   // Bv[b][0..3]
    __shared__ float4 s_bu[kSurfMaxRows];                     // Bu[a][0..3]
    __shared__ float4 s_x[kSurfWarps][kSurfMaxRows * 3];      // X[a][j][k], 12 floats per row
    __shared__ float4 s_st[kSurfWarps][2][24];                // 32 points x 3 floats, two buffers
    __shared__ float4 s_c4[kSurfWarps][12];                   // C[i][j][k]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    bernstein_table(reinterpret_cast<float*>(s_bu), a.nu, 3, tid, kSurfWarps * 32);
    bernstein_table(reinterpret_cast<float*>(s_bv), a.nv, 3, tid, kSurfWarps * 32);
    __syncthreads();

    const int nu = a.nu, nv = a.nv;
    const int64_t pts = (int64_t)nu * nv;
    const int64_t stride = (int64_t)gridDim.x * kSurfWarps;
    int64_t p = (int64_t)blockIdx.x * kSurfWarps + w;
    float c0 = 0.f, c1 = 0.f;   // this lane's control-point elements, l and 32 + l
    if (p < a.n) {
        c0 = load_elem(a.ctrl, a.dtype, p * 48 + lane);
        if (lane < 16) c1 = load_elem(a.ctrl, a.dtype, p * 48 + 32 + lane);
    }
    float* cw = reinterpret_cast<float*>(s_c4[w]);
    int buf = 0;
    for (; p < a.n; p += stride) {
        __syncwarp();  // the previous patch is done with s_c and s_x
        cw[lane] = c0;
        if (lane < 16) cw[32 + lane] = c1;
        __syncwarp();
        const int64_t pn = p + stride;  // the next patch of this warp, loaded while this one runs
        if (pn < a.n) {
            c0 = load_elem(a.ctrl, a.dtype, pn * 48 + lane);
            if (lane < 16) c1 = load_elem(a.ctrl, a.dtype, pn * 48 + 32 + lane);
        }
        const float4* cw4 = reinterpret_cast<const float4*>(cw);   // C[i][4q..4q+3] = cw4[3 i + q]
#pragma unroll 1
        for (int q = 0; q < 3; ++q) {   // columns 4q..4q+3 of the 12 per row
            const float4 k0 = cw4[q], k1 = cw4[3 + q], k2 = cw4[6 + q], k3 = cw4[9 + q];
            for (int row = lane; row < nu; row += 32) {
                const float4 bu = s_bu[row];
                float4 x;
                x.x = fmaf(bu.w, k3.x, fmaf(bu.z, k2.x, fmaf(bu.y, k1.x, bu.x * k0.x)));
                x.y = fmaf(bu.w, k3.y, fmaf(bu.z, k2.y, fmaf(bu.y, k1.y, bu.x * k0.y)));
                x.z = fmaf(bu.w, k3.z, fmaf(bu.z, k2.z, fmaf(bu.y, k1.z, bu.x * k0.z)));
                x.w = fmaf(bu.w, k3.w, fmaf(bu.z, k2.w, fmaf(bu.y, k1.w, bu.x * k0.w)));
                s_x[w][row * 3 + q] = x;
            }
        }
        __syncwarp();
        float4* out = reinterpret_cast<float4*>(a.out + p * pts * 3);
        for (int b0 = 0; b0 < nv; b0 += 32) {
            const int b = b0 + lane;
            const float4 bv = b < nv ? s_bv[b] : make_float4(0.f, 0.f, 0.f, 0.f);
            const int nvec = min(32, nv - b0) * 3 / 4;   // float4 per row segment
#pragma unroll 2
            for (int row = 0; row < nu; ++row) {
                const float4 x0 = s_x[w][row * 3], x1 = s_x[w][row * 3 + 1], x2 = s_x[w][row * 3 + 2];
                // X[row][j][k] sits at float 3 j + k of the row
                float P0 = bv.x * x0.x, P1 = bv.x * x0.y, P2 = bv.x * x0.z;
                P0 = fmaf(bv.y, x0.w, P0);
                P1 = fmaf(bv.y, x1.x, P1);
                P2 = fmaf(bv.y, x1.y, P2);
                P0 = fmaf(bv.z, x1.z, P0);
                P1 = fmaf(bv.z, x1.w, P1);
                P2 = fmaf(bv.z, x2.x, P2);
                P0 = fmaf(bv.w, x2.y, P0);
                P1 = fmaf(bv.w, x2.z, P1);
                P2 = fmaf(bv.w, x2.w, P2);
                float* st = reinterpret_cast<float*>(s_st[w][buf]);
                st[lane * 3 + 0] = P0;
                st[lane * 3 + 1] = P1;
                st[lane * 3 + 2] = P2;
                __syncwarp();
                if (lane < nvec) out[((int64_t)row * nv + b0) * 3 / 4 + lane] = s_st[w][buf][lane];
                buf ^= 1;   // the next row stages in the other buffer, so no second barrier
            }
        }
    }
}

// General grids: any degrees <= 7, dim 1..4, grid <= 256 per axis.  One warp per
// unit of work, a block of up to `rows` rows of one u slab of one volume; a
// surface is a volume of one slab (degree 0, one grid value) whose v and w are
// its u and v.  The warp forms Y[j][k][l] = sum_i Bu[i] C[i][j][l][k] and
// Z[b][k][l] = sum_j Bv[b][j] Y[j][k][l] in warp-private shared memory, l padded
// to whole float4s, then takes the rows' points in output order, 4 a lane: a
// point is L4 float4 products of Bw[c] and Z[b] a component, staged and written
// as float4s.  (The block-per-volume kernel before it wrote each row from one
// thread, 16 bytes every row length, with runtime inner loops.)  Bound by
// instruction issue (64 %) and shared memory.  A call (us, GB300): 1000 tricubic
// 3D lattices on 20 x 24 x 28 162 -> 46; 8000 on 5 x 30 x 7 147 -> 50; 30,000
// bicubic patches on 32 x 33 356 -> 95, of degree 2 x 1 261 -> 79, 5 x 5
// 364 -> 155.  4 blocks per SM (3 in 4D) measured best of 3 to 5.
constexpr int kGridRows = 32;
constexpr int kGridTile = 128;  // points a warp stages between two write-outs
constexpr int kMinUnit = 32;    // points of a unit that are worth a warp

// shared memory in floats: the tables, then each warp's C, Y, Z and stage
struct GridLayout {
    int bv, bu, warp, c, y, z, per_warp, total;
};
__host__ __device__ inline GridLayout grid_layout(const TensorArgs& a)
{
    const int lw = a.dw > 3 ? 8 : 4;
    GridLayout g;
    g.bv = a.nw * lw;
    g.bu = g.bv + a.nv * (a.dv + 1);
    g.warp = (g.bu + a.nu * (a.du + 1) + 3) & ~3;
    g.y = kGridTile * a.dim;  // after the stage
    g.z = g.y + (a.dv + 1) * a.dim * lw;
    g.c = g.z + kGridRows * a.dim * lw;
    g.per_warp = (g.c + (a.du + 1) * (a.dv + 1) * (a.dw + 1) * a.dim + 3) & ~3;
    g.total = g.warp + kSurfWarps * g.per_warp;
    return g;
}

// The units of a launch: `chunks` of `rows` rows (at most kGridRows) a slab,
// `each` a warp and one more for the first `more` warps.
struct GridUnits {
    int rows, chunks;
    int64_t each, more;
};

__device__ __forceinline__ int64_t grid_quotient(int64_t a, int b)
{
    return a >> 32 ? a / b : (int64_t)((uint32_t)a / (uint32_t)b);  // (a 64-bit division takes 0.1 us)
}

template <int L4, int DIM>
__global__ void __launch_bounds__(kSurfWarps * 32, DIM == 4 ? 3 : 4) k_grid(const TensorArgs a, const GridUnits un)
{
    constexpr int LW = 4 * L4;
    extern __shared__ float4 s_grid[];
    float* sm = reinterpret_cast<float*>(s_grid);
    const GridLayout g = grid_layout(a);
    const int tid = threadIdx.x, lane = tid & 31;
    const int du = a.du, dv = a.dv, dw = a.dw, nu = a.nu, nv = a.nv, nw = a.nw;
    // the rows of all three tables side by side (a surface's one slab has the value 1)
    const int table_rows = nw + nv + (du > 0 ? nu : 0);
    if (du == 0 && tid == 0) sm[g.bu] = 1.f;
    for (int r = tid; r < table_rows; r += kSurfWarps * 32) {
        const bool in_w = r < nw, in_v = !in_w && r < nw + nv;
        const int row = in_w ? r : in_v ? r - nw : r - nw - nv, d = in_w ? dw : in_v ? dv : du;
        const int stride = in_w ? LW : d + 1;
        bernstein_row(sm + (in_w ? 0 : in_v ? g.bv : g.bu) + row * stride, in_w ? nw : in_v ? nv : nu, d, row, stride);
    }
    __syncthreads();
    const float4* bw4 = s_grid;
    float* mine = sm + g.warp + (tid >> 5) * g.per_warp;
    float *stage = mine, *Y = mine + g.y, *Z = mine + g.z, *C = mine + g.c;
    const int ljk = (dw + 1) * DIM;  // floats of one (i, j)
    const int per = (du + 1) * (dv + 1) * ljk;
    const int q32 = 32 / nw, r32 = 32 - q32 * nw;  // 32 points on: q32 rows and r32 columns
    // a warp takes consecutive units, most of them of one volume: its control
    // points load once per volume, Y is formed once per slab
    const int64_t w = (int64_t)blockIdx.x * kSurfWarps + (tid >> 5);
    const int64_t u0 = w * un.each + min(w, un.more);
    int64_t left = un.each + (w < un.more ? 1 : 0), slab = grid_quotient(u0, un.chunks), p = grid_quotient(slab, nu);
    int64_t loaded = -1, formed = -1;
    int ch = (int)(u0 - slab * un.chunks), ai = (int)(slab - p * nu);
    for (; left > 0; --left) {
        const int b0 = ch * un.rows;
        const int rows = min(un.rows, nv - b0);
        if (p != loaded) {
            if (a.dtype == 0) {
                const float* src = static_cast<const float*>(a.ctrl) + p * per;
                for (int e = lane; e < per; e += 32) C[e] = __ldg(src + e);
            } else {
                for (int e = lane; e < per; e += 32) C[e] = load_elem(a.ctrl, a.dtype, p * per + e);
            }
            loaded = p;
            __syncwarp();
        }
        const float* bu = sm + g.bu + ai * (du + 1);
        for (int e = lane; e < (slab != formed ? (dv + 1) * DIM * LW : 0); e += 32) {
            const int j = e / (DIM * LW), k = e / LW % DIM, l = e % LW;
            float y = 0.f;
            if (l <= dw) {
                const float* src = C + j * ljk + l * DIM + k;
                for (int i = 0; i <= du; ++i) y = fmaf(bu[i], src[i * (dv + 1) * ljk], y);
            }
            Y[e] = y;
        }
        formed = slab;
        __syncwarp();
        for (int e = lane; e < rows * DIM * L4; e += 32) {
            const int b = e / (DIM * L4), r = e - b * (DIM * L4);
            const float* bv = sm + g.bv + (b0 + b) * (dv + 1);
            const float4* y4 = reinterpret_cast<const float4*>(Y) + r;
            float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int j = 0; j <= dv; ++j) {
                const float4 y = y4[j * (DIM * L4)];
                const float w = bv[j];
                z.x = fmaf(w, y.x, z.x);
                z.y = fmaf(w, y.y, z.y);
                z.z = fmaf(w, y.z, z.z);
                z.w = fmaf(w, y.w, z.w);
            }
            reinterpret_cast<float4*>(Z)[e] = z;
        }
        __syncwarp();
        const int total = rows * nw;
        float* out = a.out + ((slab * nv + b0) * (int64_t)nw) * DIM;
        int b = lane / nw, c = lane - b * nw;
        for (int t0 = 0; t0 < total; t0 += kGridTile) {
            const int cnt = min(kGridTile, total - t0);
#pragma unroll
            for (int m = 0; m < kGridTile / 32; ++m) {
                if (lane + 32 * m < cnt) {
                    const float4* z4 = reinterpret_cast<const float4*>(Z) + b * (DIM * L4);
                    float v[DIM];
#pragma unroll
                    for (int k = 0; k < DIM; ++k) v[k] = 0.f;
#pragma unroll
                    for (int q = 0; q < L4; ++q) {
                        const float4 w = bw4[c * L4 + q];
#pragma unroll
                        for (int k = 0; k < DIM; ++k) {
                            const float4 z = z4[k * L4 + q];
                            v[k] = fmaf(w.x, z.x, v[k]);
                            v[k] = fmaf(w.y, z.y, v[k]);
                            v[k] = fmaf(w.z, z.z, v[k]);
                            v[k] = fmaf(w.w, z.w, v[k]);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < DIM; ++k) stage[(lane + 32 * m) * DIM + k] = v[k];
                }
                b += q32;
                c += r32;
                if (c >= nw) {
                    c -= nw;
                    ++b;
                }
            }
            __syncwarp();
            tile_copy(out + (int64_t)t0 * DIM, stage, cnt * DIM, lane, 32);
            __syncwarp();
        }
        if (++ch == un.chunks) {
            ch = 0;
            ++slab;
            if (++ai == nu) {
                ai = 0;
                ++p;
            }
        }
    }
}

static const void* grid_kernel(int l4, int dim)
{
    switch (dim) {
    case 1: return l4 == 1 ? (const void*)k_grid<1, 1> : (const void*)k_grid<2, 1>;
    case 2: return l4 == 1 ? (const void*)k_grid<1, 2> : (const void*)k_grid<2, 2>;
    case 3: return l4 == 1 ? (const void*)k_grid<1, 3> : (const void*)k_grid<2, 3>;
    default: return l4 == 1 ? (const void*)k_grid<1, 4> : (const void*)k_grid<2, 4>;
    }
}

// The shared memory of a block-per-patch form of the contraction, which bounds
// the grids that are accepted (200 KB).
size_t tensor_smem_bytes(const TensorArgs& a)
{
    if (a.dw < 0) {
        return sizeof(float) * ((size_t)a.nu * (a.du + 1) + (size_t)a.nv * (a.dv + 1) +
                                (size_t)(a.du + 1) * (a.dv + 1) * a.dim + (size_t)a.nu * (a.dv + 1) * a.dim +
                                (size_t)kTensorThreads * a.dim);
    }
    const size_t lk = (size_t)(a.dw + 1) * a.dim;
    return sizeof(float) * ((size_t)a.nu * (a.du + 1) + (size_t)a.nv * (a.dv + 1) + (size_t)a.nw * (a.dw + 1) +
                            (size_t)(a.du + 1) * (a.dv + 1) * lk + (size_t)a.nu * (a.dv + 1) * lk +
                            (size_t)a.nu * a.nv * lk);
}

static TensorArgs to_args(const TensorLaunch& t)
{
    TensorArgs a;
    a.ctrl = t.ctrl;
    a.dtype = t.dtype;
    a.n = t.n;
    a.du = t.du;
    a.dv = t.dv;
    a.dw = t.dw;
    a.dim = t.dim;
    a.nu = t.nu;
    a.nv = t.nv;
    a.nw = t.nw;
    a.out = t.out;
    a.vparts = 1;
    return a;
}

size_t tensor_product_smem(const TensorLaunch& t) { return tensor_smem_bytes(to_args(t)); }

LaunchResult launch_tensor_product(const TensorLaunch& t, cudaStream_t s, const LaunchHooks& h)
{
    TensorArgs a = to_args(t);
    const void* kern;
    size_t smem = 0;
    int threads = kTensorThreads;
    int64_t work = a.n;
    GridUnits un{kGridRows, 1, 0, 0};
    const bool bicubic3 = a.dw < 0 && a.du == 3 && a.dv == 3 && a.dim == 3 && a.nv % 4 == 0 &&
                          ((uintptr_t)a.out & 15) == 0;
    const bool tricubic1 = a.dw == 3 && a.du == 3 && a.dv == 3 && a.dim == 1 && a.nu <= kVolMaxRows &&
                           a.nw % 4 == 0 && ((uintptr_t)a.out & 15) == 0;
    const bool general = !bicubic3 && !tricubic1;
    if (bicubic3 && a.nu <= kSurfMaxRows) {
        kern = (const void*)k_surface_bicubic3_warp;
        threads = kSurfWarps * 32;
        work = (a.n + kSurfWarps - 1) / kSurfWarps;
    } else if (tricubic1) {
        kern = (const void*)k_volume_tricubic1_warp<VOL_U_CORES>;
        threads = kSurfWarps * 32;
        a.vparts = volume_parts(a.n, a.nu, h.sm_count);
        work = (a.n * a.vparts + kSurfWarps - 1) / kSurfWarps;
    } else if (bicubic3) {
        kern = (const void*)k_surface_bicubic3;
    } else {
        if (a.dw < 0) {  // a surface: one slab, u and v in the places of v and w
            a.dw = a.dv;
            a.nw = a.nv;
            a.dv = a.du;
            a.nv = a.nu;
            a.du = 0;
            a.nu = 1;
        }
        kern = grid_kernel(a.dw > 3 ? 2 : 1, a.dim);
        threads = kSurfWarps * 32;
        // fewer rows a unit while 32 leave the SMs short of warps (us on GB300, block per
        // patch before k_grid / always 32 rows / now: one biquadratic patch on 16 x 256
        // 15.3 / 16.6 / 4.7, 64 of 31 x 31 6.6 / 8.9 / 3.9, 256 of 32 x 33 7.8 / 8.5 / 7.0,
        // 16 of degree 5 x 4, 1D, 31 x 31 5.5 / 9.4 / 4.1)
        const int64_t target = (int64_t)h.sm_count * 12;
        un.rows = a.nv < kGridRows ? a.nv : kGridRows;
        auto units = [&] { return a.n * a.nu * ((a.nv + un.rows - 1) / un.rows); };
        while (un.rows > 1 && (un.rows + 1) / 2 * a.nw >= kMinUnit && units() < target) un.rows = (un.rows + 1) / 2;
        un.chunks = (a.nv + un.rows - 1) / un.rows;
        work = (units() + kSurfWarps - 1) / kSurfWarps;
        smem = (size_t)grid_layout(a).total * sizeof(float);
        if (smem > 48 * 1024) {
            // the most a launch of this kernel takes, so that calls on several
            // threads never lower one another's limit
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            if (e != cudaSuccess) return {0, e};
        }
    }
    const int grid = persistent_grid(kern, threads, smem, h.sm_count, work);
    if (general) {
        const int64_t units = a.n * a.nu * un.chunks, warps = (int64_t)grid * kSurfWarps;
        un.each = units / warps;
        un.more = units % warps;
    }
    const SurfTexArgs no_tex{};  // the CUDA-core volume kernel reads no texture
    void* args[] = {(void*)&a, general ? (void*)&un : (void*)&no_tex};
    h.count(h.self);
    h.begin(h.self, s);
    cudaError_t e = cudaLaunchKernel(kern, dim3(grid), dim3(threads), args, smem, s);
    h.end(h.self, s);
    return {1, e};
}

}  // namespace bez
