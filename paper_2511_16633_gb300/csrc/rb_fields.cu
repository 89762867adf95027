// Field preparation: element positions and the cell-packed derivative grids
// that the ray integrator samples.
//
// The Eikonal characteristics (Eq. 6) need c and grad c along a ray and the
// dynamic ray tracing that solves the Transport equation (Eq. 7) needs the
// Hessian of c.  Discretisation: first derivatives by central differences
// over index-clamped neighbours (one-sided at the grid edge); second
// derivatives c_xx, c_yy by the three-point stencil centred at the nearest
// interior pixel; c_xy by the mixed central difference over clamped
// neighbours.  Each grid is sampled by bilinear interpolation.
//
// Layout: one 128-byte record per grid cell (i0, j0), i0 < nx-1, j0 < ny-1,
// holding for each of c, c_x, c_y, c_xx, c_xy, c_yy, alpha0 the coefficients
// (a, b, c, d) of its bilinear interpolant a + b u + c v + d u v over the cell
// (u, v in [0, 1]), from the corner values q00 = (i0, j0), q10, q01, q11:
// a = q00, b = q10 - q00, c = q01 - q00, d = q11 - q10 - q01 + q00.  The fields go
// in pairs (c, c_x), (c_y, c_xx), (c_xy, c_yy), two float4 per pair:
// {a_F, a_G, b_F, b_G}, {c_F, c_G, d_F, d_G}, so that the sampler evaluates a pair
// with packed two-lane FMAs; then alpha0's {a, b, c, d} and a pad.  A ray that enters
// a cell loads one aligned 128-byte line and keeps it in registers until it leaves
// the cell.
#include "rb_internal.cuh"

__device__ __forceinline__ void put_elem_position(const GeoDev& G, float4* xy, int t) {
    double phi = 2.0 * RB_PI_D * (double)t / (double)G.n_elem;
    double s, c;
    sincos(phi, &s, &c);
    const DF x = df_from_double(G.R_d * c), y = df_from_double(G.R_d * s);
    xy[t] = make_float4(x.hi, x.lo, y.hi, y.lo);
}

__global__ void k_elem_positions(GeoDev G, float4* xy) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < G.n_elem) put_elem_position(G, xy, t);
}

cudaError_t launch_elem_positions(const GeoDev& G, float4* elem_xy, cudaStream_t s) {
    k_elem_positions<<<(G.n_elem + 127) / 128, 128, 0, s>>>(G, elem_xy);
    return cudaGetLastError();
}

struct PixF { float c, cx, cy, cxx, cxy, cyy; };

__device__ __forceinline__ PixF pixel_fields(const float* __restrict__ c, int nx, int ny, float h, int ix, int iy) {
    const int ip = min(ix + 1, nx - 1), im = max(ix - 1, 0);
    const int jp = min(iy + 1, ny - 1), jm = max(iy - 1, 0);
    const int ic = min(max(ix, 1), nx - 2), jc = min(max(iy, 1), ny - 2);
    auto C = [&](int i, int j) { return __ldg(c + (size_t)j * nx + i); };
    const float dxs = (float)(ip - im) * h, dys = (float)(jp - jm) * h;
    const float ih2 = 1.0f / (h * h);
    PixF f;
    f.c = C(ix, iy);
    f.cx = (C(ip, iy) - C(im, iy)) / dxs;
    f.cy = (C(ix, jp) - C(ix, jm)) / dys;
    f.cxx = (C(ic + 1, iy) - 2.0f * C(ic, iy) + C(ic - 1, iy)) * ih2;
    f.cyy = (C(ix, jc + 1) - 2.0f * C(ix, jc) + C(ix, jc - 1)) * ih2;
    f.cxy = ((C(ip, jp) - C(ip, jm)) - (C(im, jp) - C(im, jm))) / (dxs * dys);
    return f;
}

// A CTA takes FT_X x FT_Y cells: it first puts the pixel fields of the (FT_X + 1) x
// (FT_Y + 1) pixels at their corners into shared memory (a thread that forms the four corners
// of its own cell does each pixel's eleven loads and three divisions four times), then each
// thread writes its cell's record with four 32-byte stores.  What is left is the write of the
// records, 128 bytes a cell.  CTAs past the cells write the element positions, which saves
// that launch.  With one thread per cell on its own, 16-byte stores and a launch of its own
// for the positions, 26 us (512 x 512 pixels, 256 elements); the whole call of ray tracing
// and linking went from 1224 to 1161 us with this form.
constexpr int FT_X = 32, FT_Y = 8, FT_N = FT_X * FT_Y;

__global__ void __launch_bounds__(FT_N) k_fields(GeoDev G, const float* __restrict__ c, const float* __restrict__ a0,
                                                 float4* __restrict__ cells, int tiles_x, int n_tiles, float4* exy) {
    if ((int)blockIdx.x >= n_tiles) {
        const int t = ((int)blockIdx.x - n_tiles) * FT_N + (int)threadIdx.x;
        if (t < G.n_elem) put_elem_position(G, exy, t);
        return;
    }
    __shared__ float S[7][FT_Y + 1][FT_X + 1];
    const int x0 = ((int)blockIdx.x % tiles_x) * FT_X, y0 = ((int)blockIdx.x / tiles_x) * FT_Y;
    for (int q = threadIdx.x; q < (FT_X + 1) * (FT_Y + 1); q += FT_N) {
        const int lx = q % (FT_X + 1), ly = q / (FT_X + 1), ix = x0 + lx, iy = y0 + ly;
        if (ix >= G.nx || iy >= G.ny) continue;   // no cell has this corner
        const PixF f = pixel_fields(c, G.nx, G.ny, G.h, ix, iy);
        S[0][ly][lx] = f.c;
        S[1][ly][lx] = f.cx;
        S[2][ly][lx] = f.cy;
        S[3][ly][lx] = f.cxx;
        S[4][ly][lx] = f.cxy;
        S[5][ly][lx] = f.cyy;
        S[6][ly][lx] = __ldg(a0 + (size_t)iy * G.nx + ix);
    }
    __syncthreads();
    const int ncx = G.nx - 1, ncy = G.ny - 1;
    const int lx = threadIdx.x % FT_X, ly = threadIdx.x / FT_X, i0 = x0 + lx, j0 = y0 + ly;
    if (i0 >= ncx || j0 >= ncy) return;
    float4* o = cells + ((size_t)j0 * ncx + i0) * 8;
    auto coef = [&](int k) {
        const float q00 = S[k][ly][lx], q10 = S[k][ly][lx + 1], q01 = S[k][ly + 1][lx], q11 = S[k][ly + 1][lx + 1];
        return make_float4(q00, q10 - q00, q01 - q00, (q11 - q10) - (q01 - q00));
    };
#pragma unroll
    for (int k = 0; k < 6; k += 2) {
        const float4 f = coef(k), g = coef(k + 1);
        stg32(o + k, make_float4(f.x, g.x, f.y, g.y), make_float4(f.z, g.z, f.w, g.w));
    }
    stg32(o + 6, coef(6), make_float4(0.f, 0.f, 0.f, 0.f));
}

cudaError_t launch_fields(const GeoDev& G, const float* c, const float* alpha0, float4* cells, float4* elem_xy,
                          cudaStream_t s) {
    const int tx = (G.nx - 1 + FT_X - 1) / FT_X, ty = (G.ny - 1 + FT_Y - 1) / FT_Y;
    const int pos = elem_xy ? (G.n_elem + FT_N - 1) / FT_N : 0;
    k_fields<<<tx * ty + pos, FT_N, 0, s>>>(G, c, alpha0, cells, tx, tx * ty, elem_xy);
    return cudaGetLastError();
}
