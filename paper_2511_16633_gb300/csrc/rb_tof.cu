// Time-of-flight initial guess (Sec. 4: a few linearisations of a ToF reconstruction
// that fits measured times of flight with times of flight along rays).
//
// One linearisation is one SIRT step in slowness s = 1/c along the current rays:
//   ds = D_col^-1 L^T D_row^-1 dT,   dT[e][r] = T_obs - T(c) on the rows used,
// where row (e, r) of L is (1 - lam) times the path of ray i plus lam times the
// path of ray i + 1 of its first-arrival link (the linked time interpolates the two
// rays' times with the same weights), a path integral is the sum over the ray's
// vertex-to-vertex segments of the segment length times the bilinear interpolant at
// the segment midpoint, D_row are the row sums (interpolated path lengths) and D_col
// the column sums.  The per-row mean slowness error dT / D_row is clamped to
// +-2e-3 s/m; rows: receivers on the opposite ~75 % of the ring, linked both in
// the data and in the current medium.  c <- 1 / (1/c + ds) on the support where
// D_col > 0.
//
// Kernels: k_tof_len (path length per ray), k_tof_coef (per fan: each ray's total
// weight sum_r w and weighted error sum_r w dT / D_row, gathered in a fixed order),
// k_tof_bp (per ray: the two coefficients spread along its segments into pixel sums),
// k_tof_apply, and k_tof_resid / k_tof_rms for the RMS ToF misfit.  The pixel sums are
// 64-bit fixed-point atomics, so they do not depend on the order of arrival.
#include <math.h>

#include "rb_internal.cuh"

namespace {

constexpr float TOF_A_MAX = 2e-3f;    // clamp of the per-row mean slowness error [s/m]
constexpr int RT = 256;
constexpr int RB = 256;

__device__ __forceinline__ bool row_used(int e, int r, int N, int gap) {
    int d = e > r ? e - r : r - e;
    d = min(d, N - d);
    return d >= gap;
}

__device__ __forceinline__ float fp_diff(float vh, float vl, float oh, float ol) {
    return __fadd_rn(__fsub_rn(vh, oh), __fsub_rn(vl, ol));
}

// Position of a vertex (the first half of its record), and of the next one minus it.
__device__ __forceinline__ float4 load_pos(const Vtx* __restrict__ p) { return __ldg(reinterpret_cast<const float4*>(p)); }

// One thread's piece of work: steps [k0 + 1, k1] of ray i of fan t.  Neighbouring threads
// take neighbouring rays at the same steps, so their vertices are contiguous.
constexpr int TOF_KC = 64;
struct TofPiece { int t, i, k0, k1; };
__device__ __forceinline__ bool tof_piece(const GeoDev& G, const rb_ray_end* __restrict__ ends, int n_pieces, TofPiece* w) {
    const long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long g = u / G.n_rays;
    if (g >= (long long)G.n_elem * n_pieces) return false;
    w->i = (int)(u - g * G.n_rays);
    w->t = (int)(g / n_pieces);
    w->k0 = (int)(g - (long long)w->t * n_pieces) * TOF_KC;
    const int nv = ends[(size_t)w->t * G.n_rays + w->i].n_vert;
    w->k1 = min(nv - 1, w->k0 + TOF_KC);
    return w->k1 > w->k0;
}

// Path length of every ray: the sum of its vertex-to-vertex segment lengths, in double and in
// order along the ray (segments of equal length bring the sum close to ties of the float it
// is kept in, and a length one ulp off moves the whole guess).  One thread per ray, eight
// vertices loaded ahead; with one load a step waited for, 260 us against 126 for 256
// elements, 256 rays, 256 x 256 pixels.
__global__ void __launch_bounds__(64) k_tof_len(GeoDev G, const Vtx* __restrict__ verts, const rb_ray_end* __restrict__ ends,
                                                float* __restrict__ len) {
    const long long ray = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (ray >= (long long)G.n_elem * G.n_rays) return;
    const int t = (int)(ray / G.n_rays), i = (int)(ray % G.n_rays);
    const int last = ends[ray].n_vert - 1;
    double acc = 0.0;
    if (last > 0) {
        const size_t step = (size_t)G.n_rays;
        const Vtx* v = verts + vtx_index(G, t, 0, i);
        float4 a = load_pos(v), b[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) b[j] = load_pos(v + step * (size_t)min(1 + j, last));
        for (int k = 1; k <= last; k += 8) {
            float4 c[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) c[j] = load_pos(v + step * (size_t)min(k + 8 + j, last));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float dx = fp_diff(b[j].x, b[j].y, a.x, a.y), dy = fp_diff(b[j].z, b[j].w, a.z, a.w);
                if (k + j <= last) acc += (double)sqrtf(dx * dx + dy * dy);
                a = b[j];
                b[j] = c[j];
            }
        }
    }
    len[ray] = (float)acc;
}

// Per fan e: the rows' mean slowness errors, then per ray i the weighted error a_i and the
// total weight b_i of the rows that use it (receivers scanned in index order); the largest
// |a| and b (as float bits, an order-independent maximum) set the fixed-point scales.
__global__ void __launch_bounds__(RT) k_tof_coef(GeoDev G, const LinkRec* __restrict__ lrec,
                                                 const double* __restrict__ t_obs, const uint8_t* __restrict__ obs_linked,
                                                 const float* __restrict__ len, float2* __restrict__ coef,
                                                 uint32_t* __restrict__ amax) {
    extern __shared__ unsigned char smem[];
    const int N = G.n_elem, n = G.n_rays, e = blockIdx.x;
    int* sb = (int*)smem;                   // [N] winning interval (-1: row not used)
    float* sl = (float*)(sb + N);           // [N] lam
    float* se = sl + N;                     // [N] mean slowness error
    const int gap = (N + 7) / 8;
    for (int r = threadIdx.x; r < N; r += RT) {
        const size_t o = (size_t)e * N + r;
        const LinkRec L = lrec[o];
        int b = -1;
        float lam = 0.f, err = 0.f;
        if (L.i >= 0 && obs_linked[o] && row_used(e, r, N, gap)) {
            lam = L.lam;
            const double drow = (1.0 - (double)lam) * (double)len[(size_t)e * n + L.i] +
                                (double)lam * (double)len[(size_t)e * n + L.i + 1];
            if (drow > 0.0) {
                b = L.i;
                const double m = (t_obs[o] - L.T) / drow;
                err = fminf(fmaxf((float)m, -TOF_A_MAX), TOF_A_MAX);
            }
        }
        sb[r] = b;
        sl[r] = lam;
        se[r] = err;
    }
    __syncthreads();
    float am = 0.f, bm = 0.f;
    for (int i = threadIdx.x; i < n; i += RT) {
        float a = 0.f, w = 0.f;
        for (int r = 0; r < N; ++r) {
            const int b = sb[r];
            if (b == i) {
                a = fmaf(1.f - sl[r], se[r], a);
                w += 1.f - sl[r];
            } else if (b == i - 1) {
                a = fmaf(sl[r], se[r], a);
                w += sl[r];
            }
        }
        coef[(size_t)e * n + i] = make_float2(a, w);
        am = fmaxf(am, fabsf(a));
        bm = fmaxf(bm, w);
    }
    if (am > 0.f) atomicMax(&amax[0], __float_as_uint(am));
    if (bm > 0.f) atomicMax(&amax[1], __float_as_uint(bm));
}

// A pixel's weight in a ray's path, in units of 2^-52 of the power of two at or above ds
// (scale: 2^30 over it), as fine as a sum in double: exact for float weights down to 2^-29 of it.
__device__ __forceinline__ unsigned long long fix_weight(float w, float scale) {
    const float t = w * scale;
    const uint32_t hi = (uint32_t)t;
    const uint32_t lo = __float2uint_rn((t - (float)hi) * 4194304.f);   // the fraction, exact, times 2^22
    return ((unsigned long long)hi << 22) + lo;
}

// A coefficient (in units of the largest one times ds over that power of two, / 2^52) times a
// weight, into a pixel sum in units of the largest coefficient x ds / 2^40, rounded to one unit:
// the product over 2^64.  |a| <= 2^53 and a piece's weights are 64 x 2^52 at most.
__device__ __forceinline__ void deposit(unsigned long long* __restrict__ dst, long long a, unsigned long long w) {
    const long long y = (long long)w;
    const long long q = __mul64hi(a, y) + (long long)(((unsigned long long)a * w) >> 63);
    if (q != 0) atomicAdd(dst, (unsigned long long)q);
}

// a_i and b_i of a ray spread along a piece of its segments into the pixel sums, in fixed
// point.  A thread keeps the weights of the four pixels of the ray's current bilinear quad
// and deposits a pixel when the ray leaves it (a move to a neighbouring quad keeps the two
// shared pixels).  Measured for 256 elements, 256 rays, 256 x 256 pixels: one thread per
// ray with all four pixels deposited at each move, their weights and products in double,
// 1774 us, most of it on the FP64 pipe (2 lanes a cycle and SM); 460 us so.
__global__ void __launch_bounds__(128) k_tof_bp(GeoDev G, const Vtx* __restrict__ verts, const rb_ray_end* __restrict__ ends,
                                                int n_pieces, const float2* __restrict__ coef,
                                                const uint32_t* __restrict__ amax, float wscale, double cscale,
                                                unsigned long long* __restrict__ num, unsigned long long* __restrict__ den) {
    TofPiece w;
    if (!tof_piece(G, ends, n_pieces, &w)) return;
    const float2 cf = coef[(size_t)w.t * G.n_rays + w.i];
    if (cf.x == 0.f && cf.y == 0.f) return;
    const float am = __uint_as_float(amax[0]), bm = __uint_as_float(amax[1]);
    const long long ca = am > 0.f ? __double2ll_rn((double)cf.x / (double)am * cscale) : 0;
    const long long cb = bm > 0.f ? __double2ll_rn((double)cf.y / (double)bm * cscale) : 0;
    unsigned long long w00 = 0, w10 = 0, w01 = 0, w11 = 0;
    int qi = -1, qj = -1;
    auto put = [&](int di, int dj, unsigned long long& wt) {
        if (wt == 0) return;
        const int px = (qj + dj) * G.nx + qi + di;
        deposit(num + px, ca, wt);
        deposit(den + px, cb, wt);
        wt = 0;
    };
    const size_t step = (size_t)G.n_rays;
    const Vtx* v = verts + vtx_index(G, w.t, w.k0, w.i);
    float4 a = load_pos(v), b = load_pos(v + step);
    for (int k = w.k0 + 1; k <= w.k1; ++k) {
        v += step;
        const float4 nx = load_pos(k < w.k1 ? v + step : v);   // in time for the next round
        const float dx = fp_diff(b.x, b.y, a.x, a.y), dy = fp_diff(b.z, b.w, a.z, a.w);
        const float l = sqrtf(dx * dx + dy * dy);
        const float mx = (a.x + a.y) + 0.5f * dx, my = (a.z + a.w) + 0.5f * dy;
        const float fu0 = fminf(fmaxf(fmaf(mx, G.inv_h, G.cxg), 0.f), (float)(G.nx - 1));
        const float fv0 = fminf(fmaxf(fmaf(my, G.inv_h, G.cyg), 0.f), (float)(G.ny - 1));
        const int i0 = min((int)fu0, G.nx - 2), j0 = min((int)fv0, G.ny - 2);
        const float fu = fu0 - (float)i0, fv = fv0 - (float)j0;
        const int di = i0 - qi, dj = j0 - qj;
        if ((di | dj) != 0) {
            if (abs(di) > 1 || abs(dj) > 1) {   // not a neighbour (or the piece's first quad)
                put(0, 0, w00);
                put(1, 0, w10);
                put(0, 1, w01);
                put(1, 1, w11);
            }
            if (di == 1) {
                put(0, 0, w00);
                put(0, 1, w01);
                w00 = w10; w01 = w11; w10 = w11 = 0;
            } else if (di == -1) {
                put(1, 0, w10);
                put(1, 1, w11);
                w10 = w00; w11 = w01; w00 = w01 = 0;
            }
            qi = i0;
            if (dj == 1) {
                put(0, 0, w00);
                put(1, 0, w10);
                w00 = w01; w10 = w11; w01 = w11 = 0;
            } else if (dj == -1) {
                put(0, 1, w01);
                put(1, 1, w11);
                w01 = w00; w11 = w10; w00 = w10 = 0;
            }
            qj = j0;
        }
        w00 += fix_weight((1.f - fu) * (1.f - fv) * l, wscale);
        w10 += fix_weight(fu * (1.f - fv) * l, wscale);
        w01 += fix_weight((1.f - fu) * fv * l, wscale);
        w11 += fix_weight(fu * fv * l, wscale);
        a = b;
        b = nx;
    }
    put(0, 0, w00);
    put(1, 0, w10);
    put(0, 1, w01);
    put(1, 1, w11);
}

__device__ __forceinline__ bool in_support_px(const GeoDev& G, int pix) {
    const int ix = pix % G.nx, iy = pix / G.nx;
    const long long jx = 2LL * ix - (G.nx - 1), jy = 2LL * iy - (G.ny - 1);
    return jx * jx + jy * jy <= G.r2max;
}

__global__ void __launch_bounds__(RT) k_tof_apply(GeoDev G, float* __restrict__ c, const unsigned long long* __restrict__ num,
                                                  const unsigned long long* __restrict__ den,
                                                  const uint32_t* __restrict__ amax) {
    const float am = __uint_as_float(amax[0]), bm = __uint_as_float(amax[1]);
    for (int p = blockIdx.x * RT + threadIdx.x; p < G.npix; p += gridDim.x * RT) {
        const long long dq = (long long)den[p];
        if (dq <= 0 || !in_support_px(G, p)) continue;
        // num / den back in physical units: (nq am ds / 2^40) / (dq bm ds / 2^40)
        const double ds = ((double)(long long)num[p] * (double)am) / ((double)dq * (double)bm);
        c[p] = (float)(1.0 / (1.0 / (double)c[p] + ds));
    }
}

// partial sums of dT^2 and of the row count over the rows used
__global__ void __launch_bounds__(RT) k_tof_resid(GeoDev G, const LinkRec* __restrict__ lrec,
                                                  const double* __restrict__ t_obs,
                                                  const uint8_t* __restrict__ obs_linked, double* __restrict__ part) {
    const int N = G.n_elem, gap = (N + 7) / 8;
    double s2 = 0.0, cnt = 0.0;
    for (long long o = (long long)blockIdx.x * RT + threadIdx.x; o < (long long)N * N; o += (long long)RB * RT) {
        const int e = (int)(o / N), r = (int)(o % N);
        const LinkRec L = lrec[o];
        if (L.i >= 0 && obs_linked[o] && row_used(e, r, N, gap)) {
            const double d = t_obs[o] - L.T;
            s2 += d * d;
            cnt += 1.0;
        }
    }
    __shared__ double a[RT], b[RT];
    a[threadIdx.x] = s2;
    b[threadIdx.x] = cnt;
    __syncthreads();
    for (int k = RT / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) {
            a[threadIdx.x] += a[threadIdx.x + k];
            b[threadIdx.x] += b[threadIdx.x + k];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[blockIdx.x] = a[0];
        part[RB + blockIdx.x] = b[0];
    }
}

__global__ void __launch_bounds__(RT) k_tof_rms(const double* __restrict__ part, double* __restrict__ out) {
    __shared__ double a[RT], b[RT];
    a[threadIdx.x] = part[threadIdx.x];
    b[threadIdx.x] = part[RB + threadIdx.x];
    __syncthreads();
    for (int k = RT / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) {
            a[threadIdx.x] += a[threadIdx.x + k];
            b[threadIdx.x] += b[threadIdx.x + k];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = b[0] > 0.0 ? sqrt(a[0] / b[0]) : 0.0;
}

__global__ void __launch_bounds__(RT) k_tof_times_out(int n2, const LinkRec* __restrict__ lrec, double* __restrict__ t_out) {
    for (int o = blockIdx.x * RT + threadIdx.x; o < n2; o += gridDim.x * RT) t_out[o] = lrec[o].i >= 0 ? lrec[o].T : 0.0;
}

}  // namespace

size_t tof_ws_bytes(int n_elem, int n_rays, int npix) {
    auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
    return al((size_t)n_elem * n_elem * sizeof(LinkRec)) + al((size_t)n_elem * n_rays * 4) +
           al((size_t)n_elem * n_rays * 8) + 2 * al((size_t)npix * 8) + 256;
}

namespace {
struct TofWs {
    LinkRec* lrec;
    float* len;
    float2* coef;
    unsigned long long* num;
    unsigned long long* den;
    uint32_t* amax;
};
TofWs carve(const GeoDev& G, void* base) {
    auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
    char* p = (char*)base;
    TofWs w;
    w.lrec = (LinkRec*)p;
    p += al((size_t)G.n_elem * G.n_elem * sizeof(LinkRec));
    w.len = (float*)p;
    p += al((size_t)G.n_elem * G.n_rays * 4);
    w.coef = (float2*)p;
    p += al((size_t)G.n_elem * G.n_rays * 8);
    w.num = (unsigned long long*)p;
    p += al((size_t)G.npix * 8);
    w.den = (unsigned long long*)p;
    p += al((size_t)G.npix * 8);
    w.amax = (uint32_t*)p;
    return w;
}
}  // namespace

cudaError_t launch_tof_link(const GeoDev& G, const float* c, const rb_ray_end* ends, void* tof_ws, uint8_t* linked,
                            cudaStream_t s) {
    FreqSet F;
    F.n = 0;
    return launch_link(G, c, ends, F, nullptr, linked, s, carve(G, tof_ws).lrec);
}

cudaError_t launch_tof_times_out(const GeoDev& G, void* tof_ws, double* t_out, cudaStream_t s) {
    k_tof_times_out<<<RB, RT, 0, s>>>(G.n_elem * G.n_elem, carve(G, tof_ws).lrec, t_out);
    return cudaGetLastError();
}

cudaError_t launch_tof_resid(const GeoDev& G, void* tof_ws, const double* t_obs, const uint8_t* obs_linked,
                             double* part, double* out, cudaStream_t s) {
    k_tof_resid<<<RB, RT, 0, s>>>(G, carve(G, tof_ws).lrec, t_obs, obs_linked, part);
    k_tof_rms<<<1, RT, 0, s>>>(part, out);
    return cudaGetLastError();
}

// one SIRT step on the current rays (vertices in verts, links in the ToF workspace)
cudaError_t launch_tof_step(const GeoDev& G, const Vtx* verts, const rb_ray_end* ends, void* tof_ws, const double* t_obs,
                            const uint8_t* obs_linked, float* c, cudaStream_t s) {
    const TofWs w = carve(G, tof_ws);
    const int n_pieces = (G.max_steps + TOF_KC - 1) / TOF_KC;
    const long long blocks = ((long long)G.n_elem * n_pieces * G.n_rays + 127) / 128;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const int rb = (int)blocks;
    const long long rays = (long long)G.n_elem * G.n_rays;
    k_tof_len<<<(int)((rays + 63) / 64), 64, 0, s>>>(G, verts, ends, w.len);
    cudaError_t e = cudaMemsetAsync(w.num, 0, (size_t)((char*)w.amax - (char*)w.num) + 8, s);
    if (e != cudaSuccess) return e;
    const size_t sm = (size_t)G.n_elem * 12;
    if (sm > 48 * 1024) {
        e = cudaFuncSetAttribute(k_tof_coef, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    k_tof_coef<<<G.n_elem, RT, sm, s>>>(G, w.lrec, t_obs, obs_linked, w.len, w.coef, w.amax);
    int ex = 0;
    const double mant = frexp(G.ds_d, &ex);   // ds = mant 2^ex, mant in [0.5, 1)
    k_tof_bp<<<rb, 128, 0, s>>>(G, verts, ends, n_pieces, w.coef, w.amax, (float)ldexp(1.0, 30 - ex),
                                4503599627370496.0 / mant, w.num, w.den);
    k_tof_apply<<<RB, RT, 0, s>>>(G, c, w.num, w.den, w.amax);
    return cudaGetLastError();
}
