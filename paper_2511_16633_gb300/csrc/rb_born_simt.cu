// Plain-FP32 (CUDA-core) Born contractions.
//
// Adjoint and Gauss-Newton diagonal (per frequency w, S = W o R), both symmetric in emitter
// and receiver, so only r <= e is multiplied out (blocks of 32 elements):
//   U[e][x] = sum_{r <= e} T[e][r] conj(G_r(x)),   g(x) = w^2 sum_e conj(G_e(x)) U[e][x]
//   V[e][x] = sum_{r <= e} Y[e][r] |G_r(x)|^2,     H(x) = w^4 sum_e |G_e(x)|^2 V[e][x]
// with T = S + S^T, Y = W + W^T below the block diagonal and T = S, Y = W inside the
// diagonal blocks.  One CTA owns a tile of 32 pixels: it synthesises G_t(x) for every
// element and the tile's pixels into shared memory (Eqs. 4-5), runs both contractions with
// T and Y streamed through shared memory, and reduces over e in a fixed order, so g and H
// never need U or V in HBM and every pixel's result is independent of scheduling.  Rings below
// 48 elements take the full sums over r instead (k_adjoint_small).
//
// Forward: d[e][r] = w^2 sum_x G_e(x) G_r(x) m(x), symmetric in (e, r).  G of the frequency is
// synthesised once into a buffer; split-K over pixel chunks: CTA (tile pair, chunk)
// accumulates a 64x64 block of the upper triangle; a second kernel sums the chunk partials
// in a fixed order and mirrors the block.
#include "rb_internal.cuh"

namespace {

constexpr int AP = 32;     // pixels per adjoint tile
constexpr int EB = 32;     // elements per block of the triangle
constexpr int AT = 256;    // threads per adjoint CTA: 4 r groups x 8 element groups x 8 pixel groups

// G tile synthesis: Gs[t][p] for t < n_pad, p < AP (zero beyond npix and beyond n).
__device__ __forceinline__ void synth_tile(const GeoDev& G, const rb_cell* __restrict__ tables, const float* __restrict__ c,
                                           const FreqC& F, int p0, int n_pad, float2* Gs) {
    const int n = G.n_elem;
    for (int idx = threadIdx.x; idx < n_pad * AP; idx += blockDim.x) {
        const int t = idx / AP, p = idx % AP;
        const int pix = p0 + p;
        float2 v = make_float2(0.f, 0.f);
        if (t < n && pix < G.npix) {
            const rb_cell rec = tables[(size_t)t * G.npix + pix];
            const int ix = pix % G.nx, iy = pix / G.nx;
            if (rec.tkey != RB_HOLE) {
                DF ex, ey;
                elem_pos(G, t, ex, ey);
                const DF dist = pixel_elem_dist(G, ix, iy, ex, ey);
                v = green_eval(rec, __ldg(c + pix), dist, F, G.j_floor);
            }
        }
        Gs[t * AP + p] = v;
    }
}

// The operand of the adjoint, per frequency, element block eb and r < 32 (eb + 1), for the 32
// elements e of the block side by side: {Re T, Im T, Y, 0} (zero beyond n).
__global__ void __launch_bounds__(256) k_prep_sym(int n, int nb, const float2* __restrict__ Rs, const uint8_t* __restrict__ Ws,
                                                  float4* __restrict__ out) {
    const int eb = blockIdx.x, fw = blockIdx.y, n_pad = nb * EB;
    const float2* R = Rs + (size_t)fw * n * n;
    const uint8_t* W = Ws + (size_t)fw * n * n;
    float4* o = out + ((size_t)fw * nb + eb) * n_pad * EB;
    for (int idx = blockIdx.z * blockDim.x + threadIdx.x; idx < EB * (eb + 1) * EB; idx += gridDim.z * blockDim.x) {
        const int r = idx / EB, e = eb * EB + idx % EB;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < n && r < n) {
            if (W[(size_t)e * n + r]) {
                const float2 s = R[(size_t)e * n + r];
                v = make_float4(s.x, s.y, 1.f, 0.f);
            }
            if (r / EB < eb && W[(size_t)r * n + e]) {
                const float2 s = R[(size_t)r * n + e];
                v.x += s.x;
                v.y += s.y;
                v.z += 1.f;
            }
        }
        o[idx] = v;
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// The 32 parts of g and H of a tile's pixels (part q of this thread's pixels 4 tx .. 4 tx + 3),
// added in order by the pixels' threads, out, and into their sums over the set.
__device__ __forceinline__ void sum_parts(const GeoDev& G, const FreqC& fc, int fw, int p0, int tx, int q, const float pg_r[4],
                                          const float pg_i[4], const float ph[4], float* red, float2* __restrict__ g_out,
                                          float* __restrict__ h_out, float& acc_g, float& acc_h) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int p = tx * 4 + j;
        red[(q * AP + p) * 3 + 0] = pg_r[j];
        red[(q * AP + p) * 3 + 1] = pg_i[j];
        red[(q * AP + p) * 3 + 2] = ph[j];
    }
    __syncthreads();
    if (threadIdx.x < AP) {
        const int p = threadIdx.x;
        float sr = 0.f, si = 0.f, sh = 0.f;
        for (int k = 0; k < 32; ++k) {
            sr += red[(k * AP + p) * 3 + 0];
            si += red[(k * AP + p) * 3 + 1];
            sh += red[(k * AP + p) * 3 + 2];
        }
        sr *= fc.w2;
        si *= fc.w2;
        sh *= fc.w4;
        const int pix = p0 + p;
        if (pix < G.npix) {
            if (g_out) g_out[(size_t)fw * G.npix + pix] = make_float2(sr, si);
            if (h_out) h_out[(size_t)fw * G.npix + pix] = sh;
        }
        acc_g += sr;
        acc_h += sh;
    }
}
__device__ __forceinline__ void store_sums(const GeoDev& G, int p0, float acc_g, float acc_h, float* __restrict__ gsum,
                                           float* __restrict__ hsum) {
    const int pix = p0 + (int)threadIdx.x;
    if (threadIdx.x >= AP || pix >= G.npix) return;
    if (gsum) gsum[pix] = acc_g;
    if (hsum) hsum[pix] = acc_h;
}

// Chunks of 32 r x 32 e (16 KB) go through two shared-memory buffers (cp.async); of each
// chunk, the CTA's four groups of 64 threads take 8 r each, and a thread accumulates 4
// elements x 4 pixels of U and V over its group's r.  g and H are linear in U and V, so the
// groups' parts meet only in the final sums.  Bound by the FP32 pipe and issue: 88 FMAs per 6
// shared-memory loads.  100 elements, 251 x 237 pixels: 370 -> 219 us; 150 elements, 260 x
// 243, two frequencies: 2553 -> 637 us (the full sums, rows of T loaded one by one).
__global__ void __launch_bounds__(AT, 2) k_adjoint_simt(GeoDev G, const rb_cell* __restrict__ tables, const float* __restrict__ c,
                                                        FreqSet F, const float4* __restrict__ sym, float2* __restrict__ g_out,
                                                        float* __restrict__ h_out, float* __restrict__ gsum,
                                                        float* __restrict__ hsum) {
    extern __shared__ float4 smem4[];
    const int n = G.n_elem, nb = (n + EB - 1) / EB, n_pad = nb * EB;
    float4* St = smem4;                              // [2][32 r][32 e]
    float2* Gs = (float2*)(smem4 + 2 * EB * EB);     // [n_pad][AP]
    float* red = (float*)St;                         // [32][AP][3], reuses the chunk buffers after the r loop
    const int tx = threadIdx.x & 7;                  // pixel group: pixels tx*4 .. tx*4+3
    const int ty = (threadIdx.x >> 3) & 7;           // element group: e = ty*4 .. ty*4+3 of the block
    const int tz = threadIdx.x >> 6;                 // r group: 8 tz .. 8 tz + 7 of a chunk
    const int p0 = blockIdx.x * AP;
    const int n_chunks = nb * (nb + 1) / 2;
    float acc_g = 0.f, acc_h = 0.f;                  // running sums over w (threads < AP)

    for (int fw = 0; fw < F.n; ++fw) {
        const FreqC& fc = F.f[fw];
        const float4* sw = sym + (size_t)fw * nb * n_pad * EB;
        auto load = [&](int eb, int rb, int buf) {
            const float4* src = sw + ((size_t)eb * n_pad + (size_t)rb * EB) * EB;
            for (int k = threadIdx.x; k < EB * EB; k += AT) cp_async16(St + buf * EB * EB + k, src + k);
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        __syncthreads();   // the previous frequency's sums are out of the buffers
        load(0, 0, 0);
        synth_tile(G, tables, c, fc, p0, n_pad, Gs);
        float pg_r[4], pg_i[4], ph[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) pg_r[j] = pg_i[j] = ph[j] = 0.f;
        float ur[4][4], ui[4][4], vv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) ur[i][j] = ui[i][j] = vv[i][j] = 0.f;
        int eb = 0, rb = 0;
        for (int ch = 0; ch < n_chunks; ++ch) {
            const int eb1 = rb == eb ? eb + 1 : eb, rb1 = rb == eb ? 0 : rb + 1;   // the next chunk
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();   // chunk ch has landed for everyone, and chunk ch - 1 is no longer read
            if (ch + 1 < n_chunks) load(eb1, rb1, (ch + 1) & 1);
            const float4* S = St + (ch & 1) * EB * EB + 8 * tz * EB + 4 * ty;
            const float4* gq = (const float4*)(Gs + (size_t)(rb * EB + 8 * tz) * AP + tx * 4);
#pragma unroll 4
            for (int rr = 0; rr < 8; ++rr) {
                const float4 g01 = gq[rr * (AP / 2)], g23 = gq[rr * (AP / 2) + 1];
                const float br[4] = {g01.x, g01.z, g23.x, g23.z};
                const float bi[4] = {-g01.y, -g01.w, -g23.y, -g23.w};   // conj(G_r)
                float a2[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) a2[j] = br[j] * br[j] + bi[j] * bi[j];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 s = S[rr * EB + i];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        ur[i][j] = fmaf(s.x, br[j], fmaf(-s.y, bi[j], ur[i][j]));
                        ui[i][j] = fmaf(s.x, bi[j], fmaf(s.y, br[j], ui[i][j]));
                        vv[i][j] = fmaf(s.z, a2[j], vv[i][j]);
                    }
                }
            }
            if (rb == eb) {
                // the block's U and V are complete (this group's part): into g and H
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4* ge = (const float4*)(Gs + (size_t)(eb * EB + 4 * ty + i) * AP + tx * 4);
                    const float4 g01 = ge[0], g23 = ge[1];
                    const float gx[4] = {g01.x, g01.z, g23.x, g23.z}, gy[4] = {g01.y, g01.w, g23.y, g23.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        pg_r[j] += gx[j] * ur[i][j] + gy[j] * ui[i][j];   // conj(G_e) U
                        pg_i[j] += gx[j] * ui[i][j] - gy[j] * ur[i][j];
                        ph[j] += (gx[j] * gx[j] + gy[j] * gy[j]) * vv[i][j];
                        ur[i][j] = ui[i][j] = vv[i][j] = 0.f;
                    }
                }
            }
            eb = eb1;
            rb = rb1;
        }
        __syncthreads();   // every thread is done with the buffers that red reuses
        sum_parts(G, fc, fw, p0, tx, tz * 8 + ty, pg_r, pg_i, ph, red, g_out, h_out, acc_g, acc_h);
    }
    store_sums(G, p0, acc_g, acc_h, gsum, hsum);
}

// The full sums over r, for the rings whose padding to blocks of 32 would cost more than the
// symmetric sums save: S and W go through shared memory eight r at a time, and a thread
// accumulates the elements ty + 32 i, i < EPT, at 4 pixels.
constexpr int RC = 8;        // r-chunk of S / W staged in shared memory
constexpr int RCP = RC + 1;  // padded row (conflict-free reads by the 4 element rows of a warp)
template <int EPT>
__global__ void __launch_bounds__(AT) k_adjoint_small(GeoDev G, const rb_cell* __restrict__ tables, const float* __restrict__ c,
                                                      FreqSet F, const float2* __restrict__ resid, const uint8_t* __restrict__ w,
                                                      float2* __restrict__ g_out, float* __restrict__ h_out,
                                                      float* __restrict__ gsum, float* __restrict__ hsum) {
    extern __shared__ float4 smem4[];
    const int n = G.n_elem;
    float2* Gs = (float2*)smem4;                 // [n][AP]
    float2* Ss = Gs + (size_t)n * AP;            // [n][RCP]
    float* Ws = (float*)(Ss + (size_t)n * RCP);  // [n][RCP]
    float* red = (float*)Ss;                     // [32][AP][3], reuses the S / W staging after the r loop
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;   // pixels tx*4 .. tx*4+3
    const int p0 = blockIdx.x * AP;
    float acc_g = 0.f, acc_h = 0.f;
    for (int fw = 0; fw < F.n; ++fw) {
        const FreqC& fc = F.f[fw];
        const float2* Rw = resid + (size_t)fw * n * n;
        const uint8_t* Ww = w + (size_t)fw * n * n;
        __syncthreads();   // the previous frequency's sums are out of the staging
        synth_tile(G, tables, c, fc, p0, n, Gs);
        float ur[EPT][4], ui[EPT][4], vv[EPT][4];
#pragma unroll
        for (int i = 0; i < EPT; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) ur[i][j] = ui[i][j] = vv[i][j] = 0.f;
        for (int r0 = 0; r0 < n; r0 += RC) {
            __syncthreads();
            for (int idx = threadIdx.x; idx < n * RC; idx += blockDim.x) {
                const int e = idx / RC, rr = idx % RC, r = r0 + rr;
                const bool used = r < n && Ww[(size_t)e * n + r];
                Ss[e * RCP + rr] = used ? Rw[(size_t)e * n + r] : make_float2(0.f, 0.f);
                Ws[e * RCP + rr] = used ? 1.f : 0.f;
            }
            __syncthreads();
            const int rmax = min(RC, n - r0);
            for (int rr = 0; rr < rmax; ++rr) {
                const float4* gp = (const float4*)(Gs + (size_t)(r0 + rr) * AP + tx * 4);
                const float4 g01 = gp[0], g23 = gp[1];
                const float br[4] = {g01.x, g01.z, g23.x, g23.z};
                const float bi[4] = {-g01.y, -g01.w, -g23.y, -g23.w};   // conj(G_r)
                float a2[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) a2[j] = br[j] * br[j] + bi[j] * bi[j];
#pragma unroll
                for (int i = 0; i < EPT; ++i) {
                    const int e = ty + 32 * i;
                    const float2 s = e < n ? Ss[e * RCP + rr] : make_float2(0.f, 0.f);
                    const float wv = e < n ? Ws[e * RCP + rr] : 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        ur[i][j] = fmaf(s.x, br[j], fmaf(-s.y, bi[j], ur[i][j]));
                        ui[i][j] = fmaf(s.x, bi[j], fmaf(s.y, br[j], ui[i][j]));
                        vv[i][j] = fmaf(wv, a2[j], vv[i][j]);
                    }
                }
            }
        }
        float pg_r[4], pg_i[4], ph[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) pg_r[j] = pg_i[j] = ph[j] = 0.f;
#pragma unroll
        for (int i = 0; i < EPT; ++i) {
            const int e = ty + 32 * i;
            if (e >= n) continue;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 ge = Gs[(size_t)e * AP + tx * 4 + j];
                pg_r[j] += ge.x * ur[i][j] + ge.y * ui[i][j];   // conj(G_e) U
                pg_i[j] += ge.x * ui[i][j] - ge.y * ur[i][j];
                ph[j] += (ge.x * ge.x + ge.y * ge.y) * vv[i][j];
            }
        }
        __syncthreads();   // every thread is done with the staging that red reuses
        sum_parts(G, fc, fw, p0, tx, ty, pg_r, pg_i, ph, red, g_out, h_out, acc_g, acc_h);
    }
    store_sums(G, p0, acc_g, acc_h, gsum, hsum);
}

// ---------------------------------------------------------------------------
// Forward
// ---------------------------------------------------------------------------
constexpr int FT = 64;      // element tile
constexpr int FS = FT + 2;  // padded row of a sub-tile (16-byte aligned)
// Threads of a forward CTA (64 rows over threads / 16 of them: 8 or 4 x 4 complex outputs a thread)
// and pixels per sub-tile.  Where the CTAs synthesise G, half their time goes by waiting for its
// special functions, and the scratch of a call without a workspace holds too few chunks for more
// than one or two CTAs an SM: twice the threads each (256 elements, 256 x 256 pixels: 2320 us,
// 3340 with 128 threads; 1000 elements, 128 x 120: 6817 and 10887; 64 elements, 64 x 64: 33 and 42).
constexpr int fwd_threads(bool from_g) { return from_g ? 128 : 256; }
constexpr int fwd_pixels(bool from_g) { return from_g ? 16 : 32; }

// FROM_G: G of the frequency comes from the buffer g [n_elem][npix]; otherwise (no workspace)
// it is synthesised from the tables, once per tile pair that uses it.  Bound by the FP32
// pipe: 128 FMAs per pixel and thread for 6 shared-memory loads.  150 elements, 260 x 243
// pixels: 416 us and 72 for G (1189 us with a 4 x 4 tile a thread and G synthesised for every
// pair, half the time the synthesis).
template <bool FROM_G>
__global__ void __launch_bounds__(fwd_threads(FROM_G)) k_forward_simt(GeoDev G, const float2* __restrict__ g, const rb_cell* __restrict__ tables,
                                                       const float* __restrict__ c, FreqC F, const float* __restrict__ m,
                                                       float2* __restrict__ partial, int n_chunks) {
    constexpr int FTHR = fwd_threads(FROM_G), FP = fwd_pixels(FROM_G), ER = FT * 16 / FTHR;   // rows e a thread
    __shared__ __align__(16) float2 Ae[FP][FS];   // G_e(x) m(x), transposed [p][e]
    __shared__ __align__(16) float2 Br[FP][FS];   // G_r(x)
    const int n = G.n_elem;
    const int nt = (n + FT - 1) / FT;
    // decode the upper-triangular tile pair from blockIdx.x
    int pair = blockIdx.x, te = 0;
    while (pair >= nt - te) { pair -= nt - te; ++te; }
    const int tr = te + pair;
    const int chunk = blockIdx.y;
    const int pix_per = (G.npix + n_chunks - 1) / n_chunks;
    const int pbeg = min(G.npix, chunk * pix_per), pend = min(G.npix, pbeg + pix_per);
    const int e0 = te * FT, r0 = tr * FT;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float ar[ER][4], ai[ER][4];
#pragma unroll
    for (int i = 0; i < ER; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) ar[i][j] = ai[i][j] = 0.f;

    for (int ps = pbeg; ps < pend; ps += FP) {
        __syncthreads();
#pragma unroll 4
        for (int idx = threadIdx.x; idx < 2 * FT * FP; idx += FTHR) {
            const int which = idx / (FT * FP);
            const int rem = idx % (FT * FP);
            const int tl = rem / FP, p = rem % FP;
            const int t = (which == 0 ? e0 : r0) + tl;
            const int pix = ps + p;
            float2 v = make_float2(0.f, 0.f);
            if (t < n && pix < pend) {
                if (FROM_G) {
                    v = g[(size_t)t * G.npix + pix];
                } else {
                    const rb_cell rec = tables[(size_t)t * G.npix + pix];
                    if (rec.tkey != RB_HOLE) {
                        const int ix = pix % G.nx, iy = pix / G.nx;
                        DF ex, ey;
                        elem_pos(G, t, ex, ey);
                        v = green_eval(rec, __ldg(c + pix), pixel_elem_dist(G, ix, iy, ex, ey), F, G.j_floor);
                    }
                }
                if (which == 0) {
                    // a hole (G = 0) adds 0 whatever m holds there, which 0 x NaN or 0 x inf would not
                    const float mv = __ldg(m + pix);
                    const bool any = v.x != 0.f || v.y != 0.f;
                    v.x = any ? v.x * mv : 0.f;
                    v.y = any ? v.y * mv : 0.f;
                }
            }
            if (which == 0) Ae[p][tl] = v; else Br[p][tl] = v;
        }
        __syncthreads();
        const int np = min(FP, pend - ps);
#pragma unroll 2
        for (int p = 0; p < np; ++p) {
            float4 a4[ER / 2], b4[2];
#pragma unroll
            for (int i = 0; i < ER / 2; ++i) a4[i] = *(const float4*)&Ae[p][ty * ER + 2 * i];
#pragma unroll
            for (int i = 0; i < 2; ++i) b4[i] = *(const float4*)&Br[p][tx * 4 + 2 * i];
            const float bx[4] = {b4[0].x, b4[0].z, b4[1].x, b4[1].z}, by[4] = {b4[0].y, b4[0].w, b4[1].y, b4[1].w};
#pragma unroll
            for (int i = 0; i < ER; ++i) {
                const float ax = (i & 1) ? a4[i >> 1].z : a4[i >> 1].x, ay = (i & 1) ? a4[i >> 1].w : a4[i >> 1].y;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    ar[i][j] = fmaf(ax, bx[j], fmaf(-ay, by[j], ar[i][j]));
                    ai[i][j] = fmaf(ax, by[j], fmaf(ay, bx[j], ai[i][j]));
                }
            }
        }
    }
    // partial[chunk][e][r] for this block (upper-triangle tile pairs only)
    float2* out = partial + (size_t)chunk * n * n;
#pragma unroll
    for (int i = 0; i < ER; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int e = e0 + ty * ER + i, r = r0 + tx * 4 + j;
            if (e < n && r < n) out[(size_t)e * n + r] = make_float2(ar[i][j], ai[i][j]);
        }
}

// d[e][r] = w^2 sum_chunk partial (fixed order), entries right of the diagonal tiles mirrored
// into the lower triangle; optional sum of W |d|^2 into per-block partials.  A CTA takes 32
// consecutive r of one e at a time; its 8 warps take every eighth chunk, warp 0 adds the
// warps' sums in order.  YS = 1, for up to eight chunks: a warp takes 32 entries by itself,
// in the same order (1000 elements, 16 x 15 pixels, the whole forward in one chunk: 270 us by
// eight warps with their barriers a run, 140 so).
template <int YS>
__global__ void __launch_bounds__(256) k_forward_reduce(GeoDev G, FreqC F, const float2* __restrict__ partial, int n_chunks,
                                                        float2* __restrict__ d_out, const uint8_t* __restrict__ w,
                                                        double* __restrict__ den_part) {
    __shared__ float2 s_sum[8][32];
    __shared__ double s_den[8];
    const int n = G.n_elem, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, y = wid % YS, nrb = (n + 31) / 32;
    const size_t total = (size_t)n * n;
    double acc = 0.0;
    constexpr int TPB = 8 / YS;   // runs of 32 entries a CTA takes at a time
    for (int tile0 = blockIdx.x * TPB; tile0 < n * nrb; tile0 += gridDim.x * TPB) {
        const int tile = tile0 + wid / YS;
        const int e = tile / nrb, rb = tile - e * nrb, r = 32 * rb + lane;
        const int te = e / FT, tr = 32 * rb / FT;   // a 32-entry run lies in one tile
        if (e >= n || tr < te) continue;            // YS = 8: the whole CTA's run
        float sr = 0.f, si = 0.f;
        if (r < n) {
            // eight chunks ahead: a chunk's load goes out as the one eight before it is added
            const float2* src = partial + (size_t)e * n + r;
            float2 nx[8];
            auto load = [&](int k, int ch) {
                nx[k] = ch < n_chunks ? __ldcg(src + (size_t)ch * total) : make_float2(0.f, 0.f);
            };
#pragma unroll
            for (int k = 0; k < 8; ++k) load(k, y + k * YS);
            for (int ch = y; ch < n_chunks; ch += 8 * YS) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    sr += nx[k].x;
                    si += nx[k].y;
                    load(k, ch + (8 + k) * YS);
                }
            }
        }
        if (YS > 1) {
            __syncthreads();
            s_sum[y][lane] = make_float2(sr, si);
            __syncthreads();
        }
        if (y == 0 && r < n) {
            for (int k = 1; k < YS; ++k) {
                sr += s_sum[k][lane].x;
                si += s_sum[k][lane].y;
            }
            sr *= F.w2;
            si *= F.w2;
            const size_t er = (size_t)e * n + r, re = (size_t)r * n + e;
            const bool mirror = te < tr;
            if (d_out) {
                d_out[er] = make_float2(sr, si);
                if (mirror) d_out[re] = make_float2(sr, si);
            }
            if (w) {
                const int cnt = (w[er] ? 1 : 0) + ((mirror && w[re]) ? 1 : 0);
                if (cnt) acc += cnt * ((double)sr * sr + (double)si * si);
            }
        }
    }
    if (den_part) {
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) s_den[wid] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < 8; ++k) acc += s_den[k];   // 0 from the warps that only helped
            den_part[blockIdx.x] = acc;
        }
    }
}

// Green's functions of one frequency from the tables, g[t][pixel], for the plain forward.
// Bound by the 24 bytes an entry it reads and writes; a CTA stays on 256 pixels and goes
// through the elements with the grid's second dimension, so that neither the entry's index
// nor the pixel's row takes a division per entry.
__global__ void __launch_bounds__(256) k_green_out(GeoDev G, const rb_cell* __restrict__ tables,
                                                   const float* __restrict__ c, FreqC F, float2* __restrict__ g) {
    const int pix = blockIdx.x * blockDim.x + threadIdx.x;
    if (pix >= G.npix) return;
    const int iy = pix / G.nx, ix = pix - iy * G.nx;
    const float cv = __ldg(c + pix);
    for (int t = blockIdx.y; t < G.n_elem; t += gridDim.y) {
        const size_t j = (size_t)t * G.npix + pix;
        DF ex, ey;
        elem_pos(G, t, ex, ey);
        g[j] = green_eval(tables[j], cv, pixel_elem_dist(G, ix, iy, ex, ey), F, G.j_floor);
    }
}

}  // namespace

size_t simt_sym_bytes(int n_elem) {
    const size_t np = (size_t)((n_elem + EB - 1) / EB) * EB;
    return np * np * sizeof(float4);
}

cudaError_t launch_adjoint_simt(const GeoDev& G, const rb_cell* tables, const float* c, const FreqSet& F,
                                const float2* resid, const uint8_t* w, float2* g_out, float* h_out, float* gsum,
                                float* hsum, void* sym, cudaStream_t s) {
    if (!simt_adjoint_supported(G.n_elem)) return cudaErrorInvalidValue;
    const int n = G.n_elem, nb = (n + EB - 1) / EB;
    const int blocks = (G.npix + AP - 1) / AP;
    // Rings below 48 elements take the full sums.  Measured at 512 x 500 pixels, symmetric against
    // full: 8 elements 134 and 59 us, 20: 178 and 123, 32: 203 and 179, 33: 330 and 261, 44: 360
    // and 343, 48: 363 and 368, 60: 403 and 473; at 64 x 64 pixels, 8 elements: 17 and 13 (the
    // operand's own launch).
    if (n < 48) {
        size_t stage = (size_t)n * RCP * (sizeof(float2) + sizeof(float));
        if (stage < (size_t)32 * AP * 3 * sizeof(float)) stage = (size_t)32 * AP * 3 * sizeof(float);
        const size_t sm = (size_t)n * AP * sizeof(float2) + stage;   // 29 KB at most
        if (n <= 32) k_adjoint_small<1><<<blocks, AT, sm, s>>>(G, tables, c, F, resid, w, g_out, h_out, gsum, hsum);
        else k_adjoint_small<2><<<blocks, AT, sm, s>>>(G, tables, c, F, resid, w, g_out, h_out, gsum, hsum);
        return cudaGetLastError();
    }
    k_prep_sym<<<dim3(nb, F.n, 8), 256, 0, s>>>(n, nb, resid, w, (float4*)sym);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t sm = (size_t)2 * EB * EB * sizeof(float4) + (size_t)nb * EB * AP * sizeof(float2);
    e = cudaFuncSetAttribute(k_adjoint_simt, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_adjoint_simt<<<blocks, AT, sm, s>>>(G, tables, c, F, (const float4*)sym, g_out, h_out, gsum, hsum);
    return cudaGetLastError();
}

// the adjoint holds a 32-pixel tile of G for every element in shared memory beside its two
// chunk buffers: rings of up to 512 elements
bool simt_adjoint_supported(int n_elem) { return n_elem >= 2 && n_elem <= 512; }

// Pixel chunks of the forward: as many as give every SM ten CTAs over the tile pairs, none
// below 32 pixels (chunks of 2048 pixels whatever the ring left 64 elements on 64 x 64
// pixels to two CTAs, 905 us, and 150 elements on 260 x 243 to 186), and none above 2048 up to
// 512 x 512 pixels (128 chunks beyond): the rounding of an accumulator grows with its run, and
// large rings have CTAs enough with few chunks (512 elements, 512 x 512 pixels, relative L2
// error against 64 bits: 9.8e-7 in 42 runs of 6242 pixels, 5.4e-7 in 128 of 2048).
int rb_fwd_chunks_for(int n_elem, int npix) {
    const int nt = (n_elem + FT - 1) / FT, pairs = nt * (nt + 1) / 2;
    const int most = (npix + 31) / 32, fill = 1520 / pairs < most ? 1520 / pairs : most;
    int run = (npix + 2047) / 2048;
    if (run > 128) run = 128;
    return fill > run ? fill : run;
}

cudaError_t launch_forward_simt(const GeoDev& G, const rb_cell* tables, const float* c, const FreqC& F, const float* m,
                                float2* g_buf, float2* partial, int n_chunks, cudaStream_t s) {
    const int nt = (G.n_elem + FT - 1) / FT;
    const dim3 grid(nt * (nt + 1) / 2, n_chunks);
    if (!g_buf) {
        k_forward_simt<false><<<grid, fwd_threads(false), 0, s>>>(G, nullptr, tables, c, F, m, partial, n_chunks);
        return cudaGetLastError();
    }
    const int bx = (G.npix + 255) / 256;
    int by = (4864 + bx - 1) / bx;   // 32 CTAs an SM: four waves of eight
    if (by > G.n_elem) by = G.n_elem;
    k_green_out<<<dim3(bx, by), 256, 0, s>>>(G, tables, c, F, g_buf);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_forward_simt<true><<<grid, fwd_threads(true), 0, s>>>(G, g_buf, tables, c, F, m, partial, n_chunks);
    return cudaGetLastError();
}

cudaError_t launch_forward_reduce(const GeoDev& G, const FreqC& F, const float2* partial, int n_chunks, float2* d_out,
                                  const uint8_t* w, double* den_part, cudaStream_t s) {
    if (n_chunks <= 8) k_forward_reduce<1><<<256, 256, 0, s>>>(G, F, partial, n_chunks, d_out, w, den_part);
    else k_forward_reduce<8><<<256, 256, 0, s>>>(G, F, partial, n_chunks, d_out, w, den_part);
    return cudaGetLastError();
}
