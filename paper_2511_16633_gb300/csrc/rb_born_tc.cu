// Tensor-core (tcgen05, BF16 x3 split products, FP32 accumulation in TMEM) Born
// adjoint and Gauss-Newton Hessian diagonal, and Born forward.
//
// Adjoint, per frequency w and tile of 128 pixels x (the MMA's M rows).  Both sums are
// symmetric in emitter and receiver, so only r <= e is multiplied out:
//   g(x) = w^2 sum_e conj(G_e(x)) U_e(x),   U_e = sum_{r <= e} T[e][r] conj(G_r),  S = W o R
//   H(x) = w^4 sum_e |G_e(x)|^2 V_e(x),     V_e = sum_{r <= e} Y[e][r] |G_r|^2
// with T = S + S^T and Y = W + W^T below the block diagonal (blocks of 8 elements for T,
// of 32 for Y) and T = S, Y = W inside the diagonal blocks: half the products of the full
// sums, the same value.
//   U[x][e'] = sum_k' A[x][k'] B[e'][k'],   k' = 2r + {0: Re, 1: Im},  A = (Re G_r, -Im G_r)
//   e' = 16 (e / 8) + e % 8:      B = (Re T[e][r], -Im T[e][r])  ->  Re U_e
//   e' = 16 (e / 8) + 8 + e % 8:  B = (Im T[e][r],  Re T[e][r])  ->  Im U_e
// Each operand is split into bf16 hi + lo and the products hi*hi + hi*lo + lo*hi
// (U) or hi*Y + lo*Y (V, Y in {0, 1, 2} is exact in bf16) accumulate in fp32 in TMEM, which
// keeps ~2^-16 relative accuracy per product.
#include <cuda.h>

#include "rb_internal.cuh"
#include "rb_tc.cuh"

namespace {

constexpr int TP = RB_TP;               // pixels per tile = MMA M
constexpr uint32_t kMaxTries = 1u << 22; // mbarrier polls before giving up (each poll suspends briefly)

// The adjoint takes the elements e in passes of ne = min(n, 256) (the accumulators of one
// pass fit TMEM); pass q covers e in [q ne, (q + 1) ne) and sums over r < (q + 1) ne.  Its
// K slices of 8 elements r: slices j < q ne / 8 lie below the block diagonal and feed all
// 2 ne columns; slice d = j - q ne / 8 on the diagonal feeds the columns from 16 d on.
// Likewise the V slices of 32 elements r and the columns from 32 d on.
struct AdjShape {
    int n, ne, ge, gv;                  // elements; per pass: elements, groups of 8, blocks of 32
    __host__ __device__ explicit AdjShape(int n_) : n(n_), ne(n_ < 256 ? n_ : 256), ge(ne / 8), gv(ne / 32) {}
    // rows e' of U slice j (rows e of V slice i) in pass q
    __host__ __device__ int u_rows(int q, int j) const { return 2 * ne - 16 * (j > q * ge ? j - q * ge : 0); }
    __host__ __device__ int v_rows(int q, int i) const { return ne - 32 * (i > q * gv ? i - q * gv : 0); }
    // bytes of the images before slice j of pass q (64 bytes a row: U hi and lo of 16 K values, V 32 K values)
    __host__ __device__ size_t u_off(int q, int j) const {
        size_t rows = 0;
        for (int p = 0; p < q; ++p) rows += (size_t)p * ge * 2 * ne + (size_t)ge * 2 * ne - 8u * (size_t)ge * (ge - 1);
        const int full = j < q * ge ? j : q * ge, d = j - full;
        rows += (size_t)full * 2 * ne + (size_t)d * 2 * ne - (d > 0 ? 8u * (size_t)d * (d - 1) : 0u);
        return rows * 64;
    }
    __host__ __device__ size_t v_off(int q, int i) const {
        size_t rows = 0;
        for (int p = 0; p < q; ++p) rows += (size_t)p * gv * ne + (size_t)gv * ne - 16u * (size_t)gv * (gv - 1);
        const int full = i < q * gv ? i : q * gv, d = i - full;
        rows += (size_t)full * ne + (size_t)d * ne - (d > 0 ? 16u * (size_t)d * (d - 1) : 0u);
        return rows * 64;
    }
};

// ---------------------------------------------------------------------------
// B operand images of every frequency of a set, in the core-matrix layouts of rb_tc.cuh,
// each slice holding the rows its pass multiplies and the slices packed in pass order:
//   bu: [pass, slice of 8 elements r][hi|lo][rows e' x 16]   (tile16_offset)
//   bw: [pass, slice of 32 elements r][rows e x 32]           (chunk_offset)
// CTA (slice, frequency, quarter); a thread takes one row's 4 (U) or 8 (V) elements r and
// writes its 16-byte core rows; one launch for all frequencies (four launches of 6.5 us
// each, one bf16 per store, before).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_prep_b(int n, const float2* __restrict__ Rs, const uint8_t* __restrict__ Ws,
                                                unsigned char* __restrict__ img, size_t img_stride, size_t w_off) {
    const AdjShape sh(n);
    const float2* R = Rs + (size_t)blockIdx.y * n * n;
    const uint8_t* W = Ws + (size_t)blockIdx.y * n * n;
    unsigned char* out = img + (size_t)blockIdx.y * img_stride;
    const int npass = n / sh.ne, nu = sh.ge * npass * (npass + 1) / 2;
    const bool is_v = (int)blockIdx.x >= nu;
    const int per = is_v ? sh.gv : sh.ge;   // slices added per pass
    int j = (int)blockIdx.x - (is_v ? nu : 0), q = 0;
    while (j >= per * (q + 1)) j -= per * ++q;
    if (!is_v) {
        const int rows = sh.u_rows(q, j), cnt = rows / 2, e0 = (q + 1) * sh.ne - cnt;
        unsigned char* dst = out + sh.u_off(q, j);
        for (int idx = blockIdx.z * blockDim.x + threadIdx.x; idx < 2 * cnt; idx += gridDim.z * blockDim.x) {
            const int el = idx % cnt, kc = idx / cnt, e = e0 + el;
            uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int r = 8 * j + 4 * kc + k;
                float2 s = make_float2(0.f, 0.f);
                if (W[(size_t)e * n + r]) s = R[(size_t)e * n + r];
                if ((e >> 3) > j && W[(size_t)r * n + e]) {
                    const float2 t = R[(size_t)r * n + e];
                    s.x += t.x;
                    s.y += t.y;
                }
                __nv_bfloat16 xh, xl, yh, yl;
                tc::split_bf16(s.x, xh, xl);
                tc::split_bf16(s.y, yh, yl);
                rh[k] = bf16_pack2(xh, __hneg(yh));
                rl[k] = bf16_pack2(xl, __hneg(yl));
                ih[k] = bf16_pack2(yh, xh);
                il[k] = bf16_pack2(yl, xl);
            }
            const uint32_t row = 16u * (uint32_t)(el >> 3) + (uint32_t)(el & 7);
            const uint32_t o = tc::tile16_offset(row, 8u * (uint32_t)kc), lo = (uint32_t)rows * 32u;
            *(uint4*)(dst + o) = make_uint4(rh[0], rh[1], rh[2], rh[3]);
            *(uint4*)(dst + lo + o) = make_uint4(rl[0], rl[1], rl[2], rl[3]);
            *(uint4*)(dst + o + tc::kRowGroupBytes16) = make_uint4(ih[0], ih[1], ih[2], ih[3]);
            *(uint4*)(dst + lo + o + tc::kRowGroupBytes16) = make_uint4(il[0], il[1], il[2], il[3]);
        }
    } else {
        const int rows = sh.v_rows(q, j), e0 = (q + 1) * sh.ne - rows;
        unsigned char* dst = out + w_off + sh.v_off(q, j);
        for (int idx = blockIdx.z * blockDim.x + threadIdx.x; idx < 4 * rows; idx += gridDim.z * blockDim.x) {
            const int el = idx % rows, core = idx / rows, e = e0 + el;
            uint32_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int r = 32 * j + 8 * core + k;
                v[k] = W[(size_t)e * n + r] ? 1u : 0u;
                if ((e >> 5) > j && W[(size_t)r * n + e]) ++v[k];
                v[k] = v[k] == 0u ? 0u : (v[k] == 1u ? 0x3f80u : 0x4000u);   // bf16 0, 1, 2
            }
            *(uint4*)(dst + tc::chunk_offset((uint32_t)el, 8u * (uint32_t)core)) =
                make_uint4(v[0] | v[1] << 16, v[2] | v[3] << 16, v[4] | v[5] << 16, v[6] | v[7] << 16);
        }
    }
}

constexpr int ADJ_MAX_ENT = 384;   // schedule entries of a pixel tile (372 for 1024 elements)
constexpr int ADJ_MAX_WORK = 24;   // work records of a quad and pixel tile (six a pass)

// One schedule entry (a pipeline stage): U slices j .. j + cnt - 1 or V slice j, and for a
// diagonal one the diagonal index d = j - (first diagonal slice of the pass).
struct AdjEnt {
    uint32_t v;
    static __host__ __device__ AdjEnt make(int j, int cnt, bool is_v, bool first, int d) {
        return AdjEnt{(uint32_t)j | (uint32_t)cnt << 8 | (is_v ? 1u << 11 : 0u) | (first ? 1u << 12 : 0u) |
                      (d >= 0 ? 1u << 16 | (uint32_t)d << 17 : 0u)};
    }
    __host__ __device__ uint32_t j() const { return v & 0xffu; }
    __host__ __device__ uint32_t cnt() const { return (v >> 8) & 7u; }
    __host__ __device__ bool is_v() const { return (v & (1u << 11)) != 0u; }
    __host__ __device__ bool first() const { return (v & (1u << 12)) != 0u; }   // first entry of its pass
    __host__ __device__ bool diag() const { return (v & (1u << 16)) != 0u; }
    __host__ __device__ uint32_t d() const { return v >> 17; }                    // 0 below the diagonal
};

// One piece of a quad's work: U unit u (groups 2u, 2u + 1 of the pass) or V slice u.  a, b:
// where the unit's two A slices (V: its stage, in a) are staged: stage ordinal (entry
// number mod NST) | KB offset << 4 | arrivals per warp << 12 | full barrier (first group
// of the entry) << 16; b = 0 when both slices are in one entry, whose second offset is
// then in off2.
struct AdjWork {
    uint32_t x, a, b, off2;
    __host__ __device__ uint32_t u() const { return x & 0xffu; }
    __host__ __device__ uint32_t q() const { return (x >> 8) & 7u; }
    __host__ __device__ bool is_v() const { return (x & (1u << 11)) != 0u; }
    __host__ __device__ bool first() const { return (x & (1u << 12)) != 0u; }   // the quad's first of its pass
    __host__ __device__ bool last() const { return (x & (1u << 13)) != 0u; }    // its last of the pass
    __host__ __device__ bool low() const { return (x & (1u << 14)) != 0u; }     // its last unit in columns V takes over
};

struct TcArgs {
    GeoDev G;
    const __nv_bfloat16* aimg; // [n_freq][tiles][hi|lo][2n / 8 rows][1024] A image (layout: aimg_put4)
    size_t aimg_stride;        // bf16 elements per frequency
    const unsigned char* bu;   // [n_freq][image]
    const unsigned char* bw;   // [n_freq][image]
    size_t b_stride;           // bytes per frequency
    __nv_bfloat16* vimg;       // [gridDim.x][2][n / 32][hi|lo][TP x 32] |G|^2 A slices of the Hessian contraction
    float2* g_out;             // [n_freq][npix] or null
    float* h_out;              // [n_freq][npix] or null
    float2* fpart;             // [n_freq][npix] (Re g, H) of each frequency for k_adjoint_sums, or null
    uint32_t* counters;
    float w2[RB_MAX_FREQ], w4[RB_MAX_FREQ];
    int n_freq, n_tiles;
    int want_h;                // the Hessian contraction is wanted (h_out or hsum set)
    uint32_t tmem_cols, v_col; // TMEM columns; first column of V (U has columns 0 .. 2 ne - 1)
    int low_groups;            // groups of U whose columns V overwrites (0: V has columns of its own)
    int n_ent, n_work[4];
    AdjEnt ent[ADJ_MAX_ENT];   // the slices of one (tile, frequency), in order
    AdjWork work[4][ADJ_MAX_WORK];   // each quad's part, in the same order
};

}  // namespace

namespace {

// Pipeline shapes of the tensor-core kernels.
constexpr int NPROD = 512;                   // adjoint epilogue threads: four quads of 128 (thread = pixel)
constexpr int NTHR_A = NPROD + 64;           // + MMA warp + loader warp
constexpr int NPROD_F = 512;                 // forward producer threads: four groups of one per A row
constexpr int NTHR_F = NPROD_F + 64;
constexpr int NST = 5;                       // pipeline stages
constexpr uint32_t ST_BYTES = 40u * 1024u;   // A hi (4 KB) + A lo (4 KB) + B (<= 32 KB)
constexpr uint32_t ST_ALO = 4096u, ST_B = 8192u;
// V slices of the adjoint (K = 32): A hi (8 KB) + A lo (8 KB) + W (n rows x 32, <= 16 KB)
constexpr uint32_t ST_VALO = 8192u, ST_VB = 16384u;

// The two bf16 halves of a packed word, hi + lo parts added (exact: lo is below hi's ulp).
__device__ __forceinline__ float sum_lo16(uint32_t h, uint32_t l) {
    return __uint_as_float(h << 16) + __uint_as_float(l << 16);
}
__device__ __forceinline__ float sum_hi16(uint32_t h, uint32_t l) {
    return __uint_as_float(h & 0xffff0000u) + __uint_as_float(l & 0xffff0000u);
}

// ---------------------------------------------------------------------------
// Operand image of one frequency set (layout: aimg_put4 in rb_internal.cuh) from the
// caller's tables, for the single-operator entry points (the update writes it from its
// resolve pass: k_resolve_images, rb_trace.cu).  The synthesis record of each entry is
// formed in registers from its table record, c at the pixel and the distance to the
// element.  The adjoint reads the image K-major (a K = 16 slice is two rows: one 4 KB
// bulk copy per plane), the forward MN-major (a 16-pixel slice of every row is one 2-D
// TMA box).  CTA (tile, element block of 16): thread (p, half) synthesises elements
// 16 eb + 8 half + k (k < 8) at pixel p for every frequency and writes rows
// 4 eb + 2 half + {0, 1} of the pixel's core row (coalesced: 128 threads, 2 KB).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_tables_images(GeoDev G, const rb_cell* __restrict__ tables,
                                                       const float* __restrict__ c, FreqSet F,
                                                       __nv_bfloat16* __restrict__ aimg, size_t a_stride) {
    const int n = G.n_elem, rcn = 2 * n / 8;
    const int neb = n / 16;
    const int tile = (int)blockIdx.x / neb, eb = (int)blockIdx.x % neb;
    const int tid = threadIdx.x, p = tid & (TP - 1), half = tid >> 7;
    const int px = tile * TP + p;
    const int e0 = 16 * eb + 8 * half;
    float4 sr[8];
    if (px < G.npix) {
        const float sqrt_c = sqrtf(__ldg(c + px));
        const int ix = px % G.nx, iy = px / G.nx;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            DF ex, ey;
            elem_pos(G, e0 + k, ex, ey);
            sr[k] = synth_record(tables[(size_t)(e0 + k) * G.npix + px], sqrt_c, pixel_elem_dist(G, ix, iy, ex, ey),
                                 G.inv_cref, G.inv_cref_lo, G.j_floor);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) sr[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int fw = 0; fw < F.n; ++fw) {
        const FreqC& fc = F.f[fw];
        __nv_bfloat16* plane = aimg + (size_t)fw * a_stride + (size_t)tile * 2 * rcn * 1024;
#pragma unroll
        for (int kg = 0; kg < 2; ++kg) {
            float2 g[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) g[q] = green_srec(sr[4 * kg + q], fc);
            aimg_put4(plane, rcn, 4 * eb + 2 * half + kg, p, g);
        }
    }
}

// ---------------------------------------------------------------------------
// Adjoint kernel: warp-specialised, NST-stage pipeline of 40 KB stages.
//   warps 0..15 four epilogue quads of four warps (thread = pixel p = tid % 128 = the TMEM
//               lane): quad u % 4 takes diagonal unit u (16 elements, two U slices).  It
//               reads G of the unit from the staged A slices, writes the unit's |G|^2 (hi /
//               lo) to the V slice in global scratch, and, once the MMAs of its second slice
//               are complete, adds conj(G_e) U_e of the unit's 32 TMEM columns to its
//               pixel's g: the columns of a unit get their last contribution from its own
//               slices, so the epilogue follows the MMAs through the tile instead of
//               waiting for its end, and G comes from slices that are in shared memory
//               anyway.  V slices alike (quad dv % 4, 32 columns, |G|^2 from the stage).
//   warp 16     MMA issuer: waits for a stage, issues its MMAs and commits their completion
//               to the stage's "empty" barrier and to the diagonal units' own;
//   warp 17     loader: bulk-copies A and B of the slices of a stage (U: the A image and T;
//               V: the |G|^2 slices and Y) as soon as it is free.
// The slice order of a (tile, frequency) is the schedule of adj_schedule(): the U slices
// with r ascending, as many of the last, short ones to a stage as fit it, and the V slices
// among them, each behind the U groups whose |G|^2 it reads and whose columns it takes.
// Barriers: full_u[d] / full_v[dv] (bulk-copy bytes of an entry on the diagonal, d its
// first group) and acc_u[u] / acc_v[dv] (MMAs complete), each used once per pass with the
// pass's parity, so that a quad waits only for its own slices (a schedule has at least NST
// entries, so no barrier can complete twice before its readers, without whom the stage is
// not free, have seen it); full[s] (the slices below the diagonal, which only the issuer
// waits for); empty[s] (the stage's MMAs, and 48 arrivals of the quads that read it, or of
// the issuer where none does), acc_low (16 warp arrivals: the U columns that V takes over
// are read), acc_empty (16 warp arrivals: every column of the pass is read), vready[dv] (8
// warp arrivals: the |G|^2 slice is written), drain (MMA completion on the error path).
// Every wait is bounded; a timeout raises a shared flag that ends all loops.
//
// What bounds it: shared-memory traffic first.  Per (tile, frequency) of 256 elements the
// MMAs need 15 k cycles, and the stages' writes (0.98 MB), the MMAs' operand reads and the
// quads' reads come to about 3 MB, 24 k cycles at 128 B a cycle (the full sums: 29 k cycles
// of MMAs and 4.6 MB).  The rest was instruction latency of the two issuing warps: one
// barrier wait per stage, polled ahead, and schedules worked out on the host keep it down.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(NTHR_A, 1) k_adjoint_tc(const __grid_constant__ TcArgs A) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t s_full[NST], s_empty[NST], s_full_u[32], s_full_v[8], s_acc_u[16], s_acc_v[8], s_vready[8];
    __shared__ uint64_t s_acc_empty, s_acc_low, s_drain;
    __shared__ uint32_t s_last[NST][2];           // loader: barrier (address) and 1 | parity << 8 of a stage's copies
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_err;
    __shared__ float s_red[2][3][3][TP];          // by item parity: partial sums of quads 1..3: Re g, Im g, H
    const GeoDev& G = A.G;
    const AdjShape sh(G.n_elem);
    const int n = sh.n;
    const uint32_t ne = (uint32_t)sh.ne;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const bool want_h = A.want_h != 0;
    const int n_ent = A.n_ent;
    constexpr uint32_t kReads = 48;               // arrivals of the readers of a stage
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) {
            tc::mbar_init(tc::smem_u32(&s_full[s]), 1);
            tc::mbar_init(tc::smem_u32(&s_empty[s]), 1 + kReads);
        }
        for (int d = 0; d < 32; ++d) tc::mbar_init(tc::smem_u32(&s_full_u[d]), 1);
        for (int d = 0; d < 16; ++d) tc::mbar_init(tc::smem_u32(&s_acc_u[d]), 1);
        for (int d = 0; d < 8; ++d) {
            tc::mbar_init(tc::smem_u32(&s_full_v[d]), 1);
            tc::mbar_init(tc::smem_u32(&s_acc_v[d]), 1);
            tc::mbar_init(tc::smem_u32(&s_vready[d]), 8);
        }
        tc::mbar_init(tc::smem_u32(&s_acc_empty), NPROD / 32);
        tc::mbar_init(tc::smem_u32(&s_acc_low), NPROD / 32);
        tc::mbar_init(tc::smem_u32(&s_drain), 1);
        s_err = 0;
    }
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(&s_tmem), A.tmem_cols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
    const size_t vslice = 2 * TP * 32;            // bf16 of one |G|^2 slice (hi and lo)
    __nv_bfloat16* vbuf = A.vimg + (size_t)blockIdx.x * 2 * (size_t)(n / 32) * vslice;
    const int n_items = A.n_tiles * A.n_freq;
    const uint32_t smem0 = tc::smem_u32(smem);
    const uint32_t full0 = tc::smem_u32(&s_full[0]), full_u0 = tc::smem_u32(&s_full_u[0]), full_v0 = tc::smem_u32(&s_full_v[0]);
    const uint32_t empty0 = tc::smem_u32(&s_empty[0]), acc_u0 = tc::smem_u32(&s_acc_u[0]), acc_v0 = tc::smem_u32(&s_acc_v[0]);
    const uint32_t vready0 = tc::smem_u32(&s_vready[0]);
    // full barrier of an entry, staged in s, and its parity (nd: parities of full[s])
    auto full_bar = [&](AdjEnt e, uint32_t s) {
        return e.diag() ? (e.is_v() ? full_v0 : full_u0) + 8u * e.d() : full0 + 8u * s;
    };

    if (warp == NPROD / 32 + 1) {
        // ------------------------------ loader ------------------------------
        const bool lead = tc::elect_one();
        int it = 0;
        uint32_t ql = 0, s = 0, ph = 0, pass = 0, nd = 0;    // passes begun; bit s: parity of full[s]
        bool ok = true;
        // the operand image streams through L2 once per launch: first out, so that it does
        // not push the CTAs' |G|^2 scratch (rewritten every tile) out to DRAM
        uint64_t stream_pol;
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream_pol));
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x, ++it) {
            const int tile = item / A.n_freq, fw = item - tile * A.n_freq;
            const unsigned char* bu = A.bu + (size_t)fw * A.b_stride;
            const unsigned char* bw = A.bw + (size_t)fw * A.b_stride;
            const unsigned char* ap = (const unsigned char*)(A.aimg + (size_t)fw * A.aimg_stride +
                                                             (size_t)tile * 2 * (n / 4) * 1024);
            const unsigned char* const ap0 = ap;
            const __nv_bfloat16* vimg = vbuf + (size_t)(it & 1) * (n / 32) * vslice;
            for (int k = 0; k < n_ent; ++k, ++ql) {
                const AdjEnt e = A.ent[k];
                if (e.first()) {
                    ++pass;
                    ap = ap0;
                }
                if (ql >= NST && !tc::mbar_wait_warp(empty0 + 8u * s, ph ^ 1u, kMaxTries, &s_err)) {
                    ok = false;
                    break;
                }
                uint32_t dst = smem0 + s * ST_BYTES;
                const uint32_t par = e.diag() ? (pass - 1u) & 1u : (nd >> s) & 1u;
                const uint32_t mb = full_bar(e, s);
                if (!e.diag()) nd ^= 1u << s;
                if (e.is_v() && e.diag() && !tc::mbar_wait_warp(vready0 + 8u * e.d(), par, kMaxTries, &s_err)) {
                    // the |G|^2 slice, written by the quads (a slice below the diagonal in an earlier
                    // pass of the item), did not come: nothing issued into this stage
                    ok = false;
                    break;
                }
                if (!e.is_v()) {
                    // rows of the entry's slices: 2 ne below the diagonal (cnt = 1), then 16 fewer each
                    const uint32_t cnt = e.cnt();
                    uint32_t bb = 64u * (2u * ne - 16u * e.d());
                    if (lead) tc::bulk_arm(mb, cnt * (ST_B + bb) - 512u * cnt * (cnt - 1u));
                    for (uint32_t c = 0; c < cnt; ++c) {
                        if (lead) {
                            // image rows 2j, 2j + 1 of the hi plane, then of the lo plane
                            tc::bulk_copy(dst + ST_B, bu, bb, mb);
                            tc::bulk_copy_hint(dst, ap, 4096u, mb, stream_pol);
                            tc::bulk_copy_hint(dst + ST_ALO, ap + (size_t)(n / 4) * 2048, 4096u, mb, stream_pol);
                        }
                        ap += 4096;
                        bu += bb;
                        dst += ST_B + bb;
                        bb -= 1024u;
                    }
                } else {
                    const uint32_t wbytes = 64u * (ne - 32u * e.d()), abytes = 2u * TP * 32 * 2;
                    if (lead) {
                        tc::bulk_arm(mb, wbytes + abytes);
                        tc::bulk_copy(dst + ST_VB, bw, wbytes, mb);
                        tc::bulk_copy(dst, vimg + (size_t)e.j() * vslice, abytes, mb);
                    }
                    bw += wbytes;
                }
                if (lead) {
                    s_last[s][0] = mb;
                    s_last[s][1] = par;
                }
                if (++s == NST) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok && lead) {
            s_err = 1;
            // bounded waits for the last copies issued into each stage
            for (uint32_t x = 0; x < (ql < NST ? ql : (uint32_t)NST); ++x) tc::mbar_wait(s_last[x][0], s_last[x][1], kMaxTries);
        }
        __syncwarp();
    } else if (warp == NPROD / 32) {
        // ------------------------------ MMA issuer ------------------------------
        const bool lead = tc::elect_one();
        const uint32_t id0 = tc::idesc_bf16_f32(128, 0);
        uint32_t s = 0, pass = 0, nd = 0;
        bool ok = true, begun = false;
        AdjEnt e = A.ent[0];
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
            bool v_begun = false;
            for (int k = 0; k < n_ent; ++k) {
                const AdjEnt nx = A.ent[k + 1 < n_ent ? k + 1 : 0];   // in time for the next round
                if (e.first()) {
                    // a new pass: every column of the previous one must have been read
                    if (pass > 0) ok = tc::mbar_wait_warp(tc::smem_u32(&s_acc_empty), (pass - 1u) & 1u, kMaxTries, &s_err);
                    ++pass;
                    v_begun = false;
                }
                if (e.is_v() && !v_begun) {
                    if (A.low_groups > 0) ok = ok && tc::mbar_wait_warp(tc::smem_u32(&s_acc_low), (pass - 1u) & 1u, kMaxTries, &s_err);
                    v_begun = true;
                }
                if (!ok) break;
                ok = tc::mbar_wait_warp(full_bar(e, s), e.diag() ? (pass - 1u) & 1u : (nd >> s) & 1u, kMaxTries, &s_err);
                if (!ok) break;
                tc::fence_after();
                const uint32_t sa0 = smem0 + s * ST_BYTES;
                if (!e.is_v()) {
                    uint32_t sa = sa0, rows = 2u * ne - 16u * e.d(), col = tmem + 16u * e.d();
                    uint32_t acc = e.j() > 0u ? 1u : 0u;
                    const uint32_t cnt = e.cnt();
                    for (uint32_t c = 0; c < cnt; ++c) {
                        // A K-major in the image's arrangement: K cores 2048 B apart (LBO), 8-pixel
                        // cores 128 B apart (SBO)
                        const uint64_t dah = tc::sdesc(sa, 2048, 128), dal = tc::sdesc(sa + ST_ALO, 2048, 128);
                        const uint64_t dbh = tc::sdesc(sa + ST_B, 128, 256), dbl = tc::sdesc(sa + ST_B + 32u * rows, 128, 256);
                        // one or two N-blocks: what exceeds 256 columns, then the last 256 (a row of B is 32 bytes)
                        const uint32_t n1 = rows > 256u ? rows - 256u : rows, id1 = id0 | ((n1 >> 3) << 17);
                        if (lead) {
                            tc::mma_bf16(col, dah, dbh, id1, acc);
                            tc::mma_bf16(col, dah, dbl, id1, 1u);
                            tc::mma_bf16(col, dal, dbh, id1, 1u);
                            if (rows > 256u) {
                                const uint32_t id2 = id0 | ((256u >> 3) << 17), c2 = col + n1;
                                const uint64_t dbh2 = dbh + 2u * n1, dbl2 = dbl + 2u * n1;
                                tc::mma_bf16(c2, dah, dbh2, id2, acc);
                                tc::mma_bf16(c2, dah, dbl2, id2, 1u);
                                tc::mma_bf16(c2, dal, dbh2, id2, 1u);
                            }
                            if (e.diag() && ((e.d() + c) & 1u)) tc::commit(acc_u0 + 8u * ((e.d() + c) >> 1));
                        }
                        sa += ST_B + 64u * rows;
                        col += 16u;
                        rows -= 16u;
                        acc = 1u;
                    }
                } else {
                    const uint32_t rows = ne - 32u * e.d(), id = id0 | ((rows >> 3) << 17);
                    const uint32_t d = tmem + A.v_col + 32u * e.d();
                    // K = 32 slice in the chunk_offset layout (SBO = 512): two K = 16 steps, 256 bytes apart
                    const uint64_t vah = tc::sdesc(sa0, 128, 512), val = tc::sdesc(sa0 + ST_VALO, 128, 512);
                    const uint64_t vb = tc::sdesc(sa0 + ST_VB, 128, 512);
                    if (lead) {
                        tc::mma_bf16(d, vah, vb, id, e.j() > 0u ? 1u : 0u);
                        tc::mma_bf16(d, val, vb, id, 1u);
                        tc::mma_bf16(d, vah + 16u, vb + 16u, id, 1u);
                        tc::mma_bf16(d, val + 16u, vb + 16u, id, 1u);
                        if (e.diag()) tc::commit(acc_v0 + 8u * e.d());
                    }
                }
                begun = true;
                if (lead) {
                    tc::commit(empty0 + 8u * s);
                    if (!e.diag()) tc::mbar_arrive_cnt(empty0 + 8u * s, kReads);
                }
                if (!e.diag()) nd ^= 1u << s;
                if (++s == NST) s = 0;
                e = nx;
            }
        }
        if (!ok && lead) {
            s_err = 1;
            atomicAdd(A.counters + CNT_TC_TIMEOUT, 1u);
            // bounded wait for the MMAs still in flight
            if (begun) {
                tc::commit(tc::smem_u32(&s_drain));
                tc::mbar_wait(tc::smem_u32(&s_drain), 0u, kMaxTries);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------ epilogue quads ------------------------------
        const uint32_t p = (uint32_t)(tid & (TP - 1));
        const int quad = warp >> 2;
        const uint32_t t0 = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const unsigned char* const a_base = smem + (p >> 3) * 128u + (p & 7u) * 16u;   // this pixel in a K core of an A slice
        const int n_work = A.n_work[quad];
        bool ok = true;
        int it = 0;
        uint32_t s0 = 0, pass = 0;    // stage of the item's first entry
        auto wait = [&](uint32_t bar, uint32_t parity) {
            if (ok) ok = tc::mbar_wait_warp(bar, parity, kMaxTries, &s_err);
            return ok;
        };
        auto arrive = [&](uint32_t bar, uint32_t cnt) {
            __syncwarp();
            if (lane == 0) tc::mbar_arrive_cnt(bar, cnt);
        };
        auto stage_of = [&](uint32_t f) {   // of a work record's a or b
            const uint32_t s = s0 + (f & 15u);
            return s >= (uint32_t)NST ? s - NST : s;
        };
        for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++it) {
            const int tile = item / A.n_freq, fw = item - tile * A.n_freq;
            __nv_bfloat16* vimg = vbuf + (size_t)(it & 1) * (n / 32) * vslice;
            float gr = 0.f, gi = 0.f, hh = 0.f;
            for (int k = 0; k < n_work && ok; ++k) {
                const AdjWork w = A.work[quad][k];
                if (w.first()) ++pass;
                const uint32_t par = (pass - 1u) & 1u, u = w.u();
                const uint32_t sa = stage_of(w.a);
                if (!w.is_v()) {
                    // G of the unit's 16 elements: K core h of a slice holds elements 4 h .. 4 h + 3
                    // as (Re G, -Im G) pairs, in a hi and a lo plane
                    uint4 hv[4], lv[4];
                    if (!wait(full_u0 + 8u * (w.a >> 16), par)) break;
                    const unsigned char* ap = a_base + sa * ST_BYTES + ((w.a >> 4) & 0xffu) * 1024u;
                    hv[0] = *(const uint4*)ap;
                    hv[1] = *(const uint4*)(ap + 2048);
                    lv[0] = *(const uint4*)(ap + ST_ALO);
                    lv[1] = *(const uint4*)(ap + ST_ALO + 2048);
                    uint32_t sb = sa;
                    if (w.b != 0u) {
                        arrive(empty0 + 8u * sa, (w.a >> 12) & 15u);
                        if (!wait(full_u0 + 8u * (w.b >> 16), par)) break;
                        sb = stage_of(w.b);
                        ap = a_base + sb * ST_BYTES + ((w.b >> 4) & 0xffu) * 1024u;
                    } else {
                        ap = a_base + sa * ST_BYTES + w.off2 * 1024u;
                    }
                    hv[2] = *(const uint4*)ap;
                    hv[3] = *(const uint4*)(ap + 2048);
                    lv[2] = *(const uint4*)(ap + ST_ALO);
                    lv[3] = *(const uint4*)(ap + ST_ALO + 2048);
                    arrive(empty0 + 8u * sb, ((w.b != 0u ? w.b : w.a) >> 12) & 15u);
                    float x[16], y[16];   // Re G, -Im G
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t hw[4] = {hv[i].x, hv[i].y, hv[i].z, hv[i].w}, lw[4] = {lv[i].x, lv[i].y, lv[i].z, lv[i].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            x[4 * i + e] = sum_lo16(hw[e], lw[e]);
                            y[4 * i + e] = sum_hi16(hw[e], lw[e]);
                        }
                    }
                    if (want_h) {
                        // elements 16 u .. 16 u + 15 of the pass: cores 2 (u % 2), + 1 of its V slice u / 2
                        __nv_bfloat16* vs = vimg + (size_t)(w.q() * (uint32_t)sh.gv + (u >> 1)) * vslice +
                                            tc::chunk_offset(p, 16u * (u & 1u)) / 2;
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            uint32_t vh[4], vl[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                __nv_bfloat16 a, b, al, bl;
                                const int e0 = 8 * c + 2 * i, e1 = e0 + 1;
                                tc::split_bf16(x[e0] * x[e0] + y[e0] * y[e0], a, al);
                                tc::split_bf16(x[e1] * x[e1] + y[e1] * y[e1], b, bl);
                                vh[i] = bf16_pack2(a, b);
                                vl[i] = bf16_pack2(al, bl);
                            }
                            *(uint4*)(vs + 64 * c) = make_uint4(vh[0], vh[1], vh[2], vh[3]);
                            *(uint4*)(vs + 64 * c + TP * 32) = make_uint4(vl[0], vl[1], vl[2], vl[3]);
                        }
                        asm volatile("fence.proxy.async.global;" ::: "memory");   // read next by the loader's bulk copies
                        arrive(vready0 + 8u * (u >> 1), 1u);
                    }
                    if (!wait(acc_u0 + 8u * u, par)) break;
                    tc::fence_after();
                    float v[32];   // per group of 8 elements: Re U, then Im U
                    tc::tmem_ld32(t0 + 32u * u, v);
                    // the columns V takes over (or the next pass) are free once read
                    if (w.low() || w.last()) tc::fence_before();
                    if (w.low()) arrive(tc::smem_u32(&s_acc_low), 1u);
                    if (w.last()) arrive(tc::smem_u32(&s_acc_empty), 1u);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float ur = v[16 * (i >> 3) + (i & 7)], ui = v[16 * (i >> 3) + 8 + (i & 7)];
                        gr = fmaf(x[i], ur, fmaf(-y[i], ui, gr));
                        gi = fmaf(x[i], ui, fmaf(y[i], ur, gi));
                    }
                } else {
                    if (!wait(full_v0 + 8u * u, par)) break;
                    const unsigned char* ap = smem + sa * ST_BYTES + (p >> 3) * 512u + (p & 7u) * 16u;
                    uint4 h[4], l[4];   // |G|^2 of elements 8 x .. 8 x + 7, hi and lo planes
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        h[x] = *(const uint4*)(ap + 128 * x);
                        l[x] = *(const uint4*)(ap + ST_VALO + 128 * x);
                    }
                    arrive(empty0 + 8u * sa, kReads / 4u);
                    if (!wait(acc_v0 + 8u * u, par)) break;
                    tc::fence_after();
                    float v[32];
                    tc::tmem_ld32(t0 + A.v_col + 32u * u, v);
                    if (w.last()) {
                        tc::fence_before();
                        arrive(tc::smem_u32(&s_acc_empty), 1u);
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const uint32_t hw[4] = {h[x].x, h[x].y, h[x].z, h[x].w}, lw[4] = {l[x].x, l[x].y, l[x].z, l[x].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            hh = fmaf(sum_lo16(hw[i], lw[i]), v[8 * x + 2 * i], hh);
                            hh = fmaf(sum_hi16(hw[i], lw[i]), v[8 * x + 2 * i + 1], hh);
                        }
                    }
                }
            }
            s0 = (s0 + (uint32_t)n_ent) % NST;
            // the quads' sums, in fixed order
            float(*red)[3][TP] = s_red[it & 1];
            if (quad > 0) {
                red[quad - 1][0][p] = gr;
                red[quad - 1][1][p] = gi;
                red[quad - 1][2][p] = hh;
            }
            if (tc::named_or(1, NPROD, !ok)) {
                ok = false;
                break;
            }
            const int px = tile * TP + (int)p;
            if (quad == 0 && px < G.npix) {
                const float fr = (gr + red[0][0][p] + red[1][0][p] + red[2][0][p]) * A.w2[fw];
                const float fi = (gi + red[0][1][p] + red[1][1][p] + red[2][1][p]) * A.w2[fw];
                const float fh = (hh + red[0][2][p] + red[1][2][p] + red[2][2][p]) * A.w4[fw];
                const size_t o = (size_t)fw * G.npix + px;
                if (A.g_out) A.g_out[o] = make_float2(fr, fi);
                if (A.h_out) A.h_out[o] = fh;
                // this frequency's Re g and H for the sums over the set (k_adjoint_sums)
                if (A.fpart) A.fpart[o] = make_float2(fr, fh);
            }
        }
        if (!ok) s_err = 1;
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, A.tmem_cols);
}

// The slices of one (tile, frequency) in order, one entry per pipeline stage, and each
// quad's work records in the same order: per pass the U slices with r ascending (the short
// diagonal ones packed up to four to a 40 KB stage), and each V slice ADJ_V_LAG U stages
// behind the last U group it depends on: the group whose |G|^2 it reads (its bulk copy
// would otherwise wait for a slice just landed) and, where V takes over U columns, the last
// of those.  False if the tables are too small (no supported ring size).
constexpr int ADJ_V_LAG = 3;
bool adj_schedule(const AdjShape& sh, bool want_h, int low_groups, TcArgs* A) {
    int k = 0;
    bool fits = true;
    for (int i = 0; i < 4; ++i) A->n_work[i] = 0;
    for (int q = 0; q < sh.n / sh.ne; ++q) {
        const int nu = (q + 1) * sh.ge, nv = want_h ? (q + 1) * sh.gv : 0, dj = q * sh.ge, dv = q * sh.gv;
        int stage_of[32];              // U stage (in this pass) of each diagonal group
        uint32_t where[32], off[32];   // its record field a / b, and its KB offset in the stage
        bool begun[4] = {false, false, false, false};
        auto put = [&](int j, int cnt, bool v, bool first, int d) {
            if (k < ADJ_MAX_ENT) A->ent[k] = AdjEnt::make(j, cnt, v, first, d);
            else fits = false;
            ++k;
        };
        auto work = [&](int quad, uint32_t x, uint32_t a, uint32_t b, uint32_t off2) {
            int& m = A->n_work[quad];
            if (m < ADJ_MAX_WORK)
                A->work[quad][m] = AdjWork{x | (uint32_t)q << 8 | (begun[quad] ? 0u : 1u << 12), a, b, off2};
            else fits = false;
            ++m;
            begun[quad] = true;
        };
        int st = 0, v = 0;
        auto put_v = [&]() {
            const int d = v - dv;
            if (d >= 0) work(d & 3, (uint32_t)d | 1u << 11, (uint32_t)(k % NST), 0u, 0u);
            put(v++, 1, true, false, d);
        };
        for (int j = 0; j < nu; ++st) {
            int cnt = 1;
            const int d0 = j - dj;
            if (d0 >= 0) {
                uint32_t bytes = ST_B + 64u * (uint32_t)sh.u_rows(q, j);
                // (64 elements: one slice a stage, which keeps the schedule at NST entries or more)
                while (cnt < 4 && j + cnt < nu && sh.ge > 8) {
                    bytes += ST_B + 64u * (uint32_t)sh.u_rows(q, j + cnt);
                    if (bytes > ST_BYTES) break;
                    ++cnt;
                }
                // readers of the entry: the quads of its units
                const uint32_t readers = (uint32_t)((d0 + cnt - 1) / 2 - d0 / 2 + 1);
                uint32_t o = 0;
                for (int c = 0; c < cnt; ++c) {
                    stage_of[d0 + c] = st;
                    off[d0 + c] = o / 1024u;
                    where[d0 + c] = (uint32_t)(k % NST) | (o / 1024u) << 4 | (12u / readers) << 12 | (uint32_t)d0 << 16;
                    o += ST_B + 64u * (uint32_t)sh.u_rows(q, j + c);
                }
            }
            put(j, cnt, false, j == 0, d0);
            j += cnt;
            const int done = j - dj;   // diagonal groups issued so far
            for (int d = d0 < 0 ? 0 : d0; d < done; ++d) {
                if (!(d & 1)) continue;
                const int u = d >> 1;
                const bool same = (where[d] >> 16) == (where[d - 1] >> 16);
                const bool low = 2 * u < low_groups && 2 * u + 8 >= low_groups;
                work(u & 3, (uint32_t)u | (low ? 1u << 14 : 0u), where[d - 1], same ? 0u : where[d], off[d]);
            }
            if (v < nv) {
                int at = low_groups > 0 ? low_groups - 1 : -1;   // the diagonal group it waits for
                if (v >= dv && 4 * (v - dv) + 3 > at) at = 4 * (v - dv) + 3;
                if (at < 0 || (at < done && st >= stage_of[at] + ADJ_V_LAG)) put_v();
            }
        }
        while (v < nv) put_v();
        for (int i = 0; i < 4; ++i)
            if (fits && A->n_work[i] > 0) A->work[i][A->n_work[i] - 1].x |= 1u << 13;   // last of the pass
    }
    A->n_ent = k;
    return fits && k >= NST;
}
}  // namespace

// rings of 64..256 elements in multiples of 64 in one pass over the elements of U and V,
// and of 512, 768 and 1024 elements in passes of 256
bool tc_adjoint_supported(int n_elem) {
    return (n_elem >= 64 && n_elem <= 256 && n_elem % 64 == 0) || (n_elem % 256 == 0 && n_elem >= 512 && n_elem <= 1024);
}


size_t tc_b_images_bytes(int n_elem) {
    const size_t n = (size_t)n_elem;
    return (2 * n) * (2 * n) * 2 * 2 + n * n * 2;   // bu (hi + lo) + bw, bf16
}

cudaError_t launch_prep_b(int n, int n_freq, const float2* R, const uint8_t* W, void* img, cudaStream_t s) {
    const AdjShape sh(n);
    const int npass = n / sh.ne, tri = npass * (npass + 1) / 2;
    const size_t w_off = (size_t)(2 * n) * (2 * n) * 4;
    k_prep_b<<<dim3((sh.ge + sh.gv) * tri, n_freq, 4), 128, 0, s>>>(n, R, W, (unsigned char*)img, tc_b_images_bytes(n), w_off);
    return cudaGetLastError();
}

size_t tc_aimage_elems(int n_elem, int npix) {
    return (size_t)((npix + TP - 1) / TP) * 2 * (size_t)(2 * n_elem / 8) * 1024;
}

cudaError_t launch_tables_images(const GeoDev& G, const rb_cell* tables, const float* c, const FreqSet& F, void* aimg,
                                 cudaStream_t s) {
    if (!tc_adjoint_supported(G.n_elem) || !tables || !c || !aimg) return cudaErrorInvalidValue;
    const int n_tiles = (G.npix + TP - 1) / TP;
    const long long blocks = (long long)n_tiles * (G.n_elem / 16);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    k_tables_images<<<(int)blocks, 256, 0, s>>>(G, tables, c, F, (__nv_bfloat16*)aimg,
                                                tc_aimage_elems(G.n_elem, G.npix));
    return cudaGetLastError();
}

namespace {
// gsum = sum over the set's frequencies of Re g, hsum of H, added in frequency order (the
// order a CTA taking all frequencies of its tile in turn would use).
__global__ void k_adjoint_sums(const float2* __restrict__ fpart, int n_freq, int npix, float* __restrict__ gsum,
                               float* __restrict__ hsum) {
    for (int px = blockIdx.x * blockDim.x + threadIdx.x; px < npix; px += gridDim.x * blockDim.x) {
        float g = 0.f, h = 0.f;
        for (int fw = 0; fw < n_freq; ++fw) {
            const float2 v = fpart[(size_t)fw * npix + px];
            g += v.x;
            h += v.y;
        }
        if (gsum) gsum[px] = g;
        if (hsum) hsum[px] = h;
    }
}
}  // namespace

cudaError_t launch_adjoint_tc(const GeoDev& G, const void* aimg, const FreqSet& F, const void* images, float2* gscr,
                              int n_ctas, float2* g_out, float* h_out, float* gsum, float* hsum, uint32_t* counters,
                              cudaStream_t s) {
    const int n = G.n_elem;
    if (!tc_adjoint_supported(n) || !aimg) return cudaErrorInvalidValue;
    const AdjShape sh(n);
    TcArgs A;
    A.G = G;
    A.n_freq = F.n;
    for (int w = 0; w < F.n; ++w) {
        A.w2[w] = F.f[w].w2;
        A.w4[w] = F.f[w].w4;
    }
    A.aimg = (const __nv_bfloat16*)aimg;
    A.aimg_stride = tc_aimage_elems(n, G.npix);
    A.bu = (const unsigned char*)images;
    A.bw = A.bu + (size_t)(2 * n) * (2 * n) * 4;
    A.b_stride = tc_b_images_bytes(n);
    A.vimg = (__nv_bfloat16*)gscr;
    A.g_out = g_out;
    A.h_out = h_out;
    // the CTAs take (tile, frequency) items in turn, so the sums over the set go through
    // the per-frequency buffer that follows the per-CTA scratch in the workspace
    A.fpart = (gsum || hsum) ? (float2*)(A.vimg + (size_t)RB_TC_MAX_CTAS * 2 * n * 256) : nullptr;
    A.counters = counters;
    A.n_tiles = (G.npix + TP - 1) / TP;
    A.want_h = (h_out || hsum) ? 1 : 0;
    // V beside U where TMEM's 512 columns hold both, else in the first columns of U
    A.v_col = 3 * sh.ne <= 512 ? 2u * (uint32_t)sh.ne : 0u;
    A.low_groups = A.v_col || !A.want_h ? 0 : sh.ne / 16;
    const int need = A.v_col ? 3 * sh.ne : 2 * sh.ne;
    A.tmem_cols = 32;
    while (A.tmem_cols < (uint32_t)need) A.tmem_cols <<= 1;
    if (!adj_schedule(sh, A.want_h != 0, A.low_groups, &A)) return cudaErrorInvalidValue;
    // most of the SM's shared memory, so one CTA (one TMEM owner) per SM
    const int sm = NST * (int)ST_BYTES;
    const int n_items = A.n_tiles * F.n;
    const int grid = n_ctas < n_items ? n_ctas : n_items;
    cudaError_t e = cudaFuncSetAttribute(k_adjoint_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e != cudaSuccess) return e;
    k_adjoint_tc<<<grid, NTHR_A, sm, s>>>(A);
    e = cudaGetLastError();
    if (e != cudaSuccess || !A.fpart) return e;
    k_adjoint_sums<<<(G.npix + 255) / 256, 256, 0, s>>>(A.fpart, F.n, G.npix, gsum, hsum);
    return cudaGetLastError();
}

// ===========================================================================
// Born forward on the tensor cores:  d[e][r] = w^2 sum_x G_e(x) G_r(x) m(x)
// Real form over K = pixels: rows e' = 2e + {0: Re, 1: -Im} of A = conj(G) m and
// columns r' = 2r + {0, 1} of B = conj(G) give D = A B^T (2n x 2n, symmetric) =
// the real form of conj(d), from which
//   Re d = D[2e][2r] - D[2e+1][2r+1],  Im d = -(D[2e][2r+1] + D[2e+1][2r]).
// Both operands come from the adjoint's A image (layout of aimg_put4), read MN-major:
// a core matrix there is 8 pixels (K) x 8 consecutive r' (16 bytes each), and a
// 16-pixel K slice of up to 32 rows of 8 r' is one 2-D TMA box per plane.  CTA (pair, s):
// the pair's 128-row block i of D and column range over pixel split s, accumulated in
// TMEM; columns left of the row block are skipped (symmetry).  Partial D blocks go to
// global memory and a second kernel sums the splits in order.
// ===========================================================================
namespace {

constexpr int FMAXB = 16;  // max row blocks (2n / 128, n <= 1024)
constexpr int FMAXG = 4;   // max column groups of 512 columns (2n / 512)
constexpr int FMAXP = 40;  // max (row block, column group) pairs (40 for n = 1024)
constexpr int FMAXST = 12; // max pipeline stages
constexpr double FWD_MIN_KB = 80.0;   // see make_fwd_args
constexpr int FBOX = 32;   // rows (of 8 r') per TMA box (16 where fewer are left)
constexpr uint32_t ST_FB = 8192u;   // forward stage: A hi (4 KB), A lo (4 KB), then B hi and B lo

struct FwdArgs {
    GeoDev G;
    float w2;
    const float* m;
    float* partial;            // [cta][128][2n] fp32 (only needed columns written)
    int n_mb;                  // row blocks
    // work pairs: row block p_i with the columns [p_c0, p_c1) (at most 512, so the accumulators
    // fit TMEM), each split over pixel ranges
    int n_pairs;
    int p_i[FMAXP], p_c0[FMAXP], p_c1[FMAXP];
    int splits[FMAXP];         // splits per pair
    int cta0[FMAXP + 1];       // first CTA of each pair
    int pidx[FMAXB][FMAXG];    // pair of (row block, column group)
    uint32_t tmem_cols;
    uint32_t* counters;
};

// Stages of a pair of `cols` columns: as many as 200 KB hold, at most FMAXST.
__host__ __device__ __forceinline__ int fwd_stages(int cols) {
    const int k = (200 * 1024) / ((int)ST_FB + 64 * cols);
    return k < FMAXST ? k : FMAXST;
}

// Forward kernel: warp-specialised pipeline over K = 16 pixel slices.
//   warps 0..15 producers, four groups of 128 threads, each on every fourth slice (a slice's
//               way through a group is mostly latency): thread u of a group takes the 16-byte
//               rows (8 r', one pixel) u and u + 128 of the row block's A slice: rows 128 i ..
//               128 i + 127 scaled by m(x) and re-split into hi / lo, once the slice has
//               landed; then the epilogue;
//   warp 16     MMA issuer; warp 17 loader (TMA boxes of the columns' rows of the slice, hi
//               and lo planes), both warp-uniform.
// SEP: some pairs load their row block's own rows separately (rings above 256 elements);
// without it every pair finds them among its B rows and the test compiles away.
template <bool SEP>
__global__ void __launch_bounds__(NTHR_F, 1) k_forward_tc(const __grid_constant__ FwdArgs A, const __grid_constant__ CUtensorMap tmap,
                                                         const __grid_constant__ CUtensorMap tmap16) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t s_full_a[FMAXST], s_full_b[FMAXST], s_empty[FMAXST], s_acc_full;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_err;
    const GeoDev& G = A.G;
    const int n = G.n_elem, n2 = 2 * n;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    int pq = 0;
    while (pq + 1 < A.n_pairs && (int)blockIdx.x >= A.cta0[pq + 1]) ++pq;
    const int i = A.p_i[pq], col0 = A.p_c0[pq], cols = A.p_c1[pq] - col0;   // needed columns (= B rows loaded)
    const int sp = (int)blockIdx.x - A.cta0[pq];
    const int S = A.splits[pq];
    const int rcn = n2 / 8, rc0 = col0 / 8;             // rows of 8 r' per plane; first one loaded
    const int nrow = cols / 8;                          // rows loaded per plane (a multiple of 16)
    const uint32_t plane_bytes = (uint32_t)nrow * 256u;
    // the row block's own 16 rows (the A operand before scaling by m): inside the loaded B
    // rows, or loaded separately into the A area of the stage
    const bool own_in = !SEP || 16 * i >= rc0;
    const uint32_t tx_bytes = 2u * plane_bytes + (own_in ? 0u : 2u * 16u * 256u);
    const uint32_t st_bytes = ST_FB + 2u * plane_bytes;
    const int nst = fwd_stages(cols);
    const int n_tiles = (G.npix + TP - 1) / TP;
    const int nsl_all = n_tiles * 8;
    const int cps = (nsl_all + S - 1) / S;
    const int sbeg = min(nsl_all, sp * cps), send = min(nsl_all, sbeg + cps);
    const int nq = send - sbeg;
    if (tid == 0) {
        for (int k = 0; k < nst; ++k) {
            tc::mbar_init(tc::smem_u32(&s_full_a[k]), 4);
            tc::mbar_init(tc::smem_u32(&s_full_b[k]), 1);
            tc::mbar_init(tc::smem_u32(&s_empty[k]), 1);
        }
        tc::mbar_init(tc::smem_u32(&s_acc_full), 1);
        s_err = 0;
    }
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(&s_tmem), A.tmem_cols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
    const uint32_t smem0 = tc::smem_u32(smem), full_a0 = tc::smem_u32(&s_full_a[0]), full_b0 = tc::smem_u32(&s_full_b[0]);
    const uint32_t empty0 = tc::smem_u32(&s_empty[0]);

    if (warp == NPROD_F / 32 + 1) {
        // ------------------------------ loader ------------------------------
        const bool lead = tc::elect_one();
        const uint64_t tm = reinterpret_cast<uint64_t>(&tmap);
        const uint64_t tm16 = reinterpret_cast<uint64_t>(&tmap16);   // 16-row boxes
        int ql = 0, k = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (; ql < nq; ++ql) {
            if (ql >= nst && !tc::mbar_wait_warp(empty0 + 8u * k, ph ^ 1u, kMaxTries, &s_err)) {
                ok = false;
                break;
            }
            const int sg = sbeg + ql, x = (sg & 7) * 128, y0 = (sg >> 3) * 2 * rcn;
            const uint32_t mb = full_b0 + 8u * k, st = smem0 + (uint32_t)k * st_bytes;
            if (lead) {
                tc::bulk_arm(mb, tx_bytes);
                for (int hl = 0; hl < 2; ++hl) {
                    const int y = y0 + hl * rcn;
                    const uint32_t dst = st + ST_FB + (uint32_t)hl * plane_bytes;
                    for (int b = 0; b < nrow; b += FBOX)
                        tc::tma_2d(dst + (uint32_t)b * 256u, nrow - b >= FBOX ? tm : tm16, x, y + rc0 + b, mb);
                    if (!own_in) tc::tma_2d(st + (uint32_t)hl * ST_ALO, tm16, x, y + 16 * i, mb);
                }
            }
            if (++k == nst) { k = 0; ph ^= 1u; }
        }
        if (!ok && lead) {
            s_err = 1;
            for (int x = (ql > nst ? ql - nst : 0); x < ql; ++x)
                tc::mbar_wait(full_b0 + 8u * (x % nst), (uint32_t)(x / nst) & 1u, kMaxTries);
        }
        __syncwarp();
    } else if (warp == NPROD_F / 32) {
        // ------------------------------ MMA issuer ------------------------------
        // both operands MN-major (transpose bits 15 and 16): LBO = stride between the
        // two 8-pixel K cores (128 B), SBO = stride between 8-r' cores (256 B)
        const bool lead = tc::elect_one();
        const uint32_t id0 = tc::idesc_bf16_f32(128, 0) | (1u << 15) | (1u << 16);
        // one or two N-blocks: what exceeds 256 columns, then the last 256
        const uint32_t n1 = cols > 256 ? (uint32_t)cols - 256u : (uint32_t)cols;
        const uint32_t id1 = id0 | ((n1 >> 3) << 17), id2 = id0 | ((256u >> 3) << 17);
        int k = 0, last = -1;
        uint32_t ph = 0, last_ph = 0;
        bool ok = true;
        for (int q = 0; q < nq; ++q) {
            ok = tc::mbar_wait_warp(full_b0 + 8u * k, ph, kMaxTries, &s_err) &&
                 tc::mbar_wait_warp(full_a0 + 8u * k, ph, kMaxTries, &s_err);
            if (!ok) break;
            tc::fence_after();
            const uint32_t sa = smem0 + (uint32_t)k * st_bytes, sb = sa + ST_FB;
            const uint64_t dah = tc::sdesc(sa, 128, 256), dal = tc::sdesc(sa + ST_ALO, 128, 256);
            const uint64_t dbh = tc::sdesc(sb, 128, 256), dbl = tc::sdesc(sb + plane_bytes, 128, 256);
            const uint32_t acc = q > 0 ? 1u : 0u;
            if (lead) {
                tc::mma_bf16(tmem, dah, dbh, id1, acc);
                tc::mma_bf16(tmem, dah, dbl, id1, 1u);
                tc::mma_bf16(tmem, dal, dbh, id1, 1u);
                if (cols > 256) {
                    const uint64_t dbh2 = dbh + 2u * n1, dbl2 = dbl + 2u * n1;   // 32 bytes a column
                    tc::mma_bf16(tmem + n1, dah, dbh2, id2, acc);
                    tc::mma_bf16(tmem + n1, dah, dbl2, id2, 1u);
                    tc::mma_bf16(tmem + n1, dal, dbh2, id2, 1u);
                }
                tc::commit(empty0 + 8u * k);
                if (q == nq - 1) tc::commit(tc::smem_u32(&s_acc_full));
            }
            last = k;
            last_ph = ph;
            if (++k == nst) { k = 0; ph ^= 1u; }
        }
        if (!ok && lead) {
            s_err = 1;
            atomicAdd(A.counters + CNT_TC_TIMEOUT, 1u);
            if (last >= 0) tc::mbar_wait(empty0 + 8u * last, last_ph, kMaxTries);   // the MMAs still in flight
        }
        __syncwarp();
    } else {
        // -------------------------------- producers --------------------------------
        // thread u of its group of 128: K core pc = (u / 8) % 2, pixel row x8 = u % 8 of that core,
        // rows rl = u / 16 and rl + 8 of 8 r' (of the row block's 16)
        constexpr int NG = 4;
        const int grp = warp >> 2, u = tid & 127;
        const int rl = u >> 4, pc = (u >> 3) & 1, x8 = u & 7;
        const uint32_t aoff = (uint32_t)(rl * 256 + pc * 128 + x8 * 16);
        // source of this thread's 16 bytes: the B rows, or the A area itself (scaled in place)
        const uint32_t soff = own_in ? ST_FB + (uint32_t)((16 * i - rc0 + rl) * 256 + pc * 128 + x8 * 16) : aoff;
        const uint32_t slo = own_in ? plane_bytes : ST_ALO;
        bool ok = true;
        auto load_m = [&](int q) -> float {
            if (q >= nq) return 0.f;
            const int px = (sbeg + q) * 16 + pc * 8 + x8;
            return px < G.npix ? __ldg(A.m + px) : 0.f;
        };
        float mnext = load_m(grp);
        int k = grp % nst;   // nst >= NG + 1
        uint32_t ph = 0;
        for (int q = grp; q < nq; q += NG) {
            const float mm = mnext;
            mnext = load_m(q + NG);
            // The stage's previous slice, another group's, has been used: without this wait the
            // test of the full barrier below could see the phase before it.  (This test cannot:
            // this group's last slice q - NG had landed, so its loader had seen slices up to
            // q - NG - nst, among them the stage's last but one, q - 2 nst, used.)
            if (q >= nst) ok = ok && tc::mbar_wait_warp(empty0 + 8u * k, ph ^ 1u, kMaxTries, &s_err);
            ok = ok && tc::mbar_wait_warp(full_b0 + 8u * k, ph, kMaxTries, &s_err);
            if (!ok) break;
            unsigned char* st = smem + (size_t)k * st_bytes;
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const unsigned char* src = st + soff + 2048u * x;
                const uint4 vh = *(const uint4*)src, vl = *(const uint4*)(src + slo);
                const uint32_t hw[4] = {vh.x, vh.y, vh.z, vh.w}, lw[4] = {vl.x, vl.y, vl.z, vl.w};
                uint32_t oh[4], ol[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    __nv_bfloat16 h0, l0, h1, l1;
                    tc::split_bf16(sum_lo16(hw[t], lw[t]) * mm, h0, l0);
                    tc::split_bf16(sum_hi16(hw[t], lw[t]) * mm, h1, l1);
                    oh[t] = bf16_pack2(h0, h1);
                    ol[t] = bf16_pack2(l0, l1);
                }
                *(uint4*)(st + aoff + 2048u * x) = make_uint4(oh[0], oh[1], oh[2], oh[3]);
                *(uint4*)(st + ST_ALO + aoff + 2048u * x) = make_uint4(ol[0], ol[1], ol[2], ol[3]);
            }
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(full_a0 + 8u * k);
            k += NG;
            if (k >= nst) { k -= nst; ph ^= 1u; }
        }
        // epilogue: this CTA's partial D block (128 rows x needed columns) to global memory
        if (nq > 0) ok = ok && tc::mbar_wait_warp(tc::smem_u32(&s_acc_full), 0u, kMaxTries, &s_err);
        tc::fence_after();
        if (ok) {
            const int row = tid & 127, g = warp >> 2;
            const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
            float* out = A.partial + ((size_t)blockIdx.x * 128 + row) * n2 + col0;
            for (int cb = 32 * g; cb < cols; cb += 128) {
                float v[32];
                if (nq > 0) {
                    tc::tmem_ld32(tmem + lane_off + (uint32_t)cb, v);
                } else {
#pragma unroll
                    for (int t = 0; t < 32; ++t) v[t] = 0.f;
                }
#pragma unroll
                for (int t = 0; t < 32; t += 4) *(float4*)(out + cb + t) = make_float4(v[t], v[t + 1], v[t + 2], v[t + 3]);
            }
        } else {
            s_err = 1;
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, A.tmem_cols);
}

// d = w^2 (sum over splits of the partial D blocks), and per-block partial sums of
// W |d|^2.  D and d are symmetric, and for e <= r the 2 x 2 block of D at (2e, 2r) lies in
// a computed block (right of its row block's first column), so entry (e, r), e <= r, is
// read row-wise and written to d[e][r] and d[r][e].  YS warps take 32 consecutive r of one e:
// each every YS-th split, the first adds the warps' sums in order.  YS = 1 where the
// entries alone fill the chip (128 to 512 elements at 511 x 389 pixels: 8 to 12 us; eight warps
// an entry, with their barriers, 43 for 256), 8 below 128 elements (64: 5 us; by single warps
// of 152 splits each, with one load under way, 27).  Loads go out eight splits ahead: left to the
// compiler, the loop of calls that write d waited for every split (256 elements, 48 splits: 45 us
// against 8).
template <int YS>
__global__ void __launch_bounds__(256) k_forward_tc_reduce(FwdArgs A, float2* __restrict__ d_out, const uint8_t* __restrict__ w,
                                                           double* __restrict__ den_part) {
    __shared__ float4 s_sum[8][32];
    __shared__ double s_den[8];
    const int n = A.G.n_elem, n2 = 2 * n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, y = wid % YS;
    double acc = 0.0;
    const int nrb = n / 32;   // n is a multiple of 64
    constexpr int TPB = 8 / YS;   // runs of 32 entries a CTA takes at a time
    for (int run0 = blockIdx.x * TPB; run0 < n * nrb; run0 += gridDim.x * TPB) {
        const int run = run0 + wid / YS;   // n nrb is a multiple of 8
        const int e = run / nrb, r = 32 * (run - e * nrb) + lane;
        const bool live = e <= r;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);   // D[2e][2r..2r+1], D[2e+1][2r..2r+1]
        if (live) {
            const int i = (2 * e) >> 7, row = (2 * e) & 127, pq = A.pidx[i][(2 * r) >> 9], ns = A.splits[pq];
            const float* blk = A.partial + ((size_t)A.cta0[pq] * 128 + row) * n2 + 2 * r;
            const size_t step = (size_t)128 * n2;
            // eight splits ahead: a split's loads go out as the one eight before it is added
            float2 n0[8], n1[8];
            auto load = [&](int k, int sp) {
                n0[k] = n1[k] = make_float2(0.f, 0.f);
                if (sp < ns) {
                    n0[k] = __ldcg((const float2*)(blk + sp * step));
                    n1[k] = __ldcg((const float2*)(blk + sp * step + n2));
                }
            };
#pragma unroll
            for (int k = 0; k < 8; ++k) load(k, y + k * YS);
            for (int sp = y; sp < ns; sp += 8 * YS) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    s.x += n0[k].x;
                    s.y += n0[k].y;
                    s.z += n1[k].x;
                    s.w += n1[k].y;
                    load(k, sp + (8 + k) * YS);
                }
            }
        }
        if (YS > 1) {
            __syncthreads();
            s_sum[wid][lane] = s;
            __syncthreads();
            if (y == 0)
                for (int k = 1; k < YS; ++k) {
                    const float4 o = s_sum[wid + k][lane];
                    s.x += o.x;
                    s.y += o.y;
                    s.z += o.z;
                    s.w += o.w;
                }
        }
        if (y == 0 && live) {
            // the image rows 2r + 1 hold -Im G_r (the conjugate, as the adjoint uses it), so the
            // product of the two images is conj(d): Re d as is, Im d negated
            const float dre = (s.x - s.w) * A.w2;
            const float dim = -(s.y + s.z) * A.w2;
            const size_t er = (size_t)e * n + r, re = (size_t)r * n + e;
            if (d_out) {
                d_out[er] = make_float2(dre, dim);
                if (e != r) d_out[re] = make_float2(dre, dim);
            }
            if (w) {
                const int cnt = (w[er] ? 1 : 0) + ((e != r && w[re]) ? 1 : 0);
                if (cnt) acc += cnt * ((double)dre * dre + (double)dim * dim);
            }
        }
    }
    if (den_part) {
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) s_den[wid] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < 8; ++k) acc += s_den[k];
            den_part[blockIdx.x] = acc;
        }
    }
}

cudaError_t forward_tc_reduce(const FwdArgs& A, float2* d_out, const uint8_t* w, double* den_part, cudaStream_t s) {
    if (A.G.n_elem < 128) k_forward_tc_reduce<8><<<256, 256, 0, s>>>(A, d_out, w, den_part);
    else k_forward_tc_reduce<1><<<256, 256, 0, s>>>(A, d_out, w, den_part);
    return cudaGetLastError();
}

FwdArgs make_fwd_args(const GeoDev& G, const FreqC& F, const float* m, float* partial, int n_ctas,
                      uint32_t* counters) {
    FwdArgs A;
    A.G = G;
    A.w2 = F.w2;
    A.m = m;
    A.partial = partial;
    A.counters = counters;
    const int n2 = 2 * G.n_elem;
    A.n_mb = n2 / 128;
    // pairs (row block i, columns from its diagonal on), in groups of 512 columns
    A.n_pairs = 0;
    int widest = 0;
    double cost[FMAXP], total = 0.0;
    for (int i = 0; i < A.n_mb; ++i) {
        for (int g = 0; g < FMAXG; ++g) A.pidx[i][g] = -1;
        for (int g = (128 * i) / 512; 512 * g < n2; ++g) {
            const int q = A.n_pairs++;
            A.p_i[q] = i;
            A.p_c0[q] = 128 * i > 512 * g ? 128 * i : 512 * g;
            A.p_c1[q] = 512 * (g + 1) < n2 ? 512 * (g + 1) : n2;
            A.pidx[i][g] = q;
            const int cols = A.p_c1[q] - A.p_c0[q];
            if (cols > widest) widest = cols;
            // A slice's cost in KB of shared-memory traffic, which sets the pace of the wide pairs:
            // the operands' arrival, the producers' 16 KB, and per N-block three MMAs reading A
            // (4 KB) and their columns of B; never below what a slice takes by latency alone.
            // Forward stage of four frequencies, 256 elements at 512 x 512 pixels, by that floor:
            // 60 KB 834 us, 80 KB 819, 100 KB 876, all pairs alike 940
            const double kb = cols / 16.0 + 16.0 + 12.0 * (cols > 256 ? 2 : 1) + 0.09375 * cols;
            cost[q] = kb > FWD_MIN_KB ? kb : FWD_MIN_KB;
            total += cost[q];
        }
    }
    A.tmem_cols = 32;
    while (A.tmem_cols < (uint32_t)widest) A.tmem_cols <<= 1;
    // splits in proportion to that cost, every pair at least one, no split below 8 slices
    const int nsl = ((G.npix + TP - 1) / TP) * 8;
    const int most = nsl / 8 > 0 ? nsl / 8 : 1;
    int left = n_ctas;
    for (int q = 0; q < A.n_pairs; ++q) {
        A.splits[q] = (int)(n_ctas * cost[q] / total);
        if (A.splits[q] < 1) A.splits[q] = 1;
        left -= A.splits[q];
    }
    while (left-- > 0) {   // what rounding left over goes to the slowest pair
        int slow = 0;
        for (int q = 1; q < A.n_pairs; ++q)
            if (cost[q] / A.splits[q] > cost[slow] / A.splits[slow]) slow = q;
        ++A.splits[slow];
    }
    int c0 = 0;
    for (int q = 0; q < A.n_pairs; ++q) {
        if (A.splits[q] > most) A.splits[q] = most;
        A.cta0[q] = c0;
        c0 += A.splits[q];
    }
    A.cta0[A.n_pairs] = c0;
    return A;
}

}  // namespace

size_t tc_forward_partial_bytes(int n_elem, int n_ctas) {
    return (size_t)(n_ctas + FMAXP) * 128 * (2 * (size_t)n_elem) * sizeof(float);
}

namespace {

// The forward kernel of one frequency on s; its arguments (which the reduce takes too) in *out.
cudaError_t forward_tc_kernel(const GeoDev& G, const void* aimg, const FreqC& F, const float* m, float* partial,
                              int n_ctas, uint32_t* counters, cudaStream_t s, FwdArgs* out) {
    if (!tc_adjoint_supported(G.n_elem) || !aimg) return cudaErrorInvalidValue;
    const FwdArgs A = make_fwd_args(G, F, m, partial, n_ctas, counters);
    // the A image of this frequency as a 2-D tensor: rows of 8 r' x 128 pixels (1024 bf16),
    // (tile, plane, row) major; boxes of 128 elements (one 16-pixel slice) x 32 or 16 rows
    const int rcn = 2 * G.n_elem / 8;
    const int n_tiles = (G.npix + TP - 1) / TP;
    CUtensorMap tmap, tmap16;
    if (!tc::encode_tmap_2d(&tmap, aimg, 1024, (uint64_t)n_tiles * 2 * rcn, 2048, 128, (uint32_t)FBOX) ||
        !tc::encode_tmap_2d(&tmap16, aimg, 1024, (uint64_t)n_tiles * 2 * rcn, 2048, 128, 16u))
        return cudaErrorUnknown;
    const int sm = NST * (int)ST_BYTES;
    const bool sep = G.n_elem > 256;   // a column group left of which a row block lies
    cudaError_t e;
    if (sep) {
        e = cudaFuncSetAttribute(k_forward_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        if (e != cudaSuccess) return e;
        k_forward_tc<true><<<A.cta0[A.n_pairs], NTHR_F, sm, s>>>(A, tmap, tmap16);
    } else {
        e = cudaFuncSetAttribute(k_forward_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        if (e != cudaSuccess) return e;
        k_forward_tc<false><<<A.cta0[A.n_pairs], NTHR_F, sm, s>>>(A, tmap, tmap16);
    }
    *out = A;
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_forward_tc(const GeoDev& G, const void* aimg, const FreqC& F, const float* m, float* partial,
                              int n_ctas, float2* d_out, const uint8_t* w, double* den_part, uint32_t* counters,
                              cudaStream_t s) {
    FwdArgs A;
    cudaError_t e = forward_tc_kernel(G, aimg, F, m, partial, n_ctas, counters, s, &A);
    if (e != cudaSuccess) return e;
    return forward_tc_reduce(A, d_out, w, den_part, s);
}

cudaError_t launch_forward_tc_overlap(const GeoDev& G, const void* aimg, const FreqC& F, const float* m,
                                      float* partial, int n_ctas, float2* d_out, const uint8_t* w, double* den_part,
                                      uint32_t* counters, cudaStream_t s, cudaStream_t r, cudaEvent_t fwd_done,
                                      cudaEvent_t red_done) {
    FwdArgs A;
    cudaError_t e = forward_tc_kernel(G, aimg, F, m, partial, n_ctas, counters, s, &A);
    if (e == cudaSuccess) e = cudaEventRecord(fwd_done, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(r, fwd_done, 0);
    if (e != cudaSuccess) return e;
    e = forward_tc_reduce(A, d_out, w, den_part, r);
    return e == cudaSuccess ? cudaEventRecord(red_done, r) : e;
}
