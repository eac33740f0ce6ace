// k_xdft.cu -- the x stages of the band transforms on the tensor cores
// (tcgen05, FP16 hi/lo splits), mixed-precision path, N = 72, 96, 120, for
// spheres whose density fits the grid (nmax <= (N - 1) / 4 < 32):
//
//   apply:   F(i) = sum_x e^{-2 pi i i x / N} s V(x) psi(x),  |i| <= nmax,
//            psi(x) = sum_i a(i) e^{+2 pi i i x / N}, in place on the planes;
//   density: sum over the bands of |psi(x)|^2.
//
// The register transforms of k_fft_impl.cuh are bound by instruction issue:
// 6500 warp instructions per 32 lines of an apply at N = 120, where the
// sphere's 41 of 120 planes make the memory floor low (0.26 of the copy
// bandwidth).  As a matrix product the transform costs the CUDA cores only
// the split into FP16 parts and the pointwise work.  Times before and now
// (us): apply mgo-120 (430 bands, nmax 20) 2325 and 1142, organic-96 (42 bands,
// nmax 20) 105 and 82; density mgo-120 1187 and 690, organic-96 90 and 56.  At
// mgo-120 a tile of 128 lines takes an SM 7.7 us / 2 (two blocks): about 1.2
// us of issued MMAs, the rest the split, the pointwise work and the waits
// between the dependent phases that two blocks do not cover; the planes' 4 GB
// read and written would take 0.62 ms.
//
// Even and odd parts.  With e(i) = a(i) + a(-i), o(i) = a(i) - a(-i) and
// likewise p, m of f = s V psi over +-x, every product is real, of 32 terms:
//   E = sum_i e(i) cos, O = sum_i o(i) sin   (real and imaginary parts each),
//   psi(+-x) = (E_re -+ O_im, E_im +- O_re),    0 <= x <= N / 2,
//   C = sum_x p(x) cos, S = sum_x m(x) sin,
//   F(+-i) = (C_re +- S_im, C_im -+ S_re),      0 <= i <= nmax,
// a quarter of the multiplications of the full matrix.  One table, cos and
// sin of 2 pi i x / N (x <= N / 2, i <= nmax; zero elsewhere), serves both ways:
// K-major for the inverse, MN-major for the forward product.
//
// Precision.  A row of the MMA is one x line (y, z); its elements are scaled
// by a power of two of its own (from its largest element; forward: from a
// bound, that element times 4 (nmax + 1) times the class's largest |V|) and
// split as hi + lo, as the table is; a product is lo.hi + hi.lo + hi.hi, and
// the last additions are those with the lowest frequencies, which are the
// largest.
//
// A tile is 128 consecutive lines of a band, a thread's line its
// tensor-memory lane; the warpgroups of a block share out the chunks of 8
// input frequencies and of 16 x.  Waits are bounded: one that runs out sets
// the contractions' flag (the call then reports ROKS_ETIMEOUT) and waits on
// with the default bound, so that nothing is read before it is there.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "roks_impl.cuh"
#include "tc_sm103.cuh"

namespace roks {

// tiled map of 64-bit words (k_stream.cu)
bool tensor_map_words(CUtensorMap* map, const void* ptr, int rank, const uint64_t* dims, const uint64_t* strides,
                      const uint32_t* box);

namespace {

constexpr int XD_I = 32, XD_X = 64;                  // table: frequencies, x
constexpr uint32_t XD_PART = XD_I * XD_X * 2;        // bytes of one part of cos or sin
constexpr uint32_t XD_TAB = 4 * XD_PART;             // cos hi, cos lo, sin hi, sin lo: 16 KB
// Input tile of a block: hi of e_re, e_im, o_re, o_im, then lo, each the
// chunks of 8 frequencies that hold any (2 KB each).  The last K-step may
// take in the first chunk of the next part: the table is zero there.
__host__ __device__ constexpr uint32_t xd_comp(int nmax) { return 2048u * (uint32_t)(nmax / 8 + 1); }
__host__ __device__ constexpr uint32_t xd_abytes(int nmax) { return 8u * xd_comp(nmax) + 2048u; }
constexpr int XD_TSH = 10;                           // the table is scaled by 2^10
constexpr uint32_t XD_WAIT = 1u << 26;
// shared memory of a block, with the next tile's planes staged or without
__host__ __device__ constexpr size_t xd_smem(int nmax, bool staged) {
    return xd_abytes(nmax) + XD_TAB + (staged ? 1024 * (2 * nmax + 1) : 0) + 1024;
}
// what lets two blocks share an SM's 228 KB: 1 KB of each is the system's, a
// little more their static arrays
constexpr size_t XD_SMEM_HALF = 111 * 1024;
constexpr size_t XD_SMEM_MAX = xd_smem(29, true);    // the largest sphere, 120^3
// What the truncating additions of an inverse product take from |psi|^2, as a
// part of it, in the mean over orbitals of many plane waves: half a unit in the
// last place of the sums, 2^-24.  It goes into the low word of the density
// (without it every density of such orbitals is 6e-8 low, which energies show:
// a DIIS step of mgo-120 2.6e-7 off 64 bits, 1.6e-7 with, 2.2e-7 with register
// transforms; an orbital of so few plane waves that nothing is truncated comes
// out half an FP32 unit high).  The apply's products are left as they are: F's
// error is 1.39e-7, the register transforms' 1.50e-7 (430 bands of mgo-120).
constexpr float XD_LOSS = 6e-8f;

__device__ __forceinline__ float xpow2(int e) { return __int_as_float((e + 127) << 23); }
__device__ __forceinline__ int xclamp(int e) { return max(-100, min(100, e)); }
// exponent of the power of two that brings a positive finite value below 2^t
__device__ __forceinline__ int below(float v, int t) { return v > 0.f && v <= 3e38f ? xclamp(t - 1 - ilogbf(v)) : 0; }

__device__ __forceinline__ uint32_t h2u(__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); }
// hi and lo of a pair of values
__device__ __forceinline__ void split2(float2 v, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __float22half2_rn(v);
    const float2 f = __half22float2(h);
    hi = h2u(h);
    lo = h2u(__float22half2_rn(csub(v, f)));
}

__device__ __forceinline__ void xwait(uint64_t* bar, uint32_t phase, uint32_t wcap, int* timeout) {
    if (!tc::mbar_wait(bar, phase & 1u, wcap)) {
        if (timeout) *timeout = 1;
        tc::mbar_wait(bar, phase & 1u, XD_WAIT);
    }
}

// Inverse products of a tile, issued by one lane: D (part c at c * dstep
// columns: E_re, E_im, -O_im, O_re) for NX x from 8 xg on; KS K-steps of 16
// frequencies.
template <int KS, int NX>
__device__ __forceinline__ void mma_inverse(uint32_t d, uint32_t dstep, uint32_t sa, uint32_t comp, uint32_t sb,
                                            int xg) {
    constexpr uint32_t idesc = tc::idesc_f16(128, NX);
    const uint64_t da0 = tc::make_desc(0, 2048, 128) + (sa >> 4), db0 = tc::make_desc(0, 1024, 128) + (sb >> 4) + 8 * xg;
    const uint32_t cs = comp >> 4;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int in = c < 2 ? c : 5 - c;                   // e_re, e_im, o_im, o_re (stored o_re, o_im)
        const uint64_t ah = da0 + in * cs, al = da0 + (4 + in) * cs;
        const uint64_t bh = db0 + (c < 2 ? 0 : 2 * XD_PART / 16), bl = bh + XD_PART / 16;
        const uint32_t id = c == 2 ? (idesc | tc::IDESC_NEG_A) : idesc;
        const uint32_t dd = d + c * dstep;
#pragma unroll
        for (int k = KS - 1; k >= 0; --k) {
            tc::mma_f16(dd, al + 256 * k, bh + 128 * k, id, k < KS - 1 ? 1 : 0);
            tc::mma_f16(dd, ah + 256 * k, bl + 128 * k, id, 1);
        }
#pragma unroll
        for (int k = KS - 1; k >= 0; --k) tc::mma_f16(dd, ah + 256 * k, bh + 128 * k, id, 1);
    }
}

// Forward products of half a tile's x: C_re, C_im, S_re, S_im at dd (32
// columns each) from the p and m in tensor memory at ta (32 columns a part:
// 16 per warpgroup, hi then lo), x from 32 hf on.
__device__ __forceinline__ void mma_forward(uint32_t dd, uint32_t ta, uint32_t sb, int hf) {
    constexpr uint32_t idesc = tc::idesc_f16(128, XD_I) | tc::IDESC_B_MN;
    const uint64_t db0 = tc::make_desc(0, 128, 1024) + (sb >> 4) + 32 * hf;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint64_t bh = db0 + (c < 2 ? 0 : 2 * XD_PART / 16), bl = bh + XD_PART / 16;
#pragma unroll
        for (int k = 1; k >= 0; --k) {
            tc::mma_f16_ta(dd + 32 * c, ta + 32 * c + 16 * k + 8, bh + 16 * k, idesc, k == 1 ? hf : 1);
            tc::mma_f16_ta(dd + 32 * c, ta + 32 * c + 16 * k, bl + 16 * k, idesc, 1);
        }
#pragma unroll
        for (int k = 1; k >= 0; --k) tc::mma_f16_ta(dd + 32 * c, ta + 32 * c + 16 * k, bh + 16 * k, idesc, 1);
    }
}

// Table to shared memory, input tiles zeroed (chunks past nmax stay zero),
// tensor memory and barriers set up, by all threads.
__device__ __forceinline__ void xd_setup(unsigned char* A, uint32_t abytes, unsigned char* B, const uint4* tab,
                                         uint32_t* tmem, uint32_t cols, uint64_t* bar, int nbar) {
    for (uint32_t t = threadIdx.x; t < XD_TAB / 16; t += blockDim.x) reinterpret_cast<uint4*>(B)[t] = tab[t];
    for (uint32_t t = threadIdx.x; t < abytes / 16; t += blockDim.x)
        reinterpret_cast<uint4*>(A)[t] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) {
        for (int i = 0; i < nbar; ++i) tc::mbar_init(bar + i, 1);
        tc::fence_mbar_init();
    }
    if (threadIdx.x < 32) tc::tmem_alloc(tmem, cols);
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}

// Eight frequencies 8 c .. 8 c + 7 of a line: a(i) and a(-i) (0 past nmax),
// planes `stride` elements apart.
__device__ __forceinline__ void load_chunk(const float2* Y, int stride, bool valid, int c, int nmax, float2 (&ap)[8],
                                           float2 (&am)[8]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int i = 8 * c + k;
        ap[k] = am[k] = make_float2(0.f, 0.f);
        if (valid && i <= nmax) {
            ap[k] = Y[(nmax + i) * stride];
            if (i > 0) am[k] = Y[(nmax - i) * stride];
        }
    }
}
__device__ __forceinline__ float chunk_max(const float2 (&ap)[8], const float2 (&am)[8]) {
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        m = fmaxf(fmaxf(m, fmaxf(fabsf(ap[k].x), fabsf(ap[k].y))), fmaxf(fabsf(am[k].x), fabsf(am[k].y)));
    return m;
}

// The chunk's e and o, scaled, as hi and lo core-matrix rows of line r.
__device__ __forceinline__ void store_chunk(unsigned char* A, uint32_t comp, int c, int r, float s, const float2 (&ap)[8],
                                            const float2 (&am)[8]) {
    uint32_t hi[4][4], lo[4][4];   // e_re, e_im, o_re, o_im
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 e0 = cscale(cadd(ap[2 * k], am[2 * k]), s), e1 = cscale(cadd(ap[2 * k + 1], am[2 * k + 1]), s);
        const float2 o0 = cscale(csub(ap[2 * k], am[2 * k]), s), o1 = cscale(csub(ap[2 * k + 1], am[2 * k + 1]), s);
        split2(make_float2(e0.x, e1.x), hi[0][k], lo[0][k]);
        split2(make_float2(e0.y, e1.y), hi[1][k], lo[1][k]);
        split2(make_float2(o0.x, o1.x), hi[2][k], lo[2][k]);
        split2(make_float2(o0.y, o1.y), hi[3][k], lo[3][k]);
    }
    unsigned char* dst = A + c * 2048 + (r >> 3) * 128 + (r & 7) * 16;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        *reinterpret_cast<uint4*>(dst + q * comp) = make_uint4(hi[q][0], hi[q][1], hi[q][2], hi[q][3]);
        *reinterpret_cast<uint4*>(dst + (4 + q) * comp) = make_uint4(lo[q][0], lo[q][1], lo[q][2], lo[q][3]);
    }
}

// The planes of a tile (all of a band's, 128 lines from l0 on) on their way
// to shared memory, issued by one lane: one tensor copy, zeros past the last
// line.  It completes bar's phase.  (41 bulk copies of 1 KB held the issuing
// warp for 2,000 cycles.)
__device__ __forceinline__ void stage_planes(float2* raw, const CUtensorMap* tm, int np, int l0, int band,
                                             uint64_t* bar) {
    tc::mbar_arrive_expect_tx(bar, 1024u * np);
    tc::tma_2d(raw, tm, l0, band * np, bar);
}

// ------------------------------------------------------------------ apply
// Two blocks of 256 threads per SM, 256 tensor-memory columns each: the x go
// in two halves of 32, D of a half (four parts of 32 columns) turning in
// place into the forward product's A (each thread overwrites the columns it
// has read), and the forward sums take the other 128 columns.  ST: the next
// tile's planes stream into shared memory meanwhile (where two blocks still
// fit an SM, nmax <= 21); otherwise they are loaded when their tile begins
// (staged in one block per SM 387 us at 160 bands on 96^3, nmax 22; loaded 293;
// the register transforms 372).  (One block
// of 512 threads with all x at once and the next tile's input split beside the
// forward products left every phase's latency in the open: 1.67 ms at mgo-120,
// against the two blocks' 1.22.)
template <int N, int KS, bool ST>
__global__ void __launch_bounds__(256, 2) k_xdft_apply(int nmax, const __grid_constant__ CUtensorMap tm,
                                                       float2* __restrict__ Yp, const float* __restrict__ Vk,
                                                       const float* __restrict__ vmax, const uint4* __restrict__ tab,
                                                       int b0, int nbb, int n_closed, float scale,
                                                       int* __restrict__ timeout, uint32_t wcap) {
    constexpr int NN = N * N, TILES = (NN + 127) / 128;
    extern __shared__ __align__(1024) unsigned char xd_dyn[];
    __shared__ float rowmax[2][128], vm[3];
    __shared__ __align__(8) uint64_t bar[3];   // D, forward sums, staged planes
    __shared__ uint32_t tmem_s;
    unsigned char* A = xd_dyn + ((1024u - (tc::smem_u32(xd_dyn) & 1023u)) & 1023u);
    const uint32_t comp = xd_comp(nmax);
    unsigned char* B = A + xd_abytes(nmax);
    float2* raw = reinterpret_cast<float2*>(B + XD_TAB);
    const int tid = threadIdx.x, warp = tc::warp_index(), h = tid >> 7, r = tid & 127, np = 2 * nmax + 1;
    if (tid < 3) vm[tid] = vmax[tid];
    xd_setup(A, xd_abytes(nmax), B, tab, &tmem_s, 256, bar, 3);
    const uint32_t tmem = tmem_s, lanes = (uint32_t)(r & 96) << 16;
    const uint32_t sa = tc::smem_u32(A), sb = tc::smem_u32(B);
    const int total = TILES * nbb;
    auto stage = [&](int t) {
        if (tc::elect_one()) stage_planes(raw, &tm, np, (t % TILES) * 128, t / TILES, &bar[2]);
        __syncwarp();
    };
    if (ST && warp == 7 && (int)blockIdx.x < total) stage(blockIdx.x);
    uint32_t ph = 0;   // tiles done: two phases of D's and the sums' barriers per tile
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++ph) {
        const int band = t / TILES, l = (t - band * TILES) * 128 + r;
        const bool valid = l < NN;
        const int b = b0 + band, cls = b < n_closed ? 0 : b - n_closed + 1;
        float2* Y = Yp + (int64_t)band * np * NN + l;
        const float* V = Vk + (int64_t)cls * N * NN + (valid ? l : 0);
        float sfw;   // 2^-e of the line's forward scale
        float c0;    // psi (scaled, times the table's 2^10) -> s psi, times the forward scale
        if (ST) xwait(&bar[2], ph, wcap, timeout);
        {
            const float2* src = ST ? raw + r : Y;
            const int stride = ST ? 128 : NN;
            float2 ap0[8], am0[8], ap1[8], am1[8];
            load_chunk(src, stride, ST || valid, h, nmax, ap0, am0);
            load_chunk(src, stride, ST || valid, h + 2, nmax, ap1, am1);
            float mx = fmaxf(chunk_max(ap0, am0), chunk_max(ap1, am1));
            rowmax[h][r] = mx;
            __syncthreads();
            if (ST && warp == 7 && t + (int)gridDim.x < total) stage(t + gridDim.x);
            mx = fmaxf(mx, rowmax[h ^ 1][r]);
            const int e = below(mx, 14);
            const float s = xpow2(e);
            if (8 * h <= nmax) store_chunk(A, comp, h, r, s, ap0, am0);
            if (8 * (h + 2) <= nmax) store_chunk(A, comp, h + 2, r, s, ap1, am1);
            const float bound = mx * (4.f * (nmax + 1)) * vm[cls] * scale;
            const int e2 = below(bound, 14);
            c0 = scale * xpow2(-e - XD_TSH) * xpow2(e2);
            sfw = xpow2(-e2 - XD_TSH);
        }
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
            if (warp == 0) {
                // (the forward products of the first half read what D overwrites)
                if (hf == 1) xwait(&bar[1], 2 * ph, wcap, timeout);
                tc::fence_after_sync();
                if (tc::elect_one()) {
                    mma_inverse<KS, 32>(tmem, 32, sa, comp, sb, 4 * hf);
                    tc::commit(&bar[0]);
                }
                __syncwarp();
            }
            const int x0 = 32 * hf + 16 * h;
            // the potential's loads run beside the products
            float wp[16], wm[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int x = x0 + k;
                wp[k] = wm[k] = 0.f;
                if (x <= N / 2) {
                    wp[k] = V[x * NN];
                    // (x = 0 and N / 2 are their own partners: p = f there)
                    if (x > 0 && x < N / 2) wm[k] = V[(N - x) * NN];
                }
            }
            xwait(&bar[0], 2 * ph + hf, wcap, timeout);
            __syncwarp();
            tc::fence_after_sync();
            const uint32_t dcol = tmem + lanes + 16 * h;
            // x in two batches of 8: this thread's 16 columns of every part
            // become hi of 8 pairs, then lo, once both have been read
            uint32_t hi[4][8], lo[4][8];   // p_re, p_im, m_re, m_im
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float d[4][8];
#pragma unroll
                for (int c = 0; c < 4; ++c) tc::tmem_ld8_nowait(dcol + 32 * c + 8 * q, d[c]);
                tc::tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int kk = 4 * q + k;
                    const float2 er = make_float2(d[0][2 * k], d[0][2 * k + 1]);
                    const float2 ei = make_float2(d[1][2 * k], d[1][2 * k + 1]);
                    const float2 oi = make_float2(d[2][2 * k], d[2][2 * k + 1]);
                    const float2 orr = make_float2(d[3][2 * k], d[3][2 * k + 1]);
                    const float2 w = cscale(make_float2(wp[2 * kk], wp[2 * kk + 1]), c0);
                    const float2 v = cscale(make_float2(wm[2 * kk], wm[2 * kk + 1]), c0);
                    const float2 frp = __fmul2_rn(cadd(er, oi), w), frm = __fmul2_rn(csub(er, oi), v);
                    const float2 fip = __fmul2_rn(cadd(ei, orr), w), fim = __fmul2_rn(csub(ei, orr), v);
                    split2(cadd(frp, frm), hi[0][kk], lo[0][kk]);
                    split2(cadd(fip, fim), hi[1][kk], lo[1][kk]);
                    split2(csub(frp, frm), hi[2][kk], lo[2][kk]);
                    split2(csub(fip, fim), hi[3][kk], lo[3][kk]);
                }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t o[16];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    o[k] = hi[c][k];
                    o[8 + k] = lo[c][k];
                }
                tc::tmem_st16(dcol + 32 * c, o);
            }
            tc::tmem_wait_st();
            tc::fence_before_sync();
            __syncthreads();
            if (warp == 0) {
                tc::fence_after_sync();
                if (tc::elect_one()) {
                    mma_forward(tmem + 128, tmem, sb, hf);
                    tc::commit(&bar[1]);
                }
                __syncwarp();
            }
        }
        // the forward sums of both halves (the first phase is over: D's second
        // half, seen above, was issued after it)
        xwait(&bar[1], 2 * ph + 1, wcap, timeout);
        __syncwarp();
        tc::fence_after_sync();
        const uint32_t fcol = tmem + lanes + 128 + 16 * h;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (16 * h + 8 * q > nmax) break;
            float cr[8], ci[8], sr[8], si[8];
            tc::tmem_ld8_nowait(fcol + 8 * q, cr);
            tc::tmem_ld8_nowait(fcol + 32 + 8 * q, ci);
            tc::tmem_ld8_nowait(fcol + 64 + 8 * q, sr);
            tc::tmem_ld8_nowait(fcol + 96 + 8 * q, si);
            tc::tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i = 16 * h + 8 * q + k;
                if (valid && i <= nmax) {
                    Y[(nmax + i) * NN] = make_float2(sfw * (cr[k] + si[k]), sfw * (ci[k] - sr[k]));
                    if (i > 0) Y[(nmax - i) * NN] = make_float2(sfw * (cr[k] - si[k]), sfw * (ci[k] + sr[k]));
                }
            }
        }
        tc::fence_before_sync();   // (the sums are overwritten after the next tile's barriers)
    }
    tc::fence_before_sync();
    __syncthreads();
    if (tid < 32) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 256);
    }
}

// ------------------------------------------------------------------ density
// Two blocks of 256 threads per SM, 256 tensor-memory columns each (D: four
// parts of 64 x), over the bands of a group for one tile of lines; ST: the
// next band's planes stream into shared memory meanwhile.  A thread keeps
// |psi|^2 of its 32 x and their partners in registers, FP32 sums of up to 16
// bands, added into the compensated grid density like the register
// transforms' (same slots, same order of bands).
template <int N, int KS, bool ST>
__global__ void __launch_bounds__(256, 2) k_xdft_density(int nmax, const __grid_constant__ CUtensorMap tm,
                                                         const float2* __restrict__ Yp,
                                                         DensAcc<float>::S* __restrict__ rho3,
                                                         DensAcc<float>::S* __restrict__ slot,
                                                         const uint4* __restrict__ tab, int b0, int nbb, int gs,
                                                         int n_closed, float2 scale, int cls_override,
                                                         int* __restrict__ timeout, uint32_t wcap) {
    using DA = DensAcc<float>;
    constexpr int NN = N * N;
    extern __shared__ __align__(1024) unsigned char xd_dyn[];
    __shared__ float rowmax[2][128];
    __shared__ __align__(8) uint64_t bar[2];   // D, staged planes
    __shared__ uint32_t tmem_s;
    unsigned char* A = xd_dyn + ((1024u - (tc::smem_u32(xd_dyn) & 1023u)) & 1023u);
    const uint32_t comp = xd_comp(nmax);
    unsigned char* B = A + xd_abytes(nmax);
    const int np = 2 * nmax + 1;
    float2* raw = reinterpret_cast<float2*>(B + XD_TAB);
    const int tid = threadIdx.x, warp = tc::warp_index(), h = tid >> 7, r = tid & 127;
    xd_setup(A, xd_abytes(nmax), B, tab, &tmem_s, 256, bar, 2);
    const uint32_t tmem = tmem_s, lanes = (uint32_t)(r & 96) << 16;
    const uint32_t sa = tc::smem_u32(A), sb = tc::smem_u32(B);
    const int l0 = blockIdx.x * 128, l = l0 + r, g = blockIdx.y;
    const bool valid = l < NN;
    const int gbeg = g * gs, gend = min(nbb, gbeg + gs);
    const int64_t N3 = (int64_t)N * NN, bstride = (int64_t)np * NN;
    DA::S* slot_g = slot ? slot + g * N3 : nullptr;
    float2 sp[16], sm[16];   // sums for x (pairs 2 k, 2 k + 1) and for N - x; x = 32 h + ...
#pragma unroll
    for (int k = 0; k < 16; ++k) sp[k] = sm[k] = make_float2(0.f, 0.f);
    bool slot_written = false;
    int cnt = 0;
    auto cls_of = [&](int bb) {
        const int b = b0 + bb;
        return cls_override >= 0 ? cls_override : (b < n_closed ? 0 : b - n_closed + 1);
    };
    // (an open class holds one band, and rho3 is zero there on entry; eight
    // values are loaded before the first is stored: one at a time they took
    // 36,000 cycles a flush)
    auto flush = [&](int cls) {
        const bool add = cls == 0 && slot_written;
        DA::S* dst = (cls == 0 ? slot_g : rho3 + cls * N3) + l;
        if (valid) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                DA::S old[8];
                auto at = [&](int k) {   // value k of the eight: x and N - x of four x
                    const int x = 32 * h + 4 * q + (k >> 1);
                    return (k & 1) ? ((x > 0 && x < N / 2) ? N - x : -1) : (x <= N / 2 ? x : -1);
                };
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    old[k] = DA::make(0.f);
                    const int e = at(k);
                    if (add && e >= 0) old[k] = dst[e * NN];
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int kk = 4 * q + (k >> 1);
                    const float2 v2 = (k & 1) ? sm[kk >> 1] : sp[kk >> 1];
                    const float u = (kk & 1) ? v2.y : v2.x, v = u * scale.x;
                    const DA::S inc = make_float2(v, fmaf(u, scale.y, fmaf(u, scale.x, -v)) + XD_LOSS * v);
                    const int e = at(k);
                    if (e >= 0) dst[e * NN] = add ? DA::add2(old[k], inc) : inc;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) sp[k] = sm[k] = make_float2(0.f, 0.f);
        cnt = 0;
        if (cls == 0) slot_written = true;
    };
    auto stage = [&](int bb) {
        if (tc::elect_one()) stage_planes(raw, &tm, np, l0, bb, &bar[1]);
        __syncwarp();
    };
    if (ST && warp == 7 && gbeg < gend) stage(gbeg);
    for (int bb = gbeg; bb < gend; ++bb) {
        if (ST) xwait(&bar[1], (uint32_t)(bb - gbeg), wcap, timeout);
        const float2* src = ST ? raw + r : Yp + bb * bstride + l;
        const int stride = ST ? 128 : NN;
        float us;   // psi's scale
        {
            // (two passes over the staged planes, or over what the first one
            // brought to L1, keep the registers for the sums)
            float2 ap[8], am[8];
            load_chunk(src, stride, ST || valid, h, nmax, ap, am);
            float mx = chunk_max(ap, am);
            {
                float2 bp[8], bm[8];
                load_chunk(src, stride, ST || valid, h + 2, nmax, bp, bm);
                mx = fmaxf(mx, chunk_max(bp, bm));
            }
            rowmax[h][r] = mx;
            __syncthreads();
            const int e = below(fmaxf(mx, rowmax[h ^ 1][r]), 14);
            const float s = xpow2(e);
            us = xpow2(-e - XD_TSH);
            if (8 * h <= nmax) store_chunk(A, comp, h, r, s, ap, am);
            if (8 * (h + 2) <= nmax) {
                load_chunk(src, stride, ST || valid, h + 2, nmax, ap, am);
                store_chunk(A, comp, h + 2, r, s, ap, am);
            }
        }
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            tc::fence_after_sync();
            if (tc::elect_one()) {
                mma_inverse<KS, XD_X>(tmem, 64, sa, comp, sb, 0);
                tc::commit(&bar[0]);
            }
            __syncwarp();
        }
        if (ST && warp == 7 && bb + 1 < gend) stage(bb + 1);
        xwait(&bar[0], (uint32_t)(bb - gbeg), wcap, timeout);
        __syncwarp();
        tc::fence_after_sync();
        const uint32_t dcol = tmem + lanes + 32 * h;
        const float2 u2 = make_float2(us, us), n2 = make_float2(-us, -us);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float d[4][8];
#pragma unroll
            for (int c = 0; c < 4; ++c) tc::tmem_ld8_nowait(dcol + 64 * c + 8 * q, d[c]);
            tc::tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 er = __fmul2_rn(make_float2(d[0][2 * k], d[0][2 * k + 1]), u2);
                const float2 ei = __fmul2_rn(make_float2(d[1][2 * k], d[1][2 * k + 1]), u2);
                const float2 oi = make_float2(d[2][2 * k], d[2][2 * k + 1]);
                const float2 orr = make_float2(d[3][2 * k], d[3][2 * k + 1]);
                const float2 prp = __ffma2_rn(oi, u2, er), prm = __ffma2_rn(oi, n2, er);
                const float2 pip = __ffma2_rn(orr, u2, ei), pim = __ffma2_rn(orr, n2, ei);
                sp[4 * q + k] = __ffma2_rn(pip, pip, __ffma2_rn(prp, prp, sp[4 * q + k]));
                sm[4 * q + k] = __ffma2_rn(pim, pim, __ffma2_rn(prm, prm, sm[4 * q + k]));
            }
        }
        tc::fence_before_sync();   // (D is overwritten after the next band's barriers)
        const int cls = cls_of(bb);
        if (++cnt == 16 || bb + 1 == gend || cls != 0 || cls_of(bb + 1) != cls) flush(cls);
    }
    if (!slot_written && slot_g && valid) {
        // a group without closed bands still owns its slot
        for (int k = 0; k < 32; ++k) {
            const int x = 32 * h + k;
            if (x > N / 2) continue;
            slot_g[x * NN + l] = DA::make(0.f);
            if (x > 0 && x < N / 2) slot_g[(N - x) * NN + l] = DA::make(0.f);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (tid < 32) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 256);
    }
}

int xd_sms() {
    int dev = 0, n = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

}  // namespace

// The grids whose kernels are instantiated, as far as their densities fit
// them: 32 frequencies and 64 x is what the tables hold, and all of these
// spheres are within it (nmax <= 29); larger spheres keep the register
// transforms, as do the exchange's fields and the packed open pair.  48^3, which
// the tables hold too, is faster in registers: half of its 64 x are empty (40
// bands, nmax 11: density 18.8 us, 29.1 here, apply 20.4 both; 160 bands 45 and
// 82, 61 and 59).
bool xdft_takes(int N, int nmax) {
    return tcg_enabled() && (N == 72 || N == 96 || N == 120) && nmax <= sphere_prune_nmax(N);
}

// Whether so many bands at once take them.  A block sets up its table and
// tensor memory first, which pays from some 1.7 million grid points on (apply and
// density in us, registers and tensor cores: 72^3, nmax 17, one band 9.0, 12.1 and
// 11.2, 15.1, six 14.2, 14.1 and 15.3, 17.3; 96^3, nmax 14, one 10.1, 10.2 and
// 13.2, 15.4, two 12.0, 11.0 and 17.3, 16.4; 120^3, nmax 20, one 13.3, 12.2 and
// 18.5, 17.4).  The density of the one sphere of 96^3 whose planes are neither
// staged nor stay in L1 (nmax 23) takes them up to 32 bands (12 bands 29.8 us,
// registers 33.8; 42 bands 76.8 and 74.7; 160 bands 242 and 230).
bool xdft_apply_takes(const Sphere& s, int nbb) { return (int64_t)s.N * s.N * s.N * nbb >= 1700000; }
bool xdft_density_takes(const Sphere& s, int nbb) {
    return xdft_apply_takes(s, nbb) && (s.N != 96 || s.nmax < 23 || nbb <= 32);
}

size_t xdft_table_bytes() { return XD_TAB; }

// Image of cos and sin of 2 pi i x / N, times 2^10, as FP16 hi and lo: element
// (x, i) of a part at (i / 8) 512 + (x / 8) 64 + (x % 8) 8 + i % 8; zero past
// x = N / 2 and i = nmax.
void xdft_table(int N, int nmax, void* host) {
    __half* t = static_cast<__half*>(host);
    for (int mat = 0; mat < 2; ++mat)
        for (int x = 0; x < XD_X; ++x)
            for (int i = 0; i < XD_I; ++i) {
                const double a = 2.0 * M_PI * ((i * x) % N) / N;
                double v = x <= N / 2 && i <= nmax ? std::ldexp(mat ? std::sin(a) : std::cos(a), XD_TSH) : 0.0;
                if (mat && 2 * x == N) v = 0.0;
                const int at = (i / 8) * 512 + (x / 8) * 64 + (x % 8) * 8 + i % 8;
                const __half hi = __double2half(v);
                t[(2 * mat) * XD_I * XD_X + at] = hi;
                t[(2 * mat + 1) * XD_I * XD_X + at] = __double2half(v - (double)__half2float(hi));
            }
}

#define XD_DISPATCH(N_, CALL)                             \
    switch (N_) {                                         \
        case 72: { constexpr int NN_ = 72; CALL; } break;   \
        case 96: { constexpr int NN_ = 96; CALL; } break;   \
        case 120: { constexpr int NN_ = 120; CALL; } break; \
        default: break;                                   \
    }

// The planes of nbb bands as rows of N^2 complex numbers, boxes of a band's
// rows x 128 lines.
static bool plane_map(CUtensorMap* tm, const Sphere& s, const float2* Yp, int nbb) {
    const uint64_t nn = (uint64_t)s.N * s.N, dims[2] = {nn, (uint64_t)s.np * nbb}, strides[1] = {8 * nn};
    const uint32_t box[2] = {128, (uint32_t)s.np};
    return tensor_map_words(tm, Yp, 2, dims, strides, box);
}

#define XD_PICK(KERNEL)                                                                    \
    (s.nmax < 16 ? (staged ? go(KERNEL<NN_, 1, true>) : go(KERNEL<NN_, 1, false>)) \
                 : (staged ? go(KERNEL<NN_, 2, true>) : go(KERNEL<NN_, 2, false>)))

// Whether the density's planes are staged where only one block then fits an SM
// (nmax >= 22).  It reads them twice, and on 120^3 those of two blocks don't stay
// in L1 meanwhile: 160 bands, nmax 22 and 29, 353 and 384 us staged, 404 and 452
// loaded (register transforms 451 and 474); on 96^3 nmax 22 they do, 230 and 224
// (230), and loading has no fewer blocks in flight for few bands.
static bool density_staged(const Sphere& s) { return xd_smem(s.nmax, true) <= XD_SMEM_HALF || s.N >= 120; }

// Bands b0 .. b0 + nbb - 1, in place on their planes Yp; vmax: the largest
// |V| of each class.
void xdft_apply(const Sphere& s, const void* tab, float2* Yp, const float* Vk, const float* vmax, int b0, int nbb,
                int n_closed, float scale, cudaStream_t st) {
    if (nbb <= 0) return;
    const int64_t total = (int64_t)((s.N * s.N + 127) / 128) * nbb;
    const int grid = (int)std::min<int64_t>(total, 2 * (int64_t)xd_sms());
    CUtensorMap tm{};
    const bool staged = xd_smem(s.nmax, true) <= XD_SMEM_HALF && plane_map(&tm, s, Yp, nbb);
    const size_t sm = xd_smem(s.nmax, staged);
    auto go = [&](auto kernel) {
        allow_smem(kernel, XD_SMEM_MAX);
        roks::count_launch(), kernel<<<grid, 256, sm, st>>>(s.nmax, tm, Yp, Vk, vmax, static_cast<const uint4*>(tab),
                                                            b0, nbb, n_closed, scale, tcg_timeout_flag(),
                                                            wait_polls());
    };
    XD_DISPATCH(s.N, XD_PICK(k_xdft_apply));
}

void xdft_density(const Sphere& s, const void* tab, const float2* Yp, double* rho3, double* slot, int gs, int ng,
                  int b0, int nbb, int n_closed, double scale, int cls_override, cudaStream_t st) {
    using DS = DensAcc<float>::S;
    // (in two words: rounded to one, it moves every density the same way, by up
    // to 6e-8; 4.3e-8 at mgo-120)
    const float2 sc = make_float2((float)scale, (float)(scale - (double)(float)scale));
    const dim3 grid((s.N * s.N + 127) / 128, ng);
    CUtensorMap tm{};
    const bool staged = density_staged(s) && plane_map(&tm, s, Yp, nbb);
    const size_t sm = xd_smem(s.nmax, staged);
    auto go = [&](auto kernel) {
        allow_smem(kernel, XD_SMEM_MAX);
        roks::count_launch(), kernel<<<grid, 256, sm, st>>>(
                                  s.nmax, tm, Yp, reinterpret_cast<DS*>(rho3), reinterpret_cast<DS*>(slot),
                                  static_cast<const uint4*>(tab), b0, nbb, gs, n_closed, sc, cls_override,
                                  tcg_timeout_flag(), wait_polls());
    };
    XD_DISPATCH(s.N, XD_PICK(k_xdft_density));
}

}  // namespace roks
