// k_mlp.cu -- the learned correction of the TPA preconditioner: a per
// (plane wave, band) network with three inputs, two tanh layers of 64 and one
// output s; the TPA step is scaled by m = exp(clip(s, -3, 3)).
//
// Training runs on the GPU in these kernels: a forward/backward pass over
// blocks of samples writes per-block gradient partials (samples summed in a
// fixed order), a second kernel sums the partials in a fixed order with
// two-sum compensation, and an Adam kernel updates the FP32 master weights.
// Inference (the fused preconditioner inside the PCG step) takes the weights
// rounded to BF16 and runs the 64 x 64 layer on the tensor cores (FP64 contexts:
// in FP32).
//
// Parameter layout (4481 floats): W1 (64 x 3, row major), b1 (64), W2
// (64 x 64, row major), b2 (64), w3 (64), b3 (1).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "roks_grid.cuh"
#include "roks_mlp.cuh"
#include "tc_sm103.cuh"

namespace roks {

namespace {

constexpr int H = kMlpHidden;
constexpr int OW1 = 0, OB1 = 3 * H, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + H;
static_assert(OB3 + 1 == kMlpParams, "layout");

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Loads the parameters into shared memory (optionally rounded to BF16).
__device__ __forceinline__ void load_params(const float* __restrict__ p, float* w, bool bf16) {
    for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) w[i] = bf16 ? bf16_round(p[i]) : p[i];
}

// tanh of two values, relative error below 3e-7 (2.5 units in the last place), in
// the form of Moshier's Cephes library, with coefficients of its own: x + x^3
// P(x^2) up to 0.625, P the least-squares polynomial of degree 4
// brought to equal ripples by Lawson's iteration (4.4e-9), and
// 1 - 2 / (1 + e^{2|x|}) beyond, the two reciprocals from one (|x| is cut
// off at 10, where tanh rounds to 1).  Half the instructions of two tanhf
// calls; the 128 of them per row are most of an evaluation.
__device__ __forceinline__ float2 tanh2(float2 x) {
    const float2 u = __fmul2_rn(x, x);
    float2 p = make_float2(-0.0057049786477133034f, -0.0057049786477133034f);
    p = __ffma2_rn(p, u, make_float2(0.020639079011511765f, 0.020639079011511765f));
    p = __ffma2_rn(p, u, make_float2(-0.053739712249969075f, -0.053739712249969075f));
    p = __ffma2_rn(p, u, make_float2(0.13331442158829518f, 0.13331442158829518f));
    p = __ffma2_rn(p, u, make_float2(-0.33333281940240483f, -0.33333281940240483f));
    const float2 sm = __ffma2_rn(__fmul2_rn(x, u), p, x);
    const float ax = fminf(fabsf(x.x), 10.f), ay = fminf(fabsf(x.y), 10.f);
    const float dx = 1.f + __expf(2.f * ax), dy = 1.f + __expf(2.f * ay);
    const float r = __fdividef(2.f, dx * dy);
    const float bx = copysignf(fmaf(-r, dy, 1.f), x.x), by = copysignf(fmaf(-r, dx, 1.f), x.y);
    // (a NaN fails the comparison and comes out of the polynomial)
    return make_float2(fabsf(x.x) > 0.625f ? bx : sm.x, fabsf(x.y) > 0.625f ? by : sm.y);
}
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// ------------------------------------------------------------------ inference on the tensor cores
// A block of 128 threads evaluates 128 feature rows at a time, thread = row =
// tensor-memory lane.  h1 goes as FP16 hi + lo (22 bits) straight into tensor
// memory, where it is the A operand of z2 = h1 W2^T; W2, scaled by a power of
// two, sits in shared memory as K-major core matrices (hi, and lo too where
// the weights are not rounded to BF16, whose 8 bits hi holds).  The 64 x 64
// layer was 4096 multiply-adds and 1024 shared-memory loads per row; what is
// left is the 128 tanh (their special-function instructions alone, three per
// pair, are 60 us for 1.44 M rows).  128 tensor-memory columns: four blocks
// per SM.  34,265 plane waves x 42 bands: 464 -> 247 us with the column sums.
constexpr int NT = 128;                       // rows (and threads) of a block
constexpr uint32_t NET_COLS = 128;            // A hi 0..31, A lo 32..63, D 64..127
constexpr uint32_t NET_WAIT = 1u << 26;       // polls before a wait is given up for good
constexpr size_t NET_PAD = 27 * 1024;         // dynamic shared memory that keeps a fifth block off the SM

struct NetShared {
    __half w2hi[H * H], w2lo[H * H];          // core (k / 8, j / 8) at (j / 8) 512 + (k / 8) 64 elements
    float4 w1[H];                             // pair j: w1[2j] = (W1[.][0], W1[.][1]), w1[2j+1] = (W1[.][2], b1)
    float4 bw[H / 2];                         // pair k: (b2, b2, w3, w3)
    float b3, unscale;
    float red[NT / 32];
    uint32_t tmem;
    uint64_t bar;
};

// Sets up the block's weights and tensor memory (all threads).
__device__ __forceinline__ void net_setup(NetShared& S, const float* __restrict__ p, bool bf16) {
    auto ld = [&](int i) { return bf16 ? bf16_round(p[i]) : p[i]; };
    const int tid = threadIdx.x;
    float m = 0.f;
    for (int i = tid; i < H * H; i += NT) m = fmaxf(m, fabsf(ld(OW2 + i)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) S.red[tid >> 5] = m;
    if (tid == 0) tc::mbar_init(&S.bar, 1);
    if (tid < 32) tc::tmem_alloc(&S.tmem, NET_COLS);
    __syncthreads();
    m = fmaxf(fmaxf(S.red[0], S.red[1]), fmaxf(S.red[2], S.red[3]));
    const int e = m > 0.f && m <= 3e38f ? min(100, 14 - ilogbf(m)) : 0;
    const float sc = __int_as_float((e + 127) << 23);
    for (int i = tid; i < H * H; i += NT) {
        const int k = i / H, j = i % H;
        const float v = sc * ld(OW2 + i);
        const __half h = __float2half_rn(v);
        const int at = (j >> 3) * 512 + (k >> 3) * 64 + (k & 7) * 8 + (j & 7);
        S.w2hi[at] = h;
        S.w2lo[at] = __float2half_rn(v - __half2float(h));
    }
    if (tid < H / 2) {
        const int j = 2 * tid;
        S.w1[j] = make_float4(ld(OW1 + 3 * j), ld(OW1 + 3 * j + 3), ld(OW1 + 3 * j + 1), ld(OW1 + 3 * j + 4));
        S.w1[j + 1] = make_float4(ld(OW1 + 3 * j + 2), ld(OW1 + 3 * j + 5), ld(OB1 + j), ld(OB1 + j + 1));
        S.bw[tid] = make_float4(ld(OB2 + j), ld(OB2 + j + 1), ld(OW3 + j), ld(OW3 + j + 1));
    }
    if (tid == 0) {
        S.b3 = ld(OB3);
        S.unscale = __int_as_float((127 - e) << 23);
        tc::fence_mbar_init();
    }
    tc::fence_async_smem();   // the weights, for the tensor cores
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}

// Network output for every thread's row; phase counts the calls.  FULL: W2
// has a low part.  A wait that runs out (wcap polls) sets the contractions' flag
// and goes on with the default bound; ok is cleared if that runs out too.
template <bool FULL>
__device__ __forceinline__ float net_eval(NetShared& S, float u0, float u1, float u2, uint32_t phase, bool& ok,
                                          int* timeout, uint32_t wcap) {
    const uint32_t tm = S.tmem, lanes = (threadIdx.x & 96u) << 16;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int j = 16 * c + q;
            const float4 a = S.w1[2 * j], b = S.w1[2 * j + 1];
            float2 z = make_float2(b.z, b.w);
            z = __ffma2_rn(make_float2(a.x, a.y), f2(u0), z);
            z = __ffma2_rn(make_float2(a.z, a.w), f2(u1), z);
            z = __ffma2_rn(make_float2(b.x, b.y), f2(u2), z);
            const float2 h = tanh2(z);
            const __half2 hh = __float22half2_rn(h);
            const float2 hf = __half22float2(hh);
            const __half2 hl = __float22half2_rn(make_float2(h.x - hf.x, h.y - hf.y));
            hi[q] = *reinterpret_cast<const uint32_t*>(&hh);
            lo[q] = *reinterpret_cast<const uint32_t*>(&hl);
        }
        tc::tmem_st16(tm + lanes + 16 * c, hi);
        tc::tmem_st16(tm + lanes + 32 + 16 * c, lo);
    }
    tc::tmem_wait_st();
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0) {
        tc::fence_after_sync();
        const uint32_t idesc = tc::idesc_f16(NT, H);
        const uint64_t bh = tc::make_desc(tc::smem_u32(S.w2hi), 1024, 128);
        const uint64_t bl = tc::make_desc(tc::smem_u32(S.w2lo), 1024, 128);
        // the small products first; K-steps of 16: 8 columns of A, two K chunks (2 KB) of B
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            tc::mma_f16_ta(tm + 64, tm + 32 + 8 * kk, bh + 128 * kk, idesc, kk > 0);
            if (FULL) tc::mma_f16_ta(tm + 64, tm + 8 * kk, bl + 128 * kk, idesc, 1);
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) tc::mma_f16_ta(tm + 64, tm + 8 * kk, bh + 128 * kk, idesc, 1);
        tc::commit(&S.bar);
    }
    ok = tc::mbar_wait(&S.bar, phase & 1u, wcap);
    if (!ok) {
        if (timeout) *timeout = 1;
        ok = tc::mbar_wait(&S.bar, phase & 1u, NET_WAIT);
    }
    tc::fence_after_sync();
    float s = S.b3;
    const float2 un = f2(S.unscale);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float v[16];
        __syncwarp();
        tc::tmem_ld16_nowait(tm + lanes + 64 + 16 * c, v);
        tc::tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 b = S.bw[8 * c + q];
            const float2 h = tanh2(__ffma2_rn(make_float2(v[2 * q], v[2 * q + 1]), un, make_float2(b.x, b.y)));
            s = fmaf(b.z, h.x, s);
            s = fmaf(b.w, h.y, s);
        }
    }
    return s;
}

__device__ __forceinline__ void net_done(NetShared& S) {
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc::fence_after_sync();
        tc::tmem_dealloc(S.tmem, NET_COLS);
    }
}

template <bool FULL>
__global__ void __launch_bounds__(NT) k_mlp_forward(int n, const float* __restrict__ U,
                                                    const float* __restrict__ params, float* __restrict__ s,
                                                    int* timeout) {
    __shared__ __align__(128) NetShared S;
    net_setup(S, params, !FULL);
    bool ok = true;
    uint32_t phase = 0;
    for (int i0 = blockIdx.x * NT; i0 < n; i0 += gridDim.x * NT, ++phase) {
        const int i = i0 + threadIdx.x;
        const float* u = U + 3 * (int64_t)min(i, n - 1);
        const float v = net_eval<FULL>(S, u[0], u[1], u[2], phase, ok, timeout, NET_WAIT);
        if (i < n) s[i] = ok ? v : __int_as_float(0x7fffffff);
    }
    net_done(S);
}

// ------------------------------------------------------------------ training
// Per-block gradient partials of sum_i w_i (s_i - t_i)^2 over the block's 128
// samples, plus [sum w r^2, sum w] at the end: part[block][kMlpParams + 2].
// FP32 throughout.  256 threads, two per sample, each with half of the hidden
// units: a thread holds its sample's row of activations (or of dz2) in
// registers and streams W2 past it in 16-byte broadcasts, one load per four
// multiply-adds; the 64 x 64 weight gradient is 4 x 4 tiles of registers over
// the samples.  Two activation tiles of 35 KB (dz1 takes h1's place once the
// weight gradient has used it), so that two blocks fit an SM.  (One thread
// per sample with a scalar load per multiply-add and three tiles, one block
// per SM, and 782 partials added one after the other: 400 us for 100,001
// samples.)
constexpr int GB = 128;      // samples per block
constexpr int GT = 256;      // threads per block
constexpr int HP = H + 4;    // padded row of the activation tiles (16-byte aligned, conflict-free)
constexpr int HH = H / 2;

// 64 floats of a tile row into registers
__device__ __forceinline__ void row_load(const float* row, float2 (&v)[HH]) {
#pragma unroll
    for (int q = 0; q < H / 4; ++q) {
        const float4 c = *reinterpret_cast<const float4*>(row + 4 * q);
        v[2 * q] = make_float2(c.x, c.y);
        v[2 * q + 1] = make_float2(c.z, c.w);
    }
}

__global__ void __launch_bounds__(GT, 2) k_mlp_grad_partial(int n, const float* __restrict__ U,
                                                            const float* __restrict__ t,
                                                            const float* __restrict__ wt,
                                                            const float* __restrict__ params,
                                                            float* __restrict__ part) {
    extern __shared__ __align__(16) float sm[];
    float* w = sm;                                // kMlpParams (+ pad to 4)
    float* h1s = w + ((kMlpParams + 3) / 4) * 4;  // h1, then dz1
    float* h2s = h1s + GB * HP;                   // h2, then dz2
    float* us = h2s + GB * HP;                    // GB x 4: features and 1
    float* dss = us + GB * 4;                     // ds
    __shared__ float sp[GB], lw[2][GB];
    load_params(params, w, false);
    __syncthreads();
    const int tid = threadIdx.x, q = tid & (GB - 1), half = tid >> 7, k0 = HH * half;
    const int i = blockIdx.x * GB + q;
    const bool valid = i < n;
    const float u0 = valid ? U[3 * (int64_t)i] : 0.f, u1 = valid ? U[3 * (int64_t)i + 1] : 0.f,
                u2 = valid ? U[3 * (int64_t)i + 2] : 0.f;
    if (half == 0) *reinterpret_cast<float4*>(us + 4 * q) = make_float4(u0, u1, u2, 1.f);
#pragma unroll 4
    for (int j = k0; j < k0 + HH; j += 2) {
        const float* a = w + OW1 + 3 * j;
        float2 z = make_float2(w[OB1 + j], w[OB1 + j + 1]);
        z = __ffma2_rn(make_float2(a[0], a[3]), f2(u0), z);
        z = __ffma2_rn(make_float2(a[1], a[4]), f2(u1), z);
        z = __ffma2_rn(make_float2(a[2], a[5]), f2(u2), z);
        *reinterpret_cast<float2*>(h1s + q * HP + j) = tanh2(z);
    }
    __syncthreads();
    float s = half == 0 ? w[OB3] : 0.f;
    {
        float2 h1[HH];
        row_load(h1s + q * HP, h1);
#pragma unroll 1
        for (int k = k0; k < k0 + HH; k += 2) {
            float2 a[2] = {make_float2(w[OB2 + k], 0.f), make_float2(w[OB2 + k + 1], 0.f)};
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4* row = reinterpret_cast<const float4*>(w + OW2 + H * (k + e));
#pragma unroll
                for (int c4 = 0; c4 < H / 4; ++c4) {
                    const float4 c = row[c4];
                    a[e] = __ffma2_rn(make_float2(c.x, c.y), h1[2 * c4], a[e]);
                    a[e] = __ffma2_rn(make_float2(c.z, c.w), h1[2 * c4 + 1], a[e]);
                }
            }
            const float2 h2 = tanh2(make_float2(a[0].x + a[0].y, a[1].x + a[1].y));
            *reinterpret_cast<float2*>(h2s + q * HP + k) = h2;
            s = fmaf(w[OW3 + k], h2.x, s);
            s = fmaf(w[OW3 + k + 1], h2.y, s);
        }
    }
    if (half == 1) sp[q] = s;
    __syncthreads();
    if (half == 0) {
        float ds = 0.f, wi = 0.f, lnum = 0.f;
        if (valid) {
            wi = wt[i];
            const float r = s + sp[q] - t[i];
            ds = 2.f * wi * r;
            lnum = wi * r * r;
        }
        dss[q] = ds;
        lw[0][q] = lnum;
        lw[1][q] = wi;
    }
    __syncthreads();
    float* P = part + (int64_t)blockIdx.x * (kMlpParams + 2);
    // output layer: gw3[k] = sum_i ds_i h2[i][k] (a warp's lanes along k), and
    // the sums of ds, w r^2 and w (one warp each); four threads per sum, the
    // samples 4 m + part, combined in order
    {
        const int col = tid >> 2, pp = tid & 3;
        float a = 0.f, b = 0.f, c = 0.f, d = 0.f;
        for (int m = pp; m < GB; m += 4) a = fmaf(dss[m], h2s[m * HP + col], a);
        if (col < 1)
            for (int m = pp; m < GB; m += 4) {
                b += dss[m];
                c += lw[0][m];
                d += lw[1][m];
            }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
            d += __shfl_xor_sync(0xffffffffu, d, o);
        }
        if (pp == 0) P[OW3 + col] = a;
        if (tid == 0) {
            P[OB3] = b;
            P[kMlpParams] = c;
            P[kMlpParams + 1] = d;
        }
    }
    __syncthreads();
    // dz2 = ds w3 (1 - h2^2), over h2 (each thread its half)
    {
        const float ds = dss[q];
#pragma unroll 4
        for (int k = k0; k < k0 + HH; k += 4) {
            float4 h = *reinterpret_cast<const float4*>(h2s + q * HP + k);
            h.x = ds * w[OW3 + k] * (1.f - h.x * h.x);
            h.y = ds * w[OW3 + k + 1] * (1.f - h.y * h.y);
            h.z = ds * w[OW3 + k + 2] * (1.f - h.z * h.z);
            h.w = ds * w[OW3 + k + 3] * (1.f - h.w * h.w);
            *reinterpret_cast<float4*>(h2s + q * HP + k) = h;
        }
    }
    __syncthreads();
    // gW2[k][j] = sum_i dz2[i][k] h1[i][j]: thread (ty, tx) rows 4 ty .. and columns 4 tx ..
    {
        const int tx = tid & 15, ty = tid >> 4;
        float2 acc[4][2];
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[a][0] = acc[a][1] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int m = 0; m < GB; ++m) {
            const float4 d = *reinterpret_cast<const float4*>(h2s + m * HP + 4 * ty);
            const float4 h = *reinterpret_cast<const float4*>(h1s + m * HP + 4 * tx);
            const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                acc[a][0] = __ffma2_rn(f2(dv[a]), make_float2(h.x, h.y), acc[a][0]);
                acc[a][1] = __ffma2_rn(f2(dv[a]), make_float2(h.z, h.w), acc[a][1]);
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                P[OW2 + (4 * ty + a) * H + 4 * tx + 2 * b] = acc[a][b].x;
                P[OW2 + (4 * ty + a) * H + 4 * tx + 2 * b + 1] = acc[a][b].y;
            }
    }
    __syncthreads();
    // dz1 = (W2^T dz2) (1 - h1^2), over h1 (each thread its half of the columns)
    {
        float2 d2[HH];
        row_load(h2s + q * HP, d2);
#pragma unroll 1
        for (int j = k0; j < k0 + HH; j += 4) {
            float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
            for (int k = 0; k < H; ++k) {
                const float4 c = *reinterpret_cast<const float4*>(w + OW2 + H * k + j);
                const float dk = (k & 1) ? d2[k >> 1].y : d2[k >> 1].x;
                a0 = __ffma2_rn(make_float2(c.x, c.y), f2(dk), a0);
                a1 = __ffma2_rn(make_float2(c.z, c.w), f2(dk), a1);
            }
            float4 h = *reinterpret_cast<const float4*>(h1s + q * HP + j);
            h.x = a0.x * (1.f - h.x * h.x);
            h.y = a0.y * (1.f - h.y * h.y);
            h.z = a1.x * (1.f - h.z * h.z);
            h.w = a1.y * (1.f - h.w * h.w);
            *reinterpret_cast<float4*>(h1s + q * HP + j) = h;
        }
    }
    __syncthreads();
    // gb2[k] = sum dz2, gW1[j][c] = sum dz1 u_c, gb1[j] = sum dz1: four threads per row
    {
        const int row = tid >> 2, pp = tid & 3;
        float b2 = 0.f, g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int m = pp; m < GB; m += 4) {
            const float4 u = *reinterpret_cast<const float4*>(us + 4 * m);
            const float d = h1s[m * HP + row];
            b2 += h2s[m * HP + row];
            g[0] = fmaf(d, u.x, g[0]);
            g[1] = fmaf(d, u.y, g[1]);
            g[2] = fmaf(d, u.z, g[2]);
            g[3] += d;
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            b2 += __shfl_xor_sync(0xffffffffu, b2, o);
#pragma unroll
            for (int c = 0; c < 4; ++c) g[c] += __shfl_xor_sync(0xffffffffu, g[c], o);
        }
        if (pp == 0) {
            P[OB2 + row] = b2;
            P[OB1 + row] = g[3];
            for (int c = 0; c < 3; ++c) P[OW1 + 3 * row + c] = g[c];
        }
    }
}

// grad[p] = sum_b part[b][p] / sum w (fixed order, two-sum); loss likewise.
// A block covers 32 columns (lanes) and its RW warps take every RW-th block's
// partial; the warps' sums are added in warp order.
constexpr int RW = 16;
__global__ void __launch_bounds__(32 * RW) k_mlp_grad_reduce(int nblk, const float* __restrict__ part,
                                                             float* __restrict__ grad, float* __restrict__ loss) {
    __shared__ float2 red[RW][32], redw[RW];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    auto add = [](float& s, float& c, float v) {
        const float t = s + v, bp = t - s;
        c += (s - (t - bp)) + (v - bp);
        s = t;
    };
    float s = 0.f, c = 0.f, ws = 0.f, wc = 0.f;
#pragma unroll 4
    for (int b = wp; b < nblk; b += RW) {
        const float* row = part + (int64_t)b * (kMlpParams + 2);
        if (p <= kMlpParams) add(s, c, row[p]);
        add(ws, wc, row[kMlpParams + 1]);
    }
    red[wp][lane] = make_float2(s, c);
    if (lane == 0) redw[wp] = make_float2(ws, wc);
    __syncthreads();
    if (wp > 0 || p > kMlpParams) return;
    for (int k = 1; k < RW; ++k) {
        add(s, c, red[k][lane].x);
        c += red[k][lane].y;
        add(ws, wc, redw[k].x);
        wc += redw[k].y;
    }
    const float sw = ws + wc;
    const float inv = sw > 0.f ? 1.f / sw : 0.f;
    if (p < kMlpParams) grad[p] = (s + c) * inv;
    else if (loss) loss[0] = (s + c) * inv;
}

__global__ void k_mlp_adam(int np, float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ g, float lr, float b1, float b2, float c1, float c2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// Network output of one row on the FP32 units, in FP32 throughout (BF16-rounded
// weights w in shared memory).  FP64 contexts take it: their results hold 1e-9
// against each other from build to build, and products of 22 significant bits
// move them by 5e-8 (though no further from 64 bits: 7.2e-8, 7.4e-8 here).  14,000
// plane waves x 40 bands: 222 us, 138 on the tensor cores.
struct SimtShared {
    float w[(kMlpParams + 3) / 4 * 4];
};
// rows (and threads) of a block of the fused preconditioner
template <typename T> __host__ __device__ constexpr int net_rows() { return sizeof(T) == 4 ? NT : 256; }
__device__ __forceinline__ float simt_eval(const float* w, float u0, float u1, float u2) {
    float h1[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
        float z = w[OB1 + j];
        z = fmaf(w[OW1 + 3 * j + 0], u0, z);
        z = fmaf(w[OW1 + 3 * j + 1], u1, z);
        z = fmaf(w[OW1 + 3 * j + 2], u2, z);
        h1[j] = tanhf(z);
    }
    float s = w[OB3];
#pragma unroll 4
    for (int k = 0; k < H; ++k) {
        const float4* row = reinterpret_cast<const float4*>(w + OW2 + H * k);
        float z = w[OB2 + k];
#pragma unroll
        for (int q = 0; q < H / 4; ++q) {
            const float4 c = row[q];
            z = fmaf(c.x, h1[4 * q + 0], z);
            z = fmaf(c.y, h1[4 * q + 1], z);
            z = fmaf(c.z, h1[4 * q + 2], z);
            z = fmaf(c.w, h1[4 * q + 3], z);
        }
        s = fmaf(w[OW3 + k], tanhf(z), s);
    }
    return s;
}

// Fused preconditioner of the PCG step: out = K m g_I with K the TPA factor
// (X_n = 1.5 T_n, T_n the kinetic energy of the residual) and m the network's
// multiplier on the features (log1p(x), log1p(|g|/rms_n), eps_n); m = 1 while
// the correction is suspended (sc->mlp_off > 0) or no weights are set.  The
// network: on the tensor cores in mixed contexts, simt_eval in FP64 ones.
template <typename T>
__global__ void __launch_bounds__(net_rows<T>())
    k_precond_mlp(int npw, const c2<T>* __restrict__ gI, int64_t ld,
                  const T* __restrict__ g2h, const double* __restrict__ sums,
                  int nb, const double2* __restrict__ Theta,
                  const double* __restrict__ wband,
                  const float* __restrict__ params, const PcgScalars* sc,
                  c2<T>* __restrict__ out, int64_t ldo, int* timeout,
                  uint32_t wcap) {
    constexpr bool TC = sizeof(T) == 4;
    __shared__ __align__(128) std::conditional_t<TC, NetShared, SimtShared> S;
    __shared__ float band[5];   // 1/X, -2/X, 1/T, 1/rms, eps
    const bool use = params != nullptr && (sc == nullptr || sc->mlp_off <= 0.0);
    if (use) {
        if constexpr (TC) net_setup(S, params, true);
        else load_params(params, S.w, true);   // (ordered by the first band's barrier)
    }
    // tiles of one row a thread of one band; a block takes a run of them, so that
    // the band's FP64 divisions are rare (FP64: one tile, like its weights)
    constexpr int R = net_rows<T>();
    const int per = (npw + R - 1) / R;
    const int64_t tiles = (int64_t)per * nb;
    const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
    int n = -1;
    bool ok = true;
    uint32_t phase = 0;
    for (int64_t t = t0; t < t1; ++t) {
        const int nt = (int)(t / per), g = (int)(t - (int64_t)nt * per) * R + threadIdx.x;
        if (nt != n) {
            n = nt;
            __syncthreads();
            if (threadIdx.x == 0) {
                const double s0 = fmax(sums[n], 1e-300), s1 = sums[nb + n];
                const double X = 1.5 * s1 / s0;           // sums carry |G|^2 |g|^2
                const double Tn = 0.5 * s1 / s0;
                band[0] = float(1.0 / X);
                band[1] = float(-2.0 / X);
                band[2] = float(1.0 / fmax(Tn, 1e-300));
                band[3] = float(1.0 / sqrt(s0 / npw));
                band[4] = float(Theta[(int64_t)n * nb + n].x / wband[n]);
            }
            __syncthreads();
        }
        const int gc = min(g, npw - 1);
        const c2<T> a = gI[(int64_t)n * ld + gc];
        const float gh = float(g2h[gc]);
        const float x = 2.f * gh * band[0];
        const float num = 27.f + x * (18.f + x * (12.f + 8.f * x));
        float K = band[1] * num / (num + 16.f * x * x * x * x);
        if (use) {
            const float amp = sqrtf(float(a.x) * float(a.x) + float(a.y) * float(a.y));
            const float u0 = log1pf(gh * band[2]), u1 = log1pf(amp * band[3]);
            float s;
            if constexpr (TC) s = net_eval<false>(S, u0, u1, band[4], phase++, ok, timeout, wcap);
            else s = simt_eval(S.w, u0, u1, band[4]);
            K *= ok ? expf(fminf(fmaxf(s, -3.f), 3.f)) : __int_as_float(0x7fffffff);
        }
        if (g < npw) out[(int64_t)n * ldo + g] = mk<T>(T(K) * a.x, T(K) * a.y);
    }
    if constexpr (TC)
        if (use) net_done(S);
}

template <typename T>
__global__ void k_mlp_features(int npw, const c2<T>* __restrict__ gI, int64_t ld, const T* __restrict__ g2h,
                               const double* __restrict__ sums, int nb, const double2* __restrict__ Theta,
                               const double* __restrict__ wband, float* __restrict__ U) {
    __shared__ float band[3];   // 1/T, 1/rms, eps
    const int n = blockIdx.y;
    if (threadIdx.x == 0) {
        const double s0 = fmax(sums[n], 1e-300), s1 = sums[nb + n];
        band[0] = float(1.0 / fmax(0.5 * s1 / s0, 1e-300));
        band[1] = float(1.0 / sqrt(s0 / npw));
        band[2] = float(Theta[(int64_t)n * nb + n].x / wband[n]);
    }
    __syncthreads();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= npw) return;
    const c2<T> a = gI[(int64_t)n * ld + g];
    const float amp = sqrtf(float(a.x) * float(a.x) + float(a.y) * float(a.y));
    float* u = U + 3 * ((int64_t)n * npw + g);
    u[0] = log1pf(float(g2h[g]) * band[0]);
    u[1] = log1pf(amp * band[1]);
    u[2] = band[2];
}

size_t grad_smem() {
    return sizeof(float) * (((kMlpParams + 3) / 4) * 4 + 2 * GB * HP + GB * 4 + GB);
}

}  // namespace

// blocks for so many tiles of rows: four per SM at most (tensor memory)
static int net_blocks(int64_t tiles) {
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (int)std::min<int64_t>(tiles, 4 * (int64_t)sms);
}

void mlp_forward(int n, const float* U, const float* params, bool bf16, float* s, cudaStream_t st) {
    if (n <= 0) return;
    const int blocks = net_blocks((n + NT - 1) / NT);
    roks::count_launch();
    if (bf16) k_mlp_forward<false><<<blocks, NT, NET_PAD, st>>>(n, U, params, s, tcg_timeout_flag());
    else k_mlp_forward<true><<<blocks, NT, NET_PAD, st>>>(n, U, params, s, tcg_timeout_flag());
}

size_t mlp_grad_work_floats(int n) { return (size_t)((n + GB - 1) / GB) * (kMlpParams + 2); }

void mlp_grad(int n, const float* U, const float* t, const float* w, const float* params, float* work, float* grad,
              float* loss, cudaStream_t st) {
    const int nblk = (n + GB - 1) / GB;
    if (nblk <= 0) return;
    const size_t sm = grad_smem();
    allow_smem(k_mlp_grad_partial, sm);
    roks::count_launch(), k_mlp_grad_partial<<<nblk, GT, sm, st>>>(n, U, t, w, params, work);
    roks::count_launch(), k_mlp_grad_reduce<<<(kMlpParams + 1 + 31) / 32, 32 * RW, 0, st>>>(nblk, work, grad, loss);
}

void mlp_adam(float* p, float* m, float* v, const float* g, int step, float lr, float b1, float b2, float eps,
              cudaStream_t st) {
    const double c1 = 1.0 / (1.0 - std::pow((double)b1, step));
    const double c2 = 1.0 / (1.0 - std::pow((double)b2, step));
    roks::count_launch(), k_mlp_adam<<<(kMlpParams + 255) / 256, 256, 0, st>>>(kMlpParams, p, m, v, g, lr, b1, b2,
                                                                             (float)c1, (float)c2, eps);
}

template <typename T>
void precondition_mlp(int npw, int nb, const c2<T>* gI, int64_t ld, const T* g2h, const double* sums,
                      const double2* Theta, const double* wband, const float* params, const PcgScalars* sc,
                      c2<T>* out, int64_t ldo, cudaStream_t st) {
    constexpr bool TC = sizeof(T) == 4;
    constexpr int R = net_rows<T>();
    const int64_t tiles = (int64_t)((npw + R - 1) / R) * nb;
    roks::count_launch(), k_precond_mlp<T><<<TC ? net_blocks(tiles) : (int)tiles, R, TC ? NET_PAD : 0, st>>>(
                              npw, gI, ld, g2h, sums, nb, Theta, wband, params, sc, out, ldo, tcg_timeout_flag(),
                              wait_polls());
}

template <typename T>
void mlp_features(int npw, int nb, const c2<T>* g, int64_t ld, const T* g2h, const double* sums,
                  const double2* Theta, const double* wband, float* U, cudaStream_t st) {
    dim3 grid((npw + 255) / 256, nb);
    roks::count_launch(), k_mlp_features<T><<<grid, 256, 0, st>>>(npw, g, ld, g2h, sums, nb, Theta, wband, U);
}
template void mlp_features<float>(int, int, const float2*, int64_t, const float*, const double*, const double2*,
                                  const double*, float*, cudaStream_t);
template void mlp_features<double>(int, int, const double2*, int64_t, const double*, const double*, const double2*,
                                   const double*, float*, cudaStream_t);

template void precondition_mlp<float>(int, int, const float2*, int64_t, const float*, const double*, const double2*,
                                      const double*, const float*, const PcgScalars*, float2*, int64_t, cudaStream_t);
template void precondition_mlp<double>(int, int, const double2*, int64_t, const double*, const double*,
                                       const double2*, const double*, const float*, const PcgScalars*, double2*,
                                       int64_t, cudaStream_t);

}  // namespace roks
