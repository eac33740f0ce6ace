// k_tcgemm.cu -- complex FP32 contractions of the large blocks (hundreds of
// bands, thousands of projectors) on the 5th-generation tensor cores
// (tcgen05, kind::f16), mixed-precision path:
//
//   CN:  C (M x N, FP64 out) = A^H B,          A: K x M, B: K x N (K: plane waves)
//   NN:  Cout (M x N) = alpha A B + beta Cin,   A: M x K tall, B: K x N small (FP64)
//
// Precision (three FP16 products per FP32 product).  Every column x of an
// operand is scaled by a power of two that puts its largest element into
// [2^14, 2^15), then split as x = hi + lo, hi = fp16(x), lo = fp16(x - hi):
// 22 significant bits for every element above 2^-29 of its column's largest
// one, and an absolute error of 2^-40 of that largest one below.  A product
// is lo.hi + hi.lo + hi.hi.  That is the accuracy of a TF32 split (the same
// 11-bit significands) at twice the MMA rate and half the operand bytes.
// The tensor cores' FP32 accumulation truncates, which biases sums of
// like-signed terms, so a few products go into a fresh tensor-memory
// accumulator, the small cross terms first, and the drain warps add its result
// into FP32 sums in registers (round to nearest).  A B: every stage (32 complex
// K).  A^H B, whose sums are a thousand stages long: every half stage, and no
// sum in registers goes on for more than GB_PIECE stages: it ends as a segment,
// and the segments are added with compensation.  (Drained by the stage, norms
// come out 2.3e-7 low; by half stages 0.8e-7; 1.2e-7 in the TF32 form this
// replaces.  At mgo-120, errors of F and of a DIIS step's psi: half stages in one
// sum 1.40e-7 and 1.79e-7, in segments of at most 128, 96 and 64 stages 1.18e-7
// and 1.77e-7, 1.15e-7 and 1.52e-7, 1.11e-7 and 1.50e-7; the TF32 form 1.48e-7 and
// 2.16e-7.  Quarter stages, whose longer sums lose more than the shorter
// accumulations gain, 1.65e-7 and 2.5e-7.  It takes 0.9% of an apply's time there,
// 1.4% with segments of 64.)  Nothing is scaled to give back what is lost: sums
// without truncation are exact.
//
// Images.  A block X (rows x cols, column major) is split once per use, by
// k_tcg_split, into an image in global memory that the MMAs can read as it
// is: for each chunk q of 8 rows, part p (hi, lo) and plane (re, im), all
// the column groups g of 8, each a 128-byte core matrix of 8 columns x 8
// rows (16 bytes per column):
//   byte ((4 q + 2 p + plane) G + g) 128 + 16 (col % 8) + 2 (row % 8).
// The planes are kept apart, so a complex product is four real ones whose
// operands the MMA descriptors choose, the minus sign being the instruction
// descriptor's negate bit; one image serves as the A or the B of A^H B
// (contraction over the rows: K-major operands) and as the A of A B
// (contraction over the columns: MN-major).  It has the size of X itself.
// A kernel that converts operands on their way through shared memory (the
// TF32 form this replaces) repeats the conversion for every tile and spent
// its time in the hand-over between conversion and MMA.
//
// One CTA per SM (192 KB of shared memory in three stages, all 512
// tensor-memory columns), three warpgroups:
//   warp 0      producer: one tensor copy per operand and stage;
//   warp 1      one thread issues the 24 MMAs of a stage (M = 128, N = tn,
//               K = 16) into one of two accumulators, 128 columns for the
//               real parts and 128 for the imaginary parts;
//   warps 4-11  drain: lane quadrant warp % 4, up to 64 complex columns each
//               (128 sums a thread: the first warpgroup gives them registers).
// Every wait is bounded (the context's wait cap); a wait that gives up sets
// a device flag and the CTA winds down: copies and MMAs in flight are waited
// for with the default bound before the tensor memory is freed.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>

#include "roks_impl.cuh"
#include "tc_sm103.cuh"

namespace roks {

// tiled map of 64-bit words (k_stream.cu)
bool tensor_map_words(CUtensorMap* map, const void* ptr, int rank, const uint64_t* dims, const uint64_t* strides,
                      const uint32_t* box);

static __device__ int g_tcg_timeout;

namespace {

constexpr int GB_M = 128;     // tile rows (tensor-memory lanes)
constexpr int GB_NT = 128;    // most complex columns of a tile
constexpr int GB_KC = 32;     // complex K per stage
constexpr int GB_ST = 3;      // stages
constexpr int GB_ACC = 2;     // accumulators (256 tensor-memory columns each)
constexpr int GB_DRAIN = 8;   // drain warps
constexpr int GB_PIECE = 96;  // A^H B: most stages of a running sum (a segment)
constexpr int GB_THREADS = (4 + GB_DRAIN) * 32;
constexpr uint32_t GB_ABYTES = GB_M * GB_KC * 8;      // 32 KB
constexpr uint32_t GB_SLOT = 2 * GB_ABYTES;           // A, then B (tn x KC x 8 bytes)
constexpr uint32_t GB_TCOLS = 512;
constexpr uint32_t GB_DEFAULT_WAIT = 1u << 26;
constexpr size_t GB_SMEM = (size_t)GB_ST * GB_SLOT + 1024;

// Bounded wait on a phase; gives up after `cap` polls, or early once another
// role of the CTA has given up (checked every 1024 polls).
__device__ __forceinline__ bool gwait(uint64_t* bar, uint32_t parity, uint32_t cap, volatile int* failed) {
    for (uint32_t i = 0; i < cap; ++i) {
        if (tc::mbar_try(bar, parity)) return true;
        if ((i & 1023u) == 1023u && *failed) return false;
    }
    return false;
}

// The same wait by every lane of a warp, with one outcome for the warp (the
// warp-wide instructions after it need all lanes): true only if every lane
// saw the phase complete.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, uint32_t cap, volatile int* failed) {
    const bool ok = gwait(bar, parity, cap, failed);
    return __all_sync(0xffffffffu, ok) != 0;
}

__device__ __forceinline__ void give_up(volatile int* failed) {
    *failed = 1;
    g_tcg_timeout = 1;
}

// 2^e as a float, e in [-126, 127]
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// CTA-loop schedules, at most one CTA per SM:
// * A^H B, stream-K: CTA c takes the units c len .. (c + 1) len - 1 of the
//   (tile, stage) sequence, stage fastest (tile t: M tile t % fast, N tile t /
//   fast), and writes the partial sums of each tile that it touches, a segment
//   for every `piece` stages of it, to its slots c * maxseg + 0, 1, ...;
// * A B, persistent: units = tiles, CTA c takes the whole tiles c, c + ctas,
//   ... (tile t: N tile t % fast, M tile t / fast), its pipeline running on
//   across them, and writes each tile's result as it completes.
struct SkPlan {
    int64_t units = 0, len = 0;
    int ctas = 0, maxseg = 0, fast = 0;
    int tn = 0;   // complex columns of a tile (a multiple of 16)
    int piece = 0;   // A^H B: stages of a segment
    // segments of so many stages of a tile
    __host__ __device__ int segments(int stages) const { return (stages + piece - 1) / piece; }
};

template <bool NN>
__global__ void __launch_bounds__(GB_THREADS, 1)
    k_tcgemm(int M, int N, int total_stages, SkPlan sk, const __grid_constant__ CUtensorMap tmA,
             const __grid_constant__ CUtensorMap tmB, const int* __restrict__ exB, float2* __restrict__ part,
             const float2* Cin, int64_t ldcin, float2* Cout, int64_t ldc, float alpha, float beta, uint32_t wcap) {
    extern __shared__ __align__(1024) unsigned char gb_smem[];
    __shared__ __align__(8) uint64_t full[GB_ST], empty[GB_ST], acc_full[GB_ACC], acc_empty[GB_ACC], mma_done;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int failed;
    unsigned char* ring = gb_smem + ((1024u - (tc::smem_u32(gb_smem) & 1023u)) & 1023u);
    const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;
    constexpr int DS = NN ? 1 : 2;   // drain steps of a stage
    const int64_t u0 = NN ? 0 : sk.len * blockIdx.x;
    // the first tile and stage (the loops then step them); after a tile's
    // last stage the next tile is t + tstep
    const int t_first = NN ? (int)blockIdx.x : (int)(u0 / total_stages);
    const int s_first = NN ? 0 : (int)(u0 - (int64_t)t_first * total_stages);
    const int tstep = NN ? sk.ctas : 1;
    const int ns = NN ? (int)((sk.units - blockIdx.x + sk.ctas - 1) / sk.ctas) * total_stages
                      : (int)(min(sk.units, u0 + sk.len) - u0);

    if (tid == 0) {
        for (int s = 0; s < GB_ST; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < GB_ACC; ++s) {
            tc::mbar_init(&acc_full[s], 1);
            tc::mbar_init(&acc_empty[s], GB_DRAIN);
        }
        tc::mbar_init(&mma_done, 1);
        failed = 0;
        tc::fence_mbar_init();
    }
    if (warp == 0) tc::tmem_alloc(&tmem_base, GB_TCOLS);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_base;
    const uint32_t wb = (uint32_t)sk.tn * 16u;   // bytes of one (q, part, plane) row of the B tile

    // 384 threads x 168 registers at launch = 128 x 56 + 256 x 224
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        // ------------------------------------------------ producer
        if (warp == 0 && tc::elect_one()) {
            int issued = 0, t_cur = t_first, s_cur = s_first;
            for (int i = 0; i < ns; ++i) {
                const int ma = NN ? t_cur / sk.fast : t_cur % sk.fast;
                const int nb_ = NN ? t_cur % sk.fast : t_cur / sk.fast;
                const int ks = s_cur;
                if (++s_cur == total_stages) {
                    s_cur = 0;
                    t_cur += tstep;
                }
                const int sl = i % GB_ST;
                if (i >= GB_ST && !gwait(&empty[sl], (uint32_t)((i / GB_ST - 1) & 1), wcap, &failed)) {
                    give_up(&failed);
                    break;
                }
                unsigned char* a = ring + (size_t)sl * GB_SLOT;
                tc::mbar_arrive_expect_tx(&full[sl], GB_ABYTES + 16u * wb);
                // A: CN 16 groups x 4 chunks of rows, NN 16 chunks x 4 groups
                if (NN) tc::tma_4d(a, &tmA, ma * 16, ks * 4, 0, &full[sl]);
                else tc::tma_2d(a, &tmA, ma * 256, ks * 16, &full[sl]);
                tc::tma_2d(a + GB_ABYTES, &tmB, nb_ * sk.tn * 2, ks * 16, &full[sl]);
                issued = i + 1;
            }
            // copies still in flight complete before the CTA may exit
            for (int i = issued > GB_ST ? issued - GB_ST : 0; i < issued; ++i)
                gwait(&full[i % GB_ST], (uint32_t)((i / GB_ST) & 1), GB_DEFAULT_WAIT, &failed);
        }
        // ------------------------------------------------ MMA issue
        if (warp == 1) {
            // (one elected lane of a whole warp issues: 57 cycles an MMA; under a
            // test of the lane the loop's bookkeeping was per lane, 85 cycles,
            // and P (D B) at mgo-120 took 479 us instead of 448)
            const bool leader = tc::elect_one();
            // A: K-major over [chunk 8192][part 4096][plane 2048][group 128], or
            // MN-major over [part 16384][plane 8192][group 2048][chunk 128];
            // B: K-major over [chunk 4 wb][part 2 wb][plane wb][group 128]
            const uint32_t idesc = tc::idesc_f16(GB_M, sk.tn) | (NN ? tc::IDESC_A_MN : 0u);
            const uint64_t da0 = NN ? tc::make_desc(0, 2048, 128) : tc::make_desc(0, 8192, 128);
            const uint64_t db0 = tc::make_desc(0, 4 * wb, 128);
            constexpr uint32_t a_part = NN ? 16384 : 4096, a_plane = NN ? 8192 : 2048, a_k = NN ? 4096 : 16384;
            bool ok = true;
            int sl = 0;
            for (int i = 0; i < ns && ok; ++i) {
                if (!warp_wait(&full[sl], (uint32_t)((i / GB_ST) & 1), wcap, &failed)) {
                    ok = false;
                    break;
                }
                const uint32_t sa = tc::smem_u32(ring + (size_t)sl * GB_SLOT), sb = sa + GB_ABYTES;
#pragma unroll
                for (int h = 0; h < DS; ++h) {
                    const int e = DS * i + h, b = e % GB_ACC;   // drain step and its accumulator
                    if (e >= GB_ACC && !warp_wait(&acc_empty[b], (uint32_t)((e / GB_ACC - 1) & 1), wcap, &failed)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    const uint32_t d = tmem + (uint32_t)(b * 256);
                    // D(out) += A(part pa, plane xa) B(part pb, plane xb) over the step's K-steps of 16
                    auto mm = [&](int out, int pa, int xa, int pb, int xb, bool neg, uint32_t first) {
#pragma unroll
                        for (int k = 0; k < 2 / DS; ++k) {
                            const int kk = h + k;
                            tc::mma_f16(d + 128u * out, da0 + ((sa + pa * a_part + xa * a_plane + kk * a_k) >> 4),
                                        db0 + ((sb + pb * 2 * wb + xb * wb + kk * 8 * wb) >> 4),
                                        neg ? (idesc | tc::IDESC_NEG_A) : idesc, (first && k == 0) ? 0u : 1u);
                        }
                    };
                    // the small cross terms first, then the hi.hi products, which alone
                    // meet a large partial sum.  CN: re = Ar.Br + Ai.Bi, im = Ar.Bi -
                    // Ai.Br; NN: re = Ar.Br - Ai.Bi, im = Ar.Bi + Ai.Br.  The last
                    // products are those with Br: in A B, where B is near a real
                    // multiple of the identity or has a real diagonal, its large
                    // elements are then truncated least often
                    if (leader) {
#pragma unroll
                        for (int o = 0; o < 2; ++o) {
                            const bool n0 = !NN && o == 1, n1 = NN && o == 0;   // the terms with Br, with Bi
                            mm(o, 1, 1 - o, 0, 1, n1, 1u);
                            mm(o, 0, 1 - o, 1, 1, n1, 0u);
                            mm(o, 1, o, 0, 0, n0, 0u);
                            mm(o, 0, o, 1, 0, n0, 0u);
                            mm(o, 0, 1 - o, 0, 1, n1, 0u);
                            mm(o, 0, o, 0, 0, n0, 0u);
                        }
                        tc::commit(&acc_full[b]);
                        if (h == DS - 1) tc::commit(&empty[sl]);   // the slot is free once these MMAs complete
                    }
                    __syncwarp();
                }
                sl = sl == GB_ST - 1 ? 0 : sl + 1;
            }
            if (!ok) give_up(&failed);
            // every MMA issued completes before the tensor memory is freed
            if (leader) tc::commit(&mma_done);
            __syncwarp();
            gwait(&mma_done, 0u, GB_DEFAULT_WAIT, &failed);
        }
        __syncwarp();   // the role's lane rejoins its warp
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        // ------------------------------------------------ drain
        const int q = warp & 3;               // lane quadrant
        // complex columns cg .. cg + ncol - 1: the tile's groups of 16 shared out
        // between the two warpgroups (64 to the first and the rest to the second
        // made half stages of 80-column tiles wait for the drain)
        const int half = 16 * ((sk.tn / 16 + 1) / 2);
        const int cg = warp < 8 ? 0 : half, ncol = warp < 8 ? half : sk.tn - half;
        const int r = 32 * q + lane;          // tile row
        float2 re[32], im[32];                // column pairs
#pragma unroll
        for (int j = 0; j < 32; ++j) re[j] = im[j] = make_float2(0.f, 0.f);
        bool ok = true;
        int left = total_stages - s_first, seg = 0, in_seg = 0, t_cur = t_first;
        for (int e = 0; e < DS * ns; ++e) {
            const int b = e % GB_ACC;
            if (!warp_wait(&acc_full[b], (uint32_t)((e / GB_ACC) & 1), wcap, &failed)) {
                ok = false;
                break;
            }
            tc::fence_after_sync();
            const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * 256 + cg);
            if (NN && beta != 0.f && left == total_stages && (lane & 15) == 0) {
                // a tile's first stage: its Cin on the way to L2
                const int no = (t_cur % sk.fast) * sk.tn + cg, m = (t_cur / sk.fast) * GB_M + r;
                const int nc = min(ncol, N - no);
                for (int j = 0; j < nc && m < M; ++j)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(Cin + (int64_t)(no + j) * ldcin + m));
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (16 * c >= ncol) break;
                float v[16], w[16];
                tc::tmem_ld16_nowait(ta + 16 * c, v);
                tc::tmem_ld16_nowait(ta + 128 + 16 * c, w);
                tc::tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    re[8 * c + j] = __fadd2_rn(re[8 * c + j], make_float2(v[2 * j], v[2 * j + 1]));
                    im[8 * c + j] = __fadd2_rn(im[8 * c + j], make_float2(w[2 * j], w[2 * j + 1]));
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&acc_empty[b]);
            if (DS > 1 && e % DS < DS - 1) continue;
            // the last stage of a tile (CN: or of a segment) in this CTA's run: its
            // sums go out (NN: the result; CN: the partial sums to the segment
            // slot) and restart
            --left;
            if (left == 0 || e == DS * ns - 1 || (!NN && ++in_seg == sk.piece)) {
                if (NN) {
                    const int m = (t_cur / sk.fast) * GB_M + r;
                    const int no = (t_cur % sk.fast) * sk.tn + cg;
                    const int nc = min(ncol, N - no);   // this warp's columns
                    if (m < M) {
                        // 32 columns at a time, every load before the first store
                        // (Cin may be Cout, so the compiler keeps their order: one
                        // load in flight per thread took 25 us a tile)
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            float2 ci[32];
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                const int jj = 32 * c + j;
                                ci[j] = make_float2(0.f, 0.f);
                                if (beta != 0.f && jj < nc) ci[j] = Cin[(int64_t)(no + jj) * ldcin + m];
                            }
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                const int jj = 32 * c + j;
                                if (jj < nc) {
                                    const float2 x = re[jj >> 1], y = im[jj >> 1];
                                    const float sc = alpha * pow2f(-exB[no + jj]);
                                    const float2 o = (j & 1) ? make_float2(sc * x.y, sc * y.y)
                                                             : make_float2(sc * x.x, sc * y.x);
                                    Cout[(int64_t)(no + jj) * ldc + m] =
                                        make_float2(fmaf(beta, ci[j].x, o.x), fmaf(beta, ci[j].y, o.y));
                                }
                            }
                        }
                    }
                } else {
                    float2* Pp = part + (((int64_t)blockIdx.x * sk.maxseg + seg) * sk.tn + cg) * GB_M + r;
#pragma unroll
                    for (int j = 0; j < 64; ++j)
                        if (j < ncol)
                            Pp[(int64_t)j * GB_M] = (j & 1) ? make_float2(re[j >> 1].y, im[j >> 1].y)
                                                            : make_float2(re[j >> 1].x, im[j >> 1].x);
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) re[j] = im[j] = make_float2(0.f, 0.f);
                ++seg;
                in_seg = 0;
                if (left == 0) {
                    t_cur += tstep;
                    left = total_stages;
                }
            }
        }
        if (!ok) give_up(&failed);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, GB_TCOLS);
    }
}

// ------------------------------------------------------------------ operand images
// Column group g = blockIdx.y, its chunks of 8 rows shared out over the
// cluster's CTAs (blockIdx.x): the columns' largest finite elements first
// (reduced over the cluster), then the split.  Lane = chunk % 4 + 4 (column
// % 8): a warp reads 256 contiguous bytes of each column and writes whole
// 128-byte core matrices.  The second read of the block mostly comes from L2.
// D: the element type (float2, or double2 for the small B of A B); exA: the
// exponents of the A image it multiplies, taken out of B's rows; VEC: 16-byte
// loads of float2 (the column bases are 16-byte aligned).
constexpr int SP_THREADS = 256;
constexpr int SP_CL = 8;

template <typename D, bool VEC>
__device__ __forceinline__ void split_load(const D* __restrict__ col, int r0, int R, const int* __restrict__ exA,
                                           float2 (&x)[8]) {
    if constexpr (VEC) {
        if (r0 + 8 <= R) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 v = *reinterpret_cast<const float4*>(col + r0 + 2 * k);
                x[2 * k] = make_float2(v.x, v.y);
                x[2 * k + 1] = make_float2(v.z, v.w);
            }
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        x[k] = make_float2(0.f, 0.f);
        if (r0 + k < R) {
            const D v = col[r0 + k];
            x[k] = make_float2((float)v.x, (float)v.y);
            if (exA) {
                const float s = pow2f(-exA[r0 + k]);
                x[k].x *= s;
                x[k].y *= s;
            }
        }
    }
}

template <typename D, bool VEC>
__global__ void __launch_bounds__(SP_THREADS) k_tcg_split(int R, int V, const D* __restrict__ X, int64_t ld, int Q,
                                                          int G, const int* __restrict__ exA,
                                                          unsigned char* __restrict__ img, int* __restrict__ ex) {
    namespace cg = cooperative_groups;
    __shared__ float red[SP_THREADS / 32][8];
    __shared__ float mine[8], top[8];
    cg::cluster_group cl = cg::this_cluster();
    const int ncl = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int g = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int vl = lane >> 2, v = 8 * g + vl;
    const int per = (Q + ncl - 1) / ncl;
    const int q1 = min(Q, (rank + 1) * per);
    const D* col = X + (int64_t)(v < V ? v : 0) * ld;
    const int R_ = v < V ? R : 0;   // columns past the end: zeros
    float m = 0.f;
    for (int q = rank * per + 4 * warp + (lane & 3); q < q1; q += SP_THREADS / 8) {
        float2 x[8];
        split_load<D, VEC>(col, 8 * q, R_, exA, x);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float a = fmaxf(fabsf(x[k].x), fabsf(x[k].y));
            if (a <= 3.4028234e38f) {   // finite (an infinity must not scale the others away)
                m = fmaxf(m, a);
            } else {
                if (fabsf(x[k].x) <= 3.4028234e38f) m = fmaxf(m, fabsf(x[k].x));
                if (fabsf(x[k].y) <= 3.4028234e38f) m = fmaxf(m, fabsf(x[k].y));
            }
        }
    }
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    if ((lane & 3) == 0) red[warp][vl] = m;
    __syncthreads();
    if (threadIdx.x < 8) {
        float t = 0.f;
        for (int w = 0; w < SP_THREADS / 32; ++w) t = fmaxf(t, red[w][threadIdx.x]);
        mine[threadIdx.x] = t;
    }
    cl.sync();
    if (threadIdx.x < 8) {
        float t = 0.f;
        for (int k = 0; k < ncl; ++k) t = fmaxf(t, cl.map_shared_rank(mine, k)[threadIdx.x]);
        top[threadIdx.x] = t;
    }
    cl.sync();
    // the exponent that puts the largest element into [2^14, 2^15)
    const float t = top[vl];
    int e = 0;
    if (t > 0.f) e = min(126, 14 - ilogbf(t));
    const float s = pow2f(e);
    if (rank == 0 && threadIdx.x < 32 && (lane & 3) == 0) ex[v] = e;
    for (int q = rank * per + 4 * warp + (lane & 3); q < q1; q += SP_THREADS / 8) {
        float2 x[8];
        split_load<D, VEC>(col, 8 * q, R_, exA, x);
        uint4 o[4];   // hi re, hi im, lo re, lo im
        __half2* h = reinterpret_cast<__half2*>(o);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 a = make_float2(s * x[2 * k].x, s * x[2 * k + 1].x);   // two real parts
            const float2 b = make_float2(s * x[2 * k].y, s * x[2 * k + 1].y);
            const __half2 ha = __float22half2_rn(a), hb = __float22half2_rn(b);
            const float2 fa = __half22float2(ha), fb = __half22float2(hb);
            h[k] = ha;
            h[4 + k] = hb;
            h[8 + k] = __float22half2_rn(make_float2(a.x - fa.x, a.y - fa.y));
            h[12 + k] = __float22half2_rn(make_float2(b.x - fb.x, b.y - fb.y));
        }
        unsigned char* dst = img + ((int64_t)4 * q * G + g) * 128 + 16 * vl;
#pragma unroll
        for (int k = 0; k < 4; ++k) *reinterpret_cast<uint4*>(dst + (int64_t)k * G * 128) = o[k];
    }
}

template <typename D, bool VEC>
bool launch_split(int R, int V, const D* X, int64_t ld, const int* exA, const TcImage& im, cudaStream_t st) {
    const int Q = (R + 7) / 8, G = (V + 7) / 8;
    cudaLaunchConfig_t cfg = {};
    // a CTA's share of a column group is at least four rounds of its warps
    int ncl = 1;
    while (ncl < SP_CL && Q > 2 * ncl * SP_THREADS / 8) ncl *= 2;
    cfg.gridDim = dim3(ncl, G, 1);
    cfg.blockDim = dim3(SP_THREADS, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ncl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    roks::count_launch();
    return cudaLaunchKernelEx(&cfg, k_tcg_split<D, VEC>, R, V, X, ld, Q, G, exA,
                              static_cast<unsigned char*>(im.data), im.ex) == cudaSuccess;
}

// ------------------------------------------------------------------ partial sums
// C (M x N, FP64) of tile t: the segments of the CTAs whose runs meet the
// tile's units t T .. (t + 1) T - 1 (one each where runs are short, else one for
// every GB_PIECE stages).  A warp covers 32 rows of one column; RG
// warps of a block take every RG-th CTA of the tile, the block's other warps
// further columns.  Compensated FP32 sums (FP64 arithmetic is slow on this
// part), combined in warp order; the operands' scales come out at the end.
// The order is fixed.
template <int RG>
__global__ void __launch_bounds__(256) k_tcg_reduce_sk(int M, int N, int mt, int T, SkPlan sk,
                                                       const int* __restrict__ exA, const int* __restrict__ exB,
                                                       const float2* __restrict__ part, double2* __restrict__ C,
                                                       int ldc) {
    constexpr int NW = 8 / RG;   // columns of a block
    __shared__ float4 red[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, wg = w % RG;
    const int m = blockIdx.x * 32 + lane, n = blockIdx.y * NW + w / RG;
    float sx = 0.f, cx = 0.f, sy = 0.f, cy = 0.f;
    auto add = [](float& s, float& e, float v) {
        const float u = s + v, bp = u - s;
        e += (s - (u - bp)) + (v - bp);
        s = u;
    };
    if (n < N) {
        const int t = (blockIdx.x * 32) / GB_M + (n / sk.tn) * mt;
        const int64_t off = (int64_t)(n % sk.tn) * GB_M + (m % GB_M);
        const int64_t ta = (int64_t)t * T;
        const int c0 = (int)(ta / sk.len), c1 = (int)((ta + T - 1) / sk.len);
        if (sk.len <= sk.piece) {
#pragma unroll 4
            for (int c = c0 + wg; c <= c1; c += RG) {
                // a run that starts before the tile has it further on
                const int seg = c == c0 ? t - (int)(c0 * sk.len / T) : 0;
                const float2 p = part[((int64_t)c * sk.maxseg + seg) * sk.tn * GB_M + off];
                add(sx, cx, p.x);
                add(sy, cy, p.y);
            }
        } else {
            for (int c = c0 + wg; c <= c1; c += RG) {
                // the segments of the run's tiles before this one, then this one's
                const int64_t u0 = c * sk.len;
                const int tb = (int)(u0 / T), sb = (int)(u0 - (int64_t)tb * T);
                const int seg = tb < t ? sk.segments(T - sb) + (t - tb - 1) * sk.segments(T) : 0;
                const int ns = sk.segments((int)(min(u0 + sk.len, ta + T) - max(u0, ta)));
                const float2* p = part + ((int64_t)c * sk.maxseg + seg) * sk.tn * GB_M + off;
#pragma unroll 4
                for (int q = 0; q < ns; ++q, p += sk.tn * GB_M) {
                    const float2 v = *p;
                    add(sx, cx, v.x);
                    add(sy, cy, v.y);
                }
            }
        }
    }
    if constexpr (RG > 1) {
        red[w][lane] = make_float4(sx, cx, sy, cy);
        __syncthreads();
        if (wg > 0) return;
        for (int k = 1; k < RG; ++k) {
            const float4 v = red[w + k][lane];
            add(sx, cx, v.x);
            add(sy, cy, v.z);
            cx += v.y;
            cy += v.w;
        }
    }
    if (m >= M || n >= N) return;
    const double sc = __hiloint2double((1023 - exA[m] - exB[n]) << 20, 0);
    C[(int64_t)n * ldc + m] =
        make_double2(sc * ((double)sx + (double)cx), sc * ((double)sy + (double)cy));
}

int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 152;
        }
    }
    return n;
}

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

int stages(int k) { return (k + GB_KC - 1) / GB_KC; }
int tile_cols(int N, int nt) { return ((N + nt - 1) / nt + 15) / 16 * 16; }

// Runs of A^H B's unit sequence, in half waves of one CTA per SM
// (tcg_set_waves): 2, one run per SM, is the default; the autotuner also
// times 5 and 8, more and shorter runs.
int g_waves_x2 = 2;

// A^H B: the fewest N tiles of equal width; runs of no fewer than four stages
// (a run that short is mostly pipeline fill, and every CTA leaves a partial
// tile to add)
SkPlan cn_plan(int M, int N, int K, int waves_x2) {
    SkPlan p;
    const int mt = (M + GB_M - 1) / GB_M, nt = (N + GB_NT - 1) / GB_NT, T = stages(K);
    p.tn = tile_cols(N, nt);
    p.fast = mt;
    p.units = (int64_t)mt * nt * T;
    p.ctas = (int)std::min<int64_t>(sm_count() * waves_x2 / 2, std::max<int64_t>(1, p.units / 4));
    p.len = (p.units + p.ctas - 1) / p.ctas;
    p.ctas = (int)((p.units + p.len - 1) / p.len);
    // segments of equal length; long runs: whole tiles, what is left over, and a
    // short segment at either end
    const int n = (int)((p.len + GB_PIECE - 1) / GB_PIECE);
    p.piece = (int)((p.len + n - 1) / n);
    p.maxseg = n == 1 ? (int)((p.len + T - 1) / T) + 1
                      : (int)(p.len / T) * p.segments(T) + (int)(p.len % T) / p.piece + 3;
    return p;
}

// A B: the number of N tiles with the least time of the busiest CTA (its
// tiles times the tile width, the A operand's share counting as 32 columns)
SkPlan nn_plan(int M, int N) {
    SkPlan best;
    double best_cost = 1e300;
    const int mt = (M + GB_M - 1) / GB_M, n0 = (N + GB_NT - 1) / GB_NT;
    for (int nt = n0; nt < n0 + 4 && 16 * (nt - 1) < N; ++nt) {
        SkPlan p;
        p.tn = tile_cols(N, nt);
        p.fast = nt;
        p.units = (int64_t)mt * nt;
        p.ctas = (int)std::min<int64_t>(sm_count(), p.units);
        const double cost = (double)((p.units + p.ctas - 1) / p.ctas) * (p.tn + 32);
        if (cost < best_cost) {
            best_cost = cost;
            best = p;
        }
    }
    return best;
}

size_t cn_part_bytes(const SkPlan& p) {
    return ((size_t)p.ctas * p.maxseg * p.tn * GB_M * sizeof(float2) + 255) / 256 * 256;
}

// tensor maps over an image: rows of 16 G 64-bit words, one per (chunk, part, plane) ...
bool image_map(CUtensorMap* map, const TcImage& im, int box_words, int box_rows) {
    const uint64_t Q = (im.rows + 7) / 8, G = (im.cols + 7) / 8;
    const uint64_t dims[2] = {16 * G, 4 * Q}, strides[1] = {128 * G};
    const uint32_t box[2] = {(uint32_t)box_words, (uint32_t)box_rows};
    return tensor_map_words(map, im.data, 2, dims, strides, box);
}
// ... or core matrices by (chunk, group, part and plane), for boxes of 16 chunks x 4 groups
bool image_map_mn(CUtensorMap* map, const TcImage& im) {
    const uint64_t Q = (im.rows + 7) / 8, G = (im.cols + 7) / 8;
    const uint64_t dims[4] = {16, Q, G, 4}, strides[3] = {512 * G, 128, 128 * G};
    const uint32_t box[4] = {16, 16, 4, 4};
    return tensor_map_words(map, im.data, 4, dims, strides, box);
}

}  // namespace

// The tensor-core path is the default for shapes it takes; ROKS_TENSOR_CORES=0
// keeps every contraction on the SIMT kernels.
bool tcg_enabled() {
    static int on = -1;
    if (on < 0) {
        const char* e = std::getenv("ROKS_TENSOR_CORES");
        on = (e && e[0] == '0') ? 0 : 1;
    }
    return on == 1;
}

// ROKS_TC_PRESPLIT=0 makes every operand's image at each call (for comparisons)
bool tcg_keep_images() {
    static int on = -1;
    if (on < 0) {
        const char* e = std::getenv("ROKS_TC_PRESPLIT");
        on = (e && e[0] == '0') ? 0 : 1;
    }
    return on == 1;
}

// Where the tensor cores take over from the streamed FP32 kernels.  P (D B) gains
// from 32 columns on (42 x 172 x 34,265 67 us streamed, 44 here; 63 bands, 320
// projectors 68 and 33; 32 bands, 160 projectors, 5600 plane waves 25 and 26).
// P^H Psi splits Psi first, and an MMA costs little less for 32 columns than for
// 64: from 8000 outputs on (9,795 plane waves, 216 x 42 43 us and 34, 144 x 56 46
// and 31), in sums of 20,000 from 6000 on (144 x 48 43 and 43 at 21,823, 82 and 74
// at 52,923); 144 x 36 is 25 and 34 us at 9,795 plane waves, 50 and 54 at 35,033.
// Fewer than 128 rows (the bands against each other) leave an M tile half empty.
bool tcg_cn_takes(int M, int N, int K) {
    return tcg_enabled() && M >= 128 && N >= 32 && K >= 1024 &&
           ((int64_t)M * N >= 8000 || ((int64_t)M * N >= 6000 && K >= 20000));
}
bool tcg_nn_takes(int M, int N, int K) { return tcg_enabled() && M >= 4096 && N >= 32 && K >= 64; }

size_t tcg_image_bytes(int rows, int cols) {
    const size_t Q = (rows + 7) / 8, G = (cols + 7) / 8;
    return 512 * Q * G + (32 * G + 255) / 256 * 256;
}

TcImage tcg_image_at(void* buf, int rows, int cols) {
    TcImage im;
    const size_t Q = (rows + 7) / 8, G = (cols + 7) / 8;
    im.data = buf;
    im.ex = reinterpret_cast<int*>(static_cast<unsigned char*>(buf) + 512 * Q * G);
    im.rows = rows;
    im.cols = cols;
    return im;
}

bool tcg_split(const TcImage& im, const float2* X, int64_t ld, cudaStream_t st) {
    const bool vec = !(ld & 1) && aligned(X, 16);
    return vec ? launch_split<float2, true>(im.rows, im.cols, X, ld, nullptr, im, st)
               : launch_split<float2, false>(im.rows, im.cols, X, ld, nullptr, im, st);
}

void tcg_set_waves(int waves_x2) { g_waves_x2 = waves_x2 >= 1 ? waves_x2 : 2; }

size_t tcg_cn_work_bytes(int M, int N, int K) {
    // the autotuner may take any of its schedules after the buffer is sized
    size_t part = 0;
    for (int w : {2, 5, 8}) part = std::max(part, cn_part_bytes(cn_plan(M, N, K, w)));
    return part + tcg_image_bytes(K, M) + tcg_image_bytes(K, N);
}

size_t tcg_nn_work_bytes(int M, int N, int K) { return tcg_image_bytes(K, N) + tcg_image_bytes(M, K); }

static long long g_tcg_launches = 0;
long long tcg_launches_take() {
    const long long n = g_tcg_launches;
    g_tcg_launches = 0;
    return n;
}

// C = A^H B on the tensor cores; false when the shape, the alignment or the
// work buffer does not allow it (the caller then takes the SIMT kernels).
// ia, ib: images of A and B that the caller has made (else they are made in
// the work buffer; one serves both when A and B are the same block).
bool gemm_cn_tcg(int M, int N, int K, const float2* A, int64_t lda, const float2* B, int64_t ldb, double2* C, int ldc,
                 void* work, size_t work_bytes, const TcImage* ia, const TcImage* ib, cudaStream_t st) {
    if (!tcg_cn_takes(M, N, K) || !work || !aligned(work, 256)) return false;
    const SkPlan sk = cn_plan(M, N, K, g_waves_x2);
    const bool same = A == B && lda == ldb && M == N;
    unsigned char* w = static_cast<unsigned char*>(work);
    size_t need = cn_part_bytes(sk);
    TcImage ma, mb;
    if (ia) ma = *ia;
    else if (same && ib) ma = *ib;
    else {
        ma = tcg_image_at(w + need, K, M);
        need += tcg_image_bytes(K, M);
    }
    if (ib) mb = *ib;
    else if (same) mb = ma;
    else {
        mb = tcg_image_at(w + need, K, N);
        need += tcg_image_bytes(K, N);
    }
    if (need > work_bytes) return false;
    CUtensorMap tmA, tmB;
    if (!image_map(&tmA, ma, 256, 16) || !image_map(&tmB, mb, 2 * sk.tn, 16)) return false;
    if (!ia && !(same && ib) && !tcg_split(ma, A, lda, st)) return false;
    if (!ib && !same && !tcg_split(mb, B, ldb, st)) return false;
    roks::count_launch();
    g_tcg_launches += 1;
    allow_smem(k_tcgemm<false>, GB_SMEM);
    const int T = stages(K);
    float2* part = reinterpret_cast<float2*>(w);
    k_tcgemm<false><<<sk.ctas, GB_THREADS, GB_SMEM, st>>>(M, N, T, sk, tmA, tmB, nullptr, part, nullptr, 0, nullptr, 0,
                                                          1.f, 0.f, wait_polls());
    roks::count_launch();
    const int mt = (M + GB_M - 1) / GB_M;
    // many CTAs per tile: their segments shared out over the warps of a block
    if ((int64_t)T > 8 * sk.len)
        k_tcg_reduce_sk<8><<<dim3((M + 31) / 32, N), 256, 0, st>>>(M, N, mt, T, sk, ma.ex, mb.ex, part, C, ldc);
    else
        k_tcg_reduce_sk<1><<<dim3((M + 31) / 32, (N + 7) / 8), 256, 0, st>>>(M, N, mt, T, sk, ma.ex, mb.ex, part, C,
                                                                           ldc);
    return true;
}

// Cout = alpha A B + beta Cin on the tensor cores (B FP64, small); false when
// not applicable.  Cout may be Cin; it must not overlap A unless ia, an image
// of A that the caller has made, is given.
bool gemm_nn_tcg(int M, int N, int K, const float2* A, int64_t lda, const double2* B, int ldb, const float2* Cin,
                 int64_t ldcin, float2* Cout, int64_t ldc, float alpha, float beta, void* work, size_t work_bytes,
                 const TcImage* ia, cudaStream_t st) {
    if (!tcg_nn_takes(M, N, K) || !work || !aligned(work, 256) || !aligned(Cout, 8)) return false;
    if (beta != 0.f && (!Cin || !aligned(Cin, 8))) return false;
    unsigned char* w = static_cast<unsigned char*>(work);
    size_t need = tcg_image_bytes(K, N);
    const TcImage mb = tcg_image_at(w, K, N);
    TcImage ma;
    if (ia) ma = *ia;
    else {
        ma = tcg_image_at(w + need, M, K);
        need += tcg_image_bytes(M, K);
    }
    if (need > work_bytes) return false;
    const SkPlan sk = nn_plan(M, N);
    CUtensorMap tmA, tmB;
    if (!image_map_mn(&tmA, ma) || !image_map(&tmB, mb, 2 * sk.tn, 16)) return false;
    if (!ia && !tcg_split(ma, A, lda, st)) return false;
    if (!launch_split<double2, false>(K, N, B, ldb, ma.ex, mb, st)) return false;
    roks::count_launch();
    g_tcg_launches += 1;
    allow_smem(k_tcgemm<true>, GB_SMEM);
    k_tcgemm<true><<<sk.ctas, GB_THREADS, GB_SMEM, st>>>(M, N, stages(K), sk, tmA, tmB, mb.ex, nullptr, Cin, ldcin,
                                                         Cout, ldc, alpha, beta, wait_polls());
    return true;
}

// device address of the flag (null if it cannot be had)
int* tcg_timeout_flag() {
    constexpr int kMaxDev = 64;
    static int* addr[kMaxDev] = {nullptr};
    int dev = 0;
    void* p = nullptr;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev ||
        (!addr[dev] && cudaGetSymbolAddress(&p, g_tcg_timeout) != cudaSuccess)) {
        cudaGetLastError();
        return nullptr;
    }
    if (!addr[dev]) addr[dev] = static_cast<int*>(p);
    return addr[dev];
}

int tcg_timeout_take() {
    int h = 0;
    if (cudaMemcpyFromSymbol(&h, g_tcg_timeout, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (h) {
        const int z = 0;
        cudaMemcpyToSymbol(g_tcg_timeout, &z, sizeof(int));
    }
    return h;
}

}  // namespace roks
