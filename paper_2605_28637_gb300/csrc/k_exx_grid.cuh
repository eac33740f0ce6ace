// k_exx_grid.cuh -- the grid work of the exact exchange, with the pointwise
// steps fused into the transform passes, on a grid of its own:
//
//   x pass, forward : rho_jn = conj(psi_j) psi_n formed while the x lines load
//   plane pass      : per x plane, in one stay in shared memory, y and z
//                     forward, times v(G) / M^3 (and the partial sums of the
//                     pair integrals), z and y inverse
//   x pass, inverse : plain (W_jn)
//   accumulation    : X_n += c(n, j) psi_j W_jn and X_j += c(j, n) psi_n
//                     conj(W_jn) over a tile of bands j x bands n, one thread
//                     per grid point
//
// The grid.  Pair densities hold frequencies up to 2 nmax, and of psi_j W_jn
// (up to 3 nmax) only those up to nmax are wanted: M >= 4 nmax + 1 points per
// side give both without aliasing, like any larger grid.  So the orbitals
// are transformed to the smallest compiled M of that kind (54 instead of 72
// for hybrid-72, 0.42 of the points), and the fields transformed back there
// and added to F|n> as coefficients.
//
// What bounds it: instruction issue in the plane pass, L2 and what spills of
// it in the others.  A batch is as many tiles of 8 x 8 bands as fit 96 MB (one
// at M = 54); a tile of 64 pairs of hybrid-72 takes 26 + 58 + 24 + 32 us in the four
// kernels, 18.8 ms an apply with its 8256 pairs.  On the density's grid, with
// y and z passes of their own and the accumulation over the list of pairs
// (a field read and written for every pair), it was 103 ms.
#pragma once

#include "k_fft_impl.cuh"
#include "roks_exx.cuh"

namespace roks {

// the compiled lengths: all of two passes (the plane pass is built on that)
#define ROKS_EXX_DISPATCH(M_, CALL)                          \
    switch (M_) {                                            \
        case 16: { constexpr int MM = 16; CALL; } break;     \
        case 24: { constexpr int MM = 24; CALL; } break;     \
        case 32: { constexpr int MM = 32; CALL; } break;     \
        case 40: { constexpr int MM = 40; CALL; } break;     \
        case 48: { constexpr int MM = 48; CALL; } break;     \
        case 54: { constexpr int MM = 54; CALL; } break;     \
        case 60: { constexpr int MM = 60; CALL; } break;     \
        case 64: { constexpr int MM = 64; CALL; } break;     \
        case 72: { constexpr int MM = 72; CALL; } break;     \
        case 80: { constexpr int MM = 80; CALL; } break;     \
        case 96: { constexpr int MM = 96; CALL; } break;     \
        case 108: { constexpr int MM = 108; CALL; } break;   \
        case 120: { constexpr int MM = 120; CALL; } break;   \
        default: break;                                      \
    }

// Threads of the passes: with 54 = 9 x 6, tiles of 64 lines hold 384 and 576
// butterflies, two and three rounds of 192 threads (an apply of 40 bands 2.10 ms,
// with 256 threads 2.14).  Elsewhere 256 against 192, the same apply: 32 0.56 and
// 0.57, 72 4.39 and 4.59, 80 6.01 and 6.57, 96 (24 bands) 5.15 and 5.33; 192 would
// be the better at 16, 24, 48, 60 and 64 by 1 to 4% and at 108 by 13%.
__host__ __device__ constexpr int exx_threads(int m) { return m == 54 ? 192 : kThreads; }
// lines of an x tile (consecutive y, z)
__host__ __device__ constexpr int exx_lines(int m, size_t elem) { return m <= 80 && elem == 8 ? 64 : 32; }

template <typename T, int M>
__global__ void __launch_bounds__(exx_threads(M)) k_exx_x_fwd(const c2<T>* __restrict__ tw,
                                                              const c2<T>* __restrict__ Phi,
                                                              const int* __restrict__ pj,
                                                              const int* __restrict__ pn, int p0,
                                                              c2<T>* __restrict__ buf) {
    using V = c2<T>;
    constexpr int TL = exx_lines(M, sizeof(V)), NT = exx_threads(M), MM = M * M;
    constexpr int64_t M3 = (int64_t)M * MM;
    extern __shared__ __align__(16) unsigned char smem[];
    V* bs = reinterpret_cast<V*>(smem);
    V* tws = bs + M * TL;
    load_twiddles<V, M>(tws, tw);
    const int l0 = blockIdx.x * TL, b = blockIdx.y;
    const V* Pj = Phi + (int64_t)pj[p0 + b] * M3 + l0;
    const V* Pn = Phi + (int64_t)pn[p0 + b] * M3 + l0;
    V* out = buf + (int64_t)b * M3 + l0;
    // (the first pass takes no twiddles; their store is ordered by its barrier)
    fft_io<V, M, -1, TL, TL, NT, false, false>(
        bs, tws,
        [&](int line, int e) {
            if (l0 + line >= MM) return mk<T>(T(0), T(0));
            return cmulc(Pj[e * MM + line], Pn[e * MM + line]);
        },
        [&](int line, int e, V v, int, int) {
            if (l0 + line < MM) out[e * MM + line] = v;
        });
}

template <typename T, int M>
__global__ void __launch_bounds__(exx_threads(M)) k_exx_x_inv(const c2<T>* __restrict__ tw, c2<T>* __restrict__ buf) {
    using V = c2<T>;
    constexpr int TL = exx_lines(M, sizeof(V)), NT = exx_threads(M), MM = M * M;
    extern __shared__ __align__(16) unsigned char smem[];
    V* bs = reinterpret_cast<V*>(smem);
    V* tws = bs + M * TL;
    load_twiddles<V, M>(tws, tw);
    const int l0 = blockIdx.x * TL;
    V* d = buf + (int64_t)blockIdx.y * M * MM + l0;
    fft_io<V, M, +1, TL, TL, NT, false, false>(
        bs, tws, [&](int line, int e) { return l0 + line < MM ? d[e * MM + line] : mk<T>(T(0), T(0)); },
        [&](int line, int e, V v, int, int) {
            if (l0 + line < MM) d[e * MM + line] = v;
        });
}

// Plane x = blockIdx.x of pair blockIdx.y.  Rows of the plane (y) lie M + 1
// apart, so that lines along either axis meet no bank twice.  The z
// transforms join in registers: the last pass of a two-pass plan R0 x R1
// leaves a thread the elements j + r R0 in place, which is what the first pass
// of the inverse plan R1 x R0 reads.  v(G) depends on |G| alone, so element
// (x, z, y) serves for (x, y, z) and the threads, whose lines run along y,
// read it in order.  The block's sum of v |rho(G)|^2 goes to
// part[pair * M + x].
template <typename T, int M>
__global__ void __launch_bounds__(exx_threads(M)) k_exx_plane(const c2<T>* __restrict__ tw, const T* __restrict__ vG,
                                                              c2<T>* __restrict__ buf, double* __restrict__ part) {
    using V = c2<T>;
    constexpr int NT = exx_threads(M), PZ = M + 1, R0 = plan_radix(M, 0), R1 = plan_radix(M, 1);
    static_assert(plan_passes(M) == 2 && R0 * R1 == M, "the plane pass joins two-pass plans");
    extern __shared__ __align__(16) unsigned char smem[];
    V* pl = reinterpret_cast<V*>(smem);
    V* tws = pl + M * PZ;
    __shared__ double red[NT / 32];
    load_twiddles<V, M>(tws, tw);
    const int x = blockIdx.x, tid = threadIdx.x;
    V* d = buf + ((int64_t)blockIdx.y * M + x) * M * M;
    auto yl = [&](int line, int e) { return pl[e * PZ + line]; };
    auto ys = [&](int line, int e, V v, int, int) { pl[e * PZ + line] = v; };
    auto zl = [&](int line, int e) { return pl[line * PZ + e]; };
    auto zs = [&](int line, int e, V v, int, int) { pl[line * PZ + e] = v; };
    pass_io<V, M, 0, -1, M, NT, false>(tws, [&](int line, int e) { return d[e * M + line]; }, ys);
    __syncthreads();
    pass_io<V, M, 1, -1, M, NT, false>(tws, yl, ys);   // in place, element by element
    __syncthreads();
    pass_io<V, M, 0, -1, M, NT, true>(tws, zl, zs);
    __syncthreads();
    T acc = T(0);
    {
        constexpr int TOT = R0 * M, PER = (TOT + NT - 1) / NT;
        V v[PER][R1];
        const T* vg = vG + (int64_t)x * M * M;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int beta = tid + q * NT;
            if (beta < TOT) {
                const int line = beta % M, j = beta / M;
#pragma unroll
                for (int r = 0; r < R1; ++r) v[q][r] = pl[line * PZ + j + r * R0];
                twiddle_dft<V, M, R1, R0, -1>(v[q], tws, j);
#pragma unroll
                for (int r = 0; r < R1; ++r) {
                    const T w = vg[(j + r * R0) * M + line];
                    const V u = v[q][r];
                    acc += w * (u.x * u.x + u.y * u.y);
                    v[q][r] = mk<T>(u.x * w, u.y * w);
                }
                twiddle_dft<V, M, R1, 1, +1>(v[q], tws, j);
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int beta = tid + q * NT;
            if (beta < TOT) {
                const int line = beta % M, j = beta / M;
#pragma unroll
                for (int r = 0; r < R1; ++r) pl[line * PZ + j * R1 + r] = v[q][r];
            }
        }
    }
    __syncthreads();
    {
        constexpr int TOT = R1 * M, PER = (TOT + NT - 1) / NT;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int beta = tid + q * NT;
            if (beta < TOT) {
                const int line = beta % M, j = beta / M;
                V v[R0];
#pragma unroll
                for (int r = 0; r < R0; ++r) v[r] = pl[line * PZ + j + r * R1];
                twiddle_dft<V, M, R0, R1, +1>(v, tws, j);
#pragma unroll
                for (int r = 0; r < R0; ++r) pl[line * PZ + j + r * R1] = v[r];
            }
        }
    }
    __syncthreads();
    pass_io<V, M, 0, +1, M, NT, true>(tws, yl, ys);
    __syncthreads();
    pass_io<V, M, 1, +1, M, NT, false>(tws, yl, [&](int line, int e, V v, int, int) { d[e * M + line] = v; });
    double s = double(acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((tid & 31) == 0) red[tid >> 5] = s;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int k = 0; k < NT / 32; ++k) t += red[k];
        part[(int64_t)blockIdx.y * M + x] = t;
    }
}

// The z part of the plane pass alone, for planes beyond the shared memory
// (FP64, M = 120), between y passes of their own: forward transform, times
// v(G) / M^3, inverse transform of the lines of plane x = blockIdx.x.
template <typename T, int N>
__global__ void __launch_bounds__(kThreads) k_exx_z_mult(const c2<T>* __restrict__ tw, const T* __restrict__ vG,
                                                         c2<T>* __restrict__ buf, double* __restrict__ part) {
    using V = c2<T>;
    constexpr int TL = tile_lines(N), LS = TL + 1;
    extern __shared__ __align__(16) unsigned char smem[];
    V* bs = reinterpret_cast<V*>(smem);
    V* tws = bs + N * LS;
    __shared__ double red[kThreads];
    load_twiddles<V, N>(tws, tw);
    const int b = blockIdx.y;
    V* d = buf + ((int64_t)b * N + blockIdx.x) * N * N;
    const T* vg = vG + (int64_t)blockIdx.x * N * N;
    T acc = T(0);
    for (int l0 = 0; l0 < N; l0 += TL) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < TL * N; idx += kThreads) {
            const int line = idx / N, e = idx - line * N;
            const int l = l0 + line;
            bs[e * LS + line] = l < N ? d[l * N + e] : mk<T>(T(0), T(0));
        }
        __syncthreads();
        tile_fft<V, N, -1, TL, LS, kThreads>(bs, tws);
        for (int idx = threadIdx.x; idx < TL * N; idx += kThreads) {
            const int line = idx / N, e = idx - line * N;
            const int l = l0 + line;
            const T w = l < N ? vg[l * N + e] : T(0);
            const V v = bs[e * LS + line];
            acc += w * (v.x * v.x + v.y * v.y);
            bs[e * LS + line] = mk<T>(v.x * w, v.y * w);
        }
        __syncthreads();
        tile_fft<V, N, +1, TL, LS, kThreads>(bs, tws);
        for (int idx = threadIdx.x; idx < TL * N; idx += kThreads) {
            const int line = idx / N, e = idx - line * N;
            const int l = l0 + line;
            if (l < N) d[l * N + e] = bs[e * LS + line];
        }
    }
    red[threadIdx.x] = double(acc);
    __syncthreads();
    for (int s = kThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(int64_t)b * N + blockIdx.x] = red[0];
}

// Exchange fields of the batch's tiles, one after the other: bands j0 .. j0 +
// bj - 1 (held in registers, as are their fields' sums) against n0 .. n0 + bn -
// 1, one thread per grid point, pairs in the list's order (n, then j; j <= n on
// the diagonal).  Bound
// by the latency of the loads: a thread has two bands n on their way to its
// own slots of shared memory (W of up to 8 pairs, psi_n and X_n each), so no
// thread waits for another.  288 threads at up to 56 registers (FP32): four
// blocks an SM, and all points of M = 54 in one wave: 32 us a tile of 64 pairs
// (loads into registers, 256 threads at 72, coefficients in FP64: 67).  An apply
// of 40 bands with 288 and with 256 threads: M = 54 2.10 ms and 2.14; 16 to 48 1 to
// 2% longer, 60 to 72 1%, from 80 on the same.
constexpr int kExxAccThreads = 288;
template <typename T> constexpr size_t exx_acc_smem() {
    return sizeof(c2<T>) * 2 * (kExxTileMax + 2) * kExxAccThreads;
}
// c[k][k'] of the classes in the element type (conversions from FP64 for every
// pair took longer than the loads)
template <typename T> struct ExxPairCoef { T c[3][3]; };
template <typename V>
__device__ __forceinline__ void exx_async(V* dst, const V* src) {
    // (memory: the slot's earlier values are read, and X written, before the copy is issued)
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(sizeof(V))
                 : "memory");
}
template <typename T>
__global__ void __launch_bounds__(kExxAccThreads, sizeof(T) == 4 ? 4 : 2)
    k_exx_accumulate(int64_t M3, const c2<T>* __restrict__ Phi, const c2<T>* __restrict__ W,
                     const ExxTile* __restrict__ tiles, int ntiles, int n_closed, ExxPairCoef<T> cf,
                     c2<T>* __restrict__ X) {
    constexpr int B = kExxTileMax, NT = kExxAccThreads;
    using V = c2<T>;
    extern __shared__ __align__(16) unsigned char smem[];
    V* ring = reinterpret_cast<V*>(smem) + threadIdx.x;
    const int64_t p = (int64_t)blockIdx.x * NT + threadIdx.x;
    if (p >= M3) return;
    W += p;
    for (int t = 0; t < ntiles; ++t) {
        const int j0 = tiles[t].j0, bj = tiles[t].bj, n0 = tiles[t].n0, bn = tiles[t].bn;
        const bool diag = j0 == n0;
        auto fetch = [&](int n) {
            V* s = ring + (n & 1) * (B + 2) * NT;
            if (n < bn) {
                const int nj = diag ? n + 1 : bj;
                for (int j = 0; j < nj; ++j) exx_async(s + j * NT, W + j * M3);
                W += nj * M3;
                exx_async(s + B * NT, Phi + (n0 + n) * M3 + p);
                exx_async(s + (B + 1) * NT, const_cast<const V*>(X) + (n0 + n) * M3 + p);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(0);
        fetch(1);
        V pj[B], xj[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
            xj[j] = mk<T>(T(0), T(0));
            pj[j] = j < bj ? Phi[(j0 + j) * M3 + p] : xj[j];
        }
        for (int n = 0; n < bn; ++n) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            const V* s = ring + (n & 1) * (B + 2) * NT;
            const V pn = s[B * NT];
            const int nj = diag ? n + 1 : bj;
            const int kn = max(0, n0 + n - n_closed + 1);
            V a = s[(B + 1) * NT];
#pragma unroll
            for (int j = 0; j < B; ++j) {
                if (j < nj) {
                    const V w = s[j * NT];
                    const int kj = max(0, j0 + j - n_closed + 1);
                    const T cnj = cf.c[kn][kj], cjn = cf.c[kj][kn];
                    const V u = cmul(pj[j], w);
                    a.x += cnj * u.x;
                    a.y += cnj * u.y;
                    if (!diag || j < n) {
                        // psi_n conj(W)
                        xj[j].x += cjn * (pn.x * w.x + pn.y * w.y);
                        xj[j].y += cjn * (pn.y * w.x - pn.x * w.y);
                    }
                }
            }
            X[(n0 + n) * M3 + p] = a;
            fetch(n + 2);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
        for (int j = 0; j < B; ++j) {
            if (j < bj) {
                const V o = X[(j0 + j) * M3 + p];
                X[(j0 + j) * M3 + p] = mk<T>(o.x + xj[j].x, o.y + xj[j].y);
            }
        }
        __threadfence_block();   // the next tile's asynchronous reads of X come after
    }
}

// Forward x transform of the exchange fields, planes of the sphere kept:
// Yp[b] (np x M^2) = scale * sum_x e^{-i G x} X_b.
template <typename T, int M>
__global__ void __launch_bounds__(exx_threads(M)) k_exx_field_x(int nmax, const c2<T>* __restrict__ tw,
                                                                const c2<T>* __restrict__ X, c2<T>* __restrict__ Yp,
                                                                T scale) {
    using V = c2<T>;
    constexpr int TL = exx_lines(M, sizeof(V)), NT = exx_threads(M), MM = M * M;
    extern __shared__ __align__(16) unsigned char smem[];
    V* bs = reinterpret_cast<V*>(smem);
    V* tws = bs + M * TL;
    load_twiddles<V, M>(tws, tw);
    const int l0 = blockIdx.x * TL;
    const V* in = X + (int64_t)blockIdx.y * M * MM + l0;
    V* out = Yp + (int64_t)blockIdx.y * (2 * nmax + 1) * MM + l0;
    fft_io<V, M, -1, TL, TL, NT, false, false>(
        bs, tws, [&](int line, int e) { return l0 + line < MM ? in[e * MM + line] : mk<T>(T(0), T(0)); },
        [&](int line, int e, V v, int, int) {
            const int i = signed_freq(e, M);
            if (l0 + line < MM && i >= -nmax && i <= nmax) out[(i + nmax) * MM + line] = mk<T>(v.x * scale, v.y * scale);
        });
}

template <typename T, int M>
struct ExxGrid {
    using V = c2<T>;
    static constexpr int TL = exx_lines(M, sizeof(V)), NT = exx_threads(M);
    static constexpr size_t SMX = sizeof(V) * (size_t)(M * TL + M);
    static constexpr size_t SMP = sizeof(V) * (size_t)(M * (M + 1) + M);
    static constexpr bool PLANE = SMP <= 220 * 1024;
    static void batch(const ExxArgs<T>& a, int t0, int t1, bool want_field, cudaStream_t st) {
        const int p0 = a.tiles[t0].p0, np = a.tiles[t1 - 1].p0 + a.tiles[t1 - 1].np - p0;
        const int64_t M3 = (int64_t)M * M * M;
        const dim3 gx((M * M + TL - 1) / TL, np);
        double* part = a.part + (int64_t)p0 * M;
        set_smem(k_exx_x_fwd<T, M>, SMX);
        roks::count_launch(), k_exx_x_fwd<T, M><<<gx, NT, SMX, st>>>(a.tw, a.Phi, a.pj, a.pn, p0, a.buf);
        if constexpr (PLANE) {
            set_smem(k_exx_plane<T, M>, SMP);
            roks::count_launch(), k_exx_plane<T, M><<<dim3(M, np), NT, SMP, st>>>(a.tw, a.vG, a.buf, part);
        } else {
            constexpr int TY = tile_lines(M);
            constexpr size_t SM = tile_smem_bytes<V, M, TY + 1>();
            const dim3 gy((M + TY - 1) / TY, M, np);
            set_smem(k_grid_fft_strided<T, M>, SM);
            set_smem(k_exx_z_mult<T, M>, SM);
            roks::count_launch(),
                k_grid_fft_strided<T, M><<<gy, kThreads, SM, st>>>(a.tw, a.buf, (int64_t)M * M, (int64_t)M, -1, M3);
            roks::count_launch(), k_exx_z_mult<T, M><<<dim3(M, np), kThreads, SM, st>>>(a.tw, a.vG, a.buf, part);
            if (want_field)
                roks::count_launch(), k_grid_fft_strided<T, M><<<gy, kThreads, SM, st>>>(
                                          a.tw, a.buf, (int64_t)M * M, (int64_t)M, +1, M3);
        }
        if (!want_field) return;
        set_smem(k_exx_x_inv<T, M>, SMX);
        roks::count_launch(), k_exx_x_inv<T, M><<<gx, NT, SMX, st>>>(a.tw, a.buf);
        ExxPairCoef<T> c;
        for (int k = 0; k < 9; ++k) c.c[k / 3][k % 3] = T(a.cf.c[k / 3][k % 3]);
        set_smem(k_exx_accumulate<T>, exx_acc_smem<T>());
        roks::count_launch(), k_exx_accumulate<T>
            <<<(unsigned)((M3 + kExxAccThreads - 1) / kExxAccThreads), kExxAccThreads, exx_acc_smem<T>(), st>>>(
                M3, a.Phi, a.buf, a.d_tiles + t0, t1 - t0, a.cf.n_closed, c, a.X);
    }
    static void orbitals(const Sphere& s, const V* tw, const V* psi, int64_t ld, int nb, V* Zc, V* Yp, V* Phi, T scale,
                         cudaStream_t st) {
        using F = BandFft<T, M>;
        if (psi) {
            F::z_inv(s, tw, psi, ld, 0, nb, Zc, st);
            F::y_inv(s, tw, Zc, Yp, nb, st);
        }
        F::x_inv_full(s, tw, Yp, Phi, 0, nb, scale, st);
    }
    static void add_fields(const Sphere& s, const V* tw, const V* X, int nb, V* Yp, V* Zc, V* out, int64_t ldo,
                           T scale, cudaStream_t st) {
        using F = BandFft<T, M>;
        set_smem(k_exx_field_x<T, M>, SMX);
        roks::count_launch(), k_exx_field_x<T, M><<<dim3((M * M + TL - 1) / TL, nb), NT, SMX, st>>>(s.nmax, tw, X, Yp,
                                                                                                   scale);
        F::y_fwd(s, tw, Yp, Zc, nb, st);
        F::z_fwd_add(s, tw, Zc, out, ldo, nb, st);
    }
};

template <typename T>
void exx_batch_grid(const ExxArgs<T>& a, int t0, int t1, bool want_field, cudaStream_t st) {
    ROKS_EXX_DISPATCH(a.M, (ExxGrid<T, MM>::batch(a, t0, t1, want_field, st)));
}
template <typename T>
void exx_orbitals(const Sphere& s, const c2<T>* tw, const c2<T>* psi, int64_t ld, int nb, c2<T>* Zc, c2<T>* Yp,
                  c2<T>* Phi, T scale, cudaStream_t st) {
    ROKS_EXX_DISPATCH(s.N, (ExxGrid<T, MM>::orbitals(s, tw, psi, ld, nb, Zc, Yp, Phi, scale, st)));
}
template <typename T>
void exx_add_fields(const Sphere& s, const c2<T>* tw, const c2<T>* X, int nb, c2<T>* Yp, c2<T>* Zc, c2<T>* out,
                    int64_t ldo, T scale, cudaStream_t st) {
    ROKS_EXX_DISPATCH(s.N, (ExxGrid<T, MM>::add_fields(s, tw, X, nb, Yp, Zc, out, ldo, scale, st)));
}

#define ROKS_INSTANTIATE_EXX(T)                                                                                    \
    template void exx_batch_grid<T>(const ExxArgs<T>&, int, int, bool, cudaStream_t);                              \
    template void exx_orbitals<T>(const Sphere&, const c2<T>*, const c2<T>*, int64_t, int, c2<T>*, c2<T>*, c2<T>*, \
                                  T, cudaStream_t);                                                                \
    template void exx_add_fields<T>(const Sphere&, const c2<T>*, const c2<T>*, int, c2<T>*, c2<T>*, c2<T>*,       \
                                    int64_t, T, cudaStream_t);

}  // namespace roks
