// k_pot_impl.cuh -- the class potentials of a density in three passes over
// the grid.  Included by one translation unit per precision.
//
//   x pass, forward : channel densities, Slater exchange (fields and energies)
//                     and V_loc rho formed while the x lines of the total
//                     density fill the tile, then their transform
//   plane pass      : y and z forward, 4 pi / G^2 and the Hartree energy, z
//                     and y inverse, each x plane in one stay in shared memory
//   x pass, inverse : the Hartree potential's lines, the class potentials
//                     V^k = w_k (V_loc + V_H) + xc^k, <o|V^c|o> and max |V^k|
//                     from the tile
//
// Bound by the launches (four with the sums, 14 when every pointwise step and
// transform direction was its own) and, from 96^3 on, by the 100 bytes a point
// that move: organic-96 mixed 85 -> 49 us, mgo-120 135 -> 74, 16^3 in FP64 81 ->
// 39, 48^3 144 -> 127.
#pragma once

#include "k_fft_impl.cuh"
#include "roks_grid.cuh"

namespace roks {

// lines of a tile: few on the small grids, so that there are blocks for the SMs
__host__ __device__ constexpr int pot_lines(int n) { return n <= 48 ? n / 4 : tile_lines(n); }

// Block sum of per-thread values in FP64, valid in thread 0; FP32: two-sums
// within a warp, FP64 across warps (conversions and FP64 additions are slow).
template <typename T, int NT>
__device__ __forceinline__ double block_total(T v, double* sh) {
    double w;
    if constexpr (sizeof(T) == 8) {
        w = v;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    } else {
        float s = v, c = 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float so = __shfl_xor_sync(0xffffffffu, s, o), co = __shfl_xor_sync(0xffffffffu, c, o);
            const float t = s + so, bp = t - s;
            c = c + co + ((s - (t - bp)) + (so - bp));
            s = t;
        }
        w = double(s) + double(c);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = w;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < NT / 32; ++k) r += sh[k];
    return r;
}

template <typename T, int N>
__global__ void __launch_bounds__(kThreads) k_pot_x_fwd(const c2<T>* __restrict__ tw,
                                                        const typename DensAcc<T>::S* __restrict__ rho3,
                                                        const T* __restrict__ vloc, PotCoefT<T> cf, T c6, T cx,
                                                        c2<T>* __restrict__ grid, T* __restrict__ xc3,
                                                        double* __restrict__ part) {
    // pointwise arithmetic in the element type T (constants come from the
    // host: FP64 arithmetic per thread is slow on this part); per-thread
    // partial energies in T over a few points, block and grid sums in FP64
    using V = c2<T>;
    using DA = DensAcc<T>;
    constexpr int TL = pot_lines(N), LS = TL + 1, NN = N * N, N3 = N * NN;
    extern __shared__ __align__(16) unsigned char smem[];
    V* buf = reinterpret_cast<V*>(smem);
    V* tws = buf + N * LS;
    __shared__ double sh[kThreads / 32];
    load_twiddles<V, N>(tws, tw);
    const int z0 = blockIdx.x * TL, y = blockIdx.y;
    T exM = 0, exT = 0, eloc = 0;
    for (int idx = threadIdx.x; idx < TL * N; idx += kThreads) {
        const int e = idx / TL, line = idx - e * TL, p = e * NN + y * N + z0 + line;
        T rho_tot = 0;
        if (z0 + line < N) {
            const T rk[3] = {T(DA::value(rho3[p])), T(DA::value(rho3[N3 + p])), T(DA::value(rho3[2 * N3 + p]))};
            T v[4];
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
                T r = 0;
#pragma unroll
                for (int k = 0; k < 3; ++k) r += cf.f[k][ch] * rk[k];
                r = r > T(0) ? r : T(0);
                const T c = cbrt(r);
                v[ch] = -cf.xscale * c6 * c;
                const T ex = -cf.xscale * cx * c * r;
                if (ch < 2) {
                    exM += ex;
                    rho_tot += r;
                } else {
                    exT += ex;
                }
            }
            eloc += vloc[p] * rho_tot;
            if (xc3) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    T s = 0;
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) s += cf.C[k][ch] * v[ch];
                    xc3[k * N3 + p] = s;
                }
            }
        }
        buf[e * LS + line] = mk<T>(rho_tot, T(0));
    }
    __syncthreads();
    V* out = grid + y * N + z0;
    fft_io<V, N, -1, TL, LS, kThreads, true, false>(
        buf, tws, [&](int line, int e) { return buf[e * LS + line]; },
        [&](int line, int e, V v, int, int) {
            if (z0 + line < N) out[e * NN + line] = v;
        });
    const double a = block_total<T, kThreads>(exM, sh), b = block_total<T, kThreads>(exT, sh),
                 c = block_total<T, kThreads>(eloc, sh);
    if (threadIdx.x == 0) {
        double* o = part + 4 * (blockIdx.y * gridDim.x + blockIdx.x);
        o[0] = a;
        o[1] = b;
        o[2] = c;
    }
}

// vmax: the largest |V^k| of each class, zeroed before (null: not wanted)
template <typename T, int N>
__global__ void __launch_bounds__(kThreads) k_pot_x_class(const c2<T>* __restrict__ tw, const c2<T>* __restrict__ grid,
                                                          const T* __restrict__ vloc, const T* __restrict__ xc3,
                                                          const typename DensAcc<T>::S* __restrict__ rho3, T w0, T w1,
                                                          T w2, T* __restrict__ Vk, double* __restrict__ part,
                                                          float* __restrict__ vmax) {
    using V = c2<T>;
    using DA = DensAcc<T>;
    constexpr int TL = pot_lines(N), LS = TL + 1, NN = N * N, N3 = N * NN;
    extern __shared__ __align__(16) unsigned char smem[];
    V* buf = reinterpret_cast<V*>(smem);
    V* tws = buf + N * LS;
    __shared__ double sh[kThreads / 32];
    __shared__ int vm[3];
    load_twiddles<V, N>(tws, tw);
    if (threadIdx.x < 3) vm[threadIdx.x] = 0;
    const int z0 = blockIdx.x * TL, y = blockIdx.y;
    const V* in = grid + y * N + z0;
    fft_io<V, N, +1, TL, LS, kThreads, false, true>(
        buf, tws, [&](int line, int e) { return z0 + line < N ? in[e * NN + line] : mk<T>(T(0), T(0)); },
        [&](int line, int e, V v, int, int) { buf[e * LS + line] = v; });
    __syncthreads();
    T ea = 0, eb = 0;
    float mc = 0.f, ma = 0.f, mb = 0.f;
    for (int idx = threadIdx.x; idx < TL * N; idx += kThreads) {
        const int e = idx / TL, line = idx - e * TL, p = e * NN + y * N + z0 + line;
        if (z0 + line >= N) continue;
        const T v0 = vloc[p] + buf[e * LS + line].x;
        const T vc = w0 * v0 + xc3[p], va = w1 * v0 + xc3[N3 + p], vb = w2 * v0 + xc3[2 * N3 + p];
        Vk[p] = vc;
        Vk[N3 + p] = va;
        Vk[2 * N3 + p] = vb;
        if (vmax) {
            mc = fmaxf(mc, fabsf(float(vc)));
            ma = fmaxf(ma, fabsf(float(va)));
            mb = fmaxf(mb, fabsf(float(vb)));
        }
        ea += vc * T(DA::value(rho3[N3 + p]));
        eb += vc * T(DA::value(rho3[2 * N3 + p]));
    }
    if (vmax) {
        // floats >= 0 order like their bits
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, o));
            ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
            mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        }
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&vm[0], __float_as_int(mc));
            atomicMax(&vm[1], __float_as_int(ma));
            atomicMax(&vm[2], __float_as_int(mb));
        }
    }
    const double a = block_total<T, kThreads>(ea, sh), b = block_total<T, kThreads>(eb, sh);
    if (vmax && threadIdx.x < 3) atomicMax(reinterpret_cast<int*>(vmax) + threadIdx.x, vm[threadIdx.x]);
    if (threadIdx.x == 0) {
        double* o = part + 2 * (blockIdx.y * gridDim.x + blockIdx.x);
        o[0] = a;
        o[1] = b;
    }
}

// The pointwise Hartree step alone, where the plane pass is not taken (FP64
// beyond 32): grid = 4 pi / G^2 grid / N^3, and the energy's partials.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_hartree_G(int N, T inv, T fpb, c2<T>* __restrict__ grid,
                                                        double* __restrict__ part) {
    __shared__ double sh[kThreads / 32];
    const int N3 = N * N * N;
    T eh = 0;
    for (int p = blockIdx.x * kThreads + threadIdx.x; p < N3; p += gridDim.x * kThreads) {
        const int z = p % N, y = (p / N) % N, x = p / (N * N);
        const int fx = signed_freq(x, N), fy = signed_freq(y, N), fz = signed_freq(z, N);
        grid[p] = hartree_point<T>(grid[p], fx * fx + fy * fy + fz * fz, inv, fpb, eh);
    }
    const double deh = block_total<T, kThreads>(eh, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = deh;
}

template <typename T, int N>
struct PotGrid {
    using V = c2<T>;
    using F = BandFft<T, N>;
    static constexpr int TL = pot_lines(N), TILES = (N + TL - 1) / TL;
    static constexpr size_t SM = tile_smem_bytes<V, N, TL + 1>();
    static int x_fwd(const PotArgs<T>& a, bool fields, cudaStream_t st) {
        set_smem(k_pot_x_fwd<T, N>, SM);
        roks::count_launch(), k_pot_x_fwd<T, N><<<dim3(TILES, N), kThreads, SM, st>>>(
                                  a.tw, a.rho3, a.vloc, a.ct, a.c6, a.cx, a.grid, fields ? a.xc3 : nullptr, a.partA);
        return TILES * N;
    }
    static int hartree(const PotArgs<T>& a, bool x_done, cudaStream_t st) {
        if (!x_done) F::grid_x(a.tw, a.grid, -1, 1, 0, st);
        if constexpr (F::PLANE) {
            set_smem(k_grid_plane<T, N, 0>, F::SMP);
            roks::count_launch(), k_grid_plane<T, N, 0><<<N, plane_threads(N), F::SMP, st>>>(
                                      a.tw, a.grid, 0, a.inv, a.fpb, a.partB, a.vmax);
            return N;
        } else {
            const int blocks = 512;
            F::grid_yz(a.tw, a.grid, -1, 1, 0, st);
            roks::count_launch(), k_hartree_G<T><<<blocks, kThreads, 0, st>>>(N, a.inv, a.fpb, a.grid, a.partB);
            F::grid_yz(a.tw, a.grid, +1, 1, 0, st);
            if (a.vmax) cudaMemsetAsync(a.vmax, 0, 3 * sizeof(float), st);
            return blocks;
        }
    }
    static int x_class(const PotArgs<T>& a, cudaStream_t st) {
        set_smem(k_pot_x_class<T, N>, SM);
        roks::count_launch(), k_pot_x_class<T, N><<<dim3(TILES, N), kThreads, SM, st>>>(
                                  a.tw, a.grid, a.vloc, a.xc3, a.rho3, a.w[0], a.w[1], a.w[2], a.Vk, a.partC, a.vmax);
        return TILES * N;
    }
};

template <typename T>
int pot_x_fwd(const PotArgs<T>& a, bool fields, cudaStream_t st) {
    int n = 0;
    ROKS_GRID_DISPATCH(a.N, (n = PotGrid<T, NN>::x_fwd(a, fields, st)));
    return n;
}
template <typename T>
int pot_hartree(const PotArgs<T>& a, bool x_done, cudaStream_t st) {
    int n = 0;
    ROKS_GRID_DISPATCH(a.N, (n = PotGrid<T, NN>::hartree(a, x_done, st)));
    return n;
}
template <typename T>
int pot_x_class(const PotArgs<T>& a, cudaStream_t st) {
    int n = 0;
    ROKS_GRID_DISPATCH(a.N, (n = PotGrid<T, NN>::x_class(a, st)));
    return n;
}

#define ROKS_INSTANTIATE_POT(T)                                          \
    template int pot_x_fwd<T>(const PotArgs<T>&, bool, cudaStream_t);    \
    template int pot_hartree<T>(const PotArgs<T>&, bool, cudaStream_t);  \
    template int pot_x_class<T>(const PotArgs<T>&, cudaStream_t);

}  // namespace roks
