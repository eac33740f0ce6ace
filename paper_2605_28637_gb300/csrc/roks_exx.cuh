// roks_exx.cuh -- exact-exchange launch arguments (internal).
#pragma once

#include <vector>

#include "roks_impl.cuh"

namespace roks {

// Coefficients derived from the occupations: c[k][k'] = -alpha Omega^{1/2}
// w(k, k') for the exchange field, fM/fT[k][k'] = sum over the spins of a
// configuration of f_k f_k', wxc[k'] = w(closed, k').
struct ExxCoef {
    double c[3][3];
    double fM[3][3];
    double fT[3][3];
    double wxc[3];
    double alpha;
    int n_closed;
};

// Points per side of the exchange's grid: the smallest compiled length that
// holds spheres of nmax without aliasing (4 nmax + 1 <= M <= N); N itself when
// the density's grid does not hold them either, or when the points saved are
// few: orbitals and fields take five launches more on a grid of their own.
int exx_grid(int N, int nmax, int nb);

// A tile of pairs: bands j0 .. j0 + bj - 1 with n0 .. n0 + bn - 1, j <= n, the
// pairs p0 .. p0 + np - 1 of the list (tile by tile, n ascending, then j).
constexpr int kExxTileMax = 8;
struct ExxTile {
    int j0, bj, n0, bn, p0, np;
};
int exx_tiles(int nb, int tile, std::vector<ExxTile>& out);   // returns the pairs

template <typename T>
struct ExxArgs {
    int M, nb, npairs, batch, ntiles;
    const ExxTile* tiles;     // host
    const ExxTile* d_tiles;   // device
    double L;
    const c2<T>* tw;      // twiddles of M
    const T* vG;          // v(G) / M^3
    const c2<T>* Phi;     // real-space orbitals, nb x M^3
    c2<T>* X;             // exchange fields, nb x M^3
    c2<T>* buf;           // batch x M^3
    const int* pj;        // pair list
    const int* pn;
    double* part;         // npairs x M
    double* Kmat;         // nb x nb
    double* hf2;          // [E_hf^M, E_hf^T] before alpha
    double* open_diag;    // exchange part of <a|F^c|a>, <b|F^c|b>
    ExxCoef cf;
};

template <typename T>
void exx_setup_kernel(int N, double L, int bare, T* vG, cudaStream_t st);
// K for all pairs, the energies and the open-band diagonal; the exchange
// fields X too when want_field.
template <typename T>
void exx_pairs(const ExxArgs<T>& a, bool want_field, cudaStream_t st);
// The grid work of the tiles t0 .. t1 - 1 (k_exx_grid.cuh): pair densities,
// transforms, v(G) and the planes' partials of the pair integrals in a.part,
// and with want_field the fields added to a.X.
template <typename T>
void exx_batch_grid(const ExxArgs<T>& a, int t0, int t1, bool want_field, cudaStream_t st);
// Real-space orbitals on the exchange's grid (s: the sphere seen from it; psi
// null: from the planes that Yp holds), and the fields' coefficients added to
// out; Zc and Yp are work space (nb columns and planes of that grid).
template <typename T>
void exx_orbitals(const Sphere& s, const c2<T>* tw, const c2<T>* psi, int64_t ld, int nb, c2<T>* Zc, c2<T>* Yp,
                  c2<T>* Phi, T scale, cudaStream_t st);
template <typename T>
void exx_add_fields(const Sphere& s, const c2<T>* tw, const c2<T>* X, int nb, c2<T>* Yp, c2<T>* Zc, c2<T>* out,
                    int64_t ldo, T scale, cudaStream_t st);

}  // namespace roks
