"""GPU: the exact exchange on its own grid (k_exx_grid.cuh) where the grid's
length changes (4 nmax + 1 just within 16, 24, 40, 54, 60, 64, 80, 108), where
the density's grid is taken (few bands; 72 and 120; planes beyond the shared
memory in FP64 at 120), where it holds the sphere with aliasing only (16^3,
nmax 6), and where tiles of 8 bands end (7, 8, 9, 17 bands, closed and open classes in one
tile), against the FP64 oracle on the density's grid.

Tolerance.  Both grids represent the same band-limited products, so FP64
differs by rounding: 1e-10 relative, the suite's bar.  Mixed: 22 to 24
significant bits per product and FP32 sums in every stage: 2e-6 for F|n>, 2e-6
of the exchange energies."""
import numpy as np
import pytest

from oracle import roks as R
from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, rel, to_dev, to_np

pytestmark = pytest.mark.gpu

CASES = [(24, 3, 7, 0), (24, 3, 8, 0), (24, 3, 6, 1), (24, 3, 7, 1), (24, 3, 15, 2), (16, 6, 3, 1), (32, 5, 9, 1),
         (48, 9, 5, 1), (72, 13, 1, 1), (72, 14, 4, 0), (72, 15, 4, 0), (72, 17, 2, 0), (96, 19, 2, 0),
         (120, 26, 2, 0), (120, 29, 2, 0)]


@pytest.mark.parametrize("N,nmax,n_closed,mode", CASES)
def test_exchange_against_the_oracle(N, nmax, n_closed, mode):
    roks = built()
    L = 12.0
    cfg = syn.with_changes(syn.make_config("tiny-16", 0), L=L, grid=N, atoms=[], n_closed=n_closed, mode=mode,
                           ecut=0.5 * (2 * np.pi / L * (nmax + 0.2)) ** 2, alpha=0.25)
    s = R.System(cfg)
    rng = np.random.default_rng(N + nmax + n_closed)
    nb = syn.n_bands(cfg)
    A = rng.standard_normal((s.npw, nb)) + 1j * rng.standard_normal((s.npw, nb))
    A *= (10.0 ** rng.uniform(-2, 0, s.npw))[:, None]
    P = np.linalg.qr(A)[0].astype(np.complex64).astype(np.complex128)
    pot = s.potentials(s.class_densities(P))
    E = s.energies(P, pot)
    F, _ = s.apply(P, pot)
    for precision, tf, te in (("fp64", 1e-10, 1e-10), ("mixed", 2e-6, 2e-6)):
        ctx = roks.Context(cfg, precision)
        psi = to_dev(ctx, P)
        ctx.density(psi)
        e = ctx.potential()
        assert abs(e["E_total"] - E["total"]) < te * sum(abs(v) for k, v in e.items() if k != "E_total"), precision
        for _ in range(2):
            assert rel(to_np(ctx.apply_h(psi)[0], ctx.npw), F) < tf, precision
        ctx.close()
