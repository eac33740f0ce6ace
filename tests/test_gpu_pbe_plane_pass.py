"""GPU: mixed precision with PBE exchange on every grid length, where the FP32 plane
pass carries all grid transforms of the gradient correction, against the FP64
path: class potentials and energies.

Tolerance: the gradient and the divergence each multiply the 2^-22 of an FP32
transform by the ratio of the largest to the mean |G| of the density, some 4:
2^-22 * 16 = 4e-6 of the largest entry; 2e-5, the suite's mixed bar for F|n>,
leaves room for points of low density.  Energies: 2e-6 of their sum."""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, rel, to_dev

pytestmark = pytest.mark.gpu

GRIDS = [(16, 10.0, 8.0), (24, 11.0, 12.0), (32, 12.0, 20.0), (48, 12.0, 35.0), (72, 14.0, 6.0), (96, 16.0, 6.0),
         (120, 16.0, 6.0)]
KEYS = ("E_loc", "E_H", "E_x_M", "E_x_T")


@pytest.mark.parametrize("N,L,ecut", GRIDS)
def test_potentials(N, L, ecut):
    roks = built()
    cfg = syn.with_changes(syn.make_config("tiny-16", 0), grid=N, L=L, ecut=ecut, n_closed=20, xc="pbe_x")
    A, out = None, []
    for precision in ("fp64", "mixed"):
        ctx = roks.Context(cfg, precision)
        if A is None:
            rng = np.random.default_rng(N)
            A = np.linalg.qr(rng.standard_normal((ctx.npw, ctx.nb)) + 1j * rng.standard_normal((ctx.npw, ctx.nb)))[0]
            A = A.astype(np.complex64).astype(np.complex128)
        psi = to_dev(ctx, A)
        for _ in range(2):
            ctx.density(psi)
            E, V = ctx.potential(want_v=True)
        out.append((E, V.cpu().numpy().astype(np.float64)))
        ctx.close()
    (E, V), (e, v) = out
    assert rel(v, V) < 2e-5
    size = sum(abs(E[k]) for k in KEYS)
    for k in KEYS:
        assert abs(e[k] - E[k]) < 2e-6 * size, k
