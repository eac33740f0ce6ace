"""GPU: the density's factor 1 / Omega on the tensor-core x stage.  The same
coefficients in two cells whose 1 / Omega rounds to FP32 by -5.5e-8 and +5.4e-8:
Omega rho is the same grid of numbers.

Tolerance: the compensated sums carry the factor in two words (2^-48); what is
left is the output's own rounding to FP32, 2^-24 random a point, in the mean
over N^3 points below 1e-9."""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nmax", [(72, 17), (96, 20), (120, 12)])
def test_two_cells(N, nmax):
    roks = built()
    got = []
    for L in (25.36, 25.04):
        cfg = syn.with_changes(syn.make_config("tiny-16", 0), L=L, grid=N, atoms=[], n_closed=20, mode=0,
                               ecut=0.5 * (2 * np.pi / L * (nmax + 0.2)) ** 2)
        ctx = roks.Context(cfg, "mixed")
        rng = np.random.default_rng(N)
        A = rng.standard_normal((ctx.npw, ctx.nb)) + 1j * rng.standard_normal((ctx.npw, ctx.nb))
        A /= np.linalg.norm(A, axis=0)
        rho = ctx.density(to_dev(ctx, A), want_rho=True)[0]
        got.append(rho.mean().item() * L ** 3)
        ctx.close()
    assert abs(got[0] / got[1] - 1.0) < 2e-9
