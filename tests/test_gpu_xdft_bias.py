"""GPU: nothing is added to what the x stage of the apply on the tensor cores
sums up.  An orbital that is one plane wave G has <G|F|G> = the mean of its class
potential plus the kinetic term; the bands are the 27 plane waves of lowest |G|,
the potentials those of eight random densities.

Tolerance.  The tensor cores' additions truncate, which can only take (at most two
units of 2^-23 in each of the two products); every other rounding is symmetric:
some 1.5e-7 of the potential a sample (the kinetic term is up to twice as large),
1e-8 in the mean over 216 samples.  Three of these: the mean error lies between
-4.8e-7 and 3e-8.  (A factor that gives back 2^-23 for each product moves it up by
2.4e-7.)"""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nmax", [(72, 17), (96, 15), (96, 22), (120, 20)])
def test_plane_waves(N, nmax):
    roks = built()
    L = 12.0
    cfg = syn.with_changes(syn.make_config("tiny-16", 0), L=L, grid=N, atoms=[], n_closed=27, mode=0,
                           ecut=0.5 * (2 * np.pi / L * (nmax + 0.2)) ** 2)
    c32, c64 = roks.Context(cfg, "mixed"), roks.Context(cfg, "fp64")
    miller = roks.roks_basis(c32.ctx)[3]
    rows = np.argsort((miller.astype(np.int64) ** 2).sum(1), kind="stable")[:27]
    waves = np.zeros((c32.npw, 27))
    waves[rows, np.arange(27)] = 1.0
    scale = float(np.float32(1.0 / N ** 3)) * N ** 3     # (1 / N^3 as the apply holds it)
    err = []
    for seed in range(8):
        rng = np.random.default_rng(seed)
        A = np.linalg.qr(rng.standard_normal((c32.npw, 27)) + 1j * rng.standard_normal((c32.npw, 27)))[0]
        diag, mean = [], []
        for ctx in (c64, c32):
            ctx.density(to_dev(ctx, A))
            V = ctx.potential(want_v=True)[1]
            mean.append(V[0].double().mean().item())
            F = to_np(ctx.apply_h(to_dev(ctx, waves))[0], ctx.npw)
            diag.append(F[rows, np.arange(27)].real)
        kinetic = diag[0] - mean[0]
        err.append((diag[1] - kinetic) / (scale * mean[1]) - 1.0)
    c32.close()
    c64.close()
    assert -4.8e-7 < np.mean(err) < 3e-8, np.mean(err)
