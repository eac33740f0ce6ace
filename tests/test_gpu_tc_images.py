"""GPU: the tensor-core contractions' operand images (k_tcgemm.cu) at the
sizes where tiles, stages, column groups and chunks of rows end, through
roks_orthonormalize on systems without projectors (S = 1): Psi L^{-H} with
Psi^H Psi = L L^H, against NumPy in FP64.

Tolerance.  Every product carries 22 significant bits (2^-22 relative per
product, random) and FP32 sums (2^-24 per stage); the band-space Cholesky of
an overlap with |O - 1| < 1/2 runs in FP32.  A few 2^-22 in the root mean
square: 1e-6 bounds the relative error of the block, and the columns' scales
(powers of ten that the images take out) change nothing in it."""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, rel, to_dev, to_np

pytestmark = pytest.mark.gpu


def system(nb, nmax):
    cfg = syn.make_config("tiny-16", 0)
    L = 12.0
    return syn.with_changes(cfg, L=L, grid=32, ecut=0.5 * (2 * np.pi / L * (nmax + 0.2)) ** 2, atoms=[],
                            n_closed=nb, mode=0)


SIZES = [(64, 10), (65, 11), (127, 10), (128, 10), (129, 11), (200, 12), (257, 11)]


# (up to 64 bands the mixed path's Cholesky takes overlaps near 1 only: no scaled columns there)
@pytest.mark.parametrize("nb,nmax,scaled", [(*s, False) for s in SIZES] + [(*s, True) for s in SIZES if s[0] > 64])
def test_orthonormalisation_at_the_edges(nb, nmax, scaled):
    roks = built()
    ctx = roks.Context(system(nb, nmax), "mixed")
    assert ctx.npw >= 4096
    rng = np.random.default_rng(nb + nmax)
    A = rng.standard_normal((ctx.npw, nb)) + 1j * rng.standard_normal((ctx.npw, nb))
    A *= (10.0 ** rng.uniform(-3, 0, ctx.npw))[:, None]     # rows of unlike size, as plane waves have
    A = np.linalg.qr(A)[0] + 0.01 * A / np.linalg.norm(A, axis=0)
    if scaled:
        A = A * 10.0 ** rng.uniform(-6, 6, nb)
    psi = to_dev(ctx, A)
    A = to_np(psi, ctx.npw)                                # as rounded to FP32
    ref = A @ np.linalg.inv(np.linalg.cholesky(A.conj().T @ A)).conj().T
    ctx.orthonormalize(psi)
    assert rel(to_np(psi, ctx.npw), ref) < 1e-6
    ctx.close()


def test_a_wait_that_runs_out_is_reported():
    """No poll at all: every wait of the contraction gives up, its copies and
    MMAs in flight are waited for, and the call returns ROKS_ETIMEOUT."""
    roks = built()
    cfg = system(128, 10)
    ctx = roks.Context(cfg, "mixed", wait_cap=-1)
    with pytest.raises(roks.RoksError) as ei:
        ctx.init_orbitals(syn.orbital_uniforms(cfg, ctx.npw))
    assert ei.value.status == roks.ROKS_ETIMEOUT
    ctx.close()
    ctx = roks.Context(cfg, "mixed")
    psi = ctx.init_orbitals(syn.orbital_uniforms(cfg, ctx.npw))
    P = to_np(psi, ctx.npw)
    assert np.abs(P.conj().T @ P - np.eye(128)).max() < 3e-6
    ctx.close()
