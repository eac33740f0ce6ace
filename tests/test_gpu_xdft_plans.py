"""GPU: how the x stages on the tensor cores are run, against the FP64 path's
register transforms on the same orbitals.

* Staged planes or loaded ones: the last sphere that is staged with two blocks an
  SM (nmax 21), the first that is not (22; the density on 120^3 stays staged).
* Two blocks an SM: an apply of the sphere beyond takes no jump in time.
* The fewest bands that take the tensor cores (5 on 72^3, 2 on 96^3, 1 on 120^3)
  and one fewer; the density of the widest sphere of 96^3 up to 32 bands; and the
  ends of the frequency chunks with more bands than that.

Tolerances as in the suite's other test of these stages: 1e-6 for densities, 2e-6
for F|n>."""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, rel, to_dev, to_np

pytestmark = pytest.mark.gpu


def system(N, nmax, **kw):
    L = 12.0
    return syn.with_changes(syn.make_config("tiny-16", 0), L=L, grid=N,
                            ecut=0.5 * (2 * np.pi / L * (nmax + 0.2)) ** 2, atoms=[], **kw)


def orbitals(ctx, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((ctx.npw, ctx.nb)) + 1j * rng.standard_normal((ctx.npw, ctx.nb))
    A *= (10.0 ** rng.uniform(-2, 0, ctx.npw))[:, None]
    return np.linalg.qr(A)[0].astype(np.complex64).astype(np.complex128)


def compare(N, nmax, **kw):
    roks = built()
    cfg = system(N, nmax, **kw)
    A, out = None, []
    for precision in ("fp64", "mixed"):
        ctx = roks.Context(cfg, precision)
        A = orbitals(ctx, N + nmax) if A is None else A
        psi = to_dev(ctx, A)
        rho = ctx.density(psi, want_rho=True).cpu().numpy()
        ctx.potential()
        out.append((rho, to_np(ctx.apply_h(psi)[0], ctx.npw)))
        ctx.close()
    (rho, F), (got, f) = out
    for k in range(3):
        if np.any(rho[k]):
            assert rel(got[k], rho[k]) < 1e-6, k
    assert rel(f, F) < 2e-6


@pytest.mark.parametrize("N,nmax", [(96, 21), (96, 22), (120, 21), (120, 22)])
def test_staged_and_loaded(N, nmax):
    compare(N, nmax, n_closed=21)


def test_two_blocks_share_an_sm_beyond_the_staged_spheres():
    """One more plane pair is 5% more work; with one block an SM the apply's x
    stage took 1.36 of the time."""
    import torch
    roks = built()
    least = []
    for nmax in (21, 22):
        ctx = roks.Context(system(96, nmax, n_closed=160, mode=0), "mixed")
        psi = to_dev(ctx, orbitals(ctx, nmax))
        ctx.density(psi)
        ctx.potential()
        t = []
        for _ in range(8):
            roks.roks_profile_enable(ctx.ctx, 1)
            ctx.apply_h(psi)
            torch.cuda.synchronize()
            t += [e["ms"] for e in roks.roks_profile_read(ctx.ctx) if e["name"] == "fft_x_apply"]
            roks.roks_profile_enable(ctx.ctx, 0)
        least.append(min(t))
        ctx.close()
    assert least[1] < 1.2 * least[0], least


@pytest.mark.parametrize("N,nmax,nb", [(72, 17, 4), (72, 17, 5), (96, 14, 1), (96, 14, 2), (120, 9, 1), (96, 23, 32),
                                       (96, 23, 33), (72, 7, 8), (72, 8, 8), (72, 15, 8), (72, 16, 8), (72, 17, 8)])
def test_few_bands(N, nmax, nb):
    compare(N, nmax, n_closed=nb, mode=0)


def test_one_band_is_no_slower_than_it_was():
    """The density's x stage of one band on 72^3 against six, which take the tensor
    cores: 11.2 and 17.3 us; 15.1 with both on them."""
    import torch
    roks = built()
    least = []
    for nb in (1, 6):
        ctx = roks.Context(system(72, 17, n_closed=nb, mode=0), "mixed")
        psi = to_dev(ctx, orbitals(ctx, nb))
        ctx.density(psi)
        ctx.potential()
        t = []
        for _ in range(20):
            roks.roks_profile_enable(ctx.ctx, 1)
            ctx.density(psi)
            torch.cuda.synchronize()
            t += [e["ms"] for e in roks.roks_profile_read(ctx.ctx) if e["name"] == "fft_x_density"]
            roks.roks_profile_enable(ctx.ctx, 0)
        least.append(min(t))
        ctx.close()
    assert least[0] < 0.78 * least[1], least
