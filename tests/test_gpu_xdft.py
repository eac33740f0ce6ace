"""GPU: the band transforms' x stages on the tensor cores (k_xdft.cu: mixed
path, N = 72, 96, 120, nmax <= (N - 1) / 4) at the ends of their frequency
chunks (nmax = 7, 8, 15, 16), of the staged planes (22 on 96^3) and of their
range, with few bands, groups of bands beyond one flush (16), a single band,
empty bands and the packed open pair of the Gamma point, against the FP64
path's register transforms on the same orbitals.

Tolerance.  A product carries 22 significant bits, the FP32 sums of the three
stages 2^-24 per addition, all relative to a line's largest value: a few
2^-22 in the root mean square, 1e-6 for the densities.  F|n> adds the mixed
path's potential (FP32 grid transforms, 2^-22 more): 2e-6."""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, rel, to_dev, to_np

pytestmark = pytest.mark.gpu


def system(N, nmax, **kw):
    L = 12.0
    return syn.with_changes(syn.make_config("tiny-16", 0), L=L, grid=N,
                            ecut=0.5 * (2 * np.pi / L * (nmax + 0.2)) ** 2, atoms=[], **kw)


CASES = [(72, 7, dict(n_closed=1)), (72, 8, dict(n_closed=2)), (72, 15, dict(n_closed=3)),
         (72, 16, dict(n_closed=1, n_empty=2)), (72, 17, dict(n_closed=2, mode=0)), (72, 7, dict(n_closed=150)),
         (96, 22, dict(n_closed=2)), (96, 23, dict(n_closed=1)), (120, 16, dict(n_closed=2)),
         (120, 29, dict(n_closed=1)), (72, 9, dict(n_closed=4, gamma=1)), (72, 12, dict(n_closed=1, mode=0))]


@pytest.mark.parametrize("N,nmax,kw", CASES)
def test_x_stages_against_fp64(N, nmax, kw):
    roks = built()
    kw = dict(kw)
    gamma = kw.pop("gamma", 0)
    cfg = system(N, nmax, **kw)
    ref = roks.Context(cfg, "fp64", gamma=gamma)
    rng = np.random.default_rng(N + nmax)
    A = rng.standard_normal((ref.npw, ref.nb)) + 1j * rng.standard_normal((ref.npw, ref.nb)) * (0 if gamma else 1)
    A *= (10.0 ** rng.uniform(-2, 0, ref.npw))[:, None]
    A = np.linalg.qr(A)[0].astype(np.complex64).astype(np.complex128)
    psi = to_dev(ref, A)
    rho = ref.density(psi, want_rho=True).cpu().numpy()
    ref.potential()
    F = to_np(ref.apply_h(psi)[0], ref.npw)
    ref.close()
    ctx = roks.Context(cfg, "mixed", gamma=gamma)
    psi = to_dev(ctx, A)
    for _ in range(2):                                   # the second time on planes the first has left
        got = ctx.density(psi, want_rho=True).cpu().numpy()
        for k in range(3):
            if np.any(rho[k]):
                assert rel(got[k], rho[k]) < 1e-6, k
        ctx.potential()
        f = to_np(ctx.apply_h(psi)[0], ctx.npw)
        assert rel(f, F) < 2e-6
    ctx.close()


def test_a_wait_that_runs_out_is_reported_and_nothing_read_early():
    """No poll at all: the density's waits run out, set the flag that the next
    checked call reports, and wait on, so the density is the same."""
    roks = built()
    cfg = system(72, 9, n_closed=20)
    ctx = roks.Context(cfg, "mixed")
    psi = ctx.init_orbitals(syn.orbital_uniforms(cfg, ctx.npw))
    rho = ctx.density(psi, want_rho=True).cpu().numpy()
    hasty = roks.Context(cfg, "mixed", wait_cap=-1)
    assert np.array_equal(hasty.density(psi, want_rho=True).cpu().numpy(), rho)
    hasty.close()
    with pytest.raises(roks.RoksError) as ei:
        ctx.orthonormalize(psi)
    assert ei.value.status == roks.ROKS_ETIMEOUT
    ctx.orthonormalize(psi)
    ctx.close()
