"""GPU: the tensor-core contractions with 32 to 63 columns (and 31, which the
streamed FP32 kernels keep): F|n>, S|n> and the gradient of systems with at
least 128 projectors and 4096 plane waves, against the FP64 path on the same
orbitals.

Tolerance: products of 22 significant bits (2^-22, random) and FP32 sums; F
adds the mixed path's transforms and potential (a few 2^-22): 2e-6."""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, rel, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [31, 32, 33, 40, 47, 49, 63])
def test_apply_against_fp64(nb):
    roks = built()
    base = syn.make_config("tiny-16", 0)
    rng = np.random.default_rng(nb)
    atoms = [{**base["atoms"][i % len(base["atoms"])], "pos": tuple(map(float, rng.uniform(0, 12.0, 3)))}
             for i in range(18 + nb % 5)]
    cfg = syn.with_changes(base, grid=48, L=12.0, ecut=0.5 * (2 * np.pi / 12.0 * 10.2) ** 2, n_closed=nb, mode=0,
                           atoms=atoms)
    out = []
    A = None
    for precision in ("fp64", "mixed"):
        ctx = roks.Context(cfg, precision)
        assert ctx.npw >= 4096
        if A is None:
            A = rng.standard_normal((ctx.npw, nb)) + 1j * rng.standard_normal((ctx.npw, nb))
            A *= (10.0 ** rng.uniform(-2, 0, ctx.npw))[:, None]
            A = np.linalg.qr(A)[0].astype(np.complex64).astype(np.complex128)
        psi = to_dev(ctx, A)
        ctx.density(psi)
        ctx.potential()
        out.append([to_np(x, ctx.npw) for x in ctx.apply_h(psi, want_grad=True)])
        ctx.close()
    for name, ref, got in zip("FSg", *out):
        assert rel(got, ref) < 2e-6, name
