"""GPU: the band-space products and the blocked Cholesky beyond 64 bands where
their tiles end (65 and 130 bands: remainders of 1 and 2 of a block of 32;
tiles of 16 with K split eight ways, tiles of 32 from 152 of them on), through
the S-orthonormalisation: the oracle's overlap of the result is 1.

Tolerance: FP64 1e-11.  Mixed: the overlap's elements are FP32 sums with 22 to 24
significant bits per product, 5e-6, the suite's bar for S-orthonormality."""
import numpy as np
import pytest

from oracle import roks as R
from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,atoms", [(65, 9), (130, 9), (130, 170)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 5e-6)])
def test_orthonormalisation(nb, atoms, precision, tol):
    roks = built()
    base = syn.make_config("tiny-16", 0)
    rng = np.random.default_rng(nb + atoms)
    species = [{**sp, "Q": 0.01 * np.asarray(sp["Q"])} for sp in base["species"]]
    cfg = syn.with_changes(base, grid=32, L=12.0, ecut=0.5 * (2 * np.pi / 12.0 * 7.2) ** 2, n_closed=nb, mode=0,
                           species=species, atoms=[{**base["atoms"][i % len(base["atoms"])],
                                                   "pos": tuple(map(float, rng.uniform(0, 12.0, 3)))}
                                                  for i in range(atoms)])
    s = R.System(cfg)
    ctx = roks.Context(cfg, precision)
    psi = ctx.init_orbitals(syn.orbital_uniforms(cfg, ctx.npw))
    ctx.orthonormalize(psi)
    O = s.overlap(to_np(psi, ctx.npw))
    assert np.abs(O - np.eye(nb)).max() < tol
    ctx.close()
