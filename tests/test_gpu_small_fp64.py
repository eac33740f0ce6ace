"""GPU: FP64 PCG steps of small systems against the oracle where the kernels
for few bands change: the exponential of one block (up to 12 bands), of a
cluster (13 .. 48) and by launches (49), tall products split over columns and
over chunks of half a slice.  Tolerance: the suite's FP64 bars, 1e-9 of the
step's energies, and an overlap of 1 to 1e-8."""
import numpy as np
import pytest

from oracle import roks as R
from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_closed,grid,ecut", [(1, 16, 8.0), (4, 16, 8.0), (10, 16, 8.0), (11, 16, 8.0),
                                                (30, 24, 12.0), (46, 24, 12.0), (47, 24, 12.0)])
def test_pcg_steps(n_closed, grid, ecut):
    roks = built()
    cfg = syn.with_changes(syn.make_config("tiny-16", 0), n_closed=n_closed, grid=grid, ecut=ecut)
    s = R.System(cfg)
    u = syn.orbital_uniforms(cfg, s.npw)
    ctx = roks.Context(cfg, "fp64")
    psi = ctx.init_orbitals(u)
    P = s.initial_orbitals(u)
    pcg = R.PCG(s)
    for _ in range(2):
        info = ctx.pcg_step(psi)
        P, ref = pcg.step(P)
        assert abs(info["E_new"] - ref.E_new) <= 1e-9 * max(1.0, abs(ref.E_new))
    O = s.overlap(to_np(psi, ctx.npw))
    assert np.abs(O - np.eye(len(O))).max() < 1e-8
    ctx.close()
