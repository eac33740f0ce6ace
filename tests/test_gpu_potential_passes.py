"""GPU: the potentials' three passes over the grid (k_pot_impl.cuh) and the plane
transforms of the gradient correction, on every grid length, against the FP64
oracle: class potentials and each energy.  (FP64 beyond 32: separate y and z
passes.)

Tolerance: FP64 1e-10 relative, the suite's bar.  Mixed, Slater: FP32 transforms
and densities, 1e-6 of the potential's norm, 1e-6 of the energies' sum."""
import numpy as np
import pytest

from oracle import roks as R
from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built, rel, to_dev

pytestmark = pytest.mark.gpu

GRIDS = [(16, 10.0, 8.0), (24, 11.0, 12.0), (32, 12.0, 20.0), (48, 12.0, 35.0), (72, 14.0, 6.0), (96, 16.0, 6.0),
         (120, 16.0, 6.0)]
KEYS = (("E_loc", "loc"), ("E_H", "H"), ("E_x_M", "x_M"), ("E_x_T", "x_T"))


@pytest.mark.parametrize("xc", ["slater", "pbe_x"])
@pytest.mark.parametrize("N,L,ecut", GRIDS)
def test_potentials(N, L, ecut, xc):
    roks = built()
    cfg = syn.with_changes(syn.make_config("tiny-16", 0), grid=N, L=L, ecut=ecut, n_closed=2, xc=xc)
    s = R.System(cfg)
    P = s.initial_orbitals(syn.orbital_uniforms(cfg, s.npw))
    P = P.astype(np.complex64).astype(np.complex128)
    pot = s.potentials(s.class_densities(P))
    ref = s.energies(P, pot)
    size = sum(abs(ref[k]) for _, k in KEYS)
    for precision, tol in (("fp64", 1e-10), ("mixed", 1e-6)):
        if precision == "mixed" and xc != "slater":
            continue
        ctx = roks.Context(cfg, precision)
        psi = to_dev(ctx, P)
        for _ in range(2):
            ctx.density(psi)
            E, V = ctx.potential(want_v=True)
            assert rel(V.cpu().numpy().astype(np.float64), pot.Vk) < tol, precision
            for g, k in KEYS:
                assert abs(E[g] - ref[k]) < tol * size, (precision, k)
        ctx.close()
