"""GPU: launches whose dynamic shared memory comes to just under 48 KB, the
limit that a launch has without asking for more and that the kernel's static
arrays share.  Each in a process of its own: a larger launch raises the limit
for all later ones of the process.

Tolerance: the orthonormality that the suite asks of these calls, 1e-12 in FP64
and 2e-6 in FP32."""
import os
import subprocess
import sys

import pytest

from tests.gpu_helpers import built

pytestmark = pytest.mark.gpu

FREE = """
import torch
from paper_2605_28637_gb300 import roks
npw, nb, f64 = {npw}, {nb}, {f64}
g = torch.Generator("cuda").manual_seed(npw + nb)
a = torch.view_as_complex(torch.randn((npw, nb, 2), generator=g, dtype=torch.float64, device="cuda"))
a = torch.linalg.qr(a)[0] + 0.02 * a / a.abs().pow(2).sum(0).sqrt()
psi = a.T.contiguous().to(torch.complex128 if f64 else torch.complex64)
torch.cuda.synchronize()
roks.roks_orthonormalize_noalloc(roks.ROKS_FP64 if f64 else roks.ROKS_MIXED, npw, nb, psi, npw, None)
x = psi.to(torch.complex128)
err = (x.conj() @ x.T - torch.eye(nb, device="cuda")).abs().max().item()
assert err < (1e-12 if f64 else 2e-6), err
"""


def alone(code):
    built()
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stderr[-2000:]


# 48,637 to 49,152 bytes: the cluster kernel's dynamic part alone fits 48 KB
@pytest.mark.parametrize("npw,nb,f64", [(3320, 7, True), (3930, 6, True), (5720, 8, False)])
def test_orthonormalize_noalloc_cluster(npw, nb, f64):
    alone(FREE.format(npw=npw, nb=nb, f64=f64))


# 39 bands: 48,672 bytes of the Cholesky kernel's matrices
@pytest.mark.parametrize("nb", [38, 39, 40])
@pytest.mark.parametrize("f64", [True, False])
def test_orthonormalize_noalloc_chain(nb, f64):
    alone(FREE.format(npw=1000, nb=nb, f64=f64))


STEP = """
import numpy as np
from oracle import roks as R
from paper_2605_28637_gb300 import roks, synthetic as syn
cfg = syn.with_changes(syn.make_config("tiny-16", 0), n_closed={nb}, grid=24, ecut=12.0, mode=0)
s = R.System(cfg)
u = syn.orbital_uniforms(cfg, s.npw)
ctx = roks.Context(cfg, "fp64")
psi = ctx.init_orbitals(u)
x = psi[:, :ctx.npw].cpu().numpy().T
assert np.abs(s.overlap(x) - np.eye({nb})).max() < 1e-12
"""


@pytest.mark.parametrize("nb", [38, 39, 40])
def test_orthonormalisation(nb):
    alone(STEP.format(nb=nb))
