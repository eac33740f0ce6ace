"""GPU: the sums of the tensor-core A^H B products.

* Orbitals that are single plane waves: no product is truncated and no sum
  rounded, the overlap is 1 and the orthonormalisation gives back its input, bit
  for bit.
* Runs of the (tile, stage) sequence below and beyond the 96 stages of a
  segment (256 bands: 18 stages a run; 512 and 640: 72 and 113 of a tile's 682,
  tiles cut by runs and runs over two tiles), against FP64 torch.  Tolerance: an element of
  the overlap is a sum of products of 22 significant bits (2^-22, random) in
  FP32, 5e-6 as elsewhere in the suite."""
import numpy as np
import pytest

from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built

pytestmark = pytest.mark.gpu


def context(roks, nb, grid, nmax):
    cfg = syn.make_config("tiny-16", 0)
    cfg["species"] = [dict(l=[], m=[], rc=[], D=np.zeros((0, 0)), Q=np.zeros((0, 0)))]
    L = cfg["L"]
    cfg = syn.with_changes(cfg, grid=grid, ecut=0.5 * (2 * np.pi / L * (nmax + 0.3)) ** 2, n_closed=nb, mode=0)
    return roks.Context(cfg, "mixed")


@pytest.mark.parametrize("nb", [128, 129, 200])
def test_plane_waves_stay_exact(nb):
    import torch
    roks = built()
    ctx = context(roks, nb, 32, 7)
    rows = np.random.default_rng(nb).permutation(ctx.npw)[:nb]
    psi = ctx.new_bands()
    psi.zero_()
    psi[torch.arange(nb), torch.from_numpy(rows)] = torch.tensor([1.0, 1j, -1.0, -1j] * (nb // 4 + 1))[:nb].to(psi)
    kept = psi.clone()
    ctx.orthonormalize(psi)
    assert torch.equal(psi, kept)
    ctx.close()


@pytest.mark.parametrize("nb", [256, 512, 640])
def test_long_runs(nb):
    import torch
    roks = built()
    ctx = context(roks, nb, 72, 17)
    assert ctx.npw > 20480
    gen = torch.Generator("cuda").manual_seed(nb)
    a = torch.view_as_complex(torch.randn((nb, ctx.npw, 2), generator=gen, dtype=torch.float32, device="cuda"))
    a *= (1.0 + torch.arange(ctx.npw, device="cuda") % 97) ** -1.0
    psi = ctx.new_bands()
    psi.zero_()
    psi[:, :ctx.npw] = a / a.abs().pow(2).sum(1, keepdim=True).sqrt()
    ctx.orthonormalize(psi)
    x = psi[:, :ctx.npw].to(torch.complex128)
    O = x.conj() @ x.T
    assert (O - torch.eye(nb, device="cuda")).abs().max().item() < 5e-6
    ctx.close()
