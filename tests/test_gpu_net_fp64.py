"""GPU: the network preconditioner of an FP64 context evaluates the network in FP32
on the CUDA cores, with the values it has always had (tests/golden/net_fp64.json):
FP64 results hold 1e-9 against each other.  (On the tensor cores, with products
of 22 significant bits, they moved by 5e-8.)

Tolerance: the inputs are exact, the evaluation has one order: 1e-9 leaves room
for the FP64 sums behind the features."""
import json
import os

import numpy as np
import pytest

from oracle import mlp as M
from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "net_fp64.json")


def test_values():
    import torch
    roks = built()
    cfg = syn.make_config("tiny-16", 0)
    ctx = roks.Context(cfg, "fp64")
    psi = ctx.init_orbitals(syn.orbital_uniforms(cfg, ctx.npw))
    ctx.density(psi)
    ctx.potential()
    ctx.apply_h(psi, want_grad=True)
    rng = np.random.default_rng(11)
    A = rng.standard_normal((ctx.nb, ctx.npw, 2)).astype(np.float32)
    A *= (10.0 ** rng.integers(-4, 1, (ctx.nb, ctx.npw, 1))).astype(np.float32)
    g = ctx.new_bands()
    g.zero_()
    g[:, :ctx.npw] = torch.view_as_complex(torch.from_numpy(A.astype(np.float64))).cuda()
    p = np.random.default_rng(5).uniform(-0.5, 0.5, M.NPARAM).astype(np.float32)
    ctx.set_preconditioner(torch.from_numpy(p).cuda())
    got = ctx.precondition(g)[0][:, :ctx.npw].cpu().numpy()[:, ::64]
    ctx.close()
    with open(GOLDEN) as f:
        want = np.array(json.load(f)["values"]) @ np.array([1.0, 1j])
    assert np.abs(got / want - 1.0).max() < 1e-9
