"""GPU: the network's wait for its tensor-core products obeys the context's wait
cap.  With no poll at all it runs out, is reported by the next checked call, and
goes on, so that nothing is read before it is there: the preconditioned block is
the same, bit for bit.  In a process of its own, without the streamed
contractions: tiny-16 in mixed precision then has no other kernel that waits."""
import os
import subprocess
import sys

import pytest

from tests.gpu_helpers import built

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np
import torch
from oracle import mlp as M
from paper_2605_28637_gb300 import roks, synthetic as syn
cfg = syn.make_config("tiny-16", 0)
p = torch.from_numpy(np.random.default_rng(5).uniform(-0.3, 0.3, M.NPARAM).astype(np.float32)).cuda()
got = []
for cap in (0, -1, 0):
    ctx = roks.Context(cfg, "mixed", wait_cap=cap)
    psi = ctx.init_orbitals(syn.orbital_uniforms(cfg, ctx.npw))
    ctx.density(psi)
    ctx.potential()
    g = ctx.apply_h(psi, want_grad=True)[2]
    ctx.set_preconditioner(p)
    got.append(ctx.precondition(g)[0].clone())
    try:
        assert np.isfinite(ctx.pcg_step(psi)["E_new"]) and cap == 0
    except roks.RoksError as e:
        assert cap < 0 and e.status == roks.ROKS_ETIMEOUT, e
    ctx.close()
assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
"""


def test_a_wait_that_runs_out_is_reported():
    built()
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       env=dict(os.environ, ROKS_STREAM="0"))
    assert r.returncode == 0, r.stderr[-2000:]
