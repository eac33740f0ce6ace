"""GPU: the network's wait for its tensor-core products obeys the context's wait
cap.  With no poll at all it runs out, is reported by the next checked call, and
goes on, so that nothing is read before it is there: the preconditioned block is
the same, bit for bit."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2605_28637_gb300 import synthetic as syn
from tests.gpu_helpers import built

pytestmark = pytest.mark.gpu


def test_a_wait_that_runs_out_is_reported():
    import torch
    roks = built()
    cfg = syn.make_config("tiny-16", 0)
    p = torch.from_numpy(np.random.default_rng(5).uniform(-0.3, 0.3, M.NPARAM).astype(np.float32)).cuda()
    u = None
    got = []
    for cap in (0, -1):
        ctx = roks.Context(cfg, "fp64", wait_cap=cap)      # (FP64: no other kernel waits)
        u = syn.orbital_uniforms(cfg, ctx.npw) if u is None else u
        psi = ctx.init_orbitals(u)
        ctx.density(psi)
        ctx.potential()
        g = ctx.apply_h(psi, want_grad=True)[2]
        ctx.set_preconditioner(p)
        got.append(ctx.precondition(g)[0].clone())
        if cap == 0:
            ctx.pcg_step(psi)
        else:
            with pytest.raises(roks.RoksError) as ei:
                ctx.pcg_step(psi)
            assert ei.value.status == roks.ROKS_ETIMEOUT
        ctx.close()
    assert torch.equal(got[0], got[1])
    # and nothing is left over for the next context
    ctx = roks.Context(cfg, "fp64")
    psi = ctx.init_orbitals(u)
    ctx.set_preconditioner(p)
    assert np.isfinite(ctx.pcg_step(psi)["E_new"])
    ctx.close()
