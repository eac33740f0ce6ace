"""GPU: the network kernels at the ends of their tiles (128 rows, and as many
tiles as blocks are resident), against the FP64 oracle.

Tolerances, for |weights| <= 0.6 and |features| of a few: an activation is good
to 3e-7, a layer sums 64 of them in FP32 (22-bit operands on the tensor
cores), so outputs of size up to 20 stay within 2e-5 and gradients within 1e-4
of the largest entry.  Saturated rows (|z| far above 10) are exact in tanh."""
import numpy as np
import pytest

from oracle import mlp as M
from tests.gpu_helpers import built

pytestmark = pytest.mark.gpu


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("n", [1, 127, 128, 129, 4 * 152 * 128 + 1])
@pytest.mark.parametrize("bf16", [0, 1])
def test_forward_rows(n, bf16):
    import torch
    roks = built()
    rng = np.random.default_rng(n)
    U = rng.normal(size=(n, 3)).astype(np.float32)
    U[0] = (40.0, -55.0, 90.0)                       # saturated units
    U[n // 2] = 0.0                                 # the polynomial alone
    p = rng.uniform(-0.6, 0.6, M.NPARAM).astype(np.float32)
    if bf16:
        p = torch.from_numpy(p).to(torch.bfloat16).float().numpy()
    s = torch.full((n + 1,), 7.0, device="cuda")
    roks.roks_mlp_forward(n, dev(U), dev(p), bf16, s)
    ref, _, _ = M.forward(p.astype(np.float64), U.astype(np.float64))
    got = s.cpu().numpy()
    assert np.abs(got[:n] - ref).max() < 2e-5
    assert got[n] == 7.0                            # nothing past the last row


def test_forward_keeps_nan_in_its_row():
    import torch
    roks = built()
    rng = np.random.default_rng(3)
    U = rng.normal(size=(200, 3)).astype(np.float32)
    U[17, 1] = np.nan
    p = rng.uniform(-0.6, 0.6, M.NPARAM).astype(np.float32)
    s = torch.empty(200, device="cuda")
    roks.roks_mlp_forward(200, dev(U), dev(p), 0, s)
    bad = np.isnan(s.cpu().numpy())
    assert bad[17] and bad.sum() == 1


@pytest.mark.parametrize("n", [1, 128, 129, 2049])
def test_gradient_rows(n):
    import torch
    roks = built()
    rng = np.random.default_rng(n + 5)
    U, t = rng.normal(size=(n, 3)), rng.normal(size=n)
    w = rng.uniform(0.1, 2.0, n)
    p = rng.uniform(-0.6, 0.6, M.NPARAM).astype(np.float32)
    U, t, w = (x.astype(np.float32) for x in (U, t, w))
    g, loss = torch.empty(M.NPARAM, device="cuda"), torch.empty(1, device="cuda")
    work = torch.empty(roks.roks_mlp_grad_work(n), device="cuda")
    roks.roks_mlp_grad(n, dev(U), dev(t), dev(w), dev(p), work, g, loss)
    L, gref = M.loss_and_grad(*(x.astype(np.float64) for x in (p, U, t, w)))
    assert abs(float(loss.item()) - L) < 1e-5 * max(1.0, abs(L))
    assert np.abs(g.cpu().numpy() - gref).max() < 1e-4 * np.abs(gref).max()
