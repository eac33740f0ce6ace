"""GPU: the allocation-free orthonormalisation's status: a singular overlap is
reported and leaves psi as it is, and the call after it, by either of its two
forms (one cluster up to 7 bands, a chain of kernels), starts clear.

Tolerance: orthonormality 1e-12 in FP64, 2e-6 in FP32, as elsewhere."""
import itertools

import numpy as np
import pytest

from tests.gpu_helpers import built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("bad,good", list(itertools.product([(200, 4), (1000, 12), (9000, 9)], [(300, 5), (900, 20)])))
def test_status_starts_clear(bad, good, f64):
    import torch
    roks = built()
    prec, dtype = (roks.ROKS_FP64, np.complex128) if f64 else (roks.ROKS_MIXED, np.complex64)
    rng = np.random.default_rng(bad[0] + good[0])

    def block(npw, nb):
        return (rng.standard_normal((nb, npw)) + 1j * rng.standard_normal((nb, npw))).astype(dtype)

    X = block(*bad)
    X[2] = 0.0
    psi = torch.from_numpy(X).cuda()
    with pytest.raises(roks.RoksError) as ei:
        roks.roks_orthonormalize_noalloc(prec, *bad, psi, bad[0], None)
    assert ei.value.status == roks.ROKS_ENOTPOSDEF
    assert np.array_equal(psi.cpu().numpy(), X)
    psi = torch.from_numpy(block(*good)).cuda()
    roks.roks_orthonormalize_noalloc(prec, *good, psi, good[0], None)
    G = psi.cpu().numpy().astype(np.complex128)
    assert np.abs(G.conj() @ G.T - np.eye(good[1])).max() < (1e-12 if f64 else 2e-6)


def test_one_call_after_another_on_three_streams():
    """The product of a call may still run when it has returned; the next call, on
    another stream, must not change the scratch under it."""
    import torch
    roks = built()
    sizes = [(40000, 24), (30000, 17), (40000, 24), (900, 9), (40000, 30), (2000, 40)]
    streams = [torch.cuda.Stream().cuda_stream, None, torch.cuda.Stream().cuda_stream]     # (None: the legacy stream)
    blocks = []
    for npw, nb in sizes:
        gen = torch.Generator("cuda").manual_seed(npw + nb)
        blocks.append(torch.view_as_complex(torch.randn((nb, npw, 2), generator=gen, dtype=torch.float64, device="cuda")))
    torch.cuda.synchronize()
    for k, X in enumerate(blocks):
        roks.roks_orthonormalize_noalloc(roks.ROKS_FP64, X.shape[1], X.shape[0], X, X.shape[1],
                                         streams[k % 3])
    torch.cuda.synchronize()
    for X in blocks:
        assert (X.conj() @ X.T - torch.eye(X.shape[0], device="cuda")).abs().max().item() < 1e-12
