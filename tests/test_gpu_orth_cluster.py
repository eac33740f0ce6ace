"""GPU: the allocation-free orthonormalisation where its one-cluster kernel
begins and ends (fewer rows than blocks, one band, odd splits, the last sizes
it takes and the first it does not), against NumPy's Cholesky in FP64, and the
failed pivot that leaves psi as it was.

Tolerance: products of the element type summed in trees (FP64: some 1e-15;
FP32: 2^-24 per product and sum, a few of them), a band-space Cholesky in FP64
of an overlap with a condition number below 10: 1e-12 and 2e-6 relative."""
import numpy as np
import pytest

from tests.gpu_helpers import built, rel

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (5, 3), (900, 7), (900, 8), (900, 9), (64, 1), (500, 2), (1045, 6), (1000, 15), (975, 16), (977, 16), (6944, 6), (6945, 6),
         (300, 28), (4000, 31), (400, 50), (700, 64)]


@pytest.mark.parametrize("npw,nb", SIZES)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_against_numpy(npw, nb, precision):
    import torch
    roks = built()
    f64 = precision == "fp64"
    rng = np.random.default_rng(npw + nb)
    A = rng.standard_normal((npw, nb)) + 1j * rng.standard_normal((npw, nb))
    A = np.linalg.qr(A)[0] + 0.3 * A / np.linalg.norm(A, axis=0)
    A = A.astype(np.complex128 if f64 else np.complex64)
    ld = npw + 3
    psi = torch.full((nb, ld), 7.0, dtype=torch.complex128 if f64 else torch.complex64, device="cuda")
    psi[:, :npw] = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
    prec = roks.ROKS_FP64 if f64 else roks.ROKS_MIXED
    A = A.astype(np.complex128)
    ref = A @ np.linalg.inv(np.linalg.cholesky(A.conj().T @ A)).conj().T
    torch.cuda.synchronize()
    roks.roks_orthonormalize_noalloc(prec, npw, nb, psi, ld, None)
    torch.cuda.synchronize()
    assert rel(psi[:, :npw].T.cpu().numpy(), ref) < (1e-12 if f64 else 2e-6)
    assert (psi[:, npw:] == 7.0).all()


@pytest.mark.parametrize("npw,nb", [(1045, 6), (20000, 6)])
def test_a_failed_pivot_keeps_psi(npw, nb):
    import torch
    roks = built()
    psi = torch.randn((nb, npw), dtype=torch.complex128, device="cuda")
    psi[3] = 0.0
    kept = psi.clone()
    torch.cuda.synchronize()
    with pytest.raises(roks.RoksError) as ei:
        roks.roks_orthonormalize_noalloc(roks.ROKS_FP64, npw, nb, psi, npw, None)
    assert ei.value.status == roks.ROKS_ENOTPOSDEF
    assert torch.equal(psi, kept)
