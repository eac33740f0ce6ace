"""GPU: long FP64 contractions (8192 rows and more) of few bands, where the
register tile and the thread grid are chosen by lanes issued: against NumPy's
Cholesky, and no slower than those of more bands.

Tolerance: FP64 sums in trees and an overlap with a condition number below 10,
1e-12 relative.  Times: least of ten; a call with half the bands does less of
everything, so 1.2 leaves room for noise (4 threads a block took 816 us at 8
bands, 533 at 17)."""
import numpy as np
import pytest

from tests.gpu_helpers import built, rel

pytestmark = pytest.mark.gpu


def block(npw, nb):
    rng = np.random.default_rng(npw + nb)
    A = rng.standard_normal((npw, nb)) + 1j * rng.standard_normal((npw, nb))
    return np.linalg.qr(A)[0] + 0.3 * A / np.linalg.norm(A, axis=0)


@pytest.mark.parametrize("npw", [8191, 8192, 20001])
@pytest.mark.parametrize("nb", [4, 6, 8, 9, 12, 17, 38])
def test_against_numpy(npw, nb):
    import torch
    roks = built()
    A = block(npw, nb)
    psi = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
    roks.roks_orthonormalize_noalloc(roks.ROKS_FP64, npw, nb, psi, npw, None)
    ref = A @ np.linalg.inv(np.linalg.cholesky(A.conj().T @ A)).conj().T
    assert rel(psi.cpu().numpy().T, ref) < 1e-12


@pytest.mark.parametrize("npw", [9000, 20000])
def test_fewer_bands_take_no_longer(npw):
    import torch
    roks = built()

    def least(nb):
        psi = torch.from_numpy(np.ascontiguousarray(block(npw, nb).T)).cuda()
        times = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            roks.roks_orthonormalize_noalloc(roks.ROKS_FP64, npw, nb, psi, npw,
                                             torch.cuda.current_stream().cuda_stream)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[2:])

    t = {nb: least(nb) for nb in (8, 9, 12, 17, 24, 34)}
    for few, many in ((8, 17), (9, 17), (12, 24), (17, 34)):
        assert t[few] < 1.2 * t[many], t
