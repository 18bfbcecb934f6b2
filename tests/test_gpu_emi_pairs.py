"""gamma_t at the edges of its pair split (odd and even date counts, every row
length) against a plain 64-bit sum over pairs, from the linked phases."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 3, 7, 8, 9, 15, 16, 17, 20, 21, 24, 25, 28, 31, 32])
def test_tcoh_of_linked_phases(N):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2511_12051_gb300 import build, plk
    build.build()
    rng = np.random.default_rng(N)
    P, ref = 301, N - 1
    z = rng.standard_normal((P, N, 60)) + 1j * rng.standard_normal((P, N, 60))
    z = z + 1.2 * (rng.standard_normal((P, 1, 60)) + 1j * rng.standard_normal((P, 1, 60)))
    S = z @ z.conj().transpose(0, 2, 1)
    d = 1 / np.sqrt(np.einsum("pii->pi", S).real)
    C = S * d[:, :, None] * d[:, None, :]
    i, k = np.triu_indices(N)
    C32 = C[:, i, k].astype(np.complex64)
    C32[:, i == k] = 1
    if N > 2:
        C32[5, 1] = 0  # an exactly-zero C_ik counts as phase 0
    r = plk.Context("cuda:0").phase_link(torch.from_numpy(np.ascontiguousarray(C32)).cuda(), N, ref)
    phase, tcoh = r["phase"].cpu().numpy().astype(np.float64), r["tcoh"].cpu().numpy()
    off = i != k
    u = np.where(C32 != 0, C32 / np.maximum(np.abs(C32), 1e-30), 1).astype(np.complex128)[:, off]
    dphi = phase[k[off]] - phase[i[off]]
    want = np.abs((u * np.exp(1j * dphi.T)).mean(1))
    # mean of at most 496 unit terms, each to a few 2^-24 in its phase and modulus
    np.testing.assert_allclose(tcoh, want, rtol=0, atol=3e-6)
