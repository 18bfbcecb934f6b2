"""|C| whose elimination first meets a pivot just above the limit of 1e-4 and
then one far below it: the inversion fails and C's own largest eigenvector
carries the phases, also where nothing is solved again in double precision
(fp64_resolve = 0, the adjoint family)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_12051_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plk():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2511_12051_gb300 import build, plk as _plk
    build.build()
    return _plk


def pivots(G):
    A, out = G.copy(), []
    with np.errstate(all="ignore"):
        for s in range(G.shape[-1]):
            out.append(A[:, s, s].copy())
            A = A - A[:, :, s, None] * A[:, None, s, :] / np.maximum(out[-1], 1e-30)[:, None, None]
    return np.array(out).T


@pytest.mark.parametrize("fp64_resolve", [1, 0])
@pytest.mark.parametrize("first", [0, -3])   # pivots follow the failing one, or none does
@pytest.mark.parametrize("N", [3, 7, 8, 15, 16, 18, 20, 24, 27, 28, 32])
def test_linked_phases(plk, N, first, fp64_resolve):
    rng = np.random.default_rng(N)
    P, a = 24, first % N
    m = np.full((P, N, N), 0.05)
    for i, k, v in ((0, 1, np.sqrt(1 - 1.1e-4)), (0, 2, 0.5), (1, 2, 0.3)):
        m[:, a + i, a + k] = v
    phi = rng.uniform(-1, 1, (P, N, N))
    i, k = np.triu_indices(N)
    C = (m * np.exp(1j * phi))[:, i, k].astype(np.complex64)
    C[:, i == k] = 1
    F = np.zeros((P, N, N), complex)
    F[:, i, k] = C
    F[:, k, i] = C.conj()
    piv = pivots(np.abs(F))
    piv[:, :a + 1] = 1
    assert np.all((piv[:, a + 1] > 1.02e-4) & (piv[:, a + 1] < 1.18e-4) & (piv[:, a + 2] < -10))
    lam, V = np.linalg.eigh(F)
    v = V[:, :, -1]
    want = np.angle(v * v[:, a, None].conj()).T
    r = plk.Context("cuda:0").phase_link(torch.from_numpy(np.ascontiguousarray(C)).cuda(), N, a,
                                         plk.default_params(fp64_resolve=fp64_resolve))
    assert np.all(r["status"].cpu().numpy() == 2)
    # entries whose phase a unit vector's rounding leaves alone: the block's, and others not near 0
    ok = (np.abs(v) > 1e-2).T & (lam[:, -1] - lam[:, -2] > 0.2)
    assert ok[a:a + 3].mean() > 0.5
    d = np.angle(np.exp(1j * (r["phase"].cpu().numpy() - want)))[ok]
    assert np.abs(d).max() <= 1e-4


@pytest.mark.parametrize("N", [12, 15, 16])
def test_adjoint(plk, N):
    win, H, W, sigma2, ref = (5, 11, 3, 6), 180, 360, 0.01, 0
    z = synth.generate(synth.config_spec(1, N=N, H=H, W=W, seed=3 + N))
    P, _ = oracle.amp_stats(z.numpy())
    mask, _ = oracle.shp_select(P, win, np.float32(oracle.glrt_threshold(1e-3, N)))
    C = oracle.covariance(z.numpy(), win, mask).reshape(-1, N * (N + 1) // 2)
    i, k = np.triu_indices(N)
    F = np.zeros((len(C), N, N), complex)
    F[:, i, k] = C
    F[:, k, i] = C.conj()
    F[:, range(N), range(N)] = 1
    piv = pivots(np.abs(F))
    low = piv <= 1.2e-4
    at = low.argmax(1)
    px = np.flatnonzero(low.any(1) & (piv[np.arange(len(piv)), at] > 1.01e-4) & ~(np.nanmin(piv, 1) > 5e-5))
    assert len(px)
    Ho, Wo = H // 3, W // 6
    dy, dx = np.divmod(np.arange(55), 11)
    y, x = (px // Wo * 3 + 1)[:, None] + dy - 2, (px % Wo * 6 + 3)[:, None] + dx - 5
    bits = (mask.reshape(-1, 1)[px].view(np.uint64) >> np.arange(55, dtype=np.uint64)) & np.uint64(1)
    inside = (y >= 0) & (y < H) & (x >= 0) & (x < W)
    flat = torch.from_numpy(np.where(inside, y * W + x, 0))
    Z = z.reshape(N, -1).to(torch.complex128)[:, flat].movedim(0, 1).requires_grad_(True)
    S = (Z * torch.from_numpy((bits.astype(bool) & inside)[:, None])) @ Z.mH
    s = S.diagonal(dim1=-2, dim2=-1).real.rsqrt()
    v = torch.linalg.eigh(S * s[:, :, None] * s[:, None, :])[1][..., -1]
    phase = torch.angle(v * v[:, ref, None].conj())
    w = torch.randn((N, len(px)), generator=torch.Generator().manual_seed(N))
    g = torch.autograd.grad((phase * w.T.double()).sum(), Z, retain_graph=True)[0]
    want = torch.zeros((N, H * W), dtype=torch.complex128)
    for d in range(N):
        want[d].index_add_(0, flat.reshape(-1), g[:, d].reshape(-1))
    want_sd = torch.zeros((N, len(px)), dtype=torch.float64)
    for d in range(1, N):
        gi = torch.autograd.grad(phase[:, d].sum(), Z, retain_graph=True)[0]
        want_sd[d] = torch.sqrt(0.5 * sigma2 * gi.abs().square().sum((1, 2)))
    ctx, mk = plk.Context("cuda:0"), torch.from_numpy(mask.view(np.int64)).cuda()
    wfull = torch.zeros((N, Ho * Wo))
    wfull[:, px] = w
    got = ctx.phase_link_backward(z.cuda(), win, mk, ref, wfull.reshape(N, Ho, Wo).cuda()).cpu().reshape(N, -1)
    sd = ctx.phase_uncertainty(z.cuda(), win, mk, ref, sigma2).cpu().reshape(N, -1)[:, px].double()
    # a definite matrix of eigenvalues within [-N, 0) some tenths below 0: a
    # hundred single-precision rounding errors
    assert (got - want).norm() < 1e-4 * want.norm()
    torch.testing.assert_close(sd, want_sd, rtol=1e-4, atol=0.0)
