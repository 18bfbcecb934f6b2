"""The adjoint kernels at the edges of their row lengths (8, 16, 20, 24, 28 and
32 entries): phase uncertainty and the gradient of the linked phases against
64-bit automatic differentiation (plain torch) on tiling windows, odd and even
date counts, regularised and not, and the closed form of a single look."""
import numpy as np
import pytest
import torch

from paper_2511_12051_gb300 import synth

pytestmark = pytest.mark.gpu

WIN = (5, 11, 5, 11)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2511_12051_gb300 import build, plk
    build.build()
    return plk.Context("cuda:0")


def windows(z):
    """[P, N, 55] complex128 samples of the tiling windows."""
    N, H, W = z.shape
    v = z.reshape(N, H // 5, 5, W // 11, 11).permute(1, 3, 0, 2, 4)
    return v.reshape(-1, N, 55).to(torch.complex128)


def phases64(Z, ref, beta):
    S = Z @ Z.mH
    s = S.diagonal(dim1=-2, dim2=-1).real.rsqrt()
    C = S * s[:, :, None] * s[:, None, :]
    eye = torch.eye(Z.shape[1], dtype=torch.float64)
    G = (1 - beta) * torch.where(eye.bool(), eye, C.abs()) + beta * eye
    lam, V = torch.linalg.eigh(torch.linalg.inv(G) * C)
    v = V[..., 0]
    return torch.angle(v * v[:, ref, None].conj()), lam[:, 1] - lam[:, 0]


@pytest.mark.parametrize("N,beta", [(2, 0.0), (7, 0.0), (8, 0.0), (9, 0.2), (15, 0.0), (16, 0.0), (17, 0.0), (20, 0.3),
                                    (21, 0.0), (24, 0.0), (25, 0.0), (28, 0.1), (29, 0.0), (32, 0.0)])
def test_rows_match_64_bit_autograd(ctx, N, beta):
    from paper_2511_12051_gb300 import plk
    ref, H, W, sigma2 = N // 2, 10, 33, 0.02
    z = synth.generate(synth.config_spec(4, N=N, H=H, W=W, seed=90 + N))
    prm = plk.default_params(beta=beta)
    mask = torch.full((H // 5, W // 11, 1), (1 << 55) - 1, dtype=torch.int64).cuda()
    sd = ctx.phase_uncertainty(z.cuda(), WIN, mask, ref, sigma2, prm).cpu().double().reshape(N, -1)
    w = torch.randn((N, H // 5, W // 11), generator=torch.Generator().manual_seed(N))
    g = ctx.phase_link_backward(z.cuda(), WIN, mask, ref, w.cuda(), prm).cpu()

    Z = windows(z).requires_grad_(True)
    phase, gap = phases64(Z, ref, beta)
    ok = (gap > 1e-2) & (phase.abs().amax(1) < np.pi - 1e-3)  # unique eigenvector, away from the wrap
    assert ok.sum() >= 3
    want_sd = torch.zeros(N, Z.shape[0], dtype=torch.float64)
    for i in range(N):
        if i != ref:
            (gi,) = torch.autograd.grad(phase[:, i].sum(), Z, retain_graph=True)
            want_sd[i] = torch.sqrt(0.5 * sigma2 * gi.abs().square().sum((1, 2)))
    (want_g,) = torch.autograd.grad((phase * w.reshape(N, -1).T).sum(), Z)
    # A single-precision solve: cond(G) eps / gap of up to about 300 x 6e-8 / 0.01
    # = 2e-3 in a gradient's relative error (the bar of the oracle comparison
    # is 1e-2).
    rel_sd = ((sd - want_sd).abs() / (want_sd + 1e-30))[:, ok]
    assert torch.all(sd[ref] == 0.0)
    others = [i for i in range(N) if i != ref]
    assert rel_sd[others].max() < 5e-3
    dg = (windows(g) - want_g).abs().square().sum((1, 2)).sqrt() / want_g.abs().square().sum((1, 2)).sqrt()
    assert dg[ok].max() < 5e-3


@pytest.mark.parametrize("N", [13, 19, 27])
def test_single_look_closed_form(ctx, N):
    # One look: C is rank one (eigenvector of C itself), phihat_i = arg z_i -
    # arg z_ref, so Var = (sigma2 / 2) (1 / |z_i|^2 + 1 / |z_ref|^2).
    ref, H, W, sigma2 = 1, 5, 22, 0.3
    z = synth.generate(synth.config_spec(4, N=N, H=H, W=W, seed=7 + N))
    mask = torch.full((1, 2, 1), 1 << 27, dtype=torch.int64).cuda()  # the centre look
    sd = ctx.phase_uncertainty(z.cuda(), WIN, mask, ref, sigma2).cpu().double()[:, 0]
    p = z[:, 2, [5, 16]].abs().double().square()
    want = torch.sqrt(0.5 * sigma2 * (1 / p + 1 / p[ref]))
    want[ref] = 0.0
    torch.testing.assert_close(sd, want, rtol=1e-4, atol=0.0)
