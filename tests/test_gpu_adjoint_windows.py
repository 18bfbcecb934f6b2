"""The gradient of the linked phases over windows from 3 x 3 to 31 x 31 (masks of
one and of several words, every share of a tile between warps, and a window too
large for a tile) against 64-bit automatic differentiation in plain torch."""
import pytest
import torch

from paper_2511_12051_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2511_12051_gb300 import build, plk
    build.build()
    return plk.Context("cuda:0")


def neighbours(H, W, win):
    """Flat indices [P, L] of every output pixel's looks and whether they lie inside."""
    wy, wx, sy, sx = win
    y = (torch.arange(H // sy) * sy + sy // 2)[:, None] + torch.arange(wy) - wy // 2
    x = (torch.arange(W // sx) * sx + sx // 2)[:, None] + torch.arange(wx) - wx // 2
    inside = ((y >= 0) & (y < H))[:, None, :, None] & ((x >= 0) & (x < W))[None, :, None, :]
    at = y.clamp(0, H - 1)[:, None, :, None] * W + x.clamp(0, W - 1)[None, :, None, :]
    return at.reshape(-1, wy * wx), inside.reshape(-1, wy * wx)


def words(sel):
    out = torch.zeros((sel.shape[0], (sel.shape[1] + 63) // 64), dtype=torch.int64)
    for b in range(sel.shape[1]):
        one = (1 << (b % 64)) if b % 64 < 63 else -(1 << 63)
        out[:, b // 64] |= torch.where(sel[:, b], one, 0)
    return out


def case(N, H, W, win):
    gen = torch.Generator().manual_seed(N * win[0])
    z = synth.generate(synth.config_spec(4, N=N, H=H, W=W, seed=11 + N))
    at, inside = neighbours(H, W, win)
    sel = inside & (torch.rand(at.shape, generator=gen) < 0.85)
    w = torch.randn((N, at.shape[0]), generator=gen)
    return z, at, sel, w


def gradient64(z, at, sel, w, ref):
    """Gradient [N, H*W] of sum w phase, and the weights used: 0 where a
    single-precision solve is not expected to give the gradient to 2e-3, i.e.
    cond(|C|) 6e-8 / gap is above that or |C|'s inversion is near its limit."""
    N = z.shape[0]
    Z = z.reshape(N, -1).to(torch.complex128)[:, at].movedim(0, 1).requires_grad_(True)
    S = (Z * sel[:, None]) @ Z.mH
    s = S.diagonal(dim1=-2, dim2=-1).real.rsqrt()
    eye = torch.eye(N, dtype=torch.bool)
    C = torch.where(eye, torch.ones((), dtype=S.dtype), S * s[:, :, None] * s[:, None, :])
    G = C.abs()
    root, info = torch.linalg.cholesky_ex(G.detach())
    pivot = root.diagonal(dim1=-2, dim2=-1).square().amin(-1)
    bad = (info > 0) | (pivot <= 1e-4)
    unsure = (info == 0) & (pivot > 5e-5) & (pivot < 2e-4)
    inv = torch.linalg.inv(torch.where(bad[:, None, None], eye.to(G.dtype), G))
    lam, V = torch.linalg.eigh(torch.where(bad[:, None, None], -C, inv * C))
    v = V[..., 0]
    phase = torch.angle(v * v[:, ref, None].conj())
    cond = torch.where(bad, 1.0, torch.linalg.cond(G.detach()))
    ok = ~unsure & (cond * 6e-8 < 2e-3 * (lam[:, 1] - lam[:, 0]).detach())
    w = w * ok
    (g,) = torch.autograd.grad((phase * w.T.double()).sum(), Z)
    grad = torch.zeros((N, z[0].numel()), dtype=torch.complex128)
    for i in range(N):
        grad[i].index_add_(0, at.reshape(-1), g[:, i].reshape(-1))
    return grad, w, ok


@pytest.mark.parametrize("N,win,H,W", [
    (2, (3, 3, 1, 1), 30, 50), (9, (3, 3, 1, 1), 17, 23), (5, (1, 55, 1, 1), 20, 70),   # up to one word
    (4, (9, 11, 1, 1), 21, 33), (15, (9, 11, 1, 1), 21, 20), (32, (9, 11, 1, 1), 12, 17),
    (3, (15, 15, 2, 3), 40, 41), (20, (15, 15, 2, 3), 30, 31),
    (8, (13, 25, 1, 1), 20, 31), (16, (13, 25, 3, 6), 40, 60),
    (2, (31, 31, 5, 6), 50, 60), (7, (31, 31, 5, 6), 40, 48), (6, (19, 39, 3, 6), 40, 60),
    (32, (19, 25, 3, 5), 27, 35),   # no tile fits
])
def test_gradient(ctx, N, win, H, W):
    ref = N // 2
    z, at, sel, w = case(N, H, W, win)
    want, w, ok = gradient64(z, at, sel, w, ref)
    assert ok.float().mean() > 0.5
    Ho, Wo = H // win[2], W // win[3]
    g = ctx.phase_link_backward(z.cuda(), win, words(sel).reshape(Ho, Wo, -1).cuda(), ref,
                                w.reshape(N, Ho, Wo).contiguous().cuda()).cpu().reshape(N, -1)
    assert (g - want).norm() < 2e-3 * want.norm()
    assert ((g - want).abs().amax(0) < 1e-2 * want.abs().max()).all()
