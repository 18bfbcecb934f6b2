"""The adjoint of a pixel with a single accepted look (an isolated persistent
scatterer), at odd and even date counts of every row length.  C is rank one and
not invertible, so its own largest eigenvector carries the phases: phihat_i =
arg z_i - arg z_ref, with closed forms for the gradient and the uncertainty."""
import pytest
import torch

from paper_2511_12051_gb300 import synth

pytestmark = pytest.mark.gpu

WIN, CENTRE = (5, 11, 5, 11), 27
NS = [2, 3, 4, 6, 8, 10, 12, 15, 16, 18, 20, 22, 24, 27, 28, 30, 32]
# The deflated matrix is -N times the identity but for rounding: a few rounding
# errors a step over at most 32 steps, 32 x 4 x 6e-8 = 8e-6 of the result.
RTOL = 2e-5


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2511_12051_gb300 import build, plk
    build.build()
    return plk.Context("cuda:0")


def stack(N):
    z = synth.generate(synth.config_spec(4, N=N, H=10, W=33, seed=40 + N))
    mask = torch.full((2, 3, 1), 1 << CENTRE, dtype=torch.int64).cuda()
    return z, mask, z[:, 2::5, 5::11].to(torch.complex128)


@pytest.mark.parametrize("N", NS)
def test_uncertainty(ctx, N):
    ref, sigma2 = N // 2, 0.3
    z, mask, look = stack(N)
    sd = ctx.phase_uncertainty(z.cuda(), WIN, mask, ref, sigma2).cpu().double()
    p = look.abs().square()
    want = torch.sqrt(0.5 * sigma2 * (1 / p + 1 / p[ref]))
    want[ref] = 0.0
    torch.testing.assert_close(sd, want, rtol=RTOL, atol=0.0)


@pytest.mark.parametrize("N", NS)
def test_gradient(ctx, N):
    # d phihat_i = Im(conj(z_i) dz_i) / |z_i|^2 - (the same of ref)
    ref = N // 2
    z, mask, look = stack(N)
    w = torch.randn((N, 2, 3), generator=torch.Generator().manual_seed(N))
    g = ctx.phase_link_backward(z.cuda(), WIN, mask, ref, w.cuda()).cpu().to(torch.complex128)
    w = w.double()
    w[ref] = 0.0
    w[ref] = -w.sum(0)
    want = 1j * w * look / look.abs().square()
    # g_i sums N terms of up to max |w| / |z_i| each
    off = ((g[:, 2::5, 5::11] - want).abs() * look.abs()).amax(0) / w.abs().amax(0)
    assert off.max() < RTOL
    g[:, 2::5, 5::11] = 0
    assert not g.any()  # no other sample is a look
