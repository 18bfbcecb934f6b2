"""Coherences and samples that are not finite, or whose squares are not: such a
pixel is not reported as solved, and has no gradient or uncertainty that looks
like one."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SOLVED = (0, 1)   # PLK_PX_EMI, PLK_PX_EMI_FP64
# every row length filled and not
NS = [8, 16, 20, 24, 28, 32, 7, 15, 18, 23, 27, 31]


@pytest.fixture(scope="module")
def plk():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2511_12051_gb300 import build, plk as _plk
    build.build()
    return _plk


def coherences(N, P=40):
    rng = np.random.default_rng(N)
    z = rng.standard_normal((P, N, 60)) + 1j * rng.standard_normal((P, N, 60))
    z = z + 1.2 * (rng.standard_normal((P, 1, 60)) + 1j * rng.standard_normal((P, 1, 60)))
    S = z @ z.conj().transpose(0, 2, 1)
    d = 1 / np.sqrt(np.einsum("pii->pi", S).real)
    i, k = np.triu_indices(N)
    C = (S * d[:, :, None] * d[:, None, :])[:, i, k].astype(np.complex64)
    C[:, i == k] = 1
    return np.ascontiguousarray(C)


def link(plk, C, N, fp64_resolve):
    r = plk.Context("cuda:0").phase_link(torch.from_numpy(C).cuda(), N, 0, plk.default_params(fp64_resolve=fp64_resolve))
    return r["status"].cpu().numpy(), r["phase"].cpu().numpy()


@pytest.mark.parametrize("fp64_resolve", [1, 0])
@pytest.mark.parametrize("N", NS)
def test_coherence_beyond_range(plk, N, fp64_resolve):
    C = coherences(N)
    want = link(plk, C, N, fp64_resolve)
    C[1::2, 3] = 1e30   # |c|^2 is infinite in single precision
    st, ph = link(plk, C, N, fp64_resolve)
    assert not np.isin(st[1::2], SOLVED).any()
    # the other pixels of the same warps are left as they are
    np.testing.assert_array_equal(st[::2], want[0][::2])
    np.testing.assert_array_equal(ph[:, ::2], want[1][:, ::2])


@pytest.mark.parametrize("fp64_resolve", [1, 0])
@pytest.mark.parametrize("N", NS)
def test_coherence_not_a_number(plk, N, fp64_resolve):
    C = coherences(N)
    C[1::2, 3] = np.nan
    assert not np.isin(link(plk, C, N, fp64_resolve)[0][1::2], SOLVED).any()


@pytest.mark.parametrize("N,groups", [(8, 2), (9, 3), (16, 4), (16, 8), (20, 4), (24, 4), (24, 8), (32, 8)])
def test_undetermined_phases_are_not_certain(plk, N, groups):
    # Groups of dates, each coherent within itself at a look of its own: C's
    # largest eigenvalue is `groups`-fold, and the phases of the other groups
    # against the reference's have no derivative.
    m, pixels = N // groups, 64
    gen = torch.Generator().manual_seed(N)
    z = torch.zeros((N, 5, 11 * pixels), dtype=torch.complex64)
    for t in range(pixels):
        v = torch.full((N,), 2.0 ** (t % 5), dtype=torch.complex64)
        if t >= 32:
            v = v * torch.polar(torch.ones(N), torch.randint(0, 4, (N,), generator=gen) * (np.pi / 2))
        for k in range(groups):
            z[k * m:(k + 1) * m, k % 5, 11 * t + k] = v[k * m:(k + 1) * m]
    mask = torch.full((1, pixels, 1), (1 << 55) - 1, dtype=torch.int64).cuda()
    sd = plk.Context("cuda:0").phase_uncertainty(z.cuda(), (5, 11, 5, 11), mask, 0, 0.1).cpu()[:, 0]
    # 0.4 at most within the group
    assert not sd[0].any() and not (sd[m:] < 100).any()


@pytest.mark.parametrize("N", [2, 4, 8, 15, 16, 20, 28, 32])
def test_power_beyond_range_gives_no_gradient(plk, N):
    # |z|^2 is infinite in the middle window: its pixel has data, but no coherence.
    ctx, win = plk.Context("cuda:0"), (5, 11, 5, 11)
    gen = torch.Generator().manual_seed(N)
    z = torch.randn((N, 5, 33), dtype=torch.complex64, generator=gen) + torch.randn((5, 33), dtype=torch.complex64, generator=gen)
    z[:, :, 11:22] *= 1e20
    mask = torch.full((1, 3, 1), (1 << 55) - 1, dtype=torch.int64).cuda()
    w = torch.randn((N, 1, 3), generator=gen).cuda()
    bad = torch.zeros(33, dtype=torch.bool)
    bad[11:22] = True
    g = ctx.phase_link_backward(z.cuda(), win, mask, 0, w).cpu()
    assert g[:, :, bad].isnan().all() and g[:, :, ~bad].isfinite().all() and (g[:, :, ~bad] != 0).all()
    dw = ctx.shp_weight_gradient(z.cuda(), win, mask, 0, w).cpu()[0]
    assert dw[1].isnan().all() and dw[[0, 2]].isfinite().all()
    sd = ctx.phase_uncertainty(z.cuda(), win, mask, 0, 0.1).cpu()[:, 0]
    assert sd[1:, 1].isnan().all() and sd[:, [0, 2]].isfinite().all() and (sd[1:, [0, 2]] > 0).all()
