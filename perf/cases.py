"""Workloads of sequential phase linking, for timing and comparing builds.

Each case is one call (or one short sequence of calls) that a program using
this package makes: a mini-stack step, a chain of steps, a batch of uneven
stacks, the single stages (coherence, phase linking), the adjoint family, the
phase similarity and the L1 network inversion.  Inputs are drawn from a seed,
on the GPU, with the value distributions of the burst-shaped stacks of
`paper_2511_12051_gb300.synth`; `exact` recomputes a case in 64 bits with plain
torch and none of the package's arithmetic.
"""
from __future__ import annotations

import math

import torch

from paper_2511_12051_gb300 import plk

ALPHA = 1e-3           # GLRT size, the library's default
PIVOT_FAIL = 1e-4      # |C| counts as not invertible at or below this pivot
DT = 12.0              # days between acquisitions
ACCEPTED = 0.87        # share of a window's looks that the GLRT keeps
BURST = dict(wy=5, wx=11, sy=3, sx=6)   # 11 x 5 window, strides 6 x 3
DENSE = dict(wy=5, wx=11, sy=1, sx=1)   # 11 x 5 window, stride 1


def listed():
    return [
        # The smallest stack in use: one mini-stack of 128 x 128, launch- and latency-bound.
        dict(name="step_small", kind="step", N=10, H=128, W=128, **DENSE, tau_lo=48.0, tau_hi=48.0, ps=0.0),
        # The full burst at the production posting.
        dict(name="step_burst", kind="step", N=15, H=4096, W=16384, **BURST, tau_lo=12.0, tau_hi=120.0, ps=0.05),
        # An archive processed mini-stack by mini-stack at full resolution: later
        # steps carry compressed SLCs (N = 15, 16, 17).
        dict(name="chain", kind="chain", steps=3, M=15, H=512, W=1024, K=3, **DENSE, tau_lo=48.0, tau_hi=48.0, ps=0.0),
        # Many independent stacks of uneven length in one recorded batch.
        dict(name="batch_uneven", kind="batch", stacks=12, n_lo=5, n_hi=30, H=509, W=1031, **BURST,
             tau_lo=48.0, tau_hi=48.0, ps=0.0),
        # Single-precision coherence alone, ragged image sides.
        dict(name="cov_fp32", kind="cov", N=15, H=1021, W=4093, precision=0, **BURST, tau_lo=12.0, tau_hi=120.0,
             ps=0.05),
        # The bfloat16 coherence mode.
        dict(name="cov_bf16", kind="cov", N=15, H=2047, W=4095, precision=1, **BURST, tau_lo=12.0, tau_hi=120.0,
             ps=0.05),
        # EMI phase linking alone, the burst's stack length, and a long stack.
        dict(name="link_n15", kind="link", N=15, npx=250_007, ref=0),
        dict(name="link_n28", kind="link", N=28, npx=65_521, ref=3),
        # The adjoint: gradient of the linked phases in the samples (training and
        # inversion), and their uncertainty.
        dict(name="backward_n20", kind="backward", N=20, H=301, W=403, **DENSE, tau_lo=48.0, tau_hi=48.0, ps=0.0,
             ref=0),
        dict(name="uncertainty_n20", kind="uncertainty", N=20, H=201, W=301, **DENSE, tau_lo=48.0, tau_hi=48.0,
             ps=0.0, ref=0),
        # Post-processing of a burst's output grid: phase cosine similarity (~200 m)
        # and the L1 inversion of the nearest-3 network.
        dict(name="similarity", kind="similarity", M=15, Ho=683, Wo=1365, radius=7),
        dict(name="invert_l1", kind="l1", dates=15, npx=932_113, iters=50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "chain", "batch", "cov", "cov", "link", "link", "backward", "uncertainty",
                       "wgrad", "similarity", "l1"])
    win = dict(rng.choice([BURST, DENSE]))
    dense = win["sy"] == 1
    lo, hi = rng.choice([(48.0, 48.0), (12.0, 120.0)])
    stack = dict(**win, tau_lo=lo, tau_hi=hi, ps=rng.choice([0.0, 0.05]))
    if kind == "link":
        N = rng.randint(4, 32)
        return dict(kind=kind, N=N, npx=_log(rng, 1000, 300_000 if N <= 16 else 80_000), ref=rng.randrange(N))
    if kind == "similarity":
        return dict(kind=kind, M=rng.randint(3, 30), Ho=_log(rng, 40, 900), Wo=_log(rng, 40, 1400),
                    radius=rng.randint(2, 9))
    if kind == "l1":
        return dict(kind=kind, dates=rng.randint(4, 17), npx=_log(rng, 2000, 1_000_000), iters=rng.choice([20, 50]))
    if kind in ("backward", "uncertainty", "wgrad"):
        N = rng.randint(6, 30)
        side = 320 if dense else 700
        return dict(kind=kind, N=N, H=_log(rng, 40, side), W=_log(rng, 60, side), ref=rng.randrange(N), **stack)
    # images: up to 4 M samples a date at the burst posting, 0.4 M at full resolution
    H = _log(rng, 64, 400 if dense else 1500)
    W = _log(rng, 64, 1000 if dense else 2700)
    if kind == "cov":
        return dict(kind=kind, N=rng.randint(4, 32), H=H, W=W, precision=rng.choice([0, 0, 1, 2]), **stack)
    if kind == "chain":
        return dict(kind=kind, steps=rng.randint(2, 4), M=rng.randint(6, 16), H=H, W=W, K=rng.randint(1, 6),
                    last=rng.choice([False, True]), regrid=rng.choice([0.0, 0.2]), **stack)
    if kind == "batch":
        return dict(kind=kind, stacks=rng.randint(3, 12), n_lo=5, n_hi=30, H=min(H, 512), W=min(W, 1024), **stack)
    return dict(kind="step", N=rng.randint(5, 30), H=H, W=W, precision=rng.choice([0, 0, 1, 2]),
                regrid=rng.choice([0.0, 0.2]), **stack)


# ------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _stack(case, N, H, W, gen, first_date=0, rho0=0.7, rho_inf=0.1, patches=0.0):
    """z [N, H, W]: circular Gaussian samples whose coherence decays as
    rho_inf + (rho0 - rho_inf) exp(-dt / tau), a phase ramp, a share of
    persistent scatterers, and patches of nearly singular coherence."""
    out = torch.empty((N, H, W), dtype=torch.complex64, device="cuda")
    near = torch.zeros((H, W), dtype=torch.bool, device="cuda")
    if patches:
        side = 32
        n = max(1, round(patches * H * W / side ** 2))
        ys = torch.randint(0, max(1, H - side), (n,), generator=gen, device="cuda").tolist()
        xs = torch.randint(0, max(1, W - side), (n,), generator=gen, device="cuda").tolist()
        for y, x in zip(ys, xs):
            near[y:y + side, x:x + side] = True

    def cn(h):
        return torch.randn((h, W), dtype=torch.complex64, generator=gen, device="cuda")

    for r0 in range(0, H, 1024):
        r1 = min(H, r0 + 1024)
        h = r1 - r0
        tau = case["tau_lo"] + (case["tau_hi"] - case["tau_lo"]) * torch.rand((h, W), generator=gen, device="cuda")
        r = torch.exp(-DT / tau)
        ar = torch.sqrt(1 - r * r)
        hot = near[r0:r1]
        s_c = torch.where(hot, 0.98, rho_inf).sqrt()
        s_a = torch.where(hot, 0.0, rho0 - rho_inf).sqrt()
        s_n = torch.where(hot, 0.02, 1 - rho0).sqrt()
        c, a = s_c * cn(h), cn(h)
        ps = torch.rand((h, W), generator=gen, device="cuda") < case["ps"]
        for i in range(N):
            if i:
                a = r * a + ar * cn(h)
            z = c + s_a * a + s_n * cn(h)
            if case["ps"]:
                z = torch.where(ps, 3.0 * (1 + 0.1 * cn(h)), z)
            phi = 0.05 * (first_date + i)
            out[i, r0:r1] = z * complex(math.cos(phi), math.sin(phi))
    return out


def _threshold(n):
    """c = F^-1_{2n,2n}(1 - alpha / 2): P(F <= c) = I_{c/(1+c)}(n, n), a binomial sum."""
    def cdf(c):
        x = c / (1 + c)
        return sum(math.comb(2 * n - 1, j) * x ** j * (1 - x) ** (2 * n - 1 - j) for j in range(n, 2 * n))
    lo, hi = 1.0, 1e9
    for _ in range(200):
        mid = math.sqrt(lo * hi)
        lo, hi = (mid, hi) if cdf(mid) < 1 - ALPHA / 2 else (lo, mid)
    return lo


def _window(case):
    return case["wy"], case["wx"], case["sy"], case["sx"]


def _neighbours(case, image):
    """[Ho, Wo, wy*wx] values of `image` in each output pixel's window, and
    whether the neighbour lies inside the image."""
    wy, wx, sy, sx = _window(case)
    H, W = image.shape
    Ho, Wo = H // sy, W // sx
    dev = image.device
    dy = torch.arange(wy, device=dev) - wy // 2
    dx = torch.arange(wx, device=dev) - wx // 2
    y = (torch.arange(Ho, device=dev) * sy + sy // 2)[:, None] + dy
    x = (torch.arange(Wo, device=dev) * sx + sx // 2)[:, None] + dx
    inside = ((y >= 0) & (y < H))[:, None, :, None] & ((x >= 0) & (x < W))[None, :, None, :]
    v = image[y.clamp(0, H - 1)[:, None, :, None], x.clamp(0, W - 1)[None, :, None, :]]
    return v.reshape(Ho, Wo, wy * wx), inside.reshape(Ho, Wo, wy * wx)


def _select(case, z):
    """SHP selection [Ho, Wo, wy*wx] (bool): two pixels' power sums over the
    dates pass the GLRT, in single precision and date order."""
    power = torch.zeros(z.shape[1:], dtype=torch.float32, device=z.device)
    for zi in z:
        power += zi.real * zi.real + zi.imag * zi.imag
    q, inside = _neighbours(case, power)
    p = q[..., q.shape[-1] // 2, None]
    c = torch.tensor(_threshold(z.shape[0]), dtype=torch.float32, device=z.device)
    return inside & (p > 0) & (q > 0) & (torch.maximum(p, q) <= c * torch.minimum(p, q))


def _mask_words(sel):
    """The selection as the library's mask: bit b of word b // 64."""
    Ho, Wo, L = sel.shape
    words = (L + 63) // 64
    out = torch.zeros((Ho, Wo, words), dtype=torch.int64, device=sel.device)
    for b in range(L):
        one = (1 << (b % 64)) if b % 64 < 63 else -(1 << 63)
        out[..., b // 64] |= torch.where(sel[..., b], one, 0)
    return out


def _coherences(case, seed):
    """Packed sample coherences [npx, N(N+1)/2] of independent pixels: 20 to 55
    looks each, decay times of 12 to 120 days, some pixels nearly singular
    and some dominated by a point target."""
    N, npx, gen = case["N"], case["npx"], _gen(seed)
    iu = torch.triu_indices(N, N, device="cuda")
    t = DT * torch.arange(N, device="cuda", dtype=torch.float32)
    lag = (t[:, None] - t[None, :]).abs()
    ramp = torch.polar(torch.ones(N, device="cuda"), 0.05 * torch.arange(N, device="cuda"))
    out = torch.empty((npx, iu.shape[1]), dtype=torch.complex64, device="cuda")
    for p0 in range(0, npx, 32768):
        P = min(32768, npx - p0)
        tau = 12.0 + 108.0 * torch.rand((P, 1, 1), generator=gen, device="cuda")
        gamma = 0.1 + 0.6 * torch.exp(-lag / tau)
        hot = torch.rand((P, 1, 1), generator=gen, device="cuda") < 0.01
        gamma = torch.where(hot, 0.98, gamma)
        gamma = torch.where(torch.eye(N, dtype=torch.bool, device="cuda"), 1.0, gamma)
        root = torch.linalg.cholesky(gamma).to(torch.complex64)
        z = root @ torch.randn((P, N, 55), dtype=torch.complex64, generator=gen, device="cuda")
        looks = torch.randint(20, 56, (P, 1, 1), generator=gen, device="cuda")
        z = z * (torch.arange(55, device="cuda") < looks)
        target = torch.rand((P,), generator=gen, device="cuda") < 0.02
        eps = torch.randn((P, N), dtype=torch.complex64, generator=gen, device="cuda")
        z[:, :, 0] = torch.where(target[:, None], 30.0 * (1 + 0.03 * eps), z[:, :, 0])
        z = z * ramp[:, None]
        S = z @ z.mH
        d = S.diagonal(dim1=1, dim2=2).real.rsqrt()
        C = S * (d[:, :, None] * d[:, None, :])
        C.diagonal(dim1=1, dim2=2).fill_(1.0)
        out[p0:p0 + P] = C[:, iu[0], iu[1]]
    return out


def _pairs(dates):
    return [(a, a + d) for a in range(dates) for d in (1, 2, 3) if a + d < dates]


def _unwrapped(case, seed):
    """Interferograms of random phase series, 2% of them off by 2 pi, with noise."""
    gen, pairs = _gen(seed), _pairs(case["dates"])
    x = torch.randn((case["dates"], case["npx"]), generator=gen, device="cuda").cumsum(0)
    b = torch.stack([x[j] - x[i] for i, j in pairs])
    jump = torch.rand(b.shape, generator=gen, device="cuda") < 0.02
    return b + 2 * math.pi * jump + 0.05 * torch.randn(b.shape, generator=gen, device="cuda")


def _phases(case, seed):
    """Linked phases [M, Ho, Wo]: a smooth history with noise, some no-data cells."""
    gen, M, Ho, Wo = _gen(seed), case["M"], case["Ho"], case["Wo"]
    y = torch.linspace(0, 6, Ho, device="cuda")[:, None]
    x = torch.linspace(0, 9, Wo, device="cuda")[None, :]
    t = torch.arange(M, device="cuda", dtype=torch.float32)[:, None, None]
    noise = 0.2 + 0.8 * torch.rand((Ho, Wo), generator=gen, device="cuda")
    phi = 0.1 * t * torch.sin(y + x) + noise * torch.randn((M, Ho, Wo), generator=gen, device="cuda")
    phi = torch.remainder(phi + math.pi, 2 * math.pi) - math.pi
    phi[:, torch.rand((Ho, Wo), generator=gen, device="cuda") < 0.002] = float("nan")
    return phi.contiguous()


def _batch_lengths(case, seed):
    g = torch.Generator()
    g.manual_seed(20 + case["stacks"])  # the lengths belong to the case, the samples to the seed
    return torch.randint(case["n_lo"], case["n_hi"] + 1, (case["stacks"],), generator=g).tolist()


def _batch_stacks(case, seed):
    gen = _gen(seed)
    return [_stack(case, N, case["H"], case["W"], gen, rho0=0.3 + 0.6 * (k % 7) / 6, patches=0.01)
            for k, N in enumerate(_batch_lengths(case, seed))]


def _dphase(case, seed):
    _, _, sy, sx = _window(case)
    return torch.randn((case["N"], case["H"] // sy, case["W"] // sx), generator=_gen(seed + 7919), device="cuda")


# ------------------------------------------------------------ the two halves


def prepare(case, seed):
    kind = case["kind"]
    ctx = plk.context()
    s = {"case": case, "ctx": ctx, "kind": kind}
    if kind in ("step", "chain"):
        steps, M = case.get("steps", 1), case.get("M", case.get("N"))
        gen = _gen(seed)
        s["z"] = [_stack(case, M, case["H"], case["W"], gen, k * M) for k in range(steps)]
        s["params"] = plk.default_params(cov_precision=case.get("precision", 0), ps_da_max=case.get("regrid", 0.0),
                                         ref_scheme=int(case.get("last", False)))
        s["state"] = plk.State(ctx, case["H"], case["W"], _window(case), K_max=case.get("K", 2), M_max=M)
    elif kind == "batch":
        s["batch"] = plk.Batch(ctx, _batch_stacks(case, seed), _window(case))
    elif kind == "link":
        s["C"], s["params"] = _coherences(case, seed), plk.default_params()
    elif kind == "similarity":
        s["phase"] = _phases(case, seed)
    elif kind == "l1":
        s["unw"], s["pairs"] = _unwrapped(case, seed), _pairs(case["dates"])
    else:
        s["z"] = _stack(case, case["N"], case["H"], case["W"], _gen(seed))
        s["mask"] = _mask_words(_select(case, s["z"]))
        if kind in ("backward", "wgrad"):
            s["dphase"] = _dphase(case, seed)
    return s


def run(state):
    case, ctx, kind = state["case"], state["ctx"], state["kind"]
    if kind == "step":
        state["state"].reset()
        return state["state"].step(state["z"][0], state["params"])
    if kind == "chain":
        st = state["state"]
        st.reset()
        outs = [st.step(z, state["params"]) for z in state["z"]]
        return {"steps": outs, "kappa": st.kappa(st.info()["K_used"] - 1)}
    if kind == "batch":
        return state["batch"].run()
    if kind == "link":
        return ctx.phase_link(state["C"], case["N"], case["ref"], state["params"])
    if kind == "similarity":
        return ctx.phase_similarity(state["phase"], case["radius"])
    if kind == "l1":
        x, r = ctx.invert_l1(state["unw"], case["dates"], state["pairs"], 1.0, case["iters"], residual=True)
        return {"x": x, "residual": r}
    win = _window(case)
    if kind == "cov":
        return ctx.estimate_covariance(state["z"], win, state["mask"], precision=case["precision"])
    if kind == "backward":
        return ctx.phase_link_backward(state["z"], win, state["mask"], case["ref"], state["dphase"])
    if kind == "wgrad":
        return ctx.shp_weight_gradient(state["z"], win, state["mask"], case["ref"], state["dphase"])
    return ctx.phase_uncertainty(state["z"], win, state["mask"], case["ref"], 0.01)


def _cov_flops(N, npx, L):
    return 4.0 * N * N * ACCEPTED * L * npx


def _link_flops(N, npx):
    # Cholesky and inverse of |C|, factor of the shifted matrix, about ten
    # inverse-iteration steps, the temporal coherence
    return (16.0 / 3 * N ** 3 + 90.0 * N * N) * npx


def work(case):
    kind = case["kind"]
    if kind == "link":
        N, npx = case["N"], case["npx"]
        return {"bytes": npx * (4.0 * N * (N + 1) + 4 * N + 9), "flops": _link_flops(N, npx)}
    if kind == "similarity":
        M, npx, r = case["M"], case["Ho"] * case["Wo"], case["radius"]
        disk = sum(1 for y in range(-r, r + 1) for x in range(-r, r + 1) if 0 < x * x + y * y <= r * r)
        return {"bytes": 4.0 * (M + 1) * npx, "flops": 18.0 * M * disk * npx}
    if kind == "l1":
        n, ifg, npx = case["dates"], len(_pairs(case["dates"])), case["npx"]
        return {"bytes": 4.0 * (2 * ifg + n - 1) * npx, "flops": case["iters"] * (10.0 * ifg + 14 * (n - 1)) * npx}
    wy, wx, sy, sx = _window(case)
    H, W, L = case["H"], case["W"], wy * wx
    px, npx, words = H * W, (H // sy) * (W // sx), (L + 63) // 64
    if kind == "batch":
        Ns = _batch_lengths(case, 0)
        return {"bytes": sum(8.0 * N * px + (4 * N + 5) * npx for N in Ns),
                "flops": sum(_cov_flops(N, npx, L) + _link_flops(N, npx) for N in Ns)}
    if kind in ("step", "chain"):
        M = case.get("M", case.get("N"))
        b = f = 0.0
        for k in range(case.get("steps", 1)):
            N = M + min(k, case.get("K", 2))
            # samples once, compressed SLCs read and written, sums, outputs
            b += 8.0 * (N + 1) * px + 16.0 * px + (4 * M + 7) * npx
            f += _cov_flops(N, npx, L) + _link_flops(N, npx) + 8.0 * M * px
        return {"bytes": b, "flops": f}
    N = case["N"]
    b, f = 8.0 * N * px + 8.0 * words * npx, _cov_flops(N, npx, L)
    if kind == "cov":
        return {"bytes": b + 4.0 * N * (N + 1) * npx, "flops": f}
    f += _link_flops(N, npx)
    pixel = 60.0 * N ** 3  # deflated inverse and the chain of N x N products behind one H
    if kind == "backward":
        return {"bytes": b + 8.0 * N * px + 4.0 * N * npx, "flops": f + (pixel + 8.0 * N * N * ACCEPTED * L) * npx}
    if kind == "wgrad":
        return {"bytes": b + 4.0 * (N + L) * npx, "flops": f + (pixel + 8.0 * N * N * L) * npx}
    return {"bytes": b + 4.0 * N * npx, "flops": f + (pixel + (N - 1) * 16.0 * N ** 3) * npx}


# ------------------------------------------------------------ 64-bit results


def _windows64(case, z, rows):
    """Samples [P, N, L] (complex128) of the windows of output rows `rows`."""
    sub = [_neighbours(case, zi.to(torch.complex128))[0][rows] for zi in z]
    Z = torch.stack(sub, dim=-2)
    return Z.reshape(-1, Z.shape[-2], Z.shape[-1])


def _normalise64(S):
    d = S.diagonal(dim1=-2, dim2=-1).real
    s = torch.where(d > 0, d, 1.0).rsqrt() * (d > 0)
    C = S * (s[:, :, None] * s[:, None, :])
    eye = torch.eye(S.shape[-1], dtype=torch.bool, device=S.device)
    return torch.where(eye, torch.ones((), dtype=S.dtype, device=S.device), C)


def _matrix64(C):
    """The matrix whose smallest eigenvector carries the phases: |C|^-1 o C, or
    -C where |C| is not invertible; and which of the two."""
    G = C.abs()
    root, info = torch.linalg.cholesky_ex(G.detach())
    bad = (info > 0) | ~(root.diagonal(dim1=-2, dim2=-1).square().amin(-1) > PIVOT_FAIL)
    eye = torch.eye(C.shape[-1], dtype=G.dtype, device=C.device)
    inv = torch.linalg.inv(torch.where(bad[:, None, None], eye, G))
    return torch.where(bad[:, None, None], -C, inv * C), bad


def _link64(C, ref):
    """(phase [P, N], gamma_t [P], lambda_min [P]) of coherences C [P, N, N]."""
    A, bad = _matrix64(C)
    lam, V = torch.linalg.eigh(A)
    v = V[..., 0]
    w = v * v[:, ref, None].conj()
    phase = torch.angle(w)
    phase[:, ref] = 0
    zeta = torch.polar(torch.ones_like(phase), phase)
    m = C.abs()
    u = torch.where(m > 0, C / torch.where(m > 0, m, 1.0), torch.ones((), dtype=C.dtype, device=C.device))
    n = C.shape[-1]
    i, k = torch.triu_indices(n, n, 1, device=C.device)
    tc = (u[:, i, k] * zeta[:, i].conj() * zeta[:, k]).sum(-1).abs() / (0.5 * n * (n - 1))
    return phase, tc, torch.where(bad, float("nan"), lam[:, 0])


def _full(packed, N):
    C = torch.zeros((packed.shape[0], N, N), dtype=torch.complex128, device=packed.device)
    i, k = torch.triu_indices(N, N, device=packed.device)
    C[:, k, i] = packed.to(torch.complex128).conj()
    C[:, i, k] = packed.to(torch.complex128)
    return C


def _row_chunks(case, N):
    _, _, sy, sx = _window(case)
    Ho, Wo = case["H"] // sy, case["W"] // sx
    rows = max(1, 40_000 * 400 // (N * N) // Wo)
    return [slice(a, min(Ho, a + rows)) for a in range(0, Ho, rows)], Ho, Wo


def _cov64(case, z, sel):
    """Coherences [Ho*Wo, N, N] of a stack and its selection."""
    out = []
    for rows in _row_chunks(case, z.shape[0])[0]:
        Z = _windows64(case, z, rows)
        m = sel[rows].reshape(Z.shape[0], 1, -1)
        out.append(_normalise64((Z * m) @ Z.mH))
    return torch.cat(out)


def _step64(case, z, ref=0):
    sel = _select(case, z)
    Ho, Wo = sel.shape[:2]
    phase, tc, _ = _link64(_cov64(case, z, sel), ref)
    return phase.T.reshape(-1, Ho, Wo), tc.reshape(Ho, Wo)


def _adjoint64(case, seed, z, sel):
    """The adjoint family by automatic differentiation in 64 bits, a band of
    output rows at a time; every output pixel holds its own copy of its window."""
    kind, N, ref = case["kind"], case["N"], case["ref"]
    wy, wx, sy, sx = _window(case)
    bands, Ho, Wo = _row_chunks(case, N)
    H, W, L = case["H"], case["W"], wy * wx
    w = _dphase(case, seed).to(torch.float64) if kind != "uncertainty" else None
    grad = torch.zeros((N, H * W), dtype=torch.complex128, device="cuda")
    index, inside = _neighbours(case, torch.arange(H * W, device="cuda").reshape(H, W))
    out = []
    for rows in bands:
        Z = _windows64(case, z, rows).requires_grad_(kind != "wgrad")
        m = sel[rows].reshape(-1, 1, L).to(torch.float64)
        if kind == "wgrad":
            m = m.clone().requires_grad_(True)
        A, _ = _matrix64(_normalise64((Z * m) @ Z.mH))
        v = torch.linalg.eigh(A)[1][..., 0]
        phase = torch.angle(v * v[:, ref, None].conj())
        if kind == "uncertainty":
            std = []
            for i in range(N):
                if i == ref:
                    std.append(torch.zeros(Z.shape[0], dtype=torch.float64, device="cuda"))
                    continue
                (g,) = torch.autograd.grad(phase[:, i].sum(), Z, retain_graph=True)
                std.append(torch.sqrt(0.5 * 0.01 * g.abs().square().sum((-2, -1))))
            out.append(torch.stack(std).reshape(N, -1, Wo))
            continue
        loss = (phase * w[:, rows].reshape(N, -1).T).sum()
        (g,) = torch.autograd.grad(loss, m if kind == "wgrad" else Z)
        if kind == "wgrad":
            out.append((g[:, 0] * inside[rows].reshape(-1, L)).reshape(-1, Wo, L))
        else:
            at = index[rows].reshape(-1)
            for i in range(N):
                grad[i].index_add_(0, at, g[:, i].reshape(-1))
    if kind == "backward":
        return grad.reshape(N, H, W)
    return torch.cat(out, dim=1 if kind == "uncertainty" else 0)


def _similarity64(case, seed):
    phi = _phases(case, seed).to(torch.float64)
    M, Ho, Wo = phi.shape
    r, net = case["radius"], [(a, a + d) for a in range(M) for d in (1, 2, 3) if a + d < M]
    v = torch.polar(torch.ones_like(phi), phi)
    e = torch.stack([v[b] * v[a].conj() for a, b in net])
    pad = torch.nn.functional.pad(torch.view_as_real(e), (0, 0, r, r, r, r), value=float("nan"))
    pad = torch.view_as_complex(pad.contiguous())
    sims = [(e * pad[:, r + y:r + y + Ho, r + x:r + x + Wo].conj()).real.mean(0)
            for y in range(-r, r + 1) for x in range(-r, r + 1) if 0 < x * x + y * y <= r * r]
    sims = torch.stack(sims)
    n = (~sims.isnan()).sum(0)
    s = torch.where(sims.isnan(), float("inf"), sims).sort(0).values
    lo = s.gather(0, ((n - 1).clamp(min=0) // 2)[None])[0]
    hi = s.gather(0, (n // 2).clamp(max=s.shape[0] - 1)[None])[0]
    return torch.where((n > 0) & ~phi.isnan().any(0), 0.5 * (lo + hi), float("nan"))


def _l164(case, seed):
    b = _unwrapped(case, seed).to(torch.float64)
    pairs, n = _pairs(case["dates"]), case["dates"]
    A = torch.zeros((len(pairs), n), dtype=torch.float64, device="cuda")
    for k, (i, j) in enumerate(pairs):
        A[k, i], A[k, j] = -1.0, 1.0
    A = A[:, 1:]
    pinv = torch.linalg.solve(A.T @ A, A.T)
    z, u = torch.zeros_like(b), torch.zeros_like(b)
    for _ in range(case["iters"]):
        x = pinv @ (b + z - u)
        t = A @ x - b + u
        z = t - t.clamp(-1.0, 1.0)
        u = t - z
    return {"x": x, "residual": b - A @ x}


def exact(case, seed):
    kind = case["kind"]
    if kind == "similarity":
        disk = math.pi * case["radius"] ** 2
        return _similarity64(case, seed) if disk * case["Ho"] * case["Wo"] < 4e8 else None
    if kind == "l1":
        return _l164(case, seed)
    if kind == "link":
        N = case["N"]
        C = _coherences(case, seed)
        got = [_link64(_full(C[a:a + 32768], N), case["ref"]) for a in range(0, case["npx"], 32768)]
        phase, tc, lam = (torch.cat(g) for g in zip(*got))
        return {"phase": phase.T, "tcoh": tc, "lam": lam, "status": None}
    if kind == "batch":
        got = []
        for z in _batch_stacks(case, seed):
            phase, tc = _step64(case, z)
            got.append({"phase": phase, "tcoh": tc, "status": None})
        return got
    _, _, sy, sx = _window(case)
    npx = (case["H"] // sy) * (case["W"] // sx)
    if kind == "chain" or npx > 300_000 or (kind == "step" and case.get("regrid", 0.0)):
        return None  # a long sequence, or too many pixels for a 64-bit eigensolver
    z = _stack(case, case["N"], case["H"], case["W"], _gen(seed))
    if kind == "step":
        phase, tc = _step64(case, z)
        return {"phase": phase, "tcoh": tc, "status": None, "count": None}
    sel = _select(case, z)
    if kind == "cov":
        C = _cov64(case, z, sel)
        i, k = torch.triu_indices(case["N"], case["N"], device="cuda")
        return C[:, i, k].reshape(*sel.shape[:2], -1)
    return _adjoint64(case, seed, z, sel)
