"""The sums over directions at block edges other than 8 and 16 (mirrored pairs,
edges 6 to 15): how far the moments are from exact sums of the library's own
intensities."""
import numpy as np
import pytest
import torch

from paper_2202_08778_gb300 import synth, vet

pytestmark = pytest.mark.gpu


def _problem(shape, B, nside, seed):
    """A thin medium lit by intensities that differ widely by face and direction: large fluxes."""
    p = synth.lognormal_problem(shape=shape, B=B, nside=nside, seed=seed)
    ctx = vet.Context(shape, B, p["h"], nside, p["q"])
    k = torch.from_numpy((0.05 * p["kappa"]).astype(np.float32)).cuda()
    S = torch.from_numpy(p["S"].astype(np.float32)).cuda()
    Ib = torch.from_numpy(np.exp(1.5 * np.random.default_rng(seed).standard_normal((6, ctx.N))).astype(np.float32)).cuda()
    return p, ctx, k, S, Ib


def _coefficients(ctx, moments):
    """[N][len(moments)] of w (1, n, nn), rounded to FP32 as the kernels hold them."""
    d = ctx.directions()
    x, y, z, w = d.T
    c = np.stack([w * m for m in (np.ones_like(x), x, y, z, x * x, y * y, z * z, x * y, x * z, y * z)], 1)
    return torch.from_numpy(c[:, moments].astype(np.float32)).cuda()


@pytest.mark.parametrize("B,nside", [(6, 4), (10, 2), (12, 4), (14, 4), (10, 8)])
def test_flux_no_further_off_than_a_ray_at_a_time(B, nside):
    """F against exact sums of the traced intensities, beside FP32 sums of four directions at a time
    with the octants in turn (what one ray a thread gave): not above them by more than the 5% that two
    samples of some 1e4 errors can differ by."""
    shape = (2 * B, B, 2 * B)
    p, ctx, k, S, Ib = _problem(shape, B, nside, 11)
    n = k.numel()
    I, M, f = (torch.empty(r, n, device="cuda") for r in (ctx.N, 10, 6))
    ctx.trace(k, S, Ib, I)
    ctx.closure(k, S, Ib, f, M)
    ctx.sync()
    c = _coefficients(ctx, [0, 1, 2, 3])
    exact = c.double().T @ I.double()
    d = ctx.directions()
    octant = (d[:, 0] < 0) + 2 * (d[:, 1] < 0) + 4 * (d[:, 2] < 0)
    turn = [list(np.flatnonzero(octant == o)) for o in range(8)]
    order = [o[r] for r in range(max(map(len, turn))) for o in turn if r < len(o)]
    total = torch.zeros(3, n, device="cuda")
    for t in range(0, ctx.N, 4):
        part = torch.zeros(3, n, device="cuda")
        for j in order[t:t + 4]:  # a fused multiply-add: the product is exact in FP64
            part = (part.double() + c[j, 1:].double()[:, None] * I[j].double()).float()
        total = total + part
    rms = lambda F: float((((F.double() - exact[1:]) / exact[0]) ** 2).mean().sqrt())  # noqa: E731
    assert rms(M[1:4]) <= 1.05 * rms(total), (rms(M[1:4]), rms(total))
