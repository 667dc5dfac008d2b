"""The sums over directions at block edges other than 8 and 16 (mirrored pairs,
edges 6 to 15): how far the moments are from exact sums of the library's own
intensities, unsplit and in the direction shares of the last partial wave."""
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


def _pair_wave(B):
    """CTAs of the paired cell pass that the device holds at once, and CTAs a block."""
    half = (B ** 3 + 1) // 2
    parts = -(-half // 512)
    threads = -(-(-(-half // parts)) // 32) * 32
    return torch.cuda.get_device_properties(0).multi_processor_count * min(8, 1024 // threads), parts


@pytest.mark.parametrize("B,nside", [(6, 2), (10, 2), (12, 2), (14, 2)])
def test_shares_of_the_last_wave(ora, B, nside):
    """A grid a little over one wave: its last blocks' directions are summed in shares.  They are (their
    bits differ from the same grid's in a batch, which does not split; the other blocks' do not), match
    the oracle, repeat, and P_ij is as close to exact sums as the unsplit ones: both round a compensated
    sum once, 25% for its compensations' own roundings."""
    wave, parts = _pair_wave(B)
    # blocks: over one wave by a twelfth to a fifth of it
    side = next(s for s in ((a, b, c) for a in range(3, 14) for b in range(a, 14) for c in range(b, 14))
                if 1 / 12 <= (s[0] * s[1] * s[2] * parts) / wave - 1 <= 1 / 5)
    shape = tuple(B * s for s in side)
    p, ctx, k, S, Ib = _problem(shape, B, nside, 12)
    n = k.numel()
    batch = vet.Batch([(shape, B, p["h"], nside, p["q"])])
    I, M, M2, Mb = (torch.empty(r, n, device="cuda") for r in (ctx.N, 10, 10, 10))
    f, f2, fb, f_alone = (torch.empty(6, n, device="cuda") for _ in range(4))
    ctx.closure(k, S, Ib, f, M)
    ctx.closure(k, S, Ib, f2, M2)
    ctx.closure(k, S, Ib, f_alone)
    ctx.trace(k, S, Ib, I)
    batch.closure([k], [S], [Ib], [fb], [Mb])
    ctx.sync()
    batch.sync()
    assert torch.equal(f, f2) and torch.equal(M, M2) and torch.equal(f, f_alone)
    blocks = int(np.prod(side))
    whole = (blocks * parts - (blocks * parts) % wave) // parts  # blocks before the last wave
    at = torch.arange(n, device="cuda")
    x, y, z = at % shape[2], at // shape[2] % shape[1], at // (shape[1] * shape[2])
    block = (z // B * side[1] + y // B) * side[2] + x // B
    first, tail = block < whole, block > whole
    assert torch.equal(M[:, first], Mb[:, first])
    assert not torch.equal(M[:, tail], Mb[:, tail])
    exact = _coefficients(ctx, [0, 7, 8, 9]).double().T @ I.double()
    rms = lambda P: float((((P[7:].double() - exact[1:]) / exact[0])[:, tail] ** 2).mean().sqrt())  # noqa: E731
    assert rms(M) <= 1.25 * rms(Mb), (rms(M), rms(Mb))
    ref = ora.vet_closure(k.cpu().numpy().astype(np.float64), S.cpu().numpy().astype(np.float64), ctx.directions(), B,
                          p["h"], Ib.cpu().numpy().astype(np.float64))
    assert float((I.cpu().double() - torch.from_numpy(ref[2].reshape(ctx.N, -1))).abs().max()
                 / np.abs(ref[2]).max()) < 1e-5
    assert float((f.cpu().double() - torch.from_numpy(ref[0].reshape(6, -1))).abs().max()) < 1e-6
