"""Small grids, whose cell pass is split into direction shares to fill the SMs:
bit for bit what the unsplit pass computes in FP32 (the same grid in a batch,
which never splits), to rounding in FP64; with and without the moments,
repeatedly and after retuning."""
import numpy as np
import pytest
import torch

from gpu_common import f_error, moment_errors, rel_err
from paper_2202_08778_gb300 import synth, vet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,B,nside", [((8, 8, 8), 8, 1),      # one CTA, two shares
                                           ((16, 16, 16), 16, 4),  # one block of two CTAs, all 24 tiles shares
                                           ((8, 24, 40), 8, 2), ((32, 32, 48), 16, 2),
                                           ((48, 48, 48), 16, 4),  # two shares an item
                                           ((56, 64, 72), 8, 1)])  # 504 CTAs of 608: one share each
def test_bits_of_the_unsplit_pass(shape, B, nside):
    p = synth.lognormal_problem(shape=shape, B=B, nside=nside, seed=7)
    n = int(np.prod(shape))
    k, S = (torch.from_numpy(p[x].astype(np.float32)).cuda() for x in ("kappa", "S"))
    ctx = vet.Context(shape, B, p["h"], nside, p["q"])
    Ib = torch.rand(6 * ctx.N, device="cuda")
    batch = vet.Batch([(shape, B, p["h"], nside, p["q"])])
    for tile in (8, 2):
        ctx.set_tuning(dir_tile=tile)
        batch.members[0].set_tuning(dir_tile=tile)
        for with_M in (True, False):
            out = [(torch.empty(6 * n, device="cuda"), torch.empty(10 * n, device="cuda") if with_M else None) for _ in range(3)]
            ctx.closure(k, S, Ib, *out[0])
            ctx.closure(k, S, Ib, *out[1])
            batch.closure([k], [S], [Ib], [out[2][0]], [out[2][1]] if with_M else None)
            ctx.sync()
            batch.sync()
            for o in out[:2]:
                assert torch.equal(o[0], out[2][0])
                assert not with_M or torch.equal(o[1], out[2][1])


@pytest.mark.parametrize("shape,B,nside", [((8, 8, 8), 8, 1),      # one CTA, three shares of one direction tile
                                           ((16, 16, 16), 16, 2),  # 8 CTAs
                                           ((48, 48, 48), 16, 2),  # 216 CTAs: one wave and a split last one
                                           ((24, 32, 48), 4, 1),   # 576 CTAs of 64 threads
                                           ((10, 15, 20), 5, 2), ((21, 14, 28), 7, 2)])
def test_fp64_shares_match_oracle(ora, shape, B, nside):
    """FP64 sums differ from the oracle in their order only: 1e-11 on the
    moments, 1e-12 on f."""
    p = synth.lognormal_problem(shape=shape, B=B, nside=nside, seed=8)
    n = int(np.prod(shape))
    ctx = vet.Context(shape, B, p["h"], nside, p["q"], precision=vet.VET_FP64)
    Ib = np.random.default_rng(8).uniform(0, 0.5, (6, ctx.N))
    k, S, ib = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (p["kappa"], p["S"], Ib))
    f_ref, M_ref, I_ref, _ = ora.vet_closure(p["kappa"], p["S"], ctx.directions(), B, p["h"], Ib)
    for tile in (0, 1, 8):
        if tile:
            ctx.set_tuning(dir_tile=tile)
        f, M, f_alone, I = (torch.full((r, n), float("nan"), dtype=torch.float64, device="cuda") for r in (6, 10, 6, ctx.N))
        for _ in range(2):
            ctx.closure(k, S, ib, f, M)
        ctx.closure(k, S, ib, f_alone)
        ctx.trace(k, S, ib, I)
        ctx.sync()
        assert rel_err(I.cpu(), I_ref.reshape(ctx.N, -1)) < 1e-11
        eE, eFP = moment_errors(M.cpu(), M_ref)
        assert eE < 1e-11 and eFP < 1e-11
        assert f_error(f.cpu(), f_ref, M_ref) < 1e-12 and f_error(f_alone.cpu(), f_ref, M_ref) < 1e-12


@pytest.mark.parametrize("shape,B,nside,precision", [((64, 64, 128), 16, 4, vet.VET_FP32),  # 256 CTAs of 152 places
                                                     ((60, 60, 70), 10, 2, vet.VET_FP32), ((48, 48, 48), 16, 2, vet.VET_FP64),
                                                     ((16, 32, 16), 16, 4, vet.VET_FP64)])
def test_repeated_calls_give_the_same_bits(shape, B, nside, precision):
    p = synth.lognormal_problem(shape=shape, B=B, nside=nside, seed=9)
    n, dtype = int(np.prod(shape)), torch.float32 if precision == vet.VET_FP32 else torch.float64
    k, S = (torch.from_numpy(np.ascontiguousarray(p[x])).to("cuda", dtype) for x in ("kappa", "S"))
    ctx = vet.Context(shape, B, p["h"], nside, p["q"], precision=precision)
    out = [torch.empty(16, n, dtype=dtype, device="cuda") for _ in range(6)]
    for o in out:
        ctx.closure(k, S, None, o[:6], o[6:])
    ctx.sync()
    assert all(torch.equal(o, out[0]) for o in out[1:])
