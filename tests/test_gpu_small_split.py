"""Small grids, whose cell pass is split into direction shares to fill the SMs:
bit for bit what the unsplit pass computes (the same grid in a batch, which
never splits), with and without the moments, repeatedly and after retuning."""
import numpy as np
import pytest
import torch

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
