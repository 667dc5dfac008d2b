"""Block edges other than 8 and 16: FP32 closures and traces on mirrored pairs
(cell pass 6 to 16, face pass 2 to 16) and past them (17) against the FP64
oracle, to the figures the closure is specified to hold."""
import numpy as np
import pytest
import torch

from gpu_common import f_error, moment_errors, rel_err
from paper_2202_08778_gb300 import synth, vet

pytestmark = pytest.mark.gpu
RTOL, FTOL = 1e-5, 1e-6


@pytest.mark.parametrize("B,blocks,nside,rotate", [
    (2, (3, 5, 4), 1, True), (3, (2, 3, 5), 2, True), (4, (3, 2, 3), 2, False), (5, (3, 1, 2), 2, True),
    (6, (2, 3, 4), 2, True), (6, (1, 1, 1), 1, False), (7, (3, 2, 1), 2, True), (7, (1, 2, 2), 1, False),
    (9, (2, 1, 3), 2, True), (10, (2, 2, 3), 2, True), (11, (1, 1, 1), 4, True), (12, (2, 3, 2), 4, True),
    (12, (2, 2, 1), 1, False), (13, (2, 1, 2), 2, True), (14, (1, 2, 2), 2, True), (15, (2, 1, 1), 2, True),
    (17, (1, 2, 1), 1, True),
    (6, (8, 8, 11), 1, True),     # 704 blocks
    (10, (6, 6, 7), 1, True)])    # 252 CTAs: the last partial wave as direction shares
def test_matches_oracle(ora, B, blocks, nside, rotate):
    shape = tuple(B * n for n in blocks)
    p = synth.lognormal_problem(shape=shape, B=B, nside=nside, seed=40 + B, rotate=rotate)
    k, S = (p[x].astype(np.float32) for x in ("kappa", "S"))
    n, N = k.size, 12 * nside * nside
    Ib = np.random.default_rng(B).uniform(0, 0.5, (6, N)).astype(np.float32)
    ctx = vet.Context(shape, B, p["h"], nside, p["q"])
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (k, S, Ib)]
    f_ref, M_ref, I_ref, _ = ora.vet_closure(k.astype(np.float64), S.astype(np.float64), ctx.directions(), B, p["h"],
                                             Ib.astype(np.float64))
    for tile in (0, 2, 8):
        if tile:
            ctx.set_tuning(dir_tile=tile)
        out = torch.full((6 + 10 + N, n), float("nan"), device="cuda")
        f, M, I = out[:6], out[6:16], out[16:]
        ctx.closure(dev[0], dev[1], dev[2], f, M)
        ctx.trace(dev[0], dev[1], dev[2], I)
        f_alone = torch.full((6, n), float("nan"), device="cuda")
        ctx.closure(dev[0], dev[1], dev[2], f_alone)
        ctx.sync()
        assert torch.equal(f_alone, f)
        assert rel_err(I.cpu(), I_ref.reshape(N, -1)) < RTOL
        eE, eFP = moment_errors(M.cpu(), M_ref)
        assert eE < RTOL and eFP < RTOL, (eE, eFP)
        assert f_error(f.cpu(), f_ref, M_ref) < FTOL


@pytest.mark.parametrize("B", [6, 7, 12])
def test_batch_gives_the_same_bits(B):
    shape = (2 * B, B, 3 * B)
    p = synth.lognormal_problem(shape=shape, B=B, nside=2, seed=B)
    k, S = (torch.from_numpy(p[x].astype(np.float32)).cuda() for x in ("kappa", "S"))
    ctx = vet.Context(shape, B, p["h"], 2, p["q"])
    batch = vet.Batch([(shape, B, p["h"], 2, p["q"])] * 2)
    f = [torch.empty(6 * k.numel(), device="cuda") for _ in range(3)]
    ctx.closure(k, S, None, f[0])
    batch.closure([k] * 2, [S] * 2, [None] * 2, f[1:])
    ctx.sync()
    batch.sync()
    assert torch.equal(f[0], f[1]) and torch.equal(f[0], f[2])
