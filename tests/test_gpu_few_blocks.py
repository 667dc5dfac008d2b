"""FP32 closures and traces of few blocks of edge 6 to 15, whose cell pass runs two threads a pair of
cells where one would leave SMs idle: the bits of one thread a pair (the same grid beside a large one
in a batch), and no slower than one ray a thread (closure_noalloc)."""
import numpy as np
import pytest
import torch

from paper_2202_08778_gb300 import synth, vet

pytestmark = pytest.mark.gpu


def _fields(shape, B, nside, seed):
    p = synth.lognormal_problem(shape=shape, B=B, nside=nside, seed=seed)
    return p, *(torch.from_numpy(p[x].astype(np.float32)).cuda() for x in ("kappa", "S"))


@pytest.mark.parametrize("B,blocks,nside", [(6, (1, 1, 1), 1), (6, (2, 3, 4), 2), (7, (3, 2, 1), 2), (9, (2, 1, 3), 1),
                                            (10, (2, 2, 3), 2), (11, (1, 1, 2), 2), (12, (2, 3, 2), 4), (12, (1, 1, 1), 1),
                                            (13, (2, 1, 2), 1), (14, (1, 2, 2), 2), (15, (2, 1, 1), 2)])
def test_bits_of_one_thread_a_pair(B, blocks, nside):
    shape = tuple(B * n for n in blocks)
    p, k, S = _fields(shape, B, nside, 60 + B)
    n = k.numel()
    big = (192, 192, 192)  # beside it the small grid's CTAs would not fit the SMs at once
    kb, Sb = (torch.full(big, v, device="cuda") for v in (1.0, 0.5))
    alone = vet.Batch([(shape, B, p["h"], nside, p["q"])])
    beside = vet.Batch([(shape, B, p["h"], nside, p["q"]), (big, 16, 1 / 192, 1, p["q"])])
    N = alone.members[0].N
    Ib = torch.rand(6 * N, device="cuda")
    for tile in (0, 2, 8):
        if tile:
            for b in (alone, beside):
                b.members[0].set_tuning(dir_tile=tile)
        for with_M in (True, False):
            out = []
            for b in (alone, beside):
                others = len(b.members) - 1
                f, M = torch.full((6, n), float("nan"), device="cuda"), torch.full((10, n), float("nan"), device="cuda")
                fs = [f] + [torch.empty(6, kb.numel(), device="cuda")] * others
                Ms = [M] + [torch.empty(10, kb.numel(), device="cuda")] * others
                b.closure([k] + [kb] * others, [S] + [Sb] * others, [Ib] + [None] * others, fs, Ms if with_M else None)
                b.sync()
                out.append((f, M))
            assert torch.isfinite(out[0][0]).all() and torch.equal(out[0][0], out[1][0])
            assert not with_M or torch.equal(out[0][1], out[1][1])
        I = [torch.full((N, n), float("nan"), device="cuda") for _ in range(2)]
        for b, i in zip((alone, beside), I):
            b.members[0].trace(k, S, Ib, i)
            b.members[0].sync()
        assert torch.isfinite(I[0]).all() and torch.equal(I[0], I[1])


def _time(fn):
    for _ in range(3):
        fn()
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(5):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 5)
    return best


@pytest.mark.parametrize("B,blocks", [(6, (4, 4, 4)), (14, (2, 2, 2))])
def test_no_slower_than_a_ray_a_thread(B, blocks):
    """192 directions.  One thread a pair took 1.67 and 1.70 times what one ray a thread took."""
    shape = tuple(B * n for n in blocks)
    p, k, S = _fields(shape, B, 4, 5)
    f = torch.empty(6, k.numel(), device="cuda")
    batch = vet.Batch([(shape, B, p["h"], 4, p["q"])])
    paired = _time(lambda: batch.closure([k], [S], None, [f]))
    single = _time(lambda: vet.closure_noalloc(shape, B, p["h"], 4, k, S, None, f, rot_q=p["q"]))
    assert paired < single, (paired, single)


def test_hand_over_that_gives_up_is_reported():
    """One poll a wait: the launch ends, the call reports the timeout, and a patient batch still gives its bits."""
    B, nside = 12, 4
    shape = (3 * B, 3 * B, 3 * B)
    p, k, S = _fields(shape, B, nside, 8)
    f, f2, lost = (torch.empty(6, k.numel(), device="cuda") for _ in range(3))
    patient, impatient = (vet.Batch([(shape, B, p["h"], nside, p["q"])], spin_limit=s) for s in (0, 1))
    patient.closure([k], [S], None, [f])
    patient.sync()
    impatient.closure([k], [S], None, [lost])
    with pytest.raises(vet.VetError) as err:
        impatient.sync()
    assert err.value.status == vet.VET_ETIMEOUT
    patient.closure([k], [S], None, [f2])
    patient.sync()
    assert torch.equal(f, f2)


@pytest.mark.parametrize("B", [6, 10, 12])
def test_listed_blocks_give_the_bits_of_the_whole_grid(B):
    """The learned closure's fallback on a few blocks (two threads a pair) against the plain closure of a
    grid that fills the SMs once (one)."""
    side = {6: 8, 10: 6, 12: 5}[B]
    shape = (side * B,) * 3
    p, k, S = _fields(shape, B, 2, 70 + B)
    n = k.numel()
    ctx = vet.Context(shape, B, p["h"], 2, p["q"])
    rng = np.random.default_rng(B)
    model = vet.Model()
    model.set_params([(rng.uniform(-0.05, 0.05, (27, co, ci)), np.zeros(co)) for ci, co in vet.layer_shapes()])
    E = torch.rand(n, device="cuda") + 0.5
    f, plain, r = torch.empty(6, n, device="cuda"), torch.empty(6, n, device="cuda"), torch.empty(n, device="cuda")
    flags = torch.empty(side ** 3, dtype=torch.int32, device="cuda")
    model.closure(ctx, k, S, E, f, threshold=float("inf"))
    model.last_indicator(r, n)
    at = torch.arange(n, device="cuda")
    x, y, z = at % shape[2], at // shape[2] % shape[1], at // (shape[1] * shape[2])
    block = (z // B * side + y // B) * side + x // B
    worst = torch.zeros(side ** 3, device="cuda").scatter_reduce(0, block, r, "amax").sort(descending=True).values
    kept = model.closure(ctx, k, S, E, f, threshold=float(worst[5]), block_flags=flags)
    ctx.closure(k, S, None, plain)
    ctx.sync()
    listed = flags.bool()[block]
    assert 0 < kept <= 5 and int(flags.bool().sum()) == kept
    assert torch.equal(f[:, listed], plain[:, listed]) and not torch.equal(f[:, ~listed], plain[:, ~listed])
