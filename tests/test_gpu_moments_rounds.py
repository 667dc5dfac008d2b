"""The quadratures' cells a thread, which follow the rounds of CTAs that the device takes: the same bits
whichever are taken, and no slower than the widest loads on grids of somewhat more than one round of two."""
import numpy as np
import pytest
import torch

from paper_2202_08778_gb300 import vet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 8, 8), (32, 64, 72), (48, 56, 64), (64, 64, 48), (64, 64, 80), (72, 88, 96),
                                   (96, 96, 96), (128, 96, 96)])
def test_bits_do_not_depend_on_the_width(shape):
    n = int(np.prod(shape))
    ctx = vet.Context(shape, 8, 1.0, 1)
    gen = torch.Generator(device="cuda").manual_seed(n)
    wide = torch.exp(3.0 * torch.randn(ctx.N * n, generator=gen, device="cuda"))
    odd = torch.empty(ctx.N * n + 1, device="cuda")[1:]  # one cell a thread: rows off the wide loads' boundary
    odd.copy_(wide)
    out = []
    for I in (wide, odd):
        M, E = torch.empty(10 * n, device="cuda"), torch.empty(n, device="cuda", dtype=torch.float64)
        alone = torch.empty(10 * n, device="cuda")
        ctx.moments(I, M, E64_out=E)
        ctx.moments(I, alone)
        ctx.sync()
        assert torch.equal(M, alone)
        out.append((M, E))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def test_somewhat_more_than_one_round_of_two_cells():
    """460800 cells, 192 directions: four cells a thread take 1.40 times a copy of as many bytes, two 1.57."""
    shape = (64, 72, 100)
    n = int(np.prod(shape))
    ctx = vet.Context(shape, 4, 1.0, 4)
    I, M = torch.rand(ctx.N * n, device="cuda"), torch.empty(10 * n, device="cuda")
    half = I[: ctx.N * n // 2]
    copy = torch.empty_like(half)

    def best(fn):
        t = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                fn()
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        return min(t)

    moments, copied = best(lambda: ctx.moments(I, M)), best(lambda: copy.copy_(half))
    assert moments < 1.55 * copied, moments / copied
