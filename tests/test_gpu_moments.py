"""The quadratures of stored intensities over their load widths (odd cell
counts, pairs, the four-cell path of large grids, rows that do not start on the
wide loads' boundary) and E in FP64, with what FP32 sums cannot hold."""
import numpy as np
import pytest
import torch

from paper_2202_08778_gb300 import synth, vet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,B,nside,offset", [((3, 3, 5 * 3), 3, 1, 0), ((2, 6, 14), 2, 2, 0), ((8, 8, 8), 8, 4, 0),
                                                  ((8, 8, 8), 8, 2, 2), ((8, 8, 8), 8, 2, 1), ((88, 96, 80), 8, 1, 0),
                                                  ((88, 96, 80), 8, 1, 2)])
def test_moments_and_e64(shape, B, nside, offset):
    n = int(np.prod(shape))
    ctx = vet.Context(shape, B, 1.0, nside, synth.rotation_quaternion(2))
    gen = torch.Generator(device="cuda").manual_seed(n)
    buf = torch.exp(6.0 * torch.randn(ctx.N * n + offset, generator=gen, device="cuda"))
    I = buf[offset:]
    M = torch.empty(10 * n, device="cuda")
    M2 = torch.empty(10 * n, device="cuda")
    E = torch.empty(n, device="cuda", dtype=torch.float64)
    ctx.moments(I, M, E64_out=E)
    ctx.moments(I, M2)
    ctx.sync()
    assert torch.equal(M, M2)
    d = torch.from_numpy(ctx.directions()).cuda()
    x, y, z, w = d[:, 0], d[:, 1], d[:, 2], d[:, 3]
    coef = torch.stack([w, w * x, w * y, w * z, w * x * x, w * y * y, w * z * z, w * x * y, w * x * z, w * y * z])
    ref = coef @ I.view(ctx.N, n).double()
    # FP64 sums of N terms, at most N roundings of 2^-53; plain FP32 sums N of 2^-24 (and the coefficients')
    assert ((E - ref[0]).abs() / ref[0]).max().item() < ctx.N * 2.0 ** -53
    assert ((M.view(10, n) - ref).abs() / ref[0]).max().item() < (ctx.N + 2) * 2.0 ** -24


def test_e64_of_what_fp32_sums_cannot_hold():
    shape, B = (4, 4, 6), 2
    n = int(np.prod(shape))
    ctx = vet.Context(shape, B, 1.0, 1, synth.rotation_quaternion(2))
    I = torch.full((ctx.N, n), 1.5, device="cuda")
    I[:, 0] = 3e38                      # a finite sum above FP32's range
    I[3, 1], I[5, 2], I[7, 3] = float("inf"), float("nan"), float("-inf")
    I[2, 4], I[3, 4] = float("inf"), float("-inf")
    I[:, 5] = 1e-42                     # denormals
    I[:, 6] = -2.25
    M, E = torch.empty(10 * n, device="cuda"), torch.empty(n, device="cuda", dtype=torch.float64)
    ctx.moments(I.reshape(-1), M, E64_out=E)
    ctx.sync()
    want = (4.0 * np.pi / ctx.N) * I.double().sum(0)
    np.testing.assert_allclose(E.cpu().numpy(), want.cpu().numpy(), rtol=1e-14, equal_nan=True)
