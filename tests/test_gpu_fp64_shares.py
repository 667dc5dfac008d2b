"""FP64 closures whose last wave of SMs is split into direction shares: E and P_ii of those blocks are as
close to exact sums of the library's own intensities as those of the unsplit ones."""
import numpy as np
import pytest
import torch

from paper_2202_08778_gb300 import synth, vet

pytestmark = pytest.mark.gpu


def test_split_sums_no_further_off_than_whole_ones():
    """Either is a compensated sum rounded once; 10% for two samples of 3000 cells of different blocks."""
    n1, B, nside = 64, 16, 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    whole = (n1 // B) ** 3 * 8 // sms * sms  # CTAs of 512 cells (two layers), one an SM
    if not 0 < whole < (n1 // B) ** 3 * 8:
        pytest.skip("the grid leaves no partial wave on this device")
    p = synth.lognormal_problem(shape=(n1,) * 3, B=B, nside=nside, seed=9)
    ctx = vet.Context((n1,) * 3, B, p["h"], nside, p["q"], precision=vet.VET_FP64)
    rng = np.random.default_rng(1)
    k, S, Ib = (torch.from_numpy(np.ascontiguousarray(a)).cuda()
                for a in (0.05 * p["kappa"], p["S"], np.exp(1.5 * rng.standard_normal((6, ctx.N)))))
    n = k.numel()
    f, M, I = (torch.empty(r, n, device="cuda", dtype=torch.float64) for r in (6, 10, ctx.N))
    ctx.closure(k, S, Ib, f, M)
    ctx.trace(k, S, Ib, I)
    ctx.sync()
    x, y, z, w = ctx.directions().T
    c = np.stack([w, w * x * x, w * y * y, w * z * z]).astype(np.longdouble)
    at = np.arange(n)
    X, Y, Z = at % n1, at // n1 % n1, at // (n1 * n1)
    cta = (((Z // B) * (n1 // B) + Y // B) * (n1 // B) + X // B) * 8 + (Z % B) // 2
    rms = []
    for sel in (cta < whole, cta >= whole):
        cells = torch.from_numpy(rng.choice(np.flatnonzero(sel), 3000, replace=False)).cuda()
        got, Is = M[:, cells].cpu().numpy(), I[:, cells].cpu().numpy().astype(np.longdouble)
        exact = np.stack([(row[:, None] * Is).sum(0) for row in c])
        err = (got[[0, 4, 5, 6]].astype(np.longdouble) - exact) / exact[0]
        rms.append(np.sqrt((err[0] ** 2).mean()).astype(float))
    assert rms[1] <= 1.1 * rms[0], rms
