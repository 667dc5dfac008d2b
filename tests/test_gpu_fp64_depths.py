"""FP64 closures whose segments take every branch of the FP64 weight: no
opacity at all, depths of every size up to far beyond e^-x's range, and
lengths and opacities outside FP32's range."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_08778_gb300 import synth, vet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h", [1.0, 1e-45, 1e40])
@pytest.mark.parametrize("B", [8, 5])
def test_all_depths(B, h):
    shape = (2 * B, B, 2 * B)
    rng = np.random.default_rng(B)
    tau = np.exp(rng.uniform(np.log(1e-9), np.log(3e3), shape))
    tau[rng.random(shape) < 0.1] = 0.0
    kappa, S = tau / h, rng.uniform(0.5, 2.0, shape)
    ctx = vet.Context(shape, B, h, 2, synth.rotation_quaternion(3), vet.VET_FP64)
    Ib = rng.uniform(0.5, 2.0, (6, ctx.N))
    n = kappa.size
    f = torch.empty(6 * n, dtype=torch.float64, device="cuda")
    M = torch.empty(10 * n, dtype=torch.float64, device="cuda")
    I = torch.empty(ctx.N * n, dtype=torch.float64, device="cuda")
    dev = [torch.from_numpy(x).cuda() for x in (kappa, S, Ib)]
    ctx.closure(*dev, f, M)
    ctx.trace(*dev, I)
    ctx.sync()
    f_ref, M_ref, I_ref, _ = oracle.vet_closure(kappa, S, ctx.directions(), B, h, Ib)
    # the FP64 tolerance of the parity tests: both sides differ in rounding alone
    assert (np.abs(I.cpu().numpy().reshape(I_ref.shape) - I_ref) / I_ref).max() < 1e-11
    assert (np.abs(M.cpu().numpy().reshape(10, -1) - M_ref.reshape(10, -1)) / M_ref[0].ravel()).max() < 1e-11
    assert np.abs(f.cpu().numpy().reshape(6, -1) - f_ref.reshape(6, -1)).max() < 1e-12
