"""The point source's walk over brick-shaped warps: grids thinner than a brick,
ragged extents, sources on faces, edges, corners and at the upper boundary (where
a source rounds to it in 32 bits), and the grids whose walks check their reads.

Tolerance: that of test_gpu_point_source.py; a uniform opacity over 65537 cells
sums as many lengths one after another, each addition half an ulp of tau_*."""
import numpy as np
import pytest
import torch

from oracle import point_source as ps
from paper_2202_08778_gb300 import vet

pytestmark = pytest.mark.gpu


def _run(kappa, h, xs):
    n = kappa.size
    k = torch.from_numpy(np.ascontiguousarray(kappa)).cuda()
    out = torch.full((5, n), np.nan, device="cuda")
    vet.point_source(kappa.shape, h, xs, 3.0, k, out[0], out[1:4])
    vet.point_source(kappa.shape, h, xs, 3.0, k, out[4], None)
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[4])
    return out[0].cpu().numpy(), out[1:4].cpu().numpy()


@pytest.mark.parametrize("shape,xs_cells", [
    ((1, 1, 1), (0.25, 0.5, 0.75)), ((1, 1, 70), (30.5, 0.5, 0.5)), ((1, 67, 1), (0.3, 40.2, 0.9)),
    ((65, 1, 1), (0.5, 0.5, 0.0)), ((1, 2, 33), (17.0, 1.0, 0.5)), ((2, 19, 3), (1.5, 0.0, 1.0)),
    ((3, 5, 17), (0.0, 0.0, 0.0)), ((17, 4, 4), (2.0, 2.0, 8.0)), ((5, 6, 7), (6.5, 5.5, 4.5)),
    ((4, 8, 16), (16 * (1 - 1e-12), 8 * (1 - 1e-12), 4 * (1 - 1e-12))), ((9, 7, 18), (18 * (1 - 1e-12), 3.0, 4.4))])
def test_every_cell_matches_oracle(shape, xs_cells):
    h = 0.125
    kappa = np.random.default_rng(sum(shape)).lognormal(0.0, 1.0, shape).astype(np.float32)
    E, p = _run(kappa, h, tuple(v * h for v in xs_cells))
    xs = tuple(float(np.float32(v)) * h for v in xs_cells)
    Er, pr = ps.deposit(kappa.astype(np.float64), h, tuple(min(x, np.nextafter(n * h, 0)) for x, n in zip(xs, shape[::-1])), 3.0)
    tau = np.array([ps.optical_depth(kappa.astype(np.float64), h, tuple(min(x, np.nextafter(n * h, 0)) for x, n in zip(xs, shape[::-1])),
                                     tuple((c + 0.5) * h for c in np.unravel_index(i, shape)[::-1]))[0]
                    if Er[i] else 0.0 for i in range(kappa.size)])
    bound = 2e-5 * (1.0 + tau) * np.abs(Er) + 1e-30
    assert np.all(np.abs(E - Er) <= bound)
    assert np.all(np.abs(p - pr) <= bound[None, :] + 1e-7 * np.abs(Er)[None, :])


@pytest.mark.parametrize("shape,axis", [((1, 2, 65537), 0), ((65537, 1, 2), 2)])
def test_extents_past_the_plain_walk(shape, axis):
    h, kap, n = 1.0, np.float32(2.0 ** -15), 65537
    src = [0.5, 0.5, 0.5]
    src[axis] = 12.25
    E, _ = _run(np.full(shape, kap), h, tuple(src))
    E = E.reshape(shape).astype(np.float64)
    line = E[0, 0] if axis == 0 else E[:, 0, 0]  # the source's own row: straight along the axis
    x = np.arange(n) + 0.5
    r = np.abs(x - src[axis])
    dr = np.where(np.arange(n) == 12, 0.75, 1.0)
    want = 3.0 * np.exp(-float(kap) * (r + 0.5 - dr)) * -np.expm1(-float(kap) * dr) / (4 * np.pi * r ** 2 * dr)
    tol = 2e-5 + (float(kap) * r) * n * 2.0 ** -24
    assert np.all(np.abs(line - want) <= tol * want)
