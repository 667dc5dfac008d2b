"""The learned closure's features against sums of the same FP32 logarithms in exact arithmetic: log S
and log E minus their volume means, and the blocks' mean and deviation of log (kappa h)."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2202_08778_gb300 import vet

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -24  # half a unit in the last place, relative at most


def _features(x, B):
    """[volumes][6][cells] of fields kappa h = S = E = x, whose logarithm is feature 1."""
    dev = torch.from_numpy(x).cuda()
    feat = torch.empty(6 * x.size, device="cuda")
    vet.Model().features(x.shape[1:], B, 1.0, dev, dev, dev, nvol=x.shape[0], feat_out=feat)
    torch.cuda.synchronize()
    return feat.cpu().numpy().astype(np.float64).reshape(x.shape[0], 6, -1)


def _check(got, shape, B, of_mean):
    """Half a unit in a feature's last place and of_mean for the mean's own error, relative to the
    logarithms; 2^-45 for the deviation's cancellation."""
    log = got[1]
    size, n = np.abs(log).max(), log.size
    mean = sum(map(Fraction, log), Fraction(0)) / n
    exact = {v: float(Fraction(v) - mean) for v in np.unique(log)}
    exact = np.array([exact[v] for v in log])
    for row in (2, 3):
        err = np.abs(got[row] - exact)
        assert (err <= EPS * (1 + 2.0 ** -10) * np.abs(exact) + of_mean * size).all(), (row, err.max())
    z, y, x = np.unravel_index(np.arange(n), shape)
    block = ((z // B) * (shape[1] // B) + y // B) * (shape[2] // B) + x // B
    for b in range(block.max() + 1):
        vals = [Fraction(v) for v in log[block == b]]
        mu = sum(vals, Fraction(0)) / len(vals)
        sd = math.sqrt(float(sum((v - mu) ** 2 for v in vals) / len(vals)))
        at = np.flatnonzero(block == b)[0]
        assert abs(got[4][at] - float(mu)) <= EPS * (1 + 2.0 ** -10) * abs(float(mu)) + of_mean * size
        assert abs(got[5][at] - sd) <= EPS * (1 + 2.0 ** -10) * sd + 2.0 ** -45 * size


@pytest.mark.parametrize("shape,B", [((12, 8, 16), 4), ((16, 16, 32), 16), ((10, 5, 15), 5)])
@pytest.mark.parametrize("kind", ["wide", "outliers", "zeros"])
def test_features_of_fields(kind, shape, B):
    """The mean's error: some 40 FP64 roundings of a sum."""
    g = np.random.default_rng(7)
    x = np.exp((4.0 if kind == "wide" else 0.5) * g.standard_normal(shape)).astype(np.float32)
    if kind != "wide":
        x.flat[::64] = 1e-12 if kind == "outliers" else 0.0  # zeros: the floor of the logarithm's argument
    _check(_features(x[None], B)[0], shape, B, 2.0 ** -47)


def test_features_of_nearly_constant_fields():
    """Fields whose logarithms differ by a few units in the last place and have one exponent: their sums
    are exact in FP64, the mean and the difference are rounded once each."""
    x = (3e-3 * (1.0 + 5e-6 * np.random.default_rng(1).standard_normal((512, 5, 5, 5)))).astype(np.float32)
    for got in _features(x, 5):
        _check(got, (5, 5, 5), 5, 2.0 ** -52)
