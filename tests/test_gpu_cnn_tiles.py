"""The network's tensor-core kernels at the edges of their tiles (columns of
8 x 16 cells marched along z, shares of slices cut anywhere): forward pass and
gradients against the FP64 oracle, with the bounds of test_gpu_learned.py,
which hold for any size."""
import numpy as np
import pytest

from oracle import cnn
from test_gpu_learned import _dev, _fields, _params, torch, vet

pytestmark = pytest.mark.gpu

# (volumes, (nz, ny, nx)): one cell; a whole tile; one cell more and less than a tile; a column longer
# than the ring of accumulators; more columns than SMs; many short runs
CASES = [(1, (1, 1, 1)), (1, (3, 16, 8)), (2, (2, 17, 9)), (1, (5, 15, 7)), (1, (61, 16, 8)), (3, (2, 40, 70)),
         (1, (1, 130, 90))]


@pytest.mark.parametrize("nvol,shape", CASES)
def test_forward_and_gradients(nvol, shape):
    rng = np.random.default_rng(nvol + shape[0])
    kappa, S, E = _fields(rng, nvol, shape)
    n = int(np.prod(shape))
    h = 1.0 / max(shape)
    params = _params(5)
    model = vet.Model()
    model.set_params(params)
    o = torch.empty(nvol * 7 * n, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    f_ref = np.stack([1.0 / 3.0 + 0.1 * rng.standard_normal((nvol, *shape)) for _ in range(6)], axis=1).astype(np.float32)
    model.features(shape, 1, h, _dev(kappa), _dev(S), _dev(E), nvol=nvol)
    model.forward(o)
    model.backward(_dev(f_ref), lam=0.01, loss_out=loss)
    x = np.concatenate([cnn.features(kappa[v], S[v], E[v], h, 1).reshape(1, 6, *shape) for v in range(nvol)])
    ref, grads, L = _reference(params, x, f_ref)
    got = o.cpu().numpy().reshape(nvol, 7, *shape)
    assert np.abs(got - ref).max() < 2e-3 * np.abs(ref).max()
    assert abs(float(loss) - L) < 1e-3 * L
    for (gW, gb), (rW, rb) in zip(model.grads(), grads):
        for a, r in ((gW, rW), (gb, rb)):
            # fewer cells average fewer rounding errors: 2^-9 per term for the single cell
            bound = 1e-3 if n * nvol > 500 else 2e-2
            assert np.linalg.norm(a - r) < bound * np.linalg.norm(r)


def _reference(params, x, f_ref):
    """Outputs, gradients and loss in 64 bits (torch autograd on the CPU)."""
    F = torch.nn.functional
    P = [(torch.tensor(W, dtype=torch.float64, requires_grad=True), torch.tensor(b, dtype=torch.float64, requires_grad=True))
         for W, b in params]
    a = torch.tensor(x, dtype=torch.float64)
    for i, (W, b) in enumerate(P):
        co, ci = W.shape[1], W.shape[2]
        a = F.conv3d(a, W.permute(1, 2, 0).reshape(co, ci, 3, 3, 3), b, padding=1)
        if i < 3:
            a = F.silu(a)
    tr = a[:, :3].sum(1, keepdim=True) / 3.0
    d = torch.cat([1.0 / 3.0 + a[:, :3] - tr, a[:, 3:6]], 1) - torch.tensor(f_ref, dtype=torch.float64)
    target = torch.log(d.detach().abs().amax(1) + 1e-4)
    loss = (d * d).mean() + 0.01 * ((a[:, 6] - target) ** 2).mean()
    loss.backward()
    return a.detach().numpy(), [(W.grad.numpy(), b.grad.numpy()) for W, b in P], float(loss.detach())


@pytest.mark.parametrize("B", [1, 3, 32, 33])
def test_features_block_edges(B):
    """Block statistics on both sides of the 32-cell edge where the block's
    indices are found another way, and of blocks of equal cells."""
    rng = np.random.default_rng(B)
    shape = (B, 2 * B, B)
    kappa, S, E = _fields(rng, 2, shape)
    kappa[1, :, :B] = 3.7  # one uniform block: standard deviation 0
    h = 0.25
    model = vet.Model()
    feat = torch.empty(2 * 6 * kappa[0].size, device="cuda")
    model.features(shape, B, h, _dev(kappa), _dev(S), _dev(E), nvol=2, feat_out=feat)
    got = feat.cpu().numpy().reshape(2, 6, *shape)
    for v in range(2):
        ref = cnn.features(kappa[v], S[v], E[v], h, B)
        assert np.abs(got[v] - ref.reshape(got[v].shape)).max() < 2e-5
    assert np.abs(got[1, 5, :, :B]).max() == 0.0


def test_features_of_infinite_fields():
    """An infinite opacity or source reaches the features as it does in plain
    sums: the block's mean depth, the volume's mean source."""
    shape, B = (4, 4, 8), 4
    kappa, S, E = (np.full((1, *shape), x, np.float32) for x in (2.0, 3.0, 5.0))
    kappa[0, 1, 2, 1] = np.inf
    S[0, 3, 3, 7] = np.inf
    model = vet.Model()
    feat = torch.empty(6 * S.size, device="cuda")
    model.features(shape, B, 1.0, _dev(kappa), _dev(S), _dev(E), feat_out=feat)
    got = feat.cpu().numpy().reshape(6, *shape)
    assert np.isposinf(got[1, 1, 2, 1]) and np.isposinf(got[4, :, :, :4]).all()
    assert np.isfinite(got[4, :, :, 4:]).all() and np.isfinite(got[3]).all()
    assert np.isneginf(np.delete(got[2].ravel(), 127)).all()
