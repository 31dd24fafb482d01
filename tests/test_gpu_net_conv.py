"""The network's implicit-GEMM convolutions at the edges of their tilings, forward and gradient
against the oracle: channel counts that are not powers of two or exceed one tile of channels, odd
channel groups, layers of one pixel, batches below max_batch, and a handle used with several batch
sizes in turn."""
import numpy as np
import pytest

from tests import _parity as P
from tests.test_gpu_warmnet import CONDS, _check_grads, _net, _rel
from oracle import warmnet as WN

pytestmark = pytest.mark.gpu

MEAN = np.array([0.1, 0.0, -0.1, 1e-4, 2e-4])
SCALE = np.array([1.0, 2.0, 0.5, 1.5e-3, 0.8e-3])


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


def _target(b, ny, nx, seed):
    r = np.random.default_rng(seed)
    phi = CONDS[:b, 1][:, None, None]
    t = r.normal(size=(b, 5, ny, nx)) * SCALE[None, :, None, None]
    t[:, 3] += phi
    t[:, 4] += 1.0 - phi
    return t.astype(np.float32)


@pytest.mark.parametrize("ny,nx,c0,hidden,batch,max_batch", [
    (16, 16, 8, 5, 2, 2),    # deepest layer 1 x 1; every forward product split over K
    (32, 48, 24, 16, 1, 2),  # 24 .. 192 channels: odd groups, ragged channel tiles, two o chunks
    (48, 32, 64, 9, 2, 3),   # 64 .. 512 channels: several tiles and chunks of channels
    (160, 144, 8, 7, 3, 3),  # tiles cut at the right and lower edges, products not split
])
def test_conv_tilings_match_oracle(ny, nx, c0, hidden, batch, max_batch):
    import torch
    net, p = _net(ny, nx, c0, hidden, max_batch, seed=7)
    cond = CONDS[:batch]
    cond32 = cond.astype(np.float32)
    c = WN.condition(*cond32.astype(np.float64).T)
    phi = cond32.astype(np.float64)[:, 1]
    net.set_normalizer(MEAN, SCALE)
    out = net.forward(torch.from_numpy(cond32)).cpu().numpy()
    norm = lambda f: WN.normalised_target(f, MEAN, SCALE, phi)  # noqa: E731
    ref = WN.predict_fields(p, c, MEAN, SCALE, ny, nx, c0, hidden, bf16=True, phi=phi)
    ref64 = WN.predict_fields(p, c, MEAN, SCALE, ny, nx, c0, hidden, phi=phi)
    # FP32 accumulation over K <= 9216 perturbs a value by about sqrt(K) 6e-8 = 6e-6, which flips
    # its rounding to BF16 with a probability of 1.5e-3: 8e-5 of a layer's norm, times the gain of
    # ten random layers. FP32 fields of phi and rho^w resolve 6e-8 of 1 in a spread of 8e-4.
    assert _rel(norm(out), norm(ref)) < 5e-3
    assert _rel(norm(out), norm(ref64)) < 3e-2
    _check_grads(net, p, ny, nx, c0, hidden, cond, _target(batch, ny, nx, 11), MEAN, SCALE, 5e-3,
                 6e-2)


def test_batch_sizes_in_turn():
    """The plans of the backward pass follow the batch size: a handle used with 3, 1, 2 and 3
    samples gives what fresh handles give, bit for bit."""
    import torch
    ny, nx, c0, hidden = 32, 32, 8, 16
    net, p = _net(ny, nx, c0, hidden, 3, seed=2)
    net.set_normalizer(MEAN, SCALE)
    for b in (3, 1, 2, 3):
        cond, target = torch.from_numpy(CONDS[:b].astype(np.float32)), _target(b, ny, nx, b)
        loss, g = net.loss_grad(cond, torch.from_numpy(target))
        fresh, _ = _net(ny, nx, c0, hidden, 3, seed=2)
        fresh.set_normalizer(MEAN, SCALE)
        loss1, g1 = fresh.loss_grad(cond, torch.from_numpy(target))
        assert loss == loss1 and torch.equal(g, g1)
