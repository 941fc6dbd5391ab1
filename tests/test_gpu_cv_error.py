"""Flatten readout against the FP64 recursion of the pixel pairs p = p' (the only
ones that readout takes): no error of one sign that grows with the layers (its
mean over a block; entries alone carry FP32's 6e-8), and column sums that leave
FP32 although the mean does not."""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_05420_gb300.api import Handle

    return Handle()


def _box(t):
    u = torch.nn.functional.pad(t, (1, 1, 1, 1))
    n, m = t.shape[-2:]
    return sum(u[..., a:a + n, b:b + m] for a in range(3) for b in range(3))


def _exact(x, y, depth, sb2):
    """Block [len(x), len(y)] in float64 (sigma_w^2 = 2)."""
    x, y = x.double(), y.double()

    def selfq(z):
        t, out = (z * z).mean(-1), []
        for _ in range(depth):
            out.append(2.0 / 9.0 * _box(t) + sb2)
            t = out[-1] / 2
        return out

    qx, qy = selfq(x), selfq(y)
    t = torch.einsum("aijc,bijc->abij", x, y) / x.shape[-1]
    for qa, qb in zip(qx, qy):
        k = 2.0 / 9.0 * _box(t) + sb2
        s = torch.sqrt(qa[:, None]) * torch.sqrt(qb[None])
        c = (k / s).clamp(-1.0, 1.0)
        t = s / (2 * math.pi) * (torch.sqrt(1 - c * c) + c * (math.pi - torch.acos(c)))
    return 2.0 * t.mean(dim=(-1, -2)) + sb2


@pytest.mark.parametrize("side,depth,sb2", [(32, 8, 0.0), (32, 8, 0.01), (16, 8, 0.01), (32, 3, 0.0)])
def test_errors_do_not_add_up(h, side, depth, sb2):
    """The map's mean error is a few 1e-9 a layer and the layers' constant is exact
    to 1e-9, so eight layers stay under 1.5e-8 (twice that at three layers, whose
    correlations reach down to where the map is off by up to 4e-8)."""
    rng = np.random.default_rng(side + depth)
    x = rng.standard_normal((200, side, side, 3))
    x = torch.nn.functional.avg_pool2d(torch.tensor(x).permute(0, 3, 1, 2), 3, 1, 1).permute(0, 2, 3, 1)
    X = (x / x.std()).float().cuda().contiguous()
    a, b = X[:100].contiguous(), X[100:].contiguous()
    qa, qb = h.self_diag(a, (depth,), 2.0, sb2), h.self_diag(b, (depth,), 2.0, sb2)
    K = h.block(a, qa, b, qb, (depth,), 2.0, sb2, prec="mixed", readout="flatten")
    h.sync_status()
    e = K.double() / _exact(a, b, depth, sb2) - 1
    assert abs(float(e.mean())) <= (1.5e-8 if depth == 8 else 3e-8)
    assert float(e.abs().max()) <= 2e-7


def test_column_sums_beyond_fp32(h):
    rng = np.random.default_rng(0)
    x = np.where(rng.random((5, 32, 32, 3)) < 0.1, -3.4e18, 3.4e18).astype(np.float32)
    X = torch.tensor(x, device="cuda")
    q = h.self_diag(X, (2,), 2.0, 0.0)
    K = h.block(X, q, X, q, (2,), 2.0, 0.0, prec="mixed", readout="flatten")
    h.sync_status()
    want = _exact(X, X, 2, 0.0)
    assert float(((K.double() - want).abs() / want).max()) <= 1e-5
