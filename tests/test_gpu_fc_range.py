"""FC block of rows whose squares leave FP32 (below 2e-19 they are subnormal,
below 3e-23 zero, above 2e19 infinite) against ordinary rows, whose products
with them are in range: against the float64 oracle, 1e-5 of each entry, the FC
block's.  Also a row with one large element, a zero row, a symmetric block, and
scales on both sides of the range that the FP32 sums take (|x|^2 in [2^-60,
2^120])."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _run(xa, xb, depth=3, symmetric=False):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_05420_gb300.api import Handle

    h = Handle()
    Xa = torch.tensor(xa, device="cuda")
    Xb = Xa if symmetric else torch.tensor(xb, device="cuda")
    K = h.fc_block(Xa, Xb, 2.0, 0.0, depth=depth, symmetric=symmetric)
    h.sync_status()
    want = oracle.fc_nngp(xa.astype(np.float64), xb.astype(np.float64), 2.0, 0.0, depth=depth).numpy()
    return K.double().cpu().numpy(), want


@pytest.mark.parametrize("d", [100, 33, 1030])
@pytest.mark.parametrize("scale", [1e-30, 1e-26, 1e-22, 1e-20, 2e-11, 5e-10, 1.0, 1e17, 1e18, 1e20, 1e25, 1e30])
def test_scaled_rows(scale, d):
    rng = np.random.default_rng(d)
    xa = (rng.standard_normal((9, d)) * scale).astype(np.float32)
    xb = rng.standard_normal((40, d)).astype(np.float32)
    for a, b in ((xa, xb), (xb, xa)):
        got, want = _run(a, b)
        assert np.isfinite(got).all()
        assert np.max(np.abs(got - want) / np.abs(want)) <= 1e-5


def test_one_large_element_and_a_zero_row():
    rng = np.random.default_rng(0)
    xa = rng.standard_normal((4, 200)).astype(np.float32)
    xa[0, 77] = 1e21
    xa[1] = 0.0
    xb = rng.standard_normal((30, 200)).astype(np.float32)
    got, want = _run(xa, xb)
    assert np.isfinite(got).all()
    assert np.max(np.abs(got - want) / np.maximum(np.abs(want), 1e-30)) <= 1e-5


def test_symmetric_small_rows():
    rng = np.random.default_rng(1)
    x = (rng.standard_normal((50, 100)) * 10.0 ** rng.uniform(-17, 1, (50, 1))).astype(np.float32)
    got, want = _run(x, x, symmetric=True)
    assert np.isfinite(got).all()
    assert np.max(np.abs(got - want) / np.abs(want)) <= 1e-5
