"""Images whose pixels fall through the FP32 range: blobs exp(-r^2 / (2 s^2))
whose tails run from 1e-12 over 1e-19 (where the product of two pixels'
factors 1 / sqrt(q) leaves FP32) and 1e-38 (subnormal) to 0, without a bias.
Such pixels add nothing that FP32 can see, so the fused forms, the tangent
kernel, the Flatten readout and the FP32 adjoint's forward recursion have to
agree with the FP64 form as anywhere: 1e-5 of each entry, the FP32 forms'."""

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


def blobs(side, seed=0):
    """Four images: blobs of three widths at different places (one against the
    border), signed noise under them, and one ordinary image."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:side, 0:side].astype(np.float64)
    out = np.empty((4, side, side, 3))
    # widths such that the far corner reaches 1e-60, 1e-40 and 1e-22
    for n, (cy, cx, low) in enumerate([(side / 2, side / 2, 60), (2, side / 3, 40), (side / 4, side - 3, 22)]):
        r2 = (y - cy) ** 2 + (x - cx) ** 2
        g = 10.0 ** (-low * r2 / r2.max())
        out[n] = g[:, :, None] * (rng.standard_normal((side, side, 3)) + (2.0 if n == 1 else 0.0))
    out[3] = rng.standard_normal((side, side, 3))
    return out.astype(np.float32)


def _close(got, want):
    assert bool(torch.isfinite(got).all())
    assert float(((got.double() - want).abs() / want.abs()).max()) <= 1e-5


BLOCKS = [(8, (2, 1, 0)), (8, (3, 3, 3)), (8, (1,)), (16, (2, 1, 0)), (16, (3, 3, 3)), (16, (1,)), (32, (2, 1, 0)),
          (32, (3, 3, 3)), (32, (1,)), (32, (1, 1)), (64, (1, 1))]


@pytest.mark.parametrize("side,convs", BLOCKS)
def test_fused_blocks(h, side, convs):
    X = torch.tensor(blobs(side), device="cuda")
    q = h.self_diag(X, convs, 2.0, 0.0)
    want = h.block(X, q, X, q, convs, 2.0, 0.0, prec="plain_fp64")
    _close(h.block(X, q, X, q, convs, 2.0, 0.0, prec="mixed"), want)
    _close(h.block(X, q, X, q, convs, 2.0, 0.0, prec="mixed", symmetric=True), want)
    h.sync_status()


@pytest.mark.parametrize("convs", [(2, 1, 0), (3, 3, 3)])
def test_tangent_kernel(h, convs):
    # off the diagonal: the derivative kernel's slope is infinite at c = 1
    X = torch.tensor(blobs(32), device="cuda")
    q = h.self_diag(X, convs, 2.0, 0.0)
    kw = dict(a_range=(0, 2), b_range=(2, 4))
    K, T = h.block_ntk(X, q, X, q, convs, 2.0, 0.0, prec="mixed", **kw)
    Kw, Tw = h.block_ntk(X, q, X, q, convs, 2.0, 0.0, prec="plain_fp64", **kw)
    h.sync_status()
    _close(K, Kw)
    _close(T, Tw)


@pytest.mark.parametrize("side", [8, 16, 32])
def test_flatten_readout(h, side):
    X = torch.tensor(blobs(side), device="cuda")
    q = h.self_diag(X, (8,), 2.0, 0.0)
    want = h.block(X, q, X, q, (8,), 2.0, 0.0, prec="plain_fp64", readout="flatten")
    _close(h.block(X, q, X, q, (8,), 2.0, 0.0, prec="mixed", readout="flatten"), want)
    h.sync_status()


@pytest.mark.parametrize("side,convs", [(16, (2, 1)), (32, (2, 1, 0)), (32, (3, 3, 3))])
def test_fp32_adjoint(h, side, convs):
    """The sigma gradients of the FP32 adjoint, whose forward passes store the
    recursion that they differentiate (image gradients of pixels below the
    FP32 range are out of its reach)."""
    X = torch.tensor(blobs(side), device="cuda")
    q = h.self_diag(X, convs, 2.0, 0.0)
    got = []
    for prec, dt in (("plain_fp64", torch.float64), ("plain_fp32", torch.float32)):
        g = torch.ones((2, 2), dtype=dt, device="cuda")
        ds, db = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
        h.block_backward(X, q, X, q, convs, 2.0, 0.0, g, None, None, ds, db, prec=prec, a_range=(0, 2), b_range=(2, 4))
        got.append(float(ds))
    h.sync_status()
    assert np.isfinite(got[1]) and abs(got[1] - got[0]) <= 1e-4 * abs(got[0])
