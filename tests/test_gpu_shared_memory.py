"""Sizes at which a kernel's dynamic shared memory alone is under 48 KB but not
together with its static tables (the launch is refused without an opt-in), in
processes of their own, so that no earlier call has raised the limit: planes
of nk_self_diag cut into two bands of 72x72, whole ones of 54x54 and 48x64;
bands of the self-variances' adjoint of 64x64 images with four and five convs
in the first stage; its D = 0 plane at 16x16 (whole, no opt-in needed)."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DIAG = """
import numpy as np, torch, oracle
from paper_2303_05420_gb300.api import Handle
H, W, n, convs = {args}
h = Handle()
x = np.random.default_rng(1).standard_normal((n, H, W, 3)).astype(np.float32)
qd, _ = h.self_diag(torch.tensor(x, device="cuda"), convs, 2.0, 0.01)
h.sync_status()
# one image takes other bands
one, _ = h.self_diag(torch.tensor(x[n - 1:], device="cuda"), convs, 2.0, 0.01)
h.sync_status()
assert bool(torch.allclose(one[0], qd[n - 1], rtol=1e-13, atol=0))
if H * W < 4000:
    arch = oracle.Arch(convs)
    want = oracle.kernels.myrtle_self_q(arch, 2.0, 0.01, torch.tensor(x[n - 1].astype(np.float64)))
    flat = torch.cat([q.reshape(-1) for q in want]).numpy()
    assert np.allclose(one[0].cpu().numpy(), flat, rtol=1e-12, atol=0)
print("ok")
"""

ADJ = """
import numpy as np, torch
from paper_2303_05420_gb300.api import Handle
side, n, convs = {args}
h = Handle()
rng = np.random.default_rng(2)
X = torch.tensor(rng.standard_normal((n, side, side, 3)).astype(np.float32), device="cuda")
Y = torch.tensor(rng.standard_normal((1, side, side, 3)).astype(np.float32), device="cuda")
qx, qy = h.self_diag(X, convs, 2.0, 0.01), h.self_diag(Y, convs, 2.0, 0.01)
g = torch.tensor(rng.standard_normal((n, 1)).astype(np.float32), device="cuda")

def grad(a0, a1):
    dX = torch.zeros_like(X)
    s = torch.zeros(2, dtype=torch.float64, device="cuda")
    h.block_backward(X, qx, Y, qy, convs, 2.0, 0.01, g[a0:a1], dX, None, s[:1], s[1:], a_range=(a0, a1))
    h.sync_status()
    return dX, s

many, sm = grad(0, n)
one = [grad(i, i + 1) for i in range(n)]  # other bands
dX, s = sum(o[0] for o in one), sum(o[1] for o in one)
# image gradients are an image's own; the targets' share of the sigma sums adds up
assert float((many - dX).abs().max()) <= 1e-6 * float(dX.abs().max())
assert float(((sm - s).abs() / s.abs()).max()) <= 1e-5
print("ok")
"""


def _run(code):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip().endswith("ok"), out.stdout + out.stderr


@pytest.mark.parametrize("args", [(72, 72, 50, (2, 1, 0)), (54, 54, 100, (2, 1)), (48, 64, 300, (2, 1))])
def test_self_diag_between_the_limits(args):
    _run(DIAG.format(args=args))


@pytest.mark.parametrize("args", [(64, 5, (4, 1, 1)), (64, 5, (5, 1, 1)), (16, 40, (2, 1))])
def test_self_adjoint_between_the_limits(args):
    _run(ADJ.format(args=args))
