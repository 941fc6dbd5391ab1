"""The resident CG run on kernel matrices whose ridge leaves kappa between 1e6
and 1e8 (Gaussian kernels of random points), where FP32 products limit what CG's
recurrences are worth: against a direct float64 solve, and against the
graph-replayed run (33 right-hand sides: the same columns repeated), which may
not need noticeably fewer iterations or, without refinement, leave a smaller
residual.  A relative residual of tol gives an error of at most kappa tol."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _problem(n, dim, ell, ridge, r):
    rng = np.random.default_rng(n)
    x = torch.tensor(rng.standard_normal((n, dim)), device="cuda")
    s = (x * x).sum(1)
    k = torch.exp(-(s[:, None] + s[None] - 2 * x @ x.T).clamp(min=0) / (2 * ell * ell)).float()
    k = torch.tril(k) + torch.tril(k, -1).T
    lam = ridge * float(torch.trace(k.double())) / n
    return k.contiguous(), lam, torch.tensor(rng.standard_normal((n, r)), device="cuda")


CASES = [(600, 8, 4.0, 1e-4), (600, 8, 4.0, 1e-5), (1000, 4, 3.0, 1e-4), (1000, 16, 8.0, 1e-6), (2048, 8, 4.0, 1e-4),
         (2700, 16, 8.0, 1e-3), (4500, 8, 4.0, 1e-3)]


@pytest.mark.parametrize("n,dim,ell,ridge", CASES)
def test_mixed_solve(n, dim, ell, ridge):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_05420_gb300.api import Handle

    h = Handle()
    K, lam, Y = _problem(n, dim, ell, ridge, 3)
    tol = 1e-8
    A, its, rel = h.pcg_solve(K, Y, lam, tol=tol, maxit=60000, refine_max=40)
    _, graph, _ = h.pcg_solve(K, Y.repeat(1, 11).contiguous(), lam, tol=tol, maxit=60000, refine_max=40)
    assert max(rel) <= tol
    M = K.double()
    M.diagonal().add_(lam)
    ev = torch.linalg.eigvalsh(M)
    want = torch.linalg.solve(M, Y)
    assert float((A - want).norm()) <= float(ev[-1] / ev[0]) * tol * float(want.norm())
    assert its <= 1.2 * graph + 64


@pytest.mark.parametrize("n,dim,ell,ridge", CASES + [(1000, 4, 3.0, 1e-5), (4500, 16, 8.0, 1e-5)])
def test_plain_fp32_solve(n, dim, ell, ridge):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_05420_gb300.api import Handle

    h = Handle()
    K, lam, Y = _problem(n, dim, ell, ridge, 3)
    kw = dict(prec="plain_fp32", tol=1e-3, maxit=30000, allow_not_converged=True)
    _, _, rel = h.pcg_solve(K, Y, lam, **kw)
    _, _, graph = h.pcg_solve(K, Y.repeat(1, 11).contiguous(), lam, **kw)
    assert max(rel) <= 3 * max(graph)


@pytest.mark.parametrize("n,dim,ell,ridge", [(600, 8, 4.0, 1e-5), (1000, 4, 3.0, 1e-4)])
def test_long_sweeps_settle_early(n, dim, ell, ridge):
    """A refinement sweep that gets long stops at the graph-replayed run's level
    (3e-2), so that the solve takes no more iterations than that run: at most
    256 in the first sweep, before it shows, and 5 % for the rounding."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_05420_gb300.api import Handle

    h = Handle()
    K, lam, Y = _problem(n, dim, ell, ridge, 3)
    _, its, _ = h.pcg_solve(K, Y, lam, tol=1e-8, maxit=60000, refine_max=40)
    _, graph, _ = h.pcg_solve(K, Y.repeat(1, 11).contiguous(), lam, tol=1e-8, maxit=60000, refine_max=40)
    assert its <= 1.05 * graph + 256
