"""The grid barriers of the resident CG run: a wait limit of 0 polls makes the
first one give up, nk_pcg_solve returns NK_ERR_TIMEOUT, and with the default
limit back the next solve on the same handle is right.  With K in shared memory,
partly read from memory, and in every precision that takes the run."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,prec", [(700, 3, "mixed"), (700, 3, "plain_fp32"), (2300, 20, "mixed"), (3500, 5, "mixed")])
def test_wait_limit_runs_out_and_the_handle_recovers(n, r, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_05420_gb300._lib import NK_ERR_TIMEOUT, NkError
    from paper_2303_05420_gb300.api import Handle

    h = Handle()
    rng = np.random.default_rng(n)
    a = torch.tensor(rng.standard_normal((n, 24)), device="cuda")
    K = (a @ a.T / 24 + torch.eye(n, dtype=torch.float64, device="cuda")).float()
    K = (K + K.T) / 2
    Y = torch.tensor(rng.standard_normal((n, r)), device="cuda")
    h.set_wait_limit(0)
    with pytest.raises(NkError) as ei:
        h.pcg_solve(K, Y, 0.5, prec=prec, tol=1e-5)
    assert ei.value.status == NK_ERR_TIMEOUT
    h.set_wait_limit(-1)
    A, _, rel = h.pcg_solve(K, Y, 0.5, prec=prec, tol=1e-5)
    assert max(rel) <= 1e-5
    M = K.double()
    M.diagonal().add_(0.5)
    assert float((M @ A - Y).norm()) <= 1.1e-5 * float(Y.norm())
