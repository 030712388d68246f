"""Float-pair CSR step: rows a thread takes from one to eight with the size of the block.

Moments of fp64_tc plans within 1e-11 of max|X| of a float64 plan's on the same operator
(the error of the float-pair recurrence and its Gram products), at sizes on both sides of
each change of the launch: 8, 4, 2 and 1 rows a thread, blocks of one chunk and wide ones,
rows that do not fill the last CTA.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_v", [(45, 3), (30011, 8), (30011, 36), (30011, 50), (30011, 101)])
def test_fp64tc_csr_rows(n, n_v):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    c = wl.er_normalized_laplacian(n, 8.0, 70 + n)
    W = torch.from_numpy(wl.random_block(n, n_v, 71 + n, "gaussian")).cuda()
    X = []
    for precision in ("fp64_tc", "fp64"):
        plan = S.ssm_plan_create(csr=c, n_v=n_v, degree=8, precision=precision)
        X.append(S.ssm_moments(plan, W, return_moments=True))
        plan.close()
    assert float((X[0] - X[1]).abs().max()) <= 1e-11 * float(X[1].abs().max())
