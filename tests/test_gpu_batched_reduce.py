"""Slab sums of batched mixed plans, few and many slabs a matrix.

Up to four slabs a matrix on average one thread sums an element (its eight chains one
after the other), beyond that eight warps share it.  The cases lie on both sides, with one
probe, a ragged count, one matrix of more slabs than chains among small ones, and more
pairs than one CTA holds.  Moments within 2e-5 of max|X| of the oracle's float64 loop (the
split-bf16 Gram error of mixed plans), and exactly symmetric.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402
from oracle import ssm_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,n_v", [((300,), 5), ((40,) * 9, 1), ((33, 64, 12), 33),
                                       ((400,) + (40,) * 30, 17), ((2000,) + (40,) * 20, 16)])
def test_moments_few_and_many_slabs(sizes, n_v):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    csrs = [wl.er_normalized_laplacian(n, 6.0, 140 + k) for k, n in enumerate(sizes)]
    M = 14
    plan = S.ssm_plan_create_batched(csrs, n_v=n_v, degree=M, precision="mixed")
    Ws = [wl.random_block(c.n, n_v, 177 + k, "rademacher") for k, c in enumerate(csrs)]
    X = S.ssm_moments(plan, torch.from_numpy(np.vstack(Ws)).cuda(), return_moments=True).cpu().numpy()
    for b, c in enumerate(csrs):
        i = S.ssm_batch_info(plan, b)
        Xr = O.moments_direct(O.transform(O.csr_matrix(c.n, c.rowptr, c.colind, c.val), i["a"], i["b"]), Ws[b], M)
        assert np.max(np.abs(X[b] - Xr)) <= 2e-5 * np.max(np.abs(Xr)), b
        assert np.array_equal(X[b], X[b].transpose(0, 2, 1))
    plan.close()
