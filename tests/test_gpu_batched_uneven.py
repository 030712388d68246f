"""Slab sums of uneven batches: large matrices among small ones, in any place.

A matrix of many slabs has its sums formed by eight warps an element, one of few by a
thread, side by side in one plan.  The large matrices come first, last and in the middle,
with one probe, a ragged count and one that takes separate even and odd products.
Moments within 2e-5 of max|X| of the oracle's float64 loop (the split-bf16 Gram error of
mixed plans), and exactly symmetric.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402
from oracle import ssm_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,n_v", [((40,) * 9 + (2000,) + (60,) * 7 + (900,), 17), ((33, 3000, 64), 1),
                                       ((1500,) + (45,) * 20 + (1200,), 130), ((50,) * 12 + (2500,), 64)])
def test_moments_of_uneven_batches(sizes, n_v):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    csrs = [wl.er_normalized_laplacian(n, 6.0, 240 + k) for k, n in enumerate(sizes)]
    M = 10
    plan = S.ssm_plan_create_batched(csrs, n_v=n_v, degree=M, precision="mixed")
    Ws = [wl.random_block(c.n, n_v, 277 + k, "rademacher") for k, c in enumerate(csrs)]
    X = S.ssm_moments(plan, torch.from_numpy(np.vstack(Ws)).cuda(), return_moments=True).cpu().numpy()
    for b, c in enumerate(csrs):
        i = S.ssm_batch_info(plan, b)
        Xr = O.moments_direct(O.transform(O.csr_matrix(c.n, c.rowptr, c.colind, c.val), i["a"], i["b"]), Ws[b], M)
        assert np.max(np.abs(X[b] - Xr)) <= 2e-5 * np.max(np.abs(Xr)), b
        assert np.array_equal(X[b], X[b].transpose(0, 2, 1))
    plan.close()
