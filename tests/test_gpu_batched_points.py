"""Batched plans with more sweep points a matrix than a batch of pencils holds (2 GiB of
K and K_Z: 128 points at 1024 probes).

The call must equal two calls of half the points each, which fit, bit for bit: every point's
arithmetic is the same.  Most points lie outside the spectrum (nothing is kept there, which
costs nothing); those inside sit at both ends of the range, on either side of the chunk's
edge.  Shared and separate coefficient tables, float64 and mixed plans, damping.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shared,damping", [("fp64", True, None), ("mixed", False, "jackson"),
                                                      ("mixed", True, None)])
def test_points_beyond_one_batch(precision, shared, damping):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    nv, n_tp, M, sigma = 1024, 130, 4, 0.3
    csrs = [wl.er_normalized_laplacian(n, 6.0, 40 + n) for n in (70, 41)]
    plan = S.ssm_plan_create_batched(csrs, n_v=nv, degree=M, precision=precision, damping=damping)
    W = np.vstack([wl.random_block(c.n, nv, 50 + c.n, "rademacher") for c in csrs])
    S.ssm_moments(plan, torch.from_numpy(W).cuda())
    t = np.full((2, n_tp), 500.0)
    t[:, [0, 1, 64, 65, 127, 128, 129]] = [0.4, 0.9, 1.1, 1.3, 0.6, 1.0, 1.6]
    if not shared:
        t[1] += 0.03
    whole = S.ssm_dos(plan, torch.from_numpy(t.reshape(-1)).cuda(), sigma)
    halves = [S.ssm_dos(plan, torch.from_numpy(np.ascontiguousarray(q).reshape(-1)).cuda(), sigma)
              for q in (t[:, :65], t[:, 65:])]
    plan.close()
    for k in range(3):
        got = whole[k].reshape(2, n_tp, -1)
        ref = torch.cat([h[k].reshape(2, 65, -1) for h in halves], dim=1)
        assert torch.equal(got, ref), k
    assert int((whole[2][:, 0] > 0).sum()) == 14
    assert bool(torch.isfinite(whole[0]).all())
