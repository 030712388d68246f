"""ssm_stats.launches counts both kernels of a solve that runs a warp a point first (eight
points an SM and more, n_v <= 32): one more than a call of one point less, for a single
and a batched plan."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
def test_small_point_solve_counts_two_launches(batched):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    c = wl.er_normalized_laplacian(60, 6.0, 11)
    n_v, edge = 3, 8 * torch.cuda.get_device_properties(0).multi_processor_count
    if batched:
        plan = S.ssm_plan_create_batched([c], n_v=n_v, degree=10, precision="mixed")
    else:
        plan = S.ssm_plan_create(csr=c, n_v=n_v, degree=10, precision="mixed")
    S.ssm_moments(plan, torch.from_numpy(wl.random_block(c.n, n_v, 12, "rademacher")).cuda())

    def launches(n_t):
        t = torch.from_numpy(np.linspace(0.1, 1.9, n_t)).cuda()
        before = S.ssm_stats_get(plan)["launches"]
        S.ssm_dos(plan, t, 0.2)
        return S.ssm_stats_get(plan)["launches"] - before

    launches(7)  # the first call prepares the moments' slices
    below, at = launches(edge - 1), launches(edge)
    plan.close()
    assert at == below + 1
