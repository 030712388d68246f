"""ssm_dos_explicit: a point's result does not depend on the chunks of the call, which go by
the free device memory, also where the solver's shape goes by the number of points.

Calls just above the number of points up to which a point gets more threads (two an SM) in
chunks below it, at probe counts with and without that rule; bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_v", [40, 66, 100])
def test_chunks_of_large_calls_give_the_same_result(n_v):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    n_t = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 6
    st = wl.laplacian2d_dirichlet_potential(13, 186)
    W = torch.from_numpy(wl.random_block(st.n, n_v, 187)).cuda()
    plan = S.ssm_plan_create(stencil=st, n_v=n_v, degree=30, precision="fp64")
    info = S.ssm_plan_info(plan)
    t = torch.from_numpy(np.linspace(info["lo"], info["hi"], n_t)).cuda()
    d_all, r_all = S.ssm_dos_explicit(plan, W, t, 0.3)
    try:
        S.ssm_debug_explicit_chunk(n_t // 2)
        d_chk, r_chk = S.ssm_dos_explicit(plan, W, t, 0.3)
    finally:
        S.ssm_debug_explicit_chunk(0)
    plan.close()
    assert torch.equal(d_all, d_chk) and torch.equal(r_all, r_chk)
