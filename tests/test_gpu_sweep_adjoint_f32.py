"""The adjoint step's sweep over the planes of a grid in float32 (mixed plans).

The gradient of a mixed stencil plan against that of a float64 one, 1e-4 of the largest
entry (the tolerance of the float32 recurrence), on blocks of 12 MiB or more, where the
sweep runs, for every number of lanes a row takes, ragged and full, on open, periodic and
inactive axes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [((64, 57, 55), (True, False, True), (-1.0, -0.7, -1.2), 14),
         ((33, 56, 64), (False, True, True), (-1.0, -0.7, -1.2), 29),
         ((17, 57, 55), (True, True, False), (-1.0, 0.0, -1.2), 64),
         ((16, 41, 43), (False, False, False), (-1.0, -0.7, -1.2), 125)]


@pytest.mark.parametrize("kind", ["scalars", "matrices"])
@pytest.mark.parametrize("dims,per,off,nv", CASES, ids=[f"{d[0]}x{d[1]}x{d[2]}-{n}" for d, _, _, n in CASES])
def test_sweep_adjoint_float32(dims, per, off, nv, kind):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    n = dims[0] * dims[1] * dims[2]
    assert n * ((nv + 3) // 4) * 16 >= 12 << 20
    rng = np.random.default_rng(n + nv)
    st = wl.Stencil(dims=dims, periodic=per, diag=rng.uniform(-2, 2, n), offdiag=off)
    M = 10
    W = torch.from_numpy(rng.standard_normal((n, nv))).cuda()
    G = torch.from_numpy(rng.standard_normal(M + 1 if kind == "scalars" else (M + 1, nv, nv))).cuda()
    got = []
    for precision in ("mixed", "fp64"):
        plan = S.ssm_plan_create(stencil=st, n_v=nv, degree=M, precision=precision, options=2, lo=-8.5, hi=8.5)
        S.ssm_moments(plan, W)
        got.append([x.cpu().numpy() for x in S.ssm_moments_adjoint(plan, G)])
        plan.close()
    (d32, o32), (d64, o64) = got
    assert np.abs(d32 - d64).max() <= 1e-4 * np.abs(d64).max()
    assert np.abs(o32 - o64).max() <= 1e-4 * np.abs(o64).max()
