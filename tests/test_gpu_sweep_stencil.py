"""The kernels that sweep the planes of a grid, at the edges of their tiles.

Forward: mixed moments against a float64 plan's (the per-item kernel), 2e-5 of the largest
entry (the tolerance of the float32 recurrence).  Grids of 64 MiB a block or more (where the
sweep runs) whose axes 1 and 2 fill 8 x 8 tiles exactly, leave ragged ones, wrap inside a
ragged tile or past an exact one, have open edges, an inactive axis, more planes than one
run, and column chunks that divide the tile evenly and unevenly.

Adjoint: the float64 gradient of a stencil plan against that of a CSR plan of the same
operator (another kernel; sums of <= 60 steps in float64, 1e-11 of the largest entry), for
every number of lanes a row takes and on open, periodic and inactive axes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [
    ((5, 120, 112), (True, True, True), (-1.0, -0.7, -1.2), 256),
    ((5, 119, 127), (False, False, False), (-1.0, -0.7, -1.2), 250),
    ((33, 47, 55), (True, False, True), (-1.0, -0.7, -1.2), 200),
    ((16, 92, 95), (False, True, False), (-1.0, -0.7, -1.2), 128),
    ((41, 64, 33), (True, True, True), (-1.0, 0.0, -1.2), 215),
]


@pytest.mark.parametrize("dims,per,off,nv", SHAPES, ids=[f"{d[0]}x{d[1]}x{d[2]}-{n}" for d, _, _, n in SHAPES])
def test_sweep_stencil_moments(dims, per, off, nv):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    n = dims[0] * dims[1] * dims[2]
    assert n * ((nv + 3) // 4) * 16 >= 64 << 20
    rng = np.random.default_rng(n + 7)
    st = wl.Stencil(dims=dims, periodic=per, diag=rng.uniform(-2, 2, n), offdiag=off)
    M = 12
    W = torch.from_numpy(wl.random_block(n, nv, 41 + n, "gaussian")).cuda()
    X = []
    for precision in ("mixed", "fp64"):
        plan = S.ssm_plan_create(stencil=st, n_v=nv, degree=M, precision=precision)
        X.append(S.ssm_moments(plan, W, return_moments=True))
        plan.close()
    assert float((X[0] - X[1]).abs().max()) <= 2e-5 * float(X[1].abs().max())


ADJ = [((23, 119, 143), (True, False, True), (-1.0, -0.7, -1.2), 6), ((33, 56, 63), (False, True, True), (-1.0, -0.7, -1.2), 15),
       ((16, 60, 64), (True, True, True), (-1.0, -0.7, -1.2), 31), ((15, 51, 47), (False, False, False), (-1.0, -0.7, -1.2), 49),
       ((36, 31, 24), (True, True, True), (-1.0, 0.0, -1.2), 64), ((5, 8, 15), (True, False, True), (-1.0, -0.7, -1.2), 6)]


@pytest.mark.parametrize("kind", ["scalars", "matrices"])
@pytest.mark.parametrize("dims,per,off,nv", ADJ, ids=[f"{d[0]}x{d[1]}x{d[2]}-{n}" for d, _, _, n in ADJ])
def test_sweep_adjoint_matches_csr_adjoint(dims, per, off, nv, kind):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    n = dims[0] * dims[1] * dims[2]  # all but the last run the sweep (12 MiB a block or more)
    assert n * ((nv + 1) // 2) * 16 >= 12 << 20 or dims == ADJ[-1][0]
    rng = np.random.default_rng(n + nv)
    st = wl.Stencil(dims=dims, periodic=per, diag=rng.uniform(-2, 2, n), offdiag=off)
    M = 10
    W = torch.from_numpy(rng.standard_normal((n, nv))).cuda()
    G = rng.standard_normal(M + 1 if kind == "scalars" else (M + 1, nv, nv))
    lo, hi = -8.5, 8.5
    got = []
    for op in (dict(stencil=st), dict(csr=wl.stencil_to_csr(st))):
        plan = S.ssm_plan_create(**op, n_v=nv, degree=M, precision="fp64", options=2, lo=lo, hi=hi)
        S.ssm_moments(plan, W)
        got.append([x.cpu().numpy() for x in S.ssm_moments_adjoint(plan, torch.from_numpy(G).cuda())])
        plan.close()
    (dd, do), (cd, cv) = got
    csr = wl.stencil_to_csr(st)
    rows = np.repeat(np.arange(n), np.diff(csr.rowptr))
    a, b = np.array(np.unravel_index(rows, dims)), np.array(np.unravel_index(csr.colind, dims))
    scale = max(np.abs(cd).max(), np.abs(cv).max())
    assert np.abs(dd - cd).max() <= 1e-11 * scale
    for ax in range(3):
        if off[ax] == 0.0:
            continue  # no stored entries of a zero coupling
        along = (a[ax] != b[ax])
        assert abs(do[ax] - cv[along].sum()) <= 1e-11 * scale * n
