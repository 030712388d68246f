"""Float32 stencil steps of large 3D grids at the row widths where the kernel changes.

Mixed moments of a stencil plan against those of a mixed CSR plan of the same operator
(another step kernel, the same Gram products): rounding of float32 steps only, 1e-5 of the
largest entry (four steps of at most 8 operations an element, each error growing linearly
with the steps after it and entering a product twice).  Blocks of 64 MiB or more: row
widths in 16-byte chunks below the sweep kernel's range (11), its narrowest even width
(12), widths between that leave idle columns (13, 23), and one, two and three idle columns
in the last tile of four (31, 26, 33).

The same for grids of large planes, where ragged tiles run the sweep too: wrapped and open
edges in a ragged tile, an inactive axis, two runs of planes, and one of small planes,
where they do not.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(dims, per, off, nv):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    n = dims[0] * dims[1] * dims[2]
    assert n * ((nv + 3) // 4) * 16 >= 64 << 20
    st = wl.Stencil(dims=dims, periodic=per, diag=np.random.default_rng(nv).uniform(-2, 2, n), offdiag=off)
    W = torch.from_numpy(wl.random_block(n, nv, 43 + nv, "gaussian")).cuda()
    X = []
    for op in (dict(stencil=st), dict(csr=wl.stencil_to_csr(st))):
        plan = S.ssm_plan_create(**op, n_v=nv, degree=8, precision="mixed", lo=-8.0, hi=8.0)
        X.append(S.ssm_moments(plan, W, return_moments=True))
        plan.close()
    assert float((X[0] - X[1]).abs().max()) <= 1e-5 * float(X[1].abs().max())


@pytest.mark.parametrize("nv", [44, 48, 49, 91, 122, 104, 130])
def test_sweep_widths(nv):
    _check((71, 72, 80), (True, False, True), (-1.0, -0.7, -1.2), nv)


@pytest.mark.parametrize("dims,per,off,nv", [((8, 101, 93), (True, True, True), (-1.0, -0.7, -1.2), 256),
                                             ((9, 99, 102), (False, True, False), (-1.0, -0.7, -1.2), 213),
                                             ((9, 101, 99), (True, True, True), (-1.0, 0.0, -1.2), 215),
                                             ((17, 211, 213), (True, True, False), (-1.0, -0.7, -1.2), 48),
                                             ((61, 60, 60), (True, False, True), (-1.0, -0.7, -1.2), 128)])
def test_sweep_planes(dims, per, off, nv):
    _check(dims, per, off, nv)
