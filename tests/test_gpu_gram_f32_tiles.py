"""Float32 CUDA-core Gram products (mixed plans without the tensor-core Gram) at the sizes
where their tile shape changes.

Entries, operator and scaled interval are chosen so that every product and every sum is
exact in float32 (V_0 of +-1, V_1 of small multiples of 1/8): the moments of degree 2,
X_0 = V_0^T V_0, X_1 = V_1^T V_0 and X_2 = 2 V_1^T V_1 - X_0, must equal the integers' to
the bit.  Sizes in 64-wide tiles, ragged and whole, and beside them in 32- and 16-wide ones
(too few tiles, too much padding).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402
from oracle import ssm_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nv", [(63, 65, 384), (63, 65, 512), (63, 65, 401), (63, 65, 300), (63, 65, 257),
                                      (127, 129, 200), (127, 129, 160), (127, 129, 129), (31, 33, 700), (9, 7, 40)])
def test_float32_gram_tiles(nx, ny, nv):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    rng = np.random.default_rng(nx + nv)
    n = nx * ny
    st = wl.Stencil(dims=(nx, ny, 1), periodic=(True, False, False), diag=rng.integers(-3, 4, n).astype(float),
                    offdiag=(-1.0, 2.0, 0.0))
    W = rng.choice([-1.0, 1.0], size=(n, nv))
    plan = S.ssm_plan_create(stencil=st, n_v=nv, degree=2, precision="mixed", options=1, lo=-16.0, hi=16.0)
    X = S.ssm_moments(plan, torch.from_numpy(W).cuda(), return_moments=True).cpu().numpy()
    plan.close()
    c = wl.stencil_to_csr(st)
    V = O.csr_matrix(c.n, c.rowptr, c.colind, c.val) @ W / 16.0
    assert np.array_equal(X[0], W.T @ W)
    assert np.array_equal(X[1], V.T @ W)
    assert np.array_equal(X[2], 2.0 * (V.T @ V) - W.T @ W)
