"""CUDA-core Gram products at the edges of their tile shapes (ssm_gram_pair).

The launch picks 32 x 32, 16 x 16 or 8 x 8 output tiles from the number of columns and
row slices; every shape sums each output in row order.  Reference: numpy float64.  A
chain of n fused multiply-adds is within n eps sum_r |a_ri b_rj| of the exact sum, and so
is the reference's, which gives the tolerance.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(1, 1), (31, 8), (33, 9), (512, 7), (513, 17), (1024, 40), (2000, 31),
                                       (4097, 33), (6000, 64), (20000, 65), (40000, 200)])
@pytest.mark.parametrize("odd", [False, True])
def test_gram_pair_tile_edges(rows, cols, odd):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    rng = np.random.default_rng(rows + cols)
    A, B = rng.standard_normal((rows, cols)), rng.standard_normal((rows, cols))
    aa, ab = S.ssm_gram_pair(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda() if odd else None)
    tol = 2 * rows * 2.0**-52
    assert np.all(np.abs(aa.cpu().numpy() - A.T @ A) <= tol * (np.abs(A).T @ np.abs(A)))
    assert torch.equal(aa, aa.T)
    if odd:
        assert np.all(np.abs(ab.cpu().numpy() - A.T @ B) <= tol * (np.abs(A).T @ np.abs(B)))
