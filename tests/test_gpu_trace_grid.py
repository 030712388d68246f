"""Alg. 8's quadrature weights (ssm_trace_weights) at grid sizes around a warp and odd ones.

The deconvolution takes its twiddles from a table and forms the quotients once.  With a
Gaussian of 0.6 grid spacings the kernel's DFT stays above 1/6 of its peak, so the two
direct DFTs of n terms are within a few n^2 eps max|h| of the oracle's FFTs: 20 n^2 2^-52.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402
from oracle import ssm_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_t", [2, 31, 32, 33, 257, 1000])
def test_trace_weights_grid_sizes(n_t):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    st = wl.make_operator("lap2d_dirichlet_32", nx=6)
    plan = S.ssm_plan_create(stencil=st, n_v=2, degree=4)
    info = S.ssm_plan_info(plan)
    dx = 2.0 * 0.5 * (info["hi"] - info["lo"]) / 0.93 / n_t
    x, w = S.ssm_trace_weights(plan, lambda v: math.exp(-0.5 * v), n_t, 0.6 * dx)
    plan.close()
    xr, dxr, ft, h = O.deconvolve_h(lambda v: np.exp(-0.5 * v), n_t, info["lo"], info["hi"], 0.6 * dx)
    assert np.max(np.abs(np.asarray(x) - xr)) <= 1e-12 * np.max(np.abs(xr))
    assert np.max(np.abs(np.asarray(w) - st.n * dxr * ft)) <= 20 * n_t**2 * 2.0**-52 * st.n * dxr * np.max(np.abs(h))
