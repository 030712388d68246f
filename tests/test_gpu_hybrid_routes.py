"""Hybrid columns on mixed plans: the factored routes of the solver against the oracle.

The RESS-DGC line of a mixed plan with hybrid columns is compared with the oracle's Alg. 7
loop on the plan's own moments and rounding floor, so only the assembly and the solve are
tested: relative L1 1e-7 on the points that the oracle does not flag as within 1e-8 of an
Alg. 4 threshold (float64 arithmetic amplified by at most 1 / tau), equal kept ranks.
The cases reach every route: everything kept with every eigenvalue inside the range filter
and with some outside, few directions dropped (duplicated probe columns), a part kept,
nothing kept, and more hybrid columns than low-rank ones.  Sweep points reach five sigma
past the spectrum (coefficients below 2^-126, farther out, are below what the assembly's
scales hold).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402
from oracle import ssm_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv,nvh,dup,sigma", [(1, 3, False, 0.3), (33, 8, False, 0.1), (40, 100, False, 0.2),
                                              (128, 70, False, 0.3), (100, 30, True, 0.3), (150, 50, True, 0.15)])
def test_hybrid_routes_match_oracle_on_own_moments(nv, nvh, dup, sigma):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    st = wl.anderson2d(40, 4600 + nv)
    W = wl.random_block(st.n, nv + nvh, 4700 + nv, "rademacher")
    if dup:
        W[:, 1] = W[:, 0]
        W[:, 3] = W[:, 2]
    M = 120
    plan = S.ssm_plan_create(stencil=st, n_v=nv, n_vh=nvh, degree=M, precision="mixed")
    info = S.ssm_plan_info(plan)
    X = S.ssm_moments(plan, torch.from_numpy(W).cuda(), return_moments=True).cpu().numpy()
    t = np.linspace(info["lo"] - 5 * sigma, info["hi"] + 5 * sigma, 97)
    ss, _, rk = (x.cpu().numpy() for x in S.ssm_dos(plan, torch.from_numpy(t).cuda(), sigma))
    plan.close()
    tab = O.coefficient_tables(t, M, sigma, st.n, info["a"], info["b"])
    r = O.ress_from_moments(X, tab, nv, O.g_max(sigma, st.n), flag_eps=1e-8, eps_floor=2.0**-36)
    ok = ~r["flagged"]
    assert ok.mean() >= 0.9
    assert np.array_equal(rk[ok, 0], r["rank_s"][ok])
    assert np.array_equal(rk[ok, 1], r["rank_xi"][ok])
    assert O.relative_l1_error(ss[ok], r["dos_ss"][ok]) <= 1e-7
