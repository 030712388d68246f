"""Per-point solver above 256 probes, where a CTA has fewer threads than K_W(t) columns.

40 x 40 Anderson model, degree 80, 13 points over the spectrum: every case has points that
keep a part of the directions (reduction of K_W) and points with eigenvalues outside the
range filter (reduction of the pencil), with few and with many directions dropped.  257 is
the last size with a thread for each column of the trailing block.

Tolerances: float64 plans and explicit blocks max(1e-10, 10 x the relative L1 spread
between two float64 evaluations of the same estimator by the oracle), mixed plans 1e-7
against the oracle on the plan's own moments and rounding floor (float64 arithmetic
amplified by at most 1 / tau); on the points that the oracle does not flag as within 1e-8
of an Alg. 4 threshold, where the kept ranks must be equal.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402
from oracle import ssm_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu

M, SIGMA, N_T = 80, 0.3, 13


@pytest.mark.parametrize("form,nv,nvh", [("fp64", 257, 0), ("fp64", 258, 0), ("fp64", 300, 0), ("fp64", 513, 0),
                                         ("mixed", 258, 0), ("mixed", 300, 0), ("mixed", 258, 40), ("mixed", 300, 310),
                                         ("pinv", 300, 0), ("explicit", 300, 0)])
def test_more_probes_than_threads(form, nv, nvh):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    st = wl.anderson2d(40, 4800 + nv)
    csr = wl.stencil_to_csr(st)
    A = O.csr_matrix(csr.n, csr.rowptr, csr.colind, csr.val)
    W = wl.random_block(st.n, nv + nvh, 4900 + nv, "rademacher")
    deg = M // 2 if form == "explicit" else M  # (the same pencils)
    plan = S.ssm_plan_create(stencil=st, n_v=nv, n_vh=nvh, degree=deg, precision="mixed" if form == "mixed" else "fp64",
                             options=8 if form == "pinv" else 0)
    info = S.ssm_plan_info(plan)
    t = np.linspace(info["lo"], info["hi"], N_T)
    Wd, td = torch.from_numpy(W).cuda(), torch.from_numpy(t).cuda()
    kw = dict(interval=(info["a"], info["b"]), flag_eps=1e-8, estimator="pinv" if form == "pinv" else "alg4")
    if form == "explicit":
        ss, rank = (x.cpu().numpy() for x in S.ssm_dos_explicit(plan, Wd, td, SIGMA))
        r = O.ss_dgc(A, W, t, deg, SIGMA, **kw)
        r2 = O.ress_dgc(A, W, nv, t, M, SIGMA, moments="doubling", **kw)
    else:
        X = S.ssm_moments(plan, Wd, return_moments=True).cpu().numpy()
        ss, _, rank = (x.cpu().numpy() for x in S.ssm_dos(plan, td, SIGMA))
        if form == "mixed":
            tab = O.coefficient_tables(t, M, SIGMA, st.n, info["a"], info["b"])
            r = r2 = O.ress_from_moments(X, tab, nv, O.g_max(SIGMA, st.n), flag_eps=1e-8, eps_floor=2.0**-36)
        else:
            r = O.ress_dgc(A, W, nv, t, M, SIGMA, **kw)
            r2 = O.ress_dgc(A, W, nv, t, M, SIGMA, moments="doubling", **kw)
    plan.close()
    ok = ~r["flagged"] & ~r2["flagged"]
    rs, rx = r["rank_s"], r["rank_xi"]
    assert ok.mean() >= 0.8
    assert np.any(ok & (rs > 0) & (rs < nv) & (3 * (nv - rs) < rs)) and np.any(ok & (rs > 0) & (3 * (nv - rs) >= rs))
    assert form == "pinv" or np.any(ok & (rx < rs))
    assert np.array_equal(rank[ok, 0], rs[ok])
    assert np.array_equal(rank[ok, 1], rx[ok])
    err = O.relative_l1_error(ss[ok], r["dos_ss"][ok])
    tol = 1e-7 if form == "mixed" else max(1e-10, 10.0 * O.relative_l1_error(r2["dos_ss"][ok], r["dos_ss"][ok]))
    assert err <= tol, (err, tol)
