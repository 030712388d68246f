"""Many sweep points of few probes, and many small matrices: the kernels that only large
counts reach.

Solver, a warp a point (n_v <= 32, eight points an SM): DOS and kept ranks of two graphs in
a batched mixed plan, and of one in a single plan, against the oracle's Alg. 7 loop on the
plan's own moments and rounding floor: relative L1 1e-7 on the points that the oracle does
not flag as within 1e-8 of an Alg. 4 threshold (float64 arithmetic amplified by at most
1 / tau), equal ranks.  Points reach five sigma past the spectrum, where nothing is kept;
inside everything is kept, or a part, with all eigenvalues inside the range filter or some
outside.  On these points a float64 plan's floor lets rounding of the coefficients through
(the ranks after the range filter differ from the oracle's whichever solver runs), so
there the call is compared with calls of fewer points, which a CTA a point solves from the
same matrices: equal ranks, 1e-7 of the largest value.

Gram products with two and four CTAs an SM (slabs for two and four an SM, n_tot <= 64 and
<= 32): moments of several hundred small graphs within 2e-5 of max|X| of the oracle's
float64 loop (the split-bf16 Gram error of mixed plans).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl  # noqa: E402
from oracle import ssm_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1504_07690_gb300 as S

    return S


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("batched", [True, False])
@pytest.mark.parametrize("n_v", [1, 17, 31, 32])
def test_warp_per_point_solver_matches_oracle(S, n_v, batched):
    M, sigma = 200, 0.05
    csrs = [wl.er_normalized_laplacian(n, 6.0, 300 + n) for n in ((240, 130) if batched else (130,))]
    Ws = [wl.random_block(c.n, n_v, 310 + c.n, "rademacher") for c in csrs]
    kw = dict(n_v=n_v, degree=M, precision="mixed")
    if batched:
        plan = S.ssm_plan_create_batched(csrs, **kw)
        infos = [S.ssm_batch_info(plan, b) for b in range(2)]
    else:
        plan = S.ssm_plan_create(csr=csrs[0], **kw)
        infos = [S.ssm_plan_info(plan)]
    n_tp = 8 * _sms() // len(csrs) + 5
    t = np.stack([np.linspace(i["lo"] - 5 * sigma, i["hi"] + 5 * sigma, n_tp) for i in infos])
    X = S.ssm_moments(plan, torch.from_numpy(np.vstack(Ws)).cuda(), return_moments=True).cpu().numpy()
    ss, _, rk = (x.cpu().numpy() for x in S.ssm_dos(plan, torch.from_numpy(t.reshape(-1)).cuda(), sigma))
    plan.close()
    kinds = set()
    for b, (c, i) in enumerate(zip(csrs, infos)):
        tab = O.coefficient_tables(t[b], M, sigma, c.n, i["a"], i["b"])
        r = O.ress_from_moments(X[b] if batched else X, tab, n_v, O.g_max(sigma, c.n), flag_eps=1e-8, eps_floor=2.0**-36)
        ok, at = ~r["flagged"], slice(b * n_tp, (b + 1) * n_tp)
        assert ok.mean() >= 0.9
        assert np.array_equal(rk[at][ok, 0], r["rank_s"][ok])
        assert np.array_equal(rk[at][ok, 1], r["rank_xi"][ok])
        assert O.relative_l1_error(ss[at][ok], r["dos_ss"][ok]) <= 1e-7
        kinds |= {(0 if s == 0 else (2 if s == n_v else 1), bool(x < s)) for s, x in zip(r["rank_s"], r["rank_xi"])}
    assert {(0, False), (2, False), (2, True)} <= kinds and (n_v == 1 or {(1, False), (1, True)} <= kinds)


@pytest.mark.parametrize("n_v", [1, 17, 31, 32])
def test_warp_per_point_solver_matches_the_cta_solver(S, n_v):
    c = wl.er_normalized_laplacian(130, 6.0, 430)
    plan = S.ssm_plan_create(csr=c, n_v=n_v, degree=200, precision="fp64")
    info, sigma = S.ssm_plan_info(plan), 0.05
    t = torch.linspace(info["lo"] - 5 * sigma, info["hi"] + 5 * sigma, 8 * _sms() + 5, dtype=torch.float64).cuda()
    S.ssm_moments(plan, torch.from_numpy(wl.random_block(c.n, n_v, 440, "rademacher")).cuda())
    ss, _, rk = S.ssm_dos(plan, t, sigma)
    parts = [S.ssm_dos(plan, q.contiguous(), sigma) for q in t.split(400)]
    plan.close()
    assert torch.equal(rk, torch.cat([p[2] for p in parts]))
    ref = torch.cat([p[0] for p in parts])
    assert float((ss - ref).abs().max()) <= 1e-7 * float(ref.abs().max())


@pytest.mark.parametrize("n_v,per_sm", [(1, 4), (31, 4), (32, 4), (32, 2), (33, 4), (64, 2)])
def test_gram_of_many_small_matrices(S, n_v, per_sm):
    B, M = per_sm * _sms() + 3, 6
    csrs = [wl.er_normalized_laplacian(33 + (17 * k) % 90, 6.0, 500 + k % 20) for k in range(B)]
    Ws = [wl.random_block(c.n, n_v, 600 + k, "rademacher") for k, c in enumerate(csrs)]
    plan = S.ssm_plan_create_batched(csrs, n_v=n_v, degree=M, precision="mixed")
    X = S.ssm_moments(plan, torch.from_numpy(np.vstack(Ws)).cuda(), return_moments=True).cpu().numpy()
    for b, c in enumerate(csrs):
        i = S.ssm_batch_info(plan, b)
        Xr = O.moments_direct(O.transform(O.csr_matrix(c.n, c.rowptr, c.colind, c.val), i["a"], i["b"]), Ws[b], M)
        assert np.max(np.abs(X[b] - Xr)) <= 2e-5 * np.max(np.abs(Xr)), b
        assert np.array_equal(X[b], X[b].transpose(0, 2, 1))
    plan.close()
