"""What the library is timed on: density-of-states work as its users call it.

A case is one call sequence of the public API on synthetic operators of this
repository's kinds (2D and 3D finite-difference Hamiltonians with a random
potential, normalised Laplacians of random graphs).  ``prepare`` makes what a
program holds before the call (operator, probe block, plan), ``run`` is the call,
``work`` the bytes and operations it cannot do without, and ``exact`` the same
result in plain float64 torch, by the definitions (Chebyshev moments by the
three-term loop, the per-point pencils by dense eigenvalues).

Tasks
    dos       ssm_moments, then ssm_dos: both estimates and the kept ranks
    kpm       ssm_moments, then the KPM line alone (no pencils)
    moments   ssm_moments with the moments copied out, then the KPM line
    trace     ssm_trace_f on a plan that holds its moments
    gradient  forward and backward of a loss of the KPM line (torch.autograd)
    explicit  ssm_dos_explicit (filtered blocks formed explicitly)
    batch     ssm_moments and ssm_dos of many small operators in one plan
    gram      ssm_gram_pair on two blocks of a caller's own recurrence
"""
import math

import numpy as np
import torch

import paper_1504_07690_gb300 as S
import workloads as wl

F64 = torch.float64
L2_BYTES = 126 << 20  # blocks that fit here need not be streamed from memory each step


def _case(name, task, op, dims, n_v, M, n_t, sigma, precision, n_vh=0, periodic=True, potential="uniform",
          probe="gaussian", damping="none", B=1, degree=8.0):
    d0, d1, d2 = dims
    c = dict(task=task, op=op, d0=d0, d1=d1, d2=d2, n_v=n_v, n_vh=n_vh, M=M, n_t=n_t, sigma=sigma,
             precision=precision, periodic=periodic, potential=potential, probe=probe, damping=damping, B=B,
             degree=degree)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest DOS call: a 32 x 32 Dirichlet Laplacian with a potential, float64
        # throughout; launches and latencies count, not bandwidth.
        _case("dirichlet_32_fp64", "dos", "stencil", (32, 32, 1), 40, 200, 101, 0.05, "fp64", periodic=False),
        # The benchmark workload: 2D Anderson model, 200 probes, degree 1000, 400 sweep
        # points, mixed precision, both estimates.
        _case("anderson_256_mixed", "dos", "stencil", (256, 256, 1), 200, 1000, 400, 0.02, "mixed",
              probe="rademacher"),
        # Its float64-accurate form: the moments themselves (which a program keeps to
        # evaluate other points later) and the KPM line.
        _case("anderson_256_fp64_tc", "moments", "stencil", (256, 256, 1), 200, 1000, 400, 0.02, "fp64_tc",
              probe="rademacher"),
        # 3D, the widest block the tensor cores take, split into low-rank and hybrid
        # probes (the robust form of the estimate): moments and 400 pencils.
        _case("lognormal_64_hybrid", "dos", "stencil", (64, 64, 64), 128, 300, 400, 0.3, "mixed", n_vh=128,
              potential="lognormal"),
        # The classic KPM line on a large ragged 3D grid: few probes, damped series.
        _case("kpm_127_mixed", "kpm", "stencil", (127, 131, 125), 17, 300, 1000, 0.1, "mixed", potential="normal",
              damping="jackson", periodic=False),
        # One sparse graph operator (CSR) of odd size at float64 accuracy: its moments.
        _case("graph_30011_fp64_tc", "moments", "graph", (30011, 1, 1), 120, 200, 200, 0.05, "fp64_tc", n_vh=40),
        # Many small graphs in one plan: about 1000 normalised Laplacians of 100 to 900
        # nodes.  Each has fewer rows than a Gram slab of any size the plan's tuner
        # tries, so what it picks by timing does not change a bit of the results.
        _case("graphs_1100_mixed", "batch", "graph", (100, 900, 1), 32, 100, 16, 0.1, "mixed", B=1100),
        # Fitting a potential: forward and backward of a KPM loss on 10^6 grid points.
        _case("gradient_100_mixed", "gradient", "stencil", (100, 100, 100), 128, 200, 400, 0.2, "mixed",
              potential="normal"),
        # A few sweep points with explicitly formed filtered blocks, float64.
        _case("explicit_128_fp64", "explicit", "stencil", (128, 128, 1), 100, 400, 16, 0.05, "fp64",
              probe="rademacher"),
        # Tr log(A + I) on a plan that holds its moments: 512 grid points, hybrid pencils.
        _case("trace_log_20_fp64", "trace", "stencil", (21, 20, 19), 96, 728, 512, 0.121, "fp64", n_vh=64,
              potential="lognormal"),
        # The Gram pair of two float64 blocks of a caller's own recurrence.
        _case("gram_pair_200", "gram", "block", (65536, 1, 1), 200, 0, 0, 0.0, "fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    task = rng.choice(["dos", "dos", "dos", "kpm", "moments", "moments", "trace", "gradient", "explicit", "batch",
                       "gram"])
    even = lambda lo, hi: 2 * _log(rng, lo // 2, hi // 2)  # noqa: E731
    periodic = rng.random() < 0.6
    if task in ("dos", "kpm", "moments"):
        three = rng.random() < 0.5
        if three:
            d0, d1, d2 = (_log(rng, 8, 64) for _ in range(3))
        else:
            d0, d1, d2 = _log(rng, 24, 256), _log(rng, 24, 256), 1
        precision = {"dos": rng.choice(["mixed", "mixed", "fp64"]), "kpm": rng.choice(["mixed", "fp64_tc"]),
                     "moments": rng.choice(["mixed", "fp64_tc", "fp64_tc"])}[task]
        n_v = _log(rng, 16, 200)
        n_vh = _log(rng, 8, 56) if rng.random() < 0.4 or precision == "fp64" else 0
        M = even(60, 400)
        if precision == "fp64":  # float64 throughout: the small problems
            d0, d1, d2, n_v = max(8, d0 // 2), max(8, d1 // 2), max(1, d2 // 2), min(n_v, 100)
        op = "graph" if task == "moments" and rng.random() < 0.4 else "stencil"
        if op == "graph":
            d0, d1, d2 = _log(rng, 2000, 60000), 1, 1
        return _case("", task, op, (d0, d1, d2), n_v, M, _log(rng, 16, 400), round(rng.uniform(0.05, 0.4), 3),
                     precision, n_vh=n_vh, periodic=periodic, probe=rng.choice(["gaussian", "rademacher"]),
                     potential=rng.choice(["uniform", "lognormal", "normal"]),
                     damping=rng.choice(["none", "none", "jackson"]))
    if task == "trace":  # the Gaussian spans a few points of the grid, the degree resolves it
        n_t = 32 * _log(rng, 4, 16)
        return _case("", task, "stencil", (_log(rng, 12, 24), _log(rng, 12, 24), _log(rng, 12, 24)),
                     _log(rng, 16, 100), 2 * int(0.71 * n_t), n_t, round(62.0 / n_t, 3), "fp64",
                     n_vh=_log(rng, 16, 64), periodic=periodic, potential="lognormal")
    if task == "gradient":
        return _case("", task, "stencil", (_log(rng, 12, 90), _log(rng, 12, 90), _log(rng, 12, 90)),
                     _log(rng, 8, 128), even(40, 200), _log(rng, 50, 400), round(rng.uniform(0.1, 0.4), 3), "mixed",
                     potential="normal", periodic=periodic)
    if task == "explicit":
        return _case("", task, "stencil", (_log(rng, 24, 128), _log(rng, 24, 128), 1), _log(rng, 16, 100),
                     even(60, 400), _log(rng, 4, 16), round(rng.uniform(0.05, 0.2), 3), "fp64", periodic=periodic,
                     probe="rademacher")
    if task == "batch":
        hi = _log(rng, 300, 900)
        return _case("", task, "graph", (max(50, hi // 8), hi, 1), _log(rng, 8, 32), even(40, 100), _log(rng, 8, 16),
                     round(rng.uniform(0.08, 0.2), 3), "mixed", B=rng.randint(1050, 1200))
    return _case("", "gram", "block", (_log(rng, 1000, 80000), 1, 1), _log(rng, 16, 256), 0, 0, 0.0, "fp64")


# ---------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _block(n, cols, kind, g):
    if kind == "rademacher":
        return torch.randint(0, 2, (n, cols), generator=g, device="cuda").to(F64).mul_(2.0).sub_(1.0)
    return torch.randn((n, cols), generator=g, device="cuda", dtype=F64)


def _diag(c, n, g):
    """Diagonal of -Laplacian + potential (3D, 2D Dirichlet) or of the Anderson model."""
    if c["d2"] == 1 and c["periodic"]:
        return torch.rand(n, generator=g, device="cuda", dtype=F64) * 4.0 - 2.0
    base = 4.0 if c["d2"] == 1 else 6.0
    if c["potential"] == "lognormal":
        return base + torch.exp(0.5 * torch.randn(n, generator=g, device="cuda", dtype=F64))
    if c["potential"] == "normal":
        return base + 0.3 * torch.randn(n, generator=g, device="cuda", dtype=F64)
    return base + torch.rand(n, generator=g, device="cuda", dtype=F64) * 2.0 - 1.0


def _graphs(sizes, degree, g):
    """Normalised Laplacians I - D^-1/2 W D^-1/2 of weighted random graphs, as one CSR
    (row pointer, columns, values) with graph b's rows after those of b - 1."""
    n = torch.as_tensor(sizes, device="cuda", dtype=torch.int64)
    off = torch.cumsum(n, 0) - n
    N = int(n.sum())
    m = (n.to(F64) * (degree / 2)).to(torch.int64)
    which = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), m)
    u = torch.rand((2, which.numel()), generator=g, device="cuda", dtype=F64)
    i, j = ((u[k] * n[which]).to(torch.int64) + off[which] for k in (0, 1))
    keep = i != j
    key = torch.unique(torch.minimum(i, j)[keep] * N + torch.maximum(i, j)[keep])
    i, j = key // N, key % N
    w = torch.rand(i.numel(), generator=g, device="cuda", dtype=F64) + 0.5
    # (summed on the host, in one order: the GPU's scatter adds in any)
    ends, twice = torch.cat([i, j]).cpu().numpy(), torch.cat([w, w]).cpu().numpy()
    deg = torch.from_numpy(np.bincount(ends, weights=twice, minlength=N)).cuda()
    dinv = torch.where(deg > 0, deg.clamp_min(1e-300).rsqrt(), torch.zeros_like(deg))
    v = -w * dinv[i] * dinv[j]
    r = torch.arange(N, device="cuda")
    rows, cols = torch.cat([i, j, r]), torch.cat([j, i, r])
    vals = torch.cat([v, v, (deg > 0).to(F64)])
    order = torch.argsort(rows * N + cols)
    ptr = torch.zeros(N + 1, device="cuda", dtype=torch.int64)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=N), 0)
    return ptr, cols[order], vals[order]


def _sizes(c, seed):
    return np.random.default_rng(seed).integers(c["d0"], c["d1"] + 1, size=c["B"]).tolist()


def _inputs(c, seed):
    """The arrays of a case: operator, probe block, target."""
    g = _gen(seed)
    x = {}
    n_tot = c["n_v"] + c["n_vh"]
    if c["op"] == "block":
        x["A"], x["B"] = _block(c["d0"], n_tot, "gaussian", g), _block(c["d0"], n_tot, "gaussian", g)
        return x
    if c["op"] == "graph":
        x["sizes"] = _sizes(c, seed) if c["task"] == "batch" else [c["d0"]]
        x["csr"] = _graphs(x["sizes"], c["degree"], g)
        n = sum(x["sizes"])
    else:
        n = c["d0"] * c["d1"] * c["d2"]
        x["diag"] = _diag(c, n, g)
    x["W"] = _block(n, n_tot, c["probe"], g)
    if c["task"] == "gradient":
        x["target"] = torch.rand(c["n_t"], generator=g, device="cuda", dtype=F64) * 0.05
    return x


GRAPH_LO, GRAPH_HI = -2e-3, 2.002  # [0, 2], padded: the spectrum of a normalised Laplacian


def _offdiag(c):
    return (-1.0, -1.0, -1.0 if c["d2"] > 1 else 0.0)


def _log1(x):
    return math.log(1.0 + x) if x > -0.999 else math.log(1e-3)


def prepare(case, seed):
    c = case
    x = _inputs(c, seed)
    if c["task"] == "gram":
        return dict(c=c, **x)
    kw = dict(n_v=c["n_v"], n_vh=c["n_vh"], degree=c["M"], precision=c["precision"], damping=c["damping"])
    if c["task"] == "batch":
        ptr, col, val = (t.cpu().numpy() for t in x["csr"])
        mats, r0 = [], 0
        for n in x["sizes"]:
            a, b = int(ptr[r0]), int(ptr[r0 + n])
            mats.append(wl.CSR(n, ptr[r0 : r0 + n + 1] - a, (col[a:b] - r0).astype(np.int32), val[a:b]))
            r0 += n
        plan = S.ssm_plan_create_batched(mats, lo=GRAPH_LO, hi=GRAPH_HI, **kw)
    elif c["op"] == "graph":
        ptr, col, val = x["csr"]
        plan = S.ssm_plan_create(csr=wl.CSR(c["d0"], ptr, col.to(torch.int32), val), lo=GRAPH_LO, hi=GRAPH_HI, **kw)
    else:
        per = (c["periodic"], c["periodic"], c["periodic"] and c["d2"] > 1)
        st = wl.Stencil((c["d0"], c["d1"], c["d2"]), per, x["diag"], _offdiag(c))
        plan = S.ssm_plan_create(stencil=st, options=2 if c["task"] == "gradient" else 0, **kw)
    s = dict(c=c, plan=plan, W=x["W"])
    if c["op"] == "graph":
        t = torch.linspace(0.0, 2.0, c["n_t"], device="cuda", dtype=F64)
        s["t"] = t.repeat(c["B"]) if c["task"] == "batch" else t
    else:
        info = S.ssm_plan_info(plan)
        t = np.linspace(info["lo"], info["hi"], c["n_t"] + (2 if c["task"] == "explicit" else 0))
        s["t"] = torch.from_numpy(t[1:-1].copy() if c["task"] == "explicit" else t).cuda()
    if c["task"] == "gradient":
        s["diag"], s["target"] = x["diag"].requires_grad_(True), x["target"]
    if c["task"] == "trace":  # the moments are there from the DOS that the program made first
        S.ssm_moments(plan, s["W"])
    return s


def run(state):
    s, c = state, state["c"]
    task = c["task"]
    if task == "gram":
        aa, ab = S.ssm_gram_pair(s["A"], s["B"])
        return {"aa": aa, "ab": ab}
    plan, t, sigma = s["plan"], s["t"], c["sigma"]
    if task in ("dos", "batch"):
        S.ssm_moments(plan, s["W"])
        ss, kpm, rank = S.ssm_dos(plan, t, sigma)
        return {"ss": ss, "kpm": kpm, "rank": rank}
    if task == "kpm":
        S.ssm_moments(plan, s["W"])
        return {"kpm": S.ssm_dos(plan, t, sigma, want_ss=False, want_rank=False)[1]}
    if task == "moments":
        X = S.ssm_moments(plan, s["W"], return_moments=True)
        return {"X": X, "kpm": S.ssm_dos(plan, t, sigma, want_ss=False, want_rank=False)[1]}
    if task == "trace":
        tr_ss, tr_kpm = S.ssm_trace_f(plan, _log1, c["n_t"], sigma)
        return {"ss": tr_ss, "kpm": tr_kpm}
    if task == "gradient":
        s["diag"].grad = None
        kpm = S.KPMDensity.apply(s["diag"], plan, s["W"], t, sigma)
        torch.sum((kpm - s["target"]) ** 2).backward()
        return {"kpm": kpm.detach(), "grad": s["diag"].grad}
    ss, rank = S.ssm_dos_explicit(plan, s["W"], t, sigma)
    return {"ss": ss, "rank": rank}


# ---------------------------------------------------------------- work


def _rows_nnz(c):
    if c["op"] == "graph":
        n = c["B"] * (c["d0"] + c["d1"]) // 2 if c["task"] == "batch" else c["d0"]
        return n, int(n * (c["degree"] + 1))
    n = c["d0"] * c["d1"] * c["d2"]
    return n, n * (7 if c["d2"] > 1 else 5)


def work(case):
    c = case
    n_tot, n_v, M, n_t = c["n_v"] + c["n_vh"], c["n_v"], c["M"], c["n_t"]
    tri = n_tot * (n_tot + 1) / 2
    if c["task"] == "gram":
        return {"bytes": 8.0 * (2 * c["d0"] * n_tot + 2 * n_tot * n_tot), "flops": 2.0 * c["d0"] * (tri + n_tot**2)}
    n, nnz = _rows_nnz(c)
    e = 4 if c["precision"] == "mixed" else 8
    blk = n * n_tot
    if c["task"] == "trace":
        steps = 0
    else:
        steps = M if c["task"] == "explicit" else M // 2
    ins = 8.0 * blk + (12.0 * nnz if c["op"] == "graph" else 8.0 * n)
    streamed = 3.0 * blk * e * steps if 3 * blk * e > L2_BYTES else 0.0
    flops = 2.0 * nnz * n_tot * steps
    points = n_t * c["B"]
    pencil = points * (2.0 * (M / 2) * tri + 2.0 * M * n_v * (n_v + 1) / 2 + 5.0 / 3 * n_v**3 + 2.0 * n_v**2 * c["n_vh"])
    if c["task"] == "explicit":
        flops += 2.0 * n * n_v * n_t * (M + 1) + n_t * 2.0 * n * 1.5 * n_v**2 + n_t * 5.0 / 3 * n_v**3
        return {"bytes": ins + streamed + 16.0 * n_t, "flops": flops}
    if c["task"] == "trace":
        return {"bytes": 8.0 * (M + 1) * tri + 8.0, "flops": pencil}
    flops += 2.0 * n * (tri + n_tot**2) * steps  # the two Gram products of a step
    out = 16.0 * points
    if c["task"] in ("dos", "batch"):
        flops += pencil
    if c["task"] == "moments":
        out += 8.0 * (M + 1) * n_tot**2
    if c["task"] == "gradient":
        flops += (2.0 * nnz * 2 + 8.0 * n) * n_tot * steps
        streamed += 6.0 * blk * e * steps
        out += 8.0 * n
    return {"bytes": ins + streamed + out, "flops": flops}


# ---------------------------------------------------------------- the same in float64 torch


def _apply_stencil(c, diag, dims=None):
    d = (c["d0"], c["d1"], c["d2"])
    off = _offdiag(c)
    per = c["periodic"]

    def apply(v):
        u = v.reshape(*d, -1)
        y = diag.reshape(*d, 1) * u
        for ax in range(3):
            if d[ax] == 1 or off[ax] == 0.0:
                continue
            for sh in (1, -1):
                r = torch.roll(u, sh, ax)
                if not per:
                    r.select(ax, 0 if sh == 1 else -1).zero_()
                y += off[ax] * r
        return y.reshape(v.shape)

    return apply


def _operator(c, x):
    """A as a function, its interval (a, b) and its spectral bounds."""
    if c["op"] == "graph":
        ptr, col, val = x["csr"]
        n = ptr.numel() - 1
        A = torch.sparse_csr_tensor(ptr, col, val, size=(n, n))
        return (lambda v: A @ v), GRAPH_LO, GRAPH_HI, GRAPH_LO, GRAPH_HI
    diag = x["diag"].detach()
    n = diag.numel()
    radius = -_apply_stencil(c, torch.zeros(n, device="cuda", dtype=F64))(torch.ones(n, 1, device="cuda", dtype=F64))
    lo, hi = float((diag - radius[:, 0]).min()), float((diag + radius[:, 0]).max())
    w = hi - lo
    return _apply_stencil(c, diag), lo - 1e-3 * w, hi + 1e-3 * w, lo, hi


def _chebyshev(apply, W, M, a, b):
    """T_l(A~) W for l = 0 .. M, by the three-term loop."""
    s, m = 2.0 / (b - a), 0.5 * (a + b)
    old, now = None, W
    yield 0, now
    for l in range(1, M + 1):
        new = (apply(now) - m * now) * s
        if old is not None:
            new = 2.0 * new - old
        old, now = now, new
        yield l, now


def _mu(t, M, n_theta, sigma, N, a, b):
    theta = np.arange(2 * n_theta) * math.pi / n_theta
    z = 0.5 * (a + b) + 0.5 * (b - a) * np.cos(theta)
    gau = np.exp(-((t[:, None] - z[None]) ** 2) / (2 * sigma**2)) / (N * math.sqrt(2 * math.pi * sigma**2))
    mu = np.fft.fft(gau, axis=1)[:, : M + 1].real / (2 * n_theta)
    mu[:, 1:] *= 2
    return mu


def _jackson(L):
    k, q = np.arange(L), math.pi / (L + 1)
    return ((L - k + 1) * np.cos(q * k) + np.sin(q * k) / math.tan(q)) / (L + 1)


def _tables(c, t, N, a, b):
    """mu to degree M, mu to degree M/2 and the square of its series, per point."""
    M = c["M"]
    half, full = _mu(t, M // 2, 2 * M, c["sigma"], N, a, b), _mu(t, M, 2 * M, c["sigma"], N, a, b)
    if c["damping"] == "jackson":
        half, full = half * _jackson(M // 2 + 1), full * _jackson(M + 1)
    theta = np.arange(4 * M) * math.pi / (2 * M)
    q = (half @ np.cos(np.outer(np.arange(M // 2 + 1), theta))) ** 2
    nu = np.fft.fft(q, axis=1)[:, : M + 1].real / (4 * M)
    nu[:, 1:] *= 2
    return full, half, nu


def _eigh(K):
    if K.shape[-1] <= 32:
        return torch.linalg.eigh(K)
    s, U = torch.linalg.eigh(K.cpu())
    return s.to(K.device), U.to(K.device)


def _pencils(KW, KZ, KC, trKH, gmax, floor, n_vh):
    """Per point: eigenvalues of the pencil (KZ, KW) restricted to what the truncation
    keeps, those in the range of the Gaussian summed, and the hybrid correction."""
    s, U = _eigh(0.5 * (KW + KW.mT))
    top = s[:, -1:]
    keep = (s >= torch.maximum(1e-7 * top, floor[:, None])) & (top > 0)
    # a dropped direction is given the weight zero: its eigenvalue is then exactly zero
    isq = torch.where(keep, s.clamp_min(1e-300).rsqrt(), torch.zeros_like(s))
    P = U * isq[:, None, :]
    xi, V = _eigh(P.mT @ KZ @ P + torch.diag_embed(torch.where(keep, 0.0, -10.0 * gmax)))
    sel = (xi >= -1e-6 * gmax) & (xi <= (1 + 1e-6) * gmax)
    phi = torch.where(sel, xi, torch.zeros_like(xi)).sum(1)
    if n_vh:
        C = P @ V * sel[:, None, :].to(F64)
        phi = phi + (trKH - ((KC @ C) ** 2).sum((1, 2))) / n_vh
    return phi


def _dos(c, X, t, N, a, b):
    """Both estimates at the points t from the moments X."""
    n_v, n_vh, M, sigma = c["n_v"], c["n_vh"], c["M"], c["sigma"]
    full, half, nu = _tables(c, t, N, a, b)
    zeta = X.diagonal(dim1=1, dim2=2).sum(1) / X.shape[1]
    kpm = torch.from_numpy(full).cuda() @ zeta
    if c["task"] in ("kpm", "moments", "gradient", "batch"):
        return None, kpm
    gmax = 1.0 / (N * math.sqrt(2 * math.pi * sigma**2))
    eps = 2.0**-36 if c["precision"] == "mixed" else 2.0**-52
    floor = 8.0 * n_v * eps * float(X[0].diagonal()[:n_v].max()) * ((np.arange(M // 2 + 1) + 1) * np.abs(half)).sum(1)
    ss = []
    for p in range(0, len(t), 128):
        h, z = torch.from_numpy(half[p : p + 128]).cuda(), torch.from_numpy(nu[p : p + 128]).cuda()
        K = torch.tensordot(h, X[: M // 2 + 1], 1)
        KZ = torch.tensordot(z, X[:, :n_v, :n_v].contiguous(), 1)
        ss.append(_pencils(K[:, :n_v, :n_v], KZ, K[:, n_v:, :n_v], K[:, n_v:, n_v:].diagonal(dim1=1, dim2=2).sum(1),
                           gmax, torch.from_numpy(floor[p : p + 128]).cuda(), n_vh))
    return torch.cat(ss), kpm


def _moments(c, x, apply, a, b):
    W = x["W"]
    X = torch.empty(c["M"] + 1, W.shape[1], W.shape[1], device="cuda", dtype=F64)
    for l, V in _chebyshev(apply, W, c["M"], a, b):
        X[l] = W.T @ V
    return 0.5 * (X + X.mT)


def _exact_trace(c, x):
    apply, a, b, lo, hi = _operator(c, x)
    n, sg, edge, st = c["n_t"], c["sigma"], 0.93, 0.016
    N = x["W"].shape[0]
    X = _moments(c, x, apply, a, b)
    mid, hw = 0.5 * (lo + hi), 0.5 * (hi - lo) / edge
    tt = -1.0 + 2.0 * np.arange(n) / n
    z, dx = mid + hw * tt, 2.0 * hw / n
    erf = lambda v: torch.erf(torch.from_numpy(v)).numpy()  # noqa: E731
    win = 0.5 * (erf((1 + edge - 2 * tt) / st) - erf((-1 - edge - 2 * tt) / st))
    end = 0.5 * (_log1(mid - hw) + _log1(mid + hw))
    h = np.array([_log1(v) for v in z]) * win + end * (1 - win)
    off = dx * (((np.arange(n) + n // 2) % n) - n // 2)
    ker = sum(np.exp(-((off + m * n * dx) ** 2) / (2 * sg**2)) for m in range(-3, 4)) / math.sqrt(2 * math.pi * sg**2)
    kh = dx * np.fft.fft(ker)
    keep = np.abs(kh) >= 1e-14 * np.abs(kh).max()
    ft = np.fft.ifft(np.where(keep, np.fft.fft(h) / np.where(keep, kh, 1.0), 0.0)).real
    w = torch.from_numpy(N * dx * ft).cuda()
    ss, kpm = _dos(c, X, z, N, a, b)
    return {"ss": float(w @ ss), "kpm": float(w @ kpm)}


def _exact_gradient(c, x):
    """The gradient by the Chebyshev identity dT_l = sum_j (2 - [j = 0]) U_{l-1-j} dA~ T_j."""
    apply, a, b, lo, hi = _operator(c, x)
    W, M = x["W"], c["M"]
    N, n_tot = W.shape
    t = np.linspace(lo, hi, c["n_t"])
    mu = torch.from_numpy(_mu(t, M, 2 * M, c["sigma"], N, a, b)).cuda()
    zeta = torch.empty(M + 1, device="cuda", dtype=F64)
    prev = None
    for l, V in _chebyshev(apply, W, M, a, b):
        zeta[l] = (W * V).sum() / n_tot
        if l == M - 1:
            prev = V
    kpm = mu @ zeta
    g = (2.0 * (kpm - x["target"])) @ mu / n_tot
    s, m = 2.0 / (b - a), 0.5 * (a + b)
    At = lambda v: (apply(v) - m * v) * s  # noqa: E731
    # B_j = sum_{l > j} g_l U_{l-1-j} W and T_j W, both from j = M - 1 down
    now, old = float(g[M]) * W, torch.zeros_like(W)
    T, Tup = prev, V
    grad = torch.zeros(N, device="cuda", dtype=F64)
    for j in range(M - 1, -1, -1):
        grad += (2.0 if j else 1.0) * (T * now).sum(1)
        if j:
            now, old = float(g[j]) * W + 2.0 * At(now) - old, now
            T, Tup = (2.0 * At(T) - Tup if j > 1 else W), T
    return {"kpm": kpm, "grad": grad * s}


def _exact_explicit(c, x):
    apply, a, b, lo, hi = _operator(c, x)
    W, M, n_v = x["W"], c["M"], c["n_v"]
    N = W.shape[0]
    t = np.linspace(lo, hi, c["n_t"] + 2)[1:-1]
    mu = _mu(t, M, 2 * M, c["sigma"], N, a, b)
    Z = torch.zeros(c["n_t"], N, n_v, device="cuda", dtype=F64)
    for l, V in _chebyshev(apply, W, M, a, b):
        for i in range(c["n_t"]):
            Z[i].add_(V, alpha=float(mu[i, l]))
    x0 = float((W * W).sum(0).max())
    floor = 8.0 * n_v * 2.0**-52 * x0 * ((np.arange(M + 1) + 1) * np.abs(mu)).sum(1)
    KW, KZ = W.T @ Z, Z.mT @ Z
    gmax = 1.0 / (N * math.sqrt(2 * math.pi * c["sigma"] ** 2))
    return {"ss": _pencils(KW, KZ, None, None, gmax, torch.from_numpy(floor).cuda(), 0), "rank": None}


def _exact_batch(c, x):
    sizes, M, n_v = x["sizes"], c["M"], c["n_v"]
    B, top = len(sizes), max(sizes)
    apply = _operator(c, x)[0]
    where = torch.cat([torch.arange(n, device="cuda") + b * top for b, n in enumerate(sizes)])
    pad = lambda v: torch.zeros(B * top, n_v, device="cuda", dtype=F64).index_copy_(0, where, v).view(B, top, n_v)  # noqa: E731
    Wp = pad(x["W"])
    X = torch.empty(B, M + 1, n_v, n_v, device="cuda", dtype=F64)
    for l, V in _chebyshev(apply, x["W"], M, GRAPH_LO, GRAPH_HI):
        X[:, l] = Wp.mT @ pad(V)
    X = 0.5 * (X + X.mT)
    t = np.linspace(0.0, 2.0, c["n_t"])
    got = [_dos(c, X[b], t, n, GRAPH_LO, GRAPH_HI) for b, n in enumerate(sizes)]
    return {"ss": None, "kpm": torch.cat([g[1] for g in got]), "rank": None}  # ss: as in exact(), small operators


def exact(case, seed):
    c = case
    x = _inputs(c, seed)
    if c["task"] == "gram":
        return {"aa": x["A"].T @ x["A"], "ab": x["A"].T @ x["B"]}
    if c["task"] == "gradient":
        return _exact_gradient(c, x)
    if c["task"] == "explicit":
        return _exact_explicit(c, x)
    if c["task"] == "batch":
        return _exact_batch(c, x)
    if c["task"] == "trace":
        return _exact_trace(c, x)
    apply, a, b, lo, hi = _operator(c, x)
    t = np.linspace(0.0, 2.0, c["n_t"]) if c["op"] == "graph" else np.linspace(lo, hi, c["n_t"])
    X = _moments(c, x, apply, a, b)
    ss, kpm = _dos(c, X, t, x["W"].shape[0], a, b)
    if c["precision"] == "mixed" and x["W"].shape[0] < 20000:
        ss = None  # float32 moments leave the low-rank estimate of a small operator few digits
    return {"dos": {"ss": ss, "kpm": kpm, "rank": None}, "kpm": {"kpm": kpm}, "moments": {"X": X, "kpm": kpm}}[c["task"]]
