"""The work that performance is measured on: what a user of the sampler has it do.

Every case is a dict of plain sizes and options.  prepare() makes what a program
holds before the call (the body, the sampler, buffers for the samples), run() makes
one call through the public binding, exact() is the same walk in plain FP64 torch.

Three kinds of work:
  sampler  Sampler(...).run(iters, thin): the walk itself, in each arithmetic mode,
           with equalities, a learned preconditioner, thinned traces, FP64 audits;
  batch    Batch(...).run(iters): many uneven polytopes advanced together;
  fit      fit_from_moments(...): the preconditioner learned from pooled moments.
"""
import math

import numpy as np
import torch

from paper_2104_07097_gb300 import mhar, workloads

_BASE = dict(kind="sampler", body="rand", precision="mixed_rs", n=0, m=0, z=0, iters=0,
             thin=0, emit=0, device_out=True, pc_rank=-1, audit_every=0, audit_walkers=0,
             check=False)


def _sampler(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # The smallest call: the 10-dimensional cube in the default precision, 100
        # walkers.  Kernel latency and launches are all of its time.
        _sampler("cube10_fp64", body="cube", precision="fp64", n=10, m=20, z=100, iters=40,
                 thin=40, device_out=False),
        # An ordinary call with every default: FP64, max(m, n) + 1 walkers, thinned
        # samples returned in host memory.  Nothing is a multiple of a tile.
        _sampler("rand37x300_fp64", precision="fp64", n=37, m=300, z=301, iters=24, thin=6,
                 device_out=False),
        # FP64 at the size of the throughput benchmark: a user who wants the default
        # precision on a large ensemble.
        _sampler("rand100x2000_fp64", precision="fp64", n=100, m=2000, z=4096, iters=4, thin=4),
        # The same body in plain FP32, the mode the tensor-core modes are judged against.
        _sampler("rand100x2000_fp32", precision="fp32", n=100, m=2000, z=4096, iters=16, thin=16),
        # The stored-slack tensor-core mode, long enough for one periodic refresh.
        _sampler("rand100x2000_stored", precision="mixed", n=100, m=2000, z=4096, iters=64,
                 thin=64),
        # The headline: the recompute tensor-core mode on that body.
        _sampler("rand100x2000_rs", n=100, m=2000, z=4096, iters=96, thin=96),
        # A checked production run: FP64 audits of a part of the ensemble on the way and
        # the feasibility check of all walkers at the end.
        _sampler("rand100x2000_rs_checked", n=100, m=2000, z=4096, iters=64, thin=64,
                 audit_every=16, audit_walkers=1024, check=True),
        # A body inside an affine subspace: the simplex with 4000 cuts, one equality.
        _sampler("simplex1000+4000_rs", body="simplex", n=1000, m=5000, z=8192, iters=16,
                 thin=16),
        # The largest: an ill-conditioned body with a frozen rank-32 + diagonal
        # preconditioner.
        _sampler("illcond500x10000_rs_pc", body="illcond", n=500, m=10000, z=16384, iters=8,
                 thin=8, pc_rank=32),
        # A long preconditioned chain on a moderate body, a trace of 64 walkers kept
        # every fifth iteration for effective-sample-size estimates.
        _sampler("illcond40x400_rs_trace", body="illcond", n=40, m=400, z=4096, iters=100,
                 thin=5, emit=64, pc_rank=32),
        # Many uneven polytopes advanced together, 512 walkers each.
        dict(kind="batch", name="batch48", count=48, nmin=20, nmax=400, z=512, iters=16),
        # Learning a preconditioner from the pooled warm-up moments of several shards.
        dict(kind="fit", name="fit500", n=500, samples=81920, rank=32, power_iters=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges; no dearer than the largest listed one."""
    u = rng.random()
    if u < 0.1:
        return dict(kind="batch", count=rng.randint(3, 48), nmin=20, nmax=rng.randint(60, 400),
                    z=_log_int(rng, 33, 512), iters=rng.randint(4, 16))
    if u < 0.2:
        n = _log_int(rng, 20, 500)
        return dict(kind="fit", n=n, samples=_log_int(rng, 40 * n, 81920),
                    rank=rng.randint(1, min(32, n)), power_iters=rng.randint(0, 6))
    precision = rng.choice(["fp64", "fp64", "fp32", "mixed", "mixed_rs", "mixed_rs"])
    c = dict(_BASE, precision=precision)
    c["body"] = rng.choice(["rand", "rand", "illcond", "simplex", "cube"])
    c["n"] = n = _log_int(rng, 5, 100 if precision in ("fp64", "fp32") else 700)
    if c["body"] == "cube":
        c["m"] = 2 * n
    elif c["body"] == "simplex":
        c["m"] = n + rng.randint(1, 4 * n)
    else:
        c["m"] = rng.randint(8 * n, 20 * n)
    c["z"] = _log_int(rng, 50, 4096 if precision in ("fp64", "fp32") else 8192)
    # As many iterations as a fixed amount of work holds: a short FP64 chain, up to 96
    # in fewer bits.
    most = {"fp64": 3e9, "fp32": 2e10, "mixed": 2e11, "mixed_rs": 3e11}[precision]
    c["iters"] = max(2, min(rng.randint(4, 12) if precision == "fp64" else rng.randint(32, 96),
                           int(most / (4.0 * c["m"] * n * c["z"]))))
    c["thin"] = rng.choice([c["iters"], c["iters"], max(1, c["iters"] // 4)])
    c["device_out"] = rng.random() < 0.5
    c["emit"] = rng.choice([0, 0, min(c["z"], 33)])
    if c["body"] == "illcond":
        c["pc_rank"] = rng.randint(0, min(32, n))
    if precision != "fp64" and rng.random() < 0.3:   # a walk in fewer bits, checked in FP64
        c["audit_every"], c["audit_walkers"] = 8, min(c["z"], 512)
        c["check"] = True
    return c


# ---- inputs ------------------------------------------------------------------

def _body(case, seed):
    n, m = case["n"], case["m"]
    if case["body"] == "cube":
        return workloads.cube(n)
    if case["body"] == "simplex":
        return workloads.simplex_cuts(n, m - n, seed)
    if case["body"] == "illcond":
        return workloads.ill_conditioned(n, m, seed, smin=1e-3 if n > 100 else 1e-2)
    return workloads.random_polytope(n, m, seed, check_bounded="auto")


def _preconditioner(case, p, seed):
    """A frozen factor such as a fit leaves: the axis extents read off the
    constraints on the diagonal, a small low-rank part in the same units."""
    extent = 1.0 / np.abs(p.A).max(axis=0)
    delta = extent / extent.max()
    r = case["pc_rank"]
    rng = np.random.default_rng([seed, 7])
    U = 0.3 * delta[:, None] * rng.standard_normal((case["n"], r)) / math.sqrt(max(r, 1))
    return delta, U


def _problems(case, seed):
    return [workloads.random_polytope(n, m, seed * 100_003 + q, check_bounded="auto")
            for q, (m, n, _, _) in enumerate(_sizes(case))]


def _moments(case, seed):
    """Sums over the warm-up points of a chain on a body with axes from 1e-3 to 1."""
    n, N = case["n"], case["samples"]
    rng = np.random.default_rng([seed, 3])
    s = np.exp(rng.uniform(math.log(1e-3), 0.0, size=n))
    mix = rng.standard_normal((n, min(n, 8))) / math.sqrt(n)
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(N, n, generator=g, device="cuda", dtype=torch.float64)
    X += (X @ torch.from_numpy(mix).cuda()) @ torch.from_numpy(mix.T.copy()).cuda()
    X = X * torch.from_numpy(s).cuda() * 0.3
    return X.sum(0).cpu().numpy(), (X.T @ X).cpu().numpy()


def prepare(case, seed):
    if case["kind"] == "batch":
        probs = [(p.A, p.b, p.x0) for p in _problems(case, seed)]
        b = mhar.Batch(probs, case["z"], seed=seed, out_on_device=True)
        outs = [torch.empty(1, case["z"], p[0].shape[1], dtype=torch.float64, device="cuda")
                for p in probs]
        return dict(case=case, batch=b, outs=outs)
    if case["kind"] == "fit":
        p = workloads.ill_conditioned(case["n"], 4 * case["n"], seed)
        s1, s2 = _moments(case, seed)
        s = mhar.Sampler(p.A, p.b, p.x0, 64, precision="mixed_rs", seed=seed)
        return dict(case=case, sampler=s, s1=s1, s2=s2)
    p = _body(case, seed)
    s = mhar.Sampler(p.A, p.b, p.x0, case["z"], AE=p.AE, bE=p.bE, precision=case["precision"],
                     seed=seed, out_on_device=case["device_out"], emit_walkers=case["emit"],
                     audit_every=case["audit_every"], audit_walkers=case["audit_walkers"])
    if case["pc_rank"] >= 0:
        delta, U = _preconditioner(case, p, seed)
        s.set_preconditioner(delta, U if case["pc_rank"] > 0 else None)
    out = None
    if case["device_out"]:
        out = torch.empty(case["iters"] // case["thin"], s.emit_walkers, p.n,
                          dtype=torch.float64, device="cuda")
    return dict(case=case, sampler=s, out=out)


def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        return state["batch"].run(c["iters"], thin=c["iters"], outs=state["outs"])
    s = state["sampler"]
    if c["kind"] == "fit":
        s.fit_from_moments(state["s1"], state["s2"], c["samples"], c["rank"], c["power_iters"])
        delta, U = s.preconditioner()
        return dict(delta=delta, U=U)
    got = dict(samples=s.run(c["iters"], thin=c["thin"], out=state["out"]))
    if c["check"]:
        st = s.check()
        got.update(max_violation=st.max_violation, run_max_violation=st.run_max_violation)
    return got


def _sizes(case):
    """(m, n, z, iterations) of every walk of a case."""
    if case["kind"] == "batch":
        rng = np.random.default_rng([case["count"], case["nmin"], case["nmax"]])
        ns = rng.integers(case["nmin"], case["nmax"] + 1, case["count"])
        return [(int(rng.integers(4 * n, 20 * n + 1)), int(n), case["z"], case["iters"])
                for n in ns]
    return [(case["m"], case["n"], case["z"], case["iters"])]


def work(case):
    if case["kind"] == "fit":
        n, r = case["n"], case["rank"]
        products = case["power_iters"] + 2
        return {"bytes": 8.0 * (n * n + n + n * (r + 1)),
                "flops": 2.0 * n * n * r * products + 6.0 * n * r * r * products}
    size = 8 if case.get("precision") == "fp64" else 4
    nbytes = flops = 0.0
    for m, n, z, iters in _sizes(case):
        # A and b read once, the points read and written once, the samples written;
        # A x and A d of every iteration (Lemma 4.2; A d alone with a stored slack).
        emitted = (case.get("emit") or z) * (iters // case.get("thin", iters))
        nbytes += size * (m * n + m) + 2.0 * size * z * n + 8.0 * emitted * n
        per = 2.0 if case.get("precision") == "mixed" else 4.0
        flops += per * m * n * z * iters
        if case.get("body") == "simplex":
            flops += 4.0 * n * z * iters              # d = h - Q^T Q h, one equality
        if case.get("pc_rank", -1) > 0:
            flops += 2.0 * n * case["pc_rank"] * z * iters
        if case.get("check"):
            audits = iters // case["audit_every"]
            flops += 2.0 * m * n * (z + audits * case["audit_walkers"])
    return {"bytes": nbytes, "flops": flops}


# ---- the same results in plain FP64 torch --------------------------------------

def _philox(ctr, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF
    c0, c1, c2, c3 = ctr
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        h0, l0 = (p0 >> 32) & mask, p0 & mask
        h1, l1 = (p1 >> 32) & mask, p1 & mask
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _words(seed, step, stream, walkers, quads, dev):
    w = torch.arange(walkers, dtype=torch.int64, device=dev)[:, None].expand(walkers, quads)
    q = torch.arange(quads, dtype=torch.int64, device=dev)[None, :].expand(walkers, quads)
    lo = torch.full_like(w, step & 0xFFFFFFFF)
    hi = torch.full_like(w, (((step >> 32) & 0xFFFFFF) << 8) | stream)
    return _philox((q, w, lo, hi), seed)


def _normals(seed, step, stream, walkers, count, dev):
    """walkers x count standard normals: Box-Muller on words (0, 1) and (2, 3)."""
    words = _words(seed, step, stream, walkers, (count + 3) // 4, dev)
    u = [(w.to(torch.float64) + 0.5) * 2.0 ** -32 for w in words]
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        out += [r * torch.cos(2.0 * math.pi * b), r * torch.sin(2.0 * math.pi * b)]
    return torch.stack(out, dim=2).reshape(walkers, -1)[:, :count]


def _walk(p, z, iters, thin, emit, seed, pre=None):
    """Algorithm 2 on {A x <= b, A_E x = b_E}: the samples after every `thin` iterations."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    def t(a):
        return torch.as_tensor(np.asarray(a, dtype=np.float64), device=dev)
    A, b = t(p.A), t(p.b)
    X = t(p.x0)[None, :].repeat(z, 1)
    Q = torch.linalg.qr(t(p.AE).T).Q if p.AE is not None else None
    inf = float("inf")
    out = []
    for s in range(iters):
        D = _normals(seed, s, 0, z, p.n, dev)
        if pre is not None:
            D = D * t(pre[0])
            if pre[1].shape[1] > 0:
                D = D + _normals(seed, s, 2, z, pre[1].shape[1], dev) @ t(pre[1]).T
        if Q is not None:
            D = D - (D @ Q) @ Q.T
        lo = torch.empty(z, dtype=torch.float64, device=dev)
        hi = torch.empty_like(lo)
        for k in range(0, z, 4096):
            G = D[k:k + 4096] @ A.T
            R = (b - X[k:k + 4096] @ A.T).clamp_(min=0.0) / G
            hi[k:k + 4096] = torch.where(G > 0, R, inf).amin(1)
            lo[k:k + 4096] = torch.where(G < 0, R, -inf).amax(1)
        u = (_words(seed, s, 1, z, 1, dev)[0][:, 0].to(torch.float64) + 0.5) * 2.0 ** -32
        X = X + (lo + u * (hi - lo))[:, None] * D
        if (s + 1) % thin == 0:
            out.append(X[:emit].clone())
    return torch.stack(out)


def _fit(case, seed):
    """delta of the rank-r + diagonal fit (U's columns have no sign of their own)."""
    n, r, N = case["n"], case["rank"], case["samples"]
    s1, s2 = _moments(case, seed)
    sigma = torch.from_numpy((s2 - np.outer(s1, s1) / N) / (N - 1.0))
    Y = sigma @ _normals(seed, 0, 3, r, n, "cpu").T
    for _ in range(case["power_iters"]):
        Y = sigma @ torch.linalg.qr(Y).Q
    Q = torch.linalg.qr(Y).Q
    T = Q.T @ sigma @ Q
    lam, V = torch.linalg.eigh(0.5 * (T + T.T))
    U = Q @ V * lam.clamp(min=0.0).sqrt()
    d = torch.diagonal(sigma)
    floor = torch.maximum(1e-2 * d, 1e-9 * d.sum() / n)
    return torch.maximum(d - (U * U).sum(1), floor).sqrt().numpy()


def exact(case, seed):
    if case["kind"] == "fit":
        return dict(delta=_fit(case, seed), U=None)
    if case["kind"] == "batch":
        z, it = case["z"], case["iters"]
        return [_walk(p, z, it, it, z, seed + q) for q, p in enumerate(_problems(case, seed))]
    p = _body(case, seed)
    pre = _preconditioner(case, p, seed) if case["pc_rank"] >= 0 else None
    got = dict(samples=_walk(p, case["z"], case["iters"], case["thin"],
                             case["emit"] or case["z"], seed, pre))
    if case["check"]:
        # How far a walk stays inside depends on that walk's own margins.
        got.update(max_violation=None, run_max_violation=None)
    return got
