"""Performance cases of the library: what a user's program has it do, through the public Python API.

Kinds of case:
  solve     one completion problem, already built (a Solver on the GPU): Algorithm 1 with the kick, up to k_max
            iterations, then what the caller takes away: the recovered values X on Omega (from the factors of X),
            the dual iterate Y and the singular values.  All values of an iterate on Omega are returned, never the
            singular vectors themselves, whose signs are arbitrary.  k_max bounds the solve: a few instances of
            every size need many times the usual 120 iterations, and their late iterates depend on the last bits.
  batch     several problems of a serving mix at once (batch_solve).
  products  the per-entry kernels on their own: Y V, Y^T U and the fused X-on-Omega + dual step, on device tensors.
  build     a new problem: Omega drawn on the device, then the context with its row- and column-major storage.

Output types: a float64 solve with lanczos_tol = 1e-9 returns float64.  With the default tolerances (1e-6 sigma_1 for
float64 values, 1e-4 for float32 and bfloat16) the iterates carry that tolerance's error, and the values are
returned in float32, as a program that stores predictions keeps them.

Problems are the planted ones of the paper's Sec. 5.2.1 (N(0,1) factors, |Omega| = ratio r (m + n - r) entries drawn
uniformly, tau = 5 sqrt(m n), delta = 1.2 m n / |Omega|), made on the GPU.
"""
from __future__ import annotations

import math

import torch

from paper_0810_3286_gb300 import Solver, batch_solve, sample_omega

MAX_RANK = 64


def listed():
    return [
        # the smallest calls: a problem of the size of the checkpoint test, where launches and latencies are all
        dict(name="solve_120x100_fp64_tight", kind="solve", m=120, n=100, r=3, ratio=5.5, precision="fp64", tol=1e-9,
             k_max=30),
        # the plain float64 workload (200 x 200, rank 5) at the tight tolerance the shrink test uses
        dict(name="solve_200_fp64_tight", kind="solve", m=200, n=200, r=5, ratio=6.0, precision="fp64", tol=1e-9,
             k_max=60),
        # Table 1's first row (1000 x 1000, rank 10) with the defaults, in both precisions: the ordinary solve
        dict(name="solve_1000_fp64", kind="solve", m=1000, n=1000, r=10, ratio=6.0, precision="fp64", tol=0.0,
             k_max=80),
        dict(name="solve_1000_fp32", kind="solve", m=1000, n=1000, r=10, ratio=6.0, precision="fp32", tol=0.0,
             k_max=80),
        # Table 1's 1000 x 1000 rank-50 row: blocks of 32, projected problems up to 128 x 128
        dict(name="solve_1000_r50_fp64", kind="solve", m=1000, n=1000, r=50, ratio=4.0, precision="fp64", tol=0.0,
             k_max=6),
        # a rectangular job of the serving distribution (m, n in [500, 8000], rank 5-20, ratio 4-6), odd sizes
        dict(name="solve_4219x2753_r13_fp32", kind="solve", m=4219, n=2753, r=13, ratio=5.2, precision="fp32", tol=0.0,
             k_max=60),
        # the "BF16 vs FP32" configuration, long enough to leave the bfloat16 phase
        dict(name="solve_10000_bf16", kind="solve", m=10000, n=10000, r=10, ratio=6.0, precision="bf16", tol=0.0,
             k_max=70),
        # Table 1's last row, the workload of bench.py, in both precisions
        dict(name="solve_30000_fp64", kind="solve", m=30000, n=30000, r=10, ratio=6.0, precision="fp64", tol=0.0,
             k_max=25),
        dict(name="solve_30000_fp32", kind="solve", m=30000, n=30000, r=10, ratio=6.0, precision="fp32", tol=0.0,
             k_max=25),
        # eight serving jobs of mixed sizes advanced in lockstep
        dict(name="batch_8_fp32", kind="batch", jobs=8, m=500, n=900, step_m=700, step_n=431, r=5, ratio=5.0,
             precision="fp32", k_max=20),
        # the sparse kernels as entry points, float64, at the block width of a rank-10 shrink
        dict(name="products_30000_fp64", kind="products", m=30000, n=30000, r=10, ratio=6.0, b=16, precision="fp64"),
        # a new problem of the 10000 x 10000 row: sampler, contexts and storage
        dict(name="build_10000_fp32", kind="build", m=10000, n=10000, r=10, ratio=6.0, precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "solve", "products", "build"])
    precision = rng.choice(["fp64", "fp64", "fp32", "fp32", "bf16"])
    m = _log_int(rng, 100, 28000)
    n = max(90, min(28000, int(round(m * math.exp(rng.uniform(-0.5, 0.5))))))
    # ranks at which the iteration settles: below them (and below ratio 5.5) the samples of a row are too few and the
    # iterate's rank runs away on many instances
    small = min(m, n) < 500
    r = rng.randint(8, 14) if not small else (rng.randint(5, 8) if min(m, n) >= 150 else 4)
    ratio = round(rng.uniform(5.5, 6.5), 2)
    case = dict(kind=kind, m=m, n=n, r=r, ratio=ratio, precision=precision)
    if kind == "products":
        case.update(precision=rng.choice(["fp64", "fp32"]), b=2 * rng.randint(4, 24), r=rng.randint(1, 40))
    elif kind == "build":
        case.update(precision=rng.choice(["fp64", "fp32"]))
    else:
        if small and precision == "bf16":
            case.update(precision="fp32")
            precision = "fp32"
        # the bfloat16 phase lasts until the residual is below 1e-2 (about 40 iterations): solves leave it
        case.update(tol=1e-9 if precision == "fp64" and max(m, n) < 400 else 0.0,
                    k_max=70 if precision == "bf16" else rng.randint(12, 60))
        if max(m, n) > 9000:
            case.update(k_max=70 if precision == "bf16" else rng.randint(8, 20))
    return case


# ------------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------------
def _nnz(m, n, r, ratio):
    return min(m * n, int(round(ratio * r * (m + n - r))))


def _problem(m, n, r, ratio, seed):
    """(rows int32, cols int32, values float64) of a planted problem, sorted row-major, on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    a = torch.randn(m, r, generator=g, device="cuda", dtype=torch.float64)
    b = torch.randn(n, r, generator=g, device="cuda", dtype=torch.float64)
    nnz = _nnz(m, n, r, ratio)
    if m * n <= 8 * nnz:
        ids = torch.randperm(m * n, generator=g, device="cuda")[:nnz]
    else:
        ids = torch.unique(torch.randint(0, m * n, (nnz + nnz // 4 + 1000,), generator=g, device="cuda"))
        ids = ids[torch.randperm(ids.numel(), generator=g, device="cuda")[:nnz]]
    ids = torch.sort(ids).values
    rows, cols = ids // n, ids % n
    vals = torch.zeros(nnz, device="cuda", dtype=torch.float64)
    for t in range(r):
        vals += a[rows, t] * b[cols, t]
    return rows.int(), cols.int(), vals


def _batch_sizes(case):
    return [(case["m"] + i * case["step_m"], case["n"] + i * case["step_n"], case["r"] + i) for i in range(case["jobs"])]


def prepare(case, seed):
    m, n, r = case["m"], case["n"], case["r"]
    if case["kind"] == "build":
        nnz = _nnz(m, n, r, case["ratio"])
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        return dict(case=case, seed=seed, vals=torch.randn(nnz, generator=g, device="cuda", dtype=torch.float64),
                    rows=torch.empty(nnz, device="cuda", dtype=torch.int32),
                    cols=torch.empty(nnz, device="cuda", dtype=torch.int32))
    if case["kind"] == "batch":
        jobs = []
        for i, (mi, ni, ri) in enumerate(_batch_sizes(case)):
            rows, cols, vals = _problem(mi, ni, ri, case["ratio"], 1000 * seed + i)
            jobs.append(Solver(mi, ni, rows, cols, vals, precision=case["precision"], k_max=case["k_max"]))
        return dict(case=case, jobs=jobs)
    rows, cols, vals = _problem(m, n, r, case["ratio"], seed)
    if case["kind"] == "products":
        s = Solver(m, n, rows, cols, vals, precision=case["precision"])
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)

        def rand(*shape):
            return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)

        b = case["b"]
        y = rand(vals.numel())
        s.set_Y(y.cpu().numpy())
        return dict(case=case, solver=s, v=rand(n, b), u=rand(m, b), ut=rand(m, r), vr=rand(n, r), y=y,
                    w=torch.empty(m, b, device="cuda", dtype=torch.float64),
                    z=torch.empty(n, b, device="cuda", dtype=torch.float64), y_out=torch.empty_like(y))
    # some 30000 x 30000 instances have an eleventh singular value close below tau for an iterate or two, and take more
    # than the default 40 Lanczos cycles to resolve it
    s = Solver(m, n, rows, cols, vals, precision=case["precision"], k_max=case["k_max"], lanczos_tol=case["tol"],
               max_cycles=200)
    return dict(case=case, solver=s, rows=rows.long(), cols=cols.long())


# ------------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------------
def _out_type(case):
    return torch.float64 if case["precision"] == "fp64" and case.get("tol", 0.0) > 0.0 else torch.float32


def run(state):
    case = state["case"]
    if case["kind"] == "build":
        sample_omega(case["m"], case["n"], state["vals"].numel(), state["seed"], state["rows"], state["cols"])
        with Solver(case["m"], case["n"], state["rows"], state["cols"], state["vals"],
                    precision=case["precision"]) as s:
            row_ptr, col_idx, col_ptr, row_idx, csc_to_csr = s.structure()
        return dict(rows=state["rows"], cols=state["cols"], row_ptr=row_ptr, col_idx=col_idx, col_ptr=col_ptr,
                    row_idx=row_idx, csc_to_csr=csc_to_csr)
    if case["kind"] == "batch":
        results, _ = batch_solve(state["jobs"], eps=1e-4, max_rank=MAX_RANK)
        return dict(y=[torch.from_numpy(s.get_Y()).float() for s in state["jobs"]],
                    iterations=[res["iterations"] for res in results], rank=[res["rank"] for res in results])
    s = state["solver"]
    if case["kind"] == "products":
        s.apply_Y(state["v"], state["w"])
        s.apply_Yt(state["u"], state["z"])
        res2 = s.sddmm_update(state["ut"], state["vr"], 1.2, state["y"], state["y_out"])
        return dict(w=state["w"], z=state["z"], y=state["y_out"], res2=res2)
    t = _out_type(case)
    res = s.solve(eps=1e-4, max_rank=MAX_RANK, raise_on_nonconvergence=False)
    u, d, v = s.factors()
    ud, vd = torch.from_numpy(u * d).cuda(), torch.from_numpy(v).cuda()
    x = (ud[state["rows"]] * vd[state["cols"]]).sum(1)
    sigma = torch.zeros(MAX_RANK, dtype=t)   # sigma_i - tau, zeros past the rank
    sigma[:d.size] = torch.from_numpy(d)
    return dict(x=x.to(t), y=torch.from_numpy(s.get_Y()).to(t), sigma=sigma,
                iterations=res["iterations"], rank=res["rank"])


# ------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------------
def _solve_work(m, n, r, nnz, k, value_bytes):
    # per iteration: Omega's indices and Y once for each of the two products of a shrink with r + 1 columns, once more
    # (with M and the new Y) for the dual step; the two bases orthonormalised once (Gram and update)
    entry = 4 + value_bytes
    nbytes = k * nnz * (2 * entry + entry + 2 * value_bytes) + 8.0 * (m + n) * (r + 1) * k
    flops = k * (2 * 2.0 * nnz * (r + 1) + 2.0 * nnz * r + 4.0 * (m + n) * (r + 1) ** 2)
    return nbytes + 8.0 * (m + n) * r + 2 * value_bytes * nnz, flops


def work(case):
    m, n, r = case["m"], case["n"], case["r"]
    nnz = _nnz(m, n, r, case["ratio"])
    vb = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "build":
        # sampled ids written and read, five index arrays written; one hash (about ten operations) per id of m n
        return {"bytes": nnz * (8.0 + 16.0 + 20.0) + 8.0 * (m + n), "flops": 10.0 * m * n}
    if case["kind"] == "products":
        b = case["b"]
        nbytes = 2 * (nnz * (4.0 + vb) + 8.0 * b * (m + n)) + nnz * (4.0 + vb + 16.0) + 8.0 * r * (m + n)
        return {"bytes": nbytes, "flops": 2 * 2.0 * nnz * b + (2.0 * r + 4.0) * nnz}
    if case["kind"] == "batch":
        parts = [_solve_work(mi, ni, ri, _nnz(mi, ni, ri, case["ratio"]), case["k_max"], vb)
                 for mi, ni, ri in _batch_sizes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    nbytes, flops = _solve_work(m, n, r, nnz, case["k_max"], vb)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------------------
# The same in 64 bits
# ------------------------------------------------------------------------------------------------
def _exact_solve(m, n, rows, cols, vals, k_max):
    """Algorithm 1 on a dense iterate, D_tau(Y) = Y V diag((sigma - tau)_+ / sigma) V^T from the eigenvectors of the
    smaller Gram matrix."""
    if m < n:
        return _exact_solve(n, m, cols, rows, vals, k_max)
    tau, delta = 5.0 * math.sqrt(m * n), 1.2 * m * n / vals.numel()
    y = torch.zeros(m, n, device="cuda", dtype=torch.float64)
    y[rows, cols] = vals
    norm2 = float(torch.linalg.eigvalsh(y.T @ y)[-1].sqrt())
    y *= math.ceil(tau / (delta * norm2)) * delta
    for k in range(k_max):
        lam, v = torch.linalg.eigh(y.T @ y)
        sig = lam.clamp_min(0.0).sqrt()
        keep = sig > tau
        v, sig = v[:, keep].flip(1), sig[keep].flip(0)
        x = ((y @ (v * ((sig - tau) / sig))) @ v.T)[rows, cols]
        e = vals - x
        if float(e.norm() / vals.norm()) <= 1e-4:
            break
        y[rows, cols] += delta * e
    sigma = torch.zeros(MAX_RANK, dtype=torch.float64)
    sigma[:sig.numel()] = (sig - tau).cpu()
    return x, y[rows, cols], sigma


def exact(case, seed):
    if case["kind"] == "products":
        m, n, r = case["m"], case["n"], case["r"]
        s = prepare(dict(case, precision="fp64"), seed)
        rows, cols, vals = _problem(m, n, r, case["ratio"], seed)
        s["solver"].close()
        rows, cols = rows.long(), cols.long()
        w = torch.zeros_like(s["w"]).index_add_(0, rows, s["y"][:, None] * s["v"][cols])
        z = torch.zeros_like(s["z"]).index_add_(0, cols, s["y"][:, None] * s["u"][rows])
        e = vals - (s["ut"][rows] * s["vr"][cols]).sum(1)
        return dict(w=w, z=z, y=s["y"] + 1.2 * e, res2=float((e * e).sum()))
    if case["kind"] != "solve" or min(case["m"], case["n"]) > 1100 or max(case["m"], case["n"]) > 4000:
        return None
    rows, cols, vals = _problem(case["m"], case["n"], case["r"], case["ratio"], seed)
    x, y, sigma = _exact_solve(case["m"], case["n"], rows.long(), cols.long(), vals, case["k_max"])
    return dict(x=x, y=y, sigma=sigma, iterations=None, rank=None)
