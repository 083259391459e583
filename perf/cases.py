"""The calls whose speed this library is judged by: its public entry points at
the sizes a program uses them at, from one operator application on a small
mesh to a whole multilevel estimate.

A case is a dict of plain values. ``kind`` names the path:

  apply    y = A(kappa) x on one mesh, FP64 or FP32 (Plan.apply, Plan.apply32)
  field    KLE coefficients and the lognormal field of one mesh, FP64 or the
           tensor-core FP32 form (Plan.draw_xi + Plan.kappa / Plan.kappa32)
  solve    a batch of solves for a caller's own kappa (Plan.solve)
  sample   coupled samples of one level (Plan.sample_level)
  run      a whole estimate: fixed sample counts, or adaptive to eps (Plan.run)
  serve    a burst of estimation requests to the server (Server.submit, drain)

Iteration counts are a property of the solver, not a result of the call: the
cases return solutions, quantities of interest, sample counts and statistics.

``exact`` computes the same results from the formulas in plain numpy and torch
(64 bits): Philox4x32-10 + Box-Muller coefficients, the closed-form
exponential-covariance KLE, the Q1 element matrices and Jacobi-preconditioned
CG run to the rounding level.
"""
import math

import numpy as np
import torch

from paper_2111_11788_gb300 import mlmc

BOX = (0.25, 0.75)

# --------------------------------------------------------------------- cases

_FIELD2 = dict(sigma2=1.0, corr_len=0.1, m=8, total_order=-1)
_FIELD3 = dict(sigma2=1.0, corr_len=0.2, m=5, total_order=-1)


def listed():
    return [
        # The smallest call: one operator application on an odd-sized mesh, as
        # a program that writes its own Krylov loop around the operator issues
        # it. Latency of the binding and of one launch.
        dict(name="apply-2d-small", kind="apply", dim=2, n=45, count=1, fp32=False, **_FIELD2),
        # The FP32 operator of the mixed form on a large 3D batch.
        dict(name="apply32-3d", kind="apply", dim=3, n=128, count=16, fp32=True, **_FIELD3),
        # The log-normal field of a batch on a fine 2D mesh, FP64.
        dict(name="field-2d", kind="field", dim=2, n=512, count=64, fp32=False, **_FIELD2),
        # The FP32 field from the tensor cores, 343 modes on a 3D mesh.
        dict(name="field32-3d", kind="field", dim=3, n=64, count=32, fp32=True, sigma2=1.0,
             corr_len=0.1, m=7, total_order=-1),
        # A caller's own coefficient on a mesh that is no power of two:
        # Jacobi-PCG, FP64, tight tolerance.
        dict(name="solve-2d-jacobi", kind="solve", dim=2, n=100, count=20, solver="jacobi", precision="fp64",
             qoi="domain", rtol=1e-11, sigma2=1.0, corr_len=0.3, m=4, total_order=-1),
        # A caller's own coefficient in 3D, multigrid, mixed form.
        dict(name="solve-3d-mixed", kind="solve", dim=3, n=64, count=16, solver="gmg", precision="mixed",
             qoi="box", rtol=1e-10, **_FIELD3),
        # An ordinary level of a 2D hierarchy: coupled samples on 256^2 and
        # 128^2, FP64 multigrid.
        dict(name="sample-2d-fp64", kind="sample", dim=2, n0=32, level=3, first=100, count=40, solver="gmg",
             precision="fp64", qoi="domain", rtol=1e-10, **_FIELD2),
        # The finest level of a 3D hierarchy (128^3 and 64^3), FP64 multigrid.
        dict(name="sample-3d-fp64", kind="sample", dim=3, n0=8, level=4, first=0, count=6, solver="gmg",
             precision="fp64", qoi="box", rtol=1e-10, **_FIELD3),
        # A whole estimate in the mixed form, 32^2..512^2, adaptive to eps.
        dict(name="run-2d-mixed", kind="run", dim=2, n0=32, levels=5, eps=1e-3, pilot=100, N="",
             solver="gmg", precision="mixed", qoi="domain", rtol=1e-10, **_FIELD2),
        # A whole estimate in 3D, mixed form, 16^3..256^3, fixed counts.
        dict(name="run-3d-mixed", kind="run", dim=3, n0=16, levels=5, eps=0.0, pilot=0, N="64,32,16,8,4",
             solver="gmg", precision="mixed", qoi="box", rtol=1e-10, sigma2=1.0, corr_len=0.1, m=7,
             total_order=-1),
        # The largest: the benchmark's estimate, 32^2..1024^2, FP64, to eps.
        dict(name="run-2d-fp64", kind="run", dim=2, n0=32, levels=6, eps=1e-3, pilot=100, N="",
             solver="gmg", precision="fp64", qoi="domain", rtol=1e-10, **_FIELD2),
        # A burst of requests of the serving mix (2D and 3D, every request
        # with its own field and tolerance), adaptive levels.
        dict(name="serve-burst", kind="serve", requests=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _field_of(rng, dim):
    corr = round(rng.uniform(0.05, 0.3), 4)
    cap = 8 if dim == 2 else 7
    f = dict(sigma2=round(rng.uniform(0.5, 2.0), 4), corr_len=corr, m=min(int(math.ceil(1.5 / corr)), cap),
             total_order=-1)
    if rng.random() < 0.25:   # a total-order truncation of a larger basis
        f.update(m=min(f["m"] + 4, 12), total_order=f["m"] + 2)
    return f


def _pow2(rng, lo, hi):
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def draw(rng):
    kind = rng.choice(["apply", "apply", "field", "field", "solve", "solve", "sample", "sample", "sample",
                       "run", "run", "serve"])
    dim = rng.choice([2, 3])
    f = _field_of(rng, dim)
    if kind == "apply":
        n = _log_int(rng, 12, 1024) if dim == 2 else _log_int(rng, 6, 144)
        count = min(_log_int(rng, 1, 256), max(1, (1 << 25) // n ** dim))
        return dict(kind=kind, dim=dim, n=n, count=count, fp32=rng.random() < 0.5, **f)
    if kind == "field":
        n = _log_int(rng, 12, 1024) if dim == 2 else _log_int(rng, 6, 128)
        count = min(_log_int(rng, 1, 256), max(1, (1 << 24) // n ** dim))
        return dict(kind=kind, dim=dim, n=n, count=count, fp32=rng.random() < 0.5, **f)
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(1, 12))
    solver = rng.choice(["gmg", "gmg", "jacobi"])
    prec = rng.choice(["fp64", "mixed"])
    # the QoI box has to fall on nodes of every mesh
    qoi = rng.choice(["domain", "box"])
    base = dict(kind=kind, dim=dim, solver=solver, precision=prec, qoi=qoi,
                rtol=rng.choice([1e-8, 1e-10, 1e-11]), **f)
    if kind == "solve":
        if solver == "gmg":
            n = _pow2(rng, 8, 1024) if dim == 2 else _pow2(rng, 4, 64)
            most = (1 << 23) if dim == 2 else (1 << 22)
        else:
            n = _log_int(rng, 9, 240) if dim == 2 else _log_int(rng, 6, 60)
            most = 1 << 19
            if qoi == "box":
                n = max(8, n // 4 * 4)
        base.update(n=n, count=min(_log_int(rng, 1, 256), max(1, most // n ** dim)))
        return base
    if kind == "sample":
        if solver == "gmg":
            n0 = _pow2(rng, 8, 64) if dim == 2 else _pow2(rng, 4, 16)
            level = rng.randint(0, 4 if dim == 2 else 3)
            most = (1 << 23) if dim == 2 else (1 << 22)
        else:
            n0 = rng.randint(5, 30) if dim == 2 else rng.randint(4, 12)
            level = rng.randint(0, 3 if dim == 2 else 2)
            most = 1 << 19
            if qoi == "box":
                n0 = max(4, n0 // 4 * 4)
        n = n0 << level
        base.update(n0=n0, level=level, first=rng.randint(0, 1 << 20),
                    count=min(_log_int(rng, 1, 256), max(1, most // n ** dim)))
        return base
    # a small to ordinary estimate with counts falling by level
    base.update(solver="gmg")
    n0 = _pow2(rng, 8, 32) if dim == 2 else _pow2(rng, 4, 16)
    levels = rng.randint(2, 4 if dim == 2 else 3)
    top = _log_int(rng, 8, 400)
    base.update(n0=n0, levels=levels, eps=0.0, pilot=0,
                N=",".join(str(max(1, top >> (l * (2 if dim == 2 else 3)))) for l in range(levels)))
    if rng.random() < 0.4:
        base.update(N="", eps=round(rng.uniform(1e-3, 5e-3), 5), pilot=rng.randint(16, 64))
    return base


# ------------------------------------------------------------ inputs, one pass

def _config(case, seed, **over):
    a = dict(dim=case["dim"], sigma2=case["sigma2"], corr_len=case["corr_len"], modes_per_dim=case["m"],
             total_order=case["total_order"], qoi=case.get("qoi", "domain"), box=BOX,
             solver=case.get("solver", "jacobi"), precision=case.get("precision", "fp64"),
             rtol=case.get("rtol", 1e-10), seed=seed, n_levels=1)
    a.update(over)
    return mlmc.config(**a)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _serve_requests(case, seed):
    """(configuration arguments, eps) of the requests of one burst."""
    rng = np.random.default_rng(seed)
    out = []
    for k in range(case["requests"]):
        eps = float(rng.uniform(5e-4, 5e-3))
        dim = 2 if rng.random() < 0.5 else 3
        sigma2, corr = float(rng.uniform(0.5, 2.0)), float(rng.uniform(0.05, 0.3))
        m = min(int(math.ceil(1.5 / corr)), 8 if dim == 2 else 7)
        out.append((dict(dim=dim, n_levels=6 if dim == 2 else 5, coarse_cells=32 if dim == 2 else 8,
                         modes_per_dim=m, sigma2=sigma2, corr_len=corr, qoi="domain" if dim == 2 else "box",
                         box=BOX, solver="gmg", precision="mixed", rtol=1e-10, seed=seed, stream_id=k), eps))
    return out


def _kappa_input(case, seed, device="cuda"):
    """A caller's log-normal coefficient on a mesh, (count, n^dim) doubles."""
    dim, n, m = case["dim"], case["n"], case["m"]
    M = len(_modes(dim, m, case["total_order"]))
    g = torch.Generator().manual_seed(seed)
    xi = torch.randn(case["count"], M, generator=g, dtype=torch.float64).to(device)
    return _lognormal(dim, n, case, xi)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        # the server is kept by a serving program; requests are what comes in
        return dict(kind=kind, server=mlmc.Server(hbm_budget=8 << 30, max_slots=8, pilot=32, adapt_from=2),
                    requests=[(mlmc.config(**a), eps) for a, eps in _serve_requests(case, seed)])
    dim = case["dim"]
    if kind in ("apply", "field", "solve"):
        n, B = case["n"], case["count"]
        ns, es = mlmc.node_stride(dim, n), mlmc.elem_stride(dim, n)
        nn, ne = (n + 1) ** dim, n ** dim
    if kind == "apply":
        plan = mlmc.Plan(_config(case, seed, coarse_cells=n), _stream())
        dt = torch.float32 if case["fp32"] else torch.float64
        kap = torch.zeros(B, es, dtype=dt, device="cuda")
        kap[:, :ne] = _kappa_input(case, seed).to(dt)
        x = torch.zeros(B, ns, dtype=dt, device="cuda")
        x[:, :nn] = _vector(case, seed).to(dt)
        y = torch.zeros(B, ns, dtype=dt, device="cuda")
        return dict(kind=kind, plan=plan, kap=kap, x=x, y=y, out=y[:, :nn], B=B,
                    call=plan.apply32 if case["fp32"] else plan.apply)
    if kind == "field":
        cfg = _config(case, seed, coarse_cells=n)
        plan = mlmc.Plan(cfg, _stream())
        xi = torch.zeros(B, mlmc.coef_count(cfg), dtype=torch.float64, device="cuda")
        kap = torch.zeros(B, es, dtype=torch.float32 if case["fp32"] else torch.float64, device="cuda")
        return dict(kind=kind, plan=plan, xi=xi, kap=kap, out=kap[:, :ne], B=B,
                    call=plan.kappa32 if case["fp32"] else plan.kappa)
    if kind == "solve":
        plan = mlmc.Plan(_config(case, seed, coarse_cells=n), _stream())
        kap = torch.zeros(B, es, dtype=torch.float64, device="cuda")
        kap[:, :ne] = _kappa_input(case, seed)
        u = torch.zeros(B, ns, dtype=torch.float64, device="cuda")
        q = torch.zeros(B, dtype=torch.float64, device="cuda")
        return dict(kind=kind, plan=plan, kap=kap, u=u, q=q, out=u[:, :nn], B=B)
    if kind == "sample":
        cfg = _config(case, seed, coarse_cells=case["n0"], n_levels=case["level"] + 1)
        return dict(kind=kind, plan=mlmc.Plan(cfg, _stream()), case=case)
    cfg = _config(case, seed, coarse_cells=case["n0"], n_levels=case["levels"])
    N = [int(v) for v in case["N"].split(",")] if case["N"] else None
    return dict(kind=kind, plan=mlmc.Plan(cfg, _stream()), N=N, eps=case["eps"], pilot=case["pilot"],
                levels=case["levels"])


def run(s):
    kind = s["kind"]
    if kind == "apply":
        s["call"](0, s["kap"].data_ptr(), s["x"].data_ptr(), s["y"].data_ptr(), s["B"])
        return s["out"]
    if kind == "field":
        s["plan"].draw_xi(0, 0, s["B"], s["xi"].data_ptr())
        s["call"](0, s["xi"].data_ptr(), s["B"], s["kap"].data_ptr())
        return dict(xi=s["xi"], kappa=s["out"])
    if kind == "solve":
        s["plan"].solve(0, s["kap"].data_ptr(), s["B"], s["u"].data_ptr(), s["q"].data_ptr(), 0)
        return dict(u=s["out"], q=s["q"])
    if kind == "sample":
        c = s["case"]
        qf, qc, _ = s["plan"].sample_level(c["level"], c["first"], c["count"])
        return dict(qf=qf, qc=qc)
    if kind == "run":
        q, v, N = s["plan"].run(eps=s["eps"], pilot=s["pilot"], N=s["N"])
        st = [s["plan"].level_stats(l) for l in range(s["levels"])]
        return dict(q=q, var=v, N=N, mean=np.array([t[1] for t in st]), m2=np.array([t[2] for t in st]))
    srv = s["server"]
    ids = [srv.submit(cfg, eps) for cfg, eps in s["requests"]]
    srv.drain(120.0)
    res = [srv.poll(i) for i in ids]
    return dict(q=np.array([r["q_hat"] for r in res]), var=np.array([r["stat_var"] for r in res]),
                N=np.array([r["N"] for r in res]), status=np.array([r["status"] for r in res]))


# ------------------------------------------------------------- work, tolerance

def work(case):
    """Bytes and operations no implementation does without: each input read
    and each output written once; for solves, one write and one read of kappa
    per mesh and one application of the operator per unknown (the number of
    iterations, and what they move, is the implementation's own)."""
    kind = case["kind"]
    if kind == "serve":
        # 32 pilot samples on the first three levels of each request
        unk = case["requests"] * 32 * 0.5 * (sum((32 << l) ** 2 for l in range(3)) + sum((8 << l) ** 3 for l in range(3)))
        return dict(bytes=16.0 * unk, flops=40.0 * unk)
    dim = case["dim"]
    ops = 17 if dim == 2 else 53   # one row of the operator
    M = len(_modes(dim, case["m"], case["total_order"]))
    if kind in ("apply", "field", "solve"):
        n, B = case["n"], case["count"]
        nn, ne = float(n + 1) ** dim, float(n) ** dim
    if kind == "apply":
        return dict(bytes=B * (2 * nn + ne) * (4 if case["fp32"] else 8), flops=B * (n - 1.0) ** dim * ops)
    if kind == "field":
        return dict(bytes=B * (ne * (4 if case["fp32"] else 8) + 8.0 * M), flops=B * ne * (2.0 * case["m"] + 10))
    if kind == "solve":
        return dict(bytes=8.0 * B * (ne + nn + 1), flops=B * nn * ops)

    def level(n, count):
        both = float(n) ** dim + (float(n // 2) ** dim)
        return np.array([16.0 * count * both, count * both * (2.0 * case["m"] + 10 + ops)])
    if kind == "sample":
        b, f = level(case["n0"] << case["level"], case["count"])
        return dict(bytes=float(b), flops=float(f))
    N = [int(v) for v in case["N"].split(",")] if case["N"] else [case["pilot"]] * case["levels"]
    b, f = sum(level(case["n0"] << l, N[l]) for l in range(case["levels"]))
    return dict(bytes=float(b), flops=float(f))


def tolerance(case):
    kind = case["kind"]
    if kind == "apply":
        # rounding of one row, a sum of 9 (2D) or 21 (3D) products: about
        # 7e-8 and 1.5e-16 seen against 64 bits
        return dict(rel=3e-7, max=1.2e-5) if case["fp32"] else dict(rel=1e-15, max=4e-14)
    if kind == "field":
        # FP32: both factors in two BF16 terms, up to 1e-5 seen; FP64: m-term
        # sums and one exp of a field of up to a few units, 3e-16 .. 1e-15 seen
        return dict(rel=4e-5, max=1.6e-3) if case["fp32"] else dict(rel=4e-15, max=1.6e-13)
    # a solve stops at ||r|| <= rtol ||b||, and any iterate that does is a
    # result: runs that differ in the smoother's damping, the initial iterate
    # or the form are up to 0.15 rtol apart in u and Q, 0.75 rtol in a variance
    r = case.get("rtol", 1e-10)
    return dict(rel=3 * r, max=60 * r)


# --------------------------------------------------- the same results, 64 bits

def _modes(dim, m, total_order):
    """Per-axis mode numbers (k_x, k_y[, k_z]) of the kept modes, x fastest."""
    idx = np.stack(np.meshgrid(*([np.arange(m)] * dim), indexing="ij"), -1).reshape(-1, dim)[:, ::-1]
    return idx[idx.sum(1) <= total_order] if total_order >= 0 else idx


def _axis_table(n, corr_len, m):
    """sqrt(theta_k) f_k at the n element centres of [0, 1], k < m."""
    c = 1.0 / corr_len
    out = np.empty((n, m))
    t = (np.arange(n) + 0.5) / n - 0.5
    for k in range(m):
        even = k % 2 == 0

        def f(w):
            return (c * math.cos(w / 2) - w * math.sin(w / 2) if even
                    else w * math.cos(w / 2) + c * math.sin(w / 2))
        lo, hi = k * math.pi, (k + 1) * math.pi
        neg = f(lo) < 0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if (f(mid) < 0) == neg:
                lo = mid
            else:
                hi = mid
        w = 0.5 * (lo + hi)
        s2 = math.sin(w) / (2 * w)
        e = np.cos(w * t) / math.sqrt(0.5 + s2) if even else np.sin(w * t) / math.sqrt(0.5 - s2)
        out[:, k] = math.sqrt(2 * c / (w * w + c * c)) * e
    return out


def _lognormal(dim, n, case, xi):
    """exp(Phi xi) at the element centres, (B, n^dim), x fastest."""
    m = case["m"]
    F = torch.from_numpy(_axis_table(n, case["corr_len"], m)).to(xi.device)
    idx = _modes(dim, m, case["total_order"])
    flat = torch.from_numpy((idx * m ** np.arange(dim)).sum(1).astype(np.int64)).to(xi.device)
    full = torch.zeros(xi.shape[0], m ** dim, dtype=torch.float64, device=xi.device)
    full[:, flat] = xi
    g = full.reshape(-1, *([m] * dim))                   # (B, [kz,] ky, kx)
    g = torch.einsum("byx,iy,jx->bij", g, F, F) if dim == 2 else \
        torch.einsum("bzyx,hz,iy,jx->bhij", g, F, F, F)
    return torch.exp(math.sqrt(case["sigma2"]) * g).reshape(xi.shape[0], -1)


def _vector(case, seed):
    n = case["n"]
    g = torch.Generator().manual_seed(seed + 77)
    return torch.randn(case["count"], (n + 1) ** case["dim"], generator=g, dtype=torch.float64).cuda()


def _philox_normals(seed, stream_id, level, first, count, M):
    """xi (count, M): Philox4x32-10, counter (pair, sample, level, stream), Box-Muller."""
    u32, mask = np.uint64(32), np.uint64(0xFFFFFFFF)
    P = (M + 1) // 2
    j, i = np.meshgrid(np.arange(P, dtype=np.uint64), np.arange(first, first + count, dtype=np.uint64))
    c = [j, i, np.full_like(j, level), np.full_like(j, stream_id)]
    k = [np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)]
    for r in range(10):
        if r:
            k = [(k[0] + np.uint64(0x9E3779B9)) & mask, (k[1] + np.uint64(0xBB67AE85)) & mask]
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> u32) ^ c[1] ^ k[0], b & mask, (a >> u32) ^ c[3] ^ k[1], a & mask]

    def uniform(hi, lo):
        return (((hi << np.uint64(20)) | (lo >> np.uint64(12))).astype(np.float64) + 0.5) * 2.0 ** -52
    r, t = np.sqrt(-2 * np.log(uniform(c[0], c[1]))), 2 * np.pi * uniform(c[2], c[3])
    xi = np.stack([r * np.cos(t), r * np.sin(t)], -1).reshape(count, 2 * P)[:, :M]
    return torch.from_numpy(np.ascontiguousarray(xi)).cuda()


def _apply(dim, n, kap, u):
    """Q1 stiffness times u: per element and corner, with S the sum of the
    element's values: 2D kappa/6 (5 u - S - opposite), 3D kappa h/12 (5 u - S +
    the three values along the edges at the corner)."""
    B = u.shape[0]
    kap, u = kap.reshape(B, *([n] * dim)), u.reshape(B, *([n + 1] * dim)).clone()
    for a in range(1, dim + 1):   # homogeneous Dirichlet: boundary values count as 0
        u.select(a, 0).zero_()
        u.select(a, n).zero_()

    def cut(t, c):
        return t[(slice(None),) + tuple(slice(b, b + n) for b in c)]
    corners = [tuple((v >> a) & 1 for a in range(dim)) for v in range(2 ** dim)]
    S = sum(cut(u, c) for c in corners)
    y = torch.zeros_like(u)
    k = kap / 6 if dim == 2 else kap / (12 * n)
    for c in corners:
        if dim == 2:
            v = 5 * cut(u, c) - S - cut(u, tuple(1 - b for b in c))
        else:
            v = 5 * cut(u, c) - S
            for a in range(3):
                v += cut(u, c[:a] + (1 - c[a],) + c[a + 1:])
        cut(y, c).add_(k * v)
    for a in range(1, dim + 1):
        y.select(a, 0).zero_()
        y.select(a, n).zero_()
    return y.reshape(B, -1)


def _solve(dim, n, kap):
    """u of A(kappa) u = b (b_i = h^dim inside) by Jacobi-PCG to the rounding
    level, with a second solve for the correction."""
    B, shape = kap.shape[0], [kap.shape[0]] + [n + 1] * dim
    k = kap.reshape(B, *([n] * dim))
    D = torch.zeros(shape, dtype=torch.float64, device=kap.device)
    for v in range(2 ** dim):
        D[(slice(None),) + tuple(slice((v >> a) & 1, ((v >> a) & 1) + n) for a in range(dim))] += k
    D *= 2.0 / 3.0 if dim == 2 else 1.0 / (3 * n)
    inner = torch.zeros(shape[1:], dtype=torch.float64, device=kap.device)
    inner[tuple(slice(1, n) for _ in range(dim))] = 1.0
    inner = inner.reshape(1, -1)
    W = inner / D.reshape(B, -1)
    b = (inner * (1.0 / n) ** dim).expand(B, -1)
    bn = b.norm(dim=1, keepdim=True)

    def pcg(rhs, tol):
        x = torch.zeros_like(rhs)
        r = rhs.clone()
        z = W * r
        p = z.clone()
        rz = (r * z).sum(1, keepdim=True)
        for it in range(40 * n + 500):
            q = _apply(dim, n, kap, p)
            a = rz / (p * q).sum(1, keepdim=True).clamp_min(1e-300)
            x += a * p
            r -= a * q
            if it % 20 == 0 and bool((r.norm(dim=1, keepdim=True) <= tol * bn).all()):
                break
            z = W * r
            new = (r * z).sum(1, keepdim=True)
            p = z + (new / rz.clamp_min(1e-300)) * p
            rz = new
        return x
    u = pcg(b.clone(), 1e-13)
    return u + pcg(b - _apply(dim, n, kap, u), 1e-15)


def _qoi(case, dim, n, u):
    h = 1.0 / n
    w = torch.zeros(n + 1, dtype=torch.float64, device=u.device)
    if case["qoi"] == "box":
        lo, hi = round(BOX[0] * n), round(BOX[1] * n)
        w[lo:hi + 1] = 1.0
        w[lo] = w[hi] = 0.5
        w *= h / (BOX[1] - BOX[0])
    else:
        w[1:n] = h
    u = u.reshape(u.shape[0], *([n + 1] * dim))
    for _ in range(dim):
        u = u @ w
    return u


def _coupled(case, seed, level, first, count):
    """(Q_l, Q_{l-1}) of samples first .. first + count - 1, in slices."""
    dim, M = case["dim"], len(_modes(case["dim"], case["m"], case["total_order"]))
    qf, qc = [], []
    step = max(1, (1 << 25) // (case["n0"] << level) ** dim)
    for s in range(first, first + count, step):
        c = min(step, first + count - s)
        xi = _philox_normals(seed, 0, level, s, c, M)
        for mesh, to in ((level, qf), (level - 1, qc)):
            if mesh < 0:
                to.append(torch.zeros(c, dtype=torch.float64))
                continue
            n = case["n0"] << mesh
            to.append(_qoi(case, dim, n, _solve(dim, n, _lognormal(dim, n, case, xi))).cpu())
    return torch.cat(qf).numpy(), torch.cat(qc).numpy()


def _cg_cost(dim, n, count):
    """Seconds of _solve, roughly: passes over the batch and launches per iteration."""
    return (4.5 if dim == 2 else 5.0) * n * (6e-4 + (60 if dim == 2 else 140) * 8.0 * count * float(n) ** dim / 4e12)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None
    dim = case["dim"]
    if kind == "apply":
        kap, x = _kappa_input(case, seed), _vector(case, seed)
        if case["fp32"]:
            kap, x = kap.float().double(), x.float().double()
        return _apply(dim, case["n"], kap, x)
    if kind == "field":
        M = len(_modes(dim, case["m"], case["total_order"]))
        xi = _philox_normals(seed, 0, 0, 0, case["count"], M)
        return dict(xi=xi, kappa=_lognormal(dim, case["n"], case, xi))
    if kind == "solve":
        if _cg_cost(dim, case["n"], case["count"]) > 10:
            return None
        u = _solve(dim, case["n"], _kappa_input(case, seed))
        return dict(u=u, q=_qoi(case, dim, case["n"], u))
    if kind == "sample":
        if 1.4 * _cg_cost(dim, case["n0"] << case["level"], case["count"]) > 10:
            return None
        qf, qc = _coupled(case, seed, case["level"], case["first"], case["count"])
        return dict(qf=qf, qc=qc)
    L = case["levels"]
    have, target = [0] * L, [int(v) for v in case["N"].split(",")] if case["N"] else [case["pilot"]] * L
    if sum(1.4 * _cg_cost(dim, case["n0"] << l, target[l]) for l in range(L)) > 10:
        return None
    n = [float(case["n0"] << l) for l in range(L)]
    cost = [(n[l] - 1) ** dim + ((n[l] / 2 - 1) ** dim if l else 0.0) for l in range(L)]
    Y = [np.zeros(0)] * L
    while True:
        for l in range(L):
            if target[l] > have[l]:
                qf, qc = _coupled(case, seed, l, have[l], target[l] - have[l])
                Y[l] = np.concatenate([Y[l], qf - qc])
                have[l] = target[l]
        if case["N"]:
            break
        V = [float(y.var()) for y in Y]
        s = sum(math.sqrt(v * c) for v, c in zip(V, cost))
        want = [math.ceil(2.0 / case["eps"] ** 2 * math.sqrt(v / c) * s) for v, c in zip(V, cost)]
        if all(w <= t for w, t in zip(want, target)):
            break
        target = [max(w, t) for w, t in zip(want, target)]
    mean, m2 = np.array([y.mean() for y in Y]), np.array([y.var() * y.size for y in Y])
    return dict(q=float(mean.sum()), var=float(sum(m2[l] / have[l] / have[l] for l in range(L))),
                N=np.array(have, dtype=np.int64), mean=mean, m2=m2)
