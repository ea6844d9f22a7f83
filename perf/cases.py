"""Workloads of the LoRADS library through its public calls, with their sizes.

Four kinds, each what a program does with the library:
  op     one operator call on device arrays (lorads_op_hessian / _spmm / _sddmm)
  solve  one solve, to the final test or to an iteration budget, and the download of its
         solution (Problem.solve, Problem.solution)
  batch  many small problems in one launch (lorads_solve_batch)
  gnn    the learned warm start: a forward pass, or a training step with its gradients and
         the updated parameters

`listed()` gives fixed cases, `draw(rng)` others of the same ranges.  `prepare(case, seed)`
makes what a program holds before the call, `run(state)` is the call, `work(case)` the bytes and
operations of one pass that nothing can save, `exact(case, seed)` the results in 64 bits.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2403_09133_gb300 import instances as I
from paper_2403_09133_gb300 import lorads as L

HID, CATW, RMAX, NLAYER, BETA = 64, 128, 16, 3, 0.1


# --------------------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest operator call: the ER n = 500 graph of the plain FP64 workload, where
        # the launch and the host path count
        dict(name="hessian_er500_f64", kind="op", op="hessian", family="er", n=500, deg=8.0, r=9,
             prec="fp64"),
        # eq. linU's operator on a grid graph beyond the L2 cache (MaxCut on 1024 x 1024)
        dict(name="hessian_torus1024_f32", kind="op", op="hessian", family="torus", a=1024, b=1024,
             r=20, prec="mixed"),
        # the same operator where every row carries hundreds of entries: matrix completion at
        # the sampling density of the n = 40,000 workload
        dict(name="hessian_mc10000_f32", kind="op", op="hessian", family="mc", n1=5000, n2=5000,
             samples=1_000_000, r=20, prec="mixed"),
        # (A^T(w) - C) V of Phase I's gradient on a sparse random graph, odd row count, FP64
        dict(name="spmm_er99991_f64", kind="op", op="spmm", family="er", n=99_991, deg=6.0, r=17,
             prec="fp64"),
        # the same product in FP32 on matrix completion, ragged block sizes
        dict(name="spmm_mc6400_f32", kind="op", op="spmm", family="mc", n1=2501, n2=3899,
             samples=500_000, r=19, prec="mixed"),
        # the residual's sampled products A(U V^T), FP64 like the dual step
        dict(name="sddmm_mc10000_f64", kind="op", op="sddmm", family="mc", n1=5000, n2=5000,
             samples=1_000_000, r=20, prec="fp64"),
        # the plain FP64 method on the ER n = 500 MaxCut: Phase I and a budget of Phase II
        # iterations, the form a program with a deadline runs
        dict(name="solve_er500_f64", kind="solve", family="er", n=500, deg=8.0, prec="fp64",
             sub="cg", cap=300),
        # the headline: the 141 x 141 toroidal MaxCut with +-1 weights, mixed form, to the final
        # test (Phase III and the eigenvalue tests included)
        dict(name="solve_torus141_mixed", kind="solve", family="torus", a=141, b=141, prec="mixed",
             sub="cg", cap=5000),
        # matrix completion: Phase I on long constraint lists, general CG
        dict(name="solve_mc1000_mixed", kind="solve", family="mc", n1=520, n2=480, samples=40_000,
             prec="mixed", sub="cg", cap=40),
        # uneven batch of ER MaxCuts, a quarter of the 512-problem workload, at a kept choice of
        # CTA size and lanes per row
        dict(name="batch_128_mixed", kind="batch", count=128, n_lo=64, n_hi=2048, prec="mixed",
             threads=384),
        # the network's proposal for the largest graphs of the learned start
        dict(name="gnn_forward_20000", kind="gnn", step="forward", n=20_000, deg=6.5),
        # one training step at the size of its training graphs
        dict(name="gnn_train_3000", kind="gnn", step="train", n=3001, deg=6.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_instance(rng, whole):
    family = rng.choice(["er", "torus", "mc"])
    if family == "er":
        n = _log_int(rng, 100, 2000) if whole else _log_int(rng, 300, 300_000)
        return dict(family="er", n=n, deg=round(rng.uniform(3.0, 12.0), 2))
    if family == "torus":
        hi = 90 if whole else 900
        return dict(family="torus", a=_log_int(rng, 12, hi), b=_log_int(rng, 12, hi))
    if whole:
        n1, n2 = _log_int(rng, 80, 700), _log_int(rng, 80, 700)
        # enough samples for recovery: several times the 5 (n1 + n2) degrees of freedom
        samples = min(int(0.6 * n1 * n2), int(rng.uniform(6.0, 9.0) * 5 * (n1 + n2)))
    else:
        n1, n2 = _log_int(rng, 200, 5000), _log_int(rng, 200, 5000)
        samples = max(1000, int(rng.uniform(0.02, 0.04) * n1 * n2))
    return dict(family="mc", n1=n1, n2=n2, samples=samples)


def draw(rng):
    kind = rng.choice(["op", "op", "op", "solve", "solve", "batch", "gnn"])
    if kind == "op":
        c = dict(kind="op", op=rng.choice(["hessian", "spmm", "sddmm"]))
        c.update(_draw_instance(rng, False))
        # the initial rank, or a rank after growth
        r = _r0(_m_of(c))
        c["r"] = min(48, int(math.ceil(r * rng.choice([1.0, 1.0, 1.5, 2.25]))))
        c["prec"] = rng.choice(["fp64", "mixed"])
        return c
    if kind == "solve":
        c = dict(kind="solve")
        c.update(_draw_instance(rng, True))
        c["prec"] = rng.choice(["fp64", "mixed"])
        c["sub"] = rng.choice(["cg", "cg", "row_direct"]) if c["family"] != "mc" else "cg"
        # a budget of iterations (the paper's instances of completion take a few)
        c["cap"] = _log_int(rng, 5, 30) if c["family"] == "mc" else _log_int(rng, 15, 100)
        return c
    if kind == "batch":
        hi = _log_int(rng, 128, 2048)
        return dict(kind="batch", count=_log_int(rng, 4, 128), n_lo=64, n_hi=hi,
                    prec=rng.choice(["fp64", "mixed"]) if hi < 1024 else "mixed",
                    threads=rng.choice([256, 384]))
    return dict(kind="gnn", step=rng.choice(["forward", "train"]), n=_log_int(rng, 300, 20_000),
                deg=round(rng.uniform(3.0, 10.0), 2))


# --------------------------------------------------------------------------------------
# problem data
# --------------------------------------------------------------------------------------
def _n_of(c):
    return {"er": lambda: c["n"], "torus": lambda: c["a"] * c["b"],
            "mc": lambda: c["n1"] + c["n2"]}[c["family"]]()


def _m_of(c):
    return c["samples"] if c["family"] == "mc" else _n_of(c)


@functools.lru_cache(maxsize=4)
def _grid_edges(a, b):
    return I.torus_edges(a, b)


def _instance(c, seed):
    if c["family"] == "er":
        return I.maxcut_er(c["n"], c["deg"], seed=seed)
    if c["family"] == "torus":
        e = _grid_edges(c["a"], c["b"])
        w = np.random.default_rng(seed).choice(np.array([-1.0, 1.0]), size=len(e))
        return I.maxcut_sdp(c["a"] * c["b"], e, w)
    return I.matrix_completion(c["n1"], c["n2"], 5, c["samples"], seed=seed)


def _prec(c):
    return L.LORADS_PREC_MIXED if c["prec"] == "mixed" else L.LORADS_PREC_FP64


def _dtype(c):
    return torch.float32 if c["prec"] == "mixed" else torch.float64


def _ld(r):
    return (r + 3) // 4 * 4


def _batch_sizes(c):
    """(n, average degree) of every graph of a batch."""
    rng = np.random.default_rng(c["count"])
    return [(int(rng.integers(c["n_lo"], c["n_hi"] + 1)), float(rng.uniform(3.0, 12.0)))
            for _ in range(c["count"])]


def _r0(m):
    return max(1, math.ceil(math.log2(m)))


def _fill(parts, size):
    """The parts one after the other in a buffer of at least `size` values, zeros after them (the
    final rank, and with it the size of a factor, depends on the instance)."""
    out = np.zeros(max(size, sum(p.size for p in parts)))
    k = 0
    for p in parts:
        out[k:k + p.size] = p.ravel()
        k += p.size
    return out


RHO, GAMMA = 37.0, 1.5


def _op_inputs(c, seed):
    """Factors and weights of an operator call (padding columns zero)."""
    n, m, r = _n_of(c), _m_of(c), c["r"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for _ in range(2):
        x = torch.zeros((n, _ld(r)), dtype=_dtype(c), device="cuda")
        x[:, :r] = torch.randn((n, r), generator=g, device="cuda", dtype=_dtype(c)) / math.sqrt(r)
        out.append(x)
    out.append(torch.randn(m, generator=g, device="cuda", dtype=torch.float64))
    return out


class _Net:
    """A network handle that is destroyed with its last reference."""

    def __init__(self, seed):
        self.handle = L.lorads_gnn_create(seed)

    def __del__(self):
        try:
            L.lorads_gnn_destroy(self.handle)
        except Exception:
            pass


def _graph(c, seed):
    """Edges with the off-diagonal entries of a MaxCut objective as weights, and targets of the
    kind a solve gives (Gram entries of unit rows, a negative dual)."""
    inst = I.maxcut_er(c["n"], c["deg"], seed=seed)
    off = inst.C_row != inst.C_col
    rng = np.random.default_rng(seed + 1)
    ei, ej, w = inst.C_row[off], inst.C_col[off], inst.C_val[off]
    Xs = np.clip(-0.6 + 0.35 * rng.standard_normal(len(ei)), -1.0, 1.0)
    ys = -1.0 - 0.5 * rng.random(c["n"])
    return ei, ej, w, Xs, ys


def _gnn_rank(c):
    return min(RMAX, max(1, math.ceil(math.log2(c["n"]))))


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "op":
        V, P, w = _op_inputs(c, seed)
        prob = L.Problem(_instance(c, seed))
        n, m = prob.n, prob.m
        out = (torch.empty(m, dtype=torch.float64, device="cuda") if c["op"] == "sddmm"
               else torch.empty((n, _ld(c["r"])), dtype=_dtype(c), device="cuda"))
        return dict(case=c, prob=prob, V=V, P=P, w=w, out=out,
                    stream=torch.cuda.current_stream())
    if c["kind"] == "solve":
        prob = L.Problem(_instance(c, seed))
        prm = prob.params(precision=_prec(c), max_admm_iter=c["cap"],
                          subsolver=(L.LORADS_SUB_ROW_DIRECT if c["sub"] == "row_direct"
                                     else L.LORADS_SUB_CG))
        return dict(case=c, prob=prob, prm=prm)
    if c["kind"] == "batch":
        probs = [L.Problem(I.maxcut_er(n, d, seed=seed + i)) for i, (n, d) in enumerate(_batch_sizes(c))]
        prm = probs[0].params(precision=_prec(c), threads=c["threads"], team_mult=1)
        return dict(case=c, probs=probs, prm=prm)
    net = _Net(seed % 1000 + 1)
    ei, ej, w, Xs, ys = _graph(c, seed)
    L.lorads_gnn_load_graph(net.handle, c["n"], ei, ej, w, seed)
    return dict(case=c, net=net, Xs=Xs, ys=ys, r=_gnn_rank(c))


# --------------------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------------------
def run(state):
    c = state["case"]
    if c["kind"] == "op":
        h, prec, r, ld = state["prob"].handle, _prec(c), c["r"], _ld(c["r"])
        V, P, w, out, s = state["V"], state["P"], state["w"], state["out"], state["stream"]
        if c["op"] == "hessian":
            rc = L.lorads_op_hessian(h, prec, r, ld, RHO, GAMMA, V, P, out, s)
        elif c["op"] == "spmm":
            rc = L.lorads_op_spmm(h, prec, r, ld, w, GAMMA, V, out, s)
        else:
            rc = L.lorads_op_sddmm(h, prec, r, ld, V, P, out, s)
        if rc != L.LORADS_OK:
            raise L.LoradsError(rc, c["op"])
        return out
    if c["kind"] == "solve":
        res = state["prob"].solve(state["prm"])
        sol = state["prob"].solution()
        return dict(objective=res["objective"], dual_objective=res["dual_objective"],
                    rank=sol["rank"], y=sol["y"],
                    U_hat=_fill([sol["U_hat"]], 4 * _r0(_m_of(c)) * _n_of(c)))
    if c["kind"] == "batch":
        res, _, _ = L.lorads_solve_batch([p.handle for p in state["probs"]], state["prm"])
        sols = [p.solution() for p in state["probs"]]
        return dict(objective=np.array([x["objective"] for x in res]),
                    rank=np.array([x["rank"] for x in sols]),
                    U_hat=_fill([x["U_hat"] for x in sols],
                                sum(4 * n * _r0(n) for n, _ in _batch_sizes(c))),
                    y=np.concatenate([x["y"] for x in sols]))
    h = state["net"].handle
    if c["step"] == "forward":
        U, y = L.lorads_gnn_forward(h, c["n"], state["r"])
        return dict(U=U, y=y)
    loss, grads = L.lorads_gnn_train_step(h, state["r"], state["Xs"], state["ys"], 1e-3,
                                          want_grads=True)
    return dict(loss=loss, grads=grads, params=L.lorads_gnn_get_params(h))


# --------------------------------------------------------------------------------------
# compulsory work
# --------------------------------------------------------------------------------------
def _nnz_c(c):
    """Entries of C, both triangles (MaxCut: the edges and the diagonal)."""
    n = _n_of(c)
    if c["family"] == "er":
        return 2 * int(n * c["deg"] / 2) + n
    return 5 * n if c["family"] == "torus" else n


def _nnz_a(c):
    return 2 * c["samples"] if c["family"] == "mc" else _n_of(c)


def work(case):
    c = dict(case)
    if c["kind"] == "op":
        n, m, r, s = _n_of(c), _m_of(c), c["r"], 4 if c["prec"] == "mixed" else 8
        if c["op"] == "hessian":      # P, V read, the product written, the entries of A once
            return dict(bytes=3 * n * r * s + (m if c["family"] == "mc" else n) * (8 + s),
                        flops=6 * _nnz_a(c) * r + 2 * n * r)
        if c["op"] == "spmm":         # V read, the product written, C, A and w once
            return dict(bytes=2 * n * r * s + (_nnz_c(c) + n) // 2 * (8 + s) + m * (8 + s) + 8 * m,
                        flops=2 * (_nnz_c(c) + _nnz_a(c)) * r + 2 * n * r)
        return dict(bytes=2 * n * r * s + m * (8 + s) + 8 * m,
                    flops=(4 if c["family"] == "mc" else 2) * m * r)
    if c["kind"] == "solve":
        # the problem read once and the solution written once; the iterations in between
        # depend on the instance
        n, m = _n_of(c), _m_of(c)
        r = math.ceil(math.log2(m))
        return dict(bytes=(_nnz_c(c) + n) // 2 * 16 + m * 28 + 8 * n * r + 8 * m,
                    flops=6 * _nnz_a(c) * r + 2 * _nnz_c(c) * r)
    if c["kind"] == "batch":
        n = c["count"] * (c["n_lo"] + c["n_hi"]) / 2
        r = math.ceil(math.log2((c["n_lo"] + c["n_hi"]) / 2))
        return dict(bytes=n * (4.75 * 16 + 28 + 8 * r + 8), flops=n * r * (6 + 2 * 8.5))
    # the layers' products and aggregations; forward reads the graph and the parameters and
    # writes U and y, a training step also reads the targets and writes gradients and parameters
    n, e = c["n"], int(c["n"] * c["deg"] / 2)
    par = NLAYER * (CATW * HID + HID) + HID * RMAX + HID + 1
    flops = n * (NLAYER * 2 * CATW * HID + 2 * HID * (RMAX + 1)) + NLAYER * 4 * e * HID
    if c["step"] == "forward":
        return dict(bytes=e * 16 + 4 * par + n * (8 * _gnn_rank(c) + 8), flops=flops)
    return dict(bytes=e * 24 + 8 * n + 16 * par, flops=3 * flops)


# --------------------------------------------------------------------------------------
# results in 64 bits
# --------------------------------------------------------------------------------------
def _scatter(n, rows, cols, vals, X):
    """sum over entries: out[rows] += vals X[cols], in pieces that fit the device."""
    out = torch.zeros((n, X.shape[1]), dtype=torch.float64, device=X.device)
    for k in range(0, len(rows), 1 << 21):
        s = slice(k, k + (1 << 21))
        out.index_add_(0, rows[s], vals[s, None] * X[cols[s]])
    return out


def _exact_op(c, seed):
    V, P, w = (x.double() for x in _op_inputs(c, seed))
    inst = _instance(c, seed)
    n = inst.n

    def dev(a, dt):
        return torch.as_tensor(np.asarray(a), device="cuda").to(dt)

    ar, ac, av = dev(inst.A_row, torch.int64), dev(inst.A_col, torch.int64), dev(inst.A_val, torch.float64)
    off = ar != ac

    def products(X, Y):      # a (X_r . Y_c + X_c . Y_r), or a X_r . Y_r on the diagonal
        q = torch.empty(len(ar), dtype=torch.float64, device="cuda")
        for k in range(0, len(ar), 1 << 21):
            s = slice(k, k + (1 << 21))
            q[s] = (X[ar[s]] * Y[ac[s]]).sum(1) + torch.where(
                off[s], (X[ac[s]] * Y[ar[s]]).sum(1), torch.zeros((), dtype=torch.float64, device="cuda"))
        return av * q

    def adjoint(wt, X):      # A^T(wt) X
        v = av * wt
        return _scatter(n, ar, ac, v, X) + _scatter(n, ac[off], ar[off], v[off], X)

    if c["op"] == "sddmm":
        return products(V, P)
    if c["op"] == "hessian":
        return RHO * adjoint(products(P, V), V) + GAMMA * P
    cr, cc, cv = dev(inst.C_row, torch.int64), dev(inst.C_col, torch.int64), dev(inst.C_val, torch.float64)
    o = cr != cc
    CV = _scatter(n, cr, cc, cv, V) + _scatter(n, cc[o], cr[o], cv[o], V)
    return adjoint(w, V) - CV + GAMMA * V


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _splitmix(key, i):
    """Output i of the SplitMix64 stream of `key`."""
    return _mix(np.uint64(key) + (i.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15))


def _normals(key, count):
    i = np.arange(count, dtype=np.uint64)
    u1 = ((_splitmix(key, 2 * i) >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
    u2 = ((_splitmix(key, 2 * i + np.uint64(1)) >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
    return np.sqrt(-2.0 * np.log(u1)) * np.cos(2.0 * np.pi * u2)


def _key(seed, stream):
    with np.errstate(over="ignore"):
        return _splitmix(seed, np.array([stream]))[0]


def _exact_gnn(c, seed):
    n, r = c["n"], _gnn_rank(c)
    ei, ej, w, Xs, ys = _graph(c, seed)
    f64 = dict(dtype=torch.float64)
    with np.errstate(over="ignore"):
        X0 = np.zeros((n, HID))
        X0[:, :8] = _normals(_key(seed, 1000), n * 8).reshape(n, 8)
        net = seed % 1000 + 1
        th = [_normals(_key(net, 2000 + l), CATW * HID).reshape(CATW, HID) / math.sqrt(CATW)
              for l in range(NLAYER)]
        thu = _normals(_key(net, 2100), HID * RMAX).reshape(HID, RMAX) / math.sqrt(HID)
        thy = _normals(_key(net, 2101), HID) / math.sqrt(HID)
    d = 1.0 + np.bincount(ei, np.abs(w), n) + np.bincount(ej, np.abs(w), n)
    X0[:, 8] = 1.0
    X0[:, 9] = np.log1p(np.bincount(ei, minlength=n) + np.bincount(ej, minlength=n))
    X0[:, 10] = d / 10.0
    X0[:, 11] = (np.bincount(ei, w, n) + np.bincount(ej, w, n)) / d
    a = torch.as_tensor(w / np.sqrt(d[ei] * d[ej]), **f64)
    i, j = torch.as_tensor(ei, dtype=torch.int64), torch.as_tensor(ej, dtype=torch.int64)
    par = []
    for l in range(NLAYER):
        par += [torch.tensor(th[l], **f64), torch.zeros(HID, **f64)]
    par += [torch.tensor(thu, **f64), torch.tensor(thy, **f64), torch.zeros(1, **f64)]
    for p in par:
        p.requires_grad_(True)
    H = torch.as_tensor(X0, **f64)
    for l in range(NLAYER):
        AH = torch.zeros((n, HID), **f64).index_add(0, i, a[:, None] * H[j]).index_add(0, j, a[:, None] * H[i])
        H = torch.relu(torch.cat([H, AH], 1) @ par[2 * l] + par[2 * l + 1])
    Z = (H @ par[-3])[:, :r]
    U = Z / Z.norm(dim=1, keepdim=True)
    y = H @ par[-2] + par[-1]
    if c["step"] == "forward":
        return dict(U=U.detach().numpy(), y=y.detach().numpy())
    loss = (((U[i] * U[j]).sum(1) - torch.as_tensor(Xs)) ** 2).mean() + BETA * ((y - torch.as_tensor(ys)) ** 2).mean()
    loss.backward()
    flat = torch.cat([p.grad.reshape(-1) for p in par])
    old = torch.cat([p.detach().reshape(-1) for p in par])
    # Adam's first step from zero moments
    new = old - 1e-3 * flat / (flat.abs() + 1e-8)
    return dict(loss=float(loss.detach()), grads=flat.numpy(), params=new.numpy())


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "op":
        out = _exact_op(c, seed)
        if c["op"] == "sddmm":
            return out
        pad = torch.zeros((out.shape[0], _ld(c["r"])), dtype=torch.float64, device=out.device)
        pad[:, :out.shape[1]] = out
        return pad
    if c["kind"] == "gnn":
        return _exact_gnn(c, seed)
    # a solve's iterates have no value of their own short of running the method
    return None
