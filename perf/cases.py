"""The workloads whose time is watched, each through the package's public calls.

A case is one step of a program that keeps an analysed pattern (a `Solver`) and solves it again and
again on new values: K shifted factorisations, R right-hand sides, the combination, and for the
training cases the gradients.  The systems are those of the paper and of `bench.py`:

* grids: distributed-slack power-flow Jacobians of random bus graphs (mean degree 2.7, 20 % PV buses)
  at a random operating point, one grid or a batch of uneven grids.  The pattern belongs to the case,
  the operating point, the right-hand sides and the gradients to the seed, as in a Newton loop or a
  contingency study, where the topology stays and the values change;
* dense: Gaussian matrices with a strong diagonal, the dense batch of the paper's own measurement.

`via` says how the program calls the library: "eager" (factor, then solve), "graph" (a step captured
once, replayed), "autograd" (forward and backward of the differentiable solve), "host" (buffers in
pinned host memory, copies inside the call).
"""
import math
import random

import numpy as np
import torch

import paper_2311_11833_gb300 as pisp

DEV = "cuda:0"
# the options the autotuner picks for a batch of a few hundred grids (bench.py's default workload)
BATCH_OPTIONS = dict(relax_small=16, relax_zeros=0.10, factor_policy=4, factor_ctas_per_sm=3, factor_smem_maxF=128,
                     solve_ctas_per_sm=4, solve_kfuse=1, solve_warp_maxF=64)


def _case(name, system, via, G, lo, hi, K, R, precision, sweeps=0, tol=0.0, one_sided=False, tuned=False):
    """`lo`..`hi`: buses of a grid (or unknowns of a dense system), log-uniform over the G instances;
    `sweeps` FP64 residual sweeps, a maximum where `tol` > 0 (each instance then stops on its own)."""
    return dict(name=name, system=system, via=via, G=G, lo=lo, hi=hi, K=K, R=R, precision=precision, sweeps=sweeps,
                tol=tol, one_sided=one_sided, tuned=tuned)


def listed():
    return [
        # one Newton step of the smallest grid in use: launches and latency are everything
        _case("newton_118", "grid", "eager", 1, 118, 118, 2, 1, "fp64"),
        # the paper's 300-bus system, replayed on new operating points
        _case("plain_300", "grid", "graph", 1, 300, 300, 4, 1, "fp64"),
        # a Newton step of a mid-size grid with 32-bit factors and a fixed number of sweeps
        _case("newton_1354_fp32", "grid", "eager", 1, 1354, 1354, 4, 1, "fp32", sweeps=3),
        # an odd one: one-sided shifts, a few right-hand sides, sweeps until converged
        _case("ragged_777", "grid", "eager", 1, 777, 777, 3, 5, "fp32", sweeps=8, tol=1e-12, one_sided=True),
        # the 2000-bus study: many shifts and right-hand sides on one grid
        _case("precision_2000", "grid", "graph", 1, 2000, 2000, 6, 16, "fp32", sweeps=8, tol=1e-12),
        # the largest grid: a wide dense root, the most right-hand sides of a replayed step
        _case("scale_10000", "grid", "graph", 1, 10000, 10000, 8, 32, "fp32", sweeps=8, tol=1e-12),
        # the benchmark's batch of uneven grids, with the options the autotuner picks for it
        _case("batch_256", "grid", "graph", 256, 118, 3000, 4, 8, "fp32", sweeps=8, tol=1e-12, tuned=True),
        # a batch of scenarios in 64-bit factors with default options
        _case("batch_48_fp64", "grid", "eager", 48, 118, 2000, 4, 3, "fp64"),
        # the end-to-end call: inputs and results in host memory
        _case("host_64", "grid", "host", 64, 118, 3000, 4, 8, "fp32", sweeps=8, tol=1e-12),
        # training: forward and backward through the solve, a minibatch of right-hand sides
        _case("train_1354", "grid", "autograd", 1, 1354, 1354, 4, 64, "fp64"),
        # training over a few grids with 32-bit factors and swept gradients
        _case("train_5_fp32", "grid", "autograd", 5, 300, 900, 4, 8, "fp32", sweeps=4),
        # the paper's dense batched systems
        _case("dense_12", "dense", "graph", 12, 64, 531, 10, 1, "fp32", sweeps=8, tol=1e-12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more program of the same kinds, sizes spread over their whole ranges."""
    kind = rng.choice(["one", "one", "large", "batch", "batch", "host", "train", "dense"])
    fp32 = rng.random() < 0.6
    prec = dict(precision="fp32", sweeps=8, tol=1e-12) if fp32 else dict(precision="fp64")
    one_sided = rng.random() < 0.25
    K = rng.choice([1, 2, 3, 4, 5]) if one_sided else rng.choice([2, 4, 6, 8])
    if kind == "one":
        n = _log(rng, 118, 3000)
        c = _case("", "grid", rng.choice(["eager", "graph"]), 1, n, n, K, _log(rng, 1, 16), **prec)
    elif kind == "large":
        n = _log(rng, 3000, 9000)
        c = _case("", "grid", rng.choice(["eager", "graph"]), 1, n, n, min(K, 6), _log(rng, 1, 24), "fp32", sweeps=8, tol=1e-12)
    elif kind == "batch":
        c = _case("", "grid", rng.choice(["eager", "graph"]), _log(rng, 4, 128), 118, _log(rng, 600, 3000), min(K, 4),
                  _log(rng, 1, 8), tuned=rng.random() < 0.5, **prec)
    elif kind == "host":
        c = _case("", "grid", "host", _log(rng, 1, 64), 118, _log(rng, 300, 3000), min(K, 4), _log(rng, 1, 8), **prec)
    elif kind == "train":
        prec = dict(precision="fp32", sweeps=4) if fp32 else prec
        c = _case("", "grid", "autograd", _log(rng, 1, 8), 118, _log(rng, 200, 1400), min(K, 4), _log(rng, 1, 64), **prec)
    else:
        c = _case("", "dense", rng.choice(["eager", "graph"]), _log(rng, 1, 16), 8, _log(rng, 32, 400), K, _log(rng, 1, 4), **prec)
    c["one_sided"] = one_sided
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs --
def _sizes(case):
    """Instance sizes (buses or unknowns), log-uniform over [lo, hi] and shuffled."""
    G = case["G"]
    q = (np.arange(G) + 0.5) / G if G > 1 else np.ones(1)
    s = np.rint(np.exp(math.log(case["lo"]) + q * (math.log(case["hi"]) - math.log(case["lo"])))).astype(np.int64)
    return np.random.default_rng(G).permutation(s)


def _grid(N, top, val):
    """CSR (row_ptr, col, val) of one power-flow Jacobian: bus graph from the generator `top`, operating
    point from `val`.  Unknowns [angles of all buses but the slack; magnitudes of the PQ buses; lambda],
    equations [P of all but the slack; Q of the PQ buses; P of the slack]."""
    relabel = top.permutation(N)
    parent = (top.random(N - 1) * np.arange(1, N)).astype(np.int64)  # a random recursive tree
    e = np.stack([relabel[np.arange(1, N)], relabel[parent]], 1)
    extra = top.integers(0, N, size=(N, 2))
    extra = extra[extra[:, 0] != extra[:, 1]]
    keys = np.concatenate([np.minimum(x[:, 0], x[:, 1]) * N + np.maximum(x[:, 0], x[:, 1]) for x in (e, extra)])
    _, first = np.unique(keys, return_index=True)
    keys = keys[np.sort(first)[:int(round(1.35 * N))]]  # the tree's edges come first
    a, b = keys // N, keys % N
    y = 1.0 / (top.uniform(0.005, 0.05, len(a)) + 1j * top.uniform(0.02, 0.3, len(a)))
    pv = 1 + top.permutation(N - 1)[:int(round(0.2 * N))]
    part = np.zeros(N)
    part[np.concatenate([[0], pv])] = top.uniform(0.5, 1.5, len(pv) + 1)
    part /= part.sum()
    V, th = val.uniform(0.95, 1.05, N), val.normal(0.0, 0.1, N)
    th[0] = 0.0
    diag = np.zeros(N, complex)
    np.add.at(diag, a, y)
    np.add.at(diag, b, y)
    i, j, yij = np.concatenate([a, b]), np.concatenate([b, a]), -np.concatenate([y, y])
    volt = V * np.exp(1j * th)
    cur = diag * volt
    np.add.at(cur, i, yij * volt[j])
    S = volt * np.conj(cur)
    pq = np.setdiff1d(np.arange(1, N), pv)
    n = N + len(pq)
    ang, mag = np.full(N, -1), np.full(N, -1)
    ang[1:] = np.arange(N - 1)
    mag[pq] = N - 1 + np.arange(len(pq))
    prow, qrow = ang.copy(), mag
    prow[0] = n - 1
    d = th[i] - th[j]
    t1 = yij.real * np.sin(d) - yij.imag * np.cos(d)
    t2 = yij.real * np.cos(d) + yij.imag * np.sin(d)
    rows = np.concatenate([prow, prow, qrow, qrow, prow[i], prow[i], qrow[i], qrow[i], prow[part != 0]])
    cols = np.concatenate([ang, mag, ang, mag, ang[j], mag[j], ang[j], mag[j], np.full((part != 0).sum(), n - 1)])
    v = np.concatenate([-S.imag - diag.imag * V ** 2, S.real / V + diag.real * V, S.real - diag.real * V ** 2,
                        S.imag / V - diag.imag * V, V[i] * V[j] * t1, V[i] * t2, -V[i] * V[j] * t2, V[i] * t1,
                        -part[part != 0]])
    keep = (rows >= 0) & (cols >= 0)
    rows, cols, v = rows[keep], cols[keep], v[keep]
    o = np.argsort(rows * n + cols)
    ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))])
    return ptr.astype(np.int64), cols[o].astype(np.int32), v[o]


def _system(case, seed):
    """(sizes, row_ptr, col, values, D, t, b, g) on the host; the instances on the block diagonal."""
    ns, ptrs, cols, vals, off = [], [np.zeros(1, np.int64)], [], [], 0
    for q, m in enumerate(_sizes(case)):
        top, val = np.random.default_rng([int(m), q]), np.random.default_rng([seed, q])
        if case["system"] == "grid":
            ptr, col, v = _grid(int(m), top, val)
        else:
            A = val.standard_normal((m, m))
            A[np.arange(m), np.arange(m)] += 2.0 * math.sqrt(m) * np.sign(val.standard_normal(m))
            ptr, col, v = np.arange(m + 1) * m, np.tile(np.arange(m), m), A.reshape(-1)
        n = len(ptr) - 1
        ns.append(n)
        ptrs.append(ptr[1:] + ptrs[-1][-1])
        cols.append(col + off)
        vals.append(v)
        off += n
    ptr, col, v = np.concatenate(ptrs), np.concatenate(cols).astype(np.int32), np.concatenate(vals)
    row = np.repeat(np.arange(off), np.diff(ptr))
    D = np.zeros(off)  # the perturbation: |A_ii|
    D[row[row == col]] = np.abs(v[row == col])
    K = case["K"]
    t = 1e-2 * np.arange(1, K + 1) if case["one_sided"] else 1e-2 * np.repeat(np.arange(1, K // 2 + 1), 2) * np.tile([1, -1], K // 2)
    rng = np.random.default_rng([seed, 1 << 20])
    b, g = rng.standard_normal((off, case["R"])), rng.standard_normal((off, case["R"]))
    return ns, ptr, col, v, D, t, b, g


# --------------------------------------------------------------- the program --
def prepare(case, seed):
    ns, ptr, col, v, D, t, b, g = _system(case, seed)
    s = pisp.Solver(ns, ptr, col, **(BATCH_OPTIONS if case["tuned"] else {}))
    if case["tol"] > 0:
        s.set_refinement(case["tol"])
    st = dict(via=case["via"], s=s, t=t, precision=case["precision"], sweeps=case["sweeps"])
    if case["via"] == "host":
        pin = lambda x: torch.from_numpy(x).pin_memory()  # noqa: E731
        st["pinned"] = [pin(x) for x in (v, D, b, np.zeros_like(b))]
        st["values"], st["D"], st["b"], st["x"] = (x.numpy() for x in st["pinned"])
        return st
    st["values"], st["D"], st["b"] = (torch.from_numpy(x).to(DEV) for x in (v, D, b))
    if case["via"] == "autograd":
        st["values"].requires_grad_(True)
        st["b"].requires_grad_(True)
        st["g"] = torch.from_numpy(g).to(DEV)
    if case["via"] == "graph":
        st["x"] = torch.empty_like(st["b"])
        s.graph_capture(st["values"], st["D"], t, st["b"], st["x"], precision=case["precision"], sweeps=case["sweeps"])
    return st


def run(st):
    s = st["s"]
    if st["via"] == "graph":
        s.graph_launch()
        return st["x"]
    if st["via"] == "host":
        return s.solve_host(st["values"], st["D"], st["t"], st["b"], precision=st["precision"], sweeps=st["sweeps"],
                            out=st["x"])
    if st["via"] == "autograd":
        x = pisp.solve(s, st["values"], st["b"], st["D"], st["t"], precision=st["precision"], sweeps=st["sweeps"])
        gv, gb = torch.autograd.grad(x, (st["values"], st["b"]), st["g"])
        return x.detach(), gv, gb
    s.factor(st["values"], st["D"], st["t"], precision=st["precision"])
    return s.solve(st["b"], sweeps=st["sweeps"])


def work(case):
    """Inputs and outputs once; the operations of the K factorisations and of one forward and one backward
    solve.  A grid's factors end in a dense block of about 0.16 unknowns a bus, the rest stays sparse."""
    by = fl = 0.0
    for m in _sizes(case):
        m = float(m)
        if case["system"] == "grid":
            n, nnz, fac, lu = 1.8 * m, 12.4 * m, (0.16 * m) ** 3 * 2 / 3 + 400 * m, (0.16 * m) ** 2 + 24 * m
        else:
            n, nnz, fac, lu = m, m * m, m ** 3 * 2 / 3, m * m
        train = 2 if case["via"] == "autograd" else 1
        by += train * (12 * nnz + 8 * n + 16 * n * case["R"])
        fl += case["K"] * (fac + train * 2 * lu * case["R"])
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------- in 64 bits --
def _solve64(A, B):
    """A^{-1} B in 64 bits: LU in 32 bits with residual corrections in 64, plain 64-bit LU where those stall."""
    lu = torch.linalg.lu_factor(A.float())
    x = torch.linalg.lu_solve(*lu, B.float()).double()
    last = math.inf
    for _ in range(25):
        d = torch.linalg.lu_solve(*lu, (B - A @ x).float()).double()
        x += d
        size = float(d.abs().max() / x.abs().max())
        if size < 1e-15 or (size < 1e-13 and size > last / 2):
            return x
        if not size < last / 1.5:
            break
        last = size
    return torch.linalg.solve(A, B)


def exact(case, seed):
    ns, ptr, col, v, D, t, b, g = _system(case, seed)
    w = [math.prod(l / (l - k) for l in t if l != k) for k in t]
    xs, gv, gb, off = [], [], [], 0
    for n in ns:
        e0, e1 = int(ptr[off]), int(ptr[off + n])
        j = torch.from_numpy(col[e0:e1].astype(np.int64) - off).to(DEV)
        i = torch.from_numpy(np.repeat(np.arange(n), np.diff(ptr[off:off + n + 1]))).to(DEV)
        A = torch.zeros(n, n, dtype=torch.float64, device=DEV)
        A[i, j] = torch.from_numpy(v[e0:e1]).to(DEV)
        d, B, C = (torch.from_numpy(x[off:off + n]).to(DEV) for x in (D, b, g))
        at = torch.arange(n, device=DEV)
        x, xb, xv = torch.zeros_like(B), torch.zeros_like(B), torch.zeros(e1 - e0, dtype=torch.float64, device=DEV)
        for tk, wk in zip(t, w):
            Ak = A.clone()
            Ak[at, at] += tk * d
            xk = _solve64(Ak, B)
            x += wk * xk
            if case["via"] == "autograd":
                lam = _solve64(Ak.T.contiguous(), C)
                xb += wk * lam
                xv -= wk * (lam[i] * xk[j]).sum(1)
        xs.append(x)
        gb.append(xb)
        gv.append(xv)
        off += n
    if case["via"] == "autograd":
        return torch.cat(xs), torch.cat(gv), torch.cat(gb)
    return torch.cat(xs)
