"""Solves at the limits of their launches: what a task may use of shared memory,
schedules rebuilt under work in flight, waits that run out, and calls that fail."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import pfgen
from _parity import entrywise_err, grad_entrywise_err
from test_abi import HostSymbolic

TOL = 1e-10  # the repository's entry-wise bound (FP64 factors, or FP32 with FP64 sweeps)
HUB = 32
ARMS = (2, 3, 5, 8, 9, 17, 32)


def _thin(p):
    """Two dense blocks of p unknowns, each tied to all of a dense hub of 32 but one:
    two fronts of p pivots and p + 31 rows under a root of 32 pivots."""
    r = np.random.default_rng(p)
    n = 2 * p + HUB
    M = np.zeros((n, n))
    M[2 * p:, 2 * p:] = r.standard_normal((HUB, HUB))
    for a in range(2):
        at = np.arange(a * p, a * p + p)
        hub = 2 * p + np.delete(np.arange(HUB), a)
        M[np.ix_(at, at)] = r.standard_normal((p, p))
        M[np.ix_(at, hub)] = r.standard_normal((p, HUB - 1))
        M[np.ix_(hub, at)] = r.standard_normal((HUB - 1, p))
    d = np.arange(n)
    M[d, d] = 2.0 * np.sqrt(n) + abs(M[d, d])
    A = sp.csr_matrix(M)
    return pfgen.Instance(n=n, row_ptr=A.indptr.astype(np.int64), col=A.indices.astype(np.int32), val=A.data,
                          D=r.uniform(0.5, 1.5, n), meta={})


def _concat(insts):
    rp, cols, off = [0], [], 0
    for I in insts:
        rp.extend((I.row_ptr[1:] + rp[-1]).tolist())
        cols.append(I.col + off)
        off += I.n
    return ([I.n for I in insts], np.array(rp, np.int64), np.concatenate(cols).astype(np.int32),
            np.concatenate([I.val for I in insts]), np.concatenate([I.D for I in insts]))


def _dev(a):
    import torch
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def test_thin_fronts_and_no_wider_pivot_blocks():
    """The systems of the next test are what it says: fronts of more than 32 rows,
    none with more than 32 pivots."""
    import paper_2311_11833_gb300._lib as L
    insts = [_thin(p) for p in ARMS]
    sizes, rp, col, _, _ = _concat(insts)
    hs = HostSymbolic(L.load(), sizes, rp, col, ordering=1, relax_small=1, relax_zeros=0.0)
    assert hs.rc == 0
    ns = hs.c1 - hs.c0
    assert ns.max() == HUB and set(ns[ns + hs.ms > 32]) == set(ARMS)
    hs.close()


@pytest.mark.gpu
@pytest.mark.parametrize("precision,sweeps", [("fp64", 0), ("fp32", 4)])
@pytest.mark.parametrize("K", [1, 4])
def test_thin_fronts_one_right_hand_side(precision, sweeps, K):
    """Fronts of more than 32 rows solved by a CTA while no front has more than 32
    pivots, whose tasks would ask for far more shared memory: the backward solve of
    one right-hand side once asked for less than its partial sums take."""
    import paper_2311_11833_gb300 as pisp
    insts = [_thin(p) for p in ARMS]
    sizes, rp, col, val, D = _concat(insts)
    t = pfgen.one_sided_shifts(K, 1e-3) if K % 2 else pfgen.symmetric_shifts(K, 1e-3)
    N = sum(sizes)
    b, g = pfgen.rhs(N, 1, 5), pfgen.rhs(N, 1, 6)
    s = pisp.Solver(sizes, rp, col, ordering=1, relax_small=1, relax_zeros=0.0)
    s.factor(_dev(val), _dev(D), t, precision)
    x = s.solve(_dev(b), sweeps=sweeps).cpu().numpy()
    gb, gv = (v.cpu().numpy() for v in s.adjoint(_dev(g), sweeps=sweeps))
    assert s.status()[0] == 0
    s.close()
    scale = float(sum(abs(w) for w in oracle.weights(t)))
    r0 = e0 = 0
    for I in insts:
        rows, ent = slice(r0, r0 + I.n), slice(e0, e0 + I.nnz)
        A = oracle.to_scipy(I)
        assert entrywise_err(x[rows], oracle.x_hat(A, I.D, t, b[rows])) <= TOL * scale, I.n
        rb, rv = oracle.adjoint(A, I.D, t, b[rows], g[rows])
        assert entrywise_err(gb[rows], rb) <= TOL * scale, I.n
        assert grad_entrywise_err(gv[ent], rv) <= TOL * scale, I.n
        r0 += I.n
        e0 += I.nnz


@pytest.mark.gpu
@pytest.mark.parametrize("precision,sweeps", [("fp64", 0), ("fp32", 4)])
@pytest.mark.parametrize("K", [12, 13, 16])
def test_two_right_hand_sides_many_shifts(precision, sweeps, K):
    """Two right-hand sides put up to 16 shifts into a group of 32 columns, each with
    coefficients of its own in shared memory: with FP64 factors 13 shifts and more
    were once refused."""
    import test_solve_shapes as shapes
    shapes.test_solve_and_adjoint_shapes(precision, sweeps, K, 2, {})


@pytest.mark.gpu
def test_schedules_rebuilt_under_work_in_flight():
    """Other numbers of right-hand sides and of shifts rebuild the task lists while
    solves and factorisations that read the old ones wait behind a long kernel on a
    stream that the legacy stream does not wait for."""
    import torch
    import paper_2311_11833_gb300 as pisp
    insts = [pfgen.grid_jacobian(n, None, n) for n in (60, 140, 200)]
    sizes, rp, col, val, D = _concat(insts)
    N = sum(sizes)
    s = pisp.Solver(sizes, rp, col)
    vals_d, D_d = _dev(val), _dev(D)
    steps = [(K, R) for K in (4, 2) for R in (12, 1, 5, 2)] + [(4, 3)]
    rhs = [_dev(pfgen.rhs(N, R, R)) for _, R in steps]
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    got, want = [], []
    with torch.cuda.stream(st):
        for out, busy in ((want, False), (got, True)):
            for (K, R), b in zip(steps, rhs):
                if busy:
                    torch.cuda._sleep(20_000_000)  # about 10 ms
                s.factor(vals_d, D_d, pfgen.symmetric_shifts(K), "fp64")
                out.append(s.solve(b))
                if not busy:
                    st.synchronize()
    st.synchronize()
    assert s.status()[0] == 0
    s.close()
    r0 = 0
    for I in insts:
        rows = slice(r0, r0 + I.n)
        A = oracle.to_scipy(I)
        for (K, R), b, x, w in zip(steps, rhs, got, want):
            assert torch.equal(x, w), (K, R)
            t = pfgen.symmetric_shifts(K)
            assert entrywise_err(x[rows].cpu().numpy(), oracle.x_hat(A, I.D, t, b[rows].cpu().numpy())) <= TOL, (K, R)
        r0 += I.n


@pytest.mark.gpu
def test_default_wait_limit_is_a_few_tenths_of_a_second():
    """2^22 polls 64 ns apart are 0.27 s of sleep, however far apart the polls of a
    long wait really are (1 us: 4.3 s); a task that gives up lets the next ones on."""
    import time
    import torch
    import paper_2311_11833_gb300 as pisp
    inst = pfgen.make_instance("plain")
    s = pisp.Solver(inst.n, inst.row_ptr, inst.col)
    s.factor(_dev(inst.val), _dev(inst.D), pfgen.symmetric_shifts(2), "fp64")
    b = _dev(pfgen.rhs(inst.n, 2, 3))
    s.solve(b)
    s.set_wait_limit(0, True)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    s.solve(b)
    torch.cuda.synchronize()
    waited = time.perf_counter() - t0
    assert s.status()[0] == 6  # PISP_ERR_TIMEOUT
    s.close()
    assert 0.05 < waited < 2.5


@pytest.mark.gpu
def test_solve_that_cannot_be_set_up_leaves_nothing_to_differentiate():
    """A solve whose workspace does not fit the card (front vectors of 2^21 right-hand
    sides and 16 shifts) has given up the workspace of the solve before it: combining
    or differentiating that one is refused, and the next solve is correct."""
    import torch
    import paper_2311_11833_gb300 as pisp
    from paper_2311_11833_gb300._lib import PispError
    inst = pfgen.make_instance("plain")
    t = pfgen.symmetric_shifts(16, 1e-3)
    b, g = pfgen.rhs(inst.n, 3, 5), pfgen.rhs(inst.n, 3, 6)
    s = pisp.Solver(inst.n, inst.row_ptr, inst.col)
    c0, c1, ms = s.supernodes()[:3]
    R = 1 << 21
    assert 16 * R * 8 * int((c1 - c0 + ms).sum()) > torch.cuda.get_device_properties(0).total_memory
    s.factor(_dev(inst.val), _dev(inst.D), t, "fp64")
    s.solve(_dev(b))
    wide = torch.zeros((inst.n, R), dtype=torch.float64, device="cuda")
    with pytest.raises(PispError, match="OOM"):
        s.solve(wide)
    del wide
    torch.cuda.empty_cache()
    with pytest.raises(PispError, match="NOT_FACTORED"):
        s.adjoint(_dev(g))
    with pytest.raises(PispError, match="NOT_FACTORED"):
        s.combine()
    x = s.solve(_dev(b)).cpu().numpy()
    gb = s.adjoint(_dev(g))[0].cpu().numpy()
    assert s.status()[0] == 0
    s.close()
    A = oracle.to_scipy(inst)
    scale = float(sum(abs(w) for w in oracle.weights(t)))
    assert entrywise_err(x, oracle.x_hat(A, inst.D, t, b)) <= TOL * scale
    assert entrywise_err(gb, oracle.adjoint(A, inst.D, t, b, g)[0]) <= TOL * scale


@pytest.mark.gpu
@pytest.mark.parametrize("precision,sweeps", [("fp64", 0), ("fp32", 4)])
@pytest.mark.parametrize("K,R,opts", [
    (1, 2, {}), (4, 2, dict(solve_kfuse=3)), (3, 3, dict(solve_schedule=1)), (2, 4, dict(solve_warp_maxF=64)),
    (2, 5, dict(solve_warp_maxF=64, solve_ctas_per_sm=4)), (4, 8, {}), (2, 9, {}), (16, 7, {}), (16, 12, {})])
def test_pivots_to_right_hand_sides(precision, sweeps, K, R, opts):
    """Fronts of 9 to 32 pivots around the numbers of right-hand sides where their
    backward solve changes from segments to columns (3 R pivots), alone and under other
    fronts, and fronts with more pivots at 1, 2 and 4 right-hand sides a task (FP64)."""
    import paper_2311_11833_gb300 as pisp
    dense = [pfgen.random_sparse(n, 1.0, seed=n, diag_boost=2.0 * np.sqrt(n))
             for n in (6, 9, 10, 12, 13, 15, 16, 17, 24, 25, 27, 28, 32, 65, 257, 300)]
    insts = dense + [_thin(p) for p in (2, 9, 12, 17, 32)] + [pfgen.grid_jacobian(140, None, 9)]
    sizes, rp, col, val, D = _concat(insts)
    t = pfgen.one_sided_shifts(K, 1e-3) if K % 2 else pfgen.symmetric_shifts(K, 1e-3)
    N = sum(sizes)
    b, g = pfgen.rhs(N, R, 5), pfgen.rhs(N, R, 6)
    s = pisp.Solver(sizes, rp, col, ordering=1, relax_small=1, relax_zeros=0.0, **opts)
    s.factor(_dev(val), _dev(D), t, precision)
    x = s.solve(_dev(b), sweeps=sweeps).cpu().numpy()
    again = s.solve(_dev(b), sweeps=sweeps).cpu().numpy()
    gb, gv = (v.cpu().numpy() for v in s.adjoint(_dev(g), sweeps=sweeps))
    assert s.status()[0] == 0
    s.close()
    assert (x == again).all()
    scale = float(sum(abs(w) for w in oracle.weights(t)))
    r0 = e0 = 0
    for I in insts:
        rows, ent = slice(r0, r0 + I.n), slice(e0, e0 + I.nnz)
        A = oracle.to_scipy(I)
        assert entrywise_err(x[rows], oracle.x_hat(A, I.D, t, b[rows])) <= TOL * scale, I.n
        rb, rv = oracle.adjoint(A, I.D, t, b[rows], g[rows])
        assert entrywise_err(gb[rows], rb) <= TOL * scale, I.n
        assert grad_entrywise_err(gv[ent], rv) <= TOL * scale, I.n
        r0 += I.n
        e0 += I.nnz
