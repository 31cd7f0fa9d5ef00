"""The solve kernels at the sizes where their task kinds change: right-hand side
counts around a chunk and around 32 columns, pivot blocks around 32 and 256 rows
(dense systems of n rows are one front of n pivots), supernodes wider than 32
pivots below the root (large amalgamation), both schedules, and the transposed
solves of the adjoint.  Against the oracle, entry by entry, at the repository's
1e-10 (FP64 factors, or FP32 with FP64 sweeps)."""
import numpy as np
import pytest

import oracle
import pfgen
from _parity import entrywise_err, grad_entrywise_err

pytestmark = pytest.mark.gpu
TOL = 1e-10


def _concat(insts):
    rp, cols, off = [0], [], 0
    for I in insts:
        rp.extend((I.row_ptr[1:] + rp[-1]).tolist())
        cols.append(I.col + off)
        off += I.n
    return ([I.n for I in insts], np.array(rp, np.int64), np.concatenate(cols).astype(np.int32),
            np.concatenate([I.val for I in insts]), np.concatenate([I.D for I in insts]))


def _systems():
    dense = [pfgen.random_sparse(n, 1.0, seed=n, diag_boost=2.0 * np.sqrt(n)) for n in (1, 31, 32, 33, 65, 255, 257, 300)]
    return dense + [pfgen.random_sparse(90, 0.05, seed=5), pfgen.grid_jacobian(140, None, 9)]


@pytest.mark.parametrize("precision,sweeps", [("fp64", 0), ("fp32", 4)])
@pytest.mark.parametrize("K,R,opts", [
    (1, 1, {}), (3, 1, dict(solve_kfuse=2)), (2, 2, {}), (3, 5, {}), (4, 8, dict(solve_warp_maxF=64)),
    (4, 9, dict(relax_small=64, relax_zeros=0.5)), (2, 33, {}), (5, 12, dict(solve_ctas_per_sm=4)),
    (16, 3, dict(solve_schedule=1)), (2, 1, dict(solve_schedule=1)), (1, 70, dict(relax_small=64, relax_zeros=0.5))])
def test_solve_and_adjoint_shapes(precision, sweeps, K, R, opts):
    import torch
    import paper_2311_11833_gb300 as pisp
    insts = _systems()
    sizes, rp, col, val, D = _concat(insts)
    t = pfgen.one_sided_shifts(K, 1e-3) if K % 2 else pfgen.symmetric_shifts(K, 1e-3)
    N = sum(sizes)
    b, g = pfgen.rhs(N, R, 5), pfgen.rhs(N, R, 6)
    dev = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    s = pisp.Solver(sizes, rp, col, **opts)
    s.factor(dev(val), dev(D), t, precision)
    x = s.solve(dev(b), sweeps=sweeps).cpu().numpy()
    gb, gv = (v.cpu().numpy() for v in s.adjoint(dev(g), sweeps=sweeps))
    assert s.status()[0] == 0
    s.close()
    r0 = e0 = 0
    for I in insts:
        rows, ent = slice(r0, r0 + I.n), slice(e0, e0 + I.nnz)
        A = oracle.to_scipy(I)
        # the weights cancel: an error of every x_k shows times their size
        scale = float(sum(abs(w) for w in oracle.weights(t)))
        assert entrywise_err(x[rows], oracle.x_hat(A, I.D, t, b[rows])) <= TOL * scale, I.n
        rb, rv = oracle.adjoint(A, I.D, t, b[rows], g[rows])
        assert entrywise_err(gb[rows], rb) <= TOL * scale, I.n
        assert grad_entrywise_err(gv[ent], rv) <= TOL * scale, I.n
        r0 += I.n
        e0 += I.nnz
