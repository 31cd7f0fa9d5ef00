"""The factorisation at the sizes where its task kinds change: fronts around 8, 16,
32, 64 and 96 rows and around a panel of 16 pivots, a parent with more children
than a warp has lanes, both precisions, level by level and in one launch.

Dense systems are one front each: its factors must reproduce the matrix within the
componentwise bound of an n-step elimination in any order of summation,
|L U - A| <= (n + 6) u (|L| |U| + |A|), u the unit roundoff (one rounding each more
for the entry, the perturbation, the reciprocal and the scaling).  Trees are
checked through the solution, entry by entry, at the repository's 1e-10."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import pfgen
from _parity import entrywise_err

pytestmark = pytest.mark.gpu

DENSE = (1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 47, 49, 63, 64, 65, 96, 97, 112, 113, 160, 161)


def _concat(insts):
    rp, cols, off = [0], [], 0
    for I in insts:
        rp.extend((I.row_ptr[1:] + rp[-1]).tolist())
        cols.append(I.col + off)
        off += I.n
    return ([I.n for I in insts], np.array(rp, np.int64), np.concatenate(cols).astype(np.int32),
            np.concatenate([I.val for I in insts]), np.concatenate([I.D for I in insts]))


def _factor(insts, K, precision, **opts):
    import torch
    import paper_2311_11833_gb300 as pisp
    sizes, rp, col, val, D = _concat(insts)
    t = pfgen.symmetric_shifts(K, 1e-3)
    s = pisp.Solver(sizes, rp, col, **opts)
    dev = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    s.factor(dev(val), dev(D), t, precision)
    assert s.status()[0] == 0
    return s, t, dev


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("opts", [{}, dict(factor_policy=4), dict(factor_policy=4, factor_ctas_per_sm=3)])
def test_dense_fronts(precision, opts):
    K = 2
    insts = [pfgen.random_sparse(n, 1.0, seed=n, diag_boost=2.0 * np.sqrt(n)) for n in DENSE]
    s, t, _ = _factor(insts, K, precision, **opts)
    perm, first = s.perm(), s.supernodes()[0].tolist()
    u = 2.0 ** -24 if precision == "fp32" else 2.0 ** -53
    r0 = 0
    for I in insts:
        p = perm[r0:r0 + I.n] - r0
        A = oracle.to_scipy(I).toarray()
        i = first.index(r0)
        for k in range(K):
            f = s.front(i, k).astype(np.float64)
            assert f.shape == (I.n, I.n)
            L, U = np.tril(f, -1) + np.eye(I.n), np.triu(f)
            B = (A + t[k] * np.diag(I.D))[np.ix_(p, p)]
            bound = (I.n + 6) * u * (abs(L) @ abs(U) + abs(B))
            assert (abs(L @ U - B) <= bound).all(), (I.n, k)
        r0 += I.n
    s.close()


def _star(hub, arms, seed):
    """A dense hub and `arms` separate unknowns, each tied to a few of the hub's."""
    r = np.random.default_rng(seed)
    n = hub + arms
    M = np.zeros((n, n))
    M[:hub, :hub] = r.standard_normal((hub, hub))
    for a in range(arms):
        at = r.choice(hub, size=int(r.integers(1, min(hub, 6) + 1)), replace=False)
        M[hub + a, at] = r.standard_normal(len(at))
        M[at, hub + a] = r.standard_normal(len(at))
    M[np.arange(n), np.arange(n)] = 3.0 + abs(M).sum(1)
    A = sp.csr_matrix(M)
    return A, r.uniform(0.5, 1.5, n)


@pytest.mark.parametrize("precision,sweeps", [("fp32", 4), ("fp64", 0)])
@pytest.mark.parametrize("policy", [0, 4])
def test_many_children(precision, sweeps, policy):
    import torch
    import paper_2311_11833_gb300 as pisp
    for hub, arms in ((6, 40), (14, 70), (30, 33), (40, 100), (100, 150)):
        A, D = _star(hub, arms, hub)
        t = pfgen.symmetric_shifts(2, 1e-3)
        n = A.shape[0]
        s = pisp.Solver([n], A.indptr.astype(np.int64), A.indices.astype(np.int32), factor_policy=policy,
                        relax_small=1, relax_zeros=0.0)
        dev = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
        s.factor(dev(A.data), dev(D), t, precision)
        b = pfgen.rhs(n, 3, 1)
        x = s.solve(dev(b), sweeps=sweeps).cpu().numpy()
        assert s.status()[0] == 0
        s.close()
        scale = float(sum(abs(w) for w in oracle.weights(t)))
        assert entrywise_err(x, oracle.x_hat(A, D, t, b)) <= 1e-10 * scale, (hub, arms)


@pytest.mark.parametrize("policy", [0, 3, 4])
@pytest.mark.parametrize("hub,arms", [(230, (27, 33, 70)), (250, (6, 40)), (480, (32, 64)), (530, (1, 95))])
def test_owner_tiles(hub, arms, policy):
    """Wide fronts around a chunk of 256 rows and a block of 32 columns: a dense hub
    and dense blocks tied to all of it, a front of (block + hub) rows each."""
    import torch
    import paper_2311_11833_gb300 as pisp
    r = np.random.default_rng(hub)
    n = hub + sum(arms)
    M = np.zeros((n, n))
    M[:hub, :] = r.standard_normal((hub, n))
    M[:, :hub] = r.standard_normal((n, hub))
    at = hub
    for a in arms:
        M[at:at + a, at:at + a] = r.standard_normal((a, a))
        at += a
    M[np.arange(n), np.arange(n)] = 2.0 * np.sqrt(n) + abs(M[np.arange(n), np.arange(n)])
    A, D = sp.csr_matrix(M), r.uniform(0.5, 1.5, n)
    t = pfgen.symmetric_shifts(2, 1e-3)
    s = pisp.Solver([n], A.indptr.astype(np.int64), A.indices.astype(np.int32), factor_policy=policy)
    dev = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    s.factor(dev(A.data), dev(D), t, "fp32")
    assert s.stats()["max_front"] >= hub + 1
    b = pfgen.rhs(n, 2, 1)
    x = s.solve(dev(b), sweeps=5).cpu().numpy()
    assert s.status()[0] == 0
    s.close()
    assert entrywise_err(x, oracle.x_hat(A, D, t, b)) <= 1e-10 * float(sum(abs(w) for w in oracle.weights(t)))
