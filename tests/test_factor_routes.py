"""Which kernels a factorisation runs, by its number of launches, and that every way
gives the same solution: one dense system of `n` unknowns (a front of n rows, owner
tiles of (n + 1) x 32 values) beside `ones` systems of one unknown (a front each)."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import pfgen
from _parity import entrywise_err

pytestmark = pytest.mark.gpu
TOL = 1e-10
K = 16


def _dev(a):
    import torch
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


# owner tiles leave room for three CTAs an SM up to 512 rows, for two up to 832; one
# launch while there are fewer than 24 x 8192 pairs with two, 4 x 8192 with one
@pytest.mark.parametrize("n,ones,single", [(500, 2200, True), (700, 2200, True), (900, 2200, False), (900, 2000, True),
                                           (700, 12300, False), (500, 12300, True), (1030, 1, False)])
def test_one_launch_or_level_by_level(n, ones, single):
    import paper_2311_11833_gb300 as pisp
    I = pfgen.random_sparse(n, 1.0, seed=n, diag_boost=2.0 * np.sqrt(n))
    r = np.random.default_rng(ones)
    a, d = r.uniform(1.0, 2.0, ones), r.uniform(0.5, 1.5, ones)
    sizes = [n] + [1] * ones
    rp = np.concatenate([I.row_ptr, I.row_ptr[-1] + 1 + np.arange(ones)])
    col = np.concatenate([I.col, n + np.arange(ones)]).astype(np.int32)
    t = pfgen.symmetric_shifts(K, 1e-3)
    b = pfgen.rhs(n + ones, 2, 1)
    for policy in (0, 4):
        s = pisp.Solver(sizes, rp, col, factor_policy=policy)
        assert s.stats()["n_supernodes"] == 1 + ones
        s.factor(_dev(np.concatenate([I.val, a])), _dev(np.concatenate([I.D, d])), t, "fp32")
        assert (s.stats()["gpu_launches"] == 1) == (single or policy == 4)
        x = s.solve(_dev(b), sweeps=4).cpu().numpy()
        assert s.status()[0] == 0
        s.close()
        scale = float(sum(abs(w) for w in oracle.weights(t)))
        assert entrywise_err(x[:n], oracle.x_hat(oracle.to_scipy(I), I.D, t, b[:n])) <= TOL * scale
        want = sum(w * b[n:] / (a + tk * d)[:, None] for w, tk in zip(oracle.weights(t), t))
        assert (abs(x[n:] - want) <= TOL * scale * abs(want).max()).all()


def _unit(precision):
    return 2.0 ** -24 if precision == "fp32" else 2.0 ** -53


# sizes of test_factor_shapes, which the default routing factors in one launch with FP32
# factors, and the widest fronts of a CTA level by level (224 rows, FP64: 160)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("policy", [2, 3])
def test_dense_fronts_level_by_level(precision, policy):
    import test_factor_shapes as shapes
    ns = shapes.DENSE + (162, 191, 223, 224, 225)
    insts = [pfgen.random_sparse(n, 1.0, seed=n, diag_boost=2.0 * np.sqrt(n)) for n in ns]
    s, t, _ = shapes._factor(insts, 2, precision, factor_policy=policy)
    assert s.stats()["gpu_launches"] > 1
    perm, first = s.perm(), s.supernodes()[0].tolist()
    r0 = 0
    for I in insts:
        p = perm[r0:r0 + I.n] - r0
        A = oracle.to_scipy(I).toarray()
        for k in range(2):
            f = s.front(first.index(r0), k).astype(np.float64)
            L, U = np.tril(f, -1) + np.eye(I.n), np.triu(f)
            B = (A + t[k] * np.diag(I.D))[np.ix_(p, p)]
            # the bound of test_factor_shapes: any order of summation
            assert (abs(L @ U - B) <= (I.n + 6) * _unit(precision) * (abs(L) @ abs(U) + abs(B))).all(), (I.n, k)
        r0 += I.n
    s.close()


@pytest.mark.parametrize("precision,sweeps", [("fp32", 4), ("fp64", 0)])
def test_many_children_level_by_level(precision, sweeps):
    import test_factor_shapes as shapes
    shapes.test_many_children(precision, sweeps, 2)


def _hub(hub, arms, seed):
    """A dense hub and dense blocks tied to all of it: a front of (block + hub) rows each."""
    r = np.random.default_rng(seed)
    n = hub + sum(arms)
    M = np.zeros((n, n))
    M[:hub, :] = r.standard_normal((hub, n))
    M[:, :hub] = r.standard_normal((n, hub))
    at = hub
    for a in arms:
        M[at:at + a, at:at + a] = r.standard_normal((a, a))
        at += a
    M[np.arange(n), np.arange(n)] = 2.0 * np.sqrt(n) + abs(M[np.arange(n), np.arange(n)])
    return sp.csr_matrix(M), r.uniform(0.5, 1.5, n)


HUBS = [(120, (31, 65)), (250, (6, 40)), (480, (32, 64)), (1010, (33, 95))]


@pytest.mark.parametrize("precision,sweeps,policy,hub,arms", [("fp64", 0, p, *h) for p in (0, 4) for h in HUBS] +
                         [("fp32", 5, 0, *HUBS[-1])])
def test_owner_tiles_by_themselves(precision, sweeps, policy, hub, arms):
    """Owner tiles of FP64 factors, level by level and in one launch, and of FP32 factors
    in launches of their own (fronts of more than 1024 rows)."""
    import paper_2311_11833_gb300 as pisp
    A, D = _hub(hub, arms, hub)
    n = A.shape[0]
    t = pfgen.symmetric_shifts(2, 1e-3)
    s = pisp.Solver([n], A.indptr.astype(np.int64), A.indices.astype(np.int32), factor_policy=policy)
    s.profile(True)
    s.factor(_dev(A.data), _dev(D), t, precision)
    s.profile_collect()
    s.profile(False)
    ran = {f for f, v in s.profile_read().items() if v["launches"]}
    assert ("factor_persistent" in ran) == (policy == 4)
    # level by level owner tiles take the fronts that a CTA's shared memory does not hold
    assert policy == 4 or ("factor_big" in ran) == (s.stats()["max_front"] > (224 if precision == "fp32" else 160))
    b = pfgen.rhs(n, 2, 1)
    x = s.solve(_dev(b), sweeps=sweeps).cpu().numpy()
    assert s.status()[0] == 0
    s.close()
    assert entrywise_err(x, oracle.x_hat(A, D, t, b)) <= TOL * float(sum(abs(w) for w in oracle.weights(t)))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("sizes,persistent", [((40, 40, 7), False), ((160, 33), False), ((200, 40), True)])
def test_fronts_that_wait_for_no_others(precision, sizes, persistent):
    """Dense systems: level by level while a CTA holds each front, whatever their number."""
    import test_factor_shapes as shapes
    G = 1000 if max(sizes) <= 40 else 1
    insts = [pfgen.random_sparse(n, 1.0, seed=n, diag_boost=2.0 * np.sqrt(n)) for n in sizes] * G
    s, t, dev = shapes._factor(insts, 4, precision)
    s.profile(True)
    s.factor(dev(np.concatenate([I.val for I in insts])), dev(np.concatenate([I.D for I in insts])), t, precision)
    s.profile_collect()
    s.profile(False)
    assert bool(s.profile_read()["factor_persistent"]["launches"]) == (persistent and precision == "fp32")
    b = pfgen.rhs(sum(I.n for I in insts), 2, 1)
    x = s.solve(dev(b), sweeps=4 if precision == "fp32" else 0).cpu().numpy()
    assert s.status()[0] == 0
    s.close()
    r0 = 0
    scale = float(sum(abs(w) for w in oracle.weights(t)))
    for I in insts[:len(sizes)]:
        assert entrywise_err(x[r0:r0 + I.n], oracle.x_hat(oracle.to_scipy(I), I.D, t, b[r0:r0 + I.n])) <= TOL * scale
        r0 += I.n
