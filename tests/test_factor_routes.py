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
