"""The default 2-opt kernels against the oracle where they can go wrong: the
edges of their launch configurations (by tour length and tours per SM), lists
that run full, and ties that a list cannot hold."""
import numpy as np
import pytest

import oracle
from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso, inputs

pytestmark = pytest.mark.gpu


def _check(C_np, tours, max_moves=0, fn=None, sample=None):
    n = C_np.shape[0]
    T = torch.from_numpy(tours.view(np.int16).copy()).to(DEV)
    cost = torch.empty(len(tours), dtype=torch.int64, device=DEV)
    pairs, moves = (fn or dpso.dpso_two_opt)(torch.from_numpy(C_np).to(DEV), n, T, len(tours),
                                             cost, max_moves)
    got_t, got_c = T.cpu().numpy().view(np.uint16), cost.cpu().numpy()
    tot_p = tot_m = 0
    for k in range(len(tours)) if sample is None else sample:
        y, f, mv, pr = oracle.two_opt(C_np, tours[k], max_moves)
        assert np.array_equal(got_t[k], y) and got_c[k] == f, (n, k)
        tot_p += pr
        tot_m += mv
    if sample is None:
        assert (pairs, moves) == (tot_p, tot_m)


@pytest.mark.parametrize("n,count,moves", [
    (7, 9, 0), (44, 5, 0), (46, 5, 0), (64, 5, 0), (65, 480, 4), (66, 480, 4), (66, 5, 0),
    (90, 5, 0), (91, 5, 0), (160, 4, 0), (160, 470, 6), (161, 4, 0), (220, 4, 0), (221, 160, 6),
    (221, 3, 0), (511, 3, 40), (512, 480, 2), (512, 620, 1), (513, 160, 2), (513, 2, 40),
    (1200, 160, 1), (1200, 2, 12), (1201, 2, 12), (5000, 1, 3), (5001, 1, 3)])
def test_launch_configurations(n, count, moves):
    C_np = inputs.random_cost_matrix(n, 31 * n, hi=1_000_000)
    _check(C_np, inputs.random_tours(n, count, 5 * n), moves)


@pytest.mark.parametrize("n,hi", [(40, 2), (90, 1), (150, 2), (300, 2), (300, 3), (640, 2)])
def test_ties_beyond_the_list(n, hi):
    # costs from {1..hi}: thousands of candidates share a delta, so the list
    # cannot hold a level and passes are taken directly
    _check(inputs.random_cost_matrix(n, n + hi, hi=hi), inputs.random_tours(n, 3, n))
    _check(inputs.random_cost_matrix(n, n + hi, hi=hi), inputs.random_tours(n, 3, n + 1),
           fn=dpso.dpso_two_opt_noalloc)


@pytest.mark.parametrize("n", [64, 200, 700])
def test_clusters_of_large_costs(n):
    # a large penalty on half of the pairs: deltas fall into dense clusters
    # far apart, so thresholds jump and lists run full
    base = inputs.random_cost_matrix(n, n, hi=50)
    pen = inputs.random_cost_matrix(n, n + 1, hi=2) // 2 * 1_000_000
    _check(np.ascontiguousarray(base + pen), inputs.random_tours(n, 4, n + 2))
