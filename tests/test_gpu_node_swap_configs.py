"""The node-swap kernel against the oracle at the edges of its launch
configurations (by tour length and tours per SM) and on ties."""
import numpy as np
import pytest

import oracle
from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso, inputs

pytestmark = pytest.mark.gpu


def _check(C_np, tours, max_moves):
    n = C_np.shape[0]
    T = torch.from_numpy(tours.view(np.int16).copy()).to(DEV)
    cost = torch.empty(len(tours), dtype=torch.int64, device=DEV)
    pairs, moves = dpso.dpso_node_swap(torch.from_numpy(C_np).to(DEV), n, T, len(tours), cost,
                                       max_moves)
    got_t, got_c = T.cpu().numpy().view(np.uint16), cost.cpu().numpy()
    tot_p = tot_m = 0
    for k, x in enumerate(tours):
        y, f, mv, pr = oracle.node_swap(C_np, x, max_moves)
        assert np.array_equal(got_t[k], y) and got_c[k] == f, (n, k)
        tot_p += pr
        tot_m += mv
    assert (pairs, moves) == (tot_p, tot_m)


@pytest.mark.parametrize("n,count,moves", [
    (6, 9, 0), (64, 3, 0), (65, 320, 3), (100, 3, 0), (101, 3, 0), (160, 310, 3), (161, 3, 0),
    (220, 3, 30), (221, 800, 2), (600, 770, 1), (601, 3, 8), (1500, 2, 3), (1501, 2, 3),
    (4497, 1, 1)])
def test_launch_configurations(n, count, moves):
    C_np = inputs.random_cost_matrix(n, 17 * n, hi=1_000_000)
    _check(C_np, inputs.random_tours(n, count, 3 * n), moves)


@pytest.mark.parametrize("n,hi", [(5, 2), (33, 1), (120, 2), (260, 3)])
def test_ties(n, hi):
    # costs from {1..hi}: most positions tie, so stale and exact values meet
    _check(inputs.random_cost_matrix(n, n + hi, hi=hi), inputs.random_tours(n, 4, n), 0)
