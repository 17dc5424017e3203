"""The node swap's first pass, which looks at every pair column block by column
block, against the oracle: the smallest tours, the edges of its blocks for each
launch configuration, costs at the limit, and tours that no swap improves."""
import numpy as np
import pytest

from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso, inputs
from test_gpu_node_swap_configs import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,count", [
    (3, 5), (4, 5), (5, 5), (31, 4), (32, 4), (33, 4), (63, 4), (64, 4), (127, 3), (128, 3),
    (255, 3), (257, 3), (511, 762), (512, 762), (513, 762), (767, 305), (768, 305), (769, 305),
    (1023, 2), (1024, 2), (1025, 2), (1500, 2), (1025, 160), (1500, 160), (2047, 1), (2048, 1), (2049, 1), (4497, 1)])
def test_block_edges(n, count):
    C_np = inputs.random_cost_matrix(n, 5 * n, hi=1_000_000)
    _check(C_np, inputs.random_tours(n, count, n), 1)


@pytest.mark.parametrize("n", [7, 150, 300, 1600])
def test_costs_at_the_limit(n):
    rng = np.random.default_rng(n)
    a = np.triu(rng.integers(0, 2, (n, n)) * dpso.NODE_SWAP_COST_MAX, 1)
    _check(np.ascontiguousarray((a + a.T).astype(np.int32)), inputs.random_tours(n, 2, n), 2)


@pytest.mark.parametrize("n,count", [(30, 6), (200, 4), (400, 4), (700, 2)])
def test_local_optima_stay(n, count):
    C = torch.from_numpy(inputs.random_cost_matrix(n, n, hi=1000)).to(DEV)
    T = torch.from_numpy(inputs.random_tours(n, count, 1).view(np.int16).copy()).to(DEV)
    cost = torch.empty(count, dtype=torch.int64, device=DEV)
    dpso.dpso_node_swap(C, n, T, count, cost, 0)
    _check(C.cpu().numpy(), T.cpu().numpy().view(np.uint16).copy(), 0)
