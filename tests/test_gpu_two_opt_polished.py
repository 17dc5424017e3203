"""The default 2-opt on tours that are 2-optimal already or nearly so, where
every row has to be known, and the allocation-free call at the lengths where its
neighbour lists move from its array to a scratch slot and where they fit
neither."""
import numpy as np
import pytest

from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso, inputs
from test_gpu_two_opt_list import _check

pytestmark = pytest.mark.gpu


def _polished(C, n, count):
    T = torch.from_numpy(inputs.random_tours(n, count, n).view(np.int16).copy()).to(DEV)
    cost = torch.empty(count, dtype=torch.int64, device=DEV)
    dpso.dpso_two_opt(C, n, T, count, cost, 0)
    return T.cpu().numpy().view(np.uint16).copy()


@pytest.mark.parametrize("n,count", [(60, 4), (150, 4), (300, 4), (300, 320), (300, 620), (700, 3),
                                     (700, 160), (1300, 2)])
def test_polished_tours_stay_and_near_ones_return(n, count):
    C_np = inputs.random_cost_matrix(n, 7 * n, hi=100_000)
    tours = _polished(torch.from_numpy(C_np).to(DEV), n, count)
    sample = None if count < 10 else (0, 1, count - 1)
    _check(C_np, tours, sample=sample)
    _check(C_np, tours, fn=dpso.dpso_two_opt_noalloc, sample=sample)
    near = tours.copy()
    near[:, [1, n // 2, n // 3]] = near[:, [n // 2, n // 3, 1]]
    _check(C_np, near, sample=sample)


@pytest.mark.parametrize("n,count", [(500, 2), (501, 2), (513, 2), (1100, 2), (1100, 1500),
                                     (4096, 1), (4097, 1)])
def test_noalloc_with_lists_in_a_slot_or_none(n, count):
    C_np = inputs.random_cost_matrix(n, 3 * n, hi=1_000_000)
    _check(C_np, inputs.random_tours(n, count, n), max_moves=5, fn=dpso.dpso_two_opt_noalloc,
           sample=None if count < 10 else (0, 1, count - 1))
