"""More pairs of one delta than the 2-opt's list holds, for every launch
configuration of it: passes that take the best move directly, by position."""
import numpy as np
import pytest

from paper_1706_04399_gb300 import inputs
from test_gpu_two_opt_list import _check

pytestmark = pytest.mark.gpu

# (viewpoints, tours): matrix in shared memory, C read in place (with and
# without few tours), warps' rows with 128 and 64 threads, the block's rows
CONFIGS = [(100, 3), (150, 4), (215, 3), (300, 4), (300, 320), (300, 630), (640, 2), (640, 160),
           (1300, 2)]


def _some(count):
    return None if count < 10 else (0, 1, count // 2, count - 1)


@pytest.mark.parametrize("n,count", CONFIGS)
def test_costs_one_and_two(n, count):
    _check(inputs.random_cost_matrix(n, n, hi=2), inputs.random_tours(n, count, n + 1),
           max_moves=0 if n < 1000 else 150, sample=_some(count))


@pytest.mark.parametrize("n,count", CONFIGS)
def test_half_of_the_pairs_blocked(n, count):
    a = (inputs.random_cost_matrix(n, n + 7, hi=2) - 1) * 1_000_000
    np.fill_diagonal(a, 0)
    _check(np.ascontiguousarray(a), inputs.random_tours(n, count, n + 2),
           max_moves=0 if n < 1000 else 150, sample=_some(count))


@pytest.mark.parametrize("n,count", [(150, 3), (300, 4), (640, 2)])
def test_lattice_costs(n, count):
    # squared distances on a lattice: many equal deltas, few of them smallest
    side = int(n ** 0.5) + 1
    p = np.stack(np.meshgrid(np.arange(side), np.arange(side)), -1).reshape(-1, 2)[:n]
    c = 500 * ((p[:, None] - p[None]) ** 2).sum(-1)
    _check(np.ascontiguousarray(c.astype(np.int32)), inputs.random_tours(n, count, n + 3))


def test_capped_calls_end_inside_a_direct_stretch():
    for cap in (1, 2, 7, 33):
        _check(inputs.random_cost_matrix(260, 5, hi=2), inputs.random_tours(260, 3, 6),
               max_moves=cap)
