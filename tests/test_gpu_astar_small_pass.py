"""A* costs of more pairs than one wave of the large shared-memory maps, so that
searches begin in the small ones: floods around the sizes that hand a search
on, and ways that are too long for the small map from the start."""
import numpy as np
import pytest

import oracle
from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso

pytestmark = pytest.mark.gpu

N = 50  # 1225 pairs, seven searches on each of 152 SMs


def _check(xyz, dims, boxes):
    ap = dpso.astar_params((0, 0, 0), 1.0, dims)
    occ = torch.empty(int(np.prod(dims)), dtype=torch.uint8, device=DEV)
    bx = torch.from_numpy(boxes).to(DEV) if len(boxes) else None
    dpso.dpso_voxel_occupancy(bx, len(boxes), ap, occ)
    occ_ref = oracle.voxel_occupancy((0, 0, 0), 1.0, dims, boxes, 0)
    C = torch.empty((N, N), dtype=torch.int32, device=DEV)
    dpso.dpso_cost_matrix_astar(torch.from_numpy(np.ascontiguousarray(xyz)).to(DEV), N, occ, ap, C)
    want, _ = oracle.cost_matrix_astar(xyz, occ_ref, (0, 0, 0), 1.0, dims, (1, 1, 1), 500, 10 ** 8,
                                       20000)
    assert np.array_equal(C.cpu().numpy(), want)


@pytest.mark.parametrize("half,depth", [(20, 30), (28, 34), (30, 34), (48, 42), (60, 42)])
def test_floods_across_the_pass_limits(half, depth):
    # a wall with one gap at its far end: a search between the two sides
    # floods about half x depth voxels
    rng = np.random.default_rng(half)
    xyz = np.column_stack([rng.uniform(0, 2 * half + 1, N), rng.uniform(0, depth / 3, N),
                           np.full(N, 0.5)])
    _check(xyz, (2 * half + 1, depth, 1), np.array([[half, 0.0, 0.0, half + 1.0, depth - 1.0, 1.0]]))


@pytest.mark.parametrize("dims", [(250, 7, 7), (250, 60, 1), (200, 2, 30), (120, 120, 9)])
def test_long_free_ways(dims):
    # 9, 15 or 19 voxels come into view per step: the longest ways pass the
    # small map's room, some the large one's
    rng = np.random.default_rng(sum(dims))
    _check(rng.uniform(0, dims, size=(N, 3)), dims, np.zeros((0, 6)))
