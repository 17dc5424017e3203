"""A* costs of searches around the sizes at which one pass hands them to the
next: the small shared-memory map, the large one, device memory."""
import numpy as np
import pytest

import oracle
from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half,depth", [(20, 30), (27, 34), (28, 34), (30, 34), (45, 42), (48, 42),
                                        (60, 42)])
def test_floods_across_the_pass_limits(half, depth):
    # a wall with one gap at its far end: a search between the two sides
    # floods about half x depth voxels
    dims = (2 * half + 1, depth, 1)
    boxes = np.array([[half, 0.0, 0.0, half + 1.0, depth - 1.0, 1.0]])
    rng = np.random.default_rng(half)
    xyz = np.column_stack([rng.uniform(0, dims[0], 12), rng.uniform(0, depth / 3, 12),
                           np.full(12, 0.5)])
    ap = dpso.astar_params((0, 0, 0), 1.0, dims)
    occ = torch.empty(int(np.prod(dims)), dtype=torch.uint8, device=DEV)
    dpso.dpso_voxel_occupancy(torch.from_numpy(boxes).to(DEV), 1, ap, occ)
    occ_ref = oracle.voxel_occupancy((0, 0, 0), 1.0, dims, boxes, 0)
    assert np.array_equal(occ.cpu().numpy().reshape(occ_ref.shape), occ_ref)
    C = torch.empty((12, 12), dtype=torch.int32, device=DEV)
    dpso.dpso_cost_matrix_astar(torch.from_numpy(np.ascontiguousarray(xyz)).to(DEV), 12, occ, ap, C)
    want, _ = oracle.cost_matrix_astar(xyz, occ_ref, (0, 0, 0), 1.0, dims, (1, 1, 1), 500, 10 ** 8,
                                       20000)
    assert np.array_equal(C.cpu().numpy(), want)
