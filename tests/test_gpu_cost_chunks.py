"""The cost matrix with boxes in several chunks, where the warps of a tile leave
a chunk at very different times: the pairs of a tile's first warp are all
blocked by the first chunk, those of the others only by a later one."""
import numpy as np
import pytest

import oracle
from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso

pytestmark = pytest.mark.gpu

CHUNK = 256


@pytest.mark.parametrize("n,chunks,last", [(96, 2, 1), (96, 5, 256), (161, 4, 37)])
def test_late_chunks_block_what_the_first_warp_no_longer_tests(n, chunks, last):
    rng = np.random.default_rng(n * 10 + chunks)
    xyz = rng.uniform(0, 20, size=(n, 3))
    xyz[:, 2] = rng.uniform(0, 1, size=n)
    # specks among the points: no tile drops them and hardly a segment meets one
    at = rng.uniform([8, 8, 0.4], [12, 12, 0.6], size=((chunks - 1) * CHUNK + last, 3))
    boxes = np.concatenate([at - 1e-4, at + 1e-4], axis=1)
    spots = [boxes[k * CHUNK:(k + 1) * CHUNK] for k in range(chunks)]

    def block(chunk, residue):  # a box around every eighth point blocks all its pairs
        pts = xyz[residue::8]
        k = min(len(pts), len(spots[chunk]))
        spots[chunk][-k:] = np.concatenate([pts[:k] - 0.01, pts[:k] + 0.01], axis=1)

    block(0, 0)  # (a warp of a tile has every eighth row)
    for chunk in range(1, chunks):
        block(chunk, 2 * chunk - 1)
    C = torch.empty((n, n), dtype=torch.int32, device=DEV)
    px, bx = torch.from_numpy(xyz).to(DEV), torch.from_numpy(np.ascontiguousarray(boxes)).to(DEV)
    ref, _ = oracle.cost_matrix(xyz, np.ascontiguousarray(boxes))
    for _ in range(50):
        C.zero_()
        dpso.dpso_cost_matrix(px, n, bx, len(boxes), dpso.default_cost_params(), C)
        assert np.array_equal(C.cpu().numpy(), ref)
