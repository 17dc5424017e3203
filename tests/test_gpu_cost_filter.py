"""The cost matrix's FP32 filter against the oracle's FP64 slab test where the
two could part: boxes that touch or nearly touch, axes on which a pair hardly
differs, magnitudes far from 1, more boxes than one chunk, tile edges."""
import numpy as np
import pytest

import oracle
from gpu_helpers import DEV, torch
from paper_1706_04399_gb300 import dpso

pytestmark = pytest.mark.gpu


def _check(xyz, boxes, radius=0.0):
    n, m = len(xyz), len(boxes)
    C = torch.empty((n, n), dtype=torch.int32, device=DEV)
    cp = dpso.default_cost_params(uav_radius_m=radius)
    dpso.dpso_cost_matrix(torch.from_numpy(np.ascontiguousarray(xyz)).to(DEV), n,
                          torch.from_numpy(np.ascontiguousarray(boxes)).to(DEV) if m else None,
                          m, cp, C)
    ref, _ = oracle.cost_matrix(np.ascontiguousarray(xyz), np.ascontiguousarray(boxes),
                                radius=radius)
    assert np.array_equal(C.cpu().numpy(), ref)


def _boxes(rng, m, extent, side):
    c = rng.uniform(0, extent, size=(m, 3))
    h = rng.uniform(0, side, size=(m, 3))
    return np.concatenate([c - h, c + h], axis=1)


@pytest.mark.parametrize("n,m", [(1, 0), (2, 1), (31, 3), (32, 32), (33, 33), (64, 0), (65, 257),
                                 (200, 600), (257, 20)])
def test_tile_and_chunk_edges(n, m):
    rng = np.random.default_rng(n * 1000 + m)
    _check(rng.uniform(0, 20, size=(n, 3)), _boxes(rng, m, 20.0, 1.5), radius=0.25)


@pytest.mark.parametrize("step", [1.0, 0.1, 1.0 / 3.0])
def test_lattice_points_on_box_faces(step):
    # points and box faces share one lattice: segments lie in faces, end on
    # edges and pass through corners
    rng = np.random.default_rng(5)
    xyz = rng.integers(0, 6, size=(150, 3)) * step
    lo = rng.integers(0, 5, size=(25, 3))
    boxes = np.concatenate([lo * step, (lo + rng.integers(0, 3, size=(25, 3))) * step], axis=1)
    _check(xyz, boxes)
    _check(xyz, boxes, radius=step)


@pytest.mark.parametrize("jitter", [0.0, 1e-300, 1e-15, 1e-9, 1e-6, 1e-4, 1e-3])
def test_nearly_planar_points(jitter):
    rng = np.random.default_rng(9)
    xyz = rng.uniform(0, 30, size=(160, 3))
    xyz[:, 1] = 3.0 + jitter * rng.integers(-2, 3, size=160)
    boxes = _boxes(rng, 20, 30.0, 3.0)
    boxes[:8, 1], boxes[:8, 4] = 3.0, 5.0            # faces in the plane
    boxes[8:12, 1], boxes[8:12, 4] = 3.0 + jitter, 5.0
    boxes[12:14, 1] = boxes[12:14, 4] = 3.0 - jitter  # flat boxes
    _check(xyz, boxes)


@pytest.mark.parametrize("scale,offset", [(1e-3, 0.0), (1e-40, 0.0), (1.0, 1e5), (0.01, 4e5),
                                          (1e4, -1e5)])
def test_magnitudes(scale, offset):
    rng = np.random.default_rng(11)
    _check(rng.uniform(0, 20, size=(120, 3)) * scale + offset,
           _boxes(rng, 30, 20.0, 2.0) * scale + offset)


@pytest.mark.parametrize("unit", [0.0005, 0.001, 0.0015, 0.25, 1.0 / 1024])
def test_lengths_at_rounding_ties(unit):
    # lattices whose lengths in mm fall on or next to half-integers
    rng = np.random.default_rng(21)
    xyz = rng.integers(0, 4000, size=(180, 3)) * unit
    xyz[:60, 1:] = 0.0
    _check(xyz, np.zeros((0, 6)))
    xyz[60:90] += rng.integers(-3, 4, size=(30, 3)) * 2.0 ** -40
    _check(xyz, np.zeros((0, 6)))
