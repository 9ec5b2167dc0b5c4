"""Sizes that no kernel takes are refused when the mesh is described, before
anything is allocated (so this needs no GPU)."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

CASES = {  # lattice, FEM block: planes of 2^30 padded nodes, blocks of 2^31 nodes
    "telegraph_plane": ((7, 140_000_000, 7), (2, 2, 2), (4, 4, 4)),
    "telegraph_block": ((1400, 1400, 1400), (2, 2, 2), (1397, 1397, 1397)),
    "refined_plane": ((40_000, 30_000, 9), (2, 2, 2), (5, 5, 5)),
}


def description(n, lo, hi, precision):
    hyb = pytest.importorskip("paper_1509_01399_gb300.hyb")
    d = hyb.hyb_mesh_desc()
    for a in range(3):
        d.n[a], d.fem_lo[a], d.fem_hi[a] = n[a], lo[a], hi[a]
    d.h, d.a_max, d.precision = 0.1, 1.0, precision
    return hyb, d


def refused(hyb, d, message):
    # (on a thread of its own: the message of the last failure is kept per thread)
    with ThreadPoolExecutor(1) as ex, pytest.raises(hyb.HybError, match=message):
        ex.submit(hyb.hyb_mesh_create, d, 0).result()


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp32_beyond_the_tile_kernel(name):
    hyb, d = description(*CASES[name], 1)
    mask = np.ones(1, np.uint8)
    if name.startswith("telegraph"):
        d.model = hyb.HYB_MODEL_TELEGRAPH
    else:
        d.refine_mask = mask.ctypes.data
    refused(hyb, d, "too large for FP32")


def test_refined_blocks_of_2_31_voxels():
    hyb, d = description((1400, 1400, 1400), (4, 4, 4), (1395, 1395, 1395), 0)
    mask = np.ones(1, np.uint8)
    d.refine_mask = mask.ctypes.data
    refused(hyb, d, "fewer than 2\\^31")
