"""The builder's four-blocks-per-warp kernels at their edges, against the test-side restatements:
resolutions around multiples of 8 and of four blocks (eight-byte loads and stores, or single
ones), occupancy that starts at an unaligned byte, any non-zero byte as occupied, full, empty
and mixed blocks; and an update of one listed block out of a slot of four."""
import numpy as np
import pytest
import torch

import _layout
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


def _occ(rng, L, R):
    occ = (rng.random((L, R, R, R)) < 0.3).astype(np.uint8)
    k = min(R, 20)
    occ[:, :k, :, : R // 2] = 0
    occ[:, R - k:, R // 3:, :] = 1
    return occ


def _map(occ):
    """The restated region map; a node cut off by the grid's edge counts as full (one region)
    when every block it has inside the grid is, as the builder's node state has it."""
    L, R = occ.shape[:2]
    m = _layout.region_map(occ)
    for l in range(L):
        for x in range(0, R, 128):
            for y in range(0, R, 128):
                for z in range(0, R, 128):
                    n = occ[l, x:x + 128, y:y + 128, z:z + 128]
                    if n.all() and all(v % 8 == 0 for v in n.shape):
                        m[l, x // 2:x // 2 + 64, y // 2:y // 2 + 64, z // 2:z // 2 + 64] = (7 << 8) | 0xFF
    return m


def _check(H, g, occ):
    v = oracle.build_vdb(occ)
    sup, sub = _layout.vdb_refinement(v)
    np.testing.assert_array_equal(g.array(H.ARRAY_LEAVES), np.asarray(v["leaves"]).reshape(-1))
    np.testing.assert_array_equal(g.array(H.ARRAY_CHILD_MASK), np.asarray(v["child"]).reshape(-1))
    np.testing.assert_array_equal(g.array(H.ARRAY_TILE_MASK), np.asarray(v["tile"]).reshape(-1))
    np.testing.assert_array_equal(g.array(H.ARRAY_NODE_SUPER), sup.reshape(-1))
    np.testing.assert_array_equal(g.array(H.ARRAY_LEAF_SUB), sub.reshape(-1))
    np.testing.assert_array_equal(g.array(H.ARRAY_REGION_MAP), _map(occ).reshape(-1))


@pytest.mark.parametrize("R", [1, 7, 8, 9, 24, 32, 33, 40, 136])
@pytest.mark.parametrize("shift", [0, 1, 4])
def test_build_and_single_block_update(H, R, shift):
    rng = np.random.default_rng(100 * R + shift)
    L = 2 if R < 100 else 1
    occ = _occ(rng, L, R)
    boxes = np.array([[-1, -1, -1, 1, 1, 1], [-2, -2, -2, 2, 2, 2]], np.float32)[:L]
    raw = torch.zeros(occ.size + shift, dtype=torch.uint8, device="cuda")
    dense = raw[shift:].view(L, R, R, R)
    values = occ * rng.integers(1, 256, occ.shape, dtype=np.uint8)  # any non-zero byte is occupied
    dense.copy_(torch.from_numpy(values))
    g = H.build_vdb(dense, boxes)
    _check(H, g, occ)
    # one voxel of one block; then the block emptied (its state changes)
    B = (R + 7) // 8
    x, y, z = (int(v) for v in rng.integers(0, R, 3))
    blk = torch.tensor([((L - 1) * B + x // 8) * B * B + (y // 8) * B + z // 8], device="cuda")
    occ[L - 1, x, y, z] ^= 1
    dense.copy_(torch.from_numpy(occ))
    g.update(dense, blk)
    _check(H, g, occ)
    b = [slice(8 * (v // 8), 8 * (v // 8) + 8) for v in (x, y, z)]
    occ[L - 1, b[0], b[1], b[2]] = 0
    dense.copy_(torch.from_numpy(occ))
    g.update(dense, blk)
    _check(H, g, occ)
