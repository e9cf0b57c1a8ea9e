"""The radix sort's tile sizes (512, 1024 and 2048 keys; prefixes added up by
the tiles themselves or scanned between the passes): keys in order and the
permutation stable, against numpy's stable sort of the same keys."""
import numpy as np
import pytest

from paper_1802_09824_gb300 import synth

pytestmark = pytest.mark.gpu


# one tile, its edge, several; the last size of each tile and the first of the
# next; beyond 64 tiles of 2048
@pytest.mark.parametrize("n", [2, 511, 512, 513, 32768, 32769, 65536, 65537, 131072, 131073, 200_003])
def test_sorted_order_is_stable(gpu_lib, n):
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=n)
    pos = ps.pos.copy()
    pos[n // 2:] = pos[: n - n // 2]          # equal keys: rows have to keep their order
    bp = ps.boxes[0]
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, 32)
    lv = B.ph_build_leaves(torch.from_numpy(pos).cuda(), None, prm)
    v = B.ph_leaves_get_view(lv)
    keys = v["keys"].cpu().numpy().view(np.uint64)
    perm = v["perm"].cpu().numpy()
    by_row = np.empty(n, np.uint64)
    by_row[perm] = keys
    np.testing.assert_array_equal(perm, np.argsort(by_row, kind="stable"))
    np.testing.assert_array_equal(np.sort(perm), np.arange(n))
    B.ph_free(lv)


def test_equal_digits_share_their_counters(gpu_lib):
    # particles on a coarse grid (low digits all alike) and in a few cells
    # (high digits alike), with lanes left over in the last warp
    import torch
    B = gpu_lib
    n = 140_003
    rng = np.random.default_rng(5)
    grid = (rng.integers(0, 8, (n, 3)) / 8.0 + 1.0 / 16).astype(np.float32)
    clump = (0.4 + 0.01 * rng.random((n, 3))).astype(np.float32)
    for pos in (grid, clump):
        lv = B.ph_build_leaves(torch.from_numpy(pos).cuda(), None, B.make_params(1.0, 1.0, 1e-3, 0.03, 0.1, 64))
        v = B.ph_leaves_get_view(lv)
        perm = v["perm"].cpu().numpy()
        by_row = np.empty(n, np.uint64)
        by_row[perm] = v["keys"].cpu().numpy().view(np.uint64)
        np.testing.assert_array_equal(perm, np.argsort(by_row, kind="stable"))
        B.ph_free(lv)
