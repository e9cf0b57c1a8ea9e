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
