"""The numbering of leaves and groups and the list's offsets, beyond one tile
of 256 particles a block (from 524,289 particles) and one run of 1024 groups."""
import numpy as np
import pytest

from paper_1802_09824_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,gs", [(300, 8), (33_000, 32), (524_288, 32), (600_001, 8)])
def test_groups_leaves_and_offsets(gpu_lib, n, gs):
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=n)
    bp = ps.boxes[0]
    rcut = 0.3 * bp.rcut
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs * 0.3, rcut, 16, 0, gs)
    lv = B.ph_build_leaves(torch.from_numpy(ps.pos).cuda(), None, prm)
    pr = B.ph_leaf_pairs(lv)
    v = B.ph_leaves_get_view(lv)
    keys = v["keys"].cpu().numpy().view(np.uint64)
    cell = keys >> np.uint64(3 * (v["key_bits"] - v["g"][0]))
    first = np.flatnonzero(np.concatenate([[True], cell[1:] != cell[:-1]]))
    sizes = np.diff(np.concatenate([first, [n]]))
    groups = np.concatenate([np.arange(f, f + s, gs) for f, s in zip(first, sizes)] + [[n]])
    np.testing.assert_array_equal(v["group_first"].cpu().numpy(), groups)
    lf = v["leaf_first"].cpu().numpy()
    assert lf[0] == 0 and lf[-1] == n
    assert 1 <= np.diff(lf).min() and np.diff(lf).max() <= 16
    assert np.isin(first, lf).all()
    clf = v["cell_leaf_first"].cpu().numpy()
    starts = np.searchsorted(cell, np.arange(clf.size - 1, dtype=np.uint64))
    np.testing.assert_array_equal(clf, np.searchsorted(lf[:-1], np.concatenate([starts, [n]])))
    p = B.ph_pairs_get_view(pr)
    off = p["group_off"].cpu().numpy()
    assert off[0] == 0 and off[-1] == p["n_pairs"] and np.diff(off).min() >= 1
    for h in (pr, lv):
        B.ph_free(h)
