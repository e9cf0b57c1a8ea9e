"""Groups whose source lists span several segments: each segment is a task of
its own, and the group's sum (segments in order, compensated) does not depend
on which warps made it."""
import numpy as np
import pytest

from helpers import check_parity, oracle_accel
from paper_1802_09824_gb300 import synth

pytestmark = pytest.mark.gpu


def _setup(B, ps, **kw):
    import torch
    bp = ps.boxes[0]
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, kw.get("leaf", 32), 0, kw.get("gs", 0),
                        queue_order=kw.get("qo", 0))
    pos, mass = torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda()
    lv = B.ph_build_leaves(pos, mass, prm)
    pr = B.ph_leaf_pairs(lv)
    return pos, mass, lv, pr


def _lists(B, pr):
    off = B.ph_pairs_get_view(pr)["group_off"].cpu().numpy()
    return np.diff(off)


# segments of 8 entries (n up to ~12,800 at leaf 32) and of 256 (leaf 1): lists
# below, at and above one segment and many segments; every lanes-per-target
# split; then the same list summed again (the tasks' counters start over), in
# the other queue order and without a list, all bit for bit
@pytest.mark.parametrize("n,leaf,gs", [(97, 32, 32), (1000, 1, 32), (4096, 32, 32), (4096, 16, 16), (9001, 32, 8),
                                       (14000, 256, 32)])
def test_split_groups_match_the_oracle_in_any_order(gpu_lib, n, leaf, gs):
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=n)
    pos, mass, lv, pr = _setup(B, ps, leaf=leaf, gs=gs)
    accs = []
    for pairs in (pr, pr, None):
        acc = torch.full((n, 3), 5.0, device="cuda")
        B.ph_pp_accel(lv, pairs, B.PH_G_EXACT, None, acc)
        accs.append(acc.cpu().numpy())
    _, _, lv1, pr1 = _setup(B, ps, leaf=leaf, gs=gs, qo=1)
    acc = torch.full((n, 3), 5.0, device="cuda")
    B.ph_pp_accel(lv1, pr1, B.PH_G_EXACT, None, acc)
    accs.append(acc.cpu().numpy())
    for a in accs[1:]:
        np.testing.assert_array_equal(a, accs[0])
    check_parity(accs[0], oracle_accel(ps))
    if n >= 4096 and leaf <= 32:
        assert _lists(B, pr).max() > 8 * 4
    for h in (pr, lv, pr1, lv1):
        B.ph_free(h)


def test_split_groups_in_active_mode(gpu_lib):
    # inactive groups have empty lists; the active ones' forces are the plain
    # step's bit for bit
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=5000)
    pos, mass, lv, pr = _setup(B, ps)
    full = torch.zeros((ps.n, 3), device="cuda")
    B.ph_pp_accel(lv, pr, B.PH_G_EXACT, None, full)
    act = torch.zeros(ps.n, dtype=torch.uint8, device="cuda")
    act[::701] = 1
    B.ph_leaves_set_active(lv, act)
    bp = ps.boxes[0]
    lv = B.ph_build_leaves(pos, mass, B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, 32), leaves=lv)
    pr = B.ph_leaf_pairs(lv, pairs=pr)
    acc = torch.full((ps.n, 3), 5.0, device="cuda")
    B.ph_pp_accel(lv, pr, B.PH_G_EXACT, None, acc)
    on = act.bool()
    assert torch.equal(acc[on], full[on])
    for h in (pr, lv):
        B.ph_free(h)


def test_noalloc_runs_out_of_task_slots(gpu_lib):
    # a clustered box whose groups ask for more tasks than the fixed array
    # holds: the groups left over are summed whole
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=3000)
    pos = ps.pos.copy()
    pos[:1500] *= np.float32(0.3)
    ps = synth.ParticleSet(pos, ps.mass, ps.boxes, ps.offsets, "clump")
    bp = ps.boxes[0]
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, 4)
    acc = torch.zeros((ps.n, 3), device="cuda")
    try:
        B.ph_accel_noalloc(torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda(), prm, acc)
    except B.PhError as e:
        assert e.code == B.PH_ERR_CAPACITY      # the documented limit of its list
        pytest.skip("the list itself does not fit")
    check_parity(acc.cpu().numpy(), oracle_accel(ps))
