"""Groups whose source lists span several segments: each segment is a task of
its own, and the group's sum (segments in order, compensated) does not depend
on which warps made it."""
import dataclasses

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


def _needed(cnt, segment):
    """Tasks of lists of cnt entries cut into segments."""
    cnt = cnt[cnt > segment]
    return int(np.sum(-(-cnt // segment)))


def _entries(n, leaf, gs=32):
    """Entries per segment (of a box with fewer than 14,592 groups)."""
    return max(min(max(n // 50, 256), 2000) // leaf, 8)


# lists that need more tasks than the no-allocation call has slots for (n / 2),
# though they fit its entries: cut into longer segments, the same in every call
# (which groups found slots was left to the order of arrival before); and lists
# with room, summed as ph_accel sums them
@pytest.mark.parametrize("n,rcut,runs_out", [(4096, 0.3, True), (16000, 0.3, True), (1000, 0.17, False),
                                             (12000, 0.17, False)])
def test_noalloc_and_its_task_slots(gpu_lib, n, rcut, runs_out):
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=n)
    bp = ps.boxes[0]
    bp = dataclasses.replace(bp, rcut=rcut, rs=rcut / 4.5)
    ps = synth.ParticleSet(ps.pos, ps.mass, [bp], ps.offsets, "wide")
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, 32)
    pos, mass = torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda()
    acc = torch.zeros((n, 3), device="cuda")
    lv, pr = B.ph_accel(pos, mass, prm, B.PH_G_EXACT, None, acc)
    want, cnt = acc.cpu().numpy().copy(), _lists(B, pr)
    assert cnt.sum() <= 32 * n
    assert (_needed(cnt, _entries(n, 32)) > n // 2) == runs_out
    got = []
    for _ in range(8):
        acc.fill_(5.0)
        B.ph_accel_noalloc(pos, mass, prm, acc)
        got.append(acc.cpu().numpy())
    for g in got[1:]:
        np.testing.assert_array_equal(g, got[0])
    if runs_out:
        check_parity(got[0], oracle_accel(ps))
    else:
        np.testing.assert_array_equal(got[0], want)
    for h in (pr, lv):
        B.ph_free(h)


# a captured step whose particles gather: many tasks where the capture saw none
def test_captured_lists_that_grow_into_segments(gpu_lib):
    import torch
    B = gpu_lib
    n = 4096
    ps = synth.workload("uniform_small", scale=n)
    bp = ps.boxes[0]
    prm = B.make_params(bp.L, bp.G, bp.eps, 0.12 / 4.5, 0.12, 1)
    pos, mass = torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda()
    lv = B.ph_build_leaves(pos, mass, prm)
    pr = B.ph_leaf_pairs(lv)
    assert _needed(_lists(B, pr), 256) == 0
    acc = torch.zeros((n, 3), device="cuda")
    g = B.ph_graph_create(lv, pr, pos, mass, B.PH_G_EXACT, None, acc, headroom=6.0)
    pos[: n // 2] = 0.5 + 0.05 * (pos[: n // 2] - 0.5)
    got = []
    for _ in range(8):
        B.ph_graph_launch(g)
        got.append(acc.cpu().numpy().copy())
        acc.fill_(5.0)
    B.ph_status(pr)
    for a in got[1:]:
        np.testing.assert_array_equal(a, got[0])
    lv1, pr1 = B.ph_accel(pos, mass, prm, B.PH_G_EXACT, None, acc)
    assert _needed(_lists(B, pr1), 256) > 400          # the capture saw none
    np.testing.assert_array_equal(acc.cpu().numpy(), got[0])
    for h in (g, pr, lv, pr1, lv1):
        B.ph_free(h)


# a handle reserved for few entries, then for many, and made for other leaves:
# the list has its tasks' slots each time, so that the sums are the direct mode's
def test_reserved_lists_get_their_slots_at_every_build(gpu_lib):
    import torch
    B = gpu_lib
    pr = None
    for n, leaf, capacity in ((300, 32, 2000), (9000, 32, 400_000), (9000, 4, 2_000_000)):
        ps = synth.workload("uniform_small", scale=n)
        bp = ps.boxes[0]
        prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, leaf)
        lv = B.ph_build_leaves(torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda(), prm)
        pr = B.ph_pairs_reserve(capacity, pairs=pr)
        pr = B.ph_leaf_pairs(lv, pairs=pr)
        acc, direct = (torch.full((n, 3), 5.0, device="cuda") for _ in range(2))
        B.ph_pp_accel(lv, pr, B.PH_G_EXACT, None, acc)
        B.ph_pp_accel(lv, None, B.PH_G_EXACT, None, direct)
        B.ph_status(pr)
        assert torch.equal(acc, direct)
        B.ph_free(lv)
    B.ph_free(pr)
