"""A capture makes room for the replays' longer lists without losing the list
at hand: its sums, view and counts are the same after ph_graph_create, before
any replay, also when the capture's allocations fail."""
import numpy as np
import pytest

from paper_1802_09824_gb300 import synth

pytestmark = pytest.mark.gpu


def _state(B, lv, pr, n):
    import torch
    acc = torch.full((n, 3), 5.0, device="cuda")
    B.ph_pp_accel(lv, pr, B.PH_G_EXACT, None, acc)
    v = B.ph_pairs_get_view(pr)
    return [acc.cpu().numpy(), v["entries"].cpu().numpy(), v["counts"].cpu().numpy(), v["group_off"].cpu().numpy(),
            B.ph_count_within(lv, pr)]


# lists with no task, with tasks, with lists of many segments; headrooms that
# leave, move and multiply the buffers
@pytest.mark.parametrize("n,headroom", [(20, 0.0), (1000, 0.0), (4096, 0.25), (4096, 4.0), (50_021, 1.0)])
def test_a_capture_keeps_the_list(gpu_lib, n, headroom):
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=n)
    bp = ps.boxes[0]
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, 32)
    pos, mass = torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda()
    lv = B.ph_build_leaves(pos, mass, prm)
    pr = B.ph_leaf_pairs(lv)
    ref = _state(B, lv, pr, n)
    out = torch.full((n, 3), 5.0, device="cuda")
    # every allocation of the growth fails in turn: refused, nothing lost
    g = None
    for k in range(8):
        B.ph_debug_fail_allocation(k)
        try:
            g = B.ph_graph_create(lv, pr, pos, mass, B.PH_G_EXACT, None, out, headroom=headroom)
        except B.PhError as e:
            assert e.code == B.PH_ERR_OOM, str(e)
        finally:
            B.ph_debug_fail_allocation(-1)
        for a, b in zip(_state(B, lv, pr, n), ref):
            np.testing.assert_array_equal(a, b)
        if g is not None:
            break
    assert k == 3 or headroom < 1.0      # entries, counts and tasks all moved
    B.ph_graph_launch(g)
    np.testing.assert_array_equal(out.cpu().numpy(), ref[0])
    for a, b in zip(_state(B, lv, pr, n), ref):
        np.testing.assert_array_equal(a, b)
    for h in (g, pr, lv):
        B.ph_free(h)


def test_a_capture_on_a_reserved_list_that_overflowed(gpu_lib):
    # the list holds its reserved entries and nothing more: before the first
    # replay its (refused) sums read no entry past them, and the replay's list
    # has the room that the capture made
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=60)
    bp = ps.boxes[0]
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, 1)
    pos, mass = torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda()
    lv = B.ph_build_leaves(pos, mass, prm)
    full = B.ph_leaf_pairs(lv)
    want = _state(B, lv, full, ps.n)
    total = int(want[3][-1])
    assert 20 <= total <= 1024            # the capture's capacity for a list of unknown length is 1024
    pr = B.ph_pairs_reserve(total // 2)
    pr = B.ph_leaf_pairs(lv, pairs=pr)
    with pytest.raises(B.PhError) as ei:
        B.ph_status(pr)
    assert ei.value.code == B.PH_ERR_CAPACITY
    part = torch.full((ps.n, 3), 5.0, device="cuda")
    B.ph_pp_accel(lv, pr, B.PH_G_EXACT, None, part)
    part, within = part.cpu().numpy(), B.ph_count_within(lv, pr)
    out = torch.full((ps.n, 3), 5.0, device="cuda")
    g = B.ph_graph_create(lv, pr, pos, mass, B.PH_G_EXACT, None, out)
    again = torch.full((ps.n, 3), 5.0, device="cuda")
    B.ph_pp_accel(lv, pr, B.PH_G_EXACT, None, again)
    np.testing.assert_array_equal(again.cpu().numpy(), part)
    assert B.ph_count_within(lv, pr) == within
    B.ph_graph_launch(g)
    B.ph_status(pr)
    np.testing.assert_array_equal(out.cpu().numpy(), want[0])
    assert B.ph_count_within(lv, pr) == want[4]
    for h in (g, pr, full, lv):
        B.ph_free(h)


def test_a_capture_of_a_list_made_on_another_stream(gpu_lib):
    # the growth waits for a list that another stream is still making, and that
    # stream need not live on
    import torch
    B = gpu_lib
    ps = synth.workload("uniform_small", scale=50_021)
    bp = ps.boxes[0]
    prm = B.make_params(bp.L, bp.G, bp.eps, bp.rs, bp.rcut, 32)
    pos, mass = torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda()
    torch.cuda.synchronize()
    lv0, pr0 = B.ph_build_leaves(pos, mass, prm), None
    pr0 = B.ph_leaf_pairs(lv0)
    ref = _state(B, lv0, pr0, ps.n)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    lv = B.ph_build_leaves(pos, mass, prm, stream=a.cuda_stream)
    pr = B.ph_leaf_pairs(lv, stream=a.cuda_stream)
    out = torch.full((ps.n, 3), 5.0, device="cuda")
    torch.cuda.current_stream().synchronize()
    g = B.ph_graph_create(lv, pr, pos, mass, B.PH_G_EXACT, None, out, headroom=1.0, stream=b.cuda_stream)
    for x, y in zip(_state(B, lv, pr, ps.n), ref):
        np.testing.assert_array_equal(x, y)
    B.ph_graph_launch(g, stream=b.cuda_stream)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), ref[0])
    for h in (g, pr, lv, pr0, lv0):
        B.ph_free(h)
