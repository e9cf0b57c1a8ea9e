"""The exact PP kernel's two forms of the softened short-range weight: the
inverse-distance form (rcut / 2R_s <= 2.3 and eps <= 2R_s / 64, dense groups)
and the general form, at both sides of the line between them, against the
oracle.  The boxes are dense: 450 sources a target."""
import dataclasses

import numpy as np
import pytest

from helpers import check_parity, gpu_accel, oracle_accel
from paper_1802_09824_gb300 import synth

pytestmark = pytest.mark.gpu


def _box(U, eps_div, scale=20_000, L=1.0):
    """A uniform box with rcut / 2R_s = U and eps = 2R_s / eps_div (0: none)."""
    ps = synth.workload("uniform_small", scale=scale)
    bp = ps.boxes[0]
    rs = bp.rcut / (2.0 * U) * L
    bx = dataclasses.replace(bp, L=bp.L * L, rcut=bp.rcut * L, rs=rs, eps=2.0 * rs / eps_div if eps_div else 0.0)
    return synth.ParticleSet((ps.pos * np.float32(L)).astype(np.float32), ps.mass, [bx], ps.offsets, "box")


# the edges of the inverse-distance form's range (U 2.3, eps 2R_s / 64), no
# softening (the kernel's floor), a narrow split, and just outside each line;
# the tolerance is the exact path's (helpers)
@pytest.mark.parametrize("U,eps_div", [(2.25, 75.0), (2.3 * (1 - 1e-12), 64.0), (2.25, 0), (0.5, 64.0), (0.05, 200.0),
                                       (2.3 * (1 + 1e-9), 64.0), (2.25, 64.0 * (1 - 1e-9)), (2.25, 2.0)])
def test_forms_match_the_oracle(gpu_lib, U, eps_div):
    ps = _box(U, eps_div)
    got, lv, pr = gpu_accel(gpu_lib, ps)
    check_parity(got, oracle_accel(ps))
    for h in (pr, lv):
        gpu_lib.ph_free(h)


@pytest.mark.parametrize("L", [1e-6, 37.0, 1e6])
def test_inverse_form_in_other_units(gpu_lib, L):
    # the lengths are scaled by a power of two near 1 / rcut
    ps = _box(2.25, 75.0, L=L)
    got, lv, pr = gpu_accel(gpu_lib, ps)
    check_parity(got, oracle_accel(ps))
    for h in (pr, lv):
        gpu_lib.ph_free(h)


def test_forms_agree_across_the_line(gpu_lib):
    # the softening a hair below and above 2R_s / 64: the same forces up to
    # both forms' FP32 errors (each within ~2e-7 of the summed terms' size)
    out = []
    for d in (64.0 * (1 + 1e-9), 64.0 * (1 - 1e-9)):
        got, lv, pr = gpu_accel(gpu_lib, _box(2.25, d))
        out.append(got.astype(np.float64))
        for h in (pr, lv):
            gpu_lib.ph_free(h)
    assert np.mean(out[0] != out[1]) > 0.5          # two forms indeed
    diff = np.linalg.norm(out[0] - out[1], axis=1) / np.linalg.norm(out[0], axis=1)
    assert np.percentile(diff, 90) <= 2e-6


def test_one_box_outside_the_range_takes_all_to_the_general_form(gpu_lib):
    # boxes summed in one launch share a form
    a, b = _box(2.25, 75.0, scale=12_000), _box(2.25, 8.0, scale=15_000)
    ps = synth.ParticleSet(np.concatenate([a.pos, b.pos]), np.concatenate([a.mass, b.mass]), a.boxes + b.boxes,
                           np.array([0, a.n, a.n + b.n]), "two")
    got, lv, pr = gpu_accel(gpu_lib, ps)
    for k in range(2):
        check_parity(got[ps.box_slice(k)], oracle_accel(ps, box=k))
    for h in (pr, lv):
        gpu_lib.ph_free(h)
