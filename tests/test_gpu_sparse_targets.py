"""Targets with few sources within the cutoff -- sparse boxes, isolated pairs
beside a dense clump, a clump's edge: as precise as those with many.

The exact kernel's two forms differ most there: near the cutoff the weight is
1/57 of the Newtonian term, from which the inverse-distance form subtracts its
polynomial in FP32 (99th percentile 8.9e-6 with one source, 2.9e-6 with five),
while the general form keeps a few 1e-7 of the weight."""
import numpy as np
import pytest

from helpers import gpu_accel, oracle_accel, rel_errors
from paper_1802_09824_gb300 import synth
from paper_1802_09824_gb300.synth import ParticleSet

pytestmark = pytest.mark.gpu

# General form: 7e-7 at the 99th percentile (SFU operations, polynomial); the
# separations are rounded to 2^-24 of at most the cutoff, and near it the weight
# falls as r^-12, so 7e-7 more.  The tests below compare targets with a source or
# more beyond half the cutoff, where every term is of one size.
TOL = 1.5e-6


def _params(**kw):
    import dataclasses
    return dataclasses.replace(synth.workload("uniform_small", scale=8).boxes[0], **kw)


def _neighbours(ps, box=0):
    from scipy.spatial import cKDTree
    bp = ps.boxes[box]
    x = np.mod(ps.pos[ps.box_slice(box)].astype(np.float64), bp.L)
    t = cKDTree(x, boxsize=bp.L)
    return t.query_ball_point(x, bp.rcut, return_length=True) - 1


def _check(B, ps, few, at_least, gs=0):
    got, lv, pr = gpu_accel(B, ps, group_size=gs)
    import torch
    direct = torch.zeros((ps.n, 3), device="cuda")
    B.ph_pp_accel(lv, None, B.PH_G_EXACT, None, direct)
    np.testing.assert_array_equal(direct.cpu().numpy(), got)      # the walk chooses alike
    e = []
    for b in range(len(ps.boxes)):
        nb = _neighbours(ps, b)
        t = np.flatnonzero((nb >= 1) & (nb <= few))
        e.append(rel_errors(got[ps.box_slice(b)][t], oracle_accel(ps, targets=t, box=b)))
    e = np.concatenate(e)
    assert e.size >= at_least
    q = float(np.percentile(e, 99))
    assert q <= TOL, f"{e.size} targets with 1..{few} sources: p99 {q:.2e}"
    for h in (pr, lv):
        B.ph_free(h)


@pytest.mark.parametrize("gs", [0, 16, 8])
@pytest.mark.parametrize("per_box,U", [(2, 2.25), (6, 2.25), (2, 2.299)])
def test_boxes_of_a_few_particles(gpu_lib, per_box, U, gs):
    # 400 boxes; two particles: 0.4 to 0.9999 cutoffs apart; six: within one another's reach
    rng = np.random.default_rng(per_box)
    bp = _params()
    bp = _params(rs=bp.rcut / (2 * U), eps=bp.rcut / U / 75)
    nb = 400
    u = rng.normal(size=(nb, per_box, 3))
    u /= np.linalg.norm(u, axis=2, keepdims=True)
    if per_box == 2:
        u[:, 0] = 0.0
        r = bp.rcut * rng.uniform(0.4, 0.9999, (nb, per_box, 1))
    else:
        r = 0.6 * bp.rcut * rng.random((nb, per_box, 1)) ** (1 / 3)
    pos = (rng.uniform(0.3, 0.7, (nb, 1, 3)) + r * u).astype(np.float32).reshape(-1, 3)
    mass = rng.uniform(0.5, 2.0, nb * per_box).astype(np.float32)
    ps = ParticleSet(pos, mass, [bp] * nb, np.arange(nb + 1) * per_box, "few")
    _check(gpu_lib, ps, per_box, nb * per_box // 2, gs)


@pytest.mark.parametrize("gs", [0, 16])
def test_isolated_pairs_beside_a_dense_clump(gpu_lib, gs):
    # the box's mean would call every target dense
    rng = np.random.default_rng(3)
    bp = _params(rcut=0.05, rs=0.05 / 4.5, eps=0.05 / 4.5 * 2 / 75)
    site = (np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.25) / 8
    site = site[1:]
    u = rng.normal(size=site.shape)
    u *= (bp.rcut * rng.uniform(0.5, 0.999, len(site)) / np.linalg.norm(u, axis=1))[:, None]
    clump = np.full(3, 0.25 / 8) + 0.02 * rng.normal(size=(400_000, 3)) / 3
    pos = np.concatenate([site, site + u, clump])
    pos = np.mod(pos, 1.0).astype(np.float32)
    ps = ParticleSet(pos, np.full(len(pos), 1.0 / len(pos), np.float32), [bp], np.array([0, len(pos)]), "void")
    n_mean = len(pos) * 4 / 3 * np.pi * bp.rcut ** 3
    assert n_mean > 200
    _check(gpu_lib, ps, 3, 900, gs)


def test_the_edge_of_a_clump(gpu_lib):
    # a Plummer sphere in an empty box: its outer particles see few sources
    rng = np.random.default_rng(5)
    bp = _params()
    n = 10_000
    r = 0.03 / np.sqrt(rng.uniform(0.02, 1, n) ** (-2 / 3) - 1 + 1e-6)
    r = np.minimum(r, 0.45)
    u = rng.normal(size=(n, 3))
    pos = (0.5 + r[:, None] * u / np.linalg.norm(u, axis=1)[:, None]).astype(np.float32)
    ps = ParticleSet(pos, np.full(n, 1.0 / n, np.float32), [bp], np.array([0, n]), "plummer")
    _check(gpu_lib, ps, 40, 30)


@pytest.mark.parametrize("n,gs", [(150, 0), (700, 0), (700, 16), (2000, 0)])
def test_sparse_uniform_boxes(gpu_lib, n, gs):
    # 3 to 46 sources a target; targets whose terms cancel are left to the other tests
    ps = synth.workload("uniform_small", scale=n)
    ref = oracle_accel(ps)
    got, lv, pr = gpu_accel(gpu_lib, ps, group_size=gs)
    e = rel_errors(got, ref)
    big = np.linalg.norm(ref.acc, axis=1) >= 0.3 * np.median(np.linalg.norm(ref.acc, axis=1))
    assert np.percentile(e[big], 99) <= 2 * TOL
    for h in (pr, lv):
        gpu_lib.ph_free(h)
