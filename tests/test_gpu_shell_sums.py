"""The contact-shell sums of both force passes against the FP64 oracle, on the
lattices where their kernels differ: species counts, offset classes, drag-only
mode, walls, sizes around the tile edges.

Bounds, as in the parity tests: accelerations of one FP32 force evaluation
within 1e-4 of the field's largest value, densities and velocities after a few
steps within 1e-5.
"""
import numpy as np
import pytest

from paper_1105_3634_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL_STATE = 1e-5
TOL_ACC = 1e-4


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_3634_gb300 import build
    build.build()
    from paper_1105_3634_gb300 import mlb
    return mlb


def site(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def check(gpu, orc, lat, n, u, steps):
    sim = gpu.Simulation(lat)
    sim.set_fields(n, u)
    f = orc.init(lat, n, u)
    on, oj = orc.moments(lat, f)
    assert site(sim.acceleration(), orc.accel(lat, on, oj)) < TOL_ACC
    sim.step(steps)
    orc.step(lat, f, steps)
    gn, gu = sim.moments()
    on, oj = orc.moments(lat, f)
    assert site(gn, on) < TOL_STATE
    assert site(gu, orc.velocity_fields(lat, on, oj)) < TOL_STATE
    sim.close()


def fields(lat, packing, seed=5):
    n0 = W.densities_from_packing(packing, lat.sigma, [1.0 / lat.nspecies] * lat.nspecies)
    return W.noise(lat, n0, 0.05, seed), W.random_velocities(lat, 0.02, seed + 1)


# reach 1: shells that are unions of axis, face and corner offsets
CUBE = {
    "one_axis_face": dict(sigma=[1.0], shape=(33, 5, 14)),
    "one_all_drag": dict(sigma=[1.5], shape=(31, 9, 3), drag_only=True),
    "two_mixed_masks": dict(sigma=[1.0, 1.5], shape=(34, 7, 13), wall_axis=2),
    "three": dict(sigma=[1.0, 1.25, 1.5], shape=(35, 6, 5), wall_axis=0),
    "three_drag": dict(sigma=[1.0, 1.25, 1.5], shape=(8, 6, 5), drag_only=True),
    "four": dict(sigma=[1.0, 1.2, 1.4, 1.5], shape=(36, 5, 4)),
}


@pytest.mark.parametrize("name", sorted(CUBE))
def test_cube_shells(gpu, orc, name):
    lat = W.Lattice(**CUBE[name])
    n, u = fields(lat, 0.12)
    check(gpu, orc, lat, n, u, 3)


# tiles of 16 x 8 sites (nx that leaves 32-wide tiles idle), full, one short and one over
NARROW = {
    "full": dict(sigma=[1.0, 1.5], shape=(16, 8, 6)),
    "short": dict(sigma=[1.0, 1.5], shape=(47, 15, 5), wall_axis=1),
    "over": dict(sigma=[1.5], shape=(12, 9, 19), drag_only=True),
    "many": dict(sigma=[1.0, 1.5], shape=(80, 40, 33), wall_axis=0),
}


@pytest.mark.parametrize("name", sorted(NARROW))
def test_narrow_tiles(gpu, orc, name):
    lat = W.Lattice(**NARROW[name])
    n, u = fields(lat, 0.12)
    check(gpu, orc, lat, n, u, 3)
    out = []
    for split in (False, True):                       # fused and split launches agree bit for bit
        sim = gpu.Simulation(lat, split_collide=split)
        sim.set_fields(n, u)
        sim.step(4)
        out.append(sim.populations()[0])
        sim.close()
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))


# rows that are no multiple of 16 bytes, walls on every axis (one site thick too)
ROWS = {
    "one_over": dict(sigma=[1.0, 1.5], shape=(33, 5, 7)),
    "two_over": dict(sigma=[1.0, 1.5], shape=(34, 8, 3), wall_axis=0),
    "narrow": dict(sigma=[1.0, 1.5], shape=(17, 9, 6), wall_axis=1),
    "three_short": dict(sigma=[1.0], shape=(61, 3, 5)),
    "one_plane": dict(sigma=[1.0, 1.5], shape=(18, 7, 1), wall_axis=2, wall_u_lo=(0.01, 0.0, 0.0),
                      wall_u_hi=(0.0, 0.02, 0.0)),
    "moving_x": dict(sigma=[1.0, 1.5], shape=(20, 7, 6), wall_axis=0, wall_u_lo=(0.0, 0.02, -0.01),
                     wall_u_hi=(0.0, -0.01, 0.02)),
    "reach2": dict(sigma=[1.5, 2.0], shape=(35, 6, 9), drag_only=True),
    "three_species": dict(sigma=[1.0, 1.25, 1.5], shape=(37, 5, 6), wall_axis=2),
}


@pytest.mark.parametrize("name", sorted(ROWS))
def test_unaligned_rows(gpu, orc, name):
    lat = W.Lattice(**ROWS[name])
    n, u = fields(lat, 0.1)
    check(gpu, orc, lat, n, u, 3)
    out = []
    for split in (False, True):
        sim = gpu.Simulation(lat, split_collide=split)
        sim.set_fields(n, u)
        sim.step(4)
        out.append(sim.populations()[0])
        sim.close()
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))


# reach 2 and 3: shells from sign groups, one to three threads per site, tiles of 32 and 16
GROUPS = {
    "one_reach2": dict(sigma=[2.0], shape=(34, 5, 9)),
    "one_reach3_drag": dict(sigma=[3.0], shape=(33, 9, 7), drag_only=True),
    "two_reach2": dict(sigma=[1.5, 2.0], shape=(31, 6, 14), wall_axis=1),
    "two_reach3": dict(sigma=[2.0, 3.0], shape=(35, 17, 6), wall_axis=2),
    "two_reach3_drag": dict(sigma=[1.0, 3.0], shape=(8, 7, 20), drag_only=True),
    "two_reach3_sweeps": dict(sigma=[2.0, 3.0], shape=(32, 8, 13), predictor_sweeps=3),
    "three_reach2": dict(sigma=[1.0, 1.5, 2.0], shape=(33, 6, 7)),
    "three_reach3": dict(sigma=[2.0, 2.5, 3.0], shape=(17, 9, 10), wall_axis=0),
    "three_reach3_drag": dict(sigma=[1.0, 2.0, 3.0], shape=(16, 8, 7), drag_only=True),
    "three_reach3_sweeps": dict(sigma=[2.0, 2.5, 3.0], shape=(31, 7, 8), predictor_sweeps=2, wall_axis=1),
    "one_reach4": dict(sigma=[4.0], shape=(9, 7, 6)),
    "two_reach8": dict(sigma=[8.0, 4.0], shape=(19, 11, 10), wall_axis=1),
    "two_reach5_drag": dict(sigma=[5.0, 1.5], shape=(33, 8, 7), wall_axis=0, drag_only=True),
    "two_reach4_sweeps": dict(sigma=[4.0, 3.0], shape=(11, 9, 13), wall_axis=2, predictor_sweeps=2),
    "three_reach4": dict(sigma=[4.0, 2.0, 3.0], shape=(10, 9, 8)),
    "four_reach3": dict(sigma=[1.5, 2.0, 2.5, 3.0], shape=(13, 9, 8), wall_axis=1),
    "four_reach2": dict(sigma=[1.0, 1.5, 1.75, 2.0], shape=(33, 5, 6), wall_axis=2),
}


@pytest.mark.parametrize("name", sorted(GROUPS))
def test_group_shells(gpu, orc, name):
    lat = W.Lattice(**GROUPS[name])
    n, u = fields(lat, 0.12)
    check(gpu, orc, lat, n, u, 3)
