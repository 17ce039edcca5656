"""Corners of the work decomposition: walls closer together than the shells reach,
and grouped launches on 16 x 8 tiles.

Bounds, as in the parity tests: accelerations of one FP32 force evaluation
within 1e-4 of the field's largest value, densities and velocities after a few
steps within 1e-5; grouped members equal the members stepped alone bit for bit.
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


def tails(S, lam, eps=0.05):
    return dict(eps=[[eps * W.KT_LATTICE] * S for _ in range(S)], lambda_c=[[lam] * S for _ in range(S)])


# the lattice's extent between the walls is below the reach, down to one site: global passes,
# tiles with several threads per site, column and far attraction
THIN = {
    "global_x1": dict(sigma=[8.0, 4.0], shape=(1, 11, 10), wall_axis=0),
    "global_x5": dict(sigma=[8.0, 4.0], shape=(5, 11, 10), wall_axis=0),
    "global_y1": dict(sigma=[4.0, 3.0], shape=(9, 1, 10), wall_axis=1),
    "global_y3": dict(sigma=[5.0], shape=(33, 3, 7), wall_axis=1, drag_only=True),
    "global_z1": dict(sigma=[4.0, 2.0, 3.0], shape=(9, 8, 1), wall_axis=2),
    "global_z2_sweeps": dict(sigma=[4.0, 3.0], shape=(11, 9, 2), wall_axis=2, predictor_sweeps=2),
    "four_x2": dict(sigma=[1.5, 2.0, 2.5, 3.0], shape=(2, 9, 8), wall_axis=0),
    "tile3_x1": dict(sigma=[2.0, 3.0], shape=(1, 9, 8), wall_axis=0),
    "tile3_y2": dict(sigma=[2.0, 2.5, 3.0], shape=(17, 2, 8), wall_axis=1),
    "tile2_z1": dict(sigma=[1.5, 2.0], shape=(33, 6, 1), wall_axis=2),
    "columns_z3": dict(sigma=[2.0, 3.0], shape=(17, 16, 3), wall_axis=2, **tails(2, 2.5)),
    "far_y4": dict(sigma=[4.0], shape=(21, 4, 11), wall_axis=1, **tails(1, 2.5)),
}


@pytest.mark.parametrize("name", sorted(THIN))
def test_walls_closer_than_the_reach(gpu, orc, name):
    lat = W.Lattice(**THIN[name])
    n0 = W.densities_from_packing(0.1, lat.sigma, [1.0 / lat.nspecies] * lat.nspecies)
    n, u = W.noise(lat, n0, 0.05, 5), W.random_velocities(lat, 0.02, 6)
    sim = gpu.Simulation(lat)
    sim.set_fields(n, u)
    f = orc.init(lat, n, u)
    on, oj = orc.moments(lat, f)
    assert site(sim.acceleration(), orc.accel(lat, on, oj)) < TOL_ACC
    sim.step(2)
    orc.step(lat, f, 2)
    gn, gu = sim.moments()
    on, oj = orc.moments(lat, f)
    assert site(gn, on) < TOL_STATE
    assert site(gu, orc.velocity_fields(lat, on, oj)) < TOL_STATE
    sim.close()


def members(shapes, **k):
    out = []
    for j, shape in enumerate(shapes):
        for wall in (-1, 0, 1, 2):
            lat = W.Lattice(shape=shape, wall_axis=wall, wall_u_lo=(0.0, 0.0, 0.01) if wall != 2 else (0.01, 0.0, 0.0), **k)
            n0 = W.densities_from_packing(0.2, lat.sigma, [1.0 / lat.nspecies] * lat.nspecies)
            out.append((lat, W.noise(lat, n0, 0.02, seed=20 + 4 * j + wall)))
    return out


# lanes of 16 x 8 tiles: every wall axis, drag-only mode, one species; the last two sets have a
# member whose own tiles are of the other width than its lane's
GROUPS = {
    "narrow": members([(16, 16, 16), (16, 12, 9)], sigma=[1.0, 1.5]),
    "narrow_drag": members([(16, 16, 16), (48, 8, 5)], sigma=[1.0, 1.5], drag_only=True),
    "narrow_one": members([(16, 9, 7), (12, 24, 6)], sigma=[1.5]),
    "wide_member": members([(16, 16, 16), (32, 12, 4)], sigma=[1.0, 1.5]),
    "narrow_member": members([(16, 16, 4), (64, 20, 16)], sigma=[1.0, 1.5]),
}


@pytest.mark.parametrize("name", sorted(GROUPS))
def test_grouped_tiles_of_both_widths(gpu, name):
    import torch

    def make(lat, n):
        sim = gpu.Simulation(lat, stream=torch.cuda.Stream())
        sim.set_fields(n, W.random_velocities(lat, 0.005, seed=11))
        return sim

    alone = []
    for lat, n in GROUPS[name]:
        sim = make(lat, n)
        sim.step(5)
        alone.append(sim.populations()[0])
        sim.close()
    sims = [make(lat, n) for lat, n in GROUPS[name]]
    batch = gpu.Batch(sims, lanes=1)
    batch.step(5)
    batch.synchronize()
    assert batch.grouped_members() == len(sims)
    for k, sim in enumerate(sims):
        assert np.array_equal(sim.populations()[0].view(np.uint32), alone[k].view(np.uint32)), k
    batch.close()
    for sim in sims:
        sim.close()
