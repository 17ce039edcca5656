"""Rounding of the FP32 mean field: no further from the 64-bit sum than a sum by
columns is.

G is a sum of some 50 column groups a species, each itself a short sum, in FP32.  A
group's sum is off by a few units of its own size and the running sum by half a
unit (2^-25 of its size) per group added: about sqrt(100) / 2 units of 2^-24, 3e-7
of the largest |G|, and the force's own last addition half a unit more.  The bound
is 2^-21 = 4.8e-7 (eight units).  Adding every plane of every column straight into
the running sum, some 780 terms, measures 5e-7 to 1.1e-6 on these fields.
"""
import math

import numpy as np
import pytest

from paper_1105_3634_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BOUND = 2.0 ** -21


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_3634_gb300 import build
    build.build()
    from paper_1105_3634_gb300 import mlb
    return mlb


EPS = 1e4 * W.KT_LATTICE          # the mean field outweighs the hard-core force, which is subtracted


def exact(lat, lam, n):
    """sum_b sum_d 6 eps sigma^6 d / |d|^8 n^b(r + d) on sigma <= |d| <= lam sigma, [S][3][N]"""
    nx, ny, nz = lat.shape
    S = lat.nspecies
    R = int(lam * max(lat.sigma)) + 1
    out = np.zeros((S, 3, nz, ny, nx))
    for b in range(S):
        v = n[b].reshape(nz, ny, nx)
        for axis in range(3):
            pad = [(0, 0)] * 3
            pad[2 - axis] = (R, R)
            v = np.pad(v, pad) if axis == lat.wall_axis else np.pad(v, pad, mode="wrap")
        for dz in range(-R, R + 1):
            for dy in range(-R, R + 1):
                for dx in range(-R, R + 1):
                    q = dx * dx + dy * dy + dz * dz
                    w = v[R + dz:R + dz + nz, R + dy:R + dy + ny, R + dx:R + dx + nx]
                    for a in range(S):
                        s = 0.5 * (lat.sigma[a] + lat.sigma[b])
                        if q and s * s <= q <= (lam * s) ** 2:
                            k = 6.0 * EPS * s ** 6 / float(q) ** 4
                            for c, d in enumerate((dx, dy, dz)):
                                if d:
                                    out[a, c] += (k * d) * w
    return out.reshape(S, 3, -1)


FIELDS = {
    "wave_x": dict(wave=(1, 0, 0)),
    "wave_y": dict(wave=(0, 1, 0)),
    "wave_z": dict(wave=(0, 0, 1)),
    "wave_xy": dict(wave=(1, 1, 0)),
    "wave_xyz": dict(wave=(1, 1, 1)),
    "wave_x_walls_y": dict(wave=(1, 0, 0), wall_axis=1),
    "wave_y_walls_x": dict(wave=(0, 1, 0), wall_axis=0),
    "one_species_y": dict(wave=(0, 1, 0), sigma=[3.0]),
    "three_species_xy": dict(wave=(1, 1, 0), sigma=[2.0, 2.5, 3.0]),
    "noise": dict(wave=None),
}


@pytest.mark.parametrize("name", sorted(FIELDS))
def test_mean_field_rounding(gpu, name):
    k = dict(FIELDS[name])
    wave = k.pop("wave")
    sigma = k.pop("sigma", [2.0, 3.0])
    S, lam = len(sigma), 2.5
    shape = (40, 20, 18)
    base = W.Lattice(shape=shape, sigma=sigma, **k)
    n0 = W.densities_from_packing(0.3, sigma, [1.0 / S] * S)
    if wave is None:
        n = W.noise(base, n0, 0.05, seed=4)
    else:
        ph = sum(c * W.coordinate(base, q) / shape[q] for q, c in enumerate(wave))
        n = np.stack([n0[a] * (1 + (-1) ** a * 0.05 * np.sin(2 * math.pi * ph + 0.3)) for a in range(S)])
    force = []
    for eps in (0.0, EPS):
        lat = W.Lattice(shape=shape, sigma=sigma, eps=[[eps] * S for _ in range(S)],
                        lambda_c=[[lam] * S for _ in range(S)], **k)
        sim = gpu.Simulation(lat)
        sim.set_fields(n)
        force.append(sim.rest_force())
        held = sim.moments()[0]                     # the densities the device holds
        sim.close()
    ref = exact(lat, lam, held)
    err = np.abs(force[1] - force[0] - ref).max() / np.abs(ref).max()
    print(name, "%.2e" % err)
    assert err < BOUND
