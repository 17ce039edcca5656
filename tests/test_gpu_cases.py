"""The 64-bit restatement of the method in perf/cases.py against the library, on a
small lattice of every kind of case (and of the explicit forcing): the two share no
code, so each pins the other.  Bound: populations within 1e-5 of their largest value,
as the densities and velocities of the parity tests."""
import importlib.util
import os

import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-5
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = {
    "binary": dict(nx=33, ny=18, nz=20, steps=4),
    "plain_order": dict(nx=128, ny=96, nz=88, steps=2),             # above 2^20 sites: launches in plain stream order
    "channel_x": dict(nx=18, ny=17, nz=20, packing=0.15, wall=0, wall_u=0.02, steps=4),
    "channel_y": dict(nx=33, ny=17, nz=12, packing=0.15, wall=1, wall_u=0.02, steps=4),
    "channel_z": dict(nx=24, ny=17, nz=13, packing=0.15, wall=2, wall_u=0.02, steps=4),
    "drag": dict(nx=20, ny=18, nz=16, drag=True, steps=4),
    "explicit": dict(nx=20, ny=18, nz=16, packing=0.1, explicit=True, steps=4),
    "sweeps": dict(nx=20, ny=18, nz=16, sigma="2,3", packing=0.2, amp=0.02, sweeps=3, steps=3),
    "tails": dict(nx=20, ny=18, nz=16, sigma="2,3", packing=0.25, amp=0.0, noise=0.01, tails=True, steps=3),
    "tails_channel": dict(nx=20, ny=12, nz=16, sigma="2,3", packing=0.2, amp=0.01, tails=True, wall=1, wall_u=0.01, steps=3),
    "tails_bf16": dict(nx=20, ny=18, nz=16, sigma="2,3", packing=0.25, amp=0.0, noise=0.01, tails=True, meanfield="bf16",
                       steps=3),
    "three": dict(nx=48, ny=12, nz=11, sigma="2,2.5,3", packing=0.211, amp=0.0, noise=0.0, wall=1, wall_u=0.05, solute=True,
                  steps=3),
    "body_force": dict(nx=20, ny=19, nz=18, sigma="8,4", packing=0.211, amp=0.01, noise=0.0, flow=0.04, steps=2),
    "upload": dict(nx=20, ny=17, nz=16, flow=0.02, upload=True, steps=3),
    "batch": dict(kind="batch", members=4, nx=16, ny=12, nz=10, packing=0.18, steps=4),
}


@pytest.fixture(scope="module")
def cases():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_3634_gb300 import build
    build.build()
    spec = importlib.util.spec_from_file_location("perf_cases", os.path.join(ROOT, "perf", "cases.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize("name", sorted(CASES))
def test_restatement_agrees(cases, name):
    import torch
    case = cases._case(name=name, **CASES[name])
    state = cases.prepare(case, 3)
    out = cases.run(state)
    f = torch.from_numpy(out["f"]).double().cuda()
    ref = cases.exact(case, 3)
    assert torch.equal(torch.from_numpy(out["n_ref"]).cuda(), ref["n_ref"])
    err = float((f - ref["f"]).abs().max() / ref["f"].abs().max())
    print(name, "%.2e" % err)
    assert err < TOL
    if state["batch"] is not None:
        state["batch"].close()
    for sim in state["sims"]:
        sim.close()
