"""Cost of the global passes by species count: a fourth, smaller species adds seven pair
shells to nine.  With one launch bound for every species count the four-species kernel kept
3 KB of its sums in local memory and took 3.6 times the three species' time."""
import pytest

from paper_1105_3634_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_3634_gb300 import build
    build.build()
    from paper_1105_3634_gb300 import mlb
    return mlb


def test_four_species_cost_by_their_pairs(gpu):
    import torch
    ms = []
    for sigma in ([6.0, 4.0, 3.0], [6.0, 4.0, 3.0, 2.0]):
        S = len(sigma)
        lat = W.Lattice(shape=(64, 64, 64), sigma=sigma)
        stream = torch.cuda.Stream()
        sim = gpu.Simulation(lat, stream=stream)
        sim.set_fields(W.noise(lat, W.densities_from_packing(0.1, sigma, [1.0 / S] * S), 0.01, 3))
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for _ in range(6):
            e0.record(stream)
            sim.step(2)
            e1.record(stream)
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        ms.append(best)
        sim.close()
    assert ms[1] < 2.5 * ms[0], ms
