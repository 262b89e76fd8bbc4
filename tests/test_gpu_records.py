"""The integer forms of FP64 conversions and comparisons in the passes over the
particles: one search and step of particles at the edges of those forms
(zeros, signed zeros, ties of the rounding, values outside the floats' range,
particles on the ends of the period) against the oracle."""
import numpy as np
import pytest

from gpu_common import lists_to_original, zdist

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_03344_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _fields(n=3000):
    rng = np.random.default_rng(4)
    f = {k: rng.uniform(-0.5, 0.5, n) for k in ("x", "y", "z")}
    f.update({k: rng.normal(0.0, 1.0, n) for k in ("vx", "vy", "vz")})
    f["h"] = rng.uniform(0.06, 0.08, n)
    f["m"] = np.full(n, 1.0 / n)
    f["u"] = rng.uniform(1.0, 2.0, n)
    # halfway between two floats, and one ulp to each side
    t = np.float64(np.float32(0.3)) + 2.0 ** -26
    f["vx"][:6] = [t, np.nextafter(t, 0), np.nextafter(t, 1), 0.0, -0.0, 1e-42]
    f["vy"][:6] = [-t, 2.0 ** -127, -2.0 ** -149, 2.0 ** -150, 1e-300, -1e-320]
    f["z"][:6] = [-0.5, np.nextafter(0.5, 0), 0.0, -0.0, 0.25, 1e-310]
    f["x"][:2] = [0.0, -0.0]
    f["h"][10:14] = 0.0625       # on an edge of the histogram of h / h_max, once
    f["h"][14] = 0.08            # ... this is h_max
    return f


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
def test_edge_values(B, orc, precision, tol):
    f = _fields()
    n = len(f["x"])
    sim = B.SPH(n, precision=precision)
    sim.set_particles(f)
    sim.find_neighbors()
    o, c = lists_to_original(*sim.neighbors(), n)
    nb = orc.neighbors(f["x"], f["y"], f["z"], f["h"], 1.0)
    assert np.array_equal(o, nb.off) and np.array_equal(c, nb.col)
    sim.step(1)
    ref = orc.Sim(f)
    ref.step(1)
    for k in ("x", "y", "vx", "vy", "vz", "u", "h"):
        assert np.abs(sim.field(k) - ref[k]).max() <= tol * np.abs(ref[k]).max(), k
    assert zdist(sim.field("z"), ref["z"]).max() <= tol
    assert sim.field("z").min() >= -0.5 and sim.field("z").max() < 0.5
    sim.close()
