"""Length units: the library takes positions, h and the period in any unit.
A power of two in front of every length changes no rounding of the search, so
the lists and n_i are those of the oracle for particles whose h is far from 1
(a parsec in metres is 3e16), by teams of lanes and by a thread per particle;
and the FP64 sums stay within their tolerance, also where squared distances
leave the range of the FP32 seeds of their square root."""
import os

import numpy as np
import pytest

from gpu_common import lists_to_original, normwise, normwise_vec
from test_gpu_rows import _cloud, _layers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_03344_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _scaled(f, unit):
    return {k: f[k] * unit if k in ("x", "y", "z", "h") else f[k] for k in f}


# 4 h^2 of every particle stays a normal float: 2^-54 gives 1e-35, 2^54 1e30 and more
@pytest.mark.parametrize("unit", [2.0 ** 54, 2.0 ** -54])
@pytest.mark.parametrize("n", [6000, 56000])     # teams; a thread each
@pytest.mark.parametrize("kind", ["faces", "big_reach", "few_z"])
def test_lists_in_any_unit(B, orc, kind, n, unit):
    f = _scaled(_cloud(kind, n), unit)
    sim = B.SPH(n, precision="fp64", max_pairs=800 * n, lz=unit)
    sim.set_particles(f)
    nb = orc.neighbors(f["x"], f["y"], f["z"], f["h"], unit, nthreads=os.cpu_count() or 1)
    for _ in range(2):           # rows counted first, then reserved from hints
        sim.find_neighbors()
        o, c = lists_to_original(*sim.neighbors(), n)
        assert np.array_equal(o, nb.off) and np.array_equal(c, nb.col)
        assert np.array_equal(sim.field("nown").astype(np.int64), nb.nown)
    sim.close()


@pytest.mark.parametrize("unit", [2.0 ** 54, 2.0 ** -54])
def test_reused_lists_in_any_unit(B, orc, unit):
    """The candidate superset is one of the two searches by teams."""
    n = 3000
    f = _scaled(_cloud("big_reach", n), unit)
    sim = B.SPH(n, precision="fp64", max_pairs=800 * n, lz=unit, list_skin=0.1)
    sim.set_particles(f)
    sim.find_neighbors()
    o, c = lists_to_original(*sim.neighbors(), n)
    nb = orc.neighbors(f["x"], f["y"], f["z"], f["h"], unit)
    assert np.array_equal(o, nb.off) and np.array_equal(c, nb.col)
    sim.close()


# at 2^63 the squared distances pass 2^120, beyond the seeds' range
@pytest.mark.parametrize("unit", [2.0 ** 63, 2.0 ** 54, 2.0 ** -54])
def test_fp64_sums_in_any_unit(B, orc, unit):
    f = _scaled(_layers("jittered", 12), unit)
    n = len(f["x"])
    rng = np.random.default_rng(8)
    f.update({k: rng.normal(0.0, 1.0, n) for k in ("vx", "vy", "vz")})
    sim = B.SPH(n, precision="fp64", max_pairs=800 * n, lz=unit)
    sim.set_particles(f)
    sim.find_neighbors()
    sim.density()
    sim.momentum_energy()
    nb = orc.neighbors(f["x"], f["y"], f["z"], f["h"], unit)
    rho = orc.density(f["x"], f["y"], f["z"], f["m"], f["h"], nb, unit)
    P, c = orc.eos(rho, f["u"])[:2]
    ref = orc.momentum_energy(f["x"], f["y"], f["z"], f["vx"], f["vy"], f["vz"], f["m"], f["h"], rho, P, c, nb, unit)
    assert normwise(sim.field("rho"), rho) < 1e-12
    assert normwise_vec([sim.field(k) for k in ("ax", "ay", "az")], ref[:3]) < 1e-12
    assert normwise(sim.field("du"), ref[3]) < 1e-12
    sim.close()
