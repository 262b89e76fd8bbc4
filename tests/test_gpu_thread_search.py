"""The search by one thread per particle, which more than 50,000 particles
take, on its rare paths: a pool that overflows, rows with words in the guard
band that are decided after the walk, rows that outgrow their reservation, and
candidate supersets of reused lists.  Lists and n_i against the oracle, bit
for bit."""
import os

import numpy as np
import pytest

from paper_1905_03344_gb300 import inputs
from gpu_common import lists_to_original
from test_gpu_parity import near_ties

pytestmark = pytest.mark.gpu

N = 56000
EDGE = 39                    # 59,319 particles
THREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def B():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_03344_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _cloud(seed, h_lo, h_hi, of, **kw):
    """A cloud of N particles as dense in h as one of `of` particles."""
    s = (of / N) ** (1.0 / 3.0)
    return inputs.random_cloud(N, seed=seed, h_lo=h_lo * s, h_hi=h_hi * s, **kw)


def _neighbors(orc, f):
    return orc.neighbors(f["x"], f["y"], f["z"], f["h"], 1.0, nthreads=THREADS)


def _check_lists(sim, nb):
    o, c = lists_to_original(*sim.neighbors(), len(nb.off) - 1)
    assert np.array_equal(o, nb.off) and np.array_equal(c, nb.col)
    assert np.array_equal(sim.field("nown").astype(np.int64), nb.nown.astype(np.int64))


def test_overflow(B, orc):
    """Rows of hundreds of neighbours, many with words in the guard band,
    against a pool far too small: warps whose reservation does not fit leave
    the pool alone, and the context goes on with lists that fit."""
    f = _cloud(3, 0.04, 0.09, 20000)
    sim = B.SPH(N, precision="fp64", max_pairs=10 * N)
    sim.set_particles(f)
    for _ in range(2):           # rows counted first, then reserved from hints
        with pytest.raises(B.SphError) as e:
            sim.find_neighbors()
        assert e.value.status == B.SPH_EOVERFLOW
    with pytest.raises(B.SphError) as e:
        sim.step(2)
    assert e.value.status == B.SPH_EOVERFLOW
    assert np.array_equal(sim.field("x"), f["x"]) and sim.dt()[2] == 0
    f["h"] = f["h"] * 0.2
    nb = _neighbors(orc, f)
    assert nb.off[-1] < 10 * N
    sim.set_particles(f)
    sim.find_neighbors()
    _check_lists(sim, nb)
    sim.close()


@pytest.mark.parametrize("cf", [0.0, 0.4])
def test_near_ties(B, orc, cf):
    f = near_ties(N // 2)
    nb = _neighbors(orc, f)
    sim = B.SPH(N, max_pairs=400 * N, cell_factor=cf)
    sim.set_particles(f)
    for _ in range(2):
        sim.find_neighbors()
        _check_lists(sim, nb)
    sim.close()


def test_rows_outgrowing_their_reservation(B, orc):
    """h grows fast (a target far above the counts), so that rows outgrow the
    space reserved from the previous step's lengths and are searched again."""
    f = _cloud(31, 0.07, 0.09, 2000, vscale=0.5)
    sim = B.SPH(N, precision="fp64", max_pairs=600 * N, n_target=150.0)
    sim.set_particles(f)
    counts = []
    for _ in range(3):
        nb = _neighbors(orc, {k: sim.field(k) for k in ("x", "y", "z", "h")})
        counts.append(np.diff(nb.off).astype(np.int64))
        sim.step(1)
        assert np.array_equal(sim.field("nnb").astype(np.int64), counts[-1])
        assert np.array_equal(sim.field("nown").astype(np.int64), nb.nown.astype(np.int64))
    sim.close()
    c0, c1 = counts[:2]
    assert np.sum(c1 > ((c0 + c0 // 3 + 8 + 7) // 8) * 8) > N // 20


@pytest.mark.parametrize("case", ["patch", "irregular", "cloud"])
def test_reused_supersets(B, orc, case):
    """Every step's exact lists from a superset, including steps that only
    filtered it."""
    f = {"patch": lambda: inputs.square_patch(EDGE),
         "irregular": lambda: inputs.irregular_patch(EDGE, seed_pos=6, seed_mass=7),
         "cloud": lambda: _cloud(31, 0.08, 0.1, 2500, vscale=0.3)}[case]()
    n = len(f["x"])
    sim = B.SPH(n, list_skin=0.25, max_pairs=400 * n)
    sim.set_particles(f)
    steps = 4
    for _ in range(steps):
        nb = _neighbors(orc, {k: sim.field(k) for k in ("x", "y", "z", "h")})
        sim.find_neighbors()
        _check_lists(sim, nb)
        sim.step(1)
        assert np.array_equal(sim.field("nnb").astype(np.int64), np.diff(nb.off))
        assert np.array_equal(sim.field("nown").astype(np.int64), nb.nown.astype(np.int64))
    assert 1 <= sim.list_rebuilds() <= steps
    sim.close()
