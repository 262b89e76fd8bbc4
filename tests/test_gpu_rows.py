"""The search over rows of cells where its runs can go wrong: rows of 128
cells (x far from the grid's origin), particles on cell faces, cells of many
particles, rows of one cell, and few z cells -- lists and n_i against the
oracle, bit for bit."""
import os

import numpy as np
import pytest

from gpu_common import lists_to_original

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_03344_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _cloud(kind, n):
    rng = np.random.default_rng(11)
    z = rng.uniform(-0.5, 0.5, n)
    if kind == "long_x":         # 128 cells along x, few along y
        x, y, h = rng.uniform(0.0, 12.0, n), rng.uniform(-0.1, 0.1, n), rng.uniform(0.03, 0.045, n)
    elif kind == "long_y":       # rows of few cells
        x, y, h = rng.uniform(-0.1, 0.1, n), rng.uniform(0.0, 12.0, n), rng.uniform(0.03, 0.045, n)
    elif kind == "faces":        # coordinates on a lattice of multiples of the cell edge and of ties at 2 h
        k = rng.integers(0, 24, (3, n))
        x, y, z = k[0] / 32.0, k[1] / 32.0, (k[2] % 16) / 16.0 - 0.5
        h = np.where(rng.random(n) < 0.5, 1.0 / 32.0, 3.0 / 64.0)
    elif kind == "clump":        # a cell of several hundred particles among sparse ones
        x, y = rng.uniform(-1.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
        x[:400], y[:400], z[:400] = (rng.normal(c, 0.004, 400) for c in (0.2, -0.3, 0.1))
        h = rng.uniform(0.05, 0.07, n)
    elif kind == "big_reach":    # a few particles whose radius spans many rows and the z period
        x, y = rng.uniform(-0.5, 0.5, n), rng.uniform(-0.5, 0.5, n)
        h = rng.uniform(0.03, 0.04, n)
        h[::97] = rng.uniform(0.15, 0.3, len(h[::97]))
    else:                        # few_z: h so large that every z cell is visited
        x, y, h = rng.uniform(-2.0, 2.0, n), rng.uniform(-2.0, 2.0, n), rng.uniform(0.14, 0.17, n)
    if kind not in ("faces", "few_z"):
        h = h * (6000.0 / n) ** (1.0 / 3.0)
    v = np.zeros(n)
    return {"x": x, "y": y, "z": z, "vx": v, "vy": v, "vz": v, "m": np.full(n, 1.0 / n), "h": h, "u": np.ones(n)}


# 6000 particles are searched by teams of lanes, 56000 by a thread each
@pytest.mark.parametrize("n,cf", [(6000, 0.0), (6000, 0.4), (6000, 1.0), (56000, 0.0), (56000, 0.4)])
@pytest.mark.parametrize("kind", ["long_x", "long_y", "faces", "clump", "big_reach", "few_z"])
def test_rows(B, orc, kind, n, cf):
    f = _cloud(kind, n)
    sim = B.SPH(n, cell_factor=cf, max_pairs=800 * n)
    sim.set_particles(f)
    nb = None
    for _ in range(2):           # rows counted first, then reserved from hints
        sim.find_neighbors()
        off, col, perm = sim.neighbors()
        o, c = lists_to_original(off, col, perm, n)
        nb = nb or orc.neighbors(f["x"], f["y"], f["z"], f["h"], 1.0, nthreads=os.cpu_count() or 1)
        assert np.array_equal(o, nb.off) and np.array_equal(c, nb.col)
        assert np.array_equal(sim.field("nown").astype(np.int64), nb.nown)
    sim.close()


def _layers(kind, e):
    """A lattice of e^3 particles whose rows are pruned by where their particles lie."""
    rng = np.random.default_rng(5)
    dx, n = 1.0 / e, e ** 3
    g = (np.arange(e) + 0.5) * dx - 0.5
    z, y, x = (t.ravel().copy() for t in np.meshgrid(g, g, g, indexing="ij"))
    h = np.full(n, 1.44 * dx)
    if kind == "sheared":        # layers along z, rows at an angle to y
        y += 0.3 * x
    elif kind == "jittered":     # with particles whose radius outgrows the stencil
        for t in (x, y):
            t += rng.uniform(-0.1, 0.1, n) * dx
        h *= rng.uniform(0.9, 1.1, n)
        h[::101] *= rng.uniform(2.0, 4.0, len(h[::101]))
    elif kind == "periodic":     # layers on the period's ends, gaps between them
        z = np.floor((z + 0.5) * e / 3.0) * 3.0 * dx - 0.5
        x += rng.uniform(-0.3, 0.3, n) * dx
    v = np.zeros(n)
    return {"x": x, "y": y, "z": z, "vx": v, "vy": v, "vz": v, "m": np.full(n, 1.0 / n), "h": h, "u": np.ones(n)}


@pytest.mark.parametrize("e,cf", [(18, 0.0), (18, 0.4), (37, 0.0), (37, 0.4), (37, 1.0)])
@pytest.mark.parametrize("kind", ["lattice", "sheared", "jittered", "periodic"])
def test_layers(B, orc, kind, e, cf):
    f = _layers(kind, e)
    n = e ** 3
    sim = B.SPH(n, cell_factor=cf, max_pairs=800 * n)
    sim.set_particles(f)
    nb = orc.neighbors(f["x"], f["y"], f["z"], f["h"], 1.0, nthreads=os.cpu_count() or 1)
    for _ in range(2):
        sim.find_neighbors()
        off, col, perm = sim.neighbors()
        o, c = lists_to_original(off, col, perm, n)
        assert np.array_equal(o, nb.off) and np.array_equal(c, nb.col)
        assert np.array_equal(sim.field("nown").astype(np.int64), nb.nown)
    sim.close()
