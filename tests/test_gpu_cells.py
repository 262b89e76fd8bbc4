"""The list search cell by cell, which more than 50,000 particles take in
patches whose h varies from cell to cell (use_cells): lattices with h graded
along x, so that the largest h around a cell is 1.1 to 1.7 times the cell's
own, alone and in a batch beside patches that are searched by rows.  Lists and
n_i against the oracle, bit for bit."""
import os

import numpy as np
import pytest

from paper_1905_03344_gb300 import inputs
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


def _graded(e, top, jitter=0.0, big=0):
    """A lattice of e^3 particles, h between 1.2 spacings and top times that,
    along x; every big-th particle's h doubled again."""
    rng = np.random.default_rng(e)
    dx, n = 1.0 / e, e ** 3
    g = (np.arange(e) + 0.5) * dx - 0.5
    z, y, x = (t.ravel().copy() for t in np.meshgrid(g, g, g, indexing="ij"))
    h = 1.2 * dx * (1.0 + (top - 1.0) * (0.5 + 0.5 * np.sin(6.0 * np.pi * x)) ** 2)
    for t in (x, y):
        t += rng.uniform(-jitter, jitter, n) * dx
    if big:
        h[::big] *= 2.0
    v = np.zeros(n)
    return {"x": x, "y": y, "z": z, "vx": v, "vy": v, "vz": v, "m": np.full(n, 1.0 / n), "h": h, "u": np.ones(n)}


def _neighbors(orc, parts):
    """The oracle's lists of independent patches, as of one particle set."""
    nb = [orc.neighbors(p["x"], p["y"], p["z"], p["h"], 1.0, nthreads=os.cpu_count() or 1) for p in parts]
    n0 = np.concatenate([[0], np.cumsum([len(p["x"]) for p in parts])])
    e0 = np.concatenate([[0], np.cumsum([q.off[-1] for q in nb])])
    off = np.concatenate([[0]] + [q.off[1:] + e for q, e in zip(nb, e0)])
    col = np.concatenate([q.col + k for q, k in zip(nb, n0)])
    return off, col, np.concatenate([q.nown for q in nb]), n0


def _check(sim, off, col, nown):
    o, c = lists_to_original(*sim.neighbors(), len(off) - 1)
    assert np.array_equal(o, off) and np.array_equal(c, col)
    assert np.array_equal(sim.field("nown").astype(np.int64), nown)


CASES = {"lattice": dict(top=2.0), "steep": dict(top=3.0), "jittered": dict(top=2.0, jitter=0.1, big=501)}


@pytest.mark.parametrize("cf", [0.0, 0.4, 0.75, 1.0])       # stencils of 2, 3, 2 and 1 cells
@pytest.mark.parametrize("case", sorted(CASES))
def test_graded_patch(B, orc, case, cf):
    f = _graded(38, **CASES[case])
    n = len(f["x"])
    off, col, nown, _ = _neighbors(orc, [f])
    sim = B.SPH(n, cell_factor=cf, max_pairs=800 * n)      # 614 entries a particle in "steep"
    sim.set_particles(f)
    for _ in range(2):           # rows counted first, then reserved from hints
        sim.find_neighbors()
        _check(sim, off, col, nown)
    sim.close()


@pytest.mark.parametrize("skin", [0.0, 0.2])
def test_batch_of_both_kinds(B, orc, skin):
    parts = [_graded(29, 2.0, 0.1, 301), inputs.square_patch(24), inputs.random_cloud(6000, seed=5, h_lo=0.05, h_hi=0.06),
             _graded(8, 2.5), inputs.square_patch(3), _graded(21, 3.0)]
    f = {k: np.concatenate([p[k] for p in parts]) for k in parts[0]}
    off, col, nown, offsets = _neighbors(orc, parts)
    n = len(f["x"])
    assert n > 50000
    sim = B.SPH(n, max_patches=len(parts), max_pairs=400 * n, list_skin=skin)
    sim.set_particles(f)
    sim.set_patches(offsets)
    for _ in range(2):
        sim.find_neighbors()
        _check(sim, off, col, nown)
    sim.close()
