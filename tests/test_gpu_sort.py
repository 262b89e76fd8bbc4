"""The radix sort at the edges of its tiles: one key, a tile less or more one,
the change from small to large tiles, many patches (a fourth digit), and a
second search of the same particles -- the order is the stable order of the
cell keys: per patch, a permutation whose cells are contiguous, with the
particles of a cell in the order they had."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_03344_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _grid_fields(n, seed):
    """Particles on the centres of a 16^3 grid, several to a centre, with a
    neighbour radius below the distance of the centres."""
    rng = np.random.default_rng(seed)
    k = rng.integers(0, 16, (3, n))
    x, y, z = ((k[q] + 0.5) / 16.0 - 0.5 for q in range(3))
    v = np.zeros(n)
    return {"x": x, "y": y, "z": z, "vx": v, "vy": v, "vz": v, "m": np.full(n, 1.0 / n),
            "h": np.full(n, 1.0 / 128.0), "u": np.ones(n)}


def _check(f, perm, offs):
    n = len(perm)
    assert np.array_equal(np.sort(perm), np.arange(n))
    cell = np.stack([f[q][perm] for q in ("x", "y", "z")], axis=1)
    for b, e in zip(offs[:-1], offs[1:]):
        if e - b < 1:
            continue
        assert perm[b:e].min() >= b and perm[b:e].max() < e
        c = cell[b:e]
        new = np.any(c[1:] != c[:-1], axis=1)
        # a centre's particles are one run, in their original order
        assert new.sum() + 1 == len(np.unique(c, axis=0))
        assert np.all(np.diff(perm[b:e])[~new] > 0)


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 40961, 622592, 622593, 625665])
def test_sort_edges(B, n):
    f = _grid_fields(n, 3)
    if n > 40961:                # more centres, so that the lists stay short
        rng = np.random.default_rng(5)
        k = rng.integers(0, 48, (3, n))
        f.update({q: (k[i] + 0.5) / 48.0 - 0.5 for i, q in enumerate(("x", "y", "z"))}, h=np.full(n, 1.0 / 384.0))
    sim = B.SPH(n, max_pairs=max(64, 40 * n))
    sim.set_particles(f)
    sim.find_neighbors()
    _, _, perm = sim.neighbors()
    _check(f, perm, [0, n])
    sim.find_neighbors()
    assert np.array_equal(sim.neighbors()[2], perm)   # sorted already: stable
    sim.close()


def test_sort_patches(B):
    offs = np.array([0, 5, 5, 1029, 2053, 9000, 9001, 20000])
    f = _grid_fields(20000, 7)
    sim = B.SPH(20000, max_patches=200, max_pairs=40 * 20000)
    sim.set_particles(f)
    sim.set_patches(np.concatenate([offs, np.full(100, 20000)]))
    sim.find_neighbors()
    _check(f, sim.neighbors()[2], offs)
    sim.close()
