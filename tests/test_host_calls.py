"""The host side of the C ABI on a device that runs nothing (fake_runtime.cpp, fake_launches.cu):
what a call launches after an earlier one failed.  A failing launch, copy or
wait is a value the fake returns, so no GPU is needed or harmed."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1905_03344_gb300 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
OVERFLOW, NONFINITE, TIMEOUT = 1, 2, 4      # bits of the device status word


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = tmp_path_factory.mktemp("host_calls")
    objs = []
    jobs = []
    for src in (os.path.join(build.CSRC, "sph_api.cu"), os.path.join(HERE, "fake_launches.cu"),
                os.path.join(HERE, "fake_runtime.cpp")):
        objs.append(str(out / (os.path.basename(src) + ".o")))
        jobs.append(subprocess.Popen([build.nvcc()] + build.ARCH + ["-std=c++17", "-Xcompiler", "-fPIC",
                                      "--expt-relaxed-constexpr", "-I", build.CSRC, "-c", src, "-o", objs[-1]]))
    assert all(j.wait() == 0 for j in jobs)
    so = str(out / "libfake.so")
    # bound to its own symbols, whatever CUDA runtime the process has loaded
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so] + objs, check=True)
    L = ctypes.CDLL(so)
    for name, (res, args) in binding.SIGNATURES.items():
        if hasattr(L, name):
            getattr(L, name).restype, getattr(L, name).argtypes = res, args
    L.fake_log.restype = ctypes.c_char_p
    L.fake_alloc.restype, L.fake_alloc.argtypes = ctypes.c_void_p, [ctypes.c_size_t, ctypes.c_int]
    return L


class Fake:
    def __init__(self, lib, n=64, **kw):
        self.lib = lib
        lib.fake_reset(b"", 0, -1)
        cfg = binding.SphConfig()
        lib.sph_config_default(ctypes.byref(cfg))
        cfg.max_particles = n
        for k, v in kw.items():
            setattr(cfg, k, v)
        self.ctx = ctypes.c_void_p()
        assert lib.sph_create(ctypes.byref(cfg), ctypes.byref(self.ctx)) == binding.SPH_OK

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.lib.sph_destroy(self.ctx)

    def expect(self, status_at="", bits=0, copies_left=-1):
        """Clears the log; the launch of that name will report bits."""
        self.lib.fake_reset(status_at.encode(), bits, copies_left)

    def log(self):
        return self.lib.fake_log().decode().split()

    def set_particles(self, n, ptrs=None, on_device=0):
        if ptrs is None:
            self.buf = np.ones((9, n))
            ptrs = [self.buf[k].ctypes.data for k in range(9)]
        return self.lib.sph_set_particles(self.ctx, n, *ptrs, on_device)

    def step(self, n=1):
        return self.lib.sph_step(self.ctx, n, None)


def test_bins_of_a_failed_call_are_not_used(lib):
    """A binning pass that gave up leaves its order unwritten; the next sum
    bins again instead of reading it."""
    with Fake(lib, pair_bins=32) as f:
        assert f.set_particles(40) == binding.SPH_OK
        assert lib.sph_find_neighbors(f.ctx) == binding.SPH_OK
        f.expect("bins", TIMEOUT)
        assert lib.sph_density(f.ctx) == binding.SPH_ETIMEOUT
        assert f.log() == ["bins", "density_binned"]
        f.expect()
        assert lib.sph_density(f.ctx) == binding.SPH_OK
        assert f.log() == ["bins", "density_binned"]
        assert lib.sph_momentum_energy(f.ctx) == binding.SPH_OK
        assert f.log() == ["bins", "density_binned", "momentum_binned"]     # the same bins


@pytest.mark.parametrize("failing", ["sort", "superset", "filter"])
def test_superset_of_a_failed_step_is_not_used(lib, failing):
    """A step that fails may leave its candidate superset incomplete, with rows
    outside the pool; no particle moves, so the check that follows every step
    finds that the superset would still hold."""
    with Fake(lib, list_skin=0.2) as f:
        assert f.set_particles(40) == binding.SPH_OK
        f.expect(failing, TIMEOUT if failing == "sort" else OVERFLOW)
        assert f.step() == (binding.SPH_ETIMEOUT if failing == "sort" else binding.SPH_EOVERFLOW)
        f.expect()
        assert f.step() == binding.SPH_OK
        assert "superset" in f.log()
        f.expect()
        assert f.step() == binding.SPH_OK       # while a good one is used again
        assert "superset" not in f.log() and "filter" in f.log()


@pytest.mark.parametrize("copies", [0, 4])
def test_failed_upload_leaves_the_particle_count(lib, copies):
    """The patch tables are sized by the particle count: an upload that fails
    changes neither."""
    with Fake(lib) as f:
        assert f.set_particles(24) == binding.SPH_OK
        f.expect(copies_left=copies)
        assert f.set_particles(40) == binding.SPH_ECUDA
        f.expect()
        f.step()        # (the runtime's last error is the copy's)
        assert f.log()[:2] == ["items=24", "keys=24"]


@pytest.mark.parametrize("where", ["here", "peer", "host"])
def test_kernels_take_only_this_devices_memory(lib, where):
    """on_device pointers are handed to a kernel where they are this device's
    memory.  Another device's is copied, as the runtime does between any two,
    and a host pointer is refused by the copy."""
    n = 32
    with Fake(lib) as f:
        def buf(k):
            if where == "host":
                f.keep = getattr(f, "keep", []) + [np.ones(k)]
                return f.keep[-1].ctypes.data
            return lib.fake_alloc(8 * k, 0 if where == "here" else 1)
        ptrs = [buf(n) for _ in range(9)]
        f.expect()
        st = f.set_particles(n, ptrs, 1)
        if where == "here":
            assert st == binding.SPH_OK and f.log() == ["load_direct"]
        elif where == "peer":
            assert st == binding.SPH_OK and f.log() == ["copy"] * 9 + ["load_own"]
        else:
            assert st == binding.SPH_ECUDA and f.log() == []
        assert f.set_particles(n) == (binding.SPH_ECUDA if where == "host" else binding.SPH_OK)
        assert lib.sph_find_neighbors(f.ctx) == binding.SPH_OK
        f.expect()
        st = lib.sph_copy_neighbors(f.ctx, buf(n + 1), buf(8), buf(n), 1)
        assert not [w for w in f.log() if w.endswith("elsewhere")]
        assert st == (binding.SPH_ECUDA if where == "host" else binding.SPH_OK)
