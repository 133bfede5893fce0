"""The library's host code against a stand-in for the CUDA runtime (no GPU):
what calls launch, within which grids, and what they leave behind when a launch
fails."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1603_08221_gb300 import binding, build, workloads

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no nvcc")
    out = tmp_path_factory.mktemp("fake") / "liblbm_fake.so"
    # PTX only and unoptimised: the device code is never run; its own runtime, not
    # one that the process has loaded
    subprocess.run([build.nvcc(), "-gencode", "arch=compute_103a,code=compute_103a",
                    "-Xcicc", "-O0", "-std=c++17", "-Xcompiler", "-fPIC", "-cudart", "none",
                    "-Xlinker", "-Bsymbolic", "-shared", build.SRC,
                    os.path.join(HERE, "fake_cudart.c"), "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    for name, (res, args) in binding._SIGS.items():
        if not name.startswith("lbm_adj"):
            fn = getattr(lib, name)
            fn.restype, fn.argtypes = res, args
    lib.fake_launch.restype = ctypes.c_char_p
    return lib


def _params(lib, **kw):
    p = binding.lbm_mix_params()
    lib.lbm_mix_default_params(ctypes.byref(p))
    for k, v in workloads.preset("heli_argon_320x16", **kw).items():
        setattr(p, k, v)
    return p


def _launches(lib):
    grid = (ctypes.c_uint * 3)()
    out = []
    for k in range(lib.fake_launches()):
        name = lib.fake_launch(k, grid).decode()
        out.append((name, tuple(grid)))
    return out


class Handle:
    def __init__(self, lib, **kw):
        self.lib, p = lib, _params(lib, **kw)
        h = ctypes.c_void_p()
        assert lib.lbm_mix_create(ctypes.byref(p), None, ctypes.byref(h)) == 0
        self.h = h
        assert lib.lbm_mix_init(h) == 0

    def __enter__(self):
        return self.h

    def __exit__(self, *exc):
        self.lib.lbm_mix_destroy(self.h)


def _steps(lib, h):
    n, nx, steps = ctypes.c_int(), ctypes.c_int(), ctypes.c_long()
    assert lib.lbm_mix_dims(h, ctypes.byref(n), ctypes.byref(nx), ctypes.byref(steps)) == 0
    return steps.value


# channels whose sweep takes batched step kernels with and without the wall
# kernel ahead of them, and tiles with their records
@pytest.mark.parametrize("count,N,Nx", [(1, 600, 100), (40, 600, 100), (12, 600, 3000),
                                        (3, 20, 600)])
def test_a_failed_launch_of_a_sweep_leaves_no_step_behind(fake, count, N, Nx):
    """Steps are counted, and the buffers change places, where their launch was
    accepted: after a failure at the k-th launch of a call every handle has taken
    the steps of the launches before it."""
    lib = fake
    ps = (binding.lbm_mix_params * count)(*[_params(lib, N=N, N_x=Nx) for _ in range(count)])
    for fail in (0, 1):
        s = ctypes.c_void_p()
        assert lib.lbm_sweep_create(ps, count, ctypes.byref(s)) == 0
        assert lib.lbm_sweep_init(s) == 0
        lib.fake_reset()
        lib.fake_fail(fail)
        status = lib.lbm_sweep_step(s, 1)
        log = _launches(lib)
        lib.fake_reset()
        if fail >= len(log):
            assert status == 0
            lib.lbm_sweep_destroy(s)
            continue
        assert status == binding.LBM_ECUDA
        accepted = [n for n, _ in log[:fail]]
        h = ctypes.c_void_p()
        taken = 0
        for k in range(count):
            assert lib.lbm_sweep_instance(s, k, ctypes.byref(h)) == 0
            taken += _steps(lib, h)
        # a launch of steps holds 32 channels of the step kernel at most, all of
        # these tiles
        most = sum(min(32, count) if "step_batch" in n else count if "tile" in n else 0
                   for n in accepted)
        assert taken == most, (fail, log)
        lib.lbm_sweep_destroy(s)


# the tallest channels that validate takes (18 N pitch below 2^31), and one row
# either side of 65535 blocks of the 56 rows that FP32 row blocks have at most
@pytest.mark.parametrize("N", [56 * 65535, 56 * 65535 + 1, 3728000])
@pytest.mark.parametrize("storage", [binding.LBM_FP32, binding.LBM_BF16])
def test_grids_of_the_tallest_channels(fake, N, storage):
    """A grid has 65535 blocks in y at most."""
    lib = fake
    with Handle(lib, N=N, N_x=8, storage=storage, diag_every=2) as h:
        lib.fake_reset()
        assert lib.lbm_mix_step(h, 3) == 0
        rows = [g[1] for n, g in _launches(lib) if "lbm_step_kernel" in n]
        assert len(rows) == 3 and max(rows) <= 65535


# tiles with records of their own and in common, single steps of wide channels,
# the step kernel with and without the wall kernel, 16-bit storage,
# re-referencing in between
@pytest.mark.parametrize("kw", [dict(N=16, N_x=320), dict(N=16, N_x=320, diag_every=1),
                                dict(N=16, N_x=320, reref_every=7),
                                dict(N=16, N_x=8000, diag_every=4),
                                dict(N=600, N_x=100), dict(N=512, N_x=32768),
                                dict(N=130, N_x=5001, storage=binding.LBM_BF16, reref_every=5)])
def test_launches_are_counted(fake, kw):
    lib = fake
    with Handle(lib, **kw) as h:
        lib.fake_reset()
        base = lib.lbm_mix_launches(h)
        for n in (1, 2, 3, 16, 400):
            assert lib.lbm_mix_step(h, n) == 0
            assert lib.lbm_mix_launches(h) - base == lib.fake_launches(), n
        if kw == dict(N=16, N_x=320):
            assert lib.fake_launches() < 422 / 4  # several steps a launch
