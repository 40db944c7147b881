"""What the library's host side launches, seen through a runtime that records
launches instead of running them (tests/_fake_cudart.cpp, linked with the
library's own objects)."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
STORAGE = {"fp64": 0, "fp32": 1, "fp16s": 2, "bf16s": 3}


@pytest.fixture()
def lib(tmp_path):
    """A fresh copy of the library (its own process-wide state) on the fake
    runtime."""
    from paper_1202_6130_gb300 import _lib, build as b
    b.build()
    so = str(tmp_path / "liblbm_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b._nvcc()))), "include")
    # -Bsymbolic: the fake, not a CUDA runtime that torch loaded into this process
    subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-O1", "-I" + inc, "-o", so,
                    os.path.join(HERE, "_fake_cudart.cpp"), *sorted(glob.glob(os.path.join(b.OBJ, "*.o"))),
                    "-Wl,-Bsymbolic", "-Wl,-z,defs", "-lpthread"], check=True)
    lib = ctypes.CDLL(so)
    for name, (res, args) in _lib.SIGNATURES.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    lib.fake_launch.restype = ctypes.c_char_p
    return lib


def _ctx(lib, nx, ny, lattice, storage):
    from paper_1202_6130_gb300 import _lib
    p = _lib.lbm_params()
    assert lib.lbm_params_default(ctypes.byref(p)) == 0
    p.nx, p.ny, p.lattice, p.storage, p.shift_rho = nx, ny, lattice, STORAGE[storage], 1.0
    ctx = ctypes.c_void_p()
    rc = lib.lbm_create(ctypes.byref(p), None, None, ctypes.byref(ctx))
    assert rc == 0, lib.lbm_last_error(None)
    rho = np.ones((ny, nx))
    zero = np.zeros((ny, nx))
    assert lib.lbm_set_equilibrium(ctx, _lib.dptr(rho), _lib.dptr(zero), _lib.dptr(zero), None) == 0
    return ctx


def _launches(lib, first=0):
    """(kernel name, device, grid x, grid y, dynamic shared memory) of each launch."""
    out = []
    for i in range(first, lib.fake_launches()):
        v = [ctypes.c_int() for _ in range(4)]
        out.append((lib.fake_launch(i, *(ctypes.byref(x) for x in v)).decode(), *(x.value for x in v)))
    return out


@pytest.mark.parametrize("lattice,storage", [(9, "fp64"), (9, "fp32"), (9, "fp16s"), (21, "fp32"),
                                             (21, "fp64"), (21, "bf16s")])
def test_a_second_device_of_the_process_runs_every_kernel(lib, lattice, storage):
    """A kernel with more than 48 KB of dynamic shared memory is launched only on
    devices on which its limit was raised: the same calls on device 0, then on
    device 1, for sizes that take different tile shapes, and for batches on
    tiles, on a march and on persistent CTAs."""
    from paper_1202_6130_gb300 import _lib
    for device in (0, 1):
        lib.fake_set_device(device)
        for nx, ny in ((130, 70), (1024, 512), (4096, 1024)):
            first = lib.fake_launches()
            ctx = _ctx(lib, nx, ny, lattice, storage)
            assert lib.lbm_step(ctx, 3) == 0, (device, nx, lib.lbm_last_error(ctx))
            d = np.empty((3, ny, nx))
            assert lib.lbm_moments_device(ctx, *(d[i].ctypes.data for i in range(3))) == 0, (device, nx)
            batch = ctypes.c_void_p()
            assert lib.lbm_batch_create(None, None, ctypes.byref(batch)) == 0
            assert lib.lbm_batch_add(batch, ctx) == 0
            for tiling in ((0, 0), (16, 0), (16, 300)):
                assert lib.lbm_batch_set_tiling(batch, *tiling) == 0
                assert lib.lbm_batch_step(batch, 1) == 0, (device, nx, tiling)
            assert lib.lbm_batch_destroy(batch) == 0 and lib.lbm_destroy(ctx) == 0
            assert {l[1] for l in _launches(lib, first)} == {device}
    big = [l for l in _launches(lib) if l[4] > 48 * 1024]
    assert not big or {l[1] for l in big} == {0, 1}


@pytest.mark.parametrize("lattice,storage", [(9, "fp32"), (9, "fp16s"), (9, "fp64"), (21, "fp32")])
@pytest.mark.parametrize("fast", ["batch_tile_kernel", "Lb0ELi1EEEv", "Lb1ELi1EEEv"],
                         ids=["tiles", "march", "persistent"])
def test_autotune_reports_a_tiling_that_can_be_set(lib, lattice, storage, fast):
    """Whichever kernel is the fastest -- tiles, a row march, a march by persistent
    CTAs -- the pair that autotuning reports selects that kernel on another batch
    of such members, and a batch that adopts the tuned tiling runs it as well."""
    def batch():
        b = ctypes.c_void_p()
        assert lib.lbm_batch_create(None, None, ctypes.byref(b)) == 0
        for nx, ny in ((130, 70), (64, 32), (257, 90)):
            assert lib.lbm_batch_add(b, _ctx(lib, nx, ny, lattice, storage)) == 0
        return b

    def step(b):
        assert lib.lbm_batch_step(b, 1) == 0
        return _launches(lib, lib.fake_launches() - 1)[0]

    lib.fake_set_fast(fast.encode())
    b = batch()
    rows, ctas, ms = ctypes.c_int32(), ctypes.c_int32(), ctypes.c_double()
    assert lib.lbm_batch_autotune(b, 4, ctypes.byref(rows), ctypes.byref(ctas), ctypes.byref(ms)) == 0
    want = step(b)
    assert fast in want[0] and ms.value == 1.0 and rows.value > 0
    again = batch()
    assert lib.lbm_batch_set_tiling(again, rows, ctas) == 0
    assert step(again) == want
    adopts = batch()
    found = ctypes.c_int32()
    assert lib.lbm_batch_use_tuned(adopts, ctypes.byref(found)) == 0 and found.value == 1
    assert step(adopts) == want
