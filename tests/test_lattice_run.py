"""The lists that the lattice kernels read (imp_run, cell_wide; csrc/lattice.cpp)
executed on the CPU (cpu_exec/lattice_run_exec.cpp): equal to the whole-grid
sweep bit for bit, with values that no level may read poisoned, and every kind
of wrong entry reported."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import test_lattice as base
from conftest import ROOT


@pytest.fixture(scope="module")
def lxr():
    here = os.path.dirname(os.path.abspath(__file__))
    csrc = os.path.join(ROOT, "paper_1011_4046_gb300", "csrc")
    lib = os.path.join(here, "cpu_exec", "_build", "liblxr.so")
    os.makedirs(os.path.dirname(lib), exist_ok=True)
    srcs = [os.path.join(here, "cpu_exec", "lattice_run_exec.cpp"), os.path.join(csrc, "lattice.cpp")]
    deps = srcs + [os.path.join(csrc, "lattice.h"), os.path.join(csrc, "sp_update.h")]
    if not os.path.exists(lib) or any(os.path.getmtime(f) > os.path.getmtime(lib) for f in deps):
        tmp = lib + f".tmp{os.getpid()}"
        subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", f"-I{csrc}", *srcs, "-o", tmp],
                       check=True)
        os.replace(tmp, lib)
    L = ctypes.CDLL(lib)
    fp = ctypes.POINTER(ctypes.c_float)
    L.lxr_run.argtypes = ([ctypes.c_int] * 6 + [ctypes.c_uint64, ctypes.c_int, ctypes.c_int, fp] + [ctypes.c_float] * 3 +
                          [fp, fp, ctypes.c_char_p, ctypes.c_int])
    return L


def _run(lxr, s, n, steps, mode, aligned, planted, phi0, pc0, coef):
    fp = ctypes.POINTER(ctypes.c_float)
    f, p = phi0.copy(), pc0.copy()
    msg = ctypes.create_string_buffer(256)
    rc = lxr.lxr_run(s, *n, steps, mode, 5, aligned, planted, coef.ctypes.data_as(fp), 0.25, 1.0, 1.0,
                     f.view(np.float32).ctypes.data_as(fp), p.ctypes.data_as(fp), msg, 256)
    return rc, msg.value.decode(), f, p


@pytest.mark.parametrize("s,n,steps", [
    (1, (4, 4, 4), 7), (1, (8, 4, 12), 9), (2, (16, 8, 24), 21), (2, (16, 16, 16), 1), (3, (12, 24, 12), 14),
    (4, (16, 16, 16), 19), (4, (32, 16, 16), 40), (4, (16, 32, 16), 3), (5, (20, 40, 20), 23), (5, (20, 20, 20), 2),
    (6, (24, 24, 24), 26),
])
def test_kernel_lists_equal_the_sweep(lx, lxr, s, n, steps):
    phi0, pc0 = base._state(n, 7 + s)
    coef = base._coef_table(steps, 2.0, 0.25, 2.0, 10.0, 10.0 + steps * 0.25)
    ref_f, ref_p = base._sweep(lx, n, steps, phi0, pc0, coef)
    for mode, aligned in ((0, 1), (1, 1), (1, 0)):
        rc, msg, f, p = _run(lxr, s, n, steps, mode, aligned, 0, phi0, pc0, coef)
        assert rc == 0, msg
        assert np.array_equal(f.view(np.uint32), ref_f.view(np.uint32))
        assert np.array_equal(p.view(np.uint32), ref_p.view(np.uint32))


@pytest.mark.parametrize("planted", range(1, 14))
@pytest.mark.parametrize("s,n,steps", [(2, (8, 16, 8), 13), (4, (16, 16, 16), 21), (6, (24, 24, 24), 27)])
def test_wrong_entries_are_reported(lxr, s, n, steps, planted):
    """Each field of the lists that a kernel decodes, wrong in every entry
    that has it: the run is refused, or (rc 1) the size has no such field."""
    phi0, pc0 = base._state(n, 3)
    coef = base._coef_table(steps, 0.0, 0.25, 2.0, 1.0, 1.0)
    absent = (s == 2 and planted in (1, 2)) or (s == 6 and planted >= 9)
    for aligned in (1, 0):
        if planted == 8 and not aligned:
            continue  # no pair copies where phi is off 16 bytes
        if planted == 1 and aligned:
            continue  # an aligned pair arrives as one copy by the pair bit alone
        rc, msg, _, _ = _run(lxr, s, n, steps, 0, aligned, planted, phi0, pc0, coef)
        assert rc == (1 if absent else -1), (rc, msg)
