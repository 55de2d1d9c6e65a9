"""The ticket order of split regions on the CPU: every region has one ticket,
its predecessors (build_preds, csrc/planner.cpp) are those whose successor it
is, and all hold earlier tickets, so waits on them end whatever the grid."""
import ctypes
import os
import subprocess

import pytest

from conftest import ROOT


@pytest.fixture(scope="module")
def tx():
    here = os.path.dirname(os.path.abspath(__file__))
    csrc = os.path.join(ROOT, "paper_1011_4046_gb300", "csrc")
    lib = os.path.join(here, "cpu_exec", "_build", "libtx.so")
    os.makedirs(os.path.dirname(lib), exist_ok=True)
    srcs = [os.path.join(here, "cpu_exec", "ticket_exec.cpp"), os.path.join(csrc, "planner.cpp")]
    deps = srcs + [os.path.join(csrc, "planner.h")]
    if not os.path.exists(lib) or any(os.path.getmtime(f) > os.path.getmtime(lib) for f in deps):
        tmp = lib + f".tmp{os.getpid()}"
        subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-I{csrc}", *srcs, "-o", tmp], check=True)
        os.replace(tmp, lib)
    L = ctypes.CDLL(lib)
    L.tx_check.argtypes = [ctypes.c_int] * 7 + [ctypes.c_char_p, ctypes.c_int]
    return L


def _check(tx, B, J, bands, reuse, planted=0):
    msg = ctypes.create_string_buffer(256)
    return tx.tx_check(B, *J, bands, reuse, planted, msg, 256), msg.value.decode()


@pytest.mark.parametrize("reuse", [0, 1])
@pytest.mark.parametrize("J, bands", [((2, 2, 2), 5), ((3, 2, 4), 4), ((5, 5, 5), 3), ((2, 7, 3), 1)])
@pytest.mark.parametrize("B", [4, 8, 16])
def test_tickets_are_a_topological_order(tx, B, J, bands, reuse):
    rc, msg = _check(tx, B, J, bands, reuse)
    assert rc == 0, msg


@pytest.mark.parametrize("planted", [1, 2, 3])
def test_planted_mistakes_are_reported(tx, planted):
    assert _check(tx, 8, (5, 4, 3), 3, 1, planted)[0] == -1
