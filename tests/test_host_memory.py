"""Device memory that the library takes to be faster (the second (pi, c) copy
of two-level sweeps) never stands in the way of what a later call needs: on a
device of a given size (cpu_exec/fake_cudart.cpp) a sweep is followed by a
plan, by a diagnostic surface and by another sweep."""
import ctypes

import numpy as np
import pytest

import fake_cuda
from paper_1011_4046_gb300 import sp

N = 160
SITES = N ** 3
STATE, PHI, COPY = 24 * SITES, 8 * SITES, 16 * SITES
TIGHT = (STATE + PHI + COPY) * 16 // 15 + (1 << 20)  # a sixteenth stays free beside all three
ROOMY = 16 * COPY + (1 << 20)


class Device:
    def __init__(self, capacity):
        self.lib = fake_cuda.load()
        self.lib.fake_reset(capacity, 0, 0)
        self.before = self.lib.fake_used()
        self.h = ctypes.c_void_p()
        p = sp.make_params(N, nu=2.0, tau0=10.0, tau_ref=20.0)
        assert self.lib.sp_grid_create(ctypes.byref(p), 1, None, 16, ctypes.byref(self.h)) == sp.SP_OK

    def sweep(self, flags=0, steps=4):
        assert self.lib.sp_evolve(self.h, steps, sp.SP_MONOLITHIC | sp.SP_RESTART | flags) == sp.SP_OK

    def plan(self, shape):
        assert self.lib.sp_set_option(self.h, sp.SP_OPT_REGION_SHAPE, shape) == sp.SP_OK
        return self.lib.sp_region_plan(self.h, 16, 0, 0, None)

    def used(self):
        return self.lib.fake_used() - self.before

    def close(self):
        if self.h:
            assert self.lib.sp_destroy(self.h) == sp.SP_OK
            self.h = None
            assert self.used() == 0


@pytest.fixture
def device():
    made = []

    def make(capacity):
        made.append(Device(capacity))
        return made[-1]

    yield make
    for d in made:
        d.close()


def test_large_copy_lasts_for_the_call(device):
    d = device(TIGHT)
    d.sweep()
    assert d.lib.fake_peak() - d.before > STATE + PHI + COPY  # two levels at a time
    assert d.used() < STATE + PHI + COPY // 8


@pytest.mark.parametrize("shape", [sp.SP_SHAPE_LATTICE, sp.SP_SHAPE_SPLIT])
@pytest.mark.parametrize("flags", [0, sp.SP_ASYNC])
def test_plan_after_sweep(device, shape, flags):
    need = device(1 << 40)
    assert need.plan(shape) == sp.SP_OK
    mailboxes = need.used() - STATE
    need.close()
    d = device(max(TIGHT, STATE + PHI + mailboxes + (1 << 20)))  # room for the plan, or just for the sweep
    d.sweep(flags)
    assert d.plan(shape) == sp.SP_OK
    assert d.used() < STATE + PHI + mailboxes + (1 << 20)
    d.sweep(flags)


def test_surface_after_sweep(device):
    d = device(TIGHT)
    d.sweep(sp.SP_ASYNC)
    assert d.used() > STATE + PHI + COPY
    d.lib.fake_set_capacity(d.lib.fake_used() + (1 << 20))  # someone else took the rest
    out = np.empty(3 * SITES, np.int8)
    assert d.lib.sp_read_surface(d.h, 0, sp.SP_SURF_WINDING, out.ctypes.data, out.nbytes, 0) == sp.SP_OK
    assert d.used() < STATE + PHI + COPY


def test_small_copy_is_kept_until_a_plan(device):
    d = device(ROOMY)
    d.sweep()
    kept = d.used()
    assert kept > STATE + PHI + COPY
    d.sweep()
    d.sweep(steps=5)
    assert d.used() < kept + (1 << 16)
    assert d.plan(sp.SP_SHAPE_LATTICE) == sp.SP_OK
    assert d.used() < STATE + 2 * PHI + COPY // 2
