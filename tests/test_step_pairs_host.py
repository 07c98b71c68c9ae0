"""Host-side decision of running steps in pairs (LBM_OPT_STEPS_PER_PASS), without a GPU."""
import ctypes
import inspect

import pytest

import bench
from paper_1803_04937_gb300 import _lib

F32, F16S = _lib.F32, _lib.F16S


class _Handle:
    """A handle with options, as Simulation has them, without device memory."""

    def __init__(self, shape, stencil=19, precision=F32, options=()):
        self.lib = _lib.load(build_if_missing=True)
        self.h = ctypes.c_void_p()
        assert self.lib.lbm_create(*shape, stencil, 0, 0, 0.8, precision, ctypes.byref(self.h)) == 0
        for key, value in options:
            assert self.lib.lbm_set_option(self.h, key, float(value)) == 0

    def __del__(self):
        self.lib.lbm_destroy(self.h)

    def option(self, key):
        v = ctypes.c_double()
        assert self.lib.lbm_get_option(self.h, key, ctypes.byref(v)) == 0
        return v.value


@pytest.mark.parametrize("n", [96, 110, 120, 127, 128, 256])
def test_bench_states_the_librarys_decision(n):
    sim = _Handle((n, n, n))
    passes = bench.steps_per_pass(sim)
    assert passes == sim.option(_lib.OPT_STEPS_PER_PASS) == (1 if n < 110 else 2)  # 2 x 76 n^3 bytes from 200 MB on
    assert bench.step_launches(passes, 23) == (23 if passes == 1 else 5 * 2 + 3)
    assert list(inspect.signature(bench.steps_per_pass).parameters) == ["sim"]  # no rule of its own


@pytest.mark.parametrize("kw", [dict(precision=F16S), dict(options=[(_lib.OPT_PATTERN, _lib.PATTERN_AA)]),
                                dict(options=[(_lib.OPT_CELLS_X, 2)]), dict(options=[(_lib.OPT_STEP_PAIRS, 0)]),
                                dict(options=[(_lib.OPT_WALLS_X, 1)])])
def test_forms_that_step_singly(kw):
    assert _Handle((256, 256, 256), **kw).option(_lib.OPT_STEPS_PER_PASS) == 1


def test_the_decision_is_read_only():
    sim = _Handle((8, 8, 8))
    assert sim.lib.lbm_set_option(sim.h, _lib.OPT_STEPS_PER_PASS, 2.0) == _lib.LBM_EINVAL
    assert b"read only" in sim.lib.lbm_last_error(sim.h)


# nx, ny, nz; whether LBM_OPT_STEP_PAIRS = 2 may run pairs: planes of 2^30 cells (32-bit byte offsets), edges of which
# three do not fit an int, more tile rows (22 rows each, D3Q27 14) than a grid may have
@pytest.mark.parametrize("shape,stencil,passes", [
    ((32768, 32767, 1), 19, 2), ((32768, 32768, 1), 19, 1), ((32768, 33000, 1), 19, 1), ((40000, 30000, 1), 19, 1),
    ((1 << 29, 1, 2), 19, 2), ((720000000, 1, 1), 19, 1), ((1, 720000000, 1), 19, 1),
    ((2, 22 * 65535, 3), 19, 2), ((2, 22 * 65535 + 1, 3), 19, 1), ((2, 14 * 65535, 3), 27, 2),
    ((2, 14 * 65535 + 1, 3), 27, 1), ((1, 1, 1), 19, 2)])
def test_lattices_that_pairs_cannot_address_step_singly(shape, stencil, passes):
    assert _Handle(shape, stencil, options=[(_lib.OPT_STEP_PAIRS, 2)]).option(_lib.OPT_STEPS_PER_PASS) == passes


def test_offsets_of_the_largest_lattices_that_run_in_pairs():
    """The kernel's coordinates and byte offsets, in Python: within int and unsigned for what the rule lets through."""
    for nx, ny in ((32768, 32767), (1 << 29, 1), (1, 1 << 29), (1 << 15, (1 << 15) - 1)):
        assert nx * ny < 1 << 30
        assert (nx + 30) + 2 * nx < 1 << 31 and (ny + 30) + 2 * ny < 1 << 31  # (xr - 1 + i + 2 nx), yr alike
        assert 4 * (nx * ny - 1) < 1 << 32                                    # ys[] + xs[]


@pytest.mark.parametrize("nx", [24, 48, 100, 256])
def test_setting_the_reported_block_again_keeps_the_librarys_choice(nx):
    sim = _Handle((nx, 512, 512))
    before = sim.option(_lib.OPT_STEPS_PER_PASS)
    bx, by = sim.option(_lib.OPT_BLOCK_X), sim.option(_lib.OPT_BLOCK_Y)
    for key, value in ((_lib.OPT_BLOCK_X, bx), (_lib.OPT_BLOCK_Y, by)):
        assert sim.lib.lbm_set_option(sim.h, key, value) == 0
        assert sim.option(_lib.OPT_STEPS_PER_PASS) == before
    assert sim.lib.lbm_set_option(sim.h, _lib.OPT_BLOCK_Y, 1.0) == 0  # another block: one step per pass
    assert sim.option(_lib.OPT_STEPS_PER_PASS) == 1
    assert sim.lib.lbm_set_option(sim.h, _lib.OPT_BLOCK_Y, by) == 0
    assert sim.option(_lib.OPT_STEPS_PER_PASS) == before


# measured on a GB300: us a step in pairs and singly
@pytest.mark.parametrize("shape,stencil,collision,walls_y,passes", [
    ((1000, 64, 64), 19, 0, 1, 1),     # 98.4, 91.4
    ((512, 128, 50), 19, 0, 1, 1),     # 78.6, 73.0
    ((171, 209, 251), 19, 0, 1, 2),    # 203.2, 210.6
    ((85, 419, 113), 19, 0, 1, 2),     # 94.1, 98.3
    ((512, 256, 256), 19, 1, 1, 2),    # 583, 741
    ((96, 500, 80), 19, 2, 0, 1),      # 90.2, 86.4
    ((300, 300, 20), 19, 2, 0, 2),     # 37.7, 41.7
    ((256, 256, 256), 19, 2, 0, 2),    # 307, 370
    ((116, 160, 279), 27, 1, 1, 1),    # 207.8, 170.7
    ((171, 209, 251), 27, 1, 1, 2)])   # 295.3, 311.2
def test_pairs_run_where_they_are_faster(shape, stencil, collision, walls_y, passes):
    sim = _Handle(shape, stencil, options=[(_lib.OPT_COLLISION, collision), (_lib.OPT_WALLS_Y, walls_y)])
    assert sim.option(_lib.OPT_STEPS_PER_PASS) == passes


@pytest.mark.parametrize("shape,rho0,passes", [((207, 376, 56), 1, 1), ((581, 332, 113), 0, 2)])
def test_walled_mrt_pairs_run_where_they_are_faster(shape, rho0, passes):
    """us a step in pairs and singly: 106.2, 96.8; 402, 531."""
    options = [(_lib.OPT_COLLISION, _lib.MRT), (_lib.OPT_WALLS_Y, 1), (_lib.OPT_RHO0_MODE, rho0)]
    assert _Handle(shape, options=options).option(_lib.OPT_STEPS_PER_PASS) == passes
