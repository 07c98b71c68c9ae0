"""The step kernels walk a lattice as one sequence of cells (or quads): lattices
whose rows, planes and total end anywhere within a warp or a block must give
the FP64 oracle's populations, cell by cell, for every pattern and storage.

Tolerances per step (largest absolute difference of a stored population, about
0.05 in size here): FP64 and FP32 by their rounding; 16-bit storage by half a
unit in the last place of the largest stored value per rounding (FP16 2^-16,
BF16 2^-13 relative to values below 2^-4), three roundings (initial state and
two steps) and a factor of two for what a step does to an earlier rounding."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from tests._helpers import gpu_pdfs_in_oracle_layout, gpu_to_oracle_order, oracle_config, random_fields

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-14, "f32": 1e-7, "f16s": 3 * 2 * 2.0 ** -16, "bf16s": 3 * 2 * 2.0 ** -13}

# nx, ny, nz: rows shorter than a warp, of odd length, one quad long, just past a block; planes of one row;
# totals of one cell, one short of and one past a block of 128
SHAPES = [(1, 1, 1), (2, 5, 3), (3, 7, 11), (4, 96, 3), (4, 1, 32), (127, 1, 1), (129, 1, 1), (31, 33, 2), (44, 9, 7),
          (160, 3, 5), (132, 2, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("pattern,stencil", [("ab", 19), ("aa", 19), ("ab", 27)])
@pytest.mark.parametrize("walls", [(0, 0, 0), (1, 1, 1)])
def test_any_row_length_matches_oracle(shape, precision, pattern, stencil, walls):
    from paper_1803_04937_gb300.lbm import Simulation
    nx, ny, nz = shape
    kw = dict(equilibrium="standard", collision="trt", tau=0.7, walls=tuple(bool(w) for w in walls),
              force=(1e-4, -5e-5, 2e-5))
    rho, u = random_fields((nz, ny, nx), seed=nx + 7 * ny)
    sim = Simulation(nx, ny, nz, precision=precision, pattern=pattern, stencil=stencil, **kw)
    sim.init(rho.cuda(), u.cuda())
    sim.step(2)
    f_g = gpu_pdfs_in_oracle_layout(sim)
    cfg = oracle_config(nx, ny, nz, stencil=stencil, **kw)
    f_o = oracle.step(cfg, oracle.init(cfg, rho.numpy(), u.numpy()), 2)
    assert np.abs(f_g - f_o).max() < TOL[precision]


@pytest.mark.parametrize("shape", [(5, 3, 2), (16, 16, 1), (127, 3, 3), (128, 2, 3), (256, 4, 2), (144, 5, 4)])
@pytest.mark.parametrize("walls", [(False, False, False), (True, True, True)])
def test_adjoint_of_any_row_length_matches_oracle(shape, walls):
    """One FP64 adjoint step, on lattices that take its grid of 128 x 2 blocks and its sequence of cells."""
    from paper_1803_04937_gb300 import _lib
    from paper_1803_04937_gb300.lbm import Simulation
    nx, ny, nz = shape
    kw = dict(equilibrium="improved", collision="trt", tau=0.7, walls=walls)
    rho, u = random_fields((nz, ny, nx), seed=3 * nx + ny)
    sim = Simulation(nx, ny, nz, precision="f64", **kw)
    sim.init(rho.cuda(), u.cuda())
    lam = torch.from_numpy(np.random.default_rng(5).standard_normal((19, nz, ny, nx))).cuda()
    out = torch.empty_like(lam)
    gw = torch.zeros(2, dtype=torch.float64, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    _lib.check(sim._lib.lbm_adjoint_step(sim.handle, p(sim.grids[0]), p(lam), p(out),
                                         ctypes.cast(p(gw), ctypes.POINTER(ctypes.c_double))), sim.handle)
    cfg = oracle_config(nx, ny, nz, **kw)
    perm = gpu_to_oracle_order()
    f_o = oracle.init(cfg, rho.numpy(), u.numpy())
    lam_o, g_o = oracle.adjoint_step(cfg, f_o, np.ascontiguousarray(np.moveaxis(lam.cpu().numpy()[perm], 0, -1)))
    got = np.moveaxis(out.cpu().numpy()[perm], 0, -1)
    assert np.abs(got - lam_o).max() < 1e-12
    assert np.abs(gw.cpu().numpy() - g_o).max() < 1e-11 * nx * ny * nz


@pytest.mark.parametrize("shape", [(2, 3, 5), (6, 1, 2), (62, 5, 3), (66, 3, 4), (130, 2, 3), (254, 1, 1)])
@pytest.mark.parametrize("precision", ["f16s", "bf16s"])
@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("walls", [(0, 0, 0), (0, 1, 0), (0, 0, 1), (1, 0, 0), (1, 1, 1)])
def test_rows_of_pairs_match_one_cell_per_thread(shape, precision, pattern, walls):
    """16-bit rows that hold pairs but no quads of cells: bitwise the one-cell kernels' populations."""
    from paper_1803_04937_gb300.lbm import Simulation
    nx, ny, nz = shape
    rho, u = random_fields((nz, ny, nx), seed=nx + ny)
    out = []
    for cells_x in (4, 1):
        sim = Simulation(nx, ny, nz, precision=precision, pattern=pattern, walls=walls, collision="trt", tau=0.7,
                         force=(1e-4, -5e-5, 2e-5), cells_x=cells_x)
        sim.init(rho.cuda(), u.cuda())
        sim.step(5)
        out.append(sim.get_pdfs())
    assert torch.equal(out[0], out[1])
