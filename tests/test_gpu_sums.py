"""The reductions' sums against exact sums of the terms that the kernels add: no
less precise than FP64 sums of those terms, for every storage precision.

The terms are formed from the velocities and densities that lbm_moments returns
in FP64 (the kernels' own FP32 or FP64 numbers, unrounded) and, for the mass,
from the populations.  Tolerance: a sum in FP64 rounds once per addition, by at
most 2^-53 of the sum of the absolute terms so far.  Cells of these lattices go
to one thread each (up to 4 roundings for its terms) and are added in trees of
at most 40 levels on the way to the result."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _sim(shape, precision, walls=(False, False, False), rho0=False, force=(0.0, 0.0, 0.0)):
    from paper_1803_04937_gb300.lbm import Simulation
    return Simulation(*shape, precision=precision, tau=0.8, walls=walls, rho0_is_rho=rho0, force=force, pattern="aa")


def _random_state(sim, seed, decades=3.0):
    """Random populations of very different sizes, so that sums round in their last bits."""
    rng = np.random.default_rng(seed)
    f = rng.standard_normal((19,) + sim.shape) * 0.02 * 10.0 ** rng.uniform(-decades, 0, (19,) + sim.shape)
    sim.set_pdfs(torch.from_numpy(f).to(sim.storage_dtype))


def _drho(sim):
    """rho - 1 of each cell as the kernels form it: the populations in order, in the compute precision."""
    f = sim.get_pdfs()
    f = f.cpu().numpy() if sim.storage_dtype == torch.float64 else f.float().cpu().numpy()
    s = f[0]
    for q in range(1, 19):
        s = s + f[q]
    return s.astype(np.float64).ravel()


def _check(sim, rho0, force, levels):
    rho, u = (t.cpu().numpy() for t in sim.moments(torch.float64))
    r = sim.reduce()
    n = sim.ncell
    tol = (4 + levels) * EPS
    drho = _drho(sim)
    # the mass is returned as n + sum(drho), which rounds once more
    assert abs(Fraction(r["mass"]) - n - sum(map(Fraction, drho))) <= tol * np.abs(drho).sum() + 2 * EPS * n
    squares = (u ** 2).ravel()  # exact for FP32 u; FP64 rounds each once, which tol covers
    assert abs(r["energy"] - 0.5 * math.fsum(squares)) <= tol * 0.5 * squares.sum()
    real = np.float64 if sim.storage_dtype == torch.float64 else np.float32
    for i in range(3):
        half = float(real(0.5 * force[i]))
        terms = (rho.ravel() if rho0 else 1.0) * u[i].ravel()
        want = math.fsum(terms) - n * half
        assert abs(r["momentum"][i] - want) <= tol * (np.abs(terms).sum() + n * abs(half))


@pytest.mark.parametrize("precision", ["f32", "f16s", "bf16s", "f64"])
@pytest.mark.parametrize("rho0", [False, True])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 1, 1), (3, 2, 2)])
def test_sums_of_few_cells(shape, rho0, precision):
    force = (1e-3, -2e-5, 0.0)
    sim = _sim(shape, precision, rho0=rho0, force=force)
    for seed in range(24):
        _random_state(sim, seed)
        _check(sim, rho0, force, levels=4)  # at most 12 cells


@pytest.mark.parametrize("precision", ["f32", "f16s", "f64"])
@pytest.mark.parametrize("rho0", [False, True])
@pytest.mark.parametrize("walls", [(False, False, False), (True, True, True)])
@pytest.mark.parametrize("shape", [(61, 33, 9), (96, 80, 70)])
def test_sums_of_many_cells(shape, walls, rho0, precision):
    """96 x 80 x 70 gives threads up to five cells each."""
    force = (1e-3, -2e-5, 0.0)
    sim = _sim(shape, precision, walls=walls, rho0=rho0, force=force)
    _random_state(sim, 5)
    _check(sim, rho0, force, levels=40)


@pytest.mark.parametrize("precision", ["f32", "f16s"])
def test_threads_of_many_cells(precision):
    """208 x 200 x 184: up to 66 cells a thread, past the 64 after which it adds them to its FP64 total."""
    sim = _sim((208, 200, 184), precision)
    _random_state(sim, 6, decades=0.5)
    rho, u = (t.cpu().numpy() for t in sim.moments(torch.float64))
    r = sim.reduce()
    tol = (8 + 40) * EPS
    drho = _drho(sim)
    assert abs((r["mass"] - sim.ncell) - math.fsum(drho)) <= tol * np.abs(drho).sum() + 2 * EPS * sim.ncell
    assert abs(r["energy"] - 0.5 * math.fsum((u ** 2).ravel())) <= tol * 0.5 * (u ** 2).sum()
    for i in range(3):
        assert abs(r["momentum"][i] - math.fsum(u[i].ravel())) <= tol * np.abs(u[i]).sum()


def _curl_square_mean(u, walls):
    """1/2 <|curl u|^2> in rational arithmetic."""
    nz, ny, nx = u.shape[1:]
    n = (nx, ny, nz)
    total = Fraction(0)

    def at(i, pos, axis, step):
        p = list(pos)
        p[axis] += step
        if not 0 <= p[axis] < n[axis]:
            if walls[axis]:
                return -Fraction(u[i, pos[2], pos[1], pos[0]])
            p[axis] %= n[axis]
        return Fraction(u[i, p[2], p[1], p[0]])

    for z in range(nz):
        for y in range(ny):
            for x in range(nx):
                pos = (x, y, z)
                d = [[at(i, pos, a, 1) - at(i, pos, a, -1) for i in range(3)] for a in range(3)]
                total += (d[1][2] - d[2][1]) ** 2 + (d[2][0] - d[0][2]) ** 2 + (d[0][1] - d[1][0]) ** 2
    return total / (8 * nx * ny * nz)


@pytest.mark.parametrize("precision", ["f32", "f16s", "f64"])
@pytest.mark.parametrize("shape,walls", [((3, 1, 1), (False, False, False)), ((1, 1, 1), (True, True, True)),
                                         ((1, 2, 3), (False, True, False)), ((5, 4, 3), (True, False, True))])
def test_enstrophy_is_no_less_precise_than_an_fp64_sum(shape, walls, precision):
    """FP64 rounds the two differences, the component, its square and the three sums: 7 per cell, then the trees."""
    sim = _sim(shape, precision, walls=walls)
    n = shape[0] * shape[1] * shape[2]
    for seed in range(24 if n < 10 else 4):
        _random_state(sim, seed, decades=6.0)
        u = sim.moments(torch.float64)[1].cpu().numpy()
        want = _curl_square_mean(u, walls)
        # (a difference of FP64 velocities may cancel: for that storage relative to the velocities)
        scale = float(want) if precision != "f64" else float(want) + float((u ** 2).max())
        assert abs(Fraction(sim.enstrophy()) - want) <= (7 + 6) * EPS * scale


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_sums_of_huge_finite_cells(precision):
    """A diverging state whose cells are finite: the sum of two densities leaves FP32's range, not FP64's."""
    sim = _sim((128, 64, 64), precision)  # more cells than threads
    f = torch.zeros((19, 64, 64, 128), dtype=sim.storage_dtype, device="cuda")
    f[0] = 3e38
    f[1] = 0.01  # an ordinary velocity
    sim.set_pdfs(f)
    r = sim.reduce()
    value = float(f[0, 0, 0, 0].double())
    assert r["nonfinite"] == 0
    assert abs(r["mass"] - value * sim.ncell) <= 48 * EPS * value * sim.ncell


@pytest.mark.parametrize("force", [(0.0, 0.0, 0.0), (1e-3, 3e-33, 0.0)])
def test_momentum_of_a_tiny_component_beside_an_ordinary_one(force):
    """rho u_y of about 1e-33: the rounding error of that product is no normal FP32 number."""
    sim = _sim((2, 2, 1), "f32", rho0=True, force=force)
    for seed in range(24):
        rng = np.random.default_rng(seed)
        f = np.zeros((19,) + sim.shape)
        f[0] = 0.05 * rng.standard_normal(sim.shape)
        f[1] = 0.01 * rng.standard_normal(sim.shape)
        f[3] = 1e-33 * rng.standard_normal(sim.shape)
        sim.set_pdfs(torch.from_numpy(f).float())
        _check(sim, True, force, levels=4)


@pytest.mark.parametrize("scale", [1.0, 1e-19, 1e-23])
def test_umax_of_tiny_velocities(scale):
    """Squares of FP32 velocities near or below FP32's smallest number: the largest |u| is still the largest.  The two
    cells are one thread's (three blocks of 256 threads on each of 152 SMs)."""
    threads = 152 * 3 * 256
    sim = _sim((threads // 64, 64, 2), "f32")
    f = torch.zeros((19, 2, 64, threads // 64), dtype=torch.float32, device="cuda")
    f[1, 0, 0, 0] = 3.0 * scale                                # |u| = 3 scale
    f[1, 1, 0, 0] = f[3, 1, 0, 0] = f[5, 1, 0, 0] = 2.5 * scale  # |u| = 4.33 scale
    sim.set_pdfs(f)
    assert sim.reduce()["umax"] == pytest.approx(2.5 * scale * 3 ** 0.5, rel=1e-6, abs=0.0)


@pytest.mark.parametrize("shape", [(4, 40, 3), (2, 70, 2), (6, 63, 4), (14, 31, 2), (62, 3, 4), (130, 2, 3), (127, 1, 2),
                                   (1, 129, 2)])
@pytest.mark.parametrize("walls", [(False, False, False), (True, True, False)])
def test_enstrophy_of_every_tile_shape(shape, walls):
    """Tiles of 4 to 128 columns, with lattices that end within and past them."""
    sim = _sim(shape, "f32", walls=walls)
    _random_state(sim, 3)
    want = _curl_square_mean(sim.moments(torch.float64)[1].cpu().numpy(), walls)
    assert abs(Fraction(sim.enstrophy()) - want) <= 40 * EPS * want
