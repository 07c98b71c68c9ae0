"""The reductions and the enstrophy against plain FP64 sums of the velocities
and densities that lbm_moments returns (the same FP32 or FP64 numbers that the
kernels sum), on lattices that end anywhere within a tile or a block, with
velocities from tiny to ordinary and with non-finite cells.

Tolerance: every term is kept to about 47 bits (double-float) and sums of n
terms in FP64 add n 2^-53 at most; 1e-12 covers both for these lattices."""
import math

import numpy as np
import pytest
import torch

from tests._helpers import random_fields

pytestmark = pytest.mark.gpu

RTOL = 1e-12


def _curl_square_mean(u, walls):
    u = u.cpu().numpy()

    def diff(i, axis):
        dim = 2 - axis
        up, down = np.roll(u[i], -1, dim), np.roll(u[i], 1, dim)
        if walls[axis]:
            up, down = np.moveaxis(up, dim, 0), np.moveaxis(down, dim, 0)
            own = np.moveaxis(u[i], dim, 0)
            up[-1], down[0] = -own[-1], -own[0]
            up, down = np.moveaxis(up, 0, dim), np.moveaxis(down, 0, dim)
        return 0.5 * (up - down)

    w = [diff(2, 1) - diff(1, 2), diff(0, 2) - diff(2, 0), diff(1, 0) - diff(0, 1)]
    return 0.5 * math.fsum((sum(a * a for a in w)).ravel()) / w[0].size


@pytest.mark.parametrize("shape", [(1, 1, 1), (30, 14, 3), (31, 15, 2), (61, 9, 40), (5, 3, 70)])
@pytest.mark.parametrize("precision,pattern,steps", [("f32", "ab", 2), ("f32", "aa", 1), ("f16s", "aa", 2),
                                                     ("f64", "ab", 1)])
@pytest.mark.parametrize("walls", [(False, False, False), (True, True, True)])
@pytest.mark.parametrize("scale", [1.0, 1e-8, 1e-18])
def test_reductions_are_fp64_sums_of_the_moments(shape, precision, pattern, steps, walls, scale):
    from paper_1803_04937_gb300.lbm import Simulation
    nx, ny, nz = shape
    if precision == "f16s" and scale < 1.0:
        pytest.skip("FP16 storage holds no such velocities")
    force = (1e-5 * scale, 0.0, -2e-5 * scale)
    sim = Simulation(nx, ny, nz, precision=precision, pattern=pattern, walls=walls, tau=0.7, force=force)
    _, u = random_fields((nz, ny, nx), seed=nx + ny)
    sim.init(None, (u * scale).cuda())
    sim.step(steps)
    rho, v = sim.moments(torch.float64)
    r = sim.reduce()
    v_np, n = v.cpu().numpy(), nx * ny * nz
    assert r["nonfinite"] == 0
    assert abs(r["mass"] - math.fsum(rho.cpu().numpy().ravel())) <= 1e-7 * n  # FP32 rho = 1 + drho is rounded
    energy = 0.5 * math.fsum((v_np ** 2).ravel())
    assert abs(r["energy"] - energy) <= RTOL * energy
    for i in range(3):
        want = math.fsum(v_np[i].ravel()) - 0.5 * force[i] * n
        assert abs(r["momentum"][i] - want) <= RTOL * (np.abs(v_np[i]).sum() + abs(force[i]) * n) + 1e-7 * abs(force[i]) * n
    assert r["umax"] == pytest.approx(math.sqrt(((v_np ** 2).sum(0)).max()), rel=RTOL)
    want = _curl_square_mean(v, walls)
    assert abs(sim.enstrophy() - want) <= RTOL * max(want, energy / n)


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16s"])
def test_non_finite_cells_are_counted(value, precision):
    from paper_1803_04937_gb300.lbm import Simulation
    sim = Simulation(33, 7, 5, precision=precision, pattern="aa")
    f = torch.zeros((19, 5, 7, 33), dtype=sim.storage_dtype, device="cuda")
    f[0, 1, 2, 3] = value
    f[7, 4, 6, 32] = value
    f[8, 4, 6, 32] = -value
    sim.set_pdfs(f)
    r = sim.reduce()
    assert r["nonfinite"] == 2 and r["status"] == 5
    assert not math.isfinite(r["mass"])
