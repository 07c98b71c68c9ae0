"""One row of nearly 2^31 cells (FP16 storage, in place): coordinates and offsets
beside its ends, which are formed in 32 bits, against a short row that has the
same cells there."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(nx):
    from paper_1803_04937_gb300.lbm import Simulation
    sim = Simulation(nx, 1, 1, precision="f16s", pattern="aa", tau=0.8)
    u = torch.zeros((3, 1, 1, nx), dtype=torch.float32, device="cuda")
    u[1, 0, 0, -1] = 0.01  # the one cell that differs, at the row's end
    u[0, 0, 0, 0] = -0.02
    sim.init(None, u)
    del u
    sim._keep = None
    torch.cuda.empty_cache()
    enstrophy = sim.enstrophy() * nx
    sim.step(4)
    late = sim.enstrophy() * nx
    r = sim.reduce()
    v = torch.empty((3, 1, 1, nx), dtype=torch.float32, device="cuda")
    sim.moments_into(None, v)
    ends = torch.cat([v[..., :16], v[..., -16:]], dim=-1).cpu()
    rest = float(v[..., 16:-16].abs().max())
    sim.close()
    return enstrophy, late, ends, rest, r


def test_ends_of_a_row_of_nearly_2_31_cells():
    short, long = _run(64), _run(2 ** 31 - 4)
    for a, b in zip(short[:2], long[:2]):
        assert a > 0 and b == pytest.approx(a, rel=1e-12)
    assert torch.equal(short[2], long[2])
    assert short[3] == long[3] == 0.0
    assert long[4]["nonfinite"] == 0 and long[4]["umax"] == short[4]["umax"]
