"""Many steps of small lattices with walls: the kernels that take the wall rows
and the rows between them in one launch, against the one-cell A/B step (which
treats all rows alike), bit for bit.  Steps follow each other without pause, as
graph replays and as single launches, so a step that began on what the step
before had not yet made visible would differ."""
import pytest
import torch

from tests._helpers import random_fields

pytestmark = pytest.mark.gpu

# nx, ny, nz: the interior fills less than one wave; no interior rows; one interior row; rows that fill rectangles of
# blocks (32 and 40 quads a row) and rows that do not
SHAPES = [(32, 32, 32), (64, 2, 5), (16, 3, 3), (128, 40, 6), (160, 7, 9), (36, 12, 10)]
WALLS = [(1, 1, 1), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 0)]


def _run(shape, steps, rho, u, **kw):
    from paper_1803_04937_gb300.lbm import Simulation
    sim = Simulation(*shape, tau=0.7, force=(1e-5, -5e-6, 2e-6), **kw)
    sim.init(rho, u)
    sim.step(steps)
    return sim.get_pdfs()


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("walls", WALLS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision,collision", [("f16s", "trt"), ("bf16s", "srt"), ("f16s", "mrt"), ("f32", "trt")])
def test_many_steps_are_bitwise_the_one_cell_steps(shape, walls, graphs, precision, collision):
    rho, u = (t.cuda() for t in random_fields((shape[2], shape[1], shape[0]), seed=sum(shape)))
    kw = dict(precision=precision, collision=collision, walls=tuple(bool(w) for w in walls), graphs=graphs)
    ref = _run(shape, 131, rho, u, cells_x=1, **kw)
    wide = 4 if precision != "f32" else 1
    assert torch.equal(ref, _run(shape, 131, rho, u, cells_x=wide, **kw))
    assert torch.equal(ref, _run(shape, 131, rho, u, cells_x=wide, pattern="aa", **kw))
    if collision != "mrt":
        assert torch.equal(ref, _run(shape, 131, rho, u, cells_x=2, pattern="aa", **kw))


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("walls", WALLS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["f16s", "bf16s"])
def test_d3q27_many_steps_are_bitwise_the_one_cell_steps(shape, walls, graphs, precision):
    rho, u = (t.cuda() for t in random_fields((shape[2], shape[1], shape[0]), seed=sum(shape)))
    kw = dict(precision=precision, collision="trt", equilibrium="standard", stencil=27, graphs=graphs,
              walls=tuple(bool(w) for w in walls))
    assert torch.equal(_run(shape, 131, rho, u, cells_x=1, **kw), _run(shape, 131, rho, u, cells_x=4, **kw))
