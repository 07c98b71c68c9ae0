"""Two steps per pass (LBM_OPT_STEP_PAIRS) give bitwise the populations of
one-step launches, in the same grid, for lattices that end anywhere within a
tile (30 x 22 columns, 30 x 18 with walls; D3Q27 30 x 14) or a block's planes."""
import pytest
import torch

from tests._helpers import random_fields

pytestmark = pytest.mark.gpu

# nx, ny, nz: one cell, rows shorter than a tile, tiles with one column or row left, exact tiles, one plane, many
SHAPES = [(1, 1, 1), (2, 2, 2), (5, 4, 3), (1, 7, 9), (60, 44, 4), (61, 45, 5), (31, 18, 33), (29, 19, 1), (91, 3, 70)]
WALLS = [(0, 0, 0), (0, 1, 0), (0, 1, 1), (0, 0, 1), (1, 0, 0), (1, 1, 1)]


def _sim(shape, pairs, **kw):
    from paper_1803_04937_gb300 import _lib
    from paper_1803_04937_gb300.lbm import Simulation
    sim = Simulation(*shape, precision="f32", tau=0.7, force=(1e-4, -5e-5, 2e-5), **kw)
    sim._set(_lib.OPT_STEP_PAIRS, pairs)
    rho, u = random_fields((shape[2], shape[1], shape[0]), seed=sum(shape))
    sim.init(rho.cuda(), u.cuda())
    return sim


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("walls", WALLS)
@pytest.mark.parametrize("collision,equilibrium,rho0", [("srt", "improved", False), ("trt", "standard", True),
                                                        ("mrt", "improved", False), ("mrt", "standard", True)])
def test_pairs_are_bitwise_single_steps(shape, walls, collision, equilibrium, rho0):
    out = []
    for pairs in (0, 2):
        sim = _sim(shape, pairs, walls=walls, collision=collision, equilibrium=equilibrium, rho0_is_rho=rho0,
                   graphs=False)
        sim.step(9)
        out.append((sim.get_pdfs(), sim.grids[1].clone(), sim.steps_done()))
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])  # nine steps leave the state in the second grid
    assert out[0][2] == out[1][2] == 9


@pytest.mark.parametrize("shape", SHAPES + [(60, 28, 7), (31, 15, 9)])
@pytest.mark.parametrize("walls", WALLS)
@pytest.mark.parametrize("rho0", [False, True])
def test_d3q27_pairs_are_bitwise_single_steps(shape, walls, rho0):
    out = []
    for pairs in (0, 2):
        sim = _sim(shape, pairs, walls=walls, collision="trt", equilibrium="standard", rho0_is_rho=rho0, stencil=27)
        sim.step(9)
        out.append(sim.get_pdfs())
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("n", [3, 4, 6, 16, 23])
@pytest.mark.parametrize("graphs", [False, True])
def test_any_number_of_steps(n, graphs):
    a, b = (_sim((40, 30, 12), pairs, graphs=graphs, walls=(0, 1, 0)) for pairs in (0, 2))
    for _ in range(3):
        a.step(n)
        b.step(n)
        assert torch.equal(a.get_pdfs(), b.get_pdfs())


def test_pairs_in_a_captured_graph_and_on_another_stream():
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a, b = (_sim((64, 40, 10), pairs, stream=stream) for pairs in (0, 2))
        graph = torch.cuda.CUDAGraph()
        b.step(4)
        stream.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            b.step(8)
        graph.replay()
        graph.replay()
        a.step(4 + 16)
        stream.synchronize()
        assert torch.equal(a.get_pdfs(), b.get_pdfs())
    stream.synchronize()


def test_unsupported_forms_step_singly():
    """Forms without a pair kernel take the option and step as before."""
    from paper_1803_04937_gb300 import _lib
    from paper_1803_04937_gb300.lbm import Simulation
    for kw in (dict(precision="f64"), dict(precision="f16s"), dict(precision="f32", pattern="aa"),
               dict(precision="f32", cells_x=2), dict(precision="f32", block=(64, 2))):
        out = []
        for pairs in (0, 2):
            sim = Simulation(36, 20, 6, tau=0.8, **kw)
            sim._set(_lib.OPT_STEP_PAIRS, pairs)
            rho, u = random_fields((6, 20, 36), seed=3)
            sim.init(rho.cuda(), u.cuda())
            sim.step(6)
            out.append(sim.get_pdfs())
        assert torch.equal(out[0], out[1]), kw
