"""Every route that lbm_step takes by size, against the one-cell, one-step kernels,
bit for bit: pairs of steps on full-size lattices and with every collision, and the
forms of the 16-bit in-place odd step that only lattices beyond the L2 cache take."""
import pytest
import torch

from tests._helpers import random_fields

pytestmark = pytest.mark.gpu


def _sim(shape, seed=1, **kw):
    from paper_1803_04937_gb300.lbm import Simulation
    sim = Simulation(*shape, **kw)
    nx, ny, nz = shape
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rho = 1 + 0.02 * (2 * torch.rand((nz, ny, nx), generator=gen, device="cuda") - 1)
    u = 0.05 * (2 * torch.rand((3, nz, ny, nx), generator=gen, device="cuda") - 1)
    sim.init(rho, u)
    return sim


@pytest.mark.parametrize("shape,walls,stencil,collision,equilibrium", [
    ((256, 256, 256), (0, 0, 0), 19, "srt", "improved"), ((256, 256, 256), (0, 0, 0), 19, "trt", "standard"),
    ((256, 256, 256), (0, 0, 0), 19, "mrt", "improved"), ((512, 256, 256), (0, 1, 0), 19, "trt", "improved"),
    ((256, 256, 256), (0, 0, 0), 27, "trt", "standard"), ((171, 209, 251), (0, 1, 1), 19, "trt", "standard")])
def test_full_size_pairs_are_bitwise_single_steps(shape, walls, stencil, collision, equilibrium):
    """The lattices on which lbm_step chooses pairs by itself: one call of four steps against four calls of one."""
    from paper_1803_04937_gb300 import _lib
    kw = dict(precision="f32", tau=0.7, force=(1e-5, -5e-6, 2e-6), walls=tuple(bool(w) for w in walls),
              stencil=stencil, collision=collision, equilibrium=equilibrium)
    a, b = _sim(shape, **kw), _sim(shape, **kw)
    assert a.option(_lib.OPT_STEPS_PER_PASS) == 2
    a.step(4)
    for _ in range(4):
        b.step(1)
    assert torch.equal(a.grids[0], b.grids[0])


@pytest.mark.parametrize("shape", [(5, 4, 3), (31, 18, 33), (61, 45, 5), (91, 3, 70)])
@pytest.mark.parametrize("walls", [(0, 0, 0), (0, 1, 1)])
@pytest.mark.parametrize("rho0", [False, True])
@pytest.mark.parametrize("collision,equilibrium", [("srt", "standard"), ("trt", "standard"), ("trt", "improved"),
                                                   ("mrt", "standard")])
def test_pairs_of_every_collision_are_bitwise_single_steps(shape, walls, rho0, collision, equilibrium):
    from paper_1803_04937_gb300 import _lib
    from paper_1803_04937_gb300.lbm import Simulation
    out = []
    for pairs in (0, 2):
        sim = Simulation(*shape, precision="f32", tau=0.6, force=(1e-4, -5e-5, 2e-5), rho0_is_rho=rho0,
                         walls=tuple(bool(w) for w in walls), collision=collision, equilibrium=equilibrium)
        sim._set(_lib.OPT_STEP_PAIRS, pairs)
        rho, u = random_fields((shape[2], shape[1], shape[0]), seed=3)
        sim.init(rho.cuda(), u.cuda())
        sim.step(13)
        out.append(sim.get_pdfs())
    assert torch.equal(out[0], out[1])


# periodic grids above 100 MiB: rows that leave lanes of their blocks idle (250 quads in blocks of 128), rows that fill
# them (64 and 32 quads), and rows taken as one sequence (40 quads)
@pytest.mark.parametrize("shape", [(1000, 60, 48), (256, 120, 97), (128, 151, 149), (160, 140, 130)])
@pytest.mark.parametrize("precision", ["f16s", "bf16s"])
@pytest.mark.parametrize("collision,rho0", [("trt", False), ("srt", True), ("mrt", False)])
def test_in_place_16_bit_steps_beyond_l2_are_bitwise_one_cell_steps(shape, precision, collision, rho0):
    assert shape[0] * shape[1] * shape[2] * 38 > 100 << 20
    kw = dict(precision=precision, tau=0.7, force=(1e-5, -5e-6, 2e-6), collision=collision, rho0_is_rho=rho0)
    a, b = _sim(shape, cells_x=1, **kw), _sim(shape, pattern="aa", cells_x=4, **kw)
    for n in (5, 1, 18):  # odd and even counts, single launches and a graph
        a.step(n)
        b.step(n)
        assert torch.equal(a.get_pdfs(), b.get_pdfs())


@pytest.mark.parametrize("shape", [(128, 3, 5), (256, 5, 2), (65, 4, 3), (64, 3, 3)])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("walls", [(0, 0, 0), (1, 1, 1)])
def test_d3q27_rows_in_rectangles_of_blocks(shape, precision, walls):
    """D3Q27 steps with walls and copies of rows of whole blocks, and the set of rows longer than 64, against the
    oracle; then a round trip through the copies."""
    from tests.test_gpu_mapping import test_any_row_length_matches_oracle as against_oracle
    against_oracle(shape, precision, "ab", 27, walls)
    a = _sim(shape, precision=precision, stencil=27, equilibrium="standard", walls=tuple(bool(w) for w in walls), cells_x=1)
    a.step(1)
    f, m = a.get_pdfs(), a.moments(torch.float64)
    a.set_pdfs(f)
    assert torch.equal(a.get_pdfs(), f)
    assert all(torch.equal(x, y) for x, y in zip(a.moments(torch.float64), m))


@pytest.mark.parametrize("kw", [dict(precision="f32"), dict(precision="f16s"), dict(precision="f32", pattern="aa"),
                                dict(precision="f16s", pattern="aa"), dict(precision="f16s", stencil=27)])
@pytest.mark.parametrize("walls", [(False, False, False), (True, True, True)])
def test_steps_captured_after_a_join_of_two_streams(kw, walls):
    """Steps launched early, recorded into a caller's graph behind work of another stream and behind a plain kernel."""
    kw = dict(kw, walls=walls, equilibrium="standard", tau=0.7)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s1):
        a, b = (_sim((48, 20, 12), stream=s1, **kw) for _ in range(2))
        for sim in (a, b):
            sim.step(2)
        f = b.get_pdfs()
        g = torch.zeros_like(f)
        s1.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s1):
            s2.wait_stream(s1)
            with torch.cuda.stream(s2):
                g.copy_(f)       # the populations that the steps start from pass through the other stream
            s1.wait_stream(s2)
            b.set_pdfs(g)
            b.step(2)
            g.add_(0)            # a plain kernel between the steps
            b.step(4)
        graph.replay()
        a.step(6)
        assert torch.equal(a.get_pdfs(), b.get_pdfs())
    s1.synchronize()
