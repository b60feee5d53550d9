"""Default and asked-for plans on meshes near the planner's lines, against the oracle: the plan taken and its weights
(FP64 <= 1e-12 relative L-infinity, FP32 <= 1e-5 relative L1, as in test_gpu_parity)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2007_12227_gb300 import inputs as I  # noqa: E402
from paper_2007_12227_gb300 import vlasov as V  # noqa: E402

PI = math.pi
AUTO, FUSED, XP = V.VP_KERNEL_AUTO, V.VP_KERNEL_FUSED, V.VP_KERNEL_FUSED_XPASS


def run(nx, np_, precision, kernel, tile=(0, 0), steps=5):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = I.Workload("t", I.Grid(nx, np_, -PI, PI, -3.0, 3.0), I.Pusher(I.PUSH_KDK, I.POT_PENDULUM, 1.0, 1.0, 0.07),
                    I.BASIS_CUBIC, precision, 0, "gaussian", dict(xc=0.0, pc=0.8, sx=0.5, sp=0.5))
    f = I.make_f0(wl)
    if precision == I.FP32:
        f = f.astype(np.float32)
    sim = V.Sim(wl.grid, wl.basis, wl.pusher, precision=precision, kernel=kernel, tile_x=tile[0], tile_p=tile[1])
    plan = sim.plan()
    sim.set_f(f)
    sim.step(steps)
    got = sim.get_f()
    sim.close()
    st = O.State(wl.grid, wl.pusher, O.CUBIC, O.GALERKIN, f.astype(np.float64))
    st.run(steps)
    if precision == I.FP64:
        assert np.abs(got - st.w).max() <= 1e-12 * np.abs(st.w).max()
    else:
        assert np.abs(got - st.w).sum() <= 1e-5 * np.abs(st.w).sum()
    return plan


@pytest.mark.parametrize("nx", [241, 255, 256, 257])
def test_separate_x_pass_fp32_on_a_mesh_little_wider_than_a_window(nx):
    assert run(nx, 60, I.FP32, XP)["kernel"] == XP


@pytest.mark.parametrize("nx,tile", [(300, (300, 128)), (357, (448, 128)), (300, (290, 0))])
def test_fp64_tile_as_wide_as_the_mesh(nx, tile):
    plan = run(nx, 130, I.FP64, AUTO, tile)
    assert plan["kernel"] == FUSED and plan["full_row"] == 1


@pytest.mark.parametrize("nx,tile,kernel", [(301, (0, 0), XP), (700, (0, 24), XP), (530, (400, 16), XP), (530, (530, 16), FUSED)])
def test_fp64_default_x_pass_in_place(nx, tile, kernel):
    """Odd rows, rows longer than a whole-period tile may be, tiles asked for (one leaves the pass's window no room)."""
    assert run(nx, 75, I.FP64, AUTO, tile)["kernel"] == kernel


@pytest.mark.parametrize("nx,np_", [(175, 90), (176, 90), (201, 300), (233, 828), (287, 61)])
def test_fp64_rows_either_side_of_the_x_pass_line(nx, np_):
    assert run(nx, np_, I.FP64, AUTO, steps=3)["kernel"] == (XP if nx >= 176 else FUSED)


def test_reset_zeroes_a_field_history_of_four_billion_words():
    """set_f zeroes the history ring: 2^32 - 4000 words here, more than a 32-bit count of the zeroing threads' steps holds."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cap = (1 << 30) - 1000
    g = I.Grid(64, 32, 0.0, 2 * PI, -0.5, 0.5)
    pu = I.Pusher(I.PUSH_FEL, I.POT_FREE, 1.0, 1.0, 0.05, 0.3, 0.0)
    if torch.cuda.mem_get_info()[0] < 18 * cap:
        pytest.skip("needs 18 GB")
    # the workspace takes this freed block, so that its history is not zero to begin with
    block = torch.empty(16 * cap + (1 << 20), dtype=torch.uint8, device="cuda").fill_(255)
    del block
    sim = V.Sim(g, I.BASIS_CUBIC, pu, precision=V.VP_FP32, history_cap=cap)
    sim.set_f(np.ones((32, 64), dtype=np.float32))
    sim.sync()
    size = sim.workspace.numel()
    margin = (size - 16 * cap + 255) // 256 * 256   # what else the workspace holds, before or behind the history
    words = sim.workspace[margin: 16 * cap // 256 * 256].view(torch.int64)
    assert not any(bool(c.any()) for c in words.split(1 << 28))
    sim.close()
    del sim, words
    torch.cuda.empty_cache()


@pytest.mark.parametrize("nx,np_,precision,tile_x", [(709, 991, I.FP64, 384), (1500, 700, I.FP32, 448)])
def test_wide_tiles_are_planned_at_one_block_an_sm(nx, np_, precision, tile_x):
    """The default height gives every SM one such tile: fewer than 152 tiles, and more than half of that."""
    plan = run(nx, np_, precision, FUSED, (tile_x, 0), steps=2)
    assert 76 < plan["ntiles_x"] * plan["ntiles_p"] <= 152


@pytest.mark.parametrize("nx,np_,tile_x", [(300, 300, 224), (1000, 200, 224), (2048, 2048, 240)])
def test_separate_x_pass_fp32_default_width(nx, np_, tile_x):
    """A multiple of the row pass's 32 nodes, or what takes one wave of tiles."""
    assert run(nx, np_, I.FP32, XP, steps=1)["tile_x"] == tile_x
