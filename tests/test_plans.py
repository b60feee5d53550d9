"""Plans that the planner has to accept, asked for through vp_workspace_size on the host."""
import math

import pytest

from paper_2007_12227_gb300 import vlasov as V


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2007_12227_gb300 import build as B
    B.build()


def size(nx, np_, precision, kernel, tile_x=0, tile_p=0):
    g = V.vp_grid(nx, np_, -math.pi, math.pi, -3.0, 3.0)
    pu = V.vp_pusher(V.VP_PUSH_LEAPFROG_KDK, V.VP_POT_PENDULUM, 1.0, 1.0, 0.05, 0.0, 0.0, 0.0, 0.0)
    o = V.vp_opts(precision, V.VP_PROJ_GALERKIN, kernel, tile_x, tile_p, 0, None)
    return V.vp_workspace_size(g, V.VP_BASIS_CUBIC_BSPLINE, pu, o)


@pytest.mark.parametrize("nx", [241, 250, 256, 257, 300])
def test_separate_x_pass_fp32_takes_meshes_little_wider_than_a_window(nx):
    """The default tile leaves the mesh wider than its window."""
    assert size(nx, 100, V.VP_FP32, V.VP_KERNEL_FUSED_XPASS) >= 2 * 4 * nx * 100


@pytest.mark.parametrize("nx,tile", [(300, (300, 128)), (357, (448, 128)), (320, (480, 256)), (288, (400, 256))])
def test_fp64_takes_tiles_as_wide_as_the_mesh(nx, tile):
    """A whole-period tile, whatever the planner would choose by itself: no third mesh-sized buffer either."""
    plain = size(nx, 130, V.VP_FP64, V.VP_KERNEL_FUSED, *tile)
    assert abs(size(nx, 130, V.VP_FP64, V.VP_KERNEL_AUTO, *tile) - plain) < 8 * nx
