"""The FP32 source walk (two columns per thread, segments of rows) where its pieces can go wrong: odd meshes
(no 8-byte loads, a last pair of one column), rows near the first and the last mesh row (exact pivots, a cut
look-ahead), tiles with one or several row segments, source rows past the cached row table, strong shear (the
rings restart on most rows) and weight that leaves the open edge.

One step's bound is the repository's FP32 bound, 1e-5 relative L1 against the FP64 oracle; the lost mass is a
sum of the same weights."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2007_12227_gb300 import inputs as I  # noqa: E402
from paper_2007_12227_gb300 import vlasov as V  # noqa: E402

PI = math.pi
FP32_TOL = 1e-5


def pend(nx, np_, dt=0.05, pr=(-3.0, 3.0), pc=0.3, s=0.5):
    return (I.Grid(nx, np_, -PI, PI, *pr), I.Pusher(I.PUSH_KDK, I.POT_PENDULUM, 1.0, 1.0, dt),
            ("gaussian", dict(xc=0.2, pc=pc, sx=s, sp=s)))


def rot(nx, np_, angle):
    return (I.Grid(nx, np_, -4.0, 4.0, -4.0, 4.0), I.Pusher(I.PUSH_ROTATION, I.POT_HARMONIC, 1.0, 1.0, angle),
            ("gaussian", dict(xc=1.0, pc=0.0, sx=0.4, sp=0.4)))


def fel(nx, np_, a0):
    return (I.Grid(nx, np_, 0.0, 2 * PI, -0.5, 0.5), I.Pusher(I.PUSH_FEL, I.POT_FREE, 1.0, 1.0, 0.05, a0, 0.0),
            ("fel_gaussian", dict(sp=0.05, eps=1e-2)))


CASES = {
    "odd_nx": (pend(357, 61), 0, 0), "odd_pair": (pend(321, 40), 97, 16), "one_row_tiles": (pend(300, 33), 64, 8),
    "short_mesh": (pend(400, 7), 0, 0), "top_rows": (pend(300, 81), 128, 64), "full_odd": (pend(101, 90), 0, 0),
    "full_wide": (pend(255, 70), 0, 32), "wide_tile": (pend(700, 50), 448, 32), "uncached_rows": (pend(500, 700, dt=0.6), 96, 64),
    "shear": (rot(420, 330, PI / 10), 0, 0), "shear_more": (rot(333, 200, 0.6), 96, 24),
    "edge_loss": (pend(300, 60, dt=0.5, pr=(-1.0, 1.0), pc=0.8, s=0.2), 96, 16),
    "edge_loss_full": (pend(120, 60, dt=0.5, pr=(-1.0, 1.0), pc=-0.8, s=0.2), 0, 0), "fel": (fel(301, 95, 0.3), 0, 32),
}


@pytest.mark.parametrize("proj", [I.PROJ_GALERKIN, I.PROJ_LUMPED], ids=["galerkin", "lumped"])
@pytest.mark.parametrize("name", CASES)
def test_walk_matches_oracle(name, proj):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    (g, pu, (f0, args)), tx, tp = CASES[name]
    wl = I.Workload(name, g, pu, I.BASIS_CUBIC, I.FP32, 3, f0, args, projection=proj)
    f = I.make_f0(wl).astype(np.float32)
    sim = V.Sim(g, wl.basis, pu, precision=V.VP_FP32, projection=proj, kernel=V.VP_KERNEL_FUSED, tile_x=tx, tile_p=tp)
    sim.set_f(f)
    sim.step(3)
    got, mom = sim.get_f(), sim.moments()
    sim.close()
    st = O.State(g, pu, O.CUBIC, O.GALERKIN if proj == I.PROJ_GALERKIN else O.LUMPED, f.astype(np.float64))
    st.run(3)
    e = np.abs(got - st.w).sum() / np.abs(st.w).sum()
    assert e <= FP32_TOL, f"{name}: rel L1 {e:.3e}"
    assert abs(mom["lost_mass"] - st.lost[0] * g.hx * g.hp) <= FP32_TOL, name
