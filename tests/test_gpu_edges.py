"""What a tile must not count and must not miss.

Lost weight: rows beyond the open momentum edge are counted by the tile that owns that edge and by no other, also
where another tile's window reaches past the mesh (tiles, or a last row of tiles, lower than the window's guard
rows) and where rows beyond the window are clamped into those guard rows.

Strong shear: where the source columns of a tile span more than a period, every node still lands once.

Bounds: weights as in the other oracle comparisons (FP64 1e-12 relative L-infinity, FP32 1e-5 relative L1 of one to
three steps). The lost weight is a sum of the same deposits: in FP32 within 1e-5 of the whole mass; in FP64 the weights'
bound over the steps' sums, 1e-10 of the loss itself."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2007_12227_gb300 import inputs as I  # noqa: E402
from paper_2007_12227_gb300 import vlasov as V  # noqa: E402

PI = math.pi
FP32_TOL, FP64_TOL = 1e-5, 1e-12
T, B3 = I.BASIS_TENT, I.BASIS_CUBIC
GAL, LUMP = I.PROJ_GALERKIN, I.PROJ_LUMPED
AUTO, FUSED, XP = V.VP_KERNEL_AUTO, V.VP_KERNEL_FUSED, V.VP_KERNEL_FUSED_XPASS


def run(wl, kernel, tile, steps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    f = I.make_f0(wl)
    if wl.precision == I.FP32:
        f = f.astype(np.float32)
    sim = V.Sim(wl.grid, wl.basis, wl.pusher, precision=wl.precision, projection=wl.projection, kernel=kernel,
                tile_x=tile[0], tile_p=tile[1])
    plan = sim.plan()
    sim.set_f(f)
    sim.step(steps)
    got, mom = sim.get_f(), sim.moments()
    sim.close()
    st = O.State(wl.grid, wl.pusher, O.TENT if wl.basis == T else O.CUBIC,
                 O.GALERKIN if wl.projection == GAL else O.LUMPED, f.astype(np.float64))
    st.run(steps)
    if wl.precision == I.FP64:
        e = np.abs(got - st.w).max() / np.abs(st.w).max()
        assert e <= FP64_TOL, f"rel Linf {e:.3e}"
    else:
        e = np.abs(got - st.w).sum() / np.abs(st.w).sum()
        assert e <= FP32_TOL, f"rel L1 {e:.3e}"
    area = wl.grid.hx * wl.grid.hp
    return mom, st.lost[0] * area, f.astype(np.float64).sum() * area, plan


# nx, np, precision, basis, projection, kernel, tile: a last row of tiles of 1 to 3 rows (FP32, four guard rows), tiles and
# last rows of tiles lower than eight (FP64), whole-period and windowed tiles, several row segments, both x passes
LOSSY = {
    "fp32_last1": (400, 49, I.FP32, B3, GAL, AUTO, (0, 16)), "fp32_default121": (300, 121, I.FP32, B3, GAL, AUTO, (0, 0)),
    "fp32_default75": (357, 75, I.FP32, B3, GAL, AUTO, (0, 0)), "fp32_lumped": (300, 73, I.FP32, B3, LUMP, AUTO, (0, 0)),
    "fp32_tent": (300, 50, I.FP32, T, GAL, AUTO, (96, 16)), "fp32_full": (120, 50, I.FP32, B3, GAL, AUTO, (0, 24)),
    "fp32_xpass": (500, 65, I.FP32, B3, GAL, XP, (96, 16)), "fp32_low": (300, 31, I.FP32, B3, GAL, FUSED, (64, 2)),
    "fp64_tent128": (128, 128, I.FP64, T, GAL, AUTO, (0, 0)), "fp64_cubic128": (128, 128, I.FP64, B3, GAL, AUTO, (0, 0)),
    "fp64_last2": (275, 66, I.FP64, B3, GAL, FUSED, (64, 64)), "fp64_last7": (400, 71, I.FP64, T, GAL, AUTO, (96, 32)),
    "fp64_xpass": (301, 67, I.FP64, B3, GAL, AUTO, (0, 0)), "fp64_low": (200, 40, I.FP64, B3, LUMP, FUSED, (64, 3)),
}


@pytest.mark.parametrize("name", LOSSY)
def test_lost_weight_is_counted_once(name):
    nx, np_, prec, basis, proj, kernel, tile = LOSSY[name]
    g = I.Grid(nx, np_, -PI, PI, -1.0, 1.0)
    for pc in (0.8, -0.8):   # kicks of several rows across the upper and the lower edge
        wl = I.Workload(name, g, I.Pusher(I.PUSH_KDK, I.POT_PENDULUM, 1.0, 1.0, 0.3), basis, prec, 2, "gaussian",
                        dict(xc=1.0, pc=pc, sx=1.2, sp=0.15), projection=proj)
        mom, lost, mass, _ = run(wl, kernel, tile, 2)
        assert lost > 0.02 * mass, "the flow has to lose weight"
        tol = 1e-10 * lost if prec == I.FP64 else FP32_TOL * mass
        assert abs(mom["lost_mass"] - lost) <= tol, f"{name}: {mom['lost_mass']:.6f} for {lost:.6f} of {mass:.6f}"


def rot(nx, np_, angle):
    return I.Grid(nx, np_, -4.0, 4.0, -4.0, 4.0), I.Pusher(I.PUSH_ROTATION, I.POT_HARMONIC, 1.0, 1.0, angle)


def stream(nx, np_, dt):
    return I.Grid(nx, np_, -PI, PI, -3.0, 3.0), I.Pusher(I.PUSH_KDK, I.POT_FREE, 1.0, 1.0, dt)


def pend(nx, np_, dt):
    return I.Grid(nx, np_, -PI, PI, -4.0, 4.0), I.Pusher(I.PUSH_KDK, I.POT_PENDULUM, 1.0, 1.0, dt)


def fel(nx, np_, dt):
    return I.Grid(nx, np_, 0.0, 2 * PI, -2.0, 2.0), I.Pusher(I.PUSH_FEL, I.POT_FREE, 1.0, 1.0, dt, 0.3, 0.0)


SHEAR = {
    "rot_fp64_255": (rot(255, 200, 1.0), I.FP64, B3, GAL, AUTO, (0, 0)),
    "rot_fp64_256": (rot(256, 200, 1.3), I.FP64, B3, GAL, AUTO, (0, 0)),
    "rot_fp64_lumped": (rot(200, 200, 1.0), I.FP64, B3, LUMP, AUTO, (0, 0)),
    "rot_fp64_xpass": (rot(333, 150, 1.3), I.FP64, B3, GAL, AUTO, (0, 0)),
    "rot_fp64_in_tile": (rot(300, 150, 1.2), I.FP64, B3, GAL, FUSED, (64, 24)),
    "rot_fp32_640": (rot(640, 512, 1.0), I.FP32, B3, GAL, AUTO, (0, 0)),
    "rot_fp32_odd": (rot(333, 200, 0.6), I.FP32, B3, GAL, AUTO, (0, 0)),
    "rot_fp32_lumped": (rot(420, 330, 1.4), I.FP32, B3, LUMP, AUTO, (0, 0)),
    "rot_fp32_tent": (rot(333, 200, 1.2), I.FP32, T, GAL, AUTO, (96, 24)),
    "rot_fp32_xpass": (rot(400, 200, 1.1), I.FP32, B3, GAL, XP, (96, 32)),
    "rot_fp32_tall": (rot(1300, 90, 1.2), I.FP32, B3, GAL, FUSED, (208, 64)),
    "stream_fp32": (stream(320, 64, 1.0), I.FP32, B3, GAL, AUTO, (0, 0)),
    "stream_fp32_far": (stream(321, 64, 9.0), I.FP32, B3, GAL, AUTO, (0, 0)),
    "stream_fp64": (stream(320, 64, 1.0), I.FP64, B3, GAL, AUTO, (0, 0)),
    "stream_fp64_tent": (stream(400, 50, 7.0), I.FP64, T, GAL, AUTO, (0, 0)),
    "pend_fp32": (pend(300, 120, 2.5), I.FP32, B3, GAL, AUTO, (0, 0)),
    "pend_fp64": (pend(300, 120, 2.5), I.FP64, B3, GAL, AUTO, (0, 0)),
    "fel_fp32": (fel(300, 120, 2.0), I.FP32, B3, GAL, AUTO, (0, 0)),
    "fel_fp64": (fel(300, 120, 2.0), I.FP64, B3, GAL, AUTO, (0, 0)),
}


@pytest.mark.parametrize("name", SHEAR)
def test_every_node_lands_once_under_strong_shear(name):
    (g, pu), prec, basis, proj, kernel, tile = SHEAR[name]
    if pu.kind == I.PUSH_FEL:
        wl = I.Workload(name, g, pu, basis, prec, 1, "fel_gaussian", dict(sp=0.8, eps=0.1), projection=proj)
    else:
        wl = I.Workload(name, g, pu, basis, prec, 1, "gaussian", dict(xc=0.5, pc=-0.3, sx=1.2, sp=1.0), projection=proj)
    mom, lost, mass, plan = run(wl, kernel, tile, 1)
    assert plan["kernel"] in (FUSED, XP), "a one-pass plan"
    assert abs(mom["lost_mass"] - lost) <= (1e-10 * lost + 1e-12 * mass if prec == I.FP64 else FP32_TOL * mass)


@pytest.mark.parametrize("prec", [I.FP32, I.FP64], ids=["fp32", "fp64"])
@pytest.mark.parametrize("basis", [T, B3], ids=["tent", "cubic"])
@pytest.mark.parametrize("nx", [4, 5, 7, 8])
def test_meshes_narrower_than_the_guard_band(nx, basis, prec):
    """Nodes that land several periods' worth of columns away, in guard columns of which some share their image."""
    for dt in (1.0, 3.0, 4.3):
        g, pu = I.Grid(nx, 40, -PI, PI, -3.0, 3.0), I.Pusher(I.PUSH_KDK, I.POT_PENDULUM, 1.0, 1.0, dt)
        wl = I.Workload("t", g, pu, basis, prec, 1, "gaussian", dict(xc=0.5, pc=-0.3, sx=1.2, sp=1.0), projection=GAL)
        run(wl, AUTO, (0, 0), 1)
