"""Boxes that are strained past the hex kernels' first screen and are still
undamaged (csrc/pdn_screen.h), next to others short of it and others past an
onset, against the FP64 oracle: nodal forces, and after one step the committed
history and which elements have one.  A free plate stretched uniformly (every
hex past the first screen, none damaged) and with a strain that grows along x
from below the screen to beyond the onset.  Tolerances relative to the largest
nodal force and to the threshold's initial 1: 1e-10 in FP64 and 1e-4 in FP32,
those of the other internal-force tests.  12,160 and 12,168 hexes are the two
sides of the rule that chooses between the FP64 forms; 2,432, 2,440, 4,864 and
4,872 those of the FP32 elements per warp."""
import dataclasses

import numpy as np
import pytest

import oracle
import pdn_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2301_05552_gb300 as p
    p.lib()
    return p


def _free_plate(nx, ny, plies, fp64):
    w = pi.damage_fp32_plate(nx=nx, ny=ny, plies=plies, Lx=0.5 * nx, Ly=0.5 * ny, H=0.275 * plies, fp64=fp64)
    p = pi.make_plate(0.5 * nx, 0.5 * ny, 0.275 * plies, nx, ny, list(w.plate.ply_angle_deg), 1, cohesive=True, clamp="none")
    return dataclasses.replace(w, plate=p)


def _state(plate, ramp):
    x, y, z = plate.X
    Lx = plate.dims[0]
    d = np.zeros_like(plate.X)
    lo, hi = (0.0005, 0.012) if ramp else (0.0035, 0.0035)
    d[0] = lo * x + 0.5 * (hi - lo) * x * x / Lx  # strain lo at x = 0, hi at x = Lx
    d[1] = -0.0012 * y + 0.001 * x
    d[2] = -0.001 * z
    return d, np.zeros_like(d)


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("nx,ny,plies", [(3, 2, 4), (5, 7, 6), (33, 13, 4), (19, 16, 8), (61, 10, 4), (38, 16, 8), (58, 21, 4),
                                         (40, 38, 8), (39, 39, 8)])
@pytest.mark.parametrize("ramp", [False, True])
def test_strained_boxes_match_oracle(pkg, nx, ny, plies, fp64, ramp):
    w = _free_plate(nx, ny, plies, fp64)
    st = _state(w.plate, ramp)
    tol = 1e-10 if fp64 else 1e-4
    g, o = pkg.Solver(w), oracle.model_for(w)
    pkg.pdn_set_state(g.ctx, *st)
    o.set_state(*st)
    fg, fo = pkg.pdn_internal_force(g.ctx), o.internal_force()
    assert np.abs(fg - fo).max() <= tol * np.abs(fo).max() and np.abs(fo).max() > 0.0
    g.step(1)
    assert o.step(1) == 0
    hg = pkg.pdn_get_history(g.ctx)[0].astype(np.float64).reshape(7, 8, -1)
    ho = o.history()[0].transpose(2, 1, 0)
    assert np.abs(hg - ho).max() <= tol
    start = np.array([1.0] * 4 + [0.0] * 3)[:, None, None]
    has_g, has_o = (hg != start).any((0, 1)), (ho != start).any((0, 1))
    barely = np.abs(ho - start).max((0, 1)) <= tol  # an onset within rounding
    assert np.array_equal(has_g | barely, has_o | barely)
    assert has_o.any() == ramp and not has_o.all()
    g.close()
    o.close()


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("nx,ny,plies", [(3, 3, 4), (33, 13, 4), (61, 10, 4), (58, 21, 4), (39, 39, 8)])
def test_plates_with_a_history_everywhere_match_oracle(pkg, nx, ny, plies, fp64):
    """Warps without one pristine element: a plate sheared past yield takes 8
    steps, and the force at its own state and history is the oracle's."""
    w = _free_plate(nx, ny, plies, fp64)
    x, y, z = w.plate.X
    d = np.stack([-0.008 * x + 0.008 * y, 0.008 * x + 0.008 * y, -0.001 * z])
    tol = 1e-10 if fp64 else 1e-4
    g, o = pkg.Solver(w), oracle.model_for(w)
    pkg.pdn_set_state(g.ctx, d, np.zeros_like(d))
    o.set_state(d, np.zeros_like(d))
    g.step(8)
    assert o.step(8) == 0
    hist, r = pkg.pdn_get_history(g.ctx)
    h = hist.reshape(7, 8, -1)
    assert ((h[:4] > 1.0).any((0, 1)) | (h[4:] != 0.0).any((0, 1))).all()
    dg, vg, _ = g.state()
    o.set_state(dg, vg)
    o.set_history(hist.astype(np.float64).transpose(2, 1, 0), r.astype(np.float64).T)
    fg, fo = pkg.pdn_internal_force(g.ctx), o.internal_force()
    assert np.abs(fo).max() > 0.0 and np.abs(fg - fo).max() <= tol * np.abs(fo).max()
    g.close()
    o.close()
