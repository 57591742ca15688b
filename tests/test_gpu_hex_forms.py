"""Hex8 internal force in its forms against the FP64 oracle: one thread per
element for boxes that stay elastic, eight lanes per element for the others, for
general hexes and for small FP64 launches.  Hex counts that leave part of a
group of four, of a warp and of a block empty, and the FP64 counts on both sides
of the rule that chooses between the two (12,160 and 12,168 hexes); states that
are elastic everywhere, damaging in part, and damaging with a history from 20
steps.  Tolerance relative to the largest nodal force: 1e-10 in FP64 and 1e-4 in
FP32, those of the repository's other internal-force tests (a node's force is a
sum of element forces that largely cancel)."""
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


def _plate(nx, ny, plies, skew, fp64):
    w = pi.damage_fp32_plate(nx=nx, ny=ny, plies=plies, Lx=0.5 * nx, Ly=0.5 * ny, H=0.275 * plies, fp64=fp64)
    if skew:
        Lx, Ly, _ = w.plate.dims
        x, y = w.plate.X[0].copy(), w.plate.X[1].copy()
        bump = np.sin(np.pi * x / Lx) * np.sin(np.pi * y / Ly)
        w.plate.X[0] = x + 0.1 * bump * np.sin(9.0 * y / Ly)
        w.plate.X[1] = y + 0.1 * bump * np.cos(7.0 * x / Lx)
    return w


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("nx,ny,plies,skew", [(3, 3, 4, False), (5, 7, 6, False), (11, 3, 4, True), (13, 9, 4, True),
                                              (40, 38, 8, False), (39, 39, 8, False)])
@pytest.mark.parametrize("state", ["elastic", "damaging", "history"])
def test_forms_match_oracle(pkg, nx, ny, plies, skew, fp64, state):
    w = _plate(nx, ny, plies, skew, fp64)
    Lx, Ly, _ = w.plate.dims
    if state == "elastic":
        st = pi.seeded_state(w.plate, 7, amp=1e-4, vamp=0.0)
    else:
        st = pi.seeded_state(w.plate, 7, amp=0.02, vamp=300.0, dimple=(0.5 * Lx, 0.5 * Ly, 0.12, 0.25 * min(Lx, Ly)))
    g, o = pkg.Solver(w), oracle.model_for(w)
    pkg.pdn_set_state(g.ctx, *st)
    o.set_state(*st)
    if state == "history":
        g.step(20)
        assert o.step(20) == 0
        # the oracle's force at the GPU's own state and history
        d, v, _ = g.state()
        o.set_state(d, v)
        hist, r = pkg.pdn_get_history(g.ctx)
        o.set_history(hist.astype(np.float64).transpose(2, 1, 0), r.astype(np.float64).T)
    fg, fo = pkg.pdn_internal_force(g.ctx), o.internal_force()
    assert np.abs(fo).max() > 0.0
    assert np.abs(fg - fo).max() <= (1e-10 if fp64 else 1e-4) * np.abs(fo).max()
    g.close()
    o.close()
