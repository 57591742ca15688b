"""General FP32 hexes on both sides of the launch size from which one thread
takes an element (194,560): internal force against FP64 element arithmetic on
the same mesh, elastic and damaging states, 1e-4 of the largest nodal force as
the other internal-force tests; the history after one step; and a repeated
step's local evaluation against a full one, bit for bit."""
import numpy as np
import pytest

import pdn_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2301_05552_gb300 as p
    p.lib()
    return p


def _plate(nx, ny, plies):
    w = pi.damage_fp32_plate(nx=nx, ny=ny, plies=plies, Lx=0.5 * nx, Ly=0.5 * ny, H=0.275 * plies)
    Lx, Ly, _ = w.plate.dims
    x, y = w.plate.X[0].copy(), w.plate.X[1].copy()
    bump = np.sin(np.pi * x / Lx) * np.sin(np.pi * y / Ly)
    w.plate.X[0] = x + 0.1 * bump * np.sin(9.0 * y / Ly)
    w.plate.X[1] = y + 0.1 * bump * np.cos(7.0 * x / Lx)
    return w


@pytest.mark.parametrize("nx,ny,plies", [(95, 127, 16), (95, 128, 16), (121, 134, 12), (95, 129, 16)])
@pytest.mark.parametrize("state", ["elastic", "damaging"])
def test_forces_and_history_match_fp64(pkg, nx, ny, plies, state):
    w = _plate(nx, ny, plies)
    Lx, Ly, _ = w.plate.dims
    if state == "elastic":
        st = pi.seeded_state(w.plate, 7, amp=1e-4, vamp=0.0)
    else:
        st = pi.seeded_state(w.plate, 7, amp=0.02, vamp=0.0, dimple=(0.5 * Lx, 0.5 * Ly, 0.12, 2.0))
    out = []
    for precision in (pkg.PDN_FP64, pkg.PDN_FP32_FORCE):
        s = pkg.Solver(w, precision=precision)
        pkg.pdn_set_state(s.ctx, *st)
        f = pkg.pdn_internal_force(s.ctx)
        s.step(1)
        h, _ = pkg.pdn_get_history(s.ctx)
        out.append((f, h.astype(np.float64)))
        s.close()
    (f64, h64), (f32, h32) = out
    assert np.abs(f32 - f64).max() <= 1e-4 * np.abs(f64).max()
    assert np.abs(h32 - h64).max() <= 1e-4 * np.abs(h64).max()
    if state == "damaging":
        assert (h64.reshape(7, 8, -1)[:4] > 1.0).any()


def test_local_repetition_equals_full(pkg, monkeypatch):
    monkeypatch.setenv("PDN_HEX_VARIANT", "0")
    w = _plate(95, 129, 16)
    Lx, Ly, H = w.plate.dims
    out = []
    for full in ("0", "1"):
        monkeypatch.setenv("PDN_FULL_REPEAT", full)
        s = pkg.Solver(w)
        # a light fast striker that rebounds within the run: nodes are released
        pkg.pdn_set_impactor(s.ctx, 8.0, 2e-8, (0.5 * Lx, 0.5 * Ly, H + 8.0005), (0.0, 0.0, -20000.0))
        s.step(1500)
        out.append(s.state()[:2] + pkg.pdn_get_history(s.ctx) + (s.info()["n_repeats"],))
        s.close()
    assert out[0][4] == out[1][4] > 0
    for a, b in zip(out[0][:4], out[1][:4]):
        assert np.array_equal(a, b)
