"""The autotuner times the hex kernels that exist: two register budgets for
FP32 boxes, nothing where one kernel runs (general hexes, boxes with the
learned law, FP64).  PDN_HEX_VARIANT fixes any of its numbers without timing."""
import numpy as np
import pytest

import pdn_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2301_05552_gb300 as p
    p.lib()
    return p


def _plate(fp64=False, skew=False):
    w = pi.damage_fp32_plate(nx=21, ny=17, plies=4, Lx=10.5, Ly=8.5, H=1.1, fp64=fp64)
    if skew:
        Lx, Ly, _ = w.plate.dims
        x, y = w.plate.X[0].copy(), w.plate.X[1].copy()
        bump = np.sin(np.pi * x / Lx) * np.sin(np.pi * y / Ly)
        w.plate.X[0] = x + 0.1 * bump * np.sin(9.0 * y / Ly)
        w.plate.X[1] = y + 0.1 * bump * np.cos(7.0 * x / Lx)
    return w


def _timed(info):
    return {k for k, ms in enumerate(info["tune_ms"]) if ms > 0.0}


@pytest.mark.parametrize("kind", ["boxes", "general", "fp64", "learned"])
def test_times_the_kernels_that_exist(pkg, monkeypatch, kind):
    monkeypatch.delenv("PDN_HEX_VARIANT", raising=False)
    w = _plate(kind == "fp64", kind == "general")
    s = pkg.Solver(w)
    law = None
    if kind == "learned":
        law = pkg.pdn_sur_create(w.material, 0.41, seed=0)
        pkg.pdn_sur_generate(law, 2000, 8, 0.01, 0.4, 0.9, seed=1)
        pkg.pdn_set_surrogate(s.ctx, law, 0.9)
    s.step(3)
    info = s.info()
    assert _timed(info) == ({0, 3} if kind == "boxes" else set())
    assert info["hex_variant"] in ({0, 3} if kind == "boxes" else {0})
    s.close()


@pytest.mark.parametrize("variant", range(8))
def test_every_variant_number_is_accepted(pkg, monkeypatch, variant):
    monkeypatch.setenv("PDN_COH_PAIRS", "0")
    out = []
    for v in (variant, variant // 4 * 4):
        monkeypatch.setenv("PDN_HEX_VARIANT", str(v))
        w = _plate()
        s = pkg.Solver(w)
        pkg.pdn_set_state(s.ctx, *pi.seeded_state(w.plate, 7, amp=0.02, vamp=300.0, dimple=(5.25, 4.25, 0.12, 1.5)))
        s.step(20)
        assert s.info()["hex_variant"] == v and not _timed(s.info())
        out.append(s.state()[0])
        s.close()
    if variant != 3:  # another register budget may contract differently
        assert np.array_equal(*out)
    assert np.abs(out[0] - out[1]).max() <= 1e-4 * np.abs(out[1]).max()
