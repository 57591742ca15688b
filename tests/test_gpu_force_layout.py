"""Which contexts keep element forces as planes (pdn_info.planes): FP32, no
column sweep, and three quarters of the hexes with each corner one node id
after their predecessor's.  Both sides of that line (rows of three and of four
hexes), the conditions one by one, PDN_PLANES=0, and the arms that
test_gpu_force_planes.py compares; and the learned law's kernel with planes
against slots, bit for bit."""
import dataclasses

import numpy as np
import pytest

import pdn_inputs as pi
from test_gpu_force_planes import _cases, _damage

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2301_05552_gb300 as p
    p.lib()
    return p


def _planes(pkg, w, **kw):
    s = pkg.Solver(w, **kw)
    p = s.info()["planes"]
    s.close()
    return p


def _hexes_shuffled(w):
    P = w.plate
    perm = np.random.default_rng(2).permutation(P.n_hex)
    return dataclasses.replace(w, plate=dataclasses.replace(P, hex=np.ascontiguousarray(P.hex[perm]),
                                                            ply_of_hex=np.ascontiguousarray(P.ply_of_hex[perm])))


@pytest.mark.parametrize("name,w", _cases(), ids=[c[0] for c in _cases()])
def test_the_compared_arms_differ(pkg, monkeypatch, name, w):
    for switch, want in (("1", 1), ("0", 0)):
        monkeypatch.setenv("PDN_PLANES", switch)
        assert _planes(pkg, w, precision=pkg.PDN_FP32_FORCE) == want


@pytest.mark.parametrize("nx,want", [(1, 0), (2, 0), (3, 0), (4, 1), (5, 1)])
def test_rule_by_row_length(pkg, monkeypatch, nx, want):
    monkeypatch.delenv("PDN_PLANES", raising=False)
    assert _planes(pkg, _damage(nx, 9, 4), precision=pkg.PDN_FP32_FORCE) == want


def test_conditions(pkg, monkeypatch):
    monkeypatch.delenv("PDN_PLANES", raising=False)
    w = _damage(33, 13, 4)
    assert _planes(pkg, w, precision=pkg.PDN_FP32_FORCE) == 1
    assert _planes(pkg, w, precision=pkg.PDN_FP64) == 0
    assert _planes(pkg, _hexes_shuffled(w), precision=pkg.PDN_FP32_FORCE) == 0
    monkeypatch.setenv("PDN_SWEEP", "1")
    assert _planes(pkg, w, precision=pkg.PDN_FP32_FORCE) == 0


def test_learned_law_planes_equal_slots(pkg, monkeypatch):
    monkeypatch.setenv("PDN_HEX_VARIANT", "0")
    w = _damage(33, 13, 6)
    law = pkg.pdn_sur_create(w.material, 0.41, seed=0)
    pkg.pdn_sur_generate(law, 4000, 8, 0.01, 0.4, 0.9, seed=1)
    pkg.pdn_sur_train(law, 100, 1024, 2e-3, seed=2)
    Lx, Ly, _ = w.plate.dims
    st = pi.seeded_state(w.plate, 7, amp=0.02, vamp=300.0, dimple=(0.5 * Lx, 0.5 * Ly, 0.12, 1.5))
    out = []
    for switch in ("1", "0"):
        monkeypatch.setenv("PDN_PLANES", switch)
        s = pkg.Solver(w, precision=pkg.PDN_FP32_FORCE)
        assert s.info()["planes"] == int(switch)
        pkg.pdn_set_surrogate(s.ctx, law, 0.9)
        pkg.pdn_set_state(s.ctx, *st)
        f = pkg.pdn_internal_force(s.ctx)
        s.step(100)
        out.append((f,) + s.state()[:2] + tuple(pkg.pdn_get_history(s.ctx)))
        s.close()
    for a, b in zip(*out):
        assert np.abs(a).max() > 0.0 and np.array_equal(a, b)
