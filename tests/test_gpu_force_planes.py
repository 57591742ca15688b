"""Element forces as planes (component x rank x node) against slots of 16
bytes per node and rank (PDN_PLANES=0, read when a context is created): the
same forces summed in the same order, so whole runs are bitwise equal.  Plates
whose node counts are no multiple of a warp's line, with and without
interfaces, boxes and general hexes, layered and other numberings with
consecutive nodes along x, in a batch; and the rule itself (three quarters of
the hexes follow their predecessor)."""
import dataclasses

import numpy as np
import pytest

import pdn_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2301_05552_gb300 as p
    p.lib()
    return p


def _rows_permuted(w, nx):
    """The plate with its rows of nodes along x in another order: each row's
    ids stay consecutive, the numbering is no longer layered."""
    P = w.plate
    rows = P.n_nodes // (nx + 1)
    perm_rows = np.random.default_rng(5).permutation(rows)
    perm = (perm_rows[:, None] * (nx + 1) + np.arange(nx + 1)).ravel()  # new id of old node
    inv = np.empty_like(perm)
    inv[perm] = np.arange(P.n_nodes)
    plate = dataclasses.replace(P, X=np.ascontiguousarray(P.X[:, inv]), hex=perm[P.hex].astype(np.int32),
                                coh=perm[P.coh].astype(np.int32), fixed=np.ascontiguousarray(P.fixed[inv]),
                                surf=np.sort(perm[P.surf]).astype(np.int32))
    return dataclasses.replace(w, plate=plate)


def _skewed(w):
    """Node columns moved in plane: general hexes, interfaces no rectangles."""
    Lx, Ly, _ = w.plate.dims
    x, y = w.plate.X[0].copy(), w.plate.X[1].copy()
    bump = np.sin(np.pi * x / Lx) * np.sin(np.pi * y / Ly)
    w.plate.X[0] = x + 0.1 * bump * np.sin(9.0 * y / Ly)
    w.plate.X[1] = y + 0.1 * bump * np.cos(7.0 * x / Lx)
    return w


def _damage(nx, ny, plies, **kw):
    return pi.damage_fp32_plate(nx=nx, ny=ny, plies=plies, Lx=0.5 * nx, Ly=0.5 * ny, H=0.275 * plies, steps=150, **kw)


def _cases():
    plain = pi.make_plate(11.5, 8.5, 1.5, 23, 17, [0.0, 90.0, 0.0], 1, cohesive=False)
    plain_w = dataclasses.replace(_damage(23, 17, 4), plate=plain)
    return [("layered_33x13x4", _damage(33, 13, 4)), ("narrow_4x7x6", _damage(4, 7, 6)),
            ("rows_permuted_21x14x4", _rows_permuted(_damage(21, 14, 4), 21)), ("skewed_19x12x4", _skewed(_damage(19, 12, 4))),
            ("no_interfaces_23x17x3", plain_w)]


def _run(pkg, w, planes, monkeypatch):
    monkeypatch.setenv("PDN_HEX_VARIANT", "0")
    monkeypatch.setenv("PDN_PLANES", "1" if planes else "0")
    s = pkg.Solver(w, precision=pkg.PDN_FP32_FORCE)
    Lx, Ly, _ = w.plate.dims
    pkg.pdn_set_state(s.ctx, *pi.seeded_state(w.plate, 7, amp=0.02, vamp=300.0, dimple=(0.5 * Lx, 0.5 * Ly, 0.12, 1.5)))
    f = pkg.pdn_internal_force(s.ctx)
    s.step(150)
    d, v, _ = s.state()
    hist, r = pkg.pdn_get_history(s.ctx)
    s.close()
    return f, d, v, hist, r


@pytest.mark.parametrize("name,w", _cases(), ids=[c[0] for c in _cases()])
def test_planes_equal_slots(pkg, monkeypatch, name, w):
    a, b = _run(pkg, w, True, monkeypatch), _run(pkg, w, False, monkeypatch)
    assert np.abs(b[0]).max() > 0.0 and np.isfinite(b[1]).all()
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_planes_equal_slots_in_a_batch(pkg, monkeypatch):
    monkeypatch.setenv("PDN_BATCH_SCHEDULE", "0")
    ws = [_damage(33, 13, 4), _damage(9, 10, 6)]
    out = []
    for planes in ("1", "0"):
        monkeypatch.setenv("PDN_PLANES", planes)
        b = pkg.pdn_batch_init([w.plate for w in ws], [w.material for w in ws])
        for w, ctx in zip(ws, b.plates):
            Lx, Ly, H = w.plate.dims
            pkg.pdn_set_impactor(ctx, 4.0, 1e-5, (0.5 * Lx, 0.5 * Ly, H + 4.001), (0.0, 0.0, -3000.0))
            pkg.pdn_set_state(ctx, *pi.seeded_state(w.plate, 7, amp=0.02, vamp=300.0,
                                                    dimple=(0.5 * Lx, 0.5 * Ly, 0.12, 1.5)))
        pkg.pdn_batch_step(b, 100)
        out.append([pkg.pdn_get_state(ctx)[:2] for ctx in b.plates])
        b.close()
    for (d1, v1), (d0, v0) in zip(*out):
        assert np.abs(d0).max() > 0.0
        assert np.array_equal(d1, d0) and np.array_equal(v1, v0)
