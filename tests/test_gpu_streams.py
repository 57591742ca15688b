"""A context on a stream that does not block on the default stream (any torch
side stream): nothing orders the two, so every upload the kernels read has to
be complete or on the context's own stream.  Whole runs equal those on the
library's own stream bit for bit (the same kernels in the same order)."""
import numpy as np
import pytest

import pdn_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2301_05552_gb300 as p
    p.lib()
    return p


def _plate(nx, ny, plies, fp64, skew=False):
    w = pi.damage_fp32_plate(nx=nx, ny=ny, plies=plies, Lx=0.5 * nx, Ly=0.5 * ny, H=0.275 * plies, fp64=fp64)
    if skew:
        Lx, Ly, _ = w.plate.dims
        x, y = w.plate.X[0].copy(), w.plate.X[1].copy()
        bump = np.sin(np.pi * x / Lx) * np.sin(np.pi * y / Ly)
        w.plate.X[0] = x + 0.1 * bump * np.sin(9.0 * y / Ly)
        w.plate.X[1] = y + 0.1 * bump * np.cos(7.0 * x / Lx)
    return w


@pytest.mark.parametrize("fp64,skew", [(True, False), (False, False), (False, True)])
def test_created_and_stepped_on_a_side_stream(pkg, monkeypatch, fp64, skew):
    import torch
    monkeypatch.setenv("PDN_HEX_VARIANT", "0")
    out = []
    for stream in (None, torch.cuda.Stream().cuda_stream):
        # a context with other ply angles first: its table is what a late
        # upload would leave in reused memory
        pkg.Solver(_plate(13, 9, 6, fp64, skew), stream=stream).close()
        s = pkg.Solver(_plate(33, 27, 4, fp64, skew), stream=stream)
        s.step(2000)  # contact after about 1,000
        out.append(s.state()[:2] + pkg.pdn_get_contact(s.ctx))
        s.close()
    assert np.abs(out[0][0]).max() > 0.0
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("fp64", [True, False])
def test_state_installed_on_a_side_stream(pkg, monkeypatch, fp64):
    import torch
    monkeypatch.setenv("PDN_HEX_VARIANT", "0")
    w = _plate(65, 49, 8, fp64)  # 42,900 nodes: copies of a megabyte, several staging buffers each
    Lx, Ly, _ = w.plate.dims
    states = [pi.seeded_state(w.plate, k, amp=0.02, vamp=300.0, dimple=(0.5 * Lx, 0.5 * Ly, 0.12, 3.0)) for k in (7, 8)]
    out = []
    for stream in (None, torch.cuda.Stream().cuda_stream):
        s = pkg.Solver(w, stream=stream)
        got = []
        for d, v in states:  # the second over the first's leftovers
            pkg.pdn_set_state(s.ctx, d, v)
            got += [pkg.pdn_internal_force(s.ctx), pkg.pdn_get_acceleration(s.ctx)]
        s.step(40)
        out.append(got + list(s.state()[:2]))
        s.close()
    for a, b in zip(*out):
        assert np.abs(a).max() > 0.0 and np.array_equal(a, b)


@pytest.mark.parametrize("schedule", ["0,0", "1,0"])
def test_batch_on_a_side_stream(pkg, monkeypatch, schedule):
    """Plate records, tile lists (one per candidate tile size while the batch
    is tuned) and counters uploaded for the batch's stream, its own (which
    never blocks on the default stream) or the caller's."""
    import torch
    monkeypatch.setenv("PDN_BATCH_SCHEDULE", schedule)
    ws = [_plate(33, 27, 4, False), _plate(13, 9, 6, False), _plate(21, 40, 8, False)]
    out = []
    for stream in (None, torch.cuda.Stream().cuda_stream):
        b = pkg.pdn_batch_init([w.plate for w in ws], [w.material for w in ws], stream=stream)
        for w, ctx in zip(ws, b.plates):
            Lx, Ly, _ = w.plate.dims
            pkg.pdn_set_impactor(ctx, *w.impactor())
            pkg.pdn_set_state(ctx, *pi.seeded_state(w.plate, 7, amp=0.02, vamp=300.0,
                                                    dimple=(0.5 * Lx, 0.5 * Ly, 0.12, 1.5)))
        pkg.pdn_batch_step(b, 100)
        out.append([x for ctx in b.plates for x in pkg.pdn_get_state(ctx)[:2]])
        b.close()
    for a, c in zip(*out):
        assert np.abs(a).max() > 0.0 and np.array_equal(a, c)
