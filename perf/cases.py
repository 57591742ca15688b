"""The work this library is run for, as cases that can be timed and compared.

A case is one call pattern of a program that uses the library: a window of
explicit impact steps on one plate (the laminates, materials and strikers of
``pdn_inputs``), on a batch of plates, or with the learned law; one
evaluation of the internal force; one stretch of training of the learned law.
``listed`` names the cases, ``draw`` gives others of the same ranges.

Impact windows.  ``prepare`` sets the plate up and runs the impact for
``preroll`` steps, as a program has before the window starts: the striker
touches the plate, the launch variant is chosen and the graph is captured.
``run`` advances ``steps`` more steps and reads the result: in FP64 the whole
state (displacement, velocity, striker, contact set and reactions); in FP32
element arithmetic the displacement in single precision and the striker, which
is what such a run is read for.  (FP32 element forces leave rounding noise of
the mesh's highest frequency in the velocities, about 1e-3 of their size after
a few hundred steps, while displacements keep six digits.)  Calling ``run``
again on the same state continues the impact.

The seed gives the striker's mass, speed and point of impact, the strengths
of the plies and, where a displacement field is an input, that field.
"""
import functools

import numpy as np
import torch

import paper_2301_05552_gb300 as pdn
import pdn_inputs as pi


# ---------------------------------------------------------------------------
# The cases.

def listed():
    return [
        # the smallest call: internal force of a coupon-sized block of hexes
        # from device buffers, FP64, for a caller that steps by itself
        dict(name="force_block_fp64", kind="force_block", nx=13, ny=17, plies=5, fp64=True),
        # the 40 x 40 x 4 mm elastic plate in FP64 (8,192 hexes): a step is a
        # chain of short launches
        dict(name="impact_plain_fp64", kind="impact", plate="plain", nx=32, ny=32, plies=8, epp=1, fp64=True,
             preroll=240, steps=160),
        # a laminate with damage and interfaces in FP64 element arithmetic
        dict(name="impact_damage_fp64", kind="impact", plate="damage", nx=48, ny=72, plies=16, epp=1, fp64=True,
             preroll=64, steps=32),
        # the 100 x 150 mm, 16-ply laminate (393,216 hexes), FP32 elements
        dict(name="impact_damage_fp32", kind="impact", plate="damage", nx=128, ny=192, plies=16, epp=1, fp64=False,
             preroll=1600, steps=192),
        # the same laminate at 400 x 600 x 32 (7.68 M hexes): memory and
        # arithmetic, little latency
        dict(name="impact_large_fp32", kind="impact", plate="damage", nx=400, ny=600, plies=16, epp=2, fp64=False,
             preroll=640, steps=192),
        # the AS4/8552 drop-weight coupon (228,528 hexes): frame, clamps,
        # gravity, dissipative integrator, node releases
        dict(name="impact_coupon_fp32", kind="impact", plate="coupon", nx=207, ny=138, plies=8, epp=1, fp64=False,
             preroll=640, steps=192),
        # the coupon divided once on the device (1.83 M hexes, a numbering
        # that is not layered)
        dict(name="impact_divided_fp32", kind="impact", plate="divided", nx=207, ny=138, plies=8, epp=1, fp64=False,
             preroll=448, steps=96),
        # a laminate whose hexes are no boxes (node columns moved in plane):
        # the general element, odd sizes
        dict(name="impact_skewed_fp32", kind="impact", plate="skewed", nx=61, ny=95, plies=12, epp=1, fp64=False,
             preroll=192, steps=96),
        # many plates in one launch (a design study): 24 plates of 8 thousand
        # to 100 thousand hexes
        dict(name="batch_fp32", kind="batch", plates=24, hex_min=8000, hex_max=100000, preroll=64, steps=64),
        # the learned law in the step, after its training
        dict(name="impact_learned_fp32", kind="learned", nx=96, ny=144, plies=16, preroll=256, steps=64),
        # internal force of a laminate at a given displacement (residual
        # checks, coupling to another integrator), to the host
        dict(name="force_plate_fp32", kind="force", nx=127, ny=191, plies=16, fp64=False),
        # training of the learned law: 256 Adam steps of 8,192 points
        dict(name="train_learned", kind="train", paths=60000, batch=8192, iters=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(np.exp(rng.uniform(np.log(lo), np.log(hi)))))


def draw(rng):
    kind = rng.choice(["impact", "impact", "impact", "impact", "impact", "force_block", "force", "batch", "learned",
                       "train"])
    if kind == "force_block":
        plies = rng.randint(2, 12)
        nx = rng.randint(4, 24)
        ny = max(2, min(rng.randint(4, 30), 8192 // (nx * plies), 16384 // ((nx + 1) * (plies + 1)) - 1))
        return dict(kind=kind, nx=nx, ny=ny, plies=plies, fp64=rng.random() < 0.5)
    if kind == "force":
        nx = _log_int(rng, 20, 260)
        return dict(kind=kind, nx=nx, ny=rng.randint(nx, 2 * nx), plies=2 * rng.randint(3, 9), fp64=rng.random() < 0.3)
    if kind == "batch":
        return dict(kind=kind, plates=rng.randint(6, 28), hex_min=8000, hex_max=_log_int(rng, 20000, 120000),
                    preroll=64, steps=rng.randint(33, 90))
    if kind == "learned":
        nx = _log_int(rng, 24, 128)
        return dict(kind=kind, nx=nx, ny=nx * 3 // 2 + rng.randint(0, 3), plies=2 * rng.randint(4, 8), preroll=128,
                    steps=rng.randint(32, 80))
    if kind == "train":
        return dict(kind=kind, paths=rng.randint(20000, 80000), batch=128 * rng.randint(8, 96),
                    iters=rng.randint(64, 300))
    plate = rng.choice(["plain", "damage", "damage", "damage", "coupon", "divided", "skewed"])
    fp64 = plate == "plain" or (plate in ("damage", "skewed") and rng.random() < 0.3)
    epp = 1
    if plate == "plain":
        nx, ny, plies = rng.randint(10, 64), rng.randint(10, 64), 8
    elif plate in ("coupon", "divided"):
        nx = _log_int(rng, 40, 207)
        ny, plies = max(28, nx * 2 // 3 + rng.randint(-2, 2)), 8
    elif plate == "skewed":
        nx = _log_int(rng, 16, 40 if fp64 else 96)
        ny, plies = nx * 3 // 2 + rng.randint(-3, 3), 2 * rng.randint(4, 8)
    else:
        nx = _log_int(rng, 16, 60 if fp64 else 320)
        ny, plies, epp = nx * 3 // 2 + rng.randint(-5, 5), 2 * rng.randint(4, 10), rng.choice([1, 1, 2])
    return dict(kind="impact", plate=plate, nx=nx, ny=ny, plies=plies, epp=epp, fp64=fp64,
                preroll=rng.randint(96, 400), steps=rng.randint(40, 200))


# ---------------------------------------------------------------------------
# Inputs.  Meshes depend on the case alone and are kept between calls, as a
# program that runs many impacts on one mesh keeps it.

SPACING = 100.0 / 128.0  # in-plane element size of the 100 x 150 mm laminate
T_PLY = 0.275            # its ply thickness (4.4 mm / 16)


def _angles(plies):
    if plies % 2 == 0:
        return pi.seeded_quasi_isotropic_layup(plies, 0)
    return [0.0, 90.0, 45.0, -45.0][:plies] + [0.0] * max(0, plies - 4)


@functools.lru_cache(maxsize=32)
def _mesh(plate, nx, ny, plies, epp):
    if plate == "plain":
        return pi.make_plate(nx * 1.25, ny * 1.25, 4.0, nx, ny, [0.0, 90.0, 0.0, 90.0, 90.0, 0.0, 90.0, 0.0], 1,
                             cohesive=False)
    if plate == "block":
        return pi.make_plate(nx * SPACING, ny * SPACING, plies * T_PLY, nx, ny, _angles(plies), 1, cohesive=False)
    if plate in ("coupon", "divided"):
        return pi.reduced_as4_frame_plate(nx=nx, ny=ny, fp64=False).plate
    h = SPACING if epp == 1 else 0.25  # two elements per ply: the 0.25 mm mesh of the refined laminate
    mesh = pi.make_plate(nx * h, ny * h, plies * T_PLY, nx, ny, _angles(plies), epp, cohesive=True)
    if plate == "skewed":
        # node columns moved in plane by a smooth field: hexes stay convex,
        # coincident interface nodes stay coincident, plies stay flat
        Lx, Ly, _ = mesh.dims
        x, y = mesh.X[0].copy(), mesh.X[1].copy()
        bump = np.sin(np.pi * x / Lx) * np.sin(np.pi * y / Ly)
        mesh.X[0] = x + 0.25 * h * bump * np.sin(9.0 * y / Ly)
        mesh.X[1] = y + 0.25 * h * bump * np.cos(7.0 * x / Lx)
    return mesh


def _striker(mesh, r, mass, speed, gap):
    """Radius, mass, centre and velocity: mass and speed within 10 %, the
    point of impact within 1 mm of the plate's centre."""
    Lx, Ly, H = mesh.dims
    dx, dy = r.uniform(-1.0, 1.0, 2)
    radius = 8.0
    return (radius, mass * r.uniform(0.9, 1.1), (0.5 * Lx + dx, 0.5 * Ly + dy, H + radius + gap),
            (0.0, 0.0, -speed * r.uniform(0.9, 1.1)))


def _smooth_field(mesh, r):
    """A displacement [3, n_nodes]: two smooth waves that vanish at the plate's
    edges, with a part linear in z, and differences of neighbouring nodes of
    1e-6 mm that open and shear the interfaces; well below damage onset."""
    Lx, Ly, H = mesh.dims
    x, y, z = mesh.X
    d = r.normal(size=mesh.X.shape) * 1e-6
    amp = 1e-4 * min(Lx, Ly)
    for _ in range(2):
        kx, ky = r.integers(1, 4, size=2)
        s = np.sin(kx * np.pi * x / Lx) * np.sin(ky * np.pi * y / Ly)
        for c in range(3):
            a, b = r.normal(size=2)
            d[c] += amp * (0.1 if c < 2 else 1.0) * s * (a + 0.02 * b * (z / H - 0.5))
    for c in range(3):
        d[c, ((mesh.fixed >> c) & 1).astype(bool)] = 0.0
    return d


def _csr(hexes, n_nodes):
    nodes = hexes.ravel().astype(np.int64)
    order = np.lexsort((np.arange(nodes.size), nodes))
    row = np.concatenate([[0], np.cumsum(np.bincount(nodes, minlength=n_nodes))])
    return row.astype(np.int32), order.astype(np.int32)


def _learned_law(seed, paths, batch, iters):
    lc = (SPACING * SPACING * T_PLY) ** (1.0 / 3.0)
    law = pdn.pdn_sur_create(pi.material_im7_like_config(t_ply=T_PLY, seed=0), lc, seed=0)
    pdn.pdn_sur_generate(law, paths, 8, 0.01, 0.4, 0.9, seed=seed)
    if iters:
        pdn.pdn_sur_train(law, iters, batch, 2e-3, seed=1)
    return law


def prepare(case, seed):
    r = np.random.default_rng(seed)
    k = case["kind"]
    if k in ("impact", "learned"):
        plate = case.get("plate", "damage")
        mesh = _mesh(plate, case["nx"], case["ny"], case["plies"], case.get("epp", 1))
        fp64 = case.get("fp64", False)
        opt = dict(precision=pdn.PDN_FP64 if fp64 else pdn.PDN_FP32_FORCE)
        state = dict(case, fp64=fp64)
        if plate in ("coupon", "divided"):
            mat = pi.material_as4_8552(t_ply=4 * 0.181, seed=int(seed))
            opt.update(phi=1.033, gravity=(0.0, 0.0, -9810.0))
            strike = _striker(mesh, r, 5.0e-3, 2780.0, 0.002)
        elif plate == "plain":
            mat = pi.material_im7_like_config(t_ply=0.5, spread=0.0)
            opt.update(damage_on=False, plasticity_on=False)
            strike = _striker(mesh, r, 1.0e-3, 1000.0, 0.005)
        else:
            mat = pi.material_im7_like_config(t_ply=T_PLY, seed=int(seed))
            strike = _striker(mesh, r, 5.5e-3, 4000.0 if case.get("epp", 1) == 2 else 3000.0, 0.001)
        if plate == "divided":
            fine = pdn.pdn_mesh_multiply(mesh, 1)
            ctx = pdn.pdn_init_refined(fine, mat, **opt)
            fine.close()
        else:
            ctx = pdn.pdn_init_mesh(mesh, mat, **opt)
        pdn.pdn_set_impactor(ctx, *strike)
        if k == "learned":
            state["law"] = _learned_law(5, 40000, 8192, 1500)
            pdn.pdn_set_surrogate(ctx, state["law"], 0.9)
        pdn.pdn_step(ctx, case["preroll"])
        state["ctx"] = ctx
        return state
    if k == "batch":
        cases = pi.batch_plates(case["plates"], seed=0, hex_min=case["hex_min"], hex_max=case["hex_max"])
        batch = pdn.pdn_batch_init([w.plate for w in cases],
                                   [dict(w.material, seed=int(seed) * 1000 + p) for p, w in enumerate(cases)])
        for w, ctx in zip(cases, batch.plates):
            pdn.pdn_set_impactor(ctx, *_striker(w.plate, r, w.mass, w.speed, 0.001))
        pdn.pdn_batch_step(batch, case["preroll"])
        return dict(case, batch=batch)
    if k == "force":
        mesh = _mesh("damage", case["nx"], case["ny"], case["plies"], 1)
        ctx = pdn.pdn_init_mesh(mesh, pi.material_im7_like_config(t_ply=T_PLY, seed=int(seed)),
                                precision=pdn.PDN_FP64 if case["fp64"] else pdn.PDN_FP32_FORCE)
        pdn.pdn_set_state(ctx, _smooth_field(mesh, r), np.zeros_like(mesh.X))
        return dict(case, ctx=ctx)
    if k == "force_block":
        mesh = _mesh("block", case["nx"], case["ny"], case["plies"], 1)
        row, col = _csr(mesh.hex, mesh.n_nodes)
        up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        d = _smooth_field(mesh, r)
        return dict(case, n=(mesh.n_nodes, mesh.n_hex), args=tuple(map(up, (mesh.hex, mesh.ply_of_hex, mesh.X, d))),
                    csr=(up(row), up(col)), mat=pi.material_im7_like_config(t_ply=T_PLY, seed=int(seed)),
                    angles=mesh.ply_angle_deg, f=torch.zeros((3, mesh.n_nodes), dtype=torch.float64, device="cuda"))
    if k == "train":
        return dict(case, law=_learned_law(int(seed), case["paths"], 0, 0), seed=int(seed))
    raise ValueError(k)


# ---------------------------------------------------------------------------
# One pass.

def _striker_out(imp, dtype):
    return np.concatenate([imp["centre"], imp["velocity"]]).astype(dtype)


def run(state):
    k = state["kind"]
    if k in ("impact", "learned"):
        ctx = state["ctx"]
        pdn.pdn_step(ctx, state["steps"])
        d, v, imp = pdn.pdn_get_state(ctx)
        if state["fp64"]:
            active, reaction = pdn.pdn_get_contact(ctx)
            return dict(d=d, v=v, striker=_striker_out(imp, np.float64), active=active, reaction=reaction)
        return dict(d=d.astype(np.float32), striker=_striker_out(imp, np.float32))
    if k == "batch":
        pdn.pdn_batch_step(state["batch"], state["steps"])
        out = []
        for ctx in state["batch"].plates:
            d, v, imp = pdn.pdn_get_state(ctx)
            out.append(np.concatenate([d.ravel(), _striker_out(imp, np.float64)]).astype(np.float32))
        return out
    if k == "force":
        f = pdn.pdn_internal_force(state["ctx"])
        return f if state["fp64"] else f.astype(np.float32)
    if k == "force_block":
        hexes, ply, X, d = state["args"]
        pdn.pdn_internal_force_noalloc(*state["n"], hexes, ply, X, d, None, *state["csr"], state["mat"], state["angles"],
                                       pdn.PDN_FP64 if state["fp64"] else pdn.PDN_FP32_FORCE, True, True, state["f"])
        return state["f"] if state["fp64"] else state["f"].float()
    if k == "train":
        loss = pdn.pdn_sur_train(state["law"], state["iters"], state["batch"], 2e-3, seed=state["seed"])
        params, scaling = pdn.pdn_sur_get_params(state["law"])
        return dict(params=params, scaling=scaling, loss=loss.astype(np.float32))
    raise ValueError(k)


# ---------------------------------------------------------------------------
# What a pass cannot do without.

def _counts(plate, nx, ny, plies, epp):
    """Nodes, hexes and interface elements of a case's mesh."""
    if plate == "plain":
        layers, inter = 9, 0
    elif plate == "block":
        layers, inter = plies + 1, 0
    else:
        ang = [45.0, 0.0, -45.0, 90.0, 90.0, -45.0, 0.0, 45.0] if plate in ("coupon", "divided") else _angles(plies)
        inter = sum(a != b for a, b in zip(ang, ang[1:]))
        layers = plies * epp + 1 + inter
    if plate == "divided":
        nx, ny, layers = 2 * nx, 2 * ny, 2 * plies * epp + 1 + inter
        return layers * (nx + 1) * (ny + 1), nx * ny * plies * epp * 2, nx * ny * inter
    return layers * (nx + 1) * (ny + 1), nx * ny * plies * epp, nx * ny * inter


# Multiply-adds of one hex8 over its eight Gauss points: displacement
# gradient, Green strain, stress in ply axes, loading functions, first
# Piola-Kirchhoff stress and the nodal forces, about 150 per point, and
# twice that in operations; an interface point is about 40 operations.
HEX_FLOPS, PAIR_FLOPS = 2 * 150 * 8, 40


def _step_work(nn, nh, nc, fp64):
    """One step: displacement and velocity (FP64) read and written, mass and
    constraint flags, reference coordinates, connectivity, ply and the
    pristine flag of each hex, an interface's connectivity and thresholds."""
    t = 8 if fp64 else 4
    return (nn * (96 + t + 1 + 3 * t) + nh * (32 + 2) + nc * (32 + 4 * t), nh * HEX_FLOPS + nc * 4 * PAIR_FLOPS)


def work(case):
    k = case["kind"]
    if k in ("impact", "learned"):
        fp64 = case.get("fp64", False)
        nn, nh, nc = _counts(case.get("plate", "damage"), case["nx"], case["ny"], case["plies"], case.get("epp", 1))
        b, f = _step_work(nn, nh, nc, fp64)
        if k == "learned":
            f += nh * 8 * 18944  # the network's products
        return dict(bytes=case["steps"] * b + nn * (24 if not fp64 else 48), flops=case["steps"] * f)
    if k == "batch":
        b = f = out = 0.0
        for w in pi.batch_plates(case["plates"], seed=0, hex_min=case["hex_min"], hex_max=case["hex_max"]):
            p = w.plate
            bb, ff = _step_work(p.n_nodes, p.n_hex, p.n_coh, False)
            b, f, out = b + bb, f + ff, out + 24 * p.n_nodes
        return dict(bytes=case["steps"] * b + out, flops=case["steps"] * f)
    if k in ("force", "force_block"):
        nn, nh, nc = _counts("damage" if k == "force" else "block", case["nx"], case["ny"], case["plies"], 1)
        t = 8 if (case["fp64"] or k == "force_block") else 4
        return dict(bytes=nn * (2 * 3 * t + 24) + nh * 33 + nc * 32, flops=nh * HEX_FLOPS + nc * 4 * PAIR_FLOPS)
    if k == "train":
        # forward, backward to the activations and to the weights
        return dict(bytes=case["iters"] * case["batch"] * 2 * 40 + 9674 * 4, flops=case["iters"] * case["batch"] * 3 * 18944)
    raise ValueError(k)


# ---------------------------------------------------------------------------
# Reference values in 64 bits.

_XI = np.array([[-1, -1, -1], [1, -1, -1], [1, 1, -1], [-1, 1, -1], [-1, -1, 1], [1, -1, 1], [1, 1, 1], [-1, 1, 1]])


def _elastic_force(mesh, mat, d):
    """Internal force of undamaged hexes (total Lagrangian, Green strain, linear
    law in ply axes, 2 x 2 x 2 points) and undamaged flat interfaces, torch
    FP64."""
    dev = torch.device("cuda")
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    X, U = t(mesh.X.T), t(d.T)
    hexes = torch.as_tensor(mesh.hex, dtype=torch.int64, device=dev)
    f = torch.zeros_like(U)
    H = np.array([[1 / mat["E1"], -mat["nu12"] / mat["E1"], -mat["nu13"] / mat["E1"]],
                  [-mat["nu12"] / mat["E1"], 1 / mat["E2"], -mat["nu23"] / mat["E2"]],
                  [-mat["nu13"] / mat["E1"], -mat["nu23"] / mat["E2"], 1 / mat["E3"]]])
    C = t(np.linalg.inv(H))
    ang = t(np.radians(mesh.ply_angle_deg))[torch.as_tensor(mesh.ply_of_hex, dtype=torch.int64, device=dev)]
    R = torch.zeros((hexes.shape[0], 3, 3), dtype=torch.float64, device=dev)  # columns: ply axes
    R[:, 0, 0], R[:, 1, 0], R[:, 0, 1], R[:, 1, 1], R[:, 2, 2] = ang.cos(), ang.sin(), -ang.sin(), ang.cos(), 1.0
    Xe, Ue = X[hexes], U[hexes]
    fe = torch.zeros_like(Ue)
    eye = torch.eye(3, dtype=torch.float64, device=dev)
    for g in _XI / np.sqrt(3.0):
        dN = t(np.stack([0.125 * _XI[:, k] * np.prod([1 + g[m] * _XI[:, m] for m in range(3) if m != k], axis=0)
                         for k in range(3)], axis=1))
        J = torch.einsum("eai,ak->eik", Xe, dN)
        G = torch.einsum("ak,ekj->eaj", dN, torch.linalg.inv(J))
        D = torch.einsum("eai,eaj->eij", Ue, G)
        E = 0.5 * (D + D.transpose(1, 2) + D.transpose(1, 2) @ D)
        P = R.transpose(1, 2) @ E @ R
        S = torch.zeros_like(P)
        S[:, [0, 1, 2], [0, 1, 2]] = P[:, [0, 1, 2], [0, 1, 2]] @ C
        for i, j, m in ((0, 1, mat["G12"]), (0, 2, mat["G13"]), (1, 2, mat["G23"])):
            S[:, i, j] = S[:, j, i] = 2 * m * P[:, i, j]
        K = (eye + D) @ (R @ S @ R.transpose(1, 2))
        fe += torch.einsum("eij,eaj->eai", K, G) * torch.linalg.det(J)[:, None, None]
    f.index_add_(0, hexes.reshape(-1), fe.reshape(-1, 3))
    if mesh.n_coh:
        coh = torch.as_tensor(mesh.coh, dtype=torch.int64, device=dev)
        lo, hi = coh[:, :4], coh[:, 4:]
        w = 0.25 * (X[coh[:, 2], 0] - X[coh[:, 0], 0]) * (X[coh[:, 2], 1] - X[coh[:, 0], 1])
        ksh = mat["KI"] * (mat["GIc"] / mat["GIIc"]) * (mat["tauII"] / mat["tauI"]) ** 2
        tau = (U[hi] - U[lo]) * t([ksh, ksh, mat["KI"]]) * w[:, None, None]
        f.index_add_(0, hi.reshape(-1), tau.reshape(-1, 3))
        f.index_add_(0, lo.reshape(-1), -tau.reshape(-1, 3))
    return f.T.contiguous()


def exact(case, seed):
    k = case["kind"]
    if k not in ("force", "force_block") or case["nx"] * case["ny"] * case["plies"] > 600000:
        return None
    r = np.random.default_rng(seed)
    mesh = _mesh("damage" if k == "force" else "block", case["nx"], case["ny"], case["plies"], 1)
    d = _smooth_field(mesh, r)
    f = _elastic_force(mesh, pi.material_im7_like_config(t_ply=T_PLY, seed=int(seed)), d)
    return f.cpu().numpy() if k == "force" else f
