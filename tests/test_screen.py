"""The hex kernels' two screens for points that keep the initial history
(csrc/pdn_screen.h, compiled here for the host) against the oracle's law at a
point (Algorithm 4): whatever a screen clears leaves every threshold and the
plastic strains at their initial values, for strengths scaled anywhere within
the spread; and the second screen clears what is strained short of an onset,
which the first does not.  No tolerance: the oracle's history is compared with
the initial one exactly (the screens keep 0.1 % to spare)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
import pdn_inputs as pi

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "pdn_screen.h"
using namespace pdn;
static double kt(const pdn_material &m) {
  const double a = m.alpha0_deg * M_PI / 180.0;
  return std::cos(a) * (std::sin(a) + std::cos(a) / std::tan(2.0 * a));
}
extern "C" double bound(const pdn_material *m, const double (*C)[3], int dm, int pl) {
  return elastic_strain_bound(*m, *reinterpret_cast<const double (*)[3][3]>(C), kt(*m), dm, pl);
}
extern "C" int cleared(const pdn_material *m, const double (*C)[3], int dm, int pl, double c, double s, const float *a) {
  const OnsetScreen o = onset_screen(*m, *reinterpret_cast<const double (*)[3][3]>(C), kt(*m), dm, pl);
  return clear_of_onset(o, (float)c, (float)s, *reinterpret_cast<const float (*)[6]>(a));
}
extern "C" float upper(uint32_t hi) { return upper_float(hi); }
"""


@pytest.fixture(scope="module")
def scr(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("screen")
    (d / "s.cpp").write_text(SRC)
    so = str(d / "s.so")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2301_05552_gb300", "csrc"), str(d / "s.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    L.bound.restype = C.c_double
    L.upper.restype = C.c_float
    L.upper.argtypes = [C.c_uint32]
    L.cleared.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_int, C.c_double, C.c_double, C.c_void_p]
    return L


class Screen:
    def __init__(self, L, mat, dm=1, pl=1):
        self.L, self.m, self.dm, self.pl = L, oracle.material(mat), dm, pl
        self.C = np.ascontiguousarray(oracle.stiffness(mat)[:3, :3])

    def bound(self):
        return self.L.bound(C.byref(self.m), self.C.ctypes.data_as(C.c_void_p), self.dm, self.pl)

    def cleared(self, angle, a):
        a = np.ascontiguousarray(a, dtype=np.float32)
        t = np.radians(angle)
        return bool(self.L.cleared(C.addressof(self.m), self.C.ctypes.data, self.dm, self.pl, np.cos(t), np.sin(t),
                                   a.ctypes.data))


def _materials():
    r = np.random.default_rng(3)
    base = [pi.material_im7_like_config(t_ply=0.275), pi.material_as4_8552(t_ply=0.724)]
    out = []
    for k in range(18):
        m = dict(base[k % 2])
        for n in ("XT", "XC", "YT", "YC", "SL", "Sp"):
            m[n] *= np.exp(r.uniform(-1.0, 1.0))
        for n in ("G12", "G13", "G23", "E1"):
            m[n] *= r.uniform(0.7, 1.4)
        m["spread"] = (0.0, 0.05, 0.3)[k % 3]
        m["GYT"] = m["GSL"] * (0.3, 1.0, 2.5)[(k // 3) % 3]
        m["alpha0_deg"] = (53.0, 46.0, 60.0)[(k // 2) % 3]
        out.append((m, (1, 1, 1, 0)[k % 4], (1, 1, 0, 1)[k % 4]))
    return [(base[0], 1, 1), (base[1], 1, 1)] + out


def _ply_strain(angle, e):
    """Ply-axis engineering strain (11 22 33 12 13 23) of a global one (xx yy zz
    xy xz yz)."""
    c, s = np.cos(np.radians(angle)), np.sin(np.radians(angle))
    return np.array([c * c * e[0] + c * s * e[3] + s * s * e[1], s * s * e[0] - c * s * e[3] + c * c * e[1], e[2],
                     2 * c * s * (e[1] - e[0]) + (c * c - s * s) * e[3], c * e[4] + s * e[5], c * e[5] - s * e[4]])


INITIAL = np.array([1.0, 1.0, 1.0, 1.0, 0.0, 0.0, 0.0])


def _keeps(mat, dm, pl, angle, e, factors):
    ep = _ply_strain(angle, e)
    return all(np.array_equal(oracle.cdm_point(mat, 0.5, ep, sf=f, damage_on=dm, plasticity_on=pl)[1], INITIAL)
               for f in factors)


def _factors(mat):
    lo, hi = 1.0 - mat["spread"], 1.0 + mat["spread"]
    return [(lo, lo, lo), (hi, hi, hi), (lo, hi, lo), (hi, lo, hi)]


@pytest.mark.parametrize("k", range(20))
def test_bound_keeps_the_initial_history(scr, k):
    mat, dm, pl = _materials()[k]
    t = 0.99 * Screen(scr, mat, dm, pl).bound()
    assert 0.0 < t < 0.1
    signs = np.array([[1.0 if (n >> b) & 1 else -1.0 for b in range(6)] for n in range(64)])
    for angle in (0.0, 17.0, 45.0, 90.0, -45.0):
        for e in signs:
            assert _keeps(mat, dm, pl, angle, t * e, _factors(mat))


@pytest.mark.parametrize("k", range(20))
def test_cleared_keeps_the_initial_history(scr, k):
    """Magnitudes at the edge of what the screen clears, in every sign."""
    mat, dm, pl = _materials()[k]
    S, r = Screen(scr, mat, dm, pl), np.random.default_rng(100 + k)
    t = S.bound()
    for angle in (0.0, 17.0, 45.0, 90.0, -60.0):
        for n in range(14):
            a = np.abs(r.normal(size=6)) if n % 2 else np.eye(6)[n // 2 % 6] + 0.02
            lo, hi = 0.0, 10.0
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                lo, hi = (mid, hi) if S.cleared(angle, mid * a) else (lo, mid)
            assert lo * a.max() >= t  # clears no less than the bound does
            for _ in range(8):
                sgn = np.where(r.random(6) < 0.5, -1.0, 1.0)
                assert _keeps(mat, dm, pl, angle, lo * a * sgn, _factors(mat))


@pytest.mark.parametrize("mat", [pi.material_im7_like_config(t_ply=0.275), pi.material_as4_8552(t_ply=0.724)],
                         ids=["im7_like", "as4_8552"])
def test_strained_short_of_onset_is_cleared(scr, mat):
    """One component in ply axes at 0.98 of its onset (the smaller of the two
    signs, which the screen does not know) with the smallest strengths: past the
    bound, and cleared; at 1.02 the law changes and it is not.  A plate strained
    so is the state an impact leaves much of it in."""
    S, lo = Screen(scr, mat), 1.0 - mat["spread"]
    past = 0
    for comp in (0, 1, 3, 5):
        e = np.eye(6)[comp]
        a, b = 0.0, 0.2
        for _ in range(80):
            mid = 0.5 * (a + b)
            keeps = all(_keeps(mat, 1, 1, 0.0, x * e, [(lo, lo, lo)]) for x in (mid, -mid))
            a, b = (mid, b) if keeps else (a, mid)
        past += 0.98 * a > S.bound()
        assert S.cleared(0.0, 0.98 * a * e)
        assert not S.cleared(0.0, 1.02 * a * e)
    assert past == 4
    # biaxial, as under bending: past the bound by a third, in every ply
    for angle in (0.0, 45.0, -45.0, 90.0):
        assert S.cleared(angle, S.bound() * np.array([1.3, 1.3, 0.3, 0.3, 0.1, 0.1]))


def test_degenerate_materials_clear_nothing(scr):
    base = pi.material_im7_like_config(t_ply=0.275)
    for change in (dict(spread=1.0), dict(spread=1.5), dict(YT=-60.0), dict(XT=0.0), dict(SL=float("nan")), dict(YC=0.0),
                   dict(GSL=0.0), dict(Sp=0.0), dict(Sp=-1.0)):
        S = Screen(scr, dict(base, **change))
        for a in (np.zeros(6), np.full(6, 1e-6), np.full(6, 1e-3)):
            assert not S.cleared(30.0, a)
    S = Screen(scr, base)
    assert S.cleared(30.0, np.zeros(6)) and S.cleared(30.0, np.full(6, 1e-5))
    for bad in (np.nan, np.inf):
        for k in range(6):
            assert not S.cleared(30.0, np.where(np.arange(6) == k, bad, 1e-5))
    off = Screen(scr, base, 0, 0)
    assert off.bound() > 1e20 and off.cleared(30.0, np.full(6, 0.5))


def test_upper_float_is_no_smaller(scr):
    r = np.random.default_rng(1)
    x = np.concatenate([np.exp(r.uniform(-750.0, 700.0, 4000)), np.exp(r.uniform(-80.0, 80.0, 4000)),
                        [0.0, 5e-324, 2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -53), np.finfo(np.float32).max, 1e308,
                         2.0 ** 128, 1.0, 1.0 - 2.0 ** -53]])
    hi = (x.view(np.uint64) >> 32).astype(np.uint32)
    up = np.array([scr.upper(int(h)) for h in hi])
    assert (up >= x).all()
    mid = (x > 2.0 ** -125) & (x < 2.0 ** 127)
    assert (up[mid] <= x[mid] * (1 + 2.0 ** -19)).all()
    assert np.isinf(scr.upper(0x7ff80000)) and np.isinf(scr.upper(0x7fffffff)) and np.isinf(scr.upper(0x7ff00000))
