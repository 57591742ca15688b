// Screens of the hex kernels for points that keep the initial history: from
// bounds on the magnitudes of the strain components alone, no yield and no
// damage onset (Algorithm 4), whatever the seeded strengths.  Plain C++, so the
// tests compile it for the host and hold it against the oracle's law.
//
// Two screens, because the first has to cost one comparison and the second has
// to clear what an impact strains without damaging:
//  * elastic_strain_bound: one bound for all components, in any axes about z.
//    A chain of worst cases (all components at the bound, every criterion by its
//    norm), about a quarter of the transverse onset strain.
//  * clear_of_onset: the criteria themselves on the magnitudes rotated to the
//    ply's axes.  On the AS4/8552 coupon at 72,000 steps the first leaves 15.7 %
//    of the hexes to the point-by-point law (1.42 rounds of four per warp), the
//    second 2.2 % (0.20), and 1.5 % have a history; on a plate of 10,800 hexes
//    late in its impact 40 % against 1.3 %.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "pdn.h"

#if defined(__CUDACC__)
#define PDN_HD __host__ __device__ __forceinline__
#else
#define PDN_HD inline
#endif

namespace pdn {

// Constants of clear_of_onset, FP32 for both element precisions (an FP64
// operation holds its scheduler 64 cycles, and the screen has 0.1 % to spare).
// A law that is off has zeros; a criterion that is not a finite number has
// infinities, which clear nothing.
struct OnsetScreen {
  float ft;                 // E1 / XT: fibre tension per e11
  float fc1, fc2, fc3;      // |C11|, |C12|, |C13| / XC: fibre compression
  float y1, y2, y3;         // |C12|, |C22|, |C23| / YT: a = s22 / YT
  float g1, g;              // matrix tension: g1 a + g a^2 + shear
  float mc2;                // matrix compression: mc2 a^2 + shear
  float h12, h13, h23;      // shear: h12 g12^2 + h13 g13^2 + h23 g23^2
  float pl;                 // yield: pl (g12^2 + g13^2)
};

namespace screen {
struct Limits {  // smallest seeded strengths; kT = ca (sa - etaT ca) of Algorithm 4
  double XT, YT, SL, ST, kT, g;
};
inline Limits limits(const pdn_material &m, double kT) {
  const double lo = 1.0 - std::fabs(m.spread);
  return {m.XT * lo, m.YT * lo, m.SL * lo, m.YC * kT, kT, m.GYT / m.GSL};
}
}  // namespace screen

// Bound on the strain components below which no point with the initial
// history yields or reaches a damage onset (Mat::e_tol).  With every normal
// component and engineering shear at most t, the tensor's Frobenius norm n is
// at most sqrt(4.5) t, the same in ply axes, and each criterion of Algorithm 4
// is bounded by a function of n: |e_ii| <= n; the 12, 13 shears together at
// most sqrt(2) n; |sigma_ii| at most the norm of the stiffness row times n.
// With the smallest seeded strengths and 0.1 % to spare for the rounding of
// the criteria; unbounded when both laws are off, 0 where a limit is no number.
inline double elastic_strain_bound(const pdn_material &m, const double (&C)[3][3], double kT, int damage_on,
                                   int plasticity_on) {
  double n = 1e30;
  auto cap = [&](double x) { n = x < n ? x : (x >= n ? n : 0.0); };
  if (plasticity_on) cap(m.Sp / (m.G12 * std::sqrt(2.0)));
  if (damage_on) {
    const screen::Limits l = screen::limits(m, kT);
    const double r1 = std::sqrt(C[0][0] * C[0][0] + C[0][1] * C[0][1] + C[0][2] * C[0][2]);
    const double r2 = std::sqrt(C[0][1] * C[0][1] + C[1][1] * C[1][1] + C[1][2] * C[1][2]);
    cap(l.XT / m.E1);
    cap(m.XC / r1);
    const double sl = std::sqrt(2.0) * std::max(m.G12, m.G13) / l.SL;
    const double sq = std::sqrt(2.0) * m.G23 / l.ST, st = r2 * l.kT / l.ST, yt = r2 / std::fabs(l.YT);
    // the matrix criteria at norm x: |1 - g| yt x + (|g| yt^2 + sh) x^2 <= 1 and (st^2 + sh) x^2 <= 1
    const double sh = sl * sl + sq * sq, q = std::fabs(l.g) * yt * yt + sh, p = std::fabs(1.0 - l.g) * yt;
    cap(2.0 / (p + std::sqrt(p * p + 4.0 * q)));
    cap(1.0 / std::sqrt(st * st + sh));
  }
  const double t = 0.999 * n / std::sqrt(4.5);
  return t > 0.0 && std::isfinite(t) ? t : 0.0;
}

inline OnsetScreen onset_screen(const pdn_material &m, const double (&C)[3][3], double kT, int damage_on,
                                int plasticity_on) {
  OnsetScreen o{};
  // an upper bound in FP32; what is negative or no number clears nothing
  auto up = [](double v) { return v >= 0.0 && v < 1e30 ? (float)(v * (1.0 + 1e-6)) : INFINITY; };
  auto pos = [](double v) { return v > 0.0 ? v : NAN; };  // a strength that is none clears nothing
  if (damage_on) {
    const screen::Limits l = screen::limits(m, kT);
    const double iXC = 1.0 / pos(m.XC), iYT = 1.0 / pos(l.YT), iSL = 1.0 / pos(l.SL), iST = 1.0 / l.ST;
    o.ft = up(m.E1 / pos(l.XT));
    o.fc1 = up(std::fabs(C[0][0]) * iXC);
    o.fc2 = up(std::fabs(C[0][1]) * iXC);
    o.fc3 = up(std::fabs(C[0][2]) * iXC);
    o.y1 = up(std::fabs(C[0][1]) * iYT);
    o.y2 = up(std::fabs(C[1][1]) * iYT);
    o.y3 = up(std::fabs(C[1][2]) * iYT);
    o.g1 = up(std::max(1.0 - l.g, 0.0));  // a negative term is left out
    o.g = up(l.g);
    const double t = l.YT * std::max(l.kT, 0.0) * iST, s = m.G23 * iST, s12 = m.G12 * iSL, s13 = m.G13 * iSL;
    o.mc2 = up(t * t);
    o.h12 = up(s12 * s12);
    o.h13 = up(s13 * s13);
    o.h23 = up(s * s);
  }
  if (plasticity_on) {
    const double s = m.G12 / pos(m.Sp);
    o.pl = up(s * s);
  }
  return o;
}

// A float no smaller than any double of magnitude whose upper word is hi
// (infinity beyond FP32 and for what is no number), without FP64 work.
PDN_HD float upper_float(uint32_t hi) {
  uint32_t b = 0x00800000u;                                             // below the normal floats
  if (hi >= (1151u << 20)) b = 0x7f800000u;                             // beyond them
  else if (hi >= (897u << 20)) b = (hi + 1u - (896u << 20)) << 3;       // the next of 20 bits
  float f;
  memcpy(&f, &b, sizeof f);
  return f;
}

// Whether points whose strain components have magnitudes of at most a (xx yy
// zz | xy xz yz, engineering shears, global axes) stay clear of yield and every
// onset in a ply at cos c, sin s: false where a bound is no number.
PDN_HD bool clear_of_onset(const OnsetScreen &o, float c, float s, const float (&a)[6]) {
  c = fabsf(c);
  s = fabsf(s);
  const float c2 = c * c, s2 = s * s, cs = c * s;
  const float e1 = c2 * a[0] + s2 * a[1] + cs * a[3], e2 = s2 * a[0] + c2 * a[1] + cs * a[3];
  const float g12 = 2.0f * cs * (a[0] + a[1]) + fabsf(c2 - s2) * a[3];
  const float g13 = c * a[4] + s * a[5], g23 = c * a[5] + s * a[4];
  const float q = o.y1 * e1 + o.y2 * e2 + o.y3 * a[2], q2 = q * q;
  const float sh = o.h12 * (g12 * g12) + o.h13 * (g13 * g13) + o.h23 * (g23 * g23);
  const float lim = 0.998f;
  return o.ft * e1 <= 0.999f && o.fc1 * e1 + o.fc2 * e2 + o.fc3 * a[2] <= 0.999f && o.g1 * q + o.g * q2 + sh <= lim &&
         o.mc2 * q2 + sh <= lim && o.pl * (g12 * g12 + g13 * g13) <= lim;
}

}  // namespace pdn
