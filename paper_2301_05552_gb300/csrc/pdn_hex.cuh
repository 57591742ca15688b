// Hex8 internal forces (Sec. 2, Eq. fcont; total Lagrangian, 2x2x2 Gauss) in
// three forms that share one formulation:
//
//  * eight lanes per element (hex_lanes8): lane = one node and the Gauss point
//    next to it.  Gradients and nodal sums go through warp shuffles, every
//    point takes the intralaminar law (Algorithm 4) by itself.
//  * one thread per element (hex_box_elastic): axis-aligned boxes whose points
//    all hold the initial history and whose strains cannot reach yield or any
//    damage onset.
//  * one thread per element, point by point (hex_points): general FP32 hexes of
//    launches that fill the GPU so.
//
// Why the second form costs less than half of a point-by-point evaluation.
// Over the 2x2x2 points of a box, du/dX_0 depends on (eta, zeta) only, and
// likewise for the other two directions: 36 distinct gradient values instead
// of 72, four distinct values of each normal strain instead of eight.  The
// stress of an undamaged point is one product with the ply's stiffness in
// global axes (Dev::ply_q, 13 constants) without rotations.  The forces of
// direction k need only sums of P_k over the pairs of points along k (four
// values per component), in which du/dX_k is a common factor.  The test for
// "cannot yield or damage" has two stages (pdn_screen.h): one bound on all
// strain components (Mat::e_tol), then the criteria on the largest magnitude of
// each component over the element's points.  Elements neither clears, or with
// history, are evaluated by hex_lanes8, four at a time by the whole warp, which
// costs about as much as the elastic form for all 32.  GB300, the point-by-point
// kernel's time, the first stage alone, both: 24 plates in a batch late in their
// impacts (up to 40 % of a plate's hexes past the first stage, 1 % damaged) 236,
// 250, 166 us per step; the AS4/8552 coupon at 60,000 to 82,000 steps 87.1, 87.5,
// 78.3 us, at its start, where the first stage clears all, 56.9, 41.2, 40.8 us.
//
// Every operation of the first two forms but the law's is rounded explicitly
// (rmul, radd, rfma), so the kernels that inline them give the same bits.
#pragma once

#include <cstdint>

#include "pdn_device.cuh"
#include "pdn_internal.h"

namespace pdn {
namespace detail {

__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// Magnitude as integer bits (the upper word of a double): compares as |x|
// does, and a NaN compares above every finite bound.  Costs no FP64 work.
// (max_mag below, of floats, drops a NaN: an element with a NaN strain may pass
// as elastic; its forces are NaN either way, and the law would leave its history.)
__device__ __forceinline__ uint32_t mag_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t mag_bits(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

template <typename T>
__device__ __forceinline__ T gauss_pt() {
  return T(0.57735026918962576451);
}

// The force slot of corner a (node nd) of element e.
template <typename T>
__device__ __forceinline__ int64_t corner_slot(const Dev<T> &D, int64_t e, int a, int nd) {
  if (D.rank == nullptr) return (int64_t)__ldg(D.pos + 8 * e + a);
  const int r = (int)((__ldg(D.rank + e) >> (3 * a)) & 7u);
  if (!D.slot_compact) return 8 * (int64_t)nd + r;
  const uint32_t lay = node_layer(D, nd);
  return compact_slot_base(D, lay, nd) + r;
}

// ---------------------------------------------------------------------------
// Eight lanes per element.  All 32 lanes of the warp call together: lane l
// belongs to element e of its group of eight (valid = false: the group does
// nothing but take part in the shuffles).  Returns the nodal force of the
// lane's node (corner a, node nd).
template <typename T>
struct LaneForce {
  T f[3];
  int nd, a;
};

template <typename T, bool BOX>
__device__ __forceinline__ LaneForce<T> hex_lanes8(const Dev<T> &D, const Mat<T> &M, int64_t e, bool &valid,
                                                   int mode) {
  using V4 = typename Vec4T<T>::type;
  constexpr uint32_t kAll = 0xffffffffu;
  const Ctl *ctl = D.ctl;
  const int lane = (int)(threadIdx.x & 31), sub = lane & 7;
  const int bit[3] = {sub & 1, (sub >> 1) & 1, sub >> 2};
  const int a = bit[2] * 4 + (bit[1] ? 3 - bit[0] : bit[0]);
  const int64_t nh = D.nh;
  const int ub = (mode == MODE_FORCES) ? (ctl->dpar ^ 1) : ctl->dpar;
  const int hb = ctl->hpar;
  const int64_t ee = valid ? e : 0;
  int nd = __ldg(D.hex + 8 * ee + a);
#ifdef PDN_CHECK
  {
    const bool in = nd >= 0 && (int64_t)nd < D.nn;
    const uint32_t bad = __ballot_sync(kAll, !in) >> (lane & 24) & 0xffu;
    if (bad != 0u) {
      if (valid && sub == 0) atomicCAS(&D.ctl->check, 0, (int32_t)CHECK_ELEMENT_NODE);
      valid = false;
      nd = 0;
    }
  }
#endif
  const V4 u = D.u4[ub][nd];
  T un[3] = {u.x, u.y, u.z};
  if constexpr (sizeof(T) == 4) {
    // from the element's first node (as raw_modes does)
#pragma unroll
    for (int i = 0; i < 3; ++i) un[i] = rsub(un[i], __shfl_sync(kAll, un[i], lane & 24));
  }
  const bool pristine = D.pflag[0] != nullptr && D.pflag[hb][ee] != 0;
  const T gp = gauss_pt<T>();
  const T al = T(0.5) + T(0.5) * gp, be = T(0.5) - T(0.5) * gp;
  // value at the lane's own Gauss coordinate along direction m of a field
  // given at the corners (and its transpose, the same formula)
  auto interp = [&](T v, int m) { return rfma(al, v, rmul(be, __shfl_xor_sync(kAll, v, 1 << m))); };
  auto diff = [&](T v, int k) {
    const T o = __shfl_xor_sync(kAll, v, 1 << k);
    return bit[k] ? rsub(v, o) : rsub(o, v);
  };
  // differences of the lane's field along the three directions, at its point
  auto grad = [&](T v, T (&g)[3]) {
    const T vz = interp(v, 2);
    g[0] = interp(diff(vz, 0), 1);
    g[1] = interp(diff(vz, 1), 0);
    g[2] = interp(interp(diff(v, 2), 0), 1);
  };
  T H[3][3], Ji[3][3], det = T(0), wk[3], vol;
  // FP64 boxes take the box record's reciprocals and volume, with the scale of
  // direction k in its last interpolation: 170 FP64 operations instead of the
  // 193 with differences and a reciprocal of the coordinates (8,192 hexes on
  // GB300: 48.6 to 45.3 us per step).  In FP32 the operations are not what
  // bounds the element, and the coordinates' differences round once less.
  constexpr bool REC = BOX && sizeof(T) == 8;
  auto scaled = [&](T v, int m, T s) {
    return rfma(rmul(al, s), v, rmul(rmul(be, s), __shfl_xor_sync(kAll, v, 1 << m)));
  };
  if constexpr (REC) {
    const V4 box = D.box[ee];
    const T jd[3] = {box.x, box.y, box.z};
    vol = rmul(T(8), box.w);
#pragma unroll
    for (int k = 0; k < 3; ++k) wk[k] = rmul(box.w, jd[k]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const T vz = interp(un[i], 2);
      H[i][0] = scaled(diff(vz, 0), 1, jd[0]);
      H[i][1] = scaled(diff(vz, 1), 0, jd[1]);
      H[i][2] = scaled(interp(diff(un[i], 2), 0), 1, jd[2]);
    }
  } else if constexpr (BOX) {
    const V4 x = D.X4[nd];
    const T xn[3] = {x.x, x.y, x.z};
    T hx[3], jd[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) hx[k] = diff(xn[k], k);
    // one reciprocal per lane, shared by the group
    const int k3 = sub % 3;
    const T r = xrcp(k3 == 0 ? hx[0] : k3 == 1 ? hx[1] : hx[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) jd[k] = __shfl_sync(kAll, r, (lane & 24) + k);
    vol = rmul(hx[0], rmul(hx[1], hx[2]));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T g[3];
      grad(un[i], g);
#pragma unroll
      for (int k = 0; k < 3; ++k) H[i][k] = rmul(g[k], jd[k]);
    }
    wk[0] = rmul(T(0.125), rmul(hx[1], hx[2]));
    wk[1] = rmul(T(0.125), rmul(hx[0], hx[2]));
    wk[2] = rmul(T(0.125), rmul(hx[0], hx[1]));
  } else {
    const V4 x = D.X4[nd];
    const T xn[3] = {x.x, x.y, x.z};
    T J[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) grad(xn[i], J[i]);  // twice the Jacobian: the differences
    // cofactors of the difference matrix; det J = det(differences) / 8
    Ji[0][0] = rfma(J[1][1], J[2][2], -rmul(J[1][2], J[2][1]));
    Ji[0][1] = rfma(J[0][2], J[2][1], -rmul(J[0][1], J[2][2]));
    Ji[0][2] = rfma(J[0][1], J[1][2], -rmul(J[0][2], J[1][1]));
    Ji[1][0] = rfma(J[1][2], J[2][0], -rmul(J[1][0], J[2][2]));
    Ji[1][1] = rfma(J[0][0], J[2][2], -rmul(J[0][2], J[2][0]));
    Ji[1][2] = rfma(J[0][2], J[1][0], -rmul(J[0][0], J[1][2]));
    Ji[2][0] = rfma(J[1][0], J[2][1], -rmul(J[1][1], J[2][0]));
    Ji[2][1] = rfma(J[0][1], J[2][0], -rmul(J[0][0], J[2][1]));
    Ji[2][2] = rfma(J[0][0], J[1][1], -rmul(J[0][1], J[1][0]));
    det = rfma(J[0][0], Ji[0][0], rfma(J[0][1], Ji[1][0], rmul(J[0][2], Ji[2][0])));
    const T id = xrcp(det);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T g[3];
      grad(un[i], g);
#pragma unroll
      for (int k = 0; k < 3; ++k) g[k] = rmul(g[k], id);
#pragma unroll
      for (int k = 0; k < 3; ++k) H[i][k] = rfma(g[0], Ji[0][k], rfma(g[1], Ji[1][k], rmul(g[2], Ji[2][k])));
    }
    // element volume: the sum of det J over the points
    T v8 = rmul(T(0.125), det);
#pragma unroll
    for (int k = 0; k < 3; ++k) v8 = radd(v8, __shfl_xor_sync(kAll, v8, 1 << k));
    vol = v8;
  }
  // Green strain: normal components and engineering shears
  T En[3], Gs[3];  // xx yy zz; xy xz yz
#pragma unroll
  for (int k = 0; k < 3; ++k)
    En[k] = rfma(T(0.5), rfma(H[0][k], H[0][k], rfma(H[1][k], H[1][k], rmul(H[2][k], H[2][k]))), H[k][k]);
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int p = s == 2 ? 1 : 0, q = s == 0 ? 1 : 2;
    Gs[s] = rfma(H[0][p], H[0][q], rfma(H[1][p], H[1][q], rfma(H[2][p], H[2][q], radd(H[p][q], H[q][p]))));
  }
  uint32_t big = mag_bits(En[0]);
  big = max(big, max(mag_bits(En[1]), mag_bits(En[2])));
  big = max(max(big, mag_bits(Gs[0])), max(mag_bits(Gs[1]), mag_bits(Gs[2])));
  T S[3][3];
  bool changed = false;
  T h[7];
#pragma unroll
  for (int f = 0; f < 7; ++f) h[f] = f < 4 ? T(1) : T(0);
  const int ply = D.ply[ee];
  if (pristine && big < mag_bits(M.e_tol)) {
    const T *qp = D.ply_q + (int64_t)kPlyStride<T> * ply;
    T q[13];
#pragma unroll
    for (int k = 0; k < 13; ++k) q[k] = __ldg(qp + kPlyRep<T> * k);
    S[0][0] = rfma(q[0], En[0], rfma(q[1], En[1], rfma(q[2], En[2], rmul(q[3], Gs[0]))));
    S[1][1] = rfma(q[1], En[0], rfma(q[4], En[1], rfma(q[5], En[2], rmul(q[6], Gs[0]))));
    S[2][2] = rfma(q[2], En[0], rfma(q[5], En[1], rfma(q[7], En[2], rmul(q[8], Gs[0]))));
    S[0][1] = rfma(q[3], En[0], rfma(q[6], En[1], rfma(q[8], En[2], rmul(q[9], Gs[0]))));
    S[1][2] = rfma(q[10], Gs[2], rmul(q[11], Gs[1]));
    S[0][2] = rfma(q[11], Gs[2], rmul(q[12], Gs[1]));
  } else {
    if (!pristine) {
      const T *hin = D.hist[hb] + ee;
#pragma unroll
      for (int f = 0; f < 7; ++f) h[f] = hin[(int64_t)(f * 8 + a) * nh];
    }
    // to ply axes (rotation about z), the law, and back
    const T cs = M.ply_c[ply], sn = M.ply_s[ply];
    const T c2 = rmul(cs, cs), s2 = rmul(sn, sn), csn = rmul(cs, sn), cd = rsub(c2, s2);
    T ep[6], sm[6];
    ep[0] = rfma(c2, En[0], rfma(csn, Gs[0], rmul(s2, En[1])));
    ep[1] = rfma(s2, En[0], rfma(-csn, Gs[0], rmul(c2, En[1])));
    ep[2] = En[2];
    ep[3] = rfma(rmul(T(2), csn), rsub(En[1], En[0]), rmul(cd, Gs[0]));
    ep[4] = rfma(cs, Gs[1], rmul(sn, Gs[2]));
    ep[5] = rfma(cs, Gs[2], rmul(-sn, Gs[1]));
    const ElemLaw<T> L = elem_law(M, ee);
    T lc = T(-1);
    cdm(M, L, (const T(*)[3]) nullptr, vol, lc, ep, h, sm);
    changed = h[0] > T(1) || h[1] > T(1) || h[2] > T(1) || h[3] > T(1) || h[4] != T(0) || h[5] != T(0) ||
              h[6] != T(0);
    const T t3 = rmul(rmul(T(2), csn), sm[3]);
    S[0][0] = rfma(c2, sm[0], rsub(rmul(s2, sm[1]), t3));
    S[1][1] = rfma(s2, sm[0], rfma(c2, sm[1], t3));
    S[2][2] = sm[2];
    S[0][1] = rfma(csn, rsub(sm[0], sm[1]), rmul(cd, sm[3]));
    S[0][2] = rfma(cs, sm[4], rmul(-sn, sm[5]));
    S[1][2] = rfma(sn, sm[4], rmul(cs, sm[5]));
  }
  S[1][0] = S[0][1];
  S[2][0] = S[0][2];
  S[2][1] = S[1][2];
  // history of the trial state: an element whose points all keep the initial
  // history writes none
  const bool dirty = ((__ballot_sync(kAll, changed) >> (lane & 24)) & 0xffu) != 0u;
  if (valid && (!pristine || dirty)) {
    T *hout = D.hist[hb ^ 1] + ee;
#pragma unroll
    for (int f = 0; f < 7; ++f) hout[(int64_t)(f * 8 + a) * nh] = h[f];
  }
  if (valid && sub == 0 && D.pflag[0] != nullptr) D.pflag[hb ^ 1][ee] = (pristine && !dirty) ? 1 : 0;
  // P = S F^T with F = I + H, weighted towards direction k, and the nodal
  // sums: along k both points of a pair, across it the transposed
  // interpolation, with the sign of the node along k
  T Q[3][3];  // [k][i]
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
      Q[k][i] = rfma(S[k][2], H[i][2], rfma(S[k][1], H[i][1], rfma(S[k][0], H[i][0], S[k][i])));
  if constexpr (BOX && !REC) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i) Q[k][i] = rmul(wk[k], Q[k][i]);
  } else if constexpr (!BOX) {
    // det J J^-1 P / 2 = cofactors P / 8
    T R[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i)
        R[k][i] = rmul(T(0.125), rfma(Ji[k][0], Q[0][i], rfma(Ji[k][1], Q[1][i], rmul(Ji[k][2], Q[2][i]))));
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i) Q[k][i] = R[k][i];
  }
  LaneForce<T> out;
  out.nd = nd;
  out.a = a;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    auto pair = [&](T v, int k) {
      const T s = radd(v, __shfl_xor_sync(kAll, v, 1 << k));
      return bit[k] ? s : -s;
    };
    T t0, t1, t2;
    if constexpr (REC) {
      t0 = scaled(pair(Q[0][i], 0), 1, wk[0]);
      t1 = scaled(pair(Q[1][i], 1), 0, wk[1]);
      t2 = scaled(interp(pair(Q[2][i], 2), 0), 1, wk[2]);
    } else {
      t0 = interp(pair(Q[0][i], 0), 1);
      t1 = interp(pair(Q[1][i], 1), 0);
      t2 = interp(interp(pair(Q[2][i], 2), 0), 1);
    }
    out.f[i] = radd(interp(radd(t0, t1), 2), t2);
  }
  return out;
}

// One item with eight lanes per element: element e = slot / 8 of the elements
// below end; the warp calls together.
template <typename T, bool BOX>
__device__ __forceinline__ void hex_lanes8_item(const Dev<T> &D, const Mat<T> &M, int64_t slot, int64_t end,
                                                int mode) {
  using V4 = typename Vec4T<T>::type;
  const int64_t e = slot >> 3;
  const int lane = (int)(threadIdx.x & 31);
  bool valid = e < end;
  if (mode == MODE_REPEAT && D.rmark_e != nullptr) {
    valid = valid && D.rmark_e[e] != 0;
    if (!__any_sync(0xffffffffu, valid)) return;
    if (valid && (lane & 7) == 0) D.rmark_e[e] = 0;
  }
  const LaneForce<T> r = hex_lanes8<T, BOX>(D, M, e, valid, mode);
  if (!valid) return;
  if (mode == MODE_REPEAT && D.rmark_n != nullptr) D.rmark_n[r.nd] = 1;
  if constexpr (sizeof(T) == 4) {
    if (D.fplane != nullptr) {
      plane_store(D.fplane, (int)((__ldg(D.rank + e) >> (3 * r.a)) & 7u), r.nd, r.f[0], r.f[1], r.f[2]);
      return;
    }
  }
  V4 o;
  o.x = r.f[0];
  o.y = r.f[1];
  o.z = r.f[2];
  o.w = T(0);
  D.fe[corner_slot(D, e, r.a, r.nd)] = o;
}

// ---------------------------------------------------------------------------
// General FP32 hex by one thread, point by point: nodal forces f (by node) of
// hex e with the node ids nd, and its history.  Geometry and displacement enter
// through their trilinear modes, taken from the first node's values, so that
// J = [dx/dxi], du/dxi and the returned force are cheap mode sums:
// f_a = sum_g sum_k dN_a/dxi_k Q_g[k][:],  Q_g = det J_g  J_g^-1 P_g.
// The next Gauss point's history is loaded while the current one computes.
// Bound by its arithmetic at 16 warps per SM (128 registers): 0.627 ms for 3.84 M
// hexes against 0.771 ms by eight lanes, whose 78 shuffles per four elements take
// four issue slots each; forces as far from FP64 either way (2.4e-5 of their
// rms on a 393,216-hex plate).
__device__ __forceinline__ void hex_points(const Dev<float> &D, const Mat<float> &M, int64_t e, int mode,
                                           const int (&nd)[8], float (&f)[8][3]) {
  using T = float;
  const Ctl *ctl = D.ctl;
  const int64_t nh = D.nh;
  const int ub = (mode == MODE_FORCES) ? (ctl->dpar ^ 1) : ctl->dpar;
  const int hb = ctl->hpar;
  const float4 *PDN_STATE_RESTRICT U = D.u4[ub];
  const T *PDN_STATE_RESTRICT hin = D.hist[hb] + e;
  T *PDN_STATE_RESTRICT hout = D.hist[hb ^ 1] + e;
  const bool pristine = D.pflag[0] != nullptr && D.pflag[hb][e] != 0;
  bool dirty = false;
  T hn[7];  // history of Gauss point 0 in flight first
#pragma unroll
  for (int k = 0; k < 7; ++k) hn[k] = pristine ? (k < 4 ? T(1) : T(0)) : hin[(int64_t)(k * 8) * nh];
  // modes of a nodal field, from its value at the first node
  auto modes = [&](const float4 *V, T (&c)[8][3]) {
    T v[8][3];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const float4 q = V[nd[a]];
      v[a][0] = q.x, v[a][1] = q.y, v[a][2] = q.z;
    }
#pragma unroll
    for (int a = 7; a >= 0; --a)
#pragma unroll
      for (int i = 0; i < 3; ++i) v[a][i] -= v[0][i];
    to_modes(v, c);
  };
  T am[8][3], bm[8][3];
  modes(U, bm);
  modes(D.X4, am);
  const int ply = D.ply[e];
  const T cs = M.ply_c[ply], sn = M.ply_s[ply];
  const T c2 = cs * cs, s2 = sn * sn, csn = cs * sn;
  const ElemLaw<T> L = elem_law(M, e);
  T lc = T(-1);
  T C[8][3];  // mode sums of the force
#pragma unroll
  for (int m = 0; m < 8; ++m) C[m][0] = C[m][1] = C[m][2] = T(0);
  const T gp = gauss_pt<T>();
#pragma unroll 1
  for (int g = 0; g < 8; ++g) {
    T h[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) h[k] = hn[k];
    if (g < 7 && !pristine) {
#pragma unroll
      for (int k = 0; k < 7; ++k) hn[k] = hin[(int64_t)(k * 8 + g + 1) * nh];
    }
    const T xi = T(sgn_x(g)) * gp, et = T(sgn_y(g)) * gp, ze = T(sgn_z(g)) * gp;
    T Du[3][3], H[3][3], Ji[3][3], J[3][3];
    jac_cols(bm, xi, et, ze, Du);
    jac_cols(am, xi, et, ze, J);
    const T det = det3(J);
    const T id = T(1) / det;
    Ji[0][0] = (J[1][1] * J[2][2] - J[1][2] * J[2][1]) * id;
    Ji[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) * id;
    Ji[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) * id;
    Ji[1][0] = (J[1][2] * J[2][0] - J[1][0] * J[2][2]) * id;
    Ji[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) * id;
    Ji[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) * id;
    Ji[2][0] = (J[1][0] * J[2][1] - J[1][1] * J[2][0]) * id;
    Ji[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) * id;
    Ji[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) * id;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) H[i][k] = Du[i][0] * Ji[0][k] + Du[i][1] * Ji[1][k] + Du[i][2] * Ji[2][k];
    // Green strain: normal components and engineering shears, to ply axes
    const T exx = H[0][0] + T(0.5) * (H[0][0] * H[0][0] + H[1][0] * H[1][0] + H[2][0] * H[2][0]);
    const T eyy = H[1][1] + T(0.5) * (H[0][1] * H[0][1] + H[1][1] * H[1][1] + H[2][1] * H[2][1]);
    const T ezz = H[2][2] + T(0.5) * (H[0][2] * H[0][2] + H[1][2] * H[1][2] + H[2][2] * H[2][2]);
    const T gxy = H[0][1] + H[1][0] + H[0][0] * H[0][1] + H[1][0] * H[1][1] + H[2][0] * H[2][1];
    const T gxz = H[0][2] + H[2][0] + H[0][0] * H[0][2] + H[1][0] * H[1][2] + H[2][0] * H[2][2];
    const T gyz = H[1][2] + H[2][1] + H[0][1] * H[0][2] + H[1][1] * H[1][2] + H[2][1] * H[2][2];
    const T ep[6] = {c2 * exx + csn * gxy + s2 * eyy,
                     s2 * exx - csn * gxy + c2 * eyy,
                     ezz,
                     T(2) * csn * (eyy - exx) + (c2 - s2) * gxy,
                     cs * gxz + sn * gyz,
                     cs * gyz - sn * gxz};
    T sm[6];
    cdm(M, L, (const T(*)[3])am, T(0), lc, ep, h, sm);
    if (!pristine) {
#pragma unroll
      for (int k = 0; k < 7; ++k) hout[(int64_t)(k * 8 + g) * nh] = h[k];
    } else {
      const bool changed = h[0] > T(1) || h[1] > T(1) || h[2] > T(1) || h[3] > T(1) || h[4] != T(0) || h[5] != T(0) ||
                           h[6] != T(0);
      if (changed && !dirty) {
        // first change in a pristine element: the earlier points keep the
        // initial history, which the output buffer does not hold yet
        for (int gg = 0; gg < g; ++gg)
#pragma unroll
          for (int k = 0; k < 7; ++k) hout[(int64_t)(k * 8 + gg) * nh] = k < 4 ? T(1) : T(0);
        dirty = true;
      }
      if (dirty) {
#pragma unroll
        for (int k = 0; k < 7; ++k) hout[(int64_t)(k * 8 + g) * nh] = h[k];
      }
    }
    // back to global axes, P = S F^T with F = I + H, Q = det J^-1 P
    T S[3][3];
    const T t3 = T(2) * csn * sm[3];
    S[0][0] = c2 * sm[0] + s2 * sm[1] - t3;
    S[1][1] = s2 * sm[0] + c2 * sm[1] + t3;
    S[2][2] = sm[2];
    S[0][1] = S[1][0] = csn * (sm[0] - sm[1]) + (c2 - s2) * sm[3];
    S[0][2] = S[2][0] = cs * sm[4] - sn * sm[5];
    S[1][2] = S[2][1] = sn * sm[4] + cs * sm[5];
    T P[3][3], Q[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) P[i][k] = S[i][k] + S[i][0] * H[k][0] + S[i][1] * H[k][1] + S[i][2] * H[k][2];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i)
        Q[k][i] = det * (Ji[k][0] * P[0][i] + Ji[k][1] * P[1][i] + Ji[k][2] * P[2][i]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      C[1][i] += Q[0][i];
      C[2][i] += Q[1][i];
      C[3][i] += Q[2][i];
      C[4][i] += et * Q[0][i] + xi * Q[1][i];
      C[5][i] += ze * Q[1][i] + et * Q[2][i];
      C[6][i] += ze * Q[0][i] + xi * Q[2][i];
      C[7][i] += et * ze * Q[0][i] + xi * ze * Q[1][i] + xi * et * Q[2][i];
    }
  }
  if (D.pflag[0] != nullptr) D.pflag[hb ^ 1][e] = (pristine && !dirty) ? 1 : 0;
  from_modes(C, f);
}

// ---------------------------------------------------------------------------
// One thread per element: boxes that stay elastic (see the head of the file).
// Largest magnitude of each strain component (xx yy zz | xy xz yz, engineering
// shears) over an element's points: FP32 values, or upper words of doubles.
template <typename T>
struct StrainMag;
template <>
struct StrainMag<float> {
  float m[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  __device__ __forceinline__ uint32_t largest() const {
    return mag_bits(fmaxf(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])), fmaxf(m[4], m[5])));
  }
  __device__ __forceinline__ float upper(int k) const { return m[k]; }
};
template <>
struct StrainMag<double> {
  uint32_t m[6] = {0u, 0u, 0u, 0u, 0u, 0u};
  __device__ __forceinline__ uint32_t largest() const { return max(max(max(m[0], m[1]), max(m[2], m[3])), max(m[4], m[5])); }
  __device__ __forceinline__ float upper(int k) const { return upper_float(m[k]); }
};

// Trilinear modes of the nodal displacements, unscaled (8 times the modes of
// to_modes), by bin: bit 0 xi, bit 1 eta, bit 2 zeta.  V: float, double or a
// packed pair of components.
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float b) { return __fmul2_rn(a, make_float2(b, b)); }

// FROM0: the values are taken from node 0's, which the modes used here do not
// depend on.  In FP32 the sums then round strains, not displacements: the
// differences of neighbouring nodes are exact, so what is left of the
// rounding of a large displacement is that of its FP32 mirror alone.
template <bool FROM0, typename V>
__device__ __forceinline__ void raw_modes(V (&r)[8]) {
  if constexpr (FROM0) {
#pragma unroll
    for (int k = 1; k < 8; ++k) r[k] = vsub(r[k], r[0]);
  }
#pragma unroll
  for (int b = 1; b < 8; b <<= 1)
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (!(k & b)) {
        const V lo = r[k], hi = r[k | b];
        if (FROM0 && b == 1 && k == 0) {
          r[0] = hi;
          continue;
        }
        if (!(b == 4 && k == 0)) r[k] = vadd(hi, lo);  // the mean is not used
        r[k | b] = vsub(hi, lo);
      }
}
// The transpose: nodal values by bin from mode sums by bin (no mean).
template <typename V>
__device__ __forceinline__ void raw_nodes(V (&r)[8]) {
#pragma unroll
  for (int b = 1; b < 8; b <<= 1)
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (!(k & b)) {
        const V c = r[k], x = r[k | b];
        if (b == 1 && k == 0) {
          r[0] = vsub(V{}, x);
        } else {
          r[k] = vsub(c, x);
          r[k | b] = vadd(c, x);
        }
      }
}

// The four values of direction K's gradient over the Gauss coordinates of
// the other two directions (A < B) from the modes: v[sA][sB].
template <int K, typename V, typename T>
__device__ __forceinline__ void column_values(const V (&r)[8], T q, T qg, T qgg, V (&p)[2], V (&s)[2]) {
  constexpr int A = K == 0 ? 1 : 0, B = K == 2 ? 1 : 2, b = 1 << K;
  const V v0 = vmul(r[b], q), va = vmul(r[b | (1 << A)], qg), vb = vmul(r[b | (1 << B)], qg), vab = vmul(r[7], qgg);
  p[0] = vsub(v0, va);
  p[1] = vadd(v0, va);
  s[0] = vsub(vb, vab);
  s[1] = vadd(vb, vab);
}

// The mode sums of direction K's four force values G[sA][sB], scaled and
// added to C by bin.
template <int K, bool FIRST, typename T>
__device__ __forceinline__ void column_sums(T g00, T g01, T g10, T g11, T t, T tg, T tgg, T (&C)[8]) {
  constexpr int A = K == 0 ? 1 : 0, B = K == 2 ? 1 : 2, b = 1 << K;
  const T a0 = radd(g00, g10), a1 = radd(g01, g11);  // over sA, at sB = 0, 1
  const T d0 = rsub(g10, g00), d1 = rsub(g11, g01);
  C[b] = rmul(t, radd(a0, a1));
  const T m = radd(d0, d1), n = rsub(a1, a0), mn = rsub(d1, d0);
  // bins shared with earlier directions: xi eta by 0, 1; xi zeta by 0, 2;
  // eta zeta by 1, 2; all three by 0, 1, 2
  C[b | (1 << A)] = (K == 0) ? rmul(tg, m) : rfma(tg, m, C[b | (1 << A)]);
  C[b | (1 << B)] = (K == 2 || false) ? rfma(tg, n, C[b | (1 << B)]) : rmul(tg, n);
  C[7] = FIRST ? rmul(tgg, mn) : rfma(tgg, mn, C[7]);
}

// FP64: nodal forces f (by node) of a box from its node displacements u (by
// node), the box record {1/hx, 1/hy, 1/hz, volume/8} and the ply's constants,
// and the largest magnitudes of the strain components.  About
// 900 FP64 operations, against about 2,500 point by point; on this part an
// FP64 operation holds a scheduler's pipe for 64 cycles, so they are the whole
// cost.
__device__ __forceinline__ void hex_box_elastic(const double (&u)[8][3], const double4_32a &box, const double *qp,
                                                double (&f)[8][3], StrainMag<double> &big) {
  const double gp = gauss_pt<double>();
  const double ih[3] = {box.x, box.y, box.z};
  double H0[3][2][2], H1[3][2][2], H2[3][2][2];  // [i][eta][zeta], [i][xi][zeta], [i][xi][eta]
  double q[3], qg[3], qgg[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q[k] = 0.25 * ih[k];
    qg[k] = rmul(q[k], gp);
    qgg[k] = rmul(qg[k], gp);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double r[8], p[2], s[2];
#pragma unroll
    for (int a = 0; a < 8; ++a) r[bin_of(a)] = u[a][i];
    raw_modes<false>(r);
    column_values<0>(r, q[0], qg[0], qgg[0], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) H0[i][m][0] = rsub(p[m], s[m]), H0[i][m][1] = radd(p[m], s[m]);
    column_values<1>(r, q[1], qg[1], qgg[1], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) H1[i][m][0] = rsub(p[m], s[m]), H1[i][m][1] = radd(p[m], s[m]);
    column_values<2>(r, q[2], qg[2], qgg[2], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) H2[i][m][0] = rsub(p[m], s[m]), H2[i][m][1] = radd(p[m], s[m]);
  }
  double c[13];
#pragma unroll
  for (int k = 0; k < 13; ++k) c[k] = __ldg(qp + k);
  auto normal = [](const double (&H)[3][2][2], int k, int m, int n) {
    return rfma(0.5, rfma(H[0][m][n], H[0][m][n], rfma(H[1][m][n], H[1][m][n], rmul(H[2][m][n], H[2][m][n]))),
                H[k][m][n]);
  };
  double E0[2][2], E1[2][2];
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      E0[m][n] = normal(H0, 0, m, n);
      E1[m][n] = normal(H1, 1, m, n);
      big.m[0] = max(big.m[0], mag_bits(E0[m][n]));
      big.m[1] = max(big.m[1], mag_bits(E1[m][n]));
    }
  double G0[3][2][2], G1[3][2][2], G2[3][2][2], T0[2][2], T1[2][2], T2[2][2];
#pragma unroll
  for (int iy = 0; iy < 2; ++iy)
#pragma unroll
    for (int ix = 0; ix < 2; ++ix) {
      const double e2 = normal(H2, 2, ix, iy);
      big.m[2] = max(big.m[2], mag_bits(e2));
#pragma unroll
      for (int iz = 0; iz < 2; ++iz) {
        const double a[3] = {H0[0][iy][iz], H0[1][iy][iz], H0[2][iy][iz]};
        const double b[3] = {H1[0][ix][iz], H1[1][ix][iz], H1[2][ix][iz]};
        const double d[3] = {H2[0][ix][iy], H2[1][ix][iy], H2[2][ix][iy]};
        const double g01 = rfma(a[0], b[0], rfma(a[1], b[1], rfma(a[2], b[2], radd(a[1], b[0]))));
        const double g02 = rfma(a[0], d[0], rfma(a[1], d[1], rfma(a[2], d[2], radd(a[2], d[0]))));
        const double g12 = rfma(b[0], d[0], rfma(b[1], d[1], rfma(b[2], d[2], radd(b[2], d[1]))));
        big.m[3] = max(big.m[3], mag_bits(g01));
        big.m[4] = max(big.m[4], mag_bits(g02));
        big.m[5] = max(big.m[5], mag_bits(g12));
        const double e0 = E0[iy][iz], e1 = E1[ix][iz];
        const double S00 = rfma(c[0], e0, rfma(c[1], e1, rfma(c[2], e2, rmul(c[3], g01))));
        const double S11 = rfma(c[1], e0, rfma(c[4], e1, rfma(c[5], e2, rmul(c[6], g01))));
        const double S22 = rfma(c[2], e0, rfma(c[5], e1, rfma(c[7], e2, rmul(c[8], g01))));
        const double S01 = rfma(c[3], e0, rfma(c[6], e1, rfma(c[8], e2, rmul(c[9], g01))));
        const double S12 = rfma(c[10], g12, rmul(c[11], g02));
        const double S02 = rfma(c[11], g12, rmul(c[12], g02));
        // P_k[i] = S_ki + sum_m S_km H_im; the term m = k is left to the end
        // (its gradient is the same along k)
        auto add = [&](double (&G)[3][2][2], double (&Tk)[2][2], int k, int m, int n, bool first, double Skk,
                       int k1, double S1, const double (&h1)[3], int k2, double S2, const double (&h2)[3]) {
          Tk[m][n] = first ? Skk : radd(Tk[m][n], Skk);
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const double base = i == k1 ? S1 : S2;
            double g;
            if (i == k)
              g = first ? rmul(S1, h1[i]) : rfma(S1, h1[i], G[i][m][n]);
            else
              g = rfma(S1, h1[i], first ? base : radd(G[i][m][n], base));
            G[i][m][n] = rfma(S2, h2[i], g);
          }
          (void)k2;
        };
        add(G0, T0, 0, iy, iz, ix == 0, S00, 1, S01, b, 2, S02, d);
        add(G1, T1, 1, ix, iz, iy == 0, S11, 0, S01, a, 2, S12, d);
        add(G2, T2, 2, ix, iy, iz == 0, S22, 0, S02, a, 1, S12, b);
      }
    }
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      G0[0][m][n] = radd(G0[0][m][n], T0[m][n]);
      G1[1][m][n] = radd(G1[1][m][n], T1[m][n]);
      G2[2][m][n] = radd(G2[2][m][n], T2[m][n]);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        G0[i][m][n] = rfma(H0[i][m][n], T0[m][n], G0[i][m][n]);
        G1[i][m][n] = rfma(H1[i][m][n], T1[m][n], G1[i][m][n]);
        G2[i][m][n] = rfma(H2[i][m][n], T2[m][n], G2[i][m][n]);
      }
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q[k] = rmul(q[k], box.w);
    qg[k] = rmul(qg[k], box.w);
    qgg[k] = rmul(qgg[k], box.w);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double C[8];
    column_sums<0, true>(G0[i][0][0], G0[i][0][1], G0[i][1][0], G0[i][1][1], q[0], qg[0], qgg[0], C);
    column_sums<1, false>(G1[i][0][0], G1[i][0][1], G1[i][1][0], G1[i][1][1], q[1], qg[1], qgg[1], C);
    column_sums<2, false>(G2[i][0][0], G2[i][0][1], G2[i][1][0], G2[i][1][1], q[2], qg[2], qgg[2], C);
    raw_nodes(C);
#pragma unroll
    for (int a = 0; a < 8; ++a) f[a][i] = C[bin_of(a)];
  }
}

// FP32, the same sums with the packed FP32 operations (two lanes per
// instruction, each rounded as the scalar operation): the lanes are the two
// zeta values of a point pair where fields depend on zeta, and the x and y
// components in the mode butterflies.  The packed form halves issue slots,
// not pipe time (measured: 17.7 T packed against 38.2 T scalar FMA/s), and
// issue is what limits the point-by-point form.
__device__ __forceinline__ float lane_sum(float2 v) { return __fadd_rn(v.x, v.y); }
__device__ __forceinline__ float max_mag(float m, float2 v) { return fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))); }

__device__ __forceinline__ void hex_box_elastic(const float (&u)[8][3], const float4 &box, const float *qp,
                                                float (&f)[8][3], StrainMag<float> &big) {
  const float gp = gauss_pt<float>();
  const float ih[3] = {box.x, box.y, box.z};
  float2 H0[3][2], H1[3][2];  // [i][eta], [i][xi]; lanes zeta
  float H2[3][2][2];          // [i][xi][eta]
  float q[3], qg[3], qgg[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q[k] = 0.25f * ih[k];
    qg[k] = rmul(q[k], gp);
    qgg[k] = rmul(qg[k], gp);
  }
  {
    float2 r[8], p[2], s[2];
#pragma unroll
    for (int a = 0; a < 8; ++a) r[bin_of(a)] = make_float2(u[a][0], u[a][1]);
    raw_modes<true>(r);
    column_values<0>(r, q[0], qg[0], qgg[0], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      H0[0][m] = make_float2(rsub(p[m].x, s[m].x), radd(p[m].x, s[m].x));
      H0[1][m] = make_float2(rsub(p[m].y, s[m].y), radd(p[m].y, s[m].y));
    }
    column_values<1>(r, q[1], qg[1], qgg[1], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      H1[0][m] = make_float2(rsub(p[m].x, s[m].x), radd(p[m].x, s[m].x));
      H1[1][m] = make_float2(rsub(p[m].y, s[m].y), radd(p[m].y, s[m].y));
    }
    column_values<2>(r, q[2], qg[2], qgg[2], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const float2 lo = vsub(p[m], s[m]), hi = vadd(p[m], s[m]);
      H2[0][m][0] = lo.x, H2[1][m][0] = lo.y, H2[0][m][1] = hi.x, H2[1][m][1] = hi.y;
    }
  }
  {
    float r[8], p[2], s[2];
#pragma unroll
    for (int a = 0; a < 8; ++a) r[bin_of(a)] = u[a][2];
    raw_modes<true>(r);
    column_values<0>(r, q[0], qg[0], qgg[0], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) H0[2][m] = make_float2(rsub(p[m], s[m]), radd(p[m], s[m]));
    column_values<1>(r, q[1], qg[1], qgg[1], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) H1[2][m] = make_float2(rsub(p[m], s[m]), radd(p[m], s[m]));
    column_values<2>(r, q[2], qg[2], qgg[2], p, s);
#pragma unroll
    for (int m = 0; m < 2; ++m) H2[2][m][0] = rsub(p[m], s[m]), H2[2][m][1] = radd(p[m], s[m]);
  }
  // the ply's constants, each as a pair (two pairs per 16-byte load)
  float2 c[14];
#pragma unroll
  for (int k = 0; k < 14; k += 2) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(qp) + k / 2);
    c[k] = make_float2(v.x, v.y);
    c[k + 1] = make_float2(v.z, v.w);
  }
  const float2 half = p2(0.5f);
  float2 E0[2], E1[2];
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    E0[m] = pfma(half, pfma(H0[0][m], H0[0][m], pfma(H0[1][m], H0[1][m], pmul(H0[2][m], H0[2][m]))), H0[0][m]);
    E1[m] = pfma(half, pfma(H1[0][m], H1[0][m], pfma(H1[1][m], H1[1][m], pmul(H1[2][m], H1[2][m]))), H1[1][m]);
    big.m[0] = max_mag(big.m[0], E0[m]);
    big.m[1] = max_mag(big.m[1], E1[m]);
  }
  float2 G0[3][2], G1[3][2], T0[2], T1[2];
  float G2[3][2][2];
#pragma unroll
  for (int iy = 0; iy < 2; ++iy)
#pragma unroll
    for (int ix = 0; ix < 2; ++ix) {
      const float d0 = H2[0][ix][iy], d1 = H2[1][ix][iy], d2 = H2[2][ix][iy];
      const float e2 = rfma(0.5f, rfma(d0, d0, rfma(d1, d1, rmul(d2, d2))), d2);
      big.m[2] = fmaxf(big.m[2], fabsf(e2));
      const float2 a[3] = {H0[0][iy], H0[1][iy], H0[2][iy]}, b[3] = {H1[0][ix], H1[1][ix], H1[2][ix]};
      const float2 d[3] = {p2(d0), p2(d1), p2(d2)};
      const float2 g01 = pfma(a[0], b[0], pfma(a[1], b[1], pfma(a[2], b[2], padd(a[1], b[0]))));
      const float2 g02 = pfma(a[0], d[0], pfma(a[1], d[1], pfma(a[2], d[2], padd(a[2], d[0]))));
      const float2 g12 = pfma(b[0], d[0], pfma(b[1], d[1], pfma(b[2], d[2], padd(b[2], d[1]))));
      big.m[3] = max_mag(big.m[3], g01);
      big.m[4] = max_mag(big.m[4], g02);
      big.m[5] = max_mag(big.m[5], g12);
      const float2 e0 = E0[iy], e1 = E1[ix], ez = p2(e2);
      const float2 S00 = pfma(c[0], e0, pfma(c[1], e1, pfma(c[2], ez, pmul(c[3], g01))));
      const float2 S11 = pfma(c[1], e0, pfma(c[4], e1, pfma(c[5], ez, pmul(c[6], g01))));
      const float2 S22 = pfma(c[2], e0, pfma(c[5], e1, pfma(c[7], ez, pmul(c[8], g01))));
      const float2 S01 = pfma(c[3], e0, pfma(c[6], e1, pfma(c[8], ez, pmul(c[9], g01))));
      const float2 S12 = pfma(c[10], g12, pmul(c[11], g02));
      const float2 S02 = pfma(c[11], g12, pmul(c[12], g02));
      auto add = [&](float2 (&G)[3][2], float2 (&Tk)[2], int k, int m, bool first, float2 Skk, int k1, float2 S1,
                     const float2 (&h1)[3], float2 S2, const float2 (&h2)[3]) {
        Tk[m] = first ? Skk : padd(Tk[m], Skk);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const float2 base = i == k1 ? S1 : S2;
          float2 g;
          if (i == k)
            g = first ? pmul(S1, h1[i]) : pfma(S1, h1[i], G[i][m]);
          else
            g = pfma(S1, h1[i], first ? base : padd(G[i][m], base));
          G[i][m] = pfma(S2, h2[i], g);
        }
      };
      add(G0, T0, 0, iy, ix == 0, S00, 1, S01, b, S02, d);
      add(G1, T1, 1, ix, iy == 0, S11, 0, S01, a, S12, d);
      const float t2 = lane_sum(S22);
      G2[0][ix][iy] = rfma(d0, t2, lane_sum(pfma(S12, b[0], pfma(S02, a[0], S02))));
      G2[1][ix][iy] = rfma(d1, t2, lane_sum(pfma(S12, b[1], pfma(S02, a[1], S12))));
      G2[2][ix][iy] = rfma(d2, t2, radd(t2, lane_sum(pfma(S12, b[2], pmul(S02, a[2])))));
    }
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    G0[0][m] = padd(G0[0][m], T0[m]);
    G1[1][m] = padd(G1[1][m], T1[m]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      G0[i][m] = pfma(H0[i][m], T0[m], G0[i][m]);
      G1[i][m] = pfma(H1[i][m], T1[m], G1[i][m]);
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q[k] = rmul(q[k], box.w);
    qg[k] = rmul(qg[k], box.w);
    qgg[k] = rmul(qgg[k], box.w);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    float C[8];
    column_sums<0, true>(G0[i][0].x, G0[i][0].y, G0[i][1].x, G0[i][1].y, q[0], qg[0], qgg[0], C);
    column_sums<1, false>(G1[i][0].x, G1[i][0].y, G1[i][1].x, G1[i][1].y, q[1], qg[1], qgg[1], C);
    column_sums<2, false>(G2[i][0][0], G2[i][0][1], G2[i][1][0], G2[i][1][1], q[2], qg[2], qgg[2], C);
    raw_nodes(C);
#pragma unroll
    for (int a = 0; a < 8; ++a) f[a][i] = C[bin_of(a)];
  }
}

// The lanes-of-eight evaluation kept out of line for the one-thread form's
// exceptions: it must not weigh on that form's registers.
template <typename T>
__device__ __noinline__ void hex_box_slow(const Dev<T> *D, const Mat<T> *M, int64_t e, bool valid, int mode, T *f) {
  const LaneForce<T> r = hex_lanes8<T, true>(*D, *M, e, valid, mode);
  f[0] = r.f[0];
  f[1] = r.f[1];
  f[2] = r.f[2];
}

// Nodal forces f (by node) of box e at the pass's displacement mirror, and
// its node ids; all 32 lanes of the warp call together, each with its own
// element (valid = false: none).  Returns valid (false too where a repeated
// pass does not evaluate the element).
template <typename T>
__device__ __forceinline__ bool hex_box_pairs_core(const Dev<T> &D, const Mat<T> &M, int64_t e, bool valid, int mode,
                                               T (&f)[8][3], int (&nd)[8]) {
  using V4 = typename Vec4T<T>::type;
  constexpr uint32_t kAll = 0xffffffffu;
  const Ctl *ctl = D.ctl;
  if (mode == MODE_REPEAT && valid) valid = repeat_take(D.rmark_e, e);
  if (!__any_sync(kAll, valid)) return false;
  const int64_t ee = valid ? e : 0;
  const int ub = (mode == MODE_FORCES) ? (ctl->dpar ^ 1) : ctl->dpar;
  const int hb = ctl->hpar;
  const V4 *PDN_STATE_RESTRICT U = D.u4[ub];
  {
    const int4 c0 = __ldg(reinterpret_cast<const int4 *>(D.hex) + 2 * ee);
    const int4 c1 = __ldg(reinterpret_cast<const int4 *>(D.hex) + 2 * ee + 1);
    nd[0] = c0.x, nd[1] = c0.y, nd[2] = c0.z, nd[3] = c0.w;
    nd[4] = c1.x, nd[5] = c1.y, nd[6] = c1.z, nd[7] = c1.w;
  }
#ifdef PDN_CHECK
  if (!nodes_in_range(D, nd)) {
    valid = false;
#pragma unroll
    for (int a = 0; a < 8; ++a) nd[a] = 0;
  }
#endif
  if (mode == MODE_REPEAT && valid) repeat_mark_nodes(D.rmark_n, nd);
  const bool pristine = D.pflag[hb][ee] != 0;
  // the elastic form, unless every element of the warp has a history (FP64, all
  // of 393,216 hexes damaged: 3,290 to 2,825 us per step)
  bool ok = false;
  if (__any_sync(kAll, valid && pristine)) {
    const V4 box = D.box[ee];
    const int ply = D.ply[ee];
    T u[8][3];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const V4 v = U[nd[a]];
      u[a][0] = v.x;
      u[a][1] = v.y;
      u[a][2] = v.z;
    }
    StrainMag<T> big;
    hex_box_elastic(u, box, D.ply_q + (int64_t)kPlyStride<T> * ply, f, big);
    ok = pristine && big.largest() < mag_bits(M.e_tol);
    if (pristine && !ok) {
      const float a[6] = {big.upper(0), big.upper(1), big.upper(2), big.upper(3), big.upper(4), big.upper(5)};
      ok = clear_of_onset(M.onset, (float)M.ply_c[ply], (float)M.ply_s[ply], a);
    }
  }
  if (valid && ok) D.pflag[hb ^ 1][ee] = 1;
  uint32_t bad = __ballot_sync(kAll, valid && !ok);
  while (bad != 0u) {
    // the next four elements, one per group of eight lanes
    const int lane = (int)(threadIdx.x & 31), grp = lane >> 3;
    int src = -1, mine = -1;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int l = bad != 0u ? __ffs(bad) - 1 : -1;
      bad &= bad - 1u;
      if (g == grp) src = l;
      if (l == lane) mine = g;
    }
    const int64_t es = __shfl_sync(kAll, (long long)ee, src < 0 ? 0 : src);
    T r[3];
    hex_box_slow<T>(&D, &M, es, src >= 0, mode, r);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      // lane of corner a in a group: xi, eta, zeta bits
      const int sub = bin_of(a);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const T v = __shfl_sync(kAll, r[i], (mine < 0 ? 0 : mine) * 8 + sub);
        if (mine >= 0) f[a][i] = v;
      }
    }
  }
  return valid;
}

}  // namespace detail
}  // namespace pdn
