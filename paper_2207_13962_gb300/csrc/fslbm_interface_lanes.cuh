// Interface update of one band cell by a warp (arXiv 2207.13962, Sec. 2.2 and
// 3), the lanes being the lattice directions: the form of interface_cell for
// short bands.
//
// A thread a cell runs 3000 to 8000 instructions in a row, so a band of a few
// warps takes 25 us (FP32) to 45 us (FP64) on a few SMs whatever its size,
// while the others idle. With a direction a lane the same update is a few
// hundred instructions, a warp a cell, over all SMs. It needs more
// instructions in all (the sums over the directions run once a cell instead
// of once for 32), so long bands keep a thread a cell; see lane_band.
//
// Every value is that of interface_cell: sums run over the lanes in direction
// order (terms that it leaves out enter as zeros), and the pair (i, ibar)
// shares products whose sign flips exactly.
#pragma once

#include "fslbm_convert.cuh"

namespace fslbm {

// A lane's direction with its weight and components in the arithmetic type.
template <int Q, class R>
struct LaneLattice {
  LaneDir l;
  int opp;  // lane of the opposite direction
  bool own; // the lane holds a PDF
  R cx, cy, cz, w;
  unsigned pos, neg;  // FP64 sums: directions the lane's component adds / subtracts
};

// Directions whose component a (0 x, 1 y, 2 z) has the sign s; all for a = -1.
template <int Q>
__host__ __device__ constexpr unsigned dirs_with(int a, int s) {
  unsigned m = 0;
  for (int i = 0; i < Q; ++i) {
    const int c = a < 0 ? 1 : a == 0 ? CX(i) : a == 1 ? CY(i) : CZ(i);
    if (c == s) m |= 1u << i;
  }
  return m;
}

template <int Q, class R>
__device__ __forceinline__ LaneLattice<Q, R> lane_lattice() {
  LaneLattice<Q, R> t;
  t.l = lane_dir<Q>();
  t.own = t.l.i < Q;
  t.opp = t.l.moving ? ((t.l.i & 1) ? t.l.i + 1 : t.l.i - 1) : t.l.i;
  t.cx = R(t.l.dx);
  t.cy = R(t.l.dy);
  t.cz = R(t.l.dz);
  t.w = lane_weight<Q, R>(t.l.dx * t.l.dx + t.l.dy * t.l.dy + t.l.dz * t.l.dz);
  constexpr unsigned kAll = dirs_with<Q>(-1, 1), kXp = dirs_with<Q>(0, 1), kXm = dirs_with<Q>(0, -1),
                     kYp = dirs_with<Q>(1, 1), kYm = dirs_with<Q>(1, -1), kZp = dirs_with<Q>(2, 1),
                     kZm = dirs_with<Q>(2, -1);
  const int q = t.l.i & 3;
  t.pos = q == 0 ? kAll : q == 1 ? kXp : q == 2 ? kYp : kZp;
  t.neg = q == 0 ? 0u : q == 1 ? kXm : q == 2 ? kYm : kZm;
  return t;
}

// sum f, sum c_x f, sum c_y f, sum c_z f over the lanes, in direction order.
// FP64: lane q < 4 forms the q-th sum (one addition a direction for all four:
// an FP64 instruction takes 16 clocks of the SM's unit whatever its lanes).
template <int Q>
__device__ __forceinline__ void lane_sums(const LaneLattice<Q, float>&, float f, float& r, float& jx, float& jy,
                                          float& jz) {
  r = jx = jy = jz = 0.f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float v = __shfl_sync(0xffffffffu, f, i);
    r = r + v;
    if (CX(i) != 0) jx = CX(i) > 0 ? jx + v : jx - v;
    if (CY(i) != 0) jy = CY(i) > 0 ? jy + v : jy - v;
    if (CZ(i) != 0) jz = CZ(i) > 0 ? jz + v : jz - v;
  }
}
template <int Q>
__device__ __forceinline__ double lane_sums64(const LaneLattice<Q, double>& t, double f) {
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const double v = __shfl_sync(0xffffffffu, f, i);
    const double a = ((t.neg >> i) & 1u) ? -v : v;
    s = s + ((((t.pos | t.neg) >> i) & 1u) ? a : 0.0);
  }
  return s;
}

// Velocity j / rho + sign g / 2 and density from the sums of f.
template <int Q>
__device__ __forceinline__ void lane_moments(const LaneLattice<Q, double>& t, double f, const KParams& p,
                                             double sign, double& rho, double u[3]) {
  const double s = lane_sums64<Q>(t, f);
  rho = __shfl_sync(0xffffffffu, s, 0);
  const int q = t.l.i & 3;
  const double g = q == 1 ? p.g[0] : q == 2 ? p.g[1] : p.g[2];
  const double v = s / rho + sign * (0.5 * g);
  u[0] = __shfl_sync(0xffffffffu, v, 1);
  u[1] = __shfl_sync(0xffffffffu, v, 2);
  u[2] = __shfl_sync(0xffffffffu, v, 3);
}

// collide() with a direction a lane: f* of the lane's direction; rho returned.
template <int Q, int COLL>
__device__ __forceinline__ double lane_collide(const LaneLattice<Q, double>& t, double& f, const KParams& p,
                                               bool& unstable) {
  using R = double;
  R rho, u[3];
  lane_moments<Q>(t, f, p, 1.0, rho, u);
  const R Fx = rho * p.g[0], Fy = rho * p.g[1], Fz = rho * p.g[2];
  const R usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  if (!(usq < R(1.0 / 3.0)) || !(rho > R(0.0))) unstable = true;
  R omega = p.omega;
  const R b = R(1.5) * usq;
  const R uF = u[0] * Fx + u[1] * Fy + u[2] * Fz;
  const R cu = t.cx * u[0] + t.cy * u[1] + t.cz * u[2];
  const R cF = t.cx * Fx + t.cy * Fy + t.cz * Fz;
  R e, eo, s, so;  // f^eq and source of the lane's direction and its opposite
  feq_pair<R>(t.w * rho, cu, b, e, eo);
  guo_pair<R>(t.w, cu, cF, uF, s, so);
  const R fo = __shfl_sync(0xffffffffu, f, t.opp);
  if constexpr (coll_les(COLL)) {
    const R dn = f - e;
    R qxx = R(0.0), qyy = R(0.0), qzz = R(0.0), qxy = R(0.0), qxz = R(0.0), qyz = R(0.0);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const R v = __shfl_sync(0xffffffffu, dn, i);
      if (CX(i) != 0) qxx = qxx + v;
      if (CY(i) != 0) qyy = qyy + v;
      if (CZ(i) != 0) qzz = qzz + v;
      if (CX(i) * CY(i) != 0) qxy = CX(i) * CY(i) > 0 ? qxy + v : qxy - v;
      if (CX(i) * CZ(i) != 0) qxz = CX(i) * CZ(i) > 0 ? qxz + v : qxz - v;
      if (CY(i) * CZ(i) != 0) qyz = CY(i) * CZ(i) > 0 ? qyz + v : qyz - v;
    }
    omega = R(1.0) / les_tau<R>(qxx, qyy, qzz, qxy, qxz, qyz, rho, omega, p.cs);
  }
  if constexpr (!coll_trt(COLL)) {
    const R pref = coll_les(COLL) ? R(1.0) - R(0.5) * omega : p.pref_p;
    f = f - omega * (f - e) + pref * s;
  } else {
    // the rest lane is its own opposite: its antisymmetric parts vanish
    R omp = p.omega, omm = p.om_m, prp = p.pref_p, prm = p.pref_m;
    if constexpr (coll_les(COLL)) {
      omp = omega;
      omm = R(1.0) / (R(0.5) + p.magic / (R(1.0) / omp - R(0.5)));
      prp = R(1.0) - R(0.5) * omp;
      prm = R(1.0) - R(0.5) * omm;
    }
    const R A = (R(0.5) * omp) * ((f + fo) - (e + eo));
    const R B = (R(0.5) * omm) * ((f - fo) - (e - eo));
    const R C = (R(0.5) * prp) * (s + so);
    const R D = (R(0.5) * prm) * (s - so);
    f = f - A - B + C + D;
  }
  return rho;
}

// collide_dev() with a direction a lane; drho returned.
template <int Q, int COLL>
__device__ __forceinline__ float lane_collide(const LaneLattice<Q, float>& t, float& d, const KParams& p,
                                              bool& unstable) {
  float dr, jx, jy, jz;
  lane_sums<Q>(t, d, dr, jx, jy, jz);
  const float rho = 1.0f + dr;
  const float gx = p.fg[0], gy = p.fg[1], gz = p.fg[2];
  const float inv = __frcp_rn(rho);
  const float ux = __fmaf_rn(jx, inv, 0.5f * gx), uy = __fmaf_rn(jy, inv, 0.5f * gy),
              uz = __fmaf_rn(jz, inv, 0.5f * gz);
  const float Fx = rho * gx, Fy = rho * gy, Fz = rho * gz;
  const float usq = __fmaf_rn(ux, ux, __fmaf_rn(uy, uy, uz * uz));
  if (!(usq < 1.0f / 3.0f) || !(rho > 0.f)) unstable = true;
  float omp = p.fomega, prp = p.fpref_p;
  float omm = coll_trt(COLL) ? p.fom_m : omp, prm = coll_trt(COLL) ? p.fpref_m : prp;
  const float base = __fmaf_rn(-1.5f * rho, usq, dr);
  const float r45 = 4.5f * rho;
  const float cu = t.cx * ux + t.cy * uy + t.cz * uz;
  const float cF = t.cx * Fx + t.cy * Fy + t.cz * Fz;
  const float es = t.w * __fmaf_rn(r45 * cu, cu, base);
  const float dd = __shfl_sync(0xffffffffu, d, t.opp);
  if constexpr (coll_les(COLL)) {
    const float dn = __fmaf_rn(-2.0f, es, d + dd);  // the same for i and ibar
    float qxx = 0.f, qyy = 0.f, qzz = 0.f, qxy = 0.f, qxz = 0.f, qyz = 0.f;
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const float v = __shfl_sync(0xffffffffu, dn, i);
      if (CX(i) != 0) qxx += v;
      if (CY(i) != 0) qyy += v;
      if (CZ(i) != 0) qzz += v;
      if (CX(i) * CY(i) != 0) qxy = CX(i) * CY(i) > 0 ? qxy + v : qxy - v;
      if (CX(i) * CZ(i) != 0) qxz = CX(i) * CZ(i) > 0 ? qxz + v : qxz - v;
      if (CY(i) * CZ(i) != 0) qyz = CY(i) * CZ(i) > 0 ? qyz + v : qyz - v;
    }
    omp = 1.0f / les_tau<float>(qxx, qyy, qzz, qxy, qxz, qyz, rho, omp, p.fcs);
    prp = 1.0f - 0.5f * omp;
    if constexpr (coll_trt(COLL)) {
      omm = 1.0f / (0.5f + p.fmagic / (1.0f / omp - 0.5f));
      prm = 1.0f - 0.5f * omm;
    } else {
      omm = omp;
      prm = prp;
    }
  }
  const float uF3 = 3.0f * __fmaf_rn(ux, Fx, __fmaf_rn(uy, Fy, uz * Fz));
  // ibar's antisymmetric parts are exact negations of i's
  const float ea = (3.0f * t.w) * rho * cu;
  const float ss = t.w * __fmaf_rn(9.0f * cu, cF, -uF3);
  const float sa = (3.0f * t.w) * cF;
  const float fp = 0.5f * (d + dd);
  const float fm = 0.5f * (d - dd);
  const float A = __fmaf_rn(omp, fp - es, -prp * ss);
  const float B = __fmaf_rn(omm, fm - ea, -prm * sa);
  const float t0 = __fmaf_rn(-t.w, base, d);
  const float rest = __fmaf_rn(-omp, t0, __fmaf_rn(-prp * t.w, uF3, d));
  d = t.l.i == 0 ? rest : d - A - B;
  return dr;
}

// interface_cell for list entry k, one warp.
template <int Q, class S, int COLL>
__device__ __forceinline__ void interface_lanes(const DPtrs& d, const KParams& p, int parity,
                                                const LaneLattice<Q, typename S::Real>& t, int k, bool& bad) {
  using R = typename S::Real;
  using T = typename S::T;
  const T* __restrict__ A = (const T*)d.pdf[parity];
  T* __restrict__ B = (T*)d.pdf[parity ^ 1];
  const long long Np = p.Np;
  const LaneDir& l = t.l;
  const int c = d.band[parity][k];
  const uint8_t fl = d.flags[c];
  const uint32_t wm = (fl & F_NEAR_WALL) ? d.wallmask[c] : 0u;
  // the lane's pull source x - c_i (-1 outside the domain) and the PDF that
  // arrives from it; at a free-slip face the mirror image
  int src = -1, dir = l.i;
  bool mir = false;
  if (fl & (F_FACE | F_WRAP)) {
    int x, y, z;
    decode(p, c, x, y, z);
    if (coll_slip(COLL)) {
      int X = x - l.dx, Y = y - l.dy, Z = z - l.dz, m = 0;
      bool out = false;
      if (X < 0 || X >= p.nx) {
        if (p.per[0]) X = X < 0 ? X + p.nx : X - p.nx;
        else if (p.slip[0]) X = x, m |= 1;
        else out = true;
      }
      if (Y < 0 || Y >= p.ny) {
        if (p.per[1]) Y = Y < 0 ? Y + p.ny : Y - p.ny;
        else if (p.slip[1]) Y = y, m |= 2;
        else out = true;
      }
      if (Z < 0 || Z >= p.nz) {
        if (p.per[2]) Z = Z < 0 ? Z + p.nz : Z - p.nz;
        else if (p.slip[2]) Z = z, m |= 4;
        else out = true;
      }
      mir = m != 0;
      if (l.moving && !out) {
        src = cidx(p, X, Y, Z);
        if (mir) dir = (int)kReflect.j[l.i][m];
      }
    } else if (l.moving) {
      src = nbr(p, x, y, z, -l.dx, -l.dy, -l.dz);
    }
  } else if (l.moving) {
    src = c - (l.dx * p.sx + l.dy * p.sy + l.dz * p.sz);
  }
  // one level of loads
  const int kind = src >= 0 ? (int)d.cls[src] : (int)T_OBST;
  R phs = R(0.0), phc;
  if constexpr (S::kDev) {
    if (src >= 0) phs = d.phif[src];
    phc = d.phif[c];
  } else {
    if (src >= 0) phs = d.phi[src];
    phc = d.phi[c];
  }
  const int clc = d.cls[c] >> 2;
  const R fx = t.own ? load_own_lane<Q, S>(A, Np, c, l.i, t.w) : R(0.0);
  R f = fx;  // the rest PDF stays in the cell
  if (l.moving) {
    // bounce-back where the source is outside or an obstacle (the wall mask,
    // but for mirror images: their type)
    const bool back = mir ? (kind & 3) == T_OBST : src < 0 || ((wm >> l.i) & 1u);
    f = load_lane<S>(A[(long long)(back ? t.opp : dir) * Np + (back ? c : src)], t.w);
  }
  const R* nhat = (const R*)d.nhat;
  const R n0 = nhat[3LL * c], n1 = nhat[3LL * c + 1], n2 = nhat[3LL * c + 2];
  const R rg = ((const R*)d.rhog)[c];  // rho^G (FP64 engine) or rho^G - 1
  const double m0 = d.mass[c];
  const bool gas = l.moving && (kind & 3) == T_GAS;
  const unsigned miss = __ballot_sync(0xffffffffu, gas);
  if (gas) f = R(0.0);
  // mass exchange: this lane forms the term of the opposite direction i, whose
  // neighbour x + c_i is the lane's source; a = f_ibar is the lane's PDF
  const R fb = __shfl_sync(0xffffffffu, fx, t.opp);
  const int ntp = l.moving ? (kind & 3) : (int)T_OBST, cln = kind >> 2;
  R v;
  if (clc == cln) v = f - fb;
  else if (clc == CL_STD) v = (cln == CL_NF) ? (S::kDev ? f + t.w : f) : -(S::kDev ? fb + t.w : fb);
  else if (clc == CL_NF) v = -(S::kDev ? fb + t.w : fb);
  else v = S::kDev ? f + t.w : f;
  double dm;
  if constexpr (S::kDev) {
    float s = 0.f, e = 0.f;
    if (ntp == T_LIQ) {
      s = __fsub_rn(f, fb);
      const float bv = __fsub_rn(s, f);
      e = __fsub_rn(__fsub_rn(f, __fsub_rn(s, bv)), __fadd_rn(fb, bv));
    } else if (ntp == T_IFACE) {
      s = __fmul_rn(__fmul_rn(0.5f, __fadd_rn(phc, phs)), v);
    }
    FAcc acc;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      acc.add(__shfl_sync(0xffffffffu, s, OPP(i)));
      acc.lo = __fadd_rn(acc.lo, __shfl_sync(0xffffffffu, e, OPP(i)));
    }
    dm = acc.value();
  } else {
    double s = 0.0;
    if (ntp == T_LIQ) s = f - fb;
    else if (ntp == T_IFACE) s = 0.5 * (phc + phs) * v;
    dm = 0.0;
#pragma unroll
    for (int i = 1; i < Q; ++i) dm = dm + __shfl_sync(0xffffffffu, s, OPP(i));
  }
  const double mn = m0 + dm;
  // BC velocity from the cell's own post-collision PDFs
  R rc, u[3];
  if constexpr (S::kDev) {
    R jx, jy, jz;
    lane_sums<Q>(t, fx, rc, jx, jy, jz);
    rc = R(1.0) + rc;
    u[0] = jx / rc - R(0.5) * p.fg[0];
    u[1] = jy / rc - R(0.5) * p.fg[1];
    u[2] = jz / rc - R(0.5) * p.fg[2];
  } else {
    lane_moments<Q>(t, fx, p, -1.0, rc, u);
  }
  // set R of the variant (Sec. 3) and reconstruction
  int var = p.variant;
  if (var == 4) var = (__popc(miss) >= 3) ? 3 : p.om3_fb;
  const R tie = R(0x1p-20);
  const R dot = t.cx * n0 + t.cy * n1 + t.cz * n2;
  const bool rec = gas || (var == 1 && dot >= -tie) || (var == 2 && dot > tie);
  {
    const R usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const R b = R(1.5) * usq;
    const R cu = t.cx * u[0] + t.cy * u[1] + t.cz * u[2];
    R e;
    if constexpr (S::kDev) {
      const R rgf = R(1.0) + rg, c3 = R(3.0) * cu, a = R(4.5) * cu * cu;
      e = t.w * (rg + rgf * (c3 + a - b)) + t.w * (rg + rgf * (a - c3 - b));
    } else {
      R ei, ej;
      feq_pair<R>(t.w * rg, cu, b, ei, ej);
      e = ei + ej;
    }
    if (rec) f = e - fb;
  }
  if (!t.own) f = R(0.0);
  long long s_in = 0;  // the mass-conserving formats: the received values in grid steps
  if constexpr (S::kExactRest) {
    s_in = t.own ? grid_steps<S>(f) : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s_in += __shfl_xor_sync(0xffffffffu, s_in, o);
  }
  double rho;
  if constexpr (S::kDev) rho = 1.0 + (double)lane_collide<Q, COLL>(t, f, p, bad);
  else rho = lane_collide<Q, COLL>(t, f, p, bad);
  // store, and the moments of the stored post-collision PDFs
  const T st = lane_store<S>(f, t.w);
  if constexpr (S::kDev) {
    R fs = t.own ? S::loadd(st) : R(0.0);
    double sd;
    if constexpr (S::kExactRest) {
      constexpr float kRange = 2147483648.0f / (float)(1LL << S::kShift);
      if (l.moving && !(fabsf(f) < kRange)) bad = true;
      long long steps = l.moving ? (long long)S::steps(st) : 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) steps += __shfl_xor_sync(0xffffffffu, steps, o);
      long long r = s_in - steps;
      if (r > 2147483647LL || r < -2147483647LL) {
        bad = true;
        r = r > 0 ? 2147483647LL : -2147483647LL;
      }
      if (l.moving) B[(long long)l.i * Np + c] = st;
      if (l.i == 0) {
        rest_slice<Q, S>(B, Np)[c] = (int)r;
        fs = from_steps<S>(r);
      }
      sd = (double)(r + steps) * (1.0 / (double)(1LL << S::kShift));
    } else {
      if (t.own) B[(long long)l.i * Np + c] = st;
    }
    R r0, jx0, jy0, jz0;
    lane_sums<Q>(t, fs, r0, jx0, jy0, jz0);
    if constexpr (!S::kExactRest) {
      FAcc sa;
#pragma unroll
      for (int i = 0; i < Q; ++i) sa.add(__shfl_sync(0xffffffffu, fs, i));
      sd = sa.value();
    }
    rho = 1.0 + sd;
    const R rr = R(rho);
    const R j = l.i == 0 ? jx0 : l.i == 1 ? jy0 : jz0;
    const R g = l.i == 0 ? p.fg[0] : l.i == 1 ? p.fg[1] : p.fg[2];
    if (l.i < 3) ((R*)d.mom_u)[3LL * c + l.i] = j / rr - R(0.5) * g;
    if (l.i == 0) d.mom_rho[c] = rho;
  } else {
    if (t.own) B[(long long)l.i * Np + c] = st;
    R r0, mu[3];
    lane_moments<Q>(t, f, p, -1.0, r0, mu);
    if (l.i < 3) ((R*)d.mom_u)[3LL * c + l.i] = l.i == 0 ? mu[0] : l.i == 1 ? mu[1] : mu[2];
    if (l.i == 0) {
      d.mom_rho[c] = r0;
      d.rho_band[c] = rho;
    }
  }
  if (fl & F_NEAR_WALL) {
    // reflected copy into the slot of an obstacle pull source (a cell of the
    // domain, never a mirror image)
    const R fo = __shfl_sync(0xffffffffu, f, t.opp);
    if (l.moving && ((wm >> l.i) & 1u)) {
      int slot = src;
      if (coll_slip(COLL) && (fl & (F_FACE | F_WRAP))) {
        int x, y, z;
        decode(p, c, x, y, z);
        slot = nbr(p, x, y, z, -l.dx, -l.dy, -l.dz);
      }
      B[(long long)l.i * Np + slot] = lane_store<S>(fo, t.w);
    }
  }
  if (l.i == 0) {
    double phin;
    if constexpr (S::kDev) {
      const double r0 = (double)__frcp_rn(d2f(rho));
      const double q0 = mn * r0;
      phin = fma(fma(-q0, rho, mn), r0, q0);
    } else {
      phin = mn / rho;
    }
    d.m_next[k] = mn;
    d.phi_next[k] = phin;
    const uint8_t mark = (phin > 1.0 + p.eps) ? CV_TOL : (phin < -p.eps) ? CV_TOG : CV_NONE;
    d.mark[c] = mark;
    if (mark != CV_NONE) append_conversion(d, parity, c);
  }
}

// Whether a band of n cells is updated a warp a cell: the line where the
// instructions of a warp on one cell's lanes cost more than the idle SMs.
// Measured (us, the stage with its launch gap; threads / lanes): FP32 D3Q19
// 266 cells 19 / 12, 4272 18 / 16, 4941 19 / 18, 11183 20 / 25; FP32 D3Q27
// 710 22 / 13, 5103 23 / 19, 11526 24 / 27; FP16SMC D3Q27 5092 27 / 19, 11583
// 28 / 27; FP64 D3Q19 66 43 / 18, 1064 43 / 33, 2136 43 / 50.
template <int Q, class S>
__device__ __forceinline__ bool lane_band(int n) {
  return n <= (S::kDev ? (Q == 19 ? 5120 : 8192) : 1280);
}

// The two forms share a kernel, whose block size and registers are those of
// the thread form; the lane form is a function of its own, not inlined, so
// that the thread form's code stays what it is alone (inlined beside it, it
// took 50 instead of 43 us on the 160x160x1024 tube; as a kernel beside it in
// the graph, the fork cost both forms 5 to 10 us).
template <int Q, class S, int COLL>
__device__ __noinline__ void interface_by_lanes(const DPtrs& d, const KParams& p, int parity, int n) {
  const LaneLattice<Q, typename S::Real> t = lane_lattice<Q, typename S::Real>();
  bool bad = false;
  for (int k = spread_warp(); k < n; k += spread_warps()) interface_lanes<Q, S, COLL>(d, p, parity, t, k, bad);
  if (bad) d.err[0] = 1;
}

// total: cells of all domains, each domain's rounded up to whole warps.
template <int Q, class S, int COLL>
__device__ __noinline__ void interface_by_lanes(const DomRec* recs, const int* off, int n, int total) {
  const LaneLattice<Q, typename S::Real> t = lane_lattice<Q, typename S::Real>();
  for (int g = spread_warp(); g < total; g += spread_warps()) {
    const int k = find_domain(off, n, g);
    const DomRec& r = recs[k];
    const int i = g - off[k];
    if (i >= r.d.counts[r.parity]) continue;
    bool bad = false;
    interface_lanes<Q, S, COLL>(r.d, r.p, r.parity, t, i, bad);
    if (bad) r.d.err[0] = 1;
  }
}

}  // namespace fslbm
