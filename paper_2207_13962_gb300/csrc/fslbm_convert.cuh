// Conversion and excess-mass stages of the FSLBM step (arXiv 2207.13962,
// Sec. 2.2: conversion thresholds, neighbour fix-up, PDFs of new interface
// cells, Eq. nm-fslbm-excess-mass) on compact lists, a warp a cell.
//
// Only a few cells of the band convert in a step (0 to a few per cent), and
// each stage is a chain of dependent neighbour reads around such a cell.  A
// thread a cell runs that chain alone, as thousands of straight-line
// instructions on a few active lanes: the stages then wait for instruction
// fetches and one lane's loads whatever the number of cells.  Here the lanes
// of a warp are the lattice directions of one cell: a level of the chain is
// one load instruction, the code is a few hundred instructions, and a stage
// visits only the cells it concerns:
//   interface kernel  appends the cells it marks to the conversion list
//   k_resolve         conflict rule and claims of the listed cells (and the
//                     commit of m and phi of the whole band)
//   k_count           receivers and shares of the listed cells; appends the
//                     interface cells that will receive to the receiver list
//   k_apply           new cells, receivers and listed cells
// Ordered sums run over the lanes in direction order, so every value is that
// of a per-direction loop.  Measured on the 37x21x11 tank (D3Q27, a few per
// cent of 700 cells converting): resolve, count and apply 10 + 10 + 33 us as
// thread-a-cell kernels.
//
// The lists live in arrays that are idle at that time: the conversion list in
// the other parity's band list (rewritten at the end of the step), the
// receiver list in the normals (dead after the interface kernel, rewritten by
// the next geometry pass).
#pragma once

#include "fslbm_cell.cuh"

namespace fslbm {

__device__ __forceinline__ int* conv_list(const DPtrs& d, int parity) { return d.band[parity ^ 1]; }
__device__ __forceinline__ int* recv_list(const DPtrs& d) { return (int*)d.nhat; }
// counters of the two lists (cleared with the step's other counters)
__device__ __forceinline__ int* conv_count(const DPtrs& d) { return &d.counts[8]; }
__device__ __forceinline__ int* recv_count(const DPtrs& d) { return &d.counts[9]; }

// rho of a band cell after its collision: the moment cache holds it in the
// deviation formats; in FP64 the cache holds the sum of the post-collision
// PDFs, whose rounding differs, so the collision's own value is kept beside it.
template <class S>
__device__ __forceinline__ double band_rho(const DPtrs& d, int c) {
  if constexpr (S::kDev) return d.mom_rho[c];
  else return d.rho_band[c];
}

// Appends a marked cell to the conversion list; called by the active lanes
// of a divergent warp (one atomic for the lanes that arrive together).
__device__ __forceinline__ void append_conversion(const DPtrs& d, int parity, int c) {
  const unsigned act = __activemask();
  const unsigned lane = threadIdx.x & 31u;
  const int lead = __ffs(act) - 1;
  int base = 0;
  if ((int)lane == lead) base = atomicAdd(conv_count(d), __popc(act));
  base = __shfl_sync(act, base, lead);
  conv_list(d, parity)[base + __popc(act & ((1u << lane) - 1u))] = c;
}

// Direction codes for lanes (dcode as a table).
struct DirCodes {
  unsigned char v[32];
};
__host__ __device__ constexpr DirCodes make_dir_codes() {
  DirCodes t{};
  for (int i = 0; i < 32; ++i) t.v[i] = (unsigned char)(i < 27 ? dcode(i) : 13);
  return t;
}
__constant__ constexpr DirCodes kDirCodes = make_dir_codes();

// Lane i of a warp stands for direction i of the cell the warp works on.
struct LaneDir {
  int i, dx, dy, dz;
  bool moving;  // a direction 1..Q-1
};
template <int Q>
__device__ __forceinline__ LaneDir lane_dir() {
  LaneDir l;
  l.i = threadIdx.x & 31;
  const int code = kDirCodes.v[l.i];
  l.dx = code % 3 - 1;
  l.dy = (code / 3) % 3 - 1;
  l.dz = code / 9 - 1;
  l.moving = l.i >= 1 && l.i < Q;
  return l;
}

// Warp number in the grid, counted over the blocks first: consecutive work
// items then go to different SMs.
__device__ __forceinline__ int spread_warp() { return (threadIdx.x >> 5) * gridDim.x + blockIdx.x; }
__device__ __forceinline__ int spread_warps() { return gridDim.x * (blockDim.x >> 5); }

// The lane's neighbour x + c_i of cell c (flag byte fl), -1 outside the
// domain (and for lanes without a direction), and its type.
__device__ __forceinline__ int lane_neighbour(const DPtrs& d, const KParams& p, const LaneDir& l, int c,
                                              uint8_t fl, int& type) {
  int n = -1;
  if (fl & (F_FACE | F_WRAP)) {
    int x, y, z;
    decode(p, c, x, y, z);
    if (l.moving) n = nbr(p, x, y, z, l.dx, l.dy, l.dz);
  } else if (l.moving) {
    n = c + l.dx * p.sx + l.dy * p.sy + l.dz * p.sz;
  }
  type = n >= 0 ? (int)(d.flags[n] & F_TYPE) : (int)T_OBST;
  return n;
}

// Sets byte 0/1 mark number n of a byte array with an atomic; true for the
// caller that set it.
__device__ __forceinline__ bool claim_byte(uint8_t* bytes, int n) {
  const unsigned bit = 1u << (8 * (n & 3));
  return !(atomicOr((unsigned*)(bytes + (n & ~3)), bit) & bit);
}

// Warp-wide append of lanes with `fresh` to a list.
__device__ __forceinline__ void warp_push(int* list, int* counter, bool fresh, int value) {
  const unsigned m = __ballot_sync(0xffffffffu, fresh);
  if (!m) return;
  const unsigned lane = threadIdx.x & 31u;
  int base = 0;
  if (lane == 0) base = atomicAdd(counter, __popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (fresh) list[base + __popc(m & ((1u << lane) - 1u))] = value;
}

// Sum over the set lanes of mask m of v, in lane (= direction) order.
__device__ __forceinline__ double ordered_sum(unsigned m, double v, double s) {
  while (m) {
    const int i = __ffs(m) - 1;
    m &= m - 1u;
    s = s + __shfl_sync(0xffffffffu, v, i);
  }
  return s;
}

// Conflict rule (a cell marked for gas stays interface next to a cell marked
// for liquid); claims of the gas neighbours of cells turning liquid and of
// the liquid neighbours of cells turning gas as new interface cells.  List
// entry j, one warp.
template <int Q>
__device__ __forceinline__ void resolve_listed(const DPtrs& d, const KParams& p, int parity, const LaneDir& l,
                                               int j) {
  const int c = conv_list(d, parity)[j];
  const uint8_t fl = d.flags[c];
  uint8_t cv = d.mark[c];
  int t;
  const int n = lane_neighbour(d, p, l, c, fl, t);
  if (cv == CV_TOG) {
    const uint8_t mk = n >= 0 ? d.mark[n] : (uint8_t)CV_NONE;
    if (__any_sync(0xffffffffu, t == T_IFACE && mk == CV_TOL)) cv = CV_NONE;
  }
  if (l.i == 0) d.conv[c] = cv;
  if (cv == CV_NONE) return;
  const int want = cv == CV_TOL ? T_GAS : T_LIQ;
  const bool fresh = t == want && claim_byte(d.claim, n);
  warp_push(d.newlist, &d.counts[2], fresh, n);
}

// Commits m and phi of band entry k (the interface kernel's neighbours read
// the old values).  A sum with +0 makes a zero positive, as the excess
// gather of a cell that receives nothing does.
__device__ __forceinline__ void commit_cell(const DPtrs& d, int parity, int k) {
  const int c = d.band[parity][k];
  d.mass[c] = d.m_next[k] + 0.0;
  set_phi(d, c, d.phi_next[k] + 0.0);
}

// Excess-mass receivers (Eq. nm-fslbm-excess-mass) of list entry j:
// interface cells after conversion in the lattice neighbourhood (interface
// cells that do not convert, and the gas or liquid cells that conversion
// claims); none -> the conversion is deferred.  The interface neighbours go
// to the receiver list.
template <int Q, class S>
__device__ __forceinline__ void count_listed(const DPtrs& d, const KParams& p, int parity, const LaneDir& l,
                                             int j) {
  const int c = conv_list(d, parity)[j];
  const uint8_t cv = d.conv[c];
  if (cv == CV_NONE) return;
  const uint8_t fl = d.flags[c];
  int t;
  const int n = lane_neighbour(d, p, l, c, fl, t);
  const uint8_t cn = n >= 0 ? d.conv[n] : (uint8_t)0, cl = n >= 0 ? d.claim[n] : (uint8_t)0;
  const bool post = t == T_IFACE ? cn == CV_NONE : t != T_OBST && cl != 0;
  const int nrecv = __popc(__ballot_sync(0xffffffffu, post));
  if (nrecv == 0) {
    if (l.i == 0) d.cfin[c] = CV_DEFER;
    return;
  }
  if (l.i == 0) {
    const double m = d.mass[c];
    const double mex = (cv == CV_TOL) ? (m - band_rho<S>(d, c)) : m;
    d.share[c] = mex / (double)nrecv;
    d.cfin[c] = cv;
  }
  const bool fresh = t == T_IFACE && claim_byte(d.rcv, n);
  warp_push(recv_list(d), recv_count(d), fresh, n);
}

__device__ __forceinline__ bool is_converted(int f) { return f == CV_TOL || f == CV_TOG; }

// A receiver: m + the shares of its converted neighbours, in direction
// order.  Cells that convert themselves, and deferred cells (they keep their
// mass), only clear their mark.
template <int Q, class S>
__device__ __forceinline__ void apply_receiver(const DPtrs& d, const KParams& p, const LaneDir& l, int c) {
  const uint8_t fl = d.flags[c];
  const uint8_t own = d.cfin[c];
  if (l.i == 0) d.rcv[c] = 0;
  if (own != CV_NONE) return;
  int t;
  const int n = lane_neighbour(d, p, l, c, fl, t);
  const int cf = n >= 0 ? (int)d.cfin[n] : (int)CV_NONE;
  const double sh = n >= 0 ? d.share[n] : 0.0;
  const bool from = t == T_IFACE && is_converted(cf);
  const double s = ordered_sum(__ballot_sync(0xffffffffu, from), sh, 0.0);
  if (l.i == 0) {
    const double m = d.mass[c] + s;
    d.mass[c] = m;
    set_phi(d, c, m / band_rho<S>(d, c));
  }
}

// A listed cell after conversion: liquid and gas cells' own fields.
template <class S>
__device__ __forceinline__ void apply_converted(const DPtrs& d, int c) {
  const uint8_t f = d.cfin[c];
  if (f == CV_TOL) {
    set_phi(d, c, 1.0);
    d.mass[c] = band_rho<S>(d, c);
  } else if (f == CV_TOG) {
    set_phi(d, c, 0.0);
    d.mass[c] = 0.0;
  }
}

// A new interface cell (gas or liquid before this step).  From gas: f* =
// f^eq(mean rho, mean u) over liquid and old interface neighbours, m = the
// received shares.  From liquid: m = rho + shares, phi = m / rho, bubble =
// the lowest id among its gas neighbours after conversion.
template <int Q, class S>
__device__ __forceinline__ void apply_new(const DPtrs& d, const KParams& p, int parity, const LaneDir& l, int c,
                                          double (*scratch)[33]) {
  using R = typename S::Real;
  using T = typename S::T;
  T* __restrict__ B = (T*)d.pdf[parity ^ 1];
  const long long Np = p.Np;
  const uint8_t fl = d.flags[c];
  int t;
  const int n = lane_neighbour(d, p, l, c, fl, t);
  // one level of loads: what a neighbour of another kind holds is not used
  const R* mu = (const R*)d.mom_u;
  const bool was_gas = (fl & F_TYPE) == T_GAS;
  int cf = CV_NONE, bn = -1;
  uint8_t cl = 0;
  double sh = 0.0, rn = 0.0;
  R un[3] = {R(0.0), R(0.0), R(0.0)};
  if (n >= 0) {
    cf = d.cfin[n];
    cl = d.claim[n];
    sh = d.share[n];
    if (was_gas) {  // moments cached by the interface kernel
      rn = d.mom_rho[n];
      un[0] = mu[3LL * n + 0];
      un[1] = mu[3LL * n + 1];
      un[2] = mu[3LL * n + 2];
    } else {
      bn = d.bid[n];
    }
  }
  if (t != T_IFACE) cf = CV_NONE;
  const bool claimed = (t == T_GAS || t == T_LIQ) && cl != 0;
  const bool from = is_converted(cf);
  const double s = ordered_sum(__ballot_sync(0xffffffffu, from), sh, 0.0);
  const bool own = l.i < Q;  // lanes that hold a PDF
  if (was_gas) {
    // neighbours that stay or turn liquid, or stay interface; liquid ones
    // (none next to a gas cell while the interface layer is closed) form
    // their moments from the stored PDFs
    const bool use = (t == T_IFACE && cf != CV_TOG) || (t == T_LIQ && !claimed);
    if (use && t == T_LIQ) post_moments<Q, S>(B, Np, n, p, rn, un);
    const unsigned um = __ballot_sync(0xffffffffu, use);
    double rb = 1.0, ub0 = 0.0, ub1 = 0.0, ub2 = 0.0;
    if (um) {
      // the four sums in lanes 0-3 at once, each in direction order (one
      // FP64 addition and one division a step for all four: an FP64
      // instruction takes 16 clocks of the SM's unit whatever its lanes)
      scratch[0][l.i] = rn;
      scratch[1][l.i] = (double)un[0];
      scratch[2][l.i] = (double)un[1];
      scratch[3][l.i] = (double)un[2];
      __syncwarp();
      const double* mine = scratch[l.i & 3];
      double sum = 0.0;
      for (unsigned m = um; m; m &= m - 1u) sum = sum + mine[__ffs(m) - 1];
      sum = sum / (double)__popc(um);
      rb = __shfl_sync(0xffffffffu, sum, 0);
      ub0 = __shfl_sync(0xffffffffu, sum, 1);
      ub1 = __shfl_sync(0xffffffffu, sum, 2);
      ub2 = __shfl_sync(0xffffffffu, sum, 3);
      __syncwarp();  // scratch is rewritten by the warp's next cell
    }
    const R ux = R(ub0), uy = R(ub1), uz = R(ub2);
    const R w = lane_weight<Q, R>(l.dx * l.dx + l.dy * l.dy + l.dz * l.dz);
    const R cu = R(l.dx) * ux + R(l.dy) * uy + R(l.dz) * uz;
    const R usq = ux * ux + uy * uy + uz * uz;
    R f;
    if constexpr (S::kDev) {
      f = w * (R(rb - 1.0) + R(rb) * (R(3.0) * cu + R(4.5) * cu * cu - R(1.5) * usq));
    } else {
      R e = R(1.0) + R(3.0) * cu;
      e = e + R(4.5) * cu * cu;
      e = e - R(1.5) * usq;
      f = w * R(rb) * e;
    }
    if constexpr (S::kExactRest) {
      // the rest PDF takes up the rounding of the others (store_cell, with
      // the sum of the stored steps taken over the lanes)
      constexpr float kRange = 2147483648.0f / (float)(1LL << S::kShift);
      bool bad = l.moving && !(fabsf(f) < kRange);
      long long steps = 0;
      if (l.moving) {
        const T v = S::stored(f);
        B[(long long)l.i * Np + c] = v;
        steps = S::steps(v);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) steps += __shfl_xor_sync(0xffffffffu, steps, o);
      if (l.i == 0) {
        long long r = __double2ll_rn((rb - 1.0) * (double)(1LL << S::kShift)) - steps;
        if (r > 2147483647LL || r < -2147483647LL) {
          bad = true;
          r = r > 0 ? 2147483647LL : -2147483647LL;
        }
        rest_slice<Q, S>(B, Np)[c] = (int)r;
      }
      if (bad) d.err[0] = 1;
    } else if (own) {
      B[(long long)l.i * Np + c] = lane_store<S>(f, w);
    }
    if (fl & F_NEAR_WALL) {
      // reflected copies into the slots of the obstacle pull sources
      const uint32_t wm = d.wallmask[c];
      const R fo = __shfl_sync(0xffffffffu, f, l.i == 0 ? 0 : (l.i & 1) ? l.i + 1 : l.i - 1);
      if (l.moving && ((wm >> l.i) & 1u)) {
        long long slot;
        if (fl & F_WRAP) {
          int x, y, z;
          decode(p, c, x, y, z);
          slot = nbr(p, x, y, z, -l.dx, -l.dy, -l.dz);
        } else {
          slot = c - (l.dx * p.sx + l.dy * p.sy + l.dz * p.sz);
        }
        B[(long long)l.i * Np + slot] = lane_store<S>(fo, w);
      }
    }
    if (l.i == 0) {
      const double m = 0.0 + s;
      d.mass[c] = m;
      set_phi(d, c, m / rb);
    }
  } else {  // from liquid
    const bool gas_after = (t == T_GAS && !claimed) || (t == T_IFACE && cf == CV_TOG);
    const int bb = gas_after ? bn : -1;
    // rho of the stored post-collision PDFs, as post_moments forms it
    if constexpr (S::kExactRest) {
      long long k = 0;
      if (l.i == 0) k = rest_slice<Q, S>(B, Np)[c];
      else if (own) k = S::steps(B[(long long)l.i * Np + c]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
      rn = 1.0 + (double)k * (1.0 / (double)(1LL << S::kShift));
    } else {
      double v = 0.0;
      if (own) {
        const T raw = B[(long long)l.i * Np + c];
        if constexpr (S::kDev) v = (double)S::loadd(raw);
        else v = raw;
      }
      double sum = 0.0;
#pragma unroll
      for (int i = 0; i < Q; ++i) sum = sum + __shfl_sync(0xffffffffu, v, i);
      rn = S::kDev ? 1.0 + sum : sum;
    }
    const unsigned best = __reduce_min_sync(0xffffffffu, bb >= 0 ? (unsigned)bb : 0xffffffffu);
    if (l.i == 0) {
      const double m = rn + s;
      d.mass[c] = m;
      set_phi(d, c, m / rn);
      d.bid[c] = best == 0xffffffffu ? -1 : (int)best;
    }
  }
}

// ------------------------------------------------------------ one domain

// The listed cells first (their chains are the longest), then the commit.
template <int Q>
__global__ void __launch_bounds__(kBlock) k_resolve(DPtrs d, KParams p, int parity) {
  stage_begin();
  const LaneDir l = lane_dir<Q>();
  const int nconv = *conv_count(d);
  for (int j = spread_warp(); j < nconv; j += spread_warps()) resolve_listed<Q>(d, p, parity, l, j);
  const int n = d.counts[parity];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
    commit_cell(d, parity, k);
}

template <int Q, class S>
__global__ void __launch_bounds__(kBlock) k_count(DPtrs d, KParams p, int parity) {
  stage_begin();
  const LaneDir l = lane_dir<Q>();
  const int nconv = *conv_count(d);
  for (int j = spread_warp(); j < nconv; j += spread_warps()) count_listed<Q, S>(d, p, parity, l, j);
}

// New cells [first, ...) and receivers of one domain by the warps first,
// first + stride, ... of a share of the grid.
template <int Q, class S>
__device__ __forceinline__ void apply_new_items(const DPtrs& d, const KParams& p, int parity, const LaneDir& l,
                                                int first, int stride) {
  __shared__ double scratch[kBlock / 32][4][33];  // a warp's moments
  const int nnew = d.counts[2];
  for (int j = first; j < nnew; j += stride)
    apply_new<Q, S>(d, p, parity, l, d.newlist[j], scratch[threadIdx.x >> 5]);
}
template <int Q, class S>
__device__ __forceinline__ void apply_old_items(const DPtrs& d, const KParams& p, int parity, const LaneDir& l,
                                                int first, int stride) {
  const int nrec = *recv_count(d);
  for (int j = first; j < nrec; j += stride) apply_receiver<Q, S>(d, p, l, recv_list(d)[j]);
  const int nconv = *conv_count(d);
  for (int j = first * 32 + l.i; j < nconv; j += stride * 32) apply_converted<S>(d, conv_list(d, parity)[j]);
}

// The kinds of cells are disjoint and read only what earlier kernels wrote
// (kNew, kOld: which parts a launch does).  In one launch the new cells (the
// longest chains) are dealt from the first warp, the others from the last.  As
// two kernels side by side in the graph, the fork and the join cost more than
// the overlap gave once the stage ran on lists (192^3 drop, a step with the
// bubbles' fork gone as well: 91.9 us forked, 89.2 in one launch).
template <int Q, class S, bool kNew, bool kOld>
__global__ void __launch_bounds__(kBlock) k_apply(DPtrs d, KParams p, int parity) {
  stage_begin();
  const LaneDir l = lane_dir<Q>();
  const int w = spread_warp(), nw = spread_warps();
  if constexpr (kNew) apply_new_items<Q, S>(d, p, parity, l, w, nw);
  if constexpr (kOld) apply_old_items<Q, S>(d, p, parity, l, nw - 1 - w, nw);
}

// --------------------------------------------------------------- batches
// The lists of n domains: the warps of the grid are dealt round-robin over
// the domains, so no prefix over the lists is needed.  f(k, first, stride):
// domain k's items first, first + stride, ... are this warp's.
template <class F>
__device__ __forceinline__ void deal_domains(int n, F f) {
  const int w = spread_warp(), nw = spread_warps();
  if (nw >= n) {
    const int k = w % n;
    f(k, w / n, (nw - k + n - 1) / n);
  } else {
    for (int k = w; k < n; k += nw) f(k, 0, 1);
  }
}

template <int Q>
__global__ void __launch_bounds__(kBlock) kb_resolve(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  const LaneDir l = lane_dir<Q>();
  deal_domains(pl.n, [&](int k, int first, int stride) {
    const DomRec& r = recs[k];
    const int nconv = *conv_count(r.d);
    for (int j = first; j < nconv; j += stride) resolve_listed<Q>(r.d, r.p, r.parity, l, j);
  });
  const int total = pl.band[pl.n];
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
    const int k = find_domain(pl.band, pl.n, g);
    const DomRec& r = recs[k];
    const int i = g - pl.band[k];
    if (i < r.d.counts[r.parity]) commit_cell(r.d, r.parity, i);
  }
}

template <int Q, class S>
__global__ void __launch_bounds__(kBlock) kb_count(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  const LaneDir l = lane_dir<Q>();
  deal_domains(pl.n, [&](int k, int first, int stride) {
    const DomRec& r = recs[k];
    const int nconv = *conv_count(r.d);
    for (int j = first; j < nconv; j += stride) count_listed<Q, S>(r.d, r.p, r.parity, l, j);
  });
}

// The apply stage of a batch (kNew, kOld as in k_apply).
template <int Q, class S, bool kNew, bool kOld>
__global__ void __launch_bounds__(kBlock) kb_apply(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  const LaneDir l = lane_dir<Q>();
  deal_domains(pl.n, [&](int k, int first, int stride) {
    const DomRec& r = recs[k];
    if constexpr (kNew) apply_new_items<Q, S>(r.d, r.p, r.parity, l, first, stride);
    if constexpr (kOld) apply_old_items<Q, S>(r.d, r.p, r.parity, l, stride - 1 - first, stride);
  });
}

}  // namespace fslbm
