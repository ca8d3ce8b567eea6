// FSLBM step kernels (arXiv 2207.13962, Sec. 2-3), templated on the lattice
// (Q = 19 / 27) and the PDF storage format S (FP64, FP32, FP16/BF16 shifted).
//
// One step, in stream order:
//   k_geometry   band   K8 smoothing, Parker-Youngs normal, FDM curvature,
//                       gas density rho^G, Thuerey class
//   k_bulk       grid   pull stream + bounce-back + collide of liquid cells
//   k_interface  band   pull, free-surface BC of the chosen variant, mass
//                       exchange, fill update, collide, conversion marks
//   k_resolve    list+band  conflict rule, claims of gas/liquid neighbours;
//                       commit of m and phi
//   k_count      list   excess-mass receivers, deferral, shares
//   k_apply      lists  excess gather, new interface cells' PDFs
//   k_finalize   band+new  final flags, tile and segment marks, bubble sums
//   k_compact_band grid the next interface list; in one more block the bubble
//                       volume pressures
// The interface work runs only on the compacted list of interface cells
// ("band") and on the cells that conversion turns into interface cells.
// Conversion and excess redistribution are gather-only: each cell computes
// its own new values from its neighbours, so the flag field is deterministic.
//
// In the FP64 instantiation the kernels are compiled without FMA contraction
// and every expression keeps the association and summation order of the
// plain CPU oracle, so results agree to the last bit.
#pragma once

#include "fslbm_bulk.cuh"
#include "fslbm_convert.cuh"
#include "fslbm_interface_lanes.cuh"
#include <type_traits>

namespace fslbm {

// ------------------------------------------------------------------ init
// Validates raw flags: values <= 3 and no liquid cell next to a gas cell.
template <int Q>
__global__ void k_init_check(const uint8_t* __restrict__ raw, KParams p, int* bad) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  uint8_t t = raw[c];
  if (t > 3) {
    atomicOr(bad, 1);
    return;
  }
  if (t != T_LIQ) return;
  int x, y, z;
  decode(p, c, x, y, z);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    int n = nbr(p, x, y, z, CX(i), CY(i), CZ(i));
    if (n >= 0 && raw[n] == T_GAS) atomicOr(bad, 2);
  }
}

// Initial fields: phi, m = phi rho (Eq. nm-fslbm-mass), f = f^eq(rho, u).
template <int Q, class S>
__global__ void k_init_cells(const uint8_t* __restrict__ raw, const double* __restrict__ fill,
                             const double* __restrict__ vel, const double* __restrict__ den,
                             DPtrs d, KParams p, int parity) {
  using R = typename S::Real;
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  const uint8_t t = raw[c];
  int x, y, z;
  decode(p, c, x, y, z);
  uint8_t fl = t;
  uint32_t wm = 0u;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    int n = nbr(p, x, y, z, CX(i), CY(i), CZ(i));
    if (n < 0) fl |= F_FACE;
    else if (raw[n] == T_OBST) fl |= F_NEAR_WALL;
    const int X = x + CX(i), Y = y + CY(i), Z = z + CZ(i);
    if (n >= 0 && (X < 0 || X >= p.nx || Y < 0 || Y >= p.ny || Z < 0 || Z >= p.nz)) fl |= F_WRAP;
    const int s = nbr(p, x, y, z, -CX(i), -CY(i), -CZ(i));
    if (s >= 0 && raw[s] == T_OBST) wm |= 1u << i;
  }
  d.flags[c] = fl;
  d.wallmask[c] = wm;
  const double r = den ? den[c] : 1.0;
  set_phi(d, c, (t == T_LIQ) ? 1.0 : (t == T_IFACE) ? fill[c] : 0.0);
  d.mass[c] = (t == T_LIQ) ? r : (t == T_IFACE) ? fill[c] * r : 0.0;
  d.cls[c] = t;
  d.mark[c] = 0;
  d.conv[c] = 0;
  d.cfin[c] = 0;
  d.claim[c] = 0;
  d.share[c] = 0.0;
  typename S::T* P = (typename S::T*)d.pdf[parity];
  typename S::T* P2 = (typename S::T*)d.pdf[parity ^ 1];
  const bool fluid = (t == T_LIQ || t == T_IFACE);
  if (!fluid) return;  // gas and obstacle slots stay as cleared (obstacle
                       // slots receive their neighbours' reflected copies)
  R fe[Q];
  if constexpr (S::kDev) {
    // deviation f^eq - w in FP32 from drho = rho - 1 taken in FP64 (every
    // term is then of the size of a deviation)
    const R ux = vel ? R(vel[c]) : R(0.0);
    const R uy = vel ? R(vel[(long long)p.N + c]) : R(0.0);
    const R uz = vel ? R(vel[2LL * p.N + c]) : R(0.0);
#pragma unroll
    for (int i = 0; i < Q; ++i) fe[i] = feq_dev<Q, R>(i, R(r - 1.0), R(r), ux, uy, uz);
  } else {
    const R ux = vel ? R(vel[c]) : R(0.0);
    const R uy = vel ? R(vel[(long long)p.N + c]) : R(0.0);
    const R uz = vel ? R(vel[2LL * p.N + c]) : R(0.0);
#pragma unroll
    for (int i = 0; i < Q; ++i) fe[i] = feq_i<Q, R>(i, R(r), ux, uy, uz);
  }
  // the mass-conserving formats store the density deviation r - 1 (to
  // their grid): the rest PDF takes up the rounding of the others
  bool over = false;
  const long long s_in = S::kExactRest ? __double2ll_rn((r - 1.0) * (double)(1LL << grid_shift<S>())) : 0;
  store_cell<Q, S>(P, p.Np, c, fe, s_in, over);
  store_cell<Q, S>(P2, p.Np, c, fe, s_in, over);
  if (wm) {
    write_reflected<Q, S>(d, p, P, c, wm, (fl & F_WRAP) != 0, fe);
    write_reflected<Q, S>(d, p, P2, c, wm, (fl & F_WRAP) != 0, fe);
  }
}

// Ordered-by-warp compaction of all interface cells into a list.
static __global__ void k_compact_full(const uint8_t* __restrict__ flags, int N, int* list,
                               int* count) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  bool pred = (c < N) && ((flags[c] & F_TYPE) == T_IFACE);
  int pos = warp_append(count, pred);
  if (pred) list[pos] = c;
}

// -------------------------------------------------------- bubble labels
// Connected gas regions (lattice neighbourhood, periodic wrap) at init, on
// the device.  Union-find with lock-free hooking: every gas cell starts as
// its own root; a union hooks the root with the larger caller index
// x + nx (y + ny z) under the other with compare-and-swap (a root is
// re-parented only while it is still a root), so every root ends as the
// cell of its component with the lowest caller index, whatever the storage
// order.  Bubbles are then numbered in the order of their roots' caller
// indices, i.e. of their lowest cell index.
__device__ __forceinline__ int cc_find(const int* lab, int x) {
  int p = lab[x];
  while (p != x) {
    x = p;
    p = lab[x];
  }
  return x;
}

static __global__ void k_cc_init(const uint8_t* __restrict__ raw, int N, int* lab) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < N) lab[c] = raw[c] == T_GAS ? c : -1;
}

template <int Q>
__global__ void k_cc_union(const uint8_t* __restrict__ raw, KParams p, int* lab) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N || raw[c] != T_GAS) return;
  int x, y, z;
  decode(p, c, x, y, z);
  for (int i = 1; i < Q; ++i) {
    const int n = nbr(p, x, y, z, CX(i), CY(i), CZ(i));
    if (n < 0 || n >= c || raw[n] != T_GAS) continue;  // each pair once (storage order)
    int a = cc_find(lab, c), b = cc_find(lab, n);
    while (a != b) {
      if (ext_index(p, a) > ext_index(p, b)) {
        const int t = a;
        a = b;
        b = t;
      }
      const int old = atomicCAS(&lab[b], b, a);  // hook root b under a
      if (old == b) break;
      b = cc_find(lab, old);
      a = cc_find(lab, a);
    }
  }
}

static __global__ void k_cc_compress(int N, int* lab) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < N && lab[c] >= 0) lab[c] = cc_find(lab, c);
}

// Storage index of the cell with caller index e.
__device__ __forceinline__ int storage_of_ext(const KParams& p, int e) {
  const int x = e % p.nx, t = e / p.nx;
  return cidx(p, x, t % p.ny, t / p.ny);
}

// Roots per block of kCcChunk cells, counted in the caller's cell order
// (pass 1 of the numbering).
constexpr int kCcChunk = 1024;
static __global__ void k_cc_count(KParams p, const int* __restrict__ lab, int* block_roots) {
  __shared__ int cnt;
  const int N = p.N;
  if (threadIdx.x == 0) cnt = 0;
  __syncthreads();
  int mine = 0;
  for (int k = threadIdx.x; k < kCcChunk; k += blockDim.x) {
    const long long e = (long long)blockIdx.x * kCcChunk + k;
    if (e < N) {
      const int c = storage_of_ext(p, (int)e);
      if (lab[c] == c) ++mine;
    }
  }
  atomicAdd(&cnt, mine);
  __syncthreads();
  if (threadIdx.x == 0) block_roots[blockIdx.x] = cnt;
}

// Exclusive scan of the per-block root counts (one block); total in off[n].
static __global__ void k_cc_scan(int nblocks, const int* __restrict__ block_roots, int* off) {
  block_prefix(nblocks, off, [&](int k) { return block_roots[k]; });
}

// Bubble id of every root in the caller's index order (pass 2): warps walk
// their block's chunk in order, so ranks within the chunk follow the index.
static __global__ void k_cc_number(KParams p, const int* __restrict__ lab, const int* __restrict__ off,
                                   int* root_id) {
  __shared__ int base;
  const int N = p.N;
  if (threadIdx.x == 0) base = off[blockIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  // one warp numbers the chunk sequentially in 32-cell steps
  if (threadIdx.x < 32) {
    int b = base;
    for (int k = 0; k < kCcChunk; k += 32) {
      const long long e = (long long)blockIdx.x * kCcChunk + k + lane;
      const int c = e < N ? storage_of_ext(p, (int)e) : -1;
      const bool root = c >= 0 && lab[c] == c;
      const unsigned m = __ballot_sync(0xffffffffu, root);
      if (root) root_id[c] = b + __popc(m & ((1u << lane) - 1u));
      b += __popc(m);
    }
  }
}

// Bubble id of gas cells (their root's number) and of interface cells (the
// lowest id among their gas neighbours); -1 elsewhere.
template <int Q>
__global__ void k_cc_assign(const uint8_t* __restrict__ raw, KParams p, const int* __restrict__ lab,
                            const int* __restrict__ root_id, int* bid) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  const uint8_t t = raw[c];
  if (t == T_GAS) {
    bid[c] = root_id[lab[c]];
    return;
  }
  int best = -1;
  if (t == T_IFACE) {
    int x, y, z;
    decode(p, c, x, y, z);
    for (int i = 1; i < Q; ++i) {
      const int n = nbr(p, x, y, z, CX(i), CY(i), CZ(i));
      if (n < 0 || raw[n] != T_GAS) continue;
      const int b = root_id[lab[n]];
      if (best < 0 || b < best) best = b;
    }
  }
  bid[c] = best;
}

// Initial bubble volumes in 2^-32 fixed point: gas cells count 1, interface
// cells 1 - phi (the same terms as the step's volume sums).
static __global__ void k_cc_volumes(const uint8_t* __restrict__ raw, const double* __restrict__ fill,
                                    int N, const int* __restrict__ bid, long long* gas_cnt,
                                    long long* iface_fix) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int b = -1;
  long long g = 0, v = 0;
  if (c < N) {
    b = bid[c];
    if (b >= 0 && raw[c] == T_GAS) g = 1;
    if (b >= 0 && raw[c] == T_IFACE) v = __double2ll_rn((1.0 - fill[c]) * 4294967296.0);
  }
  unsigned remaining = __ballot_sync(0xffffffffu, b >= 0);
  while (remaining) {
    const int leader = __ffs(remaining) - 1;
    const int bb = __shfl_sync(0xffffffffu, b, leader);
    const bool mine = b == bb;
    long long sg = mine ? g : 0, sv = mine ? v : 0;
    for (int o = 16; o > 0; o >>= 1) {
      sg += __shfl_xor_sync(0xffffffffu, sg, o);
      sv += __shfl_xor_sync(0xffffffffu, sv, o);
    }
    if (lane == leader) {
      if (sg) atomicAdd((unsigned long long*)&gas_cnt[bb], (unsigned long long)sg);
      if (sv) atomicAdd((unsigned long long*)&iface_fix[bb], (unsigned long long)sv);
    }
    remaining &= ~__ballot_sync(0xffffffffu, mine);
  }
}

static __global__ void k_cc_v0(int nb, const long long* gas_cnt, long long* iface_fix, double* V0,
                               double* Vcur, double* pV, double pv0) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  const long long acc = gas_cnt[b] * 4294967296LL + iface_fix[b];
  const double V = __ll2double_rn(acc) / 4294967296.0;
  V0[b] = V;
  Vcur[b] = V;
  pV[b] = pv0;
  iface_fix[b] = 0;
}

// ------------------------------------------------- bubble relabelling
// Coalescence and segmentation of bubbles between steps: the bubbles are
// labelled again from the current flags (the kernels above), and the gas of
// each old bubble goes to the new ones in proportion to the fixed-point
// volume of its cells that each holds (the host combines the overlaps).

// Cell types of the flags (the labelling kernels take bare types).
static __global__ void k_types(const uint8_t* __restrict__ flags, int N, uint8_t* raw) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < N) raw[c] = flags[c] & F_TYPE;
}

// Overlap of old and new bubbles in 2^-32 fixed point: M[A * W + C + 1]
// for a cell of old id A and new id C (column 0: no new bubble), fr[C] for
// the cells of new bubble C that carried no id.  Integer sums, one atomic
// per (old, new) pair present in a warp.
static __global__ void k_bubble_overlap(const uint8_t* __restrict__ raw, const double* __restrict__ phi,
                                        const int* __restrict__ old_bid, const int* __restrict__ bid, int N,
                                        int W, long long* M, long long* fr) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  long long key = -1, v = 0;
  if (c < N) {
    const uint8_t t = raw[c];
    if (t == T_GAS) v = 4294967296LL;
    else if (t == T_IFACE) v = __double2ll_rn((1.0 - phi[c]) * 4294967296.0);
    if (t == T_GAS || t == T_IFACE) {
      const int A = old_bid[c], C = bid[c];
      if (A >= 0) key = (long long)A * W + (C + 1);
      else if (C >= 0) key = -2 - (long long)C;  // fr[C]
    }
  }
  unsigned remaining = __ballot_sync(0xffffffffu, key != -1);
  while (remaining) {
    const int leader = __ffs(remaining) - 1;
    const long long kk = __shfl_sync(0xffffffffu, key, leader);
    const bool mine = key == kk;
    long long sv = mine ? v : 0;
    for (int o = 16; o > 0; o >>= 1) sv += __shfl_xor_sync(0xffffffffu, sv, o);
    if (lane == leader && sv) {
      long long* dst = kk >= 0 ? &M[kk] : &fr[-2 - kk];
      atomicAdd((unsigned long long*)dst, (unsigned long long)sv);
    }
    remaining &= ~__ballot_sync(0xffffffffu, mine);
  }
}

// Volumes and pressures of the new bubbles (p^V = p^V(0) V0 / V, as in the
// step's bubble update), with their gas reference V0 already set.
static __global__ void k_relabel_pressure(int nb, const long long* gas_cnt, long long* iface_fix,
                                          const double* V0, double* Vcur, double* pV, double pv0) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  const long long acc = gas_cnt[b] * 4294967296LL + iface_fix[b];
  const double V = __ll2double_rn(acc) / 4294967296.0;
  pV[b] = (V > 0.0) ? (pv0 * V0[b]) / V : pv0;
  Vcur[b] = V;
  iface_fix[b] = 0;
}

// ------------------------------------------------------------- geometry
// K8 weights (1 - r^2/4)^4 on the 3x3x3 block: r^2 = 0, 1, 2, 3.
template <class R>
__device__ __forceinline__ R k8w(int n2) {
  return n2 == 0 ? R(1.0) : n2 == 1 ? R(0.31640625) : n2 == 2 ? R(0.0625) : R(0.00390625);
}

// Geometry on 8^3 tiles that hold interface cells (tile list built by
// k_finalize).  The tile's fill levels with a halo of 3 sit in shared memory;
// phi~ (K8 smoothing, radius 2) lies on the 12^3 sub-box, n^ (Parker-Youngs,
// Eq. nm-fslbm-normal) on the 10^3 sub-box and kappa = -div(n^) on the
// interface cells of the tile.  Obstacle and out-of-domain stencil points
// take the stencil centre's value.  In the FP64 engine each value uses the
// same arithmetic and summation order as a per-cell evaluation.
//
// An interface is a sheet: kappa needs n^ at the interface cells and their
// face neighbours only, and these need phi~ on the 3^3 blocks around them,
// together about a third of the sub-boxes.  The points needed are marked as
// the box is loaded, compacted into two lists in shared memory and evaluated
// a thread a point, so the work follows the interface and fills the warps.
// Marching all z-columns of the sub-boxes instead (144 and 100 threads, 12
// and 10 steps) measured 99 us for the six tiles of the 32x64x1 wave in FP64,
// where the FP64 pipe of one SM (two lanes a clock) bounds a tile.
constexpr int GT = 8;                    // tile edge
constexpr int GE = GT + 6;               // box edge with halo 3
constexpr int GB = GE * GE * GE;         // 2744 box positions
constexpr int GS = GT + 4;               // phi~ sub-box edge (12)
constexpr int GN = GT + 2;               // n^ sub-box edge (10)
constexpr int kGeoBlock = 256;
// geometry blocks per interface-band block: each tile's block runs four
// dependent shared-memory phases, so many resident tiles hide the latency
#ifndef FSLBM_GEO_MULT
#define FSLBM_GEO_MULT 3
#endif
constexpr int kGeoGridMult = FSLBM_GEO_MULT;
#ifndef FSLBM_GEO_MINB
#define FSLBM_GEO_MINB 3
#endif
constexpr int kGeoMinBlocks = FSLBM_GEO_MINB;  // resident geometry blocks per SM compiled for

// Fill level stored for obstacle and out-of-domain box positions: stencils
// substitute their centre's value there (no fill level comes near it).
template <class R>
__device__ __forceinline__ R kObstacle() { return R(-1.0e30); }
template <class R>
__device__ __forceinline__ bool is_obstacle(R v) { return v < R(-1.0e29); }

// Shared memory of one tile: the fill-level box, whose space the normals
// take over once the smoothing has read it; the smoothed sub-box, whose space
// holds the marks of the needed points until the lists are made; the types;
// the lists.
constexpr int GN3 = GN * GN * GN, GS3 = GS * GS * GS;
constexpr int kGeoBoxSlots = GB > 3 * GN3 ? GB : 3 * GN3;
template <class R>
constexpr size_t geometry_smem() {
  return sizeof(R) * (kGeoBoxSlots + GS3) + GB + sizeof(unsigned short) * (GN3 + GS3);
}
static_assert(GN3 + GS3 <= 4 * GS3 && GN3 % 4 == 0 && GS3 % 4 == 0 && GB % 8 == 0, "layout of the tile's buffers");

// a / 3.6796875 (= 471 / 128, the sum of the K8 weights), correctly rounded:
// fma(a, zh, a zl) with zh + zl = 128 / 471 to twice the precision (Brisebarre,
// Muller and Raina, "Accelerating correctly rounded floating-point division
// when the divisor is known in advance", IEEE Trans. Computers 53, 2004).  A
// quotient by 471 of a binary number lies at least 1/942 of an ulp from any
// midpoint of two neighbouring numbers, and the sum before its rounding is
// within 2^-51 ulp of the quotient, so the rounding is that of the division.
__device__ __forceinline__ double div_k8(double a) {
  return fma(a, 0x1.1648d50fc3201p-2, a * 0x1.648d50fc32011p-58);
}

// Appends the positions s = t, t + NT, ... < n of thread t that have bit r of
// take set (r-th position) to a list in shared memory, one atomic a warp;
// every lane calls it.
template <int N, int NT>
__device__ __forceinline__ void push_shared(unsigned short* list, int* count, unsigned take) {
  constexpr int kPer = (N + NT - 1) / NT;
  const unsigned lane = threadIdx.x & 31u;
  unsigned m[kPer];
  int total = 0;
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    m[r] = __ballot_sync(0xffffffffu, (take >> r) & 1u);
    total += __popc(m[r]);
  }
  if (total == 0) return;
  int base = 0;
  if (lane == 0) base = atomicAdd(count, total);
  base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    if ((take >> r) & 1u)
      list[base + __popc(m[r] & ((1u << lane) - 1u))] = (unsigned short)(threadIdx.x + r * NT);
    base += __popc(m[r]);
  }
}

// phi~ at box position b (not an obstacle).  The FP32 engines group the 27
// points by z-plane: the K8 weights depend on r^2 only, so a plane gives its
// centre, the sum of its 4 in-plane face neighbours and of its 4 corners; an
// obstacle point takes the value of the stencil's centre, so a plane keeps the
// sum over its other points and, beside it, the count of its obstacle points,
// which multiplies the centre value at the end.  The FP64 engine sums in the
// oracle's order; the weights 2^-4 and 2^-8 make exact products, so a fused
// operation rounds as the product and the sum do.
template <class R, bool kSolid>
__device__ __forceinline__ R smoothed_at(const R* sphi, int b) {
  const R* q = sphi + b;
  const R pc = q[0];
  if constexpr (sizeof(R) == 4) {
    auto nz = [&](R v) { return (kSolid && is_obstacle(v)) ? R(0.0) : v; };
    auto ob = [&](R v) { return (kSolid && is_obstacle(v)) ? R(1.0) : R(0.0); };
    R c0[3], f4[3], c4[3], nf[3], nc[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const R* w = q + (k - 1) * GE * GE;
      c0[k] = w[0];
      const R a = w[-1], e = w[1], c = w[-GE], g = w[GE];
      const R u = w[-GE - 1], v = w[-GE + 1], x = w[GE - 1], y = w[GE + 1];
      f4[k] = (nz(a) + nz(e)) + (nz(c) + nz(g));
      c4[k] = (nz(u) + nz(v)) + (nz(x) + nz(y));
      if constexpr (kSolid) {
        nf[k] = (ob(a) + ob(e)) + (ob(c) + ob(g));
        nc[k] = (ob(u) + ob(v)) + (ob(x) + ob(y));
      }
    }
    const R zm = (kSolid && is_obstacle(c0[0])) ? pc : c0[0], zp = (kSolid && is_obstacle(c0[2])) ? pc : c0[2];
    R s1 = (f4[1] + zm) + zp, s2 = (c4[1] + f4[0]) + f4[2], s3 = c4[0] + c4[2];
    if constexpr (kSolid) {
      s1 = s1 + nf[1] * pc;
      s2 = s2 + (nc[1] + nf[0] + nf[2]) * pc;
      s3 = s3 + (nc[0] + nc[2]) * pc;
    }
    return (pc + k8w<R>(1) * s1 + k8w<R>(2) * s2 + k8w<R>(3) * s3) * (R(1.0) / R(3.6796875));
  } else {
    R acc = R(0.0);
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
          const int n2 = dx * dx + dy * dy + dz * dz;
          const R raw = q[dx + GE * (dy + GE * dz)];
          const R v = (kSolid && is_obstacle(raw)) ? pc : raw;
          if (n2 == 0) acc = acc + v;
          else if (n2 == 1) acc = acc + k8w<R>(1) * v;
          else acc = fma(k8w<R>(n2), v, acc);
        }
    return div_k8(acc);
  }
}

// n^ at position s of the smoothed sub-box (not an obstacle).  FP32: the
// Parker-Youngs weights (2-|d|)(2-|d'|) factor into [1 2 1] x [1 2 1] x
// [-1 0 1], formed per z-plane with the (weighted) obstacle counts beside them
// as above.  FP64: the oracle's order; the weights 1, 2 and 4 make exact
// products.
template <class R, bool kSolid>
__device__ __forceinline__ void normal_at(const R* sps, int s, R n[3]) {
  const R* q = sps + s;
  const R pc = q[0];
  if constexpr (sizeof(R) == 4) {
    auto nz = [&](R v) { return (kSolid && is_obstacle(v)) ? R(0.0) : v; };
    auto ob = [&](R v) { return (kSolid && is_obstacle(v)) ? R(1.0) : R(0.0); };
    R gx[3], gy[3], sm[3], gxo[3], gyo[3], so[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const R* w = q + (k - 1) * GS * GS;
      const R a00 = w[-GS - 1], a01 = w[-GS], a02 = w[-GS + 1];
      const R a10 = w[-1], a11 = w[0], a12 = w[1];
      const R a20 = w[GS - 1], a21 = w[GS], a22 = w[GS + 1];
      gx[k] = (nz(a02) - nz(a00)) + R(2.0) * (nz(a12) - nz(a10)) + (nz(a22) - nz(a20));
      gy[k] = (nz(a20) - nz(a00)) + R(2.0) * (nz(a21) - nz(a01)) + (nz(a22) - nz(a02));
      sm[k] = (nz(a00) + R(2.0) * nz(a01) + nz(a02)) + R(2.0) * (nz(a10) + R(2.0) * nz(a11) + nz(a12)) +
              (nz(a20) + R(2.0) * nz(a21) + nz(a22));
      if constexpr (kSolid) {
        gxo[k] = (ob(a02) - ob(a00)) + R(2.0) * (ob(a12) - ob(a10)) + (ob(a22) - ob(a20));
        gyo[k] = (ob(a20) - ob(a00)) + R(2.0) * (ob(a21) - ob(a01)) + (ob(a22) - ob(a02));
        so[k] = (ob(a00) + R(2.0) * ob(a01) + ob(a02)) + R(2.0) * (ob(a10) + R(2.0) * ob(a11) + ob(a12)) +
                (ob(a20) + R(2.0) * ob(a21) + ob(a22));
      }
    }
    R n0 = gx[0] + R(2.0) * gx[1] + gx[2];
    R n1 = gy[0] + R(2.0) * gy[1] + gy[2];
    R n2 = sm[2] - sm[0];
    if constexpr (kSolid) {
      n0 = n0 + (gxo[0] + R(2.0) * gxo[1] + gxo[2]) * pc;
      n1 = n1 + (gyo[0] + R(2.0) * gyo[1] + gyo[2]) * pc;
      n2 = n2 + (so[2] - so[0]) * pc;
    }
    const R l2 = n0 * n0 + n1 * n1 + n2 * n2;
    const R il = l2 > R(0.0) ? rsqrtf(l2) : R(0.0);
    n[0] = n0 * il;
    n[1] = n1 * il;
    n[2] = n2 * il;
  } else {
    auto at = [&](int dx, int dy, int dz) { return q[dx + GS * (dy + GS * dz)]; };
    R nn[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      R acc = R(0.0);
#pragma unroll
      for (int pp = -1; pp <= 1; ++pp)
#pragma unroll
        for (int r = -1; r <= 1; ++r) {
          const int ax = (a == 0) ? 1 : r, ay = (a == 0) ? r : (a == 1) ? 1 : pp, az = (a == 2) ? 1 : pp;
          const int bx = (a == 0) ? -1 : ax, by = (a == 1) ? -1 : ay, bz = (a == 2) ? -1 : az;
          const R rp = at(ax, ay, az), rm = at(bx, by, bz);
          const R vp = (kSolid && is_obstacle(rp)) ? pc : rp;
          const R vm = (kSolid && is_obstacle(rm)) ? pc : rm;
          const R wt = (pp == 0 && r == 0) ? R(4.0) : (pp == 0 || r == 0) ? R(2.0) : R(1.0);
          acc = fma(wt, vp - vm, acc);
        }
      nn[a] = acc;
    }
    const R len = sqrt(nn[0] * nn[0] + nn[1] * nn[1] + nn[2] * nn[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) n[a] = (len > R(0.0)) ? nn[a] / len : R(0.0);
  }
}

// One 8^3 tile of the geometry pass (all NT threads of the block call it).
template <int Q, class S, int NT = kGeoBlock>
__device__ __forceinline__ void geometry_tile(const DPtrs& d, const KParams& p, int tile,
                                              unsigned char* g_smem) {
  using R = typename S::Real;
  __shared__ int s_count[2];      // points in the lists
  __shared__ int s_off[3][16];    // offsets of the box coordinates
  R* sphi = (R*)g_smem;
  R* snh = sphi;  // written after the smoothing's last read of sphi
  R* sps = sphi + kGeoBoxSlots;
  uint8_t* need_n = (uint8_t*)sps;  // marks, until the lists are made
  uint8_t* need_s = need_n + GN3;
  uint8_t* styp = (uint8_t*)(sps + GS3);
  unsigned short* list_n = (unsigned short*)(styp + GB);
  unsigned short* list_s = list_n + GN3;
  const int ntx = (p.nx + GT - 1) / GT, nty = (p.ny + GT - 1) / GT;
  R* nhat = (R*)d.nhat;
  R* rhog = (R*)d.rhog;

  const int tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
  const int ox = tx * GT - 3, oy = ty * GT - 3, oz = tz * GT - 3;
  __syncthreads();  // the previous tile is done with the buffers
  for (int w = threadIdx.x; w < (GN3 + GS3) / 4; w += NT) ((unsigned*)need_n)[w] = 0u;
  if (threadIdx.x < 2) s_count[threadIdx.x] = 0;
  if (threadIdx.x < 48) {
    // offset of box position k along storage axis a, -1 outside the domain
    // (and outside the box)
    const int a = threadIdx.x >> 4, k = threadIdx.x & 15, x = p.ax[a];
    const int X = wrapc(sel3(x, ox, oy, oz) + k, sel3(x, p.nx, p.ny, p.nz), sel3(x, p.per[0], p.per[1], p.per[2]));
    s_off[a][k] = X < 0 || k >= GE ? -1 : X * sel3(x, p.sx, p.sy, p.sz);
  }
  __syncthreads();
  // The box in the cells' storage order: 16 lanes take the 14 positions of a
  // row along the contiguous axis (the loads of a warp coalesce whatever the
  // storage order), the threads' rows advance by NT / 16.  The offsets of the
  // coordinates along each axis come from a table.  All of a thread's global
  // reads are issued before the first result is used, without a branch around
  // them (positions outside read cell 0): a branch a position made the thread
  // wait for every load in turn, 6 to 7 us a tile.  The shared-memory box
  // itself is indexed in the caller's axes.
  constexpr int kRowStep = NT / 16;
  constexpr int kRows = (GE * GE + kRowStep - 1) / kRowStep;  // rows per thread
  static_assert(NT % 16 == 0 && kRowStep >= GE && kRowStep < 2 * GE, "row walk");
  const int o[3] = {ox, oy, oz}, size[3] = {p.nx, p.ny, p.nz};
  const int k0 = threadIdx.x & 15;
  // steps of the storage axes in the shared-memory box (caller's axes)
  int bstep[3], core[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int x = p.ax[a];
    bstep[a] = x == 0 ? 1 : x == 1 ? GE : GE * GE;
    const int left = sel3(x, size[0] - o[0], size[1] - o[1], size[2] - o[2]) - 3;
    core[a] = left < GT ? left : GT;  // the tile's cells inside the domain
  }
  bool solid_here = false;  // an obstacle or a position outside the domain
  {
    uint8_t tv[kRows];
    R pv[kRows];
    unsigned inside = 0u;  // bit r: position r lies in the domain
    int k1 = threadIdx.x >> 4, k2 = 0;
    if (k1 >= GE) k1 -= GE, k2 = 1;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int e0 = s_off[0][k0], e1 = s_off[1][k1], e2 = s_off[2][k2];
      const bool in = (e0 | e1 | e2) >= 0;
      inside |= (unsigned)in << r;
      const int c = in ? e0 + e1 + e2 : 0;
      tv[r] = d.flags[c];
      if constexpr (sizeof(R) == 4) pv[r] = d.phif[c];
      else pv[r] = d.phi[c];
      k1 += kRowStep - GE, k2 += 1;
      if (k1 >= GE) k1 -= GE, k2 += 1;
    }
    k1 = threadIdx.x >> 4, k2 = 0;
    if (k1 >= GE) k1 -= GE, k2 = 1;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      if (k0 < GE && k2 < GE) {
        const int bs = k0 * bstep[0] + k1 * bstep[1] + k2 * bstep[2];
        const uint8_t t = ((inside >> r) & 1u) ? (uint8_t)(tv[r] & F_TYPE) : (uint8_t)4;  // outside: solid
        styp[bs] = t;
        sphi[bs] = t >= T_OBST ? kObstacle<R>() : pv[r];
        solid_here |= t >= T_OBST;
        if (t == T_IFACE && (unsigned)(k0 - 3) < (unsigned)core[0] && (unsigned)(k1 - 3) < (unsigned)core[1] &&
            (unsigned)(k2 - 3) < (unsigned)core[2]) {
          // an interface cell of the tile: n^ there and at its face neighbours
          uint8_t* m = need_n + (sel3(p.inv[0], k0, k1, k2) - 2) +
                       GN * ((sel3(p.inv[1], k0, k1, k2) - 2) + GN * (sel3(p.inv[2], k0, k1, k2) - 2));
          m[0] = 1;
          m[-1] = 1;
          m[1] = 1;
          m[-GN] = 1;
          m[GN] = 1;
          m[-GN * GN] = 1;
          m[GN * GN] = 1;
        }
      }
      k1 += kRowStep - GE, k2 += 1;
      if (k1 >= GE) k1 -= GE, k2 += 1;
    }
  }
  // without an obstacle in the box the stencils below need no substitution
  // (most tiles)
  const bool solid = __syncthreads_or(solid_here) != 0;
  unsigned take = 0u;
#pragma unroll
  for (int r = 0; r < (GN3 + NT - 1) / NT; ++r) {
    const int s = threadIdx.x + r * NT;
    if (s < GN3 && need_n[s]) {
      const int i = s % GN + 2, j = (s / GN) % GN + 2, k = s / (GN * GN) + 2;
      if (styp[i + GE * (j + GE * k)] < T_OBST) {  // at an obstacle the centre's n^ stands in
        take |= 1u << r;
        uint8_t* m = need_s + (i - 1) + GS * ((j - 1) + GS * (k - 1));
#pragma unroll
        for (int e = 0; e < 27; ++e) m[(e % 3 - 1) + GS * (((e / 3) % 3 - 1) + GS * (e / 9 - 1))] = 1;
      }
    }
  }
  push_shared<GN3, NT>(list_n, &s_count[0], take);
  __syncthreads();
  take = 0u;
#pragma unroll
  for (int r = 0; r < (GS3 + NT - 1) / NT; ++r) {
    const int s = threadIdx.x + r * NT;
    take |= (unsigned)(s < GS3 && need_s[s]) << r;
  }
  push_shared<GS3, NT>(list_s, &s_count[1], take);
  __syncthreads();
  auto smooth = [&](auto SOLID) {
    constexpr bool kSolid = decltype(SOLID)::value;
    const int n = s_count[1];
    for (int q = threadIdx.x; q < n; q += NT) {
      const int s = list_s[q];
      const int b = (s % GS + 1) + GE * ((s / GS) % GS + 1 + GE * (s / (GS * GS) + 1));
      sps[s] = (kSolid && is_obstacle(sphi[b])) ? kObstacle<R>() : smoothed_at<R, kSolid>(sphi, b);
    }
  };
  if (solid) smooth(std::true_type{});
  else smooth(std::false_type{});
  __syncthreads();
  auto normals = [&](auto SOLID) {
    constexpr bool kSolid = decltype(SOLID)::value;
    const int n = s_count[0];
    for (int q = threadIdx.x; q < n; q += NT) {
      const int s = list_n[q];
      R v[3];
      normal_at<R, kSolid>(sps, (s % GN + 1) + GS * ((s / GN) % GN + 1 + GS * (s / (GN * GN) + 1)), v);
      snh[s] = v[0];
      snh[GN3 + s] = v[1];
      snh[2 * GN3 + s] = v[2];
    }
  };
  if (solid) normals(std::true_type{});
  else normals(std::false_type{});
  __syncthreads();
  // curvature, gas density and Thuerey class of the tile's interface cells
  for (int s = threadIdx.x; s < GT * GT * GT; s += blockDim.x) {
    const int i = s % GT + 3, j = (s / GT) % GT + 3, k = s / (GT * GT) + 3;
    const int X = ox + i, Y = oy + j, Z = oz + k;
    if (X >= p.nx || Y >= p.ny || Z >= p.nz) continue;
    const int b = i + GE * (j + GE * k);
    if (styp[b] != T_IFACE) continue;
    const int c = cidx(p, X, Y, Z);
    auto nh = [&](int a, int ii, int jj, int kk) {
      return snh[a * GN3 + (ii - 2) + GN * ((jj - 2) + GN * (kk - 2))];
    };
    R acc = R(0.0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int ex = (a == 0), ey = (a == 1), ez = (a == 2);
      const R vc = nh(a, i, j, k);
      const R vp = (styp[b + ex + GE * (ey + GE * ez)] >= T_OBST) ? vc : nh(a, i + ex, j + ey, k + ez);
      const R vm = (styp[b - ex - GE * (ey + GE * ez)] >= T_OBST) ? vc : nh(a, i - ex, j - ey, k - ez);
      acc = acc + (vp - vm);
    }
    const R kappa = R(-0.5) * acc;
    const int bb = p.bubble_model ? d.bid[c] : -1;
    if constexpr (S::kDev) {
      // rho^G - 1 = 3 (p^V - 1/3) + 3 sigma kappa, formed in FP64
      const double pv = bb >= 0 ? d.pV[bb] : p.pv0;
      rhog[c] = R(3.0 * (pv - 1.0 / 3.0) + 3.0 * p.sigma * (double)kappa);
    } else {
      const R pv = bb >= 0 ? R(d.pV[bb]) : R(p.pv0);
      rhog[c] = R(3.0) * (pv + R(p.sigma) * kappa);
    }
    nhat[3LL * c + 0] = nh(0, i, j, k);
    nhat[3LL * c + 1] = nh(1, i, j, k);
    nhat[3LL * c + 2] = nh(2, i, j, k);
    bool hl = false, hg = false;
#pragma unroll
    for (int q = 1; q < Q; ++q) {
      const int t = styp[b + CX(q) + GE * (CY(q) + GE * CZ(q))];
      hl |= (t == T_LIQ);
      hg |= (t == T_GAS);
    }
    d.cls[c] = T_IFACE | (((!hl && hg) ? CL_NF : (hl && !hg) ? CL_NE : CL_STD) << 2);
  }
  if (threadIdx.x == 0) d.tile_mark[tile] = 0;
}

// Resets the work-list counters that this step fills (next band list, new
// cells, next tile list, converting cells, receivers).
__device__ __forceinline__ void reset_step_counts(const DPtrs& d, int parity) {
  d.counts[parity ^ 1] = 0;
  d.counts[2] = 0;
  d.counts[3 + (parity ^ 1)] = 0;
  *conv_count(d) = 0;
  *recv_count(d) = 0;
}

template <int Q, class S>
__global__ void __launch_bounds__(kGeoBlock, kGeoMinBlocks) k_geometry(DPtrs d, KParams p, int parity) {
  stage_begin();
  extern __shared__ __align__(16) unsigned char g_smem[];
  if (blockIdx.x == 0 && threadIdx.x == 0) reset_step_counts(d, parity);
  const int ntiles = d.counts[3 + parity];
  for (int tt = blockIdx.x; tt < ntiles; tt += gridDim.x)
    geometry_tile<Q, S>(d, p, d.tiles[parity][tt], g_smem);
}

// Hand-out of n geometry tiles to the blocks of a persistent grid: block b
// takes tile b, later ones come from a per-step counter (zero at init, cleared
// again every step).  Blocks without a tile go on at once, and with at most a
// tile a block nothing waits for the counter (608 atomics on one address and
// two barriers took 2 us of every block).
template <class F>
__device__ __forceinline__ void hand_out_tiles(int n, int* counter, int* s_tile, F tile) {
  int t = blockIdx.x;
  while (t < n) {
    tile(t);
    if (n <= (int)gridDim.x) break;
    __syncthreads();  // every thread has read the previous *s_tile
    if (threadIdx.x == 0) *s_tile = gridDim.x + atomicAdd(counter, 1);
    __syncthreads();
    t = *s_tile;
  }
}

// The bulk sweep with the geometry pass folded in (FP32 and 16-bit
// engines).  The blocks of the persistent grid first take geometry tiles
// until none is left, and then bulk units.  The tiles so run at the sweep's
// occupancy with no launch boundary before the sweep.  On the 160x160x1024
// Taylor bubble: separate kernels 77.5 + 295 us, every block first on tiles
// 345 us, every second block 364 us, every fourth 361 us: the sweep needs all
// its blocks to keep HBM busy, so blocks held by tiles slow it by about what
// running the tiles beside it saves.  (Figures of when a tile took twice as
// long; the launch takes 326 to 330 us now.)
template <int Q, class S, int COLL>
__global__ void __launch_bounds__(kBulkBlock, (bulk_min_blocks<Q, S, COLL>()))
    k_bulk_geo(DPtrs d, KParams p, int parity) {
  stage_begin();
  extern __shared__ __align__(16) unsigned char g_smem[];
  __shared__ int s_tile;
  if (blockIdx.x == 0 && threadIdx.x == 0) reset_step_counts(d, parity);
  hand_out_tiles(d.counts[3 + parity], &d.counts[7], &s_tile, [&](int t) {
    geometry_tile<Q, S, kBulkBlock>(d, p, d.tiles[parity][t], g_smem);
  });
  bulk_sweep<Q, S, COLL>(d, p, parity);
}

// ------------------------------------------------------- interface update
// Directions whose neighbour data the mass exchange reads ahead at once, and
// resident blocks of 128 threads per SM the FP32/FP16 interface kernels are
// compiled for (the kernel is latency-bound: three blocks cap it at 168
// registers a thread, which every variant fits without spilling; four
// blocks at 128 registers measured 10 % slower on the Taylor bubble (118 vs
// 107 us); the FP64 engine keeps two).  FSLBM_IFACE_MINB, when defined,
// sets the bound for the FP32 and 16-bit engines.
#ifndef FSLBM_IFACE_CHUNK
#define FSLBM_IFACE_CHUNK 6
#endif

constexpr int kIfaceChunk = FSLBM_IFACE_CHUNK;
// Half-width of the band of n^.c_i values that count as a tie n.c_i = 0
// (Appendix A assumes that only c_0 ties; at mirror planes of the interface
// a component of n^ is zero in exact arithmetic and rounding-sized in any
// precision, so the sign alone would decide by rounding).  Exact in FP32
// and FP64 alike.
constexpr double kTie = 0x1p-20;
template <class S, int COLL>
constexpr int iface_min_blocks() {
#ifdef FSLBM_IFACE_MINB
  return sizeof(typename S::Real) == 4 ? FSLBM_IFACE_MINB : 2;
#else
  return sizeof(typename S::Real) == 4 ? 3 : 2;
#endif
}
// Pull with the free-surface BC (Eq. nm-fslbm-boundary-condition) on the
// variant's set R (Sec. 3), mass exchange (Eq. nm-fslbm-mass-flux) with
// Thuerey's adjustment, fill update phi = m / rho, collision, marks.
template <int Q, class S, int COLL>
__device__ __forceinline__ void interface_cell(const DPtrs& d, const KParams& p, int parity, int k,
                                               bool& bad) {
  using R = typename S::Real;
  using T = typename S::T;
  const int* __restrict__ band = d.band[parity];
  const T* __restrict__ A = (const T*)d.pdf[parity];
  T* __restrict__ B = (T*)d.pdf[parity ^ 1];
  const long long Np = p.Np;
  const uint8_t* __restrict__ flags = d.flags;
  const R* nhat = (const R*)d.nhat;
  const R* rhog = (const R*)d.rhog;

    const int c = band[k];
    const uint8_t fl = flags[c];
    const uint32_t wm = (fl & F_NEAR_WALL) ? d.wallmask[c] : 0u;
    // neighbours x + c_i (-1 outside the domain); the pull source of
    // direction i is the neighbour in direction ibar.  A cell beside a
    // free-slip face links to the mirror image of a neighbour across it,
    // whose PDF arrives with the wall-normal component reversed.
    const bool slipface = coll_slip(COLL) && (fl & F_FACE) && (p.slip[0] | p.slip[1] | p.slip[2]);
    int x = 0, y = 0, z = 0;
    int nid[Q];
    nid[0] = c;
    if (!slipface) {
      // the interior offsets, with a bit test a direction for faces and the
      // wrap distances of periodic ones (as in the bulk sweep).  A second
      // path from the coordinates beside the interior one, run by every warp
      // with a cell at a face, cost a 256x128x64 dam break 3.5 of 57 us a
      // step and 8 cylinders (FP16SMC) 11 of 142.
      unsigned faces = 0u;
      Wraps w = {};
      if (fl & (F_FACE | F_WRAP)) {
        decode(p, c, x, y, z);
        faces = faces_at(p, x, y, z);
        w = wraps_at(p, x, y, z);
      }
#pragma unroll
      for (int i = 1; i < Q; ++i) nid[i] = (faces & pull_faces(OPP(i))) ? -1 : c + p.off[i] + w.of(OPP(i));
    } else {
      decode(p, c, x, y, z);
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        int j;
        bool mir;
        nid[i] = pull_source<Q>(p, x, y, z, OPP(i), j, mir);
      }
    }
    // One level of loads: the neighbours' kind (type and class), fill level
    // and arriving PDF do not depend on one another.  Which sources bounce
    // back is static (the wall mask, or outside the domain; a mirror image
    // that is an obstacle is told by its type), and what a gas neighbour's
    // slot holds is dropped below.
    R fx[Q], f[Q];
    int nt[Q];  // type, class in bits 2-3
    nt[0] = T_IFACE;
#pragma unroll
    for (int i = 1; i < Q; ++i) nt[i] = nid[i] >= 0 ? (int)d.cls[nid[i]] : (int)T_OBST;
#pragma unroll
    for (int i = 0; i < Q; ++i) fx[i] = load_own<Q, S>(A, Np, c, i);
    f[0] = fx[0];  // the rest PDF stays in the cell
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const int src = nid[OPP(i)];
      if (!slipface) {
        // A[i Np + src]: with the neighbour at c - off[i] its offset is the
        // interior one
        const bool own = src < 0 || ((wm >> i) & 1u);
        f[i] = load_w<S, Q>(A[(long long)(own ? OPP(i) : i) * Np + (own ? c : src)], i);
      } else {
        int j;
        bool mir;
        (void)pull_source<Q>(p, x, y, z, i, j, mir);
        const bool own = (nt[OPP(i)] & 3) == T_OBST;
        f[i] = load_w<S, Q>(A[(long long)(own ? OPP(i) : j) * Np + (own ? c : src)], i);
      }
    }
    unsigned miss = 0u;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if ((nt[OPP(i)] & 3) == T_GAS) {
        miss |= 1u << i;
        f[i] = R(0.0);
      }
    }
    // mass exchange with the streamed (not yet reconstructed) PDFs:
    // a = f*_ibar(x + c_i) equals the pulled f_ibar(x).  With deviations
    // (w_i = w_ibar cancels) a liquid link's difference enters exactly, as a
    // float pair, so a liquid neighbour's PDF sum changes by exactly -dm_i;
    // an interface link's term is the float product of the same operands
    // that the neighbour negates, so the two terms cancel exactly.
    const int clc = d.cls[c] >> 2;
    double dm = 0.0;
    if constexpr (S::kDev) {
      FAcc acc;
      const float phicf = d.phif[c];
      float phn[Q];
#pragma unroll
      for (int i = 1; i < Q; ++i) phn[i] = nid[i] >= 0 ? d.phif[nid[i]] : 0.0f;
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const int ntp = nt[i] & 3;
        if (ntp == T_GAS || ntp == T_OBST) continue;
        const float fa = f[OPP(i)];
        const float fb = fx[i];
        if (ntp == T_LIQ) {
          acc.add_diff(fa, fb);
        } else {
          const float w = W<Q, float>(i);
          const int cln = nt[i] >> 2;
          float v;
          if (clc == cln) v = __fsub_rn(fa, fb);
          else if (clc == CL_STD) v = (cln == CL_NF) ? __fadd_rn(fa, w) : -__fadd_rn(fb, w);
          else if (clc == CL_NF) v = -__fadd_rn(fb, w);
          else v = __fadd_rn(fa, w);
          acc.add(__fmul_rn(__fmul_rn(0.5f, __fadd_rn(phicf, phn[i])), v));
        }
      }
      dm = acc.value();
    } else {
      const double phic = d.phi[c];
      // the interface neighbours' fill levels, read a chunk of directions at
      // a time ahead of the (ordered) accumulation
      constexpr int kChunk = kIfaceChunk;
#pragma unroll
      for (int i0 = 1; i0 < Q; i0 += kChunk) {
        double ph[kChunk];
#pragma unroll
        for (int a = 0; a < kChunk; ++a) {
          const int i = i0 + a;
          ph[a] = i < Q && nid[i] >= 0 ? d.phi[nid[i]] : 0.0;
        }
#pragma unroll
        for (int a = 0; a < kChunk; ++a) {
          const int i = i0 + a;
          if (i >= Q) continue;
          const int ntp = nt[i] & 3;
          if (ntp == T_GAS || ntp == T_OBST) continue;
          const R fa = f[OPP(i)];
          const R fb = fx[i];
          if (ntp == T_LIQ) {
            dm = dm + (double)(fa - fb);
          } else {
            const int cln = nt[i] >> 2;
            R v;
            if (clc == cln) v = fa - fb;
            else if (clc == CL_STD) v = (cln == CL_NF) ? fa : -fb;
            else if (clc == CL_NF) v = -fb;
            else v = fa;
            dm = dm + 0.5 * (phic + ph[a]) * (double)v;
          }
        }
      }
    }
    const double mn = d.mass[c] + dm;
    // BC velocity from the cell's own post-collision PDFs
    R rc, jx, jy, jz;
    sums<Q, R>(fx, rc, jx, jy, jz);
    if constexpr (S::kDev) rc = R(1.0) + rc;
    const R ux = jx / rc - R(0.5) * gpar<R>(p, 0);
    const R uy = jy / rc - R(0.5) * gpar<R>(p, 1);
    const R uz = jz / rc - R(0.5) * gpar<R>(p, 2);
    // set R of the variant (Sec. 3) and reconstruction; |n^.c_i| <= kTie
    // counts as a tie (n.c_i = 0): NBRC reconstructs ties, NBKC does not
    const R n0 = nhat[3LL * c], n1 = nhat[3LL * c + 1], n2 = nhat[3LL * c + 2];
    int v = p.variant;
    if (v == 4) v = (__popc(miss) >= 3) ? 3 : p.om3_fb;
    const R rg = rhog[c];  // rho^G (FP64 engine) or rho^G - 1
    const R tie = R(kTie);
    const R usq = ux * ux + uy * uy + uz * uz;
    if (v == 1) f[0] = feq_sum<Q, S>(0, rg, ux, uy, uz, usq) - fx[0];  // n^.c_0 = 0: a tie
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const int j = i + 1;
      const R dot = cdot<R>(i, n0, n1, n2);  // -dot for j
      const bool ri = ((miss >> i) & 1u) || (v == 1 && dot >= -tie) || (v == 2 && dot > tie);
      const bool rj = ((miss >> j) & 1u) || (v == 1 && dot <= tie) || (v == 2 && dot < -tie);
      if (ri || rj) {
        const R e = feq_sum<Q, S>(i, rg, ux, uy, uz, usq);
        if (ri) f[i] = e - fx[j];
        if (rj) f[j] = e - fx[i];
      }
    }
    long long s_in = 0;  // the mass-conserving formats: the received values in grid steps
    if constexpr (S::kExactRest) {
#pragma unroll
      for (int i = 0; i < Q; ++i) s_in += grid_steps<S>(f[i]);
    }
    double rho = collide_any<Q, S, COLL>(f, p, bad);
    // moments of the stored post-collision PDFs, in post_moments' arithmetic
    // (new interface cells average them over their neighbours)
    R mu[3];
    if constexpr (S::kDev) {
      // the density as the stored PDFs hold it (FP64 sum of the stored
      // values): the mass a conversion to liquid hands over to them
      double sd = 0.0;
      R fs[Q];
      if constexpr (S::kExactRest) {
        store_cell<Q, S>(B, Np, c, f, s_in, bad);
        const int r0 = rest_slice<Q, S>(B, Np)[c];
        long long n = r0;
        fs[0] = from_steps<S>(r0);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          const T v = S::stored(f[i]);
          fs[i] = S::loadd(v);
          n += S::steps(v);
        }
        sd = (double)n * (1.0 / (double)(1LL << S::kShift));
      } else {
        FAcc sa;  // the float sum carried as a pair: FP64 accuracy, FP32 operations
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const T v = S::stored(f[i]);
          B[(long long)i * Np + c] = v;
          fs[i] = S::loadd(v);
          sa.add(fs[i]);
        }
        sd = sa.value();
      }
      rho = 1.0 + sd;
      R r0, jx0, jy0, jz0;
      sums<Q, R>(fs, r0, jx0, jy0, jz0);
      const R rr = R(rho);
      mu[0] = jx0 / rr - R(0.5) * gpar<R>(p, 0);
      mu[1] = jy0 / rr - R(0.5) * gpar<R>(p, 1);
      mu[2] = jz0 / rr - R(0.5) * gpar<R>(p, 2);
      d.mom_rho[c] = rho;
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i) B[(long long)i * Np + c] = store_w<S, Q>(f[i], i);
      R r0, jx0, jy0, jz0;
      sums<Q, R>(f, r0, jx0, jy0, jz0);
      mu[0] = jx0 / r0 - R(0.5) * gpar<R>(p, 0);
      mu[1] = jy0 / r0 - R(0.5) * gpar<R>(p, 1);
      mu[2] = jz0 / r0 - R(0.5) * gpar<R>(p, 2);
      d.mom_rho[c] = (double)r0;
    }
    {
      R* mu_out = (R*)d.mom_u;
      mu_out[3LL * c + 0] = mu[0];
      mu_out[3LL * c + 1] = mu[1];
      mu_out[3LL * c + 2] = mu[2];
    }
    {
      if (fl & F_NEAR_WALL) write_reflected<Q, S>(d, p, B, c, wm, (fl & F_WRAP) != 0, f);
    }
    double phin;
    if constexpr (S::kDev) {
      // mn / rho from the float reciprocal and one Newton step in FP64
      // (relative error about 2^-46; an FP64 division takes tens of FP64
      // operations)
      const double r0 = (double)__frcp_rn(d2f(rho));
      const double q0 = mn * r0;
      phin = fma(fma(-q0, rho, mn), r0, q0);
    } else {
      phin = mn / rho;
    }
    d.m_next[k] = mn;
    d.phi_next[k] = phin;
    if constexpr (!S::kDev) d.rho_band[c] = rho;
    const uint8_t mark = (phin > 1.0 + p.eps) ? CV_TOL : (phin < -p.eps) ? CV_TOG : CV_NONE;
    d.mark[c] = mark;
    if (mark != CV_NONE) append_conversion(d, parity, c);
  }

// List entry that a thread of the grid starts at.  A list that needs at most
// one warp of every block is dealt a warp a block, so that it spreads over
// the SMs; a longer one runs through the blocks in order (neighbouring
// entries are neighbouring cells, whose reads share the SM's L1).
__device__ __forceinline__ int band_start(int n) {
  if (n <= (int)gridDim.x * 32) return ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
  return blockIdx.x * blockDim.x + threadIdx.x;
}

template <int Q, class S, int COLL>
__global__ void __launch_bounds__(128, (iface_min_blocks<S, COLL>())) k_interface(const __grid_constant__ DPtrs d, const __grid_constant__ KParams p, int parity) {
  stage_begin();
  const int n = d.counts[parity];
  if (lane_band<Q, S>(n)) {
    interface_by_lanes<Q, S, COLL>(d, p, parity, n);
    return;
  }
  bool bad = false;
  for (int k = band_start(n); k < n; k += gridDim.x * blockDim.x)
    interface_cell<Q, S, COLL>(d, p, parity, k, bad);
  if (bad) d.err[0] = 1;
}

// -------------------------------------------------------------- finalize
// Fixed-point bubble-volume term round((1 - phi) 2^32).
__device__ __forceinline__ long long vol_fix(double one_minus_phi) {
  return __double2ll_rn(one_minus_phi * 4294967296.0);
}

// Adds the geometry tile of cell c (c < 0: none) to a tile list once; every
// lane of the warp must call it.
__device__ __forceinline__ void mark_tile(const DPtrs& d, const KParams& p, int c, int* list,
                                          int* count) {
  int tile = -1;
  if (c >= 0) {
    int x, y, z;
    decode(p, c, x, y, z);
    const int ntx = (p.nx + 7) / 8, nty = (p.ny + 7) / 8;
    tile = (x >> 3) + ntx * ((y >> 3) + nty * (z >> 3));
  }
  const unsigned peers = __match_any_sync(0xffffffffu, tile);
  const bool lead = tile >= 0 && (int)(threadIdx.x & 31u) == __ffs(peers) - 1;
  const bool fresh = lead && atomicExch(&d.tile_mark[tile], 1) == 0;
  const int pos = warp_append(count, fresh);
  if (fresh) list[pos] = tile;
}

// Adds the kSegCells-cell group of cell c (c < 0: none) to the liquid group
// list once; every lane of the warp must call it.
__device__ __forceinline__ void mark_seg(const DPtrs& d, int c) {
  const int seg = c >= 0 ? (c / kSegCells) : -1;
  const unsigned peers = __match_any_sync(0xffffffffu, seg);
  const bool lead = seg >= 0 && (int)(threadIdx.x & 31u) == __ffs(peers) - 1;
  const bool fresh = lead && atomicExch(&d.seg_mark[seg], 1) == 0;
  const int pos = warp_append(&d.counts[5], fresh);
  if (fresh) d.segs[pos] = seg;
}

// Initial liquid group list (blocks of 256 cover whole groups).
static __global__ void k_segs_init(DPtrs d, KParams p) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool liq = c < p.N && (d.flags[c] & F_TYPE) == T_LIQ;
  const unsigned b = __ballot_sync(0xffffffffu, liq);
  const unsigned gmask = kSegCells == 32 ? 0xffffffffu : ((1u << kSegCells) - 1u);
  const bool fresh = (lane % kSegCells) == 0 && ((b >> lane) & gmask) != 0;
  if (fresh) d.seg_mark[c / kSegCells] = 1;
  const int pos = warp_append(&d.counts[5], fresh);
  if (fresh) d.segs[pos] = c / kSegCells;
}

// What the context derives from flags and fill levels (checkpoint load).
static __global__ void k_derive_fields(DPtrs d, KParams p) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  d.cls[c] = d.flags[c] & F_TYPE;
  if (d.phif) d.phif[c] = d2f(d.phi[c]);
}

// Tile list of an interface list (initial state and checkpoint load).
static __global__ void k_tiles_of_band(DPtrs d, KParams p, int parity) {
  const int n = d.counts[parity];
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (int base = wid * 32; base < n; base += warps * 32) {
    const int k = base + (threadIdx.x & 31);
    mark_tile(d, p, k < n ? d.band[parity][k] : -1, d.tiles[parity], &d.counts[3 + parity]);
  }
}

// Final flags, tile and segment marks, bubble gas counts and interface sums
// of one cell a lane (c < 0: none), a band cell or a new interface cell;
// every lane of the warp calls it.  The interface list of the next step is
// rebuilt from the flags afterwards (compact_chunk).
__device__ __forceinline__ void finalize_lane(const DPtrs& d, const KParams& p, int parity, int c,
                                              bool is_band) {
  const int lane = threadIdx.x & 31;
  bool keep = false, to_liq = false;
  int bub = -1, dgas = 0;
  long long vfix = 0;
  if (c >= 0) {
    const uint8_t fl = d.flags[c];
    const int b = d.bid[c];
    if (is_band) {
      const uint8_t f = d.cfin[c];
      if (f != CV_NONE) {  // the marks of a listed cell are spent
        d.cfin[c] = CV_NONE;
        d.conv[c] = CV_NONE;
      }
      if (f == CV_TOL) {
        d.flags[c] = (fl & ~F_TYPE) | T_LIQ;
        d.cls[c] = T_LIQ;
        d.bid[c] = -1;
        to_liq = true;
      } else if (f == CV_TOG) {
        d.flags[c] = (fl & ~F_TYPE) | T_GAS;
        d.cls[c] = T_GAS;
        dgas = 1;
      } else {
        keep = true;
      }
    } else {
      if ((fl & F_TYPE) == T_GAS) dgas = -1;
      d.flags[c] = (fl & ~F_TYPE) | T_IFACE;
      d.cls[c] = T_IFACE;  // its class follows with the next geometry pass
      d.claim[c] = 0;
      keep = true;
    }
    if (p.bubble_model && b >= 0) {
      bub = b;
      if (keep) vfix = vol_fix(1.0 - d.phi[c]);
    }
  }
  if (p.bubble_model) {
    // integer sums per bubble id present in the warp, one atomic each
    // (integer addition: the result does not depend on the order)
    unsigned remaining = __ballot_sync(0xffffffffu, bub >= 0);
    while (remaining) {
      const int leader = __ffs(remaining) - 1;
      const int bb = __shfl_sync(0xffffffffu, bub, leader);
      const bool mine = (bub == bb);
      long long sv = mine ? vfix : 0, sg = mine ? (long long)dgas : 0;
      for (int o = 16; o > 0; o >>= 1) {
        sv += __shfl_xor_sync(0xffffffffu, sv, o);
        sg += __shfl_xor_sync(0xffffffffu, sg, o);
      }
      if (lane == leader) {
        if (sv) atomicAdd((unsigned long long*)&d.iface_fix[bb], (unsigned long long)sv);
        if (sg) atomicAdd((unsigned long long*)&d.gas_cnt[bb], (unsigned long long)sg);
      }
      remaining &= ~__ballot_sync(0xffffffffu, mine);
    }
  }
  mark_tile(d, p, keep ? c : -1, d.tiles[parity ^ 1], &d.counts[3 + (parity ^ 1)]);
  mark_seg(d, to_liq ? c : -1);
}

static __global__ void __launch_bounds__(kBlock) k_finalize(DPtrs d, KParams p, int parity) {
  stage_begin();
  const int nband = d.counts[parity], nnew = d.counts[2];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    d.counts[6] = 0;  // the next step's bulk hand-out
    d.counts[7] = 0;  // and geometry-tile hand-out
  }
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (int base = wid * 32; base < nband; base += warps * 32)
    finalize_lane(d, p, parity, base + lane < nband ? d.band[parity][base + lane] : -1, true);
  for (int base = wid * 32; base < nnew; base += warps * 32)
    finalize_lane(d, p, parity, base + lane < nnew ? d.newlist[base + lane] : -1, false);
}

// ------------------------------------------------------------ observables
// Per-block partials: [0] mass, [1] max|u|^2, [2] liquid volume, [3] nan,
// [4..7] counts of gas, interface, liquid, obstacle.
//
// One read of the PDFs bounds the pass if the FP64 unit (two lanes a clock
// per SM) is kept out of it, so the deviation formats do their per-cell work
// in FP32 and integers: rho - 1 is summed in fixed point (see PartSum; grid
// steps in the mass-conserving formats), u and the candidates for the largest
// |u| are formed in FP32, and FP64 squares only where the FP32 estimate comes
// near the largest value so far (the result is the FP64 one).  The mass is the
// number of liquid cells plus their deviations plus the interface masses; |u|
// is rooted once, at the end.
// 160x160x512 tube, FP32 (8.2 M fluid cells, 0.78 GB), a call with the bubble
// pressures: 1006 us with FP64 moments and 2 blocks per SM, 290 so (284 with
// float pairs and without the liquid cells' masses and fill levels).
constexpr int kObsFields = 8;
constexpr int kObsBlocksPerSm = 4;

__device__ __forceinline__ bool is_nan_bits(double x) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}

// The sum of Q <= 27 floats, |d| < 2, by error-free extraction (Ogita, Rump and
// Oishi, "Accurate sum and dot product", SIAM J. Sci. Comput. 26, 2005): adding
// and subtracting 1.5 2^5 rounds d to a multiple of 2^-18, 1.5 2^-15 the rest
// (at most 2^-19) to one of 2^-38.  h (below 54) and m (below 2^-14) then add
// up without rounding, and l (terms of at most 2^-39) is within 2^-54 of its
// sum, so h + m + l is closer to the exact sum than an FP64 sum of 1 + d is.
// Nine operations a term in three short chains; a float pair by TwoSum takes
// seven in one chain and loses up to 2^-42 where the terms' exponents differ
// much.
struct PartSum {
  float h = 0.f, m = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float d) {
    const float a = __fsub_rn(__fadd_rn(48.f, d), 48.f), r = __fsub_rn(d, a);
    const float b = __fsub_rn(__fadd_rn(0x1.8p-15f, r), 0x1.8p-15f);
    h = __fadd_rn(h, a);
    m = __fadd_rn(m, b);
    l = __fadd_rn(l, __fsub_rn(r, b));
  }
  // 1 + the sum, rounded to float once: the rounded sum of the parts, corrected
  // by what it leaves over (1 + h, the difference and the sum with m are exact)
  __device__ __forceinline__ float one_plus() const {
    const float a = __fadd_rn(1.f, h), r = __fadd_rn(a, __fadd_rn(m, l));
    return __fadd_rn(r, __fadd_rn(__fadd_rn(__fsub_rn(a, r), m), l));
  }
};

// rho - 1 summed over cells: multiples of the units below, added as integers.
// A cell adds less than 2^46 to lo, and a thread of the grid meets fewer than
// 2^17 cells (a domain has at most 4e8), so neither overflows.
template <class S>
struct DevSum {
  long long hi = 0, lo = 0;
  __host__ __device__ static constexpr double unit_hi() { return S::kExactRest ? 1.0 / (double)(1LL << grid_shift<S>()) : 0x1p-18; }
  __host__ __device__ static constexpr double unit_lo() { return 0x1p-60; }
};

// Adds rho - 1 of a cell to `dev` if add, and gives rho in FP32 and the velocity
// (in post_moments' arithmetic).  False if the cell's deviations are outside
// the range of PartSum: then dr is their FP64 sum, and dev is left alone.
template <int Q, class S>
__device__ __forceinline__ bool obs_moments(const typename S::T* P, long long Np, int c, const KParams& p, bool add,
                                            DevSum<S>& dev, double& dr, float& rr, float u[3]) {
  bool fits = true;
  float f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = load_own<Q, S>(P, Np, c, i);
  float r, jx, jy, jz;
  sums<Q, float>(f, r, jx, jy, jz);
  if constexpr (S::kExactRest) {
    int n0 = rest_slice<Q, S>(P, Np)[c];
    long long n = n0;
#pragma unroll
    for (int i = 1; i < Q; ++i) n += grid_steps32<S>(f[i]);  // f[i] is a stored value
    rr = d2f(1.0 + (double)n * (1.0 / (double)(1LL << S::kShift)));
    if (add) dev.hi += n;
  } else {
    PartSum a;
    unsigned bits = 0u;  // bit 30 (the exponent's first) is set from 2 on, infinities and NaN included
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      a.add(f[i]);
      bits |= __float_as_uint(f[i]);
    }
    fits = !(bits & 0x40000000u);
    if (fits) {
      rr = a.one_plus();
      if (add) {
        dev.hi += __float2int_rn(a.h * 0x1p18f);
        dev.lo += ((long long)__float2int_rn(a.m * 0x1p38f) << 22) + __float2int_rn(a.l * 0x1p60f);
      }
    } else {
      dr = 0.0;
#pragma unroll 1
      for (int i = 0; i < Q; ++i) dr += (double)load_w<S, Q>(P[(long long)i * Np + c], i);
      rr = d2f(1.0 + dr);
    }
  }
  u[0] = jx / rr - 0.5f * gpar<float>(p, 0);
  u[1] = jy / rr - 0.5f * gpar<float>(p, 1);
  u[2] = jz / rr - 0.5f * gpar<float>(p, 2);
  return fits;
}

template <int Q, class S>
__global__ void __launch_bounds__(kBlock, kObsBlocksPerSm) k_obs_partial(DPtrs d, KParams p, int parity,
                                                                          double* part) {
  using R = typename S::Real;
  const typename S::T* P = (const typename S::T*)d.pdf[parity];
  // interface masses (and all masses in FP64) are summed per thread with
  // Neumaier's compensation, then pairwise across threads and blocks
  double mass = 0.0, mcomp = 0.0, u2max = 0.0, vol = 0.0;
  DevSum<S> dev;  // of the liquid cells (deviation formats)
  float near_max = -1.0f;  // a float bound below the largest |u|^2 so far
  int nan = 0, cnt[4] = {0, 0, 0, 0};
  auto add_mass = [&](double x) {
    const double s = mass + x;
    mcomp += (fabs(mass) >= fabs(x)) ? ((mass - s) + x) : ((x - s) + mass);
    mass = s;
  };
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < p.N; c += gridDim.x * blockDim.x) {
    const int t = d.flags[c] & F_TYPE;
#pragma unroll
    for (int k = 0; k < 4; ++k) cnt[k] += t == k;
    if (t != T_LIQ && t != T_IFACE) continue;
    // mass and fill level of every fluid cell (a checkpoint may hold anything);
    // a liquid cell's are checked with integer operations and enter the sums
    // through the count of liquid cells
    const double m = d.mass[c], ph = d.phi[c];
    if (is_nan_bits(m)) nan = 1;
    if (t == T_IFACE) vol += ph;
    else if (__double_as_longlong(ph) != 0x3ff0000000000000LL) vol += ph - 1.0;
    if constexpr (S::kDev) {
      double dr = 0.0;
      float rr, u[3];
      const bool fits = obs_moments<Q, S>(P, p.Np, c, p, t == T_LIQ, dev, dr, rr, u);
      const float q = __fmaf_rn(u[0], u[0], __fmaf_rn(u[1], u[1], u[2] * u[2]));
      if (!(q == q) || !(rr > 0.0f)) nan = 1;
      if (q >= near_max) {
        const double uu = (double)u[0] * u[0] + (double)u[1] * u[1] + (double)u[2] * u[2];
        if (uu > u2max) u2max = uu;
        near_max = (float)u2max * 0.9999f;
      }
      if (t == T_IFACE) add_mass(m);
      else if (!fits) add_mass(dr);
    } else {
      double r;
      R u[3];
      post_moments<Q, S>(P, p.Np, c, p, r, u);
      const double uu = (double)u[0] * u[0] + (double)u[1] * u[1] + (double)u[2] * u[2];
      if (!(uu == uu) || !(r > 0.0)) nan = 1;
      if (uu > u2max) u2max = uu;
      add_mass((t == T_LIQ) ? r : m);
    }
  }
  if constexpr (S::kDev) {
    add_mass((double)dev.hi * dev.unit_hi());
    add_mass((double)dev.lo * dev.unit_lo());
    add_mass((double)cnt[T_LIQ]);
  }
  vol += (double)cnt[T_LIQ];
  __shared__ double sh[kObsFields][kBlock / 32];
  double v[kObsFields] = {mass + mcomp, u2max, vol, (double)nan, (double)cnt[0], (double)cnt[1], (double)cnt[2],
                          (double)cnt[3]};
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int f = 0; f < kObsFields; ++f) {
    double a = v[f];
    for (int o = 16; o > 0; o >>= 1) {
      const double b = __shfl_down_sync(0xffffffffu, a, o);
      a = (f == 1 || f == 3) ? fmax(a, b) : a + b;
    }
    if (lane == 0) sh[f][w] = a;
  }
  __syncthreads();
  if (threadIdx.x < kObsFields) {
    const int f = threadIdx.x;
    double a = sh[f][0];
    for (int i = 1; i < kBlock / 32; ++i) a = (f == 1 || f == 3) ? fmax(a, sh[f][i]) : a + sh[f][i];
    part[blockIdx.x * kObsFields + f] = a;
  }
}

// One warp a field: each lane adds every 32nd partial, then the lanes add up
// (a single thread a field reads the partials one after another: 46 us for
// 304 blocks).
static __global__ void __launch_bounds__(32 * kObsFields) k_obs_final(const double* part, int nblocks, double* out) {
  const int f = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool mx = f == 1 || f == 3;
  double a = 0.0;  // of a sum and of maxima of values >= 0
  for (int b = lane; b < nblocks; b += 32) {
    const double v = part[b * kObsFields + f];
    a = mx ? fmax(a, v) : a + v;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double b = __shfl_down_sync(0xffffffffu, a, o);
    a = mx ? fmax(a, b) : a + b;
  }
  if (lane == 0) out[f] = f == 1 ? sqrt(a) : a;
}

// PDFs of the current buffer as FP64 (zero on gas and obstacle cells), in
// the caller's cell order: thread e writes the cell with caller index e.
template <int Q, class S>
__global__ void k_pdf_out(DPtrs d, KParams p, int parity, double* out) {
  using R = typename S::Real;
  const typename S::T* P = (const typename S::T*)d.pdf[parity];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= p.N) return;
  const int c = storage_of_ext(p, e);
  const int t = d.flags[c] & F_TYPE;
  const bool fluid = (t == T_LIQ || t == T_IFACE);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    double v;
    if constexpr (S::kExactRest) {
      if (i == 0) {
        out[(long long)i * p.N + e] =
            fluid ? (double)rest_slice<Q, S>(P, p.Np)[c] * (1.0 / (double)(1LL << S::kShift)) + W<Q, double>(0)
                  : 0.0;
        continue;
      }
    }
    if constexpr (S::kDev)
      v = (double)S::loadd(P[(long long)i * p.Np + c]) + W<Q, double>(i);
    else
      v = (double)S::load(P[(long long)i * p.Np + c], W<Q, R>(i));
    out[(long long)i * p.N + e] = fluid ? v : 0.0;
  }
}

// ------------------------------------------------------------ storage order
// Liquid-holding kSegCells-cell groups of the storage order p over flags
// given in the caller's order (one warp = one 32-cell group): the work list
// length of the bulk sweep if the cells were stored that way.
static __global__ void k_layout_census(const uint8_t* __restrict__ raw_ext, KParams p,
                                       unsigned long long* groups) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const bool liq = c < p.N && raw_ext[ext_index(p, c)] == T_LIQ;
  const unsigned b = __ballot_sync(0xffffffffu, liq);
  if ((threadIdx.x & 31) == 0 && b) {
    int n = 0;
    for (int g = 0; g < 32; g += kSegCells) n += ((b >> g) & (kSegCells == 32 ? 0xffffffffu : ((1u << kSegCells) - 1u))) != 0u;
    atomicAdd(groups, (unsigned long long)n);
  }
}

// Arrays between the caller's cell order and the storage order: ncomp
// consecutive arrays of N entries each.
template <class T>
__global__ void k_to_storage(const T* __restrict__ ext, T* __restrict__ st, KParams p, int ncomp) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  const int e = ext_index(p, c);
  for (int k = 0; k < ncomp; ++k) st[(long long)k * p.N + c] = ext[(long long)k * p.N + e];
}
template <class T>
__global__ void k_to_caller(const T* __restrict__ st, T* __restrict__ ext, KParams p) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= p.N) return;
  ext[e] = st[storage_of_ext(p, e)];
}

// Cell types of the flags in the caller's cell order.
static __global__ void k_types_to_caller(const uint8_t* __restrict__ flags, uint8_t* __restrict__ ext, KParams p) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < p.N) ext[e] = flags[storage_of_ext(p, e)] & F_TYPE;
}

// ---------------------------------------------------------------- batches
// Many domains of different sizes advance in one launch per phase.  The
// block table is an array of DomRec; the plan kernels turn each domain's
// device-side list counts into prefix offsets, and every batched kernel maps
// its global work index to (domain, local index) by binary search over the
// offsets.  Domain ranges of the cell lists are padded to multiples of 32,
// so a warp never straddles two domains and the warp-collective code of the
// single-domain bodies runs unchanged.

// Plan of the first phase (before geometry): resets the counters this step
// fills and lays out tiles, bulk warp units and band cells.
static __global__ void kb_plan_front(DomRec* recs, BatchPlan pl) {
  stage_begin();
  constexpr int kGroups = 32 / kSegCells;
  if (threadIdx.x == 0) {
    pl.ctr[0] = 0;  // the bulk sweep's hand-out counter
    pl.ctr[1] = 0;  // and the fused sweep's tile counter
  }
  for (int k = threadIdx.x; k < pl.n; k += blockDim.x) reset_step_counts(recs[k].d, recs[k].parity);
  __syncthreads();
  block_prefix(pl.n, pl.tiles, [&](int k) { return recs[k].d.counts[3 + recs[k].parity]; });
  block_prefix(pl.n, pl.bulk, [&](int k) { return (recs[k].d.counts[5] + kGroups - 1) / kGroups; });
  block_prefix(pl.n, pl.band, [&](int k) { return round32(recs[k].d.counts[recs[k].parity]); });
}

template <int Q, class S>
__global__ void __launch_bounds__(kGeoBlock, kGeoMinBlocks) kb_geometry(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  extern __shared__ __align__(16) unsigned char g_smem[];
  const int total = pl.tiles[pl.n];
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    const int k = find_domain(pl.tiles, pl.n, t);
    const DomRec& r = recs[k];
    geometry_tile<Q, S>(r.d, r.p, r.d.tiles[r.parity][t - pl.tiles[k]], g_smem);
  }
}

// Units of all domains handed out as in k_bulk.
template <int Q, class S, int COLL>
__device__ __forceinline__ void batch_bulk_sweep(const DomRec* __restrict__ recs, const BatchPlan& pl) {
  const int total = pl.bulk[pl.n];
  auto unit = [&](int w) {
    const int k = find_domain(pl.bulk, pl.n, w);
    const DomRec& r = recs[k];
    bulk_unit<Q, S, COLL>(r.d, r.p, r.parity, w - pl.bulk[k], r.d.counts[5]);
  };
  hand_out_units<S>(total, &pl.ctr[0], unit);
}

template <int Q, class S, int COLL>
__global__ void __launch_bounds__(kBulkBlock, (bulk_min_blocks<Q, S, COLL>()))
    kb_bulk(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  batch_bulk_sweep<Q, S, COLL>(recs, pl);
}

// The batch's bulk sweep with the geometry tiles of all domains folded in,
// as k_bulk_geo: the blocks first take tiles from the plan's tile counter,
// then bulk units.
template <int Q, class S, int COLL>
__global__ void __launch_bounds__(kBulkBlock, (bulk_min_blocks<Q, S, COLL>()))
    kb_bulk_geo(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  extern __shared__ __align__(16) unsigned char g_smem[];
  __shared__ int s_tile;
  hand_out_tiles(pl.tiles[pl.n], &pl.ctr[1], &s_tile, [&](int t) {
    const int k = find_domain(pl.tiles, pl.n, t);
    const DomRec& r = recs[k];
    geometry_tile<Q, S, kBulkBlock>(r.d, r.p, r.d.tiles[r.parity][t - pl.tiles[k]], g_smem);
  });
  batch_bulk_sweep<Q, S, COLL>(recs, pl);
}

template <int Q, class S, int COLL>
__global__ void __launch_bounds__(128, (iface_min_blocks<S, COLL>())) kb_interface(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  const int total = pl.band[pl.n];  // with each domain's cells rounded up to whole warps
  if (lane_band<Q, S>(total)) {
    interface_by_lanes<Q, S, COLL>(recs, pl.band, pl.n, total);
    return;
  }
  for (int g = band_start(total); g < total; g += gridDim.x * blockDim.x) {
    const int k = find_domain(pl.band, pl.n, g);
    const DomRec& r = recs[k];
    const int i = g - pl.band[k];
    if (i >= r.d.counts[r.parity]) continue;
    bool bad = false;
    interface_cell<Q, S, COLL>(r.d, r.p, r.parity, i, bad);
    if (bad) r.d.err[0] = 1;
  }
}

static __global__ void __launch_bounds__(kBlock) kb_finalize(const DomRec* __restrict__ recs, BatchPlan pl) {
  stage_begin();
  const int total = pl.band[pl.n];
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (int base = wid * 32; base < total; base += warps * 32) {
    const int k = find_domain(pl.band, pl.n, base);
    const DomRec& r = recs[k];
    const int i = base - pl.band[k] + lane;
    finalize_lane(r.d, r.p, r.parity, i < r.d.counts[r.parity] ? r.d.band[r.parity][i] : -1, true);
  }
  deal_domains(pl.n, [&](int k, int first, int stride) {
    const DomRec& r = recs[k];
    const int nnew = r.d.counts[2];
    for (int b = first * 32; b < nnew; b += stride * 32)
      finalize_lane(r.d, r.p, r.parity, b + lane < nnew ? r.d.newlist[b + lane] : -1, false);
  });
}

// Bubble pressures of every domain (one block each), then the step is done
// and the domain's buffers swap.
static __global__ void kb_bubble_end(DomRec* recs) {
  stage_begin();
  DomRec& r = recs[blockIdx.x];
  if (r.p.bubble_model && r.d.nb > 0) bubble_update(r.d, r.p);
  __syncthreads();
  if (threadIdx.x == 0) r.parity ^= 1;
}

}  // namespace fslbm
