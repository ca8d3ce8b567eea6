// Bulk sweep of the FSLBM step (arXiv 2207.13962, Sec. 2.1): the pull
// stream-collide of liquid cells over the liquid segment list.  Kept in its
// own header so that the recorded DRAM traffic of this kernel is tied to the
// sources it is built from (this file, the cell layer and the common types).
#pragma once

#include "fslbm_cell.cuh"

namespace fslbm {
// ------------------------------------------------------------ bulk sweep
// Pull stream-collide of liquid cells (Eqs. nm-lbm-streaming, -collision)
// with bounce-back at obstacles.  Interface and gas cells are skipped.
//
// Bounce-back through the obstacle's slot: a fluid cell x whose pull source
// x - c_i is an obstacle cell writes, besides its own PDFs, f*_ibar(x) into
// slot i of that obstacle cell.  That slot is pulled by x alone, so the write
// is race-free, and next step x pulls its bounced-back PDF from the constant
// offset like any interior cell: the bulk sweep reads at constant offsets
// except next to a non-periodic domain face (own-slot bounce-back) or across
// a periodic face (wrap distances; see below).  Every kernel that produces post-collision PDFs of a fluid cell (bulk, interface,
// new interface cells, init) writes these reflected copies.
constexpr int kBulkBlock = 256;

// How a warp finds the pull sources of its cells: all inside the domain; some
// across a no-slip face (bounce-back from the cell's own slot); some across a
// periodic face as well.  With free-slip faces the last two are one.
//
// A row of a closed box begins and ends at a face, so with rows of a few
// segments a third to all of the warps meet one.  Indexing every direction
// from the coordinates there (compare, wrap, multiply) took more instructions
// than the collision; the offset table with a bit test a direction, and a sum
// of wrap distances at periodic faces, take a few.  Sweep with tiles, indexing
// from coordinates against this: 96x96x384 tube in FP16SMC 92 / 74.5 us, 192^3
// drop 47.5 / 43, 160x160x1024 tube 333 / 326, 37x21x11 tank 18.6 / 15.4.
enum { kInterior = 0, kFace = 1, kWrap = 2 };

// Bits 2a / 2a + 1: the cell touches the lower / upper no-slip face of axis a.
__device__ __forceinline__ unsigned faces_at(const KParams& p, int x, int y, int z) {
  unsigned m = 0u;
  if (!p.per[0]) m |= (x == 0 ? 1u : 0u) | (x == p.nx - 1 ? 2u : 0u);
  if (!p.per[1]) m |= (y == 0 ? 4u : 0u) | (y == p.ny - 1 ? 8u : 0u);
  if (!p.per[2]) m |= (z == 0 ? 16u : 0u) | (z == p.nz - 1 ? 32u : 0u);
  return m;
}
// The faces that direction i is pulled through (its source is x - c_i).
__host__ __device__ constexpr unsigned pull_faces(int i) {
  return (CX(i) > 0 ? 1u : CX(i) < 0 ? 2u : 0u) | (CY(i) > 0 ? 4u : CY(i) < 0 ? 8u : 0u) |
         (CZ(i) > 0 ? 16u : CZ(i) < 0 ? 32u : 0u);
}
// Storage distance from x - c_i to its image across the periodic faces.
struct Wraps {
  int lo[3], hi[3];  // per axis: added when the source lies below / above
  __device__ __forceinline__ int of(int i) const {
    return (CX(i) > 0 ? lo[0] : CX(i) < 0 ? hi[0] : 0) + (CY(i) > 0 ? lo[1] : CY(i) < 0 ? hi[1] : 0) +
           (CZ(i) > 0 ? lo[2] : CZ(i) < 0 ? hi[2] : 0);
  }
};
__device__ __forceinline__ Wraps wraps_at(const KParams& p, int x, int y, int z) {
  Wraps w;
  w.lo[0] = p.per[0] && x == 0 ? p.nx * p.sx : 0;
  w.hi[0] = p.per[0] && x == p.nx - 1 ? -p.nx * p.sx : 0;
  w.lo[1] = p.per[1] && y == 0 ? p.ny * p.sy : 0;
  w.hi[1] = p.per[1] && y == p.ny - 1 ? -p.ny * p.sy : 0;
  w.lo[2] = p.per[2] && z == 0 ? p.nz * p.sz : 0;
  w.hi[2] = p.per[2] && z == p.nz - 1 ? -p.nz * p.sz : 0;
  return w;
}

// One liquid cell, loads straight from global memory.
template <int Q, class S, int COLL>
__device__ __forceinline__ void bulk_cell(const DPtrs& d, const KParams& p, int parity, int c,
                                          uint8_t fl, int path) {
  using R = typename S::Real;
  using T = typename S::T;
  const T* __restrict__ A = (const T*)d.pdf[parity];
  T* __restrict__ B = (T*)d.pdf[parity ^ 1];
  const long long Np = p.Np;
  R f[Q];
  // the mass-conserving formats hold the rest PDF in an int32 slice
  constexpr int i0 = S::kExactRest ? 1 : 0;
  if (path == kInterior) {
    const T* Ac = A + c;
#pragma unroll
    for (int i = i0; i < Q; ++i) f[i] = load_w<S, Q>(Ac[p.dofs[i]], i);
  } else {
    int x, y, z;
    decode(p, c, x, y, z);
    if constexpr (coll_slip(COLL)) {
#pragma unroll
      for (int i = i0; i < Q; ++i)
        f[i] = load_w<S, Q>(A[pull_index_slip<Q>(p, d.flags, c, x, y, z, i)], i);
    } else {
      // a bit per no-slip face the cell touches, tested against the faces a
      // direction is pulled through
      const unsigned faces = faces_at(p, x, y, z);
      const T* Ac = A + c;
      if (path == kFace) {
#pragma unroll
        for (int i = i0; i < Q; ++i)
          f[i] = load_w<S, Q>(Ac[(faces & pull_faces(i)) ? (long long)OPP(i) * Np : p.dofs[i]], i);
      } else {
        const Wraps w = wraps_at(p, x, y, z);
#pragma unroll
        for (int i = i0; i < Q; ++i)
          f[i] = load_w<S, Q>(Ac[(faces & pull_faces(i)) ? (long long)OPP(i) * Np : p.dofs[i] + w.of(i)], i);
      }
    }
  }
  long long s_in = 0;
  if constexpr (S::kExactRest) {
    // the received stored values in grid steps, summed exactly
    const int r0 = rest_slice<Q, S>(A, Np)[c];
    f[0] = from_steps<S>(r0);
    s_in = r0;
#pragma unroll
    for (int i = 1; i < Q; ++i) s_in += grid_steps32<S>(f[i]);
  }
  bool bad = false;
  collide_any<Q, S, COLL>(f, p, bad);
  store_cell<Q, S, true>(B, Np, c, f, s_in, bad);
  if (fl & F_NEAR_WALL) write_reflected<Q, S>(d, p, B, c, d.wallmask[c], path == kWrap, f);
  if (bad) d.err[0] = 1;
}

// One warp's share of the direct bulk sweep: groups [w G, w G + G) of the
// liquid group list, G = 32 / kSegCells (every lane of the warp calls it).
// Gas lanes that share a 32-byte sector of a PDF slice with a liquid lane
// store zero PDFs (gas values are never read): the sector is then written
// whole, which spares HBM a read-modify-write of it.  Interface lanes (the
// interface kernel writes them concurrently) and obstacle lanes (reflected
// copies) store nothing.
#ifndef FSLBM_BULK_FILL
#define FSLBM_BULK_FILL 1
#endif
template <int Q, class S, int COLL>
__device__ __forceinline__ void bulk_unit(const DPtrs& d, const KParams& p, int parity, int w,
                                          int nseg) {
  using T = typename S::T;
  using R = typename S::Real;
  constexpr int kGroups = 32 / kSegCells;
  constexpr int kFill = (32 / (int)sizeof(T)) < kSegCells ? (32 / (int)sizeof(T)) : kSegCells;
  const int lane = threadIdx.x & 31;
  const int e = w * kGroups + lane / kSegCells;
  const int c = e < nseg ? d.segs[e] * kSegCells + (lane % kSegCells) : p.N;
  const uint8_t fl = c < p.N ? d.flags[c] : (uint8_t)T_IFACE;
  const int t = fl & F_TYPE;
  const bool liq = t == T_LIQ;
  // the whole warp takes the path that its most demanding cell needs
  const bool wrap = __any_sync(0xffffffffu, liq && (fl & F_WRAP));
  const bool face = __any_sync(0xffffffffu, liq && (fl & F_FACE));
  const int path = wrap ? kWrap : face ? kFace : kInterior;
  const unsigned lm = __ballot_sync(0xffffffffu, liq);
  if (liq) {
    bulk_cell<Q, S, COLL>(d, p, parity, c, fl, path);
  } else if (FSLBM_BULK_FILL) {
    const unsigned grp = (lm >> (lane & ~(kFill - 1))) & ((1u << kFill) - 1u);
    if (grp && t == T_GAS) {
      T* __restrict__ B = (T*)d.pdf[parity ^ 1];
#pragma unroll
      for (int i = S::kExactRest ? 1 : 0; i < Q; ++i) B[(long long)i * p.Np + c] = S::store(R(0.0), W<Q, R>(i));
    }
    if constexpr (S::kExactRest) {
      // the int32 rest slice: 8 cells per 32-byte sector
      if (((lm >> (lane & ~7)) & 0xffu) && t == T_GAS) rest_slice<Q, S>(d.pdf[parity ^ 1], p.Np)[c] = 0;
    }
  }
}

// Hand-out of n warp-sized units of work to the warps of a persistent grid.
//
// Each warp's first chunk is fixed by its number, later ones come from a
// per-step counter (zero at init, cleared again every step).  Long lists are
// handed out kBulkChunk consecutive units at a time: a warp then sweeps
// neighbouring segments one after another while the 32-byte sectors they
// share are still in L2, and the grid works on one front of the list.  A
// list of less than short_rounds units a warp is handed out unit by unit:
// in whole chunks it would fill a part of the warps only or leave a last
// round that is nearly empty, and its sectors stay in L2 anyway.  The line
// lies where the counter's atomics (one address, so one after another) cost
// more than that: 4 units a warp for the formats whose units are short, 6 for
// FP32MC, whose units are longer (integer rest sums) but whose sectors leave
// L2 as FP32's do, 16 where a unit is long and the sectors are half as many or
// the arithmetic hides them (FP16SMC, FP64).  Step with units one by one /
// chunks of 4, us (domain, units a warp):
//   FP32     64x64x256 tube, 2.9: 53.9 / 56.4; 256x128x64 dam, 3.3: 65.1 / 63.7
//   FP32MC   256x128x64 dam (D3Q27), 4.4: 87 / 92; 192^3 cylinder (D3Q27), 5.6: 113 / 119;
//            320x160x80 dam, 6.5: 98 / 94; 224^3 drop, 8.1: 122 / 117;
//            384x192x96 dam, 11: 152 / 114; the same in D3Q27, 15: 210 / 164
//   FP16SMC  256x128x64 dam (D3Q27), 4.4: 86 / 92; 320x160x80 dam, 6.5: 98 / 101;
//            96x96x384 tube, 10: 118 / 121; 256^3 cylinder (D3Q27), 15: 215 / 214
//   FP64     192^3 cylinder (D3Q27), 8.4: 1090 / 1145; 192^3 drop, 10: 962 / 981;
//            208^3 cylinder (D3Q27), 13: 1643 / 1636
// Warps are numbered over the blocks first and from the last block down, so
// that a short list is spread over the SMs, one unit a warp, and starts on
// the blocks that hold no geometry tile.
// FSLBM_BULK_DYN = 0: no hand-out, a fixed stride over the list.
#ifndef FSLBM_BULK_DYN
#define FSLBM_BULK_DYN 4
#endif
constexpr int kBulkChunk = FSLBM_BULK_DYN;
static_assert(kBulkChunk >= 0, "units a chunk, or 0 for a fixed stride");
template <class S>
__host__ __device__ constexpr int short_rounds() {
  return !S::kDev ? 16 : !S::kExactRest ? 4 : sizeof(typename S::T) == 4 ? 6 : 16;
}

template <class S, class F>
__device__ __forceinline__ void hand_out_units(int n, int* counter, F unit) {
  const int warps = gridDim.x * (kBulkBlock / 32);
  if constexpr (kBulkChunk == 0) {
    for (int w = blockIdx.x * (kBulkBlock / 32) + (threadIdx.x >> 5); w < n; w += warps) unit(w);
    return;
  }
  constexpr int kShort = short_rounds<S>();
  const int chunk = n >= warps * kShort ? kBulkChunk : 1;
  int base = ((threadIdx.x >> 5) * gridDim.x + (gridDim.x - 1 - blockIdx.x)) * chunk;
  while (base < n) {
    const int end = base + chunk < n ? base + chunk : n;
    for (int w = base; w < end; ++w) unit(w);
    int next = 0;
    if ((threadIdx.x & 31) == 0) next = atomicAdd(counter, chunk);
    base = warps * chunk + __shfl_sync(0xffffffffu, next, 0);
  }
}

// Resident blocks per SM a bulk sweep is compiled for: the FP32 engines
// kBulkMinBlocks32 (64 registers), 3 with the Smagorinsky model (its
// momentum flux needs more) and in the mass-conserving formats with 27
// directions, the FP64 engine 2.  Step with three / four blocks, us: D3Q27
// FP16SMC, 8 cylinders in a batch 128 / 131; D3Q27 FP32MC, 160x160x384 tube
// 298 / 304, 8 cylinders in a batch 274 / 280; D3Q27 FP32, the same tube 272 /
// 264, cylinders 246 / 244; D3Q19 FP16SMC, the tube 239 / 227, 8 drops in a
// batch 326 / 320; D3Q19 FP32MC 224 / 209 and 313 / 306.
template <int Q, class S, int COLL>
constexpr int bulk_min_blocks() {
  return sizeof(typename S::Real) == 4 ? (coll_les(COLL) || (S::kExactRest && Q == 27) ? 3 : kBulkMinBlocks32) : 2;
}

// The sweep over the liquid segments by the warps of a persistent grid.
template <int Q, class S, int COLL>
__device__ __forceinline__ void bulk_sweep(const DPtrs& d, const KParams& p, int parity) {
  constexpr int kGroups = 32 / kSegCells;
  const int nseg = d.counts[5];
  hand_out_units<S>((nseg + kGroups - 1) / kGroups, &d.counts[6],
                    [&](int w) { bulk_unit<Q, S, COLL>(d, p, parity, w, nseg); });
}

template <int Q, class S, int COLL>
__global__ void __launch_bounds__(kBulkBlock, (bulk_min_blocks<Q, S, COLL>()))
    k_bulk(DPtrs d, KParams p, int parity) {
  stage_begin();
  bulk_sweep<Q, S, COLL>(d, p, parity);
}

}  // namespace fslbm
