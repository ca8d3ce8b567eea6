// Host-side launch sequence of one FSLBM step for a given lattice and PDF
// storage format.  Included by the per-precision translation units, each of
// which exports one table of entry points (Ops) to the C-ABI layer.
#pragma once

#include "fslbm_internal.h"
#include <type_traits>

#include "fslbm_kernels.cuh"
#include "fslbm_band_list.cuh"

namespace fslbm {

// Calls f with the collision variant as a compile-time constant
// (bit 0: TRT, bit 1: Smagorinsky model, bit 2: free-slip faces).
template <class F>
inline void with_coll(int coll, F&& f) {
  switch (coll) {
    case 0: f(std::integral_constant<int, 0>{}); break;
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    default: f(std::integral_constant<int, 7>{}); break;
  }
}

// The kernels' variant: the collision variant and, in bit 2, whether the
// domain has free-slip faces (the free-slip logic is compiled only then).
inline int iface_coll(const KParams& p) { return coll_of(p) | slip_bit(p); }

template <int Q, class S>
struct Engine {
  // persistent bulk blocks per SM the sweep is compiled for
  static constexpr int bulk_blocks_per_sm() {
    return sizeof(typename S::Real) == 4 ? kBulkMinBlocks32 : 2;
  }
  static int grid_cells(const KParams& p) { return (p.N + kBlock - 1) / kBlock; }
  // blocks of k_compact_band: one chunk of kCompactChunk cells each, at most
  // 4 per band block (8 per SM; the grid loops over the remaining chunks)
  static int compact_grid(const KParams& p, int band_grid) {
    const long long chunks = ((long long)p.N + kCompactChunk - 1) / kCompactChunk;
    const long long cap = 4LL * band_grid;
    return (int)(chunks < cap ? chunks : cap);
  }
  // the FP32 and 16-bit engines fold the geometry pass into the bulk sweep
  static constexpr bool kFusedGeo = sizeof(typename S::Real) == 4;
  // shared-memory carveout (percent of the 228 KB) that holds a tile buffer
  // for every persistent block of the fused sweep; the rest stays L1
  static constexpr int fused_carveout() {
    return (kBulkMinBlocks32 * ((int)geometry_smem<typename S::Real>() + 1024) * 100 + 228 * 1024 - 1) /
           (228 * 1024);
  }

  static void init_cells(const DPtrs& d, const KParams& p, const uint8_t* raw, const double* fill,
                         const double* vel, const double* den, cudaStream_t st) {
    k_init_cells<Q, S><<<grid_cells(p), kBlock, 0, st>>>(raw, fill, vel, den, d, p, 0);
  }
  static void init_check(const KParams& p, const uint8_t* raw, int* bad, cudaStream_t st) {
    k_init_check<Q><<<grid_cells(p), kBlock, 0, st>>>(raw, p, bad);
  }
  static void cc_union(const uint8_t* raw, const KParams& p, int* lab, cudaStream_t st) {
    k_cc_union<Q><<<grid_cells(p), kBlock, 0, st>>>(raw, p, lab);
  }
  static void cc_assign(const uint8_t* raw, const KParams& p, const int* lab, const int* root_id,
                        int* bid, cudaStream_t st) {
    k_cc_assign<Q><<<grid_cells(p), kBlock, 0, st>>>(raw, p, lab, root_id, bid);
  }

  // One step reading pdf[parity], band[parity]; writing the other buffers.
  // Returns the first error of its launches.
  // With a Fork (and no stage events) the bulk sweep runs on the side stream
  // while geometry, interface update and the first conversion passes run on
  // the main stream; the streams join before k_apply, the first kernel that
  // reads post-collision PDFs of liquid cells.
  static cudaError_t step(const DPtrs& d, const KParams& p, int parity, int band_grid, int bulk_grid,
                          cudaStream_t st, StageEvents* ev, const Fork* fk) {
    FirstError keep;
    const int coll = iface_coll(p);
    const bool bub = p.bubble_model && d.nb > 0;
    const bool chained = !ev;  // with an event between two kernels there is nothing to chain
    // the next list, and the bubble pressures in a block of the same launch (a
    // launch of its own while stages are timed)
    auto list_and_bubbles = [&]() {
      const int beside = bub && !ev;
      keep(launch_stage(chained, k_compact_band, compact_grid(p, band_grid) + beside, kBlock, 0, st, d, p, parity,
                        beside));
      if (ev) ev->mark(7, st);
      if (bub && ev) keep(launch_stage(false, k_compact_band, 1, kBlock, 0, st, d, p, parity, 1));
      if (ev) ev->mark(8, st);
    };
    if constexpr (kFusedGeo) {
      // geometry and bulk in one persistent launch, then the band chain
      constexpr size_t sm = geometry_smem<typename S::Real>();
      if (ev) {
        ev->mark(0, st);
        ev->mark(1, st);
      }
      with_coll(coll, [&](auto C) {
        keep(launch_stage(false, k_bulk_geo<Q, S, decltype(C)::value>, bulk_grid, kBulkBlock, sm, st, d, p, parity));
      });
      if (ev) ev->mark(2, st);
      with_coll(coll, [&](auto C) {
        keep(launch_stage(chained, k_interface<Q, S, decltype(C)::value>, band_grid * 2, 128, 0, st, d, p, parity));
      });
      if (ev) ev->mark(3, st);
      keep(launch_stage(chained, k_resolve<Q>, band_grid * 2, kBlock, 0, st, d, p, parity));
      if (ev) ev->mark(4, st);
      keep(launch_stage(chained, k_count<Q, S>, band_grid * 2, kBlock, 0, st, d, p, parity));
      if (ev) ev->mark(5, st);
      if (ev) {  // its two parts one after the other while stages are timed
        keep(launch_stage(false, k_apply<Q, S, true, false>, band_grid * 2, kBlock, 0, st, d, p, parity));
        keep(launch_stage(false, k_apply<Q, S, false, true>, band_grid * 2, kBlock, 0, st, d, p, parity));
      } else {
        keep(launch_stage(chained, k_apply<Q, S, true, true>, band_grid * 2, kBlock, 0, st, d, p, parity));
      }
      if (ev) ev->mark(6, st);
      keep(launch_stage(chained, k_finalize, band_grid, kBlock, 0, st, d, p, parity));
      list_and_bubbles();
    } else {
      auto bulk = [&](cudaStream_t s2) {
        with_coll(coll, [&](auto C) {
          keep(launch_stage(false, k_bulk<Q, S, decltype(C)::value>, bulk_grid, kBulkBlock, 0, s2, d, p, parity));
        });
      };
      const bool forked = fk && !ev;
      auto fork_bulk = [&]() {
        keep(cudaEventRecord(fk->fork, st));
        keep(cudaStreamWaitEvent(fk->side, fk->fork, 0));
        bulk(fk->side);
        keep(cudaEventRecord(fk->join, fk->side));
      };
      if (ev) ev->mark(0, st);
      if (forked) fork_bulk();
      keep(launch_stage(false, k_geometry<Q, S>, band_grid * kGeoGridMult, kGeoBlock,
                        geometry_smem<typename S::Real>(), st, d, p, parity));
      if (ev) ev->mark(1, st);
      if (!forked) bulk(st);
      if (ev) ev->mark(2, st);
      with_coll(coll, [&](auto C) {
        keep(launch_stage(chained, k_interface<Q, S, decltype(C)::value>, band_grid * 2, 128, 0, st, d, p, parity));
      });
      if (ev) ev->mark(3, st);
      keep(launch_stage(chained, k_resolve<Q>, band_grid * 2, kBlock, 0, st, d, p, parity));
      if (ev) ev->mark(4, st);
      keep(launch_stage(chained, k_count<Q, S>, band_grid * 2, kBlock, 0, st, d, p, parity));
      if (ev) ev->mark(5, st);
      if (forked) keep(cudaStreamWaitEvent(st, fk->join, 0));
      keep(launch_stage(chained && !forked, k_apply<Q, S, true, true>, band_grid * 2, kBlock, 0, st, d, p, parity));
      if (ev) ev->mark(6, st);
      keep(launch_stage(chained, k_finalize, band_grid, kBlock, 0, st, d, p, parity));
      list_and_bubbles();
    }
    return keep.e;
  }

  // One step of all domains of a block table.  Same stages and stream fork
  // as step(); the plan kernels lay out each phase's work on the device, and
  // the last kernel swaps every domain's buffers.  collision: the variant
  // shared by the members (coll_of), with bit 2 set when one of them has
  // free-slip faces.
  static cudaError_t batch_step(DomRec* recs, const BatchPlan& pl, int band_grid, int bulk_grid,
                                int collision, cudaStream_t st, const Fork* fk) {
    FirstError keep;
    keep(launch_stage(false, kb_plan_front, 1, 1024, 0, st, recs, pl));
    constexpr size_t sm = geometry_smem<typename S::Real>();
    if constexpr (kFusedGeo) {
      with_coll(collision, [&](auto C) {
        keep(launch_stage(true, kb_bulk_geo<Q, S, decltype(C)::value>, bulk_grid, kBulkBlock, sm, st, recs, pl));
      });
      with_coll(collision, [&](auto C) {
        keep(launch_stage(true, kb_interface<Q, S, decltype(C)::value>, band_grid * 2, 128, 0, st, recs, pl));
      });
      keep(launch_stage(true, kb_resolve<Q>, band_grid * 2, kBlock, 0, st, recs, pl));
      keep(launch_stage(true, kb_count<Q, S>, band_grid * 2, kBlock, 0, st, recs, pl));
      keep(launch_stage(true, kb_apply<Q, S, true, true>, band_grid * 2, kBlock, 0, st, recs, pl));
      keep(launch_stage(true, kb_finalize, band_grid, kBlock, 0, st, recs, pl));
      keep(launch_stage(true, kb_bubble_end, pl.n, 256, 0, st, recs));
      (void)fk;
    } else {
      keep(cudaEventRecord(fk->fork, st));
      keep(cudaStreamWaitEvent(fk->side, fk->fork, 0));
      with_coll(collision, [&](auto C) {
        keep(launch_stage(false, kb_bulk<Q, S, decltype(C)::value>, bulk_grid, kBulkBlock, 0, fk->side, recs, pl));
      });
      keep(cudaEventRecord(fk->join, fk->side));
      keep(launch_stage(false, kb_geometry<Q, S>, band_grid * kGeoGridMult, kGeoBlock, sm, st, recs, pl));
      with_coll(collision, [&](auto C) {
        keep(launch_stage(true, kb_interface<Q, S, decltype(C)::value>, band_grid * 2, 128, 0, st, recs, pl));
      });
      keep(launch_stage(true, kb_resolve<Q>, band_grid * 2, kBlock, 0, st, recs, pl));
      keep(launch_stage(true, kb_count<Q, S>, band_grid * 2, kBlock, 0, st, recs, pl));
      keep(cudaStreamWaitEvent(st, fk->join, 0));
      // the new cells' FP64 chains beside the receivers' (4 drops of 48 to 80
      // cells a side: 315.2 us a step so, 315.4 in one launch)
      keep(cudaEventRecord(fk->fork, st));
      keep(cudaStreamWaitEvent(fk->side, fk->fork, 0));
      keep(launch_stage(false, kb_apply<Q, S, true, false>, band_grid * 2, kBlock, 0, fk->side, recs, pl));
      keep(cudaEventRecord(fk->join, fk->side));
      keep(launch_stage(false, kb_apply<Q, S, false, true>, band_grid * 2, kBlock, 0, st, recs, pl));
      keep(cudaStreamWaitEvent(st, fk->join, 0));
      keep(launch_stage(false, kb_finalize, band_grid, kBlock, 0, st, recs, pl));
      keep(launch_stage(true, kb_bubble_end, pl.n, 256, 0, st, recs));
    }
    return keep.e;
  }

  static void observables(const DPtrs& d, const KParams& p, int parity, double* out,
                          cudaStream_t st) {
    k_obs_partial<Q, S><<<d.red_blocks, kBlock, 0, st>>>(d, p, parity, d.red);
    k_obs_final<<<1, 32 * kObsFields, 0, st>>>(d.red, d.red_blocks, out);
  }

  static void pdf_out(const DPtrs& d, const KParams& p, int parity, double* out, cudaStream_t st) {
    k_pdf_out<Q, S><<<grid_cells(p), kBlock, 0, st>>>(d, p, parity, out);
  }

  static Ops ops() {
    if constexpr (!kFusedGeo) {
      cudaFuncSetAttribute(k_geometry<Q, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)geometry_smem<typename S::Real>());
      cudaFuncSetAttribute(kb_geometry<Q, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)geometry_smem<typename S::Real>());
    }
    Ops o;
    o.init_cells = &init_cells;
    o.init_check = &init_check;
    o.cc_union = &cc_union;
    o.cc_assign = &cc_assign;
    o.step = &step;
    o.observables = &observables;
    o.pdf_out = &pdf_out;
    o.elem_size = sizeof(typename S::T);
    o.real_size = sizeof(typename S::Real);
    o.rest_size = S::kExactRest ? sizeof(int) : 0;
    if constexpr (kFusedGeo) {
      const void* fns[8] = {(const void*)&k_bulk_geo<Q, S, 0>, (const void*)&k_bulk_geo<Q, S, 1>,
                            (const void*)&k_bulk_geo<Q, S, 2>, (const void*)&k_bulk_geo<Q, S, 3>,
                            (const void*)&k_bulk_geo<Q, S, 4>, (const void*)&k_bulk_geo<Q, S, 5>,
                            (const void*)&k_bulk_geo<Q, S, 6>, (const void*)&k_bulk_geo<Q, S, 7>};
      for (int c = 0; c < 8; ++c) {
        o.bulk_fn[c] = fns[c];
        cudaFuncSetAttribute(fns[c], cudaFuncAttributePreferredSharedMemoryCarveout, fused_carveout());
      }
    } else {
        o.bulk_fn[0] = (const void*)&k_bulk<Q, S, 0>;
        o.bulk_fn[1] = (const void*)&k_bulk<Q, S, 1>;
        o.bulk_fn[2] = (const void*)&k_bulk<Q, S, 2>;
        o.bulk_fn[3] = (const void*)&k_bulk<Q, S, 3>;
        o.bulk_fn[4] = (const void*)&k_bulk<Q, S, 4>;
        o.bulk_fn[5] = (const void*)&k_bulk<Q, S, 5>;
        o.bulk_fn[6] = (const void*)&k_bulk<Q, S, 6>;
        o.bulk_fn[7] = (const void*)&k_bulk<Q, S, 7>;
    }
    o.bulk_blocks_per_sm = bulk_blocks_per_sm();
    // bulk and geometry (one launch when fused), interface, resolve, count,
    // apply, finalize, list rebuild with the bubbles; while stages are timed
    // the apply stage is two launches when fused and the bubbles are their own
    o.step_launches = kFusedGeo ? 7 : 8;
    o.bulk_smem = kFusedGeo ? geometry_smem<typename S::Real>() : 0;
    o.batch_step = &batch_step;
    // plan, geometry and bulk sweep (one launch when fused), interface update,
    // resolve, count, apply (two in FP64), finalize,
    // bubbles + buffer swap, and kb_compact_band, launched by the batch
    o.batch_step_launches = kFusedGeo ? 9 : 11;
    if constexpr (kFusedGeo) {
      const void* fns[8] = {(const void*)&kb_bulk_geo<Q, S, 0>, (const void*)&kb_bulk_geo<Q, S, 1>,
                            (const void*)&kb_bulk_geo<Q, S, 2>, (const void*)&kb_bulk_geo<Q, S, 3>,
                            (const void*)&kb_bulk_geo<Q, S, 4>, (const void*)&kb_bulk_geo<Q, S, 5>,
                            (const void*)&kb_bulk_geo<Q, S, 6>, (const void*)&kb_bulk_geo<Q, S, 7>};
      for (int c = 0; c < 8; ++c) {
        o.batch_bulk_fn[c] = fns[c];
        cudaFuncSetAttribute(fns[c], cudaFuncAttributePreferredSharedMemoryCarveout, fused_carveout());
      }
    } else {
        o.batch_bulk_fn[0] = (const void*)&kb_bulk<Q, S, 0>;
        o.batch_bulk_fn[1] = (const void*)&kb_bulk<Q, S, 1>;
        o.batch_bulk_fn[2] = (const void*)&kb_bulk<Q, S, 2>;
        o.batch_bulk_fn[3] = (const void*)&kb_bulk<Q, S, 3>;
        o.batch_bulk_fn[4] = (const void*)&kb_bulk<Q, S, 4>;
        o.batch_bulk_fn[5] = (const void*)&kb_bulk<Q, S, 5>;
        o.batch_bulk_fn[6] = (const void*)&kb_bulk<Q, S, 6>;
        o.batch_bulk_fn[7] = (const void*)&kb_bulk<Q, S, 7>;
    }
    return o;
  }
};

}  // namespace fslbm
