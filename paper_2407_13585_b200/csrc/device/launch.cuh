// Host-side launcher of a cluster instantiation: picks the skeleton from the cluster's
// roots, the vector width from the shapes, sizes the grid to the machine and the scratch
// region to the grid.
#pragma once
#include <algorithm>

#include "../graph.h"
#include "../registry.h"
#include "hist.cuh"
#include "scanring.cuh"
#include "segfold.cuh"
#include "skeletons.cuh"
#include "slabgather.cuh"
#include "stencil.cuh"
#include "tile.cuh"

namespace acc {

// Opt-in to `smem` bytes of dynamic shared memory for a kernel, asked of the driver once per device
// and size: `granted` (one per kernel, 64 zeroed words) remembers the largest size already granted.
template <class K>
inline bool opt_in_shared_memory(K kern, size_t smem, int* granted) {
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) {
    cudaGetLastError();
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
  }
  if (granted[device] >= (int)smem + 1) return true;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
  granted[device] = (int)smem + 1;
  return true;
}

// Blocks of `kern` (no dynamic shared memory) that are resident at once on the current device, 0 if the device
// cannot launch a grid cooperatively; asked of the driver once per kernel and device (`fit_on`: 64 zeroed words).
inline int resident_grid(const void* kern, int block, int* fit_on) {
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) { cudaGetLastError(); return 0; }
  if (fit_on[device] == 0) {
    int fit = 0;
    if (!cooperative_launch_ok() || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, block, 0) != cudaSuccess) {
      cudaGetLastError();
      fit = 0;
    }
    fit_on[device] = fit + 1;
  }
  return (fit_on[device] - 1) * sm_count();
}

template <class CL>
struct Launcher {
  static constexpr int N = CL::c.n;
  static constexpr bool kHasScan = dev::count_if<CL>(dev::is_scan_root) > 0;
  static constexpr bool kHasRowFold = dev::count_if<CL>(dev::is_row_fold) > 0;
  static constexpr int kScalarFolds = dev::count_if<CL>(dev::is_scalar_fold);
  static constexpr int kScanBlock = dev::scan_block<CL>();
  static constexpr int kScanTile = kScanBlock * dev::scan_rows<CL>() * 4;
  static constexpr bool kHasSegFold = dev::count_if<CL>(dev::is_segfold_root) > 0;
  // exactly one scatter, fp32 '+': its bins can live in shared memory (k_hist)
  static constexpr bool kHistShape = !kHasScan && !kHasRowFold && dev::count_if<CL>(dev::is_permute_root) == 1 &&
                                     dev::count_if<CL>(dev::is_f32_add_permute) == 1;

  // Local id of the array whose index space root `i` iterates over, -1 if i is no root.
  static int domain_of(int i) {
    const CNode& n = CL::c.nodes[i];
    if (dev::is_store_root(n) || dev::is_scan_root(n) || dev::is_segfold_root(n)) return i;
    if (dev::is_fold_root(n)) return n.in[0];
    if (dev::is_permute_root(n)) return n.in[1];
    return -1;
  }

  // Iteration domain: shape of the first root's index space.
  static bool domain(const ClusterLaunch& L, int& R, int& C) {
    for (int i = 0; i < N; ++i) {
      const int at = domain_of(i);
      if (at >= 0) { R = L.nodes[at].R; C = L.nodes[at].C; return true; }
    }
    return false;
  }

  // Every root must iterate over the same domain (a legal cluster has one iteration size).
  static bool domains_agree(const ClusterLaunch& L, int R, int C) {
    for (int i = 0; i < N; ++i) {
      const int at = domain_of(i);
      if (at >= 0 && (L.nodes[at].R != R || L.nodes[at].C != C)) return false;
    }
    return true;
  }

  // 128-bit accesses need every array's innermost extent and base address to allow them.
  static bool vec_ok(const ClusterLaunch& L, int C) {
    if (C % 4) return false;
    for (int i = 0; i < N; ++i) {
      const CNode& n = CL::c.nodes[i];
      if (!n.member) {
        bool as_array = false;                         // free variables are scalar reads
        for (int j = 0; j < N; ++j)
          for (int s = 0; s < CL::c.nodes[j].narr; ++s)
            if (CL::c.nodes[j].member && CL::c.nodes[j].in[s] == i) as_array = true;
        if (!as_array) continue;
      } else if (!dev::is_store_root(n) && !dev::is_scan_root(n)) {
        continue;                                      // never written with a vector store
      }
      if (L.nodes[i].C % 4 || (reinterpret_cast<uintptr_t>(L.nodes[i].ptr) & 15)) return false;
    }
    return true;
  }

  // The streaming kernels over a rank-1 domain take any length 128 bits at a time (all but its last few elements): every
  // array they read at the domain's own index starts on 16 bytes.  Only a reversal asks whether the length is a multiple of
  // four.  (142458709 elements of the chain: 152 -> 111 us; 10^8 + 1 keys into 4096 bins: 291 -> 118 us.)
  static bool stream_vec_ok(const ClusterLaunch& L, bool vec) { return vec || (dev::domain_rank<CL>() <= 1 && !dev::has_reversal<CL>()); }

  static int stream_grid(int R, int C, bool vec) {
    const int64_t per_row = C / (vec || dev::domain_rank<CL>() <= 1 ? 4 : 1);
    const int64_t trips = dev::domain_rank<CL>() <= 1
                              ? (per_row + dev::kBlock - 1) / dev::kBlock
                              : ((per_row + 31) / 32) * ((R + dev::kStreamTileRows - 1) / dev::kStreamTileRows);
    return (int)std::max<int64_t>(1, std::min<int64_t>(trips, (int64_t)sm_count() * 8));
  }

  // folds of few elements, over all arrays that are read or stored: one cluster of blocks (k_stream_few, where both sides' times are)
  static constexpr bool kFewShape = dev::few_eligible<CL>();
  static constexpr int kFewElements = 1 << 18;
  static bool use_few(const ClusterLaunch&, int R, int C) { return kFewShape && (int64_t)R * C * dev::few_arrays<CL>() <= kFewElements; }

  // transposes staged through shared-memory tile pairs (k_tile_pair)
  static constexpr bool kTileShape = dev::tile_eligible<CL>();
  static constexpr int kRowFolds = dev::count_if<CL>(dev::is_row_fold);

  // ... or, where there are few (and more than one), by a cluster of blocks to every block of rows (k_tile_rows, where both sides'
  // times are).  Two arrays, up to 33 blocks of rows: with two blocks per SM 33 clusters run at once, a 34th afterwards (us, the pair kernels /
  // this one: 2048 rows 14.4 / 11.4, 2111 21.9 / 16.4, 2112 14.3 / 13.0; 2176 14.3 / 18.4, 2177 21.5 / 23.6, 2559 20.5 / 28.3).  One array,
  // up to 2559 rows: it stays ahead to about 3100 (2624 rows 16.4 / 12.3, 3000 16.4 / 14.2, 3100 18.3 / 16.4, 3300 17.6 / 18.5), measured
  // with nothing else in the L2; where other arrays go through it between two runs is not measured there.
  static constexpr bool kTileRowsShape = dev::tile_rows_eligible<CL>();
  static constexpr int kTileRowsMost = dev::staged_externals<CL>() == 1 ? 2559 : 33 * dev::kTile;
  static bool use_tile_rows(int n) { return kTileRowsShape && n > dev::kTile && n <= kTileRowsMost; }

  // The tile-pair kernel wants a square domain of at least one tile, and every staged
  // external of that same shape.
  static bool use_tiles(const ClusterLaunch& L, int R, int C) {
    if constexpr (kTileShape) {
      if (R != C || R < dev::kTile) return false;
      for (int i = 0; i < N; ++i)
        if (dev::is_staged_external<CL>(i) && (L.nodes[i].R != R || L.nodes[i].C != C)) return false;
      return true;
    } else {
      return false;
    }
  }

  // blocks of k_segfold: one per eight warps' runs of the folds' source (its records are laid out for them)
  static int seg_grid(const ClusterLaunch& L) {
    if constexpr (kHasSegFold) {
      const int src = CL::c.nodes[dev::first_segfold<CL>()].in[0];
      const int64_t n_src = (int64_t)L.nodes[src].R * L.nodes[src].C;
      const int64_t span = (int64_t)dev::seg_run(n_src, sm_count()) * (dev::kBlock / 32);
      return (int)std::max<int64_t>(1, (n_src + span - 1) / span);
    } else {
      return 0;
    }
  }

  // 128-bit reads of a segmented fold's operands: every array read as an array has 16-byte rows and base
  static bool seg_vec_ok(const ClusterLaunch& L) {
    for (int i = 0; i < N; ++i) {
      if (CL::c.nodes[i].member) continue;
      bool as_array = false;
      for (int j = 0; j < N; ++j)
        for (int s = 0; s < CL::c.nodes[j].narr; ++s)
          if (CL::c.nodes[j].member && CL::c.nodes[j].in[s] == i) as_array = true;
      if (as_array && (L.nodes[i].C % 4 || (reinterpret_cast<uintptr_t>(L.nodes[i].ptr) & 15))) return false;
    }
    return true;
  }

  // Scans through the shared-memory ring (k_scan_ring), or a warp or block per row where rows are short (k_scan_rows);
  // without them, where a chunk behind an index map would not be a 128-bit access, or where rows are long and the ring does
  // not serve the scan's operand or the device cannot launch a grid with all blocks resident, k_scan, which also takes what
  // it is quicker at.
  static constexpr bool kRingShape = kHasScan && dev::scan_ring_eligible<CL>();
  static constexpr bool kRingServes = kHasScan && dev::ring_serves<CL>();
  static bool use_ring(const ClusterLaunch& L, int R, int C) {
    if constexpr (!kRingShape) return false;
    else return (!dev::has_index_map<CL>() || vec_ok(L, C)) && (C <= dev::kScanBlockRow || (kRingServes && cooperative_launch_ok())) && !look_back_is_quicker(L, R, C);
  }
  // One scan of a size at which the ring has not got going: its tiles wait for a round's totals to be exchanged, k_scan's for
  // their neighbours only, and most of them are there at once.  us for two scans of rows, ring against k_scan with resident
  // blocks: 64 x 17000 23.6 / 14.4, 148 x 17000 27.1 / 18.6, 148 x 33000 36.1 / 33.3, 8 x 200000 24.7 / 18.4; 300 x 17000 equal
  // (600 tiles), 1000 x 17000 84 / 88.  One row: 300000 15.4 / 14.5, 500000 17.7 / 15.3, 2^20 23.1 / 17.6, 2^21 25.3 / 23.1,
  // 3 * 10^6 27.1 / 27.4 (184 tiles).  Element by element (rows without 128-bit accesses), where the ring takes more than a round:
  // 32 x 30001 23.9 / 18.6, 3 x 500001 24.0 / 22.2, 900001 23.0 / 21.0; 757761 (149 tiles of the ring) 19.5 / 20.5, 2^21 + 1 25.3 / 26.2,
  // 148 x 33001 36.5 / 47.1.  A staged gather below the scan: one row of few elements (30000: ticketed tiles 8.7, ring 12.4).
  // Few rows with a gather below the scan, which a block per row would leave to few SMs: one row of 6000 from 4 MB equal, of
  // 8000 9.2 / 7.2, of 16000 13.3 / 7.2 (two such scans 26.6 / 14.4).
  static bool look_back_is_quicker(const ClusterLaunch& L, int R, int C) {
    if constexpr (!kRingShape || dev::count_if<CL>(dev::is_scan_root) != 1) {
      return false;                                      // (k_scan takes one scan; several share the ring's walk)
    } else {
      const int64_t per_row = (C + kScanTile - 1) / kScanTile, tiles = R * per_row;
      if (C <= dev::kScanBlockRow) return dev::costly_members<CL>() > 0 && dev::scan_gathers<CL>() && C > dev::kScanGatherRow && tiles <= sm_count();
      if constexpr (dev::costly_members<CL>() > 0) return R == 1 && C <= dev::kScanFewElements;
      if constexpr (dev::scan_gathers<CL>()) return false;   // (with what reads the scan: smaller tiles, not measured)
      if (vec_ok(L, C)) return tiles <= 3 * sm_count() && per_row <= 160;
      return tiles <= sm_count() && per_row <= 64 && 8 * (int64_t)R * ring_tiles_per_row(R, C) > 9 * sm_count();
    }
  }
  // (a row of C elements may begin up to three words into its first 16-byte chunk)
  static int ring_tiles_per_row(int R, int C) {
    if constexpr (kRingShape) return (C + (R > 1 && C % 4 ? 3 : 0) + dev::RingTile<CL>::TILE - 1) / dev::RingTile<CL>::TILE;
    else return 0;
  }
  static int64_t scan_scratch_bytes(const ClusterLaunch& L, int R, int C) {
    if (use_ring(L, R, C)) {
      int per_row = ring_tiles_per_row(R, C);
      if constexpr (kRingShape) {
        if constexpr (dev::can_stage<CL>()) per_row = std::max(per_row, Launcher<dev::StagedScan<CL>>::ring_tiles_per_row(R, C));
      }
      return 16 + (per_row > 1 ? 2 * (int64_t)dev::count_if<CL>(dev::is_scan_root) * R * per_row * 8 : 0);
    }
    return 16 + (int64_t)R * ((C + kScanTile - 1) / kScanTile) * 8;
  }

  // WHOLE: the cluster whose costly members are staged first (this one is then what is left of it), or void.
  template <class WHOLE = void>
  static int launch_ring(const ClusterLaunch& L, dev::Args<N>& a, int R, int C, dev::StageArgs<WHOLE, N> whole = {}) {
    if constexpr (kRingShape) {
      constexpr int kForms = std::is_void<WHOLE>::value ? dev::ScanForms<CL>::value : 2;
      if constexpr ((kForms & 1) != 0) {
        if (C <= dev::kScanWarpRow) {
          const int warps = dev::kBlock / 32;
          dev::k_scan_rows<CL, 1, 4><<<(int)std::min<int64_t>((R + warps - 1) / warps, (int64_t)sm_count() * 8), dev::kBlock, 0, L.stream>>>(a);
        } else if (C <= dev::kScanBlockRow) {
          // (a thread's chunks are all under way together, those beyond the row's end for nothing: rows of 5000 in sixteen warps
          // of four chunks 19.5 us for 2000 of them, of eight 29.7; and a warp beyond the row's end takes another block's place: as
          // many warps as have chunks instead of sixteen, two scans of 4099 x 3001 45.1 -> 39.0 us, 8000 x 1200 66.9 -> 28.7, 2443 x 5825 53.3 ->
          // 45.1, 3000 x 9000 92.1 -> 71.5)
          const int chunks = C <= 4096 - 3 ? 2 : C <= 8192 - 3 ? 4 : 8;
          const int warps = (C + (R > 1 && C % 4 ? 3 : 0) + chunks * 128 - 1) / (chunks * 128);
          const int grid = (int)std::min<int64_t>(R, (int64_t)sm_count() * 16);
          if (chunks == 2) dev::k_scan_rows<CL, 16, 2><<<grid, warps * 32, 0, L.stream>>>(a);
          else if (chunks == 4) dev::k_scan_rows<CL, 16, 4><<<grid, warps * 32, 0, L.stream>>>(a);
          else dev::k_scan_rows<CL, 16, 8><<<grid, warps * 32, 0, L.stream>>>(a);
        }
      }
      if constexpr ((kForms & 2) != 0 && kRingServes) {
        if (C > dev::kScanBlockRow) {
          int per_row = ring_tiles_per_row(R, C);
          const int64_t tiles = (int64_t)R * per_row;
          if (tiles >= (int64_t(1) << 31)) return set_error(ACC_ERR_SHAPE, "too many rows to scan in one launch");
          if constexpr (std::is_void<WHOLE>::value && dev::can_stage<CL>()) {
            dev::Args<N> rest = a;
            for (int i = 0; i < N; ++i)
              if (dev::is_costly<CL>(i)) {
                rest.n[i].ptr = a.n[dev::stage_target<CL>(i)].ptr;
                rest.n[i].R = R;
                rest.n[i].C = C;
              }
            return Launcher<dev::StagedScan<CL>>::template launch_ring<CL>(L, rest, R, C, dev::StageArgs<CL, N>{a});
          } else {
            using K = dev::Ring<CL, dev::ring_resident<CL>()>;
            int n_tiles = (int)tiles;
            const void* kern = reinterpret_cast<const void*>(dev::k_scan_ring<CL, WHOLE>);
            static int granted[64];
            if (!opt_in_shared_memory(kern, K::SMEM, granted))
              return set_error(ACC_ERR_CUDA, "shared-memory opt-in failed: %s", cudaGetErrorString(cudaGetLastError()));
            // (blocks read one another's totals: all of them resident)
            void* params[] = {&a, &per_row, &n_tiles, &whole};
            cudaLaunchCooperativeKernel(kern, dim3((unsigned)std::min<int64_t>(tiles, std::min(sm_count(), dev::kRingMaxBlocks))), dim3(K::THREADS), params, K::SMEM, L.stream);
          }
        }
      }
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
      return ACC_OK;
    } else {
      return set_error(ACC_ERR_NO_KERNEL, "not a cluster of scans");
    }
  }

  // k_scan: tiles that look back one after the other, claimed from a ticket, or walked by blocks that are all resident.
  static int launch_look_back(const ClusterLaunch& L, dev::Args<N>& a, bool vec, int tiles_per_row, int64_t tiles, bool resident = false) {
    if constexpr (dev::count_if<CL>(dev::is_scan_root) == 1) {
      if (resident) {
        const void* kern = vec ? reinterpret_cast<const void*>(dev::k_scan<CL, true>) : reinterpret_cast<const void*>(dev::k_scan<CL, false>);
        static int fit_on[2][64];
        const int at_once = resident_grid(kern, kScanBlock, fit_on[vec ? 1 : 0]);
        if (at_once > 0) {
          int n_tiles = (int)tiles, yes = 1;
          void* params[] = {&a, &tiles_per_row, &n_tiles, &yes};
          cudaLaunchCooperativeKernel(kern, dim3((unsigned)std::min<int64_t>(tiles, at_once)), dim3(kScanBlock), params, 0, L.stream);
          const cudaError_t e = cudaGetLastError();
          if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
          return ACC_OK;
        }
      }
      const int grid = (int)std::min<int64_t>(tiles, (int64_t)sm_count() * (1536 / kScanBlock));
      if (vec) dev::k_scan<CL, true><<<grid, kScanBlock, 0, L.stream>>>(a, tiles_per_row, (int)tiles, 0);
      else dev::k_scan<CL, false><<<grid, kScanBlock, 0, L.stream>>>(a, tiles_per_row, (int)tiles, 0);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
      return ACC_OK;
    } else {
      return set_error(ACC_ERR_NO_KERNEL, "several scans walk together through the ring only");
    }
  }

  // Whether the gather below the scan runs as slab passes: decided by shapes alone, so that the scratch
  // layout (which is fixed before any pointer is known) and the launch agree.
  static constexpr bool kSlabShape = dev::slab_gather_eligible<CL>();
  static bool slab_shapes_ok(const ClusterLaunch& L, int R, int C) {
    if constexpr (kSlabShape) {
      const int src = CL::c.nodes[dev::the_gather<CL>()].in[1];
      const int64_t src_bytes = (int64_t)L.nodes[src].R * L.nodes[src].C * 4;
      return R == 1 && C >= dev::kSlabMinElements && C % 4 == 0 && src_bytes >= dev::kSlabMinSourceBytes && src_bytes <= dev::kSlabMaxSourceBytes;
    } else {
      return false;
    }
  }

  // The same for a cluster of element-wise roots only (k_stream_merge): every root a rank-1 array of the domain's length.
  static constexpr bool kStreamSlabShape = dev::slab_stream_eligible<CL>();
  static bool stream_slab_shapes_ok(const ClusterLaunch& L, int R, int C) {
    if constexpr (kStreamSlabShape) {
      const int src = CL::c.nodes[dev::the_gather<CL>()].in[1];
      const int64_t src_bytes = (int64_t)L.nodes[src].R * L.nodes[src].C * 4;
      for (int i = 0; i < N; ++i)
        if (dev::is_store_root(CL::c.nodes[i]) && (L.nodes[i].R != 1 || L.nodes[i].C != C)) return false;
      return R == 1 && C >= dev::kSlabMinElements && C % 4 == 0 && src_bytes >= dev::kSlabMinSourceBytes && src_bytes <= dev::kSlabMaxSourceBytes;
    } else {
      return false;
    }
  }
  // bytes of the group sizes and slab codes of the slab passes, which lie behind `base` bytes of other scratch
  static int64_t with_slab_area(int64_t base, int C) {
    const int64_t full = C / dev::kSlabWarpTile;
    return ((base + 15) & ~int64_t(15)) + full * 4 + full * 32 * 4;
  }

  // k_hist's scratch behind `words` of counters and accumulators: private overflow bins per CTA, then (from a multiple of 16
  // bytes) what the CTAs exchange.
  static int64_t hist_exchange_off(int64_t words, const dev::HistPlan& plan) { return (words + (int64_t)sm_count() * plan.overflow + 3) & ~int64_t(3); }

  static int64_t scratch_bytes(const ClusterLaunch& L) {
    int R, C;
    if (!domain(L, R, C)) return ACC_ERR_NO_KERNEL;
    if (use_tiles(L, R, C)) {
      const int blocks = (R + dev::kTile - 1) / dev::kTile;
      return (dev::tile_partials_off(blocks) + (int64_t)kRowFolds * blocks * R) * 4;
    }
    if (kHasScan) {
      if (slab_shapes_ok(L, R, C)) {                      // + group sizes and slab codes of the slab passes (slabgather.cuh)
        const int64_t bytes = 16 + (int64_t)R * ((C + kScanTile - 1) / kScanTile) * 8, full = C / dev::kSlabWarpTile;
        return ((bytes + 15) & ~int64_t(15)) + full * 4 + full * 32 * 4;
      }
      return scan_scratch_bytes(L, R, C);
    }
    if (kHasSegFold) return dev::seg_scratch_words(dev::count_if<CL>(dev::is_segfold_root), seg_grid(L)) * 4;
    if (kHasRowFold) return 0;
    int64_t words = dev::stream_acc64_off(kScalarFolds, sm_count() * 8);
    for (int i = 0; i < N; ++i)
      if (dev::is_f32_add_permute(CL::c.nodes[i])) words += 2 * (int64_t)L.nodes[i].R * L.nodes[i].C;
    dev::HistPlan plan;
    if (use_hist(L, R, C, plan)) words = hist_exchange_off(words, plan) + (int64_t)sm_count() * plan.exchange;
    if (stream_slab_shapes_ok(L, R, C)) return with_slab_area(words * 4, C);
    return words * 4;
  }

  // Counters, tickets, tile states and accumulators start from zero; what a kernel writes before it reads
  // (partial sums per tile, the codes and group sizes of the slab passes) need not be cleared, and lies last.
  static int64_t zeroed_bytes(const ClusterLaunch& L) {
    int R, C;
    if (!domain(L, R, C)) return 0;
    if (use_tiles(L, R, C)) return use_tile_rows(R) ? 0 : dev::tile_partials_off((R + dev::kTile - 1) / dev::kTile) * 4;
    if (kHasSegFold) return 0;
    if (kHasScan && slab_shapes_ok(L, R, C)) return ((16 + (int64_t)R * ((C + kScanTile - 1) / kScanTile) * 8) + 15) & ~int64_t(15);
    if (kHasScan && use_ring(L, R, C) && (scan_scratch_bytes(L, R, C) == 16 || C <= dev::kScanBlockRow)) return 0;
    if (stream_slab_shapes_ok(L, R, C)) return (((int64_t)dev::stream_acc64_off(kScalarFolds, sm_count() * 8) * 4) + 15) & ~int64_t(15);
    if (use_few(L, R, C)) return 0;
    dev::HistPlan plan;
    if (use_hist(L, R, C, plan)) return scratch_bytes(L) - (int64_t)sm_count() * plan.exchange * 4;   // (what is exchanged is written first)
    return scratch_bytes(L);
  }

  static void fill(const ClusterLaunch& L, dev::Args<N>& a, int R, int C) {
    for (int i = 0; i < N; ++i) a.n[i] = L.nodes[i];
    a.R = R;
    a.C = C;
    a.scratch = L.scratch;
    a.status = L.status;
    a.run_id = L.run_id;
    a.spin_limit = L.spin_limit;
    a.grid = sm_count() * 8;             // the partials' layout is sized for the largest grid
  }

  static int launch_hist(const ClusterLaunch& L, dev::Args<N>& a, int R, int C, bool vec);

  // clamped shifts served from halo tiles copied by cp.async.bulk.tensor (k_stencil)
  static constexpr bool kStencilShape = dev::stencil_eligible<CL>();

  // Returns ACC_OK after a launch, an error, or 1 when k_stream should run instead: no
  // 128-bit rows, an external of another shape, a shift by more than one, or a domain too
  // small to fill the machine with tiles.
  static int launch_stencil(const ClusterLaunch& L, dev::Args<N>& a, int R, int C, bool vec) {
    if constexpr (kStencilShape) {
      if (R < 1 || (int64_t)R * C < (int64_t)dev::kStRows * dev::kStCols * 64) return 1;
      constexpr int depth = dev::max_shift_depth<CL>();
      // (rows that do not start on 16 bytes are copied word by word, which pays where iterates are kept on chip: 4000 x 3999,
      // four iterations in twos 360 -> 141 us, one by one 204 -> 201 us, 1000 x 1001 one by one 27 -> 35 us)
      if (!vec && depth < 2) return 1;
      dev::StencilMaps maps;
      for (int i = 0; i < N; ++i) {
        const CNode& n = CL::c.nodes[i];
        if (n.member && n.kind == ACC_BACKPERMUTE && n.idxfn == ACC_IDX_SHIFT_CLAMP &&
            (L.nodes[i].ip0 < -1 || L.nodes[i].ip0 > 1 || L.nodes[i].ip1 < -1 || L.nodes[i].ip1 > 1))
          return 1;
        if (dev::is_staged_external<CL>(i)) {
          if (L.nodes[i].R != R || L.nodes[i].C != C) return 1;
          if (vec && !make_tensor_map_2d(&maps.m[dev::tile_slot<CL>(i)], L.nodes[i].ptr, R, C, dev::st_box_rows(depth), dev::kStBoxCols)) return 1;
        }
      }
      auto kern = dev::k_stencil<CL, true>;
      if constexpr (depth >= 2) {
        if (!vec) kern = dev::k_stencil<CL, false>;
      }
      // two stages of every external's box, one box per member kept on chip
      const size_t smem = (size_t)(dev::kStStages * dev::staged_externals<CL>() + dev::staged_members<CL>()) * dev::st_box_stride(depth) * 4 +
                          (vec ? 0 : (size_t)dev::kBlock / 32 * dev::kStCols * 4);
      static int granted[2][64];
      if (!opt_in_shared_memory(kern, smem, granted[vec ? 1 : 0]))
        return set_error(ACC_ERR_CUDA, "shared-memory opt-in failed: %s", cudaGetErrorString(cudaGetLastError()));
      const int64_t tiles = (int64_t)((C + dev::kStCols - 1) / dev::kStCols) * ((R + dev::kStRows - 1) / dev::kStRows);
      const int per_sm = std::max(1, std::min(3, (int)((size_t)220 * 1024 / (smem + 1024))));
      const int grid = (int)std::min<int64_t>(tiles, (int64_t)sm_count() * per_sm);
      kern<<<grid, dev::kBlock, smem, L.stream>>>(a, maps);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
      return ACC_OK;
    } else {
      return 1;
    }
  }

  // Tile pairs staged by tensor copies (k_tile_pair_tma): clusters whose roots are row folds, rows
  // 16-byte friendly.
  // Returns ACC_OK after a launch, an error, or 1 when k_tile_pair should run instead.
  static int launch_tiles_tma(const ClusterLaunch& L, dev::Args<N>& a, int n, bool vec) {
    if constexpr (dev::tile_tma_eligible<CL>()) {
      if (!cooperative_launch_ok()) return 1;
      // (word-by-word copies and the meeting at the end pay from about here on, for two arrays more than for one; us staged by threads
      // against copied, one array and two: 2561 rows 18.3 / 20.5 and 22.7 / 28.7, 2717 18.4 / 20.5 and 25.6 / 26.7, 2721 18.4 / 20.5 and
      // 25.7 / 26.6, 2749 18.4 / 18.5 and 25.5 / 22.5, 2901 20.4 / 20.5 and 27.8 / 28.9, 3001 20.5 / 18.5 and 28.7 / 24.6, 3101 20.5 / 22.5
      // and 28.7 / 30.7, 3501 23.9 / 24.0 and 42.7 / 39.1)
      if (!vec && n < 2720) return 1;
      dev::TileMaps maps;
      for (int i = 0; i < N; ++i)
        if (vec && dev::is_staged_external<CL>(i) &&
            !make_tensor_map_2d(&maps.m[dev::tile_slot<CL>(i)], L.nodes[i].ptr, n, n, dev::kTile, dev::kTile))
          return 1;
      auto kern = vec ? dev::k_tile_pair_tma<CL, true> : dev::k_tile_pair_tma<CL, false>;
      const int threads = vec ? dev::tp_threads<true>() : dev::tp_threads<false>();
      constexpr int E = dev::staged_externals<CL>();
      const size_t smem = (size_t)dev::tp_stages<E>() * E * dev::kTpSlotWords * 4 + 128;   // + room to align the copies
      static int fit_on_[2][64];                               // blocks of this kernel per SM, + 1, by device (asked once each)
      int* fit_on = fit_on_[vec ? 1 : 0];
      int device = 0;
      if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) { cudaGetLastError(); return 1; }
      int per_sm = fit_on[device] - 1;
      if (per_sm < 0) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
          return set_error(ACC_ERR_CUDA, "shared-memory opt-in failed: %s", cudaGetErrorString(cudaGetLastError()));
        int fit = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, threads, smem) != cudaSuccess) {
          cudaGetLastError();
          fit = 0;
        }
        per_sm = fit;
        fit_on[device] = fit + 1;
      }
      if (per_sm < 1) return 1;
      const int64_t blocks = (n + dev::kTile - 1) / dev::kTile;
      const int64_t pairs = blocks * (blocks + 1) / 2;
      const int grid = (int)std::min<int64_t>(pairs, (int64_t)sm_count() * per_sm);
      void* params[] = {&a, &maps};                        // all blocks resident: they meet at a counter after their walk
      cudaLaunchCooperativeKernel(reinterpret_cast<void*>(kern), dim3(grid), dim3(threads), params, smem, L.stream);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
      return ACC_OK;
    } else {
      return 1;
    }
  }

  // Whether the scatter's bins go on chip: they must fit (see hist_plan) and there must be
  // enough elements per bin to repay clearing and flushing them.
  static bool use_hist(const ClusterLaunch& L, int R, int C, dev::HistPlan& plan) {
    if constexpr (kHistShape) {
      constexpr int P = dev::the_f32_add_permute<CL>();
      const int64_t bins = (int64_t)L.nodes[P].R * L.nodes[P].C;
      if (bins <= 0 || (int64_t)R * C < 8 * bins) return false;
      return dev::hist_plan(bins, sm_count(), plan);
    } else {
      return false;
    }
  }

  static int launch(const ClusterLaunch& L) {
    int R, C;
    if (!domain(L, R, C)) return set_error(ACC_ERR_NO_KERNEL, "cluster without a root");
    if (!domains_agree(L, R, C)) return set_error(ACC_ERR_SHAPE, "members of one cluster iterate over different sizes");
    const bool vec = vec_ok(L, C);
    // scatters on integers work in place on a copy of the defaults
    for (int i = 0; i < N; ++i) {
      const CNode& n = CL::c.nodes[i];
      if (dev::is_permute_root(n) && !dev::is_f32_add_permute(n)) {
        const size_t bytes = (size_t)L.nodes[i].R * L.nodes[i].C * 4;
        if (bytes && cudaMemcpyAsync(const_cast<void*>(L.nodes[i].ptr), L.nodes[n.in[0]].ptr, bytes,
                                     cudaMemcpyDeviceToDevice, L.stream) != cudaSuccess)
          return set_error(ACC_ERR_CUDA, "copy of scatter defaults failed: %s", cudaGetErrorString(cudaGetLastError()));
      }
    }
    dev::Args<N> a;
    fill(L, a, R, C);
    if constexpr (dev::rowfold_then_eligible<CL>()) {
      // row folds consumed by element-wise members: the block walks the folds' source rows
      int src = -1;
      for (int i = 0; i < N && src < 0; ++i)
        if (dev::is_inner_row_fold(CL::c.nodes[i])) src = CL::c.nodes[i].in[0];
      bool same = true;                                  // every fold reduces an array of one shape
      for (int i = 0; i < N; ++i)
        if (dev::is_inner_row_fold(CL::c.nodes[i]))
          same = same && L.nodes[CL::c.nodes[i].in[0]].R == L.nodes[src].R && L.nodes[CL::c.nodes[i].in[0]].C == L.nodes[src].C;
      if (same && L.nodes[src].C >= 64) {                // short rows are as well off pulled through
        a.R = L.nodes[src].R;
        a.C = L.nodes[src].C;
        if (a.R == 0) return ACC_OK;
        const int grid = std::min(a.R, sm_count() * 16);
        const bool v4 = vec_ok(L, a.C);
        if (v4) dev::k_rowfold_then<CL, true><<<grid, dev::kBlock, 0, L.stream>>>(a);
        else dev::k_rowfold_then<CL, false><<<grid, dev::kBlock, 0, L.stream>>>(a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
        return ACC_OK;
      }
    }
    if (use_tiles(L, R, C)) {
      if constexpr (kTileShape) {
        if constexpr (kTileRowsShape) {
          if (use_tile_rows(R)) {
            auto kern = vec ? dev::k_tile_rows<CL, true> : dev::k_tile_rows<CL, false>;
            const size_t smem = (size_t)dev::staged_externals<CL>() * 2 * dev::kTileWords * 4;
            static int granted[2][64];
            if (!opt_in_shared_memory(kern, smem, granted[vec ? 1 : 0]))
              return set_error(ACC_ERR_CUDA, "shared-memory opt-in failed: %s", cudaGetErrorString(cudaGetLastError()));
            kern<<<(R + dev::kTile - 1) / dev::kTile * dev::kTrBlocks, dev::kBlock, smem, L.stream>>>(a);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
            return ACC_OK;
          }
        }
        const int rc = launch_tiles_tma(L, a, R, vec);
        if (rc != 1) return rc;                          // 1 = no tensor copies here: the threads stage the tiles
        auto kern = vec ? dev::k_tile_pair<CL, true> : dev::k_tile_pair<CL, false>;
        const size_t smem = (size_t)dev::staged_externals<CL>() * 2 * dev::kTileWords * 4;
        static int granted[2][64];
        if (!opt_in_shared_memory(kern, smem, granted[vec ? 1 : 0]))
          return set_error(ACC_ERR_CUDA, "shared-memory opt-in failed: %s", cudaGetErrorString(cudaGetLastError()));
        const int blocks = (R + dev::kTile - 1) / dev::kTile;
        kern<<<blocks * (blocks + 1) / 2, dev::kBlock, smem, L.stream>>>(a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
      }
      return ACC_OK;
    }
    if constexpr (kHasSegFold) {
      if constexpr (dev::segfold_eligible<CL>()) {
        if (C == 0) return ACC_OK;
        const int grid = seg_grid(L);
        // (chunks of four start on 16 bytes whatever the length; behind an index map they need 128-bit rows)
        const int src = CL::c.nodes[dev::first_segfold<CL>()].in[0];
        const int run = dev::seg_run((int64_t)L.nodes[src].R * L.nodes[src].C, sm_count());
        if (!dev::has_index_map<CL>() || seg_vec_ok(L)) {
          constexpr size_t smem = dev::seg_landing_bytes<CL, true>();
          static int granted[64];
          if (!opt_in_shared_memory(dev::k_segfold<CL, true>, smem, granted))
            return set_error(ACC_ERR_CUDA, "shared-memory opt-in failed: %s", cudaGetErrorString(cudaGetLastError()));
          dev::k_segfold<CL, true><<<grid, dev::kBlock, smem, L.stream>>>(a, run);
        } else dev::k_segfold<CL, false><<<grid, dev::kBlock, 0, L.stream>>>(a, run);
        dev::k_segfold_across<CL><<<(grid + dev::kBlock / 32 - 1) / (dev::kBlock / 32), dev::kBlock, 0, L.stream>>>(a, grid);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
        return ACC_OK;
      } else {
        return set_error(ACC_ERR_NO_KERNEL, "segmented folds share a kernel only with each other and over one offsets array");
      }
    }
    if constexpr (kStencilShape) {
      const int rc = launch_stencil(L, a, R, C, vec);
      if (rc != 1) return rc;                            // 1 = shapes or shifts it does not cover: stream instead
    }
    if constexpr (kHasScan) {
      if ((int64_t)R * C == 0) return ACC_OK;
      const int per_row = (C + kScanTile - 1) / kScanTile;
      const int64_t tiles = (int64_t)R * per_row;
      if (tiles >= (int64_t(1) << 31)) return set_error(ACC_ERR_SHAPE, "too many rows to scan in one launch");
      const int grid = (int)std::min<int64_t>(tiles, (int64_t)sm_count() * (1536 / kScanBlock));
      if constexpr (kSlabShape) {
        if (vec && slab_shapes_ok(L, R, C)) {
          // partition the indices by slab, gather slab by slab from L2, merge and scan (slabgather.cuh)
          const int src = CL::c.nodes[dev::the_gather<CL>()].in[1];
          const int64_t n_src = (int64_t)L.nodes[src].R * L.nodes[src].C;
          const uint32_t mul = (uint32_t)(((uint64_t)dev::kSlabs << 32) / (uint64_t)n_src);
          const int full = C / dev::kSlabWarpTile;
          const int64_t states = ((16 + tiles * 8) + 15) & ~int64_t(15);
          uint32_t* counts = L.scratch + states / 4;
          uint32_t* codes = counts + full;
          const int warps = dev::kBlock / 32;
          const int pgrid = (int)std::min<int64_t>((full + warps - 1) / warps, (int64_t)sm_count() * 4);
          const int ggrid = (int)std::min<int64_t>((full + warps - 1) / warps, (int64_t)sm_count() * 8);
          // (word 1 of the scratch, cleared with the tile states: how many sampled warp tiles have local indices)
          const int probes = (int)std::min<int64_t>((full + warps - 1) / warps, (int64_t)sm_count());
          const dev::SlabIn slab{codes, counts, full, L.scratch + 1, (uint32_t)(probes * warps)};
          dev::k_slab_probe<CL><<<probes, dev::kBlock, 0, L.stream>>>(a, full, L.scratch + 1);
          dev::k_slab_partition<CL><<<pgrid, dev::kBlock, 0, L.stream>>>(a, codes, counts, full, mul, slab);
          for (int k = 0; k < dev::kSlabs; ++k) dev::k_slab_gather<CL><<<ggrid, dev::kBlock, 0, L.stream>>>(a, counts, full, (uint32_t)k, slab);
          {
            int per_row_arg = per_row, tiles_arg = (int)tiles;
            dev::SlabIn slab_arg = slab;
            void* params[] = {&a, &per_row_arg, &tiles_arg, &slab_arg};
            static int fit_on[64];
            const int resident = resident_grid(reinterpret_cast<const void*>(dev::k_scan_merge_pipelined<CL>), kScanBlock + 32, fit_on);
            if (resident > 0)
              cudaLaunchCooperativeKernel(reinterpret_cast<void*>(dev::k_scan_merge_pipelined<CL>), dim3((unsigned)std::min<int64_t>(tiles, resident)),
                                          dim3(kScanBlock + 32), params, 0, L.stream);
            else
              dev::k_scan_merge<CL><<<grid, kScanBlock, 0, L.stream>>>(a, per_row, (int)tiles, slab);
          }
          L.extra_launches += 2 + dev::kSlabs;
          const cudaError_t e = cudaGetLastError();
          if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
          return ACC_OK;
        }
      }
      if (use_ring(L, R, C)) return launch_ring(L, a, R, C);
      // (a gather's latency covers the ticket's: sums over two gathers of 2^24 elements 222 us with tickets, 330 without)
      return launch_look_back(L, a, vec, per_row, tiles, dev::scan_gathers<CL>() ? C <= dev::kScanBlockRow && tiles <= sm_count() : tiles <= 3 * sm_count());
    } else if constexpr (kHasRowFold) {
      if (R == 0) return ACC_OK;
      const int grid = std::min(R, sm_count() * 16);
      if (vec) dev::k_rowfold<CL, true><<<grid, dev::kBlock, 0, L.stream>>>(a);
      else dev::k_rowfold<CL, false><<<grid, dev::kBlock, 0, L.stream>>>(a);
    } else {
      if constexpr (kHistShape) {
        const int rc = launch_hist(L, a, R, C, stream_vec_ok(L, vec));
        if (rc != 1) return rc;                        // 1 = not worth it or does not fit: stream instead
      }
      if constexpr (kStreamSlabShape) {
        if (vec && stream_slab_shapes_ok(L, R, C)) {
          // the gather's source does not fit L2: partition the indices by slab, gather slab by slab, store from the merged values
          const int src = CL::c.nodes[dev::the_gather<CL>()].in[1];
          const int64_t n_src = (int64_t)L.nodes[src].R * L.nodes[src].C;
          const uint32_t mul = (uint32_t)(((uint64_t)dev::kSlabs << 32) / (uint64_t)n_src);
          const int full = C / dev::kSlabWarpTile;
          const int64_t base = (((int64_t)dev::stream_acc64_off(kScalarFolds, sm_count() * 8) * 4) + 15) & ~int64_t(15);
          uint32_t* counts = L.scratch + base / 4;
          uint32_t* codes = counts + full;
          const int warps = dev::kBlock / 32;
          const int pgrid = (int)std::min<int64_t>((full + warps - 1) / warps, (int64_t)sm_count() * 4);
          const int ggrid = (int)std::min<int64_t>((full + warps - 1) / warps, (int64_t)sm_count() * 8);
          const int probes = (int)std::min<int64_t>((full + warps - 1) / warps, (int64_t)sm_count());
          const dev::SlabIn slab{codes, counts, full, L.scratch + 1, (uint32_t)(probes * warps)};
          dev::k_slab_probe<CL><<<probes, dev::kBlock, 0, L.stream>>>(a, full, L.scratch + 1);
          dev::k_slab_partition<CL><<<pgrid, dev::kBlock, 0, L.stream>>>(a, codes, counts, full, mul, slab);
          for (int k = 0; k < dev::kSlabs; ++k) dev::k_slab_gather<CL><<<ggrid, dev::kBlock, 0, L.stream>>>(a, counts, full, (uint32_t)k, slab);
          dev::k_stream_merge<CL><<<pgrid, dev::kBlock, 0, L.stream>>>(a, slab);
          L.extra_launches += 2 + dev::kSlabs;
          const cudaError_t e = cudaGetLastError();
          if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
          return ACC_OK;
        }
      }
      if constexpr (kFewShape) {
        if (use_few(L, R, C)) {
          if (stream_vec_ok(L, vec)) dev::k_stream_few<CL, true><<<dev::kFewBlocks, dev::kFewThreads, 0, L.stream>>>(a);
          else dev::k_stream_few<CL, false><<<dev::kFewBlocks, dev::kFewThreads, 0, L.stream>>>(a);
          const cudaError_t e = cudaGetLastError();
          if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
          return ACC_OK;
        }
      }
      // an empty domain still runs one block: a scatter must copy its defaults out
      const bool v4 = stream_vec_ok(L, vec);
      const int grid = stream_grid(R, C, v4);
      if (v4) dev::k_stream<CL, true><<<grid, dev::kBlock, 0, L.stream>>>(a);
      else dev::k_stream<CL, false><<<grid, dev::kBlock, 0, L.stream>>>(a);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
    return ACC_OK;
  }
};

// On-chip histogram path.  Returns ACC_OK after a launch, an error, or 1 when the generic
// streaming kernel should run instead.
template <class CL>
int Launcher<CL>::launch_hist(const ClusterLaunch& L, dev::Args<N>& a, int R, int C, bool vec) {
  if constexpr (kHistShape) {
    dev::HistPlan plan;
    if (!use_hist(L, R, C, plan)) return 1;
    constexpr int P = dev::the_f32_add_permute<CL>();
    const int64_t bins = (int64_t)L.nodes[P].R * L.nodes[P].C;
    auto kern = vec ? dev::k_hist<CL, true> : dev::k_hist<CL, false>;
    const size_t smem = std::max<size_t>(((size_t)plan.per_cta + 3) / 4 * 16, (size_t)(sm_count() + dev::kHistBlock / 2) * 8);
    static int granted[2][64];
    if (!opt_in_shared_memory(kern, smem, granted[vec ? 1 : 0]))
      return set_error(ACC_ERR_CUDA, "shared-memory opt-in failed: %s", cudaGetErrorString(cudaGetLastError()));
    const int64_t chunks = (int64_t)R * C / (vec ? 4 : 1);
    const int64_t per_team = (int64_t)dev::kHistBlock * dev::kHistUnroll;
    const int64_t want = (chunks + per_team - 1) / per_team;
    const int teams = (int)std::max<int64_t>(1, std::min<int64_t>(want, sm_count() / plan.group));
    const int grid = teams * plan.group;                  // one CTA per SM: all of them are resident together
    plan.polls = dev::hist_polls((int64_t)R * C, teams);
    int* overflow = reinterpret_cast<int*>(L.scratch + dev::stream_acc64_off(kScalarFolds, a.grid) + 2 * bins);
    int* exchange = reinterpret_cast<int*>(L.scratch + hist_exchange_off(dev::stream_acc64_off(kScalarFolds, a.grid) + 2 * bins, plan));
    if (plan.exchange && cooperative_launch_ok()) {
      void* params[] = {&a, &plan, &overflow, &exchange};
      cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kern), dim3(grid), dim3(dev::kHistBlock), params, smem, L.stream);
    } else {
      plan.exchange = 0;
      kern<<<grid, dev::kHistBlock, smem, L.stream>>>(a, plan, overflow, exchange);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
    return ACC_OK;
  } else {
    return 1;
  }
}

// A cluster whose accumulating roots no single skeleton walks together (two scans; a scan beside a
// fold or a scatter; row folds beside a scatter) runs as several passes over the same description.
// Each pass keeps one group of those roots and treats the others as absent; only the first pass writes
// the element-wise roots.  Producers that the groups share are evaluated again in every pass, from
// the cluster's inputs: nothing beyond the cluster's own manifest arrays reaches memory.
constexpr int kMaxPasses = 6;
struct PassPlan {
  int n = 0;
  uint64_t keep[kMaxPasses] = {};     // bit i: accumulating root i runs in this pass
};

constexpr bool is_accumulating_root(const CNode& n) {
  return dev::is_fold_root(n) || dev::is_scan_root(n) || dev::is_permute_root(n);
}

// The scan whose values element-wise member i consumes inside the cluster, -1 if none.
constexpr int scan_needed_by(const CCluster& c, int i) {
  for (int s = 0; s < c.n; ++s)
    if (dev::is_scan_root(c.nodes[s]) && dev::needs_scan(c, i, s)) return s;
  return -1;
}

constexpr CNode unread_array(const CNode& n) {
  return CNode{ACC_INPUT, n.dtype, n.rank, 0, 0, 0, 0, {-1, -1, -1, -1, -1, -1}, false, true};
}

// The description of one pass: the accumulating roots in `keep` stay; element-wise roots that consume a
// scan are written by that scan's pass, the other element-wise roots by the first pass; members that no
// root of the pass reaches any more, and the roots of other passes, become arrays nobody reads.
constexpr CCluster pass_cluster(CCluster c, uint64_t keep, bool first) {
  const CCluster whole = c;
  for (int i = 0; i < c.n; ++i) {
    if (is_accumulating_root(whole.nodes[i]) && !((keep >> i) & 1)) {
      c.nodes[i] = unread_array(whole.nodes[i]);
    } else if (dev::is_store_root(whole.nodes[i])) {
      const int needs = scan_needed_by(whole, i);
      if (needs >= 0 ? ((keep >> needs) & 1) == 0 : !first) c.nodes[i].manifest = false;
    }
  }
  bool live[kMaxCluster] = {};
  for (int i = c.n - 1; i >= 0; --i) {
    const CNode& n = c.nodes[i];
    if (!n.member) continue;
    if (is_accumulating_root(n) || dev::is_store_root(n) || dev::is_segfold_root(n)) live[i] = true;
    if (live[i])
      for (int k = 0; k < n.nin; ++k) live[n.in[k]] = true;
  }
  for (int i = 0; i < c.n; ++i)
    if (c.nodes[i].member && !live[i]) c.nodes[i] = unread_array(c.nodes[i]);
  return c;
}

constexpr uint64_t scans_of_kind(const CCluster& c, int kind) {
  uint64_t m = 0;
  for (int i = 0; i < c.n; ++i)
    if (dev::is_scan_root(c.nodes[i]) && c.nodes[i].kind == kind) m |= 1ull << i;
  return m;
}
// Whether the scans of one direction can share a walk: as one pass they must be something k_scan_ring serves, whatever
// the shapes.  (Each array is then read once for all of them.)
template <class CL, int KIND>
struct ScansTogether {
  static constexpr CCluster c = pass_cluster(CL::c, scans_of_kind(CL::c, KIND), true);
};
template <class CL, int KIND> constexpr bool scans_share_a_pass() {
  if constexpr (scans_of_kind(CL::c, KIND) == 0) return false;
  else return dev::ring_serves<ScansTogether<CL, KIND>>() && !dev::has_index_map<ScansTogether<CL, KIND>>();
}

// TOGETHER: the scans of one direction share a pass where they can.
template <class CL, bool TOGETHER> constexpr PassPlan pass_plan() {
  PassPlan p;
  uint64_t folds = 0, permutes = 0;
  for (int kind : {(int)ACC_SCANL, (int)ACC_SCANR}) {
    const uint64_t scans = scans_of_kind(CL::c, kind);
    const bool together = TOGETHER && (kind == ACC_SCANL ? scans_share_a_pass<CL, ACC_SCANL>() : scans_share_a_pass<CL, ACC_SCANR>());
    if (scans && together) p.keep[p.n++] = scans;                   // one walk for all scans of a direction
    else
      for (int i = 0; i < CL::c.n; ++i)
        if ((scans >> i) & 1) p.keep[p.n++] = 1ull << i;             // a scan walks alone
  }
  for (int i = 0; i < CL::c.n; ++i) {
    const CNode& n = CL::c.nodes[i];
    if (dev::is_fold_root(n)) folds |= 1ull << i;
    else if (dev::is_permute_root(n)) permutes |= 1ull << i;
  }
  // whole-array folds and scatters share the streaming kernel; row folds have a kernel of their own
  const bool together = dev::domain_rank<CL>() <= 1 || !folds || !permutes;
  if (together) {
    if (p.n == 0 || (folds | permutes)) p.keep[p.n++] = folds | permutes;
  } else {
    p.keep[p.n++] = folds;
    p.keep[p.n++] = permutes;
  }
  return p;
}

// How many of the scans, each in a pass of its own, gather in a way that slab passes can serve (slabgather.cuh).
template <class CL, int P>
struct SinglePass {
  static constexpr CCluster c = pass_cluster(CL::c, pass_plan<CL, false>().keep[P], P == 0);
};
template <class CL, int P = 0> constexpr int slab_passes() {
  if constexpr (P < pass_plan<CL, false>().n) return (dev::slab_gather_eligible<SinglePass<CL, P>>() ? 1 : 0) + slab_passes<CL, P + 1>();
  else return 0;
}

template <class CL, bool TOGETHER, int P>
struct PassOf {
  static constexpr int kScanForms = pass_plan<CL, false>().n == pass_plan<CL, true>().n ? 3 : TOGETHER ? 2 : slab_passes<CL>() == 1 ? 3 : 1;
  static constexpr CCluster c = pass_cluster(CL::c, pass_plan<CL, TOGETHER>().keep[P], P == 0);
};

template <class CL>
struct Passes {
  static constexpr int kSingly = pass_plan<CL, false>().n, kTogether = pass_plan<CL, true>().n;

  // Scans share a pass where they go through the ring (long rows); k_scan_rows keeps a row's operands in registers and
  // takes one scan at a time.  A scan whose gather runs as slab passes keeps a pass of its own, for a shared walk gathers
  // from DRAM (2^26 indices into 256 MB beside a running sum: 890 us apart, 1354 shared); two such scans over one gather
  // are no slower shared (1341 against 1347 us, with the sum 1505 against 1621).
  static bool together(const ClusterLaunch& L) {
    if constexpr (kSingly == kTogether) return false;
    else {
      int R, C;
      return Launcher<CL>::domain(L, R, C) && C > dev::kScanBlockRow && cooperative_launch_ok() && !(slab_passes<CL>() == 1 && slab_shapes<0>(L, R, C));
    }
  }
  template <int P> static bool slab_shapes(const ClusterLaunch& L, int R, int C) {
    if constexpr (P < kSingly) return Launcher<PassOf<CL, false, P>>::slab_shapes_ok(L, R, C) || slab_shapes<P + 1>(L, R, C);
    else return false;
  }

  template <bool T, int P>
  static int64_t scratch_from(const ClusterLaunch& L) {
    if constexpr (P < pass_plan<CL, T>().n) {
      const int64_t here = Launcher<PassOf<CL, T, P>>::scratch_bytes(L);
      if (here < 0) return here;
      const int64_t rest = scratch_from<T, P + 1>(L);
      return rest < 0 ? rest : ((here + 255) & ~int64_t(255)) + rest;
    } else {
      return 0;
    }
  }
  template <bool T> static int64_t all_scratch(const ClusterLaunch& L) {
    if constexpr (pass_plan<CL, T>().n <= 1) return Launcher<CL>::scratch_bytes(L);
    else return scratch_from<T, 0>(L);
  }
  static int64_t scratch_bytes(const ClusterLaunch& L) {
    if constexpr (kSingly != kTogether) {
      if (together(L)) return all_scratch<true>(L);
    }
    return all_scratch<false>(L);
  }
  static int64_t zeroed_bytes(const ClusterLaunch& L) {
    if constexpr (kSingly <= 1) return Launcher<CL>::zeroed_bytes(L);
    else return scratch_bytes(L);                     // the passes' regions follow one another: all of it
  }

  template <bool T, int P>
  static int launch_from(ClusterLaunch& L) {
    if constexpr (P < pass_plan<CL, T>().n) {
      const int64_t here = Launcher<PassOf<CL, T, P>>::scratch_bytes(L);
      if (here < 0) return (int)here;
      const int rc = Launcher<PassOf<CL, T, P>>::launch(L);
      if (rc != ACC_OK) return rc;
      L.scratch += ((here + 255) & ~int64_t(255)) / 4;
      return launch_from<T, P + 1>(L);
    } else {
      return ACC_OK;
    }
  }
  template <bool T> static int launch_all(const ClusterLaunch& L) {
    if constexpr (pass_plan<CL, T>().n <= 1) {
      return Launcher<CL>::launch(L);
    } else {
      ClusterLaunch pass = L;
      pass.extra_launches = 0;                        // (L's own are counted already)
      const int rc = launch_from<T, 0>(pass);
      L.extra_launches += pass.extra_launches;
      return rc;
    }
  }
  static int launch(const ClusterLaunch& L) {
    if constexpr (kSingly != kTogether) {
      if (together(L)) {
        L.extra_launches += kTogether - kSingly;      // (the entry counts a pass per scan)
        return launch_all<true>(L);
      }
    }
    return launch_all<false>(L);
  }
};

template <class CL>
struct Registrar {
  explicit Registrar(const char* name) {
    // (a cluster of segmented folds is a walk over the elements and a small second launch for the segments that
    // cross its blocks)
    register_kernel(KernelEntry{signature(CL::c), name, &Passes<CL>::scratch_bytes, &Passes<CL>::zeroed_bytes, &Passes<CL>::launch,
                                Passes<CL>::kSingly > 1 ? Passes<CL>::kSingly : (dev::count_if<CL>(dev::is_segfold_root) > 0 ? 2 : 1)});
  }
};

// A file of many clusters is compiled in ACC_PARTS parts, each of which registers every ACC_PARTS-th cluster (the build sets
// both; one part where they are not set).
#ifndef ACC_PARTS
#define ACC_PARTS 1
#define ACC_PART 0
#endif
template <class CL, bool HERE> struct PartRegistrar : Registrar<CL> { using Registrar<CL>::Registrar; };
template <class CL> struct PartRegistrar<CL, false> { explicit PartRegistrar(const char*) {} };

#define ACC_CAT2(a, b) a##b
#define ACC_CAT(a, b) ACC_CAT2(a, b)
// Instantiates the kernels of cluster MASK of program PROG and registers them under NAME.
#define ACC_CLUSTER(PROG, MASK, NAME)                                              \
  struct ACC_CAT(Cl_, NAME) { static constexpr CCluster c = extract(PROG, MASK); }; \
  static PartRegistrar<ACC_CAT(Cl_, NAME), __COUNTER__ % ACC_PARTS == ACC_PART> ACC_CAT(reg_, NAME)(#NAME);

}  // namespace acc
