// k_scan_ring and k_scan_rows: scans along the innermost extent, with what reads them and what they are computed from.
//
// k_scan_ring.  A scan reads and writes every element once, so it should run at the rate of a copy; what kept the
// look-back scan of skeletons.cuh at half of that is that a block's loads, its scan, its look-back and its stores ran
// one after the other.  Here they overlap:
//
//   * one block per SM walks tiles b, b + G, b + 2G, ... of the array (a "round" is one such step of all G blocks).  Copy
//     warps keep the block's next tiles coming into rings of shared-memory stages (cp.async.bulk, one copy per array and
//     tile), results leave by bulk copies from the stages: no load or store of array data waits in a register;
//   * reducing warps visit a tile first and post the totals of its parts;
//   * look-back warps, one per round in flight, need no chain of look-backs: a tile's predecessors in its round are the
//     other blocks' tiles, so a look-back warp posts its tile's total, reads the totals of all G tiles of the round at
//     once and adds those before its own to the total of the earlier rounds, which it carries along: one exchange
//     through L2, whatever the distance, and the same order of additions in every run.  (In a long walk the first
//     block's look-back warps do this for all tiles of the round, and the others read what they post: 148 blocks that
//     poll 148 words each cost as much as they gained, 286 + 266 against 230 + 170 us for the passes below);
//   * scanning warps, two groups in turn, visit the tile again when the total of everything before it is known: they
//     scan it, evaluate what reads the scan and hand the results to bulk copies.
//
// Between a tile's first visit and its second lies the slowest copy of its round and an exchange: 10 us and more where
// memory is busy (copies land 2 to 6 us after they are asked for; a load of the posted totals queues behind its own SM's
// copies).  Held in shared memory for that long, the tiles in waiting fill the ring and the walk runs at 3.9 TB/s.  So the
// first visit has a ring of its own, runs up to a dozen rounds ahead, and leaves its tiles in L2, from where the second
// visit gets them again.  (RESIDENT: one ring serves both visits, where a cluster has too many arrays for two.)
//
// Measured on 2^26 floats, two arrays read and two written per pass: two sums in one walk 208 us, one maximum 171 us =
// 6.3 TB/s (a scan to a pass, tiles of 16384 elements with look-back: three passes of 218 us).
//
// Rows need no alignment: a tile is a 16-byte aligned range of the flat array, clipped to its row; chunks of four that
// straddle a row's ends are masked, and stored element by element.  Arrays that the cluster reads at its own index come
// through the ring, anything else (gather sources, arrays behind index maps) is read from global memory.
//
// A gather below a scan would be evaluated in both visits, and its reads want room in L1 to land in (a line each), which
// the ring takes: 5 * 10^6 gathers from 20 MB took 53 us inside the ring, 40 us with a ring of half the size.  So before
// the walk the whole block stages the gathered values of its own tiles in one of the cluster's output arrays
// (stage_costly): 16-byte asynchronous copies around each wanted word land in the ring's shared memory, past L1, and the
// ring then reads the array of values like any other (2 * 10^7 gathers and their scan: 171 us, with plain loads 265 us).
//
// Several scans of one direction share the walk (each array is read once for all of them).
//
// k_scan_rows: rows of up to 16384 elements, by a warp or by a block each, without shared-memory stages.
//
// Waits: every mbarrier wait is bounded (wait_phase), a look-back warp gives up after spin_limit polls; either raises the
// time-out status.  The copy warps wait (bounded) for copies in flight before they leave.
#pragma once
#include "skeletons.cuh"
#include "tile.cuh"

namespace acc {
namespace dev {

// ---- index kinds: four (one) consecutive elements whose arrays lie in a ring stage -----------------
struct IxRg  { int r, c; const uint32_t* stage; int at; };     // `at`: word offset of element (r, c) in a slot of the stage
struct IxRg1 { int r, c; const uint32_t* stage; int at; };
template <> struct width_of<IxRg1> { static constexpr int value = 1; };
__device__ __forceinline__ Ix lane(const IxRg& i, int j) { return Ix{i.r, i.c + j}; }
__device__ __forceinline__ Ix lane(const IxRg1& i, int) { return Ix{i.r, i.c}; }
template <int F, int P0 = kRunTime, int P1 = kRunTime>
__device__ __forceinline__ auto map_index(const IxRg& i, const NodeArg& self, const NodeArg& src) {
  if constexpr (F == ACC_IDX_IDENTITY) return i;
  else return map_index<F, P0, P1>(Ix4{i.r, i.c}, self, src);
}
template <int F, int P0 = kRunTime, int P1 = kRunTime>
__device__ __forceinline__ auto map_index(const IxRg1& i, const NodeArg& self, const NodeArg& src) {
  if constexpr (F == ACC_IDX_IDENTITY) return i;
  else return map_index<F, P0, P1>(Ix{i.r, i.c}, self, src);
}
// the same index with the values of the cluster's scans there
template <class B, int K> struct IxScN : B { val_of<B> sv[K]; };
template <class B, int K> struct width_of<IxScN<B, K>> { static constexpr int value = width_of<B>::value; };

// ---- compile-time layout ----------------------------------------------------------------------------
// Whether member i evaluated at a chunk reads node `leaf` at that same chunk (scans are where such a path ends: what
// lies below one is read by the scan's own operand).
constexpr bool reads_at_index(const CCluster& c, int i, int leaf) {
  if (i == leaf) return true;
  const CNode& n = c.nodes[i];
  if (!n.member) return false;
  int slots = 0;
  if (n.kind == ACC_MAP || n.kind == ACC_ZIPWITH) slots = n.narr;
  else if (n.kind == ACC_GATHER) slots = 1;                        // (its index operand)
  else if (n.kind == ACC_BACKPERMUTE && n.idxfn == ACC_IDX_IDENTITY) slots = 1;
  for (int k = 0; k < slots; ++k)
    if (reads_at_index(c, n.in[k], leaf)) return true;
  return false;
}
template <class CL> constexpr int scan_ord(int i) { return count_if<CL>(is_scan_root, i); }
// costly members that a scan's operand reads at its own index: staged (evaluated once, by stage_costly)
template <class CL> constexpr bool is_costly(int i) {
  const CNode& n = CL::c.nodes[i];
  if (!n.member || (n.kind != ACC_GATHER && n.kind != ACC_FOLD && n.kind != ACC_FOLDSEG)) return false;
  for (int s = 0; s < CL::c.n; ++s)
    if (is_scan_root(CL::c.nodes[s]) && reads_at_index(CL::c, CL::c.nodes[s].in[0], i)) return true;
  return false;
}
template <class CL> constexpr int costly_members() {
  int k = 0;
  for (int i = 0; i < CL::c.n; ++i) k += is_costly<CL>(i) ? 1 : 0;
  return k;
}
constexpr int kRingMaxSlots = 4;
// arrays from outside that come through the ring: read at the cluster's own index by a scan's operand or a store root
template <class CL> constexpr bool wants_ring(int i) {
  const CNode& n = CL::c.nodes[i];
  if (n.member || n.rank != domain_rank<CL>()) return false;
  for (int j = 0; j < CL::c.n; ++j) {
    const CNode& m = CL::c.nodes[j];
    if (is_scan_root(m) && reads_at_index(CL::c, m.in[0], i)) return true;
    if (is_store_root(m) && reads_at_index(CL::c, j, i)) return true;
  }
  return false;
}
// (those that the scans' operands read come first: the first visit needs no others)
template <class CL> constexpr bool feeds_scan(int i) {
  for (int j = 0; j < CL::c.n; ++j)
    if (is_scan_root(CL::c.nodes[j]) && reads_at_index(CL::c, CL::c.nodes[j].in[0], i)) return true;
  return false;
}
template <class CL> constexpr int ring_slot(int i) {
  int k = 0;
  for (int j = 0; j < CL::c.n; ++j)
    if (wants_ring<CL>(j) && (feeds_scan<CL>(i) ? feeds_scan<CL>(j) && j < i : feeds_scan<CL>(j) || j < i)) ++k;
  return k;
}
template <class CL> constexpr int ring_wanted(bool feeding_only) {
  int k = 0;
  for (int j = 0; j < CL::c.n; ++j) k += wants_ring<CL>(j) && (!feeding_only || feeds_scan<CL>(j)) ? 1 : 0;
  return k;
}
template <class CL> constexpr int ring_arrays() {                  // (what does not fit is read directly)
  return ring_wanted<CL>(false) < kRingMaxSlots ? ring_wanted<CL>(false) : kRingMaxSlots;
}
template <class CL> constexpr bool in_ring(int i) { return wants_ring<CL>(i) && ring_slot<CL>(i) < ring_arrays<CL>(); }
constexpr bool is_ring_output(const CNode& n) { return is_store_root(n) || (is_scan_root(n) && n.manifest); }
template <class CL> constexpr int ring_outputs() { return count_if<CL>(is_ring_output); }

template <class CL> constexpr bool has_index_map() {
  for (int i = 0; i < CL::c.n; ++i)
    if (CL::c.nodes[i].member && CL::c.nodes[i].kind == ACC_BACKPERMUTE && CL::c.nodes[i].idxfn != ACC_IDX_IDENTITY) return true;
  return false;
}
// whether a chunk may be evaluated although some of its elements lie outside the row (nothing is read through a value)
template <class CL> constexpr bool harmless_outside() {
  for (int i = 0; i < CL::c.n; ++i) {
    const CNode& n = CL::c.nodes[i];
    if (wants_ring<CL>(i) && !in_ring<CL>(i)) return false;
    if (n.member && !is_scan_root(n) && n.kind != ACC_MAP && n.kind != ACC_ZIPWITH && n.kind != ACC_GENERATE) return false;
  }
  return true;
}

// Scans of one direction, none of which feeds another, and element-wise roots.
constexpr bool scans_walk_together(const CCluster& c) {
  int first = -1;
  for (int i = 0; i < c.n; ++i) {
    const CNode& n = c.nodes[i];
    if (is_fold_root(n) || is_permute_root(n) || is_segfold_root(n)) return false;
    if (!is_scan_root(n)) continue;
    if (first >= 0 && n.kind != c.nodes[first].kind) return false;
    if (first < 0) first = i;
    for (int s = 0; s < c.n; ++s)
      if (is_scan_root(c.nodes[s]) && s != i && (n.in[0] == s || needs_scan(c, n.in[0], s))) return false;
  }
  return first >= 0;
}
template <class CL> constexpr bool scan_ring_eligible() {
  if (!scans_walk_together(CL::c)) return false;
  for (int i = 0; i < CL::c.n; ++i)
    if (is_store_root(CL::c.nodes[i]) && CL::c.nodes[i].rank != domain_rank<CL>()) return false;
  return ring_outputs<CL>() >= 1 && ring_outputs<CL>() <= kRingMaxSlots && count_if<CL>(is_scan_root) <= 4;
}

template <class CL, int I, class B, int K> struct reads_staged<CL, I, IxScN<B, K>> { static constexpr bool value = is_scan_root(CL::c.nodes[I]); };

// Where costly member p is staged: in its own array if it is stored anyway, else in the array of an output that is no
// other's staging area; -1 if there is none.  (Every output has the shape of the domain, and a tile of it is written only
// after the tile has been read for the last time, by the same block.)
template <class CL> constexpr int stage_target(int p) {
  if (CL::c.nodes[p].manifest) return p;
  int skip = 0;
  for (int i = 0; i < p; ++i) skip += is_costly<CL>(i) && !CL::c.nodes[i].manifest ? 1 : 0;
  for (int k = 0; k < CL::c.n; ++k)
    if (is_ring_output(CL::c.nodes[k]) && !is_costly<CL>(k) && skip-- == 0) return k;
  return -1;
}
template <class CL> constexpr bool has_stage_targets() {
  for (int i = 0; i < CL::c.n; ++i)
    if (is_costly<CL>(i) && stage_target<CL>(i) < 0) return false;
  return costly_members<CL>() > 0;
}
// The cluster once its costly members are staged: they are arrays, and members that only they needed are gone.
constexpr CCluster with_arrays(CCluster c, uint64_t arrays) {
  for (int i = 0; i < c.n; ++i)
    if ((arrays >> i) & 1) c.nodes[i] = CNode{ACC_INPUT, c.nodes[i].dtype, c.nodes[i].rank, 0, 0, 0, 0, {-1, -1, -1, -1, -1, -1}, false, true};
  bool live[kMaxCluster] = {};
  for (int i = c.n - 1; i >= 0; --i) {
    const CNode& n = c.nodes[i];
    if (!n.member) continue;
    if (is_scan_root(n) || is_store_root(n)) live[i] = true;
    if (live[i])
      for (int k = 0; k < n.nin; ++k) live[n.in[k]] = true;
  }
  for (int i = 0; i < c.n; ++i)
    if (c.nodes[i].member && !live[i]) c.nodes[i] = CNode{ACC_INPUT, c.nodes[i].dtype, c.nodes[i].rank, 0, 0, 0, 0, {-1, -1, -1, -1, -1, -1}, false, true};
  return c;
}
template <class CL> constexpr uint64_t costly_mask() {
  uint64_t m = 0;
  for (int i = 0; i < CL::c.n; ++i) m |= is_costly<CL>(i) ? 1ull << i : 0ull;
  return m;
}
template <class CL> struct StagedScan { static constexpr CCluster c = with_arrays(CL::c, costly_mask<CL>()); };
// (the staged arrays must come through the ring: they are written and read in one kernel)
template <class CL> constexpr bool can_stage() { return has_stage_targets<CL>() && ring_wanted<StagedScan<CL>>(true) <= kRingMaxSlots; }

// Whether everything the scans are computed from comes through the ring, element by element.  The ring evaluates the
// operands in both of its visits: what it would have to read from memory at other positions, it would read twice (the sum of
// two gathers stored nowhere, scanned: 2^24 elements 1101 us, by k_scan 222; a reversed array, 2^26 elements: 205 and 157).
template <class CL> constexpr bool fed_by_ring(int i) {
  const CNode& n = CL::c.nodes[i];
  if (!n.member) return in_ring<CL>(i);
  if (n.kind == ACC_GENERATE) return true;
  if (n.kind != ACC_MAP && n.kind != ACC_ZIPWITH && (n.kind != ACC_BACKPERMUTE || n.idxfn != ACC_IDX_IDENTITY)) return false;
  for (int k = 0; k < n.narr; ++k)
    if (!fed_by_ring<CL>(n.in[k])) return false;
  return true;
}
template <class CL> constexpr bool operands_fed_by_ring() {
  for (int i = 0; i < CL::c.n; ++i)
    if (is_scan_root(CL::c.nodes[i]) && !fed_by_ring<CL>(CL::c.nodes[i].in[0])) return false;
  return true;
}
// ... as they are, or once the costly members are staged
template <class CL> constexpr bool ring_serves() {
  if constexpr (!scan_ring_eligible<CL>()) return false;
  else if constexpr (can_stage<CL>()) return operands_fed_by_ring<StagedScan<CL>>();
  else return operands_fed_by_ring<CL>();
}

constexpr int kRingPerLane = 5;        // totals of a round that a lane of a look-back warp takes
constexpr int kRingMaxBlocks = 32 * kRingPerLane;   // and so the most blocks a round may have
constexpr int kRingDirectRounds = 8;   // rounds up to which every block adds the totals of a round up for itself
constexpr int kRingPollPause = 50;     // ns between two looks at totals that were missing
// Rows of up to kScanWarpRow elements get a warp each, up to kScanBlockRow a block each (a row may begin three words into its
// first 16-byte chunk).
constexpr int kScanWarpRow = 1024, kScanBlockRow = 16384 - 3;
constexpr int kScanGatherRow = 6144;        // ... but few rows with a gather below the scan up to so many elements only
constexpr int kScanFewElements = 1 << 17;   // a gather below a scan of up to so many elements is not staged

// ---- shape of the kernel --------------------------------------------------------------------------------
template <class CL>
struct RingTile {
  static constexpr int SCANS = count_if<CL>(is_scan_root);
  static constexpr int ARRAYS = ring_arrays<CL>(), OUTS = ring_outputs<CL>();
  static constexpr int FEEDING = ring_wanted<CL>(true) < ARRAYS ? ring_wanted<CL>(true) : ARRAYS;   // arrays of the first visit
  static constexpr int SLOTS = ARRAYS > OUTS ? ARRAYS : OUTS;
  // consecutive elements per thread, read and written as 128-bit accesses at a stride of an odd multiple of 16 bytes,
  // which eight lanes make without a bank conflict
  static constexpr int E = SLOTS == 1 ? 20 : 12;
  static constexpr int PARTS = 8;                                  // parts of a tile, one warp's share each
  static constexpr int PART = 32 * E, TILE = PARTS * PART;
};
constexpr int kRingRoom = 222 * 1024;                              // of the 227 KB a block may have
template <class CL, bool RESIDENT>
struct Ring : RingTile<CL> {
  using T = RingTile<CL>;
  static constexpr int GROUPS = 2;                                 // groups of PARTS scanning warps, taking rounds in turn
  static constexpr int REDUCERS = RESIDENT ? 8 : 4;                // reducing warps (4: two parts each)
  static constexpr int ROUND_BYTES = T::SCANS * T::PARTS * (32 * 4 + 12) + 64;   // kept per round between the visits (what precedes each thread, each part)
  static constexpr int STAGE_BYTES = T::SLOTS * T::TILE * 4;
  static constexpr int ROUNDS_AHEAD = 12;
  static constexpr int STAGES1 = RESIDENT ? 0 : 3;                 // of the first visit's own ring
  static constexpr int STAGE1_WORDS = T::FEEDING * T::TILE;
  static constexpr int ROOM = RESIDENT ? kRingRoom / (STAGE_BYTES + ROUND_BYTES)
                                       : (kRingRoom - STAGES1 * STAGE1_WORDS * 4 - ROUNDS_AHEAD * ROUND_BYTES) / STAGE_BYTES;
  static constexpr int MOST = RESIDENT ? 12 : 6;
  static constexpr int STAGES = ROOM < MOST ? ROOM : MOST;
  static constexpr bool FITS = STAGES >= (RESIDENT ? 4 : 3);        // (otherwise not instantiated)
  static constexpr int SLOTS_ROUNDS = RESIDENT ? STAGES : ROUNDS_AHEAD;   // rounds whose totals are kept
  // tiles whose copies are in flight, of either ring: what the memory's latency needs, no more (see above)
  static constexpr int COPIES = STAGE_BYTES <= 24 * 1024 ? 2 : 1;
  static constexpr int LB = SLOTS_ROUNDS < 6 ? SLOTS_ROUNDS : 6;   // look-back warps
  // A barrier is waited for by the parity of its phase, so whoever waits for round i must know that the round that used
  // the barrier before has passed it.  Warps that take every g-th round know that round i - g has; whose copy was issued
  // after all but COPIES of the earlier ones had landed; and rounds of one group pass in order.
  static_assert(!FITS || (STAGES >= GROUPS + COPIES && (RESIDENT || STAGES1 > COPIES) && LB <= SLOTS_ROUNDS && (RESIDENT || SLOTS_ROUNDS % GROUPS == 0)),
                "see above");
  static constexpr int W_RED = GROUPS * T::PARTS, W_LB = W_RED + REDUCERS, W_COPY = W_LB + LB;   // first warp of each kind
  static constexpr int THREADS = (W_COPY + (RESIDENT ? 1 : 2)) * 32;
  static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + (size_t)STAGES1 * STAGE1_WORDS * 4 + (size_t)SLOTS_ROUNDS * T::SCANS * T::PARTS * 32 * 4 + 128;
};
// one ring for both visits: where there is no room for two
template <class CL> constexpr bool ring_resident() { return !Ring<CL, false>::FITS; }
// Which kernels a cluster of scans needs: those for short rows (1), for long ones (2) or both (3).  A cluster of several
// scans is walked together where rows are long and scan by scan where they are short (see Passes in launch.cuh).
template <class CL, class = void> struct ScanForms { static constexpr int value = 3; };
template <class CL> struct ScanForms<CL, std::void_t<decltype(CL::kScanForms)>> { static constexpr int value = CL::kScanForms; };

template <class CL, int I, class A> __device__ __forceinline__ V4 ld_ext(const A& a, const IxRg& ix) {
  if constexpr (in_ring<CL>(I)) {
    const uint4 v = *reinterpret_cast<const uint4*>(ix.stage + ring_slot<CL>(I) * RingTile<CL>::TILE + ix.at);
    return V4{{v.x, v.y, v.z, v.w}};
  } else {
    return ld(reinterpret_cast<const uint32_t*>(a.n[I].ptr), a.n[I].C, Ix4{ix.r, ix.c});
  }
}
template <class CL, int I, class A> __device__ __forceinline__ uint32_t ld_ext(const A& a, const IxRg1& ix) {
  if constexpr (in_ring<CL>(I)) return ix.stage[ring_slot<CL>(I) * RingTile<CL>::TILE + ix.at];
  else return ld1(reinterpret_cast<const uint32_t*>(a.n[I].ptr), a.n[I].C, Ix{ix.r, ix.c});
}
template <class CL, int I, class A, int K> __device__ __forceinline__ V4 ld_ext(const A& a, const IxScN<IxRg, K>& ix) {
  return ld_ext<CL, I>(a, static_cast<const IxRg&>(ix));
}
template <class CL, int I, class A, int K> __device__ __forceinline__ uint32_t ld_ext(const A& a, const IxScN<IxRg1, K>& ix) {
  return ld_ext<CL, I>(a, static_cast<const IxRg1&>(ix));
}
template <class CL, int I, class A, class B, int K> __device__ __forceinline__ val_of<B> ld_staged(const A&, const IxScN<B, K>& ix) {
  return ix.sv[scan_ord<CL>(I)];
}

// A running total: fp32 sums are carried in fp64 (a chain over thousands of tiles), everything else as it is.
template <int FN, int DT> struct Running {
  static constexpr bool WIDE = FN == ACC_FN_ADD && DT == ACC_F32;
  using T = std::conditional_t<WIDE, double, uint32_t>;
  static __device__ __forceinline__ T identity() { if constexpr (WIDE) return 0.0; else return identity_of<FN, DT>(); }
  static __device__ __forceinline__ T of(uint32_t v) { if constexpr (WIDE) return (double)f_(v); else return v; }
  static __device__ __forceinline__ T add(T a, T b) { if constexpr (WIDE) return a + b; else return combine<FN, DT>(a, b); }
  static __device__ __forceinline__ uint32_t narrow(T a) { if constexpr (WIDE) return u_((float)a); else return a; }
  static __device__ __forceinline__ uint64_t bits(T a) { if constexpr (WIDE) return (uint64_t)__double_as_longlong(a); else return a; }
  static __device__ __forceinline__ T from(uint64_t b) { if constexpr (WIDE) return __longlong_as_double((long long)b); else return (uint32_t)b; }
  static __device__ __forceinline__ T up(T a, int d) { return __shfl_up_sync(0xFFFFFFFFu, a, d); }
  static __device__ __forceinline__ T across(T a, int d) { return __shfl_xor_sync(0xFFFFFFFFu, a, d); }
  // in a posted word, whose lowest bit says that it is there: an fp32 sum as two floats (the last bit of the second dropped)
  static __device__ __forceinline__ uint64_t state(T a) {
    if constexpr (WIDE) {
      const float hi = (float)a, lo = isfinite(hi) ? (float)(a - (double)hi) : 0.0f;    // an overflowed sum stays infinite
      return ((uint64_t)__float_as_uint(hi) << 32) | (__float_as_uint(lo) | 1u);
    } else {
      return ((uint64_t)a << 32) | 1u;
    }
  }
  static __device__ __forceinline__ T of_state(uint64_t s) {
    if constexpr (WIDE) return (double)__uint_as_float((uint32_t)(s >> 32)) + (double)__uint_as_float((uint32_t)s & ~1u);
    else return (uint32_t)(s >> 32);
  }
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint64_t ld_posted(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void post(uint64_t* p, uint64_t v) { asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory"); }

// A position in the ring: the stage of a round, and the parity its barriers have in that round.
template <int S> struct RingAt {
  int s;
  uint32_t parity = 0;
  __device__ explicit RingAt(int round) : s(round) {}             // round < S
  __device__ __forceinline__ void advance(int rounds) {            // by less than S
    s += rounds;
    if (s >= S) { s -= S; parity ^= 1u; }
  }
};

// ---- staging -------------------------------------------------------------------------------------------
// The one array that gather p reads through its source, if that is an array or an element-wise chain over one array; else -1.
template <class CL> constexpr int gathered_array(int p) {
  const CNode& n = CL::c.nodes[p];
  if (n.kind != ACC_GATHER) return -1;
  int i = n.in[1];
  while (CL::c.nodes[i].member) {
    const CNode& m = CL::c.nodes[i];
    if (m.kind != ACC_MAP || m.narr != 1) return -1;
    i = m.in[0];
  }
  return i;
}
// the source of a gather at one element, whose array's word has been fetched
struct IxWord { int r, c; uint32_t word; };
template <> struct width_of<IxWord> { static constexpr int value = 1; };
__device__ __forceinline__ Ix lane(const IxWord& i, int) { return Ix{i.r, i.c}; }
template <class CL, int I, class A> __device__ __forceinline__ uint32_t ld_ext(const A&, const IxWord& ix) { return ix.word; }

// The block's tiles (blockIdx.x, blockIdx.x + gridDim.x, ...) of costly member P, stored in the array stage_target names.
// `landing`: 32 words of shared memory per thread of the block.
template <class CL, int P, int TILE, int THREADS, class A, class L>
__device__ __forceinline__ void stage_costly(const A& a, int rounds, const L& locate, uint32_t* landing) {
  constexpr int X = gathered_array<CL>(P);
  constexpr CNode nd = CL::c.nodes[P];
  constexpr int CHUNKS = TILE / 4, U = 2;                              // chunks of four under way per thread
  uint32_t* out = reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[stage_target<CL>(P)].ptr));
  const uint32_t total = (uint32_t)rounds * CHUNKS;
  for (uint32_t q0 = threadIdx.x; q0 < total; q0 += THREADS * U) {
    int f[U], row[U], col[U];
    bool whole[U];
    uint32_t key[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t q = q0 + u * THREADS;
      whole[u] = false;
      if (q < total) {
        const uint32_t i = q / CHUNKS;
        const auto w = locate((int)(blockIdx.x + i * gridDim.x));
        f[u] = w.lo + (int)(q - i * CHUNKS) * 4;
        row[u] = w.row;
        col[u] = f[u] - w.row_lo;
        whole[u] = f[u] >= w.row_lo && f[u] + 4 <= w.row_hi;
        if (!whole[u]) {                                               // a chunk across a row's end: element by element
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (f[u] + e >= w.row_lo && f[u] + e < w.row_hi) out[f[u] + e] = eval<CL, P>(a, Ix{w.row, col[u] + e});
        } else if constexpr (X >= 0) {
          const V4 k = eval<CL, nd.in[0]>(a, Ix4{row[u], col[u]});
          const uint32_t n_src = (uint32_t)(a.n[X].R * a.n[X].C);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            key[u][e] = min(k.v[e], n_src - 1u);                       // (an index outside the source is the caller's error; it reads no foreign memory here)
            const uint32_t at = key[u][e] & ~3u, bytes = min(n_src - at, 4u) * 4u;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(landing + ((u * 4 + e) * THREADS + threadIdx.x) * 4)),
                         "l"(reinterpret_cast<const uint32_t*>(a.n[X].ptr) + at), "r"(bytes) : "memory");
          }
        }
      }
    }
    if constexpr (X >= 0) {
      asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (!whole[u]) continue;
        uint32_t v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t word = landing[((u * 4 + e) * THREADS + threadIdx.x) * 4 + (key[u][e] & 3u)];
          const Ix at = gather1<CL::c.nodes[nd.in[1]].rank>(key[u][e], a.n[nd.in[1]]);
          v[e] = eval<CL, nd.in[1]>(a, IxWord{at.r, at.c, word});
        }
        *reinterpret_cast<uint4*>(out + f[u]) = make_uint4(v[0], v[1], v[2], v[3]);
      }
    } else {
      V4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (whole[u]) v[u] = eval<CL, P>(a, Ix4{row[u], col[u]});
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (whole[u]) *reinterpret_cast<uint4*>(out + f[u]) = make_uint4(v[u].v[0], v[u].v[1], v[u].v[2], v[u].v[3]);
    }
  }
}

// Scratch: from byte 16 one 64-bit word per scan and tile, (total << 32) | 1 once it is posted, then (not RESIDENT) one for
// what precedes the tile.  Not used (and not cleared) where every row is one tile.
// WHOLE: the cluster whose costly members the block stages first (`whole`: its arguments); CL is then what is left of it,
// StagedScan<WHOLE>.  void: nothing is staged.
template <class WHOLE, int N> struct StageArgs { Args<N> a; };
template <int N> struct StageArgs<void, N> {};
template <class CL, class WHOLE = void, bool RESIDENT = ring_resident<CL>()>
__global__ void __launch_bounds__((Ring<CL, RESIDENT>::THREADS), 1) k_scan_ring(const __grid_constant__ Args<CL::c.n> a, int tiles_per_row, int n_tiles,
                                                                               const __grid_constant__ StageArgs<WHOLE, CL::c.n> whole) {
  using K = Ring<CL, RESIDENT>;
  constexpr int N = CL::c.n, E = K::E, CH = E / 4, TILE = K::TILE, S = K::STAGES, S1 = RESIDENT ? S : K::STAGES1, H = K::SLOTS_ROUNDS;
  constexpr int PARTS = K::PARTS, NS = K::SCANS;
  constexpr bool REV = CL::c.nodes[first_scan<CL>()].kind == ACC_SCANR;
  constexpr bool HARMLESS = harmless_outside<CL>();
  extern __shared__ uint32_t ring_raw[];
  // full / empty: a stage of the (second visit's) ring; full1 / empty1: of the first visit's; the others: a round
  __shared__ __align__(8) uint64_t full[S], empty[S], full1[S1], empty1[S1], posted[H], known[H], carried[H];
  __shared__ uint32_t part_total[H][NS][PARTS];
  __shared__ uint64_t part_before[H][NS][PARTS], carry[H][NS];
  __shared__ uint32_t rounds_asked;                                    // rounds whose copies for the second visit have been issued
  uint32_t* const ring = ring_raw + ((128u - (smem_addr(ring_raw) & 127u)) & 127u) / 4;
  uint32_t* const ring1 = RESIDENT ? ring : ring + S * K::SLOTS * TILE;
  constexpr int kStage1 = RESIDENT ? K::SLOTS * TILE : K::STAGE1_WORDS;
  uint32_t* const thread_before = RESIDENT ? ring + S * K::SLOTS * TILE : ring1 + S1 * kStage1;        // [round][scan][part][lane]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int G = (int)gridDim.x, n = a.C, count = a.R * a.C;
  const int rounds = ((int)blockIdx.x < n_tiles) ? (n_tiles - 1 - (int)blockIdx.x) / G + 1 : 0;   // tiles of this block
  const bool chain = tiles_per_row > 1;
  const bool direct = n_tiles <= kRingDirectRounds * G;               // how the blocks learn of one another's totals (see the look-back warps)

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], PARTS); }
    for (int s = 0; s < S1; ++s) { mbar_init(&full1[s], 1); mbar_init(&empty1[s], PARTS); }
    for (int h = 0; h < H; ++h) { mbar_init(&posted[h], PARTS); mbar_init(&known[h], 1); mbar_init(&carried[h], 1); }
    rounds_asked = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // a tile's row, the flat position of its first word (a multiple of four) and the row's range
  struct Where { int row, lo, row_lo, row_hi; };
  auto locate = [&](int tile) {
    Where w;
    w.row = tiles_per_row == n_tiles ? 0 : tile / tiles_per_row;
    const int k = tile - w.row * tiles_per_row;
    w.row_lo = w.row * n;
    w.row_hi = w.row_lo + n;
    w.lo = (w.row_lo & ~3) + (REV ? tiles_per_row - 1 - k : k) * TILE;
    return w;
  };

  if constexpr (!std::is_void<WHOLE>::value) {
    static_assert(K::SMEM >= K::THREADS * 128 + 128, "the ring is where the gathered words land");
    static_for<0, N>([&](auto ic) {
      constexpr int p = decltype(ic)::value;
      if constexpr (is_costly<WHOLE>(p)) stage_costly<WHOLE, p, TILE, K::THREADS>(whole.a, rounds, locate, ring);
    });
    asm volatile("fence.proxy.async;" ::: "memory");                    // the staged values and the ring's words, before copies touch either
    __syncthreads();
  }

  if (warp >= K::W_COPY) {
    // ---- the copy warps: one lane each ----------------------------------------------------------------
    if (lane != 0) return;
    auto feed = [&](auto first_c) {
      constexpr bool FIRST = decltype(first_c)::value;                   // the first visit's ring (not RESIDENT)
      constexpr int STAGES = FIRST ? S1 : S, ARRAYS = FIRST ? K::FEEDING : K::ARRAYS;
      uint64_t* const landed = FIRST ? full1 : full;
      uint64_t* const freed = FIRST ? empty1 : empty;
      RingAt<STAGES> at(0), behind(0);
      int i = 0;
      bool ok = true;
      for (; i < rounds; ++i, at.advance(1)) {
        if (i >= STAGES) ok = wait_phase(&freed[at.s], at.parity ^ 1u);
        if (ok && i >= K::COPIES) {                                      // no more copies in flight than the memory's latency needs
          ok = wait_phase(&landed[behind.s], behind.parity);
          behind.advance(1);
        }
        if constexpr (FIRST) {
          // as far ahead as there is room for rounds: those asked for by the second visit, less its stages, are done with
          for (uint32_t spins = 0; ok && *reinterpret_cast<volatile uint32_t*>(&rounds_asked) + H <= (uint32_t)(i + S); ++spins) {
            ok = spins < kCopySpinLimit * 16u;
            __nanosleep(100);
          }
        }
        if (!ok) break;
        const Where w = locate((int)blockIdx.x + i * G);
        const int hi = min(w.lo + TILE, w.row_hi);
        const int end = min((hi + 3) & ~3, count & ~3);                // whole chunks that lie inside the arrays
        const uint32_t bytes = end > w.lo ? (uint32_t)(end - w.lo) * 4u : 0u, bar = smem_addr(&landed[at.s]);
        uint32_t* stage = FIRST ? ring1 + at.s * kStage1 : ring + at.s * K::SLOTS * TILE;
        static_for<0, N>([&](auto ic) {                                 // the last words of arrays that end within a chunk
          constexpr int k = decltype(ic)::value;
          if constexpr (in_ring<CL>(k) && ring_slot<CL>(k) < ARRAYS) {
            const volatile uint32_t* src = reinterpret_cast<const volatile uint32_t*>(a.n[k].ptr);
            for (int f = max(end, w.lo); f < hi; ++f) stage[ring_slot<CL>(k) * TILE + (f - w.lo)] = src[f];
          }
        });
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes * (uint32_t)ARRAYS) : "memory");
        if (bytes) {
          static_for<0, N>([&](auto ic) {
            constexpr int k = decltype(ic)::value;
            if constexpr (in_ring<CL>(k) && ring_slot<CL>(k) < ARRAYS)
              bulk_load(smem_addr(stage + ring_slot<CL>(k) * TILE), reinterpret_cast<const uint32_t*>(a.n[k].ptr) + w.lo, bytes, bar);
          });
        }
        if constexpr (!FIRST && !RESIDENT) *reinterpret_cast<volatile uint32_t*>(&rounds_asked) = (uint32_t)i + 1u;
      }
      if (!ok) raise_status(a, kStatusTimeout);
      // copies still in flight must not land in the shared memory of a block that has gone
      for (int q = max(0, i - K::COPIES - 1); q < i; ++q) wait_phase(&landed[q % STAGES], (uint32_t)(q / STAGES) & 1u);
    };
    if (RESIDENT || warp == K::W_COPY) feed(std::false_type{});
    else feed(std::true_type{});
    return;
  }

  if (warp >= K::W_LB) {
    // ---- a look-back warp: every LB-th round -------------------------------------------------------
    uint64_t* states = reinterpret_cast<uint64_t*>(a.scratch + 4);
    const int l = warp - K::W_LB;
    for (int i = l; i < rounds; i += K::LB) {
      const int s = i % H;
      const uint32_t parity = (uint32_t)(i / H) & 1u;
      if (!__all_sync(0xFFFFFFFFu, wait_phase(&posted[s], parity))) { raise_status(a, kStatusTimeout); return; }
      const int tile = (int)blockIdx.x + i * G, first = i * G;         // (first tile of the round)
      const int after = s + 1 == H ? 0 : s + 1;
      uint64_t earlier[NS];                                            // per lane: the parts of this tile before part `lane` (bits of a running total)
      uint64_t here[NS];                                               // what of the row lies before this tile
      static_for<0, N>([&](auto ic) {
        constexpr int sc = decltype(ic)::value;
        if constexpr (is_scan_root(CL::c.nodes[sc])) {
          constexpr int o = scan_ord<CL>(sc);
          using Run = Running<CL::c.nodes[sc].fn, CL::c.nodes[sc].dtype>;
          auto incl = lane < PARTS ? Run::of(part_total[s][o][lane]) : Run::identity();
#pragma unroll
          for (int d = 1; d < PARTS; d <<= 1) {
            const auto t = Run::up(incl, d);
            if (lane >= d) incl = Run::add(t, incl);
          }
          if (chain && lane == PARTS - 1) post(states + (size_t)o * n_tiles + tile, ((uint64_t)Run::narrow(incl) << 32) | 1u);
          const auto before = Run::up(incl, 1);
          earlier[o] = Run::bits(lane == 0 ? Run::identity() : before);
          here[o] = Run::bits(Run::identity());
        }
      });
      // the totals of tiles base + step * u of scan o, u = 0 .. kRingPerLane - 1, where these lie below `limit`: waits until they are posted
      auto totals = [&](int o, int base, int step, int limit, uint64_t (&v)[kRingPerLane]) {
        const uint64_t* at = states + (size_t)o * n_tiles + base;
#pragma unroll
        for (int u = 0; u < kRingPerLane; ++u) v[u] = base + step * u < limit ? 0u : 1u;
        for (uint32_t spins = 0;;) {
          bool missing = false;
#pragma unroll
          for (int u = 0; u < kRingPerLane; ++u)                                   // (only what is still missing is asked for again)
            if ((v[u] & 1u) == 0u) v[u] = ld_posted(at + step * u);
#pragma unroll
          for (int u = 0; u < kRingPerLane; ++u) missing = missing || (v[u] & 1u) == 0u;
          if (!__any_sync(0xFFFFFFFFu, missing)) return true;
          if (++spins > a.spin_limit) return false;
          __nanosleep(kRingPollPause);
        }
      };
      bool in_time = true;
      if (chain) {
        if (direct) {
          // every block reads the totals of the whole round itself: the shortest way, for few rounds
          const int row_first = tile - tile % tiles_per_row;               // first tile of this tile's row
          const bool more = i + 1 < rounds;                                // then the totals of the whole round are carried on
          const int limit = more ? first + G : tile;
          const int last_first = more ? (first + G - 1) - (first + G - 1) % tiles_per_row : 0;   // first tile of the row that the next round may go on with
          uint64_t next[NS];
          static_for<0, N>([&](auto ic) {
            constexpr int sc = decltype(ic)::value;
            if constexpr (is_scan_root(CL::c.nodes[sc])) {
              constexpr int o = scan_ord<CL>(sc);
              using Run = Running<CL::c.nodes[sc].fn, CL::c.nodes[sc].dtype>;
              auto h = Run::identity(), x = Run::identity();
              for (int base = max(first, row_first); base < limit; base += 32 * kRingPerLane) {
                uint64_t v[kRingPerLane];
                in_time = in_time && totals(o, base + lane, 32, limit, v);
                if (!in_time) break;
#pragma unroll
                for (int u = 0; u < kRingPerLane; ++u) {
                  const int j = base + 32 * u + lane;
                  const auto t = j < limit ? Run::of((uint32_t)(v[u] >> 32)) : Run::identity();
                  if (j < tile) h = Run::add(h, t);
                  if (j >= last_first) x = Run::add(x, t);
                }
              }
#pragma unroll
              for (int d = 16; d > 0; d >>= 1) {
                h = Run::add(h, Run::across(h, d));
                if (more) x = Run::add(x, Run::across(x, d));
              }
              here[o] = Run::bits(h);
              next[o] = Run::bits(x);
            }
          });
          if (i > 0 && !__all_sync(0xFFFFFFFFu, wait_phase(&carried[s], parity ^ (s == 0 ? 1u : 0u)))) { raise_status(a, kStatusTimeout); return; }
          static_for<0, N>([&](auto ic) {
            constexpr int sc = decltype(ic)::value;
            if constexpr (is_scan_root(CL::c.nodes[sc])) {
              constexpr int o = scan_ord<CL>(sc);
              using Run = Running<CL::c.nodes[sc].fn, CL::c.nodes[sc].dtype>;
              const auto before = i > 0 ? Run::from(carry[s][o]) : Run::identity();
              if (row_first < first) here[o] = Run::bits(Run::add(before, Run::from(here[o])));
              if (more && lane == 0) carry[after][o] = Run::bits(last_first < first ? Run::add(before, Run::from(next[o])) : Run::from(next[o]));
            }
          });
          __syncwarp();
          if (lane == 0 && more) mbar_arrive(&carried[after]);
        } else if (blockIdx.x == 0) {
          // the first block scans the totals of the round (a row's first tile starts anew) and posts what precedes each tile
          const int limit = min(first + G, n_tiles), j0 = first + kRingPerLane * lane;
          uint64_t excl[NS][kRingPerLane], lane_before[NS], lane_after[NS];
          bool resets[kRingPerLane], any = false;                                     // a row begins at tile j0 + u; one begins in this lane's tiles
#pragma unroll
          for (int u = 0; u < kRingPerLane; ++u) {
            resets[u] = j0 + u < limit && (j0 + u) % tiles_per_row == 0;
            any = any || resets[u];
          }
          const unsigned begins = __ballot_sync(0xFFFFFFFFu, any);
          const unsigned below = begins & ((1u << lane) - 1u);              // lanes before this one in which a row begins
          const int run_from = below ? 31 - __clz(below) : -1;              // the last of them: nothing before its row matters
          static_for<0, N>([&](auto ic) {
            constexpr int sc = decltype(ic)::value;
            if constexpr (is_scan_root(CL::c.nodes[sc])) {
              constexpr int o = scan_ord<CL>(sc);
              using Run = Running<CL::c.nodes[sc].fn, CL::c.nodes[sc].dtype>;
              uint64_t v[kRingPerLane];
              in_time = in_time && totals(o, j0, 1, limit, v);
              auto run = Run::identity();
#pragma unroll
              for (int u = 0; u < kRingPerLane; ++u) {
                if (resets[u]) run = Run::identity();
                excl[o][u] = Run::bits(run);
                if (in_time && j0 + u < limit) run = Run::add(run, Run::of((uint32_t)(v[u] >> 32)));
              }
#pragma unroll
              for (int d = 1; d < 32; d <<= 1) {                            // (a lane in which a row begins takes nothing from before)
                const auto t = Run::up(run, d);
                if (lane >= d && !any && lane - d >= run_from) run = Run::add(t, run);
              }
              lane_after[o] = Run::bits(run);
              const auto t = Run::up(run, 1);
              lane_before[o] = Run::bits(lane == 0 ? Run::identity() : t);
            }
          });
          if (i > 0 && !__all_sync(0xFFFFFFFFu, wait_phase(&carried[s], parity ^ (s == 0 ? 1u : 0u)))) { raise_status(a, kStatusTimeout); return; }
          static_for<0, N>([&](auto ic) {
            constexpr int sc = decltype(ic)::value;
            if constexpr (is_scan_root(CL::c.nodes[sc])) {
              constexpr int o = scan_ord<CL>(sc);
              using Run = Running<CL::c.nodes[sc].fn, CL::c.nodes[sc].dtype>;
              const auto sofar = i > 0 ? Run::from(carry[s][o]) : Run::identity();
              if (lane == 31) carry[after][o] = Run::bits(begins ? Run::from(lane_after[o]) : Run::add(sofar, Run::from(lane_after[o])));
              auto before = Run::from(lane_before[o]);
              if (run_from < 0) before = Run::add(sofar, before);
              bool fresh = false;
#pragma unroll
              for (int u = 0; u < kRingPerLane; ++u) {
                fresh = fresh || resets[u];
                const auto p = fresh ? Run::from(excl[o][u]) : Run::add(before, Run::from(excl[o][u]));
                if (u == 0) here[o] = Run::bits(p);                         // (lane 0: this block's tile)
                if (j0 + u < limit && j0 + u > tile) post(states + (size_t)(NS + o) * n_tiles + j0 + u, Run::state(p));
              }
              here[o] = __shfl_sync(0xFFFFFFFFu, here[o], 0);
            }
          });
          __syncwarp();
          if (lane == 31) mbar_arrive(&carried[after]);
        } else {
          // ... every other block waits for what the first one posts for its tile
          uint64_t v = lane < NS ? 0u : 1u;
          for (uint32_t spins = 0;;) {
            if ((v & 1u) == 0u) v = ld_posted(states + (size_t)(NS + lane) * n_tiles + tile);
            if (!__any_sync(0xFFFFFFFFu, (v & 1u) == 0u)) break;
            if (++spins > a.spin_limit) { in_time = false; break; }
            __nanosleep(kRingPollPause);
          }
          static_for<0, N>([&](auto ic) {
            constexpr int sc = decltype(ic)::value;
            if constexpr (is_scan_root(CL::c.nodes[sc])) {
              constexpr int o = scan_ord<CL>(sc);
              using Run = Running<CL::c.nodes[sc].fn, CL::c.nodes[sc].dtype>;
              here[o] = Run::bits(Run::of_state(__shfl_sync(0xFFFFFFFFu, v, o)));
            }
          });
        }
        if (!in_time) raise_status(a, kStatusTimeout);
      }
      static_for<0, N>([&](auto ic) {
        constexpr int sc = decltype(ic)::value;
        if constexpr (is_scan_root(CL::c.nodes[sc])) {
          constexpr int o = scan_ord<CL>(sc);
          using Run = Running<CL::c.nodes[sc].fn, CL::c.nodes[sc].dtype>;
          if (lane < PARTS) part_before[s][o][lane] = Run::bits(Run::add(Run::from(here[o]), Run::from(earlier[o])));
        }
      });
      __syncwarp();
      if (lane == 0) mbar_arrive(&known[s]);
    }
    return;
  }

  // ---- reducing and scanning warps -----------------------------------------------------------------
  // Part p of a tile (in the order of the walk) is a warp's share; its lanes hold E consecutive elements each.
  const int mem_lane = REV ? 31 - lane : lane;
  auto start_of = [&](int part) { return ((REV ? PARTS - 1 - part : part) * 32 + mem_lane) * E; };   // the thread's first word in a slot
  auto mask_of = [&](int f, const Where& w) {                           // which of elements f .. f + 3 belong to the row
    uint32_t m = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) m |= (f + e >= w.row_lo && f + e < w.row_hi) ? 1u << e : 0u;
    return m;
  };
  // whether a part lies wholly inside its row (the same for the whole warp)
  auto is_whole = [&](const Where& w, int part) {
    const int lo = w.lo + (REV ? PARTS - 1 - part : part) * K::PART;
    return lo >= w.row_lo && lo + K::PART <= w.row_hi;
  };
  // the value of member I at a chunk, of which the elements in `inside` exist (the others: anything)
  auto value = [&](auto member, const auto& ix, uint32_t inside) {
    constexpr int I = decltype(member)::value;
    using IX = std::decay_t<decltype(ix)>;
    if constexpr (HARMLESS) {
      return eval<CL, I>(a, ix);
    } else {
      if (inside == 15u) return eval<CL, I>(a, ix);
      V4 v{{0u, 0u, 0u, 0u}};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if ((inside >> e) & 1u) {
          if constexpr (std::is_same<IX, IxRg>::value) {
            v.v[e] = eval<CL, I>(a, IxRg1{ix.r, ix.c + e, ix.stage, ix.at + e});
          } else {
            IxScN<IxRg1, NS> one;
            one.r = ix.r; one.c = ix.c + e; one.stage = ix.stage; one.at = ix.at + e;
#pragma unroll
            for (int o = 0; o < NS; ++o) one.sv[o] = ix.sv[o].v[e];
            v.v[e] = eval<CL, I>(a, one);
          }
        }
      return v;
    }
  };

  if (warp >= K::W_RED) {
    // ---- first visit: the totals of the parts -------------------------------------------------------
    auto reduce = [&](auto whole_c, const Where& w, int part, uint32_t* stage, int h) {
      constexpr bool WHOLE_PART = decltype(whole_c)::value;
      const int at0 = start_of(part);
      static_for<0, N>([&](auto ic) {
        constexpr int sc = decltype(ic)::value;
        constexpr CNode sn = CL::c.nodes[sc];
        if constexpr (is_scan_root(sn)) {
          constexpr int o = scan_ord<CL>(sc);
          uint32_t incl = identity_of<sn.fn, sn.dtype>();
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const int f = w.lo + at0 + 4 * j;
            const uint32_t inside = WHOLE_PART ? 15u : mask_of(f, w);
            V4 v = value(std::integral_constant<int, sn.in[0]>{}, IxRg{w.row, f - w.row_lo, stage, at0 + 4 * j}, inside);
            if constexpr (!WHOLE_PART) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (!((inside >> e) & 1u)) v.v[e] = identity_of<sn.fn, sn.dtype>();
            }
            const uint32_t four = combine<sn.fn, sn.dtype>(combine<sn.fn, sn.dtype>(v.v[0], v.v[1]), combine<sn.fn, sn.dtype>(v.v[2], v.v[3]));
            incl = j == 0 ? four : combine<sn.fn, sn.dtype>(incl, four);
          }
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= d) incl = combine<sn.fn, sn.dtype>(t, incl);
          }
          const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
          thread_before[((h * NS + o) * PARTS + part) * 32 + lane] = lane == 0 ? identity_of<sn.fn, sn.dtype>() : before;
          if (lane == 31) part_total[h][o][part] = incl;
        }
      });
      __syncwarp();                                                     // (every lane's words are in place)
      if (lane == 31) mbar_arrive(&posted[h]);
    };
    RingAt<S1> at(0);
    RingAt<H> slot(0);
    for (int i = 0; i < rounds; ++i, at.advance(1), slot.advance(1)) {
      const Where w = locate((int)blockIdx.x + i * G);
      if (!__all_sync(0xFFFFFFFFu, wait_phase(RESIDENT ? &full[at.s] : &full1[at.s], at.parity))) { raise_status(a, kStatusTimeout); return; }
      uint32_t* stage = ring1 + at.s * kStage1;
#pragma unroll 1
      for (int part = warp - K::W_RED; part < PARTS; part += K::REDUCERS) {
        if (is_whole(w, part)) reduce(std::true_type{}, w, part, stage, slot.s);
        else reduce(std::false_type{}, w, part, stage, slot.s);
        if constexpr (!RESIDENT)
          if (lane == 31) mbar_arrive(&empty1[at.s]);                    // (behind the part's __syncwarp: its words have been read)
      }
    }
    return;
  }

  // ---- second visit: scan, evaluate what reads the scan, store ------------------------------------------
  const int part = warp % PARTS, at0 = start_of(part), part_lo = (REV ? PARTS - 1 - part : part) * K::PART;
  auto scan = [&](auto whole_c, const Where& w, int s, int h) {
    constexpr bool WHOLE_PART = decltype(whole_c)::value;
    uint32_t* stage = ring + s * K::SLOTS * TILE;
    uint32_t base[NS], run[NS];                                         // what precedes the thread's elements; their running scan
    static_for<0, N>([&](auto ic) {
      constexpr int sc = decltype(ic)::value;
      constexpr CNode sn = CL::c.nodes[sc];
      if constexpr (is_scan_root(sn)) {
        constexpr int o = scan_ord<CL>(sc);
        using Run = Running<sn.fn, sn.dtype>;
        auto b = Run::add(Run::from(part_before[h][o][part]), Run::of(thread_before[((h * NS + o) * PARTS + part) * 32 + lane]));
        if constexpr (sn.p0 == 1) b = Run::add(Run::of(sn.dtype == ACC_F32 ? u_(a.n[sc].fp0) : (uint32_t)a.n[sc].ip0), b);   // the seed comes first
        base[o] = Run::narrow(b);
        run[o] = identity_of<sn.fn, sn.dtype>();
      }
    });
#pragma unroll
    for (int jj = 0; jj < CH; ++jj) {
      const int j = REV ? CH - 1 - jj : jj;
      const int f = w.lo + at0 + 4 * j;
      const uint32_t inside = WHOLE_PART ? 15u : mask_of(f, w);
      const IxRg ix{w.row, f - w.row_lo, stage, at0 + 4 * j};
      IxScN<IxRg, NS> with;
      static_cast<IxRg&>(with) = ix;
      static_for<0, N>([&](auto ic) {
        constexpr int sc = decltype(ic)::value;
        constexpr CNode sn = CL::c.nodes[sc];
        if constexpr (is_scan_root(sn)) {
          constexpr int o = scan_ord<CL>(sc);
          const V4 v = value(std::integral_constant<int, sn.in[0]>{}, ix, inside);
#pragma unroll
          for (int ee = 0; ee < 4; ++ee) {
            const int e = REV ? 3 - ee : ee;
            const uint32_t upto = WHOLE_PART || ((inside >> e) & 1u) ? combine<sn.fn, sn.dtype>(run[o], v.v[e]) : run[o];
            with.sv[o].v[e] = combine<sn.fn, sn.dtype>(base[o], sn.p0 == 1 ? run[o] : upto);
            run[o] = upto;
          }
        }
      });
      V4 out[K::OUTS];
      static_for<0, N>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        if constexpr (is_ring_output(CL::c.nodes[k])) {
          constexpr int o = count_if<CL>(is_ring_output, k);
          if constexpr (is_scan_root(CL::c.nodes[k])) out[o] = with.sv[scan_ord<CL>(k)];
          else out[o] = value(std::integral_constant<int, k>{}, with, inside);
          if (!WHOLE_PART && inside != 15u && inside != 0u) {            // a chunk across a row's end is stored element by element
            uint32_t* dst = reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[k].ptr));
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if ((inside >> e) & 1u) dst[f + e] = out[o].v[e];
          }
        }
      });
      // (the chunk's operands have been read, by this thread and nobody else: the results take their place)
#pragma unroll
      for (int o = 0; o < K::OUTS; ++o)
        *reinterpret_cast<uint4*>(stage + o * TILE + at0 + 4 * j) = make_uint4(out[o].v[0], out[o].v[1], out[o].v[2], out[o].v[3]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) {
      const int from = WHOLE_PART ? w.lo + part_lo : max(w.lo + part_lo, (w.row_lo + 3) & ~3);
      const int to = WHOLE_PART ? from + K::PART : min(w.lo + part_lo + K::PART, w.row_hi & ~3);
      if (to > from) {
        static_for<0, N>([&](auto ic) {
          constexpr int k = decltype(ic)::value;
          if constexpr (is_ring_output(CL::c.nodes[k])) {
            constexpr int o = count_if<CL>(is_ring_output, k);
            bulk_store(reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[k].ptr)) + from, smem_addr(stage + o * TILE + (from - w.lo)), (uint32_t)(to - from) * 4u);
          }
        });
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");     // the results have left the stage
      mbar_arrive(&empty[s]);
    }
  };
  const int group = warp / PARTS;
  RingAt<S> at(group);
  RingAt<H> slot(group);
  for (int i = group; i < rounds; i += K::GROUPS, at.advance(K::GROUPS), slot.advance(K::GROUPS)) {
    const Where w = locate((int)blockIdx.x + i * G);
    if (!__all_sync(0xFFFFFFFFu, wait_phase(&full[at.s], at.parity) && wait_phase(&known[slot.s], slot.parity))) { raise_status(a, kStatusTimeout); break; }
    if (is_whole(w, part)) scan(std::true_type{}, w, at.s, slot.s);
    else scan(std::false_type{}, w, at.s, slot.s);
  }
  if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// =========================================================================================
// A warp per row (WARPS = 1: kBlock / 32 rows to a block), or a block per row with as many warps as the row has work for, up to WARPS;
// CH chunks of four per lane at a time: all of a row's loads are under way together, which is what bounds these rows.  A warp takes a
// longer row in several spans; a block takes its row in one, so whoever launches it sees to it that its warps cover the row
// and the up to three words of its first chunk that precede it: blockDim.x / 32 * CH * 128 >= C + 3 (C, where rows start on 16 bytes).
template <class CL, int WARPS, int CH>
__global__ void __launch_bounds__(WARPS == 1 ? kBlock : WARPS * 32, WARPS == 1 ? 1 : CH == 2 ? 3 : 2) k_scan_rows(const __grid_constant__ Args<CL::c.n> a) {
  constexpr int N = CL::c.n, NS = count_if<CL>(is_scan_root), SPAN = WARPS * CH * 128, ROWS = WARPS == 1 ? kBlock / 32 : 1;
  constexpr bool REV = CL::c.nodes[first_scan<CL>()].kind == ACC_SCANR;
  __shared__ uint32_t warp_total[2][NS][WARPS];
  const int lane = threadIdx.x & 31, mem_lane = REV ? 31 - lane : lane;
  const int warp = WARPS == 1 ? 0 : (int)threadIdx.x >> 5, mem_warp = WARPS > 1 && REV ? (int)blockDim.x / 32 - 1 - warp : warp;
  const int n = a.C;
  int half = 0;                                                       // which half of warp_total this row uses
  for (int row = blockIdx.x * ROWS + (WARPS == 1 ? (int)threadIdx.x >> 5 : 0); row < a.R; row += gridDim.x * ROWS, half ^= 1) {
    const int row_lo = row * n, row_hi = row_lo + n, first = row_lo & ~3;
    const int spans = WARPS == 1 ? (row_hi - first + SPAN - 1) / SPAN : 1;
    auto mask_of = [&](int f) {                                        // which of elements f .. f + 3 belong to the row
      uint32_t m = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) m |= (f + e >= row_lo && f + e < row_hi) ? 1u << e : 0u;
      return m;
    };
    uint64_t carry[NS];
    static_for<0, N>([&](auto ic) {
      constexpr int s = decltype(ic)::value;
      constexpr CNode sn = CL::c.nodes[s];
      if constexpr (is_scan_root(sn)) {
        using Run = Running<sn.fn, sn.dtype>;
        carry[scan_ord<CL>(s)] = Run::bits(sn.p0 == 1 ? Run::of(sn.dtype == ACC_F32 ? u_(a.n[s].fp0) : (uint32_t)a.n[s].ip0) : Run::identity());
      }
    });
    for (int q = 0; q < spans; ++q) {
      const int lo = first + (REV ? spans - 1 - q : q) * SPAN + mem_warp * CH * 128;
      // Whether the warp's elements all belong to the row.  Then nothing below branches: a load whose value is used inside a
      // branch is waited for before the next chunk's is issued (rows of 16000 through a map: 155 us, without the branch 80 us).
      const bool whole = lo >= row_lo && lo + CH * 128 <= row_hi;
      // ... and whether chunks beyond the row's ends may be read all the same (they lie inside the arrays, and nothing is read
      // through a value), so that only what is stored needs the row's ends
      const bool safe = whole || (harmless_outside<CL>() && lo >= 0 && lo + CH * 128 <= (a.R * n & ~3));
      V4 v[NS][CH];
      auto operands = [&](auto safe_c) {
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          const int f = lo + (j * 32 + mem_lane) * 4;
          const uint32_t inside = decltype(safe_c)::value ? 15u : mask_of(f);
          static_for<0, N>([&](auto ic) {
            constexpr int s = decltype(ic)::value;
            constexpr CNode sn = CL::c.nodes[s];
            if constexpr (is_scan_root(sn)) {
              constexpr int o = scan_ord<CL>(s);
              if (inside == 15u) {
                v[o][j] = eval<CL, sn.in[0]>(a, Ix4{row, f - row_lo});
              } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  v[o][j].v[e] = ((inside >> e) & 1u) ? eval<CL, sn.in[0]>(a, Ix{row, f + e - row_lo}) : identity_of<sn.fn, sn.dtype>();
              }
            }
          });
        }
      };
      const bool any = lo < row_hi && lo + CH * 128 > row_lo;          // (a warp beyond the row's end has nothing to read or store)
      if (safe && any) operands(std::true_type{});
      else operands(std::false_type{});
      if (safe && !whole) {
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          const uint32_t inside = mask_of(lo + (j * 32 + mem_lane) * 4);
          static_for<0, N>([&](auto ic) {
            constexpr int s = decltype(ic)::value;
            constexpr CNode sn = CL::c.nodes[s];
            if constexpr (is_scan_root(sn)) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (!((inside >> e) & 1u)) v[scan_ord<CL>(s)][j].v[e] = identity_of<sn.fn, sn.dtype>();
            }
          });
        }
      }
      // what precedes each chunk within the warp's part, and the part's total
      uint32_t before[NS][CH], total[NS];
      static_for<0, N>([&](auto ic) {
        constexpr int s = decltype(ic)::value;
        constexpr CNode sn = CL::c.nodes[s];
        if constexpr (is_scan_root(sn)) {
          constexpr int o = scan_ord<CL>(s);
          uint32_t incl[CH];
#pragma unroll
          for (int j = 0; j < CH; ++j)
            incl[j] = combine<sn.fn, sn.dtype>(combine<sn.fn, sn.dtype>(v[o][j].v[0], v[o][j].v[1]), combine<sn.fn, sn.dtype>(v[o][j].v[2], v[o][j].v[3]));
#pragma unroll
          for (int d = 1; d < 32; d <<= 1)
#pragma unroll
            for (int j = 0; j < CH; ++j) {
              const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl[j], d);
              if (lane >= d) incl[j] = combine<sn.fn, sn.dtype>(t, incl[j]);
            }
          uint32_t run = identity_of<sn.fn, sn.dtype>();
#pragma unroll
          for (int jj = 0; jj < CH; ++jj) {
            const int j = REV ? CH - 1 - jj : jj;
            const uint32_t e = __shfl_up_sync(0xFFFFFFFFu, incl[j], 1);
            before[o][j] = lane == 0 ? run : combine<sn.fn, sn.dtype>(run, e);
            run = combine<sn.fn, sn.dtype>(run, __shfl_sync(0xFFFFFFFFu, incl[j], 31));
          }
          total[o] = run;
          if (WARPS > 1 && lane == 0) warp_total[half][o][warp] = run;
        }
      });
      if constexpr (WARPS > 1) {
        __syncthreads();                                                // (the next row writes the other half, and the one after it is a barrier away)
        static_for<0, N>([&](auto ic) {
          constexpr int s = decltype(ic)::value;
          constexpr CNode sn = CL::c.nodes[s];
          if constexpr (is_scan_root(sn)) {
            constexpr int o = scan_ord<CL>(s);
            using Run = Running<sn.fn, sn.dtype>;
            // (a lane per warp: one conversion instead of a chain of sixteen conversions and additions in every warp: 4099 x 3001
            // in two directions 48.8 -> 45.0 us, 8000 x 1200 77.5 -> 66.4)
            static_assert((WARPS & (WARPS - 1)) == 0 && WARPS <= 32, "a lane per warp, the sums in every lane");
            const int w = lane & (WARPS - 1);
            auto sum = w < warp ? Run::of(warp_total[half][o][w]) : Run::identity();
#pragma unroll
            for (int d = WARPS / 2; d > 0; d >>= 1) sum = Run::add(sum, Run::across(sum, d));
            carry[o] = Run::bits(Run::add(Run::from(carry[o]), sum));
          }
        });
      }
      auto results = [&](auto whole_c, auto safe_c) {
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          const int f = lo + (j * 32 + mem_lane) * 4;
          const uint32_t inside = decltype(whole_c)::value ? 15u : mask_of(f);
          IxScN<Ix4, NS> with;
          with.r = row;
          with.c = f - row_lo;
          static_for<0, N>([&](auto ic) {
            constexpr int s = decltype(ic)::value;
            constexpr CNode sn = CL::c.nodes[s];
            if constexpr (is_scan_root(sn)) {
              constexpr int o = scan_ord<CL>(s);
              using Run = Running<sn.fn, sn.dtype>;
              const uint32_t base = Run::narrow(Run::add(Run::from(carry[o]), Run::of(before[o][j])));
              uint32_t run = identity_of<sn.fn, sn.dtype>();
#pragma unroll
              for (int ee = 0; ee < 4; ++ee) {
                const int e = REV ? 3 - ee : ee;
                const uint32_t earlier = run;
                run = combine<sn.fn, sn.dtype>(run, v[o][j].v[e]);
                with.sv[o].v[e] = combine<sn.fn, sn.dtype>(base, sn.p0 == 1 ? earlier : run);
              }
            }
          });
          static_for<0, N>([&](auto ic) {
            constexpr int k = decltype(ic)::value;
            if constexpr (is_ring_output(CL::c.nodes[k])) {
              uint32_t* dst = reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[k].ptr));
              if (decltype(safe_c)::value || inside == 15u) {
                V4 x;
                if constexpr (is_scan_root(CL::c.nodes[k])) x = with.sv[scan_ord<CL>(k)];
                else x = eval<CL, k>(a, with);
                if (inside == 15u) {
                  *reinterpret_cast<uint4*>(dst + f) = make_uint4(x.v[0], x.v[1], x.v[2], x.v[3]);
                } else {
#pragma unroll
                  for (int e = 0; e < 4; ++e)
                    if ((inside >> e) & 1u) dst[f + e] = x.v[e];
                }
              } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if ((inside >> e) & 1u) {
                    IxScN<Ix, NS> one;
                    one.r = row;
                    one.c = f + e - row_lo;
#pragma unroll
                    for (int o = 0; o < NS; ++o) one.sv[o] = with.sv[o].v[e];
                    if constexpr (is_scan_root(CL::c.nodes[k])) dst[f + e] = one.sv[scan_ord<CL>(k)];
                    else dst[f + e] = eval<CL, k>(a, one);
                  }
              }
            }
          });
        }
      };
      if (whole) results(std::true_type{}, std::true_type{});
      else if (any && safe) results(std::false_type{}, std::true_type{});
      else if (any) results(std::false_type{}, std::false_type{});
      if constexpr (WARPS == 1) {
        static_for<0, N>([&](auto ic) {
          constexpr int s = decltype(ic)::value;
          constexpr CNode sn = CL::c.nodes[s];
          if constexpr (is_scan_root(sn)) {
            constexpr int o = scan_ord<CL>(s);
            using Run = Running<sn.fn, sn.dtype>;
            carry[o] = Run::bits(Run::add(Run::from(carry[o]), Run::of(total[o])));
          }
        });
      }
    }
  }
}

}  // namespace dev
}  // namespace acc
