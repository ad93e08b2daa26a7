// k_segfold: the skeleton for clusters whose roots are segmented folds over one offsets
// array:  ys[s] = fold(op) of xs[off[s] .. off[s+1]),  xs evaluated in registers from the
// fused producers.
//
// The work is cut by elements, not by segments, so that a few very long segments among many
// short ones (skewed lengths) cost what their elements cost:
//
//  * a warp owns up to kSegMaxRun consecutive elements (seg_run) and walks them 512 at a time, without a barrier: the
//    warps of a block meet once, at the end;
//  * where no segment begins among the 512, every lane adds its elements to a compensated running
//    value of its own;
//  * otherwise the offsets that fall among them become bits, the operands go through shared memory so
//    that a lane holds 16 consecutive ones, and a segmented scan (inside the lane, then once across the
//    warp by shuffles that stop at a lane holding a start) leaves the value of every prefix there; a
//    lane per start then takes the value in front of it, which is the segment that ends;
//  * a segment that crosses warps is put together by one thread of the block (fp32 sums in fp64); one
//    that crosses blocks leaves a record per block (the part after its start: `tail`; a part that
//    continues one begun earlier: `head`), and a second, small launch (k_segfold_across) combines the
//    records in block order.
//
// (A block that walked tiles of 4096 elements with ten barriers each took 243 us for a sum and a maximum of 2^27 elements in 2^20
// segments of Zipf lengths, 184 in 2^15 segments, 450 in 2^24, 42.5 for 10^6 in 10^4.  Warps on their own, with loads into
// registers ahead of a step's work, 176, 144, 407 and 17.1; with operands that land in shared memory two steps ahead, below, and
// without records cleared beforehand, 156, 130, 405 and 13.7: 53 % of the issue slots, the rest mostly a warp's waits for offsets
// and for the shuffles of its scan.)
//
// Several segmented folds of one cluster (say a sum and a maximum over the same segments) share
// the walk.  Results do not depend on timing: every order of combination is fixed by the layout.
//
// Offsets are data, so they are checked here, every one of them: a segment that leaves the
// source is reported as ACC_ERR_INDEX_RANGE, an empty or descending one as ACC_ERR_SHAPE (a fold
// without a seed has no value for it).
#pragma once
#include "scanring.cuh"
#include "skeletons.cuh"

namespace acc {
namespace dev {

constexpr int kSegStep = 512;                  // elements of a warp's step
constexpr int kSegMaxRun = 4096;               // consecutive elements of a warp, at most: what amortises finding its first segment
constexpr int kSegStride = 20;                 // words a lane's 16 elements take in shared memory: an odd multiple of 16 bytes, no bank conflicts
// ... without room to spare, where operands land: a lane's 16 elements side by side, chunks of four swapped so that eight lanes
// that read theirs 128 bits at a time meet no bank twice.  Word of chunk c of lane l:
__device__ __forceinline__ int seg_chunk(int l, int c) { return l * 16 + ((c ^ ((l >> 1) & 3)) << 2); }
constexpr int kSegResident = 4;                // blocks per SM the kernel is built for (5: 191 -> 257 us for 2^27 elements)
// Elements of a warp's run: what leaves the fewest steps (2 to 3 us each, mostly latency) to the blocks that an SM's places see
// one after another, counting one for finding a run's first segment.  As many steps as fit the first time round, which leaves
// a last round nearly empty, took 49.9 against 48.5 us for 2 * 10^7 elements in 20000 segments, 215.6 against 211 for
// 6 * 10^7 in 7 * 10^6; runs of up to 2048 or 8192 elements 216 and 192 against 191 for 2^27 Zipf lengths, 211 and 252 for
// 6 * 10^7.
inline int seg_run(int64_t n, int sms) {
  int64_t best = 1, best_cost = INT64_MAX;
  for (int64_t steps = 1; steps <= kSegMaxRun / kSegStep; ++steps) {
    const int64_t span = steps * kSegStep * (kBlock / 32), blocks = (n + span - 1) / span, at_once = (int64_t)sms * kSegResident;
    const int64_t cost = (blocks + at_once - 1) / at_once * (steps + 1);
    if (cost < best_cost) { best = steps; best_cost = cost; }
  }
  return (int)best * kSegStep;
}

template <class CL> constexpr int first_segfold() {
  for (int i = 0; i < CL::c.n; ++i)
    if (is_segfold_root(CL::c.nodes[i])) return i;
  return -1;
}

// All segmented folds of the cluster must read one offsets array, and nothing else may be a root.
template <class CL> constexpr bool segfold_eligible() {
  const int f = first_segfold<CL>();
  if (f < 0) return false;
  for (int i = 0; i < CL::c.n; ++i) {
    const CNode& n = CL::c.nodes[i];
    if (is_store_root(n) || is_fold_root(n) || is_scan_root(n) || is_permute_root(n)) return false;
    if (is_segfold_root(n) && n.in[1] != CL::c.nodes[f].in[1]) return false;
  }
  return true;
}

// Scratch of k_segfold (32-bit words): from word 4 two records per block, `head`
// then `tail`, of 2 + NF words each: segment id + 1 (0: no record), unused, one value per fold.  Every block writes its own.
__host__ __device__ inline int seg_record_words(int n_folds) { return 2 + n_folds; }
__host__ __device__ inline int64_t seg_scratch_words(int n_folds, int grid) { return 4 + (int64_t)grid * 2 * seg_record_words(n_folds); }

// Largest s in [0, S) with off[s] <= x, for off[0] <= x < off[S] (any s for other x): a 32-way search by one warp.
__device__ __forceinline__ int seg_containing(const int32_t* off, int S, int x, int lane) {
  int lo = 0, hi = S;                                          // off[lo] <= x < off[hi]
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32;
    const int p = lo + (lane + 1) * step;
    const bool ok = p < hi && __ldg(off + p) <= x;             // true for a prefix of the lanes
    const int k = __popc(__ballot_sync(0xFFFFFFFFu, ok));
    const int nlo = lo + k * step;
    hi = min(hi, nlo + step);
    lo = nlo;
  }
  return lo;
}

// ---- operands that land in shared memory before they are wanted ------------------------------------------------
// Several folds whose operands are computed from one array, element by element, have a warp's next two steps of that array under way
// in asynchronous copies, straight to where a lane finds its 16 consecutive elements: no step waits for memory, no operand is
// written to shared memory to be read again in another order, and no registers hold what another fold will need.  Two steps of
// 2 KB a warp are what four blocks per SM have room for; three steps and three blocks 174 against 156 us (2^27 elements,
// Zipf lengths).  The search for a run's first segment comes behind the first copies: in front of them 50.2 -> 50.6 us for 5 * 10^7
// elements in 16 segments, 53.4 -> 54.5 in 5000, 19.0 -> 20.0 for 5 * 10^6 in 10^4, but 186.9 -> 186.8 for 2^27 in 2.7 * 10^6.
// One fold alone takes its operands through registers: it has them all before it begins, and the 128 KB per SM that copies would
// land in are worth more as L1 to the offsets, which are read three times (us, landed / registers: 2^27 elements in segments of 4
// 428 / 397, of 16 193 / 179, of 500 101 / 102; 5 * 10^7 in segments of 2.5 248 / 232, of 500 46.4 / 48.0; 2 * 10^7 in 6 segments
// 23.6 / 19.4).
struct IxLd4 { int r, c; const uint32_t* landed; };                 // four consecutive elements, and where their array's lie
__device__ __forceinline__ Ix lane(const IxLd4& i, int j) { return Ix{i.r, i.c + j}; }
template <int F, int P0 = kRunTime, int P1 = kRunTime>
__device__ __forceinline__ auto map_index(const IxLd4& i, const NodeArg&, const NodeArg&) {
  static_assert(F == ACC_IDX_IDENTITY, "operands that land ahead are read in place");
  return i;
}
template <class CL, int I, class A> __device__ __forceinline__ V4 ld_ext(const A&, const IxLd4& ix) {
  const uint4 v = *reinterpret_cast<const uint4*>(ix.landed);
  return V4{{v.x, v.y, v.z, v.w}};
}
// the one array that member i is computed from, element by element; -1: none yet, -2: anything else
template <class CL> constexpr int seg_array_below(int i, int so_far) {
  const CNode& n = CL::c.nodes[i];
  if (so_far == -2) return -2;
  if (!n.member) return n.rank == 1 && (so_far == -1 || so_far == i) ? i : -2;
  if (n.kind == ACC_GENERATE) return so_far;
  if (n.kind != ACC_MAP && n.kind != ACC_ZIPWITH && (n.kind != ACC_BACKPERMUTE || n.idxfn != ACC_IDX_IDENTITY)) return -2;
  for (int k = 0; k < n.narr; ++k) so_far = seg_array_below<CL>(n.in[k], so_far);
  return so_far;
}
template <class CL> constexpr int seg_landing_array() {
  if (count_if<CL>(is_segfold_root) < 2) return -2;
  int x = -1;
  for (int i = 0; i < CL::c.n; ++i)
    if (is_segfold_root(CL::c.nodes[i])) x = seg_array_below<CL>(CL::c.nodes[i].in[0], x);
  return x;
}
constexpr int kSegAhead = 2;                   // steps whose copies are under way
template <class CL, bool VEC> constexpr size_t seg_landing_bytes() { return VEC && seg_landing_array<CL>() >= 0 ? (size_t)kSegAhead * kSegStep * 4 * (kBlock / 32) : 0; }

template <class CL, bool VEC>
__global__ void __launch_bounds__(kBlock, kSegResident) k_segfold(const __grid_constant__ Args<CL::c.n> a, int run_length) {
  constexpr int N = CL::c.n;
  constexpr int F = first_segfold<CL>();
  constexpr int NF = count_if<CL>(is_segfold_root);
  constexpr int WARPS = kBlock / 32, ROWS = 4, STEP = kSegStep;
  constexpr int REC = 2 + NF;
  __shared__ uint32_t bits[WARPS][STEP / 32];                    // bit p: element p of the warp's step begins a segment
  __shared__ __align__(16) uint32_t staged[WARPS][32 * kSegStride];   // the value of every prefix within its lane (before that a step's operands, if they do not land ahead)
  // what a warp leaves for the block: the segment that is open at its end and its value there, and, where a segment begins
  // in the warp's run, that segment and the value of the one that ends at the first start
  __shared__ int open_seg[WARPS], first_seg[WARPS];              // first_seg: -1 if none begins; open_seg -1: no elements
  __shared__ bool has_head[WARPS];                               // the segment that ends at the first start has elements in the run
  __shared__ uint32_t open_val[NF][WARPS], head_val[NF][WARPS];
  constexpr int LAND = VEC ? seg_landing_array<CL>() : -2;         // the array that lands ahead
  extern __shared__ __align__(16) uint32_t landing_smem[];       // [warp][step % kSegAhead][STEP]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int S = a.C;                                             // segments
  constexpr int OFF = CL::c.nodes[F].in[1], SRC = CL::c.nodes[F].in[0];
  const int32_t* off = reinterpret_cast<const int32_t*>(a.n[OFF].ptr);
  const int n_src = a.n[SRC].R * a.n[SRC].C;
  uint32_t* rec = a.scratch + 4;
  auto fold_slot_of = [](int i) { return count_if<CL>(is_segfold_root, i); };

  // every offset is looked at once, whatever the walk below does with it
  for (int s = blockIdx.x * kBlock + threadIdx.x; s < S; s += gridDim.x * kBlock) {
    const int lo = __ldg(off + s), hi = __ldg(off + s + 1);
    if (lo < 0 || hi > n_src) raise_status(a, kStatusIndex);
    else if (hi <= lo) raise_status(a, kStatusEmptySegment);
  }

  const int e_lo = max(__ldg(off), 0), e_hi = min(__ldg(off + S), n_src);   // elements that belong to segments
  const int64_t run_lo = ((int64_t)blockIdx.x * WARPS + warp) * run_length;
  const int lo0 = (int)(run_lo > e_lo ? run_lo : e_lo), hi0 = (int)(run_lo + run_length < e_hi ? run_lo + run_length : e_hi);
  if (lane == 0) { open_seg[warp] = -1; first_seg[warp] = -1; }
  if (threadIdx.x < 2) rec[((size_t)blockIdx.x * 2 + threadIdx.x) * REC] = 0;    // no record yet (nobody clears them beforehand)
  if (lo0 < hi0) {                                               // uniform
    uint32_t* const landing = landing_smem + (size_t)warp * kSegAhead * STEP;
    int slot = 0;                                                // of the step that is worked on
    auto land = [&](int base) {                                  // (a group is closed for every step, so that they can be counted)
      if constexpr (LAND >= 0) {
        const int last = (n_src & ~3) - 4;
        if (base < hi0 && last >= 0) {
          const uint32_t* src = reinterpret_cast<const uint32_t*>(a.n[LAND].ptr);
          const uint32_t to = (uint32_t)__cvta_generic_to_shared(landing + slot * STEP);
#pragma unroll
          for (int j = 0; j < ROWS; ++j) {
            const int q = j * 32 + lane;                         // chunk of the step
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + seg_chunk(q >> 2, q & 3) * 4), "l"(src + min(base + q * 4, last)) : "memory");
          }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    };
    // the elements of a step; what lies outside [lo0, hi0) reads as the operator's identity.  A lane takes chunks of four:
    // those of its 16 consecutive elements where they have landed, else every 32nd.
    auto chunk_begin = [&](int base, int j) { return base + (LAND >= 0 ? lane * 16 + j * 4 : (j * 32 + lane) * 4); };
    auto operands = [&](auto ic, int base, uint32_t (&x)[ROWS][4]) {
      constexpr int i = decltype(ic)::value;
      constexpr CNode nd = CL::c.nodes[i];
      if constexpr (VEC) {
        // (chunks outside the array read its last whole chunk instead, without a branch: a load whose value is used inside a
        // branch is waited for before the next one is issued)
        const int last = (n_src & ~3) - 4;
        const bool whole = base >= lo0 && base + STEP <= hi0;     // uniform
        if (last >= 0) {
#pragma unroll
          for (int j = 0; j < ROWS; ++j) {
            const int c = chunk_begin(base, j);
            V4 v;
            if constexpr (LAND >= 0) v = eval<CL, nd.in[0]>(a, IxLd4{0, c, landing + slot * STEP + seg_chunk(lane, j)});
            else v = eval<CL, nd.in[0]>(a, Ix4{0, min(c, last)});
#pragma unroll
            for (int e = 0; e < 4; ++e) x[j][e] = v.v[e];
          }
        }
        if (!whole) {
#pragma unroll
          for (int j = 0; j < ROWS; ++j) {
            const int c = chunk_begin(base, j);
            if (c > last && c < n_src) {                         // the array's last few elements
#pragma unroll
              for (int e = 0; e < 3; ++e)
                if (c + e < n_src) x[j][e] = eval<CL, nd.in[0]>(a, Ix{0, c + e});
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (c + e < lo0 || c + e >= hi0) x[j][e] = identity_of<nd.fn, nd.dtype>();
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < ROWS; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int p = chunk_begin(base, j) + e;
            x[j][e] = p >= lo0 && p < hi0 ? eval<CL, nd.in[0]>(a, Ix{0, p}) : identity_of<nd.fn, nd.dtype>();
          }
      }
    };
    const int base0 = (int)run_lo + (lo0 - (int)run_lo) / STEP * STEP;   // the first step with elements of a segment
    if constexpr (LAND >= 0) {
#pragma unroll
      for (slot = 0; slot < kSegAhead; ++slot) land(base0 + slot * STEP);
      slot = 0;
    }
    const int s0 = seg_containing(off, S, lo0, lane);
    int next = __ldg(off + s0) == lo0 ? s0 : s0 + 1;             // the next segment to begin
    const int first = next;
    const bool starts_with_run = __ldg(off + s0) == lo0;
    // where segments next .. next + 32 * AHEAD - 1 begin: enough for a step of short segments, loaded while the step before is
    // worked on (a refill within the step is a wait)
    constexpr int AHEAD = 3;
    int o[AHEAD];
    auto refill = [&](int from) {
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) o[u] = from + 32 * u + lane < S ? __ldg(off + from + 32 * u + lane) : 0x7FFFFFFF;
    };
    refill(next);
    uint32_t acc[N], open[N];                                    // the open segment: this lane's share of rows without a start, and the rest
    float comp[N] = {};
    uint32_t head[N];                                            // (in the lane that finds it)
    bool found_head = false;
    static_for<0, N>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr CNode nd = CL::c.nodes[i];
      if constexpr (is_segfold_root(nd)) acc[i] = open[i] = identity_of<nd.fn, nd.dtype>();
    });
    for (int base = base0; base < hi0; base += STEP) {
      if constexpr (VEC && LAND < 0) {
        // steps far inside a long segment, two at a time: twice the loads under way (2^24 elements in one segment 24.6 -> 20.6 us,
        // 2^27 Zipf lengths 189 -> 178)
        while (base + 2 * STEP <= hi0 && base >= lo0 && __shfl_sync(0xFFFFFFFFu, o[0], 0) >= base + 2 * STEP) {
          uint32_t q[N][2 * ROWS];                                // a chunk of four each
          static_for<0, N>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            constexpr CNode nd = CL::c.nodes[i];
            if constexpr (is_segfold_root(nd)) {
              V4 v[2 * ROWS];
#pragma unroll
              for (int j = 0; j < 2 * ROWS; ++j) v[j] = eval<CL, nd.in[0]>(a, Ix4{0, base + (j * 32 + lane) * 4});
#pragma unroll
              for (int j = 0; j < 2 * ROWS; ++j)
                q[i][j] = combine<nd.fn, nd.dtype>(combine<nd.fn, nd.dtype>(v[j].v[0], v[j].v[1]), combine<nd.fn, nd.dtype>(v[j].v[2], v[j].v[3]));
            }
          });
          static_for<0, N>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            constexpr CNode nd = CL::c.nodes[i];
            if constexpr (is_segfold_root(nd)) {
#pragma unroll
              for (int j = 0; j < 2 * ROWS; ++j) fold_step<nd.fn, nd.dtype>(acc[i], comp[i], q[i][j]);
            }
          });
          base += 2 * STEP;
        }
        if (base >= hi0) break;
      }
      uint32_t x[LAND >= 0 ? 1 : N][ROWS][4];                     // (of one fold after another where they have landed)
      auto ahead = [&]() {                                        // every lane has its last values of the step: its room goes to a later one
        if constexpr (LAND >= 0) {
          __syncwarp();
          land(base + kSegAhead * STEP);
          slot = slot + 1 == kSegAhead ? 0 : slot + 1;
        }
      };
      if constexpr (LAND >= 0) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kSegAhead - 1) : "memory");
        __syncwarp();
      } else {
        static_for<0, N>([&](auto ic) {
          constexpr int i = decltype(ic)::value;
          if constexpr (is_segfold_root(CL::c.nodes[i])) operands(ic, base, x[i]);
        });
      }
      if constexpr (VEC && LAND < 0) {                                       // the next step's lines, asked into L2
        if (base + 2 * STEP <= hi0 && (lane & 7) == 0) {
          static_for<0, N>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            if constexpr (is_segfold_root(CL::c.nodes[i])) {
#pragma unroll
              for (int j = 0; j < ROWS; ++j) eval<CL, CL::c.nodes[i].in[0]>(a, IxPF4{0, base + STEP + (j * 32 + lane) * 4});
            }
          });
        }
      }
      const int step_hi = min(base + STEP, hi0);
      if (__shfl_sync(0xFFFFFFFFu, o[0], 0) >= step_hi) {            // uniform: the step belongs to the open segment
        static_for<0, N>([&](auto ic) {
          constexpr int i = decltype(ic)::value;
          constexpr CNode nd = CL::c.nodes[i];
          if constexpr (is_segfold_root(nd)) {
            constexpr int at = LAND >= 0 ? 0 : i;
            if constexpr (LAND >= 0) operands(ic, base, x[at]);
#pragma unroll
            for (int j = 0; j < ROWS; ++j)
              fold_step<nd.fn, nd.dtype>(acc[i], comp[i], combine<nd.fn, nd.dtype>(combine<nd.fn, nd.dtype>(x[at][j][0], x[at][j][1]),
                                                                                   combine<nd.fn, nd.dtype>(x[at][j][2], x[at][j][3])));
          }
        });
        ahead();
        continue;
      }
      if (lane < STEP / 32) bits[warp][lane] = 0;
      __syncwarp();
      int begun = 0;                                             // segments that begin in this step
      for (bool more = true; more;) {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
          const unsigned beyond = __ballot_sync(0xFFFFFFFFu, o[u] >= step_hi);
          const int k = !more ? 0 : beyond ? __ffs(beyond) - 1 : 32;   // (offsets behind one beyond the step do not count, whatever they are)
          if (lane < k && o[u] >= base) atomicOr(&bits[warp][(o[u] - base) >> 5], 1u << ((o[u] - base) & 31));
          begun += k;
          more = more && k == 32;
        }
        refill(next + begun);
      }
      __syncwarp();
      const uint32_t b = (bits[warp][lane >> 1] >> ((lane & 1) * 16)) & 0xFFFFu;   // starts among the lane's 16 elements
      const unsigned H = __ballot_sync(0xFFFFFFFFu, b != 0);
      const unsigned upto = H & (0xFFFFFFFFu >> (31 - lane));
      const int lower = upto ? 31 - __clz(upto) : 0;             // the segment open at the lane's end began in that lane, or before the step
      const bool led = (H & ((1u << lane) - 1u)) == 0;           // no start in earlier lanes
      static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr CNode nd = CL::c.nodes[i];
        if constexpr (is_segfold_root(nd)) {
          uint32_t t = acc[i];                                    // the lanes' shares of the open segment
#pragma unroll
          for (int d = 16; d > 0; d >>= 1) t = combine<nd.fn, nd.dtype>(t, __shfl_xor_sync(0xFFFFFFFFu, t, d));
          open[i] = combine<nd.fn, nd.dtype>(open[i], t);
          acc[i] = identity_of<nd.fn, nd.dtype>();
          comp[i] = 0.0f;
          uint32_t* mine = staged[warp];
          constexpr int at = LAND >= 0 ? 0 : i;
          if constexpr (LAND >= 0) {
            operands(ic, base, x[at]);
            if constexpr (count_if<CL>(is_segfold_root, i + 1) == NF) ahead();   // (the last fold)
          } else {
#pragma unroll
            for (int j = 0; j < ROWS; ++j) {
              const int q = j * 32 + lane;                        // chunk of four: the (q % 4)-th of lane q / 4
              *reinterpret_cast<uint4*>(mine + (q >> 2) * kSegStride + (q & 3) * 4) = make_uint4(x[at][j][0], x[at][j][1], x[at][j][2], x[at][j][3]);
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < ROWS; ++j) {
              const uint4 v = *reinterpret_cast<const uint4*>(mine + lane * kSegStride + j * 4);
              x[at][j][0] = v.x; x[at][j][1] = v.y; x[at][j][2] = v.z; x[at][j][3] = v.w;
            }
          }
          uint32_t run = identity_of<nd.fn, nd.dtype>();
#pragma unroll
          for (int c = 0; c < 4; ++c) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint32_t v = x[at][c][e];
              x[at][c][e] = run = ((b >> (4 * c + e)) & 1u) ? v : combine<nd.fn, nd.dtype>(run, v);
            }
            *reinterpret_cast<uint4*>(mine + lane * kSegStride + c * 4) = make_uint4(x[at][c][0], x[at][c][1], x[at][c][2], x[at][c][3]);
          }
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, run, d);
            if (lane - d >= lower) run = combine<nd.fn, nd.dtype>(u, run);
          }
          uint32_t into = __shfl_up_sync(0xFFFFFFFFu, run, 1);    // what runs into the lane's elements
          if (lane == 0) into = open[i];
          else if (led) into = combine<nd.fn, nd.dtype>(open[i], into);
          mine[lane * kSegStride + 16] = into;                    // (a word of the lane's padding)
          open[i] = __shfl_sync(0xFFFFFFFFu, run, 31);            // (some segment begins in the step, so this began in it)
          __syncwarp();
          // a lane per start: the segment before it ends in front of it
          uint32_t* out = reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[i].ptr));
          for (int k = lane; k < begun; k += 32) {
            const int seg = next + k, pos = __ldg(off + seg) - base;
            if (pos < 0 || pos >= STEP) continue;                 // (offsets that descend)
            uint32_t v;
            if (pos == 0) {
              v = mine[16];
            } else {
              const int l = (pos - 1) >> 4, e = (pos - 1) & 15;
              const uint32_t lb = (bits[warp][l >> 1] >> ((l & 1) * 16)) & ((2u << e) - 1u);   // starts in that lane up to the element
              v = mine[l * kSegStride + e];
              if (lb == 0) v = combine<nd.fn, nd.dtype>(mine[l * kSegStride + 16], v);
            }
            if (seg == first) { head[i] = v; found_head = true; }
            else out[seg - 1] = v;
          }
          __syncwarp();                                           // (the next fold, or step, writes there)
        }
      });
      next += begun;
    }
    if constexpr (LAND >= 0) asm volatile("cp.async.wait_all;" ::: "memory");
    static_for<0, N>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr CNode nd = CL::c.nodes[i];
      if constexpr (is_segfold_root(nd)) {
        uint32_t t = acc[i];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) t = combine<nd.fn, nd.dtype>(t, __shfl_xor_sync(0xFFFFFFFFu, t, d));
        if (lane == 0) open_val[fold_slot_of(i)][warp] = combine<nd.fn, nd.dtype>(open[i], t);
      }
    });
    if (found_head) {                                             // (one lane's)
      static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (is_segfold_root(CL::c.nodes[i])) head_val[fold_slot_of(i)][warp] = head[i];
      });
    }
    if (lane == 0) {
      open_seg[warp] = next - 1;
      first_seg[warp] = next > first ? first : -1;
      has_head[warp] = !starts_with_run && first > 0;
    }
  }
  __syncthreads();

  // segments that cross warps: one thread per fold goes over the warps in order
  if (threadIdx.x < NF) {
    static_for<0, N>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr CNode nd = CL::c.nodes[i];
      if constexpr (is_segfold_root(nd)) {
        const int f = fold_slot_of(i);
        if ((int)threadIdx.x != f) return;
        using Run = Running<nd.fn, nd.dtype>;
        uint32_t* out = reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[i].ptr));
        uint32_t* head = rec + (size_t)blockIdx.x * 2 * REC;
        uint32_t* tail = head + REC;
        auto value = Run::identity();
        int seg = -1;                                             // the open segment; -1: nothing of one in this block yet
        bool from_here = false, any = false;
        auto close = [&]() {
          if (seg < 0 || seg >= S || !any) return;
          if (from_here) { out[seg] = Run::narrow(value); return; }
          head[0] = (uint32_t)seg + 1u;
          head[2 + f] = Run::narrow(value);
        };
        for (int w = 0; w < WARPS; ++w) {
          if (open_seg[w] < 0 && first_seg[w] < 0) continue;      // (a run without elements)
          if (first_seg[w] >= 0) {
            if (has_head[w]) {
              if (!any) { seg = first_seg[w] - 1; any = true; }
              value = Run::add(value, Run::of(head_val[f][w]));
            }
            close();
            seg = open_seg[w];
            value = Run::of(open_val[f][w]);
            from_here = any = true;
          } else {
            if (!any) { seg = open_seg[w]; any = true; }
            value = Run::add(value, Run::of(open_val[f][w]));
          }
        }
        if (any) {
          const int64_t block_hi = (int64_t)(blockIdx.x + 1) * WARPS * run_length;
          if (e_hi <= block_hi) {
            close();                                              // the last segment ends in this block
          } else {
            uint32_t* r = from_here ? tail : head;
            if (seg >= 0 && seg < S) {
              r[0] = (uint32_t)seg + 1u;
              r[2 + f] = Run::narrow(value);
            }
          }
        }
      }
    });
  }
}

// Second launch of a segmented-fold cluster: segments that cross the blocks of k_segfold.  A warp per block
// that left a `tail` (the part of a segment after its start): its lanes look at the blocks that follow, 32 at a
// time, take the `head` records that continue the segment, and combine them in a fixed order.
template <class CL>
__global__ void __launch_bounds__(kBlock) k_segfold_across(const __grid_constant__ Args<CL::c.n> a, int n_blocks) {
  constexpr int N = CL::c.n;
  constexpr int NF = count_if<CL>(is_segfold_root);
  constexpr int REC = 2 + NF;
  auto fold_slot_of = [](int i) { return count_if<CL>(is_segfold_root, i); };
  const int lane = threadIdx.x & 31;
  const int b = blockIdx.x * (kBlock / 32) + ((int)threadIdx.x >> 5);
  if (b >= n_blocks) return;
  const uint32_t* rec = a.scratch + 4;
  const uint32_t* tail = rec + ((size_t)b * 2 + 1) * REC;
  const uint32_t key = tail[0];
  if (key == 0) return;                                          // the same for the whole warp
  uint32_t v[N];
  static_for<0, N>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (is_segfold_root(CL::c.nodes[i])) v[i] = tail[2 + fold_slot_of(i)];
  });
  // G times 32 blocks from `base` on, all of whose records are asked for together; whether the segment goes on behind them
  auto go_on = [&](auto groups_c, int base) {
    constexpr int G = decltype(groups_c)::value;
    bool same[G];
    uint32_t x[N][G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int b2 = base + 32 * g + lane;
      const uint32_t* head = rec + (size_t)min(b2, n_blocks - 1) * 2 * REC;
      same[g] = b2 < n_blocks && head[0] == key;
      static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (is_segfold_root(CL::c.nodes[i])) x[i][g] = head[2 + fold_slot_of(i)];
      });
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const unsigned others = ~__ballot_sync(0xFFFFFFFFu, same[g]);
      const int n = others ? __ffs(others) - 1 : 32;             // blocks of these 32 that continue the segment
      static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr CNode nd = CL::c.nodes[i];
        if constexpr (is_segfold_root(nd))
          v[i] = combine<nd.fn, nd.dtype>(v[i], warp_reduce<nd.fn, nd.dtype>(lane < n ? x[i][g] : identity_of<nd.fn, nd.dtype>()));
      });
      if (n < 32) return false;
    }
    return base + 32 * G < n_blocks;
  };
  // (few segments cross more than 33 blocks; those that do may cross all of them: 2^27 elements in one segment, 4096 records,
  // 156 -> 133 us)
  if (b + 1 < n_blocks && go_on(std::integral_constant<int, 1>{}, b + 1)) {
    int base = b + 33;
    while (go_on(std::integral_constant<int, 8>{}, base)) base += 8 * 32;
  }
  if (lane == 0) {
    static_for<0, N>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if constexpr (is_segfold_root(CL::c.nodes[i])) reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[i].ptr))[key - 1] = v[i];
    });
  }
}

}  // namespace dev
}  // namespace acc
