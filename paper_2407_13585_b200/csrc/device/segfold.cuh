// k_segfold: the skeleton for clusters whose roots are segmented folds over one offsets
// array:  ys[s] = fold(op) of xs[off[s] .. off[s+1]),  xs evaluated in registers from the
// fused producers.
//
// The work is cut by elements, not by segments, so that a few very long segments among many
// short ones (skewed lengths) cost what their elements cost:
//
//  * a warp owns kSegRun consecutive elements and walks them 512 at a time, without a barrier: the
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
// (Before, a block walked tiles of 4096 elements with ten barriers each, about 800 instructions per
// thread where a tile held several segments, and sources without 128-bit rows went through shared
// memory element by element.  2^27 elements, a sum and a maximum: 2^20 segments of
// Zipf lengths 243 -> 178 us, 2^15 segments 184 -> 143, 2^24 segments 450 -> 413; 10^6 elements in 10^4 segments 42.5 ->
// 16.5.  What bounds it now is latency: a warp's step waits for its loads, then for the scan's shuffles, with 42 % of the issue
// slots used.)
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
// then `tail`, of 2 + NF words each: segment id + 1 (0: no record), unused, one value per fold.
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

template <class CL, bool VEC>
__global__ void __launch_bounds__(kBlock, kSegResident) k_segfold(const __grid_constant__ Args<CL::c.n> a, int run_length) {
  constexpr int N = CL::c.n;
  constexpr int F = first_segfold<CL>();
  constexpr int NF = count_if<CL>(is_segfold_root);
  constexpr int WARPS = kBlock / 32, ROWS = 4, STEP = kSegStep;
  constexpr int REC = 2 + NF;
  __shared__ uint32_t bits[WARPS][STEP / 32];                    // bit p: element p of the warp's step begins a segment
  __shared__ __align__(16) uint32_t staged[WARPS][32 * kSegStride];   // a step's operands, then the value of every prefix within its lane
  // what a warp leaves for the block: the segment that is open at its end and its value there, and, where a segment begins
  // in the warp's run, that segment and the value of the one that ends at the first start
  __shared__ int open_seg[WARPS], first_seg[WARPS];              // first_seg: -1 if none begins; open_seg -1: no elements
  __shared__ bool has_head[WARPS];                               // the segment that ends at the first start has elements in the run
  __shared__ uint32_t open_val[NF][WARPS], head_val[NF][WARPS];
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
  if (lo0 < hi0) {                                               // uniform
    // the elements of a step; what lies outside [lo0, hi0) reads as the operator's identity
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
            const V4 v = eval<CL, nd.in[0]>(a, Ix4{0, min(base + (j * 32 + lane) * 4, last)});
#pragma unroll
            for (int e = 0; e < 4; ++e) x[j][e] = v.v[e];
          }
        }
        if (!whole) {
#pragma unroll
          for (int j = 0; j < ROWS; ++j) {
            const int c = base + (j * 32 + lane) * 4;
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
            const int p = base + (j * 32 + lane) * 4 + e;
            x[j][e] = p >= lo0 && p < hi0 ? eval<CL, nd.in[0]>(a, Ix{0, p}) : identity_of<nd.fn, nd.dtype>();
          }
      }
    };
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
    for (int base = (int)run_lo; base < hi0; base += STEP) {
      if (base + STEP <= lo0) continue;
      if constexpr (VEC) {
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
      uint32_t x[N][ROWS][4];
      static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (is_segfold_root(CL::c.nodes[i])) operands(ic, base, x[i]);
      });
      if constexpr (VEC) {                                       // the next step's lines, asked into L2
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
#pragma unroll
            for (int j = 0; j < ROWS; ++j)
              fold_step<nd.fn, nd.dtype>(acc[i], comp[i], combine<nd.fn, nd.dtype>(combine<nd.fn, nd.dtype>(x[i][j][0], x[i][j][1]),
                                                                                   combine<nd.fn, nd.dtype>(x[i][j][2], x[i][j][3])));
          }
        });
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
#pragma unroll
          for (int j = 0; j < ROWS; ++j) {
            const int q = j * 32 + lane;                          // chunk of four: the (q % 4)-th of lane q / 4
            *reinterpret_cast<uint4*>(mine + (q >> 2) * kSegStride + (q & 3) * 4) = make_uint4(x[i][j][0], x[i][j][1], x[i][j][2], x[i][j][3]);
          }
          __syncwarp();
          uint32_t run = identity_of<nd.fn, nd.dtype>();
          uint32_t* own = mine + lane * kSegStride;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint4 v = *reinterpret_cast<const uint4*>(own + 4 * c);
            v.x = run = ((b >> (4 * c + 0)) & 1u) ? v.x : combine<nd.fn, nd.dtype>(run, v.x);
            v.y = run = ((b >> (4 * c + 1)) & 1u) ? v.y : combine<nd.fn, nd.dtype>(run, v.y);
            v.z = run = ((b >> (4 * c + 2)) & 1u) ? v.z : combine<nd.fn, nd.dtype>(run, v.z);
            v.w = run = ((b >> (4 * c + 3)) & 1u) ? v.w : combine<nd.fn, nd.dtype>(run, v.w);
            *reinterpret_cast<uint4*>(own + 4 * c) = v;
          }
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, run, d);
            if (lane - d >= lower) run = combine<nd.fn, nd.dtype>(u, run);
          }
          uint32_t into = __shfl_up_sync(0xFFFFFFFFu, run, 1);    // what runs into the lane's elements
          if (lane == 0) into = open[i];
          else if (led) into = combine<nd.fn, nd.dtype>(open[i], into);
          own[16] = into;                                         // (a word of the lane's padding)
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
