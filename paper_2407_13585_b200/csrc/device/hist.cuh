// k_hist: the skeleton for a cluster whose permute is an fp32 '+' scatter into few enough
// bins to keep them on chip.
//
// Measured on B200 (2^27 Zipf-skewed keys): shared-memory integer atomics sustain about
// 1000 G updates/s, fp32 shared-memory atomics about 56 G/s (they retry on every collision,
// and a hot bin collides all the time), atomics into a partner CTA's shared memory 140 G/s.
// So the bins are 32-bit *integers* in the CTA's own shared memory:
//
//  * a value x is added as the integer x * 2^S when that product is an integer of magnitude
//    below `cap` -- exact, one fire-and-forget native atomic.  `cap` is 2^31 divided by the
//    number of elements the CTA can meet, so a bin cannot overflow; S is picked per CTA from
//    the largest magnitude among the first elements it sees;
//  * any other value (not a multiple of 2^-S, too large, not finite) is added to the global
//    fp64 accumulator of its bin directly -- exact as well, slower;
//  * at the end the CTAs' bins are put together.  Many bins: every CTA writes its own to scratch, all meet at a counter
//    (the launch is cooperative), and each CTA adds up a slice of the bins over the CTAs and stores the fp32 result on
//    top of the defaults.  Few bins: every CTA adds its bins into the fp64 accumulators, and the block that finishes last
//    turns those into the result.  (With 2^16 bins the second way was 148 x 2^16 fp64 atomics and 64 rounds of one block:
//    2^27 keys 221 -> 186 us, 13101521 keys into 47631 bins 63 -> 46 us.)
//
// Every partial sum is exact, so the result is the fp32 rounding of the exact fp64-combined
// sum whatever the order of arrival.
//
// Bins beyond one CTA's shared memory: up to kHistOverflowBins more live in a private slice
// of global memory per CTA (integer atomics again; private, so a hot bin is not shared
// between SMs).  Beyond that a group of G = 2, 4 or 8 neighbouring CTAs splits the bins:
// all CTAs of a group walk the same elements (the later readers hit L2) and each updates
// only the bins it owns; store roots and whole-array folds of an element are handled by one
// CTA of the group.
#pragma once
#include "skeletons.cuh"
#include "tile.cuh"

namespace acc {
namespace dev {

constexpr int kHistBlock = 1024;
constexpr int kHistMaxBinsPerCta = 56 * 1024;   // 224 KiB of 32-bit bins per CTA
constexpr int kHistOverflowBins = 16 * 1024;    // further bins kept per CTA in global memory
constexpr int kHistUnroll = 2;                  // independent chunks in flight per thread (4 measured no faster)
constexpr int kHistAhead = 2;                   // trips between asking L2 for a chunk and reading it

struct HistPlan {
  int group;        // CTAs that split the bins
  int per_cta;      // bins in each CTA's shared memory
  int shift;        // log2(per_cta) when it is a power of two and group > 1, else -1
  int overflow;     // bins per CTA kept in global memory (group == 1 only)
  int exchange;     // words per CTA of the scratch in which the CTAs exchange their bins; 0: they add them up with atomics
  uint32_t polls;   // looks at the meeting counter (a tenth of a microsecond at the least) before a CTA gives the others up
};
constexpr int kHistExchangeBins = 20000;        // bins from which exchanging them is worth a meeting of all CTAs (1246656 keys: 10000 bins 25.7 against 22.5 us, 20000 bins the same, 60000 bins 33 against 46)

// A CTA that has walked its share waits for the others', which may take longer: a value that the integer bins do not take is
// an fp64 atomic on global memory, and where all such values meet in one bin a CTA's turn comes once in as many of these
// (some nanoseconds each) as there are CTAs.  Eight polls for every element of a share cover that; a short walk gets the usual limit.
inline uint32_t hist_polls(int64_t elements, int teams) {
  return (uint32_t)std::min<int64_t>((int64_t)kCopySpinLimit + 8 * (elements / std::max(teams, 1)), 0xFFFFFFFFll);
}

// How the bins are laid out, or false when they do not fit eight CTAs.
inline bool hist_plan(int64_t bins, int sms, HistPlan& p) {
  p = HistPlan{1, 0, -1, 0, 0, kCopySpinLimit};
  if (bins <= 0) return false;
  if (bins <= kHistMaxBinsPerCta + kHistOverflowBins) {
    p.per_cta = (int)std::min<int64_t>(bins, kHistMaxBinsPerCta);
    p.overflow = (int)(bins - p.per_cta);
    if (bins >= kHistExchangeBins) p.exchange = ((p.per_cta + 3) & ~3) + 4;
    return true;
  }
  while (p.group <= 8 && (bins + p.group - 1) / p.group > kHistMaxBinsPerCta) p.group *= 2;
  if (p.group > 8 || p.group > sms) return false;
  p.per_cta = (int)((bins + p.group - 1) / p.group);
  if ((p.per_cta & (p.per_cta - 1)) == 0)
    for (p.shift = 0; (1 << p.shift) < p.per_cta; ++p.shift) {}
  p.exchange = ((p.per_cta + 3) & ~3) + 4;              // (the bins, then the CTA's scale)
  return true;
}

// Fire-and-forget integer add on global memory (no value comes back, so nothing waits for it).
__device__ __forceinline__ void red_add_global(int* p, int v) {
  asm volatile("red.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Adds v to bin k: bins below `per_cta` are words of shared memory from `bins_addr`, the others
// words of global memory from `rest` (which already points per_cta words before the first of
// them).  One comparison and two predicated fire-and-forget adds, no branch.
__device__ __forceinline__ void red_add_bin(uint32_t k, uint32_t per_cta, uint32_t bins_addr, const int* rest, int v) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .u32 sa;\n\t.reg .u64 ga;\n\t"
      "setp.lt.u32 p, %0, %1;\n\t"
      "mad.lo.u32 sa, %0, 4, %2;\n\t"
      "mad.wide.u32 ga, %0, 4, %3;\n\t"
      "@p red.shared.add.s32 [sa], %4;\n\t"
      "@!p red.global.add.s32 [ga], %4;\n\t}"
      ::"r"(k), "r"(per_cta), "r"(bins_addr), "l"(rest), "r"(v) : "memory");
}
// Four updates of bins that may lie in either, or (rest == nullptr: all bins are in shared memory) without the choice per
// element (10^8 keys into 4096 bins 118 -> 96 us, 13101521 keys into 47631 bins 46 -> 42 us).
__device__ __forceinline__ void red_add_four(const uint32_t (&k)[4], uint32_t per_cta, uint32_t bins_addr, const int* rest, const int (&v)[4]) {
  if (rest == nullptr) {
#pragma unroll
    for (int j = 0; j < 4; ++j) asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(bins_addr + k[j] * 4u), "r"(v[j]) : "memory");
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) red_add_bin(k[j], per_cta, bins_addr, rest, v[j]);
  }
}
__device__ __forceinline__ void red_add_global(double* p, double v) {
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

// Whether member I can only take integer values in [0, iparam[0]), known from its function alone
// (then a scatter of it needs no per-value test of what the integer bins can hold).
template <class CL> constexpr bool yields_small_integers(int i) {
  const CNode& n = CL::c.nodes[i];
  return n.member && n.kind == ACC_GENERATE && n.dtype == ACC_F32 && n.fn == ACC_FN_IMOD_TO_F32;
}

template <class CL> constexpr int the_f32_add_permute() {
  for (int i = 0; i < CL::c.n; ++i)
    if (is_f32_add_permute(CL::c.nodes[i])) return i;
  return -1;
}

template <class CL, bool VEC>
__global__ void __launch_bounds__(kHistBlock, 1)
k_hist(const __grid_constant__ Args<CL::c.n> a, const HistPlan plan, int* overflow_base, int* exchange_base) {
  constexpr int N = CL::c.n;
  constexpr int W = VEC ? 4 : 1;
  constexpr int U = kHistUnroll;
  constexpr int DR = domain_rank<CL>();
  constexpr int NF = count_if<CL>(is_scalar_fold);
  constexpr int P = the_f32_add_permute<CL>();
  static_assert(P >= 0, "k_hist needs an fp32 '+' permute");
  constexpr CNode pn = CL::c.nodes[P];
  using IX = std::conditional_t<VEC, Ix4, Ix>;
  using VAL = val_of<IX>;
  extern __shared__ __align__(16) int bins_smem[];
  __shared__ uint32_t red[kHistBlock / 32];
  __shared__ bool last_block;
  __shared__ float sample_max;

  const int per_cta = plan.per_cta;
  const uint32_t group = (uint32_t)plan.group;
  const uint32_t rank = blockIdx.x % group;                    // which slice of the bins this CTA owns
  const uint32_t team = blockIdx.x / group;                    // which share of the elements its group walks
  const uint32_t n_teams = gridDim.x / group;
  int* const spill = overflow_base + (size_t)blockIdx.x * plan.overflow;   // zeroed by the host with the scratch
  for (int i = threadIdx.x; i < per_cta; i += kHistBlock) bins_smem[i] = 0;

  uint32_t acc[N];
  float comp[N] = {};                                          // see fold_step
  static_for<0, N>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr CNode nd = CL::c.nodes[i];
    if constexpr (is_scalar_fold(nd)) acc[i] = identity_of<nd.fn, nd.dtype>();
  });
  const uint32_t n_bins = (uint32_t)(a.n[P].R * a.n[P].C);
  const uint32_t per_row = (uint32_t)a.C / W;
  const uint32_t total = (uint32_t)a.R * per_row;
  const uint32_t stride = n_teams * kHistBlock;
  double* acc64 = reinterpret_cast<double*>(a.scratch + stream_acc64_off(NF, a.grid));

  auto index_of = [&](uint32_t q) {
    IX ix;
    if constexpr (DR <= 1) { ix.r = 0; ix.c = (int)(q * W); }
    else { const uint32_t r = q / per_row; ix.r = (int)r; ix.c = (int)((q - r * per_row) * W); }
    return ix;
  };

  // scale: the first chunk of every thread gives the magnitude to expect
  {
    float m = 0.0f;
    const uint32_t q = team * kHistBlock + threadIdx.x;
    if (q < total) {
      const VAL v = eval<CL, pn.in[2]>(a, index_of(q));
      if constexpr (VEC) {
#pragma unroll
        for (int j = 0; j < 4; ++j) m = fmaxf(m, fabsf(f_(v.v[j])));
      } else {
        m = fabsf(f_(v));
      }
    }
    if (!(m < 3.0e38f)) m = 0.0f;                              // ignore infinities and NaNs here
    const uint32_t top = block_reduce_n<ACC_FN_MAX, ACC_F32, kHistBlock>(u_(m), red);
    if (threadIdx.x == 0) sample_max = f_(top);
  }
  __syncthreads();
  // a bin receives at most `mine` addends of magnitude < cap each: |sum| < 2^31
  const uint32_t mine = ((total + n_teams - 1) / n_teams + 1) * W;
  const int cap_log2 = min(30 - (32 - __clz(mine)), 22);      // 2^cap_log2 * mine < 2^30
  constexpr bool INTS = yields_small_integers<CL>(pn.in[2]);
  // values known to be integers below m: m - 1 is the magnitude to scale for, whatever the sample says
  const float largest = INTS ? (float)max(a.n[pn.in[2]].ip0 - 1, 0) : sample_max;
  int S = 0;
  if (largest > 0.0f) {
    int e;
    frexpf(largest, &e);                                       // largest = f * 2^e, f in [0.5, 1)
    S = min(max(cap_log2 - 1 - e, -100), 100);                 // largest * 2^S < cap / 2
  }
  const float cap = exp2f((float)cap_log2);
  const float up = exp2f((float)S);
  // the denormal 2^(S - 149): a value in [0, 2^23) times it has the integer value * 2^S as its bits (one product, without the
  // conversion and the test that other values need: 2^27 keys 186.2 -> 184.5 us; used where S >= 0 and the values are known
  // to be integers, which makes S <= 21)
  const float up_bits = __uint_as_float(S >= 0 && S < 23 ? 1u << S : 0u);
  const double down = exp2((double)-S);

  auto scatter_one = [&](uint32_t k, uint32_t xbits) {
    if (k >= n_bins) { raise_status(a, kStatusIndex); return; }
    uint32_t at = k;                                           // position among this CTA's bins
    if (group != 1) {
      const uint32_t owner = plan.shift >= 0 ? (k >> plan.shift) : (k / (uint32_t)per_cta);
      if (owner != rank) return;
      at = k - owner * (uint32_t)per_cta;
    }
    const float x = f_(xbits);
    if (x == 0.0f) return;
    const float t = __fmul_rn(x, up);                          // exact whenever |t| >= 1 (no underflow)
    // nearest integer without the conversion unit: adding 1.5 * 2^23 leaves |t| < 2^22 rounded
    // to an integer in the low mantissa bits (cap <= 2^22 keeps |t| in that range)
    const float shifted = __fadd_rn(t, 12582912.0f);
    const float rounded = __fadd_rn(shifted, -12582912.0f);
    if (fabsf(t) >= 1.0f && fabsf(t) < cap && t == rounded) {
      const int v = __float_as_int(shifted) - 0x4B400000;      // bits of 12582912.0f
      // two calls, so that each is an atomic on a known address space (shared / global)
      if (at < (uint32_t)per_cta) atomicAdd(bins_smem + at, v);
      else red_add_global(spill + (at - (uint32_t)per_cta), v);
    } else {
      red_add_global(acc64 + k, (double)x);
    }
  };

  const bool fast_ok = group == 1 && S >= 0;
  const int* const rest = plan.overflow ? spill - per_cta : nullptr;
  const uint32_t bins_addr = (uint32_t)__cvta_generic_to_shared(bins_smem);
  uint32_t it = 0;
  // FULL: every chunk of the trip and of the trips prefetched from it lies inside the array (no test per chunk)
  auto trip = [&](auto full_c, uint32_t q0) {
    constexpr bool FULL = decltype(full_c)::value;
    if constexpr (VEC) {
      // ask L2 for what the trip after next will read: there are too few registers to keep
      // enough loads in flight to cover DRAM latency, so the loads should find their lines in L2
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t q = q0 + (kHistAhead * U + u) * stride;
        if (FULL || q < total) {
          const IX ix = index_of(q);
          eval<CL, pn.in[1]>(a, IxPF4{ix.r, ix.c});
          eval<CL, pn.in[2]>(a, IxPF4{ix.r, ix.c});
        }
      }
    }
    // evaluate U independent chunks first so that their loads are in flight together
    VAL key[U], val[U];
    bool live[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t q = q0 + u * stride;
      live[u] = FULL || q < total;
      if (live[u]) {
        const IX ix = index_of(q);
        key[u] = eval<CL, pn.in[1]>(a, ix);
        val[u] = eval<CL, pn.in[2]>(a, ix);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!FULL && !live[u]) continue;
      if (group == 1 || (it + u) % group == rank) {            // this CTA's turn for the element-wise side
        const IX ix = index_of(q0 + u * stride);
        static_for<0, N>([&](auto ic) {
          constexpr int i = decltype(ic)::value;
          constexpr CNode nd = CL::c.nodes[i];
          if constexpr (is_store_root(nd)) {
            st(reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[i].ptr)), a.n[i].C, ix, eval<CL, i>(a, ix));
          } else if constexpr (is_scalar_fold(nd)) {
            // a fold over the scatter's own value or index operand shares its registers
            VAL v;
            if constexpr (nd.in[0] == CL::c.nodes[P].in[2]) v = val[u];
            else if constexpr (nd.in[0] == CL::c.nodes[P].in[1]) v = key[u];
            else v = eval<CL, nd.in[0]>(a, ix);
            // a thread adds thousands of chunks to its running value: that step is compensated; the four
            // elements of a chunk are of one magnitude and are combined as a small tree first
            if constexpr (VEC) {
              const uint32_t four = combine<nd.fn, nd.dtype>(combine<nd.fn, nd.dtype>(v.v[0], v.v[1]),
                                                             combine<nd.fn, nd.dtype>(v.v[2], v.v[3]));
              fold_step<nd.fn, nd.dtype>(acc[i], comp[i], four);
            } else {
              fold_step<nd.fn, nd.dtype>(acc[i], comp[i], v);
            }
          }
        });
      }
      if constexpr (VEC) {
        // The usual case in one piece, without a branch per element: all four indices in range and
        // all four values exact integers below `cap` after scaling.  (With up >= 1 a non-zero x
        // cannot underflow to a zero product; otherwise the careful path below is taken.)
        const uint32_t kmax = max(max(key[u].v[0], key[u].v[1]), max(key[u].v[2], key[u].v[3]));
        if constexpr (INTS) {
          // integers below m, and (m - 1) * 2^S below cap / 2 by the choice of S: every product is an
          // exact integer the bins can take, so only the indices are looked at
          if (fast_ok & (kmax < n_bins)) {
            int v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = __float_as_int(__fmul_rn(f_(val[u].v[j]), up_bits));
            red_add_four(key[u].v, (uint32_t)per_cta, bins_addr, rest, v);
            continue;
          }
        }
        float t[4], shifted[4], off = 0.0f, big = 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          t[j] = __fmul_rn(f_(val[u].v[j]), up);
          shifted[j] = __fadd_rn(t[j], 12582912.0f);
          off = __fadd_rn(off, fabsf(__fadd_rn(__fadd_rn(shifted[j], -12582912.0f), -t[j])));   // 0 iff t is an integer (NaN otherwise)
          big = fmaxf(big, fabsf(t[j]));
        }
        if (fast_ok & (kmax < n_bins) & (off == 0.0f) & (big < cap)) {
          // (a zero is added like any other value: skipping it would cost more than it saves)
          int v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = __float_as_int(shifted[j]) - 0x4B400000;
          red_add_four(key[u].v, (uint32_t)per_cta, bins_addr, rest, v);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) scatter_one(key[u].v[j], val[u].v[j]);
        }
      } else {
        scatter_one(key[u], val[u]);
      }
    }
  };
  {
    const uint64_t step = (uint64_t)stride * U;
    const uint64_t reach = (uint64_t)(kHistAhead * U + U - 1) * stride;     // the furthest chunk a trip touches, from its first
    uint64_t q0 = (uint64_t)team * kHistBlock + threadIdx.x;
    for (; q0 + reach < total; q0 += step, it += U) trip(std::true_type{}, (uint32_t)q0);
    for (; q0 < total; q0 += step, it += U) trip(std::false_type{}, (uint32_t)q0);
  }
  if constexpr (VEC && DR <= 1) {
    // the last elements of an array whose length is no multiple of four: every CTA of the first team takes those whose bin it owns
    const int c = (int)(per_row * 4u + threadIdx.x);
    if (team == 0 && c < a.C) {
      const Ix ix{0, c};
      if (rank == 0) {
        static_for<0, N>([&](auto ic) {
          constexpr int i = decltype(ic)::value;
          constexpr CNode nd = CL::c.nodes[i];
          if constexpr (is_store_root(nd)) reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[i].ptr))[c] = eval<CL, i>(a, ix);
          else if constexpr (is_scalar_fold(nd)) fold_step<nd.fn, nd.dtype>(acc[i], comp[i], eval<CL, nd.in[0]>(a, ix));
        });
      }
      scatter_one(eval<CL, pn.in[1]>(a, ix), eval<CL, pn.in[2]>(a, ix));
    }
  }

  __syncthreads();
  if (plan.exchange) {
    int* mine = exchange_base + (size_t)blockIdx.x * plan.exchange;
    for (int i = threadIdx.x * 4; i < per_cta; i += kHistBlock * 4)      // (the words behind the last bin are nobody's)
      *reinterpret_cast<int4*>(mine + i) = *reinterpret_cast<const int4*>(bins_smem + i);
    if (threadIdx.x == 0) *reinterpret_cast<double*>(mine + plan.exchange - 4) = down;
  } else {
  // every CTA starts its sweep somewhere else, so that the CTAs that finish together do not all
  // queue up on the same accumulators
  const int turn = (int)((blockIdx.x * 2654435761u) >> 8);
  for (int i0 = threadIdx.x; i0 < per_cta; i0 += kHistBlock) {
    const int i = (int)((uint32_t)(i0 + turn) % (uint32_t)per_cta);
    const int v = bins_smem[i];
    const uint32_t bin = rank * (uint32_t)per_cta + i;
    if (v != 0 && bin < n_bins) red_add_global(acc64 + bin, (double)v * down);
  }
  for (int i0 = threadIdx.x; i0 < plan.overflow; i0 += kHistBlock) {
    const int i = (int)((uint32_t)(i0 + turn) % (uint32_t)plan.overflow);
    const int v = *reinterpret_cast<volatile int*>(spill + i);
    if (v != 0) red_add_global(acc64 + per_cta + i, (double)v * down);
  }
  }

  static_for<0, N>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr CNode nd = CL::c.nodes[i];
    if constexpr (is_scalar_fold(nd)) {
      constexpr int ord = count_if<CL>(is_scalar_fold, i);
      const uint32_t v = block_reduce_n<nd.fn, nd.dtype, kHistBlock>(acc[i], red);
      if (threadIdx.x == 0) a.scratch[stream_partials_off() + ord * a.grid + blockIdx.x] = v;
    }
  });
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t before = atomicAdd(a.scratch, 1u);
    last_block = plan.exchange ? blockIdx.x == 0 : before == gridDim.x - 1;
    if (plan.exchange) {                                       // all CTAs are resident: wait until each has written its bins
      uint32_t spins = 0;
      while (*reinterpret_cast<volatile uint32_t*>(a.scratch) < gridDim.x) {
        if (++spins > plan.polls) { raise_status(a, kStatusTimeout); break; }
        __nanosleep(100);
      }
    }
  }
  __syncthreads();
  __threadfence();
  const float* defaults = reinterpret_cast<const float*>(a.n[pn.in[0]].ptr);
  float* out = reinterpret_cast<float*>(const_cast<void*>(a.n[P].ptr));
  if (plan.exchange) {
    // this CTA's slice of the bins: half of the threads take the even teams, half the odd ones
    double* scale = reinterpret_cast<double*>(bins_smem);       // (the bins have been written out)
    double* other = scale + gridDim.x;                          // what the second half found
    for (int c = threadIdx.x; c < (int)gridDim.x; c += kHistBlock)
      scale[c] = __ldcg(reinterpret_cast<const double*>(exchange_base + (size_t)(c + 1) * plan.exchange - 4));
    __syncthreads();
    const uint32_t lo = (uint32_t)((uint64_t)n_bins * blockIdx.x / gridDim.x), hi = (uint32_t)((uint64_t)n_bins * (blockIdx.x + 1) / gridDim.x);
    const uint32_t side = threadIdx.x / (kHistBlock / 2), at0 = threadIdx.x % (kHistBlock / 2);
    for (uint32_t b0 = lo; b0 < hi; b0 += kHistBlock / 2) {
      const uint32_t b = b0 + at0;
      double sum = 0.0;
      if (b < hi) {
        const uint32_t owner = group == 1 ? 0u : b / (uint32_t)per_cta, at = group == 1 ? b : b - owner * (uint32_t)per_cta;
        const bool spilled = at >= (uint32_t)per_cta;
        const int* src = spilled ? overflow_base + (at - (uint32_t)per_cta) : exchange_base + at;
        const size_t step = spilled ? (size_t)plan.overflow : (size_t)plan.exchange;
#pragma unroll 8
        for (uint32_t t = side; t < n_teams; t += 2) {
          const uint32_t c = t * group + owner;
          sum += (double)__ldcg(src + c * step) * scale[c];
        }
        if (side == 1) other[at0] = sum;
      }
      __syncthreads();
      if (b < hi && side == 0) out[b] = (float)((double)defaults[b] + __ldcg(acc64 + b) + (sum + other[at0]));
      __syncthreads();
    }
  }
  if (!last_block) return;
  static_for<0, N>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr CNode nd = CL::c.nodes[i];
    if constexpr (is_scalar_fold(nd)) {
      constexpr int ord = count_if<CL>(is_scalar_fold, i);
      const volatile uint32_t* part = a.scratch + stream_partials_off() + ord * a.grid;
      uint32_t v = identity_of<nd.fn, nd.dtype>();
      for (int b = threadIdx.x; b < (int)gridDim.x; b += kHistBlock) v = combine<nd.fn, nd.dtype>(v, part[b]);
      v = block_reduce_n<nd.fn, nd.dtype, kHistBlock>(v, red);
      if (threadIdx.x == 0) *reinterpret_cast<uint32_t*>(const_cast<void*>(a.n[i].ptr)) = v;
    }
  });
  if (plan.exchange) return;
  const volatile double* sums = acc64;
  for (uint32_t b = threadIdx.x; b < n_bins; b += kHistBlock) out[b] = (float)((double)defaults[b] + sums[b]);
}

}  // namespace dev
}  // namespace acc
