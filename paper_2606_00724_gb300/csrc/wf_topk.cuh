// The deterministic Top-K (Eq. 9) of the kernels that keep a unit's ranking
// keys in shared memory, run by the unit's compute warps: one warpgroup, or
// two (WIDE).  Keys must be followed by the caller's own barrier after the
// last one is written and before the call.
#pragma once

#include <float.h>
#include <stddef.h>
#include <stdint.h>

#include "wf_sm100.cuh"

namespace wf {
namespace topk {

using namespace sm100;

constexpr int NCW = 4;              // warps of a warpgroup
constexpr int NCT = 32 * NCW;       // threads of a warpgroup
constexpr int kMaxCand = 64 * NCT;  // largest candidate list (64 keys a thread of one warpgroup)
constexpr uint32_t kCsyncId = 1;    // named barriers 1, 2: the compute warps of unit 0, 1 (1 for both when WIDE)

// A unit's compute warps: one warpgroup (one per unit of a two-unit cluster),
// or both warpgroups (WIDE) when the cluster serves one unit; then the
// warpgroups take alternate tiles and share the Top-K.  Thread index within
// the unit's compute warps, their count and their barrier.
template <bool WIDE>
__host__ __device__ constexpr int unit_warps() {
  return WIDE ? 2 * NCW : NCW;
}
template <bool WIDE>
__device__ __forceinline__ int ctid() {
  return threadIdx.x & (32 * unit_warps<WIDE>() - 1);
}
template <bool WIDE>
__device__ __forceinline__ void csync() {
  named_sync(kCsyncId + (WIDE ? 0u : (threadIdx.x >> 7)), 32 * unit_warps<WIDE>());
}
// Top-K scratch, in shared memory.  The histogram, the list counter and the
// masks are zero between calls (zeroed at kernel start, cleared again at the
// end of every call).
constexpr int NB = 2048;     // histogram buckets
constexpr int MAXUW = 2 * NCW;  // most compute warps of a unit
struct SelScratch {
  uint32_t hist[NB];
  float2 blist[32 * MAXUW];  // boundary-bucket keys (key, position)
  float2 sred[2][MAXUW];     // (min, max) per warp, alternating rounds
  int wsum[4][MAXUW];        // per-warp sums of the scans (slot per scan, 32 bytes)
  uint32_t taken[2 * 32 * MAXUW];  // boundary keys taken, as each owner's position mask (zero between uses)
  uint32_t bcnt;
};
static_assert((NB / NCT) % 8 == 0, "buckets are cleared four at a time by up to twice NCT threads");
static_assert(offsetof(SelScratch, wsum) % 16 == 0, "the scan's warp sums are read 16 bytes at a time");

#define SC_ADDR(sc_a, field) ((sc_a) + (uint32_t)offsetof(SelScratch, field))

// Positions a Top-K thread owns for a list of m: the smallest power of two
// (at least 4) with R times the unit's compute threads >= m.
template <bool WIDE>
__host__ __device__ constexpr int topk_run(int m) {
  int R = 4;
  while (R * 32 * unit_warps<WIDE>() < m) R <<= 1;
  return R;
}

// Exclusive prefix sum over the unit's compute threads (thread order), with
// its per-warp sums in the words at wsum_a.  One barrier: the caller does not
// reuse those words before another barrier has passed.
template <bool WIDE>
__device__ __forceinline__ int cta_excl_scan(int v, uint32_t wsum_a) {
  const int lane = threadIdx.x & 31, warp = ctid<WIDE>() >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) sts_u32(wsum_a + 4u * warp, (uint32_t)incl);
  csync<WIDE>();
  int before = 0;
#pragma unroll
  for (int q = 0; q < unit_warps<WIDE>() / 4; ++q) {
    const uint4 w = lds_v4(wsum_a + 16u * q);
    before += (warp > 4 * q ? (int)w.x : 0) + (warp > 4 * q + 1 ? (int)w.y : 0) + (warp > 4 * q + 2 ? (int)w.z : 0) +
              (warp > 4 * q + 3 ? (int)w.w : 0);
  }
  return before + incl - v;
}

// Bucket of key v in NB buckets linear over [lo, hi): the same fp32
// operations in every pass and every CTA give the same bucket.
__device__ __forceinline__ int bucket_of(float v, float lo, float scale) {
  // floor(x) for 0 <= x < 2^23: adding 2^23 rounded toward -inf leaves
  // floor(x) in the low mantissa bits.
  const float x = fmaxf((v - lo) * scale, 0.f);
  return min(NB - 1, __float_as_int(__fadd_rd(x, 8388608.f)) - 0x4B000000);
}

// Bit counts of the Top-K's position masks (32 or 64 positions a thread).
__device__ __forceinline__ int popc_m(uint32_t x) { return __popc(x); }
__device__ __forceinline__ int popc_m(unsigned long long x) { return __popcll(x); }
__device__ __forceinline__ int ffs_m(uint32_t x) { return __ffs(x); }
__device__ __forceinline__ int ffs_m(unsigned long long x) { return __ffsll((long long)x); }

// (min, max) of the undecided keys (bit i of act: position j0 + i of the key
// array) over the compute threads, via slot `par`.
template <typename MT, bool WIDE>
__device__ __forceinline__ float2 cta_minmax(uint32_t keys_a, int j0, MT act, uint32_t sc_a, int par) {
  const int lane = threadIdx.x & 31, warp = ctid<WIDE>() >> 5;
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll 1
  for (MT a = act; a; a &= a - 1) {
    const float v = lds_f32(keys_a + 4u * (uint32_t)(j0 + ffs_m(a) - 1));
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
  }
  lo = warp_min_f32(lo);
  hi = warp_max_f32(hi);
  if (lane == 0) sts_v2(SC_ADDR(sc_a, sred) + 8u * (par * MAXUW + warp), __float_as_uint(lo), __float_as_uint(hi));
  csync<WIDE>();
#pragma unroll
  for (int w = 0; w < unit_warps<WIDE>(); ++w) {
    const uint2 r = lds_v2(SC_ADDR(sc_a, sred) + 8u * (par * MAXUW + w));
    lo = fminf(lo, __uint_as_float(r.x));
    hi = fmaxf(hi, __uint_as_float(r.y));
  }
  return make_float2(lo, hi);
}

// Every warp locates the boundary bucket in the histogram by itself, with no
// barrier or broadcast: the bucket holding the need-th largest undecided key
// (buckets ranked high to low), how many of its keys are still needed, and
// how many it holds.  Lane l sums the 64 buckets [NB - 64 (l + 1), NB - 64 l)
// (reading them in a lane-rotated order, free of bank conflicts); a scan over
// the lanes finds the chunk, and a second scan over that chunk's buckets, two
// a lane, the bucket.
__device__ __forceinline__ uint3 warp_boundary(uint32_t hist_a, uint32_t need, int lane) {
  const uint32_t cbase = hist_a + 4u * (uint32_t)(NB - 64 * (lane + 1));
  uint32_t tot = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint4 v = lds_v4(cbase + 16u * (uint32_t)((i + lane) & 15));
    tot += v.x + v.y + v.z + v.w;
  }
  uint32_t incl = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  // Some lane always qualifies (need never exceeds the keys counted); the
  // clamp only keeps the reads in the histogram should a wait have given up.
  const int lc = max(0, __ffs(__ballot_sync(0xffffffffu, incl >= need)) - 1);
  const uint32_t above = __shfl_sync(0xffffffffu, incl - tot, lc);
  const int bb = NB - 1 - 64 * lc - 2 * lane;                 // this lane's buckets bb and bb - 1
  const uint2 pr = lds_v2(hist_a + 4u * (uint32_t)(bb - 1));  // .x = bucket bb - 1, .y = bucket bb
  const uint32_t pair = pr.x + pr.y;
  uint32_t inc2 = pair;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc2, o);
    if (lane >= o) inc2 += t;
  }
  const int l2 = max(0, __ffs(__ballot_sync(0xffffffffu, above + inc2 >= need)) - 1);
  const uint32_t before = above + inc2 - pair;
  const bool upper = before + pr.y >= need;
  const uint32_t b = upper ? (uint32_t)bb : (uint32_t)(bb - 1);
  const uint32_t nd = upper ? need - before : need - before - pr.y;
  const uint32_t ct = upper ? pr.y : pr.x;
  return make_uint3(__shfl_sync(0xffffffffu, b, l2), __shfl_sync(0xffffffffu, nd, l2),
                    __shfl_sync(0xffffffffu, ct, l2));
}

// The boundary bucket of the histogram: the bucket holding the need-th largest
// undecided key (buckets ranked high to low), how many of its keys are still
// needed, and how many it holds.  Thread t sums the BPT buckets
// [NB - BPT (t + 1), NB - BPT t) (reading them in a lane-rotated order, free of
// bank conflicts); a scan over the threads finds the one whose buckets reach
// `need`, which searches them and publishes the result.  For two warpgroups:
// with each warp searching the whole histogram by itself as below, its reads
// were 1100 cycles of a Top-K of 5300 (128K step 90.2 -> 88.1 us).  One
// warpgroup keeps that: two more barriers a Top-K cost two-unit clusters more
// than they saved (64 units x 32K 68.6 -> 68.9 us).
template <bool WIDE>
__device__ __forceinline__ uint3 unit_boundary(uint32_t hist_a, uint32_t need, uint32_t sc_a) {
  constexpr int TN = 32 * unit_warps<WIDE>(), BPT = NB / TN, NV = BPT / 4;
  static_assert(NV == 4 || NV == 2, "the rotation below");
  const int tid = ctid<WIDE>(), lane = tid & 31;
  const uint32_t own = hist_a + 4u * (uint32_t)(NB - BPT * (tid + 1));
  uint32_t tot = 0;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const uint4 v = lds_v4(own + 16u * (uint32_t)((i + (lane >> (NV == 4 ? 1 : 2))) & (NV - 1)));
    tot += (v.x + v.y) + (v.z + v.w);
  }
  const uint32_t excl = (uint32_t)cta_excl_scan<WIDE>((int)tot, SC_ADDR(sc_a, wsum));
  if (excl < need && need <= excl + tot) {  // one thread
    uint32_t cum = excl, b = 0, nd = 0, ct = 0;
    bool found = false;
#pragma unroll
    for (int g = NV - 1; g >= 0; --g) {
      const uint4 v = lds_v4(own + 16u * (uint32_t)g);
      const uint32_t c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 3; e >= 0; --e) {
        const bool hit = !found && cum + c[e] >= need;
        b = hit ? (uint32_t)(NB - BPT * (tid + 1) + 4 * g + e) : b;
        nd = hit ? need - cum : nd;
        ct = hit ? c[e] : ct;
        found |= hit;
        cum += c[e];
      }
    }
    sts_v4(SC_ADDR(sc_a, wsum) + 32u, make_uint4(b, nd, ct, 0u));
  }
  csync<WIDE>();
  const uint4 r = lds_v4(SC_ADDR(sc_a, wsum) + 32u);
  return make_uint3(r.x, r.y, r.z);
}

// Top-K of the m keys at keys_a (largest first, lower position wins ties):
// the kk chosen candidate indices, in ascending position order, overwrite the
// key array.  A candidate's index is its position at the top scale, else
// 2 J[j/2] + j%2 with J the previous selection at jprev_a (Eq. 10).
// [lo, hi] is the range of the keys (sent along with them).
// Each thread owns the run of R positions j0 = tid R .. j0 + R - 1 (R a power
// of two, 4 to 64), with one bit per position for "undecided" and "taken" in
// a mask of type MT (32 bits up to R = 32, else 64).
// The keys stay in shared memory; every pass re-reads them four at a time
// (16-byte loads, the G = R / 4 groups of a run visited in a lane-rotated
// order so that the 8 lanes of a quarter warp hit distinct banks).  Each
// round spreads the undecided keys over NB buckets linear in [lo, hi] (fp32
// arithmetic is monotone, so a key in a higher bucket is strictly larger);
// the bucket holding the boundary is found from the counts: keys above it are
// taken, keys below it dropped.  A boundary bucket of at most
// as many keys as the unit has threads is resolved exactly: its keys go to a
// list and are ranked on (key, -position) against the whole list.  Up to 32
// keys (the common case: a few), every warp does that by itself with an entry
// a lane and the owners take their winners from the lanes, with no further
// barrier; more are ranked by their owners (one warpgroup) or by the list
// entries' threads, which mark winners in the owners' position masks (both
// warpgroups: measured 116.9 -> 110.6 us at 128K, while one warpgroup ran
// slower that way).  A larger bucket is bucketed again over its own range.
// If only equal keys remain, the lowest positions are taken.
template <typename MT, bool WIDE>
__device__ __noinline__ void select_keys(uint32_t keys_a, int m, int kk, uint32_t jprev_a, int top, uint32_t sc_a,
                                         float lo, float hi, int R) {
  constexpr int MB = 8 * (int)sizeof(MT);       // positions a mask holds
  constexpr int TN = 32 * unit_warps<WIDE>();   // the unit's compute threads
  constexpr int BPT = NB / TN;                  // buckets each thread clears
  const int tid = ctid<WIDE>(), lane = tid & 31;
  const int j0 = tid * R;
  const int G = R >> 2;                         // groups of four keys in a run
  const int rotg = ((lane * G) >> 3) & (G - 1);  // first group this lane visits
  const int nv = max(0, min(R, m - j0));        // valid positions of the run
  const uint32_t m4 = (uint32_t)((m + 3) & ~3);  // the key array holds m4 >= 4 words
  MT act = nv >= MB ? ~(MT)0 : (((MT)1 << nv) - 1), took = 0;
  // The four keys of group g (clamped into the array; positions past m are
  // never undecided).
  auto group = [&](int g) {
    const uint4 v = lds_v4(keys_a + 4u * min((uint32_t)(j0 + 4 * g), m4 - 4u));
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
  };
  // body(g, keys of group g) for every group of the run, up to four groups'
  // loads in flight (shared-memory accesses keep their order, so a load issued
  // between another group's updates would be waited for by itself).
  auto for_groups = [&](auto&& body) {
    if (G < 4) {
#pragma unroll 1
      for (int gg = 0; gg < G; ++gg) {
        const int g = (gg + rotg) & (G - 1);
        body(g, group(g));
      }
      return;
    }
#pragma unroll 1
    for (int g4 = 0; g4 < G; g4 += 4) {
      float4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = group((g4 + k + rotg) & (G - 1));
#pragma unroll
      for (int k = 0; k < 4; ++k) body((g4 + k + rotg) & (G - 1), v[k]);
    }
  };
  const uint32_t hist_a = SC_ADDR(sc_a, hist);
  const uint32_t own_a = hist_a + 4u * (uint32_t)(BPT * tid);  // the buckets this thread clears
  uint32_t need = (uint32_t)kk;
  bool resolved = false;
#pragma unroll 1
  for (int iter = 0; iter < 6; ++iter) {
    // A key of -inf (a row of weight 0) does not stretch the buckets to an
    // infinite width, which would put every key into the lowest one.
    lo = fmaxf(lo, -FLT_MAX);
    if (!(hi > lo)) break;  // every undecided key is equal (or none is left)
    const float scale = (float)NB / (hi - lo);
    for_groups([&](int g, const float4& v) {
      const uint32_t a4 = (uint32_t)(act >> (4 * g));
      const int b0 = bucket_of(v.x, lo, scale), b1 = bucket_of(v.y, lo, scale);
      const int b2 = bucket_of(v.z, lo, scale), b3 = bucket_of(v.w, lo, scale);
      reds_add_if(a4 & 1u, hist_a + 4u * b0, 1u);
      reds_add_if(a4 & 2u, hist_a + 4u * b1, 1u);
      reds_add_if(a4 & 4u, hist_a + 4u * b2, 1u);
      reds_add_if(a4 & 8u, hist_a + 4u * b3, 1u);
    });
    csync<WIDE>();
    const uint3 bd = WIDE ? unit_boundary<WIDE>(hist_a, need, sc_a) : warp_boundary(hist_a, need, lane);
    const int sb = (int)bd.x;
    need = bd.y;
    const uint32_t cnt = bd.z;
    for_groups([&](int g, const float4& v) {
      const int bk[4] = {bucket_of(v.x, lo, scale), bucket_of(v.y, lo, scale), bucket_of(v.z, lo, scale),
                         bucket_of(v.w, lo, scale)};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const MT bit = act & ((MT)1 << (4 * g + e));  // 0 for a decided position
        took |= bk[e] > sb ? bit : (MT)0;
        act &= bk[e] != sb ? ~bit : ~(MT)0;
      }
    });
    if (cnt == need) {
      took |= act;
      act = 0;
      resolved = true;
      break;
    }
    if (cnt <= (uint32_t)TN) {
      // Append the boundary keys, one atomic each: there are few, and their
      // order in the list does not matter.
#pragma unroll 1
      for (MT a = act; a; a &= a - 1) {
        const int i = ffs_m(a) - 1;
        const uint32_t key = lds_u32(keys_a + 4u * (uint32_t)(j0 + i));
        const uint32_t slot = atoms_add(SC_ADDR(sc_a, bcnt), 1u);
        // slot < TN always (the list holds cnt <= TN keys); the predicate
        // keeps the store in the list should a wait have given up.
        sts_v2_if(slot < (uint32_t)TN, SC_ADDR(sc_a, blist) + 8u * slot, key, (uint32_t)(j0 + i));
      }
      csync<WIDE>();
      if (cnt <= 32u) {
        // Every warp ranks the whole list by itself, entry l on lane l, on
        // (key, -position); the owners then take their winners from the lanes.
        const uint2 me = lds_v2(SC_ADDR(sc_a, blist) + 8u * min((uint32_t)lane, cnt - 1));
        const float kx = __uint_as_float(me.x);
        const int jx = (int)me.y;
        uint32_t rank = 0;
#pragma unroll 4
        for (int v = 0; v < (int)cnt; ++v) {
          const float ko = __shfl_sync(0xffffffffu, kx, v);
          const int jo = __shfl_sync(0xffffffffu, jx, v);
          rank += (ko > kx) || (ko == kx && jo < jx);
        }
        const bool win = (uint32_t)lane < cnt && rank < need;
#pragma unroll 1
        for (uint32_t w = __ballot_sync(0xffffffffu, win); w; w &= w - 1) {
          const int off = __shfl_sync(0xffffffffu, jx, __ffs(w) - 1) - j0;
          took |= (uint32_t)off < (uint32_t)R ? act & ((MT)1 << off) : (MT)0;
        }
        act = 0;
        resolved = true;
        break;
      }
      if (!WIDE) {
        // Every owner ranks its own boundary keys on (key, -position)
        // against the list (measured faster with one warpgroup).
#pragma unroll 1
        for (MT a = act; a; a &= a - 1) {
          const int i = ffs_m(a) - 1;
          const float kx = lds_f32(keys_a + 4u * (uint32_t)(j0 + i));
          const int jx = j0 + i;
          uint32_t rank = 0;
#pragma unroll 1
          for (uint32_t v0 = 0; v0 < cnt; v0 += 4) {
            uint2 o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = lds_v2(SC_ADDR(sc_a, blist) + 8u * min(v0 + k, cnt - 1));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float ko = __uint_as_float(o[k].x);
              rank += (v0 + k < cnt) && ((ko > kx) || (ko == kx && (int)o[k].y < jx));
            }
          }
          if (rank < need) took |= (MT)1 << i;
        }
        act = 0;
        resolved = true;
        break;
      }
      // WIDE: thread t ranks list entry t on (key, -position) against the
      // whole list (every thread reads the same entry at a time: broadcasts)
      // and marks a winner in its owner's mask; then each owner takes its bits.
      constexpr int MW = (int)sizeof(MT) / 4;  // 32-bit words of a mask
      if ((uint32_t)tid < cnt) {
        const uint2 me = lds_v2(SC_ADDR(sc_a, blist) + 8u * (uint32_t)tid);
        const float kx = __uint_as_float(me.x);
        const int jx = (int)me.y;
        uint32_t rank = 0;
#pragma unroll 1
        for (uint32_t v0 = 0; v0 < cnt; v0 += 4) {
          uint2 o[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) o[k] = lds_v2(SC_ADDR(sc_a, blist) + 8u * min(v0 + k, cnt - 1));
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float ko = __uint_as_float(o[k].x);
            rank += (v0 + k < cnt) && ((ko > kx) || (ko == kx && (int)o[k].y < jx));
          }
        }
        if (rank < need) {
          const int owner = jx / R, bit = jx - owner * R;
          // owner < TN always; the bound keeps the store in the masks should a wait have given up
          const uint32_t w = (uint32_t)min(owner, TN - 1) * MW + (uint32_t)(bit >> 5);
          reds_or(SC_ADDR(sc_a, taken) + 4u * w, 1u << (bit & 31));
        }
      }
      csync<WIDE>();
      {
        const uint32_t ta = SC_ADDR(sc_a, taken) + 4u * (uint32_t)(tid * MW);
        MT mine = (MT)lds_u32(ta);
        if (MW == 2) mine |= (MT)((unsigned long long)lds_u32(ta + 4u) << 32);
        took |= mine & act;
        sts_u32(ta, 0u);
        if (MW == 2) sts_u32(ta + 4u, 0u);
      }
      act = 0;
      resolved = true;
      break;
    }
    // The boundary bucket again over its own range, with a cleared histogram.
    csync<WIDE>();  // every warp has read the histogram
#pragma unroll
    for (int i = 0; i < BPT / 4; ++i) sts_v4(own_a + 16u * i, make_uint4(0, 0, 0, 0));
    const float2 lh = cta_minmax<MT, WIDE>(keys_a, j0, act, sc_a, iter & 1);  // its barrier also publishes the cleared buckets
    lo = lh.x;
    hi = lh.y;
  }
  MT take = took;
  if (!resolved) {
    // Only equal keys are undecided: the first `need` by position are taken.
    const int eq_base = cta_excl_scan<WIDE>(popc_m(act), SC_ADDR(sc_a, wsum) + 96u);
    int remaining = (int)need - eq_base;
    for (MT e = act; e && remaining > 0; --remaining) {
      const MT low = e & (~e + 1);
      take |= low;
      e ^= low;
    }
  }
  // Each winner at its output rank, four positions at a time (positions
  // 4g .. 4g + 3 of the run are the children of the previous selection's
  // entries (j0 + 4g) / 2 and that + 1).  The scan's barrier orders every read
  // of the keys, the histogram and the boundary list before the key array is
  // overwritten and the scratch cleared.
  int r = cta_excl_scan<WIDE>(popc_m(take), SC_ADDR(sc_a, wsum) + 64u);
  // (Four groups a turn, so that their entries of the previous selection load
  // together; a run shorter than that has entries of its last group repeated.)
#pragma unroll 1
  for (int g4 = 0; g4 < G; g4 += 4) {
    uint2 pj[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = j0 + 4 * min(g4 + k, G - 1);
      // Entries past the previous selection (positions past m) are not used;
      // the clamp keeps the load in the array.
      pj[k] = top ? make_uint2(0u, 0u) : lds_v2(jprev_a + 4u * min((uint32_t)(j >> 1), (m4 >> 1) - 2u));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = j0 + 4 * (g4 + k);
      const uint32_t t4 = g4 + k < G ? (uint32_t)(take >> (4 * (g4 + k))) & 15u : 0u;
      const int c[4] = {top ? j : 2 * (int)pj[k].x, top ? j + 1 : 2 * (int)pj[k].x + 1, top ? j + 2 : 2 * (int)pj[k].y,
                        top ? j + 3 : 2 * (int)pj[k].y + 1};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        // r < kk <= m always; the bound keeps the store in the array should a
        // wait have given up.
        sts_u32_if(((t4 >> e) & 1u) && (uint32_t)r < (uint32_t)m, keys_a + 4u * (uint32_t)r, (uint32_t)c[e]);
        r += (t4 >> e) & 1u;
      }
    }
  }
  csync<WIDE>();
  // The scratch is cleared after the selection's last barrier: nothing uses it
  // again before another barrier of these threads.
#pragma unroll
  for (int i = 0; i < BPT / 4; ++i) sts_v4(own_a + 16u * i, make_uint4(0, 0, 0, 0));
  if (tid == 0) sts_u32(SC_ADDR(sc_a, bcnt), 0u);
}

// Top-K dispatch: R = the smallest power of two (at least 4) with R TN >= m
// (m <= 64 NCT, TN the unit's compute threads); 64-bit position masks only
// for R = 64.
template <bool WIDE>
__device__ __forceinline__ void select_topk(uint32_t keys_a, int m, int kk, uint32_t jprev_a, int top, uint32_t sc_a,
                                            float lo, float hi) {
  const int R = topk_run<WIDE>(m);
  if (WIDE || R <= 32) select_keys<uint32_t, WIDE>(keys_a, m, kk, jprev_a, top, sc_a, lo, hi, R);
  else select_keys<unsigned long long, WIDE>(keys_a, m, kk, jprev_a, top, sc_a, lo, hi, R);
}

}  // namespace topk
}  // namespace wf
