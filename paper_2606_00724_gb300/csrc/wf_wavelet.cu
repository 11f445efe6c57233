// Approximation rows of the periodized DWT of a gathered key sub-sequence
// (Eq. 6 for the whole prompt, Eq. 11 for the blocks of the candidates kept
// one scale up), for the Haar and db2 filter banks.
//
// The sequence of a unit is the keys of blocks [2^b c, 2^b (c + 1)) for the
// unit's candidates c, in candidate order, taken as periodic.  One level of
// analysis is a[j] = sum_k h[k] x[(2j + k) mod len]; b levels give one
// approximation row per candidate.
//
// Scales 1 to 5 stream the rows through registers (approx_stream_kernel).
// Deeper ones go through shared memory (approx_kernel):
// one CTA computes TO consecutive level-b rows for DS head-dim channels: it
// gathers the TO 2^b input rows plus the (taps - 2)(2^b - 1) rows the filter
// reaches past them (wrapping around the gathered sequence) into shared
// memory with 16-byte cp.async copies, and runs the b levels of the cascade
// there in fp32.  A thread owns one 16-byte vector of channels (8 for bf16,
// 4 for fp32) and a run of consecutive outputs of each level: it slides its
// filter window two rows per output, so an input row is one 16-byte load
// (plus the widening of its bf16 lanes), and every output is taps packed
// multiply-adds a channel pair.  Intermediate levels stay in shared memory as
// fp32 in 16-byte planes (conflict-free loads); the last level goes from
// registers to global memory.  Arithmetic, the storage rule: Haar:
// fl32(x0 + x1) * fl32(1 / sqrt 2), as the stored pyramid; db2:
// fl32(fl32(h[0]) x0), then fused multiply-adds with fl32(h[1..3]) in order.
// The packed fp32 instructions round each lane as the scalar ones do.  Only
// the last level is rounded to the key dtype.
#include <math.h>

#include <map>
#include <mutex>

#include "wf_internal.cuh"
#include "wf_sm100.cuh"

namespace wf {
namespace {

using namespace sm100;

constexpr int NTH = 256;      // threads per CTA
constexpr int IN_ROWS = 128;  // gathered rows per CTA before the filter's reach

// Output rows per CTA at scale `level`.
__host__ __device__ inline int outputs_per_cta(int level) { return (IN_ROWS >> level) > 0 ? (IN_ROWS >> level) : 1; }

// Rows needed l levels below the output so that the output level yields `to`
// rows: to 2^l + (taps - 2)(2^l - 1).
__host__ __device__ inline int rows_needed(int to, int l, int taps) { return (to << l) + (taps - 2) * ((1 << l) - 1); }

struct Taps {
  float h[4];
};

// A vector of VEC channels as VEC / 2 packed fp32 pairs.
template <typename T>
struct Lanes {
  static constexpr int VEC = Vec<T>::N;
  f32x2 v[VEC / 2];
};

// Widen one 16-byte vector of T (as loaded) to fp32 pairs (exact).
__device__ __forceinline__ void widen(const uint4& w, Lanes<bf16>& o) {
  const uint32_t a[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) o.v[i] = pk2(__uint_as_float(a[i] << 16), __uint_as_float(a[i] & 0xffff0000u));
}
__device__ __forceinline__ void widen(const uint4& w, Lanes<float>& o) {
  o.v[0] = pk2(__uint_as_float(w.x), __uint_as_float(w.y));
  o.v[1] = pk2(__uint_as_float(w.z), __uint_as_float(w.w));
}
// Round to T and pack one 16-byte vector.
__device__ __forceinline__ uint4 narrow(const Lanes<bf16>& x) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = up2(x.v[i]);
    w[i] = pack_bf16(f.x, f.y);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ uint4 narrow(const Lanes<float>& x) {
  const float2 a = up2(x.v[0]), b = up2(x.v[1]);
  return make_uint4(__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(b.x), __float_as_uint(b.y));
}

// Outputs of one unrolled pass of the cascade (longer runs take several
// passes, each reloading the window's first taps - 2 rows).
constexpr int PMAX = 2;

// One level of the cascade for this thread's channel vector vt and its run
// of outputs [jb, jb + cnt), cnt <= PMAX: out[j] = sum_k h[k] in[2 j + k].
// RAW: the input is the gathered rows (T, row-major DS channels); else fp32
// rows in 16-byte planes (plane p of vector vt at byte p * 16 VT + 16 vt of
// the row).  LAST: outputs go to global memory rounded to T (rows below
// `valid` only); else to the fp32 rows at dst.  The run is unrolled, so the
// sliding window lives in renamed registers.
template <typename T, int TAPS, int DS, bool RAW>
__device__ __forceinline__ void cascade_level(const uint8_t* src, uint8_t* dst, int jb, int cnt, int vt, bool last,
                                              int valid, T* ob, int64_t out_row, const f32x2 (&h2)[4], f32x2 c2) {
  constexpr int VEC = Vec<T>::N, VT = DS / VEC, NP = VEC / 4;
  constexpr int IN_ROW = RAW ? DS * (int)sizeof(T) : DS * 4;  // bytes per input row
  const uint8_t* sp = src + (2 * jb) * IN_ROW + 16 * vt;
  auto load = [&](int row, Lanes<T>& o) {
    if (RAW) {
      widen(*reinterpret_cast<const uint4*>(sp + row * IN_ROW), o);
    } else {
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(sp + row * IN_ROW + p * 16 * VT);
        o.v[2 * p] = q.x;
        o.v[2 * p + 1] = q.y;
      }
    }
  };
  Lanes<T> x[2 * PMAX + TAPS - 2];  // rows 2 jb + i of the run's window
#pragma unroll
  for (int i = 0; i < TAPS - 2; ++i) load(i, x[i]);
#pragma unroll
  for (int t = 0; t < PMAX; ++t) {
    if (t < cnt) {
      load(2 * t + TAPS - 2, x[2 * t + TAPS - 2]);
      load(2 * t + TAPS - 1, x[2 * t + TAPS - 1]);
      Lanes<T> y;
#pragma unroll
      for (int i = 0; i < VEC / 2; ++i) {
        if (TAPS == 2) {
          y.v[i] = mul2(add2(x[2 * t].v[i], x[2 * t + 1].v[i]), c2);
        } else {
          f32x2 a = mul2(h2[0], x[2 * t].v[i]);
#pragma unroll
          for (int k = 1; k < TAPS; ++k) a = fma2(h2[k], x[2 * t + k].v[i], a);
          y.v[i] = a;
        }
      }
      const int j = jb + t;
      if (last) {
        if (j < valid) *reinterpret_cast<uint4*>(ob + (int64_t)j * out_row + vt * VEC) = narrow(y);
      } else {
#pragma unroll
        for (int p = 0; p < NP; ++p)
          *reinterpret_cast<ulonglong2*>(dst + j * DS * 4 + p * 16 * VT + 16 * vt) =
              make_ulonglong2(y.v[2 * p], y.v[2 * p + 1]);
      }
    }
  }
}

// Quotient and remainder by an invariant divisor with a multiply and a shift
// (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994): for 0 <= x < 2^31 and d >= 1, with
// l = ceil(log2 d) and mul = floor(2^32 (2^l - d) / d) + 1,
// x / d = (umulhi(mul, x) + x) >> l.
struct FastDiv {
  uint32_t d, mul, shift;
};
inline FastDiv make_fastdiv(uint32_t d) {
  FastDiv f;
  f.d = d;
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;
  f.shift = l;
  f.mul = (uint32_t)((((1ull << l) - d) << 32) / d + 1);
  return f;
}
__device__ __forceinline__ uint32_t fastdiv(uint32_t x, const FastDiv& f) {
  return (__umulhi(f.mul, x) + x) >> f.shift;
}

// Shared memory: the gathered rows as loaded (T), then the fp32 levels
// alternating between a second buffer and the first one (which holds at
// least as many fp32 rows as the level after the first needs), then the
// gathered rows' token indices.
template <typename T, int TAPS, int DS>
__global__ void __launch_bounds__(NTH, 3) approx_kernel(const T* __restrict__ K, int64_t ksb, int64_t ksh, int64_t kss,
                                                     int64_t n, FastDiv heads, const int32_t* __restrict__ cand,
                                                     int64_t cand_stride, int m, int level, Taps taps,
                                                     T* __restrict__ out, int64_t out_unit, int64_t out_row) {
  extern __shared__ __align__(16) uint8_t sbuf[];
  constexpr int VEC = Vec<T>::N;
  constexpr int VT = DS / VEC;   // vector threads across a row
  constexpr int RT = NTH / VT;   // run threads
  static_assert(NTH % VT == 0 && (VT & (VT - 1)) == 0, "a row's vectors split evenly");
  const int to = outputs_per_cta(level);
  const int nin = rows_needed(to, level, TAPS);
  uint8_t* X = sbuf;                                                             // raw rows, later fp32 levels
  uint8_t* Y = sbuf + ((size_t)nin * DS * sizeof(T) + 15) / 16 * 16;             // fp32 levels 1, 3, ...
  int* tok = reinterpret_cast<int*>(Y + (size_t)(nin / 2 + 1) * DS * 4);         // token of each gathered row
  // The channel slice varies fastest, so the slices of the same rows are read
  // by neighbouring CTAs at about the same time.
  const int u = blockIdx.z;
  const int j0 = blockIdx.y * to;
  const int c0 = blockIdx.x * DS;
  const uint32_t bb = fastdiv((uint32_t)u, heads), hh = (uint32_t)u - bb * heads.d;
  const int len = m << level;  // the gathered sequence (< 2^31 tokens)
  const int blk_mask = (1 << level) - 1;
  const int32_t* cd = cand ? cand + (int64_t)u * cand_stride : nullptr;
  const int tid = threadIdx.x;
  grid_dep_wait();  // the candidates (and the output's previous readers) come from the grids before
  grid_dep_launch();

  // Row r is gathered position (j0 2^b + r) mod len: its token first, then
  // 16-byte copies, VT a row.
  const int base = j0 << level;  // j0 < m, so base < len
  for (int r = tid; r < nin; r += NTH) {
    int p = base + r;
    if (p >= len) p = p - len < len ? p - len : p % len;  // the filter's reach wraps around
    int64_t tl = cd ? ((int64_t)cd[p >> level] << level) + (p & blk_mask) : p;
    tok[r] = (int)(tl < 0 ? 0 : (tl >= n ? n - 1 : tl));  // out-of-range block indices are clamped
  }
  __syncthreads();
  {
    const T* src = K + (int64_t)bb * ksb + (int64_t)hh * ksh + c0 + (tid % VT) * VEC;
    const uint32_t xs = (uint32_t)__cvta_generic_to_shared(X) + (uint32_t)((tid % VT) * VEC * sizeof(T));
#pragma unroll 4
    for (int r = tid / VT; r < nin; r += RT)
      cp_async16(xs + (uint32_t)(r * DS * sizeof(T)), src + (int64_t)tok[r] * kss);
  }
  cp_async_wait_all();
  __syncthreads();

  const float c32 = 0.70710678118654752440f;  // fl32(1 / sqrt 2)
  const f32x2 c2 = pk2(c32, c32);
  f32x2 h2[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) h2[k] = pk2(taps.h[k], taps.h[k]);
  const int vt = tid % VT, rt = tid / VT;
  // The last level's outputs are rows j0 .. j0 + to - 1, those below m written.
  T* obl = out + (int64_t)u * out_unit + c0 + (int64_t)j0 * out_row;
  const int valid = m - j0;
#pragma unroll 1
  for (int l = 1; l <= level; ++l) {
    const int nout = rows_needed(to, level - l, TAPS);
    const bool last = l == level;
    uint8_t* dst = (l & 1) ? Y : X;
    const int per = (nout + RT - 1) / RT;
    const int je = min(nout, (rt + 1) * per);
#pragma unroll 1
    for (int jb = rt * per; jb < je; jb += PMAX) {
      const int cnt = min(je - jb, PMAX);
      if (l == 1)
        cascade_level<T, TAPS, DS, true>(X, dst, jb, cnt, vt, last, valid, obl, out_row, h2, c2);
      else
        cascade_level<T, TAPS, DS, false>((l & 1) ? X : Y, dst, jb, cnt, vt, last, valid, obl, out_row, h2, c2);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Scales 1 to 5: the cascade streamed through registers.
// ---------------------------------------------------------------------------
// A thread owns one 16-byte vector of channels and a run of consecutive
// outputs.  It reads its input rows in order, one candidate block of 2^L rows
// after the other (the sequence is made of whole blocks, so a block needs one
// index), and pushes each row through all L levels at once.  Level l keeps of
// its past inputs only the first half of the next output's sum,
// fma(h[1], x1, h[0] x0), plus an unpaired input; every output is finished by
// two more fused multiply-adds, in the order of the storage rule above, so
// the results are the same bits.  A db2 output reaches 2 (2^L - 1) rows past
// its own block: a run reads two blocks more than it has outputs (one at
// L = 1), wrapping around the sequence.
//
// What bounds it: HBM.  Nothing goes through shared memory and no barrier
// separates loading from computing: a thread loads its next 8 rows before it
// works on the current 8, and the 16 warps an SM holds keep about 64 KB in
// flight.  (Gathering 128 rows into shared memory, then transforming them
// level by level between barriers, left DRAM at 44 % at scale 3.)  Measured:
// the db2 step of 64 units x 32K tokens 233.1 -> 218.1 us (187.7 with one unit
// a cluster); its three transforms move 546 MB through DRAM, one by one and cold
// in 98.6 us (5.5 TB/s, 0.81 of a copy's rate), in the step in about 84, 99 us
// before.  Scales 6 to 10 (a long halo, few outputs) keep the shared-memory kernel
// below.
template <typename T, int TAPS, int L>
struct Cascade {
  static constexpr int VEC = Vec<T>::N;
  static constexpr float c = 0.70710678118654752440f;  // fl32(1 / sqrt 2)
  f32x2 h2[4];
  Lanes<T> half[L + 1];  // an input whose pair is still to come
  Lanes<T> acc[L + 1];   // h[0] x0 + h[1] x1 of the pair before
  // Input E of the chunk (2^(L - LV + 1) inputs of level LV a block).  A db2
  // output needs the pair after its own, so level 1 gives output j - 1 with
  // pair j: the inputs of level 2 start at an odd index; level 2's shift of
  // one more makes the later levels even again.
  template <int LV, int E, typename F>
  __device__ __forceinline__ void push(const Lanes<T>& x, F&& emit) {
    constexpr int off = TAPS == 4 && LV == 2 ? 1 : 0;
    if constexpr (((E + off) & 1) == 0) {
      half[LV] = x;
    } else {
      Lanes<T> y;
#pragma unroll
      for (int i = 0; i < VEC / 2; ++i) {
        if constexpr (TAPS == 2) {
          // Scalar: the compiler merges a packed product with the next
          // level's packed sum, which would skip the product's rounding.
          const float2 a = up2(half[LV].v[i]), b = up2(x.v[i]);
          y.v[i] = pk2(__fmul_rn(__fadd_rn(a.x, b.x), c), __fmul_rn(__fadd_rn(a.y, b.y), c));
        } else {
          y.v[i] = fma2(h2[3], x.v[i], fma2(h2[2], half[LV].v[i], acc[LV].v[i]));
          acc[LV].v[i] = fma2(h2[1], x.v[i], mul2(h2[0], half[LV].v[i]));
        }
      }
      if constexpr (LV == L) emit(y);
      else push<LV + 1, (E + off - 1) / 2>(y, emit);
    }
  }
  // Rows E .. E + N - 1 of a block, as loaded.
  template <int E, int N, typename F>
  __device__ __forceinline__ void rows(const uint4* w, F&& emit) {
    if constexpr (N > 0) {
      Lanes<T> x;
      widen(*w, x);
      push<1, E>(x, emit);
      rows<E + 1, N - 1>(w + 1, emit);
    }
  }
};

constexpr int kStreamThreads = 128;
constexpr int kStreamMaxLevel = 5;

// CTAs an SM: 128 registers a thread hold the cascade's state up to scale 3;
// eight db2 channels at scales 4 and 5 need more.
template <typename T, int TAPS, int L>
__host__ __device__ constexpr int stream_ctas() {
  return Vec<T>::N == 8 && TAPS == 4 && L >= 4 ? 3 : 4;
}

template <typename T, int TAPS, int L, int D>
__global__ void __launch_bounds__(kStreamThreads, (stream_ctas<T, TAPS, L>()))
    approx_stream_kernel(const T* __restrict__ K, int64_t ksb, int64_t ksh, int64_t kss, int64_t n, FastDiv heads,
                         const int32_t* __restrict__ cand, int64_t cand_stride, int m, int run, Taps taps,
                         T* __restrict__ out, int64_t out_unit) {
  constexpr int VEC = Vec<T>::N, LPR = D / VEC;    // lanes a row
  constexpr int DLY = TAPS == 2 ? 0 : (L == 1 ? 1 : 2);  // blocks read before the first output
  constexpr int RG = 8;                              // rows a load group
  constexpr int BPG = L < 3 ? RG >> L : 1;           // blocks a group, or
  constexpr int GPB = L > 3 ? (1 << L) / RG : 1;     // groups a block
  constexpr int BR = L < 3 ? 1 << L : RG;            // rows of a block in a group
  grid_dep_wait();  // the candidates (and the output's previous readers) come from the grids before
  grid_dep_launch();
  const int u = blockIdx.y;
  const int t = (int)blockIdx.x * kStreamThreads + (int)threadIdx.x;
  const int vt = t % LPR, j0 = t / LPR * run;
  if (j0 >= m) return;
  const int cnt = min(run, m - j0);  // outputs of this thread
  const uint32_t bb = fastdiv((uint32_t)u, heads), hh = (uint32_t)u - bb * heads.d;
  const T* src = K + (int64_t)bb * ksb + (int64_t)hh * ksh + vt * VEC;
  T* dst = out + (int64_t)u * out_unit + (int64_t)j0 * D + vt * VEC;
  const int32_t* cd = cand ? cand + (int64_t)u * cand_stride : nullptr;
  const int blocks = cnt + DLY;

  Cascade<T, TAPS, L> cas;
#pragma unroll
  for (int k = 0; k < 4; ++k) cas.h2[k] = pk2(taps.h[k], taps.h[k]);
#pragma unroll
  for (int l = 0; l <= L; ++l)
#pragma unroll
    for (int i = 0; i < VEC / 2; ++i) cas.half[l].v[i] = cas.acc[l].v[i] = pk2(0.f, 0.f);

  // The block indices of the next group to load, read a group ahead of their
  // rows.  Block b of the run is position j0 + b of the sequence,
  // modulo m.
  int pos = j0;
  int32_t ci[BPG];
  auto fetch = [&]() {
#pragma unroll
    for (int b = 0; b < BPG; ++b) {
      ci[b] = cd ? cd[pos] : pos;
      if (++pos >= m) pos = 0;
    }
  };
  // Load group g: BPG whole blocks, or part g % GPB of a block.  A block's
  // row step is 0 for an index outside [0, n >> L): every token of the block is
  // then clamped to the same one.
  const T* row = src;
  int64_t step = 0;
  auto load = [&](int g, uint4 (&w)[RG]) {
#pragma unroll
    for (int b = 0; b < BPG; ++b) {
      if (GPB == 1 || g % GPB == 0) {
        const int64_t t0 = (int64_t)ci[b] << L;
        const bool in = t0 >= 0 && t0 < n;
        row = src + (in ? t0 : (t0 < 0 ? 0 : n - 1)) * kss;
        step = in ? kss : 0;
      }
#pragma unroll
      for (int i = 0; i < BR; ++i) {
        w[b * BR + i] = __ldg(reinterpret_cast<const uint4*>(row));
        row += step;
      }
    }
    if (GPB == 1 || g % GPB == 0) fetch();
  };
  int blk = 0;
  auto emit = [&](const Lanes<T>& y) {
    const int j = blk - DLY;
    if (j >= 0 && j < cnt) *reinterpret_cast<uint4*>(dst + (int64_t)j * D) = narrow(y);
  };
  const int groups = GPB > 1 ? blocks * GPB : (blocks + BPG - 1) / BPG;
  uint4 w[2][RG];
  fetch();
  load(0, w[0]);
#pragma unroll 1
  for (int g = 0; g < groups; g += 2 * GPB) {
    // Two blocks (GPB > 1) or two groups of blocks a turn, so that the buffers
    // and the parts of a block have fixed places.
#pragma unroll
    for (int h = 0; h < 2 * GPB; ++h) {
      if (g + h + 1 < groups) load(h + 1, w[(h + 1) & 1]);
      if (g + h < groups) {
        if constexpr (GPB == 1) {
#pragma unroll
          for (int b = 0; b < BPG; ++b) {
            cas.template rows<0, BR>(w[h & 1] + b * BR, emit);
            ++blk;
          }
        } else if (GPB == 2) {
          if (h % 2 == 0) cas.template rows<0, RG>(w[h & 1], emit);
          else cas.template rows<GPB == 2 ? RG : 0, RG>(w[h & 1], emit);
          if (h % 2 == 1) ++blk;
        } else {
          if (h % 4 == 0) cas.template rows<0, RG>(w[h & 1], emit);
          else if (h % 4 == 1) cas.template rows<GPB == 4 ? RG : 0, RG>(w[h & 1], emit);
          else if (h % 4 == 2) cas.template rows<GPB == 4 ? 2 * RG : 0, RG>(w[h & 1], emit);
          else cas.template rows<GPB == 4 ? 3 * RG : 0, RG>(w[h & 1], emit);
          if (h % 4 == 3) ++blk;
        }
      }
    }
  }
}

// Outputs a thread: as many CTAs as the SMs hold at once, an equal number a
// unit, so that the runs are long enough to hide the two extra blocks and no
// partial second wave is left; at least 4.  But one while that fills at most
// half of the chip: a run's blocks are read one after the other, and a short
// list is bound by that (one unit, 1024 blocks of scale 5, db2, bf16: 11.1 us
// with runs of 4, 6.6 with 1, 10.4 through shared memory; the db2 step of one
// unit x 32K in six scales 96.8 -> 87.5).
inline int stream_run(int64_t units, int m, int lpr, int ctas) {
  int sms = sm_count();
  if (sms <= 0) sms = 148;
  const int64_t per_unit = (int64_t)sms * ctas / units;
  const int64_t runs = (per_unit < 1 ? 1 : per_unit) * (kStreamThreads / lpr);
  if (per_unit >= 1 && m <= runs / 2) return 1;
  const int64_t run = (m + runs - 1) / runs;
  return (int)(run < 4 ? 4 : run);
}

template <typename T, int TAPS, int L, int D>
cudaError_t run_stream(const void* K, const wf_tensor& kv, const int32_t* cand, int64_t cand_stride, int m,
                       const Taps& taps, void* out, int64_t out_unit, cudaStream_t s) {
  constexpr int LPR = D / Vec<T>::N;
  const int64_t units = (int64_t)kv.batch * kv.heads;
  const int run = stream_run(units, m, LPR, stream_ctas<T, TAPS, L>());
  const int64_t threads = (int64_t)((m + run - 1) / run) * LPR;
  return Launch(dim3((unsigned)((threads + kStreamThreads - 1) / kStreamThreads), (unsigned)units), kStreamThreads, 0,
                s)(approx_stream_kernel<T, TAPS, L, D>, static_cast<const T*>(K), kv.stride_b, kv.stride_h, kv.stride_s,
                   (int64_t)kv.seq, make_fastdiv((uint32_t)kv.heads), cand, cand_stride, m, run, taps,
                   static_cast<T*>(out), out_unit);
}

// Shared memory of one CTA for DS channels: the raw rows, the first fp32
// level (the raw buffer holds the later ones) and the row tokens.
template <typename T, int TAPS>
size_t approx_smem(int level, int ds) {
  const int nin = rows_needed(outputs_per_cta(level), level, TAPS);
  return ((size_t)nin * ds * sizeof(T) + 15) / 16 * 16 + sizeof(float) * ds * (size_t)(nin / 2 + 1) +
         sizeof(int) * (size_t)nin;
}

template <typename T, int TAPS, int DS>
cudaError_t run_ds(const void* K, const wf_tensor& kv, const int32_t* cand, int64_t cand_stride, int m, int level,
                   const Taps& taps, void* out, int64_t out_unit, cudaStream_t s) {
  const int to = outputs_per_cta(level);
  const size_t smem = approx_smem<T, TAPS>(level, DS);
  // The shared-memory limit, raised per device to the largest size requested
  // so far (not on every launch).
  static std::mutex mu;
  static std::map<int, size_t> raised;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lock(mu);
    size_t& cur = raised[dev];
    if (cur < smem) {
      e = cudaFuncSetAttribute(approx_kernel<T, TAPS, DS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      cur = smem;
    }
  }
  return Launch(dim3((unsigned)(kv.head_dim / DS), (unsigned)((m + to - 1) / to), (unsigned)(kv.batch * kv.heads)), NTH,
                smem, s)(approx_kernel<T, TAPS, DS>, static_cast<const T*>(K), kv.stride_b, kv.stride_h, kv.stride_s,
                         (int64_t)kv.seq, make_fastdiv((uint32_t)kv.heads), cand, cand_stride, m, level, taps,
                         static_cast<T*>(out), out_unit, (int64_t)kv.head_dim);
}

// Scales above kStreamMaxLevel: whole rows of 128 channels per CTA (each row's
// token resolved once, 256-byte copies of bf16) while the shared memory
// allows, else 64 channels, else 16 (the deepest scales).
template <typename T, int TAPS, int D>
cudaError_t run_d(const void* K, const wf_tensor& kv, const int32_t* cand, int64_t cand_stride, int m, int level,
                  const Taps& taps, void* out, int64_t out_unit, cudaStream_t s) {
  switch (level) {
    case 1: return run_stream<T, TAPS, 1, D>(K, kv, cand, cand_stride, m, taps, out, out_unit, s);
    case 2: return run_stream<T, TAPS, 2, D>(K, kv, cand, cand_stride, m, taps, out, out_unit, s);
    case 3: return run_stream<T, TAPS, 3, D>(K, kv, cand, cand_stride, m, taps, out, out_unit, s);
    case 4: return run_stream<T, TAPS, 4, D>(K, kv, cand, cand_stride, m, taps, out, out_unit, s);
    default: return run_stream<T, TAPS, 5, D>(K, kv, cand, cand_stride, m, taps, out, out_unit, s);
  }
}

template <typename T, int TAPS>
cudaError_t run(const void* K, const wf_tensor& kv, const int32_t* cand, int64_t cand_stride, int m, int level,
                const Taps& taps, void* out, int64_t out_unit, cudaStream_t s) {
  if (level <= kStreamMaxLevel && kv.batch * kv.heads <= 65535)
    return kv.head_dim == 64 ? run_d<T, TAPS, 64>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s)
                             : run_d<T, TAPS, 128>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s);
  if (kv.head_dim == 128 && approx_smem<T, TAPS>(level, 128) <= 200 * 1024)
    return run_ds<T, TAPS, 128>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s);
  if (approx_smem<T, TAPS>(level, 64) <= 200 * 1024)
    return run_ds<T, TAPS, 64>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s);
  return run_ds<T, TAPS, 16>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s);
}

}  // namespace

int wavelet_taps(int wavelet) { return wavelet == WF_WAVELET_HAAR ? 2 : (wavelet == WF_WAVELET_DB2 ? 4 : 0); }

int wavelet_max_level(int wavelet) { return wavelet == WF_WAVELET_DB2 ? 8 : 10; }

cudaError_t launch_wavelet_approx(const void* K, const wf_tensor& kv, const int32_t* cand, int64_t cand_stride, int m,
                                  int level, int wavelet, void* out, int64_t out_unit, cudaStream_t s) {
  Taps taps{};
  if (wavelet == WF_WAVELET_DB2) {
    // Daubechies' two-vanishing-moment scaling filter, from its closed form.
    const double r = sqrt(3.0), q = 4.0 * sqrt(2.0);
    const double h[4] = {(1.0 + r) / q, (3.0 + r) / q, (3.0 - r) / q, (1.0 - r) / q};
    for (int k = 0; k < 4; ++k) taps.h[k] = (float)h[k];
    return kv.dtype == WF_BF16 ? run<bf16, 4>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s)
                               : run<float, 4>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s);
  }
  return kv.dtype == WF_BF16 ? run<bf16, 2>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s)
                             : run<float, 2>(K, kv, cand, cand_stride, m, level, taps, out, out_unit, s);
}

}  // namespace wf
