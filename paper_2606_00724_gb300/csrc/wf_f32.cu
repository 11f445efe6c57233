// One layer in fp32 in one launch: the multi-scale filter (Eq. 7-11) and the
// sparse attention, for one query head per key head with at most 64 query
// rows and head_dim 64 or 128.
//
// A thread-block cluster serves one (batch, head) unit; each CTA (8 warps)
// holds one contiguous slice of the unit's candidate list at every scale, and
// finally of its sparse key list:
//   rows    the slice's rows gathered into shared memory (16-byte cp.async),
//           all at once where they fit;
//   logits  2 rows x QM / 4 queries a thread in packed fp32 FMAs, queries read
//           as warp-wide broadcasts, kept in shared memory as [query][row];
//   stats   (max, sum of exp) per query over the slice, four queries a warp at a
//           time, exchanged over the cluster;
//   keys    log W_j of each row (the sum over the queries against the cluster's
//           normalisers), written into every CTA's key array;
//   Top-K   the same selection in every CTA, giving the next scale's rows;
//   attention over the slice with a running max per query, partial outputs
//           combined from the cluster's shared memories.
// Exact fp32 throughout: fused multiply-adds, expf and logf.
//
// What bounds it: the chain of dependent phases of a scale (gather, FMAs,
// two cluster exchanges, Top-K), so the cluster is as wide as the SMs and 8
// CTAs allow, which shortens the gather and the FMAs.  A 2 x 8 register tile
// takes 16 shared-memory wavefronts for 64 FMAs a lane, which is the most that
// the reads allow; the FMAs are packed pairs of channels, so that they do not
// also fill the issue slots.  Measured against three kernels a scale
// and two for the attention: 4 heads x 1K tokens (d 64) 64.9 -> 19.2 us a
// step, 16 heads x 8K (d 128) 170.6 -> 73.2 us, the error against 64 bits
// no larger (3.1e-7 and 2.3e-6; 5.6e-7 and 3.8e-6 before).
#include <float.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "wf_internal.cuh"
#include "wf_sm100.cuh"
#include "wf_topk.cuh"

namespace wf {
namespace {

using namespace sm100;
using namespace topk;

constexpr int NTH = 2 * NCT;  // threads: both warpgroups of a WIDE Top-K
constexpr int NW = NTH / 32;
constexpr int MAXCS = 8;

struct F32Params {
  const float* Q;
  int64_t qsb, qsh, qss;
  const float* K;
  const float* V;
  int64_t ksb, ksh, kss;
  const float* Kg;
  const float* Vg;
  int64_t gsb, gsh, gss;
  const float* coeffs;
  int64_t rows_total;
  float* O;
  int64_t osb, osh, oss;
  int32_t* idx;
  int32_t* level_sets;
  int64_t sets_stride;
  int q, n, ng, H, L, trim, attn;
  int trow, srow, bufw;  // rows of the row buffer, floats of a query's logit row, words of a key buffer
  int32_t keep[12];
  float scale;
};

// Shared memory (byte offsets).
struct F32Layout {
  uint32_t q, tile, s, buf, sel, stat, total;
};
struct F32Stat {
  float2 xstat[MAXCS][64];  // (max, sum of exp) per query of every CTA's slice
  float2 kmm[MAXCS][NW];    // (min, max) of every warp's keys
  float xch[128];           // second half's sum per row
  float ms[64];             // the normalisers; the attention's running max
  float l[64];              // the attention's running row sums
  float alpha[64];          // this tile's factor of the partial output
};
__host__ __device__ inline F32Layout f32_layout(int D, int QM, int trow, int srow, int bufw) {
  F32Layout y;
  y.q = 0;
  y.tile = y.q + 4u * (uint32_t)(QM * D);
  y.s = y.tile + 4u * (uint32_t)(trow * (D + 4));
  y.buf = y.s + 4u * (uint32_t)(QM * srow);
  y.sel = y.buf + 2u * 4u * (uint32_t)bufw;
  y.stat = y.sel + (uint32_t)((sizeof(SelScratch) + 15) / 16 * 16);
  y.total = y.stat + (uint32_t)((sizeof(F32Stat) + 15) / 16 * 16);
  return y;
}

// CTA `rank`'s part of a list of m candidates, sibling pairs kept together
// (unit 2), or of m keys (unit 1): the rows [g0, g0 + mc).
__host__ __device__ inline void slice_of(int m, int unit, int rank, int cs, int& g0, int& mc) {
  const int items = (m + unit - 1) / unit;
  g0 = min(m, unit * (rank * items / cs));
  mc = min(m, unit * ((rank + 1) * items / cs)) - g0;
}

__device__ __forceinline__ float4 ld_cluster_v4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}

// Rows [t0, t0 + cnt) of a list into a tile (row stride D + 4 floats); row(j)
// is the address of the list's row j.
template <int D, typename F>
__device__ __forceinline__ void gather(float* tile, int t0, int cnt, F&& row) {
  constexpr int LPR = D / 4;  // lanes a row
  const int c = threadIdx.x % LPR;
#pragma unroll 4
  for (int r = threadIdx.x / LPR; r < cnt; r += NTH / LPR)
    cp_async16(smem_u32(tile + r * (D + 4) + 4 * c), row(t0 + r) + 4 * c);
}

// Rows of a tile for a list of mc rows in tiles of at most cap: equal tiles,
// a multiple of 4.
__device__ __forceinline__ int tile_rows(int mc, int cap) {
  const int nt = max((mc + cap - 1) / cap, 1);
  return ((mc + nt - 1) / nt + 3) & ~3;
}

// Logits (x scale) of rows r0 + lane (+ 32 i, i < RPL) of a tile against QG
// queries from q0 into S[query][t0 + row].  Rows past the tile's cnt compute
// whatever the tile holds and are not stored.  Each accumulator is a packed
// pair, the sums over the even and the odd channels.
template <int D, int RPL, int QG>
__device__ __forceinline__ void score_item(const float* Qs, const float* tile, float* S, int srow, int t0, int cnt,
                                           int r0, int q0, float scale) {
  const int r = r0 + (threadIdx.x & 31);
  const ulonglong2* p[RPL];
#pragma unroll
  for (int i = 0; i < RPL; ++i) p[i] = reinterpret_cast<const ulonglong2*>(tile + min(r + 32 * i, cnt - 1) * (D + 4));
  f32x2 a[RPL][QG];
#pragma unroll
  for (int i = 0; i < RPL; ++i)
#pragma unroll
    for (int k = 0; k < QG; ++k) a[i][k] = pk2(0.f, 0.f);
#pragma unroll 2
  for (int c = 0; c < D / 4; ++c) {
    ulonglong2 x[RPL];
#pragma unroll
    for (int i = 0; i < RPL; ++i) x[i] = p[i][c];
#pragma unroll
    for (int k = 0; k < QG; ++k) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(Qs + (q0 + k) * D + 4 * c);
#pragma unroll
      for (int i = 0; i < RPL; ++i) a[i][k] = fma2(v.y, x[i].y, fma2(v.x, x[i].x, a[i][k]));
    }
  }
#pragma unroll
  for (int k = 0; k < QG; ++k) {
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const float2 z = up2(a[i][k]);
      if (r + 32 * i < cnt) S[(q0 + k) * srow + t0 + r + 32 * i] = (z.x + z.y) * scale;
    }
  }
}

// A tile's rows against every query: a tile of at most 32 rows splits its
// queries over all the warps, a larger one goes 64 rows x QM / 4 queries a warp
// at a time.
template <int D, int QM>
__device__ __forceinline__ void score_tile(const float* Qs, const float* tile, float* S, int srow, int t0, int cnt,
                                           float scale) {
  const int w = threadIdx.x >> 5;
  if (cnt <= 32) {
    if (cnt > 0) score_item<D, 1, QM / NW>(Qs, tile, S, srow, t0, cnt, 0, QM / NW * w, scale);
    return;
  }
#pragma unroll 1
  for (int it = w; it < 4 * ((cnt + 63) / 64); it += NW)
    score_item<D, 2, QM / 4>(Qs, tile, S, srow, t0, cnt, 64 * (it >> 2), QM / 4 * (it & 3), scale);
}

// Four queries' rows of S (srow apart) over cnt rows, by one warp: their maxima
// (at least m0) and the sums of exp(s - max); with P, the exponentials replace
// the logits and zeros follow up to row pad.
template <bool P>
__device__ __forceinline__ void row_stats(float* s, int srow, int cnt, int pad, float (&mx)[4], float (&z)[4]) {
  const int lane = threadIdx.x & 31;
  for (int j = lane; j < cnt; j += 32)
#pragma unroll
    for (int k = 0; k < 4; ++k) mx[k] = fmaxf(mx[k], s[k * srow + j]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    mx[k] = warp_max_f32(mx[k]);
    z[k] = 0.f;
  }
  for (int j = lane; j < (P ? pad : cnt); j += 32)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float e = !P || j < cnt ? expf(s[k * srow + j] - mx[k]) : 0.f;
      if (P) s[k * srow + j] = e;
      z[k] += e;
    }
#pragma unroll
  for (int o = 16; o; o >>= 1)
#pragma unroll
    for (int k = 0; k < 4; ++k) z[k] += __shfl_xor_sync(0xffffffffu, z[k], o);
}

template <int D, int QM>
__global__ void __launch_bounds__(NTH, 1) wf_f32_kernel(const __grid_constant__ F32Params p) {
  extern __shared__ __align__(16) uint8_t smem[];
  const F32Layout ly = f32_layout(D, QM, p.trow, p.srow, p.bufw);
  float* Qs = reinterpret_cast<float*>(smem + ly.q);
  float* T0 = reinterpret_cast<float*>(smem + ly.tile);
  float* S = reinterpret_cast<float*>(smem + ly.s);
  F32Stat& st = *reinterpret_cast<F32Stat*>(smem + ly.stat);
  const uint32_t sc_a = smem_u32(smem + ly.sel);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster_rank(), cs = (int)cluster_size();
  const int u = (int)cluster_id_x();
  const int64_t bb = u / p.H, hh = u % p.H;
  auto buf = [&](int lev) { return reinterpret_cast<int32_t*>(smem + ly.buf) + ((p.L - lev) & 1) * p.bufw; };

  grid_dep_wait();
  grid_dep_launch();
  // The query block (rows past q zero) with the first tile's copies; the
  // Top-K scratch starts zeroed.
  for (int e = tid; e < QM * (D / 4); e += NTH) {
    const int i = e / (D / 4), c = e % (D / 4);
    cp_async16_zfill(smem_u32(Qs + i * D + 4 * c),
                     p.Q + bb * p.qsb + hh * p.qsh + (int64_t)min(i, p.q - 1) * p.qss + 4 * c, i < p.q);
  }
  for (int e = tid; e < (int)((sizeof(SelScratch) + 15) / 16); e += NTH)
    *reinterpret_cast<uint4*>(smem + ly.sel + 16 * e) = make_uint4(0, 0, 0, 0);
  cluster_sync();  // every CTA of the cluster runs before any remote store

  // S = scale Q rows^T of a list of mc rows.
  auto score_list = [&](int mc, auto&& row) {
    const int tr = tile_rows(mc, p.trow);
    for (int t0 = 0; t0 < mc; t0 += tr) {
      const int cnt = min(tr, mc - t0);
      gather<D>(T0, t0, cnt, row);
      cp_async_wait_all();
      __syncthreads();
      score_tile<D, QM>(Qs, T0, S, p.srow, t0, cnt, p.scale);
      __syncthreads();
    }
    cp_async_wait_all();  // (an empty list's query block)
    __syncthreads();
  };

  int64_t sets_off = 0;
  const int lev_end = p.trim ? 0 : 1;
#pragma unroll 1
  for (int lev = p.L; lev >= lev_end; --lev) {
    const bool top = lev == p.L;
    const int m = top ? p.n >> p.L : 2 * p.keep[lev + 1];
    int g0, mc;
    slice_of(m, 2, rank, cs, g0, mc);
    const int32_t* Jp = buf(lev + 1);  // the selection one scale up
    {
      const float* base;
      int64_t rs;
      if (lev >= 1) {
        base = p.coeffs + ((int64_t)u * p.rows_total + ((int64_t)p.n - ((int64_t)p.n >> (lev - 1)))) * D;
        rs = D;
      } else {
        base = p.K + bb * p.ksb + hh * p.ksh;
        rs = p.kss;
      }
      score_list(mc, [&](int j) {
        const int pos = g0 + j;
        return base + (int64_t)(top ? pos : 2 * Jp[pos >> 1] + (pos & 1)) * rs;
      });
    }
    // (max, sum of exp) of every query over the slice, to every CTA.
    for (int i = 4 * warp; i < QM; i += 4 * NW) {
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY}, z[4];
      row_stats<false>(S + i * p.srow, p.srow, mc, 0, mx, z);
      if (lane < cs)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          st_cluster_v2f32(map_rank(smem_u32(&st.xstat[rank][i + k]), (uint32_t)lane), mx[k], z[k]);
    }
    cluster_sync();
    if (tid < QM) {
      float2 x[MAXCS];
      float M = -INFINITY;
#pragma unroll
      for (int r = 0; r < MAXCS; ++r) {
        x[r] = r < cs ? st.xstat[r][tid] : make_float2(-INFINITY, 0.f);
        if (x[r].y > 0.f) M = fmaxf(M, x[r].x);
      }
      float z = 0.f;
#pragma unroll
      for (int r = 0; r < MAXCS; ++r)
        if (x[r].y > 0.f) z = fmaf(x[r].y, expf(x[r].x - M), z);
      st.ms[tid] = M + logf(z);
    }
    __syncthreads();
    // Ranking keys: the two warpgroups take half the queries each of 128 rows.
    int32_t* J = buf(lev);  // receives this scale's keys, then its selection
    float kmin = INFINITY, kmax = -INFINITY;
    {
      // Every exponent s - ms is at most 0 (ms is the log of a sum that contains
      // the row's own term), so the sum is taken unshifted; a row whose sum is
      // tiny (below 1e-28, where flushed terms could matter) is taken again
      // shifted by its largest exponent.
      const int h = tid >> 7, rl = tid & 127;
      const int i0 = h * ((p.q + 1) / 2), i1 = h ? p.q : (p.q + 1) / 2;
      for (int t0 = 0; t0 < mc; t0 += 128) {
        const int j = t0 + rl;
        float z = 0.f;
        if (j < mc) {
#pragma unroll 8
          for (int i = i0; i < i1; ++i) z += expf(S[i * p.srow + j] - st.ms[i]);
        }
        if (h) st.xch[rl] = z;
        __syncthreads();
        if (!h && j < mc) {
          z += st.xch[rl];
          float key = logf(z);
          if (z < 1e-28f) {
            float mx = -INFINITY;
            for (int i = 0; i < p.q; ++i) mx = fmaxf(mx, S[i * p.srow + j] - st.ms[i]);
            z = 0.f;
            for (int i = 0; i < p.q && mx > -INFINITY; ++i) z += expf((S[i * p.srow + j] - st.ms[i]) - mx);
            key = mx + logf(z);
          }
          kmin = fminf(kmin, key);
          kmax = fmaxf(kmax, key);
          const uint32_t dst = smem_u32(J + g0 + j);
          for (int r = 0; r < cs; ++r) st_cluster_f32(map_rank(dst, (uint32_t)r), key);
        }
        __syncthreads();
      }
    }
    kmin = warp_min_f32(kmin);
    kmax = warp_max_f32(kmax);
    if (lane < cs) st_cluster_v2f32(map_rank(smem_u32(&st.kmm[rank][warp]), (uint32_t)lane), kmin, kmax);
    cluster_sync();
    float lo = INFINITY, hi = -INFINITY;
    for (int e = lane; e < cs * NW; e += 32) {
      const float2 v = st.kmm[e / NW][e % NW];
      lo = fminf(lo, v.x);
      hi = fmaxf(hi, v.y);
    }
    lo = warp_min_f32(lo);
    hi = warp_max_f32(hi);
    // Eq. 9 (the same result in every CTA; ends on a barrier).
    const int kb = p.keep[lev];
    select_topk<true>(smem_u32(J), m, kb, smem_u32(Jp), top, sc_a, lo, hi);
    if (rank == 0) {
      int32_t* ls = p.level_sets ? p.level_sets + (int64_t)u * p.sets_stride + sets_off : nullptr;
      if (lev >= 1 && ls)
        for (int i = tid; i < kb; i += NTH) ls[i] = J[i];
      if (lev == lev_end) {
        // mu^0: the children of J^1, or the trimmed level-0 selection.
        const int kk = p.keep[0];
        int32_t* out = p.idx + (int64_t)u * kk;
        int32_t* ls0 = ls ? ls + (lev >= 1 ? kb : 0) : nullptr;
        for (int t = tid; t < kk; t += NTH) {
          const int tok = p.trim ? J[t] : 2 * J[t >> 1] + (t & 1);
          out[t] = tok;
          if (ls0) ls0[t] = tok;
        }
      }
    }
    if (lev >= 1) sets_off += kb;
  }

  if (p.attn) {
    // The slice [a0, a0 + mc) of the sparse key list [mu^0; generation rows].
    int a0, mc;
    slice_of(p.keep[0] + p.ng, 1, rank, cs, a0, mc);
    const int32_t* J = buf(lev_end);
    const int64_t kb0 = bb * p.ksb + hh * p.ksh, gb0 = bb * p.gsb + hh * p.gsh;
    auto row_of = [&](const float* base, const float* gbase, int j) {
      const int pos = a0 + j;
      if (pos >= p.keep[0]) return gbase + gb0 + (int64_t)(pos - p.keep[0]) * p.gss;
      const int tok = p.trim ? J[pos] : 2 * J[pos >> 1] + (pos & 1);
      return base + kb0 + (int64_t)tok * p.kss;
    };
    auto krow = [&](int j) { return row_of(p.K, p.Kg, j); };
    auto vrow = [&](int j) { return row_of(p.V, p.Vg, j); };
    if (tid < 64) {
      st.ms[tid] = -FLT_MAX;  // finite, so that a tile of logits -inf has P = 0, not exp(-inf + inf)
      st.l[tid] = 0.f;
    }
    // Output accumulators: a thread holds 4 channels of QG queries over one of
    // NS interleaved subsets of the tile's keys (4 keys at a time).
    constexpr int LPR = D / 4, QG = QM / 4, NS = 2 * (32 / LPR);
    const int d4 = 4 * (lane % LPR), q0 = QG * (warp & 3), sub = (warp >> 2) * (32 / LPR) + lane / LPR;
    float acc[QG][4];
#pragma unroll
    for (int i = 0; i < QG; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
    // K and V tiles in the two halves of the row buffer; the next tile's K rows
    // are copied under the softmax, its V rows under the next logits.
    const int cap = min(p.trow / 8 * 4, p.srow - 4), tr = tile_rows(mc, cap);
    float* T1 = T0 + cap * (D + 4);
    gather<D>(T0, 0, min(tr, mc), krow);
    cp_async_commit();
    gather<D>(T1, 0, min(tr, mc), vrow);
    cp_async_commit();
    for (int t0 = 0; t0 < mc; t0 += tr) {
      const int cnt = min(tr, mc - t0), pad = (cnt + 3) & ~3, nxt = min(tr, max(mc - t0 - tr, 0));
      cp_async_wait<1>();  // K (V's copies are the newest group)
      __syncthreads();
      score_tile<D, QM>(Qs, T0, S, p.srow, 0, cnt, p.scale);
      __syncthreads();
      gather<D>(T0, t0 + tr, nxt, krow);
      cp_async_commit();
      // P = exp(s - m) against the running max, zeros up to a multiple of 4 keys.
      for (int i = 4 * warp; i < QM; i += 4 * NW) {
        float mo[4], mx[4], z[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) mx[k] = mo[k] = st.ms[i + k];
        row_stats<true>(S + i * p.srow, p.srow, cnt, pad, mx, z);
        __syncwarp();
        if (lane == 0)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float a = expf(mo[k] - mx[k]);
            st.alpha[i + k] = a;
            st.ms[i + k] = mx[k];
            st.l[i + k] = fmaf(st.l[i + k], a, z[k]);
          }
      }
      // The padding keys' V rows are zero: P is 0 there, and the buffer may
      // hold anything (infinities included).
      for (int e = tid; e < (pad - cnt) * LPR; e += NTH)
        *reinterpret_cast<float4*>(T1 + (cnt + e / LPR) * (D + 4) + 4 * (e % LPR)) = make_float4(0.f, 0.f, 0.f, 0.f);
      cp_async_wait<1>();  // V
      __syncthreads();
      if (t0 > 0) {
#pragma unroll
        for (int i = 0; i < QG; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[i][e] *= st.alpha[q0 + i];
      }
#pragma unroll 1
      for (int j = 4 * sub; j < cnt; j += 4 * NS) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = *reinterpret_cast<const float4*>(T1 + (j + k) * (D + 4) + d4);
#pragma unroll
        for (int i = 0; i < QG; ++i) {
          const float4 w = *reinterpret_cast<const float4*>(S + (q0 + i) * p.srow + j);
          acc[i][0] = fmaf(w.w, v[3].x, fmaf(w.z, v[2].x, fmaf(w.y, v[1].x, fmaf(w.x, v[0].x, acc[i][0]))));
          acc[i][1] = fmaf(w.w, v[3].y, fmaf(w.z, v[2].y, fmaf(w.y, v[1].y, fmaf(w.x, v[0].y, acc[i][1]))));
          acc[i][2] = fmaf(w.w, v[3].z, fmaf(w.z, v[2].z, fmaf(w.y, v[1].z, fmaf(w.x, v[0].z, acc[i][2]))));
          acc[i][3] = fmaf(w.w, v[3].w, fmaf(w.z, v[2].w, fmaf(w.y, v[1].w, fmaf(w.x, v[0].w, acc[i][3]))));
        }
      }
      __syncthreads();
      gather<D>(T1, t0 + tr, nxt, vrow);
      cp_async_commit();
    }
    cp_async_wait_all();
    // The subsets' sums meet in the tile buffer: Op[query][channel].
    float* Op = T0;
    for (int k = NS - 1; k >= 0; --k) {
      if (sub == k) {
#pragma unroll
        for (int i = 0; i < QG; ++i) {
          float4* o = reinterpret_cast<float4*>(Op + (q0 + i) * D + d4);
          float4 v = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
          if (k < NS - 1) {
            const float4 w = *o;
            v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
          }
          *o = v;
        }
      }
      __syncthreads();
    }
    if (tid < QM)
      for (int r = 0; r < cs; ++r)
        st_cluster_v2f32(map_rank(smem_u32(&st.xstat[rank][tid]), (uint32_t)r), st.ms[tid], st.l[tid]);
    cluster_sync();
    // This CTA's share of the outputs, 4 channels an item, from every CTA's
    // partials in CTA order (one without keys weighs 0).
    const int items = p.q * LPR;
    float* ob = p.O + bb * p.osb + hh * p.osh;
    const uint32_t op_a = smem_u32(Op);
    for (int e = rank * items / cs + tid; e < (rank + 1) * items / cs; e += NTH) {
      const int i = e / LPR, c = 4 * (e % LPR);
      float M = -INFINITY;
      for (int r = 0; r < cs; ++r)
        if (st.xstat[r][i].y > 0.f) M = fmaxf(M, st.xstat[r][i].x);
      float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
      float den = 0.f;
#pragma unroll 4
      for (int r = 0; r < cs; ++r) {
        const float2 ml = st.xstat[r][i];
        const float w = ml.y > 0.f ? expf(ml.x - M) : 0.f;
        const float4 v = ld_cluster_v4(map_rank(op_a + 4u * (uint32_t)(i * D + c), (uint32_t)r));
        den = fmaf(ml.y, w, den);
        num.x = fmaf(v.x, w, num.x);
        num.y = fmaf(v.y, w, num.y);
        num.z = fmaf(v.z, w, num.z);
        num.w = fmaf(v.w, w, num.w);
      }
      *reinterpret_cast<float4*>(ob + (int64_t)i * p.oss + c) =
          make_float4(num.x / den, num.y / den, num.z / den, num.w / den);
    }
  }
  cluster_sync();  // no CTA leaves while another may still address its shared memory
}

typedef void (*F32Kernel)(F32Params);
F32Kernel f32_kernel(int d, int q) {
  if (d == 64) return q <= 32 ? wf_f32_kernel<64, 32> : wf_f32_kernel<64, 64>;
  return q <= 32 ? wf_f32_kernel<128, 32> : wf_f32_kernel<128, 64>;
}

// Clusters of cs CTAs that can be resident at once; cached per configuration.
int resident_clusters(F32Kernel k, int cs, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, F32Kernel, int, size_t>, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const auto key = std::make_tuple(dev, k, cs, smem);
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  Launch one(dim3((unsigned)cs), NTH, smem, nullptr, cs);
  int n = 0;
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k), smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &one.cfg);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    n = 0;
  }
  cache.emplace(key, n);
  return n;
}

// fp32, one query head per key head, candidate lists within the Top-K's 8192.
// The largest cluster (up to 8) whose grid fits the SMs in one wave, all
// clusters resident, and whose slice's logits and at least 64 rows fit shared
// memory; else the smallest whose logits fit.
F32Plan fit_f32(const wf_tensor& q, const wf_tensor& kv, int levels, const int32_t* keep, int n_g, int num_sms) {
  F32Plan fp{};
  if (kv.dtype != WF_F32 || q.heads != kv.heads || q.seq > kMaxQ || levels > 10) return fp;
  const int D = kv.head_dim, QM = q.seq <= 32 ? 32 : 64;
  const int U = kv.batch * kv.heads;
  fp.trim = keep[0] < 2 * keep[1];
  int cmax = kv.seq >> levels, kmax = 0;
  for (int l = 0; l <= levels; ++l) kmax = kmax > keep[l] ? kmax : keep[l];
  for (int l = 1; l <= levels; ++l) cmax = cmax > 2 * keep[l] ? cmax : 2 * keep[l];
  if (cmax > kMaxCand || kmax > kMaxCand) return fp;
  fp.bufw = ((cmax > kmax ? cmax : kmax) + 3) / 4 * 4;
  const size_t kMaxSmem = 227 * 1024;
  const F32Kernel k = f32_kernel(D, q.seq);
  auto fit = [&](int cs) {
    // The widest slices of candidates and of keys; the row buffer takes all of
    // the first, and the second's K and V, as far as there is room.
    const int rows = 2 * (((cmax + 1) / 2 + cs - 1) / cs), keys = n_g < 0 ? 0 : (keep[0] + n_g + cs - 1) / cs;
    const int want = std::max({rows, 2 * ((keys + 3) / 4 * 4), 64});
    fp.srow = (std::max(rows, std::min(keys, 128)) + 3) / 4 * 4 + 4;
    const size_t rest = f32_layout(D, QM, 0, fp.srow, fp.bufw).total, row = 4 * (size_t)(D + 4);
    if (rest + 64 * row > kMaxSmem) return false;
    fp.trow = std::min(want, (int)((kMaxSmem - rest) / row)) / 8 * 8;
    fp.smem = f32_layout(D, QM, fp.trow, fp.srow, fp.bufw).total;
    fp.tiles = (rows + fp.trow - 1) / fp.trow;
    return true;
  };
  for (int cs = MAXCS; cs >= 1 && fp.cs == 0; --cs)
    if (U * cs <= num_sms && fit(cs) && U <= resident_clusters(k, cs, fp.smem)) fp.cs = cs;
  for (int cs = 1; cs <= MAXCS && fp.cs == 0; ++cs)
    if (fit(cs) && resident_clusters(k, cs, fp.smem) > 0) fp.cs = cs;
  if (fp.cs == 0) return fp;
  const int at_once = resident_clusters(k, fp.cs, fp.smem);
  fp.waves = (U + at_once - 1) / at_once;
  fp.U = U;
  fp.ok = true;
  return fp;
}

// What the routes of an fp32 call take, in ns, for up to 32 query rows and
// slices of several tiles or waves: fitted to 690 (head_dim 64) and 888 (128)
// measured shapes of that kind, 1 to 304 units, lists of up to 4096, 1 to 32
// query rows; each fit is within 5 % of half of them and 15 % of 95 in 100.
struct F32Cost {
  float f0, frow, fkey;        // one-launch filter: in all; a wave, per gathered row of a CTA, per candidate
  float s0, srow, skey, scan;  // one-launch step: the same; per attended key of a CTA
  float scale, cand, candq, sel;  // kernels per scale: a scale; a unit's candidate, the same per 32 query rows; Top-K
  float a0, att, attq;         // split attention: in all; a unit's key, the same per 32 query rows
};
constexpr F32Cost kCost64 = {5100.f, 33.f, 1.9f, 3900.f, 36.f, 2.8f, 52.f, 17000.f, 0.19f, 0.21f, 1.3f, 12000.f, 0.40f, 0.041f};
constexpr F32Cost kCost128 = {0.f, 63.f, 1.1f, 0.f, 71.f, 1.4f, 87.f, 19000.f, 0.38f, 0.26f, 0.44f, 16000.f, 1.0f, 0.11f};

}  // namespace

// The one launch where it is the faster route (on a near tie too: its sums
// are the more accurate ones).  It always is above 32 query rows, and where all
// clusters run at once with slices of at most two tiles.  Elsewhere (more units than
// clusters at once, slices that do not fit the row buffer) its CTAs compute 32
// query rows for any block, with one CTA an SM, and the kernels per scale catch
// up for small blocks.  Head_dim 64, 8 query rows, 16K tokens, a step: two scales,
// 40 units 219 us against 145, 16 units 67 against 91; four scales, 80 units 292
// against 238, 128 units 296 against 326; with 32 rows 80 units 297 against 318.
// So there the routes' costs are compared.
F32Plan plan_f32(const wf_tensor& q, const wf_tensor& kv, int levels, const int32_t* keep, int n_g, int num_sms) {
  F32Plan fp = fit_f32(q, kv, levels, keep, n_g, num_sms);
  auto at_once = [](const F32Plan& p) { return p.waves == 1 && p.tiles <= 2; };
  if (!fp.ok || q.seq > 32 || at_once(fp)) return fp;
  const F32Cost& c = kv.head_dim == 64 ? kCost64 : kCost128;
  // The candidate lists: their number and lengths.
  const int lists = levels + (fp.trim ? 1 : 0);
  auto list = [&](int i) { return i == 0 ? kv.seq >> levels : 2 * keep[levels + 1 - i]; };
  float cands = 0.f;
  for (int i = 0; i < lists; ++i) cands += (float)list(i);
  auto gathered = [&](int cs) {
    int rows = 0;
    for (int i = 0; i < lists; ++i) rows += (list(i) + cs - 1) / cs;
    return (float)rows;
  };
  const float U = (float)std::max(fp.U, 6);  // (fewer units leave the kernels per scale without CTAs)
  const float q32 = (float)q.seq / 32.f, near_tie = 1.03f;
  const float per_scale = c.scale * lists + U * cands * (c.cand + c.candq * q32) + c.sel * cands;
  auto filter_cost = [&](const F32Plan& p) {
    return c.f0 + (float)p.waves * (c.frow * gathered(p.cs) + c.fkey * cands);
  };
  if (n_g < 0) {
    fp.ok = filter_cost(fp) <= near_tie * per_scale;
    return fp;
  }
  const F32Plan ff = fit_f32(q, kv, levels, keep, -1, num_sms);
  const float one_filter = ff.ok ? filter_cost(ff) : per_scale;
  const float filter = ff.ok && (at_once(ff) || one_filter <= near_tie * per_scale) ? one_filter : per_scale;
  const float keys = (float)(keep[0] + n_g);
  const float split = c.a0 + U * keys * (c.att + c.attq * q32);
  const float one = c.s0 + (float)fp.waves * (c.srow * gathered(fp.cs) + c.skey * cands +
                                              c.scan * (float)((keep[0] + n_g + fp.cs - 1) / fp.cs));
  fp.ok = one <= near_tie * (filter + split);
  return fp;
}

cudaError_t launch_f32(const F32Plan& fp, const void* Q, const wf_tensor& qd, const void* K, const void* V,
                       const wf_tensor& kv, const void* Kg, const void* Vg, const wf_tensor* g, const void* coeffs,
                       int levels, const int32_t* keep, int32_t* idx, int32_t* level_sets, void* O,
                       const wf_tensor& od, cudaStream_t s) {
  F32Params p;
  memset(&p, 0, sizeof(p));
  p.Q = static_cast<const float*>(Q);
  p.qsb = qd.stride_b; p.qsh = qd.stride_h; p.qss = qd.stride_s;
  p.K = static_cast<const float*>(K);
  p.V = static_cast<const float*>(V);
  p.ksb = kv.stride_b; p.ksh = kv.stride_h; p.kss = kv.stride_s;
  p.Kg = static_cast<const float*>(Kg);
  p.Vg = static_cast<const float*>(Vg);
  if (g) { p.gsb = g->stride_b; p.gsh = g->stride_h; p.gss = g->stride_s; }
  p.coeffs = static_cast<const float*>(coeffs);
  p.rows_total = (int64_t)kv.seq - ((int64_t)kv.seq >> levels);
  p.O = static_cast<float*>(O);
  p.osb = od.stride_b; p.osh = od.stride_h; p.oss = od.stride_s;
  p.idx = idx;
  p.level_sets = level_sets;
  for (int l = 0; l <= levels; ++l) p.sets_stride += keep[l];
  p.q = qd.seq; p.n = kv.seq; p.ng = g ? g->seq : 0; p.H = kv.heads; p.L = levels;
  p.trim = fp.trim;
  p.attn = O != nullptr;
  p.trow = fp.trow; p.srow = fp.srow; p.bufw = fp.bufw;
  for (int l = 0; l <= levels; ++l) p.keep[l] = keep[l];
  p.scale = 1.0f / sqrtf((float)kv.head_dim);
  const F32Kernel k = f32_kernel(kv.head_dim, qd.seq);
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k), fp.smem);
  if (e != cudaSuccess) return e;
  return Launch(dim3((unsigned)(fp.U * fp.cs)), NTH, fp.smem, s, fp.cs)(k, p);
}

}  // namespace wf
