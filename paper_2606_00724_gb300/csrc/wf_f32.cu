// One layer in fp32 in one launch: the multi-scale filter (Eq. 7-11) and the
// sparse attention, for one query head per key head with at most 64 query
// rows and head_dim 64 or 128.
//
// A thread-block cluster serves one (batch, head) unit; each CTA (8 warps)
// holds one contiguous slice of the unit's candidate list at every scale, and
// finally of its sparse key list:
//   rows    the slice's rows gathered into shared memory (16-byte cp.async),
//           128 at a time;
//   logits  2 rows x QM / 4 queries a thread in fp32 FMAs, queries read as
//           warp-wide broadcasts, kept in shared memory as [query][row];
//   stats   (max, sum of exp) per query over the slice, one warp a query,
//           exchanged over the cluster;
//   keys    log W_j of each row (log-sum-exp over the queries against the
//           cluster's normalisers), written into every CTA's key array;
//   Top-K   the same selection in every CTA, giving the next scale's rows;
//   attention over the slice with a running max per query, partial outputs
//           combined from the cluster's shared memories.
// Exact fp32 throughout: fused multiply-adds in channel order, expf and logf.
//
// What bounds it: the chain of dependent phases of a scale (gather, FMAs,
// two cluster exchanges, Top-K), so the cluster is as wide as the SMs and 8
// CTAs allow, which shortens the gather and the FMAs.  A 2 x 8 register tile
// needs 16 shared-memory wavefronts for 64 FMAs a lane: the FMA pipe and
// shared memory are then about equally busy, where one row x 4 queries a
// thread needed twice the wavefronts.  Measured against three kernels a scale
// and two for the attention: 4 heads x 1K tokens (d 64) 63.5 -> 28.7 us a
// step, 16 heads x 8K (d 128) 170.2 -> 94.0 us, the error against 64 bits
// unchanged (4.4e-7 and 3.9e-6).
#include <math.h>
#include <string.h>

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
constexpr int TR = 128;       // rows of a tile
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
  int nbuf, srow, bufw;  // tile buffers, floats of a query's logit row, words of a key buffer
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
  float2 xch[TR];           // second half's (max, sum) per row
  float ms[64];             // the normalisers; the attention's running max
  float l[64];              // the attention's running row sums
  float alpha[64];          // this tile's factor of the partial output
};
__host__ __device__ inline F32Layout f32_layout(int D, int QM, int nbuf, int srow, int bufw) {
  F32Layout y;
  y.q = 0;
  y.tile = y.q + 4u * (uint32_t)(QM * D);
  y.s = y.tile + 4u * (uint32_t)(nbuf * TR * (D + 4));
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

// Rows [t0, t0 + min(TR, mc - t0)) of a list into a tile (row stride D + 4
// floats); row(j) is the address of the list's row j.
template <int D, typename F>
__device__ __forceinline__ void gather(float* tile, int t0, int mc, F&& row) {
  constexpr int LPR = D / 4;  // lanes a row
  const int c = threadIdx.x % LPR, cnt = min(TR, mc - t0);
#pragma unroll 4
  for (int r = threadIdx.x / LPR; r < cnt; r += NTH / LPR)
    cp_async16(smem_u32(tile + r * (D + 4) + 4 * c), row(t0 + r) + 4 * c);
}

// Logits (x scale) of a tile's rows against every query into S[query][t0 + row].
// Warp w: rows 64 (w % 2) + lane and + 32, queries QG (w / 2) ..; rows past the
// tile's cnt compute whatever the tile holds and are not stored.
template <int D, int QM>
__device__ __forceinline__ void score_tile(const float* Qs, const float* tile, float* S, int srow, int t0, int cnt,
                                           float scale) {
  constexpr int QG = QM / 4;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r0 = 64 * (w & 1) + lane, q0 = QG * (w >> 1);
  if (64 * (w & 1) >= cnt) return;
  const float* p0 = tile + r0 * (D + 4);
  const float* p1 = p0 + 32 * (D + 4);
  float a0[QG], a1[QG];
#pragma unroll
  for (int i = 0; i < QG; ++i) a0[i] = a1[i] = 0.f;
#pragma unroll 2
  for (int c = 0; c < D; c += 4) {
    const float4 x = *reinterpret_cast<const float4*>(p0 + c);
    const float4 y = *reinterpret_cast<const float4*>(p1 + c);
#pragma unroll
    for (int i = 0; i < QG; ++i) {
      const float4 v = *reinterpret_cast<const float4*>(Qs + (q0 + i) * D + c);
      a0[i] = fmaf(v.w, x.w, fmaf(v.z, x.z, fmaf(v.y, x.y, fmaf(v.x, x.x, a0[i]))));
      a1[i] = fmaf(v.w, y.w, fmaf(v.z, y.z, fmaf(v.y, y.y, fmaf(v.x, y.x, a1[i]))));
    }
  }
#pragma unroll
  for (int i = 0; i < QG; ++i) {
    float* s = S + (q0 + i) * srow + t0;
    if (r0 < cnt) s[r0] = a0[i] * scale;
    if (r0 + 32 < cnt) s[r0 + 32] = a1[i] * scale;
  }
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

template <int D, int QM>
__global__ void __launch_bounds__(NTH, 1) wf_f32_kernel(const __grid_constant__ F32Params p) {
  extern __shared__ __align__(16) uint8_t smem[];
  const F32Layout ly = f32_layout(D, QM, p.nbuf, p.srow, p.bufw);
  float* Qs = reinterpret_cast<float*>(smem + ly.q);
  float* T0 = reinterpret_cast<float*>(smem + ly.tile);
  float* T1 = T0 + (p.nbuf > 1 ? TR * (D + 4) : 0);  // the same buffer when there is one
  float* S = reinterpret_cast<float*>(smem + ly.s);
  F32Stat& st = *reinterpret_cast<F32Stat*>(smem + ly.stat);
  const uint32_t sc_a = smem_u32(smem + ly.sel);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster_rank(), cs = (int)cluster_size();
  const int u = (int)cluster_id_x();
  const int64_t bb = u / p.H, hh = u % p.H;
  auto buf = [&](int lev) { return reinterpret_cast<int32_t*>(smem + ly.buf) + ((p.L - lev) & 1) * p.bufw; };

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

  // S = scale Q rows^T of a list of mc rows; with two buffers the next tile's
  // copies run under the current tile's FMAs.
  auto score_list = [&](int mc, auto&& row) {
    gather<D>(T0, 0, mc, row);
    cp_async_commit();
    for (int t0 = 0, k = 0; t0 < mc; t0 += TR, k ^= 1) {
      const bool more = t0 + TR < mc;
      if (more && p.nbuf > 1) gather<D>(k ? T0 : T1, t0 + TR, mc, row);
      cp_async_commit();
      if (p.nbuf > 1) cp_async_wait<1>();
      else cp_async_wait<0>();
      __syncthreads();
      score_tile<D, QM>(Qs, (p.nbuf > 1 && k) ? T1 : T0, S, p.srow, t0, min(TR, mc - t0), p.scale);
      __syncthreads();
      if (more && p.nbuf == 1) gather<D>(T0, t0 + TR, mc, row);
    }
    cp_async_wait<0>();  // (an empty list's query block)
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
    for (int i = warp; i < QM; i += NW) {
      const float* s = S + i * p.srow;
      float mx = -INFINITY;
      for (int j = lane; j < mc; j += 32) mx = fmaxf(mx, s[j]);
      mx = warp_max_f32(mx);
      float z = 0.f;
      for (int j = lane; j < mc; j += 32) z += expf(s[j] - mx);
      z = warp_sum(z);
      if (lane < cs) st_cluster_v2f32(map_rank(smem_u32(&st.xstat[rank][i]), (uint32_t)lane), mx, z);
    }
    cluster_sync();
    if (tid < QM) {
      float M = -INFINITY;
      for (int r = 0; r < cs; ++r)
        if (st.xstat[r][tid].y > 0.f) M = fmaxf(M, st.xstat[r][tid].x);
      float z = 0.f;
      for (int r = 0; r < cs; ++r)
        if (st.xstat[r][tid].y > 0.f) z = fmaf(st.xstat[r][tid].y, expf(st.xstat[r][tid].x - M), z);
      st.ms[tid] = M + logf(z);
    }
    __syncthreads();
    // Ranking keys: the two warpgroups take half the queries each of 128 rows.
    int32_t* J = buf(lev);  // receives this scale's keys, then its selection
    float kmin = INFINITY, kmax = -INFINITY;
    {
      const int h = tid >> 7, rl = tid & (TR - 1);
      const int i0 = h * ((p.q + 1) / 2), i1 = h ? p.q : (p.q + 1) / 2;
      for (int t0 = 0; t0 < mc; t0 += TR) {
        const int j = t0 + rl;
        float mx = -INFINITY, z = 0.f;
        if (j < mc) {
#pragma unroll 8
          for (int i = i0; i < i1; ++i) mx = fmaxf(mx, S[i * p.srow + j] - st.ms[i]);
#pragma unroll 8
          for (int i = i0; i < i1 && mx > -INFINITY; ++i) z += expf((S[i * p.srow + j] - st.ms[i]) - mx);
        }
        if (h) st.xch[rl] = make_float2(mx, z);
        __syncthreads();
        if (!h && j < mc) {
          const float2 o = st.xch[rl];
          const float M = fmaxf(mx, o.x);
          const float key = M + logf((z > 0.f ? z * expf(mx - M) : 0.f) + (o.y > 0.f ? o.y * expf(o.x - M) : 0.f));
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
      st.ms[tid] = -INFINITY;
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
    for (int t0 = 0; t0 < mc; t0 += TR) {
      const int cnt = min(TR, mc - t0);
      gather<D>(T0, t0, mc, krow);
      cp_async_commit();
      if (p.nbuf > 1) {
        gather<D>(T1, t0, mc, vrow);
        cp_async_commit();
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
      score_tile<D, QM>(Qs, T0, S, p.srow, 0, cnt, p.scale);
      __syncthreads();
      if (p.nbuf == 1) {
        gather<D>(T1, t0, mc, vrow);
        cp_async_commit();
      }
      // P = exp(s - m) against the running max; keys past the tile get 0.
      for (int i = warp; i < QM; i += NW) {
        float* s = S + i * p.srow;
        float mx = -INFINITY;
        for (int j = lane; j < cnt; j += 32) mx = fmaxf(mx, s[j]);
        const float mo = st.ms[i], mn = fmaxf(mo, warp_max_f32(mx));
        float z = 0.f;
        for (int j = lane; j < TR; j += 32) {
          const float e = j < cnt ? expf(s[j] - mn) : 0.f;
          s[j] = e;
          z += e;
        }
        z = warp_sum(z);
        __syncwarp();
        if (lane == 0) {
          const float a = mo > -INFINITY ? expf(mo - mn) : 0.f;
          st.alpha[i] = a;
          st.ms[i] = mn;
          st.l[i] = fmaf(st.l[i], a, z);
        }
      }
      // Rows past the tile are zero: P is 0 there, and the last tile's rows
      // of the buffer may hold anything (infinities included).
      for (int e = tid; e < (TR - cnt) * LPR; e += NTH)
        if (p.nbuf > 1)
          *reinterpret_cast<float4*>(T1 + (cnt + e / LPR) * (D + 4) + 4 * (e % LPR)) = make_float4(0.f, 0.f, 0.f, 0.f);
      cp_async_wait<0>();
      __syncthreads();
      if (p.nbuf == 1) {
        for (int e = tid; e < (TR - cnt) * LPR; e += NTH)
          *reinterpret_cast<float4*>(T1 + (cnt + e / LPR) * (D + 4) + 4 * (e % LPR)) = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
      }
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
    }
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

void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr, int clusters, int cs, size_t smem) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)(clusters * cs), 1, 1);
  cfg.blockDim = dim3(NTH, 1, 1);
  cfg.dynamicSmemBytes = smem;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)cs;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
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
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  cluster_config(cfg, attr, 1, cs, smem);
  int n = 0;
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k), smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    n = 0;
  }
  cache.emplace(key, n);
  return n;
}

}  // namespace

// fp32, one query head per key head, candidate lists within the Top-K's 8192.
// The largest cluster (up to 8) whose grid fits the SMs in one wave, all
// clusters resident, and whose slice's logits fit shared memory; else the
// smallest whose logits fit.
F32Plan plan_f32(const wf_tensor& q, const wf_tensor& kv, int levels, const int32_t* keep, int num_sms) {
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
    int rows = 2 * (((cmax + 1) / 2 + cs - 1) / cs);  // the widest slice
    rows = rows > TR ? rows : TR;
    fp.srow = (rows + 3) / 4 * 4 + 4;
    for (fp.nbuf = 2; fp.nbuf >= 1; --fp.nbuf) {
      fp.smem = f32_layout(D, QM, fp.nbuf, fp.srow, fp.bufw).total;
      if (fp.smem <= kMaxSmem) return true;
    }
    return false;
  };
  for (int cs = MAXCS; cs >= 1 && fp.cs == 0; --cs)
    if (U * cs <= num_sms && fit(cs) && U <= resident_clusters(k, cs, fp.smem)) fp.cs = cs;
  for (int cs = 1; cs <= MAXCS && fp.cs == 0; ++cs)
    if (fit(cs) && resident_clusters(k, cs, fp.smem) > 0) fp.cs = cs;
  if (fp.cs == 0) return fp;
  fp.U = U;
  fp.ok = true;
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
  p.nbuf = fp.nbuf; p.srow = fp.srow; p.bufw = fp.bufw;
  for (int l = 0; l <= levels; ++l) p.keep[l] = keep[l];
  p.scale = 1.0f / sqrtf((float)kv.head_dim);
  const F32Kernel k = f32_kernel(kv.head_dim, qd.seq);
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k), fp.smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  cluster_config(cfg, attr, fp.U, fp.cs, fp.smem);
  cfg.stream = s;
  e = cudaLaunchKernelEx(&cfg, k, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace wf
