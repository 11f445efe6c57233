// Fused WaveFilter step (Algorithm 1 body): multi-scale skim/scan filtering
// (Eq. 7-11) and the final sparse attention, in one kernel.
//
// A thread-block cluster of CS CTAs serves P (1 or 2) (batch, head) units;
// every CTA holds one contiguous slice of each unit's candidate list at every
// scale (and finally of its sparse key list).  The warps of a CTA specialise:
//   * producer warps gather candidate rows (pyramid level b, raw keys for the
//     level-0 trim, or K/V rows of mu^0 and the generation rows) with 16-byte
//     cp.async copies into 128-byte-swizzled tiles of 128 rows, through a ring
//     of stages; each copy's completion arrives on the stage's mbarrier;
//   * one MMA thread issues tcgen05.mma (bf16 in, fp32 out) per landed tile,
//     writing S^T = rows . Q^T into the unit's TMEM region (32 columns per
//     tile), and in the attention O^T += V_s^T P^T;
//   * four compute warps per unit (one per TMEM lane quarter, one candidate
//     row per thread; both warpgroups, taking alternate tiles, when a
//     cluster serves one unit with long candidate lists) read the logits
//     back (tcgen05.ld), form the per-query max and
//     sum of exp of the slice, exchange them with the cluster (st.async into
//     every CTA, completion counted on its mbarrier), compute the ranking key
//     log2 W_j (Eq. 8) of each candidate, all-gather the keys the same way,
//     and run the same deterministic Top-K (Eq. 9, lowest position first on
//     ties) in every CTA, giving J_b and hence the next scale's candidates
//     {2j, 2j+1} (Eq. 10).
// The units of a cluster alternate: while the compute warps score, exchange
// and select one unit, the producers already stream the other unit's rows, so
// copies overlap the latency-bound phases.  In the attention the compute warps
// turn S into P = 2^(s - m) (bf16) for the MMA thread, and each CTA's partial
// (m, l, O^T) is reduce-scattered over head-dimension slices: CTA r combines
// rows d of O for its slice and writes them.
//
// A launch may also run part of the chain (a range of scales, the previous
// selection handed in, the last one handed out, the attention optional): the
// literal-basis path runs one launch per scale.  Launches are programmatic
// dependents of the kernel before them (every thread waits for that grid
// before its first global access).
//
// Every wait is bounded (~1 s): on timeout the CTA records a status word,
// stops issuing MMAs and skips the remaining waits, so every thread reaches
// the final cluster barrier.
#include <float.h>
#include <math.h>
#include <string.h>

#include <map>
#include <mutex>
#include <tuple>

#include "wf_internal.cuh"
#include "wf_sm100.cuh"
#include "wf_topk.cuh"

// The file is compiled once per head_dim (wf_fused_d64.cu defines 64 and
// includes it), and for head_dim 128 once more for the filter and the attention
// as calls of their own (wf_fused_stages.cu defines WF_STAGE_CALLS and includes
// it); the entry points live in a namespace of each.
#ifndef WF_HEAD_DIM
#define WF_HEAD_DIM 128
#endif
#ifndef WF_STAGE_CALLS
#define WF_STAGE_CALLS 0
#endif
#if WF_STAGE_CALLS
#define WF_HD stage128
#elif WF_HEAD_DIM == 128
#define WF_HD hd128
#else
#define WF_HD hd64
#endif

namespace wf {
namespace WF_HD {
namespace {

using namespace sm100;
using namespace topk;

constexpr int D = WF_HEAD_DIM;             // head_dim
static_assert(D == 64 || D == 128, "a row is one or two 128-byte swizzle rows");
constexpr int TM = 128;                    // rows per MMA tile (M)
constexpr int NQ = 32;                     // query rows per MMA (N), zero padded
constexpr int MAXP = 2;                    // units per cluster
// A unit has NCW = 4 compute warps (one per TMEM lane quarter), NCT threads.
constexpr int MMA_WARP = MAXP * NCW;       // TMEM allocation and MMA issue (lane 0)
constexpr int NPW = 3;                     // producer warps
constexpr int NPT = 32 * NPW;              // producer threads
constexpr int P0 = 32 * (MMA_WARP + 1);    // first producer thread
constexpr int NT = 32 * (MMA_WARP + 1 + NPW);  // threads per CTA
constexpr int MAXCS = 8;                   // CTAs per cluster
constexpr int HALF_BYTES = TM * 128;       // one 64-column half of a tile, 128-byte rows
constexpr int HALVES = D / 64;               // 128-byte halves of a row
constexpr int TILE_BYTES = HALVES * HALF_BYTES;
// Ring stages: as many bytes for either head_dim.
constexpr int MAXS = 4 * 128 / D;          // most stages of an instance
constexpr int QGRP = (D / 8) * 128;        // bytes per 8-row group of a query tile (core matrices)
constexpr int Q_BYTES = NQ * D * 2;
// The attention's P = 2^(s - m) is the bf16 operand of the PV product.  For
// head_dim 128 P is rounded to bf16.  For head_dim 64 P keeps its 24 bits, as
// three bf16 terms (each the rounding of what the terms before it leave) that
// multiply V one after the other into the same fp32 accumulator.  An attention
// of its own at head_dim 128 keeps 16 bits, as two terms (wf_fused_stages.cu).
constexpr int PTERMS = D == 64 ? 3 : 1;
constexpr bool kLowTerm = WF_STAGE_CALLS != 0;
// Whether a launch may be the attention alone.  Its code is left out of the
// other instance, whose first pass fetches all of it from memory (64 units x
// 32K with L2 flushed 79.3 -> 78.2 us).
constexpr bool kAlone = D == 64 || WF_STAGE_CALLS != 0;
constexpr int PT_BYTES = NQ * TM * 2;      // one term of one P tile
constexpr int P_BYTES = PTERMS * PT_BYTES;
constexpr int MAXCS_PAD_BYTES = 8 * NQ * 4;  // the ragged head-dim slices of a cluster of up to 8 CTAs
// A unit's P double buffer; also its Top-K scratch and its combine buffer
// (the partial O rows of this CTA's head-dim slice from every cluster CTA:
// at most (D + cs) rows of 32 fp32 when cs does not divide D).
constexpr int UNIT_P_BYTES = 2 * P_BYTES + MAXCS_PAD_BYTES;
constexpr float kLog2e = 1.4426950408889634f;
// Named barriers 1 and 2 (kCsyncId) are the compute warps' of unit 0 and 1.
constexpr uint32_t kSetupSyncId = 3;       // named barrier 3: the set-up threads (all but the producers)

constexpr uint32_t kIdescScore = idesc_bf16(TM, NQ, 0, 0);  // A = rows (K-major), B = Q (K-major)
// A = V^T (MN-major), B = P^T (MN-major).  M is 128 for head_dim 64 too: the
// upper 64 accumulator rows are products of whatever follows the value tile
// in shared memory (always inside the CTA's allocation) and nothing reads them.
constexpr uint32_t kIdescPV = idesc_bf16(128, NQ, 1, 1);

constexpr int MAXT = 16;  // TMEM tiles of one unit's region (512 columns / 32)

// The Top-K scratch lives in the unit's P buffers, which nothing uses before
// the attention.
static_assert((sizeof(SelScratch) + 15) / 16 * 16 <= UNIT_P_BYTES, "Top-K scratch must fit the P buffers");

struct UnitState {
  float2 xstat[MAXCS][NQ];  // (stabiliser, sum of exp) of every cluster CTA's slice
  float2 cstat[MAXCS][NQ];  // attention (max, row sum) of every CTA (d-slice owner side)
  // Per-warp slots (warp w of the unit at slot w; a WIDE unit's warps 4-7 use
  // the second unit's slots, which nothing else uses then).
  float2 kmm[MAXCS][NCW];   // (min, max) of the ranking keys of every cluster warp
  float2 wstat[NCW][NQ];    // (stabiliser, sum of exp) of each compute warp's rows
  float cw[NCW][NQ];        // softmax normaliser c_i, one copy per compute warp
  float fw[NCW][NQ];        // 2^(stabiliser - c_i) of each warp (keys from stored exponentials)
  float mloc[NQ], lacc[NQ];
  float alpha[NQ];          // attention: factor 2^(m_old - m_new) of a raised stabiliser
  float red[NCW][32];
};

constexpr int MAXREG = 8;  // grouped filter: most TMEM regions of pass 2

struct Misc {
  unsigned long long full[MAXS], empty[MAXS];
  unsigned long long mdone[MAXP], jready[MAXP], xbar[MAXP], kbar[MAXP];
  unsigned long long tdone[MAXP][MAXT];  // scale tile t of a unit scored (one phase per scale)
  unsigned long long pfull[MAXP][2], pempty[MAXP][2], cbar[MAXP], cready[MAXP];
  UnitState us[MAXP];
  unsigned long long qfull;     // the query blocks have landed (the producers' first copies)
  // Grouped filter: pass 1's TMEM buffers and pass 2's regions ready / read.
  unsigned long long p1done[2], p1free[2], rdone[MAXREG], rfree[MAXREG];
  unsigned long long stallbar;  // completed by nothing (the test-only stalled first wait)
  unsigned long long drainbar;  // the MMA thread's final commit
  long long wait_limit;         // bound of the waits that can give up (cycles)
  int abort;
  uint32_t tmem_base;
};

// The UnitState holding the per-warp slots of unit warp w (index w % 4).
template <bool WIDE>
__device__ __forceinline__ UnitState& wslots(Misc& ms, int pp, int w) {
  return WIDE ? ms.us[w >> 2] : ms.us[pp];
}

// Shared-memory layout (byte offsets; the stage ring starts at 0, 1024-byte
// aligned for the 128-byte swizzle).
struct SmemLayout {
  uint32_t q, p, misc, buf, bufw, lo, total;
};
__host__ __device__ inline SmemLayout smem_layout(int stages, int P, int cmax, int kmax, bool alone) {
  SmemLayout l;
  l.q = (uint32_t)stages * TILE_BYTES;
  l.p = l.q + (uint32_t)P * Q_BYTES;
  l.misc = l.p + (uint32_t)P * UNIT_P_BYTES;
  // Two buffers per unit alternate by scale: one receives the scale's keys and
  // then its selection J_b, the other still holds J_{b+1}.
  l.buf = (l.misc + (uint32_t)sizeof(Misc) + 127u) / 128u * 128u;
  l.bufw = (uint32_t)((max(cmax, kmax) + 3) / 4 * 4);
  l.lo = l.buf + (uint32_t)P * 2u * 4u * l.bufw;  // the second terms' double buffer
  l.total = l.lo + (kLowTerm && alone ? (uint32_t)P * 2u * PT_BYTES : 0u);
  return l;
}

struct FusedParams {
  const bf16* Q;
  int64_t qsb, qsh, qss;
  const bf16* K;
  const bf16* V;
  int64_t ksb, ksh, kss;
  const bf16* Kg;
  const bf16* Vg;
  int64_t gsb, gsh, gss;
  const bf16* coeffs;
  int64_t rows_total;
  bf16* O;
  int64_t osb, osh, oss;
  int32_t* idx;
  int32_t* level_sets;
  int64_t sets_stride;
  int* status;
  int q, n, ng, U, H, L, trim, P, cmax, kmax;
  uint32_t tmem_cols, ucols;  // TMEM allocation; columns per unit region
  uint32_t ecol;              // column of the stored exponentials in a unit region (0: none)
  long long wait_limit;       // bound of the waits that can give up (cycles)
  int stall;                  // test-only: the MMA thread's first wait never completes
  int G, nch;                 // grouped filter: query heads per key head, 32-row chunks of the stacked block
  int32_t keep[12];
  float scale_log2;           // log2(e) / sqrt(d)
  // The scales this launch runs, lev_top down to lev_bot (the whole chain, L
  // down to 1 or 0, for the pyramid step).  A launch that starts below L reads
  // the previous selection J_{lev_top+1} as the children list jin (candidate
  // block indices of scale lev_top, 2 J[i] and 2 J[i] + 1); one that ends
  // above the final scale writes the children of its last selection to jout.
  int lev_top, lev_bot, final_sel, attn;
  const int32_t* jin;
  int32_t* jout;
  int64_t jstride;  // entries per unit of jin and jout
  // Attention alone (no scale; L = 0, trim): the caller's token list
  // [units][keep[0]], any order, clamped to the prompt; else null.
  const int32_t* sel;
  // Literal-basis rows: scale lev_top's candidate rows in candidate order
  // (row j of unit u at lrows + u lrows_unit + j D); null for the pyramid.
  const bf16* lrows;
  int64_t lrows_unit;
};

// Per-CTA constants and shared-memory addresses.
struct Ctx {
  uint8_t* smem;
  Misc* ms;
  SmemLayout ly;
  uint32_t rank, cs, tmem;
  int np, u0, lev_top, lev_end, stages;
};

// The warpgroup of a compute thread within its unit (0 unless WIDE), the
// first tile it takes and its tile stride.
template <bool WIDE>
__device__ __forceinline__ int unit_wg() {
  return WIDE ? (int)((threadIdx.x >> 7) & 1) : 0;
}
template <bool WIDE>
__host__ __device__ constexpr int tile_step() {
  return WIDE ? 2 : 1;
}

__device__ __forceinline__ bool aborted(const Misc& ms) { return abort_set(smem_u32(&ms.abort)); }

__device__ __forceinline__ void set_abort(Misc& ms, int* status) {
  ms.abort = 1;
  atomicExch(status, 1);
}

__device__ __noinline__ void wait_or_abort(uint32_t bar, uint32_t parity, Misc& ms, int* status) {
  if (!aborted(ms) && !mbar_wait_bounded(bar, parity, ms.wait_limit, smem_u32(&ms.abort))) set_abort(ms, status);
}

// Wait for a phase completed by other CTAs of the cluster (acquire, cluster scope).
__device__ __noinline__ void wait_cluster_or_abort(uint32_t bar, uint32_t parity, Misc& ms, int* status) {
  if (!aborted(ms) && !mbar_wait_cluster_bounded(bar, parity, ms.wait_limit, smem_u32(&ms.abort)))
    set_abort(ms, status);
}

__device__ __forceinline__ uint32_t bar_addr(const unsigned long long& b) { return smem_u32(&b); }

// Candidate count of scale `lev`: the top coefficients, or the children of
// the coefficients kept one scale up (Eq. 10).
__device__ __forceinline__ int m_total(const FusedParams& p, int lev) {
  return lev == p.L ? (p.n >> p.L) : 2 * p.keep[lev + 1];
}

// This CTA's slice [g0, g0 + mc) of a candidate list of m (sibling pairs kept
// together).
__device__ __forceinline__ void scale_slice(int m, uint32_t rank, uint32_t cs, int& g0, int& mc) {
  const int pairs = (m + 1) >> 1;
  // 32-bit arithmetic: rank <= 8 and pairs <= 2^16 (a 64-bit division is a
  // called routine on the path between two scales).
  g0 = min(m, 2 * (int)(rank * (uint32_t)pairs / cs));
  const int g1 = min(m, 2 * (int)((rank + 1u) * (uint32_t)pairs / cs));
  mc = g1 - g0;
}

// This CTA's slice of the sparse key list of `total` rows.
__device__ __forceinline__ void attn_slice(int total, uint32_t rank, uint32_t cs, int& a0, int& mc) {
  a0 = (int)(rank * (uint32_t)total / cs);
  mc = (int)((rank + 1u) * (uint32_t)total / cs) - a0;
}

__device__ __forceinline__ int tiles_of(int mc) { return (mc + TM - 1) / TM; }

// Head-dim slice [dlo(r), dlo(r + 1)) whose output rows CTA r combines.
__device__ __forceinline__ int dlo(int r, int cs) { return r * D / cs; }

// Where the rows of a candidate or key list come from.
//  kind 0: position j -> row j (top scale);
//  kind 1: position j -> row 2 J[j/2] + j%2 (children of the kept coefficients);
//  kind 2: sparse key list, positions < kk -> token 2 J[j/2] + j%2, then
//          generation rows;
//  kind 3: the same with a trimmed level 0, positions < kk -> token J[j].
struct RowSrc {
  const bf16* base;
  int64_t stride;
  const bf16* gbase;
  int64_t gstride;
  uint32_t J;  // shared address of the selection the rows derive from
  int kind, g0, mc, kk;
  int rows;  // rows of the source: indices from a selection are clamped below it
};

// Row r of a slice.  Kinds 0 and 1: the row index in the source; kinds 2
// and 3: the row's address (a key row or a generation row).  Indices read
// from a selection are valid rows; the clamp keeps every address inside the
// source even when a wait gave up and the selection was made from stale data
// (the status word then reports the failure).
template <int KIND>
__device__ __forceinline__ uint32_t row_index(const RowSrc& s, int r) {
  const int pos = s.g0 + (r < s.mc ? r : 0);  // rows past the slice repeat its first row
  const uint32_t row = KIND == 0 ? (uint32_t)pos
                                 : 2u * lds_u32(s.J + 4u * (uint32_t)(pos >> 1)) + (uint32_t)(pos & 1);
  return min(row, (uint32_t)s.rows - 1u);
}
template <int KIND>
__device__ __forceinline__ const bf16* row_ptr(const RowSrc& s, int r) {
  const int pos = s.g0 + (r < s.mc ? r : 0);
  const int pk = min(pos, s.kk - 1);
  const uint32_t tok0 = KIND == 3 ? lds_u32(s.J + 4u * (uint32_t)pk)
                                  : 2u * lds_u32(s.J + 4u * (uint32_t)(pk >> 1)) + (uint32_t)(pk & 1);
  const bf16* key = s.base + (int64_t)min(tok0, (uint32_t)s.rows - 1u) * s.stride;
  const bf16* gen = s.gbase + (int64_t)(pos - s.kk) * s.gstride;
  return pos < s.kk ? key : gen;
}

// Buffer k (0, 1) of unit pp; scale lev's keys and selection use buffer
// (L - lev) % 2.
__device__ __forceinline__ int32_t* unit_buf(const Ctx& c, int pp, int k) {
  return reinterpret_cast<int32_t*>(c.smem + c.ly.buf) + (pp * 2 + k) * (int)c.ly.bufw;
}
// Buffer holding the selection J made at scale lev.
__device__ __forceinline__ int32_t* unit_J(const Ctx& c, const FusedParams& p, int pp, int lev) {
  return unit_buf(c, pp, (p.L - lev) & 1);
}

// Rows of unit u at scale lev (pyramid level lev, or the raw keys at level 0).
__device__ __forceinline__ RowSrc scale_src(const Ctx& c, const FusedParams& p, int pp, int lev, int g0, int mc) {
  const int u = c.u0 + pp;
  const bool lit = p.lrows && lev >= 1 && lev == c.lev_top;  // literal-basis rows of this launch's scale
  RowSrc s;
  if (lit) {
    s.base = p.lrows + (int64_t)u * p.lrows_unit;  // row j: candidate j's transform (kind 0 below)
    s.stride = D;
  } else if (lev >= 1) {
    s.base = p.coeffs + ((int64_t)u * p.rows_total + ((int64_t)p.n - ((int64_t)p.n >> (lev - 1)))) * D;
    s.stride = D;
  } else {
    s.base = p.K + (int64_t)(u / p.H) * p.ksb + (int64_t)(u % p.H) * p.ksh;
    s.stride = p.kss;
  }
  s.gbase = nullptr;
  s.gstride = 0;
  s.J = smem_u32(unit_J(c, p, pp, lev + 1));  // the children of the selection one scale up (unused at the top)
  s.kind = (lev == p.L || lit) ? 0 : 1;
  s.g0 = g0;
  s.mc = mc;
  s.kk = 0;
  s.rows = lit ? m_total(p, lev) : (lev >= 1 ? (int)(p.n >> lev) : (int)p.n);
  return s;
}

// Sparse key list [K[mu^0]; Kg] (or the V rows) of unit pp.
__device__ __forceinline__ RowSrc attn_src(const Ctx& c, const FusedParams& p, int pp, bool values, int a0,
                                           int mc) {
  const int u = c.u0 + pp;
  const int64_t b = u / p.H, h = u % p.H;
  RowSrc s;
  s.base = (values ? p.V : p.K) + b * p.ksb + h * p.ksh;
  s.stride = p.kss;
  s.gbase = (values ? p.Vg : p.Kg) + b * p.gsb + h * p.gsh;
  s.gstride = p.gss;
  s.J = smem_u32(unit_J(c, p, pp, p.trim ? 0 : 1));  // mu^0 from the last selection
  s.kind = p.trim ? 3 : 2;
  s.g0 = a0;
  s.mc = mc;
  s.kk = p.keep[0];
  s.rows = (int)p.n;
  return s;
}

// ---------------------------------------------------------------------------
// Producer warps.
// ---------------------------------------------------------------------------

// This producer thread's share of one 128-row tile: 16-byte chunk c = pt % LPR
// of rows r0 + RSTEP j (r0 = pt / LPR, j < RROWS), written in the
// 128-byte-swizzled K-major layout (row r, chunk c at half c/8, byte
// r*128 + ((c%8) ^ (r%8))*16).  The LPR lanes of a row's chunks copy the same
// rows, so each lane forms one row's index or address per LPR rows and they
// share them by shuffles.  The swizzle term of a thread's rows repeats every
// 4 rows (RSTEP j mod 8 takes at most 4 values), so each destination is one
// add.
constexpr int LPR = D / 8;                       // lanes (16-byte chunks) a row
constexpr int RSTEP = NPT / LPR;
constexpr int RROWS = (TM + RSTEP - 1) / RSTEP;  // most rows of one thread
static_assert(RSTEP * LPR <= TM && LPR <= RROWS, "a lane's first resolved row needs no clamp");
static_assert(RSTEP % 2 == 0 && RROWS <= 2 * LPR, "4 swizzle terms and two resolved rows a lane cover a thread's rows");
template <int KIND>
__device__ __forceinline__ void load_share(uint32_t st, int t, const RowSrc& src, int pt) {
  const int c = pt & (LPR - 1), r0 = (int)((unsigned)pt / LPR), grp = pt & (32 - LPR);
  const uint32_t dbase = st + ((c >> 3) << 14) + (uint32_t)r0 * 128u;
  uint32_t xr[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) xr[m] = (uint32_t)((c ^ (r0 + RSTEP * m)) & 7) << 4;
  // Rows j = c and j = LPR + c of these lanes (the second clamped into the tile).
  const int ra = t * TM + r0 + RSTEP * c;
  const int rb = t * TM + min(r0 + RSTEP * min(LPR + c, RROWS - 1), TM - 1);
  if (KIND <= 1) {
    const char* cb = reinterpret_cast<const char*>(src.base) + c * 16;
    const uint32_t sb = (uint32_t)src.stride * 2u;  // row stride in bytes
    const uint32_t ia = row_index<KIND>(src, ra), ib = row_index<KIND>(src, rb);
#pragma unroll
    for (int j = 0; j < RROWS; ++j) {
      const uint32_t idx = __shfl_sync(0xffffffffu, j < LPR ? ia : ib, grp | (j & (LPR - 1)));
      if (RSTEP * j + RSTEP - 1 < TM || r0 + RSTEP * j < TM)
        cp_async16(dbase + 128u * RSTEP * j + xr[j & 3], cb + (size_t)idx * sb);
    }
  } else {
    const unsigned long long pa = reinterpret_cast<unsigned long long>(row_ptr<KIND>(src, ra));
    const unsigned long long pb = reinterpret_cast<unsigned long long>(row_ptr<KIND>(src, rb));
#pragma unroll
    for (int j = 0; j < RROWS; ++j) {
      const unsigned long long ak = __shfl_sync(0xffffffffu, j < LPR ? pa : pb, grp | (j & (LPR - 1)));
      if (RSTEP * j + RSTEP - 1 < TM || r0 + RSTEP * j < TM)
        cp_async16(dbase + 128u * RSTEP * j + xr[j & 3], reinterpret_cast<const bf16*>(ak) + c * 8);
    }
  }
}

// Tiles t0 .. t0 + ntl - 1 of the source into ring slots it0, it0 + 1, ...
template <int S>
__device__ __noinline__ void produce(Misc& ms, int* status, uint32_t ring, int it0, int t0, int ntl, const RowSrc src,
                                     int pt) {
#pragma unroll 1
  for (int t = t0; t < t0 + ntl; ++t) {
    const int it = it0 + t - t0, s = it % S, n = it / S;
    if (n > 0) wait_or_abort(bar_addr(ms.empty[s]), (uint32_t)(n - 1) & 1u, ms, status);
    if (!aborted(ms)) {
      const uint32_t st = ring + s * TILE_BYTES;
      switch (src.kind) {
        case 0: load_share<0>(st, t, src, pt); break;
        case 1: load_share<1>(st, t, src, pt); break;
        case 2: load_share<2>(st, t, src, pt); break;
        default: load_share<3>(st, t, src, pt); break;
      }
    }
    cp_async_arrive_noinc(bar_addr(ms.full[s]));
  }
}

template <int S>
__device__ void producer_role(const Ctx& c, const FusedParams& p) {
  Misc& ms = *c.ms;
  const int pt = threadIdx.x - P0;
  // The query blocks go first, ahead of every row copy: they are the MMA
  // thread's first operands, and requests queued behind the whole grid's
  // first burst of rows would reach it only after that burst.  K-major core
  // matrices; rows >= q are zero-filled (no bytes read).
  for (int pp = 0; pp < c.np; ++pp) {
    const int u = c.u0 + pp;
    const bf16* qb = p.Q + (int64_t)(u / p.H) * p.qsb + (int64_t)(u % p.H) * p.qsh;
    const uint32_t sq = smem_u32(c.smem + c.ly.q + pp * Q_BYTES);
    for (int e = pt; e < NQ * (D / 8); e += NPT) {
      const int rr = e & 7, ch = (e >> 3) & (D / 8 - 1), g = e / D;
      const int i = g * 8 + rr;
      cp_async16_zfill(sq + (uint32_t)(g * QGRP + ch * 128 + rr * 16), qb + (int64_t)min(i, p.q - 1) * p.qss + ch * 8,
                       i < p.q);
    }
  }
  cp_async_arrive_noinc(bar_addr(ms.qfull));
  int it = 0;
  for (int lev = c.lev_top; lev >= c.lev_end; --lev) {
    for (int pp = 0; pp < c.np; ++pp) {
      // The rows of a lower scale are the children of the unit's last selection.
      if (lev != c.lev_top) wait_or_abort(bar_addr(ms.jready[pp]), (uint32_t)(c.lev_top - lev - 1) & 1u, ms, p.status);
      int g0, mc;
      scale_slice(m_total(p, lev), c.rank, c.cs, g0, mc);
      const int ntl = tiles_of(mc);
      produce<S>(ms, p.status, smem_u32(c.smem), it, 0, ntl, scale_src(c, p, pp, lev, g0, mc), pt);
      it += ntl;
    }
  }
  const int nsel = kAlone && p.sel ? 1 : c.lev_top - c.lev_end + 1;  // selections made (or handed in)
  for (int pp = 0; pp < c.np && p.attn; ++pp) {
    wait_or_abort(bar_addr(ms.jready[pp]), (uint32_t)(nsel - 1) & 1u, ms, p.status);
    int a0, mc;
    attn_slice(p.keep[0] + p.ng, c.rank, c.cs, a0, mc);
    const int ntl = tiles_of(mc);
    // The key tiles, then the value tiles.  A key tile's slot frees as soon
    // as its S product is done and a value tile's once its PV product is,
    // whose P the compute warps form from each S tile as it lands, so the
    // value stream follows the key stream without waiting for all of S.
    produce<S>(ms, p.status, smem_u32(c.smem), it, 0, ntl, attn_src(c, p, pp, false, a0, mc), pt);
    it += ntl;
    produce<S>(ms, p.status, smem_u32(c.smem), it, 0, ntl, attn_src(c, p, pp, true, a0, mc), pt);
    it += ntl;
  }
  // Copies still in flight (only after a wait gave up) land before the CTA
  // can leave.
  cp_async_wait_all();
}

// ---------------------------------------------------------------------------
// MMA thread.
// ---------------------------------------------------------------------------

// S^T = rows . Q^T of the landed tile in ring slot `it` into TMEM columns
// [dcol, dcol + 32); its completion frees the slot and completes `tbar`, so the
// compute warps start on the tile at once.
template <int S>
__device__ __forceinline__ void mma_score_tile(const Ctx& c, const FusedParams& p, int it, uint32_t dcol, uint32_t sq,
                                               uint32_t tbar) {
  Misc& ms = *c.ms;
  const int s = it % S, n = it / S;
  wait_or_abort(bar_addr(ms.full[s]), (uint32_t)n & 1u, ms, p.status);
  fence_proxy_async();
  if (!aborted(ms)) {
    tc_fence_after();
    const uint32_t st = smem_u32(c.smem) + s * TILE_BYTES;
#pragma unroll
    for (int h = 0; h < HALVES; ++h)
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        mma_bf16(dcol, smem_desc_sw128(st + h * HALF_BYTES + kk * 32, 16, 1024),
                 smem_desc(sq + (4 * h + kk) * 256, 128, QGRP), kIdescScore, (h | kk) != 0);
  }
  mma_commit(bar_addr(ms.empty[s]));
  mma_commit(tbar);
}

// O^T += V_t^T P_t^T for the value tile in ring slot `it` and unit pp's P tile
// t (the P double buffer t % 2, filled by the compute warps).
template <int S>
__device__ __forceinline__ void mma_pv_tile(const Ctx& c, const FusedParams& p, int pp, int it, int t, uint32_t ocol) {
  Misc& ms = *c.ms;
  const uint32_t pa = smem_u32(c.smem + c.ly.p + pp * UNIT_P_BYTES);
  const int s = it % S, n = it / S;
  const uint32_t pb = (uint32_t)t & 1u, pn = (uint32_t)t >> 1;
  wait_or_abort(bar_addr(ms.full[s]), (uint32_t)n & 1u, ms, p.status);
  wait_or_abort(bar_addr(ms.pfull[pp][pb]), pn & 1u, ms, p.status);
  fence_proxy_async();
  if (!aborted(ms)) {
    tc_fence_after();
    const uint32_t st = smem_u32(c.smem) + s * TILE_BYTES;
#pragma unroll
    for (int kq = 0; kq < TM / 16; ++kq)
#pragma unroll
      for (int e = 0; e < PTERMS; ++e)
        mma_bf16(ocol, smem_desc_sw128(st + kq * 2048, HALF_BYTES, 1024),
                 smem_desc(pa + pb * P_BYTES + e * PT_BYTES + kq * 1024, 512, 128), kIdescPV,
                 (t > 0 || kq > 0 || e > 0) ? 1u : 0u);
    if (kLowTerm && p.sel) {
      const uint32_t lo = smem_u32(c.smem + c.ly.lo) + (2u * pp + pb) * PT_BYTES;
#pragma unroll
      for (int kq = 0; kq < TM / 16; ++kq)
        mma_bf16(ocol, smem_desc_sw128(st + kq * 2048, HALF_BYTES, 1024), smem_desc(lo + kq * 1024, 512, 128),
                 kIdescPV, 1u);
    }
  }
  mma_commit(bar_addr(ms.empty[s]));
  mma_commit(bar_addr(ms.pempty[pp][pb]));
}

template <int S>
__device__ void mma_role_body(const Ctx& c, const FusedParams& p) {
  Misc& ms = *c.ms;
  wait_or_abort(bar_addr(ms.qfull), 0u, ms, p.status);
  fence_proxy_async();
  int it = 0;
  for (int lev = c.lev_top; lev >= c.lev_end; --lev) {
    for (int pp = 0; pp < c.np; ++pp) {
      int g0, mc;
      scale_slice(m_total(p, lev), c.rank, c.cs, g0, mc);
      const int ntl = tiles_of(mc);
      const uint32_t tb = c.tmem + pp * p.ucols, sq = smem_u32(c.smem + c.ly.q + pp * Q_BYTES);
#pragma unroll 1
      for (int t = 0; t < ntl; ++t) mma_score_tile<S>(c, p, it + t, tb + 32 * t, sq, bar_addr(ms.tdone[pp][t]));
      it += ntl;
    }
  }
  for (int pp = 0; pp < c.np && p.attn; ++pp) {
    int a0, mc;
    attn_slice(p.keep[0] + p.ng, c.rank, c.cs, a0, mc);
    const int ntl = tiles_of(mc);
    const uint32_t tb = c.tmem + pp * p.ucols, sq = smem_u32(c.smem + c.ly.q + pp * Q_BYTES);
    if (ntl == 0) continue;
    // S_t as each key tile lands (its completion on the tile's barrier), then
    // the PV products as the value tiles land and their P tiles are formed.
#pragma unroll 1
    for (int t = 0; t < ntl; ++t) mma_score_tile<S>(c, p, it + t, tb + 32 * t, sq, bar_addr(ms.tdone[pp][t]));
    it += ntl;
#pragma unroll 1
    for (int t = 0; t < ntl; ++t) mma_pv_tile<S>(c, p, pp, it + t, t, tb + p.ucols - 32);
    it += ntl;
    mma_commit(bar_addr(ms.mdone[pp]));  // every PV product of the unit is done
  }
}

// The MMA thread: an optional stalled first wait (test-only), the MMAs, then
// a commit that it waits for (default bound), so that no MMA is still
// writing TMEM when it is freed, also after a wait gave up.
template <int S>
__device__ void mma_role(const Ctx& c, const FusedParams& p) {
  Misc& ms = *c.ms;
  if (p.stall) wait_or_abort(bar_addr(ms.stallbar), 0u, ms, p.status);
  mma_role_body<S>(c, p);
  mma_commit(bar_addr(ms.drainbar));
  (void)mbar_wait_bounded(bar_addr(ms.drainbar), 0u, kDefaultWaitLimit);
}

// ---------------------------------------------------------------------------
// Compute warps.
// ---------------------------------------------------------------------------

// Reduce 32 values per lane across the warp's 32 lanes; afterwards lane i
// holds the reduction of column i (31 shuffles).
template <bool MAX>
__device__ __forceinline__ float transpose_reduce32(float (&v)[32], int lane) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < off; ++j) {
      const float keep = up ? v[j + off] : v[j];
      const float send = up ? v[j] : v[j + off];
      const float recv = __shfl_xor_sync(0xffffffffu, send, off);
      v[j] = MAX ? fmaxf(keep, recv) : keep + recv;
    }
  }
  return v[0];
}


// The warp's (stabiliser, sum of 2^(l sl2 - stabiliser)) per query over its
// rows of TMEM tiles 0..ntl-1, with the stabiliser the column maximum over
// all those rows: the overflow path of scale_sums, one query column at a
// time (compact code for a path that real inputs never take).
template <bool WIDE>
__device__ __noinline__ float2 warp_sums_exact(uint32_t tb, int ntl, int mc, float sl2) {
  const int tid = ctid<WIDE>(), lane = tid & 31, warp = tid >> 5, row = tid & (TM - 1);
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  float2 out = make_float2(-INFINITY, 0.f);
#pragma unroll 1
  for (int i = 0; i < 32; ++i) {
    float mx = -INFINITY;
#pragma unroll 1
    for (int t = unit_wg<WIDE>(); t < ntl; t += tile_step<WIDE>()) {
      const float v = tmem_ld1(tb + lane_base + 32 * t + i);
      if (t * TM + row < mc) mx = fmaxf(mx, v);
    }
    const float mi = warp_max_f32(mx) * sl2;
    float sum = 0.f;
#pragma unroll 1
    for (int t = unit_wg<WIDE>(); t < ntl; t += tile_step<WIDE>()) {
      const float v = tmem_ld1(tb + lane_base + 32 * t + i);
      if (t * TM + row < mc) sum += ex2(fmaf(v, sl2, -mi));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == i) out = make_float2(mi, sum);
  }
  return out;
}

// Softmax statistics of one scale (Eq. 7-8), tile by tile as the MMA thread
// completes them, so that the exponentials of early tiles overlap the
// copies of later ones.  Each compute warp takes as its stabiliser per query
// the largest logit (x sl2, log2 units) of its rows in the first tile (a
// warp with no row there has none in later tiles either) and accumulates the
// sum of 2^(l sl2 - m) over its rows.  A later logit more than ~127 above the
// stabiliser would overflow the sum; the warp then redoes its sums with the
// maximum over all its rows.  The four warps' (m, sum) merge into the CTA's
// (M, S) per query, which goes to slot `rank` of every cluster CTA's xstat.
// tpar holds the parity of each tile barrier's next phase.
template <bool WIDE>
__device__ __noinline__ bool scale_sums(uint32_t rank, uint32_t cs, Misc& ms, int pp, uint32_t tb, int ntl, int mc,
                                        float sl2, uint32_t ecol, uint32_t& tpar, int* status) {
  const int tid = ctid<WIDE>(), lane = tid & 31, warp = tid >> 5, row = tid & (TM - 1);
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  UnitState& us = ms.us[pp];
  const f32x2 s2 = pk2(sl2, sl2);
  f32x2 nml[16], acc[16];
  float mcol = -INFINITY;  // lane i: this warp's stabiliser of query i
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    acc[k] = pk2(0.f, 0.f);
    nml[k] = pk2(0.f, 0.f);
  }
#pragma unroll 1
  for (int t = unit_wg<WIDE>(); t < ntl; t += tile_step<WIDE>()) {
    wait_or_abort(bar_addr(ms.tdone[pp][t]), (tpar >> t) & 1u, ms, status);
    tpar ^= 1u << t;
    tc_fence_after();
    uint32_t ra[32];
    tmem_ld32_issue(tb + lane_base + 32 * t, ra);
    tmem_wait_ld();
    const bool valid = t * TM + row < mc;
    if (t == unit_wg<WIDE>()) {
      float m2[2];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        m2[i & 1] = warp_max_f32(valid ? __uint_as_float(ra[i]) : -INFINITY) * sl2;
        mcol = lane == i ? m2[i & 1] : mcol;
        if (i & 1) nml[i >> 1] = pk2(-m2[0], -m2[1]);
      }
    }
    if (valid) {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const float2 x = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, nml[k]));
        const float e0 = ex2(x.x), e1 = ex2(x.y);
        acc[k] = add2(acc[k], pk2(e0, e1));
        ra[2 * k] = __float_as_uint(e0);
        ra[2 * k + 1] = __float_as_uint(e1);
      }
    }
    // The exponentials stay in TMEM for the ranking keys (rows past the
    // slice store whatever they hold; no key is formed for them).
    if (ecol) tmem_st32(tb + ecol + lane_base + 32 * t, ra);
  }
  if (ecol) tmem_wait_st();
  float a[32];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float2 v = up2(acc[k]);
    a[2 * k] = v.x;
    a[2 * k + 1] = v.y;
  }
  float2 st = make_float2(mcol, transpose_reduce32<false>(a, lane));
  const bool overflow = __any_sync(0xffffffffu, !(st.y <= 3.0e38f));
  if (overflow) st = warp_sums_exact<WIDE>(tb, ntl, mc, sl2);
  sts_v2(smem_u32(&wslots<WIDE>(ms, pp, warp).wstat[warp & 3][lane]), __float_as_uint(st.x), __float_as_uint(st.y));
  csync<WIDE>();
  if (tid < 32) {
    constexpr int NW = unit_warps<WIDE>();
    float2 w[NW];
#pragma unroll
    for (int k = 0; k < NW; ++k) {
      const uint2 v = lds_v2(smem_u32(&wslots<WIDE>(ms, pp, k).wstat[k & 3][tid]));
      w[k] = make_float2(__uint_as_float(v.x), __uint_as_float(v.y));
    }
    float M = -INFINITY;
#pragma unroll
    for (int k = 0; k < NW; ++k)
      if (w[k].y > 0.f) M = fmaxf(M, w[k].x);
    float S = 0.f;
#pragma unroll
    for (int k = 0; k < NW; ++k)
      if (w[k].y > 0.f) S = fmaf(w[k].y, ex2(w[k].x - M), S);
    const uint32_t dst = smem_u32(&us.xstat[rank][tid]);
    const uint32_t bar = bar_addr(ms.xbar[pp]);
    // After a wait gave up, this CTA sends nothing to the cluster.
    const uint32_t nr = aborted(ms) ? 0u : cs;
#pragma unroll 1
    for (uint32_t r = 0; r < nr; ++r)
      st_async_v2(map_rank(dst, r), __float_as_uint(M), __float_as_uint(S), map_rank(bar, r));
  }
  return ecol != 0 && !overflow;  // the stored exponentials are relative to this warp's stabilisers
}

// Softmax normaliser per query, c_i = M + log2 S over the whole candidate
// set from the cluster's (M, S) pairs (padded query columns get +inf and
// weigh 0), into this warp's slot of cw.  Every warp forms its own copy,
// so no barrier across the warps is needed.
template <bool WIDE>
__device__ __forceinline__ void warp_normaliser(Misc& ms, int pp, uint32_t cs, int q) {
  const int lane = threadIdx.x & 31, warp = ctid<WIDE>() >> 5;
  UnitState& us = ms.us[pp];
  UnitState& ws = wslots<WIDE>(ms, pp, warp);
  float2 st[MAXCS];
#pragma unroll
  for (int r = 0; r < MAXCS; ++r) {
    const uint2 v = lds_v2(smem_u32(&us.xstat[min(r, (int)cs - 1)][lane]));
    st[r] = make_float2(__uint_as_float(v.x), __uint_as_float(v.y));
  }
  float M = -INFINITY;
#pragma unroll
  for (int r = 0; r < MAXCS; ++r)
    if (r < (int)cs && st[r].y > 0.f) M = fmaxf(M, st[r].x);
  float S = 0.f;
#pragma unroll
  for (int r = 0; r < MAXCS; ++r)
    if (r < (int)cs && st[r].y > 0.f) S = fmaf(st[r].y, ex2(st[r].x - M), S);
  const float c = lane < q ? M + lg2(S) : INFINITY;
  ws.cw[warp & 3][lane] = c;
  ws.fw[warp & 3][lane] = ex2(ws.wstat[warp & 3][lane].x - c);  // 0 for padded columns and for a warp without rows
  __syncwarp();
}

// Ranking key log2 W_j of each valid row (Eq. 8), stored at position g0 + j
// of every cluster CTA's key array of the unit; each warp's (min, max) key
// goes to slot (rank, warp) of every CTA's kmm on the same barrier.
// With the scale's exponentials e = 2^(l sl2 - m) stored in TMEM at column
// ecol (eok: the warp's sums used those stabilisers m), W_j = sum_i e_ij f_i
// with f_i = 2^(m_i - c_i) from us.fw: fused multiply-adds, no exponentials.
// Otherwise, and for a row whose W is tiny (below 2^-96, where flushed terms
// could matter), the key is a log-sum-exp of the logits over the query rows
// against the normaliser c_i (us.cw): every exponent l sl2 - c_i is at most 0
// (c_i is the log of a sum that contains the row's own term), so the sum
// cannot overflow; padded query columns have c_i = +inf and add 0; a tiny sum
// is taken again shifted by its largest exponent.
// The exact key of one row from its logits (the slow path of pass_keys):
// the log-sum-exp over the query rows of l sl2 - c_i, with c_i at cw_a
// (+inf for padded columns); a tiny sum is taken again shifted by its largest
// exponent.
__device__ __forceinline__ float key_from_logits(const uint32_t (&ra)[32], uint32_t cw_a, float sl2) {
  const f32x2 s2 = pk2(sl2, sl2);
  f32x2 ncv[16];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint4 v = lds_v4(cw_a + 16u * k);
    ncv[2 * k] = pk2(-__uint_as_float(v.x), -__uint_as_float(v.y));
    ncv[2 * k + 1] = pk2(-__uint_as_float(v.z), -__uint_as_float(v.w));
  }
  f32x2 z2 = pk2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float2 v = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, ncv[k]));
    z2 = add2(z2, pk2(ex2(v.x), ex2(v.y)));
  }
  float2 zz = up2(z2);
  float key = lg2(zz.x + zz.y);
  if (zz.x + zz.y < 0x1p-96f) {
    float mx = -INFINITY;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float2 v = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, ncv[k]));
      mx = fmax3(mx, v.x, v.y);
    }
    z2 = pk2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float2 v = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, ncv[k]));
      z2 = add2(z2, pk2(ex2(v.x - mx), ex2(v.y - mx)));
    }
    zz = up2(z2);
    key = mx + lg2(zz.x + zz.y);
  }
  return key;
}

template <bool WIDE>
__device__ __noinline__ void pass_keys(uint32_t rank, uint32_t cs, Misc& ms, int pp, uint32_t tb, int ntl, int mc,
                                       int g0, float sl2, uint32_t keys_a, uint32_t ecol, bool eok) {
  const int tid = ctid<WIDE>(), lane = tid & 31, warp = tid >> 5, row = tid & (TM - 1);
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  const uint32_t bar = bar_addr(ms.kbar[pp]);
  UnitState& ws = wslots<WIDE>(ms, pp, warp);
  const uint32_t cw_a = smem_u32(&ws.cw[warp & 3][0]);
  float kmin = INFINITY, kmax = -INFINITY;
  // After a wait gave up, this CTA sends nothing to the cluster.
  const uint32_t nr = aborted(ms) ? 0u : cs;
  auto emit = [&](int j, float key) {
    if (j < mc) {
      // A row whose logits are all -inf has no weight: its key is a NaN here
      // (-inf - -inf, or the zero rows that pad the queries times an infinity)
      // and must be -inf, below every other.
      key = fmaxf(key, -INFINITY);
      kmin = fminf(kmin, key);
      kmax = fmaxf(kmax, key);
      const uint32_t dst = keys_a + 4u * (uint32_t)(g0 + j);
#pragma unroll 1
      for (uint32_t r = 0; r < nr; ++r) st_async_b32(map_rank(dst, r), __float_as_uint(key), map_rank(bar, r));
    }
  };
  if (eok) {
    f32x2 fv[16];
    const uint32_t fw_a = smem_u32(&ws.fw[warp & 3][0]);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint4 f = lds_v4(fw_a + 16u * k);
      fv[2 * k] = pk2(__uint_as_float(f.x), __uint_as_float(f.y));
      fv[2 * k + 1] = pk2(__uint_as_float(f.z), __uint_as_float(f.w));
    }
#pragma unroll 1
    for (int t = unit_wg<WIDE>(); t < ntl; t += tile_step<WIDE>()) {
      uint32_t ra[32];
      tmem_ld32_issue(tb + ecol + lane_base + 32 * t, ra);
      tmem_wait_ld();
      f32x2 z2 = pk2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 16; ++k) z2 = fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), fv[k], z2);
      const float2 zz = up2(z2);
      float key = lg2(zz.x + zz.y);
      const int j = t * TM + row;
      const bool slow = zz.x + zz.y < 0x1p-96f;
      if (__any_sync(0xffffffffu, slow && j < mc)) {
        // A tiny W: the exact key from the logits (the whole warp reloads them;
        // TMEM loads are warp-wide).
        uint32_t sa[32];
        tmem_ld32_issue(tb + lane_base + 32 * t, sa);
        tmem_wait_ld();
        const float k2 = key_from_logits(sa, cw_a, sl2);
        key = slow ? k2 : key;
      }
      emit(j, key);
    }
  } else {
#pragma unroll 1
    for (int t = unit_wg<WIDE>(); t < ntl; t += tile_step<WIDE>()) {
      uint32_t ra[32];
      tmem_ld32_issue(tb + lane_base + 32 * t, ra);
      tmem_wait_ld();
      emit(t * TM + row, key_from_logits(ra, cw_a, sl2));
    }
  }
  // The warp's key range goes with the keys (the Top-K's first bucket range).
  kmin = warp_min_f32(kmin);
  kmax = warp_max_f32(kmax);
  if (lane == 0) {
    const uint32_t dst = smem_u32(&ws.kmm[rank][warp & 3]);
#pragma unroll 1
    for (uint32_t r = 0; r < nr; ++r)
      st_async_v2(map_rank(dst, r), __float_as_uint(kmin), __float_as_uint(kmax), map_rank(bar, r));
  }
  // Every TMEM read of the scale is done before the Top-K's barriers.
  tc_fence_before();
}

// OR of a predicate over the unit's compute threads (a barrier of theirs).
template <bool WIDE>
__device__ __forceinline__ bool csync_or(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\tsetp.ne.u32 pi, %1, 0;\n\tbar.red.or.pred po, %2, %3, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(kCsyncId + (WIDE ? 0u : (threadIdx.x >> 7))), "r"(32u * unit_warps<WIDE>())
      : "memory");
  return r != 0;
}

// Attention of unit pp over its key slice, tile by tile as the MMA thread
// completes each S tile: P = 2^(s sl2 - m) (bf16, P^T MN-major core matrices)
// into the unit's P double buffer for the MMA thread, so the value tiles are
// consumed while later key tiles still stream.  The stabiliser m_i (x sl2,
// log2 units) is the largest logit of query i in the first step's tiles (one
// tile, or one per warpgroup in the WIDE mode).  A later step whose logits
// exceed m_i by more than kRaise raises m_i to that step's maximum first (a
// decision taken jointly by the unit's threads; real inputs do not take it):
// every PV product issued so far completes, column i of the O^T accumulator
// and the running sums are scaled by 2^(m_old - m_new), and the step's P uses
// the new m.  Otherwise P <= 2^kRaise, which bf16 holds and fp32 sums over
// any key list accumulate without overflow; terms more than 2^126 below the
// stabiliser flush to zero, as they do below the largest term.  Rows past the
// slice get P = 0.  The final m -> us.mloc, the row sums of P -> us.lacc.
// WIDE: warpgroup w forms the P tiles t = w, w + 2, ... (always P buffer w).
// LOW: P has a second term, in the unit's buffers lo.
constexpr float kRaise = 64.f;
template <bool WIDE, bool LOW>
__device__ __noinline__ void attn_online(Misc& ms, int* status, float sl2, uint8_t* pbase, uint8_t* lo, int pp,
                                         uint32_t tb, int ntl, int mc, uint32_t& tpar, uint32_t ocol) {
  const int tid = ctid<WIDE>(), lane = tid & 31, warp = tid >> 5, row = tid & (TM - 1);
  const int wg = unit_wg<WIDE>();
  constexpr int NW = unit_warps<WIDE>();
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  UnitState& us = ms.us[pp];
  UnitState& ws = wslots<WIDE>(ms, pp, warp);
  const f32x2 s2 = pk2(sl2, sl2);
  f32x2 nml[16], lsum2[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    nml[k] = pk2(0.f, 0.f);
    lsum2[k] = pk2(0.f, 0.f);
  }
  const int nsteps = (ntl + tile_step<WIDE>() - 1) / tile_step<WIDE>();
#pragma unroll 1
  for (int j = 0; j < nsteps; ++j) {
    const int t = j * tile_step<WIDE>() + wg;
    const bool has = t < ntl;  // warp-uniform
    uint32_t ra[32];
    if (has) {
      wait_or_abort(bar_addr(ms.tdone[pp][t]), (tpar >> t) & 1u, ms, status);
      tpar ^= 1u << t;
      tc_fence_after();
      tmem_ld32_issue(tb + lane_base + 32 * t, ra);
      tmem_wait_ld();
    }
    const bool valid = has && t * TM + row < mc;
    bool raise = j == 0;
    if (j > 0) {
      bool over = false;
      if (valid) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float2 x = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, nml[k]));
          over |= fmaxf(x.x, x.y) > kRaise;
        }
      }
      raise = csync_or<WIDE>(over);
    }
    if (raise) {
      // The step's column maxima: lane i of each warp keeps column i's.
      float mcol = -INFINITY;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float m = warp_max_f32(valid ? __uint_as_float(ra[i]) : -INFINITY);
        mcol = lane == i ? m : mcol;
      }
      ws.red[warp & 3][lane] = mcol;
      csync<WIDE>();
      if (tid < 32) {
        float m = -INFINITY;
#pragma unroll
        for (int w = 0; w < NW; ++w) m = fmaxf(m, wslots<WIDE>(ms, pp, w).red[w & 3][tid]);
        m = fmaxf(m * sl2, -FLT_MAX);  // finite also where every logit so far is -inf: P is 0 there, not 2^(-inf + inf)
        const float mn = j == 0 ? m : fmaxf(us.mloc[tid], m);
        us.alpha[tid] = j == 0 ? 1.f : ex2(us.mloc[tid] - mn);
        us.mloc[tid] = mn;
      }
      csync<WIDE>();
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        nml[k] = pk2(-us.mloc[2 * k], -us.mloc[2 * k + 1]);
        lsum2[k] = mul2(lsum2[k], pk2(us.alpha[2 * k], us.alpha[2 * k + 1]));
      }
      if (j > 0 && wg == 0) {
        // Every PV product issued so far (through tile tl) completes; then the
        // accumulator's columns take the factor.  The tile's P is not
        // announced before, so the next product sees the scaled O^T.
        const int tl = j * tile_step<WIDE>() - 1;
        if (lane == 0) wait_or_abort(bar_addr(ms.pempty[pp][tl & 1]), (uint32_t)(tl >> 1) & 1u, ms, status);
        __syncwarp();
        tc_fence_after();
        uint32_t o[32];
        tmem_ld32_issue(ocol + lane_base, o);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * us.alpha[i]);
        tmem_st32(ocol + lane_base, o);
        tmem_wait_st();
        tc_fence_before();
      }
    }
    if (has) {
      const uint32_t pb = (uint32_t)t & 1u, pn = (uint32_t)t >> 1;
      if (t >= 2) {
        if (lane == 0) wait_or_abort(bar_addr(ms.pempty[pp][pb]), (pn - 1) & 1u, ms, status);
        __syncwarp();
      }
      // P^T, MN-major core matrices: key group r / 8, query chunk ch.  Rows
      // past the slice: P = 0.
      const int at = (row >> 3) * 512 + (row & 7) * 16;
      uint8_t* dst = pbase + pb * P_BYTES + at;
      if (PTERMS == 1 && !LOW) {
        uint32_t w[16];
        if (valid) {
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float2 x = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, nml[k]));
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(ex2(x.x), ex2(x.y));
            lsum2[k] = add2(lsum2[k], pk2(__low2float(h2), __high2float(h2)));
            w[k] = *reinterpret_cast<const uint32_t*>(&h2);
          }
        } else {
#pragma unroll
          for (int k = 0; k < 16; ++k) w[k] = 0u;
        }
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
          *reinterpret_cast<uint4*>(dst + ch * 128) =
              make_uint4(w[4 * ch], w[4 * ch + 1], w[4 * ch + 2], w[4 * ch + 3]);
      } else {
        // The exponentials take the logits' registers; each term is stored
        // and taken off what is left.
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float2 x = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, nml[k]));
          const float e0 = valid ? ex2(x.x) : 0.f, e1 = valid ? ex2(x.y) : 0.f;
          lsum2[k] = add2(lsum2[k], pk2(e0, e1));
          ra[2 * k] = __float_as_uint(e0);
          ra[2 * k + 1] = __float_as_uint(e1);
        }
#pragma unroll
        for (int e = 0; e < (LOW ? 2 : PTERMS); ++e) {
          uint8_t* de = LOW && e == 1 ? lo + pb * PT_BYTES + at : dst + e * PT_BYTES;
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int i = 8 * ch + 2 * k;
              const __nv_bfloat162 h2 =
                  __floats2bfloat162_rn(__uint_as_float(ra[i]), __uint_as_float(ra[i + 1]));
              ra[i] = __float_as_uint(__uint_as_float(ra[i]) - __low2float(h2));
              ra[i + 1] = __float_as_uint(__uint_as_float(ra[i + 1]) - __high2float(h2));
              w[k] = *reinterpret_cast<const uint32_t*>(&h2);
            }
            *reinterpret_cast<uint4*>(de + ch * 128) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      }
      fence_proxy_async();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_addr(ms.pfull[pp][pb]));
    }
  }
  float lsum[32];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float2 v = up2(lsum2[k]);
    lsum[2 * k] = v.x;
    lsum[2 * k + 1] = v.y;
  }
  ws.red[warp & 3][lane] = transpose_reduce32<false>(lsum, lane);
  csync<WIDE>();
  if (tid < 32) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) sum += wslots<WIDE>(ms, pp, w).red[w & 3][tid];
    us.lacc[tid] = sum;
    if (nsteps == 0) us.mloc[tid] = -INFINITY;  // no keys in this CTA's slice
  }
  csync<WIDE>();
}

// Rows of a query group in the combine buffer for a slice of `rows`: one of
// padding, against bank conflicts, where the buffer has the room.
__device__ __forceinline__ int comb_rows(int rows, int cs) { return rows + ((rows + 1) * cs <= D + MAXCS ? 1 : 0); }

// Attention combine of unit pp: this CTA's partial O^T rows go to the CTA
// owning their head-dim slice (with the CTA's (m, l) per query), and this
// CTA combines the cluster's partials of its own slice and writes those
// columns of O (bf16).  The partials land in each owner's P buffers of the
// unit, which are free once the owner's own PV products are done; owners
// announce that before any partial is sent.
// (Run by one warpgroup of the unit: four warps, one per TMEM lane quarter.)
__device__ __noinline__ void attn_combine(Misc& ms, const FusedParams& p, uint32_t rank, uint32_t cs, int u,
                                          uint8_t* comb, UnitState& us, int pp, uint32_t ocol) {
  const int tid = threadIdx.x & (NCT - 1), warp = tid >> 5;
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  uint32_t orow[32];
  tmem_ld32_issue(ocol + lane_base, orow);
  tmem_wait_ld();
  const uint32_t ready = bar_addr(ms.cready[pp]);
  // One arrival per CTA, each from its own thread (every thread has seen
  // this unit's PV products complete), so the remote arrivals overlap.  A CTA
  // whose wait gave up announces nothing and sends nothing: its P buffers
  // may still be in use, and the partials of others must not land there.
  if (tid < (int)cs && !aborted(ms)) mbar_arrive_cluster(map_rank(ready, (uint32_t)tid));
  wait_cluster_or_abort(ready, 0u, ms, p.status);
  const uint32_t comb_a = smem_u32(comb);
  const uint32_t cbar = bar_addr(ms.cbar[pp]);
  const bool send = !aborted(ms);  // every owner has announced its buffers free
  if (send && tid < D) {
    // Owner of head-dim row d = tid, and the row's place in its buffer.
    int owner = tid * (int)cs / D;
    while (owner + 1 < (int)cs && dlo(owner + 1, cs) <= tid) ++owner;
    const int orows = dlo(owner + 1, cs) - dlo(owner, cs);
    const int dl = tid - dlo(owner, cs);
    // Four queries a store, at [source][query / 4][row] (comb_rows a group): the
    // lanes of a warp hold consecutive rows, so each store of theirs
    // covers consecutive addresses, and the owner's reads (a lane a query) hit
    // distinct banks.
    const uint32_t step = 16u * (uint32_t)comb_rows(orows, (int)cs);
    const uint32_t dst = map_rank(comb_a + 8u * rank * step + 16u * (uint32_t)dl, (uint32_t)owner);
    const uint32_t rb = map_rank(cbar, (uint32_t)owner);
#pragma unroll
    for (int i = 0; i < 32; i += 4)
      st_async_v4(dst + (uint32_t)(i / 4) * step, orow[i], orow[i + 1], orow[i + 2], orow[i + 3], rb);
  }
  if (tid < 32 && send) {
    const uint32_t dst = smem_u32(&us.cstat[rank][tid]);
#pragma unroll 1
    for (uint32_t r = 0; r < cs; ++r)
      st_async_v2(map_rank(dst, r), __float_as_uint(us.mloc[tid]), __float_as_uint(us.lacc[tid]),
                  map_rank(cbar, r));
  }
  wait_cluster_or_abort(cbar, 0u, ms, p.status);
  // A thread always serves query qi = tid % 32: the weight 2^(m_r - M) of
  // every source CTA and the denominator are formed once.
  const int qi = tid & (NQ - 1);
  const uint32_t cst_a = smem_u32(&us.cstat[0][qi]);
  float2 st[MAXCS];
#pragma unroll
  for (int r = 0; r < MAXCS; ++r) {
    const uint2 v = lds_v2(cst_a + (uint32_t)(min(r, (int)cs - 1) * NQ * 8));
    st[r] = make_float2(__uint_as_float(v.x), __uint_as_float(v.y));
  }
  float M = -INFINITY;
#pragma unroll
  for (int r = 0; r < MAXCS; ++r)
    if (r < (int)cs && st[r].y > 0.f) M = fmaxf(M, st[r].x);
  float f[MAXCS], den = 0.f;
#pragma unroll
  for (int r = 0; r < MAXCS; ++r) {
    f[r] = (r < (int)cs && st[r].y > 0.f) ? ex2(st[r].x - M) : 0.f;  // a CTA with no keys contributes nothing
    den = fmaf(st[r].y, f[r], den);
  }
  const float inv = 1.f / den;
  bf16* ob = p.O + (int64_t)(u / p.H) * p.osb + (int64_t)(u % p.H) * p.osh;
  const int d0 = dlo((int)rank, cs), rows = dlo((int)rank + 1, cs) - d0;
  const int crows = comb_rows(rows, (int)cs);
  auto out = [&](int dl) {
    float n = 0.f;
#pragma unroll
    for (int r = 0; r < MAXCS; ++r)
      if (r < (int)cs)
        n = fmaf(lds_f32(comb_a + 16u * (uint32_t)((r * 8 + (qi >> 2)) * crows + dl) + 4u * (uint32_t)(qi & 3)),
                 f[r], n);
    return n * inv;
  };
  // A slice of a multiple of 8 rows (clusters of a power of two): warp w
  // writes its quarter of the 8-row pieces of its query, 16 bytes a store;
  // otherwise one element a store.
  const bool vec = rows % 8 == 0 && d0 % 8 == 0 && p.oss % 8 == 0 && (reinterpret_cast<uintptr_t>(ob) & 15) == 0;
  if (qi < p.q && vec) {
    const int np8 = rows / 8;
#pragma unroll 1
    for (int c0 = 8 * (warp * np8 / NCW); c0 < 8 * ((warp + 1) * np8 / NCW); c0 += 8) {
      uint32_t w4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(out(c0 + 2 * e), out(c0 + 2 * e + 1));
        w4[e] = *reinterpret_cast<const uint32_t*>(&h);
      }
      *reinterpret_cast<uint4*>(ob + (int64_t)qi * p.oss + d0 + c0) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
    }
  } else if (qi < p.q) {
#pragma unroll 1
    for (int dl = tid >> 5; dl < rows; dl += NCT / NQ) ob[(int64_t)qi * p.oss + d0 + dl] = __float2bfloat16_rn(out(dl));
  }
}

// The compute warps of unit pp = threadIdx.x / NCT of the cluster's units.
// WIDE: both warpgroups serve the cluster's one unit.
template <bool WIDE>
__device__ void compute_role(const Ctx& c, const FusedParams& p) {
  Misc& ms = *c.ms;
  constexpr int TN = 32 * unit_warps<WIDE>();  // the unit's compute threads
  const int tid = ctid<WIDE>();
  const int pp = WIDE ? 0 : threadIdx.x / NCT;
  if (pp >= c.np) return;
  UnitState& us = ms.us[pp];
  uint8_t* ubuf = c.smem + c.ly.p + pp * UNIT_P_BYTES;  // P buffers, Top-K scratch, combine buffer
  const uint32_t sc_a = smem_u32(ubuf);
  const uint32_t tb = c.tmem + pp * p.ucols;
  const int u = c.u0 + pp;
  const float sl2 = p.scale_log2;
  int64_t sets_off = 0;  // the level sets of the scales above this launch's first
  for (int l = p.L; l > c.lev_top; --l) sets_off += p.keep[l];
  // The unit's mdone barrier completes one phase, when the attention's PV
  // products are done (the MMA thread commits it only for a non-empty slice).
  auto wait_mdone = [&]() {
    wait_or_abort(bar_addr(ms.mdone[pp]), 0u, ms, p.status);
    tc_fence_after();
  };
  // A launch that starts below the top scale (its rows dense, so the
  // producers do not need it): the previous selection J_{lev_top+1}, for the
  // first Top-K's winners, from the children list it was handed (halved).
  // The Top-K's first barrier orders it.
  if (c.lev_top < p.L) {
    const int32_t* src = p.jin + (int64_t)u * p.jstride;
    int32_t* Jp = unit_J(c, p, pp, c.lev_top + 1);
#pragma unroll 1
    for (int i = tid; i < p.keep[c.lev_top + 1]; i += TN) Jp[i] = src[2 * i] >> 1;
  }
  if (kAlone && p.sel) {
    const int32_t* src = p.sel + (int64_t)u * p.keep[0];
    int32_t* J = unit_J(c, p, pp, 0);
#pragma unroll 1
    for (int i = tid; i < p.keep[0]; i += TN) J[i] = min(max(src[i], 0), p.n - 1);
    csync<WIDE>();
    if (tid == 0) mbar_arrive(bar_addr(ms.jready[pp]));
  }
  // The first pass through the Top-K's code fetches its instructions from
  // memory, where they queue behind the first scale's row streams (several us
  // at 32K).  In a two-unit cluster unit 1's warpgroup, which waits for its
  // first rows until unit 0's have streamed, runs the Top-K once on synthetic
  // keys with the first scale's list length, so unit 0's first selection
  // finds the code cached (measured: 32K step 82.6 -> 80.5 us; in one-unit
  // clusters the warm-up delays the unit's own first scale and the 128K step
  // was 2 us slower).  Its key buffer is the one the scale below receives,
  // which no CTA fills before this one has finished its first selection; the
  // Top-K leaves its scratch cleared.
  if (!WIDE && pp == 1 && c.lev_top == p.L && c.lev_top > c.lev_end) {
    const int m0 = m_total(p, c.lev_top);
    int32_t* wk = unit_J(c, p, pp, c.lev_top - 1);
    // 512 distinct values, each several times: one bucket round whose
    // boundary bucket holds more keys than it needs, like real keys.
#pragma unroll 1
    for (int i = tid; i < m0; i += TN) wk[i] = __float_as_int((float)((((uint32_t)i * 2654435761u) >> 8) & 511u));
    csync<WIDE>();
    select_topk<WIDE>(smem_u32(wk), m0, p.keep[c.lev_top], 0u, 1, sc_a, 0.f, 511.f);
  }
  uint32_t tpar = 0;  // parity of each scale-tile barrier's next phase
#pragma unroll 1
  for (int lev = c.lev_top; lev >= c.lev_end; --lev) {
    const uint32_t ph = (uint32_t)(c.lev_top - lev) & 1u;  // phase of the per-scale barriers
    const int m = m_total(p, lev);
    int g0, mc;
    scale_slice(m, c.rank, c.cs, g0, mc);
    const int ntl = tiles_of(mc);
    const int kb = p.keep[lev];
    int32_t* J = unit_J(c, p, pp, lev);  // receives this scale's keys, then its selection
    const uint32_t keys_a = smem_u32(J);
    const bool eok = scale_sums<WIDE>(c.rank, c.cs, ms, pp, tb, ntl, mc, sl2, p.ecol, tpar, p.status);
    wait_cluster_or_abort(bar_addr(ms.xbar[pp]), ph, ms, p.status);
    // This phase is complete for tid 0, so the arrival arms the next one.
    // After a wait gave up the phase may still be pending (its bytes never
    // came): a second arrival would then underflow the phase's arrival
    // count, so an aborted CTA arms nothing.
    if (tid == 0 && lev > c.lev_end && !aborted(ms)) mbar_arrive_expect_tx(bar_addr(ms.xbar[pp]), c.cs * NQ * 8u);
    warp_normaliser<WIDE>(ms, pp, c.cs, p.q);
    pass_keys<WIDE>(c.rank, c.cs, ms, pp, tb, ntl, mc, g0, sl2, keys_a, p.ecol, eok);
    wait_cluster_or_abort(bar_addr(ms.kbar[pp]), ph, ms, p.status);
    // The keys' range from the cluster warps' (min, max).
    float lo, hi;
    {
      constexpr int NW = unit_warps<WIDE>();
      const int lane = tid & 31;
      float2 mm = make_float2(INFINITY, -INFINITY);
#pragma unroll 1
      for (int e = lane; e < (int)c.cs * NW; e += 32) {  // entry (CTA e / NW, warp e % NW)
        const int w = e % NW;
        const uint2 v = lds_v2(smem_u32(&wslots<WIDE>(ms, pp, w).kmm[e / NW][w & 3]));
        mm = make_float2(fminf(mm.x, __uint_as_float(v.x)), fmaxf(mm.y, __uint_as_float(v.y)));
      }
      lo = warp_min_f32(mm.x);
      hi = warp_max_f32(mm.y);
    }
    // Eq. 9: Top-K (the same result in every CTA of the cluster).
    select_topk<WIDE>(keys_a, m, kb, smem_u32(unit_J(c, p, pp, lev + 1)), lev == p.L, sc_a, lo, hi);
    if (tid == 0) {
      if (lev > c.lev_end && !aborted(ms))  // as for xbar above
        mbar_arrive_expect_tx(bar_addr(ms.kbar[pp]),
                              4u * (uint32_t)m_total(p, lev - 1) + c.cs * unit_warps<WIDE>() * 8u);
      mbar_arrive(bar_addr(ms.jready[pp]));  // the selection is complete (the Top-K ends on a barrier)
    }
    if (c.rank == 0) {
      int32_t* ls = p.level_sets ? p.level_sets + (int64_t)u * p.sets_stride + sets_off : nullptr;
      if (lev >= 1 && ls) {
#pragma unroll 1
        for (int i = tid; i < kb; i += TN) ls[i] = J[i];
      }
      if (lev == c.lev_end && !p.final_sel) {
        // A launch that ends above the final scale hands on the children of
        // its last selection (the next launch's candidates).
        int32_t* out = p.jout + (int64_t)u * p.jstride;
#pragma unroll 1
        for (int t = tid; t < 2 * kb; t += TN) out[t] = 2 * J[t >> 1] + (t & 1);
      } else if (lev == c.lev_end) {
        // mu^0: the children of J^1, or the trimmed level-0 selection.
        const int kk = p.keep[0];
        int32_t* out = p.idx + (int64_t)u * kk;
        int32_t* ls0 = ls ? ls + (lev >= 1 ? kb : 0) : nullptr;
#pragma unroll 1
        for (int t = tid; t < kk; t += TN) {
          const int tok = p.trim ? J[t] : 2 * J[t >> 1] + (t & 1);
          out[t] = tok;
          if (ls0) ls0[t] = tok;
        }
      }
    }
    if (lev >= 1) sets_off += kb;
  }
  if (!p.attn) return;

  // Attention: S of the key slice, P for the MMA thread, then the combine.
  int a0, mc;
  attn_slice(p.keep[0] + p.ng, c.rank, c.cs, a0, mc);
  const int ntl = tiles_of(mc);
  attn_online<WIDE, kLowTerm>(ms, p.status, sl2, ubuf, c.smem + c.ly.lo + 2 * pp * PT_BYTES, pp, tb, ntl, mc, tpar,
                              tb + p.ucols - 32);
  if (ntl > 0) wait_mdone();  // every PV product of the unit is done
  if (unit_wg<WIDE>() != 0) return;  // one warpgroup combines
  attn_combine(ms, p, c.rank, c.cs, u, ubuf, us, pp, tb + p.ucols - 32);
}

template <int S, bool WIDE>
__global__ void __launch_bounds__(NT, 1) wf_fused_kernel(const __grid_constant__ FusedParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  Ctx c;
  c.smem = smem;
  c.ly = smem_layout(S, p.P, p.cmax, p.kmax, p.sel != nullptr);
  c.ms = reinterpret_cast<Misc*>(smem + c.ly.misc);
  Misc& ms = *c.ms;
  c.rank = cluster_rank();
  c.cs = cluster_size();
  c.u0 = (int)cluster_id_x() * p.P;
  c.np = min(p.P, p.U - c.u0);
  c.lev_top = p.lev_top;
  c.lev_end = p.lev_bot;
  c.stages = S;
  const int tid = threadIdx.x, warp = tid >> 5;

  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(bar_addr(ms.full[s]), NPT);
      mbar_init(bar_addr(ms.empty[s]), 1);
    }
    for (int pp = 0; pp < MAXP; ++pp) {
      mbar_init(bar_addr(ms.mdone[pp]), 1);
      mbar_init(bar_addr(ms.jready[pp]), 1);
      mbar_init(bar_addr(ms.xbar[pp]), 1);
      mbar_init(bar_addr(ms.kbar[pp]), 1);
      for (int t = 0; t < MAXT; ++t) mbar_init(bar_addr(ms.tdone[pp][t]), 1);
    }
    for (int pp = 0; pp < MAXP; ++pp) {
      for (int i = 0; i < 2; ++i) {
        mbar_init(bar_addr(ms.pfull[pp][i]), NCW);
        mbar_init(bar_addr(ms.pempty[pp][i]), 1);
      }
      mbar_init(bar_addr(ms.cbar[pp]), 1);
      mbar_init(bar_addr(ms.cready[pp]), c.cs);
    }
    mbar_init(bar_addr(ms.qfull), NPT);
    mbar_init(bar_addr(ms.stallbar), 1);
    mbar_init(bar_addr(ms.drainbar), 1);
    ms.wait_limit = p.wait_limit;
    ms.abort = 0;
    fence_mbar_init();
  }
  __syncthreads();  // this CTA's barriers exist
  if (warp > MMA_WARP) {
    // The producers touch only this CTA's ring and barriers, so they start at
    // once: they join the cluster barrier's first phase now (nothing of theirs
    // needs ordering before other CTAs' remote stores) and wait for it at the
    // end, while the other warps finish the set-up.
    cluster_arrive_relaxed();
    grid_dep_wait();  // the rows come from the grids before a programmatic launch
    producer_role<S>(c, p);
    cluster_wait();
  } else {
    constexpr int NS = NT - NPT;  // the set-up threads: compute warps and the MMA warp
    if (tid == 0) {
      // Arm the first phase of every receive barrier (bytes this CTA expects).
      for (int pp = 0; pp < c.np; ++pp) {
        if (!kAlone || c.lev_top >= c.lev_end) {
          mbar_arrive_expect_tx(bar_addr(ms.xbar[pp]), c.cs * NQ * 8u);
          mbar_arrive_expect_tx(bar_addr(ms.kbar[pp]),
                                4u * (uint32_t)m_total(p, c.lev_top) + c.cs * unit_warps<WIDE>() * 8u);
        }
        const uint32_t rows = (uint32_t)(dlo((int)c.rank + 1, c.cs) - dlo((int)c.rank, c.cs));
        mbar_arrive_expect_tx(bar_addr(ms.cbar[pp]), c.cs * rows * NQ * 4u + c.cs * NQ * 8u);
      }
    }
    if (warp == MMA_WARP) {
      tmem_alloc(smem_u32(&ms.tmem_base), p.tmem_cols);
      tmem_relinquish();
    }
    // The Top-K scratch starts zeroed (histogram, list counter, masks).
    for (int pp = 0; pp < c.np; ++pp) {
      uint8_t* sc = smem + c.ly.p + pp * UNIT_P_BYTES;
      for (int e = tid; e < (int)((sizeof(SelScratch) + 15) / 16); e += NS)
        *reinterpret_cast<uint4*>(sc + 16 * e) = make_uint4(0, 0, 0, 0);
    }
    // Global memory only after the grids this launch depends on are done (the
    // set-up above overlaps their tail when the launch is programmatic).
    grid_dep_wait();
    tc_fence_before();
    named_sync(kSetupSyncId, NS);
    tc_fence_after();
    grid_dep_launch();  // after the barrier that publishes the tensor memory (see Launch)
    c.tmem = ms.tmem_base;
    cluster_sync();  // every CTA's barriers are armed before any remote arrival
    if (warp < MMA_WARP) {
      compute_role<WIDE>(c, p);
    } else {
      if ((tid & 31) == 0) mma_role<S>(c, p);
      __syncwarp();
    }
  }

  tc_fence_before();
  __syncthreads();
  // No CTA leaves while another may still address its shared memory.
  cluster_arrive();
  cluster_wait();
  if (warp == MMA_WARP) {
    if (aborted(ms)) {
      // After a wait gave up, asynchronous stores from cluster CTAs that were
      // not waited for may still be landing in this CTA's shared memory:
      // every CTA has issued its last one (all are past the cluster
      // barrier), so a short pause lets them complete before the CTA leaves.
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 20000ull) {
      }
    }
    tc_fence_after();
    tmem_dealloc(c.tmem, p.tmem_cols);
  }
}

#if !WF_STAGE_CALLS

// ---------------------------------------------------------------------------
// Grouped query heads (reading 21): the filter of one key head for the
// stacked query rows of its G query heads, W_j summed over every row of the
// group (Eq. 7-11; Dream-7B's 7 query heads per key head give 224 rows).
// ---------------------------------------------------------------------------
//
// One cluster of CS CTAs per (batch, key head) unit, both compute warpgroups
// on the unit, the same producers and Top-K as the one-head kernel.  Every
// scale runs two passes over the CTA's rows, each with the side of the
// product on the TMEM lanes that its sums run along, so that both are serial
// sums of a thread:
//   1. query rows on the lanes (S = Q rows^T, M tiles of 128 stacked query
//      rows, 128 candidates a tile): each thread holds one query row's
//      stabiliser (x sl2, raised when a logit exceeds it by 2^64) and sum of
//      exponentials over the tile's columns.  Two M tiles: warpgroup w takes M
//      tile w of every tile; one: the warpgroups take alternate tiles, and a
//      block of at most 64 rows stands 2 or 4 times in the M tile, so that
//      every warp has real rows and takes that part of the columns.  The
//      cluster exchanges the (M, S) into the normalisers c_i = M + log2 S.
//   2. candidates on the lanes (S^T = rows Q^T, the stacked block's chunks of
//      32 query rows as 32 nch columns): each thread sums its candidate's
//      ranking key log2 W_j = log2 sum_i 2^(l_ij sl2 - c_i), all-gathered, then
//      the Top-K (Eq. 9).  Warpgroup w reads every other TMEM region.  The last
//      tiles of pass 1 (as many as the ring has stages) stay in shared memory
//      and are multiplied again from there; only earlier ones are streamed
//      again.
// With two M tiles the passes use the same TMEM columns in turn; with one,
// pass 2 has columns of its own (as many regions as fit), and its products
// follow pass 1's at once.  (With the candidates on the lanes in both passes,
// pass 1 needed a warp-wide maximum and a 31-shuffle transpose per 32 x 32
// logits, about 7 instructions a logit against 2.5: 32 key heads x 32K tokens
// with 224 stacked rows, 85.3 us a launch against 72.  Each tile's pass 2
// product issued right behind its pass 1 product delayed the next tile's:
// 64 stacked rows x 16K, 62 us a launch against 56.)
// The selection is written as mu^0 (and the level sets); the attention runs
// afterwards on the per-stage tensor-core kernels.
constexpr int GQ_MAXCH = 8;  // chunks of 32 stacked query rows (G q <= 256)

// How often the stacked block stands in its M tile (nch <= 2).
__host__ __device__ constexpr int gqa_copies(int nch) { return nch <= 2 ? 4 / nch : 1; }
// TMEM regions of pass 2 (an even number: warpgroup w reads regions w, w + 2,
// ..) and the column of the first: beside pass 1's two buffers of 128 columns
// (one M tile), or in their place (two).
__host__ __device__ constexpr int gqa_regions(int nch) { return nch > 4 ? 2 : (256 / (32 * nch)) & ~1; }
__host__ __device__ constexpr uint32_t gqa_region0(int nch) { return nch > 4 ? 0u : 256u; }

struct GqaLayout {
  uint32_t q, sc, misc, wst, xst, cvec, buf, bufw, total;
};
__host__ __device__ inline GqaLayout gqa_layout(int stages, int nch, int cs, int cmax, int kmax) {
  GqaLayout l;
  const uint32_t nq = 32u * (uint32_t)nch;
  l.q = (uint32_t)stages * TILE_BYTES;
  l.sc = l.q + (uint32_t)(nch * gqa_copies(nch)) * Q_BYTES;        // Top-K scratch
  l.misc = (l.sc + (uint32_t)sizeof(SelScratch) + 127u) / 128u * 128u;
  l.wst = (l.misc + (uint32_t)sizeof(Misc) + 15u) / 16u * 16u;     // [256] float2: each thread's statistics (one M tile)
  l.xst = l.wst + 256u * 8u;                                       // [cs][nq] float2: every CTA's (M, S) per column
  l.cvec = l.xst + (uint32_t)cs * nq * 8u;                         // [nq] float: the normalisers c_i
  l.buf = (l.cvec + nq * 4u + 127u) / 128u * 128u;                 // two key / selection buffers
  l.bufw = (uint32_t)((max(cmax, kmax) + 3) / 4 * 4);
  l.total = l.buf + 2u * 4u * l.bufw;
  return l;
}

// (m, s) pairs of sums of 2^(x - m): the pair of their union.
__device__ __forceinline__ float2 merge_ms(float2 a, float2 b) {
  if (!(b.y > 0.f)) return a;
  if (!(a.y > 0.f)) return b;
  const float M = fmaxf(a.x, b.x);
  return make_float2(M, a.y * ex2(a.x - M) + b.y * ex2(b.x - M));
}

// The stacked query block, by the compute warps (idle until the first tile is
// multiplied) while the producers start on the rows: up to 56 KB of copies took
// the producers several us ahead of their first row.
__device__ void gqa_load_queries(const Ctx& c, const FusedParams& p) {
  const int tid = threadIdx.x;
  // Row i = g q + r is row r of query head
  // h G + g; chunk ch holds rows 32 ch .. 32 ch + 31 (K-major core matrices),
  // rows >= G q zero-filled.
  const int64_t b = c.u0 / p.H, h = c.u0 % p.H;
  const int nq = p.G * p.q;
  for (int cc = 0; cc < p.nch * gqa_copies(p.nch); ++cc) {
    const uint32_t sq = smem_u32(c.smem + c.ly.q + cc * Q_BYTES);
    const int ch = cc % p.nch;
    for (int e = tid; e < NQ * (D / 8); e += 64 * NCW) {
      const int rr = e & 7, c16 = (e >> 3) & (D / 8 - 1), g8 = e / D;
      const int i = ch * NQ + g8 * 8 + rr;
      const int ic = min(i, nq - 1), hd = ic / p.q, r = ic - hd * p.q;
      const bf16* src = p.Q + b * p.qsb + (h * p.G + hd) * p.qsh + (int64_t)r * p.qss + c16 * 8;
      cp_async16_zfill(sq + (uint32_t)(g8 * QGRP + c16 * 128 + rr * 16), src, i < nq);
    }
  }
  cp_async_arrive_noinc(bar_addr(c.ms->qfull));
}

template <int S>
__device__ void gqa_producer_role(const Ctx& c, const FusedParams& p) {
  Misc& ms = *c.ms;
  const int pt = threadIdx.x - P0;
  int it = 0;
  for (int lev = c.lev_top; lev >= c.lev_end; --lev) {
    if (lev != c.lev_top) wait_or_abort(bar_addr(ms.jready[0]), (uint32_t)(c.lev_top - lev - 1) & 1u, ms, p.status);
    int g0, mc;
    scale_slice(m_total(p, lev), c.rank, c.cs, g0, mc);
    const int ntl = tiles_of(mc);
    const RowSrc src = scale_src(c, p, 0, lev, g0, mc);
    produce<S>(ms, p.status, smem_u32(c.smem), it, 0, ntl, src, pt);  // pass 1
    it += ntl;
    // Pass 2: the same rows again, but for the last tiles, which stay in the
    // ring from pass 1.
    const int nre = max(ntl - S, 0);
    produce<S>(ms, p.status, smem_u32(c.smem), it, 0, nre, src, pt);
    it += nre;
  }
  cp_async_wait_all();
}

// Pass 1 of every scale: tile t's logits with the query rows on the lanes
// into TMEM buffer t % 2 (128 columns an M tile); pass 2: with the candidates
// on the lanes into region k % 2, the kept tiles first.
template <int S>
__device__ void gqa_mma_role(const Ctx& c, const FusedParams& p) {
  Misc& ms = *c.ms;
  if (p.stall) wait_or_abort(bar_addr(ms.stallbar), 0u, ms, p.status);
  wait_or_abort(bar_addr(ms.qfull), 0u, ms, p.status);
  fence_proxy_async();
  const uint32_t sq = smem_u32(c.smem + c.ly.q);
  const int nmt = (p.nch + 3) / 4;                // M tiles of 128 query rows
  const uint32_t rcols = 32u * (uint32_t)p.nch;   // columns of a pass 2 region
  const uint32_t bcols = 128u * (uint32_t)nmt;    // columns of a pass 1 buffer
  const int nreg = gqa_regions(p.nch);
  const uint32_t tm2 = c.tmem + gqa_region0(p.nch);
  const bool shared = nmt > 1;                    // the passes share their columns
  const uint32_t idesc1 = idesc_bf16(TM, TM, 0, 0);          // A = query rows, B = candidate rows (both K-major)
  const uint32_t idesc2 = idesc_bf16(TM, 32 * p.nch, 0, 0);  // A = candidate rows, B = the stacked queries
  uint32_t used1 = 0, used2 = 0;  // pass 1 buffers and pass 2 regions filled so far: use i takes buffer i % 2, region i % nreg
  // Buffer use % ring has been read since its use before.
  auto wait_free = [&](const unsigned long long* bar, uint32_t use, uint32_t ring) {
    if (use >= ring) wait_or_abort(bar_addr(bar[use % ring]), (use / ring - 1u) & 1u, ms, p.status);
  };
  // Pass 2's product of the tile in ring slot `slot` into the next region.
  auto pass2 = [&](int slot) {
    const int s = slot % S, r = (int)(used2 % (uint32_t)nreg);
    wait_free(ms.rfree, used2, (uint32_t)nreg);
    ++used2;
    wait_or_abort(bar_addr(ms.full[s]), (uint32_t)(slot / S) & 1u, ms, p.status);
    fence_proxy_async();
    if (!aborted(ms)) {
      tc_fence_after();
      const uint32_t st = smem_u32(c.smem) + s * TILE_BYTES;
      // One MMA per K step over every query chunk at once (N = 32 nch: the
      // chunks' 8-row groups follow each other at the same stride).
#pragma unroll
      for (int h = 0; h < HALVES; ++h)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16(tm2 + (uint32_t)r * rcols, smem_desc_sw128(st + h * HALF_BYTES + kk * 32, 16, 1024),
                   smem_desc(sq + (4 * h + kk) * 256, 128, QGRP), idesc2, (h | kk) != 0);
    }
    mma_commit(bar_addr(ms.empty[s]));
    mma_commit(bar_addr(ms.rdone[r]));
  };
  // Every read of the last `ring` uses is done.
  auto wait_all_free = [&](const unsigned long long* bar, uint32_t used, uint32_t ring) {
    for (uint32_t i = used < ring ? 0u : used - ring; i < used; ++i)
      wait_or_abort(bar_addr(bar[i % ring]), (i / ring) & 1u, ms, p.status);
  };
  int it = 0;
  for (int lev = c.lev_top; lev >= c.lev_end; --lev) {
    int g0, mc;
    scale_slice(m_total(p, lev), c.rank, c.cs, g0, mc);
    const int ntl = tiles_of(mc), nkeep = min(ntl, S), nre = ntl - nkeep;
    // Shared columns change hands between the passes: every read of the other
    // pass is done first.
    if (shared) wait_all_free(ms.rfree, used2, (uint32_t)nreg);
#pragma unroll 1
    for (int t = 0; t < ntl; ++t) {
      const int r = (int)(used1 & 1u), slot = it + t, s = slot % S;
      wait_free(ms.p1free, used1, 2u);
      ++used1;
      wait_or_abort(bar_addr(ms.full[s]), (uint32_t)(slot / S) & 1u, ms, p.status);
      fence_proxy_async();
      if (!aborted(ms)) {
        tc_fence_after();
        const uint32_t st = smem_u32(c.smem) + s * TILE_BYTES;
        // Query rows past the stacked block (up to the M tile's 128) are
        // whatever follows it in shared memory; nothing reads their rows.
#pragma unroll 1
        for (int m = 0; m < nmt; ++m)
#pragma unroll
          for (int h = 0; h < HALVES; ++h)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_bf16(c.tmem + (uint32_t)r * bcols + 128u * (uint32_t)m,
                       smem_desc(sq + (uint32_t)m * 16u * QGRP + (4 * h + kk) * 256, 128, QGRP),
                       smem_desc_sw128(st + h * HALF_BYTES + kk * 32, 16, 1024), idesc1, (h | kk) != 0);
      }
      if (t < nre) mma_commit(bar_addr(ms.empty[s]));
      mma_commit(bar_addr(ms.p1done[r]));
    }
    if (shared) wait_all_free(ms.p1free, used1, 2u);
    // The kept tiles (slots it + nre ..), then the streamed ones (it + ntl ..).
#pragma unroll 1
    for (int k = 0; k < ntl; ++k) pass2(k < nkeep ? it + nre + k : it + ntl + k - nkeep);
    it += ntl + nre;
  }
  mma_commit(bar_addr(ms.drainbar));
  (void)mbar_wait_bounded(bar_addr(ms.drainbar), 0u, kDefaultWaitLimit);
}

template <int S>
__device__ void gqa_compute_role(const Ctx& c, const FusedParams& p, const GqaLayout gl) {
  Misc& ms = *c.ms;
  constexpr int TN = 32 * unit_warps<true>();
  const int tid = ctid<true>(), lane = tid & 31, warp = tid >> 5, wg = tid >> 7, qd = warp & 3, row = tid & (TM - 1);
  const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
  const int nch = p.nch, nqp = 32 * nch, nq = p.G * p.q;
  const uint32_t nreg = (uint32_t)gqa_regions(nch);
  uint32_t treg = 0;   // the TMEM region that pass 2 reads
  const uint32_t sc_a = smem_u32(c.smem + gl.sc);
  float2* wst = reinterpret_cast<float2*>(c.smem + gl.wst);
  float2* xst = reinterpret_cast<float2*>(c.smem + gl.xst);
  float* cvec = reinterpret_cast<float*>(c.smem + gl.cvec);  // -c_i
  const uint32_t ncvec_a = smem_u32(cvec);
  const float sl2 = p.scale_log2;
  const int u = c.u0;
  int64_t sets_off = 0;
  uint32_t used = 0;   // tiles of the scales before: the uses of pass 1's buffers and of pass 2's regions
  const bool two = nch > 4;  // two M tiles of query rows
  const int copies = gqa_copies(nch);
  const f32x2 s2 = pk2(sl2, sl2);
  // body(ra, ch) for every query chunk of the tile in the region.
  auto for_chunks = [&](auto&& body) {
#pragma unroll 1
    for (int ch = 0; ch < nch; ++ch) {
      uint32_t ra[32];
      tmem_ld32_issue(treg + 32u * ch + lane_base, ra);
      tmem_wait_ld();
      body(ra, ch);
    }
  };
#pragma unroll 1
  for (int lev = c.lev_top; lev >= c.lev_end; --lev) {
    const uint32_t ph = (uint32_t)(c.lev_top - lev) & 1u;
    const int m = m_total(p, lev);
    int g0, mc;
    scale_slice(m, c.rank, c.cs, g0, mc);
    const int ntl = tiles_of(mc);
    const int kb = p.keep[lev];
    int32_t* J = unit_J(c, p, 0, lev);
    const uint32_t keys_a = smem_u32(J);

    // Pass 1: this thread's query row over the tile's candidates, 32 columns at
    // a time.
    const int ncol = TM / (two ? 1 : copies);            // this thread's columns of a tile:
    const int ccol = two ? 0 : row / nqp * ncol;           // from ccol on
    float rmax = -INFINITY;  // the row's stabiliser (log2 units)
    f32x2 rsum = pk2(0.f, 0.f);
#pragma unroll 1
    for (int t = two ? 0 : (int)(((uint32_t)wg - used) & 1u); t < ntl; t += two ? 1 : 2) {
      const uint32_t use = used + (uint32_t)t;
      const int b = (int)(use & 1u);
      wait_or_abort(bar_addr(ms.p1done[b]), (use >> 1) & 1u, ms, p.status);
      tc_fence_after();
      const uint32_t tc = c.tmem + lane_base + (two ? 256u * (uint32_t)b + 128u * (uint32_t)wg : 128u * (uint32_t)b);
      const int nv = min(mc - t * TM, TM);  // candidates of the tile
#pragma unroll 1
      for (int c0 = ccol; c0 < min(nv, ccol + ncol); c0 += 32) {
        uint32_t ra[32];
        tmem_ld32_issue(tc + (uint32_t)c0, ra);
        tmem_wait_ld();
        if (nv - c0 < 32) {
#pragma unroll
          for (int i = 0; i < 32; ++i) ra[i] = i < nv - c0 ? ra[i] : __float_as_uint(-INFINITY);
        }
        float vm = -INFINITY;
#pragma unroll
        for (int i = 0; i < 32; i += 2) vm = fmax3(vm, __uint_as_float(ra[i]), __uint_as_float(ra[i + 1]));
        const float xm = vm * sl2;
        if (xm > rmax + kRaise) {  // also the first columns (rmax = -inf)
          const float f = ex2(rmax - xm);
          rsum = mul2(rsum, pk2(f, f));
          rmax = xm;
        }
        const float nm = rmax > -INFINITY ? -rmax : 0.f;
        const f32x2 nm2 = pk2(nm, nm);
        f32x2 z[2] = {pk2(0.f, 0.f), pk2(0.f, 0.f)};
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float2 x = up2(fma2(pk2(__uint_as_float(ra[2 * k]), __uint_as_float(ra[2 * k + 1])), s2, nm2));
          z[k & 1] = add2(z[k & 1], pk2(ex2(x.x), ex2(x.y)));
        }
        rsum = add2(rsum, add2(z[0], z[1]));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_addr(ms.p1free[b]));
    }
    // The CTA's (M, S) per query row, sent to every cluster CTA.
    {
      const float2 rs2 = up2(rsum);
      float2 st = make_float2(rmax, rs2.x + rs2.y);
      if (!two) {
        wst[tid] = st;
        csync<true>();
        // Query row `tid` from both warpgroups and every copy of the block.
        if (tid < nqp) {
          st = wst[tid];
#pragma unroll 1
          for (int e = 1; e < 2 * copies; ++e) st = merge_ms(st, wst[(e & 1) * TM + (e >> 1) * nqp + tid]);
        }
      }
      const int col = tid;  // (two M tiles: warpgroup w's row is query row 128 w + row)
      const bool own = col < nqp;
      const uint32_t xbar = bar_addr(ms.xbar[0]);
      const uint32_t nr = aborted(ms) || !own ? 0u : c.cs;  // after a wait gave up, nothing goes to the cluster
      const uint32_t dst = smem_u32(&xst[c.rank * nqp + (own ? col : 0)]);
#pragma unroll 1
      for (uint32_t r = 0; r < nr; ++r)
        st_async_v2(map_rank(dst, r), __float_as_uint(st.x), __float_as_uint(st.y), map_rank(xbar, r));
    }
    wait_cluster_or_abort(bar_addr(ms.xbar[0]), ph, ms, p.status);
    if (tid == 0 && lev > c.lev_end && !aborted(ms))
      mbar_arrive_expect_tx(bar_addr(ms.xbar[0]), c.cs * (uint32_t)nqp * 8u);
#pragma unroll 1
    for (int col = tid; col < nqp; col += TN) {
      float2 a = make_float2(-INFINITY, 0.f);
#pragma unroll 1
      for (uint32_t r = 0; r < c.cs; ++r) a = merge_ms(a, xst[r * nqp + col]);
      cvec[col] = col < nq ? -(a.x + lg2(a.y)) : -INFINITY;  // -c_i; padded rows weigh 0
    }
    csync<true>();

    // Pass 2: each row's ranking key over every stacked query row.
    float kmin = INFINITY, kmax = -INFINITY;
    const uint32_t kbar = bar_addr(ms.kbar[0]);
    const uint32_t nr = aborted(ms) ? 0u : c.cs;
    const int nkeep = min(ntl, S), nre = ntl - nkeep;
#pragma unroll 1
    for (int k = (int)(((uint32_t)wg - used) & 1u); k < ntl; k += 2) {
      const int t = k < nkeep ? nre + k : k - nkeep;
      const uint32_t use = used + (uint32_t)k, reg = use % nreg;
      wait_or_abort(bar_addr(ms.rdone[reg]), (use / nreg) & 1u, ms, p.status);
      tc_fence_after();
      treg = c.tmem + gqa_region0(nch) + reg * 32u * (uint32_t)nch;
      // Every exponent l sl2 - c_i is at most 0 (c_i is the log of a sum that
      // holds the row's own term), so the sum is taken unshifted; a row whose
      // sum is tiny (below 2^-96, where flushed terms could matter) is taken
      // again shifted by its largest exponent (the warp together).
      float rm = 0.f, rs = 0.f;
      f32x2 z[2] = {pk2(0.f, 0.f), pk2(0.f, 0.f)};
      for_chunks([&](const uint32_t (&ra)[32], int ch) {
#pragma unroll
        for (int k4 = 0; k4 < 8; ++k4) {
          const uint4 cv = lds_v4(ncvec_a + 16u * (uint32_t)(8 * ch + k4));
          const float2 x = up2(fma2(pk2(__uint_as_float(ra[4 * k4]), __uint_as_float(ra[4 * k4 + 1])), s2,
                                    pk2(__uint_as_float(cv.x), __uint_as_float(cv.y))));
          const float2 y = up2(fma2(pk2(__uint_as_float(ra[4 * k4 + 2]), __uint_as_float(ra[4 * k4 + 3])), s2,
                                    pk2(__uint_as_float(cv.z), __uint_as_float(cv.w))));
          z[0] = add2(z[0], pk2(ex2(x.x), ex2(x.y)));
          z[1] = add2(z[1], pk2(ex2(y.x), ex2(y.y)));
        }
      });
      {
        const float2 zz = up2(add2(z[0], z[1]));
        rs = zz.x + zz.y;
      }
      if (__any_sync(0xffffffffu, rs < 0x1p-96f && t * TM + row < mc)) {
        float mxr = -INFINITY;
        for_chunks([&](const uint32_t (&ra)[32], int ch) {
#pragma unroll
          for (int k4 = 0; k4 < 8; ++k4) {
            const uint4 cv = lds_v4(ncvec_a + 16u * (uint32_t)(8 * ch + k4));
            mxr = fmaxf(mxr, fmax3(fmaf(__uint_as_float(ra[4 * k4]), sl2, __uint_as_float(cv.x)),
                                   fmaf(__uint_as_float(ra[4 * k4 + 1]), sl2, __uint_as_float(cv.y)),
                                   fmaxf(fmaf(__uint_as_float(ra[4 * k4 + 2]), sl2, __uint_as_float(cv.z)),
                                         fmaf(__uint_as_float(ra[4 * k4 + 3]), sl2, __uint_as_float(cv.w)))));
          }
        });
        float z2 = 0.f;
        for_chunks([&](const uint32_t (&ra)[32], int ch) {
#pragma unroll
          for (int k4 = 0; k4 < 8; ++k4) {
            const uint4 cv = lds_v4(ncvec_a + 16u * (uint32_t)(8 * ch + k4));
            z2 += ex2(fmaf(__uint_as_float(ra[4 * k4]), sl2, __uint_as_float(cv.x)) - mxr);
            z2 += ex2(fmaf(__uint_as_float(ra[4 * k4 + 1]), sl2, __uint_as_float(cv.y)) - mxr);
            z2 += ex2(fmaf(__uint_as_float(ra[4 * k4 + 2]), sl2, __uint_as_float(cv.z)) - mxr);
            z2 += ex2(fmaf(__uint_as_float(ra[4 * k4 + 3]), sl2, __uint_as_float(cv.w)) - mxr);
          }
        });
        if (rs < 0x1p-96f) {
          rm = mxr;
          rs = z2;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_addr(ms.rfree[reg]));
      const int j = t * TM + row;
      if (j < mc) {
        const float key = fmaxf(rm + lg2(rs), -INFINITY);  // (a row of -inf logits: see pass_keys)
        kmin = fminf(kmin, key);
        kmax = fmaxf(kmax, key);
        const uint32_t dst = keys_a + 4u * (uint32_t)(g0 + j);
#pragma unroll 1
        for (uint32_t r = 0; r < nr; ++r) st_async_b32(map_rank(dst, r), __float_as_uint(key), map_rank(kbar, r));
      }
    }
    kmin = warp_min_f32(kmin);
    kmax = warp_max_f32(kmax);
    if (lane == 0) {
      const uint32_t dst = smem_u32(&wslots<true>(ms, 0, warp).kmm[c.rank][warp & 3]);
#pragma unroll 1
      for (uint32_t r = 0; r < nr; ++r)
        st_async_v2(map_rank(dst, r), __float_as_uint(kmin), __float_as_uint(kmax), map_rank(kbar, r));
    }
    wait_cluster_or_abort(kbar, ph, ms, p.status);
    float lo, hi;
    {
      constexpr int NW = unit_warps<true>();
      float2 mm = make_float2(INFINITY, -INFINITY);
#pragma unroll 1
      for (int e = lane; e < (int)c.cs * NW; e += 32) {  // entry (CTA e / NW, warp e % NW)
        const int w = e % NW;
        const uint2 v = lds_v2(smem_u32(&wslots<true>(ms, 0, w).kmm[e / NW][w & 3]));
        mm = make_float2(fminf(mm.x, __uint_as_float(v.x)), fmaxf(mm.y, __uint_as_float(v.y)));
      }
      lo = warp_min_f32(mm.x);
      hi = warp_max_f32(mm.y);
    }
    used += (uint32_t)ntl;
    // Eq. 9: Top-K (the same result in every CTA of the cluster).
    select_topk<true>(keys_a, m, kb, smem_u32(unit_J(c, p, 0, lev + 1)), lev == p.L, sc_a, lo, hi);
    if (tid == 0) {
      if (lev > c.lev_end && !aborted(ms))
        mbar_arrive_expect_tx(kbar, 4u * (uint32_t)m_total(p, lev - 1) + c.cs * unit_warps<true>() * 8u);
      mbar_arrive(bar_addr(ms.jready[0]));
    }
    if (c.rank == 0) {
      int32_t* ls = p.level_sets ? p.level_sets + (int64_t)u * p.sets_stride + sets_off : nullptr;
      if (lev >= 1 && ls) {
#pragma unroll 1
        for (int i = tid; i < kb; i += TN) ls[i] = J[i];
      }
      if (lev == c.lev_end) {
        // mu^0: the children of J^1, or the trimmed level-0 selection.
        const int kk = p.keep[0];
        int32_t* out = p.idx + (int64_t)u * kk;
        int32_t* ls0 = ls ? ls + (lev >= 1 ? kb : 0) : nullptr;
#pragma unroll 1
        for (int t = tid; t < kk; t += TN) {
          const int tok = p.trim ? J[t] : 2 * J[t >> 1] + (t & 1);
          out[t] = tok;
          if (ls0) ls0[t] = tok;
        }
      }
    }
    if (lev >= 1) sets_off += kb;
  }
}

template <int S>
__global__ void __launch_bounds__(NT, 1) wf_gqa_filter_kernel(const __grid_constant__ FusedParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const GqaLayout gl = gqa_layout(S, p.nch, (int)cluster_size(), p.cmax, p.kmax);
  Ctx c;
  c.smem = smem;
  c.ly.q = gl.q;
  c.ly.p = gl.sc;
  c.ly.misc = gl.misc;
  c.ly.buf = gl.buf;
  c.ly.bufw = gl.bufw;
  c.ly.total = gl.total;
  c.ms = reinterpret_cast<Misc*>(smem + gl.misc);
  Misc& ms = *c.ms;
  c.rank = cluster_rank();
  c.cs = cluster_size();
  c.u0 = (int)cluster_id_x();
  c.np = 1;
  c.lev_top = p.L;
  c.lev_end = p.trim ? 0 : 1;
  c.stages = S;
  const int tid = threadIdx.x, warp = tid >> 5;

  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(bar_addr(ms.full[s]), NPT);
      mbar_init(bar_addr(ms.empty[s]), 1);
    }
    mbar_init(bar_addr(ms.jready[0]), 1);
    mbar_init(bar_addr(ms.xbar[0]), 1);
    mbar_init(bar_addr(ms.kbar[0]), 1);
    for (int r = 0; r < 2; ++r) {
      mbar_init(bar_addr(ms.p1done[r]), 1);
      mbar_init(bar_addr(ms.p1free[r]), p.nch > 4 ? 2 * NCW : NCW);
    }
    for (int r = 0; r < MAXREG; ++r) {
      mbar_init(bar_addr(ms.rdone[r]), 1);
      mbar_init(bar_addr(ms.rfree[r]), NCW);
    }
    mbar_init(bar_addr(ms.qfull), 64 * NCW);
    mbar_init(bar_addr(ms.stallbar), 1);
    mbar_init(bar_addr(ms.drainbar), 1);
    ms.wait_limit = p.wait_limit;
    ms.abort = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (warp > MMA_WARP) {
    cluster_arrive_relaxed();
    grid_dep_wait();
    gqa_producer_role<S>(c, p);
    cluster_wait();
  } else {
    constexpr int NS = NT - NPT;
    if (tid == 0) {
      mbar_arrive_expect_tx(bar_addr(ms.xbar[0]), c.cs * 32u * (uint32_t)p.nch * 8u);
      mbar_arrive_expect_tx(bar_addr(ms.kbar[0]),
                            4u * (uint32_t)m_total(p, c.lev_top) + c.cs * unit_warps<true>() * 8u);
    }
    if (warp == MMA_WARP) {
      tmem_alloc(smem_u32(&ms.tmem_base), p.tmem_cols);
      tmem_relinquish();
    }
    // The Top-K scratch starts zeroed (histogram, list counter, masks).
    for (int e = tid; e < (int)((sizeof(SelScratch) + 15) / 16); e += NS)
      *reinterpret_cast<uint4*>(smem + gl.sc + 16 * e) = make_uint4(0, 0, 0, 0);
    grid_dep_wait();
    if (warp < MMA_WARP) gqa_load_queries(c, p);
    tc_fence_before();
    named_sync(kSetupSyncId, NS);
    tc_fence_after();
    grid_dep_launch();  // after the barrier that publishes the tensor memory (see Launch)
    c.tmem = ms.tmem_base;
    cluster_sync();  // every CTA's barriers are armed before any remote arrival
    if (warp < MMA_WARP) {
      gqa_compute_role<S>(c, p, gl);
      cp_async_wait_all();  // (query copies still in flight only after a wait gave up)
    } else {
      if ((tid & 31) == 0) gqa_mma_role<S>(c, p);
      __syncwarp();
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  if (warp == MMA_WARP) {
    if (aborted(ms)) {
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 20000ull) {
      }
    }
    tc_fence_after();
    tmem_dealloc(c.tmem, p.tmem_cols);
  }
}
#endif  // !WF_STAGE_CALLS
}  // namespace

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
namespace {

// The kernel instance for a stage count and unit width (one-unit plans with
// long candidate lists run the WIDE instance, whose two warpgroups both serve
// the unit).
typedef void (*FusedKernel)(FusedParams);
constexpr int kStagesMin = D == 64 ? 4 : 3;  // (two units' P terms leave head_dim 64 four stages of 16 KB)
FusedKernel fused_kernel(int stages, bool wide) {
  if (stages == MAXS) return wide ? wf_fused_kernel<MAXS, true> : wf_fused_kernel<MAXS, false>;
  return wide ? wf_fused_kernel<kStagesMin, true> : wf_fused_kernel<kStagesMin, false>;
}

// The kernel's dynamic shared-memory limit, raised once per device and
// instance to the largest size requested so far instead of on every launch.
cudaError_t ensure_smem_limit(int stages, bool wide, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, bool>, size_t> raised;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t& cur = raised[std::make_tuple(dev, stages, wide)];
  if (cur >= smem) return cudaSuccess;
  e = cudaFuncSetAttribute(fused_kernel(stages, wide), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) cur = smem;
  return e;
}

// How many clusters of cs CTAs (with `smem` bytes each) can be resident at
// once on the current device; cached per configuration.
int max_active_clusters(int stages, bool wide, int cs, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, bool, int, size_t>, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const auto key = std::make_tuple(dev, stages, wide, cs, smem);
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)cs, 1, 1);
  cfg.blockDim = dim3(NT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  cudaError_t e;
  e = ensure_smem_limit(stages, wide, smem);  // only ever raised, so a launch's earlier limit still holds
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, fused_kernel(stages, wide), &cfg);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    n = 0;
  }
  cache.emplace(key, n);
  return n;
}

}  // namespace

FusedPlan plan_fused(const wf_tensor& q, const wf_tensor& kv, int levels, const int32_t* keep, int n_g, int num_sms,
                     bool split) {
  FusedPlan fp{};
  fp.ok = false;
  if (kv.dtype != WF_BF16 || kv.head_dim != D || q.seq > NQ || levels > 10) return fp;
  const int U = kv.batch * kv.heads;
  const int n = kv.seq;
  const bool filter = levels > 0;  // else the attention alone, over a list of keep[0] tokens
  const bool trim = !filter || keep[0] < 2 * keep[1];
  int cmax = filter ? n >> levels : 0, kmax = 0;
  for (int l = 0; l <= levels; ++l) kmax = kmax > keep[l] ? kmax : keep[l];
  for (int l = 1; l <= levels; ++l) cmax = cmax > 2 * keep[l] ? cmax : 2 * keep[l];
  if (cmax > kMaxCand || kmax > kMaxCand) return fp;
  const int total = n_g < 0 ? 0 : keep[0] + n_g;  // keys of the attention
  // TMEM columns of one unit's region at cluster size cs: the widest scale
  // slice, or the attention slice plus the O^T accumulator.
  // TMEM tiles of the widest scale slice at cluster size cs.
  auto scale_tiles = [&](int cs) {
    auto slice_tiles = [&](int m) { return (2 * (((m + 1) / 2 + cs - 1) / cs) + TM - 1) / TM; };
    int tmax = filter ? slice_tiles(n >> levels) : 0;
    for (int l = levels; l >= 1; --l) {
      const int t = slice_tiles(2 * keep[l]);
      tmax = tmax > t ? tmax : t;
    }
    return tmax;
  };
  auto unit_cols = [&](int cs) {
    int tmax = scale_tiles(cs);
    const int ta = total > 0 ? ((total + cs - 1) / cs + TM - 1) / TM + 1 : 0;
    tmax = tmax > ta ? tmax : ta;
    return 32 * tmax;
  };
  const size_t kMaxSmem = 227 * 1024;
  // A one-unit plan runs both warpgroups on its unit unless the candidate lists
  // are too short for the halved per-thread work to outweigh the wider barriers
  // (32 heads, head_dim 128, a step: lists of 512 22.0 -> 22.5 us; of 1024 38.5
  // -> 38.4; of 1638 46.7 -> 45.2).  Where outlying keys leave more in the
  // Top-K's boundary bucket than one warpgroup lists at once, whatever the
  // length, both save a second round (47 -> 35 us at 1024).  The one-unit plans of
  // filter and attention calls take the same instance at any size: alternating
  // two costs 5 us of code fetches.
  const bool wide1 = split || D == 64 || cmax >= 1024;
  // For P units per cluster (1, or 2 so that one unit's copies overlap the
  // other's exchanges and Top-K): the largest cluster (any size up to 8)
  // whose grid fits the SMs in one wave, all clusters resident at once, and
  // whose slices fit TMEM; else the smallest one that fits TMEM.
  struct Choice {
    int P, cs, stages;
    size_t smem;
    bool resident;
  };
  auto choose = [&](int P) {
    Choice ch{P, 0, MAXS, 0, false};
    const int clusters = (U + P - 1) / P;
    if (smem_layout(MAXS, P, cmax, kmax, !filter).total > kMaxSmem) ch.stages = kStagesMin;
    ch.smem = smem_layout(ch.stages, P, cmax, kmax, !filter).total;
    if (ch.smem > kMaxSmem) return ch;
    for (int c = MAXCS; c >= 1 && ch.cs == 0; --c)
      if (clusters * c <= num_sms && P * unit_cols(c) <= 512 &&
          clusters <= max_active_clusters(ch.stages, P == 1 && wide1, c, ch.smem))
        ch.cs = c;
    ch.resident = ch.cs > 0;
    for (int c = 1; c <= MAXCS && ch.cs == 0; ++c)
      if (P * unit_cols(c) <= 512) ch.cs = c;
    return ch;
  };
  // Units per SM (P / cs) set each SM's share of the rows: take the smaller.
  // On a tie two units per cluster, so that one's copies run under the other's
  // reductions over the whole chain of a step (64 units x 32K 71.6 -> 68.9 us,
  // 128 units 106 -> 92), but one, on both warpgroups, where the chain is split
  // over launches and there is little to overlap (64 units: filter and
  // attention at 16K 82.3 -> 68.5 us, the db2 step at 32K 217.9 -> 189.0), and
  // where the lists are short (at most 128 KB of rows: 64 units x 2K 26.3 ->
  // 23.6 us, x 8K of head_dim 64 46.1 -> 43.3; 96 units x 8K, 256 KB, 60.4
  // against 63.2).
  const bool one_unit = split || cmax * D <= 1 << 16;
  const Choice c2 = U >= 2 ? choose(2) : Choice{2, 0, MAXS, 0, false};
  const Choice c1 = choose(1);
  Choice best = c2;
  if (c2.cs == 0 || (c1.cs > 0 && c2.cs < 2 * c1.cs + (one_unit ? 1 : 0))) best = c1;
  if (best.cs == 0) return fp;
  const int P = best.P, cs = best.cs, stages = best.stages;
  const size_t smem = best.smem;
  const int clusters = (U + P - 1) / P;
  int ucols = unit_cols(cs);
  // Room for the scale's exponentials beside its logits (the ranking keys
  // then need no exponentials of their own): the widest scale slice twice.
  const int stiles = scale_tiles(cs);
  int ecol = 0;
  const int ecols = ucols > 64 * stiles ? ucols : 64 * stiles;
  if (filter && P * ecols <= 512) {
    ecol = 32 * stiles;
    ucols = ecols;
  }
  int cols = 32;
  while (cols < P * ucols) cols *= 2;
  fp.ok = true;
  fp.cs = cs;
  fp.P = P;
  fp.wide = P == 1 && wide1;
  fp.resident = best.resident;
  fp.full_ring = stages == MAXS;
  fp.stages = stages;
  fp.smem = smem;
  fp.tmem_cols = cols;
  fp.ucols = ucols;
  fp.ecol = ecol;
  fp.cmax = cmax;
  fp.kmax = kmax;
  fp.trim = trim;
  fp.U = U;
  fp.clusters = clusters;
  return fp;
}

cudaError_t launch_fused(const FusedPlan& fp, const void* Q, const wf_tensor& qd, const void* K, const void* V,
                         const wf_tensor& kv, const void* Kg, const void* Vg, const wf_tensor* g,
                         const void* coeffs, int levels, const int32_t* keep, int32_t* idx, int32_t* level_sets,
                         void* O, const wf_tensor& od, int* status, cudaStream_t s, const FusedRange* range) {
  FusedParams p;
  memset(&p, 0, sizeof(p));
  p.Q = static_cast<const bf16*>(Q);
  p.qsb = qd.stride_b; p.qsh = qd.stride_h; p.qss = qd.stride_s;
  p.K = static_cast<const bf16*>(K);
  p.V = static_cast<const bf16*>(V);
  p.ksb = kv.stride_b; p.ksh = kv.stride_h; p.kss = kv.stride_s;
  p.Kg = static_cast<const bf16*>(Kg);
  p.Vg = static_cast<const bf16*>(Vg);
  if (g) { p.gsb = g->stride_b; p.gsh = g->stride_h; p.gss = g->stride_s; }
  p.coeffs = static_cast<const bf16*>(coeffs);
  p.rows_total = (int64_t)kv.seq - ((int64_t)kv.seq >> levels);
  p.O = static_cast<bf16*>(O);
  p.osb = od.stride_b; p.osh = od.stride_h; p.oss = od.stride_s;
  p.idx = idx;
  p.level_sets = level_sets;
  int64_t stride = 0;
  for (int l = 0; l <= levels; ++l) stride += keep[l];
  p.sets_stride = stride;
  p.status = status;
  p.q = qd.seq; p.n = kv.seq; p.ng = g ? g->seq : 0; p.U = fp.U; p.H = kv.heads; p.L = levels;
  p.trim = fp.trim ? 1 : 0;
  p.P = fp.P;
  p.cmax = fp.cmax; p.kmax = fp.kmax;
  p.tmem_cols = (uint32_t)fp.tmem_cols;
  p.ucols = (uint32_t)fp.ucols;
  p.ecol = (uint32_t)fp.ecol;
  const WaitControls wc = wait_controls();
  p.wait_limit = wc.limit;
  p.stall = wc.stall;
  for (int l = 0; l <= levels; ++l) p.keep[l] = keep[l];
  p.scale_log2 = kLog2e / sqrtf((float)D);
  if (range) {
    // A launch below the top scale reads its first scale's rows densely: the
    // producers never wait for the handed-in selection.
    if (range->lev_top < levels && !range->lrows) return cudaErrorInvalidValue;
    p.lev_top = range->lev_top;
    p.lev_bot = range->lev_bot;
    p.final_sel = range->final_sel;
    p.attn = range->attn;
    p.jin = range->jin;
    p.jout = range->jout;
    p.jstride = range->jstride;
    p.sel = range->sel;
    if (range->scale > 0.f) p.scale_log2 = kLog2e * range->scale;
    p.lrows = static_cast<const bf16*>(range->lrows);
    p.lrows_unit = range->lrows_unit;
  } else {
    p.lev_top = levels;
    p.lev_bot = fp.trim ? 0 : 1;
    p.final_sel = 1;
    p.attn = 1;
  }

  cudaError_t e = ensure_smem_limit(fp.stages, fp.wide, fp.smem);
  if (e != cudaSuccess) return e;
  return Launch(dim3((unsigned)(fp.clusters * fp.cs)), NT, fp.smem, s, fp.cs,
                range && range->plain)(fused_kernel(fp.stages, fp.wide), p);
}

#if !WF_STAGE_CALLS
// The grouped filter (wf_gqa_filter_kernel): bf16, at most 256 stacked
// query rows a key head of grouped heads, or of one head with a block of more
// than 32 rows (up to 32 are the fused kernel's), candidate lists within the
// Top-K's 8192.  (32 heads x 16K tokens with blocks of 64: a step took 171 us
// with 20 launches for the filter and takes 73 us with this one.)
// One unit per cluster; the largest cluster of up to 8 CTAs
// whose grid fits the SMs in one wave with every cluster resident.
constexpr int kGqaStages = 3 * 128 / D;  // least stages: beside 256 stacked query rows
typedef void (*GqaKernel)(FusedParams);
GqaKernel gqa_kernel(int stages) {
  return stages == MAXS ? wf_gqa_filter_kernel<MAXS> : wf_gqa_filter_kernel<kGqaStages>;
}
GqaPlan plan_gqa(const wf_tensor& q, const wf_tensor& kv, int levels, const int32_t* keep, int num_sms) {
  GqaPlan gp{};
  gp.ok = false;
  if (kv.dtype != WF_BF16 || kv.head_dim != D || q.dtype != WF_BF16 || kv.heads <= 0 || levels > 10) return gp;
  if (q.heads % kv.heads != 0 || q.batch != kv.batch) return gp;
  const int G = q.heads / kv.heads;
  if ((G == 1 && q.seq <= NQ) || q.seq > kMaxQ || G * q.seq > GQ_MAXCH * NQ) return gp;
  const int U = kv.batch * kv.heads;
  int cmax = kv.seq >> levels, kmax = 0;
  for (int l = 0; l <= levels; ++l) kmax = kmax > keep[l] ? kmax : keep[l];
  for (int l = 1; l <= levels; ++l) cmax = cmax > 2 * keep[l] ? cmax : 2 * keep[l];
  if (cmax > kMaxCand || kmax > kMaxCand) return gp;
  const int nch = (G * q.seq + NQ - 1) / NQ;
  // As many stages as fit: tiles kept in the ring are not streamed again.
  int stages = 0;
  const size_t kMaxSmem = 227 * 1024;
  int cs = 0;
  size_t smem = 0;
  auto layout = [&](int c) {
    stages = MAXS;
    smem = gqa_layout(stages, nch, c, cmax, kmax).total;
    if (smem <= kMaxSmem) return;
    stages = kGqaStages;
    smem = gqa_layout(stages, nch, c, cmax, kmax).total;
  };
  for (int c = MAXCS; c >= 1 && cs == 0; --c) {
    layout(c);
    if (smem > kMaxSmem || U * c > num_sms) continue;
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, size_t>, int> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return gp;
    int n = 0;
    {
      std::lock_guard<std::mutex> lock(mu);
      const auto key = std::make_tuple(dev, stages, c, smem);
      auto it = cache.find(key);
      if (it != cache.end()) {
        n = it->second;
      } else {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)c, 1, 1);
        cfg.blockDim = dim3(NT, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = c;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const GqaKernel k = gqa_kernel(stages);
        cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k), smem);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
        if (e != cudaSuccess) {
          (void)cudaGetLastError();
          n = 0;
        }
        cache.emplace(key, n);
      }
    }
    if (U <= n) cs = c;
  }
  if (cs == 0) {  // more units than one wave holds: single-CTA clusters in several waves
    cs = 1;
    layout(1);
    if (smem > kMaxSmem) return gp;
  }
  gp.trim = keep[0] < 2 * keep[1];
  if (D == 128 && nch == 1 && cs == 1) {
    // One CTA a unit and at most 32 stacked rows, on half-empty M tiles: in a
    // last wave that is nearly empty the kernels per scale, spread over every
    // SM, are faster on long lists (160 units x 16K tokens, one scale, 8 heads x 4
    // rows: 242 us against 192; x 32K, four scales 263 against 247; 8K, three
    // scales 141 against 154).  Both sides in us, fitted to 280 shapes of 80 to
    // 384 units (within 4 % of half of them and 16 % of 95 in 100; the choice is at most
    // 5 % slower than the better side).
    const int lists = levels + (gp.trim ? 1 : 0), waves = (U + num_sms - 1) / num_sms;
    float cands = (float)(kv.seq >> levels);
    for (int l = levels; l > levels + 1 - lists; --l) cands += 2.f * (float)keep[l];
    const float one = 6.1f * (float)lists + 0.0147f * (float)waves * cands;
    const float rows32 = (float)(G * q.seq) / 32.f;
    const float per_scale =
        20.7f * (float)lists + 1e-3f * cands * ((float)U * (0.112f + 0.011f * rows32) + 0.6f);
    if (one > per_scale) return gp;
  }
  const int cols = 512;  // both passes' columns
  gp.ok = true;
  gp.cs = cs;
  gp.stages = stages;
  gp.smem = smem;
  gp.tmem_cols = cols;
  gp.nch = nch;
  gp.G = G;
  gp.cmax = cmax;
  gp.kmax = kmax;
  gp.U = U;
  return gp;
}

cudaError_t launch_gqa_filter(const GqaPlan& gp, const void* Q, const wf_tensor& qd, const void* K,
                              const wf_tensor& kv, const void* coeffs, int levels, const int32_t* keep, int32_t* idx,
                              int32_t* level_sets, int* status, cudaStream_t s) {
  FusedParams p;
  memset(&p, 0, sizeof(p));
  p.Q = static_cast<const bf16*>(Q);
  p.qsb = qd.stride_b; p.qsh = qd.stride_h; p.qss = qd.stride_s;
  p.K = static_cast<const bf16*>(K);
  p.ksb = kv.stride_b; p.ksh = kv.stride_h; p.kss = kv.stride_s;
  p.coeffs = static_cast<const bf16*>(coeffs);
  p.rows_total = (int64_t)kv.seq - ((int64_t)kv.seq >> levels);
  p.idx = idx;
  p.level_sets = level_sets;
  int64_t stride = 0;
  for (int l = 0; l <= levels; ++l) stride += keep[l];
  p.sets_stride = stride;
  p.status = status;
  p.q = qd.seq; p.n = kv.seq; p.U = gp.U; p.H = kv.heads; p.L = levels;
  p.trim = gp.trim ? 1 : 0;
  p.P = 1;
  p.cmax = gp.cmax; p.kmax = gp.kmax;
  p.tmem_cols = (uint32_t)gp.tmem_cols;
  const WaitControls wc = wait_controls();
  p.wait_limit = wc.limit;
  p.stall = wc.stall;
  for (int l = 0; l <= levels; ++l) p.keep[l] = keep[l];
  p.scale_log2 = kLog2e / sqrtf((float)D);
  p.lev_top = levels;
  p.lev_bot = gp.trim ? 0 : 1;
  p.final_sel = 1;
  p.G = gp.G;
  p.nch = gp.nch;
  const GqaKernel k = gqa_kernel(gp.stages);
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k), gp.smem);
  if (e != cudaSuccess) return e;
  return Launch(dim3((unsigned)(gp.U * gp.cs)), NT, gp.smem, s, gp.cs)(k, p);
}

cudaError_t launch_literal_fused(const FusedPlan& fp, const FilterPlan& fl, const void* Q, const wf_tensor& qd,
                                 const void* top, const void* K, const void* V, const wf_tensor& kv, const void* Kg,
                                 const void* Vg, const wf_tensor* g, int wavelet, int32_t* idx, int32_t* level_sets,
                                 void* O, const wf_tensor* od, void* ws, int* status, cudaStream_t s) {
  char* base = static_cast<char*>(ws);
  int32_t* cur = reinterpret_cast<int32_t*>(base + fl.off_cand_a);  // candidates of the scale being filtered
  int32_t* nxt = reinterpret_cast<int32_t*>(base + fl.off_cand_b);
  void* arows = base + align_up(fl.total, 256);
  const int L = fl.L;
  int m = fl.n >> L;
  cudaError_t e;
  for (int l = L; l >= 1; --l) {
    // Scale l's rows: the whole prompt's scale-L rows at the top, else the
    // transform of the candidates' gathered blocks, in candidate order.
    if (l < L && (e = launch_wavelet_approx(K, kv, cur, fl.cmax, m, l, wavelet, arows, (int64_t)fl.cmax * D,
                                            s)) != cudaSuccess)
      return e;
    FusedRange r{};
    r.plain = l == L;  // every launch after the first follows one of this pipeline's own
    r.lev_top = l;
    r.lev_bot = (l == 1 && fl.trim) ? 0 : l;
    r.final_sel = l == 1;
    r.attn = l == 1 && O != nullptr;
    r.jin = cur;
    r.jout = nxt;
    r.jstride = fl.cmax;
    r.lrows = l == L ? top : arows;
    r.lrows_unit = l == L ? (int64_t)m * D : (int64_t)fl.cmax * D;
    if ((e = WF_HD::launch_fused(fp, Q, qd, K, V, kv, Kg, Vg, g, nullptr, L, fl.keep, idx, level_sets, O, od ? *od : qd,
                          status, s, &r)) != cudaSuccess)
      return e;
    m = 2 * fl.keep[l];
    int32_t* t = cur;
    cur = nxt;
    nxt = t;
  }
  return cudaSuccess;
}
#endif  // !WF_STAGE_CALLS

}  // namespace WF_HD
}  // namespace wf
