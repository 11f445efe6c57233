// Multi-level Haar DWT of the cached keys (Eq. 5 recursion, Eq. 6).
//
// One thread owns one 16-byte column slice (4 fp32 / 8 bf16 channels) of one
// aligned block of 2^L tokens.  It streams the block in chunks of 2^LC tokens
// (LC = min(L, 3)): a chunk's levels 1..LC are evaluated in registers, and the
// chunk's level-LC value feeds a binary-counter carry for levels LC+1..L, so
// every key row is read once and every pyramid row written once.  Lanes that
// share a row are adjacent, so each warp reads and writes whole 256-byte row
// segments.  The arithmetic is the fp32 add-then-multiply of wf_dwt_build
// (no fused multiply-add: __fadd_rn / __fmul_rn).
//
// The update mode (wf_cache_update) runs the same cascade over only the blocks
// that contain token positions [pos, pos + count): a thread takes its slice of
// a new row from the update buffer and writes it into the cache, and takes
// every other row of the block from the cache, so the coefficients it writes
// equal those of a full build of the updated keys.  The value rows are copied
// by CTAs of their own.  An update moves a few MB over a few thousand threads,
// so it is bound by its chain of memory latencies: every load of a chunk is
// issued before the first store (the row's source is chosen as an address, not
// by a branch around the load), the next chunk's loads before this one's
// arithmetic, and CTAs are small, to use more SMs (32 rows of 64 units at 32K,
// four scales: 9.3 -> 3.2 us a launch).  Large updates are bound by HBM, and a
// value CTA then copies up to eight slices a thread: with one, starting the CTAs took
// longer than the copies (16K rows of 64 units of 128 fp32 channels, four
// scales: 786 -> 375 us).
#include <algorithm>

#include "wf_internal.cuh"

namespace wf {
namespace {

// Rows [pos, pos + count) of the cache, replaced by an update buffer.
template <typename T>
struct Update {
  const T* Kn;  // [B, H, count, D] new key rows
  const T* Vn;  // new value rows, or null
  T* V;         // value cache (null with Vn)
  int64_t nsb, nsh, nss;  // strides of the update buffers
  int64_t pos, count;
  int64_t blk0;           // first block of the unit that holds a new row
  uint32_t vctas;         // CTAs of a unit's value rows
  int vper;               // 16-byte slices a thread of theirs copies, at most kMaxSlices
};

constexpr int kBuildThreads = 256, kUpdateThreads = 64, kMaxSlices = 8;

template <typename T, int L, bool UPDATE>
__global__ void __launch_bounds__(UPDATE ? kUpdateThreads : kBuildThreads) dwt_kernel(const T* K_in, T* K_out, int64_t sb, int64_t sh,
                                                  int64_t ss, int H, int n, int D, T* __restrict__ coeffs,
                                                  int64_t rows_total, int64_t nblk, int64_t total_items,
                                                  int64_t key_ctas, Update<T> up) {
  constexpr int VEC = Vec<T>::N;
  constexpr int LC = L < 3 ? L : 3;
  constexpr int CH = 1 << LC;
  constexpr int NP = L > LC ? L - LC : 1;
  const int lanes = D / VEC;
  if (UPDATE && blockIdx.x >= key_ctas) {
    // 16-byte slices of a unit's new value rows: every load before the first store.
    const uint32_t vb = blockIdx.x - (uint32_t)key_ctas, u = vb / up.vctas;
    const int64_t bb = u / (uint32_t)H, hh = u % (uint32_t)H;
    const T* src = up.Vn + bb * up.nsb + hh * up.nsh;
    T* dst = up.V + bb * sb + hh * sh + up.pos * ss;
    const int64_t e0 = (int64_t)(vb - u * up.vctas) * (kUpdateThreads * up.vper) + threadIdx.x;
    const int shift = __ffs(lanes) - 1;  // (8, 16 or 32 slices a row)
    auto here = [&](int i) { return i < up.vper && (e0 + i * kUpdateThreads) >> shift < up.count; };
    auto at = [&](int i, int64_t row_stride) {
      const int64_t e = e0 + i * kUpdateThreads;
      return (e >> shift) * row_stride + (e & (lanes - 1)) * VEC;
    };
    uint4 w[kMaxSlices];
#pragma unroll
    for (int i = 0; i < kMaxSlices; ++i)
      if (here(i)) w[i] = __ldg(reinterpret_cast<const uint4*>(src + at(i, up.nss)));
#pragma unroll
    for (int i = 0; i < kMaxSlices; ++i)
      if (here(i)) *reinterpret_cast<uint4*>(dst + at(i, ss)) = w[i];
    return;
  }
  const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (item >= total_items) return;
  const int lane = (int)(item % lanes);
  const int64_t rest = item / lanes;
  const int64_t blk = rest % nblk + (UPDATE ? up.blk0 : 0);
  const int64_t u = rest / nblk;
  const int64_t bb = u / H, hh = u % H;
  const int64_t tok0 = blk << L;
  const T* src = K_in + bb * sb + hh * sh + tok0 * ss + (int64_t)lane * VEC;
  T* dst = coeffs + u * rows_total * D + (int64_t)lane * VEC;
  const float c = 0.70710678118654752440f;  // fl32(1/sqrt 2)

  float pend[NP][VEC];
  // Update mode: the chunk's rows as loaded, and which of them are new.
  uint4 raw[CH];
  auto is_new = [&](int64_t tok) { return tok >= up.pos && tok < up.pos + up.count; };
  auto fetch = [&](int ch) {
#pragma unroll
    for (int t = 0; t < CH; ++t) {
      const int64_t tok = tok0 + ch * CH + t;
      const T* row = is_new(tok) ? up.Kn + bb * up.nsb + hh * up.nsh + (tok - up.pos) * up.nss + (int64_t)lane * VEC
                                 : src + (int64_t)(ch * CH + t) * ss;
      raw[t] = __ldg(reinterpret_cast<const uint4*>(row));
    }
  };
  if (UPDATE) fetch(0);
#pragma unroll 1
  for (int ch = 0; ch < (1 << (L - LC)); ++ch) {
    float v[CH][VEC];
    if (UPDATE) {
#pragma unroll
      for (int t = 0; t < CH; ++t) widen_vec(src, raw[t], v[t]);
      uint4 own[CH];
#pragma unroll
      for (int t = 0; t < CH; ++t) own[t] = raw[t];
      if (ch + 1 < (1 << (L - LC))) fetch(ch + 1);
#pragma unroll
      for (int t = 0; t < CH; ++t) {
        const int64_t tok = tok0 + ch * CH + t;
        if (is_new(tok))
          *reinterpret_cast<uint4*>(K_out + bb * sb + hh * sh + tok * ss + (int64_t)lane * VEC) = own[t];
      }
    } else {
#pragma unroll
      for (int t = 0; t < CH; ++t) ld_vec(src + (int64_t)(ch * CH + t) * ss, v[t]);
    }
    const int64_t gc = (blk << (L - LC)) + ch;  // chunk index within the unit
#pragma unroll
    for (int lev = 1; lev <= LC; ++lev) {
      const int cnt = CH >> lev;
      const int64_t off = (int64_t)n - ((int64_t)n >> (lev - 1));
#pragma unroll
      for (int j = 0; j < cnt; ++j) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) v[j][e] = __fmul_rn(__fadd_rn(v[2 * j][e], v[2 * j + 1][e]), c);
        st_vec(dst + (off + gc * cnt + j) * D, v[j]);
      }
    }
    if (L > LC) {
      float x[VEC];
#pragma unroll
      for (int e = 0; e < VEC; ++e) x[e] = v[0][e];
#pragma unroll
      for (int lev = LC + 1; lev <= L; ++lev) {
        const int bit = lev - LC - 1;
        if (((ch >> bit) & 1) == 0) {
#pragma unroll
          for (int e = 0; e < VEC; ++e) pend[bit][e] = x[e];
          break;
        }
#pragma unroll
        for (int e = 0; e < VEC; ++e) x[e] = __fmul_rn(__fadd_rn(pend[bit][e], x[e]), c);
        const int64_t off = (int64_t)n - ((int64_t)n >> (lev - 1));
        st_vec(dst + (off + (gc >> (lev - LC))) * D, x);
      }
    }
  }
}

// Full build (up.count == 0) or the update of the blocks holding the new rows.
template <typename T, int L>
cudaError_t run(const void* K, void* K_out, const wf_tensor& kv, void* coeffs, const Update<T>& up, cudaStream_t s) {
  const int U = kv.batch * kv.heads;
  const int lanes = kv.head_dim / Vec<T>::N;
  const int64_t rows_total = (int64_t)kv.seq - ((int64_t)kv.seq >> L);
  const int64_t nblk = up.count > 0 ? ((up.pos + up.count - 1) >> L) - (up.pos >> L) + 1 : ((int64_t)kv.seq >> L);
  const int64_t items = (int64_t)U * nblk * lanes;
  const int threads = up.count > 0 ? kUpdateThreads : kBuildThreads;
  const int64_t blocks = (items + threads - 1) / threads;
  if (up.count > 0) {
    Update<T> u2 = up;
    u2.blk0 = up.pos >> L;
    // Value rows: as many slices a thread as leave the SMs eight CTAs each.
    const int64_t slices = up.Vn ? up.count * lanes : 0;
    u2.vper = 1;
    if (U * slices > 8 * 100 * threads) {
      const int sms = sm_count();
      if (sms > 0) u2.vper = (int)std::clamp<int64_t>(U * slices / (8 * (int64_t)sms * threads), 1, kMaxSlices);
    }
    u2.vctas = (uint32_t)((slices + threads * u2.vper - 1) / (threads * u2.vper));
    const int64_t vblocks = (int64_t)U * u2.vctas;
    dwt_kernel<T, L, true><<<(unsigned)(blocks + vblocks), threads, 0, s>>>(
        static_cast<const T*>(K), static_cast<T*>(K_out), kv.stride_b, kv.stride_h, kv.stride_s, kv.heads, kv.seq,
        kv.head_dim, static_cast<T*>(coeffs), rows_total, nblk, items, blocks, u2);
  } else {
    dwt_kernel<T, L, false><<<(unsigned)blocks, threads, 0, s>>>(
        static_cast<const T*>(K), nullptr, kv.stride_b, kv.stride_h, kv.stride_s, kv.heads, kv.seq, kv.head_dim,
        static_cast<T*>(coeffs), rows_total, nblk, items, blocks, up);
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t dispatch(const void* K, void* K_out, const wf_tensor& kv, int levels, void* coeffs, const Update<T>& up,
                     cudaStream_t s) {
  switch (levels) {
    case 1: return run<T, 1>(K, K_out, kv, coeffs, up, s);
    case 2: return run<T, 2>(K, K_out, kv, coeffs, up, s);
    case 3: return run<T, 3>(K, K_out, kv, coeffs, up, s);
    case 4: return run<T, 4>(K, K_out, kv, coeffs, up, s);
    case 5: return run<T, 5>(K, K_out, kv, coeffs, up, s);
    case 6: return run<T, 6>(K, K_out, kv, coeffs, up, s);
    case 7: return run<T, 7>(K, K_out, kv, coeffs, up, s);
    case 8: return run<T, 8>(K, K_out, kv, coeffs, up, s);
    case 9: return run<T, 9>(K, K_out, kv, coeffs, up, s);
    case 10: return run<T, 10>(K, K_out, kv, coeffs, up, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
Update<T> make_update(const void* Kn, const void* Vn, void* V, const wf_tensor* nt, int64_t pos) {
  Update<T> up{};
  if (nt) {
    up.Kn = static_cast<const T*>(Kn);
    up.Vn = static_cast<const T*>(Vn);
    up.V = static_cast<T*>(V);
    up.nsb = nt->stride_b;
    up.nsh = nt->stride_h;
    up.nss = nt->stride_s;
    up.pos = pos;
    up.count = nt->seq;
  }
  return up;
}

}  // namespace

cudaError_t launch_dwt(const void* K, const wf_tensor& kv, int levels, void* coeffs, cudaStream_t s) {
  if (kv.dtype == WF_BF16) return dispatch<bf16>(K, nullptr, kv, levels, coeffs, make_update<bf16>(0, 0, 0, 0, 0), s);
  return dispatch<float>(K, nullptr, kv, levels, coeffs, make_update<float>(0, 0, 0, 0, 0), s);
}

cudaError_t launch_cache_update(const void* Kn, const void* Vn, const wf_tensor& nt, void* K, void* V,
                                const wf_tensor& kv, int64_t pos, int levels, void* coeffs, cudaStream_t s) {
  if (kv.dtype == WF_BF16)
    return dispatch<bf16>(K, K, kv, levels, coeffs, make_update<bf16>(Kn, Vn, V, &nt, pos), s);
  return dispatch<float>(K, K, kv, levels, coeffs, make_update<float>(Kn, Vn, V, &nt, pos), s);
}

}  // namespace wf
