// rowfinish.cuh -- one warp finishes one query row: the order of its kept keys
// (when the selection is an output), the softmax over them (Eq. 4) and the
// weighted sum of their value rows.
//
// The row's n <= 32 KPL kept (score, index) pairs sit in registers, entry
// 32 c + lane in lane `lane`'s slot c.  The value rows are gathered with
// 16-byte loads, D / 8 lanes per row, 32 / (D / 8) rows per load, 16 loads in
// flight: a load instruction touches 2 to 4 whole 128-byte lines.  (A thread
// per query row reading its own value rows touches 32 lines per load and
// occupies the load pipe 8 to 16 times as long.)
#pragma once

#include <stdint.h>

#include "common.cuh"
#include "rowlist.cuh"

namespace topk {

__device__ __forceinline__ float warp_max_f(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

__device__ __forceinline__ float warp_sum_f(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Sorts the warp's 32 KPL keys in descending order (a bitonic network; strides
// of 32 and more stay within a lane).
template <int KPL>
__device__ __forceinline__ void warp_sort_desc(uint64_t (&key)[KPL]) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int kk = 2; kk <= 32 * KPL; kk <<= 1) {
#pragma unroll
    for (int jc = KPL / 2; jc >= 1; jc >>= 1) {
      if (32 * jc < kk) {
#pragma unroll
        for (int c = 0; c < KPL; ++c) {
          if (c & jc) continue;
          const uint64_t a = key[c], b = key[c | jc];
          const bool desc = ((32 * c) & kk) == 0;
          const bool swap = (a < b) == desc;
          key[c] = swap ? b : a;
          key[c | jc] = swap ? a : b;
        }
      }
    }
#pragma unroll 1
    for (int j = kk < 64 ? kk >> 1 : 16; j >= 1; j >>= 1) {
#pragma unroll
      for (int c = 0; c < KPL; ++c) {
        const uint64_t a = key[c], b = __shfl_xor_sync(0xffffffffu, a, j);
        const bool desc = ((32 * c + lane) & kk) == 0;
        const bool first = (lane & j) == 0;
        key[c] = ((a < b) == (desc == first)) ? b : a;
      }
    }
  }
}

// The selection outputs of one row: the sorted keys, then -1 / -inf.
template <int KPL>
__device__ __forceinline__ void write_selection(const uint64_t (&key)[KPL], int n, int topk, int32_t* idx_row,
                                                float* score_row) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < KPL; ++c) {
    const int t = 32 * c + lane;
    if (t < topk) {
      if (idx_row) idx_row[t] = t < n ? static_cast<int32_t>(key_index(key[c])) : -1;
      if (score_row) score_row[t] = t < n ? key_score(key[c]) : -INFINITY;
    }
  }
}

template <typename T>
struct Vec16;  // 16 bytes of a value row as floats
template <>
struct Vec16<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ __forceinline__ static void fma(float w, const uint4& u, float (&acc)[8]) {
    const uint32_t x[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[2 * i] = fmaf(w, __uint_as_float(x[i] << 16), acc[2 * i]);
      acc[2 * i + 1] = fmaf(w, __uint_as_float(x[i] & 0xffff0000u), acc[2 * i + 1]);
    }
  }
  __device__ __forceinline__ static uint4 pack(const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
};
template <>
struct Vec16<float> {
  static constexpr int N = 4;
  __device__ __forceinline__ static void fma(float w, const uint4& u, float (&acc)[4]) {
    acc[0] = fmaf(w, __uint_as_float(u.x), acc[0]);
    acc[1] = fmaf(w, __uint_as_float(u.y), acc[1]);
    acc[2] = fmaf(w, __uint_as_float(u.z), acc[2]);
    acc[3] = fmaf(w, __uint_as_float(u.w), acc[3]);
  }
  __device__ __forceinline__ static uint4 pack(const float (&f)[4]) {
    return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
  }
};

// out row = sum_t softmax(s)_t V[j_t] over the first n entries; entries at and
// past n are not read (a value row that no key selects may hold anything).  A
// row with no entry writes zeros.
template <typename T, int D, int KPL>
__device__ __forceinline__ void softmax_gather(const float (&s)[KPL], const uint32_t (&j)[KPL], int n,
                                               const T* __restrict__ vb, T* __restrict__ orow) {
  using V = Vec16<T>;
  constexpr int LPR = D / V::N;  // lanes per value row
  constexpr int G = 32 / LPR;    // rows per load
  static_assert(LPR >= 1 && LPR <= 32 && 32 % LPR == 0, "a value row spans 1..32 lanes");
  constexpr int STEPS = 32 / G;                               // loads per 32 entries
  constexpr int CB = STEPS >= 16 ? 1 : (16 / STEPS < KPL ? 16 / STEPS : KPL);  // 32-entry slots per batch
  constexpr int UB = STEPS < 16 ? STEPS : 16;                 // loads per slot and batch
  const int lane = threadIdx.x & 31;
  const int grp = lane / LPR, col = lane % LPR;
  float m = -INFINITY;
#pragma unroll
  for (int c = 0; c < KPL; ++c)
    if (32 * c + lane < n) m = fmaxf(m, s[c]);
  m = warp_max_f(m);
  float w[KPL], z = 0.f;
#pragma unroll
  for (int c = 0; c < KPL; ++c) {
    w[c] = 32 * c + lane < n ? expf(s[c] - m) : 0.f;
    z += w[c];
  }
  z = warp_sum_f(z);
  float acc[V::N];
#pragma unroll
  for (int e = 0; e < V::N; ++e) acc[e] = 0.f;
  const T* vc = vb + col * V::N;
#pragma unroll
  for (int c0 = 0; c0 < KPL; c0 += CB) {
    if (32 * c0 >= n) break;
#pragma unroll
    for (int u0 = 0; u0 < STEPS; u0 += UB) {
      uint4 raw[CB][UB];
#pragma unroll
      for (int b = 0; b < CB; ++b)
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const int tl = (u0 + u) * G + grp;
          const uint32_t jj = __shfl_sync(0xffffffffu, j[c0 + b], tl);
          raw[b][u] = make_uint4(0u, 0u, 0u, 0u);
          if (32 * (c0 + b) + tl < n) raw[b][u] = __ldg(reinterpret_cast<const uint4*>(vc + static_cast<size_t>(jj) * D));
        }
#pragma unroll
      for (int b = 0; b < CB; ++b)
#pragma unroll
        for (int u = 0; u < UB; ++u)
          V::fma(__shfl_sync(0xffffffffu, w[c0 + b], (u0 + u) * G + grp), raw[b][u], acc);
    }
  }
#pragma unroll
  for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
    for (int e = 0; e < V::N; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
  const float inv = n > 0 ? 1.0f / z : 0.0f;
#pragma unroll
  for (int e = 0; e < V::N; ++e) acc[e] *= inv;
  if (grp == 0) *(reinterpret_cast<uint4*>(orow) + col) = V::pack(acc);
}

// The exact top k (a row of m <= 32 KH candidates, entry 32 c + lane in slot c,
// in index order) moved in order into buf (k entries of shared memory); returns
// how many there are, and in `low` a score that at least k entries reach (-inf
// unless m > k).  The k-th score is found bit by bit on the ordered scores,
// below the bits that all candidates share; ties at it go to the lower entries.
template <int KH>
__device__ __forceinline__ int select_into(const float (&s)[KH], const uint32_t (&j)[KH], int m, int k, uint2* buf,
                                           float& low) {
  const int lane = threadIdx.x & 31;
  uint32_t o[KH];
  uint32_t hi = 0u, lo = 0xffffffffu;
#pragma unroll
  for (int c = 0; c < KH; ++c) {
    const bool in = 32 * c + lane < m;
    o[c] = in ? ord_f32(s[c]) : 0u;  // 0: below every score
    hi = max(hi, o[c]);
    lo = in ? min(lo, o[c]) : lo;
  }
  uint32_t thr = 1u;
  int eq_left = 32 * KH;  // entries equal to thr still to take
  if (m > k) {
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    int c_thr = m;  // entries >= thr
    thr = lo;
    if (lo != hi) {
      const int top = 31 - __clz(lo ^ hi);
      thr = hi & ~((2u << top) - 1u);
#pragma unroll 1
      for (int b = top; b >= 0 && c_thr != k; --b) {
        const uint32_t cand = thr | (1u << b);
        unsigned n = 0;
#pragma unroll
        for (int c = 0; c < KH; ++c) n += o[c] >= cand ? 1u : 0u;
        const int all = static_cast<int>(__reduce_add_sync(0xffffffffu, n));
        if (all >= k) {
          thr = cand;
          c_thr = all;
        }
      }
    }
    if (c_thr != k) {
      unsigned n = 0;
#pragma unroll
      for (int c = 0; c < KH; ++c) n += o[c] > thr ? 1u : 0u;
      eq_left = k - static_cast<int>(__reduce_add_sync(0xffffffffu, n));
    }
  }
  low = m > k ? unord_f32(thr) : -INFINITY;
  const uint32_t below = (1u << lane) - 1u;
  int w = 0;
#pragma unroll
  for (int c = 0; c < KH; ++c) {
    bool take = o[c] >= thr;
    if (eq_left < 32 * KH) {  // a tie at thr that not all entries equal to it fit in
      const unsigned beq = __ballot_sync(0xffffffffu, o[c] == thr);
      take = o[c] > thr || (o[c] == thr && __popc(beq & below) < eq_left);
      eq_left -= __popc(beq);
    }
    const unsigned bt = __ballot_sync(0xffffffffu, take);
    if (take) buf[w + __popc(bt & below)] = make_uint2(__float_as_uint(s[c]), j[c]);
    w += __popc(bt);
  }
  __syncwarp();
  return w;
}

// One row from its n <= 32 KPL kept pairs load(t) -> (score bits, index), in
// index order: used in that order, or sorted (and written) first if the
// selection is an output.
template <typename T, int D, int KPL, typename Load>
__device__ __forceinline__ void finish_kept(Load&& load, int n, int topk, const T* __restrict__ vb,
                                            T* __restrict__ orow, int32_t* idx_row, float* score_row) {
  const int lane = threadIdx.x & 31;
  float s[KPL];
  uint32_t j[KPL];
#pragma unroll
  for (int c = 0; c < KPL; ++c) {
    const int t = 32 * c + lane;
    const uint2 e = t < n ? load(t) : make_uint2(0u, 0u);
    s[c] = __uint_as_float(e.x);
    j[c] = e.y;
  }
  if (idx_row || score_row) {
    uint64_t key[KPL];
#pragma unroll
    for (int c = 0; c < KPL; ++c) key[c] = 32 * c + lane < n ? make_key(s[c], j[c]) : 0ull;
    warp_sort_desc<KPL>(key);
    write_selection<KPL>(key, n, topk, idx_row, score_row);
#pragma unroll
    for (int c = 0; c < KPL; ++c) {
      s[c] = key_score(key[c]);
      j[c] = key_index(key[c]);
    }
  }
  softmax_gather<T, D, KPL>(s, j, n, vb, orow);
}

// One row from its m <= 32 KH candidates load(t) -> (score bits, index) in index
// order, which hold its top k <= 32 KPL: the exact top k, used in index order, or
// sorted (and written) first if the selection is an output.  buf: k entries of
// this warp's shared memory.
template <typename T, int D, int KH, int KPL, typename Load>
__device__ __forceinline__ void finish_row(Load&& load, int m, int topk, uint2* buf, const T* __restrict__ vb,
                                           T* __restrict__ orow, int32_t* idx_row, float* score_row) {
  const int lane = threadIdx.x & 31;
  int n;
  {
    float s[KH];
    uint32_t j[KH];
#pragma unroll
    for (int c = 0; c < KH; ++c) {
      const int t = 32 * c + lane;
      const uint2 e = t < m ? load(t) : make_uint2(0u, 0u);
      s[c] = __uint_as_float(e.x);
      j[c] = e.y;
    }
    float low;
    __syncwarp();  // buf may be where the candidates were read from
    n = select_into<KH>(s, j, m, topk, buf, low);
  }
  finish_kept<T, D, KPL>([buf](int t) { return buf[t]; }, n, topk, vb, orow, idx_row, score_row);
  __syncwarp();  // buf is free again
}

}  // namespace topk
