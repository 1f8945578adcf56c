// attn_simt.cuh -- top-k attention (Eq. 4) with scores on the CUDA cores.
//
// Serves the fp32 path (scores by sequential fp32 FMA, never TF32, as the
// paper's own fp32 runs had TF32 disabled) and bf16 inputs under Eq. 2's
// arbitrary bit masks (bf16 products are exact in fp32, accumulation fp32).
//
// A CTA of NW warps takes NW * RPW query rows of one (b, h), RPW per warp.  Keys
// come in tiles of 64, staged in shared memory as fp32; the next tile's global
// loads are in flight while one is used.  Lane l of a warp scores keys l and
// l + 32 of the tile for the warp's rows, so a row's 64 new scores sit in its
// warp's registers: two votes pick those above the row's threshold and append
// them, in key order, to the row's list of up to 32 KH candidates in shared
// memory.  A list without room for 64 more is cut to its exact top k
// (select_into() of rowfinish.cuh), whose lowest score is the new threshold.
// After the last key the warp finishes its rows one by one (rowfinish.cuh).  No
// score matrix is stored anywhere.
//
// A thread per query row, as before, left the smallest calls on a handful of
// SMs and ran the selection in divergent lockstep: B1 H1 L512 d64 k32 fp32 took
// 204 us and takes 18 here; B8 H12 L512 d64 k64 bf16 under a bit mask 859 and
// 285.  What bounds the latter: shared-memory reads of the key tile (192 cycles
// per warp and tile against 128 of FMA issue) and the rows' finishing latency.
#pragma once

#include "kernels.h"
#include "rowfinish.cuh"

namespace topk {

namespace {

constexpr int KT = 64;  // keys per staged tile

// 16 bytes of T as floats in shared memory
template <typename T>
__device__ __forceinline__ void stage16(float* dst, const uint4& u);
template <>
__device__ __forceinline__ void stage16<float>(float* dst, const uint4& u) {
  *reinterpret_cast<uint4*>(dst) = u;
}
template <>
__device__ __forceinline__ void stage16<__nv_bfloat16>(float* dst, const uint4& u) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 2; ++i)
    *reinterpret_cast<uint4*>(dst + 4 * i) =
        make_uint4(w[2 * i] << 16, w[2 * i] & 0xffff0000u, w[2 * i + 1] << 16, w[2 * i + 1] & 0xffff0000u);
}

template <int D, int NW, int RPW, int KH>
struct SimtShape {
  static constexpr int ROWS = NW * RPW;
  static constexpr int LDK = D + 4;  // padded key row: lanes' 16-byte reads of 8 rows touch all banks once
  static constexpr size_t kKeys = static_cast<size_t>(KT) * LDK * 4;
  static constexpr size_t kQ = static_cast<size_t>(ROWS) * D * 4;
  static constexpr size_t kLists = static_cast<size_t>(ROWS) * KH * 32 * sizeof(uint2);
  static constexpr size_t kBytes = kKeys + kQ + kLists;
  static constexpr int kMaxK = KH * 32 - KT;  // a list holds the top k and one tile
};

template <typename T, int D, int NW, int RPW, int KH, int KPL>
__global__ void __launch_bounds__(NW * 32)
    attn_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* __restrict__ out,
                     int BH, int H, int Lq, int Lk, int topk, int causal, const int32_t* __restrict__ kv_len,
                     const uint32_t* __restrict__ mask, long long mask_bs, long long mask_hs,
                     int32_t* __restrict__ idx, float* __restrict__ score) {
  using S = SimtShape<D, NW, RPW, KH>;
  constexpr int ROWS = S::ROWS, LDK = S::LDK, THREADS = NW * 32;
  constexpr int VEC = 16 / sizeof(T);                    // elements per 16-byte load
  constexpr int NV = KT * D / VEC;                       // 16-byte loads per key tile
  constexpr int PT = (NV + THREADS - 1) / THREADS;       // of them per thread
  constexpr int CAP = KH * 32;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  float* ks = reinterpret_cast<float*>(smem_raw);                       // [KT][LDK]
  float* qs = reinterpret_cast<float*>(smem_raw + S::kKeys);            // [ROWS][D]
  uint2* lists = reinterpret_cast<uint2*>(smem_raw + S::kKeys + S::kQ);  // [ROWS][CAP]

  const int n_qt = (Lq + ROWS - 1) / ROWS;
  const int unit = blockIdx.x;
  // causal: heaviest query tiles first
  const int qt = causal ? (n_qt - 1 - unit / BH) : (unit % n_qt);
  const int bh = causal ? (unit % BH) : (unit / n_qt);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0 = warp * RPW, i0 = qt * ROWS + r0;  // the warp's first row

  for (int e = tid; e < ROWS * D / VEC; e += THREADS) {
    const int r = e / (D / VEC), i = qt * ROWS + r;
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    if (i < Lq) u = __ldg(reinterpret_cast<const uint4*>(q + (static_cast<size_t>(bh) * Lq + i) * D) + e % (D / VEC));
    stage16<T>(qs + r * D + (e % (D / VEC)) * VEC, u);
  }

  // Eq. 2's masks.  Causal: the queries are the last Lq positions, key j is
  // valid for query i iff j <= i + Lk - Lq.  kv_len: the batch's key count.
  // Both give each row a valid key prefix [0, lim); the bit mask (1 = valid)
  // then removes keys anywhere in it.
  const int coff = Lk - Lq;
  const int kv_end = kv_len ? min(max(__ldg(kv_len + bh / H), 0), Lk) : Lk;
  const int kend = min(kv_end, causal ? min((qt + 1) * ROWS, Lq) + coff : Lk);
  const T* kb = k + static_cast<size_t>(bh) * Lk * D;
  const int words = (Lk + 31) / 32;
  const uint32_t* mrow = mask ? mask + (bh / H) * mask_bs + (bh % H) * mask_hs + static_cast<long long>(i0) * words : nullptr;

  int cnt[RPW], lim[RPW];
  float tau[RPW];
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    cnt[r] = 0;
    tau[r] = -INFINITY;
    const int i = i0 + r;
    lim[r] = i < Lq ? min(kv_end, causal ? min(i + 1 + coff, Lk) : Lk) : 0;
  }

  uint4 nx[PT];
  auto fetch = [&](int j0) {
#pragma unroll
    for (int p = 0; p < PT; ++p) {
      const int e = tid + p * THREADS, jj = j0 + e / (D / VEC);
      nx[p] = make_uint4(0u, 0u, 0u, 0u);
      if (e < NV && jj < Lk)
        nx[p] = __ldg(reinterpret_cast<const uint4*>(kb + static_cast<size_t>(jj) * D) + e % (D / VEC));
    }
  };
  if (kend > 0) fetch(0);
  for (int j0 = 0; j0 < kend; j0 += KT) {
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PT; ++p) {
      const int e = tid + p * THREADS;
      if (e < NV) stage16<T>(ks + (e / (D / VEC)) * LDK + (e % (D / VEC)) * VEC, nx[p]);
    }
    __syncthreads();
    if (j0 + KT < kend) fetch(j0 + KT);
    uint32_t bits[RPW][2];
#pragma unroll
    for (int r = 0; r < RPW; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        bits[r][h] = mask && i0 + r < Lq && j0 / 32 + h < words ? __ldg(mrow + static_cast<long long>(r) * words + j0 / 32 + h)
                                                                : (mask ? 0u : 0xffffffffu);
    float s[RPW][2];
#pragma unroll
    for (int r = 0; r < RPW; ++r) s[r][0] = s[r][1] = 0.0f;
    const float* k0 = ks + lane * LDK;
    const float* k1 = k0 + 32 * LDK;
    const float* qr = qs + r0 * D;
#pragma unroll 8
    for (int t = 0; t < D; t += 4) {
      const float4 a = *reinterpret_cast<const float4*>(k0 + t), b = *reinterpret_cast<const float4*>(k1 + t);
#pragma unroll
      for (int r = 0; r < RPW; ++r) {
        const float4 x = *reinterpret_cast<const float4*>(qr + r * D + t);
        s[r][0] = fmaf(x.x, a.x, s[r][0]);
        s[r][1] = fmaf(x.x, b.x, s[r][1]);
        s[r][0] = fmaf(x.y, a.y, s[r][0]);
        s[r][1] = fmaf(x.y, b.y, s[r][1]);
        s[r][0] = fmaf(x.z, a.z, s[r][0]);
        s[r][1] = fmaf(x.z, b.z, s[r][1]);
        s[r][0] = fmaf(x.w, a.w, s[r][0]);
        s[r][1] = fmaf(x.w, b.w, s[r][1]);
      }
    }
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      uint2* lst = lists + (r0 + r) * CAP;
      if (cnt[r] > CAP - KT) {  // no room for a whole tile: the exact top k so far
        float x[KH];
        uint32_t jx[KH];
#pragma unroll
        for (int c = 0; c < KH; ++c) {
          const int t = 32 * c + lane;
          const uint2 e = t < cnt[r] ? lst[t] : make_uint2(0u, 0u);
          x[c] = __uint_as_float(e.x);
          jx[c] = e.y;
        }
        __syncwarp();
        float low;
        cnt[r] = select_into<KH>(x, jx, cnt[r], topk, lst, low);
        tau[r] = fmaxf(tau[r], low);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = j0 + 32 * h + lane;
        const bool pass = s[r][h] > tau[r] && j < lim[r] && ((bits[r][h] >> lane) & 1u);
        const uint32_t bal = __ballot_sync(0xffffffffu, pass);
        if (bal) {
          if (pass) lst[cnt[r] + __popc(bal & ((1u << lane) - 1u))] = make_uint2(__float_as_uint(s[r][h]), j);
          cnt[r] += __popc(bal);
        }
      }
    }
  }
  __syncwarp();

  // the rows' results; a row's own list is its buffer
  const T* vb = v + static_cast<size_t>(bh) * Lk * D;
#pragma unroll 1
  for (int r = 0; r < RPW; ++r) {
    if (i0 + r >= Lq) break;
    const size_t orow = static_cast<size_t>(bh) * Lq + i0 + r;
    uint2* lst = lists + (r0 + r) * CAP;
    int m = cnt[0];
#pragma unroll
    for (int c = 1; c < RPW; ++c) m = r == c ? cnt[c] : m;
    finish_row<T, D, KH, KPL>([lst](int t) { return lst[t]; }, m, topk, lst, vb, out + orow * D,
                              idx ? idx + orow * topk : nullptr, score ? score + orow * topk : nullptr);
  }
}

template <typename T, int D, int NW, int RPW, int KH, int KPL>
int launch_simt_k(const AttnArgs& a, cudaStream_t st) {
  using S = SimtShape<D, NW, RPW, KH>;
  auto kern = attn_simt_kernel<T, D, NW, RPW, KH, KPL>;
  if (S::kBytes > 48 * 1024 &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(S::kBytes)) !=
          cudaSuccess)
    return -1;
  const int BH = a.B * a.H;
  const long long grid = static_cast<long long>(BH) * ((a.Lq + S::ROWS - 1) / S::ROWS);
  kern<<<static_cast<unsigned>(grid), NW * 32, S::kBytes, st>>>(
      static_cast<const T*>(a.q), static_cast<const T*>(a.k), static_cast<const T*>(a.v), static_cast<T*>(a.out),
      BH, a.H, a.Lq, a.Lk, a.topk, a.causal, a.kv_len, a.mask, a.mask_bs, a.mask_hs, a.idx, a.score);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

// k up to 128: 32 rows per CTA (four per warp share each key read) where that
// still gives every SM a few CTAs, else 4 rows per CTA; larger k: 8 rows, one
// per warp, with longer lists.
template <typename T, int D>
int launch_simt(const AttnArgs& a, int num_sms, cudaStream_t st) {
  if (a.topk > 128) {
    static_assert(SimtShape<D, 8, 1, 18>::kMaxK >= kSimtMaxK, "list size");
    return launch_simt_k<T, D, 8, 1, 18, 16>(a, st);
  }
  const long long rows = static_cast<long long>(a.B) * a.H * a.Lq;
  if (rows >= 64LL * num_sms) return launch_simt_k<T, D, 8, 4, 8, 4>(a, st);
  return launch_simt_k<T, D, 4, 1, 8, 4>(a, st);
}

}  // namespace

}  // namespace topk
