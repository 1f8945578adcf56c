// attn_tc.cuh -- fused top-k attention (Eq. 4) for bf16 inputs on sm_103a.
//
// One persistent CTA per SM walks work units: a unit is RT query tiles of 128
// rows of one (b, h).  For a unit the query tiles (Sec. 2.2 "Query chunking",
// C = 128 RT) are loaded once by TMA, then the keys stream through in tiles of
// N that all RT query tiles share:
//
//   warp 0       TMA producer: the query tiles, then K tiles into a ring
//   warps 1, 2   MMA issuers, one per query tile: S = Q K_tile^T with
//                tcgen05.mma (bf16 in, fp32 accumulate) into that query tile's
//                TMEM accumulators [128 x N]
//   warps 4 ..   filters, four per query tile: lane t of warp w owns TMEM lane
//                / query row 32 (w % 4) + t.  It reads its scores with
//                tcgen05.ld.red, which returns each group of eight together
//                with its maximum, and keeps the row's candidates in its list
//                (rowlist.cuh).  After the unit's last key tile it cuts the
//                lists to the top k, or near it (Layout::hand), and hands them
//                over.
//   the rest     epilogue: a warp per row makes the cut exact, orders the kept
//                keys if the selection is an output, applies the softmax over
//                them and gathers the matching value rows (rowfinish.cuh),
//                while the filters stream the next unit.
//
// The score tile never leaves TMEM/registers: no [C x Lk] matrix is written
// to device memory (Sec. 2.2 "Query chunking": memory O(C Lk) becomes
// O(C k) here, in shared memory).  The scale of Eq. 1 is folded into Q by
// the caller.  Causal masking (Eq. 2) skips key tiles past the query tile
// and masks keys j > i inside the diagonal tile.
//
// Every pipeline wait is bounded (common.cuh); on expiry the CTA stops,
// drains its in-flight copies and MMAs, frees TMEM and returns.
#pragma once

#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "rowfinish.cuh"
#include "rowlist.cuh"

namespace topk {

namespace {

constexpr int BM = 128;        // rows of an MMA tile
constexpr int kThreads = 512;  // 4 control warps, 4 RT filter warps, the rest epilogue
constexpr size_t kMaxSmem = 232448;  // shared memory that a CTA may ask for

// D: head size; RT: query tiles per unit; RPU: query rows of a tile that
// belong to the unit.  The MMA tile always has 128 rows; with RPU = 64 or 32
// (RT = 1) only the first RPU of them are the unit's, so that one row's list
// can hold several hundred keys.
// LONG: rows of more than 65,536 keys.  RECS: records per row (rowlist.cuh); which
// of four and eight of them, and with how many scores per offer, see with_variant_i.
template <int D, bool LONG, int RT, int RPU, int RECS>
struct Layout {
  static_assert(RT == 1 || RPU == BM, "reduced-row units take one query tile");
  static constexpr int N = D == 64 ? 128 : 64;  // keys per tile: 16 KB of K
  static constexpr int S = RT == 2 || RPU < BM ? 2 : 3;  // K stages
  static constexpr int R = D / 64;  // 128-byte column blocks per row
  static constexpr int OFFER = RT == 1 && RECS == 4 ? 16 : 32;  // scores per offer
  using List = RowList<RECS, LONG>;
  static constexpr int NQ = RPU / 32;      // filter warps per query tile
  static constexpr int NJ = RT * NQ;       // filter warps in all
  static constexpr int NE = 12 - 4 * RT;   // epilogue warps
  static constexpr int NS = NE > NJ ? NE / NJ : 1;  // epilogue warps that share a filter warp's rows
  static constexpr int RS = 32 / NS;       // rows each of them takes
  // The kept lists go through a device buffer of SL slots per filter warp, so
  // that the epilogue of one unit overlaps the filtering of the next.  Large-k
  // kernels hand their lists over in place: a unit's filtering is long against
  // its epilogue there.
  static constexpr bool kPark = RPU == BM;
  static constexpr int SL = 4 / RT;  // the same buffer size for both RT
  static constexpr uint32_t Q_BYTES = BM * D * 2;  // one query tile
  static constexpr uint32_t KST_BYTES = N * D * 2;
  static constexpr size_t OFF_Q = 0;
  static constexpr size_t OFF_K = OFF_Q + static_cast<size_t>(RT) * Q_BYTES;
  static constexpr size_t OFF_CTRL = OFF_K + static_cast<size_t>(S) * KST_BYTES;
  // TMEM accumulators per query tile: as many N-column buffers as fit in 512
  // columns, at most 4, so that the MMAs run ahead of a filter that prunes
  static constexpr int NACC = 512 / (RT * N) < 4 ? 512 / (RT * N) : 4;
  static constexpr uint32_t TMEM_COLS = RT * NACC * N;
  static constexpr int NBARS = 2 * S + 2 + 2 * RT * NACC + RT;
  static constexpr size_t CTRL_BYTES = (static_cast<size_t>(NBARS) * 8 + 8 + 2 * 8 * 4 + RPU * 4 + 127) & ~size_t(127);
  // Entries of a row that the filters hand over at most: the exact top k, or up to
  // k + 63 candidates that the epilogue cuts (a warp per row).  Parked lists are cut by
  // the filters, 32 rows in lockstep (B8 H12 L512 k = 64: 185 us against 153; B32 H12
  // L128 k = 16: 129 against 89), but where rows are so long that the filters bound
  // the kernel (L = 65,536, k = 64: 17.9 ms against 18.1).  Lists of large k that stay
  // in place are cut by the epilogue: the filters wait for it anyhow (L = 8,192,
  // k = 256: 3.0 ms against 5.4).
  // The buffer has room for hand_max entries per row in any case, so that its size does
  // not depend on Lk; LONG rows give the last ones up for their break counts.
  static constexpr int hand_max(int topk) { return (topk + 63) & ~31; }
  static constexpr int hand(int topk, int Lk) {
    if (!kPark) return hand_max(topk);
    if (!LONG) return Lk < 32768 ? topk : hand_max(topk);
    const int given = (breaks(Lk) + 4 * SL - 1) / (4 * SL);  // 8 SL bytes each, 2 per break
    return hand_max(topk) - given > topk ? hand_max(topk) - given : topk;
  }
  static constexpr int breaks(int Lk) { return (Lk - 1) / 65536; }
  static constexpr bool breaks_in_park(int topk, int Lk) {  // up to 16 million keys
    return kPark && breaks(Lk) <= 4 * SL * (hand_max(topk) - hand(topk, Lk));
  }
  static constexpr size_t OFF_LIST = OFF_CTRL + CTRL_BYTES;
  static constexpr size_t kFixed = 1024 + OFF_LIST;

  static constexpr int min_cap(int topk) { return (topk + kListSlack + 8 + 7) & ~7; }
  // the epilogue warps' buffers, behind the lists
  static constexpr size_t buf_bytes(int topk) { return static_cast<size_t>(NE) * topk * sizeof(uint2); }
  // List slots per row: what fits, up to about 2.5 k + 64 (longer lists prune
  // less often but let their thresholds lag further behind).
  static int cap(int topk) {
    const int want = (5 * topk / 2 + 64 + 7) & ~7;
    int c = static_cast<int>((kMaxSmem - kFixed) / NJ / (kListStride * 6)) & ~7;
    while (c > 0 && kFixed + buf_bytes(topk) + NJ * List::bytes(c) > kMaxSmem) c -= 8;
    c = std::min(c, std::max(want, min_cap(topk)));
    return c >= min_cap(topk) ? c : 0;
  }
  static bool fits(int topk) { return cap(topk) > 0; }
  // Classes of the bound stretch (RowList): 2 k, or what the warp's memory holds,
  // in multiples of the slots that a tile takes at most (groups of four keys).
  static constexpr int kTileSlots = N / 4;
  static int classes(int topk) {
    const int mem = static_cast<int>(List::bytes(cap(topk)) / (kListStride * 4));
    const int want = std::max(2 * topk, 16) + kTileSlots - 1;
    return std::min(want, mem) / kTileSlots * kTileSlots;
  }
  static size_t bytes(int topk) { return kFixed + buf_bytes(topk) + NJ * List::bytes(cap(topk)); }

  static constexpr size_t park_keys_per_cta(int topk) { return kPark ? static_cast<size_t>(NJ) * SL * 32 * hand_max(topk) : 0; }
  static constexpr size_t park_bytes(int grid, int topk) {
    return kPark ? static_cast<size_t>(grid) * (park_keys_per_cta(topk) * 8 + NJ * SL * 32 * 4) : 0;
  }
};

// How the bound pass sorts its nb key tiles of N keys into classes (RowList): the
// tiles' maxima over groups of `group` keys go to slots 0 .. n - 1 in turn, N / group
// of them per tile.  Groups of 64 keys, or as many fewer as leave a group per class.
// n is a multiple of a tile's slots, so that a tile never writes past slot n - 1
// (32 slots per tile at N = 128, group = 4), and of 16.
struct BoundSplit {
  int group, n;
};
__host__ __device__ constexpr BoundSplit bound_split(int N, int nb, int classes) {
  int group = 64;
  while (group > 4 && nb * N < group * classes) group >>= 1;
  const int per = N / group, unit = per > 16 ? per : 16;
  const int n = nb * per < classes ? nb * per : classes;
  return BoundSplit{group, n & ~(unit - 1)};
}

// Waits for an mbarrier phase: every lane tries once, then lane 0 polls.  The
// whole warp leaves together.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, const DevCtl& ctl,
                                          volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  int ok = 0;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait_slow<true>(bar, parity, ctl, abort_flag) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (ok) (void)mbar_try_wait(bar, parity);  // every lane observes the completed phase
  return ok != 0;
}

// Waits (bounded; lane 0 polls) until the shared-memory counter *ctr, which
// only grows, reaches target; every lane then reads it with acquire
// semantics itself, so that what the releasing warp wrote before it is
// visible to the whole warp.  False if the CTA aborts or the limit runs out.
__device__ __forceinline__ bool wait_count(uint32_t* ctr, uint32_t target, const DevCtl& ctl,
                                           volatile int* abort_flag) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0 && static_cast<int>(ld_acquire_u32(ctr) - target) < 0) {
    const unsigned long long t0 = global_ns();
    for (uint32_t spin = 0;; ++spin) {
      if (static_cast<int>(ld_acquire_u32(ctr) - target) >= 0) break;
      if ((spin & 15u) == 15u) {
        if (*abort_flag) {
          ok = 0;
          break;
        }
        if (global_ns() - t0 > ctl.wait_limit_ns) {
          atomicOr(ctl.error, kDevErrTimeout);
          *abort_flag = 1;
          ok = 0;
          break;
        }
      }
      __nanosleep(32u << (spin < 4u ? spin : 4u));
    }
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (ok) (void)ld_acquire_u32(ctr);
  return ok != 0;
}

// Bounded wait that ignores the abort flag: used only to drain in-flight
// asynchronous work before the CTA exits.
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity, const DevCtl& ctl) {
  const unsigned long long t0 = global_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_ns() - t0 > ctl.wait_limit_ns) {
      atomicOr(ctl.error, kDevErrTimeout);
      return;
    }
  }
}

template <int D, bool LONG, int RT, int RPU, int RECS>
__global__ void __launch_bounds__(kThreads, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                   const __nv_bfloat16* __restrict__ v, __nv_bfloat16* __restrict__ out, int BH, int H, int Lq,
                   int Lk, int topk, int cap, int hand, int classes, int bound_den, int causal,
                   const int32_t* __restrict__ kv_len, int n_units, int parts, uint2* __restrict__ part_keys, int* __restrict__ part_n, int32_t* __restrict__ idx,
                   float* __restrict__ score, uint2* __restrict__ park, int* __restrict__ park_n, uint16_t* breaks,
                   DevCtl ctl) {
  using L = Layout<D, LONG, RT, RPU, RECS>;
  using List = typename L::List;
  constexpr int kOffer = L::OFFER;
  constexpr int N = L::N, S = L::S, R = L::R, NACC = L::NACC, NQ = L::NQ, NJ = L::NJ, NE = L::NE;
  constexpr uint32_t IDESC = idesc_bf16_f32(BM, N);
  constexpr int RU = RPU * RT;  // query rows per unit

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* q_s = smem + L::OFF_Q;
  uint8_t* k_s = smem + L::OFF_K;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::OFF_CTRL);
  uint64_t* full_k = bars;
  uint64_t* empty_k = bars + S;
  uint64_t* q_full = bars + 2 * S;
  uint64_t* q_empty = bars + 2 * S + 1;
  uint64_t* acc_full = bars + 2 * S + 2;                  // [RT][NACC]
  uint64_t* acc_empty = bars + 2 * S + 2 + RT * NACC;     // [RT][NACC]
  uint64_t* drain = bars + 2 * S + 2 + 2 * RT * NACC;     // [RT]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + L::NBARS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint32_t* pk_done = tmem_slot + 2;                      // [8] units handed over by each filter warp
  uint32_t* ep_done = tmem_slot + 10;                     // [8] units finished by the epilogue, per warp or job
  int* row_n = reinterpret_cast<int*>(tmem_slot + 18);    // [RPU] kept counts (lists handed over in place)
  uint8_t* list_mem = smem + L::OFF_LIST;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full_k[s], 1);
      mbar_init(&empty_k[s], RT);
    }
    mbar_init(q_full, 1);
    mbar_init(q_empty, RT);
    for (int b = 0; b < RT * NACC; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], NQ);
    }
    for (int rt = 0; rt < RT; ++rt) mbar_init(&drain[rt], 1);
    *abort_flag = 0;
    for (int q = 0; q < 8; ++q) pk_done[q] = ep_done[q] = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, L::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int n_qt = (Lq + RU - 1) / RU;
  // A unit is (b, h, query rows, key part): with parts > 1 (grids that would
  // leave SMs idle, as decoding a few positions against a long cache does)
  // each query tile's key tiles are split into `parts` ranges, each part keeps
  // its own top k, and a merge kernel combines them.
  auto decode = [&](int u_, int& bh, int& qt, int& part) {
    part = u_ % parts;
    const int u = u_ / parts;
    if (causal) {  // heaviest query tiles first
      qt = n_qt - 1 - u / BH;
      bh = u % BH;
    } else {  // consecutive units share a head, so its K/V stay in L2
      bh = u / n_qt;
      qt = u % n_qt;
    }
  };
  // Eq. 2's masks as a valid key prefix per row: causal (queries are the
  // last Lq positions: key j is valid for query i iff j <= i + Lk - Lq) and
  // the batch's key count.  A unit streams at least one key tile, all of it
  // masked if its rows have no key, so that every pipeline stage runs.
  const int coff = Lk - Lq;
  auto kv_end = [&](int bh) { return kv_len ? min(max(__ldg(kv_len + bh / H), 0), Lk) : Lk; };
  auto key_tiles = [&](int bh, int i_end) {  // key tiles of the query rows below i_end
    int kend = min(kv_end(bh), causal ? min(i_end + coff, Lk) : Lk);
    kend = max(kend, 1);
    return (kend + N - 1) / N;
  };
  auto row_limit = [&](int bh, int i) {  // keys j < limit are valid for query i
    return static_cast<uint32_t>(min(kv_end(bh), causal ? min(i + 1 + coff, Lk) : Lk));
  };
  // key tiles [t0, t1) of a unit's part; a part left without tiles streams one
  // fully masked tile (empty = true) so that every stage keeps its handshakes
  auto tile_range = [&](int bh, int qt, int part, int& t0, int& t1, bool& empty) {
    const int nk = key_tiles(bh, (qt + 1) * RU);
    t0 = static_cast<int>(static_cast<long long>(part) * nk / parts);
    t1 = static_cast<int>(static_cast<long long>(part + 1) * nk / parts);
    empty = t1 <= t0;
    if (empty) {
      t0 = 0;
      t1 = 1;
    }
  };

  // The bound pass: the n_full key tiles that are valid for every row of the
  // unit are scored twice, first only for their group maxima, so that the main
  // pass starts with a threshold (RowList::bound_begin).  The second GEMM costs
  // less than the candidates it saves: bounds over a quarter, three quarters and
  // all of the keys took 20.3, 19.3 and 18.4 ms at L = 65536, k = 64.  Where rows have
  // many keys per k it covers a share of them (bound_divisor()).  Fewer than
  // 6 k keys give no useful bound.
  auto bound_tiles = [&](int bh, int qt, int t0, int t1, bool empty) {
    if (empty) return 0;
    const int nb = (min(t1, static_cast<int>(row_limit(bh, qt * RU)) / N) - t0) / bound_den;
    return nb * N >= 6 * topk ? nb : 0;
  };

  // Rows of more than 65,536 keys: where a filter warp's break counts lie, and how
  // many of them a unit's key tiles [t0, t1) leave.
  constexpr int kStretch = 65536 / N;  // key tiles
  auto breaks_of = [&](int job) {
    return breaks + (static_cast<size_t>(blockIdx.x) * NJ + job) * L::breaks(Lk) * 32;
  };
  auto n_breaks = [&](int t0, int t1) { return (t1 - 1) / kStretch - t0 / kStretch; };

  // entry t of row r of filter warp `job`'s lists, of a unit's key tiles [t0, t1)
  auto list_at = [&](int job, int r, int t, int t0, int t1) {
    const uint32_t base = smem_u32(list_mem + job * List::bytes(cap)) + List::M::kRecBytes;
    uint32_t j = lds_u16(base + cap * kScStep + t * kIxStep + r * 2);
    if constexpr (LONG) {
      const uint16_t* b = breaks_of(job) + r;
      uint32_t hi = t0 / kStretch;
      for (int e = n_breaks(t0, t1); e > 0; --e, b += 32) hi += t >= *b ? 1u : 0u;
      j |= hi << 16;
    }
    return make_uint2(__float_as_uint(lds_f32(base + t * kScStep + r * 4)), j);
  };

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      tma_prefetch_desc(&tmq);
      tma_prefetch_desc(&tmk);
    }
    uint32_t it = 0, q_issued = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
      int bh, qt, part;
      decode(u, bh, qt, part);
      if (!warp_wait(q_empty, (q_issued & 1u) ^ 1u, ctl, abort_flag)) break;
      if (lane == 0) {
        mbar_arrive_expect_tx(q_full, RT * L::Q_BYTES);
        for (int rt = 0; rt < RT; ++rt)
          for (int r = 0; r < R; ++r)
            tma_load_3d(q_s + rt * L::Q_BYTES + r * BM * 128, &tmq, q_full, r * 64, qt * RU + rt * BM, bh);
      }
      ++q_issued;
      int t0, t1;
      bool empty;
      tile_range(bh, qt, part, t0, t1, empty);
      const int nb = bound_tiles(bh, qt, t0, t1, empty);
      for (int i = -nb; i < t1 - t0; ++i) {
        const int kt = t0 + (i < 0 ? i + nb : i);
        const int s = it % S;
        const uint32_t ph = (it / S) & 1u;
        if (!warp_wait(&empty_k[s], ph ^ 1u, ctl, abort_flag)) {
          ok = false;
          break;
        }
        if (lane == 0) {
          if (ctl.debug_skip_arrive && it == 1) {
            // testing hook: withhold this stage so the consumers' waits run out
          } else {
            mbar_arrive_expect_tx(&full_k[s], L::KST_BYTES);
            for (int r = 0; r < R; ++r)
              tma_load_3d(k_s + static_cast<size_t>(s) * L::KST_BYTES + r * N * 128, &tmk, &full_k[s], r * 64,
                          kt * N, bh);
          }
        }
        ++it;
      }
    }
    // drain: every issued copy must have landed before the CTA may exit
    if (lane == 0) {
      for (uint32_t back = 1; back <= static_cast<uint32_t>(S) && back <= it; ++back) {
        const uint32_t t = it - back;
        if (ctl.debug_skip_arrive && t == 1) continue;
        mbar_drain(&full_k[t % S], (t / S) & 1u, ctl);
      }
      if (q_issued > 0) mbar_drain(q_full, (q_issued - 1) & 1u, ctl);
    }
    __syncwarp();
  } else if (warp <= RT) {
    // ------------------------------------------------------------ MMA issuers
    const int rt = warp - 1;
    uint32_t it = 0, acc_it = 0, qi = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x, ++qi) {
      int bh, qt, part;
      decode(u, bh, qt, part);
      if (!warp_wait(q_full, qi & 1u, ctl, abort_flag)) break;
      tc_fence_after();
      int t0, t1;
      bool empty;
      tile_range(bh, qt, part, t0, t1, empty);
      const int nb = bound_tiles(bh, qt, t0, t1, empty);
      for (int i = -nb; i < t1 - t0; ++i, ++it, ++acc_it) {
        const int s = it % S;
        const int b = rt * NACC + acc_it % NACC;
        if (!warp_wait(&full_k[s], (it / S) & 1u, ctl, abort_flag) ||
            !warp_wait(&acc_empty[b], ((acc_it / NACC) & 1u) ^ 1u, ctl, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (lane == 0) {
          const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(b * N);
          const uint32_t qa = smem_u32(q_s) + rt * L::Q_BYTES;
          const uint32_t ka = smem_u32(k_s + static_cast<size_t>(s) * L::KST_BYTES);
#pragma unroll
          for (int st = 0; st < D / 16; ++st) {
            const uint32_t r = st / 4, off = (st % 4) * 32;
            mma_bf16_ss(d_tmem, sdesc_k128(qa + r * BM * 128 + off), sdesc_k128(ka + r * N * 128 + off), IDESC,
                        st > 0 ? 1u : 0u);
          }
          mma_commit(&empty_k[s]);
          mma_commit(&acc_full[b]);
        }
        __syncwarp();
      }
      if (!ok) break;
      if (lane == 0) mma_commit(q_empty);
      __syncwarp();
    }
    // drain: all issued MMAs must complete before TMEM is freed
    if (lane == 0) {
      mma_commit(&drain[rt]);
      mbar_drain(&drain[rt], 0, ctl);
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 4 + 4 * RT) {
    // ------------------------------------------------------------ filters
    const int quad = warp & 3;       // TMEM lane quarter
    const int rt = (warp - 4) >> 2;  // query tile
    if (quad < NQ) {                 // lanes of the MMA tile that belong to the unit
      const int job = rt * NQ + quad;
      const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
      uint32_t acc_it = 0;
      List list;
      list.bind(list_mem + job * List::bytes(cap), cap, topk);
      if constexpr (LONG) list.brk.p = breaks_of(job) + lane;
      bool ok = true;
      uint32_t s = 0;  // units done
      for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x, ++s) {
        int bh, qt, part;
        decode(u, bh, qt, part);
        const int i0 = qt * RU + rt * BM + quad * 32;  // the warp's first query row
        const int i_row = i0 + lane;
        if (!L::kPark && parts == 1 && s > 0) {  // the lists handed over in place are free again
          for (int h = 0; ok && h < L::NS; ++h)
            ok = wait_count(&ep_done[job * L::NS + h], s, ctl, abort_flag);
          if (!ok) break;
        }
        float tau0 = i_row < Lq ? -INFINITY : INFINITY;
        int t0, t1;
        bool empty;
        tile_range(bh, qt, part, t0, t1, empty);
        const uint32_t lim = empty ? 0u : row_limit(bh, i_row);
        const int lim_min = empty ? 0 : static_cast<int>(row_limit(bh, i0));  // smallest limit of the warp's rows
        const int nb = bound_tiles(bh, qt, t0, t1, empty);
        if (nb > 0) {
          const BoundSplit split = bound_split(N, nb, classes);
          const int group = split.group, M = split.n;
          list.bound_begin(M);
          int slot = 0;
          auto stretch = [&](auto g) {
            constexpr int G = decltype(g)::value;
            for (int i = 0; i < nb; ++i, ++acc_it) {
              const int b = rt * NACC + acc_it % NACC;
              if (!warp_wait(&acc_full[b], (acc_it / NACC) & 1u, ctl, abort_flag)) {
                ok = false;
                break;
              }
              tc_fence_after();
              list.template bound_tile<N, G>(tmem_base + lane_base + static_cast<uint32_t>(b * N), slot);
              tc_fence_before();
              __syncwarp();
              mbar_arrive_if(lane == 0, &acc_empty[b]);
              slot = slot + N / G >= M ? 0 : slot + N / G;
            }
          };
          if (group == 64)
            stretch(std::integral_constant<int, 64>{});
          else if (group == 32)
            stretch(std::integral_constant<int, 32>{});
          else if (group == 16)
            stretch(std::integral_constant<int, 16>{});
          else if (group == 8)
            stretch(std::integral_constant<int, 8>{});
          else
            stretch(std::integral_constant<int, 4>{});
          if (!ok) break;
          const float t = list.bound_end(M);
          if (i_row < Lq) tau0 = t;
        }
        list.begin(tau0);
        for (int kt = t0; kt < t1; ++kt, ++acc_it) {
          if constexpr (LONG)
            if (kt % kStretch == 0 && kt > t0) list.next_stretch();
          const int b = rt * NACC + acc_it % NACC;
          if (!warp_wait(&acc_full[b], (acc_it / NACC) & 1u, ctl, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t taddr = tmem_base + lane_base + static_cast<uint32_t>(b * N);
          const uint32_t jt = static_cast<uint32_t>(kt * N);
          const bool masked = static_cast<int>(jt) + N > lim_min;  // some key is not valid for some row
#pragma unroll 1
          for (int c = 0; c < N; c += kOffer) {
            float va[kOffer], ma[kOffer / 8];
            load_chunk<kOffer / 8>(taddr + c, va, ma);
            tmem_wait_tied(va, ma);
            if (c + kOffer == N) {
              tc_fence_before();
              __syncwarp();
              mbar_arrive_if(lane == 0, &acc_empty[b]);
            }
            if (masked) {  // a group's maximum is then taken over its valid keys
#pragma unroll
              for (int e = 0; e < kOffer; ++e)
                if (jt + c + e >= lim) va[e] = -INFINITY;
#pragma unroll
              for (int g = 0; g < kOffer / 8; ++g)
                ma[g] = max3f(max3f(va[8 * g], va[8 * g + 1], va[8 * g + 2]),
                              max3f(va[8 * g + 3], va[8 * g + 4], va[8 * g + 5]), fmaxf(va[8 * g + 6], va[8 * g + 7]));
            }
            list.template offer<kOffer / 8>(va, ma, jt + c);
          }
        }
        if (!ok) break;
        list.finish(parts > 1 ? 0 : hand - topk);
        const int list_n = list.count();
        __syncwarp();  // the lists are read across lanes below
        if (parts > 1) {  // this part's kept keys, for the merge
          const size_t prow0 = (static_cast<size_t>(part) * BH + bh) * Lq + i0;
          for (int r = 0; r < 32 && i0 + r < Lq; ++r) {
            const int n = __shfl_sync(0xffffffffu, list_n, r);
            for (int t = lane; t < n; t += 32) part_keys[(prow0 + r) * topk + t] = list_at(job, r, t, t0, t1);
          }
          if (i_row < Lq) part_n[prow0 + lane] = list_n;
          __syncwarp();
        } else if constexpr (L::kPark) {
          // slot s % SL last held unit s - SL, whose epilogue must be done
          if (s >= L::SL) {
            for (int h = 0; ok && h < L::NS; ++h)
              ok = wait_count(&ep_done[job * L::NS + h], s - L::SL + 1, ctl, abort_flag);
            if (!ok) break;
          }
          const size_t slot = (static_cast<size_t>(blockIdx.x) * NJ + job) * L::SL + s % L::SL;
          uint2* pk = park + slot * 32 * hand;
          for (int r = 0; r < 32; ++r) {
            const int n = __shfl_sync(0xffffffffu, list_n, r);
            for (int t = lane; t < n; t += 32) pk[r * hand + t] = list_at(job, r, t, t0, t1);
          }
          park_n[slot * 32 + lane] = list_n;
          __syncwarp();
          st_release_u32(&pk_done[job], s + 1);
        } else {
          row_n[job * 32 + lane] = list_n;
          __syncwarp();
          st_release_u32(&pk_done[job], s + 1);
        }
      }
    }
  } else if (warp >= 4 && parts == 1) {
    // ------------------------------------------------------------ epilogue
    // Warp e takes RS rows of filter warp e / NS, then of filter warp
    // (e + NE) / NS ..., unit by unit.
    const int e = warp - (4 + 4 * RT);
    uint2* buf = reinterpret_cast<uint2*>(list_mem + NJ * List::bytes(cap)) + e * topk;
    uint32_t s = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x, ++s) {
      int bh, qt, part;
      decode(u, bh, qt, part);
      int t0, t1;
      bool empty;
      tile_range(bh, qt, part, t0, t1, empty);
      for (int w = e; w < NJ * L::NS; w += NE) {
        const int job = w / L::NS, r0 = (w % L::NS) * L::RS;
        if (!wait_count(&pk_done[job], s + 1, ctl, abort_flag)) {
          ok = false;
          break;
        }
        const int i0 = qt * RU + (job / NQ) * BM + (job % NQ) * 32 + r0;
        const __nv_bfloat16* vb = v + static_cast<size_t>(bh) * Lk * D;
        const size_t slot = (static_cast<size_t>(blockIdx.x) * NJ + job) * L::SL + s % L::SL;
        int nv = 0;  // lane r: the kept count of row r
        if (lane < L::RS) {
          if constexpr (L::kPark)
            nv = __ldcg(park_n + slot * 32 + r0 + lane);
          else
            nv = row_n[job * 32 + r0 + lane];
        }
        for (int r = 0; r < L::RS && i0 + r < Lq; ++r) {
          const int n = __shfl_sync(0xffffffffu, nv, r);
          const size_t orow = static_cast<size_t>(bh) * Lq + i0 + r;
          int32_t* ir = idx ? idx + orow * topk : nullptr;
          float* fr = score ? score + orow * topk : nullptr;
          auto go = [&](auto&& load) {
            // k + 32 candidates at most, rounded up to whole slots of 32
            if constexpr (L::kPark) {
              if (topk <= 32)
                finish_row<__nv_bfloat16, D, 2, 1>(load, n, topk, buf, vb, out + orow * D, ir, fr);
              else if (topk <= 64)
                finish_row<__nv_bfloat16, D, 3, 2>(load, n, topk, buf, vb, out + orow * D, ir, fr);
              else if (topk <= 128)
                finish_row<__nv_bfloat16, D, 5, 4>(load, n, topk, buf, vb, out + orow * D, ir, fr);
              else if constexpr (RT == 1)
                finish_row<__nv_bfloat16, D, 9, 8>(load, n, topk, buf, vb, out + orow * D, ir, fr);
            } else {
              if (topk <= 256)
                finish_row<__nv_bfloat16, D, 9, 8>(load, n, topk, buf, vb, out + orow * D, ir, fr);
              else
                finish_row<__nv_bfloat16, D, 17, 16>(load, n, topk, buf, vb, out + orow * D, ir, fr);
            }
          };
          if constexpr (L::kPark) {
            const uint2* pk = park + (slot * 32 + r0 + r) * hand;
            go([pk](int t) { return __ldcg(pk + t); });
          } else {
            go([&, r](int t) { return list_at(job, r0 + r, t, t0, t1); });
          }
        }
        __syncwarp();
        st_release_u32(&ep_done[w], s + 1);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, L::TMEM_COLS);
  }
}

// Key parts per query tile: split only grids that would leave at least half
// the SMs idle (a few query tiles against many keys), into as many parts as
// fill the SMs in one wave, each with at least 4 key tiles.
constexpr int kMaxParts = 8;
int tc_parts(const AttnArgs& a, int num_sms, int N, int ru) {
  const long long units = static_cast<long long>(a.B) * a.H * ((a.Lq + ru - 1) / ru);
  if (units * 2 > num_sms) return 1;
  const int kend_min = a.causal ? std::min(a.Lk, ru + (a.Lk - a.Lq)) : a.Lk;  // query tile 0's key range
  const int nk_min = (kend_min + N - 1) / N;
  long long p = num_sms / units;
  p = std::min<long long>(p, nk_min / 4);
  p = std::min<long long>(p, kMaxParts);
  return static_cast<int>(std::max<long long>(p, 1));
}

size_t parts_bytes(const AttnArgs& a, int parts) {
  if (parts <= 1) return 0;
  const size_t rows = static_cast<size_t>(a.B) * a.H * a.Lq;
  return static_cast<size_t>(parts) * rows * (static_cast<size_t>(a.topk) * 8 + 4);
}

// The bound pass covers 1 / divisor of the keys.  A share f of n keys costs f n and
// leaves about k / f candidates to append, so the best share goes with the root of
// k / n: the divisor is the largest power of two up to sqrt(n / (k per)).  `per` is
// smaller where a key of the bound pass costs more: at d = 128 (twice the MMA work),
// and where every call reads the keys from device memory (few positions per head
// against more keys than several times the 129 MB of L2).  At d = 64 lists of less
// than 1.5 k slots prune for every few candidates, and there all of the keys pay.
// us, all of the keys / the divisor's share:
//   d = 64    131,072 keys, 2 heads, k = 16: 9242 / 7920 (4); k = 64: 12191, halved 13453
//             16,384 keys, 1 head, k = 8: 233 / 219 (2); k = 32: 262, halved 269
//   d = 128   8,192 keys, 12 heads, k = 1: 857 / 614 (8); k = 16: 967 / 878 (2)
//             32,768 keys, 8 heads, causal, k = 128: 7134, halved 7453
//   one position, 256 heads, 65,536 keys, d = 64, k = 16: 1391 / 850 (8); k = 128: 1488 / 1375 (2)
int bound_divisor(const AttnArgs& a, int cap, int recs) {
  const bool from_memory = a.Lq <= BM / 2 && 2.0 * a.B * a.H * a.Lk * a.d > 512e6;
  if (!from_memory && a.d == 64 && 2 * cap < 3 * a.topk) return 1;
  const int per = from_memory ? (a.d == 64 ? 40 : 16) : a.d == 64 ? 512 : recs == 8 ? 64 : 128;
  const long long keys = a.causal ? a.Lk - a.Lq / 2 : a.Lk;
  int div = 1;
  while (div < 16 && 4LL * div * div * per * a.topk <= keys) div *= 2;
  return div;
}

// Rows (warps) per block of the merge: eight, or what their candidates leave room
// for (8 parts of k = 455 and more).
constexpr size_t merge_row_bytes(int parts, int topk) { return static_cast<size_t>(parts) * topk * sizeof(uint2); }
constexpr int kMergeWarps = 8;
constexpr int merge_warps(int parts, int topk) {
  const size_t fit = kMaxSmem / merge_row_bytes(parts, topk);
  return fit < kMergeWarps ? static_cast<int>(fit) : kMergeWarps;
}

// Merges a row's `parts` kept lists (each the exact top k of its key range, in
// index order, so their union holds the row's top k), one warp per row.  The
// k-th largest score of the union is found bit by bit on the ordered scores
// (below the bits all of them share), the keys above it and the first ties at
// it are compacted in place (part-major order is index order), and the row is
// finished as in the single-pass kernel.
template <int D, int KPL>
__global__ void __launch_bounds__(kMergeWarps * 32)
    attn_merge_kernel(const uint2* __restrict__ part_keys, const int* __restrict__ part_n, int parts, int BH, int Lq,
                      int Lk, int topk, const __nv_bfloat16* __restrict__ v, __nv_bfloat16* __restrict__ out,
                      int32_t* __restrict__ idx, float* __restrict__ score) {
  extern __shared__ uint2 mk_all[];  // [warps][parts * topk]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  uint2* mk = mk_all + static_cast<size_t>(warp) * parts * topk;
  const long long rows = static_cast<long long>(BH) * Lq;
  for (long long r = static_cast<long long>(blockIdx.x) * warps + warp; r < rows;
       r += static_cast<long long>(gridDim.x) * warps) {
    int P = 0;
    uint32_t hi = 0u, lo = 0xffffffffu;
    for (int p = 0; p < parts; ++p) {
      const long long pr = static_cast<long long>(p) * rows + r;
      // counts and keys are checked before use: after a kernel that stopped
      // early (a wait ran out) they may never have been written
      const int n = min(max(__ldg(part_n + pr), 0), topk);
      for (int t0 = 0; t0 < n; t0 += 32) {
        const int t = t0 + lane;
        uint2 e = make_uint2(0u, 0u);
        bool live = t < n;
        if (live) {
          e = __ldg(part_keys + pr * topk + t);
          live = e.y < static_cast<uint32_t>(Lk);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, live);
        if (live) {
          const uint32_t o = ord_f32(__uint_as_float(e.x));
          mk[P + __popc(bal & ((1u << lane) - 1u))] = make_uint2(o, e.y);
          hi = max(hi, o);
          lo = min(lo, o);
        }
        P += __popc(bal);
      }
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    __syncwarp();
    int n = P;
    if (P > topk) {
      uint32_t thr = hi;
      int c_thr = 0;  // entries >= thr, once a probe has counted them
      if (lo != hi) {
        const int top = 31 - __clz(lo ^ hi);
        thr = top == 31 ? 0u : hi & ~((2u << top) - 1u);
        c_thr = P;
        for (int b = top; b >= 0 && c_thr != topk; --b) {
          const uint32_t cand = thr | (1u << b);
          int c = 0;
          for (int i = lane; i < P; i += 32) c += mk[i].x >= cand ? 1 : 0;
          c = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(c)));
          if (c >= topk) {
            thr = cand;
            c_thr = c;
          }
        }
      }
      // keep what is above thr and, where more than k entries reach it, the
      // first of those equal to it
      int above = 0;
      for (int i = lane; i < P; i += 32) above += mk[i].x > thr ? 1 : 0;
      above = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(above)));
      int eq_left = c_thr == topk ? P : topk - above;
      int w = 0;
      for (int i0 = 0; i0 < P; i0 += 32) {
        const int i = i0 + lane;
        const uint2 e = i < P ? mk[i] : make_uint2(0u, 0u);
        const bool eq = i < P && (c_thr == topk ? e.x >= thr : e.x == thr);
        const unsigned beq = __ballot_sync(0xffffffffu, eq);
        const unsigned below = (1u << lane) - 1u;
        const bool take = (i < P && e.x > thr) || (eq && __popc(beq & below) < eq_left);
        const unsigned bt = __ballot_sync(0xffffffffu, take);
        eq_left -= __popc(beq);
        if (take) mk[w + __popc(bt & below)] = e;
        w += __popc(bt);
        __syncwarp();
      }
      n = min(w, topk);
    }
    const int bh = static_cast<int>(r / Lq);
    finish_kept<__nv_bfloat16, D, KPL>(
        [mk](int t) { return make_uint2(__float_as_uint(unord_f32(mk[t].x)), mk[t].y); }, n, topk,
        v + static_cast<size_t>(bh) * Lk * D, out + r * D, idx ? idx + r * topk : nullptr,
        score ? score + r * topk : nullptr);
    __syncwarp();
  }
}

template <int D, int KPL>
int launch_merge(const AttnArgs& a, const uint2* part_keys, const int* part_n, int parts, int num_sms,
                 cudaStream_t st) {
  const int warps = merge_warps(parts, a.topk);
  const size_t msmem = warps * merge_row_bytes(parts, a.topk);
  auto merge = attn_merge_kernel<D, KPL>;
  if (msmem > 48 * 1024 &&
      cudaFuncSetAttribute(merge, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(msmem)) != cudaSuccess)
    return -1;
  const long long rows = static_cast<long long>(a.B) * a.H * a.Lq;
  long long mgrid = (rows + warps - 1) / warps;
  if (mgrid > 16LL * num_sms) mgrid = 16LL * num_sms;
  merge<<<static_cast<unsigned>(mgrid), warps * 32, msmem, st>>>(
      part_keys, part_n, parts, a.B * a.H, a.Lq, a.Lk, a.topk, static_cast<const __nv_bfloat16*>(a.v),
      static_cast<__nv_bfloat16*>(a.out), a.idx, a.score);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// What a kernel variant needs for a call.
struct TcPlan {
  int parts = 1, n_units = 0, grid = 0;
  size_t park = 0, bytes = 0;  // of device scratch: parked lists, in all
  size_t breaks = 0;           // where in it the break counts begin
  bool fits = false;           // the lists of topk entries fit in shared memory
};

template <int D, bool LONG, int RT, int RPU, int RECS>
struct Variant {
  using L = Layout<D, LONG, RT, RPU, RECS>;

  static TcPlan plan(const AttnArgs& a, int num_sms) {
    TcPlan p;
    constexpr int RU = RT * RPU;
    p.fits = L::fits(a.topk);
    p.parts = RT == 1 ? tc_parts(a, num_sms, L::N, RPU) : 1;
    p.n_units = a.B * a.H * ((a.Lq + RU - 1) / RU) * p.parts;
    p.grid = p.n_units < num_sms ? p.n_units : num_sms;
    if (!p.fits) return p;
    // for as many CTAs as units of one query tile would have: whether two share a
    // unit may depend on what topk_attn_workspace_bytes() is not told
    const int ctas = std::min(RT * p.n_units, num_sms);
    p.park = p.parts == 1 ? L::park_bytes(ctas, a.topk) : 0;
    p.bytes = p.park + parts_bytes(a, p.parts);
    if (LONG && p.parts == 1 && L::breaks_in_park(a.topk, a.Lk)) {
      p.breaks = static_cast<size_t>(p.grid) * L::NJ * L::SL * 32 * L::hand(a.topk, a.Lk) * sizeof(uint2);
    } else if (LONG) {
      p.breaks = p.bytes;
      p.bytes += static_cast<size_t>(ctas) * L::NJ * L::breaks(a.Lk) * 32 * sizeof(uint16_t);
    }
    return p;
  }

  static int launch(const AttnArgs& a, const DevCtl& ctl, int num_sms, cudaStream_t st) {
    const int BH = a.B * a.H;
    const TcPlan p = plan(a, num_sms);
    if (!p.fits) return 0;
    CUtensorMap tmq, tmk;
    if (!make_tmap_bf16_3d(&tmq, a.q, D, a.Lq, BH, BM)) return -1;
    if (!make_tmap_bf16_3d(&tmk, a.k, D, a.Lk, BH, L::N)) return -1;
    // At least 120 KB so that a second CTA never shares the SM: each CTA takes
    // all TMEM columns it needs for its whole (persistent) lifetime.
    const size_t smem = std::max<size_t>(L::bytes(a.topk), 120 * 1024);
    auto kern = attn_tc_kernel<D, LONG, RT, RPU, RECS>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) !=
        cudaSuccess)
      return -1;
    if (p.bytes && (!a.workspace || a.workspace_bytes < p.bytes)) return -1;
    uint8_t* ws = static_cast<uint8_t*>(a.workspace);
    uint2* park = nullptr;
    int* park_n = nullptr;
    if (p.park) {
      park = reinterpret_cast<uint2*>(ws);
      park_n = reinterpret_cast<int*>(park + static_cast<size_t>(p.grid) * L::park_keys_per_cta(a.topk));
    }
    uint2* part_keys = nullptr;
    int* part_n = nullptr;
    if (p.parts > 1) {
      const size_t rows = static_cast<size_t>(BH) * a.Lq;
      part_keys = reinterpret_cast<uint2*>(ws + p.park);
      part_n = reinterpret_cast<int*>(part_keys + static_cast<size_t>(p.parts) * rows * a.topk);
      // counts start at 0, so that rows a stopped kernel never reached merge as empty
      if (cudaMemsetAsync(part_n, 0, static_cast<size_t>(p.parts) * rows * sizeof(int), st) != cudaSuccess) return -1;
    }
    kern<<<p.grid, kThreads, smem, st>>>(tmq, tmk, static_cast<const __nv_bfloat16*>(a.v),
                                         static_cast<__nv_bfloat16*>(a.out), BH, a.H, a.Lq, a.Lk, a.topk,
                                         L::cap(a.topk), L::hand(a.topk, a.Lk), L::classes(a.topk),
                                         bound_divisor(a, L::cap(a.topk), RECS), a.causal, a.kv_len, p.n_units,
                                         p.parts, part_keys, part_n, a.idx, a.score, park, park_n,
                                         LONG ? reinterpret_cast<uint16_t*>(ws + p.breaks) : nullptr, ctl);
    if (cudaGetLastError() != cudaSuccess) return -1;
    if (p.parts == 1) return 1;
    int rc;
    if (a.topk <= 64)
      rc = launch_merge<D, 2>(a, part_keys, part_n, p.parts, num_sms, st);
    else if (a.topk <= 128)
      rc = launch_merge<D, 4>(a, part_keys, part_n, p.parts, num_sms, st);
    else if (a.topk <= 256)
      rc = launch_merge<D, 8>(a, part_keys, part_n, p.parts, num_sms, st);
    else
      rc = launch_merge<D, 16>(a, part_keys, part_n, p.parts, num_sms, st);
    return rc == 0 ? 2 : -1;
  }
};

// Whether units of two query tiles are faster than units of one.  They share each
// key tile and give an SM eight filter warps instead of four (L = 65,536, k = 64:
// 17.9 ms against 31.8), but they leave the epilogue four warps for 256 rows instead
// of eight for 128.  It has to keep up with the filters, so rows need 8,192 keys
// (L = 4,096, k = 16, H = 12: 353 us against 263) and 128 k of them, twice that where
// it also orders the selection (L = 16,384, causal, H = 8, k = 64: 1505 against 1328;
// k = 32: 1036 against 1091).  And a grid of half the units, each 1.4 (from 512 k keys
// on) to 1.6 times as long, has to end sooner: waves of units over the SMs are
// compared (L = 8,192, k = 64, H = 6: three waves 517, two 609; L = 16,384, k = 16,
// H = 3: three waves 654, two 537; 8,192 rows, 131,072 keys, k = 64, H = 4: 2729, 2085).
bool two_query_tiles(const AttnArgs& a, int num_sms) {
  const long long keys = a.causal ? a.Lk - a.Lq / 2 : a.Lk, k = a.topk;
  if (keys < 8192 || keys < (a.idx || a.score ? 256 : 128) * k) return false;
  auto waves = [&](int rows) {
    return (static_cast<long long>(a.B) * a.H * ((a.Lq + rows - 1) / rows) + num_sms - 1) / num_sms;
  };
  const long long w1 = waves(BM), w2 = waves(2 * BM);
  // a single tile's rows: the second tile is empty, but with four records an offer
  // that no row passes takes one vote less (one position, 256 heads, 65,536 keys,
  // k = 16: 870 us against 1078)
  if (a.Lq <= BM) return w1 > 1 && !a.idx && !a.score;
  if (w2 == 1 && keys < 256 * k) return false;  // 8,192 keys, k = 64, H = 4: 376 us against 358
  return 5 * w1 > (keys >= 512 * k ? 7 : 8) * w2;
}

// Which variant serves a call: f is called with the Variant, which may not fit
// (TcPlan::fits); the call is then not served here.
// - Two query tiles per unit where their lists fit (d = 64, k up to 68) and
//   two_query_tiles() says so.
// - Else one query tile; and, for k beyond what 128 rows' lists can hold, units
//   of 64 or 32 query rows.
// Eight records per row and 32 scores per offer, but two query tiles leave room
// for four records.  At d = 128 the larger query and key tiles do so as well once
// k is large: the lists there have to hold 1.5 k (k up to 90), or they prune all
// the time, and four records with 16 scores per offer are the better split.
// L = 8,192, H = 12, d = 128, four records and eight: k = 16: 1105 and 967 us,
// k = 64: 1420 and 1222; L = 1,000, k = 100: 163 and 167.
// Units of 128 rows whose lists hold fewer than k + 16 entries (k = 137 to 140) pay
// only for rows of 16 k keys: short ones have no bound pass, and every eighth entry
// prunes (H = 12, k = 140: L = 300: 231 us against 93 with units of 64 rows, 2,048:
// 466 against 349, 4,096: 852 against 957).
template <typename L>
bool lists_pay(const AttnArgs& a) {
  return L::fits(a.topk) && (L::cap(a.topk) >= a.topk + 16 || (a.causal ? a.Lk - a.Lq / 2 : a.Lk) >= 16 * a.topk);
}

template <int D, bool LONG, typename F>
auto with_variant_i(const AttnArgs& a, int num_sms, F&& f) {
  if constexpr (D == 64) {
    if (Layout<D, LONG, 2, BM, 4>::fits(a.topk) && two_query_tiles(a, num_sms))
      return f(Variant<D, LONG, 2, BM, 4>{});
    if (lists_pay<Layout<D, LONG, 1, BM, 8>>(a)) return f(Variant<D, LONG, 1, BM, 8>{});
  } else {
    if (2 * Layout<D, LONG, 1, BM, 8>::cap(a.topk) >= 3 * a.topk) return f(Variant<D, LONG, 1, BM, 8>{});
    if (lists_pay<Layout<D, LONG, 1, BM, 4>>(a)) return f(Variant<D, LONG, 1, BM, 4>{});
  }
  if (Layout<D, LONG, 1, 64, 8>::fits(a.topk)) return f(Variant<D, LONG, 1, 64, 8>{});
  return f(Variant<D, LONG, 1, 32, 8>{});
}

template <int D, typename F>
auto with_variant(const AttnArgs& a, int num_sms, F&& f) {
  return a.Lk <= 65536 ? with_variant_i<D, false>(a, num_sms, f) : with_variant_i<D, true>(a, num_sms, f);
}

// The two calls of attn_tc.cu for one head size.
template <int D>
size_t tc_bytes(const AttnArgs& a, int num_sms) {
  return with_variant<D>(a, num_sms, [&](auto v) { return decltype(v)::plan(a, num_sms).bytes; });
}

template <int D>
int tc_launch(const AttnArgs& a, const DevCtl& ctl, int num_sms, cudaStream_t st) {
  return with_variant<D>(a, num_sms, [&](auto v) { return decltype(v)::launch(a, ctl, num_sms, st); });
}

}  // namespace

}  // namespace topk
