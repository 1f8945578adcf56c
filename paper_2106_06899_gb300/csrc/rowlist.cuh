// rowlist.cuh -- exact streaming top-k of 32 rows by one warp, one row per lane.
//
// The kept set of a row is the first k entries of the total order (score
// descending, key index ascending): the top-k of Eq. 4 with ties broken toward
// the lower key index.  Keys stream in by ascending index.
//
// Each row keeps a list of candidates (score, index) in shared memory, in index
// order, and a threshold tau such that at least k entries of the list score
// >= tau.  A key can enter the top k only if it scores strictly above tau (an
// equal score has a higher index and ranks below those k), so most keys cost
// the compare of their group's maximum.  When a list is full the warp prunes
// all 32 of its lists in lockstep: a threshold with k to k + kSlack entries at
// or above it is found by counting, the entries below it are dropped in place
// (order kept) and tau rises to it.
//
// Why lists and not a heap: a heap replaces its root for every key above the
// running k-th score, k (1 + ln(n/k)) times per row, and each replacement is a
// dependent chain of about 150 instructions that the warp's lanes rarely share.
// Here a bound taken from group maxima in a first pass over the keys (RowList)
// leaves about 1.4 k candidates per row, each of them an append.  Measured,
// heaps and lists: k = 64, L = 65,536, d = 64: 19.7 and 17.9 ms; k = 128,
// L = 16,384 causal, d = 128: 15.8 and 8.8 ms; k = 256, L = 8,192: 11.3 and
// 3.0 ms; k = 64, L = 512: 250 and 165 us.  What bounds it: the filters' issue
// latency (about five cycles per instruction and warp, two filter warps per SM
// sub-partition at most), not the tensor pipe.  Heaps were faster where one
// filter warp per sub-partition meets few candidates: d = 64, one query tile per
// unit, k up to 32 of more than 8,000 keys (128 positions against 65,536 keys,
// k = 16: 256 and 308 us), and where scores rise along the keys (L = 8,192, k = 64:
// 6.4 and 10.0 ms).
//
// Indices take 16 bits.  Rows of more than 65,536 keys (LONG) also keep, per 65,536
// keys after the first, how many entries of the list come before them (Breaks):
// the list is in key order, so an entry's position gives the rest of its index.
// With 32 bits in the list instead, two query tiles' lists do not fit at k = 64 and
// no lists at all at d = 128, k > 462.  L = 131,072, k = 64, d = 64, two heads: 20.5
// and 12.3 ms; 8,192 rows, 131,072 keys, d = 128, k = 128, four heads: 9.2 and 5.4.
//
// Layout: [slot][row] with a row stride of 33, so that a warp's lockstep passes
// (one slot, 32 rows) and a row's list read by 32 lanes are both free of bank
// conflicts.
#pragma once

#include <stdint.h>

#include "common.cuh"

namespace topk {

// Order-preserving map of fp32 to unsigned integers (-0 folded onto +0).
__device__ __forceinline__ uint32_t ord_f32(float s) {
  const uint32_t u = __float_as_uint(s + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float unord_f32(uint32_t o) {
  const uint32_t u = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
  return __uint_as_float(u);
}

// A (score, index) pair as one 64-bit key whose unsigned order is the total order.
__device__ __forceinline__ uint64_t make_key(float s, uint32_t j) {
  return (static_cast<uint64_t>(ord_f32(s)) << 32) | static_cast<uint64_t>(~j);
}

__device__ __forceinline__ float key_score(uint64_t key) { return unord_f32(static_cast<uint32_t>(key >> 32)); }

__device__ __forceinline__ uint32_t key_index(uint64_t key) { return ~static_cast<uint32_t>(key); }

constexpr int kListStride = 33;  // words between a list's slots (32 rows + 1)
constexpr int kListSlack = 4;    // a prune keeps at most k + kListSlack entries (ties aside)

// Shared-memory accesses by 32-bit address: the prune is a function of its own
// (one copy, so that the filters' loop stays small in the instruction cache),
// which could not tell that a pointer argument is a shared one.
__device__ __forceinline__ float lds_f32(uint32_t a) {
  float x;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
  return x;
}
__device__ __forceinline__ void sts_f32(uint32_t a, float x) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory");
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  unsigned short x;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x) : "r"(a) : "memory");
  return x;
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t x) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(static_cast<unsigned short>(x)) : "memory");
}

// An entry (x, j) stored at as, ai where x passes thr (GE: x >= thr, else
// x > thr), without a branch; as, ai step to the next slot.  The steps go to new
// registers: a store reads its address late, and a predicated step in place
// would wait for that (eight appends take 107 cycles instead of 151).
template <bool GE>
__device__ __forceinline__ void append_if(float x, float thr, uint32_t j, uint32_t& as, uint32_t& ai) {
  if constexpr (GE)
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ge.f32 q, %2, %3;\n\t@q st.shared.f32 [%0], %2;\n\t"
        "@q st.shared.u16 [%1], %4;\n\t}" ::"r"(as),
        "r"(ai), "f"(x), "f"(thr), "h"(static_cast<unsigned short>(j))
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.gt.f32 q, %2, %3;\n\t@q st.shared.f32 [%0], %2;\n\t"
        "@q st.shared.u16 [%1], %4;\n\t}" ::"r"(as),
        "r"(ai), "f"(x), "f"(thr), "h"(static_cast<unsigned short>(j))
        : "memory");
  const bool p = GE ? x >= thr : x > thr;
  as += p ? 4u * kListStride : 0u;
  ai += p ? 2u * kListStride : 0u;
}

constexpr uint32_t kScStep = kListStride * 4;  // bytes between a row's scores
constexpr uint32_t kIxStep = kListStride * 2;  // bytes between their indices

// Entries of a list at or above x among slots 0 .. cr - 1 (cr > 0, pads are -inf),
// counted in floats: the adds then run on the FMA pipe, next to the compares on
// the ALU pipe, which issues at half its rate.
static __device__ __noinline__ float list_count_ge(uint32_t sc, float x, int cr) {
  float c[4] = {0.f, 0.f, 0.f, 0.f};
  float s[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) s[e] = lds_f32(sc + e * kScStep);
#pragma unroll 2
  for (int i = 8; i < cr; i += 8) {  // the next slots' loads are in flight while these are counted
    sc += 8 * kScStep;
    float n[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) n[e] = lds_f32(sc + e * kScStep);
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (s[e] >= x) c[e & 3] += 1.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) s[e] = n[e];
  }
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if (s[e] >= x) c[e & 3] += 1.f;
  return (c[0] + c[1]) + (c[2] + c[3]);
}

// Sum and maximum of the entries in slots 0 .. cr - 1 (pads left out of the sum).
struct ListStats {
  float sum, mx;
};
static __device__ __noinline__ ListStats list_stats(uint32_t sc, int cr) {
  float sum0 = 0.f, sum1 = 0.f, mx = -INFINITY;
#pragma unroll 2
  for (int i = 0; i < cr; i += 8, sc += 8 * kScStep) {
    float s[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) s[e] = lds_f32(sc + e * kScStep);
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      mx = max3f(mx, s[e], s[e + 1]);
      if (s[e] > -INFINITY) sum0 += s[e];
      if (s[e + 1] > -INFINITY) sum1 += s[e + 1];
    }
  }
  return ListStats{sum0 + sum1, mx};
}

// A threshold that at least k of a row's cnt entries reach and, ties aside, at
// most k + slack do (slack 0: the k-th score's own set).  Called by the whole
// warp, one row per lane; lanes with cnt <= k + slack keep their tau.  The
// slots from cnt up to the warp's largest count (rounded up to 8) become -inf.
//
// The k-th score is bracketed by counts, count(>= lo) >= k > count(>= hi), lo
// and hi as ordered integers.  The first probe assumes an exponential tail
// above the old threshold (the mean excess times ln(count / k)), the next ones
// interpolate between the counts, and after kInterp of them the bracket is
// halved, so at most kInterp + 32 passes end with lo the k-th score itself.
// `eq` is then how many entries equal to tau belong to the k best (the others
// above it do), else a number no list reaches.
struct Threshold {
  float tau;
  int eq;
};
static __device__ __noinline__ Threshold list_threshold(uint32_t sc, int k, int slack, int cnt, float tau) {
  constexpr int kInterp = 6;
  const bool active = cnt > k + slack;
  const int cr = (static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(cnt))) + 7) & ~7;
#pragma unroll 1
  for (int i = cnt; i < cr; ++i) sts_f32(sc + i * kScStep, -INFINITY);
  const ListStats st = list_stats(sc, cr);
  const float mx = st.mx;
  const float target = static_cast<float>(k) + 0.5f * static_cast<float>(slack);
  const float mean = __fdividef(st.sum, static_cast<float>(cnt));
  float flo = tau > -INFINITY ? tau : 2.f * mean - mx, fhi = mx;  // for the interpolation
  uint32_t lo = ord_f32(tau), hi = ord_f32(mx) + 1u;
  float clo = static_cast<float>(cnt), chi = 0.f;
  const float kf = static_cast<float>(k), enough = static_cast<float>(k + slack);
  float t = flo + (mean - flo) * __logf(__fdividef(clo, target));
  bool done = !active;
#pragma unroll 1
  for (int it = 0;; ++it) {
    done = done || clo <= enough || hi - lo <= 1u;
    if (__all_sync(0xffffffffu, done)) break;
    uint32_t mid = it < kInterp ? ord_f32(t) : lo + ((hi - lo) >> 1);
    mid = min(max(mid, lo + 1u), hi - 1u);
    const float x = unord_f32(mid);
    const float c = list_count_ge(sc, x, cr);
    if (!done) {
      if (c >= kf) {
        lo = mid;
        clo = c;
        flo = x;
      } else {
        hi = mid;
        chi = c;
        fhi = x;
      }
      t = flo + (fhi - flo) * __fdividef(clo - target, clo - chi);
    }
  }
  Threshold r;
  r.eq = active && clo > enough ? k - static_cast<int>(chi) : 0x3fffffff;
  r.tau = active ? unord_f32(lo) : tau;
  return r;
}

// Keeps the entries >= thr of slots 0 .. cr - 1, in order; returns the address
// after the last one kept.
static __device__ __noinline__ uint32_t list_compact(uint32_t sc, uint32_t ix, int cr, float thr) {
  uint32_t ws = sc, wi = ix;
#pragma unroll 1
  for (int i = 0; i < cr; i += 8, sc += 8 * kScStep, ix += 8 * kIxStep) {
    float s[8];
    uint32_t j[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      s[e] = lds_f32(sc + e * kScStep);
      j[e] = lds_u16(ix + e * kIxStep);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) append_if<true>(s[e], thr, j[e], ws, wi);
  }
  return ws;
}

// How many of a row's entries come before each further stretch of 65,536 keys
// (device memory, [stretch][row]; p is the lane's column).  Nothing for rows of
// one stretch.
template <bool LONG>
struct Breaks {};
template <>
struct Breaks<true> {
  uint16_t* p;
  int n;  // stretches begun after the unit's first

  // The counts once the entries from thr on (of those equal to it the first eq)
  // are all that is left of slots 0 .. cr - 1.
  __device__ __forceinline__ void move(uint32_t sc, int cr, float thr, int eq) const {
    int e = 0, next = p[0], w = 0;
#pragma unroll 1
    for (int i = 0; i < cr; ++i) {
      while (next == i) {
        p[e * 32] = static_cast<uint16_t>(w);
        next = ++e < n ? p[e * 32] : -1;
      }
      const float s = lds_f32(sc + i * kScStep);
      w += s > thr || (s == thr && eq > 0) ? 1 : 0;
      eq -= s == thr ? 1 : 0;
    }
    for (; e < n; ++e) p[e * 32] = static_cast<uint16_t>(w);
  }
};

// Drops entries that cannot be in the top k, keeping the list order: lists of
// more than k + slack entries go down to between k and k + slack of them (ties
// cut exactly), the others stay as they are; slack 0 leaves the exact top k.
struct Pruned {
  int cnt;
  float tau;
};
template <bool LONG>
static __device__ __noinline__ Pruned list_prune(uint32_t sc, uint32_t ix, int k, int slack, int cnt, float tau0,
                                                 Breaks<LONG> brk) {
  const bool active = cnt > k + slack;
  if (!__any_sync(0xffffffffu, active)) return Pruned{cnt, tau0};
  const Threshold th = list_threshold(sc, k, slack, cnt, tau0);
  int eq = th.eq;
  const int cr = (static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(cnt))) + 7) & ~7;
  const float thr = active ? th.tau : -INFINITY;
  if constexpr (LONG) {
    if (active && brk.n > 0) brk.move(sc, cr, thr, eq);
    __syncwarp();
  }
  uint32_t ws = sc;
  if (__all_sync(0xffffffffu, eq == 0x3fffffff)) {
    ws = list_compact(sc, ix, cr, thr);
  } else {  // some row keeps only the first of its entries equal to thr
    uint32_t wi = ix;
#pragma unroll 1
    for (int i = 0; i < cr; ++i) {
      const float s = lds_f32(sc + i * kScStep);
      const uint32_t j = lds_u16(ix + i * kIxStep);
      const bool is_eq = s == thr;
      if (s > thr || (is_eq && eq > 0)) {
        sts_f32(ws, s);
        sts_u16(wi, j);
        ws += kScStep;
        wi += kIxStep;
      }
      eq -= is_eq ? 1 : 0;
    }
  }
  return active ? Pruned{static_cast<int>((ws - sc) / kScStep), thr} : Pruned{cnt, tau0};
}

// A record (a group's eight scores and its first key index) stored where its
// maximum m passes tau, without a branch.
template <int HI>
__device__ __forceinline__ void record_if(float m, float tau, const float* v, uint32_t j, uint32_t ra, uint32_t rx) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.gt.f32 q, %2, %3;\n\t@q st.shared.v4.f32 [%0], {%4, %5, %6, %7};\n\t"
      "@q st.shared.v4.f32 [%0+%13], {%8, %9, %10, %11};\n\t@q st.shared.u16 [%1], %12;\n\t}" ::"r"(ra),
      "r"(rx), "f"(m), "f"(tau), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]),
      "f"(v[7]), "h"(static_cast<unsigned short>(j)), "n"(HI)
      : "memory");
}
__device__ __forceinline__ void lds_v4(uint32_t a, float& x, float& y, float& z, float& w) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x), "=f"(y), "=f"(z), "=f"(w) : "r"(a) : "memory");
}

// Where a warp's records and lists lie in its shared memory `mem`; lane r's row.
// R records per row.
template <int R>
struct ListMem {
  static constexpr uint32_t kRecStep = 512;  // bytes between a row's records
  static constexpr uint32_t kRixStep = 64;
  static constexpr uint32_t kRecHi = R * kRecStep;  // from a record's scores 0..3 to 4..7
  static constexpr uint32_t kRecBytes = 2 * R * kRecStep + R * kRixStep;

  uint32_t rec;  // shared address of the row's record 0 (scores 0..3)
  uint32_t rix;  // the same of its index
  uint32_t sc;   // shared address of the row's score in list slot 0
  uint32_t ix;   // the same of its index

  __device__ __forceinline__ ListMem(uint32_t mem, int cap) {
    const uint32_t lane = threadIdx.x & 31;
    rec = mem + lane * 16;
    rix = mem + 2 * R * kRecStep + lane * 2;
    sc = mem + kRecBytes + lane * 4;
    ix = mem + kRecBytes + cap * kScStep + lane * 2;
  }
};

// Appends what still passes of every row's records (up to ra) to its list,
// which ends at `as`, pruning the lists when one gets too full; returns the new
// end and tau.
struct ListEnd {
  uint32_t as;
  float tau;
};
template <int R, bool LONG>
static __device__ __noinline__ ListEnd list_expand(uint32_t mem, int cap, int k, uint32_t ra, uint32_t as, float tau,
                                                   Breaks<LONG> brk) {
  using M = ListMem<R>;
  const M l(mem, cap);
  const int rc = static_cast<int>((ra - l.rec) / M::kRecStep);
  const int steps = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(rc)));
  uint32_t ai = l.ix + (as - l.sc) / 2;
  const uint32_t tight = l.sc + (cap - 8) * kScStep;
#pragma unroll 1
  for (int i = 0; i < steps; ++i) {
    float x[8];
    const uint32_t a = l.rec + i * M::kRecStep;
    lds_v4(a, x[0], x[1], x[2], x[3]);
    lds_v4(a + M::kRecHi, x[4], x[5], x[6], x[7]);
    const uint32_t j = lds_u16(l.rix + i * M::kRixStep);
    const bool live = i < rc;
    if (__any_sync(0xffffffffu, as > tight)) {
      const int n = static_cast<int>((as - l.sc) / kScStep);
      int pc = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) pc += live && x[e] > tau ? 1 : 0;
      if (__any_sync(0xffffffffu, n + pc > cap)) {
        const Pruned pr = list_prune<LONG>(l.sc, l.ix, k, kListSlack, n, tau, brk);
        as = l.sc + pr.cnt * kScStep;
        ai = l.ix + pr.cnt * kIxStep;
        tau = pr.tau;
      }
    }
    const float thr = live ? tau : INFINITY;
#pragma unroll
    for (int e = 0; e < 8; ++e) append_if<false>(x[e], thr, j + e, as, ai);
  }
  return ListEnd{as, tau};
}

// The filter's view of its 32 rows.  Every call is made by all 32 lanes.
//
// Scores arrive in groups of eight.  A group whose maximum beats its row's
// threshold is set aside whole (8 scores and its first key index, three
// stores) among the row's R records; when some row gets near R of them, the
// warp expands the records of all its rows in lockstep into the lists.  That keeps
// the work on the path that every passing group takes, mostly for one lane out
// of 32, to a few instructions.
template <int R, bool LONG>
struct RowList {
  using M = ListMem<R>;
  uint32_t mem;  // the warp's memory: records, then lists
  int cap;       // list slots, a multiple of 8, at least k + kListSlack + 8
  int k;
  uint32_t ra;   // where the next record goes
  uint32_t as;   // where the next entry's score goes
  float tau;     // at least k keys seen score >= tau (-inf until that is known)
  Breaks<LONG> brk;

  // bytes of one warp's records and lists (a multiple of 16)
  __host__ __device__ static constexpr size_t bytes(int cap_) {
    return M::kRecBytes + ((static_cast<size_t>(cap_) * kListStride * 6 + 15) & ~size_t(15));
  }

  __device__ __forceinline__ void bind(const uint8_t* mem_, int cap_, int k_) {
    mem = smem_u32(mem_);
    cap = cap_;
    k = k_;
  }

  // Empty lists under the threshold tau (+inf for a row that takes no part).
  __device__ __forceinline__ void begin(float tau_) {
    if constexpr (LONG) brk.n = 0;
    ra = mem + (threadIdx.x & 31) * 16;
    as = M(mem, cap).sc;
    tau = tau_;
  }

  __device__ __forceinline__ int count() const { return static_cast<int>((as - M(mem, cap).sc) / kScStep); }

  // A bound before the first key.  The keys of a first stretch fall into M
  // classes (M > k); the k-th largest of the class maxima is a lower bound of
  // the k-th score, since k different keys reach it.  The maxima take the
  // warp's memory, one slot after the other.
  __device__ __forceinline__ void bound_begin(int M) {
    const uint32_t a = mem + (threadIdx.x & 31) * 4;
#pragma unroll 8
    for (int b = 0; b < M; ++b) sts_f32(a + b * kScStep, -INFINITY);
  }
  // One tile of N columns at TMEM address taddr, in groups of G: slots slot ..
  // slot + N / G - 1.
  template <int N, int G>
  __device__ __forceinline__ void bound_tile(uint32_t taddr, int slot) const {
    constexpr int W = G == 64 ? 64 : 32;  // columns at a time: their loads hold W registers
    constexpr int NG = W / G;
    const uint32_t a = mem + (threadIdx.x & 31) * 4 + slot * kScStep;
#pragma unroll
    for (int h = 0; h < N / W; ++h) {
      float m[NG], c[NG];
#pragma unroll
      for (int g = 0; g < NG; ++g) m[g] = tmem_ld_max<G>(taddr + h * W + g * G);
#pragma unroll
      for (int g = 0; g < NG; ++g) c[g] = lds_f32(a + (h * NG + g) * kScStep);
      tmem_wait_ld();
#pragma unroll
      for (int g = 0; g < NG; ++g) asm volatile("" : "+f"(m[g]));
#pragma unroll
      for (int g = 0; g < NG; ++g) sts_f32(a + (h * NG + g) * kScStep, fmaxf(c[g], m[g]));
    }
  }
  // The largest number below the bound: a key that scores exactly the bound
  // still passes, as the k keys that support it may have any index.
  __device__ __forceinline__ float bound_end(int M) const {
    const float t = list_threshold(mem + (threadIdx.x & 31) * 4, k, max(kListSlack, k / 8), M, -INFINITY).tau;
    __syncwarp();
    const uint32_t below = ord_f32(t) - 1u;
    return t > -INFINITY ? unord_f32(below == 0x7fffffffu ? below - 1u : below) : t;  // below +0 comes -0, its equal
  }

  // Offer 8 G scores with key indices j0 ..; m[g] is the maximum of group g of
  // eight (NaN ignored).  The votes of all groups come first, so that their
  // latencies overlap; a group that no lane passes costs a branch more.  With
  // more than G records per row they are expanded between offers only, when a
  // row may not have room for G more: the scores are out of their registers
  // then.  With G or fewer, as soon as a row has R.
  template <int G>
  __device__ __forceinline__ void offer(const float (&v)[8 * G], const float (&m)[G], uint32_t j0) {
    const float t = tau;
    bool any[G];
#pragma unroll
    for (int g = 0; g < G; ++g) any[g] = __any_sync(0xffffffffu, m[g] > t);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (any[g]) {
        const uint32_t rx = mem + 2 * R * M::kRecStep + (ra - mem) / 8;
        record_if<static_cast<int>(M::kRecHi)>(m[g], t, v + 8 * g, j0 + 8 * g, ra, rx);
        ra += m[g] > t ? M::kRecStep : 0u;
        if (R <= G && __any_sync(0xffffffffu, ra >= mem + R * M::kRecStep)) expand();
      }
    }
    if (R > G && __any_sync(0xffffffffu, ra >= mem + (R - G + 1) * M::kRecStep)) expand();
  }

  __device__ __forceinline__ void expand() {
    const ListEnd r = list_expand<R, LONG>(mem, cap, k, ra, as, tau, brk);
    as = r.as;
    tau = r.tau;
    ra = mem + (threadIdx.x & 31) * 16;
  }

  // The next keys' indices are the first of another stretch of 65,536.
  __device__ __forceinline__ void next_stretch() {
    expand();
    brk.p[brk.n * 32] = static_cast<uint16_t>(count());
    ++brk.n;
  }

  // The unit's last records, then lists of at most k + slack entries.
  __device__ __forceinline__ void finish(int slack) {
    expand();
    const M l(mem, cap);
    as = l.sc + list_prune<LONG>(l.sc, l.ix, k, slack, count(), tau, brk).cnt * kScStep;
  }
};

}  // namespace topk
