// Host-side check of the tensor-core attention kernel's shared-memory plans: prints one line per
// violation and exits non-zero if there is any.  No kernel is launched.
#include <cstdio>

#include "attn_tc.cuh"

using namespace topk;

namespace {

int bad = 0;

// Every number of bound tiles (until the split no longer changes): the slots that the tiles write, one
// tile after the other, lie below the class count and inside the warp's memory, and there are more than k.
template <int D, int RT, int RPU, int RECS>
void bound_slots() {
  using L = Layout<D, false, RT, RPU, RECS>;
  for (int k = 1; k <= kTcMaxK; ++k) {
    if (!L::fits(k)) continue;
    const int classes = L::classes(k);
    const size_t mem = L::List::bytes(L::cap(k));
    for (int nb = (6 * k + L::N - 1) / L::N; (nb - 1) * L::N <= 64 * classes; ++nb) {
      const BoundSplit s = bound_split(L::N, nb, classes);
      const int per = L::N / s.group;
      int top = 0;
      for (int i = 0, slot = 0; i < nb && top <= s.n; ++i) {
        top = slot + per > top ? slot + per : top;
        slot = slot + per >= s.n ? 0 : slot + per;
      }
      if (top > s.n || s.n <= k || static_cast<size_t>(top) * kScStep > mem) {
        std::printf("D %d RT %d RPU %d RECS %d k %d: %d bound tiles write %d of %d slots, %zu bytes of memory\n", D, RT, RPU,
                    RECS, k, nb, top, s.n, mem);
        ++bad;
        break;
      }
    }
  }
}

// Every call is served, by a variant that has room for its lists.
template <int D>
void picked() {
  for (int Lk : {600, 65536, 65537, 1000000})
    for (int Lq : {1, 130, 5000})
      for (int k = 1; k <= kTcMaxK; ++k) {
        AttnArgs a{};
        a.B = 1, a.H = 8, a.Lq = Lq, a.Lk = Lk, a.d = D, a.topk = k, a.dtype = 1;
        with_variant<D>(a, 152, [&](auto v) {
          using V = decltype(v);
          const TcPlan p = V::plan(a, 152);
          const int cap = V::L::cap(k);
          const bool room = cap >= V::L::min_cap(k) && V::L::bytes(k) <= kMaxSmem;
          if (!p.fits || !room) {
            std::printf("D %d Lq %d Lk %d k %d: fits %d, %d list slots\n", D, Lq, Lk, k, p.fits, cap);
            ++bad;
          }
          return 0;
        });
      }
}

// The break counts of long rows lie inside the scratch and apart from the lists and counts in it; where
// lists are parked they take none of their own up to 16 million keys.
template <int D>
void breaks() {
  for (int Lk : {65537, 131072, 131073, 1 << 20, 16000000, 40000000})
    for (int Lq : {1, 200, 9000, 40000})
      for (int k = 1; k <= kTcMaxK; ++k) {
        AttnArgs a{};
        a.B = 1, a.H = 8, a.Lq = Lq, a.Lk = Lk, a.d = D, a.topk = k, a.dtype = 1;
        with_variant<D>(a, 152, [&](auto v) {
          using V = decltype(v);
          using L = typename V::L;
          const TcPlan p = V::plan(a, 152);
          const size_t need = static_cast<size_t>(p.grid) * L::NJ * L::breaks(Lk) * 64, end = p.breaks + need;
          const size_t keys = static_cast<size_t>(p.grid) * L::NJ * L::SL * 32 * L::hand(k, Lk) * 8;
          bool ok = end <= p.bytes && L::hand(k, Lk) >= k;
          if (p.park > 0)
            ok = ok && ((p.breaks >= keys && end <= p.grid * L::park_keys_per_cta(k) * 8) || p.breaks >= p.park) &&
                 (p.bytes == p.park || Lk > 16000000);
          else
            ok = ok && p.breaks >= parts_bytes(a, p.parts);
          if (!ok) {
            std::printf("D %d Lq %d Lk %d k %d: breaks at %zu .. %zu of %zu bytes, lists %zu, parked %zu\n", D, Lq, Lk, k,
                        p.breaks, end, p.bytes, keys, p.park);
            ++bad;
          }
          return 0;
        });
      }
}

// The merge of a call's key parts fits in shared memory.
void merges() {
  for (int parts = 2; parts <= kMaxParts; ++parts)
    for (int k = 1; k <= kTcMaxK; ++k) {
      const int w = merge_warps(parts, k);
      if (w < 1 || w > kMergeWarps || w * merge_row_bytes(parts, k) > kMaxSmem) {
        std::printf("merge of %d parts, k %d: %d warps\n", parts, k, w);
        ++bad;
      }
    }
}

template <int D>
void check() {
  bound_slots<D, 2, BM, 4>();
  bound_slots<D, 1, BM, 4>();
  bound_slots<D, 1, BM, 8>();
  bound_slots<D, 1, 64, 8>();
  bound_slots<D, 1, 32, 8>();
  picked<D>();
  breaks<D>();
}

}  // namespace

int main() {
  check<64>();
  check<128>();
  merges();
  std::printf("%d violations\n", bad);
  return bad != 0;
}
