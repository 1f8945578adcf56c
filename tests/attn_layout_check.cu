// Host-side check of the tensor-core attention kernel's shared-memory plans: prints one line per
// violation and exits non-zero if there is any.  No kernel is launched.
#include <cstdio>

#include "attn_tc.cuh"

using namespace topk;

namespace {

int bad = 0;

// Every number of bound tiles (until the split no longer changes): the slots that the tiles write, one
// tile after the other, lie below the class count and inside the warp's memory, and there are more than k.
template <int D, typename IdxT, int RT, int RPU>
void bound_slots() {
  using L = Layout<D, IdxT, RT, RPU>;
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
        std::printf("D %d index bytes %zu RT %d RPU %d k %d: %d bound tiles write %d of %d slots, %zu bytes of memory\n", D,
                    sizeof(IdxT), RT, RPU, k, nb, top, s.n, mem);
        ++bad;
        break;
      }
    }
  }
}

template <int D, typename IdxT>
void check() {
  bound_slots<D, IdxT, 2, BM>();
  bound_slots<D, IdxT, 1, BM>();
  bound_slots<D, IdxT, 1, 64>();
  bound_slots<D, IdxT, 1, 32>();
}

}  // namespace

int main() {
  check<64, uint16_t>();
  check<64, uint32_t>();
  check<128, uint16_t>();
  check<128, uint32_t>();
  std::printf("%d violations\n", bad);
  return bad != 0;
}
