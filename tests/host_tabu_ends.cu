// Host-only check of the rotation layout's tabu ends (RotEnds in
// qap_rotation.cuh): no GPU, no CUDA calls.  Replays the order of an iteration,
// the pairs' slots, the marks and the ring against a plain table of ends, with
// pairs applied again while tabu, over iterations around multiples of 2^15
// (where 16-bit marks wrap) and at the start of a search.  Built and run by
// tests/test_host_tabu_ends.py; prints "ok" and exits 0, or the first violations.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <utility>
#include <vector>

#include "../paper_2307_11248_gb300/csrc/qap_host.cuh"

namespace {
int fails = 0;

template <int RING>
struct HostMem {
  static uint32_t ring_[RING], node_[2 * RING];
  static uint32_t* ring() { return ring_; }
  static uint32_t* node() { return node_; }
};
template <int RING>
uint32_t HostMem<RING>::ring_[RING];
template <int RING>
uint32_t HostMem<RING>::node_[2 * RING];

// Iterations first..last of a search of `iters` (ends beyond it reach no scan,
// and hang nowhere); the moves draw from a few pairs, so that most are tabu when
// applied.
template <int NT, int C, bool LATE>
void replay(int n, int first, int last, int iters, unsigned seed) {
  constexpr int RING = qapk::rot_ring(NT);
  using Mem = HostMem<RING>;
  const int n2 = (n + 1) / 2, J = qapk::rot_chunks(n, NT, C), pairs = n * (n - 1) / 2;
  if (J == 0) {
    std::printf("FAIL shape (%d, %d) does not hold n = %d\n", NT, C, n);
    ++fails;
    return;
  }
  std::vector<int32_t> marks(pairs + 1, 0);
  std::fill(Mem::ring_, Mem::ring_ + RING, 0xffffffffu);
  qapk::RotEnds<NT, C, Mem> ends(n2, qapk::rot_circle(n, C), J, iters, marks.data());
  std::vector<int> tab((size_t)(J * n2) << qapk::rot_slot_bits(NT), 0);  // tabu bits, by slot
  std::vector<int> until(pairs, 0);
  auto tri = [](int u, int v) { return std::max(u, v) * (std::max(u, v) - 1) / 2 + std::min(u, v); };
  auto set = [&](int u, int v, int x) {
    const int2 w = ends.slots(std::min(u, v), std::max(u, v));
    tab[w.x] = x;
    if (w.y >= 0) tab[w.y] = x;
  };
  auto live = [&](int at, int it) {  // as phase X reads a mark
    return NT == qapk::kRotBig
               ? qapk::rot_tabu16(reinterpret_cast<const uint16_t*>(marks.data())[at], it)
               : marks[at] > it + 1;
  };
  for (int u = 0; u < n; ++u)
    for (int v = u + 1; v < n; ++v) {
      const int2 w = ends.slots(u, v);
      if (ends.pair_at(w.x) != tri(u, v) || (w.y >= 0 && ends.pair_at(w.y) != tri(u, v)))
        if (fails++ < 10) std::printf("FAIL slot of (%d, %d): n=%d shape=%d\n", u, v, n, NT);
    }
  std::mt19937 rng(seed);
  std::vector<std::pair<int, int>> pool = {{0, 1}, {0, n - 1}, {n - 2, n - 1}};
  while (pool.size() < 24) {
    const int u = rng() % n, v = rng() % n;
    if (u < v) pool.push_back({u, v});
  }
  for (int it = first; it <= last; ++it) {
    const auto [r, s] = pool[rng() % pool.size()];
    // up to the longest of the ring, the shortest often
    const int t = rng() % 3 == 0 ? 1 + (int)(rng() % 4) : 1 + (int)(rng() % (RING - 2));
    if (LATE && it % 2) ends.finish();  // beside the reads below, in either order
    for (uint32_t x = Mem::ring()[(it + 1) & (RING - 1)]; x != 0xffffffffu;
         x = x >> 16 == 0xffffu ? 0xffffffffu : Mem::node()[x >> 16])
      --tab[x & 0xffffu];
    if (LATE && it % 2 == 0) ends.finish();
    for (int k = 0; k < n; ++k) {
      if (k == r || k == s) continue;
      set(r, k, live(tri(r, k), it));
      set(s, k, live(tri(s, k), it));
    }
    set(r, s, t > 1);
    ends.template apply<LATE>(r, s, it, it + t);
    until[tri(r, s)] = it + t;
    for (int u = 0; u < n; ++u)
      for (int v = u + 1; v < n; ++v) {
        const int2 w = ends.slots(u, v);
        const int want = until[tri(u, v)] > it + 1;
        if (tab[w.x] != want || (w.y >= 0 && tab[w.y] != want)) {
          if (fails++ < 10)
            std::printf("FAIL pair (%d, %d) after iteration %d: tabu until %d, its slot says %d "
                        "(n=%d shape=%d c=%d)\n", u, v, it, until[tri(u, v)], tab[w.x], n, NT, C);
          return;
        }
      }
  }
}

template <int NT, int C>
void shape(int n) {
  for (int base : {0, 32768, 65536, 20 * 32768}) {
    const int first = std::max(1, base - 540), last = base + 560;
    replay<NT, C, false>(n, first, last, last + 200, 7 + base);
    replay<NT, C, true>(n, first, last, last + 1, 8 + base);
  }
}
}  // namespace

int main() {
  // the large-n shape (16-bit marks), odd and even circles; two with 32-bit marks
  shape<qapk::kRotBig, 10>(152);
  shape<qapk::kRotBig, 12>(183);
  shape<qapk::kRotBig, 22>(255);
  shape<256, 3>(50);
  shape<512, 13>(139);
  if (fails) return 1;
  std::printf("ok\n");
  return 0;
}
