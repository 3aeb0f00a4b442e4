// Host-only check of what qap_batch_search_noalloc plans with (no GPU, no CUDA
// calls): batch_takes_workspace allocates nothing on the heap, and refuses for
// int32 elements exactly the sizes that int64 ones need a workspace for (against
// copies of the instances with the wide strides).  Built and run by
// tests/test_host_noalloc.py; prints "ok" and exits 0, or the first violations.
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>

#include "../paper_2307_11248_gb300/csrc/qap_host.cuh"

namespace {
long news = 0;
int fails = 0;
}  // namespace
#ifndef __CUDA_ARCH__
void* operator new(std::size_t n) {
  ++news;
  void* const p = std::malloc(n);
  if (!p) std::abort();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
#endif

int main() {
  constexpr int kOptin = 232448;
  int taken = 0, refused = 0;
  for (int n = 3; n <= 256; ++n)
    for (int sym = 0; sym < 2; ++sym)
      for (int mixed = 0; mixed < 2; ++mixed)
        for (int threads : {0, 256, 512, 1024})
          for (int many = 0; many < 2; ++many) {
            std::vector<qaph::DevInstance> d(mixed ? 3 : 1), d8;
            for (size_t i = 0; i < d.size(); ++i) {
              d[i].n = n - (int)i > 2 ? n - (int)i : 2;
              d[i].symF = d[i].symD = (sym + (int)i) % 2;
              d[i].wide = d[i].mid = 1;
              d[i].bound = (int64_t)1 << 40;
              d[i].ldF = qaph::pad_ldF(d[i].n, 4);
              d[i].ldP = qaph::pad_ldP(d[i].n, 4);
            }
            d8 = d;
            for (auto& x : d8) {
              x.ldF = qaph::pad_ldF(x.n, 8);
              x.ldP = qaph::pad_ldP(x.n, 8);
            }
            qap_search_params sp{};
            sp.starts = 4;
            sp.iters = 10;
            sp.tenure = {2, 5, 0};
            sp.threads_per_walk = threads;
            auto plan = [&](const std::vector<qaph::DevInstance>& x, int fb, qaph::Plan* p) {
              return qaph::search_plan(n, many != 0, x.data(), (int)x.size(), fb, 8, false, kOptin,
                                       16, n > 181, &sp, p);
            };
            qaph::Plan p4, p8;
            if (!plan(d, 4, &p4)) continue;
            const bool ok8 = plan(d8, 8, &p8);
            const bool want = qaph::ws_layout(p4, 8, 4, n, &sp).stride != 0 || !ok8 ||
                              qaph::ws_layout(p8, 8, 8, n, &sp).stride != 0;
            bool bad = false;
            const long before = news;
            const bool got = qaph::batch_takes_workspace(p4, n, many != 0, d.data(), (int)d.size(),
                                                         4, 8, false, kOptin, &sp, &bad);
            if (news != before && fails++ < 10) std::printf("FAIL allocates: n=%d\n", n);
            if (got != want && fails++ < 10)
              std::printf("FAIL n=%d sym=%d mixed=%d threads=%d many=%d: %d for %d\n", n, sym, mixed,
                          threads, many, got, want);
            ++(got ? refused : taken);
          }
  if (news == 0) ++fails, std::printf("FAIL allocations are not counted\n");
  if (!taken || !refused) ++fails, std::printf("FAIL one answer only\n");
  if (fails) return 1;
  std::printf("ok\n");
  return 0;
}
