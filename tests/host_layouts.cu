// Host-only checks of which layout a search takes (search_plan in qap_host.cuh; no
// GPU, no CUDA calls): for every n, flow width, symmetry and number of walks the
// ranges that the documents state, and a rotation plan whose shared memory, with
// the kernel's static part, would pass the limit is not taken; every compiled number
// of partner blocks is the fewest for some n.  Built and run by
// tests/test_host_layouts.py; prints "ok" and exits 0, or the first violations.
#include <cstdio>
#include <string>

#include "../paper_2307_11248_gb300/csrc/qap_host.cuh"

namespace {
constexpr int kOptin = 232448;
int fails = 0;

qaph::DevInstance instance(int n, int fb, int sym) {
  qaph::DevInstance d;
  d.n = n;
  d.symF = d.symD = sym;
  d.bytevec = fb == 1;
  d.diff16 = 1;
  d.rotX = 1000;
  d.bound = 1000000;
  d.ldF = qaph::pad_ldF(n, fb);
  d.ldP = qaph::pad_ldP(n, 1);
  return d;
}

qap_search_params params() {
  qap_search_params sp{};
  sp.starts = 4;
  sp.iters = 10;
  sp.tenure = {2, 5, 0};
  return sp;
}

// As the entry points call it: a batch (and a served request) leaves room for its
// own static word and may take a workspace for M where the rows take none.
bool plan(const qaph::DevInstance& d, int fb, bool many, bool batch, int optin, qaph::Plan* p) {
  const qap_search_params sp = params();
  return qaph::search_plan(d.n, many, &d, 1, fb, 4, false, optin, batch ? 16 : 0,
                           batch || d.n > 181, &sp, p);
}

const char* name(const qaph::Plan& p) {
  return !p.rot ? "rows" : p.store & qapk::kGlobalM ? "large" : "rotation";
}

const char* expected(int n, int fb, bool batch) {
  if (n < 3) return "rows";
  if (fb == 2) return n <= 149 ? "rotation" : "rows";
  return n <= 146 ? "rotation" : n >= (batch ? 152 : 182) ? "large" : "rows";
}
}  // namespace

int main() {
  for (int n = 2; n <= 256; ++n)
    for (int fb = 1; fb <= 2; ++fb)
      for (int sym = 0; sym < 2; ++sym)
        for (int many = 0; many < 2; ++many)
          for (int batch = 0; batch < 2; ++batch) {
            const qaph::DevInstance d = instance(n, fb, sym);
            qaph::Plan p;
            if (!plan(d, fb, many != 0, batch != 0, kOptin, &p) ||
                std::string(name(p)) != expected(n, fb, batch != 0)) {
              if (fails++ < 10)
                std::printf("FAIL layout: n=%d fb=%d sym=%d many=%d batch=%d -> %s\n", n, fb, sym,
                            many, batch, name(p));
              continue;
            }
            if (!p.rot) continue;
            // a device that has just the plan's dynamic shared memory
            const int smem = qaph::plan_smem(p, &d, 1, fb, 4);
            qaph::Plan tight;
            if (plan(d, fb, many != 0, batch != 0, smem, &tight) && tight.rot &&
                qaph::plan_smem(tight, &d, 1, fb, 4) + qaph::kRotStatic > smem && fails++ < 10)
              std::printf("FAIL beyond shared memory: n=%d fb=%d sym=%d many=%d batch=%d\n", n, fb,
                          sym, many, batch);
          }
  for (int nt : {128, 256, 512, 1024, qapk::kRotBig})
    for (int c = 1; c <= qapk::kRotMaxC; ++c) {
      if (!qapk::rot_compiled(nt, c)) continue;
      bool fewest = false;
      for (int n = 3; n <= 256 && !fewest; ++n) {
        qaph::Plan p;
        const bool products = nt == qapk::kRotBig
                                  ? n >= 152
                                  : n <= 181 && qaph::plan_for(n, nt, &p) && qaph::has_product_form(p, 2);
        int k = 1;
        while (k < c && !(qapk::rot_compiled(nt, k) && qapk::rot_chunks(n, nt, k) > 0)) ++k;
        fewest = products && k == c && qapk::rot_chunks(n, nt, c) > 0;
      }
      if (!fewest && fails++ < 10) std::printf("FAIL shape (%d, %d) is never taken\n", nt, c);
    }
  if (fails) return 1;
  std::printf("ok\n");
  return 0;
}
