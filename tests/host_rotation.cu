// Host-only checks of the rotation layout's geometry and admission
// (qap_rotation.cuh, qap_host.cuh): no GPU, no CUDA calls.  For every n, thread
// count and compiled number of partner blocks that rot_chunks admits: every
// pair has a slot, no slot pairs an index with itself, window positions stay on
// the doubled circle, phase X has a thread per index, ranks fit their bits, and
// the fixed arrays hold n.  Built and run by tests/test_host_rotation.py.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_2307_11248_gb300/csrc/qap_host.cuh"

namespace {
int fails = 0;
void fail(const char* what, int n, int nt, int c) {
  if (fails++ < 10) std::printf("FAIL %s: n=%d threads=%d c=%d\n", what, n, nt, c);
}

void check(int n, int nt, int c) {
  const int J = qapk::rot_chunks(n, nt, c);
  if (J == 0) return;
  const int n2 = (n + 1) / 2, nc = qapk::rot_circle(n, c), nE = 2 * nc;
  if (nc % c != 0 || nc < n2) fail("circle", n, nt, c);
  if (n > qapk::rot_max_n(nt) || nE > qapk::rot_max_e(nt)) fail("fixed arrays too small", n, nt, c);
  if (qapk::ld_m(n) > qapk::rot_max_n(nt) + 4) fail("pending words too small", n, nt, c);
  if (J * n2 > qapk::rot_owners(nt)) fail("too many pair threads", n, nt, c);
  if (n > qapk::rot_kx(nt) * (qapk::rot_threads(nt) - qapk::rot_owners(nt)))
    fail("no thread per index", n, nt, c);
  if (qapk::rot_rank(nt) ? 2 * c >= 1 << (qapk::rot_key_bits(nt) - 1)
                         : n > 1 << qapk::rot_key_bits(nt))
    fail("partner does not fit the key bits", n, nt, c);
  if (4 * c >= 1 << qapk::rot_slot_bits(nt) ||
      (J * n2 - 1) << qapk::rot_slot_bits(nt) >= 0xffff - (1 << qapk::rot_slot_bits(nt)))
    fail("a slot does not fit 16 bits", n, nt, c);
  std::vector<char> held((size_t)nE * nE, 0);
  for (int tid = 0; tid < J * n2; ++tid) {
    const int j = tid / n2, m = tid - j * n2, pb = m + 1 + j * c, c0 = pb % c;
    if (j == 0) held[(size_t)2 * m * nE + 2 * m + 1] = 1;
    for (int i = 0; i < c; ++i) {
      // the block of residue i in the window [pb, pb + c)
      const int pos = pb - c0 + i + (i < c0 ? c : 0), b = pos % nc;
      if (pos < pb || pos >= pb + c || b % c != i) fail("slot group off its window", n, nt, c);
      if (pos >= 2 * nc) fail("window beyond the doubled circle", n, nt, c);
      if (b == m) fail("a block against itself", n, nt, c);
      for (int q = 0; q < 4; ++q) {
        const int v = 2 * m + (q >> 1), u = 2 * b + (q & 1);
        held[(size_t)std::min(u, v) * nE + std::max(u, v)] = 1;
      }
    }
  }
  for (int u = 0; u < n; ++u)
    for (int v = u + 1; v < n; ++v)
      if (!held[(size_t)u * nE + v]) return fail("a pair without a slot", n, nt, c);
}
}  // namespace

int main() {
  for (int n = 2; n <= 256; ++n)
    for (int nt : {128, 256, 512, 1024, qapk::kRotBig})
      for (int c = 1; c <= qapk::kRotMaxC; ++c)
        if (qapk::rot_compiled(nt, c)) check(n, nt, c);
  // every size that the automatic int8 products plans take has a layout
  for (int n = 3; n <= 150; ++n)
    for (int many = 0; many < 2; ++many) {
      qaph::Plan p;
      if (!qaph::choose_plan(n, 0, many != 0, &p)) continue;
      bool any = false;
      for (int c = 1; c <= qapk::kRotMaxC; ++c)
        any |= qapk::rot_compiled(p.nt, c) && qapk::rot_chunks(n, p.nt, c) > 0;
      if (!any && p.nt < 1024) fail("no layout", n, p.nt, many);
    }
  // and every larger size the workspace shape
  for (int n = 152; n <= 256; ++n) {
    bool any = false;
    for (int c = 1; c <= qapk::kRotMaxC; ++c)
      any |= qapk::rot_compiled(qapk::kRotBig, c) && qapk::rot_chunks(n, qapk::kRotBig, c) > 0;
    if (!any) fail("no large-n layout", n, 512, 0);
    const int ld = qaph::pad_ldF(n, 1);
    if (qapk::rot_layout(n, ld, 1, ld, 0, 0, 1, 1, qapk::rot_fixed_bytes(qapk::kRotBig, 1)).bytes +
            16 > 232448)
      fail("large n beyond shared memory", n, 512, 0);
  }
  // the scan candidates' bound: by brute force over permutations and pairs it
  // holds every delta and g; F of any sign, skewed or dense
  std::mt19937 rng(3);
  for (int kind = 0; kind < 6; ++kind) {
    const int n = 9 + kind;
    std::vector<int64_t> F(n * n), D(n * n);
    for (auto& f : F) f = kind % 3 == 0 ? rng() % 100 : kind % 3 == 1 ? rng() % 9000 * (rng() % 4 == 0)
                                                                 : (int)(rng() % 2001) - 1000;
    for (auto& d : D) d = kind < 3 ? rng() % 100 : (int)(rng() % 120) - 60;
    qaph::DevInstance d;
    if (qaph::inspect_instance(F.data(), D.data(), n, &d) != QAP_OK || !d.diff16)
      fail("inspect", n, 0, kind);
    std::vector<int> p(n);
    for (int i = 0; i < n; ++i) p[i] = i;
    auto cost = [&]() {
      int64_t c = 0;
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) c += F[i * n + j] * D[p[i] * n + p[j]];
      return c;
    };
    for (int rep = 0; rep < 40; ++rep) {
      std::shuffle(p.begin(), p.end(), rng);
      const int64_t c0 = cost();
      int64_t g1 = 0, dmax = 0;
      for (int u = 0; u < n; ++u) {
        int64_t g = -d.g0;
        for (int j = 0; j < n; ++j)
          g += F[u * n + j] * D[p[u] * n + p[j]] + F[j * n + u] * D[p[j] * n + p[u]];
        g1 = std::max(g1, std::abs(g));
        for (int v = u + 1; v < n; ++v) {
          std::swap(p[u], p[v]);
          dmax = std::max(dmax, std::abs(cost() - c0));
          std::swap(p[u], p[v]);
        }
      }
      if (g1 + dmax >= d.rotX) fail("values beyond the bound", n, 0, kind);
    }
  }
  qaph::DevInstance d;
  d.rotX = ((int64_t)1 << 23) - 1;
  if (!qaph::rot_fits_keys(d, 256)) fail("largest value at 7 low bits", 0, 256, 0);
  ++d.rotX;
  if (qaph::rot_fits_keys(d, 256) || !qaph::rot_fits_keys(d, 512)) fail("key bound", 0, 256, 0);
  // tenures: up to the ring's length less 2
  qap_search_params sp{};
  sp.iters = 10;
  for (int nt : {128, 256, 512, 1024}) {
    qaph::Plan p{nt, 8, qapk::kProductM, 1, qapk::kProductM, nt};
    sp.tenure = {1, qapk::rot_ring(nt) - 2, 0};
    if (!qaph::rot_holds_tenures(p, &sp, 50)) fail("longest tenure", 50, nt, 0);
    ++sp.tenure.tmax;
    if (qaph::rot_holds_tenures(p, &sp, 50)) fail("tenure beyond the ring", 50, nt, 0);
    sp.tenure_per_n = 1;
    sp.tenure = {90, 110, 200};
    if (!qaph::rot_holds_tenures(p, &sp, 181)) fail("tenure per n", 181, nt, 0);
    sp.tenure_per_n = 0;
  }
  if (fails) return 1;
  std::printf("ok\n");
  return 0;
}
