// Rotation layout of the walk kernels (sm_103a): int8 or int16 flows, the
// paper's own tabu criterion, phase X from the maintained products M.
//
// Same search and same two barriers per iteration as qap_kernels.cuh; what
// differs is how a walk's pairs lie in the registers, what a pair costs, and
// that warps have roles.
//
// Layout.  The n indices form n2 = ceil(n / 2) blocks of two (a phantom index
// fills an odd n), on a circle of nc blocks, nc the next multiple of C.
// Thread (m, j) holds block m against the C partner blocks from m + 1 + jC on
// (mod nc): 4 pairs each, and the pair inside block m.  Going round, every
// unordered pair of blocks lies within nc / 2 steps of one of its members, so
// J threads per block with J C >= nc / 2 hold every pair; steps past nc / 2
// hold pairs a second time, which changes nothing (equal values, equal keys).
// No slot is ever invalid, so the loops carry no bounds checks; consecutive
// threads read consecutive 16-byte words (two partners' operands, 4 pairs),
// free of bank conflicts; and a thread's own operands stay in registers for
// all its slots.  Among a thread's slots a partner block lies at its residue
// mod C: the same slot in every thread, so that a move's columns, and a slot
// whose tabu time ends, are found by one branch for the whole warp (against
// slots in the window's order, where each thread compares each slot, n = 100
// went from 3385 to 3230 warp instructions per walk-iteration).

// What a pair costs.  The table holds d(u, v) = delta(u, v) + g[u] + g[v]
// (with g less its mid-range), whose O(1) update is one dp4a accumulating into
// it: the w terms of the plain delta's update are exactly the changes of g.
// The scan's candidate is e = d 2^S + psi[u], one multiply-add: delta + g[v]
// in the high bits, an index of the partner in the low S, so that a running
// minimum carries its argument (the lowest partner is also the lowest pair of
// a fixed v).  A tabu pair's d carries 2^(31 - S) on top, the sign bit of e:
// with psi lowered by 2^30 the others are negative and tabu pairs are not, the
// signed minimum of e is the best pair that is not tabu and the unsigned one
// the best that is.  The 2 C pairs with r or s as partner, and the rows of r
// and s, take phase X's values before the scan; those bring their tabu bits
// along (phase X reads the pairs' end times), so marking the applied pair
// costs nothing, and the end of a tabu time is an event: the slots that end at
// an iteration hang on that iteration's word of a ring.
//
// Roles.  The first warps hold the pairs, then come phase X's (one thread per
// index), the rest help to bring M up to date; an iteration is phase X, a
// barrier, then table and scan beside M's update, a barrier.  The last warp
// keeps tabu times and hash; a serial chain, so with few warps it does no more
// than that, and it hangs slots in the shadow of the next phase X (n = 50, 256
// walks 0.94 -> 0.85 us per iteration of all, n = 23, 100 walks 0.64 -> 0.50,
// against the first warp of phase X doing it on top of its share of M).
//
// M's update is put off: the byte operands of up to 2 moves (4 on symmetric
// instances, whose two products are equal) collect in one word per index, one
// dp4a per entry of M then applies them together, and phase X corrects the
// four entries per index that it reads by one dp4a each.
//
// Bound: the fixed latencies of one iteration's chain (arg-min, phase X,
// table, scan, two barriers) with one or two walks on an SM, integer issue
// with more.  Measured against the row layout's products form (one GB300, same
// box): n = 100 grid, 1024 walks x (2opt + 10^4) 150.0 -> 47.4 ms; n = 50
// asymmetric, 256 walks x 5000 7.85 -> 4.16 ms; n = 139 asymmetric, 150 walks
// x 2000 8.74 -> 2.83 ms; n = 23, 100 walks x 1000 in one blocking call 1.21 ->
// 0.58 ms; 2opt from 32 starts at n = 12 16.4 -> 11-12 us.  Warp instructions per
// walk-iteration: n = 100 grid 10360 -> 3196, n = 50 asymmetric 3606 -> 1924.
// int16 flows (two dp2a per pair): 96 lognormal instances of n = 20-150, 64
// walks x 1000 each, 103.4 -> 38.9 ms; their costs need 64 bits, their deltas
// do not: the rows' sums of |F| bound them (rot_bounds), where the row layout
// holds every delta as wide as the cost.
// Large n (M in the workspace, two dp4a words of pending moves): n = 256 grid,
// 64 walks x (2opt + 1000) 21.4 -> 6.25 ms, n = 203 asymmetric, 48 walks x 1000
// 15.9 -> 3.27 ms against the workspace plan, that keeps deltas and marks in L2
// and recomputes dot products; 24 requests of n = 12-256 24.5 -> 6.6 ms.
// Tried and slower: every warp holding pairs and phase X on some of them
// (n = 100 2.33 against 1.44 us per iteration of two walks per SM); tabu times
// checked by each thread through its earliest (0.3 us per iteration on the
// critical path); M updated by 4 moves at once every fourth move (the burst
// outlasts the scan beside it).
#pragma once
#include "qap_kernels.cuh"

namespace qapk {

// A shape: the threads of a CTA, or kRotBig, the one of 512 threads for large
// n, where M does not fit shared memory and lies in the CTA's workspace (L2).
constexpr int kRotBig = 513;
__host__ __device__ constexpr bool rot_big(int nt) { return nt == kRotBig; }
__host__ __device__ constexpr int rot_threads(int nt) { return rot_big(nt) ? 512 : nt; }

// Threads that may hold pairs: the same number of warps on each of an SM's
// four schedulers (from 256 threads).
__host__ __device__ constexpr int rot_owners(int nt) {
  return rot_big(nt) ? 384 : nt == 1024 ? 768 : nt / 2;
}

// Indices per phase X thread.
__host__ __device__ constexpr int rot_kx(int nt) { return rot_big(nt) ? 2 : 1; }

// Phase X threads: whole warps.
__host__ __device__ constexpr int rot_px(int n, int nt) {
  return (n + 32 * rot_kx(nt) - 1) / (32 * rot_kx(nt)) * 32;
}

// Indices, with a phantom, that a shape holds at most.
__host__ __device__ constexpr int rot_max_n(int nt) {
  return rot_big(nt) ? 256 : nt == 128 ? 64 : nt == 256 ? 128 : 192;
}

// The partner blocks per thread (C) compiled for a shape: below 16 (large n: 32)
// for their ranks.
constexpr int kRotMaxC = 22;
__host__ __device__ constexpr bool rot_compiled(int nt, int c) {
  return rot_big(nt)  ? c == 10 || c == 12 || c == 17 || c == 19 || c == 21 || c == 22
         : nt == 128  ? c == 1 || c == 2 || c == 4 || c == 7
         : nt == 256  ? c <= 4 || c == 6 || c == 7 || c == 12 || c == 13
         : nt == 512  ? c <= 3 || c == 5 || c == 7 || c == 8 || c == 12 || c == 13
                      : c == 2 || c == 4;
}

// Blocks on the circle: a multiple of c, with phantom blocks at the end.
__host__ __device__ inline int rot_circle(int n, int c) { return ((n + 1) / 2 + c - 1) / c * c; }

// Indices on the circle that a shape's arrays hold (a multiple of 4: the
// arrays behind them stay on 16-byte boundaries).
__host__ __device__ constexpr int rot_max_e(int nt) {
  return rot_big(nt) ? 264 : rot_max_n(nt);
}

// Threads per block of two (J) at c partner blocks each: the fewest that hold
// every pair; 0 when the shape does not hold n (its pairs, or its indices).
__host__ __device__ inline int rot_chunks(int n, int nt, int c) {
  const int n2 = (n + 1) / 2, nc = rot_circle(n, c), j = (nc / 2 + c - 1) / c;
  return n >= 3 && n <= rot_max_n(nt) && 2 * nc <= rot_max_e(nt) && j * n2 <= rot_owners(nt) &&
                 rot_px(n, nt) <= rot_threads(nt) - rot_owners(nt) && j * c <= nc - 1
             ? j
             : 0;
}

// Low bits S of a scan candidate.  Up to 256 threads (n <= 128) they are the
// partner itself; beyond, its rank in the thread's window, below the top bit,
// that is set before the circle's wrap: half an addition more per pair.
__host__ __device__ constexpr bool rot_rank(int nt) { return nt >= 512; }
__host__ __device__ constexpr int rot_key_bits(int nt) {
  return rot_rank(nt) && !rot_big(nt) ? 6 : 7;
}

// A slot of a thread in 16 bits: the low bits for the slot.
__host__ __device__ constexpr int rot_slot_bits(int nt) { return rot_big(nt) ? 7 : 6; }

// Ends of tabu times that lie ahead are kept in a ring of this many
// iterations; searches with longer tenures take the row layout.
__host__ __device__ constexpr int rot_ring(int nt) { return nt <= 256 ? 256 : 512; }
__host__ __device__ inline bool rot_ring_holds(int nt, int tmax) {
  return tmax <= rot_ring(nt) - 2;
}

// Pending moves of M: words of 32 bits per row and per column, and the moves
// they hold (symmetric instances twice as many): one dp4a takes 2 asymmetric
// moves of int8 flows, one dp2a 1 of int16 flows.  Large n keeps two dp4a
// words: half the traffic with M.
template <int NT, typename FE>
struct RotPending {
  static constexpr int RW = sizeof(FE) == 2 || rot_big(NT) ? 2 : 1;
  static constexpr int LW = sizeof(FE) == 1 ? RW : 1;
  template <bool SYM>
  static constexpr int Q = (rot_big(NT) ? 4 : 2) * (SYM ? 2 : 1);
};

// Barrier of the CTA; the warps of each role reach it from their own code.  bar.sync
// is the aligned form: all lanes of a warp come to it together, so a __syncwarp()
// stands where lanes part before one.  (Measured, one box: with it there, n = 139
// 2.83 ms, n = 203 3.24, n = 50 4.15, n = 100 grid 47.3; in this function 2.95, 3.66,
// 4.30, 49.2.  The form for diverged warps, barrier.sync, takes 3 to 7 registers
// more, 40 to 140 bytes of spill at large n.)
__device__ __forceinline__ void rot_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// What a walk is, for the functions of its roles: in shared memory, so that
// no register holds it through the iterations.
struct RotWalkArgs {
  InstArgs I;
  SearchArgs s;
  int64_t cost;    // of the start permutation
  const int32_t* start;
  int row, notr;
  uint32_t wid;
  int32_t* M;      // large n: M in the workspace
};
constexpr int kRotArgsBytes = (sizeof(RotWalkArgs) + 15) / 16 * 16;

// Words of an index in the pairs' update: one (int8 flows: bytes b, e, a, c,
// one dp4a) or two (int16: halves a, c, and bytes b, e, one dp2a each way).
template <typename FE>
constexpr int kRotWords = sizeof(FE) == 1 ? 1 : 2;

// Shared memory: arrays of a fixed size per thread count first, so that their
// addresses are constants, then the instance's own.
template <int NT, typename FE>
struct RotFixed {
  static constexpr int NE = rot_max_e(NT), N = rot_max_n(NT);
  static constexpr int W = kRotWords<FE>;
  // per position (the circle's indices, then again): update word(s), scan
  // addend, d of the pairs {r, k}, and of {s, k}, after the move
  static constexpr int X = 0;
  static constexpr int X2 = X + 8 * NE;
  static constexpr int psi = X + 8 * W * NE;
  static constexpr int Rr = psi + 8 * NE;
  static constexpr int Rs = Rr + 8 * NE;
  // per index: the negated words that meet a partner's (W); label (row of
  // P0); start permutation
  static constexpr int own = Rs + 8 * NE;
  static constexpr int sigma = own + 4 * W * NE;
  static constexpr int p0 = sigma + 4 * N;
  // pending operands of M's update (two buffers, by the move's parity): rows
  // by index (RW words), columns by label (LW)
  static constexpr int NW = N + 4;  // ld_m(n) at most
  static constexpr int RW = RotPending<NT, FE>::RW, LW = RotPending<NT, FE>::LW;
  static constexpr int vw = p0 + 4 * N;
  static constexpr int vwu = vw + 8 * RW * NW;
  // ring: the slots whose tabu time ends at iteration i, at i mod its length:
  // the first (thread and slot) in the low half, node of the rest in the high
  // half; nodes: such words moved aside, two for each iteration
  static constexpr int ring = vwu + 8 * LW * NW;
  static constexpr int node = ring + 4 * rot_ring(NT);
  // tenures of the iterations, at (it - 1) mod 64
  static constexpr int ten = node + 8 * rot_ring(NT);
  // arg-min candidates of the warps (int2) and, at 32, whether the walk is
  // over, at 33 the move for the keeper; block sums
  static constexpr int red = ten + 4 * 64;
  static constexpr int sum = red + 8 * 34;
  // what the walk is (RotWalkArgs)
  static constexpr int args = sum + 8 * 32;
  static constexpr int bytes = args + kRotArgsBytes;
  static_assert(own % 16 == 0 && vw % 16 == 0 && vwu % 16 == 0 && ring % 16 == 0 &&
                    args % 16 == 0 && bytes % 16 == 0 && psi % 8 == 0 && Rr % 8 == 0,
                "aligned for the widest access of each array");
};

struct RotLayout {
  int F, Ft, P, Pt, M, mark, bytes;
};

// notr: no transposed copies of F and P (kNoTransposed plans)
__host__ __device__ inline RotLayout rot_layout(int n, int ldF, int fbytes, int ldP, int symF,
                                                int symD, int notr, int big, int fixed) {
  RotLayout L;
  int o = fixed;
  L.F = o;    o = align16(o + n * ldF * fbytes);
  L.Ft = o;   o = (symF || notr) ? o : align16(o + n * ldF * fbytes);
  L.P = o;    o = align16(o + n * ldP);
  L.Pt = o;   o = (symD || notr) ? o : align16(o + n * ldP);
  L.M = o;    o = big ? o : align16(o + n * ld_m(n) * 4);
  // one entry more: the thread of k = r reads past the triangle's end at
  // r = n - 1 (and drops it)
  L.mark = o; o = align16(o + (n * (n - 1) / 2 + 1) * (big ? 2 : 4));
  L.bytes = o;
  return L;
}

template <typename FE>
__host__ __device__ inline int rot_fixed_of(int nt) {
  return nt == 128   ? RotFixed<128, FE>::bytes
         : nt == 256 ? RotFixed<256, FE>::bytes
         : nt == 512 ? RotFixed<512, FE>::bytes
         : rot_big(nt) ? RotFixed<kRotBig, FE>::bytes
                     : RotFixed<1024, FE>::bytes;
}
__host__ __device__ inline int rot_fixed_bytes(int nt, int fbytes) {
  return fbytes == 1 ? rot_fixed_of<int8_t>(nt) : rot_fixed_of<int16_t>(nt);
}

extern __shared__ __align__(16) unsigned char rot_smem[];

template <typename T>
__device__ __forceinline__ T* rot_at(int off) {
  return reinterpret_cast<T*>(rot_smem + off);
}

// Views of the shared memory.
template <int NT, typename FE>
struct RotSmem {
  using X_ = RotFixed<NT, FE>;
  RotLayout L;
  int ft, pt;          // offsets that F^T and P0^T are read from:
  int fr, fk, pr, pk;  // entry [r][k] at r fr + k fk
  __device__ __forceinline__ RotSmem(const InstArgs& I, int n, bool notr) {
    L = rot_layout(n, I.ldF, sizeof(FE), I.ldP, I.symF, I.symD, notr, rot_big(NT), X_::bytes);
    ft = I.symF || notr ? L.F : L.Ft;
    pt = I.symD || notr ? L.P : L.Pt;
    // without copies F^T is read from F's columns
    const bool fc = !I.symF && notr, pc = !I.symD && notr;
    fr = fc ? 1 : I.ldF;
    fk = fc ? I.ldF : 1;
    pr = pc ? 1 : I.ldP;
    pk = pc ? I.ldP : 1;
  }
  __device__ __forceinline__ FE* F() const { return rot_at<FE>(L.F); }
  __device__ __forceinline__ FE* Ft() const { return rot_at<FE>(ft); }
  __device__ __forceinline__ int8_t* P() const { return rot_at<int8_t>(L.P); }  // P0 = D[p0][p0]
  __device__ __forceinline__ int8_t* Pt() const { return rot_at<int8_t>(pt); }
  // M[x][label], halved on symmetric instances
  __device__ __forceinline__ int32_t* M() const {
    return rot_big(NT) ? args().M : rot_at<int32_t>(L.M);
  }
  // tabu_until of pair u < v at v (v - 1) / 2 + u (large n: see rot_mark16)
  __device__ __forceinline__ int32_t* mark() const { return rot_at<int32_t>(L.mark); }
  __device__ __forceinline__ static int32_t* X() { return rot_at<int32_t>(X_::X); }
  __device__ __forceinline__ static int32_t* X2() { return rot_at<int32_t>(X_::X2); }
  __device__ __forceinline__ static int32_t* psi() { return rot_at<int32_t>(X_::psi); }
  __device__ __forceinline__ static int32_t* Rr() { return rot_at<int32_t>(X_::Rr); }
  __device__ __forceinline__ static int32_t* Rs() { return rot_at<int32_t>(X_::Rs); }
  __device__ __forceinline__ static int32_t* own() { return rot_at<int32_t>(X_::own); }
  __device__ __forceinline__ static int32_t* sigma() { return rot_at<int32_t>(X_::sigma); }
  __device__ __forceinline__ static int32_t* p0() { return rot_at<int32_t>(X_::p0); }
  __device__ __forceinline__ static int32_t* vw() { return rot_at<int32_t>(X_::vw); }
  __device__ __forceinline__ static int32_t* vwu() { return rot_at<int32_t>(X_::vwu); }
  __device__ __forceinline__ static uint32_t* ring() { return rot_at<uint32_t>(X_::ring); }
  __device__ __forceinline__ static uint32_t* node() { return rot_at<uint32_t>(X_::node); }
  __device__ __forceinline__ static int32_t* ten() { return rot_at<int32_t>(X_::ten); }
  __device__ __forceinline__ static int2* red() { return rot_at<int2>(X_::red); }
  __device__ __forceinline__ static int64_t* sum() { return rot_at<int64_t>(X_::sum); }
  __device__ __forceinline__ static RotWalkArgs& args() { return *rot_at<RotWalkArgs>(X_::args); }
};

// The course of a walk, as the pairs' warps and phase X's follow it.
template <typename FE>
struct RotCourse {
  // costs: int8 flows have int32 deltas by the bound on the cost
  using Cost = std::conditional_t<sizeof(FE) == 1, int, int64_t>;
  Cost cur, best;
  int it, dmoves, iters, cap, ow;
  int bd, r, s;          // the move
  bool tabu_phase, stalled;

  __device__ __forceinline__ RotCourse(const RotWalkArgs& w, int warps)
      : cur((Cost)w.cost), best(cur), it(0), dmoves(0), iters(w.s.iters),
        cap(w.s.max_descent >= 0 ? w.s.max_descent : kDescentCap), ow(warps), bd(0), r(0), s(1),
        tabu_phase(!w.s.descend), stalled(false) {}

  // The arg-min over the warps' candidates, after the barrier that ends a
  // scan; false when the walk is over.
  __device__ __forceinline__ bool next(int2* red) {
    const int lane = threadIdx.x & 31;
    rot_barrier();
    const int2 c = lane < ow ? red[lane] : make_int2(INT_MAX, (int)kNoMove);
    bd = __reduce_min_sync(kFull, c.x);
    const uint32_t bk = __reduce_min_sync(kFull, c.x == bd ? (uint32_t)c.y : kNoMove);
    stalled = bk == kNoMove;
    if (__builtin_expect(!tabu_phase, 0)) {
      if (stalled || bd >= 0 || dmoves == cap) {
        // the descent ends; its last arg-min is also that of tabu iteration
        // 1, where no pair is tabu
        tabu_phase = true;
        best = cur;
      } else {
        ++dmoves;
      }
    }
    if (tabu_phase) {
      if (__builtin_expect(it == iters || stalled, 0)) {
        if (lane == 0) red[32].x = 1;  // for the helpers
        __syncwarp();
        rot_barrier();
        return false;
      }
      ++it;
    }
    r = (int)(bk >> 8);
    s = (int)(bk & 0xffu);
    cur += bd;
    return true;
  }
};

// What an instance fixes for a thread.
struct RotThread {
  int n, n2;        // indices, blocks of two (with a phantom index when n is odd)
  int nc, nE;       // blocks and indices on the circle
  int J;            // threads per block
  int role;         // of the thread's warp: 0 holds pairs, 1 phase X, 2 helps with M
  int m;            // role 0: block of two that the thread holds
  int pb, pbm;      // role 0: first partner block, as position and mod nc
  bool extra;       // role 0: past the last chunk; the thread offers no candidates
  bool keeper;      // the thread's warp keeps tabu times and hash: the last one
  int pt, pxt;      // role 1: the thread among phase X's, their number
  int ow;           // warps with role 0
  int ug, ux, urows;  // roles 1, 2: column group and first row of M, rows at once
};

template <int NT, int C>
__device__ __forceinline__ RotThread rot_thread(int n) {
  RotThread t;
  const int tid = threadIdx.x;
  t.n = n;
  t.n2 = (n + 1) / 2;
  t.nc = rot_circle(n, C);
  t.nE = 2 * t.nc;
  const int J = t.J = rot_chunks(n, NT, C);
  const int jt = tid / t.n2;
  t.m = tid - jt * t.n2;
  const int j = jt < J ? jt : 0;
  t.extra = jt >= J;
  t.pb = t.m + 1 + j * C;
  t.pbm = t.pb < t.nc ? t.pb : t.pb - t.nc;
  t.ow = (J * t.n2 + 31) / 32;
  t.pt = tid - rot_owners(NT);
  t.pxt = rot_px(n, NT);
  t.role = tid < 32 * t.ow ? 0 : t.pt >= 0 && t.pt < t.pxt ? 1 : 2;
  t.keeper = tid >= rot_threads(NT) - 32;
  // a keeper that is no phase X warp leaves M to the others (8 warps or fewer:
  // with more the keeper is done before its share)
  const int mt = rot_threads(NT) - 32 * t.ow -
                 (NT <= 256 && t.pxt + rot_owners(NT) <= NT - 32 ? 32 : 0);
  const int gpr = ld_m(n) / 4, f = tid - 32 * t.ow;
  t.ug = f % gpr;
  t.ux = f / gpr;
  t.urows = mt / gpr;
  return t;
}

// Shared-memory loads and stores by 32-bit address.
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ int lds32(uint32_t at) {
  int v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ int lds8(uint32_t at) {
  int v;
  asm volatile("ld.shared.s8 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ int lds16(uint32_t at) {
  int v;
  asm volatile("{.reg .b16 t; ld.shared.s16 t, [%1]; cvt.s32.s16 %0, t;}"
               : "=r"(v)
               : "r"(at)
               : "memory");
  return v;
}
// an element of F
template <typename FE>
__device__ __forceinline__ int ldsf(uint32_t at) {
  return sizeof(FE) == 1 ? lds8(at) : lds16(at);
}
__device__ __forceinline__ int2 lds64(uint32_t at) {
  int2 v;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ int4 lds128(uint32_t at) {
  int4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(at)
               : "memory");
  return v;
}
__device__ __forceinline__ void sts32(uint32_t at, int v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t at, int x, int y) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t at, int4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}

__device__ __forceinline__ int lds16u(uint32_t at) {
  int v;
  asm volatile("{.reg .b16 t; ld.shared.u16 t, [%1]; cvt.u32.u16 %0, t;}"
               : "=r"(v)
               : "r"(at)
               : "memory");
  return v;
}
// A tabu time's end in 16 bits: 0 for a pair that is not tabu.
__host__ __device__ __forceinline__ int rot_mark16(int end) { return (end & 0x7fff) | 0x8000; }
// Whether a pair with that mark is tabu after iteration `it`.
__host__ __device__ __forceinline__ bool rot_tabu16(int mark, int it) {
  return mark != 0 && mark != rot_mark16(it + 1);
}
// Entries of M at byte offset `at`: in shared memory, or (large n) in the
// workspace, past L1.
template <int NT>
__device__ __forceinline__ int ldm32(const char* g, uint32_t at) {
  if constexpr (rot_big(NT)) {
    int v;
    asm volatile("ld.global.cg.b32 %0, [%1];" : "=r"(v) : "l"(g + at) : "memory");
    return v;
  } else {
    return lds32(at);
  }
}
template <int NT>
__device__ __forceinline__ int4 ldm128(const char* g, uint32_t at) {
  if constexpr (rot_big(NT)) {
    int4 v;
    asm volatile("ld.global.cg.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(g + at)
                 : "memory");
    return v;
  } else {
    return lds128(at);
  }
}
template <int NT>
__device__ __forceinline__ void stm128(char* g, uint32_t at, int4 v) {
  if constexpr (rot_big(NT))
    asm volatile("st.global.cg.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(g + at), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
  else
    sts128(at, v);
}

__device__ __forceinline__ uint32_t pack2(int h0, int h1) {
  return __byte_perm((uint32_t)h0, (uint32_t)h1, 0x5410u);
}
__device__ __forceinline__ uint32_t pack4(int b0, int b1, int b2, int b3) {
  return __byte_perm(__byte_perm((uint32_t)b0, (uint32_t)b1, 0x0040u),
                     __byte_perm((uint32_t)b2, (uint32_t)b3, 0x0040u), 0x5410u);
}

// M at the start of a walk, from F and P0: one dot product per entry over
// rows, a second over columns when F or D is asymmetric.  A warp takes four
// rows of F at once (each 16-byte chunk of a row of P0 serves four dot
// products), its lanes the columns.  Symmetric instances keep half of M.
template <int NT, typename FE>
__device__ __forceinline__ void rot_compute_m(const RotSmem<NT, FE>& S, int n, int ldF, int ldP,
                                              bool sym, bool notr) {
  using C = Chunk<FE>;
  using FV = typename C::FV;
  using QV = typename C::QV;
  const int nc = (n + C::W - 1) / C::W, ldm = ld_m(n);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int x0 = 4 * warp; x0 < n; x0 += rot_threads(NT) / 8) {
    const int xm = n - 1;
    const int x1 = min(x0 + 1, xm), x2 = min(x0 + 2, xm), x3 = min(x0 + 3, xm);
    for (int k = lane; k < n; k += 32) {
      int a0 = 0, a1 = 0, a2 = 0, a3 = 0;
      auto rows = [&](const FE* F, const int8_t* P) {
        const QV* q = reinterpret_cast<const QV*>(P + k * ldP);
        const FV* f0 = reinterpret_cast<const FV*>(F + x0 * ldF);
        const FV* f1 = reinterpret_cast<const FV*>(F + x1 * ldF);
        const FV* f2 = reinterpret_cast<const FV*>(F + x2 * ldF);
        const FV* f3 = reinterpret_cast<const FV*>(F + x3 * ldF);
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {
          const QV v = q[c];
          a0 = C::dot(f0[c], v, a0);
          a1 = C::dot(f1[c], v, a1);
          a2 = C::dot(f2[c], v, a2);
          a3 = C::dot(f3[c], v, a3);
        }
      };
      rows(S.F(), S.P());
      if (!sym && !notr) rows(S.Ft(), S.Pt());
      if (!sym && notr) {
        // columns x0..x0+3 of F (x0 a multiple of 4) and column k of P0
#pragma unroll 4
        for (int j = 0; j < n; ++j) {
          using F4 = std::conditional_t<sizeof(FE) == 1, char4, short4>;
          const F4 f = *reinterpret_cast<const F4*>(S.F() + j * ldF + x0);
          const int p = S.P()[j * ldP + k];
          a0 += f.x * p;
          a1 += f.y * p;
          a2 += f.z * p;
          a3 += f.w * p;
        }
      }
      S.M()[x0 * ldm + k] = a0;
      if (x0 + 1 < n) S.M()[x1 * ldm + k] = a1;
      if (x0 + 2 < n) S.M()[x2 * ldm + k] = a2;
      if (x0 + 3 < n) S.M()[x3 * ldm + k] = a3;
    }
  }
}

// The marks, after the pairs' warps have taken the table from their place (or
// made it); by the other warps.
template <int NT>
__device__ __forceinline__ void rot_clear_marks(int32_t* mark, int n, int ow) {
  rot_barrier();
  const int words = rot_big(NT) ? (n * (n - 1) / 2 + 1) / 2 : n * (n - 1) / 2;
  for (int x = (int)threadIdx.x - 32 * ow; x < words; x += rot_threads(NT) - 32 * ow) mark[x] = 0;
  __syncwarp();
}

// Tenure of iteration it (from 1).
struct RotTenure {
  int tmin, tmax, period;
  __device__ __forceinline__ RotTenure(const SearchArgs& a, int n)
      : tmin(a.tmin), tmax(a.tmax), period(a.period) {
    if (a.tenure_per_n) {
      tmin = max(1, a.tmin * n / 100);
      tmax = max(tmin, (a.tmax * n + 99) / 100);
      period = a.period * n / 100;
    }
  }
  __device__ __forceinline__ int of(uint64_t seed, uint32_t wid, int it) const {
    const uint32_t i = (uint32_t)(it - 1);
    const uint32_t x = walk_draw(seed, wid, 1u, period > 0 ? i / (uint32_t)period : i);
    return tmin + (int)below(x, (uint32_t)(tmax - tmin + 1));
  }
};

// An entry of M with its pending moves: row words, column words.
template <int NT, typename FE>
__device__ __forceinline__ int rot_entry(int2 w, int2 u, int m) {
  using P = RotPending<NT, FE>;
  if constexpr (P::RW == 1) return __dp4a(w.x, u.x, m);
  else if constexpr (P::LW == 2) return __dp4a(w.y, u.y, __dp4a(w.x, u.x, m));
  else return __dp2a_hi(w.y, u.x, __dp2a_lo(w.x, u.x, m));
}

// M[x][.] after a move, for the rows x = slot mod Q, with the pending words:
// a group of 4 columns of every urows-th such row per thread, 4 rows (large n:
// 8) in flight.
template <int NT, typename FE>
__device__ __forceinline__ void rot_update_m(const RotThread& T, char* gM, uint32_t aM,
                                             uint32_t aVw, uint32_t aVwu, int n, int ldm,
                                             int Q, int slot) {
  using P = RotPending<NT, FE>;
  constexpr int B = rot_big(NT) ? 8 : 4;
  if (T.ux >= T.urows) return;
  int4 w, w2 = make_int4(0, 0, 0, 0);
  if constexpr (P::LW == 1) {
    w = lds128(aVwu + 16 * T.ug);
  } else {
    const int4 a = lds128(aVwu + 32 * T.ug), b = lds128(aVwu + 32 * T.ug + 16);
    w = make_int4(a.x, a.z, b.x, b.z);
    w2 = make_int4(a.y, a.w, b.y, b.w);
  }
  const int step = Q * T.urows;
  auto upd = [&](int2 u, int4 v) {
    v.x = rot_entry<NT, FE>(u, make_int2(w.x, w2.x), v.x);
    v.y = rot_entry<NT, FE>(u, make_int2(w.y, w2.y), v.y);
    v.z = rot_entry<NT, FE>(u, make_int2(w.z, w2.z), v.z);
    v.w = rot_entry<NT, FE>(u, make_int2(w.w, w2.w), v.w);
    return v;
  };
  uint32_t am = aM + 16 * T.ug + 4 * ldm * (slot + Q * T.ux);
  uint32_t av = aVw + 4 * P::RW * (slot + Q * T.ux);
  const uint32_t sm = 4 * ldm * step, sv = 4 * P::RW * step;
#pragma unroll 1
  for (int x = slot + Q * T.ux; x < n; x += B * step) {
    // rows past the last repeat the first: the same entry, loaded before it
    // is stored, takes the same value again
    int4 a[B];
    int2 b[B];
    uint32_t at[B];
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const bool in = x + i * step < n;
      at[i] = am + (in ? i * sm : 0);
      a[i] = ldm128<NT>(gM, at[i]);
      const uint32_t ab = av + (in ? i * sv : 0);
      if constexpr (P::RW == 1) b[i] = make_int2(lds32(ab), 0);
      else b[i] = lds64(ab);
    }
#pragma unroll
    for (int i = 0; i < B; ++i) stm128<NT>(gM, at[i], upd(b[i], a[i]));
    am += B * sm;
    av += B * sv;
  }
}

// d[q] less `big`, q the same in every lane: a branch tree.
template <int LO, int HI, int NS>
__device__ __forceinline__ void clear_tabu(int (&d)[NS], int q, int big) {
  if constexpr (HI - LO > 3) {
    constexpr int MID = (LO + HI) / 2;
    if (q < MID) clear_tabu<LO, MID>(d, q, big);
    else clear_tabu<MID, HI>(d, q, big);
  } else {
#pragma unroll
    for (int i = LO; i < HI; ++i) d[i] -= q == i ? big : 0;
  }
}

// A pair's entry of the table at the start of a walk: M[u][v] + M[v][u] + the
// 2x2 term of Eq. 2, less twice g's mid-range.
template <int NT, typename FE>
__device__ __forceinline__ int rot_pair(const RotSmem<NT, FE>& S, const InstArgs& I, int u, int v) {
  const int ldF = I.ldF, ldP = I.ldP, ldm = ld_m(I.n);
  const FE* F = S.F();
  const int8_t* P = S.P();
  const int32_t* M = S.M();
  const int f = (int)F[u * ldF + u] - F[u * ldF + v] - F[v * ldF + u] + F[v * ldF + v];
  const int p = (int)P[u * ldP + u] - P[u * ldP + v] - P[v * ldP + u] + P[v * ldP + v];
  return ((M[u * ldm + v] + M[v * ldm + u]) << (I.symF && I.symD ? 1 : 0)) + f * p - 2 * I.g0;
}

// d's slots with the partner of residue and parity x (the same in every lane),
// where the lane holds it: a branch tree.
template <int LO, int HI, int NS>
__device__ __forceinline__ void put_partner(int (&d)[NS], int x, bool hold, int w0, int w1) {
  if constexpr (HI - LO > 4) {
    constexpr int MID = (LO + HI) / 2;
    if (x < MID) put_partner<LO, MID>(d, x, hold, w0, w1);
    else put_partner<MID, HI>(d, x, hold, w0, w1);
  } else {
#pragma unroll
    for (int y = LO; y < HI; ++y) {
      const bool here = hold && x == y;
      constexpr int STEP = 2;
      const int q = 4 * (y >> 1) + (y & 1);
      d[q] = here ? w0 : d[q];
      d[q + STEP] = here ? w1 : d[q + STEP];
    }
  }
}

// The warps that hold pairs: the table, its update after each move, and the
// scan for the next iteration.  Slot group i of a thread holds the partner
// block of residue i mod C in its window: a block has the same group in every
// thread, so that the two columns of a move are written by one uniform branch.
template <int NT, int C, typename FE>
__device__ __forceinline__ void rot_owner() {
  using S = RotSmem<NT, FE>;
  const RotWalkArgs& W = S::args();
  const InstArgs& I = W.I;
  const int aspiration = W.s.aspiration;
  const RotThread T = rot_thread<NT, C>(I.n);
  const int n = T.n, nc = T.nc, nE = T.nE, m = T.m;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int v0 = 2 * m, v1 = v0 + 1;
  const bool half = v1 >= n || T.extra;  // no candidates from the second row: a phantom
  constexpr bool RANK = rot_rank(NT);
  constexpr int SB = rot_key_bits(NT);
  constexpr uint32_t MUL = 1u << SB;
  constexpr int TOP = (int)(MUL / 2);  // with RANK: on the partners before the wrap
  static_assert(!RANK || 2 * C < TOP, "ranks fit below the top bit");
  constexpr int BIG = 1 << (31 - SB);  // on top of a tabu pair's d
  constexpr int NS = 4 * C + 1;        // slots; the last holds the pair inside the block

  // position of slot group i's block, and its offset in arrays of two words
  // per block
  const int c0 = T.pb % C;
  int o0 = 8 * (T.pb - c0), o1 = o0 + 8 * C;
  auto off = [&](int i) { return (i < c0 ? o1 : o0) + 8 * i; };
  // many slots leave no registers to hold the offsets from one use to the next
  auto again = [&] {
    if constexpr (C > 13) asm volatile("" : "+r"(o0), "+r"(o1));
  };

  // the table: from where rot_start left it, or (large n) by the pairs
  int32_t* const mark = S(I, n, W.notr != 0).mark();
  int d[NS];
  auto d_init = [&](int u, int v) -> int {
    const int hi = max(u, v), lo = min(u, v);
    if (hi >= n) return 0;
    if constexpr (rot_big(NT)) return rot_pair(S(I, n, W.notr != 0), I, lo, hi);
    else return mark[hi * (hi - 1) / 2 + lo];
  };
#pragma unroll
  for (int i = 0; i < C; ++i) {
    const int b = off(i) / 8 < nc ? off(i) / 8 : off(i) / 8 - nc;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      d[4 * i + q] = d_init(v0 + (q >> 1), 2 * b + (q & 1));
      // large n: one after the other (together they take more registers
      // than the iterations have)
      if constexpr (rot_big(NT)) asm volatile("" : "+r"(d[4 * i + q])::"memory");
    }
  }
  d[4 * C] = d_init(v0, v1);
  __syncwarp();
  rot_barrier();  // the others now clear the marks

  // arrays of two words per block, by byte offset
  auto two = [](const int32_t* a, int at) {
    return *reinterpret_cast<const int2*>(reinterpret_cast<const char*>(a) + at);
  };

  // Scan of the table: the warp's candidate into red.  A tabu pair aspires
  // when its delta is below `lim` (at most 0, at least NOLIM).
  constexpr int NOLIM = -(INT_MAX >> SB);
  auto scan = [&](int lim) {
    again();
    int m0 = INT_MAX, m1 = INT_MAX;
    uint32_t t0 = 0xffffffffu, t1 = 0xffffffffu;
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const int2 y = two(S::psi(), off(i));
      // rank: twice the block's place in the window, from 1 (the pair inside: 0)
      const uint32_t rk = RANK ? (uint32_t)((i < c0 ? 2 * C : 0) - 2 * c0) : 0u;
      const uint32_t y0 = (uint32_t)y.x + rk + (RANK ? 2 * i + 1 : 0);
      const uint32_t y1 = (uint32_t)y.y + rk + (RANK ? 2 * i + 2 : 0);
      const uint32_t e00 = (uint32_t)d[4 * i] * MUL + y0;
      const uint32_t e01 = (uint32_t)d[4 * i + 1] * MUL + y1;
      const uint32_t e10 = (uint32_t)d[4 * i + 2] * MUL + y0;
      const uint32_t e11 = (uint32_t)d[4 * i + 3] * MUL + y1;
      m0 = min(m0, min((int)e00, (int)e01));
      m1 = min(m1, min((int)e10, (int)e11));
      t0 = min(t0, min(e00, e01));
      t1 = min(t1, min(e10, e11));
    }
    const int2 o = two(S::psi(), 8 * m);
    {
      // the pair inside the block: its first thread offers it
      uint32_t e = (uint32_t)d[4 * C] * MUL + (uint32_t)o.y;
      e = warp * 32 + lane == m ? e : INT_MAX;
      m0 = min(m0, (int)e);
      t0 = min(t0, e);
    }
    // delta 2^S + index of each row's best, by the own index's psi: q is
    // 2^30 less g[v]
    const uint32_t q0 = (uint32_t)o.x - (RANK ? TOP : v0) + 0x80000000u;
    const uint32_t q1 = (uint32_t)o.y - (RANK ? TOP : v1) + 0x80000000u;
    const int ls = (int)((uint32_t)lim * MUL);
    int b0 = m0 < 0 ? (int)((uint32_t)m0 + q0) : INT_MAX;
    int b1 = m1 < 0 ? (int)((uint32_t)m1 + q1) : INT_MAX;
    const int x0 = (int)(t0 + q0 + 0x80000000u), x1 = (int)(t1 + q1 + 0x80000000u);
    if ((int)t0 >= 0 && x0 < ls) b0 = min(b0, x0);
    if ((int)t1 >= 0 && x1 < ls) b1 = min(b1, x1);
    if (half) b1 = INT_MAX;
    if (T.extra) b0 = INT_MAX;
    // the lower pair of the two rows
    const int d0 = b0 >> SB, d1 = b1 >> SB;
    int u0 = b0 & (int)(MUL - 1), u1 = b1 & (int)(MUL - 1);
    if (RANK) {
      u0 = (u0 & (TOP - 1)) + 2 * T.pb - 1;
      u0 = u0 >= nE ? u0 - nE : u0;
      u0 = (b0 & (TOP - 1)) == 0 ? v1 : u0;
      u1 = (u1 & (TOP - 1)) + 2 * T.pb - 1;
      u1 = u1 >= nE ? u1 - nE : u1;
    }
    const uint32_t k0 = (uint32_t)(min(u0, v0) << 8 | max(u0, v0));
    const uint32_t k1 = (uint32_t)(min(u1, v1) << 8 | max(u1, v1));
    const bool second = d1 < d0 || (d1 == d0 && k1 < k0);
    const int dd = second ? d1 : d0;
    const uint32_t kk = second ? k1 : k0;
    const int wd = __reduce_min_sync(kFull, dd);
    const uint32_t wk = __reduce_min_sync(kFull, dd == wd ? kk : kNoMove);
    const bool none = wd == INT_MAX >> SB;
    // (by every lane: lanes that part cost more)
    S::red()[warp] = make_int2(none ? INT_MAX : wd, (int)(none ? kNoMove : wk));
  };

  scan(NOLIM);

  RotCourse<FE> c(W, T.ow);
  while (c.next(S::red())) {
    const int r = c.r, s = c.s, it = c.it;
    c.best = c.tabu_phase ? min(c.best, c.cur) : c.cur;
    using Cost = typename RotCourse<FE>::Cost;
    const int lim = aspiration ? (int)max(c.best - c.cur, (Cost)NOLIM) : NOLIM;
    // slots whose tabu time ends with the next iteration
    uint32_t w = S::ring()[(it + 1) & (rot_ring(NT) - 1)];
    while (w != 0xffffffffu) {
      const int at = (int)(w & 0xffffu) >> rot_slot_bits(NT);
      if (at >> 5 == warp)
        clear_tabu<0, NS>(d, (int)w & ((1 << rot_slot_bits(NT)) - 1),
                          (at & 31) == lane ? BIG : 0);
      w = w >> 16 == 0xffffu ? 0xffffffffu : S::node()[w >> 16];
    }
    const int br = r >> 1, bs = s >> 1;
    // slot groups of r and s as partners, and whether the thread holds them
    const int xr = 2 * (br % C) + (r & 1), xs = 2 * (bs % C) + (s & 1);
    int kr = br - T.pbm, ks = bs - T.pbm;
    kr = kr < 0 ? kr + nc : kr;
    ks = ks < 0 ? ks + nc : ks;
    const bool hold_r = kr < C, hold_s = ks < C;
    const bool row0 = v0 == r || v0 == s, row1 = v1 == r || v1 == s;
    rot_barrier();

    // the new table
    again();
    const int2 wr = two(S::Rr(), 8 * m), ws = two(S::Rs(), 8 * m);  // v0, v1 with r, with s
    if constexpr (sizeof(FE) == 1) {
      const int2 A = two(S::own(), 8 * m);
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int2 x = two(S::X(), off(i));
        d[4 * i] = __dp4a(A.x, x.x, d[4 * i]);
        d[4 * i + 1] = __dp4a(A.x, x.y, d[4 * i + 1]);
        d[4 * i + 2] = __dp4a(A.y, x.x, d[4 * i + 2]);
        d[4 * i + 3] = __dp4a(A.y, x.y, d[4 * i + 3]);
      }
      d[4 * C] = __dp4a(A.x, S::X()[v1], d[4 * C]);
    } else {
      // (-a, -c) of a row with the partner's (b, e), its (-b, -e) with (a, c)
      const int4 A = reinterpret_cast<const int4*>(S::own())[m];
      auto upd = [](int ac, int be, int x, int x2, int t) {
        return __dp2a_lo(x, be, __dp2a_lo(ac, x2, t));
      };
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int2 x = two(S::X(), off(i)), x2 = two(S::X2(), off(i));
        d[4 * i] = upd(A.x, A.y, x.x, x2.x, d[4 * i]);
        d[4 * i + 1] = upd(A.x, A.y, x.y, x2.y, d[4 * i + 1]);
        d[4 * i + 2] = upd(A.z, A.w, x.x, x2.x, d[4 * i + 2]);
        d[4 * i + 3] = upd(A.z, A.w, x.y, x2.y, d[4 * i + 3]);
      }
      d[4 * C] = upd(A.x, A.y, S::X()[v1], S::X2()[v1], d[4 * C]);
    }
    // the columns of r and s
    put_partner<0, 2 * C>(d, xr, hold_r, wr.x, wr.y);
    put_partner<0, 2 * C>(d, xs, hold_s, ws.x, ws.y);
    // their rows
    if (row0 || row1) {
      again();
      if (row0) {
        const int32_t* const x = v0 == r ? S::Rr() : S::Rs();
#pragma unroll
        for (int i = 0; i < C; ++i) {
          const int2 y = two(x, off(i));
          d[4 * i] = y.x;
          d[4 * i + 1] = y.y;
        }
        d[4 * C] = x[v1];
      }
      if (row1) {
        const int32_t* const x = v1 == r ? S::Rr() : S::Rs();
#pragma unroll
        for (int i = 0; i < C; ++i) {
          const int2 y = two(x, off(i));
          d[4 * i + 2] = y.x;
          d[4 * i + 3] = y.y;
        }
        d[4 * C] = x[v0];
      }
    }
    scan(lim);
  }
}

// The ends of a walk's tabu times: each pair's mark, and the ring that the slots
// whose time ends hang on.  Kept by one thread.  Mem says where the ring and its
// nodes lie: shared memory, or (to check the bookkeeping on the host) an array.
template <int NT, int C, typename Mem>
struct RotEnds {
  static constexpr bool M16 = rot_big(NT);
  static constexpr int RING = rot_ring(NT), SL = rot_slot_bits(NT);
  static_assert(0x8000 % RING == 0, "a 16-bit mark gives its end modulo the ring's length");
  const int n2, nc, J, iters;
  int32_t* const mark;
  int2 late;     // the last move, while its slots are to be hung
  int late_end;  // the end of its tabu time (0: none)

  __host__ __device__ __forceinline__ RotEnds(int blocks, int circle, int chunks, int its,
                                              int32_t* marks)
      : n2(blocks), nc(circle), J(chunks), iters(its), mark(marks), late(make_int2(0, 0)),
        late_end(0) {}

  // The slot that block u's threads hold pair (u, v) in, or -1 when v is not
  // in their windows.
  __host__ __device__ __forceinline__ int slot(int u, int v) const {
    const int bu = u >> 1, bv = v >> 1;
    int o = bv - bu;
    o = (o < 0 ? o + nc : o) - 1;
    const int j = o / C;
    return j < J ? (j * n2 + bu) << SL | (4 * (bv % C) + 2 * (u & 1) + (v & 1)) : -1;
  }
  // The slots of a pair, one or two (the one inside a block is its first
  // thread's).
  __host__ __device__ __forceinline__ int2 slots(int r, int s) const {
    if (r >> 1 == s >> 1) return make_int2((r >> 1) << SL | 4 * C, -1);
    const int a = slot(r, s), b = slot(s, r);
    return a >= 0 ? make_int2(a, b) : make_int2(b, -1);
  }
  // The pair of a slot, as its place in the triangle of marks.
  __host__ __device__ __forceinline__ int pair_at(int w) const {
    const int t = w >> SL, q = w & ((1 << SL) - 1), j = t / n2, m = t - j * n2;
    int v = 2 * m, u = v + 1;
    if (q < 4 * C) {
      const int pb = m + 1 + j * C, c0 = pb % C, i = q >> 2;
      const int b = pb - c0 + i + (i < c0 ? C : 0);
      v += q >> 1 & 1;
      u = 2 * (b < nc ? b : b - nc) + (q & 1);
    }
    const int hi = u > v ? u : v, lo = u > v ? v : u;
    return hi * (hi - 1) / 2 + lo;
  }
#pragma nv_exec_check_disable
  __host__ __device__ __forceinline__ void hang(uint32_t w, int end, uint32_t node) const {
    uint32_t* const at = Mem::ring() + (end & (RING - 1));
    const uint32_t old = *at;
    if (old != 0xffffffffu) Mem::node()[node] = old;
    *at = w | (old != 0xffffffffu ? node : 0xffffu) << 16;
  }
  // Take a slot off the ring word of iteration `end`.
#pragma nv_exec_check_disable
  __host__ __device__ __noinline__ static void unhang(uint32_t w, int end) {
    uint32_t* at = Mem::ring() + (end & (RING - 1));
    while (*at != 0xffffffffu) {
      const uint32_t next = *at >> 16;
      if ((*at & 0xffffu) == w) {
        *at = next == 0xffffu ? 0xffffffffu : Mem::node()[next];
      } else {
        if (next == 0xffffu) break;
        at = Mem::node() + next;
      }
    }
  }

  // Move (r, s) of iteration `it`, tabu up to `end`.  With LATE the slots are
  // hung by finish(), after the next barrier, unless the pairs' warps may read
  // the ring word by then.
#pragma nv_exec_check_disable
  template <bool LATE>
  __host__ __device__ __forceinline__ void apply(int r, int s, int it, int end) {
    const int at = s * (s - 1) / 2 + r;
    // a pair applied while tabu: its old end no longer counts
    int old = 0;
    if constexpr (M16) {
      uint16_t* const m = reinterpret_cast<uint16_t*>(mark);
      // the marks that end with the next iteration
      for (uint32_t x = Mem::ring()[(it + 1) & (RING - 1)]; x != 0xffffffffu;
           x = x >> 16 == 0xffffu ? 0xffffffffu : Mem::node()[x >> 16])
        m[pair_at((int)(x & 0xffffu))] = 0;
      old = m[at];  // with its top bit: the other 15 are 0 at multiples of 2^15
      m[at] = end > it + 1 ? (uint16_t)rot_mark16(end) : 0;
    } else {
      old = mark[at] > it + 1 ? mark[at] : 0;
      mark[at] = end;
    }
    // the ring word of the iteration just served is free again
    Mem::ring()[(it + 1) & (RING - 1)] = 0xffffffffu;
    late = make_int2(r << 8 | s, it);
    late_end = end;
    if (old != 0) {
      int2 w = slots(r, s);
#pragma unroll 1
      for (; w.x >= 0; w = make_int2(w.y, -1)) unhang((uint32_t)w.x, old);
    }
    if (!LATE || end <= it + 2) finish();
  }
  // The last move's slots on the ring.
  __host__ __device__ __forceinline__ void finish() {
    const int it = late.y;
    if (late_end > it + 1 && late_end <= iters) {
      int2 w = slots(late.x >> 8, late.x & 0xff);
      uint32_t node = 2 * ((uint32_t)it & (RING - 1));
#pragma unroll 1
      for (; w.x >= 0; w = make_int2(w.y, -1)) hang((uint32_t)w.x, late_end, node++);
    }
    late_end = 0;
  }
};

// The tabu times and the hash of a walk, kept by one warp beside the scan.
template <int NT, int C, typename FE>
struct RotKeeper : RotEnds<NT, C, RotSmem<NT, FE>> {
  using S = RotSmem<NT, FE>;
  static constexpr uint64_t kH0 = 14695981039346656037ull;
  const int p_stride;
  int32_t* const fq;
  uint64_t h, dh;
  bool was_tabu;

  __device__ __forceinline__ RotKeeper(const RotWalkArgs& W, const RotThread& T, int32_t* marks)
      : RotEnds<NT, C, S>(T.n2, T.nc, T.J, W.s.iters, marks), p_stride(W.s.p_stride),
        fq(W.s.freq ? W.s.freq + (size_t)W.row * W.s.p_stride * W.s.p_stride : nullptr), h(kH0),
        dh(kH0), was_tabu(!W.s.descend) {}

  // The tenure of an iteration, one of the 32 that the warp draws ahead.
  __device__ __noinline__ static void tenures(int it) {
    const RotWalkArgs& W = S::args();
    S::ten()[(it - 1) & 63] = RotTenure(W.s, W.I.n).of(W.s.seed, W.wid, it);
  }

  // Move (r, s) of iteration `it` (0 in the descent), by the whole warp.
  template <bool LATE>
  __device__ __forceinline__ void move(int r, int s, int it) {
    const int lane = threadIdx.x & 31;
    if (it > 0) {
      const int end = it + S::ten()[(it - 1) & 63];
      __syncwarp();  // (its place takes the tenure of iteration it + 64)
      if ((it & 31) == 0) tenures(it + 33 + lane);
      if (lane == 0) {
        this->template apply<LATE>(r, s, it, end);
        if (fq) atomicAdd(fq + s * p_stride + r, 1);
      }
      if (!was_tabu) {  // the first tabu move
        was_tabu = true;
        dh = h;
        h = kH0;
      }
    }
    h = fnv_step(h, r, s);
  }

  __device__ __forceinline__ void results(const SearchArgs& a, int row) {
    if ((threadIdx.x & 31) != 0) return;
    if (!was_tabu) {
      dh = h;
      h = kH0;
    }
    if (a.hash) a.hash[row] = h;
    if (a.descent_hash) a.descent_hash[row] = dh;
  }
};

// The phase X warps: one thread per index k (large n: two indices) computes what
// move (r, s) changes (see phase_m_prep for the algebra), and keeps the labels, the pending words,
// the tabu times and the walk's results.
//
// M's rows are brought up to date in turn, those with x mod Q = t mod Q after
// move t, by the last Q moves at once: byte (pair) t mod Q of the pending
// words belongs to move t.  A row's word is cleared when the row is done, so
// its entries' correction is one dp4a whatever the row's place in the turn.
template <int NT, int C, bool SYM, typename FE>
__device__ __forceinline__ void rot_phase_x() {
  constexpr int FB = sizeof(FE), KX = rot_kx(NT);
  // the last warp may be one of these
  constexpr bool KEEPS = rot_px(rot_max_n(NT), NT) + rot_owners(NT) > rot_threads(NT) - 32;
  constexpr bool PW2 = kRotWords<FE> == 2;
  using P = RotPending<NT, FE>;
  constexpr int RW = P::RW, LW = P::LW, Q = P::template Q<SYM>;
  constexpr bool M16 = rot_big(NT);
  constexpr int SB = rot_key_bits(NT);
  constexpr int BIG = 1 << (31 - SB);
  constexpr int TOP = 1 << (SB - 1);
  using X_ = RotFixed<NT, FE>;
  const RotWalkArgs& W = RotSmem<NT, FE>::args();
  const InstArgs& I = W.I;
  const RotThread T = rot_thread<NT, C>(I.n);
  const RotSmem<NT, FE> S(I, T.n, W.notr != 0);
  const int n = T.n, ldF = I.ldF, ldP = I.ldP, ldm = ld_m(n), nE = T.nE;
  const int g0 = I.g0, g2 = 2 * g0;
  // addresses
  const uint32_t base = smem_addr(rot_smem);
  const uint32_t aF = base + S.L.F, aP = base + S.L.P, aM = rot_big(NT) ? 0 : base + S.L.M;
  const uint32_t aFt = base + S.ft, aPt = base + S.pt, aMark = base + S.L.mark;
  const uint32_t aVw = base + X_::vw, aVwu = base + X_::vwu, aSig = base + X_::sigma;
  const uint32_t aX = base + X_::X, aPsi = base + X_::psi, aOwn = base + X_::own;
  const uint32_t aRr = base + X_::Rr, aRs = base + X_::Rs, aTen = base + X_::ten;
  char* const gM = reinterpret_cast<char*>(W.M);
  // per index of the thread (past the last: a repeat of n - 1 that stores
  // nothing)
  int k[KX], uk[KX], best_uk[KX], Fkk[KX], Qkk[KX], gk[KX];
  int2 wk[KX];  // the pending word(s) of row k
  bool live[KX];
#pragma unroll
  for (int j = 0; j < KX; ++j) {
    const int kj = T.pt + j * T.pxt;
    live[j] = kj < n;
    k[j] = min(kj, n - 1);
    uk[j] = best_uk[j] = k[j];
    wk[j] = make_int2(0, 0);
    Fkk[j] = S.F()[k[j] * ldF + k[j]];
    Qkk[j] = S.P()[k[j] * ldP + k[j]];
    gk[j] = (S.M()[k[j] * ldm + k[j]] << (SYM ? 1 : 0)) - g0;
  }
  int best_iter = 0, mv = 0;
  rot_clear_marks<NT>(S.mark(), n, T.ow);
  RotCourse<FE> course(W, T.ow);
  RotKeeper<NT, C, FE> keeper(W, T, S.mark());

  while (course.next(S.red())) {
    const int r = course.r, s = course.s, it = course.it;
    const bool tabu_phase = course.tabu_phase;
    const uint32_t oFr = aF + r * ldF * FB, oFs = aF + s * ldF * FB;
    const uint32_t oMr = aM + 4 * r * ldm, oMs = aM + 4 * s * ldm;
    const int ur = lds32(aSig + 4 * r), us = lds32(aSig + 4 * s);
    // the moves that the rows r, s and k of M do not hold yet
    const int rd = (mv & 1) * 4 * ldm, wt = 4 * ldm - rd;  // this move's buffers
    const int done = (mv - 1) & (Q - 1);                   // rows finished after the last move
    auto pending = [&](int x) {
      int2 w = make_int2(lds32(aVw + RW * rd + 4 * RW * x), 0);
      if constexpr (RW == 2) w.y = lds32(aVw + RW * rd + 4 * RW * x + 4);
      return (x & (Q - 1)) == done ? make_int2(0, 0) : w;
    };
    auto column = [&](int u) {
      int2 w = make_int2(lds32(aVwu + LW * rd + 4 * LW * u), 0);
      if constexpr (LW == 2) w.y = lds32(aVwu + LW * rd + 4 * LW * u + 4);
      return w;
    };
    // M's entries first: with large n they come from L2
    int Ar[KX], As[KX], Bs[KX], Br[KX];
#pragma unroll
    for (int j = 0; j < KX; ++j) {
      const uint32_t oMk = aM + 4 * ldm * k[j], u4 = 4 * (uint32_t)uk[j];
      Ar[j] = ldm32<NT>(gM, oMr + u4);
      As[j] = ldm32<NT>(gM, oMs + u4);
      Bs[j] = ldm32<NT>(gM, oMk + 4 * us);
      Br[j] = ldm32<NT>(gM, oMk + 4 * ur);
    }
    int mrs = ldm32<NT>(gM, oMr + 4 * us), msr = ldm32<NT>(gM, oMs + 4 * ur);
    const int2 wr = pending(r), ws = pending(s);
    const int fRR = ldsf<FE>(oFr + FB * r), fRS = ldsf<FE>(oFr + FB * s);
    const int fSS = ldsf<FE>(oFs + FB * s), fSR = SYM ? fRS : ldsf<FE>(oFs + FB * r);
    const int rtri = r * (r - 1) / 2, stri = s * (s - 1) / 2;
    const int ten = lds32(aTen + 4 * ((it - 1) & 63));
    const uint32_t oQr = aP + ur * ldP, oQs = aP + us * ldP;
    const int2 wur = column(ur), wus = column(us);
    const int qRR = lds8(oQr + ur), qRS = lds8(oQr + us), qSS = lds8(oQs + us);
    const int qSR = SYM ? qRS : lds8(oQs + ur);
    // the byte (pair) of the pending words that this move takes
    const int slot = mv & (Q - 1);
    const uint32_t selb = (0x3210u & ~(0xfu << (4 * (slot & 3)))) | 4u << (4 * (slot & 3));
    const uint32_t selh = slot & 1 ? 0x5410u : 0x3254u;
    const uint32_t sel = SYM ? selb : selh;
    const bool high = (SYM ? slot >> 2 : slot >> 1) != 0;  // of two dp4a words
    mrs = rot_entry<NT, FE>(wr, wus, mrs);
    msr = rot_entry<NT, FE>(ws, wur, msr);
    int gr, gs;
    if (SYM) {
      gr = 2 * (mrs - (fRR - fRS) * (qRS - qSS)) - g0;
      gs = 2 * (msr - (fRS - fSS) * (qRR - qRS)) - g0;
    } else {
      gr = mrs - (fRR - fRS) * (qSR - qSS) - (fRR - fSR) * (qRS - qSS) - g0;
      gs = msr - (fSR - fSS) * (qRR - qRS) - (fRS - fSS) * (qRR - qSR) - g0;
    }
    // the pair (r, s) itself only changes sign, and turns tabu
    const int drs = gr + gs - course.bd + (tabu_phase && ten > 1 ? BIG : 0);
#pragma unroll
    for (int j = 0; j < KX; ++j) {
      const int kj = k[j], uj = uk[j];
      const int Frk = ldsf<FE>(oFr + FB * kj), Fsk = ldsf<FE>(oFs + FB * kj);
      const int Fkr = SYM ? Frk : ldsf<FE>(aFt + FB * (r * S.fr + kj * S.fk));
      const int Fks = SYM ? Fsk : ldsf<FE>(aFt + FB * (s * S.fr + kj * S.fk));
      // whether the pairs {r, k} and {s, k} are tabu at the next iteration
      const int ktri = kj * (kj - 1) / 2;
      const int ar = kj < r ? rtri + kj : ktri + r, as = kj < s ? stri + kj : ktri + s;
      bool tabu_r, tabu_s;
      if constexpr (M16) {
        tabu_r = rot_tabu16(lds16u(aMark + 2 * ar), it);
        tabu_s = rot_tabu16(lds16u(aMark + 2 * as), it);
      } else {
        tabu_r = lds32(aMark + 4 * ar) > it + 1;
        tabu_s = lds32(aMark + 4 * as) > it + 1;
      }
      int2 wuk = column(uj);
      const int Qrk = lds8(oQr + uj), Qsk = lds8(oQs + uj);
      const int Qkr = SYM ? Qrk : lds8(aPt + ur * S.pr + uj * S.pk);
      const int Qks = SYM ? Qsk : lds8(aPt + us * S.pr + uj * S.pk);
      const int2 wkj = (kj & (Q - 1)) == done ? make_int2(0, 0) : wk[j];
      const int mAr = rot_entry<NT, FE>(wr, wuk, Ar[j]), mAs = rot_entry<NT, FE>(ws, wuk, As[j]);
      const int mBs = rot_entry<NT, FE>(wkj, wus, Bs[j]), mBr = rot_entry<NT, FE>(wkj, wur, Br[j]);
      const int av = Frk - Fsk, b = Qrk - Qsk;
      const int c = Fkr - Fks, e = Qkr - Qks;
      // the words of k in the pairs' update (int16 flows: (a, c), then (b, e))
      uint32_t own, word, own2 = 0, word2 = 0;
      if constexpr (PW2) {
        own = pack2(-av, -c);
        word = pack2(av, c);
        own2 = __byte_perm((uint32_t)-b, (uint32_t)-e, 0x0040u);
        word2 = __byte_perm((uint32_t)b, (uint32_t)e, 0x0040u);
      } else if constexpr (SYM) {
        own = __byte_perm((uint32_t)-av, (uint32_t)-b, 0x4400u);
        word = __byte_perm((uint32_t)b, (uint32_t)av, 0x4400u);
      } else {
        own = pack4(-av, -c, -b, -e);
        word = pack4(b, e, av, c);
      }
      int gn, Rr, Rs;
      if (SYM) {
        gn = gk[j] - 2 * av * b;
        Rr = 2 * (mAr + mBs + (qSS - qRS) * av - (fRR - fRS) * b) - g2 +
             (fRR + Fkk[j] - 2 * Frk) * (qSS + Qkk[j] - 2 * Qsk);
        Rs = 2 * (mAs + mBr + (qRS - qRR) * av - (fRS - fSS) * b) - g2 +
             (fSS + Fkk[j] - 2 * Fsk) * (qRR + Qkk[j] - 2 * Qrk);
      } else {
        gn = gk[j] - av * b - c * e;
        Rr = mAr + mBs - g2 + (fRR - Frk - Fkr + Fkk[j]) * (qSS - Qsk - Qks + Qkk[j]) -
             (fRR - fRS) * e - (fRR - fSR) * b + (qSS - qSR) * c + (qSS - qRS) * av;
        Rs = mAs + mBr - g2 + (fSS - Fsk - Fks + Fkk[j]) * (qRR - Qrk - Qkr + Qkk[j]) -
             (fSR - fSS) * e - (fRS - fSS) * b + (qRS - qRR) * c + (qSR - qRR) * av;
      }
      Rr += tabu_r ? BIG : 0;
      Rs += tabu_s ? BIG : 0;
      // M's operands of this move: (-a, -c) by index, bytes (b, e) by label
      // (symmetric: -a and b)
      int2 wn = wkj;
      if constexpr (PW2) {
        if constexpr (SYM) {
          const int hw = (int)__byte_perm((uint32_t)(slot & 2 ? wkj.y : wkj.x), own, selh);
          wn.x = slot & 2 ? wn.x : hw;
          wn.y = slot & 2 ? hw : wn.y;
        } else {
          wn.x = slot ? wn.x : (int)own;
          wn.y = slot ? (int)own : wn.y;
        }
        wuk.x = (int)__byte_perm((uint32_t)wuk.x, word2, sel);
      } else if constexpr (RW == 1) {
        wn.x = (int)__byte_perm((uint32_t)wkj.x, own, sel);
        wuk.x = (int)__byte_perm((uint32_t)wuk.x, word, sel);
      } else {
        const int hr = (int)__byte_perm((uint32_t)(high ? wkj.y : wkj.x), own, sel);
        const int hc = (int)__byte_perm((uint32_t)(high ? wuk.y : wuk.x), word, sel);
        wn.x = high ? wn.x : hr;
        wn.y = high ? hr : wn.y;
        wuk.x = high ? wuk.x : hc;
        wuk.y = high ? hc : wuk.y;
      }
      wk[j] = wn;
      const bool isr = kj == r, iss = kj == s;
      gn = isr ? gr : iss ? gs : gn;
      Rr = isr || iss ? drs : Rr;
      Rs = isr || iss ? drs : Rs;
      gk[j] = gn;
      if (live[j]) {
        const int psi = (int)(0u - ((uint32_t)gn << SB) - (1u << 30)) + (rot_rank(NT) ? TOP : kj);
        sts32(aX + 4 * kj, (int)word);
        sts32(aX + 4 * nE + 4 * kj, (int)word);
        if constexpr (PW2) {
          sts32(base + X_::X2 + 4 * kj, (int)word2);
          sts32(base + X_::X2 + 4 * nE + 4 * kj, (int)word2);
        }
        sts32(aPsi + 4 * kj, psi);
        sts32(aPsi + 4 * nE + 4 * kj, rot_rank(NT) ? psi - TOP : psi);
        if constexpr (!PW2) sts32(aOwn + 4 * kj, (int)own);
        else sts64(aOwn + 8 * kj, (int)own, (int)own2);
        sts32(aRr + 4 * kj, Rr);
        sts32(aRr + 4 * nE + 4 * kj, Rr);
        sts32(aRs + 4 * kj, Rs);
        sts32(aRs + 4 * nE + 4 * kj, Rs);
        if constexpr (RW == 1) sts32(aVw + wt + 4 * kj, wn.x);
        else sts64(aVw + 2 * wt + 8 * kj, wn.x, wn.y);
        if constexpr (LW == 1) sts32(aVwu + wt + 4 * uj, wuk.x);
        else sts64(aVwu + 2 * wt + 8 * uj, wuk.x, wuk.y);
      }
    }
    if (T.pt == 0) S.red()[33] = make_int2(r << 8 | s, tabu_phase ? it : 0);  // for the keeper
    __syncwarp();
    rot_barrier();
    // while the other warps bring the table up to date: M, the labels and the
    // best solution
    rot_update_m<NT, FE>(T, gM, aM, aVw + RW * wt, aVwu + LW * wt, n, ldm, Q, slot);
    ++mv;
    const bool better = !tabu_phase || course.cur < course.best;
#pragma unroll
    for (int j = 0; j < KX; ++j) {
      const bool isr = k[j] == r, iss = k[j] == s;
      uk[j] = isr ? us : iss ? ur : uk[j];
      Qkk[j] = isr ? qSS : iss ? qRR : Qkk[j];
      if (live[j] && (isr || iss)) sts32(aSig + 4 * k[j], uk[j]);
      best_uk[j] = better ? uk[j] : best_uk[j];
    }
    course.best = better ? course.cur : course.best;
    best_iter = better ? it : best_iter;  // 0 in the descent
    if (KEEPS && T.keeper) keeper.template move<false>(r, s, tabu_phase ? it : 0);
    __syncwarp();
  }

  // ---- outputs
  const SearchArgs& a = W.s;
  const int row = W.row;
#pragma unroll
  for (int j = 0; j < KX; ++j)
    if (a.best_p && live[j]) a.best_p[(size_t)row * a.p_stride + k[j]] = S.p0()[best_uk[j]];
  if (T.pt == 0) {
    a.best_cost[row] = (int64_t)course.best;
    if (a.final_cost) a.final_cost[row] = (int64_t)course.cur;
    if (a.best_iter) a.best_iter[row] = best_iter;
    if (a.iters_done) a.iters_done[row] = course.it;
    if (a.status) a.status[row] = course.stalled && course.it < course.iters ? 1 : 0;
    if (a.descent_moves) a.descent_moves[row] = course.dmoves;
  }
  if (KEEPS && T.keeper) keeper.results(a, row);
}

// The other warps: M's update, until the flag beside the candidates is set.
template <int NT, int C, typename FE>
__device__ __forceinline__ void rot_helper() {
  using P = RotPending<NT, FE>;
  using X_ = RotFixed<NT, FE>;
  const RotWalkArgs& W = RotSmem<NT, FE>::args();
  const RotThread T = rot_thread<NT, C>(W.I.n);
  const RotSmem<NT, FE> S(W.I, T.n, W.notr != 0);
  const int n = T.n, ldm = ld_m(n);
  const int Q = W.I.symF && W.I.symD ? P::template Q<true> : P::template Q<false>;
  const uint32_t base = smem_addr(rot_smem);
  rot_clear_marks<NT>(S.mark(), n, T.ow);
  RotKeeper<NT, C, FE> keeper(W, T, S.mark());
  for (int mv = 0;; ++mv) {
    rot_barrier();
    if (T.keeper) {
      if ((threadIdx.x & 31) == 0) keeper.finish();
      __syncwarp();
    }
    rot_barrier();
    if (lds32(base + X_::red + 8 * 32)) break;
    const int2 move = lds64(base + X_::red + 8 * 33);
    const uint32_t wt = mv & 1 ? 0 : 4 * ldm;
    if (T.keeper) keeper.template move<true>(move.x >> 8, move.x & 0xff, move.y);
    rot_update_m<NT, FE>(T, reinterpret_cast<char*>(W.M), rot_big(NT) ? 0 : base + S.L.M,
                         base + X_::vw + P::RW * wt, base + X_::vwu + P::LW * wt, n, ldm, Q,
                         mv & (Q - 1));
    __syncwarp();
  }
  if (T.keeper) keeper.results(W.s, W.row);
}

// The start of a walk: permutation, P0, M, the scan addends and the cost.
// Starts and ends with every thread of the CTA together.
template <int NT, int C, typename FE>
__device__ __forceinline__ void rot_start() {
  constexpr int TH = rot_threads(NT);
  RotWalkArgs& W = RotSmem<NT, FE>::args();
  const InstArgs& I = W.I;
  const SearchArgs& a = W.s;
  const bool notr = W.notr != 0;
  const int32_t* const start = W.start;
  const uint32_t wid = W.wid;
  const int n = I.n, ldF = I.ldF, ldP = I.ldP, tid = threadIdx.x;
  const RotSmem<NT, FE> S(I, n, notr);
  const int lane = tid & 31, warp = tid >> 5;
  const bool sym = I.symF && I.symD;
  const int ldm = ld_m(n), nE = 2 * rot_circle(n, C), g0 = I.g0;
  const int hsh = sym ? 1 : 0;  // M is stored halved
  constexpr int SB = rot_key_bits(NT);

  // ---- start permutation: given, or Fisher-Yates on stream 0 (the draws by
  // all threads, the exchanges by one)
  if (start) {
#pragma unroll 1
    for (int x = tid; x < n; x += TH) S.p0()[x] = start[x];
  } else {
#pragma unroll 1
    for (int i = tid; i < n; i += TH) {
      S.p0()[i] = i;
      if (i >= 1) S.vw()[i] = (int)below(walk_draw(a.seed, wid, 0u, (uint32_t)(n - 1 - i)),
                                         (uint32_t)(i + 1));
    }
    __syncthreads();
    if (tid == 0)
      for (int i = n - 1; i >= 1; --i) {
        const int j = S.vw()[i];
        const int32_t t = S.p0()[i];
        S.p0()[i] = S.p0()[j];
        S.p0()[j] = t;
      }
  }
  __syncthreads();

  // ---- P0 = D[p0][p0] gathered from global memory, and the walk's state
  {
    const int8_t* Dg = static_cast<const int8_t*>(I.D);
    const bool tr = !I.symD && !notr;
    int8_t* Pt = S.Pt();
#pragma unroll 1
    for (int i = warp; i < n; i += TH / 32) {
      const int8_t* Di = Dg + (size_t)S.p0()[i] * n;
      for (int j = lane; j < n; j += 32) {
        const int8_t v = Di[S.p0()[j]];
        S.P()[i * ldP + j] = v;
        if (tr) Pt[j * ldP + i] = v;
      }
    }
#pragma unroll 1
    for (int x = tid; x < n; x += TH) S.sigma()[x] = x;
    // phantom indices: never candidates, never updated
#pragma unroll 1
    for (int x = n + tid; x < nE; x += TH) {
      S.X()[x] = S.X()[x + nE] = 0;
      S.psi()[x] = S.psi()[x + nE] = INT_MAX - 128;
      S.Rr()[x] = S.Rr()[x + nE] = S.Rs()[x] = S.Rs()[x + nE] = 0;
      for (int w = 0; w < kRotWords<FE>; ++w) S.own()[kRotWords<FE> * x + w] = 0;
      if (kRotWords<FE> == 2) S.X2()[x] = S.X2()[x + nE] = 0;
    }
    // no pending moves; M's padding columns take updates from these words only
    using Pd = RotPending<NT, FE>;
#pragma unroll 1
    for (int x = tid; x < 2 * Pd::LW * ldm; x += TH) S.vwu()[x] = 0;
#pragma unroll 1
    for (int x = tid; x < 2 * Pd::RW * ldm; x += TH) S.vw()[x] = 0;
#pragma unroll 1
    for (int x = tid; x < rot_ring(NT); x += TH) S.ring()[x] = 0xffffffffu;
    if (a.iters > 0) {
      const RotTenure tenure(a, n);
#pragma unroll 1
      for (int x = tid; x < 64; x += TH) S.ten()[x] = tenure.of(a.seed, wid, x + 1);
    }
    if (tid == 0) S.red()[32] = make_int2(0, 0);
  }
  __syncthreads();
  rot_compute_m<NT, FE>(S, n, ldF, ldP, sym, notr);
  __syncthreads();

  // ---- the pairs' table, in the marks' place (large n: they are too small)
  if (!rot_big(NT))
    for (int v = 1 + warp; v < n; v += rot_threads(NT) / 32)
      for (int u = lane; u < v; u += 32) S.mark()[v * (v - 1) / 2 + u] = rot_pair(S, I, u, v);

  // ---- scan addends of every index; the walk's cost (Eq. 1): M's diagonal
  // sums to twice the cost
  int64_t c0 = 0;
#pragma unroll 1
  for (int x = tid; x < n; x += TH) {
    const int mxx = S.M()[x * ldm + x];
    c0 += mxx;
    const uint32_t psi = 0u - ((uint32_t)((mxx << hsh) - g0) << SB) - (1u << 30);
    S.psi()[x] = (int)(psi + (rot_rank(NT) ? 1 << (SB - 1) : x));
    S.psi()[x + nE] = (int)(psi + (rot_rank(NT) ? 0 : x));
  }
  c0 = block_sum<TH>(c0, S.sum());
  if (tid == 0) W.cost = sym ? c0 : c0 >> 1;
  if (a.freq) {
    int32_t* fq = a.freq + (size_t)W.row * a.p_stride * a.p_stride;
    for (int c = tid; c < a.p_stride * a.p_stride; c += TH) fq[c] = 0;
  }
  __syncthreads();
}

// One whole walk of the instance in shared memory (see RotWalkArgs).  Starts
// and ends with every thread of the CTA together.
template <int NT, int C, typename FE>
__device__ __forceinline__ void rot_walk() {
  rot_start<NT, C, FE>();
  const RotWalkArgs& W = RotSmem<NT, FE>::args();
  const int role = rot_thread<NT, C>(W.I.n).role;
  const bool sym = W.I.symF && W.I.symD;
  if (role == 0) rot_owner<NT, C, FE>();
  else if (role == 1 && sym) rot_phase_x<NT, C, true, FE>();
  else if (role == 1) rot_phase_x<NT, C, false, FE>();
  else rot_helper<NT, C, FE>();
  __syncthreads();
}

// The instance into shared memory: F (and F^T); P (and P^T) zeroed so that
// their padding columns stay zero.  Ends with a barrier.
template <int NT, typename FE>
__device__ __forceinline__ void rot_load(const InstArgs& I, bool notr) {
  const RotLayout L = rot_layout(I.n, I.ldF, sizeof(FE), I.ldP, I.symF, I.symD, notr,
                                 rot_big(NT), RotFixed<NT, FE>::bytes);
  const bool ft = !I.symF && !notr, pt = !I.symD && !notr;
  const int tid = threadIdx.x;
  const int fvec = I.n * I.ldF * (int)sizeof(FE) / 16, pvec = I.n * I.ldP / 16;
  const int4* gF = static_cast<const int4*>(I.F);
  const int4* gFt = static_cast<const int4*>(I.Ft);
#pragma unroll 2
  for (int i = tid; i < fvec; i += rot_threads(NT)) {
    rot_at<int4>(L.F)[i] = gF[i];
    if (ft) rot_at<int4>(L.Ft)[i] = gFt[i];
  }
  const int4 zero = make_int4(0, 0, 0, 0);
#pragma unroll 2
  for (int i = tid; i < pvec; i += rot_threads(NT)) {
    rot_at<int4>(L.P)[i] = zero;
    if (pt) rot_at<int4>(L.Pt)[i] = zero;
  }
  __syncthreads();
}

// CTAs per SM to compile for.
constexpr int rot_min_blocks(int nt) { return nt == 128 ? 4 : nt == 256 ? 2 : 1; }

// Walks of one instance (b.single: CTAs step over its walks) or of many (CTAs
// take items from the counter and reload the instance when it changes).
template <int NT, int C, typename FE>
__global__ void __launch_bounds__(rot_threads(NT), rot_min_blocks(NT)) rot_kernel(const BatchArgs b) {
  __shared__ int item_s;
  RotWalkArgs& W = RotSmem<NT, FE>::args();
  int cur_inst = -1, item = blockIdx.x;
  for (;; item += gridDim.x) {
    if (!b.single) {
      if (threadIdx.x == 0) item_s = atomicAdd(b.counter, 1);
      __syncthreads();
      item = item_s;
    }
    if (item >= b.items) break;
    const int inst = b.single ? 0 : b.item_inst[item];
    const InstArgs* const I = b.single ? &b.inst : b.insts + inst;
    if (inst != cur_inst) rot_load<NT, FE>(*I, b.notr != 0);
    if (threadIdx.x == 0) {
      if (inst != cur_inst) {
        W.I = *I;
        W.s = b.s;
        W.notr = b.notr;
        W.M = reinterpret_cast<int32_t*>(b.ws ? b.ws + b.ws_stride * blockIdx.x : nullptr);
      }
      const int w = b.single ? b.walk_offset + item : b.item_walk[item];
      W.row = b.single ? w : b.row_base[inst] + w;
      W.wid = b.s.walk_base + (uint32_t)w;
      W.start = b.starts ? b.starts + (size_t)w * I->n : nullptr;
    }
    cur_inst = inst;
    __syncthreads();
    rot_walk<NT, C, FE>();
  }
}

}  // namespace qapk
