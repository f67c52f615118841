// smem.cuh -- certificates and bridges of one graph of up to 4,096 vertices in shared memory, by a
// group of threads: the batched kernels, the one-block forms of small calls (batched.cu) and the
// core of the final stage's reduced graph (final.cu, up to 3,616 vertices) share this code.  Nothing here is visible through the C ABI.
#pragma once

#include "../../include/bridges.h"
#include "batched.h"
#include "common.cuh"
#include "stream.cuh"

namespace bridges {
namespace {

constexpr int kT = 1024;           // threads per block
constexpr int kVmax = kBatchVmax;  // 4096: a whole block's graph
constexpr int kHalfT = kT / 2;     // threads of a half-block group
constexpr int kHalfVmax = kBatchHalfVmax;  // 3008: a half-block group's graph
constexpr int kQuarterT = kT / 4;     // threads of a quarter-block group
constexpr int kQuarterVmax = kBatchQuarterVmax;  // 1024: a quarter-block (certification) group's graph
constexpr uint16_t kNone16 = 0xffff;
constexpr int kRuleGap = 8;  // list ranking: a ruler every kRuleGap arcs (by index)

constexpr int a16(int x) { return (x + 15) & ~15; }
// Shared-memory layout for graphs of up to VM vertices (bytes, each region a multiple of 16),
// in address order R0, R2, R1, R3, ...:
//   R0  P1 (int32[V]); later each arc's ruler (u16[2V]); later aoff + vbase (u16[V+1] each);
//       later the chunk tables of the range test
//   R1  P2 (int32[V]); later root + cur (u16[V+2] each)
//   R2  F list (u32[V]); later the reduced graph's tree edges (s_contract); later the bridges found
//   R3  F' list (u32[V]); later the reduced graph's further edges, from the front, and its tree edges'
//       original ends, from the back
//   R4  chunk minima / maxima (int32[V/32] each)
//   R5  head (int32[V]); later lo (int32[V]); before the stage the reduced vertices' numbers, or,
//       with R6, a merge's staging copy
//   R6  next (u16[2V]); later each arc's place in its sublist; later hi (int32[V]); before the stage
//       the F edges between F' components (places in F1, then tokens)
//   R7  succ (u16[2V]); before the stage the reduced ends of R6's edges; later dflag / dscan (u16[2V+1]); later in-chunk prefix extrema (u16[V] x 2)
//   R8  rnk (u16[2V]); later the vertex at each preorder position
//   R9  pre, sz, par (u16[V] each); earlier the rulers' two packed buffers (3 VM / 4 words each)
template <int VM>
struct Layout {
  static constexpr int kU16 = a16(2 * (VM + 16));  // a u16[V+2] array
  static constexpr int R0 = 2 * kU16 > 4 * VM ? 2 * kU16 : 4 * VM;
  static constexpr int R1 = R0;
  static constexpr int R2 = 4 * VM;
  static constexpr int R3 = 4 * VM;
  static constexpr int R4 = VM / 4;
  static constexpr int R5 = 4 * VM;
  static constexpr int R6 = 4 * VM;
  static constexpr int R7 = a16(2 * (2 * VM + 8));
  static constexpr int R8 = 4 * VM;
  static constexpr int R9 = 6 * VM;
  static constexpr int kBytes = R0 + R1 + R2 + R3 + R4 + R5 + R6 + R7 + R8 + R9;
};
constexpr int cmax(int a, int b) { return a > b ? a : b; }
// a half block's share holds one half-group layout
constexpr int kHalfBytes = Layout<kHalfVmax>::kBytes;
constexpr int kSmem = cmax(Layout<kVmax>::kBytes, 2 * kHalfBytes);
static_assert(kHalfVmax % 32 == 0 && kHalfBytes % 16 == 0, "half layouts: whole chunks, 16-byte regions");
static_assert(kSmem + 2048 <= 227 * 1024, "the bridge kernel's shared memory (with its static part) fits a block");

struct Smem {
  int32_t* P1;
  int32_t* P2;
  uint32_t* F1;
  uint32_t* F2;
  uint16_t* aoff;
  uint16_t* vbase;
  uint16_t* root;
  uint16_t* cur;
  uint32_t* keys;
  int32_t* chunk;
  uint16_t* dst;
  int32_t* head;
  uint16_t* next;
  int32_t* lo;
  int32_t* hi;
  uint16_t* succ;
  uint16_t* dflag;
  uint16_t* rnk;
  uint16_t* pre;
  uint16_t* sz;
  uint16_t* par;
};

template <int VM>
__device__ Smem carve_smem(char* base) {
  using L = Layout<VM>;
  Smem s;
  char* c = base;
  s.P1 = reinterpret_cast<int32_t*>(c);
  s.aoff = reinterpret_cast<uint16_t*>(c);
  s.vbase = reinterpret_cast<uint16_t*>(c + L::kU16);
  c += L::R0;
  s.F1 = reinterpret_cast<uint32_t*>(c);
  s.keys = s.F1;
  c += L::R2;
  s.P2 = reinterpret_cast<int32_t*>(c);
  s.root = reinterpret_cast<uint16_t*>(c);
  s.cur = reinterpret_cast<uint16_t*>(c + L::kU16);
  c += L::R1;
  s.F2 = reinterpret_cast<uint32_t*>(c);
  c += L::R3;
  s.chunk = reinterpret_cast<int32_t*>(c);
  c += L::R4;
  s.dst = reinterpret_cast<uint16_t*>(c);
  s.head = reinterpret_cast<int32_t*>(c);
  s.lo = reinterpret_cast<int32_t*>(c);
  c += L::R5;
  s.next = reinterpret_cast<uint16_t*>(c);
  s.hi = reinterpret_cast<int32_t*>(c);
  c += L::R6;
  s.succ = reinterpret_cast<uint16_t*>(c);
  s.dflag = s.succ;
  c += L::R7;
  s.rnk = reinterpret_cast<uint16_t*>(c);
  c += L::R8;
  s.pre = reinterpret_cast<uint16_t*>(c);
  s.sz = s.pre + VM;
  s.par = s.sz + VM;
  return s;
}

// A group of NT threads (whole block, a half or a quarter) working on one task: its thread index
// and its barrier (0 = the block's; named barriers 1, 2 for the bridge kernel's halves and 1 to 4
// for the certification groups, the quarters).
template <int NT>
struct Grp {
  int tid;
  int bar;
  __device__ __forceinline__ void sync() const {
    if (NT == kT)
      __syncthreads();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(NT) : "memory");
  }
};

// Per-group scalars in shared memory.
struct GroupShared {
  int32_t red[kT / 32];
  int32_t red_b[kT / 32];
  int32_t task, n1, n2, err, sh;
  int32_t kept, verts, tree, rest;  // the reduced graph (s_contract)
};

// Concurrent union-find in shared memory: the algorithm of uf_link (common.cuh) -- parents are
// compared first (a grandparent equal to the other end's parent also proves one set), a root is
// hooked under the other end's parent, a smaller vertex, so P[x] <= x always.
__device__ __forceinline__ bool s_link(int32_t* P, int32_t a, int32_t b) {
  volatile int32_t* VP = P;
  int32_t x = a, y = b;
  while (true) {
    int32_t px = VP[x], py = VP[y];
    if (px == py) return false;
    if (px < py) {
      int32_t t = x;
      x = y;
      y = t;
      t = px;
      px = py;
      py = t;
    }
    if (px == x) {
      if (atomicCAS(P + x, x, py) == x) return true;
      continue;
    }
    const int32_t g = VP[px];
    if (g == py) {
      VP[x] = g;
      return false;
    }
    if (g == px) {
      if (atomicCAS(P + px, px, py) == px) return true;
      continue;
    }
    VP[x] = g;
    x = g;
  }
}

// Block-wide exclusive scan of n (<= 2*NT*... ) u16 values in place; returns the total.
template <int NT>
__device__ int32_t block_scan16(const Grp<NT>& G, uint16_t* a, int32_t n, int32_t* red) {
  const int per = (n + NT - 1) / NT;  // contiguous items per thread
  const int lo = min(n, G.tid * per), hi = min(n, lo + per);
  int32_t s = 0;
  for (int i = lo; i < hi; i++) s += a[i];
  const int lane = G.tid & 31, w = G.tid >> 5;
  int32_t incl = s;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) red[w] = incl;
  G.sync();
  int32_t base = 0, tot = 0;
  for (int k = 0; k < (NT / 32); k++) {
    if (k < w) base += red[k];
    tot += red[k];
  }
  int32_t run = base + incl - s;
  for (int i = lo; i < hi; i++) {
    const int32_t v = a[i];
    a[i] = (uint16_t)run;
    run += v;
  }
  G.sync();
  return tot;
}

// The same for two arrays of equal length at once (one pair of block barriers for both).
template <int NT>
__device__ void block_scan16_pair(const Grp<NT>& G, uint16_t* a, uint16_t* b, int32_t n, int32_t* red,
                                  int32_t* red_b) {
  const int per = (n + NT - 1) / NT;
  const int lo = min(n, G.tid * per), hi = min(n, lo + per);
  int32_t sa = 0, sb = 0;
  for (int i = lo; i < hi; i++) {
    sa += a[i];
    sb += b[i];
  }
  const int lane = G.tid & 31, w = G.tid >> 5;
  int32_t ia = sa, ib = sb;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t ya = __shfl_up_sync(kFull, ia, o), yb = __shfl_up_sync(kFull, ib, o);
    if (lane >= o) {
      ia += ya;
      ib += yb;
    }
  }
  if (lane == 31) {
    red[w] = ia;
    red_b[w] = ib;
  }
  G.sync();
  int32_t ba = 0, bb = 0;
  for (int k = 0; k < w; k++) {
    ba += red[k];
    bb += red_b[k];
  }
  int32_t ra = ba + ia - sa, rb = bb + ib - sb;
  for (int i = lo; i < hi; i++) {
    const int32_t va = a[i], vb = b[i];
    a[i] = (uint16_t)ra;
    b[i] = (uint16_t)rb;
    ra += va;
    rb += vb;
  }
  G.sync();
}

// Offers edge (a, b) to F, then F'; put(which, place, a, b) takes each winner (1: F, 2: F'), the places
// counted warp-aggregated.  Every lane calls it.
template <class Put>
__device__ __forceinline__ void s_settle(int32_t* P1, int32_t* P2, bool need, int32_t a, int32_t b, int32_t* n1,
                                         int32_t* n2, Put put) {
  if (!__any_sync(kFull, need)) return;
  int r = 0;
  if (need) r = s_link(P1, a, b) ? 1 : (s_link(P2, a, b) ? 2 : 0);
  const unsigned m1 = __ballot_sync(kFull, r == 1), m2 = __ballot_sync(kFull, r == 2);
  const int lane = threadIdx.x & 31;  // groups are whole warps
  int32_t b1 = 0, b2 = 0;
  if (m1 && lane == __ffs(m1) - 1) b1 = atomicAdd(n1, __popc(m1));
  if (m2 && lane == __ffs(m2) - 1) b2 = atomicAdd(n2, __popc(m2));
  if (m1) b1 = __shfl_sync(kFull, b1, __ffs(m1) - 1);
  if (m2) b2 = __shfl_sync(kFull, b2, __ffs(m2) - 1);
  if (r == 1)
    put(1, b1 + __popc(m1 & lanemask_lt()), a, b);
  else if (r == 2)
    put(2, b2 + __popc(m2 & lanemask_lt()), a, b);
}

// The same with the winners packed into S's lists.
__device__ __forceinline__ void s_settle(const Smem& S, bool need, int32_t a, int32_t b, int32_t* n1, int32_t* n2,
                                         int32_t V) {
  s_settle(S.P1, S.P2, need, a, b, n1, n2, [&](int which, int32_t i, int32_t x, int32_t y) {
    if (i < V) (which == 1 ? S.F1 : S.F2)[i] = (uint32_t)x | ((uint32_t)y << 16);
  });
}

// Points every vertex straight at its root (no link runs meanwhile), so that afterwards "equal
// parents" recognises every pair that shares a set.
template <int NT>
__device__ __forceinline__ void s_flatten(const Grp<NT>& G, int32_t* P, int32_t V) {
  G.sync();
  for (int x = G.tid; x < V; x += NT) {
    int32_t r = x, p = P[x];
    while (p != r) {
      r = p;
      p = P[r];
    }
    P[x] = r;
  }
  G.sync();
}

// Scalar certification of edges [lo, hi): every lane takes one edge per step.
template <int NT>
__device__ void s_certify_scalar(const Grp<NT>& G, const Smem& S, const int32_t* __restrict__ u, const int32_t* __restrict__ v,
                                 int64_t lo, int64_t hi, int32_t V, int32_t* n1, int32_t* n2, int32_t* err,
                                 uint32_t stride = 0) {
  volatile int32_t* P2 = S.P2;
  // the next step's edge is loaded before this step's union-find work, so the load's latency
  // overlaps it instead of adding to every step
  int64_t i = lo + G.tid;
  int32_t a = i < hi ? __ldcs(u + i) : 0, b = i < hi ? __ldcs(v + i) : 0;
  for (int64_t t0 = lo; t0 < hi; t0 += NT, i += NT) {
    const bool valid = i < hi;
    const int64_t j = i + NT;
    const int32_t na = j < hi ? __ldcs(u + j) : 0, nb = j < hi ? __ldcs(v + j) : 0;
    bool need = valid;
    if (need && ((uint32_t)a >= (uint32_t)V || (uint32_t)b >= (uint32_t)V)) {
      *err = BRIDGES_ERANGE;
      need = false;
    }
    if (need && (a == b || P2[a] == P2[b] || excluded(i, stride))) need = false;
    s_settle(S, need, a, b, n1, n2, V);
    a = na;
    b = nb;
  }
}

// The lanes' flagged edges of one tile go through the union-finds (bit 4k+c of m: element
// 4*(base + k*NT + tid) + c of ub / vb).  Out of line: rare after the flatten.
template <int NT>
__device__ __noinline__ void s_offer_misses(const Grp<NT>& G, const Smem& S, uint32_t m, const int32_t* __restrict__ ub,
                                            const int32_t* __restrict__ vb, int64_t base, int32_t V, int32_t* n1,
                                            int32_t* n2, int32_t* err, int64_t first, uint32_t stride) {
  while (__any_sync(kFull, m != 0)) {
    int32_t a = 0, b = 0;
    bool go = false;
    if (m) {
      const int bit = __ffs(m) - 1;
      m &= m - 1;
      const int64_t e = 4 * (base + (int64_t)(bit >> 2) * NT + G.tid) + (bit & 3);
      a = ub[e];
      b = vb[e];
      if ((uint32_t)a >= (uint32_t)V || (uint32_t)b >= (uint32_t)V)
        *err = BRIDGES_ERANGE;
      else
        go = a != b && !excluded(first + e, stride);
    }
    s_settle(S, go, a, b, n1, n2, V);
  }
}

// Certifies edges [lo, hi) of (u, v) with 16-byte loads when u and v share their alignment (a
// scalar head and tail otherwise), four units of four edges per thread in flight, a per-thread
// miss mask (the ends' F' parents differ, or an id is out of range) and one warp vote per tile.
template <int NT, int VM>
__device__ __forceinline__ void s_certify_vec(const Grp<NT>& G, const Smem& S, const int32_t* __restrict__ u, const int32_t* __restrict__ v, int64_t lo,
                              int64_t hi, int32_t V, int32_t* n1, int32_t* n2, int32_t* err, uint32_t stride = 0) {
  constexpr int U = 4;
  if (lo >= hi) return;
  // the vector body starts on a 128-byte line of both arrays when they share their offset within
  // a line (a warp's 512 bytes of loads then touch four lines, not five), else on a 16-byte boundary
  const uintptr_t d = reinterpret_cast<uintptr_t>(u) ^ reinterpret_cast<uintptr_t>(v);
  const uintptr_t amask = (d & 127) == 0 ? 127 : 15;
  int64_t body = lo;
  if ((d & 15) == 0) {
    while (body < hi && (reinterpret_cast<uintptr_t>(u + body) & amask)) body++;
  } else {
    body = hi;
  }
  s_certify_scalar(G, S, u, v, lo, body, V, n1, n2, err, stride);
  const int64_t nunits = (hi - body) >> 2;
  const int32_t* ub = u + body;
  const int32_t* vb = v + body;
  const int4* u4 = reinterpret_cast<const int4*>(ub);
  const int4* v4 = reinterpret_cast<const int4*>(vb);
  volatile int32_t* P2 = S.P2;
  const uint32_t cl = (uint32_t)(VM - 1);
  for (int64_t base = 0; base < nunits; base += (int64_t)NT * U) {
    int4 ua[U], va[U];
#pragma unroll
    for (int k = 0; k < U; k++) {
      const int64_t idx = base + (int64_t)k * NT + G.tid;
      if (idx < nunits) {
        ua[k] = __ldcs(u4 + idx);
        va[k] = __ldcs(v4 + idx);
      } else {
        ua[k] = make_int4(0, 0, 0, 0);
        va[k] = make_int4(0, 0, 0, 0);
      }
    }
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < U; k++) {
      if (base + (int64_t)k * NT + G.tid >= nunits) continue;
      const int32_t as[4] = {ua[k].x, ua[k].y, ua[k].z, ua[k].w};
      const int32_t bs[4] = {va[k].x, va[k].y, va[k].z, va[k].w};
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const uint32_t a = (uint32_t)as[c], b = (uint32_t)bs[c];
        const bool bad = a >= (uint32_t)V || b >= (uint32_t)V;
        const bool same_set = P2[min(a, cl)] == P2[min(b, cl)];
        m |= (uint32_t)(bad || !same_set) << (4 * k + c);
      }
    }
    if (__any_sync(kFull, m != 0)) s_offer_misses(G, S, m, ub, vb, base, V, n1, n2, err, body, stride);
  }
  s_certify_scalar(G, S, u, v, body + 4 * nunits, hi, V, n1, n2, err, stride);
}

// Certifies edges [lo, hi) of (u, v) into S.F1 / S.F2 (appending to *n1 / *n2); ids outside
// [0, V) set *err.  A warm-up prefix goes edge by edge (most of its edges still link; a vector
// tile's miss loop would run as long as its busiest lane), then both union-finds are flattened,
// so that "equal F' parents" afterwards recognises nearly every pair inside one F' component,
// and the rest streams through the vector loop.
template <int NT, int VM>
__device__ void s_certify_range(const Grp<NT>& G, const Smem& S, const int32_t* __restrict__ u, const int32_t* __restrict__ v,
                                int64_t lo, int64_t hi, int64_t warm_edges, int32_t V, int32_t* n1, int32_t* n2,
                                int32_t* err) {
  // the task's prefix (the host's plan: 4V + 2048 unless tuned)
  const int64_t warm = min(hi - lo, max(warm_edges, (int64_t)0));
  s_certify_scalar(G, S, u, v, lo, lo + warm, V, n1, n2, err);
  lo += warm;
  if (lo >= hi) return;
  s_flatten(G, S.P1, V);
  s_flatten(G, S.P2, V);
  s_certify_vec<NT, VM>(G, S, u, v, lo, hi, V, n1, n2, err);
}

// ---- a sample certified in rounds, in shared memory ----
// The rounds of sample_kernel (sample.cu) for one group and a graph of up to kVmax vertices: all edges
// of the sample advance together, and a round's two barriers are block barriers.  (Edge by edge through
// the union-finds a step of 1,024 edges takes 3.5 us while the sets form: every lane's chain of
// dependent accesses and retries, and the warp waits for its longest.)
constexpr int kLoBits = 12;  // a hook: the edge's key, and the vertex above in the low bits
static_assert(kVmax <= 1 << kLoBits, "a vertex fits the low bits of a hook");
constexpr uint32_t kKeyMask = (1u << (32 - kLoBits)) - 1;
constexpr uint32_t kKeyMul = 0x9e3779b1u & kKeyMask;  // odd: slots and keys are in bijection
constexpr uint32_t inverse_mod_2_32(uint32_t x) {     // of an odd number, by Newton's iteration
  uint32_t y = x;
  for (int i = 0; i < 5; i++) y *= 2 - x * y;
  return y;
}
constexpr uint32_t kKeyInv = inverse_mod_2_32(kKeyMul) & kKeyMask;
static_assert(((kKeyMul * kKeyInv) & kKeyMask) == 1, "the key's inverse");
constexpr uint32_t kFree = 0xffffffffu;  // no hook (vertex 4095 never stands above another one)

// Slots of a sample of `groups` groups of 2^kSampleShift edges, every stride-th one of a list of n:
// loads them packed into ed (loops and, with *err set, edges out of range as 0, a loop).
template <int NT>
__device__ void s_load_sample(const Grp<NT>& G, uint32_t* ed, const int32_t* __restrict__ u,
                              const int32_t* __restrict__ v, int64_t n, int64_t stride, int32_t groups, int32_t V,
                              int32_t* err) {
  constexpr int kAhead = 4;
  const int32_t slots = groups << kSampleShift;
  for (int32_t base = G.tid; base < slots; base += kAhead * NT) {
    int32_t a[kAhead], b[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; k++) {
      const int32_t i = base + k * NT;
      const int64_t e = ((i >> kSampleShift) * stride << kSampleShift) | (i & ((1 << kSampleShift) - 1));
      a[k] = b[k] = -1;
      if (i < slots && e < n) {
        a[k] = __ldg(u + e);
        b[k] = __ldg(v + e);
      } else if (i < slots) {
        a[k] = b[k] = 0;
      }
    }
#pragma unroll
    for (int k = 0; k < kAhead; k++) {
      const int32_t i = base + k * NT;
      if (i >= slots) continue;
      const bool past = ((i >> kSampleShift) * stride << kSampleShift | (i & ((1 << kSampleShift) - 1))) >= n;
      const bool bad = !past && ((uint32_t)a[k] >= (uint32_t)V || (uint32_t)b[k] >= (uint32_t)V);
      if (bad) *err = BRIDGES_ERANGE;
      ed[i] = bad || past || a[k] == b[k] ? 0u : (uint32_t)a[k] | ((uint32_t)b[k] << 16);
    }
  }
  G.sync();
}

// F and F' of the slots in ed (consumed).  R: V words, left holding each vertex's root in F (low half)
// and in F' (high half); H1, H2: V words of scratch each.  put(which, a, b, warp-aggregated place)
// takes the winners, counted in *n1 and *n2.
template <int NT, class Put>
__device__ void s_certify_rounds(const Grp<NT>& G, uint32_t* ed, int32_t slots, int32_t V, uint32_t* R, uint32_t* H1,
                                 uint32_t* H2, int32_t* n1, int32_t* n2, int32_t* any, Put put) {
  volatile uint32_t* Rv = R;
  for (int x = G.tid; x < V; x += NT) {
    R[x] = (uint32_t)x * 0x10001u;
    H1[x] = kFree;
    H2[x] = kFree;
  }
  if (G.tid < 2) any[G.tid] = 0;
  G.sync();
  for (int t = 0;; t++) {
    // A: offers
    const int32_t in = min(slots, t < 3 ? 2 * V : (t == 3 ? 4 * V : slots));
    bool live = in < slots;
    for (int32_t i = G.tid; i < in; i += NT) {
      const uint32_t p = ed[i];
      if (p == 0) continue;
      const uint32_t ra = R[p & 0xffff], rb = R[p >> 16];
      if (ra == rb) {
        ed[i] = 0;
        continue;
      }
      uint32_t x = ra & 0xffff, y = rb & 0xffff;
      const bool second = x == y;
      if (second) {
        x = ra >> 16;
        y = rb >> 16;
        if (x == y) {  // (the F roots differ: not reached)
          ed[i] = 0;
          continue;
        }
      }
      live = true;
      const uint32_t hi = max(x, y), mine = (((uint32_t)i * kKeyMul) & kKeyMask) << kLoBits | min(x, y);
      uint32_t* h = (second ? H2 : H1) + hi;
      if (*reinterpret_cast<volatile uint32_t*>(h) > mine) atomicMin(h, mine);
    }
    if (__any_sync(kFull, live) && (threadIdx.x & 31) == 0) any[t & 1] = 1;
    G.sync();
    const bool more = any[t & 1] != 0;
    if (G.tid == 0) any[(t + 1) & 1] = 0;  // (last read before the barrier that ended round t - 1)
    if (!more) break;
    // B: each root hooked in this round names its edge; C: new roots
    const int lane = threadIdx.x & 31;
    for (int32_t base = G.tid - lane; base < V; base += NT) {
      const int32_t x = base + lane;
      uint32_t r = x < V ? R[x] : 0;
      uint32_t r1 = r & 0xffff, r2 = r >> 16;
      uint32_t h1 = x < V ? H1[r1] : kFree, h2 = x < V ? H2[r2] : kFree;
      const bool w1 = h1 != kFree && r1 == (uint32_t)x, w2 = h2 != kFree && r2 == (uint32_t)x;
      const unsigned m1 = __ballot_sync(kFull, w1), m2 = __ballot_sync(kFull, w2);
      int32_t b1 = 0, b2 = 0;
      if (lane == 0) {
        if (m1) b1 = atomicAdd(n1, __popc(m1));
        if (m2) b2 = atomicAdd(n2, __popc(m2));
      }
      b1 = __shfl_sync(kFull, b1, 0) + __popc(m1 & lanemask_lt());
      b2 = __shfl_sync(kFull, b2, 0) + __popc(m2 & lanemask_lt());
      if (w1) {
        const uint32_t slot = ((h1 >> kLoBits) * kKeyInv) & kKeyMask, p = ed[slot];
        put(1, b1, p);
        ed[slot] = 0;  // an edge of F is never one of F'
      }
      if (w2) put(2, b2, ed[((h2 >> kLoBits) * kKeyInv) & kKeyMask]);
      if (h1 == kFree && h2 == kFree) continue;
      // a long chain shortens as all its vertices walk it (climb, sample.cu)
      for (int k = 0; h1 != kFree || h2 != kFree; k++) {
        const bool a = h1 != kFree, b = h2 != kFree;
        if (a) r1 = h1 & ((1u << kLoBits) - 1);
        if (b) r2 = h2 & ((1u << kLoBits) - 1);
        if (k >= 6) {
          if (a) r1 = Rv[r1] & 0xffff;
          if (b) r2 = Rv[r2] >> 16;
          Rv[x] = r1 | r2 << 16;
        }
        const uint32_t n1 = a ? H1[r1] : kFree, n2 = b ? H2[r2] : kFree;
        h1 = n1;
        h2 = n2;
      }
      Rv[x] = r1 | r2 << 16;
    }
    G.sync();
  }
}

// Certifies packed edges (a | b << 16) of a list in shared memory.
template <int NT>
__device__ void s_certify_packed(const Grp<NT>& G, const Smem& S, const uint32_t* e, int32_t n, int32_t V, int32_t* n1, int32_t* n2) {
  volatile int32_t* P2 = S.P2;
  for (int32_t t0 = 0; t0 < n; t0 += NT) {
    const int32_t i = t0 + G.tid;
    const bool valid = i < n;
    const uint32_t x = valid ? e[i] : 0;
    const int32_t a = (int32_t)(x & 0xffff), b = (int32_t)(x >> 16);
    const bool need = valid && a != b && P2[a] != P2[b];
    s_settle(S, need, a, b, n1, n2, V);
  }
}

// The reduced graph of the certificate in S (F1: the nt edges of F, packed; P2: every vertex's root in
// F'): its vertices are the F' components that an F edge leaves, its edges the F edges between them.
//
// Two ends of an F' edge are joined by F as well (F' takes only edges that F rejected), so the edge lies
// on a cycle, and with it each F' component lies in one 2-edge-connected component.  Contracting those
// changes no bridge and makes none: the bridges of F u F' are those of the reduced graph, whose edges
// all come from F.  In a dense graph one component holds nearly every vertex, and what is left is the
// sparse fringe (2,088 vertices in 8 dense clusters: 60 vertices).
//
// Leaves a spanning forest of the reduced graph in F1 (packed reduced ends; each edge's token, from the
// back of R3: orig_of), its other edges in F2 and the forest's union-find in P1; returns the number of
// reduced vertices, *nt2 and *nx2 the numbers of edges.  token(e): what stands for F1's edge e (its ends,
// packed, when F1 is the graph's own forest).
template <int VM>
__device__ __forceinline__ uint32_t& orig_of(const Smem& S, int32_t e) {
  return S.F2[VM - 1 - e];
}

template <int NT, int VM, class Token>
__device__ int32_t s_contract(const Grp<NT>& G, const Smem& S, int32_t V, int32_t nt, GroupShared& gs, int32_t* nt2,
                              int32_t* nx2, Token token) {
  const int lane = threadIdx.x & 31;  // groups are whole warps
  int32_t* id = S.head;               // R5
  uint32_t* kept = reinterpret_cast<uint32_t*>(S.next);  // R6
  for (int x = G.tid; x < V; x += NT) {
    id[x] = 0;
    S.P1[x] = x;
  }
  if (G.tid == 0) {
    gs.kept = 0;
    gs.verts = 0;
    gs.tree = 0;
    gs.rest = 0;
  }
  G.sync();
  for (int base = G.tid - lane; base < nt; base += NT) {
    const int e = base + lane;
    const uint32_t p = e < nt ? S.F1[e] : 0;
    const int32_t ra = S.P2[p & 0xffff], rb = S.P2[p >> 16];
    const bool keep = ra != rb;
    if (keep) {
      id[ra] = 1;
      id[rb] = 1;
    }
    const unsigned m = __ballot_sync(kFull, keep);
    if (m) {
      int32_t at = 0;
      if (lane == __ffs(m) - 1) at = atomicAdd(&gs.kept, __popc(m));
      at = __shfl_sync(kFull, at, __ffs(m) - 1) + __popc(m & lanemask_lt());
      if (keep) kept[at] = (uint32_t)e;
    }
  }
  G.sync();
  const int32_t nk = gs.kept;
  if (nk == 0) {
    *nt2 = *nx2 = 0;
    return 0;
  }
  for (int base = G.tid - lane; base < V; base += NT) {
    const int x = base + lane;
    const bool is = x < V && id[x] != 0;
    const unsigned m = __ballot_sync(kFull, is);
    if (m) {
      int32_t at = 0;
      if (lane == __ffs(m) - 1) at = atomicAdd(&gs.verts, __popc(m));
      at = __shfl_sync(kFull, at, __ffs(m) - 1) + __popc(m & lanemask_lt());
      if (is) id[x] = at;
    }
  }
  G.sync();
  // (the ends' numbers replace the edges' places in two steps: F1 is rewritten as the forest forms)
  uint32_t* ends = reinterpret_cast<uint32_t*>(S.succ);  // R7
  for (int i = G.tid; i < nk; i += NT) {
    const uint32_t e = kept[i], p = S.F1[e];
    ends[i] = (uint32_t)id[S.P2[p & 0xffff]] | (uint32_t)id[S.P2[p >> 16]] << 16;
    kept[i] = token((int32_t)e);
  }
  G.sync();
  for (int base = G.tid - lane; base < nk; base += NT) {
    const int i = base + lane;
    const bool live = i < nk;
    const uint32_t packed = live ? ends[i] : 0;
    const bool tree = live && s_link(S.P1, (int32_t)(packed & 0xffff), (int32_t)(packed >> 16));
    const unsigned m1 = __ballot_sync(kFull, tree), m2 = __ballot_sync(kFull, live && !tree);
    int32_t b1 = 0, b2 = 0;
    if (lane == 0) {
      if (m1) b1 = atomicAdd(&gs.tree, __popc(m1));
      if (m2) b2 = atomicAdd(&gs.rest, __popc(m2));
    }
    b1 = __shfl_sync(kFull, b1, 0);
    b2 = __shfl_sync(kFull, b2, 0);
    if (tree) {
      const int32_t at = b1 + __popc(m1 & lanemask_lt());
      S.F1[at] = packed;
      orig_of<VM>(S, at) = kept[i];
    } else if (live) {
      S.F2[b2 + __popc(m2 & lanemask_lt())] = packed;
    }
  }
  G.sync();
  *nt2 = gs.tree;
  *nx2 = gs.rest;
  return gs.verts;
}

// Bridges of the graph in S with V >= 1 vertices (F1: a spanning forest, P1 its union-find, nt edges;
// extra(e), e < nx: the further edges, packed); leaves the bridges' places in F1 in S.keys, in no order,
// and returns their number.
template <int NT, int VM, class Extra>
__device__ int32_t s_bridges(const Grp<NT>& G, const Smem& S, int32_t V, int32_t nt, int32_t nx, int32_t* red,
                             int32_t* red_b, int32_t* sh, Extra extra) {
  const int tid = G.tid;
  // roots (minimum vertex of each tree)
  for (int x = tid; x < V; x += NT) {
    int32_t r = x, p = S.P1[x];
    while (p != r) {
      r = p;
      p = S.P1[r];
    }
    S.root[x] = (uint16_t)r;  // P2 region: F' union-find no longer needed
    S.head[x] = -1;
  }
  G.sync();
  // arcs 2e (a -> b) and 2e + 1 (b -> a) of tree edge e = F1[e] = (a, b): each vertex's outgoing
  // arcs in a list (head, next) built by one atomic exchange per arc
  const int32_t narcs = 2 * nt;
  for (int e = tid; e < nt; e += NT) {
    const uint32_t p = S.F1[e];
    S.next[2 * e] = (uint16_t)atomicExch(S.head + (p & 0xffff), 2 * e);
    S.next[2 * e + 1] = (uint16_t)atomicExch(S.head + (p >> 16), 2 * e + 1);
  }
  G.sync();
  // Euler-tour successors, cut at each root: after arc i into y comes the arc that follows i's
  // twin (y's arc back) in y's list, wrapping to its first arc except at the root
  uint16_t* succ = S.succ;  // R7
  for (int i = tid; i < narcs; i += NT) {
    const uint32_t p = S.F1[i >> 1];
    const int32_t y = (int32_t)((i & 1) ? (p & 0xffff) : (p >> 16));
    uint16_t s = S.next[i ^ 1];
    if (s == kNone16 && S.root[y] != y) s = (uint16_t)S.head[y];
    succ[i] = s;
  }
  if (tid == 0) *sh = 0;
  G.sync();
  // List ranking (rank = arcs after the arc in its tour) by a ruling set: every kRuleGap-th arc
  // by index and the head of every tour (a root's first arc, which no arc points to) start a
  // sublist that ends before the next ruler; one lane walks each sublist, recording for each arc
  // its ruler and its place in the sublist; the rulers' own list is ranked by pointer jumping,
  // four hops per round; then every arc subtracts its place from its ruler's count.  Random
  // shared-memory loads bound this step, and this reads each arc about three times in all where
  // pointer jumping over every arc reads it four times a round.
  //   R0 (free now) and R6 (next, free now): per arc, its ruler and its place (u16 each)
  //   R9 (pre / sz / par, written later): two buffers of packed (next ruler | arcs << 16) words
  //   R1's cur half (free now): the first arc of each extra ruler (heads off the kRuleGap grid)
  // A forest with t trees has at most (2V - 2t) / kRuleGap + t + 1 <= 5V/8 + 1 rulers.
  {
    const int32_t nreg = (narcs + kRuleGap - 1) / kRuleGap;
    for (int x = tid; x < V; x += NT) {
      const int32_t h = S.head[x];
      if (S.root[x] == x && h >= 0 && h % kRuleGap != 0) S.cur[atomicAdd(sh, 1)] = (uint16_t)h;
    }
    G.sync();
    const int32_t nrul = nreg + *sh;
    uint16_t* oruler = reinterpret_cast<uint16_t*>(S.P1);  // R0
    uint16_t* oplace = S.next;                             // R6
    uint32_t* ra = reinterpret_cast<uint32_t*>(S.pre);  // R9: 3 VM / 4 words each
    uint32_t* rb = ra + 3 * VM / 4;
    for (int k = tid; k < nrul; k += NT) {
      uint32_t i = k < nreg ? (uint32_t)(k * kRuleGap) : S.cur[k - nreg];
      uint32_t place = 0, next = kNone16;
      for (int32_t step = 0; step < narcs; step++) {  // a tour is a path: a sublist has < narcs arcs
        oruler[i] = (uint16_t)k;
        oplace[i] = (uint16_t)place;
        place++;
        const uint32_t s = succ[i];
        if (s == kNone16) break;
        if (s % kRuleGap == 0) {
          next = s / kRuleGap;
          break;
        }
        i = s;
      }
      ra[k] = next | (place << 16);
    }
    G.sync();
    int rounds = 0;
    while ((1 << (2 * rounds)) < max(nrul, 1)) rounds++;
    for (int r = 0; r < rounds; r++) {
      for (int k = tid; k < nrul; k += NT) {
        const uint32_t w = ra[k];
        uint32_t nx = w & 0xffffu, acc = w >> 16;
#pragma unroll
        for (int h = 0; h < 3 && nx != kNone16; h++) {
          const uint32_t x = ra[nx];
          acc += x >> 16;
          nx = x & 0xffffu;
        }
        rb[k] = nx | (acc << 16);
      }
      G.sync();
      uint32_t* t = ra;
      ra = rb;
      rb = t;
    }
    // ra[k] >> 16: the arcs from ruler k's first arc to the end of its tour
    for (int i = tid; i < narcs; i += NT) S.rnk[i] = (uint16_t)((ra[oruler[i]] >> 16) - oplace[i] - 1);
    G.sync();
  }
  // per root: tour arcs (aoff) and tree vertices (vbase); P1 region is free now
  if (nt == V - 1) {
    // one spanning tree, whose root is vertex 0 (the minimum of its set): its tour takes every
    // arc and its vertices every preorder number, and no other entry is read
    if (tid == 0) {
      S.aoff[0] = 0;
      S.aoff[1] = (uint16_t)narcs;
      S.vbase[0] = 0;
    }
  } else {
    for (int x = tid; x <= V; x += NT) {
      uint16_t L = 0, nv = 0;
      if (x < V && S.root[x] == x) {
        L = S.head[x] >= 0 ? (uint16_t)(S.rnk[S.head[x]] + 1) : 0;
        nv = (uint16_t)(L / 2 + 1);
      }
      S.aoff[x] = L;
      S.vbase[x] = nv;
    }
    G.sync();
    block_scan16_pair(G, S.aoff, S.vbase, V + 1, red, red_b);
  }
  // tour positions; down arcs (dflag reuses succ, free after ranking)
  for (int i = tid; i <= narcs; i += NT) S.dflag[i] = 0;
  G.sync();
  for (int i = tid; i < narcs; i += NT) {
    const uint32_t pe = S.F1[i >> 1];
    const int32_t a = (int32_t)(pe & 0xffff), b = (int32_t)(pe >> 16);
    const int32_t x = (i & 1) ? b : a, y = (i & 1) ? a : b;  // arc i: x -> y
    const int32_t ri = S.rnk[i], rt = S.rnk[i ^ 1];
    // the tour of x's root r fills positions [aoff[r], aoff[r + 1]); arc i is ri arcs from its end
    const int32_t g = S.aoff[S.root[x] + 1] - 1 - ri;
    if (g < 0 || g >= narcs) continue;
    if (ri > rt) {
      S.dflag[g] = 1;
      S.par[y] = (uint16_t)(i >> 1);  // its tree edge
      S.pre[y] = (uint16_t)g;
      S.sz[y] = (uint16_t)((ri - rt + 1) / 2);
    }
  }
  G.sync();
  block_scan16(G, S.dflag, narcs, red);  // dscan in place
  // preorder numbers; lo / hi (dst and twin are free now)
  for (int x = tid; x < V; x += NT) {
    const int32_t r = S.root[x];
    int32_t p;
    if (r == x) {
      p = S.vbase[x];
      S.sz[x] = (uint16_t)((S.aoff[x + 1] - S.aoff[x]) / 2 + 1);
      S.par[x] = kNone16;
    } else {
      const int32_t g = S.pre[x], a0 = S.aoff[r];
      p = (g < narcs && a0 < narcs) ? S.vbase[r] + 1 + S.dflag[g] - S.dflag[a0] : 0;
    }
    const int32_t q = min(max(p, 0), V - 1);
    S.pre[x] = (uint16_t)q;
    S.rnk[q] = (uint16_t)x;  // the vertex at each preorder position (rnk is free now)
    S.lo[q] = q;
    S.hi[q] = q;
  }
  G.sync();
  for (int e = tid; e < nx; e += NT) {
    const uint32_t p = extra(e);
    const int32_t a = (int32_t)(p & 0xffff), b = (int32_t)(p >> 16);
    if (a == b) continue;
    const int32_t pa = S.pre[a], pb = S.pre[b];
    atomicMin(S.lo + pa, pb);
    atomicMin(S.lo + pb, pa);
    atomicMax(S.hi + pa, pb);
    atomicMax(S.hi + pb, pa);
  }
  G.sync();
  // per chunk of 32 preorder positions: the in-chunk prefix minima of lo and maxima of hi (u16, in
  // the dflag region, free now) and the chunk's minimum / maximum
  uint16_t* plo = S.dflag;
  uint16_t* phi = S.dflag + VM;
  int32_t* cmin = S.chunk;
  int32_t* cmax = cmin + VM / 32;
  const int nch = (V + 31) / 32;
  const int lane = tid & 31;
  for (int c = tid >> 5; c < nch; c += (NT / 32)) {  // warp-uniform
    const int i = c * 32 + lane;
    int32_t mn = i < V ? S.lo[i] : INT32_MAX, mx = i < V ? S.hi[i] : INT32_MIN;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t a = __shfl_up_sync(kFull, mn, o), b = __shfl_up_sync(kFull, mx, o);
      if (lane >= o) mn = min(mn, a), mx = max(mx, b);
    }
    if (i < V) {
      plo[i] = (uint16_t)mn;
      phi[i] = (uint16_t)mx;
    }
    if (lane == 31) {
      cmin[c] = mn;
      cmax[c] = mx;
    }
  }
  if (tid == 0) *sh = 0;
  G.sync();
  // superchunks of 32 chunks, a warp each: the extrema of windows of 2^j chunks (j < 6, cut at
  // the superchunk's end), the in-superchunk prefix and suffix extrema and each superchunk's
  // extrema (int32, in the P1 region, free now), so that any run of whole chunks is a few loads
  constexpr int NC = VM / 32;
  static_assert((16 * NC + 2 * (NC / 32 + 1)) * 4 <= Layout<VM>::R0, "the chunk tables fit the P1 region");
  int32_t* wcl = S.P1;           // [6][NC] window minima of lo
  int32_t* wch = wcl + 6 * NC;   // [6][NC] window maxima of hi
  int32_t* pcl = wch + 6 * NC;   // in-superchunk prefix
  int32_t* pch = pcl + NC;
  int32_t* scl = pch + NC;       // in-superchunk suffix
  int32_t* sch = scl + NC;
  int32_t* sml = sch + NC;       // [NC / 32 + 1] superchunk extrema
  int32_t* smh = sml + NC / 32 + 1;
  const int nsc = (nch + 31) / 32;
  if ((tid >> 5) < nsc) {  // warp-uniform
    const int w = tid >> 5, c = w * 32 + lane;
    const int32_t a0 = c < nch ? cmin[c] : INT32_MAX, b0 = c < nch ? cmax[c] : INT32_MIN;
    int32_t wa = a0, wb = b0;
#pragma unroll
    for (int j = 0; j < 6; j++) {
      if (c < nch) {
        wcl[j * NC + c] = wa;
        wch[j * NC + c] = wb;
      }
      if (j < 5) {
        const int o = 1 << j;
        const int32_t ta = __shfl_down_sync(kFull, wa, o), tb = __shfl_down_sync(kFull, wb, o);
        if (lane + o < 32) wa = min(wa, ta), wb = max(wb, tb);
      }
    }
    int32_t pa = a0, pb = b0, sa = a0, sb = b0;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t x1 = __shfl_up_sync(kFull, pa, o), x2 = __shfl_up_sync(kFull, pb, o);
      const int32_t y1 = __shfl_down_sync(kFull, sa, o), y2 = __shfl_down_sync(kFull, sb, o);
      if (lane >= o) pa = min(pa, x1), pb = max(pb, x2);
      if (lane + o < 32) sa = min(sa, y1), sb = max(sb, y2);
    }
    if (c < nch) {
      pcl[c] = pa;
      pch[c] = pb;
      scl[c] = sa;
      sch[c] = sb;
    }
    if (lane == 31) {
      sml[w] = pa;
      smh[w] = pb;
    }
  }
  G.sync();
  // test every tree edge (par(y), y), whose subtree holds the preorder positions [p, p + sz(y)),
  // p = pre(y): a warp takes a chunk of 32 positions, a lane one position.  The subtree's part in
  // the chunk, [p, e), is covered by two power-of-two windows, [p, p + 2^k) and [e - 2^k, e),
  // whose extrema the warp builds and exchanges by shuffles; past the chunk come the whole
  // chunks (two windows within a superchunk, else a suffix, a prefix and the superchunks between)
  // and the last chunk's prefix.
  const uint16_t* vtx = S.rnk;
  for (int c = tid >> 5; c < nch; c += (NT / 32)) {  // warp-uniform
    const int32_t p = c * 32 + lane;
    int32_t wa[6], wb[6];  // extrema of [p, p + 2^j), cut at the chunk's end
    wa[0] = p < V ? S.lo[p] : INT32_MAX;
    wb[0] = p < V ? S.hi[p] : INT32_MIN;
#pragma unroll
    for (int j = 1; j < 6; j++) {
      const int o = 1 << (j - 1);
      const int32_t a = __shfl_down_sync(kFull, wa[j - 1], o), b = __shfl_down_sync(kFull, wb[j - 1], o);
      wa[j] = lane + o < 32 ? min(wa[j - 1], a) : wa[j - 1];
      wb[j] = lane + o < 32 ? max(wb[j - 1], b) : wb[j - 1];
    }
    int32_t y = 0, py = kNone16, r = p;
    if (p < V) {
      y = min((int32_t)vtx[p], V - 1);
      py = S.par[y];
      r = min(V, p + max((int32_t)S.sz[y], 1));
    }
    const bool live = p < V && py != kNone16;
    const int32_t e = min(r, c * 32 + 32);
    const int32_t len = max(e - p, 1);  // lane + len <= 32
    const int k = 31 - __clz(len);
    int32_t mn = INT32_MAX, mx = INT32_MIN;
#pragma unroll
    for (int j = 0; j < 6; j++) {
      const int src = min(max(lane + len - (1 << j), 0), 31);
      const int32_t a = __shfl_sync(kFull, wa[j], src), b = __shfl_sync(kFull, wb[j], src);
      if (k == j) {
        mn = min(wa[j], a);
        mx = max(wb[j], b);
      }
    }
    // past the chunk: whole chunks [c + 1, cr), then chunk cr's prefix up to r - 1
    if (live && r > e) {
      const int32_t cl = c + 1, cr = (r - 1) >> 5;
      mn = min(mn, (int32_t)plo[r - 1]);
      mx = max(mx, (int32_t)phi[r - 1]);
      if (cl < cr) {
        const int32_t s0 = cl >> 5, s1 = (cr - 1) >> 5;
        if (s0 == s1) {
          const int j = 31 - __clz(cr - cl);
          const int32_t c2 = cr - (1 << j);
          mn = min(mn, min(wcl[j * NC + cl], wcl[j * NC + c2]));
          mx = max(mx, max(wch[j * NC + cl], wch[j * NC + c2]));
        } else {
          mn = min(mn, min(scl[cl], pcl[cr - 1]));
          mx = max(mx, max(sch[cl], pch[cr - 1]));
          for (int32_t q = s0 + 1; q < s1; q++) mn = min(mn, sml[q]), mx = max(mx, smh[q]);
        }
      }
    }
    if (live && mn >= p && mx < r) {
      const int32_t kk = atomicAdd(sh, 1);
      if (kk < V) S.keys[kk] = (uint32_t)py;
    }
  }
  G.sync();
  return min(*sh, max(V - 1, 0));
}

// Sorts the n bridges that s_bridges left in S.keys by their original ends and writes the pairs.
template <int NT, int VM>
__device__ void s_write_sorted(const Grp<NT>& G, const Smem& S, int32_t n, int32_t* out) {
  const int tid = G.tid;
  for (int i = tid; i < n; i += NT) {
    const uint32_t p = orig_of<VM>(S, (int32_t)S.keys[i]);
    const uint32_t a = p & 0xffff, b = p >> 16;
    S.keys[i] = min(a, b) << 12 | max(a, b);
  }
  G.sync();
  if (n <= NT) {
    // rank sort: keys are unique (a bridge has no parallel copy), every thread ranks one key
    // against all n with broadcast reads; one pass, no barrier
    if (tid < n) {
      const uint32_t mine = S.keys[tid];
      int32_t rank = 0;
      for (int j = 0; j < n; j++) rank += S.keys[j] < mine;
      out[2 * rank] = (int32_t)(mine >> 12);
      out[2 * rank + 1] = (int32_t)(mine & 0xfff);
    }
    G.sync();
    return;
  }
  int np = 1;
  while (np < n) np <<= 1;
  if (np > VM) {
    // more keys than the threads and a power of two above the key array's capacity: every thread
    // ranks several keys against all n (keys are unique)
    for (int i = tid; i < n; i += NT) {
      const uint32_t mine = S.keys[i];
      int32_t rank = 0;
      for (int j = 0; j < n; j++) rank += S.keys[j] < mine;
      out[2 * rank] = (int32_t)(mine >> 12);
      out[2 * rank + 1] = (int32_t)(mine & 0xfff);
    }
    G.sync();
    return;
  }
  // bitonic sort of n keys (padded to a power of two with ~0)
  for (int i = n + tid; i < np; i += NT) S.keys[i] = 0xffffffffu;
  G.sync();
  for (int k = 2; k <= np; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < np; i += NT) {
        const int l = i ^ j;
        if (l > i) {
          const uint32_t x = S.keys[i], y = S.keys[l];
          const bool up = (i & k) == 0;
          if ((x > y) == up) {
            S.keys[i] = y;
            S.keys[l] = x;
          }
        }
      }
      G.sync();
    }
  }
  for (int i = tid; i < n; i += NT) {
    out[2 * i] = (int32_t)(S.keys[i] >> 12);
    out[2 * i + 1] = (int32_t)(S.keys[i] & 0xfff);
  }
  G.sync();
}

// The bridges of the certificate in S (F1: nt edges; P2: F' roots, flat), sorted, to out; returns their
// number.
template <int NT, int VM>
__device__ int32_t s_certificate_bridges(const Grp<NT>& G, const Smem& S, int32_t V, int32_t nt, int32_t* out,
                                         GroupShared& gs) {
  int32_t nt2, nx2;
  const int32_t VH = s_contract<NT, VM>(G, S, V, nt, gs, &nt2, &nx2, [&](int32_t e) { return S.F1[e]; });
  if (VH == 0) return 0;
  const int32_t n = s_bridges<NT, VM>(G, S, VH, nt2, nx2, gs.red, gs.red_b, &gs.sh, [&](int32_t e) { return S.F2[e]; });
  s_write_sorted<NT, VM>(G, S, n, out);
  return n;
}


}  // namespace
}  // namespace bridges
