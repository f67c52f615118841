// sample.cu -- the sampled certificate: F and F' of a sample of the list (Alg. 2 on one partition),
// the label snapshot of F', in one cooperative kernel.
//
// The forest pass streams the list against a snapshot of F' (certify.cu), so some edges have to be
// certified before it.  Linking them one by one through the concurrent union-finds is a chain of
// dependent, contended accesses per edge (2.5 M-edge list of 64 clusters, 473 k edges first: 208 us;
// a list of 2,000 edges: 30 us).  Here all edges of the sample advance together, in rounds of
// Boruvka's kind: no edge waits for another, and only the two grid barriers of a round are serial.
//
//   R: at the start of a round every vertex's root in F and in F', exactly (one word of both: the
//      rounds are bound by L2 sectors, and each gather is one).
//   H1, H2: for every vertex, the hook that took it under a smaller root: the key of the edge that
//      joined them (one number per edge, scrambled) and that root, in one word.
//   A  every live edge (a, b) reads its ends' roots.  F roots differ: it is a candidate for F and
//      offers its hook to the larger root (a minimum that returns nothing).  F roots equal, F'
//      roots differ: a candidate for F', the same on H2 -- its ends are joined by F edges, which F'
//      never holds, so F stays a spanning forest without it.  Both equal: the edge is redundant and
//      leaves.
//   B  an edge that finds its own word in the hook has won it, belongs to F or F', and leaves.
//   C  every vertex walks from its old root along the hooks to its new one.
//
// A root is hooked at most once and only under a smaller root, so the hooks are acyclic and every
// winner joins two different sets: F and F' are forests.  A round that finds no candidate has F
// spanning every edge of the sample and F' spanning every edge that is not in F: a certificate, as
// Alg. 2 builds one in list order.  Once few edges are live, they take the union-finds one by one
// (a round costs 5 us at the least, and the last few sets would take several).
//
// The scrambled keys make each root take a random smaller neighbour.  (Taking the smallest one needs
// a round less, but gives the smallest vertices all their edges in F and none in F', and a vertex
// outside F' sends its whole list down the stream's slow path: 1.29 -> 1.61 ms for the stream of a
// 1.07 G-edge list.)  A thread holds up to eight edges and lets the grid's first 2V in at once, the rest
// in rounds 4 and 5: the first ones join most of the sets, the rest meet few roots (594 k edges on
// 73,719 vertices: 103 us with all edges at once, 100 us so; 279 k on 37,147: 69 and 65 us).  Rounds with one barrier, edges and
// vertices climbing hooks of earlier rounds themselves, took longer: 82 us against 68 for 279 k edges
// on 37,147 vertices (a climb is a chain of L2 accesses, and a warp waits for its longest).
//
// The sample is every `stride`-th group of 8 edges (a 32-byte sector of each array), so a list sorted
// by its ends is sampled as evenly as a shuffled one: 8V edges in all give every vertex's run of
// edges two groups or so (128-byte lines would leave half of the runs out).  The stream reads the
// whole list and passes over the sampled edges among its misses (excluded, stream.cuh).  A list no
// longer than the sample is certified here whole.
#include <algorithm>

#include "batched.h"
#include "grid.cuh"
#include "forest.cuh"

namespace bridges {

namespace {

constexpr int kThreads = 1024;
constexpr int kMaxRounds = 24;  // rounds before the remaining edges take the union-finds one by one
// Live edges that take the union-finds one by one, and at most V / 4.  They gain a round or two where they are
// the last ones, but where their sets have yet to meet (sparse random lists around the densities at which F or
// F' forms its large set), every link chases the others' roots.  Over random lists of 0.55 V to 10 V edges on 5,000
// to 113,000 vertices and lists of clusters and R-MAT graphs, mean and worst against the best of eleven limits:
// 32,768 and V / 2 84.6 us and 4.0 times (60,000 vertices, 123,000 edges: 299 us instead of 74), 8,192 and V / 4
// 70.6 and 2.2 times, 4,096 and V / 4 70.3 and 1.27, 1,024 and V / 16 72.2 and 1.36.
constexpr unsigned kFewLive = 4096;
constexpr int kGroup = 8;       // edges per group of the sample (kSampleShift)
static_assert(kGroup == 1 << kSampleShift, "the stream's test of a sampled edge");

struct SampleArgs {
  const int32_t* u;
  const int32_t* v;
  int64_t n;       // edges [0, n) of the list are sampled from
  int64_t stride;  // every stride-th group of kGroup
  int64_t groups;  // groups sampled
  int32_t V;
  int32_t snap;  // whether the labels are wanted
  int32_t first;  // a thread's edges let in from the start
  unsigned bar_polls;  // polls a barrier waits before it gives up
  int32_t hold_polls;  // > 0: the last block sleeps this many ~100 ns polls before its first barrier
  int2* R;
  unsigned long long* H1;
  unsigned long long* H2;
  CertBufs b;
};

constexpr unsigned long long kNoHook = ~0ull;

// The hook that the edge in `slot` offers: its key (an odd multiple of the slot: unique) and the root
// above.
__device__ __forceinline__ unsigned long long hook_of(uint32_t slot, int32_t lo) {
  return (unsigned long long)(slot * 0x9e3779b1u) << 32 | (uint32_t)lo;
}

// Vertex x's new roots in F and F', its last ones r having hooks h1 and h2; the two walks run side by side (one
// after the other: 67.3 us for the sample of 2.5 M edges on 37,147 vertices, 65.0 so).
// A long chain (a path in list order) shortens as all its vertices walk it: past a few hooks the walk goes
// on from what R holds for the vertex reached and leaves its own progress in R[x], so jumps double.
__device__ __forceinline__ int2 climb(int2* R, const unsigned long long* H1, const unsigned long long* H2, int64_t x,
                                      int2 r, unsigned long long h1, unsigned long long h2) {
  int32_t* roots = reinterpret_cast<int32_t*>(R);
  for (int k = 0; h1 != kNoHook || h2 != kNoHook; k++) {
    const bool a = h1 != kNoHook, b = h2 != kNoHook;
    if (a) r.x = (int32_t)(uint32_t)h1;
    if (b) r.y = (int32_t)(uint32_t)h2;
    if (k >= 6) {
      const int32_t ra = a ? ld_relaxed(roots + 2 * (int64_t)r.x) : 0;
      const int32_t rb = b ? ld_relaxed(roots + 2 * (int64_t)r.y + 1) : 0;
      if (a) st_relaxed(roots + 2 * x, r.x = ra);
      if (b) st_relaxed(roots + 2 * x + 1, r.y = rb);
    }
    const unsigned long long n1 = a ? H1[r.x] : kNoHook, n2 = b ? H2[r.y] : kNoHook;
    h1 = n1;
    h2 = n2;
  }
  return r;
}

// The grid barrier of grid.cuh with a number to say: the blocks' *n add up, and every block learns the
// sum (*sum) from the word it polls, with no further access.  Bits 0-31 count arrivals, bits 32-63
// the numbers so far; `seen` is what they were before.  A barrier without numbers (n null) leaves
// `seen` alone, and one stands between any two with numbers: a fast block may add its number for the
// next barrier while a slow one still polls this one, but not for the one after.
// What a block keeps between its barriers is in shared memory (as arguments it cost the kernel registers).
struct SumBarrier {
  unsigned long long* word;
  int32_t* status;
  unsigned polls;  // before it gives up
  unsigned epoch, seen;
  unsigned sum;
  int ok;
};

static __device__ __noinline__ bool sum_barrier(SumBarrier* s, const unsigned* n) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned target = (s->epoch += 1) * gridDim.x;
    unsigned long long* const word = s->word;
    const unsigned long long add = (unsigned long long)(n ? *n : 0u) << 32 | 1ull;
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(add) : "memory");
    unsigned long long w = 0;
    const bool ok = bounded_poll(
        [&] {
          asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(word) : "memory");
          return (int)((unsigned)w - target) >= 0;
        },
        s->polls);
    if (!ok) set_status(s->status, BRIDGES_ETIMEDOUT_CODE);
    s->ok = ok;
    if (n) {
      s->sum = (unsigned)(w >> 32) - s->seen;
      s->seen = (unsigned)(w >> 32);
    }
  }
  __syncthreads();
  return s->ok != 0;
}

// K edges per thread.
template <int K>
__global__ void __launch_bounds__(kThreads, 1) sample_kernel(SampleArgs A) {
  __shared__ SumBarrier bar;
  __shared__ unsigned nlive, won[2];
  if (threadIdx.x == 0) {
    bar.word = reinterpret_cast<unsigned long long*>(A.b.ctl);
    bar.status = A.b.status;
    bar.polls = A.bar_polls;
    bar.epoch = bar.seen = nlive = won[0] = won[1] = 0;
  }
  hold_last_block(A.hold_polls);
  const Job J = job_of(A.b, A.V, 0);
  const int32_t V = A.V;
  int2* const R = A.R;
  unsigned long long* const H1 = A.H1;
  unsigned long long* const H2 = A.H2;
  unsigned* const ctl = A.b.ctl;
  const int lane = threadIdx.x & 31;
  const uint32_t slot0 = (uint32_t)gspread(), nslots = (uint32_t)gstride();
  unsigned left = 0;  // live edges of the grid
  auto barrier = [&](const unsigned* n) {
    if (!sum_barrier(&bar, n)) return false;
    if (n) left = bar.sum;
    return true;
  };

  for (int64_t x = gspread(); x < V; x += gstride()) {
    R[x] = make_int2((int32_t)x, (int32_t)x);
    H1[x] = kNoHook;
    H2[x] = kNoHook;
    if (A.snap && V > (int32_t)kNoLabel) A.b.tmp[x] = -1;
  }
  if (gtid() < 2) J.cnt[gtid()] = 0;
  // this thread's edges: one of each of groups q, q + Q, ... (Q groups to a pass of the grid)
  int32_t ea[K], eb[K];
  uint32_t live = 0;
#pragma unroll
  for (int k = 0; k < K; k++) {
    const int64_t q = (gspread() + k * gstride()) / kGroup;
    const int64_t e = q * A.stride * kGroup + lane % kGroup;
    ea[k] = eb[k] = 0;
    if (q < A.groups && e < A.n) {
      ea[k] = __ldg(A.u + e);
      eb[k] = __ldg(A.v + e);
      live |= 1u << k;
    }
  }
  bool bad = false;
#pragma unroll
  for (int k = 0; k < K; k++) {
    if ((live >> k & 1) && ((uint32_t)ea[k] >= (uint32_t)V || (uint32_t)eb[k] >= (uint32_t)V)) {
      bad = true;
      live &= ~(1u << k);
    }
    if (ea[k] == eb[k]) live &= ~(1u << k);
  }
  if (!barrier(nullptr)) return;
  if (bad) set_status(A.b.status, BRIDGES_ERANGE_CODE);

  uint32_t won1 = 0, won2 = 0;  // edges of F and of F'
  uint32_t joined = 0;          // edges whose ends F has joined: candidates for F' only
  for (int t = 1; t <= kMaxRounds; t++) {
    // A: candidates; hi / lo: the larger and the smaller root of the edge's pair
    int32_t hi[K], lo[K];
    const int admitted = t <= 3 ? A.first : (t == 4 ? 2 * A.first : K);
    const bool all_in = admitted >= K;
    const uint32_t in = (1u << min(admitted, K)) - 1;
    uint32_t offers = live & in;
    if (t == 1) {
#pragma unroll
      for (int k = 0; k < K; k++) {
        hi[k] = max(ea[k], eb[k]);
        lo[k] = min(ea[k], eb[k]);
      }
    } else {
      int2 ra[K], rb[K];
#pragma unroll
      for (int k = 0; k < K; k++) {
        if (!(offers >> k & 1)) continue;
        ra[k] = R[ea[k]];
        rb[k] = R[eb[k]];
      }
#pragma unroll
      for (int k = 0; k < K; k++) {
        if (!(offers >> k & 1)) continue;
        int32_t x = ra[k].x, y = rb[k].x;
        if (x == y) {
          joined |= 1u << k;
          x = ra[k].y;
          y = rb[k].y;
        }
        hi[k] = max(x, y);
        lo[k] = min(x, y);
        if (x == y) {
          live &= ~(1u << k);
          offers &= ~(1u << k);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < K; k++) {
      if (!(offers >> k & 1)) continue;
      unsigned long long* h = ((joined >> k & 1) ? H2 : H1) + hi[k];
      const unsigned long long mine = hook_of(slot0 + k * nslots, lo[k]);
      // an entry only falls, so a stale value (L1) that is already lower settles it
      if (*h > mine) atomicMin(h, mine);
    }
    const unsigned mine = __reduce_add_sync(kFull, (unsigned)__popc(live));
    if (lane == 0 && mine) atomicAdd(&nlive, mine);
    if (!barrier(&nlive)) return;
    if (left == 0) break;

    // B: winners
#pragma unroll
    for (int k = 0; k < K; k++) {
      if (!(offers >> k & 1)) continue;
      const bool f2 = joined >> k & 1;
      if ((f2 ? H2 : H1)[hi[k]] == hook_of(slot0 + k * nslots, lo[k])) {
        if (f2)
          won2 |= 1u << k;
        else
          won1 |= 1u << k;
        live &= ~(1u << k);
      }
    }
    if (threadIdx.x == 0) nlive = 0;

    // C: new roots, at the end also for the union-finds
    const bool last = all_in && left <= min(kFewLive, (unsigned)V / 4);
    for (int64_t x = gspread(); x < V; x += gstride()) {
      int2 r = R[x];
      const unsigned long long h1 = H1[r.x], h2 = H2[r.y];
      r = climb(R, H1, H2, x, r, h1, h2);
      R[x] = r;
      if (last || t == kMaxRounds) {
        J.P1[x] = r.x;
        J.P2[x] = r.y;
      }
    }
    if (!barrier(nullptr)) return;
    if (last) break;
  }
  if (left != 0) {  // what the rounds left links edge by edge
#pragma unroll
    for (int k = 0; k < K; k++) {
      const int r = (live >> k & 1) ? offer(J, ea[k], eb[k]) : 0;
      if (r == 1) won1 |= 1u << k;
      if (r == 2) won2 |= 1u << k;
    }
    if (!barrier(nullptr)) return;
  }
  for (int64_t x = gspread(); x < V; x += gstride()) {
    int2 r = R[x];
    if (left != 0) r = make_int2(uf_root_static(J.P1, (int32_t)x), uf_root_static(J.P2, (int32_t)x));
    J.P1[x] = r.x;
    J.P2[x] = r.y;
  }

  // the winners to the lists: places counted per warp, then per block, one global add per list and block
  {
    const int n1 = __popc(won1), n2 = __popc(won2);
    int incl = n1 | (n2 << 16);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    const int tot = __shfl_sync(kFull, incl, 31);
    unsigned w1 = 0, w2 = 0;
    if (lane == 0) {
      if (tot & 0xffff) w1 = atomicAdd(won + 0, tot & 0xffff);
      if (tot >> 16) w2 = atomicAdd(won + 1, tot >> 16);
    }
    __syncthreads();
    if (threadIdx.x < 2 && won[threadIdx.x])
      won[threadIdx.x] = (unsigned)atomicAdd(J.cnt + threadIdx.x, (int)won[threadIdx.x]);
    __syncthreads();
    int32_t at1 = (int32_t)(won[0] + __shfl_sync(kFull, w1, 0)) + (incl & 0xffff) - n1;
    int32_t at2 = (int32_t)(won[1] + __shfl_sync(kFull, w2, 0)) + (incl >> 16) - n2;
#pragma unroll
    for (int k = 0; k < K; k++) {
      const bool f2 = won2 >> k & 1;
      if (!f2 && !(won1 >> k & 1)) continue;
      const int32_t at = f2 ? at2++ : at1++;
      if (at < V) {
        (f2 ? J.f2u : J.f1u)[at] = ea[k];
        (f2 ? J.f2v : J.f1v)[at] = eb[k];
      } else {
        set_status(A.b.status, BRIDGES_EINTERNAL_CODE);
      }
    }
  }

  // the snapshot of F'
  const int64_t Vpad = A.b.Vpad;
  if (A.snap && V <= (int32_t)kNoLabel) {
    // 16 bits name every root: the label is the root (a vertex alone in its component shares it
    // with no other vertex)
    for (int64_t x = gspread(); x < Vpad; x += gstride()) A.b.lab[x] = x < V ? (uint16_t)J.P2[x] : kNoLabel;
  } else if (A.snap) {
    // number the components of two or more vertices: marked, numbered at their roots, then read
    for (int64_t x = gspread(); x < V; x += gstride()) {
      const int32_t r = J.P2[x];  // (written by this thread)
      if (r != x && A.b.tmp[r] == -1) A.b.tmp[r] = -2;
    }
    if (!barrier(nullptr)) return;
    for (int64_t base = gspread() & ~31LL; base < V; base += gstride()) {
      const int64_t x = base + lane;
      const bool is = x < V && A.b.tmp[x] == -2;
      const unsigned m = __ballot_sync(kFull, is);
      if (m) {
        int32_t at = 0;
        if (lane == __ffs(m) - 1) at = (int32_t)atomicAdd(ctl + kCtlLabels, (unsigned)__popc(m));
        at = __shfl_sync(kFull, at, __ffs(m) - 1) + __popc(m & lanemask_lt());
        if (is) A.b.tmp[x] = at;
      }
    }
    if (!barrier(nullptr)) return;
    for (int64_t x = gspread(); x < Vpad; x += gstride()) {
      const int32_t id = x < V ? A.b.tmp[J.P2[x]] : -1;
      A.b.lab[x] = (id >= 0 && id < (int32_t)kNoLabel) ? (uint16_t)id : kNoLabel;
    }
  }
}

template <int K>
void launch_sample(const Launch& L, SampleArgs& a, int blocks) {
  void* args[] = {&a};
  cudaLaunchCooperativeKernel((void*)sample_kernel<K>, dim3(blocks), dim3(kThreads), args, 0, L.stream);
  *L.launches += 1;
}

}  // namespace

int64_t sample_capacity(int num_sms) { return (int64_t)num_sms * kThreads * 8; }

void cert_sample(const Launch& L, const CertPlan& p, const CertBufs& b, const int32_t* u, const int32_t* v) {
  SampleArgs a{};
  a.u = u;
  a.v = v;
  a.n = p.stride > 0 ? p.E : std::min(p.warm, p.E);
  a.stride = std::max<int64_t>(p.stride, 1);
  a.groups = ceil_div(ceil_div(a.n, kGroup), a.stride);
  a.V = p.V;
  a.snap = p.cache;
  a.bar_polls = L.bar_polls > 0 ? L.bar_polls : kSpinCap;
  a.hold_polls = L.hold_polls;
  a.H1 = b.hook;
  a.H2 = b.hook + std::max(p.V, 1);
  a.R = b.roots;
  a.b = b;
  const int64_t slots = a.groups * kGroup;
  if (slots <= kBlockCertSlots && p.V <= kBatchVmax) {
    const BlockCertArgs ba{u, v, a.n, a.stride, (int32_t)a.groups, p.V, a.snap, b};
    block_certify_launch(L.stream, ba);  // a launch error is caught by the caller's error check
    *L.launches += 1;
    return;
  }
  // one thread per sampled edge and per vertex, at most one block per SM (fewer blocks make the
  // barriers cheaper) or per SM of the call's share, at most 8 edges a thread (the plan keeps the
  // sample below that for all SMs; a share takes more blocks if it must)
  const int64_t work = std::max<int64_t>({a.groups * kGroup, (int64_t)p.V, 1});
  const int64_t most = std::max<int64_t>(L.coop_blocks, ceil_div(a.groups, kThreads));
  const int blocks = (int)std::min<int64_t>({ceil_div(work, kThreads), most, (int64_t)L.num_sms});
  const int64_t per = ceil_div(a.groups * kGroup, (int64_t)blocks * kThreads);
  a.first = (int32_t)std::min<int64_t>(8, ceil_div(2 * (int64_t)std::max(p.V, 1), (int64_t)blocks * kThreads));
  if (per <= 1)
    launch_sample<1>(L, a, blocks);
  else if (per <= 2)
    launch_sample<2>(L, a, blocks);
  else if (per <= 4)
    launch_sample<4>(L, a, blocks);
  else
    launch_sample<8>(L, a, blocks);
}

}  // namespace bridges
