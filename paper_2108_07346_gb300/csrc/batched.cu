// batched.cu -- many small graphs in two persistent launches, and the one-block kernels of single
// small graphs.
//
// Certification (certify_kernel): four 256-thread groups per block take tasks from a queue with
// two ends (most edges first; one group per block starts with the fewest).  A task is a whole
// graph (V <= 4096) or one partition of its edge list (Sec. 3: the edges split into contiguous
// sets).  The group certifies the task's edges with two concurrent union-finds in SHARED memory
// (Alg. 2: F, then F' from the edges F rejects) and appends the winners to the task's slot in
// global memory, so it holds only the union-finds (8 bytes per vertex) and four graphs share an
// SM: while one runs its warm-up prefix edge by edge (latency bound), the others stream their
// edges.  A graph of up to 1,024 vertices (one task) is certified straight into the bridge
// stage's shared-memory layout and its bridge stage runs right there, beside the other groups'
// streams.
//
// Bridges (bridge_kernel), for the larger graphs: per graph, a group copies F and the roots of F' from
// the first task's slot, offers the other tasks' edges (several: the Sec. 3 merge with fan-in = the
// number of partitions) and runs the bridge stage.  The stage contracts the F' components first
// (s_contract: what is left of a dense graph is a small fringe); if cycles are left it is the same
// Euler-tour / preorder-range test as final.cu, on 16-bit arrays with barriers between phases (list
// ranking by a ruling set, subtree ranges from shuffle windows and chunk extrema); then a rank sort
// of the packed (a << 12 | b) keys (bitonic above the group's thread count).  A graph's fixed cost is its barriers, so graphs of
// up to 3,008 vertices run two per block: the block splits into 512-thread groups with their own
// half of shared memory and their own named barrier, so that one graph's barrier waits overlap
// with the other's work.  Nothing waits on another block, so there is no spin anywhere.
#include <algorithm>

#include "smem.cuh"

namespace bridges {

namespace {

constexpr int kAT = 256;               // threads of a certification group
constexpr int kAGroups = kT / kAT;     // certification groups per block
static_assert(kAT == kQuarterT, "a certification group runs the quarter-class bridge stages");
// a certification group's shared memory: the union-finds (P1, P2) of a graph of up to kVmax
// vertices, or the whole bridge-stage layout of a quarter-class graph
constexpr int kABytes = cmax(8 * kVmax, Layout<kQuarterVmax>::kBytes);
static_assert(kABytes % 16 == 0, "group regions stay 16-byte aligned");

// The certificate slot of task T (batch_slot_words).
__device__ __forceinline__ uint32_t* task_slot(const BatchArgs& A, const BatchTask& T) { return A.slots + T.slot; }

// Whether T's descriptor can be used (a malformed one is skipped, never used to index memory).
__device__ __forceinline__ bool task_ok(const BatchArgs& A, const BatchTask& T) {
  const int64_t stride = batch_slot_words(T.V);
  return T.V >= 0 && T.V <= kVmax && T.lo >= 0 && T.hi >= T.lo && T.g >= 0 && T.g < A.G && T.nparts >= 1 &&
         T.part >= 0 && T.part < T.nparts && T.count && (T.V <= 1 || T.out) && T.slot >= (int64_t)T.part * stride &&
         T.slot + (int64_t)(T.nparts - T.part) * stride <= A.slot_words;
}

// Certifies task T by group G of NT threads.  A quarter-class graph (one task, at most
// kQuarterVmax vertices) is certified into the bridge stage's layout in the group's shared memory
// and finished here; any other task keeps only its two union-finds in shared memory and appends
// its winners to its slot (the graph's first task also leaves the roots of its forests there).
template <int NT>
__device__ void certify_task(const BatchArgs& A, const BatchTask& T, char* smem, const Grp<NT>& G,
                             GroupShared& gs) {
  const int tid = G.tid;
  if (!task_ok(A, T)) {
    if (tid == 0 && T.g >= 0 && T.g < A.G) atomicExch(A.gerr + T.g, BRIDGES_EINTERNAL);
    return;
  }
  const int32_t V = T.V;
  if (T.cls == 2) {
    if (V > kQuarterVmax || T.nparts != 1) {  // not a quarter-class task: never run past the layout
      if (tid == 0) *T.count = BRIDGES_EINTERNAL;
      return;
    }
    // a quarter-class graph (one task, at most kQuarterVmax vertices): certified straight into the
    // bridge stage's shared-memory layout, then its bridge stage runs here, beside the other
    // groups' streams, instead of in bridge_kernel
    const Smem S = carve_smem<kQuarterVmax>(smem);
    for (int x = tid; x < V; x += NT) {
      S.P1[x] = x;
      S.P2[x] = x;
    }
    if (tid == 0) {
      gs.n1 = 0;
      gs.n2 = 0;
      gs.err = 0;
    }
    G.sync();
    s_certify_range<NT, kQuarterVmax>(G, S, T.u, T.v, T.lo, T.hi, T.warm, V, &gs.n1, &gs.n2, &gs.err);
    s_flatten(G, S.P2, V);
    const int32_t nt = min(gs.n1, V), err = gs.err;
    if (err) {
      if (tid == 0) *T.count = err;
      return;
    }
    const int32_t nb = s_certificate_bridges<NT, kQuarterVmax>(G, S, V, nt, T.out, gs);
    if (tid == 0) *T.count = nb;
    return;
  }
  uint32_t* slot = task_slot(A, T);
  Smem S{};
  S.P1 = reinterpret_cast<int32_t*>(smem);
  S.P2 = S.P1 + kVmax;
  S.F1 = slot + 2;      // global: winners are appended straight to the slot
  S.F2 = slot + 2 + V;
  for (int x = tid; x < V; x += NT) {
    S.P1[x] = x;
    S.P2[x] = x;
  }
  if (tid == 0) {
    gs.n1 = 0;
    gs.n2 = 0;
    gs.err = 0;
  }
  G.sync();
  s_certify_range<NT, kVmax>(G, S, T.u, T.v, T.lo, T.hi, T.warm, V, &gs.n1, &gs.n2, &gs.err);
  if (T.part == 0) {
    // the graph's first task: the roots of its F' trees (and, when more tasks follow, of its F
    // trees), so that the bridge stage starts from this task's union-finds as they stand and
    // offers only the other tasks' edges
    if (T.nparts > 1) s_flatten(G, S.P1, V);
    s_flatten(G, S.P2, V);
    uint16_t* roots2 = reinterpret_cast<uint16_t*>(slot + 2 + 2 * (int64_t)V);
    uint16_t* roots1 = reinterpret_cast<uint16_t*>(slot + 2 + 2 * (int64_t)V + (V + 1) / 2);
    for (int x = tid; x < V; x += NT) {
      roots2[x] = (uint16_t)S.P2[x];
      if (T.nparts > 1) roots1[x] = (uint16_t)S.P1[x];
    }
  }
  G.sync();
  if (tid == 0) {
    slot[0] = (uint32_t)min(gs.n1, V);
    slot[1] = (uint32_t)min(gs.n2, V);
    if (gs.err) atomicExch(A.gerr + T.g, gs.err);
  }
}

// Copies words [0, n) of src (global) to dst(i) (shared memory) with eight loads per thread in
// flight before their stores: a plain copy loop waits for one load per round.
template <int NT, class Dst>
__device__ __forceinline__ void copy_in(const uint32_t* __restrict__ src, int32_t n, int tid, Dst dst) {
  for (int32_t base = 0; base < n; base += 8 * NT) {
    uint32_t r[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int32_t i = base + k * NT + tid;
      r[k] = i < n ? __ldcg(src + i) : 0u;
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int32_t i = base + k * NT + tid;
      if (i < n) dst(i, r[k]);
    }
  }
}

// Bridges of the graph whose first task is T (later partitions are skipped): its slots' F and F'
// edges offered to fresh union-finds (one slot: the same two forests again; several: the Sec. 3
// merge), then the bridge stage, by a group of NT threads whose graphs have at most VM vertices.
template <int NT, int VM>
__device__ void bridge_task(const BatchArgs& A, const BatchTask& T, const Smem& S, const Grp<NT>& G, GroupShared& gs) {
  const int tid = G.tid;
  if (T.part != 0 || T.cls == 2) return;  // quarter-class graphs are finished by certify_kernel
  if (!task_ok(A, T) || T.V > VM) {
    if (tid == 0 && T.count) *T.count = BRIDGES_EINTERNAL;
    return;
  }
  const int32_t V = T.V;
  const int64_t stride = batch_slot_words(V);
  if (tid == 0) {
    gs.n1 = 0;
    gs.n2 = 0;
    gs.err = ld_relaxed(A.gerr + T.g);
  }
  // the first task's F as it stands, with the roots of its F' trees (and, when other tasks' edges
  // follow, of its F trees: P1 and P2 then hold each vertex's root -- offering its lists again to
  // fresh union-finds would rebuild exactly these forests).  The F' edges themselves are not needed:
  // each lies inside one vertex of the reduced graph.
  const uint32_t* sp = task_slot(A, T);
  const int32_t nf = min((int32_t)__ldcg(sp), V);
  const int32_t rw = (V + 1) / 2;  // words of a roots array (two 16-bit roots a word)
  copy_in<NT>(sp + 2, nf, tid, [&](int32_t i, uint32_t w) { S.F1[i] = w; });
  copy_in<NT>(sp + 2 + 2 * (int64_t)V, T.nparts > 1 ? 2 * rw : rw, tid, [&](int32_t j, uint32_t w) {
    int32_t* P = j < rw ? S.P2 : S.P1;
    const int32_t x = 2 * (j < rw ? j : j - rw);
    if (x < V) P[x] = min((int32_t)(w & 0xffffu), V - 1);
    if (x + 1 < V) P[x + 1] = min((int32_t)(w >> 16), V - 1);
  });
  if (tid == 0) {
    gs.n1 = nf;
    gs.n2 = 0;
  }
  G.sync();
  // the other tasks: the Sec. 3 merge -- each slot's F and F' edges offered to the union-finds.
  // Each slot is read with all of a thread's loads in flight and filtered on the way: an edge
  // whose ends already have the same F' parent is joined in both forests (F' components lie
  // inside F components, and sets only grow), so only the others are staged in shared memory
  // (the dst region, 2 VM words, free until the bridge stage) and offered, in any order (every
  // order leaves F a spanning forest of the offered edges and F' one of the rest).
  uint32_t* stage = reinterpret_cast<uint32_t*>(S.dst);
  volatile int32_t* P2v = S.P2;
  // two staging counters used in turn (red_b is free until the bridge stage): slot p counts in
  // cnt[p & 1], and cnt[(p + 1) & 1], last read in slot p - 1's pass, is reset after the barrier
  // that ends that pass
  int32_t* cnt = gs.red_b;
  if (tid == 0) {
    cnt[0] = 0;
    cnt[1] = 0;
  }
  for (int p = 1; p < T.nparts; p++) {
    const uint32_t* pp = sp + (int64_t)p * stride;
    const int32_t mf = min((int32_t)__ldcg(pp), V), mx = min((int32_t)__ldcg(pp + 1), V);
    G.sync();  // the previous slot's edges are settled: the stage is free
    if (tid == 0) cnt[(p + 1) & 1] = 0;
    copy_in<NT>(pp + 2, 2 * V, tid, [&](int32_t i, uint32_t w) {
      if (i < V ? i >= mf : i - V >= mx) return;
      const int32_t a = (int32_t)(w & 0xffff), b = (int32_t)(w >> 16);
      if (a < V && b < V && a != b && P2v[a] != P2v[b]) stage[atomicAdd(cnt + (p & 1), 1)] = w;
    });
    G.sync();
    s_certify_packed(G, S, stage, min(cnt[p & 1], 2 * V), V, &gs.n1, &gs.n2);
  }
  if (T.nparts > 1)
    s_flatten(G, S.P2, V);
  else
    G.sync();
  const int32_t nt = min(gs.n1, V);
  if (gs.err) {
    G.sync();  // every thread has read gs.err before the next task resets it
    if (tid == 0) *T.count = gs.err;
    return;
  }
  const int32_t nb = s_certificate_bridges<NT, VM>(G, S, V, nt, T.out, gs);
  if (tid == 0) *T.count = nb;
}

// Takes tasks first + 0, 1, ... from `queue` until `last` and runs their bridge stage on group G.
template <int NT, int VM>
__device__ void run_queue(const BatchArgs& A, char* smem, const Grp<NT>& G, GroupShared& gs, int32_t* queue,
                          int32_t first, int32_t last) {
  const Smem S = carve_smem<VM>(smem);
  while (true) {
    G.sync();  // every thread of the group is done with the previous task (and with gs.task)
    if (G.tid == 0) gs.task = first + atomicAdd(queue, 1);
    G.sync();
    const int32_t t = gs.task;
    if (t >= last) break;
    bridge_task<NT, VM>(A, A.tasks[t], S, G, gs);
  }
}

// Claims the next position of corder, or -1 when none is left.  One 64-bit word counts the claims
// at both ends (the front's in the low half, the back's in the high half), so one atomic add
// sees both: a front claim f succeeds while f + min(b, nback) < n, a back claim b while b < nback
// and f + b < n (task n - 1 - b).  No position is claimed twice, and none is missed: after a back
// claim fails, every later one fails too and its group claims from the front.
__device__ __noinline__ int32_t claim_task(unsigned long long* q, int32_t n, int32_t nback, bool& back) {
  if (back) {
    const unsigned long long old = atomicAdd(q, 1ull << 32);
    const int64_t f = (int64_t)(old & 0xffffffffull), b = (int64_t)(old >> 32);
    if (b < nback && f + b < n) return (int32_t)(n - 1 - b);
    back = false;
  }
  const unsigned long long old = atomicAdd(q, 1ull);
  const int64_t f = (int64_t)(old & 0xffffffffull), b = (int64_t)(old >> 32);
  return f + min(b, (int64_t)nback) < n ? (int32_t)f : -1;
}

// Certifies tasks on group G in corder: most edges first, or, for a back group, the fewest edges
// first while the last nback tasks last, then from the front.
template <int NT>
__device__ void certify_queue(const BatchArgs& A, char* smem, const Grp<NT>& G, GroupShared& gs, bool back,
                              int32_t ntasks) {
  unsigned long long* q = reinterpret_cast<unsigned long long*>(A.queue + 4);
  const int32_t nback = min(max(A.nback, 0), ntasks);
  while (true) {
    G.sync();
    if (G.tid == 0) gs.task = claim_task(q, ntasks, nback, back);
    G.sync();
    const int32_t t = gs.task;
    if (t < 0) break;
    certify_task<NT>(A, A.tasks[A.corder[t]], smem, G, gs);
  }
}

// Persistent certification: four 256-thread groups per block (named barriers 1-4), each with a
// quarter of the shared memory, take the tasks in corder (most edges first, so that the longest
// lists start early); one group's warm-up prefix (edge by edge, latency bound) overlaps the other
// groups' streams.  The last group of each block starts from the back of corder: the smallest
// graphs are almost all prefix, and taken last they would leave HBM idle at the end of the
// launch; taken beside the long streams they are hidden.  (Whole blocks for the long tasks were
// measured slower: a block alone on its SM has no other group's stream to hide its own prefix
// behind.)
__global__ void __launch_bounds__(kT, 1) certify_kernel(const BatchArgs* __restrict__ dA) {
  const BatchArgs A = *dA;
  extern __shared__ __align__(16) char smem_raw[];
  __shared__ GroupShared gs[kAGroups];
  const int32_t ntasks = *A.d_ntasks;
  const int k = (int)threadIdx.x / kAT;
  certify_queue<kAT>(A, smem_raw + k * kABytes, Grp<kAT>{(int)threadIdx.x % kAT, 1 + k}, gs[k],
                     k == kAGroups - 1, ntasks);
}

// Persistent bridge stages: whole-block tasks first (graphs above kHalfVmax vertices and
// partitioned graphs); then the block splits into two independent half-block groups, each with
// half the shared memory and its own named barrier, for graphs of up to kHalfVmax vertices.  A
// small graph's cost is mostly its barriers, and this overlaps two of them on one SM.  No barrier
// spans groups after the split.  (Quarter-class graphs were finished by certify_kernel.)
__global__ void __launch_bounds__(kT, 1) bridge_kernel(const BatchArgs* __restrict__ dA) {
  const BatchArgs A = *dA;
  extern __shared__ __align__(16) char smem_raw[];
  __shared__ GroupShared gs[3];  // [0] the block, then [1 + h] each half
  const int32_t ntasks = *A.d_ntasks;
  const int32_t nbig = min(max(A.nbig, 0), ntasks);
  const int32_t nmid = min(max(A.nmid, 0), ntasks - nbig);
  run_queue<kT, kVmax>(A, smem_raw, Grp<kT>{(int)threadIdx.x, 0}, gs[0], A.queue, 0, nbig);
  __syncthreads();  // the halves reuse the shared memory
  const int h = (int)threadIdx.x / kHalfT;
  char* half = smem_raw + h * kHalfBytes;
  const Grp<kHalfT> gh{(int)threadIdx.x % kHalfT, 1 + h};
  run_queue<kHalfT, kHalfVmax>(A, half, gh, gs[1 + h], A.queue + 1, nbig, nbig + nmid);
}

// ---- the plan of a batch ----
//
// Every graph's partitions, classes and slots, and the two orders of the tasks, by one block: the sums over
// the graphs as block scans, the orders as counting sorts by class and by edges (16 sizes to an octave, which
// is as fine as the orders need; tasks of one size come in any order).  Bound by its few passes over the
// graphs and their barriers.  The host took 90 us to plan 1,024 graphs (1,640 tasks), half of it the sorts,
// before the first kernel could start; this takes 22, and 13 KB go up instead of 150 (the call 597 -> 534 us).
constexpr int kPlanSizes = 1024;

// The size class of e edges, the largest first.
__device__ __forceinline__ int plan_size(int64_t e) {
  int b = (int)e;
  if (e >= 16) {
    const int lg = 63 - __clzll(e);
    b = ((lg - 3) << 4) | (int)((e >> (lg - 4)) & 15);
  }
  return kPlanSizes - 1 - b;
}

// Exclusive block scan (kT threads) of one value per thread; *total gets the sum.  red: kT / 32 words.
template <class T>
__device__ __forceinline__ T plan_scan(T v, T* red, T* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T incl = v;
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  __syncthreads();
  if (lane == 31) red[w] = incl;
  __syncthreads();
  T before = 0, all = 0;
  for (int k = 0; k < kT / 32; k++) {
    if (k < w) before += red[k];
    all += red[k];
  }
  *total = all;
  return before + incl - v;
}

__global__ void __launch_bounds__(kT, 1) plan_kernel(const char* plan, BatchArgs* dA) {
  __shared__ BatchPlanArgs H;
  __shared__ int32_t by_class[3 * kPlanSizes], by_size[kPlanSizes];
  __shared__ int64_t red[kT / 32];
  __shared__ int32_t red32[kT / 32];
  const int tid = threadIdx.x;
  if (tid == 0) H = *reinterpret_cast<const BatchPlanArgs*>(plan);
  for (int i = tid; i < 3 * kPlanSizes; i += kT) by_class[i] = 0;
  by_size[tid] = 0;
  static_assert(kPlanSizes == kT, "a thread per size");
  __syncthreads();
  const int64_t* const off = reinterpret_cast<const int64_t*>(plan + kPlanHeader);
  const int32_t* const Vs = reinterpret_cast<const int32_t*>(off + H.G + 1);
  const int32_t per = (H.G + kT - 1) / kT;
  const int32_t g0 = min(H.G, tid * per), g1 = min(H.G, g0 + per);
  // sizes, and the sums over this thread's graphs
  int64_t pairs = 0, words = 0;
  for (int32_t g = g0; g < g1; g++) {
    const int64_t lo = off[g], E = off[g + 1] - lo;
    const int32_t V = Vs[g];
    pairs += 2 * (int64_t)max(V - 1, 0);
    if (V > kVmax) continue;
    const int32_t np = batch_parts(E, H.split);
    words += np * batch_slot_words(V);
    const int cls = batch_min_class(V, np);
    for (int32_t p = 0; p < np; p++) {
      const int size = plan_size(E * (p + 1) / np - E * p / np);
      atomicAdd(by_class + cls * kPlanSizes + size, 1);
      atomicAdd(by_size + size, 1);
    }
  }
  int64_t all;
  int64_t out_at = plan_scan<int64_t>(pairs, red, &all);
  int64_t slot_at = plan_scan<int64_t>(words, red, &all);
  // the counts to first places
  {
    int32_t c[3], t = 0, n;
    for (int k = 0; k < 3; k++) {
      c[k] = by_class[3 * tid + k];
      t += c[k];
    }
    int32_t at = plan_scan<int32_t>(t, red32, &n);
    for (int k = 0; k < 3; k++) {
      by_class[3 * tid + k] = at;
      at += c[k];
    }
    const int32_t b = by_size[tid];
    const int32_t first = plan_scan<int32_t>(b, red32, &n);
    by_size[tid] = first;
    __syncthreads();
    if (tid == 0) {
      BatchArgs A = H.args;
      A.nbig = by_class[kPlanSizes];
      A.nmid = by_class[2 * kPlanSizes] - A.nbig;
      const int back = plan_size(H.back_edges) + 1;  // the sizes below it
      A.nback = back < kPlanSizes ? n - by_size[back] : 0;
      *dA = A;
      *const_cast<int32_t*>(A.d_ntasks) = n;
    }
    __syncthreads();  // the places are handed out below
  }
  for (int32_t g = g0; g < g1; g++) {
    const int64_t lo = off[g], E = off[g + 1] - lo;
    const int32_t V = Vs[g];
    if (V <= kVmax) {
      BatchTask T{};
      T.u = H.u;
      T.v = H.v;
      T.out = H.out ? H.out + out_at : nullptr;
      T.count = H.counts + g;
      T.g = g;
      T.V = V;
      T.nparts = batch_parts(E, H.split);
      T.cls = batch_min_class(V, T.nparts);
      T.warm = batch_warm(V);
      for (int32_t p = 0; p < T.nparts; p++) {
        T.lo = lo + E * p / T.nparts;
        T.hi = lo + E * (p + 1) / T.nparts;
        T.slot = slot_at;
        T.part = p;
        slot_at += batch_slot_words(V);
        const int size = plan_size(T.hi - T.lo);
        const int32_t at = atomicAdd(by_class + T.cls * kPlanSizes + size, 1);
        const_cast<BatchTask*>(H.args.tasks)[at] = T;
        const_cast<int32_t*>(H.args.corder)[atomicAdd(by_size + size, 1)] = at;
      }
    }
    out_at += 2 * (int64_t)max(V - 1, 0);
  }
}

// The bridge stage of one graph of 2..kVmax vertices on one block, in place of the grid-wide
// final stage when only the sorted bridges and their count are wanted: F (in global memory) is packed
// into the shared-memory layout, F's union-find copied, and the reduced graph's bridges found with
// block barriers only -- no grid barrier, no cooperative launch.
__global__ void __launch_bounds__(kT, 1) small_final_kernel(const SmallFinalArgs A) {
  extern __shared__ __align__(16) char smem_raw[];
  __shared__ GroupShared gs;
  const Smem S = carve_smem<kVmax>(smem_raw);
  const Grp<kT> G{(int)threadIdx.x, 0};
  const int tid = (int)threadIdx.x;
  const int32_t V = min(max(A.V, 0), kVmax);
  const int32_t nt = min(max(ld_relaxed(A.d_nt), 0), max(V - 1, 0));
  for (int x = tid; x < V; x += kT) {
    const int32_t p = __ldcg(A.P2 + x);
    S.P2[x] = (p >= 0 && p <= x) ? p : x;
  }
  int bad = 0;  // a certificate edge out of range (never expected: its edges passed the range test)
  for (int e = tid; e < nt; e += kT) {
    const int32_t a = __ldcg(A.tu + e), b = __ldcg(A.tv + e);
    bad |= (uint32_t)a >= (uint32_t)V || (uint32_t)b >= (uint32_t)V;
    S.F1[e] = (uint32_t)(a & 0xffff) | ((uint32_t)(b & 0xffff) << 16);
  }
  const bool any_bad = __syncthreads_or(bad) != 0;
  int32_t st = ld_relaxed(A.status);  // the same value for every thread: no stage writes it now
  if (st == 0 && any_bad) st = BRIDGES_EINTERNAL;
  if (st != 0) {
    if (tid == 0) *A.count = st;
    return;
  }
  s_flatten(G, S.P2, V);
  const int32_t nb = s_certificate_bridges<kT, kVmax>(G, S, V, nt, A.out, gs);
  if (tid == 0) *A.count = nb;
}

// The certificate of a sample of a graph of up to kVmax vertices on one block, in rounds in shared
// memory: what sample_kernel (sample.cu) leaves, without its grid barriers.
__global__ void __launch_bounds__(kT, 1) block_certify_kernel(const BlockCertArgs A) {
  extern __shared__ __align__(16) char smem_raw[];
  __shared__ int32_t n[2], any[2], err;
  const Grp<kT> G{(int)threadIdx.x, 0};
  const int tid = (int)threadIdx.x;
  const int32_t V = min(max(A.V, 0), kVmax);
  uint32_t* R = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* H1 = R + kVmax;
  uint32_t* H2 = H1 + kVmax;
  uint32_t* ed = H2 + kVmax;
  if (tid == 0) n[0] = n[1] = err = 0;
  __syncthreads();
  s_load_sample(G, ed, A.u, A.v, A.n, A.stride, A.groups, V, &err);
  s_certify_rounds(G, ed, A.groups << kSampleShift, V, R, H1, H2, n, n + 1, any, [&](int which, int32_t i, uint32_t p) {
    if (i < V) {
      (which == 1 ? A.b.f1u : A.b.f2u)[i] = (int32_t)(p & 0xffff);
      (which == 1 ? A.b.f1v : A.b.f2v)[i] = (int32_t)(p >> 16);
    }
  });
  for (int x = tid; x < V; x += kT) {
    A.b.P1[x] = (int32_t)(R[x] & 0xffff);
    A.b.P2[x] = (int32_t)(R[x] >> 16);
  }
  if (A.snap)
    for (int x = tid; x < A.b.Vpad; x += kT) A.b.lab[x] = x < V ? (uint16_t)(R[x] >> 16) : kNoLabel;
  if (tid == 0) {
    A.b.cnt[0] = n[0];
    A.b.cnt[1] = n[1];
    if (err) set_status(A.b.status, err);
  }
}

// A whole call on one block: a sample certified in rounds, the rest of the list streamed against its
// union-finds (live ones, in shared memory), the reduced graph's bridges sorted and written.
__global__ void __launch_bounds__(kT, 1) small_call_kernel(const SmallCallArgs A) {
  extern __shared__ __align__(16) char smem_raw[];
  __shared__ GroupShared gs;
  __shared__ int32_t any[2];
  const Smem S = carve_smem<kVmax>(smem_raw);
  const Grp<kT> G{(int)threadIdx.x, 0};
  const int tid = (int)threadIdx.x;
  const int32_t V = min(max(A.V, 0), kVmax);
  if (tid == 0) gs.n1 = gs.n2 = gs.err = 0;
  __syncthreads();
  // the sample in R5-R9 (free until the reduced graph), the roots in P1's region, the hooks in P2's
  // and in R3 (the F' edges are not needed: each lies inside one vertex of the reduced graph)
  uint32_t* ed = reinterpret_cast<uint32_t*>(S.head);
  uint32_t* R = reinterpret_cast<uint32_t*>(S.P1);
  s_load_sample(G, ed, A.u, A.v, A.E, A.stride, A.groups, V, &gs.err);
  s_certify_rounds(G, ed, A.groups << kSampleShift, V, R, reinterpret_cast<uint32_t*>(S.P2), S.F2, &gs.n1, &gs.n2, any,
                   [&](int which, int32_t i, uint32_t p) {
                     if (which == 1 && i < V) S.F1[i] = p;
                   });
  __syncthreads();
  for (int x = tid; x < V; x += kT) {
    const uint32_t r = R[x];
    S.P1[x] = (int32_t)(r & 0xffff);
    S.P2[x] = (int32_t)(r >> 16);
  }
  __syncthreads();
  if (A.stride > 1) {
    s_certify_vec<kT, kVmax>(G, S, A.u, A.v, 0, A.E, V, &gs.n1, &gs.n2, &gs.err, (uint32_t)A.stride);
    s_flatten(G, S.P2, V);
  }
  const int32_t nt = min(gs.n1, V), err = gs.err;
  const int32_t nb = err ? 0 : s_certificate_bridges<kT, kVmax>(G, S, V, nt, A.out, gs);
  if (tid == 0) *A.count = err ? err : nb;
}

}  // namespace

bool block_certify_launch(cudaStream_t s, const BlockCertArgs& a) {
  const size_t smem = 3 * sizeof(uint32_t) * kVmax + sizeof(uint32_t) * ((size_t)a.groups << kSampleShift);
  block_certify_kernel<<<1, kT, smem, s>>>(a);
  return cudaPeekAtLastError() == cudaSuccess;
}

bool small_call_launch(cudaStream_t s, const int32_t* u, const int32_t* v, int64_t E, int32_t V, int64_t* count,
                       int32_t* out) {
  // the sample: the whole list, or every stride-th group so that 4V + 2048 edges at most are taken
  using L = Layout<kVmax>;
  constexpr int64_t kRoom = (L::R5 + L::R6 + L::R7 + L::R8 + L::R9) / 4;
  static_assert(4 * kVmax + 2048 <= kRoom, "the sample fits beside the union-finds");
  const int64_t groups = ceil_div(E, 1 << kSampleShift);
  const int64_t most = std::min<int64_t>(kRoom, E <= 2 * (4 * (int64_t)V + 2048) ? E + 7 : 4 * (int64_t)V + 2048) >> kSampleShift;
  const int64_t stride = std::max<int64_t>(1, ceil_div(groups, std::max<int64_t>(most, 1)));
  const SmallCallArgs a{u, v, E, stride, (int32_t)ceil_div(groups, stride), V, count, out};
  small_call_kernel<<<1, kT, L::kBytes, s>>>(a);
  return cudaPeekAtLastError() == cudaSuccess;
}

bool batched_prepare() {
  const struct {
    const void* kernel;
    size_t bytes;
  } most[] = {{(const void*)small_final_kernel, Layout<kVmax>::kBytes},
              {(const void*)block_certify_kernel, sizeof(uint32_t) * (3 * kVmax + kBlockCertSlots)},
              {(const void*)small_call_kernel, Layout<kVmax>::kBytes},
              {(const void*)certify_kernel, kAGroups * kABytes},
              {(const void*)bridge_kernel, kSmem}};
  for (const auto& m : most)
    if (cudaFuncSetAttribute(m.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m.bytes) != cudaSuccess)
      return false;
  return true;
}

size_t batched_smem_bytes() { return (size_t)kSmem; }

bool small_final_launch(cudaStream_t s, const SmallFinalArgs& a) {
  if (a.V < 2 || a.V > kVmax) return false;
  small_final_kernel<<<1, kT, Layout<kVmax>::kBytes, s>>>(a);
  return cudaPeekAtLastError() == cudaSuccess;
}

bool batched_plan_launch(cudaStream_t s, const void* plan, BatchArgs* dev_args) {
  plan_kernel<<<1, kT, 0, s>>>(static_cast<const char*>(plan), dev_args);
  return cudaGetLastError() == cudaSuccess;
}

bool batched_launch(cudaStream_t s, const BatchArgs* dev_args, int num_sms) {
  certify_kernel<<<num_sms, kT, kAGroups * kABytes, s>>>(dev_args);
  bridge_kernel<<<num_sms, kT, kSmem, s>>>(dev_args);
  return cudaGetLastError() == cudaSuccess;
}

}  // namespace bridges
