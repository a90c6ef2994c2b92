// k_pairs.cu -- persistence pairs of the critical cells.
//
// The critical cells left by the lower-star gradient are paired exactly as
// the plain reduction of the lexicographic filtration would pair them:
//   D0 (minimum, 1-saddle): integral lines from both ends of each critical
//     edge down to minima, then the elder rule over critical edges in
//     increasing order (union-find);
//   D2 (2-saddle, maximum): by duality, integral lines from the two
//     tetrahedra (or the outside) of each critical triangle up to maxima, then
//     the elder rule over critical triangles in decreasing order, the outside
//     of the domain being the oldest node;
//   D1 (1-saddle, 2-saddle): the column reduction of the critical triangles
//     left over, restricted to positive edges, where a gradient-paired edge is
//     eliminated with its triangle's reduced column.
// The elder rule is a column reduction with two entries per column: every item
// runs on its own thread, without rounds (k_uf_items), which gives exactly the
// sequential result whatever the schedule.
#include <atomic>
#include <utility>

#include "tsf_grid.cuh"
#include "tsf_group.cuh"
#include "tsf_kernels.cuh"
#include "tsf_star.cuh"

namespace tsf {

// Process-wide knobs (tsf_debug_set changes them for tests).  Of the union-
// find: two without effect any more, and a cap on an item's steps (0: none).
// The limit after which device waits and walks give up: polls at a grid
// barrier, steps of a union-find item.
std::atomic<int64_t> g_uf_grid_min{1 << 16};
std::atomic<int64_t> g_uf_handoff{1 << 13};
std::atomic<int64_t> g_uf_round_cap{0};
std::atomic<int64_t> g_barrier_limit{1 << 24};
// Of the D1 reduction: columns from which it starts with rounds over
// the whole GPU, active columns below which they go on on warps.  Measured on
// one diagram: 2.0 M columns (256^3) 2.50 ms with a handoff at 2^17, 2.87 ms
// at 2^12, 2.90 ms without rounds; 62 k columns (97 x 61 x 130) 0.41 ms with
// rounds down to 2^12, 0.33 ms without
std::atomic<int64_t> g_d1_grid_min{1 << 18};
std::atomic<int64_t> g_d1_handoff{1 << 17};
// schedule of the D1 Morse boundaries' phase A, as threads per column and its
// frontier + stage entries: 0 the default (8 for diagrams of at least 2^19
// critical triangles, 4 below 2^13, else 6), 1 and 2 one warp with 128 + 256 and
// 256 + 512, 3 one warp with 64 + 128 uncapped, 4 capped, 5 half a warp with 32 +
// 64, 6 a quarter of a warp with 16 + 32, 7 half a warp with 64 + 128, 8 a
// quarter of a warp with 32 + 64
std::atomic<int64_t> g_d1_phase_a{0};
// blocks per SM the lower-star gradient kernels are compiled for: 0 the
// default (six), 1 no register cap, 2 five
std::atomic<int64_t> g_gradient_blocks{0};
// entries of a column that a warp of the D1 reduction keeps in shared memory
// (at most 256; longer columns go to a block)
std::atomic<int64_t> g_chain_cap{256};
// D1 Morse boundaries: visits a thread chains per round along single-target
// updates (0: the default), rounds of the first phase before a column moves
// to a block (0: the default); both defaults depend on the diagram's size
std::atomic<int64_t> g_morse_chain{0};
std::atomic<int64_t> g_morse_rounds{0};
// D1 reduction: additions a column makes on a warp before it goes to a block
// (0: the default), groups of 1024 rows that a block keeps in shared memory
// (0: all that fit)
std::atomic<int64_t> g_chain_max{0};
std::atomic<int64_t> g_long_window{0};
// words of the D1 column pool per critical triangle in the first attempt (0:
// the default, see compute_diagram)
std::atomic<int64_t> g_pool_words{0};
// polls of a sort's look-back before it gives up (k_sort.cu; 0: the default,
// negative: none at all)
std::atomic<int64_t> g_sort_polls{0};
// device allocations of the fields until one is refused (0: none is)
std::atomic<int64_t> g_alloc_fail{0};

static std::atomic<int64_t>* knob(int what) {
  return what == 1   ? &g_uf_grid_min
         : what == 2 ? &g_uf_handoff
         : what == 3 ? &g_uf_round_cap
         : what == 4 ? &g_barrier_limit
         : what == 5 ? &g_d1_grid_min
         : what == 6 ? &g_d1_handoff
         : what == 7 ? &g_d1_phase_a
         : what == 8 ? &g_gradient_blocks
         : what == 9 ? &g_chain_cap
         : what == 10 ? &g_morse_chain
         : what == 11 ? &g_morse_rounds
         : what == 12 ? &g_chain_max
         : what == 13 ? &g_long_window
         : what == 14 ? &g_pool_words
         : what == 15 ? &g_sort_polls
         : what == 16 ? &g_alloc_fail
                     : nullptr;
}

int64_t get_knob(int what) {
  std::atomic<int64_t>* k = knob(what);
  return k ? k->load() : -1;
}

bool refuse_allocation() {
  int64_t k = g_alloc_fail.load(std::memory_order_relaxed);
  while (k > 0)
    if (g_alloc_fail.compare_exchange_weak(k, k - 1)) return k == 1;
  return false;
}

int64_t set_knob(int what, int64_t value) {
  std::atomic<int64_t>* k = knob(what);
  if (!k) return -1;
  return k->exchange(value);
}

// ---------------------------------------------------------------------------
// integral lines
// ---------------------------------------------------------------------------
// A descending line visits each vertex at most once (ranks decrease), so it
// has at most nv steps; an ascending dual line crosses into a higher vertex's
// star at most nv times and takes at most 24 steps inside one star.
__device__ __forceinline__ int32_t trace_down(uint32_t w, const uint8_t* __restrict__ vnext8,
                                              const uint32_t* __restrict__ cidx, const NbrDelta& nd, int64_t nv) {
  for (int64_t s = 0; s <= nv; ++s) {
    int k = vnext8[w];
    if (k == kVnextMin) return (int32_t)cidx[w];
    w = (uint32_t)((int32_t)w + nd.d[k]);
  }
  return -1;
}

// A union-find word: an item's priority and a node, or nothing.
constexpr unsigned long long kUfNone = ~0ull;

// Nothing has happened to any node or item yet.
__device__ __forceinline__ void uf_clear(int64_t t, int64_t threads, int nn, PairScratch S) {
  for (int64_t x = t; x < nn; x += threads) {
    S.rec[x] = kUfNone;
    S.skip[x] = kUfNone;
  }
}

__device__ __forceinline__ Rec ld_rec(const Rec* rec, uint32_t v) {
  const uint4* p = reinterpret_cast<const uint4*>(rec + v);
  uint4 a = __ldg(p), b = __ldg(p + 1);
  Rec r;
  r.w[0] = a.x; r.w[1] = a.y; r.w[2] = a.z; r.w[3] = a.w;
  r.w[4] = b.x; r.w[5] = b.y; r.w[6] = b.z; r.w[7] = b.w;
  return r;
}

// The integral lines of both stages run in one launch (the stages do not
// depend on each other and each is bound by its longest lines), D2's first as
// they take longer.  Both stages, one after the other with D2's walk holding a
// whole record in local memory / now: 0.266 / 0.097 ms for the 128^3 filament
// field, 0.59 / 0.23 for the 97 x 61 x 130 field, 3.69 / 1.26 for a 256^3 one.
struct TraceArgs {
  Dims d;
  NbrDelta nd;
  CritLists L;
  int n0, n1, n2, n3;
  const uint32_t* rank;
  const Rec* rec;
  const uint8_t* vnext8;
  const uint32_t* cidx;
  PairScratch S0, S2;
  PairOut P;
};
constexpr int kTraceT = 128;

// D0: one thread per endpoint of each critical edge; also clears the
// union-find.
__device__ void d0_trace(const TraceArgs& A, int64_t t, int64_t threads, uint32_t* status) {
  uf_clear(t, threads, A.n0, A.S0);
  if (t >= 2 * (int64_t)A.n1) return;
  uint32_t vn = A.L.c1_vn[t >> 1];
  uint32_t v = vn >> 4;
  if (!(t & 1)) {
    A.P.d0_min[t >> 1] = -1;
    A.P.d0_killed[t >> 1] = 0;
    A.P.d0mask[v] = 0u;
  }
  if (t & 1) v = (uint32_t)((int32_t)v + A.nd.d[vn & 15u]);
  int32_t a = trace_down(v, A.vnext8, A.cidx, A.nd, A.d.nv);
  if (a < 0) atomicOr(status, kErrTrace);
  A.S0.ends[t] = a < 0 ? 0 : a;
}

// Code of tetrahedron tau in a record in memory: the two words that hold its
// seven bits (rec_tet_code of the whole record, whose words a run-time index
// would send through local memory).
__device__ __forceinline__ int ld_tet_code(const Rec* __restrict__ rec, uint32_t w, int tau) {
  const int off = 56 + 7 * tau;
  const uint32_t* p = rec[w].w + (off >> 5);  // off <= 217: word 7 is the last
  return (int)(__funnelshift_r(__ldg(p), __ldg(p + 1), off & 31) & 127u);
}

// Ascending integral line in the dual: from tetrahedron (w, tau) follow the
// record codes to a maximum (its index) or to the outside (returns n3).
// Bound: one dependent L2 or memory access per star crossed, the steps inside
// a star hit L1.
__device__ int32_t trace_up(uint32_t w, int tau, const Rec* __restrict__ rec, const uint32_t* __restrict__ cidx,
                            const int32_t* nd, int n3, const UpStep* up, int64_t nv) {
  for (int64_t s = 0; s <= 25 * nv; ++s) {
    const int code = ld_tet_code(rec, w, tau);
    if (code < 24) {
      tau = code;
      continue;
    }
    if (code >= 96) return code == kCodeMax ? (int32_t)cidx[w] : code == kCodeOut ? n3 : -1;
    const UpStep u = up[code - 24];
    tau = u.tau;
    w = (uint32_t)((int32_t)w + nd[u.c]);
  }
  return -1;
}

// D2: one thread per (critical triangle, side): the ascending dual line from
// the tetrahedron on that side to a maximum or the outside.  Also clears the
// union-find.
__device__ void d2_trace(const TraceArgs& A, int64_t tt, int64_t threads, const int32_t* snd, const UpStep* sup,
                         uint32_t* status) {
  const Dims& d = A.d;
  const int n3 = A.n3;
  const Rec* __restrict__ rec = A.rec;
  const uint32_t* __restrict__ cidx = A.cidx;
  uf_clear(tt, threads, n3 + 1, A.S2);
  if (tt >= 2 * (int64_t)A.n2) return;
  int i = (int)(tt >> 1), k = (int)(tt & 1);
  if (!k) A.P.d2_max[i] = -1;
  const Geo& G = c_geo;
  uint32_t ve = A.L.c2_ve[i];
  uint32_t v = ve >> 6;
  int e = (int)(ve & 63u);
  int a = G.edge[e][0], b = G.edge[e][1];
  int x, y, z;
  vxyz(d, v, x, y, z);
  int t = G.edge_tri[e][k];
  int j = 0;
  while (G.tri[t][j] == a || G.tri[t][j] == b) ++j;
  int c = G.tri[t][j];
  int nx, ny, nz;
  int32_t res;
  if (!nbr_xyz(d, x, y, z, c, nx, ny, nz)) {
    res = n3;
  } else {
    uint32_t wc = vid(d, nx, ny, nz);
    if (__ldg(A.rank + wc) < __ldg(A.rank + v)) {
      res = trace_up(v, t, rec, cidx, snd, n3, sup, d.nv);
    } else {
      int i0 = nbr_index(G, -G.off[c][0], -G.off[c][1], -G.off[c][2]);
      int i1 = nbr_index(G, G.off[a][0] - G.off[c][0], G.off[a][1] - G.off[c][1], G.off[a][2] - G.off[c][2]);
      int i2 = nbr_index(G, G.off[b][0] - G.off[c][0], G.off[b][1] - G.off[c][1], G.off[b][2] - G.off[c][2]);
      int tau = (i0 >= 0 && i1 >= 0 && i2 >= 0) ? G.tri_of3[i0][i1][i2] : -1;
      res = tau < 0 ? -1 : trace_up(wc, tau, rec, cidx, snd, n3, sup, d.nv);
    }
  }
  if (res < 0) {
    atomicOr(status, kErrTrace);
    res = n3;
  }
  A.S2.ends[tt] = res;
}

__global__ void __launch_bounds__(kTraceT) k_traces(const __grid_constant__ TraceArgs A, unsigned blocks2,
                                                    uint32_t* status) {
  __shared__ UpStep sup[72];
  __shared__ int32_t snd[14];
  if (blockIdx.x < blocks2) {
    if (threadIdx.x < 14) snd[threadIdx.x] = A.nd.d[threadIdx.x];
    if (threadIdx.x < 72) sup[threadIdx.x] = c_up.s[threadIdx.x];
    __syncthreads();
    d2_trace(A, (int64_t)blockIdx.x * kTraceT + threadIdx.x, (int64_t)blocks2 * kTraceT, snd, sup, status);
  } else {
    d0_trace(A, (int64_t)(blockIdx.x - blocks2) * kTraceT + threadIdx.x,
             (int64_t)(gridDim.x - blocks2) * kTraceT, status);
  }
}

// ---------------------------------------------------------------------------
// Elder-rule union-find
// ---------------------------------------------------------------------------
// An item (critical edge, or triangle in decreasing order) with the components
// a and b of its ends is a column {a, b}: its low is the younger one, and the
// elder rule is the reduction by additions of earlier columns.  Each node's
// record holds the smallest priority that has it as its low, with the other
// entry of that column, in one 64-bit word, so that a single atomicMin both
// claims the low and returns the column to go on with: the claimant's own plus
// an earlier owner's, or the later owner's that it displaced plus its own.
// Nobody waits, and any schedule ends with the same lows.
//
// Before claiming, a thread replaces its entries by their records while these
// are earlier (also additions of earlier columns).  Such walks follow the merge
// tree, which may be deep, so each halves its path: skip[x] = (p, y) says that
// {x, y} is a sum of columns of priority at most p, which later items may use
// instead of two records; a stale word stays true.
// Bound: dependent L2 round trips along the deepest walk.  Rounds of
// reservations (one block, or the whole GPU behind barriers) took 0.34 ms for
// stage D0 of the 97 x 61 x 130 field and 1.42 ms for a 256^3 one, now 0.14
// and 0.75 ms (traces included, each stage on its own).
__device__ __forceinline__ unsigned long long uf_word(int pr, int node) {
  return ((unsigned long long)(uint32_t)pr << 32) | (uint32_t)node;
}

// The best word of node x that an item of priority pr may use, or kUfNone.
__device__ __forceinline__ unsigned long long uf_step(const PairScratch& S, int x, int pr) {
  const unsigned long long s = __ldcg(S.skip + x), r = __ldcg(S.rec + x);
  if ((uint32_t)(s >> 32) < (uint32_t)pr) return s;
  return (uint32_t)(r >> 32) < (uint32_t)pr ? r : kUfNone;
}

__device__ __forceinline__ int uf_walk(const PairScratch& S, int x, int pr, int nn) {
  for (int hop = 0; hop <= nn; ++hop) {  // every hop goes to an older node
    const unsigned long long s = uf_step(S, x, pr);
    if (s == kUfNone) return x;
    const int y = (int)(uint32_t)s;
    const unsigned long long t = uf_step(S, y, pr);
    if (t == kUfNone) return y;
    const uint32_t p = max((uint32_t)(s >> 32), (uint32_t)(t >> 32));
    __stcg(S.skip + x, uf_word((int)p, (int)(uint32_t)t));
    x = (int)(uint32_t)t;
  }
  return x;
}

// n items (priority i, or n-1-i for D2), nn nodes.  Younger node = larger
// index (D0) or smaller index (D2).  No blocks and no nodes: nothing to do.
struct UfSide {
  int n, nn;
  unsigned blocks;  // of k_uf_items
  PairScratch S;
  int32_t* kill;
};

// Both stages in one launch, D2's blocks first.
__global__ void __launch_bounds__(256) k_uf_items(const __grid_constant__ UfSide U2, const __grid_constant__ UfSide U0,
                                                  int limit, uint32_t* status) {
  const bool two = blockIdx.x < U2.blocks;
  const UfSide& U = two ? U2 : U0;
  const PairScratch S = U.S;
  const int n = U.n, nn = U.nn;
  const int threads = U.blocks * 256;
  for (int t = (blockIdx.x - (two ? 0u : U2.blocks)) * 256 + threadIdx.x; t < n; t += threads) {  // in priority order
    const int i = two ? n - 1 - t : t;
    int pr = t, a = S.ends[2 * i], b = S.ends[2 * i + 1];
    for (int step = 0;; ++step) {
      if (step >= limit) {
        atomicOr(status, kErrRounds);
        return;
      }
      a = uf_walk(S, a, pr, nn);
      b = uf_walk(S, b, pr, nn);
      if (a == b) break;  // closes a cycle
      const int young = two ? min(a, b) : max(a, b), old = a + b - young;
      const unsigned long long was = atomicMin(S.rec + young, uf_word(pr, old));
      if (was == kUfNone) break;
      const int wp = (int)(was >> 32);
      a = (int)(uint32_t)was;
      b = old;
      if (wp > pr) pr = wp;  // go on with the displaced item
    }
  }
}

// kill[i] = node killed by item i; for D0 also the marks of killed edges.
__global__ void __launch_bounds__(256) k_uf_kills(const __grid_constant__ UfSide U2, const __grid_constant__ UfSide U0,
                                                  CritLists L, PairOut P) {
  const unsigned blocks2 = (unsigned)(U2.nn + 255) / 256;
  const bool two = blockIdx.x < blocks2;
  const UfSide& U = two ? U2 : U0;
  const int x = (blockIdx.x - (two ? 0u : blocks2)) * 256 + threadIdx.x;
  if (x >= U.nn) return;
  const unsigned long long r = U.S.rec[x];
  if (r == kUfNone) return;
  const int pr = (int)(r >> 32), i = two ? U.n - 1 - pr : pr;
  U.kill[i] = x;
  if (!two) {
    P.d0_killed[i] = 1;
    const uint32_t vn = L.c1_vn[i];
    atomicOr(&P.d0mask[vn >> 4], 1u << (vn & 15u));
  }
}

// Threads in flight: enough to hide the round trips, few enough that the items
// run nearly in priority order (an item far ahead claims lows that earlier
// items take back).  Stages D0 and D2, each on its own with its traces, of the 97 x 61 x 130 field (8e4 items):
// 0.29 and 0.44 ms with 2^12 threads, 0.14 and 0.37 with 2^14, 0.19 and 0.45
// with 2^16; of a 256^3 field (2.6e6 items): 1.58 and 3.75 ms with 2^14, 0.75
// and 2.95 with 2^16, 0.76 and 3.02 with all.
static int uf_blocks(int n) { return (std::min(n, std::max(1 << 14, n / 32)) + 255) / 256; }

static int uf_limit() {
  int64_t limit = std::min<int64_t>(std::max<int64_t>(g_barrier_limit.load(), 1), 1 << 30);
  const int64_t cap = g_uf_round_cap.load();
  return (int)(cap > 0 ? std::min(limit, cap) : limit);
}

void launch_traces(const Dims& d, const NbrDelta& nd, const CritLists& L, int n0, int n1, int n2, int n3,
                   const uint32_t* rank, const Rec* rec, const uint8_t* vnext8, const uint32_t* cidx, PairScratch& S0,
                   PairScratch& S2, PairOut& P, uint32_t* status, cudaStream_t st) {
  const TraceArgs A{d, nd, L, n0, n1, n2, n3, rank, rec, vnext8, cidx, S0, S2, P};
  const unsigned b2 = (unsigned)((2 * (int64_t)n2 + kTraceT - 1) / kTraceT);
  const unsigned b0 = (unsigned)((2 * (int64_t)n1 + kTraceT - 1) / kTraceT);
  if (b0 + b2 == 0) return;
  k_traces<<<b2 + b0, kTraceT, 0, st>>>(A, b2, status); note_launch();
}

void launch_union_find(const CritLists& L, int n0, int n1, int n2, int n3, PairScratch& S0, PairScratch& S2,
                       PairOut& P, uint32_t* status, cudaStream_t st) {
  if (n1 == 0 && n2 == 0) return;
  const UfSide U2{n2, n2 ? n3 + 1 : 0, (unsigned)uf_blocks(n2), S2, P.d2_max};
  const UfSide U0{n1, n1 ? n0 : 0, (unsigned)uf_blocks(n1), S0, P.d0_min};
  k_uf_items<<<U2.blocks + U0.blocks, 256, 0, st>>>(U2, U0, uf_limit(), status); note_launch();
  k_uf_kills<<<(U2.nn + 255) / 256 + (U0.nn + 255) / 256, 256, 0, st>>>(U2, U0, L, P); note_launch();
}

// ---------------------------------------------------------------------------
// D1: column reduction of the critical triangles not paired in D2
// ---------------------------------------------------------------------------
struct D1Ctx {
  Dims d;
  NbrDelta nd;
  const uint32_t* rank;
  const uint32_t* order;
  const Rec* rec;
  const D1Tab* tab;
  const uint32_t* c1base;
  CritLists L;
  const uint8_t* d0_killed;
  const uint32_t* d0mask;
  int chain;  // visits one thread makes per round along single-target updates
};

__device__ __forceinline__ int nbr_of_pair(const Dims& d, uint32_t hi, uint32_t lo) {
  int hx, hy, hz, lx, ly, lz;
  vxyz(d, hi, hx, hy, hz);
  vxyz(d, lo, lx, ly, lz);
  return nbr_index(lx - hx, ly - hy, lz - hz);
}
__device__ __forceinline__ int nbr_of_pair(const Dims& d, uint32_t hi, uint32_t lo, const Geo& G) {
  int hx, hy, hz, lx, ly, lz;
  vxyz(d, hi, hx, hy, hz);
  vxyz(d, lo, lx, ly, lz);
  return nbr_index(G, lx - hx, ly - hy, lz - hz);
}

__device__ int crit_edge_index(const D1Ctx& c, uint32_t hi, const Rec& r, int k) {
  int cnt = __popc(rec_crit_edges(r));
  uint32_t base = c.c1base[hi];
  for (int j = 0; j < cnt; ++j)
    if ((int)(c.L.c1_vn[base + j] & 15u) == k) return (int)(base + j);
  return -1;
}

// 0: negative edge (not a row of the D1 matrix), 1: positive and critical,
// 2: positive and paired with a triangle in its lower star.
__device__ int edge_status(const D1Ctx& c, uint32_t p, uint32_t q, unsigned long long& key, int& ci) {
  uint32_t rp = c.rank[p], rq = c.rank[q];
  uint32_t hi = rp > rq ? p : q, lo = rp > rq ? q : p;
  key = ((unsigned long long)max(rp, rq) << 32) | min(rp, rq);
  int k = nbr_of_pair(c.d, hi, lo);
  Rec r = ld_rec(c.rec, hi);
  if (rec_vnext(r) == k) return 0;
  if ((rec_crit_edges(r) >> k) & 1u) {
    ci = crit_edge_index(c, hi, r, k);
    if (ci < 0) return 0;
    return c.d0_killed[ci] ? 0 : 1;
  }
  return 2;
}

struct Heap {
  unsigned long long* h;
  uint32_t off, cap, size;
};

__device__ bool heap_push(D1Work& W, Heap& H, unsigned long long key, uint32_t* status) {
  if (H.size == H.cap) {
    uint32_t ncap = H.cap * 2;
    uint32_t noff = atomicAdd(W.pool_head, ncap);
    if ((unsigned long long)noff + ncap > W.pool_cap) {
      atomicOr(status, kErrPool);
      return false;
    }
    unsigned long long* nh = W.pool + noff;
    for (uint32_t i = 0; i < H.size; ++i) nh[i] = H.h[i];
    H.h = nh;
    H.off = noff;
    H.cap = ncap;
  }
  uint32_t i = H.size++;
  H.h[i] = key;
  while (i > 0) {
    uint32_t p = (i - 1) >> 1;
    if (H.h[p] >= H.h[i]) break;
    unsigned long long t = H.h[p];
    H.h[p] = H.h[i];
    H.h[i] = t;
    i = p;
  }
  return true;
}

__device__ unsigned long long heap_pop(Heap& H) {
  unsigned long long top = H.h[0];
  unsigned long long last = H.h[--H.size];
  uint32_t i = 0;
  while (true) {
    uint32_t l = 2 * i + 1;
    if (l >= H.size) break;
    uint32_t r = l + 1;
    uint32_t m = (r < H.size && H.h[r] > H.h[l]) ? r : l;
    if (H.h[m] <= last) break;
    H.h[i] = H.h[m];
    i = m;
  }
  if (H.size > 0) H.h[i] = last;
  return top;
}

// largest entry present an odd number of times (Z/2), 0 if the column is empty
__device__ unsigned long long heap_low(Heap& H) {
  while (H.size > 0) {
    unsigned long long top = heap_pop(H);
    int c = 1;
    while (H.size > 0 && H.h[0] == top) {
      heap_pop(H);
      ++c;
    }
    if (c & 1) return top;
  }
  return 0ull;
}

__device__ __forceinline__ Heap heap_of(D1Work& W, int j) {
  Heap H;
  H.off = W.hoff[j];
  H.cap = W.hcap[j];
  H.size = W.hsize[j];
  H.h = W.pool + H.off;
  return H;
}
__device__ __forceinline__ void heap_store(D1Work& W, int j, const Heap& H) {
  W.hoff[j] = H.off;
  W.hcap[j] = H.cap;
  W.hsize[j] = H.size;
}

__device__ void push_if_positive(const D1Ctx& c, D1Work& W, Heap& H, uint32_t p, uint32_t q, uint32_t* status) {
  unsigned long long key;
  int ci;
  if (edge_status(c, p, q, key, ci) != 0) heap_push(W, H, key, status);
}

__global__ void k_d1_select(int n2, const int32_t* __restrict__ d2_max, uint32_t* __restrict__ flag) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n2) flag[i] = d2_max[i] < 0 ? 1u : 0u;
}
// Every column starts with kOut0 words of the pool of its own, from j kOut0 on.
constexpr uint32_t kOut0 = 64;
__device__ __forceinline__ uint32_t d1_reserved(int ncols) {
  return (uint32_t)min((unsigned long long)kOut0 * (unsigned)ncols, 1ull << 31);
}

__global__ void k_d1_gather(int n2, const uint32_t* __restrict__ flag, const uint32_t* __restrict__ pos,
                            int32_t* __restrict__ cols, int32_t* __restrict__ d1_edge, int32_t* __restrict__ ncols,
                            uint32_t* __restrict__ pool_head) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n2) {
    d1_edge[i] = -1;
    if (flag[i]) cols[pos[i]] = i;
    if (i == n2 - 1) {
      *ncols = (int32_t)(pos[i] + flag[i]);
      *pool_head = d1_reserved(*ncols);
    }
  }
}

// The same by one block, for up to kSelectOne triangles (four launches less:
// 22 us before on 2e3 triangles).
constexpr int kSelectT = 1024, kSelectOne = 8 * kSelectT;
__global__ void __launch_bounds__(kSelectT) k_d1_select_one(int n2, const int32_t* __restrict__ d2_max,
                                                            int32_t* __restrict__ cols, int32_t* __restrict__ d1_edge,
                                                            int32_t* __restrict__ ncols,
                                                            uint32_t* __restrict__ pool_head) {
  __shared__ int wsum[kSelectT / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (n2 + kSelectT - 1) / kSelectT;
  const int i0 = min(tid * per, n2), i1 = min(i0 + per, n2);
  uint32_t keep = 0;
  for (int i = i0; i < i1; ++i) {
    d1_edge[i] = -1;
    if (d2_max[i] < 0) keep |= 1u << (i - i0);
  }
  const int c = __popc(keep);
  int inc = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    const int x = wsum[lane];
    int xi = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, xi, o);
      if (lane >= o) xi += y;
    }
    wsum[lane] = xi - x;
    if (lane == 31) {
      *ncols = xi;
      *pool_head = d1_reserved(xi);
    }
  }
  __syncthreads();
  int at = wsum[w] + inc - c;
  for (; keep; keep &= keep - 1) cols[at++] = i0 + __ffs((int)keep) - 1;
}

// Growable array in the pool (a column's heap or its Morse boundary).
struct Vec {
  unsigned long long* h;
  uint32_t off, cap, size;
};

__device__ bool vec_alloc(D1Work& W, Vec& v, uint32_t cap, uint32_t* status) {
  uint32_t off = atomicAdd(W.pool_head, cap);
  if ((unsigned long long)off + cap > W.pool_cap) {
    atomicOr(status, kErrPool);
    return false;
  }
  v.off = off;
  v.cap = cap;
  v.size = 0;
  v.h = W.pool + off;
  return true;
}

__device__ bool vec_push(D1Work& W, Vec& v, unsigned long long x, uint32_t* status) {
  if (v.size == v.cap) {
    Vec n;
    if (!vec_alloc(W, n, v.cap * 2, status)) return false;
    for (uint32_t i = 0; i < v.size; ++i) n.h[i] = v.h[i];
    n.size = v.size;
    v = n;
  }
  v.h[v.size++] = x;
  return true;
}

__device__ __forceinline__ Heap as_heap(const Vec& v) {
  Heap H;
  H.h = v.h;
  H.off = v.off;
  H.cap = v.cap;
  H.size = v.size;
  return H;
}

constexpr int kD1StepLimit = 1 << 24;

// Phase 1: Morse boundary of each candidate triangle t: its boundary (positive
// edges) with every gradient-paired edge eliminated by its triangle's reduced
// column, largest first, one lower star at a time.  Output: the critical
// edges left (C1 indices), in decreasing lexicographic order.
__global__ void k_d1_morse(D1Ctx c, D1Work W, uint32_t* status) {
  const int ncols = W.flags[1];
  __shared__ Geo sg;
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  const bool mine = j < ncols && W.redo[j] != 0;
  if (!__syncthreads_or(mine)) return;  // almost always: nothing outgrew its buffers
  geo_to_shared(sg);
  if (!mine) return;
  W.hsize[j] = 0;
  W.hoff[j] = 0;
  Vec hv, out;
  if (!vec_alloc(W, hv, 32, status) || !vec_alloc(W, out, 8, status)) return;
  Heap H = as_heap(hv);
  uint32_t ve = c.L.c2_ve[W.cols[j]];
  uint32_t v0 = ve >> 6;
  int e0 = (int)(ve & 63u);
  uint32_t a0 = (uint32_t)((int32_t)v0 + c.nd.d[c_geo.edge[e0][0]]);
  uint32_t b0 = (uint32_t)((int32_t)v0 + c.nd.d[c_geo.edge[e0][1]]);
  push_if_positive(c, W, H, v0, a0, status);
  push_if_positive(c, W, H, v0, b0, status);
  push_if_positive(c, W, H, a0, b0, status);
  int nblocks = 0;
  for (int step = 0;; ++step) {
    if (step >= kD1StepLimit) {
      atomicOr(status, kErrRounds);
      return;
    }
    unsigned long long top = heap_low(H);
    if (top == 0) break;
    uint32_t rv = (uint32_t)(top >> 32);
    uint32_t v = c.order[rv];
    // every entry of v's lower star, with its parity, by neighbour index
    uint32_t m = 1u << nbr_of_pair(c.d, v, c.order[(uint32_t)(top & 0xFFFFFFFFull)]);
    while (H.size > 0 && (uint32_t)(H.h[0] >> 32) == rv) {
      unsigned long long e = heap_pop(H);
      m ^= 1u << nbr_of_pair(c.d, v, c.order[(uint32_t)(e & 0xFFFFFFFFull)]);
    }
    if (!m) continue;
    ++nblocks;
    Rec r = ld_rec(c.rec, v);
    uint32_t crit = rec_crit_edges(r);
    Star s;
    star_load(s, c.d, v, c.rank);
    int8_t y_of[14];
    uint64_t path_of[14];
    star_chains(s, y_of, path_of, sg);
    for (int p = s.nl - 1; p >= 1; --p) {
      int x = s.by_pos[p];
      if (!((m >> x) & 1u)) continue;
      m &= ~(1u << x);
      if ((crit >> x) & 1u) {
        int ci = crit_edge_index(c, v, r, x);
        if (ci >= 0 && !c.d0_killed[ci]) vec_push(W, out, (unsigned long long)ci, status);
        continue;
      }
      int y = y_of[x];
      if (y < 0) {
        atomicOr(status, kErrInconsistent);
        return;
      }
      if (y != s.by_pos[0]) m ^= 1u << y;  // w*y stays in this lower star (w*y negative if y is the lowest)
      for (uint64_t pm = path_of[x]; pm; pm &= pm - 1) {
        int le = __ffsll((long long)pm) - 1;
        uint32_t pa = (uint32_t)((int32_t)v + c.nd.d[c_geo.edge[le][0]]);
        uint32_t pb = (uint32_t)((int32_t)v + c.nd.d[c_geo.edge[le][1]]);
        push_if_positive(c, W, H, pa, pb, status);
      }
    }
  }
  W.hoff[j] = out.off;
  W.hsize[j] = out.size;
  atomicAdd(&W.stats[0], (unsigned long long)nblocks);
  atomicMax(&W.stats[1], (unsigned long long)nblocks);
}

// ---------------------------------------------------------------------------
// Phase 1, one group of threads per column.  The pending entries of a column
// are lower stars with a parity mask over their 14 edge directions.  All of
// a column's updates come from its own group, so they live in the group's
// shared memory: the frontier, sorted by descending key = value_key << 32 |
// vertex (the rank order), one entry per star.  Each round the group takes
// the GS highest entries, one per thread; every visit appends its updates of
// target stars to a stage; the stage is sorted, merged into the rest of the
// frontier and equal keys are combined (xor of masks, zero masks dropped).
// The projection is linear, so a star that receives entries after it was
// processed simply comes back, and the order only decides how often.
// ---------------------------------------------------------------------------
// Frontier entries are FEnt: key = value_key << 32 | vertex (0 never occurs,
// NaN is rejected), payload = the pending parity mask.  Entries saved in the
// pool (8-byte aligned) are two 64-bit words.
__device__ __forceinline__ void fent_save(unsigned long long* p, const FEnt& e) {
  p[0] = e.key;
  p[1] = e.mask;
}
__device__ __forceinline__ FEnt fent_restore(const unsigned long long* p) {
  FEnt e;
  e.key = p[0];
  e.mask = (uint32_t)p[1];
  e.pad = 0u;
  return e;
}

__device__ __forceinline__ unsigned long long star_key(uint32_t vkey, uint32_t v) {
  return ((unsigned long long)vkey << 32) | v;
}

// Link edge (a, b) left by a visit goes to the lower star of whichever
// endpoint ranks higher, as the direction towards the other one.  le: a, b,
// direction a -> b, direction b -> a, four bits each; at[x][0] / at[x][1]: the
// edges that have x as their a / their b.  Copied to shared
// memory: the index differs from lane to lane (constant memory would
// serialise), and read from global memory they did not stay in L1 (21 % hits).
struct D1Links {
  unsigned long long at[14][2];
  uint16_t le[36];
};
constexpr D1Links make_links() {
  D1Links t{};
  for (int e = 0; e < 36; ++e) {
    const int a = geo_edge(e, 0), b = geo_edge(e, 1);
    t.le[e] = (uint16_t)(a | b << 4 | geo_dir(a, b) << 8 | geo_dir(b, a) << 12);
    t.at[a][0] |= 1ull << e;
    t.at[b][1] |= 1ull << e;
  }
  return t;
}
__device__ const D1Links g_links = make_links();

// One lower-star visit: apply the closures of the star's pending edges
// (linear over Z/2), keep the positive critical edges left as (v << 4 | x),
// and append the link edges left to the stage as updates of the target
// stars.  One dependent global access: the star's table row, of which only
// the closures asked for are read.  The loops run over the bits that are set:
// a visit has little more than one pending edge and 1.1 targets on average.
// With `chain` set, a visit whose link edges all go to one target star hands
// that update back in *next instead of staging it, and the caller visits it at
// once (a star reached again later by another part of its mask is simply
// visited again: the projection is linear).
// Unrolling all 14 closures and 36 link edges at compile time needed the whole
// row in registers (64 are what 32 warps per SM leave: it spilled) and issued a
// fifth more instructions; the loops are worth it only where the groups of a
// warp share them (tsf_group.cuh): Morse boundaries of a 256^3 field 13.0 ms
// unrolled, 25.5 with loops and a barrier per group, 10.9 in lockstep.
template <int SCAP>
__device__ __forceinline__ bool d1_visit(const D1Ctx& c, FEnt fe, const int32_t* snd, const D1Links& links,
                                         FEnt* stage, int* s_ntot, int* s_flag, unsigned long long* myouts, int& myout,
                                         int& updates, bool chain, FEnt* next, uint32_t* status) {
  const uint32_t v = (uint32_t)fe.key;
  if ((int64_t)v >= c.d.nv) {  // never for a valid entry: report and let the column be recomputed
    atomicOr(status, kErrInconsistent);
    atomicOr(s_flag, 1);
    return false;
  }
  const uint32_t* row = reinterpret_cast<const uint32_t*>(c.tab + v);
  const uint4 q89 = __ldg(reinterpret_cast<const uint4*>(row + 16));
  uint4 nk[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) nk[k] = __ldg(reinterpret_cast<const uint4*>(row + 20) + k);
  const uint64_t ends = (uint64_t)q89.y << 32 | q89.x, above = (uint64_t)q89.w << 32 | q89.z;
  uint64_t path = fe.pad ? 1ull << (fe.pad - 1) : 0ull;  // a column's first entry brings a link edge
  uint32_t em = 0;
  for (uint32_t mm = fe.mask & 0x3FFFu; mm; mm &= mm - 1) {
    const int x = __ffs((int)mm) - 1, off = 36 * x;  // off <= 468: words 14 and 15 of the closures' 16
    const uint32_t* p = row + (off >> 5);
    path ^= ((uint64_t)__ldg(p + 1) << 32 | __ldg(p)) >> (off & 31);  // 36 bits from a multiple of 4 <= 28
    em ^= 1u << ((uint32_t)(ends >> (4 * x)) & 15u);
  }
  path &= (1ull << 36) - 1;
  em &= 0x3FFFu;
  if (em) {
    em &= ~__ldg(c.d0mask + v);  // negative critical edges are not rows
    if (em) {  // their indices are looked up at the column's end: bring them to L2
      asm volatile("prefetch.global.L2 [%0];" ::"l"(c.rec + v));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(c.c1base + v));
    }
    for (; em; em &= em - 1) myouts[myout++] = ((unsigned long long)v << 4) | (unsigned)(__ffs((int)em) - 1);
  }
  while (path) {
    const int e0 = __ffsll((long long)path) - 1;
    const uint32_t l0 = (uint32_t)links.le[e0];
    const int hn = (int)((above >> e0) & 1ull ? l0 & 15u : (l0 >> 4) & 15u);
    // all of them that go to the same star
    uint64_t same = path & ((above & links.at[hn][0]) | (~above & links.at[hn][1]));
    path ^= same;
    uint32_t mask = 0;
    for (; same; same &= same - 1) {
      const int e = __ffsll((long long)same) - 1;
      const uint32_t l = (uint32_t)links.le[e];
      mask |= 1u << ((above >> e) & 1ull ? (l >> 8) & 15u : l >> 12);
    }
    const uint32_t hv = (uint32_t)((int32_t)v + snd[hn]);
    FEnt t;
    t.mask = mask;
    t.pad = 0;
    ++updates;
    const uint4 k4 = hn < 8 ? (hn < 4 ? nk[0] : nk[1]) : (hn < 12 ? nk[2] : nk[3]);
    t.key = star_key(hn & 2 ? (hn & 1 ? k4.w : k4.z) : (hn & 1 ? k4.y : k4.x), hv);
    if (chain && !path) {  // the only one
      *next = t;
      return true;
    }
    chain = false;
    const int off = atomicAdd(s_ntot, 1);
    if (off >= SCAP) {
      atomicOr(s_flag, 1);
      return false;
    }
    stage[off] = t;
    // the star is likely visited in a later round: bring its row to L2
    const char* trow = reinterpret_cast<const char*>(c.tab + hv);
    asm volatile("prefetch.global.L2 [%0];" ::"l"(trow));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(trow + 128));
  }
  return false;
}

// Sorts a stage of n <= SCAP entries (a[] holds SCAP entries, a power of
// two): in registers for up to two entries per thread (the usual case),
// else in shared memory (compact code: the unrolled networks for more
// entries per thread only crowd the instruction cache).
template <int GS, int SCAP>
__device__ void group_sort_stage(FEnt* a, int n) {
  static_assert(SCAP % GS == 0 && (SCAP & (SCAP - 1)) == 0, "a stage is a power of two");
  const int most = gmax<GS>(n);
  if (most <= GS) group_sort_reg<GS, 1>(a, n);
  else if (most <= 2 * GS && SCAP >= 2 * GS) group_sort_reg<GS, (SCAP >= 2 * GS ? 2 : 1)>(a, n);
  else group_sort_smem<GS>(a, n);
}

// New frontier from the untaken rest (front[nb..nf), descending) and the
// stage (ntot updates, any order): sort the stage, merge, combine equal keys.
// Returns the new frontier size.  All threads of the group call it.
template <int GS, int SCAP>
__device__ int group_combine(FEnt* front, int nb, int nf, FEnt* other, FEnt* stage, int ntot, int* scan_sm) {
  const int tid = gtid<GS>();
  int rest = nf - nb;
  group_sort_stage<GS, SCAP>(stage, ntot);
  int total = rest + ntot;
  for (int k = tid; k < total; k += GS) {  // merge path
    int lo = max(0, k - ntot), hi = min(k, rest);
    while (lo < hi) {
      int mid = (lo + hi) >> 1;
      if (front[nb + mid].key >= stage[k - mid - 1].key) lo = mid + 1;
      else hi = mid;
    }
    int i = lo, jb = k - lo;
    other[k] = (i < rest && (jb >= ntot || front[nb + i].key >= stage[jb].key)) ? front[nb + i] : stage[jb];
  }
  gsync<GS>();
  int kept = 0;
  const int most = gmax<GS>(total);
  for (int base = 0; base < most; base += GS) {
    int k = base + tid;
    int keep = 0;
    FEnt e;
    e.key = 0ull;
    e.mask = 0u;
    e.pad = 0u;
    if (k < total) {
      e = other[k];
      if (k == 0 || other[k - 1].key != e.key) {
        for (int q = k + 1; q < total && other[q].key == e.key; ++q) e.mask ^= other[q].mask;
        keep = e.mask != 0u;
      }
    }
    int t;
    int off = gscan<GS>(keep, t, scan_sm);
    if (keep) front[kept + off] = e;
    kept += t;
  }
  gsync<GS>();
  return kept;
}

// Visits one thread makes per round along a chain of single-target updates;
// room for the critical edges those visits keep; rounds of phase A before a
// column moves to a block.  The defaults depend on the diagram's size.  A
// large diagram (at least kLargeD1 critical triangles) keeps enough columns
// in flight in phase A to fill the GPU, so its columns stay there (no
// chaining, 128 rounds); a smaller one gains from moving its long columns to
// 128-thread blocks early (chains of 2, 16 rounds).  Stage time, ms: 256^3
// field (2.6e6 triangles) at 16 / 24 / 64 / 128 rounds 11.3 / 8.5 / 8.1 / 8.1;
// 97 x 61 x 130 field (8e4) at 6 / 12 / 16 / 24: 0.68 / 0.48 / 0.50 / 0.52.
constexpr int kOutCap = 28;
constexpr int kLargeD1 = 1 << 19;
constexpr int kChainLarge = 1, kRoundsLarge = 128;  // defaults of knobs 10 and 11, large diagrams
constexpr int kChainSmall = 2, kRoundsSmall = 16;   // ... small diagrams
// Below 2^13 critical triangles every column can have its block at once, so
// phase A only keeps the columns that end after a few rounds.  At 2 / 4 / 6 /
// 12 rounds: 32^3 field (3e3 triangles) 0.136 / 0.105 / 0.107 / 0.138 ms, 128^3
// filament field (2e3) 0.38 / 0.39 / 0.43 / 0.44, but 1.8 / 1.2 / 0.68 / 0.48
// for the 97 x 61 x 130 field.
constexpr int kTinyD1 = 1 << 13, kRoundsTiny = 4;

// One column.  Phase A (max_rounds > 0): every column, one group of GS threads
// (a quarter, a half or a whole warp); a column still open after max_rounds,
// or whose frontier outgrows the group's buffers, saves its entries and is
// listed for phase B (NT = GS = 128, one block per listed column).  Groups of
// a warp run in lockstep: a group without a column (not `live`), or whose
// column has stopped, goes along without changing anything.  Groups of one
// block otherwise share only the tables.
template <int NT, int FCAP, int SCAP, int GS>
__device__ __forceinline__ void d1_column(const D1Ctx& c, D1Work& W, int j, bool live, bool phase_b, int max_rounds,
                                          FEnt* front, const int32_t* snd, const D1Links& links, int* scan_sm,
                                          unsigned long long* acc, uint32_t* status) {
  constexpr int G = NT / GS;
  const int gi = (int)threadIdx.x / GS;
  FEnt* other = front + FCAP;
  FEnt* stage = other + FCAP;
  __shared__ int sg_nf[G], sg_flag[G], sg_full[G], sg_ntot[G], sg_otot[G];
  __shared__ Vec sg_out[G], sg_grow[G], sg_fr[G];
  int& s_nf = sg_nf[gi];
  // s_flag: a visit's updates were dropped (set by any thread between two
  // barriers, read after the second).  s_full: the pool had no room (set by
  // thread 0 right before a barrier at each allocation, read right after it): a
  // word of its own, as slower warps may still be reading s_flag when thread 0
  // allocates.  Every branch with barriers depends on such settled words only.
  int& s_flag = sg_flag[gi];
  int& s_full = sg_full[gi];
  int& s_ntot = sg_ntot[gi];
  int& s_otot = sg_otot[gi];
  Vec& s_out = sg_out[gi];
  Vec& s_grow = sg_grow[gi];
  Vec& s_fr = sg_fr[gi];
  const int tid = gtid<GS>();
  if (tid == 0) {
    s_flag = 0;
    s_nf = 0;
    s_ntot = 0;
    s_otot = 0;
    if (live && phase_b) {
      uint4 cs = W.cont[j];
      s_ntot = (int)cs.y;  // saved entries, combined below like a stage
      s_out.off = cs.z;
      s_out.size = cs.w;
      s_out.cap = W.cont_cap[j];
      s_out.h = W.pool + s_out.off;
    } else if (live) {
      s_out.off = kOut0 * (uint32_t)j;
      s_out.size = 0;
      s_out.cap = kOut0;
      s_out.h = W.pool + s_out.off;
      if ((unsigned long long)kOut0 * (unsigned)j + kOut0 > W.pool_cap) {
        atomicOr(status, kErrPool);
        s_flag = 1;
      }
      // seed: the boundary of the critical triangle.  Its highest vertex is v0;
      // the edge opposite goes to its lower star as a link edge of v0.
      const uint32_t ve = c.L.c2_ve[W.cols[j]];
      const int e0 = (int)(ve & 63u);
      FEnt e;
      e.key = ve >> 6;  // alone in the frontier: not compared
      e.mask = 1u << (links.le[e0] & 15) | 1u << (links.le[e0] >> 4 & 15);
      e.pad = (uint32_t)e0 + 1;
      front[0] = e;
      s_nf = 1;
    }
  }
  gsync<GS>();
  if (phase_b) {
    uint4 cs = W.cont[j];
    for (int i = tid; i < (int)cs.y; i += GS) stage[i] = fent_restore(W.pool + cs.x + 2 * (size_t)i);
    gsync<GS>();
    int n0 = group_combine<GS, SCAP>(front, 0, 0, other, stage, s_ntot, scan_sm);
    if (tid == 0) {
      s_nf = n0;
      s_ntot = 0;
    }
    gsync<GS>();
  }
  int visits = 0, updates = 0, rounds = 0;
  bool failed = s_flag != 0;
  gsync<GS>();  // before the first visits, which may set it
  bool handoff = false;
  bool run = live && !failed;
  for (;;) {
    const int nf = run ? s_nf : 0;
    if (nf == 0 || (!phase_b && rounds >= max_rounds)) run = false;
    // every target is a lower neighbour of the visited vertex, so the
    // frontier's highest key drops each round: at most nv rounds
    if (run && rounds > c.d.nv) {
      if (tid == 0) atomicOr(status, kErrRounds);
      failed = true;
      run = false;
    }
    if (!gany<GS>(run)) break;
    rounds += run ? 1 : 0;
    const int nb = run ? min(GS, nf) : 0;
    int myout = 0;
    unsigned long long myouts[kOutCap];
    if (tid < nb) {
      FEnt cur = front[tid];
      for (int k = 0;; ++k) {
        ++visits;
        FEnt nxt;
        bool more = k + 1 < c.chain && myout + 14 <= kOutCap;
        if (!d1_visit<SCAP>(c, cur, snd, links, stage, &s_ntot, &s_flag, myouts, myout, updates, more, &nxt, status))
          break;
        cur = nxt;
      }
    }
    const int ooff = myout ? atomicAdd(&s_otot, myout) : 0;
    gsync<GS>();
    if (run && s_flag) {  // stage overflow: updates were dropped, recompute the column
      failed = true;
      run = false;
    }
    // outputs: append to the column's list in the pool (grown by the group)
    const int otot = run ? s_otot : 0;
    if (gany<GS>(otot > 0)) {
      if (tid == 0) {
        s_grow.h = nullptr;
        s_full = 0;
        if (otot > 0 && s_out.size + otot > s_out.cap) {
          uint32_t cap = s_out.cap;
          while (cap < s_out.size + otot) cap *= 2;
          if (!vec_alloc(W, s_grow, cap, status)) {
            s_grow.h = nullptr;
            s_full = 1;
          }
        }
      }
      gsync<GS>();
      if (run && s_full) {
        failed = true;
        run = false;
      }
      const bool grow = run && otot > 0 && s_grow.h;
      if (gany<GS>(grow)) {
        if (grow)
          for (uint32_t i = tid; i < s_out.size; i += GS) s_grow.h[i] = s_out.h[i];
        gsync<GS>();
        if (grow && tid == 0) {
          s_grow.size = s_out.size;
          s_out = s_grow;
        }
        gsync<GS>();
      }
      if (run)
        for (int k = 0; k < myout; ++k) s_out.h[s_out.size + ooff + k] = myouts[k];
      gsync<GS>();
      if (tid == 0 && run) {
        s_out.size += otot;
        s_otot = 0;
      }
    }
    const int ntot = run ? s_ntot : 0;
    const int rest = nf - nb;
    const bool over = run && rest + ntot > FCAP;  // the new frontier would not fit
    if (gany<GS>(over)) {
      const bool save = over && !phase_b;  // phase A: the rest and the stage go to phase B as they are
      if (over) {
        failed = true;
        run = false;
      }
      if (save && tid == 0) s_full = vec_alloc(W, s_fr, 2u * (uint32_t)(rest + ntot), status) ? 0 : 1;
      gsync<GS>();
      if (save && !s_full) {
        handoff = true;
        for (int i = tid; i < rest; i += GS) fent_save(s_fr.h + 2 * i, front[nb + i]);
        for (int i = tid; i < ntot; i += GS) fent_save(s_fr.h + 2 * (rest + i), stage[i]);
      }
      gsync<GS>();
      if (handoff && save && tid == 0) {
        W.cont[j] = make_uint4(s_fr.off, (uint32_t)(rest + ntot), s_out.off, s_out.size);
        W.cont_cap[j] = s_out.cap;
        W.big[atomicAdd(W.nbig, 1)] = j;
      }
    }
    if (!gany<GS>(run && !(rest == 0 && ntot <= GS))) {
      // every entry is taken next round, so neither their order nor
      // combining equal keys matters (a star listed twice is visited twice
      // with parts of its mask: the projection is linear)
      if (run)
        for (int i = tid; i < ntot; i += GS) front[i] = stage[i];
      gsync<GS>();  // every thread has read s_ntot before it is reset
      if (tid == 0 && run) {
        s_nf = ntot;
        s_ntot = 0;
      }
      gsync<GS>();
      continue;
    }
    gsync<GS>();
    // a group that has stopped keeps its frontier: it combines nothing
    const int nn = group_combine<GS, SCAP>(front, run ? nb : 0, run ? nf : 0, other, stage, run ? ntot : 0, scan_sm);
    if (tid == 0 && run) {
      s_nf = nn;
      s_ntot = 0;
    }
    gsync<GS>();
  }
  // visits and target updates of the whole group
  int vtot, utot;
  gscan<GS>(visits, vtot, scan_sm);
  gscan<GS>(updates, utot, scan_sm);
  bool redo = live && failed && !handoff;
  const bool open = live && !failed && !phase_b && s_nf > 0;  // still open after max_rounds: save the frontier for phase B
  if (gany<GS>(open)) {
    if (open && tid == 0) s_full = vec_alloc(W, s_fr, 2u * (uint32_t)s_nf, status) ? 0 : 1;
    gsync<GS>();
    redo = redo || (open && s_full);
    if (open && !redo)
      for (int i = tid; i < s_nf; i += GS) fent_save(s_fr.h + 2 * i, front[i]);
    gsync<GS>();
    if (open && !redo && tid == 0) {
      W.cont[j] = make_uint4(s_fr.off, (uint32_t)s_nf, s_out.off, s_out.size);
      W.cont_cap[j] = s_out.cap;
      W.big[atomicAdd(W.nbig, 1)] = j;
    }
  }
  const bool goes_on = live && !redo && (handoff || open);
  if (goes_on && tid == 0) {
    W.redo[j] = 0;
    W.hsize[j] = 0;
    acc[0] += (unsigned long long)vtot;
    acc[2] += (unsigned long long)rounds;
    acc[4] += (unsigned long long)utot;
  }
  // finished: (v, x) -> C1 index, sort descending, keep the entries present
  // an odd number of times (Z/2)
  bool fin = live && !redo && !goes_on;
  int nout = fin ? (int)s_out.size : 0;
  int n2 = 1;
  while (n2 < nout) n2 <<= 1;
  n2 = gmax<GS>(n2);
  unsigned long long* a = reinterpret_cast<unsigned long long*>(stage);
  if (n2 > 2 * SCAP) {  // too long for shared memory: sort in the pool
    if (fin && tid == 0) s_full = vec_alloc(W, s_grow, (uint32_t)n2, status) ? 0 : 1;
    gsync<GS>();
    if (fin && s_full) {
      redo = true;
      fin = false;
      nout = 0;
    }
    if (fin) a = s_grow.h;
  }
  if (redo && tid == 0) {
    W.redo[j] = 1;
    W.hsize[j] = 0;
  }
  if (!gany<GS>(fin)) return;
  for (int i = tid; fin && i < n2; i += GS) {
    unsigned long long ci = 0;
    if (i < nout) {
      uint32_t v = (uint32_t)(s_out.h[i] >> 4);
      int x = (int)(s_out.h[i] & 15ull);
      int cnt = __popc(rec_crit_edges(ld_rec(c.rec, v)));
      uint32_t base = c.c1base[v];
      int found = -1;
      for (int k2 = 0; k2 < cnt; ++k2)
        if ((int)(c.L.c1_vn[base + k2] & 15u) == x) found = (int)(base + k2);
      if (found < 0) atomicOr(status, kErrInconsistent);
      ci = (unsigned long long)(found < 0 ? 0 : found);
    }
    a[i] = ci;
  }
  gsync<GS>();
  group_sort_desc<GS>(a, n2, fin);
  int kept = 0;
  const int most = gmax<GS>(nout);
  for (int base = 0; base < most; base += GS) {
    int k = base + tid;
    int keep = 0;
    unsigned long long x = 0;
    if (k < nout) {
      x = a[k];
      if (k == 0 || a[k - 1] != x) {
        int e = k + 1;
        while (e < nout && a[e] == x) ++e;
        keep = (e - k) & 1;
      }
    }
    int t;
    int off = gscan<GS>(keep, t, scan_sm);
    if (keep) s_out.h[kept + off] = x;
    kept += t;
  }
  gsync<GS>();
  if (fin && tid == 0) {
    W.hoff[j] = s_out.off;
    W.hsize[j] = (uint32_t)kept;
    W.redo[j] = 0;
    acc[0] += (unsigned long long)vtot;
    acc[1] = max(acc[1], (unsigned long long)vtot);
    acc[2] += (unsigned long long)rounds;
    acc[3] = max(acc[3], (unsigned long long)rounds);
    acc[4] += (unsigned long long)utot;
  }
}

// Groups take columns by ticket (W.flags[2] in phase A, [3] in phase B), so a
// launch is as large as the GPU and not as the diagram: phase B's blocks with
// nothing to do took 0.29 ms for 4.9e5 triangles.
template <int NT, int FCAP, int SCAP, int MINB = (NT == 32 ? 12 : 4), int GS = NT>
__global__ void __launch_bounds__(NT, MINB) k_d1_morse_group(D1Ctx c, D1Work W, int max_rounds, uint32_t* status) {
  static_assert(GS == NT || GS < 32, "several groups only within one warp");
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ D1Links links;
  __shared__ int32_t snd[16];
  __shared__ int scan_sm[16];  // GS/32 + 1 <= 16 (blocks only)
  __shared__ int s_ticket;
  const bool phase_b = max_rounds <= 0;
  const int total = phase_b ? *W.nbig : W.flags[1];
  FEnt* front = reinterpret_cast<FEnt*>(smem) + (size_t)(threadIdx.x / GS) * (2 * FCAP + SCAP);
  if (threadIdx.x < 14) snd[threadIdx.x] = c.nd.d[threadIdx.x];
  for (int i = threadIdx.x; i < (int)(sizeof(D1Links) / 4); i += NT)
    reinterpret_cast<uint32_t*>(&links)[i] = __ldg(reinterpret_cast<const uint32_t*>(&g_links) + i);
  if (NT > 32) __syncthreads();
  else __syncwarp();  // read by every group
  // the group's share of W.stats (added once: per column the atomics on one
  // line took as long as a round)
  __shared__ unsigned long long s_acc[NT / GS][kD1Stats];
  unsigned long long* acc = s_acc[threadIdx.x / GS];
  if (gtid<GS>() == 0)
    for (int k = 0; k < kD1Stats; ++k) acc[k] = 0;
  int* const tickets = W.flags + (phase_b ? 3 : 2);
  // With many columns to come the next ticket is drawn before the column, else
  // after it (a ticket drawn early waits behind a long column).
  const bool early = !phase_b && total > 8 * (int)gridDim.x * (NT / GS);
  int next = gtid<GS>() == 0 ? atomicAdd(tickets, 1) : 0;
  for (;;) {
    int t;
    if (GS > 32) {
      if (threadIdx.x == 0) s_ticket = next;
      __syncthreads();
      t = s_ticket;
    } else {
      t = __shfl_sync(0xFFFFFFFFu, next, 0, GS);
    }
    const bool live = t < total;
    if (!gany<GS>(live)) break;
    if (early && gtid<GS>() == 0) next = atomicAdd(tickets, 1);
    gsync<GS>();  // the group is done with the last column's shared words and ticket
    d1_column<NT, FCAP, SCAP, GS>(c, W, !live ? 0 : phase_b ? W.big[t] : t, live, phase_b, max_rounds, front, snd,
                                  links, scan_sm, acc, status);
    if (!early && gtid<GS>() == 0) next = atomicAdd(tickets, 1);
  }
  if (gtid<GS>() == 0 && acc[0]) {
    atomicAdd(&W.stats[0], acc[0]);
    atomicMax(&W.stats[1], acc[1]);
    atomicAdd(&W.stats[2], acc[2]);
    atomicMax(&W.stats[3], acc[3]);
    atomicAdd(&W.stats[4], acc[4]);
  }
}

// Phase A is bound by the latency of its rounds (a table row from L2 or memory,
// then a few hundred instructions; ncu: 43 % of issue slots, 60 % of the stalls
// on loads), so what counts is columns in flight and lanes in use: a round
// visits 4 lower stars on average on noise, 30 on long filaments.  Registers
// are held to 64 so that 32 one-warp blocks share an SM; a column that outgrows
// its tile continues in phase B.  Stage time, ms, with a quarter warp and
// 32 + 64 entries (8) / a quarter and 16 + 32 (6) / half a warp and 32 + 64 (5) /
// a whole warp and 64 + 128 (4):
//   256^3 field, 2.6e6 triangles        8.1 / 9.5 / 8.7 / 10.4   -> 8
//   96^3 field, 7e4 triangles           0.78 / 0.71 / 0.83 / 0.93 -> 6
//   97 x 61 x 130 field, 8e4 triangles  0.54 / 0.50 / 0.61 / 0.71 -> 6
//   32^3 field, 3e3 triangles           0.116 / 0.112 / 0.103 / 0.105
//   128^3 filament field, 2e3           0.42 / 0.40 / 0.44 / 0.39 -> 4
// Before (half-warp groups on their own, whole rows in local memory, a launch
// block per column): 15.2, 1.03, 0.77, 0.103 and 0.50 ms.
constexpr int kThreadsB = 128;
constexpr int kFrontA = 64, kStageA = 128;
constexpr int kFrontH = 32, kStageH = 64;
constexpr int kFrontQ = 16, kStageQ = 32;
constexpr int kFrontB = 1024, kStageB = 1024;
static_assert(kFrontA + kStageA <= kStageB, "a phase A handoff fits phase B's stage");

static size_t d1_group_smem(int fcap, int scap) { return (2 * (size_t)fcap + scap) * sizeof(FEnt); }

// Candidate columns in increasing triangle order; their number stays on the
// device (W.flags[1]), the later D1 launches are sized by n2.
void launch_d1_prepare(int n2, D1Work& W, PairOut& P, cudaStream_t st) {
  if (n2 == 0) {
    cudaMemsetAsync(W.flags + 1, 0, sizeof(int32_t), st);
    return;
  }
  if (n2 <= kSelectOne) {
    k_d1_select_one<<<1, kSelectT, 0, st>>>(n2, P.d2_max, W.cols, P.d1_edge, W.flags + 1, W.pool_head); note_launch();
    return;
  }
  uint32_t* flag = reinterpret_cast<uint32_t*>(W.lowc);  // scratch (n2 entries available)
  uint32_t* pos = reinterpret_cast<uint32_t*>(W.hsize);
  uint32_t* sums = reinterpret_cast<uint32_t*>(W.hcap);
  k_d1_select<<<(n2 + 255) / 256, 256, 0, st>>>(n2, P.d2_max, flag); note_launch();
  exclusive_scan_u32(flag, pos, n2, sums, st);
  k_d1_gather<<<(n2 + 255) / 256, 256, 0, st>>>(n2, flag, pos, W.cols, P.d1_edge, W.flags + 1, W.pool_head); note_launch();
}

void launch_d1_morse(const Dims& d, const NbrDelta& nd, const CritLists& L, int n1, int n2, const uint32_t* rank,
                     const uint32_t* order, const Rec* rec, const D1Tab* tab, const uint32_t* c1base, D1Work& W,
                     PairOut& P, uint32_t* status, cudaStream_t st) {
  if (n2 == 0) return;
  D1Ctx c;
  c.d = d;
  c.nd = nd;
  c.rank = rank;
  c.order = order;
  c.rec = rec;
  c.tab = tab;
  c.c1base = c1base;
  c.L = L;
  c.d0_killed = P.d0_killed;
  c.d0mask = P.d0mask;
  {
    const int64_t ch = g_morse_chain.load();
    c.chain = ch > 0 ? (int)std::min<int64_t>(ch, 8) : (n2 >= kLargeD1 ? kChainLarge : kChainSmall);
  }
  const int64_t mr = g_morse_rounds.load();
  const int roundsA =
      mr > 0 ? (int)std::min<int64_t>(mr, 1 << 20) : (n2 >= kLargeD1 ? kRoundsLarge : n2 >= kTinyD1 ? kRoundsSmall : kRoundsTiny);
  cudaMemsetAsync(W.stats, 0, kD1Stats * sizeof(unsigned long long), st);
  cudaMemsetAsync(W.nbig, 0, sizeof(int32_t), st);
  cudaMemsetAsync(W.flags + 2, 0, 2 * sizeof(int32_t), st);  // the tickets
  size_t sb = d1_group_smem(kFrontB, kStageB);
  int dev = 0;
  cudaGetDevice(&dev);
  static std::atomic<bool> attr[64] = {};  // fields may be driven from several host threads
  if (dev >= 0 && dev < 64 && !attr[dev].load(std::memory_order_acquire)) {
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontA, kStageA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)d1_group_smem(kFrontA, kStageA));
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontA * 2, kStageA * 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)d1_group_smem(kFrontA * 2, kStageA * 2));
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontA * 4, kStageA * 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)d1_group_smem(kFrontA * 4, kStageA * 4));
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontA, kStageA, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)d1_group_smem(kFrontA, kStageA));
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontA, kStageA, 32, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(2 * d1_group_smem(kFrontA, kStageA)));
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontH, kStageH, 32, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(2 * d1_group_smem(kFrontH, kStageH)));
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontH, kStageH, 32, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(4 * d1_group_smem(kFrontH, kStageH)));
    cudaFuncSetAttribute(k_d1_morse_group<32, kFrontQ, kStageQ, 32, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(4 * d1_group_smem(kFrontQ, kStageQ)));
    cudaFuncSetAttribute(k_d1_morse_group<kThreadsB, kFrontB, kStageB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sb);
    attr[dev].store(true, std::memory_order_release);
  }
  // blocks of g columns, at most what an SM holds of them
  const auto blocks = [&](int g, int per_sm) { return std::min((n2 + g - 1) / g, d1_sms() * per_sm); };
  // knob 7 = 0: by size, see the figures at kThreadsB
  int64_t phase_a = g_d1_phase_a.load();
  if (phase_a == 0) phase_a = n2 >= kLargeD1 ? 8 : n2 >= kTinyD1 ? 6 : 4;
  switch (phase_a) {
    case 1:
      k_d1_morse_group<32, kFrontA * 2, kStageA * 2><<<blocks(1, 12), 32, d1_group_smem(kFrontA * 2, kStageA * 2), st>>>(
          c, W, roundsA, status);
      break;
    case 2:
      k_d1_morse_group<32, kFrontA * 4, kStageA * 4><<<blocks(1, 12), 32, d1_group_smem(kFrontA * 4, kStageA * 4), st>>>(
          c, W, roundsA, status);
      break;
    case 3:  // one warp per column without the register cap
      k_d1_morse_group<32, kFrontA, kStageA><<<blocks(1, 12), 32, d1_group_smem(kFrontA, kStageA), st>>>(c, W, roundsA,
                                                                                             status);
      break;
    case 4:  // one warp per column, registers capped (63) so that 32 warps fit an SM
      k_d1_morse_group<32, kFrontA, kStageA, 32><<<blocks(1, 32), 32, d1_group_smem(kFrontA, kStageA), st>>>(c, W, roundsA,
                                                                                                  status);
      break;
    case 5:  // half a warp per column with the smaller tile
      k_d1_morse_group<32, kFrontH, kStageH, 32, 16><<<blocks(2, 32), 32, 2 * d1_group_smem(kFrontH, kStageH), st>>>(
          c, W, roundsA, status);
      break;
    case 6:  // a quarter of a warp per column with the smallest tile
      k_d1_morse_group<32, kFrontQ, kStageQ, 32, 8><<<blocks(4, 32), 32, 4 * d1_group_smem(kFrontQ, kStageQ), st>>>(
          c, W, roundsA, status);
      break;
    case 8:  // a quarter of a warp per column with half a warp's tile
      k_d1_morse_group<32, kFrontH, kStageH, 32, 8><<<blocks(4, 32), 32, 4 * d1_group_smem(kFrontH, kStageH), st>>>(
          c, W, roundsA, status);
      break;
    default:  // (7) half a warp per column (two columns per warp), registers capped for 32 warps per SM
      k_d1_morse_group<32, kFrontA, kStageA, 32, 16><<<blocks(2, 32), 32, 2 * d1_group_smem(kFrontA, kStageA), st>>>(
          c, W, roundsA, status);
  }
  note_launch();
  k_d1_morse_group<kThreadsB, kFrontB, kStageB><<<blocks(1, 4), kThreadsB, sb, st>>>(c, W, 0, status); note_launch();
  k_d1_morse<<<(n2 + 63) / 64, 64, 0, st>>>(c, W, status); note_launch();
}

}  // namespace tsf
