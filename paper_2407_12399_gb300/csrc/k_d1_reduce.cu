// k_d1_reduce.cu -- D1 (1-saddle, 2-saddle) pairs: column reduction over Z/2
// of the Morse boundaries (k_pairs.cu), every addition of an earlier column.
//
// The pairs are the lows of any reduction made by left-to-right additions, so
// the schedule is free.  Three kernels share one state, a record {column,
// pool offset, length} per row (critical edge) of the smallest column so far
// that holds the row as its low:
//   k_d1_reduce_grid (large diagrams): rounds over the whole GPU while many
//     columns are active;
//   k_d1_columns: one warp per column, no rounds and no barriers.  A column
//     adds the owner of its low while that owner is an earlier column; it
//     claims a low whose owner is later or absent by a 128-bit compare and
//     swap of the record, and the warp then goes on with the column that it
//     displaced.  A record names an immutable copy of the owner's entries in
//     the bump-allocated pool, so a reader never waits and never sees a
//     column half written;
//   k_d1_long: a column that took many additions, or outgrew the warp's
//     buffers, gets a block.  Its entries are a bit set in shared memory, and
//     each round adds the owners of many of its highest entries at once.
#include <algorithm>
#include <atomic>

#include "tsf_grid.cuh"
#include "tsf_kernels.cuh"

namespace tsf {

constexpr int kUFT = 1024;
constexpr uint32_t kNoOwner = 0x7FFFFFFFu;
constexpr uint32_t kLongAdd = 64;  // whole-GPU rounds: column additions at least this long run on a warp
constexpr int kLongCap = 1024;     // ... at most this many per block and round (the rest on one thread)

// Stage failures after which nothing is reduced (results are discarded).
__device__ __forceinline__ bool d1_failed(const uint32_t* status) {
  return (*reinterpret_cast<const volatile uint32_t*>(status) & (kErrSpin | kErrRounds | kErrPool | kErrTrace)) != 0u;
}

// Nobody owns a row yet: a launch of its own, ahead of kernels that return
// early after a failed stage, so that every record is one of this diagram's.
__global__ void k_d1_init(int n1, D1Work W) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n1) return;
  W.owner[i] = kNoOwner;
  W.orec[i] = make_uint4(kNoOwner, 0u, 0u, 0u);
}

// Number of entries of a strictly decreasing column greater than v (loads
// from L2: other SMs may have written the column in this kernel).
__device__ __forceinline__ uint32_t d1_count_greater(unsigned long long v, const unsigned long long* arr,
                                                    uint32_t len) {
  uint32_t lo = 0, hi = len;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldcg(arr + mid) > v) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// One warp writes the sum over Z/2 of two strictly decreasing columns a (n)
// and b (nb) to d, decreasing, and returns its length.  An entry x of a that
// b lacks lands at x + (entries of b above it) - 2 (entries of a above it
// that b also has): everything above it, minus the cancelled pairs.  Same
// for b.  Positions outside [0, n + nb) set kErrInconsistent.
__device__ uint32_t d1_warp_add(const unsigned long long* a, uint32_t n, const unsigned long long* b, uint32_t nb,
                                unsigned long long* d, uint32_t* status) {
  const int lane = threadIdx.x & 31;
  const uint32_t cap = n + nb;
  uint32_t common = 0;
  for (int pass = 0; pass < 2; ++pass) {
    const unsigned long long* p = pass == 0 ? a : b;
    const unsigned long long* q = pass == 0 ? b : a;
    const uint32_t np_ = pass == 0 ? n : nb, nq = pass == 0 ? nb : n;
    uint32_t before = 0;
    for (uint32_t x0 = 0; x0 < np_; x0 += 32) {
      const uint32_t x = x0 + lane;
      bool found = false;
      uint32_t c = 0;
      unsigned long long v = 0;
      if (x < np_) {
        v = __ldcg(p + x);
        c = d1_count_greater(v, q, nq);
        found = c < nq && __ldcg(q + c) == v;
      }
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, found);
      if (x < np_ && !found) {
        const uint32_t pos = x + c - 2u * (before + __popc(bal & ((1u << lane) - 1u)));
        if (pos < cap) d[pos] = v;
        else atomicOr(status, kErrInconsistent);
      }
      before += __popc(bal);
    }
    common = before;
  }
  return cap - 2u * common;
}

__device__ __forceinline__ void d1_list_push(int32_t* next, int* n_next, int32_t* mark, int j, int round) {
  if (atomicExch(&mark[j], round) != round) next[atomicAdd(n_next, 1)] = j;
}


// Rounds over the whole GPU (cooperative launch, grid barriers between the
// phases) while at least `handoff` columns are active; the columns still
// active then go on in k_d1_columns.  In a round every listed column claims
// its low (atomicMin), then every listed column that does not own its low
// adds the owner's column (owners do not change in that phase) and is listed
// again; a settled owner that a smaller column displaces is listed for the
// next round.  Every read of state that another SM may have written in this
// kernel goes to L2.
__global__ void __launch_bounds__(kUFT) k_d1_reduce_grid(D1Work W, int n1, D1Ctl* ctl, int handoff, unsigned limit,
                                                         uint32_t* status) {
  const int ncols = W.flags[1];
  int32_t* listA = W.lowc;
  int32_t* listB = reinterpret_cast<int32_t*>(W.hcap);
  int32_t* mark = W.redo;
  __shared__ int s_nlong;
  __shared__ int32_t s_long[kLongCap];
  const unsigned nb = gridDim.x;
  const int gt = blockIdx.x * kUFT + threadIdx.x, gn = nb * kUFT;
  const long long c_start = clock64();
  // an earlier stage failed (its results are discarded): every block returns
  // before the first barrier, and the later kernels see the same bits
  if (d1_failed(status)) return;
  for (int j = gt; j < ncols; j += gn) {
    mark[j] = -1;
    if (W.hsize[j] > 0) listA[atomicAdd(&ctl->n[0], 1)] = j;
  }
  if (!grid_barrier(ctl->bar, nb, status, limit)) return;
  int which = 0;
  for (int round = 0;; ++round) {
    const int na = *reinterpret_cast<volatile int*>(&ctl->n[which]);
    if (na == 0 || na < handoff) break;
    if (round > ncols + 2) {
      if (gt == 0) atomicOr(status, kErrRounds);
      break;
    }
    const long long c_round = clock64();
    const int32_t* cur = which ? listB : listA;
    int32_t* nxt = which ? listA : listB;
    int* n_next = &ctl->n[which ^ 1];
    if (threadIdx.x == 0) s_nlong = 0;
    for (int i = gt; i < na; i += gn) {
      const int j = __ldcg(&cur[i]);
      const int old = atomicMin(&W.owner[(int)__ldcg(&W.pool[__ldcg(&W.hoff[j])])], j);
      if (old > j && old != (int)kNoOwner) d1_list_push(nxt, n_next, mark, old, round);  // displaced owner
    }
    if (!grid_barrier(ctl->bar, nb, status, limit)) return;
    for (int i = gt; i < na; i += gn) {
      const int j = __ldcg(&cur[i]);
      const uint32_t n = __ldcg(&W.hsize[j]);
      const unsigned long long* a = W.pool + __ldcg(&W.hoff[j]);
      const int o = __ldcg(&W.owner[(int)__ldcg(a)]);
      if (o == j) {  // owns its low: its record
        W.orec[(int)__ldcg(a)] = make_uint4((uint32_t)j, __ldcg(&W.hoff[j]), n, 0u);
        continue;
      }
      const uint32_t no = __ldcg(&W.hsize[o]);
      if (n + no >= kLongAdd) {  // long: one warp of this block adds it below
        const int q = atomicAdd(&s_nlong, 1);
        if (q < kLongCap) {
          s_long[q] = j;
          continue;
        }
      }
      const unsigned long long* b = W.pool + __ldcg(&W.hoff[o]);
      const uint32_t cap = n + no;
      const uint32_t off = atomicAdd(W.pool_head, cap);
      if ((unsigned long long)off + cap > W.pool_cap) {
        atomicOr(status, kErrPool);
        continue;
      }
      unsigned long long* d = W.pool + off;
      uint32_t x = 0, y = 0, m = 0;
      unsigned long long ax = x < n ? __ldcg(a) : 0, by = y < no ? __ldcg(b) : 0;
      while (x < n && y < no) {  // both decreasing: symmetric difference
        if (ax > by) {
          d[m++] = ax;
          ax = ++x < n ? __ldcg(a + x) : 0;
        } else if (by > ax) {
          d[m++] = by;
          by = ++y < no ? __ldcg(b + y) : 0;
        } else {
          ax = ++x < n ? __ldcg(a + x) : 0;
          by = ++y < no ? __ldcg(b + y) : 0;
        }
      }
      for (; x < n; ++x) d[m++] = __ldcg(a + x);
      for (; y < no; ++y) d[m++] = __ldcg(b + y);
      W.hoff[j] = off;
      W.hsize[j] = m;
      atomicAdd(&W.stats[6], (unsigned long long)m);
      atomicMax(&W.stats[7], (unsigned long long)m);
      if (m == 0) atomicOr(status, kErrEmptyColumn);
      else d1_list_push(nxt, n_next, mark, j, round);
    }
    __syncthreads();
    {  // this block's long additions, one warp each
      const int nlong = min(s_nlong, kLongCap), lane = threadIdx.x & 31;
      for (int q = threadIdx.x >> 5; q < nlong; q += kUFT / 32) {
        const int j = s_long[q];
        const uint32_t n = __ldcg(&W.hsize[j]);
        const unsigned long long* a = W.pool + __ldcg(&W.hoff[j]);
        const int o = __ldcg(&W.owner[(int)__ldcg(a)]);
        const uint32_t no = __ldcg(&W.hsize[o]);
        const unsigned long long* b = W.pool + __ldcg(&W.hoff[o]);
        const uint32_t cap = n + no;
        uint32_t off = 0;
        if (lane == 0) off = atomicAdd(W.pool_head, cap);
        off = __shfl_sync(0xFFFFFFFFu, off, 0);
        if ((unsigned long long)off + cap > W.pool_cap) {
          if (lane == 0) atomicOr(status, kErrPool);
          continue;
        }
        const uint32_t m = d1_warp_add(a, n, b, no, W.pool + off, status);
        if (lane == 0) {
          W.hoff[j] = off;
          W.hsize[j] = m;
          atomicAdd(&W.stats[6], (unsigned long long)m);
          atomicMax(&W.stats[7], (unsigned long long)m);
          if (m == 0) atomicOr(status, kErrEmptyColumn);
          else d1_list_push(nxt, n_next, mark, j, round);
        }
      }
    }
    which ^= 1;
    if (gt == 0) {
      ctl->n[which ^ 1] = 0;  // the list the next round fills
      ctl->which = which;
      W.stats[5] = (unsigned long long)(round + 1);
      W.stats[8] += 1;
      W.stats[9] += (unsigned long long)(clock64() - c_round);
    }
    if (!grid_barrier(ctl->bar, nb, status, limit)) return;
  }
  if (gt == 0) W.stats[10] += (unsigned long long)(clock64() - c_start);
}

// d = a (n) + b (nb) over Z/2 by one warp, all in shared memory, strictly
// decreasing.  Merge path: lane t walks positions [t*per, (t+1)*per) of the
// merged order (ties: a first, so a common entry is a[i] directly followed by
// b[j]); an entry is cancelled when the other column holds it, which each
// lane sees from its neighbour in the walk (b[j] from a[i-1], a[i] from
// b[j]).  A counting walk, a warp scan, then the writing walk.  Returns the
// length of d; the warp sees d complete.
__device__ uint32_t warp_merge_add(const uint32_t* a, uint32_t n, const uint32_t* b, uint32_t nb, uint32_t* d) {
  const int lane = threadIdx.x & 31;
  const uint32_t N = n + nb, per = (N + 31u) / 32u;
  const uint32_t k0 = min(N, (uint32_t)lane * per), k1 = min(N, k0 + per);
  // split: i = entries of a among the first k0 of the merged order
  uint32_t lo = k0 > nb ? k0 - nb : 0u, hi = min(k0, n);
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (a[mid] >= b[k0 - 1 - mid]) lo = mid + 1;
    else hi = mid;
  }
  const uint32_t i0 = lo, j0 = k0 - lo;
  uint32_t cnt = 0, total = 0;
  for (int pass = 0; pass < 2; ++pass) {
    uint32_t i = i0, j = j0, out = 0;
    if (pass == 1) {
      uint32_t inc = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += t;
      }
      total = __shfl_sync(0xFFFFFFFFu, inc, 31);
      out = inc - cnt;
    }
    uint32_t ai = i < n ? a[i] : 0u, bj = j < nb ? b[j] : 0u, ap = i > 0 ? a[i - 1] : 0xFFFFFFFFu;
    for (uint32_t k = k0; k < k1; ++k) {
      bool cancel;
      uint32_t v;
      if (i < n && (j >= nb || ai >= bj)) {
        v = ai;
        cancel = j < nb && ai == bj;
        ap = ai;
        ++i;
        ai = i < n ? a[i] : 0u;
      } else {
        v = bj;
        cancel = i > 0 && ap == bj;
        ++j;
        bj = j < nb ? b[j] : 0u;
      }
      if (!cancel) {
        if (pass == 1) d[out] = v;
        ++out;
      }
    }
    if (pass == 0) cnt = out;
  }
  __syncwarp();
  return total;
}

// ---------------------------------------------------------------------------
// Records: 16 bytes per row, read and replaced as one 128-bit word
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 rec_of(unsigned long long lo, unsigned long long hi) {
  return make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
}

// The acquire pairs with the release of rec_claim: the entries that the
// record names are visible after it.
__device__ __forceinline__ uint4 rec_load(const uint4* p) {
  unsigned long long lo, hi;
  asm volatile(
      "{\n\t.reg .b128 t;\n\t"
      "ld.acquire.gpu.global.b128 t, [%2];\n\t"
      "mov.b128 {%0, %1}, t;\n\t}"
      : "=l"(lo), "=l"(hi)
      : "l"(p)
      : "memory");
  return rec_of(lo, hi);
}

__device__ __forceinline__ uint4 rec_claim(uint4* p, const uint4& was, const uint4& now) {
  unsigned long long lo, hi;
  const unsigned long long wl = was.x | ((unsigned long long)was.y << 32), wh = was.z | ((unsigned long long)was.w << 32);
  const unsigned long long nl = now.x | ((unsigned long long)now.y << 32), nh = now.z | ((unsigned long long)now.w << 32);
  asm volatile(
      "{\n\t.reg .b128 c, n, o;\n\t"
      "mov.b128 c, {%3, %4};\n\t"
      "mov.b128 n, {%5, %6};\n\t"
      "atom.acq_rel.gpu.global.cas.b128 o, [%2], c, n;\n\t"
      "mov.b128 {%0, %1}, o;\n\t}"
      : "=l"(lo), "=l"(hi)
      : "l"(p), "l"(wl), "l"(wh), "l"(nl), "l"(nh)
      : "memory");
  return rec_of(lo, hi);
}

__device__ __forceinline__ bool rec_same(const uint4& a, const uint4& b) {
  return a.x == b.x && a.y == b.y && a.z == b.z && a.w == b.w;
}

// A record's column lies in the pool (an absent owner has none).
__device__ __forceinline__ bool rec_ok(const uint4& r, uint32_t pool_cap) {
  return r.x == kNoOwner || (r.z > 0u && (unsigned long long)r.y + r.z <= pool_cap);
}

// ---------------------------------------------------------------------------
// One warp per column
// ---------------------------------------------------------------------------
constexpr int kColWarps = 8;           // warps per block
constexpr uint32_t kColCap = 256;      // entries of a column kept in shared memory (three buffers per warp)
constexpr int kColSteps = 24;          // additions before a column moves to a block (default of knob 12)
constexpr int kColStepsMax = 1 << 16;  // ... at most
constexpr int kStepLimit = 1 << 22;    // loop bound (steps of a warp, rounds of a block) above any reduction

// Columns are taken in list order (all columns, in increasing order, or the
// list that the whole-GPU rounds left).  A warp keeps its column's entries in
// shared memory as 32-bit row indices; they reach the pool when the column
// claims a low or moves to the long list.
// Bound: each addition costs two dependent L2 round trips (the record of the
// low, then the owner's entries); the warps of all columns in flight overlap
// them, and no column waits for another.  kColSteps: a column of many
// additions is faster on a block (k_d1_long); 6, 12, 24, 40 and 80 additions
// before the move took 0.41, 0.39, 0.39, 0.40 and 0.45 ms on the 96^3
// mixture's diagram and 0.101, 0.093, 0.093, 0.083 and 0.079 ms on the 32^3
// one.
__global__ void __launch_bounds__(kColWarps * 32) k_d1_columns(D1Work W, int n1, D1Ctl* ctl, bool listed,
                                                               uint32_t cap, int max_adds, uint32_t* status) {
  __shared__ uint32_t bufs[kColWarps][3 * kColCap];
  const int lane = threadIdx.x & 31;
  uint32_t* A = bufs[threadIdx.x >> 5];
  uint32_t* B = A + kColCap;
  uint32_t* D = B + kColCap;
  if (__any_sync(0xFFFFFFFFu, d1_failed(status))) return;
  const int32_t* list = nullptr;
  int nlist = W.flags[1];
  if (listed) {
    list = ctl->which ? reinterpret_cast<const int32_t*>(W.hcap) : W.lowc;
    nlist = ctl->n[ctl->which];
  }
  int32_t* heavy = W.heavy;
  const long long c_start = clock64();
  unsigned long long t_merged = 0, t_adds = 0, t_longest = 0, t_chain = 0;
  for (int item = 0; item <= nlist; ++item) {  // a warp takes at most every item
    int k = 0;
    if (lane == 0) k = atomicAdd(&ctl->next, 1);
    k = __shfl_sync(0xFFFFFFFFu, k, 0);
    if (k >= nlist) break;
    uint32_t j = list ? (uint32_t)list[k] : (uint32_t)k;
    uint32_t n = W.hsize[j], off = W.hoff[j];
    if (n == 0) continue;  // no Morse boundary: an earlier stage reported why
    bool loaded = false, dirty = false;
    int adds = 0;
    for (int step = 0;; ++step) {
      if (step >= kStepLimit || (!loaded && (unsigned long long)off + n > W.pool_cap)) {
        if (lane == 0) atomicOr(status, step >= kStepLimit ? kErrRounds : kErrInconsistent);
        break;
      }
      if (n > cap || adds >= max_adds) {  // to a block
        if (dirty) {
          uint32_t o = 0;
          if (lane == 0) o = atomicAdd(W.pool_head, n);
          o = __shfl_sync(0xFFFFFFFFu, o, 0);
          if ((unsigned long long)o + n > W.pool_cap) {
            if (lane == 0) atomicOr(status, kErrPool);
            break;
          }
          for (uint32_t i = lane; i < n; i += 32) W.pool[o + i] = A[i];
          off = o;
        }
        if (lane == 0) {
          W.hoff[j] = off;
          W.hsize[j] = n;
          heavy[atomicAdd(&ctl->nheavy, 1)] = (int32_t)j;
        }
        break;
      }
      if (!loaded) {
        for (uint32_t i = lane; i < n; i += 32) A[i] = (uint32_t)__ldcg(W.pool + off + i);
        __syncwarp();
        loaded = true;
      }
      const uint32_t r = A[0];
      if (r >= (uint32_t)n1) {
        if (lane == 0) atomicOr(status, kErrInconsistent);
        break;
      }
      uint4 rec = rec_load(W.orec + r);
      // every lane acts on one view of the record
      rec.x = __shfl_sync(0xFFFFFFFFu, rec.x, 0);
      rec.y = __shfl_sync(0xFFFFFFFFu, rec.y, 0);
      rec.z = __shfl_sync(0xFFFFFFFFu, rec.z, 0);
      rec.w = __shfl_sync(0xFFFFFFFFu, rec.w, 0);
      __syncwarp();
      if (!rec_ok(rec, W.pool_cap) || rec.x == j) {
        if (lane == 0) atomicOr(status, kErrInconsistent);
        break;
      }
      if (rec.x < j) {  // an earlier owner: add it
        if (rec.z > cap || n + rec.z > cap) {
          adds = max_adds;  // outgrows the buffers: to a block
          continue;
        }
        for (uint32_t i = lane; i < rec.z; i += 32) B[i] = (uint32_t)__ldcg(W.pool + rec.y + i);
        __syncwarp();
        const uint32_t m = warp_merge_add(A, n, B, rec.z, D);
        uint32_t* t = A;
        A = D;
        D = t;
        n = m;
        dirty = true;
        ++adds;
        t_merged += m;
        t_longest = max(t_longest, (unsigned long long)m);
        if (m == 0) {
          if (lane == 0) atomicOr(status, kErrEmptyColumn);
          break;
        }
        continue;
      }
      // absent or later owner: claim the row
      if (dirty) {
        uint32_t o = 0;
        if (lane == 0) o = atomicAdd(W.pool_head, n);
        o = __shfl_sync(0xFFFFFFFFu, o, 0);
        if ((unsigned long long)o + n > W.pool_cap) {
          if (lane == 0) atomicOr(status, kErrPool);
          break;
        }
        for (uint32_t i = lane; i < n; i += 32) W.pool[o + i] = A[i];
        off = o;
        dirty = false;
        __threadfence();
        __syncwarp();
      }
      uint32_t won = 0;
      if (lane == 0) won = rec_same(rec_claim(W.orec + r, rec, make_uint4(j, off, n, 0u)), rec) ? 1u : 0u;
      won = __shfl_sync(0xFFFFFFFFu, won, 0);
      if (!won) continue;  // the record changed: look again
      t_adds += adds;
      t_chain = max(t_chain, (unsigned long long)adds);
      if (rec.x == kNoOwner) break;
      j = rec.x;  // go on with the displaced column
      off = rec.y;
      n = rec.z;
      loaded = false;
      adds = 0;
    }
    __syncwarp();
  }
  if (lane == 0) {
    if (t_adds) atomicAdd(&W.stats[11], t_adds);
    if (t_merged) atomicAdd(&W.stats[6], t_merged);
    if (t_longest) atomicMax(&W.stats[7], t_longest);
    if (t_chain) atomicMax(&W.stats[12], t_chain);
    atomicMax(&W.stats[15], (unsigned long long)(clock64() - c_start));
  }
}

// ---------------------------------------------------------------------------
// One block per long column
// ---------------------------------------------------------------------------
// The column is a bit set over the rows: the words of its highest rows in
// shared memory, the rest (diagrams of more rows than fit) in the block's
// slice of W.hbits, which is zero between columns.  A summary bit per 1024
// rows (32 words) says where a bit may be set.
//
// A round reads the highest 1024-row groups, looks up the owners of all their
// entries, and adds the owner of every entry above the highest one that has
// no earlier owner: each must go before that entry can be the low, and every
// addition is of an earlier column, so it is left-to-right.  An entry that a
// higher one's owner would have cancelled is added in vain and goes in a
// later round (the sum is over Z/2), so a round still lowers the top.  Once
// the highest entry has no earlier owner it is the low, and the block claims
// it like a warp of k_d1_columns.
// Bound: latency.  A round costs two dependent L2 round trips (records, then
// entries) and a few block barriers for the additions of up to 64 groups'
// entries, where one warp pays two round trips per addition.  One 256^3
// diagram holds columns of more than 10^4 additions: reducing such columns
// one addition at a time on a single block took 99 of that diagram's 103 ms
// of reduction; with this kernel the whole reduction takes 2.5 ms (97 x 61 x
// 130 8-bit field: 4.19 to 0.33 ms; 32^3 mixture: 0.32 to 0.09 ms).
constexpr int kLT = 512;                 // threads per block
constexpr int kLongGroups = kLT / 8;     // 1024-row groups read per round (8 lanes each)
constexpr uint32_t kLongEnts = 1024;     // entries per round, at most (one full group always fits)
constexpr size_t kLongSmem = 208 * 1024;  // summary, entries and bit set

struct LongShared {
  uint32_t ent[kLongEnts], off[kLongEnts], len[kLongEnts];
  int group[kLongGroups];
  uint32_t wsum[kLT / 32];
  uint32_t total, stuck, nent;
  int ngroup, top, item, go, base, npos;
  uint32_t j, poff, plen, row;
};

__host__ __device__ inline int long_groups(int n1) { return (n1 + 1023) / 1024; }
// groups whose words fit shared memory next to the summary
inline int long_window(int n1) {
  const long long left = (long long)kLongSmem - (long long)sizeof(LongShared) - 4ll * ((long_groups(n1) + 31) / 32) - 64;
  const long long w = std::min<long long>(std::max<long long>(left / 128, 0), long_groups(n1));
  const int64_t knob = get_knob(13);
  return (int)(knob > 0 ? std::min<long long>(w, knob) : w);
}

struct LongSet {
  uint32_t* words;    // shared: groups [base, base + window)
  uint32_t* gwords;   // global: groups below base
  uint32_t* summary;  // shared: bit per group
  int base;
};

// Flips row x; returns the change of the number of set rows.
__device__ __forceinline__ int long_flip(const LongSet& S, uint32_t x) {
  const int g = (int)(x >> 10);
  const uint32_t bit = 1u << (x & 31u);
  uint32_t* w = g >= S.base ? S.words + ((x >> 5) - (uint32_t)S.base * 32u) : S.gwords + (x >> 5);
  const uint32_t old = atomicXor(w, bit);
  const uint32_t sb = 1u << (g & 31);
  if (!(*reinterpret_cast<volatile uint32_t*>(S.summary + (g >> 5)) & sb)) atomicOr(S.summary + (g >> 5), sb);
  return (old & bit) ? -1 : 1;
}

// Words 4 * q .. 4 * q + 3 of group g.
__device__ __forceinline__ uint4 long_words(const LongSet& S, int g, int q) {
  return g >= S.base ? *reinterpret_cast<const uint4*>(S.words + (size_t)(g - S.base) * 32 + 4 * q)
                     : __ldcg(reinterpret_cast<const uint4*>(S.gwords + (size_t)g * 32 + 4 * q));
}

// Exclusive sum over the block (thread order); total in sh.total.
__device__ __forceinline__ uint32_t long_scan(LongShared& sh, uint32_t v) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) sh.wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    uint32_t x = lane < kLT / 32 ? sh.wsum[lane] : 0u, xi = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, xi, o);
      if (lane >= o) xi += t;
    }
    if (lane < kLT / 32) sh.wsum[lane] = xi - x;
    if (lane == 31) sh.total = xi;
  }
  __syncthreads();
  return sh.wsum[w] + inc - v;
}

// The highest groups (at most kLongGroups, descending, at or below summary
// word `top`) whose summary bit is set: sh.group[0 .. sh.ngroup).  Warp 0.
__device__ void long_top_groups(LongShared& sh, const LongSet& S, int top) {
  const int lane = threadIdx.x & 31;
  int cnt = 0, newtop = -1;
  for (int w0 = top; w0 >= 0 && cnt < kLongGroups; w0 -= 32) {
    const int wi = w0 - lane;
    uint32_t bits = wi >= 0 ? S.summary[wi] : 0u;
    const unsigned any = __ballot_sync(0xFFFFFFFFu, bits != 0u);
    if (any && newtop < 0) newtop = w0 - (__ffs(any) - 1);
    int c = __popc(bits), inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += t;
    }
    int at = cnt + inc - c;
    for (; bits && at < kLongGroups; ++at) {
      const int b = 31 - __clz(bits);
      bits &= ~(1u << b);
      sh.group[at] = wi * 32 + b;
    }
    cnt += __shfl_sync(0xFFFFFFFFu, inc, 31);
  }
  if (lane == 0) {
    sh.ngroup = min(cnt, kLongGroups);
    if (newtop >= 0) sh.top = newtop;
  }
}

__global__ void __launch_bounds__(kLT, 1) k_d1_long(D1Work W, int n1, D1Ctl* ctl, int window, uint32_t* status) {
  extern __shared__ __align__(16) uint32_t lsm[];
  __shared__ LongShared sh;
  const int nheavy = ctl->nheavy;
  if ((int)blockIdx.x >= nheavy) return;
  if (__syncthreads_or(d1_failed(status))) return;
  const int ngroups = long_groups(n1), nsum = (ngroups + 31) / 32;
  LongSet S;
  S.words = lsm;
  S.summary = lsm + (size_t)window * 32;
  S.gwords = W.hbits + (size_t)blockIdx.x * ((size_t)ngroups * 32);
  S.base = 0;
  const int tid = threadIdx.x, sub = tid >> 3, sl = tid & 7;
  const long long c_start = clock64();
  for (int i = tid; i < window * 32 + nsum; i += kLT) lsm[i] = 0u;
  unsigned long long t_adds = 0, t_merged = 0, t_rounds = 0, t_longest = 0;
  __syncthreads();
  for (int item = 0; item <= nheavy; ++item) {
    if (tid == 0) {
      sh.item = atomicAdd(&ctl->next_heavy, 1);
      sh.go = 0;
      if (sh.item < nheavy) {
        sh.go = 1;
        sh.j = (uint32_t)W.heavy[sh.item];
        sh.poff = W.hoff[sh.j];
        sh.plen = W.hsize[sh.j];
      }
    }
    __syncthreads();
    if (!sh.go) break;
    bool alive = true;
    // one iteration per column: the listed one, then each that it displaces
    for (int col = 0; alive && col < kStepLimit; ++col) {
      const uint32_t j = sh.j, poff = sh.poff, plen = sh.plen;
      if (plen == 0 || (unsigned long long)poff + plen > W.pool_cap || __ldcg(W.pool + poff) >= (unsigned long long)n1) {
        if (tid == 0) atomicOr(status, kErrInconsistent);
        break;
      }
      const int topg = (int)(__ldcg(W.pool + poff) >> 10);
      S.base = max(0, topg + 1 - window);
      if (tid == 0) sh.top = topg >> 5;
      int cnt = 0;  // this thread's share of the number of set rows
      for (uint32_t i = tid; i < plen; i += kLT) {
        const unsigned long long x = __ldcg(W.pool + poff + i);
        if (x < (unsigned long long)n1) cnt += long_flip(S, (uint32_t)x);
      }
      __syncthreads();
      int adds_here = 0;
      bool claimed = false;
      for (int round = 0; !claimed; ++round) {
        // a round lowers the top or takes it to a claim; a claim that fails
        // meets a smaller owner
        if (round >= kStepLimit) {
          if (tid == 0) atomicOr(status, kErrRounds);
          alive = false;
          break;
        }
        if (tid < 32) long_top_groups(sh, S, sh.top);
        if (tid == 0) sh.stuck = 0u;
        __syncthreads();
        const int ng = sh.ngroup;
        if (ng == 0) {  // nothing left: never for a valid reduction
          if (tid == 0) atomicOr(status, kErrEmptyColumn);
          alive = false;
          break;
        }
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        const int g = sub < ng ? sh.group[sub] : -1;
        if (g >= 0) q = long_words(S, g, 7 - sl);  // lane 0 of a group holds its highest words
        const uint32_t c = (uint32_t)(__popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w));
        uint32_t gsum = c;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) gsum += __shfl_xor_sync(0xFFFFFFFFu, gsum, o);
        if (g >= 0 && sl == 0 && gsum == 0u) atomicAnd(S.summary + (g >> 5), ~(1u << (g & 31)));
        const uint32_t at0 = long_scan(sh, c);
        // whole groups only, so that the entries taken are the highest ones:
        // the end of a thread's group is its last lane's position plus count
        const uint32_t gend = __shfl_sync(0xFFFFFFFFu, at0 + c, (tid & 31) | 7);
        if (tid == 0) sh.nent = 0u;
        __syncthreads();
        if (gend <= kLongEnts) {
          uint32_t at = at0;
          const uint32_t w4[4] = {q.w, q.z, q.y, q.x};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t b = w4[i];
            const uint32_t wbase = (uint32_t)g * 1024u + (uint32_t)(7 - sl) * 128u + (uint32_t)(3 - i) * 32u;
            for (; b; ++at) {
              const int p = 31 - __clz(b);
              b &= ~(1u << p);
              sh.ent[at] = wbase + (uint32_t)p;
            }
          }
          if (c) atomicMax(&sh.nent, at);
        }
        __syncthreads();
        const uint32_t ne = sh.nent;
        if (ne == 0u) {  // stale summary bits only
          __syncthreads();
          continue;
        }
        for (uint32_t i = tid; i < ne; i += kLT) {
          const uint32_t e = sh.ent[i];
          uint4 rec = make_uint4(kNoOwner, 0u, 0u, 0u);
          if (e < (uint32_t)n1) rec = rec_load(W.orec + e);
          if (e >= (uint32_t)n1 || !rec_ok(rec, W.pool_cap) || rec.x == j) {
            atomicOr(status, kErrInconsistent);
            rec.x = kNoOwner;
          }
          sh.len[i] = 0u;
          if (rec.x < j) {
            sh.off[i] = rec.y;
            sh.len[i] = rec.z;
          } else {
            atomicMax(&sh.stuck, e + 1u);
          }
        }
        __syncthreads();
        const uint32_t stuck = sh.stuck;
        if (sh.ent[0] + 1u > stuck) {
          // entries are descending: the ones above the stuck one are a prefix
          for (uint32_t i = sub; i < ne; i += kLongGroups) {
            if (sh.ent[i] + 1u <= stuck) break;
            const uint32_t off = sh.off[i], len = sh.len[i];
            for (uint32_t k = sl; k < len; k += 8) {
              const unsigned long long x = __ldcg(W.pool + off + k);
              if (x < (unsigned long long)n1) cnt += long_flip(S, (uint32_t)x);
            }
            if (sl == 0) {
              ++t_adds;
              ++adds_here;
              t_merged += len;
            }
          }
          if (tid == 0) ++t_rounds;
          __syncthreads();
          continue;
        }
        // the highest entry has no earlier owner: it is the low.  Write the
        // column to the pool (clearing the set) and claim the row.
        const uint32_t n = [&] {
          long_scan(sh, (uint32_t)cnt);  // the shares may be negative; their sum is not
          return sh.total;
        }();
        if (tid == 0) {
          const uint32_t o = atomicAdd(W.pool_head, n);
          sh.go = (unsigned long long)o + n <= W.pool_cap;
          if (!sh.go) atomicOr(status, kErrPool);
          sh.poff = o;
          sh.row = stuck - 1u;
          sh.npos = 0;
        }
        __syncthreads();
        if (!sh.go) {
          alive = false;
          break;
        }
        const uint32_t noff = sh.poff;
        for (int pass = 0; pass <= ngroups; ++pass) {
          if (tid < 32) long_top_groups(sh, S, sh.top);
          __syncthreads();
          const int mg = sh.ngroup;
          if (mg == 0) break;
          uint4 x = make_uint4(0u, 0u, 0u, 0u);
          const int gg = sub < mg ? sh.group[sub] : -1;
          if (gg >= 0) x = long_words(S, gg, 7 - sl);
          const uint32_t cc = (uint32_t)(__popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w));
          uint32_t at = (uint32_t)sh.npos + long_scan(sh, cc);
          const uint32_t w4[4] = {x.w, x.z, x.y, x.x};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t b = w4[i];
            const uint32_t wbase = (uint32_t)gg * 1024u + (uint32_t)(7 - sl) * 128u + (uint32_t)(3 - i) * 32u;
            for (; b; ++at) {
              const int p = 31 - __clz(b);
              b &= ~(1u << p);
              if (at < n) W.pool[noff + at] = wbase + (uint32_t)p;
            }
          }
          if (cc) {
            uint32_t* w = gg >= S.base ? S.words + (size_t)(gg - S.base) * 32 : S.gwords + (size_t)gg * 32;
            *reinterpret_cast<uint4*>(w + 4 * (7 - sl)) = make_uint4(0u, 0u, 0u, 0u);
          }
          if (gg >= 0 && sl == 0) atomicAnd(S.summary + (gg >> 5), ~(1u << (gg & 31)));
          __syncthreads();
          if (tid == 0) sh.npos += (int)sh.total;
          __syncthreads();
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) {
          if ((uint32_t)sh.npos != n) atomicOr(status, kErrInconsistent);
          sh.plen = n;
          const uint4 mine = make_uint4(j, noff, n, 0u);
          uint4 was = rec_load(W.orec + sh.row);
          sh.go = 0;
          for (int t = 0; t < kStepLimit; ++t) {  // each failure meets a smaller owner
            if (!rec_ok(was, W.pool_cap) || was.x == j) {
              atomicOr(status, kErrInconsistent);
              sh.go = 3;
              break;
            }
            if (was.x < j) {  // an earlier column claimed the row meanwhile: go on reducing
              sh.go = 1;
              break;
            }
            const uint4 got = rec_claim(W.orec + sh.row, was, mine);
            if (rec_same(got, was)) {
              sh.go = was.x == kNoOwner ? 0 : 2;
              if (sh.go == 2) {  // go on with the displaced column
                sh.j = was.x;
                sh.poff = was.y;
                sh.plen = was.z;
              }
              break;
            }
            was = got;
          }
        }
        __syncthreads();
        claimed = true;
        alive = sh.go == 1 || sh.go == 2;
      }
      t_longest = max(t_longest, (unsigned long long)plen);
      if (adds_here) atomicMax(&W.stats[12], (unsigned long long)adds_here);
      __syncthreads();
    }
    const uint32_t bad = *reinterpret_cast<const volatile uint32_t*>(status) &
                         (kErrPool | kErrRounds | kErrInconsistent | kErrEmptyColumn);
    if (__syncthreads_or(bad != 0u)) break;  // the set may hold leftovers: results are discarded
  }
  if (t_adds) {
    atomicAdd(&W.stats[11], t_adds);
    atomicAdd(&W.stats[6], t_merged);
  }
  if (tid == 0) {
    atomicAdd(&W.stats[13], t_rounds);
    atomicMax(&W.stats[7], t_longest);
    atomicMax(&W.stats[14], (unsigned long long)(clock64() - c_start));
  }
}

// Every row's owner is paired with it.
__global__ void k_d1_edges(int n1, D1Work W, int32_t* d1_edge, uint32_t* status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) W.stats[10] += W.stats[14] + W.stats[15];
  if (i >= n1) return;
  const uint32_t j = W.orec[i].x, ncols = (uint32_t)W.flags[1];
  if (j == kNoOwner || d1_failed(status)) return;
  if (j < ncols) d1_edge[W.cols[j]] = i;
  else atomicOr(status, kErrInconsistent);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
int d1_sms() {
  static std::atomic<int> sms[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  int n = dev >= 0 && dev < 64 ? sms[dev].load(std::memory_order_relaxed) : 0;
  if (n == 0) {
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (dev >= 0 && dev < 64) sms[dev].store(n, std::memory_order_relaxed);
  }
  return std::max(n, 1);
}

size_t d1_long_words(int n1) {
  if (long_window(n1) >= long_groups(n1)) return 0;
  return (size_t)d1_sms() * long_groups(n1) * 32;
}

void launch_d1_reduce(int n1, int n2, D1Work& W, PairOut& P, uint32_t* status, D1Ctl* ctl, cudaStream_t st) {
  if (n2 == 0 || n1 == 0) return;
  int dev = 0;
  cudaGetDevice(&dev);
  static std::atomic<bool> attr[64] = {};
  if (dev >= 0 && dev < 64 && !attr[dev].load(std::memory_order_acquire)) {
    cudaFuncSetAttribute(k_d1_long, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(kLongSmem - sizeof(LongShared)));
    attr[dev].store(true, std::memory_order_release);
  }
  const uint32_t cap = (uint32_t)std::min<int64_t>(std::max<int64_t>(get_knob(9), 0), kColCap);
  const int64_t cm = get_knob(12);
  const int max_adds = cm > 0 ? (int)std::min<int64_t>(cm, kColStepsMax) : kColSteps;
  const int window = long_window(n1);
  const size_t words = d1_long_words(n1);
  cudaMemsetAsync(ctl, 0, sizeof(D1Ctl), st);
  if (words) cudaMemsetAsync(W.hbits, 0, words * sizeof(uint32_t), st);
  k_d1_init<<<(n1 + 255) / 256, 256, 0, st>>>(n1, W); note_launch();
  bool listed = false;
  const int nb = n2 >= get_knob(5) ? cooperative_blocks((const void*)k_d1_reduce_grid, kUFT) : 0;
  if (nb > 0) {
    int handoff = (int)std::min<int64_t>(get_knob(6), 1 << 30);
    unsigned limit = (unsigned)std::min<int64_t>(std::max<int64_t>(get_knob(4), 1), 1u << 30);
    void* args[] = {&W, &n1, &ctl, &handoff, &limit, &status};
    listed = cooperative_launch((const void*)k_d1_reduce_grid, dim3(nb), dim3(kUFT), args, st) == cudaSuccess;
    if (!listed) cudaGetLastError();  // not launched: the warps take every column
  }
  const int sms = d1_sms();
  const int warps = std::min((n2 + kColWarps - 1) / kColWarps, sms * 4);
  k_d1_columns<<<warps, kColWarps * 32, 0, st>>>(W, n1, ctl, listed, cap, max_adds, status); note_launch();
  const size_t lsm = (size_t)window * 128 + 4 * (size_t)((long_groups(n1) + 31) / 32);
  k_d1_long<<<sms, kLT, lsm, st>>>(W, n1, ctl, window, status); note_launch();
  k_d1_edges<<<(n1 + 255) / 256, 256, 0, st>>>(n1, W, P.d1_edge, status); note_launch();
}

}  // namespace tsf
