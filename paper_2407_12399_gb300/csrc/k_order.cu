// k_order.cu -- incremental update of the vertex order (Section 2.1) after a
// gradient step that changed few values.  The vertices the step left alone
// keep their relative order, so the new order is the merge of the old order
// without the updated vertices and the updated vertices sorted by their new
// (value key, id):
//   a kept vertex at old position i lands at  i - #{updated u : rank(u) < i}
//                                               + #{updated u : key'(u) < key(i)}
//   the q-th updated vertex (by new key) at     q + #{kept vertices with key < key'(u)}.
// The old order's sorted keys (kept from the previous ordering) give the
// second count by a binary search, even though the updated vertices' old
// values are gone.
#include "../../include/tsf.h"
#include "tsf_kernels.cuh"

namespace tsf {

// The old ranks of the updated vertices as a bitmap over positions, and their
// new keys value_key << 32 | id in K (in the order of upd).
__global__ void k_order_mark(const uint32_t* __restrict__ upd, int nu, const float* __restrict__ f,
                             const uint32_t* __restrict__ rank, uint32_t* __restrict__ ubits,
                             unsigned long long* __restrict__ K, uint32_t* status) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < nu) {
    const uint32_t u = upd[q];
    const uint32_t r = __ldg(rank + u);
    const float x = __ldg(f + u);
    if (!isfinite(x)) atomicOr(status, kErrNaN);
    K[q] = ((unsigned long long)value_key(x) << 32) | u;
    atomicOr(ubits + (r >> 5), 1u << (r & 31));
  }
}

constexpr int kCntT = 1024;  // words per counting block

// ucnt[w] = set bits in ubits[blk*1024 .. w) for w's block blk, btot[blk] =
// the block's total (coalesced, one word per thread).
__global__ void __launch_bounds__(kCntT) k_order_count(const uint32_t* __restrict__ ubits, int64_t nw,
                                                       uint32_t* __restrict__ ucnt, uint32_t* __restrict__ btot) {
  __shared__ uint32_t wsum[kCntT / 32];
  const int64_t w = (int64_t)blockIdx.x * kCntT + threadIdx.x;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  uint32_t c = w < nw ? (uint32_t)__popc(__ldg(ubits + w)) : 0u;
  uint32_t inc = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[wi] = inc;
  __syncthreads();
  if (wi == 0) {
    uint32_t x = wsum[lane], xi = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t t = __shfl_up_sync(0xFFFFFFFFu, xi, o);
      if (lane >= o) xi += t;
    }
    wsum[lane] = xi - x;
    if (lane == 31) btot[blockIdx.x] = xi;
  }
  __syncthreads();
  if (w < nw) ucnt[w] = wsum[wi] + inc - c;
}

// B = K ascending, by rank counting: a block ranks 32 keys, one per lane, and
// each of its warps counts the smaller ones in its share of K (a broadcast
// load per step, no dependence between steps).  The keys are distinct, as the
// vertices are.  The last block also turns the counting blocks' totals into
// boff[b] = set bits before block b.  Bound by the n^2 comparisons.  A
// bitonic sort by one block took 46 us of the stage's 102 us for the 128^3
// filament field (about 3e3 keys); the stage now takes 63 us.
constexpr int kRankT = 256;
constexpr int kRankW = kRankT / 32;
__global__ void __launch_bounds__(kRankT) k_order_rank(const unsigned long long* __restrict__ K, int nu,
                                                       unsigned long long* __restrict__ B,
                                                       const uint32_t* __restrict__ btot, int nblk,
                                                       uint32_t* __restrict__ boff) {
  __shared__ int cnt[kRankW][32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (blockIdx.x == gridDim.x - 1) {
    uint32_t* part = reinterpret_cast<uint32_t*>(&cnt[0][0]);
    const int per = (nblk + kRankT - 1) / kRankT;
    const int b0 = min(tid * per, nblk), b1 = min(b0 + per, nblk);
    uint32_t mine = 0;
    for (int b = b0; b < b1; ++b) mine += btot[b];
    part[tid] = mine;
    __syncthreads();
    for (int o = 1; o < kRankT; o <<= 1) {  // inclusive scan of the runs' totals
      const uint32_t x = tid >= o ? part[tid - o] : 0u;
      __syncthreads();
      part[tid] += x;
      __syncthreads();
    }
    uint32_t run = part[tid] - mine;
    for (int b = b0; b < b1; ++b) {
      boff[b] = run;
      run += btot[b];
    }
    return;
  }
  const int q = blockIdx.x * 32 + lane;
  const unsigned long long k = q < nu ? __ldg(K + q) : 0ull;
  const int per = (nu + kRankW - 1) / kRankW;
  const int j1 = min((w + 1) * per, nu);
  int c = 0;
#pragma unroll 8
  for (int j = w * per; j < j1; ++j) c += __ldg(K + j) < k ? 1 : 0;
  cnt[w][lane] = c;
  __syncthreads();
  if (w == 0 && q < nu) {
    c = 0;
#pragma unroll
    for (int i = 0; i < kRankW; ++i) c += cnt[i][lane];
    B[c] = k;
  }
}

__device__ __forceinline__ int count_below(const unsigned long long* __restrict__ s, int n, unsigned long long x) {
  int lo = 0, hi = n;  // #{k : s[k] < x}, s ascending
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (__ldg(s + mid) < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}
// #{updated vertices with old rank < i}
__device__ __forceinline__ int updated_below(const uint32_t* __restrict__ ubits, const uint32_t* __restrict__ ucnt,
                                             const uint32_t* __restrict__ boff, int64_t i) {
  int64_t w = i >> 5;
  return (int)(__ldg(boff + (w >> 10)) + __ldg(ucnt + w) + __popc(__ldg(ubits + w) & ((1u << (i & 31)) - 1u)));
}

constexpr int kKeepT = 256, kKeepC = 16;  // threads, positions per lane
constexpr int kKeepTile = kKeepT * kKeepC;

// The new order.  The first blocks place the updated vertices, one thread
// each (a binary search of the old order, latency bound: it runs beside the
// copy below); in the others each lane walks kept positions i0, i0 + 32, ...
// and advances its count of smaller new keys (non-decreasing in i).
__global__ void __launch_bounds__(kKeepT) k_order_place(int64_t n, const uint32_t* __restrict__ order,
                                                        const uint32_t* __restrict__ skey,
                                                        const uint32_t* __restrict__ ubits,
                                                        const uint32_t* __restrict__ ucnt,
                                                        const uint32_t* __restrict__ boff, int nu,
                                                        const unsigned long long* __restrict__ B,
                                                        uint32_t* __restrict__ order2, uint32_t* __restrict__ skey2,
                                                        uint32_t* __restrict__ rank) {
  const int moved_blocks = (nu + kKeepT - 1) / kKeepT;
  if ((int)blockIdx.x < moved_blocks) {
    const int q = blockIdx.x * kKeepT + threadIdx.x;
    if (q >= nu) return;
    const unsigned long long key = B[q];
    int64_t lo = 0, hi = n;  // old positions whose (old key, id) is below key
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      const unsigned long long k = ((unsigned long long)__ldg(skey + mid) << 32) | __ldg(order + mid);
      if (k < key) lo = mid + 1;
      else hi = mid;
    }
    const int la = lo < n ? updated_below(ubits, ucnt, boff, lo) : nu;
    const uint32_t ni = (uint32_t)(q + lo - la);
    const uint32_t u = (uint32_t)key;
    order2[ni] = u;
    skey2[ni] = (uint32_t)(key >> 32);
    rank[u] = ni;
    return;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t i0 = (int64_t)(blockIdx.x - moved_blocks) * kKeepTile + (int64_t)w * (32 * kKeepC) + lane;
  if (i0 >= n) return;
  int b = count_below(B, nu, ((unsigned long long)__ldg(skey + i0) << 32) | __ldg(order + i0));
#pragma unroll 4
  for (int k = 0; k < kKeepC; ++k) {
    int64_t i = i0 + 32 * k;
    if (i >= n) break;
    uint32_t v = __ldg(order + i);
    uint32_t kk = __ldg(skey + i);
    if ((__ldg(ubits + (i >> 5)) >> (i & 31)) & 1u) continue;  // updated: placed by its own thread
    unsigned long long key = ((unsigned long long)kk << 32) | v;
    while (b < nu && __ldg(B + b) < key) ++b;
    uint32_t ni = (uint32_t)(i - updated_below(ubits, ucnt, boff, i) + b);
    order2[ni] = v;
    skey2[ni] = kk;
    rank[v] = ni;
  }
}

void vertex_order_incremental(const float* f, int64_t n, const uint32_t* upd, int nu, const uint32_t* order,
                              const uint32_t* skey, uint32_t* order2, uint32_t* skey2, uint32_t* rank,
                              uint32_t* ubits, uint32_t* ucnt, unsigned long long* B, uint32_t* status,
                              cudaStream_t st) {
  if (nu <= 0 || nu > kIncOrderMax) return;
  const int64_t nw = (n + 31) / 32;
  const int nblk = (int)((nw + kCntT - 1) / kCntT);
  uint32_t* btot = ucnt + nw;  // ucnt holds nw + 2 * nblk words
  uint32_t* boff = btot + nblk;
  unsigned long long* K = B + kIncOrderMax;
  cudaMemsetAsync(ubits, 0, sizeof(uint32_t) * (size_t)nw, st);
  k_order_mark<<<(nu + 255) / 256, 256, 0, st>>>(upd, nu, f, rank, ubits, K, status); note_launch();
  k_order_count<<<nblk, kCntT, 0, st>>>(ubits, nw, ucnt, btot); note_launch();
  k_order_rank<<<(nu + 31) / 32 + 1, kRankT, 0, st>>>(K, nu, B, btot, nblk, boff); note_launch();
  const int64_t place = (nu + kKeepT - 1) / kKeepT + (n + kKeepTile - 1) / kKeepTile;
  k_order_place<<<(unsigned)place, kKeepT, 0, st>>>(n, order, skey, ubits, ucnt, boff, nu, B, order2, skey2, rank);
  note_launch();
}

int64_t order_count_words(int64_t n) {
  const int64_t nw = (n + 31) / 32;
  return nw + 2 * ((nw + kCntT - 1) / kCntT);
}

}  // namespace tsf
