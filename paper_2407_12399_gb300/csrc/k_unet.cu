// k_unet.cu -- kernels of the learned warm start: a 3-level 3D U-Net
// (channels 16/32/64, 3x3x3 convolutions, bf16 storage, fp32 accumulation)
// whose forward and backward passes run here.  The paper has no learned
// component; the network only proposes a starting field that the solver of
// Algorithm 1 then refines.
//
// Activation layout ("chunk planes"): a tensor of C channels on an
// (lz, ly, lx) grid is C/8 planes of lz*ly*lx voxels x 8 bf16 channels,
//   act[c / 8][z][y][x][c % 8],
// so one voxel's 8 channels of a plane are one 16-byte row.  A concatenated
// input is just more planes of the same buffer.
//
// Convolution (forward, and the data gradient as a convolution with the
// flipped, transposed kernel) is an implicit GEMM on the tcgen05 tensor
// cores; k_conv_tc says how.

// Weight gradients, pooling, upsampling, the 1x1 head, the loss and Adam are
// bandwidth-bound and run on the CUDA cores.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "tsf_unet.cuh"

namespace tsf {
namespace unet {

// ---------------------------------------------------------------------------
// PTX wrappers (tcgen05, TMA, mbarrier)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase with the given parity; false after ~2^22 polls
// (seconds), so a kernel that would wait forever reports and returns.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 22); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (it > 64) __nanosleep(32);
  }
  return false;
}

// The same for a whole warp that goes on in step: the branch is warp-uniform.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 22); ++it) {
    if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) return true;
    if (it > 64) __nanosleep(32);
  }
  return false;
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor, no swizzle: start address, leading byte
// offset (between core matrices adjacent along K), stride byte offset
// (between core matrices adjacent along M or N), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr >> 4) & 0x3FFFu);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  return d;
}

// Instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, M x N.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(m >> 4) << 24);
}

// Issued by one elected lane; the whole warp calls them, with values that are
// the same in every lane, so that descriptors stay in uniform registers (from
// one lane of a diverged warp an MMA took about 150 cycles to issue).
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "elect.sync _|q, 0xFFFFFFFF;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xFFFFFFFF;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);  // .x = a (low half), .y = b
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void unpack8(const uint4& q, float* v) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(w[i] << 16);
    v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

__device__ __forceinline__ uint4 pack8(const float* v) {
  return make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                    pack_bf16x2(v[6], v[7]));
}

// q to two adjacent 16-byte rows, as one 32-byte store (p is 32-byte aligned).
__device__ __forceinline__ void store_twice(uint4* p, const uint4& q) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %1, %2, %3, %4};" ::"l"(p), "r"(q.x), "r"(q.y), "r"(q.z),
               "r"(q.w)
               : "memory");
}

// ---------------------------------------------------------------------------
// Convolution as an implicit GEMM on tcgen05
// ---------------------------------------------------------------------------
// A block computes tx x ty x tz output voxels.  For each pair of input planes
// (16 channels, one K step) it walks the tz + 2 input z-planes; TMA brings a
// plane's (ty + 2) x (tx + 2) voxels (zero outside the grid: the padding) as
// 16-byte rows, one after the other.  In the no-swizzle K-major operand layout
// 128 consecutive rows are an A tile, so a tile of 128 outputs (flattened with
// pitch tx + 2; the two halo columns of a row give outputs that nobody keeps)
// reads its (dy, dx) neighbours by a shift of the operand's start address: one
// load serves nine taps.  The three dz taps of an input plane go to three
// output planes, whose accumulators lie next to each other in TMEM, so the
// three weight matrices form one B operand of 3 x cout columns and one MMA
// does all three.
// A block per SM walks over tiles: one warp issues the loads (they run ahead
// into the next tile), two the MMAs (half of a tile's operand tiles each),
// eight turn accumulators into outputs
// while the other half of TMEM (256 columns) takes the next tile's MMAs.
// Weights that fit stay in shared memory for the whole launch.
// Bound: the A operand.  An MMA reads 4 KB of A (32 cycles of shared-memory
// bandwidth) and 96 x cout bytes of B, 32 + 3 x cout / 4 cycles in all, for
// 3 x cout / 2 cycles of math, so 16 output channels reach about half of the
// tensor rate.
// A single input plane (8 channels) takes two dx neighbours as its K step:
// the second K half is the first one shifted by one row.
constexpr int kConvEpiWarps = 8;
constexpr int kConvMmaWarps = 2;
constexpr int kConvThreads = (kConvEpiWarps + 1 + kConvMmaWarps) * 32;

struct ConvBars {
  uint64_t full_a[kConvStagesMax], empty_a[kConvStagesMax], full_b[kConvBSlotsMax], empty_b[kConvBSlotsMax];
  uint64_t tfull[2], tempty[2], done;
  uint32_t taddr;
  int gave_up, issued_a, issued_b;
  float bias[96], head[17];
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// The MMAs of one input plane: every (dy, dx) tap on kM operand tiles.
struct PlaneMmas {
  uint64_t a, b;         // operand descriptors of the first tile and tap
  uint32_t t0, tcols;    // accumulators of d = 0 and the distance of two tiles'
  uint32_t cout, pitch;
  int dlo, dhi;          // dz taps that stay in the tile
  bool first;            // first K step: output plane d = 2 starts its sums here
};

// dz taps d .. d + n - 1 of one (dy, dx) tap.
template <int kM>
__device__ __forceinline__ void issue_tap(const PlaneMmas& f, uint64_t ad, uint64_t bd, int d, int n, uint32_t acc) {
  const uint32_t idesc = instr_desc(128, n * static_cast<int>(f.cout));
  bd += static_cast<uint32_t>(d) * f.cout;
  const uint32_t td = f.t0 + static_cast<uint32_t>(d) * f.cout;
#pragma unroll
  for (int m = 0; m < kM; ++m) mma_bf16(td + m * f.tcols, ad + m * 128u, bd, idesc, acc);
}

// Unrolled: an MMA of 48 columns takes 44 cycles, and the loop has to issue
// one in as many.  256^3 voxels, 16 to 16 channels: rolled over taps and tiles
// 1046 us, over tiles only 645, unrolled 437 (66 cycles per MMA: about 72 per
// tap and 49 per tile); two warps that share the tiles take the whole layer
// from 479 to 403 us.
template <bool kSingle, int kM>
__device__ __forceinline__ void issue_plane(const PlaneMmas& f) {
  constexpr int kDx = kSingle ? 2 : 3;
  const int n = f.dhi - f.dlo + 1;
  const bool upper = f.dhi == 2 && f.dlo < 2;                       // d = 2 next to others
  const bool wide = upper && n * static_cast<int>(f.cout) > 256;  // N <= 256
  const bool split = wide || (f.first && upper);
  issue_tap<kM>(f, f.a, f.b, f.dlo, split ? 2 - f.dlo : n, f.first && f.dlo == 2 ? 0u : 1u);
  if (split) issue_tap<kM>(f, f.a, f.b, 2, 1, f.first ? 0u : 1u);
  if (!wide) {
#pragma unroll
    for (int t = 1; t < 3 * kDx; ++t)
      issue_tap<kM>(f, f.a + static_cast<uint32_t>(t / kDx) * f.pitch + t % kDx,
                    f.b + static_cast<uint32_t>(t) * (6u * f.cout), f.dlo, n, 1u);
  } else {
#pragma unroll 1
    for (int t = 1; t < 3 * kDx; ++t) {
      const uint64_t ad = f.a + static_cast<uint32_t>(t / kDx) * f.pitch + t % kDx;
      const uint64_t bd = f.b + static_cast<uint32_t>(t) * (6u * f.cout);
      issue_tap<kM>(f, ad, bd, f.dlo, 2 - f.dlo, 1u);
      issue_tap<kM>(f, ad, bd, 2, 1, 1u);
    }
  }
}

template <bool kSingle>
__global__ void __launch_bounds__(kConvThreads, 1) k_conv_tc(const __grid_constant__ CUtensorMap in_map, ConvArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ ConvBars sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const ConvPlan& p = a.plan;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* sb0 = smem + p.stages * p.a_bytes;
  volatile int* gave_up = &sh.gave_up;
  const int tiles = p.tiles_x * p.tiles_y * p.tiles_z;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&sh.full_a[s], 1);
      mbar_init(&sh.empty_a[s], kConvMmaWarps);
    }
    for (int s = 0; s < p.b_slots; ++s) {
      mbar_init(&sh.full_b[s], 1);
      mbar_init(&sh.empty_b[s], kConvMmaWarps);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sh.tfull[s], kConvMmaWarps);
      mbar_init(&sh.tempty[s], kConvEpiWarps);
    }
    mbar_init(&sh.done, kConvMmaWarps);
    sh.gave_up = 0;
    sh.issued_a = 0;
    sh.issued_b = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (a.mode != kConvDgrad && threadIdx.x < a.cout) sh.bias[threadIdx.x] = a.bias[threadIdx.x];
  if (a.mode == kConvHead && threadIdx.x < 17) sh.head[threadIdx.x] = a.head[threadIdx.x];
  __syncwarp();
  if (warp == 0) {  // TMEM accumulators: two halves of p.tmem_cols / 2 fp32 columns x 128 lanes
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.taddr)),
                 "r"(static_cast<uint32_t>(p.tmem_cols))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t taddr = __shfl_sync(0xFFFFFFFFu, sh.taddr, 0);
  const int role = __shfl_sync(0xFFFFFFFFu, warp, 0);  // the same value, known to be warp-uniform
  const uint32_t thalf = static_cast<uint32_t>(p.tmem_cols / 2);

  if (role == kConvEpiWarps && lane == 0) {
    // producer: per tile and K step the weights (once, if all stay resident),
    // then the input planes
    int it = 0, bt = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      const int x0 = (tile % p.tiles_x) * p.tx, y0 = ((tile / p.tiles_x) % p.tiles_y) * p.ty,
                z0 = tile / (p.tiles_x * p.tiles_y) * p.tz;
      for (int kk = 0; kk < p.ksteps && ok; ++kk) {
        if (!p.b_resident || bt < p.ksteps) {
          const int bs = bt % p.b_slots;
          if (bt >= p.b_slots && !mbar_wait(&sh.empty_b[bs], ((bt / p.b_slots) - 1) & 1)) ok = false;
          if (!ok || *gave_up) {
            ok = false;
            break;
          }
          mbar_expect_tx(&sh.full_b[bs], p.b_bytes);
          bulk_load(sb0 + bs * p.b_bytes, a.wpack + static_cast<size_t>(kk) * (p.b_bytes / 2), p.b_bytes,
                    &sh.full_b[bs]);
          sh.issued_b = ++bt;
        }
        for (int zi = 0; zi < p.tz + 2; ++zi, ++it) {
          const int slot = it % p.stages;
          if (it >= p.stages && !mbar_wait(&sh.empty_a[slot], ((it / p.stages) - 1) & 1)) ok = false;
          if (!ok || *gave_up) {
            ok = false;
            break;
          }
          mbar_expect_tx(&sh.full_a[slot], p.a_tx);
          tma_load_4d(smem + slot * p.a_bytes, &in_map, 2 * (x0 - 1), y0 - 1, z0 - 1 + zi, kk * p.kchunks,
                      &sh.full_a[slot]);
          sh.issued_a = it + 1;
        }
      }
    }
    if (!ok) {
      if (!*gave_up) atomicOr(a.status, kUnetErrSpin);
      *gave_up = 1;
    }
  } else if (role > kConvEpiWarps) {
    // MMA issuers: descriptors are built once per plane and advanced by adds to
    // their address fields (in units of 16 bytes)
    const int m0 = role == kConvEpiWarps + 1 ? 0 : (p.mtiles + 1) / 2;
    const int nm = role == kConvEpiWarps + 1 ? (p.mtiles + 1) / 2 : p.mtiles / 2;
    const uint32_t a_lbo = kSingle ? 16u : static_cast<uint32_t>((p.ty + 2) * p.pitch) * 16u;
    const uint32_t b_lbo = static_cast<uint32_t>(3 * a.cout) * 16u;
    const uint32_t tcols = static_cast<uint32_t>(p.tz * a.cout), cout = static_cast<uint32_t>(a.cout);
    int it = 0, bt = 0, nt = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++nt) {
      const int half = nt & 1;
      if (nt >= 2 && !mbar_wait_warp(&sh.tempty[half], ((nt >> 1) - 1) & 1)) {
        ok = false;
        break;
      }
      tc_fence_after();
      for (int kk = 0; kk < p.ksteps && ok; ++kk, ++bt) {
        const int bs = bt % p.b_slots;
        if ((!p.b_resident || nt == 0) &&
            !mbar_wait_warp(&sh.full_b[bs], p.b_resident ? 0 : (bt / p.b_slots) & 1)) {
          ok = false;
          break;
        }
        const uint64_t bbase = smem_desc(smem_u32(sb0 + bs * p.b_bytes), b_lbo, 128u);
        for (int zi = 0; zi < p.tz + 2; ++zi, ++it) {
          const int slot = it % p.stages;
          if (!mbar_wait_warp(&sh.full_a[slot], (it / p.stages) & 1) || __any_sync(0xFFFFFFFFu, *gave_up)) {
            ok = false;
            break;
          }
          tc_fence_after();
          // input plane zi feeds output planes zi - 2 + d (dz tap 2 - d)
          const int dlo = max(0, 2 - zi), dhi = min(2, p.tz + 1 - zi);
          const uint64_t abase = smem_desc(smem_u32(smem + slot * p.a_bytes), a_lbo, 128u);
          const PlaneMmas f{abase + static_cast<uint32_t>(m0) * 128u, bbase,
                            taddr + (half ? thalf : 0u) + static_cast<uint32_t>(m0) * tcols +
                                static_cast<uint32_t>((zi - 2) * a.cout),
                            tcols, cout, static_cast<uint32_t>(p.pitch), dlo, dhi, kk == 0};
          if (nm == 1) issue_plane<kSingle, 1>(f);
          else if (nm == 2) issue_plane<kSingle, 2>(f);
          mma_commit(&sh.empty_a[slot]);  // the slot is free once these MMAs have read it
        }
        if (ok && !p.b_resident) mma_commit(&sh.empty_b[bs]);
      }
      if (ok) mma_commit(&sh.tfull[half]);
    }
    if (!ok && lane == 0) {
      if (!*gave_up) atomicOr(a.status, kUnetErrSpin);
      *gave_up = 1;
    }
    __syncwarp();
    mma_commit(&sh.done);  // every MMA issued above is complete before TMEM is freed
    mbar_wait(&sh.done, 0);
  } else if (role < kConvEpiWarps) {
    // epilogue: warp w reads TMEM lanes 32 * (w % 4) ..; the two warps of a
    // lane quarter take every other output row of the tile
    const size_t nv = static_cast<size_t>(a.lx) * a.ly * a.lz;
    const uint32_t tlane = static_cast<uint32_t>((warp & 3) * 32) << 16;
    int nt = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++nt) {
      const int x0 = (tile % p.tiles_x) * p.tx, y0 = ((tile / p.tiles_x) % p.tiles_y) * p.ty,
                z0 = tile / (p.tiles_x * p.tiles_y) * p.tz;
      const int half = nt & 1;
      const bool ready = mbar_wait(&sh.tfull[half], (nt >> 1) & 1);
      if (__any_sync(0xFFFFFFFFu, !ready || *gave_up)) {
        if (lane == 0) {
          if (!*gave_up) atomicOr(a.status, kUnetErrSpin);
          *gave_up = 1;
        }
        break;
      }
      tc_fence_after();
      const uint32_t tbase = taddr + (half ? thalf : 0u) + tlane;
      int turn = warp >> 2;
      for (int m = 0; m < p.mtiles; ++m) {
        const int q = m * 128 + (warp & 3) * 32 + lane;  // flattened position in the tile's planes
        const int yy = q / p.pitch, xx = q - yy * p.pitch;
        const int x = x0 + xx, y = y0 + yy;
        const bool in_xy = xx < p.tx && yy < p.ty && x < a.lx && y < a.ly;
        for (int zo = 0; zo < p.tz; ++zo, turn ^= 1) {
          const int z = z0 + zo;
          if (turn || z >= a.lz) continue;
          const size_t vox = (static_cast<size_t>(z) * a.ly + y) * a.lx + x;
          const uint32_t tcol = tbase + static_cast<uint32_t>((m * p.tz + zo) * a.cout);
          float head = 0.0f;
          for (int c16 = 0; c16 < a.cout / 16; ++c16) {
            float v[16];
            __syncwarp();
            tmem_ld16(tcol + static_cast<uint32_t>(c16 * 16), v);  // warp-wide
            if (!in_xy) continue;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int c8 = 2 * c16 + h;
              float* w = v + 8 * h;
              if (a.mode == kConvDgrad) {  // masked by the ReLU of the activation it flows into
                if (a.mask) {
                  float mk[8];
                  unpack8(reinterpret_cast<const uint4*>(a.mask)[(a.mask_plane0 + c8) * nv + vox], mk);
#pragma unroll
                  for (int i = 0; i < 8; ++i) w[i] = mk[i] > 0.0f ? w[i] : 0.0f;
                }
                reinterpret_cast<uint4*>(a.out)[(a.out_plane0 + c8) * nv + vox] = pack8(w);
                continue;
              }
#pragma unroll
              for (int i = 0; i < 8; ++i) w[i] = fmaxf(w[i] + sh.bias[c8 * 8 + i], 0.0f);
              const uint4 o = pack8(w);
              if (a.mode == kConvHead) {  // the 1x1 head on the stored (bf16) values
                float u[8];
                unpack8(o, u);
#pragma unroll
                for (int i = 0; i < 8; ++i) head = fmaf(u[i], sh.head[c8 * 8 + i], head);
              } else if (a.up) {  // nearest x2 upsampling: the voxel's 2x2x2 block of the fine grid
                const int fx = a.lx * 2, fy = a.ly * 2;
                const size_t fnv = nv * 8;
                uint4* base = reinterpret_cast<uint4*>(a.out) + (a.out_plane0 + c8) * fnv;
#pragma unroll
                for (int k = 0; k < 4; ++k)  // two voxels along x per store
                  store_twice(base + (static_cast<size_t>(2 * z + (k >> 1)) * fy + (2 * y + (k & 1))) * fx + 2 * x, o);
              } else {
                reinterpret_cast<uint4*>(a.out)[(a.out_plane0 + c8) * nv + vox] = o;
              }
            }
          }
          if (a.mode == kConvHead && in_xy) {
            const float r = __bfloat162float(__float2bfloat16_rn(head + sh.head[16]));
            a.g0[vox] = a.f[vox] + r;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.tempty[half]);
    }
  }
  __syncthreads();
  // after giving up, wait (bounded) for the copies still in flight before the
  // shared memory they target is released
  if (threadIdx.x == 0 && *gave_up) {
    for (int s = max(0, sh.issued_a - p.stages); s < sh.issued_a; ++s)
      mbar_wait(&sh.full_a[s % p.stages], (s / p.stages) & 1);
    for (int s = max(0, sh.issued_b - p.b_slots); s < sh.issued_b; ++s)
      mbar_wait(&sh.full_b[s % p.b_slots], (s / p.b_slots) & 1);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                 "r"(static_cast<uint32_t>(p.tmem_cols))
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Bandwidth-bound layers on the CUDA cores
// ---------------------------------------------------------------------------
// Network input: plane 0 = (f, tau, 0, ..., 0) rounded to bf16.
__global__ void k_pack_input(const float* __restrict__ f, float tau, int64_t nv, uint4* __restrict__ x) {
  const int64_t v = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (v >= nv) return;
  const float c[8] = {f[v], tau, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  x[v] = pack8(c);
}

// 2x2x2 average pooling of `planes` planes (fine grid lx, ly, lz).
__global__ void k_avgpool(const uint4* __restrict__ in, int in_plane0, int planes, int lx, int ly, int lz,
                          uint4* __restrict__ out) {
  const int cx = lx / 2, cy = ly / 2, cz = lz / 2;
  const int64_t cnv = static_cast<int64_t>(cx) * cy * cz, fnv = static_cast<int64_t>(lx) * ly * lz;
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= cnv * planes) return;
  const int p = static_cast<int>(i / cnv);
  const int64_t v = i % cnv;
  const int x = static_cast<int>(v % cx), y = static_cast<int>((v / cx) % cy), z = static_cast<int>(v / (static_cast<int64_t>(cx) * cy));
  float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int k = 0; k < 8; ++k) {
    const int64_t fv = (static_cast<int64_t>(2 * z + (k >> 2)) * ly + 2 * y + ((k >> 1) & 1)) * lx + 2 * x + (k & 1);
    float t[8];
    unpack8(in[(in_plane0 + p) * fnv + fv], t);
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] += t[c];
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] *= 0.125f;
  out[p * cnv + v] = pack8(acc);
}

// Backward of "upsample, then concatenate": the gradient of the coarse
// activation is the sum of its 2x2x2 fine gradients, masked by its ReLU.
// g: fine gradient planes [g_plane0, g_plane0 + planes); act: the coarse
// activation (read through the upsampled copy: any of its 8 fine voxels).
__global__ void k_upsample_back(const uint4* __restrict__ g, int g_plane0, int planes, int lx, int ly, int lz,
                                const uint4* __restrict__ act_up, int act_plane0, uint4* __restrict__ out) {
  const int cx = lx / 2, cy = ly / 2, cz = lz / 2;
  const int64_t cnv = static_cast<int64_t>(cx) * cy * cz, fnv = static_cast<int64_t>(lx) * ly * lz;
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= cnv * planes) return;
  const int p = static_cast<int>(i / cnv);
  const int64_t v = i % cnv;
  const int x = static_cast<int>(v % cx), y = static_cast<int>((v / cx) % cy), z = static_cast<int>(v / (static_cast<int64_t>(cx) * cy));
  float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  int64_t fv0 = 0;
  for (int k = 0; k < 8; ++k) {
    const int64_t fv = (static_cast<int64_t>(2 * z + (k >> 2)) * ly + 2 * y + ((k >> 1) & 1)) * lx + 2 * x + (k & 1);
    if (k == 0) fv0 = fv;
    float t[8];
    unpack8(g[(g_plane0 + p) * fnv + fv], t);
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] += t[c];
  }
  float a[8];
  unpack8(act_up[(act_plane0 + p) * fnv + fv0], a);
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = a[c] > 0.0f ? acc[c] : 0.0f;
  out[p * cnv + v] = pack8(acc);
}

// Gradient of a skip activation s (fine grid): its share from the
// concatenation plus the average-pooling backward of the coarse gradient gp,
// masked by s's ReLU.
__global__ void k_skip_back(const uint4* __restrict__ gs, int gs_plane0, const uint4* __restrict__ gp,
                            const uint4* __restrict__ s, int s_plane0, int planes, int lx, int ly, int lz,
                            uint4* __restrict__ out) {
  const int64_t fnv = static_cast<int64_t>(lx) * ly * lz;
  const int cx = lx / 2, cy = ly / 2;
  const int64_t cnv = fnv / 8;
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= fnv * planes) return;
  const int p = static_cast<int>(i / fnv);
  const int64_t v = i % fnv;
  const int x = static_cast<int>(v % lx), y = static_cast<int>((v / lx) % ly), z = static_cast<int>(v / (static_cast<int64_t>(lx) * ly));
  const int64_t cv = (static_cast<int64_t>(z / 2) * cy + y / 2) * cx + x / 2;
  float a[8], b[8], m[8];
  unpack8(gs[(gs_plane0 + p) * fnv + v], a);
  unpack8(gp[p * cnv + cv], b);
  unpack8(s[(s_plane0 + p) * fnv + v], m);
#pragma unroll
  for (int c = 0; c < 8; ++c) a[c] = m[c] > 0.0f ? a[c] + b[c] * 0.125f : 0.0f;
  out[p * fnv + v] = pack8(a);
}

// Head, backward for the loss mean((g0 - g)^2): per voxel gg = 2 (g0 - g) / nv;
// the u1 gradient gg * w masked by u1's ReLU; block partial sums (fp64) of
// the loss, of gg and of gg * u1[c] (the head's bias and weight gradients).
__global__ void __launch_bounds__(256) k_head_backward(const uint4* __restrict__ u1, const float* __restrict__ hw,
                                                       int64_t nv, const float* __restrict__ f,
                                                       const float* __restrict__ g, uint4* __restrict__ gz,
                                                       double* __restrict__ partial) {
  __shared__ double red[18][8];
  const float hb = hw[16];
  const int64_t v = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  double acc[18];
#pragma unroll
  for (int k = 0; k < 18; ++k) acc[k] = 0.0;
  if (v < nv) {
    float a[16];
    unpack8(u1[v], a);
    unpack8(u1[nv + v], a + 8);
    float r = 0.0f;
#pragma unroll
    for (int c = 0; c < 16; ++c) r = fmaf(a[c], hw[c], r);
    r = __bfloat162float(__float2bfloat16_rn(r + hb));
    const float d = (f[v] + r) - g[v];
    const float gg = 2.0f * d / static_cast<float>(nv);
    acc[0] = static_cast<double>(d) * d;
    acc[1] = gg;
    float o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      acc[2 + c] = static_cast<double>(gg) * a[c];
      o[c] = a[c] > 0.0f ? gg * hw[c] : 0.0f;
    }
    gz[v] = pack8(o);
    gz[nv + v] = pack8(o + 8);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 18; ++k) {
    double x = acc[k];
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    if (lane == 0) red[k][w] = x;
  }
  __syncthreads();
  if (threadIdx.x < 18) {
    double x = 0.0;
    for (int i = 0; i < 8; ++i) x += red[threadIdx.x][i];
    partial[static_cast<int64_t>(blockIdx.x) * 18 + threadIdx.x] = x;
  }
}

// Sums the head's block partials in block order: out[0] = loss (mean),
// grad[hw_off + c] = sum gg u1[c], grad[hb_off] = sum gg.
__global__ void k_head_reduce(const double* __restrict__ partial, int nblocks, int64_t nv, double* __restrict__ loss,
                              float* __restrict__ grad, int64_t hw_off, int64_t hb_off) {
  const int k = threadIdx.x;
  if (k >= 18) return;
  double s = 0.0;
  for (int b = 0; b < nblocks; ++b) s += partial[static_cast<int64_t>(b) * 18 + k];
  if (k == 0) *loss = s / static_cast<double>(nv);
  else if (k == 1) grad[hb_off] = static_cast<float>(s);
  else grad[hw_off + (k - 2)] = static_cast<float>(s);
}

// Weight gradient of one convolution: gw[o][c][tap] = sum over voxels p of
// gz[o][p] x[c][p + tap - 1] (zero outside the grid), gb[o] = sum gz[o][p].
// Block (tap, chunk of kWgV voxels in linear order); each thread owns a
// 4 (o) x 4 (c) register tile and a share of the voxels; partial sums per
// block, reduced in block order by k_wgrad_reduce (deterministic).
constexpr int kWgV = 64;     // voxels staged in shared memory at a time
constexpr int kWgChunk = 1024;  // voxels per block

__global__ void __launch_bounds__(256) k_wgrad(const uint4* __restrict__ x, int x_plane0, int cin,
                                               const uint4* __restrict__ gz, int cout, int lx, int ly, int lz,
                                               float* __restrict__ partial) {
  extern __shared__ float wsm[];
  float* sg = wsm;                    // [cout][kWgV]
  float* sx = wsm + cout * kWgV;      // [cin][kWgV]
  float* sred = sx + cin * kWgV;      // reduction across voxel groups
  const int tap = blockIdx.y;
  const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
  const int64_t nv = static_cast<int64_t>(lx) * ly * lz;
  const int64_t v0 = static_cast<int64_t>(blockIdx.x) * kWgChunk;
  const int to = cout / 4, tc = cin / 4, ntile = to * tc;
  const int groups = max(1, 256 / ntile);  // voxel groups sharing the tiles
  const int tid = threadIdx.x;
  const int tile = tid % ntile, grp = tid / ntile;
  const bool active = tid < ntile * groups;
  const int o0 = (tile / tc) * 4, c0 = (tile % tc) * 4;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  for (int64_t vb = v0; vb < v0 + kWgChunk && vb < nv; vb += kWgV) {
    __syncthreads();
    // stage gz (cout planes) and the tap-shifted x (cin planes) as fp32
    for (int i = tid; i < (cout / 8) * kWgV; i += 256) {
      const int p = i / kWgV, k = i % kWgV;
      const int64_t v = vb + k;
      float t[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      if (v < nv) unpack8(gz[p * nv + v], t);
#pragma unroll
      for (int c = 0; c < 8; ++c) sg[(p * 8 + c) * kWgV + k] = t[c];
    }
    for (int i = tid; i < (cin / 8) * kWgV; i += 256) {
      const int p = i / kWgV, k = i % kWgV;
      const int64_t v = vb + k;
      float t[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      if (v < nv) {
        const int vx = static_cast<int>(v % lx) + dx, vy = static_cast<int>((v / lx) % ly) + dy,
                  vz = static_cast<int>(v / (static_cast<int64_t>(lx) * ly)) + dz;
        if (vx >= 0 && vx < lx && vy >= 0 && vy < ly && vz >= 0 && vz < lz)
          unpack8(x[(x_plane0 + p) * nv + (static_cast<int64_t>(vz) * ly + vy) * lx + vx], t);
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) sx[(p * 8 + c) * kWgV + k] = t[c];
    }
    __syncthreads();
    if (active) {
      for (int k = grp; k < kWgV; k += groups) {
        float go[4], xc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) go[i] = sg[(o0 + i) * kWgV + k];
#pragma unroll
        for (int j = 0; j < 4; ++j) xc[j] = sx[(c0 + j) * kWgV + k];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(go[i], xc[j], acc[i][j]);
      }
    }
  }
  // combine the voxel groups (fixed order), then write the block's partial
  __syncthreads();
  float* out = partial + (static_cast<int64_t>(tap) * gridDim.x + blockIdx.x) * cout * cin;
  for (int g = 0; g < groups; ++g) {
    if (active && grp == g) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float* p = &sred[(o0 + i) * cin + c0 + j];
          *p = (g == 0 ? 0.0f : *p) + acc[i][j];
        }
    }
    __syncthreads();
  }
  for (int i = tid; i < cout * cin; i += 256) out[i] = sred[i];
}

// gw in the reference layout (cout, cin_real, 3, 3, 3) = sum over blocks of
// the partials, in block order.
__global__ void k_wgrad_reduce(const float* __restrict__ partial, int nblk, int cout, int cin, int cin_real,
                               float* __restrict__ gw) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // over 27 * cout * cin_real
  if (i >= 27 * cout * cin_real) return;
  const int tap = i % 27, c = (i / 27) % cin_real, o = i / (27 * cin_real);
  const float* p = partial + static_cast<int64_t>(tap) * nblk * cout * cin + o * cin + c;
  float s = 0.0f;
  for (int b = 0; b < nblk; ++b) s += p[static_cast<int64_t>(b) * cout * cin];
  gw[i] = s;
}

// gb[o] = sum over voxels of gz[o]: block partials, then an ordered sum.
__global__ void __launch_bounds__(256) k_bias_partial(const uint4* __restrict__ gz, int cout, int64_t nv,
                                                      float* __restrict__ partial) {
  __shared__ float red[8][96];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t v0 = static_cast<int64_t>(blockIdx.x) * 2048;
  for (int p = 0; p < cout / 8; ++p) {
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t v = v0 + threadIdx.x; v < v0 + 2048 && v < nv; v += 256) {
      float t[8];
      unpack8(gz[p * nv + v], t);
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[c] += t[c];
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float x = acc[c];
      for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
      if (lane == 0) red[w][p * 8 + c] = x;
    }
  }
  __syncthreads();
  if (threadIdx.x < cout) {
    float s = 0.0f;
    for (int i = 0; i < 8; ++i) s += red[i][threadIdx.x];
    partial[static_cast<int64_t>(blockIdx.x) * cout + threadIdx.x] = s;
  }
}

__global__ void k_bias_reduce(const float* __restrict__ partial, int nblk, int cout, float* __restrict__ gb) {
  const int o = threadIdx.x;
  if (o >= cout) return;
  float s = 0.0f;
  for (int b = 0; b < nblk; ++b) s += partial[static_cast<int64_t>(b) * cout + o];
  gb[o] = s;
}

// Weights of one layer from the fp32 master copy (reference layout
// (cout, cin_real, 3, 3, 3)) into the bf16 B operand of k_conv_tc:
// pack[K step][tap][K half][d * n_out + o][8], d = 0..2 for the dz tap 2 - d.
// Two input planes make a K step of nine (dy, dx) taps; a single one makes a
// K step of three dy times the dx pairs (0, 1) and (-, 2).  The data-gradient
// packing transposes and flips: B[o'][c'][tap] = w[c'][o'][26 - tap] (o' over
// the forward inputs, c' over its outputs).
__global__ void k_pack_weights(const float* __restrict__ w, int cout_f, int cin_real, int cin_pad, int transpose,
                               int64_t total, __nv_bfloat16* __restrict__ pack) {
  const int n_out = transpose ? cin_pad : cout_f;   // N of the GEMM
  const int n_in = transpose ? cout_f : cin_pad;    // input channels of the GEMM
  const bool single = n_in == 8;
  const int taps = single ? 6 : 9;
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= total) return;
  const int e = static_cast<int>(i % 8);
  const int n = static_cast<int>((i / 8) % (3 * n_out));
  const int half = static_cast<int>((i / (24 * n_out)) % 2);
  const int t = static_cast<int>((i / (48 * n_out)) % taps);
  const int kk = static_cast<int>(i / (static_cast<int64_t>(48) * n_out * taps));
  const int o = n % n_out, dz = 2 - n / n_out;
  const int dy = single ? t >> 1 : t / 3, dx = single ? (t & 1) + half : t % 3;
  const int ci = single ? e : (kk * 2 + half) * 8 + e;
  const int tap = (dz * 3 + dy) * 3 + dx;
  float val = 0.0f;
  if (!(single && (t & 1) && half == 0)) {  // dx = 1 is in the first pair
    if (!transpose) {
      if (ci < cin_real) val = w[(static_cast<int64_t>(o) * cin_real + ci) * 27 + tap];
    } else {  // GEMM output o = forward input channel, GEMM input ci = forward output channel
      if (o < cin_real) val = w[(static_cast<int64_t>(ci) * cin_real + o) * 27 + (26 - tap)];
    }
  }
  pack[i] = __float2bfloat16_rn(val);
}

// Biases and head weights rounded to bf16 (kept as fp32 values).
__global__ void k_round_bf16(const float* __restrict__ in, int64_t n, float* __restrict__ out) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i < n) out[i] = __bfloat162float(__float2bfloat16_rn(in[i]));
}

// Adam (Kingma & Ba, Algorithm 1) on the fp32 master parameters; bc1 and bc2
// are 1 - beta1^t and 1 - beta2^t.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float beta1, float beta2, float eps, float bc1,
                       float bc2) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = beta1 * m[i] + (1.0f - beta1) * gi;
  const float vi = beta2 * v[i] + (1.0f - beta2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float mh = mi / bc1, vh = vi / bc2;
  p[i] -= lr * mh / (sqrtf(vh) + eps);
}

// Planes (bf16) -> fp32 in the reference layout (C, z, y, x), `c_real`
// channels of the planes starting at plane0.
__global__ void k_unpack_planes(const uint4* __restrict__ in, int plane0, int c_real, int64_t nv,
                                float* __restrict__ out) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= nv * c_real) return;
  const int c = static_cast<int>(i / nv);
  const int64_t v = i % nv;
  float t[8];
  unpack8(in[(plane0 + c / 8) * nv + v], t);
  out[i] = t[c % 8];
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
namespace {
// cuTensorMapEncodeTiled, looked up through the runtime (no link to libcuda)
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
bool g_attr_set[64] = {};
}  // namespace

// Planes as (2 * lx, ly, lz, chunks) 8-byte elements, two per voxel, so that a
// row of voxels is one run of a box's innermost dimension (at most 256
// elements): TMA takes three to five cycles per innermost run, and with
// 16-byte runs it, not the tensor cores, set the time.  x coordinates are
// multiples of two elements, 16 bytes.
int encode_planes_map(CUtensorMap* map, const void* base, int lx, int ly, int lz, int chunks, int bx, int by,
                      int bchunks) {
  if (!g_encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
      return -1;
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  }
  const uint64_t nv = static_cast<uint64_t>(lx) * ly * lz;
  cuuint64_t dims[4] = {2 * static_cast<cuuint64_t>(lx), static_cast<cuuint64_t>(ly), static_cast<cuuint64_t>(lz),
                        static_cast<cuuint64_t>(chunks)};
  cuuint64_t strides[3] = {16ull * lx, 16ull * lx * ly, 16ull * nv};
  cuuint32_t box[4] = {2 * static_cast<cuuint32_t>(bx), static_cast<cuuint32_t>(by), 1,
                       static_cast<cuuint32_t>(bchunks)};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, const_cast<void*>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -1;
}

// Tile of a convolution: the shape of least estimated time, in cycles.  An MMA
// of n dz taps takes 32 + n x cout / 4 (its operands' shared-memory reads); a
// tile's tz + 2 planes feed one, two or three output planes each; loads and
// epilogue run beside the MMAs.  Small grids take smaller tiles so that every
// SM has one.
ConvPlan plan_conv(int lx, int ly, int lz, int chunks, int cout) {
  ConvPlan best{};
  double best_time = 0.0;
  const int kchunks = chunks == 1 ? 1 : 2;
  const int ksteps = (chunks + 1) / 2, taps = chunks == 1 ? 6 : 9;
  const int b_bytes = taps * 2 * 3 * cout * 16;
  const int room = static_cast<int>(kConvSmem) - kConvSmemFixed;
  const int min_x = (lx + kConvTx - 1) / kConvTx;
  for (int tiles_x = min_x; tiles_x <= min_x + 3; ++tiles_x) {
    const int tx = (lx + tiles_x - 1) / tiles_x, pitch = tx + 2;
    for (int tz = 1; tz <= 16; ++tz) {
      for (int mt = 1; mt <= 4 && mt * tz * cout <= 256; ++mt) {
        if (mt * 128 < tx) continue;
        int ty = std::min((mt * 128 - tx) / pitch + 1, ly);
        const int tiles_y = (ly + ty - 1) / ty;
        ty = (ly + tiles_y - 1) / tiles_y;
        if (ty + 2 > 256) continue;
        ConvPlan p{};
        p.tx = tx;
        p.ty = ty;
        p.tz = tz;
        p.pitch = pitch;
        p.mtiles = ((ty - 1) * pitch + tx + 127) / 128;
        p.tiles_x = tiles_x;
        p.tiles_y = tiles_y;
        p.tiles_z = (lz + tz - 1) / tz;
        p.kchunks = kchunks;
        p.ksteps = ksteps;
        p.taps = taps;
        p.a_tx = (ty + 2) * pitch * 16 * kchunks;
        p.a_bytes = (p.a_tx + 127) / 128 * 128;
        p.b_bytes = b_bytes;
        p.b_resident = ksteps <= kConvBSlotsMax && room - ksteps * b_bytes >= 4 * p.a_bytes;
        p.b_slots = p.b_resident ? ksteps : room - 2 * b_bytes >= 4 * p.a_bytes ? 2 : 1;
        p.stages = std::min((room - p.b_slots * b_bytes) / p.a_bytes, kConvStagesMax);
        if (p.stages < 2) continue;
        const int cols = 2 * p.mtiles * tz * cout;
        p.tmem_cols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
        double mma = 0.0;
        for (int zi = 0; zi < tz + 2; ++zi)
          mma += 32.0 + (std::min(2, tz + 1 - zi) - std::max(0, 2 - zi) + 1) * cout / 4.0;
        // ... or what its issue takes: about 72 cycles per tap, 49 per tile
        mma = std::max(mma * p.mtiles, (tz + 2) * (72.0 + 49.0 * ((p.mtiles + 1) / 2))) * ksteps * taps;
        const double loads = ksteps * (tz + 2) * p.a_tx / 30.0 + (p.b_resident ? 0.0 : ksteps * b_bytes / 30.0);
        const double epilogue = 120.0 * p.mtiles * tz * (cout / 16);
        const int64_t tiles = static_cast<int64_t>(tiles_x) * tiles_y * p.tiles_z;
        const double time = static_cast<double>((tiles + kConvSms - 1) / kConvSms) *
                                std::max(std::max(mma, loads), epilogue) + std::min(mma, loads) / 2 + epilogue;
        if (best.tx == 0 || time < best_time) {
          best = p;
          best_time = time;
        }
      }
    }
  }
  return best;
}

int launch_conv(const ConvArgs& a0, const void* in_planes, int in_chunks, cudaStream_t st) {
  ConvArgs a = a0;
  if (a.cout % 16 != 0 || a.cout > 96 || (in_chunks != 1 && in_chunks % 2 != 0)) return -1;
  a.plan = plan_conv(a.lx, a.ly, a.lz, in_chunks, a.cout);
  const ConvPlan& p = a.plan;
  if (p.tx == 0) return -3;
  CUtensorMap map;
  if (encode_planes_map(&map, in_planes, a.lx, a.ly, a.lz, in_chunks, p.pitch, p.ty + 2, p.kchunks) != 0) return -2;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !g_attr_set[dev]) {
    cudaFuncSetAttribute(k_conv_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kConvSmem));
    cudaFuncSetAttribute(k_conv_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kConvSmem));
    g_attr_set[dev] = true;
  }
  const size_t smem = static_cast<size_t>(kConvSmemFixed) + static_cast<size_t>(p.stages) * p.a_bytes +
                      static_cast<size_t>(p.b_slots) * p.b_bytes;
  const auto kernel = in_chunks == 1 ? k_conv_tc<true> : k_conv_tc<false>;
  kernel<<<std::min(p.tiles_x * p.tiles_y * p.tiles_z, kConvSms), kConvThreads, smem, st>>>(map, a);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -4;
}

void launch_pack_input(const float* f, float tau, int64_t nv, void* x, cudaStream_t st) {
  k_pack_input<<<static_cast<unsigned>((nv + 255) / 256), 256, 0, st>>>(f, tau, nv, static_cast<uint4*>(x));
}

void launch_avgpool(const void* in, int in_plane0, int planes, int lx, int ly, int lz, void* out, cudaStream_t st) {
  const int64_t n = static_cast<int64_t>(lx / 2) * (ly / 2) * (lz / 2) * planes;
  k_avgpool<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(static_cast<const uint4*>(in), in_plane0, planes,
                                                                    lx, ly, lz, static_cast<uint4*>(out));
}

void launch_upsample_back(const void* g, int g_plane0, int planes, int lx, int ly, int lz, const void* act_up,
                          int act_plane0, void* out, cudaStream_t st) {
  const int64_t n = static_cast<int64_t>(lx / 2) * (ly / 2) * (lz / 2) * planes;
  k_upsample_back<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(
      static_cast<const uint4*>(g), g_plane0, planes, lx, ly, lz, static_cast<const uint4*>(act_up), act_plane0,
      static_cast<uint4*>(out));
}

void launch_skip_back(const void* gs, int gs_plane0, const void* gp, const void* s, int s_plane0, int planes, int lx,
                      int ly, int lz, void* out, cudaStream_t st) {
  const int64_t n = static_cast<int64_t>(lx) * ly * lz * planes;
  k_skip_back<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(
      static_cast<const uint4*>(gs), gs_plane0, static_cast<const uint4*>(gp), static_cast<const uint4*>(s), s_plane0,
      planes, lx, ly, lz, static_cast<uint4*>(out));
}

int head_blocks(int64_t nv) { return static_cast<int>((nv + 255) / 256); }

void launch_head_backward(const void* u1, const float* hw, int64_t nv, const float* f, const float* g, void* gz,
                          double* partial, double* loss, float* grad, int64_t hw_off, int64_t hb_off, cudaStream_t st) {
  const int nb = head_blocks(nv);
  k_head_backward<<<nb, 256, 0, st>>>(static_cast<const uint4*>(u1), hw, nv, f, g, static_cast<uint4*>(gz), partial);
  k_head_reduce<<<1, 32, 0, st>>>(partial, nb, nv, loss, grad, hw_off, hb_off);
}

int64_t wgrad_partial_floats(int64_t nv, int cout, int cin) {
  const int64_t nblk = (nv + kWgChunk - 1) / kWgChunk;
  return 27 * nblk * cout * cin;
}

int64_t bias_partial_floats(int64_t nv, int cout) { return ((nv + 2047) / 2048) * cout; }

void launch_wgrad(const void* x, int x_plane0, int cin, int cin_real, const void* gz, int cout, int lx, int ly, int lz,
                  float* partial, float* gw, float* bpartial, float* gb, cudaStream_t st) {
  const int64_t nv = static_cast<int64_t>(lx) * ly * lz;
  const int nblk = static_cast<int>((nv + kWgChunk - 1) / kWgChunk);
  const size_t smem = (static_cast<size_t>(cout + cin) * kWgV + static_cast<size_t>(cout) * cin) * sizeof(float);
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr[dev]) {
    cudaFuncSetAttribute(k_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    attr[dev] = true;
  }
  k_wgrad<<<dim3(nblk, 27), 256, smem, st>>>(static_cast<const uint4*>(x), x_plane0, cin,
                                             static_cast<const uint4*>(gz), cout, lx, ly, lz, partial);
  const int n = 27 * cout * cin_real;
  k_wgrad_reduce<<<(n + 255) / 256, 256, 0, st>>>(partial, nblk, cout, cin, cin_real, gw);
  const int nb = static_cast<int>((nv + 2047) / 2048);
  k_bias_partial<<<nb, 256, 0, st>>>(static_cast<const uint4*>(gz), cout, nv, bpartial);
  k_bias_reduce<<<1, 128, 0, st>>>(bpartial, nb, cout, gb);
}

void launch_pack_weights(const float* w, int cout_f, int cin_real, int cin_pad, int transpose, void* pack,
                         cudaStream_t st) {
  const int64_t total = pack_elems(cout_f, cin_pad, transpose);
  k_pack_weights<<<static_cast<unsigned>((total + 255) / 256), 256, 0, st>>>(
      w, cout_f, cin_real, cin_pad, transpose, total, static_cast<__nv_bfloat16*>(pack));
}

int64_t pack_elems(int cout_f, int cin_pad, int transpose) {
  const int n_in = transpose ? cout_f : cin_pad;
  const int n_out = transpose ? cin_pad : cout_f;
  return static_cast<int64_t>(n_in == 8 ? 1 : n_in / 16) * (n_in == 8 ? 6 : 9) * 2 * 3 * n_out * 8;
}

void launch_round_bf16(const float* in, int64_t n, float* out, cudaStream_t st) {
  k_round_bf16<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(in, n, out);
}

void launch_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float beta1, float beta2,
                 float eps, float bc1, float bc2, cudaStream_t st) {
  k_adam<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(p, g, m, v, n, lr, beta1, beta2, eps, bc1, bc2);
}

void launch_unpack_planes(const void* in, int plane0, int c_real, int64_t nv, float* out, cudaStream_t st) {
  const int64_t n = nv * c_real;
  k_unpack_planes<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(static_cast<const uint4*>(in), plane0,
                                                                         c_real, nv, out);
}

}  // namespace unet
}  // namespace tsf
