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
// cores; k_conv_tc says how.  The weight gradients are GEMMs over the voxels
// (k_wgrad_tc).  Pooling, upsampling, the head's backward pass, the loss and
// Adam are bandwidth-bound and run on the CUDA cores.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
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
// K-major (or both MN-major), M x N.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n, bool mn_major = false) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major ? 3u << 15 : 0u) | (static_cast<uint32_t>(n >> 3) << 17) |
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

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
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
// A block computes tx x ty x tz output voxels, walking the tz + 2 input
// z-planes.  TMA brings a plane's (ty + 2) x (tx + 2) voxels of every input
// channel (zero outside the grid: the padding) as 16-byte rows, one after the
// other.  In the no-swizzle K-major operand layout 128 consecutive rows are an
// A tile, so a tile of 128 outputs (flattened with pitch tx + 2; the two halo
// columns of a row give outputs that nobody keeps) reads its (dy, dx)
// neighbours by a shift of the operand's start address: one load serves nine
// taps.  The three dz taps of an input plane go to three output planes, whose
// accumulators lie next to each other in TMEM, so the three weight matrices
// form one B operand of 3 x cout columns and one MMA does all three.  Every
// output still sums its taps in (dz, dy, dx) order, 16 channels at a time.
// A block per SM walks over tiles: one warp issues the loads (they run ahead
// into the next tile), two the MMAs (half of a tile's operand tiles each),
// eight turn accumulators into outputs while the other half of TMEM (256
// columns) takes the next tile's MMAs.  Weights that fit stay in shared memory
// for the whole launch, others come again for every plane.
// Bound: the A operand.  An MMA reads 4 KB of A (32 cycles of shared-memory
// bandwidth) and 96 x cout bytes of B, 32 + 3 x cout / 4 cycles in all, for
// 3 x cout / 2 cycles of math, so 16 output channels reach about half of the
// tensor rate.
// A single input plane (8 channels, kSteps = 0) makes K steps of two taps: the
// second half of K is the next tap's rows, at their distance from the first's.
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

// The MMAs of one input plane on kM operand tiles.
struct PlaneMmas {
  uint64_t a;            // operand descriptor of the first tile, tap and K step
  uint32_t kstep;        // ... distance of two K steps (16-byte units)
  uint32_t t0, tcols;    // accumulators of d = 0 and the distance of two tiles'
  uint32_t cout, pitch;
  int dlo, dhi;          // dz taps that stay in the tile
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

// One (dy, dx) tap on every K step; at, bt its operand rows and weights.
// `first` (tap 0): input plane zi is the first to reach output plane zi
// (d = 2), which starts its sums here.  kWide: three dz taps are more than 256
// columns, so d = 2 always has an MMA of its own.
template <int kSteps, int kM, bool kWide>
__device__ __forceinline__ void issue_tap_steps(const PlaneMmas& f, uint64_t at, uint64_t bt, bool first) {
  const int n = f.dhi - f.dlo + 1;
  const bool upper = f.dhi == 2 && f.dlo < 2;  // d = 2 next to others
#pragma unroll
  for (int kk = 0; kk < kSteps; ++kk) {
    const uint64_t ad = at + static_cast<uint32_t>(kk) * f.kstep, bd = bt + static_cast<uint32_t>(kk) * (6u * f.cout);
    const bool start = kk == 0 && first;
    if ((kWide || start) && upper) {
      issue_tap<kM>(f, ad, bd, f.dlo, 2 - f.dlo, 1u);
      issue_tap<kM>(f, ad, bd, 2, 1, start ? 0u : 1u);
    } else {
      issue_tap<kM>(f, ad, bd, f.dlo, n, start && f.dlo == 2 ? 0u : 1u);
    }
  }
}

// Every tap of one input plane (resident weights at b, btap apart).  An MMA of
// 48 columns takes 44 cycles, and the loop has to issue one in as many.
// 256^3 voxels, 16 to 16 channels: rolled over taps and tiles 1046 us, over
// tiles only 645, unrolled 437 (66 cycles per MMA: about 72 per tap and 49 per
// tile); two warps that share the tiles take the whole layer from 479 to 403
// us.  With two or more K steps the tap loop stays rolled: a small grid's one
// pass through a long unrolled body waits for its instructions (32^3, 32 to
// 32 channels: 22 us unrolled, 14 rolled).
template <int kSteps, int kM, bool kWide>
__device__ __forceinline__ void issue_plane(const PlaneMmas& f, uint64_t b, uint32_t btap) {
  issue_tap_steps<kSteps, kM, kWide>(f, f.a, b, true);
#pragma unroll(kSteps == 1 ? 8 : 1)
  for (int tap = 1; tap < 9; ++tap)
    issue_tap_steps<kSteps, kM, kWide>(f, f.a + static_cast<uint32_t>(tap / 3) * f.pitch + static_cast<uint32_t>(tap % 3),
                                       b + static_cast<uint32_t>(tap) * btap, false);
}

// A single input plane of 8 channels: the 14 K steps (27 taps in pairs; the
// last tap's partner has zero weights) of one output plane, from the input
// planes at a, a + dplane, a + 2 dplane.
template <int kM>
__device__ __forceinline__ void issue_single(const PlaneMmas& f, uint32_t dplane, uint64_t bt) {
  const uint32_t idesc = instr_desc(128, static_cast<int>(f.cout));
#pragma unroll
  for (int t = 0; t < 14; ++t) {
    const int t0 = 2 * t, t1 = t == 13 ? 26 : 2 * t + 1;
    const uint32_t o0 = static_cast<uint32_t>(t0 / 9) * dplane + static_cast<uint32_t>(t0 / 3 % 3) * f.pitch + t0 % 3;
    const uint32_t o1 = static_cast<uint32_t>(t1 / 9) * dplane + static_cast<uint32_t>(t1 / 3 % 3) * f.pitch + t1 % 3;
    const uint64_t ad = f.a + o0 + (static_cast<uint64_t>(o1 - o0) << 16);  // the distance of the K halves
    const uint64_t bd = bt + static_cast<uint32_t>(t) * (2u * f.cout);
#pragma unroll
    for (int m = 0; m < kM; ++m) mma_bf16(f.t0 + m * f.tcols, ad + m * 128u, bd, idesc, t > 0 ? 1u : 0u);
  }
}

template <int kSteps, bool kWide = false>
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
    for (int s = 0; s < kConvBSlotsMax; ++s) {
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
    // producer: each plane, then its taps' weights (once, if all stay, after
    // the first plane; else again as the ring frees up)
    int it = 0, bt = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      const int x0 = (tile % p.tiles_x) * p.tx, y0 = ((tile / p.tiles_x) % p.tiles_y) * p.ty,
                z0 = tile / (p.tiles_x * p.tiles_y) * p.tz;
      for (int zi = 0; zi < p.tz + 2 && ok; ++zi, ++it) {
        const int slot = it % p.stages;
        if (it >= p.stages && !mbar_wait(&sh.empty_a[slot], ((it / p.stages) - 1) & 1)) ok = false;
        if (!ok || *gave_up) {
          ok = false;
          break;
        }
        mbar_expect_tx(&sh.full_a[slot], p.a_tx);
        tma_load_4d(smem + slot * p.a_bytes, &in_map, 2 * (x0 - 1), y0 - 1, z0 - 1 + zi, 0, &sh.full_a[slot]);
        sh.issued_a = it + 1;
        for (int tap = 0; (!p.b_resident || it == 0) && tap < p.taps; ++tap, ++bt) {
          const int bs = bt % p.b_slots;
          if (bt >= p.b_slots && !mbar_wait(&sh.empty_b[bs], ((bt / p.b_slots) - 1) & 1)) ok = false;
          if (!ok || *gave_up) {
            ok = false;
            break;
          }
          mbar_expect_tx(&sh.full_b[bs], p.b_bytes);
          bulk_load(sb0 + bs * p.b_bytes, a.wpack + static_cast<size_t>(tap) * (p.b_bytes / 2), p.b_bytes,
                    &sh.full_b[bs]);
          sh.issued_b = bt + 1;
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
    const uint32_t a_lbo = kSteps == 0 ? 0u : static_cast<uint32_t>((p.ty + 2) * p.pitch) * 16u;
    const uint32_t b_lbo = static_cast<uint32_t>((kSteps == 0 ? 1 : 3) * a.cout) * 16u;
    const uint32_t tcols = static_cast<uint32_t>(p.tz * a.cout);
    int it = 0, bt = 0, nt = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++nt) {
      const int half = nt & 1;
      if (nt >= 2 && !mbar_wait_warp(&sh.tempty[half], ((nt >> 1) - 1) & 1)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t tmine = taddr + (half ? thalf : 0u) + static_cast<uint32_t>(m0) * tcols;
      for (int zi = 0; zi < p.tz + 2 && ok; ++zi, ++it) {
        const int slot = it % p.stages;
        if (!mbar_wait_warp(&sh.full_a[slot], (it / p.stages) & 1) || __any_sync(0xFFFFFFFFu, *gave_up)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (kSteps == 0) {
          // planes zi - 2 .. zi make output plane zi - 2 (a tile's planes lie
          // one after the other: stages is a multiple of tz + 2)
          for (int tap = 0; it == 0 && tap < p.taps && ok; ++tap) ok = mbar_wait_warp(&sh.full_b[tap], 0);
          if (zi < 2) continue;
          const uint64_t abase = smem_desc(smem_u32(smem + (slot - 2) * p.a_bytes), a_lbo, 128u);
          const PlaneMmas f{abase + static_cast<uint32_t>(m0) * 128u, 0u, tmine + static_cast<uint32_t>((zi - 2) * a.cout),
                            tcols, static_cast<uint32_t>(a.cout), static_cast<uint32_t>(p.pitch), 0, 0};
          const uint64_t bd = smem_desc(smem_u32(sb0), b_lbo, 128u);
          if (nm == 1) issue_single<1>(f, static_cast<uint32_t>(p.a_bytes / 16), bd);
          else if (nm == 2) issue_single<2>(f, static_cast<uint32_t>(p.a_bytes / 16), bd);
          mma_commit(&sh.empty_a[slot - 2]);  // the slot is free once these MMAs have read it
          if (zi == p.tz + 1) {
            mma_commit(&sh.empty_a[slot - 1]);
            mma_commit(&sh.empty_a[slot]);
          }
          continue;
        }
        // input plane zi feeds output planes zi - 2 + d (dz tap 2 - d)
        const uint64_t abase = smem_desc(smem_u32(smem + slot * p.a_bytes), a_lbo, 128u);
        const PlaneMmas f{abase + static_cast<uint32_t>(m0) * 128u, 2u * (a_lbo >> 4),
                          tmine + static_cast<uint32_t>((zi - 2) * a.cout), tcols, static_cast<uint32_t>(a.cout),
                          static_cast<uint32_t>(p.pitch), max(0, 2 - zi), min(2, p.tz + 1 - zi)};
        constexpr int kS = kSteps > 0 ? kSteps : 1;
        if (p.b_resident && it > 0) {
          const uint64_t bbase = smem_desc(smem_u32(sb0), b_lbo, 128u);
          const uint32_t btap = static_cast<uint32_t>(p.b_bytes) >> 4;
          if (nm == 1) issue_plane<kS, 1, kWide>(f, bbase, btap);
          else if (nm == 2) issue_plane<kS, 2, kWide>(f, bbase, btap);
        } else {  // weights arrive tap by tap
          for (int tap = 0; tap < 9; ++tap, ++bt) {
            const int bs = bt % p.b_slots;
            if (!mbar_wait_warp(&sh.full_b[bs], (bt / p.b_slots) & 1)) {
              ok = false;
              break;
            }
            const uint64_t bd = smem_desc(smem_u32(sb0 + bs * p.b_bytes), b_lbo, 128u);
            const uint64_t at = f.a + static_cast<uint32_t>(tap / 3) * f.pitch + static_cast<uint32_t>(tap % 3);
            if (nm == 1) issue_tap_steps<kS, 1, kWide>(f, at, bd, tap == 0);
            else if (nm == 2) issue_tap_steps<kS, 2, kWide>(f, at, bd, tap == 0);
            if (!p.b_resident) mma_commit(&sh.empty_b[bs]);
          }
          if (!ok) break;
        }
        mma_commit(&sh.empty_a[slot]);
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
// Bound: fp64 arithmetic (two operations per clock on an SM), most of all the
// warp sums, so a block per SM loops over the voxels and sums across a warp
// once: 64^3 voxels 71 us with a block per 256 voxels, 32 us now.
__global__ void __launch_bounds__(256) k_head_backward(const uint4* __restrict__ u1, const float* __restrict__ hw,
                                                       int64_t nv, const float* __restrict__ f,
                                                       const float* __restrict__ g, uint4* __restrict__ gz,
                                                       double* __restrict__ partial) {
  __shared__ double red[18][8];
  const float hb = hw[16];
  double acc[18];
#pragma unroll
  for (int k = 0; k < 18; ++k) acc[k] = 0.0;
  for (int64_t v = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; v < nv;
       v += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    float a[16];
    unpack8(u1[v], a);
    unpack8(u1[nv + v], a + 8);
    float r = 0.0f;
#pragma unroll
    for (int c = 0; c < 16; ++c) r = fmaf(a[c], hw[c], r);
    r = __bfloat162float(__float2bfloat16_rn(r + hb));
    const float d = (f[v] + r) - g[v];
    const float gg = 2.0f * d / static_cast<float>(nv);
    acc[0] += static_cast<double>(d) * d;
    acc[1] += gg;
    float o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      acc[2 + c] += static_cast<double>(gg) * a[c];
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

// Sums the head's block partials, one warp per value, in a fixed order: out[0]
// = loss (mean), grad[hw_off + c] = sum gg u1[c], grad[hb_off] = sum gg.
__global__ void __launch_bounds__(18 * 32) k_head_reduce(const double* __restrict__ partial, int nblocks, int64_t nv,
                                                         double* __restrict__ loss, float* __restrict__ grad,
                                                         int64_t hw_off, int64_t hb_off) {
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s = 0.0;
  for (int b = lane; b < nblocks; b += 32) s += partial[static_cast<int64_t>(b) * 18 + k];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if (lane != 0) return;
  if (k == 0) *loss = s / static_cast<double>(nv);
  else if (k == 1) grad[hb_off] = static_cast<float>(s);
  else grad[hw_off + (k - 2)] = static_cast<float>(s);
}

// Weight gradient of one convolution: gw[o][c][tap] = sum over voxels p of
// gz[o][p] x[c][p + tap - 1] (zero outside the grid), gb[o] = sum gz[o][p],
// as a GEMM over the voxels on the tensor cores.  The chunk planes are
// MN-major operands as they lie: 8 channels of a voxel are one 16-byte row, 8
// consecutive voxels a core matrix, so 16 voxels along x are a K step.
//   M: the cout channels of gz, three times: shifted by the dy taps (copies
//      that TMA loads; with 64 channels one copy, and a third of the blocks
//      per dy).
//   N: a block of input channels at the planes z - 1, z, z + 1 (dz taps).
//   The three dx taps are shifts of the N operand's start address by one row,
//   each with its own accumulator, issued by its own warp.
// gz is zero outside the grid and tx is a multiple of 16, so every pair of a
// voxel and a tap counts once.  A step is one z-plane of a tx x ty tile; a
// block takes a range of steps, keeps its sums in TMEM, and writes one partial
// per launch; k_wgrad_reduce adds the partials in a fixed order.
// Bound: loads (gz and x three times each, from L2).  64^3 voxels, 48 to 16
// channels: 2264 us on the CUDA cores with operands converted to fp32 in
// shared memory, 23 us here.
constexpr int kWgThreads = 256;  // warps 0-3 bias and epilogue, 4 loads, 5-7 MMAs of one dx tap each
constexpr int kWgStagesMax = 4;

struct WgBars {
  uint64_t full[kWgStagesMax], empty[kWgStagesMax], done;
  uint32_t taddr;
  int gave_up, issued;
  float bias[128 * 8];
};

__global__ void __launch_bounds__(kWgThreads, 1) k_wgrad_tc(const __grid_constant__ CUtensorMap x_map,
                                                            const __grid_constant__ CUtensorMap g_map, WgradPlan p,
                                                            float* __restrict__ partial, float* __restrict__ bpartial,
                                                            uint32_t* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ WgBars sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* gave_up = &sh.gave_up;
  const int cb = blockIdx.y % p.cin_blocks, dyi = blockIdx.y / p.cin_blocks;  // input channel block, dy tap (one copy)
  const int s0 = static_cast<int>(static_cast<int64_t>(p.steps) * blockIdx.x / gridDim.x);
  const int s1 = static_cast<int>(static_cast<int64_t>(p.steps) * (blockIdx.x + 1) / gridDim.x);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 3 + 4);
    }
    mbar_init(&sh.done, 3);
    sh.gave_up = 0;
    sh.issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.taddr)),
                 "r"(static_cast<uint32_t>(p.tmem_cols))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t taddr = __shfl_sync(0xFFFFFFFFu, sh.taddr, 0);
  const int role = __shfl_sync(0xFFFFFFFFu, warp, 0);
  const int n = 24 * p.cin_chunks;  // N: dz taps x 8 channels per plane

  if (role == 4 && lane == 0) {
    bool ok = true;
    for (int s = s0, it = 0; s < s1; ++s, ++it) {
      const int slot = it % p.stages;
      if (it >= p.stages && !mbar_wait(&sh.empty[slot], ((it / p.stages) - 1) & 1)) ok = false;
      if (!ok || *gave_up) {
        ok = false;
        break;
      }
      const int z = s % p.lz, t = s / p.lz;
      const int x0 = (t % p.tiles_x) * p.tx, y0 = (t / p.tiles_x) * p.ty;
      uint8_t* sg = smem + slot * p.stage_bytes;
      mbar_expect_tx(&sh.full[slot], p.tx_bytes);
      for (int c = 0; c < p.copies; ++c) {  // row y of copy c holds gz at y - dy, dy = c - 1
        const int dy = p.copies == 3 ? c : dyi;
        tma_load_4d(sg + c * p.copy_bytes, &g_map, 2 * x0, y0 + 1 - dy, z, 0, &sh.full[slot]);
      }
      tma_load_4d(sg + p.copies * p.copy_bytes, &x_map, 2 * (x0 - 1), y0, z - 1, cb * p.cin_chunks, &sh.full[slot]);
      sh.issued = it + 1;
    }
    if (!ok) {
      if (!*gave_up) atomicOr(status, kUnetErrSpin);
      *gave_up = 1;
    }
  } else if (role > 4) {
    const int dx = role - 5;
    const uint32_t idesc = instr_desc(p.m, n, true);
    const uint32_t td = taddr + static_cast<uint32_t>(dx * n);
    const uint32_t g_sbo = static_cast<uint32_t>(p.tx * p.ty) * 16u, x_sbo = static_cast<uint32_t>(p.pitch * p.ty) * 16u;
    const int kx = p.tx / 16;
    uint32_t acc = 0u;
    bool ok = true;
    for (int s = s0, it = 0; s < s1; ++s, ++it) {
      const int slot = it % p.stages;
      if (!mbar_wait_warp(&sh.full[slot], (it / p.stages) & 1) || __any_sync(0xFFFFFFFFu, *gave_up)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t sg = smem_u32(smem + slot * p.stage_bytes);
      uint64_t ad = smem_desc(sg, 128u, g_sbo);
      uint64_t brow = smem_desc(sg + static_cast<uint32_t>(p.copies * p.copy_bytes), 128u, x_sbo) + dx;
      for (int y = 0; y < p.ty; ++y) {
        uint64_t bd = brow;
#pragma unroll 4
        for (int k = 0; k < kx; ++k) {
          mma_bf16(td, ad, bd, idesc, acc);
          acc = 1u;
          ad += 16u;
          bd += 16u;
        }
        brow += static_cast<uint32_t>(p.pitch);
      }
      mma_commit(&sh.empty[slot]);
    }
    if (!ok && lane == 0) {
      if (!*gave_up) atomicOr(status, kUnetErrSpin);
      *gave_up = 1;
    }
    __syncwarp();
    mma_commit(&sh.done);
    mbar_wait_warp(&sh.done, 0);
  } else if (role < 4) {
    // bias: thread t sums channels of plane t / per over the rows t % per,
    // t % per + per, ... of the unshifted copy
    const bool bias = cb == 0 && (p.copies == 3 || dyi == 1);
    const int per = 128 / p.cout_chunks, plane = threadIdx.x / per, rows = p.tx * p.ty;
    const int copy = p.copies == 3 ? 1 : 0;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    bool ok = true;
    for (int s = s0, it = 0; s < s1; ++s, ++it) {
      const int slot = it % p.stages;
      if (!mbar_wait_warp(&sh.full[slot], (it / p.stages) & 1) || __any_sync(0xFFFFFFFFu, *gave_up)) {
        ok = false;
        break;
      }
      if (bias) {
        const uint4* g = reinterpret_cast<const uint4*>(smem + slot * p.stage_bytes + copy * p.copy_bytes) +
                         static_cast<size_t>(plane) * rows;
        for (int r = threadIdx.x % per; r < rows; r += per) {
          float t[8];
          unpack8(g[r], t);
#pragma unroll
          for (int c = 0; c < 8; ++c) acc[c] += t[c];
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.empty[slot]);
    }
    if (ok && !mbar_wait_warp(&sh.done, 0)) ok = false;
    if (__any_sync(0xFFFFFFFFu, !ok || *gave_up)) {
      if (lane == 0) {
        if (!*gave_up) atomicOr(status, kUnetErrSpin);
        *gave_up = 1;
      }
    } else {
      tc_fence_after();
      // M = 64: row 16 w + l in lane l < 16 of warp w; M = 128: row 32 w + l
      const int row = p.m == 64 ? (lane < 16 ? warp * 16 + lane : p.m) : warp * 32 + lane;
      const int mrows = p.copies * p.cout_chunks * 8;
      float* out = partial + (static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x) * (3 * mrows * n);
      for (int dx = 0; dx < 3; ++dx)
        for (int c = 0; c < n; c += 8) {
          float v[8];
          __syncwarp();
          tmem_ld8(taddr + (static_cast<uint32_t>(warp * 32) << 16) + static_cast<uint32_t>(dx * n + c), v);
          if (s0 >= s1) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = 0.0f;
          }
          if (row < mrows) {
            float4* o = reinterpret_cast<float4*>(out + (static_cast<size_t>(dx) * mrows + row) * n + c);
            o[0] = make_float4(v[0], v[1], v[2], v[3]);
            o[1] = make_float4(v[4], v[5], v[6], v[7]);
          }
        }
      tc_fence_before();
    }
    if (bias) {
#pragma unroll
      for (int c = 0; c < 8; ++c) sh.bias[threadIdx.x * 8 + c] = acc[c];
    }
  }
  __syncthreads();
  if (cb == 0 && (p.copies == 3 || dyi == 1) && threadIdx.x < p.cout_chunks * 8) {
    const int per = 128 / p.cout_chunks, plane = threadIdx.x / 8, c = threadIdx.x % 8;
    float sum = 0.0f;
    for (int t = 0; t < per; ++t) sum += sh.bias[(plane * per + t) * 8 + c];
    bpartial[static_cast<size_t>(blockIdx.x) * p.cout_chunks * 8 + threadIdx.x] = sum;
  }
  // after giving up, wait (bounded) for the copies still in flight before the
  // shared memory they target is released
  if (threadIdx.x == 0 && *gave_up) {
    for (int s = max(0, sh.issued - p.stages); s < sh.issued; ++s)
      mbar_wait(&sh.full[s % p.stages], (s / p.stages) & 1);
  }
  __syncthreads();
  tc_fence_after();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                 "r"(static_cast<uint32_t>(p.tmem_cols))
                 : "memory");
  }
}

// gw in the reference layout (cout, cin_real, 3, 3, 3) and gb: the partials
// summed as eight interleaved shares of the blocks, then the shares, in fixed
// order.  Thread (i, share): element i of a partial's order, so that reads are
// coalesced.
__global__ void __launch_bounds__(256) k_wgrad_reduce(WgradPlan p, const float* __restrict__ partial,
                                                      const float* __restrict__ bpartial, int cin_real,
                                                      float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, share = threadIdx.x >> 5;
  const int n = 24 * p.cin_chunks, cout = p.cout_chunks * 8, mrows = p.copies * cout;
  const int per = 3 * mrows * n, total = p.groups * per;
  const int i = blockIdx.x * 32 + lane;
  const bool weight = i < total, bias = !weight && i < total + cout;
  const float* src = weight ? partial + static_cast<size_t>(i / per) * p.blocks * per + i % per : bpartial + (i - total);
  const size_t step = weight ? per : cout;
  float s = 0.0f;
  if (weight || bias) {
#pragma unroll 8
    for (int b = share; b < p.blocks; b += 8) s += src[static_cast<size_t>(b) * step];
  }
  red[share][lane] = s;
  __syncthreads();
  if (share != 0) return;
#pragma unroll
  for (int k = 1; k < 8; ++k) s += red[k][lane];
  if (bias) gb[i - total] = s;
  if (!weight) return;
  const int grp = i / per, cb = grp % p.cin_blocks, dyg = grp / p.cin_blocks;
  const int col = i % n, row = (i % per) / n % mrows, dx = (i % per) / n / mrows;
  const int e = col % 8, dz = col / 8 % 3, c = (cb * p.cin_chunks + col / 24) * 8 + e;
  const int o = row % cout, dy = p.copies == 3 ? row / cout : dyg;
  if (c < cin_real) gw[(static_cast<int64_t>(o) * cin_real + c) * 27 + (dz * 3 + dy) * 3 + dx] = s;
}

// Weights of one layer from the fp32 master copy (reference layout
// (cout, cin_real, 3, 3, 3)) into the bf16 B operand of k_conv_tc:
// pack[(dy, dx) tap][K step][K half][d * n_out + o][8], d = 0..2 for the dz
// tap 2 - d; for a single input plane pack[pair of taps][K half][o][8].  The
// data-gradient packing transposes and flips: B[o'][c'][tap] =
// w[c'][o'][26 - tap] (o' over the forward inputs, c' over its outputs).
__global__ void k_pack_weights(const float* __restrict__ w, int cout_f, int cin_real, int cin_pad, int transpose,
                               int64_t total, __nv_bfloat16* __restrict__ pack) {
  const int n_out = transpose ? cin_pad : cout_f;   // N of the GEMM
  const int n_in = transpose ? cout_f : cin_pad;    // input channels of the GEMM
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= total) return;
  const int e = static_cast<int>(i % 8);
  int o, ci, tap;
  if (n_in == 8) {
    o = static_cast<int>((i / 8) % n_out);
    tap = static_cast<int>(i / (8 * n_out));  // pair and half
    ci = e;
  } else {
    const int ksteps = n_in / 16;
    const int n = static_cast<int>((i / 8) % (3 * n_out));
    const int half = static_cast<int>((i / (24 * n_out)) % 2);
    const int kk = static_cast<int>((i / (48 * n_out)) % ksteps);
    const int t = static_cast<int>(i / (static_cast<int64_t>(48) * n_out * ksteps));
    o = n % n_out;
    ci = (kk * 2 + half) * 8 + e;
    tap = (2 - n / n_out) * 9 + t;
  }
  float val = 0.0f;
  if (tap < 27) {
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
std::atomic<EncodeTiledFn> g_encode{nullptr};  // networks may run in several host threads
std::atomic<bool> g_attr_set[64] = {};
}  // namespace

// Planes as (2 * lx, ly, lz, chunks) 8-byte elements, two per voxel, so that a
// row of voxels is one run of a box's innermost dimension (at most 256
// elements): TMA takes three to five cycles per innermost run, and with
// 16-byte runs it, not the tensor cores, set the time.  x coordinates are
// multiples of two elements, 16 bytes.
int encode_planes_map(CUtensorMap* map, const void* base, int lx, int ly, int lz, int chunks, int bx, int by, int bz,
                      int bchunks) {
  EncodeTiledFn encode = g_encode.load(std::memory_order_acquire);
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
      return -1;
    encode = reinterpret_cast<EncodeTiledFn>(fn);
    g_encode.store(encode, std::memory_order_release);
  }
  const uint64_t nv = static_cast<uint64_t>(lx) * ly * lz;
  cuuint64_t dims[4] = {2 * static_cast<cuuint64_t>(lx), static_cast<cuuint64_t>(ly), static_cast<cuuint64_t>(lz),
                        static_cast<cuuint64_t>(chunks)};
  cuuint64_t strides[3] = {16ull * lx, 16ull * lx * ly, 16ull * nv};
  cuuint32_t box[4] = {2 * static_cast<cuuint32_t>(bx), static_cast<cuuint32_t>(by), static_cast<cuuint32_t>(bz),
                       static_cast<cuuint32_t>(bchunks)};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, const_cast<void*>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -1;
}

// Tile of a convolution: the shape of least estimated time, in cycles.  An MMA
// of n dz taps takes 32 + n x cout / 4 (its operands' shared-memory reads); a
// tile's tz + 2 planes feed one, two or three output planes each; loads and
// epilogue run beside the MMAs, and a change of tiles costs about 1200.  Small
// grids take smaller tiles so that every SM has one.
ConvPlan plan_conv(int lx, int ly, int lz, int chunks, int cout, int sms) {
  ConvPlan best{};
  double best_time = 0.0;
  const bool single = chunks == 1;
  const int ksteps = chunks / 2, taps = single ? 14 : 9;
  const int b_bytes = single ? 2 * cout * 16 : ksteps * 2 * 3 * cout * 16;  // weights of a tap (of a pair of taps)
  const int room = static_cast<int>(kConvSmem) - kConvSmemFixed;
  const int min_x = (lx + kConvTx - 1) / kConvTx;
  const unsigned usms = static_cast<unsigned>(sms);
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
        p.chunks = chunks;
        p.taps = taps;
        p.a_tx = (ty + 2) * pitch * 16 * chunks;
        p.a_bytes = (p.a_tx + 127) / 128 * 128;
        p.b_bytes = b_bytes;
        p.b_resident = room - taps * b_bytes >= 3 * p.a_bytes;
        p.b_slots = taps;
        if (p.b_resident) {
          p.stages = std::min((room - taps * b_bytes) / p.a_bytes, kConvStagesMax);
        } else {  // up to three planes, the rest of the room for weights
          p.stages = std::min((room - 3 * b_bytes) / p.a_bytes, 3);
          p.b_slots = std::min((room - p.stages * p.a_bytes) / b_bytes, taps);
        }
        if (single) p.stages = p.stages / (tz + 2) * (tz + 2);
        if (single ? !p.b_resident || p.stages < tz + 2 : p.stages < 2) continue;
        const int cols = 2 * p.mtiles * tz * cout;
        p.tmem_cols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
        const int groups = single ? tz * taps : (tz + 2) * taps * ksteps;  // operand pairs issued per tile
        double mma = 0.0;
        for (int zi = 0; zi < tz + 2; ++zi)
          mma += 32.0 + (std::min(2, tz + 1 - zi) - std::max(0, 2 - zi) + 1) * cout / 4.0;
        mma = single ? tz * 14 * 40.0 : mma * taps * ksteps;
        // ... or what its issue takes: about 72 cycles per tap, 49 per tile
        mma = std::max(mma * p.mtiles, groups * (72.0 + 49.0 * ((p.mtiles + 1) / 2)));
        const double loads = (tz + 2) * (p.a_tx + (p.b_resident ? 0.0 : static_cast<double>(taps) * b_bytes)) / 30.0;
        const double epilogue = 120.0 * p.mtiles * tz * (cout / 16);
        const unsigned tiles = static_cast<unsigned>(tiles_x * tiles_y * p.tiles_z);  // a 32-bit division each
        const double time = static_cast<double>((tiles + usms - 1) / usms) *
                                std::max(std::max(mma + 1200.0, loads), epilogue) + std::min(mma, loads) / 2 + epilogue;
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
  using Kernel = void (*)(const CUtensorMap, ConvArgs);
  // the network's layers; more than 85 output channels: from 32 inputs only
  const Kernel kernel = in_chunks == 1    ? k_conv_tc<0>
                        : in_chunks == 2  ? k_conv_tc<1>
                        : in_chunks == 4  ? (a.cout > 85 ? k_conv_tc<2, true> : k_conv_tc<2>)
                        : in_chunks == 6  ? k_conv_tc<3>
                        : in_chunks == 8  ? k_conv_tc<4>
                        : in_chunks == 12 ? k_conv_tc<6>
                                          : nullptr;
  if (!kernel || a.cout % 16 != 0 || a.cout > 96 || (a.cout > 85 && in_chunks != 4)) return -1;
  a.plan = plan_conv(a.lx, a.ly, a.lz, in_chunks, a.cout, a.sms);
  const ConvPlan& p = a.plan;
  if (p.tx == 0) return -3;
  CUtensorMap map;
  if (encode_planes_map(&map, in_planes, a.lx, a.ly, a.lz, in_chunks, p.pitch, p.ty + 2, 1, in_chunks) != 0) return -2;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !g_attr_set[dev].load(std::memory_order_acquire)) {
    for (const Kernel k : {k_conv_tc<0>, k_conv_tc<1>, k_conv_tc<2>, k_conv_tc<2, true>, k_conv_tc<3>, k_conv_tc<4>,
                           k_conv_tc<6>})
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kConvSmem));
    g_attr_set[dev].store(true, std::memory_order_release);
  }
  const size_t smem = static_cast<size_t>(kConvSmemFixed) + static_cast<size_t>(p.stages) * p.a_bytes +
                      static_cast<size_t>(p.b_slots) * p.b_bytes;
  kernel<<<std::min(p.tiles_x * p.tiles_y * p.tiles_z, a.sms), kConvThreads, smem, st>>>(map, a);
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

int head_blocks(int64_t nv, int sms) { return static_cast<int>(std::min<int64_t>((nv + 255) / 256, sms)); }

void launch_head_backward(const void* u1, const float* hw, int64_t nv, const float* f, const float* g, void* gz,
                          double* partial, double* loss, float* grad, int64_t hw_off, int64_t hb_off, int sms,
                          cudaStream_t st) {
  const int nb = head_blocks(nv, sms);
  k_head_backward<<<nb, 256, 0, st>>>(static_cast<const uint4*>(u1), hw, nv, f, g, static_cast<uint4*>(gz), partial);
  k_head_reduce<<<1, 18 * 32, 0, st>>>(partial, nb, nv, loss, grad, hw_off, hb_off);
}

WgradPlan plan_wgrad(int lx, int ly, int lz, int cin, int cout, int sms) {
  WgradPlan p{};
  p.lz = lz;
  p.cout_chunks = cout / 8;
  p.copies = 3 * cout <= 128 ? 3 : 1;
  p.cin_blocks = cin > 48 ? 2 : 1;
  p.cin_chunks = cin / 8 / p.cin_blocks;
  p.groups = p.cin_blocks * (3 / p.copies);
  p.m = p.copies * cout <= 64 ? 64 : 128;
  const int cols = 3 * 24 * p.cin_chunks;
  p.tmem_cols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
  p.tiles_x = (lx + kWgTx - 1) / kWgTx;
  p.tx = ((lx + p.tiles_x - 1) / p.tiles_x + 15) / 16 * 16;
  p.pitch = p.tx + 2;
  // rows per step: four stages in shared memory, and four steps for every
  // block (each block's partial is written and read once more)
  const int row_bytes = 16 * (3 * p.cin_chunks * p.pitch + p.copies * p.cout_chunks * p.tx);
  int blocks = std::max(sms / p.groups, 1);
  const int by_smem = std::max(static_cast<int>(kWgSmem / kWgStagesMax) / row_bytes, 1);
  const int by_steps = std::max(static_cast<int>(static_cast<int64_t>(ly) * lz * p.tiles_x / (4 * blocks)), 1);
  p.ty = std::min(std::min(by_smem, by_steps), std::min(ly, 256));
  p.tiles_y = (ly + p.ty - 1) / p.ty;
  p.ty = (ly + p.tiles_y - 1) / p.tiles_y;
  p.steps = p.tiles_x * p.tiles_y * lz;
  blocks = std::min(blocks, std::max(p.steps / 4, 1));
  p.blocks = blocks;
  p.copy_bytes = p.ty * p.tx * 16 * p.cout_chunks;
  p.tx_bytes = p.ty * row_bytes;
  p.stage_bytes = (p.tx_bytes + 127) / 128 * 128;
  p.stages = std::min(static_cast<int>(kWgSmem) / p.stage_bytes, kWgStagesMax);
  return p;
}

int64_t wgrad_partial_floats(int lx, int ly, int lz, int cin, int cout, int sms) {
  return static_cast<int64_t>(plan_wgrad(lx, ly, lz, cin, cout, sms).blocks) * 27 * cin * cout;
}

int64_t bias_partial_floats(int lx, int ly, int lz, int cin, int cout, int sms) {
  return static_cast<int64_t>(plan_wgrad(lx, ly, lz, cin, cout, sms).blocks) * cout;
}

int launch_wgrad(const void* x, int cin, int cin_real, const void* gz, int cout, int lx, int ly, int lz,
                 float* partial, float* gw, float* bpartial, float* gb, uint32_t* status, int sms,
                 cudaStream_t st) {
  const WgradPlan p = plan_wgrad(lx, ly, lz, cin, cout, sms);
  if (p.stages < 1 || cout % 16 != 0 || cout > 64 || cin > 96) return -1;
  CUtensorMap xm, gm;
  if (encode_planes_map(&xm, x, lx, ly, lz, cin / 8, p.pitch, p.ty, 3, p.cin_chunks) != 0 ||
      encode_planes_map(&gm, gz, lx, ly, lz, p.cout_chunks, p.tx, p.ty, 1, p.cout_chunks) != 0)
    return -2;
  static std::atomic<bool> attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr[dev].load(std::memory_order_acquire)) {
    cudaFuncSetAttribute(k_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kWgSmem) + 1024);
    attr[dev].store(true, std::memory_order_release);
  }
  k_wgrad_tc<<<dim3(p.blocks, p.groups), kWgThreads, static_cast<size_t>(p.stages) * p.stage_bytes + 1024, st>>>(
      xm, gm, p, partial, bpartial, status);
  const int n = 27 * cin * cout + cout;
  k_wgrad_reduce<<<(n + 31) / 32, 256, 0, st>>>(p, partial, bpartial, cin_real, gw, gb);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -4;
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
  return n_in == 8 ? static_cast<int64_t>(14) * 2 * n_out * 8 : static_cast<int64_t>(9) * n_in * 3 * n_out;
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
