// tsf_unet.cuh -- declarations shared by the warm-start network's kernels
// (k_unet.cu) and its C ABI (tsf_unet.cu).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace tsf {
namespace unet {

constexpr int kConvStagesMax = 12;             // input planes in flight in a convolution block
constexpr int kConvBSlotsMax = 14;             // taps' weights in shared memory
constexpr size_t kConvSmem = 220 * 1024;       // dynamic shared memory, one block per SM
constexpr int kConvSmemFixed = 1024;           // ... of which alignment
constexpr int kConvTx = 126;                   // voxels of a tile along x: a row with its halo is one TMA run
constexpr uint32_t kUnetErrSpin = 1u << 5;     // a bounded wait gave up (same bit as the solver's)

enum ConvMode { kConvForward = 0, kConvDgrad = 1, kConvHead = 2 };

// Tile, pipeline and grid of one convolution launch (plan_conv).
struct ConvPlan {
  int tx, ty, tz;                   // output voxels of a block
  int pitch, mtiles;                // row pitch tx + 2; operand tiles of 128 flattened positions
  int tiles_x, tiles_y, tiles_z;
  int chunks, taps;                 // input planes; (dy, dx) taps (pairs of taps for a single input plane)
  int stages, b_slots, b_resident;  // z-planes and taps' weights in shared memory; all weights stay
  int a_tx, a_bytes, b_bytes;       // bytes of a z-plane (loaded, reserved) and of a tap's weights
  int tmem_cols;
};

// One 3x3x3 'same' convolution as an implicit GEMM (k_conv_tc).  launch_conv
// fills the plan.
struct ConvArgs {
  int lx, ly, lz;     // grid of input and output (the output of an `up` launch is 2x)
  int cout;           // output channels (multiple of 16, <= 96)
  int mode;           // kConvForward: relu(acc + bias); kConvDgrad: acc masked by mask > 0;
                      // kConvHead: forward, then g0 = f + the 1x1 head, nothing else stored
  int up;             // forward only: store every voxel to its 2x2x2 block of a 2x grid
  void* out;          // output planes (bf16)
  int64_t out_plane0; // first output plane
  const void* mask;   // dgrad: activation whose ReLU masks the output (may be null)
  int64_t mask_plane0;
  const float* bias;  // forward: cout biases (bf16 values)
  const __nv_bfloat16* wpack;  // packed weights (k_pack_weights)
  const float* head;  // kConvHead: 16 weights, then the bias (bf16 values)
  const float* f;
  float* g0;
  uint32_t* status;   // device status word (kUnetErrSpin)
  int sms;            // of the device
  ConvPlan plan;
};

ConvPlan plan_conv(int lx, int ly, int lz, int chunks, int cout, int sms);
int launch_conv(const ConvArgs& a, const void* in_planes, int in_chunks, cudaStream_t st);

void launch_pack_input(const float* f, float tau, int64_t nv, void* x, cudaStream_t st);
void launch_avgpool(const void* in, int in_plane0, int planes, int lx, int ly, int lz, void* out, cudaStream_t st);
void launch_upsample_back(const void* g, int g_plane0, int planes, int lx, int ly, int lz, const void* act_up,
                          int act_plane0, void* out, cudaStream_t st);
void launch_skip_back(const void* gs, int gs_plane0, const void* gp, const void* s, int s_plane0, int planes, int lx,
                      int ly, int lz, void* out, cudaStream_t st);
int head_blocks(int64_t nv, int sms);
void launch_head_backward(const void* u1, const float* hw, int64_t nv, const float* f, const float* g, void* gz,
                          double* partial, double* loss, float* grad, int64_t hw_off, int64_t hb_off, int sms,
                          cudaStream_t st);
// Weight gradient of one convolution (k_wgrad_tc): tile, operand blocks and
// grid (blocks x groups).
struct WgradPlan {
  int tx, ty, pitch, tiles_x, tiles_y, lz, steps;  // voxels of a step, row pitch of x, steps = tiles x z-planes
  int cout_chunks, cin_chunks, cin_blocks;         // planes of gz; planes of x per block, blocks of input channels
  int copies, groups, m, tmem_cols;                // dy copies of gz; launches side by side; M of the MMAs
  int copy_bytes, tx_bytes, stage_bytes, stages;
  int blocks;                                      // blocks per group = partials
};
constexpr int kWgTx = 112;                // voxels of a step along x, at most
constexpr size_t kWgSmem = 208 * 1024;    // stages of a block
WgradPlan plan_wgrad(int lx, int ly, int lz, int cin, int cout, int sms);
int64_t wgrad_partial_floats(int lx, int ly, int lz, int cin, int cout, int sms);
int64_t bias_partial_floats(int lx, int ly, int lz, int cin, int cout, int sms);
int launch_wgrad(const void* x, int cin, int cin_real, const void* gz, int cout, int lx, int ly, int lz,
                 float* partial, float* gw, float* bpartial, float* gb, uint32_t* status, int sms,
                 cudaStream_t st);
void launch_pack_weights(const float* w, int cout_f, int cin_real, int cin_pad, int transpose, void* pack,
                         cudaStream_t st);
int64_t pack_elems(int cout_f, int cin_pad, int transpose);
void launch_round_bf16(const float* in, int64_t n, float* out, cudaStream_t st);
void launch_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float beta1, float beta2,
                 float eps, float bc1, float bc2, cudaStream_t st);
void launch_unpack_planes(const void* in, int plane0, int c_real, int64_t nv, float* out, cudaStream_t st);

}  // namespace unet
}  // namespace tsf
