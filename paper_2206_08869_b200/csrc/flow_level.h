// Flow levels of three-conv couplings whose geometry and requantisation fit the compact kernel
// (flow_level.cu): the launch-time plan, the packed meta blocks and the launch interface.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "iodf_dev.h"
#include "level_kernel.h"

namespace iodf {

constexpr int kFlowWarps = 16;                       // requantising warps, four per TMEM lane quarter
constexpr int kFlowWorkers = kFlowWarps * 32;
constexpr int kFlowThreads = kFlowWorkers + 3 * 32;  // + an MMA-issuing warp per tile slot and the weight-loading warp
constexpr int kFlowMaxRing = 12;                     // slots of the weight ring
constexpr int kFlowMaxTiles = 32;                    // of a CTA
constexpr int kFlowMaxSteps = 18;                    // K steps of the first conv
constexpr int kFlowMaxRounds = 5;                    // blocks of 32 columns that a warp requantises of a layer

enum FlowDirect : int { kFlowNine = 1, kFlowRows = 2 };   // forms of the last conv on the hidden operand: an MMA per tap, per row of taps

constexpr int kFlowMaxBlocks = 8;                    // CTAs that share an image (portable cluster size)

// Everything about a level that the kernel needs and that is the same for all its couplings; passed
// by value (constant bank), so that no index computation waits for a global load.
struct FlowPlan {
  int32_t c, h, w, px, ca, cb;   // (h, w, px: of the CTA's block where an image is split)
  int32_t nbx, nby;              // blocks of an image; more than one: a cluster of CTAs, group = 1
  int32_t fh, fw, fpx;           // the whole image
  int32_t halo_bytes[3];         // bytes that a position takes from a neighbour: above / below, beside, at a corner
  int32_t reds[kFlowMaxBlocks];  // products per channel that block r's neighbours add to its accumulator
  int32_t n_couplings, has_prior, is_first, is_last, keep_c;
  int32_t group;                 // images per CTA
  int32_t pg;                    // pixels of the CTA (group * px): plane stride of the flow variable
  // GEMM tiles. A tile is an 8-column block of an image, 16 (m = 128) or 8 (m = 64) rows high, or, at
  // 4 x 4 levels (im2col), up to four whole images of 16 pixels each (m = 64)
  int32_t m, im2col;
  int32_t copies;                // 4 x 4: operand rows hold every image that often, in a lane quarter each (1, or up to four rows of images)
  int32_t tiles;                 // of the CTA
  int32_t tiles_img, tiles_x;    // of an image; 8-column blocks per row
  int32_t rec;                   // bytes of a position's record in the network-input frame
  int32_t paired;                // records are [pixel j | pixel j + 1], eight bytes each
  int32_t wp, frame;             // frame of an image: (h + 2) rows of wp = w + 2 positions
  int32_t plane16;               // 16-byte units between the 16-byte planes of a record
  int32_t sbo16;                 // 16-byte units between 8-row groups of the first conv's operand
  int32_t ks1;                   // its K steps; step s: offset of the first 16-byte chunk from the tile's first position
  uint32_t step[kFlowMaxSteps];  // (mod 2^32) + distance of the second chunk << 16, in 16-byte units
  int32_t pitch;                 // bytes between 16-byte K chunks of the hidden operands
  int32_t acc_stride;            // words per channel plane of the translation accumulator (pg + 4: no bank conflicts)
  // 8 x 8 images, one tile each: the last conv on the hidden operand itself, in a zero-bordered frame (planes of 16 channels,
  // s_h), rather than per-tap partials and their shifted sum. kFlowRows where its accumulators fit, else kFlowNine
  int32_t direct;
  // 1: the second (third) GEMM's K steps start as the blocks of its operand are written, a round of blocks at a time
  int32_t chunk2, chunk3;
  int32_t alias;                 // 1: the third matrix travels through the first one's slot
  int32_t ring;                  // > 0: hidden widths above 256: one tile in flight, weights streamed for every tile in K
  uint32_t ring_slot_bytes;      // steps of 32 bytes through a ring of that many slots at s_w[0]
  int32_t d_col, d3_col, d3_step;// TMEM columns: slot s has its accumulators at s * d_col (the second GEMM's d2_col further
  int32_t d2_col;                // on), those of the last one at d3_col + s * d3_step
  int32_t n_prior;               // columns of the prior head (padded to 16)
  int32_t tmem_cols;
  uint32_t s_v, s_xa, s_xa_end, s_acc, s_a[2], s_h[2], s_h_end, s_meta[2], s_w[3], s_total;
  uint32_t mul_per_img, mul_4px, mul_w2, mul_px, mul_w;
  int64_t z_off, prior_off, z_final_off, d, d_fact;
};
static_assert(sizeof(FlowPlan) < 1024, "travels as a kernel parameter");

// Meta part of a coupling's packed block. Followed by colA[ca], colB[cb] (physical columns of the flow
// variable), OutRq[cb], and per hidden layer the FloatRq constants of its 32-column blocks in thread order (lane & 3, eight
// columns; so that the four addresses of a 16-byte load lie in different banks): 32 multipliers a block, then 32 addends a
// block from the first that has any.
struct __align__(16) FlowLayer { // what a hidden epilogue needs, in one load
  uint8_t ks, nfull, last, plain;// 32-column blocks written, blocks that are full of columns, last block with any, blocks
                                 // that are full and without an addend
  uint16_t off, off_c;           // multipliers of block 0, addends of block nfb, in 16-byte units
  uint32_t beyond;               // what its output holds where the last blocks have no columns
  uint8_t half, nfb, nfi, us;    // half 1: block nfull has 16 columns; blocks from nfb on may have addends, from nfi on a channel
                                 // without floating-point constants: integer form with shift us, multipliers M0
};
struct FlowMeta {
  int32_t in_m0, in_s;
  int32_t n1, n2, n3;            // MMA N of the three GEMMs
  int32_t n3d;                   // N of the last conv in its direct form
  int32_t ks2, ks3;              // K steps of the second and third GEMM = 32-column blocks of their operands
  FlowLayer layer[2];
  int32_t off_colA, off_colB, off_out;
  int32_t pad[13];
};
static_assert(sizeof(FlowMeta) == 128, "meta header is 128 bytes");

cudaError_t configure_flow_kernels(uint32_t max_smem_bytes);
// clusters of `ctas` CTAs that can be resident at once (0 if that cannot be determined); smem_limit: what the
// device allows a block
int max_flow_clusters(int ctas, uint32_t smem_bytes, uint32_t smem_limit);
cudaError_t launch_flow_level(const LevelArgs& args, const FlowPlan& plan, bool inverse, int grid, cudaStream_t stream);

}  // namespace iodf
