// Residual levels (Eq. 3 with the scatter add of Sec. 4.5) whose geometry and requantisation fit the
// overlapped kernel (res_flow.cu): launch-time plan, packed records and the launch interface.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "iodf_dev.h"
#include "level_kernel.h"

namespace iodf {

constexpr int kRfWarps = 16;                        // requantising warps, four per TMEM lane quarter
constexpr int kRfWorkers = kRfWarps * 32;
constexpr int kRfThreads = kRfWorkers + 3 * 32;     // + two MMA-issuing warps and the weight-loading warp
constexpr int kRfTmemCols = 512;                    // two convs of two accumulators of 128 columns
constexpr int kRfMaxSlots = 4;                      // weight ring
constexpr int kRfChunks = 4;                        // 32-channel chunks of the widest activation (128 channels)

// What a conv's epilogue does (see res_flow.cu).
enum RfKind : int32_t { kRfHidden = 0, kRfBranch = 1, kRfOut = 2, kRfPrior = 3 };

// One 3x3 conv: what the loader needs (global memory).
struct RfConv {
  uint32_t w_off, meta_off, meta_bytes;
  int32_t n_pad, nk;             // MMA N, 32-channel chunks of K
  int32_t pad[3];
};
static_assert(sizeof(RfConv) == 32, "32-byte records");
// Its weights: for every chunk kc nine taps [2][n_pad][16 bytes], preceded in the first chunk by the bias rows
// [2][n_pad][16] (they meet a constant operand row 1, c, c, ...). A ring slot holds a chunk.

// Head of a conv's meta block (shared memory), followed by kRfHidden / kRfBranch: float or int32 constants
// [chunk][lane & 3][8] (multipliers), then kRfHidden: addends in the same order; kRfOut / kRfPrior: OutRq[n].
struct RfMeta {
  int32_t kind, n, n_pad, nb;    // nb: 32-column chunks written
  int32_t nk, src, dst;          // buffers: 0 network input of couplings, 1 X, 2 MID (and the prior head's network
                                 // input: a neighbour may write the next one while this CTA still reads it)
  int32_t a_unsigned;
  int32_t nfi;                   // kRfHidden: chunks from here on in integer form
  int32_t us;                    // the conv's shift (integer forms)
  float short_m;                 // kRfBranch: shortcut multiplier (subnormal form)
  int32_t input;                 // first conv of a coupling, prior head: the network input is requantised first,
  int32_t in_m0, in_s;           // with these constants
  uint32_t cols_off;             // offset in the block: colA[] of such a conv, colB[] of kRfOut
  int32_t ls_lo, ls_hi;
  int32_t pad[3];
};
static_assert(sizeof(RfMeta) == 80, "a multiple of 16 bytes");

struct RfPlan {
  int32_t c, h, w, px, ca, cb;
  int32_t n_couplings, convs_per_coupling, has_prior, is_first, is_last, keep_c;
  int32_t bw, bh, nbx, nby;      // block of an image that a CTA holds; blocks per row and column (a cluster per image)
  int32_t group, pg;             // whole images per CTA (one block per image), pixels per CTA
  int32_t m, tiles, small;       // MMA rows, tiles; small: 4 x 4 images
  int32_t wp, plane16;           // frame row pitch and positions per 16-channel plane (16-byte units)
  int32_t xa_chunks;             // 32-channel chunks of the network input
  int32_t n_slots;
  uint32_t slot_bytes, conv_off; // conv_off: RfConv[] in the blob (prior head last)
  uint32_t s_v, s_buf[3], s_buf_end, s_const, s_meta[3], s_ring, s_total;
  int64_t z_off, prior_off, z_final_off, d, d_fact;
};
static_assert(sizeof(RfPlan) < 1024, "travels as a kernel parameter");

cudaError_t configure_res_flow_kernels(uint32_t max_smem_bytes);
// clusters of `ctas` CTAs that can be resident at once (0 if that cannot be determined)
int max_res_flow_clusters(int ctas, uint32_t smem_bytes);
cudaError_t launch_res_flow(const LevelArgs& args, const RfPlan& plan, bool inverse, int ctas, cudaStream_t stream);

}  // namespace iodf
