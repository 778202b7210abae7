// One flow level of three-conv couplings (the arithmetic of level_kernel.cu) in a kernel built to be
// short: a coupling is a chain of a dozen phases that every warp runs once or a few times, so what a
// phase costs is latency (hand-overs, tensor-memory loads, MMA round trips) and instruction fetch. The
// general kernel's 209 KB of code does not fit the instruction caches: its phases took 1 000 - 2 000
// clocks each for fewer than a hundred instructions per warp. This one is a few KB per phase loop.
//
//   * No im2col. The requantised network input sits in shared memory as a zero-bordered frame of
//     16-byte records, and the first conv's operand descriptors point straight into it: a tile is an
//     8-column block of the image, so its 8-row core-matrix groups are image rows, one frame row apart
//     (the descriptor's stride offset), and a tap is a start address. Two 16-byte chunks make a K step;
//     the leading offset is whatever lies between them (the next tap, or the record's next plane).
//     Up to six input channels: a record holds its own pixel and the right neighbour (eight bytes each), so
//     that a row of three taps is one K step. 4 x 4 levels build the operand by hand: whoever
//     requantises a word writes it to the (up to) nine places that need it.
//   * Bias columns are bytes of the records that no channel uses.
//   * Hidden epilogues read 16 rows x 32 columns per unit: four threads share a row, a thread meets the same
//     eight columns in two rows, which halves the loads of constants; the order of the channels within the
//     next GEMM's K is free, so a thread's eight results are eight adjacent operand bytes.
//   * The per-tap partial products of the last conv are added to a pixel-major accumulator (odd
//     stride) with one shared-memory reduction each. 8 x 8 images, one tile each, need none of that (P.direct): their hidden
//     operand is a zero-bordered frame too, and the last conv is taps of it. An MMA of 64 rows takes 23 clocks up to 24 columns and N / 2
//     beyond, and this warp 28 to issue, so with an MMA per tap (kFlowNine) 45 of them took longer than the epilogues before them. With one
//     per row of taps (kFlowRows) it is fifteen of three times the columns; the three products of a pixel lie in neighbouring lanes and
//     meet by shuffles as the translation is applied. K steps start as the blocks of 32 channels are written. 128 images of 48
//     channels: 48 us with per-tap partials, 40 by taps, 37.5 by rows; 256 of 24, two to a CTA: 65, 49.5, 45. The three products
//     need columns: where those of both slots do not fit beside the hidden layers' and a slot has more tiles than one, taps stay.
//   * A lane quarter of a 4 x 4 level's tile is an image. Of a CTA's one image (two) the operands' rows can hold four (two) copies,
//     so that all sixteen warps, not four, share its columns (P.copies; the host's rule says where there is enough to share): 64 images
//     of 96 channels, eight couplings of width 128: 40 -> 37 us, of width 512 95 -> 86.
//   * CTAs of several tiles have two in flight (slots), each with eight of the sixteen workers and an MMA
//     warp of its own, so that one slot's hand-overs and MMAs run under the other's requantisation; CTAs of
//     one tile put all sixteen workers on it. One lane of another warp streams weights and meta blocks.
//   * Weights that do not fit beside two tiles (hidden widths above 256) go through a ring of K steps, one tile in
//     flight (P.ring).
//   * An image may be split over a cluster of CTAs (kSplit): edge pixels of the network input are stored into the
//     neighbours' frames and products across a border added to their accumulators, both asynchronously; the
//     receiver's barriers count the bytes, so that no CTA waits for more than it needs. A neighbour's products of
//     the next coupling must not come before this CTA's sums have been read and cleared. Nothing in an
//     asynchronous store orders the stores that its thread made earlier, so one lane per neighbour releases them at
//     cluster scope: an arrival on the neighbour's network-input barrier after the barrier that ends the
//     translation, acquired by the neighbour's MMA warp, without whose MMAs there are no products. (Overwriting a
//     frame needs no release: the MMAs that read it have completed before anything is sent that lets a neighbour go on.)
//
// What bounds it: the chain of a coupling (7 000 - 9 000 clocks where a CTA has one tile) and 3 000 clocks per tile of 128 pixels:
// requantisation, shifted sum and their hand-overs, at five to nine clocks an instruction and warp (54 % of an SM's issue slots at
// 32 x 32, 41 % at 8 x 8, 34 % at 4 x 4; of 32 x 32's 133 us the phases' skeleton of waits, hand-overs and MMAs takes half). Measured for eight
// couplings of hidden widths 103 - 179 (mean 143), 128 images (general kernel before): 32 x 32 x 12 channels 218 -> 133 us,
// 16 x 16 85 -> 53, 8 x 8 63 -> 37, 4 x 4 70 -> 45; one image, 32 x 32 split in eight: 48. Width 512, 64 images of
// 32 x 32, split in two: 2 357 -> 286 us, the tensor core busy a third of it.
#include <stddef.h>

#include "flow_level.h"
#include "level_device.cuh"

namespace iodf {

namespace {

// Shape of a level's tiles: rows of a tile of images whose sides are multiples of eight, or images of 4 x 4.
enum FlowShapeKind : int { kRows128, kRows64, kImages4x4 };

struct __align__(16) FlowCtl {
  uint64_t xa_ready[2];   // workers (and the neighbours' edge bytes) -> MMA warp, loader: network input of an even / odd
                          // step written (count kFlowWarps and the neighbours' releases; a neighbour may be one step ahead)
  uint64_t acc_full;      // split images: the neighbours' products of a coupling have been added
  uint64_t peers_done;    // split images: the neighbours have read the prior head's input
  uint64_t a_ready[2][kFlowMaxRounds];  // slot's workers -> its MMA warp: a round of blocks of the next hidden operand is
                          // written (all of them: in the first barrier, unless P.chunk2 / chunk3)
  uint64_t dm_ready[2];   // tensor core -> workers: first / second GEMM of the slot's tile complete
  uint64_t d3_ready[2];   // tensor core -> workers: per-tap partials of the slot's tile complete
  uint64_t w_full[kFlowMaxRing], w_empty[kFlowMaxRing];   // weight slots: copy landed / last MMAs (of each tile slot) that read it complete
  uint64_t meta_full[2];
  uint32_t tmem_base;
  uint32_t abort;
  int32_t sink[32];                 // sums of products that no pixel of the CTA takes, one word a lane
  int4 tile[kFlowMaxTiles];         // {image, first row, first column, 16-byte units from the frame's start to that position}
};

static_assert(sizeof(FlowCtl) <= 1024, "the host leaves this much for static shared memory");

struct Flow {
  uint8_t* smem;
  FlowCtl* ctl;
  uint32_t* status;
  uint32_t tmem;
  int tid, warp, lane;
  int nimg, pvalid, tiles;      // images, pixels and tiles of this CTA
  int slots;                    // tile slots in use: 1 or 2
  int rank, by, bx;             // split images: this CTA's block
  uint32_t halo;                // ... and the bytes of network input that its neighbours send each step
  int sl, cs, ncs;              // worker: its slot, its share of a lane quarter's work (cs of ncs warps; of an image's, 4 x 4)
  int image;                    // 4 x 4: image of the tile in this warp's lane quarter
};

// One test, then suspended (spinning warps take issue slots and shared-memory bandwidth from the others).
// Out of line: a dozen inlined copies cost more in instruction fetch than the call does.
__device__ __noinline__ void flow_wait_at(uint32_t bar, uint32_t parity, FlowCtl* ctl, uint32_t* status) {
  if (ptx::mbar_test_wait(bar, parity)) return;
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    if (ptx::mbar_try_wait(bar, parity)) return;
    if (*reinterpret_cast<volatile uint32_t*>(&ctl->abort)) return;      // bounded: see ptx::bounded_wait
  }
  *reinterpret_cast<volatile uint32_t*>(&ctl->abort) = 1;
  atomicExch(status, 1u);
}
__device__ __forceinline__ void flow_wait(const Flow& f, uint64_t* bar, uint32_t parity) {
  const uint32_t b = ptx::smem_u32(bar);
  if (ptx::mbar_try_wait(b, parity)) return;
  flow_wait_at(b, parity, f.ctl, f.status);
}
// for phases that neighbours take part in (split images)
__device__ __forceinline__ void flow_wait_cluster(const Flow& f, uint64_t* bar, uint32_t parity) {
  const uint32_t b = ptx::smem_u32(bar);
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    if (ptx::mbar_try_wait_cluster(b, parity)) return;
    if (*reinterpret_cast<volatile uint32_t*>(&f.ctl->abort)) return;
  }
  *reinterpret_cast<volatile uint32_t*>(&f.ctl->abort) = 1;
  atomicExch(f.status, 1u);
}
__device__ __forceinline__ void flow_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(ptx::smem_u32(bar)) : "memory");
}
// this warp's shared-memory writes (towards the tensor core) and tensor-memory reads are done
// (bytes: what neighbours' asynchronous stores add to the phase, announced by one warp)
__device__ __forceinline__ void flow_hand_over(const Flow& f, uint64_t* bar, uint32_t bytes = 0u) {
  ptx::tc_fence_before();
  ptx::fence_async_smem();
  __syncwarp();
  if (f.lane == 0) {
    if (bytes) ptx::mbar_expect_tx(ptx::smem_u32(bar), bytes);
    else flow_arrive(bar);
  }
}
// the MMA warp's wait for the network input of step i; a neighbour's bytes came through the generic proxy
__device__ __forceinline__ void flow_wait_input(const Flow& f, int i) {
  uint64_t* bar = &f.ctl->xa_ready[i & 1];
  if (!f.halo) {
    flow_wait(f, bar, (uint32_t)(i >> 1) & 1u);
  } else {
    flow_wait_cluster(f, bar, (uint32_t)(i >> 1) & 1u);
    asm volatile("fence.proxy.async;" ::: "memory");
  }
}
// ---- between the CTAs of a split image ----
__device__ __forceinline__ uint32_t flow_peer(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// a word into / a sum onto a neighbour's shared memory; its barrier counts the four bytes when they are there
__device__ __forceinline__ void flow_store_async(uint32_t addr, uint32_t bar, uint32_t v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void flow_red_async(uint32_t addr, uint32_t bar, int32_t v) {
  asm volatile("red.async.relaxed.cluster.shared::cluster.mbarrier::complete_tx::bytes.add.s32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void flow_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ bool flow_block_exists(const FlowPlan& P, const Flow& f, int dy, int dx) {
  return (uint32_t)(f.by + dy) < (uint32_t)P.nby && (uint32_t)(f.bx + dx) < (uint32_t)P.nbx;
}

// Lane L < 9 of the calling warp arrives on barrier `bar` of the neighbour in direction (L / 3 - 1, L % 3 - 1), releasing at
// cluster scope what this CTA's workers wrote before their last barrier.
__device__ __forceinline__ void flow_release_to_neighbours(const FlowPlan& P, const Flow& f, uint64_t* bar) {
  const int dy = f.lane / 3 - 1, dx = f.lane % 3 - 1;
  if (f.lane < 9 && (dy || dx) && flow_block_exists(P, f, dy, dx))
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                     flow_peer(ptx::smem_u32(bar), (uint32_t)(f.rank + dy * P.nbx + dx))) : "memory");
  __syncwarp();
}

__device__ __forceinline__ void worker_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kFlowWorkers) : "memory"); }
__device__ __forceinline__ void mma_barrier() { asm volatile("bar.sync 2, %0;" ::"n"(2 * 32) : "memory"); }      // both slots' MMA warps

// ---- weight and meta loader (one lane) -----------------------------------------------------------------
__device__ void flow_loader(const Flow& f, const FlowPlan& P, const LevelArgs& a, const Steps& st) {
  FlowCtl* ctl = f.ctl;
  uint32_t nl[3] = {0u, 0u, 0u};
  auto copy = [&](uint32_t off, uint32_t bytes, uint32_t dst, uint64_t* bar) {
    const uint32_t b = ptx::smem_u32(bar);
    ptx::mbar_expect_tx(b, bytes);
    ptx::bulk_g2s(ptx::smem_u32(f.smem + dst), a.blob + off, bytes, b);
  };
  auto meta = [&](int step) {
    if (step >= st.nsteps) return;
    const BlockRef& br = step_ref(*a.plan, st, step);
    copy(br.meta_off, br.meta_bytes, P.s_meta[step & 1], &ctl->meta_full[step & 1]);
  };
  auto load = [&](int step, int g) {
    if (step >= st.nsteps || (g > 0 && st.is_prior(step))) return;
    const int s = (P.alias && g == 2) ? 0 : g, part = P.direct && g == 2 ? 3 : g;
    const BlockRef& br = step_ref(*a.plan, st, step);
    const uint32_t off = br.w_off[part], bytes = br.w_bytes[part];
    if (nl[s] > 0) flow_wait(f, &ctl->w_empty[s], (nl[s] - 1u) & 1u);
    ++nl[s];
    copy(off, bytes, P.s_w[s], &ctl->w_full[s]);
  };
  meta(0);
  load(0, 0);
  load(0, 1);
  if (!P.alias) load(0, 2);
  meta(1);
#pragma unroll 1
  for (int i = 0; i < st.nsteps; ++i) {
    if (P.alias) {          // in the order in which the slots become free
      load(i, 2);
      load(i + 1, 1);
      load(i + 1, 0);
    } else {
      load(i + 1, 0);
      load(i + 1, 1);
      load(i + 1, 2);
    }
    // meta slot of step i: its last reader is the pixel pass of step i + 1
    if (i + 2 < st.nsteps) {
      flow_wait(f, &ctl->xa_ready[(i + 1) & 1], (uint32_t)((i + 1) >> 1) & 1u);
      meta(i + 2);
    }
  }
}

// Streamed weights (P.ring): for every tile the K steps of its GEMMs, in order, through the ring, as many to a slot as it
// holds. A copy takes its warp 290 clocks whatever its size, 135 with two warps that take the slots in turn, and runs at over 100 bytes per
// clock and SM. Neither bounds the stream while a slot carries several steps (one warp for all slots: 0.1 % faster on average over
// 192 levels and batches of widths 264 - 512, 3 % either way above 100 us); what does is one tile's GEMMs and epilogues in series.
__device__ __forceinline__ int flow_slot_steps(const FlowPlan& P, int n) { return max(1, (int)(P.ring_slot_bytes >> 5) / n); }

__device__ void flow_loader_ring(const Flow& f, const FlowPlan& P, const LevelArgs& a, const Steps& st, uint32_t which) {
  FlowCtl* ctl = f.ctl;
  const bool lead = ptx::elect_one();
  uint32_t slot = 0, round = 0, turn = which;          // slot of a GEMM's first step; 0 if that is this warp's, else 1
#pragma unroll 1
  for (int i = 0; i < st.nsteps; ++i) {
    const BlockRef& br = step_ref(*a.plan, st, i);
    // meta slot of step i: its last reader was the pixel pass of step i - 1
    if (i >= 2) flow_wait(f, &ctl->xa_ready[(i - 1) & 1], (uint32_t)((i - 1) >> 1) & 1u);
    if (which == 0 && lead) {
      const uint32_t b = ptx::smem_u32(&ctl->meta_full[i & 1]);
      ptx::mbar_expect_tx(b, br.meta_bytes);
      ptx::bulk_g2s(ptx::smem_u32(f.smem + P.s_meta[i & 1]), a.blob + br.meta_off, br.meta_bytes, b);
    }
    const int gemms = st.is_prior(i) ? 1 : 3;
#pragma unroll 1
    for (int t = 0; t < f.tiles; ++t)
#pragma unroll 1
      for (int g = 0; g < gemms; ++g) {
        const uint32_t step = br.w_bytes[g] / br.k_slices[g], all = br.w_bytes[g], bytes = (uint32_t)flow_slot_steps(P, (int)(step >> 5)) * step;
        uint32_t off = turn * bytes, count = (all + bytes - 1) / bytes;
        auto advance = [&](uint32_t& sl, uint32_t& ro, uint32_t by) {
          for (sl += by; sl >= (uint32_t)P.ring; sl -= (uint32_t)P.ring) ++ro;
        };
        uint32_t sl = slot, ro = round;
        advance(sl, ro, turn);
#pragma unroll 1
        for (; off < all; off += 2 * bytes) {
          if (ro > 0) flow_wait(f, &ctl->w_empty[sl], (ro - 1u) & 1u);
          if (lead) {
            const uint32_t b = ptx::smem_u32(&ctl->w_full[sl]), now = min(bytes, all - off);
            ptx::mbar_expect_tx(b, now);
            ptx::bulk_g2s(ptx::smem_u32(f.smem + P.s_w[0] + sl * P.ring_slot_bytes), a.blob + br.w_off[g] + off, now, b);
          }
          advance(sl, ro, 2);
        }
        advance(slot, round, count);
        turn ^= count & 1u;
      }
  }
}

// ---- MMA warp --------------------------------------------------------------------------------------------
// K steps k0 .. k1 - 1 (32 K bytes each) of D (+)= A B^T, n above 256 in two parts, issued by one lane as a straight row. An
// instruction of this warp takes about 13 clocks beside the four workers of its scheduler, so a loop that decided per step whether
// to wait, to issue and to accumulate took 230 clocks a step, the row about 100: 128 images of 32 x 32 144.5 -> 136 us, of 16 x 16
// 57.7 -> 56, of 8 x 8 43.3 -> 40.5.
__device__ __forceinline__ void flow_gemm(uint32_t d, uint32_t al, uint32_t a_step, uint32_t bl, int n, int k0, int k1, uint32_t idesc_m) {
  const uint32_t hi = ptx::kUmmaDescHi, b_step = 2u * (uint32_t)n;
  const int na = n > 256 ? 256 : n;
  const uint32_t idesc = idesc_m | ((uint32_t)(na >> 3) << 17);
  al += (uint32_t)k0 * a_step;
  bl += (uint32_t)k0 * b_step;
  if (ptx::elect_one()) {
    if (n <= 256) {
      ptx::umma_i8_hl(d, al, hi, bl, hi, idesc, k0 > 0 ? 1u : 0u);
#pragma unroll 4
      for (int k = k0 + 1; k < k1; ++k) {
        al += a_step;
        bl += b_step;
        ptx::umma_i8_hl(d, al, hi, bl, hi, idesc, 1u);
      }
    } else {
      const uint32_t idesc2 = idesc_m | ((uint32_t)((n - na) >> 3) << 17);
#pragma unroll 2
      for (int k = k0; k < k1; ++k) {
        ptx::umma_i8_hl(d, al, hi, bl, hi, idesc, k > 0 ? 1u : 0u);
        ptx::umma_i8_hl(d + 256u, al, hi, bl + 256u, hi, idesc2, k > 0 ? 1u : 0u);
        al += a_step;
        bl += b_step;
      }
    }
  }
  __syncwarp();
}

// The last conv in its direct forms, 32-channel chunks k0 .. k1 - 1: a tap is a start address of the operand, and the weights of a
// chunk's tap row are [2][three taps of n rows][16 bytes]. kFlowNine: an MMA of n columns per tap. kFlowRows: one of 3 n columns per
// row of taps, its three products summed by the epilogue.
__device__ __forceinline__ void flow_taps(const FlowPlan& P, uint32_t d, uint32_t al, uint32_t a_hi, uint32_t bl, int n, int k0, int k1,
                                          uint32_t idesc_m) {
  if (ptx::elect_one()) {
    if (P.direct == kFlowRows) {
      const uint32_t idesc = idesc_m | ((uint32_t)((3 * n + 15) >> 4) << 18);
#pragma unroll 1
      for (int k = k0; k < k1; ++k) {
        const uint32_t a = al + (uint32_t)k * 2u * (uint32_t)P.frame + 1u, b = bl + (uint32_t)k * 18u * (uint32_t)n;
#pragma unroll
        for (int u = 0; u < 3; ++u)
          ptx::umma_i8_hl(d, a + (uint32_t)(u * P.wp), a_hi, b + (uint32_t)(6 * u * n), ptx::kUmmaDescHi, idesc, u > 0 || k > 0 ? 1u : 0u);
      }
    } else {
      const uint32_t idesc = idesc_m | ((uint32_t)(n >> 3) << 17);
#pragma unroll 1
      for (int k = k0; k < k1; ++k) {
        const uint32_t a = al + (uint32_t)k * 2u * (uint32_t)P.frame, b = bl + (uint32_t)k * 18u * (uint32_t)n;
#pragma unroll
        for (int u = 0; u < 3; ++u)
#pragma unroll
          for (int v = 0; v < 3; ++v)
            ptx::umma_i8_hl(d, a + (uint32_t)(u * P.wp + v), a_hi, b + (uint32_t)((6 * u + v) * n), ptx::kUmmaDescHi, idesc,
                            u + v > 0 || k > 0 ? 1u : 0u);
      }
    }
  }
  __syncwarp();
}

// MMA warp of tile slot `sl`: tiles sl, sl + 2, ...
template <int kShape>
__device__ void flow_mma(const Flow& f, const FlowPlan& P, const Steps& st, int sl) {
  if (sl >= f.slots) return;
  FlowCtl* ctl = f.ctl;
  uint8_t* smem = f.smem;
  const bool lead = ptx::elect_one();
  const uint32_t idesc_m = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.m >> 4) << 24);     // s8 x s8 -> s32
  // (in a cluster a shared-memory address also carries the CTA's rank above the descriptor's 14 bits)
  const uint32_t xa16 = (ptx::smem_u32(smem + P.s_xa) >> 4) & 0x3FFFu;
  const uint32_t a1_hi = (uint32_t)P.sbo16 | (1u << 14);
  const uint32_t pitch16 = (uint32_t)P.pitch >> 4;
  const uint32_t a_lo = ((ptx::smem_u32(smem + P.s_a[sl]) >> 4) & 0x3FFFu) | (pitch16 << 16);
  const uint32_t dm = f.tmem + (uint32_t)(sl * P.d_col), d2 = dm + (uint32_t)P.d2_col, d3 = f.tmem + (uint32_t)(P.d3_col + sl * P.d3_step);
  const uint32_t h_lo = ((ptx::smem_u32(smem + P.s_h[sl]) >> 4) & 0x3FFFu) | ((uint32_t)P.frame << 16), h_hi = (uint32_t)P.wp | (1u << 14);
  const int s3 = P.alias ? 0 : 2;
  auto commit = [&](uint64_t* bar) { if (lead) ptx::umma_commit(ptx::smem_u32(bar)); };
  uint32_t used[3] = {0u, 0u, 0u}, apar = 0u;
  auto wait_w = [&](int s) { flow_wait(f, &ctl->w_full[s], used[s] & 1u); };
  // the K steps of a hidden operand, issue(k0, k1): written a round of ncs blocks at a time, or all at once
  auto hidden = [&](int ks, bool chunked, auto issue) {
    const int round = kShape != kRows128 && chunked ? f.ncs : ks;
#pragma unroll 1
    for (int k = 0, r = 0; k < ks; k += round, ++r) {
      flow_wait(f, &ctl->a_ready[sl][r], (apar >> r) & 1u);
      apar ^= 1u << r;
      ptx::tc_fence_after();
      issue(k, min(k + round, ks));
    }
  };
#pragma unroll 1
  for (int i = 0; i < st.nsteps; ++i) {
    const bool prior = st.is_prior(i);
    flow_wait(f, &ctl->meta_full[i & 1], (uint32_t)(i >> 1) & 1u);
    const FlowMeta* M = reinterpret_cast<const FlowMeta*>(smem + P.s_meta[i & 1]);
    // (through a shuffle: tells the compiler that the values are the same in all lanes, so that the operands of
    // the MMAs are computed in uniform registers)
    auto uniform = [](int x) { return __shfl_sync(0xFFFFFFFFu, x, 0); };
    const int n1 = prior ? P.n_prior : uniform(M->n1), n2 = uniform(M->n2), n3 = uniform(kShape == kRows64 && P.direct ? M->n3d : M->n3);
    const int ks2 = uniform(M->ks2), ks3 = uniform(M->ks3);
    wait_w(0);
    ++used[0];
    const uint32_t b1 = ((ptx::smem_u32(smem + P.s_w[0]) >> 4) & 0x3FFFu) | ((uint32_t)n1 << 16);
    const uint32_t b2 = ((ptx::smem_u32(smem + P.s_w[1]) >> 4) & 0x3FFFu) | ((uint32_t)n2 << 16);
    const uint32_t b3 = ((ptx::smem_u32(smem + P.s_w[s3]) >> 4) & 0x3FFFu) | ((uint32_t)(kShape == kRows64 && P.direct ? 3 * n3 : n3) << 16);
    const uint32_t idesc1 = idesc_m | ((uint32_t)(n1 >> 3) << 17);
    // first conv of a tile: steps from the table {start offset, leading offset}
    auto first_conv = [&](int t, uint32_t d) {
      const uint32_t base = xa16 + (uint32_t)uniform(ctl->tile[t].w);
      uint32_t bl = b1;
      if (ptx::elect_one()) {
        ptx::umma_i8_hl(d, base + P.step[0], a1_hi, bl, ptx::kUmmaDescHi, idesc1, 0u);
#pragma unroll 4
        for (int s = 1; s < P.ks1; ++s) {
          bl += 2u * (uint32_t)n1;
          ptx::umma_i8_hl(d, base + P.step[s], a1_hi, bl, ptx::kUmmaDescHi, idesc1, 1u);
        }
      }
      __syncwarp();
    };
    flow_wait_input(f, i);
    ptx::tc_fence_after();
    if (prior) {
#pragma unroll 1
      for (int t = sl; t < f.tiles; t += 2) first_conv(t, f.tmem + (uint32_t)(t * P.n_prior));
      commit(&ctl->dm_ready[sl]);
      commit(&ctl->w_empty[0]);
      continue;
    }
#pragma unroll 1
    for (int t = sl; t < f.tiles; t += 2) {
      // the slot's accumulator has been drained: its last tile's third GEMM was issued after that
      const bool last = t + 2 >= f.tiles;
      // A step starts both slots at once, and MMAs issued in turn complete together: both slots would wait for the sum of their GEMMs, at
      // this one and, in step, at every later one. Slot 0's go first (two images of 8 x 8 with 48 channels 53 -> 49 us, of 24 45 -> 43,
      // 128 images of 16 x 16 55.2 -> 53.2, of 32 x 32 132 -> 131.5; slot 1 a whole GEMM and epilogue behind: 32 x 32 133). Both
      // warps wait, slot 0's for one that is there by then: a warp that only arrived would run ahead once a wait has given up, and two
      // of its arrivals would stand for one of the other's, which would then wait for good.
      const bool order = f.slots == 2 && t == sl;
      if (order && sl == 1) mma_barrier();
      first_conv(t, dm);
      commit(&ctl->dm_ready[sl]);
      if (order && sl == 0) mma_barrier();
      if (last) commit(&ctl->w_empty[0]);
      if (t == sl) wait_w(1);
      hidden(ks2, P.chunk2, [&](int k0, int k1) { flow_gemm(d2, a_lo, 2u * pitch16, b2, n2, k0, k1, idesc_m); });
      commit(&ctl->dm_ready[sl]);
      if (last) commit(&ctl->w_empty[1]);
      if (t == sl) wait_w(s3);
      if (kShape == kRows64 && P.direct) {
        hidden(ks3, P.chunk3, [&](int k0, int k1) { flow_taps(P, d3, h_lo, h_hi, b3, n3, k0, k1, idesc_m); });
      } else {
        hidden(ks3, false, [&](int k0, int k1) { flow_gemm(d3, a_lo, 2u * pitch16, b3, n3, k0, k1, idesc_m); });
      }
      commit(&ctl->d3_ready[sl]);
      if (last) commit(&ctl->w_empty[s3]);
    }
    ++used[1];
    ++used[s3];
  }
}

// MMA warp of levels with streamed weights: one tile at a time, all accumulators from column 0 on. A step of 32 K bytes keeps
// the tensor core 256 clocks at width 512, and a wait, a commit and the bookkeeping of a slot took this warp 450 (with a copy
// per step for every GEMM and a wait for each): 64 images of 32 x 32 360 -> 288 us, of 4 x 4 112 -> 98.
__device__ void flow_mma_ring(const Flow& f, const FlowPlan& P, const Steps& st) {
  FlowCtl* ctl = f.ctl;
  uint8_t* smem = f.smem;
  auto uniform = [](int x) { return __shfl_sync(0xFFFFFFFFu, x, 0); };
  const uint32_t idesc_m = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.m >> 4) << 24);
  const uint32_t xa16 = (ptx::smem_u32(smem + P.s_xa) >> 4) & 0x3FFFu, hi = ptx::kUmmaDescHi;
  const uint32_t a1_hi = (uint32_t)P.sbo16 | (1u << 14), pitch16 = (uint32_t)P.pitch >> 4;
  const uint32_t a_lo = ((ptx::smem_u32(smem + P.s_a[0]) >> 4) & 0x3FFFu) | (pitch16 << 16);
  const uint32_t w16 = (ptx::smem_u32(smem + P.s_w[0]) >> 4) & 0x3FFFu, slot16 = P.ring_slot_bytes >> 4;
  const uint32_t full0 = ptx::smem_u32(&ctl->w_full[0]), last = full0 + 8u * (uint32_t)(P.ring - 1);
  constexpr uint32_t kToEmpty = (uint32_t)(offsetof(FlowCtl, w_empty) - offsetof(FlowCtl, w_full));
  const bool lead = ptx::elect_one();
  uint32_t bar = full0, bw = w16, wpar = 0, apar = 0;          // next slot: its barrier, its address, the phase's parity
  bool full = false;                           // its copy has landed (asked ahead: a wait takes a hundred clocks)
  // one GEMM: K step s reads A at `al`, then step(s, al) is the next one; N above 256 in two parts
  auto gemm = [&](uint32_t d, int n, int ks, uint32_t al, auto step, uint32_t ahi, uint64_t* done) {
    const int na = min(n, 256), sp = flow_slot_steps(P, n);
    const uint32_t idesc = idesc_m | ((uint32_t)(na >> 3) << 17), idesc2 = idesc_m | ((uint32_t)((n - na) >> 3) << 17), lbo = (uint32_t)n << 16;
    uint32_t acc = 0;
    int left = sp;
#pragma unroll 1
    for (int s = 0; s < ks;) {
      if (!full) flow_wait_at(bar, wpar, ctl, f.status);
      ptx::tc_fence_after();
      const uint32_t empty = bar + kToEmpty;
      uint32_t bl = bw | lbo;
      if (bar == last) { bar = full0; bw = w16; wpar ^= 1u; }
      else { bar += 8u; bw += slot16; }
      full = ptx::mbar_test_wait(bar, wpar);
      for (left = sp; ; bl += 2u * (uint32_t)n) {
        if (lead) ptx::umma_i8_hl(d, al, ahi, bl, hi, idesc, acc);
        if (n > 256 && lead) ptx::umma_i8_hl(d + 256u, al, ahi, bl + 256u, hi, idesc2, acc);
        acc = 1u;
        ++s;
        al = step(s, al);
        if (--left == 0 || s == ks) break;
      }
      if (lead) ptx::umma_commit(empty);
    }
    if (done && lead) ptx::umma_commit(ptx::smem_u32(done));
  };
  auto wait_a = [&]() {
    flow_wait(f, &ctl->a_ready[0][0], apar);
    apar ^= 1u;
    ptx::tc_fence_after();
  };
  auto hidden = [&](int, uint32_t al) { return al + 2u * pitch16; };
#pragma unroll 1
  for (int i = 0; i < st.nsteps; ++i) {
    const bool prior = st.is_prior(i);
    flow_wait(f, &ctl->meta_full[i & 1], (uint32_t)(i >> 1) & 1u);
    const FlowMeta* M = reinterpret_cast<const FlowMeta*>(smem + P.s_meta[i & 1]);
    const int n1 = prior ? P.n_prior : uniform(M->n1), n2 = uniform(M->n2), n3 = uniform(M->n3);
    const int ks2 = uniform(M->ks2), ks3 = uniform(M->ks3);
    flow_wait_input(f, i);
    ptx::tc_fence_after();
#pragma unroll 1
    for (int t = 0; t < f.tiles; ++t) {
      const uint32_t base = xa16 + (uint32_t)uniform(ctl->tile[t].w);
      auto first = [&](int s, uint32_t) { return base + P.step[min(s, kFlowMaxSteps - 1)]; };
      if (prior) {
        gemm(f.tmem + (uint32_t)(t * P.n_prior), n1, P.ks1, first(0, 0u), first, a1_hi, t + 1 == f.tiles ? &ctl->dm_ready[0] : nullptr);
        continue;
      }
      if (t > 0) wait_a();                     // the last tile's partials have been summed
      gemm(f.tmem, n1, P.ks1, first(0, 0u), first, a1_hi, &ctl->dm_ready[0]);
      wait_a();
      gemm(f.tmem, n2, ks2, a_lo, hidden, hi, &ctl->dm_ready[0]);
      wait_a();
      gemm(f.tmem, n3, ks3, a_lo, hidden, hi, &ctl->d3_ready[0]);
    }
  }
}

// ---- workers ---------------------------------------------------------------------------------------------
// Integer form (rare: blocks with a channel that has no floating-point constants)
__device__ __forceinline__ uint32_t flow_integer_one(uint32_t acc, float m, int us) {
  const long long p = (long long)(int)acc * (long long)__float_as_int(m) + (1ll << (30 + us));
  return (uint32_t)max(0, (int)(p >> 32) >> (us - 1));
}

// Where a hidden epilogue writes: this thread's first row, block 0; bytes to the next block and to the row eight further on
struct HiddenOut {
  uint8_t* at;
  int block, row;
};

// Hidden epilogue of one tile: accumulator columns at `taddr` (this warp's lane quarter) -> bytes of the next GEMM's
// operand, 32-column blocks, dealt to the quarter's warps; rows in halves of 16. A thread meets the same eight columns in all
// its rows, so their constants are loaded once per block: the four bytes per channel that a broadcast load returns to every
// lane bound the epilogue (addends loaded for all channels: 161 -> 178 us for a 32 x 32 level). Beyond the columns the operand
// holds constants.
template <int kShape>
__device__ __forceinline__ void flow_hidden(const Flow& f, const FlowPlan& P, uint32_t taddr, const uint8_t* __restrict__ mb, int layer,
                                            const HiddenOut ho, bool chunked, uint64_t* ready, uint32_t parity) {
  constexpr int kHalves = kShape == kRows128 ? 2 : 1;
  // everything that does not depend on the accumulator comes before the wait for it
  const FlowLayer L = reinterpret_cast<const FlowMeta*>(mb)->layer[layer];
  const uint8_t* t = mb + 16 * L.off + (f.lane & 3) * 32;
  const int row = kShape == kRows64 ? ho.row : 128;
  auto put = [&](uint8_t* to, uint2 w) {
    *reinterpret_cast<uint2*>(to) = w;
    if constexpr (kShape == kImages4x4)
#pragma unroll
      for (int c = 1; c < 4; ++c)
        if (c < P.copies) *reinterpret_cast<uint2*>(to + 256 * c) = w;
  };
  uint64_t* done = f.ctl->a_ready[f.sl];
  flow_wait(f, ready, parity);
  ptx::tc_fence_after();
#pragma unroll 1
  for (int b0 = 0; b0 < L.ks; b0 += f.ncs) {
    const int b = b0 + f.cs;
    if (b < L.ks) {
      uint32_t r[kHalves][16];
      const uint32_t ta = taddr + (uint32_t)(min(b, (int)L.last) << 5);
#pragma unroll
      for (int h = 0; h < kHalves; ++h) ptx::tmem_ld_16x32(ta + ((uint32_t)h << 20), r[h]);
      const float4* tb = reinterpret_cast<const float4*>(t + b * 128);
      const float4 m0 = tb[0], m1 = tb[1];
      const float m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
      uint8_t* o = ho.at + b * ho.block;
      // the eight bytes of a thread's row (e = 0: the upper one, 1: eight further on) of a half
      auto pack = [&](int h, int e) {
        return make_uint2(pack4_sat((int)r[h][2 * e], (int)r[h][2 * e + 1], (int)r[h][2 * e + 4], (int)r[h][2 * e + 5]),
                          pack4_sat((int)r[h][2 * e + 8], (int)r[h][2 * e + 9], (int)r[h][2 * e + 12], (int)r[h][2 * e + 13]));
      };
      ptx::tmem_ld_wait16(r[0]);
#pragma unroll
      for (int h = 1; h < kHalves; ++h) ptx::tmem_ld_wait16_nosync(r[h]);
      if (b < L.plain) {                           // (in one piece: nothing between the multiplications and the stores)
#pragma unroll
        for (int h = 0; h < kHalves; ++h) {
#pragma unroll
          for (int k = 0; k < 16; ++k) r[h][k] = (uint32_t)FloatRq::one(r[h][k], m[2 * (k >> 2) + (k & 1)], 0.f);
#pragma unroll
          for (int e = 0; e < 2; ++e) put(o + (2 * h + e) * row, pack(h, e));
        }
      } else {
        if (b < L.nfi) {
          float4 c0 = make_float4(0.f, 0.f, 0.f, 0.f), c1 = c0;
          if (b >= L.nfb) {
            const float4* tc = reinterpret_cast<const float4*>(mb + 16 * L.off_c + (f.lane & 3) * 32 + (b - L.nfb) * 128);
            c0 = tc[0];
            c1 = tc[1];
          }
          const float c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
          for (int h = 0; h < kHalves; ++h)
#pragma unroll
            for (int k = 0; k < 16; ++k) r[h][k] = (uint32_t)FloatRq::one(r[h][k], m[2 * (k >> 2) + (k & 1)], c[2 * (k >> 2) + (k & 1)]);
        } else {
#pragma unroll
          for (int h = 0; h < kHalves; ++h)
#pragma unroll
            for (int k = 0; k < 16; ++k) r[h][k] = flow_integer_one(r[h][k], m[2 * (k >> 2) + (k & 1)], L.us);
        }
        const bool tail = b >= L.nfull, none = b > L.nfull || !L.half;
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            uint2 w = pack(h, e);
            if (tail) w = make_uint2(none ? L.beyond : w.x, L.beyond);
            put(o + (2 * h + e) * row, w);
          }
      }
    }
    if (kShape != kRows128 && chunked) flow_hand_over(f, done++);
  }
  if (kShape == kRows128 || !chunked) flow_hand_over(f, done);
}

// rq with the shift folded to the high word; the host admits only shifts s >= 1 to this kernel
__device__ __forceinline__ int32_t rq_hi(int32_t a, const OutRq o) {
  const long long c64 = (long long)(((unsigned long long)o.c_hi << 32) | (unsigned long long)o.c_lo);
  return (int32_t)(((long long)a * (long long)o.m0 + c64) >> 32) >> (o.s - 1);
}

// Per-tap partials of tile t -> accumulator. A lane quarter is kR rows of the tile's eight columns, and a
// thread holds a column: the three vertical taps of one horizontal tap v meet in its registers, so unit
// (granule of 8 channels, v) costs kR + 2 reductions per channel instead of 3 kR. Products whose output
// pixel is outside the image are dropped (zero padding), or added to the neighbour's accumulator where an image is split.
template <int kR, bool kSplit>
__device__ __forceinline__ void flow_sum(const Flow& f, const FlowPlan& P, int t, uint32_t taddr, int32_t* __restrict__ acc,
                                         uint64_t* ready, uint32_t parity) {
  const int ng = (P.cb + 7) >> 3;
  const int4 tp = f.ctl->tile[t];
  const int i0 = tp.y + (f.warp & 3) * kR, j0 = tp.z + (f.lane >> 2) + 1, ch0 = 2 * (f.lane & 3);
  const uint32_t row = (uint32_t)P.w * 4u, next_ch = (uint32_t)P.acc_stride * 4u, du = (uint32_t)(3 * ng) << 3;
  // output row i0 - 1, the column right of the thread's (v = 0), the thread's channels of granule 0
  const uint32_t dst0 = ptx::smem_u32(acc + ch0 * P.acc_stride + tp.x * P.px + (i0 - 1) * P.w + j0);
  const bool top = i0 > 0, bottom = i0 + kR < P.h;
  const uint32_t sink = ptx::smem_u32(&f.ctl->sink[f.lane]);
  int g = 0, v = f.ncs == 2 ? (f.cs ^ (t >> 1)) & 1 : f.cs;       // (two warps: which of them has the odd unit alternates)
  flow_wait(f, ready, parity);
  ptx::tc_fence_after();
#pragma unroll 1
  for (;; v += f.ncs) {
    while (v >= 3) { v -= 3; ++g; }
    if (g >= ng) break;
    uint32_t r[3][kR / 2][4];
    const uint32_t col = taddr + (uint32_t)((v * ng + g) << 3);
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
      for (int h = 0; h < kR / 2; ++h) ptx::tmem_ld_16x8(col + ((uint32_t)h << 20) + (uint32_t)u * du, r[u][h]);
    uint32_t dst = dst0 + (uint32_t)(g * 8) * next_ch - (uint32_t)(4 * v);
    // Products that belong nowhere go to the lane's sink: a predicated reduction is compiled to branches, forty of them in a
    // unit, which took longer than all the rest of it (128 images of 32 x 32: 161 -> 145 us, of 16 x 16: 63.5 -> 57).
    const bool ok = (uint32_t)(j0 - v) < (uint32_t)P.w && g * 8 + ch0 < P.cb;
    const uint32_t to0 = ok ? dst : sink, to1 = ok ? dst + next_ch : sink, step = ok ? row : 0u;
    // split images: where the row above, the quarter's own rows and the row below go if not to this CTA (-1: nowhere)
    int away[3] = {-1, -1, -1};
    uint32_t away_at[3] = {0, 0, 0};
    bool any = false;
    if constexpr (kSplit) {
      const int dx = j0 < v ? -1 : (j0 - v >= P.w ? 1 : 0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int dy = k == 0 && i0 == 0 ? -1 : (k == 2 && i0 + kR == P.h ? 1 : 0);
        if ((dy || dx) && flow_block_exists(P, f, dy, dx) && g * 8 + ch0 < P.cb) {
          away[k] = f.rank + dy * P.nbx + dx;
          away_at[k] = (uint32_t)(dy * P.h * P.w + dx * P.w) * 4u;
        }
      }
      any = __any_sync(0xFFFFFFFFu, away[0] >= 0 || away[1] >= 0 || away[2] >= 0);
    }
    ptx::tmem_ld_wait4(r[0][0]);
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
      for (int h = 0; h < kR / 2; ++h) ptx::tmem_ld_wait4_nosync(r[u][h]);
#pragma unroll
    for (int o = -1; o <= kR; ++o) {
      int sum[2] = {0, 0};
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int i = o + u - 1;
        if (i < 0 || i >= kR) continue;
        sum[0] += (int)r[u][i >> 1][2 * (i & 1)];
        sum[1] += (int)r[u][i >> 1][2 * (i & 1) + 1];
      }
      const bool in = o < 0 ? top : (o < kR || bottom);
      ptx::red_add_s32_always(in ? to0 + (uint32_t)(o + 1) * step : sink, sum[0]);
      ptx::red_add_s32_always(in ? to1 + (uint32_t)(o + 1) * step : sink, sum[1]);
      if constexpr (kSplit) {
        const int k = o < 0 ? 0 : (o == kR ? 2 : 1);
        if (any && away[k] >= 0) {
          const uint32_t at = flow_peer(dst - away_at[k], (uint32_t)away[k]), bar = flow_peer(ptx::smem_u32(&f.ctl->acc_full), (uint32_t)away[k]);
          flow_red_async(at, bar, sum[0]);
          flow_red_async(at + next_ch, bar, sum[1]);
        }
      }
      dst += row;
    }
  }
}

// 4 x 4 levels: a lane quarter is a whole image, so the nine taps meet by shuffles and the translation is
// applied on the spot, without an accumulator. Lane T holds pixels T / 4 and T / 4 + 8: rows 0, 2 in the lower
// half-warp, 1, 3 in the upper one.
template <bool kInv>
__device__ __forceinline__ void flow_sum_4x4(const Flow& f, const FlowPlan& P, int t, uint32_t taddr, const uint8_t* mb,
                                             int32_t* __restrict__ v, uint64_t* ready, uint32_t parity) {
  const int ng = (P.cb + 7) >> 3, lane = f.lane, j = (lane >> 2) & 3;
  const FlowMeta* M = reinterpret_cast<const FlowMeta*>(mb);
  const int32_t* colB = reinterpret_cast<const int32_t*>(mb + M->off_colB);
  const OutRq* orq = reinterpret_cast<const OutRq*>(mb + M->off_out);
  const bool odd = lane >= 16;
  // a unit's constants and its part of the flow variable, which nobody else writes: the first unit's before the wait
  int32_t* vq = v + (4 * t + f.image) * 16 + (lane >> 2);
  OutRq o[2];
  int32_t* vp[2];
  uint32_t x[2][2];
  bool okc = false;
  auto fetch = [&](int g) {
    const int ch = g * 8 + 2 * (lane & 3);
    okc = ch < P.cb;                             // (cb is even)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      o[e] = orq[okc ? ch + e : 0];
      vp[e] = vq + colB[okc ? ch + e : 0] * P.pg;
      x[e][0] = (uint32_t)vp[e][0];
      x[e][1] = (uint32_t)vp[e][8];
    }
  };
  fetch(f.cs);
  flow_wait(f, ready, parity);
  ptx::tc_fence_after();
#pragma unroll 1
  for (int g = f.cs; g < ng;) {
    int lo[2] = {0, 0}, hi[2] = {0, 0};
    uint32_t ra[3][3][4];
#pragma unroll
    for (int tv = 0; tv < 3; ++tv)
#pragma unroll
      for (int u = 0; u < 3; ++u) ptx::tmem_ld_16x8(taddr + (uint32_t)(((3 * u + tv) * ng + g) << 3), ra[tv][u]);
    ptx::tmem_ld_wait4(ra[0][0]);
#pragma unroll
    for (int tv = 0; tv < 3; ++tv) {
#pragma unroll
      for (int u = 0; u < 3; ++u) ptx::tmem_ld_wait4_nosync(ra[tv][u]);
      const uint32_t (&r)[3][4] = ra[tv];
      const bool ok = (uint32_t)(j + tv - 1) < 4u;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int a0 = __shfl_xor_sync(0xFFFFFFFFu, (int)r[0][e], 16), a2 = __shfl_xor_sync(0xFFFFFFFFu, (int)r[0][e + 2], 16);
        const int b0 = __shfl_xor_sync(0xFFFFFFFFu, (int)r[2][e], 16), b2 = __shfl_xor_sync(0xFFFFFFFFu, (int)r[2][e + 2], 16);
        const int s0 = (int)r[1][e] + (odd ? a0 + b2 : b0), s2 = (int)r[1][e + 2] + (odd ? a2 : a0 + b2);
        const int t0 = __shfl_sync(0xFFFFFFFFu, s0, lane + 4 * (tv - 1)), t2 = __shfl_sync(0xFFFFFFFFu, s2, lane + 4 * (tv - 1));
        lo[e] += ok ? t0 : 0;
        hi[e] += ok ? t2 : 0;
      }
    }
    if (okc) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint32_t y0 = (uint32_t)rq_hi(lo[e], o[e]), y8 = (uint32_t)rq_hi(hi[e], o[e]);
        vp[e][0] = (int32_t)(kInv ? x[e][0] - y0 : x[e][0] + y0);
        vp[e][8] = (int32_t)(kInv ? x[e][1] - y8 : x[e][1] + y8);
      }
    }
    g += f.ncs;
    if (g < ng) fetch(g);
  }
}

// Last conv in its direct form: the accumulators of tile t (a lane quarter: 16 pixels) are the translation. Unit = 8 channels.
template <bool kInv>
__device__ __forceinline__ void flow_out(const Flow& f, const FlowPlan& P, int t, uint32_t taddr, const uint8_t* mb, int32_t* __restrict__ v,
                                         uint64_t* ready, uint32_t parity) {
  const FlowMeta* M = reinterpret_cast<const FlowMeta*>(mb);
  const int32_t* colB = reinterpret_cast<const int32_t*>(mb + M->off_colB);
  const OutRq* orq = reinterpret_cast<const OutRq*>(mb + M->off_out);
  int32_t* vq = v + (4 * t + (f.warp & 3)) * 16 + (f.lane >> 2);
  // a unit's constants and its part of the flow variable, which nobody else writes: the first unit's before the wait
  OutRq o[2];
  int32_t* vp[2];
  uint32_t x[2][2];
  bool ok = false;
  auto fetch = [&](int g) {
    const int ch = 8 * g + 2 * (f.lane & 3);
    ok = ch < P.cb;                              // (cb is even)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      o[e] = orq[ok ? ch + e : 0];
      vp[e] = vq + colB[ok ? ch + e : 0] * P.pg;
      x[e][0] = (uint32_t)vp[e][0];
      x[e][1] = (uint32_t)vp[e][8];
    }
  };
  int g = f.cs;
  fetch(g);
  flow_wait(f, ready, parity);
  ptx::tc_fence_after();
#pragma unroll 1
  while (8 * g < P.cb) {
    uint32_t r[4];
    if (P.direct == kFlowRows) {       // products of the taps left, middle and right: of the columns x - 1, x and x + 1
      uint32_t r0[4], r2[4];
      const uint32_t at = taddr + (uint32_t)(8 * g), n = (uint32_t)M->n3d;
      ptx::tmem_ld_16x8(at, r0);
      ptx::tmem_ld_16x8(at + n, r);
      ptx::tmem_ld_16x8(at + 2u * n, r2);
      ptx::tmem_ld_wait4(r0);
      ptx::tmem_ld_wait4_nosync(r);
      ptx::tmem_ld_wait4_nosync(r2);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t left = __shfl_up_sync(0xFFFFFFFFu, r0[k], 4), right = __shfl_down_sync(0xFFFFFFFFu, r2[k], 4);
        r[k] += (f.lane >= 4 ? left : 0u) + (f.lane < 28 ? right : 0u);
      }
    } else {
      ptx::tmem_ld_16x8(taddr + (uint32_t)(8 * g), r);
      ptx::tmem_ld_wait4(r);
    }
    if (ok) {
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint32_t y = (uint32_t)rq_hi((int32_t)r[e + 2 * k], o[e]);
          vp[e][8 * k] = (int32_t)(kInv ? x[e][k] - y : x[e][k] + y);
        }
    }
    g += f.ncs;
    if (8 * g < P.cb) fetch(g);
  }
}

// Prior head: accumulators of all tiles -> mu and clipped log-scale index in global memory. Unit = (tile, 8 columns). Constants
// are loaded ahead of the stores, which the compiler must not move them across, and a column's place and bounds are the same in all
// lanes: a unit took a warp 1 700 clocks, a quarter of them for eight 64-bit addresses (with flow_out's and flow_sum_4x4's loads ahead
// of their waits, 128 images of 64 x 64: 255.2 -> 253.9 us; 256 of 32 x 32: 152.1 -> 150.7).
template <bool kSplit, int kShape>
__device__ void flow_prior(const Flow& f, const FlowPlan& P, const LevelArgs& a, const PriorMeta* M, int img0) {
  const int wq = f.warp & 3, hs = kShape == kRows128 ? 1 : 0;
  const OutRq* orq = reinterpret_cast<const OutRq*>(reinterpret_cast<const uint8_t*>(M) + M->off_out);
  const int ng = (2 * P.cb + 7) >> 3, ls_lo = M->ls_lo, ls_hi = M->ls_hi;
  const int lane_row = (wq << (4 + hs)) + (f.lane & (hs ? 31 : 15)), plane = kSplit ? P.fpx : P.px;
  const uint32_t to_scale = (uint32_t)(P.d_fact - P.cb * plane);          // from a channel's mu on to the channel's scale, less P.cb planes
  int t = f.sl, g = f.cs;
#pragma unroll 1
  for (; ; g += f.ncs) {
    while (g >= ng) { g -= ng; t += f.slots; }
    if (t >= f.tiles) break;
    uint32_t r[8];
    ptx::tmem_ld8(f.tmem + (uint32_t)(t * P.n_prior + g * 8) + ((uint32_t)(wq * 32) << 16), r);
    const int4 tp = f.ctl->tile[t];
    int img = tp.x, at = (tp.y + (lane_row >> 3)) * P.w + tp.z + (lane_row & 7);
    if constexpr (kSplit) at = (f.by * P.h + tp.y + (lane_row >> 3)) * P.fw + f.bx * P.w + tp.z + (lane_row & 7);
    if (kShape == kImages4x4) { img += f.image; at = lane_row & 15; }
    int32_t* mu = a.prior + (size_t)(img0 + img) * (size_t)(2 * P.d_fact) + P.prior_off + at;
    OutRq o[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = orq[min(g * 8 + e, 2 * P.cb - 1)];
    ptx::tmem_ld_wait8(r);
    if (!(hs || f.lane < 16) || img >= f.nimg) continue;
    // (the same place for all lanes: offsets and bounds in uniform registers)
    uint32_t off = (uint32_t)(g * 8 * plane);
#pragma unroll
    for (int e = 0; e < 8; ++e, off += (uint32_t)plane) {
      const int col = g * 8 + e;
      const bool scale = col >= P.cb;
      const int32_t y = clampi(rq_hi((int32_t)r[e], o[e]), scale ? ls_lo : INT32_MIN, scale ? ls_hi : INT32_MAX);
      if (col < 2 * P.cb) mu[off + (scale ? to_scale : 0u)] = y;
    }
  }
}

// Work split of the pixel pass: thread -> (pair of neighbouring pixels, part) with `parts` threads per
// pair. With one part a thread has all channels of its pixels and needs no barrier between the two halves of the pass.
struct PixelMap {
  int p, j, parts;              // first pixel (-1: none), part
  int32_t* v;                   // the pair in plane 0 of the flow variable
  int32_t* acc;                 // and of the accumulator
  uint8_t* rec;                 // its first pixel's record (4 x 4 levels: operand row)
  int dy, dx;                   // split images: the edge of the block that the pair is on (at most one of each: blocks are
                                // eight rows and columns or more)
  uint32_t taps;                // 4 x 4 levels: bit t (16 + t): the first (second) pixel's value is read by tap t of a pixel
};

template <bool kInv>
__device__ __forceinline__ void flow_translate(const FlowPlan& P, const PixelMap& pm, const uint8_t* mb) {
  const FlowMeta* M = reinterpret_cast<const FlowMeta*>(mb);
  const int32_t* colB = reinterpret_cast<const int32_t*>(mb + M->off_colB);
  const OutRq* orq = reinterpret_cast<const OutRq*>(mb + M->off_out);
#pragma unroll 1
  for (int c = pm.j; c < P.cb; c += pm.parts) {
    int2* ap = reinterpret_cast<int2*>(pm.acc + c * P.acc_stride);
    uint2* vp = reinterpret_cast<uint2*>(pm.v + colB[c] * P.pg);
    const OutRq o = orq[c];
    const int2 s = *ap;
    uint2 x = *vp;
    *ap = make_int2(0, 0);
    const uint32_t t0 = (uint32_t)rq_hi(s.x, o), t1 = (uint32_t)rq_hi(s.y, o);
    x.x = kInv ? x.x - t0 : x.x + t0;
    x.y = kInv ? x.y - t1 : x.y + t1;
    *vp = x;
  }
}

// network input: words of four requantised channels (then the constants 1, 127, 127, ...) into the frame
template <bool kSplit, int kShape>
__device__ __forceinline__ void flow_requant(const Flow& f, const FlowPlan& P, const PixelMap& pm, uint64_t* input, const int32_t* cols, int32_t m0, int32_t s) {
  const int nw = (P.ca + 3) >> 2;
  const long long rnd = 1ll << (30 + s);
  // Whole images of 1 024 pixels, up to six channels: a thread has both words of its two pixels, so its first record is one 16-byte store and
  // its part of either neighbour's one of eight; word by word the four-byte stores of a warp, 32 bytes apart, met in four banks
  // (128 images 267.5 -> 264.9 us for the whole call, four calls in flight 840 -> 832).
  if constexpr (kShape == kRows128 && !kSplit) {
    if (P.paired && pm.parts == 1) {
      if (pm.j != 0) return;
      uint32_t w[2][2];
#pragma unroll
      for (int wd = 0; wd < 2; ++wd) {
        const int4 c4 = *reinterpret_cast<const int4*>(cols + min(wd, nw - 1) * 4);
        const int col[4] = {c4.x, c4.y, c4.z, c4.w};
        int y[2][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int2 x = *reinterpret_cast<const int2*>(pm.v + col[e] * P.pg);
          y[0][e] = (int32_t)(((long long)x.x * (long long)m0 + rnd) >> 32) >> (s - 1);
          y[1][e] = (int32_t)(((long long)x.y * (long long)m0 + rnd) >> 32) >> (s - 1);
        }
        const int over = wd * 4 + 4 - P.ca;        // (six channels or two: as below; none: the constants alone)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          w[wd][k] = pack4_sat(y[k][0], y[k][1], y[k][2], y[k][3]);
          if (over >= 4) w[wd][k] = over == 4 ? 0x7F7F7F01u : 0x7F7F7F7Fu;
          else if (over > 0) w[wd][k] = (w[wd][k] & 0xFFFFu) | 0x7F010000u;
        }
      }
      const uint2 a = make_uint2(w[0][0], w[1][0]), b = make_uint2(w[0][1], w[1][1]);
      *reinterpret_cast<uint4*>(pm.rec) = make_uint4(a.x, a.y, b.x, b.y);
      *reinterpret_cast<uint2*>(pm.rec - 8) = a;
      *reinterpret_cast<uint2*>(pm.rec + 16) = b;
      return;
    }
  }
#pragma unroll 1
  for (int wd = pm.j; wd < nw; wd += pm.parts) {
    const int4 c4 = *reinterpret_cast<const int4*>(cols + wd * 4);       // (entries beyond ca: any column)
    const int col[4] = {c4.x, c4.y, c4.z, c4.w};
    int y[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int2 x = *reinterpret_cast<const int2*>(pm.v + col[e] * P.pg);
      y[0][e] = (int32_t)(((long long)x.x * (long long)m0 + rnd) >> 32) >> (s - 1);
      y[1][e] = (int32_t)(((long long)x.y * (long long)m0 + rnd) >> 32) >> (s - 1);
    }
    // the clip to -128..127 is the pack's saturation
    uint32_t w0 = pack4_sat(y[0][0], y[0][1], y[0][2], y[0][3]), w1 = pack4_sat(y[1][0], y[1][1], y[1][2], y[1][3]);
    const int over = wd * 4 + 4 - P.ca;          // bytes of the word that hold no channel (two, C being a multiple of four)
    if (over > 0) {
      w0 = (w0 & 0xFFFFu) | 0x7F010000u;
      w1 = (w1 & 0xFFFFu) | 0x7F010000u;
    }
    if constexpr (kShape != kImages4x4) {
      uint32_t* rec = reinterpret_cast<uint32_t*>(pm.rec + (wd >> 2) * P.plane16 * 16 + (wd & 3) * 4);
      rec[0] = w0;
      rec[4] = w1;
      if (P.paired) {                            // second half of the left neighbour's record
        rec[-2] = w0;
        rec[2] = w1;
      }
      if constexpr (kSplit) {                    // pixels on an edge of the block also go to the neighbours' frames
        const uint32_t base = ptx::smem_u32(rec), bar = ptx::smem_u32(input);
        auto put = [&](int dy, int dx, uint32_t at, uint32_t w) {
          if (!flow_block_exists(P, f, dy, dx)) return;
          const uint32_t rank = (uint32_t)(f.rank + dy * P.nbx + dx), b = flow_peer(bar, rank);
          const uint32_t d = flow_peer(at - (uint32_t)((dy * P.h * P.wp + dx * P.w) * 16), rank);
          flow_store_async(d, b, w);
          if (P.paired && dx == 0) flow_store_async(d - 8u, b, w);
        };
        if (pm.dy) {
          put(pm.dy, 0, base, w0);
          put(pm.dy, 0, base + 16u, w1);
        }
        if (pm.dx) {                             // the left edge's first pixel or the right edge's second one
          const uint32_t at = pm.dx < 0 ? base : base + 16u, w = pm.dx < 0 ? w0 : w1;
          put(0, pm.dx, at, w);
          if (pm.dy) put(pm.dy, pm.dx, at, w);
        }
      }
    } else {
      // word (tap, wd) of the rows of the pixels that read this one: row - 4 (u - 1) - (v - 1)
      int k = wd;
#pragma unroll
      for (int t = 0; t < 9; ++t, k += P.ca >> 2) {
        uint8_t* d = pm.rec + (k >> 2) * P.plane16 * 16 + (k & 3) * 4 - ((t / 3 - 1) * 4 + (t % 3 - 1)) * 16;
        if (pm.taps >> t & 1u) *reinterpret_cast<uint32_t*>(d) = w0;
        if (pm.taps >> (16 + t) & 1u) *reinterpret_cast<uint32_t*>(d + 16) = w1;
      }
    }
  }
}

// ---- a level's input and output index maps (four neighbouring elements per thread and step) ----------------
__device__ __forceinline__ size_t patch_index(const FlowPlan& P, const LevelArgs& a, int b, int ci, int y, int x) {
  const int by = fdiv(b, a.mul_patches_x), bx = b - by * a.patches_x;
  return ((size_t)ci * a.img_h + (size_t)(by * 2 * P.fh + y)) * a.img_w + (size_t)(bx * 2 * P.fw + x);
}

// pre-squeeze element e (a multiple of four, image-major over the CTA's images) -> address in the level's
// input / output array and the flow variable's two planes (dx = 0 at d0, dx = 1 at d0 + pg)
template <bool kSplit>
__device__ __forceinline__ void squeeze_map(const Flow& f, const FlowPlan& P, const LevelArgs& a, int img0, int e, size_t* at, int* d0) {
  const int per_img = P.c * P.px, w2 = 2 * P.w;
  const int g = fdiv(e, P.mul_per_img), r = e - g * per_img;
  const int ci = fdiv(r, P.mul_4px), r2 = r - ci * 4 * P.px;
  const int y = fdiv(r2, P.mul_w2), x = r2 - y * w2;
  const int fy = kSplit ? f.by * 2 * P.h + y : y, fx = kSplit ? f.bx * w2 + x : x;
  if (P.is_first && a.img_w > 0) *at = patch_index(P, a, img0 + g, ci, fy, fx);
  else if (kSplit) *at = (size_t)img0 * P.c * P.fpx + (size_t)ci * 4 * P.fpx + (size_t)fy * 2 * P.fw + fx;
  else *at = (size_t)(img0 + g) * per_img + r;
  *d0 = (ci * 4 + (y & 1) * 2) * P.pg + g * P.px + (y >> 1) * P.w + (x >> 1);
}

// logical element e (a multiple of four) of the level's channels -> its place in z, in the kept channels
// (stride `keep_stride` per image) and in the flow variable
template <bool kSplit, typename Fn>
__device__ __forceinline__ void split_map(const Flow& f, const FlowPlan& P, const LevelArgs& a, const int32_t* col_out, int img0, int e,
                                          int32_t* keep, size_t keep_stride, Fn fn) {
  const int per_img = P.c * P.px;
  const int g = fdiv(e, P.mul_per_img), r = e - g * per_img;
  const int k = fdiv(r, P.mul_px), q = r - k * P.px;
  const size_t b = (size_t)(img0 + g);
  int at = q, plane = P.px;
  if constexpr (kSplit) {
    const int y = fdiv(q, P.mul_w), x = q - y * P.w;
    at = (f.by * P.h + y) * P.fw + f.bx * P.w + x;
    plane = P.fpx;
  }
  int32_t* dst = k >= P.keep_c ? a.z + b * P.d + P.z_off + (size_t)(k - P.keep_c) * plane + at
                               : keep + b * keep_stride + (size_t)k * plane + at;
  fn(k, dst, col_out[k] * P.pg + g * P.px + q);
}

template <bool kInv, bool kSplit>
__device__ __forceinline__ void flow_load(const Flow& f, const FlowPlan& P, const LevelArgs& a, int img0, int32_t* v) {
  const int n = f.nimg * P.c * P.px;
  if (!kInv) {
#pragma unroll 1
    for (int e = 4 * f.tid; e < n; e += 4 * kFlowWorkers) {
      size_t at; int d0;
      squeeze_map<kSplit>(f, P, a, img0, e, &at, &d0);
      int4 q;
      if (P.is_first) {
        const uint32_t b4 = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint8_t*>(a.in) + at);
        q = make_int4((int)(b4 & 0xFFu), (int)((b4 >> 8) & 0xFFu), (int)((b4 >> 16) & 0xFFu), (int)(b4 >> 24));
      } else {
        q = *reinterpret_cast<const int4*>(reinterpret_cast<const int32_t*>(a.in) + at);
      }
      *reinterpret_cast<int2*>(v + d0) = make_int2(q.x, q.z);
      *reinterpret_cast<int2*>(v + d0 + P.pg) = make_int2(q.y, q.w);
    }
  } else {
    int32_t* keep = const_cast<int32_t*>(reinterpret_cast<const int32_t*>(a.in));
#pragma unroll 1
    for (int e = 4 * f.tid; e < n; e += 4 * kFlowWorkers)
      split_map<kSplit>(f, P, a, a.plan->col_out, img0, e, keep, (size_t)a.in_stride, [&](int k, const int32_t* src, int d) {
        // (prior head only: z's block is not read)
        if (a.phase != 1 || k < P.keep_c) *reinterpret_cast<int4*>(v + d) = *reinterpret_cast<const int4*>(src);
      });
  }
}

template <bool kInv, bool kSplit>
__device__ __forceinline__ void flow_store(const Flow& f, const FlowPlan& P, const LevelArgs& a, int img0, const int32_t* v) {
  const int n = f.nimg * P.c * P.px;
  if (!kInv) {
    int32_t* keep = P.is_last ? a.z + P.z_final_off : reinterpret_cast<int32_t*>(a.out);
    const size_t keep_stride = P.is_last ? (size_t)P.d : (size_t)P.keep_c * P.fpx;
#pragma unroll 1
    for (int e = 4 * f.tid; e < n; e += 4 * kFlowWorkers)
      split_map<kSplit>(f, P, a, a.plan->col_out, img0, e, keep, keep_stride,
                [&](int, int32_t* dst, int d) { *reinterpret_cast<int4*>(dst) = *reinterpret_cast<const int4*>(v + d); });
  } else if (a.phase != 1) {
    uint32_t bad = 0;
#pragma unroll 1
    for (int e = 4 * f.tid; e < n; e += 4 * kFlowWorkers) {
      size_t at; int d0;
      squeeze_map<kSplit>(f, P, a, img0, e, &at, &d0);
      const int2 x0 = *reinterpret_cast<const int2*>(v + d0), x1 = *reinterpret_cast<const int2*>(v + d0 + P.pg);
      if (P.is_first) {
        *reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(a.out) + at) = pack4(x0.x, x1.x, x0.y, x1.y);
        bad += (uint32_t)((uint32_t)x0.x > 255u) + (uint32_t)((uint32_t)x1.x > 255u) + (uint32_t)((uint32_t)x0.y > 255u) +
               (uint32_t)((uint32_t)x1.y > 255u);
      } else {
        *reinterpret_cast<int4*>(reinterpret_cast<int32_t*>(a.out) + at) = make_int4(x0.x, x1.x, x0.y, x1.y);
      }
    }
    if (P.is_first && a.oor != nullptr) {
      bad = __reduce_add_sync(0xFFFFFFFFu, bad);
      if (f.lane == 0 && bad) atomicAdd(a.oor, bad);
    }
  }
}

template <bool kInv, bool kSplit, int kShape>
__device__ void flow_workers(const Flow& f, const FlowPlan& P, const LevelArgs& a, const Steps& st, int img0) {
  FlowCtl* ctl = f.ctl;
  uint8_t* smem = f.smem;
  int32_t* v = reinterpret_cast<int32_t*>(smem + P.s_v);
  int32_t* acc = reinterpret_cast<int32_t*>(smem + P.s_acc);
  const uint32_t lane_field = (uint32_t)((f.warp & 3) * 32) << 16;
  // (4 x 4 levels: a lane quarter is an image, or a copy of one; quarters without one only take part in the hand-overs)
  PixelMap pm;
  const int pairs = P.pg >> 1;
  pm.parts = kFlowWorkers / pairs;
  pm.j = f.tid / pairs;
  pm.p = 2 * (f.tid - pm.j * pairs);
  int copy = 0;                                 // (4 x 4: threads of their own for each copy of the operand)
  if (kShape == kImages4x4) {
    pm.parts /= P.copies;
    copy = pm.j / pm.parts;
    pm.j -= copy * pm.parts;
    if (copy >= P.copies) pm.j = 1 << 20;
  }
  if (pm.j >= pm.parts || pm.p >= f.pvalid) pm.j = 1 << 20;      // no work
  {
    const int img = fdiv(pm.p, P.mul_px), px = pm.p - img * P.px, r = fdiv(px, P.mul_w), c = px - r * P.w;
    pm.v = v + pm.p;
    pm.acc = acc + pm.p;
    pm.rec = smem + P.s_xa + 16 * (P.im2col ? (img * P.copies + copy) * 16 + px : img * P.frame + (r + 1) * P.wp + c + 1);
    pm.dy = r == 0 ? -1 : (r == P.h - 1 ? 1 : 0);
    pm.dx = c == 0 ? -1 : (c == P.w - 2 ? 1 : 0);
    pm.taps = 0;
    for (int t = 0; t < 9; ++t) {
      const int oi = r - (t / 3 - 1), oj = c - (t % 3 - 1);
      if ((uint32_t)oi < (uint32_t)P.h && (uint32_t)oj < (uint32_t)P.w) pm.taps |= 1u << t;
      if ((uint32_t)oi < (uint32_t)P.h && (uint32_t)(oj + 1) < (uint32_t)P.w) pm.taps |= 1u << (16 + t);
    }
  }
  const uint32_t dm = f.tmem + (uint32_t)(f.sl * P.d_col) + lane_field, d3 = f.tmem + (uint32_t)(P.d3_col + f.sl * P.d3_step) + lane_field;
  uint32_t dpar = 0u, tpar = 0u, npar = 0u;
  const uint8_t* prev = nullptr;                // coupling whose translation is still to be applied
#pragma unroll 1
  for (int i = 0; i <= st.nsteps; ++i) {
    if (kShape != kImages4x4 && prev && !(kShape == kRows64 && P.direct)) {
      flow_translate<kInv>(P, pm, prev);
      // the network input may read channels that were just updated; what was cleared is released as a whole
      if (kSplit || pm.parts > 1) worker_barrier();
    }
    const uint8_t* mb = smem + P.s_meta[i & 1];
    const FlowMeta* M = reinterpret_cast<const FlowMeta*>(mb);
    const bool prior = i < st.nsteps && st.is_prior(i);
    if (i < st.nsteps) {
    flow_wait(f, &ctl->meta_full[i & 1], (uint32_t)(i >> 1) & 1u);
    // (the first two words of both kinds of meta block)
    uint64_t* input = &ctl->xa_ready[i & 1];
    if (kSplit && f.warp == kFlowWarps - 1) flow_release_to_neighbours(P, f, input);
    flow_requant<kSplit, kShape>(f, P, pm, input, prior ? a.plan->col_out : reinterpret_cast<const int32_t*>(mb + M->off_colA), M->in_m0, M->in_s);
    flow_hand_over(f, input, kSplit && f.warp == 0 ? f.halo : 0u);
    prev = prior ? nullptr : mb;
    }
    // the flow variable is complete: it is stored, under the prior head's GEMM where that is the last step
    if (i == (kInv ? st.nsteps : st.n_couplings)) {
      worker_barrier();
      flow_store<kInv, kSplit>(f, P, a, img0, v);
    }
    if (i == st.nsteps) break;
    if (prior) {
      flow_wait(f, &ctl->dm_ready[f.sl], dpar);
      dpar ^= 1u;
      ptx::tc_fence_after();
      flow_prior<kSplit, kShape>(f, P, a, reinterpret_cast<const PriorMeta*>(mb), img0);
    } else {
#pragma unroll 1
      for (int t = f.sl; t < f.tiles; t += f.slots) {
        const bool quarter = kShape != kImages4x4 || 4 * t + f.image < f.nimg;
#pragma unroll 1
        for (int layer = 0; layer < 2; ++layer) {
          const bool chunked = kShape != kRows128 && (layer ? P.chunk3 : P.chunk2);
          const uint32_t d = kShape != kRows128 && layer ? dm + (uint32_t)P.d2_col : dm;
          const int q = f.lane & 3, row = f.lane >> 2;
          HiddenOut ho;
          if (kShape == kRows64 && layer && P.direct) {
            ho.at = smem + P.s_h[f.sl] + ((q >> 1) * P.frame + ((f.warp & 3) * 2 + 1) * P.wp + 1 + row) * 16 + (q & 1) * 8;
            ho.block = 32 * P.frame;
            ho.row = 16 * P.wp;
          } else {
            const int first = kShape == kImages4x4 ? f.image * P.copies * 16 : (f.warp & 3) * (kShape == kRows128 ? 32 : 16);
            ho.at = smem + P.s_a[f.sl] + (q >> 1) * P.pitch + (first + row) * 16 + (q & 1) * 8;
            ho.block = 2 * P.pitch;
            ho.row = 128;
          }
          if (quarter) {
            flow_hidden<kShape>(f, P, d, mb, layer, ho, chunked, &ctl->dm_ready[f.sl], dpar);
          } else {
            flow_wait(f, &ctl->dm_ready[f.sl], dpar);      // (never a phase ahead in its arrivals)
            const int ks = layer ? M->ks3 : M->ks2;
            for (int b0 = 0, r = 0; b0 < (chunked ? ks : 1); b0 += f.ncs, ++r) flow_hand_over(f, &ctl->a_ready[f.sl][r]);
          }
          dpar ^= 1u;
        }
        if (kShape == kRows64 && P.direct) {
          flow_out<kInv>(f, P, t, d3, mb, v, &ctl->d3_ready[f.sl], tpar);
        } else if constexpr (kShape == kImages4x4) {
          if (quarter) flow_sum_4x4<kInv>(f, P, t, d3, mb, v, &ctl->d3_ready[f.sl], tpar);
        } else {
          flow_sum<kShape == kRows128 ? 4 : 2, kSplit>(f, P, t, d3, acc, &ctl->d3_ready[f.sl], tpar);
        }
        tpar ^= 1u;
        // (streamed weights: the next tile's first GEMM writes where the partials were)
        if (P.ring && t + 1 < f.tiles) flow_hand_over(f, &ctl->a_ready[0][0]);
      }
    }
    ptx::tc_fence_before();
    if (kSplit && !prior && f.tid == 0) ptx::mbar_expect_tx(ptx::smem_u32(&ctl->acc_full), (uint32_t)(P.reds[f.rank] * P.cb * 4));
    worker_barrier();                           // every product has been added
    if constexpr (kSplit) {
      if (!prior) {
        flow_wait_cluster(f, &ctl->acc_full, npar);
        npar ^= 1u;
      } else if (i + 1 < st.nsteps) {
        // The next step's edge pixels overwrite what the neighbours' prior heads read. (After a coupling their products
        // say that they are past it.)
        if (f.warp == 0) flow_release_to_neighbours(P, f, &ctl->peers_done);
        flow_wait_cluster(f, &ctl->peers_done, 0u);
      }
    }
  }
}

template <bool kInv, bool kSplit, int kShape>
__global__ void __launch_bounds__(kFlowThreads, 1) flow_level_kernel(const LevelArgs a, const __grid_constant__ FlowPlan P) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ FlowCtl ctl;
  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;

  ptx::grid_launch_dependents();         // the next kernel in the stream may start its prologue
  const int nblk = kSplit ? P.nbx * P.nby : 1;
  const int img0 = (kSplit ? blockIdx.x / nblk : blockIdx.x) * P.group, nimg = min(P.group, a.batch - img0);
  const int tiles = P.im2col ? (nimg + 3) >> 2 : nimg * P.tiles_img, slots = P.ring ? 1 : min(2, tiles);
  Flow f;
  f.halo = 0;
  f.rank = kSplit ? blockIdx.x % nblk : 0;
  f.by = kSplit ? f.rank / P.nbx : 0;
  f.bx = kSplit ? f.rank - f.by * P.nbx : 0;
  int neighbours = 0;
  if constexpr (kSplit)
    for (int dy = -1; dy <= 1; ++dy)
      for (int dx = -1; dx <= 1; ++dx)
        if ((dy || dx) && flow_block_exists(P, f, dy, dx)) {
          ++neighbours;
          f.halo += (uint32_t)(dx == 0 ? P.w * P.halo_bytes[0] : (dy == 0 ? P.h * P.halo_bytes[1] : P.halo_bytes[2]));
        }
  if (tid == 0) {
    ptx::mbar_init(ptx::smem_u32(&ctl.acc_full), 1);
    ptx::mbar_init(ptx::smem_u32(&ctl.peers_done), (uint32_t)max(neighbours, 1));
    for (int s = 0; s < 2; ++s) {
      ptx::mbar_init(ptx::smem_u32(&ctl.xa_ready[s]), (uint32_t)(kFlowWarps + neighbours));
      for (int r = 0; r < kFlowMaxRounds; ++r) ptx::mbar_init(ptx::smem_u32(&ctl.a_ready[s][r]), (uint32_t)(kFlowWarps / slots));
      ptx::mbar_init(ptx::smem_u32(&ctl.dm_ready[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.d3_ready[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.meta_full[s]), 1);
    }
    for (int s = 0; s < kFlowMaxRing; ++s) {
      ptx::mbar_init(ptx::smem_u32(&ctl.w_full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.w_empty[s]), (uint32_t)slots);
    }
    ptx::mbar_init_fence();
    ctl.abort = 0;
  }
  if (warp == 0) ptx::tmem_alloc(ptx::smem_u32(&ctl.tmem_base), (uint32_t)P.tmem_cols);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();

  f.smem = smem; f.ctl = &ctl; f.status = a.status; f.tmem = ctl.tmem_base;
  f.tid = tid; f.warp = warp; f.lane = lane;
  f.nimg = nimg; f.pvalid = nimg * P.px; f.tiles = tiles; f.slots = slots;
  const int copies = kShape == kImages4x4 ? P.copies : 1;
  f.ncs = kFlowWarps / 4 / slots * copies;
  f.sl = slots == 2 && warp >= kFlowWarps / 2 ? 1 : 0;
  f.cs = ((warp - f.sl * (kFlowWarps / 2)) >> 2) * copies + (warp & 3) % copies;
  f.image = (warp & 3) / copies;
  Steps st;
  st.n_couplings = (kInv && a.phase == 1) ? 0 : P.n_couplings;
  st.do_prior = P.has_prior && a.prior != nullptr && !(kInv && a.phase == 2);
  st.nsteps = st.n_couplings + (st.do_prior ? 1 : 0);
  st.inverse = kInv;

  if (warp >= kFlowWarps && kSplit) flow_cluster_sync();        // (the workers below, after the frame)
  // (packed blocks were written once, at model creation)
  if (warp == kFlowWarps + 2 && !P.ring) {
    if (lane == 0) flow_loader(f, P, a, st);
  } else if (warp >= kFlowWarps) {
    if (!P.ring) flow_mma<kShape>(f, P, st, warp - kFlowWarps);
    else if (warp == kFlowWarps) flow_mma_ring(f, P, st);
    else flow_loader_ring(f, P, a, st, (uint32_t)(warp - kFlowWarps - 1));
  } else {
    // frame of the network input: zero channels, and the constants that multiply the bias rows in the
    // bytes that no channel uses (at 4 x 4 levels: after the nine taps)
    const int lim = P.im2col ? 9 * P.ca : P.ca, unit = P.paired ? 8 : P.plane16 * 16;
    for (uint32_t o = 16 * tid; o < P.s_xa_end - P.s_xa; o += 16 * kFlowWorkers) {
      const int first = P.paired ? 0 : (int)(o / (uint32_t)unit) * 16;       // first byte of the 16-byte plane in a record
      // word of bytes b .. b + 3: zeros up to lim (an even number), then 1, 127, 127, ...
      auto word = [&](int b) { return b + 4 <= lim ? 0u : (b > lim ? 0x7F7F7F7Fu : (b == lim ? 0x7F7F7F01u : 0x7F010000u)); };
      const uint32_t w0 = word(first), w1 = word(first + 4), w2 = P.paired ? w0 : word(first + 8), w3 = P.paired ? w1 : word(first + 12);
      *reinterpret_cast<uint4*>(smem + P.s_xa + o) = make_uint4(w0, w1, w2, w3);
    }
    if (tid < f.tiles) {
      int4 tp = make_int4(4 * tid, 0, 0, 64 * tid);                          // (im2col: first of four images)
      if (!P.im2col) {
        tp.x = tid / P.tiles_img;
        const int tt = tid - tp.x * P.tiles_img;
        tp.y = tt / P.tiles_x * (P.m >> 3);
        tp.z = tt % P.tiles_x * 8;
        tp.w = tp.x * P.frame + (tp.y + 1) * P.wp + tp.z + 1;
      }
      ctl.tile[tid] = tp;
    }
    if (P.direct)                        // zero border of the last conv's operand
      for (uint32_t o = P.s_h[0] + 16 * tid; o < P.s_h_end; o += 16 * kFlowWorkers) *reinterpret_cast<uint4*>(smem + o) = make_uint4(0u, 0u, 0u, 0u);
    for (int o = tid; o < (P.im2col || P.direct ? 0 : P.cb * P.acc_stride); o += kFlowWorkers) reinterpret_cast<int32_t*>(smem + P.s_acc)[o] = 0;
    int32_t* v = reinterpret_cast<int32_t*>(smem + P.s_v);
    if constexpr (kSplit) flow_cluster_sync();     // frame, accumulator and barriers are ready for the neighbours
    ptx::grid_dependency_wait();         // from here on: what the previous kernel in the stream wrote
    flow_load<kInv, kSplit>(f, P, a, img0, v);
    worker_barrier();
    flow_workers<kInv, kSplit, kShape>(f, P, a, st, img0);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if constexpr (kSplit) flow_cluster_sync();       // nothing is on its way to this CTA's memory any more
  if (warp == 0) ptx::tmem_dealloc(ctl.tmem_base, (uint32_t)P.tmem_cols);
}

}  // namespace

namespace {
template <bool kInv, bool kSplit, int kShape>
cudaError_t launch(const LevelArgs& args, const FlowPlan& plan, int grid, cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)kFlowThreads);
  cfg.dynamicSmemBytes = plan.s_total;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)(plan.nbx * plan.nby);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = kSplit ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, flow_level_kernel<kInv, kSplit, kShape>, args, plan);
}
}  // namespace

namespace {
template <bool kInv>
cudaError_t launch_shape(const LevelArgs& args, const FlowPlan& plan, int grid, cudaStream_t stream) {
  const bool split = plan.nbx * plan.nby > 1;
  if (plan.im2col) return launch<kInv, false, kImages4x4>(args, plan, grid, stream);
  if (plan.m == 128) return split ? launch<kInv, true, kRows128>(args, plan, grid, stream) : launch<kInv, false, kRows128>(args, plan, grid, stream);
  return split ? launch<kInv, true, kRows64>(args, plan, grid, stream) : launch<kInv, false, kRows64>(args, plan, grid, stream);
}
}  // namespace

cudaError_t launch_flow_level(const LevelArgs& args, const FlowPlan& plan, bool inverse, int grid, cudaStream_t stream) {
  return inverse ? launch_shape<true>(args, plan, grid, stream) : launch_shape<false>(args, plan, grid, stream);
}

int max_flow_clusters(int ctas, uint32_t smem_bytes, uint32_t smem_limit) {
  if (configure_flow_kernels(smem_limit) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3((unsigned)kFlowThreads);
  cfg.dynamicSmemBytes = smem_bytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, flow_level_kernel<false, true, kRows128>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t configure_flow_kernels(uint32_t max_smem_bytes) {
  const auto set = [&](const void* k) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem_bytes); };
  const void* kernels[] = {
      reinterpret_cast<const void*>(flow_level_kernel<false, false, kRows128>), reinterpret_cast<const void*>(flow_level_kernel<true, false, kRows128>),
      reinterpret_cast<const void*>(flow_level_kernel<false, true, kRows128>), reinterpret_cast<const void*>(flow_level_kernel<true, true, kRows128>),
      reinterpret_cast<const void*>(flow_level_kernel<false, false, kRows64>), reinterpret_cast<const void*>(flow_level_kernel<true, false, kRows64>),
      reinterpret_cast<const void*>(flow_level_kernel<false, true, kRows64>), reinterpret_cast<const void*>(flow_level_kernel<true, true, kRows64>),
      reinterpret_cast<const void*>(flow_level_kernel<false, false, kImages4x4>), reinterpret_cast<const void*>(flow_level_kernel<true, false, kImages4x4>)};
  for (const void* k : kernels)
    if (const cudaError_t e = set(k); e != cudaSuccess) return e;
  return cudaSuccess;
}

}  // namespace iodf
