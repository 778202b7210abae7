// One flow level with residual coupling networks (Eq. 3; scatter add, Sec. 4.5), convs overlapped.
//
// As in res_level.cu the activations of an image (xa: requantised network input, X: block tensor, MID:
// first conv's output) stay in shared memory in the K-major operand layout with a zero border, a conv
// tap is an offset of the operand's start address, and the scatter add is applied to the weights when the
// level is packed. There a conv took 10 000 clocks at a one-tile level, of which the tensor core worked 2 300:
// multiply, requantise and barrier followed one another. What is different here:
//
//   * A conv's K runs chunk by chunk (32 channels, nine taps each). The epilogue of the conv before it
//     hands over its outputs in the same chunks (an mbarrier each), so a conv starts as soon as its first 32
//     input channels exist at all positions; accumulators alternate between two tensor-memory ranges.
//   * Tiles are 8-column blocks (row groups of the operand are image rows, one frame row apart, as in
//     flow_level.cu): 16 x 16 images are two tiles instead of three and no border position is computed; 8 x 8
//     images are one tile of 64 rows; 4 x 4 images are rows of eight positions of which four count, up to
//     three images to a tile.
//   * Biases are a tenth operand row group: one more K step against a constant operand (1, c, ..., c).
//     Hidden outputs are then one fma.rn.sat each (FloatRq), the branch of a block one high multiply-add
//     and shift, its shortcut one multiply on the byte as a subnormal.
//   * Larger images are cut into blocks of 16 x 16 or 8 x 16, one CTA of a cluster each, and so are 16 x 16 images whose convs
//     have more than one chunk, while a batch leaves SMs for it. Edge positions are also stored
//     into the neighbours' frames, asynchronously: the neighbours' chunk barriers count the bytes, and there is no
//     cluster barrier between convs.
//   * Two warps issue the MMAs (a chunk's nine taps per wait: waits and commits cost a lane 150 clocks
//     each, an MMA 40): a tile each, or, where there is one tile, its chunks in turn, with an accumulator each that the
//     epilogue adds. One lane of another streams weights and the convs' meta blocks.
//
// What bounds it: a conv's chain of first chunk -> 36 MMAs (1 500 - 2 400 clocks) -> last chunk's epilogue -> hand-over,
// 3 300 clocks at 8 x 8 and 4 x 4 images, 5 700 at 16 x 16 (in two blocks), 145 convs one after another. Measured at width 128 with
// eight blocks, eight couplings (res_level.cu before): 64 images of 16 x 16 1 610 -> 420 us, 8 x 8 750 -> 240,
// 4 x 4 740 -> 245; 32 images of 32 x 32 1 750 -> 627.
#include "res_flow.h"
#include "level_device.cuh"

namespace iodf {

namespace {

struct __align__(16) RfCtl {
  uint64_t chunk_ready[2][kRfChunks];  // workers (and the neighbours' edge bytes) -> MMA warp: 32 channels of the output of
                                       // an even / odd conv (a neighbour may be one conv ahead)
  uint64_t xa_ready;                // the same for the network input
  uint64_t d_ready[2][2];           // tensor core -> workers: accumulators of an even / odd conv complete, by tile (one tile: both)
  uint64_t w_full[kRfMaxSlots];     // weight slots: copy landed
  uint64_t w_empty[kRfMaxSlots];    // ... and both MMA warps are past it (count 2)
  uint64_t meta_full[3];
  uint32_t tmem_base, abort;
};

struct Rf {
  uint8_t* smem;
  RfCtl* ctl;
  uint32_t* status;
  uint32_t tmem;
  int tid, warp, lane;
  int nimg;
  int rank, by, bx;                 // CTA of the cluster, its block
  uint32_t halo;                    // positions of this CTA's frame that neighbours write (0: no neighbours)
};

__device__ __noinline__ void rf_wait_slow(uint32_t bar, uint32_t parity, RfCtl* ctl, uint32_t* status) {
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    if (ptx::mbar_try_wait(bar, parity)) return;
    if (*reinterpret_cast<volatile uint32_t*>(&ctl->abort)) return;
  }
  *reinterpret_cast<volatile uint32_t*>(&ctl->abort) = 1;
  atomicExch(status, 1u);
}
__device__ __forceinline__ void rf_wait(const Rf& f, uint64_t* bar, uint32_t parity) {
  const uint32_t b = ptx::smem_u32(bar);
  if (ptx::mbar_test_wait(b, parity) || ptx::mbar_try_wait(b, parity)) return;
  rf_wait_slow(b, parity, f.ctl, f.status);
}

// ---- thread-block cluster ---------------------------------------------------------------------------------
__device__ __forceinline__ void rf_cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t rf_peer(uint32_t saddr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
  return a;
}
__device__ __forceinline__ void rf_arrive_local(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(ptx::smem_u32(bar)) : "memory");
}
// this warp's part of an activation is written; `bytes`: what the neighbours' asynchronous stores will add to the
// phase (announced by one warp; others pass 0)
__device__ __forceinline__ void rf_hand_over(const Rf& f, uint64_t* bar, uint32_t bytes) {
  ptx::tc_fence_before();
  ptx::fence_async_smem();
  __syncwarp();
  if (f.lane == 0) {
    if (bytes) ptx::mbar_expect_tx(ptx::smem_u32(bar), bytes);
    else rf_arrive_local(bar);
  }
}
// store of an edge position into a neighbour's frame: its barrier counts the bytes when they have landed, so the
// writer needs no fence and no arrival of its own (a release at cluster scope per chunk and warp stalled the
// edge warps: 0.84 -> 0.69 ms for the 32 x 32 level of config R64)
__device__ __forceinline__ void rf_store_async8(uint32_t addr, uint32_t bar, const uint2 v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(bar) : "memory");
}
__device__ __forceinline__ void rf_store_async4(uint32_t addr, uint32_t bar, const uint32_t v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
// The MMA warp's wait for an operand. The neighbours' bytes came through the generic proxy and are released at cluster
// scope by the completion that counts them: the phase, complete by now, is read once more with an acquire of that
// scope. (As the waiting loop itself the acquire made every wait's code longer: 1 033 -> 1 061 us for 64 images of
// 32 x 32, none of them cut into blocks; read again: 1 024.)
__device__ __forceinline__ void rf_wait_operand(const Rf& f, uint64_t* bar, uint32_t parity) {
  rf_wait(f, bar, parity);
  if (f.halo) {
    ptx::mbar_acquire_cluster(ptx::smem_u32(bar), parity);
    asm volatile("fence.proxy.async;" ::: "memory");
  }
  ptx::tc_fence_after();
}

// ---- the sequence of convs ----------------------------------------------------------------------------------
struct RfSeq {
  int n_couplings, cpc;         // couplings that run, convs of each
  bool prior_first, prior_last, inverse;
  int count;                    // convs in all
  int all_couplings;
  // conv record of the q-th conv
  __device__ __forceinline__ int index(int q) const {
    const int p = prior_first ? 1 : 0;
    if (q < p || q - p >= n_couplings * cpc) return all_couplings * cpc;          // prior head
    const int k = (q - p) / cpc, i = q - p - k * cpc;
    return (inverse ? n_couplings - 1 - k : k) * cpc + i;
  }
};

// ---- weight and meta loader (one lane) -----------------------------------------------------------------------
__device__ void rf_loader(const Rf& f, const RfPlan& P, const LevelArgs& a, const RfSeq& sq) {
  RfCtl* ctl = f.ctl;
  const RfConv* convs = reinterpret_cast<const RfConv*>(a.blob + P.conv_off);
  uint32_t slot = 0, round = 0;
  int ms = 0;
#pragma unroll 1
  for (int q = 0; q < sq.count; ++q) {
    const RfConv c = convs[sq.index(q)];
    // meta slot: its last readers were the workers at the epilogue of conv q - 3, over when conv q - 2 is
    // complete (whose barrier cannot complete again before conv q, so the wait cannot miss its phase)
    if (q >= 3) rf_wait(f, &ctl->d_ready[q & 1][0], (uint32_t)((q - 2) >> 1) & 1u);
    {
      const uint32_t b = ptx::smem_u32(&ctl->meta_full[ms]);
      ptx::mbar_expect_tx(b, c.meta_bytes);
      ptx::bulk_g2s(ptx::smem_u32(f.smem + P.s_meta[ms]), a.blob + c.meta_off, c.meta_bytes, b);
      ms = ms == 2 ? 0 : ms + 1;
    }
    const uint8_t* src = a.blob + c.w_off;
#pragma unroll 1
    for (int g = 0; g < c.nk; ++g) {
      const uint32_t bytes = (uint32_t)(g == 0 ? 10 : 9) * 32u * (uint32_t)c.n_pad;
      if (round > 0) rf_wait(f, &ctl->w_empty[slot], (round - 1u) & 1u);
      const uint32_t b = ptx::smem_u32(&ctl->w_full[slot]);
      ptx::mbar_expect_tx(b, bytes);
      ptx::bulk_g2s(ptx::smem_u32(f.smem + P.s_ring + slot * P.slot_bytes), src, bytes, b);
      src += bytes;
      if (++slot == (uint32_t)P.n_slots) { slot = 0; ++round; }
    }
  }
}

// ---- MMA warps -----------------------------------------------------------------------------------------------
// Two tiles: a warp each. One tile: the warps take its chunks in turn, each into an accumulator of its own (the epilogue adds
// them), so that one warp's waits and commit, 250 - 450 clocks a chunk, pass under the other's MMAs (360 - 570): 64 images of 8 x 8
// 285 -> 248 us, of 4 x 4 289 -> 260, three of 32 x 32 in 8 x 16 blocks 539 -> 438; with two tiles a chunk's MMAs hid them already
// (16 x 16 466 -> 465).
// Every copy is seen by both warps, and a slot is empty when both are past it. A barrier's parity tells a phase only from the one before
// it: a warp that tested a slot whose last copy had been the other's (rings of three slots, convs of three chunks) could take the
// phase before that for its own, if that copy was late, and multiply with what was in the slot. (The other's copies cost it a test and an
// arrival each: 64 images of 32 x 32 873 -> 890 us for the whole call.)
__device__ void rf_mma(const Rf& f, const RfPlan& P, const RfSeq& sq, int which) {
  RfCtl* ctl = f.ctl;
  uint8_t* smem = f.smem;
  auto uniform = [](int x) { return __shfl_sync(0xFFFFFFFFu, x, 0); };
  // (in a cluster a shared-memory address also carries the CTA's rank above the descriptor's 14 bits)
  auto addr16 = [&](uint32_t s) { return (ptx::smem_u32(smem + s) >> 4) & 0x3FFFu; };
  const uint32_t a_hi = (uint32_t)P.wp | (1u << 14), plane = (uint32_t)P.plane16;
  const bool one = P.tiles == 1;
  uint32_t slot = 0, round = 0, ready = 0, xa_par = 0;     // ready: bit 4 s + c: parity of chunk barrier [s][c]
  int ms = 0;
  uint32_t mpar = 0;
#pragma unroll 1
  for (int q = 0; q < sq.count; ++q) {
    rf_wait(f, &ctl->meta_full[ms], mpar);
    const RfMeta* M = reinterpret_cast<const RfMeta*>(smem + P.s_meta[ms]);
    const int n = uniform(M->n_pad), nk = uniform(M->nk), src = uniform(M->src), uns = uniform(M->a_unsigned), input = uniform(M->input);
    if (++ms == 3) { ms = 0; mpar ^= 1u; }
    const uint32_t idesc = (2u << 4) | ((uns ? 0u : 1u) << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(P.m >> 4) << 24);
    const uint32_t d0 = f.tmem + (uint32_t)((q & 1) * 256 + which * 128);
    const uint32_t b_lbo = (uint32_t)n << 16, tap_step = 2u * (uint32_t)n;
    // first position of the tile's first tap in the source, chunk 0
    uint32_t a_chunk = addr16(P.s_buf[src]) + (plane << 16) + (one ? 0u : 8u * (uint32_t)which);
    uint32_t acc = 0u;
    const int set = (q - 1) & 1;
    auto wait_chunk = [&](int kc) {
      if (!input) rf_wait_operand(f, &ctl->chunk_ready[set][kc], (ready >> (4 * set + kc)) & 1u);
      else if (kc < 2) rf_wait_operand(f, &ctl->xa_ready, xa_par);
    };
    // (a warp without a chunk of this conv commits no sooner than the other one: never a phase ahead)
    if (one && which >= nk) wait_chunk(0);
#pragma unroll 1
    for (int kc = 0; kc < nk; ++kc) {
      if (one && (kc & 1) != which) {
        rf_wait(f, &ctl->w_full[slot], round & 1u);
        if (ptx::elect_one()) rf_arrive_local(&ctl->w_empty[slot]);
      } else {
        // (all that the wait need not precede: an instruction of this warp takes about 13 clocks)
        uint32_t bl = addr16(P.s_ring + slot * P.slot_bytes) | b_lbo;
        const uint32_t a_bias = addr16(P.s_const + (uns ? 0u : 2304u)) | (8u << 16);
        rf_wait(f, &ctl->w_full[slot], round & 1u);
        wait_chunk(kc);
        if (ptx::elect_one()) {
          if (kc == 0) {                    // bias rows: the operand is the same constant row everywhere
            ptx::umma_i8_hl(d0, a_bias, ptx::kUmmaDescHi, bl, ptx::kUmmaDescHi, idesc, 0u);
            bl += tap_step;
            acc = 1u;
          }
          uint32_t al = a_chunk;
#pragma unroll
          for (int u = 0; u < 3; ++u) {
#pragma unroll
            for (int v = 0; v < 3; ++v) {
              ptx::umma_i8_hl(d0, al + (uint32_t)v, a_hi, bl, ptx::kUmmaDescHi, idesc, u + v > 0 ? 1u : acc);
              bl += tap_step;
            }
            al += (uint32_t)P.wp;
          }
          ptx::umma_commit(ptx::smem_u32(&ctl->w_empty[slot]));
        }
        acc = 1u;
      }
      __syncwarp();
      if (++slot == (uint32_t)P.n_slots) { slot = 0; ++round; }
      a_chunk += 2u * plane;
    }
    if (input) xa_par ^= 1u;
    else ready ^= ((1u << nk) - 1u) << (4 * set);
    if (ptx::elect_one()) ptx::umma_commit(ptx::smem_u32(&ctl->d_ready[q & 1][one ? 0 : which]));
    __syncwarp();
  }
}

// ---- workers ---------------------------------------------------------------------------------------------------
struct RfPos {             // a thread's two positions of a tile half (rows of the operand: lane / 4 and lane / 4 + 8)
  bool ok0, ok1;
  int p0, p1;              // pixels of the CTA
};

// 8 (4) bytes of an activation, stored at `d` in this CTA's frame, into the neighbours' frames if the pixel (i, j) of the block lies on
// an edge. (Apart from the store itself, so that whole images test once for neighbours: 64 images of 4 x 4 260 -> 254 us.)
template <typename V>
__device__ __forceinline__ void rf_send(const Rf& f, const RfPlan& P, uint8_t* d, const V v, int i, int j, uint64_t* bar) {
  const int dy = i == 0 ? -1 : (i == P.bh - 1 ? 1 : 0), dx = j == 0 ? -1 : (j == P.bw - 1 ? 1 : 0);
  const bool ny = dy && (uint32_t)(f.by + dy) < (uint32_t)P.nby, nx = dx && (uint32_t)(f.bx + dx) < (uint32_t)P.nbx;
  const uint32_t s = ptx::smem_u32(d), b = ptx::smem_u32(bar);
  auto put = [&](int oy, int ox) {
    const uint32_t rank = (uint32_t)(f.rank + oy * P.nbx + ox), at = rf_peer(s - (uint32_t)((oy * P.bh * P.wp + ox * P.bw) * 16), rank);
    if constexpr (sizeof(V) == 8) rf_store_async8(at, rf_peer(b, rank), v);
    else rf_store_async4(at, rf_peer(b, rank), v);
  };
  if (ny) put(dy, 0);
  if (nx) put(0, dx);
  if (ny && nx) put(dy, dx);
}

// One unit: 16 rows (half `h` of this warp's lane quarter of tile `t`) x 32 columns (chunk b) of a hidden or branch conv.
__device__ __forceinline__ void rf_unit(const Rf& f, const RfPlan& P, const RfMeta* __restrict__ M, uint32_t d, int t, int h, int b,
                                        uint64_t* ready, uint32_t parity, uint64_t* chunk) {
  const bool both = P.tiles == 1 && M->nk > 1;           // two accumulators
  const int q = f.lane & 3, x = f.lane >> 2, hs = P.m >> 7;
  // (what does not depend on the accumulator comes before the wait for it)
  uint32_t r[16];
  const uint8_t* tab = reinterpret_cast<const uint8_t*>(M) + sizeof(RfMeta) + b * 128 + q * 32;
  const float4 m0 = *reinterpret_cast<const float4*>(tab), m1 = *reinterpret_cast<const float4*>(tab + 16);
  const float m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
  // operand rows: row group g is a frame row; the thread's two rows are neighbours in a column
  const int g = ((f.warp & 3) << (1 + hs)) + 2 * h;
  uint8_t* o = f.smem + P.s_buf[M->dst] + ((2 * b + (q >> 1)) * P.plane16 + (g + 1) * P.wp + 1 + t * 8 + x) * 16 + (q & 1) * 8;
  bool ok0 = true, ok1 = true;
  if (P.small) {          // 4 x 4 images, five row groups each
    ok0 = x < 4 && g % 5 < 4 && g / 5 < f.nimg;
    ok1 = x < 4 && (g + 1) % 5 < 4 && (g + 1) / 5 < f.nimg;
  }
  const uint32_t row = (uint32_t)P.wp * 16u;
  const int j = t * 8 + x;
  auto accumulator = [&]() {
    rf_wait(f, ready, parity);
    ptx::tc_fence_after();
    const uint32_t at = d + (uint32_t)(t * 128 + b * 32) + ((uint32_t)h << 20) + ((uint32_t)((f.warp & 3) * 32) << 16);
    ptx::tmem_ld_16x32(at, r);
    if (both) {
      uint32_t r2[16];
      ptx::tmem_ld_16x32(at + 128u, r2);
      ptx::tmem_ld_wait16(r);
      ptx::tmem_ld_wait16_nosync(r2);
#pragma unroll
      for (int k = 0; k < 16; ++k) r[k] += r2[k];
    } else {
      ptx::tmem_ld_wait16(r);
    }
  };
  if (M->kind == kRfHidden) {
    float4 c0 = make_float4(0.f, 0.f, 0.f, 0.f), c1 = c0;
    if (b < M->nfi) {
      c0 = *reinterpret_cast<const float4*>(tab + kRfChunks * 128);
      c1 = *reinterpret_cast<const float4*>(tab + kRfChunks * 128 + 16);
    }
    const float c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
    const bool integer = b >= M->nfi;
    accumulator();
    if (!integer) {
#pragma unroll
      for (int k = 0; k < 16; ++k) r[k] = (uint32_t)FloatRq::one(r[k], m[2 * (k >> 2) + (k & 1)], c[2 * (k >> 2) + (k & 1)]);
    } else {
      const long long rnd = 1ll << (30 + M->us);
      const int sh = M->us - 1;
#pragma unroll
      for (int k = 0; k < 16; ++k)
        r[k] = (uint32_t)((int)(((long long)(int)r[k] * (long long)__float_as_int(m[2 * (k >> 2) + (k & 1)]) + rnd) >> 32) >> sh);
    }
  } else {
    uint2 x0 = make_uint2(0u, 0u), x1 = x0;
    if (ok0) x0 = *reinterpret_cast<const uint2*>(o);
    if (ok1) x1 = *reinterpret_cast<const uint2*>(o + row);
    const float ms = M->short_m;
    const long long rnd = 1ll << (30 + M->us);
    const int sh = M->us - 1;
    accumulator();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const uint32_t word = (k & 8) ? ((k & 2) ? x1.y : x0.y) : ((k & 2) ? x1.x : x0.x);
      const uint32_t byte = __byte_perm(word, 0u, 0x4440u | (uint32_t)(2 * ((k >> 2) & 1) + (k & 1)));
      float s;              // the shortcut: the byte as a subnormal, times the multiplier, rounded to an integer
      asm("fma.rn.f32 %0, %1, %2, %3;" : "=f"(s) : "f"(__uint_as_float(byte)), "f"(ms), "f"(0.f));
      const int br = (int)(((long long)(int)r[k] * (long long)__float_as_int(m[2 * (k >> 2) + (k & 1)]) + rnd) >> 32) >> sh;
      r[k] = (uint32_t)(__float_as_int(s) + br);
    }
  }
  // ReLU and clip to 0..255 are the pack's saturation
  const uint2 v0 = make_uint2(pack4_sat_u8((int)r[0], (int)r[1], (int)r[4], (int)r[5]), pack4_sat_u8((int)r[8], (int)r[9], (int)r[12], (int)r[13]));
  const uint2 v1 = make_uint2(pack4_sat_u8((int)r[2], (int)r[3], (int)r[6], (int)r[7]), pack4_sat_u8((int)r[10], (int)r[11], (int)r[14], (int)r[15]));
  if (ok0) *reinterpret_cast<uint2*>(o) = v0;
  if (ok1) *reinterpret_cast<uint2*>(o + row) = v1;
  if (f.halo) {
    rf_send(f, P, o, v0, g, j, chunk);
    rf_send(f, P, o + row, v1, g + 1, j, chunk);
  }
}

// thread's two pixels (of the CTA) for operand rows g, g + 1 of tile t; -1: none
__device__ __forceinline__ void rf_pixels(const Rf& f, const RfPlan& P, int t, int g, int* p0, int* p1) {
  const int x = f.lane >> 2;
  if (P.small) {
    *p0 = x < 4 && g % 5 < 4 && g / 5 < f.nimg ? g / 5 * 16 + g % 5 * 4 + x : -1;
    ++g;
    *p1 = x < 4 && g % 5 < 4 && g / 5 < f.nimg ? g / 5 * 16 + g % 5 * 4 + x : -1;
  } else {
    *p0 = g * P.bw + t * 8 + x;
    *p1 = *p0 + P.bw;
  }
}

// Last conv of a coupling: the translation is added to (subtracted from) the flow variable; prior head:
// parameters to global memory. Unit: (tile, half, 8 columns).
template <bool kInv>
__device__ void rf_out(const Rf& f, const RfPlan& P, const LevelArgs& a, const RfMeta* __restrict__ M, uint32_t d, int32_t* v, int b0) {
  const uint8_t* mb = reinterpret_cast<const uint8_t*>(M);
  const OutRq* orq = reinterpret_cast<const OutRq*>(mb + sizeof(RfMeta));
  const int32_t* colB = reinterpret_cast<const int32_t*>(mb + M->cols_off);
  const int hs = P.m >> 7, ng = (M->n + 7) >> 3, units = (P.tiles << hs) * ng;
#pragma unroll 1
  for (int un = f.warp >> 2; un < units; un += 4) {
    const int gr = un / (P.tiles << hs), th = un - gr * (P.tiles << hs), h = th & hs, t = th >> hs;
    uint32_t r[4], r2[4] = {0u, 0u, 0u, 0u};
    const uint32_t at = d + (uint32_t)(t * 128 + gr * 8) + ((uint32_t)h << 20) + ((uint32_t)((f.warp & 3) * 32) << 16);
    ptx::tmem_ld_16x8(at, r);
    if (P.tiles == 1 && M->nk > 1) ptx::tmem_ld_16x8(at + 128u, r2);
    int p[2];
    rf_pixels(f, P, t, ((f.warp & 3) << (1 + hs)) + 2 * h, &p[0], &p[1]);
    ptx::tmem_ld_wait4(r);
    ptx::tmem_ld_wait4_nosync(r2);
#pragma unroll
    for (int k = 0; k < 4; ++k) r[k] += r2[k];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int ch = gr * 8 + 2 * (f.lane & 3) + e;
      if (ch >= M->n) continue;
      const OutRq o = orq[ch];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (p[k] < 0) continue;
        const int32_t y = rq_out((int32_t)r[2 * k + e], o);
        if (M->kind == kRfOut) {
          uint32_t* vp = reinterpret_cast<uint32_t*>(v + colB[ch] * P.pg + p[k]);
          *vp = kInv ? *vp - (uint32_t)y : *vp + (uint32_t)y;
        } else {
          const int img = P.small ? p[k] >> 4 : 0, pp = P.small ? p[k] & 15 : p[k];
          const int i = P.small ? pp >> 2 : pp / P.bw, j = P.small ? pp & 3 : pp - i * P.bw;
          int32_t* mu = a.prior + (size_t)(b0 + img) * (size_t)(2 * P.d_fact) + P.prior_off + (f.by * P.bh + i) * P.w + f.bx * P.bw + j;
          const int half = M->n >> 1;
          if (ch < half) mu[(size_t)ch * P.px] = y;
          else mu[P.d_fact + (size_t)(ch - half) * P.px] = clampi(y, M->ls_lo, M->ls_hi);
        }
      }
    }
  }
}

// network input: words of four requantised channels at the pixels' positions (and the neighbours' edges)
__device__ __forceinline__ void rf_requant(const Rf& f, const RfPlan& P, const RfMeta* __restrict__ M, const int32_t* __restrict__ v) {
  const int32_t* cols = reinterpret_cast<const int32_t*>(reinterpret_cast<const uint8_t*>(M) + M->cols_off);
  const int nw = (P.ca + 3) >> 2, pv = f.nimg * P.bw * P.bh, m0 = M->in_m0, s = M->in_s;
#pragma unroll 1
  for (int it = f.tid; it < nw * P.pg; it += kRfWorkers) {
    const int wd = it / P.pg, p = it - wd * P.pg;
    if (p >= pv) continue;
    int y[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      y[e] = 0;
      if (wd * 4 + e < P.ca) y[e] = rq_exact(v[cols[wd * 4 + e] * P.pg + p], m0, s);
    }
    const int row = P.small ? (p >> 4) * 5 + ((p >> 2) & 3) : p / P.bw, j = P.small ? p & 3 : p - row * P.bw;
    uint8_t* d = f.smem + P.s_buf[M->src] + ((wd >> 2) * P.plane16 + (row + 1) * P.wp + 1 + j) * 16 + (wd & 3) * 4;
    const uint32_t word = pack4_sat(y[0], y[1], y[2], y[3]);
    *reinterpret_cast<uint32_t*>(d) = word;
    if (f.halo) rf_send(f, P, d, word, row, j, &f.ctl->xa_ready);
  }
}

template <bool kInv>
__device__ void rf_workers(const Rf& f, const RfPlan& P, const LevelArgs& a, const RfSeq& sq, int b0) {
  RfCtl* ctl = f.ctl;
  int32_t* v = reinterpret_cast<int32_t*>(f.smem + P.s_v);
  const int cs = f.warp >> 2, hs = P.m >> 7;
  // units of a chunk in a lane quarter: (tile, half); the quarter's warps take them and, where there are
  // fewer than four, successive chunks
  const int per = P.tiles << hs, me = cs & (per - 1), c0 = cs / per, cstep = 4 / per;
  const int t = me >> hs, h = me & hs;
  int ms = 0;
  uint32_t mpar = 0;
#pragma unroll 1
  for (int q = 0; q < sq.count; ++q) {
    rf_wait(f, &ctl->meta_full[ms], mpar);
    const RfMeta* M = reinterpret_cast<const RfMeta*>(f.smem + P.s_meta[ms]);
    if (++ms == 3) { ms = 0; mpar ^= 1u; }
    if (M->input) {
      rf_requant(f, P, M, v);
      rf_hand_over(f, &ctl->xa_ready, f.warp == 0 ? f.halo * 4u * (uint32_t)((P.ca + 3) >> 2) : 0u);
    }
    const uint32_t d = f.tmem + (uint32_t)((q & 1) * 256);
    const int nb = M->nb, kind = M->kind;
    uint64_t* dr = &ctl->d_ready[q & 1][t];
    const uint32_t dp = (uint32_t)(q >> 1) & 1u;
    if (kind == kRfHidden || kind == kRfBranch) {
      if (c0 != 0) {                       // every warp arrives once per conv: nobody can miss a phase
        rf_wait(f, dr, dp);
        __syncwarp();
        if (f.lane == 0) rf_arrive_local(&ctl->chunk_ready[q & 1][0]);
        // The next conv starts with chunk 0, so that chunk's warps go first: with all at once each takes longer and the MMAs wait
        // (arrivals ahead of the wait, without the delay that this wait is: 64 images of 32 x 32 927 -> 970 us for the whole call; with
        // the pauses 895 -> 870). A pause is a hint, of nothing to twice its length, and nothing but time depends on it. At width 128
        // convs take 1 - 3 % longer without, at 16 - 64 the same, with three 4 x 4 images to a CTA 2 - 4 % less.
        if (per == 2) __nanosleep(120);
        else if (c0 >= 2) __nanosleep(c0 == 2 ? 200 : 300);
      }
#pragma unroll 1
      for (int b = c0; b < nb; b += cstep) {
        uint64_t* cr = &ctl->chunk_ready[q & 1][b];
        rf_unit(f, P, M, d, t, h, b, dr, dp, cr);
        rf_hand_over(f, cr, me == 0 && (f.warp & 3) == 0 ? f.halo * 32u : 0u);
      }
    } else {
      rf_wait(f, &ctl->d_ready[q & 1][0], dp);
      if (P.tiles == 2) rf_wait(f, &ctl->d_ready[q & 1][1], dp);
      ptx::tc_fence_after();
      rf_out<kInv>(f, P, a, M, d, v, b0);
      ptx::tc_fence_before();
      asm volatile("bar.sync 1, %0;" ::"n"(kRfWorkers) : "memory");      // the next network input reads what was updated
    }
  }
}

// ---- level input and output: four neighbouring elements per thread and step -------------------------------------
template <bool kInv, bool kStore>
__device__ __forceinline__ void rf_io(const Rf& f, const RfPlan& P, const LevelArgs& a, int32_t* v, int b0) {
  const int32_t* col_out = a.plan->col_out;
  uint32_t bad = 0;
  if (kInv == kStore) {
    // pre-squeeze array [c/4][2h][2w] <-> planes: rows 2 by bh .., columns 2 bx bw ..
    const int w2 = 2 * P.bw, per = P.c * P.bw * P.bh, w2full = 2 * P.w;
#pragma unroll 1
    for (int e = 4 * f.tid; e < f.nimg * per; e += 4 * kRfWorkers) {
      const int g = e / per, r = e - g * per, ci = r / (4 * P.bw * P.bh), r2 = r - ci * 4 * P.bw * P.bh, y = r2 / w2, x = r2 - y * w2;
      const int gy = 2 * f.by * P.bh + y, gx = 2 * f.bx * P.bw + x, bi = b0 + g;
      size_t at = ((size_t)bi * (P.c / 4) + ci) * (size_t)(4 * P.px) + (size_t)gy * w2full + gx;
      if (P.is_first && a.img_w > 0) {
        const int py = fdiv(bi, a.mul_patches_x), px = bi - py * a.patches_x;
        at = ((size_t)ci * a.img_h + (size_t)(py * 2 * P.h + gy)) * a.img_w + (size_t)(px * w2full + gx);
      }
      int32_t* d0 = v + (ci * 4 + (y & 1) * 2) * P.pg + g * P.bw * P.bh + (y >> 1) * P.bw + (x >> 1);
      if (!kStore) {
        int4 q;
        if (P.is_first) {
          const uint32_t b4 = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint8_t*>(a.in) + at);
          q = make_int4((int)(b4 & 0xFFu), (int)((b4 >> 8) & 0xFFu), (int)((b4 >> 16) & 0xFFu), (int)(b4 >> 24));
        } else {
          q = *reinterpret_cast<const int4*>(reinterpret_cast<const int32_t*>(a.in) + at);
        }
        *reinterpret_cast<int2*>(d0) = make_int2(q.x, q.z);
        *reinterpret_cast<int2*>(d0 + P.pg) = make_int2(q.y, q.w);
      } else {
        const int2 x0 = *reinterpret_cast<const int2*>(d0), x1 = *reinterpret_cast<const int2*>(d0 + P.pg);
        if (P.is_first) {
          *reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(a.out) + at) = pack4(x0.x, x1.x, x0.y, x1.y);
          bad += (uint32_t)((uint32_t)x0.x > 255u) + (uint32_t)((uint32_t)x1.x > 255u) + (uint32_t)((uint32_t)x0.y > 255u) +
                 (uint32_t)((uint32_t)x1.y > 255u);
        } else {
          *reinterpret_cast<int4*>(reinterpret_cast<int32_t*>(a.out) + at) = make_int4(x0.x, x1.x, x0.y, x1.y);
        }
      }
    }
    if (kStore && P.is_first && a.oor != nullptr) {
      bad = __reduce_add_sync(0xFFFFFFFFu, bad);
      if (f.lane == 0 && bad) atomicAdd(a.oor, bad);
    }
  } else {
    // logical channels: kept ones <-> the other level's buffer (or z's final block), the rest <-> z's block
    const int per = P.c * P.bw * P.bh;
    int32_t* keep = kInv ? const_cast<int32_t*>(reinterpret_cast<const int32_t*>(a.in))
                         : (P.is_last ? a.z + P.z_final_off : reinterpret_cast<int32_t*>(a.out));
    const size_t keep_stride = kInv ? (size_t)a.in_stride : (P.is_last ? (size_t)P.d : (size_t)P.keep_c * P.px);
#pragma unroll 1
    for (int e = 4 * f.tid; e < f.nimg * per; e += 4 * kRfWorkers) {
      const int g = e / per, r = e - g * per, k = r / (P.bw * P.bh), q = r - k * P.bw * P.bh, i = q / P.bw, j = q - i * P.bw;
      const size_t bi = (size_t)(b0 + g), px = (size_t)(f.by * P.bh + i) * P.w + f.bx * P.bw + j;
      if (kInv && a.phase == 1 && k >= P.keep_c) continue;
      int32_t* at = k >= P.keep_c ? a.z + bi * P.d + P.z_off + (size_t)(k - P.keep_c) * P.px + px
                                  : keep + bi * keep_stride + (size_t)k * P.px + px;
      int4* d = reinterpret_cast<int4*>(v + col_out[k] * P.pg + g * P.bw * P.bh + q);
      if (kStore) *reinterpret_cast<int4*>(at) = *d;
      else *d = *reinterpret_cast<const int4*>(at);
    }
  }
}

template <bool kInv>
__global__ void __launch_bounds__(kRfThreads, 1) res_flow_kernel(const LevelArgs a, const __grid_constant__ RfPlan P) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ RfCtl ctl;
  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
  const int nblk = P.nbx * P.nby;
  ptx::grid_launch_dependents();

  Rf f;
  f.smem = smem; f.ctl = &ctl; f.status = a.status;
  f.tid = tid; f.warp = warp; f.lane = lane;
  f.rank = nblk > 1 ? (int)(blockIdx.x % nblk) : 0;
  f.by = f.rank / P.nbx; f.bx = f.rank - f.by * P.nbx;
  const int b0 = (int)(blockIdx.x / nblk) * P.group;
  f.nimg = min(P.group, a.batch - b0);
  f.halo = 0;
  for (int dy = -1; dy <= 1; ++dy)
    for (int dx = -1; dx <= 1; ++dx)
      if ((dy || dx) && (uint32_t)(f.by + dy) < (uint32_t)P.nby && (uint32_t)(f.bx + dx) < (uint32_t)P.nbx)
        f.halo += (uint32_t)((dy ? 1 : P.bh) * (dx ? 1 : P.bw));
  if (tid == 0) {
    // (chunk 0 takes every warp's arrival, the others those of the warps that work on them)
    for (int c = 0; c < 2 * kRfChunks; ++c)
      ptx::mbar_init(ptx::smem_u32(&ctl.chunk_ready[c >> 2][c & 3]), (c & 3) ? (uint32_t)(4 * (P.tiles * (P.m >> 6))) : (uint32_t)kRfWarps);
    ptx::mbar_init(ptx::smem_u32(&ctl.xa_ready), (uint32_t)kRfWarps);
    for (int s = 0; s < 4; ++s) ptx::mbar_init(ptx::smem_u32(&ctl.d_ready[s >> 1][s & 1]), P.tiles == 1 ? 2u : 1u);
    for (int s = 0; s < 3; ++s) ptx::mbar_init(ptx::smem_u32(&ctl.meta_full[s]), 1);
    for (int s = 0; s < kRfMaxSlots; ++s) {
      ptx::mbar_init(ptx::smem_u32(&ctl.w_full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.w_empty[s]), 2);
    }
    ptx::mbar_init_fence();
    ctl.abort = 0;
  }
  if (warp == 0) ptx::tmem_alloc(ptx::smem_u32(&ctl.tmem_base), kRfTmemCols);
  // activation buffers start at zero (borders, channels beyond a conv's outputs); the constant operand rows
  for (uint32_t o = P.s_buf[0] + 16 * tid; o < P.s_buf_end; o += 16 * kRfThreads) *reinterpret_cast<uint4*>(smem + o) = make_uint4(0u, 0u, 0u, 0u);
  for (uint32_t o = 16 * tid; o < 2u * 2304u; o += 16 * kRfThreads) {
    const uint32_t w = o < 2304u ? 0xFFFFFFFFu : 0x7F7F7F7Fu;
    *reinterpret_cast<uint4*>(smem + P.s_const + o) = make_uint4((w & ~0xFFu) | 1u, w, w, w);
  }
  ptx::fence_async_smem();
  ptx::tc_fence_before();
  if (nblk > 1) rf_cluster_barrier(); else __syncthreads();
  ptx::tc_fence_after();
  f.tmem = ctl.tmem_base;

  RfSeq sq;
  sq.n_couplings = (kInv && a.phase == 1) ? 0 : P.n_couplings;
  sq.all_couplings = P.n_couplings;
  sq.cpc = P.convs_per_coupling;
  const bool prior = P.has_prior && a.prior != nullptr && !(kInv && a.phase == 2);
  sq.prior_first = prior && kInv; sq.prior_last = prior && !kInv; sq.inverse = kInv;
  sq.count = sq.n_couplings * sq.cpc + (prior ? 1 : 0);

  if (warp == kRfWarps + 2) {
    if (lane == 0) rf_loader(f, P, a, sq);
  } else if (warp >= kRfWarps) {
    rf_mma(f, P, sq, warp - kRfWarps);
  } else {
    int32_t* v = reinterpret_cast<int32_t*>(smem + P.s_v);
    ptx::grid_dependency_wait();
    rf_io<kInv, false>(f, P, a, v, b0);
    asm volatile("bar.sync 1, %0;" ::"n"(kRfWorkers) : "memory");
    rf_workers<kInv>(f, P, a, sq, b0);
    if (!(kInv && a.phase == 1)) rf_io<kInv, true>(f, P, a, v, b0);
  }
  __syncwarp();
  ptx::tc_fence_before();
  // (a neighbour may still be storing edges here: nobody leaves before everybody is done)
  if (nblk > 1) rf_cluster_barrier(); else __syncthreads();
  if (warp == 0) ptx::tmem_dealloc(ctl.tmem_base, kRfTmemCols);
}

}  // namespace

cudaError_t launch_res_flow(const LevelArgs& args, const RfPlan& plan, bool inverse, int ctas, cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3((unsigned)kRfThreads);
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
  cfg.numAttrs = plan.nbx * plan.nby > 1 ? 2 : 1;
  return inverse ? cudaLaunchKernelEx(&cfg, res_flow_kernel<true>, args, plan) : cudaLaunchKernelEx(&cfg, res_flow_kernel<false>, args, plan);
}

int max_res_flow_clusters(int ctas, uint32_t smem_bytes) {
  if (configure_res_flow_kernels(smem_bytes) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3((unsigned)kRfThreads);
  cfg.dynamicSmemBytes = smem_bytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, res_flow_kernel<false>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t configure_res_flow_kernels(uint32_t max_smem_bytes) {
  cudaError_t e = cudaFuncSetAttribute(res_flow_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem_bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(res_flow_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem_bytes);
}

}  // namespace iodf
