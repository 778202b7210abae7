// Entropy coding of the flow's latents on the GPU: the discrete logistic prior of Sec. 3 in integer
// table form and range-ANS (App. A) with a 32-bit state renormalised in 16-bit words, one chain
// per stream. The streams are independent (an image's coded blocks are cut into streams of about
// `elems_per_stream` interleaved elements), so a batch of 128 ImageNet64-sized latents in streams of 128 is 12 288
// streams: the GPU coder that Sec. 5.3 names as future work (the paper codes on the CPU).
//
//   symbol of an element   k = clamp(z - mu, -2048, 2048) + 2048          (0 and 4096: escapes, then
//                                                                          z follows as 2 x 16 raw bits)
//   cumulative counts      Cum(k) = k + G[clamp(floor((2(k-2048)-1) R[ls] / 2^16), -umax, umax) + umax]
//                          Cum(0) = 0, Cum(4097) = M = 2^16
//   encode step            if x >= F * 2^16: move the low 16 bits of x out;  x = (x / F) * M + (x mod F) + C
//   decode step            slot = x mod M; k: Cum(k) <= slot < Cum(k+1);  x = F * (x / M) + slot - C;
//                          if x < 2^16: x = x * 2^16 + next word
//
// The encoder walks a stream's elements last to first and appends words, then the state (low half,
// high half); the decoder starts at the end of the words and walks back, producing the elements
// first to last. Consecutive threads own consecutive streams of a block, whose i-th elements are
// consecutive in memory: the loads of z and of the prior parameters are coalesced.
#include "rans_kernel.h"

namespace iodf {

namespace {

constexpr int kWin = 2048;
constexpr uint32_t kM = 1u << 16;
constexpr int kThreadsPerBlock = 128;        // of the decoder
constexpr int kEncodeStreams = 128, kEncodeThreads = 3 * kEncodeStreams, kBatch = 8;
__host__ __device__ inline size_t encode_buffers_at(const RansArgs& a) {       // offset in the encoder's shared memory, after the tables
  return (4 * (size_t)a.n_scales + 2 * (size_t)(2 * a.umax + 1) + 15) / 16 * 16;
}
// More streams of a block than this per SM: half a warp each. A warp per stream then has six warps and more per scheduler, and issue
// slots bound it. Where the line lies depends on the residuals, which a launch does not know: us for streams of 128 at 148 SMs, residuals
// distributed as the prior says (scales 1 - 32) | uniform over +-3 000, a third of them escapes:
//   streams per SM        5          10          16          21          28          36          49
//   a warp each     40 | 46     42 | 50     52 | 60     58 | 68     66 | 78     83 | 97   109 | 126
//   half of one     49 | 70     50 | 70     46 | 72     46 | 75     50 | 79     54 | 87    68 | 110
// Blocks without prior parameters have one scale, whose look-up table stays in the L1 cache: 36 | 46, 40 | 48, 48 | 58, 56 | 68, 64 | 77
// a warp each and 40 | 52, 42 | 52, 45 | 56, 46 | 56, 50 | 62 half of one.
constexpr long kHalfWarpStreamsPerSm = 24, kHalfWarpStreamsPerSmOneScale = 12;

struct Tables {
  const uint16_t* G;       // shared memory
  const uint32_t* R;       // shared memory
  int umax, n_scales;
};

__device__ __forceinline__ uint32_t cum_of(const Tables& t, uint32_t R, int k) {
  if (k <= 0) return 0u;
  if (k >= 2 * kWin + 1) return kM;
  // floor(edge2 * R / 2^16) in 32-bit pieces: with R = Rh 2^16 + Rl it is edge2 * Rh + floor(edge2 * Rl /
  // 2^16) exactly (|edge2| < 2^13, Rl < 2^16, Rh < 2^15 for the scales a codec accepts)
  const int edge2 = 2 * (k - kWin) - 1;
  int u = edge2 * (int)(R >> 16) + ((edge2 * (int)(R & 0xFFFFu)) >> 16);      // arithmetic shift: floor
  u = max(-t.umax, min(t.umax, u));
  return (uint32_t)k + t.G[u + t.umax];
}

// The same for 0 < k < 4097 (any value otherwise), one wide multiplication and a shift: fewer instructions in a row, 37 -> 35 us for a
// chain of 128; but where issue slots count the pieces are cheaper (encoder 29 against 33 us).
__device__ __forceinline__ uint32_t inner_cum_of(const Tables& t, uint32_t R, int k) {
  const int u = (int)(((long long)(2 * (k - kWin) - 1) * (long long)(int)R) >> 16);       // (fits: above)
  return (uint32_t)k + t.G[max(-t.umax, min(t.umax, u)) + t.umax];
}

// x / F and x mod F for 0 < F <= 2^16 and x < F 2^16, inv = 1 / F rounded: the quotient is below 2^16, so that x * inv
// is off by less than one before truncation (one rounding of 2^-23, x truncated to 24 bits, and two of 2^-24, on a value
// below 2^16), and two conditional corrections make it exact. A 32-bit division is several times as long, and it sits on the chain.
__device__ __forceinline__ uint32_t divide(uint32_t x, uint32_t F, float inv, uint32_t* rem) {
  uint32_t q = __float2uint_rz(__uint2float_rz(x) * inv);
  uint32_t r = x - q * F;
  if ((int32_t)r < 0) { --q; r += F; }
  if (r >= F) { ++q; r -= F; }
  *rem = r;
  return q;
}

// (four bytes at a time and eight loads in flight: one entry after the other the tables took a tenth of a short kernel)
template <int kThreads>
__device__ __forceinline__ void load_tables(const RansArgs& a, uint16_t* sG, uint32_t* sR) {
  const uint32_t* g = reinterpret_cast<const uint32_t*>(a.G);
#pragma unroll 8
  for (int i = threadIdx.x; i < a.umax; i += kThreads) reinterpret_cast<uint32_t*>(sG)[i] = g[i];
  if (threadIdx.x == 0) sG[2 * a.umax] = a.G[2 * a.umax];
  for (int i = threadIdx.x; i < a.n_scales; i += kThreads) sR[i] = a.R[i];
  __syncthreads();
}

// the element's prior parameters; a block without a prior head has mu = 0 and the fixed scale index
__device__ __forceinline__ void prior_of(const RansArgs& a, const RansBlock& blk, const int32_t* prior_img, long e,
                                         int32_t* mu, int* ls, uint32_t* bad) {
  if (blk.prior_off < 0) { *mu = 0; *ls = a.final_ls; return; }
  *mu = prior_img[blk.prior_off + e];
  int l = prior_img[a.d_fact + blk.prior_off + e];
  if (l < 0 || l >= a.n_scales) { *bad = 1u; l = l < 0 ? 0 : a.n_scales - 1; }
  *ls = l;
}

// Encode: a thread per stream walks the chain (symbol, renormalisation, division), and two more prepare its symbols: the
// element, its prior parameters, its counts and their reciprocal depend on no state. A launch has about one chain warp per
// scheduler, which took 650 clocks per symbol, most of them the latencies of what the other two warps now do beside it. Symbols
// go from the preparing to the coding threads in batches of eight, two buffers in shared memory.
// 12 288 streams of 128 elements: 44 -> 30 us, 57 600 94 -> 88.
struct EncodeSymbol {
  uint32_t counts;          // C | F << 16 (F < 2^16: there are 4 097 symbols); 0: no symbol
  float inv;                // 1 / F
};
__global__ void __launch_bounds__(kEncodeThreads) rans_encode_kernel(const RansArgs a, const int32_t* __restrict__ z,
                                                                     const int32_t* __restrict__ prior,
                                                                     uint16_t* __restrict__ words,
                                                                     uint32_t* __restrict__ counts) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ int most;                         // elements of the CTA's longest stream
  __shared__ uint32_t bad[kEncodeStreams];
  uint32_t* sR = reinterpret_cast<uint32_t*>(smem);
  uint16_t* sG = reinterpret_cast<uint16_t*>(smem + 4 * a.n_scales);
  EncodeSymbol* sym = reinterpret_cast<EncodeSymbol*>(smem + encode_buffers_at(a));          // [2][kBatch][kEncodeStreams]
  int32_t* val = reinterpret_cast<int32_t*>(sym + 2 * kBatch * kEncodeStreams);              // the same
  const int me = threadIdx.x & (kEncodeStreams - 1), role = threadIdx.x / kEncodeStreams;    // 0: codes, 1, 2: prepare half a batch each
  const long gid = (long)blockIdx.x * kEncodeStreams + me;
  const bool valid = gid < (long)a.batch * a.n_streams;
  if (threadIdx.x == 0) most = 0;
  if (role == 0) bad[me] = 0;
  load_tables<kEncodeThreads>(a, sG, sR);
  const Tables t{sG, sR, a.umax, a.n_scales};
  const int b = valid ? (int)(gid / a.n_streams) : 0, s = valid ? (int)(gid - (long)b * a.n_streams) : 0;
  int q = 0;
  while (q + 1 < a.n_blocks && s >= a.blocks[q + 1].first_stream) ++q;
  const RansBlock blk = a.blocks[q];
  const int j = s - blk.first_stream, ns = blk.n_streams;
  const int n_el = valid ? (int)((blk.n - j + ns - 1) / ns) : 0;
  if (role == 0) atomicMax(&most, n_el);
  __syncthreads();
  const int batches = (most + kBatch - 1) / kBatch;
  if (role > 0) {
    constexpr int kMine = kBatch / 2;
    const bool has_prior = blk.prior_off >= 0;
    const int32_t* zb = z + (long)b * a.d + blk.z_off + j;
    const int32_t* mub = prior + (has_prior ? (long)b * 2 * a.d_fact + blk.prior_off + j : 0);
    const int32_t* lsb = mub + a.d_fact;
    // elements and prior parameters are on their way a batch ahead: a trip to memory is longer than several symbols
    int32_t zn[kMine], mun[kMine];
    int lsn[kMine], i0 = n_el - 1 - (role - 1) * kMine;          // element of this thread's first symbol of the batch
    auto fetch = [&](int k, int i) {
      zn[k] = 0; mun[k] = 0; lsn[k] = a.final_ls;
      if (i < 0) return;
      const long e = (long)i * ns;
      zn[k] = zb[e];
      if (has_prior) {
        mun[k] = mub[e];
        lsn[k] = lsb[e];
      }
    };
#pragma unroll
    for (int k = 0; k < kMine; ++k) fetch(k, i0 - k);
    for (int n = 0; n < batches; ++n, i0 -= kBatch) {
      const int at = ((n & 1) * kBatch + (role - 1) * kMine) * kEncodeStreams + me;
#pragma unroll
      for (int k = 0; k < kMine; ++k) {
        const int32_t zv = zn[k], mu = mun[k];
        int ls = lsn[k];
        fetch(k, i0 - k - kBatch);
        if (ls < 0 || ls >= a.n_scales) { bad[me] = 1u; ls = ls < 0 ? 0 : a.n_scales - 1; }
        int r;
        asm("sub.sat.s32 %0, %1, %2;" : "=r"(r) : "r"(zv), "r"(mu));
        const int sy = max(-kWin, min(kWin, r)) + kWin;
        const uint32_t R = t.R[ls], C = cum_of(t, R, sy), F = cum_of(t, R, sy + 1) - C;
        EncodeSymbol e;
        e.counts = i0 - k < 0 ? 0u : C | F << 16;
        e.inv = __frcp_rn(__uint2float_rn(F));
        sym[at + k * kEncodeStreams] = e;
        val[at + k * kEncodeStreams] = zv;
      }
      __syncthreads();                                   // batch n is there; the coder is done with batch n - 1
    }
    __syncthreads();
    return;
  }
  uint16_t* out = words + gid * a.cap;
  uint32_t pos = 0, x = 1u << 16;
  __syncthreads();
  for (int n = 0; n < batches; ++n) {
    const int at = (n & 1) * kBatch * kEncodeStreams + me;
    EncodeSymbol e[kBatch];
    int32_t zv[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      e[k] = sym[at + k * kEncodeStreams];
      zv[k] = val[at + k * kEncodeStreams];
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      // (selections rather than branches: some lane of the warp takes either at nearly every symbol)
      const uint32_t C = e[k].counts & 0xFFFFu, F = e[k].counts >> 16;
      const bool some = e[k].counts != 0u, escape = some && (C == 0u || C + F == kM);       // the first or the last symbol
      // an escape: two symbols of frequency 1, the value's lower and upper half: each moves the state's lower 16 bits out (the
      // state is never below 2^16) and takes their place
      if (escape) {
        out[pos] = (uint16_t)x;
        out[pos + 1] = (uint16_t)zv[k];
      }
      pos += escape ? 2u : 0u;
      uint32_t y = escape ? (x & 0xFFFF0000u) | ((uint32_t)zv[k] >> 16) : x;
      const bool full = some && (y >> 16) >= F;
      if (full) out[pos] = (uint16_t)y;
      pos += full ? 1u : 0u;
      y = full ? y >> 16 : y;
      uint32_t r;
      const uint32_t qu = divide(y, F, e[k].inv, &r);
      x = some ? (qu << 16) + r + C : x;
    }
    __syncthreads();
  }
  if (!valid) return;
  out[pos++] = (uint16_t)(x & 0xFFFFu);
  out[pos++] = (uint16_t)(x >> 16);
  counts[gid] = pos;
  if (bad[me] && a.errors) atomicAdd(a.errors, 1u);
}

// Decode: one WARP per stream. The state, the word pointer and every step are the same in all 32
// lanes; what the lanes share out is everything that would otherwise be a dependent trip to memory
// or a dependent search step on the stream's serial chain (state -> symbol -> state):
//   * the symbol search: the lanes hold Cum(32), Cum(64), .. Cum(4096) of the element's scale, four each, from a table made with the
//     codec; they do not depend on the state and are asked for a symbol ahead. Four ballots select 32 symbols; lane L tests one
//     and a ballot picks the largest k with Cum(k) <= slot. The same values give C = Cum(k) and Cum(k + 1) by shuffle;
//   * the prior parameters: the (mu, scale index) of the next 32 elements are loaded by the 32 lanes
//     in one go, a round ahead, and handed out by shuffle, so no global-memory latency sits between two symbols;
//   * the coded words: the lanes hold a window of the stream's next 32 words (the decoder reads the
//     stream backwards).
// What bounds it is a stream's chain, the instructions of a warp that has its scheduler nearly to itself: 35 - 37 us for 768 - 1 536
// streams of 128, 530 clocks per symbol. So the symbols that need more code (escapes, the last of a group of 32) take a branch of
// their own: 47 us with that code in line. With the first look-up in a table of 256 slot ranges per scale, as in the kernel below,
// it was 50: 64 KB of ranges do not stay in the L1 cache, and the load was on the chain.
__global__ void __launch_bounds__(kThreadsPerBlock) rans_decode_kernel(const RansArgs a, int q,
                                                                       const uint16_t* __restrict__ words,
                                                                       const uint32_t* __restrict__ counts,
                                                                       const int32_t* __restrict__ prior,
                                                                       int32_t* __restrict__ z) {
  extern __shared__ __align__(16) uint8_t smem[];
  uint32_t* sR = reinterpret_cast<uint32_t*>(smem);
  uint16_t* sG = reinterpret_cast<uint16_t*>(smem + 4 * a.n_scales);
  load_tables<kThreadsPerBlock>(a, sG, sR);
  const Tables t{sG, sR, a.umax, a.n_scales};
  const RansBlock blk = a.blocks[q];
  const int lane = threadIdx.x & 31;
  const long wid = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;       // one stream per warp
  if (wid >= (long)a.batch * blk.n_streams) return;
  const int b = (int)(wid / blk.n_streams), j = (int)(wid - (long)b * blk.n_streams), ns = blk.n_streams;
  const long sid = (long)b * a.n_streams + blk.first_stream + j;
  const int n_el = (int)((blk.n - j + ns - 1) / ns);
  const uint16_t* in = words + sid * a.cap;
  int top = (int)min((long)counts[sid], (long)a.cap);  // words not yet consumed when the window was filled: in[0 .. top)
  int used = 0;                                        // words taken from the window since
  uint32_t bad = 0;
  // window of the next 32 words: lane L holds in[top - 1 - L], 0 before the stream's first word
  auto fill = [&]() { return top > lane ? (uint32_t)in[top - 1 - lane] : 0u; };
  uint32_t win = fill();
  uint32_t x = __shfl_sync(0xFFFFFFFFu, win, 0) << 16 | __shfl_sync(0xFFFFFFFFu, win, 1);
  used = 2;
  int32_t* zb = z + (long)b * a.d + blk.z_off + j;
  const int32_t* pb = prior + (long)b * 2 * a.d_fact;
  // this lane's element of the next 32: its prior parameters, a round ahead
  int32_t mu_n = 0;
  int ls_n = a.final_ls;
  if (lane < n_el) prior_of(a, blk, pb, j + (long)lane * ns, &mu_n, &ls_n, &bad);
  const uint2* coarse = reinterpret_cast<const uint2*>(a.coarse) + lane;
  uint2 next = __ldg(coarse + (__shfl_sync(0xFFFFFFFFu, ls_n, 0) << 5));
  for (int i0 = 0; i0 < n_el; i0 += 32) {
    const int32_t mu_l = mu_n;
    const int ls_l = ls_n;
    const uint32_t R_l = t.R[ls_l];
    if (i0 + 32 + lane < n_el) prior_of(a, blk, pb, j + (long)(i0 + 32 + lane) * ns, &mu_n, &ls_n, &bad);
    int32_t zv_l = 0;
    const int n_here = min(32, n_el - i0);
    for (int ii = 0; ii < n_here; ++ii) {
      if (used > 29) {                             // (a symbol takes up to three words)
        top -= used;
        used = 0;
        win = fill();
      }
      // what does not depend on the state is on its way during the search
      const uint2 edge = next;
      next = __ldg(coarse + (__shfl_sync(0xFFFFFFFFu, ii == 31 ? ls_n : ls_l, ii + 1) << 5));
      const uint32_t w0 = __shfl_sync(0xFFFFFFFFu, win, used), R = __shfl_sync(0xFFFFFFFFu, R_l, ii);
      const uint32_t slot = x & 0xFFFFu, high = x >> 16;
      // largest k with Cum(k) <= slot: how many of Cum(32), Cum(64), .. Cum(4096) are not above the slot (a prefix: Cum is monotone),
      // then the lanes' 32 symbols from there on
      const int k0 = 32 * (__popc(__ballot_sync(0xFFFFFFFFu, (edge.x & 0xFFFFu) <= slot)) + __popc(__ballot_sync(0xFFFFFFFFu, (edge.x >> 16) <= slot)) +
                           __popc(__ballot_sync(0xFFFFFFFFu, (edge.y & 0xFFFFu) <= slot)) + __popc(__ballot_sync(0xFFFFFFFFu, (edge.y >> 16) <= slot)));
      const uint32_t c = inner_cum_of(t, R, k0 + lane);
      const int sel = 31 - __clz((int)__ballot_sync(0xFFFFFFFFu, c <= slot));
      const uint32_t C = __shfl_sync(0xFFFFFFFFu, c, sel), Cn = __shfl_sync(0xFFFFFFFFu, c, sel + 1);
      int32_t zv;
      if (k0 > 0 && k0 < 2 * kWin && sel < 31) {
        x = (Cn - C) * high + slot - C;
        zv = (int32_t)((uint32_t)mu_l + (uint32_t)(k0 + sel - kWin));             // (lane ii's is the one that counts)
        if (x < (1u << 16)) {
          x = (x << 16) | w0;
          ++used;
        }
      } else {
        // the first and the last symbols, and a group's last one, whose upper end is another group's
        const uint32_t w1 = __shfl_sync(0xFFFFFFFFu, win, used + 1), w2 = __shfl_sync(0xFFFFFFFFu, win, used + 2);
        const int k = k0 + 31 - __clz((int)__ballot_sync(0xFFFFFFFFu, cum_of(t, R, k0 + lane) <= slot));
        const uint32_t Ck = cum_of(t, R, k);
        x = (cum_of(t, R, k + 1) - Ck) * high + slot - Ck;
        const bool more = x < (1u << 16);
        if (more) x = (x << 16) | w0;
        used += more ? 1 : 0;
        zv = (int32_t)((uint32_t)mu_l + (uint32_t)(k - kWin));
        if (k == 0 || k == 2 * kWin) {
          // an escape: two symbols of frequency 1, the value's upper and lower half; each takes the state's lower 16 bits and
          // a word in their place (x >> 16 is always below 2^16)
          const uint32_t wa = more ? w1 : w0, wb = more ? w2 : w1;
          zv = (int32_t)((x << 16) | wa);
          x = (x & 0xFFFF0000u) | wb;
          used += 2;
        }
      }
      if (lane == ii) zv_l = zv;
    }
    if (i0 + lane < n_el) zb[(long)(i0 + lane) * ns] = zv_l;
  }
  if (top != used || x != (1u << 16)) bad = 1u;    // every word used, none missing, and the state back at its start
  bad = __any_sync(0xFFFFFFFFu, bad != 0) ? 1u : 0u;
  if (bad && lane == 0 && a.errors) atomicAdd(a.errors, 1u);
}

// The same with HALF a warp per stream, for blocks of so many streams that issue slots bound the time and not a stream's chain, which
// is longer here. The slot's upper eight bits select, for the element's scale, the symbols
// that it can mean (a table made with the codec: first and count, usually a handful, 257 at most); a lane tests one candidate,
// after a round in steps where there are more than fifteen. A warp's two streams go side by side, so steps that only some symbols take (escapes, a word more)
// are selections, not branches. Words: the lanes hold the next 16, replaced lane by lane every four symbols from the ones after
// them, which were asked for four symbols earlier; prior parameters are loaded 16 symbols ahead.
// 128 elements per stream: 6 144 streams 88 us, 28 800 305. (No gain: the first look-up in shared memory, 34 clocks instead of 106 but
// 33 KB to load per CTA; warp reductions instead of ballot and shuffles; the wide multiplication of inner_cum_of.)
__global__ void __launch_bounds__(kThreadsPerBlock) rans_decode_half_kernel(const RansArgs a, int q,
                                                                       const uint16_t* __restrict__ words,
                                                                       const uint32_t* __restrict__ counts,
                                                                       const int32_t* __restrict__ prior,
                                                                       int32_t* __restrict__ z) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  constexpr int kLanes = 16;
  extern __shared__ __align__(16) uint8_t smem[];
  uint32_t* sR = reinterpret_cast<uint32_t*>(smem);
  uint16_t* sG = reinterpret_cast<uint16_t*>(smem + 4 * a.n_scales);
  load_tables<kThreadsPerBlock>(a, sG, sR);
  const Tables t{sG, sR, a.umax, a.n_scales};
  const RansBlock blk = a.blocks[q];
  const int lane = threadIdx.x & (kLanes - 1), shift = threadIdx.x & 31 & ~(kLanes - 1);      // in the stream's lanes; the first of them
  const long wid = ((long)blockIdx.x * blockDim.x + threadIdx.x) / kLanes, total = (long)a.batch * blk.n_streams;
  if (((long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) / kLanes >= total) return;       // (no stream in the whole warp)
  const long me = min(wid, total - 1);                 // (a warp's second half may have none: it decodes nothing)
  const int b = (int)(me / blk.n_streams), j = (int)(me - (long)b * blk.n_streams), ns = blk.n_streams;
  const long sid = (long)b * a.n_streams + blk.first_stream + j;
  const int n_el = wid < total ? (int)((blk.n - j + ns - 1) / ns) : 0;
  const int top = (int)min((long)counts[sid], (long)a.cap);
  const uint16_t* in = words + sid * a.cap + top - 1;
  // word i from the stream's end, 0 before its first word
  auto word = [&](int i) { return i < top ? (uint32_t)in[-i] : 0u; };
  int used = 2, mine = lane;                           // words taken; the one that this lane holds (of used .. used + kLanes - 1)
  uint32_t win = word(lane), next = word(lane + kLanes), bad = 0;
  uint32_t x = __shfl_sync(kAll, win, 0, kLanes) << 16 | __shfl_sync(kAll, win, 1, kLanes);
  int32_t* zb = z + (long)b * a.d + blk.z_off + j;
  const int32_t* pb = prior + (long)b * 2 * a.d_fact;
  // this lane's element of the next kLanes: its prior parameters, a round ahead
  int32_t mu_n = 0;
  int ls_n = a.final_ls;
  if (lane < n_el) prior_of(a, blk, pb, j + (long)lane * ns, &mu_n, &ls_n, &bad);
  const int n_most = (int)__reduce_max_sync(kAll, (unsigned)n_el);      // (a warp's streams differ by one element at most)
  for (int i0 = 0; i0 < n_most; i0 += kLanes) {
    const int32_t mu_l = mu_n;
    const uint32_t R_l = t.R[ls_n], row_l = (uint32_t)ls_n << 8;
    if (i0 + kLanes + lane < n_el) prior_of(a, blk, pb, j + (long)(i0 + kLanes + lane) * ns, &mu_n, &ls_n, &bad);
    int32_t zv_l = 0;
    const int n_here = min(kLanes, n_most - i0);
    for (int ii = 0; ii < n_here; ++ii) {
      if ((ii & (kLanes / 4 - 1)) == 0 && mine < used) {          // (kLanes / 4 symbols take three quarters of the words at most)
        win = next;
        mine += kLanes;
        next = word(mine + kLanes);
      }
      // what does not depend on the state is on its way during the search
      const uint32_t R = __shfl_sync(kAll, R_l, ii, kLanes), row = __shfl_sync(kAll, row_l, ii, kLanes);
      const uint32_t w0 = __shfl_sync(kAll, win, used, kLanes), w1 = __shfl_sync(kAll, win, used + 1, kLanes);
      const uint32_t w2 = __shfl_sync(kAll, win, used + 2, kLanes);
      const uint32_t slot = x & 0xFFFFu;
      // largest k with Cum(k) <= slot, among the symbols that the slot can mean
      const uint32_t range = __ldg(a.ranges + row + (slot >> 8));
      int k = (int)(range & 0xFFFFu), d = (int)(range >> 16) - 1;            // k .. k + d
      auto last_below = [&](uint32_t c) {              // lane of the stream's last value that is not above the slot (Cum is monotone)
        return 31 - __clz((int)((__ballot_sync(kAll, c <= slot) >> shift) & (kAll >> (32 - kLanes))));
      };
      while (__any_sync(kAll, d > kLanes - 2)) {       // (at most twice)
        const int step = d > kLanes - 2 ? (d + kLanes) / kLanes : 1;
        k += last_below(cum_of(t, R, k + lane * step)) * step;
        d = step - 1;
      }
      const uint32_t cl = cum_of(t, R, k + lane);
      const int sel = last_below(cl);                  // at most kLanes - 2
      const uint32_t C = __shfl_sync(kAll, cl, sel, kLanes), Cn = __shfl_sync(kAll, cl, sel + 1, kLanes);
      k += sel;
      uint32_t y = (Cn - C) * (x >> 16) + slot - C;
      const bool more = y < (1u << 16), escape = k == 0 || k == 2 * kWin;
      if (more) y = (y << 16) | w0;
      // an escape: two symbols of frequency 1, the value's upper and lower half; each takes the state's lower 16 bits and
      // a word in their place (x >> 16 is always below 2^16)
      const uint32_t wa = more ? w1 : w0, wb = more ? w2 : w1;
      const int32_t zv = escape ? (int32_t)((y << 16) | wa) : (int32_t)((uint32_t)mu_l + (uint32_t)(k - kWin));      // (lane ii's counts)
      if (escape) y = (y & 0xFFFF0000u) | wb;
      if (lane == ii) zv_l = zv;
      if (i0 + ii < n_el) {
        x = y;
        used += (more ? 1 : 0) + (escape ? 2 : 0);
      }
    }
    if (i0 + lane < n_el) zb[(long)(i0 + lane) * ns] = zv_l;
  }
  if (n_el > 0 && (top != used || x != (1u << 16))) bad = 1u;    // every word used, none missing, and the state back at its start
  const unsigned any = __ballot_sync(kAll, bad != 0) >> shift & (kAll >> (32 - kLanes));
  if (any && lane == 0 && wid < total && a.errors) atomicAdd(a.errors, 1u);
}

// ---- compact byte stream -----------------------------------------------------------------------------
// Packed form of a batch's container (little endian):
//   uint32 offset[B + 1]      byte offset of image b's record from the start of the payload; offset[B] =
//                             payload bytes
//   payload, per image:       uint16 count[n_streams], then the words of stream 0, 1, ... back to back
// so an image's record is 2 * (n_streams + sum of its counts) bytes.

// exclusive scan of n values by one warp, 32 at a time; returns the total (in every lane)
template <typename Load, typename Store>
__device__ __forceinline__ uint32_t warp_scan(int n, int lane, Load load, Store store) {
  uint32_t run = 0;
  for (int base = 0; base < n; base += 32) {
    const int i = base + lane;
    const uint32_t v = i < n ? load(i) : 0u;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, inc, d);
      if (lane >= d) inc += o;
    }
    if (i < n) store(i, run + inc - v);
    run += __shfl_sync(0xFFFFFFFFu, inc, 31);
  }
  return run;
}

// record size of every image, in bytes
__global__ void pack_sizes_kernel(const uint32_t* __restrict__ counts, int n_streams, int cap, uint32_t* __restrict__ sizes) {
  __shared__ uint32_t part[8];
  const int b = blockIdx.x;
  uint32_t sum = 0;
  for (int s = threadIdx.x; s < n_streams; s += blockDim.x) sum += min(counts[(long)b * n_streams + s], (uint32_t)cap);
  sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
    sizes[b] = 2u * ((uint32_t)n_streams + t);
  }
}

// offset[0 .. B] from the sizes (one warp)
__global__ void pack_offsets_kernel(const uint32_t* __restrict__ sizes, int B, uint32_t* __restrict__ offset) {
  const int lane = threadIdx.x;
  const uint32_t total = warp_scan(B, lane, [&](int i) { return sizes[i]; }, [&](int i, uint32_t v) { offset[i] = v; });
  if (lane == 0) offset[B] = total;
}

// kPack: container -> records; !kPack: records -> container. One CTA per image.
constexpr int kCopyThreads = 1024;
template <bool kPack>
__global__ void __launch_bounds__(kCopyThreads) pack_copy_kernel(uint16_t* __restrict__ words, uint32_t* __restrict__ counts,
                                                        int n_streams, int cap, uint8_t* __restrict__ packed,
                                                        int B, unsigned long long payload_bytes, uint32_t* errors) {
  extern __shared__ uint32_t start[];       // word offset of every stream inside the record, after the counts
  __shared__ uint32_t bad;
  const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t* offset = reinterpret_cast<const uint32_t*>(packed);
  uint8_t* payload = packed + 4 * (size_t)(B + 1);
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  const uint32_t off = offset[b], end = offset[b + 1];
  // a record that does not fit the payload, or that cannot even hold its counts, is skipped
  const bool fits = kPack || (off <= end && end <= payload_bytes && (end - off) >= 2u * (uint32_t)n_streams && (off & 1u) == 0);
  uint16_t* rec = reinterpret_cast<uint16_t*>(payload + off);
  uint32_t* cnt = counts + (long)b * n_streams;
  if (!fits) {
    for (int s = threadIdx.x; s < n_streams; s += blockDim.x) cnt[s] = 0;
    if (threadIdx.x == 0 && errors) atomicAdd(errors, 1u);
    return;
  }
  if (warp == 0) {
    const uint32_t total = warp_scan(n_streams, lane,
        [&](int s) { return min(kPack ? cnt[s] : (uint32_t)rec[s], (uint32_t)cap); },
        [&](int s, uint32_t v) { start[s] = v; });
    if (lane == 0) {
      start[n_streams] = total;
      if (!kPack && 2u * ((uint32_t)n_streams + total) != end - off) bad = 1;    // counts disagree with the record size
    }
  }
  __syncthreads();
  if (bad) {
    for (int s = threadIdx.x; s < n_streams; s += blockDim.x) cnt[s] = 0;
    if (threadIdx.x == 0 && errors) atomicAdd(errors, 1u);
    return;
  }
  for (int s = threadIdx.x; s < n_streams; s += blockDim.x) {
    if (kPack) rec[s] = (uint16_t)min(cnt[s], (uint32_t)cap);
    else cnt[s] = min((uint32_t)rec[s], (uint32_t)cap);
  }
  uint16_t* body = rec + n_streams;
  for (int s = warp; s < n_streams; s += nwarps) {
    const uint32_t n = start[s + 1] - start[s];
    uint16_t* w = words + ((long)b * n_streams + s) * cap;
    uint16_t* r = body + start[s];
    for (uint32_t i = lane; i < n; i += 32) {
      if (kPack) r[i] = w[i]; else w[i] = r[i];
    }
  }
}

}  // namespace

cudaError_t launch_rans_pack(const RansArgs& a, const uint16_t* words, const uint32_t* counts, uint32_t* sizes,
                             uint8_t* packed, cudaStream_t stream) {
  pack_sizes_kernel<<<a.batch, 256, 0, stream>>>(counts, a.n_streams, a.cap, sizes);
  pack_offsets_kernel<<<1, 32, 0, stream>>>(sizes, a.batch, reinterpret_cast<uint32_t*>(packed));
  pack_copy_kernel<true><<<a.batch, kCopyThreads, 4 * (a.n_streams + 1), stream>>>(
      const_cast<uint16_t*>(words), const_cast<uint32_t*>(counts), a.n_streams, a.cap, packed, a.batch, 0ull, a.errors);
  return cudaGetLastError();
}

cudaError_t launch_rans_unpack(const RansArgs& a, const uint8_t* packed, unsigned long long payload_bytes,
                               uint16_t* words, uint32_t* counts, cudaStream_t stream) {
  pack_copy_kernel<false><<<a.batch, kCopyThreads, 4 * (a.n_streams + 1), stream>>>(
      words, counts, a.n_streams, a.cap, const_cast<uint8_t*>(packed), a.batch, payload_bytes, a.errors);
  return cudaGetLastError();
}

static size_t encode_smem(const RansArgs& a) { return encode_buffers_at(a) + 2 * kBatch * kEncodeStreams * (sizeof(EncodeSymbol) + 4); }

// The encoder's dynamic shared memory may exceed what a kernel has without asking: 48 KB, its static part included (tables of
// more than 5 947 entries a side with 64 scales). The limit belongs to the kernel, not to a codec or a launch: it is always
// the largest codec's, so that one codec cannot lower it under another's launch from a second thread.
cudaError_t configure_rans_kernels() {
  RansArgs largest{};
  largest.umax = kMaxRansUmax;
  largest.n_scales = kMaxRansScales;
  return cudaFuncSetAttribute(rans_encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)encode_smem(largest));
}

static size_t table_smem(const RansArgs& a) { return 4 * (size_t)a.n_scales + 2 * (size_t)(2 * a.umax + 1) + 16; }

// (No programmatic launch of the coder: started under a level's kernel, whose CTAs fill their SMs, the coder's CTAs all land
// on the few SMs that kernel leaves idle, +110 us on a decompression of 128 images.)
cudaError_t launch_rans_encode(const RansArgs& a, const int32_t* z, const int32_t* prior, uint16_t* words,
                               uint32_t* counts, cudaStream_t stream) {
  const long total = (long)a.batch * a.n_streams;
  const unsigned grid = (unsigned)((total + kEncodeStreams - 1) / kEncodeStreams);
  rans_encode_kernel<<<grid, kEncodeThreads, encode_smem(a), stream>>>(a, z, prior, words, counts);
  return cudaGetLastError();
}

cudaError_t launch_rans_decode(const RansArgs& a, int block, const uint16_t* words, const uint32_t* counts,
                               const int32_t* prior, int32_t* z, cudaStream_t stream) {
  const long streams = (long)a.batch * a.blocks[block].n_streams;
  const bool half = streams > (a.blocks[block].prior_off < 0 ? kHalfWarpStreamsPerSmOneScale : kHalfWarpStreamsPerSm) * a.n_sms;
  const long total = streams * (half ? 16 : 32);
  const unsigned grid = (unsigned)((total + kThreadsPerBlock - 1) / kThreadsPerBlock);
  if (half) rans_decode_half_kernel<<<grid, kThreadsPerBlock, table_smem(a), stream>>>(a, block, words, counts, prior, z);
  else rans_decode_kernel<<<grid, kThreadsPerBlock, table_smem(a), stream>>>(a, block, words, counts, prior, z);
  return cudaGetLastError();
}

}  // namespace iodf
