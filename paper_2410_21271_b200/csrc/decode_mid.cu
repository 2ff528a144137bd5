// Medium batches (9 to 32 tokens): one kernel computes Eq. 4 for a whole layer,
//     Y = X . deq(Wq) + (X . A) . B,
// in one pass over the weights, on mma.sync with the tokens as the narrow operand.
//
// Why not the tcgen05 kernel of prefill.cu.  With one token tile that kernel is bound by turning the weights into an fp16
// operand in shared memory and by a chain over the reduction axis per CTA, and t = X.A is a launch of its own in front: 134
// us for a block of LLaMA3-8B layers at 16 tokens, 14 % of HBM's rate.  Here the dequantised weights never leave
// the registers of the warp that multiplies them (a blob of 16 x 128 costs about 130 instructions and 16 mma per eight
// tokens: the tensor pipe and the issue slots are about even at 16 tokens, the tensor pipe leads at 32), and the layer
// is cut like in decode.cu: clusters of two CTAs own row tiles and split the reduction axis, sums meet in shared memory,
// t travels as self-validating words from clusters of its own.
//
// Work of a CTA.  Its row tiles go in pairs (32 rows share every activation fragment that is read from shared memory); kWarps /
// (pairs of row tiles) warps share one and take turns along the reduction axis, 128 elements at a time.  A warp keeps its
// sums in registers to the end; t . B is the end of the reduction axis (a CTA's half of every 128 columns of t).  X comes by TMA
// into a ring of 128-element slots, laid out as [32 k][token][32 fp16]: the eight tokens x 64 bytes that a
// fragment load of a warp reads are 512 contiguous bytes.  The warp that is the last to read a slot refills it.  The weights come through a ring per warp.  Weights
// are RN((q - z) * s) in fp16, as in prefill.cu, or, up to 16 tokens, exact q - z with the scale applied to the group's sums.
//
// Several adapters (EXACT): such a batch may as well go through decode.cu, eight tokens at a time, and its results must not
// depend on how many requests it happens to hold.  All operands are then multiplied as there: exact q - z at every number of tokens, t sent
// in fp32 and multiplied as an fp16 high and low part.  Rounding t once, and the weights from 17 tokens on, was 2.6 to 2000 times further
// from float64 (2048 x 1024, three adapters of rank 64, fp32 Y, 9 to 32 tokens: 3e-5 to 2e-4 of Y).
//
// Measured: four LLaMA3-8B blocks, 4-bit backbone and adapters, 16 tokens 544 -> 261 us (see also mid_supported).
#include <cuda.h>
#include "decode_common.cuh"

namespace eora {
namespace {
using namespace dec;

// Sixteen warps of 128 registers; a seventeenth as the producer of X would leave 96 (five warps share a scheduler's registers).
constexpr int kWarps = 16, kThreads = kWarps * 32;
constexpr int kMaxTokens = 32;            // tokens per launch
constexpr int kSegPitch = 36;             // floats from one token's 32 row sums to the next (36: the four token pairs of a store hit different banks)
constexpr int kMaxSmem = 226 * 1024;
constexpr int kMaxSlots = 4;
constexpr int kMaxXSlots = 32;

struct MidArgs {
  const uint8_t* a_q; const uint8_t* w_q; const uint8_t* b_q;
  int a_fmt;                              // format of A and B (FMT_NONE: no adapter)
  uint32_t a_sz2, b_sz2, a_blob;
  uint32_t np, pairs0;                    // pairs of the reduction axis; of its first half (rank 0's)
  uint32_t ks;                            // CTAs per cluster (1 if there is one pair only)
  uint32_t a_nt, n_a;                     // row tiles of A; CTAs that hold A
  Share a_tiles;                          // row tiles of A dealt to their clusters
  uint32_t w_nt;                          // row tiles of W
  Share w_dbl;                            // pairs of row tiles of W dealt to their clusters
  uint32_t xslots, a_xslots;              // slots of X, one pair each (W, A)
  uint32_t slots, ring_pitch;             // ring of a warp (W): slots of one pair of two row tiles
  uint32_t a_slots, a_pitch;              // ring of a warp (A): slots of one blob
  uint32_t off_ring, a_off_ring, off_inbox;      // shared memory: X slots | rings; later, over both, the warps' sums | the partner's sums
  void* ys[4];
  uint32_t sub_tile0[5];                  // layer i owns row tiles [sub_tile0[i], sub_tile0[i + 1]) and pairs [i, i + 1) * sub_pairs of t
  int sub_dout[4];
  int n_sub;
  uint32_t sub_pairs, b_np;               // as in decode.cu
  uint32_t t_chunk;                       // pairs of t in shared memory at a time
  uint32_t adp_pairs;                     // several adapters: pair p of t belongs to adapter p / adp_pairs (0: one adapter)
  signed char adp[kMaxTokens];              // adapter of every token (-1: none)
  unsigned long long* t_part;             // [m][t_cols / 2] words (two columns as fp16, launch number); EXACT: [m][t_cols] words (fp32, launch number)
  unsigned long long* launches;
  int* dev_status;
  int m, m_log, t_cols, y_dtype;
  unsigned long long wait_ns;
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
               ::"r"(dst), "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t h2mul(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// Scale entry of a tile: scales of rows g / g + 8 as fp16 pairs, zero-point constants.
struct SZ { uint32_t s[2]; ZC zc; };
template <int FMT>
__device__ __forceinline__ void load_sz(SZ& z, uint32_t entry, int lane) {
  const uint32_t sw = lds_u1(entry + (lane >> 2) * 4);
  z.s[0] = prmt(sw, 0u, 0x1010u); z.s[1] = prmt(sw, 0u, 0x3232u);
  make_zc<FMT>(z.zc, lds_u16(entry + 32 + (lane >> 2) * 2));
}

// The wide operand of a 32-element block's two mma: RN((q - z) * s) in fp16, or (SCALED false) the exact q - z.
template <int FMT, bool SCALED>
__device__ __forceinline__ void weights_half(const RawTile<FMT>& r, int blk, const SZ& z, uint32_t lut, uint32_t (&a)[2][4]) {
  half_frags<FMT>(r, z.zc, blk, a[0], a[1], lut);
  if constexpr (SCALED && fmt_quantised(FMT)) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) a[i][e] = h2mul(a[i][e], z.s[e & 1]);
  }
}

// One pair of T row tiles (blobs `stride` apart) times the activations of 8 NT tokens at x: [4 blocks of 32 k][8 NT tokens][32 fp16],
// x already at this lane's token and piece.  Up to 16 tokens the scale of a quantised group is applied to the group's sums (8 NT T multiplications
// a lane instead of 32 T on the weights); with more the sums would need as many registers again.
// EXACT: the scale is always applied to the sums.
template <int FMT, bool SZ2, int NT, int T, bool EXACT>
__device__ __forceinline__ void product(uint32_t blob, uint32_t stride, int lane, uint32_t x, uint32_t lut, float (*acc)[NT][4]) {
  constexpr int tb = tile_bytes(FMT);
  constexpr bool late = fmt_quantised(FMT) && (NT <= 2 || EXACT);
  SZ z[T];
  float d[late ? T : 1][late ? NT : 1][4];
  if constexpr (late) {
#pragma unroll
    for (int u = 0; u < T; ++u)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) d[u][n][i] = 0.f;
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    RawTile<FMT> r[T];
#pragma unroll
    for (int u = 0; u < T; ++u) {
      if constexpr (fmt_quantised(FMT)) { if (c == 0 || SZ2) load_sz<FMT>(z[u], blob + u * stride + 2 * tb + c * kSzEntryBytes, lane); }
      load_tile_s<FMT>(r[u], blob + u * stride + c * tb, lane);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      uint32_t a[T][2][4];
#pragma unroll
      for (int u = 0; u < T; ++u) weights_half<FMT, !late>(r[u], b, z[u], lut, a[u]);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const uint4 v = lds_u4(x + (2 * c + b) * (NT * 512) + n * 512);
#pragma unroll
        for (int u = 0; u < T; ++u) mma16816(late ? d[late ? u : 0][late ? n : 0] : acc[u][n], a[u][0], v.x, v.y);
#pragma unroll
        for (int u = 0; u < T; ++u) mma16816(late ? d[late ? u : 0][late ? n : 0] : acc[u][n], a[u][1], v.z, v.w);
      }
    }
    if constexpr (late) {
      if (c == 1 || SZ2) {
#pragma unroll
        for (int u = 0; u < T; ++u) {
          const float sa = __half2float(__ushort_as_half((unsigned short)z[u].s[0])), sb = __half2float(__ushort_as_half((unsigned short)z[u].s[1]));
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              acc[u][n][i] = fmaf(d[u][n][i], i < 2 ? sa : sb, acc[u][n][i]);
              d[u][n][i] = 0.f;
            }
        }
      }
    }
  }
}

// The sums of exact products join a row tile's, with the group's scales.
template <int NT>
__device__ __forceinline__ void add_scaled(float (&acc)[NT][4], float (&d)[NT][4], const SZ& z) {
  const float sa = __half2float(__ushort_as_half((unsigned short)z.s[0])), sb = __half2float(__ushort_as_half((unsigned short)z.s[1]));
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[n][i] = fmaf(d[n][i], i < 2 ? sa : sb, acc[n][i]);
      d[n][i] = 0.f;
    }
}

// A and B: the format is known at run time only (one uniform branch per blob).
// A: a blob times a pair of X, as above.
template <int FMT, int NT, bool EXACT>
__device__ __forceinline__ void product_a1(uint32_t blob, uint32_t sz2, int lane, uint32_t x, float (&acc)[NT][4]) {
  constexpr int tb = tile_bytes(FMT);
  constexpr bool late = EXACT && fmt_quantised(FMT);
  float d[late ? NT : 1][4];
  if constexpr (late) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) d[n][i] = 0.f;
  }
  SZ z;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if constexpr (fmt_quantised(FMT)) { if (c == 0 || sz2) load_sz<FMT>(z, blob + 2 * tb + c * kSzEntryBytes, lane); }
    RawTile<FMT> r;
    load_tile_s<FMT>(r, blob + c * tb, lane);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      uint32_t a[2][4];
      weights_half<FMT, !late>(r, b, z, 0u, a);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const uint4 v = lds_u4(x + (2 * c + b) * (NT * 512) + n * 512);
        mma16816(late ? d[late ? n : 0] : acc[n], a[0], v.x, v.y);
        mma16816(late ? d[late ? n : 0] : acc[n], a[1], v.z, v.w);
      }
    }
    if constexpr (late) { if (c == 1 || sz2) add_scaled<NT>(acc, d, z); }
  }
}
template <int NT, bool EXACT>
__device__ __forceinline__ void product_a(int fmt, uint32_t sz2, uint32_t blob, int lane, uint32_t x, float (&acc)[NT][4]) {
  switch (fmt) {
    case FMT_F16: product_a1<FMT_F16, NT, EXACT>(blob, 0u, lane, x, acc); break;
    case FMT_Q8: product_a1<FMT_Q8, NT, EXACT>(blob, 0u, lane, x, acc); break;
    case FMT_Q4: product_a1<FMT_Q4, NT, EXACT>(blob, sz2, lane, x, acc); break;
    case FMT_Q3: product_a1<FMT_Q3, NT, EXACT>(blob, sz2, lane, x, acc); break;
    default: break;
  }
}
// B: one 64-element tile of each of two row tiles, each with its scale entry behind it (kBStride bytes apart), times 64 columns of t
// (EXACT: their high part, the low part behind it).
template <int FMT> constexpr uint32_t kBStride = tile_bytes(FMT) + 64;
template <int FMT, int NT, bool EXACT>
__device__ __forceinline__ void product_b1(uint32_t buf, int lane, uint32_t x, float (&acc)[2][NT][4]) {
  constexpr bool late = EXACT && fmt_quantised(FMT);
  float d[late ? NT : 1][4];
  if constexpr (late) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) d[n][i] = 0.f;
  }
  // one row tile after the other: an fp16 tile is 16 registers a lane
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    SZ z;
    if constexpr (fmt_quantised(FMT)) load_sz<FMT>(z, buf + u * kBStride<FMT> + tile_bytes(FMT), lane);
    RawTile<FMT> r;
    load_tile_s<FMT>(r, buf + u * kBStride<FMT>, lane);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      uint32_t a[2][4];
      weights_half<FMT, !late>(r, b, z, 0u, a);
#pragma unroll
      for (int p = 0; p < (EXACT ? 2 : 1); ++p)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint4 v = lds_u4(x + p * (NT * 1024) + b * (NT * 512) + n * 512);
          mma16816(late ? d[late ? n : 0] : acc[u][n], a[0], v.x, v.y);
          mma16816(late ? d[late ? n : 0] : acc[u][n], a[1], v.z, v.w);
        }
    }
    if constexpr (late) add_scaled<NT>(acc[u], d, z);
  }
}
template <int NT, bool EXACT>
__device__ __forceinline__ void product_b(int fmt, uint32_t buf, int lane, uint32_t x, float (&acc)[2][NT][4]) {
  switch (fmt) {
    case FMT_F16: product_b1<FMT_F16, NT, EXACT>(buf, lane, x, acc); break;
    case FMT_Q8: product_b1<FMT_Q8, NT, EXACT>(buf, lane, x, acc); break;
    case FMT_Q4: product_b1<FMT_Q4, NT, EXACT>(buf, lane, x, acc); break;
    case FMT_Q3: product_b1<FMT_Q3, NT, EXACT>(buf, lane, x, acc); break;
    default: break;
  }
}

__device__ __forceinline__ int sub_of(const MidArgs& p, uint32_t tile) {
  if (p.n_sub == 1) return 0;
  int s = 0;
#pragma unroll
  for (int i = 1; i < 4; ++i)
    if (i < p.n_sub && tile >= p.sub_tile0[i]) s = i;
  return s;
}
// NT: tokens / 8.  EXACT: several adapters (see above).
template <int WF, bool SZ2, int NT, bool EXACT>
__global__ void __launch_bounds__(kThreads, 1) k_mid(const __grid_constant__ CUtensorMap tm, const __grid_constant__ MidArgs p) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(256) uint32_t lut_s[16];
  __shared__ __align__(8) uint64_t xbars_s[kMaxXSlots], bars_s[kWarps * kMaxSlots];
  __shared__ uint32_t readers_s[kMaxXSlots];       // warps that are done with a slot of X
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  asm volatile("griddepcontrol.launch_dependents;");
  const bool is_a = blockIdx.x < p.n_a;
  const uint32_t cta = is_a ? blockIdx.x : blockIdx.x - p.n_a;
  const uint32_t cl = p.ks == 2 ? cta >> 1 : cta, rank = p.ks == 2 ? cta & 1 : 0;
  const uint32_t d0 = share_lo(is_a ? p.a_tiles : p.w_dbl, cl), nD = share_n(is_a ? p.a_tiles : p.w_dbl, cl);
  const uint32_t P = rank ? p.np - p.pairs0 : p.pairs0, pr0 = rank ? p.pairs0 : 0u;
  const uint32_t xs = smem_u32(smem), xfull = smem_u32(xbars_s);
  constexpr uint32_t kXSlot = NT * 2048, kTHalf = EXACT ? NT * 2048 : NT * 1024;      // bytes of a pair of X; of 64 columns of t
  uint32_t lut = 0;
  if constexpr (WF == FMT_SP24 || WF == FMT_SQ4) lut = sp24_lut(lut_s);
  if (warp == 0 && lane < kMaxXSlots) {
    mbar_init_a(xfull + 8 * lane, 1);
    readers_s[lane] = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }

  // this warp's place: unit d (row tile of A, pair of row tiles of W), every wpt-th pair of the reduction axis from j on
  // The slots of X are a multiple of wpt, so a slot's pairs are always read by the same warps: none of them can be a phase of the
  // slot's barrier ahead.
  const uint32_t max_x = is_a ? p.a_xslots : p.xslots, wpt = min(kWarps / nD, max_x), xslots = max_x - max_x % wpt;
  const uint32_t d = warp / wpt, j = warp - d * wpt;
  const bool active = d < nD;
  Ring ring;
  const uint32_t blob_b = is_a ? p.a_blob : (uint32_t)blob_bytes(WF, SZ2 ? 1 : 0);
  const uint32_t slot_b = is_a ? p.a_blob : 2 * blob_b, slots = is_a ? p.a_slots : p.slots;
  ring.base = smem_u32(smem + (is_a ? p.a_off_ring : p.off_ring)) + warp * (is_a ? p.a_pitch : p.ring_pitch);
  ring.bytes = slots * slot_b; ring.bars = ring.bar = smem_u32(bars_s) + warp * (kMaxSlots * 8); ring.so = 0; ring.parity = 0;
  // first blob of the unit's first row tile in this half of the reduction axis, and from there to its second row tile
  const uint8_t* w0 = is_a ? p.a_q + ((size_t)(d0 + d) * p.np + pr0) * blob_b
                           : p.w_q + ((size_t)rank * p.w_nt * p.pairs0 + (size_t)(d0 + d) * 2 * P) * blob_b;
  uint32_t l_q = j;                                // the next pair to be asked for
  auto ask = [&](uint32_t so, uint32_t bar) {
    if (l_q >= P) return;
    if (lane == 0) {
      const uint8_t* src = w0 + (size_t)l_q * blob_b;
      mbar_expect_tx_a(bar, slot_b);
      bulk_g2s_a(ring.base + so, src, blob_b, bar);
      if (!is_a) bulk_g2s_a(ring.base + so + blob_b, src + (size_t)P * blob_b, blob_b, bar);
    }
    l_q += wpt;
  };
  if (active) {
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < kMaxSlots; ++i) mbar_init_a(ring.bars + 8 * i, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    for (uint32_t i = 0, so = 0, b = ring.bars; i < slots; ++i, so += slot_b, b += 8) ask(so, b);
  }
  if (!is_a && p.n_a) {                            // blobs of B towards L2 (the partner reads the other halves of them)
    const uint32_t per = p.b_np * (uint32_t)blob_bytes(p.a_fmt, (int)p.b_sz2), bytes = 2 * nD * per;
    const uint8_t* b_part = p.b_q + (size_t)(2 * d0) * per;
    for (uint32_t o = (threadIdx.x * p.ks + rank) << 13; o < bytes; o += (kThreads * p.ks) << 13) prefetch_l2(b_part + o, min(8192u, bytes - o));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();                                 // the barriers of X are set up
  const uint32_t launch = launch_number(p.launches);
  bool ok = true;
  constexpr int T = 2;
  float acc[T][NT][4];
#pragma unroll
  for (int u = 0; u < T; ++u)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[u][n][i] = 0.f;

  auto load_x = [&](uint32_t q, uint32_t s) {      // pair q into slot s; one lane
    mbar_expect_tx_a(xfull + 8 * s, kXSlot);
    tma_load_3d(xs + s * kXSlot, &tm, 0, 0, (int)((pr0 + q) * 4), xfull + 8 * s);
  };
  if (lane == 0)
    for (uint32_t q = warp; q < min(P, xslots); q += kWarps) load_x(q, q);
  if (active) {
    const uint32_t xl = xs + (lane >> 2) * 64 + (lane & 3) * 16;
    uint32_t s = j, par = 0;
#pragma unroll 1
    for (uint32_t q = j; q < P; q += wpt) {
      if (ok && !mbar_try_wait_a(ring.bar, ring.parity) && !mbar_wait_lane(ring.bar, ring.parity, p.dev_status)) ok = false;
      if (ok && !mbar_try_wait_a(xfull + 8 * s, par) && !mbar_wait_lane(xfull + 8 * s, par, p.dev_status)) ok = false;
      if (!__all_sync(0xffffffffu, ok)) {          // gave up: what is in flight for this warp must land first, weights and the slots of X that it reads
        ok = false;
        for (uint32_t i = 0; i < slots; ++i) mbar_drain_warp(ring.bars + 8 * i, ring.bars + 8 * i < ring.bar ? ring.parity ^ 1u : ring.parity, lane);
        for (uint32_t i = j; i < xslots; i += wpt) mbar_drain_warp(xfull + 8 * i, i < s ? par ^ 1u : par, lane);
        break;
      }
      const uint32_t src = ring.base + ring.so, x = xl + s * kXSlot;
      if (is_a) {
        product_a<NT, EXACT>(p.a_fmt, p.a_sz2, src, lane, x, acc[0]);
      } else if constexpr (EXACT && NT > 2 && fmt_quantised(WF)) {      // one row tile after the other: sums of both would not fit the registers
#pragma unroll
        for (int u = 0; u < T; ++u) product<WF, SZ2, NT, 1, true>(src + u * blob_b, blob_b, lane, x, lut, acc + u);
      } else {
        product<WF, SZ2, NT, T, EXACT>(src, blob_b, lane, x, lut, acc);
      }
      __syncwarp();                                // every lane is done with both slots
      if (lane == 0 && q + xslots < P) {           // a pair of X is read by one warp per unit
        uint32_t done = nD - 1;
        if (nD > 1) asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], %2;" : "=r"(done) : "r"(smem_u32(readers_s + s)), "r"(1u) : "memory");
        if (done == nD - 1) { readers_s[s] = 0u; load_x(q + xslots, s); }
      }
      ask(ring.so, ring.bar);
      ring_next(ring, slot_b);
      s += wpt;
      if (s >= xslots) { s = j; par ^= 1u; }
    }
  }

  // ---- + t . B: this CTA's 64 of every 128 columns of t (all, if it has no partner)
  if (!is_a && p.n_a) {
    const uint32_t tile = 2 * (d0 + d), base = p.sub_pairs && active ? (uint32_t)sub_of(p, tile) * p.sub_pairs : 0u;
    const uint32_t h_log = p.ks == 2 ? 0u : 1u, m_mask = (1u << p.m_log) - 1;      // halves of a pair that are this CTA's
    uint32_t c0 = 0, c_end = p.b_np;               // chunk of t (pairs), end of all chunks
    if (p.sub_pairs) { c0 = (uint32_t)sub_of(p, 2 * d0) * p.sub_pairs; c_end = (uint32_t)(sub_of(p, 2 * (d0 + nD) - 1) + 1) * p.sub_pairs; }
    const uint32_t tb = (uint32_t)tile_bytes(p.a_fmt), stride = tb + 64, sz = fmt_quantised(p.a_fmt) ? (uint32_t)kSzEntryBytes : 0u;
    const uint32_t b_blob = (uint32_t)blob_bytes(p.a_fmt, (int)p.b_sz2);
    // unit h of a chunk: pair c0 + (h >> h_log), half `c` of it; a warp takes every wpt-th one of its layer's
    auto half_of = [&](uint32_t h) { return p.ks == 2 ? rank : h & 1u; };
    auto ask_b = [&](uint32_t h) {                 // to the start of the (empty) ring
      if (lane == 0) {
        const uint32_t c = half_of(h), pair = c0 + (h >> h_log) - base;
        mbar_expect_tx_a(ring.bar, 2 * (tb + sz));
#pragma unroll
        for (uint32_t u = 0; u < 2; ++u) {
          const uint8_t* blob = p.b_q + ((size_t)(tile + u) * p.b_np + pair) * b_blob;
          bulk_g2s_a(ring.base + u * stride, blob + c * tb, tb, ring.bar);
          if (sz) bulk_g2s_a(ring.base + u * stride + tb, blob + 2 * tb + (p.b_sz2 ? c * sz : 0u), sz, ring.bar);
        }
      }
    };
    auto span = [&](uint32_t& h, uint32_t& h_end) {          // the warp's first unit of the chunk, the end of its layer's
      const uint32_t lo = max(c0, base), hi = min(min(c0 + p.t_chunk, c_end), base + p.b_np);
      h = hi > lo ? ((lo - c0) << h_log) + j : 0u;
      h_end = hi > lo ? (hi - c0) << h_log : 0u;
    };
    // step e of a chunk: two words of one token, i.e. four columns (16 steps per half and token) or, EXACT, two (32 steps)
    constexpr uint32_t kSLog = EXACT ? 5 : 4, kSteps = 1u << kSLog, kWordCols = EXACT ? 1 : 2;
    auto t_src = [&](uint32_t e, uint32_t& tok, uint32_t& col) {
      const uint32_t h = e >> (kSLog + p.m_log);
      tok = (e >> kSLog) & m_mask;
      col = (c0 + (h >> h_log)) * 128 + half_of(h) * 64 + (e & (kSteps - 1)) * (2 * kWordCols);
      return p.t_part + ((size_t)tok * p.t_cols + col) / kWordCols;
    };
    uint32_t h, h_end, tok, col;
    span(h, h_end);
    if (ok && active && h < h_end) ask_b(h);
    bool asked = true;
#pragma unroll 1
    for (;;) {
      // t as fp16 (EXACT: high and low part, error 2^-22 of the value), zero for tokens that do not use the pair's adapter and in the columns past A's rows (padding); the loads of a batch
      // go out together (each is a round trip to L2), those of the first before the barrier
      constexpr int kBatch = 2;
      const uint32_t steps = (min(p.t_chunk, c_end - c0) << h_log) << (kSLog + p.m_log);
#pragma unroll 1
      for (uint32_t e0 = 0; e0 < steps; e0 += kBatch * kThreads) {
        TWords tw[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
          const uint32_t e = e0 + k * kThreads + threadIdx.x;
          const unsigned long long* src = t_src(e, tok, col);
          if (e < steps && tok < (uint32_t)p.m) load_t(tw[k], src);
        }
        if (e0 == 0) __syncthreads();              // every warp is done with X (with the chunk before)
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
          const uint32_t e = e0 + k * kThreads + threadIdx.x;
          const unsigned long long* src = t_src(e, tok, col);
          if (e >= steps || tok >= (uint32_t)p.m) continue;
          uint32_t v0 = 0u, v1 = 0u;
          if (col < p.a_nt * 16 && !(p.adp_pairs && p.adp[tok] != (int)((col >> 7) / p.adp_pairs)) &&
              wait_t(tw[k], src, launch, p.wait_ns, p.dev_status)) { v0 = (uint32_t)tw[k].a; v1 = (uint32_t)tw[k].b; }
          const uint32_t i = e & (kSteps - 1), blk = i >> (kSLog - 1), in_blk = i & (kSteps / 2 - 1);      // 32 columns = 64 bytes
          const uint32_t dst = xs + (e >> (kSLog + p.m_log)) * kTHalf + blk * (NT * 512) + tok * 64 + in_blk * (128 / kSteps);
          if constexpr (EXACT) {
            const float f0 = __uint_as_float(v0), f1 = __uint_as_float(v1);
            const uint32_t hi = pack_h2(f0, f1);
            const float2 hf = __half22float2(*reinterpret_cast<const __half2*>(&hi));
            sts_u1(dst, hi);
            sts_u1(dst + NT * 1024, pack_h2(f0 - hf.x, f1 - hf.y));
          } else {
            asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(dst), "r"(v0), "r"(v1) : "memory");
          }
        }
      }
      __syncthreads();
      if (active) {
#pragma unroll 1
        for (; ok && h < h_end; h += wpt, asked = false) {      // (a warp that gave up asks for nothing more)
          if (!asked) ask_b(h);
          if (!mbar_try_wait_a(ring.bar, ring.parity) && !mbar_wait_lane(ring.bar, ring.parity, p.dev_status)) ok = false;
          if (!__all_sync(0xffffffffu, ok)) {
            ok = false;
            mbar_drain_warp(ring.bar, ring.parity, lane);
            break;
          }
          ring.parity ^= 1u;
          // (columns of tokens past m hold whatever was there: their sums are not read)
          product_b<NT, EXACT>(p.a_fmt, ring.base, lane, xs + h * kTHalf + (lane >> 2) * 64 + (lane & 3) * 16, acc);
          __syncwarp();
        }
      }
      c0 += p.t_chunk;
      if (c0 >= c_end) break;
      asked = false;
      span(h, h_end);
    }
  }

  // ---- sums: every warp's into a slot of its own, over X and the rings; the partner's row tiles to the partner
  if (p.ks == 2) { cluster_arrive(); cluster_wait(); } else __syncthreads();       // nobody needs X and the rings any more
  float* const seg = reinterpret_cast<float*>(smem);
  float* const inbox = reinterpret_cast<float*>(smem + p.off_inbox);
  constexpr uint32_t kSlot = NT * 8 * kSegPitch;   // floats of a warp's slot: [token][32 rows, pitch 36]
  if (active) {
    float* s = seg + warp * kSlot + (lane & 3) * (2 * kSegPitch) + (lane >> 2);
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int u = 0; u < T; ++u) {
        float* q = s + n * 8 * kSegPitch + u * 16;
        q[0] = acc[u][n][0]; q[kSegPitch] = acc[u][n][1]; q[8] = acc[u][n][2]; q[kSegPitch + 8] = acc[u][n][3];
      }
  }
  __syncthreads();
  // this CTA finishes row tiles [first, first + nf) of the cluster's nT
  const uint32_t nT = is_a ? nD : 2 * nD, first = rank ? nT >> 1 : 0u, nf = (p.ks == 2 && rank == 0 ? nT >> 1 : nT) - first;
  const uint32_t hw = threadIdx.x >> 4, row = threadIdx.x & 15, m = p.m, OT = 16 * m;
  constexpr uint32_t kHalfWarps = kThreads / 16;
  // four tokens of a row tile at once (independent loads: in a rolled loop each costs its latency), summed over the warps that share it
  auto tile_sum = [&](uint32_t f, uint32_t tok, float (&v)[4]) {
    const float* s = seg + tok * kSegPitch + row + (is_a ? f * wpt * kSlot : (f >> 1) * wpt * kSlot + (f & 1) * 16);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = s[i * kSegPitch];
#pragma unroll 2
    for (uint32_t k = 1; k < wpt; ++k) {
      s += kSlot;
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] += s[i * kSegPitch];
    }
  };
  const uint32_t q_log = p.m_log - 2, q_mask = (1u << q_log) - 1;      // groups of four tokens
  if (p.ks == 2) {                                 // the partner's row tiles
    const uint32_t s0 = rank ? 0u : nf, ns = nT - nf;
    const uint32_t to = mapa(smem_u32(inbox), rank ^ 1u) + row * 4;
    for (uint32_t u = hw; u < ns << q_log; u += kHalfWarps) {
      const uint32_t f = u >> q_log, tok = (u & q_mask) * 4;
      float v[4];
      tile_sum(s0 + f, tok, v);
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i)
        if (tok + i < m) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to + (f * OT + (tok + i) * 16) * 4), "f"(v[i]) : "memory");
    }
    cluster_arrive();
    cluster_wait();
  }
  // (m_log >= 4: nf << q_log is even, so the halves of a warp take part alike)
  for (uint32_t u = hw; u < nf << q_log; u += kHalfWarps) {
    const uint32_t f = u >> q_log, tok = (u & q_mask) * 4;
    float v[4];
    tile_sum(first + f, tok, v);
    if (p.ks == 2) {
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) v[i] += inbox[f * OT + min(tok + i, m - 1) * 16 + row];      // (past m: any, not stored)
    }
    if (is_a && EXACT) {                           // a column of t per word
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i)
        if (tok + i < m) {
          const unsigned long long word = ((unsigned long long)launch << 32) | __float_as_uint(v[i]);
          asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p.t_part + (size_t)(tok + i) * p.t_cols + (d0 + first + f) * 16 + row), "l"(word) : "memory");
        }
    } else if (is_a) {                             // two columns of t per word
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        const float o = __shfl_down_sync(0xffffffffu, v[i], 1);
        if (tok + i < m && !(row & 1)) {
          const unsigned long long word = ((unsigned long long)launch << 32) | pack_h2(v[i], o);
          asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p.t_part + ((size_t)(tok + i) * p.t_cols + (d0 + first + f) * 16 + row) / 2), "l"(word) : "memory");
        }
      }
    } else {
      const uint32_t tg = 2 * d0 + first + f;
      void* y = p.ys[0];
      uint32_t st0 = 0;
      int dout = p.sub_dout[0];
      if (p.n_sub > 1) {
#pragma unroll
        for (int k = 1; k < 4; ++k)
          if (k < p.n_sub && tg >= p.sub_tile0[k]) { y = p.ys[k]; st0 = p.sub_tile0[k]; dout = p.sub_dout[k]; }
      }
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i)
        if (tok + i < m) store_y(y, p.y_dtype, (int64_t)(tok + i) * dout + (tg - st0) * 16 + row, v[i]);
    }
  }
  __syncthreads();                                 // every thread of the CTA has read the launch counter
  if (threadIdx.x == 0) count_launch(p.launches);
}

// ---------------------------------------------------------------------------------------------- host
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    return cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess ? reinterpret_cast<EncodeTiledFn>(p) : nullptr;
  }();
  return fn;
}

// X [m][d_in] fp16 as (k within a block of 32, token, block of 32 k); the box brings a pair (4 blocks) of all tokens (zeros past m)
bool make_map(CUtensorMap* tm, const void* x, int m, int d_in, int tokens) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {32, (cuuint64_t)m, (cuuint64_t)d_in / 32};
  cuuint64_t strides[2] = {(cuuint64_t)d_in * 2, 64};
  cuuint32_t box[3] = {32, (cuuint32_t)tokens, 4};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <auto KERNEL>
cudaError_t launch_kernel(const cudaLaunchConfig_t& cfg, const CUtensorMap& tm, const MidArgs& a, int device) {
  static bool attr_set[64] = {};
  if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[device]) {
    cudaError_t e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e != cudaSuccess) return e;
    attr_set[device] = true;
  }
  return cudaLaunchKernelEx(&cfg, KERNEL, tm, a);
}
template <int WF, bool SZ2>
cudaError_t launch_nt(const cudaLaunchConfig_t& cfg, const CUtensorMap& tm, const MidArgs& a, int nt, int device) {
  if (a.adp_pairs) return nt == 2 ? launch_kernel<k_mid<WF, SZ2, 2, true>>(cfg, tm, a, device) : launch_kernel<k_mid<WF, SZ2, 4, true>>(cfg, tm, a, device);
  return nt == 2 ? launch_kernel<k_mid<WF, SZ2, 2, false>>(cfg, tm, a, device) : launch_kernel<k_mid<WF, SZ2, 4, false>>(cfg, tm, a, device);
}
cudaError_t launch_any(const cudaLaunchConfig_t& cfg, const CUtensorMap& tm, const MidArgs& a, int wf, bool sz2, int nt, int device) {
  switch (wf) {
    case FMT_Q4: return sz2 ? launch_nt<FMT_Q4, true>(cfg, tm, a, nt, device) : launch_nt<FMT_Q4, false>(cfg, tm, a, nt, device);
    case FMT_Q3: return sz2 ? launch_nt<FMT_Q3, true>(cfg, tm, a, nt, device) : launch_nt<FMT_Q3, false>(cfg, tm, a, nt, device);
    case FMT_SQ4: return sz2 ? launch_nt<FMT_SQ4, true>(cfg, tm, a, nt, device) : launch_nt<FMT_SQ4, false>(cfg, tm, a, nt, device);
    case FMT_SP24: return launch_nt<FMT_SP24, false>(cfg, tm, a, nt, device);
    default: return cudaErrorInvalidValue;
  }
}

Share make_share(uint32_t total, uint32_t n) { return {n ? total / n : 0, n ? total % n : 0}; }

struct Plan { MidArgs a; int grid, smem, nt; };

// How a launch of m (at most 32) tokens is cut up; false if its shared memory does not fit.
bool make_plan(const Handle* h, int m, Plan& pl) {
  MidArgs& a = pl.a;
  a = MidArgs();
  const bool ab = h->cfg.rank > 0;
  const int NT = m <= 16 ? 2 : 4;
  pl.nt = NT;
  a.m = m;
  while ((1 << a.m_log) < m) ++a.m_log;
  a.w_q = h->w.q; a.w_nt = h->w.nt; a.np = h->w.np; a.pairs0 = h->w.half;
  a.ks = h->w.np >= 2 ? 2 : 1;
  const uint32_t sms = (uint32_t)h->sm_count / a.ks * a.ks, cls = sms / a.ks, nd = h->w.nt / 2;
  const uint32_t most_x = 131072u / (NT * 2048) < (uint32_t)kMaxXSlots ? 131072u / (NT * 2048) : kMaxXSlots;
  auto blobs = [&](uint32_t per) {                 // blobs of a CTA with `per` units, idle turns included
    uint32_t wpt = per >= (uint32_t)kWarps ? 1u : (uint32_t)kWarps / per;
    if (wpt > most_x) wpt = most_x;
    return (double)per * wpt * ((a.pairs0 + wpt - 1) / wpt);
  };
  if (ab) {
    a.a_fmt = h->a.fmt; a.a_q = h->a.q; a.a_nt = h->a.nt; a.a_sz2 = h->a.sz2; a.a_blob = h->a.blob;
    a.b_q = h->b.q; a.b_np = h->b.np; a.b_sz2 = h->b.sz2;
    // Clusters for A: t should be there when the products with W are done (an exchange through L2 takes about as long as 24
    // blobs of a CTA's).
    double best = 1e30;
    uint32_t best_n = 1;
    for (uint32_t n = 1; n <= cls / 2 && n <= (uint32_t)h->a.nt; ++n) {
      const uint32_t per_a = (h->a.nt + n - 1) / n, per_w = (nd + cls - n - 1) / (cls - n);
      if (per_a > (uint32_t)kWarps || per_w > (uint32_t)kWarps) continue;
      const double ta = 24.0 + 1.2 * blobs(per_a), tw = 2.0 * blobs(per_w), t = ta > tw ? ta : tw;
      if (t < 0.99 * best) { best = t; best_n = n; }
    }
    if ((h->a.nt + best_n - 1) / best_n > (uint32_t)kWarps) best_n = (h->a.nt + (uint32_t)kWarps - 1) / (uint32_t)kWarps;
    a.n_a = best_n * a.ks;
    a.a_tiles = make_share(h->a.nt, best_n);
    a.sub_pairs = h->n_sub > 1 ? (uint32_t)h->r_pad / 128 : 0u;
  }
  uint32_t ncl = cls > a.n_a / a.ks ? cls - a.n_a / a.ks : 1;
  if (ncl > nd) ncl = nd;
  if ((nd + ncl - 1) / ncl > (uint32_t)kWarps) ncl = (nd + (uint32_t)kWarps - 1) / (uint32_t)kWarps;      // more than fit at once: in waves
  a.w_dbl = make_share(nd, ncl);
  pl.grid = (int)(a.n_a + ncl * a.ks);
  if (pl.grid >= (1 << kLaunchShift)) return false;
  const uint32_t nD = a.w_dbl.per + (a.w_dbl.rem ? 1 : 0);
  auto up = [](uint32_t v) { return (v + 127u) & ~127u; };
  const uint32_t t_half = (h->multi ? 2u : 1u) * NT * 1024 * (a.ks == 2 ? 1 : 2);      // bytes of a CTA's part of 128 columns of t
  const uint32_t x_slot = NT * 2048, seg_b = kWarps * 8 * NT * kSegPitch * 4;
  a.off_inbox = up(seg_b);
  const uint32_t per_a = a.a_tiles.per + (a.a_tiles.rem ? 1 : 0);
  uint32_t total = a.off_inbox + (a.ks == 2 ? (nD > (per_a + 1) / 2 ? nD : (per_a + 1) / 2) * 64 * m : 0u);
  // Slots of X: as many as there are warps to read different pairs at a time, within 128 KB; a ring of up to four slots from what is
  // left, fewer slots of X where that would be less than two.  (A ring also takes half a blob of B per row tile.)
  const uint32_t b_need = ab ? 2u * ((uint32_t)tile_bytes(a.a_fmt) + 64u) : 0u;
  auto fit = [&](uint32_t slot_b, uint32_t need, uint32_t least, uint32_t& xslots, uint32_t& off_ring, uint32_t& slots, uint32_t& pitch) {
    xslots = most_x;
    if (xslots > a.pairs0) xslots = a.pairs0;
    for (;; --xslots) {
      off_ring = up(xslots * x_slot > least ? xslots * x_slot : least);
      const uint32_t room = ((uint32_t)kMaxSmem - off_ring) / kWarps;
      slots = room / slot_b;
      if ((slots >= 2 && room >= need) || xslots <= 2) break;
    }
    if (slots > (uint32_t)kMaxSlots) slots = kMaxSlots;
    pitch = slots * slot_b > need ? slots * slot_b : need;
    const uint32_t end = off_ring + kWarps * pitch;
    if (end > total) total = end;
    return slots >= 1;
  };
  if (!fit(2 * (uint32_t)h->w.blob, b_need, ab ? t_half : 0u, a.xslots, a.off_ring, a.slots, a.ring_pitch)) return false;
  if (ab && !fit(a.a_blob, 0u, 0u, a.a_xslots, a.a_off_ring, a.a_slots, a.a_pitch)) return false;
  a.t_chunk = a.off_ring / t_half;                 // t goes where X was
  pl.smem = (int)total;
  return total <= (uint32_t)kMaxSmem;
}

}  // namespace

// Above eight tokens (one decode pass is cheaper) and up to 32.  Three LLaMA3-8B blocks, 4-bit, fp16 adapters of rank 128, against
// the tcgen05 kernel: 12 tokens 196 against 412 us, 32 tokens 256 against 421.  Forms for 64 tokens lost: two launches 510
// against 431 us; one with twice the accumulators 464 (the sums of 64 tokens fill the registers, and only eight pairs of X fit).
bool mid_supported(const Handle* h, int m) {
  if (m <= 8 || m > kMaxTokens || h->sm_count < 4 || h->cfg.kernel_policy == EORA_POLICY_GENERIC) return false;
  if (h->w.fmt != FMT_Q4 && h->w.fmt != FMT_Q3 && h->w.fmt != FMT_SP24 && h->w.fmt != FMT_SQ4) return false;
  if (!encode_fn()) return false;
  Plan pl;
  return make_plan(h, m, pl);
}

int mid_grid(const Handle* h, int m) {
  Plan pl;
  return make_plan(h, m, pl) ? pl.grid : 0;
}

// x16: fp16 activations (device).
cudaError_t launch_mid_forward(const Handle* h, const void* x16, int m, void* const* ys, cudaStream_t st, const int32_t* adapter_ids) {
  Plan pl;
  MidArgs& a = pl.a;
  if (!make_plan(h, m, pl)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cfg.gridDim = dim3(pl.grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = pl.smem;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = a.ks; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  a.n_sub = h->n_sub;
  for (int k = 0; k < 5; ++k) a.sub_tile0[k] = (uint32_t)(k <= h->n_sub ? h->sub_tile0[k] : h->w.nt);
  for (int k = 0; k < h->n_sub; ++k) { a.sub_dout[k] = h->sub_dout[k]; a.ys[k] = ys[k]; }
  a.t_part = h->t_part; a.launches = h->launches; a.dev_status = h->dev_status;
  a.t_cols = h->t_cols; a.y_dtype = h->cfg.y_dtype; a.wait_ns = h->wait_limit_ns;
  if (h->multi) {
    a.adp_pairs = (uint32_t)h->r_pad / 128;
    for (int k = 0; k < m; ++k) {
      const int id = adapter_ids ? adapter_ids[k] : -1;
      a.adp[k] = (signed char)(id >= 0 && id < h->n_adapters ? id : -1);
    }
  }
  CUtensorMap tm;
  if (!make_map(&tm, x16, m, h->cfg.d_in, 8 * pl.nt)) return cudaErrorInvalidValue;
  return launch_any(cfg, tm, a, h->w.fmt, h->w.sz2 != 0, pl.nt, h->device);
}

}  // namespace eora
