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
// Work of a CTA.  Its row tiles go in pairs (32 rows share every activation fragment that is read from shared memory); kWarps / (pairs of
// row tiles) warps share one and cut the reduction axis among them, chunk by chunk.  A warp keeps its sums in registers
// from the first chunk to the last.  X comes by TMA in chunks of pairs, double-buffered, as [32 k][token][32 fp16]: the
// eight tokens x 64 bytes that a fragment load of a warp reads are 512 contiguous bytes.  The weights come
// through a ring per warp.  Weights are RN((q - z) * s) in fp16, as in prefill.cu, so scales need no accumulators of
// their own.
//
// Measured: four LLaMA3-8B blocks, 4-bit backbone and adapters, 16 tokens 544 -> 270 us (see also mid_supported).
#include <cuda.h>
#include "decode_common.cuh"

namespace eora {
namespace {
using namespace dec;

constexpr int kWarpLog = 4, kWarps = 1 << kWarpLog, kThreads = kWarps * 32;
constexpr int kMaxPass = 32;              // tokens per launch
constexpr int kSegPitch = 36;             // floats from one token's 32 row sums to the next (36: the four token pairs of a store hit different banks)
constexpr int kMaxSmem = 226 * 1024;
constexpr int kMaxSlots = 4;
constexpr uint32_t kBox = 4;              // pairs of X per copy

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
  uint32_t chunk, a_chunk;                // pairs of X per buffer (W, A)
  uint32_t slots, slot_pairs, ring_pitch; // ring of a warp (W): slots of slot_pairs pairs of two row tiles
  uint32_t a_slots, a_pitch;              // ring of a warp (A): slots of one blob
  uint32_t off_ring, off_inbox, off_bseg, off_t;      // shared memory, W (X buffers first; later the warps' sums over them)
  uint32_t a_off_ring, a_off_inbox;
  void* ys[4];
  uint32_t sub_tile0[5];                  // layer i owns row tiles [sub_tile0[i], sub_tile0[i + 1]) and pairs [i, i + 1) * sub_pairs of t
  int sub_dout[4];
  int n_sub;
  uint32_t sub_pairs, b_np, t_chunk, b_log;           // as in decode.cu
  uint32_t adp_pairs;                     // several adapters: pair p of t belongs to adapter p / adp_pairs (0: one adapter)
  signed char adp[kMaxPass];              // adapter of every token (-1: none)
  unsigned long long* t_part;             // [m][t_cols / 2] words (two columns as fp16, launch number)
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

// The wide operand of the tile's four mma: RN((q - z) * s) in fp16, or (SCALED false) the exact q - z.
template <int FMT, bool SCALED>
__device__ __forceinline__ void weights_f16(uint32_t tile, int lane, const SZ& z, uint32_t lut, uint32_t (&a)[4][4]) {
  RawTile<FMT> r;
  load_tile_s<FMT>(r, tile, lane);
  tile_frags<FMT>(r, z.zc, a, lut);
  if constexpr (SCALED && fmt_quantised(FMT)) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) a[i][e] = h2mul(a[i][e], z.s[e & 1]);
  }
}

// One pair of T row tiles (blobs `stride` apart) times the activations at x: [4 blocks of 32 k][8 NT tokens][32 fp16], x already at
// this lane's token and piece.  Up to 16 tokens the scale of a quantised group is applied to the group's sums (8 NT T multiplications
// a lane instead of 32 T on the weights); with more the sums would need as many registers again.
template <int FMT, bool SZ2, int NT, int T>
__device__ __forceinline__ void product(uint32_t blob, uint32_t stride, int lane, uint32_t x, uint32_t lut, float (&acc)[T][NT][4]) {
  constexpr int tb = tile_bytes(FMT);
  constexpr bool late = fmt_quantised(FMT) && NT <= 2;
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
    uint32_t a[T][4][4];
#pragma unroll
    for (int u = 0; u < T; ++u) {
      if constexpr (fmt_quantised(FMT)) { if (c == 0 || SZ2) load_sz<FMT>(z[u], blob + u * stride + 2 * tb + c * kSzEntryBytes, lane); }
      weights_f16<FMT, !late>(blob + u * stride + c * tb, lane, z[u], lut, a[u]);
    }
#pragma unroll
    for (int n = 0; n < NT; ++n) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const uint4 v = lds_u4(x + (2 * c + b) * (NT * 512) + n * 512);
#pragma unroll
        for (int u = 0; u < T; ++u) {
          float (&o)[4] = late ? d[late ? u : 0][late ? n : 0] : acc[u][n];
          mma16816(o, a[u][2 * b], v.x, v.y);
          mma16816(o, a[u][2 * b + 1], v.z, v.w);
        }
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

// A or B: the format is known at run time only (one uniform branch per blob).  x_step: bytes from one block of eight tokens to the
// next, k_step: from one block of 32 k to the next.
template <int FMT, bool SZ2, int NT>
__device__ __forceinline__ void product_ab1(uint32_t blob, int lane, uint32_t x, uint32_t x_step, uint32_t k_step, float (&acc)[NT][4]) {
  constexpr int tb = tile_bytes(FMT);
  SZ z;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if constexpr (fmt_quantised(FMT)) { if (c == 0 || SZ2) load_sz<FMT>(z, blob + 2 * tb + c * kSzEntryBytes, lane); }
    uint32_t a[4][4];
    weights_f16<FMT, true>(blob + c * tb, lane, z, 0u, a);
#pragma unroll
    for (int n = 0; n < NT; ++n) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const uint4 v = lds_u4(x + (2 * c + b) * k_step + n * x_step);
        mma16816(acc[n], a[2 * b], v.x, v.y);
        mma16816(acc[n], a[2 * b + 1], v.z, v.w);
      }
    }
  }
}
template <int NT>
__device__ __forceinline__ void product_ab(int fmt, uint32_t sz2, uint32_t blob, int lane, uint32_t x, uint32_t x_step, uint32_t k_step, float (&acc)[NT][4]) {
  switch (fmt) {
    case FMT_F16: product_ab1<FMT_F16, false, NT>(blob, lane, x, x_step, k_step, acc); break;
    case FMT_Q8: product_ab1<FMT_Q8, false, NT>(blob, lane, x, x_step, k_step, acc); break;
    case FMT_Q4: if (sz2) product_ab1<FMT_Q4, true, NT>(blob, lane, x, x_step, k_step, acc); else product_ab1<FMT_Q4, false, NT>(blob, lane, x, x_step, k_step, acc); break;
    case FMT_Q3: if (sz2) product_ab1<FMT_Q3, true, NT>(blob, lane, x, x_step, k_step, acc); else product_ab1<FMT_Q3, false, NT>(blob, lane, x, x_step, k_step, acc); break;
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
struct Span { uint32_t a, b, base; };              // pairs of t that row tile `tile` takes part in, within [c0, c1)
__device__ __forceinline__ Span t_span(const MidArgs& p, uint32_t tile, uint32_t c0, uint32_t c1) {
  Span s;
  s.base = p.sub_pairs ? (uint32_t)sub_of(p, tile) * p.sub_pairs : 0u;
  s.a = max(c0, s.base); s.b = min(c1, s.base + p.b_np);
  return s;
}

// The chunks of a CTA's part of the reduction axis (P pairs, chunk of them per buffer) and a warp's share of each: of a chunk's n
// pairs warp j of wpt takes [j n / wpt, (j + 1) n / wpt).
struct Walk {
  uint32_t P, chunk, j, wpt_inv;
  uint32_t c, q, end;                     // chunk's first pair; next pair of the share, its end (counted from c)
};
__device__ __forceinline__ void walk_open(Walk& w, uint32_t c) {
  w.c = c;
  const uint32_t n = min(w.chunk, w.P - c), lo = w.j * n, hi = lo + n;
  w.q = w.wpt_inv ? __umulhi(lo, w.wpt_inv) : lo;
  w.end = w.wpt_inv ? __umulhi(hi, w.wpt_inv) : hi;
}
__device__ __forceinline__ bool walk_next_chunk(Walk& w) {          // to the next chunk with something in it
  while (w.q == w.end) {
    if (w.c + w.chunk >= w.P) return false;
    walk_open(w, w.c + w.chunk);
  }
  return true;
}

template <int WF, bool SZ2, int NT>
__global__ void __launch_bounds__(kThreads, 1) k_mid(const __grid_constant__ CUtensorMap tm, const __grid_constant__ MidArgs p) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint32_t lut_s[16];
  __shared__ __align__(8) uint64_t bars_s[2 + kWarps * kMaxSlots];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  asm volatile("griddepcontrol.launch_dependents;");
  const bool is_a = blockIdx.x < p.n_a;
  const uint32_t cta = is_a ? blockIdx.x : blockIdx.x - p.n_a;
  const uint32_t cl = p.ks == 2 ? cta >> 1 : cta, rank = p.ks == 2 ? cta & 1 : 0;
  if (p.ks == 2) cluster_arrive();                 // (that the partner runs at all, before anything is written to it)
  if constexpr (WF == FMT_SP24 || WF == FMT_SQ4) { if (threadIdx.x < 16) lut_s[threadIdx.x] = sp24_selectors(threadIdx.x); }
  const uint32_t lut = smem_u32(lut_s), xbar = smem_u32(bars_s), bars = xbar + 16 + warp * (kMaxSlots * 8);
  if (threadIdx.x == 0) { mbar_init_a(xbar, 1); mbar_init_a(xbar + 8, 1); }
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kMaxSlots; ++i) mbar_init_a(bars + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncwarp();

  // this CTA's units (row tiles of A, or pairs of row tiles of W) and this warp's place: unit d, share j of wpt
  const uint32_t d0 = share_lo(is_a ? p.a_tiles : p.w_dbl, cl), nD = share_n(is_a ? p.a_tiles : p.w_dbl, cl);
  const uint32_t wpt = kWarps / nD, d = warp / wpt, j = warp - d * wpt;
  const bool active = d < nD;
  const uint32_t P = rank ? p.np - p.pairs0 : p.pairs0, pr0 = rank ? p.pairs0 : 0u, chunk = is_a ? p.a_chunk : p.chunk;
  const uint32_t xbuf = smem_u32(smem), xbuf_b = (chunk + kBox - 1) / kBox * (kBox * NT * 2048);
  Walk in = {P, chunk, j, wpt > 1 ? 0xffffffffu / wpt + 1u : 0u, 0, 0, 0}, out;
  walk_open(in, 0);
  if (!active) { in.q = in.end = 0; in.c = P; }
  out = in;

  Ring ring;
  const uint32_t blob_b = is_a ? p.a_blob : (uint32_t)blob_bytes(WF, SZ2 ? 1 : 0);
  const uint32_t slot_n = is_a ? 1u : p.slot_pairs, slot_b = is_a ? p.a_blob : 2 * slot_n * blob_b, slots = is_a ? p.a_slots : p.slots;
  ring.base = smem_u32(smem + (is_a ? p.a_off_ring : p.off_ring)) + warp * (is_a ? p.a_pitch : p.ring_pitch);
  ring.bytes = slots * slot_b; ring.bars = ring.bar = bars; ring.so = 0; ring.parity = 0;
  // first blob of the unit's first row tile in this half of the reduction axis, and from there to its second row tile
  const uint8_t* w0 = is_a ? p.a_q + ((size_t)(d0 + d) * p.np + pr0) * blob_b
                           : p.w_q + ((size_t)rank * p.w_nt * p.pairs0 + (size_t)(d0 + d) * 2 * P) * blob_b;
  const size_t to_second = (size_t)P * blob_b;
  auto ask = [&](uint32_t so, uint32_t bar) {      // the next copy of the warp's share
    if (!walk_next_chunk(in)) return;
    const uint32_t cnt = min(slot_n, in.end - in.q);
    if (lane == 0) {
      const uint8_t* src = w0 + (size_t)(in.c + in.q) * blob_b;
      mbar_expect_tx_a(bar, (is_a ? 1u : 2u) * cnt * blob_b);
      bulk_g2s_a(ring.base + so, src, cnt * blob_b, bar);
      if (!is_a) bulk_g2s_a(ring.base + so + slot_n * blob_b, src + to_second, cnt * blob_b, bar);
    }
    in.q += cnt;
  };
  for (uint32_t i = 0, so = 0, b = bars; i < slots; ++i, so += slot_b, b += 8) ask(so, b);
  const uint32_t f0 = is_a ? 0u : (rank ? nD : 0u), nT = is_a ? nD : 2 * nD;      // W: rank 0 finishes the first nD row tiles, rank 1 the others
  const uint32_t a_f0 = rank ? nD >> 1 : 0u, a_f1 = p.ks == 2 && rank == 0 ? nD >> 1 : nD;
  const uint32_t first = is_a ? a_f0 : (p.ks == 2 ? f0 : 0u), nf = is_a ? a_f1 - a_f0 : (p.ks == 2 ? nD : nT);
  if (!is_a && p.n_a) {                            // blobs of B towards L2
    const uint32_t per = p.b_np * (uint32_t)blob_bytes(p.a_fmt, (int)p.b_sz2), bytes = nf * per;
    const uint8_t* b_part = p.b_q + (size_t)(2 * d0 + first) * per;
    for (uint32_t o = threadIdx.x << 14; o < bytes; o += kThreads << 14) prefetch_l2(b_part + o, min(16384u, bytes - o));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();                                 // the X barriers are set up
  const uint32_t launch = launch_number(p.launches);
  auto load_x = [&](uint32_t c) {                  // chunk c / chunk of X: one warp per copy, the first of them says how much comes
    const uint32_t i = (c / chunk) & 1, b = xbar + 8 * i;
    if (threadIdx.x == 0) mbar_expect_tx_a(b, xbuf_b);
    for (uint32_t k = warp * kBox; k < chunk && lane == 0; k += kWarps * kBox) tma_load_3d(xbuf + i * xbuf_b + k * (NT * 2048), &tm, 0, 0, (int)((pr0 + c + k) * 4), b);
  };
  load_x(0);
  if (chunk < P) load_x(chunk);

  constexpr int T = 2;
  float acc[T][NT][4];
#pragma unroll
  for (int u = 0; u < T; ++u)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[u][n][i] = 0.f;
  bool ok = true;
  uint32_t xpar = 0;                               // bit i: phase that buffer i completes next
#pragma unroll 1
  for (uint32_t c = 0, xi = 0; c < P; c += chunk, xi ^= 1) {
    if (ok && !mbar_try_wait_a(xbar + 8 * xi, (xpar >> xi) & 1) && !mbar_wait_lane(xbar + 8 * xi, (xpar >> xi) & 1, p.dev_status)) ok = false;
    xpar ^= 1u << xi;
    if (c > 0 && active) walk_open(out, c);
    const uint32_t xl = xbuf + xi * xbuf_b + (lane >> 2) * 64 + (lane & 3) * 16;
#pragma unroll 1
    while (out.q < out.end) {
      uint32_t cnt = min(slot_n, out.end - out.q);
      if (ok && !mbar_try_wait_a(ring.bar, ring.parity) && !mbar_wait_lane(ring.bar, ring.parity, p.dev_status)) ok = false;
      __syncwarp();
      uint32_t src = ring.base + ring.so, x = xl + out.q * (NT * 2048);
      out.q += cnt;
#pragma unroll 1
      for (; cnt > 0; --cnt, src += blob_b, x += NT * 2048) {
        if (is_a) product_ab<NT>(p.a_fmt, p.a_sz2, src, lane, x, 512u, NT * 512u, acc[0]);
        else product<WF, SZ2, NT, T>(src, slot_n * blob_b, lane, x, lut, acc);
      }
      __syncwarp();                                // every lane is done with the slot
      if (ok) ask(ring.so, ring.bar);
      ring_next(ring, slot_b);
    }
    if (c + chunk < P) {
      __syncthreads();                             // every warp is done with the buffer
      if (c + 2 * chunk < P) load_x(c + 2 * chunk);
    }
  }
  if (!__all_sync(0xffffffffu, ok)) {              // gave up: what is in flight must land first
    for (uint32_t i = 0; i < slots; ++i) mbar_drain_warp(bars_s + 2 + warp * kMaxSlots + i, ring.bars + 8 * i < ring.bar ? ring.parity ^ 1u : ring.parity, lane);
    for (int i = 0; i < 2; ++i) mbar_drain_warp(bars_s + i, (xpar >> i) & 1, lane);
  }

  // ---- the CTA's sums: every warp's into a slot of its own (over the X buffers), then added up per element
  const bool ab = p.n_a != 0;
  auto ask_b = [&](uint32_t tile, uint32_t pair, uint32_t b_blob) {                 // a blob of B to the start of the (empty) ring
    if (lane == 0) {
      mbar_expect_tx_a(ring.bar, b_blob);
      bulk_g2s_a(ring.base, p.b_q + ((size_t)tile * p.b_np + pair) * b_blob, b_blob, ring.bar);
    }
  };
  const uint32_t first_tile = 2 * d0 + first, b_blob = (uint32_t)blob_bytes(p.a_fmt, (int)p.b_sz2);
  uint32_t c0 = 0, c_end = p.b_np;                 // chunk of t, end of all chunks
  TWords tw = {0ull, 0ull};
  // step e of a chunk of t: four columns of one token (32 steps per pair and token)
  auto t_tok = [&](uint32_t e) { return (e >> 5) & ((1u << p.m_log) - 1); };
  auto t_col = [&](uint32_t e) { return (e >> (5 + p.m_log)) * 128 + (e & 31) * 4; };
  if (!is_a && ab) {
    if (p.sub_pairs) { c0 = (uint32_t)sub_of(p, first_tile) * p.sub_pairs; c_end = (uint32_t)(sub_of(p, first_tile + nf - 1) + 1) * p.sub_pairs; }
    if (warp < (int)(nf << p.b_log)) {
      const uint32_t tile = first_tile + (warp >> p.b_log);
      const Span s = t_span(p, tile, c0, c0 + p.t_chunk);
      const uint32_t q = s.a + (warp & ((1u << p.b_log) - 1));
      if (q < s.b) ask_b(tile, q - s.base, b_blob);
    }
    if (t_tok(threadIdx.x) < (uint32_t)p.m && c0 * 128 + t_col(threadIdx.x) < (uint32_t)p.t_cols)
      load_t(tw, p.t_part + ((size_t)t_tok(threadIdx.x) * p.t_cols + c0 * 128 + t_col(threadIdx.x)) / 2);
  }
  __syncthreads();                                 // every warp is done with X
  float* const seg = reinterpret_cast<float*>(smem);
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
  const uint32_t hw = threadIdx.x >> 4, row = threadIdx.x & 15, m = p.m, OT = 16 * m, m_mask = (1u << p.m_log) - 1;
  float* const inbox = reinterpret_cast<float*>(smem + (is_a ? p.a_off_inbox : p.off_inbox));
  // four tokens of a row tile at once (independent loads: in a rolled loop each costs its latency), summed over the warps that share it
  auto tile_sum = [&](uint32_t f, uint32_t tok, float (&v)[4]) {
    const float* s = is_a ? seg + f * wpt * kSlot + tok * kSegPitch + row : seg + (f >> 1) * wpt * kSlot + tok * kSegPitch + (f & 1) * 16 + row;
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
    cluster_wait();
    const uint32_t s0 = rank ? 0u : first + nf, ns = nT - nf;
    const uint32_t to = mapa(smem_u32(inbox), rank ^ 1u) + row * 4;
    for (uint32_t u = hw; u < ns << q_log; u += 2 * kWarps) {
      const uint32_t f = u >> q_log, tok = (u & q_mask) * 4;
      float v[4];
      tile_sum(s0 + f, tok, v);
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i)
        if (tok + i < m) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to + (f * OT + (tok + i) * 16) * 4), "f"(v[i]) : "memory");
    }
    cluster_arrive();
  }
  float* const bseg = reinterpret_cast<float*>(smem + p.off_bseg);
  if (!is_a && ab) {
    const uint32_t pitch = p.t_chunk * 256 + 64, th = smem_u32(smem + p.off_t);
    uint32_t parity = ring.parity;
    bool fresh = true;
#pragma unroll 1
    for (;;) {
      // t of this chunk as fp16, zero for tokens that do not use the pair's adapter and in the columns past A's rows (padding)
      const uint32_t steps = min(p.t_chunk, c_end - c0) << (5 + p.m_log);
      for (uint32_t e = threadIdx.x; e < steps; e += kThreads) {
        const uint32_t tok = t_tok(e), col = t_col(e);
        if (tok >= m) continue;
        uint2 v = make_uint2(0u, 0u);
        if (c0 * 128 + col < p.a_nt * 16 && !(p.adp_pairs && p.adp[tok] != (int)((c0 + (col >> 7)) / p.adp_pairs))) {
          const unsigned long long* src = p.t_part + ((size_t)tok * p.t_cols + c0 * 128 + col) / 2;
          if (!fresh || e != threadIdx.x) load_t(tw, src);
          if (wait_t(tw, src, launch, p.wait_ns, p.dev_status)) v = make_uint2((uint32_t)tw.a, (uint32_t)tw.b);
        }
        sts_u1(th + tok * pitch + col * 2, v.x);
        sts_u1(th + tok * pitch + col * 2 + 4, v.y);
      }
      __syncthreads();
#pragma unroll 1
      for (uint32_t u = warp; u < nf << p.b_log; u += kWarps) {
        const uint32_t tile = first_tile + (u >> p.b_log);
        const Span s = t_span(p, tile, c0, c0 + p.t_chunk);
        float bacc[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) bacc[n][i] = 0.f;
#pragma unroll 1
        for (uint32_t q = s.a + (u & ((1u << p.b_log) - 1)), k = 0; q < s.b; q += 1u << p.b_log, ++k) {
          if (!fresh || u != (uint32_t)warp || k) ask_b(tile, q - s.base, b_blob);
          if (!mbar_try_wait_a(ring.bar, parity)) mbar_wait_lane(ring.bar, parity, p.dev_status);
          parity ^= 1u;
          __syncwarp();
          product_ab<NT>(p.a_fmt, p.b_sz2, ring.base, lane, th + (lane >> 2) * pitch + (lane & 3) * 16 + (q - c0) * 256, 8 * pitch, 64u, bacc);
          __syncwarp();
        }
        float* b = bseg + u * OT + (lane >> 2) + (lane & 3) * 32;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint32_t tok = n * 8 + 2 * (lane & 3);
          if (tok < m) { b[n * 128] = bacc[n][0]; b[n * 128 + 8] = bacc[n][2]; }
          if (tok + 1 < m) { b[n * 128 + 16] = bacc[n][1]; b[n * 128 + 24] = bacc[n][3]; }
        }
      }
      c0 += p.t_chunk;
      if (c0 >= c_end) break;
      fresh = false;
      __syncthreads();
      for (uint32_t u = hw; u < nf << p.m_log; u += 2 * kWarps) {      // this chunk's products join the first warp's sums of the row tile
        const uint32_t f = u >> p.m_log, tok = u & m_mask;
        if (tok >= m) continue;
        float v = 0.f;
        for (uint32_t k = 0; k < 1u << p.b_log; ++k) v += bseg[((f << p.b_log) + k) * OT + tok * 16 + row];
        seg[((first + f) >> 1) * wpt * kSlot + tok * kSegPitch + ((first + f) & 1) * 16 + row] += v;
      }
    }
  }
  if (p.ks == 2) cluster_wait();
  __syncthreads();
  // (m_log >= 4: nf << q_log is even, so the halves of a warp take part alike)
  for (uint32_t u = hw; u < nf << q_log; u += 2 * kWarps) {
    const uint32_t f = u >> q_log, tok = (u & q_mask) * 4;
    float v[4];
    tile_sum(first + f, tok, v);
    if (p.ks == 2) {
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) v[i] += inbox[f * OT + (tok + i < m ? tok + i : tok) * 16 + row];
    }
    if (is_a) {                                    // two columns of t per word
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        const float o = __shfl_down_sync(0xffffffffu, v[i], 1);
        if (tok + i < m && !(row & 1)) {
          const unsigned long long word = ((unsigned long long)launch << 32) | pack_h2(v[i], o);
          asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p.t_part + ((size_t)(tok + i) * p.t_cols + (d0 + first + f) * 16 + row) / 2), "l"(word) : "memory");
        }
      }
    } else {
      if (ab) {
        for (uint32_t k = 0; k < 1u << p.b_log; ++k)
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i) v[i] += bseg[((f << p.b_log) + k) * OT + (tok + i < m ? tok + i : tok) * 16 + row];
      }
      const uint32_t tg = first_tile + f;
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

// X [m][d_in] fp16 as (k within a block of 32, token, block of 32 k); the box brings `blocks` blocks of all tokens (zeros past m)
bool make_map(CUtensorMap* tm, const void* x, int m, int d_in, int tokens, int blocks) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {32, (cuuint64_t)m, (cuuint64_t)d_in / 32};
  cuuint64_t strides[2] = {(cuuint64_t)d_in * 2, 64};
  cuuint32_t box[3] = {32, (cuuint32_t)tokens, (cuuint32_t)blocks};
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
  return nt == 2 ? launch_kernel<k_mid<WF, SZ2, 2>>(cfg, tm, a, device) : launch_kernel<k_mid<WF, SZ2, 4>>(cfg, tm, a, device);
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
  const int NT = m <= 16 ? 2 : 4, Mr = 8 * NT;
  pl.nt = NT;
  a.m = m;
  while ((1 << a.m_log) < m) ++a.m_log;
  a.w_q = h->w.q; a.w_nt = h->w.nt; a.np = h->w.np; a.pairs0 = h->w.half;
  a.ks = h->w.np >= 2 ? 2 : 1;
  const uint32_t sms = (uint32_t)h->sm_count / a.ks * a.ks, cls = sms / a.ks, nd = h->w.nt / 2;
  a.chunk = NT == 2 ? 16 : 8;                      // 64 KB of X per buffer (one buffer if that is all)
  if (a.chunk > a.pairs0) a.chunk = a.pairs0;
  if (ab) {
    a.a_fmt = h->a.fmt; a.a_q = h->a.q; a.a_nt = h->a.nt; a.a_sz2 = h->a.sz2; a.a_blob = h->a.blob;
    a.b_q = h->b.q; a.b_np = h->b.np; a.b_sz2 = h->b.sz2;
    // Clusters for A: t should be there when the products with W are done (an exchange through L2 takes about as long as 24
    // blobs of a CTA's).
    double best = 1e30;
    uint32_t best_n = 1;
    for (uint32_t n = 1; n <= cls / 2 && n <= (uint32_t)h->a.nt; ++n) {
      const uint32_t per_a = (h->a.nt + n - 1) / n, per_w = (nd + cls - n - 1) / (cls - n);
      if (per_a > (uint32_t)kWarps) continue;
      const double ta = 24.0 + (double)per_a * a.pairs0 * 1.2, tw = 2.0 * per_w * a.pairs0, t = ta > tw ? ta : tw;
      if (t < 0.99 * best) { best = t; best_n = n; }
    }
    if ((h->a.nt + best_n - 1) / best_n > (uint32_t)kWarps) best_n = (h->a.nt + kWarps - 1) / kWarps;
    a.n_a = best_n * a.ks;
    a.a_tiles = make_share(h->a.nt, best_n);
    a.sub_pairs = h->n_sub > 1 ? (uint32_t)h->r_pad / 128 : 0u;
  }
  uint32_t ncl = cls > a.n_a / a.ks ? cls - a.n_a / a.ks : 1;
  if (ncl > nd) ncl = nd;
  if ((nd + ncl - 1) / ncl > (uint32_t)kWarps) ncl = (nd + kWarps - 1) / kWarps;      // more than fit at once: in waves
  a.w_dbl = make_share(nd, ncl);
  pl.grid = (int)(a.n_a + ncl * a.ks);
  if (pl.grid >= (1 << kLaunchShift)) return false;
  const uint32_t nD = a.w_dbl.per + (a.w_dbl.rem ? 1 : 0), nF = a.ks == 2 ? nD : 2 * nD;
  const uint32_t t_pairs = (uint32_t)h->t_cols / 128;
  a.t_chunk = NT == 2 ? 4 : 2;
  if (a.t_chunk > t_pairs) a.t_chunk = t_pairs;
  while ((2u << a.b_log) * nF <= (uint32_t)kWarps && (1u << a.b_log) < a.t_chunk && (1u << a.b_log) < a.b_np) ++a.b_log;
  auto up = [](uint32_t v) { return (v + 127u) & ~127u; };
  const uint32_t seg_b = up(kWarps * Mr * kSegPitch * 4);
  const uint32_t bseg_b = ab ? up((nF > (uint32_t)kWarps ? nF : (uint32_t)kWarps) * 64 * m) : 0u, t_b = ab ? up(Mr * (a.t_chunk * 256 + 64)) : 0u;
  a.off_bseg = seg_b; a.off_t = seg_b + bseg_b;
  const uint32_t late = seg_b + bseg_b + t_b, inbox_b = a.ks == 2 ? up(nD * 64 * m) : 0u;
  // ring: what is left, in up to four slots of one or two pairs of two row tiles; it also takes a blob of B.  Smaller chunks of X
  // where that leaves less than two slots.
  const uint32_t pair_b = 2 * (uint32_t)h->w.blob, b_blob = ab ? (uint32_t)h->b.blob : 0u;
  uint32_t room = 0;
  for (;; a.chunk = (a.chunk + 1) / 2) {
    const uint32_t x_b = (a.chunk < a.pairs0 ? 2 : 1) * ((a.chunk + kBox - 1) / kBox) * (kBox * NT * 2048);
    a.off_inbox = x_b > late ? x_b : late;
    a.off_ring = a.off_inbox + inbox_b;
    room = a.off_ring < (uint32_t)kMaxSmem ? ((uint32_t)kMaxSmem - a.off_ring) / kWarps / pair_b : 0u;
    if (room >= 2 || a.chunk <= 2 || x_b <= late) break;
  }
  if (room < 1) return false;
  a.slot_pairs = room >= 4 ? 2 : 1;
  a.slots = room / a.slot_pairs < (uint32_t)kMaxSlots ? room / a.slot_pairs : kMaxSlots;
  a.ring_pitch = a.slots * a.slot_pairs * pair_b;
  if (a.ring_pitch < b_blob) a.ring_pitch = b_blob;
  uint32_t total = a.off_ring + kWarps * a.ring_pitch;
  if (ab) {
    const uint32_t per_a = a.a_tiles.per + (a.a_tiles.rem ? 1 : 0);
    // A's clusters have few row tiles, so their warps cut the reduction axis finely: as much of X at once as leaves a blob per warp
    uint32_t a_room = 0;
    for (a.a_chunk = a.pairs0 < 32 ? a.pairs0 : 32;; a.a_chunk = (a.a_chunk + 1) / 2) {
      const uint32_t bufs = a.a_chunk < a.pairs0 ? 2 : 1, ax = bufs * ((a.a_chunk + kBox - 1) / kBox) * (kBox * NT * 2048);
      a.a_off_inbox = ax > seg_b ? ax : seg_b;
      a.a_off_ring = a.a_off_inbox + (a.ks == 2 ? up(((per_a + 1) / 2) * 64 * m) : 0u);
      a_room = a.a_off_ring < (uint32_t)kMaxSmem ? ((uint32_t)kMaxSmem - a.a_off_ring) / kWarps / a.a_blob : 0u;
      if (a_room >= 2 || a.a_chunk <= 8) break;
    }
    if (a_room < 1) return false;
    a.a_slots = a_room < (uint32_t)kMaxSlots ? a_room : kMaxSlots;
    a.a_pitch = a.a_slots * a.a_blob;
    if (a.a_off_ring + kWarps * a.a_pitch > total) total = a.a_off_ring + kWarps * a.a_pitch;
  }
  pl.smem = (int)total;
  return total <= (uint32_t)kMaxSmem;
}

}  // namespace

// Above eight tokens (one decode pass is cheaper) and up to what one launch takes.  Three LLaMA3-8B blocks, 4-bit, fp16 adapters of
// rank 128, against the tcgen05 kernel: 12 tokens 204 against 412 us, 32 tokens 293 against 421; 64 tokens in two launches
// would be 567 against 431.
bool mid_supported(const Handle* h, int m) {
  if (m <= 8 || m > kMaxPass || h->sm_count < 4 || h->cfg.kernel_policy == EORA_POLICY_GENERIC) return false;
  if (h->w.fmt != FMT_Q4 && h->w.fmt != FMT_Q3 && h->w.fmt != FMT_SP24 && h->w.fmt != FMT_SQ4) return false;
  if (!encode_fn()) return false;
  Plan pl;
  return make_plan(h, m < kMaxPass ? m : kMaxPass, pl);
}

int mid_launch_count(const Handle*, int m) { return (m + kMaxPass - 1) / kMaxPass; }

// x16: fp16 activations (device).
cudaError_t launch_mid_forward(const Handle* h, const void* x16, int m, void* const* ys, cudaStream_t st, const int32_t* adapter_ids) {
  Plan pl;
  MidArgs& a = pl.a;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cfg.blockDim = dim3(kThreads);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const size_t ybytes = h->cfg.y_dtype == EORA_Y_F32 ? 4 : 2;
  const int passes = mid_launch_count(h, m);
  for (int i = 0, m0 = 0; i < passes; ++i) {
    const int mp = (m - m0 + passes - i - 1) / (passes - i);      // even passes
    if (!make_plan(h, mp, pl)) return cudaErrorInvalidValue;
    a.n_sub = h->n_sub;
    for (int k = 0; k < 5; ++k) a.sub_tile0[k] = (uint32_t)(k <= h->n_sub ? h->sub_tile0[k] : h->w.nt);
    for (int k = 0; k < h->n_sub; ++k) {
      a.sub_dout[k] = h->sub_dout[k];
      a.ys[k] = reinterpret_cast<uint8_t*>(ys[k]) + (size_t)m0 * h->sub_dout[k] * ybytes;
    }
    a.t_part = h->t_part; a.launches = h->launches; a.dev_status = h->dev_status;
    a.t_cols = h->t_cols; a.y_dtype = h->cfg.y_dtype; a.wait_ns = h->wait_limit_ns;
    if (h->multi) {
      a.adp_pairs = (uint32_t)h->r_pad / 128;
      for (int k = 0; k < mp; ++k) {
        const int id = adapter_ids ? adapter_ids[m0 + k] : -1;
        a.adp[k] = (signed char)(id >= 0 && id < h->n_adapters ? id : -1);
      }
    }
    CUtensorMap tm;
    if (!make_map(&tm, reinterpret_cast<const uint8_t*>(x16) + (size_t)m0 * h->cfg.d_in * 2, mp, h->cfg.d_in, 8 * pl.nt, 4 * kBox)) return cudaErrorInvalidValue;
    cfg.gridDim = dim3(pl.grid);
    cfg.dynamicSmemBytes = pl.smem;
    attr[1].val.clusterDim.x = a.ks;
    cudaError_t e = launch_any(cfg, tm, a, h->w.fmt, h->w.sz2 != 0, pl.nt, h->device);
    if (e != cudaSuccess) return e;
    m0 += mp;
  }
  return cudaSuccess;
}

}  // namespace eora
