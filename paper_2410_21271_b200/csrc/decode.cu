// Decode path (m <= 8 tokens per launch): one kernel computes Eq. 4 for a whole layer,
//     Y = X . deq(Wq) + (X . A) . B,
// streaming every weight byte exactly once.
//
// What bounds it.  A decode launch moves 3 - 50 MB, 0.5 - 7 us at the HBM's rate, and is one of a chain of dependent
// launches; most of its time is latency, not bandwidth: instructions at 6 to 10 cycles each in the parts that run once per
// CTA, an L2 round trip for the activations and one for t, and the products themselves (about 100 instructions per blob).
// So the kernel is built around the chain
//     previous launch ends -> activations arrive -> products -> sums -> Y
// and keeps everything that is not in it out of the way:
//   * A CTA owns whole row tiles of the output over half of the reduction axis, its cluster partner the other half.  The
//     sums of a row tile meet in the shared memory of the two CTAs; nothing goes through atomics or tickets in global
//     memory (a release, a ticket and a read-back cost 1.8 us of a 2.8 us launch measured on their own).
//   * A's rows belong to CTAs of their own ([0, n_a), dispatched first), which send t = X . A to everybody as 8-byte
//     words of (value, launch number): a reader that sees the number has the value, so the exchange is one store and
//     one polling load, no fence, counter or reset.  Only t is waited for, and only by CTAs that come later in the
//     grid than the ones they wait for, which themselves never wait.  The wait is bounded.
//   * One token: eight warps of 128 registers and half of an SM's shared memory, so that the next launch's CTAs are
//     resident and have their first weights in their rings while this one runs (programmatic dependent launch), and four
//     blobs at once per warp.  More tokens: sixteen warps and a whole SM, for the rings beside their activations and
//     sums.  (The issue slots are not what asks for it: 1.35 of 4 are used at eight tokens, and the first stall is a missing instruction.)
//     Asking for all of the next launch's weights ahead (bulk prefetches into L2) was slower, 183 against 172 us for four
//     blocks: the activations and t, which the launch in front is waiting for, then queue behind that traffic.
// Measured, four LLaMA3-8B blocks of four launches, fp16 adapters of rank 128: 3-bit, one token 194 -> 173 us; eight tokens
// 303 -> 259 us; two blocks of a 2:4 backbone, one token 143 -> 132 us (the figures before: warps that added their
// partial sums of single blobs to global memory and counted tickets).
//
// Work of a CTA.  Its blobs (16 rows x 128 reduction elements, see eora_common.cuh) in the order (chunk of the reduction
// axis, row tile, pair) are cut into equal runs, one per warp.  The activations of a chunk sit in shared memory
// in the form the products read: for one token and a 3/4-bit backbone as the byte planes of a 16-bit block fixed point
// number (integer tensor-core product, decode_common.cuh), else as fp16.  A warp keeps the sums of a row tile in
// registers and leaves them in a slot of its own when its run goes on to the next tile.
#include <type_traits>
#include "decode_common.cuh"

namespace eora {
namespace {
using namespace dec;

// Warps per CTA (log2), by the kind of product.
__host__ __device__ constexpr int warp_log(int mode) { return mode == 1 ? 3 : 4; }
constexpr int kMaxTok = 8;                // tokens per launch (the n8 side of the mma)
constexpr int kMaxSlices = 4;             // parts of the reduction axis that t may be sent in
constexpr int kMaxTiles = 48;             // row tiles per cluster (what its shared memory is sized for); more: further CTAs, in waves
constexpr int kMaxSmem = 226 * 1024;
constexpr int kHalfSmem = 112 * 1024;     // what two CTAs of an SM may use each
constexpr int kMaxSlots = 4;
constexpr uint32_t kRingLeast = 48 * 1024;      // bytes of weights in flight per CTA that keep HBM busy (148 x 48 KB = 7 MB, a microsecond's worth)
constexpr int kPlaneBytes = 272;          // integer path: two byte planes of a pair (256 B), scale and two sums

struct DecodeArgs {
  const uint8_t* a_q; const uint8_t* w_q; const uint8_t* b_q;
  int a_fmt;                              // format of A and B (FMT_NONE: no adapter)
  uint32_t a_sz2, b_sz2;
  uint32_t a_nt, a_np;                    // A: row tiles, pairs
  uint32_t n_a, a_slices, a_slice_pairs;  // CTAs that hold A; parts of its reduction axis, pairs per part
  uint32_t ks;                            // CTAs per cluster = parts of W's reduction axis (1 or 2)
  uint32_t w_nt, w_np, pairs;             // W: row tiles, pairs; pairs per part (of the first)
  uint32_t chunk;                         // pairs whose activations are in shared memory at a time
  Share tiles;                            // row tiles of W dealt to the clusters
  // Of each part: its pairs, and for CTAs with tiles.per / tiles.per + 1 row tiles ceil(2^32 / blobs) (whole runs) -- reciprocals
  // for the places where a CTA would divide.
  struct Part { uint32_t pairs, inv_pairs, inv_blobs[2]; } part[2];
  uint32_t b_np;                          // pairs of B per row tile
  uint32_t t_chunk;                       // pairs of t in shared memory at a time
  uint32_t b_log;                         // log2 of the warps that share a row tile's pairs of a chunk
  uint32_t slots, slot_blobs, ring_pitch; // a warp's ring of weights: slots of whole blobs; bytes from one warp's ring to the next
  uint32_t off_bar, off_ring, off_seg, off_inbox, off_sum, off_bseg, off_t;   // shared memory (bytes from the start): see the kernel
  const void* x;
  void* ys[4];                            // outputs of the fused layers (one for a plain layer)
  uint32_t sub_tile0[5];                  // layer i owns row tiles [sub_tile0[i], sub_tile0[i + 1]) and pairs [i, i + 1) * sub_pairs of t
  int sub_dout[4];
  int n_sub;
  uint32_t sub_pairs;                     // 0: every row tile takes part in all pairs of t (plain layer, several adapters)
  // Several adapters on one backbone: pair p of t belongs to adapter p / adp_pairs, and token i uses adapter
  // adp[i] (-1: none).  adp_pairs == 0: one adapter for all tokens.
  uint32_t adp_pairs;
  int adp[kMaxTok];
  unsigned long long* t_part;             // [slices][m][t_cols] words (value, launch number)
  unsigned long long* launches;           // launch counter
  int* dev_status;
  int m, m_log;                           // tokens; log2 of the next power of two
  int d_in, t_cols, x_dtype, y_dtype;
  unsigned long long wait_ns;             // limit of the wait for t
  unsigned long long* trace;
};

// Reads a word of every 64 bytes of the arguments.  They are new with every launch, and the first read of a line of them goes to
// L2; done here, that happens while the launch in front still runs instead of piece by piece in the middle of the kernel.
__device__ __forceinline__ void touch_args(const DecodeArgs& p) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(&p);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(DecodeArgs) / 4); i += 16) asm volatile("" ::"r"(w[i]));
  asm volatile("" ::"r"(w[sizeof(DecodeArgs) / 4 - 1]));
}

// ---- activations -> shared memory ------------------------------------------------------------------------------
// Sixteen lanes take the 128 activations of one (pair, token), eight consecutive ones each.

// Integer path (one token): pair q of the chunk at xs + q * kPlaneBytes: [half h of the MMAs][plane][t][16 bytes = MMAs 2h, 2h + 1],
// i.e. lane (g < 2, t) of the product reads its narrow-operand registers of MMAs 2h and 2h + 1 with one 16-byte load; then
// the block scale and the sums of the two 64-element tiles.  A warp takes a pair, four consecutive activations a lane.
template <int FMT, int kWarps>
__device__ __forceinline__ void stage_x_i8(uint32_t xs, const void* x, bool bf16, uint32_t pair0, uint32_t n, int warp, int lane) {
  constexpr int B = 4;                             // loads in flight: each is a round trip to a busy L2
  for (uint32_t q0 = warp; q0 < n; q0 += B * kWarps) {
  uint2 raw[B];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    raw[b] = make_uint2(0u, 0u);
    if (q0 + b * kWarps < n)
      asm volatile("ld.global.cg.v2.u32 {%0,%1}, [%2];" : "=r"(raw[b].x), "=r"(raw[b].y)
                   : "l"(reinterpret_cast<const uint16_t*>(x) + (size_t)(pair0 + q0 + b * kWarps) * 128 + 4 * lane) : "memory");
  }
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const uint32_t q = q0 + b * kWarps;
    if (q >= n) break;
    const uint2 u = raw[b];
    float f[4];
    if (bf16) {
      f[0] = __uint_as_float(u.x << 16); f[1] = __uint_as_float(u.x & 0xffff0000u);
      f[2] = __uint_as_float(u.y << 16); f[3] = __uint_as_float(u.y & 0xffff0000u);
    } else {
      const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
      f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
    }
    float am = fmaxf(fmaxf(fabsf(f[0]), fabsf(f[1])), fmaxf(fabsf(f[2]), fabsf(f[3])));
    am = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(am)));      // non-negative floats order like integers
    const uint32_t eb = __float_as_uint(am * 1.00396f) >> 23;           // biased exponent of a value just above the maximum
    const bool live = eb >= 15u && eb < 255u;
    const float inv = live ? __uint_as_float((268u - eb) << 23) : 0.f;   // 2^(14 - exponent): |v| <= 32639 = 127 * 256 + 127
    int v[4], s = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) { v[e] = __float2int_rn(f[e] * inv); s += v[e]; }
    // the low plane is the low byte of v as it is (a signed byte), the high plane byte 1 of v + 128
    uint32_t lo = prmt(prmt(v[0], v[1], 0x0040u), prmt(v[2], v[3], 0x0040u), 0x5410u);
    uint32_t hi = prmt(prmt(v[0] + 128, v[1] + 128, 0x0051u), prmt(v[2] + 128, v[3] + 128, 0x0051u), 0x5410u);
    if constexpr (FMT == FMT_Q4) {                 // the and delivers the codes as (0, 4, 1, 5) and (2, 6, 3, 7): neighbouring lanes swap
      const uint32_t ol = __shfl_xor_sync(0xffffffffu, lo, 1), oh = __shfl_xor_sync(0xffffffffu, hi, 1);
      lo = (lane & 1) ? prmt(ol, lo, 0x7362u) : prmt(lo, ol, 0x5140u);
      hi = (lane & 1) ? prmt(oh, hi, 0x7362u) : prmt(hi, oh, 0x5140u);
    }
    const int s_all = __reduce_add_sync(0xffffffffu, s), s_first = __reduce_add_sync(0xffffffffu, lane < 16 ? s : 0);
    // this lane's elements belong to MMA j = lane / 8 (32 elements each) and lane t of the product
    const uint32_t j = lane >> 3, t = (lane >> 1) & 3, d = xs + q * kPlaneBytes + (j >> 1) * 128 + t * 16 + (j & 1) * 8 + (lane & 1) * 4;
    sts_u1(d, lo);
    sts_u1(d + 64, hi);
    if (lane == 0) {
      const uint32_t meta = xs + q * kPlaneBytes + 256;
      sts_u1(meta, live ? (eb - 14u) << 23 : 0u);                        // 2^(exponent - 14)
      sts_u1(meta + 4, (uint32_t)s_first);
      sts_u1(meta + 8, (uint32_t)(s_all - s_first));
    }
  }
  }
}

// fp16 path: rows of tokens, `pitch` bytes apart (64 bytes past a multiple of 128: the 16-byte reads of a quarter warp, two
// rows of 64 bytes, then touch every bank once).  Every 16-byte piece (8 elements) holds the four register pairs in
// the order in which the products of FMT use them.  For the quantised formats also the sums of a tile's activations
// (the zero-point's factor): xsum[2 * pair + tile][token], and for bf16 activations, which may lie outside fp16's range, a
// power of two per (pair, token): the fp16 values are x / scale.
template <int FMT, int kWarps>
__device__ __forceinline__ void stage_x_f16(uint8_t* xs, uint32_t pitch, float* xsum, float* xscale, const void* x, bool bf16, int m, int d_in,
                                            uint32_t pair0, uint32_t n) {
  constexpr bool sums = FMT == FMT_Q4 || FMT == FMT_Q3;
  const uint32_t hw = threadIdx.x >> 4, l = threadIdx.x & 15, total = n * (uint32_t)m;
  constexpr int B = 4;                            // loads in flight per lane
  for (uint32_t u0 = hw; u0 < ((total + 1) & ~1u); u0 += B * 2 * kWarps) {
    uint4 raw[B];
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const uint32_t u = u0 + i * 2 * kWarps;
      if (u < total) {
        const uint32_t tok = u / n, q = u - tok * n;
        raw[i] = ld_cg_u4(reinterpret_cast<const uint16_t*>(x) + (size_t)tok * d_in + (size_t)(pair0 + q) * 128 + 8 * l);
      } else {
        raw[i] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const uint32_t u = u0 + i * 2 * kWarps;
      if ((u & ~1u) >= total) continue;                   // uniform over the warp: its halves take u and u + 1, u even
      uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
      const uint32_t tok = u / n, q = u - tok * n;
      float sc = 1.f;
      if (bf16) {
        float f[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) { f[2 * e] = __uint_as_float(w[e] << 16); f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
        float inv = 1.f;
        if constexpr (sums) {
          float am = 0.f;
#pragma unroll
          for (int e = 0; e < 8; ++e) am = fmaxf(am, fabsf(f[e]));
#pragma unroll
          for (int o = 1; o < 16; o <<= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
          const uint32_t eb = __float_as_uint(am) >> 23;
          if (eb >= 14u && eb < 255u) { inv = __uint_as_float((267u - eb) << 23); sc = __uint_as_float((eb - 13u) << 23); }   // largest magnitude in [2^13, 2^14); both factors are normal numbers
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = pack_h2(f[2 * e] * inv, f[2 * e + 1] * inv);
      }
      if constexpr (sums) {
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) { const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w[e])); s += v.x + v.y; }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (u < total) {
          if ((l & 7) == 0) xsum[(2 * q + (l >> 3)) * kMaxTok + tok] = s;
          if (l == 0) xscale[q * kMaxTok + tok] = sc;
        }
      }
      if (u < total) {
        uint4 o = make_uint4(w[0], w[1], w[2], w[3]);
        if constexpr (FMT == FMT_Q4) { o.y = w[2]; o.z = w[1]; }
        else if constexpr (FMT == FMT_Q3) o = make_uint4(prmt(w[0], w[1], 0x5410u), prmt(w[0], w[1], 0x7632u), prmt(w[2], w[3], 0x5410u), prmt(w[2], w[3], 0x7632u));
        *reinterpret_cast<uint4*>(xs + (size_t)tok * pitch + q * 256 + l * 16) = o;
      }
    }
  }
}

// ---- products ---------------------------------------------------------------------------------------------------
// Blobs and activations are addressed by 32-bit shared-memory addresses: what bounds the loop over the blobs is the number
// of instructions around the tensor-core products, and generic pointers cost two per step.

// One token, 3/4-bit backbone.  xa: this lane's planes of the pair (stage_x_i8; a block of zeros for the lanes that hold
// no column), xm: the pair's scale and sums.  acc[0] / acc[1] += rows g / g + 8 on the lanes with t == 0.
template <int FMT, bool SZ2>
__device__ __forceinline__ void product_i8(const RawBlob<FMT, SZ2>& r, uint32_t xa, uint32_t xm, float (&acc)[2]) {
  const uint4 xb[2] = {lds_u4(xa), lds_u4(xa + 128)};
  const uint4 meta = lds_u4(xm);
  const float scale = __uint_as_float(meta.x);
  const int xsum[2] = {(int)meta.y, (int)meta.z};
  int d[4] = {0, 0, 0, 0};             // rows g / g + 8 x columns (low, high plane) on the lanes with t == 0
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint32_t q[4][2];
    code_quads<FMT>(r.t[c], q);
    mma16832_s8(d, q[0][0], q[1][0], q[0][1], q[1][1], xb[c].x, xb[c].y);
    mma16832_s8(d, q[2][0], q[3][0], q[2][1], q[3][1], xb[c].z, xb[c].w);
    if (c == 1 || SZ2) {
      const int k = SZ2 ? c : 0;
      const int xs = SZ2 ? xsum[c] : xsum[0] + xsum[1];
      const float2 s = __half22float2(*reinterpret_cast<const __half2*>(&r.s[k]));
      const int z_a = (int)(r.z[k] & 255u), z_b = (int)(r.z[k] >> 8);
      acc[0] = fmaf((float)(d[1] * 256 + d[0] - z_a * xs), s.x * scale, acc[0]);
      acc[1] = fmaf((float)(d[3] * 256 + d[2] - z_b * xs), s.y * scale, acc[1]);
      d[0] = d[1] = d[2] = d[3] = 0;
    }
  }
}

// This lane's activation registers of a pair for tile c, four per half of the tile.
__device__ __forceinline__ void load_xf(uint32_t (&xr)[8], uint32_t row, int c) {
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const uint4 v = lds_u4(row + (2 * c + b) * 64);
    xr[4 * b] = v.x; xr[4 * b + 1] = v.y; xr[4 * b + 2] = v.z; xr[4 * b + 3] = v.w;
  }
}

// Two to eight tokens, 3/4-bit backbone, fp16 activations.  The codes go into the product as they lie in their words: as
// fp16 bit patterns they are the numbers q * 2^-24 (subnormals, which the tensor core multiplies exactly), or 16 (8 for 3-bit)
// times that where they sit four (three) bits higher; those go to an accumulator chain of their own.  One logic
// instruction per two codes instead of two, and nothing is rounded that was not before.
//   sum w x = s * (2^24 (chain 0 + chain 1 / 16) - z * sum x)
// row: this lane's activations of the pair; xsum: the sums of tokens 2t, 2t + 1 over the pair's first tile (32 bytes further: over
// its second); xscale: their scales (bf16 activations).  acc: (row g, token 2t), (g, 2t + 1), (g + 8, 2t), (g + 8, 2t + 1).
template <int FMT, bool SZ2>
__device__ __forceinline__ void product_codes(const RawBlob<FMT, SZ2>& r, uint32_t row, uint32_t xsum, uint32_t xscale, bool bf16, float (&acc)[4]) {
  constexpr float kUp = 16777216.f, kDown = FMT == FMT_Q4 ? 1.f / 16.f : 1.f / 8.f;
  float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
  float2 xs = make_float2(0.f, 0.f);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint32_t xr[8];
    load_xf(xr, row, c);
    uint32_t a[4][4];
    code_frags<FMT>(r.t[c], a);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      mma16816(d0, a[2 * b], xr[4 * b], xr[4 * b + 1]);
      mma16816(d1, a[2 * b + 1], xr[4 * b + 2], xr[4 * b + 3]);
    }
    const uint2 xc = lds_u2(xsum + c * 4 * kMaxTok);
    xs.x += __uint_as_float(xc.x); xs.y += __uint_as_float(xc.y);
    if (c == 1 || SZ2) {
      const int k = SZ2 ? c : 0;
      const float2 s = __half22float2(*reinterpret_cast<const __half2*>(&r.s[k]));
      const float za = -(float)(r.z[k] & 255u) * s.x, zb = -(float)(r.z[k] >> 8) * s.y;
      const float sa = s.x * kUp, sb = s.y * kUp;
      float v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        v[i] = fmaf(fmaf(d1[i], kDown, d0[i]), i < 2 ? sa : sb, (i < 2 ? za : zb) * ((i & 1) ? xs.y : xs.x));
        d0[i] = 0.f; d1[i] = 0.f;
      }
      if (bf16) {
        const uint2 sc = lds_u2(xscale);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] *= __uint_as_float((i & 1) ? sc.y : sc.x);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] += v[i];
      xs = make_float2(0.f, 0.f);
    }
  }
}

// Any format as exact fp16 values (q - z, or the 2:4 pattern expanded), times fp16 activations; LO: a second set of
// activations (the low part of t) `lo` bytes further.  blob: in shared memory; it is read tile by tile (an fp16 blob is 32
// registers a lane).
template <int FMT, bool SZ2, bool LO>
__device__ __forceinline__ void product_exact(uint32_t blob, int lane, uint32_t row, uint32_t lo, uint32_t lut, float (&acc)[4]) {
  constexpr bool quant = fmt_quantised(FMT);
  constexpr int tb = tile_bytes(FMT);
  float d[2][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { d[0][i] = 0.f; d[1][i] = 0.f; }
  ZC zc;
  float2 s = make_float2(1.f, 1.f);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if constexpr (quant) {
      if (c == 0 || SZ2) {
        const uint32_t sz = blob + 2 * tb + c * kSzEntryBytes, sw = lds_u1(sz + (lane >> 2) * 4);
        make_zc<FMT>(zc, lds_u16(sz + 32 + (lane >> 2) * 2));
        s = __half22float2(*reinterpret_cast<const __half2*>(&sw));
      }
    }
    RawTile<FMT> r;
    load_tile_s<FMT>(r, blob + c * tb, lane);
    uint32_t a[4][4];
    tile_frags<FMT>(r, zc, a, lut);
    uint32_t xr[8];
    load_xf(xr, row, c);
#pragma unroll
    for (int i = 0; i < 4; ++i) mma16816(d[i & 1], a[i], xr[2 * i], xr[2 * i + 1]);
    if constexpr (LO) {
      load_xf(xr, row + lo, c);
#pragma unroll
      for (int i = 0; i < 4; ++i) mma16816(d[i & 1], a[i], xr[2 * i], xr[2 * i + 1]);
    }
    if (c == 1 || (quant && SZ2)) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[i] = fmaf(d[0][i] + d[1][i], i < 2 ? s.x : s.y, acc[i]);
        d[0][i] = 0.f; d[1][i] = 0.f;
      }
    }
  }
}

// ---- A: t = X . A ---------------------------------------------------------------------------------------------------
// Unit u = (row tile of A, part of the reduction axis); its pairs go round the sixteen warps, whose sums meet in shared
// memory; the 16 x m results leave as words (value, launch number).
// Returns (thread 0) g_last_entry as it was when the launch in front had ended: asked for here, it costs nothing later (see hold_place).
__device__ unsigned long long g_last_entry;        // globaltimer when the last one-token launch on this device entered
template <int ABF, bool SZ2, int kWarps>
__device__ __forceinline__ unsigned long long run_a(const DecodeArgs& p, float* red, int warp, int lane, unsigned long long* tr) {
  constexpr uint32_t blob_b = blob_bytes(ABF, SZ2 ? 1 : 0);
  const uint32_t units = p.a_nt * p.a_slices;
  const int g = lane >> 2, t = lane & 3;
  const bool has = g < p.m;
  // weights ahead of the dependency: everything of this CTA towards L2 (A and B are small: 173 against 189 us without)
  for (uint32_t u = blockIdx.x + p.n_a * threadIdx.x; u < units; u += p.n_a * (kWarps * 32)) {
    const uint32_t tile = u % p.a_nt, s = u / p.a_nt, p0 = s * p.a_slice_pairs;
    if (p0 < p.a_np) prefetch_l2(p.a_q + ((size_t)tile * p.a_np + p0) * blob_b, min(p.a_slice_pairs, p.a_np - p0) * blob_b);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tr && lane == 0) tr[1] = globaltimer_ns();
  const uint32_t launch = launch_number(p.launches);
  unsigned long long seen = 0;
  if (threadIdx.x == 0) seen = ld_volatile_u64(&g_last_entry);
  const uint16_t* xrow = reinterpret_cast<const uint16_t*>(p.x) + (size_t)(has ? g : 0) * p.d_in + 8 * t;
  int flip = 0;
  for (uint32_t u = blockIdx.x; u < units; u += p.n_a, flip ^= 1) {
    const uint32_t tile = u % p.a_nt, s = u / p.a_nt;
    const uint32_t p0 = s * p.a_slice_pairs, p1 = min(p.a_np, p0 + p.a_slice_pairs);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (uint32_t q = p0 + warp; q < p1; q += kWarps) {
      const uint8_t* blob = p.a_q + ((size_t)tile * p.a_np + q) * blob_b;
      RawBlob<ABF, SZ2> r;
      load_blob(r, blob, lane);
      float d[2][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { d[0][i] = 0.f; d[1][i] = 0.f; }
      ZC zc;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint4 xv[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          xv[b] = has ? ld_cg_u4(xrow + (size_t)q * 128 + 32 * (2 * c + b)) : make_uint4(0u, 0u, 0u, 0u);
          if (p.x_dtype == EORA_X_BF16) { xv[b].x = bf2_to_h2(xv[b].x); xv[b].y = bf2_to_h2(xv[b].y); xv[b].z = bf2_to_h2(xv[b].z); xv[b].w = bf2_to_h2(xv[b].w); }
        }
        if constexpr (fmt_quantised(ABF)) { if (c == 0 || SZ2) make_zc<ABF>(zc, r.z[SZ2 ? c : 0]); }
        uint32_t a[4][4];
        tile_frags<ABF>(r.t[c], zc, a, 0u);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          mma16816(d[0], a[2 * b], xv[b].x, xv[b].y);
          mma16816(d[1], a[2 * b + 1], xv[b].z, xv[b].w);
        }
        if (c == 1 || (fmt_quantised(ABF) && SZ2)) {
          float2 sc = make_float2(1.f, 1.f);
          if constexpr (fmt_quantised(ABF)) sc = __half22float2(*reinterpret_cast<const __half2*>(&r.s[SZ2 ? c : 0]));
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            acc[i] = fmaf(d[0][i] + d[1][i], i < 2 ? sc.x : sc.y, acc[i]);
            d[0][i] = 0.f; d[1][i] = 0.f;
          }
        }
      }
    }
    float* mine = red + (flip * kWarps + warp) * 16 * kMaxTok;
    mine[(2 * t) * 16 + g] = acc[0]; mine[(2 * t + 1) * 16 + g] = acc[1];
    mine[(2 * t) * 16 + g + 8] = acc[2]; mine[(2 * t + 1) * 16 + g + 8] = acc[3];
    __syncthreads();
    if (threadIdx.x < 16u * p.m) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) v += red[(flip * kWarps + w) * 16 * kMaxTok + threadIdx.x];
      const uint32_t tok = threadIdx.x >> 4, col = tile * 16 + (threadIdx.x & 15);
      const unsigned long long word = ((unsigned long long)launch << 32) | __float_as_uint(v);
      asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p.t_part + ((size_t)s * p.m + tok) * p.t_cols + col), "l"(word) : "memory");
    }
  }
  if (tr && lane == 0) tr[2] = globaltimer_ns();
  return seen;
}

// One token: an SM has room for two CTAs, one of this launch and one of the launch behind it.  A CTA that holds A is done long before the
// others.  If it left before the launch behind had been placed (calls that are enqueued one by one arrive during the launch in front), that launch
// would put two of its CTAs on this SM and none on another, would take as long as those two, and hand the imbalance on: gate|up at one token 22
// us instead of 15, four blocks 248 us enqueued against 178 in a graph.  So the CTA keeps its place until a launch has entered after its own, or the
// first of the others is about to store its sums, or for kHoldNs (with many streams such CTAs could otherwise fill the chip).  Only timing
// depends on it.  Kept always until the others' end, four blocks in a graph took 183 us instead of 178: the launch after next is placed later.
constexpr unsigned long long kHoldNs = 30000ull, kEntrySpreadNs = 1000ull;      // (CTAs of one launch enter within 0.6 us on a free chip)
__device__ __forceinline__ void hold_place(const unsigned long long* launches, unsigned long long entry, unsigned long long seen) {
  if (seen > entry + kEntrySpreadNs) return;
  const unsigned long long t0 = globaltimer_ns();
  while (ld_volatile_u64(&g_last_entry) <= entry + kEntrySpreadNs && (ld_volatile_u64(launches) & ((1ull << kLaunchShift) - 1)) == 0 &&
         globaltimer_ns() - t0 < kHoldNs) __nanosleep(100);
}

// ---- after the backbone: + t . B, the partner's sums, Y ---------------------------------------------------------------
__device__ __forceinline__ int sub_of(const DecodeArgs& p, uint32_t tile) {
  if (p.n_sub == 1) return 0;
  int s = 0;
#pragma unroll
  for (int i = 1; i < 4; ++i)
    if (i < p.n_sub && tile >= p.sub_tile0[i]) s = i;
  return s;
}

// x / n for small x; inv = ceil(2^32 / n), 0 for n == 1
__device__ __forceinline__ uint32_t div_by(uint32_t x, uint32_t inv) { return inv ? __umulhi(x, inv) : x; }
// The warps whose runs hold blobs of row tile f of a chunk of n pairs: those of its first to its last blob.  Warp w's run is
// [w L / kWarps, (w + 1) L / kWarps) of the L blobs; inv = ceil(2^32 / L).
struct Owners { uint32_t a, b; };
template <int kWarps>
__device__ __forceinline__ Owners owners_of(uint32_t f, uint32_t n, uint32_t inv) {
  const uint32_t x = (f * n + 1) * kWarps - 1;
  return {div_by(x, inv), div_by(x + (n - 1) * kWarps, inv)};
}

// Pairs of t that row tile `tile` takes part in, within [c0, c1): [a, b).
struct Span { uint32_t a, b, base; };
__device__ __forceinline__ Span t_span(const DecodeArgs& p, uint32_t tile, uint32_t c0, uint32_t c1) {
  Span s;
  s.base = p.sub_pairs ? (uint32_t)sub_of(p, tile) * p.sub_pairs : 0u;
  s.a = max(c0, s.base); s.b = min(c1, s.base + p.b_np);
  return s;
}

// What a CTA does once its warps' runs are in `seg`: adds up the row tiles that its partner finishes and sends it the sums,
// adds t . B and the partner's sums to its own, and stores Y.  Everything that has to come from L2 (the first words of t, the
// first blob of B, which goes to the warp's ring) is asked for before the barrier that the warps meet at.  All of it is
// latency -- a shared-memory load in a rolled loop costs 60 cycles -- so every element has a thread of its own: half a warp
// per (row tile, token), tokens counted up to a power of two (1 << p.m_log).  Few values live across its phases: with two
// CTAs of 512 threads an SM has 64 registers a thread, and a spill goes to L2 (shared memory takes nearly all of the L1).
//
// The product with B: unit u = (row tile u >> b_log, every (1 << b_log)-th of its pairs in the chunk of t, from u's low bits on);
// units go round the warps.  bar, parity: the barrier of the warp's (empty) ring that a blob of B arrives at.  ok: false in a warp whose wait
// ran out, which asks for nothing more.
template <int ABF, bool SZ2, int kWarps>
__device__ __forceinline__ void finish(const DecodeArgs& p, uint8_t* smem, uint32_t ring, uint32_t bar, uint32_t parity, uint32_t t0, uint32_t nT,
                                       uint32_t rank, uint32_t n, uint32_t inv, uint32_t launch, bool ok, unsigned long long* tr) {
  constexpr bool ab = ABF != FMT_NONE;
  constexpr uint32_t blob_b = blob_bytes(ABF, SZ2 ? 1 : 0);
  const uint32_t OT = 16u * p.m;
  const uint32_t f0 = rank ? nT >> 1 : 0u, nf = (p.ks == 2 && rank == 0 ? nT >> 1 : nT) - f0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* const seg = reinterpret_cast<float*>(smem + p.off_seg);
  const uint32_t hw = threadIdx.x >> 4, row = threadIdx.x & 15;
  const uint32_t first_tile = t0 + f0;

  auto ask_b = [&](uint32_t tile, uint32_t pair) {
    if (lane == 0) {
      mbar_expect_tx_a(bar, blob_b);
      bulk_g2s_a(ring, p.b_q + ((size_t)tile * p.b_np + pair) * blob_b, blob_b, bar);
    }
  };
  // step e of a chunk of t: two columns of one token (64 steps per pair and token)
  auto t_tok = [&](uint32_t e) { return (e >> 6) & ((1u << p.m_log) - 1); };
  auto t_col = [&](uint32_t e) { return (e >> (6 + p.m_log)) * 128 + (e & 63) * 2; };
  uint32_t c0 = 0, c_end = p.b_np;                 // the chunk of t and the end of all chunks
  TWords tw = {0ull, 0ull};
  if constexpr (ab) {
    if (p.sub_pairs && nf) { c0 = (uint32_t)sub_of(p, first_tile) * p.sub_pairs; c_end = (uint32_t)(sub_of(p, first_tile + nf - 1) + 1) * p.sub_pairs; }
    if (ok && warp < (int)(nf << p.b_log)) {
      const uint32_t tile = first_tile + (warp >> p.b_log);
      const Span s = t_span(p, tile, c0, c0 + p.t_chunk);
      const uint32_t q = s.a + (warp & ((1u << p.b_log) - 1));
      if (q < s.b) ask_b(tile, q - s.base);
    }
    if (t_tok(threadIdx.x) < (uint32_t)p.m && c0 * 128 + t_col(threadIdx.x) < (uint32_t)p.t_cols)
      load_t(tw, p.t_part + (size_t)t_tok(threadIdx.x) * p.t_cols + c0 * 128 + t_col(threadIdx.x));
  }
  __syncthreads();
  if (tr && lane == 0) tr[2] = globaltimer_ns();

  auto tile_sum = [&](uint32_t f, uint32_t i) {    // element i of the sums of row tile f: of all warps that hold blobs of it
    const Owners o = owners_of<kWarps>(f, n, inv);
    const float* src = seg + (o.a + f) * OT + i;
    float v0 = 0.f, v1 = 0.f;
    if ((rank ? p.w_np - p.pairs : p.pairs) > p.chunk) v0 = reinterpret_cast<const float*>(smem + p.off_sum)[f * OT + i];     // of the chunks before
    uint32_t k = o.b - o.a + 1;
    for (; k >= 4; k -= 4, src += 4 * OT) { v0 += src[0] + src[OT]; v1 += src[2 * OT] + src[3 * OT]; }
    if (k > 0) v0 += src[0];
    if (k > 1) v1 += src[OT];
    if (k > 2) v0 += src[2 * OT];
    return v0 + v1;
  };
  if (p.ks == 2) {
    // the partner's tiles: [nf, nT) for rank 0, [0, f0) for rank 1
    cluster_wait();
    const uint32_t to = mapa(smem_u32(smem + p.off_inbox), rank ^ 1u) + row * 4;
    for (uint32_t u = hw; u < (nT - nf) << p.m_log; u += 2 * kWarps) {
      const uint32_t f = u >> p.m_log, tok = u & ((1u << p.m_log) - 1);
      if (tok < (uint32_t)p.m)
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to + (f * OT + tok * 16) * 4), "f"(tile_sum(rank ? f : nf + f, tok * 16 + row)) : "memory");
    }
    cluster_arrive();
  }
  if constexpr (ab) {
    const uint32_t pitch = p.t_chunk * 256 + 64;
    const uint32_t th = smem_u32(smem + p.off_t);
    float* const bseg = reinterpret_cast<float*>(smem + p.off_bseg);
    bool first = true;
#pragma unroll 1
    while (nf) {
      // t of this chunk as fp16 high and low parts (error 2^-22 of the value), zero for tokens that do not use the pair's adapter
      // and in the columns past A's rows (padding)
      const uint32_t steps = min(p.t_chunk, c_end - c0) << (6 + p.m_log);
      for (uint32_t e = threadIdx.x; e < steps; e += (kWarps * 32)) {
        const uint32_t tok = t_tok(e), col = t_col(e);
        if (tok >= (uint32_t)p.m) continue;
        float v0 = 0.f, v1 = 0.f;
        if (c0 * 128 + col < p.a_nt * 16 && !(p.adp_pairs && p.adp[tok] != (int)((c0 + (col >> 7)) / p.adp_pairs))) {
          const unsigned long long* src = p.t_part + (size_t)tok * p.t_cols + c0 * 128 + col;
#pragma unroll 1
          for (uint32_t s = 0; s < p.a_slices; ++s, src += (size_t)p.m * p.t_cols) {
            if (!first || s || e != threadIdx.x) load_t(tw, src);
            if (!wait_t(tw, src, launch, p.wait_ns, p.dev_status)) break;
            v0 += __uint_as_float((uint32_t)tw.a); v1 += __uint_as_float((uint32_t)tw.b);
          }
        }
        const uint32_t hi = pack_h2(v0, v1);
        const float2 hf = __half22float2(*reinterpret_cast<const __half2*>(&hi));
        const uint32_t d = th + tok * pitch + col * 2;
        sts_u1(d, hi);
        sts_u1(d + p.m * pitch, pack_h2(v0 - hf.x, v1 - hf.y));
      }
      __syncthreads();
#pragma unroll 1
      for (uint32_t u = warp; u < nf << p.b_log; u += kWarps) {
        const uint32_t tile = first_tile + (u >> p.b_log);
        const Span s = t_span(p, tile, c0, c0 + p.t_chunk);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (uint32_t q = s.a + (u & ((1u << p.b_log) - 1)), k = 0; ok && q < s.b; q += 1u << p.b_log, ++k) {
          if (!first || u != (uint32_t)warp || k) ask_b(tile, q - s.base);
          ok = __all_sync(0xffffffffu, mbar_try_wait_a(bar, parity) || mbar_wait_lane(bar, parity, p.dev_status));
          if (!ok) { mbar_drain_warp(bar, parity, lane); break; }
          parity ^= 1u;
          // columns past the tokens repeat the last one; their sums are not stored
          product_exact<ABF, SZ2, true>(ring, lane, th + min((uint32_t)lane >> 2, (uint32_t)p.m - 1) * pitch + (lane & 3) * 16 + (q - c0) * 256, p.m * pitch, 0u, acc);
          __syncwarp();
        }
        float* d = bseg + u * OT + (lane >> 2) + (lane & 3) * 32;
        if (2 * (lane & 3) < p.m) { d[0] = acc[0]; d[8] = acc[2]; }
        if (2 * (lane & 3) + 1 < p.m) { d[16] = acc[1]; d[24] = acc[3]; }
      }
      c0 += p.t_chunk;
      if (c0 >= c_end) break;
      first = false;
      __syncthreads();
      // more chunks of t: this one's products join the first of the tile's partial sums
      for (uint32_t e = threadIdx.x; e < nf * OT; e += (kWarps * 32)) {
        const uint32_t f = e / OT, i = e - f * OT;
        float v = 0.f;
        for (uint32_t k = 0; k < 1u << p.b_log; ++k) v += bseg[((f << p.b_log) + k) * OT + i];
        seg[(owners_of<kWarps>(f0 + f, n, inv).a + f0 + f) * OT + i] += v;
      }
    }
  }
  if (p.ks == 2) cluster_wait();
  __syncthreads();
  if (threadIdx.x == 0) count_launch(p.launches);  // (every thread of the CTA has read the counter)
  for (uint32_t u = hw; u < nf << p.m_log; u += 2 * kWarps) {
    const uint32_t f = u >> p.m_log, tok = u & ((1u << p.m_log) - 1), i = tok * 16 + row;
    if (tok >= (uint32_t)p.m) continue;
    float v = tile_sum(f0 + f, i);
    if (p.ks == 2) v += reinterpret_cast<const float*>(smem + p.off_inbox)[f * OT + i];
    if constexpr (ab)
      for (uint32_t k = 0; k < 1u << p.b_log; ++k) v += reinterpret_cast<const float*>(smem + p.off_bseg)[((f << p.b_log) + k) * OT + i];
    const uint32_t tg = first_tile + f;
    void* y = p.ys[0];
    uint32_t st0 = 0;
    int dout = p.sub_dout[0];
    if (p.n_sub > 1) {
#pragma unroll
      for (int k = 1; k < 4; ++k)
        if (k < p.n_sub && tg >= p.sub_tile0[k]) { y = p.ys[k]; st0 = p.sub_tile0[k]; dout = p.sub_dout[k]; }
    }
    store_y(y, p.y_dtype, (int64_t)tok * dout + (tg - st0) * 16 + row, v);
  }
}

// MODE 1: one token through the integer product, 0: fp16 activations.
// Blobs that a warp multiplies at once.
__host__ __device__ constexpr uint32_t fast_blobs(int fmt, int mode) { return mode == 1 ? 4 : fmt == FMT_Q4 || fmt == FMT_Q3 ? 2 : 1; }

// 120 registers a thread, not 128: two CTAs of the one-token form (one of the larger form) then leave an SM 4096 registers, enough for a CTA
// of the staging kernel of the host-buffer calls.  With all registers taken, the SMs that held such a CTA had no room for the launch behind it,
// which put its last CTAs in pairs on other SMs (see hold_place): four 3-bit blocks of host-buffer calls in a graph 264 us, so 214; enqueued 358 and 313.
template <int WF, int MODE, bool SZ2>
__global__ void __maxnreg__(120) k_decode(const __grid_constant__ DecodeArgs p) {
  constexpr int kWarpLog = warp_log(MODE), kWarps = 1 << kWarpLog;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(256) uint32_t lut_s[16];
  __shared__ __align__(16) uint32_t zero_s[52];    // what lanes without a token read as their activations: up to 208 bytes (load_xf)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  asm volatile("griddepcontrol.launch_dependents;");
  touch_args(p);
  unsigned long long entry = 0;
  if (MODE == 1 && threadIdx.x == 0 && blockIdx.x < max(p.n_a, 1u)) {
    entry = globaltimer_ns();
    if (blockIdx.x == 0) asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(&g_last_entry), "l"(entry) : "memory");
  }
  unsigned long long* tr = p.trace ? p.trace + (size_t)(blockIdx.x * 16 + warp) * 4 : nullptr;
  if (tr && lane == 0) tr[0] = globaltimer_ns();

  if (blockIdx.x < p.n_a) {
    float* red = reinterpret_cast<float*>(smem);
    unsigned long long seen = 0;
    switch (p.a_fmt) {
      case FMT_F16: seen = run_a<FMT_F16, false, kWarps>(p, red, warp, lane, tr); break;
      case FMT_Q8: seen = run_a<FMT_Q8, false, kWarps>(p, red, warp, lane, tr); break;
      case FMT_Q4: if (p.a_sz2) seen = run_a<FMT_Q4, true, kWarps>(p, red, warp, lane, tr); else seen = run_a<FMT_Q4, false, kWarps>(p, red, warp, lane, tr); break;
      case FMT_Q3: if (p.a_sz2) seen = run_a<FMT_Q3, true, kWarps>(p, red, warp, lane, tr); else seen = run_a<FMT_Q3, false, kWarps>(p, red, warp, lane, tr); break;
      default: break;
    }
    __syncthreads();                               // every thread of the CTA has read the launch counter
    if (threadIdx.x == 0) {
      if constexpr (MODE == 1) hold_place(p.launches, entry, seen);
      count_launch(p.launches);
    }
  } else {
    constexpr uint32_t blob_b = blob_bytes(WF, SZ2 ? 1 : 0);
    const uint32_t cta = blockIdx.x - p.n_a, cl = p.ks == 2 ? cta >> 1 : cta, rank = p.ks == 2 ? cta & 1 : 0;
    const uint32_t t0 = share_lo(p.tiles, cl), nT = share_n(p.tiles, cl);
    const DecodeArgs::Part part = p.part[rank];
    const uint32_t pr0 = rank * p.pairs, P = part.pairs;
    const uint32_t OT = 16u * p.m;
    uint8_t* xs = smem;
    float* seg = reinterpret_cast<float*>(smem + p.off_seg);
    // the CTA's blobs are one contiguous range: the two halves of the reduction axis are stored one after the other
    const uint8_t* w_part = p.w_q + ((size_t)rank * p.w_nt * p.pairs + (size_t)t0 * P) * blob_b;
    if (p.ks == 2) cluster_arrive();               // (that the partner runs at all, before anything is written to it)
    uint32_t lut = 0;
    if constexpr (WF == FMT_SP24 || WF == FMT_SQ4) lut = sp24_lut(lut_s);
    if (threadIdx.x < 52) zero_s[threadIdx.x] = 0u;

    // A warp's run of a chunk of n pairs: blobs [lo, hi) in (row tile, pair) order.  They come through the warp's own ring in
    // shared memory, one bulk copy of up to slot_blobs blobs per slot.
    const uint32_t slot_b = p.slot_blobs * blob_b;
    Ring ring;
    ring.bytes = p.slots * slot_b; ring.base = smem_u32(smem + p.off_ring) + warp * p.ring_pitch;
    ring.bars = ring.bar = smem_u32(smem + p.off_bar) + warp * (kMaxSlots * 8);
    ring.so = 0; ring.parity = 0;
    if (lane == 0) {
      for (uint32_t i = 0; i < p.slots; ++i) mbar_init_a(ring.bars + 8 * i, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    uint32_t left = 0, tile = 0, pr = 0;           // blobs of the run still to be multiplied; the next one
    uint32_t l_left = 0, l_pr = 0;                 // copies: blobs of the run still to be asked for, pair of the next one
    const uint8_t* l_ptr = w_part;
    const bool whole = P <= p.chunk;                     // one chunk: the run is contiguous in memory
    auto open_run = [&](uint32_t c, uint32_t n) {
      const uint32_t L = nT * n, lo = ((uint32_t)warp * L) >> kWarpLog;
      left = (((uint32_t)(warp + 1) * L) >> kWarpLog) - lo;
      tile = whole ? div_by(lo, part.inv_pairs) : lo / n;
      pr = lo - tile * n;
      l_pr = pr; l_left = left;
      l_ptr = w_part + ((size_t)tile * P + c + pr) * blob_b;
    };
    auto ask = [&](uint32_t dst_o, uint32_t b, uint32_t n) {
      uint32_t cnt = min(p.slot_blobs, l_left);
      if (!whole) cnt = min(cnt, n - l_pr);
      if (cnt == 0) return;
      const uint32_t bytes = cnt * blob_b;
      if (lane == 0) {
        mbar_expect_tx_a(b, bytes);
        bulk_g2s_a(ring.base + dst_o, l_ptr, bytes, b);
      }
      l_left -= cnt; l_ptr += bytes;
      if (!whole) { l_pr += cnt; if (l_pr == n) { l_pr = 0; l_ptr += (P - n) * blob_b; } }
    };
    auto fill = [&](uint32_t n) {                  // the first copies of a run, into the slots from the reading position on
      uint32_t o = ring.so, b = ring.bar;
#pragma unroll 1
      for (uint32_t i = 0; i < p.slots; ++i) {
        ask(o, b, n);
        o += slot_b; b += 8;
        if (o == ring.bytes) { o = 0; b = ring.bars; }
      }
    };
    const uint32_t chunk0 = min(p.chunk, P);
    open_run(0, chunk0);
    fill(chunk0);
    if (p.n_a) {
      const uint32_t f0 = rank ? nT >> 1 : 0u, nf = (p.ks == 2 && rank == 0 ? nT >> 1 : nT) - f0;
      const uint32_t per_tile = p.b_np * (uint32_t)blob_bytes(p.a_fmt, (int)p.b_sz2), bytes = nf * per_tile;
      const uint8_t* b_part = p.b_q + (size_t)(t0 + f0) * per_tile;
      for (uint32_t o = threadIdx.x << 14; o < bytes; o += (kWarps * 32) << 14) prefetch_l2(b_part + o, min(16384u, bytes - o));
    }
    const int g = lane >> 2, t = lane & 3;
    const bool bf16 = p.x_dtype == EORA_X_BF16;
    bool ok = true;

    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tr && lane == 0) tr[1] = globaltimer_ns();
    const uint32_t launch = launch_number(p.launches);

    uint32_t n = 0, inv = 0;
#pragma unroll 1
    for (uint32_t c = 0; c < P; c += p.chunk) {
      n = min(p.chunk, P - c);
      inv = whole ? part.inv_blobs[nT - p.tiles.per] : 0xffffffffu / (nT * n) + 1u;
      const uint32_t pitch = p.chunk * 256 + 64;
      float* xsum = reinterpret_cast<float*>(xs + (size_t)p.m * pitch);          // fp16 path: [2 chunk][8] sums, [chunk][8] scales
      float* xscale = xsum + 2 * p.chunk * kMaxTok;
      if (c > 0) {
        open_run(c, n);
        if (ok) fill(n); else left = 0;
      }
      if constexpr (MODE == 1) stage_x_i8<WF, kWarps>(smem_u32(xs), p.x, bf16, pr0 + c, n, warp, lane);
      else stage_x_f16<WF, kWarps>(xs, pitch, xsum, xscale, p.x, bf16, p.m, p.d_in, pr0 + c, n);
      __syncthreads();
      float acc[MODE == 1 ? 2 : 4];
#pragma unroll
      for (int i = 0; i < (MODE == 1 ? 2 : 4); ++i) acc[i] = 0.f;
      // this lane's activations of a pair: base and step per pair (lanes without a token stay on the zeros)
      const bool has = MODE == 1 ? g < 2 : g < p.m;
      const uint32_t x_step = has ? (MODE == 1 ? kPlaneBytes : 256u) : 0u;
      const uint32_t x_base = has ? smem_u32(xs) + (MODE == 1 ? (g * 4 + t) * 16 : g * pitch + t * 16) : smem_u32(zero_s);
      const uint32_t x_meta = MODE == 1 ? smem_u32(xs) + 256 : smem_u32(xsum) + 8 * t;
      float* d = seg + (warp + tile) * OT + g;
      auto flush = [&]() {
        if constexpr (MODE == 1) {
          if (t == 0) { d[0] = acc[0]; d[8] = acc[1]; }
          acc[0] = acc[1] = 0.f;
        } else {
          if (2 * t < p.m) { d[(2 * t) * 16] = acc[0]; d[(2 * t) * 16 + 8] = acc[2]; }
          if (2 * t + 1 < p.m) { d[(2 * t + 1) * 16] = acc[1]; d[(2 * t + 1) * 16 + 8] = acc[3]; }
          acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
        }
        d += OT;
      };
      uint32_t xa = x_base + pr * x_step, xm = x_meta + pr * (MODE == 1 ? (uint32_t)kPlaneBytes : 8u * kMaxTok);
      bool open = left == 0;                       // something to leave in the slot at the end (an empty run leaves zeros)
#pragma unroll 1
      while (left > 0) {
        uint32_t cnt = min(p.slot_blobs, left);
        if (!whole) cnt = min(cnt, n - pr);
        if (!__all_sync(0xffffffffu, mbar_try_wait_a(ring.bar, ring.parity) || mbar_wait_lane(ring.bar, ring.parity, p.dev_status))) {
          ok = false;                              // gave up: nothing more is asked for (and the ring stays where it is, to say what is in flight)
          break;
        }
        uint32_t src = ring.base + ring.so;
        left -= cnt;
        // NB blobs of one row tile at once (independent chains hide one another's latency), one at a time around its end
        constexpr uint32_t NB = fast_blobs(WF, MODE), xm_step = MODE == 1 ? (uint32_t)kPlaneBytes : 8u * kMaxTok;
        open = true;
        auto blobs = [&](auto count) {
          constexpr int N = decltype(count)::value;
          if constexpr (WF == FMT_Q4 || WF == FMT_Q3) {
            RawBlob<WF, SZ2> raw[N];
#pragma unroll
            for (int k = 0; k < N; ++k) load_blob_s(raw[k], src + k * blob_b, lane);
#pragma unroll
            for (int k = 0; k < N; ++k) {
              if constexpr (MODE == 1) product_i8<WF, SZ2>(raw[k], xa + k * x_step, xm + k * xm_step, acc);
              else product_codes<WF, SZ2>(raw[k], xa + k * x_step, xm + k * xm_step, smem_u32(xscale) + ((pr + k) * kMaxTok + 2 * t) * 4, bf16, acc);
            }
          } else {
#pragma unroll
            for (int k = 0; k < N; ++k) product_exact<WF, SZ2, false>(src + k * blob_b, lane, xa + k * x_step, 0u, lut, acc);
          }
          src += N * blob_b; xa += N * x_step; xm += N * xm_step; pr += N; cnt -= N;
          if (pr == n) { flush(); open = false; pr = 0; xa = x_base; xm = x_meta; }
        };
#pragma unroll 1
        while (cnt > 0) {
          if (NB > 1 && cnt >= NB && pr + NB <= n) { open = true; blobs(std::integral_constant<int, NB>()); }
          else { open = true; blobs(std::integral_constant<int, 1>()); }
        }
        __syncwarp();                              // every lane is done with the slot
        ask(ring.so, ring.bar, n);
        ring_next(ring, slot_b);
      }
      if (open) flush();
      if (c + p.chunk < P) {                       // more chunks: add up what there is
        __syncthreads();
        float* sum = reinterpret_cast<float*>(smem + p.off_sum);
        for (uint32_t f = threadIdx.x >> 4; f < nT; f += 2 * kWarps) {
          const Owners o = owners_of<kWarps>(f, n, inv);
          for (uint32_t i = threadIdx.x & 15; i < OT; i += 16) {
            float v = c ? sum[f * OT + i] : 0.f;
            for (uint32_t w = o.a; w <= o.b; ++w) v += seg[(w + f) * OT + i];
            sum[f * OT + i] = v;
          }
        }
      }
    }
    if (!ok) {                                     // what is in flight must land before its memory is used for anything else
      for (uint32_t i = 0; i < p.slots; ++i) mbar_drain_warp(ring.bars + 8 * i, ring.bars + 8 * i < ring.bar ? ring.parity ^ 1u : ring.parity, lane);
    }
    switch (p.a_fmt) {
      case FMT_F16: finish<FMT_F16, false, kWarps>(p, smem, ring.base, ring.bar, ring.parity, t0, nT, rank, n, inv, launch, ok, tr); break;
      case FMT_Q8: finish<FMT_Q8, false, kWarps>(p, smem, ring.base, ring.bar, ring.parity, t0, nT, rank, n, inv, launch, ok, tr); break;
      case FMT_Q4: if (p.b_sz2) finish<FMT_Q4, true, kWarps>(p, smem, ring.base, ring.bar, ring.parity, t0, nT, rank, n, inv, launch, ok, tr);
                   else finish<FMT_Q4, false, kWarps>(p, smem, ring.base, ring.bar, ring.parity, t0, nT, rank, n, inv, launch, ok, tr); break;
      case FMT_Q3: if (p.b_sz2) finish<FMT_Q3, true, kWarps>(p, smem, ring.base, ring.bar, ring.parity, t0, nT, rank, n, inv, launch, ok, tr);
                   else finish<FMT_Q3, false, kWarps>(p, smem, ring.base, ring.bar, ring.parity, t0, nT, rank, n, inv, launch, ok, tr); break;
      default: finish<FMT_NONE, false, kWarps>(p, smem, ring.base, ring.bar, ring.parity, t0, nT, rank, n, inv, launch, ok, tr); break;
    }
  }
  if (tr && lane == 0) tr[3] = globaltimer_ns();
}

template <auto KERNEL>
cudaError_t launch_kernel(const cudaLaunchConfig_t& cfg, const DecodeArgs& args, int device) {
  static bool attr_set[64] = {};  // per kernel (KERNEL is a template argument) and device: the attribute belongs to the current device
  if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[device]) {
    cudaError_t e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e != cudaSuccess) return e;
    attr_set[device] = true;
  }
  return cudaLaunchKernelEx(&cfg, KERNEL, args);
}

cudaError_t launch_any(const cudaLaunchConfig_t& cfg, const DecodeArgs& a, int wf, bool sz2, int device) {
  const bool one = a.m == 1;
  switch (wf) {
    case FMT_Q4:
      if (one) return sz2 ? launch_kernel<k_decode<FMT_Q4, 1, true>>(cfg, a, device) : launch_kernel<k_decode<FMT_Q4, 1, false>>(cfg, a, device);
      return sz2 ? launch_kernel<k_decode<FMT_Q4, 0, true>>(cfg, a, device) : launch_kernel<k_decode<FMT_Q4, 0, false>>(cfg, a, device);
    case FMT_Q3:
      if (one) return sz2 ? launch_kernel<k_decode<FMT_Q3, 1, true>>(cfg, a, device) : launch_kernel<k_decode<FMT_Q3, 1, false>>(cfg, a, device);
      return sz2 ? launch_kernel<k_decode<FMT_Q3, 0, true>>(cfg, a, device) : launch_kernel<k_decode<FMT_Q3, 0, false>>(cfg, a, device);
    case FMT_SQ4: return sz2 ? launch_kernel<k_decode<FMT_SQ4, 0, true>>(cfg, a, device) : launch_kernel<k_decode<FMT_SQ4, 0, false>>(cfg, a, device);
    case FMT_SP24: return launch_kernel<k_decode<FMT_SP24, 0, false>>(cfg, a, device);
    default: return cudaErrorInvalidValue;
  }
}

// SM cycles per blob of the backbone / of A or B (only the ratios matter, to deal the CTAs).
double blob_cost(int fmt, bool int8) {
  switch (fmt) {
    case FMT_Q3: case FMT_Q4: return int8 ? 32.0 : 42.0;
    case FMT_SQ4: return 50.0;
    case FMT_SP24: return 100.0;          // 2304 bytes: HBM's rate
    default: return 45.0;
  }
}

Share make_share(uint32_t total, uint32_t n) {
  Share s;
  s.per = n ? total / n : 0;
  s.rem = n ? total % n : 0;
  return s;
}

struct Plan { DecodeArgs a; int grid; int warps; int smem; uint32_t ring; };

// How a launch of m (at most eight) tokens is cut up, with the activations in `chunks` parts and at most max_tiles row tiles per cluster;
// false if its shared memory does not fit.
bool cut(const Handle* h, int m, uint32_t chunks, uint32_t max_tiles, Plan& pl) {
  DecodeArgs& a = pl.a;
  a = DecodeArgs();
  const bool ab = h->cfg.rank > 0;
  const bool int8 = m == 1 && (h->w.fmt == FMT_Q4 || h->w.fmt == FMT_Q3);
  const uint32_t kWarps = 1u << warp_log(int8 ? 1 : 0);
  pl.warps = (int)kWarps;
  a.w_q = h->w.q; a.w_nt = h->w.nt; a.w_np = h->w.np;
  a.ks = h->w.np >= 2 ? 2 : 1;
  a.pairs = h->w.half;
  a.m = m;
  while ((1 << a.m_log) < m) ++a.m_log;
  const uint32_t nt = h->w.nt, sms = (uint32_t)h->sm_count / a.ks * a.ks;
  a.a_fmt = FMT_NONE;
  a.a_slices = 1;
  if (ab) {
    a.a_fmt = h->a.fmt; a.a_q = h->a.q; a.a_nt = h->a.nt; a.a_np = h->a.np; a.a_sz2 = h->a.sz2;
    a.b_q = h->b.q; a.b_np = h->b.np; a.b_sz2 = h->b.sz2;
    // CTAs for A.  They work beside the others; what counts is the later of "the backbone's products are done" and "t
    // has arrived" (an exchange through L2 takes about 2500 cycles).  Row tiles are dealt whole, so some CTAs are often
    // free; of equal choices the one with the earliest t is taken.
    const double cw = blob_cost(h->w.fmt, int8), ca = blob_cost(h->a.fmt, false);
    double best = 1e30, best_a = 1e30;
    for (uint32_t na = a.ks; na <= sms / 3; na += a.ks) {
      const uint32_t ncl = (sms - na) / a.ks, per = (nt + ncl - 1) / ncl;
      const double tw = per * a.pairs * cw;
      uint32_t sl = 1;
      while (sl < (uint32_t)kMaxSlices && a.a_nt * sl < na && a.a_np >= 32 * sl) sl *= 2;
      const uint32_t sp = (a.a_np + sl - 1) / sl, rounds = (a.a_nt * sl + na - 1) / na;
      const double ta = 2500.0 + rounds * (300.0 + ((sp + kWarps - 1) / kWarps) * kWarps * ca);
      const double t = tw > ta ? tw : ta;
      if (t < 0.98 * best || (t <= 1.02 * best && ta < 0.98 * best_a)) { best = t; best_a = ta; a.n_a = na; a.a_slices = sl; a.a_slice_pairs = sp; }
    }
    if (a.n_a == 0) return false;
    a.sub_pairs = h->n_sub > 1 ? (uint32_t)h->r_pad / 128 : 0u;
  }
  uint32_t ncl = (sms - a.n_a) / a.ks;
  if (ncl > nt) ncl = nt;
  if ((nt + ncl - 1) / ncl > max_tiles) ncl = (nt + max_tiles - 1) / max_tiles;
  a.tiles = make_share(nt, ncl);
  auto inverse = [](uint32_t n) { return (uint32_t)((0x100000000ull + n - 1) / n); };      // 0 for n == 1
  for (int r = 0; r < 2; ++r) {
    const uint32_t P = r ? a.w_np - a.pairs : a.pairs;
    if (P == 0) continue;
    a.part[r].pairs = P; a.part[r].inv_pairs = inverse(P);
    for (int k = 0; k < 2; ++k) a.part[r].inv_blobs[k] = inverse((a.tiles.per + k) * P);
  }
  pl.grid = (int)(a.n_a + ncl * a.ks);
  if (pl.grid >= (1 << kLaunchShift)) return false;
  const uint32_t nT = a.tiles.per + (a.tiles.rem ? 1 : 0), nF = (nT + a.ks - 1) / a.ks;
  const bool codes = h->w.fmt == FMT_Q4 || h->w.fmt == FMT_Q3;
  const uint32_t per_pair = int8 ? (uint32_t)kPlaneBytes : (uint32_t)m * 256 + (codes ? 3 * kMaxTok * 4 : 0);
  a.chunk = (a.pairs + chunks - 1) / chunks;
  if ((uint64_t)kWarps * (nT * a.chunk) * (nT * a.chunk) >> 32) return false;      // (div_by is exact below that)
  const uint32_t t_pairs = (uint32_t)h->t_cols / 128;
  a.t_chunk = 32u / (uint32_t)m < t_pairs ? 32u / (uint32_t)m : t_pairs;
  // Shared memory: activations | barriers | rings (later blobs of B) | sums of the warps' runs | the partner's sums, and, after
  // the backbone's products (over the activations where they fit and no later chunk needs those): sums of the chunks before |
  // t . B | t.
  auto up = [](uint32_t v) { return (v + 127u) & ~127u; };
  const uint32_t OT = 64u * m;                     // bytes of a row tile's sums
  const uint32_t x_b = up(a.chunk * per_pair + (int8 ? 0u : 64u * m));
  while ((2u << a.b_log) * nF <= (uint32_t)kWarps && (1u << a.b_log) < a.t_chunk && (1u << a.b_log) < a.b_np) ++a.b_log;
  const uint32_t sum_b = a.chunk < a.pairs ? up(nT * OT) : 0u, bseg_b = ab ? up((nF > (uint32_t)kWarps ? nF : (uint32_t)kWarps) * OT) : 0u;
  const uint32_t t_b = ab ? up(2u * m * (a.t_chunk * 256 + 64)) : 0u, late_b = sum_b + bseg_b + t_b;
  const uint32_t keep_b = up((kWarps + nT) * OT) + (a.ks == 2 ? up(nF * OT) : 0u) + (a.chunk < a.pairs || late_b > x_b ? late_b : 0u);
  const uint32_t bar_b = kWarps * kMaxSlots * 8;
  // The ring takes what is left of half an SM, in two to four slots of one, two or four blobs; at least two
  // slots even if the CTA then needs an SM of its own.
  const uint32_t budget = int8 ? kHalfSmem : kMaxSmem;
  const uint32_t blob = (uint32_t)h->w.blob, fixed = x_b + bar_b + keep_b;
  const uint32_t room = fixed < budget ? (budget - fixed) / kWarps / blob : 0u;   // blobs per warp
  pl.ring = room * blob * kWarps;
  if (room >= 4) { a.slot_blobs = room >= 8 ? 4 : 2; a.slots = room / a.slot_blobs < kMaxSlots ? room / a.slot_blobs : kMaxSlots; }
  else { a.slot_blobs = 1; a.slots = room < 2 ? 2 : room; }
  a.off_bar = x_b;
  a.off_ring = a.off_bar + bar_b;
  a.ring_pitch = a.slots * a.slot_blobs * blob;
  if (ab && a.ring_pitch < (uint32_t)h->b.blob) a.ring_pitch = h->b.blob;      // (a blob of B at a time)
  uint32_t off = a.off_ring + up(kWarps * a.ring_pitch);
  a.off_seg = off; off += up((kWarps + nT) * OT);
  a.off_inbox = off; off += a.ks == 2 ? up(nF * OT) : 0u;
  if (a.chunk < a.pairs || late_b > x_b) { a.off_sum = off; off += late_b; }
  else a.off_sum = 0;                              // over the activations
  a.off_bseg = a.off_sum + sum_b;
  a.off_t = a.off_bseg + bseg_b;
  pl.smem = (int)off;
  if (pl.smem < (int)(2 * kWarps * 16 * kMaxTok * 4)) pl.smem = (int)(2 * kWarps * 16 * kMaxTok * 4);      // the A CTAs' sums
  return pl.smem <= kMaxSmem;
}

// The fewest parts of the activations with which the rings hold kRingLeast: every further part is a barrier, a round trip to L2 and rings
// that run empty (3-bit 14336 x 4096 at eight tokens, adapters of rank 128: three parts of 58 KB 24.2 us, one of 118 KB 19.4).  If none does (large blobs,
// many row tiles), the one with the largest ring; if nothing fits, fewer row tiles per cluster.
bool make_plan(const Handle* h, int m, Plan& pl) {
  for (uint32_t max_tiles = kMaxTiles; max_tiles >= 8; max_tiles -= 8) {
    uint32_t best = 0, best_ring = 0;
    for (uint32_t chunks = 1; chunks <= (uint32_t)h->w.half && chunks <= 64; ++chunks) {
      if (!cut(h, m, chunks, max_tiles, pl)) continue;
      if (pl.ring >= kRingLeast) return true;
      if (best == 0 || pl.ring > best_ring) { best = chunks; best_ring = pl.ring; }
      else break;
    }
    if (best) return cut(h, m, best, max_tiles, pl);
  }
  return false;
}

}  // namespace

// One thread waits, bounded by the handle's limit, for a word that nobody sends, after leaving a stale one where t's would
// be.  See eora_linear_selftest_wait_timeout.
__global__ void k_wait_selftest(unsigned long long* t_part, const unsigned long long* launches, int* dev_status, unsigned long long limit_ns) {
  if (threadIdx.x == 0) {
    t_part[0] = 0x3f800000ull;                     // 1.0f, sent by launch 0 (the first is number 1)
    const uint32_t want = launch_number(launches);
    const unsigned long long t0 = dec::globaltimer_ns();
    while ((uint32_t)(ld_volatile_u64(t_part) >> 32) != want) {
      if (dec::globaltimer_ns() - t0 > limit_ns) { atomicExch(dev_status, EORA_ERR_DEVICE_TIMEOUT); break; }
      __nanosleep(32);
    }
  }
}

cudaError_t launch_wait_selftest(const Handle* h, cudaStream_t st) {
  k_wait_selftest<<<1, 32, 0, st>>>(h->t_part, h->launches, h->dev_status, h->wait_limit_ns);
  return cudaGetLastError();
}

size_t decode_part_bytes(int t_cols) { return (size_t)kMaxSlices * kMaxTok * t_cols * 8; }

bool decode_supported(const Handle* h, int m) {
  if (m < 1 || m > 64) return false;
  if (h->sm_count < 2) return false;
  if (h->w.fmt != FMT_Q4 && h->w.fmt != FMT_Q3 && h->w.fmt != FMT_SP24 && h->w.fmt != FMT_SQ4) return false;
  Plan pl;
  return make_plan(h, m < kMaxTok ? m : kMaxTok, pl);
}

int decode_launch_count(const Handle*, int m) { return (m + kMaxTok - 1) / kMaxTok; }

int decode_grid(const Handle* h, int m) {
  Plan pl;
  return make_plan(h, m < kMaxTok ? m : kMaxTok, pl) ? pl.grid : 0;
}

cudaError_t launch_decode_forward(const Handle* h, const void* x, int m, void* const* ys, cudaStream_t st,
                                  const int32_t* adapter_ids) {
  Plan pl;
  DecodeArgs& a = pl.a;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const size_t ybytes = h->cfg.y_dtype == EORA_Y_F32 ? 4 : 2;
  int planned = 0;
  for (int m0 = 0; m0 < m; m0 += kMaxTok) {        // eight tokens per pass (the n8 side of the mma)
    const int mp = m - m0 < kMaxTok ? m - m0 : kMaxTok;
    if (mp != planned) {
      if (!make_plan(h, mp, pl)) return cudaErrorInvalidValue;
      planned = mp;
      a.n_sub = h->n_sub;
      for (int i = 0; i < 5; ++i) a.sub_tile0[i] = (uint32_t)(i <= h->n_sub ? h->sub_tile0[i] : h->w.nt);
      for (int i = 0; i < h->n_sub; ++i) a.sub_dout[i] = h->sub_dout[i];
      a.t_part = h->t_part; a.launches = h->launches; a.dev_status = h->dev_status;
      a.d_in = h->cfg.d_in; a.t_cols = h->t_cols;
      a.x_dtype = h->cfg.x_dtype; a.y_dtype = h->cfg.y_dtype;
      a.trace = reinterpret_cast<unsigned long long*>(h->trace);
      a.wait_ns = h->wait_limit_ns;
      cfg.gridDim = dim3(pl.grid);
      cfg.blockDim = dim3(pl.warps * 32);
      cfg.dynamicSmemBytes = pl.smem;
      attr[1].val.clusterDim.x = a.ks;
    }
    a.x = reinterpret_cast<const uint8_t*>(x) + (size_t)m0 * h->cfg.d_in * 2;
    for (int i = 0; i < h->n_sub; ++i) a.ys[i] = reinterpret_cast<uint8_t*>(ys[i]) + (size_t)m0 * h->sub_dout[i] * ybytes;
    if (h->multi) {
      a.adp_pairs = (uint32_t)h->r_pad / 128;
      for (int i = 0; i < kMaxTok; ++i) {
        const int id = (adapter_ids && m0 + i < m) ? adapter_ids[m0 + i] : -1;
        a.adp[i] = (id >= 0 && id < h->n_adapters) ? id : -1;
      }
    }
    cudaError_t e = launch_any(cfg, a, h->w.fmt, h->w.sz2 != 0, h->device);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace eora
