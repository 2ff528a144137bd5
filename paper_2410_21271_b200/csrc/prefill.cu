// Prefill kernel family (more than 32 tokens; fewer where decode_mid.cu does not take the layer): Y = X.deq(Wq) + (X.A).B
// (paper Eq. 4) as a tcgen05 GEMM.
//
// The paper measures only batch-1 decoding (Section 4.5); for many tokens the layer is a dense
// contraction, so it runs on the 5th-generation tensor cores.  The product is computed transposed,
// Yt[n][m] = sum_k w[n][k] X[m][k], so that the operand that has to be produced on chip is the small one:
//   * MMA "A" operand (128 rows): a tile of 128 output columns n of the weights.  Sixteen dequant warps
//     turn the packed tiles of the shared layout into fp16 RN((q - z) * s) in registers and store them in tensor memory (TM, see
//     tm_tile), or, where the accumulators fill that (256 rows x more than 160 tokens), as a K-major,
//     128-byte-swizzled operand tile in shared memory (bank-conflict-free stores);
//   * MMA "B" operand (up to 256 rows): a tile of tokens of X, K-major, brought in by TMA
//     (cp.async.bulk.tensor, 128-byte swizzle, no multicast) into the same ring of k-block stages as
//     the dequantised weight tile;
//   * an elected lane of one warp issues tcgen05.mma (M = 128, N = tokens, K = 16) with the fp32 accumulator in
//     tensor memory; tcgen05.commit releases the ring slots when the MMAs have drained;
//   * where whole tiles would leave SMs idle, a cluster of two to eight CTAs shares a tile's reduction axis and
//     adds its parts through distributed shared memory (pick_tilings chooses tile and cluster for both launches);
//   * the low-rank term is a K-extension: after the d_in/64 backbone k-blocks come r/64 k-blocks whose
//     token operand is t = X.A (fp16, from a first launch of the same kernel with A as the weight) and
//     whose weight operand is B, so (X.A).B lands in the same accumulator.  The two launches overlap:
//     the main one is a programmatic dependent launch that waits for t only in front of the K-extension;
//   * epilogue (all sixteen dequant warps): tcgen05.ld -> fp16/bf16/fp32 -> transpose through shared
//     memory -> 16-byte row stores, so Y is written once.
// Launches per forward: 1 (rank 0) or 2 (t = X.A, then the main product), plus a conversion launch
// when X is bf16 (the f16 MMA kind needs both operands in fp16; weights are kept fp16 because
// bf16 weights alone cost 1.7e-3 of the 2e-3 error budget).
#include <cuda.h>
#include "decode_common.cuh"
#include "tcgen05.cuh"

namespace eora {
using namespace dec;
namespace {

constexpr int BN_W = 128, BK = 64;               // weight rows per MMA (its M), k-block; a CTA owns up to two such halves
constexpr int kDqWarps = 16;                    // dequant warps (warps 4..19): one 16-row tile of the 256 weight rows each
constexpr int kThreadsP = (4 + kDqWarps) * 32;  // warp 0: TMA, warp 1: MMA, warp 2: TMEM alloc, warp 3: idle
constexpr int kMaxWStages = 6;                  // ring of k-block stages (token tile + dequantised weight tile)
constexpr int kSmallTile = 128;                // rows and tokens of the small tiles that fill a launch's last wave

struct PrefillArgs {
  WMat w;            // weight operand of the first nkb_w k-blocks (rows = output columns)
  WMat b;            // weight operand of the K-extension (FMT_NONE if none)
  void* out;         // [m][ld_out]
  int out_dtype;     // EORA_Y_*
  int ld_out;        // leading dimension of out (elements)
  int n_valid;       // columns of out to write
  int m;
  int bt;            // token tile (the MMA N): multiple of 16, at most 256
  int rows;          // weight rows per CTA: 256 (two MMA halves) or 128 (small matrices: more CTAs, half the dequant work each)
  // The grid is one-dimensional.  CTAs [0, n_small) take tiles of 128 rows x 128 tokens of the weight rows
  // [n_split, n_valid) (small_x row tiles per token tile); the others take tiles of rows x bt of the weight rows
  // [0, n_split) (big_x row tiles per token tile).  Without small tiles n_small = 0 and n_split = n_valid.
  int n_small, small_x, n_split, big_x;
  int nkb_w, nkb_b;  // k-blocks of each part
  int sw;            // stages of the ring (token tiles first, weight tiles from w_off on)
  int w_off, w_slot; // byte offset of the weight ring (after sw token tiles of bt*128 bytes), bytes of a weight tile (rows * 128)
  // Weights in tensor memory (TM): the warps' rings of packed weights start at w_off, w_slot bytes apart; columns of tensor memory from one 128-row
  // half's accumulator to the next; first column of the ring of weight tiles, columns of a stage (32 per half).
  int acc_cols, a_col0, a_cols;
  // Where the tiles leave SMs idle, the reduction axis of a tile is split over the ksplit CTAs of a cluster (the first one
  // also takes the K-extension; split_lo says which backbone k-blocks are whose).  The
  // partial accumulators meet in distributed shared memory: every CTA finishes every ksplit-th chunk of 32 tokens.
  // Fused layers (stacked along the weight rows): layer i owns rows [sub_row0[i], sub_row0[i + 1]),
  // writes to outs[i] (leading dimension sub_ld[i]) and takes columns [i * t_sub, (i + 1) * t_sub) of t in the
  // K-extension.  A plain layer: n_sub = 1, sub_row0 = {0, n_valid}, outs[0] = out.
  int n_sub;
  int sub_row0[5];
  void* outs[4];
  int sub_ld[4];
  int t_sub;
  int ksplit;
  int wait_x;          // X comes from the launch in front: wait for it before the first token tile (else only before t)
  int* dev_status;
  long long* trace;  // optional: for CTA (0,0), 4 clock64() stamps per k-block (token copy requested, W ready, X ready, MMA issued),
                     // then one more row: kernel entry, set-up done, accumulators complete, epilogue done
};

#define PTRACE(it, slot) do { if (p.trace && blockIdx.x == 0 && blockIdx.y == 0) p.trace[(it) * 4 + (slot)] = clock64(); } while (0)

struct PrefillState {
  __half* x16;       // fp16 copy of a bf16 X, [max_m][d_in] (bf16 handles only)
};

// First backbone k-block of split s: even shares of all k-blocks, the extension being part of the first; if the extension is more than
// a share, the others share the backbone.  (each_tiling sees to it that every split has some.)
__host__ __device__ __forceinline__ int split_lo(const PrefillArgs& p, int s) {
  if (s <= 0) return 0;
  if (s >= p.ksplit) return p.nkb_w;
  const int w = p.nkb_w / 2, b = p.nkb_b / 2, total = w + b;      // in pairs: a blob is not split
  return 2 * (b > total / p.ksplit ? (s - 1) * w / (p.ksplit - 1) : s * total / p.ksplit - b);
}

// k-blocks of a dequant warp's unit of work: a blob, or one tile where the blob has no scales (TM) or is 32 registers.
__host__ __device__ constexpr int unit_blocks(int fmt, bool tm) { return tm ? (fmt_quantised(fmt) ? 2 : 1) : fmt == FMT_F16 ? 1 : 2; }
// Two warps that share a row tile take its units alternately, and go on alternately from W's last unit to B's first: the first unit of B of the warp that
// began W with unit `phase`.  So no warp passes over more than one unit of the other, three k-blocks at most from one of its own to the next; a wait by
// parity cannot tell a stage's phase from the one two before, which a longer step than there are stages would ask of it.
__host__ __device__ constexpr int b_phase(int phase, int step, int units_w) { return step == 2 ? (units_w + phase) & 1 : 0; }

// ---------------------------------------------------------------------------------------------- PTX
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int c0, int c1, uint64_t* bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(smem_u32(dst)), "l"(tm), "r"(c0), "r"(c1), "r"(smem_u32(bar)) : "memory");
}
// The same with the 128-row operand in tensor memory: lane = row, one 32-bit column = two reduction elements.
__device__ __forceinline__ void umma_f16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// 16 lanes x 32 columns as fragments of 8 x 8 blocks (the inverse of tmem_ld16x32 below).
__device__ __forceinline__ void tmem_st16x32(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
               ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
                 "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
// 16 lanes x 32 columns as fragments of 8 x 8 blocks: registers 4 c .. 4 c + 3 hold columns 8 c + 2 (lane % 4) and the next one of
// lane lane / 4, then of lane lane / 4 + 8.
__device__ __forceinline__ void tmem_ld16x32(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                 "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
               : "r"(taddr));
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
               "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
                 "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
                 "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
                 "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
               : "r"(taddr) : "memory");
}

// packed tile payload of one lane, by format
template <int FMT> struct Packed;
template <> struct Packed<FMT_Q4> { uint4 v; };
template <> struct Packed<FMT_Q3> { uint2 v; uint32_t w2; };
template <> struct Packed<FMT_Q8> { uint4 v[2]; };
template <> struct Packed<FMT_F16> { uint4 v[4]; };
template <> struct Packed<FMT_SP24> { uint4 v[2]; uint32_t meta; };
template <> struct Packed<FMT_SQ4> { uint2 v; uint32_t meta; };

// Lanes with an odd row index g store the two 32-element halves of their rows in the opposite order
// (see dequant_store), so they take them in the opposite order too: where a half is a separate piece of
// the tile the swap is done here, by address (sw = 1 for such lanes); otherwise swap_halves does it on
// the loaded words, at the time they are used.
template <int FMT>
__device__ __forceinline__ void load_packed(Packed<FMT>& r, const uint8_t* blob, int lane, int sw) {
  if constexpr (FMT == FMT_Q4) r.v = __ldg(reinterpret_cast<const uint4*>(blob) + lane);
  else if constexpr (FMT == FMT_Q3) {
    r.v = __ldg(reinterpret_cast<const uint2*>(blob) + lane);
    r.w2 = __ldg(reinterpret_cast<const uint32_t*>(blob + 256) + lane);
  } else if constexpr (FMT == FMT_Q8) {
    r.v[0] = __ldg(reinterpret_cast<const uint4*>(blob + 512 * sw) + lane);
    r.v[1] = __ldg(reinterpret_cast<const uint4*>(blob + 512 * (sw ^ 1)) + lane);
  } else if constexpr (FMT == FMT_F16) {
#pragma unroll
    for (int p = 0; p < 4; ++p) r.v[p] = __ldg(reinterpret_cast<const uint4*>(blob + 512 * (p ^ (2 * sw))) + lane);
  } else if constexpr (FMT == FMT_SQ4) {
    r.v = __ldg(reinterpret_cast<const uint2*>(blob) + lane);
    r.meta = __ldg(reinterpret_cast<const uint32_t*>(blob + 256) + lane);
  } else {
    r.v[0] = __ldg(reinterpret_cast<const uint4*>(blob + 512 * sw) + lane);
    r.v[1] = __ldg(reinterpret_cast<const uint4*>(blob + 512 * (sw ^ 1)) + lane);
    r.meta = __ldg(reinterpret_cast<const uint32_t*>(blob + 1024) + lane);
  }
}
__device__ __forceinline__ void cswap(uint32_t& a, uint32_t& b, bool sw) {
  const uint32_t x = sw ? b : a, y = sw ? a : b;
  a = x; b = y;
}
// The value-level part of the swap (formats whose halves share a load; the position bytes of the 2:4 formats).
template <int FMT>
__device__ __forceinline__ void swap_halves(Packed<FMT>& r, bool sw) {
  if constexpr (FMT == FMT_Q4) { cswap(r.v.x, r.v.z, sw); cswap(r.v.y, r.v.w, sw); }
  else if constexpr (FMT == FMT_SQ4) { cswap(r.v.x, r.v.y, sw); r.meta = __funnelshift_l(r.meta, r.meta, sw ? 16 : 0); }
  else if constexpr (FMT == FMT_SP24) r.meta = __funnelshift_l(r.meta, r.meta, sw ? 16 : 0);
}

__device__ __forceinline__ uint32_t h2mul(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Byte offsets, inside one stage of the weight ring, of the four 16-byte chunks (8 consecutive reduction
// elements of one row each) that a lane stores per tile.  Store k holds row g + 8 * (k & 1) and the half
// (k >> 1) ^ (g & 1) of the 64 reduction elements: in step k lanes with even g write one half and lanes
// with odd g the other, so that the 8 lanes of a quarter warp (two rows) hit 8 different 16-byte columns
// of the 128-byte swizzle.
__device__ __forceinline__ void store_offsets(uint32_t (&off)[4], int tile, int lane) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int row = tile * 16 + g + 8 * (k & 1);
    const int chunk = (((k >> 1) ^ (g & 1)) << 2) + t;          // 16-byte chunk index along K inside the 128-byte row
    off[k] = (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4));
  }
}

// Per-tile constants (1024 + z), -(64 + z) as fp16x2 for the two rows of a lane, one byte permute each.
template <int FMT>
__device__ __forceinline__ void make_zc_p(ZC& zc, uint32_t zz) {
  zc.c[0][0] = prmt(zz, 0x64646464u, 0x4040u);
  zc.c[1][0] = prmt(zz, 0x64646464u, 0x4141u);
  if constexpr (FMT == FMT_Q4) {
    const uint32_t z4 = zz << 4;                                  // bytes: z_a << 4, z_b << 4 (zero-points < 16)
    zc.c[0][1] = prmt(z4, 0xD4D4D4D4u, 0x4040u);
    zc.c[1][1] = prmt(z4, 0xD4D4D4D4u, 0x4141u);
  }
}

// Dequantise one 16 x 64 tile to fp16 RN((q - z) * s) and store this lane's four chunks into the swizzled
// operand of the stage at shared address `stage`.  The lane's words arrive with their halves in storage
// order; `odd` (= g & 1) says that this lane stores them in the opposite order (store_offsets).
template <int FMT>
__device__ __forceinline__ void dequant_store(Packed<FMT> r, uint32_t sc2, uint32_t zz2, uint32_t stage, const uint32_t (&off)[4], bool odd,
                                              uint32_t lut) {
  swap_halves<FMT>(r, odd);
  uint32_t out[4][4];     // [part][pair]; part = 2 * (half as stored by this lane) + (row g or g + 8)
  if constexpr (FMT == FMT_F16) {
#pragma unroll
    for (int p = 0; p < 4; ++p) { out[p][0] = r.v[p].x; out[p][1] = r.v[p].y; out[p][2] = r.v[p].z; out[p][3] = r.v[p].w; }
  } else if constexpr (FMT == FMT_SP24 || FMT == FMT_SQ4) {
    // A quad's two kept values (one register) are spread over its four positions (two registers) with two byte
    // permutes.  Their selectors (sp24_selectors) are four bytes of 0x44, zero, with 0x10 at the first value's position and 0x32
    // at the second's: two shifts and one three-input xor.  From a table in shared memory, as in the decode kernels, they cost fewer
    // instructions, but the loads compete with the MMAs' operands (2:4 14336 x 4096, 2048 tokens: 242 -> 219 us without them).  4-bit
    // kept values, which need the issue slots more, take every other selector from the table (a block at 2048 tokens 905 -> 880 us,
    // at 64 tokens 133.5 against 134.3).
    const uint32_t at0[2] = {(r.meta << 3) & 0x18181818u, (r.meta >> 1) & 0x18181818u};      // 8 * position of the first value, even / odd quads
    const uint32_t at1[2] = {(r.meta << 1) & 0x18181818u, (r.meta >> 3) & 0x18181818u};      // of the second
    [[maybe_unused]] ZC zc;
    if constexpr (FMT == FMT_SQ4) make_zc_p<FMT>(zc, zz2);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      uint32_t vq[2];                                                         // (val0,val1) of quad 0, of quad 1
      if constexpr (FMT == FMT_SP24) {
        const uint4 u = r.v[p >> 1];
        vq[0] = (p & 1) ? u.z : u.x; vq[1] = (p & 1) ? u.w : u.y;
      } else {                                                                // kept codes -> RN((q - z) * s)
        const int hf = p & 1;
        const uint32_t w = (p >> 1) ? r.v.y : r.v.x;
        const uint32_t s2 = prmt(sc2, 0u, hf ? 0x3232u : 0x1010u);
        vq[0] = h2mul(h2sub(and_or(w >> (8 * hf), 0x000f000fu, kMagic), zc.c[hf][0]), s2);
        vq[1] = h2mul(h2sub(and_or(w >> (8 * hf + 4), 0x000f000fu, kMagic), zc.c[hf][0]), s2);
      }
#pragma unroll
      for (int quad = 0; quad < 2; ++quad) {
        uint32_t sel;
        if (FMT == FMT_SQ4 && quad == 1) {
          asm volatile("ld.shared.u32 %0, [%1];" : "=r"(sel) : "r"(lut + ((r.meta >> (8 * p + 2)) & 0x3Cu)));
        } else {                                                              // (shifts modulo 32: the bits above a byte's position are those of the bytes behind it)
          sel = 0x44444444u ^ __funnelshift_l(0u, 0x54u, at0[quad] >> (8 * p)) ^ __funnelshift_l(0u, 0x76u, at1[quad] >> (8 * p));
        }
        out[p][2 * quad] = prmt(vq[quad], 0u, sel);
        out[p][2 * quad + 1] = prmt(vq[quad], 0u, sel >> 16);
      }
    }
  } else {
    ZC zc;
    make_zc_p<FMT>(zc, zz2);
    uint32_t a[4][4];
    if constexpr (FMT == FMT_Q4) {
      const uint32_t w[4] = {r.v.x, r.v.y, r.v.z, r.v.w};
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        const int hf = part & 1;
        uint32_t lo = w[part], hi = w[part] >> 8;
        a[part][0] = h2sub(and_or(lo, 0x000f000fu, kMagic), zc.c[hf][0]);
        a[part][1] = h2fma(and_or(lo, 0x00f000f0u, kMagic), 0x2C002C00u, zc.c[hf][1]);
        a[part][2] = h2sub(and_or(hi, 0x000f000fu, kMagic), zc.c[hf][0]);
        a[part][3] = h2fma(and_or(hi, 0x00f000f0u, kMagic), 0x2C002C00u, zc.c[hf][1]);
      }
    } else if constexpr (FMT == FMT_Q3) {
      uint32_t q[4][2];
      q3_quads(r.v.x, r.v.y, r.w2, q);
#pragma unroll
      for (int j = 0; j < 2; ++j) { cswap(q[0][j], q[2][j], odd); cswap(q[1][j], q[3][j], odd); }
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        const int hf = part & 1;
#pragma unroll
        for (int j = 0; j < 4; ++j) a[part][j] = h2sub(quad_pair(q[part][j >> 1], j & 1), zc.c[hf][0]);
      }
    } else {   // FMT_Q8
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        const int hf = part & 1;
        const uint4 u = r.v[part >> 1];
        const uint32_t w0 = hf ? u.z : u.x, w1 = hf ? u.w : u.y;
        a[part][0] = h2sub(and_or(w0, 0x00ff00ffu, kMagic), zc.c[hf][0]);
        a[part][1] = h2sub(and_or(w0 >> 8, 0x00ff00ffu, kMagic), zc.c[hf][0]);
        a[part][2] = h2sub(and_or(w1, 0x00ff00ffu, kMagic), zc.c[hf][0]);
        a[part][3] = h2sub(and_or(w1 >> 8, 0x00ff00ffu, kMagic), zc.c[hf][0]);
      }
    }
    const uint32_t s_a = prmt(sc2, 0u, 0x1010u), s_b = prmt(sc2, 0u, 0x3232u);
#pragma unroll
    for (int part = 0; part < 4; ++part)
#pragma unroll
      for (int j = 0; j < 4; ++j) out[part][j] = h2mul(a[part][j], (part & 1) ? s_b : s_a);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int part = (k >> 1) * 2 + (k & 1);
    st_shared_v4(stage + off[k], out[part][0], out[part][1], out[part][2], out[part][3]);
  }
}

// One part (W or the K-extension B) of a dequant warp's work.  The warp owns row tile `tile` (0..15) of
// the CTA's 256 weight rows; k-blocks [kb_lo, kb_hi) of `mat` (both even) land in pipeline iterations it0, it0 + 1, ...
// A unit of work is a blob (two k-blocks, one set of scales) or, for fp16 weights, whose blob is 32 registers, one k-block;
// the warp takes units phase, phase + step, ... (step = 2 when two warps share a row tile, which is how a CTA with 128 rows
// keeps all sixteen warps and twice the loads in flight).  Units are loaded PF of the warp's own ahead.  The loop is what bounds
// the kernel (four of these warps share a scheduler), so everything that does not change per k-block is computed once per
// blob or once altogether: constants from scales and zero-points, running addresses, the ring position as a (slot, wrap) pair.
template <int FMT>
__device__ __forceinline__ bool dequant_part(const WMat& mat, int n0, int kb_lo, int kb_hi, int it0, int tile, int phase,
                                             int step, int lane, uint8_t* smem, const PrefillArgs& p, uint64_t* full_w,
                                             uint64_t* empty_w, uint32_t lut) {
  if constexpr (FMT == FMT_NONE) {
    return true;
  } else {
    constexpr int U = unit_blocks(FMT, false), PF = FMT == FMT_F16 ? 3 : 2;
    constexpr bool quant = fmt_quantised(FMT);
    constexpr int tb = tile_bytes(FMT);
    const int rt = (n0 >> 4) + tile;                     // this warp's row tile of the matrix
    const bool active = rt < mat.nt;
    const int g = lane >> 2;
    const int odd = g & 1;
    uint32_t off[4];
    store_offsets(off, tile, lane);
    const uint32_t ring = smem_u32(smem + p.w_off), full0 = smem_u32(full_w), empty0 = smem_u32(empty_w);
    const int u_hi = kb_hi / U;                          // units [kb_lo / U + phase, u_hi), every step-th
    int u_next = kb_lo / U + phase;                      // the next unit to load, and where it is
    const uint8_t* next = wmat_blob(mat, rt, u_next * U / 2) + (U == 1 ? (u_next & 1) * tb : 0);
    const int64_t to_second = wmat_blob(mat, rt, mat.half) - (wmat_blob(mat, rt, 0) + (int64_t)mat.half * mat.blob);   // what the second half of the pairs is further
    const int half_u = u_next * U / 2 < mat.half ? 2 * mat.half / U : 0x7fffffff;      // the unit that the second half begins with, if it is ahead
    const bool two = mat.sz2 != 0;
    Packed<FMT> pk[PF][U];
    uint32_t scq[PF][U], zzq[PF][U];
    bool crossed = false;
    auto issue = [&](int slot) {
      if (!active || u_next >= u_hi) return;
      if (!crossed && u_next >= half_u) { next += to_second; crossed = true; }
#pragma unroll
      for (int c = 0; c < U; ++c) load_packed<FMT>(pk[slot][c], next + c * tb, lane, odd);
      if constexpr (quant) {
        const uint8_t* sz = next + 2 * tb + 4 * g;
        scq[slot][0] = __ldg(reinterpret_cast<const uint32_t*>(sz));
        zzq[slot][0] = __ldg(reinterpret_cast<const uint16_t*>(sz + 32 - 2 * g));
        if (two) {
          scq[slot][U - 1] = __ldg(reinterpret_cast<const uint32_t*>(sz + kSzEntryBytes));
          zzq[slot][U - 1] = __ldg(reinterpret_cast<const uint16_t*>(sz + kSzEntryBytes + 32 - 2 * g));
        }
      }
      u_next += step;
      next += U == 1 ? (step == 2 ? mat.blob : (u_next & 1) ? tb : mat.blob - tb) : step * mat.blob;
    };
#pragma unroll
    for (int j = 0; j < PF; ++j) issue(j);
    int it = it0 + phase * U;
    int s = it % p.sw, wrap = it / p.sw;                 // ring slot of iteration `it`, and how often it has been used before
    auto advance = [&](int by) {                         // by <= 3 <= stages (b_phase: across the seam too)
      it += by;
      s += by;
      if (s >= p.sw) { s -= p.sw; ++wrap; }
    };
    for (int ub = kb_lo / U + phase; ub < u_hi; ub += PF * step) {
#pragma unroll
      for (int j = 0; j < PF; ++j) {
        if (ub + j * step < u_hi) {
#pragma unroll
          for (int c = 0; c < U; ++c) {
            if (wrap > 0 && !__all_sync(0xffffffffu, mbar_try_wait_a(empty0 + 8 * s, (wrap - 1) & 1)) &&
                !mbar_wait_warp(empty_w + s, (wrap - 1) & 1, p.dev_status, lane)) return false;
            const uint32_t stage = ring + (uint32_t)s * p.w_slot;
            if (active) {
              const bool own = U == 2 && c == 1 && two;
              dequant_store<FMT>(pk[j][c], own ? scq[j][U - 1] : scq[j][0], own ? zzq[j][U - 1] : zzq[j][0], stage, off, odd != 0, lut);
            } else {                                      // rows past the matrix: keep the operand finite
#pragma unroll
              for (int k = 0; k < 4; ++k) st_shared_v4(stage + off[k], 0u, 0u, 0u, 0u);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> visible to the MMA
            __syncwarp();
            if (lane == 0) {
              asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(full0 + 8 * s) : "memory");
              if (tile == 0) PTRACE(it, 1);
            }
            if (c + 1 < U) advance(1);
          }
          issue(j);
          advance(step * U - U + 1);
        }
      }
    }
    return true;
  }
}

// ---------------------------------------------------------------------------------------------- weights in tensor memory
// Up to 160 tokens (256 with 128 rows) the accumulators leave tensor memory for the dequantised weights.  Through shared memory a k-block of 256 rows x
// 64 tokens moved 32 KB of weights in and out of it, 512 cycles of its bandwidth, and each hand-over waited for the stores to become visible to the
// MMAs (1215 cycles a k-block); here the weights go from registers to tensor memory and the MMAs read only the tokens from shared memory (790).  A 4-bit
// LLaMA3-8B block of 64 tokens with 8-bit adapters of rank 512: 139 -> 114 us; of 128 tokens, rank 128, 124 -> 105; of a prompt of 333 238 -> 218.
// Tried and not kept: two chains of MMAs with accumulators of their own (128 rows 515 -> 562 cycles).
//
// tcgen05.st writes a tile of 16 rows x 64 reduction elements as fragments of 8 x 8 32-bit blocks: lane (g, t) holds, for each of the four MMAs j of a
// k-block, elements 16 j + 4 t .. + 3 of rows g and g + 8.  In the packed layout these are half (t & 1) of the eight codes that
// lane (g, 2 (j & 1) + (t >> 1)) owns of the 32-element block j / 2.  So every warp brings its blobs to shared memory (a ring of its own;
// the first of W are asked for as soon as the barriers and tensor memory are set up, those of B behind all of W) and its lanes read the words of those two lanes.
// out[4 j + 2 hf + i]: elements 16 j + 4 t + 2 i, + 1 of row g + 8 hf, as fp16 RN((q - z) * s).
template <int FMT>
__device__ __forceinline__ void tm_tile(uint32_t tile, int lane, const ZC& zc, uint32_t s_a, uint32_t s_b, uint32_t (&out)[16]) {
  const int g = lane >> 2, t = lane & 3, half = t & 1;
  const uint32_t at = (uint32_t)(g * 4 + (t >> 1));  // lane of the packed layout for even j; two further for odd j
  auto put = [&](int j, int hf, uint32_t a, uint32_t b) {
    out[4 * j + 2 * hf] = h2mul(a, hf ? s_b : s_a); out[4 * j + 2 * hf + 1] = h2mul(b, hf ? s_b : s_a);
  };
  if constexpr (FMT == FMT_Q4) {
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
      const uint4 u = lds_u4(tile + (at + 2 * jj) * 16);
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        const int hf = part & 1;
        const uint32_t v = w[part] >> (8 * half);
        put(2 * (part >> 1) + jj, hf, h2sub(and_or(v, 0x000f000fu, kMagic), zc.c[hf][0]), h2fma(and_or(v, 0x00f000f0u, kMagic), 0x2C002C00u, zc.c[hf][1]));
      }
    }
  } else if constexpr (FMT == FMT_Q3) {
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
      const uint2 u = lds_u2(tile + (at + 2 * jj) * 8);
      const uint32_t w2 = lds_u1(tile + 256 + (at + 2 * jj) * 4), w[3] = {u.x, u.y, w2};
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        const int hf = part & 1;
        const uint32_t q = part < 3 ? (w[part < 3 ? part : 0] >> (3 * half)) & 0x07070707u
                                    : and_or(w2 >> (4 + half), 0x04040404u, ((half ? u.y : u.x) >> 6) & 0x03030303u);
        put(2 * (part >> 1) + jj, hf, h2sub(quad_pair(q, 0), zc.c[hf][0]), h2sub(quad_pair(q, 1), zc.c[hf][0]));
      }
    }
  } else if constexpr (FMT == FMT_Q8) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const uint32_t w = lds_u1(tile + (j >> 1) * 512 + (at + 2 * (j & 1)) * 16 + hf * 8 + half * 4);
        put(j, hf, h2sub(and_or(w, 0x00ff00ffu, kMagic), zc.c[hf][0]), h2sub(and_or(w >> 8, 0x00ff00ffu, kMagic), zc.c[hf][0]));
      }
  } else if constexpr (FMT == FMT_F16) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const uint2 w = lds_u2(tile + (2 * (j >> 1) + hf) * 512 + (at + 2 * (j & 1)) * 16 + half * 8);
        out[4 * j + 2 * hf] = w.x; out[4 * j + 2 * hf + 1] = w.y;
      }
  } else {                                           // 2:4 formats: the quad `half` of each part (selectors as in dequant_store)
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
      const uint32_t meta = lds_u1(tile + (FMT == FMT_SP24 ? 1024 : 256) + (at + 2 * jj) * 4) >> (4 * half);
      const uint32_t at0 = (meta << 3) & 0x18181818u, at1 = (meta << 1) & 0x18181818u;
      uint2 u = make_uint2(0u, 0u);
      if constexpr (FMT == FMT_SQ4) { u = lds_u2(tile + (at + 2 * jj) * 8); u.x >>= 4 * half; u.y >>= 4 * half; }
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        const int hf = part & 1, j = 2 * (part >> 1) + jj;
        uint32_t v;
        if constexpr (FMT == FMT_SP24) v = lds_u1(tile + (part >> 1) * 512 + (at + 2 * jj) * 16 + hf * 8 + half * 4);
        else v = h2mul(h2sub(and_or(((part >> 1) ? u.y : u.x) >> (8 * hf), 0x000f000fu, kMagic), zc.c[hf][0]), hf ? s_b : s_a);
        const uint32_t sel = 0x44444444u ^ __funnelshift_l(0u, 0x54u, at0 >> (8 * part)) ^ __funnelshift_l(0u, 0x76u, at1 >> (8 * part));
        out[4 * j + 2 * hf] = prmt(v, 0u, sel); out[4 * j + 2 * hf + 1] = prmt(v, 0u, sel >> 16);
      }
    }
  }
}

// Weights to shared memory, 16 bytes a lane and instruction; a group per slot of a ring.
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All but the PENDING newest groups have landed, for every lane of the warp.
template <int PENDING>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
  __syncwarp();
}
// BYTES (a multiple of 16) by a warp.
template <int BYTES>
__device__ __forceinline__ void cp_block(uint32_t dst, const uint8_t* src, int lane) {
#pragma unroll
  for (int o = 0; o < BYTES; o += 512)
    if (o + 512 <= BYTES || o + lane * 16 < BYTES) cp16(dst + o + lane * 16, src + o + lane * 16);
}

// A warp's ring of packed weights: slots of one unit (a blob, or one tile where there are no scales), one group of copies each.
__host__ __device__ constexpr int tm_unit_most(int fmt) { return fmt == FMT_NONE ? 0 : fmt_quantised(fmt) ? blob_bytes(fmt, 1) : tile_bytes(fmt); }
__host__ __device__ constexpr int tm_slots(int fmt) { return tm_unit_most(fmt) <= 1536 ? 4 : 2; }      // (16 warps: 68 KB of 4-bit weights, 64 KB of fp16 in flight)
__host__ __device__ constexpr int tm_ring(int fmt) { return tm_slots(fmt) * tm_unit_most(fmt); }

// The counterpart of dequant_part: the same units, in the same order.  `tile`: row tile of the CTA's 256 weight rows.  ring: the warp's ring.  The loop
// is bound by its instructions (130 a tile took 907 cycles per k-block of 256 rows, of which the arithmetic is 150), so it carries nothing that could be
// worked out before.
template <int FMT>
__device__ __forceinline__ bool dequant_part_tm(const WMat& mat, int n0, int kb_lo, int kb_hi, int it0, int tile, int phase, int step, int lane,
                                                const PrefillArgs& p, uint32_t ring, uint32_t tmem_a, uint64_t* full_w, uint64_t* empty_w) {
  if constexpr (FMT == FMT_NONE) {
    return true;
  } else {
    constexpr int U = unit_blocks(FMT, true), D = tm_slots(FMT), tb = tile_bytes(FMT);
    constexpr bool quant = fmt_quantised(FMT);
    constexpr int kUnit = quant ? blob_bytes(FMT, 0) : tb;
    const int rt = (n0 >> 4) + tile;
    const bool active = rt < mat.nt;                     // (else: rows past the matrix, zeros keep the operand finite)
    const bool two = quant && mat.sz2 != 0;
    const uint32_t unit_b = quant ? (uint32_t)mat.blob : (uint32_t)tb, ring_b = D * unit_b;
    const int u_lo = kb_lo / U + phase, u_hi = kb_hi / U;
    // the next unit to ask for, and where it is; where the second half of the pairs begins, it is elsewhere
    int u_next = active ? u_lo : u_hi;
    const uint8_t* next = wmat_blob(mat, rt, u_next * U / 2) + (U == 1 ? (u_next & 1) * tb : 0);
    const int64_t to_second = wmat_blob(mat, rt, mat.half) - (wmat_blob(mat, rt, 0) + (int64_t)mat.half * mat.blob);
    int cross = u_next * U / 2 < mat.half ? 2 * mat.half / U : 0x7fffffff;
    const int stride = U == 1 ? (step == 2 ? mat.blob : tb) : step * mat.blob;      // (two tiles of an unquantised blob are contiguous, and so are its blobs)
    auto ask = [&](uint32_t to) {
      if (u_next < u_hi) {
        if (u_next >= cross) { next += to_second; cross = 0x7fffffff; }
        cp_block<kUnit>(to, next, lane);
        if (two && lane < kSzEntryBytes / 16) cp16(to + kUnit + lane * 16, next + kUnit + lane * 16);
        u_next += step;
        next += stride;
      }
      cp_commit();                                       // (also if there is nothing left: the count of groups stays in step)
    };
#pragma unroll 1
    for (uint32_t o = 0; o < ring_b; o += unit_b) ask(ring + o);
    const uint32_t sz_at = 2 * tb + 4 * (lane >> 2), zz_at = 2 * tb + 32 + 2 * (lane >> 2);
    const int stages = p.sw;
    const uint32_t cols = p.a_cols;
    int s = (it0 + phase * U) % stages;
    uint32_t ph = (uint32_t)((it0 + phase * U) / stages) & 1u;
    uint32_t full = smem_u32(full_w) + 8 * s, empty = smem_u32(empty_w) + 8 * s, at = tmem_a + s * cols;      // of stage s
    auto advance = [&](int by) {
      s += by; full += 8 * by; empty += 8 * by; at += by * cols;
      if (s >= stages) { s -= stages; full -= 8 * stages; empty -= 8 * stages; at -= stages * cols; ph ^= 1u; }
    };
    const bool traced = p.trace && blockIdx.x == 0 && tile == 0 && lane == 0;
    int it = it0 + phase * U;
    // A tile is handed over when the next one has been dequantised: by then its way to tensor memory, some hundred cycles, is over.
    uint32_t sent = 0;                                   // its stage's barrier, 0: none
    auto hand_over = [&]() {
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0 && sent) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sent) : "memory");
    };
    uint32_t so = 0;                                     // slot of the unit
    bool ok = true;
#pragma unroll 1
    for (int u = u_lo; u < u_hi; u += step) {
      cp_wait<D - 1>();
      const uint32_t src = ring + so;
      ZC zc;
      uint32_t s_a = 0u, s_b = 0u;
#pragma unroll
      for (int c = 0; c < U; ++c) {
        uint32_t out[16];
        if (active) {
          if constexpr (quant) {
            if (c == 0 || two) {
              const uint32_t sc2 = lds_u1(src + sz_at + (c ? kSzEntryBytes : 0)), zz = lds_u16(src + zz_at + (c ? kSzEntryBytes : 0));
              s_a = prmt(sc2, 0u, 0x1010u); s_b = prmt(sc2, 0u, 0x3232u);
              make_zc_p<FMT>(zc, zz);
            }
          }
          tm_tile<FMT>(src + c * tb, lane, zc, s_a, s_b, out);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) out[i] = 0u;
        }
        hand_over();
        if (!__all_sync(0xffffffffu, mbar_try_wait_a(empty, ph ^ 1u)) && !mbar_wait_warp_fast(empty_w + s, ph ^ 1u, p.dev_status, lane)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_st16x32(at, out);
        sent = full;
        if (traced) p.trace[it * 4 + 1] = clock64();
        it += c + 1 < U ? 1 : step * U - U + 1;
        advance(c + 1 < U ? 1 : step * U - U + 1);       // (by at most 3 <= stages; b_phase: across the seam too)
      }
      if (!ok) break;
      __syncwarp();                                      // every lane has read the slot
      ask(src);
      so += unit_b;
      if (so == ring_b) so = 0;
    }
    if (ok) hand_over();
    else cp_wait<0>();                                   // gave up: what is in flight lands first
    return ok;
  }
}

// TM: the dequantised weights go to tensor memory instead of shared memory.
template <int WF, int BF, bool TM>
__global__ void __launch_bounds__(kThreadsP, 1) k_prefill(const __grid_constant__ CUtensorMap tm_x,
                                                          const __grid_constant__ CUtensorMap tm_t,
                                                          const __grid_constant__ CUtensorMap tm_x_small,
                                                          const __grid_constant__ CUtensorMap tm_t_small, const PrefillArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // One ring for both operands: stage s holds the token tile and the dequantised weight tile of a k-block, full_w[s]
  // collects the copy's bytes and the dequant warps' arrivals, empty_w[s] one commit: one wait and one commit per k-block for
  // the warp that issues the MMAs.
  __shared__ __align__(8) uint64_t full_w[kMaxWStages], empty_w[kMaxWStages], acc_full;
  __shared__ uint32_t tmem_base_s;
  __shared__ uint32_t sp_lut[16];        // 2:4 expansion selectors (2:4 backbones of 4-bit codes only)
  __shared__ int fail_s;                 // set by an epilogue warp whose bounded wait ran out
  // 1024-byte alignment of the operand tiles (the swizzle pattern is anchored at 1 KB)
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

  // Programmatic dependent launch: a kernel launched behind this one with the serialisation attribute may start early.  A launch
  // that waits for X lets it go only after that wait: the main product behind the launch that computes t starts
  // without waiting for anything, and reads the same X.
  if (!p.wait_x) asm volatile("griddepcontrol.launch_dependents;");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool small = (int)blockIdx.x < p.n_small;
  const int big_id = (int)blockIdx.x - p.n_small;
  const int bt = small ? kSmallTile : p.bt;                 // tokens of this CTA's tile (the MMA N)
  const int rows = small ? kSmallTile : p.rows;
  // big tiles: the split of the reduction axis fastest (a cluster), then the row tile, then the token tile
  const int tile = big_id / p.ksplit, split = small ? 0 : big_id - tile * p.ksplit;
  const int tile_x = tile % p.big_x, tile_y = tile / p.big_x;
  const int n0 = small ? p.n_split + ((int)blockIdx.x % p.small_x) * kSmallTile : tile_x * rows;
  const int m0 = small ? ((int)blockIdx.x / p.small_x) * kSmallTile : tile_y * bt;
  int sub = 0;                                              // fused layers: whose rows these are (tiles never straddle)
#pragma unroll
  for (int i = 1; i < 4; ++i)
    if (i < p.n_sub && n0 >= p.sub_row0[i]) sub = i;
  const int n_end = min(small ? p.n_valid : p.n_split, p.sub_row0[sub + 1]);   // this CTA writes columns n0 .. n_end - 1 at most
  void* const out_p = p.outs[sub];
  const int ld_o = p.sub_ld[sub], col0 = p.sub_row0[sub];   // output column of weight row n: n - col0
  const int nh = (rows > BN_W && n_end - n0 > BN_W) ? 2 : 1;   // 128-row halves of this CTA that hold real rows
  const CUtensorMap* map_x = small ? &tm_x_small : &tm_x;
  const CUtensorMap* map_t = small ? &tm_t_small : &tm_t;
  const int kw_lo = split_lo(p, split), kw_hi = split_lo(p, split + 1);
  const int nkw = kw_hi - kw_lo;
  const int nkb_ext = split == 0 ? p.nkb_b : 0;             // the K-extension goes with the first split
  const int nkb = nkw + nkb_ext;
  const uint32_t xbytes = (uint32_t)bt * 128;               // bytes of a token tile; the ring's slots are p.bt * 128 apart
  const uint32_t xslot = (uint32_t)p.bt * 128;

  if constexpr (WF == FMT_SQ4 && !TM) {
    if (threadIdx.x >= 32 && threadIdx.x < 48) sp_lut[threadIdx.x - 32] = sp24_selectors(threadIdx.x - 32);
  }
  const uint32_t lut = smem_u32(sp_lut);
  if (threadIdx.x == 96) {                                  // (their first use would pay for a trip to L2)
    asm volatile("prefetch.tensormap [%0];" ::"l"(map_x) : "memory");
    if (nkb_ext > 0) asm volatile("prefetch.tensormap [%0];" ::"l"(map_t) : "memory");
  }
  if (threadIdx.x == 0) {
    PTRACE(nkb, 0);
    fail_s = 0;
    for (int i = 0; i < p.sw; ++i) { mbar_init(full_w + i, 8 * nh + 1); mbar_init(empty_w + i, 1); }
    mbar_init(&acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {   // tensor memory: two accumulators of 128 lanes x 256 fp32 columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = tmem_base_s;
  if (threadIdx.x == 0) PTRACE(nkb, 1);

  if constexpr (TM && BF != FMT_NONE) {                     // the CTA's blobs of B towards L2: they are needed at once, at the end
    if (warp == 3 && nkb_ext > 0) {
      const int t_lo = n0 >> 4, t_n = min(8 * nh, p.b.nt - t_lo);
      const uint8_t* src = wmat_blob(p.b, t_lo, 0);
      const int64_t bytes = (int64_t)t_n * p.b.np * p.b.blob;
      for (int64_t o = (int64_t)lane << 13; o < bytes; o += 32 << 13) prefetch_l2(src + o, (uint32_t)(bytes - o < 8192 ? bytes - o : 8192));
    }
  }
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (token tiles)
    if (lane == 0) {
      if (p.wait_x) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;");
      }
      int s = 0, wrap = 0;                          // ring slot of iteration `it`, and how often it has been used before
      for (int it = 0; it < nkb; ++it) {
        if (wrap > 0 && !mbar_wait(empty_w + s, (wrap - 1) & 1, p.dev_status)) break;
        PTRACE(it, 0);
        mbar_expect_tx(full_w + s, xbytes);
        uint8_t* xt = smem + (size_t)s * xslot;
        if (it < nkw) {
          tma_load_2d(xt, map_x, (kw_lo + it) * BK, m0, full_w + s);
        } else {
          // t comes from the previous launch, which may still be running: everything up to here overlapped with it
          if (it == nkw && !p.wait_x) asm volatile("griddepcontrol.wait;" ::: "memory");
          tma_load_2d(xt, map_t, (it - nkw) * BK + sub * p.t_sub, m0, full_w + s);
        }
        if (++s == p.sw) { s = 0; ++wrap; }
      }
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == 1) {      // (warp-uniform for the compiler)
    // ------------------------------------------------------------------ MMA issuer
    // The whole warp walks through the loop and one elected lane issues: descriptors and addresses are then warp-uniform values
    // that stay in uniform registers.  Inside an `if (lane == 0)` every operand of every MMA was moved there first, ~90 cycles
    // per MMA, which bounded a k-block of 256 rows at 1050 cycles whatever the tokens.
    // instruction descriptor: fp32 accumulate, fp16 x fp16, both operands K-major, M = 128 weight rows, N = bt tokens
    const uint32_t idesc = (1u << 4) | ((uint32_t)(bt >> 3) << 17) | ((uint32_t)(BN_W >> 4) << 24);
    const bool elected = elect_one();
    const uint64_t bdesc0 = make_desc<128>(smem_u32(smem)), adesc0 = make_desc<128>(smem_u32(smem + p.w_off));
    const uint32_t bstep = xslot >> 4, astep = (uint32_t)p.w_slot >> 4;       // from one ring slot to the next, in 16-byte units
    const uint32_t full0 = smem_u32(full_w), empty0 = smem_u32(empty_w);
    bool ok = true;
    uint32_t sw = 0, pw = 0;                        // ring slot of iteration `it` and its phase
    for (int it = 0; it < nkb; ++it) {
      // token tile copied and weight tile dequantised?
      if (!mbar_try_wait_a(full0 + 8 * sw, pw)) ok = mbar_wait(full_w + sw, pw, p.dev_status);
      if (!__all_sync(0xffffffffu, ok)) break;
      if (elected) PTRACE(it, 2);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t bdesc = bdesc0 + sw * bstep, adesc = adesc0 + sw * astep;
      if (elected) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          // half j / 4 of the weight rows is 128 rows = 16 KB further (+1024 in the address field), each K step of
          // 16 fp16 is 32 bytes further (+2)
          if (j < 4 * nh)
            if constexpr (TM)                           // (16 reduction elements are 8 columns)
              umma_f16_ts(tmem_d + (j >> 2) * p.acc_cols, tmem_d + p.a_col0 + sw * p.a_cols + (j >> 2) * 32 + 8 * (j & 3), bdesc + 2 * (j & 3),
                          idesc, (it > 0 || (j & 3) > 0) ? 1u : 0u);
            else
              umma_f16(tmem_d + (j >> 2) * 256, adesc + (uint64_t)((j >> 2) * ((BN_W * 128) >> 4) + 2 * (j & 3)), bdesc + 2 * (j & 3),
                       idesc, (it > 0 || (j & 3) > 0) ? 1u : 0u);
        }
        umma_commit_a(empty0 + 8 * sw);             // arrives when these MMAs have finished reading their operands
        PTRACE(it, 3);
      }
      if (++sw == (uint32_t)p.sw) { sw = 0; pw ^= 1u; }
    }
    if (elected) umma_commit(&acc_full);            // arrives when every MMA above has completed
    __syncwarp();
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ dequant warps, then epilogue
    const int dw = warp - 4;
    bool ok = true;
    if constexpr (TM) {
      // A warp writes to the quarter of the lanes that its number selects: row tiles 2 (warp % 4) and the next one of each half.  Two halves: one
      // row tile per warp; one half: two warps per row tile, alternating units.
      const int q = dw >> 2, kstep = 3 - nh, kphase = nh == 2 ? 0 : q >> 1;
      const int in_half = 2 * (dw & 3) + (q & 1), hh = nh == 2 ? q >> 1 : 0, tile = hh * 8 + in_half;
      const uint32_t ring = smem_u32(smem + p.w_off) + (uint32_t)(dw * p.w_slot);
      const uint32_t tmem_a = tmem_d + ((uint32_t)(in_half * 16) << 16) + p.a_col0 + hh * 32;
      ok = dequant_part_tm<WF>(p.w, n0, kw_lo, kw_hi, 0, tile, kphase, kstep, lane, p, ring, tmem_a, full_w, empty_w);
      if (ok && nkb_ext > 0)
        ok = dequant_part_tm<BF>(p.b, n0, 0, nkb_ext, nkw, tile, b_phase(kphase, kstep, nkw / unit_blocks(WF, true)), kstep, lane, p, ring, tmem_a, full_w, empty_w);
    } else {
      // two halves: one row tile per warp; one half: two warps per row tile, alternating k-blocks
      const int kstep = 3 - nh, tile = nh == 2 ? dw : (dw & 7), kphase = nh == 2 ? 0 : (dw >> 3);
      ok = dequant_part<WF>(p.w, n0, kw_lo, kw_hi, 0, tile, kphase, kstep, lane, smem, p, full_w, empty_w, lut);
      if (ok && nkb_ext > 0)
        ok = dequant_part<BF>(p.b, n0, 0, nkb_ext, nkw, tile, b_phase(kphase, kstep, nkw / unit_blocks(WF, false)), kstep, lane, smem, p, full_w, empty_w, lut);
    }
    if (ok) ok = mbar_wait_warp(&acc_full, 0, p.dev_status, lane);
    // the warps meet at barriers below: they must all take the same way
    if (!ok) *reinterpret_cast<volatile int*>(&fail_s) = 1;
    asm volatile("bar.sync 1, 512;" ::: "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (dw == 0 && lane == 0) PTRACE(nkb, 2);
  }

  // Epilogue: all sixteen dequant warps, as four groups of four.  A warp can read the quarter of the TMEM lanes that its index
  // selects (warp % 4), i.e. accumulator rows (= weight rows n) 32 * (warp % 4) ... of each half; columns are tokens.  The
  // accumulator goes out in units of 32 tokens x 128 rows, dealt round-robin to the CTAs of the cluster and to the groups.
  const int dw = warp - 4, grp = dw >> 2, lq = warp & 3;
  const int nl = lq * 32 + lane;                         // local weight row inside the half = thread index inside the group
  const int nchunk = (bt + 31) >> 5, units = nh * nchunk;
  const uint32_t lane_base = tmem_d + ((uint32_t)(lq * 32) << 16);
  const uint32_t acc_cols = TM ? (uint32_t)p.acc_cols : 256u;
  const uint32_t parts = smem_u32(smem) + 65536;         // split: the other CTAs' shares of this CTA's units, 16 KB each
  const bool out16 = p.out_dtype != EORA_Y_F32;
  // A unit's accumulators: for a 16-bit Y as fragments of 8 x 8 blocks, for a float Y one row of W per lane (32 tokens).
  auto load_unit = [&](uint32_t taddr, uint32_t (&v)[32]) {
    if (out16) {
      tmem_ld16x32(taddr, v);
      tmem_ld16x32(taddr + (16u << 16), v + 16);
    } else {
      tmem_ld32(taddr, v);
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  };
  if (p.ksplit > 1) {
    __syncwarp();
    cluster_arrive(); cluster_wait();                    // every CTA's MMAs have completed: the rings are free everywhere
    const bool live = warp >= 4 && *reinterpret_cast<volatile int*>(&fail_s) == 0;
    for (int u = grp; live && u < units; u += 4) {
      const int owner = u % p.ksplit;
      if (owner == split) continue;
      const int hh = u / nchunk, c0 = (u - hh * nchunk) * 32;
      uint32_t v[32];
      load_unit(lane_base + hh * acc_cols + (uint32_t)c0, v);
      const int slot = (u / p.ksplit) * (p.ksplit - 1) + (split < owner ? split : split - 1);
      const uint32_t to = mapa(parts + slot * 16384 + nl * 16, (uint32_t)owner);      // (the same thread of the owner adds it to the same registers)
#pragma unroll
      for (int j = 0; j < 32; j += 4)
        asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to + j * 512), "r"(v[j]), "r"(v[j + 1]), "r"(v[j + 2]), "r"(v[j + 3]) : "memory");
    }
    __syncwarp();
    cluster_arrive(); cluster_wait();
  }
  if (warp >= 4 && *reinterpret_cast<volatile int*>(&fail_s) == 0) {
    // A unit goes through shared memory as [32 tokens][128 n] so that the global stores are 16-byte pieces of rows of Y: a 16-bit
    // Y by transposing stores of 8 x 8 blocks, rows 16 bytes apart modulo the banks; a float Y word by word.  (Storing it element
    // by element, the type decided at each, took 7400 of the 10700 cycles of a 256 x 256 tile; the stores to Y take 1000.)
    // Without a split each group has two buffers of 16 KB (a 32 x 128 block of floats) and alternates: a buffer is rewritten two
    // units later, after a barrier that every thread of the group passes only when it has read the buffer out, so one barrier
    // per unit is enough.  With a split it has one buffer and takes two barriers.
    const uint32_t gbuf = smem_u32(smem) + grp * (p.ksplit > 1 ? 16384 : 32768);
    const uint32_t pitch = out16 ? 272 : 512;            // bytes from one token's row in the buffer to the next
    const int esz = out16 ? 2 : 4, row_sh = out16 ? 4 : 5;      // log2 of the 16-byte pieces per token row (128 n)
    int flip = 0;
    for (int i = grp; i * p.ksplit + split < units; i += 4) {
      const int u = i * p.ksplit + split, hh = u / nchunk, c0 = (u - hh * nchunk) * 32;
      const uint32_t tbuf = gbuf + flip * 16384;
      if (p.ksplit == 1) flip ^= 1;
      uint32_t v[32];
      load_unit(lane_base + hh * acc_cols + (uint32_t)c0, v);
      for (int q = 0; q < p.ksplit - 1; ++q) {
        const uint32_t src = parts + (i * (p.ksplit - 1) + q) * 16384 + nl * 16;
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const uint4 o = lds128(src + j * 512);
          v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(o.x));
          v[j + 1] = __float_as_uint(__uint_as_float(v[j + 1]) + __uint_as_float(o.y));
          v[j + 2] = __float_as_uint(__uint_as_float(v[j + 2]) + __uint_as_float(o.z));
          v[j + 3] = __float_as_uint(__uint_as_float(v[j + 3]) + __uint_as_float(o.w));
        }
      }
      if (out16) {
        uint32_t h[16];                                  // pairs of tokens of a row
        if (p.out_dtype == EORA_Y_F16) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const __half2 w = __floats2half2_rn(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
            h[j] = *reinterpret_cast<const uint32_t*>(&w);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const __nv_bfloat162 w = __floats2bfloat162_rn(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
            h[j] = *reinterpret_cast<const uint32_t*>(&w);
          }
        }
        // block q of a store: rows 8 q .. of this warp's 32, tokens 8 c ..;  lane 8 q + i gives the address of token i
        const uint32_t at = tbuf + (lane & 7) * 272 + (lq * 32 + (lane >> 3) * 8) * 2;
#pragma unroll
        for (int c = 0; c < 4; ++c) stmatrix_x4_trans(at + c * 8 * 272, h[2 * c], h[2 * c + 1], h[8 + 2 * c], h[8 + 2 * c + 1]);
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) asm volatile("st.shared.u32 [%0], %1;" ::"r"(tbuf + j * 512 + nl * 4), "r"(v[j]) : "memory");
      }
      asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
      const int pieces = 32 << row_sh;
      for (int e = nl; e < pieces; e += 128) {
        const int tok = e >> row_sh, piece = e & ((1 << row_sh) - 1);
        const int row = m0 + c0 + tok, col = n0 + hh * BN_W + piece * (16 / esz);
        if (c0 + tok < bt && row < p.m && col < n_end)       // a unit may reach past the tile's tokens
          *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(out_p) + ((int64_t)row * ld_o + col - col0) * esz) = lds128(tbuf + tok * pitch + piece * 16);
      }
      if (p.ksplit > 1) asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
    }
    if (dw == 0 && lane == 0) PTRACE(nkb, 3);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(512u) : "memory");
}

// n is a multiple of 8 (d_in is a multiple of 128): 16 bytes in, 16 bytes out per step
__global__ void k_bf16_to_f16(const __nv_bfloat16* in, __half* out, int64_t n) {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");         // `out` may still be read by the launch in front
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 8; i < n; i += (int64_t)gridDim.x * blockDim.x * 8) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(in + i));
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __half2 h = __floats2half2_rn(__uint_as_float(w[j] << 16), __uint_as_float(w[j] & 0xffff0000u));
      o[j] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(out + i) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// ---------------------------------------------------------------------------------------------- host
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess || !p) return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// fp16 [rows][cols] row-major, box = 64 columns x box_rows rows, 128-byte swizzle, zero fill out of bounds
bool make_map(CUtensorMap* tm, const void* base, int rows, int cols, int ld, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kSmemP = 225 * 1024;

// The launch may begin while the previous kernel of the stream is still running (it waits, on the device, before it touches what
// that kernel writes).
template <auto KERNEL>
cudaError_t launch_p(dim3 grid, int smem, cudaStream_t st, const CUtensorMap& tx, const CUtensorMap& tt, const CUtensorMap& txs,
                     const CUtensorMap& tts, const PrefillArgs& a) {
  static bool attr_set[64] = {};   // per kernel and device: the attribute belongs to the device that is current at the call
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[device]) {
    cudaError_t e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemP);
    if (e != cudaSuccess) return e;
    attr_set[device] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreadsP);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = a.ksplit; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, KERNEL, tx, tt, txs, tts, a);
}

template <int WF, int BF>
cudaError_t launch_tm(dim3 grid, int smem, cudaStream_t st, const CUtensorMap& tx, const CUtensorMap& tt, const CUtensorMap& txs, const CUtensorMap& tts,
                      const PrefillArgs& a) {
  return a.a_cols ? launch_p<k_prefill<WF, BF, true>>(grid, smem, st, tx, tt, txs, tts, a) : launch_p<k_prefill<WF, BF, false>>(grid, smem, st, tx, tt, txs, tts, a);
}
template <int WF>
cudaError_t launch_bf(int bf, dim3 grid, int smem, cudaStream_t st, const CUtensorMap& tx, const CUtensorMap& tt,
                      const CUtensorMap& txs, const CUtensorMap& tts, const PrefillArgs& a) {
  switch (bf) {
    case FMT_F16: return launch_tm<WF, FMT_F16>(grid, smem, st, tx, tt, txs, tts, a);
    case FMT_Q4: return launch_tm<WF, FMT_Q4>(grid, smem, st, tx, tt, txs, tts, a);
    case FMT_Q8: return launch_tm<WF, FMT_Q8>(grid, smem, st, tx, tt, txs, tts, a);
    case FMT_Q3: return launch_tm<WF, FMT_Q3>(grid, smem, st, tx, tt, txs, tts, a);
    default: return launch_tm<WF, FMT_NONE>(grid, smem, st, tx, tt, txs, tts, a);
  }
}

cudaError_t launch_any(int wf, int bf, dim3 grid, int smem, cudaStream_t st, const CUtensorMap& tx, const CUtensorMap& tt,
                       const CUtensorMap& txs, const CUtensorMap& tts, const PrefillArgs& a) {
  switch (wf) {
    case FMT_Q4: return launch_bf<FMT_Q4>(bf, grid, smem, st, tx, tt, txs, tts, a);
    case FMT_Q3: return launch_bf<FMT_Q3>(bf, grid, smem, st, tx, tt, txs, tts, a);
    case FMT_SP24: return launch_bf<FMT_SP24>(bf, grid, smem, st, tx, tt, txs, tts, a);
    case FMT_SQ4: return launch_bf<FMT_SQ4>(bf, grid, smem, st, tx, tt, txs, tts, a);
    // A as the weight of the first launch (t = X.A): no K-extension there
    case FMT_F16: return launch_tm<FMT_F16, FMT_NONE>(grid, smem, st, tx, tt, txs, tts, a);
    case FMT_Q8: return launch_tm<FMT_Q8, FMT_NONE>(grid, smem, st, tx, tt, txs, tts, a);
    default: return cudaErrorInvalidValue;
  }
}

// Weights in tensor memory: beside the accumulators there is room for at least kTmLeast stages of the tile's weights.
constexpr int kTmLeast = 3;
bool tm_fits(int rows, int bt) { return rows / BN_W * (bt + kTmLeast * 32) <= 512; }

int fill_stages(PrefillArgs& a) {      // returns the dynamic shared memory to request
  if (tm_fits(a.rows, a.bt)) {
    const int nh = a.rows / BN_W;
    a.acc_cols = a.bt; a.a_col0 = nh * a.bt; a.a_cols = 32 * nh;
    // stages as tensor memory has room for, if the warps' rings fit beside their token tiles
    const int w_ring = tm_ring(a.w.fmt), b_ring = tm_ring(a.b.fmt);
    a.w_slot = w_ring > b_ring ? w_ring : b_ring;
    a.sw = (512 - a.a_col0) / a.a_cols;
    if (a.sw > kMaxWStages) a.sw = kMaxWStages;
    while (a.sw > kTmLeast && a.sw * a.bt * 128 + kDqWarps * a.w_slot > kSmemP - 1024) --a.sw;
    a.w_off = a.sw * a.bt * 128;
    const int smem = a.w_off + kDqWarps * a.w_slot, units = nh * ((a.bt + 31) / 32);
    const int out = a.ksplit > 1 ? 65536 + (units + a.ksplit - 1) / a.ksplit * (a.ksplit - 1) * 16384 : 131072;      // the epilogue's
    return (out > smem ? out : smem) + 1024;
  }
  a.a_cols = 0;
  a.w_slot = a.rows * 128;
  const int stage = a.bt * 128 + a.w_slot;             // token tile + weight tile of one k-block
  a.sw = (kSmemP - 1024) / stage;
  if (a.sw > kMaxWStages) a.sw = kMaxWStages;
  a.w_off = a.sw * a.bt * 128;
  int smem = a.w_off + a.sw * a.w_slot;
  const int units = a.rows / BN_W * ((a.bt + 31) / 32);
  const int out = a.ksplit > 1 ? 65536 + (units + a.ksplit - 1) / a.ksplit * (a.ksplit - 1) * 16384 : 131072;      // the epilogue's
  return (out > smem ? out : smem) + 1024;
}

// Tiles of a launch: weight rows and tokens per CTA, CTAs that share a tile's reduction axis.
struct Tiling { int rows, bt, ks; };

// Shared memory of the split epilogue: four buffers of 16 KB and (ks - 1) shares of every ks-th unit.
bool split_fits(int rows, int bt, int ks) {
  const int units = rows / BN_W * ((bt + 31) / 32);
  return 65536 + (units + ks - 1) / ks * (ks - 1) * 16384 <= kSmemP - 1024;
}
// CTAs of clusters of ks that run at once, one per SM (the occupancy calculator's figures for 148 SMs; of seven only 15 clusters).
int at_once(int ks, int sm_count) {
  constexpr int clusters[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
  return sm_count * clusters[ks] / 148 * ks;
}

// Cycles of a k-block, measured with 64 to 256 tokens.  Weights in tensor memory: 128 rows 515 whatever the tokens, 256 rows 790, which is as long as
// sixteen warps take to dequantise them.  Through shared memory, where the accumulators leave no room: 256 rows 1100, and with 256 tokens, whose eight MMAs
// alone take 1024, 1150.  Many tokens come close to what L2 delivers when the SMs are full throughout several waves (128 rows x 256 tokens: 740).
float kblock_cycles(const Tiling& t, bool one_wave) {
  if (t.rows == BN_W) return one_wave || t.bt <= 176 ? (t.bt <= 224 ? 515.f : 540.f) : 2.9f * (float)t.bt;
  return tm_fits(t.rows, t.bt) ? 790.f : t.bt <= 192 ? 1100.f : 1150.f;
}
// Estimated cycles of a launch: its k-blocks, set-up and first operands 3200, the epilogue 900 and 5000 per 256 x 256 of the tile; sharing a
// reduction axis costs two cluster barriers and the way of the tile's sums through distributed shared memory, 1000 + 1600 per
// doubling + 5500 per 256 x 256.  A last partial wave of 256-row tiles that is at most a quarter of the SMs is covered by small tiles
// inside the first wave (launch_prefill_forward), counted as half a wave.
float tiling_cost(const Tiling& t, int n_rows, int m, int nkb, int sm_count) {
  const int tiles = (n_rows + t.rows - 1) / t.rows * ((m + t.bt - 1) / t.bt), cap = at_once(t.ks, sm_count), ctas = tiles * t.ks;
  float waves = (float)((ctas + cap - 1) / cap);
  const int over = tiles % sm_count;
  if (t.ks == 1 && t.rows == 2 * BN_W && t.bt == 256 && tiles > sm_count && over > 0 && 4 * over <= sm_count) waves -= 0.5f;
  constexpr float log2s[9] = {0.f, 0.f, 1.f, 1.5849625f, 2.f, 2.3219281f, 2.5849625f, 2.807355f, 3.f};
  const float area = (float)(t.rows * t.bt) / 65536.f, doublings = log2s[t.ks];
  // Three, five, six or seven CTAs deal a tile's units unevenly (q|k|v at 100 tokens with five 21.4 us, with two CTAs of half the rows 19.5, estimated 4 % slower).
  const float uneven = t.ks & (t.ks - 1) ? 2000.f : 0.f;
  return waves * ((float)((nkb + t.ks - 1) / t.ks) * kblock_cycles(t, ctas <= cap) + 4100.f + 5000.f * area +
                  (t.ks > 1 ? 1000.f + 1600.f * doublings + 5500.f * area + uneven : 0.f));
}

int token_tile(int m, int most) {      // the MMA N: a multiple of 16 up to `most`, even tiles
  const int tiles = (m + most - 1) / most;
  return ((m + tiles - 1) / tiles + 15) / 16 * 16;
}

// The tilings of the main product and of t = X.A (t_cols == 0: none) that take least time together.  A CTA of either launch needs
// an SM of its own and clusters need theirs side by side: if the main launch fits into one wave beside the one for t they
// overlap to the main product's K-extension; if not, it starts with what t leaves and its last CTAs wait for t.
struct Tilings { Tiling main, t; };
// A reduction axis is shared only by clusters that all run at once: in a second wave a cluster waits for SMs side by side (192 CTAs
// in pairs take 50 us where 96 take 27).
// A tiling that can be taken, its CTAs and its time.
struct Candidate { Tiling t; int ctas; float cost; };
constexpr int kMaxCandidates = 32;                   // two token tiles x two row sizes x eight cluster sizes
int candidates(int n_rows, int m, int nkb_w, int nkb, int sm_count, bool only128, Candidate (&out)[kMaxCandidates]) {
  // Even tiles up to 1024 tokens, whole ones beyond.  Beyond, even ones are 1 to 3 % faster up to 1100 tokens (4096 x 14336 at 1025: 103.3 against
  // 106.9 us), within 2 % from there on and 5 % slower at 1800 to 1900 of that shape (198.9 against 188.4).
  // Or tiles of at most 160, where the weights of 256 rows fit into tensor memory.
  const int wide = m > 1024 ? 256 : token_tile(m, 256), narrow = m > 1024 ? 256 : token_tile(m, 160);
  int n = 0;
  for (int bt = wide; bt == wide || bt == narrow; bt = bt == narrow ? 0 : narrow) {
    for (int rows = BN_W; rows <= (only128 ? BN_W : 2 * BN_W); rows += BN_W) {
      const int tiles = (n_rows + rows - 1) / rows * ((m + bt - 1) / bt);
      for (int ks = 1; ks <= 8 && (ks == 1 || nkb_w / ks >= 4); ++ks) {
        const Tiling t{rows, bt, ks};
        if (ks == 1 || (split_fits(rows, bt, ks) && tiles * ks <= at_once(ks, sm_count))) out[n++] = {t, tiles * ks, tiling_cost(t, n_rows, m, nkb, sm_count)};
      }
    }
  }
  return n;
}
// This runs in every call: each candidate's time is worked out once, and a main product that alone takes as long as the best pair does is not paired
// (200 tokens, 1024 outputs, rank 512: 17 us with the times worked out for every pair, now 1.5).
Tilings pick_tilings(int n_rows, int t_cols, int m, int nkb_w, int nkb_b, int sm_count, bool only128) {
  Candidate mains[kMaxCandidates], ts[kMaxCandidates];
  const int n_main = candidates(n_rows, m, nkb_w, nkb_w + nkb_b, sm_count, only128, mains);
  const int n_t = t_cols > 0 ? candidates(t_cols, m, nkb_w, nkb_w, sm_count, t_cols <= BN_W, ts) : 0;
  int room[9] = {};
  for (int ks = 1; ks <= 8; ++ks) room[ks] = at_once(ks, sm_count);
  Tilings best = {};
  float best_c = -1.f;
  for (int i = 0; i < n_main; ++i) {
    const Candidate& a = mains[i];
    const float cm = a.cost, tail = (float)nkb_b * kblock_cycles(a.t, true);
    if (best_c >= 0.f && cm >= best_c) continue;
    if (n_t == 0) { best_c = cm; best = {a.t, Tiling{}}; continue; }
    const bool one_wave = a.ctas <= room[a.t.ks];
    for (int j = 0; j < n_t; ++j) {
      const Candidate& t = ts[j];
      const float ct = t.cost;
      const bool beside = one_wave && a.ctas + t.ctas <= room[a.t.ks > t.t.ks ? a.t.ks : t.t.ks];
      // (of equal ones the earlier t: three blocks of 64 tokens with adapters of rank 512, down 31.6 -> 28.6 us)
      const float c = 0.02f * ct + (beside ? (cm > ct + tail ? cm : ct + tail) : one_wave ? cm + ct : cm + ct * (float)t.ctas / (float)sm_count);
      if (best_c < 0.f || c < best_c) { best_c = c; best = {a.t, t.t}; }
    }
  }
  return best;
}

Tilings plan_tilings(const Handle* h, int m) {
  const bool ab = h->cfg.rank > 0;
  const int n_rows = h->n_sub > 1 ? 16 * h->sub_tile0[h->n_sub] : h->cfg.d_out;
  bool only128 = false;                                       // fused layers: every layer a whole number of tiles
  for (int i = 0; i < h->n_sub && h->n_sub > 1; ++i) only128 = only128 || h->sub_dout[i] % (2 * BN_W) != 0;
  return pick_tilings(n_rows, ab ? h->t_cols : 0, m, h->cfg.d_in / BK, ab ? h->r_pad / BK : 0, h->sm_count, only128);
}

// The most k-blocks from one that a dequant warp takes to the next it takes, over the CTAs of a launch whose rows end in a tile of one half.
int longest_step(const PrefillArgs& a) {
  const bool tm = a.a_cols > 0;
  const int uw = unit_blocks(a.w.fmt, tm), ub = unit_blocks(a.b.fmt, tm);
  int longest = 1;
  for (int split = 0; split < a.ksplit; ++split)
    for (int phase = 0; phase < 2; ++phase) {
      const int nkw = split_lo(a, split + 1) - split_lo(a, split), nb = split == 0 ? a.nkb_b : 0;
      int last = -1;                                     // (the first ones need no wait: as if the k-block in front of the first were this warp's)
      auto part = [&](int it0, int units, int u, int from) {
        for (int i = from; i < units; i += 2) {
          if (it0 + i * u - last > longest) longest = it0 + i * u - last;
          last = it0 + i * u + u - 1;
        }
      };
      part(0, nkw / uw, uw, phase);
      if (nb > 0) part(nkw, nb / ub, ub, b_phase(phase, 2, nkw / uw));
    }
  return longest;
}

}  // namespace

int prefill_plan(const Handle* h, int m, eora_prefill_tiling* out) {
  if (h->multi || h->w.group % 64) return EORA_ERR_UNSUPPORTED;
  for (int i = 0; i < h->n_sub && h->n_sub > 1; ++i)
    if (h->sub_dout[i] % BN_W) return EORA_ERR_UNSUPPORTED;
  const Tilings tls = plan_tilings(h, m);
  for (int i = 0; i < 2; ++i) {
    out[i] = eora_prefill_tiling();
    if (i == 1 && h->cfg.rank == 0) break;
    const Tiling& t = i ? tls.t : tls.main;
    PrefillArgs a = {};
    a.w.fmt = i ? h->a.fmt : h->w.fmt;
    a.b.fmt = i || h->cfg.rank == 0 ? FMT_NONE : h->b.fmt;
    a.rows = t.rows; a.bt = t.bt; a.ksplit = t.ks;
    a.nkb_w = h->cfg.d_in / BK; a.nkb_b = i || h->cfg.rank == 0 ? 0 : h->r_pad / BK;
    fill_stages(a);
    out[i].rows = t.rows; out[i].tokens = t.bt; out[i].cluster = t.ks;
    out[i].stages = a.sw; out[i].in_tensor_memory = a.a_cols > 0; out[i].longest_step = longest_step(a);
  }
  return EORA_OK;
}

bool prefill_supported(const Handle* h, int m) {
  if (m <= 8) return false;              // one decode pass is always cheaper
  if (h->multi) return false;            // per-token adapters: decode family only
  if (h->n_sub > 1) {                    // fused layers: tiles of 128 rows must not straddle two layers
    for (int i = 0; i < h->n_sub; ++i)
      if (h->sub_dout[i] % BN_W) return false;
  }
  if (h->w.group % 64) return false;
  return encode_fn() != nullptr;
}

int prefill_launch_count(const Handle* h, int m) {
  return (mid_supported(h, m) ? 1 : h->cfg.rank > 0 ? 2 : 1) + (h->cfg.x_dtype == EORA_X_BF16 ? 1 : 0);
}

cudaError_t prefill_init(Handle* h) {
  h->prefill_state = nullptr;
  if (h->cfg.max_m <= 8) return cudaSuccess;
  PrefillState* ps = new PrefillState();
  *ps = PrefillState();
  cudaError_t e = cudaSuccess;
  if (h->cfg.x_dtype == EORA_X_BF16) e = cudaMalloc(&ps->x16, (size_t)h->cfg.max_m * h->cfg.d_in * 2);
  if (e != cudaSuccess) { delete ps; return e; }
  h->prefill_state = ps;
  return cudaSuccess;
}

void prefill_free(Handle* h) {
  PrefillState* ps = reinterpret_cast<PrefillState*>(h->prefill_state);
  if (!ps) return;
  cudaFree(ps->x16);
  delete ps;
  h->prefill_state = nullptr;
}

cudaError_t launch_prefill_forward(const Handle* h, const void* x, int m, void* const* ys, cudaStream_t st) {
  const eora_linear_config& c = h->cfg;
  const void* x16 = x;
  if (c.x_dtype == EORA_X_BF16) {
    PrefillState* ps = reinterpret_cast<PrefillState*>(h->prefill_state);
    if (!ps || !ps->x16) return cudaErrorInvalidValue;
    int64_t n = (int64_t)m * c.d_in;
    int64_t blocks = (n / 8 + 255) / 256;
    if (blocks > h->sm_count * 8) blocks = h->sm_count * 8;
    cudaLaunchConfig_t cc = {};
    cc.gridDim = dim3((unsigned)blocks);
    cc.blockDim = dim3(256);
    cc.stream = st;
    cudaLaunchAttribute ca[1];
    ca[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    ca[0].val.programmaticStreamSerializationAllowed = 1;
    cc.attrs = ca;
    cc.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cc, k_bf16_to_f16, reinterpret_cast<const __nv_bfloat16*>(x), ps->x16, n);
    if (e != cudaSuccess) return e;
    x16 = ps->x16;
  }
  if (mid_supported(h, m)) return launch_mid_forward(h, x16, m, ys, st);
  const bool ab = c.rank > 0;
  const Tilings tls = plan_tilings(h, m);
  const Tiling tl = tls.main;
  const int bt = tl.bt;
  CUtensorMap tm_x, tm_t;
  if (!make_map(&tm_x, x16, m, c.d_in, c.d_in, bt)) return cudaErrorInvalidValue;
  if (ab) {
    if (!make_map(&tm_t, h->t16, m, h->t_cols, h->t_cols, bt)) return cudaErrorInvalidValue;
    // launch 1: t = X.A with A as the weight (rows = r_pad), written as fp16.  It is a small product, and the main launch
    // behind it starts on the other SMs while it runs (programmatic dependent launch): the main product needs t only
    // for its last k-blocks and waits for this launch there.
    const int rows_t = tls.t.rows, bt_t = tls.t.bt;
    CUtensorMap tm_xt;
    if (!make_map(&tm_xt, x16, m, c.d_in, c.d_in, bt_t)) return cudaErrorInvalidValue;
    PrefillArgs a = {};
    a.w = h->a; a.b = WMat(); a.b.fmt = FMT_NONE;
    a.out = h->t16; a.out_dtype = EORA_Y_F16; a.ld_out = h->t_cols; a.n_valid = h->t_cols; a.m = m; a.bt = bt_t;
    a.nkb_w = c.d_in / BK; a.nkb_b = 0; a.dev_status = h->dev_status; a.trace = nullptr;
    a.rows = rows_t;
    a.n_small = 0; a.small_x = 1; a.n_split = a.n_valid; a.big_x = (h->t_cols + a.rows - 1) / a.rows;
    a.n_sub = 1; a.sub_row0[0] = 0; a.outs[0] = a.out; a.sub_ld[0] = a.ld_out; a.t_sub = 0;
    for (int i = 1; i < 5; ++i) a.sub_row0[i] = a.n_valid;
    a.ksplit = tls.t.ks; a.wait_x = 1;
    const int smem_t = fill_stages(a);
    dim3 grid(a.big_x * a.ksplit * ((m + bt_t - 1) / bt_t), 1, 1);
    cudaError_t e = launch_any(h->a.fmt, FMT_NONE, grid, smem_t, st, tm_xt, tm_xt, tm_xt, tm_xt, a);
    if (e != cudaSuccess) return e;
  } else {
    tm_t = tm_x;
  }
  PrefillArgs a = {};
  a.w = h->w; a.b = h->b;
  if (!ab) a.b.fmt = FMT_NONE;
  // fused layers: the stacked rows; a plain layer has one part
  const int n_all = h->w.n_rows < 16 * h->sub_tile0[h->n_sub] ? h->w.n_rows : 16 * h->sub_tile0[h->n_sub];
  const int n_valid = h->n_sub > 1 ? n_all : c.d_out;
  a.out = ys[0]; a.out_dtype = c.y_dtype; a.ld_out = c.d_out; a.n_valid = n_valid; a.m = m; a.bt = bt;
  a.n_sub = h->n_sub; a.t_sub = h->n_sub > 1 ? h->r_pad : 0;
  for (int i = 0; i < 5; ++i) a.sub_row0[i] = n_valid;
  for (int i = 0; i < h->n_sub; ++i) {
    a.sub_row0[i] = h->n_sub > 1 ? 16 * h->sub_tile0[i] : 0;
    a.outs[i] = ys[i];
    a.sub_ld[i] = h->n_sub > 1 ? h->sub_dout[i] : c.d_out;
  }
  a.nkb_w = c.d_in / BK; a.nkb_b = ab ? h->r_pad / BK : 0; a.dev_status = h->dev_status;
  a.trace = reinterpret_cast<long long*>(h->trace);
  a.rows = tl.rows;
  a.n_small = 0; a.small_x = 1; a.n_split = n_valid; a.big_x = (n_valid + a.rows - 1) / a.rows;
  a.ksplit = tl.ks; a.wait_x = ab ? 0 : 1;
  const int big_y = (m + bt - 1) / bt;
  // Wave quantisation: a CTA needs an SM of its own, so a few tiles more than a whole number of waves cost a whole
  // wave (gate / up at M = 2048: 448 tiles on 148 SMs).  Then the last row tiles are taken out of the big grid until
  // it fits, and their rows are covered by small tiles (128 x 128, about half the time of a big one each) that are
  // dispatched first and share the launch's first wave with the big tiles.
  CUtensorMap tm_xs = tm_x, tm_ts = tm_t;
  const int tiles = a.big_x * big_y, over = tiles % h->sm_count;
  if (a.ksplit == 1 && a.rows == 2 * BN_W && bt == 256 && tiles > h->sm_count && over > 0 && 4 * over <= h->sm_count) {
    const int peel = (over + big_y - 1) / big_y;                 // row tiles to take out
    if (peel < a.big_x) {
      a.big_x -= peel;
      a.n_split = a.big_x * a.rows;
      a.small_x = (n_valid - a.n_split + kSmallTile - 1) / kSmallTile;
      a.n_small = a.small_x * ((m + kSmallTile - 1) / kSmallTile);
      if (!make_map(&tm_xs, x16, m, c.d_in, c.d_in, kSmallTile)) return cudaErrorInvalidValue;
      if (ab && !make_map(&tm_ts, h->t16, m, h->t_cols, h->t_cols, kSmallTile)) return cudaErrorInvalidValue;
      if (!ab) tm_ts = tm_xs;
    }
  }
  const int smem_y = fill_stages(a);
  dim3 grid(a.n_small + a.big_x * a.ksplit * big_y, 1, 1);
  return launch_any(h->w.fmt, ab ? h->b.fmt : FMT_NONE, grid, smem_y, st, tm_x, tm_t, tm_xs, tm_ts, a);
}

}  // namespace eora
