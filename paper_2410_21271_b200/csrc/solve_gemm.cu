// fp32 products on the 5th-generation tensor cores, for the large contractions of the offline solve.
//
// Why.  On the CUDA cores these products are bound by the FFMA pipe (42 of 74 TFLOP/s reached; P = dW X~ of a 4096 x 4096 layer with 2048
// calibration columns 1650 us, its Gram matrix 460).  Here every fp32 value is the sum of three bf16 numbers of eight bits each, which is
// exact but for a part of 2^-27, and a product is six bf16 MMAs: high x high and the five next larger ones; what is left out is 2^-26 of
// |a| |b| at most.
//
// Sums.  The tensor core adds to its fp32 accumulator with truncation, so a long chain in it drifts; fp32 arithmetic on the CUDA cores rounds.
// high x high therefore goes to an accumulator of its own that is emptied every 256 reduction elements (16 MMAs) into registers,
// where the parts are added with rounding; the five small products, 2^-8 as large, share a second accumulator to the end.
//
// Shape.  A tile of 128 x 256 (or 128 x 128, where that fills the GPU better, and for symmetric results) per CTA, stages of 32 reduction
// elements (72 KB: three of them), one copying thread, one issuing warp, sixteen warps that empty the accumulators while the
// issuing warp goes on with the small products.  The tensor core needs 1536 cycles per stage of 128 x 256, the copies 47 bytes a cycle and SM.
// Operands are split and laid out as the tensor core reads them by a pass of their own (2 x 3 x 2 bytes per value, 15 to 35 us).
#include <cuda_bf16.h>
#include "decode_common.cuh"
#include "tcgen05.cuh"
#include "solve_gemm.cuh"

namespace eora {
namespace {
using namespace dec;

// x = h + m + l, eight significant bits each.
__device__ __forceinline__ void split3(float x, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = __bfloat16_as_ushort(__float2bfloat16_rn(x));
  if ((h & 0x7f80u) == 0x7f80u) {                    // rounded up to infinity: cut instead; infinities and NaN stay what they are
    if ((__float_as_uint(x) & 0x7f800000u) == 0x7f800000u) { m = l = 0u; return; }
    h = __float_as_uint(x) >> 16;
  }
  const float r1 = x - __uint_as_float(h << 16);     // (exact)
  m = __bfloat16_as_ushort(__float2bfloat16_rn(r1));
  l = __bfloat16_as_ushort(__float2bfloat16_rn(r1 - __uint_as_float(m << 16)));
}
// Eight consecutive reduction elements of row r of a block, piece c (of 4).
__device__ __forceinline__ void store_piece(uint8_t* block, int r, int c, const float (&v)[8]) {
  uint32_t o[3][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    uint32_t a[3], b[3];
    split3(v[2 * e], a[0], a[1], a[2]);
    split3(v[2 * e + 1], b[0], b[1], b[2]);
#pragma unroll
    for (int p = 0; p < 3; ++p) o[p][e] = a[p] | b[p] << 16;
  }
  uint8_t* at = block + r * 64 + ((c ^ ((r >> 1) & 3)) << 4);
#pragma unroll
  for (int p = 0; p < 3; ++p) *reinterpret_cast<uint4*>(at + p * kSplitPlane) = make_uint4(o[p][0], o[p][1], o[p][2], o[p][3]);
}

// A CTA takes 128 rows x 128 columns.
__global__ void __launch_bounds__(256) k_split_rows(const float* __restrict__ a, const float* __restrict__ b, int rows, int cols, int lda, bool vec,
                                                    int cols_p, uint8_t* __restrict__ out, float* __restrict__ copy, int ld_copy) {
  const int c = threadIdx.x & 3;
  for (int i = 0; i < 8; ++i) {
    const int r = (threadIdx.x >> 2) + (i & 1) * 64, kb = blockIdx.x * 4 + (i >> 1);
    const int64_t row = (int64_t)blockIdx.y * kSplitRows + r;
    const int k0 = kb * kSplitCols + 8 * c;
    float v[8];
    if (vec) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < rows && k0 + 4 * h < cols) {
          u = *reinterpret_cast<const float4*>(a + row * lda + k0 + 4 * h);
          if (b) { const float4 w = *reinterpret_cast<const float4*>(b + row * lda + k0 + 4 * h); u.x -= w.x; u.y -= w.y; u.z -= w.z; u.w -= w.w; }
        }
        v[4 * h] = u.x; v[4 * h + 1] = u.y; v[4 * h + 2] = u.z; v[4 * h + 3] = u.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        v[e] = 0.f;
        if (row < rows && k0 + e < cols) { v[e] = a[row * lda + k0 + e]; if (b) v[e] -= b[row * lda + k0 + e]; }
      }
    }
    if (copy) {
      float4* to = reinterpret_cast<float4*>(copy + row * ld_copy + k0);
      to[0] = make_float4(v[0], v[1], v[2], v[3]); to[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
    if (out) store_piece(out + ((int64_t)blockIdx.y * (cols_p / kSplitCols) + kb) * kSplitBlock, r, c, v);
  }
}

// A CTA takes 32 rows x 128 columns of a: 128 rows x 32 columns of the operand.  (A pitch of 129 words: the eight values of a piece are read
// from different banks by the four pieces x eight rows of a warp.)
__global__ void __launch_bounds__(256) k_split_cols(const float* __restrict__ a, int rows, int cols, int lda, int rows_p, int cols_p, uint8_t* __restrict__ out,
                                                    float* __restrict__ copy) {
  __shared__ float s[kSplitCols][129];
  const int n0 = blockIdx.x * kSplitRows, k0 = blockIdx.y * kSplitCols;
  float v[16];                                       // (all loads out together: the pass is latency)
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int k = (threadIdx.x >> 7) + 2 * i, n = threadIdx.x & 127;
    v[i] = k0 + k < rows && n0 + n < cols ? a[(int64_t)(k0 + k) * lda + n0 + n] : 0.f;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int k = (threadIdx.x >> 7) + 2 * i, n = threadIdx.x & 127;
    s[k][n] = v[i];
    if (copy) copy[(int64_t)(k0 + k) * cols_p + n0 + n] = v[i];
  }
  __syncthreads();
  const int c = threadIdx.x & 3;
  uint8_t* block = out + ((int64_t)blockIdx.x * (rows_p / kSplitCols) + blockIdx.y) * kSplitBlock;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = (threadIdx.x >> 2) + i * 64;
    float w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = s[8 * c + e][r];
    store_piece(block, r, c, w);
  }
}

// ---------------------------------------------------------------------------------------------- product
constexpr int kGemmThreads = 640;                  // warp 0: copies, 1: MMA, 2: tensor memory, 4..19: accumulators
constexpr int kChunk = 8;                          // stages after which the accumulator of high x high is emptied
__host__ __device__ constexpr int gemm_stage(int nt) { return (kSplitRows + nt) * 64 * 3; }
__host__ __device__ constexpr int gemm_stages(int nt) { return nt == 256 ? 3 : 4; }
constexpr int gemm_smem(int nt) { return gemm_stage(nt) * gemm_stages(nt) + 1024; }

__device__ __forceinline__ void tmem_add8(uint32_t taddr, float* acc) {
  uint32_t v[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] += __uint_as_float(v[i]);
}

// The barriers of a CTA and its tensor memory: high x high in columns [0, NT), the rest in [256, 256 + NT).
struct GemmShared { uint64_t full[4], empty[4], d0_full, d0_free, d1_full; uint32_t tmem; };
constexpr uint32_t kSmallCol = 256;
template <int S>
__device__ __forceinline__ void gemm_setup(GemmShared& sh, int warp) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) { mbar_init(sh.full + i, 1); mbar_init(sh.empty + i, 1); }
    mbar_init(&sh.d0_full, 1); mbar_init(&sh.d0_free, 16); mbar_init(&sh.d1_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void gemm_release(GemmShared& sh, int warp) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh.tmem), "r"(512u) : "memory");
}

// The sums of a tile of 128 rows x NT columns over nkb stages.  ap: the row block of A at the first stage.  b: all of B; rows [n0, n0 + NT) of it, stages
// from kb0 on, of nkb_b in all.  Warps 4..19 return the sums of row 32 (warp % 4) + lane and NT / 4 columns from (warp - 4) / 4 * NT / 4 on in acc
// (warps whose wait ran out return false); the others take part.
template <int NT, int S>
__device__ __forceinline__ bool gemm_tile(GemmShared& sh, uint32_t smem, int warp, int lane, const uint8_t* ap, const uint8_t* b, int n0, int kb0,
                                          int nkb_b, int nkb, int* status, float (&acc)[NT / 4]) {
  constexpr int kStage = gemm_stage(NT), kA = kSplitBlock, kPlaneB = NT * 64;
  if (warp == 0) {
    if (lane == 0) {
      int s = 0, wrap = 0, it = 0;
      bool ok = true;
      for (; it < nkb; ++it) {
        if (wrap > 0 && !mbar_wait(sh.empty + s, (wrap - 1) & 1, status)) { ok = false; break; }
        const uint32_t at = smem + s * kStage, bar = smem_u32(sh.full + s);
        mbar_expect_tx_a(bar, kStage);
        bulk_g2s_a(at, ap + (int64_t)it * kSplitBlock, kSplitBlock, bar);
        for (int r = 0; r < NT;) {                   // the rows of B lie in one to three row blocks (n0 is a multiple of 32: the swizzle fits)
          const int in = (n0 + r) % kSplitRows, cnt = min(kSplitRows - in, NT - r);
          const uint8_t* src = b + ((int64_t)((n0 + r) / kSplitRows) * nkb_b + kb0 + it) * kSplitBlock + in * 64;
          if (NT == kSplitRows && cnt == NT) {
            bulk_g2s_a(at + kA, src, kSplitBlock, bar);
          } else {
#pragma unroll
            for (int q = 0; q < 3; ++q) bulk_g2s_a(at + kA + q * kPlaneB + r * 64, src + q * kSplitPlane, cnt * 64, bar);
          }
          r += cnt;
        }
        if (++s == S) { s = 0; ++wrap; }
      }
      if (!ok) {                                     // gave up: what is in flight lands first
        const int issued = it < S ? it : S;
        for (int i = 0; i < issued; ++i) {
          const int at_it = it - 1 - i, slot = at_it % S;
          const unsigned long long t0 = globaltimer_ns();
          while (!mbar_try_wait(sh.full + slot, (at_it / S) & 1) && globaltimer_ns() - t0 < 2000000ull) __nanosleep(200);
        }
      }
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == 1) {
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) | ((128u >> 4) << 24);      // fp32 += bf16 x bf16
    const bool elected = elect_one();
    const uint32_t tmem = sh.tmem, small = tmem + kSmallCol;
    const uint64_t a0 = make_desc<64>(smem), b0 = make_desc<64>(smem + kA);
    constexpr uint32_t pa = kSplitPlane >> 4, pb = kPlaneB >> 4;
    bool ok = true;
    uint32_t s = 0, ph = 0;
    for (int it = 0, pos = 0; it < nkb; ++it) {
      if (!mbar_try_wait_a(smem_u32(sh.full + s), ph)) ok = mbar_wait(sh.full + s, ph, status);
      if (ok && pos == 0 && it > 0) ok = mbar_wait(&sh.d0_free, (it / kChunk - 1) & 1, status);
      if (!__all_sync(0xffffffffu, ok)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t ad = a0 + s * (kStage >> 4), bd = b0 + s * (kStage >> 4);
      const bool last = pos == kChunk - 1 || it == nkb - 1;
      if (elected) {
#pragma unroll
        for (int k = 0; k < 2; ++k) umma_f16(tmem, ad + 2 * k, bd + 2 * k, idesc, pos > 0 || k > 0 ? 1u : 0u);
        if (last) umma_commit(&sh.d0_full);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          umma_f16(small, ad + 2 * k, bd + pb + 2 * k, idesc, it > 0 || k > 0 ? 1u : 0u);
          umma_f16(small, ad + pa + 2 * k, bd + 2 * k, idesc, 1u);
          umma_f16(small, ad + 2 * k, bd + 2 * pb + 2 * k, idesc, 1u);
          umma_f16(small, ad + 2 * pa + 2 * k, bd + 2 * k, idesc, 1u);
          umma_f16(small, ad + pa + 2 * k, bd + pb + 2 * k, idesc, 1u);
        }
        umma_commit(sh.empty + s);
      }
      if (++pos == kChunk) pos = 0;
      if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
    }
    if (elected) umma_commit(&sh.d1_full);
    __syncwarp();
  } else if (warp >= 4) {
    constexpr int W = NT / 4;                        // columns of a warp: a quarter of the tile's, of the 32 rows its number selects
    const uint32_t at = sh.tmem + ((uint32_t)((warp & 3) * 32) << 16) + ((warp - 4) >> 2) * W;
#pragma unroll
    for (int i = 0; i < W; ++i) acc[i] = 0.f;
    const int chunks = (nkb + kChunk - 1) / kChunk;
    for (int ch = 0; ch < chunks; ++ch) {
      if (!mbar_wait_warp_fast(&sh.d0_full, ch & 1, status, lane)) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int i = 0; i < W; i += 8) tmem_add8(at + i, acc + i);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&sh.d0_free)) : "memory");
    }
    if (!mbar_wait_warp_fast(&sh.d1_full, 0, status, lane)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
    for (int i = 0; i < W; i += 8) tmem_add8(at + kSmallCol + i, acc + i);
  }
  return true;
}

template <int NT, bool SYM>
__global__ void __launch_bounds__(kGemmThreads, 1) k_split_gemm(const uint8_t* __restrict__ a, const uint8_t* __restrict__ b, int nkb,
                                                                 float* __restrict__ c, int ldc, bool add, int* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) GemmShared sh;
  const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int by = blockIdx.y, bx = blockIdx.x;
  if (SYM) {                                         // tile number -> (row, column <= row)
    by = (int)((sqrtf(8.f * bx + 1.f) - 1.f) * 0.5f);
    while ((by + 1) * (by + 2) / 2 <= bx) ++by;
    while (by * (by + 1) / 2 > bx) --by;
    bx -= by * (by + 1) / 2;
  }
  gemm_setup<gemm_stages(NT)>(sh, warp);
  float acc[NT / 4];
  const bool ok = gemm_tile<NT, gemm_stages(NT)>(sh, smem, warp, lane, a + (int64_t)by * nkb * kSplitBlock, b, bx * NT, 0, nkb, nkb, status, acc);
  if (warp >= 4 && ok) {
    const int64_t row = (int64_t)by * 128 + (warp & 3) * 32 + lane, col = (int64_t)bx * NT + ((warp - 4) >> 2) * (NT / 4);
    float4* to = reinterpret_cast<float4*>(c + row * ldc + col);
    if (add) {
#pragma unroll
      for (int i = 0; i < NT / 16; ++i) {
        const float4 o = to[i];
        acc[4 * i] += o.x; acc[4 * i + 1] += o.y; acc[4 * i + 2] += o.z; acc[4 * i + 3] += o.w;
      }
    }
#pragma unroll
    for (int i = 0; i < NT / 16; ++i) to[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
    if (SYM && by != bx) {
#pragma unroll
      for (int i = 0; i < NT / 4; ++i) c[(col + i) * ldc + row] = acc[i];
    }
  }
  gemm_release(sh, warp);
}

// Products with an iterate: C [m][ldc] = A B^T - *shift Y, B having a few hundred rows (the iterate's columns), of which a CTA takes NT.  A cluster
// shares a tile of 128 rows along the reduction axis; the parts meet in distributed shared memory and are added in a fixed order.
// 2048 x 2048 x 160 are 16 tiles, 64 CTAs of sixteen stages.
constexpr int kPartPad = 4;                          // floats between the rows of a part (16-byte stores of 32 rows hit all banks)
template <int NT>
__global__ void __launch_bounds__(kGemmThreads, 1) k_split_skinny(const uint8_t* __restrict__ a, const uint8_t* __restrict__ b, int nkb,
                                                                   float* __restrict__ c, int ldc, const float* __restrict__ y, const float* __restrict__ shift, int* status) {
  constexpr int S = 3, pitch = NT + kPartPad;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) GemmShared sh;
  uint8_t* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t smem = smem_u32(base);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ks = gridDim.x, rank = blockIdx.x;
  const int n0 = blockIdx.z * NT, lo = rank * nkb / ks, hi = (rank + 1) * nkb / ks;
  gemm_setup<S>(sh, warp);
  float acc[NT / 4];
  const bool ok = gemm_tile<NT, S>(sh, smem, warp, lane, a + ((int64_t)blockIdx.y * nkb + lo) * kSplitBlock, b, n0, lo, nkb, hi - lo, status, acc);
  // (every MMA has completed when a warp has its sums, so the stages may be overwritten; a CTA that gave up sends what it has: the status says so)
  float* part = reinterpret_cast<float*>(base);
  if (warp >= 4 && ok) {
    float4* to = reinterpret_cast<float4*>(part + ((warp & 3) * 32 + lane) * pitch + ((warp - 4) >> 2) * (NT / 4));
#pragma unroll
    for (int i = 0; i < NT / 16; ++i) to[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
  }
  __syncwarp();
  cluster_arrive(); cluster_wait();
  const int per = 128 / ks;                          // rows of the tile that this CTA adds up
  const float rho = shift ? *shift : 0.f;
  for (int e = threadIdx.x; e < per * (NT / 4); e += kGemmThreads) {
    const int r = rank * per + e / (NT / 4), q = (e % (NT / 4)) * 4;
    const uint32_t at = smem + (r * pitch + q) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < ks; ++k) {
      float4 u;
      asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(u.x), "=f"(u.y), "=f"(u.z), "=f"(u.w) : "r"(mapa(at, (uint32_t)k)));
      v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
    }
    const int64_t to = ((int64_t)blockIdx.y * 128 + r) * ldc + n0 + q;
    if (shift) {
      const float4 u = *reinterpret_cast<const float4*>(y + to);
      v.x = fmaf(-rho, u.x, v.x); v.y = fmaf(-rho, u.y, v.y); v.z = fmaf(-rho, u.z, v.z); v.w = fmaf(-rho, u.w, v.w);
    }
    *reinterpret_cast<float4*>(c + to) = v;
  }
  cluster_arrive(); cluster_wait();                  // nobody leaves while its sums are being read
  gemm_release(sh, warp);
}

template <int NT, bool SYM>
cudaError_t launch_gemm(dim3 grid, cudaStream_t st, const uint8_t* a, const uint8_t* b, int k, float* c, int ldc, bool add, int* status) {
  static bool set[64] = {};                          // per device
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
  if (!set[device]) {
    e = cudaFuncSetAttribute(k_split_gemm<NT, SYM>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem(NT));
    if (e != cudaSuccess) return e;
    set[device] = true;
  }
  k_split_gemm<NT, SYM><<<grid, kGemmThreads, gemm_smem(NT), st>>>(a, b, k / kSplitCols, c, ldc, add, status);
  return cudaGetLastError();
}

}  // namespace

cudaError_t split_rows(cudaStream_t st, const float* a, const float* b, int rows, int cols, int lda, int rows_p, int cols_p, uint8_t* out, float* copy, int ld_copy) {
  const bool vec = cols % 4 == 0 && lda % 4 == 0 && ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
  k_split_rows<<<dim3(cols_p / 128, rows_p / 128), 256, 0, st>>>(a, b, rows, cols, lda, vec, cols_p, out, copy, ld_copy);
  return cudaGetLastError();
}
cudaError_t split_cols(cudaStream_t st, const float* a, int rows, int cols, int lda, int rows_p, int cols_p, uint8_t* out, float* copy) {
  k_split_cols<<<dim3(cols_p / kSplitRows, rows_p / kSplitCols), 256, 0, st>>>(a, rows, cols, lda, rows_p, cols_p, out, copy);
  return cudaGetLastError();
}
cudaError_t split_gemm(cudaStream_t st, const uint8_t* a, const uint8_t* b, int m, int n, int k, float* c, int ldc, bool sym, bool add, int sm_count, int* status) {
  const int mt = m / 128, nt = n / 128;
  if (sym) return launch_gemm<128, true>(dim3(mt * (mt + 1) / 2), st, a, b, k, c, ldc, add, status);
  // Cycles of a stage: 1536 of MMAs for 256 columns; 768 for 128, of which the copies (48 KB) take about 900.
  const int waves256 = (mt * (nt / 2) + sm_count - 1) / sm_count, waves128 = (mt * nt + sm_count - 1) / sm_count;
  if (nt % 2 == 0 && waves256 * 1536 <= waves128 * 900) return launch_gemm<256, false>(dim3(nt / 2, mt), st, a, b, k, c, ldc, add, status);
  return launch_gemm<128, false>(dim3(nt, mt), st, a, b, k, c, ldc, add, status);
}

namespace {
template <int NT>
cudaError_t launch_skinny(cudaStream_t st, const uint8_t* a, const uint8_t* b, int m, int n, int k, float* c, int ldc, const float* y, const float* shift, int* status) {
  // More than half of an SM's shared memory, so that no two such CTAs (of solves on different streams) share an SM: each takes all of tensor memory, and
  // clusters whose CTAs wait for one another's would wait for good.
  constexpr int own = 3 * gemm_stage(NT) + 1024, smem = own > 120 * 1024 ? own : 120 * 1024;
  static_assert(128 * (NT + kPartPad) * 4 <= 3 * gemm_stage(NT), "a CTA's sums take the place of its stages");
  static bool set[64] = {};                          // per device
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
  if (!set[device]) {
    e = cudaFuncSetAttribute(k_split_skinny<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    set[device] = true;
  }
  // as many CTAs per tile as run at once (15 clusters of eight, 33 of four, 74 of two, measured with one CTA per SM), each with at least four stages.  (A
  // sixteenth cluster of eight waits for the others: 25 us instead of 17.)
  const int tiles = m / 128 * (n / NT), nkb = k / kSplitCols;
  int ks = 8;
  while (ks > 1 && (tiles > (ks == 8 ? 15 : ks == 4 ? 33 : 74) || nkb / ks < 4)) ks >>= 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ks, m / 128, n / NT);
  cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_split_skinny<NT>, a, b, nkb, c, ldc, y, shift, status);
}
}  // namespace

cudaError_t split_skinny(cudaStream_t st, int width, const uint8_t* a, const uint8_t* b, int m, int n, int k, float* c, int ldc, const float* y, const float* shift, int* status) {
  switch (width) {
    case 64: return launch_skinny<64>(st, a, b, m, n, k, c, ldc, y, shift, status);
    case 96: return launch_skinny<96>(st, a, b, m, n, k, c, ldc, y, shift, status);
    case 128: return launch_skinny<128>(st, a, b, m, n, k, c, ldc, y, shift, status);
    default: return launch_skinny<160>(st, a, b, m, n, k, c, ldc, y, shift, status);
  }
}

}  // namespace eora
