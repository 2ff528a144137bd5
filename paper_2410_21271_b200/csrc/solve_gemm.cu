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
    store_piece(out + ((int64_t)blockIdx.y * (cols_p / kSplitCols) + kb) * kSplitBlock, r, c, v);
  }
}

// A CTA takes 32 rows x 128 columns of a: 128 rows x 32 columns of the operand.  (A pitch of 129 words: the eight values of a piece are read
// from different banks by the four pieces x eight rows of a warp.)
__global__ void __launch_bounds__(256) k_split_cols(const float* __restrict__ a, int rows, int cols, int lda, int rows_p, int cols_p, uint8_t* __restrict__ out,
                                                    float* __restrict__ copy) {
  __shared__ float s[kSplitCols][129];
  const int n0 = blockIdx.x * kSplitRows, k0 = blockIdx.y * kSplitCols;
  for (int e = threadIdx.x; e < kSplitCols * kSplitRows; e += 256) {
    const int k = e >> 7, n = e & 127;
    const float v = k0 + k < rows && n0 + n < cols ? a[(int64_t)(k0 + k) * lda + n0 + n] : 0.f;
    s[k][n] = v;
    if (copy) copy[(int64_t)(k0 + k) * cols_p + n0 + n] = v;
  }
  __syncthreads();
  const int c = threadIdx.x & 3;
  uint8_t* block = out + ((int64_t)blockIdx.x * (rows_p / kSplitCols) + blockIdx.y) * kSplitBlock;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = (threadIdx.x >> 2) + i * 64;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = s[8 * c + e][r];
    store_piece(block, r, c, v);
  }
}

// ---------------------------------------------------------------------------------------------- product
constexpr int kGemmThreads = 640;                  // warp 0: copies, 1: MMA, 2: tensor memory, 4..19: accumulators
constexpr int kChunk = 8;                          // stages after which the accumulator of high x high is emptied
__host__ __device__ constexpr int gemm_stage(int nt) { return (kSplitRows + nt) * 64 * 3; }
__host__ __device__ constexpr int gemm_stages(int nt) { return nt == 256 ? 3 : 4; }
constexpr int gemm_smem(int nt) { return gemm_stage(nt) * gemm_stages(nt) + 1024; }

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tmem_add16(uint32_t taddr, float* acc) {
  uint32_t v[16];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                 "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
               : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] += __uint_as_float(v[i]);
}
// K-major, 64-byte swizzle operand descriptor: rows of 64 B, 8-row groups 512 B apart.
__device__ __forceinline__ uint64_t make_desc64(uint32_t addr) {
  const uint32_t lo = ((addr & 0x3FFFFu) >> 4) | (1u << 16);
  const uint32_t hi = (512u >> 4) | (1u << 14) | (4u << 29);
  return ((uint64_t)hi << 32) | lo;
}

template <int NT, bool SYM>
__global__ void __launch_bounds__(kGemmThreads, 1) k_split_gemm(const uint8_t* __restrict__ a, const uint8_t* __restrict__ b, int nkb,
                                                                 float* __restrict__ c, int ldc, bool add, int* status) {
  constexpr int S = gemm_stages(NT), kStage = gemm_stage(NT), kA = kSplitBlock, kPlaneB = NT * 64;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[S], empty[S], d0_full, d0_free, d1_full;
  __shared__ uint32_t tmem_s;
  const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int by = blockIdx.y, bx = blockIdx.x;
  if (SYM) {                                         // tile number -> (row, column <= row)
    by = (int)((sqrtf(8.f * bx + 1.f) - 1.f) * 0.5f);
    while ((by + 1) * (by + 2) / 2 <= bx) ++by;
    while (by * (by + 1) / 2 > bx) --by;
    bx -= by * (by + 1) / 2;
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
    mbar_init(&d0_full, 1); mbar_init(&d0_free, 16); mbar_init(&d1_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {                                   // high x high in columns [0, NT), the rest in [NT, 2 NT)
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)), "r"(2u * NT) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_s;

  if (warp == 0) {
    if (lane == 0) {
      const uint8_t* ap = a + (int64_t)by * nkb * kSplitBlock;
      const uint8_t* bp = b + (int64_t)bx * (NT / kSplitRows) * nkb * kSplitBlock;
      int s = 0, wrap = 0, it = 0;
      bool ok = true;
      for (; it < nkb; ++it) {
        if (wrap > 0 && !mbar_wait(empty + s, (wrap - 1) & 1, status)) { ok = false; break; }
        const uint32_t at = smem + s * kStage, bar = smem_u32(full + s);
        mbar_expect_tx_a(bar, kStage);
        bulk_g2s_a(at, ap + (int64_t)it * kSplitBlock, kSplitBlock, bar);
        if (NT == kSplitRows) {
          bulk_g2s_a(at + kA, bp + (int64_t)it * kSplitBlock, kSplitBlock, bar);
        } else {                                     // a plane of both row blocks, one behind the other
#pragma unroll
          for (int q = 0; q < 6; ++q)
            bulk_g2s_a(at + kA + (q >> 1) * kPlaneB + (q & 1) * kSplitPlane, bp + ((int64_t)(q & 1) * nkb + it) * kSplitBlock + (q >> 1) * kSplitPlane, kSplitPlane, bar);
        }
        if (++s == S) { s = 0; ++wrap; }
      }
      if (!ok) {                                     // gave up: what is in flight lands first
        const int issued = it < S ? it : S;
        for (int i = 0; i < issued; ++i) {
          const int at_it = it - 1 - i, slot = at_it % S;
          const unsigned long long t0 = globaltimer_ns();
          while (!mbar_try_wait(full + slot, (at_it / S) & 1) && globaltimer_ns() - t0 < 2000000ull) __nanosleep(200);
        }
      }
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == 1) {
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) | ((128u >> 4) << 24);      // fp32 += bf16 x bf16
    const bool elected = elect_one();
    const uint64_t a0 = make_desc64(smem), b0 = make_desc64(smem + kA);
    constexpr uint32_t pa = kSplitPlane >> 4, pb = kPlaneB >> 4;
    bool ok = true;
    uint32_t s = 0, ph = 0;
    for (int it = 0, pos = 0; it < nkb; ++it) {
      if (!mbar_try_wait_a(smem_u32(full + s), ph)) ok = mbar_wait(full + s, ph, status);
      if (ok && pos == 0 && it > 0) ok = mbar_wait(&d0_free, (it / kChunk - 1) & 1, status);
      if (!__all_sync(0xffffffffu, ok)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t ad = a0 + s * (kStage >> 4), bd = b0 + s * (kStage >> 4);
      const bool last = pos == kChunk - 1 || it == nkb - 1;
      if (elected) {
#pragma unroll
        for (int k = 0; k < 2; ++k) umma_bf16(tmem, ad + 2 * k, bd + 2 * k, idesc, pos > 0 || k > 0 ? 1u : 0u);
        if (last) umma_commit(&d0_full);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          umma_bf16(tmem + NT, ad + 2 * k, bd + pb + 2 * k, idesc, it > 0 || k > 0 ? 1u : 0u);
          umma_bf16(tmem + NT, ad + pa + 2 * k, bd + 2 * k, idesc, 1u);
          umma_bf16(tmem + NT, ad + 2 * k, bd + 2 * pb + 2 * k, idesc, 1u);
          umma_bf16(tmem + NT, ad + 2 * pa + 2 * k, bd + 2 * k, idesc, 1u);
          umma_bf16(tmem + NT, ad + pa + 2 * k, bd + pb + 2 * k, idesc, 1u);
        }
        umma_commit(empty + s);
      }
      if (++pos == kChunk) pos = 0;
      if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
    }
    if (elected) umma_commit(&d1_full);
    __syncwarp();
  } else if (warp >= 4) {
    constexpr int W = NT / 4;                        // columns of a warp: a quarter of the tile's, of the 32 rows its number selects
    const int lq = warp & 3, cg = (warp - 4) >> 2;
    const uint32_t at = tmem + ((uint32_t)(lq * 32) << 16) + cg * W;
    float acc[W];
#pragma unroll
    for (int i = 0; i < W; ++i) acc[i] = 0.f;
    bool ok = true;
    const int chunks = (nkb + kChunk - 1) / kChunk;
    for (int ch = 0; ch < chunks && ok; ++ch) {
      ok = mbar_wait_warp_fast(&d0_full, ch & 1, status, lane);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int i = 0; i < W; i += 16) tmem_add16(at + i, acc + i);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&d0_free)) : "memory");
    }
    if (ok) ok = mbar_wait_warp_fast(&d1_full, 0, status, lane);
    if (ok) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int i = 0; i < W; i += 16) tmem_add16(at + NT + i, acc + i);
      const int64_t row = (int64_t)by * 128 + lq * 32 + lane, col = (int64_t)bx * NT + cg * W;
      float4* to = reinterpret_cast<float4*>(c + row * ldc + col);
      if (add) {
#pragma unroll
        for (int i = 0; i < W / 4; ++i) {
          const float4 o = to[i];
          acc[4 * i] += o.x; acc[4 * i + 1] += o.y; acc[4 * i + 2] += o.z; acc[4 * i + 3] += o.w;
        }
      }
#pragma unroll
      for (int i = 0; i < W / 4; ++i) to[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
      if (SYM && by != bx) {
#pragma unroll
        for (int i = 0; i < W; ++i) c[(col + i) * ldc + row] = acc[i];
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2u * NT) : "memory");
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

}  // namespace eora
