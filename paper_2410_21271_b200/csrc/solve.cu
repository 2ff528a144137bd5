// Offline EoRA solve (Algorithm 1, steps 1-6) on the GPU; the interface and the mathematics are in eora_solve.h.
//
//   1.  dW = W - W^                                                    (k_split_rows, on the way to its three parts)
//   2-4 the paper projects dW into the eigenspace of X~ X~^T, dW' = dW Q sqrt(L).  Only dW' dW'^T = P P^T with P = dW X~
//       (d x n) is needed here.
//   5.  top-r eigenpairs (U', S'^2) of P P^T by subspace iteration on m = r + oversample vectors:
//         Y = C Q;  Q = orth(Y)  by Cholesky-QR (Gram matrix, factor and substitution in fp64);  repeated `iters` times, or by
//       default fourteen times, the last ten of them with a Chebyshev filter (see eora_solve).
//       C is the smaller of P P^T (d x d) and P^T P (n x n), whose leading eigenvectors P carries into each other.  Then a
//       Rayleigh-Ritz step in the d-dimensional basis Y:  H = (P^T Y)^T (P^T Y)  (m x m, fp64),  H = V diag(lam) V^T by
//       one-sided Jacobi,  U' = Y V[:, top r],  S' = sqrt(lam)
//   6.  B' = U' S',  A = S'^{-1} U'^T dW
//
// The products are fp32 in accuracy, because the quality of the eigenvectors near the cut depends on the small differences between
// neighbouring eigenvalues: on the tensor cores with three bf16 numbers per value (solve_gemm.cu), or, small ones and those with the
// result's r columns, on the CUDA cores.  All matrices are padded with zeros to whole tiles, so there is one form of each product.  The
// (r + oversample)^2 problems run in fp64.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include "../../include/eora_linear.h"
#include "../../include/eora_solve.h"
#include "solve_gemm.cuh"

namespace {

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ------------------------------------------------------------------------------------------------ SGEMM
constexpr int BM = 128, BN = 128, BKS = 16, PAD = 4;

// C[M][N] (ldc) = sum_p opA[m][p] opB[p][n];  opA[m][p] = ta ? A[p * lda + m] : A[m * lda + p];
// opB[p][n] = tb ? B[n * ldb + p] : B[p * ldb + n].  Out-of-range elements read as zero.
__global__ void __launch_bounds__(256) k_sgemm(int M, int N, int P, const float* __restrict__ A, int lda, int ta,
                                               const float* __restrict__ B, int ldb, int tb, float* __restrict__ C, int ldc) {
  __shared__ float As[BKS][BM + PAD];
  __shared__ float Bs[BKS][BN + PAD];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  for (int p0 = 0; p0 < P; p0 += BKS) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = t + 256 * i;
      {
        const int m = ta ? (e & (BM - 1)) : (e >> 4), p = ta ? (e >> 7) : (e & 15);
        const int gm = m0 + m, gp = p0 + p;
        float v = 0.f;
        if (gm < M && gp < P) v = ta ? A[(int64_t)gp * lda + gm] : A[(int64_t)gm * lda + gp];
        As[p][m] = v;
      }
      {
        const int n = tb ? (e >> 4) : (e & (BN - 1)), p = tb ? (e & 15) : (e >> 7);
        const int gn = n0 + n, gp = p0 + p;
        float v = 0.f;
        if (gn < N && gp < P) v = tb ? B[(int64_t)gn * ldb + gp] : B[(int64_t)gp * ldb + gn];
        Bs[p][n] = v;
      }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < BKS; ++p) {
      float a[8], b[8];
      const float4 a0 = *reinterpret_cast<const float4*>(&As[p][ty * 4]), a1 = *reinterpret_cast<const float4*>(&As[p][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[p][tx * 4]), b1 = *reinterpret_cast<const float4*>(&Bs[p][64 + tx * 4]);
      a[0] = a0.x; a[1] = a0.y; a[2] = a0.z; a[3] = a0.w; a[4] = a1.x; a[5] = a1.y; a[6] = a1.z; a[7] = a1.w;
      b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w; b[4] = b1.x; b[5] = b1.y; b[6] = b1.z; b[7] = b1.w;
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int gm = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4);
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int gn = n0 + (j < 4 ? tx * 4 + j : 64 + tx * 4 + j - 4);
      if (gn < N) C[(int64_t)gm * ldc + gn] = acc[i][j];
    }
  }
}

// Two fp32 fused multiply-adds per instruction (the pair of neighbouring columns).
__device__ __forceinline__ void ffma2(float2& d, const float2& a, const float2& b) {
  unsigned long long& dd = reinterpret_cast<unsigned long long&>(d);
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(dd) : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
}

// The same product for whole tiles, nothing transposed (M, N multiples of 128, P of 16, rows 16-byte aligned): 16-byte global loads, the
// next k-slice fetched into registers while the current one is multiplied, 8 x 8 outputs per thread.
__global__ void __launch_bounds__(256, 2) k_sgemm_full(int P, const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
                                                    float* __restrict__ C, int ldc) {
  __shared__ __align__(16) float As[2][BKS][BM + PAD];
  __shared__ __align__(16) float Bs[2][BKS][BN + PAD];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  // this thread's two 16-byte pieces of each operand tile: A 128 rows x 16 p, 4 pieces per row; B 16 p x 128 columns, 32 pieces per p
  int a_r[2], a_c[2], b_r[2], b_c[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int e = t + 256 * i;
    a_r[i] = e >> 2; a_c[i] = (e & 3) * 4;
    b_r[i] = e >> 5; b_c[i] = (e & 31) * 4;
  }
  auto load_a = [&](int p0, int i) -> float4 { return *reinterpret_cast<const float4*>(A + (int64_t)(m0 + a_r[i]) * lda + p0 + a_c[i]); };
  auto load_b = [&](int p0, int i) -> float4 { return *reinterpret_cast<const float4*>(B + (int64_t)(p0 + b_r[i]) * ldb + n0 + b_c[i]); };
  auto store_a = [&](int buf, int i, const float4& v) {
    As[buf][a_c[i]][a_r[i]] = v.x; As[buf][a_c[i] + 1][a_r[i]] = v.y; As[buf][a_c[i] + 2][a_r[i]] = v.z; As[buf][a_c[i] + 3][a_r[i]] = v.w;
  };
  auto store_b = [&](int buf, int i, const float4& v) { *reinterpret_cast<float4*>(&Bs[buf][b_r[i]][b_c[i]]) = v; };
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  float4 ra[2], rb[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) { ra[i] = load_a(0, i); rb[i] = load_b(0, i); }
#pragma unroll
  for (int i = 0; i < 2; ++i) { store_a(0, i, ra[i]); store_b(0, i, rb[i]); }
  __syncthreads();
  int buf = 0;
  for (int p0 = 0; p0 < P; p0 += BKS) {
    const bool more = p0 + BKS < P;
    if (more) {
#pragma unroll
      for (int i = 0; i < 2; ++i) { ra[i] = load_a(p0 + BKS, i); rb[i] = load_b(p0 + BKS, i); }
    }
#pragma unroll
    for (int p = 0; p < BKS; ++p) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][p][ty * 4]), a1 = *reinterpret_cast<const float4*>(&As[buf][p][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][p][tx * 4]), b1 = *reinterpret_cast<const float4*>(&Bs[buf][p][64 + tx * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 aa = make_float2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) ffma2(acc[i][j], aa, b[j]);
      }
    }
    if (more) {
#pragma unroll
      for (int i = 0; i < 2; ++i) { store_a(buf ^ 1, i, ra[i]); store_b(buf ^ 1, i, rb[i]); }
    }
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float* row = C + (int64_t)(m0 + (i & 3) + ty * 4 + (i & 4) * 16) * ldc + n0;
    *reinterpret_cast<float4*>(row + tx * 4) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
    *reinterpret_cast<float4*>(row + 64 + tx * 4) = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
  }
}

// Skinny products C[M][ldc] = op(A) B with B [P][ldb] of a few hundred columns (the iterates): M a multiple of 64, P of 16 times the
// cluster size; opA[m][p] = TA ? A[p * lda + m] : A[m * lda + p].  A cluster owns a tile of 64 rows x 16 NC columns and splits P; the
// partial sums meet in distributed shared memory and are added in a fixed order, so the result does not depend on timing.
// 4 x NC outputs per thread (two instructions' worth of shared-memory reads per ten of arithmetic at NC = 10; 2 x 10 was bound
// by the reads), and enough CTAs without padding columns: 2048 x 2048 x 160 are 32 tiles, 128 CTAs.
// shift (may be null; op(A) square): C = op(A) B - *shift B.
template <int NC, bool TA>
__global__ void __launch_bounds__(256) k_skinny(int P, const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
                                                float* __restrict__ C, int ldc, const float* __restrict__ shift) {
  constexpr int W = 16 * NC, NP = NC / 2, RM = 64;
  constexpr int BQ = (BKS * W / 4 + 255) / 256;      // 16-byte pieces of the B slice per thread
  constexpr int kAb = 2 * BKS * (RM + PAD), kBb = 2 * BKS * (W + PAD), kSm = kAb + kBb > RM * W ? kAb + kBb : RM * W;
  __shared__ __align__(16) float sm[kSm];
  float (*As)[BKS][RM + PAD] = reinterpret_cast<float (*)[BKS][RM + PAD]>(sm);
  float (*Bs)[BKS][W + PAD] = reinterpret_cast<float (*)[BKS][W + PAD]>(sm + kAb);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int ks = gridDim.x, rank = blockIdx.x, m0 = blockIdx.y * RM, n0 = blockIdx.z * W;
  const int span = P / ks, lo = rank * span;
  const int a_r = TA ? t >> 4 : t >> 2, a_c = TA ? (t & 15) * 4 : (t & 3) * 4;
  auto load_a = [&](int p0) -> float4 {
    return TA ? __ldg(reinterpret_cast<const float4*>(A + (int64_t)(p0 + a_r) * lda + m0 + a_c))
              : __ldg(reinterpret_cast<const float4*>(A + (int64_t)(m0 + a_r) * lda + p0 + a_c));
  };
  auto store_a = [&](int buf, const float4& v) {
    if (TA) *reinterpret_cast<float4*>(&As[buf][a_r][a_c]) = v;
    else { As[buf][a_c][a_r] = v.x; As[buf][a_c + 1][a_r] = v.y; As[buf][a_c + 2][a_r] = v.z; As[buf][a_c + 3][a_r] = v.w; }
  };
  auto has_b = [&](int i) { return (i + 1) * 256 <= BKS * W / 4 || t + 256 * i < BKS * W / 4; };
  auto load_b = [&](int p0, int i) -> float4 {
    const int e = t + 256 * i;
    return __ldg(reinterpret_cast<const float4*>(B + (int64_t)(p0 + e / (W / 4)) * ldb + n0 + (e % (W / 4)) * 4));
  };
  auto store_b = [&](int buf, int i, const float4& v) { const int e = t + 256 * i; *reinterpret_cast<float4*>(&Bs[buf][e / (W / 4)][(e % (W / 4)) * 4]) = v; };
  // columns of a thread: four of every 64, two of a last 32
  float2 acc[4][NP];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NP; ++j) acc[i][j] = make_float2(0.f, 0.f);
  float4 ra = load_a(lo), rb[BQ];
#pragma unroll
  for (int i = 0; i < BQ; ++i) if (has_b(i)) rb[i] = load_b(lo, i);
  store_a(0, ra);
#pragma unroll
  for (int i = 0; i < BQ; ++i) if (has_b(i)) store_b(0, i, rb[i]);
  __syncthreads();
  int buf = 0;
  for (int p0 = lo; p0 < lo + span; p0 += BKS) {
    const bool more = p0 + BKS < lo + span;
    if (more) {
      ra = load_a(p0 + BKS);
#pragma unroll
      for (int i = 0; i < BQ; ++i) if (has_b(i)) rb[i] = load_b(p0 + BKS, i);
    }
#pragma unroll
    for (int p = 0; p < BKS; ++p) {
      const float4 a = *reinterpret_cast<const float4*>(&As[buf][p][ty * 4]);
      float2 b[NP];
#pragma unroll
      for (int c = 0; c < NC / 4; ++c) {
        const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][p][64 * c + tx * 4]);
        b[2 * c] = make_float2(v.x, v.y); b[2 * c + 1] = make_float2(v.z, v.w);
      }
      if (NC % 4) b[NP - 1] = *reinterpret_cast<const float2*>(&Bs[buf][p][64 * (NC / 4) + tx * 2]);
      const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 aa = make_float2(av[i], av[i]);
#pragma unroll
        for (int j = 0; j < NP; ++j) ffma2(acc[i][j], aa, b[j]);
      }
    }
    if (more) {
      store_a(buf ^ 1, ra);
#pragma unroll
      for (int i = 0; i < BQ; ++i) if (has_b(i)) store_b(buf ^ 1, i, rb[i]);
    }
    __syncthreads();
    buf ^= 1;
  }
  auto col = [&](int j) { return j / 2 < NC / 4 ? 64 * (j / 2) + tx * 4 + 2 * (j & 1) : 64 * (NC / 4) + tx * 2; };
  const float rho = shift ? *shift : 0.f;
  if (ks == 1) {
    if (shift) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          const float2 q = *reinterpret_cast<const float2*>(B + (int64_t)(m0 + ty * 4 + i) * ldb + n0 + col(j));
          acc[i][j].x = fmaf(-rho, q.x, acc[i][j].x); acc[i][j].y = fmaf(-rho, q.y, acc[i][j].y);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < NP; ++j) *reinterpret_cast<float2*>(C + (int64_t)(m0 + ty * 4 + i) * ldc + n0 + col(j)) = acc[i][j];
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NP; ++j) *reinterpret_cast<float2*>(sm + (ty * 4 + i) * W + col(j)) = acc[i][j];
  cluster_sync_all();
  const int per = RM / ks;                           // rows of the tile that this CTA adds up
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm) + rank * per * W * 4;
  for (int e = t; e < per * W / 4; e += 256) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r = 0; r < ks; ++r) {
      float4 u;
      uint32_t a;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(base + 16 * e), "r"(r));
      asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(u.x), "=f"(u.y), "=f"(u.z), "=f"(u.w) : "r"(a));
      v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
    }
    const int row = m0 + rank * per + e / (W / 4), at = n0 + (e % (W / 4)) * 4;
    if (shift) {
      const float4 q = *reinterpret_cast<const float4*>(B + (int64_t)row * ldb + at);
      v.x = fmaf(-rho, q.x, v.x); v.y = fmaf(-rho, q.y, v.y); v.z = fmaf(-rho, q.z, v.z); v.w = fmaf(-rho, q.w, v.w);
    }
    *reinterpret_cast<float4*>(C + (int64_t)row * ldc + at) = v;
  }
  cluster_sync_all();                                // nobody leaves while its sums are being read
}

template <int NC, bool TA>
cudaError_t launch_skinny(cudaStream_t st, int M, int P, const float* A, int lda, const float* B, int ldb, int N, float* C, int ldc, const float* shift) {
  // as many CTAs per tile as there is room for (two per SM), each with at least eight slices of P
  const int tiles = M / 64 * (N / (16 * NC));
  int ks = 4;
  while (ks > 1 && (tiles * ks > 300 || P % (BKS * ks) || P / ks < 8 * BKS)) ks >>= 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ks, M / 64, N / (16 * NC));
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_skinny<NC, TA>, P, A, lda, B, ldb, C, ldc, shift);
}
// N: a multiple of the width `w` (64, 96, 128 or 160) that make_plan chose.
template <bool TA>
cudaError_t skinny(cudaStream_t st, int w, int M, int P, const float* A, int lda, const float* B, int ldb, int N, float* C, int ldc, const float* shift = nullptr) {
  switch (w) {
    case 64: return launch_skinny<4, TA>(st, M, P, A, lda, B, ldb, N, C, ldc, shift);
    case 96: return launch_skinny<6, TA>(st, M, P, A, lda, B, ldb, N, C, ldc, shift);
    case 128: return launch_skinny<8, TA>(st, M, P, A, lda, B, ldb, N, C, ldc, shift);
    default: return launch_skinny<10, TA>(st, M, P, A, lda, B, ldb, N, C, ldc, shift);
  }
}

// The general product (the loss check: any sizes).
cudaError_t sgemm(cudaStream_t st, int M, int N, int P, const float* A, int lda, bool ta, const float* B, int ldb, bool tb, float* C, int ldc) {
  dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
  const bool full = !ta && !tb && M % BM == 0 && N % BN == 0 && P % BKS == 0 && lda % 4 == 0 && ldb % 4 == 0 && ldc % 4 == 0 &&
                    ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) | reinterpret_cast<uintptr_t>(C)) & 15) == 0;
  if (full) k_sgemm_full<<<grid, 256, 0, st>>>(P, A, lda, B, ldb, C, ldc);
  else k_sgemm<<<grid, 256, 0, st>>>(M, N, P, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, C, ldc);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------ small pieces
__global__ void k_sub(const float* __restrict__ a, const float* __restrict__ b, float* __restrict__ c, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) c[i] = a[i] - b[i];
}
// A fixed start for the iteration: values in (-1, 1) from a counter hash (any full-rank start converges).  The iterate
// is stored with a leading dimension ld >= m and rows_p >= rows rows (whole tiles); the padding is zero and stays zero.
__global__ void k_init(float* y, int rows, int rows_p, int m, int ld) {
  const int64_t n = (int64_t)rows_p * ld;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t z = (uint64_t)i * 0x9E3779B97F4A7C15ull + 0xD1B54A32D192ED03ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    y[i] = (int)(i % ld) < m && i / ld < rows ? (float)((double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0) : 0.f;
  }
}

// S[i][j] = sum_row A[row][i] A[row][j] for a [rows][m] fp32 matrix, products and sums in fp64, lower triangle.
// One CTA per 32 x 32 block on or below the diagonal and per part of the rows (blockIdx.y; `chunk` rows each), 2 x 2 elements per
// thread; slices of 32 rows go through shared memory as fp64 (every element is converted once per CTA: a conversion per operand of
// every product is what bounded the earlier form, 64 us for 4096 x 160).  Part z writes its sums to parts[z][m][m]; k_sum_parts adds
// the parts in a fixed order, so the result does not depend on the order the CTAs ran in.
constexpr int kGramParts = 32;
__global__ void __launch_bounds__(256) k_gram64(const float* __restrict__ A, int rows, int chunk, int m, int ld, double* __restrict__ parts) {
  __shared__ __align__(16) double sa[32][34], sb[32][34];
  int bi = (int)((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((bi + 1) * (bi + 2) / 2 <= (int)blockIdx.x) ++bi;
  while (bi * (bi + 1) / 2 > (int)blockIdx.x) --bi;
  const int bj = blockIdx.x - bi * (bi + 1) / 2;
  const int t = threadIdx.x, ti = t >> 4, tj = t & 15, lr = t >> 3, lc = (t & 7) * 4;
  const int r_lo = blockIdx.y * chunk, r_hi = min(rows, r_lo + chunk);
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = va;
  // (ld is a multiple of 32 and the columns past m are zero, so whole pieces can be read)
  auto fetch = [&](int r0) {
    const int rr = r0 + lr;
    va = vb = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rr < r_hi) {
      va = *reinterpret_cast<const float4*>(A + (int64_t)rr * ld + bi * 32 + lc);
      vb = *reinterpret_cast<const float4*>(A + (int64_t)rr * ld + bj * 32 + lc);
    }
  };
  fetch(r_lo);
  for (int r0 = r_lo; r0 < r_hi; r0 += 32) {
    sa[lr][lc] = va.x; sa[lr][lc + 1] = va.y; sa[lr][lc + 2] = va.z; sa[lr][lc + 3] = va.w;
    sb[lr][lc] = vb.x; sb[lr][lc + 1] = vb.y; sb[lr][lc + 2] = vb.z; sb[lr][lc + 3] = vb.w;
    __syncthreads();
    fetch(r0 + 32);
#pragma unroll 8
    for (int r = 0; r < 32; ++r) {
      const double2 a = *reinterpret_cast<const double2*>(&sa[r][2 * ti]), b = *reinterpret_cast<const double2*>(&sb[r][2 * tj]);
      acc[0][0] = fma(a.x, b.x, acc[0][0]); acc[0][1] = fma(a.x, b.y, acc[0][1]);
      acc[1][0] = fma(a.y, b.x, acc[1][0]); acc[1][1] = fma(a.y, b.y, acc[1][1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int gi = bi * 32 + 2 * ti + i, gj = bj * 32 + 2 * tj + j;
      if (gi < m && gj <= gi) parts[((int64_t)blockIdx.y * m + gi) * m + gj] = acc[i][j];
    }
}
// The parts' sum; MIRROR: both triangles, else the lower one.
template <bool MIRROR>
__global__ void k_sum_parts(const double* __restrict__ parts, int n_parts, int m, double* __restrict__ S) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = e / m, j = e - i * m;
  if (i >= m || j > i) return;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  int z = 0;
  for (; z + 4 <= n_parts; z += 4)
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] += parts[((int64_t)(z + k) * m + i) * m + j];
  for (; z < n_parts; ++z) v[0] += parts[((int64_t)z * m + i) * m + j];
  const double sum = (v[0] + v[1]) + (v[2] + v[3]);
  S[(int64_t)i * m + j] = sum;
  if (MIRROR) S[(int64_t)j * m + i] = sum;
}
// S = A^T A over all rows: the parts, then their sum.
template <bool MIRROR>
cudaError_t gram64(cudaStream_t st, const float* A, int rows, int m, int ld, double* parts, double* S) {
  const int nb = (m + 31) / 32, tiles = nb * (nb + 1) / 2;
  int n_parts = (rows + 127) / 128;                  // 128 rows per part, or more where that would be too many
  if (n_parts > kGramParts) n_parts = kGramParts;
  const int chunk = ((rows + n_parts - 1) / n_parts + 31) / 32 * 32;
  n_parts = (rows + chunk - 1) / chunk;
  k_gram64<<<dim3(tiles, n_parts), 256, 0, st>>>(A, rows, chunk, m, ld, parts);
  k_sum_parts<MIRROR><<<(m * m + 255) / 256, 256, 0, st>>>(parts, n_parts, m, S);
  return cudaGetLastError();
}

// The power of two next to 1 / v.
__device__ __forceinline__ float pow2_scale(double v) {
  const int ex = min(max((__double2hiint(v) >> 20) - 1023, -120), 120);
  return __int_as_float((127 - ex) << 23);
}
// 1 / sqrt(d) in fp64 from the fp32 value by Newton's method (each step doubles the digits; the argument's exponent is taken
// out first, so every positive d works).
__device__ __forceinline__ double rsqrt_newton(double d) {
  const int e = (__double2hiint(d) >> 20) - 1023, half = e >> 1;          // d = 2^(2 half) * [1, 4)
  const double x = __hiloint2double(__double2hiint(d) - (half << 21), __double2loint(d));
  double y = (double)rsqrtf((float)x);
#pragma unroll
  for (int i = 0; i < 2; ++i) y = fma(y * 0.5, fma(-x * y, y, 1.0), y);
  return __hiloint2double(__double2hiint(y) - (half << 20), __double2loint(y));
}

// Cholesky S = L L^T (fp64) of an m x m Gram matrix by one CTA, right-looking in panels of 16 columns:
//   (A) one warp factors the 16 x 16 diagonal block in registers (lane = row) and inverts it,
//   (B) the rows below are multiplied with the inverse, one element per thread,
//   (C) the trailing lower triangle is updated in 4 x 4 tiles.  Warp 0 takes the tiles of the next diagonal block first and goes on
//       with (A) for the next panel while the others update the rest.
// The chain of (A)s is what bounds it: a pivot, its root, a column and an update, 16 times per panel.
// Writes L over S (lower triangle, global) and the inverses of the diagonal blocks; Q = Y L^{-T} follows by k_trsm.  Every diagonal
// element first grows by 1e-13 of itself, so that a rank-deficient iterate still factors; relative to itself, because the columns of
// an iterate are graded (column j has about the norm of the j-th eigenvalue, or of its square).
// L0: the whole matrix, rows ld apart; this launch factors the m x m block (m <= kCholSmem, what shared memory holds) whose first row and column
// are j_base, of m_all; least_g: [m_all], the smallest pivots of later blocks.  Larger matrices go block by block (orthonormalise).
constexpr int kCholSmem = 160;
constexpr int kCholThreads = 512;
__host__ __device__ constexpr int pan_pitch(int m) { return (m + 5) / 4 * 4 + 2; }      // (even, and rows of the panel on different banks)
__host__ __device__ constexpr int chol_smem(int m) { return (m * (m | 1) + m + 16 * pan_pitch(m)) * 8 + 16; }
//
// f (may be null): the filter's state.  With prev the iterate went through a pair of products with (C - f->rho[0] I) and (C - f->rho[1] I), starting from
// columns of norm 1 / f->scale, else through one with C: the diagonal of L then says where the eigenvalues of the iterate's columns are.
// The next pair's shifts are lo and hi times the smallest of them.
struct Filter { float rho[2]; double scale; };
constexpr double kFilterEdge = 0.95;                 // the estimate comes from below, but not always (measured 0.8 to 1.07 of eigenvalue m after four steps; 1.3 on a plateau with few extra vectors, where the points then lie a little high and the loss is still half the plain iteration's)
__global__ void __launch_bounds__(kCholThreads) k_chol64(double* L0, int ld, int m_all, int j_base, int m, double* __restrict__ Dinv, double* least_g, Filter* f, bool prev, double lo, double hi) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double dv[16][17];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  double* Sg = L0 + (int64_t)j_base * (ld + 1);
  const int ls = m | 1, lp = pan_pitch(m);
  double* pan = sm;                                  // [16][lp]: the panel by columns
  double* least = sm + 16 * lp;                      // [m]: the smallest pivot of a column that is taken as it is
  double* S = least + m;
  for (int i = warp; i < m; i += 2 * (kCholThreads / 32)) {      // two rows' loads go out together (one at a time each was a round trip to L2: 20 us)
    double v[2][kCholSmem / 32];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int k = 0; k < kCholSmem / 32; ++k) {
        const int r = i + h * (kCholThreads / 32), j = lane + 32 * k;
        v[h][k] = r < m && j <= r ? Sg[(int64_t)r * ld + j] : 0.0;
      }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int k = 0; k < kCholSmem / 32; ++k) {
        const int r = i + h * (kCholThreads / 32), j = lane + 32 * k;
        if (r < m && j <= r) S[r * ls + j] = v[h][k];
      }
  }
  __syncthreads();
  if (j_base == 0) {                                 // (for all blocks: a later one's diagonal is a difference by then)
    for (int i = t; i < m_all; i += kCholThreads) {
      double& d = i < m ? S[(int64_t)i * ls + i] : L0[(int64_t)i * (ld + 1)];
      const double shift = 1e-13 * d + 1e-300;
      d += shift;
      if (i < m) least[i] = 1e-3 * shift; else least_g[i] = 1e-3 * shift;
    }
  } else {
    for (int i = t; i < m; i += kCholThreads) least[i] = least_g[j_base + i];
  }
  __syncthreads();
  auto diagonal = [&](int j0) {                      // (A), one warp; lanes 16..31 repeat lanes 0..15
    const int r = lane & 15, gi = j0 + r;
    double a[16], x[16], rinv = 0.0;
    const double fl = gi < m ? least[gi] : 0.0;
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] = gi < m && q <= r ? S[(int64_t)gi * ls + j0 + q] : (q == r ? 1.0 : 0.0);      // past m: identity
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      double d = __shfl_sync(0xffffffffu, a[k], k);
      const double f = __shfl_sync(0xffffffffu, fl, k);
      d = d > f ? d : f;
      const double ri = rsqrt_newton(d);
      a[k] = r == k ? d * ri : a[k] * ri;            // (rows above k: never read)
      if (r == k) rinv = ri;
#pragma unroll
      for (int c = k + 1; c < 16; ++c) a[c] = fma(-a[k], __shfl_sync(0xffffffffu, a[k], c), a[c]);
    }
    // column r of the inverse by forward substitution
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      double v = i == r ? 1.0 : 0.0, u = 0.0;
#pragma unroll
      for (int q = 0; q < i; ++q) {
        const double l = __shfl_sync(0xffffffffu, a[q], i);
        if (q & 1) u = fma(-l, x[q], u); else v = fma(-l, x[q], v);
      }
      x[i] = (v + u) * __shfl_sync(0xffffffffu, rinv, i);
    }
    if (lane < 16) {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        if (gi < m && q <= r) S[(int64_t)gi * ls + j0 + q] = a[q];
        dv[q][r] = x[q];
        Dinv[(int64_t)(j0 + q) * 16 + r] = x[q];
      }
    }
  };
  if (warp == 0) diagonal(0);
  __syncthreads();
  for (int j0 = 0; j0 < m; j0 += 16) {
    const int j1 = j0 + 16, R = m - j1;
    if (R <= 0) break;
    for (int e = t; e < R * 16; e += kCholThreads) {       // (B)
      const int i = j1 + (e >> 4), c = e & 15;
      const double* ri = S + (int64_t)i * ls + j0;
      double v = 0.0, u = 0.0;
#pragma unroll
      for (int q = 0; q < 16; q += 2) { v = fma(ri[q], dv[c][q], v); u = fma(ri[q + 1], dv[c][q + 1], u); }      // (zeros past c)
      pan[c * lp + i] = v + u;
    }
    __syncthreads();
    const int T = (R + 3) / 4, head = T < 4 ? T * (T + 1) / 2 : 10, tiles = T * (T + 1) / 2;      // the first `head` tiles: the next diagonal block
    auto update = [&](int e) {                              // (C)
      int ti = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
      while ((ti + 1) * (ti + 2) / 2 <= e) ++ti;
      while (ti * (ti + 1) / 2 > e) --ti;
      const int i0 = j1 + 4 * ti, c0 = j1 + 4 * (e - ti * (ti + 1) / 2);
      double acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = 0.0;
#pragma unroll 4
      for (int q = 0; q < 16; ++q) {                        // (the panel's columns are padded: reading past m is in bounds, the sums are not stored)
        const double2 l0 = *reinterpret_cast<const double2*>(pan + q * lp + i0), l1 = *reinterpret_cast<const double2*>(pan + q * lp + i0 + 2);
        const double2 m0 = *reinterpret_cast<const double2*>(pan + q * lp + c0), m1 = *reinterpret_cast<const double2*>(pan + q * lp + c0 + 2);
        const double li[4] = {l0.x, l0.y, l1.x, l1.y}, lc[4] = {m0.x, m0.y, m1.x, m1.y};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[i][c] = fma(li[i], lc[c], acc[i][c]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (i0 + i < m && c0 + c <= i0 + i) S[(int64_t)(i0 + i) * ls + c0 + c] -= acc[i][c];
    };
    if (warp == 0) {
      if (lane < head) update(lane);
      __syncwarp();
      diagonal(j1);                                         // (dv was read in (B))
    } else {
      const int wt = t - 32;
      for (int e = wt; e < R * 16; e += kCholThreads - 32) S[(int64_t)(j1 + (e >> 4)) * ls + j0 + (e & 15)] = pan[(e & 15) * lp + j1 + (e >> 4)];
      for (int e = head + wt; e < tiles; e += kCholThreads - 32) update(e);
    }
    __syncthreads();
  }
  if (f && warp == 0) {
    double least_l = 1e300;
    for (int i = lane; i < m; i += 32) least_l = fmin(least_l, S[(int64_t)i * ls + i]);
    for (int i = lane; i < j_base; i += 32) least_l = fmin(least_l, L0[(int64_t)i * (ld + 1)]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) least_l = fmin(least_l, __shfl_xor_sync(0xffffffffu, least_l, o));
    if (lane == 0) {
      double at = least_l;                           // (x - rho0)(x - rho1) = L f->scale
      if (prev) {
        const double r0 = f->rho[0], r1 = f->rho[1], half = 0.5 * (r0 - r1);
        at = 0.5 * (r0 + r1) + sqrt(half * half + least_l * f->scale);
      }
      f->rho[0] = (float)(lo * kFilterEdge * at); f->rho[1] = (float)(hi * kFilterEdge * at);
      f->scale = 1.0 / (double)pow2_scale(j_base ? L0[0] : S[0]);
    }
  }
  for (int i = warp; i < m; i += kCholThreads / 32)
    for (int j = lane; j <= i; j += 32) Sg[(int64_t)i * ld + j] = S[i * ls + j];
}

// Q = Y L^{-T}, row by row (fp64 inside): a CTA takes 16 rows, half a warp each (lane = column of the panel); panel by panel of 16
// columns  q_p = (y_p - sum_{c < 16 p} q_c L[p][c]^T) Dinv_p^T.  A panel's 16 rows of L and its Dinv come by cp.async, one panel
// ahead, its column of Y by a load one panel ahead.  With `scaled`, Q is divided by the power of two next to L[0][0].
// T: float (an iterate; rows are a multiple of 16 and Q's columns past m become zero) or double (rows of the Gram matrix below a block, in place).
__host__ __device__ constexpr int trsm_pitch(int m) { return (m + 15) / 16 * 16 + 2; }
__host__ __device__ constexpr int trsm_smem(int m) { return (3 * 16 * trsm_pitch(m) + 2 * 16 * 18) * 8; }
template <typename T>
__global__ void __launch_bounds__(256) k_trsm(const T* Y, const double* __restrict__ L, int ll, const double* __restrict__ Dinv, int m, int ld, int rows,
                                              T* Q, bool scaled) {
  extern __shared__ __align__(16) double smt[];
  const int lq = trsm_pitch(m);
  double* qd = smt;                                  // [16][lq]
  double* lp = smt + 16 * lq;                        // [2][16][lq]
  double* di = smt + 48 * lq;                        // [2][16][18]
  const int t = threadIdx.x, r = t >> 4, c = t & 15;
  const int64_t row = (int64_t)blockIdx.x * 16 + r;
  const int np = (m + 15) / 16;
  auto copy8 = [](double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
  };
  auto fetch = [&](int p) {                          // rows 16 p .. of L, columns before 16 p
    double* dst = lp + (p & 1) * 16 * lq;
    copy8(di + (p & 1) * 16 * 18 + r * 18 + c, Dinv + (int64_t)(16 * p + r) * 16 + c);
    for (int q = c; q < 16 * p; q += 16) {
      if (16 * p + r < m) copy8(dst + r * lq + q, L + (int64_t)(16 * p + r) * ll + q);
      else dst[r * lq + q] = 0.0;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0);
  const bool live = row < rows;
  T y = live ? Y[row * ld + c] : (T)0;
  const float scale = scaled ? pow2_scale(L[0]) : 1.f;
  for (int p = 0; p < np; ++p) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                 // panel p is there, and panel p - 1 has been read
    if (p + 1 < np) fetch(p + 1);
    double v[4] = {(double)y, 0.0, 0.0, 0.0};
    if (live && p + 1 < np) y = Y[row * ld + 16 * (p + 1) + c];
    const double* lr = lp + (p & 1) * 16 * lq + c * lq;
    const double* qr = qd + r * lq;
#pragma unroll 4
    for (int q = 0; q < 16 * p; q += 4) {
      const double2 a = *reinterpret_cast<const double2*>(qr + q), b = *reinterpret_cast<const double2*>(lr + q);
      const double2 a2 = *reinterpret_cast<const double2*>(qr + q + 2), b2 = *reinterpret_cast<const double2*>(lr + q + 2);
      v[0] = fma(-a.x, b.x, v[0]); v[1] = fma(-a.y, b.y, v[1]); v[2] = fma(-a2.x, b2.x, v[2]); v[3] = fma(-a2.y, b2.y, v[3]);
    }
    const double w = (v[0] + v[1]) + (v[2] + v[3]);
    const double* dr = di + (p & 1) * 16 * 18 + c * 18;
    double o[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 16; ++q) o[q & 3] = fma(__shfl_sync(0xffffffffu, w, q, 16), dr[q], o[q & 3]);      // (Dinv is lower triangular: zeros past c)
    const double res = (o[0] + o[1]) + (o[2] + o[3]);
    qd[r * lq + 16 * p + c] = res;
    if (live) Q[row * ld + 16 * p + c] = (T)res * (T)scale;
    __syncwarp();
  }
  if constexpr (sizeof(T) == 4)
    for (int i = 16 * np + c; i < ld; i += 16) Q[row * ld + i] = 0.f;
}

// S22 -= L21 L21^T, lower triangle: rows [j1, m) of the matrix, the block's columns [j0, j1) (a multiple of 32 of them).  One CTA per 32 x 32 tile.
__global__ void __launch_bounds__(256) k_syrk64(double* __restrict__ S, int ld, int m, int j0, int j1) {
  __shared__ double sa[32][33], sb[32][33];
  int bi = (int)((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((bi + 1) * (bi + 2) / 2 <= (int)blockIdx.x) ++bi;
  while (bi * (bi + 1) / 2 > (int)blockIdx.x) --bi;
  const int bj = blockIdx.x - bi * (bi + 1) / 2;
  const int t = threadIdx.x, x = t & 31, y = t >> 5, ti = t >> 4, tj = t & 15;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int q0 = j0; q0 < j1; q0 += 32) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = j1 + bi * 32 + y + 8 * k, j = j1 + bj * 32 + y + 8 * k;
      sa[y + 8 * k][x] = i < m ? S[(int64_t)i * ld + q0 + x] : 0.0;
      sb[y + 8 * k][x] = j < m ? S[(int64_t)j * ld + q0 + x] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int q = 0; q < 32; ++q) {
      const double a0 = sa[2 * ti][q], a1 = sa[2 * ti + 1][q], b0 = sb[2 * tj][q], b1 = sb[2 * tj + 1][q];
      acc[0][0] = fma(a0, b0, acc[0][0]); acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]); acc[1][1] = fma(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int gi = j1 + bi * 32 + 2 * ti + i, gj = j1 + bj * 32 + 2 * tj + j;
      if (gi < m && gj <= gi) S[(int64_t)gi * ld + gj] -= acc[i][j];
    }
}

// Symmetric positive semi-definite eigenproblem H = V diag(lam) V^T, m x m, fp64, by one-sided (Hestenes) Jacobi: pairs of
// columns of H are rotated until they are orthogonal.  With J the product of the rotations the result is H J = V diag(lam): column i
// has norm lam_i and direction v_i, so the eigenvectors are the normalised columns and no separate accumulation of the
// rotations is needed (a column whose norm is zero up to rounding has no direction; its eigenvalue is far below the kept ones).
//
// A warp holds two blocks of B columns in registers (E elements of each per lane); blocks meet by the round-robin tournament
// and travel between the warps of a cluster through distributed shared memory, one cluster barrier per meeting.  In a
// meeting every column of one block is rotated against every column of the other, B disjoint pairs at a time whose latencies
// overlap; the pairs inside a block take their turn once per sweep.  Squared norms are carried along (recomputed every
// sweep), so a rotation needs one dot product.  The angle is computed in fp32 -- a rotation by a slightly different angle is
// still a rotation, and the next sweep works on what it left -- its cosine in fp64.  The last sweep is the one that finds every pair
// orthogonal to 1e-8 before it rotates them (convergence is quadratic by then, and the results are fp32).  One CTA that kept the columns in shared
// memory and went through it for every pair took 4.5 ms at m = 160.
template <int B, int E>
struct JacobiShape {
  static constexpr int kElems = 32 * E;              // elements per column (>= m, zero-padded)
  static constexpr int kBlock = B * kElems + B;      // doubles of a block: its columns, their squared norms
};
template <int B, int E>
__global__ void __launch_bounds__(B == 4 ? 160 : 320, 1) k_jacobi_cl(const double* __restrict__ Hg, int m, double* lam, float* __restrict__ Vf, int ldv, int max_sweeps) {
  using Sh = JacobiShape<B, E>;
  extern __shared__ __align__(16) double smj[];      // [2 buffers][warps][2 sides][B][kElems]
  __shared__ int moved_s[2];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
  const int cs = gridDim.x, rank = blockIdx.x, G = cs * nw, g = rank * nw + warp;      // groups of the tournament, this warp's
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(smj);
  const uint32_t buf_b = (uint32_t)nw * 2 * Sh::kBlock * 8;
  // scale so that the largest norm is about one (a power of two: exact)
  double tr = 0.0;
  for (int i = lane; i < m; i += 32) tr += Hg[(int64_t)i * m + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
  int ex = 0;
  if (tr > 0.0) frexp(tr, &ex);
  const double down = ldexp(1.0, -ex), up = ldexp(1.0, ex);
  double h[2][B][E], nrm[2][B];
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int col = (2 * g + s) * B + b;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = lane + 32 * e;
        h[s][b][e] = col < m && i < m ? Hg[(int64_t)col * m + i] * down : 0.0;
      }
    }
  if (t < 2) moved_s[t] = 0;
  constexpr double kStop = 1e-16;
  int any = 0;
  auto norms = [&]() {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int b = 0; b < B; ++b) {
        double v = 0.0;
#pragma unroll
        for (int e = 0; e < E; ++e) v = fma(h[s][b][e], h[s][b][e], v);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        nrm[s][b] = v;
      }
  };
  auto rotate = [&](double (&x)[E], double (&y)[E], double& al, double& be, double ga) {
    if (ga * ga <= 1e-22 * al * be) return;          // orthogonal far beyond what the fp32 operands carry
    if (ga * ga > kStop * al * be) any = 1;
    // both scaled by one power of two, so that fp32 neither overflows nor loses what is small
    const double zd = be - al, wd = 2.0 * ga;
    const int e_max = max(__double2hiint(zd) & 0x7ff00000, __double2hiint(wd) & 0x7ff00000);
    if (e_max < 0x01000000) return;
    const double unit = __hiloint2double(0x7fe00000 - e_max, 0);
    const float z = (float)(zd * unit), w = (float)(wd * unit);
    const float tf = copysignf(w / (fabsf(z) + sqrtf(fmaf(z, z, w * w))), z >= 0.f ? w : -w);
    const double tt = (double)tf, c = rsqrt(fma(tt, tt, 1.0)), sn = c * tt;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const double a = x[e], b = y[e];
      x[e] = c * a - sn * b;
      y[e] = fma(sn, a, c * b);
    }
    // exact for any angle: |c a - s b|^2 = c^2 al - 2 c s ga + s^2 be
    const double c2 = c * c, s2 = sn * sn, cs2 = 2.0 * c * sn * ga, na = c2 * al - cs2 + s2 * be, nb = s2 * al + cs2 + c2 * be;
    al = na > 0.0 ? na : 0.0; be = nb > 0.0 ? nb : 0.0;
  };
  auto dot = [&](const double (&x)[E], const double (&y)[E]) {
    double v = 0.0;
#pragma unroll
    for (int e = 0; e < E; ++e) v = fma(x[e], y[e], v);
    return v;
  };
  cluster_sync_all();
  int flip = 0, sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    any = 0;
    norms();
    if (B > 1) {                                     // the pairs inside the blocks: rounds of B / 2 disjoint pairs in each
#pragma unroll
      for (int k = 1; k < B; ++k) {
        double ga[2][B];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int b = 0; b < B; ++b) if ((b ^ k) > b) ga[s][b] = dot(h[s][b], h[s][b ^ k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int b = 0; b < B; ++b) if ((b ^ k) > b) ga[s][b] += __shfl_xor_sync(0xffffffffu, ga[s][b], o);
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int b = 0; b < B; ++b) if ((b ^ k) > b) rotate(h[s][b], h[s][b ^ k], nrm[s][b], nrm[s][b ^ k], ga[s][b]);
      }
    }
    // Meetings.  The B disjoint pairs of a round are dealt to B groups of lanes: their dot products are reduced into the groups
    // (6 shuffles instead of 20 for B = 4), every group computes its pair's angle, all at the same time and without a branch, and
    // keeps the squared norms of its two columns; cosines and sines are then read from the groups.  One pair after the other, each
    // behind a branch, a round took 2.5 times as long.
    constexpr int GL = 32 / B;                       // lanes of a group
    const int pb = lane / GL;
    double al = nrm[0][0], be = nrm[1][0];           // of column pb of the one block and column (pb + k) % B of the other
#pragma unroll
    for (int b = 1; b < B; ++b) if (pb == b) { al = nrm[0][b]; be = nrm[1][b]; }
    for (int step = 0; step < 2 * G - 1; ++step) {
#pragma unroll
      for (int k = 0; k < B; ++k) {
        double ga[B];
#pragma unroll
        for (int b = 0; b < B; ++b) ga[b] = dot(h[0][b], h[1][(b + k) % B]);
        double g;
        if constexpr (B == 4) {
          const bool hi = lane & 16, odd = lane & 8;
          double k0 = hi ? ga[2] : ga[0], k1 = hi ? ga[3] : ga[1];
          k0 += __shfl_xor_sync(0xffffffffu, hi ? ga[0] : ga[2], 16);
          k1 += __shfl_xor_sync(0xffffffffu, hi ? ga[1] : ga[3], 16);
          g = (odd ? k1 : k0) + __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, 8);
        } else {
          const bool hi = lane & 16;
          g = (hi ? ga[1] : ga[0]) + __shfl_xor_sync(0xffffffffu, hi ? ga[0] : ga[1], 16);
          g += __shfl_xor_sync(0xffffffffu, g, 8);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        // (as in rotate above)
        const double zd = be - al, wd = 2.0 * g;
        const int e_max = max(__double2hiint(zd) & 0x7ff00000, __double2hiint(wd) & 0x7ff00000);
        const bool act = g * g > 1e-22 * al * be && e_max >= 0x01000000;
        const double unit = __hiloint2double(0x7fe00000 - e_max, 0);
        const float z = (float)(zd * unit), w = (float)(wd * unit);
        const float tf = act ? copysignf(w / (fabsf(z) + sqrtf(fmaf(z, z, w * w))), z >= 0.f ? w : -w) : 0.f;
        const double tt = (double)tf, c = act ? rsqrt(fma(tt, tt, 1.0)) : 1.0, sn = c * tt;
        if (__any_sync(0xffffffffu, act)) {
          if (__any_sync(0xffffffffu, g * g > kStop * al * be)) any = 1;
          const double c2 = c * c, s2 = sn * sn, cs2 = 2.0 * c * sn * g, na = c2 * al - cs2 + s2 * be, nb = s2 * al + cs2 + c2 * be;
          al = na > 0.0 ? na : 0.0; be = nb > 0.0 ? nb : 0.0;
#pragma unroll
          for (int b = 0; b < B; ++b) {
            const double cb = __shfl_sync(0xffffffffu, c, b * GL), sb = __shfl_sync(0xffffffffu, sn, b * GL);
#pragma unroll
            for (int e = 0; e < E; ++e) {
              const double x = h[0][b][e], y = h[1][(b + k) % B][e];
              h[0][b][e] = cb * x - sb * y;
              h[1][(b + k) % B][e] = fma(sb, x, cb * y);
            }
          }
        }
        be = __shfl_sync(0xffffffffu, be, ((pb + 1) % B) * GL);
      }
      if (G == 1) break;
      // circle method: the top block of group 0 stays, the others move on by one place of the ring of blocks
      flip ^= 1;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        int tg, ts;
        if (s == 0) { if (g == 0) { tg = 0; ts = 0; } else if (g < G - 1) { tg = g + 1; ts = 0; } else { tg = g; ts = 1; } }
        else { if (g == 0) { tg = 1; ts = 0; } else { tg = g - 1; ts = 1; } }
        const uint32_t off = base + flip * buf_b + (uint32_t)((tg % nw) * 2 + ts) * (Sh::kBlock * 8) + lane * 8;
        uint32_t dst;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(off), "r"(tg / nw));
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
          for (int e = 0; e < E; ++e)
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst + (b * Sh::kElems + 32 * e) * 8), "d"(h[s][b][e]) : "memory");
        if (lane % GL == 0) asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst + (B * Sh::kElems + pb - lane) * 8), "d"(s ? be : al) : "memory");
      }
      cluster_sync_all();
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const double* src = smj + (size_t)flip * nw * 2 * Sh::kBlock + (size_t)(warp * 2 + s) * Sh::kBlock + lane;
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
          for (int e = 0; e < E; ++e) h[s][b][e] = src[b * Sh::kElems + 32 * e];
        (s ? be : al) = src[B * Sh::kElems + pb - lane];
      }
    }
    // did anybody rotate?  every CTA's flag, by every warp that did
    if (any && lane == 0) {
      for (int r = 0; r < cs; ++r) {
        uint32_t a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(&moved_s[sweep & 1])), "r"(r));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(1) : "memory");
      }
    }
    cluster_sync_all();
    const int moved = *reinterpret_cast<volatile int*>(&moved_s[sweep & 1]);
    if (t == 0) moved_s[(sweep & 1) ^ 1] = 0;
    cluster_sync_all();
    if (!moved) break;
  }
  // eigenvalues = column norms; order them (descending; ties by place)
  norms();
  const int nc = 2 * G * B;
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int b = 0; b < B; ++b)
      if (lane == 0) lam[m + (2 * g + s) * B + b] = sqrt(nrm[s][b]);      // unsorted, behind the sorted ones
  __threadfence();
  cluster_sync_all();
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int me = (2 * g + s) * B + b;
      const double mine = __ldcg(lam + m + me);
      int rk = 0;
      for (int o = lane; o < nc; o += 32) { const double v = __ldcg(lam + m + o); rk += (v > mine || (v == mine && o < me)) ? 1 : 0; }
      rk = __reduce_add_sync(0xffffffffu, rk);
      if (rk < m) {
        if (lane == 0) lam[rk] = mine * up;
        const double inv = mine > 0.0 ? 1.0 / mine : 0.0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int i = lane + 32 * e;
          if (i < m) Vf[(int64_t)i * ldv + rk] = (float)(h[s][b][e] * inv);
        }
      }
    }
}

// The same in one CTA, for matrices whose blocks do not fit into a cluster's shared memory (m > 320): pairs of rows of H (= columns, H is symmetric) are rotated until they are orthogonal.  With J the product of the
// rotations the result is J^T H = diag(lam) J^T: row i has norm lam_i and direction v_i, so the eigenvectors are the
// normalised rows and no separate accumulation of the rotations is needed (a row whose norm is zero up to rounding has
// no direction; its eigenvalue is far below the ones that are kept).
// Pairs follow the round-robin tournament (m' / 2 disjoint pairs per step, m' - 1 steps per sweep); a warp takes a pair.
// Output: eigenvalues in descending order (lam) and the matching eigenvectors as fp32 columns of Vf ([m][ldv] row-major).
__global__ void __launch_bounds__(1024) k_jacobi64(double* H, int m, double* lam, float* Vf, int ldv, int max_sweeps) {
  __shared__ int moved_s;
  __shared__ int rank_s[512];
  const int t = threadIdx.x, nt = blockDim.x, warp = t >> 5, lane = t & 31, nwarp = nt >> 5;
  const int mp = (m + 1) & ~1;                       // players of the tournament (one bye if m is odd)
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    if (t == 0) moved_s = 0;
    __syncthreads();
    for (int step = 0; step < mp - 1; ++step) {
      for (int pr = warp; pr < mp / 2; pr += nwarp) {
        // circle method: player mp - 1 is fixed, the others rotate
        int p = pr == 0 ? mp - 1 : (step + pr) % (mp - 1);
        int q = (step + mp - 1 - pr) % (mp - 1);
        if (p > q) { const int x = p; p = q; q = x; }
        if (q >= m) continue;                        // the bye
        // columns p and q of H (column c of the symmetric start is stored as row c: H[c * m + i])
        double* hp = H + (int64_t)p * m; double* hq = H + (int64_t)q * m;
        double al = 0.0, be = 0.0, ga = 0.0;
        for (int i = lane; i < m; i += 32) { const double a = hp[i], b = hq[i]; al += a * a; be += b * b; ga += a * b; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o); be += __shfl_xor_sync(0xffffffffu, be, o); ga += __shfl_xor_sync(0xffffffffu, ga, o);
        }
        if (fabs(ga) <= 1e-11 * sqrt(al * be) || ga == 0.0) continue;      // orthogonal far beyond what the fp32 operands carry
        const double zeta = (be - al) / (2.0 * ga);
        const double tt = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
        const double c = 1.0 / sqrt(1.0 + tt * tt), s = c * tt;
        for (int i = lane; i < m; i += 32) {
          const double a = hp[i], b = hq[i];
          hp[i] = c * a - s * b; hq[i] = s * a + c * b;
        }
        if (lane == 0) moved_s = 1;
      }
      __syncthreads();
    }
    const int moved = moved_s;
    __syncthreads();
    if (!moved) break;
  }
  // eigenvalues = column norms; order them (descending; ties by index)
  for (int c = warp; c < m; c += nwarp) {
    double al = 0.0;
    for (int i = lane; i < m; i += 32) { const double a = H[(int64_t)c * m + i]; al += a * a; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) al += __shfl_xor_sync(0xffffffffu, al, o);
    if (lane == 0) lam[m + c] = sqrt(al);            // unsorted, behind the sorted ones
  }
  __syncthreads();
  for (int c = t; c < m; c += nt) {
    int rk = 0;
    const double mine = lam[m + c];
    for (int o = 0; o < m; ++o) { const double v = lam[m + o]; rk += (v > mine || (v == mine && o < c)) ? 1 : 0; }
    rank_s[c] = rk;
  }
  __syncthreads();
  for (int c = t; c < m; c += nt) lam[rank_s[c]] = lam[m + c];
  __syncthreads();
  for (int e = t; e < m * m; e += nt) {
    const int c = e / m, i = e % m;                  // eigenvector c, component i  ->  Vf[i][rank of c]
    const double nrm = lam[rank_s[c]];
    Vf[(int64_t)i * ldv + rank_s[c]] = nrm > 0.0 ? (float)(H[e] / nrm) : 0.f;
  }
}

// Sums of squares of the first r columns of V [v_rows][ld] and U [u_rows][ld], fp64: part z of the rows writes parts[z][0][r] and [z][1][r].
constexpr int kSigmaParts = 32;
__global__ void __launch_bounds__(256) k_colsq(const float* __restrict__ V, int v_rows, const float* __restrict__ U, int u_rows, int ld, int r, double* __restrict__ parts) {
  __shared__ double sm[8][33];
  const int c = threadIdx.x & 31, y = threadIdx.x >> 5, col = blockIdx.x * 32 + c;
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const float* a = w ? U : V;
    const int rows = w ? u_rows : v_rows, per = (rows + kSigmaParts - 1) / kSigmaParts, hi = min(rows, (int)(blockIdx.y + 1) * per);
    double s = 0.0;
    if (col < r)
      for (int i = blockIdx.y * per + y; i < hi; i += 8) { const double v = a[(int64_t)i * ld + col]; s = fma(v, v, s); }
    sm[y][c] = s;
    __syncthreads();
    if (y == 0 && col < r) {
#pragma unroll
      for (int i = 1; i < 8; ++i) s += sm[i][c];
      parts[((int64_t)blockIdx.y * 2 + w) * r + col] = s;
    }
    __syncthreads();
  }
}
// lam_i = |V_i|^2 / |U_i|^2; zero for a direction that is zero, and NaN where either is NaN (so no comparison that a NaN would fail decides here or below).
__global__ void k_sigma(const double* __restrict__ parts, int r, double* __restrict__ lam) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= r) return;
  double v = 0.0, u = 0.0;
  for (int z = 0; z < kSigmaParts; ++z) { v += parts[(int64_t)z * 2 * r + i]; u += parts[((int64_t)z * 2 + 1) * r + i]; }
  lam[i] = u == 0.0 ? 0.0 : v / u;
}
// sigma_i = sqrt(lam_i);  B'[row][i] = U[row][i] sigma_i  (U: [d][ld]).  status: not zero if a product gave up; the results are then NaN.
__global__ void k_finish_b(const float* __restrict__ U, int ld, const double* __restrict__ lam, int d, int r, float* __restrict__ Bp, float* __restrict__ sigma,
                           const int* __restrict__ status) {
  const int64_t n = (int64_t)d * r;
  const float bad = *status ? __int_as_float(0x7fffffff) : 0.f;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % r);
    Bp[e] = U[e / r * ld + i] * (float)sqrt(lam[i]) + bad;
    if (e < r) sigma[e] = (float)sqrt(lam[e]) + bad;
  }
}
// A[i][j] = T[j][i] / sigma_i  (T: [k][ld], holding dW^T U); 32 x 32 tiles through shared memory, 32 x 8 threads
__global__ void k_finish_a(const float* __restrict__ T, int ld, const double* __restrict__ lam, int r, int k, float* __restrict__ A,
                           const int* __restrict__ status) {
  __shared__ float tile[32][33];
  const float bad = *status ? __int_as_float(0x7fffffff) : 0.f;
  const int j0 = blockIdx.x * 32, i0 = blockIdx.y * 32, x = threadIdx.x, y = threadIdx.y;
  for (int q = y; q < 32; q += 8) tile[q][x] = j0 + q < k && i0 + x < r ? T[(int64_t)(j0 + q) * ld + i0 + x] : 0.f;
  __syncthreads();
  for (int q = y; q < 32; q += 8) {
    if (i0 + q >= r || j0 + x >= k) continue;
    const double s = sqrt(lam[i0 + q]);
    A[(int64_t)(i0 + q) * k + j0 + x] = (s == 0.0 ? 0.f : (float)((double)tile[x][q] / s)) + bad;
  }
}
// sum of squares of a matrix, fp64, into *out (zeroed by the caller)
__global__ void k_sumsq(const float* __restrict__ a, int64_t n, double* out) {
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) acc += (double)a[i] * (double)a[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}
__global__ void k_axpy_neg(float* __restrict__ c, const float* __restrict__ a, int64_t n) {      // c = a - c
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) c[i] = a[i] - c[i];
}

// ------------------------------------------------------------------------------------------------ workspace
struct Plan {
  int d, k, n, r, m;
  int iters;                  // plain products; 0: the filter
  int dp, kp, np;             // d, k, n in whole 128-tiles
  bool tensor;                // products with the iterate on the tensor cores (with C's three parts in the workspace)
  bool keep_dw;               // dW stays where P's product leaves it; else its place is used in between, and it is formed again for step 6
  int kc, lc;                 // of the reduction axes of P and of its square: what is split at a time
  int py, pz;                 // rows of P, and columns of it, that are split at a time for the products with the iterate
  bool n_side, pad_x;         // iterate with P^T P instead of P P^T; X~ is needed in whole tiles
  int s, sp;                  // size of the matrix that is iterated with, in whole tiles
  int w, ldm;                 // width of the skinny products' tiles, leading dimension of the iterates (a multiple of it)
  int wr, ldr;                // the same for the products with r columns
  size_t off_x, off_p, off_dw, off_big, off_c, off_parts, off_sq, off_it, off_y, off_q, off_z, off_s, off_sp, off_d, off_h, off_lam, off_vf, total;
};
size_t up256(size_t v) { return (v + 255) & ~size_t(255); }
int up128(int v) { return (v + 127) & ~127; }
// The width with the fewest padding columns (the widest of those).
int pick_width(int cols) {
  int best = 160;
  for (int w : {128, 96, 64})
    if ((cols + w - 1) / w * w < (cols + best - 1) / best * best) best = w;
  return best;
}
// What the workspace has room for.  ROOMY: what makes no product go in more parts than is good for it, or as much of that as kRoomy or a quarter of the
// matrices themselves.  TIGHT: the matrices (and C's three parts where they are larger).  LEAN: the matrices; products with the iterate on the CUDA cores.
// Parts cost some 10 us each in a small solve, 2 to 4 % of it, and 80 us at 4096 x 4096 x 16384 (seven parts 8.26 ms, one 7.7, with 330 MB more; three, with 110 MB more, 7.8).
enum Room { ROOMY, TIGHT, LEAN };
constexpr size_t kRoomy = 48u << 20;
constexpr size_t kSmall = 8u << 20;                  // (one or two parts more at most; the reported workspace is the smallest one then)

// Offsets and parts for a given region `big`; whole: nothing goes in more parts than is good for it.
bool lay_out(Plan& p, size_t big, bool& whole) {
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o += up256(bytes); return at; };
  const size_t rows = p.dp > p.np ? p.dp : p.np, tall = rows > (size_t)p.kp ? rows : p.kp, c_b = (size_t)p.sp * p.sp * 4;
  p.off_x = take(p.pad_x ? (size_t)p.kp * p.np * 4 : 0);
  p.off_p = take((size_t)p.dp * p.np * 4);                        // P = dW X~; the loss check keeps (dW - B'A) X~ here
  p.off_dw = take((size_t)p.dp * p.kp * 4);
  // One region for what is not needed at the same time, with room for C or, in the loss check, dW - B'A:
  //   dW and X~^T split, as much of the reduction axis at a time as there is room for up to off_lam (at least two parts where all would take more than 32 MB);
  //   C at the region's end, and P split for its square in front of it or behind it;
  //   C split from the region's front on, over C itself (slabs of rows, in order);
  //   in the end P split, as many of the result's rows at a time as there is room for.
  // Without keep_dw it begins with dW's place.  An iterate's parts are at its end, or, if they fit there, among the small problems, which are not in use when it is
  // multiplied with.
  p.off_big = take(big);
  p.off_c = p.off_big + big - c_b;
  const size_t end = o;
  p.off_y = take(rows * p.ldm * 4);
  p.off_q = take(rows * p.ldm * 4);
  p.off_z = take(tall * p.ldm * 4);
  p.off_s = take((size_t)p.m * p.m * 8);                          // (in the end, with the next one: 64 r partial sums for sigma)
  p.off_sp = take((size_t)kGramParts * p.m * p.m * 8);
  p.off_d = take((size_t)((p.m + 15) / 16) * 256 * 8);
  p.off_h = take((size_t)p.m * p.m * 8);
  p.off_lam = take((size_t)(2 * p.m + 128) * 8);                  // (the last 32 doubles: status and the filter's state)
  p.off_vf = take((size_t)p.ldm * p.ldm * 4);
  p.total = o;
  p.off_it = p.keep_dw ? p.off_big : p.off_dw;
  size_t s_q = eora::split_bytes(up128(p.ldm), p.dp);             // an iterate of either side (np <= dp with n_side)
  const bool among = s_q <= p.off_lam - p.off_s;
  p.off_sq = among ? p.off_s : end - s_q;
  if (among) s_q = 0;
  // How much at a time.
  auto in_parts = [](int len, int parts) { return ((len / 128 + parts - 1) / parts) * 128; };
  auto at_once = [&](int len, size_t each, size_t room, int least) {      // (each: bytes of 128 of len)
    const size_t most = room / each;
    if (most < 1) return 0;
    int parts = least;
    while ((size_t)in_parts(len, parts) > most * 128) ++parts;
    return in_parts(len, parts);
  };
  const size_t dx = eora::split_bytes(p.dp, 128) + eora::split_bytes(p.np, 128);
  const int halves = dx * (p.kp / 128) > (32u << 20) ? 2 : 1;
  p.kc = at_once(p.kp, dx, p.off_lam - p.off_it, halves);
  const int len = p.n_side ? p.dp : p.np;                         // reduction axis of P's square
  const size_t front = p.off_c - p.off_it, behind = p.off_lam - p.off_y;
  p.off_parts = front >= behind ? p.off_it : p.off_y;
  p.lc = at_once(len, eora::split_bytes(p.sp, 128), front >= behind ? front : behind, 1);
  if (p.kc < 1 || p.lc < 1) return false;
  whole = p.kc == in_parts(p.kp, halves) && p.lc == len;
  p.py = p.pz = 0;
  if (p.tensor) {
    if (end - p.off_it < s_q || eora::split_bytes(p.sp, p.sp) > end - p.off_it - s_q) return false;
    // (a slab of C takes at least one row block: the last one with what C's rows in front of it have left)
    if (front + (size_t)(p.sp - 128) * p.sp * 4 < eora::split_bytes(p.sp, p.sp)) return false;
    const size_t room = end - p.off_it - s_q;
    p.pz = at_once(p.np, eora::split_bytes(128, p.dp), room, 1);
    if (p.pz < 1) return false;
    whole = whole && p.pz == p.np;
    if (p.n_side) {
      p.py = at_once(p.dp, eora::split_bytes(128, p.np), room, 1);
      if (p.py < 1) return false;
      whole = whole && p.py == p.dp;
    }
  }
  return true;
}
bool make_plan(const eora_solve_config* c, Plan& p, Room room) {
  if (!c || c->d < 1 || c->k < 1 || c->n < 1 || c->rank < 1) return false;
  p.d = c->d; p.k = c->k; p.n = c->n; p.r = c->rank;
  int over = c->oversample > 0 ? c->oversample : 32;
  p.m = p.r + over;
  if (p.m > p.d) p.m = p.d;
  if (p.r > p.m || p.m > 512) return false;
  p.iters = c->iters > 0 ? c->iters : 0;
  p.dp = up128(p.d); p.kp = up128(p.k); p.np = up128(p.n);
  p.pad_x = p.k % 128 || p.n % 128;
  // The smaller side (every iteration is a product with its square); it has to hold m directions.
  p.n_side = p.n < p.d && p.n >= p.m;
  p.s = p.n_side ? p.n : p.d;
  p.sp = p.n_side ? p.np : p.dp;
  p.w = pick_width(p.m); p.ldm = (p.m + p.w - 1) / p.w * p.w;
  p.wr = pick_width(p.r); p.ldr = (p.r + p.wr - 1) / p.wr * p.wr;
  if (p.ldr > p.ldm) { p.wr = p.w; p.ldr = p.ldm; }
  // The products with an iterate: on the tensor cores, the iterate being split for each, or, small ones, on the CUDA cores in one launch.  512 x 512 x 64: 9
  // against 6 us on the CUDA cores, 768 x 768 x 64 about even; 2048 x 2048 x 160: 21 against 50.
  p.tensor = room != LEAN && (double)p.sp * p.sp * p.ldm >= 8e7;
  const size_t c_b = (size_t)p.sp * p.sp * 4, e_b = (size_t)p.d * p.k * 4, least = up256(c_b > e_b ? c_b : e_b);
  // The matrices' own size if that will do, with dW left alone or formed again; else a larger one.
  bool whole = false;
  p.keep_dw = true;
  if (lay_out(p, least, whole) && whole) return true;
  if (room == ROOMY && p.total >= kSmall) {
    // what is asked of the region: dW and X~^T split, C and P split, C's three parts, each with an iterate's
    const int len = p.n_side ? p.dp : p.np;
    const size_t sq = eora::split_bytes(up128(p.ldm), p.dp), c_p = c_b + eora::split_bytes(p.sp, len), c_3 = eora::split_bytes(p.sp, p.sp) + sq;
    const int kh = eora::split_bytes(p.dp, p.kp) + eora::split_bytes(p.np, p.kp) > (32u << 20) ? (p.kp / 128 + 1) / 2 * 128 : p.kp;
    const size_t a = eora::split_bytes(p.dp, kh) + eora::split_bytes(p.np, kh), own = p.off_lam - p.off_y, p_3 = eora::split_bytes(p.dp, p.np) + sq;
    size_t need = least;
    for (size_t v : {a > own ? a - own : 0, c_p, p.tensor ? c_3 : 0, p.tensor ? p_3 : 0})
      if (up256(v) > need) need = up256(v);
    const size_t most = p.total / 4 > kRoomy ? up256(p.total / 4) : kRoomy;
    if (need - least <= most && lay_out(p, need, whole) && whole) return true;
    p.keep_dw = false;
    const size_t dw_b = up256((size_t)p.dp * p.kp * 4);
    if (lay_out(p, least, whole) && whole) return true;
    const size_t more = need > dw_b ? need - dw_b : 0;
    if (more > least && lay_out(p, more - least <= most ? more : least + most, whole)) return true;
  }
  // In parts.
  for (int i = 0; i < 2; ++i) {
    p.keep_dw = i == 0 && !p.tensor;
    if (lay_out(p, least, whole)) return true;
  }
  // C's three parts are larger than C and dW (14336 x 4096, n 16384).
  const size_t three = up256(eora::split_bytes(p.sp, p.sp) + eora::split_bytes(up128(p.ldm), p.dp) + eora::split_bytes(128, p.dp)), dw_b = up256((size_t)p.dp * p.kp * 4);
  p.keep_dw = false;
  return lay_out(p, three - dw_b, whole);
}
inline bool aligned16(const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; }

#define CK(x) do { cudaError_t e__ = (x); if (e__ != cudaSuccess) return EORA_ERR_CUDA; } while (0)

// Shared-memory limits are set once per kernel and device.
template <auto KERNEL>
cudaError_t allow_smem(int bytes) {
  static bool done[64] = {};
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
  if (done[device]) return cudaSuccess;
  e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done[device] = true;
  return e;
}

constexpr int kSingleSteps = 4;        // products that are orthogonalised one by one before the pairs begin

// Q = orth(Y) by Cholesky-QR: Gram matrix, its factor and Q = Y L^{-T} in fp64.  Y, Q: [rows][ldm], rows a multiple of 16.  parts: the Gram matrix's
// partial sums, then the smallest pivots.
int orthonormalise(cudaStream_t st, const Plan& p, int rows, const float* Y, float* Q, double* S, double* parts, double* D,
                   bool scaled = false, Filter* f = nullptr, bool prev = false, double lo = 0.0, double hi = 0.0) {
  CK(gram64<false>(st, Y, rows, p.m, p.ldm, parts, S));
  CK(allow_smem<k_chol64>(chol_smem(kCholSmem)));
  CK(allow_smem<k_trsm<float>>(trsm_smem(512)));
  CK(allow_smem<k_trsm<double>>(trsm_smem(kCholSmem)));
  // Up to 160 columns one CTA factors the matrix in shared memory.  More go in blocks of 160: factor, rows below, update of the rest (2048 x 3072, n 2048, 288
  // columns: 6.28 ms, with one CTA that kept such a matrix in L2 7.72).
  for (int j0 = 0; j0 < p.m; j0 += kCholSmem) {
    const int w = p.m - j0 < kCholSmem ? p.m - j0 : kCholSmem, j1 = j0 + w, below = p.m - j1;
    k_chol64<<<1, kCholThreads, chol_smem(w), st>>>(S, p.m, p.m, j0, w, D + j0 * 16, parts, below ? nullptr : f, prev, lo, hi);
    if (below > 0) {
      double* l21 = S + (int64_t)j1 * p.m + j0;
      k_trsm<double><<<(below + 15) / 16, 256, trsm_smem(w), st>>>(l21, S + (int64_t)j0 * (p.m + 1), p.m, D + j0 * 16, w, p.m, below, l21, false);
      const int nb = (below + 31) / 32;
      k_syrk64<<<nb * (nb + 1) / 2, 256, 0, st>>>(S, p.m, p.m, j0, j1);
    }
  }
  k_trsm<float><<<rows / 16, 256, trsm_smem(p.m), st>>>(Y, S, p.m, D, p.m, p.ldm, rows, Q, scaled);
  CK(cudaGetLastError());
  return EORA_OK;
}

template <int B, int E>
cudaError_t launch_jacobi(cudaStream_t st, const double* H, int m, double* lam, float* Vf, int ldv) {
  constexpr int cs = B == 4 ? 4 : 8;                 // CTAs: five warps each at m = 160, ten at m = 320
  const int groups = (m + 2 * B - 1) / (2 * B), nw = (groups + cs - 1) / cs;
  const int smem = 2 * nw * 2 * JacobiShape<B, E>::kBlock * 8;
  cudaError_t e = allow_smem<k_jacobi_cl<B, E>>(2 * (B == 4 ? 5 : 10) * 2 * JacobiShape<B, E>::kBlock * 8);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs);
  cfg.blockDim = dim3(32 * nw);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_jacobi_cl<B, E>, H, m, lam, Vf, ldv, 40);
}
cudaError_t jacobi(cudaStream_t st, double* H, int m, double* lam, float* Vf, int ldv) {
  if (m <= 64) return launch_jacobi<4, 2>(st, H, m, lam, Vf, ldv);
  if (m <= 96) return launch_jacobi<4, 3>(st, H, m, lam, Vf, ldv);
  if (m <= 128) return launch_jacobi<4, 4>(st, H, m, lam, Vf, ldv);
  if (m <= 160) return launch_jacobi<4, 5>(st, H, m, lam, Vf, ldv);
  if (m <= 224) return launch_jacobi<2, 7>(st, H, m, lam, Vf, ldv);
  if (m <= 320) return launch_jacobi<2, 10>(st, H, m, lam, Vf, ldv);
  k_jacobi64<<<1, 1024, 0, st>>>(H, m, lam, Vf, ldv, 40);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

size_t eora_solve_workspace_bytes(const eora_solve_config* cfg) {
  Plan p;
  return make_plan(cfg, p, ROOMY) ? p.total : 0;
}

int eora_solve(const eora_solve_config* cfg, const float* w, const float* w_hat, const float* x_tilde, float* b_prime, float* a,
               float* sigma, void* workspace, size_t workspace_bytes, void* stream) {
  if (!cfg || !w || !w_hat || !x_tilde || !b_prime || !a || !sigma || !workspace) return EORA_ERR_NULL_ARG;
  Plan p;
  bool fits = false;
  for (Room room : {ROOMY, TIGHT, LEAN}) fits = fits || (make_plan(cfg, p, room) && workspace_bytes >= p.total);
  if (!fits) return EORA_ERR_BAD_SHAPE;
  if (!aligned16(w) || !aligned16(w_hat) || !aligned16(x_tilde) || !aligned16(b_prime) || !aligned16(a) || !aligned16(workspace)) return EORA_ERR_MISALIGNED;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  char* ws = reinterpret_cast<char*>(workspace);
  float* dW = reinterpret_cast<float*>(ws + p.off_dw);
  float* Pm = reinterpret_cast<float*>(ws + p.off_p);
  float* C = reinterpret_cast<float*>(ws + p.off_c);
  float* Y = reinterpret_cast<float*>(ws + p.off_y);
  float* Q = reinterpret_cast<float*>(ws + p.off_q);
  float* Z = reinterpret_cast<float*>(ws + p.off_z);
  double* S = reinterpret_cast<double*>(ws + p.off_s);
  double* Sp = reinterpret_cast<double*>(ws + p.off_sp);
  double* D = reinterpret_cast<double*>(ws + p.off_d);
  double* H = reinterpret_cast<double*>(ws + p.off_h);
  double* lam = reinterpret_cast<double*>(ws + p.off_lam);
  float* Vf = reinterpret_cast<float*>(ws + p.off_vf);
  const int dp = p.dp, kp = p.kp, np = p.np, sp = p.sp, ldm = p.ldm;

  uint8_t* it_mem = reinterpret_cast<uint8_t*>(ws + p.off_it);
  uint8_t* parts = reinterpret_cast<uint8_t*>(ws + p.off_parts);
  int* status = reinterpret_cast<int*>(lam + 2 * p.m + 96);
  static_assert(sizeof(Filter) <= 30 * 8, "behind the eigenvalues");
  int device = 0, sms = 0;
  CK(cudaGetDevice(&device));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
  CK(cudaMemsetAsync(status, 0, 4, st));
  // steps 1-4: dW, P = dW X~, and the smaller of P P^T and P^T P
  float* xp = p.pad_x ? reinterpret_cast<float*>(ws + p.off_x) : nullptr;
  for (int k0 = 0; k0 < kp; k0 += p.kc) {
    const int kc = kp - k0 < p.kc ? kp - k0 : p.kc, kr = p.k - k0 < kc ? p.k - k0 : kc;      // columns of dW, without the padding
    uint8_t* xs = it_mem + eora::split_bytes(dp, p.kc);
    CK(eora::split_rows(st, w + k0, w_hat + k0, p.d, kr, p.k, dp, kc, it_mem, p.keep_dw ? dW + k0 : nullptr, kp));
    CK(eora::split_cols(st, x_tilde + (size_t)k0 * p.n, kr, p.n, p.n, kc, np, xs, xp ? xp + (size_t)k0 * np : nullptr));
    CK(eora::split_gemm(st, it_mem, xs, dp, np, kc, Pm, np, false, k0 > 0, sms, status));
  }
  const int len = p.n_side ? dp : np;
  for (int l0 = 0; l0 < len; l0 += p.lc) {
    const int lc = len - l0 < p.lc ? len - l0 : p.lc;
    if (p.n_side) CK(eora::split_cols(st, Pm + (size_t)l0 * np, lc, np, np, lc, np, parts));
    else CK(eora::split_rows(st, Pm + l0, nullptr, dp, lc, np, dp, lc, parts, nullptr, 0));
    CK(eora::split_gemm(st, parts, parts, sp, sp, lc, C, sp, true, l0 > 0, sms, status));
  }
  uint8_t* sq = reinterpret_cast<uint8_t*>(ws + p.off_sq);
  if (p.tensor) {
    // C's parts take 6 bytes where C has 4: a slab of rows ends before the first row that is not yet split.
    for (int r0 = 0; r0 < sp;) {
      const size_t room = p.off_c - p.off_it + (size_t)r0 * sp * 4;
      const int most = (int)(room / eora::split_bytes(128, sp) < (size_t)sp / 128 ? room / eora::split_bytes(128, sp) : (size_t)sp / 128) * 128, r1 = most < sp ? most : sp;
      if (r1 <= r0) return EORA_ERR_BAD_SHAPE;       // (never: lay_out has seen to it)
      CK(eora::split_rows(st, C + (size_t)r0 * sp, nullptr, r1 - r0, sp, sp, r1 - r0, sp, it_mem + eora::split_bytes(r0, sp), nullptr, 0));
      r0 = r1;
    }
  }
  // V [rows_out][ldm] = M U - *shift U for an iterate U; M = mat split (rows_out x rows_in); to: where U is split
  auto product = [&](const uint8_t* mat, const uint8_t* u_split, int rows_out, int rows_in, const float* U, float* V, const float* shift) -> int {
    CK(eora::split_skinny(st, p.w, mat, u_split, rows_out, ldm, rows_in, V, ldm, U, shift, status));
    return EORA_OK;
  };
  auto split_iterate = [&](const float* U, int rows_in, uint8_t* to) { return eora::split_cols(st, U, rows_in, ldm, ldm, rows_in, up128(ldm), to); };
  auto times_c = [&](const float* U, float* V, const float* shift) -> int {
    if (p.tensor) {
      CK(split_iterate(U, sp, sq));
      return product(it_mem, sq, sp, sp, U, V, shift);
    }
    CK(skinny<true>(st, p.w, sp, sp, C, sp, U, ldm, ldm, V, ldm, shift));      // (C is symmetric: read by columns)
    return EORA_OK;
  };
  // step 5: subspace iteration
  k_init<<<592, 256, 0, st>>>(Y, p.s, sp, p.m, ldm);
  CK(cudaGetLastError());
  if (int rc = orthonormalise(st, p, sp, Y, Q, S, Sp, D)) return rc;
  // Orthogonalising costs twice a product with C (a chain of m pivots).  Once the columns are graded -- column j close to the j-th
  // eigenvector, which the first steps see to -- it is needed only every second product: the part of the larger eigenvectors that
  // rounding brings into a column stays in the span and is taken out with the next factor, and what lies outside the span
  // is damped by every product.  The iterate that goes through two products is scaled to norm 1 / lam_1, which keeps
  // C C Q in the range of the products of one step.
  //
  // By default four single products are followed by kPairs pairs whose second factors are C - rho I with rho at the Chebyshev points of degree 2 kPairs
  // of [0, lam_m]: what is left of an eigenvalue there is 1 / T_10(2 lam_r / lam_m - 1) of eigenvalue r's part instead of (lam_m / lam_r)^10.
  // A pair takes a point and its mirror image, so no pair lets anything in the interval grow against what lies above it, whatever their order.  The
  // diagonal of the factor says where lam_m is (k_chol64), each time anew.  14 products and 12 factorisations come as close as 24 and 17 of
  // the plain iteration, or closer (error of the projector where the plain one has not converged: flat spectra 1.1e-2 -> 8e-4 and 2.1e-4 -> 3e-5).
  const bool filter = p.iters == 0;
  constexpr int kPairs = 5, kOrder[kPairs] = {3, 1, 4, 0, 2};
  auto node = [&](int i) { return 0.5 + 0.5 * cos((2 * i + 1) * 3.14159265358979323846 / (4 * kPairs)); };
  const int iters = filter ? kSingleSteps + 2 * kPairs : p.iters;
  Filter* f = filter ? reinterpret_cast<Filter*>(lam + 2 * p.m + 98) : nullptr;
  for (int it = 0, pairs = 0; it < iters;) {
    const bool pair = it >= kSingleSteps && iters - it >= 2;
    if (int rc = times_c(Q, Y, pair && f ? f->rho : nullptr)) return rc;
    if (pair) {
      if (int rc = times_c(Y, Q, f ? f->rho + 1 : nullptr)) return rc;
      float* y = Y; Y = Q; Q = y;
    }
    it += pair ? 2 : 1;
    const bool next_pair = it >= kSingleSteps && iters - it >= 2;
    const int i = next_pair && f ? kOrder[pairs++] : 0;
    if (int rc = orthonormalise(st, p, sp, Y, Q, S, Sp, D, next_pair, next_pair ? f : nullptr, pair, node(i), node(2 * kPairs - 1 - i))) return rc;
  }
  if (p.n_side) {                                                             // to the d-dimensional side
    if (p.tensor) {
      CK(split_iterate(Q, np, sq));
      for (int r0 = 0; r0 < dp; r0 += p.py) {
        const int rc = dp - r0 < p.py ? dp - r0 : p.py;
        CK(eora::split_rows(st, Pm + (size_t)r0 * np, nullptr, rc, np, np, rc, np, it_mem, nullptr, 0));
        if (int e = product(it_mem, sq, rc, np, Q, Y + (size_t)r0 * ldm, nullptr)) return e;
      }
    } else {
      CK(skinny<false>(st, p.w, dp, np, Pm, np, Q, ldm, ldm, Y, ldm));
    }
    if (int rc = orthonormalise(st, p, dp, Y, Q, S, Sp, D)) return rc;
  }
  if (int rc = orthonormalise(st, p, dp, Q, Y, S, Sp, D)) return rc;          // second pass: orthogonal to fp32 rounding
  // Rayleigh-Ritz on span(Y)
  if (p.tensor) {                                                             // Z = P^T Y
    CK(split_iterate(Y, dp, sq));
    for (int n0 = 0; n0 < np; n0 += p.pz) {
      const int nc = np - n0 < p.pz ? np - n0 : p.pz;
      CK(eora::split_cols(st, Pm + n0, dp, nc, np, dp, nc, it_mem));
      if (int e = product(it_mem, sq, nc, dp, Y, Z + (size_t)n0 * ldm, nullptr)) return e;
    }
  } else {
    CK(skinny<true>(st, p.w, np, dp, Pm, np, Y, ldm, ldm, Z, ldm));
  }
  CK(gram64<true>(st, Z, np, p.m, ldm, Sp, H));                               // H = Z^T Z = Y^T P P^T Y
  CK(cudaMemsetAsync(Vf, 0, (size_t)ldm * ldm * 4, st));
  CK(jacobi(st, H, p.m, lam, Vf, ldm));
  CK(skinny<false>(st, p.wr, dp, ldm, Y, ldm, Vf, ldm, p.ldr, Q, ldm));       // U' = Y V[:, :r]
  // step 6.  The tensor cores' sums are 2e-7 too small (truncation), which the eigenvectors do not notice but the eigenvalues would (sigma 2e-7 off instead
  // of 3e-8): sigma_i = |X~^T dW^T u_i| / |u_i| is taken from fp32 products on the CUDA cores.
  if (!p.keep_dw) CK(eora::split_rows(st, w, w_hat, p.d, p.k, p.k, dp, kp, nullptr, dW, kp));
  CK(skinny<true>(st, p.wr, kp, dp, dW, kp, Q, ldm, p.ldr, Z, ldm));          // dW^T U'
  CK(skinny<true>(st, p.wr, np, kp, xp ? xp : x_tilde, np, Z, ldm, p.ldr, Y, ldm));
  k_colsq<<<dim3((p.r + 31) / 32, kSigmaParts), 256, 0, st>>>(Y, np, Q, dp, ldm, p.r, S);
  k_sigma<<<(p.r + 127) / 128, 128, 0, st>>>(S, p.r, lam);
  k_finish_b<<<592, 256, 0, st>>>(Q, ldm, lam, p.d, p.r, b_prime, sigma, status);
  k_finish_a<<<dim3((p.k + 31) / 32, (p.r + 31) / 32), dim3(32, 8), 0, st>>>(Z, ldm, lam, p.r, p.k, a, status);
  CK(cudaGetLastError());
  return EORA_OK;
}

int eora_solve_loss(const eora_solve_config* cfg, const float* w, const float* w_hat, const float* x_tilde, const float* b_prime,
                    const float* a, double* loss_sq, void* workspace, size_t workspace_bytes, void* stream) {
  if (!cfg || !w || !w_hat || !x_tilde || !b_prime || !a || !loss_sq || !workspace) return EORA_ERR_NULL_ARG;
  Plan p;
  if (!make_plan(cfg, p, LEAN) || workspace_bytes < p.total) return EORA_ERR_BAD_SHAPE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  char* ws = reinterpret_cast<char*>(workspace);
  float* dW = reinterpret_cast<float*>(ws + p.off_dw);
  float* R = reinterpret_cast<float*>(ws + p.off_big);     // B'A, then the residual
  float* E = reinterpret_cast<float*>(ws + p.off_p);       // (dW - B'A) X~  (d x n)
  k_sub<<<592, 256, 0, st>>>(w, w_hat, dW, (int64_t)p.d * p.k);
  CK(sgemm(st, p.d, p.k, p.r, b_prime, p.r, false, a, p.k, false, R, p.k));    // B' A
  k_axpy_neg<<<592, 256, 0, st>>>(R, dW, (int64_t)p.d * p.k);                  // dW - B'A
  CK(sgemm(st, p.d, p.n, p.k, R, p.k, false, x_tilde, p.n, false, E, p.n));
  CK(cudaMemsetAsync(loss_sq, 0, sizeof(double), st));
  k_sumsq<<<592, 256, 0, st>>>(E, (int64_t)p.d * p.n, loss_sq);
  CK(cudaGetLastError());
  return EORA_OK;
}

}  // extern "C"
