// Device helpers shared by the decode kernels: PTX wrappers (mbarrier, bulk copy, mma) and the
// in-register dequantisation of one 16 x 64 tile into tensor-core operand registers.
#pragma once
#include "eora_common.cuh"

namespace eora {
namespace dec {

// ------------------------------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// The same test, but the thread may stay suspended (taking no issue slots) until the phase completes or `ns` nanoseconds
// have passed: what a waiting loop polls with, so that many waiting warps do not crowd out the working ones.
__device__ __forceinline__ bool mbar_try_wait_susp(uint64_t* bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(ns) : "memory");
  return ok != 0;
}
// The same on 32-bit shared addresses.
__device__ __forceinline__ void mbar_init_a(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx_a(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_a(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_g2s_a(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
constexpr unsigned long long kWaitLimitNs = 1000000000ull;   // every device-side wait gives up after 1 s
// Bounded wait: returns false (and latches the status word) if the phase does not complete in time.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* dev_status) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
#pragma unroll 1
    for (int it = 0; it < 64; ++it)
      if (mbar_try_wait_susp(bar, parity, 20000u)) return true;
    if (globaltimer_ns() - t0 > kWaitLimitNs) break;
  }
  atomicExch(dev_status, EORA_ERR_DEVICE_TIMEOUT);
  return false;
}
// The slow path of a wait that every lane of a warp does for itself (the caller brings the lanes together afterwards).
__device__ __forceinline__ bool mbar_wait_lane(uint32_t bar, uint32_t parity, int* dev_status) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
#pragma unroll 1
    for (int it = 0; it < 64; ++it)
      if (mbar_try_wait_a(bar, parity)) return true;
    if (globaltimer_ns() - t0 > kWaitLimitNs) break;
  }
  atomicExch(dev_status, EORA_ERR_DEVICE_TIMEOUT);
  return false;
}
// The same wait for a whole warp.  Only lane 0 polls, and it backs off between polls: a warp-wide
// spin costs a shared-memory access per poll, and a dozen spinning warps are enough to starve the
// bulk-copy engine and the tensor core of shared-memory bandwidth.  Once lane 0 has seen the phase
// complete, every lane tests it once itself (which succeeds at once) so that each thread has its own
// acquire of the data behind the barrier.  The vote makes the lanes take the same way even if they arrive one after the
// other: a lane that saw the phase complete and left would miss the shuffle below, whose result would then be undefined.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, int* dev_status, int lane) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity) ? 1 : 0)) return true;
  int ok = 1;
  if (lane == 0) {
    const unsigned long long t0 = globaltimer_ns();
    ok = 0;
    for (;;) {
#pragma unroll 1
      for (int it = 0; it < 64 && !ok; ++it) {
        __nanosleep(40);
        ok = mbar_try_wait(bar, parity) ? 1 : 0;
      }
      if (ok || globaltimer_ns() - t0 > kWaitLimitNs) break;
    }
    if (!ok) atomicExch(dev_status, EORA_ERR_DEVICE_TIMEOUT);
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (ok) { while (!mbar_try_wait(bar, parity)) {} }
  return ok != 0;
}
// The same without the back-off, for hand-overs that are short and sit on the critical path of a pipeline (a sleeping
// poll adds up to its period to every hand-over).  The polling try_wait suspends the thread until the phase completes.
__device__ __forceinline__ bool mbar_wait_warp_fast(uint64_t* bar, uint32_t parity, int* dev_status, int lane) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity) ? 1 : 0)) return true;
  int ok = 1;
  if (lane == 0) {
    const unsigned long long t0 = globaltimer_ns();
    ok = 0;
    for (;;) {
#pragma unroll 1
      for (int it = 0; it < 256 && !ok; ++it) ok = mbar_try_wait_susp(bar, parity, 20000u) ? 1 : 0;
      if (ok || globaltimer_ns() - t0 > kWaitLimitNs) break;
    }
    if (!ok) atomicExch(dev_status, EORA_ERR_DEVICE_TIMEOUT);
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (ok) { while (!mbar_try_wait(bar, parity)) {} }
  return ok != 0;
}

// Wait, for at most two milliseconds and without touching the status word, for a bulk copy that may still be in flight:
// used by a warp that has already given up and only has to let its copies land before it leaves.
__device__ __forceinline__ void mbar_drain_warp(uint32_t bar, uint32_t parity, int lane) {
  if (lane == 0) {
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_try_wait_a(bar, parity) && globaltimer_ns() - t0 < 2000000ull) __nanosleep(200);
  }
  __syncwarp();
}

// Bounded spin on a global counter reaching `target`.
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p);
__device__ __forceinline__ bool counter_wait(const uint32_t* cnt, uint32_t target, int* dev_status,
                                             unsigned long long limit_ns = kWaitLimitNs) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
#pragma unroll 1
    for (int it = 0; it < 64; ++it) {
      if (ld_acquire(cnt) >= target) return true;
      __nanosleep(32);
    }
    if (globaltimer_ns() - t0 > limit_ns) break;
  }
  atomicExch(dev_status, EORA_ERR_DEVICE_TIMEOUT);
  return false;
}
// global -> shared bulk copy of `bytes` (multiple of 16; both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float ld_cg(const float* p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_add(float* p, float v) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ uint32_t h2sub(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t h2fma(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ------------------------------------------------------------------------------------------ dequant
// Per-quantum constants of the two rows a lane owns: fp16x2 values that turn the magic-number
// form of a code (1024 + q * 2^s as fp16) into the exact integer q - z.
struct ZC { uint32_t c[2][3]; };

template <int FMT>
__device__ __forceinline__ void make_zc(ZC& zc, uint32_t zz) {
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    uint32_t z = (zz >> (8 * hf)) & 255u;
    zc.c[hf][0] = (0x6400u | z) * 0x00010001u;                                      //  1024 + z
    if constexpr (FMT == FMT_Q4) zc.c[hf][1] = (0xD400u | (z << 4)) * 0x00010001u;   // -(64 + z)
  }
}

constexpr uint32_t kMagic = 0x64006400u;   // fp16x2 (1024, 1024)

// (a & mask) | c in ONE instruction.  Written as `(a & mask) | kMagic` with two immediates the compiler
// emits two logic instructions (an instruction holds only one 32-bit immediate), and those run on the
// half-rate integer pipe that bounds the decode kernel; with the constant in a register it is one LOP3.
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t mask, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(mask), "r"(c));
  return d;
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// 2:4 expansion table: for the position nibble p0 | p1 << 2 of a quad, the two byte-permute selectors that
// spread the quad's two kept fp16 values (one register) over its four positions (two registers), zero
// elsewhere.  Low half: selector of positions (0, 1), high half: of positions (2, 3).  Selector bytes: 0x10 =
// first value, 0x32 = second value, 0x44 = zero (the permute's other operand).
__host__ __device__ constexpr uint32_t sp24_selectors(uint32_t nib) {
  const uint32_t p0 = nib & 3u, p1 = nib >> 2;
  uint32_t r = 0;
  for (uint32_t e = 0; e < 4; ++e) {
    const uint32_t sel = e == p0 ? 0x10u : e == p1 ? 0x32u : 0x44u;
    r |= sel << (8 * e);
  }
  return r;
}
// The table in shared memory: 16 words, each in a bank of its own; `mem` is aligned to 256 bytes (half_frags).  Returns its address.
__device__ __forceinline__ uint32_t sp24_lut(uint32_t (&mem)[16]) {
  if (threadIdx.x < 16) mem[threadIdx.x] = sp24_selectors(threadIdx.x);
  return smem_u32(mem);
}

// The eight byte quads (one code per byte) of a lane's 32 codes of a 3-bit tile: q[part][quad].
__device__ __forceinline__ void q3_quads(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t (&q)[4][2]) {
  const uint32_t w[3] = {w0, w1, w2};
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    q[p][0] = w[p] & 0x07070707u;
    q[p][1] = (w[p] >> 3) & 0x07070707u;
  }
  q[3][0] = and_or(w2 >> 4, 0x04040404u, (w0 >> 6) & 0x03030303u);
  q[3][1] = and_or(w2 >> 5, 0x04040404u, (w1 >> 6) & 0x03030303u);
}
// Two neighbouring codes of a byte quad as fp16x2 (1024 + c0, 1024 + c1): which = 0: bytes 0, 1; 1: bytes 2, 3.
__device__ __forceinline__ uint32_t quad_pair(uint32_t quad, int which) {
  return prmt(quad, 0x64646464u, which ? 0x4342u : 0x4140u);
}

// ------------------------------------------------------------------------------------------ blobs in registers
// One lane's payload of a tile and of a blob (two tiles and their scale entries), as loaded from global memory.  The
// weights are read once per launch: no L1 line is allocated for them.
__device__ __forceinline__ uint4 ldw_u4(const uint8_t* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ldw_u2(const uint8_t* p) {
  uint2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ldw_u1(const uint8_t* p) {
  uint32_t v;
  asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ldw_u16(const uint8_t* p) {
  uint16_t v;
  asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(v) : "l"(p));
  return v;
}

template <int FMT> struct RawTile;
template <> struct RawTile<FMT_Q4> { uint4 v; };
template <> struct RawTile<FMT_Q3> { uint2 v; uint32_t w2; };
template <> struct RawTile<FMT_Q8> { uint4 v[2]; };
template <> struct RawTile<FMT_F16> { uint4 v[4]; };
template <> struct RawTile<FMT_SP24> { uint4 v[2]; uint32_t meta; };
template <> struct RawTile<FMT_SQ4> { uint2 v; uint32_t meta; };

template <int FMT> __device__ __forceinline__ void load_tile(RawTile<FMT>& r, const uint8_t* tile, int lane) {
  if constexpr (FMT == FMT_Q4) {
    r.v = ldw_u4(tile + lane * 16);
  } else if constexpr (FMT == FMT_Q3) {
    r.v = ldw_u2(tile + lane * 8);
    r.w2 = ldw_u1(tile + 256 + lane * 4);
  } else if constexpr (FMT == FMT_SQ4) {
    r.v = ldw_u2(tile + lane * 8);
    r.meta = ldw_u1(tile + 256 + lane * 4);
  } else if constexpr (FMT == FMT_F16) {
#pragma unroll
    for (int i = 0; i < 4; ++i) r.v[i] = ldw_u4(tile + i * 512 + lane * 16);
  } else {                                          // Q8, SP24
    r.v[0] = ldw_u4(tile + lane * 16);
    r.v[1] = ldw_u4(tile + 512 + lane * 16);
    if constexpr (FMT == FMT_SP24) r.meta = ldw_u1(tile + 1024 + lane * 4);
  }
}

// s, z: scales (s[row g] | s[row g + 8] << 16) and zero-points (z | z << 8) of the pair, or of each tile (SZ2: groups that are
// not a multiple of 128).
template <int FMT, bool SZ2> struct RawBlob {
  RawTile<FMT> t[2];
  uint32_t s[SZ2 ? 2 : 1], z[SZ2 ? 2 : 1];
};
template <int FMT, bool SZ2> __device__ __forceinline__ void load_blob(RawBlob<FMT, SZ2>& r, const uint8_t* blob, int lane) {
  constexpr int tb = tile_bytes(FMT);
  load_tile<FMT>(r.t[0], blob, lane);
  load_tile<FMT>(r.t[1], blob + tb, lane);
  if constexpr (fmt_quantised(FMT)) {
    const int g = lane >> 2;
#pragma unroll
    for (int i = 0; i < (SZ2 ? 2 : 1); ++i) {
      r.s[i] = ldw_u1(blob + 2 * tb + i * kSzEntryBytes + 4 * g);
      r.z[i] = ldw_u16(blob + 2 * tb + i * kSzEntryBytes + 32 + 2 * g);
    }
  }
}

// The same from a blob in shared memory (32-bit shared addresses).
__device__ __forceinline__ uint4 lds_u4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 lds_u2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u1(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_u1(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
template <int FMT> __device__ __forceinline__ void load_tile_s(RawTile<FMT>& r, uint32_t tile, int lane) {
  if constexpr (FMT == FMT_Q4) {
    r.v = lds_u4(tile + lane * 16);
  } else if constexpr (FMT == FMT_Q3 || FMT == FMT_SQ4) {
    r.v = lds_u2(tile + lane * 8);
    const uint32_t w = lds_u1(tile + 256 + lane * 4);
    if constexpr (FMT == FMT_Q3) r.w2 = w; else r.meta = w;
  } else if constexpr (FMT == FMT_F16) {
#pragma unroll
    for (int i = 0; i < 4; ++i) r.v[i] = lds_u4(tile + i * 512 + lane * 16);
  } else {                                          // Q8, SP24
    r.v[0] = lds_u4(tile + lane * 16);
    r.v[1] = lds_u4(tile + 512 + lane * 16);
    if constexpr (FMT == FMT_SP24) r.meta = lds_u1(tile + 1024 + lane * 4);
  }
}
template <int FMT, bool SZ2> __device__ __forceinline__ void load_blob_s(RawBlob<FMT, SZ2>& r, uint32_t blob, int lane) {
  constexpr int tb = tile_bytes(FMT);
  load_tile_s<FMT>(r.t[0], blob, lane);
  load_tile_s<FMT>(r.t[1], blob + tb, lane);
  if constexpr (fmt_quantised(FMT)) {
    const int g = lane >> 2;
#pragma unroll
    for (int i = 0; i < (SZ2 ? 2 : 1); ++i) {
      r.s[i] = lds_u1(blob + 2 * tb + i * kSzEntryBytes + 4 * g);
      r.z[i] = lds_u16(blob + 2 * tb + i * kSzEntryBytes + 32 + 2 * g);
    }
  }
}

// The wide operand of two of the tile's four mma.m16n8k16 as exact fp16 values: those of its 32-element block blk (0, 1).  `aux`:
// shared-memory address of the 2:4 expansion table (a multiple of 256); unused by other formats.
template <int FMT>
__device__ __forceinline__ void half_frags(const RawTile<FMT>& r, const ZC& zc, int blk, uint32_t (&a0)[4], uint32_t (&a1)[4], uint32_t aux) {
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {                   // row g, row g + 8: part 2 * blk + hf
    if constexpr (FMT == FMT_Q4) {
      const uint32_t lo = blk ? (hf ? r.v.w : r.v.z) : (hf ? r.v.y : r.v.x), hi = lo >> 8;
      a0[hf] = h2sub(and_or(lo, 0x000f000fu, kMagic), zc.c[hf][0]);
      a0[hf + 2] = h2fma(and_or(lo, 0x00f000f0u, kMagic), 0x2C002C00u, zc.c[hf][1]);   // * 1/16
      a1[hf] = h2sub(and_or(hi, 0x000f000fu, kMagic), zc.c[hf][0]);
      a1[hf + 2] = h2fma(and_or(hi, 0x00f000f0u, kMagic), 0x2C002C00u, zc.c[hf][1]);
    } else if constexpr (FMT == FMT_Q3) {
      uint32_t q0, q1;                               // the part's two byte quads of codes (q3_quads)
      if (blk == 1 && hf == 1) {
        q0 = and_or(r.w2 >> 4, 0x04040404u, (r.v.x >> 6) & 0x03030303u);
        q1 = and_or(r.w2 >> 5, 0x04040404u, (r.v.y >> 6) & 0x03030303u);
      } else {
        const uint32_t w = blk ? r.w2 : hf ? r.v.y : r.v.x;
        q0 = w & 0x07070707u; q1 = (w >> 3) & 0x07070707u;
      }
      a0[hf] = h2sub(quad_pair(q0, 0), zc.c[hf][0]); a0[hf + 2] = h2sub(quad_pair(q0, 1), zc.c[hf][0]);
      a1[hf] = h2sub(quad_pair(q1, 0), zc.c[hf][0]); a1[hf + 2] = h2sub(quad_pair(q1, 1), zc.c[hf][0]);
    } else if constexpr (FMT == FMT_Q8) {
      const uint32_t w0 = hf ? r.v[blk].z : r.v[blk].x, w1 = hf ? r.v[blk].w : r.v[blk].y;
      a0[hf] = h2sub(and_or(w0, 0x00ff00ffu, kMagic), zc.c[hf][0]);
      a0[hf + 2] = h2sub(and_or(w0 >> 8, 0x00ff00ffu, kMagic), zc.c[hf][0]);
      a1[hf] = h2sub(and_or(w1, 0x00ff00ffu, kMagic), zc.c[hf][0]);
      a1[hf + 2] = h2sub(and_or(w1 >> 8, 0x00ff00ffu, kMagic), zc.c[hf][0]);
    } else if constexpr (FMT == FMT_F16) {
      const uint4 u = r.v[2 * blk + hf];
      a0[hf] = u.x; a0[hf + 2] = u.y; a1[hf] = u.z; a1[hf + 2] = u.w;
    } else {
      // 2:4 formats: a quad's two kept values (SQ4: two codes made exact fp16 values first) are spread over its four
      // positions with two byte permutes whose selectors come from the table.
#pragma unroll
      for (int quad = 0; quad < 2; ++quad) {
        uint32_t kept;
        if constexpr (FMT == FMT_SP24) {
          const uint4 u = r.v[blk];
          kept = hf ? (quad ? u.w : u.z) : (quad ? u.y : u.x);
        } else {
          kept = h2sub(and_or((blk ? r.v.y : r.v.x) >> (8 * hf + 4 * quad), 0x000f000fu, kMagic), zc.c[hf][0]);
        }
        // Nibble * 4 = byte offset into the table; one permute puts it under the table's address.
        const uint32_t offs = (quad ? r.meta >> 2 : r.meta << 2) & 0x3C3C3C3Cu;
        uint32_t sel;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(sel) : "r"(prmt(offs, aux, 0x7650u + (uint32_t)(blk * 2 + hf))));
        (quad ? a1 : a0)[hf] = prmt(kept, 0u, sel);
        (quad ? a1 : a0)[hf + 2] = prmt(kept, 0u, sel >> 16);
      }
    }
  }
}
// All four: a[2 * blk + sub][*].
template <int FMT>
__device__ __forceinline__ void tile_frags(const RawTile<FMT>& r, const ZC& zc, uint32_t (&a)[4][4], uint32_t aux) {
  half_frags<FMT>(r, zc, 0, a[0], a[1], aux);
  half_frags<FMT>(r, zc, 1, a[2], a[3], aux);
}

// 3/4-bit codes as the fp16 bit patterns they are in their words (subnormals q * 2^-24): a[2 * blk] with the codes at the low end of
// their half-words, a[2 * blk + 1] with those four (three) bits up, i.e. 16 (8) times as large.
template <int FMT>
__device__ __forceinline__ void code_frags(const RawTile<FMT>& r, uint32_t (&a)[4][4]) {
  if constexpr (FMT == FMT_Q4) {
    const uint32_t w[4] = {r.v.x, r.v.y, r.v.z, r.v.w};
#pragma unroll
    for (int part = 0; part < 4; ++part) {
      const int hf = part & 1, blk = part >> 1;
      const uint32_t hi = w[part] >> 8;
      a[blk * 2 + 0][hf] = w[part] & 0x000f000fu; a[blk * 2 + 0][hf + 2] = hi & 0x000f000fu;       // elements (0, 1), (4, 5)
      a[blk * 2 + 1][hf] = w[part] & 0x00f000f0u; a[blk * 2 + 1][hf + 2] = hi & 0x00f000f0u;       // elements (2, 3), (6, 7)
    }
  } else {
    const uint32_t w[3] = {r.v.x, r.v.y, r.w2};
#pragma unroll
    for (int part = 0; part < 3; ++part) {
      const int hf = part & 1, blk = part >> 1;
      const uint32_t hi = w[part] >> 8;
      a[blk * 2 + 0][hf] = w[part] & 0x00070007u; a[blk * 2 + 0][hf + 2] = hi & 0x00070007u;       // elements (0, 2), (1, 3)
      a[blk * 2 + 1][hf] = w[part] & 0x00380038u; a[blk * 2 + 1][hf + 2] = hi & 0x00380038u;       // elements (4, 6), (5, 7)
    }
    // part 3 from the spare bits (see the layout)
    a[2][1] = and_or(r.w2 >> 4, 0x00040004u, (w[0] >> 6) & 0x00030003u);
    a[2][3] = and_or(r.w2 >> 12, 0x00040004u, (w[0] >> 14) & 0x00030003u);
    a[3][1] = and_or(r.w2 >> 2, 0x00200020u, (w[1] >> 3) & 0x00180018u);
    a[3][3] = and_or(r.w2 >> 10, 0x00200020u, (w[1] >> 11) & 0x00180018u);
  }
}

// ------------------------------------------------------------------------------------------ integer path (M = 1)
// With a single token the fp16 tensor-core product wastes seven of its eight columns and needs the codes as fp16 pairs.
// The integer product keeps the codes as bytes (one and extracts four of them) and multiplies them with mma.m16n8k32
// (s8 x s8 -> s32): a 16 x 128 blob is four instructions.  The 128 activations of a pair are turned once into a 16-bit
// block fixed-point number, x = v * 2^e with |v| <= 32639 and one power-of-two scale per pair (so the products are exact
// and one-hot inputs reproduce the weights bit for bit), split into two signed byte planes (v = 256 * high + low) that
// are columns 0 and 1 of the MMA's narrow operand.  Zero-point and scales follow per group, in fp32:
//   y += s * 2^e * (sum q v - z * sum v).
__device__ __forceinline__ void mma16832_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Byte quads of a tile's parts (8 codes of one row): q[part][0] the codes an and delivers first, q[part][1] the others.
template <int FMT>
__device__ __forceinline__ void code_quads(const RawTile<FMT>& r, uint32_t (&q)[4][2]) {
  if constexpr (FMT == FMT_Q4) {
    const uint32_t w[4] = {r.v.x, r.v.y, r.v.z, r.v.w};
#pragma unroll
    for (int part = 0; part < 4; ++part) {
      q[part][0] = w[part] & 0x0f0f0f0fu;
      q[part][1] = (w[part] >> 4) & 0x0f0f0f0fu;
    }
  } else {
    q3_quads(r.v.x, r.v.y, r.w2, q);
  }
}

// ------------------------------------------------------------------------------------------ deal, exchange of t
struct Share { uint32_t per, rem; };      // items dealt to n takers: taker i gets per + (i < rem)
__device__ __forceinline__ uint32_t share_lo(const Share& s, uint32_t i) { return i * s.per + (i < s.rem ? i : s.rem); }
__device__ __forceinline__ uint32_t share_n(const Share& s, uint32_t i) { return s.per + (i < s.rem ? 1u : 0u); }

__device__ __forceinline__ uint4 ld_cg_u4(const void* p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
  __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t bf2_to_h2(uint32_t v) {
  return pack_h2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }


// Launches of a handle are numbered from 1 (the kernels of the decode family share the count).  A launch adds 2^16 in all: a
// CTA's 1, and the last CTA of the grid the rest, so that the count never reaches the next multiple before every CTA has
// read it (a CTA adds its share after its reads, at most 65535 CTAs: 25 million outputs).
constexpr uint32_t kLaunchShift = 16;
__device__ __forceinline__ uint32_t launch_number(const unsigned long long* launches) {
  return (uint32_t)(ld_volatile_u64(launches) >> kLaunchShift) + 1u;
}
__device__ __forceinline__ void count_launch(unsigned long long* launches) {
  const unsigned long long v = blockIdx.x + 1 == gridDim.x ? (1ull << kLaunchShift) - (gridDim.x - 1) : 1ull;
  asm volatile("red.global.add.u64 [%0], %1;" ::"l"(launches), "l"(v) : "memory");
}

// Two neighbouring columns of t, one part of the reduction axis: asked for (load) and, until the launch's words are there, again.
struct TWords { unsigned long long a, b; };
__device__ __forceinline__ void load_t(TWords& w, const unsigned long long* src) {
  asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.a), "=l"(w.b) : "l"(src) : "memory");
}
__device__ __forceinline__ bool wait_t(TWords& w, const unsigned long long* src, uint32_t launch, unsigned long long limit_ns, int* dev_status) {
  unsigned long long t0 = 0;
  for (uint32_t tries = 1;; ++tries) {
    if ((uint32_t)(w.a >> 32) == launch && (uint32_t)(w.b >> 32) == launch) return true;
    if ((tries & 63u) == 0u) {
      const unsigned long long now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) { atomicExch(dev_status, EORA_ERR_DEVICE_TIMEOUT); return false; }
    }
    load_t(w, src);
  }
}

// A warp's ring of weights in shared memory: position of the slot that is read next, its barrier and the phase it completes.
struct Ring { uint32_t base, bytes, bars, so, bar, parity; };
__device__ __forceinline__ void ring_next(Ring& r, uint32_t slot_b) {
  r.so += slot_b; r.bar += 8;
  if (r.so == r.bytes) { r.so = 0; r.bar = r.bars; r.parity ^= 1u; }
}

__device__ __forceinline__ void store_y(void* y, int dtype, int64_t i, float v) {
  if (dtype == EORA_Y_F16) reinterpret_cast<__half*>(y)[i] = __float2half_rn(v);
  else if (dtype == EORA_Y_BF16) reinterpret_cast<__nv_bfloat16*>(y)[i] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(y)[i] = v;
}

}  // namespace dec
}  // namespace eora
