// A tile's logits in the epilogues of the persistent kernels: tensor-memory
// loads of 32 keys x 32 query rows, packed fp32 arithmetic on them and their
// sums over keys and over query rows.
#pragma once

#include "ckv_device.cuh"

namespace ckv {
namespace {

// `p` points to shared memory: plain shared-memory instructions instead of
// generic ones, in functions that are not inlined.
template <class T>
__device__ __forceinline__ void assume_shared(const T* p) {
  __builtin_assume(__isShared(p));
}

// Two fp32 numbers in a register pair, and packed arithmetic on them.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t exp2_2(uint64_t v) {
  float a, b;
  unpack2(v, a, b);
  return pack2(ex2_approx(a), ex2_approx(b));
}

// True in one lane of the warp (the same one every time).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "elect.sync _|P, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, P;\n\t}"
      : "=r"(p));
  return p != 0u;
}

// A 32-key x 32-column block of logits in the 16x256b shape: r[16 h + 4 j +
// 2 b + a] is key 16 h + 8 b + lane / 4, column 8 j + 2 (lane % 4) + a.
__device__ __forceinline__ void tmem_load_block(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr), "r"(taddr + (16u << 16))
      : "memory");
}

// Sum of v[i] over the 8 lanes that share lane % 4; on return the lane holds
// column slot i = block_slot(lane).
__device__ __forceinline__ int block_slot(int lane) {
  return ((lane & 16) >> 2) | ((lane & 8) >> 2) | ((lane & 4) >> 2);
}
__device__ __forceinline__ int block_col(int lane) {  // column of that slot
  const int i = block_slot(lane);
  return 8 * (i >> 1) + 2 * (lane & 3) + (i & 1);
}
__device__ __forceinline__ float sum_over_keys(float (&v)[8], int lane) {
#pragma unroll
  for (int half = 4, bit = 16; half >= 1; half >>= 1, bit >>= 1) {
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = up ? v[i] : v[i + half];
      const float keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
  }
  return v[0];
}
// Sum of the 4 keys' values over the 4 lanes that share lane / 4; on return
// the lane holds key block_key(lane).
__device__ __forceinline__ int block_key(int lane) {
  return (lane >> 2) + 8 * (lane & 1) + 8 * (lane & 2);
}
__device__ __forceinline__ float sum_over_cols(float (&v)[4], int lane) {
#pragma unroll
  for (int half = 2, bit = 2; half >= 1; half >>= 1, bit >>= 1) {
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = up ? v[i] : v[i + half];
      const float keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
  }
  return v[0];
}

// Which of a lane's 32 elements of a block are attended: key < L, key no
// later than the row's position (window position + n), column < lim.
__device__ __noinline__ uint32_t block_mask(int c0, int window, int lim, int tok0, int n, int L,
                                            int lane) {
  int wpos[8];  // window positions of the lane's columns
#pragma unroll
  for (int i = 0; i < 8; ++i) wpos[i] = (c0 + 8 * (i >> 1) + 2 * (lane & 3) + (i & 1)) % window;
  uint32_t m = 0u;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const int tok = tok0 + 16 * h + 8 * b + (lane >> 2);
          const int col = 8 * j + 2 * (lane & 3) + a;
          const bool ok = col < lim && tok < L && wpos[2 * j + a] >= tok - n;
          m |= (ok ? 1u : 0u) << (16 * h + 4 * j + 2 * b + a);
        }
  return m;
}

}  // namespace
}  // namespace ckv
