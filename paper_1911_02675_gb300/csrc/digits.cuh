// digits.cuh -- FP64 values as balanced base-256 digits in BF16, for exact products on the tensor cores
// (gram.cu, gauss64.cu).  A column is put in fixed point on the scale of its largest element:
//   T = x 2^(1084 - emax), |T| < 2^62,  T = sum_i D_i 256^(7-i), |D_i| <= 128 (exact in BF16),
// emax the exponent field of the largest magnitude.  A value loses only bits below 2^-62 of it.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace lsq_digits {

constexpr unsigned long long BIAS = 0x8080808080808080ull;  // T + BIAS holds the digits + 128 as bytes

// T + BIAS for x on the scale emax >= its exponent field
__device__ __forceinline__ unsigned long long biased_digits(double x, int emax) {
  const uint32_t hi = (uint32_t)__double2hiint(x);
  const int ec = (int)((hi >> 20) & 0x7FFu);
  const unsigned long long M =
      ((unsigned long long)((hi & 0xFFFFFu) | (ec ? 0x100000u : 0u)) << 32) | (uint32_t)__double2loint(x);
  const int sh = emax - max(ec, 1) - 9;  // M 2^-sh below 2^62
  const unsigned long long t = sh <= 0 ? M << -sh : sh < 64 ? M >> sh : 0ull;
  return BIAS + ((hi >> 31) ? 0ull - t : t);
}

// digits i of two values, as a pair of BF16: 2^23 + byte - (2^23 + 128) is the digit, exact in the
// upper 16 bits of its FP32 form
__device__ __forceinline__ uint32_t digit_pair(unsigned long long u0, unsigned long long u1, int i) {
  const uint32_t b0 = (uint32_t)(u0 >> (56 - 8 * i)) & 0xFFu, b1 = (uint32_t)(u1 >> (56 - 8 * i)) & 0xFFu;
  const float f0 = __uint_as_float(0x4B000000u | b0) - 8388736.f, f1 = __uint_as_float(0x4B000000u | b1) - 8388736.f;
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
}

// largest magnitude of every column (high words): mag[c], zeroed before
template <typename TA>
__global__ void __launch_bounds__(256) column_max_kernel(const TA* __restrict__ A, int64_t n, int d, int64_t ld,
                                                         uint32_t* __restrict__ mag) {
  const int c = blockIdx.x * 32 + (threadIdx.x & 31);
  const int w = threadIdx.x >> 5;
  if (c >= d) return;
  uint32_t v = 0;
  const int64_t step = 8 * (int64_t)gridDim.y;
  for (int64_t r = blockIdx.y * 8 + w; r < n; r += step)
    v = max(v, (uint32_t)__double2hiint((double)__ldg(A + r * ld + c)) & 0x7FFFFFFFu);
  atomicMax(mag + c, v);
}

// digits of rows [r0, r0 + rows) of A (zeros from n on): plane i at out + i rows dq, row pitch dq; two
// columns a thread, 64 columns a block and every 8 gridDim.y-th row.  Of each column's elements there,
// counts[c] (zeroed before) counts those whose exponent is at most `gap` below the column's largest, and
// with NZ counts[d + c] those that are not zero.
template <typename TA, int NS, bool NZ>
__global__ void __launch_bounds__(256) digits_kernel(const TA* __restrict__ A, int64_t n, int d, int64_t ld, int dq,
                                                     int64_t r0, int rows, const uint32_t* __restrict__ mag, int gap,
                                                     uint32_t* __restrict__ counts, uint32_t* __restrict__ out) {
  __shared__ uint32_t cnt[NZ ? 2 : 1][64];
  const int half = dq / 2, p = 2 * (threadIdx.x & 31), c = blockIdx.x * 64 + p;
  const int64_t plane = (int64_t)rows * half;
  int emax[2], least[2];
  uint32_t large[2] = {0u, 0u}, nonzero[2] = {0u, 0u};
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    emax[q] = c + q < d ? max((int)(mag[c + q] >> 20), 1) : 1;
    least[q] = max(emax[q] - gap, 1);
  }
  for (int e = threadIdx.x; e < (NZ ? 128 : 64); e += 256) cnt[e >> 6][e & 63] = 0u;
  for (int r = blockIdx.y * 8 + (threadIdx.x >> 5); r < rows; r += 8 * gridDim.y) {
    unsigned long long U[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const double x = r0 + r < n && c + q < d ? (double)__ldg(A + (r0 + r) * ld + c + q) : 0.0;
      U[q] = biased_digits(x, emax[q]);
      large[q] += (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7FFu) >= least[q] ? 1u : 0u;
      if (NZ) nonzero[q] += ((uint32_t)__double2hiint(x) << 1 | (uint32_t)__double2loint(x)) != 0u ? 1u : 0u;
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) out[i * plane + (int64_t)r * half + c / 2] = digit_pair(U[0], U[1], i);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (large[q]) atomicAdd(&cnt[0][p + q], large[q]);
    if (NZ && nonzero[q]) atomicAdd(&cnt[NZ ? 1 : 0][p + q], nonzero[q]);
  }
  __syncthreads();
  const int col = blockIdx.x * 64 + threadIdx.x;
  if (threadIdx.x < 64 && col < d) {
#pragma unroll
    for (int k = 0; k < (NZ ? 2 : 1); ++k)
      if (cnt[k][threadIdx.x]) atomicAdd(counts + k * d + col, cnt[k][threadIdx.x]);
  }
}

// its grid: a row a warp, at most eight blocks an SM
inline dim3 lsq_digits_grid(int dq, int rows, int sm_count) {
  const int gx = dq / 64;
  return dim3((unsigned)gx, (unsigned)std::max(1, std::min((rows + 7) / 8, (8 * sm_count + gx - 1) / gx)));
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(p)));
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// 2^k for any k that FP64 holds, subnormal powers included
__device__ __forceinline__ double pow2(int k) {
  return k >= -1022 ? __longlong_as_double((long long)(k + 1023) << 52) : __longlong_as_double(1ll << (k + 1074));
}

}  // namespace lsq_digits
