// apassdg.cuh -- the dot products of the FP64 pass over A on the tensor cores, from digit products.
// Internal, not part of the ABI.
//
// The FP64 pass spends 4 flops an element on a pipe that does 1.75 multiply-adds a clock an SM; here
// the products w = A p take none of it, and only v = A^T w stays there.  p is written once per pass as
// p_j = T_j 2^(e_j - 1076), T_j an integer below 2^54 in 7 balanced base-256 digits.  The elements of a
// row's 64 columns are put on one scale with the exponents of p taken in, E = max (e(a_ij) + e_j):
//   a_ij = U_ij 2^(E - e_j - 1084), |U_ij| < 2^62, 8 digits,   a_ij p_j = U_ij T_j 2^(E - 2160),
// so an element loses only what lies 2^-61 below the row's largest |a_ij p_j| there, whatever the
// scales of rows and columns: w is at least as near to A p as with FP64 additions, which round at
// 2^-53 of the partial sums.  The digits of a 16 x 16 tile of A are formed in registers, in the layout
// that an m16n8k16 MMA wants of its first operand, as FP16 subnormals (byte b is b 2^-24: one byte
// permutation, no arithmetic); the second operand of digit i holds in column s the digit s - i of p, so
// that the 8 columns collect the sums over i + k = s of digits i of A and k of p (i + k > 7 lies below
// 2^-59).  A product is at most 255 x 128 and 7 of them in 64 columns stay below 2^24: the FP32
// accumulators are exact.  (The bytes are digits + 128: 128 times the sums of p's digits comes off.)
// Elements 2^-64 or more below the scale, zeros and subnormals among them, become 0; rows that hold an
// infinity or a NaN, or whose largest product is outside 2^-796 ... 2^854, take FP64 arithmetic, and so
// does the pass if p is not finite or its largest entry is outside 2^-600 ... 2^600.
#pragma once

#include <cuda_fp16.h>

namespace lsq_apass {

constexpr int DG = 7;              // digits of an entry of p (an element of A has 8)
constexpr int DG_ROWS = 2 * DG + 1;  // rows of the table of p's digits: 7 of zeros, the digits, 1 of zeros
constexpr int DG_MIN_ROWS = 384;   // rows of a CTA from which the 16-row tiles of its 8 warps are even enough

// the tables, in the shared memory of the (not yet used) reduction buffer: 34.5 dk + 480 bytes of its
// 64 dp, dk = d rounded up to 64
struct DigitTab {
  uint32_t* epk;   // dk: exponent fields of p << 20, the columns of a lane's fragment adjacent
  int* corr;       // dk / 64 x 8: what the digits' + 128 adds to the 8 sums of 64 columns
  __half* dig;     // DG_ROWS x pitch: digits of p, in the order of epk
  int pitch;       // halves: 32 bytes past a multiple of 128, distinct banks for a half-warp's rows
  int lo;          // rows with E <= lo are left to FP64
};

__device__ __forceinline__ DigitTab digit_tab(double* wred, int dk) {
  DigitTab t;
  t.epk = reinterpret_cast<uint32_t*>(wred);
  t.corr = reinterpret_cast<int*>(t.epk + dk);
  t.dig = reinterpret_cast<__half*>(t.corr + dk / 8);
  t.pitch = dk + 16;
  t.lo = 0;
  return t;
}

// fills the tables from p (all threads); false if p is out of range.  red: 8 ints of scratch.
__device__ inline bool digit_prep(DigitTab& t, int d, int dk, const double* vec_s, int* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t mx = 0;
  for (int c = threadIdx.x; c < d; c += blockDim.x) mx = max(mx, (uint32_t)__double2hiint(vec_s[c]) & 0x7FFFFFFFu);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) red[warp] = (int)mx;
  for (int c = threadIdx.x; c < t.pitch; c += blockDim.x) {
#pragma unroll
    for (int r = 0; r < DG; ++r) t.dig[r * t.pitch + c] = __ushort_as_half(0);
    t.dig[(DG_ROWS - 1) * t.pitch + c] = __ushort_as_half(0);
  }
  for (int ch = warp; ch < dk / 64; ch += LSQ_WARPS) {
    int sum[DG];
#pragma unroll
    for (int k = 0; k < DG; ++k) sum[k] = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = 64 * ch + 32 * h + lane;
      const double p = c < d ? vec_s[c] : 0.0;
      const uint32_t hi = (uint32_t)__double2hiint(p);
      const uint32_t ep = (hi >> 20) & 0x7FFu;
      long long T = (long long)((((unsigned long long)((hi & 0xFFFFFu) | (ep ? 0x100000u : 0u)) << 32) |
                                 (uint32_t)__double2loint(p)) << 1);
      if (hi >> 31) T = -T;
      const unsigned long long b = (unsigned long long)T + 0x0080808080808080ull;
      const int pos = (c & ~15) + 4 * (c & 3) + ((c >> 2) & 3);
      t.epk[pos] = max(ep, p != 0.0 ? 1u : 0u) << 20;
#pragma unroll
      for (int k = 0; k < DG; ++k) {
        const int D = (int)((uint32_t)(b >> (8 * (DG - 1 - k))) & 0xFFu) - 128;
        t.dig[(DG + k) * t.pitch + pos] = __int2half_rn(D);
        sum[k] += D;
      }
    }
#pragma unroll
    for (int k = 0; k < DG; ++k) sum[k] = __reduce_add_sync(0xffffffffu, sum[k]);
    if (lane < 8) {
      // sum s takes the digits k = s - i of p, one for each digit i of A
      int v = 0;
#pragma unroll
      for (int k = 0; k < DG; ++k) v += k <= lane ? sum[k] : 0;
      t.corr[8 * ch + lane] = 128 * v;
    }
  }
  __syncthreads();
  uint32_t m = 0;
#pragma unroll
  for (int w = 0; w < LSQ_WARPS; ++w) m = max(m, (uint32_t)red[w]);
  __syncthreads();  // red is read before a warp leaves its q there
  const int e = (int)(m >> 20);
  t.lo = max(e + 64, 1250);
  return e >= 1023 - 600 && e <= 1023 + 600;
}

constexpr int DG_HI = 2900;  // rows with E >= DG_HI are left to FP64

// biased digits of a, sh bits below the scale: digit i in byte 7 - i
__device__ __forceinline__ void digit_bytes(double a, int sh, uint32_t& u0, uint32_t& u1) {
  uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t neg = (uint32_t)((int)hi >> 31);
  hi = (hi & 0xFFFFFu) | 0x100000u;
  hi = __funnelshift_l(lo, hi, 9);
  lo <<= 9;
  if (sh >= 32) {
    lo = hi;
    hi = 0;
    sh -= 32;
  }
  lo = __funnelshift_rc(lo, hi, sh);
  hi = __funnelshift_rc(hi, 0u, sh);
  asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
      : "=r"(u0), "=r"(u1)
      : "r"(lo ^ neg), "r"(hi ^ neg), "r"(0x80808080u - neg), "r"(0x80808080u));
}

__device__ __forceinline__ void mma_f16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the contribution of columns [c0, c0 + 64) to w of rows g (pa) and g + 8 (pb); false if a row's scale
// is out of range.  Columns from d on read column d - 1 against zero digits of p.
template <bool FULL, typename TA>
__device__ __forceinline__ bool digit_chunk(const TA* __restrict__ pa, const TA* __restrict__ pb, int c0, int d,
                                            const DigitTab& t, double& w0, double& w1) {
  const int lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
  auto col = [&](int kt, int e) { return FULL ? c0 + 16 * kt + tq + 4 * e : min(c0 + 16 * kt + tq + 4 * e, d - 1); };
  // the scales: a first look at the high words (the second finds the elements in L1)
  uint32_t k0 = 0, k1 = 0, m0 = 0, m1 = 0;
#pragma unroll
  for (int kt = 0; kt < 4; ++kt)
    if (FULL || c0 + 16 * kt < d) {
      const uint4 q4 = *reinterpret_cast<const uint4*>(t.epk + c0 + 16 * kt + 4 * tq);
      const uint32_t ep[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t x = (uint32_t)__double2hiint(ld_elem(pa + col(kt, e))) & 0x7FFFFFFFu;
        const uint32_t y = (uint32_t)__double2hiint(ld_elem(pb + col(kt, e))) & 0x7FFFFFFFu;
        m0 = max(m0, x);
        m1 = max(m1, y);
        k0 = max(k0, x + ep[e]);
        k1 = max(k1, y + ep[e]);
      }
    }
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    k0 = max(k0, __shfl_xor_sync(0xffffffffu, k0, o));
    k1 = max(k1, __shfl_xor_sync(0xffffffffu, k1, o));
    m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
    m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
  }
  int E0 = (int)(k0 >> 20), E1 = (int)(k1 >> 20);
  const bool ok = (m0 == 0 || (m0 < 0x7FF00000u && E0 > t.lo && E0 < DG_HI)) &&
                  (m1 == 0 || (m1 < 0x7FF00000u && E1 > t.lo && E1 < DG_HI));
  // a row of zeros: every shift past 64
  if (m0 == 0) E0 = 4095;
  if (m1 == 0) E1 = 4095;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int kt = 0; kt < 4; ++kt)
    if (FULL || c0 + 16 * kt < d) {
      const uint4 q4 = *reinterpret_cast<const uint4*>(t.epk + c0 + 16 * kt + 4 * tq);
      const uint32_t ep[4] = {q4.x, q4.y, q4.z, q4.w};
      uint32_t x0[4], x1[4], y0[4], y1[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double x = ld_elem(pa + col(kt, e)), y = ld_elem(pb + col(kt, e));
        const uint32_t kx = ((uint32_t)__double2hiint(x) & 0x7FFFFFFFu) + ep[e];
        const uint32_t ky = ((uint32_t)__double2hiint(y) & 0x7FFFFFFFu) + ep[e];
        digit_bytes(x, E0 - (int)(kx >> 20), x0[e], x1[e]);
        digit_bytes(y, E1 - (int)(ky >> 20), y0[e], y1[e]);
      }
      // two bytes of two elements at a time, then each pair of bytes widened
      const __half* dp = t.dig + (g + DG) * t.pitch + c0 + 16 * kt + 4 * tq;
#pragma unroll
      for (int h = 0; h < 4; ++h) {  // bytes 2h, 2h + 1
        const uint32_t sel = (h & 1) ? 0x7632u : 0x5410u;
        const uint32_t p0 = h < 2 ? __byte_perm(x0[0], x0[1], sel) : __byte_perm(x1[0], x1[1], sel);
        const uint32_t p1 = h < 2 ? __byte_perm(y0[0], y0[1], sel) : __byte_perm(y1[0], y1[1], sel);
        const uint32_t p2 = h < 2 ? __byte_perm(x0[2], x0[3], sel) : __byte_perm(x1[2], x1[3], sel);
        const uint32_t p3 = h < 2 ? __byte_perm(y0[2], y0[3], sel) : __byte_perm(y1[2], y1[3], sel);
        const int i0 = 7 - 2 * h;  // digit of the even byte
        {
          const uint2 b = *reinterpret_cast<const uint2*>(dp - i0 * t.pitch);
          const uint32_t a[4] = {p0 & 0x00FF00FFu, p1 & 0x00FF00FFu, p2 & 0x00FF00FFu, p3 & 0x00FF00FFu};
          mma_f16_16816(acc, a, b.x, b.y);
        }
        {
          const uint2 b = *reinterpret_cast<const uint2*>(dp - (i0 - 1) * t.pitch);
          const uint32_t a[4] = {__byte_perm(p0, 0u, 0x4341u), __byte_perm(p1, 0u, 0x4341u),
                                 __byte_perm(p2, 0u, 0x4341u), __byte_perm(p3, 0u, 0x4341u)};
          mma_f16_16816(acc, a, b.x, b.y);
        }
      }
    }
  // lane's sums s = 2 tq, 2 tq + 1 of both rows, as one integer below 2^31 in magnitude each
  const int2 cr = *reinterpret_cast<const int2*>(t.corr + c0 / 8 + 2 * tq);
  const int X0 = (__float2int_rn(acc[0] * 16777216.f) - cr.x) * 256 + (__float2int_rn(acc[1] * 16777216.f) - cr.y);
  const int X1 = (__float2int_rn(acc[2] * 16777216.f) - cr.x) * 256 + (__float2int_rn(acc[3] * 16777216.f) - cr.y);
  // 2^52 + 2^31 + X as bits, less 2^52 + 2^31
  const double f0 = __hiloint2double(0x43300000, (int)((uint32_t)X0 ^ 0x80000000u)) - 4503601774854144.0;
  const double f1 = __hiloint2double(0x43300000, (int)((uint32_t)X1 ^ 0x80000000u)) - 4503601774854144.0;
  const int s = 1023 - 2064 - 16 * tq;  // X 256^(12 - 2 tq) 2^(E - 2160)
  w0 = fma(f0, __hiloint2double((m0 == 0 || !ok ? 1023 : E0 + s) << 20, 0), w0);
  w1 = fma(f1, __hiloint2double((m1 == 0 || !ok ? 1023 : E1 + s) << 20, 0), w1);
  return ok;
}

// w of 16 rows in FP64 (rows the digits do not take)
template <typename TA>
__device__ __noinline__ void tile_dots_f64(const TA* __restrict__ A, int64_t ld, int d, int nr, const double* vec_s,
                                           double* out /* w0, w1 of this lane */) {
  const int lane = threadIdx.x & 31, g = lane >> 2;
  for (int r = 0; r < nr; ++r) {
    double s = 0.0;
    for (int c = lane; c < d; c += 32) s = fma(ld_elem(A + (int64_t)r * ld + c), vec_s[c], s);
    s = warp_sum(s);
    if (g == (r & 7)) out[r >> 3] = s;
  }
}

// fused_rows with the dot products from digits, 16 rows of a warp at a time
template <typename TA, int NK>
__device__ __forceinline__ void digit_rows(const TA* __restrict__ A, int64_t ld, int d, int64_t r0, int64_t r1,
                                           const double* vec_s, const DigitTab& t, double (&acc)[NK], double& q) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2;
#pragma unroll
  for (int k = 0; k < NK; ++k) acc[k] = 0.0;
  q = 0.0;
  for (int64_t i = r0 + 16 * warp; i < r1; i += 16 * LSQ_WARPS) {
    const int nr = (int)min((int64_t)16, r1 - i);
    const TA* tile = A + i * ld;
    const TA* pa = tile + min(g, nr - 1) * ld;
    const TA* pb = tile + min(g + 8, nr - 1) * ld;
    double w[2] = {0.0, 0.0};
    bool ok = true;
    int c0 = 0;
#pragma unroll 1
    for (; c0 + 64 <= d; c0 += 64) ok &= digit_chunk<true>(pa, pb, c0, d, t, w[0], w[1]);
    if (c0 < d) ok &= digit_chunk<false>(pa, pb, c0, d, t, w[0], w[1]);
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      w[0] += __shfl_xor_sync(0xffffffffu, w[0], o);
      w[1] += __shfl_xor_sync(0xffffffffu, w[1], o);
    }
    if (!__all_sync(0xffffffffu, ok)) {
      double f[2] = {0.0, 0.0};
      tile_dots_f64(tile, ld, d, nr, vec_s, f);
      w[0] = f[0];
      w[1] = f[1];
    }
    if (g < nr) q = fma(w[0], w[0], q);
    if (g + 8 < nr) q = fma(w[1], w[1], q);
#pragma unroll 1
    for (int j = 0; j < 8 && j < nr; ++j) {
      const double wa = __shfl_sync(0xffffffffu, w[0], 4 * j), wb = __shfl_sync(0xffffffffu, w[1], 4 * j);
      const TA* ra = tile + j * ld + lane;
      const TA* rb = ra + 8 * ld;
      const bool two = j + 8 < nr;
      double x[NK], y[NK];
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        const bool in = k < NK - 2 || lane + 32 * k < d;
        x[k] = in ? ld_elem(ra + 32 * k) : 0.0;
        y[k] = in && two ? ld_elem(rb + 32 * k) : 0.0;
      }
#pragma unroll
      for (int k = 0; k < NK; ++k) acc[k] = fma(wa, x[k], acc[k]);
      if (two) {
#pragma unroll
        for (int k = 0; k < NK; ++k) acc[k] = fma(wb, y[k], acc[k]);
      }
    }
  }
  // the four lanes of a row hold the same q: add the rows
#pragma unroll
  for (int o = 4; o <= 16; o <<= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
}

}  // namespace lsq_apass
