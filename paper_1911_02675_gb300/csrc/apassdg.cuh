// apassdg.cuh -- the dot products of the FP64 pass over A on the tensor cores, from digit products.
// Internal, not part of the ABI.
//
// The FP64 pass spends 4 flops an element on a pipe that does 1.75 multiply-adds a clock an SM; here
// the products w = A p take almost none of it, and only v = A^T w stays there.  p is written once per
// pass as p_j = T_j 2^(e_j - 1076), T_j an integer below 2^54 in 7 balanced base-256 digits.  The
// elements of a row's 32 columns are put on one scale with the exponents of p taken in,
// E = max (e(a_ij) + e_j):
//   a_ij = U_ij 2^(E - e_j - 1084), |U_ij| < 2^62, 8 bytes and a sign,   a_ij p_j = U_ij T_j 2^(E - 2160),
// so an element loses only what lies 2^-61 below the row's largest |a_ij p_j| there, whatever the
// scales of rows and columns: w is at least as near to A p as with FP64 additions, which round at
// 2^-53 of the partial sums.  The bytes of a 16 x 16 tile of A are formed in registers, in the layout
// that an m16n8k16 MMA wants of its first operand, as FP16 subnormals (byte b is b 2^-24, with the sign of
// its element: byte permutations, no arithmetic); the second operand of byte i holds in column s the digit
// s - i of p, so that the 8 columns collect the sums over i + k = s of bytes i of A and digits k of p
// (i + k > 7 lies below 2^-59).  A product is at most 255 x 128 and 7 of them in 32 columns stay below
// 2^24: the FP32 accumulators are exact.  With signs and magnitudes (and not complements), elements that
// fit their scale are exact whatever their sign, so sums of products that FP64 forms without rounding
// (integers, A p = 0) are the same here: their nonzero bytes and digits have i + k <= 7.
// Elements 2^-64 or more below the scale, zeros and subnormals among them, become 0, and so do those that
// meet a zero of p (they would set the scale of products that do not exist; 600011 x 333 with 64 zeros in
// p, 619 us, with 111 of them everywhere 667); rows that hold an
// infinity or a NaN, or whose largest product is outside 2^-796 ... 2^854, take FP64 arithmetic, and so
// does the pass if p is not finite, its largest entry is outside 2^-600 ... 2^600 or it has subnormal ones
// (whose digits do not fill their scale).
//
// Bound by the FP64 pipe, now with one multiply-add an element and two instructions per 32 columns of 16
// rows: 70% busy by its counter.  (The rest is the integer work of the digits, about 25 instructions an element, and
// loads of 8 rows each, whose 8 cache lines take as many cycles: chunks of 64 columns, looked at twice,
// spent more there than they saved in FP64.  More warps or rows prefetched into L2 gave nothing.)
// Measured: 600011 x 333, FP64 sums 859 us, chunks of 64 columns 661, this 605; 1200011 x 160, 540 us.
// FP32 rows keep FP64 sums (widening twice costs more: 1231 against 1618 us at 622592 x 301), and so do
// rows of more than 512 columns (8 warps an SM, too few for both pipes: 1173 against 1323 us at
// 311296 x 1000).
#pragma once

#include <cuda_fp16.h>

namespace lsq_apass {

constexpr int DG = 7;              // digits of an entry of p (an element of A has 8)
constexpr int DG_ROWS = 2 * DG + 1;  // rows of the table of p's digits: 7 of zeros, the digits, 1 of zeros
// rows of a CTA from which the 16-row tiles of its 8 warps are even enough (d = 301, FP64 sums against
// digits: at 128 rows 88 and 89 us, at 192 rows 114 and 111, at 256 rows 134 and 120)
constexpr int DG_MIN_ROWS = 192;

// FP64 rows of 65 to 512 columns
template <typename TA, int EPL>
constexpr __host__ __device__ bool digit_pass() {
  return sizeof(TA) == 8 && EPL >= 4 && EPL <= 16;
}

// the tables, in the shared memory of the (not yet used) reduction buffer: 34 dk + 480 bytes of its
// 64 dp, dk = d rounded up to 32
struct DigitTab {
  uint32_t* epk;   // dk: exponent fields of p << 20, the columns of a lane's fragment adjacent
  __half* dig;     // DG_ROWS x pitch: digits of p, in the order of epk
  int pitch;       // halves: 32 or 96 bytes past a multiple of 128, distinct banks for a half-warp's rows
  int lo;          // rows with E <= lo are left to FP64
  uint32_t zeros;  // bit per 32 columns: some meet a zero of p, or lie past d
};

__device__ __forceinline__ DigitTab digit_tab(double* wred, int dk) {
  DigitTab t;
  t.epk = reinterpret_cast<uint32_t*>(wred);
  t.dig = reinterpret_cast<__half*>(t.epk + dk);
  t.pitch = dk + 16;
  t.lo = 0;
  t.zeros = 0;
  return t;
}

// fills the tables from p (all threads); false if p is out of range.  red: 16 ints of scratch.
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
  uint32_t zeros = 0;
  bool sub = false;
  for (int ch = warp; ch < dk / 32; ch += LSQ_WARPS) {
    const int c = 32 * ch + lane;
    const double p = c < d ? vec_s[c] : 0.0;
    const uint32_t hi = (uint32_t)__double2hiint(p);
    const uint32_t ep = (hi >> 20) & 0x7FFu;
    if (__any_sync(0xffffffffu, p == 0.0)) zeros |= 1u << ch;
    sub |= ep == 0 && p != 0.0;
    long long T = (long long)((((unsigned long long)((hi & 0xFFFFFu) | (ep ? 0x100000u : 0u)) << 32) |
                               (uint32_t)__double2loint(p)) << 1);
    if (hi >> 31) T = -T;
    const unsigned long long b = (unsigned long long)T + 0x0080808080808080ull;
    const int pos = (c & ~15) + 4 * (c & 3) + ((c >> 2) & 3);
    t.epk[pos] = ep << 20;
#pragma unroll
    for (int k = 0; k < DG; ++k)
      t.dig[(DG + k) * t.pitch + pos] = __int2half_rn((int)((uint32_t)(b >> (8 * (DG - 1 - k))) & 0xFFu) - 128);
  }
  if (lane == 0) red[LSQ_WARPS + warp] = (int)zeros;
  sub = __syncthreads_or(sub) != 0;
  uint32_t m = 0;
#pragma unroll
  for (int w = 0; w < LSQ_WARPS; ++w) {
    m = max(m, (uint32_t)red[w]);
    t.zeros |= (uint32_t)red[LSQ_WARPS + w];
  }
  __syncthreads();  // red is read before a warp leaves its q there
  const int e = (int)(m >> 20);
  t.lo = max(e + 64, 1250);
  return e >= 1023 - 600 && e <= 1023 + 600 && !sub;
}

constexpr int DG_HI = 2900;  // rows with E >= DG_HI are left to FP64

// |a|, sh bits below the scale, as bytes: digit i in byte 7 - i
__device__ __forceinline__ void digit_bytes(double a, int sh, uint32_t& u0, uint32_t& u1) {
  uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  hi = (hi & 0xFFFFFu) | 0x100000u;
  hi = __funnelshift_l(lo, hi, 9);
  lo <<= 9;
  if (sh >= 32) {
    lo = hi;
    hi = 0;
    sh -= 32;
  }
  u0 = __funnelshift_rc(lo, hi, sh);
  u1 = __funnelshift_rc(hi, 0u, sh);
}

// the signs of two elements, in bits 15 and 31
__device__ __forceinline__ uint32_t sign_pair(double a, double b) {
  return __byte_perm((uint32_t)__double2hiint(a), (uint32_t)__double2hiint(b), 0x7030u) & 0x80008000u;
}

__device__ __forceinline__ void mma_f16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// elements of 32 columns of rows g (pa) and g + 8 (pb); columns from d on repeat column d - 1, against
// zero digits of p
template <bool FULL>
__device__ __forceinline__ void digit_load(double (&x)[8], double (&y)[8], const double* __restrict__ pa,
                                           const double* __restrict__ pb, int c0, int d) {
  const int tq = threadIdx.x & 3;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int c = FULL ? c0 + tq + 4 * i : min(c0 + tq + 4 * i, d - 1);
    x[i] = ld_elem(pa + c);
    y[i] = ld_elem(pb + c);
  }
}

// the contribution of 32 columns to w: of row g in the even lanes, of row g + 8 in the odd ones; false
// if a row's scale is out of range
__device__ __forceinline__ bool digit_chunk(double (&x)[8], double (&y)[8], int c0, const DigitTab& t, double& w) {
  const int lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
  uint32_t ep[8];
  {
    const uint4 q0 = *reinterpret_cast<const uint4*>(t.epk + c0 + 4 * tq);
    const uint4 q1 = *reinterpret_cast<const uint4*>(t.epk + c0 + 16 + 4 * tq);
    ep[0] = q0.x; ep[1] = q0.y; ep[2] = q0.z; ep[3] = q0.w;
    ep[4] = q1.x; ep[5] = q1.y; ep[6] = q1.z; ep[7] = q1.w;
  }
  if ((t.zeros >> (c0 >> 5)) & 1u) {
    // finite elements against a zero of p take no part; infinities and NaNs stay and are seen below
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (ep[i] == 0u) {
        if (((uint32_t)__double2hiint(x[i]) & 0x7FFFFFFFu) < 0x7FF00000u) x[i] = 0.0;
        if (((uint32_t)__double2hiint(y[i]) & 0x7FFFFFFFu) < 0x7FF00000u) y[i] = 0.0;
      }
  }
  uint32_t k0 = 0, k1 = 0, m0 = 0, m1 = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t a = (uint32_t)__double2hiint(x[i]) & 0x7FFFFFFFu, b = (uint32_t)__double2hiint(y[i]) & 0x7FFFFFFFu;
    m0 = max(m0, a);
    m1 = max(m1, b);
    k0 = max(k0, a + ep[i]);
    k1 = max(k1, b + ep[i]);
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
  const uint32_t F0 = ((uint32_t)E0 << 20) | 0xFFFFFu, F1 = ((uint32_t)E1 << 20) | 0xFFFFFu;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int kt = 0; kt < 2; ++kt) {
    uint32_t x0[4], x1[4], y0[4], y1[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * kt + e;
      // E - e(a) - e(p): no borrow from the bits below
      digit_bytes(x[i], (int)((F0 - ((uint32_t)__double2hiint(x[i]) & 0x7FFFFFFFu) - ep[i]) >> 20), x0[e], x1[e]);
      digit_bytes(y[i], (int)((F1 - ((uint32_t)__double2hiint(y[i]) & 0x7FFFFFFFu) - ep[i]) >> 20), y0[e], y1[e]);
    }
    const uint32_t s0 = sign_pair(x[4 * kt], x[4 * kt + 1]), s1 = sign_pair(y[4 * kt], y[4 * kt + 1]);
    const uint32_t s2 = sign_pair(x[4 * kt + 2], x[4 * kt + 3]), s3 = sign_pair(y[4 * kt + 2], y[4 * kt + 3]);
    // two bytes of two elements at a time, then each byte of the two with their signs
    const __half* dp = t.dig + (g + DG) * t.pitch + c0 + 16 * kt + 4 * tq;
#pragma unroll
    for (int h = 0; h < 4; ++h) {  // bytes 2h, 2h + 1
      const uint32_t sel = (h & 1) ? 0x7632u : 0x5410u;
      const uint32_t p0 = h < 2 ? __byte_perm(x0[0], x0[1], sel) : __byte_perm(x1[0], x1[1], sel);
      const uint32_t p1 = h < 2 ? __byte_perm(y0[0], y0[1], sel) : __byte_perm(y1[0], y1[1], sel);
      const uint32_t p2 = h < 2 ? __byte_perm(x0[2], x0[3], sel) : __byte_perm(x1[2], x1[3], sel);
      const uint32_t p3 = h < 2 ? __byte_perm(y0[2], y0[3], sel) : __byte_perm(y1[2], y1[3], sel);
      const int i0 = 7 - 2 * h;  // digit of the even byte
      const uint2 b = *reinterpret_cast<const uint2*>(dp - i0 * t.pitch);
      const uint32_t a[4] = {__byte_perm(p0, s0, 0x7250u), __byte_perm(p1, s1, 0x7250u),
                             __byte_perm(p2, s2, 0x7250u), __byte_perm(p3, s3, 0x7250u)};
      mma_f16_16816(acc, a, b.x, b.y);
      const uint2 b1 = *reinterpret_cast<const uint2*>(dp - (i0 - 1) * t.pitch);
      const uint32_t a1[4] = {__byte_perm(p0, s0, 0x7351u), __byte_perm(p1, s1, 0x7351u),
                              __byte_perm(p2, s2, 0x7351u), __byte_perm(p3, s3, 0x7351u)};
      mma_f16_16816(acc, a1, b1.x, b1.y);
    }
  }
  // sums s = 2 tq, 2 tq + 1 of both rows as one integer each, below 2^32; then the lanes of a pair join
  // theirs, 2^16 apart, the even one for row g, the odd one for row g + 8
  const long long X0 = (long long)__float2int_rn(acc[0] * 16777216.f) * 256 + __float2int_rn(acc[1] * 16777216.f);
  const long long X1 = (long long)__float2int_rn(acc[2] * 16777216.f) * 256 + __float2int_rn(acc[3] * 16777216.f);
  const bool odd = tq & 1;
  const long long got = __shfl_xor_sync(0xffffffffu, odd ? X0 : X1, 1);
  const long long Y = odd ? (got << 16) + X1 : (X0 << 16) + got;
  // 2^52 + 2^51 + Y as bits, less 2^52 + 2^51
  const double f = __longlong_as_double(0x4338000000000000ll + Y) - 6755399441055744.0;
  // Y 256^(12 - 4 (tq / 2) - 2) 2^(E - 2160)
  const int s = 1023 - 2080 - 32 * (tq >> 1);
  const uint32_t mm = odd ? m1 : m0;
  w = fma(f, __hiloint2double(mm == 0 || !ok ? 0 : ((odd ? E1 : E0) + s) << 20, 0), w);
  return ok;
}

// w of 16 rows in FP64 (rows the digits do not take)
static __device__ __noinline__ void tile_dots_f64(const double* __restrict__ A, int64_t ld, int d, int nr, const double* vec_s,
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
template <int NK>
__device__ __forceinline__ void digit_rows(const double* __restrict__ A, int64_t ld, int d, int64_t r0, int64_t r1,
                                           const double* vec_s, const DigitTab& t, double (&acc)[NK], double& q) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2;
#pragma unroll
  for (int k = 0; k < NK; ++k) acc[k] = 0.0;
  q = 0.0;
  for (int64_t i = r0 + 16 * warp; i < r1; i += 16 * LSQ_WARPS) {
    const int nr = (int)min((int64_t)16, r1 - i);
    const double* tile = A + i * ld;
    const double* pa = tile + min(g, nr - 1) * ld;
    const double* pb = tile + min(g + 8, nr - 1) * ld;
    double wl = 0.0;
    bool ok = true;
    double x[8], y[8];
#pragma unroll 1
    for (int c0 = 0; c0 < d; c0 += 32) {
      if (c0 + 32 <= d) digit_load<true>(x, y, pa, pb, c0, d);
      else digit_load<false>(x, y, pa, pb, c0, d);
      ok &= digit_chunk(x, y, c0, t, wl);
    }
    // row g in every even lane of its four, row g + 8 in the odd ones
    wl += __shfl_xor_sync(0xffffffffu, wl, 2);
    if (!__all_sync(0xffffffffu, ok)) {
      double f[2] = {0.0, 0.0};
      tile_dots_f64(tile, ld, d, nr, vec_s, f);
      wl = f[lane & 1];
    }
    if (g + 8 * (lane & 1) < nr) q = fma(wl, wl, q);
#pragma unroll 1
    for (int j = 0; j < 8 && j < nr; ++j) {
      const double wa = __shfl_sync(0xffffffffu, wl, 4 * j), wb = __shfl_sync(0xffffffffu, wl, 4 * j + 1);
      const double* ra = tile + j * ld + lane;
      const double* rb = ra + 8 * ld;
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
  // the two lanes of a row hold the same q: add the rows, and both halves of a lane pair
  q += __shfl_xor_sync(0xffffffffu, q, 1);
#pragma unroll
  for (int o = 4; o <= 16; o <<= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
}

}  // namespace lsq_apass
