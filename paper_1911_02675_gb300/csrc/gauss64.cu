// gauss64.cu -- the Gaussian sketch SA = S A in FP64 (Section 2; the definition of lsq.h: Box-Muller on
// 53-bit uniforms), its dense contraction from exact digit products (digits.cuh) on the tensor cores.
//
// FP64 multiply-adds run at 1.75 a clock an SM and the FP64 logarithm, square root, sine and cosine of a
// pair of entries took ~100 FP64 instructions: 4096 x 64, m = 256, 219 us, where the 0.13 GFLOP and the
// 2 MB of A are nothing.  Here a CTA owns a 64 x 64 tile of SA and a range of rows.  Per 16 rows it draws
// its entries of S (table-driven log, sine and cosine with Taylor polynomials, a Goldschmidt square
// root: ~40 FP64 instructions a pair), writes them as 8 base-256 digits in fixed point (2^-58) to shared
// memory, and multiplies them with the digits of A's columns (columns in fixed point on the scale M of their
// largest element, digits_kernel): 36 digit products, each summed exactly in FP32 over 128 rows, then in
// 64-bit integers.  S stays in shared memory.
//
// An entry of SA differs from its value by about 2^-58 M sqrt(nonzero elements of the column) (digit pairs that
// are dropped, S in fixed point).  FP64 rounds every z a at 2^-53 |z a| and the partial sums of its row splits,
// which is more once the elements of M/8 and above are a 16th of the column's nonzero ones, or as many as
// the splits (2 an SM); and with 16 of them no entry hangs on one small z.  A tile with a column that has
// fewer (a few dominant rows) is summed in FP64, from FP64 Box-Muller entries (direct_tile).
//
// Bound by the FP64 pipe (Box-Muller).  Measured (the sketch's kernels before its last
// reduction): 4096 x 64, m = 256: 219 -> 77 us; m = 512: 381 -> 130 us.  With a dominant row in every column the whole
// sketch takes 227 us (m = 256; 231 without digits, 97 with even columns).
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "digits.cuh"

using namespace lsq_digits;

namespace {

constexpr int NS = 8;                // digits
constexpr int T = 256;               // 8 warps, each 16 sketch rows x 32 columns of the tile
constexpr int BM = 64, BN = 64, KC = 16, FOLD = 128;
constexpr int PITCH = 64 + 8;        // row pitch in shared memory
constexpr int OPER = NS * KC * PITCH;  // one operand's digits of a stage
constexpr size_t SMEM = (size_t)4 * OPER * 2 + 128 * 16 + 64 * 16;

constexpr int GAP = 2;                // exponents below its largest's at which an element of A counts as large

struct Tables {
  double2 lg[128];  // c ~ 1 / m of the interval, 2 ln c
  double2 sc[64];   // sine and cosine at the middle of each 64th of a turn
};

// interval i of the mantissa [1, 2) in 128ths, the upper ones halved, so that the reduced argument lies
// in [0.707, 1.414); c = 1 on both intervals that touch 1, which keeps ln near 1 accurate
__device__ __forceinline__ bool upper(int i) { return i >= 53; }

__device__ void fill_tables(Tables& tb) {
  for (int i = threadIdx.x; i < 128; i += T) {
    const double mid = (1.0 + (i + 0.5) / 128.0) * (upper(i) ? 0.5 : 1.0);
    const double c = i == 0 || i == 127 ? 1.0 : 1.0 / mid;
    tb.lg[i] = make_double2(c, 2.0 * log(c));
  }
  for (int i = threadIdx.x; i < 64; i += T) {
    double s, c;
    sincospi((i + 0.5) / 32.0, &s, &c);
    tb.sc[i] = make_double2(s, c);
  }
}

// the uniform (k + 1/2) 2^-53 of a word pair, evaluated in FP64, as a multiple of 2^-54: from k = 2^52 on,
// k + 1/2 has 54 bits and rounds to the even neighbour (at the top to 1)
__device__ __forceinline__ unsigned long long uniform54(uint32_t hi, uint32_t lo) {
  const unsigned long long k = (((unsigned long long)hi << 32) | lo) >> 11;
  return 2 * k + ((hi >> 31) ? 2 * (k & 1ull) : 1ull);
}

// z(2q, i) and z(2q + 1, i) from the words of Philox(i, q, t, TAG_GAUSS)
__device__ __forceinline__ void normal_pair(const Tables& tb, uint4 w, double& zc, double& zs) {
  const unsigned long long k1 = uniform54(w.x, w.y), k2 = uniform54(w.z, w.w);  // 53 bits at most each
  // -2 ln u1: u1 = m 2^e, m c = 1 + r
  const int lz = __clzll((long long)k1);
  const unsigned long long n1 = k1 << lz;
  const int i1 = (int)(n1 >> 56) & 127;
  const bool up = upper(i1);
  const double m = __longlong_as_double((long long)(((up ? 0x3FEull : 0x3FFull) << 52) | ((n1 >> 11) & 0xFFFFFFFFFFFFFull)));
  const double2 lg = tb.lg[i1];
  const double r = fma(m, lg.x, -1.0);
  double p = fma(r, -2.0 / 7.0, 2.0 / 6.0);
  p = fma(r, p, -2.0 / 5.0);
  p = fma(r, p, 2.0 / 4.0);
  p = fma(r, p, -2.0 / 3.0);
  p = fma(r, p, 1.0);
  p = fma(r * r, p, -2.0 * r);
  const double x = fma((double)(lz - 9 - (up ? 1 : 0)), 2.0 * 0.69314718055994530942, lg.y + p);
  // its square root: two Goldschmidt steps from the hardware's approximation, one correction
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double g = x * y, h = 0.5 * y;
  double e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  h = fma(h, e, h);
  e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  const double rad = lz > 9 ? fma(fma(-g, g, x), h, g) : 0.0;  // (lz = 9: u1 rounded to 1, x = 0)
  // sine and cosine of 2 pi u2 from the middle of its 64th of a turn
  const double2 sc = tb.sc[(int)(k2 >> 48) & 63];  // (u2 rounded to 1 is a whole turn)
  const double a = (__longlong_as_double(0x4330000000000000ll | (long long)(k2 & 0xFFFFFFFFFFFFull)) - (0x1p52 + 0x1p47)) *
                   (6.28318530717958647692 * 0x1p-54);
  const double a2 = a * a;
  double ps = fma(a2, -1.0 / 5040.0, 1.0 / 120.0);
  ps = fma(a2, ps, -1.0 / 6.0);
  const double sa = fma(a * a2, ps, a);
  double pcs = fma(a2, 1.0 / 40320.0, -1.0 / 720.0);
  pcs = fma(a2, pcs, 1.0 / 24.0);
  pcs = fma(a2, pcs, -0.5);
  const double cm = a2 * pcs;
  zs = rad * (sc.x + fma(sc.x, cm, sc.y * sa));
  zc = rad * (sc.y + fma(sc.y, cm, -(sc.x * sa)));
}

// out[j][c] (+)= sum over rows [i_begin, i_end) of z(j, i) A[i][c] for the tile at (j0, c0), in FP64
template <typename TA>
__device__ __noinline__ void direct_tile(const TA* __restrict__ A, int64_t i_begin, int64_t i_end, int d, int64_t ld, int m,
                                         uint64_t seed, uint32_t t, int64_t grow0, int j0, int c0, void* smem,
                                         int accumulate, double* __restrict__ out) {
  double (*Ss)[BM] = reinterpret_cast<double (*)[BM]>(smem);
  double (*As)[BN] = reinterpret_cast<double (*)[BN]>(Ss + KC);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4] = {};
  for (int64_t i0 = i_begin; i0 < i_end; i0 += KC) {
    __syncthreads();  // the rows before are no longer read
    for (int e = threadIdx.x; e < KC * BM / 2; e += T) {
      const int jp = e / KC, k = e % KC;
      double zc = 0.0, zs = 0.0;
      if (i0 + k < i_end) {
        const uint4 w = philox_at(seed, (uint32_t)(i0 + k + grow0), (uint32_t)((j0 >> 1) + jp), t, TAG_GAUSS);
        const double rad = sqrt(-2.0 * log((double)uniform54(w.x, w.y) * 0x1p-54));
        double sn, cs;
        sincospi((double)uniform54(w.z, w.w) * 0x1p-53, &sn, &cs);
        zc = rad * cs;
        zs = rad * sn;
      }
      Ss[k][2 * jp] = zc;
      Ss[k][2 * jp + 1] = zs;
    }
    for (int e = threadIdx.x; e < KC * BN; e += T) {
      const int k = e / BN, c = e % BN;
      As[k][c] = i0 + k < i_end && c0 + c < d ? (double)__ldg(A + (i0 + k) * ld + c0 + c) : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < KC; ++k) {
      double s[4], a[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) s[r] = Ss[k][ty + 16 * r];
#pragma unroll
      for (int c = 0; c < 4; ++c) a[c] = As[k][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fma(s[r], a[c], acc[r][c]);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = j0 + ty + 16 * r, col = c0 + tx + 16 * c;
      if (j < m && col < d) {
        double* o = out + (int64_t)j * d + col;
        *o = accumulate ? *o + acc[r][c] : acc[r][c];
      }
    }
}

// part[split][j][c] (+)= sum over the split's rows of the panel of z(j, i) A[i][c]; planes: the digits of
// the panel's rows (from row i0 of A, `rows` a multiple of KC), with their counts (digits_kernel)
template <typename TA>
__global__ void __launch_bounds__(T, 1) gauss64_kernel(const uint16_t* __restrict__ planes, int rows, int dq,
                                                       const TA* __restrict__ A, int64_t n, int d, int64_t ld, int m,
                                                       uint64_t seed, uint32_t t, int64_t i0, int64_t grow0,
                                                       int rows_per_split, const uint32_t* __restrict__ mag,
                                                       const uint32_t* __restrict__ counts, uint32_t enough,
                                                       int accumulate, double* __restrict__ part) {
  extern __shared__ __align__(16) uint16_t sm[];  // [2] digits of S, [2] digits of A, tables
  Tables& tb = *reinterpret_cast<Tables*>(sm + 4 * OPER);
  const int j0 = blockIdx.x * BM, c0 = blockIdx.y * BN;
  const int k0 = blockIdx.z * rows_per_split, k1 = min(rows, k0 + rows_per_split);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wa = (warp & 3) * 16, wb = (warp >> 2) * 32;
  const int64_t plane = (int64_t)rows * dq;
  double* out = part + (int64_t)blockIdx.z * m * d;
  auto load = [&](int k, int st) {
    uint16_t* dst = sm + (2 + st) * OPER;
    for (int e = tid; e < NS * KC * BN / 8; e += T) {
      const int row = e / (BN / 8), p = e % (BN / 8), i = row / KC, r = row % KC;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                       (unsigned)__cvta_generic_to_shared(dst + row * PITCH + 8 * p)),
                   "l"(planes + i * plane + (int64_t)(k + r) * dq + c0 + 8 * p)
                   : "memory");
    }
  };
  // 16 rows of S: row k + (tid mod 16), pairs tid / 16 and tid / 16 + 16
  auto draw = [&](int k, int st) {
    uint32_t* dst = reinterpret_cast<uint32_t*>(sm + st * OPER);
    const int r = tid & 15;
    const int64_t i = i0 + k + r;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = (tid >> 4) + 16 * h;
      unsigned long long uc = BIAS, us = BIAS;
      if (k + r < k1 && i < n) {
        double zc, zs;
        normal_pair(tb, philox_at(seed, (uint32_t)(i + grow0), (uint32_t)((j0 >> 1) + q), t, TAG_GAUSS), zc, zs);
        uc = biased_digits(zc, 1026);  // 2^-58 units (|z| < 16)
        us = biased_digits(zs, 1026);
      }
#pragma unroll
      for (int x = 0; x < NS; ++x) dst[(x * KC + r) * (PITCH / 2) + q] = digit_pair(uc, us, x);
    }
  };
  float acc[NS][4][4];
  long long hi[4][4], lo[4][4];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      hi[c][x] = lo[c][x] = 0;
#pragma unroll
      for (int w = 0; w < NS; ++w) acc[w][c][x] = 0.f;
    }
  auto fold = [&]() {
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        long long h = 0, l = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) h = h * 256 + __float2int_rn(acc[w][c][x]);
#pragma unroll
        for (int w = 4; w < 8; ++w) l = l * 256 + __float2int_rn(acc[w][c][x]);
        hi[c][x] += h;
        lo[c][x] += l;
#pragma unroll
        for (int w = 0; w < NS; ++w) acc[w][c][x] = 0.f;
      }
  };
  const int lr = (lane & 7) + ((lane >> 4) & 1) * 8, lc = ((lane >> 3) & 1) * 8;
  const int br = (lane & 7) + ((lane >> 3) & 1) * 8, bc = ((lane >> 4) & 1) * 8;
  fill_tables(tb);
  if (k0 < k1) load(k0, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  // (columns of zeros are exact either way; those with infinities or NaNs are seen at the end)
  bool few = false;
  if (tid < BN && c0 + tid < d) {
    const uint32_t mg = mag[c0 + tid];
    few = mg != 0u && mg < 0x7FF00000u && counts[c0 + tid] < max(16u, min(counts[d + c0 + tid] / 16u, enough));
  }
  if (__syncthreads_or(few)) {  // (the tables are there, too)
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // (direct_tile starts with a barrier)
    direct_tile(A, i0 + k0, min(n, i0 + k1), d, ld, m, seed, t, grow0, j0, c0, sm, accumulate, out);
    return;
  }
  if (k0 < k1) draw(k0, 0);
  int since = 0;
  for (int k = k0, st = 0; k < k1; k += KC, st ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // this stage is complete, and the other one no longer read
    if (k + KC < k1) load(k + KC, st ^ 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint16_t* As = sm + st * OPER + lr * PITCH + wa + lc;
    const uint16_t* Bs = sm + (2 + st) * OPER + br * PITCH + wb + bc;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      uint32_t b0[4], b1[4];
      ldsm4t(b0, Bs + j * KC * PITCH);
      ldsm4t(b1, Bs + j * KC * PITCH + 16);
#pragma unroll
      for (int i = 0; i < NS; ++i)
        if (i + j < NS) {
          uint32_t a[4];
          ldsm4t(a, As + i * KC * PITCH);
          mma_bf16_16816(acc[i + j][0], a, b0[0], b0[1]);
          mma_bf16_16816(acc[i + j][1], a, b0[2], b0[3]);
          mma_bf16_16816(acc[i + j][2], a, b1[0], b1[1]);
          mma_bf16_16816(acc[i + j][3], a, b1[2], b1[3]);
        }
    }
    if (k + KC < k1) draw(k + KC, st ^ 1);
    since += KC;
    if (since == FOLD) {
      fold();
      since = 0;
    }
  }
  fold();
  // (hi 2^32 + lo) 2^56 2^-58 2^(emax - 1084); a column with infinities or NaNs: what its non-finite
  // elements give in floating point
  const int g = lane >> 2, tq = lane & 3;
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int j = j0 + wa + g + (x >> 1) * 8, col = c0 + wb + c * 8 + 2 * tq + (x & 1);
      if (j < m && col < d) {
        const int e = (int)(mag[col] >> 20);
        // (two factors: e - 1086 alone lies below the smallest power for columns under 2^-1011)
        double v = fma((double)hi[c][x], 4294967296.0, (double)lo[c][x]) * 0x1p-58 * pow2(max(e, 1) - 1028);
        if (e == 0x7FF) {
          v = 0.0;
          for (int k = k0; k < k1 && i0 + k < n; ++k) {
            const double xa = (double)A[(i0 + k) * ld + col];
            if (isfinite(xa)) continue;
            double zc, zs;
            normal_pair(tb, philox_at(seed, (uint32_t)(i0 + k + grow0), (uint32_t)(j >> 1), t, TAG_GAUSS), zc, zs);
            v = fma((j & 1) ? zs : zc, xa, v);
          }
        }
        double* o = out + (int64_t)j * d + col;
        *o = accumulate ? *o + v : v;
      }
    }
}

constexpr int64_t PANEL_BYTES = (int64_t)256 << 20;  // digit planes of a panel of rows at most

template <typename TA>
lsq_status run(lsq_ctx* ctx, const lsq_matrix* A, int m, uint64_t seed, uint32_t t, int64_t grow0, LsqGauss64* out) {
  const TA* data = static_cast<const TA*>(A->data);
  const int d = (int)A->d, dq = (d + BN - 1) / BN * BN;
  const int64_t n = A->n;
  const int64_t cap = PANEL_BYTES / ((int64_t)NS * dq * 2) / FOLD * FOLD;
  const int64_t panel = std::min<int64_t>((n + KC - 1) / KC * KC, std::max<int64_t>(FOLD, cap));
  const int gx = lsq_ceil_div(m, BM), gy = dq / BN;
  // whole waves of one CTA per SM; a CTA's start (tables, first stage) costs about a stage of rows
  const int64_t stages = panel / KC;
  const int64_t pcap = std::max<int64_t>(1, ((int64_t)256 << 20) / ((int64_t)m * d * 8));
  int64_t splits = 1;
  double best = 1e300;
  for (int64_t s = 1; s <= std::min<int64_t>(std::min(stages, pcap), 1024); ++s) {
    const double cost = (double)((gx * gy * s + ctx->sm_count - 1) / ctx->sm_count) * ((double)((stages + s - 1) / s) + 1.0);
    if (cost < best * (1.0 - 1e-9)) {
      best = cost;
      splits = s;
    }
  }
  const int rows_per_split = (int)((stages + splits - 1) / splits) * KC;
  splits = (panel + rows_per_split - 1) / rows_per_split;
  // the columns' largest magnitudes, then the two counts of every panel
  const int64_t mag_words = d * (1 + 2 * ((n + panel - 1) / panel));
  const size_t need = lsq_align256((size_t)splits * m * d * 8) + lsq_align256((size_t)NS * panel * dq * 2) +
                      lsq_align256((size_t)mag_words * 4);
  lsq_status st = lsq_ensure_scratch(ctx, need);
  if (st != LSQ_OK) return st;
  Carver cv{reinterpret_cast<char*>(ctx->scratch), 0};
  double* part = cv.take<double>((size_t)splits * m * d);
  uint32_t* planes = cv.take<uint32_t>((size_t)NS * panel * dq / 2);
  uint32_t* mag = cv.take<uint32_t>(mag_words);
  cudaStream_t s = ctx->stream;
  LSQ_CUDA_TRY(cudaMemsetAsync(mag, 0, (size_t)mag_words * 4, s));
  const int cb = (d + 31) / 32;
  const int rb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 7) / 8, (4 * ctx->sm_count + cb - 1) / cb));
  column_max_kernel<TA><<<dim3((unsigned)cb, (unsigned)rb), 256, 0, s>>>(data, n, d, A->ld, mag);
  LSQ_LAUNCH_CHECK();
  LSQ_CUDA_TRY(cudaFuncSetAttribute(gauss64_kernel<TA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM));
  uint32_t* counts = mag + d;
  for (int64_t i0 = 0; i0 < n; i0 += panel, counts += 2 * d) {
    const int rows = (int)std::min<int64_t>(panel, (n - i0 + KC - 1) / KC * KC);
    digits_kernel<TA, NS, true>
        <<<lsq_digits_grid(dq, rows, ctx->sm_count), 256, 0, s>>>(data, n, d, A->ld, dq, i0, rows, mag, GAP, counts, planes);
    LSQ_LAUNCH_CHECK();
    gauss64_kernel<TA><<<dim3((unsigned)gx, (unsigned)gy, (unsigned)splits), T, SMEM, s>>>(
        reinterpret_cast<const uint16_t*>(planes), rows, dq, data, n, d, A->ld, m, seed, t, i0, grow0, rows_per_split, mag,
        counts, 2u * ctx->sm_count, i0 > 0 ? 1 : 0, part);
    LSQ_LAUNCH_CHECK();
  }
  out->part = part;
  out->splits = (int)splits;
  return LSQ_OK;
}

}  // namespace

// the partial sums [splits][m][d] of sqrt(m) SA, in the context's scratch
lsq_status lsq_gauss64_run(lsq_ctx* ctx, const lsq_matrix* A, int m, uint64_t seed, uint32_t t, int64_t grow0,
                           LsqGauss64* out) {
  return A->dtype == LSQ_F64 ? run<double>(ctx, A, m, seed, t, grow0, out) : run<float>(ctx, A, m, seed, t, grow0, out);
}
