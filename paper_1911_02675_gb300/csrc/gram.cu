// gram.cu -- the Gram matrix H_S = (SA)^T (SA) of a sketch (Section 1, PCG paragraph) on the tensor
// cores, from exact products of 8-bit digits.
//
// The FP64 pipe does 1.75 multiply-adds a clock an SM, warp-level BF16 MMAs 1024.  Each column of SA is
// written in fixed point on the scale of its largest element, as NS balanced base-256 digits
// (|D| <= 128, exact in BF16):  SA[r][a] = sum_i D_i[r][a] 256^(7-i) 2^(e_a - 1084),  63 bits below the
// largest element at NS = 8.  A product of two digits is at most 2^14, so the FP32 accumulators hold
// the sum over 128 rows of every pair with the same i + j exactly (8 pairs x 128 x 2^14 = 2^24); pairs
// with i + j >= NS are dropped.  The sums are folded into 64-bit integers every 128 rows, and one FP64
// rounding per element follows.
//
// What is dropped is on the scale of the columns' largest elements, M_a M_b: about 2^-62 M_a M_b sqrt(m)
// at NS = 8 and 2^-54 at 7 (rms over random digits).  FP64 multiply-adds round at 2^-54 of the partial
// sums, which is more as long as the products themselves are not far below M_a M_b.  So a column takes
// digits only if more than 5/8 of its elements lie within 2^5 of its largest: two such columns share at
// least a quarter of their rows, their products there are 2^-10 M_a M_b or more, and over 64 rows and
// more the FP64 sums' own error is no smaller (double-FP32, LSQ_PREC_MIXED: the 45 bits of its
// elements).  A tile with any other column (a few dominant rows, mostly zeros) is summed with FP64 or
// double-FP32 multiply-adds as the precision asks (direct_tile).  The sketch of a matrix of many rows has
// columns near N(0, s): 80% of their elements lie within the 2^5 at 4 s.
//
// Bound by the MMAs, NS (NS + 1) / 2 for each 16 x 8 x 16 product, and the latency of a stage.  Measured
// (maximum, digits and product; before: FP64 or double-FP32 multiply-adds in tiles of 64 x 64):
// 4096 x 1024 mixed 1100 -> 568 us, 1204 x 301 FP64 169 -> 49 us, 256 x 64 FP64 75 -> 19 us; the counts cost
// 2 us a Gram.
#include <algorithm>

#include "apass.cuh"
#include "common.cuh"
#include "digits.cuh"

using namespace lsq_digits;

namespace {

constexpr int GT = 256;                 // threads of the product kernel: 8 warps of 16 x 16 outputs
constexpr int BA = 64, BB = 32;         // its tile of H_S
constexpr int KC = 32;                  // rows of SA per stage (of 16: 3% slower at 4096 x 1024)
constexpr int FOLD = 128;               // rows between folds
constexpr int PA = BA + 8, PB = BB + 8;  // row pitches in shared memory (16-byte pieces of 8 rows: distinct banks)

constexpr int GAP = 4;                   // exponents below its largest element's at which an element counts as large
constexpr int TK = 16;                   // rows of SA per step of direct_tile

// exponent field of column c's largest element, 1 for zeros and subnormals
__device__ __forceinline__ int column_exp(const uint32_t* mag, int c) { return max((int)(mag[c] >> 20), 1); }

// 2^k as the scale of column c: NaN where the column is not finite, 0 past the last column
__device__ __forceinline__ double column_scale(const uint32_t* mag, int c, int d, int k) {
  if (c >= d) return 0.0;
  return column_exp(mag, c) == 0x7FF ? __longlong_as_double(0x7FF8000000000000ll) : pow2(k);
}

// what brings a column whose largest element lies outside 2^-20 .. 2^50 into the range of FP32 products
__device__ __forceinline__ int df_shift(const uint32_t* mag, int c, int d) {
  const int e = c < d ? column_exp(mag, c) : 1023;
  return e > 1073 ? 1073 - e : e < 1003 ? 1023 - e : 0;
}

// out (+)= the sum over rows [r0, r1) of SA for the tile at (a0, b0), by multiply-adds: FP64, or DF:
// double-FP32 (elements split into a 21-bit head and the FP32 rounding of the rest, exact products, sums
// as (head, tail) pairs).  Thread (ty, tx) owns rows
// ty + 16 i and columns tx + 16 j of the tile.
template <bool DF>
__device__ __noinline__ void direct_tile(const double* __restrict__ SA, int d, int dp, int r0, int r1, int a0, int b0,
                                         const uint32_t* __restrict__ mag, void* smem, int accumulate,
                                         double* __restrict__ out) {
  using E = typename std::conditional<DF, float2, double>::type;
  E (*Xa)[BA] = reinterpret_cast<E (*)[BA]>(smem);
  E (*Xb)[BB] = reinterpret_cast<E (*)[BB]>(Xa + TK);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][2] = {};
  float ah[4][2] = {}, al[4][2] = {};
  for (int k0 = r0; k0 < r1; k0 += TK) {
    __syncthreads();  // the rows before are no longer read
    for (int e = threadIdx.x; e < TK * (BA + BB); e += GT) {
      const int k = e / (BA + BB), p = e - k * (BA + BB);
      const int c = p < BA ? a0 + p : b0 + p - BA;
      const double v = k0 + k < r1 && c < d ? SA[(int64_t)(k0 + k) * d + c] : 0.0;
      E* o = p < BA ? &Xa[k][p] : &Xb[k][p - BA];
      if constexpr (DF) {
        // (by the exponent fields; what leaves the range, or is subnormal, is zero)
        const uint32_t hi = (uint32_t)__double2hiint(v);
        const int ec = (int)((hi >> 20) & 0x7FFu), es = ec + df_shift(mag, c, d);
        const double u = __hiloint2double((int)((hi & 0x800FFFFFu) | ((uint32_t)es << 20)), __double2loint(v));
        lsq_apass::split_df(ec > 0 && es > 0 ? u : 0.0, o->x, o->y);
      } else {
        *o = v;
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < TK; ++k) {
      E x[4], y[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = Xa[k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 2; ++j) y[j] = Xb[k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if constexpr (DF) lsq_apass::df_fma(x[i].x, x[i].y, y[j].x, y[j].y, ah[i][j], al[i][j]);
          else acc[i][j] = fma(x[i], y[j], acc[i][j]);
        }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int a = a0 + ty + 16 * i, b = b0 + tx + 16 * j;
      if (a < dp && b < dp) {
        double v = acc[i][j];
        if constexpr (DF)
          v = ((double)ah[i][j] + (double)al[i][j]) * column_scale(mag, a, d, -df_shift(mag, a, d)) *
              column_scale(mag, b, d, -df_shift(mag, b, d));
        double* o = out + (int64_t)a * dp + b;
        *o = accumulate ? *o + v : v;
      }
    }
}

// whether a column of the tile at (a0, b0) is left to direct_tile, given the digit kernel's counts over
// `live` rows (columns of zeros are exact either way, those with infinities or NaNs end as NaN); each
// thread looks at one column
__device__ __forceinline__ bool uneven_column(const uint32_t* mag, const uint32_t* large, int live, int a0, int b0,
                                              int d) {
  const int tid = threadIdx.x, c = tid < BA ? a0 + tid : b0 + tid - BA;
  if (tid >= BA + BB || c >= d) return false;
  const uint32_t m = mag[c];
  return m != 0u && m < 0x7FF00000u && 8ull * large[c] <= 5ull * (unsigned)live;
}

// the tiles that gram_mma_kernel leaves to it, on the same grid: at three CTAs an SM, where the product
// kernel's registers allow one
template <bool DF>
__global__ void __launch_bounds__(GT, 3) gram_direct_kernel(int rows, int dp, int rows_per_split,
                                                            const int2* __restrict__ tiles,
                                                            const uint32_t* __restrict__ mag,
                                                            const uint32_t* __restrict__ large,
                                                            const double* __restrict__ SA, int row0, int live, int d,
                                                            int accumulate, double* __restrict__ part) {
  __shared__ __align__(16) double sm[TK * (BA + BB)];
  const int2 tl = tiles[blockIdx.x];
  const int a0 = tl.x * BA, b0 = tl.y * BB;
  if (!__syncthreads_or(uneven_column(mag, large, live, a0, b0, d))) return;
  const int k0 = blockIdx.y * rows_per_split, k1 = min(rows, k0 + rows_per_split);
  direct_tile<DF>(SA, d, dp, row0 + min(k0, live), row0 + min(k1, live), a0, b0, mag, sm, accumulate,
                  part + (int64_t)blockIdx.y * dp * dp);
}

// part[split][a][b] (+)= the sum over the split's rows of the panel, for one tile of H_S that meets its
// upper triangle; planes as digits_kernel writes them for the panel's `rows` (a multiple of KC, `live` of
// them in SA, the first one row row0), with its counts `large`.  direct: tiles with an uneven column are
// summed here, too, else left to gram_direct_kernel.
template <int NS>
__global__ void __launch_bounds__(GT, 1) gram_mma_kernel(const uint16_t* __restrict__ planes, int rows, int dq, int dp,
                                                         int rows_per_split, const int2* __restrict__ tiles,
                                                         const uint32_t* __restrict__ mag,
                                                         const uint32_t* __restrict__ large,
                                                         const double* __restrict__ SA, int row0, int live, int d,
                                                         int accumulate, int direct, double* __restrict__ part) {
  extern __shared__ __align__(16) uint16_t sm[];  // two stages of [NS][KC][PA] and [NS][KC][PB]
  constexpr int SA_E = NS * KC * PA, SB_E = NS * KC * PB, ST = SA_E + SB_E;
  const int2 tl = tiles[blockIdx.x];
  const int a0 = tl.x * BA, b0 = tl.y * BB;
  const int k0 = blockIdx.y * rows_per_split, k1 = min(rows, k0 + rows_per_split);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wa = (warp & 3) * 16, wb = (warp >> 2) * 16;
  const int64_t plane = (int64_t)rows * dq;
  double* out = part + (int64_t)blockIdx.y * dp * dp;
  auto load = [&](int k, int st) {
    uint16_t* dst = sm + st * ST;
    for (int e = tid; e < NS * KC * (BA + BB) / 8; e += GT) {
      const int row = e / ((BA + BB) / 8), p = e - row * ((BA + BB) / 8);
      const int i = row / KC, r = row - i * KC;
      const bool isa = p < BA / 8;
      const uint16_t* src = planes + i * plane + (int64_t)(k + r) * dq + (isa ? a0 + 8 * p : b0 + 8 * (p - BA / 8));
      uint16_t* o = isa ? dst + row * PA + 8 * p : dst + SA_E + row * PB + 8 * (p - BA / 8);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(o)), "l"(src)
                   : "memory");
    }
  };
  float acc[NS][2][4];
  long long hi[2][4], lo[2][4];
#pragma unroll
  for (int w = 0; w < NS; ++w)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[w][n][x] = 0.f;
#pragma unroll
  for (int n = 0; n < 2; ++n)
#pragma unroll
    for (int x = 0; x < 4; ++x) hi[n][x] = lo[n][x] = 0;
  // hi: sums of i + j <= 3 on the scale of 3, lo: of 4 .. 7 on the scale of 7
  auto fold = [&]() {
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        long long h = 0, l = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) h = h * 256 + __float2int_rn(acc[w][n][x]);
#pragma unroll
        for (int w = 4; w < 8; ++w) l = l * 256 + (w < NS ? __float2int_rn(acc[w < NS ? w : 0][n][x]) : 0);
        hi[n][x] += h;
        lo[n][x] += l;
#pragma unroll
        for (int w = 0; w < NS; ++w) acc[w][n][x] = 0.f;
      }
  };
  // ldmatrix rows of this lane: A tile (16 columns of H_S's row range as M, 16 rows of SA as K), both
  // stored [k][column] and read transposed
  const int lr = (lane & 7) + ((lane >> 4) & 1) * 8, lc = ((lane >> 3) & 1) * 8;    // A: matrices (m, k) 00 10 01 11
  const int br = (lane & 7) + ((lane >> 3) & 1) * 8, bc = ((lane >> 4) & 1) * 8;    // B: (k, n) 00 10 01 11
  if (k0 < k1) load(k0, 0);  // (a short last panel leaves splits empty)
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (__syncthreads_or(uneven_column(mag, large, live, a0, b0, d))) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // (direct_tile starts with a barrier)
    if (direct) direct_tile<NS < 8>(SA, d, dp, row0 + min(k0, live), row0 + min(k1, live), a0, b0, mag, sm, accumulate,
                        out);
    return;
  }
  int since = 0;
  for (int k = k0, st = 0; k < k1; k += KC, st ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (k + KC < k1) load(k + KC, st ^ 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
    for (int ks = 0; ks < KC; ks += 16) {
      const uint16_t* As = sm + st * ST + (ks + lr) * PA + wa + lc;
      const uint16_t* Bs = sm + st * ST + SA_E + (ks + br) * PB + wb + bc;
      uint32_t b[NS][4];
#pragma unroll
      for (int j = 0; j < NS; ++j) ldsm4t(b[j], Bs + j * KC * PB);
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        uint32_t a[4];
        ldsm4t(a, As + i * KC * PA);
#pragma unroll
        for (int j = 0; j < NS; ++j)
          if (i + j < NS) {
            mma_bf16_16816(acc[i + j][0], a, b[j][0], b[j][1]);
            mma_bf16_16816(acc[i + j][1], a, b[j][2], b[j][3]);
          }
      }
    }
    since += KC;
    if (since == FOLD) {
      fold();
      since = 0;
    }
  }
  fold();
  // H_S[a][b] = (hi 2^32 + lo) 2^56 2^(e_a - 1084) 2^(e_b - 1084), NaN where a column is not finite
  const int g = lane >> 2, t = lane & 3;
  auto scale = [&](int c) { return column_scale(mag, c, d, c < d ? column_exp(mag, c) - 1084 + 28 : 0); };
#pragma unroll
  for (int n = 0; n < 2; ++n)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int a = a0 + wa + g + (x >> 1) * 8, bcol = b0 + wb + n * 8 + 2 * t + (x & 1);
      if (a < dp && bcol < dp) {
        const double v = fma((double)hi[n][x], 4294967296.0, (double)lo[n][x]) * scale(a) * scale(bcol);
        double* o = out + (int64_t)a * dp + bcol;
        *o = accumulate ? *o + v : v;
      }
    }
}

template <int NS>
lsq_status run(lsq_ctx* ctx, const double* SA, int m, int d, int dp, int dq, int panel, int splits, int rows_per_split,
               const int2* d_tiles, int ntiles, uint32_t* mag, uint32_t* planes, double* part) {
  cudaStream_t s = ctx->stream;
  uint32_t* large = mag + d;  // of each panel
  // a launch for the uneven tiles, most often empty, is worth its 2 us where tiles are many (factor of 4096 x
  // 1024 with all columns uneven, in the product kernel and in one of their own: FP64 6.69 and 6.00 ms, mixed
  // 3.77 and 3.21; 6.23 and 3.19 without digits)
  const bool direct = dp <= 256;
  constexpr size_t smem = (size_t)2 * (NS * KC * PA + NS * KC * PB) * 2;
  LSQ_CUDA_TRY(cudaFuncSetAttribute(gram_mma_kernel<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  for (int r0 = 0; r0 < m; r0 += panel) {
    const int rows = std::min(panel, (m - r0 + KC - 1) / KC * KC);
    const dim3 grid = lsq_digits_grid(dq, rows, ctx->sm_count);
    digits_kernel<double, NS, false><<<grid, 256, 0, s>>>(SA, m, d, d, dq, r0, rows, mag, GAP, large, planes);
    LSQ_LAUNCH_CHECK();
    gram_mma_kernel<NS><<<dim3((unsigned)ntiles, (unsigned)splits), GT, smem, s>>>(
        reinterpret_cast<const uint16_t*>(planes), rows, dq, dp, rows_per_split, d_tiles, mag, large, SA, r0,
        std::min(rows, m - r0), d, r0 > 0 ? 1 : 0, direct ? 1 : 0, part);
    LSQ_LAUNCH_CHECK();
    if (!direct) {
      gram_direct_kernel<NS < 8><<<dim3((unsigned)ntiles, (unsigned)splits), GT, 0, s>>>(
          rows, dp, rows_per_split, d_tiles, mag, large, SA, r0, std::min(rows, m - r0), d, r0 > 0 ? 1 : 0, part);
      LSQ_LAUNCH_CHECK();
    }
    large += d;
  }
  return LSQ_OK;
}

constexpr int64_t PANEL_BYTES = (int64_t)256 << 20;  // digit planes of a panel of rows at most

}  // namespace

LsqGramPlan lsq_gram_plan(const lsq_ctx* ctx, int m, int d, bool mixed) {
  LsqGramPlan p;
  p.dp = (d + 31) / 32 * 32;
  p.dq = (d + BA - 1) / BA * BA;
  for (int a = 0; a * BA < p.dp; ++a)
    for (int b = 0; b * BB < p.dp; ++b)
      if (b * BB + BB > a * BA) p.tiles.push_back(make_int2(a, b));
  p.ns = mixed ? 7 : 8;
  // panels of whole folds; the splits of a panel in whole stages, at least 64 rows, about two CTAs an SM
  const int64_t cap = PANEL_BYTES / ((int64_t)p.ns * p.dq * 2) / FOLD * FOLD;
  const int mk = (m + KC - 1) / KC * KC;
  p.panel = (int)std::min<int64_t>(mk, std::max<int64_t>(FOLD, cap));
  int splits = std::max(1, (2 * ctx->sm_count + (int)p.tiles.size() - 1) / (int)p.tiles.size());
  splits = std::min(splits, std::max(1, p.panel / 64));
  p.rows_per_split = ((p.panel + splits - 1) / splits + KC - 1) / KC * KC;
  p.splits = (p.panel + p.rows_per_split - 1) / p.rows_per_split;
  p.plane_bytes = (size_t)p.ns * p.panel * p.dq * 2;
  p.mag_words = (size_t)d * (1 + (m + p.panel - 1) / p.panel);
  return p;
}

lsq_status lsq_gram_run(lsq_ctx* ctx, const LsqGramPlan& p, const double* SA, int m, int d, const int2* d_tiles,
                        uint32_t* mag, uint32_t* planes, double* part) {
  const int cb = (d + 31) / 32;
  const int rb = std::max(1, std::min((m + 7) / 8, (4 * ctx->sm_count + cb - 1) / cb));
  column_max_kernel<double><<<dim3((unsigned)cb, (unsigned)rb), 256, 0, ctx->stream>>>(SA, m, d, d, mag);
  LSQ_LAUNCH_CHECK();
  const int nt = (int)p.tiles.size();
  return p.ns == 8 ? run<8>(ctx, SA, m, d, p.dp, p.dq, p.panel, p.splits, p.rows_per_split, d_tiles, nt, mag, planes, part)
                   : run<7>(ctx, SA, m, d, p.dp, p.dq, p.panel, p.splits, p.rows_per_split, d_tiles, nt, mag, planes, part);
}
