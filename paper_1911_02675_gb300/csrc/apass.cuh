// apass.cuh -- the fused pass over A (v = A^T (A p), q = ||A p||^2, one read of each row)
// shared by the solver and the standalone pass entry points.  Internal, not part of the ABI.
#pragma once

#include "common.cuh"

namespace lsq_apass {

// an element of A as FP64.  FP32 elements are widened with integer operations (the conversion
// instruction runs on the FP64 pipe, which bounds the pass); the conversion is left to
// subnormals, infinities and NaNs.
__device__ __forceinline__ double ld_elem(const double* p) { return __ldg(p); }
__device__ __forceinline__ double ld_elem(const float* p) {
  const float x = __ldg(p);
  const uint32_t u = __float_as_uint(x), m = u & 0x7FFFFFFFu;
  if (m - 0x00800000u < 0x7F000000u || m == 0u) {
    const uint32_t hi = (u & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u);
    return __hiloint2double((int)hi, (int)(u << 29));
  }
  return (double)x;
}

// ------------------------------------------------------------------------------------
// Fused pass over the rows [r0, r1): per-warp accumulators of v = A^T (A p) in
// registers (lane owns columns lane + 32 k), q = sum (a_i . p)^2; then a fixed-order
// CTA reduction into part[c * P + cta].
//
// The FP64 pipe bounds it: an FP64 warp instruction holds a sub-partition for ~64 cycles, so
// what counts is their number, 2 per 32 elements at best.  A warp therefore computes only the
// NK = ceil(d / 32) column groups that exist (not the power of two the layout pads to), and
// takes R rows at a time: their R dot products are summed over the lanes together (each
// exchange halves the rows a lane still sums, R - 1 + 5 - log2 R additions instead of 5 R), and
// q takes one FMA for the R rows.  Loads need no prefetch: the other warps' FP64 work covers
// them.  Measured, pass over 600011 x 333 FP64 (1.6 GB): 1220 us with padded groups and a sum
// per row, 859 us now (0.79 ms is the FP64 pipe's time for the 4 n d flops).
// ------------------------------------------------------------------------------------
template <typename TA, int NK, int R>
__device__ __forceinline__ void fused_rows(const TA* __restrict__ A, int64_t ld, int d, int64_t r0, int64_t r1,
                                           const double* vec_s, double (&acc)[NK], double& q) {
  static_assert(R == 2 || R == 4, "rows per step");
  constexpr bool PV_REG = NK <= 8;  // keep p in registers while they are plentiful
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0;
  double pv[PV_REG ? NK : 1];
  if (PV_REG) {
#pragma unroll
    for (int k = 0; k < NK; ++k) pv[PV_REG ? k : 0] = lane + 32 * k < d ? vec_s[lane + 32 * k] : 0.0;
  }
#pragma unroll
  for (int k = 0; k < NK; ++k) acc[k] = 0.0;
  q = 0.0;
  for (int64_t i = r0 + (int64_t)R * warp; i < r1; i += (int64_t)R * LSQ_WARPS) {
    const int nr = (int)min((int64_t)R, r1 - i);  // rows of this step (fewer at the end)
    double a[R][NK], w[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const TA* src = A + (i + r) * ld + lane;
      if (r < nr) {
#pragma unroll
        for (int k = 0; k < NK; ++k) a[r][k] = (k < NK - 2 || lane + 32 * k < d) ? ld_elem(src + 32 * k) : 0.0;  // d > 32 (NK - 2)
      } else {
#pragma unroll
        for (int k = 0; k < NK; ++k) a[r][k] = 0.0;
      }
      w[r] = 0.0;
    }
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const double pk = PV_REG ? pv[PV_REG ? k : 0] : vec_s[lane + 32 * k];
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r < nr) w[r] = fma(a[r][k], pk, w[r]);
    }
    // lanes with bit 4 (and bit 3) set keep the upper half of the rows they still sum
    double s;
    if constexpr (R == 4) {
      const double u0 = __shfl_xor_sync(0xffffffffu, b4 ? w[0] : w[R - 2], 16);
      const double u1 = __shfl_xor_sync(0xffffffffu, b4 ? w[1] : w[R - 1], 16);
      const double k0 = (b4 ? w[R - 2] : w[0]) + u0, k1 = (b4 ? w[R - 1] : w[1]) + u1;
      const double u2 = __shfl_xor_sync(0xffffffffu, b3 ? k0 : k1, 8);
      s = (b3 ? k1 : k0) + u2;
    } else {
      s = (b4 ? w[1] : w[0]) + __shfl_xor_sync(0xffffffffu, b4 ? w[0] : w[1], 16);
      s += __shfl_xor_sync(0xffffffffu, s, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    q = fma(s, s, q);
#pragma unroll
    for (int r = 0; r < R; ++r) w[r] = __shfl_sync(0xffffffffu, s, R == 4 ? 8 * r : 16 * r);
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < nr) {
#pragma unroll
        for (int k = 0; k < NK; ++k) acc[k] = fma(w[r], a[r][k], acc[k]);
      }
  }
  // the lanes that summed one row hold the same q: add the rows' groups
  q += __shfl_xor_sync(0xffffffffu, q, 16);
  if (R == 4) q += __shfl_xor_sync(0xffffffffu, q, 8);
}

}  // namespace lsq_apass

#include "apassdg.cuh"

namespace lsq_apass {

// the row loop for ceil(d / 32) = NK column groups, the accumulators into the warp's wred row; dg: the
// digit tables stand in wred
template <typename TA, int NK>
__device__ __forceinline__ void fused_rows_to(const TA* __restrict__ A, int64_t ld, int d, int dp, int64_t r0,
                                              int64_t r1, const double* vec_s, double* wred, double* qred,
                                              bool dg, const DigitTab& tab) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double acc[NK], q;
  bool done = false;
  if constexpr (digit_pass<TA, (NK + 1) / 2 * 2>()) {
    if (dg) {
      digit_rows<NK>(A, ld, d, r0, r1, vec_s, tab, acc, q);
      __syncthreads();  // every warp is done with the tables
      done = true;
    }
  }
  if (!done) fused_rows<TA, NK, (NK <= 6 ? 4 : 2)>(A, ld, d, r0, r1, vec_s, acc, q);
#pragma unroll
  for (int k = 0; k < NK; ++k) wred[warp * dp + lane + 32 * k] = acc[k];
  if (lane == 0) qred[warp] = q;
}

// (one body per type and width: the solver calls it from several places)
template <typename TA, int EPL>
__device__ __noinline__ void fused_pass(const TA* __restrict__ A, int64_t ld, int d, int dp, int64_t r0, int64_t r1,
                           const double* vec_s, double* wred, double* qred, double* part, int P, int cta) {
#define LSQ_FP_CASE(N) \
  case N: fused_rows_to<TA, N>(A, ld, d, dp, r0, r1, vec_s, wred, qred, dg, tab); break;
  DigitTab tab{};
  bool dg = false;
  if constexpr (digit_pass<TA, EPL>()) {
    if (r1 - r0 >= DG_MIN_ROWS) {
      const int dk = (d + 31) & ~31;
      tab = digit_tab(wred, dk);
      dg = digit_prep(tab, d, dk, vec_s, reinterpret_cast<int*>(qred));
    }
  }
  const int nk = (d + 31) >> 5;
  if constexpr (EPL <= 2) {
    fused_rows_to<TA, EPL>(A, ld, d, dp, r0, r1, vec_s, wred, qred, dg, tab);
  } else if constexpr (EPL == 4) {
    switch (nk) { LSQ_FP_CASE(3) default: LSQ_FP_CASE(4) }
  } else if constexpr (EPL == 8) {
    switch (nk) { LSQ_FP_CASE(5) LSQ_FP_CASE(6) LSQ_FP_CASE(7) default: LSQ_FP_CASE(8) }
  } else if constexpr (EPL == 16) {
    switch (nk) {
      LSQ_FP_CASE(9) LSQ_FP_CASE(10) LSQ_FP_CASE(11) LSQ_FP_CASE(12) LSQ_FP_CASE(13) LSQ_FP_CASE(14)
      LSQ_FP_CASE(15) default: LSQ_FP_CASE(16)
    }
  } else {
    switch (nk) {  // every second width: at most one empty group of 17 to 31
      case 17: LSQ_FP_CASE(18) case 19: LSQ_FP_CASE(20) case 21: LSQ_FP_CASE(22) case 23: LSQ_FP_CASE(24)
      case 25: LSQ_FP_CASE(26) case 27: LSQ_FP_CASE(28) case 29: LSQ_FP_CASE(30) default: LSQ_FP_CASE(32)
    }
  }
#undef LSQ_FP_CASE
  __syncthreads();
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < LSQ_WARPS; ++w) s += wred[w * dp + c];
    part[(int64_t)c * P + cta] = s;
  }
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < LSQ_WARPS; ++w) s += qred[w];
    part[(int64_t)dp * P + cta] = s;
  }
  __syncthreads();
}


// ------------------------------------------------------------------------------------
// FP32 arithmetic variant of the pass (the inner passes of the mixed-precision solve).
// FP64 elements are narrowed to FP32 by integer operations on their bit pattern (the
// FP64->FP32 conversion instruction runs at the FP64 rate, about 2 per clock per SM on
// this part, below the ~3 elements per clock per SM that the HBM rate needs):
// mantissa truncated to 23 bits, exponent clamped so that values below the FP32 normal
// range become (tiny) subnormal-or-zero patterns and values above it become non-finite,
// which the solver reports as a breakdown.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ float narrow_f32(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const uint32_t lo = (uint32_t)u, hi = (uint32_t)(u >> 32);
  const uint32_t e = (hi >> 20) & 0x7FFu;
  const uint32_t ec = min(max(e, 896u), 1151u) - 896u;
  const uint32_t mant = __funnelshift_l(lo, hi, 3) & 0x7FFFFFu;
  return __uint_as_float((ec << 23) | mant | (hi & 0x80000000u));
}

__device__ __forceinline__ float narrow_f32(float x) { return x; }

// column of element k of a lane's row slice: lane + 32 k, or, at EPL >= 16, 128 (k / 4) + 4 lane + k % 4
// (four adjacent columns per lane, the layout of the bulk-copy pass below, so both compute with
// the same values in the same order)
template <int EPL>
__device__ __forceinline__ int f32_col(int k, int lane) {
  return EPL >= 16 ? 128 * (k >> 2) + 4 * lane + (k & 3) : lane + 32 * k;
}

template <typename TA, int EPL>
__device__ void fused_pass_f32(const TA* __restrict__ A, int64_t ld, int d, int dp, int64_t r0, int64_t r1,
                               const double* vec_s, double* wred, double* qred, double* part, int P, int cta) {
  // two rows in flight per warp while the registers allow it (raw FP64 rows are 2 registers
  // per element); p from shared memory at the widest rows
  constexpr bool PREFETCH = sizeof(TA) == 4 || EPL <= 16;
  constexpr bool PV_REG = EPL <= 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // FP32 copy of p in the (not yet used) reduction buffer: one conversion per entry per pass
  float* pf = reinterpret_cast<float*>(wred);
  for (int c = threadIdx.x; c < dp; c += blockDim.x) pf[c] = (float)vec_s[c];
  __syncthreads();
  float pv[PV_REG ? EPL : 1], acc[EPL];
  TA cur[EPL];
  bool ok[EPL];
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    const int c = f32_col<EPL>(k, lane);
    ok[k] = c < d;
    if (PV_REG) pv[PV_REG ? k : 0] = ok[k] ? pf[c] : 0.0f;
    acc[k] = 0.0f;
  }
  double q = 0.0;
  int64_t i = r0 + warp;
  if (PREFETCH && i < r1) {
    const TA* a = A + i * ld;
#pragma unroll
    for (int k = 0; k < EPL; ++k) cur[k] = ok[k] ? __ldg(a + f32_col<EPL>(k, lane)) : (TA)0;
  }
  for (; i < r1; i += LSQ_WARPS) {
    if (!PREFETCH) {
      const TA* a = A + i * ld;
#pragma unroll
      for (int k = 0; k < EPL; ++k) cur[k] = ok[k] ? __ldg(a + f32_col<EPL>(k, lane)) : (TA)0;
    }
    // narrow the row first (its raw registers die here), then put the next row in flight
    float af[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) af[k] = narrow_f32(cur[k]);
    if (PREFETCH) {
      const int64_t inext = i + LSQ_WARPS;
      if (inext < r1) {
        const TA* a = A + inext * ld;
#pragma unroll
        for (int k = 0; k < EPL; ++k) cur[k] = ok[k] ? __ldg(a + f32_col<EPL>(k, lane)) : (TA)0;
      }
    }
    float w = 0.0f;
#pragma unroll
    for (int k = 0; k < EPL; ++k) w = fmaf(af[k], PV_REG ? pv[PV_REG ? k : 0] : pf[f32_col<EPL>(k, lane)], w);
    w = warp_sumf(w);
#pragma unroll
    for (int k = 0; k < EPL; ++k) acc[k] = fmaf(w, af[k], acc[k]);
    q = fma((double)w, (double)w, q);
  }
  __syncthreads();  // every warp is done with pf before wred is overwritten
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    const int c = f32_col<EPL>(k, lane);
    if (c < dp) wred[warp * dp + c] = (double)acc[k];
  }
  if (lane == 0) qred[warp] = q;
  __syncthreads();
  for (int c = threadIdx.x; c < dp; c += blockDim.x) {
    double s = 0.0;
#pragma unroll
    for (int w2 = 0; w2 < LSQ_WARPS; ++w2) s += wred[w2 * dp + c];
    part[(int64_t)c * P + cta] = s;
  }
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w2 = 0; w2 < LSQ_WARPS; ++w2) s += qred[w2];
    part[(int64_t)dp * P + cta] = s;
  }
  __syncthreads();
}


// ------------------------------------------------------------------------------------
// The FP32 pass for wide FP32 rows (128 < d <= 1024, d a multiple of 4, 16-byte aligned rows)
// with the rows staged by bulk copies: each warp keeps ring_ns(EPL) of its rows in flight in a ring
// of shared-memory slots, one cp.async.bulk per row started by lane 0 and counted in bytes on
// the slot's mbarrier, instead of one row prefetched in registers.  The registers that frees
// hold p, and the deeper queue keeps HBM busy with one 256-thread CTA per SM.  Lane l owns the
// columns f32_col(k, l), as in the pass above, and both add in one order: the same bits.
// Rows of 129 to 256 columns: two mixed solves over 262144 x 256, 6.76 -> 6.64 ms.
// Every wait is bounded: on a time-out the pass records LSQ_ERR_TIMEOUT, waits (bounded) for
// its copies still in flight and returns; the caller checks the flag at its next barrier.
// ------------------------------------------------------------------------------------
// rows of a warp in flight: 16 KB a warp at most, and no less than 8 KB at 1 KB rows
constexpr __host__ __device__ int ring_ns(int epl) { return epl == 8 ? 8 : 4; }
constexpr uint32_t RING_SPIN = 1u << 24;

__device__ __forceinline__ uint32_t smem_u32a(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ring_init(uint64_t* bars, int n) {
  // thread 0, before a CTA barrier: one arrival (the expect-tx) per phase
  for (int e = 0; e < n; ++e)
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32a(bars + e)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void ring_issue(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32a(bar)), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32a(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32a(bar))
      : "memory");
}

__device__ __forceinline__ bool ring_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t spins = 0; spins < RING_SPIN; ++spins) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32a(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// ring: LSQ_WARPS x ring_ns(EPL) slots of `slot_floats` floats; bars: as many mbarriers;
// phase: this thread's parity bits of its warp's slots (kept across passes by the caller)
template <int EPL>
__device__ inline void fused_pass_f32_ring(const float* __restrict__ A, int64_t ld, int d, int dp, int64_t r0,
                                           int64_t r1, const double* vec_s, double* wred, double* qred, double* part,
                                           int P, int cta, float* ring, int slot_floats, uint64_t* bars,
                                           uint32_t& phase, int* err) {
  static_assert(EPL == 8 || EPL == 16 || EPL == 32, "rows of 256, 512 or 1024 padded columns");
  constexpr int NS = ring_ns(EPL);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* pf = reinterpret_cast<float*>(wred);
  for (int c = threadIdx.x; c < dp; c += blockDim.x) pf[c] = (float)vec_s[c];
  __syncthreads();
  float pv[EPL], acc[EPL];
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    const int c = f32_col<EPL>(k, lane);
    pv[k] = c < d ? pf[c] : 0.0f;
    acc[k] = 0.0f;
  }
  double q = 0.0;
  float* slots = ring + (size_t)warp * NS * slot_floats;
  uint64_t* bar = bars + warp * NS;
  const uint32_t bytes = (uint32_t)d * 4u;
  const int64_t first = r0 + warp;
  // rows first + LSQ_WARPS j of this warp; slot j % NS
  int64_t issued = 0, done = 0;
  const int64_t nrows = first < r1 ? (r1 - first + LSQ_WARPS - 1) / LSQ_WARPS : 0;
  for (; issued < nrows && issued < NS; ++issued)
    if (lane == 0) ring_issue(slots + issued * slot_floats, A + (first + LSQ_WARPS * issued) * ld, bytes, bar + issued);
  bool good = true;
  for (; done < nrows; ++done) {
    const int s = (int)(done % NS);
    const bool landed = __all_sync(0xffffffffu, ring_wait(bar + s, (phase >> s) & 1u));
    if (!landed) {
      good = false;
      break;
    }
    phase ^= 1u << s;
    const float* row = slots + s * slot_floats;
    float af[EPL];
    if constexpr (EPL >= 16) {
      // four adjacent columns a lane; d is a multiple of 4, so they are in or out together
#pragma unroll
      for (int k = 0; k < EPL; k += 4) {
        const int c = f32_col<EPL>(k, lane);
        const float4 v = c < d ? *reinterpret_cast<const float4*>(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        af[k] = v.x;
        af[k + 1] = v.y;
        af[k + 2] = v.z;
        af[k + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int k = 0; k < EPL; ++k) {
        const int c = f32_col<EPL>(k, lane);
        af[k] = c < d ? row[c] : 0.0f;
      }
    }
    __syncwarp();  // every lane has its values: the slot may be refilled
    if (issued < nrows) {
      if (lane == 0) ring_issue(slots + s * slot_floats, A + (first + LSQ_WARPS * issued) * ld, bytes, bar + s);
      ++issued;
    }
    float w = 0.0f;
#pragma unroll
    for (int k = 0; k < EPL; ++k) w = fmaf(af[k], pv[k], w);
    w = warp_sumf(w);
#pragma unroll
    for (int k = 0; k < EPL; ++k) acc[k] = fmaf(w, af[k], acc[k]);
    q = fma((double)w, (double)w, q);
  }
  if (!good) {
    if (lane == 0) atomicCAS(err, 0, (int)LSQ_ERR_TIMEOUT);
    // the copies still in flight land before the slots are given up (bounded)
    for (; done < issued; ++done) {
      const int s = (int)(done % NS);
      if (ring_wait(bar + s, (phase >> s) & 1u)) phase ^= 1u << s;
    }
  }
  __syncthreads();  // every warp is done with pf before wred is overwritten
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    const int c = f32_col<EPL>(k, lane);
    if (c < dp) wred[warp * dp + c] = (double)acc[k];
  }
  if (lane == 0) qred[warp] = q;
  __syncthreads();
  for (int c = threadIdx.x; c < dp; c += blockDim.x) {
    double s2 = 0.0;
#pragma unroll
    for (int w2 = 0; w2 < LSQ_WARPS; ++w2) s2 += wred[w2 * dp + c];
    part[(int64_t)c * P + cta] = s2;
  }
  if (threadIdx.x == 0) {
    double s2 = 0.0;
    for (int w2 = 0; w2 < LSQ_WARPS; ++w2) s2 += qred[w2];
    part[(int64_t)dp * P + cta] = s2;
  }
  __syncthreads();
}

// ------------------------------------------------------------------------------------
// Exact pass in double-FP32 arithmetic (the residual replacements of the mixed solve).
// Each FP64 element a is split into a head of 21 significant bits and the FP32 rounding
// of its remaining 32 mantissa bits (about 45 significant bits in all); products are made
// error-free with an FMA (TwoProduct) and sums are carried as unevaluated (hi, lo) FP32
// pairs with Knuth's TwoSum (Dekker 1971; Knuth, TAOCP vol. 2).  v = A^T (A x) comes out
// with a relative error of a few 1e-14 per component, far below what the solver's
// tolerance needs, at the throughput of the FP32 and integer pipes.
// Elements with |a| < 2^-74 keep only their head (their tail would underflow FP32).
// ------------------------------------------------------------------------------------
struct dfl {
  float hi, lo;
};

__device__ __forceinline__ void split_df(double x, float& head, float& tail) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const uint32_t lo32 = (uint32_t)u, hi32 = (uint32_t)(u >> 32);
  const uint32_t sign = hi32 & 0x80000000u;
  const uint32_t e = (hi32 >> 20) & 0x7FFu;
  const uint32_t ec = min(max(e, 896u), 1151u);
  head = __uint_as_float(sign | ((ec - 896u) << 23) | ((hi32 & 0xFFFFFu) << 3));
  // tail = lo32 * 2^(e - 1075), sign of x; zero when that scale leaves the FP32 range
  const float scale = __uint_as_float(sign | ((e - 948u) << 23));
  tail = (e >= 949u && e <= 1151u) ? __fmul_rn(__uint2float_rn(lo32), scale) : 0.0f;
}

__device__ __forceinline__ void split_df(float x, float& head, float& tail) {
  head = x;
  tail = 0.0f;
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& err) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// (sh, sl) += (ah + al) * (bh + bl), dropping only al * bl
__device__ __forceinline__ void df_fma(float ah, float al, float bh, float bl, float& sh, float& sl) {
  const float p = __fmul_rn(ah, bh);
  const float pe = __fmaf_rn(ah, bh, -p);
  const float cross = __fmaf_rn(ah, bl, __fmaf_rn(al, bh, pe));
  float s, e;
  two_sum(sh, p, s, e);
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(e, cross));
}

__device__ __forceinline__ void df_add(float& ah, float& al, float bh, float bl) {
  float s, e;
  two_sum(ah, bh, s, e);
  ah = s;
  al = __fadd_rn(al, __fadd_rn(e, bl));
}

// v partials only (the residual needs no q); part[dp * P + cta] is written as 0
template <typename TA, int EPL>
__device__ void fused_pass_df(const TA* __restrict__ A, int64_t ld, int d, int dp, int64_t r0, int64_t r1,
                              const double* vec_s, double* wred, double* qred, double* part, int P, int cta) {
  constexpr bool PREFETCH = sizeof(TA) == 4 || EPL <= 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2* xs = reinterpret_cast<float2*>(wred);  // (head, tail) of x, dp entries
  for (int c = threadIdx.x; c < dp; c += blockDim.x) {
    const double xv = vec_s[c];
    const float xh = (float)xv;
    xs[c] = make_float2(xh, (float)(xv - (double)xh));
  }
  __syncthreads();
  float vh[EPL], vl[EPL];
  TA cur[EPL];
  bool ok[EPL];
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    ok[k] = lane + 32 * k < d;
    vh[k] = 0.0f;
    vl[k] = 0.0f;
  }
  int64_t i = r0 + warp;
  if (PREFETCH && i < r1) {
    const TA* a = A + i * ld;
#pragma unroll
    for (int k = 0; k < EPL; ++k) cur[k] = ok[k] ? __ldg(a + lane + 32 * k) : (TA)0;
  }
  for (; i < r1; i += LSQ_WARPS) {
    if (!PREFETCH) {
      const TA* a = A + i * ld;
#pragma unroll
      for (int k = 0; k < EPL; ++k) cur[k] = ok[k] ? __ldg(a + lane + 32 * k) : (TA)0;
    }
    float ah[EPL], al[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) split_df(cur[k], ah[k], al[k]);
    if (PREFETCH) {
      const int64_t inext = i + LSQ_WARPS;
      if (inext < r1) {
        const TA* a = A + inext * ld;
#pragma unroll
        for (int k = 0; k < EPL; ++k) cur[k] = ok[k] ? __ldg(a + lane + 32 * k) : (TA)0;
      }
    }
    float wh = 0.0f, wl = 0.0f;
#pragma unroll
    for (int k = 0; k < EPL; ++k) {
      const float2 xv = xs[lane + 32 * k];
      df_fma(ah[k], al[k], xv.x, xv.y, wh, wl);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, wh, o);
      const float ol = __shfl_xor_sync(0xffffffffu, wl, o);
      df_add(wh, wl, oh, ol);
    }
    // renormalise w to a clean (head, tail) pair
    float nh, nl;
    two_sum(wh, wl, nh, nl);
#pragma unroll
    for (int k = 0; k < EPL; ++k) df_fma(ah[k], al[k], nh, nl, vh[k], vl[k]);
  }
  __syncthreads();  // every warp is done with xs before wred is overwritten
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    const int c = lane + 32 * k;
    if (c < dp) wred[warp * dp + c] = (double)vh[k] + (double)vl[k];
  }
  if (lane == 0) qred[warp] = 0.0;
  __syncthreads();
  for (int c = threadIdx.x; c < dp; c += blockDim.x) {
    double sum = 0.0;
#pragma unroll
    for (int w2 = 0; w2 < LSQ_WARPS; ++w2) sum += wred[w2 * dp + c];
    part[(int64_t)c * P + cta] = sum;
  }
  if (threadIdx.x == 0) part[(int64_t)dp * P + cta] = 0.0;
  __syncthreads();
}

// The same pass for FP64 rows, staged through shared memory: each warp has one row slot
// (slots: LSQ_WARPS x dp doubles, which may lie in wred past its first dp entries) and, as
// soon as the current row is split into registers, has the next row copied into the slot
// with cp.async while it computes, so a row is in flight without holding registers (the
// split row and the double-FP32 accumulators already fill them).  Each lane copies and reads
// only its own elements (columns lane + 32 k): its own cp.async.wait_group orders the data,
// and a __syncwarp (which orders the memory operations of the lanes it joins) separates the
// loads of the current row from the copy of the next one into the same slot.  Same
// arithmetic, in the same order, as fused_pass_df.
__device__ __forceinline__ void cp_async_8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_none() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <int EPL>
__device__ void fused_pass_df_staged(const double* __restrict__ A, int64_t ld, int d, int dp, int64_t r0, int64_t r1,
                                     const double* vec_s, double* wred, double* qred, double* part, int P, int cta,
                                     double* slots) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2* xs = reinterpret_cast<float2*>(wred);  // (head, tail) of x, dp entries
  for (int c = threadIdx.x; c < dp; c += blockDim.x) {
    const double xv = vec_s[c];
    const float xh = (float)xv;
    xs[c] = make_float2(xh, (float)(xv - (double)xh));
  }
  double* slot = slots + (int64_t)warp * dp + lane;
  float vh[EPL], vl[EPL];
  bool ok[EPL];
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    ok[k] = lane + 32 * k < d;
    vh[k] = 0.0f;
    vl[k] = 0.0f;
    // columns at or past d are never copied: zero in the slot for the whole pass
    if (!ok[k]) slot[32 * k] = 0.0;
  }
  __syncthreads();  // xs complete; no warp still reads wred from before the pass
  int64_t i = r0 + warp;
  if (i < r1) {
    const double* a = A + i * ld + lane;
#pragma unroll
    for (int k = 0; k < EPL; ++k)
      if (ok[k]) cp_async_8(slot + 32 * k, a + 32 * k);
  }
  cp_async_commit_group();
  for (; i < r1; i += LSQ_WARPS) {
    cp_async_wait_none();  // row i has landed
    float ah[EPL], al[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) split_df(slot[32 * k], ah[k], al[k]);
    __syncwarp();
    const int64_t inext = i + LSQ_WARPS;
    if (inext < r1) {
      const double* a = A + inext * ld + lane;
#pragma unroll
      for (int k = 0; k < EPL; ++k)
        if (ok[k]) cp_async_8(slot + 32 * k, a + 32 * k);
    }
    cp_async_commit_group();
    float wh = 0.0f, wl = 0.0f;
#pragma unroll
    for (int k = 0; k < EPL; ++k) {
      const float2 xv = xs[lane + 32 * k];
      df_fma(ah[k], al[k], xv.x, xv.y, wh, wl);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, wh, o);
      const float ol = __shfl_xor_sync(0xffffffffu, wl, o);
      df_add(wh, wl, oh, ol);
    }
    float nh, nl;
    two_sum(wh, wl, nh, nl);
#pragma unroll
    for (int k = 0; k < EPL; ++k) df_fma(ah[k], al[k], nh, nl, vh[k], vl[k]);
  }
  cp_async_wait_none();
  __syncthreads();  // every warp is done with xs and its slot before wred is overwritten
#pragma unroll
  for (int k = 0; k < EPL; ++k) {
    const int c = lane + 32 * k;
    if (c < dp) wred[warp * dp + c] = (double)vh[k] + (double)vl[k];
  }
  if (lane == 0) qred[warp] = 0.0;
  __syncthreads();
  for (int c = threadIdx.x; c < dp; c += blockDim.x) {
    double sum = 0.0;
#pragma unroll
    for (int w2 = 0; w2 < LSQ_WARPS; ++w2) sum += wred[w2 * dp + c];
    part[(int64_t)c * P + cta] = sum;
  }
  if (threadIdx.x == 0) part[(int64_t)dp * P + cta] = 0.0;
  __syncthreads();
}

// sum_{j < P} src[j] by one warp, fixed order
__device__ __forceinline__ double warp_sum_strip(const double* src, int P) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int j = lane; j < P; j += 32) s += src[j];
  return warp_sum(s);
}

// standalone pass: CTA b handles rows [b * rows_per_cta, (b + 1) * rows_per_cta)
template <typename TA, int EPL>
__global__ void __launch_bounds__(LSQ_THREADS, (EPL <= 16 ? 2 : 1)) hmatvec_kernel(const void* A, int64_t n, int d, int dp, int64_t ld,
                                                                  int64_t rows_per_cta, const double* p, double* part) {
  extern __shared__ __align__(16) double smem[];
  double* vec = smem;
  double* wred = vec + dp;
  double* qred = wred + LSQ_WARPS * dp;
  for (int c = threadIdx.x; c < dp; c += blockDim.x) vec[c] = c < d ? p[c] : 0.0;
  __syncthreads();
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_cta;
  const int64_t r1 = min(n, r0 + rows_per_cta);
  fused_pass<TA, EPL>(reinterpret_cast<const TA*>(A), ld, d, dp, r0, r1, vec, wred, qred, part, gridDim.x,
                      blockIdx.x);
}

// v[c] = sum_j part[c][j] (c < d), q = sum_j part[dp][j]; one warp per output, fixed order
static __global__ void reduce_part_kernel(const double* part, int P, int d, int dp, double* v, double* q) {
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int c = gw; c <= d; c += nw) {
    const int src = c < d ? c : dp;
    const double s = warp_sum_strip(part + (int64_t)src * P, P);
    if (lane == 0) {
      if (c < d) v[c] = s;
      else *q = s;
    }
  }
}

// elements per lane: the smallest power of two with 32 * EPL >= d
static inline int epl_for(int d) {
  int e = 1;
  while (32 * e < d) e <<= 1;
  return e;
}

template <typename TA>
static void* pick_hmv(int epl) {
  switch (epl) {
    case 1: return (void*)hmatvec_kernel<TA, 1>;
    case 2: return (void*)hmatvec_kernel<TA, 2>;
    case 4: return (void*)hmatvec_kernel<TA, 4>;
    case 8: return (void*)hmatvec_kernel<TA, 8>;
    case 16: return (void*)hmatvec_kernel<TA, 16>;
    default: return (void*)hmatvec_kernel<TA, 32>;
  }
}

static inline size_t hmatvec_smem_bytes(int dp) { return (size_t)(dp + LSQ_WARPS * dp + LSQ_WARPS) * 8; }

}  // namespace lsq_apass
