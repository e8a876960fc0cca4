// btile.cuh -- the exact passes of the mixed-precision batched solves over FP32 A (included by batch.cu
// inside its namespace, after BProb / BatchArgs): V = A^T (A X) in double-FP32 for the active
// right-hand sides of a chunk of rows, one read of the rows (the residual replacements; Section 1,
// eq. (PCG) per right-hand side).
//
// The active right-hand sides are taken 8 or 4 at a time (KP), so one that has stopped costs nothing.  A
// stage of R rows (about 16 K elements) sits in shared memory, the next one to three on their way in
// with cp.async:
//   product 1  Y = A_stage X: a thread owns 2 rows x KP right-hand sides of registers and every
//              ncs-th column (Q = ceil(d / ncs) of them); a warp covers CSW column slices, so that a
//              row of X is read by 32 / CSW lanes at once.  The slices' partial sums are added over
//              the lanes (each exchange halves the values a lane keeps), then, for d > 136, over 2
//              or 4 warps through shared memory.
//   product 2  V += A_stage^T Y: a thread owns 2 columns x KP sums and every RS-th block of 4 rows.
//              The row splits are added in FP64 at the end of the chunk.
// The row stride in shared memory is congruent to CSW modulo 2 CSW, so the lanes of product 1
// (32 / CSW rows apart, CSW consecutive columns) meet 32 distinct banks; the rows of X are spaced
// so that 8 consecutive ones do.
//
// Bound by the FP32 pipe: 11 additions and multiplications per product (TwoProduct, TwoSum), 2 KP
// products an element.  Two right-hand sides share an instruction (f32x2: the same pipe rate, half the
// issue slots).  Measured over the 256 problems of a batch (n 2^12..2^18, d 32..512, k 1..16; 9.2 GB of A,
// all right-hand sides active): 38.8 ms a pass with a warp per group of rows and lanes on columns, 27 ms.
#pragma once

constexpr int TT = 512;                        // threads of a pass CTA
constexpr int TW = TT / 32;
constexpr size_t TSMEM = 226 * 1024;           // dynamic shared memory
constexpr int TSTAGE = 17920;                  // most floats of a stage

struct TileShape {
  int CSW, u, ncs, Q, R, stride, rep;  // slices per warp, column groups of warps, slices, columns per slice
};

__device__ __forceinline__ TileShape tile_shape(int d) {
  TileShape t;
  t.CSW = d >= 64 ? 8 : d >= 32 ? 4 : 2;
  t.u = d <= 136 ? 1 : d <= 272 ? 2 : 4;
  t.ncs = t.CSW * t.u;
  t.Q = (d + t.ncs - 1) / t.ncs;
  // smallest stride >= d congruent to CSW modulo 2 CSW
  t.stride = (d + t.CSW - 1) / (2 * t.CSW) * (2 * t.CSW) + t.CSW;
  if (t.stride < d) t.stride += 2 * t.CSW;
  const int base = 2 * (TW / t.u) * (32 / t.CSW);  // rows one round of the warps covers
  t.rep = max(1, min(512, TSTAGE / t.stride) / base);
  t.R = base * t.rep;
  return t;
}

// ---- two FP32 values in a 64-bit register
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// (sh, sl) += a (bh + bl) with a exact in FP32 and na = -a: TwoProduct by FMA, the tail product
// folded into the error term, TwoSum into the head (Dekker 1971; Knuth)
__device__ __forceinline__ void f2_df_fma(f2 a, f2 na, f2 bh, f2 bl, f2& sh, f2& sl) {
  const f2 np = f2_mul(na, bh);  // minus the product
  const f2 cross = f2_fma(a, bl, f2_fma(a, bh, np));
  const f2 s = f2_sub(sh, np);
  const f2 bb = f2_sub(s, sh);
  const f2 e = f2_sub(f2_sub(sh, f2_sub(s, bb)), f2_add(np, bb));
  sh = s;
  sl = f2_add(sl, f2_add(e, cross));
}

template <int F>
__device__ __forceinline__ void tp_copy(float* dst, const float* src, int nbytes) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (F == 4)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(a), "l"(src), "r"(nbytes) : "memory");
  else if constexpr (F == 2)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(a), "l"(src), "r"(nbytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(a), "l"(src), "r"(nbytes) : "memory");
}

// rows [lo, lo + R) of A (zeros from r1 on) into a stage, F floats a copy
template <int F>
__device__ __forceinline__ void tp_load(const float* __restrict__ A, int64_t ld, int d, int64_t lo, int64_t r1, int R,
                                        int stride, float* buf) {
  const int pc = (d + F - 1) / F;                          // copies per row
  const unsigned magic = 0xFFFFFFFFu / (unsigned)pc + 1u;  // e / pc for e < 2^18 (pc = 1: not used)
  for (int e = threadIdx.x; e < R * pc; e += TT) {
    const int r = pc == 1 ? e : (int)__umulhi((unsigned)e, magic), c = (e - r * pc) * F;
    const bool in = lo + r < r1;
    tp_copy<F>(buf + r * stride + c, A + (in ? (lo + r) * ld + c : 0), in ? 4 * min(F, d - c) : 0);
  }
}

// KP values of a 16-byte aligned row, in pairs
template <int KP>
__device__ __forceinline__ void tp_row(const float* p, f2 (&v)[KP / 2]) {
#pragma unroll
  for (int j = 0; j < KP; j += 4) {
    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(p + j);
    v[j / 2] = x.x;
    v[j / 2 + 1] = x.y;
  }
}

// one exchange of the lane sums: lanes with `bit` set keep the upper half of the 2 H values
template <int H, int N>
__device__ __forceinline__ void tp_halve_df(float (&h)[N], float (&l)[N], int bit) {
  const bool up = (threadIdx.x & bit) != 0;
#pragma unroll
  for (int x = 0; x < H; ++x) {
    const float gh = up ? h[x] : h[x + H], gl = up ? l[x] : l[x + H];
    float kh = up ? h[x + H] : h[x], kl = up ? l[x + H] : l[x];
    lsq_apass::df_add(kh, kl, __shfl_xor_sync(0xffffffffu, gh, bit), __shfl_xor_sync(0xffffffffu, gl, bit));
    h[x] = kh;
    l[x] = kl;
  }
}

// One exact chunk, rows [r0, r1) of problem pr, for the right-hand sides jl[0 .. na), na <= KP:
//   out[jl[x] dp + c] = sum_rows a_c (a . x_j) for c < d,  out[kp dp + jl[x]] = 0 (an exact pass needs no q).
// Called by every thread of the CTA.
template <int KP>
__device__ __forceinline__ void tp_chunk(const BProb& pr, int64_t r0, int64_t r1, double* __restrict__ out,
                                         float* smf, const int* jl, int na) {
  constexpr int KW = 2 * KP;             // floats of a row of X and of Y: heads, then tails
  constexpr int PS = KW == 16 ? 20 : 12;  // their spacing in X
  constexpr int CW = 2;
  const int d = pr.d, dp = pr.dp, kp = pr.kp;
  const TileShape ts = tile_shape(d);
  const int R = ts.R, stride = ts.stride, Q = ts.Q, ncs = ts.ncs, u = ts.u, CSW = ts.CSW;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* Xs = smf;                                                  // [d][PS]
  float* Ys = Xs + d * PS;                                          // [R][KW]
  float* Yp = u > 1 ? Ys + R * KW : Ys;                             // [u][R][KW]
  float* stage0 = Ys + (u > 1 ? u + 1 : 1) * R * KW;
  const int sf = R * stride;                                        // floats of a stage
  const int NS = min(4, ((int)(TSMEM / 4) - (int)(stage0 - smf)) / sf);  // stages: 2 to 4
  const float* A = reinterpret_cast<const float*>(pr.A);
  const int64_t ld = pr.ld;
  const int F = CSW >= 4 && pr.vec ? 4 : (ld % 2 == 0 && ((uintptr_t)A % 8) == 0) ? 2 : 1;
  const int nst = (int)((r1 - r0 + R - 1) / R);
  auto load = [&](int t) {
    if (t < nst) {
      float* buf = stage0 + (t % NS) * sf;
      const int64_t lo = r0 + (int64_t)t * R;
      if (F == 4) tp_load<4>(A, ld, d, lo, r1, R, stride, buf);
      else if (F == 2) tp_load<2>(A, ld, d, lo, r1, R, stride, buf);
      else tp_load<1>(A, ld, d, lo, r1, R, stride, buf);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int t = 0; t < NS - 1; ++t) load(t);
  // heads and tails of x, zero past the active right-hand sides
  for (int e = tid; e < d * KP; e += TT) {
    const int c = e / KP, x = e - c * KP;
    const int64_t at = (int64_t)c * kp + (x < na ? jl[x] : 0);
    Xs[c * PS + x] = x < na ? pr.Xh[at] : 0.f;
    Xs[c * PS + KP + x] = x < na ? pr.Xl[at] : 0.f;
  }
  // product 1: this thread's slice and its two rows of each round (rg0 and rg0 + NRG)
  const int csg = warp % u, cs = csg * CSW + lane % CSW;
  const int RGW = 32 / CSW, rg0 = (warp / u) * RGW + lane / CSW;
  const int NRG = (TW / u) * RGW;
  // product 2: columns g and g + G, blocks of 4 rows rs, rs + RS, ...
  const int G = (d + CW - 1) / CW, RS = TT / G;
  const int g = tid % G, rs = tid / G;
  const int colb = min(g + G, d - 1);  // (sums past d are not written)
  f2 vh[CW][KP / 2], vl[CW][KP / 2];
#pragma unroll
  for (int i = 0; i < CW; ++i)
#pragma unroll
    for (int j = 0; j < KP / 2; ++j) vh[i][j] = vl[i][j] = 0ull;
  // the sum over the column groups: this thread's right-hand side tid % KP, rows tid / KP, + TT / KP, ...
  const int qj = tid % KP, qr = tid / KP;
  constexpr int QS = TT / KP;
  for (int t = 0; t < nst; ++t) {
    const float* As = stage0 + (t % NS) * sf;
    // stage t has landed (NS - 2 younger groups may be in flight)
    if (NS == 2) asm volatile("cp.async.wait_group 0;" ::: "memory");
    else if (NS == 3) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 2;" ::: "memory");
    __syncthreads();  // for every thread; stage t - 1 and Y are no longer read
    load(t + NS - 1);
    for (int rep = 0; rep < ts.rep; ++rep) {
      const int row = rep * 2 * NRG + rg0;
      const float* a0 = As + row * stride + cs;
      const float* a1 = a0 + NRG * stride;
      const float* p = Xs + cs * PS;
      f2 yh[KP], yl[KP];  // rows 0 and 1, KP / 2 pairs each
#pragma unroll
      for (int x = 0; x < KP; ++x) yh[x] = yl[x] = 0ull;
      auto step = [&](float x0, float x1, const float* pp) {
        f2 ph[KP / 2], pl[KP / 2];
        tp_row<KP>(pp, ph);
        tp_row<KP>(pp + KP, pl);
        const f2 d0 = f2_pack(x0, x0), d1 = f2_pack(x1, x1), n0 = f2_pack(-x0, -x0), n1 = f2_pack(-x1, -x1);
#pragma unroll
        for (int j = 0; j < KP / 2; ++j) {
          f2_df_fma(d0, n0, ph[j], pl[j], yh[j], yl[j]);
          f2_df_fma(d1, n1, ph[j], pl[j], yh[KP / 2 + j], yl[KP / 2 + j]);
        }
      };
#pragma unroll 2
      for (int q = 0; q < Q - 1; ++q) {
        step(*a0, *a1, p);
        a0 += ncs;
        a1 += ncs;
        p += ncs * PS;
      }
      if (cs + ncs * (Q - 1) < d) step(*a0, *a1, p);  // only a slice's last column can lie past d
      // sums over the CSW slices of the warp: the rows are halved first, then the right-hand sides
      float h[2 * KP], l[2 * KP];
#pragma unroll
      for (int x = 0; x < KP; ++x) {
        f2_unpack(yh[x], h[2 * x], h[2 * x + 1]);
        f2_unpack(yl[x], l[2 * x], l[2 * x + 1]);
      }
      const int b0 = lane & 1, b1 = (lane >> 1) & 1, b2 = (lane >> 2) & 1;
      tp_halve_df<KP>(h, l, 1);
      int n = KP, j0 = 0;  // values left and the first one's right-hand side
      if (CSW >= 4) {
        tp_halve_df<KP / 2>(h, l, 2);
        n = KP / 2;
        j0 = b1 * (KP / 2);
      }
      if (CSW == 8) {
        tp_halve_df<KP / 4>(h, l, 4);
        n = KP / 4;
        j0 += b2 * (KP / 4);
      }
      float* yo = Yp + (csg * R + row + b0 * NRG) * KW + j0;
#pragma unroll
      for (int x = 0; x < KP; ++x)
        if (x < n) {
          float sh = h[x], sl = l[x];
          if (u == 1) lsq_apass::two_sum(h[x], l[x], sh, sl);  // a clean (head, tail) pair
          yo[x] = sh;
          yo[KP + x] = sl;
        }
    }
    __syncthreads();
    if (u > 1) {  // Y from the column groups of warps, in order
      for (int r = qr; r < R; r += QS) {
        float yv = Yp[r * KW + qj], tl = Yp[r * KW + KP + qj];
        for (int x = 1; x < u; ++x) lsq_apass::df_add(yv, tl, Yp[(x * R + r) * KW + qj], Yp[(x * R + r) * KW + KP + qj]);
        float sh, sl;
        lsq_apass::two_sum(yv, tl, sh, sl);
        Ys[r * KW + qj] = sh;
        Ys[r * KW + KP + qj] = sl;
      }
      __syncthreads();
    }
    if (rs < RS) {
      for (int rb = rs * 4; rb < R; rb += RS * 4) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const float* ar = As + (rb + x) * stride;
          const float x0 = ar[g], x1 = ar[colb];
          const f2 d0 = f2_pack(x0, x0), d1 = f2_pack(x1, x1), n0 = f2_pack(-x0, -x0), n1 = f2_pack(-x1, -x1);
          f2 yh[KP / 2], yl[KP / 2];
          tp_row<KP>(Ys + (rb + x) * KW, yh);
          tp_row<KP>(Ys + (rb + x) * KW + KP, yl);
#pragma unroll
          for (int j = 0; j < KP / 2; ++j) {
            f2_df_fma(d0, n0, yh[j], yl[j], vh[0][j], vl[0][j]);
            f2_df_fma(d1, n1, yh[j], yl[j], vh[1][j], vl[1][j]);
          }
        }
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();  // the stages are free for the reduction (66 KB at most)
  double* red = reinterpret_cast<double*>(stage0);  // [RS][KP][CW][G]
  if (rs < RS) {
#pragma unroll
    for (int i = 0; i < CW; ++i)
#pragma unroll
      for (int j = 0; j < KP / 2; ++j) {
        float a, b, al, bl;
        f2_unpack(vh[i][j], a, b);
        f2_unpack(vl[i][j], al, bl);
        red[((size_t)(rs * KP + 2 * j) * CW + i) * G + g] = (double)a + (double)al;
        red[((size_t)(rs * KP + 2 * j + 1) * CW + i) * G + g] = (double)b + (double)bl;
      }
  }
  __syncthreads();
  for (int e = tid; e < na * d; e += TT) {
    const int x = e / d, c = e - x * d;
    double sum = 0.0;
    for (int y = 0; y < RS; ++y) sum += red[(size_t)(y * KP + x) * CW * G + c];  // c = g + G i
    out[(size_t)jl[x] * dp + c] = sum;
  }
  if (tid < na) out[(size_t)kp * dp + jl[tid]] = 0.0;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // a bulk copy may come into this memory next
  __syncthreads();
}
