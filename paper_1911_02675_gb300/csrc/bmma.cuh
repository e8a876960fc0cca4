// bmma.cuh -- the FP32 pass of the batched solves over FP32 A on the tensor cores (included by
// batch.cu inside its namespace, after btile.cuh): V = A^T (A P), q_j = ||A p_j||^2 for the active
// directions of a chunk of rows (Section 1, eq. (PCG) per right-hand side), one read of the rows.
//
// A stage of R rows (up to 16 K elements) sits in shared memory, the next ones on their way in.
//   product 1  Y = A_stage P by m16n8k8 TF32 MMAs: a warp takes one 16-row tile and one of KS runs
//              of at most 8 k-steps (KS nrt = 16 warps), the partial tiles go to shared memory;
//   Y          the KS partial tiles summed in a fixed order, q_j += y_j^2, Y split for product 2;
//   product 2  V_stage = A_stage^T Y: a warp owns up to three 16-column tiles of V, each with a share
//              of the stage's 8-row k-steps; V_stage is added to the running V by FP32 additions
//              (the tensor cores' own accumulation is kept to one stage: over thousands of steps its
//              rounding drifts).
// Each product is three MMAs over a split of both operands into a TF32 head (rounded to nearest)
// and the FP32 remainder: a_h b_h + a_h b_l + a_l b_h, the dropped a_l b_l below 2^-22 of the
// product (the remainder itself is read as TF32, a relative 2^-11 of it).
//
// A's elements are read twice from shared memory, as 4-byte words: product 1 by lanes (row g,
// column t), product 2 by lanes (row pair t, column g).  Both are free of bank conflicts when the
// row stride is 4 x odd: the columns of a k-step and the rows of a tile may be taken in any order,
// so with a stride of 2 x odd (odd) the eight rows of a tile half lie 2 (4) apart, and the row pairs
// of a k-step 4 (8).  That covers the rows as they lie in memory unless d is a multiple of 8; those
// are copied one by one to a stride 4 more than a multiple of 8.  (Rows are contiguous and 16-byte
// aligned: batch.cu sends other problems to the tiled pass.)
//
// Why warp-level MMAs: at HBM rate an SM has ~20 instructions per element and thread slot; FP32 FMAs
// took 53 at 16 right-hand sides (packed two to an instruction) and ran at 1.2 TB/s, bound by issue
// and by shared-memory reads of P and Y.  The MMAs alone take 3 to 6, and the 512 TF32 products a clock an SM
// allow 5.3 elements a clock (HBM: 5.7).  tcgen05 would need A in shared memory twice (as A and as
// A^T) and split in two.  16 warps of 128 registers, with P's fragments in shared memory, rather than 8
// of 255 with the fragments in registers and rows as they lie in memory (2.3-way bank conflicts on
// average): 5.8 -> 4.2 ms a pass over the 256 problems of a batch (n 2^12..2^18, d 32..512, k 1..16; 9.2 GB);
// 2.3 TB/s at 4 right-hand sides of d = 512 and 1.8 at 16.  What bounds it now is issue (33 instructions
// an element at 4 right-hand sides at 2 a clock): addresses, barriers and the fold of each stage's sums.  (At
// 128 registers the kernel, the exact pass with it, spills 48 bytes.)
#pragma once

constexpr int YP = 36;                   // floats between rows of Y (16 pairs of head and remainder)

struct MmaShape {
  int lgks, R, kd, kps, stride, lgm;  // log2 of the K runs, rows, k-steps, k-steps per run, row stride, row spacing
  bool rows;                           // rows copied one by one (else one bulk copy a stage)
};

__device__ __forceinline__ MmaShape mma_shape(const BProb& pr) {
  MmaShape s;
  const int d = pr.d;
  s.kd = (d + 7) >> 3;
  s.lgks = s.kd <= 8 ? 0 : s.kd <= 16 ? 1 : s.kd <= 32 ? 2 : 3;
  s.R = 256 >> s.lgks;
  s.kps = (s.kd + (1 << s.lgks) - 1) >> s.lgks;
  s.rows = d % 8 == 0;
  s.stride = s.rows ? ((d + 3) & ~7) + 4 : d;
  s.lgm = s.rows || d % 4 == 0 ? 0 : d % 2 == 0 ? 1 : 2;
  return s;
}

__device__ __forceinline__ uint32_t tf32_head(float x) { return (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u; }

__device__ __forceinline__ void mma_tf32(float (&dd)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(dd[0]), "+f"(dd[1]), "+f"(dd[2]), "+f"(dd[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void tf32_split4(const float (&a)[4], uint32_t (&h)[4], uint32_t (&l)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = tf32_head(a[i]);
    l[i] = __float_as_uint(a[i] - __uint_as_float(h[i]));
  }
}

// One FP32 chunk, rows [r0, r1) of problem pr, for the right-hand sides jl[0 .. na), na <= 8 NT:
// out[jl[x] dp + c] = sum_rows a_c (a . p) for c < d, out[kp dp + jl[x]] = sum_rows (a . p)^2.  `phase`:
// the parities of the four stage barriers (each fills by one bulk copy), kept across chunks.  Called by every
// thread of the CTA; false if a wait gave up (every copy started has then been waited for, bounded).
template <int NT>
__device__ __forceinline__ bool tm_chunk(const BProb& pr, int64_t r0, int64_t r1, double* __restrict__ out, float* smf,
                                         const int* jl, int na, uint64_t* full, uint32_t& phase) {
  constexpr int KPAD = 8 * NT;
  const int d = pr.d, dp = pr.dp, kp = pr.kp;
  const MmaShape ms = mma_shape(pr);
  const int R = ms.R, stride = ms.stride, lgm = ms.lgm, m = 1 << lgm, KS = 1 << ms.lgks, kps = ms.kps;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  float4* Pf = reinterpret_cast<float4*>(smf);                   // [kd][NT][32] fragments of P: heads, remainders
  float* Yb = smf + ms.kd * NT * 128;                            // [R][YP] Y by k-step, (head, remainder) pairs
  float* Yp = Yb + R * YP;                                       // [16 warps][16][KPAD] partial tiles
  float* stage0 = Yp + 16 * 16 * KPAD;
  const int sf = (R * stride + 8 + 31) & ~31;                    // floats of a stage
  const int NS = min(4, ((int)(TSMEM / 4) - (int)(stage0 - smf)) / sf);  // 2 to 4 stages
  const float* A = reinterpret_cast<const float*>(pr.A);
  const int64_t ld = pr.ld;
  const int nst = (int)((r1 - r0 + R - 1) / R);
  bool ok = true;
  // row-by-row copies: this thread's 4 columns of a row (from column lc) and its first row of a sweep of
  // TT / pc rows (pc <= 128 pieces a row)
  const int pc = max(1, d >> 2), lsweep = TT / pc, lrow = tid / pc, lc = (tid - lrow * pc) * 4;
  auto load_rows = [&](int64_t lo, float* buf) {
    const float* src = A + (lo + lrow) * ld + lc;
    float* dst = buf + lrow * stride + lc;
    const int left = (int)min((int64_t)R, r1 - lo);
    for (int r = lrow; r < R; r += lsweep) {
      tp_copy<4>(dst, r < left ? src : A, r < left ? 16 : 0);
      src += (int64_t)lsweep * ld;
      dst += lsweep * stride;
    }
  };
  auto load = [&](int t, int slot) {
    float* buf = stage0 + slot * sf;
    const int64_t lo = r0 + (int64_t)t * R;
    if (ms.rows) {
      if (t < nst && lrow < lsweep) load_rows(lo, buf);
      asm volatile("cp.async.commit_group;" ::: "memory");
    } else if (t < nst && tid == 0) {
      // the stage's element range rounded out to 16 bytes; where that would read past the matrix the
      // copy stops at the last 16-byte boundary and plain loads fetch the last < 4 elements
      const int64_t e_lo = lo * d, e_hi = min(r1, lo + R) * d, a_lo = e_lo & ~(int64_t)3;
      int64_t a_hi = (e_hi + 3) & ~(int64_t)3;
      if (a_hi > pr.n * d) {
        a_hi = e_hi & ~(int64_t)3;
        for (int64_t e = a_hi; e < e_hi; ++e) buf[e - a_lo] = __ldg(A + e);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier reads and writes of the slot
      const uint32_t bytes = (uint32_t)(a_hi - a_lo) * 4u;
      if (bytes) lsq_apass::ring_issue(buf, A + a_lo, bytes, full + slot);
      else asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(lsq_apass::smem_u32a(full + slot)) : "memory");
    }
  };
  for (int t = 0; t < NS - 1; ++t) load(t, t);
  // P's fragments: b0 = P[8 k + tq][8 nt + g], b1 = P[8 k + tq + 4][..], zero past d and the active
  // right-hand sides
  for (int e = warp; e < ms.kd * NT; e += TW) {
    const int x = (e % NT) * 8 + g, c = (e / NT) * 8 + tq;
    const float v0 = c < d && x < na ? pr.Pf[(int64_t)c * kp + jl[x]] : 0.f;
    const float v1 = c + 4 < d && x < na ? pr.Pf[(int64_t)(c + 4) * kp + jl[x]] : 0.f;
    const float h0 = __uint_as_float(tf32_head(v0)), h1 = __uint_as_float(tf32_head(v1));
    Pf[e * 32 + lane] = make_float4(h0, h1, v0 - h0, v1 - h1);
  }
  const int ks = warp & (KS - 1), rt = warp >> ms.lgks;
  const int k0 = ks * kps, nk = max(0, min(kps, ms.kd - k0));
  // product 1: rows ra (lanes' g) and rb of the tile: the low and high halves
  const int ra = lgm == 0 ? rt * 16 + g : ((rt >> (lgm - 1)) << (3 + lgm)) + m * g + 2 * (rt & (m / 2 - 1));
  const int rb = lgm == 0 ? ra + 8 : ra + 1;
  // the k-steps of this warp's run that lie inside d, and the columns of the one that does not
  const int nfull = nk > 0 && (k0 + nk) * 8 > d ? nk - 1 : nk, dtail = d - (ms.kd - 1) * 8;
  // product 2: tasks (column tile, share of the k-steps) warp, warp + 16, warp + 32
  const int nct = (d + 15) >> 4, K8 = R >> 3;
  int tpw = 1, rspl = 0;
  {
    int best = 1 << 30;
    for (int t = 1; t <= 3; ++t) {
      const int rs = min(16 * t / nct, K8);
      if (rs < 1) continue;
      const int cost = t * ((K8 + rs - 1) / rs);
      if (cost < best) {
        best = cost;
        tpw = t;
        rspl = rs;
      }
    }
  }
  __shared__ int shk[17];  // the shares' first k-steps
  if (tid <= rspl) shk[tid] = (K8 * tid) / rspl;
  int tshare[3], tcols[3];  // each task's share and first column
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    tshare[i] = min((warp + 16 * i) / nct, rspl - 1);
    tcols[i] = ((warp + 16 * i) % nct) * 16;
  }
  const int ntask = nct * rspl, skip = (6 * m + 2) * stride;  // to the next k-step's rows past a block's end
  float vrun[3][NT][4];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int x = 0; x < 4; ++x) vrun[i][nt][x] = 0.f;
  float qrun = 0.f;
  __syncthreads();  // the fragments of P are there
  int s = 0;  // stage t's slot
  for (int t = 0; t < nst; ++t, s = s + 1 == NS ? 0 : s + 1) {
    float* slot = stage0 + s * sf;
    const int64_t lo = r0 + (int64_t)t * R;
    const int nrows = (int)min((int64_t)R, r1 - lo);
    if (ms.rows) {
      if (NS == 2) asm volatile("cp.async.wait_group 0;" ::: "memory");
      else if (NS == 3) asm volatile("cp.async.wait_group 1;" ::: "memory");
      else asm volatile("cp.async.wait_group 2;" ::: "memory");
    } else {
      ok = lsq_apass::ring_wait(full + s, (phase >> s) & 1u);
      phase ^= 1u << s;
    }
    if (__syncthreads_or(!ok)) {  // stage t has landed; stage t - 1 and Y are no longer read
      ok = false;
      // the copies of stages t + 1 .. t + NS - 2 are still in flight: wait for them (bounded)
      if (!ms.rows)
        for (int x = t + 1; x < min(nst, t + NS - 1); ++x) {
          lsq_apass::ring_wait(full + x % NS, (phase >> (x % NS)) & 1u);
          phase ^= 1u << (x % NS);
        }
      break;
    }
    load(t + NS - 1, s == 0 ? NS - 1 : s - 1);
    const float* raw = slot + (ms.rows ? 0 : (int)((lo * d) & 3));
    if (nrows < R && !ms.rows) {  // the last stage's missing rows read as zeros
      float* z = slot + (int)((lo * d) & 3);
      for (int e = nrows * d + tid; e < R * d; e += TT) z[e] = 0.f;
      __syncthreads();
    }
    // ---- product 1
    {
      float dh[NT][4], d1[NT][4], d2[NT][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) dh[nt][i] = d1[nt][i] = d2[nt][i] = 0.f;
      const float* pa = raw + ra * stride + k0 * 8 + tq;
      const float* pb = raw + rb * stride + k0 * 8 + tq;
      const float4* pf = Pf + k0 * NT * 32 + lane;
      auto step = [&](const float (&a)[4]) {
        uint32_t ah[4], al[4];
        tf32_split4(a, ah, al);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const float4 b = pf[nt * 32];
          mma_tf32(dh[nt], ah, __float_as_uint(b.x), __float_as_uint(b.y));
          mma_tf32(d1[nt], ah, __float_as_uint(b.z), __float_as_uint(b.w));
          mma_tf32(d2[nt], al, __float_as_uint(b.x), __float_as_uint(b.y));
        }
      };
#pragma unroll 4
      for (int kk = 0; kk < nfull; ++kk) {
        const float a[4] = {pa[0], pb[0], pa[4], pb[4]};
        step(a);
        pa += 8;
        pb += 8;
        pf += NT * 32;
      }
      if (nfull < nk) {  // the last k-step: what lies past d is another row's, or nothing's
        const bool in0 = tq < dtail, in1 = tq + 4 < dtail;
        const float a[4] = {in0 ? pa[0] : 0.f, in0 ? pb[0] : 0.f, in1 ? pa[4] : 0.f, in1 ? pb[4] : 0.f};
        step(a);
      }
      float* yp = Yp + warp * 16 * KPAD;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        *reinterpret_cast<float2*>(yp + g * KPAD + nt * 8 + 2 * tq) =
            make_float2(dh[nt][0] + (d1[nt][0] + d2[nt][0]), dh[nt][1] + (d1[nt][1] + d2[nt][1]));
        *reinterpret_cast<float2*>(yp + (g + 8) * KPAD + nt * 8 + 2 * tq) =
            make_float2(dh[nt][2] + (d1[nt][2] + d2[nt][2]), dh[nt][3] + (d1[nt][3] + d2[nt][3]));
      }
    }
    __syncthreads();
    // ---- Y: the KS partial tiles in order; q; the split, stored by k-step (row pair t of step i of a
    // block of 8 m rows at 8 i + 2 t)
    {
      float qs = 0.f;
      for (int e = tid; e < R * KPAD; e += TT) {
        const int tr = e / KPAD, x = e % KPAD;             // row of the tiles (16 rt + r16)
        const float* yp = Yp + ((tr >> 4) << ms.lgks) * 16 * KPAD + (tr & 15) * KPAD + x;
        float y = yp[0];
#pragma unroll
        for (int k = 1; k < 8; ++k)
          if (k < KS) y += yp[k * 16 * KPAD];
        qs = fmaf(y, y, qs);
        int pos = tr;
        if (lgm > 0) {
          const int tl = tr >> 4;
          pos = ((tl >> (lgm - 1)) << (3 + lgm)) + ((m / 2) * (tr & 1) + (tl & (m / 2 - 1))) * 8 + (tr & 6) + ((tr >> 3) & 1);
        }
        const uint32_t h = tf32_head(y);
        *reinterpret_cast<float2*>(Yb + pos * YP + 2 * x) = make_float2(__uint_as_float(h), y - __uint_as_float(h));
      }
      qrun += qs;
    }
    __syncthreads();
    // ---- product 2
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int task = warp + 16 * i;
      if (i < tpw && task < ntask) {
        float vh[NT][4], vx[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int x = 0; x < 4; ++x) vh[nt][x] = vx[nt][x] = 0.f;
        // k-step kr: row pairs 2 m tq + 2 (kr mod m) of block kr / m; a share's k-steps are consecutive
        const int rsl = tshare[i], kb = shk[rsl], ke = shk[rsl + 1];
        const float* ar = raw + tcols[i] + g + (2 * m * tq + ((kb >> lgm) << (3 + lgm)) + 2 * (kb & (m - 1))) * stride;
        const float2* yr = reinterpret_cast<const float2*>(Yb + (kb * 8 + 2 * tq) * YP) + g;
#pragma unroll 4
        for (int kr = kb; kr < ke; ++kr) {
          const float a[4] = {ar[0], ar[8], ar[stride], ar[stride + 8]};
          ar += (kr + 1) & (m - 1) ? 2 * stride : skip;
          uint32_t ah[4], al[4];
          tf32_split4(a, ah, al);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const float2 y0 = yr[nt * 8], y1 = yr[nt * 8 + YP / 2];
            mma_tf32(vh[nt], ah, __float_as_uint(y0.x), __float_as_uint(y1.x));
            mma_tf32(vx[nt], ah, __float_as_uint(y0.y), __float_as_uint(y1.y));
            mma_tf32(vx[nt], al, __float_as_uint(y0.x), __float_as_uint(y1.x));
          }
          yr += 4 * YP;
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int x = 0; x < 4; ++x) vrun[i][nt][x] += vh[nt][x] + vx[nt][x];
      }
    }
  }
  if (ms.rows) asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();  // the stages are free for the reduction
  if (!ok) return false;
  // ---- V: the row shares in FP64, [rspl][KPAD][16 nct]
  double* red = reinterpret_cast<double*>(stage0);
  const int cp = 16 * nct;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int task = warp + 16 * i;
    if (i < tpw && task < ntask) {
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        double* o = red + (size_t)(tshare[i] * KPAD + nt * 8 + 2 * tq) * cp + tcols[i] + g;
        o[0] = (double)vrun[i][nt][0];
        o[cp] = (double)vrun[i][nt][1];
        o[8] = (double)vrun[i][nt][2];
        o[cp + 8] = (double)vrun[i][nt][3];
      }
    }
  }
  float* qf = Yp;  // q: thread tid summed right-hand side tid % KPAD
  qf[tid] = qrun;
  __syncthreads();
  for (int e = tid; e < na * d; e += TT) {
    const int x = e / d, c = e - x * d;
    double sum = 0.0;
    for (int q = 0; q < rspl; ++q) sum += red[(size_t)(q * KPAD + x) * cp + c];
    out[(size_t)jl[x] * dp + c] = sum;
  }
  if (tid < na) {
    double sum = 0.0;
    for (int y = tid; y < TT; y += KPAD) sum += (double)qf[y];
    out[(size_t)kp * dp + jl[tid]] = sum;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the next chunk's bulk copies come after this
  __syncthreads();
  return true;
}

// The pass: CTAs take chunks from the iteration's queue (costliest first), as bpass_kernel does.
__global__ void __launch_bounds__(TT, 1) btile_kernel(BatchArgs a, int force_exact) {
  extern __shared__ __align__(128) float tsm[];
  __shared__ __align__(8) uint64_t full[4];
  __shared__ int next, nact, jl[KPMAX];
  if (threadIdx.x == 0) {
    for (int s = 0; s < 4; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(lsq_apass::smem_u32a(full + s)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  uint32_t phase = 0u;
  const int it = *(volatile int*)a.iter;
  int* head = a.qhead + it % 3;
  for (;;) {
    if (threadIdx.x == 0) next = atomicAdd(head, 1);
    __syncthreads();
    const int unit = next;
    if (unit >= a.nchunks) break;
    const int ch = a.order[unit];
    const int4 cd = a.chunks[ch];
    const BProb& pr = a.probs[cd.x];
    if (threadIdx.x == 0) {  // the active right-hand sides, in order
      int n = 0;
      if (prob_active(pr, it))
        for (int j = 0; j < pr.k; ++j)
          if (pr.flags[(it & 1) * pr.kp + j] & F_ACTIVE) jl[n++] = j;
      nact = n;
    }
    __syncthreads();
    const int n = nact;
    if (n == 0) continue;
    double* out = a.part + a.part_off[ch];
    if (force_exact != 0 || exact_step(pr, it)) {
      for (int j = 0; j < n; j += 8) {
        if (n - j > 4) tp_chunk<8>(pr, cd.y, cd.z, out, tsm, jl + j, min(8, n - j));
        else tp_chunk<4>(pr, cd.y, cd.z, out, tsm, jl + j, n - j);
      }
    } else {
      const bool ok = n > 8 ? tm_chunk<2>(pr, cd.y, cd.z, out, tsm, jl, n, full, phase)
                            : tm_chunk<1>(pr, cd.y, cd.z, out, tsm, jl, n, full, phase);
      if (!ok) {
        if (threadIdx.x == 0) atomicCAS(a.err, 0, (int)LSQ_ERR_TIMEOUT);
        break;
      }
    }
  }
}
