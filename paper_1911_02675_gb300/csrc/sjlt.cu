// sjlt.cu -- the SJLT (Section 2, last paragraph) in FP32 arithmetic: SA = S A with s entries
// +-1/sqrt(s) per column of S, for one matrix or for many at once, and the hash pass of the other
// SJLT sketches.
//
// S A is a sum over the rows of A: row i is added, signed, to s rows of SA.  Scattering them with
// shared-memory additions runs at ~3.4 additions per clock per SM whatever the shape.  Here the
// sum is turned round: for each chunk of up to 2048 rows one CTA first sorts the chunk's (row,
// sign) entries by target row of SA (lists_kernel; all column tiles use the lists), then each
// target row gathers its entries (gather_kernel), so the sums stay in registers and run in a
// fixed order (the sketch repeats bit for bit).  A partial sum per (group of chunks, target) and
// a reduction over the groups in double-FP32 give SA.
#include <math.h>

#include <algorithm>
#include <vector>

#include <cuda_bf16.h>

#include "apass.cuh"
#include "common.cuh"

namespace {

// The s target rows of data row i in SJLT instance t: Lemire's bounded integers in [0, m) from the
// successive words of Philox(i, draw, t, TAG_SJLT), duplicates skipped (at most 4096 draws).
template <int SMAX>
__device__ __forceinline__ void sjlt_targets(uint64_t seed, int64_t i, uint32_t t, int m, int s,
                                             int32_t (&picked)[SMAX]) {
  const uint32_t range = (uint32_t)m;
  const uint32_t threshold = (uint32_t)(0u - range) % range;
  int got = 0;
  if constexpr (SMAX <= 8) {
    // every index static, so that the picks stay in registers (unused places hold -1)
#pragma unroll
    for (int q = 0; q < SMAX; ++q) picked[q] = -1;
    for (uint32_t draw = 0; got < s && draw < 4096u; ++draw) {
      const uint4 w = philox_at(seed, (uint32_t)i, draw, t, TAG_SJLT);
      const uint32_t words[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int32_t v = (int32_t)__umulhi(words[k], range);
        bool take = got < s && words[k] * range >= threshold;
#pragma unroll
        for (int q = 0; q < SMAX; ++q) take = take && picked[q] != v;
#pragma unroll
        for (int q = 0; q < SMAX; ++q) picked[q] = take && q == got ? v : picked[q];
        got += take ? 1 : 0;
      }
    }
#pragma unroll
    for (int q = 0; q < SMAX; ++q) picked[q] = max(picked[q], 0);  // every index in range
  } else {
    for (uint32_t draw = 0; got < s && draw < 4096u; ++draw) {
      const uint4 w = philox_at(seed, (uint32_t)i, draw, t, TAG_SJLT);
      const uint32_t words[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (got >= s) break;
        const unsigned long long prod = (unsigned long long)words[k] * range;
        const uint32_t low = (uint32_t)prod;
        if (low < range && low < threshold) continue;
        const int32_t v = (int32_t)(prod >> 32);
        bool dup = false;
        for (int q = 0; q < got; ++q) dup |= (picked[q] == v);
        if (!dup) picked[got++] = v;
      }
    }
    for (int k = got; k < SMAX; ++k) picked[k] = 0;  // unreachable for s <= m; keeps every index in range
  }
}

__global__ void sjlt_hash_kernel(int64_t n, int m, int s, uint64_t seed, uint32_t t, int32_t* __restrict__ h,
                                 uint32_t* __restrict__ signs, int64_t grow0) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t picked[32];
    sjlt_targets<32>(seed, i + grow0, t, m, s, picked);  // column i + grow0 of S
    for (int k = 0; k < s; ++k) h[i * s + k] = picked[k];
    signs[i] = philox_at(seed, (uint32_t)(i + grow0), 0u, t, TAG_SJLT_SIGN).x;
  }
}

constexpr int GT = 512;             // threads of both kernels
constexpr int G_QUADS = 4096;       // 4-column pieces of rows in a chunk of a gather tile
constexpr int G_ENTRIES = 16384;    // most entries of a chunk (rows x s)
constexpr int G_MT = 16;            // most target rows per thread group
constexpr size_t G_LIST_SMEM = 221 * 1024;  // shared memory the list kernel may take

// target rows of a grid.z slice with L threads per target
__host__ __device__ constexpr int slice_of(int L) { return G_MT * (GT / L); }

// entries of a chunk's list with its padding, and its pitch
__host__ __device__ constexpr int list_pitch(int m, int R, int s) { return (R * s + m + 7) & ~7; }

// one sketch; L threads gather a target row (4 L columns a tile), R rows per chunk, the entries of
// chunk k at list + k list_pitch, the offsets of its targets (in pairs of entries) at offs + k pitch
// (m + 1 of them), cpg chunks per group, its partial sums [group][m][d]
struct SjltJob {
  const void* A;
  int64_t n, ld, grow0;
  float* part;
  uint16_t* list;
  uint16_t* offs;
  int dtype, d, m, s, L, R, nchunk, cpg, pitch, vec, bf16;
  uint32_t t;
  double scale;  // 1 / sqrt(s)
};

// ------------------------------------------------------------------------------------
// One chunk's entries (row of the chunk, bit 15: negative) sorted by target row, by row within a
// target, each target's run padded to an even length with the entry R (a row of zeros), so that
// the gather reads entries two at a time: counts and placement with shared-memory integer
// atomics (16-bit counters, two to a word), then each target's few entries are put in order (a
// thread per target; a warp for the long lists of a small m).  offs[e] counts pairs.
// ------------------------------------------------------------------------------------
template <int SMAX>
__global__ void __launch_bounds__(GT) sjlt_lists_kernel(const SjltJob* __restrict__ jobs,
                                                        const __grid_constant__ SjltJob one,
                                                        const int2* __restrict__ items, uint64_t seed) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t wsum[GT / 32];
  const int2 it = items ? items[blockIdx.x] : make_int2(0, (int)blockIdx.x);
  const SjltJob jb = jobs ? jobs[it.x] : one;
  const int m = jb.m, s = jb.s, R = jb.R;
  uint32_t* cnt2 = reinterpret_cast<uint32_t*>(smem_raw);         // [m] 16-bit counts, then positions
  uint16_t* cnt = reinterpret_cast<uint16_t*>(cnt2);
  uint16_t* ent = cnt + ((m + 1) & ~1);                           // [entries]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t row0 = (int64_t)it.y * R;
  const int rows = (int)min((int64_t)R, jb.n - row0);
  for (int e = tid; e < (m + 1) / 2; e += GT) cnt2[e] = 0u;
  __syncthreads();
  auto bump = [&](int t) -> uint32_t {  // the count (position) of target t before adding one
    const int sh = 16 * (t & 1);
    return (atomicAdd(&cnt2[t >> 1], 1u << sh) >> sh) & 0xFFFFu;
  };
  int32_t tg[SMAX];
  for (int r = tid; r < rows; r += GT) {
    sjlt_targets<SMAX>(seed, row0 + r + jb.grow0, jb.t, m, s, tg);
#pragma unroll
    for (int k = 0; k < SMAX; ++k)
      if (k < s) bump(tg[k]);
  }
  __syncthreads();
  // exclusive scan of the padded counts: thread t owns an even run of them
  const int per = ((m + GT - 1) / GT + 1) & ~1;
  const int e0 = min(m, tid * per), e1 = min(m, e0 + per);
  uint32_t mine = 0;
  for (int e = e0; e < e1; ++e) mine += (cnt[e] + 1u) & ~1u;
  uint32_t inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  uint32_t base = inc - mine;
  for (int w = 0; w < warp; ++w) base += wsum[w];
  uint16_t* offs = jb.offs + (int64_t)it.y * jb.pitch;
  for (int e = e0; e < e1; ++e) {
    const uint32_t c = cnt[e];
    cnt[e] = (uint16_t)base;
    offs[e] = (uint16_t)(base >> 1);
    base += (c + 1u) & ~1u;
    if (e == m - 1) offs[m] = (uint16_t)(base >> 1);
  }
  __syncthreads();
  for (int r = tid; r < rows; r += GT) {
    // (a chunk of at most GT rows: the thread's one row is still in registers)
    if (rows > GT) sjlt_targets<SMAX>(seed, row0 + r + jb.grow0, jb.t, m, s, tg);
    const uint32_t sw = philox_at(seed, (uint32_t)(row0 + r + jb.grow0), 0u, jb.t, TAG_SJLT_SIGN).x;
#pragma unroll
    for (int k = 0; k < SMAX; ++k)
      if (k < s) ent[bump(tg[k])] = (uint16_t)(r | (((sw >> k) & 1u) << 15));
  }
  __syncthreads();
  // cnt[e] is now the end of target e's entries, which start at the end of target e - 1, rounded up
  uint16_t* out = jb.list + (int64_t)it.y * list_pitch(jb.m, R, s);
  constexpr int SHORT = 24;
  for (int e = tid; e < m; e += GT) {
    const int b = e ? (cnt[e - 1] + 1) & ~1 : 0, n_e = (int)cnt[e] - b;
    if (n_e & 1) out[b + n_e] = (uint16_t)R;
    if (n_e > SHORT) continue;
    for (int i = 1; i < n_e; ++i) {
      const uint16_t x = ent[b + i];
      int j = i;
      for (; j > 0 && (ent[b + j - 1] & 0x7FFFu) > (x & 0x7FFFu); --j) ent[b + j] = ent[b + j - 1];
      ent[b + j] = x;
    }
    for (int i = 0; i < n_e; ++i) out[b + i] = ent[b + i];
  }
  // long lists: an entry's place is the number of entries of its target with a smaller row
  for (int e = warp; e < m; e += GT / 32) {
    const int b = e ? (cnt[e - 1] + 1) & ~1 : 0, n_e = (int)cnt[e] - b;
    if (n_e <= SHORT) continue;
    for (int i0 = 0; i0 < n_e; i0 += 32) {
      const uint32_t x = i0 + lane < n_e ? ent[b + i0 + lane] : 0xFFFFu;
      int rank = 0;
      for (int j = 0; j < n_e; ++j) rank += (ent[b + j] & 0x7FFFu) < (x & 0x7FFFu) ? 1 : 0;
      if (i0 + lane < n_e) out[b + rank] = (uint16_t)x;
    }
  }
}

// ------------------------------------------------------------------------------------
// The gather.  A CTA owns 4 L columns, a range of chunks and a slice of target rows.  A chunk's
// 4096 / L rows sit in shared memory as FP32 (two buffers: the next chunk's rows are loaded,
// narrowed and stored between the targets of the current one, so that no thread waits for
// them); its lists are copied in with cp.async.  L threads take the target rows slot,
// slot + GT / L, ... (MT of them): per entry one 16-byte read of the row and four additions each;
// the chunk's sum is then added to the target's registers, which keeps the FP32 chains short.
// With few targets several slots share a target's entries and their sums are added at the end.
// Bound by shared memory (random rows: conflicts of 16-byte reads fall as the rows widen, 2.1
// ways at 32 bytes, 1.5 at 64, none at 128) and by the steps of the longest list of a warp, so a
// tile is as wide as the registers of its target sums allow: 32 columns up to m = 1024, 16 up to
// 2048, 8 above (slices of 4096).  Measured, whole sketch of 2^20 x 512 FP64, m = 2048, s = 8:
// 6.54 ms with shared-memory additions, 2.97 ms gathered in 8-column tiles, 2.37 ms so.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// BF16 sketches: an element of A rounded to FP32, then to BF16 (nearest, ties to even)
__device__ __forceinline__ float round_bf16(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// 4 columns of one row as loaded
struct RawQuad {
  uint4 a, b;  // FP32: a; FP64: a, b
};

__device__ __forceinline__ RawQuad quad_load(const SjltJob& jb, int64_t row, int c) {
  RawQuad q;
  q.a = q.b = make_uint4(0u, 0u, 0u, 0u);
  if (jb.dtype == LSQ_F64) {
    const double* p = reinterpret_cast<const double*>(jb.A) + row * jb.ld + c;
    if (jb.vec && c + 4 <= jb.d) {
      q.a = __ldg(reinterpret_cast<const uint4*>(p));
      q.b = __ldg(reinterpret_cast<const uint4*>(p) + 1);
    } else {
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = c + k < jb.d ? __ldg(p + k) : 0.0;
      q.a = make_uint4(__double2loint(v[0]), __double2hiint(v[0]), __double2loint(v[1]), __double2hiint(v[1]));
      q.b = make_uint4(__double2loint(v[2]), __double2hiint(v[2]), __double2loint(v[3]), __double2hiint(v[3]));
    }
  } else {
    const float* p = reinterpret_cast<const float*>(jb.A) + row * jb.ld + c;
    if (jb.vec && c + 4 <= jb.d) {
      q.a = __ldg(reinterpret_cast<const uint4*>(p));
    } else {
      float v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = c + k < jb.d ? __ldg(p + k) : 0.f;
      q.a = make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
    }
  }
  return q;
}

__device__ __forceinline__ float4 quad_narrow(const SjltJob& jb, const RawQuad& q) {
  float4 v;
  if (jb.dtype == LSQ_F64) {
    using lsq_apass::narrow_f32;
    v = make_float4(narrow_f32(__hiloint2double((int)q.a.y, (int)q.a.x)), narrow_f32(__hiloint2double((int)q.a.w, (int)q.a.z)),
                    narrow_f32(__hiloint2double((int)q.b.y, (int)q.b.x)), narrow_f32(__hiloint2double((int)q.b.w, (int)q.b.z)));
  } else {
    v = make_float4(__uint_as_float(q.a.x), __uint_as_float(q.a.y), __uint_as_float(q.a.z), __uint_as_float(q.a.w));
  }
  if (jb.bf16) v = make_float4(round_bf16(v.x), round_bf16(v.y), round_bf16(v.z), round_bf16(v.w));
  return v;
}

// a += v sg with sg = +-1 (exact products: one rounding, as an addition)
__device__ __forceinline__ void add_signed(float4& a, const float4& v, float sg) {
  a.x = fmaf(v.x, sg, a.x);
  a.y = fmaf(v.y, sg, a.y);
  a.z = fmaf(v.z, sg, a.z);
  a.w = fmaf(v.w, sg, a.w);
}

template <int L, int MT>
__device__ __forceinline__ void gather_body(const SjltJob& jb, int tile, int group, int slice, unsigned char* smem) {
  constexpr int SLOTS = GT / L, SLICE = slice_of(L);
  constexpr int NU = G_QUADS / GT;           // quads of a chunk per thread: 8
  constexpr int NG = MT < 4 ? MT : 4;        // groups of them, one after another through the targets
  constexpr int NB = NU / NG;                // quads in flight per thread
  constexpr int SPG = MT / NG;               // targets per group
  const int R = jb.R, m = jb.m;
  const int tid = threadIdx.x, col = tid & (L - 1), slot = tid / L;
  float4* Z = reinterpret_cast<float4*>(smem);                              // [2][R + 1][L], row R zero
  uint16_t* list = reinterpret_cast<uint16_t*>(Z + (size_t)2 * (R + 1) * L);  // [2][lpitch]
  const int lpitch = list_pitch(min(m, SLICE), R, jb.s) + 8;
  uint16_t* offs = list + 2 * lpitch;                                       // [2][pitch of the slice]
  const int c0 = tile * 4 * L;
  const int t0 = slice * SLICE, mt = min(m - t0, SLICE);                    // targets of the slice
  const int opitch = ((min(m, SLICE) + 1 + 7) & ~7) + 8;
  // with few targets, 2^lgp slots each take a piece of a target's entries
  int lgp = 0;
  if (MT == 1)
    while ((mt << (lgp + 1)) <= SLOTS) ++lgp;
  const int target0 = MT == 1 ? slot >> lgp : slot;
  const int part = MT == 1 ? slot & ((1 << lgp) - 1) : 0;
  const int k_begin = group * jb.cpg, k_end = min(jb.nchunk, k_begin + jb.cpg);
  // the slice's part of a chunk's list, from the multiple of 8 entries before it; its first entry
  // (of two, by buffer) is what the target offsets count from
  int first0 = 0, first1 = 0;
  auto copy_lists = [&](int k, int b) {
    const uint16_t* go = jb.offs + (int64_t)k * jb.pitch + t0;
    int from = 0, to = list_pitch(m, R, jb.s);
    if (m > SLICE) {
      from = (2 * (int)__ldg(go)) & ~7;
      to = 2 * (int)__ldg(go + mt);
    }
    if (b) first1 = from;
    else first0 = from;
    const uint16_t* gl = jb.list + (int64_t)k * list_pitch(m, R, jb.s);
    for (int e = from + 8 * tid; e < to; e += 8 * GT) cp_async16(list + b * lpitch + e - from, gl + e);
    for (int e = 8 * tid; e < mt + 1; e += 8 * GT) cp_async16(offs + b * opitch + e, go + e);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // quad u of this thread: row (tid + GT u) / L of the chunk, column quad tid mod L
  auto load_quad = [&](int k, int u) -> RawQuad {
    const int r = slot + SLOTS * u;
    const int64_t row = (int64_t)k * R + r;
    if (k < k_end && r < R && row < jb.n) return quad_load(jb, row, c0 + 4 * col);
    return RawQuad{make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
  };
  auto store_quad = [&](int b, int u, const RawQuad& q) {
    if (slot + SLOTS * u < R) Z[(size_t)b * (R + 1) * L + tid + GT * u] = quad_narrow(jb, q);
  };
  float4 acc[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid < 2 * L) Z[((size_t)(tid / L) * (R + 1) + R) * L + col] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (k_begin < k_end) {
    copy_lists(k_begin, 0);
#pragma unroll
    for (int g = 0; g < NU; g += 4) {
      RawQuad q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = load_quad(k_begin, g + u);
#pragma unroll
      for (int u = 0; u < 4; ++u) store_quad(0, g + u, q[u]);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  __syncthreads();
  for (int k = k_begin; k < k_end; ++k) {
    const int b = (k - k_begin) & 1;
    if (k + 1 < k_end) copy_lists(k + 1, b ^ 1);
    const uint32_t* lst = reinterpret_cast<const uint32_t*>(list + b * lpitch - (b ? first1 : first0));
    const uint16_t* off = offs + b * opitch;
    const float4* z = Z + (size_t)b * (R + 1) * L + col;
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      RawQuad q[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) q[u] = load_quad(k + 1, g * NB + u);
#pragma unroll
      for (int i = g * SPG; i < (g + 1) * SPG; ++i) {
        const int t = target0 + SLOTS * i;
        int e = (b ? first1 : first0) >> 1, end = e;  // (an empty run inside the buffer)
        if (t < mt) {
          e = off[t];
          end = off[t + 1];
          if (MT == 1 && lgp) {
            const int len = end - e;
            end = e + ((len * (part + 1)) >> lgp);
            e += (len * part) >> lgp;
          }
        }
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t x = lst[e];  // two entries; the next two are read a step ahead (inside the buffer)
        while (e < end) {
          const uint32_t x1 = lst[++e];
          const float4 v0 = z[L * (x & 0xFFFu)], v1 = z[L * ((x >> 16) & 0xFFFu)];
          add_signed(sum, v0, __uint_as_float(((x << 16) & 0x80000000u) | 0x3F800000u));
          add_signed(sum, v1, __uint_as_float((x & 0x80000000u) | 0x3F800000u));
          x = x1;
        }
        acc[i].x += sum.x;
        acc[i].y += sum.y;
        acc[i].z += sum.z;
        acc[i].w += sum.w;
      }
#pragma unroll
      for (int u = 0; u < NB; ++u) store_quad(b ^ 1, g * NB + u, q[u]);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // the next chunk is complete, and this one is no longer read
  }
  if (MT == 1 && lgp) {
    // the parts of a target in order (Z is free)
    Z[tid] = acc[0];
    __syncthreads();
    if (part == 0)
      for (int p = 1; p < (1 << lgp); ++p) {
        const float4 v = Z[tid + L * p];
        acc[0].x += v.x;
        acc[0].y += v.y;
        acc[0].z += v.z;
        acc[0].w += v.w;
      }
  }
  if (part == 0) {
    float* out = jb.part + (int64_t)group * m * jb.d;
    const int c = c0 + 4 * col;
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      const int t = target0 + SLOTS * i;
      if (t >= mt) continue;
      const float v[4] = {acc[i].x, acc[i].y, acc[i].z, acc[i].w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c + j < jb.d) out[(int64_t)(t0 + t) * jb.d + c + j] = v[j];
    }
  }
}

// one CTA per (job, column tile, group, slice)
__global__ void __launch_bounds__(GT, 1) sjlt_gather_kernel(const SjltJob* __restrict__ jobs,
                                                            const __grid_constant__ SjltJob one,
                                                            const int4* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int4 it = items ? items[blockIdx.x] : make_int4(0, (int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z);
  const SjltJob jb = jobs ? jobs[it.x] : one;
  const int L = jb.L, mt = min(jb.m - it.w * slice_of(L), slice_of(L)), per = (mt * L + GT - 1) / GT;
#define GATHER(L_, MT_) gather_body<L_, MT_>(jb, it.y, it.z, it.w, smem_raw)
  if (L == 8) {
    if (per <= 1) GATHER(8, 1);
    else if (per <= 2) GATHER(8, 2);
    else if (per <= 4) GATHER(8, 4);
    else if (per <= 8) GATHER(8, 8);
    else GATHER(8, 16);
  } else if (L == 4) {
    if (per <= 1) GATHER(4, 1);
    else if (per <= 4) GATHER(4, 4);
    else GATHER(4, 16);
  } else {
    if (per <= 1) GATHER(2, 1);
    else if (per <= 4) GATHER(2, 4);
    else GATHER(2, 16);
  }
#undef GATHER
}

// SA_p = scale_p * sum over the groups of problem p's partials (double-FP32 sums), one launch;
// element e of the concatenation belongs to the problem whose prefix range holds it
__global__ void sjlt_reduce_kernel(const SjltJob* __restrict__ jobs, const __grid_constant__ SjltJob one,
                                   const int64_t* __restrict__ prefix, double* const* __restrict__ SA,
                                   double* __restrict__ SA_one, int nprob, int64_t total) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = nprob - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (prefix[mid] <= e) lo = mid;
      else hi = mid - 1;
    }
    const SjltJob& jb = jobs ? jobs[lo] : one;
    const int64_t md = (int64_t)jb.m * jb.d, k = jobs ? e - prefix[lo] : e;
    const int groups = (jb.nchunk + jb.cpg - 1) / jb.cpg;
    float h = 0.f, t = 0.f;
    for (int g = 0; g < groups; ++g) lsq_apass::df_add(h, t, jb.part[(int64_t)g * md + k], 0.f);
    (jobs ? SA[lo] : SA_one)[k] = ((double)h + (double)t) * jb.scale;
  }
}

// ------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------
size_t lists_smem(int m, int R, int s) { return ((size_t)m + 1 + list_pitch(m, R, s)) * 2; }

size_t gather_smem(const SjltJob& jb) {
  const int ms = std::min(jb.m, slice_of(jb.L));
  const size_t opitch = (((size_t)ms + 1 + 7) & ~(size_t)7) + 8;
  return (size_t)2 * (jb.R + 1) * jb.L * 16 + 2 * ((size_t)list_pitch(ms, jb.R, jb.s) + 8 + opitch) * 2;
}

// the fields of a job that follow from the matrix and the sketch (part, list, offs and cpg are the
// caller's)
SjltJob make_job(const lsq_matrix& a, int m, int s, uint32_t t, int64_t grow0, bool bf16) {
  SjltJob jb = {};
  const size_t es = a.dtype == LSQ_F64 ? 8 : 4;
  jb.A = a.data;
  jb.n = a.n;
  jb.ld = a.ld;
  jb.grow0 = grow0;
  jb.dtype = a.dtype;
  jb.d = (int)a.d;
  jb.m = m;
  jb.s = s;
  // the widest tile whose target sums fit the registers in one slice, no wider than A
  jb.L = m <= slice_of(8) ? 8 : m <= slice_of(4) ? 4 : 2;
  while (jb.L > 2 && 2 * jb.L >= jb.d) jb.L >>= 1;
  // a chunk's rows fill a buffer; fewer where s or m is large (the entries and the counts share the
  // list kernel's shared memory), multiples of 64 so that every chunk's lists are 16-byte aligned
  jb.R = G_QUADS / jb.L;
  while (jb.R > 64 && (jb.R * s > G_ENTRIES || lists_smem(m, jb.R, s) > G_LIST_SMEM)) jb.R >>= 1;
  jb.nchunk = (int)((a.n + jb.R - 1) / jb.R);
  jb.cpg = jb.nchunk;
  jb.pitch = ((m + 1 + 7) & ~7) + 8;  // 16-byte aligned; room for the copies' last vector
  jb.vec = (((uintptr_t)a.data % 16) == 0 && ((size_t)a.ld * es) % 16 == 0) ? 1 : 0;
  jb.bf16 = bf16 ? 1 : 0;
  jb.t = t;
  jb.scale = 1.0 / sqrt((double)s);
  return jb;
}

size_t list_elems(const SjltJob& jb) { return (size_t)jb.nchunk * list_pitch(jb.m, jb.R, jb.s); }
size_t offs_elems(const SjltJob& jb) { return (size_t)jb.nchunk * jb.pitch; }

lsq_status launch_lists(lsq_ctx* ctx, const SjltJob* jobs, const SjltJob& one, const int2* items, unsigned nitems,
                        int smax, size_t smem, uint64_t seed) {
  auto run = [&](auto kern) -> lsq_status {
    LSQ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<nitems, GT, smem, ctx->stream>>>(jobs, one, items, seed);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
  };
  return smax <= 8 ? run(sjlt_lists_kernel<8>) : run(sjlt_lists_kernel<32>);
}

}  // namespace

// the hash pass of the other SJLT sketches (target rows in draw order and the sign word of every
// row of A)
lsq_status lsq_sjlt_hash_launch(lsq_ctx* ctx, int64_t n, int m, int s, uint64_t seed, uint32_t t, int64_t grow0,
                                int32_t* h, uint32_t* signs) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 16 * (int64_t)ctx->sm_count));
  sjlt_hash_kernel<<<grid, 256, 0, ctx->stream>>>(n, m, s, seed, t, h, signs, grow0);
  LSQ_LAUNCH_CHECK();
  return LSQ_OK;
}

// Whether one matrix is gathered (else the scatter of sketch.cu).  The gather adds in registers, but sorts
// n s entries and visits m targets a chunk, whatever d is: it wants many additions for its targets,
// s n d >= 12 m^2, no more than 4096 sqrt(s) targets (every slice of 4096 reads A again, and a row's lists grow
// with m / R) and more columns than a tile's 16, unless s is large or a wide chunk has few targets.  Embeddings
// of 8 d rows at most are gathered at any n: up to 8192 rows the lists cost them 10 to 30 us, with half
// the error.  Measured over 2400 sizes (n 2^11..2^20, d 4..1000, m 16..51200, s 1..32), scatter against
// gather: 2^20 x 512 FP64, m = 2048, s = 8, 6.54 and 2.37 ms; 2^18 x 512, m = 16384, 2.45 and 2.56;
// m = 51200, 3.40 and 9.03; 2^18 x 64, m = 51200, 0.87 and 1.75; 2^20 x 4, m = 16, 0.40 and 2.1;
// 32768 x 4, m = 1024, 32 and 53 us; 8192 x 100, m = 8192, 42 and 112 us.
bool lsq_sjlt_gathers(int64_t n, int d, int m, int s) {
  if (d > 16 && s >= 4 && m <= 8 * d && m <= 4096) return true;
  const double mm = (double)m * m, adds = (double)s * n * d;
  if (mm > 16777216.0 * s) return false;
  if (s > 16) return 4.0 * mm <= adds && m >= 4 * s;
  if ((s < 4 ? 24.0 : 12.0) * mm > adds || adds < 4194304.0) return false;
  return d > 16 || (d > 8 && n >= (1 << 19) && m >= 8 * s && m <= 1024);
}

// SA (m x d FP64) of one matrix; m <= 51200 (the list kernel's counts)
lsq_status lsq_sjlt_f32(lsq_ctx* ctx, const lsq_matrix* A, int m, int s, uint64_t seed, uint32_t t, double* SA,
                        int64_t grow0) {
  if ((size_t)m * 4 > 200 * 1024) return LSQ_ERR_ARG;
  SjltJob jb = make_job(*A, m, s, t, grow0, false);
  const int d = (int)A->d;
  const int tiles = lsq_ceil_div(d, 4 * jb.L), slices = lsq_ceil_div(m, slice_of(jb.L));
  // whole waves of one CTA per SM; at most 256 MB of partial sums
  const int64_t cap = std::max<int64_t>(1, ((int64_t)256 << 20) / ((int64_t)m * d * 4));
  int64_t groups = 1;
  double best = 1e300;
  for (int64_t g = 1; g <= std::min<int64_t>(std::min<int64_t>(jb.nchunk, cap), 64); ++g) {
    const int64_t cpg = (jb.nchunk + g - 1) / g;
    const double cost = (double)(((int64_t)tiles * slices * g + ctx->sm_count - 1) / ctx->sm_count) * ((double)cpg + 0.5);
    if (cost < best * (1.0 - 1e-9)) {
      best = cost;
      groups = g;
    }
  }
  jb.cpg = (int)((jb.nchunk + groups - 1) / groups);
  groups = (jb.nchunk + jb.cpg - 1) / jb.cpg;
  const int64_t md = (int64_t)m * d;
  const size_t need = lsq_align256(list_elems(jb) * 2) + lsq_align256(offs_elems(jb) * 2) +
                      lsq_align256((size_t)groups * md * 4);
  lsq_status st = lsq_ensure_scratch(ctx, need);
  if (st != LSQ_OK) return st;
  Carver cv{reinterpret_cast<char*>(ctx->scratch), 0};
  jb.list = cv.take<uint16_t>(list_elems(jb));
  jb.offs = cv.take<uint16_t>(offs_elems(jb));
  jb.part = cv.take<float>((size_t)groups * md);
  st = launch_lists(ctx, nullptr, jb, nullptr, (unsigned)jb.nchunk, s, lists_smem(m, jb.R, s), seed);
  if (st != LSQ_OK) return st;
  const size_t smem = gather_smem(jb);
  LSQ_CUDA_TRY(cudaFuncSetAttribute(sjlt_gather_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  sjlt_gather_kernel<<<dim3(tiles, (unsigned)groups, slices), GT, smem, ctx->stream>>>(nullptr, jb, nullptr);
  LSQ_LAUNCH_CHECK();
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((md + 255) / 256, 4 * (int64_t)ctx->sm_count));
  sjlt_reduce_kernel<<<grid, 256, 0, ctx->stream>>>(nullptr, jb, nullptr, nullptr, SA, 1, md);
  LSQ_LAUNCH_CHECK();
  return LSQ_OK;
}

// Sketches of many problems in three launches (lists, gather, reduction): problem p draws
// instance t = p of `seed` into SA[p] (m[p] x d FP64), exactly the embedding lsq_sketch would
// draw, over BF16-rounded A where bf16 is set.
lsq_status lsq_sjlt_batched(lsq_ctx* ctx, int nprob, const lsq_matrix* A, const int* m, int s, uint64_t seed,
                            double* const* SA, int bf16) {
  if (nprob <= 0) return LSQ_OK;
  std::vector<SjltJob> jobs(nprob);
  std::vector<int4> items;
  std::vector<int2> chunks;
  std::vector<int64_t> prefix(nprob);
  int64_t total = 0;
  size_t part_elems = 0, lists = 0, offs = 0, smem_l = 0, smem_g = 0;
  for (int p = 0; p < nprob; ++p) {
    const int sp = std::min(s, m[p]);
    if ((size_t)m[p] * 32 > 200 * 1024 || sp < 1 || sp > 32) return LSQ_ERR_ARG;
    SjltJob& jb = jobs[p];
    jb = make_job(A[p], m[p], sp, (uint32_t)p, 0, bf16 != 0);
    // about 16k rows per work item, at most 64 groups
    const int64_t g = std::max<int64_t>(1, std::min<int64_t>(64, (A[p].n + 16383) / 16384));
    jb.cpg = (int)((jb.nchunk + g - 1) / g);
    const int groups = (jb.nchunk + jb.cpg - 1) / jb.cpg;
    prefix[p] = total;
    total += (int64_t)jb.m * jb.d;
    part_elems += (size_t)groups * jb.m * jb.d;
    lists += (list_elems(jb) + 7) & ~(size_t)7;
    offs += offs_elems(jb);
    smem_l = std::max(smem_l, lists_smem(jb.m, jb.R, sp));
    smem_g = std::max(smem_g, gather_smem(jb));
    for (int sl = 0; sl < lsq_ceil_div(jb.m, slice_of(jb.L)); ++sl)
      for (int ct = 0; ct < lsq_ceil_div(jb.d, 4 * jb.L); ++ct)
        for (int gg = 0; gg < groups; ++gg) items.push_back(make_int4(p, ct, gg, sl));
    for (int k = 0; k < jb.nchunk; ++k) chunks.push_back(make_int2(p, k));
  }
  // the costliest items first (chunks of the group)
  std::stable_sort(items.begin(), items.end(), [&](const int4& x, const int4& y) {
    auto cost = [&](const int4& i) {
      const SjltJob& jb = jobs[i.x];
      return std::min(jb.cpg, jb.nchunk - i.z * jb.cpg) * jb.R;
    };
    return cost(x) > cost(y);
  });
  const size_t need = lsq_align256(part_elems * 4) + lsq_align256(lists * 2) + lsq_align256(offs * 2) +
                      lsq_align256(nprob * sizeof(SjltJob)) + lsq_align256(items.size() * sizeof(int4)) +
                      lsq_align256(chunks.size() * sizeof(int2)) + lsq_align256(nprob * 8) +
                      lsq_align256(nprob * sizeof(double*));
  lsq_status st = lsq_ensure_scratch(ctx, need);
  if (st != LSQ_OK) return st;
  Carver cv{reinterpret_cast<char*>(ctx->scratch), 0};
  float* part = cv.take<float>(part_elems);
  uint16_t* d_lists = cv.take<uint16_t>(lists);
  uint16_t* d_offs = cv.take<uint16_t>(offs);
  SjltJob* d_jobs = cv.take<SjltJob>(nprob);
  int4* d_items = cv.take<int4>(items.size());
  int2* d_chunks = cv.take<int2>(chunks.size());
  int64_t* d_prefix = cv.take<int64_t>(nprob);
  double** d_sa = cv.take<double*>(nprob);
  for (int p = 0; p < nprob; ++p) {
    SjltJob& jb = jobs[p];
    jb.part = part;
    jb.list = d_lists;
    jb.offs = d_offs;
    part += (size_t)((jb.nchunk + jb.cpg - 1) / jb.cpg) * jb.m * jb.d;
    d_lists += (list_elems(jb) + 7) & ~(size_t)7;
    d_offs += offs_elems(jb);
  }
  cudaStream_t str = ctx->stream;
  LSQ_CUDA_TRY(cudaMemcpyAsync(d_jobs, jobs.data(), nprob * sizeof(SjltJob), cudaMemcpyHostToDevice, str));
  LSQ_CUDA_TRY(cudaMemcpyAsync(d_items, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice, str));
  LSQ_CUDA_TRY(cudaMemcpyAsync(d_chunks, chunks.data(), chunks.size() * sizeof(int2), cudaMemcpyHostToDevice, str));
  LSQ_CUDA_TRY(cudaMemcpyAsync(d_prefix, prefix.data(), nprob * 8, cudaMemcpyHostToDevice, str));
  LSQ_CUDA_TRY(cudaMemcpyAsync(d_sa, SA, nprob * sizeof(double*), cudaMemcpyHostToDevice, str));
  st = launch_lists(ctx, d_jobs, jobs[0], d_chunks, (unsigned)chunks.size(), s, smem_l, seed);
  if (st != LSQ_OK) return st;
  LSQ_CUDA_TRY(cudaFuncSetAttribute(sjlt_gather_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_g));
  sjlt_gather_kernel<<<(unsigned)items.size(), GT, smem_g, str>>>(d_jobs, jobs[0], d_items);
  LSQ_LAUNCH_CHECK();
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 8 * (int64_t)ctx->sm_count));
  sjlt_reduce_kernel<<<grid, 256, 0, str>>>(d_jobs, jobs[0], d_prefix, d_sa, nullptr, nprob, total);
  LSQ_LAUNCH_CHECK();
  return LSQ_OK;
}
