// Seeded sampling from the full softmax at a given temperature (training
// rollouts sample at temperature 1, top-p 1: App. A, training configuration).
//
// A draw is a deterministic function of (logits row, seed, draw number,
// inverse temperature), defined bit-exactly so that any device reproduces it:
//   bits_v  = word v % 4 of Philox4x32-10(counter = (v / 4, draw_lo, draw_hi, 0),
//             key = (seed_lo, seed_hi))   (Salmon et al., SC 2011)
//   u_v     = (2 (bits_v >> 9) + 1) 2^-24                       in (0, 1), exact
//   s_v     = fl(l_v c) - lg2(-lg2(u_v)),   c = fl(fp32(log2 e) * inv_temperature)
//   token   = argmax_v s_v, ties to the lower id
// with lg2 the fixed fp32 procedure below and every product and sum rounded
// to fp32 on its own (no fused multiply-add).  This is the Gumbel-max trick in
// base 2: l c - lg2(-lg2 u) = log2(e) (l / T - ln(-ln u)) - log2(ln 2).
//
// Most entries are ruled out by an upper bound of their score instead of having
// it evaluated: with x = 1 - u (exact), -log2 u >= x log2 e, so
//   s_v <= l_v c - (log2 x + log2(log2 e)).
// Eight entries at a time are held against the best score found so far (shared
// by a CTA's warps) by their largest logit and largest random word, one
// hardware log2 for the eight, where each score takes two eight-term
// polynomials; the few vectors that reach it take the bound entry by entry,
// and only the entries that still reach it get the defined score, so the draw
// stays bit-exact.
//
// Kernels: the sampled rows' 8-entry vectors form one flat range cut into one
// wave of equal pieces, one per CTA (a piece meets at most two rows).  A CTA
// stores its largest (score, -id) key per row it meets; a second kernel
// reduces each row's keys (max is order-free, so the result does not depend
// on the schedule).
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace {

constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;
constexpr uint32_t kLog2eBits = 0x3FB8AA3Bu;
// Two CTAs an SM with two vectors of a thread in work at once: fewer warps find
// their first threshold, longer stretches use it, and the two vectors' Philox
// chains fill the issue slots.  192 / 1000 rows of 151,936, us a call: 34.1 / 130.9;
// one vector at a time with four CTAs 39.2 / -, three 36.6 / 139.5, two 35.1 /
// 136.0; two vectors with three CTAs 37.3 / 138.2, with one CTA of 512 threads
// 45.0 / 142.5.
constexpr int kSampleThreads = 256;
constexpr int kSampleCtas = 2;  // resident CTAs per SM
constexpr int kSampleVecs = 2;  // vectors of a thread worked on at once
constexpr int kSampleGridCap = 2048;  // CTAs of one launch when the rows are fewer

// The ten round keys of one seed (key + i * Weyl increment), passed by value
// so that the rounds read them from the kernel's parameter bank.
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
};

PhiloxKeys philox_keys(uint64_t seed) {
  PhiloxKeys k;
  uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
  for (int i = 0; i < 10; ++i) {
    k.k0[i] = a;
    k.k1[i] = b;
    a += kPhiloxW0;
    b += kPhiloxW1;
  }
  return k;
}

// What the first two rounds of Philox leave constant over a row: the counter
// is (v / 4, draw_lo, draw_hi, 0), so round 1's second product and round 2's
// first do not depend on v.
struct PhiloxRow {
  uint32_t x2, z2, w2;  // round 2's xor terms of words 0 and 2, and its word 3
};

__device__ __forceinline__ void mul_wide(uint32_t a, uint32_t b, uint32_t &hi, uint32_t &lo) {
  const uint64_t p = (uint64_t)a * b;
  lo = (uint32_t)p;
  hi = (uint32_t)(p >> 32);
}

__device__ __forceinline__ PhiloxRow philox_row(uint32_t draw_lo, uint32_t draw_hi,
                                                const PhiloxKeys &key) {
  uint32_t h1, l1, h2, l2;
  mul_wide(kPhiloxM1, draw_hi, h1, l1);                      // round 1
  mul_wide(kPhiloxM0, h1 ^ draw_lo ^ key.k0[0], h2, l2);     // round 2
  return PhiloxRow{l1 ^ key.k0[1], h2 ^ key.k1[1], l2};
}

// Philox4x32 with 10 rounds of counter (g, draw_lo, draw_hi, 0).
__device__ __forceinline__ uint4 philox10(uint32_t g, const PhiloxRow &r, const PhiloxKeys &key) {
  uint32_t h0, l0, h1, l1;
  mul_wide(kPhiloxM0, g, h0, l0);                  // round 1
  mul_wide(kPhiloxM1, h0 ^ key.k1[0], h1, l1);     // round 2
  uint4 c = make_uint4(h1 ^ r.x2, l1, l0 ^ r.z2, r.w2);
#pragma unroll
  for (int i = 2; i < 10; ++i) {
    mul_wide(kPhiloxM0, c.x, h0, l0);
    mul_wide(kPhiloxM1, c.z, h1, l1);
    c = make_uint4(h1 ^ c.y ^ key.k0[i], l1, h0 ^ c.w ^ key.k1[i], l0);
  }
  return c;
}

// a score's order code: monotone, -0 folded onto +0
__device__ __forceinline__ uint32_t score_code(float s) {
  uint32_t b = __float_as_uint(s);
  if (b == 0x80000000u) b = 0u;
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float code_score(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// (score, -id) as one ordered 64-bit key; 0 = no entry
__device__ __forceinline__ unsigned long long score_key(float s, int v) {
  if (v < 0) return 0ull;
  return ((unsigned long long)score_code(s) << 32) |
         (unsigned long long)(0xffffffffu - (uint32_t)v);
}

__device__ __forceinline__ unsigned long long max_u64(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}

IPD_DEVINL unsigned long long f2_mul(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// log2 on the special-function unit (absolute error below 2^-22 on (0.5, 2),
// relative 2^-22 elsewhere), for bounds only
IPD_DEVINL float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The fixed lg2 of the sampler, of two positive values at once: for x =
// 2^e m with m in (sqrt(1/2), sqrt(2)], lg2(x) = e + t P(t) with t = m - 1
// and P by Horner's rule; P's coefficients are a least-squares fit of
// log2(1 + t) / t on Chebyshev nodes of [sqrt(1/2) - 1, sqrt(2) - 1], rounded
// to fp32 (|lg2(x) - log2(x)| <= 1.1e-6 for normal x).  The integer steps run
// per lane, the fp32 steps on packed pairs (each lane rounded exactly like the
// scalar operation, no fused multiply-add).  The reduction to m in (sqrt(1/2), sqrt(2)] subtracts the bit
// pattern just above sqrt(1/2) and shifts arithmetically: e = floor((b -
// bits(sqrt(1/2))^+) / 2^23), m = b - e 2^23 -- the same (m, e) as halving m
// when it exceeds sqrt(2); e enters as (1.5 2^23 + e) - 1.5 2^23, exact.
__device__ __forceinline__ unsigned long long lg2_x2(unsigned long long x2) {
  float x0, x1;
  f2_unpack(x2, x0, x1);
  const uint32_t b0 = __float_as_uint(x0), b1 = __float_as_uint(x1);
  const int e0 = (int)(b0 - 0x3f3504f4u) >> 23, e1 = (int)(b1 - 0x3f3504f4u) >> 23;
  const uint32_t m0 = b0 - ((uint32_t)e0 << 23), m1 = b1 - ((uint32_t)e1 << 23);
  const unsigned long long ef = f2_sub(
      f2_pack(__uint_as_float(0x4b400000u + (uint32_t)e0), __uint_as_float(0x4b400000u + (uint32_t)e1)),
      f2_pack(12582912.0f, 12582912.0f));
  const unsigned long long t =
      f2_sub(f2_pack(__uint_as_float(m0), __uint_as_float(m1)), f2_pack(1.0f, 1.0f));
  const float c7 = __uint_as_float(0xBE15B661u), c6 = __uint_as_float(0x3E6FD4B5u),
              c5 = __uint_as_float(0xBE7ECB25u), c4 = __uint_as_float(0x3E92FB93u),
              c3 = __uint_as_float(0xBEB871A3u), c2 = __uint_as_float(0x3EF63BADu),
              c1 = __uint_as_float(0xBF38AA93u), c0 = __uint_as_float(0x3FB8AA3Au);
  unsigned long long p = f2_pack(c7, c7);
  p = f2_add(f2_mul(p, t), f2_pack(c6, c6));
  p = f2_add(f2_mul(p, t), f2_pack(c5, c5));
  p = f2_add(f2_mul(p, t), f2_pack(c4, c4));
  p = f2_add(f2_mul(p, t), f2_pack(c3, c3));
  p = f2_add(f2_mul(p, t), f2_pack(c2, c2));
  p = f2_add(f2_mul(p, t), f2_pack(c1, c1));
  p = f2_add(f2_mul(p, t), f2_pack(c0, c0));
  return f2_add(ef, f2_mul(t, p));
}

// scores of two entries: u = (2 (bits >> 9) + 1) 2^-24, formed exactly as
// (1 + (bits >> 9) 2^-23) - (1 - 2^-24); s = l c - lg2(-lg2 u)
__device__ __forceinline__ void score_x2(uint32_t lbits2, uint32_t r0, uint32_t r1,
                                         unsigned long long c2, float &s0, float &s1) {
  const unsigned long long u = f2_sub(
      f2_pack(__uint_as_float(0x3f800000u | (r0 >> 9)), __uint_as_float(0x3f800000u | (r1 >> 9))),
      f2_pack(__uint_as_float(0x3f7fffffu), __uint_as_float(0x3f7fffffu)));
  const unsigned long long e = f2_mul(lg2_x2(u), f2_pack(-1.0f, -1.0f));  // -lg2 u > 0
  const unsigned long long g = lg2_x2(e);                                    // lg2(-lg2 u)
  const unsigned long long l = f2_pack(bf16lo(lbits2), bf16hi(lbits2));
  f2_unpack(f2_sub(f2_mul(l, c2), g), s0, s1);
}

// Upper bounds of two scores, short of the constant log2(log2 e): fl(l c) -
// lg2.approx(1 - u).  1 - u = (2 (2^23 - 1 - (bits >> 9)) + 1) 2^-24 is exact,
// formed like u from the complemented bits.  The products are the score's own
// (rounded once), so the bound meets the score through one monotone
// subtraction.
__device__ __forceinline__ void bound_x2(uint32_t lbits2, uint32_t r0, uint32_t r1,
                                         unsigned long long c2, float &b0, float &b1) {
  const unsigned long long x = f2_sub(
      f2_pack(__uint_as_float((r0 >> 9) ^ 0x3fffffffu), __uint_as_float((r1 >> 9) ^ 0x3fffffffu)),
      f2_pack(__uint_as_float(0x3f7fffffu), __uint_as_float(0x3f7fffffu)));
  float x0, x1;
  f2_unpack(x, x0, x1);
  const unsigned long long g = f2_pack(lg2_approx(x0), lg2_approx(x1));
  const unsigned long long l = f2_pack(bf16lo(lbits2), bf16hi(lbits2));
  f2_unpack(f2_sub(f2_mul(l, c2), g), b0, b1);
}

// Bounds are clamped here (an infinite logit's), so that a number can be put
// into their low bits.
constexpr float kMaxBound = 3.0e38f, kFltMax = 3.402823466e38f;

// The least bound_x2 value of an entry whose score can reach `best`: a score
// is at most bound - log2(log2 e) (0.52877); 0.5 leaves 0.028 for the errors
// of lg2.approx (below 1e-5 at |log2 x| <= 24) and of the score's own two
// fixed logarithms (below 2e-5 together), and 2^-18 |best| covers the rounding
// of the two subtractions and the three bits taken from a bound.
__device__ __forceinline__ float bound_threshold(float best) {
  return fminf(fmaf(fabsf(best), -3.814697265625e-6f, best + 0.5f), 2.9e38f);
}

__device__ __forceinline__ float max8(const float (&v)[8]) {
  return fmax3(fmax3(v[0], v[1], v[2]), fmax3(v[3], v[4], v[5]), fmaxf(v[6], v[7]));
}

// The entries of row vectors [v_lo, v_hi): every thread's best score and its
// id.  Equal scores keep the lower id (-0 == +0 too), and a thread whose
// entries all score -inf keeps the first id it met (-1: none).  s_thr is the
// largest threshold any warp of the CTA has published: a plain word, since any
// value ever written to it is a valid threshold; finite, so that a row of -inf
// ends the search at once.
__device__ __forceinline__ void scan_row(const uint16_t *__restrict__ row, int v_lo, int v_hi,
                                         uint32_t draw_lo, uint32_t draw_hi, const PhiloxKeys &key,
                                         float cf, volatile float *s_thr, float &bs, int &bv) {
  const int lane = threadIdx.x & 31;
  const unsigned long long c2 = f2_pack(cf, cf);
  const PhiloxRow pr = philox_row(draw_lo, draw_hi, key);
  const uint4 *src = reinterpret_cast<const uint4 *>(row);
  int vec = v_lo + (int)threadIdx.x;
  bs = -INFINITY;
  bv = vec < v_hi ? vec * 8 : -1;

  // a vector whose bound reaches the threshold, with its random words
  auto examine = [&](int vec, const uint4 &raw, const uint4 &ra, const uint4 &rb, float &thr) {
    // the entries' own bounds, the entry's number in the low three bits
    float ub[8];
    bound_x2(raw.x, ra.x, ra.y, c2, ub[0], ub[1]);
    bound_x2(raw.y, ra.z, ra.w, c2, ub[2], ub[3]);
    bound_x2(raw.z, rb.x, rb.y, c2, ub[4], ub[5]);
    bound_x2(raw.w, rb.z, rb.w, c2, ub[6], ub[7]);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      ub[j] = __uint_as_float((__float_as_uint(fminf(ub[j], kMaxBound)) & ~7u) | (uint32_t)j);
    float top = vec < v_hi ? max8(ub) : -INFINITY;
    // score each lane's largest bound that reaches the threshold, which follows
    // the warp's best score; then the next, usually none
    while (__any_sync(0xffffffffu, top >= thr)) {
      const uint32_t e = __float_as_uint(top) & 7u;
      const bool e0 = e & 1u, e1 = e & 2u, e2 = e & 4u;
      const uint32_t rlo = e1 ? (e0 ? ra.w : ra.z) : (e0 ? ra.y : ra.x);
      const uint32_t rhi = e1 ? (e0 ? rb.w : rb.z) : (e0 ? rb.y : rb.x);
      const uint32_t lw = e2 ? (e1 ? raw.w : raw.z) : (e1 ? raw.y : raw.x);
      const uint32_t rr = e2 ? rhi : rlo;
      float s, unused;
      score_x2(e0 ? lw >> 16 : lw, rr, rr, c2, s, unused);
      const int v = vec * 8 + (int)e;
      if (top >= thr && (s > bs || (s == bs && v < bv))) {
        bs = s;
        bv = v;
      }
      thr = fmaxf(thr, bound_threshold(code_score(__reduce_max_sync(0xffffffffu, score_code(bs)))));
      float rest[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) rest[j] = ub[j] < top ? ub[j] : -INFINITY;
      top = max8(rest);
    }
    if (lane == 0 && thr > *s_thr) *s_thr = thr;
  };

  uint4 nxt[kSampleVecs];
#pragma unroll
  for (int u = 0; u < kSampleVecs; ++u) {
    nxt[u] = make_uint4(0, 0, 0, 0);
    if (vec + u * kSampleThreads < v_hi) nxt[u] = __ldg(src + vec + u * kSampleThreads);
  }
  constexpr int kStep = kSampleVecs * kSampleThreads;
#pragma unroll 1
  for (int first = vec - lane; first < v_hi; first += kStep, vec += kStep) {
    uint4 raw[kSampleVecs], ra[kSampleVecs], rb[kSampleVecs];
    float b8[kSampleVecs];
#pragma unroll
    for (int u = 0; u < kSampleVecs; ++u) {
      const int v = vec + u * kSampleThreads;
      raw[u] = nxt[u];
      if (v + kStep < v_hi) nxt[u] = __ldg(src + v + kStep);
      ra[u] = philox10(2u * (uint32_t)v, pr, key);
      rb[u] = philox10(2u * (uint32_t)v + 1u, pr, key);
      // the vector's bound: its largest logit with its largest random word.  With
      // y = 2^32 - 1 - bits, y 2^-32 is at most 2 (1 - u), so the bound needs one
      // more unit of slack than an entry's own; y = 0 gives +inf
      const uint32_t r8 = max(max(max(ra[u].x, ra[u].y), max(ra[u].z, ra[u].w)),
                              max(max(rb[u].x, rb[u].y), max(rb[u].z, rb[u].w)));
      b8[u] = __fsub_rn(__fmul_rn(bf16x8_max(raw[u]), cf), lg2_approx(__uint2float_rn(~r8)));
      if (v >= v_hi) b8[u] = -INFINITY;
    }
    float thr = *s_thr;
    bool reach = false;
#pragma unroll
    for (int u = 0; u < kSampleVecs; ++u) reach |= b8[u] >= thr - 33.f;
    if (!__any_sync(0xffffffffu, reach)) continue;
#pragma unroll
    for (int u = 0; u < kSampleVecs; ++u)
      examine(vec + u * kSampleThreads, raw[u], ra[u], rb[u], thr);
  }
}

// How the rows' vectors are cut: CTA i takes `len` of them, one more if i < rem,
// from piece_begin(i) on.
struct Pieces {
  int len, rem;
};
__device__ __forceinline__ long long piece_begin(const Pieces &p, int i) {
  return (long long)i * p.len + min(i, p.rem);
}
// a / b, in 32 bits where a fits (a 64-bit division takes over a hundred
// instructions of every warp)
__device__ __forceinline__ int div_small(long long a, int b) {
  return (a >> 32) == 0 ? (int)((uint32_t)a / (uint32_t)b) : (int)(a / b);
}
__device__ __forceinline__ int piece_of(const Pieces &p, long long x) {
  const long long longer = (long long)(p.len + 1) * p.rem;
  return x < longer ? div_small(x, p.len + 1) : p.rem + div_small(x - longer, p.len);
}

// One draw per row of a list of rows.  mode 0: row r is row r of `rows0`
// with draw number draw_id[r].  mode 1 (after a verdict): request r draws the
// first token of its next span from the next driver's row n_emit[r] of its
// span (rows0 = student, rows1 = teacher) with draw number draw_id[r] +
// prefix_len[r] + n_emit[r]; a request that ended or emitted every span token
// draws nothing.
//
// Bound: the integer pipes.  Philox's 36 wide multiplies a vector keep the
// heavy half of the FMA pipe over half busy, and the rows are read at 1.7 TB/s.
// 192 rows of 151,936: 57.3 us a call with every entry scored (44 warp
// instructions an entry), 34.1 now.
//
// Work split: the rows' 8-entry vectors form one flat range that is cut into
// gridDim.x equal pieces, one per CTA (grid >= rows, so a piece meets at most
// two rows).  Each CTA stores its best key for the first and the second row
// it meets (0 where it meets none).
__global__ void __launch_bounds__(kSampleThreads, kSampleCtas) sample_partial_kernel(
    int mode, const uint16_t *__restrict__ rows0, const uint16_t *__restrict__ rows1, int vocab,
    int n_rows, const Pieces pieces, const PhiloxKeys key, const uint64_t *__restrict__ draw_id,
    float inv_temperature, const int32_t *__restrict__ cu_span,
    const int32_t *__restrict__ prefix_len, const int32_t *__restrict__ n_emit,
    const uint8_t *__restrict__ next_driver, const uint8_t *__restrict__ done,
    unsigned long long *__restrict__ partial) {
  __shared__ unsigned long long s_best[2][kSampleThreads / 32];
  __shared__ const uint16_t *s_row[2];
  __shared__ uint32_t s_draw[2][2];
  __shared__ float s_thr[2];
  dependency_wait();  // the verdict, when the draw follows one
  const int nv = vocab >> 3;  // vectors per row
  const long long lo = piece_begin(pieces, blockIdx.x), hi = piece_begin(pieces, blockIdx.x + 1);
  const int row_lo = div_small(lo, nv);
  if (threadIdx.x < 2) {
    const int r = row_lo + (int)threadIdx.x;
    const uint16_t *row = nullptr;
    uint64_t draw = 0ull;
    if (r < n_rows) {
      draw = draw_id ? draw_id[r] : 0ull;
      if (mode == 1) {
        const int t0 = cu_span[r], t1 = cu_span[r + 1], n = n_emit[r];
        if (!(done[r] || t0 < 0 || n < 0 || n >= t1 - t0)) {
          row = (next_driver[r] ? rows1 : rows0) + (size_t)(t0 + n) * vocab;
          draw += (uint64_t)(int64_t)(prefix_len[r] + n);
        }
      } else {
        row = rows0 + (size_t)r * vocab;
      }
    }
    s_row[threadIdx.x] = row;
    s_draw[threadIdx.x][0] = (uint32_t)draw;
    s_draw[threadIdx.x][1] = (uint32_t)(draw >> 32);
    s_thr[threadIdx.x] = -kFltMax;  // every finite bound reaches it, -inf never does
  }
  __syncthreads();
  const float cf = __fmul_rn(__uint_as_float(kLog2eBits), inv_temperature);
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    // this CTA's vectors of row row_lo + k
    const long long base = (long long)(row_lo + k) * nv;
    const int v_lo = (int)(lo > base ? lo - base : 0);
    const int v_hi = (int)(hi - base < nv ? (hi > base ? hi - base : 0) : nv);
    float bs = -INFINITY;
    int bv = -1;
    if (s_row[k] != nullptr)
      scan_row(s_row[k], v_lo, v_hi, s_draw[k][0], s_draw[k][1], key, cf, &s_thr[k], bs, bv);
    unsigned long long b = score_key(bs, bv);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b = max_u64(b, __shfl_xor_sync(0xffffffffu, b, o));
    if ((threadIdx.x & 31) == 0) s_best[k][threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    unsigned long long b = 0ull;
#pragma unroll
    for (int i = 0; i < kSampleThreads / 32; ++i) b = max_u64(b, s_best[threadIdx.x][i]);
    partial[2 * (size_t)blockIdx.x + threadIdx.x] = b;
  }
}

// one warp per row: the best key over the CTAs whose piece meets the row ->
// token id (-1: none)
__global__ void __launch_bounds__(256) sample_finalize_kernel(
    const unsigned long long *__restrict__ partial, int n_rows, int vocab, const Pieces pieces,
    int32_t *__restrict__ tokens) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  dependency_wait();  // the CTAs' partials
  if (r >= n_rows) return;
  unsigned long long b = 0ull;
  if (partial) {
    const int nv = vocab >> 3;
    const int i0 = piece_of(pieces, (long long)r * nv);
    const int i1 = piece_of(pieces, (long long)(r + 1) * nv - 1);
    for (int i = i0 + lane; i <= i1; i += 32) {
      // row r is the first of its CTA's two unless the piece began before it
      const int second = piece_begin(pieces, i) < (long long)r * nv ? 1 : 0;
      b = max_u64(b, partial[2 * (size_t)i + second]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b = max_u64(b, __shfl_xor_sync(0xffffffffu, b, o));
  if (lane == 0) tokens[r] = b ? (int32_t)(0xffffffffu - (uint32_t)b) : -1;
}

// CTAs of one launch: every resident slot of the GPU once (so the equal
// pieces run as one wave), at least one per row
int sample_grid(int n_rows) {
  static int cap[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  if (cap[dev] == 0) {
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sample_partial_kernel,
                                                      kSampleThreads, 0) != cudaSuccess)
      return -1;
    const int c = sms * (per_sm > 0 ? per_sm : 1);
    cap[dev] = c < kSampleGridCap ? c : kSampleGridCap;
  }
  return n_rows > cap[dev] ? n_rows : cap[dev];
}

Pieces sample_pieces(int n_rows, int vocab, int grid) {
  const long long total = (long long)n_rows * (vocab >> 3);
  return Pieces{(int)(total / grid), (int)(total % grid)};
}

}  // namespace

extern "C" __attribute__((visibility("hidden"))) size_t ipd_internal_sample_ws(int n_rows,
                                                                              int vocab) {
  (void)vocab;
  const size_t g = n_rows > kSampleGridCap ? (size_t)n_rows : (size_t)kSampleGridCap;
  return 2 * g * sizeof(unsigned long long);
}

// The draw after a verdict, launched by ipd_score_span_ex (ws: ipd_internal_sample_ws bytes,
// or NULL when the step has no span tokens).
extern "C" __attribute__((visibility("hidden"))) int ipd_internal_sample_after_verdict(
    const uint16_t *ls, const uint16_t *lt, int num_reqs, int total_tokens, int vocab,
    uint64_t seed, const uint64_t *draw_base, float inv_temperature, const int32_t *cu_span,
    const int32_t *prefix_len, const int32_t *n_emit, const uint8_t *next_driver,
    const uint8_t *done, int32_t *next_token, void *ws, cudaStream_t st) {
  unsigned long long *partial = nullptr;
  int grid = 1;
  if (total_tokens > 0) {
    grid = sample_grid(num_reqs);
    if (grid < 0) return IPD_ERR_CUDA;
    partial = static_cast<unsigned long long *>(ws);
    if (launch_dependent(sample_partial_kernel, grid, kSampleThreads, 0, st, 1, ls, lt, vocab,
                         num_reqs, sample_pieces(num_reqs, vocab, grid), philox_keys(seed), draw_base, inv_temperature, cu_span,
                         prefix_len, n_emit, next_driver, done, partial) != cudaSuccess)
      return IPD_ERR_CUDA;
  }
  if (launch_dependent(sample_finalize_kernel, (num_reqs + 7) / 8, 256, 0, st, partial, num_reqs,
                       vocab, sample_pieces(num_reqs, vocab, grid), next_token) != cudaSuccess)
    return IPD_ERR_CUDA;
  return IPD_OK;
}

extern "C" size_t ipd_sample_workspace_size(int n_rows, int vocab) {
  if (n_rows < 0 || vocab < 1) return 0;
  return ipd_internal_sample_ws(n_rows, vocab);
}

extern "C" int ipd_sample(const uint16_t *logits, int n_rows, int vocab, uint64_t seed,
                          const uint64_t *draw_id, float inv_temperature, int32_t *tokens,
                          void *workspace, size_t workspace_bytes, ipd_stream_t stream) {
  if (n_rows < 0) return IPD_ERR_INVALID_ARG;
  if (vocab < 8 || vocab % 8) return IPD_ERR_UNSUPPORTED;
  if (!(inv_temperature > 0.f) || !(inv_temperature - inv_temperature == 0.f))
    return IPD_ERR_INVALID_ARG;  // not positive and finite
  if (n_rows == 0) return IPD_OK;
  if (!logits || !tokens || ((uintptr_t)logits & 15)) return IPD_ERR_INVALID_ARG;
  if ((long long)n_rows * (vocab >> 3) > 0x3fffffffffffLL) return IPD_ERR_UNSUPPORTED;
  if (!workspace || workspace_bytes < ipd_internal_sample_ws(n_rows, vocab) ||
      ((uintptr_t)workspace & 7))
    return IPD_ERR_WORKSPACE;
  const int grid = sample_grid(n_rows);
  if (grid < 0) return IPD_ERR_CUDA;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  unsigned long long *partial = static_cast<unsigned long long *>(workspace);
  sample_partial_kernel<<<grid, kSampleThreads, 0, st>>>(
      0, logits, nullptr, vocab, n_rows, sample_pieces(n_rows, vocab, grid), philox_keys(seed), draw_id,
      inv_temperature, nullptr, nullptr, nullptr, nullptr, nullptr, partial);
  if (cudaGetLastError() != cudaSuccess) return IPD_ERR_CUDA;
  if (launch_dependent(sample_finalize_kernel, (n_rows + 7) / 8, 256, 0, st, partial, n_rows, vocab,
                       sample_pieces(n_rows, vocab, grid), tokens) != cudaSuccess)
    return IPD_ERR_CUDA;
  return IPD_OK;
}
