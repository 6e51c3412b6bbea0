// The transforms of the FP64 engine, in 64-bit block fixed point.
//
// GB300 issues one FP64 instruction per 76 cycles and SM sub-partition, a 64-bit integer addition (two
// instructions) in 4 and a high 32 x 32 bit product in 4.  So a line is transformed as 64-bit integers that
// share one exponent, value = v 2^e: sums are exact and products keep the high 64 of their 128 bits.
// Measured on chip (radix-16 stages of 4096-point lines, exchanges included, time per point and stage):
// FP64 24.4 ps, double-float 3.49 ps, this 2.58 ps; error of one transform of N(0,1) data, against
// extended precision: FP64 2.1e-16, double-float 7.1e-15, this 7e-17.
//
// Scaling.  Before each twiddled stage the line is shifted left until its largest component fills bits
// 0..61 (an OR of the magnitude bits over the line's threads gives the shift).  Twiddles carry 60 fraction
// bits, so that a product's high word is the product over 16, the growth of the radix-16 DFT that follows:
// complex magnitudes stay below 2^62.5 and the rounding unit is 2^-58 of the line's largest value, against
// FP64's 2^-53.  The scale follows the data and not a growth bound, so lines whose spectra are concentrated
// (smooth fields) lose nothing.
//
// The DF64 engine sets the scale of the first stage's rows of at most kQStaticMax points once, on entry.  The unit
// after the last butterfly is then 2^-60 L times the row's largest value: N(0,1) and smooth rows lose
// nothing to speak of, since their largest value grows with the transform, rows of one spike over noise most.
// Normwise difference from the F64 engine over lambda_max ||u||, at worst over spikes, noise and alpha: 1.3e-15 at L =
// 512; it was 1.9e-15 at 1024 and 3.9e-15 at 2048 and 4096 (double-float arithmetic: 5e-15), where the scale now
// follows the data and both engines agree bit for bit.  (Columns and inverse transforms need the data's scale: the
// columns of a smooth field at high frequencies, and spectra, lost up to 28 bits without it.)
//
// Between kernels a line's values are stored as integers with the line's exponent beside them
// (apply_q.cuh); a kernel whose lines run across those aligns their exponents as it loads.
#pragma once

#include "common.cuh"
#include "fft.cuh"

namespace frlap {

struct cq {
  long long x, y;
};

__device__ __forceinline__ cq operator+(cq a, cq b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cq operator-(cq a, cq b) { return {a.x - b.x, a.y - b.y}; }

// the signed 32-bit halves of a = h 2^32 + l (|a| < 2^63 - 2^32)
struct QHalf {
  int h, l;
};
__host__ __device__ __forceinline__ QHalf q_half(long long a) {
  const int l = (int)a;
  return {(int)(a >> 32) + (int)((unsigned)l >> 31), l};
}
__device__ __forceinline__ long long q_wide(int a, int b) { return (long long)a * b; }

// Products a w / 2^64 as a1 w1 + (a1 w0 + a0 w1) / 2^32 on the signed halves: one 64-bit and two high
// 32-bit products (a0 w0 stays below the unit).  A high product rounds down; a sum takes them in pairs, one
// as p and one as -(-p), which rounds up, so that the offsets cancel and zero stays zero.  (Summing the cross
// products in 64 bits and rounding once is no more exact and takes multiply-adds with 64-bit addends, 5.5
// cycles each against 4: 3.04 against 2.72 ps per point and stage.)

// a w (CONJ = false) or a conj(w), over 16 (w: 60 fraction bits)
template <bool CONJ>
__device__ __forceinline__ cq q_cmul(cq a, int4 w) {
  const QHalf x = q_half(a.x), y = q_half(a.y);
  const int nrh = -w.x, nih = -w.z;
  cq r;
  if constexpr (!CONJ) {
    const int mx = __mulhi(x.h, w.y) - __mulhi(x.l, nrh) - __mulhi(y.h, w.w) + __mulhi(y.l, nih);
    const int my = __mulhi(x.h, w.w) - __mulhi(x.l, nih) + __mulhi(y.h, w.y) - __mulhi(y.l, nrh);
    r.x = q_wide(x.h, w.x) + (q_wide(y.h, nih) + (long long)mx);
    r.y = q_wide(x.h, w.z) + (q_wide(y.h, w.x) + (long long)my);
  } else {
    const int mx = __mulhi(x.h, w.y) - __mulhi(x.l, nrh) + __mulhi(y.h, w.w) - __mulhi(y.l, nih);
    const int my = __mulhi(y.h, w.y) - __mulhi(y.l, nrh) - __mulhi(x.h, w.w) + __mulhi(x.l, nih);
    r.x = q_wide(x.h, w.x) + (q_wide(y.h, w.z) + (long long)mx);
    r.y = q_wide(x.h, nih) + (q_wide(y.h, w.x) + (long long)my);
  }
  return r;
}
// a w / 2^64 for a real w
__device__ __forceinline__ long long q_rmul(QHalf a, QHalf w) {
  return q_wide(a.h, w.h) + (long long)(__mulhi(a.h, w.l) - __mulhi(a.l, -w.h));
}

// Constants of the 8- and 16-point DFTs with 64 fraction bits: 1 - cos(pi/8), sin(pi/8), 1 - 1/sqrt 2
// (factors above 1/2 enter as a - a (1 - c), so that their halves fit 32 bits).
constexpr long long kQ1mC1 = 0x137ca1866b95cebbLL, kQS1 = 0x61f78a9abaa58b47LL, kQ1mR2 = 0x4afb0ccc06219b7cLL;
constexpr int qhi(long long w) { return (int)((w - (long long)(int)(w & 0xffffffffLL)) >> 32); }
constexpr int qlo(long long w) { return (int)(w & 0xffffffffLL); }

// a / sqrt 2
__device__ __forceinline__ long long q_r2(long long a) {
  const QHalf t = q_half(a);
  constexpr int h = qhi(kQ1mR2), l = qlo(kQ1mR2);
  return a + (q_wide(t.h, -h) - (long long)(__mulhi(t.h, l) - __mulhi(t.l, -h)));
}
// a cos(pi/8) + b sin(pi/8) and a cos(pi/8) - b sin(pi/8)
__device__ __forceinline__ long long q_cs_add(long long a, long long b) {
  const QHalf s = q_half(a), t = q_half(b);
  constexpr int ch = qhi(kQ1mC1), cl = qlo(kQ1mC1), sh = qhi(kQS1), sl = qlo(kQS1);
  const int m = (__mulhi(t.h, sl) + __mulhi(t.l, sh)) - (__mulhi(s.h, cl) + __mulhi(s.l, ch));
  return a + (q_wide(s.h, -ch) + (q_wide(t.h, sh) + (long long)m));
}
__device__ __forceinline__ long long q_cs_sub(long long a, long long b) {
  const QHalf s = q_half(a), t = q_half(b);
  constexpr int ch = qhi(kQ1mC1), cl = qlo(kQ1mC1), sh = qhi(kQS1), sl = qlo(kQS1);
  const int m = (__mulhi(t.h, sl) - __mulhi(t.l, -sh)) + (__mulhi(s.h, cl) - __mulhi(s.l, -ch));
  return a + (q_wide(s.h, -ch) + (q_wide(t.h, -sh) - (long long)m));
}
// v W_16^m, m = 1, 2, 3, 6, 9 (W = exp(SIGN 2 pi i / 16))
template <int SIGN>
__device__ __forceinline__ cq q_w16(cq v, int m) {
  // multiply by exp(SIGN i t): (x cos t - SIGN y sin t, y cos t + SIGN x sin t)
  switch (m) {
    case 1: return SIGN < 0 ? cq{q_cs_add(v.x, v.y), q_cs_sub(v.y, v.x)} : cq{q_cs_sub(v.x, v.y), q_cs_add(v.y, v.x)};
    case 2: return SIGN < 0 ? cq{q_r2(v.x + v.y), q_r2(v.y - v.x)} : cq{q_r2(v.x - v.y), q_r2(v.y + v.x)};
    case 3:  // cos 3pi/8 = sin pi/8, sin 3pi/8 = cos pi/8
      return SIGN < 0 ? cq{q_cs_add(v.y, v.x), -q_cs_sub(v.x, v.y)} : cq{-q_cs_sub(v.y, v.x), q_cs_add(v.x, v.y)};
    case 6:  // cos = -1/sqrt 2, sin = 1/sqrt 2
      return SIGN < 0 ? cq{q_r2(v.y - v.x), -q_r2(v.x + v.y)} : cq{-q_r2(v.x + v.y), q_r2(v.x - v.y)};
    default:  // 9: minus the case m = 1
      return SIGN < 0 ? cq{-q_cs_add(v.x, v.y), -q_cs_sub(v.y, v.x)} : cq{-q_cs_sub(v.x, v.y), -q_cs_add(v.y, v.x)};
  }
}

template <int SIGN>
__device__ __forceinline__ void q_dft4(cq& a, cq& b, cq& c, cq& d) {
  const cq s0 = a + c, d0 = a - c, s1 = b + d, t = b - d;
  const cq d1 = mul_i<SIGN>(t);
  a = s0 + s1;
  c = s0 - s1;
  b = d0 + d1;
  d = d0 - d1;
}
template <int SIGN>
__device__ __forceinline__ void q_dft8(cq* v) {
  q_dft4<SIGN>(v[0], v[2], v[4], v[6]);
  q_dft4<SIGN>(v[1], v[3], v[5], v[7]);
  const cq e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
  const cq t1 = q_w16<SIGN>(v[3], 2), t2 = mul_i<SIGN>(v[5]), t3 = q_w16<SIGN>(v[7], 6);
  v[0] = e0 + o0; v[4] = e0 - o0;
  v[1] = e1 + t1; v[5] = e1 - t1;
  v[2] = e2 + t2; v[6] = e2 - t2;
  v[3] = e3 + t3; v[7] = e3 - t3;
}
template <int SIGN>
__device__ __forceinline__ void q_dft16(cq* v) {
#pragma unroll
  for (int j = 0; j < 4; ++j) q_dft4<SIGN>(v[j], v[4 + j], v[8 + j], v[12 + j]);
#pragma unroll
  for (int k = 1; k < 4; ++k)
#pragma unroll
    for (int j = 1; j < 4; ++j) v[4 * k + j] = j * k == 4 ? mul_i<SIGN>(v[4 * k + j]) : q_w16<SIGN>(v[4 * k + j], j * k);
  cq out[16];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    cq a = v[4 * k], b = v[4 * k + 1], c = v[4 * k + 2], d = v[4 * k + 3];
    q_dft4<SIGN>(a, b, c, d);
    out[k] = a; out[k + 4] = b; out[k + 8] = c; out[k + 12] = d;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = out[i];
}
template <int R, int SIGN>
__device__ __forceinline__ void q_dftR(cq* v) {
  if constexpr (R == 2) {
    const cq t = v[0] - v[1];
    v[0] = v[0] + v[1];
    v[1] = t;
  } else if constexpr (R == 4) {
    q_dft4<SIGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    q_dft8<SIGN>(v);
  } else {
    q_dft16<SIGN>(v);
  }
}

// ---- the line's scale

// Shared words through which the threads of a line that spans several warps agree on its scale: one per
// reduction of a kernel (at most kQSlots) and line (at most kQLines such lines per CTA), zero at first.
constexpr int kQSlots = 10, kQLines = 8;
__device__ __forceinline__ void q_slots_clear(unsigned* slots) {
  for (int i = threadIdx.x; i < kQSlots * kQLines; i += blockDim.x) slots[i] = 0u;
}

// OR (or maximum) of o over the line's threads.  A line of at most 32 threads has it at once.  A longer
// one: *slot collects it, and q_fetch reads it after the line's next barrier.
template <bool MAX>
__device__ __forceinline__ unsigned q_publish(unsigned o, int logL, unsigned* slot) {
  if (logL >= 9) {
    if constexpr (MAX) o = __reduce_max_sync(0xffffffffu, o);
    else o = __reduce_or_sync(0xffffffffu, o);
    if (logL > 9 && (threadIdx.x & 31) == 0) {
      if constexpr (MAX) atomicMax(slot, o);
      else atomicOr(slot, o);
    }
  } else {
    for (int s = 1 << (logL - 4) >> 1; s > 0; s >>= 1) {
      const unsigned t = __shfl_xor_sync(0xffffffffu, o, s);
      if constexpr (MAX) o = t > o ? t : o;
      else o |= t;
    }
  }
  return o;
}
__device__ __forceinline__ unsigned q_fetch(unsigned o, int logL, const unsigned* slot) {
  return logL > 9 ? *reinterpret_cast<const volatile unsigned*>(slot) : o;
}
// both, with the barrier in between
template <bool MAX>
__device__ __forceinline__ unsigned q_reduce(unsigned o, int logL, unsigned* slot) {
  o = q_publish<MAX>(o, logL, slot);
  if (logL > 9) line_sync<double>(logL);
  return q_fetch(o, logL, slot);
}

// magnitude bits of the components' high words
__device__ __forceinline__ unsigned q_bits(cq v) {
  const int a = (int)(v.x >> 32), b = (int)(v.y >> 32);
  return (unsigned)(a ^ (a >> 31)) | (unsigned)(b ^ (b >> 31));
}
__device__ __forceinline__ long long q_shl(long long a, int s) {  // 0 <= s <= 31
  const unsigned l = (unsigned)a;
  const unsigned h = __funnelshift_l(l, (unsigned)(a >> 32), s);
  return (long long)(((unsigned long long)h << 32) | (l << s));
}
// Shift of a line with magnitude bits o to bits 0..61: components below 2^62, or magnitudes still below 2^62.5.
__device__ __forceinline__ int q_fill_shift(unsigned o) {
  const int sh = __clz((int)o) - 2;
  return sh < 0 ? 0 : (sh > 30 ? 30 : sh);
}
// The line's entries v[0..N) (all threads') shifted so.
template <int N>
__device__ __forceinline__ void q_fill(cq* v, int& e, int logL, unsigned* slot) {
  unsigned o = 0u;
#pragma unroll
  for (int m = 0; m < N; ++m) o |= q_bits(v[m]);
  const int sh = q_fill_shift(q_reduce<false>(o, logL, slot));
#pragma unroll
  for (int m = 0; m < N; ++m) v[m] = {q_shl(v[m].x, sh), q_shl(v[m].y, sh)};
  e -= sh;
}
template <int SH>
__device__ __forceinline__ long long q_shr_round(long long a) {
  return (a + (1LL << (SH - 1))) >> SH;
}
template <int SH>
__device__ __forceinline__ cq q_shr_round(cq a) {
  return {q_shr_round<SH>(a.x), q_shr_round<SH>(a.y)};
}

// To nearest, ties to even where few bits go: ties are frequent there, and rounding them all one way puts
// the same offset on every bin of a spectrum, an error concentrated at one grid point.
template <int SH>
__device__ __forceinline__ long long q_shr_even(long long a) {
  return SH >= 4 ? q_shr_round<SH>(a) : (a + ((1LL << (SH - 1)) - 1 + ((a >> SH) & 1))) >> SH;
}
template <int SH>
__device__ __forceinline__ cq q_shr_even(cq a) {
  return {q_shr_even<SH>(a.x), q_shr_even<SH>(a.y)};
}

// ---- double <-> fixed point.  Scaling by a power of two is an addition to the exponent field.

// Exponents that mark a line with a non-finite entry, and a line of zeros: further stages shift an
// exponent by a few thousand at most, so a maximum over lines keeps the first and drops the second.
constexpr int kQNan = 1 << 24, kQZero = -(1 << 24);
struct QIn {
  int kadd, thr, e;
  bool small;
};
// hm: the high word of the line's largest |x|.  x 2^k < 2^58 for every x of the line; e = -k.
__device__ __forceinline__ QIn q_in_scale(unsigned hm) {
  int E = (int)(hm >> 20);
  QIn q;
  q.small = E < 64;  // near the subnormal range: the entries are scaled by 2^300 first
  if (q.small) E = (E < 1 ? 1 : E) + 300;
  const int k = 1080 - E;
  q.kadd = k << 20;
  q.thr = (k < 999 ? 1000 - k : 1) << 20;  // below: less than 2^-23 of a unit
  q.e = E == 2047 ? kQNan : (hm == 0u ? kQZero : (q.small ? -k - 300 : -k));
  return q;
}
__device__ __forceinline__ unsigned q_mag(double x) {
  const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
  return h == 0u && __double2loint(x) != 0 ? 1u : h;
}
__device__ __forceinline__ long long q_in(double x, const QIn& q) {
  if (q.small) x *= 0x1p300;
  const int h = __double2hiint(x);
  const int hs = (h & 0x7ff00000) < q.thr ? 0 : h + q.kadd;
  return __double2ll_rn(__hiloint2double(hs, __double2loint(x)));
}

__device__ __forceinline__ bool q_out_fast(int e) { return e > -1000 && e < 900; }
__device__ __forceinline__ double q_out(long long v, int e) {  // q_out_fast(e)
  const double d = __ll2double_rn(v);
  const int h = __double2hiint(d);
  return __hiloint2double(h == 0 ? 0 : h + e * (1 << 20), __double2loint(d));
}
// any exponent: the two factors of 2^e overflow and underflow as FP64 products do
__device__ __forceinline__ double q_out_any(long long v, int e) {
  if (q_out_fast(e)) return q_out(v, e);
  if (e > kQNan / 2) return __longlong_as_double(0x7ff8000000000000LL);
  e = e < -2040 ? -2040 : (e > 2040 ? 2040 : e);
  const int e1 = e / 2, e2 = e - e1;
  return __ll2double_rn(v) * __hiloint2double((1023 + e1) << 20, 0) * __hiloint2double((1023 + e2) << 20, 0);
}

// ---- the transform

// A twiddle, loaded where it stands in the code: hoisted over a stage, a stage's fifteen spill.
__device__ __forceinline__ int4 q_ld_tw(const int4* p) {
#ifdef FRLAP_BOUNDS_CHECK
  if (!bc_ok(p, sizeof(int4))) return make_int4(0, 0, 0, 0);
#endif
  int4 v;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

template <int SIGN>
__device__ __forceinline__ void q_stage16(cq* v, int lane, int logNs, const int4* __restrict__ tw, int logPtab) {
  const int Ns = 1 << logNs, k = lane & (Ns - 1);
  const int4* st = tw + (1 << logPtab) + 15 * (Ns - 1) - Ns + k;  // layout: twiddle_entries
  v[0] = q_shr_round<4>(v[0]);
#pragma unroll
  for (int r = 1; r < 16; ++r) v[r] = q_cmul<(SIGN > 0)>(v[r], q_ld_tw(st + r * Ns));
  q_dft16<SIGN>(v);
}
template <int R, int SIGN>
__device__ __forceinline__ void q_last_stage(cq* v, int lane, int G, const int4* __restrict__ tw, int shift) {
  constexpr int B = 16 / R;
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const int j = lane + b * G;
    cq t[R];
    t[0] = q_shr_round<4>(v[b]);
#pragma unroll
    for (int r = 1; r < R; ++r) t[r] = q_cmul<(SIGN > 0)>(v[b + r * B], q_ld_tw(tw + ((r * j) << shift)));
    q_dftR<R, SIGN>(t);
#pragma unroll
    for (int r = 0; r < R; ++r) v[b + r * B] = t[r];
  }
}

// Bits that a line's transform of log2 length = REM mod 4 ends below 2^62.5: a last stage of radix 2 or 4
// grows by that, but its products divide by 16.
template <int REM, int E = 16, int LOGL = 0>
constexpr int kQDrop = E == 4 ? ((REM & 1) ? 3 : 2) : E == 8 ? (LOGL % 3 == 0 ? 1 : LOGL % 3 == 1 ? 3 : 2)
                                                    : REM == 1 ? 3 : REM == 2 ? 2 : 0;

// Transforms with E = 4 or 8 entries a thread, in stages of radix E (a last one of 2 or 4 for the rest).
// For launches of few lines: every thread of a sixteen-entry line issues some 1500 instructions a stage, and with
// less than a warp per SM sub-partition their latency is the time.  E = 4 has a quarter of the entries and a fifth
// of the instructions a stage, twice the stages and four times the threads; E = 8 lies between.  Lines of at most
// 2^kQThinLog points.
// v[m] = x[lane + m L/E] on entry and X[lane + m L/E] on exit, scaled as in q_fft (magnitudes below
// 2^(62.5 - kQDrop<REM, E, LOGL>)).  With DYN = false the line is shifted by what its stage leaves free instead.
constexpr int kQThinLog = 10;
// Longest line whose scale may be set once (DYN = false): see above.
constexpr int kQStaticMax = 512;
template <int E>
constexpr int kQCta = E == 8 ? 1024 : 512;  // threads per CTA the kernels are compiled for
template <int E>
constexpr int kQLogE = E == 4 ? 2 : E == 8 ? 3 : 4;
// What stands for log2 of the line length where that tells the threads of a line (line_sync, q_reduce).
template <int E>
__host__ __device__ constexpr int q_lg(int logL) {
  return logL + 4 - kQLogE<E>;
}
template <int E, bool DYN, int SIGN, bool ZIN>
__device__ __forceinline__ void q_fft_e(cq* v, int& e, cq* buf, int logL, int lane, const int4* __restrict__ tw,
                                        int logPtab, bool sync_first, unsigned* slots, int& si) {
  constexpr int LE = kQLogE<E>;
  const int G = 1 << (logL - LE), lg = q_lg<E>(logL);
  if constexpr (ZIN) {
#pragma unroll
    for (int m = E / 2; m < E; ++m) v[m] = {0, 0};
  }
  q_dftR<E, SIGN>(v);
  int logNs = 0;  // of the stage whose results v holds
  while (true) {
    const int next = logNs + LE;
    // E = 4: the next stage's twiddles are in flight over the exchange (E = 8 has no registers for them)
    int4 w[3];
    if constexpr (E == 4) {
      if (next + 1 == logL) {
#pragma unroll
        for (int b = 0; b < 2; ++b) w[b] = q_ld_tw(tw + ((lane + b * G) << (logPtab - logL)));
      } else {
        const int k = lane & ((1 << next) - 1);
#pragma unroll
        for (int r = 1; r < 4; ++r) w[r - 1] = q_ld_tw(tw + ((r * k) << (logPtab - next - 2)));
      }
    }
    unsigned o = 0u;
    if (DYN) {
#pragma unroll
      for (int m = 0; m < E; ++m) o |= q_bits(v[m]);
      o = q_publish<false>(o, lg, slots + si);
    }
    if (logNs > 0 || sync_first) line_sync<double>(lg);
    const int Ns = 1 << logNs, kw = lane & (Ns - 1), ob = (lane - kw) * E + kw;
    const bool ns16 = (Ns & 15) == 0;
    const int obase = spad(ob), sstep = Ns + (Ns >> 4);
#pragma unroll
    for (int r = 0; r < E; ++r) buf[ns16 ? obase + r * sstep : spad(ob + r * Ns)] = v[r];
    line_sync<double>(lg);
    const bool g16 = (G & 15) == 0;
    const int rbase = spad(lane), rstep = G + (G >> 4);
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = buf[g16 ? rbase + m * rstep : spad(lane + m * G)];
    const int sh = DYN ? q_fill_shift(q_fetch(o, lg, slots + si)) : 4 - LE;
    if (DYN) ++si;
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = {q_shl(v[m].x, sh), q_shl(v[m].y, sh)};
    e += 4 - sh;
    logNs = next;
    if (logNs + 1 == logL) {  // radix 2
#pragma unroll
      for (int b = 0; b < E / 2; ++b) {
        const int4 wb = E == 4 ? w[b & 1] : q_ld_tw(tw + ((lane + b * G) << (logPtab - logL)));
        const cq s = q_shr_round<4>(v[b]), t = q_cmul<(SIGN > 0)>(v[b + E / 2], wb);
        v[b] = s + t;
        v[b + E / 2] = s - t;
      }
      return;
    }
    if constexpr (E == 8) {
      if (logNs + 2 == logL) {  // radix 4
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const int j = lane + b * G;
          v[b] = q_shr_round<4>(v[b]);
#pragma unroll
          for (int r = 1; r < 4; ++r)
            v[b + 2 * r] = q_cmul<(SIGN > 0)>(v[b + 2 * r], q_ld_tw(tw + ((r * j) << (logPtab - logL))));
          q_dft4<SIGN>(v[b], v[b + 2], v[b + 4], v[b + 6]);
        }
        return;
      }
    }
    v[0] = q_shr_round<4>(v[0]);
    if constexpr (E == 4) {
#pragma unroll
      for (int r = 1; r < 4; ++r) v[r] = q_cmul<(SIGN > 0)>(v[r], w[r - 1]);
    } else {
      // W_{8 Ns}^{r k} = W_{16 Ns}^{2 r k}, in the table's radix-16 stage entries, or in its last part
      const int k = lane & ((1 << logNs) - 1);
      const bool st16 = logNs + 4 <= logPtab;
      const int4* st = st16 ? tw + (1 << logPtab) + 15 * ((1 << logNs) - 1) - (1 << logNs) + k
                            : tw + twiddle_entries(1 << logPtab) - (1 << logNs) + k;
      const int step = st16 ? 2 << logNs : 1 << logNs;
#pragma unroll
      for (int r = 1; r < 8; ++r) v[r] = q_cmul<(SIGN > 0)>(v[r], q_ld_tw(st + r * step));
    }
    q_dftR<E, SIGN>(v);
    if (logNs + LE == logL) return;
  }
}

// As fft_regs: v[m] = x[lane + m G] on entry (components below 2^58), X[lane + m G] on exit (magnitudes
// below 2^(62.5 - kQDrop)); e, the line's exponent, follows.  DYN: the scale follows the data between stages;
// else it stays as set on entry (lines of at most kQStaticMax points).  ZIN: v[8..15] are zero.  slots:
// the line's reduction words, used from index si on.  E < 16: see q_fft_e.
template <bool DYN, int SIGN, bool ZIN, int REM, int E = 16>
__device__ __forceinline__ void q_fft(cq* v, int& e, cq* buf, int logL, int lane, const int4* __restrict__ tw,
                                      int logPtab, bool sync_first, unsigned* slots, int& si) {
  if constexpr (E < 16) {
    q_fft_e<E, DYN, SIGN, ZIN>(v, e, buf, logL, lane, tw, logPtab, sync_first, slots, si);
    return;
  } else {
  const int G = 1 << (logL - 4);
  if constexpr (ZIN) {
#pragma unroll
    for (int m = 8; m < 16; ++m) v[m] = {0, 0};
  }
  // between stages: write, agree on the scale, read, shift
  auto exchange = [&](int logNs, bool first8, bool pre_sync) {
    unsigned o = 0u;
    if (DYN) {
#pragma unroll
      for (int m = 0; m < 16; ++m) o |= q_bits(v[m]);
      o = q_publish<false>(o, logL, slots + si);
    }
    if (pre_sync) line_sync<double>(logL);
    if (first8) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int ob = spad((lane + b * G) * 8);
#pragma unroll
        for (int r = 0; r < 8; ++r) buf[ob + r] = v[b + r * 2];
      }
    } else {
      const int Ns = 1 << logNs, k = lane & (Ns - 1);
      const int ob = (lane - k) * 16 + k;
      const bool ns16 = (Ns & 15) == 0;
      const int obase = spad(ob), sstep = Ns + (Ns >> 4);
#pragma unroll
      for (int r = 0; r < 16; ++r) buf[ns16 ? obase + r * sstep : spad(ob + r * Ns)] = v[r];
    }
    line_sync<double>(logL);
    const bool g16 = (G & 15) == 0;
    const int rbase = spad(lane), rstep = G + (G >> 4);
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = buf[g16 ? rbase + m * rstep : spad(lane + m * G)];
    e += 4;
    if (DYN) {
      const int sh = q_fill_shift(q_fetch(o, logL, slots + si));
      ++si;
#pragma unroll
      for (int m = 0; m < 16; ++m) v[m] = {q_shl(v[m].x, sh), q_shl(v[m].y, sh)};
      e -= sh;
    }
  };
  int logNs;
  if constexpr (REM == 3) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      cq t[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) t[r] = v[b + r * 2];
      q_dft8<SIGN>(t);
#pragma unroll
      for (int r = 0; r < 8; ++r) v[b + r * 2] = t[r];
    }
    exchange(0, true, sync_first);
    logNs = 3;
  } else {
    q_dft16<SIGN>(v);
    if (REM == 0 && logL == 4) return;
    exchange(0, false, sync_first);
    logNs = 4;
  }
  while (true) {
    if constexpr (REM == 1 || REM == 2) {
      if (logNs + REM == logL) {
        q_last_stage<(1 << REM), SIGN>(v, lane, G, tw, logPtab - logL);
        return;
      }
    }
    q_stage16<SIGN>(v, lane, logNs, tw, logPtab);
    if (logNs + 4 == logL) return;
    exchange(logNs, false, true);
    logNs += 4;
  }
  }
}

}  // namespace frlap
