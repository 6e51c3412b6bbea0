// The apply's stages in the FP64 and the DF64 engine: the pipeline of apply_impl.cuh on 64-bit block fixed point
// (fft_q.cuh).  Vectors and symbol are FP64.  The DF64 engine's first stage sets the scale of a row of at most 512 points
// once (DYN = false); all else is common.  In the workspace a complex value is two 64-bit integers
// below 2^62.5, as a transform leaves them, in the same S1 / S2 layout and 16 bytes as an FP64 pair, and each line that a kernel wrote
// has its exponent in an array behind S1 and S2:
//   ex_row[row]           after the first stage, for S1[.][row]
//   ex_line[kx n_z + z]   3D, for the y lines of both directions
//   ex_col[kx] (2D), ex_col[kx P_y + ky] (3D) after the middle stage
// A kernel whose lines run across those shifts its entries to a common exponent as it loads them: the bits it drops
// are below the rounding unit of its own line.
//
// Native FP64 stages were bound by the FP64 pipe (84% busy) at a ninth of these stages' rate; conversions
// from and to FP64 (64 cycles a warp) remain only at the vectors.
#pragma once

#include "apply_impl.cuh"
#include "fft_q.cuh"

namespace frlap {

namespace {

// Exponent arrays of one instance, in ints.
struct QExpLayout {
  size_t row, line, col, total;
};
inline QExpLayout q_exp_layout(const Plan& p) {
  const size_t Hx1 = p.P[0] / 2 + 1;
  QExpLayout l;
  l.row = 0;
  const size_t nrows = (size_t)p.n[1] * (p.d == 3 ? p.n[2] : 1);
  l.line = align256(nrows * 4) / 4;
  l.col = l.line + (p.d == 3 ? align256(Hx1 * p.n[2] * 4) / 4 : 0);
  // 2D with the split middle stage: a second array for the even half
  const size_t ncol = p.d == 3 ? Hx1 * p.P[1] : Hx1 * (p.P[1] > kMaxLine ? 2 : 1);
  l.total = l.col + align256(ncol * 4) / 4;
  return l;
}

__device__ __forceinline__ unsigned q_ord(int e) { return (unsigned)e ^ 0x80000000u; }
__device__ __forceinline__ int q_unord(unsigned u) { return (int)(u ^ 0x80000000u); }
// v 2^(e - top), e <= top, to nearest, ties up or, with down, down.  Ties are frequent where few bits go.  Callers
// alternate down with the parity of a frequency index along which a line's exponent (and so the offset of a rounding) is
// the same: the offset then sits at the middle of the axis' embedding, outside the box, instead of adding up at its first
// point.
__device__ __forceinline__ cq q_align(cq v, int e, int top, bool down) {
  const int d = min(top - e, 63);
  const unsigned c = ((1u << min(d, 31)) - (down ? 1u : 0u)) >> 1;
  return {(v.x + c) >> d, (v.y + c) >> d};
}

// The shift that brings a line with magnitude bits o of its components' high words to components below 2^58, what a
// transform starts from.
__device__ __forceinline__ int q_excess(unsigned o) { return max(6 - __clz((int)o), 0); }

#define FRLAP_Q_PROLOGUE(logLine)                                        \
  extern __shared__ __align__(16) unsigned char smem_raw[];              \
  __shared__ unsigned q_slot_words[kQSlots * kQLines];                   \
  if (skip && FRLAP_GLD(skip)) return;                                   \
  if ((logLine) > 9) {                                                   \
    q_slots_clear(q_slot_words);                                         \
    __syncthreads();                                                     \
  }                                                                      \
  cq* smem = reinterpret_cast<cq*>(smem_raw);

template <bool DYN, int REM, int LOGL, int E>
__global__ void __launch_bounds__(kQCta<E>, 1)
    k_q_r2c(const double* __restrict__ in, cq* __restrict__ out, int* __restrict__ ex, int nlines, int n, size_t ldo,
            int logH, int TL, const int4* __restrict__ tw, const int* __restrict__ skip, Batch bt, size_t ex_inst) {
  logH = LOGL;
  constexpr int lg = q_lg<E>(LOGL);
  {
    const size_t bi = blockIdx.y;
    in += bi * bt.in;
    out += bi * bt.out;
    ex += bi * ex_inst;
    if (skip) skip += bi * bt.skip;
  }
  FRLAP_Q_PROLOGUE(lg)
  const int H = 1 << logH, G = H / E, LS = sline(H);
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int line0 = blockIdx.x * TL, line = line0 + l;
  const bool valid = line < nlines;
  const double* src = in + (size_t)(valid ? line : 0) * n;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * LS;
  // packed samples z[q] = x[2q] + i x[2q+1], as in k_r2c_T
  double xr[E / 2], xi[E / 2];
  const bool pair_aligned = (reinterpret_cast<uintptr_t>(src) % sizeof(double2)) == 0;
  unsigned hm = 0u;
#pragma unroll
  for (int m = 0; m < E / 2; ++m) {
    const int q = lane + m * G;
    double a = 0.0, b = 0.0;
    if (valid) {
      if (pair_aligned && 2 * q + 1 < n) {
        const double2 t = FRLAP_GLD(reinterpret_cast<const double2*>(src + 2 * q));
        a = t.x;
        b = t.y;
      } else {
        if (2 * q < n) a = FRLAP_GLD(src + 2 * q);
        if (2 * q + 1 < n) b = FRLAP_GLD(src + 2 * q + 1);
      }
    }
    xr[m] = a;
    xi[m] = b;
  }
#pragma unroll
  for (int m = 0; m < E / 2; ++m) hm = max(hm, max(q_mag(xr[m]), q_mag(xi[m])));
  int si = 0;
  const QIn qs = q_in_scale(q_reduce<true>(hm, lg, slots + si));
  ++si;
  cq v[E];
#pragma unroll
  for (int m = 0; m < E / 2; ++m) v[m] = {q_in(xr[m], qs), q_in(xi[m], qs)};
  int e = qs.e;
  q_fft<DYN, -1, true, REM, E>(v, e, buf, logH, lane, tw, logH + 1, false, slots, si);
  if constexpr (!DYN) q_fill<E>(v, e, lg, slots + si);
  line_sync<double>(lg);
#pragma unroll
  for (int m = 0; m < E; ++m) buf[spad(lane + m * G)] = v[m];
  int4 wk[E / 2];  // W^k of this thread's pairs, in flight over the barrier
#pragma unroll
  for (int j = 0; j < E / 2; ++j) wk[j] = FRLAP_GLD(tw + lane + j * G);
  line_sync<double>(lg);
  // Real-data split in place, one product per pair (see r2c_tile): X[k] = s + W^k d,
  // X[H-k] = conj(s - W^k d), s = (a + b) / 2, d = -i (a - b) / 2, over 2^F, below 2^61.5 (D = kQDrop, 0 after q_fill:
  // a and b are below 2^(62.5 - D)).  A product's unit is 16: where a and b leave the room, a - b goes in 16 times
  // larger, so that the high frequencies of a smooth row, which the symbol weighs most, carry units of 2^-61.5 of the
  // row's largest value and not of 2^-58 (stored at 58 bits, F64 applies of smooth fields had 2.4e-16 lambda_max ||u|| on
  // 4096-interval rows, native FP64 8.8e-17; now 3.8e-17).  With D = 0, a + b can take 64 bits, so both are shifted first.
  constexpr int D = DYN ? kQDrop<REM, E, LOGL> : 0, F = D < 2 ? 2 - D : 0;
  auto split = [&](int k, const int4 wk) {
    const int km = H - k;
    const cq a = buf[spad(k)];
    const cq b = conjg(buf[spad(km & (H - 1))]);
    const bool room = (q_bits(a) | q_bits(b)) < (1u << (25 + F));
    constexpr int kRoom = 3 - F, kElse = D - 1;  // shifts of a - b
    cq d, s;
    if constexpr (D == 0) {
      const int r = room ? 0 : 1;
      d = {(a.x >> r) - (b.x >> r), (a.y >> r) - (b.y >> r)};
      if (room) d = {d.x << kRoom, d.y << kRoom};
      s = {((a.x >> 2) + (b.x >> 2) + 1) >> 1, ((a.y >> 2) + (b.y >> 2) + 1) >> 1};
    } else {
      const int r = room ? kRoom : kElse;
      d = a - b;
      d = {d.x << r, d.y << r};
      s = q_shr_even<1 + F>(a + b);
    }
    cq t = q_cmul<false>(mul_i<-1>(d), wk);
    const int up = room ? 0 : kRoom - kElse;
    t = {t.x << up, t.y << up};
    buf[spad(k)] = s + t;
    if (k != km) buf[spad(km)] = conjg(s - t);
  };
#pragma unroll
  for (int j = 0; j < E / 2; ++j) split(lane + j * G, wk[j]);
  if (lane == 0) split(H / 2, FRLAP_GLD(tw + H / 2));
  if (valid && lane == 0) FRLAP_GST(ex + line, e + F);
  __syncthreads();
  const int logTL = __ffs(TL) - 1;
  const int lt = threadIdx.x & (TL - 1);
  if (line0 + lt < nlines) {
    const cq* trow = smem + (size_t)lt * LS;
    int k = (int)threadIdx.x >> logTL;
    cq* gp = out + (size_t)k * ldo + line0 + lt;
    const size_t gstep = (size_t)G * ldo;
#pragma unroll 4
    for (; k <= H; k += G, gp += gstep) FRLAP_GST(gp, trow[spad(k)]);
  }
}

// Entries v[m], m < M, of a line that runs across lines of other exponents, aligned to an exponent at which all fit 58
// bits, which it returns (down: see q_align).  Entries are stored with up to 63 bits: what a line drops here is below the
// unit of its own largest value, where dropped before it was stored it would be one of the crossing line's.
template <int M>
__device__ __forceinline__ int q_load_aligned(cq* v, const cq* line, const int* ex, bool down, int lane, int G, int n,
                                              bool valid, int logL, unsigned* slot) {
  int e[M];
  int top = kQZero;
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int i = lane + m * G;
    const bool ok = valid && i < n;
    v[m] = ok ? ld_stream(line + i) : cq{0, 0};
    e[m] = ok ? FRLAP_GLD(ex + i) : kQZero;
  }
#pragma unroll
  for (int m = 0; m < M; ++m) top = max(top, e[m] + q_excess(q_bits(v[m])));
  top = q_unord(q_reduce<true>(q_ord(top), logL, slot));
#pragma unroll
  for (int m = 0; m < M; ++m) v[m] = q_align(v[m], e[m], top, down);
  return top;
}

// Loads that stay where they are written (not merged with an earlier one of the same address).
__device__ __forceinline__ unsigned q_ld_hi(const double* p) {
#ifdef FRLAP_BOUNDS_CHECK
  if (!bc_ok(p, 8)) return 0u;
#endif
  unsigned h;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(h) : "l"(reinterpret_cast<const unsigned*>(p) + 1));
  return h;
}
__device__ __forceinline__ double q_ld(const double* p) {
#ifdef FRLAP_BOUNDS_CHECK
  if (!bc_ok(p, 8)) return 0.0;
#endif
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

// The symbol product v <- lambda v at a common exponent for the line, components below 2^58.  lambda enters by
// its mantissa, so every entry has full precision whatever lambda's range along the line; the line's
// exponent is what its largest |lambda_k| |v_k| needs.  lambda is not negative: A is strictly diagonally dominant
// and so is its circulant embedding (a rounding below zero is cut off in the table).
// plain: every lambda is finite and normal (Plan::lam_plain).  Otherwise a subnormal or zero lambda has no leading bit,
// and a non-finite one makes its line NaN, even one of zeros.  A flag of the plan, because to look at each
// lambda costs a single 2047^2 apply 1%.
// lrow[idx(m)] is entry m's lambda; its words are read twice (the second time from L1), since held over the
// reduction they spill.
template <int E, typename I>
__device__ __forceinline__ void q_symbol(cq* v, int& e, const double* __restrict__ lrow, I idx, bool plain, int logL,
                                         unsigned* slot) {
  int top = 0;
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const unsigned h = q_ld_hi(lrow + idx(m));
    // leading bit of |v| above bit 31 (the conversion rounds it up by at most one), plus 127
    const int pos = __float_as_int(__uint2float_rn(q_bits(v[m]))) >> 23;
    top = max(top, (int)(h >> 20) + max(pos, 126));
  }
  if (!plain) {
#pragma unroll 1
    for (int m = 0; m < E; ++m)
      if (q_ld_hi(lrow + idx(m)) >= 0x7ff00000u) top = 2 * kQNan;
  }
  top = (int)q_reduce<true>((unsigned)top, logL, slot);
  auto product = [&](auto normal) {
#pragma unroll
    for (int m = 0; m < E; ++m) {
      // lambda v = (mant v / 2^64) 2^(el - 1020), 2^61 <= mant < 2^62, and |v| 2^(el - top + 127) < 2^33: the
      // shift s = el - top + 152 brings the product below 2^58.  A right shift is one of the mantissa (its
      // dropped bits weigh less than a unit of the product), a left one is one of v.
      const double lam = q_ld(lrow + idx(m));
      const unsigned h = (unsigned)__double2hiint(lam), l = (unsigned)__double2loint(lam);
      const int s = (int)(h >> 20) - top + 152;
      unsigned long long mant =
          ((unsigned long long)__funnelshift_l(l, (h & 0xfffffu) | 0x100000u, 9) << 32) | (l << 9);
      if (!decltype(normal)::value && h < 0x100000u) mant = (mant - (1ull << 61)) << 1;  // el = 0 stands for 1
      mant >>= min(max(-s, 0), 63);
      const int sl = min(max(s, 0), 31);
      const QHalf w = q_half((long long)mant);
      v[m] = {q_rmul(q_half(q_shl(v[m].x, sl)), w), q_rmul(q_half(q_shl(v[m].y, sl)), w)};
    }
  };
  if (plain) product(std::true_type{});
  else product(std::false_type{});
  e += top - 1172;
}

// A column's entries of one line: element i of instance-local column col at data[col ld + i].
template <int REM, int LOGP, int E>
__global__ void __launch_bounds__(kQCta<E>, 1)
    k_q_colmul(cq* __restrict__ data, const int* __restrict__ ex_in, int* __restrict__ ex_out, int ncols, int n,
               size_t ld, int logP, int TL, const double* __restrict__ lam, LamMap map, int nz,
               const int4* __restrict__ tw, const int* __restrict__ skip, Batch bt, size_t ex_inst) {
  logP = LOGP;
  constexpr int lg = q_lg<E>(LOGP);
  {
    const size_t bi = blockIdx.y;
    data += bi * bt.in;
    lam += bi * bt.lam;
    ex_in += bi * ex_inst;
    ex_out += bi * ex_inst;
    if (skip) skip += bi * bt.skip;
  }
  FRLAP_Q_PROLOGUE(lg)
  const int P = 1 << logP, G = P / E;
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int col = blockIdx.x * TL + l;
  const bool valid = col < ncols;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * sline(P);
  const int c = valid ? col : 0;
  int si = 0;
  cq v[E];
  const int kx = map.d == 2 ? c : c >> map.logPy;
  const int* exi = ex_in + (map.d == 2 ? 0 : (size_t)kx * nz);
  int e = q_load_aligned<E / 2>(v, data + (size_t)c * ld, exi, kx & 1, lane, G, n, valid, lg, slots + si);
  ++si;
  q_fft<true, -1, true, REM, E>(v, e, buf, logP, lane, tw, logP, false, slots, si);
  const int ky = c & (map.Py - 1);
  const double* lrow = map.d == 2 ? lam + (size_t)c * map.Hy1
                                  : lam + ((size_t)kx * map.Hy1 + min(ky, map.Py - ky)) * map.Hz1;
  q_symbol<E>(v, e, lrow, [&](int m) { return min(lane + m * G, P - lane - m * G); }, map.plain, lg,
              slots + si);
  ++si;
  q_fft<true, 1, false, REM, E>(v, e, buf, logP, lane, tw, logP, true, slots, si);
  if (valid && lane == 0) FRLAP_GST(ex_out + col, e);
  store_line<E>(v, data, ncols, n, ld, logP, TL);
}

// The middle stage of a 16384-point y embedding in two halves (see k_colmul_split).  ODD = false: the even
// frequencies' half of the column into tmp; ODD = true: the odd half, added to it, in place.
template <bool ODD>
__global__ void __launch_bounds__(512, 1)
    k_q_colmul_split(cq* __restrict__ data, cq* __restrict__ tmp, const int* __restrict__ ex_in,
                     int* __restrict__ ex_out, int* __restrict__ ex_tmp, int ncols, int n, size_t ld, int TL,
                     const double* __restrict__ lam, int Hy1, bool plain, const int4* __restrict__ tw,
                     const int* __restrict__ skip, Batch bt, size_t ex_inst) {
  constexpr int logL = 13, L = 1 << logL, P = 2 * L, G = L >> 4, REM = logL & 3;
  {
    const size_t bi = blockIdx.y;
    data += bi * bt.in;
    tmp += bi * bt.out;
    lam += bi * bt.lam;
    ex_in += bi * ex_inst;
    ex_out += bi * ex_inst;
    ex_tmp += bi * ex_inst;
    if (skip) skip += bi * bt.skip;
  }
  FRLAP_Q_PROLOGUE(logL)
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int col = blockIdx.x * TL + l;
  const bool valid = col < ncols;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * sline(L);
  cq* line = data + (size_t)(valid ? col : 0) * ld;
  cq* tline = tmp + (size_t)(valid ? col : 0) * ld;
  int si = 0;
  cq v[16];
  int e = q_load_aligned<16>(v, line, ex_in, col & 1, lane, G, n, valid, logL, slots + si);
  ++si;
  if constexpr (ODD) {  // times W_P^j: from below 2^62.5 (a shift by 4) back to below 2^58.5
#pragma unroll
    for (int m = 0; m < 16; ++m)
      v[m] = q_cmul<false>(cq{q_shl(v[m].x, 4), q_shl(v[m].y, 4)}, FRLAP_GLD(tw + lane + m * G));
  }
  q_fft<true, -1, false, REM>(v, e, buf, logL, lane, tw, logL + 1, false, slots, si);
  // the half's symbol entries are every second one
  const double* lrow = lam + (size_t)(valid ? col : 0) * Hy1;
  q_symbol<16>(
      v, e, lrow,
      [&](int m) {
        const int k = 2 * (lane + m * G) + (ODD ? 1 : 0);
        return min(k, P - k);
      },
      plain, logL, slots + si);
  ++si;
  q_fft<true, 1, false, REM>(v, e, buf, logL, lane, tw, logL + 1, true, slots, si);
  if (!valid) return;
  if constexpr (!ODD) {
    if (lane == 0) FRLAP_GST(ex_tmp + col, e);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int j = lane + m * G;
      if (j < n) FRLAP_GST(tline + j, v[m]);
    }
  } else {
    // y_j = even_j + W_P^-j odd_j: the product divides by 16, and the even half is aligned to that
    const int et = FRLAP_GLD(ex_tmp + col);
    const int eo = e + 4, top = max(et + 4, eo);
    if (lane == 0) FRLAP_GST(ex_out + col, top);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int j = lane + m * G;
      if (j < n) {
        const cq o = q_cmul<true>(v[m], FRLAP_GLD(tw + j));
        FRLAP_GST(line + j, q_align(o, eo, top, col & 1) + q_align(FRLAP_GLD(tline + j), et, top, col & 1));
      }
    }
  }
}

// groups of contiguous lines of length n -> pad, FFT, transposed store out[g][k][line]
template <int REM, int LOGL, int E>
__global__ void __launch_bounds__(kQCta<E>, 1)
    k_q_c2cT_fwd(const cq* __restrict__ in, cq* __restrict__ out, const int* __restrict__ ex_in,
                 int* __restrict__ ex_out, int nlines, int tiles, int n, size_t gin, int ldi, size_t gout, int ldo,
                 int logP, int TL, const int4* __restrict__ tw, const int* __restrict__ skip, Batch bt,
                 size_t ex_inst) {
  logP = LOGL;
  constexpr int lg = q_lg<E>(LOGL);
  {
    const size_t bi = blockIdx.y;
    in += bi * bt.in;
    out += bi * bt.out;
    ex_in += bi * ex_inst;
    ex_out += bi * ex_inst;
    if (skip) skip += bi * bt.skip;
  }
  FRLAP_Q_PROLOGUE(lg)
  const int P = 1 << logP, G = P / E, LS = sline(P);
  const int g = blockIdx.x / tiles, tile = blockIdx.x % tiles;
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int line0 = tile * TL, line = line0 + l;
  const bool valid = line < nlines;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * LS;
  const int c = valid ? line : 0;
  int si = 0;
  cq v[E];
  // rows (z, y) of this line z: exponents ex_in[z n + y]
  int e = q_load_aligned<E / 2>(v, in + g * gin + (size_t)c * ldi, ex_in + (size_t)c * n, g & 1, lane, G, n, valid,
                            lg, slots + si);
  ++si;
  q_fft<true, -1, true, REM, E>(v, e, buf, logP, lane, tw, logP, false, slots, si);
  if (valid && lane == 0) FRLAP_GST(ex_out + (size_t)g * nlines + line, e);
  line_sync<double>(lg);
#pragma unroll
  for (int m = 0; m < E; ++m) buf[spad(lane + m * G)] = v[m];
  __syncthreads();
  const int logTL = __ffs(TL) - 1;
  const int lt = threadIdx.x & (TL - 1);
  if (line0 + lt < nlines) {
    const cq* trow = smem + (size_t)lt * LS;
    int k = (int)threadIdx.x >> logTL;
    cq* gp = out + g * gout + (size_t)k * ldo + line0 + lt;
    const size_t gstep = (size_t)G * ldo;
#pragma unroll 4
    for (; k < P; k += G, gp += gstep) FRLAP_GST(gp, trow[spad(k)]);
  }
}

// transposed in[g][k][line] (k < P) -> IFFT along k, crop to n, store out[g][line][i]
template <int REM, int LOGL, int E>
__global__ void __launch_bounds__(kQCta<E>, 1)
    k_q_c2cT_inv(const cq* __restrict__ in, cq* __restrict__ out, const int* __restrict__ ex_in,
                 int* __restrict__ ex_out, int nlines, int tiles, int n, size_t gin, int ldi, size_t gout, int ldo,
                 int logP, int TL, const int4* __restrict__ tw, const int* __restrict__ skip, Batch bt,
                 size_t ex_inst) {
  logP = LOGL;
  constexpr int lg = q_lg<E>(LOGL);
  {
    const size_t bi = blockIdx.y;
    in += bi * bt.in;
    out += bi * bt.out;
    ex_in += bi * ex_inst;
    ex_out += bi * ex_inst;
    if (skip) skip += bi * bt.skip;
  }
  FRLAP_Q_PROLOGUE(lg)
  const int P = 1 << logP, G = P / E, LS = sline(P);
  const int g = blockIdx.x / tiles, tile = blockIdx.x % tiles;
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int line0 = tile * TL, line = line0 + l;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * LS;
  int ek[E];
#pragma unroll
  for (int m = 0; m < E; ++m) ek[m] = FRLAP_GLD(ex_in + (size_t)g * P + lane + m * G);
  load_transposed<cq>(smem, in + g * gin, TL * P, TL, LS, ldi, line0, nlines);
  __syncthreads();
  int si = 0;
  cq v[E];
  int e = kQZero;  // (by the entries, as in q_load_aligned: a column's exponent is that of its largest line)
#pragma unroll
  for (int m = 0; m < E; ++m) {
    v[m] = buf[spad(lane + m * G)];
    e = max(e, ek[m] + q_excess(q_bits(v[m])));
  }
  e = q_unord(q_reduce<true>(q_ord(e), lg, slots + si));
  ++si;
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = q_align(v[m], ek[m], e, (lane + m * G) & 1);
  q_fft<true, 1, false, REM, E>(v, e, buf, logP, lane, tw, logP, true, slots, si);
  if (line < nlines) {
    if (lane == 0) FRLAP_GST(ex_out + (size_t)g * nlines + line, e);
    cq* dst = out + g * gout + (size_t)line * ldo;
#pragma unroll
    for (int m = 0; m < E / 2; ++m) {
      const int i = lane + m * G;
      if (i < n) FRLAP_GST(dst + i, v[m]);
    }
  }
}

// Last stage.  Bin k of row r has exponent ex[k ex_k + (r / rows_per) ].
template <int REM, int LOGL, int E>
__global__ void __launch_bounds__(kQCta<E>, 1)
    k_q_c2r(const cq* __restrict__ in, double* __restrict__ out, const int* __restrict__ ex, int ex_k, int rows_per,
            int nlines, int n, size_t ldi, int logH, int TL, const int4* __restrict__ tw,
            const int* __restrict__ skip, Batch bt, size_t ex_inst) {
  logH = LOGL;
  constexpr int lg = q_lg<E>(LOGL);
  {
    const size_t bi = blockIdx.y;
    in += bi * bt.in;
    out += bi * bt.out;
    ex += bi * ex_inst;
    if (skip) skip += bi * bt.skip;
  }
  FRLAP_Q_PROLOGUE(lg)
  const int H = 1 << logH, G = H / E, LS = sline(H);
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int line0 = blockIdx.x * TL, line = line0 + l;
  const bool valid = line < nlines;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * LS;
  // this thread's pairs (k, H - k): k = lane + j G <= H/2 (j = E/2: lane 0 alone)
  int ea[E / 2 + 1], eb[E / 2 + 1];
  const int* exl = ex + (valid ? line / rows_per : 0);
#pragma unroll
  for (int j = 0; j < E / 2 + 1; ++j) {
    const int k = lane + j * G;
    if (k <= H / 2) {
      ea[j] = FRLAP_GLD(exl + (size_t)k * ex_k);
      eb[j] = FRLAP_GLD(exl + (size_t)(H - k) * ex_k);
    }
  }
  load_transposed<cq>(smem, in, TL * (H + 1), TL, LS, ldi, line0, nlines);
  int4 wk[E / 2];  // W^k of this thread's pairs, in flight over the barrier
#pragma unroll
  for (int j = 0; j < E / 2; ++j) wk[j] = FRLAP_GLD(tw + lane + j * G);
  __syncthreads();
  int si = 0;
  // The row's exponent, at which its bins fit 60 bits, by the bins themselves: a column's exponent is that of its largest
  // row, and a row that crosses one with a high wall in another row lost what that one is above it (a wall of height 1
  // over noise of 1e-3, 2047 x 511: 1.6e-15 lambda_max ||u||, now 4.6e-16).
  int e = kQZero;
#pragma unroll
  for (int j = 0; j < E / 2 + 1; ++j) {
    const int k = lane + j * G;
    if (k <= H / 2) {
      e = max(e, ea[j] + max(4 - __clz((int)q_bits(buf[spad(k)])), 0));
      e = max(e, eb[j] + max(4 - __clz((int)q_bits(buf[spad(H - k)])), 0));
    }
  }
  e = q_unord(q_reduce<true>(q_ord(e), lg, slots + si));
  ++si;
  // Repack in place (see k_c2r_T): Z[k] = A + i T, Z[H-k] = conj(A - i T), A = X[k] + conj X[H-k],
  // T = W^-k (X[k] - conj X[H-k]), magnitudes below 2^62.5.  A product's unit is 16: where the pair leaves
  // the room, its difference goes in 16 times larger, so that small bins keep a unit of 2^-60 of the row's largest.
  // Then the line is shifted to what the transform takes, by its own largest value.
  unsigned o = 0u;
#pragma unroll
  for (int j = 0; j < E / 2 + 1; ++j) {
    const int k = lane + j * G;
    if (k <= H / 2) {
      const int km = H - k;
      const cq xk = q_align(buf[spad(k)], ea[j], e, k & 1);
      const cq b = conjg(q_align(buf[spad(km)], eb[j], e, k & 1));
      const int r = (q_bits(xk) | q_bits(b)) < (1u << 24) ? 4 : 0;
      const cq A = xk + b, d = xk - b;
      const int4 w = j < E / 2 ? wk[j & (E / 2 - 1)] : FRLAP_GLD(tw + k);
      const cq t = q_cmul<true>(cq{d.x << r, d.y << r}, w);
      const cq iT = mul_i<1>(cq{t.x << (4 - r), t.y << (4 - r)});
      const cq z0 = A + iT, z1 = conjg(A - iT);
      buf[spad(k)] = z0;
      o |= q_bits(z0);
      if (k != km && km != H) {
        buf[spad(km)] = z1;
        o |= q_bits(z1);
      }
    }
  }
  o = q_publish<false>(o, lg, slots + si);
  line_sync<double>(lg);
  const int drop = q_excess(q_fetch(o, lg, slots + si));
  ++si;
  cq v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = q_align(buf[spad(lane + m * G)], 0, drop, (lane + m * G) & 1);
  e += drop;
  q_fft<true, 1, false, REM, E>(v, e, buf, logH, lane, tw, logH + 1, true, slots, si);
  if (!valid) return;
  double* dst = out + (size_t)line * n;
  const bool pair_aligned = (reinterpret_cast<uintptr_t>(dst) % sizeof(double2)) == 0;
#pragma unroll
  for (int m = 0; m < E / 2; ++m) {
    const int q = lane + m * G;
    if (2 * q < n) {
      const double a = q_out_any(v[m].x, e), b = q_out_any(v[m].y, e);
      if (pair_aligned && 2 * q + 1 < n) {
        FRLAP_GST(reinterpret_cast<double2*>(dst + 2 * q), make_double2(a, b));
      } else {
        FRLAP_GST(dst + 2 * q, a);
        if (2 * q + 1 < n) FRLAP_GST(dst + 2 * q + 1, b);
      }
    }
  }
}

}  // namespace
}  // namespace frlap

namespace frlap {

// Workspace arrays of one instance: S1, S2 (16-byte complex entries), then the exponents.
struct QWork {
  cq* S1;
  cq* S2;
  int *row, *line, *col;
  size_t stride;     // to the next instance, in complex entries
  size_t ex_stride;  // the same in ints
};
inline QWork q_work(const Plan& p, void* work) {
  unsigned char* w = reinterpret_cast<unsigned char*>(work);
  const QExpLayout l = q_exp_layout(p);
  QWork q;
  q.S1 = reinterpret_cast<cq*>(w);
  q.S2 = reinterpret_cast<cq*>(w + align256(p.s1_elems * 16));
  int* ex = reinterpret_cast<int*>(w + align256(p.s1_elems * 16) + align256(p.s2_elems * 16));
  q.row = ex + l.row;
  q.line = ex + l.line;
  q.col = ex + l.col;
  q.stride = apply_work_bytes(p, 8) / 16;
  q.ex_stride = q.stride * 4;
  return q;
}

// One launch: the kernel's shared memory limit, then the grid of (tiles, instances).
template <typename K, typename... A>
static cudaError_t q_launch(K kern, unsigned grid, int B, int threads, size_t sm, cudaStream_t s, A... args) {
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  kern<<<dim3(grid, B), threads, sm, s>>>(args...);
  return cudaGetLastError();
}

// Lines per CTA and the launch numbers that follow, for `lines` lines (per group: `tiles`) of length L.
struct QShape {
  int tl, threads, tiles;
  size_t sm;
  int e;  // entries a thread
};
// Entries a thread.  Sixteen (the fewest stages, exchanges and barriers) for launches that fill the chip.  Fewer
// where, at sixteen, a vector's lines leave most of the 608 sub-partitions without a warp: then a thread's chain of
// instructions is the time.  The lines depend on the plan alone, so that a batch equals its vectors' applies bit for
// bit; a batch of 8 at the first line still has at most a warp per sub-partition.  One F64 vector, us per stage (with
// its launch; r2c, colmul, c2r), sixteen -> four: 32^2 12.2, 10.8, 10.2 -> 9.6, 7.9, 7.2, 128^2 13.1, 11.9, 10.2 ->
// 10.6, 8.9, 8.2; 8 x 128^2 4.7 -> 4.1 a vector.  Sixteen -> eight: 256^2 14.2, 14.9, 11.6 -> 11.7, 11.3, 10.2; above
// the second line the further stage costs more: 512^2 colmul 17.0 -> 19.3, 8 x 255^2 3.2 -> 3.4
// a vector, 8 x 2048^2 165 -> 206 a vector.  Rows of at most
// 128 points are bound by their loads and conversions: with eight entries and twice the warps 128^3 r2c 36.9 -> 33.0,
// c2r 32.7 -> 28.7.
constexpr long long kQThin4 = 152 * 16, kQThin8 = 152 * 64;
enum class QKind { Line, Row, Split };
static QShape q_shape(int tuned, int L, long long lines, int B, int lines_per_group, QKind k = QKind::Line) {
  QShape q;
  const long long t16 = lines * (L >> 4);
  q.e = k == QKind::Split || L > (1 << kQThinLog) ? 16
        : t16 <= kQThin4                          ? 4
        : t16 <= kQThin8 || (k == QKind::Row && L <= 128) ? 8
                                                          : 16;
  const int G = L / q.e;
  q.tl = pick_tl_tuned(q.e == 4 ? 0 : tuned, sline(L), 16, G, 96 * 1024, lines * B);
  while (q.tl > 1 && q.tl * G > 512) q.tl /= 2;  // (a tuned choice is one for sixteen entries)
  q.threads = q.tl * G;
  q.tiles = (lines_per_group + q.tl - 1) / q.tl;
  q.sm = (size_t)q.tl * sline(L) * 16;
  return q;
}

// The shape of apply stage st: 2D rows, middle, rows; 3D rows, y lines, middle, y lines, rows.
static QShape q_stage_shape(const Plan& p, int st, int tuned, int B) {
  const int Hx1 = p.P[0] / 2 + 1, nrows = p.n[1] * p.n[2];
  if (st == 0 || st == (p.d == 2 ? 2 : 4)) return q_shape(tuned, p.P[0] / 2, nrows, B, nrows, QKind::Row);
  if (p.d == 3 && st != 2) return q_shape(tuned, p.P[1], (long long)p.n[2] * Hx1, B, p.n[2]);
  if (p.d == 2 && p.P[1] > kMaxLine) return q_shape(tuned, kMaxLine, Hx1, B, Hx1, QKind::Split);
  const int ncols = p.d == 3 ? Hx1 * p.P[1] : Hx1;
  return q_shape(tuned, p.P[p.d - 1], ncols, B, ncols);
}
template <typename T>
int q_stage_tl(const Plan& p, int st, int tuned, int B) {
  return q_stage_shape(p, st, tuned, B).tl;
}

// f(tag) for the kernel instance of a line of 2^logL points: tag::rem, tag::logp and tag::e entries a thread.
template <int R, int L, int E>
struct QTag : ShapeTag<R, L> {
  static constexpr int e = E;
};
template <typename F>
static cudaError_t q_with_shape(const QShape& q, int logL, F&& f) {
  return with_line_shape(logL, [&](auto tag) {
    constexpr int R = decltype(tag)::rem, L = decltype(tag)::logp;
    if constexpr (L <= kQThinLog) {
      if (q.e == 4) return f(QTag<R, L, 4>{});
      if (q.e == 8) return f(QTag<R, L, 8>{});
    }
    return f(QTag<R, L, 16>{});
  });
}

static LamMap q_lam_map(const Plan& p) {
  LamMap map;
  map.d = p.d;
  map.Hx1 = p.P[0] / 2 + 1;
  map.logPy = p.logP[1];
  map.Py = p.P[1];
  map.Hy1 = p.P[1] / 2 + 1;
  map.Hz1 = p.d == 3 ? p.P[2] / 2 + 1 : 1;
  map.plain = p.lam_plain;
  return map;
}

#ifdef FRLAP_BOUNDS_CHECK
static cudaError_t q_register(const Plan& p, BcRanges r, void* work, int B, cudaStream_t s) {
  r.add(work, (size_t)B * apply_work_bytes(p, 8));
  for (int a = 0; a < p.d; ++a) r.add(p.twq[a], (size_t)twq_entries(p.P[a]) * sizeof(int4));
  return r.commit(s);
}
#endif

// The stages, one launch each over B instances (per-instance strides in elements).
template <bool DYN>
static cudaError_t q_stage_r2c(const Plan& p, const QWork& w, int B, const double* u, size_t ustride, int tuned,
                               const int* skip, int skip_stride, cudaStream_t s) {
  const int nrows = p.n[1] * p.n[2];
  const QShape q = q_stage_shape(p, 0, tuned, B);
  Batch b;
  b.in = ustride;
  b.out = w.stride;
  b.skip = skip_stride;
  return q_with_shape(q, p.logP[0] - 1, [&](auto tag) {
    using K = decltype(tag);
    return q_launch(k_q_r2c<DYN || ((1 << K::logp) > kQStaticMax), K::rem, K::logp, K::e>, q.tiles, B, q.threads, q.sm, s, u, w.S1, w.row,
                    nrows, p.n[0], (size_t)nrows, p.logP[0] - 1, q.tl, (const int4*)p.twq[0], skip, b, w.ex_stride);
  });
}
static cudaError_t q_stage_yz_fwd(const Plan& p, const QWork& w, int B, int tuned, const int* skip, int skip_stride,
                                  cudaStream_t s) {
  const int Py = p.P[1], ny = p.n[1], nz = p.n[2], Hx1 = p.P[0] / 2 + 1;
  const QShape q = q_stage_shape(p, 1, tuned, B);
  Batch b;
  b.in = b.out = w.stride;
  b.skip = skip_stride;
  return q_with_shape(q, p.logP[1], [&](auto tag) {
    using K = decltype(tag);
    return q_launch(k_q_c2cT_fwd<K::rem, K::logp, K::e>, Hx1 * q.tiles, B, q.threads, q.sm, s, (const cq*)w.S1,
                    w.S2, (const int*)w.row, w.line, nz, q.tiles, ny, (size_t)nz * ny, ny, (size_t)Py * nz, nz, p.logP[1],
                    q.tl, (const int4*)p.twq[1], skip, b, w.ex_stride);
  });
}
static cudaError_t q_stage_yz_inv(const Plan& p, const QWork& w, int B, int tuned, const int* skip, int skip_stride,
                                  cudaStream_t s) {
  const int Py = p.P[1], ny = p.n[1], nz = p.n[2], Hx1 = p.P[0] / 2 + 1;
  const QShape q = q_stage_shape(p, 1, tuned, B);
  Batch b;
  b.in = b.out = w.stride;
  b.skip = skip_stride;
  return q_with_shape(q, p.logP[1], [&](auto tag) {
    using K = decltype(tag);
    return q_launch(k_q_c2cT_inv<K::rem, K::logp, K::e>, Hx1 * q.tiles, B, q.threads, q.sm, s, (const cq*)w.S2,
                    w.S1, (const int*)w.col, w.line, nz, q.tiles, ny, (size_t)Py * nz, nz, (size_t)nz * ny, ny, p.logP[1],
                    q.tl, (const int4*)p.twq[1], skip, b, w.ex_stride);
  });
}
static cudaError_t q_stage_c2r(const Plan& p, const QWork& w, int B, double* y, size_t ystride, int tuned,
                               const int* skip, int skip_stride, cudaStream_t s) {
  const int nrows = p.n[1] * p.n[2];
  const QShape q = q_stage_shape(p, p.d == 2 ? 2 : 4, tuned, B);
  Batch b;
  b.in = w.stride;
  b.out = ystride;
  b.skip = skip_stride;
  return q_with_shape(q, p.logP[0] - 1, [&](auto tag) {
    using K = decltype(tag);
    return q_launch(k_q_c2r<K::rem, K::logp, K::e>, q.tiles, B, q.threads, q.sm, s, (const cq*)w.S1, y,
                    (const int*)(p.d == 3 ? w.line : w.col), p.d == 3 ? p.n[2] : 1, p.d == 3 ? p.n[1] : nrows, nrows,
                    p.n[0], (size_t)nrows, p.logP[0] - 1, q.tl, (const int4*)p.twq[0], skip, b, w.ex_stride);
  });
}

template <typename T>
cudaError_t q_apply_launch_b(const Plan& p, int B, const double* u, double* y, size_t vstride, void* work,
                             cudaStream_t s, const int* skip, int skip_stride, cudaEvent_t const* ev,
                             const double* lam_override, size_t lam_stride) {
  constexpr bool DYN = std::is_same<T, double>::value;
  int stage = 0;
  auto mark = [&]() -> cudaError_t {
    if (ev && ev[stage]) {
      cudaError_t e = cudaEventRecord(ev[stage], s);
      if (e != cudaSuccess) return e;
    }
    ++stage;
    return cudaSuccess;
  };
  const int* tuned = p.tl_tuned[engine_index<T>()];
  const double* lam = lam_override ? lam_override : p.lamL64;
  const QWork w = q_work(p, work);
  const int ny = p.n[1], nz = p.n[2], Hx1 = p.P[0] / 2 + 1, nrows = ny * nz;
  const LamMap map = q_lam_map(p);
  cudaError_t e;
#ifdef FRLAP_BOUNDS_CHECK
  {
    BcRanges r;
    const size_t vext = ((size_t)(B - 1) * vstride + p.M) * sizeof(double);
    r.add(u, vext);
    r.add(y, vext);
    r.add(lam, ((size_t)(B - 1) * lam_stride + p.lam_count) * sizeof(double));
    if (skip) r.add(skip, ((size_t)(B - 1) * skip_stride + 1) * sizeof(int));
    if ((e = q_register(p, r, work, B, s)) != cudaSuccess) return e;
  }
#endif
  Batch b;
  b.in = b.out = w.stride;
  b.lam = lam_stride;
  b.skip = skip_stride;
  if ((e = mark()) != cudaSuccess) return e;
  if ((e = q_stage_r2c<DYN>(p, w, B, u, vstride, tuned[0], skip, skip_stride, s)) != cudaSuccess) return e;
  if ((e = mark()) != cudaSuccess) return e;
  if (p.d == 2 && p.P[1] > kMaxLine) {
    const QShape q = q_stage_shape(p, 1, tuned[1], B);
    int* ex_tmp = w.col + Hx1;
    e = q_launch(k_q_colmul_split<false>, q.tiles, B, q.threads, q.sm, s, w.S1, w.S2, (const int*)w.row, w.col, ex_tmp,
                 Hx1, ny, (size_t)nrows, q.tl, lam, map.Hy1, map.plain, (const int4*)p.twq[1], skip, b, w.ex_stride);
    if (e == cudaSuccess)
      e = q_launch(k_q_colmul_split<true>, q.tiles, B, q.threads, q.sm, s, w.S1, w.S2, (const int*)w.row, w.col,
                   ex_tmp, Hx1, ny, (size_t)nrows, q.tl, lam, map.Hy1, map.plain, (const int4*)p.twq[1], skip, b, w.ex_stride);
    if (e != cudaSuccess) return e;
  } else {
    if (p.d == 3) {
      if ((e = q_stage_yz_fwd(p, w, B, tuned[1], skip, skip_stride, s)) != cudaSuccess) return e;
      if ((e = mark()) != cudaSuccess) return e;
    }
    // the middle stage: columns over y in S1 (2D), over z in S2 (3D)
    const int ax = p.d == 3 ? 2 : 1;
    const int ncols = p.d == 3 ? Hx1 * p.P[1] : Hx1;
    const QShape q = q_stage_shape(p, ax, tuned[ax], B);
    e = q_with_shape(q, p.logP[ax], [&](auto tag) {
      using K = decltype(tag);
      return q_launch(k_q_colmul<K::rem, K::logp, K::e>, q.tiles, B, q.threads, q.sm, s, p.d == 3 ? w.S2 : w.S1,
                      (const int*)(p.d == 3 ? w.line : w.row), w.col, ncols, p.n[ax], (size_t)(p.d == 3 ? nz : nrows),
                      p.logP[ax], q.tl, lam, map, nz, (const int4*)p.twq[ax], skip, b, w.ex_stride);
    });
    if (e != cudaSuccess) return e;
    if (p.d == 3) {
      if ((e = mark()) != cudaSuccess) return e;
      if ((e = q_stage_yz_inv(p, w, B, tuned[3], skip, skip_stride, s)) != cudaSuccess) return e;
    }
  }
  if ((e = mark()) != cudaSuccess) return e;
  if ((e = q_stage_c2r(p, w, B, y, vstride, tuned[p.d == 2 ? 2 : 4], skip, skip_stride, s)) != cudaSuccess) return e;
  return mark();
}

}  // namespace frlap
