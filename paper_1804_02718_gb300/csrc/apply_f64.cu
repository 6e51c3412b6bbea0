// The FP64 and DF64 engines' apply and the spectrum transforms of the learned preconditioner (kernels and launchers in
// apply_q.cuh, dispatch in apply_impl.cuh), plus the engine-independent entry points.
#include "apply_q.cuh"

namespace frlap {

size_t apply_spectra_bytes(const Plan& p, int real_bytes) {
  const size_t cb = 2 * (size_t)real_bytes;
  return align256(p.s1_elems * cb) + align256(p.s2_elems * cb);
}

size_t apply_work_bytes(const Plan& p, int real_bytes) {
  size_t b = apply_spectra_bytes(p, real_bytes);
  if (real_bytes == 8) b += q_exp_layout(p).total * sizeof(int);  // the fixed-point engines' exponents
  return b;
}

cudaError_t apply64(const Plan& p, const double* u, double* y, void* work, cudaStream_t s, const int* skip,
                    cudaEvent_t const* ev) {
  if (p.df64) return apply_launch<df64>(p, u, y, work, s, skip, ev, nullptr);
  return apply_launch<double>(p, u, y, work, s, skip, ev, nullptr);
}

template cudaError_t apply_batch_launch<double>(const Plan&, int, const double*, double*, size_t, void*, cudaStream_t,
                                                const int*, int, const double*, size_t, cudaEvent_t const*);
template cudaError_t apply_launch<double>(const Plan&, const double*, double*, void*, cudaStream_t, const int*,
                                          cudaEvent_t const*, const double*, bool);
template cudaError_t apply_batch_launch<df64>(const Plan&, int, const double*, double*, size_t, void*, cudaStream_t,
                                              const int*, int, const double*, size_t, cudaEvent_t const*);
template cudaError_t apply_launch<df64>(const Plan&, const double*, double*, void*, cudaStream_t, const int*,
                                        cudaEvent_t const*, const double*, bool);

size_t spectrum_elems(const Plan& p) {
  const size_t Hx1 = p.P[0] / 2 + 1;
  return (p.d == 2) ? Hx1 * p.P[1] : Hx1 * p.P[1] * p.P[2];
}

namespace {

// Spectrum columns of the learned preconditioner: columns of n entries -> zero-pad to P, forward FFT, all P
// outputs in FP64 (stride ldo).
template <int REM, int LOGP, int E>
__global__ void __launch_bounds__(kQCta<E>, 1)
    k_q_col_fwd(const cq* __restrict__ in, const int* __restrict__ ex, double2* __restrict__ out, int ncols, int n,
                size_t ld, size_t ldo, int logP, int TL, int cols_per, const int4* __restrict__ tw,
                const int* __restrict__ skip, Batch bt, size_t ex_inst) {
  in += blockIdx.y * bt.in;
  out += blockIdx.y * bt.out;
  ex += blockIdx.y * ex_inst;
  logP = LOGP;
  constexpr int lg = q_lg<E>(LOGP);
  FRLAP_Q_PROLOGUE(lg)
  const int P = 1 << logP, G = P / E;
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int col = blockIdx.x * TL + l;
  const bool valid = col < ncols;
  const int c = valid ? col : 0;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * sline(P);
  int si = 0;
  cq v[E];
  // exponents: 2D ex[i] for every column; 3D ex[(col / P_y) n + i]
  const int kx = cols_per ? c / cols_per : c;
  int e = q_load_aligned<E / 2>(v, in + (size_t)c * ld, ex + (cols_per ? (size_t)kx * n : 0), kx & 1, lane, G, n, valid,
                            lg, slots + si);
  ++si;
  q_fft<true, -1, true, REM, E>(v, e, buf, logP, lane, tw, logP, false, slots, si);
  if (!valid) return;
  double2* dst = out + (size_t)col * ldo;
#pragma unroll
  for (int m = 0; m < E; ++m)
    FRLAP_GST(dst + lane + m * G, make_double2(q_out_any(v[m].x, e), q_out_any(v[m].y, e)));
}

// Columns of P FP64 spectrum values times a multiplier (natural octant order) -> inverse FFT, crop to n.
template <int REM, int LOGP, int E>
__global__ void __launch_bounds__(kQCta<E>, 1)
    k_q_col_mulinv(const double2* __restrict__ in, cq* __restrict__ out, int* __restrict__ ex, int ncols, int n,
                   size_t ld, size_t ldo, int logP, int TL, const double* __restrict__ lam, LamMap map,
                   const int4* __restrict__ tw, const int* __restrict__ skip, Batch bt, size_t ex_inst) {
  in += blockIdx.y * bt.in;
  out += blockIdx.y * bt.out;
  ex += blockIdx.y * ex_inst;
  logP = LOGP;
  constexpr int lg = q_lg<E>(LOGP);
  FRLAP_Q_PROLOGUE(lg)
  const int P = 1 << logP, G = P / E;
  const int l = threadIdx.x / G, lane = threadIdx.x % G;
  const int col = blockIdx.x * TL + l;
  const bool valid = col < ncols;
  const int c = valid ? col : 0;
  unsigned* slots = q_slot_words + (l & (kQLines - 1)) * kQSlots;
  cq* buf = smem + (size_t)l * sline(P);
  const double2* src = in + (size_t)c * ld;
  size_t lam_base;
  int lam_stride;
  if (map.d == 2) {
    lam_base = c;
    lam_stride = map.Hx1;
  } else {
    const int kx = c >> map.logPy, ky = c & (map.Py - 1);
    lam_base = (size_t)min(ky, map.Py - ky) * map.Hx1 + kx;
    lam_stride = map.Hy1 * map.Hx1;
  }
  double2 x[E];
  unsigned hm = 0u;
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int k = lane + m * G;
    x[m] = valid ? FRLAP_GLD(lam + lam_base + (size_t)min(k, P - k) * lam_stride) * FRLAP_GLD(src + k)
                 : make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int m = 0; m < E; ++m) hm = max(hm, max(q_mag(x[m].x), q_mag(x[m].y)));
  int si = 0;
  const QIn qs = q_in_scale(q_reduce<true>(hm, lg, slots + si));
  ++si;
  cq v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = {q_in(x[m].x, qs), q_in(x[m].y, qs)};
  int e = qs.e;
  q_fft<true, 1, false, REM, E>(v, e, buf, logP, lane, tw, logP, false, slots, si);
  if (valid && lane == 0) FRLAP_GST(ex + col, e);
  store_line<E>(v, out, ncols, n, ldo, logP, TL);
}

}  // namespace

// SP = F R^T u on the half spectrum in FP64: 2D [kx][ky], 3D [kx][ky][kz] (kx <= P_x/2, full ky, kz).
cudaError_t spectrum_forward(const Plan& p, int nb, const double* u, double2* SP, size_t sstride, void* work,
                             cudaStream_t s) {
  cudaError_t e;
#ifdef FRLAP_BOUNDS_CHECK
  {
    BcRanges r;
    r.add(u, nb * p.M * sizeof(double));
    r.add(SP, nb * sstride * sizeof(double2));
    if ((e = q_register(p, r, work, nb, s)) != cudaSuccess) return e;
  }
#endif
  const QWork w = q_work(p, work);
  if ((e = q_stage_r2c<true>(p, w, nb, u, p.M, 0, nullptr, 0, s)) != cudaSuccess) return e;
  if (p.d == 3 && (e = q_stage_yz_fwd(p, w, nb, 0, nullptr, 0, s)) != cudaSuccess) return e;
  const int ax = p.d == 3 ? 2 : 1, Hx1 = p.P[0] / 2 + 1, nrows = p.n[1] * p.n[2];
  const int ncols = p.d == 3 ? Hx1 * p.P[1] : Hx1;
  const QShape q = q_shape(0, p.P[ax], (long long)ncols, nb, ncols);
  Batch b;
  b.in = w.stride;
  b.out = sstride;
  return q_with_shape(q, p.logP[ax], [&](auto tag) {
    using K = decltype(tag);
    return q_launch(k_q_col_fwd<K::rem, K::logp, K::e>, q.tiles, nb, q.threads, q.sm, s,
                    (const cq*)(p.d == 3 ? w.S2 : w.S1), (const int*)(p.d == 3 ? w.line : w.row), SP, ncols, p.n[ax],
                    (size_t)(p.d == 3 ? p.n[2] : nrows), (size_t)p.P[ax], p.logP[ax], q.tl, p.d == 3 ? p.P[1] : 0,
                    (const int4*)p.twq[ax], (const int*)nullptr, b, w.ex_stride);
  });
}

// y = R F^-1 (mult * SP), mult = a symbol octant with the 1/prod(P) factor folded in.
cudaError_t spectrum_inverse(const Plan& p, int nb, const double2* SP, size_t sstride, const double* mult, double* y,
                             void* work, cudaStream_t s) {
  cudaError_t e;
#ifdef FRLAP_BOUNDS_CHECK
  {
    BcRanges r;
    r.add(SP, nb * sstride * sizeof(double2));
    r.add(mult, p.lam_count * sizeof(double));
    r.add(y, nb * p.M * sizeof(double));
    if ((e = q_register(p, r, work, nb, s)) != cudaSuccess) return e;
  }
#endif
  const QWork w = q_work(p, work);
  const int ax = p.d == 3 ? 2 : 1, Hx1 = p.P[0] / 2 + 1, nrows = p.n[1] * p.n[2];
  const int ncols = p.d == 3 ? Hx1 * p.P[1] : Hx1;
  const QShape q = q_shape(0, p.P[ax], (long long)ncols, nb, ncols);
  const LamMap map = q_lam_map(p);
  Batch b;
  b.in = sstride;
  b.out = w.stride;
  e = q_with_shape(q, p.logP[ax], [&](auto tag) {
    using K = decltype(tag);
    return q_launch(k_q_col_mulinv<K::rem, K::logp, K::e>, q.tiles, nb, q.threads, q.sm, s, SP, p.d == 3 ? w.S2 : w.S1,
                    w.col, ncols, p.n[ax], (size_t)p.P[ax], (size_t)(p.d == 3 ? p.n[2] : nrows), p.logP[ax], q.tl, mult,
                    map, (const int4*)p.twq[ax], (const int*)nullptr, b, w.ex_stride);
  });
  if (e != cudaSuccess) return e;
  if (p.d == 3 && (e = q_stage_yz_inv(p, w, nb, 0, nullptr, 0, s)) != cudaSuccess) return e;
  return q_stage_c2r(p, w, nb, y, p.M, 0, nullptr, 0, s);
}

template cudaError_t autotune_engine<double>(Plan&, int, double*, double*, void*, cudaStream_t);
template cudaError_t autotune_engine<df64>(Plan&, int, double*, double*, void*, cudaStream_t);

template cudaError_t bc_collect<double>(unsigned long long*, unsigned long long*);

#ifdef FRLAP_BOUNDS_CHECK
static __device__ double g_bc_probe[16];

// 8 loads inside the registered range, 5 just past it (still inside g_bc_probe, so harmless
// whether or not the checks skip them), one store to the registered sink
__global__ void k_bc_selftest(const double* buf, double* sink) {
  double s = 0.0;
  for (int i = 0; i < 8; ++i) s += FRLAP_GLD(buf + i);
  for (int i = 8; i < 13; ++i) s += FRLAP_GLD(buf + i);
  FRLAP_GST(sink, s);
}
#endif

cudaError_t bc_selftest(unsigned long long* flagged) {
#ifdef FRLAP_BOUNDS_CHECK
  unsigned long long c = 0, f = 0;
  cudaError_t e = bc_collect<double>(&c, &f);  // reset
  double* probe = nullptr;
  if (e == cudaSuccess) e = cudaGetSymbolAddress(reinterpret_cast<void**>(&probe), g_bc_probe);
  if (e != cudaSuccess) return e;
  BcRanges r;
  r.add(probe, 8 * sizeof(double));
  r.add(probe + 15, sizeof(double));
  if ((e = r.commit(nullptr)) != cudaSuccess) return e;
  k_bc_selftest<<<1, 1>>>(probe, probe + 15);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) return e;
  e = bc_collect<double>(&c, &f);
  *flagged = c;
  if (e == cudaSuccess && c > 0 && f != reinterpret_cast<unsigned long long>(probe + 8)) *flagged = ~0ull;
  return e;
#else
  *flagged = 0ull;
  return cudaErrorNotSupported;
#endif
}

}  // namespace frlap
