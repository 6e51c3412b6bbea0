// The FP64 engine's apply and the spectrum transforms of the learned preconditioner (kernels and launchers in
// apply_q.cuh, dispatch in apply_impl.cuh), plus the engine-independent entry points.
#include "apply_q.cuh"

namespace frlap {

// instantiated in apply_dfl.cu
extern template cudaError_t apply_launch<dfl>(const Plan&, const double*, double*, void*, cudaStream_t, const int*,
                                              cudaEvent_t const*, const dfl*, bool);

size_t apply_work_bytes(const Plan& p, int real_bytes) {
  const size_t cb = 2 * (size_t)real_bytes;
  size_t b = align256(p.s1_elems * cb);
  b += align256(p.s2_elems * cb);
  if (real_bytes == 8) b += q_exp_layout(p).total * sizeof(int);  // the FP64 engine's exponents
  return b;
}

cudaError_t apply64(const Plan& p, const double* u, double* y, void* work, cudaStream_t s, const int* skip,
                    cudaEvent_t const* ev) {
  if (p.df64) return apply_launch<dfl>(p, u, y, work, s, skip, ev, nullptr);
  return apply_launch<double>(p, u, y, work, s, skip, ev, nullptr);
}

template cudaError_t apply_batch_launch<double>(const Plan&, int, const double*, double*, size_t, void*, cudaStream_t,
                                                const int*, int, const double*, size_t, cudaEvent_t const*);
template cudaError_t apply_launch<double>(const Plan&, const double*, double*, void*, cudaStream_t, const int*,
                                          cudaEvent_t const*, const double*, bool);

size_t spectrum_elems(const Plan& p) {
  const size_t Hx1 = p.P[0] / 2 + 1;
  return (p.d == 2) ? Hx1 * p.P[1] : Hx1 * p.P[1] * p.P[2];
}

template cudaError_t autotune_engine<double>(Plan&, int, double*, double*, void*, cudaStream_t);

template cudaError_t bc_collect<double>(unsigned long long*, unsigned long long*);
template cudaError_t wait_collect<double>(unsigned long long*);

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

// The give-up path of the bounded mbarrier wait: one warp waits on a phase that nothing
// completes (no arrival, no copy in flight), gives up after the wait's bound, and records it.
__global__ void k_wait_selftest() {
  __shared__ unsigned long long bar;
  if (threadIdx.x == 0) mbar_init(&bar, 1);
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0u);
  if (!__syncthreads_and(ok) && threadIdx.x == 0) atomicAdd(&g_wait_timeouts, 1ull);
}

cudaError_t wait_selftest(unsigned long long* timeouts) {
  unsigned long long c = 0;
  cudaError_t e = wait_collect<double>(&c);  // reset
  if (e != cudaSuccess) return e;
  k_wait_selftest<<<1, 32>>>();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) return e;
  return wait_collect<double>(timeouts);
}

}  // namespace frlap
