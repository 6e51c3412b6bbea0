// The learned Fourier-multiplier preconditioner: a per-frequency MLP over
// (alpha, kappa_x, kappa_y, kappa_z), kappa_r = k_r / (P_r/2) on the symbol octant,
// two tanh layers of 64 units, output s; multiplier m(k) = exp(s(k)) / lambda(k)
// (lambda = A's embedding symbol, so a zero network is the inverse-embedding
// preconditioner).  M^-1 r = R F^-1 (m . F R^T r).
//
// Training pairs (r_b, e_b = A^-1 r_b) come from the plain CG solver.  The loss is
// the relative A-norm error of z_b = M^-1 r_b as an approximation of e_b:
//   L = mean_b ||e_b - z_b||_A^2 / ||e_b||_A^2 = mean_b (1 - 2 a_b / c_b + b_b / c_b),
//   a = r.z,  b = z.Az,  c = r.e.
// (For the untrained network M A >= I, with most eigenvalues at 1, so the loss pins the
// overall scale of M; a per-pair scale-free form let bands of frequencies rescale
// independently and spread the spectrum of M A.)
// With ^ the P-point DFT of a zero-padded field, R = r^, W = (Az)^:
//   dL/dm(k) = mean_b [ -(2/c) |R(k)|^2 + (1/c) 2 Re(conj(W(k)) R(k)) ] / prod(P),
// summed over the mirror images of each octant entry, and dL/ds(k) = dL/dm(k) m(k);
// the network gradient follows by backpropagation.
// Spectra and residuals are FP64; the network is FP32 (weights, activations),
// its gradient is reduced in FP64.
#include <math.h>

#include "common.cuh"

namespace frlap {

namespace {

constexpr int HID = FRLAP_MLP_HIDDEN;
constexpr int NF = FRLAP_MLP_NFEAT;
constexpr int NPAR = FRLAP_MLP_NPARAM;
// parameter offsets (W1 [HID][NF], b1, W2 [HID][HID] (out, in), b2, w3, b3)
constexpr int OW1 = 0, OB1 = OW1 + HID * NF, OW2 = OB1 + HID, OB2 = OW2 + HID * HID, OW3 = OB2 + HID,
              OB3 = OW3 + HID;
static_assert(OB3 + 1 == NPAR, "parameter layout");

struct Oct {
  int d;
  int Hx1, Hy1, Hz1;  // octant extents
  float ix, iy, iz;   // 1 / (P_r / 2)
  float alpha;
};

__device__ __forceinline__ void features(const Oct& o, size_t f, float* phi) {
  const int kx = (int)(f % o.Hx1);
  const int ky = (int)((f / o.Hx1) % o.Hy1);
  const int kz = (int)(f / ((size_t)o.Hx1 * o.Hy1));
  phi[0] = o.alpha;
  phi[1] = kx * o.ix;
  phi[2] = ky * o.iy;
  phi[3] = (o.d == 3) ? kz * o.iz : 0.0f;
}

// m(f) = exp(s(f)) / lambda(f); optional caches of the two hidden layers for backprop, [HID][F] so that a
// warp's stores of one unit are contiguous.  The weights are read four per shared-memory load (one per load
// took 98 us at 257 x 257 entries).
__global__ void __launch_bounds__(128) k_mlp_fwd(const float* __restrict__ params, Oct o, const double* __restrict__ lam,
                                                 double lamscale, size_t F, double* m, double* m_scaled,
                                                 double mscale, float* h1c, float* h2c) {
  __shared__ __align__(16) float W[NPAR + 3];
  for (int i = threadIdx.x; i < NPAR; i += blockDim.x) W[i] = params[i];
  __syncthreads();
  const size_t f = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  float phi[NF];
  features(o, f, phi);
  float h1[HID];
  static_assert(NF == 4 && OW1 % 4 == 0 && OW2 % 4 == 0 && HID % 4 == 0, "float4 rows");
#pragma unroll
  for (int h = 0; h < HID; ++h) {
    const float4 w = *reinterpret_cast<const float4*>(&W[OW1 + h * NF]);
    float a = W[OB1 + h];
    a = fmaf(w.x, phi[0], a);
    a = fmaf(w.y, phi[1], a);
    a = fmaf(w.z, phi[2], a);
    a = fmaf(w.w, phi[3], a);
    h1[h] = tanhf(a);
    if (h1c) h1c[h * F + f] = h1[h];
  }
  float s = W[OB3];
#pragma unroll 2
  for (int q = 0; q < HID; ++q) {
    float a = W[OB2 + q];
#pragma unroll
    for (int i = 0; i < HID; i += 4) {
      const float4 w = *reinterpret_cast<const float4*>(&W[OW2 + q * HID + i]);
      a = fmaf(w.x, h1[i], a);
      a = fmaf(w.y, h1[i + 1], a);
      a = fmaf(w.z, h1[i + 2], a);
      a = fmaf(w.w, h1[i + 3], a);
    }
    const float h2 = tanhf(a);
    if (h2c) h2c[q * F + f] = h2;
    s = fmaf(W[OW3 + q], h2, s);
  }
  const double l = lam[f] * lamscale;
  const double mv = (l > 0.0) ? exp((double)s) / l : 0.0;
  m[f] = mv;
  if (m_scaled) m_scaled[f] = mv * mscale;
}

// Gradient of sum_f g_s(f) s(f), g_s = g_m * m.  A CTA walks tiles of BENT = 64 entries; per tile the two
// 64 x 64 x 64 products run as register tiles (4 x 4 outputs a thread, operands four per load; one operand
// per load was 115 us at 257 x 257 entries), their FP32 sums over the tile's entries added to FP64
// accumulators in registers.  partial[CTA][NPAR].
constexpr int BENT = 64, BST = BENT + 4;  // row stride of a tile in shared memory: 16-byte rows, spread banks
constexpr int kBwdCtas = 304;
constexpr size_t kBwdSmem = (size_t)(HID * BST + 4 * BENT * BST + BENT * NF + BENT) * sizeof(float);
__global__ void __launch_bounds__(256, 2) k_mlp_bwd(const float* __restrict__ params, Oct o,
                                                    const double* __restrict__ g_m, const double* __restrict__ m,
                                                    const float* __restrict__ h1c, const float* __restrict__ h2c,
                                                    size_t F, double* partial) {
  static_assert(HID == 64 && BENT == 64, "16 x 16 threads of 4 x 4 outputs");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* W2 = reinterpret_cast<float*>(smem_raw);  // [q][h]
  float* sh1 = W2 + HID * BST;                     // [e][h] (and the next three)
  float* sh2 = sh1 + BENT * BST;
  float* sga2 = sh2 + BENT * BST;
  float* sga1 = sga2 + BENT * BST;
  float* sphi = sga1 + BENT * BST;                 // [e][NF]
  float* sgs = sphi + BENT * NF;                   // [e]
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  for (int i = t; i < HID * HID; i += 256) W2[(i >> 6) * BST + (i & 63)] = params[OW2 + i];
  double acc2[4][4] = {};  // W2[4 ty + i][4 tx + j]
  double acc1 = 0.0;       // W1[t / NF][t % NF]
  double accb = 0.0;       // t < 64: b1, < 128: b2, < 192: w3, 192: b3
  const size_t ntiles = (F + BENT - 1) / BENT;
  for (size_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const size_t f0 = tile * BENT;
    __syncthreads();  // the previous tile's readers are done
    for (int i = t; i < BENT * HID; i += 256) {
      const int e = i & 63, h = i >> 6;
      const size_t f = f0 + e;
      sh1[e * BST + h] = f < F ? h1c[(size_t)h * F + f] : 0.0f;
      sh2[e * BST + h] = f < F ? h2c[(size_t)h * F + f] : 0.0f;
    }
    if (t < BENT) {
      const size_t f = f0 + t;
      float phi[NF];
      features(o, f < F ? f : 0, phi);
      for (int j = 0; j < NF; ++j) sphi[t * NF + j] = phi[j];
      sgs[t] = (f < F) ? (float)(g_m[f] * m[f]) : 0.0f;
    }
    __syncthreads();
    // g_a2[e][q] = g_s[e] w3[q] (1 - h2^2)
    for (int i = t; i < BENT * HID; i += 256) {
      const int e = i >> 6, q = i & 63;
      const float h2 = sh2[e * BST + q];
      sga2[e * BST + q] = sgs[e] * params[OW3 + q] * (1.0f - h2 * h2);
    }
    __syncthreads();
    // g_a1[e][h] = (sum_q W2[q][h] g_a2[e][q]) (1 - h1^2): rows e = 4 ty + i, columns h = 4 tx + j
    {
      float a[4][4] = {};
#pragma unroll 4
      for (int q = 0; q < HID; q += 4) {
        float4 g[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) g[i] = *reinterpret_cast<const float4*>(&sga2[(4 * ty + i) * BST + q]);
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = *reinterpret_cast<const float4*>(&W2[(q + k) * BST + 4 * tx]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float gq[4] = {g[i].x, g[i].y, g[i].z, g[i].w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            a[i][0] = fmaf(w[k].x, gq[k], a[i][0]);
            a[i][1] = fmaf(w[k].y, gq[k], a[i][1]);
            a[i][2] = fmaf(w[k].z, gq[k], a[i][2]);
            a[i][3] = fmaf(w[k].w, gq[k], a[i][3]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 h1 = *reinterpret_cast<const float4*>(&sh1[(4 * ty + i) * BST + 4 * tx]);
        *reinterpret_cast<float4*>(&sga1[(4 * ty + i) * BST + 4 * tx]) =
            make_float4(a[i][0] * (1.0f - h1.x * h1.x), a[i][1] * (1.0f - h1.y * h1.y),
                        a[i][2] * (1.0f - h1.z * h1.z), a[i][3] * (1.0f - h1.w * h1.w));
      }
    }
    // W2[q][i]: sum_e g_a2[e][q] h1[e][i], q = 4 ty + i, columns 4 tx + j
    {
      float a[4][4] = {};
#pragma unroll 8
      for (int e = 0; e < BENT; ++e) {
        const float4 g = *reinterpret_cast<const float4*>(&sga2[e * BST + 4 * ty]);
        const float4 h = *reinterpret_cast<const float4*>(&sh1[e * BST + 4 * tx]);
        const float gq[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          a[i][0] = fmaf(gq[i], h.x, a[i][0]);
          a[i][1] = fmaf(gq[i], h.y, a[i][1]);
          a[i][2] = fmaf(gq[i], h.z, a[i][2]);
          a[i][3] = fmaf(gq[i], h.w, a[i][3]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc2[i][j] += (double)a[i][j];
    }
    __syncthreads();  // g_a1 is complete
    float a1 = 0.0f, ab = 0.0f;
    for (int e = 0; e < BENT; ++e) a1 = fmaf(sga1[e * BST + t / NF], sphi[e * NF + t % NF], a1);
    if (t < 64) {
      for (int e = 0; e < BENT; ++e) ab += sga1[e * BST + t];
    } else if (t < 128) {
      for (int e = 0; e < BENT; ++e) ab += sga2[e * BST + t - 64];
    } else if (t < 192) {
      for (int e = 0; e < BENT; ++e) ab = fmaf(sgs[e], sh2[e * BST + t - 128], ab);
    } else if (t == 192) {
      for (int e = 0; e < BENT; ++e) ab += sgs[e];
    }
    acc1 += (double)a1;
    accb += (double)ab;
  }
  double* out = partial + (size_t)blockIdx.x * NPAR;
  out[OW1 + t] = acc1;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) out[OW2 + (4 * ty + i) * HID + 4 * tx + j] = acc2[i][j];
  if (t < 64) out[OB1 + t] = accb;
  else if (t < 128) out[OB2 + t - 64] = accb;
  else if (t < 192) out[OW3 + t - 128] = accb;
  else if (t == 192) out[OB3] = accb;
}
static_assert(HID * NF == 256, "one W1 entry per thread of k_mlp_bwd");

// grad[p] = sum over the CTAs of the partials, in a fixed order: 32 parameters per CTA, 8 threads each
__global__ void __launch_bounds__(256) k_param_reduce(const double* __restrict__ partial, int nblocks, float* grad) {
  __shared__ double red[8][33];
  const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  double acc = 0.0;
  if (p < NPAR)
    for (int b = seg; b < nblocks; b += 8) acc += partial[(size_t)b * NPAR + p];
  red[seg][lane] = acc;
  __syncthreads();
  if (seg == 0 && p < NPAR) {
    for (int k = 1; k < 8; ++k) acc += red[k][lane];
    grad[p] = (float)acc;
  }
}

__device__ __forceinline__ double bsum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  if (w == 0) {
    t = (lane < (int)(blockDim.x >> 5)) ? red[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  __syncthreads();
  return t;
}

// part[pair][k][block]: the blocks' sums of r.z, z.w and r.e of each pair (blockIdx.y)
constexpr int kDotBlocks = 64;
__global__ void __launch_bounds__(256) k_dots3(const double* __restrict__ r, const double* __restrict__ z,
                                               const double* __restrict__ w, const double* __restrict__ e, size_t n,
                                               double* part) {
  __shared__ double red[32];
  const size_t off = blockIdx.y * n;
  double a = 0.0, b = 0.0, c = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double ri = r[off + i], zi = z[off + i];
    a += ri * zi;
    b += zi * w[off + i];
    c += ri * e[off + i];
  }
  const double ta = bsum(a, red);
  const double tb = bsum(b, red);
  const double tc = bsum(c, red);
  if (threadIdx.x == 0) {
    double* out = part + (size_t)blockIdx.y * 3 * kDotBlocks + blockIdx.x;
    out[0] = ta;
    out[kDotBlocks] = tb;
    out[2 * kDotBlocks] = tc;
  }
}
// dots[3 pair + k]: the blocks' sums added in a fixed order (one warp per dot product)
__global__ void k_dots3_sum(const double* __restrict__ part, double* dots) {
  const double* p = part + (size_t)blockIdx.x * kDotBlocks;
  double v = p[threadIdx.x] + p[threadIdx.x + 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (threadIdx.x == 0) dots[blockIdx.x] = v;
}
static_assert(kDotBlocks == 64, "k_dots3_sum");

// g_m[f] += (x weight) * sum over nb pairs and the y (z) mirror images of
//           [ -(2/c) |R|^2 + (1/c) 2 Re(conj(W) R) ] / (B prod(P))
__global__ void k_grad_accum(const double2* __restrict__ SR, const double2* __restrict__ SW, size_t sstride, Oct o,
                             int Py, int Pz, const double* __restrict__ dots, int nb, int B, double invP,
                             double* g_m) {
  const size_t F = (size_t)o.Hx1 * o.Hy1 * o.Hz1;
  const size_t f = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const int kx = (int)(f % o.Hx1);
  const int ky = (int)((f / o.Hx1) % o.Hy1);
  const int kz = (int)(f / ((size_t)o.Hx1 * o.Hy1));
  const int ny_img = (ky == 0 || 2 * ky == Py) ? 1 : 2;
  const int nz_img = (o.d == 2) ? 1 : ((kz == 0 || 2 * kz == Pz) ? 1 : 2);
  const double wx = (kx == 0 || kx == o.Hx1 - 1) ? 1.0 : 2.0;
  double g = g_m[f];
  for (int pair = 0; pair < nb; ++pair) {
    const double c = dots[3 * pair + 2];
    if (!(c > 0.0)) continue;  // degenerate pair (zero error): no contribution
    const double ca = -2.0 / c, cb = 2.0 / c;
    double acc = 0.0;
    for (int i = 0; i < ny_img; ++i) {
      const int yy = i == 0 ? ky : Py - ky;
      for (int j = 0; j < nz_img; ++j) {
        const int zz = j == 0 ? kz : Pz - kz;
        const size_t idx =
            pair * sstride + ((o.d == 2) ? (size_t)kx * Py + yy : ((size_t)kx * Py + yy) * Pz + zz);
        const double2 rv = SR[idx], wv = SW[idx];
        acc += ca * (rv.x * rv.x + rv.y * rv.y) + cb * (wv.x * rv.x + wv.y * rv.y);
      }
    }
    g += wx * acc * invP / B;
  }
  g_m[f] = g;
}

__global__ void k_loss(const double* __restrict__ dots, int B, double* loss) {
  double L = 0.0;  // one warp; lane i takes pairs i, i + 32, ...
  for (int i = threadIdx.x; i < B; i += 32) {
    const double a = dots[3 * i], b = dots[3 * i + 1], c = dots[3 * i + 2];
    if (c > 0.0) L += (1.0 - 2.0 * a / c + b / c) / B;
  }
  for (int o = 16; o > 0; o >>= 1) L += __shfl_down_sync(0xffffffffu, L, o);
  if (threadIdx.x == 0) *loss = L;
}

__global__ void k_adam(float* p, const float* __restrict__ g, float* m1, float* m2, int n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float a = b1 * m1[i] + (1.0f - b1) * gi;
  const float v = b2 * m2[i] + (1.0f - b2) * gi * gi;
  m1[i] = a;
  m2[i] = v;
  p[i] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
}

Oct make_oct(const Plan& p) {
  Oct o;
  o.d = p.d;
  o.Hx1 = p.P[0] / 2 + 1;
  o.Hy1 = p.P[1] / 2 + 1;
  o.Hz1 = (p.d == 3) ? p.P[2] / 2 + 1 : 1;
  o.ix = 2.0f / p.P[0];
  o.iy = 2.0f / p.P[1];
  o.iz = (p.d == 3) ? 2.0f / p.P[2] : 0.0f;
  o.alpha = (float)p.alpha;
  return o;
}

double prodP(const Plan& p) {
  double s = 1.0;
  for (int r = 0; r < p.d; ++r) s *= (double)p.P[r];
  return s;
}

// Pairs whose transforms share a launch: their spectra and workspaces are held at once, so at most eight, and
// on large grids no more than 2 GB of them (one pair at least).
int learn_chunk(const Plan& p, int B) {
  const size_t pair = apply_work_bytes(p, 8) + 2 * align256(spectrum_elems(p) * 16) + 2 * p.M * 8;
  const size_t fit = ((size_t)2 << 30) / pair;
  const int c = fit < 1 ? 1 : fit > 8 ? 8 : (int)fit;
  return B < c ? B : c;
}

struct LearnBufs {
  void* awork;    // [chunk] apply workspaces
  double2* SR;    // [chunk] spectra, sstride entries apart
  double2* SD;
  size_t sstride;
  double* z;      // [chunk][M]
  double* w;
  double* m;
  double* ms;
  double* gm;
  float* h1;
  float* h2;
  double* partial;
  double* dpart;
  double* norms;
  size_t bytes;
};

LearnBufs carve_learn(const Plan& p, void* work, int B) {
  LearnBufs b;
  const size_t F = p.lam_count, C = learn_chunk(p, B);
  unsigned char* const w0 = reinterpret_cast<unsigned char*>(work);
  unsigned char* w = w0;
  auto take = [&](size_t bytes) {
    unsigned char* q = w;
    w += align256(bytes);
    return q;
  };
  b.sstride = align256(spectrum_elems(p) * 16) / 16;
  b.awork = take(C * apply_work_bytes(p, 8));
  b.SR = reinterpret_cast<double2*>(take(C * b.sstride * 16));
  b.SD = reinterpret_cast<double2*>(take(C * b.sstride * 16));
  b.z = reinterpret_cast<double*>(take(C * p.M * 8));
  b.w = reinterpret_cast<double*>(take(C * p.M * 8));
  b.m = reinterpret_cast<double*>(take(F * 8));
  b.ms = reinterpret_cast<double*>(take(F * 8));
  b.gm = reinterpret_cast<double*>(take(F * 8));
  b.h1 = reinterpret_cast<float*>(take(F * HID * 4));
  b.h2 = reinterpret_cast<float*>(take(F * HID * 4));
  b.partial = reinterpret_cast<double*>(take((size_t)kBwdCtas * NPAR * 8));
  b.dpart = reinterpret_cast<double*>(take(C * 3 * kDotBlocks * 8));
  b.norms = reinterpret_cast<double*>(take((size_t)3 * B * 8));
  b.bytes = (size_t)(w - w0);
  return b;
}

}  // namespace

size_t learn_work_bytes(const Plan& p, int B) { return carve_learn(p, nullptr, B).bytes + 256; }

cudaError_t mlp_multiplier_launch(const Plan& p, const float* params, double* m, cudaStream_t s) {
  const Oct o = make_oct(p);
  const size_t F = p.lam_count;
  k_mlp_fwd<<<(unsigned)((F + 127) / 128), 128, 0, s>>>(params, o, p.lam64, prodP(p), F, m, nullptr, 1.0, nullptr,
                                                        nullptr);
  return cudaGetLastError();
}

cudaError_t learn_grad_launch(const Plan& p, const float* params, const double* r, const double* e, int B,
                              float* grad, double* loss, void* work, cudaStream_t s) {
  const LearnBufs b = carve_learn(p, work, B);
  const Oct o = make_oct(p);
  const size_t F = p.lam_count;
  const double PP = prodP(p);
  cudaError_t err;
  k_mlp_fwd<<<(unsigned)((F + 127) / 128), 128, 0, s>>>(params, o, p.lam64, PP, F, b.m, b.ms, 1.0 / PP, b.h1, b.h2);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if ((err = cudaMemsetAsync(b.gm, 0, F * sizeof(double), s)) != cudaSuccess) return err;
  const int Py = p.P[1], Pz = (p.d == 3) ? p.P[2] : 1;
  const int C = learn_chunk(p, B);
  for (int i = 0; i < B; i += C) {
    const int nb = B - i < C ? B - i : C;
    const double* ri = r + (size_t)i * p.M;
    const double* ei = e + (size_t)i * p.M;
    if ((err = spectrum_forward(p, nb, ri, b.SR, b.sstride, b.awork, s)) != cudaSuccess) return err;
    if ((err = spectrum_inverse(p, nb, b.SR, b.sstride, b.ms, b.z, b.awork, s)) != cudaSuccess) return err;
    if ((err = apply_batch_launch<double>(p, nb, b.z, b.w, p.M, b.awork, s, nullptr, 0, nullptr, 0)) != cudaSuccess)
      return err;
    if ((err = spectrum_forward(p, nb, b.w, b.SD, b.sstride, b.awork, s)) != cudaSuccess) return err;
    k_dots3<<<dim3(kDotBlocks, nb), 256, 0, s>>>(ri, b.z, b.w, ei, p.M, b.dpart);
    k_dots3_sum<<<3 * nb, 32, 0, s>>>(b.dpart, b.norms + 3 * i);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    k_grad_accum<<<(unsigned)((F + 255) / 256), 256, 0, s>>>(b.SR, b.SD, b.sstride, o, Py, Pz, b.norms + 3 * i, nb, B,
                                                            1.0 / PP, b.gm);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  k_loss<<<1, 32, 0, s>>>(b.norms, B, loss);
  const size_t ntiles = (F + BENT - 1) / BENT;
  const int ctas = ntiles < (size_t)kBwdCtas ? (int)ntiles : kBwdCtas;
  if ((err = cudaFuncSetAttribute(k_mlp_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBwdSmem)) !=
      cudaSuccess)
    return err;
  k_mlp_bwd<<<ctas, 256, kBwdSmem, s>>>(params, o, b.gm, b.m, b.h1, b.h2, F, b.partial);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  k_param_reduce<<<(NPAR + 31) / 32, 256, 0, s>>>(b.partial, ctas, grad);
  return cudaGetLastError();
}

cudaError_t adam_launch(float* p, const float* g, float* m1, float* m2, int n, float lr, float b1, float b2, float eps,
                        int t, cudaStream_t s) {
  const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
  k_adam<<<(n + 255) / 256, 256, 0, s>>>(p, g, m1, m2, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace frlap
