// Parametric density model and optimiser kernels for reconstructions that
// differentiate through the projector (Sec. 4.5 Eq. 7 / Listing 8; Sec. 6
// Eq. 10 uses spherical harmonics per shell).
//
// Model: rho[ir, ie, ia] = sum_j sum_q B[ir, j] c[j, q] Y[(ie, ia), q]
//   B: clamped cubic B-splines in r (Cox-de Boor recursion, de Boor 1972),
//   Y: real orthonormal spherical harmonics, q = l^2 + l + m, |m| <= l <= L,
//      from the normalised associated Legendre recurrence:
//        Y_l0 = N_l0 P_l(cos t), Y_lm = sqrt(2) N_lm P_l^m(cos t) cos(m p) (m > 0),
//        Y_l,-m = sqrt(2) N_lm P_l^m(cos t) sin(m p), N_lm = sqrt((2l+1)/(4 pi) (l-m)!/(l+m)!)
//      (no Condon-Shortley phase in P_l^m).
// Both bases are evaluated on the host in double at the voxel centres and
// uploaded as float32 tables (B as [Nr][nb], Y transposed as [nq][Ne*Na]).
//
// Also here: Adam (Kingma and Ba, 2015) and the squared-residual loss.
#include <cmath>
#include <vector>

#include "tsp_internal.h"

struct tsp_shbs_s {
  int Nr = 0, nang = 0, nb = 0, L = 0, nq = 0;
  float* B = nullptr;   // [Nr][nb]
  float* Yt = nullptr;  // [nq][nang]
  float* T = nullptr;   // [Nr][nq] scratch for the render and its adjoint
  bool shells = false;  // a coefficient set per shell: B is the identity
  int device = 0;
};

namespace tsp {
namespace {

const double kPi = 3.14159265358979323846;

// Clamped cubic B-spline basis values at x (nb functions, uniform interior knots).
void bspline_row(double x, double x0, double x1, int nb, double* out) {
  const int deg = 3, nk = nb + deg + 1;
  std::vector<double> t(nk);
  const int n_int = nb - deg - 1;  // interior knots
  for (int i = 0; i <= deg; ++i) {
    t[i] = x0;
    t[nk - 1 - i] = x1;
  }
  for (int i = 1; i <= n_int; ++i) t[deg + i] = x0 + (x1 - x0) * i / (n_int + 1);
  // degree-0 indicators; the right end belongs to the last non-empty interval
  std::vector<double> N(nk - 1, 0.0);
  for (int i = 0; i + 1 < nk; ++i) {
    if (t[i] < t[i + 1] && ((x >= t[i] && x < t[i + 1]) || (x == x1 && t[i + 1] == x1 && i + 1 == nk - 1 - deg)))
      N[i] = 1.0;
  }
  for (int k = 1; k <= deg; ++k) {
    for (int i = 0; i + k + 1 < nk; ++i) {
      double a = 0.0, b = 0.0;
      if (t[i + k] > t[i]) a = (x - t[i]) / (t[i + k] - t[i]) * N[i];
      if (t[i + k + 1] > t[i + 1]) b = (t[i + k + 1] - x) / (t[i + k + 1] - t[i + 1]) * N[i + 1];
      N[i] = a + b;
    }
  }
  for (int j = 0; j < nb; ++j) out[j] = N[j];
}

// Real orthonormal spherical harmonics up to degree L at (theta, phi).
void sh_row(double theta, double phi, int L, double* out) {
  const double x = std::cos(theta), s = std::sin(theta);
  // normalised associated Legendre functions Pbar_l^m = N_lm P_l^m (no CS phase)
  std::vector<double> P((L + 1) * (L + 1), 0.0);
  auto at = [&](int l, int m) -> double& { return P[l * (L + 1) + m]; };
  at(0, 0) = std::sqrt(1.0 / (4.0 * kPi));
  for (int m = 1; m <= L; ++m) at(m, m) = std::sqrt((2.0 * m + 1.0) / (2.0 * m)) * s * at(m - 1, m - 1);
  for (int m = 0; m < L; ++m) at(m + 1, m) = std::sqrt(2.0 * m + 3.0) * x * at(m, m);
  for (int m = 0; m <= L; ++m) {
    for (int l = m + 2; l <= L; ++l) {
      const double a = std::sqrt((4.0 * l * l - 1.0) / (double(l) * l - double(m) * m));
      const double b = std::sqrt(((l - 1.0) * (l - 1.0) - double(m) * m) / (4.0 * (l - 1.0) * (l - 1.0) - 1.0));
      at(l, m) = a * (x * at(l - 1, m) - b * at(l - 2, m));
    }
  }
  for (int l = 0; l <= L; ++l) {
    out[l * l + l] = at(l, 0);
    for (int m = 1; m <= l; ++m) {
      const double v = std::sqrt(2.0) * at(l, m);
      out[l * l + l + m] = v * std::cos(m * phi);
      out[l * l + l - m] = v * std::sin(m * phi);
    }
  }
}

// T[ir][q] = sum_j B[ir][j] c[j][q]
__global__ void shbs_t_kernel(const float* __restrict__ B, const float* __restrict__ c, float* __restrict__ T, int Nr,
                              int nb, int nq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Nr * nq) return;
  const int ir = i / nq, q = i - ir * nq;
  float acc = 0.0f;
  for (int j = 0; j < nb; ++j) acc = fmaf(B[ir * nb + j], c[j * nq + q], acc);
  T[i] = acc;
}

// rho[ir][a] = sum_q T[ir][q] Yt[q][a]: a thread takes one angle of RENDER_R
// shells, whose T rows lie in shared memory, so Yt is read once per RENDER_R
// shells (128 shells x 8192 angles, degree 8, on GB300: 28 us with
// one shell per block, 15 now).
constexpr int RENDER_R = 8;
__global__ void __launch_bounds__(128) shbs_render_kernel(const float* __restrict__ T, const float* __restrict__ Yt,
                                                          float* __restrict__ rho, int Nr, int nang, int nq) {
  extern __shared__ __align__(16) float tr[];  // [nq][RENDER_R]
  const int r0 = blockIdx.y * RENDER_R, nr = min(RENDER_R, Nr - r0);
  for (int i = threadIdx.x; i < nq * RENDER_R; i += blockDim.x) {
    const int q = i / RENDER_R, k = i % RENDER_R;
    tr[i] = k < nr ? T[(r0 + k) * nq + q] : 0.0f;
  }
  __syncthreads();
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= nang) return;
  float acc[RENDER_R];
#pragma unroll
  for (int k = 0; k < RENDER_R; ++k) acc[k] = 0.0f;
#pragma unroll 4
  for (int q = 0; q < nq; ++q) {
    const float y = __ldg(Yt + size_t(q) * nang + a);
    const float4 t0 = *reinterpret_cast<const float4*>(tr + q * RENDER_R);
    const float4 t1 = *reinterpret_cast<const float4*>(tr + q * RENDER_R + 4);
    const float t[RENDER_R] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
    for (int k = 0; k < RENDER_R; ++k) acc[k] = fmaf(t[k], y, acc[k]);
  }
#pragma unroll
  for (int k = 0; k < RENDER_R; ++k)
    if (k < nr) rho[size_t(r0 + k) * nang + a] = acc[k];
}

// dT[ir][q] = sum_a G[ir][a] Yt[q][a]: a block takes one harmonic and DT_R
// shells, so each value of Yt read serves DT_R of them (128 shells x 8192
// angles, degree 8: 115 us with a block per shell and harmonic, 29 now; two or
// four harmonics a block, reading G less often from L2 with fewer warps per
// harmonic, 39 and 45). Two shells a block where eight leave SMs idle (DT_FEW).
// Fixed order.
template <int DT_R>
__global__ void __launch_bounds__(256) shbs_dt_kernel(const float* __restrict__ G, const float* __restrict__ Yt,
                                                      float* __restrict__ dT, int Nr, int nang, int nq) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = blockIdx.x, r0 = blockIdx.y * DT_R, nr = min(DT_R, Nr - r0);
  const float* y = Yt + size_t(q) * nang;
  const float* g = G + size_t(r0) * nang;
  float acc[DT_R];
#pragma unroll
  for (int k = 0; k < DT_R; ++k) acc[k] = 0.0f;
  if (nr == DT_R) {
#pragma unroll 4
    for (int a = threadIdx.x; a < nang; a += 256) {
      const float yv = __ldg(y + a);
#pragma unroll
      for (int k = 0; k < DT_R; ++k) acc[k] = fmaf(__ldg(g + size_t(k) * nang + a), yv, acc[k]);
    }
  } else {
    for (int a = threadIdx.x; a < nang; a += 256) {
      const float yv = __ldg(y + a);
#pragma unroll
      for (int k = 0; k < DT_R; ++k)
        if (k < nr) acc[k] = fmaf(__ldg(g + size_t(k) * nang + a), yv, acc[k]);
    }
  }
  __shared__ float part[8][DT_R];
#pragma unroll
  for (int k = 0; k < DT_R; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], o);
    if (lane == 0) part[warp][k] = acc[k];
  }
  __syncthreads();
  if (threadIdx.x < nr) {  // (in double: a float32 chain would lose the smaller of the eight sums one by one)
    double v = part[0][threadIdx.x];
    for (int w = 1; w < 8; ++w) v += double(part[w][threadIdx.x]);
    dT[(r0 + threadIdx.x) * nq + q] = float(v);
  }
}

// dc[j][q] = sum_ir B[ir][j] dT[ir][q], a warp each
__global__ void __launch_bounds__(256) shbs_dc_kernel(const float* __restrict__ B, const float* __restrict__ dT,
                                                      float* __restrict__ dc, int Nr, int nb, int nq) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= nb * nq) return;
  const int j = i / nq, q = i - j * nq;
  float acc = 0.0f;
  for (int ir = lane; ir < Nr; ir += 32) acc = fmaf(B[ir * nb + j], dT[ir * nq + q], acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) dc[i] = acc;
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float wd,
                            float c1, float c2) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float gi = fmaf(wd, p[i], g[i]);
    const float mi = fmaf(b1, m[i], (1.0f - b1) * gi);
    const float vi = fmaf(b2, v[i], (1.0f - b2) * gi * gi);
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// grad = 2 (yhat - y) (if grad != NULL); loss += sum (yhat - y)^2 in double.
__global__ void sq_residual_kernel(const float* __restrict__ yhat, const float* __restrict__ y, int64_t n,
                                   float* __restrict__ grad, double* __restrict__ loss) {
  double acc = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float r = yhat[i] - y[i];
    if (grad) grad[i] = 2.0f * r;
    acc += double(r) * double(r);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0 && loss) atomicAdd(loss, v);
  }
}

// loss += lambda sum_{ir < Nr-1, q} (c[ir+1][q] - c[ir][q])^2 (double) and
// grad[ir][q] += its derivative: one thread per coefficient.
__global__ void tikhonov_radial_kernel(const float* __restrict__ c, int Nr, int nq, float lambda,
                                       float* __restrict__ grad, double* __restrict__ loss) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double part = 0.0;
  if (i < Nr * nq) {
    const int ir = i / nq;
    const float here = c[i];
    float g = 0.0f;
    if (ir > 0) g = fmaf(2.0f * lambda, here - c[i - nq], g);
    if (ir + 1 < Nr) {
      const float d = c[i + nq] - here;
      g = fmaf(-2.0f * lambda, d, g);
      part = double(lambda) * double(d) * double(d);
    }
    if (grad) grad[i] += g;
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0 && loss) atomicAdd(loss, part);
}

// loss += sum (w yhat - y)^2 (double); grad = 2 w (w yhat - y).
__global__ void weighted_residual_kernel(const float* __restrict__ yhat, const float* __restrict__ w,
                                         const float* __restrict__ y, int64_t n, float* __restrict__ grad,
                                         double* __restrict__ loss) {
  double acc = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float wi = w[i];
    const float r = fmaf(wi, yhat[i], -y[i]);
    if (grad) grad[i] = 2.0f * wi * r;
    acc += double(r) * double(r);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0 && loss) atomicAdd(loss, v);
  }
}

// out += sum x y (double), grid-stride with a block reduction.
__global__ void vec_dot_kernel(const float* __restrict__ x, const float* __restrict__ y, int64_t n,
                               double* __restrict__ out) {
  double acc = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    acc += double(x[i]) * double(y[i]);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) atomicAdd(out, v);
  }
}

// y = a x + b y
__global__ void vec_axpby_kernel(float a, const float* __restrict__ x, float b, float* __restrict__ y, int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    y[i] = fmaf(a, x[i], b * y[i]);
}

// out = w x (elementwise)
__global__ void vec_mul_kernel(const float* __restrict__ w, const float* __restrict__ x, float* __restrict__ out,
                               int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = w[i] * x[i];
}

// Adds the block's values of acc to *out.
__device__ __forceinline__ void block_add(double acc, double* out) {
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) atomicAdd(out, v);
  }
}

// The vector work of CGLS, a kernel between each two operators. Vectors of
// this length (rays or coefficients: 10^4 to 10^6 values) take a few us, so a
// kernel costs its launch, not its bytes: they are fused, and the scalars stay
// on the device, each iteration's in slots of its own (gamma[k], den[k], zeroed
// once), so that no host read separates the launches. On GB300, 50 x 45 x 90
// voxels, 20 polar views of 50 x 50, 4 iterations, a dot, an update or a product per
// kernel and two host reads an iteration: 1554 us a solve, 769 now (554 in the projections).
struct CglsVecs {
  const float* w;  // [n] Eq. 9's factor
  float *q, *r, *wr;  // [n]
  float *x, *p, *s;  // [rows][nq]
  int64_t n;
  int rows, nq;
  float lambda;
};

// An iteration acts while both are positive (or NaN); a gamma that was not
// added to stays 0, so a solver that has stopped remains so.
__device__ __forceinline__ bool cgls_runs(double gamma, double den) { return !(gamma <= 0.0) && !(den <= 0.0); }

// r = y, wr = w y, first += y . y; x = 0
__global__ void cgls_start_kernel(CglsVecs v, const float* __restrict__ y, double* __restrict__ first) {
  const int64_t i0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, step = int64_t(gridDim.x) * blockDim.x;
  double acc = 0.0;
  for (int64_t i = i0; i < v.n; i += step) {
    const float yi = y[i];
    v.r[i] = yi;
    v.wr[i] = v.w[i] * yi;
    acc += double(yi) * double(yi);
  }
  for (int64_t i = i0; i < int64_t(v.rows) * v.nq; i += step) v.x[i] = 0.0f;
  block_add(acc, first);
}

// q = w q (F M p before), den += q . q + lambda ||D_r p||^2
__global__ void cgls_image_kernel(CglsVecs v, double* __restrict__ den) {
  const int64_t i0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, step = int64_t(gridDim.x) * blockDim.x;
  double acc = 0.0;
  for (int64_t i = i0; i < v.n; i += step) {
    const float qi = v.w[i] * v.q[i];
    v.q[i] = qi;
    acc += double(qi) * double(qi);
  }
  for (int64_t i = i0; i < int64_t(v.rows - 1) * v.nq; i += step) {
    const float d = v.p[i + v.nq] - v.p[i];
    acc += double(v.lambda) * double(d) * double(d);
  }
  block_add(acc, den);
}

// x += alpha p, r -= alpha q, wr = w r with alpha = gamma / den. (The scalars
// stay double, here and below: a step rounded to float32 leaves the directions
// less conjugate. With the render's transpose above: the coefficients' error
// against 64 bits, geometric mean over 28 problems of 20 to 60 shells, 6.7e-7
// with both in float32, 6.0e-7 now, which is that of the pieces' lengths; the
// eight runs of a problem lay up to 2 times apart and lie within a third now.)
__global__ void cgls_update_kernel(CglsVecs v, const double* __restrict__ gamma, const double* __restrict__ den) {
  if (!cgls_runs(*gamma, *den)) return;
  const int64_t i0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, step = int64_t(gridDim.x) * blockDim.x;
  const double alpha = *gamma / *den;
  for (int64_t i = i0; i < v.n; i += step) {
    const float ri = float(fma(-alpha, double(v.q[i]), double(v.r[i])));
    v.r[i] = ri;
    v.wr[i] = v.w[i] * ri;
  }
  for (int64_t i = i0; i < int64_t(v.rows) * v.nq; i += step) v.x[i] = float(fma(alpha, double(v.p[i]), double(v.x[i])));
}

// s -= lambda D^T D x (s: M^T F^T w r before), next += s . s, unless the
// iteration (gamma, den; NULL before the first) was a stop.
__global__ void cgls_gradient_kernel(CglsVecs v, const double* __restrict__ gamma, const double* __restrict__ den,
                                     double* __restrict__ next) {
  if (gamma && !cgls_runs(*gamma, *den)) return;
  const int64_t i0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, step = int64_t(gridDim.x) * blockDim.x;
  double acc = 0.0;
  for (int64_t i = i0; i < int64_t(v.rows) * v.nq; i += step) {
    const double here = v.x[i];
    double g = 0.0;
    if (i >= v.nq) g += here - double(v.x[i - v.nq]);
    if (i + v.nq < int64_t(v.rows) * v.nq) g -= double(v.x[i + v.nq]) - here;
    const float si = float(fma(-double(v.lambda), g, double(v.s[i])));
    v.s[i] = si;
    acc += double(si) * double(si);
  }
  block_add(acc, next);
}

// p = s + (next / gamma) p; p = s before the first iteration (gamma NULL)
__global__ void cgls_direction_kernel(CglsVecs v, const double* __restrict__ gamma, const double* __restrict__ next) {
  if (gamma && *gamma <= 0.0) return;
  const double beta = gamma ? *next / *gamma : 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < int64_t(v.rows) * v.nq;
       i += int64_t(gridDim.x) * blockDim.x)
    v.p[i] = gamma ? float(fma(beta, double(v.p[i]), double(v.s[i]))) : v.s[i];
}

int vec_blocks(int64_t n) { return int(std::min<int64_t>((n + 255) / 256, 152 * 8)); }

}  // namespace
}  // namespace tsp

using namespace tsp;

extern "C" tsp_status tsp_shbs_create(int n_basis_r, int L, const double* r_centres, int Nr, const double* theta_centres,
                                      int Ne, const double* phi_centres, int Na, double r_min, double r_max,
                                      tsp_shbs* out) {
  if (!out) return fail(TSP_EINVAL, "tsp_shbs_create: out is NULL");
  *out = nullptr;
  if (n_basis_r < 4 || L < 0 || L > 32 || Nr <= 0 || Ne <= 0 || Na <= 0 || !r_centres || !theta_centres || !phi_centres ||
      !(r_max > r_min))
    return fail(TSP_EINVAL, "tsp_shbs_create: bad argument");
  tsp_shbs h = new (std::nothrow) tsp_shbs_s();
  if (!h) return fail(TSP_ENOMEM, "tsp_shbs_create: host allocation");
  h->Nr = Nr;
  h->nang = Ne * Na;
  h->nb = n_basis_r;
  h->L = L;
  h->nq = (L + 1) * (L + 1);
  std::vector<float> B(size_t(Nr) * h->nb), Yt(size_t(h->nq) * h->nang);
  std::vector<double> row(std::max(h->nb, h->nq));
  for (int ir = 0; ir < Nr; ++ir) {
    bspline_row(std::min(std::max(r_centres[ir], r_min), r_max), r_min, r_max, h->nb, row.data());
    for (int j = 0; j < h->nb; ++j) B[size_t(ir) * h->nb + j] = float(row[j]);
  }
  for (int ie = 0; ie < Ne; ++ie) {
    for (int ia = 0; ia < Na; ++ia) {
      sh_row(theta_centres[ie], phi_centres[ia], L, row.data());
      for (int q = 0; q < h->nq; ++q) Yt[size_t(q) * h->nang + ie * Na + ia] = float(row[q]);
    }
  }
  cudaError_t e = cudaGetDevice(&h->device);
  if (e == cudaSuccess) e = cudaMalloc(&h->B, sizeof(float) * B.size());
  if (e == cudaSuccess) e = cudaMalloc(&h->Yt, sizeof(float) * Yt.size());
  if (e == cudaSuccess) e = cudaMalloc(&h->T, sizeof(float) * size_t(Nr) * h->nq);
  if (e == cudaSuccess) e = cudaMemcpy(h->B, B.data(), sizeof(float) * B.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(h->Yt, Yt.data(), sizeof(float) * Yt.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    tsp_shbs_destroy(h);
    return cuda_fail(e, "tsp_shbs_create: upload");
  }
  *out = h;
  return TSP_OK;
}

extern "C" tsp_status tsp_shbs_create_shells(int L, int Nr, const double* theta_centres, int Ne,
                                             const double* phi_centres, int Na, tsp_shbs* out) {
  if (!out) return fail(TSP_EINVAL, "tsp_shbs_create_shells: out is NULL");
  *out = nullptr;
  if (L < 0 || L > 32 || Nr <= 0 || Ne <= 0 || Na <= 0 || !theta_centres || !phi_centres)
    return fail(TSP_EINVAL, "tsp_shbs_create_shells: bad argument");
  tsp_shbs h = new (std::nothrow) tsp_shbs_s();
  if (!h) return fail(TSP_ENOMEM, "tsp_shbs_create_shells: host allocation");
  h->Nr = Nr;
  h->nang = Ne * Na;
  h->nb = Nr;
  h->L = L;
  h->nq = (L + 1) * (L + 1);
  h->shells = true;
  std::vector<float> B(size_t(Nr) * Nr, 0.0f), Yt(size_t(h->nq) * h->nang);
  for (int ir = 0; ir < Nr; ++ir) B[size_t(ir) * Nr + ir] = 1.0f;  // one coefficient set per shell
  std::vector<double> row(h->nq);
  for (int ie = 0; ie < Ne; ++ie) {
    for (int ia = 0; ia < Na; ++ia) {
      sh_row(theta_centres[ie], phi_centres[ia], L, row.data());
      for (int q = 0; q < h->nq; ++q) Yt[size_t(q) * h->nang + ie * Na + ia] = float(row[q]);
    }
  }
  cudaError_t e = cudaGetDevice(&h->device);
  if (e == cudaSuccess) e = cudaMalloc(&h->B, sizeof(float) * B.size());
  if (e == cudaSuccess) e = cudaMalloc(&h->Yt, sizeof(float) * Yt.size());
  if (e == cudaSuccess) e = cudaMalloc(&h->T, sizeof(float) * size_t(Nr) * h->nq);
  if (e == cudaSuccess) e = cudaMemcpy(h->B, B.data(), sizeof(float) * B.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(h->Yt, Yt.data(), sizeof(float) * Yt.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    tsp_shbs_destroy(h);
    return cuda_fail(e, "tsp_shbs_create_shells: upload");
  }
  *out = h;
  return TSP_OK;
}

extern "C" void tsp_shbs_destroy(tsp_shbs h) {
  if (!h) return;
  if (h->B) cudaFree(h->B);
  if (h->Yt) cudaFree(h->Yt);
  if (h->T) cudaFree(h->T);
  delete h;
}

extern "C" tsp_status tsp_shbs_tables(tsp_shbs h, float* B_host, float* Yt_host) {
  if (!h) return fail(TSP_EINVAL, "tsp_shbs_tables: NULL handle");
  if (B_host) TSP_CUDA(cudaMemcpy(B_host, h->B, sizeof(float) * size_t(h->Nr) * h->nb, cudaMemcpyDeviceToHost));
  if (Yt_host) TSP_CUDA(cudaMemcpy(Yt_host, h->Yt, sizeof(float) * size_t(h->nq) * h->nang, cudaMemcpyDeviceToHost));
  return TSP_OK;
}

extern "C" tsp_status tsp_shbs_render(tsp_shbs h, const float* coeffs, float* rho, void* stream) {
  if (!h || !coeffs || !rho) return fail(TSP_EINVAL, "tsp_shbs_render: NULL argument");
  tsp_status st = check_device(h->device);
  if (st != TSP_OK) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  const int n = h->Nr * h->nq;
  if (!h->shells) shbs_t_kernel<<<(n + 127) / 128, 128, 0, cs>>>(h->B, coeffs, h->T, h->Nr, h->nb, h->nq);
  const dim3 grid((h->nang + 127) / 128, (h->Nr + RENDER_R - 1) / RENDER_R);
  shbs_render_kernel<<<grid, 128, sizeof(float) * h->nq * RENDER_R, cs>>>(h->shells ? coeffs : h->T, h->Yt, rho, h->Nr,
                                                                          h->nang, h->nq);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_shbs_render_adjoint(tsp_shbs h, const float* grad_rho, float* grad_coeffs, void* stream) {
  if (!h || !grad_rho || !grad_coeffs) return fail(TSP_EINVAL, "tsp_shbs_render_adjoint: NULL argument");
  tsp_status st = check_device(h->device);
  if (st != TSP_OK) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  float* dT = h->shells ? grad_coeffs : h->T;
  // (DT_FEW: 50 shells x 4050 angles, degree 3: 112 blocks of eight shells take
  // 13.6 us, 400 of two 9.0.)
  constexpr int DT_FEW = 2 * 152;
  if (h->nq * ((h->Nr + 7) / 8) >= DT_FEW) {
    shbs_dt_kernel<8><<<dim3(h->nq, (h->Nr + 7) / 8), 256, 0, cs>>>(grad_rho, h->Yt, dT, h->Nr, h->nang, h->nq);
  } else {
    shbs_dt_kernel<2><<<dim3(h->nq, (h->Nr + 1) / 2), 256, 0, cs>>>(grad_rho, h->Yt, dT, h->Nr, h->nang, h->nq);
  }
  const int n = h->nb * h->nq;
  if (!h->shells) shbs_dc_kernel<<<(n + 7) / 8, 256, 0, cs>>>(h->B, h->T, grad_coeffs, h->Nr, h->nb, h->nq);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_adam(float* params, const float* grads, float* m, float* v, int64_t n, float lr, float beta1,
                               float beta2, float eps, float weight_decay, int step, void* stream) {
  if (!params || !grads || !m || !v || n <= 0 || step < 1) return fail(TSP_EINVAL, "tsp_adam: bad argument");
  const float c1 = float(1.0 - std::pow(double(beta1), step));
  const float c2 = float(1.0 - std::pow(double(beta2), step));
  const int blocks = int(std::min<int64_t>((n + 255) / 256, 152 * 8));
  adam_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(params, grads, m, v, n, lr, beta1, beta2, eps,
                                                                     weight_decay, c1, c2);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_sq_residual(const float* yhat, const float* y, int64_t n, float* grad, double* loss,
                                      void* stream) {
  if (!yhat || !y || n <= 0) return fail(TSP_EINVAL, "tsp_sq_residual: bad argument");
  const int blocks = int(std::min<int64_t>((n + 255) / 256, 152 * 8));
  sq_residual_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(yhat, y, n, grad, loss);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_tikhonov_radial(const float* coeffs, int n_r, int n_q, float lambda, float* grad,
                                          double* loss, void* stream) {
  if (!coeffs || n_r <= 0 || n_q <= 0 || !(lambda >= 0.0f))
    return fail(TSP_EINVAL, "tsp_tikhonov_radial: bad argument");
  const int n = n_r * n_q;
  tikhonov_radial_kernel<<<(n + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(coeffs, n_r, n_q, lambda,
                                                                                          grad, loss);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_sq_residual_weighted(const float* yhat, const float* w, const float* y, int64_t n,
                                               float* grad, double* loss, void* stream) {
  if (!yhat || !w || !y || n <= 0) return fail(TSP_EINVAL, "tsp_sq_residual_weighted: bad argument");
  const int blocks = int(std::min<int64_t>((n + 255) / 256, 152 * 8));
  weighted_residual_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(yhat, w, y, n, grad, loss);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_vec_dot(const float* x, const float* y, int64_t n, double* out, void* stream) {
  if (!x || !y || !out || n < 0) return fail(TSP_EINVAL, "tsp_vec_dot: bad argument");
  if (n == 0) return TSP_OK;
  vec_dot_kernel<<<vec_blocks(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(x, y, n, out);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_vec_axpby(float a, const float* x, float b, float* y, int64_t n, void* stream) {
  if (!x || !y || n < 0) return fail(TSP_EINVAL, "tsp_vec_axpby: bad argument");
  if (n == 0) return TSP_OK;
  vec_axpby_kernel<<<vec_blocks(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(a, x, b, y, n);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_vec_mul(const float* w, const float* x, float* out, int64_t n, void* stream) {
  if (!w || !x || !out || n < 0) return fail(TSP_EINVAL, "tsp_vec_mul: bad argument");
  if (n == 0) return TSP_OK;
  vec_mul_kernel<<<vec_blocks(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(w, x, out, n);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_shbs_cgls(tsp_shbs model, tsp_grid grid, tsp_geom geom, const float* w, const float* y,
                                    float lambda, int n_iter, float* x, float* ws, int64_t ws_floats, double* scalars,
                                    void* stream) {
  if (!model || !grid || !geom || !w || !y || !x || !ws || !scalars || n_iter < 0 || !(lambda >= 0.0f))
    return fail(TSP_EINVAL, "tsp_shbs_cgls: bad argument");
  if (model->Nr != grid->Nr || model->nang != grid->Ne * grid->Na)
    return fail(TSP_EINVAL, "tsp_shbs_cgls: the model and the grid differ in shape");
  tsp_status st = check_device(model->device);
  if (st != TSP_OK) return st;
  const int64_t n = geom->n_rays, nc = int64_t(model->nb) * model->nq;
  if (ws_floats < 3 * n + 2 * nc + grid->voxels()) return fail(TSP_EINVAL, "tsp_shbs_cgls: workspace too small");
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  float* vol = ws;  // rho of the projection, then the gradient that comes back
  CglsVecs v;
  v.w = w;
  v.q = vol + grid->voxels();
  v.r = v.q + n;
  v.wr = v.r + n;
  v.x = x;
  v.p = v.wr + n;
  v.s = v.p + nc;
  v.n = n;
  v.rows = model->nb;
  v.nq = model->nq;
  v.lambda = lambda;
  double* gamma = scalars + 2;    // [n_iter]
  double* den = gamma + n_iter;   // [n_iter]
  const int bn = vec_blocks(std::max(n, nc)), bc = vec_blocks(nc);
  TSP_CUDA(cudaMemsetAsync(scalars, 0, sizeof(double) * (2 * size_t(n_iter) + 2), cs));
  cgls_start_kernel<<<bn, 256, 0, cs>>>(v, y, scalars);
  for (int k = 0; k < n_iter; ++k) {
    // s = A^T r - lambda D^T D x and the next direction
    if ((st = tsp_adjoint_ex(grid, geom, v.wr, vol, 1, 0, nullptr, stream)) != TSP_OK) return st;
    if ((st = tsp_shbs_render_adjoint(model, vol, v.s, stream)) != TSP_OK) return st;
    const double *g_last = k ? gamma + k - 1 : nullptr, *d_last = k ? den + k - 1 : nullptr;
    cgls_gradient_kernel<<<bc, 256, 0, cs>>>(v, g_last, d_last, gamma + k);
    if (k % 32 == 31) {  // (a solver that has stopped launches no more than this many idle iterations)
      double g = 0.0;
      TSP_CUDA(cudaMemcpyAsync(&g, gamma + k, sizeof(double), cudaMemcpyDeviceToHost, cs));
      TSP_CUDA(cudaStreamSynchronize(cs));
      if (g <= 0.0) break;
    }
    cgls_direction_kernel<<<bc, 256, 0, cs>>>(v, g_last, gamma + k);
    // alpha = gamma / (||A p||^2 + lambda ||D p||^2) and the step
    if ((st = tsp_shbs_render(model, v.p, vol, stream)) != TSP_OK) return st;
    if ((st = tsp_forward_ex(grid, geom, vol, v.q, 1, nullptr, stream)) != TSP_OK) return st;
    cgls_image_kernel<<<bn, 256, 0, cs>>>(v, den + k);
    cgls_update_kernel<<<bn, 256, 0, cs>>>(v, gamma + k, den + k);
  }
  vec_dot_kernel<<<vec_blocks(n), 256, 0, cs>>>(v.r, v.r, n, scalars + 1);
  tikhonov_radial_kernel<<<unsigned((nc + 255) / 256), 256, 0, cs>>>(x, v.rows, v.nq, lambda, nullptr, scalars + 1);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}
