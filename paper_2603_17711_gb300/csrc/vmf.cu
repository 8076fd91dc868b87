// Kernels of the direct integration (vmf, Sec. 2.3 and Sec. 7.5), FP64.
//
// The node equations of the multilayer-MCTDH form need, on every edge p -> c,
// the single-hole density matrix rho and the mean fields M(kappa) of the part
// of the tree above c, weighted by the root. With the upper part brought into
// an orthonormal basis by a QR gauge move toward c (V_p = Q R), they are
//     rho = R^H R,   M(kappa) = R^H E(kappa) R,
// E(kappa) the ordinary (isometric) environment of class kappa. The equation
// of c, rho_reg dU_c/dt = (1 - P_c) G_c with rho_reg = rho + vmf_atol * 1, is
// evaluated as
//     dU_c/dt = (1 - P_c) [ H~ U_c + (D - 1) x_parent G_down ],
//     H~      = the node operator with E~(kappa) = rho_reg^-1 M(kappa) on the
//               parent leg, D = rho_reg^-1 rho,
// G_down the part of the node operator without a parent-leg factor (rho_reg^-1
// then multiplies rho, not the identity, for those terms). P_c projects onto
// the span of U_c's rows (parent index fixed): (1 - P) X = X - (X U^H) U.
//
//  k_vmf_inv    one CTA: rho = R^H R, rho_reg^-1 by Gauss-Jordan elimination with
//               partial pivoting, D - 1 = -vmf_atol rho_reg^-1
//  k_vmf_class  one cluster per class: E~ = rho_reg^-1 (R^H (E R)), in place
//  k_vmf_addmul K += (D - 1) G_down; K -= X U
//  k_vmf_px     X = K U^H (one CTA per entry, fixed-order sums)
//  k_vmf_stage  out = y + sum_l c_l K_l over the flat state
//  k_vmf_err    scaled squared error of the embedded pair, block partials;
//  k_vmf_sum    the partials added in order
#include <algorithm>

#include <cooperative_groups.h>

#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace ttn {

namespace {

constexpr int kT = 256;

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {  // conj(a) b
  return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// Component comp (0 real, 1 imaginary) of s + a b and of s + conj(a) b.
__device__ __forceinline__ double fma_part(double2 a, double2 b, int comp, double s) {
  return fma(a.y, comp ? b.x : -b.y, fma(a.x, comp ? b.y : b.x, s));
}
__device__ __forceinline__ double fma_conj_part(double2 a, double2 b, int comp, double s) {
  return fma(a.y, comp ? -b.x : b.y, fma(a.x, comp ? b.y : b.x, s));
}

// inv = (rho + eps)^-1 with rho = R^H R, dmi = (rho + eps)^-1 rho - 1 = -eps inv, by
// Gauss-Jordan on [rho + eps | 1], held in shared memory (in `aug` above
// kGjSmemMaxR). Pivot: the largest |re| + |im| of the column among the rows not
// yet used. Rows are neither swapped nor scaled until the end, so a pivot takes
// two barriers: warp 0 finds it and divides the column's entries by it, then
// all threads eliminate; of the left block only the columns still to come are
// updated. A chain of latencies on one CTA (an FP64 instruction holds an SM
// sub-partition for 64 cycles): r = 12 took 38 us with six barriers a pivot, the
// matrix in global memory and rho as a third block.
constexpr int kGjSmemMaxR = 64;
size_t inv_smem(int r) { return sizeof(double2) * (size_t)(2 * r + (r <= kGjSmemMaxR ? 2 * r * r : 0)) + sizeof(int) * r; }
__global__ void __launch_bounds__(kT) k_vmf_inv(const double2* __restrict__ R, int r, double eps, double2* aug,
                                                double2* __restrict__ inv, double2* __restrict__ dmi) {
  extern __shared__ double2 gj[];
  const int tid = threadIdx.x, nt = blockDim.x, w = 2 * r;
  double2* f = gj;       // multipliers of the current pivot
  double2* sc = gj + r;  // 1 / pivot
  double2* A = r <= kGjSmemMaxR ? gj + 2 * r : aug;
  int* perm = (int*)(gj + 2 * r + (r <= kGjSmemMaxR ? 2 * r * r : 0));  // row of pivot j
  grid_wait();
  for (int e = tid; e < 2 * r * r; e += nt) {
    const int comp = e & 1, i = (e >> 1) / r, j = (e >> 1) % r;
    double s = 0.0;
    for (int k = 0; k < r; ++k) s = fma_conj_part(R[k * r + i], R[k * r + j], comp, s);
    reinterpret_cast<double*>(A + i * w + j)[comp] = i == j && comp == 0 ? s + eps : s;
    reinterpret_cast<double*>(A + i * w + r + j)[comp] = i == j && comp == 0 ? 1.0 : 0.0;
  }
  __syncthreads();
  for (int j = 0; j < r; ++j) {
    if (tid < 32) {
      // nonnegative doubles compare as integers (a NaN above all numbers); + 1: a zero still beats no row
      unsigned long long best = 0;
      int bi = r;
      for (int i = tid; i < r; i += 32) {
        bool used = false;
        for (int q = 0; q < j; ++q) used |= perm[q] == i;
        const double2 v = A[i * w + j];
        const unsigned long long a = used ? 0 : (unsigned long long)__double_as_longlong(fabs(v.x) + fabs(v.y)) + 1;
        if (a > best) {
          best = a;
          bi = i;
        }
      }
      const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32));
      const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
      const bool top = best == (((unsigned long long)hi << 32) | lo);
      const int pv = (int)__reduce_min_sync(0xffffffffu, top ? (unsigned)bi : (unsigned)r);
      const double2 p = A[pv * w + j];
      const double n = fma(p.x, p.x, p.y * p.y), q = ((tid & 1) ? -p.y : p.x) / n;  // even lanes real, odd imaginary
      const double2 pi = make_double2(__shfl_sync(0xffffffffu, q, 0), __shfl_sync(0xffffffffu, q, 1));
      for (int i = tid; i < r; i += 32) f[i] = cmul(A[i * w + j], pi);
      if (tid == 0) {
        perm[j] = pv;
        sc[j] = pi;
      }
    }
    __syncthreads();
    const int pv = perm[j], nc = w - j - 1;
    for (int e = tid; e < r * nc; e += nt) {
      const int i = e / nc, c = j + 1 + e % nc;
      if (i == pv) continue;
      const double2 p = A[pv * w + c], m = f[i];
      double2 a = A[i * w + c];
      a.x = fma(-m.x, p.x, fma(m.y, p.y, a.x));
      a.y = fma(-m.x, p.y, fma(-m.y, p.x, a.y));
      A[i * w + c] = a;
    }
    __syncthreads();
  }
  grid_release();
  for (int e = tid; e < r * r; e += nt) {
    const int i = e / r, c = e % r;
    const double2 v = cmul(A[perm[i] * w + r + c], sc[i]);
    inv[e] = v;
    dmi[e] = make_double2(-eps * v.x, -eps * v.y);
  }
}

// E~ = inv (R^H (E R)) for one class matrix per cluster, in place; a CTA makes
// its own columns of all three products (one thread per component), the two
// intermediate ones in `tmp` (2 r^2 per class), and E is overwritten once every
// CTA has read it. FP64 issue of one SM bound a CTA per class: r = 12 12.7 us.
__global__ void __launch_bounds__(128) k_vmf_class(double2* const* mats, const int* __restrict__ slots,
                                                   const double2* __restrict__ R, const double2* __restrict__ inv, int r,
                                                   double2* tmp) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CC = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), cls = blockIdx.x / CC;
  const int j0 = rank * r / CC, nj = (rank + 1) * r / CC - j0, n = 2 * r * nj;
  double2* E = mats[slots[cls]];
  double2* A = tmp + (size_t)cls * 2 * r * r;  // E R
  double2* B = A + r * r;                      // R^H E R
  grid_wait();
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int comp = e & 1, i = (e >> 1) / nj, j = j0 + (e >> 1) % nj;
    double s = 0.0;
    for (int k = 0; k < r; ++k) s = fma_part(E[i * r + k], R[k * r + j], comp, s);
    reinterpret_cast<double*>(A + i * r + j)[comp] = s;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int comp = e & 1, i = (e >> 1) / nj, j = j0 + (e >> 1) % nj;
    double s = 0.0;
    for (int k = 0; k < r; ++k) s = fma_conj_part(R[k * r + i], A[k * r + j], comp, s);
    reinterpret_cast<double*>(B + i * r + j)[comp] = s;
  }
  grid_release();
  cluster.sync();
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int comp = e & 1, i = (e >> 1) / nj, j = j0 + (e >> 1) % nj;
    double s = 0.0;
    for (int k = 0; k < r; ++k) s = fma_part(inv[i * r + k], B[k * r + j], comp, s);
    reinterpret_cast<double*>(E + i * r + j)[comp] = s;
  }
}

// K (r x nc) += sgn M (r x r) G (r x nc): dmi G_down added, X U taken off. One
// thread per component and CTAs of two warps: at r = 12 (1728 elements) eight-warp
// CTAs of one thread per element took 6.7 us, bound by the FP64 issue of the 7 SMs used.
constexpr int kTs = 64;
__global__ void __launch_bounds__(kTs) k_vmf_addmul(double2* __restrict__ K, const double2* __restrict__ G,
                                                    const double2* __restrict__ M, double sgn, int r, int64_t nc) {
  grid_wait();
  grid_release();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < 2 * (int64_t)r * nc;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int comp = (int)(e & 1);
    int64_t c;
    const int a = (int)idivmod(e >> 1, nc, c);
    double s = 0.0;
    for (int b = 0; b < r; ++b) s = fma_part(M[a * r + b], G[(int64_t)b * nc + c], comp, s);
    double* k = reinterpret_cast<double*>(K) + e;
    *k = fma(sgn, s, *k);
  }
}

// X[a][b] = sum_c K[a][c] conj(U[b][c]); one CTA per entry
__global__ void k_vmf_px(const double2* __restrict__ K, const double2* __restrict__ U, int r, int64_t nc,
                         double2* __restrict__ X) {
  __shared__ double2 red[kT / 32];
  const int a = blockIdx.x / r, b = blockIdx.x % r;
  grid_wait();
  double2 s = make_double2(0.0, 0.0);
  for (int64_t c = threadIdx.x; c < nc; c += blockDim.x)
    s = cadd(s, cmulc(U[(int64_t)b * nc + c], K[(int64_t)a * nc + c]));
  grid_release();
  for (int o = 16; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double2 t = make_double2(0.0, 0.0);
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t = cadd(t, red[q]);
    X[blockIdx.x] = t;
  }
}

__global__ void k_vmf_stage(double2* __restrict__ out, const double2* __restrict__ y, VmfComb cb, int64_t n) {
  grid_wait();
  grid_release();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double2 s = y[e];
    for (int l = 0; l < cb.n; ++l) {
      const double2 k = cb.K[l][e];
      s.x = fma(cb.c[l], k.x, s.x);
      s.y = fma(cb.c[l], k.y, s.y);
    }
    out[e] = s;
  }
}

constexpr int kErrBlocks = 1024;
__global__ void k_vmf_err(const double2* __restrict__ y, const double2* __restrict__ y5, VmfComb cb, double rtol,
                          double atol, int64_t n, double* __restrict__ part) {
  __shared__ double red[kT / 32];
  double acc = 0.0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double ex = 0.0, ey = 0.0;
    for (int l = 0; l < cb.n; ++l) {
      const double2 k = cb.K[l][e];
      ex = fma(cb.c[l], k.x, ex);
      ey = fma(cb.c[l], k.y, ey);
    }
    const double a = sqrt(y[e].x * y[e].x + y[e].y * y[e].y), b = sqrt(y5[e].x * y5[e].x + y5[e].y * y5[e].y);
    const double sc = atol + rtol * fmax(a, b);
    acc += (ex * ex + ey * ey) / (sc * sc);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < kT / 32; ++q) t += red[q];
    part[blockIdx.x] = t;
  }
}
__global__ void k_vmf_sum(const double* __restrict__ part, int n, double* __restrict__ out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < n; ++i) t += part[i];
    out[0] = t;
  }
}

int grid_of(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + kT - 1) / kT, 4096)); }

}  // namespace

void launch_vmf_edge(double2* const* mats_dev, const int* slots_dev, int n_classes, const double2* R, int r,
                     double eps, double2* aug, double2* dmi, double2* tmp, cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_vmf_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)inv_smem(kGjSmemMaxR));
    attr = true;
  }
  double2* inv = aug + 2 * (int64_t)r * r;
  launch_dep(k_vmf_inv, dim3(1), dim3(kT), inv_smem(r), s, 0, R, r, eps, aug, inv, dmi);
  const int cc = std::min(8, (r + 3) / 4);
  if (n_classes > 0)
    launch_dep(k_vmf_class, dim3((unsigned)(n_classes * cc)), dim3(128), 0, s, cc, mats_dev, slots_dev, R, inv, r, tmp);
}

void launch_vmf_finish(double2* K, const double2* Gdown, const double2* dmi, const double2* U, int r, int64_t nc,
                       double2* X, cudaStream_t s) {
  const int64_t n = 2 * (int64_t)r * nc;
  const dim3 grid((unsigned)std::min<int64_t>((n + kTs - 1) / kTs, 8192));
  launch_dep(k_vmf_addmul, grid, dim3(kTs), 0, s, 0, K, Gdown, dmi, 1.0, r, nc);
  launch_dep(k_vmf_px, dim3(r * r), dim3(kT), 0, s, 0, K, U, r, nc, X);
  launch_dep(k_vmf_addmul, grid, dim3(kTs), 0, s, 0, K, U, X, -1.0, r, nc);
}

void launch_vmf_stage(double2* out, const double2* y, const VmfComb& cb, int64_t n, cudaStream_t s) {
  launch_dep(k_vmf_stage, dim3(grid_of(n)), dim3(kT), 0, s, 0, out, y, cb, n);
}

void launch_vmf_err(const double2* y, const double2* y5, const VmfComb& cb, double rtol, double atol, int64_t n,
                    double* part, double* out, cudaStream_t s) {
  k_vmf_err<<<counted(kErrBlocks), kT, 0, s>>>(y, y5, cb, rtol, atol, n, part);
  k_vmf_sum<<<counted(1), 32, 0, s>>>(part, kErrBlocks, out);
}

}  // namespace ttn
