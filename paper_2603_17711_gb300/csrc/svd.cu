// One-sided (Hestenes) Jacobi SVD spread over several CTAs, FP64 -- the
// factorisation that splits a merged pair in the adaptive-rank scheme (Sec. 2.3,
// last paragraph), for matrices too wide for one CTA.
//
// The working matrix holds the columns of Theta (or of Theta^H when Theta is
// wider than tall), column-major; V starts as the identity. A sweep visits every
// column pair once, in the rounds of the circle method: the pairs of one round
// are disjoint, so they are dealt to the CTAs. Between rounds stands the hardware
// barrier of a thread-block cluster when the pairs fit one cluster (at most 16
// CTAs); in the grid form (one cooperative launch) a CTA waits for its two columns
// only, handed over by a counter each, and a grid barrier ends the sweep.
// A pair is handled by one CTA of four warps: its threads split the rows, the three
// Gram entries a = |x|^2, b = |y|^2, c = x^H y are summed in a fixed order (threads
// -> warps -> a butterfly over the warps), warp 0 computes the complex rotation
// (rotate_warp: skipped when |c| <= tol sqrt(a b) or a column is rounding
// noise) and the threads apply it to the pair's rows of the working matrix and
// of V. GB300 retires about one FP64 warp instruction per 19 cycles per SM, and
// a square root or quotient is a dozen of them: computing the rotation in one
// warp instead of all keeps the FP64 pipe for the rows.
// A sweep without a rotation, or of small rotations only (kBigCos, kBigSin), ends
// the iteration: every CTA reads the sweep's counts after the sweep's last barrier.
// Which CTA handles a pair, and what ends a round, does not change the arithmetic,
// so the result does not depend on the launch shape.
//
// The convergence threshold tol = 2 sqrt(max(rows, 64)) * DBL_EPSILON sits above
// the rounding noise of the Gram entries summed over the rows, so a converged
// matrix stops rotating; a run that reaches max_sweeps reports it (info[0] ==
// max_sweeps) and the host refuses the result.
//
// Every grid wait is bounded (wait_ns from the moment the CTA starts waiting);
// a CTA whose wait gives up sets bit 4 (value 16) of *flag and returns. Nothing
// is in flight when it does (plain loads and stores only), so any CTA may leave
// at any time; the others give up at their next wait. The cluster barrier is
// the hardware's: all CTAs of a cluster are resident together and every CTA
// passes the same number of barriers.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include <cooperative_groups.h>

#include "../../include/ttn_heom.h"
#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace ttn {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
// Jacobi: four warps, one per SM sub-partition. Eight would share the FP64 pipes
// two by two and double the time of the lane sums.
constexpr int kJThreads = 128;
constexpr int kJWarps = kJThreads / 32;
constexpr int kBarLanes = 8;
constexpr int kSvdMaxVer = 2048;  // more columns than this keep one barrier a round
constexpr int kSmallOff = kBarLanes + kJacMaxSweeps;  // first counter of small rotations
static_assert(kSmallOff + kJacMaxSweeps <= kSvdSyncInts, "the counters of all sweeps fit");

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double wsum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier: CTA c adds one to lane c % kBarLanes after a CTA barrier (which
// orders the CTA's writes before thread 0's release); warp 0 polls the lanes
// with acquire loads until their sum reaches target, then a CTA barrier orders
// the other CTAs' writes before this CTA's later reads. Returns false when the
// wait gave up.
__device__ bool grid_sync(unsigned* lanes, unsigned target, uint64_t wait_ns, int* flag) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    if (lane == 0) red_release_add(lanes + blockIdx.x % kBarLanes, 1u);
    const uint64_t t0 = now_ns();
    int ok = 1;
    for (unsigned it = 0;; ++it) {
      unsigned v = lane < kBarLanes ? ld_acquire(lanes + lane) : 0u;
      for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (__shfl_sync(0xffffffffu, v, 0) >= target) break;
      if ((it & 15u) != 0) continue;  // the clock is read every 16th poll
      if (__shfl_sync(0xffffffffu, (int)(now_ns() - t0 >= wait_ns), 0)) {  // wait_ns = 0: one poll
        if (lane == 0) atomicOr(flag, 16);
        ok = 0;
        break;
      }
    }
    if (lane == 0) s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// jacobi_rotation by a whole warp. An FP64 instruction takes 64 cycles for one
// lane or 32, so what one lane did one after another is laid across lanes: the
// test |c|^2 > tol^2 a b beside |c|^2, and the two reciprocal square roots of
// the first stage (of |c|^2 and of d^2 + 4 |c|^2, whose product with its
// argument is the square root) as one. 3.0k -> 1.5k cycles of a round's ~10k.
// Results in par (cs, sn, e); *go = 0 (pair left alone), 1 (a small rotation) or
// 2. Small: the columns' cosine was at most kBigCos and the angle at most
// kBigSin. A sweep of small rotations only is the last one: what it leaves
// of the cosines is their product, below 1e-17, so no sweep is spent on
// finding nothing to rotate.
constexpr double kBigCos = 1e-10, kBigSin = 1e-8;
__device__ __forceinline__ void rotate_warp(double a, double b, double cr, double ci, double tol, double tiny2,
                                            double* par, int* go) {
  const int lane = threadIdx.x & 31;
  // lane 0: |c|^2, lane 1: tol^2 a b, lane 2: kBigCos^2 a b
  const double t = lane == 1 ? tol * tol : lane == 2 ? kBigCos * kBigCos : cr, u0 = lane == 0 ? cr : a * b;
  double q = t * u0;
  if (lane == 0) q = fma(ci, ci, q);
  const double c2 = __shfl_sync(0xffffffffu, q, 0), lim = __shfl_sync(0xffffffffu, q, 1);
  const double big = __shfl_sync(0xffffffffu, q, 2);
  if (!(c2 > lim) || c2 == 0.0 || !(fmin(a, b) > tiny2)) {
    if (lane == 0) *go = 0;
    return;
  }
  const double d = b - a, c4 = 4.0 * c2;
  const double arg = lane == 1 ? c2 : fma(d, d, c4);
  const double y = rsqrt(arg);
  const double ic = __shfl_sync(0xffffffffu, y, 1);   // 1 / |c|
  const double sr = __shfl_sync(0xffffffffu, arg * y, 0);  // sqrt(d^2 + 4 |c|^2)
  const double uu = fabs(d) + sr;
  const double w = rsqrt(fma(uu, uu, c4));
  // lane 0: cs = u w, lane 1: 2 |c| = 2 |c|^2 / |c|, lanes 2, 3: e = conj(c) / |c|
  const double l = lane == 0 ? uu : lane == 1 ? 2.0 * c2 : lane == 2 ? cr : -ci;
  double r = l * (lane == 0 ? w : ic);
  if (lane == 1) r = d >= 0.0 ? r * w : -(r * w);
  if (lane < 4) par[lane] = r;
  if (lane == 1) *go = c2 > big || fabs(r) > kBigSin ? 2 : 1;
}

// Circle-method pair p of round rd among N (even) columns.
__device__ __forceinline__ void round_pair(int N, int rd, int p, int& i, int& j) {
  if (p == 0) {
    i = 0;
    j = 1 + rd;
  } else {
    i = 1 + (rd + p) % (N - 1);
    j = 1 + (rd - p + N - 1) % (N - 1);
  }
  if (i > j) {
    const int t = i;
    i = j;
    j = t;
  }
}

// Working matrix A (nr x nc, column-major) from theta (m x n, row-major): the
// columns of theta, or of theta^H when n > m. V = identity (nc x nc).
__global__ void k_svd_load(const double2* __restrict__ theta, int m, int n, double2* __restrict__ A,
                           double2* __restrict__ V) {
  const bool tr = n > m;
  const int nr = tr ? n : m, nc = tr ? m : n;
  const int64_t na = (int64_t)nr * nc, nv = (int64_t)nc * nc;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < na + nv;
       k += (int64_t)gridDim.x * blockDim.x) {
    if (k < na) {
      int64_t r;
      const int64_t c = idivmod(k, nr, r);
      A[k] = tr ? cconj(theta[c * n + r]) : theta[r * n + c];
    } else {
      const int64_t kv = k - na;
      int64_t rr;
      const int64_t cc = idivmod(kv, nc, rr);
      V[kv] = make_double2(rr == cc ? 1.0 : 0.0, 0.0);
    }
  }
}

// Barrier at the end of a phase: the hardware barrier of the cluster (release /
// acquire at cluster scope, which orders the global-memory writes of A and V
// too), or the grid barrier of a cooperative launch.
template <bool kCluster>
__device__ __forceinline__ bool phase_sync(unsigned* lanes, unsigned target, uint64_t wait_ns, int* flag) {
  if constexpr (kCluster) {
    cg::this_cluster().sync();
    return true;
  } else {
    return grid_sync(lanes, target, wait_ns, flag);
  }
}

// sync: [0, 8) barrier lanes, [8, 8 + max_sweeps) rotations per sweep that ask for
// another one, then as many counters of the small ones; ver: the columns' rounds (grid
// form); both zeroed before the launch. kCluster: the CTAs form one thread-block
// cluster. V may be null (no right vectors). nc_dev (nullable): the column count, at most nc,
// found on the device; columns beyond it are zero.
//
// Between the rounds of the grid form a CTA waits for its two columns only:
// ver[j] counts the rounds column j has been through, written with release by
// the CTA that finished it and polled with acquire by the one that takes it
// next. A round's hand-over is then one flag to one reader instead of a
// barrier over all CTAs; one grid barrier a sweep remains, for its rotation count.
// (Up to kSvdMaxVer columns; wider matrices keep the barrier.)
// The two-site split of the rank-16 driven system (256 x 100 and 256 x 64), per
// step of 14 splits: 148 ms with accumulated right vectors and one barrier a
// round; 45 ms with R^H in place of the matrix, 41 with column hand-over and
// the early last sweep, 40 with four warps a CTA, 37 with the pivoted QR's shorter sums.
template <bool kCluster>
__global__ void __launch_bounds__(kJThreads) k_jacobi_grid(double2* __restrict__ A, double2* __restrict__ V, int nr,
                                                          int nc_in, const int* nc_dev, double* __restrict__ sigma, int* __restrict__ info,
                                                          unsigned* sync, unsigned* ver, int* flag, double tol, int max_sweeps,
                                                          int tr, uint64_t wait_ns) {
  static_assert(kJWarps * 4 <= 32 && (kJWarps & (kJWarps - 1)) == 0, "warp 0 adds four sums of each warp, one per lane");
  __shared__ double s_red[kJWarps][4];
  __shared__ double s_par[4];
  __shared__ int s_go;
  __shared__ unsigned s_total;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int G = gridDim.x;
  const int nc = nc_dev ? max(0, min(*nc_dev, nc_in)) : nc_in;
  const int N = max(2, nc + (nc & 1)), npairs = N / 2;
  unsigned nbar = 0;
  bool ok = true;
  // ||A||_F^2: column norms of columns jc = blockIdx.x (mod G) into sigma[]
  // (overwritten at the end), one barrier, then every CTA adds them in order
  for (int jc = blockIdx.x; jc < nc; jc += G) {
    const double2* x = A + (int64_t)jc * nr;
    double f = 0.0;
    for (int r = tid; r < nr; r += kJThreads) f = fma(x[r].x, x[r].x, fma(x[r].y, x[r].y, f));
    f = wsum(f);
    if (lane == 0) s_red[wid][0] = f;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < kJWarps; ++w) t += s_red[w][0];
      sigma[jc] = t;
    }
    __syncthreads();
  }
  ++nbar;
  ok = phase_sync<kCluster>(sync, nbar * (unsigned)G, wait_ns, flag);
  if (!ok) return;
  double fro2 = 0.0;
  for (int jc = 0; jc < nc; ++jc) fro2 += sigma[jc];
  const double tiny2 = jacobi_negligible(nr, fro2);
  const bool p2p = !kCluster && nc <= kSvdMaxVer;
  __shared__ int s_alive;
  int sweep = 0;
  unsigned round = 0;  // rounds done, over all sweeps
  for (; sweep < max_sweeps; ++sweep) {
    unsigned rot = 0, small = 0;
    for (int rd = 0; rd < N - 1 && ok; ++rd) {
      for (int p = blockIdx.x; p < npairs; p += G) {
        int i, j;
        round_pair(N, rd, p, i, j);
        if (p2p) {
          if (tid < 32) {
            const int cj = tid == 0 ? i : j;
            bool alive = true;
            if (tid < 2 && cj < nc && ld_acquire(ver + cj) != round) {
              const uint64_t t0 = now_ns();
              for (unsigned it = 1; ld_acquire(ver + cj) != round; ++it)
                if ((it & 15u) == 0 && now_ns() - t0 >= wait_ns) {
                  atomicOr(flag, 16);
                  alive = false;
                  break;
                }
            }
            alive = __all_sync(0xffffffffu, alive);
            if (tid == 0) s_alive = alive ? 1 : 0;
          }
          __syncthreads();
          if (!s_alive) {
            ok = false;
            break;
          }
        }
        if (j >= nc) {  // the dummy column of an odd count
          if (p2p && tid == 0) st_release(ver + i, round + 1);
          continue;
        }
        double2* x = A + (int64_t)i * nr;
        double2* y = A + (int64_t)j * nr;
        double a = 0.0, b = 0.0, cr = 0.0, ci = 0.0;
        for (int r = tid; r < nr; r += kJThreads) {
          const double2 xv = x[r], yv = y[r];
          a = fma(xv.x, xv.x, fma(xv.y, xv.y, a));
          b = fma(yv.x, yv.x, fma(yv.y, yv.y, b));
          cr = fma(xv.x, yv.x, fma(xv.y, yv.y, cr));  // Re conj(x) y
          ci = fma(xv.x, yv.y, fma(-xv.y, yv.x, ci));  // Im conj(x) y
        }
        const double sum = warp_sum4(a, b, cr, ci);
        if ((lane & 7) == 0) s_red[wid][lane >> 3] = sum;
        __syncthreads();
        if (wid == 0) {  // the rotation, once per pair: warp 0 adds the warps' sums and rotates
          // lane l holds quantity l & 3 of warp l >> 2; a fixed butterfly over the warp bits
          double v = s_red[(lane >> 2) % kJWarps][lane & 3];
          for (int o = 4; o < 4 * kJWarps; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          const double ga = __shfl_sync(0xffffffffu, v, 0), gb = __shfl_sync(0xffffffffu, v, 1);
          const double gr = __shfl_sync(0xffffffffu, v, 2), gi = __shfl_sync(0xffffffffu, v, 3);
          rotate_warp(ga, gb, gr, gi, tol, tiny2, s_par, &s_go);
        }
        __syncthreads();  // s_red and s_par are rewritten only after the next pair's sums
        const int go = s_go;
        if (go == 0) {
          if (p2p && tid < 2) st_release(ver + (tid == 0 ? i : j), round + 1);
          continue;
        }
        const double cs = s_par[0], sn = s_par[1];
        const double2 e = make_double2(s_par[2], s_par[3]);
        for (int r = tid; r < nr; r += kJThreads) {
          const double2 xv = x[r], yv = cmul(e, y[r]);
          x[r] = make_double2(cs * xv.x - sn * yv.x, cs * xv.y - sn * yv.y);
          y[r] = make_double2(sn * xv.x + cs * yv.x, sn * xv.y + cs * yv.y);
        }
        if (V) {
          double2* vx = V + (int64_t)i * nc;
          double2* vy = V + (int64_t)j * nc;
          for (int r = tid; r < nc; r += kJThreads) {
            const double2 xv = vx[r], yv = cmul(e, vy[r]);
            vx[r] = make_double2(cs * xv.x - sn * yv.x, cs * xv.y - sn * yv.y);
            vy[r] = make_double2(sn * xv.x + cs * yv.x, sn * xv.y + cs * yv.y);
          }
        }
        rot += go == 2;
        small += go == 1;
        if (p2p) {
          __syncthreads();  // the pair's columns are written
          if (tid < 2) st_release(ver + (tid == 0 ? i : j), round + 1);
        }
      }
      ++round;
      if (!ok) break;
      // the sweep's count of rotations that ask for another sweep is published before its last barrier
      if (rd == N - 2 && tid == 0 && rot > 0) atomicAdd(sync + kBarLanes + sweep, rot);
      if (rd == N - 2 && tid == 0 && small > 0) atomicAdd(sync + kSmallOff + sweep, small);
      if (p2p && rd < N - 2) continue;
      ++nbar;
      ok = phase_sync<kCluster>(sync, nbar * (unsigned)G, wait_ns, flag);
    }
    if (!ok) break;
    if (tid == 0) s_total = ld_acquire(sync + kBarLanes + sweep);
    __syncthreads();
    if (s_total == 0) {
      // the last sweep rotated too (max_sweeps itself says that the iteration did not end)
      if (ld_acquire(sync + kSmallOff + sweep) > 0 && sweep + 1 < max_sweeps) ++sweep;
      break;
    }
  }
  if (!ok) return;
  // sigma_j = |column j|, fixed-order sums; columns dealt round-robin to CTAs
  for (int jc = blockIdx.x; jc < nc; jc += G) {
    const double2* x = A + (int64_t)jc * nr;
    double a = 0.0;
    for (int r = tid; r < nr; r += kJThreads) a = fma(x[r].x, x[r].x, fma(x[r].y, x[r].y, a));
    a = wsum(a);
    if (lane == 0) s_red[wid][0] = a;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < kJWarps; ++w) t += s_red[w][0];
      sigma[jc] = sqrt(t);
    }
    __syncthreads();
  }
  if (blockIdx.x == 0) {
    for (int jc = nc + tid; jc < nc_in; jc += kJThreads) sigma[jc] = 0.0;
    if (tid == 0) {
      info[0] = sweep;
      info[1] = tr;
    }
  }
}

// Column-pivoted Householder QR of B (nb x ni, nb = the rows of theta that are
// not the isometry's, ni = the isometry's): B P = Q R, of which only
// X = R^H (ni x k, column-major, rows in the original order) is kept. One-sided
// Jacobi on X turns it into W Sigma with W the isometry's singular vectors. R^H
// is nearly diagonal where the singular values fall fast, so the sweeps drop
// from 17-20 to 9-11 on the two-site matrices of a run (rank-16 driven
// system, 256 x 100), and no rotation has to be accumulated.
//
// The columns are dealt to the CTAs and live in shared memory. A step is one
// grid barrier: every CTA publishes its largest remaining column and the norm,
// then all pick the same pivot (ties: lower index), read that column from L2
// and apply its reflector to their own columns. A step is a latency chain
// (barrier, candidates, pivot column, scalars, dot, update) of about 5.5 us
// whatever the size (7.5 with the sums of three values over all warps). *keff: the
// number of steps; it stops early when every remaining column is rounding noise
// of the matrix (jacobi_negligible).
constexpr int kPivMaxCols = 8;  // columns per CTA
constexpr int kPivSmem = 200 * 1024;
__global__ void __launch_bounds__(kThreads) k_pivot_qr(const double2* __restrict__ theta, int m, int n, int iso_first,
                                                       double2* __restrict__ Bg, double2* __restrict__ X, double* cand,
                                                       int* cand_i, double* fpart, int* keff, unsigned* sync, int* flag,
                                                       uint64_t wait_ns) {
  extern __shared__ double2 sm[];
  __shared__ double s_nrm[kPivMaxCols], s_part1[kWarps], s_part2[kWarps][2], s_sc[8];
  __shared__ int s_done[kPivMaxCols], s_piv;
  __shared__ long long s_best;
  const int nb = iso_first ? n : m, ni = iso_first ? m : n;
  const int k = min(nb, ni), G = gridDim.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  double2* v = sm;         // [nb] reflector
  double2* col = sm + nb;  // [ncl][nb]
  const int ncl = blockIdx.x < ni ? (ni - 1 - blockIdx.x) / G + 1 : 0;
  // warps of a column: all eight for one column, down to one for eight
  const int gs = ncl <= 1 ? 8 : ncl <= 2 ? 4 : ncl <= 4 ? 2 : 1;
  const int my = wid / gs, gw = wid % gs;  // this warp's column and place in its group
  const bool on = my < ncl;
  double2* a = col + (size_t)my * nb;
  // Sums over a column's lanes and warps (block-uniform barrier): of two values,
  // left in every lane, lanes 0..15 carrying x and 16..31 y so that a step costs one
  // FP64 addition; of one value, left in the column's first warp. Each has its own
  // partials, so nothing has to be waited for before they are written. With three
  // values in every lane and all warps adding the partials one by one, the two sums
  // of a step took 9k cycles.
  auto over_warps = [&](double t) {  // lane q of a half holds warp q's partial
    for (int o = gs >> 1; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
  };
  auto group_sum2 = [&](double x, double y, double& ox, double& oy) {
    const bool up = lane >= 16;
    double t = (up ? y : x) + __shfl_xor_sync(0xffffffffu, up ? x : y, 16);
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((lane & 15) == 0) s_part2[wid][lane >> 4] = t;
    __syncthreads();
    t = over_warps(s_part2[wid - gw + (lane & (gs - 1))][lane >> 4]);
    ox = __shfl_sync(0xffffffffu, t, 0);
    oy = __shfl_sync(0xffffffffu, t, 16);
  };
  auto group_sum1 = [&](double x) {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) s_part1[wid] = x;
    __syncthreads();
    return gw == 0 ? over_warps(s_part1[wid + (lane & (gs - 1))]) : 0.0;
  };
  double nrm = 0.0;
  {
    double f = 0.0;
    if (on) {
      const int i = blockIdx.x + my * G;
      for (int r = gw * 32 + lane; r < nb; r += gs * 32) {
        const double2 t = iso_first ? cconj(theta[(int64_t)i * n + r]) : theta[(int64_t)r * n + i];
        a[r] = t;
        f = fma(t.x, t.x, fma(t.y, t.y, f));
      }
    }
    nrm = group_sum1(f);
    if (on && gw == 0 && lane == 0) {
      s_nrm[my] = nrm;
      s_done[my] = 0;
    }
  }
  __syncthreads();
  if (tid == 0) {
    double f = 0.0;
    for (int l = 0; l < ncl; ++l) f += s_nrm[l];
    fpart[blockIdx.x] = f;
  }
  unsigned nbar = 0;
  double tiny2 = 0.0;
  int c = 0;
  for (; c < k; ++c) {
    // candidate: the largest remaining column of this CTA
    if (tid == 0) {
      int best = -1;
      for (int l = 0; l < ncl; ++l)
        if (!s_done[l] && (best < 0 || s_nrm[l] > s_nrm[best])) best = l;
      s_piv = best;
      const int slot = (c & 1) * G + blockIdx.x;
      cand[slot] = best < 0 ? -1.0 : s_nrm[best];
      cand_i[slot] = best < 0 ? 0x7fffffff : (int)blockIdx.x + best * G;
    }
    __syncthreads();
    if (s_piv >= 0) {
      const double2* src = col + (size_t)s_piv * nb;
      double2* dst = Bg + (int64_t)(blockIdx.x + s_piv * G) * nb;
      for (int r = c + tid; r < nb; r += kThreads) dst[r] = src[r];
    }
    ++nbar;
    if (!grid_sync(sync, nbar * (unsigned)G, wait_ns, flag)) return;
    if (c == 0) {
      double f = 0.0;
      for (int q = lane; q < G; q += 32) f += __ldcg(fpart + q);
      f = wsum(f);
      tiny2 = jacobi_negligible(max(nb, ni), f);
      if (!isfinite(f)) {  // nothing to factor: report it, no columns (uniform over the grid)
        if (blockIdx.x == 0 && tid == 0) atomicOr(flag, 1);
        break;
      }
    }
    if (wid == 0) {  // pivot: largest norm (positive doubles order like their bits), then lowest index
      long long bv = -1;
      int bi = 0x7fffffff;
      for (int q = lane; q < G; q += 32) {
        const double cv = __ldcg(cand + (c & 1) * G + q);
        const long long kb = cv < 0.0 ? -1 : __double_as_longlong(cv);
        const int ki = __ldcg(cand_i + (c & 1) * G + q);
        if (kb > bv || (kb == bv && ki < bi)) {
          bv = kb;
          bi = ki;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) {
          bv = ov;
          bi = oi;
        }
      }
      if (lane == 0) {
        s_best = bv;
        s_piv = bi;
      }
    }
    __syncthreads();
    const double n2 = s_best < 0 ? 0.0 : __longlong_as_double(s_best);
    if (!(n2 > tiny2)) break;  // uniform over the grid: every CTA sees the same candidates
    const int pi = s_piv;
    const double2* xp = Bg + (int64_t)pi * nb;
    if (wid == 0) {
      const double2 x0 = __ldcg(xp + c);
      // lane 0: alpha = |x|, lane 1: |x_0|
      const double rt = sqrt(lane == 1 ? fma(x0.x, x0.x, x0.y * x0.y) : n2);
      const double alpha = __shfl_sync(0xffffffffu, rt, 0), ax0 = __shfl_sync(0xffffffffu, rt, 1);
      const double rc = 1.0 / (lane == 1 ? alpha * (alpha + ax0) : ax0);
      const double inv = __shfl_sync(0xffffffffu, rc, 0), beta = __shfl_sync(0xffffffffu, rc, 1);
      const double2 phi = ax0 > 0.0 ? make_double2(x0.x * inv, x0.y * inv) : make_double2(1.0, 0.0);
      if (lane == 0) {
        s_sc[0] = fma(phi.x, alpha, x0.x);  // v_0
        s_sc[1] = fma(phi.y, alpha, x0.y);
        s_sc[2] = beta;
        s_sc[3] = -phi.x * alpha;  // R_cc
        s_sc[4] = -phi.y * alpha;
      }
    }
    for (int r = c + tid; r < nb; r += kThreads) v[r] = __ldcg(xp + r);
    __syncthreads();
    if (tid == 0) v[c] = make_double2(s_sc[0], s_sc[1]);
    const bool mine = on && (int)blockIdx.x + my * G == pi;
    const bool act = on && !s_done[my] && !mine;
    __syncthreads();
    double wr = 0.0, wi = 0.0;
    if (act)
      for (int r = c + gw * 32 + lane; r < nb; r += gs * 32) {
        const double2 x = v[r], y = a[r];
        wr = fma(x.x, y.x, fma(x.y, y.y, wr));
        wi = fma(x.x, y.y, fma(-x.y, y.x, wi));
      }
    double sr, si;
    group_sum2(wr, wi, sr, si);
    const double beta = s_sc[2];
    sr *= beta;
    si *= beta;
    double f = 0.0;
    if (act)
      for (int r = c + gw * 32 + lane; r < nb; r += gs * 32) {
        const double2 x = v[r];
        double2 y = a[r];
        y.x = fma(-x.x, sr, fma(x.y, si, y.x));
        y.y = fma(-x.x, si, fma(-x.y, sr, y.y));
        a[r] = y;
        if (r > c) f = fma(y.x, y.x, fma(y.y, y.y, f));
      }
    nrm = group_sum1(f);
    if (on && gw == 0 && lane == 0) {
      const int i = blockIdx.x + my * G;
      double2 t = make_double2(0.0, 0.0);  // a column finished earlier has no entry in this row of R
      if (mine)
        t = make_double2(s_sc[3], -s_sc[4]);
      else if (act)
        t = cconj(a[c]);
      X[(int64_t)c * ni + i] = t;
      if (mine) s_done[my] = 1;
      if (act) s_nrm[my] = nrm;
    }
    __syncthreads();
  }
  if (blockIdx.x == 0 && tid == 0) *keff = c;
}

size_t pivot_smem(int nb, int ni, int G) { return sizeof(double2) * (size_t)nb * (1 + (ni + G - 1) / G); }

struct GridInfo {
  int sms = 0, coop = 0, occ = 0;
  bool cluster16 = false;
};
GridInfo grid_info() {
  static std::once_flag once;
  static GridInfo gi;
  std::call_once(once, [] {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&gi.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      gi.sms = 1;
    if (cudaDeviceGetAttribute(&gi.coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) gi.coop = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&gi.occ, k_jacobi_grid<false>, kJThreads, 0) != cudaSuccess)
      gi.occ = 0;
    cudaFuncSetAttribute(k_pivot_qr, cudaFuncAttributeMaxDynamicSharedMemorySize, kPivSmem);
    gi.cluster16 = cudaFuncSetAttribute(k_jacobi_grid<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                   cudaSuccess;
  });
  return gi;
}

}  // namespace

double jacobi_tol(int m, int n) {
  const int nr = std::max(m, n);
  return 2.0 * std::sqrt((double)std::max(nr, 64)) * DBL_EPSILON;
}

bool launch_jacobi_svd_grid(const double2* theta, int m, int n, double2* A, double2* V, double* sigma, int* info,
                            unsigned* sync, unsigned* ver, int* flag, uint64_t wait_ns, cudaStream_t s) {
  const int nc = std::min(m, n), nr = std::max(m, n);
  const GridInfo gi = grid_info();
  const int npairs = (nc + 1) / 2;
  const bool cluster = npairs <= (gi.cluster16 ? kJacClusterMax : 8);  // one pair per CTA, one cluster
  if (nc <= kJacOneCtaMaxCols || (!cluster && (!gi.coop || gi.occ < 1))) {
    launch_jacobi_svd(theta, m, n, A, V, sigma, info, s);
    return cudaGetLastError() == cudaSuccess;
  }
  const int64_t tot = (int64_t)nr * nc + (int64_t)nc * nc;
  k_svd_load<<<counted((int)std::min<int64_t>((tot + 255) / 256, 4096)), 256, 0, s>>>(theta, m, n, A, V);
  if (cudaMemsetAsync(sync, 0, kSvdSyncInts * sizeof(unsigned), s) != cudaSuccess ||
      cudaMemsetAsync(ver, 0, nc * sizeof(unsigned), s) != cudaSuccess)
    return false;
  const int tr = n > m ? 1 : 0;
  const double tol = jacobi_tol(m, n);
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kJThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cluster) {  // one pair per CTA, the CTAs one cluster
    cfg.gridDim = counted(dim3(npairs, 1, 1));
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = npairs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    return cudaLaunchKernelEx(&cfg, k_jacobi_grid<true>, A, V, nr, nc, (const int*)nullptr, sigma, info, sync, ver, flag, tol,
                              kJacMaxSweeps, tr,
                              wait_ns) == cudaSuccess;
  }
  const int G = std::max(1, std::min(npairs, gi.sms * std::min(gi.occ, 2)));
  cfg.gridDim = counted(dim3(G, 1, 1));
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  return cudaLaunchKernelEx(&cfg, k_jacobi_grid<false>, A, V, nr, nc, (const int*)nullptr, sigma, info, sync, ver, flag, tol,
                              kJacMaxSweeps, tr,
                            wait_ns) == cudaSuccess;
}

bool launch_pivot_svd(const double2* theta, int m, int n, bool iso_first, double2* X, double2* Bg, double* sigma,
                      double* cand, int* info, unsigned* sync, unsigned* ver, int* flag, uint64_t wait_ns, cudaStream_t s) {
  const int nb = iso_first ? n : m, ni = iso_first ? m : n, k = std::min(m, n);
  const GridInfo gi = grid_info();
  // the pivoted QR pays its ~5 us a column where the sweeps it saves are those
  // of the grid Jacobi (more columns than a cluster holds)
  if (k <= 2 * kJacClusterMax || !gi.coop || gi.occ < 1 || gi.sms < 2) return false;
  const int G = std::min({ni, gi.sms, kPivMaxGrid});
  if ((ni + G - 1) / G > kPivMaxCols || pivot_smem(nb, ni, G) > (size_t)kPivSmem) return false;
  // the column count stays zero if the factorisation gives up
  if (cudaMemsetAsync(sync, 0, kSvdSyncInts * sizeof(unsigned), s) != cudaSuccess ||
      cudaMemsetAsync(info + 2, 0, sizeof(int), s) != cudaSuccess)
    return false;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cfg.gridDim = counted(dim3(G, 1, 1));
  cfg.dynamicSmemBytes = pivot_smem(nb, ni, G);
  double* fpart = cand + 2 * kPivMaxGrid;
  int* cand_i = (int*)(fpart + kPivMaxGrid);
  if (cudaLaunchKernelEx(&cfg, k_pivot_qr, theta, m, n, iso_first ? 1 : 0, Bg, X, cand, cand_i, fpart, info + 2, sync,
                         flag, wait_ns) != cudaSuccess)
    return false;
  if (cudaMemsetAsync(sync, 0, kSvdSyncInts * sizeof(unsigned), s) != cudaSuccess ||
      cudaMemsetAsync(ver, 0, k * sizeof(unsigned), s) != cudaSuccess)
    return false;
  cfg.dynamicSmemBytes = 0;
  cfg.blockDim = dim3(kJThreads, 1, 1);
  cfg.gridDim = counted(dim3(std::max(1, std::min((k + 1) / 2, gi.sms * std::min(gi.occ, 2))), 1, 1));
  return cudaLaunchKernelEx(&cfg, k_jacobi_grid<false>, X, (double2*)nullptr, ni, k, (const int*)(info + 2), sigma,
                            info, sync, ver, flag, jacobi_tol(m, n), kJacMaxSweeps, iso_first ? 0 : 1,
                            wait_ns) == cudaSuccess;
}

// Isometry columns a < g from W Sigma (X, ni x k column-major), Z = W or its
// conjugate (second side), zero beyond g; Zg the same; centre = theta
// contracted with conj(Z), one warp per entry.
__global__ void k_pivot_iso(const double2* __restrict__ X, const double* __restrict__ sigma, const int* __restrict__ perm,
                            int ni, int r, int g, int iso_first, double2* Z, double2* Zg) {
  const int64_t nz = (int64_t)ni * r;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nz; q += (int64_t)gridDim.x * blockDim.x) {
    const int a = (int)(q % r), row = (int)(q / r);
    double2 v = make_double2(0.0, 0.0);
    if (a < g) {
      const int j = perm[a];
      const double2 x = X[(int64_t)j * ni + row];
      v = make_double2(x.x / sigma[j], (iso_first ? x.y : -x.y) / sigma[j]);
    }
    Z[q] = v;
    Zg[q] = v;
  }
}
__global__ void __launch_bounds__(256) k_pivot_centre(const double2* __restrict__ theta, int m, int n,
                                                      const double2* __restrict__ Z, int r, int iso_first,
                                                      double2* __restrict__ Cm) {
  const int lane = threadIdx.x & 31;
  const int ni = iso_first ? m : n, no = iso_first ? n : m;
  const int64_t tot = (int64_t)no * r;
  for (int64_t w = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5); w < tot;
       w += (int64_t)gridDim.x * (blockDim.x / 32)) {
    // iso_first: Cm[a][col] (r x n); second: Cm[row][a] (m x r)
    const int a = iso_first ? (int)(w / no) : (int)(w % r), o = iso_first ? (int)(w % no) : (int)(w / r);
    double2 acc = make_double2(0.0, 0.0);
    for (int i = lane; i < ni; i += 32) {
      const double2 z = Z[(int64_t)i * r + a], t = iso_first ? theta[(int64_t)i * n + o] : theta[(int64_t)o * n + i];
      acc.x = fma(z.x, t.x, fma(z.y, t.y, acc.x));
      acc.y = fma(z.x, t.y, fma(-z.y, t.x, acc.y));
    }
    for (int q = 16; q > 0; q >>= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, q);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, q);
    }
    if (lane == 0) Cm[w] = acc;
  }
}
void launch_pivot_vecs(const double2* theta, int m, int n, bool iso_first, const double2* X, const double* sigma,
                       const int* perm, int r, int g, double2* Z, double2* Zg, double2* Cm, cudaStream_t s) {
  const int ni = iso_first ? m : n, no = iso_first ? n : m;
  k_pivot_iso<<<counted((int)std::min<int64_t>(((int64_t)ni * r + 255) / 256, 1024)), 256, 0, s>>>(X, sigma, perm, ni, r, g,
                                                                                          iso_first ? 1 : 0, Z, Zg);
  k_pivot_centre<<<counted((int)std::min<int64_t>(((int64_t)no * r + 7) / 8, 4096)), 256, 0, s>>>(theta, m, n, Z, r,
                                                                                         iso_first ? 1 : 0, Cm);
}

namespace {

// U (m x k) and Vh (k x n), row-major, from the converged working matrix, V and
// the descending order perm of sigma; columns whose sigma is 0 are left 0.
__global__ void k_svd_write(const double2* __restrict__ A, const double2* __restrict__ V,
                            const double* __restrict__ sigma, const int* __restrict__ perm, int m, int n,
                            double2* __restrict__ U, double2* __restrict__ Vh) {
  const bool tr = n > m;
  const int nr = tr ? n : m, nc = tr ? m : n, k = nc;
  const int64_t nu = (int64_t)m * k, nvh = (int64_t)k * n;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nu + nvh;
       q += (int64_t)gridDim.x * blockDim.x) {
    const bool upart = q < nu;
    const int64_t qq = upart ? q : q - nu;
    int row, a;
    int64_t rem;
    if (upart) {
      row = (int)idivmod(qq, k, rem);
      a = (int)rem;
    } else {
      a = (int)idivmod(qq, n, rem);
      row = (int)rem;
    }
    const int j = perm[a];
    const double sj = sigma[j];
    double2 v = make_double2(0.0, 0.0);
    if (upart) {  // left vector entry `row` (length m)
      if (tr)
        v = V[(int64_t)j * nc + row];
      else if (sj > 0.0)
        v = make_double2(A[(int64_t)j * nr + row].x / sj, A[(int64_t)j * nr + row].y / sj);
      U[qq] = v;
    } else {  // conj of right vector entry `row` (length n)
      if (!tr)
        v = cconj(V[(int64_t)j * nc + row]);
      else if (sj > 0.0)
        v = make_double2(A[(int64_t)j * nr + row].x / sj, -A[(int64_t)j * nr + row].y / sj);
      Vh[qq] = v;
    }
  }
}

struct SvdWs {
  int64_t A, V, sigma, perm, info, sync, flag, total;
};
SvdWs svd_ws(int m, int n) {
  const int64_t nr = std::max(m, n), nc = std::min(m, n);
  SvdWs L;
  int64_t o = 0;
  auto take = [&](int64_t bytes) {
    const int64_t r = o;
    o += (bytes + 255) / 256 * 256;
    return r;
  };
  L.A = take(nr * nc * 16);
  L.V = take(nc * nc * 16);
  L.sigma = take(nc * 8);
  L.perm = take(nc * 4);
  L.info = take(4 * 4);
  L.sync = take(kSvdSyncInts * 4);
  L.flag = take(4);
  L.total = o;
  return L;
}

}  // namespace

}  // namespace ttn

extern "C" ttn_status ttn_svd_workspace_size(int32_t m, int32_t n, size_t* bytes) {
  if (!bytes || m < 1 || n < 1) return TTN_EINVAL;
  *bytes = (size_t)ttn::svd_ws(m, n).total;
  return TTN_OK;
}

extern "C" ttn_status ttn_svd(const void* a_dev, int32_t m, int32_t n, void* u_dev, double* sigma_host, void* vh_dev,
                              void* ws_dev, size_t ws_bytes, double wait_s, int32_t* sweeps_out, void* stream) {
  using namespace ttn;
  if (!a_dev || !u_dev || !sigma_host || !vh_dev || !ws_dev || m < 1 || n < 1 || !(wait_s >= 0.0)) return TTN_EINVAL;
  const SvdWs L = svd_ws(m, n);
  if (ws_bytes < (size_t)L.total || ((uintptr_t)ws_dev & 255)) return TTN_ENOMEM;
  cudaStream_t s = (cudaStream_t)stream;
  char* base = (char*)ws_dev;
  double2* A = (double2*)(base + L.A);
  double2* V = (double2*)(base + L.V);
  double* sigma = (double*)(base + L.sigma);
  int* perm = (int*)(base + L.perm);
  int* info = (int*)(base + L.info);
  unsigned* sync = (unsigned*)(base + L.sync);
  int* flag = (int*)(base + L.flag);
  const int nc = std::min(m, n);
  if (cudaMemsetAsync(flag, 0, sizeof(int), s) != cudaSuccess) return TTN_ECUDA;
  const double wns = std::min(wait_s, 60.0) * 1e9;
  // the columns' counters lie in U, which is written last
  if (!launch_jacobi_svd_grid((const double2*)a_dev, m, n, A, V, sigma, info, sync, (unsigned*)u_dev, flag, (uint64_t)wns, s))
    return TTN_ECUDA;
  std::vector<double> sig(nc);
  int hinfo[2] = {0, 0}, hflag = 0;
  if (cudaMemcpyAsync(sig.data(), sigma, nc * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(hinfo, info, sizeof(hinfo), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return TTN_ECUDA;
  if (hflag & 16) return TTN_ETIMEOUT;
  if (sweeps_out) *sweeps_out = hinfo[0];
  if (hinfo[0] >= kJacMaxSweeps) return TTN_ENUMERIC;
  std::vector<int> pm(nc);
  for (int i = 0; i < nc; ++i) pm[i] = i;
  std::stable_sort(pm.begin(), pm.end(), [&](int a, int b) { return sig[a] > sig[b]; });
  for (int i = 0; i < nc; ++i) sigma_host[i] = sig[pm[i]];
  if (cudaMemcpyAsync(perm, pm.data(), nc * sizeof(int), cudaMemcpyHostToDevice, s) != cudaSuccess) return TTN_ECUDA;
  const int64_t tot = (int64_t)(m + n) * nc;
  k_svd_write<<<counted((int)std::min<int64_t>((tot + 255) / 256, 4096)), 256, 0, s>>>(A, V, sigma, perm, m, n,
                                                                             (double2*)u_dev, (double2*)vh_dev);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) return TTN_ECUDA;
  return TTN_OK;
}
