// Householder QR of a node tensor spread over a thread-block cluster (FP64).
//
// GB300 retires FP64 at a small fraction of its FP32 rate: a warp issues one
// FP64 instruction per ~64 cycles, an SM about one per ~19 cycles, and an FP64
// square root or division costs ~600 cycles. The kernel is therefore laid out
// to keep the number of FP64 warp instructions on the critical path small:
//
//  * the m rows are split over C <= 16 CTAs of one cluster, each keeping its
//    row block in shared memory;
//  * a column costs ONE exchange: every CTA pushes (st.async into the other
//    CTAs' shared memory, completing bytes on their mbarrier) its partial
//    squared norm of column j and its partial dots u_k = x_j^H a_k, k > j, and
//    the CTA owning row j adds x_0 and row j of the trailing columns. With
//    v = x + phi*alpha*e_0 the reflector dot is then w_k = sum u_k + alpha
//    conj(phi) a_k[j], so norm and dots need no second round trip;
//  * alpha, phi and beta are computed by one warp (two lanes share each sqrt
//    and division) while the other warps sum the pushed dot partials;
//  * the update and the next column's partials use groups of 8 lanes per
//    trailing column (rows strided over the group), so each warp instruction
//    covers 4 columns;
//  * Q is formed from the compact WY form H_0..H_{n-1} = I - V T V^H, but
//    instead of the sequential recurrence for T, M = T V_top^H is obtained by
//    back substitution with T^{-1} = diag(1/beta) + strictly-upper(V^H V)
//    (Joffrain, Low, Quintana-Orti, van de Geijn, Van Zee 2006), one column of
//    M per warp, spread over the cluster.
//
// The arithmetic convention is the one of the CPU oracle and of the one-CTA
// kernel: for column j with remainder x of norm alpha, alpha <= tol*||A||_F
// means no reflector (R_jj = 0, Q column H_0..H_{j-1} e_j); otherwise
// v = x + phi*alpha*e_0, phi = x_0/|x_0| (1 if x_0 = 0), beta = 1/(alpha(alpha+|x_0|)),
// and finally row j of R / column j of Q are rescaled by the phase -phi so
// that diag(R) >= 0. All reductions run in a fixed order, so results are
// bitwise reproducible. Every wait on a peer is bounded (2 s from the kernel
// start): on expiry bit 2 of *flag is set and the kernel runs to its end
// without further exchanges.
#include <cooperative_groups.h>

#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace ttn {

namespace {

constexpr int kThreads = 256;
constexpr int kNW = kThreads / 32;
// G = lanes per trailing-column group (8 for whole small matrices, 32 for
// panels of tall matrices, whose row blocks are long)
template <int G> struct Grp {
  static constexpr int kGPW = 32 / G;             // column groups per warp
  static constexpr int kSlots = (kNW - 1) * kGPW;  // column groups of warps 1..7
  static constexpr int kMaxPass = (kQrClusterMaxN - 1 + kSlots - 1) / kSlots;
};
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ double2 cfmaj(double2 a, double2 b, double2 c) {  // conj(a)*b + c
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(-a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ double2 cfms(double2 a, double2 b, double2 c) {  // c - a*b
  c.x = fma(-a.x, b.x, c.x);
  c.x = fma(a.y, b.y, c.x);
  c.y = fma(-a.x, b.y, c.y);
  c.y = fma(-a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ double wsum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
// Sum over aligned groups of G lanes: lanes of the group's lower half get the
// real part, the upper half the imaginary part (the first exchange gives each
// half one component, so a level costs one FP64 addition, 64 cycles, not two;
// the sums are those of the plain butterfly).
template <int G>
__device__ __forceinline__ double gsum_split(double2 v) {
  const bool up = (threadIdx.x & (G / 2)) != 0;
  double k = up ? v.y : v.x;
  k += __shfl_xor_sync(kFull, up ? v.x : v.y, G / 2);
  for (int o = G / 4; o > 0; o >>= 1) k += __shfl_xor_sync(kFull, k, o);
  return k;
}
// (real, imaginary) in every lane from the split form
template <int G>
__device__ __forceinline__ double2 join_split(double k) {
  const bool up = (threadIdx.x & (G / 2)) != 0;
  const double o = __shfl_xor_sync(kFull, k, G / 2);
  return up ? make_double2(o, k) : make_double2(k, o);
}
// block sum in a fixed order; every thread gets the result
__device__ double bsum(double v, double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = wsum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < nw; ++w) s += red[w];
  __syncthreads();
  return s;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// address of the same shared variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_init(uint64_t* mb, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mb)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* mb, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mb)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* mb, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(mb)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait for the phase of the given parity; false (and bit 2 of *flag) once the
// kernel-wide deadline has passed.
__device__ __forceinline__ bool mbar_wait(uint64_t* mb, uint32_t parity, uint64_t deadline, int* flag) {
  for (unsigned it = 1; !mbar_try(mb, parity); ++it) {
    if ((it & 31u) == 0 && gtimer() > deadline) {
      atomicOr(flag, 2);
      return false;
    }
  }
  return true;
}
// remote stores into another CTA's shared memory that complete bytes on its mbarrier
__device__ __forceinline__ void push_f64(uint32_t raddr, double v, uint32_t rmb) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(raddr), "d"(v),
               "r"(rmb)
               : "memory");
}
__device__ __forceinline__ void push_c64(uint32_t raddr, double2 v, uint32_t rmb) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(raddr),
               "d"(v.x), "d"(v.y), "r"(rmb)
               : "memory");
}

}  // namespace

// Shared-memory layout (dynamic, double2 units):
//   A   [n][rp]     my row block, column-major (v_j overwrites rows >= j of column j)
//   SU  [2][16][n]  per-parity dot partials u_k pushed by each CTA
//   RJ  [2][n]      per-parity row j of the trailing columns (from the owner of row j)
//   GF  [n][n]      strictly-upper Gram of V, transposed
//   M   [n][n]      M; its own region where that fits, else GF's (one more
//                   cluster barrier). When not even GF fits, both are single
//                   copies in global memory behind the CTAs' partial Grams.
template <int GL>
__global__ void __launch_bounds__(kThreads) k_qr_cluster(double2* U, int d0, int d1, int d2, int leg,
                                                         double tol, double2* R, int* flag, float2* U_lo,
                                                         float2* R_lo, QrPanel pn) {
  using Gp = Grp<GL>;
  constexpr int kGPW = Gp::kGPW, kSlots = Gp::kSlots, kMaxPass = Gp::kMaxPass;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int me = (int)cluster.block_rank();
  const int dd[3] = {d0, d1, d2};
  const int64_t st[3] = {(int64_t)d1 * d2, d2, 1};
  const int la = leg == 0 ? 1 : 0, lb = leg == 2 ? 1 : 2;
  // panel mode: factor columns [c0, c0+nb) of the column-major m x n matrix
  // pn.A over rows [c0, m) -- an (m - c0) x nb matrix in its own right
  const bool panel = pn.A != nullptr;
  const int n = panel ? pn.nb : dd[leg];
  const int m = panel ? pn.m - pn.c0 : dd[la] * dd[lb];
  const int rp = (m + C - 1) / C;
  const int r0 = me * rp;
  const int nr = max(0, min(m, r0 + rp) - r0);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5;
  // column groups: warps 1..7, or, when six warps hold all columns, without
  // warp 4: it shares its SM sub-partition, and so its FP64 pipe, with warp 0, whose
  // scalar chain everything waits for
  const bool six = n <= 6 * kGPW;
  const int slots = six ? 6 * kGPW : kSlots;
  const int cw = !six ? wid - 1 : wid < 4 ? wid - 1 : wid == 4 ? -1 : wid - 2;  // place among the column warps, -1: none

  extern __shared__ double2 smem[];
  double2* A = smem;
  double2* SU = A + (size_t)n * rp;
  double2* RJ = SU + 32 * (size_t)n;
  const bool gt = !panel && pn.gtail != nullptr;
  const size_t n2 = (size_t)n * n;
  double2* GF = gt ? pn.gtail : RJ + 2 * (size_t)n;
  double2* M = gt ? pn.gtail + n2 : pn.m_apart ? GF + n2 : GF;
  __shared__ __align__(8) uint64_t mb[2], mbg[2];
  __shared__ double SN[2][16];
  __shared__ double2 SX[2];
  __shared__ double red[kNW];
  __shared__ double s_part, s_frob;
  __shared__ double s_beta[kQrClusterMaxN], s_alpha[kQrClusterMaxN];
  __shared__ int s_skip[kQrClusterMaxN];
  __shared__ double2 s_phase[kQrClusterMaxN];
  __shared__ double2 s_gam;
  if (tid == 0) {
    mbar_init(&mb[0], 1);
    mbar_init(&mb[1], 1);
    mbar_init(&mbg[0], 1);
    mbar_init(&mbg[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  grid_wait();
  const uint64_t deadline = gtimer() + 2000000000ull;
  // gather my rows: A[c][i] = U[.. row r0+i, column c ..] (panel: pn.A[c0+c][c0+r0+i])
  double fro = 0.0;
  for (int k = tid; k < n * rp; k += nt) {
    const int c = k / rp, i = k % rp;
    double2 v = make_double2(0.0, 0.0);
    if (i < nr) {
      const int r = r0 + i;
      v = panel ? pn.A[(int64_t)(pn.c0 + c) * pn.m + pn.c0 + r]
                : U[c * st[leg] + (int64_t)(r / dd[lb]) * st[la] + (int64_t)(r % dd[lb]) * st[lb]];
    }
    A[k] = v;
    fro = fma(v.x, v.x, fma(v.y, v.y, fro));
  }
  fro = bsum(fro, red);
  if (tid == 0) s_part = fro;
  cluster.sync();  // partial norms visible, mbarriers initialised cluster-wide
  if (wid == 0) {  // lane c reads CTA c's partial; fixed butterfly order
    double v = lane < C ? *cluster.map_shared_rank(&s_part, lane) : 0.0;
    v = wsum(v);
    if (lane == 0) s_frob = sqrt(v);
  }
  __syncthreads();
  // the threshold of a panel is the one of the whole matrix (NaN: abort)
  const double frob = panel ? *pn.thr : s_frob;
  if (!isfinite(frob)) {  // uniform across the cluster
    if (tid == 0 && me == 0 && !panel) atomicOr(flag, 1);
    cluster.sync();
    return;
  }
  const double thr = panel ? frob : tol * frob;  // s_part stays untouched until the final cluster barrier
  bool alive = true;

  // Partials of step j over my rows >= j, pushed into every CTA's slots of
  // parity j&1: ||x_j||^2 (warp 0), u_k = x_j^H a_k for k > j (column groups);
  // the CTA owning row j also pushes x_0 and a_k[j].
  auto push_partials = [&](int j) {
    const int p = j & 1;
    const int i0 = max(0, j - r0);
    const double2* x = A + (size_t)j * rp;
    const bool own = j >= r0 && j < r0 + nr;
    const int lrow = j - r0;
    if (tid == 0) {
      const uint32_t nk = (uint32_t)(n - j - 1);
      mbar_arrive_tx(&mb[p], 8u * C + 16u * C * nk + (j < m ? 16u + 16u * nk : 0u));
    }
    if (wid == 0) {
      double ss = 0.0;
      for (int i = i0 + lane; i < nr; i += 32) ss = fma(x[i].x, x[i].x, fma(x[i].y, x[i].y, ss));
      ss = wsum(ss);
      if (alive && lane < C) {
        const uint32_t rmb = mapa(smem_u32(&mb[p]), lane);
        push_f64(mapa(smem_u32(&SN[p][me]), lane), ss, rmb);
        if (own) push_c64(mapa(smem_u32(&SX[p]), lane), x[lrow], rmb);
      }
    } else if (cw >= 0) {
      const int q = cw * kGPW + lane / GL, sl = lane % GL;
      for (int kb = j + 1; kb < n; kb += slots) {  // block-uniform trip count
        const int k = kb + q;
        const double2* a = A + (size_t)min(k, n - 1) * rp;
        double2 u = make_double2(0.0, 0.0);
        if (k < n)
          for (int i = i0 + sl; i < nr; i += GL) u = cfmaj(x[i], a[i], u);
        u = join_split<GL>(gsum_split<GL>(u));
        if (alive && k < n) {
          const uint32_t su = smem_u32(&SU[((size_t)p * 16 + me) * n + k]);
          const uint32_t rj = smem_u32(&RJ[(size_t)p * n + k]);
          const uint32_t lmb = smem_u32(&mb[p]);
          for (int c = sl; c < C; c += GL) {
            const uint32_t rmb = mapa(lmb, c);
            push_c64(mapa(su, c), u, rmb);
            if (own) push_c64(mapa(rj, c), a[lrow], rmb);
          }
        }
      }
    }
  };

  // Column loop (see the header): wait for step j's partials, scalars in warp
  // 0 / dot sums in warps 1..7, barrier, update, barrier, push step j+1.
  // A push for step j+2 (same parity as j) can only leave a CTA after every
  // CTA has pushed for step j+1, i.e. after all threads here have passed the
  // second barrier of step j and are done with step j's slots and phase.
  push_partials(0);
  uint32_t ph[2] = {0u, 0u};
  for (int j = 0; j < n; ++j) {
    const int p = j & 1;
    const int i0 = max(0, j - r0);
    double2* x = A + (size_t)j * rp;
    const bool own = j >= r0 && j < r0 + nr;
    const int lrow = j - r0;
    if (alive) alive = mbar_wait(&mb[p], ph[p], deadline, flag);
    ph[p] ^= 1u;
    double W[kMaxPass];  // split form
    if (wid == 0) {
      // C <= 16: a half-warp carries the sum, both halves alike (a zero in any lane
      // would send the whole warp through the square root's slow path)
      double a2 = (lane & 15) < C ? SN[p][lane & 15] : 0.0;
      for (int o = 8; o > 0; o >>= 1) a2 += __shfl_xor_sync(kFull, a2, o);
      const double2 x0 = j < m ? SX[p] : make_double2(0.0, 0.0);
      // lane 0: alpha = sqrt(sum), lane 1: |x_0| (one sqrt for both)
      const double rt = sqrt(lane == 1 ? fma(x0.x, x0.x, x0.y * x0.y) : a2);
      const double alpha = __shfl_sync(kFull, rt, 0);
      const double ax0 = __shfl_sync(kFull, rt, 1);
      if (!(alpha > thr)) {
        for (int i = i0 + lane; i < nr; i += 32) x[i] = make_double2(0.0, 0.0);
        if (lane == 0) {
          s_skip[j] = 1;
          s_beta[j] = 0.0;
          s_alpha[j] = 0.0;
          s_phase[j] = make_double2(1.0, 0.0);
        }
      } else {
        // even lanes: 1/|x_0|, odd lanes: beta (one division for both)
        const double rc = 1.0 / ((lane & 1) ? alpha * (alpha + ax0) : ax0);
        const double inv = __shfl_sync(kFull, rc, 0);
        // lane 0 the real, lane 1 the imaginary part of phi, alpha conj(phi) and v_0
        const double xc = (lane & 1) ? x0.y : x0.x;
        const double phi = ax0 > 0.0 ? xc * inv : ((lane & 1) ? 0.0 : 1.0);
        const double ap = alpha * phi;
        if (lane < 2) {
          if (lane == 1) s_beta[j] = rc;
          if (lane == 0) {
            s_skip[j] = 0;
            s_alpha[j] = alpha;
          }
          reinterpret_cast<double*>(&s_phase[j])[lane] = -phi;
          reinterpret_cast<double*>(&s_gam)[lane] = lane == 0 ? ap : -ap;
          if (own) reinterpret_cast<double*>(&x[lrow])[lane] = fma(phi, alpha, xc);
        }
      }
    } else if (cw >= 0) {
      const int q = cw * kGPW + lane / GL, sl = lane % GL;
#pragma unroll
      for (int ps = 0; ps < kMaxPass; ++ps) {
        const int k = j + 1 + ps * slots + q;
        if (j + 1 + ps * slots >= n) break;  // block-uniform
        double2 w = make_double2(0.0, 0.0);
        if (k < n)
          for (int c = sl; c < C; c += GL) {
            const double2 t = SU[((size_t)p * 16 + c) * n + k];
            w.x += t.x;
            w.y += t.y;
          }
        W[ps] = gsum_split<GL>(w);
      }
    }
    __syncthreads();
    if (wid > 0 && cw >= 0 && !s_skip[j]) {
      const double beta = s_beta[j];
      const double2 gam = s_gam;
      const int q = cw * kGPW + lane / GL, sl = lane % GL;
#pragma unroll
      for (int ps = 0; ps < kMaxPass; ++ps) {
        const int k = j + 1 + ps * slots + q;
        if (j + 1 + ps * slots >= n) break;
        const double2 rj = RJ[(size_t)p * n + min(k, n - 1)];
        // w += gam rj, one component a lane: (gam.x rj.x - gam.y rj.y, gam.x rj.y + gam.y rj.x)
        const bool up = (lane & (GL / 2)) != 0;
        const double w = fma(gam.x, up ? rj.y : rj.x, fma(up ? gam.y : -gam.y, up ? rj.x : rj.y, W[ps]));
        const double2 bw = join_split<GL>(beta * w);
        if (k < n) {
          double2* a = A + (size_t)k * rp;
          for (int i = i0 + sl; i < nr; i += GL) a[i] = cfms(x[i], bw, a[i]);
        }
      }
    }
    __syncthreads();
    if (j + 1 < n) push_partials(j + 1);
  }
  cluster.sync();  // all reflectors final everywhere, every pushed slot consumed
  if (panel) {
    // write the panel back (v below the diagonal, R entries above), the
    // per-column scalars, and the WY factor T of the panel:
    // T^{-1} = diag(1/beta) + strictly-upper(V^H V), column c of T solved by
    // back substitution from e_c (skipped reflectors give zero rows/columns)
    for (int k = tid; k < n * nr; k += nt) {
      const int c = k / nr, i = k % nr;
      pn.A[(int64_t)(pn.c0 + c) * pn.m + pn.c0 + r0 + i] = A[(size_t)c * rp + i];
    }
    if (me == 0)
      for (int c = tid; c < n; c += nt) {
        pn.beta[pn.c0 + c] = s_beta[c];
        pn.alpha[pn.c0 + c] = s_alpha[c];
        pn.phase[pn.c0 + c] = s_phase[c];
        pn.skip[pn.c0 + c] = s_skip[c];
      }
  }

  // R rows owned here (global rows < n), diag(R) = alpha >= 0 after the phase fix
  for (int k = tid; !panel && k < n * n; k += nt) {
    const int i = k / n, c = k % n;
    if (i < r0 || i >= r0 + nr) continue;
    double2 v = make_double2(0.0, 0.0);
    if (c == i) {
      v = make_double2(s_skip[i] ? 0.0 : s_alpha[i], 0.0);
    } else if (c > i) {
      const double2 a = A[(size_t)c * rp + (i - r0)];
      const double2 p = s_phase[i];
      v = make_double2(a.x * p.x + a.y * p.y, a.y * p.x - a.x * p.y);  // conj(p) * a
    }
    R[k] = v;
    if (R_lo) R_lo[k] = make_float2((float)v.x, (float)v.y);
  }
  // Strictly-upper Gram of V (v_a vanishes above row a; skipped reflectors are
  // zero columns): one thread per pair a < b sums its rows; the partials of pair
  // t go to CTA t mod C, which adds them in CTA order and sends the sum to every
  // CTA (stored transposed, GF[b][a], so that the solves read along lanes).
  // Reading all partials of all CTAs everywhere took 11k cycles, this 4k.
  const int npair = n * (n - 1) / 2;
  auto pair_of = [](int t, int& a, int& b) {  // t = b(b-1)/2 + a
    b = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)t)) * 0.5f);
    while (b * (b - 1) / 2 > t) --b;
    while ((b + 1) * b / 2 <= t) ++b;
    a = t - b * (b - 1) / 2;
  };
  const int nown = me < npair ? (npair - 1 - me) / C + 1 : 0;  // pairs summed here
  const int nslot = (npair + C - 1) / C;
  if (tid == 0 && !gt) {
    mbar_arrive_tx(&mbg[0], 16u * C * nown);
    mbar_arrive_tx(&mbg[1], 16u * npair);
  }
  for (int t = tid; t < npair; t += nt) {
    int a, b;
    pair_of(t, a, b);
    double2 g = make_double2(0.0, 0.0);
    const double2* va = A + (size_t)a * rp;
    const double2* vb = A + (size_t)b * rp;
    for (int i = max(b - r0, 0); i < nr; ++i) g = cfmaj(va[i], vb[i], g);
    if (gt)
      pn.gtail[(size_t)(2 + me) * n2 + a * n + b] = g;
    else if (alive)  // SU is free after the column loop
      push_c64(mapa(smem_u32(&SU[(size_t)me * nslot + t / C]), t % C), g, mapa(smem_u32(&mbg[0]), t % C));
  }
  if (gt) {
    cluster.sync();
    for (int e = tid; e < nown; e += nt) {
      int a, b;
      pair_of(me + C * e, a, b);
      double2 g = make_double2(0.0, 0.0);
      for (int c = 0; c < C; ++c) {
        const double2 v = pn.gtail[(size_t)(2 + c) * n2 + a * n + b];
        g.x += v.x;
        g.y += v.y;
      }
      GF[b * n + a] = g;
    }
    cluster.sync();
  } else {
    if (alive) alive = mbar_wait(&mbg[0], 0u, deadline, flag);
    // one lane per component
    for (int e = tid; e < 2 * nown; e += nt) {
      const double* p = reinterpret_cast<const double*>(SU) + 2 * (size_t)(e >> 1) + (e & 1);
      double g = 0.0;
      for (int c = 0; c < C; ++c) g += p[2 * (size_t)c * nslot];
      int a, b;
      pair_of(me + C * (e >> 1), a, b);
      if (alive) {
        const uint32_t dst = smem_u32(reinterpret_cast<double*>(GF + b * n + a) + (e & 1)), lmb = smem_u32(&mbg[1]);
        for (int c = 0; c < C; ++c) push_f64(mapa(dst, c), g, mapa(lmb, c));
      }
    }
    if (alive) alive = mbar_wait(&mbg[1], 0u, deadline, flag);
  }
  __syncthreads();
  // Back substitution of one column, T^{-1} y = rhs with T^{-1} = diag(1/beta) +
  // strictly-upper Gram, from a = c down: lanes 0..15 carry real parts, 16..31
  // imaginary parts of entries 16 q + (lane & 15), so a step is one product and
  // two FMAs per block of 16 entries (an FP64 instruction costs 64 cycles
  // whatever the lanes). put(a, v) stores component lane >> 4 of entry a.
  auto solve = [&](int c, double (&acc)[kQrClusterMaxN / 16], auto&& put) {
    const int comp = lane >> 4, e = lane & 15;
    double beta = s_beta[c];
#pragma unroll
    for (int qa = kQrClusterMaxN / 16 - 1; qa >= 0; --qa) {
      if (c < 16 * qa) continue;
      double2 g[kQrClusterMaxN / 16];  // row a of the transposed Gram, read a step ahead
      const int a0 = min(c, 16 * qa + 15);
#pragma unroll
      for (int q = 0; q <= qa; ++q) g[q] = 16 * q + e < a0 ? GF[a0 * n + 16 * q + e] : make_double2(0.0, 0.0);
      for (int a = a0; a >= 16 * qa; --a) {
        const double t = beta * acc[qa];
        double2 gn[kQrClusterMaxN / 16];
        if (a > 0) {
          beta = s_beta[a - 1];
#pragma unroll
          for (int q = 0; q <= qa; ++q)
            gn[q] = 16 * q + e < a - 1 ? GF[(a - 1) * n + 16 * q + e] : make_double2(0.0, 0.0);
        }
        const double tx = __shfl_sync(kFull, t, a & 15), ty = __shfl_sync(kFull, t, 16 + (a & 15));
        if (e == (a & 15)) put(a, t);
        const double t1 = comp == 0 ? tx : ty, t2 = comp == 0 ? ty : tx;
#pragma unroll
        for (int q = 0; q <= qa; ++q) {
          if (16 * q < a && 16 * q + e < a) {
            acc[q] = fma(-g[q].x, t1, acc[q]);
            acc[q] = fma(comp == 0 ? g[q].y : -g[q].y, t2, acc[q]);
          }
          if (a > 0) g[q] = gn[q];
        }
      }
    }
  };
  if (panel) {
    for (int c = me + C * wid; c < n; c += C * kNW) {
      double acc[kQrClusterMaxN / 16];
#pragma unroll
      for (int q = 0; q < kQrClusterMaxN / 16; ++q) acc[q] = lane < 16 && 16 * q + lane == c ? 1.0 : 0.0;
      double* T = reinterpret_cast<double*>(pn.T);
      solve(c, acc, [&](int a, double v) { T[2 * (a * n + c) + (lane >> 4)] = v; });
      for (int a = c + 1 + lane; a < n; a += 32) pn.T[a * n + c] = make_double2(0.0, 0.0);
    }
    cluster.sync();  // keep shared memory alive until every remote read has finished
    return;
  }
  // M = T V_top^H column by column: T^{-1} M[:, c] = conj(V_top[c, :])^T
  // (M[a][c] = 0 for a > c). Column c is solved by CTA c mod C, one warp.
  for (int c = me + C * wid; c < n; c += C * kNW) {
    double acc[kQrClusterMaxN / 16];
#pragma unroll
    for (int q = 0; q < kQrClusterMaxN / 16; ++q) acc[q] = 0.0;
    if (c < m) {
      const int oc = c / rp;
      const double2* Ar = cluster.map_shared_rank(A, oc);
      const int lr = c - oc * rp;
#pragma unroll
      for (int q = 0; q < kQrClusterMaxN / 16; ++q) {
        const int i = 16 * q + (lane & 15);
        if (i <= c && i < n && !s_skip[i]) {
          const double2 v = Ar[(size_t)i * rp + lr];
          acc[q] = lane < 16 ? v.x : -v.y;
        }
      }
    }
    // the column waits in SU (free since the Gram sums) until every CTA may receive it
    double2* buf = SU + ((size_t)(c / (C * kNW)) * kNW + wid) * n;
    solve(c, acc, [&](int a, double v) { reinterpret_cast<double*>(buf)[2 * a + (lane >> 4)] = v; });
  }
  if (!gt && !pn.m_apart) cluster.sync();  // M takes GF's place: every solve is done
  for (int c = me + C * wid; c < n; c += C * kNW) {
    __syncwarp();
    const double2* buf = SU + ((size_t)(c / (C * kNW)) * kNW + wid) * n;
    const int copies = gt ? 1 : C;
    for (int k = lane; k < (c + 1) * copies; k += 32) {
      const int a = k % (c + 1), to = k / (c + 1);
      double2* dst = gt ? M : cluster.map_shared_rank(M, to);
      dst[a * n + c] = buf[a];
    }
  }
  grid_release();
  cluster.sync();  // M complete in every CTA; nobody reads another's rows any more
  // Q rows: Q[r][c] = delta_rc - sum_{a <= min(r,c)} v_a[r] M[a][c], column c scaled by phase_c
  // Entries (c, row) are laid along the lanes column after column, so that few
  // rows per CTA still fill the warps; a task is 32 entries and costs as many
  // steps as its last column needs, so tasks go to the warps forth and back.
  const int ntask = (n * nr + 31) / 32;
  for (int rnd = 0; rnd * kNW < ntask; ++rnd) {
    const int task = rnd * kNW + ((rnd & 1) ? kNW - 1 - wid : wid), e = task * 32 + lane;
    if (task >= ntask || e >= n * nr) continue;
    const int c = e / nr, i = e % nr;
    const int r = r0 + i;
    double2 q = make_double2(r == c ? 1.0 : 0.0, 0.0);
    const int amax = min(c, r);
    for (int a = 0; a <= amax; ++a) q = cfms(A[(size_t)a * rp + i], M[a * n + c], q);
    const double2 p = s_phase[c];
    const double2 qp = make_double2(q.x * p.x - q.y * p.y, q.x * p.y + q.y * p.x);
    const int64_t at = c * st[leg] + (int64_t)(r / dd[lb]) * st[la] + (int64_t)(r % dd[lb]) * st[lb];
    U[at] = qp;
    if (U_lo) U_lo[at] = make_float2((float)qp.x, (float)qp.y);
  }
}

constexpr size_t kQrSmemCap = 200 * 1024;

// nn: n x n buffers in shared memory (2: GF and M, 1: shared, 0: global memory)
size_t qr_cluster_smem(int m, int n, int C, int nn) {
  const int rp = (m + C - 1) / C;
  return sizeof(double2) * ((size_t)n * rp + 34 * (size_t)n + (size_t)nn * n * n);
}

// Cluster size for an m x n QR (0: does not fit); *nn as above.
int qr_cluster_size(int m, int n, int* nn) {
  *nn = 0;
  if (n > kQrClusterMaxN) return 0;
  int C = (m + 7) / 8;  // about 8 rows per CTA: the factorisation is FP64-issue bound
  C = C < 1 ? 1 : (C > 16 ? 16 : C);
  if (n > 4 * kNW * C) return 0;  // solved columns wait in four rounds of warps
  for (*nn = 2; *nn >= 0; --*nn)
    if (qr_cluster_smem(m, n, C, *nn) <= kQrSmemCap) return C;
  return 0;
}

template <int G>
static bool launch_cluster(double2* U, int d0, int d1, int d2, int leg, double tol, double2* R, int* flag,
                           float2* U_lo, float2* R_lo, const QrPanel& pn, int m, int n, int C, cudaStream_t s) {
  static bool attr_done = false;
  if (!attr_done) {
    cudaFuncSetAttribute(k_qr_cluster<G>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaFuncSetAttribute(k_qr_cluster<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQrSmemCap);
    attr_done = true;
  }
  const size_t smem = qr_cluster_smem(m, n, C, pn.A ? 1 : pn.gtail ? 0 : pn.m_apart ? 2 : 1);
  return launch_dep(k_qr_cluster<G>, dim3(C), dim3(kThreads), smem, s, C, U, d0, d1, d2, leg, tol, R, flag, U_lo, R_lo,
                    pn) == cudaSuccess;
}

bool launch_qr_cluster(double2* U, int d0, int d1, int d2, int leg, double tol, double2* R, int* flag,
                       float2* U_lo, float2* R_lo, double2* scratch, int64_t scratch_elems, cudaStream_t s) {
  const int dd[3] = {d0, d1, d2};
  const int n = dd[leg];
  const int m = (int)((int64_t)d0 * d1 * d2 / n);
  int nn = 0;
  const int C = qr_cluster_size(m, n, &nn);
  if (C == 0) return false;
  QrPanel pn = {};
  pn.m_apart = nn == 2;
  if (nn == 0) {
    if (!scratch || scratch_elems < (C + 2) * (int64_t)n * n) return false;
    pn.gtail = scratch;
  }
  return launch_cluster<8>(U, d0, d1, d2, leg, tol, R, flag, U_lo, R_lo, pn, m, n, C, s);
}

int qr_panel_cluster(int m_act, int nb) {
  int C = (m_act + 7) / 8;
  C = C < 1 ? 1 : (C > 16 ? 16 : C);
  return qr_cluster_smem(m_act, nb, C, 1) > kQrSmemCap ? 0 : C;
}

bool launch_qr_panel(const QrPanel& pn, cudaStream_t s) {
  const int m_act = pn.m - pn.c0;
  const int C = qr_panel_cluster(m_act, pn.nb);
  if (C == 0 || pn.nb > kQrPanelMaxNb) return false;
  return launch_cluster<32>(nullptr, 1, 1, 1, 0, 0.0, nullptr, nullptr, nullptr, nullptr, pn, m_act, pn.nb, C, s);
}

}  // namespace ttn
