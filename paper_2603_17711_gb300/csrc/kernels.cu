// Device kernels of the TTN-HEOM library, FP64 path (sm_103a).
//
// On GB300 the FP64 pipe issues about 2 FMA per SM per clock, so every kernel
// here is bound by FP64 issue, not by memory: the data (node tensors of at most
// a few hundred KB, environments of r x r) stays in L2 and L1.
#include <algorithm>
#include <cooperative_groups.h>
#include <mutex>
#include <type_traits>

#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace ttn {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {  // a*b + c
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(-a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ double2 cfma_conj(double2 a, double2 b, double2 c) {  // conj(a)*b + c
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(-a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 cscale(double s, double2 a) { return make_double2(s * a.x, s * a.y); }

// ---------------------------------------------------------------------------
// Complex arithmetic in the contraction type (double2 or float2).
// ---------------------------------------------------------------------------
template <typename R> struct Cx;
template <> struct Cx<double> {
  using T = double2;
  __device__ static T zero() { return make_double2(0.0, 0.0); }
  __device__ static T fma(T a, T b, T c) { return cfma(a, b, c); }
  __device__ static T fmaj(T a, T b, T c) { return cfma_conj(a, b, c); }
  __device__ static T add(T a, T b) { return cadd(a, b); }
  // component comp (0 real, 1 imaginary) of fma(), the same operations in the same order
  __device__ static double fma_part(T a, T b, int comp, double c) {
    return ::fma(a.y, comp ? b.x : -b.y, ::fma(a.x, comp ? b.y : b.x, c));
  }
  __device__ static double2 wide(T a) { return a; }
  __device__ static T narrow(double2 a) { return a; }
};
template <> struct Cx<float> {
  using T = float2;
  __device__ static T zero() { return make_float2(0.f, 0.f); }
  __device__ static T fma(T a, T b, T c) {
    c.x = fmaf(a.x, b.x, c.x);
    c.x = fmaf(-a.y, b.y, c.x);
    c.y = fmaf(a.x, b.y, c.y);
    c.y = fmaf(a.y, b.x, c.y);
    return c;
  }
  __device__ static T fmaj(T a, T b, T c) {
    c.x = fmaf(a.x, b.x, c.x);
    c.x = fmaf(a.y, b.y, c.x);
    c.y = fmaf(a.x, b.y, c.y);
    c.y = fmaf(-a.y, b.x, c.y);
    return c;
  }
  __device__ static T add(T a, T b) { return make_float2(a.x + b.x, a.y + b.y); }
  __device__ static double2 wide(T a) { return make_double2(a.x, a.y); }
  __device__ static T narrow(double2 a) { return make_float2((float)a.x, (float)a.y); }
};

// ---------------------------------------------------------------------------
// Sum of mode products: out_o[idx] = sum_t M_t x_{leg_t} src_t.
// An output tile is 32 consecutive elements (one per lane). Its work is cut
// into units -- an identity term, or kApChunk consecutive positions x of one
// mode product -- dealt round-robin to the NW*k warps of the k CTAs (one
// thread-block cluster) that share the tile. Each warp sums its units in
// order, the CTA sums its warps in order, and CTA 0 of the cluster sums the
// CTAs in order (through distributed shared memory), so results are bitwise
// reproducible for a given tile shape (NW, k). GB300 issues one FP64
// instruction per warp every ~64 cycles, so short dependency chains (4
// positions per unit, loads issued before the FMAs) and many warps per tile
// make a small contraction fast; when many lists run at once (batched
// instances) fewer warps per tile waste less on idle warps and reductions.
// NW (warps per CTA: 2, 4 or 8) and k are chosen per list (ApList::w, k).
//
// A small launch is a latency chain, so the chain is kept short: job tables in
// the constant bank (three dependent L2 reads saved), the next unit of a warp by
// addition instead of a modulo per term, real and imaginary sums on two
// sub-partitions, the stage update's state and accumulator loaded before the
// sum, its step coefficient divided on the host. Same sums in the same order.
// Small FP64 launches (CS) give an output two lanes, one component each: half a
// tile per CTA, twice the CTAs, and half the FP64 instructions on a warp's
// chain (8 a unit instead of 16, 64 cycles each), again the same sums.
// Measured in the rank-10 spin-boson train: 8-CTA bond lists 5.0 -> 3.9 us,
// 1-CTA lists 5.0 -> 3.6 us; rank-20 chain, 160-CTA lists 6.1 -> 4.6 us, 500-CTA
// (FP64-issue bound) 20 -> 20 us.
// ---------------------------------------------------------------------------

// Job tables as seen by the kernels: in global memory (any list), or as kernel
// parameters (lists of at most NT terms and NO outputs, all addresses resolved).
template <typename V>
struct ApTermV {
  const V* M;  // null: identity
  const V* X;
  int leg;
  int diag;  // ApTerm::pad: packed diagonals of a sparse operator, 0: dense
};
template <typename V>
struct ApOutV {
  int d0, d1, d2, d3, tb, te, tile0;
  V* dst;
};
template <typename V>
struct ApMem {
  DevTables T;
  __device__ __forceinline__ int find(const ApList& L, int tile) const {
    return list_output(T.outs, L.out_begin, L.out_end, L.tpo, tile);
  }
  __device__ __forceinline__ ApOutV<V> out(int o) const {
    const ApOut u = T.outs[o];
    return ApOutV<V>{u.d0, u.d1, u.d2, u.d3, u.term_begin, u.term_end, u.tile0, u.dst >= 0 ? (V*)T.bufs[u.dst] : nullptr};
  }
  __device__ __forceinline__ ApTermV<V> term(int t) const {
    const ApTerm a = T.terms[t];
    return ApTermV<V>{a.mat < 0 ? nullptr : (const V*)T.mats[a.mat], (const V*)T.bufs[a.src], a.leg, a.pad};
  }
};
template <typename V, int NT, int NO>
struct ApPar {
  ApOutV<V> outs[NO];
  ApTermV<V> terms[NT];
  __device__ __forceinline__ int find(const ApList& L, int tile) const {
    return list_output(outs, 0, L.out_end - L.out_begin, L.tpo, tile);
  }
  __device__ __forceinline__ const ApOutV<V>& out(int o) const { return outs[o]; }
  __device__ __forceinline__ const ApTermV<V>& term(int t) const { return terms[t]; }
};

// Leg geometry of one output element (kept in registers: selected by switch,
// never indexed dynamically).
struct Geo {
  int d0, d1, d2, d3;
  int i0, i1, i2, i3;
  int64_t s0, s1, s2;  // s3 = 1
};
__device__ __forceinline__ void geo_leg(const Geo& g, int leg, int& dl, int& il, int64_t& stride) {
  switch (leg) {
    case 0: dl = g.d0; il = g.i0; stride = g.s0; break;
    case 1: dl = g.d1; il = g.i1; stride = g.s1; break;
    case 2: dl = g.d2; il = g.i2; stride = g.s2; break;
    default: dl = g.d3; il = g.i3; stride = 1; break;
  }
}

// What a lane sums: an output's complex value, or (CS) component comp of it.
template <typename R, bool CS>
struct LaneSum {
  using C = Cx<R>;
  using V = typename C::T;
  using A = std::conditional_t<CS, R, V>;
  __device__ static A zero() {
    if constexpr (CS) return R(0);
    else return C::zero();
  }
  __device__ static A add(A a, A b) {
    if constexpr (CS) return a + b;
    else return C::add(a, b);
  }
  __device__ static A fma(V a, V b, int comp, A c) {
    if constexpr (CS) return C::fma_part(a, b, comp, c);
    else return C::fma(a, b, c);
  }
  __device__ static A load(const V* p, int64_t i, int comp) {
    if constexpr (CS) return reinterpret_cast<const R*>(p)[2 * i + comp];
    else return p[i];
  }
};

// contribution of positions [x0, x0 + kApChunk) of one term (the whole term if
// identity or sparse)
template <typename R, bool CS>
__device__ __forceinline__ typename LaneSum<R, CS>::A unit_dot(const ApTermV<typename Cx<R>::T>& term, int64_t idx,
                                                               const Geo& g, int x0, int comp) {
  using C = Cx<R>;
  using V = typename C::T;
  using S = LaneSum<R, CS>;
  if (!term.M) return S::load(term.X, idx, comp);
  int dl, il;
  int64_t stride;
  geo_leg(g, term.leg, dl, il, stride);
  const V* __restrict__ row = term.M + (int64_t)il * dl;
  const V* __restrict__ col = term.X + (idx - (int64_t)il * stride);
  V mv[kApChunk], sv[kApChunk];
  if (sizeof(R) == 8 && term.diag) {  // at most three diagonals: x = il + offset
    const int nd = term.diag >> 24;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int x = il + (int)(int8_t)(term.diag >> (8 * k));
      const bool in = k < nd && x >= 0 && x < dl;
      mv[k] = in ? row[x] : C::zero();
      sv[k] = in ? col[(int64_t)x * stride] : C::zero();
    }
    typename S::A acc = S::zero();
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (k < nd) acc = S::fma(mv[k], sv[k], comp, acc);
    return acc;
  }
#pragma unroll
  for (int k = 0; k < kApChunk; ++k) {
    const int x = x0 + k;
    if (x < dl) {
      mv[k] = row[x];
      sv[k] = col[(int64_t)x * stride];
    }
  }
  typename S::A acc = S::zero();
#pragma unroll
  for (int k = 0; k < kApChunk; ++k)
    if (x0 + k < dl) acc = S::fma(mv[k], sv[k], comp, acc);
  return acc;
}

// Sum of n per-warp (or per-CTA) partials of one tile, in order: warp 0 adds the
// real parts, warp 1 the imaginary parts. An FP64 addition holds an SM
// sub-partition for 64 cycles whatever the lane count, so the two components
// on two sub-partitions take half the time of one warp adding complex values,
// with the same sums; the epilogue follows the same split. Where the lanes hold
// components already (CS), warp 0 does both.
template <typename R, bool CS = false>
__device__ __forceinline__ R comp_sum(const void* part, int n) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  R acc = R(0);
  if (wid < (CS ? 1 : 2)) {
    const R* p = reinterpret_cast<const R*>(part) + (CS ? lane : 2 * lane + wid);
    acc = p[0];
    for (int w = 1; w < n; ++w) acc += p[(CS ? 32 : 64) * w];
  }
  return acc;
}

// Sum of one output tile over the units of CTA `rank` of the k sharing it;
// the CTA's total (fixed order over warps) is returned in warps 0 (real part)
// and 1 (imaginary part), or in warp 0 (CS).
template <typename R, int NW, bool CS, typename TAB>
__device__ __forceinline__ R tile_sum(const TAB& tab, const ApOutV<typename Cx<R>::T>& out, const Geo& g, int64_t idx,
                                      int comp, bool in, int rank, int K, typename LaneSum<R, CS>::A (*part)[32]) {
  using V = typename Cx<R>::T;
  using S = LaneSum<R, CS>;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  typename S::A acc = S::zero();
  const int W = K * NW;
  int off = rank * NW + wid;  // this warp's first unit, relative to the current term's
  for (int t = out.tb; t < out.te; ++t) {
    const ApTermV<V> term = tab.term(t);
    int nch = 1;
    if (term.M && !(sizeof(R) == 8 && term.diag)) {
      const int dl = term.leg == 0 ? g.d0 : term.leg == 1 ? g.d1 : term.leg == 2 ? g.d2 : g.d3;
      nch = (dl + kApChunk - 1) / kApChunk;
    }
    int c = off;
    for (; c < nch; c += W)
      if (in) acc = S::add(acc, unit_dot<R, CS>(term, idx, g, c * kApChunk, comp));
    off = c - nch;
  }
  part[wid][lane] = acc;
  __syncthreads();
  return comp_sum<R, CS>(part, NW);
}

// Epilogue of one component of one output element (at = 2 idx + comp); y0, a0: the state and the stage
// accumulator, loaded ahead of the sum.
template <typename R>
__device__ __forceinline__ void tile_store(R* dst, const Epi& ep, int64_t at, R acc, double y0, double a0) {
  if (ep.mode == EPI_STORE) {
    dst[at] = acc;
    return;
  }
  const double k = acc;
  if (ep.mode == EPI_RK4) {
    const double yn = y0 + ep.c * (a0 + k);
    ((double*)ep.y)[at] = yn;
    if ((void*)ep.y_lo != (void*)ep.y) ((R*)ep.y_lo)[at] = (R)yn;
    return;
  }
  ((double*)ep.acc)[at] = ep.mode == EPI_RK1 ? k : a0 + 2.0 * k;
  ((R*)ep.ys)[at] = (R)(y0 + ep.c * k);
}

template <typename R, int NW, bool CS, typename TAB>
__global__ void __launch_bounds__(32 * NW, 32 / NW) k_apply(const __grid_constant__ TAB tab, ApList L, Epi ep) {
  using V = typename Cx<R>::T;
  using A = typename LaneSum<R, CS>::A;
  __shared__ A part[NW][32];
  __shared__ A slot[kMaxSplit][32];
  const int K = L.k;
  const int block = blockIdx.x / K, rank = blockIdx.x % K;  // rank == block rank in the cluster
  const int tile = CS ? block >> 1 : block;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const ApOutV<V> out = tab.out(tab.find(L, tile));
  Geo g;
  g.d0 = out.d0; g.d1 = out.d1; g.d2 = out.d2; g.d3 = out.d3;
  g.s2 = g.d3;
  g.s1 = (int64_t)g.d2 * g.d3;
  g.s0 = g.s1 * g.d1;
  const int64_t P = g.s0 * g.d0, idx = (int64_t)(tile - out.tile0) * kApTile +
                                    (CS ? (block & 1) * (kApTile / 2) + (lane >> 1) : lane);
  const bool in = idx < P;
  const int comp = CS ? lane & 1 : wid & 1;  // of the lane's sum, or of the warp's share of the epilogue
  const bool last = wid < (CS ? 1 : 2);      // warps that finish the tile
  g.i0 = g.i1 = g.i2 = g.i3 = 0;
  const int64_t at = 2 * idx + comp;
  grid_wait();
  double y0 = 0.0, a0 = 0.0;
  if (in) {
    if (ep.mode != EPI_STORE && last && rank == 0) {
      y0 = ((const double*)ep.y)[at];
      if (ep.mode != EPI_RK1) a0 = ((const double*)ep.acc)[at];
    }
    if (P <= 0x7fffffff) {  // every tensor of these trees: 32-bit index arithmetic
      const unsigned x = (unsigned)idx, s1 = (unsigned)g.s1, s2 = (unsigned)g.s2;
      const unsigned q2 = x / s2, q1 = x / s1;
      g.i0 = (int)(x / (unsigned)g.s0);
      g.i1 = (int)(q1 % (unsigned)g.d1);
      g.i2 = (int)(q2 % (unsigned)g.d2);
      g.i3 = (int)(x - q2 * s2);
    } else {
      g.i0 = (int)(idx / g.s0);
      g.i1 = (int)((idx / g.s1) % g.d1);
      g.i2 = (int)((idx / g.s2) % g.d2);
      g.i3 = (int)(idx % g.d3);
    }
  }
  R acc = tile_sum<R, NW, CS>(tab, out, g, idx, comp, in, rank, K, part);
  grid_release();
  if (K > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    if (last)
      reinterpret_cast<R*>(cluster.map_shared_rank(&slot[0][0], 0))[CS ? rank * 32 + lane
                                                                       : rank * 64 + 2 * lane + wid] = acc;
    cluster.sync();
    if (rank > 0) return;
    acc = comp_sum<R, CS>(slot, K);
  }
  if (!last || !in) return;
  tile_store<R>(reinterpret_cast<R*>(out.dst), ep, at, acc, y0, a0);
}

// Launch n_tiles * k CTAs; k > 1 makes every k consecutive CTAs one cluster.
template <typename Kern, typename... Args>
static void launch_split(Kern kern, int n_tiles, int k, int warps, cudaStream_t s, const Args&... args) {
  launch_dep(kern, dim3((unsigned)(n_tiles * k)), dim3(32 * warps), 0, s, k > 1 ? k : 0, args...);
}

// CS: lists of at most half the SMs' number of CTAs, which still have an SM each
// when doubled. Rank-10 train / rank-19 tree / Table 1 / FMO step: 10.27 / 17.83 / 14.39 /
// 31.59 ms without, 9.97 / 17.62 / 14.23 / 31.41 up to 76 CTAs, 10.12 / 17.71 / 14.37 /
// 31.41 up to 152, 10.11 / 18.38 / 14.46 / 31.52 up to 304 (the pipes are shared).
constexpr int kCsMaxCtas = 76;
template <typename R, typename TAB>
static void launch_apply_w(const TAB& tab, const ApList& L, const Epi& e, cudaStream_t s) {
  if constexpr (sizeof(R) == 8) {
    if (L.w != 2 && L.w != 4 && L.n_tiles * L.k <= kCsMaxCtas) {
      launch_split(k_apply<R, 8, true, TAB>, 2 * L.n_tiles, L.k, 8, s, tab, L, e);
      return;
    }
  }
  switch (L.w) {
    case 2: launch_split(k_apply<R, 2, false, TAB>, L.n_tiles, L.k, 2, s, tab, L, e); break;
    case 4: launch_split(k_apply<R, 4, false, TAB>, L.n_tiles, L.k, 4, s, tab, L, e); break;
    default: launch_split(k_apply<R, 8, false, TAB>, L.n_tiles, L.k, 8, s, tab, L, e); break;
  }
}

template <typename R, int NT, int NO>
static bool apply_par(const HostTables& H, const ApList& L, const Epi& e, cudaStream_t s) {
  using V = typename Cx<R>::T;
  const int t0 = H.outs[L.out_begin].term_begin, t1 = H.outs[L.out_end - 1].term_end;
  if (L.out_end - L.out_begin > NO || t1 - t0 > NT) return false;
  ApPar<V, NT, NO> tab{};
  for (int o = L.out_begin; o < L.out_end; ++o) {
    const ApOut& u = H.outs[o];
    tab.outs[o - L.out_begin] = ApOutV<V>{u.d0, u.d1, u.d2, u.d3, u.term_begin - t0, u.term_end - t0, u.tile0,
                                          u.dst >= 0 ? (V*)H.bufs[u.dst] : nullptr};
  }
  for (int t = t0; t < t1; ++t) {
    const ApTerm& a = H.terms[t];
    tab.terms[t - t0] = ApTermV<V>{a.mat < 0 ? nullptr : (const V*)H.mats[a.mat], (const V*)H.bufs[a.src], a.leg, a.pad};
  }
  launch_apply_w<R>(tab, L, e, s);
  return true;
}

// Three parameter sizes (a launch's parameters are copied whole), then the tables in memory.
template <typename R>
static void launch_apply_r(const DevTables& T, const HostTables& H, const ApList& L, const Epi& e, cudaStream_t s) {
  if (apply_par<R, 12, 4>(H, L, e, s)) return;
  if (apply_par<R, 32, 32>(H, L, e, s)) return;
  if (apply_par<R, 120, 40>(H, L, e, s)) return;
  launch_apply_w<R>(ApMem<typename Cx<R>::T>{T}, L, e, s);
}

void launch_apply(int prec, const DevTables& T, const HostTables& H, const ApList& L, const Epi& e, cudaStream_t s) {
  if (L.n_tiles <= 0) return;
  if (prec == PREC_F32)
    launch_apply_r<float>(T, H, L, with_coef(e), s);
  else
    launch_apply_r<double>(T, H, L, with_coef(e), s);
}

// ---------------------------------------------------------------------------
// Environment projection E[x', x] = sum_r conj(U[.. x' ..]) W[.. x ..] over all
// legs except `leg`. A tile is 32 output entries (one per lane); the reduction
// range r is dealt round-robin to the 8*k warps of the k CTAs (one cluster)
// sharing the tile, four positions per batch with loads issued first, and the
// partial sums are added in a fixed order (warps, then CTAs via distributed
// shared memory).
// ---------------------------------------------------------------------------
constexpr int kPjWarps = kSplitWarps;

template <typename V>
struct PjOutV {
  int d0, d1, d2, leg, tile0;
  const V* u;
  const V* w;
  V* dst;
};
template <typename V>
struct PjMem {
  DevTables T;
  __device__ __forceinline__ PjOutV<V> out(const PjList& L, int tile) const {
    const PjOut p = T.pjs[list_output(T.pjs, L.out_begin, L.out_end, L.tpo, tile)];
    return PjOutV<V>{p.d0, p.d1, p.d2, p.leg, p.tile0, (const V*)T.bufs[p.u_buf], (const V*)T.bufs[p.w_buf], (V*)T.mats[p.dst_mat]};
  }
};
template <typename V, int NO>
struct PjPar {
  PjOutV<V> outs[NO];
  __device__ __forceinline__ PjOutV<V> out(const PjList& L, int tile) const {
    return outs[list_output(outs, 0, L.out_end - L.out_begin, L.tpo, tile)];
  }
};

template <typename R, typename TAB>
__global__ void __launch_bounds__(32 * kPjWarps, 4) k_project(const __grid_constant__ TAB tab, PjList L) {
  using C = Cx<R>;
  using V = typename C::T;
  __shared__ V part[kPjWarps][32];
  __shared__ V slot[kMaxSplit][32];
  const int K = L.k;
  const int tile = blockIdx.x / K, rank = blockIdx.x % K;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const PjOutV<V> pj = tab.out(L, tile);
  const int dd[3] = {pj.d0, pj.d1, pj.d2};
  const int64_t st[3] = {(int64_t)pj.d1 * pj.d2, pj.d2, 1};
  const int l = pj.leg;
  const int d = dd[l];
  const int e = (tile - pj.tile0) * kPjTile + lane;
  const int la = l == 0 ? 1 : 0, lb = l == 2 ? 1 : 2;  // the two other legs
  const int nrest = dd[la] * dd[lb];
  grid_wait();
  V acc = C::zero();
  if (e < d * d) {
    const int xp = e / d, x = e % d;
    const V* __restrict__ U = pj.u + (int64_t)xp * st[l];
    const V* __restrict__ Wt = pj.w + (int64_t)x * st[l];
    const int W = K * kPjWarps, me = rank * kPjWarps + wid;
    for (int r0 = me; r0 < nrest; r0 += 4 * W) {
      V uv[4], wv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = r0 + k * W;
        if (r < nrest) {
          const int64_t off = (int64_t)(r / dd[lb]) * st[la] + (int64_t)(r % dd[lb]) * st[lb];
          uv[k] = U[off];
          wv[k] = Wt[off];
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (r0 + k * W < nrest) acc = C::fmaj(uv[k], wv[k], acc);
    }
  }
  part[wid][lane] = acc;
  __syncthreads();
  R sum = comp_sum<R>(part, kPjWarps);
  grid_release();
  if (K > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    if (wid < 2) reinterpret_cast<R*>(cluster.map_shared_rank(&slot[0][0], 0))[rank * 64 + 2 * lane + wid] = sum;
    cluster.sync();
    if (rank > 0) return;
    sum = comp_sum<R>(slot, K);
  }
  if (wid > 1 || e >= d * d) return;
  reinterpret_cast<R*>(pj.dst)[2 * e + wid] = sum;
}

// Projection of wide bonds (d >= 32, reduction range >= 1024): 32 x 32 output
// tiles, reduction range in chunks of 32 staged through shared memory with
// coalesced loads (along the reduction index, or along the leg when the leg
// is the contiguous one), 2 x 2 outputs per thread. The range is split over
// KS CTAs of one cluster, whose partial tiles CTA 0 adds in rank order
// through distributed shared memory, so results are reproducible.
constexpr int kPtT = 32;  // output tile edge
constexpr int kPtR = 32;  // reduction chunk

template <typename R>
__global__ void __launch_bounds__(256) k_project_tiled(DevTables T, PjList L, int ntx, int KS) {
  using C = Cx<R>;
  using V = typename C::T;
  extern __shared__ __align__(16) unsigned char psm[];
  V(*Us)[kPtR + 1] = (V(*)[kPtR + 1])psm;
  V(*Ws)[kPtR + 1] = Us + kPtT;
  V* slot = (V*)(Ws + kPtT);  // CTA 0: [KS-1][kPtT * kPtT] partial tiles of the other ranks
  __shared__ int64_t base[kPtR];
  const int tid = threadIdx.x;
  const int rank = blockIdx.x % KS, item = blockIdx.x / KS;
  const int per_out = ntx * ntx;
  const int o = L.out_begin + item / per_out, tt = item % per_out;
  const PjOut pj = T.pjs[o];
  const int dd[3] = {pj.d0, pj.d1, pj.d2};
  const int64_t st[3] = {(int64_t)pj.d1 * pj.d2, pj.d2, 1};
  const int l = pj.leg, d = dd[l];
  const int la = l == 0 ? 1 : 0, lb = l == 2 ? 1 : 2;
  const int nrest = dd[la] * dd[lb];
  const int X0 = (tt / ntx) * kPtT, Y0 = (tt % ntx) * kPtT;  // rows x' (conjugated side), columns x
  const V* __restrict__ U = (const V*)T.bufs[pj.u_buf];
  const V* __restrict__ W = (const V*)T.bufs[pj.w_buf];
  const int nch = (nrest + kPtR - 1) / kPtR;
  const int c0 = (int)((int64_t)rank * nch / KS), c1 = (int)((int64_t)(rank + 1) * nch / KS);
  const bool leg_fast = l == 2;  // the leg index is the contiguous one
  const int ty = (tid >> 4) * 2, tx = (tid & 15) * 2;
  V acc[2][2] = {{C::zero(), C::zero()}, {C::zero(), C::zero()}};
  grid_wait();
  for (int c = c0; c < c1; ++c) {
    const int r0 = c * kPtR;
    if (tid < kPtR) {
      const int r = r0 + tid;
      base[tid] = r < nrest ? (int64_t)(r / dd[lb]) * st[la] + (int64_t)(r % dd[lb]) * st[lb] : 0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < (kPtT * kPtR) / 256; ++q) {
      const int e = tid + q * 256;
      const int row = leg_fast ? (e & 31) : (e >> 5), rr = leg_fast ? (e >> 5) : (e & 31);
      const bool rin = r0 + rr < nrest;
      const int xu = X0 + row, xw = Y0 + row;
      Us[row][rr] = (xu < d && rin) ? U[(int64_t)xu * st[l] + base[rr]] : C::zero();
      Ws[row][rr] = (xw < d && rin) ? W[(int64_t)xw * st[l] + base[rr]] : C::zero();
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < kPtR; ++rr) {
      const V u0 = Us[ty][rr], u1 = Us[ty + 1][rr], w0 = Ws[tx][rr], w1 = Ws[tx + 1][rr];
      acc[0][0] = C::fmaj(u0, w0, acc[0][0]);
      acc[0][1] = C::fmaj(u0, w1, acc[0][1]);
      acc[1][0] = C::fmaj(u1, w0, acc[1][0]);
      acc[1][1] = C::fmaj(u1, w1, acc[1][1]);
    }
    __syncthreads();
  }
  grid_release();
  if (KS > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    if (rank > 0) {
      V* dst = cluster.map_shared_rank(slot, 0) + (size_t)(rank - 1) * kPtT * kPtT;
      for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) dst[(ty + i) * kPtT + tx + j] = acc[i][j];
    }
    cluster.sync();
    if (rank > 0) return;
    for (int r = 1; r < KS; ++r)
      for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) acc[i][j] = C::add(acc[i][j], slot[(size_t)(r - 1) * kPtT * kPtT + (ty + i) * kPtT + tx + j]);
  }
  V* E = (V*)T.mats[pj.dst_mat];
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const int xp = X0 + ty + i, x = Y0 + tx + j;
      if (xp < d && x < d) E[xp * d + x] = acc[i][j];
    }
}

bool launch_project_tiled(int prec, const DevTables& T, const PjList& L, int d, int64_t nrest, int sm_count,
                          cudaStream_t s) {
  const int n_outs = L.out_end - L.out_begin;
  // FP64 projections are bound by FP64 issue either way and measured faster
  // on the per-entry kernel (rank-64 env update 100 vs 117 ms/step)
  if (prec != PREC_F32 || n_outs <= 0 || d < 32 || nrest < 1024) return false;
  const int ntx = (d + kPtT - 1) / kPtT;
  const int items = n_outs * ntx * ntx;
  const int nch = (int)((nrest + kPtR - 1) / kPtR);
  const int kmax = prec == PREC_F32 ? 8 : 4;
  int KS = 1;
  while (KS < kmax && KS < nch && items * KS < 2 * sm_count) ++KS;
  const size_t vb = prec == PREC_F32 ? sizeof(float2) : sizeof(double2);
  const size_t smem = vb * (2 * kPtT * (kPtR + 1) + (size_t)(KS - 1) * kPtT * kPtT);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_project_tiled<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    cudaFuncSetAttribute(k_project_tiled<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    attr = true;
  }
  const dim3 grid((unsigned)(items * KS));
  if (prec == PREC_F32)
    return launch_dep(k_project_tiled<float>, grid, dim3(256), smem, s, KS, T, L, ntx, KS) == cudaSuccess;
  return launch_dep(k_project_tiled<double>, grid, dim3(256), smem, s, KS, T, L, ntx, KS) == cudaSuccess;
}

template <typename R, int NO>
static bool project_par(const HostTables& H, const PjList& L, cudaStream_t s) {
  using V = typename Cx<R>::T;
  if (L.out_end - L.out_begin > NO) return false;
  PjPar<V, NO> tab{};
  for (int o = L.out_begin; o < L.out_end; ++o) {
    const PjOut& p = H.pjs[o];
    tab.outs[o - L.out_begin] = PjOutV<V>{p.d0, p.d1, p.d2, p.leg, p.tile0, (const V*)H.bufs[p.u_buf],
                                          (const V*)H.bufs[p.w_buf], (V*)H.mats[p.dst_mat]};
  }
  launch_split(k_project<R, PjPar<V, NO>>, L.n_tiles, L.k, kPjWarps, s, tab, L);
  return true;
}
template <typename R>
static void launch_project_r(const DevTables& T, const HostTables& H, const PjList& L, cudaStream_t s) {
  if (project_par<R, 8>(H, L, s) || project_par<R, 48>(H, L, s)) return;
  launch_split(k_project<R, PjMem<typename Cx<R>::T>>, L.n_tiles, L.k, kPjWarps, s, PjMem<typename Cx<R>::T>{T}, L);
}

void launch_project(int prec, const DevTables& T, const HostTables& H, const PjList& L, cudaStream_t s) {
  if (L.n_tiles <= 0) return;
  if (prec == PREC_F32)
    launch_project_r<float>(T, H, L, s);
  else
    launch_project_r<double>(T, H, L, s);
}

// Clusters of more than 8 CTAs are non-portable: allowed once per process for
// every contraction and projection kernel, before any launch (and outside any
// graph capture).
template <typename K>
static void allow_wide(K kern) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
template <typename R, typename TAB>
static void allow_wide_apply() {
  allow_wide(k_apply<R, 8, false, TAB>);
  allow_wide(k_apply<R, 4, false, TAB>);
  allow_wide(k_apply<R, 2, false, TAB>);
  if constexpr (sizeof(R) == 8) allow_wide(k_apply<R, 8, true, TAB>);
}
template <typename R>
static void allow_wide_r() {
  using V = typename Cx<R>::T;
  allow_wide_apply<R, ApPar<V, 12, 4>>();
  allow_wide_apply<R, ApPar<V, 32, 32>>();
  allow_wide_apply<R, ApPar<V, 120, 40>>();
  allow_wide_apply<R, ApMem<V>>();
  allow_wide(k_project<R, PjPar<V, 8>>);
  allow_wide(k_project<R, PjPar<V, 48>>);
  allow_wide(k_project<R, PjMem<V>>);
}
void allow_wide_splits() {
  static std::once_flag once;
  std::call_once(once, [] {
    allow_wide_r<double>();
    allow_wide_r<float>();
    cudaGetLastError();
  });
}


// ---------------------------------------------------------------------------
// Householder QR (one CTA). A (m x n, m = P / d_leg, n = d_leg) is gathered
// column-major into `work`; rows enumerate the two other legs in order.
// Convention (identical to the CPU oracle): for column j with remainder x of
// norm alpha, alpha <= tol*||A||_F means no reflector (R_jj = 0, Q column
// H_0..H_{j-1} e_j); otherwise v = x + phi*alpha*e_0 with phi = x_0/|x_0|
// (1 if x_0 = 0), H = I - beta v v^H, beta = 2 / (v^H v) = 1/(alpha(alpha+|x_0|)).
// Afterwards rows of R and columns of Q are rescaled so that diag(R) >= 0.
// ---------------------------------------------------------------------------
constexpr int kQrThreads = 512;
constexpr int kQrMaxN = 256;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double2 warp_sum2(double2 v) {
  v.x = warp_sum(v.x);
  v.y = warp_sum(v.y);
  return v;
}
// Block-wide sum with a fixed reduction order (deterministic).
__device__ double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < nw; ++w) s += red[w];
  return s;
}

__global__ void __launch_bounds__(kQrThreads) k_qr(double2* U, int d0, int d1, int d2, int leg,
                                                   double tol, double2* A, double2* Q, double2* R, int* flag,
                                                   float2* U_lo, float2* R_lo) {
  __shared__ double red[kQrThreads / 32];
  __shared__ double s_beta[kQrMaxN];
  __shared__ int s_skip[kQrMaxN];
  __shared__ double2 s_rdiag[kQrMaxN];
  __shared__ double2 s_phase[kQrMaxN];
  const int dd[3] = {d0, d1, d2};
  const int64_t st[3] = {(int64_t)d1 * d2, d2, 1};
  const int n = dd[leg];
  const int la = leg == 0 ? 1 : 0, lb = leg == 2 ? 1 : 2;
  const int64_t m = (int64_t)dd[la] * dd[lb];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  // gather A[r, c] (column-major), r = (a, b) over the two other legs
  double fro = 0.0;
  for (int64_t k = tid; k < m * n; k += nt) {
    const int64_t c = k / m, r = k % m;
    const int64_t a = r / dd[lb], b = r % dd[lb];
    const double2 v = U[c * st[leg] + a * st[la] + b * st[lb]];
    A[k] = v;
    fro += v.x * v.x + v.y * v.y;
  }
  fro = sqrt(block_sum(fro, red));
  if (!isfinite(fro)) {  // non-finite or overflowing input: report, leave U untouched
    if (tid == 0) atomicOr(flag, 1);
    return;
  }
  const double thr = tol * fro;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    double2* x = A + (int64_t)j * m;
    double ss = 0.0;
    for (int64_t r = j + tid; r < m; r += nt) ss += x[r].x * x[r].x + x[r].y * x[r].y;
    const double alpha = sqrt(block_sum(ss, red));
    if (alpha <= thr) {
      for (int64_t r = j + tid; r < m; r += nt) x[r] = make_double2(0.0, 0.0);
      if (tid == 0) {
        s_skip[j] = 1;
        s_beta[j] = 0.0;
        s_rdiag[j] = make_double2(0.0, 0.0);
        s_phase[j] = make_double2(1.0, 0.0);
      }
      __syncthreads();
      continue;
    }
    const double2 x0 = x[j];
    const double ax0 = hypot(x0.x, x0.y);
    const double2 phi = ax0 > 0.0 ? make_double2(x0.x / ax0, x0.y / ax0) : make_double2(1.0, 0.0);
    const double beta = 1.0 / (alpha * (alpha + ax0));
    __syncthreads();
    if (tid == 0) {
      x[j] = make_double2(x0.x + phi.x * alpha, x0.y + phi.y * alpha);  // v_0
      s_skip[j] = 0;
      s_beta[j] = beta;
      s_rdiag[j] = make_double2(-phi.x * alpha, -phi.y * alpha);
      s_phase[j] = make_double2(-phi.x, -phi.y);  // R_jj / |R_jj|
    }
    __syncthreads();
    // apply H_j to the remaining columns: one warp per column
    for (int k = j + 1 + wid; k < n; k += nw) {
      double2* a = A + (int64_t)k * m;
      double2 w = make_double2(0.0, 0.0);
      for (int64_t r = j + lane; r < m; r += 32) w = cfma_conj(x[r], a[r], w);
      w = warp_sum2(w);
      const double2 bw = cscale(beta, w);
      for (int64_t r = j + lane; r < m; r += 32) {
        const double2 t = cmul(x[r], bw);
        a[r] = make_double2(a[r].x - t.x, a[r].y - t.y);
      }
    }
    __syncthreads();
  }
  // R (row-major n x n) with diag(R) real >= 0: row j scaled by conj(phase_j)
  for (int k = tid; k < n * n; k += nt) {
    const int i = k / n, c = k % n;
    double2 v = make_double2(0.0, 0.0);
    if (c == i) {
      v = s_skip[i] ? make_double2(0.0, 0.0) : make_double2(hypot(s_rdiag[i].x, s_rdiag[i].y), 0.0);
    } else if (c > i) {
      const double2 a = A[(int64_t)c * m + i];
      const double2 p = s_phase[i];
      v = make_double2(a.x * p.x + a.y * p.y, a.y * p.x - a.x * p.y);  // conj(p) * a
    }
    R[k] = v;
    if (R_lo) R_lo[k] = make_float2((float)v.x, (float)v.y);
  }
  // Q = H_0 ... H_{n-1} [I; 0], column-major in Q
  for (int64_t k = tid; k < m * n; k += nt) {
    const int64_t c = k / m, r = k % m;
    Q[k] = make_double2(r == c ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  for (int j = n - 1; j >= 0; --j) {
    if (s_skip[j]) continue;
    const double2* v = A + (int64_t)j * m;
    const double beta = s_beta[j];
    for (int k = j + wid; k < n; k += nw) {
      double2* q = Q + (int64_t)k * m;
      double2 w = make_double2(0.0, 0.0);
      for (int64_t r = j + lane; r < m; r += 32) w = cfma_conj(v[r], q[r], w);
      w = warp_sum2(w);
      const double2 bw = cscale(beta, w);
      for (int64_t r = j + lane; r < m; r += 32) {
        const double2 t = cmul(v[r], bw);
        q[r] = make_double2(q[r].x - t.x, q[r].y - t.y);
      }
    }
    __syncthreads();
  }
  // scatter Q (columns scaled by phase) back into the node layout
  for (int64_t k = tid; k < m * n; k += nt) {
    const int64_t c = k / m, r = k % m;
    const int64_t a = r / dd[lb], b = r % dd[lb];
    const double2 q = cmul(Q[k], s_phase[c]);
    const int64_t at = c * st[leg] + a * st[la] + b * st[lb];
    U[at] = q;
    if (U_lo) U_lo[at] = make_float2((float)q.x, (float)q.y);
  }
}

void launch_qr(double2* U, int d0, int d1, int d2, int leg, double tol, double2* work, int64_t work_elems,
               double2* qbuf, double2* R, int* flag, float2* U_lo, float2* R_lo, cudaStream_t s,
               uint64_t grid_wait_ns) {
  if (launch_qr_cluster(U, d0, d1, d2, leg, tol, R, flag, U_lo, R_lo, work, work_elems, s)) return;
  if (launch_qr_blocked(U, d0, d1, d2, leg, tol, work, work_elems, qbuf, R, flag, U_lo, R_lo, s, grid_wait_ns))
    return;
  k_qr<<<counted(1), kQrThreads, 0, s>>>(U, d0, d1, d2, leg, tol, work, qbuf, R, flag, U_lo, R_lo);
}

__global__ void k_copy(double2* dst, float2* dst_lo, const double2* src, int64_t n) {
  grid_wait();
  grid_release();  // nothing but the copy itself is left
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = src[i];
    dst[i] = v;
    if (dst_lo) dst_lo[i] = make_float2((float)v.x, (float)v.y);
  }
}
void launch_copy(double2* dst, float2* dst_lo, const double2* src, int64_t n, cudaStream_t s) {
  if (n <= 0) return;
  int blocks = (int)std::min<int64_t>((n + 255) / 256, 1024);
  launch_dep(k_copy, dim3(blocks), dim3(256), 0, s, 0, dst, dst_lo, src, n);
}

// ---------------------------------------------------------------------------
// Reduced density matrix (rho_S = <0|Omega>): contraction of one node with
// the vectors of its two child legs (the n = 0 unit vector on open legs).
// ---------------------------------------------------------------------------
// All nodes of one tree level in one launch, one CTA per output. Lanes own the
// positions c of the last leg, warp w the rows b = w, w + 8, ...: a lane adds
// w1[b] U[a, b, c] over its rows, multiplies by w2[c] once, and only that is
// summed over lanes (fixed butterfly) and warps (in order), so an element costs
// four FP64 operations; a butterfly per row, as one launch per node had it, costs
// ten more per row. 21-node chain at rank 20: 21 launches of 4.2 us -> 7 of about 3 us.
struct RdmLevel {
  int n;
  RdmJob job[kRdmLevelMax];
};
__global__ void __launch_bounds__(256) k_rdm_level(const __grid_constant__ RdmLevel lv, const int* flag,
                                                   double2* flag_out) {
  __shared__ double part[8][2];
  int q = 0;
  while (q + 1 < lv.n && (int)blockIdx.x >= lv.job[q + 1].cta0) ++q;
  const RdmJob jb = lv.job[q];
  const int e = blockIdx.x - jb.cta0, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  grid_wait();
  // root: e = i*d1 + j, out[e] = sum_c U[i, j, c] w2[c]; else out[a] = sum_{b,c} U[a, b, c] w1[b] w2[c]
  const int nb = jb.w1 ? jb.d1 : 1, nc = jb.w2 ? jb.d2 : 1;
  const double2* blk = jb.U + (int64_t)e * (jb.root ? jb.d2 : (int64_t)jb.d1 * jb.d2);
  double2 acc = make_double2(0.0, 0.0);
  if (jb.w2) {
    for (int c = lane; c < nc; c += 32) {
      double2 t = make_double2(0.0, 0.0);
      if (jb.w1) {
        for (int b = warp; b < nb; b += 8) t = cfma(jb.w1[b], blk[(int64_t)b * jb.d2 + c], t);
      } else if (warp == 0) {
        t = blk[c];
      }
      acc = cfma(t, jb.w2[c], acc);
    }
  } else if (jb.w1) {  // the n = 0 position of the last leg: threads over the rows
    for (int b = threadIdx.x; b < nb; b += 256) acc = cfma(jb.w1[b], blk[(int64_t)b * jb.d2], acc);
  } else if (threadIdx.x == 0) {
    acc = blk[0];
  }
  for (int o = 16; o > 0; o >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
  }
  grid_release();
  if (lane == 0) {
    part[warp][0] = acc.x;
    part[warp][1] = acc.y;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double t = part[0][threadIdx.x];
    for (int w = 1; w < 8; ++w) t += part[w][threadIdx.x];
    reinterpret_cast<double*>(jb.out)[2 * e + threadIdx.x] = t;
  }
  // the error flag beside rho, so that one copy brings both to the host
  if (flag_out && blockIdx.x == 0 && threadIdx.x == 0) flag_out->x = (double)*flag;
}
void launch_rdm_level(RdmJob* jobs, int n, const int* flag, double2* flag_out, cudaStream_t s) {
  for (int i0 = 0; i0 < n; i0 += kRdmLevelMax) {
    RdmLevel lv{};
    int ctas = 0;
    for (int i = i0; i < n && lv.n < kRdmLevelMax; ++i) {
      RdmJob j = jobs[i];
      j.cta0 = ctas;
      ctas += j.n_out;
      lv.job[lv.n++] = j;
    }
    if (ctas > 0) launch_dep(k_rdm_level, dim3(ctas), dim3(256), 0, s, 0, lv, flag, flag_out);
  }
}

__global__ void k_drive(double2* const* mats, float2* const* mats32, const DriveMat* list, int n, DriveArgs g) {
  const DriveMat dm = list[blockIdx.x];
  const int dd = dm.d * dm.d;
  double2* cur = mats[dm.cur];
  float2* cur32 = mats32 ? mats32[dm.cur] : nullptr;
  const double2* st = mats[dm.stat];
  for (int e = threadIdx.x; e < dd; e += blockDim.x) {
    double2 v = st[e];
    for (int d = 0; d < kMaxDrives; ++d)
      if (dm.part[d] >= 0) {
        const double2 p = mats[dm.part[d]][e];
        v.x += g.g[d] * p.x;
        v.y += g.g[d] * p.y;
      }
    cur[e] = v;
    if (cur32) cur32[e] = make_float2((float)v.x, (float)v.y);
  }
}
void launch_drive(double2* const* mats_dev, float2* const* mats32, const DriveMat* list, int n,
                  const DriveArgs& g, cudaStream_t s) {
  if (n <= 0) return;
  k_drive<<<counted(n), 128, 0, s>>>(mats_dev, mats32, list, n, g);
}

__global__ void k_check_finite(const double2* x, int64_t n, int* flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = x[i];
    if (!isfinite(v.x) || !isfinite(v.y)) atomicOr(flag, 1);
  }
}
void launch_check_finite(const double2* x, int64_t n, int* flag, cudaStream_t s) {
  int blocks = (int)std::min<int64_t>((n + 255) / 256, 64);
  k_check_finite<<<counted(blocks), 256, 0, s>>>(x, n, flag);
}

}  // namespace ttn
