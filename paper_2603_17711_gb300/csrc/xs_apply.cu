// FP64 mode products on the tensor cores by an exact split into 8-bit digits.
//
// What bounds the FP64 contractions is the FP64 pipe: an SM sub-partition of
// GB300 retires one FP64 warp instruction per 64-76 cycles (0.42 FMA/clk),
// while a warp-level m16n8k16 f16 MMA (2048 multiply-adds, f32 accumulators)
// takes 8.2 cycles, both measured. Here a real FP64 operand becomes a 62-bit
// fixed-point integer, scaled by the largest exponent of its row (operator) or
// fiber (tensor), and the integer eight signed 8-bit digits, held exactly in
// f16. The product of two digits is below 2^14 and at most 8 * 128 of them
// enter one f32 accumulator (2d <= 128, digit pairs i + j = g <= 7), so every
// accumulator is an exact integer below 2^24: the only errors are the two
// truncations at 2^-62 and the dropped digit pairs i + j > 7, together below
// 2^-56.8 of (row scale x position scale) for each real product (2^-60 as a root
// mean square), where a chain of FP64 FMAs loses 2^-53 of the sum per addition. 36
// digit products replace 64-cycle FMAs by MMAs at 2048 * 592 / (36 * 8.2) = 4.1k
// multiply-adds per clock against 259 FMAs.
//
// One term Y += M x_l X (complex, d = d_l <= 64) is a real GEMM: output index
// i gives rows i (real part) and i + 8 (imaginary part) of an MMA tile, leg
// index x the two K columns (Re, Im), a position n of the other legs one N
// column. A lane loads the complex values of its own fragment slots from
// global memory (L1 / L2), so there is no shared-memory staging and no barrier
// in the term loop; the digits live in registers. A warp owns 8 output indices x
// 16 positions.
//
// Scales. X[x] of the tile is scaled to equal size over x and the scale moved to
// operator column x. The operator's fixed point of row i is then set by the
// largest |M[i][x]| S[x], S[x] = max_n |X[x][n]| over the tile's 16 positions, the
// tensor's of position n by its largest scaled element |X[x][n]| / S[x]. Where the
// grading is a row factor times a position factor these are the size of the output's own
// largest product. (With the columns of M scaled to equal size instead, a
// rank-20 chain's bond directions of weight 1e-9 differed by 2e-9 from the FMA chain
// after 30 steps.)
//
// Weak outputs. Otherwise row and position may reach their scales at different x,
// and an output that is small against both would keep few digits of its own: 1e-6
// for a row that sees only x = 0 at a position where X[0] is 1e-12 of S[0]. A run from
// the product state is full of them (padded directions), and they decide its weakly
// occupied directions: without what follows the nodes of chains of rank 20 to 32 were
// 6e-7 to 5e-6 from the FMA chain's after 20 to 60 steps and as far from those of
// another max_split (the chain's, in another order of sums: 1e-13 to 2e-11), rho up to
// 1e-12 (1e-17). So the products' magnitudes are summed too (powers of two, two MMAs
// per 8 x), and an output below kXsWeak of the scales is made from the operands by
// FMAs: nodes within 4e-14 to 1e-11 again. (Only where the row's scale also exceeds the position's
// largest output by 2^12, 2^16, 2^20: cheaper, but up to 2e-4 away.)
// What the split keeps is within 2 d 2^-44.8 sum |a b| of the exact sum whatever
// the operands. Largest and root mean square error over sum |a b| in units of 2^-53
// over the 64^3 outputs of a product, chain / split: flat operands 1.5, 0.22 / 0.38,
// 0.07; graded as the perf cases' states 6.6, 1.0 / 2.1, 0.29; tensor 10^(-0.6 |x - n|)
// 8.0, 1.0 / 9.3, 0.36; operator 1 + 1e-9 G on a graded tensor 7.1, 1.2 / 38, 0.42; rows
// that see what is small 1.8, 0.40 / 2.2, 0.31 (4e10, 4e8 without). One output's
// parts are not told apart: a part that is small beside the other is as accurate as
// the other.
// Cost: from a generic state, where 3e-4 of the outputs are below 2^-8 and none below
// 2^-12, the check alone (rank-64 chain 100.0 -> 101.4 ms; at 2^-8 102.3); in a run from the
// product state a third of the work at rank 64 (94 -> 156 ms, FMA chain 288), more
// than the split gives at rank 20; hence the line (xs_min_flops). Sharing the weak outputs
// of a CTA among its warps at the end, or leaving out the MMAs of warps that have no
// others, is no cheaper.
//
// A non-finite operand makes its whole row or column of outputs NaN; it sets no
// scale, so the outputs beside them are what they are without it.
//
// Measured without the check for weak outputs (graph replay, CUDA-core kernel /
// this one): 64^3 node, 14 terms
// 1799 / 244 us (7.7 TFLOP/s of FP64 results against the 1.1 of the FP64 pipe;
// the tensor pipe is half busy, the rest is operand latency and digit
// arithmetic); 20^3, 12 terms 22.9 / 12.9 us; 20x25x25, 12 terms 38.4 / 16.8 us.
// A product takes two group barriers (scales alternate between two sets; a
// tensor row's scale is known to the warp that loaded it): with the scale of an
// operator column, which all warps have to agree on, it took three and 249 us.
// Relative 2-norm error against 128-bit sums: 1.15e-16 / 2.35e-16 (64^3),
// 1.14e-16 / 1.70e-16 (20^3), 4.7e-17 / 1.4e-16 for a single product.
#include <algorithm>
#include <cstdint>

#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace ttn {

namespace {

constexpr int kXsWarps = 8;
constexpr int kXsThreads = 32 * kXsWarps;
constexpr int kXsNT = 2;              // n tiles (8 positions) per warp
constexpr int kXsCols = 8 * kXsNT;    // positions per warp
constexpr int kXsTermSplit = 2;       // more terms than this on a leg: the warp groups split the terms
constexpr int kXsMaxD = 64;           // 2 d <= 128: exactness of the f32 accumulators
// An output whose products sum to less than this of row scale x position scale is
// made by FP64 multiply-adds (weak outputs, above).
constexpr float kXsWeak = 1.0f / 4096;
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The same with 8 rows (the other 8 zero) and 8 K positions, for the magnitudes.
__device__ __forceinline__ void mma_f16_k8(float (&c)[4], uint32_t a, uint32_t b) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a), "r"(0), "r"(b));
}

__device__ __forceinline__ int exp_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ int exp_c(double2 v) { return max(exp_field(v.x), exp_field(v.y)); }
// an exponent that sets a scale: not of a zero, and not of a non-finite value
__device__ __forceinline__ bool scales(int e) { return (unsigned)(e - 1) < 0x7feu; }
__device__ __forceinline__ uint32_t pack2(int lo, int hi) { return (uint32_t)lo | ((uint32_t)hi << 16); }
__device__ __forceinline__ uint32_t both(int v) { return (uint32_t)(v & 0xffff) * 0x10001u; }
__device__ __forceinline__ uint32_t nonzero2(uint32_t e) { return __vminu2(e, 0x00010001u) * 0xffffu; }  // mask of 16-bit halves
// two exponents e <= 0 as f16x2 magnitudes 2^(e + 15), e at least -29; 0 where the mask is
__device__ __forceinline__ uint32_t magnitudes(uint32_t e, uint32_t mask) {
  return (__vmaxs2(__vadd2(e, both(30)), 0x00010001u) & mask) << 10;
}

// v as a fixed-point integer with 62 bits below 2^(top + 1 - 1023), plus the
// bias that turns its bytes into digits - 128 .. 127 offset by 128. Subnormal v
// is zero; so is everything where top is out of range (no scale): a shift by
// 64 or more (or a negative count, taken as unsigned) gives zero.
constexpr int kXsBias = 4096;  // above every exponent field and difference of two
__device__ __forceinline__ uint64_t fixed_biased(double v, int top) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t e = (hi >> 20) & 0x7ffu, mh = (hi & 0xfffffu) | 0x100000u;
  const uint32_t s = e == 0 ? 64u : (uint32_t)(top - (int)e);
  uint64_t f;
  asm("{\n .reg .b64 m;\n mov.b64 m, {%2, %1};\n shl.b64 m, m, 9;\n shr.u64 %0, m, %3;\n}" : "=l"(f) : "r"(mh), "r"(lo), "r"(s));
  const uint32_t sg = (uint32_t)((int)hi >> 31);
  uint32_t tl, th;
  asm("{\n .reg .b32 a, b, n;\n mov.b64 {a, b}, %2;\n xor.b32 a, a, %3;\n xor.b32 b, b, %3;\n and.b32 n, %3, 1;\n"
      " add.u32 n, n, 0x80808080;\n add.cc.u32 %0, a, n;\n addc.u32 %1, b, 0x80808080;\n}"
      : "=r"(tl), "=r"(th)
      : "l"(f), "r"(sg));
  return ((uint64_t)th << 32) | tl;
}
// Digit i (0 = most significant) of the pair (re, im) as f16x2.
template <int I>
__device__ __forceinline__ uint32_t digit_pair(uint64_t re, uint64_t im) {
  constexpr int b = 7 - I;
  const uint32_t wr = b >= 4 ? (uint32_t)(re >> 32) : (uint32_t)re;
  const uint32_t wi = b >= 4 ? (uint32_t)(im >> 32) : (uint32_t)im;
  constexpr uint32_t sel = (uint32_t)(b & 3) | ((uint32_t)(4 + (b & 3)) << 8);  // byte 0: re, byte 2: im
  uint32_t r = (__byte_perm(wr, wi, sel) & 0x00ff00ffu) | 0x64006400u;          // 1024 + byte
  const __half2 h = __hsub2(*reinterpret_cast<__half2*>(&r), __half2half2(__ushort_as_half(0x6480)));  // - 1152
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void digits8(double2 v, int top, uint32_t (&d)[8]) {
  const uint64_t re = fixed_biased(v.x, top), im = fixed_biased(v.y, top);
  d[0] = digit_pair<0>(re, im);
  d[1] = digit_pair<1>(re, im);
  d[2] = digit_pair<2>(re, im);
  d[3] = digit_pair<3>(re, im);
  d[4] = digit_pair<4>(re, im);
  d[5] = digit_pair<5>(re, im);
  d[6] = digit_pair<6>(re, im);
  d[7] = digit_pair<7>(re, im);
}

// acc += sum_g C_g 2^(8 (7 - g)) 2^ex. The sum is a 76-bit integer H 2^32 + l;
// its top 63 bits (all of it unless |H| is near its bound) go through one
// conversion and one FMA on the FP64 pipe, which the digit arithmetic leaves idle:
// building the double from integers took 60 instructions instead of 30.
__device__ __forceinline__ double join(const float (&c)[8], int ex, double acc) {
  int C[8];
#pragma unroll
  for (int g = 0; g < 8; ++g) C[g] = __float2int_rn(c[g]);
  const int64_t lo = (int64_t)C[4] * (1 << 24) + (int64_t)C[5] * (1 << 16) + (int64_t)C[6] * 256 + C[7];
  const int64_t H = (int64_t)C[0] * (1 << 24) + (int64_t)C[1] * (1 << 16) + (int64_t)C[2] * 256 + C[3] + (lo >> 32);
  const uint32_t l = (uint32_t)lo, hh = (uint32_t)(H >> 32), hl = (uint32_t)H;
  // shift the 96-bit value right by sh (0 .. 14) until 64 bits hold it with its sign
  const int top = 32 - __clz((int)hh ^ ((int)hh >> 31));
  const int sh = top > 0 ? top + 1 : (int)((hl ^ hh) >> 31);
  const uint32_t vl = __funnelshift_r(l, hl, sh), vh = __funnelshift_r(hl, hh, sh);
  const double d = (double)(int64_t)(((uint64_t)vh << 32) | vl);
  const int E = 1023 + ex + sh;
  if (E > 0 && E < 0x7ff) return fma(d, __hiloint2double(E << 20, 0), acc);
  return acc + scalbn(d, ex + sh);  // the scale itself is out of range
}

// One block product: 8 MT output indices (8 per warp of a group of MT warps) x 16
// positions, K <= 8 MT complex K positions. The tensor operand's digits are
// made once per group (warp m makes those of K positions 8m .. 8m+7) and
// shared through shared memory; the operator's are made by the warp that uses
// them.
struct XsGroup {
  int m, MT, bar;   // warp of the group, warps, named barrier
  int* sc;          // [2][96] scales, two sets used in turn (one is cleared while the other is in use):
                    //   [64] scale of every K position: its largest tensor exponent over the 16 positions
                    //   [16] largest scaled tensor exponent of every position, offset by kXsBias
                    //   [16] largest raw tensor exponent (0x7ff: not finite)
  uint4* bd;        // [MT][8][32] digits: x, y = K halves of positions 0..7, z, w = of positions 8..15
  uint2* be;        // [MT][32] magnitudes of the same values: x of positions 0..7, y of 8..15, f16x2 of the K halves
  uint8_t* weak;    // [128] this warp's list of weak outputs
};
struct XsSrc {
  const double2* a;  // operator row of this lane, or null
  const double2* b[kXsNT];  // tensor fiber of this lane's positions, or null
};
__device__ __forceinline__ void gsync(const XsGroup& G) {
  if (G.MT == 1)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(G.bar), "r"(32 * G.MT) : "memory");
}

// The outputs of the masks `weak` (bit 2 t + j of a lane: row lane >> 2, position
// 8 t + 2 (lane & 3) + j) by FP64 multiply-adds, into add. The warp lists them and takes
// up to 32 at a time, 32 / (their number) lanes each, so a few cost the latency of a
// short chain (four at a time, without a list: 4 % of a rank-20 chain's step more).
// Not inlined: its registers would be the product's spills (300 bytes against 208;
// rank-64 chain 102.8 ms against 101.4).
template <bool PROJ, typename KA, typename KB>
__device__ __noinline__ void weak_sums(uint8_t* list, const double2* sa, const double2* sb0, const double2* sb1, int K,
                                       KA ka, KB kb, uint32_t weak, double* add) {
  const int lane = threadIdx.x & 31, cnt = __popc(weak);
  int end = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, end, o);
    if (lane >= o) end += v;
  }
  const int total = __shfl_sync(kFull, end, 31), off = end - cnt;
  __syncwarp();  // the previous product's list is done with
#pragma unroll 1
  for (uint32_t w = weak, q = off; w != 0; w &= w - 1, ++q) list[q] = (uint8_t)(lane << 2 | (__ffs(w) - 1));
  __syncwarp();
#pragma unroll 1
  for (int base = 0; base < total;) {
    const int rem = total - base, lg = max(0, __clz(rem - 1) - 27), nb = 32 >> lg;
    const int slot = lane >> lg, L = 1 << lg;
    const bool on = slot < rem;
    const int code = on ? list[base + slot] : 0;
    const int from = code >> 2, t = code >> 1 & 1, pos = (2 * (from & 3) + (code & 1)) * 4;
    const double2* a = (const double2*)__shfl_sync(kFull, (unsigned long long)sa, from);
    const double2* b0 = (const double2*)__shfl_sync(kFull, (unsigned long long)sb0, pos);
    const double2* b1 = (const double2*)__shfl_sync(kFull, (unsigned long long)sb1, pos);
    const double2* b = t == 0 ? b0 : b1;
    double x = 0.0, y = 0.0;
#pragma unroll 2
    for (int k = lane & (L - 1); on && k < K; k += L) {
      const double2 u = a[ka(k)];
      double2 v = b[kb(k)];
      if (PROJ) v.y = -v.y;
      x = fma(u.x, v.x, fma(-u.y, v.y, x));
      y = fma(u.x, v.y, fma(u.y, v.x, y));
    }
#pragma unroll 1
    for (int o = L >> 1; o > 0; o >>= 1) {
      x += __shfl_xor_sync(kFull, x, o);
      y += __shfl_xor_sync(kFull, y, o);
    }
    int q = off - base;
#pragma unroll
    for (int e = 0; e < 2 * kXsNT; ++e) {  // back to the owners
      const int at = (q & (nb - 1)) << lg;
      const double gx = __shfl_sync(kFull, x, at), gy = __shfl_sync(kFull, y, at);
      if (weak >> e & 1u) {
        if (q >= 0 && q < nb) {
          add[2 * e] += gx;
          add[2 * e + 1] += gy;
        }
        ++q;
      }
    }
    base += nb;
  }
}

// acc += block product. PROJ: conj(B) instead of B.
template <bool PROJ, typename KA, typename KB>
__device__ __forceinline__ void xs_block(const XsGroup& G, int turn, const XsSrc& S, int K, KA ka, KB kb,
                                         double (&acc)[kXsNT][4]) {
  int* const scx = G.sc + 96 * (turn & 1);
  int* const scol = scx + 64;
  int* const scraw = scx + 80;
  const int lane = threadIdx.x & 31, kq = lane & 3;
  const double2 zero = make_double2(0.0, 0.0);
  const int KS = (K + 7) >> 3;
  // 1: raw tensor values of this warp's K positions, their scales (the largest
  // exponent over the positions) and the position scales; operator exponents
  double2 braw[kXsNT][2];
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int k = G.m * 8 + 4 * hf + kq;
#pragma unroll
    for (int t = 0; t < kXsNT; ++t) braw[t][hf] = (k < K && S.b[t]) ? S.b[t][kb(k)] : zero;
  }
  uint32_t ep[8];  // operator exponents of both K halves, so the operator is read once more only for its digits
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
    ep[ks] = 0;
    if (ks < KS) {
      const int k = ks * 8 + kq;
      const int e0 = (k < K && S.a) ? exp_c(S.a[ka(k)]) : 0;
      const int e1 = (k + 4 < K && S.a) ? exp_c(S.a[ka(k + 4)]) : 0;
      ep[ks] = (uint32_t)e0 | ((uint32_t)e1 << 16);
    }
  }
  int eb[kXsNT][2];
  uint32_t xr = 0;  // both K halves (packed 16-bit maxima)
#pragma unroll
  for (int t = 0; t < kXsNT; ++t) {
    eb[t][0] = exp_c(braw[t][0]);
    eb[t][1] = exp_c(braw[t][1]);
    xr = __vmaxu2(xr, pack2(scales(eb[t][0]) ? eb[t][0] : 0, scales(eb[t][1]) ? eb[t][1] : 0));
  }
  xr = __vmaxu2(xr, __shfl_xor_sync(kFull, xr, 4));
  xr = __vmaxu2(xr, __shfl_xor_sync(kFull, xr, 8));
  xr = __vmaxu2(xr, __shfl_xor_sync(kFull, xr, 16));
  const int xk[2] = {(int)(xr & 0xffff), (int)(xr >> 16)};
  if (lane < 8) scx[G.m * 8 + lane] = lane < 4 ? xk[0] : xk[1];
#pragma unroll
  for (int t = 0; t < kXsNT; ++t) {
    int c = 0, r = 0;
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      if (scales(eb[t][hf])) c = max(c, eb[t][hf] - xk[hf] + kXsBias);
      r = max(r, eb[t][hf]);
    }
    c = max(c, __shfl_xor_sync(kFull, c, 1));
    c = max(c, __shfl_xor_sync(kFull, c, 2));
    r = max(r, __shfl_xor_sync(kFull, r, 1));
    r = max(r, __shfl_xor_sync(kFull, r, 2));
    if (kq == 0) {
      atomicMax(&scol[8 * t + (lane >> 2)], c);
      atomicMax(&scraw[8 * t + (lane >> 2)], r);
    }
  }
  gsync(G);  // also: every warp is done with the previous product's scales and digits
  for (int e = 64 + G.m * 32 + lane; e < 96; e += 32 * G.MT) G.sc[96 * ((turn & 1) ^ 1) + e] = 0;
  // 2: row scale of the scaled operator; tensor digits of this warp's K positions
  uint32_t rowp = 0, rawp = 0;
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
    if (ks < KS) {
      const uint32_t x = pack2(scx[ks * 8 + kq], scx[ks * 8 + 4 + kq]);
      rawp = __vmaxu2(rawp, ep[ks]);
      const uint32_t fin = pack2(scales(ep[ks] & 0xffff) ? 0xffff : 0, scales(ep[ks] >> 16) ? 0xffff : 0);
      ep[ks] = (ep[ks] + x) & fin & nonzero2(x);  // exponents of the scaled operator
      rowp = __vmaxu2(rowp, ep[ks]);
    }
  int row = max((int)(rowp & 0xffff), (int)(rowp >> 16)), rraw = max((int)(rawp & 0xffff), (int)(rawp >> 16));
  if (row == 0) row = -kXsBias;
  row = max(row, __shfl_xor_sync(kFull, row, 1));
  row = max(row, __shfl_xor_sync(kFull, row, 2));
  rraw = max(rraw, __shfl_xor_sync(kFull, rraw, 1));
  rraw = max(rraw, __shfl_xor_sync(kFull, rraw, 2));
  {
    uint32_t d[kXsNT][2][8], q[kXsNT];
#pragma unroll
    for (int t = 0; t < kXsNT; ++t) {
      const int top = scol[8 * t + (lane >> 2)] - kXsBias;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) digits8(braw[t][hf], top + xk[hf], d[t][hf]);
      const uint32_t e = pack2(scales(eb[t][0]) ? eb[t][0] : 0, scales(eb[t][1]) ? eb[t][1] : 0);
      q[t] = magnitudes(__vsub2(__vsub2(e, xr), both(top)), nonzero2(e));
    }
    G.be[G.m * 32 + lane] = make_uint2(q[0], q[1]);
#pragma unroll
    for (int j = 0; j < 8; ++j) G.bd[(G.m * 8 + j) * 32 + lane] = make_uint4(d[0][0][j], d[0][1][j], d[1][0][j], d[1][1][j]);
  }
  gsync(G);
  // 3: this lane's weak outputs (bit 2 t + j: row lane >> 2, position 8 t + 2 kq + j)
  uint32_t weak = 0;
  {
    float s[kXsNT][4] = {};
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
      if (ks < KS) {
        const uint32_t a = magnitudes(__vsub2(ep[ks], both(row)), nonzero2(ep[ks]));
        const uint2 b = G.be[ks * 32 + lane];
        mma_f16_k8(s[0], a, b.x);
        mma_f16_k8(s[1], a, b.y);
      }
#pragma unroll
    for (int t = 0; t < kXsNT; ++t)
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if (s[t][j] > 0.f && s[t][j] < kXsWeak * 0x1p30f) weak |= 1u << (2 * t + j);
  }
  // 4: operator digits and MMAs
  float c[kXsNT][8][4];
#pragma unroll
  for (int t = 0; t < kXsNT; ++t)
#pragma unroll
    for (int g = 0; g < 8; ++g)
#pragma unroll
      for (int r = 0; r < 4; ++r) c[t][g][r] = 0.f;
  auto ld_a = [&](int k) { return (k < K && S.a) ? S.a[ka(k)] : zero; };
  double2 nv[2] = {ld_a(kq), ld_a(4 + kq)};
#pragma unroll 1
  for (int ks = 0; ks < KS; ++ks) {
    uint32_t a[8][4];
    const double2 v[2] = {nv[0], nv[1]};
    if (ks + 1 < KS) {
      nv[0] = ld_a(ks * 8 + 8 + kq);
      nv[1] = ld_a(ks * 8 + 12 + kq);
    }
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      uint32_t ad[8];
      digits8(v[hf], row - scx[ks * 8 + 4 * hf + kq], ad);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t sw = __byte_perm(ad[i], ad[i], 0x1032);  // (im, re)
        a[i][2 * hf] = PROJ ? ad[i] : ad[i] ^ 0x80000000u;      // (re, -+im)
        a[i][2 * hf + 1] = PROJ ? sw ^ 0x80000000u : sw;        // (im, +-re)
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint4 b = G.bd[(ks * 8 + j) * 32 + lane];
#pragma unroll
      for (int i = 0; i + j < 8; ++i) {
        mma_f16(c[0][i + j], a[i], b.x, b.y);
        mma_f16(c[1][i + j], a[i], b.z, b.w);
      }
    }
  }
  // lane holds rows (lane >> 2) re / im of columns 2 kq, 2 kq + 1
#pragma unroll
  for (int t = 0; t < kXsNT; ++t)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int n = 8 * t + 2 * kq + j, ec = scol[n];
      const int ex = row + ec - kXsBias;  // no scale: the sums are zero, and 2^0 keeps join() off its slow path
      const bool none = row < 0 || ec == 0;
      const bool bad = rraw == 0x7ff || scraw[n] == 0x7ff;
      if (bad) weak &= ~(1u << (2 * t + j));
      if (weak >> (2 * t + j) & 1u) continue;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float cc[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) cc[g] = c[t][g][2 * p + j];
        // both fixed points: value = integer * 2^(scale - 1084); the digit pairs of
        // group g weigh 2^(8 (14 - g)), 2^56 of it outside join()
        acc[t][2 * j + p] = bad ? __longlong_as_double(0x7ff8000000000000ll)
                                : join(cc, none ? 0 : ex - 2 * 1084 + 56, acc[t][2 * j + p]);
      }
    }
  if (__any_sync(kFull, weak != 0)) {
    double add[4 * kXsNT] = {};
    weak_sums<PROJ>(G.weak, S.a, S.b[0], S.b[1], K, ka, kb, weak, add);
#pragma unroll
    for (int t = 0; t < kXsNT; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[t][q] += add[4 * t + q];
  }
}

// Leg geometry: element = outer * (d * inner) + x * inner + in, position n = outer * inner + in.
struct XsLeg {
  int d, inner, rest;  // all below 2^30 (xs_applicable)
};
__device__ __forceinline__ XsLeg leg_of(const int (&dd)[4], int leg) {
  XsLeg g;
  g.d = dd[leg];
  g.inner = 1;
  for (int l = 3; l > leg; --l) g.inner *= dd[l];
  g.rest = dd[0] * dd[1] * dd[2] * dd[3] / g.d;
  return g;
}

}  // namespace

// Work of one launch, passed by value: operands and term lists sit in the
// constant bank, where a table in global memory costs three dependent L2 round
// trips (about 1.4 us of a launch) before the first operand can be loaded.
constexpr int kXsMaxTerms = 192, kXsMaxOuts = 96;
struct XsTerm {
  const double2* M;
  const double2* X;
};
struct XsWork {
  int dims[4];      // of every output
  int leg;          // -1: one output, all legs, planes; -2: every output's terms share one leg; else this leg
  // -1: CTAs [lt[l], lt[l+1]) of grid.x work on leg l, parts[l] term parts x
  // tiles; part j writes plane plane[l] + j
  int lt[5], parts[4], plane[4];
  double2* planes;
  double2* dst[kXsMaxOuts];
  short tb[kXsMaxOuts][5];  // terms of output o on leg l: [tb[o][l], tb[o][l+1])
  XsTerm term[kXsMaxTerms];
};

// CTA = (output, leg, tile, part). With MT = ceil(d / 8) row blocks the 8 warps
// form G = 8 / MT groups; the groups split the terms (split_terms, one 16-position
// tile per CTA, summed in group order through shared memory) or the positions
// (one 16-position tile per group, no sum).
__global__ void __launch_bounds__(kXsThreads, 2) k_xs_apply(const __grid_constant__ XsWork w) {
  __shared__ __align__(16) uint4 sm_bd[kXsWarps * 8 * 32];  // digits; the groups' sums at the end
  __shared__ uint2 sm_be[kXsWarps * 32];
  __shared__ uint8_t sm_weak[kXsWarps][128];
  __shared__ int sm_sc[kXsWarps][2 * 96];
  double2(*red)[kXsCols * 8] = reinterpret_cast<double2(*)[kXsCols * 8]>(sm_bd);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int o = blockIdx.y;
  int leg = w.leg, bx = blockIdx.x, part = 0, nparts = 1;
  const bool pl = leg == -1;
  if (leg == -2) {
    leg = 0;
    while (leg < 3 && w.tb[o][leg + 1] == w.tb[o][0]) ++leg;
  }
  if (pl) {
    leg = 0;
    while (leg < 3 && bx >= w.lt[leg + 1]) ++leg;
    nparts = w.parts[leg];
    const int nt = (w.lt[leg + 1] - w.lt[leg]) / nparts;
    bx -= w.lt[leg];
    part = bx / nt;
    bx = bx % nt;
  }
  const XsLeg g = leg_of(w.dims, leg);
  const int MT = (g.d + 7) >> 3, G = kXsWarps / MT;
  const int t_begin = w.tb[o][leg], nterm = w.tb[o][leg + 1] - t_begin;
  const bool earlier = !pl && t_begin > w.tb[o][0];  // an earlier leg's launch wrote the destination
  if (nterm == 0) return;  // uniform over the CTA
  const bool split_terms = pl || nterm > kXsTermSplit;
  const int tiles = (g.rest + kXsCols - 1) / kXsCols;
  if (!split_terms && bx * G >= tiles) return;
  const int mt = wid % MT, grp = wid / MT;
  const int tile = split_terms ? bx : bx * G + grp;
  const bool on = grp < G && tile < tiles;
  double acc[kXsNT][4];
#pragma unroll
  for (int t = 0; t < kXsNT; ++t)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[t][r] = 0.0;
  const int i = mt * 8 + (lane >> 2);
  const XsGroup gp{mt, MT, 1 + grp, sm_sc[grp], sm_bd + (size_t)grp * MT * 8 * 32, sm_be + (size_t)grp * MT * 32, sm_weak[wid]};
  for (int e = threadIdx.x; e < kXsWarps * 2 * 96; e += kXsThreads) sm_sc[0][e] = 0;
  __syncthreads();
  if (on) {
    const int n_split = split_terms ? nparts * G : 1, me = split_terms ? part * G + grp : 0;
    int boff[kXsNT];
#pragma unroll
    for (int t = 0; t < kXsNT; ++t) {
      const int n = tile * kXsCols + 8 * t + (lane >> 2);
      boff[t] = n < g.rest ? (n / g.inner) * (g.d * g.inner) + n % g.inner : -1;
    }
    const int inner = g.inner;
    auto src = [&](int q) {
      XsSrc S;
      const XsTerm tm = w.term[t_begin + q];
      S.a = i < g.d ? tm.M + (int64_t)i * g.d : nullptr;
#pragma unroll
      for (int t = 0; t < kXsNT; ++t) S.b[t] = boff[t] >= 0 ? tm.X + boff[t] : nullptr;
      return S;
    };
    int turn = 0;
    for (int q = me; q < nterm; q += n_split, ++turn) {
      xs_block<false>(gp, turn, src(q), g.d, [](int k) { return k; }, [inner](int k) { return k * inner; }, acc);
    }
  }
  double2* Y = pl ? w.planes + (int64_t)(w.plane[leg] + part) * ((int64_t)g.rest * g.d) : w.dst[o];
  auto put = [&](int n, int ii, double2 v) {
    if (n >= g.rest || ii >= g.d) return;
    const int at = (n / g.inner) * (g.d * g.inner) + n % g.inner + ii * g.inner;
    if (earlier) {
      const double2 y = Y[at];
      v.x += y.x;
      v.y += y.y;
    }
    Y[at] = v;
  };
  if (!split_terms || G == 1) {
    if (on)
#pragma unroll
      for (int t = 0; t < kXsNT; ++t)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          put(tile * kXsCols + 8 * t + 2 * (lane & 3) + j, i, make_double2(acc[t][2 * j], acc[t][2 * j + 1]));
    return;
  }
  // groups added in order; slot = column * 8 + row of the block
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kXsNT; ++t)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      red[wid][(8 * t + 2 * (lane & 3) + j) * 8 + (lane >> 2)] = make_double2(acc[t][2 * j], acc[t][2 * j + 1]);
  __syncthreads();
  for (int e = threadIdx.x; e < MT * kXsCols * 8; e += kXsThreads) {
    // consecutive threads along the faster of (row, position) in the destination
    int cc, ii;
    if (g.inner == 1) {
      ii = e % (MT * 8);
      cc = e / (MT * 8);
    } else {
      cc = e % kXsCols;
      ii = e / kXsCols;
    }
    const int m = ii >> 3, slot = cc * 8 + (ii & 7);
    double2 v = red[m][slot];
    for (int q = 1; q < G; ++q) {
      const double2 w = red[q * MT + m][slot];
      v.x += w.x;
      v.y += w.y;
    }
    put(tile * kXsCols + cc, ii, v);
  }
}

// RK4 stage update of element e with the computed derivative k (kernels.cuh, Epi), FP64.
__device__ __forceinline__ void rk_update(const Epi& ep, int64_t e, double2 k) {
  const double2 y = ep.y[e];
  const double c = ep.c;
  if (ep.mode == EPI_RK4) {
    const double2 a = ep.acc[e];
    ep.y[e] = make_double2(y.x + c * (a.x + k.x), y.y + c * (a.y + k.y));
    return;
  }
  if (ep.mode == EPI_RK1) {
    ep.acc[e] = k;
  } else {
    const double2 a = ep.acc[e];
    ep.acc[e] = make_double2(a.x + 2.0 * k.x, a.y + 2.0 * k.y);
  }
  ((double2*)ep.ys)[e] = make_double2(y.x + c * k.x, y.y + c * k.y);
}

// Sum of the planes of a one-output list, in order, the list's sparse terms (at
// most three entries a row: a few FMAs an element, not worth a tensor-core
// term) and its epilogue.
constexpr int kXsMaxSparse = 24;
struct XsSparse {
  int n;
  int dims[4];
  XsTerm term[kXsMaxSparse];
  int leg[kXsMaxSparse], diag[kXsMaxSparse];
};
__global__ void __launch_bounds__(128) k_xs_epilogue(const double2* planes, int n_planes, int64_t P, Epi ep,
                                                     double2* dst, const __grid_constant__ XsSparse sp) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= P) return;
  double2 k = n_planes > 0 ? planes[e] : make_double2(0.0, 0.0);
  for (int q = 1; q < n_planes; ++q) {
    const double2 v = planes[(int64_t)q * P + e];
    k.x += v.x;
    k.y += v.y;
  }
  for (int t = 0; t < sp.n; ++t) {
    int inner = 1;
    for (int l = 3; l > sp.leg[t]; --l) inner *= sp.dims[l];
    const int d = sp.dims[sp.leg[t]], i = (int)(e / inner) % d, nd = sp.diag[t] >> 24;
    for (int q = 0; q < nd; ++q) {
      const int off = (int)(int8_t)(sp.diag[t] >> (8 * q)), x = i + off;
      if (x < 0 || x >= d) continue;
      const double2 m = sp.term[t].M[i * d + x], v = sp.term[t].X[e + (int64_t)off * inner];
      k.x = fma(m.x, v.x, fma(-m.y, v.y, k.x));
      k.y = fma(m.x, v.y, fma(m.y, v.x, k.y));
    }
  }
  if (ep.mode == EPI_STORE) {
    dst[e] = k;
    return;
  }
  rk_update(ep, e, k);
}

// ---------------------------------------------------------------------------
// Environment projections E[x', x] = sum_r conj(U[x', r]) W[x, r] of wide bonds
// by the same split, W as the operator and the isometry conj(U) as the tensor
// operand (its scales leave W's rows as they are, so weakly occupied x keep their relative
// accuracy): x in blocks of 8 (one per warp of a group), x' in tiles of 16, the reduction range in chunks of 8 MT positions, one
// exact block product per chunk with its own scales, added in FP64. The chunks of
// a tile are dealt to the groups of KS CTAs (one cluster), whose sums CTA 0 adds
// in order through distributed shared memory.
// ---------------------------------------------------------------------------
constexpr int kXsMaxPj = 96;
struct XsPj {
  int dims[3], leg, KS;
  const double2* u;
  const double2* w[kXsMaxPj];
  double2* dst[kXsMaxPj];
};
__global__ void __launch_bounds__(kXsThreads, 2) k_xs_project(const __grid_constant__ XsPj w) {
  __shared__ __align__(16) uint4 sm_bd[kXsWarps * 8 * 32];
  __shared__ uint2 sm_be[kXsWarps * 32];
  __shared__ uint8_t sm_weak[kXsWarps][128];
  __shared__ int sm_sc[kXsWarps][2 * 96];
  __shared__ double2 tot[kXsWarps * kXsCols * 8];  // this CTA's 8 MT x 16 tile
  double2(*red)[kXsCols * 8] = reinterpret_cast<double2(*)[kXsCols * 8]>(sm_bd);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int dd[4] = {w.dims[0], w.dims[1], w.dims[2], 1};
  const XsLeg g = leg_of(dd, w.leg);
  const int MT = (g.d + 7) >> 3, G = kXsWarps / MT;
  const int mt = wid % MT, grp = wid / MT;
  const int rank = blockIdx.x % w.KS, tile = blockIdx.x / w.KS, o = blockIdx.y;
  const XsGroup gp{mt, MT, 1 + grp, sm_sc[grp], sm_bd + (size_t)grp * MT * 8 * 32, sm_be + (size_t)grp * MT * 32, sm_weak[wid]};
  for (int e = threadIdx.x; e < kXsWarps * 2 * 96; e += kXsThreads) sm_sc[0][e] = 0;
  __syncthreads();
  double acc[kXsNT][4];
#pragma unroll
  for (int t = 0; t < kXsNT; ++t)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[t][r] = 0.0;
  const int chunk = 8 * MT, nch = (g.rest + chunk - 1) / chunk;
  if (grp < G) {
    const int i = mt * 8 + (lane >> 2), inner = g.inner, span = g.d * g.inner;
    XsSrc S;
    S.a = i < g.d ? w.w[o] + (int64_t)i * inner : nullptr;
#pragma unroll
    for (int t = 0; t < kXsNT; ++t) {
      const int x = tile * kXsCols + 8 * t + (lane >> 2);
      S.b[t] = x < g.d ? w.u + (int64_t)x * inner : nullptr;
    }
    int turn = 0;
    for (int c = rank * G + grp; c < nch; c += w.KS * G, ++turn) {
      const int r0 = c * chunk, K = min(chunk, g.rest - r0);
      auto at = [=](int k) { return (r0 + k) / inner * span + (r0 + k) % inner; };
      xs_block<true>(gp, turn, S, K, at, at, acc);
    }
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kXsNT; ++t)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      red[wid][(8 * t + 2 * (lane & 3) + j) * 8 + (lane >> 2)] = make_double2(acc[t][2 * j], acc[t][2 * j + 1]);
  __syncthreads();
  const int ne = MT * kXsCols * 8;
  for (int e = threadIdx.x; e < ne; e += kXsThreads) {
    const int m = e / (kXsCols * 8), slot = e % (kXsCols * 8);
    double2 v = red[m][slot];
    for (int q = 1; q < G; ++q) {
      const double2 x = red[q * MT + m][slot];
      v.x += x.x;
      v.y += x.y;
    }
    tot[e] = v;
  }
  if (w.KS > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    // every CTA adds its share of the tile's entries over the CTAs, in order
    for (int e = rank * kXsThreads + threadIdx.x; e < ne; e += w.KS * kXsThreads) {
      double2 v = *cluster.map_shared_rank(&tot[e], 0);
      for (int q = 1; q < w.KS; ++q) {
        const double2 x = *cluster.map_shared_rank(&tot[e], q);
        v.x += x.x;
        v.y += x.y;
      }
      const int ii = (e / (kXsCols * 8)) * 8 + (e & 7), x = tile * kXsCols + (e % (kXsCols * 8)) / 8;
      if (ii < g.d && x < g.d) w.dst[o][(int64_t)x * g.d + ii] = v;
    }
    cluster.sync();  // shared memory stays until every CTA has read it
    return;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < ne; e += kXsThreads) {
    const int ii = (e / (kXsCols * 8)) * 8 + (e & 7), x = tile * kXsCols + (e % (kXsCols * 8)) / 8;
    if (ii < g.d && x < g.d) w.dst[o][(int64_t)x * g.d + ii] = tot[e];
  }
}

namespace {

int sm_count() {
  static int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
      v = 152;
    return v;
  }();
  return n;
}

}  // namespace

// Lists that take this path: contracted legs of at most 64, all outputs alike,
// fewer than 2^30 elements an output, no more outputs and terms than a launch
// has room for (everything else stays on the CUDA-core kernel and its tile
// shapes, so ttn_autotune asks here too), and enough multiply-adds that the CUDA-core kernel
// would be bound by FP64 issue instead of by its launch.
bool xs_applicable(const ApList& L, const ApOut* outs, const ApTerm* terms, int max_split) {
  if (L.n_tiles <= 0) return false;
  const ApOut& f = outs[L.out_begin];
  const int64_t P = (int64_t)f.d0 * f.d1 * f.d2 * f.d3;
  double dense = 0.0;  // sparse operators are cheap on the CUDA cores
  if (P >= (int64_t)1 << 30 || L.out_end - L.out_begin > kXsMaxOuts) return false;
  if (outs[L.out_end - 1].term_end - f.term_begin > kXsMaxTerms) return false;
  for (int o = L.out_begin; o < L.out_end; ++o) {
    const ApOut& u = outs[o];
    if (u.d0 != f.d0 || u.d1 != f.d1 || u.d2 != f.d2 || u.d3 != f.d3) return false;
    const int dd[4] = {u.d0, u.d1, u.d2, u.d3};
    if (u.term_begin == u.term_end) return false;
    for (int t = u.term_begin; t < u.term_end; ++t) {
      const ApTerm& tm = terms[t];
      if (tm.mat < 0 || tm.leg < 0 || tm.leg > 3 || dd[tm.leg] > kXsMaxD) return false;
      if (!tm.pad) dense += 8.0 * P * dd[tm.leg];
    }
  }
  return dense >= xs_min_flops(max_split);
}

bool launch_apply_xs(double2* const* bufs, double2* const* mats, const ApList& L, const Epi& e, const ApOut* outs,
                     const ApTerm* terms, double2* planes, int64_t plane_elems, int max_split,
                     cudaStream_t s) {
  const int n_outs = L.out_end - L.out_begin;
  const ApOut& u = outs[L.out_begin];
  const int dd[4] = {u.d0, u.d1, u.d2, u.d3};
  const int64_t P = (int64_t)u.d0 * u.d1 * u.d2 * u.d3;
  int nterm[4] = {0, 0, 0, 0};
  bool multi_leg = false;
  for (int o = L.out_begin; o < L.out_end; ++o)
    for (int t = outs[o].term_begin; t < outs[o].term_end; ++t) {
      ++nterm[terms[t].leg];
      multi_leg = multi_leg || terms[t].leg != terms[outs[o].term_begin].leg;
    }
  int tiles[4];
  for (int l = 0; l < 4; ++l) tiles[l] = (int)((P / dd[l] + kXsCols - 1) / kXsCols);
  XsWork gr{};
  XsSparse sp{};
  int nq = 0;
  for (int i = 0; i < 4; ++i) gr.dims[i] = sp.dims[i] = dd[i];
  for (int o = 0; o < n_outs; ++o) {
    const ApOut& v = outs[L.out_begin + o];
    gr.dst[o] = v.dst >= 0 ? bufs[v.dst] : nullptr;
    gr.tb[o][0] = (short)nq;
    for (int l = 0; l < 4; ++l) {
      for (int t = v.term_begin; t < v.term_end; ++t)
        if (terms[t].leg == l && n_outs == 1 && terms[t].pad && sp.n < kXsMaxSparse) {
          sp.leg[sp.n] = l;
          sp.diag[sp.n] = terms[t].pad;
          sp.term[sp.n++] = XsTerm{mats[terms[t].mat], bufs[terms[t].src]};
        } else if (terms[t].leg == l)
          gr.term[nq++] = XsTerm{mats[terms[t].mat], bufs[terms[t].src]};
      gr.tb[o][l + 1] = (short)nq;
    }
  }
  if (n_outs == 1) {
    for (int l = 0; l < 4; ++l) nterm[l] = gr.tb[0][l + 1] - gr.tb[0][l];
    // all legs in one launch, each leg's terms cut into parts while a warp
    // still has more than one term and the launch stays below four CTAs per SM
    // (two are resident at a time)
    int ctas = 0, n_planes = 0, groups[4];
    for (int l = 0; l < 4; ++l) {
      // a leg without a dense term may be of any size, also above the kXsWarps row blocks of a CTA
      groups[l] = nterm[l] ? kXsWarps / ((dd[l] + 7) / 8) : 0;
      gr.parts[l] = 1;
      if (nterm[l]) {
        ctas += tiles[l];
        ++n_planes;
      }
    }
    if ((int64_t)n_planes * P > plane_elems) return false;
    for (;;) {
      int best = -1;
      double chain = 1.0;
      for (int l = 0; l < 4; ++l) {
        if (!nterm[l]) continue;
        const int q = groups[l] * gr.parts[l];
        const double c = (double)((nterm[l] + q - 1) / q) * ((dd[l] + 7) / 8);
        if (nterm[l] > q && gr.parts[l] < max_split && c > chain) {
          chain = c;
          best = l;
        }
      }
      if (best < 0 || ctas + tiles[best] > 4 * sm_count() || (int64_t)(n_planes + 1) * P > plane_elems) break;
      ++gr.parts[best];
      ctas += tiles[best];
      ++n_planes;
    }
    int q = 0;
    for (int l = 0; l < 4; ++l) {
      gr.plane[l] = q;
      gr.lt[l + 1] = gr.lt[l] + (nterm[l] ? tiles[l] * gr.parts[l] : 0);
      if (nterm[l]) q += gr.parts[l];
    }
    gr.leg = -1;
    gr.planes = planes;
    k_xs_apply<<<counted(dim3(gr.lt[4], 1)), kXsThreads, 0, s>>>(gr);
    k_xs_epilogue<<<counted((int)((P + 127) / 128)), 128, 0, s>>>(planes, q, P, with_coef(e), gr.dst[0], sp);
    return true;
  }
  if (e.mode != EPI_STORE) return false;
  // several outputs: one launch when no output has terms on two legs, else one
  // launch per leg, later legs adding to what earlier ones wrote. Outputs of
  // at most two terms a leg use the groups for positions, so fewer CTAs.
  int most[4] = {0, 0, 0, 0};
  for (int o = L.out_begin; o < L.out_end; ++o) {
    int c[4] = {0, 0, 0, 0};
    for (int t = outs[o].term_begin; t < outs[o].term_end; ++t) ++c[terms[t].leg];
    for (int l = 0; l < 4; ++l) most[l] = std::max(most[l], c[l]);
  }
  int gx[4], gmax = 0;
  for (int l = 0; l < 4; ++l) {
    const int G = kXsWarps / ((dd[l] + 7) / 8);
    gx[l] = nterm[l] == 0 ? 0 : most[l] > kXsTermSplit ? tiles[l] : (tiles[l] + G - 1) / G;
    gmax = std::max(gmax, gx[l]);
  }
  if (!multi_leg) {
    gr.leg = -2;
    k_xs_apply<<<counted(dim3(gmax, n_outs)), kXsThreads, 0, s>>>(gr);
    return true;
  }
  for (int l = 0; l < 4; ++l)
    if (nterm[l]) {
      gr.leg = l;
      k_xs_apply<<<counted(dim3(gx[l], n_outs)), kXsThreads, 0, s>>>(gr);
    }
  return true;
}

bool launch_project_xs(double2* const* bufs, double2* const* mats, const PjList& L, const PjOut* pjs, int max_split,
                       cudaStream_t s) {
  const int n = L.out_end - L.out_begin;
  if (n < 1 || n > kXsMaxPj) return false;
  const PjOut& f = pjs[L.out_begin];
  if (L.flops < xs_min_flops(max_split)) return false;
  const int dd[3] = {f.d0, f.d1, f.d2}, d = dd[f.leg];
  const int64_t P = (int64_t)f.d0 * f.d1 * f.d2;
  if (d > kXsMaxD || d < 8 || P >= (int64_t)1 << 30) return false;
  XsPj w{};
  for (int i = 0; i < 3; ++i) w.dims[i] = dd[i];
  w.leg = f.leg;
  w.u = bufs[f.u_buf];
  for (int o = 0; o < n; ++o) {
    const PjOut& q = pjs[L.out_begin + o];
    if (q.d0 != f.d0 || q.d1 != f.d1 || q.d2 != f.d2 || q.leg != f.leg || q.u_buf != f.u_buf) return false;
    w.w[o] = bufs[q.w_buf];
    w.dst[o] = mats[q.dst_mat];
  }
  // split the range while the launch is below two CTAs per SM and a group keeps a chunk
  const int MT = (d + 7) / 8, G = kXsWarps / MT, tiles = (d + kXsCols - 1) / kXsCols;
  const int nch = (int)((P / d + 8 * MT - 1) / (8 * MT));
  w.KS = 1;
  while (w.KS < std::min(8, max_split) && w.KS * G < nch && (int64_t)tiles * n * w.KS < 2 * sm_count()) ++w.KS;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = counted(dim3((unsigned)(tiles * w.KS), (unsigned)n, 1));
  cfg.blockDim = dim3(kXsThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)w.KS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_xs_project, w) == cudaSuccess;
}

}  // namespace ttn
