// Compensated FP32 arithmetic for the statevector pass kernels.
//
// An amplitude of a stage group is held as a sum q + l of two FP32 complex
// numbers.  The high parts q of the whole group are multiples of one grid
// unit u, a power of two chosen from the group's largest component, and are
// kept biased: H = C + q with C = 1.5 * 2^23 u, so that H lies in the binade
// [2^23 u, 2^24 u) whose FP32 spacing is u.  Adding a product to H in one
// FMA then rounds it to the grid, sums of high parts are exact without any
// TwoSum, and the part of the product that the grid dropped is recovered by
// one more FMA:
//   H' = fma(c, yq, H)         (rounds c*yq to a multiple of u)
//   d  = H' - H                (exact: the rounded product)
//   e  = fma(c, yq, -d)        (what the grid dropped, |e| <= u/2)
// The low part l collects e, the products with the operands' low parts and
// those with the constants' own FP32 remainders.
//
// The grid: components of a unitary's group stay within sqrt(32) of the
// largest one, and the unnormalized rotations below stretch them by at most
// sqrt(2) each (four per stage), together less than 2^5; with the largest
// component below 2^E the unit u = 2^(E + 5 - 22) keeps every q within
// 2^22 u.  The low parts are a few u (at most 5.2 after four rotations of
// 20000 random groups), so one operation errs by about 2^-24 * 4 u = 2^-39 of
// the group's largest amplitude (the four rotations of those groups: 2^-41.1
// rms, 2^-38.1 at most), far below the FP32 rounding (2^-25) of the amplitudes
// that the stage stores.  An amplitude below half a unit, 2^-18 of the
// largest one, lies in its low part alone: plain FP32 precision.
//
// Constants are FP32 pairs throughout.  Rotations were tried with quotients
// made exact in FP32 and a factor on the inputs (one instruction less per
// output, 24-qubit sweep of 64 tasks 93.9 against 97.0 ms): the factor put
// hundreds of units into the low parts and erred by 2^-34, always the same
// way for one angle, so that 5000 repeats of it moved amplitudes by 3e-7.
//
// A two-term output costs 11 packed instructions and an unnormalized
// rotation output 6 (and one more to un-bias its operand), against 16 for
// the double-float arithmetic this replaced (products split by FMA, sums by
// TwoSum): a full rotation stage takes 44 packed instructions per amplitude
// instead of 80, and the kernels that run it are bound by the FMA pipe.
//
// Without compensation, the FP32 roundings of the ~600 rotations that every
// amplitude of a 24-qubit, 24-layer ansatz goes through move a Pauli-sum
// energy by about 1e-6 of its typical size; with it, the state is rounded
// only when it is written back to FP32 storage.
//
// Both components of a complex amplitude go through the same real
// coefficients, so the arithmetic is written on float2 with the packed
// two-lane FP32 instructions.
#pragma once

#include <cuda_runtime.h>

namespace qw {

__device__ __forceinline__ float2 f2s(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 f2neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 f2swap(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __fadd2_rn(a, f2neg(b)); }

// H <- H + c y on the grid, what the grid drops and the low-order products
// into r: c = ch + cl, y = yq + yl
__device__ __forceinline__ void gd_mac(float2 ch, float2 cl, float2 yq, float2 yl, float2 &H, float2 &r) {
  const float2 h1 = __ffma2_rn(ch, yq, H);
  float2 e = __ffma2_rn(ch, yq, f2sub(H, h1));
  e = __ffma2_rn(ch, yl, e);
  r = __ffma2_rn(cl, yq, e);
  H = h1;
}

// the same added to the amplitude H, l
__device__ __forceinline__ void gd_rot(float2 ch, float2 cl, float2 yq, float2 yl, float2 &H, float2 &l) {
  const float2 h1 = __ffma2_rn(ch, yq, H);
  float2 e = __ffma2_rn(ch, yq, f2sub(H, h1));
  e = __ffma2_rn(cl, yq, e);
  l = __fadd2_rn(__ffma2_rn(ch, yl, l), e);
  H = h1;
}

// H, l <- c1 x + c2 y (coefficients and operands as pairs)
__device__ __forceinline__ void gd_lin2(float2 C, float2 c1h, float2 c1l, float2 xq, float2 xl, float2 c2h, float2 c2l,
                                        float2 yq, float2 yl, float2 &H, float2 &l) {
  float2 h = C, r1, r2;
  gd_mac(c1h, c1l, xq, xl, h, r1);
  gd_mac(c2h, c2l, yq, yl, h, r2);
  H = h;
  l = __fadd2_rn(r1, r2);
}

// z <- w z for a complex constant w = (wr, wi), both parts as pairs:
// (wr zr - wi zi, wr zi + wi zr) = wr (zr, zi) + (-wi, wi) (zi, zr)
__device__ __forceinline__ void gd_cmul(float2 C, float wrh, float wrl, float wih, float wil, float2 &H, float2 &l) {
  const float2 q = f2sub(H, C), ql = l;
  gd_lin2(C, f2s(wrh), f2s(wrl), q, ql, make_float2(-wih, wih), make_float2(-wil, wil), f2swap(q), f2swap(ql), H, l);
}

// ---- register operations on the N = 2^G amplitudes of a stage group ------
// m / ml: the op's parameters (see SvKind) and their FP32 remainders.

// Unnormalized rotation on position P, t = {t0, t1} and their remainders:
//   x' = x + t0 y,  y' = y + t1 x
// (a real orthogonal 2x2 with its diagonal taken out into the factors of the
// stage's table; the host arranges |t| <= 1)
__device__ __forceinline__ void gd_pair(float2 C, float4 t, float2 &Hx, float2 &lx, float2 &Hy, float2 &ly) {
  const float2 xq = f2sub(Hx, C), yq = f2sub(Hy, C), xl = lx, yl = ly;
  gd_rot(f2s(t.x), f2s(t.z), yq, yl, Hx, lx);
  gd_rot(f2s(t.y), f2s(t.w), xq, xl, Hy, ly);
}
template <int P, int N>
__device__ __forceinline__ void gdop_rot(float2 C, float2 (&H)[N], float2 (&l)[N], float4 t) {
#pragma unroll
  for (int i = 0; i < N; i++)
    if (!(i & (1 << P))) gd_pair(C, t, H[i], l[i], H[i | (1 << P)], l[i | (1 << P)]);
}
// real 2x2 {r00, r01; r10, r11} on position P
template <int P, int N>
__device__ __forceinline__ void gdop_real(float2 C, float2 (&H)[N], float2 (&l)[N], float r00, float r01, float r10,
                                          float r11, float e00, float e01, float e10, float e11) {
#pragma unroll
  for (int i = 0; i < N; i++) {
    if (i & (1 << P)) continue;
    const int j = i | (1 << P);
    const float2 xq = f2sub(H[i], C), yq = f2sub(H[j], C), xl = l[i], yl = l[j];
    gd_lin2(C, f2s(r00), f2s(e00), xq, xl, f2s(r01), f2s(e01), yq, yl, H[i], l[i]);
    gd_lin2(C, f2s(r10), f2s(e10), xq, xl, f2s(r11), f2s(e11), yq, yl, H[j], l[j]);
  }
}
// K_RP layout {r00, r01, r10, r11, pr, pi}: the real 2x2, then diag(1, p)
template <int P, int N>
__device__ __forceinline__ void gdop_rp(float2 C, float2 (&H)[N], float2 (&l)[N], const float (&m)[8],
                                        const float (&ml)[8]) {
  gdop_real<P, N>(C, H, l, m[0], m[1], m[2], m[3], ml[0], ml[1], ml[2], ml[3]);
#pragma unroll
  for (int i = 0; i < N; i++)
    if (i & (1 << P)) gd_cmul(C, m[4], ml[4], m[5], ml[5], H[i], l[i]);
}
// K_R layout {r00, 0, r01, 0, r10, 0, r11, 0}
template <int P, int N>
__device__ __forceinline__ void gdop_r(float2 C, float2 (&H)[N], float2 (&l)[N], const float (&m)[8],
                                       const float (&ml)[8]) {
  gdop_real<P, N>(C, H, l, m[0], m[2], m[4], m[6], ml[0], ml[2], ml[4], ml[6]);
}
// general 2x2 {u00, u01; u10, u11}, complex entries (re, im) in m[0..7]
template <int P, int N>
__device__ __forceinline__ void gdop_u1(float2 C, float2 (&H)[N], float2 (&l)[N], const float (&m)[8],
                                        const float (&ml)[8]) {
#pragma unroll
  for (int i = 0; i < N; i++) {
    if (i & (1 << P)) continue;
    const int j = i | (1 << P);
    const float2 xq = f2sub(H[i], C), yq = f2sub(H[j], C), xl = l[i], yl = l[j];
#pragma unroll
    for (int r = 0; r < 2; r++) {
      // u_r0 x + u_r1 y = Re u_r0 x + Im u_r0 (-xi, xr) + [same for y]
      const int o = 4 * r;
      float2 h = C, e0, e1, e2, e3;
      gd_mac(f2s(m[o]), f2s(ml[o]), xq, xl, h, e0);
      gd_mac(make_float2(-m[o + 1], m[o + 1]), make_float2(-ml[o + 1], ml[o + 1]), f2swap(xq), f2swap(xl), h, e1);
      gd_mac(f2s(m[o + 2]), f2s(ml[o + 2]), yq, yl, h, e2);
      gd_mac(make_float2(-m[o + 3], m[o + 3]), make_float2(-ml[o + 3], ml[o + 3]), f2swap(yq), f2swap(yl), h, e3);
      const float2 e = __fadd2_rn(__fadd2_rn(e0, e1), __fadd2_rn(e2, e3));
      if (r == 0) { H[i] = h; l[i] = e; }
      else { H[j] = h; l[j] = e; }
    }
  }
}
// diag(d0, d1): m = {d0r, d0i, d1r, d1i}
template <int P, int N>
__device__ __forceinline__ void gdop_d1(float2 C, float2 (&H)[N], float2 (&l)[N], const float (&m)[8],
                                        const float (&ml)[8]) {
#pragma unroll
  for (int i = 0; i < N; i++) {
    const int o = (i & (1 << P)) ? 2 : 0;
    gd_cmul(C, m[o], ml[o], m[o + 1], ml[o + 1], H[i], l[i]);
  }
}
// diag(1, p): m = {pr, pi}
template <int P, int N>
__device__ __forceinline__ void gdop_p1(float2 C, float2 (&H)[N], float2 (&l)[N], const float (&m)[8],
                                        const float (&ml)[8]) {
#pragma unroll
  for (int i = 0; i < N; i++)
    if (i & (1 << P)) gd_cmul(C, m[0], ml[0], m[1], ml[1], H[i], l[i]);
}
// amplitudes with bits A and B set times p = {pr, pi}; p = -1 (CZ) negates
template <int A, int B, int N>
__device__ __forceinline__ void gdop_cd(float2 C, float2 (&H)[N], float2 (&l)[N], const float (&m)[8],
                                        const float (&ml)[8]) {
  const bool neg = m[0] == -1.f && m[1] == 0.f && ml[0] == 0.f && ml[1] == 0.f;
#pragma unroll
  for (int i = 0; i < N; i++) {
    if (!(i & (1 << A)) || !(i & (1 << B))) continue;
    if (neg) {
      H[i] = f2sub(C, f2sub(H[i], C));  // exact on the grid
      l[i] = f2neg(l[i]);
    } else {
      gd_cmul(C, m[0], ml[0], m[1], ml[1], H[i], l[i]);
    }
  }
}
// [[c, -is], [-is, c]]: m = {c, s}
//   x' = c x - i s y = c (xr, xi) + (s, -s) (yi, yr)
//   y' = c y - i s x = c (yr, yi) + (s, -s) (xi, xr)
template <int P, int N>
__device__ __forceinline__ void gdop_rx(float2 C, float2 (&H)[N], float2 (&l)[N], const float (&m)[8],
                                        const float (&ml)[8]) {
  const float2 c = f2s(m[0]), cl = f2s(ml[0]);
  const float2 s = make_float2(m[1], -m[1]), sl = make_float2(ml[1], -ml[1]);
#pragma unroll
  for (int i = 0; i < N; i++) {
    if (i & (1 << P)) continue;
    const int j = i | (1 << P);
    const float2 xq = f2sub(H[i], C), yq = f2sub(H[j], C), xl = l[i], yl = l[j];
    gd_lin2(C, c, cl, xq, xl, s, sl, f2swap(yq), f2swap(yl), H[i], l[i]);
    gd_lin2(C, c, cl, yq, yl, s, sl, f2swap(xq), f2swap(xl), H[j], l[j]);
  }
}

// dispatch on the dense op index (the same table as the plain kernels);
// positions beyond the group (1 << P >= N) never occur in its programs
template <int N>
__device__ __forceinline__ void gd_apply_op(uint32_t code, const float (&m)[8], const float (&ml)[8], float2 C,
                                            float2 (&H)[N], float2 (&l)[N]) {
  switch (code) {
#define QW_ONE(K, P, F) \
  case sv_op_index(K, P, 0): if constexpr ((1 << P) < N) F<P, N>(C, H, l, m, ml); break;
#define QW_ALL(K, F) QW_ONE(K, 0, F) QW_ONE(K, 1, F) QW_ONE(K, 2, F) QW_ONE(K, 3, F)
    QW_ALL(K_U1, gdop_u1)
    QW_ALL(K_D1, gdop_d1)
    QW_ALL(K_P1, gdop_p1)
    QW_ALL(K_R, gdop_r)
    QW_ALL(K_RX, gdop_rx)
    QW_ALL(K_RP, gdop_rp)
#undef QW_ALL
#undef QW_ONE
#define CD(x, y) case sv_op_index(K_CD, x, y): if constexpr ((1 << y) < N) gdop_cd<x, y, N>(C, H, l, m, ml); break;
    CD(0, 1) CD(0, 2) CD(0, 3) CD(1, 2) CD(1, 3) CD(2, 3)
#undef CD
    default: break;
  }
}

}  // namespace qw
