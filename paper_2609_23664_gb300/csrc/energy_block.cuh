// Pauli-sum energy over one block of amplitudes, shared by the stand-alone
// energy kernel and by the persistent suffix kernel, which runs energy
// blocks as a second kind of work item.
//
// E = sum_k c_k <psi|P_k|psi> / <psi|psi>, P|x> = i^{#Y} (-1)^{popc(x&z)}|x^m>.
// For m != 0 the pair (x, x^m) is visited once and contributes
// 2 Re(i^{#Y} (-1)^{popc(x&z)} conj(psi[x^m]) psi[x]); the host folds 2, the
// sign of i^{#Y} and the coefficient into EnTerm::coef and the choice of real
// or imaginary part into EnTerm::code.
//
// Terms are evaluated in groups of up to four independent flip masks.  With V
// the span of a group's masks, a thread loads the 16 amplitudes of one coset
// x0 ^ V into registers, where every pair of every term whose mask lies in V
// is at hand: the state is read once per four terms instead of half of it
// once per term, which halves the L2 -> SM traffic that bounds the kernel
// (200 random terms at 24 qubits: 52 sweeps of the state, 6.7 GB, instead of
// 14 GB; the SMs take at most 64 bytes per clock each from L2).
//
// A coset is represented by its element with zeros at the pivot bits of V
// (its leading bits), so consecutive representatives are consecutive
// addresses except at the pivots and a warp's loads stay coalesced.  Groups
// are formed within a class of terms that flip the same bits above an
// L2-sized chunk: the blocks of one class then sweep one pair of chunks at a
// time, which stays in L2 while all groups of the class visit it.
#pragma once

#include <cuda_runtime.h>

#include "qw_internal.h"

namespace qw {

template <typename T> struct EnC;
template <> struct EnC<float> { typedef float2 t; };
template <> struct EnC<double> { typedef double2 t; };

struct DFAcc {  // double-float accumulator (two-sum of the high part)
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float p) {
    const float s = hi + p;
    const float bp = s - hi;
    const float err = (hi - (s - bp)) + (p - bp);
    hi = s;
    lo += err;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
struct DAcc {
  double v = 0.0;
  __device__ __forceinline__ void add(double p) { v += p; }
  __device__ __forceinline__ double value() const { return v; }
};
template <typename T> struct AccOf;
template <> struct AccOf<float> { typedef DFAcc t; };
template <> struct AccOf<double> { typedef DAcc t; };

__device__ __forceinline__ double en_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Warp sums of the lanes' accumulators.  FP32 blocks add in double-float:
// FP64 adds run at 1/64 of the FP32 rate, and a block is short enough (13
// groups per class) that 12 of them per thread showed.  Where 32 lanes'
// sums leave the FP32 range (amplitudes of about 10^18) they add in FP64.
__device__ __forceinline__ double en_warp_total(const DFAcc in) {
  DFAcc a = in;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_xor_sync(0xffffffffu, a.hi, o), l = __shfl_xor_sync(0xffffffffu, a.lo, o);
    a.add(h);
    a.lo += l;
  }
  if (__any_sync(0xffffffffu, !(fabsf(a.hi) <= 3.402823466e38f)))
    // (an infinite sum has no low part)
    return en_warp_sum(fabsf(in.hi) <= 3.402823466e38f ? in.value() : (double)in.hi);
  return a.value();
}
__device__ __forceinline__ double en_warp_total(DAcc a) { return en_warp_sum(a.v); }

// NC: the state is read-only for the whole launch (read-only cache path);
// otherwise it was written earlier in the same launch by other CTAs and is
// read from L2.
template <bool NC, typename C>
__device__ __forceinline__ C en_ld(const C *p) {
  if (NC) return __ldg(p);
  return __ldcg(p);
}

// Amplitudes of a thread: index i = combination of the four basis masks, and
// below it in FP32 blocks of aligned states (PAIR) the two neighbours 2x, 2x+1
// that one 16-byte load brings: the span then has bit 0 as a fifth direction,
// and everything that is per thread and term (addresses, signs, branches) is
// paid once for 32 amplitudes.
template <typename T, bool PAIR> struct EnAmp {
  typedef typename EnC<T>::t C;
  static constexpr int N = PAIR ? 32 : 16;
};

// k-th pair {x, x ^ m} for m = basis combination MC, and bit 0 when E (PAIR):
// index of its first member, whose highest flipped direction is clear
template <int MC, int E, bool PAIR>
__device__ __forceinline__ constexpr int en_low(int k) {
  constexpr int m = PAIR ? 2 * MC + E : MC;
  constexpr int h = m >= 16 ? 4 : m >= 8 ? 3 : m >= 4 ? 2 : m >= 2 ? 1 : 0;
  return m ? (((k >> h) << (h + 1)) | (k & ((1 << h) - 1))) : k;
}

// Sum over those pairs of (-1)^{popc(x & z)} times the real (IM: imaginary)
// part of conj(a[x ^ m]) a[x]; m = 0: over all amplitudes, with |a[x]|^2.
// FP32 adds through a butterfly of +-1 multiply-adds (exact products, no
// branch) with the signs s of the pair index's bits, the real part on both
// components at once (packed instructions: the kernel is bound by
// instruction issue); FP64, whose pipe runs at 1/64 of the FP32 rate, flips
// signs on the integer pipe instead and accumulates straight into its
// multiply-adds (16 FP64 operations per 8 pairs, not 23).
template <int MC, int E, bool IM, bool PAIR>
__device__ __forceinline__ float en_pairs(const float2 (&a)[EnAmp<float, PAIR>::N], const float (&s)[5]) {
  constexpr int m = PAIR ? 2 * MC + E : MC, N = EnAmp<float, PAIR>::N, NP = m ? N / 2 : N;
  if constexpr (IM) {
    float v[NP];
#pragma unroll
    for (int k = 0; k < NP; k++) {
      const float2 x = a[en_low<MC, E, PAIR>(k)], p = a[en_low<MC, E, PAIR>(k) ^ m];
      v[k] = p.x * x.y - p.y * x.x;
    }
#pragma unroll
    for (int w = NP / 2, b = 0; w > 0; w /= 2, b++)
#pragma unroll
      for (int k = 0; k < w; k++) v[k] = fmaf(s[b], v[2 * k + 1], v[2 * k]);
    return v[0];
  } else {
    // the first level takes every second product unrounded: its sign goes
    // to one factor (exact), the product into the multiply-add
    float2 v[NP / 2];
#pragma unroll
    for (int k = 0; k < NP / 2; k++) {
      const int i = en_low<MC, E, PAIR>(2 * k), j = en_low<MC, E, PAIR>(2 * k + 1);
      v[k] = __ffma2_rn(__fmul2_rn(make_float2(s[0], s[0]), a[j ^ m]), a[j], __fmul2_rn(a[i ^ m], a[i]));
    }
#pragma unroll
    for (int w = NP / 4, b = 1; w > 0; w /= 2, b++) {
      const float2 sb = make_float2(s[b], s[b]);
#pragma unroll
      for (int k = 0; k < w; k++) v[k] = __ffma2_rn(sb, v[2 * k + 1], v[2 * k]);
    }
    return v[0].x + v[0].y;
  }
}
template <int MC, int E, bool IM, bool PAIR>
__device__ __forceinline__ double en_pairs(const double2 (&a)[16], uint32_t zz) {
  static_assert(!PAIR, "FP64 amplitudes are 16 bytes each");
  double s0 = 0, s1 = 0;
#pragma unroll
  for (int k = 0; k < (MC ? 8 : 16); k++) {
    const int i = en_low<MC, 0, false>(k);
    const int sgn = (__popc((uint32_t)i & zz) & 1) << 31;
    const double2 p = a[i ^ MC];
    const double px = __hiloint2double(__double2hiint(p.x) ^ sgn, __double2loint(p.x));
    const double py = __hiloint2double(__double2hiint(p.y) ^ sgn, __double2loint(p.y));
    s0 = fma(px, IM ? a[i].y : a[i].x, s0);
    s1 = fma(IM ? -py : py, IM ? a[i].x : a[i].y, s1);
  }
  return s0 + s1;
}
// Squared norm of the amplitudes [LO, LO + CNT), added in a tree: the error of
// 32 FP32 squares added one after another is the same in every thread of a
// state of constant amplitude (5e-7 of the norm, and of every energy).
template <int LO, int CNT, int N>
__device__ __forceinline__ float2 en_squares(const float2 (&a)[N]) {
  if constexpr (CNT == 2) return __ffma2_rn(a[LO], a[LO], __fmul2_rn(a[LO + 1], a[LO + 1]));
  else return __fadd2_rn(en_squares<LO, CNT / 2>(a), en_squares<LO + CNT / 2, CNT / 2>(a));
}
template <int N>
__device__ __forceinline__ float en_norm(const float2 (&a)[N]) {
  const float2 s = en_squares<0, N>(a);
  return s.x + s.y;
}
template <int N>
__device__ __forceinline__ double en_norm(const double2 (&a)[N]) {
  double s = 0;
#pragma unroll
  for (int k = 0; k < N; k++) s += a[k].x * a[k].x + a[k].y * a[k].y;
  return s;
}
// the term's sign data in the form its precision takes
template <typename T> struct EnSign;
template <> struct EnSign<float> {
  float s[5];
  __device__ __forceinline__ EnSign(const EnTerm *t, uint32_t code) {
    const float4 v = __ldg((const float4 *)t + 1);
    s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
    s[4] = (code & EN_LAST_SIGN) ? -1.f : 1.f;  // only a term without flips has five
  }
  __device__ __forceinline__ const float (&get() const)[5] { return s; }
};
template <> struct EnSign<double> {
  uint32_t zz;
  __device__ __forceinline__ EnSign(const EnTerm *, uint32_t code) : zz((code >> 8) & 15u) {}
  __device__ __forceinline__ uint32_t get() const { return zz; }
};
// code bits 0-3: MC, bit 4: imaginary part, bit 5: E
template <typename T, bool PAIR, typename C>
__device__ __forceinline__ T en_pairs_rt(const C (&a)[EnAmp<T, PAIR>::N], uint32_t code, const EnSign<T> &sg) {
  switch (code & (PAIR ? 63u : 31u)) {
#define QW_PR(S) case S: return en_pairs<(S & 15), 0, (S >= 16), PAIR>(a, sg.get());
    QW_PR(0) QW_PR(1) QW_PR(2) QW_PR(3) QW_PR(4) QW_PR(5) QW_PR(6) QW_PR(7)
    QW_PR(8) QW_PR(9) QW_PR(10) QW_PR(11) QW_PR(12) QW_PR(13) QW_PR(14) QW_PR(15)
    QW_PR(17) QW_PR(18) QW_PR(19) QW_PR(20) QW_PR(21) QW_PR(22) QW_PR(23)
    QW_PR(24) QW_PR(25) QW_PR(26) QW_PR(27) QW_PR(28) QW_PR(29) QW_PR(30)
#undef QW_PR
    default: break;
  }
  if constexpr (PAIR) {
    switch (code & 63u) {
#define QW_PR(S) case 32 + S: return en_pairs<(S & 15), 1, (S >= 16), PAIR>(a, sg.get());
      QW_PR(0) QW_PR(1) QW_PR(2) QW_PR(3) QW_PR(4) QW_PR(5) QW_PR(6) QW_PR(7)
      QW_PR(8) QW_PR(9) QW_PR(10) QW_PR(11) QW_PR(12) QW_PR(13) QW_PR(14) QW_PR(15)
      QW_PR(16) QW_PR(17) QW_PR(18) QW_PR(19) QW_PR(20) QW_PR(21) QW_PR(22) QW_PR(23)
      QW_PR(24) QW_PR(25) QW_PR(26) QW_PR(27) QW_PR(28) QW_PR(29) QW_PR(30) QW_PR(31)
#undef QW_PR
      default: break;
    }
  }
  return en_pairs<15, 0, true, PAIR>(a, sg.get());
}

template <typename T> __device__ __forceinline__ T en_coef(const uint4 &q);
template <> __device__ __forceinline__ float en_coef<float>(const uint4 &q) { return __uint_as_float(q.z); }
template <> __device__ __forceinline__ double en_coef<double>(const uint4 &q) {
  return __hiloint2double((int)q.w, (int)q.z);
}

// Keeps the compiler from hoisting the pair products of every case of the
// switch out of the term loop (they do not change in it, and their 240
// values would be spilled).
template <int N>
__device__ __forceinline__ void en_pin(float2 (&a)[N]) {
#pragma unroll
  for (int k = 0; k < N; k++) asm volatile("" : "+f"(a[k].x), "+f"(a[k].y));
}
template <int N>
__device__ __forceinline__ void en_pin(double2 (&a)[N]) {
#pragma unroll
  for (int k = 0; k < N; k++) asm volatile("" : "+d"(a[k].x), "+d"(a[k].y));
}

// one term on the basis mask of combination MC
template <typename T, int MC, bool PAIR, typename C>
__device__ __forceinline__ void en_slot(const C (&a)[EnAmp<T, PAIR>::N], const EnTerm *t, uint32_t x0, typename AccOf<T>::t &acc) {
  const uint4 q = __ldg((const uint4 *)t);
  const T coef = en_coef<T>(q);
  const EnSign<T> sg(t, q.y);
  const T c = (__popc(x0 & q.x) & 1) ? -coef : coef;
  T s;
  if constexpr (PAIR) {
    if (q.y & 32u) {
      if (q.y & 16u) s = en_pairs<MC, 1, true, PAIR>(a, sg.get());
      else s = en_pairs<MC, 1, false, PAIR>(a, sg.get());
      acc.add(c * s);
      return;
    }
  }
  if (q.y & 16u) s = en_pairs<MC, 0, true, PAIR>(a, sg.get());
  else s = en_pairs<MC, 0, false, PAIR>(a, sg.get());
  acc.add(c * s);
}

// Block `jb` of energy job J: 2^J.rep_bits coset representatives of each of
// its class's groups, one per thread (blockDim.x = 2^J.rep_bits, at most
// EN_THREADS), 2^J.iter_bits times; thread 0 writes {sum_k c_k term_k, squared norm
// of the block} to out[0..1].  PAIR: FP32 states on a 16-byte boundary with a
// layout built for pairs.
template <typename T, bool PAIR, bool NC>
__device__ __forceinline__ void energy_block(const EnJob &J, uint32_t jb, const EnTables &tab, double *out) {
  typedef typename EnC<T>::t C;
  constexpr int N = EnAmp<T, PAIR>::N;
  uint32_t c = J.class_begin;
  const uint32_t ce = J.class_begin + J.n_classes;
  while (c + 1 < ce && tab.classes[c + 1].block_begin <= jb) c++;
  const EnClass K = tab.classes[c];
  const C *psi = (const C *)J.state;
  typename AccOf<T>::t acc, nrm;
  const uint32_t n_rep = 1u << (J.n - EN_RANK - (PAIR ? 1 : 0));
#pragma unroll 1
  for (uint32_t it = 0; it < (1u << J.iter_bits); it++) {
    const uint32_t j = ((((jb - K.block_begin) << J.iter_bits) + it) << J.rep_bits) | threadIdx.x;
    if (j >= n_rep) break;
#pragma unroll 1
    for (uint32_t g = K.group_begin; g < K.group_end; g++) {
      const uint4 b = __ldg((const uint4 *)(tab.groups + g)), w = __ldg((const uint4 *)(tab.groups + g) + 1);
      const uint32_t basis[EN_RANK] = {b.x, b.y, b.z, b.w};
      // zeros at the pivots, ascending (and at bit 0 of a pair)
      uint32_t x = PAIR ? j << 1 : j;
#pragma unroll
      for (int k = 0; k < EN_RANK; k++) {
        const uint32_t lo = x & ((1u << ((w.x >> (8 * k)) & 31u)) - 1u);
        x = ((x ^ lo) << 1) | lo;
      }
      const uint32_t x0 = x;
      C a[N];
#pragma unroll
      for (int k = 0; k < 16; k++) {  // Gray-code order, one XOR per address
        if (k) x ^= basis[(k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : 3];
        const int i = k ^ (k >> 1);
        if constexpr (PAIR) {
          const float4 v = en_ld<NC>((const float4 *)(psi + x));
          a[2 * i] = make_float2(v.x, v.y);
          a[2 * i + 1] = make_float2(v.z, v.w);
        } else {
          a[i] = en_ld<NC>(psi + x);
        }
      }
      if (w.w & EN_GROUP_NORM) nrm.add(en_norm(a));
      uint32_t t = w.y;
      // the first terms flip the basis masks, one each: straight-line code, a
      // uniform branch or two each (random Hamiltonians hold few others)
      const uint32_t ns = w.w >> EN_GROUP_SLOTS_SHIFT;
      if (ns > 0) en_slot<T, 1, PAIR>(a, tab.terms + t, x0, acc);
      if (ns > 1) en_slot<T, 2, PAIR>(a, tab.terms + t + 1, x0, acc);
      if (ns > 2) en_slot<T, 4, PAIR>(a, tab.terms + t + 2, x0, acc);
      if (ns > 3) en_slot<T, 8, PAIR>(a, tab.terms + t + 3, x0, acc);
      t += ns;
#pragma unroll 1
      for (; t < w.z; t++) {
        const uint4 q = __ldg((const uint4 *)(tab.terms + t));  // zm, code, coef
        const T coef = en_coef<T>(q);
        const EnSign<T> sg(tab.terms + t, q.y);
        en_pin(a);
        const T s = en_pairs_rt<T, PAIR>(a, q.y, sg);
        acc.add(((__popc(x0 & q.x) & 1) ? -coef : coef) * s);
      }
    }
  }
  __shared__ double en_red[2][8];
  const double e = en_warp_total(acc), nn = en_warp_total(nrm);
  const int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
  if (ln == 0) { en_red[0][w] = e; en_red[1][w] = nn; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double se = 0, sn = 0;
    for (uint32_t i = 0; i < blockDim.x / 32; i++) { se += en_red[0][i]; sn += en_red[1][i]; }
    out[0] = se;
    out[1] = sn;
  }
  __syncthreads();
}

}  // namespace qw
