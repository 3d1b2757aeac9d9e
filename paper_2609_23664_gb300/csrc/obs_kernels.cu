// Observables: Pauli-sum energy and computational-basis sampling (sm_103a).
//
// Energy (the repeated expectation evaluation of the VQE workloads, Sec. V,
// Table III): E = sum_k c_k <psi|P_k|psi> / <psi|psi> with
// P|x> = i^{#Y} (-1)^{popc(x&z)} |x^m>, evaluated in groups of terms on the
// cosets of their flip masks (energy_block.cuh).  Products are FP32; every
// thread keeps a double-float (two-sum) accumulator across groups, and block
// and final reductions are FP64, in a fixed order.
//
// Sampling: p_x = |psi_x|^2 summed in FP64 into a CDF that is never written
// out: per 4096-amplitude block a lane sums 128 contiguous probabilities and
// the 32 lane sums are chained in lane order; block offsets are an FP64 scan;
// a shot finds its block by binary search and its index by rescanning that
// block with the additions of the block sums.
#include <cuda_runtime.h>

#include <algorithm>
#include <unordered_map>

#include "energy_block.cuh"
#include "qw_internal.h"

namespace qw {

template <typename T> struct V2o;
template <> struct V2o<float> { typedef float2 t; };
template <> struct V2o<double> { typedef double2 t; };

// ---------------------------------------------------------------------------
// energy layout (host)
// ---------------------------------------------------------------------------
EnLayout build_energy_layout(const qw_pauli_term *terms, uint64_t n_terms, uint32_t n, bool fp64, bool pair,
                             uint32_t rep_bits, uint32_t max_class_bits) {
  const uint32_t amp_bytes = fp64 ? 16u : 8u;
  const uint32_t low = pair ? 1u : 0u;  // bit 0 is a direction of every pair layout's cosets
  EnLayout L;
  L.rep_bits = rep_bits;
  // chunks of at most EN_CHUNK_BYTES, so that the chunk pair a class reads
  // stays in L2, and large enough for a coset's in-chunk pivots
  uint32_t chunk_bits = n;
  while (chunk_bits > (uint32_t)(EN_RANK + 8) && n - chunk_bits < max_class_bits &&
         ((uint64_t)amp_bytes << chunk_bits) > EN_CHUNK_BYTES)
    chunk_bits--;
  const uint32_t u = n - chunk_bits;
  // per class: distinct masks (but for a pair's bit 0) in order of appearance, each with its terms
  struct Flip {
    uint32_t mask;
    std::vector<uint64_t> terms;
    bool used = false;
  };
  std::vector<std::vector<Flip>> by_class(1u << u);
  std::vector<std::unordered_map<uint32_t, size_t>> at(1u << u);
  for (uint64_t k = 0; k < n_terms; k++) {
    const uint32_t m = (uint32_t)terms[k].xmask & ~low, d = (uint32_t)((uint64_t)m >> chunk_bits);
    auto it = at[d].emplace(m, by_class[d].size());
    if (it.second) by_class[d].push_back(Flip{m, {}});
    by_class[d][it.first->second].terms.push_back(k);
  }
  L.iter_bits = en_iter_bits(n, rep_bits);
  const uint32_t reps = n - EN_RANK - low;
  const uint32_t blocks = reps > rep_bits + L.iter_bits ? 1u << (reps - rep_bits - L.iter_bits) : 1u;
  uint32_t blk = 0;
  for (uint32_t d = 0; d < (1u << u); d++) {
    std::vector<Flip> &F = by_class[d];
    if (d != 0 && F.empty()) continue;
    EnClass c{};
    c.group_begin = (uint32_t)L.groups.size();
    size_t next = 0;
    bool first = true;
    for (;;) {
      while (next < F.size() && F[next].used) next++;
      if (next == F.size() && !(d == 0 && first)) break;
      EnGroup g{};
      uint32_t ech[EN_RANK] = {0}, rank = 0;  // echelon form of the basis (distinct leading bits)
      auto reduce = [&](uint32_t v) {
        for (uint32_t i = 0; i < rank; i++) v = std::min(v, v ^ ech[i]);
        return v;
      };
      auto push = [&](uint32_t v) {
        const uint32_t r = reduce(v);
        if (!r) return false;
        g.basis[rank] = v;
        // kept descending, so that reducing in order clears leading bits once
        uint32_t i = rank++;
        for (; i > 0 && ech[i - 1] < r; i--) ech[i] = ech[i - 1];
        ech[i] = r;
        return true;
      };
      for (size_t i = next; i < F.size() && rank < (uint32_t)EN_RANK; i++)
        if (!F[i].used && F[i].mask) push(F[i].mask);
      // fewer masks than EN_RANK: unit vectors, from bit 5 up so that a
      // warp's representatives stay consecutive
      for (uint32_t i = 0; i < chunk_bits && rank < (uint32_t)EN_RANK; i++)
        push((1u << ((i + 5) % chunk_bits)) & ~low);
      uint32_t piv[EN_RANK];
      for (uint32_t i = 0; i < (uint32_t)EN_RANK; i++) piv[i] = 31u - (uint32_t)__builtin_clz(ech[EN_RANK - 1 - i]);
      for (uint32_t i = 0; i < (uint32_t)EN_RANK; i++) g.pivots |= piv[i] << (8 * i);
      if (d == 0 && first) g.flags |= EN_GROUP_NORM;
      // every term whose mask lies in the span
      g.term_begin = (uint32_t)L.terms.size();
      auto put = [&](uint64_t k, uint32_t comb) {
        const uint64_t m = terms[k].xmask, z = terms[k].zmask;
        const int y = __builtin_popcountll(m & z);
        EnTerm t{};
        t.zm = (uint32_t)z;
        t.code = comb | ((uint32_t)(y & 1) << 4);
        if (m & low) t.code |= 32u;
        float sg[EN_RANK + 1];
        uint32_t ns = 0;
        // the highest flipped direction has no sign: a basis vector, bit 0
        // of a pair, or none
        const int top = comb ? 31 - __builtin_clz(comb) : ((m & low) ? -1 : EN_RANK);
        if (pair && top != -1) sg[ns++] = (z & 1u) ? -1.f : 1.f;
        for (int i = 0; i < EN_RANK; i++) {
          const uint32_t par = (uint32_t)(__builtin_popcountll(g.basis[i] & z) & 1);
          t.code |= par << (8 + i);
          if (i != top) sg[ns++] = par ? -1.f : 1.f;
        }
        if (ns == EN_RANK + 1 && sg[EN_RANK] < 0) t.code |= EN_LAST_SIGN;
        for (uint32_t i = 0; i < std::min<uint32_t>(ns, EN_RANK); i++) t.sign[i] = sg[i];
        const double coef = terms[k].coef * (((y & 3) == 0 || (y & 3) == 3) ? 1.0 : -1.0) * (m ? 2.0 : 1.0);
        if (amp_bytes == 16) t.coef64 = coef;
        else t.coef32 = (float)coef;
        L.terms.push_back(t);
      };
      auto flip_of = [&](uint32_t comb) -> Flip * {
        uint32_t m = 0;
        for (uint32_t i = 0; i < (uint32_t)EN_RANK; i++)
          if ((comb >> i) & 1u) m ^= g.basis[i];
        auto it = at[d].find(m);
        return (it == at[d].end() || F[it->second].used) ? nullptr : &F[it->second];
      };
      // one term of each basis mask that is a term's mask (the first ones of
      // the basis) first
      uint32_t slots = 0;
      while (slots < (uint32_t)EN_RANK) {
        const Flip *f = flip_of(1u << slots);
        if (!f) break;
        put(f->terms[0], 1u << slots++);
      }
      g.flags |= slots << EN_GROUP_SLOTS_SHIFT;
      for (uint32_t comb = (d == 0 && first) ? 0u : 1u; comb < (1u << EN_RANK); comb++) {
        Flip *f = flip_of(comb);
        if (!f) continue;
        f->used = true;
        const bool slotted = comb && (comb & (comb - 1)) == 0 && comb < (1u << slots);
        for (size_t i = slotted ? 1 : 0; i < f->terms.size(); i++) put(f->terms[i], comb);
      }
      g.term_end = (uint32_t)L.terms.size();
      L.groups.push_back(g);
      first = false;
    }
    c.group_end = (uint32_t)L.groups.size();
    c.block_begin = blk;
    blk += blocks;
    L.classes.push_back(c);
  }
  L.n_blocks = blk;
  return L;
}

// ---------------------------------------------------------------------------
// energy kernels
// ---------------------------------------------------------------------------
// one CTA per block; the block's job is found by binary search.  The 64
// registers of an FP32 pair coset leave five CTAs of 128 threads per SM (96
// registers): 64 24-qubit states, 200 terms: 27.7 ms, against 30.9 ms with
// four CTAs, 33.6 ms with six (which spill), 31.6 ms with two of 256 threads,
// 33.1 ms for cosets of 16 amplitudes on 32 warps per SM (bound by
// instruction issue) and 47 ms term by term.  A two-sum per term instead of
// one per group makes it 28.6 ms and the energy of a random state err by
// 5.3e-8 of its typical size instead of 6.6e-8 (6.5e-8 term by term).
template <typename T, bool PAIR>
__global__ void __launch_bounds__(EN_THREADS, sizeof(T) == 8 ? 4 : PAIR ? 5 : 8)
energy_kernel(EnTables t, uint32_t n_jobs) {
  const uint32_t gb = blockIdx.x;
  uint32_t lo = 0, hi = n_jobs;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (t.jobs[mid].block_begin <= gb) lo = mid; else hi = mid;
  }
  const EnJob J = t.jobs[lo];
  energy_block<T, PAIR, true>(J, gb - J.block_begin, t, t.partials + 2 * (size_t)gb);
}

// one CTA per job; fixed summation order.  (One warp per job took 2.2 ms for
// the 262144 partials of a 26-qubit state, as long as the energy kernel.)
constexpr int EN_RED_THREADS = 256;
__global__ void __launch_bounds__(EN_RED_THREADS)
energy_reduce_kernel(const EnJob *__restrict__ jobs, const double2 *__restrict__ partials) {
  const EnJob J = jobs[blockIdx.x];
  double se = 0, sn = 0;
#pragma unroll 8
  for (uint32_t i = threadIdx.x; i < J.n_blocks; i += EN_RED_THREADS) {
    const double2 v = partials[J.block_begin + i];
    se += v.x;
    sn += v.y;
  }
  __shared__ double red[2][EN_RED_THREADS / 32];
  se = en_warp_sum(se);
  sn = en_warp_sum(sn);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = se;
    red[1][threadIdx.x >> 5] = sn;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    se = sn = 0;
    for (int i = 0; i < EN_RED_THREADS / 32; i++) {
      se += red[0][i];
      sn += red[1][i];
    }
    J.out[0] = se / sn;
    J.out[1] = sn;
  }
}

void launch_energy_reduce(const EnJob *jobs, uint32_t n_jobs, const double *partials, void *stream) {
  if (n_jobs == 0) return;
  energy_reduce_kernel<<<n_jobs, EN_RED_THREADS, 0, (cudaStream_t)stream>>>(jobs, (const double2 *)partials);
}

void launch_energy(bool fp64, bool pair, const EnTables &t, uint32_t n_jobs, uint32_t total_blocks, uint32_t rep_bits,
                   void *stream) {
  if (n_jobs == 0 || total_blocks == 0) return;
  cudaStream_t s = (cudaStream_t)stream;
  const unsigned threads = 1u << rep_bits;
  if (fp64)
    energy_kernel<double, false><<<total_blocks, threads, 0, s>>>(t, n_jobs);
  else if (pair)
    energy_kernel<float, true><<<total_blocks, threads, 0, s>>>(t, n_jobs);
  else
    energy_kernel<float, false><<<total_blocks, threads, 0, s>>>(t, n_jobs);
  launch_energy_reduce(t.jobs, n_jobs, t.partials, stream);
}

// ---------------------------------------------------------------------------
// sampling kernels
// ---------------------------------------------------------------------------
constexpr int SMP_PER_LANE = (1 << SMP_BLOCK_BITS) / 32;  // 128


__device__ __forceinline__ uint32_t find_source(const SmpSource *srcs, uint32_t n_src, uint32_t gb) {
  uint32_t lo = 0, hi = n_src;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (srcs[mid].block_begin <= gb) lo = mid; else hi = mid;
  }
  return lo;
}

// Running sum of one lane's probabilities in index order.  FP64 states add
// in FP64; FP32 states add their FP32 probabilities in double-float (a
// two-sum of the high part, about 2^-44 relative, FP32 arithmetic at 64
// times GB300's FP64 rate) and hand the sum on in FP64.  The lane sums and
// the element scan of the shot kernel make the same additions in the same
// order, so their partial sums agree bit for bit.
template <typename T> struct SmpAcc;
template <> struct SmpAcc<double> {
  double v = 0.0;
  __device__ __forceinline__ void add(double p) { v += p; }
  __device__ __forceinline__ double value() const { return v; }
  typedef double raw;  // the running sum as it is kept in shared memory
  __device__ __forceinline__ raw get() const { return v; }
  static __device__ __forceinline__ double value_of(const raw &r) { return r; }
};
template <> struct SmpAcc<float> {
  DFAcc a;
  __device__ __forceinline__ void add(float p) { a.add(p); }
  __device__ __forceinline__ double value() const { return a.value(); }
  typedef float2 raw;
  __device__ __forceinline__ raw get() const { return make_float2(a.hi, a.lo); }
  static __device__ __forceinline__ double value_of(const raw &r) { return (double)r.x + (double)r.y; }
};
__device__ __forceinline__ float prob32(const float2 &v) { return fmaf(v.x, v.x, v.y * v.y); }
__device__ __forceinline__ double prob32(const double2 &v) { return fma(v.x, v.x, v.y * v.y); }

// lane-serial sum of the lane's 128 probabilities, lane sums chained in order
template <typename T>
__device__ void lane_sums(const typename V2o<T>::t *psi, uint32_t dim, uint32_t off, int ln,
                          double *lane_sum, int32_t *lane_last) {
  SmpAcc<T> s;
  int32_t last = -1;
  const uint32_t b0 = off + (uint32_t)ln * SMP_PER_LANE;
  if constexpr (sizeof(T) == 4) {
    // FP32, whole segment of a state on a 16-byte boundary: two amplitudes per load
    if (b0 + SMP_PER_LANE <= dim && ((uintptr_t)psi & 15u) == 0) {
      const float4 *q = reinterpret_cast<const float4 *>(psi + b0);
#pragma unroll 8
      for (int i = 0; i < SMP_PER_LANE / 2; i++) {
        const float4 v = q[i];
        const float p0 = fmaf(v.x, v.x, v.y * v.y), p1 = fmaf(v.z, v.z, v.w * v.w);
        s.add(p0);
        if (p0 > 0) last = ln * SMP_PER_LANE + 2 * i;
        s.add(p1);
        if (p1 > 0) last = ln * SMP_PER_LANE + 2 * i + 1;
      }
      *lane_sum = s.value();
      *lane_last = last;
      return;
    }
  }
  for (int i = 0; i < SMP_PER_LANE; i++) {
    const uint32_t x = b0 + i;
    if (x < dim) {
      const auto p = prob32(psi[x]);
      s.add(p);
      if (p > 0) last = ln * SMP_PER_LANE + i;
    }
  }
  *lane_sum = s.value();
  *lane_last = last;
}

// chained (sequential in lane order) inclusive scan: S_l = S_{l-1} + s_l
__device__ __forceinline__ double chain_scan(double s, int ln) {
  double S = (ln == 0) ? s : 0.0;
  for (int l = 1; l < 32; l++) {
    const double prev = __shfl_sync(0xffffffffu, S, l - 1);
    if (ln == l) S = prev + s;
  }
  return S;
}

// The lane sums of a whole FP32 block on a 16-byte boundary, read in memory
// order: 16 amplitudes of every lane's segment at a time (32 lines of 128
// bytes) are copied to shared memory, eight lanes to a line, two such pieces
// in flight, and each lane then adds its own row (rows padded to 144 bytes:
// a quarter warp's 16-byte reads cover every bank).  Each lane reading its
// segment directly touches 32 lines per load instruction, which the L1 takes
// one per clock (4.2 TB/s).
constexpr int SMP_PIECE = 16, SMP_ROW = SMP_PIECE * 8 + 16;  // amplitudes, padded bytes
struct SmpStage {
  unsigned char b[2][32 * SMP_ROW];
};
__device__ __forceinline__ void smp_fetch(SmpStage &st, const float2 *blk, int piece, int ln) {
  const uint32_t sm = (uint32_t)__cvta_generic_to_shared(st.b[piece & 1]);
#pragma unroll
  for (int u = 0; u < 8; u++) {
    const int r = u * 4 + (ln >> 3), c = ln & 7;
    const float2 *g = blk + r * SMP_PER_LANE + piece * SMP_PIECE + 2 * c;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sm + (uint32_t)(r * SMP_ROW + c * 16)), "l"(g)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void lane_sums_staged(SmpStage &st, const float2 *blk, int ln, double *lane_sum,
                                                 int32_t *lane_last) {
  constexpr int PIECES = SMP_PER_LANE / SMP_PIECE;
  SmpAcc<float> s;
  int32_t last = -1;
  smp_fetch(st, blk, 0, ln);
#pragma unroll 1
  for (int p = 0; p < PIECES; p++) {
    if (p + 1 < PIECES) {
      smp_fetch(st, blk, p + 1, ln);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncwarp();
    const float4 *q = (const float4 *)(st.b[p & 1] + ln * SMP_ROW);
#pragma unroll
    for (int i = 0; i < SMP_PIECE / 2; i++) {
      const float4 v = q[i];
      const float p0 = fmaf(v.x, v.x, v.y * v.y), p1 = fmaf(v.z, v.z, v.w * v.w);
      const int at = ln * SMP_PER_LANE + p * SMP_PIECE + 2 * i;
      s.add(p0);
      if (p0 > 0) last = at;
      s.add(p1);
      if (p1 > 0) last = at + 1;
    }
    __syncwarp();  // the piece is overwritten by the fetch after next
  }
  *lane_sum = s.value();
  *lane_last = last;
}

// One warp per block; the lane sums of the CTA's blocks are chained by one
// thread per block, all of them at once (the 31 dependent FP64 adds of a
// chain cost a warp the same for one block as for 32, and at 1/64 of the
// FP32 rate they showed beside the loads).
constexpr int SMP_WARPS = 4;
template <typename T>
__global__ void __launch_bounds__(SMP_WARPS * 32)
smp_blocksum_kernel(const SmpSource *__restrict__ srcs, uint32_t n_src, uint32_t total, double *bsum, int32_t *blast) {
  typedef typename V2o<T>::t C;
  __shared__ double ls[SMP_WARPS][33];
  __shared__ int32_t ll[SMP_WARPS];
  __shared__ __align__(16) unsigned char stage[sizeof(T) == 4 ? SMP_WARPS * sizeof(SmpStage) : 16];
  const uint32_t w = threadIdx.x / 32, gb = blockIdx.x * SMP_WARPS + w;
  const int ln = threadIdx.x & 31;
  if (gb < total) {
    const SmpSource S = srcs[find_source(srcs, n_src, gb)];
    const uint32_t blk = gb - S.block_begin;
    const C *psi = (const C *)S.state;
    double s;
    int32_t last;
    bool done = false;
    if constexpr (sizeof(T) == 4) {
      if (S.n >= (uint32_t)SMP_BLOCK_BITS && ((uintptr_t)psi & 15u) == 0) {
        lane_sums_staged(((SmpStage *)stage)[w], psi + ((size_t)blk << SMP_BLOCK_BITS), ln, &s, &last);
        done = true;
      }
    }
    if (!done) lane_sums<T>(psi, 1u << S.n, blk << SMP_BLOCK_BITS, ln, &s, &last);
    ls[w][ln] = s;
    last = __reduce_max_sync(0xffffffffu, last);
    if (ln == 0) ll[w] = last;
  }
  __syncthreads();
  const uint32_t b = blockIdx.x * SMP_WARPS + threadIdx.x;
  if (threadIdx.x < SMP_WARPS && b < total) {
    double S = ls[threadIdx.x][0];
    for (int l = 1; l < 32; l++) S = S + ls[threadIdx.x][l];
    bsum[b] = S;
    blast[b] = ll[threadIdx.x];
  }
}

// one CTA per source: boff[b] = sum of the blocks before b, the entry after
// the last block is the total.  Each thread adds a run of blocks in order,
// the runs' sums are scanned across the CTA.  (One thread per source, block
// by block, took 1.87 ms for the 16384 blocks of 26 qubits.)  The scan rounds
// in another order than the runs do, so the offsets may step by an ulp from
// one run to the next: an empty block takes the offset of the next block that
// is not empty, so that no target falls into it.
constexpr int SMP_OFF_THREADS = 256;
__global__ void __launch_bounds__(SMP_OFF_THREADS)
smp_offsets_kernel(const SmpSource *__restrict__ srcs, const double *__restrict__ bsum,
                   const int32_t *__restrict__ blast, double *boff, int64_t *lastnz) {
  const uint32_t s = blockIdx.x, t = threadIdx.x;
  const SmpSource S = srcs[s];
  double *o = boff + S.block_begin + s;  // n_blocks + 1 entries per source
  const uint32_t run = (S.n_blocks + SMP_OFF_THREADS - 1) / SMP_OFF_THREADS;
  const uint32_t b0 = min(t * run, S.n_blocks), b1 = min(b0 + run, S.n_blocks);
  double acc = 0;
  int64_t last = -1;
#pragma unroll 8
  for (uint32_t b = b0; b < b1; b++) {
    acc = acc + bsum[S.block_begin + b];
    const int32_t l = blast[S.block_begin + b];
    if (l >= 0) last = ((int64_t)b << SMP_BLOCK_BITS) + l;
  }
  // exclusive scan of the runs' sums: within a warp, then of the warps
  __shared__ double wsum[SMP_OFF_THREADS / 32];
  __shared__ int64_t wlast[SMP_OFF_THREADS / 32];
  __shared__ unsigned wfilled[SMP_OFF_THREADS / 32];
  __shared__ double base[SMP_OFF_THREADS + 1];  // offset of each run, the total
  double incl = acc;
#pragma unroll
  for (int d = 1; d < 32; d *= 2) {
    const double up = __shfl_up_sync(0xffffffffu, incl, d);
    if ((t & 31) >= (uint32_t)d) incl = incl + up;
  }
  double excl = __shfl_up_sync(0xffffffffu, incl, 1);
  if ((t & 31) == 0) excl = 0;
  const uint32_t end = last >= 0 ? (uint32_t)(last >> SMP_BLOCK_BITS) + 1 : b0;  // past the run's last filled block
  const unsigned filled = __ballot_sync(0xffffffffu, last >= 0);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, d));
  if ((t & 31) == 31) wsum[t >> 5] = incl;
  if ((t & 31) == 0) {
    wlast[t >> 5] = last;
    wfilled[t >> 5] = filled;
  }
  __syncthreads();
  double before = 0;
  for (uint32_t w = 0; w < (t >> 5); w++) before = before + wsum[w];
  acc = before + excl;
  base[t] = acc;
  if (t == SMP_OFF_THREADS - 1) base[SMP_OFF_THREADS] = before + incl;
  __syncthreads();
#pragma unroll 8
  for (uint32_t b = b0; b < end; b++) {
    o[b] = acc;
    acc = acc + bsum[S.block_begin + b];
  }
  if (end < b1) {  // the run ends with empty blocks: the next filled run's offset
    uint32_t w = t >> 5;
    unsigned m = (t & 31) == 31 ? 0u : wfilled[w] >> ((t & 31) + 1) << ((t & 31) + 1);
    while (!m && ++w < SMP_OFF_THREADS / 32) m = wfilled[w];
    const double next = base[m ? 32 * w + (uint32_t)__ffs(m) - 1 : SMP_OFF_THREADS];
    for (uint32_t b = end; b < b1; b++) o[b] = next;
  }
  if (t == SMP_OFF_THREADS - 1) {
    o[S.n_blocks] = base[SMP_OFF_THREADS];
    for (int w = 0; w < SMP_OFF_THREADS / 32; w++) last = max(last, wlast[w]);
    lastnz[s] = last;
  }
}

// One warp per shot: binary search for its block, then the block's lane sums,
// then the running sums of the lane's 128 probabilities.  Those are FP32 pairs
// (FP64 for FP64 states), formed by that lane alone and left in shared
// memory; the 32 lanes then compare four of them each with the target in
// FP64 (compared one by one by a single lane, 128 times three FP64 adds at
// 1/64 of the FP32 rate took 145 of the 177 us of 4096 shots).
constexpr int SMP_SHOT_WARPS = 4;
template <typename T>
__global__ void __launch_bounds__(SMP_SHOT_WARPS * 32)
smp_shot_kernel(const SmpSource *__restrict__ srcs, const SmpShot *__restrict__ shots,
                uint32_t n_shots, const double *boff, const int64_t *lastnz) {
  typedef typename V2o<T>::t C;
  __shared__ typename SmpAcc<T>::raw run[SMP_SHOT_WARPS][SMP_PER_LANE];
  const uint32_t w = threadIdx.x / 32, sh = blockIdx.x * SMP_SHOT_WARPS + w;
  const int ln = threadIdx.x & 31;
  if (sh >= n_shots) return;  // whole warps; no block-wide barrier below
  const SmpShot Q = shots[sh];
  const SmpSource S = srcs[Q.source];
  const double *o = boff + S.block_begin + Q.source;
  const double total = o[S.n_blocks];
  const double target = Q.u * total;
  const uint32_t dim = 1u << S.n;
  if (!(target < total)) {
    if (ln == 0) *Q.out = (uint64_t)lastnz[Q.source];
    return;
  }
  // first block whose end exceeds target
  uint32_t lo = 0, hi = S.n_blocks - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (o[mid + 1] > target) hi = mid; else lo = mid + 1;
  }
  const uint32_t blk = lo;
  const double ob = o[blk];
  const C *psi = (const C *)S.state;
  double s;
  int32_t last;
  lane_sums<T>(psi, dim, blk << SMP_BLOCK_BITS, ln, &s, &last);
  const double incl = chain_scan(s, ln);
  const double excl = __shfl_up_sync(0xffffffffu, incl, 1);
  const double lane_start = (ln == 0) ? 0.0 : excl;
  const unsigned hit = __ballot_sync(0xffffffffu, ob + incl > target);
  if (hit == 0) {
    // the rounding of the block offsets left the target at the block's end:
    // its last outcome of nonzero probability
    last = __reduce_max_sync(0xffffffffu, last);
    if (ln == 0)
      *Q.out = last >= 0 ? ((uint64_t)blk << SMP_BLOCK_BITS) + (uint64_t)last : (uint64_t)lastnz[Q.source];
    return;
  }
  const int L = __ffs(hit) - 1;
  const uint32_t b0 = (blk << SMP_BLOCK_BITS) + (uint32_t)L * SMP_PER_LANE;
  const uint32_t cnt = min((uint32_t)SMP_PER_LANE, dim > b0 ? dim - b0 : 0u);
  if (ln == L) {
    SmpAcc<T> pre;
    for (uint32_t i = 0; i < cnt; i++) {
      pre.add(prob32(psi[b0 + i]));
      run[w][i] = pre.get();
    }
  }
  const double from = __shfl_sync(0xffffffffu, lane_start, L);
  const int32_t lane_last = __shfl_sync(0xffffffffu, last, L);
  __syncwarp();
  for (uint32_t c = 0; c < cnt; c += 32) {
    const uint32_t i = c + (uint32_t)ln;
    const bool over = i < cnt && ob + (from + SmpAcc<T>::value_of(run[w][i])) > target;
    const unsigned m = __ballot_sync(0xffffffffu, over);
    if (m) {
      if (ln == 0) *Q.out = (uint64_t)b0 + c + (uint32_t)(__ffs(m) - 1);
      return;
    }
  }
  // no running sum exceeds the target: the lane's last nonzero outcome
  if (ln == 0)
    *Q.out = lane_last >= 0 ? ((uint64_t)blk << SMP_BLOCK_BITS) + (uint64_t)lane_last
                            : (uint64_t)b0 + SMP_PER_LANE - 1;
}

void launch_sampling(bool fp64, const SmpSource *srcs, uint32_t n_src, uint32_t total_blocks,
                     double *bsum, int32_t *blast, double *boff, int64_t *lastnz,
                     const SmpShot *shots, uint32_t n_shots, void *stream) {
  if (n_src == 0) return;
  cudaStream_t s = (cudaStream_t)stream;
  const uint32_t g1 = (total_blocks + SMP_WARPS - 1) / SMP_WARPS;
  if (fp64)
    smp_blocksum_kernel<double><<<g1, SMP_WARPS * 32, 0, s>>>(srcs, n_src, total_blocks, bsum, blast);
  else
    smp_blocksum_kernel<float><<<g1, SMP_WARPS * 32, 0, s>>>(srcs, n_src, total_blocks, bsum, blast);
  smp_offsets_kernel<<<n_src, SMP_OFF_THREADS, 0, s>>>(srcs, bsum, blast, boff, lastnz);
  if (n_shots == 0) return;
  const uint32_t g3 = (n_shots + SMP_SHOT_WARPS - 1) / SMP_SHOT_WARPS;
  if (fp64)
    smp_shot_kernel<double><<<g3, SMP_SHOT_WARPS * 32, 0, s>>>(srcs, shots, n_shots, boff, lastnz);
  else
    smp_shot_kernel<float><<<g3, SMP_SHOT_WARPS * 32, 0, s>>>(srcs, shots, n_shots, boff, lastnz);
}

}  // namespace qw
