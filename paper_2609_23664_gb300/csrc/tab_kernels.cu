// Stabilizer-tableau kernels (sm_103a), 64-bit words.
//
// The GPU keeps the INVERSE tableau T: for every generator X_i / Z_i of the
// initial frame it stores the Pauli string T(P) = C^-1 P C (C = circuit so
// far) as x-words, z-words and a sign, row-major, 2n rows in shared memory.
// A gate G of the circuit updates T by T'(P) = T(G^-1 P G), which is a
// product or a swap of ROWS (word-parallel over all qubits: W = ceil(n/64)
// words per half-row).  Measuring Z_a reads row T(Z_a): without an X part
// the outcome is its sign (deterministic); otherwise the outcome is random
// and the tableau is collapsed by conjugating every row with a few column
// operations in the initial frame (CNOTs, S^dagger, H, X), which leave
// |0...0> invariant up to the projected outcome.  This is the Heisenberg-
// picture formulation used by the stabilizer simulator the paper cites
// [gidney2021stim]; the CPU oracle uses the textbook forward tableau
// [aaronson2004stabilizer], so the two share no algorithm.  Measurement
// outcomes agree bit for bit: a deterministic outcome is fixed by the state,
// and a random one takes the outcome bit carried by the gate record.
//
// Row products keep Paulis in the Hermitian form (-1)^r i^{x.z} X^x Z^z:
// P1 P2 = (-1)^{r1+r2} i^{x1.z1 + x2.z2 - x3.z3 + 2 z1.x2 + e0} P3 where e0
// is an extra power of i (S: 3, S^dagger: 1) and the exponent is 0 or 2.
#include <cuda_runtime.h>

#include "qw_internal.h"

namespace qw {

// The kernel is compiled per row width W (64-bit words per half row, 1..10),
// so every word loop is unrolled.  CTAs of 128 threads serve registers up to
// 128 qubits, 256 up to 256, 512 above: one thread takes one row operation,
// and a layer has at most about 2n of them.
constexpr int TAB_MAX_W = (QW_TABLEAU_MAX_QUBITS + 63) / 64;
QW_HD constexpr int tab_threads(int W) { return W <= 2 ? 128 : (W <= 4 ? 256 : 512); }
// slots of a layer staged in shared memory at a time (at least n, so that a
// measurement layer fits)
QW_HD constexpr int tab_stage(int W) { return 2 * tab_threads(W); }
constexpr size_t TAB_SMEM_LIMIT = 227 * 1024 - 64;  // beside the kernel's static shared memory

// Shared memory of a tableau of n qubits with `stride` words per row and
// `bufs` slot staging buffers.
QW_HD inline size_t tab_smem_of(uint32_t n, uint32_t stride, uint32_t bufs) {
  const int W = (int)((n + 63) / 64);
  return (size_t)2 * n * stride * 8 + ((2 * n + 15) & ~15u) + ((n + 15) & ~15u) +
         (size_t)bufs * tab_stage(W) * sizeof(TabSlot) + 16;
}
// Row stride: 2W words and one more, so that word c of consecutive rows
// falls into different banks; without the pad where it does not fit (the
// largest registers).  Two staging buffers where they fit (a layer's slots
// are then staged while the previous layer runs, saving a barrier).
QW_HD inline uint32_t tab_stride(uint32_t n) {
  const uint32_t W = (n + 63) / 64;
  return tab_smem_of(n, 2 * W + 1, 1) <= TAB_SMEM_LIMIT ? 2 * W + 1 : 2 * W;
}
QW_HD inline uint32_t tab_bufs(uint32_t n) { return tab_smem_of(n, tab_stride(n), 2) <= TAB_SMEM_LIMIT ? 2u : 1u; }

template <int W>
struct TabSm {
  uint64_t *R;     // rows of `stride` words: x words 0..W-1, z words W..2W-1
  uint8_t *sign;   // rows
  uint8_t *pending;
  TabSlot *sl;     // tab_stage(W) staged slots of the current layer
  TabSlot *sl_alt; // the other staging buffer (== sl when single-buffered)
  uint32_t *any_random;
  uint32_t stride;
  __device__ __forceinline__ uint64_t *row(uint32_t r) const { return R + (size_t)r * stride; }
};

// Row product P1 P2: words into x3, z3, the power of i (mod 4) returned.
// The exponent x1.z1 + x2.z2 - x3.z3 + 2 z1.x2 is a sum over qubits of terms
// 0 or +-1 (nonzero where the two anticommute); they are added bit-sliced,
// two counter bits per word position, as the stabilizer simulator the paper
// cites does [gidney2021stim], so a product takes two population counts
// instead of four per word (POPC runs at a quarter of the logic rate).
template <int W>
__device__ __forceinline__ int tab_product(const uint64_t *r1, const uint64_t *r2, uint64_t *rd) {
  uint64_t c0 = 0, c1 = 0;
#pragma unroll
  for (int c = 0; c < W; c++) {
    const uint64_t x1 = r1[c], z1 = r1[W + c], x2 = r2[c], z2 = r2[W + c];
    const uint64_t x3 = x1 ^ x2, z3 = z1 ^ z2, xz = x1 & z2;
    const uint64_t anti = (x2 & z1) ^ xz;
    c1 ^= (c0 ^ x3 ^ z3 ^ xz) & anti;
    c0 ^= anti;
    rd[c] = x3;
    rd[W + c] = z3;
  }
  return __popcll(c0) + 2 * __popcll(c1);
}

// One unitary slot by one thread.
template <int W>
__device__ __forceinline__ void tab_slot(const TabSm<W> &S, const TabSlot &sl) {
  uint64_t *rd = S.row(sl.dst);
  if (sl.kind == T_PROD) {
    const int t = tab_product<W>(S.row(sl.s1), S.row(sl.s2), rd);
    S.sign[sl.dst] = S.sign[sl.s1] ^ S.sign[sl.s2] ^ (uint8_t)((((t + sl.flags) & 3) >> 1) & 1);
  } else if (sl.kind == T_SWAP2) {
    uint64_t *r2 = S.row(sl.s2);
#pragma unroll
    for (int c = 0; c < 2 * W; c++) {
      const uint64_t a0 = rd[c];
      rd[c] = r2[c];
      r2[c] = a0;
    }
    const uint8_t tmp = S.sign[sl.dst];
    S.sign[sl.dst] = S.sign[sl.s2];
    S.sign[sl.s2] = tmp;
  } else if (sl.kind == T_SIGN) {
    S.sign[sl.dst] ^= 1;
  }
}

// Random outcome of measuring Z_a with T(Z_a) = row sl.dst: p is the first
// qubit of its X part, S the others.  The collapse conjugates every row by
// CNOT(p -> q) for q in S, then S^dagger_p when T(Z_a) holds Z at p, then
// H_p and X_p^(outcome xor sign).  A row takes the whole sequence in one
// word-parallel visit: with x_p set, the CNOTs flip x on S, and their sign
//   sum over q in S with z_q of (x_q + 1 + z_p + number of earlier such q)
//     = |z & x & S| + k (1 + z_p) + k (k - 1) / 2,  k = |z & S|  (mod 2)
// where z_p itself takes the parity of k; the last two touch p's bits only.
// Two barriers per outcome and O(W) work per row.  (One CNOT at a time, as
// before, was O(n) dependent bit operations per row and nine barriers: a
// 100-qubit task with 100 random outcomes took 0.85 ms.)
template <int W>
__device__ void tab_collapse(const TabArgs &A, const TabSm<W> &S, const TabSlot &sl, uint32_t bits_base,
                             uint32_t out_base) {
  const uint32_t row = sl.dst;
  uint64_t Sx[W];
  uint64_t any = 0, zs = 0, k0 = 0, k1 = 0;
  uint32_t p = 0;
  int pw = -1;
  const uint64_t *rr = S.row(row);
#pragma unroll
  for (int w = 0; w < W; w++) {
    Sx[w] = rr[w];
    if (pw < 0 && Sx[w]) {
      pw = w;
      p = (uint32_t)__ffsll((long long)Sx[w]) - 1u;
      Sx[w] &= Sx[w] - 1;
      any = 1;
      zs = (rr[W + w] >> p) & 1ull;
    }
    const uint64_t t = rr[W + w] & Sx[w];
    k1 ^= k0 & t;
    k0 ^= t;
  }
  const uint8_t m = A.bits[bits_base + sl.aux] & 1;
  const uint8_t row_sign = S.sign[row];
  __syncthreads();
  if (!any) {  // became deterministic
    if (threadIdx.x == 0) {
      if (sl.aux2 != 0xFFFFFFFFu) A.outs[out_base + sl.aux2] = row_sign;
      if ((sl.flags & 1) && row_sign) S.sign[row] ^= 1;
    }
    __syncthreads();
    return;
  }
  if (threadIdx.x == 0) *S.any_random = 1u;
  // the row itself (x_p = 1, x = S elsewhere) after the CNOTs: z at p, sign
  const uint32_t kr = (uint32_t)(__popcll(k0) + 2 * __popcll(k1)) & 3u;
  const uint32_t zp_row = (uint32_t)zs ^ (kr & 1u);
  const uint32_t s_row = row_sign ^ ((kr + kr * (1u + (uint32_t)zs) + (kr * (kr - 1u)) / 2u) & 1u);
  const uint32_t bb = m ^ s_row;
  for (uint32_t r = threadIdx.x; r < A.rows; r += blockDim.x) {
    uint64_t *q = S.row(r);
    const uint64_t xw = q[pw], zw = q[W + pw];
    const uint32_t xp = (uint32_t)(xw >> p) & 1u;
    uint32_t zp = (uint32_t)(zw >> p) & 1u, sg = 0;
    uint64_t c0 = 0, c1 = 0, zx = 0;
#pragma unroll
    for (int w = 0; w < W; w++) {
      const uint64_t t = q[W + w] & Sx[w];
      if (xp) {
        const uint64_t x = q[w];
        c1 ^= c0 & t;
        zx ^= t & x;
        q[w] = x ^ Sx[w];
      }
      c0 ^= t;
    }
    if (xp) {
      const uint32_t k = (uint32_t)(__popcll(c0) + 2 * __popcll(c1)) & 3u;
      sg = (uint32_t)__popcll(zx) + k * (1u + zp) + (k * (k - 1u)) / 2u;
      zp ^= k & 1u;
    } else {
      zp ^= (uint32_t)__popcll(c0) & 1u;
    }
    if (zp_row) {  // S^dagger_p: Y -> X
      sg ^= xp & (zp ^ 1u);
      zp ^= xp;
    }
    sg ^= (xp & zp) ^ (bb & xp);  // H_p, then X_p when bb
    const uint64_t bit = 1ull << p;
    const uint64_t xn = q[pw];
    q[pw] = zp ? xn | bit : xn & ~bit;
    q[W + pw] = xp ? zw | bit : zw & ~bit;
    S.sign[r] ^= (uint8_t)(sg & 1u);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (sl.aux2 != 0xFFFFFFFFu) A.outs[out_base + sl.aux2] = m;
    if ((sl.flags & 1) && m) S.sign[row] ^= 1;
  }
  __syncthreads();
}

template <int W>
__device__ void tab_run_program(const TabArgs &A, const TabSm<W> &S, const TabProgram &P, uint32_t bits_base,
                                uint32_t out_base) {
  constexpr int NT = tab_threads(W);
  constexpr uint32_t STAGE = (uint32_t)tab_stage(W);
  // The first STAGE slots of the next layer are loaded into registers while
  // the current layer runs, and the descriptor of the layer after it as
  // well, so that neither staging a layer nor starting its prefetch waits on
  // a dependent global load.
  constexpr int PRE = (int)STAGE / NT;
  TabSlot pre[PRE];
  TabLayer Lnext = {}, Lafter = {};
  auto desc = [&](uint32_t li) {
    TabLayer d = {};
    if (li < P.n_layers) d = A.layers[P.layer_begin + li];
    return d;
  };
  // slots of layer li (descriptor Lnext) into pre[], descriptor of li + 1
  // into Lafter
  auto prefetch = [&](uint32_t li) {
    if (li >= P.n_layers) return;
    const uint32_t cn = min(STAGE, Lnext.n_slots);
#pragma unroll
    for (int k = 0; k < PRE; k++) {
      const uint32_t i = threadIdx.x + (uint32_t)k * NT;
      if (i < cn) pre[k] = A.slots[Lnext.slot_begin + i];
    }
    Lafter = desc(li + 1);
  };
  // with two staging buffers, a small layer writes the next layer's first
  // slots into the other buffer before its closing barrier
  TabSlot *sl_cur = S.sl, *sl_alt = S.sl_alt;
  const bool db = sl_alt != sl_cur;
  auto stage_next = [&](uint32_t li) {
    if (!db || li + 1 >= P.n_layers) return false;
    const uint32_t cn = min(STAGE, Lnext.n_slots);
#pragma unroll
    for (int k = 0; k < PRE; k++) {
      const uint32_t i = threadIdx.x + (uint32_t)k * NT;
      if (i < cn) sl_alt[i] = pre[k];
    }
    return true;
  };
  bool staged = false;  // this layer's slots are already in S.sl_alt
  Lnext = desc(0);
  prefetch(0);
  for (uint32_t li = 0; li < P.n_layers; li++) {
    const TabLayer cur = Lnext;
    Lnext = Lafter;
    if (staged) {
      TabSlot *t = sl_cur;
      sl_cur = sl_alt;
      sl_alt = t;
    } else {
      const uint32_t cn = min(STAGE, cur.n_slots);
#pragma unroll
      for (int k = 0; k < PRE; k++) {
        const uint32_t i = threadIdx.x + (uint32_t)k * NT;
        if (i < cn) sl_cur[i] = pre[k];
      }
      __syncthreads();
    }
    staged = false;
    if (cur.n_slots <= STAGE) prefetch(li + 1);
    if (!cur.is_measure) {
      // the layer's slots are staged in shared memory (one coalesced read
      // instead of a dependent global load per slot)
      for (uint32_t c0 = 0; c0 < cur.n_slots; c0 += STAGE) {
        const uint32_t cn = min(STAGE, cur.n_slots - c0);
        if (c0 > 0) {
          for (uint32_t i = threadIdx.x; i < cn; i += NT) sl_cur[i] = A.slots[cur.slot_begin + c0 + i];
          __syncthreads();
        }
        for (uint32_t i = threadIdx.x; i < cn; i += NT) tab_slot<W>(S, sl_cur[i]);
        if (cur.n_slots <= STAGE) staged = stage_next(li);
        __syncthreads();
      }
      if (cur.n_slots > STAGE) prefetch(li + 1);
    } else {
      // a measurement layer holds at most one slot per qubit, so all of its
      // slots are in the staging buffer already
      // phase 1: deterministic outcomes in parallel, random ones flagged
      int my_pending = 0;
      for (uint32_t si = threadIdx.x; si < cur.n_slots; si += NT) {
        const TabSlot sl = sl_cur[si];
        const uint64_t *rr = S.row(sl.dst);
        uint64_t v = 0;
#pragma unroll
        for (int c = 0; c < W; c++) v |= rr[c];
        if (v == 0) {
          const uint8_t oc = S.sign[sl.dst];
          if (sl.aux2 != 0xFFFFFFFFu) A.outs[out_base + sl.aux2] = oc;
          if ((sl.flags & 1) && oc) S.sign[sl.dst] ^= 1;
          S.pending[si] = 0;
        } else {
          S.pending[si] = 1;
          my_pending = 1;
        }
      }
      staged = stage_next(li);
      // phase 2 (only when some outcome is random): one at a time, in
      // program order
      if (__syncthreads_or(my_pending)) {
        for (uint32_t si = 0; si < cur.n_slots; si++)
          if (S.pending[si]) tab_collapse<W>(A, S, sl_cur[si], bits_base, out_base);
        __syncthreads();
      }
    }
  }
}

template <int W>
__global__ void __launch_bounds__(tab_threads(W), W <= 4 ? 2 : 1) tab_kernel(TabArgs A) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ uint32_t s_any_random;
  if (A.run_if && *A.run_if == 0u) return;  // uniform over the grid
  const uint32_t rows = A.rows;
  TabSm<W> S;
  S.any_random = &s_any_random;
  if (threadIdx.x == 0) s_any_random = 0u;
  S.stride = tab_stride(A.n);
  S.sl = (TabSlot *)smraw;
  S.sl_alt = tab_bufs(A.n) == 2 ? S.sl + tab_stage(W) : S.sl;
  S.R = (uint64_t *)(S.sl_alt + tab_stage(W));
  S.sign = (uint8_t *)(S.R + (size_t)rows * S.stride);
  S.pending = S.sign + ((rows + 15) & ~15u);
  const uint32_t nwords = rows * 2 * W;
  const TabTaskDesc T = A.tasks[blockIdx.x];
  if (T.init_rows) {
    const uint8_t *init_sign = (const uint8_t *)(T.init_rows + nwords);
    for (uint32_t i = threadIdx.x; i < nwords; i += blockDim.x) S.row(i / (2 * W))[i % (2 * W)] = __ldg(T.init_rows + i);
    for (uint32_t i = threadIdx.x; i < rows; i += blockDim.x) S.sign[i] = __ldg(init_sign + i);
  } else {
    for (uint32_t i = threadIdx.x; i < nwords; i += blockDim.x) {
      const uint32_t r = i / (2 * W), c = i % (2 * W);
      // row r < n: X_r (bit r in the x half); row n+i: Z_i (bit i in the z half)
      uint64_t v = 0;
      if (r < A.n) {
        if (c < W && (r >> 6) == c) v = 1ull << (r & 63);
      } else {
        const uint32_t q = r - A.n;
        if (c >= W && (q >> 6) == c - W) v = 1ull << (q & 63);
      }
      S.row(r)[c] = v;
    }
    for (uint32_t i = threadIdx.x; i < rows; i += blockDim.x) S.sign[i] = 0;
  }
  __syncthreads();
  for (uint32_t si = 0; si < T.n_segs; si++) {
    const TabSegment sg = A.segs[T.seg_begin + si];
    const TabProgram P = A.progs[sg.prog];
    tab_run_program<W>(A, S, P, sg.bit_base, T.out_base + sg.out_base);
  }
  __syncthreads();
  if (A.rand_any && threadIdx.x == 0) A.rand_any[blockIdx.x] = s_any_random;
  if (T.out_rows) {
    for (uint32_t i = threadIdx.x; i < nwords; i += blockDim.x) T.out_rows[i] = S.row(i / (2 * W))[i % (2 * W)];
    for (uint32_t i = threadIdx.x; i < rows; i += blockDim.x) T.out_sign[i] = S.sign[i];
  }
}

typedef void (*TabKernel)(TabArgs);
static TabKernel tab_kernel_of(uint32_t W) {
  static const TabKernel k[TAB_MAX_W] = {tab_kernel<1>, tab_kernel<2>, tab_kernel<3>, tab_kernel<4>, tab_kernel<5>,
                                         tab_kernel<6>, tab_kernel<7>, tab_kernel<8>, tab_kernel<9>, tab_kernel<10>};
  static_assert(TAB_MAX_W == 10, "one kernel per row width");
  return k[W - 1];
}

size_t tab_smem_bytes(uint32_t n) { return tab_smem_of(n, tab_stride(n), tab_bufs(n)); }

// every register of a width fits below the 227 KB opt-in limit together with
// the kernel's static shared memory
cudaError_t tab_init_attrs() {
  for (uint32_t W = 1; W <= (uint32_t)TAB_MAX_W; W++) {
    const cudaError_t e = cudaFuncSetAttribute((const void *)tab_kernel_of(W),
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAB_SMEM_LIMIT);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void launch_tab(const TabArgs &a, uint32_t n_tasks, void *stream) {
  if (n_tasks == 0) return;
  tab_kernel_of(a.W)<<<n_tasks, tab_threads((int)a.W), tab_smem_bytes(a.n), (cudaStream_t)stream>>>(a);
}

}  // namespace qw
