// Pauli-sum energy of a caller-owned device state without any device
// allocation: qw_sv_energy_noalloc_dev.
//
// Some callers cannot allocate device memory: programs whose device memory
// is fully owned by another allocator (for example a framework's caching
// allocator that has reserved the whole pool, where a cudaMalloc beside it
// fails or fragments it), and latency-bound loops with a fixed memory
// footprint that cannot accept the implicit device synchronization of
// cudaFree.  They pass the state and an output buffer; everything else the
// energy kernels need (term layout, job record, per-block partial sums)
// lives in one file-scope device array of fixed size, which every GPU that
// loads this library holds until the process exits.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <mutex>
#include <new>

#include "qw_internal.h"

namespace qw {

namespace {

constexpr uint32_t NA_CLASS_BITS = 3, NA_MAX_CLASSES = 1u << NA_CLASS_BITS;
// every group of a class but its last holds EN_RANK independent masks, so at
// least as many terms
constexpr uint32_t NA_MAX_GROUPS = QW_NOALLOC_MAX_TERMS / EN_RANK + NA_MAX_CLASSES + 1;
// blocks of the largest register
constexpr uint32_t NA_REP_BITS = en_rep_bits(QW_NOALLOC_MAX_QUBITS);
constexpr uint32_t NA_MAX_BLOCKS = NA_MAX_CLASSES << (QW_NOALLOC_MAX_QUBITS - EN_RANK - NA_REP_BITS -
                                                      en_iter_bits(QW_NOALLOC_MAX_QUBITS, NA_REP_BITS));

struct alignas(16) NaHeader {
  alignas(16) EnJob job;
  alignas(16) EnClass classes[NA_MAX_CLASSES];
  EnGroup groups[NA_MAX_GROUPS];
  EnTerm terms[QW_NOALLOC_MAX_TERMS];
};
struct NaScratch {
  NaHeader h;
  alignas(16) double partials[2 * NA_MAX_BLOCKS];
};

}  // namespace

// The scratch array (about 1.1 MB).  In host code this name is only a
// stand-in for the device object: its device address comes from
// cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char qw_noalloc_scratch[sizeof(NaScratch)];

namespace {

std::mutex g_mu;
void *g_dev_ptr[256];  // device address of the scratch array, per device

qw_status scratch_address(int dev, NaScratch **out) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (dev < 0 || dev >= 256) {
    set_last_error("device ordinal out of range");
    return QW_ERR_INVALID_ARG;
  }
  if (!g_dev_ptr[dev]) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, qw_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      set_last_error(std::string("cudaGetSymbolAddress failed: ") + cudaGetErrorString(e));
      return QW_ERR_CUDA;
    }
    g_dev_ptr[dev] = p;
  }
  *out = (NaScratch *)g_dev_ptr[dev];
  return QW_OK;
}

// Copies a piece of the host-built layout, passed by value as the kernel's
// parameter (the device reads no host memory), into the scratch array.
struct NaPiece {
  uint4 w[1024];
};
static_assert(sizeof(NaPiece) <= 32000 && sizeof(NaHeader) % 16 == 0, "pieces fit the kernel parameter space");
__global__ void na_setup_kernel(const NaPiece h, uint4 *dst, uint32_t n) {
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) dst[i] = h.w[i];
}

}  // namespace
}  // namespace qw

extern "C" qw_status qw_sv_energy_noalloc_dev(uint32_t mode, uint32_t n, const void *state,
                                              const qw_pauli_term *terms, uint64_t n_terms, double *out,
                                              void *stream) {
  using namespace qw;
  set_last_error("");
  if (mode > QW_MODE_SV_FP32) {
    set_last_error("statevector modes only");
    return QW_ERR_INVALID_ARG;
  }
  if (!state || !out || (n_terms && !terms)) {
    set_last_error("NULL argument");
    return QW_ERR_INVALID_ARG;
  }
  if (n < SV_G) {
    set_last_error("n must be at least 5 (states are padded to 5 qubits)");
    return QW_ERR_INVALID_ARG;
  }
  if (n > QW_NOALLOC_MAX_QUBITS) {
    set_last_error("n must be at most " + std::to_string(QW_NOALLOC_MAX_QUBITS) +
                   " for the non-allocating energy's scratch array");
    return QW_ERR_BUDGET;
  }
  if (n_terms > QW_NOALLOC_MAX_TERMS) {
    set_last_error("at most " + std::to_string(QW_NOALLOC_MAX_TERMS) +
                   " terms fit the non-allocating energy's scratch array");
    return QW_ERR_BUDGET;
  }
  const uint64_t mask = (1ull << n) - 1;
  for (uint64_t k = 0; k < n_terms; k++)
    if ((terms[k].xmask | terms[k].zmask) & ~mask) {
      set_last_error("a term acts outside the register");
      return QW_ERR_INVALID_ARG;
    }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    set_last_error("no current CUDA device");
    return QW_ERR_CUDA;
  }
  NaScratch *S = nullptr;
  qw_status st = scratch_address(dev, &S);
  if (st != QW_OK) return st;

  // The term layout of the allocating entry point with at most 3 class bits,
  // so that it fits the fixed arrays (chunks of an eighth of the state above
  // 25 qubits, where the allocating one takes smaller ones: the same terms,
  // added in another order)
  const bool fp64 = mode == QW_MODE_SV_FP64, pair = en_pair(fp64, state);
  NaHeader h;  // built on the host stack, handed to the device as a kernel parameter
  uint32_t n_blocks = 0;
  try {
    const EnLayout L = build_energy_layout(terms, n_terms, n, fp64, pair, en_rep_bits(n), NA_CLASS_BITS);
    if (L.classes.size() > NA_MAX_CLASSES || L.groups.size() > NA_MAX_GROUPS || L.n_blocks > NA_MAX_BLOCKS) {
      set_last_error("the term layout exceeds the scratch array");
      return QW_ERR_BUDGET;
    }
    std::copy(L.classes.begin(), L.classes.end(), h.classes);
    std::copy(L.groups.begin(), L.groups.end(), h.groups);
    std::copy(L.terms.begin(), L.terms.end(), h.terms);
    h.job.state = state;
    h.job.out = out;
    h.job.n = n;
    h.job.rep_bits = L.rep_bits;
    h.job.iter_bits = L.iter_bits;
    h.job.class_begin = 0;
    h.job.n_classes = (uint32_t)L.classes.size();
    h.job.block_begin = 0;
    h.job.n_blocks = n_blocks = L.n_blocks;
  } catch (const std::bad_alloc &) {
    set_last_error("host allocation failed");
    return QW_ERR_OOM;
  }
  // every partial is written by its block before the reduction reads it, so
  // nothing in the array needs clearing between calls
  cudaStream_t s = (cudaStream_t)stream;
  char *base = (char *)S;  // device address: offsets only, never dereferenced here
  EnJob *d_job = (EnJob *)(base + offsetof(NaScratch, h) + offsetof(NaHeader, job));
  EnClass *d_classes = (EnClass *)(base + offsetof(NaScratch, h) + offsetof(NaHeader, classes));
  EnGroup *d_groups = (EnGroup *)(base + offsetof(NaScratch, h) + offsetof(NaHeader, groups));
  EnTerm *d_terms = (EnTerm *)(base + offsetof(NaScratch, h) + offsetof(NaHeader, terms));
  double *d_partials = (double *)(base + offsetof(NaScratch, partials));
  const size_t hdr = offsetof(NaHeader, terms) + sizeof(EnTerm) * (size_t)n_terms;
  for (size_t o = 0; o < hdr; o += sizeof(NaPiece)) {
    NaPiece piece;
    const size_t k = std::min(sizeof(NaPiece), hdr - o);
    memcpy(&piece, (const char *)&h + o, k);
    na_setup_kernel<<<1, 256, 0, s>>>(piece, (uint4 *)(base + offsetof(NaScratch, h) + o), (uint32_t)(k / 16));
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string("layout copy failed: ") + cudaGetErrorString(e));
    return QW_ERR_CUDA;
  }
  launch_energy(fp64, pair, EnTables{d_job, d_classes, d_groups, d_terms, d_partials}, 1, n_blocks,
                en_rep_bits(n), s);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string("energy launch failed: ") + cudaGetErrorString(e));
    return QW_ERR_CUDA;
  }
  return QW_OK;
}
