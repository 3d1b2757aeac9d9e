// Engine: device memory, boundary-state store, execution of a plan,
// CUDA-graph capture, autotuning of the tile schedule and the learned cost
// model's training loop.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <functional>
#include <map>
#include <random>

#include "dense.h"
#include "plan.h"

namespace qw {
qw_dense_prog *dense_prog_autotune(Engine *E, uint32_t mode, uint32_t n, const qw_gate *gates, uint64_t n_gates,
                                   uint32_t kmax, uint32_t engine);
void dense_prog_config(const qw_dense_prog *p, uint32_t *engine, uint32_t *kmax, uint32_t *nacc, double *est_ms);
uint64_t dense_prog_blocks(const qw_dense_prog *p);
void dense_prog_run(qw_dense_prog *p, void *state, void *stream);
qw_status dense_prog_check(qw_dense_prog *p);
void dense_prog_destroy(qw_dense_prog *p);

#define CK(x)                                                                       \
  do {                                                                              \
    cudaError_t e_ = (x);                                                           \
    if (e_ != cudaSuccess)                                                          \
      fail(e_ == cudaErrorMemoryAllocation ? QW_ERR_OOM : QW_ERR_CUDA, "%s: %s (%s:%d)", #x, \
           cudaGetErrorString(e_), __FILE__, __LINE__);                             \
  } while (0)

// ---------------------------------------------------------------------------
// small kernels
// ---------------------------------------------------------------------------
// |0...0>: every amplitude 0, the first 1
__global__ void basis_zero_kernel(void *state, bool fp64, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    if (fp64) ((double2 *)state)[i] = make_double2(i == 0 ? 1.0 : 0.0, 0.0);
    else ((float2 *)state)[i] = make_float2(i == 0 ? 1.f : 0.f, 0.f);
  }
}

__global__ void convert_kernel(const void *src, bool src64, void *dst, bool dst64, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double re, im;
  if (src64) { const double2 v = ((const double2 *)src)[i]; re = v.x; im = v.y; }
  else { const float2 v = ((const float2 *)src)[i]; re = v.x; im = v.y; }
  if (dst64) ((double2 *)dst)[i] = make_double2(re, im);
  else ((float2 *)dst)[i] = make_float2((float)re, (float)im);
}

void launch_copy(const void *src, void *dst, size_t bytes, void *stream) {
  if (bytes) cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// device-side tables of a set of statevector programs
// ---------------------------------------------------------------------------
// A stage of one rotation without a phase runs as a general op: its two-term
// outputs (compensated: 17 packed instructions per amplitude with the split
// and the rounding, FP64: 4 operations) cost less than an unnormalized
// rotation and the factors of the table (24 and 6).
static bool lone_rotation(const HostStage &st) {
  return st.ops.size() == 1 && st.ops[0].kind == K_R && st.gphase[0] == 1.0 && st.gphase[1] == 0.0;
}

// Factors of FP64 rotation stages are products of up to eleven numbers, and an
// error of theirs is the same in every amplitude: they are formed as unevaluated
// sums of two doubles (products split by FMA, sums by TwoSum) and rounded once
// (states of 7-qubit sweeps err by 7.3e-16, 8.3e-16 with products in FP64).
struct Dd {
  double h, l;
};
static Dd dd_sum(double a, double b) {
  const double s = a + b, z = s - a;
  return {s, (a - (s - z)) + (b - z)};
}
static Dd dd_add(Dd a, Dd b) {
  const Dd s = dd_sum(a.h, b.h);
  return dd_sum(s.h, s.l + (a.l + b.l));
}
static Dd dd_mul(Dd a, Dd b) {
  const double p = a.h * b.h;
  return dd_sum(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
struct DdC {
  Dd re, im;
};
static DdC dd_cmul(const DdC &a, const DdC &b) {
  const Dd p = dd_mul(a.im, b.im);
  return {dd_add(dd_mul(a.re, b.re), Dd{-p.h, -p.l}), dd_add(dd_mul(a.re, b.im), dd_mul(a.im, b.re))};
}
// The diagonal entry r of a rotation's row {1, t} r, corrected so that the
// row has length 1 with t as it is stored: r (1 + e / 2), e = 1 - r^2 (1 + t^2).
static Dd dd_unit_row(double r, double t) {
  const Dd n = dd_mul(dd_mul({r, 0}, {r, 0}), dd_add({1, 0}, dd_mul({t, 0}, {t, 0})));
  const double e = (1.0 - n.h) - n.l;
  return std::fabs(e) < 1e-12 ? dd_sum(r, 0.5 * r * e) : Dd{r, 0};
}

struct SvTableBuilder {
  std::vector<SvPassDesc> passes;
  std::vector<SvStageDesc> stages;
  std::vector<SvOpDesc<float>> ops32;
  std::vector<float> ops32lo;  // m[t] - (float)m[t] per FP32 op (compensated passes)
  std::vector<float> ph;       // blocks of the compensated rotation stages (see SvStageDesc::ph_block)
  std::vector<double> ph64;    // and of FP64 ones
  std::vector<SvOpDesc<double>> ops64;
  bool fp64;
  explicit SvTableBuilder(bool f) : fp64(f) {}
  // appends the program; returns the index of its first pass
  uint32_t add(const SvProgram &pr) {
    const uint32_t first = (uint32_t)passes.size();
    for (const HostPass &hp : pr.passes) {
      SvPassDesc d;
      memset(&d, 0, sizeof(d));
      d.k = (uint32_t)hp.q.size();
      d.b = hp.b;
      d.n_stages = (uint32_t)hp.stages.size();
      d.stage_begin = (uint32_t)stages.size();
      uint32_t inq = 0;
      for (uint32_t q : hp.q) inq |= 1u << q;
      uint32_t nh = 0;
      for (uint32_t q = 0; q < pr.n; q++)
        if (!(inq & (1u << q))) d.hi_pos[nh++] = (uint8_t)q;
      d.n_hi = nh;
      // local bit i (>= b) -> global qubit hp.q[i]
      for (uint32_t v = 0; v < 64; v++) {
        uint32_t g = 0;
        for (uint32_t j = 0; j < 6; j++)
          if ((v >> j) & 1u) { const uint32_t li = d.b + j; if (li < d.k) g |= 1u << hp.q[li]; }
        d.lo_tab[v] = g;
      }
      for (uint32_t v = 0; v < 32; v++) {
        uint32_t g = 0;
        for (uint32_t j = 0; j < 5; j++)
          if ((v >> j) & 1u) { const uint32_t li = d.b + 6 + j; if (li < d.k) g |= 1u << hp.q[li]; }
        d.hi_tab[v] = g;
      }
      // byte offset of the swizzled slot of a (pre-swizzle) tile index
      const uint32_t asz = fp64 ? 16u : 8u;
      auto slot = [&](uint32_t v) { return (fp64 ? sv_swz64(v) : sv_swz32(v)) * asz; };
      auto phi_of = [&](const uint32_t *mcol, uint32_t mc, uint32_t l) {
        uint32_t v = mc;
        for (uint32_t t = 0; t < d.k; t++)
          if ((l >> t) & 1u) v ^= mcol[t];
        return v;
      };
      // every tile map must be a bijection of the k-bit tile index: the
      // kernels address shared memory through it
      auto check_phi = [&](const uint32_t *mcol, uint32_t mc) {
        const uint32_t km = (1u << d.k) - 1u;
        uint32_t basis[32] = {0};
        bool ok = (mc & ~km) == 0;
        for (uint32_t t = 0; t < d.k && ok; t++) {
          uint32_t v = mcol[t];
          if (v & ~km) { ok = false; break; }
          for (int bit = 31; bit >= 0 && v; bit--)
            if ((v >> bit) & 1u) {
              if (!basis[bit]) { basis[bit] = v; break; }
              v ^= basis[bit];
            }
          ok = v != 0;
        }
        if (!ok) fail(QW_ERR_STATE, "internal: tile map of a pass is not a bijection");
      };
      check_phi(hp.mcol, hp.mc);
      for (const HostStage &hs : hp.stages) check_phi(hs.mcol, hs.mc);
      // outside control qubits -> tile-index bits; their per-tile terms
      // must stay inside the tile like every column of the map
      if (hp.ctl_q.size() > (size_t)SV_MAX_OUT_CTL) fail(QW_ERR_STATE, "internal: too many outside controls");
      uint32_t ctl_tb[SV_MAX_OUT_CTL] = {0, 0, 0, 0};
      for (size_t c = 0; c < hp.ctl_q.size(); c++) {
        uint32_t tb = 0xFFFFFFFFu;
        for (uint32_t i = 0; i < d.n_hi; i++)
          if (d.hi_pos[i] == hp.ctl_q[c]) tb = i;
        if (tb == 0xFFFFFFFFu) fail(QW_ERR_STATE, "internal: outside control %u is a tile qubit", hp.ctl_q[c]);
        ctl_tb[c] = tb;
      }
      auto check_ctl = [&](const uint32_t *w) {
        for (int c = 0; c < SV_MAX_OUT_CTL; c++)
          if ((w[c] >> d.k) != 0 || (w[c] != 0 && (size_t)c >= hp.ctl_q.size()))
            fail(QW_ERR_STATE, "internal: per-tile map term outside the tile");
      };
      check_ctl(hp.ctl_w);
      for (const HostStage &hs : hp.stages) check_ctl(hs.ctl_w);
      for (int c = 0; c < SV_MAX_OUT_CTL; c++) {
        d.ctl_tb[c] = ctl_tb[c];
        d.ctl_w[c] = slot(hp.ctl_w[c]);
      }
      {
        bool ident = hp.mc == 0;
        for (uint32_t t = 0; t < d.k; t++) ident = ident && hp.mcol[t] == (1u << t);
        for (int c = 0; c < SV_MAX_OUT_CTL; c++) ident = ident && hp.ctl_w[c] == 0;
        d.phi_ident = ident ? 1u : 0u;
        const uint32_t apu_bits = fp64 ? 0u : 1u;  // amplitudes per 16-byte unit: 2^apu_bits
        for (uint32_t v = 0; v < 64; v++) d.st_lo[v] = slot(phi_of(hp.mcol, hp.mc, v << apu_bits));
        for (uint32_t v = 0; v < 128; v++) d.st_hi[v] = slot(phi_of(hp.mcol, 0, v << (6 + apu_bits)));
        d.phi_pair = fp64 ? 0u : slot(hp.mcol[0]);
        bool unit16 = true;  // FP64: a unit is one amplitude
        if (!fp64) {
          unit16 = d.phi_pair == 8u;
          for (uint32_t v = 0; v < 64 && unit16; v++) unit16 = (d.st_lo[v] & 8u) == 0;
          for (uint32_t v = 0; v < 128 && unit16; v++) unit16 = (d.st_hi[v] & 8u) == 0;
          for (int c = 0; c < SV_MAX_OUT_CTL && unit16; c++) unit16 = (d.ctl_w[c] & 8u) == 0;
        }
        d.phi_unit16 = unit16 ? 1u : 0u;
      }
      for (const HostStage &hs : hp.stages) {
        SvStageDesc sd;
        memset(&sd, 0, sizeof(sd));
        uint32_t pm = 0;
        for (uint32_t j = 0; j < pr.g; j++) {
          sd.roff[j] = slot(hs.mcol[hs.pos[j]]);
          pm |= 1u << hs.pos[j];
        }
        sd.cst = slot(hs.mc);
        for (int c = 0; c < SV_MAX_OUT_CTL; c++) {
          sd.ctl_tb[c] = ctl_tb[c];
          sd.ctl_w[c] = slot(hs.ctl_w[c]);
        }
        // group bits: the first four (the lanes of a half warp) chosen so
        // that their slots differ in the bank bits (slot bits 0-3 of 8-byte
        // FP32 slots, 0-2 of 16-byte FP64 slots), the rest ascending
        std::vector<uint32_t> free_pos;
        for (uint32_t t = 0; t < d.k; t++)
          if (!(pm & (1u << t))) free_pos.push_back(t);
        const uint32_t bank_mask = fp64 ? 7u : 15u;
        std::vector<uint32_t> order, basis;
        std::vector<uint8_t> used(free_pos.size(), 0);
        for (int pick = 0; pick < 4; pick++) {
          int best = -1;
          for (size_t c = 0; c < free_pos.size() && best < 0; c++) {
            if (used[c]) continue;
            uint32_t v = (fp64 ? sv_swz64(hs.mcol[free_pos[c]]) : sv_swz32(hs.mcol[free_pos[c]])) & bank_mask;
            for (uint32_t bv : basis) v = std::min(v, v ^ bv);  // reduce against the echelon basis
            if (v) { best = (int)c; basis.push_back(v); std::sort(basis.rbegin(), basis.rend()); }
          }
          if (best < 0) break;
          used[best] = 1;
          order.push_back(free_pos[best]);
        }
        for (size_t c = 0; c < free_pos.size(); c++)
          if (!used[c]) order.push_back(free_pos[c]);
        if (order.size() > (size_t)SV_MAX_GBITS) fail(QW_ERR_STATE, "internal: tile wider than the stage descriptor");
        for (size_t t = 0; t < order.size(); t++) sd.gcol[t] = slot(hs.mcol[order[t]]);
        // a stage of real rotations (with or without a |1>-phase) on
        // distinct positions runs as one straight-line sequence: the ops
        // commute, so they are stored in position order as K_RP records
        std::vector<HostOp> sops = hs.ops;
        uint32_t rp_mask = 0;
        bool rp_stage = !sops.empty();
        for (const HostOp &o : sops) {
          if ((o.kind != K_RP && o.kind != K_R) || (rp_mask & (1u << o.a))) { rp_stage = false; break; }
          rp_mask |= 1u << o.a;
        }
        if ((fp64 || pr.g == 4) && lone_rotation(hs)) rp_stage = false;
        if (rp_stage) {
          std::sort(sops.begin(), sops.end(), [](const HostOp &x, const HostOp &y) { return x.a < y.a; });
          for (HostOp &o : sops)
            if (o.kind == K_R) {  // {r00, 0, r01, 0, r10, 0, r11, 0} -> {r00, r01, r10, r11, 1, 0}
              const double r[4] = {o.m[0], o.m[2], o.m[4], o.m[6]};
              o.m[0] = r[0]; o.m[1] = r[1]; o.m[2] = r[2]; o.m[3] = r[3];
              o.m[4] = 1.0; o.m[5] = 0.0; o.m[6] = 0.0; o.m[7] = 0.0;
              o.kind = K_RP;
            }
        }
        sd.rp_mask = rp_stage ? rp_mask : 0u;
        // a compensated or FP64 stage of rotations: each real orthogonal 2x2
        // {r00, r01; r10, r11} is diag(r00, r11) {1, r01/r00; r10/r11, 1};
        // where |r01| is the larger entry the columns are exchanged first
        // (the group is read with that position's halves exchanged), so the
        // off-diagonal quotients stay within 1.  The diagonals commute with
        // the other positions' rotations: amplitude e takes their product,
        // with the |1>-phases of its set positions.  Quotients and products
        // are computed here in FP64 and, for compensated stages, stored as
        // FP32 pairs (to 2^-48: the same angle repeated thousands of times
        // adds its constants' error up)
        sd.ph_block = 0xFFFFFFFFu;
        const bool gfold = hs.gphase[0] != 1.0 || hs.gphase[1] != 0.0;
        if (gfold && (!rp_stage || (!fp64 && pr.g != 4))) fail(QW_ERR_STATE, "internal: a global phase on a stage without a table");
        if (rp_stage && (fp64 || pr.g == 4)) {
          sd.ph_block = fp64 ? (uint32_t)(ph64.size() / (2 * SV_PH64_BLOCK)) : (uint32_t)stages.size();
          double t[SV_G][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
          // factors of the amplitudes so far, doubled position by position
          std::complex<double> f32[16] = {{hs.gphase[0], hs.gphase[1]}};
          DdC f64[32] = {{{hs.gphase[0], 0}, {hs.gphase[1], 0}}};
          uint32_t next = 0;
          auto double_table = [&](uint32_t pos, double r0, double r1, const double *ph1) {
            const uint32_t n = 1u << pos;
            if (fp64) {
              const Dd d0 = ph1 ? dd_unit_row(r0, t[pos][0]) : Dd{1, 0}, d1 = ph1 ? dd_unit_row(r1, t[pos][1]) : Dd{1, 0};
              const DdC w{dd_mul(d1, {ph1 ? ph1[0] : 1.0, 0}), dd_mul(d1, {ph1 ? ph1[1] : 0.0, 0})};
              for (uint32_t e = 0; e < n; e++) {
                f64[e | n] = ph1 ? dd_cmul(f64[e], w) : f64[e];
                if (ph1) f64[e] = {dd_mul(f64[e].re, d0), dd_mul(f64[e].im, d0)};
              }
            } else {
              const std::complex<double> w = ph1 ? r1 * std::complex<double>(ph1[0], ph1[1]) : 1.0;
              for (uint32_t e = 0; e < n; e++) {
                f32[e | n] = f32[e] * w;
                if (ph1) f32[e] *= r0;
              }
            }
            next = pos + 1;
          };
          for (const HostOp &o : sops) {
            double r00 = o.m[0], r01 = o.m[1], r10 = o.m[2], r11 = o.m[3];
            if (std::fabs(r01) > std::fabs(r00)) {
              std::swap(r00, r01);
              std::swap(r10, r11);
              sd.ld_xor ^= sd.roff[o.a];
            }
            t[o.a][0] = r01 / r00;
            t[o.a][1] = r10 / r11;
            while (next < o.a) double_table(next, 1.0, 1.0, nullptr);  // (ops are in position order)
            double_table(o.a, r00, r11, o.m + 4);
          }
          while (next < pr.g) double_table(next, 1.0, 1.0, nullptr);
          for (uint32_t q = 0; q < pr.g; q++) {
            if (fp64) {
              ph64.insert(ph64.end(), {t[q][0], t[q][1]});
            } else {
              const float h0 = (float)t[q][0], h1 = (float)t[q][1];
              ph.insert(ph.end(), {h0, h1, (float)(t[q][0] - (double)h0), (float)(t[q][1] - (double)h1)});
            }
          }
          for (uint32_t e = 0; e < (1u << pr.g); e++) {
            if (fp64) {
              ph64.insert(ph64.end(), {f64[e].re.h, f64[e].im.h});
            } else {
              for (const double v : {f32[e].real(), f32[e].imag()})
                ph.insert(ph.end(), {(float)v, (float)(v - (double)(float)v)});
            }
          }
          sops.clear();  // the stage runs from its block alone
        }
        sd.n_ops = (uint32_t)sops.size();
        sd.op_begin = (uint32_t)(fp64 ? ops64.size() : ops32.size());
        for (const HostOp &o : sops) {
          const uint32_t lo = std::min(o.a, o.b), hi = std::max(o.a, o.b);
          const uint32_t code = o.kind == K_CD ? sv_op_index(o.kind, lo, hi) : sv_op_index(o.kind, o.a, 0);
          if (code >= SV_N_OP_INDEX || o.a >= pr.g || (o.kind == K_CD && (hi >= pr.g || lo == hi)))
            fail(QW_ERR_STATE, "internal: op outside the stage dispatch table");
          if (fp64) {
            SvOpDesc<double> od{};
            od.code = code;
            for (int t = 0; t < 8; t++) od.m[t] = o.m[t];
            ops64.push_back(od);
          } else {
            SvOpDesc<float> od{};
            od.code = code;
            for (int t = 0; t < 8; t++) {
              od.m[t] = (float)o.m[t];
              ops32lo.push_back((float)(o.m[t] - (double)od.m[t]));
            }
            ops32.push_back(od);
          }
        }
        stages.push_back(sd);
        // compensated programs have a block per stage (zero where unused), so
        // that a stage's descriptor and block are fetched together
        if (!fp64 && pr.g == 4) ph.resize(stages.size() * SV_PH_BLOCK, 0.f);
      }
      passes.push_back(d);
    }
    return first;
  }
};

// device allocation tracked for release
struct DevArena {
  Engine *eng = nullptr;  // when set, blocks come from and return to the engine's cache
  std::vector<std::pair<void *, size_t>> blocks;
  uint64_t h2d = 0;  // bytes uploaded from the host
  void *alloc(size_t bytes) {
    void *p = nullptr;
    if (bytes == 0) bytes = 16;
    size_t got = bytes;
    if (eng) p = eng->dev_alloc(bytes, &got);
    else CK(cudaMalloc(&p, bytes));
    blocks.push_back({p, got});
    return p;
  }
  template <typename T>
  T *upload(const std::vector<T> &v, cudaStream_t s) {
    T *p = (T *)alloc(v.size() * sizeof(T));
    if (!v.empty()) CK(cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, s));
    h2d += v.size() * sizeof(T);
    return p;
  }
  void release() {
    for (auto &b : blocks) {
      if (eng) eng->dev_free(b.first, b.second);
      else cudaFree(b.first);
    }
    blocks.clear();
  }
};

struct Wave {
  bool fp64 = false;
  bool per_pass = false;                  // one launch per pass (else one persistent launch)
  int ar = SV_AR_PLAIN;                   // arithmetic of the wave's FP32 passes
  uint32_t k_max = 13;
  int grid = 0;
  std::vector<uint32_t> tasks;            // tasks run in this wave (own buffers)
  std::vector<uint32_t> obs_tasks;        // tasks whose observables are evaluated in this wave
  std::vector<SvJob> jobs;                // pass jobs, in list order
  bool few = false;                       // at most SV_FEW_TILES tiles side by side
  bool fused_energy = false;              // energy blocks run inside the persistent launch
  uint32_t seg_bits = 0;
  std::vector<SvSeg> segs;
  uint32_t total_items = 0;
  SvJob *d_jobs = nullptr;
  SvSeg *d_segs = nullptr;
  unsigned int *d_ctr = nullptr;
  size_t ctr_words = 0;
  std::vector<EnJob> en;
  std::vector<uint32_t> obs_tasks_en;     // task of each energy job
  uint32_t en_blocks = 0;
  EnJob *d_en = nullptr;
  std::vector<SmpSource> src;
  uint32_t smp_blocks = 0;
  SmpSource *d_src = nullptr;
  std::vector<SmpShot> shots;
  SmpShot *d_shots = nullptr;
  std::vector<std::pair<uint32_t, std::pair<const void *, void *>>> converts;  // task, (src, dst)
};

struct DeviceState {
  DevArena arena;
  cudaStream_t stream = nullptr;
  SvTables t32{}, t64{};
  // FP32 arithmetic: of the boundaries' passes and per-task launches
  // (ar_chain: SV_AR_REM, or SV_AR_PLAIN) and of the persistent suffix
  // launches (ar_batch: SV_AR_COMP or SV_AR_PLAIN); `rem` is the remainder
  // array those chains share (they run one after another on the stream)
  int ar_chain = SV_AR_PLAIN, ar_batch = SV_AR_PLAIN;
  void *rem = nullptr;
  std::vector<uint32_t> mat_pass0, task_pass0;
  std::vector<void *> mat_buf;
  std::vector<void *> mat_export[2];   // per mode (FP64, FP32): statevector exported from a tableau node
  std::vector<StabBasis *> mat_basis;  // scratch of each exporting tableau node
  std::vector<qw_dense_prog *> mat_dense;  // boundary evolved by a dense-block program, else NULL
  // statevector boundaries of one precision in one persistent launch (a
  // boundary's first pass waits for its parent's last); empty = per-pass launches
  struct MatBatch {
    bool fp64 = false;
    int ar = SV_AR_PLAIN;
    uint32_t k_max = 5, seg_bits = 0, total_items = 0;
    bool few = false;  // at most SV_FEW_TILES tiles side by side
    int grid = 0;
    size_t n_jobs = 0, ctr_words = 0;
    SvJob *d_jobs = nullptr;
    SvSeg *d_segs = nullptr;
    unsigned int *d_ctr = nullptr;
  };
  std::vector<MatBatch> mat_batches;
  std::vector<void *> task_state;  // state a task's observables read
  std::vector<Wave> waves;
  EnClass *d_classes = nullptr;
  EnGroup *d_groups = nullptr;
  EnTerm *d_terms = nullptr;
  std::vector<uint32_t> ham_class_off;
  double *d_partials = nullptr;
  double *d_bsum = nullptr, *d_boff = nullptr;
  int32_t *d_blast = nullptr;
  int64_t *d_lastnz = nullptr;
  double *d_energy = nullptr;
  uint64_t *d_samples = nullptr;
  // tableau
  TabProgram *d_progs = nullptr;
  TabLayer *d_layers = nullptr;
  TabSlot *d_slots = nullptr;
  uint8_t *d_bits = nullptr;
  uint8_t *d_outs = nullptr, *d_mat_outs = nullptr;
  struct TabLaunch {
    TabArgs a;
    uint32_t n_tasks;
    int frame;  // >= 0: preceded by the reference run and the frame launch of this frame group
  };
  std::vector<TabLaunch> tab_mat_launches, tab_task_launches;
  // final inverse tableau of each tableau task submitted with
  // QW_TASK_KEEP_STATE: 2n rows of 2W words, then 2n sign bytes elsewhere
  std::vector<std::pair<const uint64_t *, const uint8_t *>> tab_keep;
  struct FrameLaunch {
    TabArgs ref;  // the reference suffix on the tableau (one CTA), outcomes and random flag
    FrameArgs fa;
  };
  std::vector<FrameLaunch> frame_launches;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  cudaEvent_t ev[8] = {nullptr};
  std::vector<cudaEvent_t> wave_ev;  // 4 per wave: start, after suffix, after energy, after sampling
  ~DeviceState() {
    if (gexec) cudaGraphExecDestroy(gexec);
    if (graph) cudaGraphDestroy(graph);
    for (auto &e : ev) if (e) cudaEventDestroy(e);
    for (auto &e : wave_ev) cudaEventDestroy(e);
    arena.release();
  }
};

// remainder arrays that the boundaries of a plan may hold together
constexpr uint64_t MAT_REM_BYTES = 2ull << 30;

static size_t sv_state_bytes(bool fp64, uint32_t n_eff) { return (size_t)(fp64 ? 16 : 8) << n_eff; }

// HBM bytes of a chain of `passes` passes over a state of S bytes: the state
// is read and written once per pass; with a remainder array (SV_AR_REM)
// every pass but the first also reads it and every pass but the last writes it
static double chain_bytes(double S, size_t passes, int ar) {
  const double p = (double)passes;
  return 2.0 * S * p + ((ar == SV_AR_REM && passes > 1) ? 2.0 * S * (p - 1.0) : 0.0);
}
// remainder arrays of pass p of a chain of n passes (SV_AR_REM)
static const void *chain_src_lo(const DeviceState *D, int ar, size_t p) {
  return (ar == SV_AR_REM && p > 0) ? D->rem : nullptr;
}
static void *chain_dst_lo(const DeviceState *D, int ar, size_t p, size_t n) {
  return (ar == SV_AR_REM && p + 1 < n) ? D->rem : nullptr;
}
// Algorithmic floating-point operations of one pass over 2^n amplitudes
// (an FMA counts two, an add or a multiply one), from its stages' register
// ops under the arithmetic `ar`, per group of A = 2^g amplitudes:
//   plain: a real rotation output costs 6 (packed multiply + FMA on both
//   components), a complex product 6, a general 2x2 output 14;
//   compensated (sv_df.cuh): a multiply-accumulate on the grid is 4 FMAs
//   and a subtraction per component (18 for the amplitude's two), so with
//   the un-biasing of the operand a two-term output costs 40, an
//   unnormalized rotation output 22, a general 2x2 output 80, and every
//   stage splits (6) and rounds (4) each amplitude.
static double pass_flops(const HostPass &hp, uint32_t n, uint32_t g, int ar) {
  const bool comp = ar != SV_AR_PLAIN;
  const double groups = std::ldexp(1.0, (int)n - (int)g), A = std::ldexp(1.0, (int)g);
  const double lin = comp ? 40.0 : 6.0, cm = comp ? 40.0 : 6.0, u1 = comp ? 80.0 : 14.0;
  double f = 0;
  for (const HostStage &st : hp.stages) {
    double fg = comp ? A * 10.0 : 0.0;
    if (comp) {
      uint32_t mask = 0;
      bool rot = !st.ops.empty();
      for (const HostOp &o : st.ops) {
        rot = rot && (o.kind == K_RP || o.kind == K_R) && !(mask & (1u << o.a));
        mask |= 1u << o.a;
      }
      if (rot && !lone_rotation(st)) {  // unnormalized rotations, then one product per amplitude
        f += (fg + A * (22.0 * (double)st.ops.size() + cm)) * groups;
        continue;
      }
    }
    for (const HostOp &o : st.ops) {
      switch (o.kind) {
        case K_R: case K_RX: fg += A * lin; break;
        case K_RP: fg += A * lin + A / 2 * cm; break;
        case K_U1: fg += A * u1; break;
        case K_D1: fg += A * cm; break;
        case K_P1: fg += A / 2 * cm; break;
        case K_CD: fg += (comp && o.m[0] == -1.0 && o.m[1] == 0.0) ? 0.0 : A / 4 * cm; break;
        default: break;
      }
    }
    f += fg * groups;
  }
  return f;
}

int plan_ar_batch(const qw_plan *P) { return P->fp32_compensated ? SV_AR_COMP : SV_AR_PLAIN; }

// Segment size of a persistent work list: the largest power of two (at most
// 64) that no job's unit count falls below, so that few items are empty.
static uint32_t segment_bits(const std::vector<SvJob> &jobs) {
  uint32_t mn = 64;
  for (const SvJob &j : jobs) mn = std::min<uint32_t>(mn, std::max<uint32_t>(1, j.n_tiles));
  uint32_t b = 0;
  while ((2u << b) <= mn) b++;
  return b;
}

// Orders the work of one persistent launch into segments.  jobs[0, n_pass)
// are pass jobs, already in list order (a task's passes in sequence); the
// rest are energy jobs sorted by the pass job they wait for.  An energy job
// is released once its dependency has been listed and `lag` more items have
// gone by (by then its last tiles have been taken, so the wait is short);
// released energy work is interleaved so that the pass and energy streams
// advance at the same fraction of their totals, which keeps the two kinds
// of work (ALU-bound tiles, L2-bound energy blocks) running side by side.
static void build_segments(const std::vector<SvJob> &jobs, size_t n_pass, uint32_t seg_bits, uint64_t lag,
                           std::vector<SvSeg> &segs) {
  const uint64_t G = 1ull << seg_bits;
  auto nseg = [&](const SvJob &j) { return (uint64_t)(j.n_tiles + G - 1) / G; };
  uint64_t pass_total = 0, en_total = 0;
  for (size_t i = 0; i < jobs.size(); i++) (i < n_pass ? pass_total : en_total) += nseg(jobs[i]);
  segs.clear();
  segs.reserve(pass_total + en_total);
  std::vector<int64_t> end_seg(jobs.size(), -1);  // one past the job's last segment
  std::vector<int64_t> first_seg(jobs.size(), -1);
  size_t pi = 0, ei = n_pass;
  uint32_t pu = 0, eu = 0;
  uint64_t pass_done = 0, en_done = 0;
  const uint64_t lag_segs = (lag + G - 1) / G;
  while (pi < n_pass || ei < jobs.size()) {
    // skip jobs without units
    if (pi < n_pass && jobs[pi].n_tiles == 0) { end_seg[pi] = first_seg[pi] = (int64_t)segs.size(); pi++; continue; }
    if (ei < jobs.size() && jobs[ei].n_tiles == 0) { ei++; continue; }
    bool e_ready = false;
    if (ei < jobs.size()) {
      const int dep = jobs[ei].dep;
      e_ready = dep < 0 || (end_seg[dep] >= 0 && (pi >= n_pass || (uint64_t)segs.size() - end_seg[dep] >= lag_segs));
    }
    bool take_e;
    if (pi >= n_pass) take_e = true;
    else if (!e_ready) take_e = false;
    else take_e = en_done * pass_total <= pass_done * en_total;
    const size_t j = take_e ? ei : pi;
    uint32_t &u = take_e ? eu : pu;
    if (first_seg[j] < 0) first_seg[j] = (int64_t)segs.size();
    segs.push_back(SvSeg{(uint32_t)j, u});
    u += (uint32_t)G;
    (take_e ? en_done : pass_done) += 1;
    if (u >= jobs[j].n_tiles) {
      end_seg[j] = (int64_t)segs.size();
      u = 0;
      if (take_e) ei++; else pi++;
    }
  }
  // every dependency lies wholly before its dependent (the launch drains)
  for (size_t j = 0; j < jobs.size(); j++) {
    const int d = jobs[j].dep;
    if (d >= 0 && jobs[j].n_tiles && jobs[d].n_tiles && end_seg[d] > first_seg[j])
      fail(QW_ERR_STATE, "internal: work list orders a job before its dependency");
  }
}

// ---------------------------------------------------------------------------
// prepare: allocate, upload, build launch descriptors
// ---------------------------------------------------------------------------
static void prepare(qw_plan *P) {
  Engine *E = P->eng;
  DeviceState *D = new DeviceState();
  D->arena.eng = E;
  P->dev = D;
  D->stream = (cudaStream_t)E->stream;
  cudaStream_t s = D->stream;
  const uint32_t nt = (uint32_t)P->tasks.size();

  // statevector programs
  SvTableBuilder b32(false), b64(true);
  D->mat_pass0.assign(P->mats.size(), 0);
  D->task_pass0.assign(nt, 0);
  D->ar_batch = plan_ar_batch(P);
  D->ar_chain = D->ar_batch == SV_AR_COMP ? SV_AR_REM : SV_AR_PLAIN;
  size_t rem_bytes = 0;      // largest FP32 chain launched pass by pass that keeps a remainder
  size_t mat_rem_bytes = 0;  // and boundary
  for (size_t m = 0; m < P->mats.size(); m++) {
    const MatNode &M = P->mats[m];
    if (M.mode == QW_MODE_TABLEAU) continue;
    D->mat_pass0[m] = (M.mode == QW_MODE_SV_FP64 ? b64 : b32).add(M.sv);
    const bool f64 = M.mode == QW_MODE_SV_FP64;
    const int ar = f64 ? SV_AR_PLAIN : D->ar_chain;
    const size_t S = sv_state_bytes(f64, M.n_eff);
    // algorithmic bytes of the boundary's passes (state, and the remainder between passes)
    P->prefix_alg_bytes += chain_bytes((double)S, M.sv.passes.size(), ar);
    for (const HostPass &hp : M.sv.passes) P->prefix_alg_flops += pass_flops(hp, M.n_eff, M.sv.g, ar);
    if (ar == SV_AR_REM && M.sv.passes.size() > 1) mat_rem_bytes = std::max(mat_rem_bytes, S);
  }
  for (uint32_t t = 0; t < nt; t++) {
    const TaskPlan &tp = P->tasks[t];
    if (tp.mode == QW_MODE_TABLEAU) continue;
    D->task_pass0[t] = (tp.mode == QW_MODE_SV_FP64 ? b64 : b32).add(tp.sv);
  }
  D->t32.passes = D->arena.upload(b32.passes, s);
  D->t32.stages = D->arena.upload(b32.stages, s);
  D->t32.ops = D->arena.upload(b32.ops32, s);
  D->t32.ops_lo = D->arena.upload(b32.ops32lo, s);
  D->t32.ph = D->arena.upload(b32.ph, s);
  D->t64.passes = D->arena.upload(b64.passes, s);
  D->t64.stages = D->arena.upload(b64.stages, s);
  D->t64.ops = D->arena.upload(b64.ops64, s);
  D->t64.ph = D->arena.upload(b64.ph64, s);

  // boundary store (budget was enforced by the planner)
  D->mat_buf.assign(P->mats.size(), nullptr);
  D->mat_export[0].assign(P->mats.size(), nullptr);
  D->mat_export[1].assign(P->mats.size(), nullptr);
  D->mat_basis.assign(P->mats.size(), nullptr);
  for (size_t m = 0; m < P->mats.size(); m++) {
    const MatNode &M = P->mats[m];
    if (M.mode == QW_MODE_TABLEAU) {
      const uint32_t W = (M.n + 63) / 64;
      D->mat_buf[m] = D->arena.alloc((size_t)2 * M.n * 2 * W * 8 + 2 * M.n + 64);
      if (M.export_modes) {
        if (M.n > QW_SV_MAX_QUBITS) fail(QW_ERR_STATE, "internal: tableau export above the statevector cap");
        D->mat_basis[m] = (StabBasis *)D->arena.alloc(sizeof(StabBasis));
        const uint32_t n_eff = std::max<uint32_t>(M.n, SV_G);
        for (uint32_t md = 0; md < 2; md++)
          if ((M.export_modes >> md) & 1u)
            D->mat_export[md][m] = D->arena.alloc(sv_state_bytes(md == QW_MODE_SV_FP64, n_eff));
      }
    } else {
      D->mat_buf[m] = D->arena.alloc(sv_state_bytes(M.mode == QW_MODE_SV_FP64, M.n_eff));
      // lower-precision copy for the consumers of another precision
      for (uint32_t md = 0; md < 2; md++)
        if (md != M.mode && ((M.export_modes >> md) & 1u))
          D->mat_export[md][m] = D->arena.alloc(sv_state_bytes(md == QW_MODE_SV_FP64, M.n_eff));
    }
  }
  // ---- statevector boundaries as dense-block programs (dense_boundaries) --
  D->mat_dense.assign(P->mats.size(), nullptr);
  P->dense_choices.clear();
  if (P->opts.dense_boundaries) {
    for (size_t m = 0; m < P->mats.size(); m++) {
      const MatNode &M = P->mats[m];
      if (M.mode == QW_MODE_TABLEAU || M.sv.passes.empty() || M.gates.empty()) continue;
      if (M.parent >= 0 && P->mats[M.parent].mode != M.mode) continue;
      const bool fp64 = M.mode == QW_MODE_SV_FP64;
      qw_dense_prog *dp = dense_prog_autotune(E, M.mode, M.n_eff, M.gates.data(), M.gates.size(), 0, QW_DENSE_AUTO);
      DenseChoice c;
      c.mat = (int)m;
      dense_prog_config(dp, &c.engine, &c.width, nullptr, &c.est_ms);
      c.blocks = (uint32_t)dense_prog_blocks(dp);
      c.over_budget = !fp64 && D->ar_chain == SV_AR_REM && c.blocks > DENSE_COMP_MAX_BLOCKS;
      bool use = P->opts.dense_boundaries == 2 && !c.over_budget;
      if (!use && !c.over_budget) {
        // both candidates timed once from |0...0> on a scratch state
        const size_t bytes = sv_state_bytes(fp64, M.n_eff), n_amp = (size_t)1 << M.n_eff;
        void *scratch = nullptr, *scratch_lo = nullptr;
        const int ar = fp64 ? SV_AR_PLAIN : D->ar_chain;
        CK(cudaMalloc(&scratch, bytes));
        if (ar == SV_AR_REM) CK(cudaMalloc(&scratch_lo, bytes));
        const SvTables &T = fp64 ? D->t64 : D->t32;
        cudaEvent_t e[4];
        for (auto &x : e) CK(cudaEventCreate(&x));
        CK(cudaEventRecord(e[0], s));
        const size_t np = M.sv.passes.size();
        for (size_t p = 0; p < np; p++)
          launch_sv_pass(fp64, T, D->mat_pass0[m] + (uint32_t)p, (uint32_t)M.sv.passes[p].q.size(), M.n_eff,
                         p == 0 ? nullptr : scratch, scratch, s, ar, (ar == SV_AR_REM && p > 0) ? scratch_lo : nullptr,
                         (ar == SV_AR_REM && p + 1 < np) ? scratch_lo : nullptr);
        CK(cudaEventRecord(e[1], s));
        CK(cudaEventRecord(e[2], s));
        basis_zero_kernel<<<(unsigned)std::min<size_t>((n_amp + 255) / 256, (size_t)E->sm_count * 16), 256, 0, s>>>(
            scratch, fp64, n_amp);
        dense_prog_run(dp, scratch, s);
        CK(cudaEventRecord(e[3], s));
        CK(cudaEventSynchronize(e[3]));
        float a = 0, b = 0;
        CK(cudaEventElapsedTime(&a, e[0], e[1]));
        CK(cudaEventElapsedTime(&b, e[2], e[3]));
        for (auto &x : e) cudaEventDestroy(x);
        cudaFree(scratch);
        if (scratch_lo) cudaFree(scratch_lo);
        dense_prog_check(dp);
        c.pass_ms = a;
        c.dense_ms = b;
        use = b < a;
      }
      c.used = use;
      P->dense_choices.push_back(c);
      if (use) D->mat_dense[m] = dp;
      else dense_prog_destroy(dp);
    }
  }

  // the state a statevector consumer of node m reads (the node itself, or its
  // export into the consumer's precision)
  auto sv_source = [&](int m, uint32_t mode) -> void * {
    if (P->mats[m].mode == mode) return D->mat_buf[m];
    return D->mat_export[mode][m] ? D->mat_export[mode][m] : D->mat_buf[m];
  };
  auto needs_convert = [&](const TaskPlan &tp) {
    return tp.src >= 0 && P->mats[tp.src].mode != QW_MODE_TABLEAU && P->mats[tp.src].mode != tp.mode &&
           !D->mat_export[tp.mode][tp.src];
  };

  // ---- statevector boundaries: one persistent launch per precision --------
  // Used when every boundary has passes and continues from |0...0> or from a
  // statevector boundary of its own precision (no export or conversion in
  // between); a boundary's first pass then waits for its parent's last, and
  // sibling boundaries run side by side.  Otherwise: pass by pass.
  uint64_t mat_rem = 0;  // remainder arrays of every boundary
  {
    bool ok = P->opts.batched != 0;
    size_t n_sv = 0;
    for (const qw_dense_prog *dp : D->mat_dense)
      if (dp) ok = false;  // a dense-block boundary is launched block by block
    for (const MatNode &M : P->mats) {
      if (M.mode == QW_MODE_TABLEAU) continue;
      n_sv++;
      if (M.sv.passes.empty()) ok = false;
      if (M.parent >= 0 && P->mats[M.parent].mode != M.mode) ok = false;
      // compensated FP32 boundaries keep their remainder between passes, an
      // array each in a persistent launch
      if (M.mode == QW_MODE_SV_FP32 && D->ar_chain == SV_AR_REM && M.sv.passes.size() > 1)
        mat_rem += sv_state_bytes(false, M.n_eff);
    }
    // beyond a small share of the budget: one array, pass by pass
    if (mat_rem > std::min<uint64_t>(MAT_REM_BYTES, E->task_budget / 8)) ok = false;
    // a single boundary is a chain of dependent passes: separate launches
    // serve it as well, without CTAs waiting on the previous pass
    ok = ok && n_sv > 1;
    if (!ok) {
      mat_rem = 0;
      rem_bytes = mat_rem_bytes;
    } else {
      std::vector<uint32_t> level(P->mats.size(), 0);
      uint32_t max_level = 0;
      size_t max_p = 0;
      for (size_t m = 0; m < P->mats.size(); m++) {  // parents precede their children
        const MatNode &M = P->mats[m];
        if (M.mode == QW_MODE_TABLEAU) continue;
        level[m] = (M.parent >= 0) ? level[M.parent] + 1 : 0;
        max_level = std::max(max_level, level[m]);
        max_p = std::max(max_p, M.sv.passes.size());
      }
      for (uint32_t prec : {(uint32_t)QW_MODE_SV_FP32, (uint32_t)QW_MODE_SV_FP64}) {
        std::vector<SvJob> jobs;
        std::vector<int> last_job(P->mats.size(), -1);
        const int ar = prec == QW_MODE_SV_FP32 ? D->ar_chain : SV_AR_PLAIN;
        std::vector<void *> rems(P->mats.size(), nullptr);
        if (ar == SV_AR_REM)
          for (size_t m = 0; m < P->mats.size(); m++)
            if (P->mats[m].mode == prec && P->mats[m].sv.passes.size() > 1)
              rems[m] = D->arena.alloc(sv_state_bytes(false, P->mats[m].n_eff));
        uint32_t kmax = 5;
        for (uint32_t L = 0; L <= max_level; L++)
          for (size_t pi = 0; pi < max_p; pi++)
            for (size_t m = 0; m < P->mats.size(); m++) {
              const MatNode &M = P->mats[m];
              if (M.mode != prec || level[m] != L || pi >= M.sv.passes.size()) continue;
              const uint32_t k = (uint32_t)M.sv.passes[pi].q.size();
              SvJob j{};
              j.src = (pi == 0) ? (M.parent >= 0 ? D->mat_buf[M.parent] : nullptr) : D->mat_buf[m];
              j.dst = D->mat_buf[m];
              j.pass = D->mat_pass0[m] + (uint32_t)pi;
              j.n_tiles = 1u << (M.n_eff - k);
              j.dep = (pi == 0) ? (M.parent >= 0 ? last_job[M.parent] : -1) : last_job[m];
              j.kind = SVJ_PASS;
              j.n = M.n_eff;
              j.src_lo = pi > 0 ? rems[m] : nullptr;
              j.dst_lo = pi + 1 < M.sv.passes.size() ? rems[m] : nullptr;
              last_job[m] = (int)jobs.size();
              jobs.push_back(j);
              kmax = std::max(kmax, k);
            }
        if (jobs.empty()) continue;
        DeviceState::MatBatch B;
        B.fp64 = prec == QW_MODE_SV_FP64;
        B.k_max = kmax;
        B.ar = ar;
        std::vector<uint64_t> tiles(max_level + 1, 0);  // of the siblings of each level
        for (size_t m = 0; m < P->mats.size(); m++)
          if (P->mats[m].mode == prec) tiles[level[m]] += 1ull << (P->mats[m].n_eff - std::min(P->mats[m].n_eff, kmax));
        B.few = *std::max_element(tiles.begin(), tiles.end()) <= SV_FEW_TILES;
        B.grid = sv_batch_grid(B.fp64, kmax, E->sm_count, ar, false, B.few);
        B.seg_bits = segment_bits(jobs);
        std::vector<SvSeg> segs;
        build_segments(jobs, jobs.size(), B.seg_bits, 2ull * (uint64_t)B.grid, segs);
        if (((uint64_t)segs.size() << B.seg_bits) > 0xFFFFFFF0ull)
          fail(QW_ERR_BUDGET, "the boundaries' work list exceeds 2^32 items");
        B.total_items = (uint32_t)(segs.size() << B.seg_bits);
        B.n_jobs = jobs.size();
        B.d_jobs = D->arena.upload(jobs, s);
        B.d_segs = D->arena.upload(segs, s);
        B.ctr_words = 2 + jobs.size();
        B.d_ctr = (unsigned int *)D->arena.alloc(B.ctr_words * sizeof(unsigned int));
        D->mat_batches.push_back(B);
      }
    }
  }

  // Hamiltonians
  std::vector<EnClass> cls;
  std::vector<EnGroup> grp;
  std::vector<EnTerm> trm;
  for (auto &H : P->hams) {
    D->ham_class_off.push_back((uint32_t)cls.size());
    const uint32_t goff = (uint32_t)grp.size(), toff = (uint32_t)trm.size();
    for (EnClass c : H.en.classes) {
      c.group_begin += goff;
      c.group_end += goff;
      cls.push_back(c);
    }
    for (EnGroup g : H.en.groups) {
      g.term_begin += toff;
      g.term_end += toff;
      grp.push_back(g);
    }
    trm.insert(trm.end(), H.en.terms.begin(), H.en.terms.end());
  }
  D->d_classes = D->arena.upload(cls, s);
  D->d_groups = D->arena.upload(grp, s);
  D->d_terms = D->arena.upload(trm, s);

  // results
  D->d_energy = (double *)D->arena.alloc(sizeof(double) * 2 * std::max<uint32_t>(nt, 1));
  P->sample_off.assign(nt + 1, 0);
  for (uint32_t t = 0; t < nt; t++) P->sample_off[t + 1] = P->sample_off[t] + P->tasks[t].shots;
  D->d_samples = (uint64_t *)D->arena.alloc(sizeof(uint64_t) * std::max<uint64_t>(1, P->sample_off[nt]));

  // ---- statevector tasks: buffers and waves --------------------------------
  D->task_state.assign(nt, nullptr);
  std::map<std::pair<int, uint32_t>, std::vector<uint32_t>> groups;  // (fp64, n_eff) -> tasks
  for (uint32_t t = 0; t < nt; t++) {
    const TaskPlan &tp = P->tasks[t];
    if (tp.mode == QW_MODE_TABLEAU) continue;
    groups[{tp.mode == QW_MODE_SV_FP64 ? 1 : 0, tp.n_eff}].push_back(t);
  }
  size_t max_partials = 1, max_smp_blocks = 1, max_src = 1;
  const bool batched = P->opts.batched != 0;
  // Compensated FP32 tasks with long programs keep their remainder between
  // passes.  Where a pass alone leaves much of the chip idle, several tasks
  // advance together in a persistent launch, each with its remainder array:
  // where its tiles take at most half of the resident CTAs (up to 19 qubits:
  // 64 tiles of 18 qubits left 86 % idle), or where they take two or three
  // rounds of them and the last is less than half full (21 and 22 qubits: 512
  // and 1024 tiles on 456 CTAs).  Other registers run one task after another,
  // pass by pass.  From 23 qubits on they fill the chip alone; 20 qubits (256
  // tiles) would leave 44 % of it idle, but sharing there makes a rerun of two
  // tasks cheaper than Eq. 2, which prices passes of one state, estimates it.
  auto long_chain = [&](const TaskPlan &tp) { return batched && tp.chain; };
  const uint32_t rem_slots = (uint32_t)sv_batch_grid(false, SV_MAX_TILE_FP32_REM, E->sm_count, SV_AR_REM);
  auto shares_launch = [&](const TaskPlan &tp) {
    if (tp.sv.passes.empty()) return false;
    const uint64_t tiles = 1ull << (tp.n_eff - (uint32_t)tp.sv.passes[0].q.size());
    const uint64_t rounds = (tiles + rem_slots - 1) / rem_slots, last = tiles - (rounds - 1) * rem_slots;
    return 2 * tiles <= rem_slots || ((rounds == 2 || rounds == 3) && 2 * last < rem_slots);
  };
  // Task buffers of every group coexist for the plan's lifetime, so the
  // groups share one task budget: each group with pooled tasks gets one
  // buffer, then the rest of the budget goes to the groups in order of
  // state size (smallest first) for up to one buffer per pooled task, and
  // for up to one state and remainder per long chain.
  std::map<std::pair<int, uint32_t>, size_t> pool_size, long_size;
  {
    std::map<std::pair<int, uint32_t>, size_t> n_long;
    std::map<std::pair<int, uint32_t>, bool> n_share;
    std::vector<std::pair<size_t, std::pair<int, uint32_t>>> order;  // (S, group)
    std::map<std::pair<int, uint32_t>, size_t> n_pooled;
    uint64_t committed = mat_rem;  // the boundaries' remainder arrays come out of it too
    for (auto &g : groups) {
      size_t np = 0, nl = 0;
      bool pooled_long = false;
      for (uint32_t t : g.second) {
        const TaskPlan &tp = P->tasks[t];
        if (tp.sv.passes.empty() && !needs_convert(tp)) continue;
        if (long_chain(tp)) {
          nl++;
          n_share[g.first] = shares_launch(tp);
          pooled_long = pooled_long || !(tp.flags & QW_TASK_KEEP_STATE);
        } else if (!(tp.flags & QW_TASK_KEEP_STATE)) {
          np++;
        }
      }
      if (pooled_long && np == 0) np = 1;
      const size_t S = sv_state_bytes(g.first.first != 0, g.first.second);
      n_pooled[g.first] = np;
      n_long[g.first] = nl;
      pool_size[g.first] = np ? 1 : 0;
      long_size[g.first] = nl ? 1 : 0;
      if (np) committed += S;
      if (nl) committed += S;  // the remainder of one chain
      if (np || nl) order.push_back({S, g.first});
    }
    std::sort(order.begin(), order.end());
    uint64_t left = E->task_budget > committed ? E->task_budget - committed : 0;
    for (auto &o : order) {
      if (!batched) break;
      const size_t S = o.first;
      const size_t np = n_pooled[o.second], nl = n_long[o.second];
      const size_t extra = std::min<size_t>(np ? np - 1 : 0, (size_t)(left / S));
      pool_size[o.second] += extra;
      left -= (uint64_t)extra * S;
      // chains share the pooled states (their waves run at other times)
      for (size_t k = 1; k < nl && n_share[o.second]; k++) {
        const size_t need = S + (long_size[o.second] >= pool_size[o.second] ? S : 0);
        if (left < need) break;
        left -= need;
        long_size[o.second]++;
        pool_size[o.second] = std::max(pool_size[o.second], long_size[o.second]);
      }
    }
  }
  for (auto &g : groups) {
    const bool fp64 = g.first.first != 0;
    const uint32_t n_eff = g.first.second;
    const size_t S = sv_state_bytes(fp64, n_eff);
    std::vector<uint32_t> own, shared_src;
    for (uint32_t t : g.second) {
      const TaskPlan &tp = P->tasks[t];
      const bool convert = needs_convert(tp);
      if (!tp.sv.passes.empty() || convert) own.push_back(t);
      else { shared_src.push_back(t); D->task_state[t] = sv_source(tp.src, tp.mode); }
    }
    // KEEP_STATE tasks get dedicated buffers; the others share a pool
    std::vector<uint32_t> pooled;
    for (uint32_t t : own) {
      if (P->tasks[t].flags & QW_TASK_KEEP_STATE) D->task_state[t] = D->arena.alloc(S);
      else pooled.push_back(t);
    }
    // waves: dedicated tasks first (one wave), then pooled chunks; long
    // compensated chains one task per wave, launched pass by pass
    std::vector<uint32_t> dedicated, ded_short, pool_short, longs;
    for (uint32_t t : own) if (P->tasks[t].flags & QW_TASK_KEEP_STATE) dedicated.push_back(t);
    for (uint32_t t : dedicated) (long_chain(P->tasks[t]) ? longs : ded_short).push_back(t);
    bool pooled_long = false;
    for (uint32_t t : pooled) {
      if (long_chain(P->tasks[t])) { longs.push_back(t); pooled_long = true; }
      else pool_short.push_back(t);
    }
    const size_t long_n = std::min(long_size[g.first], longs.size());
    const size_t pool_n = std::min(pool_size[g.first], std::max(pool_short.size(), pooled_long ? long_n : (size_t)0));
    std::vector<void *> pool(pool_n);
    for (auto &p : pool) p = D->arena.alloc(S);
    // remainder arrays of the chains of one wave (a single chain at a time
    // shares the boundaries' array, as it is launched pass by pass)
    std::vector<void *> rems(long_n > 1 ? long_n : 0);
    for (auto &p : rems) p = D->arena.alloc(S);
    std::vector<std::pair<std::vector<uint32_t>, bool>> wave_tasks;  // (tasks, per-pass launches)
    if (batched) {
      if (!ded_short.empty()) wave_tasks.push_back({ded_short, false});
      for (size_t i = 0; i < pool_short.size(); i += pool_n)
        wave_tasks.push_back({std::vector<uint32_t>(pool_short.begin() + i,
                                                    pool_short.begin() + std::min(pool_short.size(), i + pool_n)),
                              false});
      const size_t lw = std::max<size_t>(1, long_n);
      for (size_t i = 0; i < longs.size(); i += lw)
        wave_tasks.push_back({std::vector<uint32_t>(longs.begin() + i, longs.begin() + std::min(longs.size(), i + lw)),
                              lw == 1});
    } else {
      for (uint32_t t : own) wave_tasks.push_back({{t}, true});
    }
    if (wave_tasks.empty()) wave_tasks.push_back({{}, !batched});
    for (size_t w = 0; w < wave_tasks.size(); w++) {
      Wave W;
      W.fp64 = fp64;
      W.per_pass = wave_tasks[w].second;
      W.tasks = wave_tasks[w].first;
      const bool chains = !W.tasks.empty() && long_chain(P->tasks[W.tasks[0]]);  // (a wave holds one kind)
      W.ar = fp64 ? SV_AR_PLAIN : (W.per_pass || chains ? D->ar_chain : D->ar_batch);
      uint32_t kmax = 5;
      for (size_t i = 0; i < W.tasks.size(); i++) {
        const uint32_t t = W.tasks[i];
        if (!(P->tasks[t].flags & QW_TASK_KEEP_STATE)) D->task_state[t] = pool[i % std::max<size_t>(1, pool_n)];
        for (const HostPass &hp : P->tasks[t].sv.passes) kmax = std::max<uint32_t>(kmax, (uint32_t)hp.q.size());
      }
      W.k_max = kmax;
      {
        uint32_t b_first = 0;
        for (uint32_t t : W.tasks)
          if (!P->tasks[t].sv.passes.empty()) { b_first = P->tasks[t].sv.passes[0].b; break; }
        P->wave_tiles.push_back({kmax, b_first});
      }
      W.obs_tasks = W.tasks;
      if (w == 0) W.obs_tasks.insert(W.obs_tasks.end(), shared_src.begin(), shared_src.end());
      // jobs, round-robin over pass index within windows of tasks
      std::map<uint32_t, int> last_pass;  // task -> its last pass job
      uint32_t window = P->opts.window ? P->opts.window : (uint32_t)W.tasks.size();
      window = std::max<uint32_t>(1, window);
      for (size_t w0 = 0; w0 < W.tasks.size(); w0 += window) {
        const size_t w1 = std::min(W.tasks.size(), w0 + window);
        size_t max_p = 0;
        for (size_t i = w0; i < w1; i++) max_p = std::max(max_p, P->tasks[W.tasks[i]].sv.passes.size());
        std::vector<int> last(W.tasks.size(), -1);
        for (size_t p = 0; p < max_p; p++) {
          for (size_t i = w0; i < w1; i++) {
            const uint32_t t = W.tasks[i];
            const TaskPlan &tp = P->tasks[t];
            if (p >= tp.sv.passes.size()) continue;
            SvJob j{};
            const bool convert = needs_convert(tp);
            j.src = (p == 0 && !convert) ? (tp.src >= 0 ? sv_source(tp.src, tp.mode) : nullptr) : D->task_state[t];
            j.dst = D->task_state[t];
            j.pass = D->task_pass0[t] + (uint32_t)p;
            j.n_tiles = 1u << (tp.n_eff - (uint32_t)tp.sv.passes[p].q.size());
            P->batch_alg_flops += pass_flops(tp.sv.passes[p], tp.n_eff, tp.sv.g, W.ar);
            j.dep = last[i];
            j.kind = SVJ_PASS;
            j.n = tp.n_eff;
            if (chains && !W.per_pass) {
              j.src_lo = p > 0 ? rems[i] : nullptr;
              j.dst_lo = p + 1 < tp.sv.passes.size() ? rems[i] : nullptr;
            }
            last[i] = (int)W.jobs.size();
            last_pass[t] = (int)W.jobs.size();
            W.jobs.push_back(j);
          }
        }
      }
      for (uint32_t t : W.tasks) {
        const TaskPlan &tp = P->tasks[t];
        if (needs_convert(tp)) W.converts.push_back({t, {D->mat_buf[tp.src], D->task_state[t]}});
      }
      // energy jobs
      for (uint32_t t : W.obs_tasks) {
        const TaskPlan &tp = P->tasks[t];
        if (tp.ham < 0) continue;
        const HamLayout &H = P->hams[tp.ham];
        EnJob j{};
        j.state = D->task_state[t];
        j.out = D->d_energy + 2 * (size_t)t;
        j.n = H.n_eff;
        j.rep_bits = H.en.rep_bits;
        j.iter_bits = H.en.iter_bits;
        j.class_begin = D->ham_class_off[tp.ham];
        j.n_classes = (uint32_t)H.en.classes.size();
        j.block_begin = W.en_blocks;
        j.n_blocks = H.en.n_blocks;
        W.en_blocks += H.en.n_blocks;
        W.en.push_back(j);
        W.obs_tasks_en.push_back(t);
      }
      max_partials = std::max<size_t>(max_partials, W.en_blocks);
      // sampling sources (deduplicated by state) and shots
      std::map<const void *, uint32_t> sid;
      for (uint32_t t : W.obs_tasks) {
        const TaskPlan &tp = P->tasks[t];
        if (!tp.shots) continue;
        const void *st = D->task_state[t];
        auto it = sid.find(st);
        uint32_t si;
        if (it == sid.end()) {
          SmpSource so{};
          so.state = st;
          so.n = tp.n_eff;
          so.n_blocks = (tp.n_eff >= (uint32_t)SMP_BLOCK_BITS) ? (1u << (tp.n_eff - SMP_BLOCK_BITS)) : 1u;
          so.block_begin = W.smp_blocks;
          W.smp_blocks += so.n_blocks;
          si = (uint32_t)W.src.size();
          W.src.push_back(so);
          sid[st] = si;
        } else {
          si = it->second;
        }
        for (uint32_t k = 0; k < tp.shots; k++) {
          SmpShot q{};
          q.u = tp.uniforms[k];
          q.source = si;
          q.out = D->d_samples + P->sample_off[t] + k;
          W.shots.push_back(q);
        }
      }
      max_smp_blocks = std::max<size_t>(max_smp_blocks, W.smp_blocks);
      max_src = std::max<size_t>(max_src, W.src.size());
      // algorithmic bytes: every pass reads and writes its state once; the
      // energy of a task reads every amplitude once per term class
      if (W.ar == SV_AR_REM) {
        for (uint32_t t : W.tasks) P->batch_alg_bytes += chain_bytes((double)S, P->tasks[t].sv.passes.size(), W.ar);
        if (W.per_pass && W.jobs.size() > 1) rem_bytes = std::max(rem_bytes, S);
      } else {
        for (const SvJob &j : W.jobs) { (void)j; P->batch_alg_bytes += 2.0 * (double)S; }
      }
      for (size_t e = 0; e < W.en.size(); e++) {
        const EnJob &j = W.en[e];
        const double Sj = (double)sv_state_bytes(fp64, j.n);
        P->energy_alg_bytes += (double)j.n_classes * Sj;
        // L2 -> SM reads: the state once per group of terms
        P->energy_l2_bytes += (double)P->hams[P->tasks[W.obs_tasks_en[e]].ham].en.groups.size() * Sj;
      }
      // persistent work list: pass jobs, then (fused) the energy jobs,
      // released in the order their states finish
      std::vector<SvJob> up = W.jobs;
      W.fused_energy =
          !W.per_pass && W.ar != SV_AR_REM && P->opts.fuse_energy && !W.en.empty() && sv_threads_for_k(W.k_max, W.ar, fp64) == 128;
      W.few = ((uint64_t)W.tasks.size() << (n_eff - std::min(n_eff, W.k_max))) <= SV_FEW_TILES;
      W.grid = !W.per_pass ? sv_batch_grid(fp64, W.k_max, E->sm_count, W.ar, W.fused_energy, W.few) : 0;
      if (W.fused_energy) {
        std::vector<SvJob> ej;
        for (size_t e = 0; e < W.en.size(); e++) {
          SvJob j{};
          const uint32_t t = W.obs_tasks_en[e];
          auto it = last_pass.find(t);
          j.dep = (it == last_pass.end()) ? -1 : it->second;
          j.kind = SVJ_ENERGY;
          j.pass = (uint32_t)e;
          j.n_tiles = W.en[e].n_blocks;
          j.n = W.en[e].n;
          ej.push_back(j);
        }
        std::stable_sort(ej.begin(), ej.end(), [](const SvJob &a, const SvJob &b) { return a.dep < b.dep; });
        up.insert(up.end(), ej.begin(), ej.end());
      }
      if (!W.per_pass) {
        W.seg_bits = segment_bits(up);
        build_segments(up, W.jobs.size(), W.seg_bits, 2ull * (uint64_t)W.grid, W.segs);
        if (((uint64_t)W.segs.size() << W.seg_bits) > 0xFFFFFFF0ull)
          fail(QW_ERR_BUDGET, "a wave's work list exceeds 2^32 items; lower task_budget");
        W.total_items = (uint32_t)(W.segs.size() << W.seg_bits);
        if (W.fused_energy) P->energy_fused = true;
      }
      // With fault injection (tests only) the first job waits on an extra
      // job that has no segment, so no CTA ever takes it: its counter never
      // reaches the one unit it needs and the bounded wait runs out.
      if (P->opts.fault_injection && !W.per_pass && !up.empty()) {
        SvJob ph{};
        ph.n_tiles = 1;
        ph.dep = -1;
        up[0].dep = (int32_t)up.size();
        up.push_back(ph);
      }
      W.d_jobs = D->arena.upload(up, s);
      W.d_segs = D->arena.upload(W.segs, s);
      W.ctr_words = 2 + up.size();
      W.d_ctr = (unsigned int *)D->arena.alloc(W.ctr_words * sizeof(unsigned int));
      CK(cudaMemsetAsync(W.d_ctr, 0, W.ctr_words * sizeof(unsigned int), s));
      W.d_en = D->arena.upload(W.en, s);
      W.d_src = D->arena.upload(W.src, s);
      W.d_shots = D->arena.upload(W.shots, s);
      D->waves.push_back(std::move(W));
    }
  }
  D->d_partials = (double *)D->arena.alloc(sizeof(double) * 2 * max_partials);
  if (rem_bytes) D->rem = D->arena.alloc(rem_bytes);
  D->d_bsum = (double *)D->arena.alloc(sizeof(double) * max_smp_blocks);
  D->d_blast = (int32_t *)D->arena.alloc(sizeof(int32_t) * max_smp_blocks);
  D->d_boff = (double *)D->arena.alloc(sizeof(double) * (max_smp_blocks + max_src));
  D->d_lastnz = (int64_t *)D->arena.alloc(sizeof(int64_t) * max_src);

  // ---- tableau --------------------------------------------------------------
  std::vector<TabProgram> progs;
  std::vector<TabLayer> layers;
  std::vector<TabSlot> slots;
  for (const TabHostProgram &hp : P->tab_progs) {
    TabProgram pg{};
    pg.layer_begin = (uint32_t)layers.size();
    pg.n_layers = (uint32_t)hp.layers.size();
    pg.n_bits = hp.n_bits;
    pg.n_outs = hp.n_outs;
    const uint32_t soff = (uint32_t)slots.size();
    for (TabLayer L : hp.layers) { L.slot_begin += soff; layers.push_back(L); }
    slots.insert(slots.end(), hp.slots.begin(), hp.slots.end());
    progs.push_back(pg);
  }
  bool any_tab = !P->tab_progs.empty();
  if (any_tab) {
    D->d_progs = D->arena.upload(progs, s);
    D->d_layers = D->arena.upload(layers, s);
    D->d_slots = D->arena.upload(slots, s);
    D->d_bits = D->arena.upload(P->tab_bits, s);
    // outcome layout
    P->outs_off.assign(nt + 1, 0);
    for (uint32_t t = 0; t < nt; t++) P->outs_off[t + 1] = P->outs_off[t] + P->tasks[t].tab_outs;
    P->outs_mat_off.assign(P->mats.size() + 1, 0);
    for (size_t m = 0; m < P->mats.size(); m++) P->outs_mat_off[m + 1] = P->outs_mat_off[m] + P->mats[m].tab_outs;
    D->d_outs = (uint8_t *)D->arena.alloc(std::max<uint32_t>(1, P->outs_off[nt]));
    D->d_mat_outs = (uint8_t *)D->arena.alloc(std::max<uint32_t>(1, P->outs_mat_off[P->mats.size()]));
    auto sign_of = [](uint64_t *rows, uint32_t n) {
      return rows ? (uint8_t *)(rows + (size_t)2 * n * 2 * ((n + 63) / 64)) : nullptr;
    };
    auto add_launch = [&](std::vector<DeviceState::TabLaunch> &dst, uint32_t n, const std::vector<TabTaskDesc> &descs,
                          const std::vector<TabSegment> &segs, uint8_t *outs) {
      TabArgs a{};
      a.n = n;
      a.W = (n + 63) / 64;
      a.rows = 2 * n;
      a.tasks = D->arena.upload(descs, s);
      a.segs = D->arena.upload(segs, s);
      a.progs = D->d_progs;
      a.layers = D->d_layers;
      a.slots = D->d_slots;
      a.bits = D->d_bits;
      a.outs = outs;
      dst.push_back({a, (uint32_t)descs.size(), -1});
    };
    // appends one CTA: its segments (outcomes relative to out_base) and descriptor
    auto add_desc = [&](std::vector<TabTaskDesc> &descs, std::vector<TabSegment> &segs,
                        const std::vector<std::pair<uint32_t, uint32_t>> &tab_segs, uint32_t out_base,
                        const void *init, uint64_t *out_rows, uint8_t *out_sign) {
      TabTaskDesc d{};
      d.seg_begin = (uint32_t)segs.size();
      d.n_segs = (uint32_t)tab_segs.size();
      d.out_base = out_base;
      d.init_rows = (const uint64_t *)init;
      d.out_rows = out_rows;
      d.out_sign = out_sign;
      uint32_t oo = 0;
      for (auto &sg : tab_segs) {
        segs.push_back({sg.first, sg.second, oo, 0});
        oo += P->tab_progs[sg.first].n_outs;
      }
      descs.push_back(d);
    };
    // Boundaries: every boundary of one register size whose parent is ready
    // runs in one launch, a CTA each (level by level; parents precede their
    // children in the list).  A launch per boundary left one SM busy at a
    // time: 129 boundaries of a random-outcome workload took 129 launches.
    {
      std::vector<uint32_t> level(P->mats.size(), 0);
      std::map<std::pair<uint32_t, uint32_t>, std::vector<size_t>> by_level;  // (level, n) -> boundaries
      for (size_t m = 0; m < P->mats.size(); m++) {
        const MatNode &M = P->mats[m];
        if (M.mode != QW_MODE_TABLEAU) continue;
        if (M.parent >= 0) level[m] = level[M.parent] + 1;
        by_level[{level[m], M.n}].push_back(m);
      }
      for (auto &lv : by_level) {
        std::vector<TabTaskDesc> descs;
        std::vector<TabSegment> segs;
        const uint32_t n = lv.first.second;
        for (size_t m : lv.second) {
          const MatNode &M = P->mats[m];
          uint64_t *out = (uint64_t *)D->mat_buf[m];
          add_desc(descs, segs, M.tab_segs, P->outs_mat_off[m], M.parent >= 0 ? D->mat_buf[M.parent] : nullptr, out,
                   sign_of(out, n));
        }
        add_launch(D->tab_mat_launches, n, descs, segs, D->d_mat_outs);
      }
    }
    // Tasks: those of one register size run in one launch, each from its own
    // boundary, except Pauli-frame groups, whose launch is gated by their
    // own reference run
    std::map<std::pair<int, uint32_t>, std::vector<uint32_t>> by_src;
    for (uint32_t t = 0; t < nt; t++)
      if (P->tasks[t].mode == QW_MODE_TABLEAU)
        by_src[{P->task_frame_group[t] >= 0 ? P->tasks[t].src : -1, P->tasks[t].n}].push_back(t);
    D->tab_keep.assign(nt, {nullptr, nullptr});
    for (auto &g : by_src) {
      std::vector<TabTaskDesc> descs;
      std::vector<TabSegment> segs;
      const uint32_t kn = g.first.second;
      const size_t kwords = (size_t)2 * kn * 2 * ((kn + 63) / 64);
      for (uint32_t t : g.second) {
        const TaskPlan &tp = P->tasks[t];
        uint64_t *keep = nullptr;  // final tableau of a task that keeps its state
        if (tp.flags & QW_TASK_KEEP_STATE) {
          keep = (uint64_t *)D->arena.alloc(kwords * 8 + 2 * kn);
          D->tab_keep[t] = {keep, sign_of(keep, kn)};
        }
        add_desc(descs, segs, tp.tab_segs, P->outs_off[t], tp.src >= 0 ? D->mat_buf[tp.src] : nullptr, keep,
                 sign_of(keep, kn));
      }
      add_launch(D->tab_task_launches, kn, descs, segs, D->d_outs);
      const int fg = P->task_frame_group[g.second[0]];
      if (fg >= 0) {
        // Pauli frames: the reference suffix once on the tableau, then the
        // frame launch; the per-task launch above runs only if a reference
        // outcome was random (decided on the device, no host round trip)
        const FrameGroup &G = P->frame_groups[fg];
        if (G.tasks != g.second) fail(QW_ERR_STATE, "internal: frame group and tableau group differ");
        uint8_t *ref_out = (uint8_t *)D->arena.alloc(std::max<uint32_t>(1, G.n_outs));
        uint32_t *rand = (uint32_t *)D->arena.alloc(sizeof(uint32_t));
        std::vector<TabSegment> rsegs;
        std::vector<TabTaskDesc> rd;
        add_desc(rd, rsegs, G.ref_segs, 0, D->mat_buf[G.src], nullptr, nullptr);
        std::vector<DeviceState::TabLaunch> tmp;
        add_launch(tmp, G.n, rd, rsegs, ref_out);
        DeviceState::FrameLaunch fl{};
        fl.ref = tmp[0].a;
        fl.ref.rand_any = rand;
        FrameArgs &fa = fl.fa;
        fa.n = G.n;
        fa.n_tasks = (uint32_t)G.tasks.size();
        fa.n_words = G.n_words;
        fa.n_layers = (uint32_t)G.prog.layers.size();
        fa.layers = D->arena.upload(G.prog.layers, s);
        fa.ops = D->arena.upload(G.prog.ops, s);
        fa.ev_x = D->arena.upload(G.ev_x, s);
        fa.ev_z = D->arena.upload(G.ev_z, s);
        fa.ref_out = ref_out;
        fa.rand_any = rand;
        std::vector<uint32_t> ob;
        for (uint32_t t : G.tasks) ob.push_back(P->outs_off[t]);
        fa.out_base = D->arena.upload(ob, s);
        fa.outs = D->d_outs;
        D->tab_task_launches.back().a.run_if = rand;
        D->tab_task_launches.back().frame = (int)D->frame_launches.size();
        D->frame_launches.push_back(fl);
      }
    }
  }
  for (auto &e : D->ev) CK(cudaEventCreate(&e));
  CK(cudaStreamSynchronize(s));
  P->h2d_bytes = D->arena.h2d;
  P->d2h_bytes = 16ull * nt + 8ull * P->sample_off[nt] +
                 (any_tab ? (uint64_t)P->outs_off[nt] + P->outs_mat_off[P->mats.size()] : 0ull);
}

// ---------------------------------------------------------------------------
// launch sequence of a prepared plan (captured once into a graph)
// ---------------------------------------------------------------------------
static void enqueue(qw_plan *P, cudaStream_t s, bool capturing) {
  DeviceState *D = P->dev;
  uint64_t nl = 0;  // kernels launched by one execution
  // timing events: inside a capture they become external event-record nodes
  auto rec = [&](cudaEvent_t e) {
    return capturing ? cudaEventRecordWithFlags(e, s, cudaEventRecordExternal) : cudaEventRecord(e, s);
  };
  CK(rec(D->ev[0]));
  // 1) shared prefixes (boundary states): the tableaus level by level, then
  // the statevectors in creation order (parents first)
  for (const DeviceState::TabLaunch &L : D->tab_mat_launches) {
    launch_tab(L.a, L.n_tasks, s);
    nl += 1;
  }
  for (size_t m = 0; m < P->mats.size(); m++) {
    const MatNode &M = P->mats[m];
    if (M.mode == QW_MODE_TABLEAU) {
      // Table II STAB -> SV: the statevectors its consumers continue from
      for (uint32_t md = 0; md < 2; md++)
        if (D->mat_export[md][m]) {
          launch_stab_export(D->mat_buf[m], M.n, D->mat_basis[m], md == QW_MODE_SV_FP64,
                             std::max<uint32_t>(M.n, SV_G), D->mat_export[md][m], P->eng->sm_count, s);
          nl += 2;
        }
      continue;
    }
    if (!D->mat_batches.empty()) continue;  // statevector boundaries run in the batches below
    const bool fp64 = M.mode == QW_MODE_SV_FP64;
    const SvTables &T = fp64 ? D->t64 : D->t32;
    const void *psrc = nullptr;
    if (M.parent >= 0) {
      const MatNode &PM = P->mats[M.parent];
      if (PM.mode == M.mode) psrc = D->mat_buf[M.parent];
      else psrc = D->mat_export[M.mode][M.parent];
    }
    if (D->mat_dense[m]) {
      const size_t n_amp = (size_t)1 << M.n_eff;
      if (psrc) launch_copy(psrc, D->mat_buf[m], sv_state_bytes(fp64, M.n_eff), s);
      else
        basis_zero_kernel<<<(unsigned)std::min<size_t>((n_amp + 255) / 256, (size_t)P->eng->sm_count * 16), 256, 0,
                            s>>>(D->mat_buf[m], fp64, n_amp);
      dense_prog_run(D->mat_dense[m], D->mat_buf[m], s);
      nl += 1 + dense_prog_blocks(D->mat_dense[m]);
    } else if (M.sv.passes.empty()) {
      if (psrc) launch_copy(psrc, D->mat_buf[m], sv_state_bytes(fp64, M.n_eff), s);
    } else {
      // compensated FP32: the remainder stays in D->rem between the passes
      // and the last pass rounds the state once, into the boundary
      const int ar = fp64 ? SV_AR_PLAIN : D->ar_chain;
      const size_t np = M.sv.passes.size();
      nl += np;
      for (size_t p = 0; p < np; p++) {
        launch_sv_pass(fp64, T, D->mat_pass0[m] + (uint32_t)p, (uint32_t)M.sv.passes[p].q.size(), M.n_eff,
                       p == 0 ? psrc : D->mat_buf[m], D->mat_buf[m], s, ar, chain_src_lo(D, ar, p),
                       chain_dst_lo(D, ar, p, np));
      }
    }
    // the boundary rounded once into the other precision its consumers use
    for (uint32_t md = 0; md < 2; md++)
      if (md != M.mode && D->mat_export[md][m]) {
        const size_t n = (size_t)1 << M.n_eff;
        convert_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(D->mat_buf[m], fp64, D->mat_export[md][m],
                                                                  md == QW_MODE_SV_FP64, n);
        nl += 1;
      }
  }
  if (!D->mat_batches.empty()) {
    for (const DeviceState::MatBatch &B : D->mat_batches) {
      CK(cudaMemsetAsync(B.d_ctr, 0, B.ctr_words * sizeof(unsigned int), s));
      launch_sv_batch(B.fp64, B.fp64 ? D->t64 : D->t32, B.d_jobs, B.d_segs, B.seg_bits, B.total_items, B.k_max,
                      B.d_ctr, EnTables{}, B.grid, s, B.ar, B.few);
      nl += 1;
    }
    // each boundary rounded once into the other precision its consumers use
    for (size_t m = 0; m < P->mats.size(); m++) {
      const MatNode &M = P->mats[m];
      if (M.mode == QW_MODE_TABLEAU) continue;
      for (uint32_t md = 0; md < 2; md++)
        if (md != M.mode && D->mat_export[md][m]) {
          const size_t n = (size_t)1 << M.n_eff;
          convert_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
              D->mat_buf[m], M.mode == QW_MODE_SV_FP64, D->mat_export[md][m], md == QW_MODE_SV_FP64, n);
          nl += 1;
        }
    }
  }
  CK(rec(D->ev[1]));
  // 2) task suffixes, observables
  size_t wi = 0;
  for (auto &W : D->waves) {
    const SvTables &T = W.fp64 ? D->t64 : D->t32;
    CK(rec(D->wave_ev[4 * wi]));
    nl += W.converts.size();
    for (auto &c : W.converts) {
      const TaskPlan &tp = P->tasks[c.first];
      const size_t n = (size_t)1 << tp.n_eff;
      convert_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
          c.second.first, P->mats[tp.src].mode == QW_MODE_SV_FP64, c.second.second, W.fp64, n);
    }
    if (!W.per_pass) {
      if (W.total_items) {
        CK(cudaMemsetAsync(W.d_ctr, 0, W.ctr_words * sizeof(unsigned int), s));
        const EnTables et =
            W.fused_energy ? EnTables{W.d_en, D->d_classes, D->d_groups, D->d_terms, D->d_partials} : EnTables{};
        launch_sv_batch(W.fp64, T, W.d_jobs, W.d_segs, W.seg_bits, W.total_items, W.k_max, W.d_ctr, et,
                        W.grid, s, W.ar, W.few);
        nl += 1;
      }
    } else {
      // one task per wave, its passes in order (SV_AR_REM: one rounding, at the end)
      nl += W.jobs.size();
      for (size_t i = 0; i < W.jobs.size(); i++) {
        const SvJob &j = W.jobs[i];
        const uint32_t k = j.n - (uint32_t)std::log2((double)j.n_tiles);
        launch_sv_pass(W.fp64, T, j.pass, k, j.n, j.src, j.dst, s, W.ar, chain_src_lo(D, W.ar, i),
                       chain_dst_lo(D, W.ar, i, W.jobs.size()));
      }
    }
    CK(rec(D->wave_ev[4 * wi + 1]));
    if (W.fused_energy) {
      launch_energy_reduce(W.d_en, (uint32_t)W.en.size(), D->d_partials, s);
      nl += 1;
    } else {
      const EnTables et{W.d_en, D->d_classes, D->d_groups, D->d_terms, D->d_partials};
      launch_energy(W.fp64, !W.fp64, et, (uint32_t)W.en.size(), W.en_blocks, W.en.empty() ? 0u : W.en[0].rep_bits, s);
      if (!W.en.empty()) nl += 2;
    }
    if (!W.src.empty()) nl += W.shots.empty() ? 2 : 3;
    CK(rec(D->wave_ev[4 * wi + 2]));
    launch_sampling(W.fp64, W.d_src, (uint32_t)W.src.size(), W.smp_blocks, D->d_bsum, D->d_blast, D->d_boff,
                    D->d_lastnz, W.d_shots, (uint32_t)W.shots.size(), s);
    CK(rec(D->wave_ev[4 * wi + 3]));
    wi++;
  }
  CK(rec(D->ev[2]));
  // 3) tableau tasks
  for (auto &L : D->tab_task_launches) {
    if (L.frame >= 0) {
      const DeviceState::FrameLaunch &F = D->frame_launches[L.frame];
      launch_tab(F.ref, 1, s);
      launch_frames(F.fa, s);
      nl += 2;
    }
    launch_tab(L.a, L.n_tasks, s);
  }
  nl += D->tab_task_launches.size();
  CK(rec(D->ev[3]));
  P->n_launches = nl;
  CK(cudaGetLastError());
}

void plan_execute(qw_plan *P, void *stream) {
  Engine *E = P->eng;
  if (!E) fail(QW_ERR_STATE, "plan has no engine (created without one, or its engine was destroyed)");
  CK(cudaSetDevice(E->device));
  const auto t0 = std::chrono::steady_clock::now();
  if (!P->dev) {
    prepare(P);
    P->t_upload_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    DeviceState *D = P->dev;
    for (size_t w = 0; w < 4 * D->waves.size(); w++) {
      cudaEvent_t e;
      CK(cudaEventCreate(&e));
      D->wave_ev.push_back(e);
    }
  }
  DeviceState *D = P->dev;
  cudaStream_t s = stream ? (cudaStream_t)stream : D->stream;
  if (P->opts.use_graph) {
    if (!D->gexec) {
      cudaStream_t cs = D->stream;
      CK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
      try {
        enqueue(P, cs, true);
      } catch (...) {
        cudaGraph_t g = nullptr;
        if (cudaStreamEndCapture(cs, &g) == cudaSuccess && g) cudaGraphDestroy(g);
        cudaGetLastError();
        throw;
      }
      CK(cudaStreamEndCapture(cs, &D->graph));
      CK(cudaGraphInstantiate(&D->gexec, D->graph, 0));
    }
    CK(cudaGraphLaunch(D->gexec, s));
  } else {
    enqueue(P, s, false);
  }
  P->executed = true;
}

void plan_wait(qw_plan *P) {
  DeviceState *D = P->dev;
  if (!D || !P->eng) fail(QW_ERR_STATE, "qw_wait before qw_execute, or the engine was destroyed");
  CK(cudaSetDevice(P->eng->device));
  CK(cudaEventSynchronize(D->ev[3]));
  CK(cudaGetLastError());
  const uint32_t nt = (uint32_t)P->tasks.size();
  // device error flags of the persistent launches
  for (auto &W : D->waves) {
    if (!W.total_items || W.per_pass) continue;
    unsigned int flag = 0;
    CK(cudaMemcpy(&flag, W.d_ctr + 1, sizeof(flag), cudaMemcpyDeviceToHost));
    if (flag) fail(QW_ERR_DEVICE_TIMEOUT, "a bounded dependency wait of the persistent batch expired");
  }
  for (const DeviceState::MatBatch &B : D->mat_batches) {
    unsigned int flag = 0;
    CK(cudaMemcpy(&flag, B.d_ctr + 1, sizeof(flag), cudaMemcpyDeviceToHost));
    if (flag) fail(QW_ERR_DEVICE_TIMEOUT, "a bounded dependency wait of the boundaries' launch expired");
  }
  for (qw_dense_prog *dp : D->mat_dense)
    if (dp) dense_prog_check(dp);
  std::vector<double> en(2 * (size_t)nt);
  if (nt) CK(cudaMemcpy(en.data(), D->d_energy, en.size() * sizeof(double), cudaMemcpyDeviceToHost));
  P->energy.assign(nt, 0);
  P->norm2.assign(nt, 0);
  for (uint32_t t = 0; t < nt; t++) { P->energy[t] = en[2 * t]; P->norm2[t] = en[2 * t + 1]; }
  P->samples.assign(P->sample_off[nt], 0);
  if (!P->samples.empty())
    CK(cudaMemcpy(P->samples.data(), D->d_samples, P->samples.size() * sizeof(uint64_t), cudaMemcpyDeviceToHost));
  if (D->d_outs) {
    P->outs_suffix.assign(P->outs_off[nt], 0);
    if (!P->outs_suffix.empty())
      CK(cudaMemcpy(P->outs_suffix.data(), D->d_outs, P->outs_suffix.size(), cudaMemcpyDeviceToHost));
    P->outs_mat.assign(P->outs_mat_off.back(), 0);
    if (!P->outs_mat.empty())
      CK(cudaMemcpy(P->outs_mat.data(), D->d_mat_outs, P->outs_mat.size(), cudaMemcpyDeviceToHost));
  }
  float ms = 0;
  cudaEventElapsedTime(&ms, D->ev[0], D->ev[1]);
  P->t_prefix_ms = ms;
  P->t_suffix_ms = P->t_energy_ms = P->t_sample_ms = 0;
  P->batch_ms.assign(D->waves.size(), 0.0);
  for (size_t w = 0; w < D->waves.size(); w++) {
    cudaEventElapsedTime(&ms, D->wave_ev[4 * w], D->wave_ev[4 * w + 1]);
    P->t_suffix_ms += ms;
    P->batch_ms[w] = ms;
    cudaEventElapsedTime(&ms, D->wave_ev[4 * w + 1], D->wave_ev[4 * w + 2]);
    P->t_energy_ms += ms;
    cudaEventElapsedTime(&ms, D->wave_ev[4 * w + 2], D->wave_ev[4 * w + 3]);
    P->t_sample_ms += ms;
  }
  cudaEventElapsedTime(&ms, D->ev[2], D->ev[3]);
  P->t_tab_ms = ms;
  cudaEventElapsedTime(&ms, D->ev[0], D->ev[3]);
  P->t_total_ms = ms;
  P->timed++;
}

void plan_release(qw_plan *P) {
  if (P->dev) {
    if (P->eng) cudaSetDevice(P->eng->device);
    // the plan may have run on a caller's stream: its blocks go back to the
    // engine's cache only once the device has finished with them
    cudaDeviceSynchronize();
    for (qw_dense_prog *dp : P->dev->mat_dense) dense_prog_destroy(dp);
    delete P->dev;
    P->dev = nullptr;
  }
}

void *plan_state_ptr(const qw_plan *P, uint64_t t) {
  return P->dev ? P->dev->task_state[t] : nullptr;
}

bool plan_tableau_keep(const qw_plan *P, uint64_t t, const uint64_t **rows, const uint8_t **sign) {
  if (!P->dev || t >= P->dev->tab_keep.size() || !P->dev->tab_keep[t].first) return false;
  *rows = P->dev->tab_keep[t].first;
  *sign = P->dev->tab_keep[t].second;
  return true;
}

// ---------------------------------------------------------------------------
// engine
// ---------------------------------------------------------------------------
__global__ void bw_probe_kernel(const float4 *a, float4 *b, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = a[i];
}

// L2 read probe: 64 KB blocks of an L2-resident buffer in hashed order (the
// access pattern of the energy kernel's partner reads: independent blocks
// at scattered places), 16 independent 16-byte loads per thread per block.
// Every block index is reduced modulo the block count, so all loads stay in
// the buffer.
__global__ void l2_probe_kernel(const float4 *__restrict__ buf, uint64_t n_blocks, int iters, float *sink) {
  float acc = 0.f;
  for (int it = 0; it < iters; it++) {
    const uint64_t b = ((((uint64_t)blockIdx.x * iters + it) * 0x9E3779B97F4A7C15ull) >> 20) % n_blocks;
    float4 v[16];
#pragma unroll
    for (int j = 0; j < 16; j++) v[j] = __ldg(buf + b * 4096 + j * 256 + threadIdx.x);
#pragma unroll
    for (int j = 0; j < 16; j++) acc += (v[j].x + v[j].y) + (v[j].z + v[j].w);
  }
  if (acc == 1.5e30f) sink[0] = acc;  // keeps the loads; the buffer holds zeros
}

double engine_probe_l2(Engine *E) {
  CK(cudaSetDevice(E->device));
  cudaStream_t s = (cudaStream_t)E->stream;
  const size_t bytes = std::min<size_t>((size_t)64 << 20, (size_t)(E->l2_bytes / 2) & ~(size_t)0xFFFF);
  if (bytes < ((size_t)1 << 20)) fail(QW_ERR_UNSUPPORTED, "L2 of %llu bytes is too small to probe", (unsigned long long)E->l2_bytes);
  float4 *buf = nullptr;
  float *sink = nullptr;
  CK(cudaMalloc(&buf, bytes));
  CK(cudaMalloc(&sink, sizeof(float)));
  CK(cudaMemsetAsync(buf, 0, bytes, s));
  const int grid = E->sm_count * 8, iters = 64;
  const uint64_t nb = bytes / (size_t)65536;
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  float best = 1e30f;
  for (int r = 0; r < 4; r++) {
    CK(cudaEventRecord(e0, s));
    l2_probe_kernel<<<grid, 256, 0, s>>>(buf, nb, iters, sink);
    CK(cudaEventRecord(e1, s));
    CK(cudaEventSynchronize(e1));
    float ms;
    CK(cudaEventElapsedTime(&ms, e0, e1));
    if (r) best = std::min(best, ms);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(buf);
  cudaFree(sink);
  CK(cudaGetLastError());
  return (double)grid * iters * 65536.0 / (best * 1e-3) / 1e9;
}

void engine_init(Engine *E, const qw_engine_opts *o) {
  E->device = o ? o->device : 0;
  CK(cudaSetDevice(E->device));
  cudaDeviceProp prop;
  CK(cudaGetDeviceProperties(&prop, E->device));
  E->sm_count = prop.multiProcessorCount;
  E->l2_bytes = prop.l2CacheSize;
  cudaStream_t s;
  CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  E->stream = s;
  size_t fr = 0, tot = 0;
  CK(cudaMemGetInfo(&fr, &tot));
  E->store_budget = (o && o->store_budget_bytes) ? o->store_budget_bytes : (uint64_t)(0.4 * fr);
  E->task_budget = (o && o->task_budget_bytes) ? o->task_budget_bytes : (uint64_t)(0.4 * fr);
  if (o && o->hbm_gbs > 0) {
    E->hbm_gbs = o->hbm_gbs;
  } else {
    const size_t n = (size_t)1 << 26;  // 1 GiB of float4 per buffer
    float4 *a = nullptr, *b = nullptr;
    CK(cudaMalloc(&a, n * sizeof(float4)));
    CK(cudaMalloc(&b, n * sizeof(float4)));
    CK(cudaMemsetAsync(a, 0, n * sizeof(float4), s));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    for (int r = 0; r < 4; r++) {
      cudaEventRecord(e0, s);
      bw_probe_kernel<<<E->sm_count * 8, 256, 0, s>>>(a, b, n);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float ms;
      cudaEventElapsedTime(&ms, e0, e1);
      if (r) best = std::min(best, ms);
    }
    E->hbm_gbs = 2.0 * n * sizeof(float4) / (best * 1e-3) / 1e9;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(a);
    cudaFree(b);
  }
  // Workspaces of the calls on caller buffers come from a pool of the
  // engine's own that keeps up to CALL_POOL_BYTES between calls (the device's
  // default pool unmaps everything at each synchronization: a 24-qubit gate
  // list then maps its 128 MB remainder array anew, 0.7 ms)
  {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = E->device;
    cudaMemPool_t pool;
    CK(cudaMemPoolCreate(&pool, &props));
    E->call_pool = pool;
    uint64_t keep = CALL_POOL_BYTES;
    CK(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep));
  }
  // kernel attributes are set before any capture
  CK(sv_init_attrs());
  CK(tab_init_attrs());
  CK(dense_init_attrs());
  CK(frame_init_attrs());
  CK(cudaGetLastError());
}

void *Engine::dev_alloc(size_t bytes, size_t *got) {
  const size_t want = (bytes + 511) & ~(size_t)511;
  auto it = free_blocks.lower_bound(want);
  if (it != free_blocks.end() && it->first <= want + want / 4 + 4096) {
    void *p = it->second;
    *got = it->first;
    cached_bytes -= it->first;
    free_blocks.erase(it);
    return p;
  }
  void *p = nullptr;
  cudaError_t e = cudaMalloc(&p, want);
  if (e != cudaSuccess) {  // give the cached blocks back and try once more
    cudaGetLastError();
    trim_cache();
    e = cudaMalloc(&p, want);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    fail(QW_ERR_OOM, "device allocation of %zu bytes failed: %s", want, cudaGetErrorString(e));
  }
  *got = want;
  return p;
}

void Engine::dev_free(void *p, size_t bytes) {
  free_blocks.insert({bytes, p});
  cached_bytes += bytes;
}

void Engine::trim_cache() {
  cudaSetDevice(device);
  if (call_pool) cudaMemPoolTrimTo((cudaMemPool_t)call_pool, 0);
  if (free_blocks.empty()) return;
  cudaDeviceSynchronize();
  for (auto &b : free_blocks) cudaFree(b.second);
  free_blocks.clear();
  cached_bytes = 0;
}

void engine_release(Engine *E) {
  cudaSetDevice(E->device);
  E->trim_cache();
  if (E->scratch) cudaFree(E->scratch);
  if (E->d_mlp) cudaFree(E->d_mlp);
  if (E->call_pool) {
    cudaDeviceSynchronize();  // its memory may still be in use on a caller's stream
    cudaMemPoolDestroy((cudaMemPool_t)E->call_pool);
  }
  if (E->stream) cudaStreamDestroy((cudaStream_t)E->stream);
}

void *Engine::ensure_scratch(size_t bytes) {
  if (bytes > scratch_bytes) {
    if (scratch) { cudaStreamSynchronize((cudaStream_t)stream); cudaFree(scratch); scratch = nullptr; }
    CK(cudaMalloc(&scratch, bytes));
    scratch_bytes = bytes;
  }
  return scratch;
}

// Autotuner: times one synthetic hardware-efficient layer stack under each
// candidate (tile qubits, contiguous low qubits) and keeps the fastest per
// (qubit count, precision).
TileConfig Engine::tile_config(uint32_t n_eff, bool fp64, int ar, uint32_t mix) {
  const uint32_t key_n = std::min<uint32_t>(n_eff, 26);
  if (fp64 || ar == SV_AR_REM) ar = SV_AR_PLAIN;
  mix &= 1u;
  const uint64_t key = tile_key(n_eff, fp64, ar, mix);
  auto it = tiles.find(key);
  if (it != tiles.end()) return it->second;
  TileConfig best;
  best.k_max = sv_max_tile(ar, fp64);
  best.b = 4;
  best.g = sv_stage_width(ar, fp64);
  CK(cudaSetDevice(device));
  cudaStream_t s = (cudaStream_t)stream;
  std::mt19937_64 rng(12345);
  std::uniform_real_distribution<double> U(0, 6.283185307179586);
  // the tuning circuits of the gate mix: layered (hardware-efficient layers,
  // rotations on every qubit and a CNOT chain, 1 to 4 layers as in a sweep's
  // suffixes; their times are summed) or entangling (a random circuit, half
  // of its gates CNOT / CZ on random pairs)
  std::vector<std::vector<qw_gate>> circuits;
  if (mix == 0) {
    for (int layers = 1; layers <= 4; layers++) {
      std::vector<qw_gate> g;
      for (int l = 0; l < layers; l++) {
        for (uint32_t q = 0; q < key_n; q++) g.push_back({QW_OP_RY, q, 0, 0, U(rng)});
        for (uint32_t q = 0; q < key_n; q++) g.push_back({QW_OP_RZ, q, 0, 0, U(rng)});
        for (uint32_t q = 0; q + 1 < key_n; q++) g.push_back({QW_OP_CNOT, q, q + 1, 0, 0.0});
      }
      circuits.push_back(std::move(g));
    }
  } else {
    std::vector<qw_gate> g;
    for (int i = 0; i < 40 * (int)key_n; i++) {
      const uint32_t a = (uint32_t)(rng() % key_n), b = (uint32_t)((a + 1 + rng() % (key_n - 1)) % key_n);
      const uint32_t r = (uint32_t)(rng() % 4);
      const uint32_t op = r == 0 ? QW_OP_CZ : r == 1 ? QW_OP_CNOT : r == 2 ? QW_OP_RX : QW_OP_RZ;
      g.push_back({op, a, r < 2 ? b : 0, 0, U(rng)});
    }
    circuits.push_back(std::move(g));
  }
  // independent states advanced together, as a wave's tasks are: as many as
  // make a pass of the widest tile at least eight rounds of the resident CTAs
  // (with fewer, its last, partly empty round decides between shapes: 8
  // states of 20 qubits chose 12-qubit tiles, 3.30 ms against 2.92 ms for the
  // 64-task suffix), 2 to 32, within 1 GB
  const size_t S = sv_state_bytes(fp64, key_n);
  const uint32_t wide = std::min<uint32_t>(key_n, (uint32_t)sv_max_tile(ar, fp64));
  const size_t rounds = (8ull * 3ull * (size_t)sm_count) >> (key_n - wide);
  const uint32_t chains = (uint32_t)std::max<size_t>(
      1, std::min<size_t>(std::min<size_t>(32, std::max<size_t>(2, rounds)), ((size_t)1 << 30) / S));
  void *buf = nullptr;
  CK(cudaMalloc(&buf, S * chains));
  CK(cudaMemsetAsync(buf, 0, S * chains, s));
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const uint32_t ks32[5] = {12, 13, 14, 0, 0}, ks64[5] = {11, 12, 13, 9, 10}, bs[3] = {3, 4, 5};
  float best_ms = 1e30f;
  const uint32_t best_cap = best.k_max;
  // a register that fits one tile is timed with that single shape (its
  // per-pass time calibrates the analytic cost model)
  // Small FP64 registers are timed with smaller tiles too: a state that fits
  // one tile runs on one SM, whose FP64 pipe (1/64 of the FP32 rate) it then
  // waits for, 0.9 ms for a 6-layer 12-qubit prefix.
  const bool small64 = fp64 && key_n <= 16;
  const bool one_tile = key_n <= best.k_max && !(small64 && key_n >= 11);
  for (int ki = 0; ki < (small64 ? 5 : 3); ki++) {
    for (int bi = 0; bi < 3; bi++) {
      TileConfig tc;
      tc.k_max = fp64 ? ks64[ki] : ks32[ki];
      tc.b = bs[bi];
      tc.g = best.g;
      if (one_tile) {
        if (ki || bi) continue;
        tc.k_max = best.k_max;
        tc.b = best.b;
      }
      if (tc.b + 2 > tc.k_max || tc.k_max > best_cap) continue;
      float tot = 0;
      for (const auto &g : circuits) {
        SvProgram pr = fuse_sv(g.data(), g.size(), key_n, tc, fp64);
        SvTableBuilder tb(fp64);
        tb.add(pr);
        SvTables T;
        DevArena dar;
        T.passes = dar.upload(tb.passes, s);
        T.stages = dar.upload(tb.stages, s);
        T.ops = fp64 ? (const void *)dar.upload(tb.ops64, s) : (const void *)dar.upload(tb.ops32, s);
        T.ops_lo = fp64 ? nullptr : dar.upload(tb.ops32lo, s);
        T.ph = fp64 ? (const void *)dar.upload(tb.ph64, s) : (const void *)dar.upload(tb.ph, s);
        // timed in the persistent batch kernel that runs the suffixes: each
        // state's passes a chain of jobs (each waiting for the last), the
        // chains interleaved pass by pass
        std::vector<SvJob> jobs;
        uint32_t kmax = 5;
        for (size_t p = 0; p < pr.passes.size(); p++) {
          const uint32_t kp = (uint32_t)pr.passes[p].q.size();
          for (uint32_t c = 0; c < chains; c++) {
            SvJob j{};
            j.src = (char *)buf + (size_t)c * S;
            j.dst = (char *)buf + (size_t)c * S;
            j.pass = (uint32_t)p;
            j.n_tiles = 1u << (key_n - kp);
            j.dep = p ? (int32_t)jobs.size() - (int32_t)chains : -1;
            j.kind = SVJ_PASS;
            j.n = key_n;
            jobs.push_back(j);
          }
          kmax = std::max(kmax, kp);
        }
        const int grid = sv_batch_grid(fp64, kmax, sm_count, ar);
        const uint32_t seg_bits = segment_bits(jobs);
        std::vector<SvSeg> segs;
        build_segments(jobs, jobs.size(), seg_bits, 2ull * (uint64_t)grid, segs);
        const uint32_t total = (uint32_t)(segs.size() << seg_bits);
        const SvJob *dj = dar.upload(jobs, s);
        const SvSeg *dsg = dar.upload(segs, s);
        const size_t ctr_bytes = (2 + jobs.size()) * sizeof(unsigned int);
        unsigned int *ctr = (unsigned int *)dar.alloc(ctr_bytes);
        const EnTables no_energy{};
        for (int r = 0; r < 3; r++) {  // one warm-up, two timed
          CK(cudaMemsetAsync(ctr, 0, ctr_bytes, s));
          cudaEventRecord(e0, s);
          launch_sv_batch(fp64, T, dj, dsg, seg_bits, total, kmax, ctr, no_energy, grid, s, ar);
          cudaEventRecord(e1, s);
          CK(cudaEventSynchronize(e1));
          float ms;
          cudaEventElapsedTime(&ms, e0, e1);
          if (r) tot += ms;
        }
        CK(cudaStreamSynchronize(s));
        dar.release();
      }
      if (tot < best_ms) {
        best_ms = tot;
        best = tc;
      }
    }
  }
  // the analytic cost's calibration (Eq. 2): the chosen shape's time per
  // pass on one state, its passes launched one by one, as the cost probe
  // times the segments of one task
  {
    float tot = 0;
    size_t n_passes = 0;
    for (const auto &g : circuits) {
      SvProgram pr = fuse_sv(g.data(), g.size(), key_n, best, fp64);
      SvTableBuilder tb(fp64);
      tb.add(pr);
      SvTables T;
      DevArena dar;
      T.passes = dar.upload(tb.passes, s);
      T.stages = dar.upload(tb.stages, s);
      T.ops = fp64 ? (const void *)dar.upload(tb.ops64, s) : (const void *)dar.upload(tb.ops32, s);
      T.ops_lo = fp64 ? nullptr : dar.upload(tb.ops32lo, s);
      T.ph = fp64 ? (const void *)dar.upload(tb.ph64, s) : (const void *)dar.upload(tb.ph, s);
      for (int r = 0; r < 3; r++) {  // one warm-up, two timed
        cudaEventRecord(e0, s);
        for (size_t p = 0; p < pr.passes.size(); p++)
          launch_sv_pass(fp64, T, (uint32_t)p, (uint32_t)pr.passes[p].q.size(), key_n, buf, buf, s, ar);
        cudaEventRecord(e1, s);
        CK(cudaEventSynchronize(e1));
        float ms;
        cudaEventElapsedTime(&ms, e0, e1);
        if (r) tot += ms;
      }
      CK(cudaStreamSynchronize(s));
      dar.release();
      n_passes += pr.passes.size();
    }
    best.pass_ns = (double)tot * 1e6 / 2.0 / std::max<double>(1.0, (double)n_passes);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(buf);
  CK(cudaGetLastError());
  tiles[key] = best;
  tuning_runs++;
  return best;
}

double Engine::predict_log2ns(const float *feat, uint32_t rows, float *out) {
  CK(cudaSetDevice(device));
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<float> x((size_t)rows * QW_MLP_IN);
  for (uint32_t r = 0; r < rows; r++)
    for (int i = 0; i < QW_MLP_IN; i++)
      x[(size_t)r * QW_MLP_IN + i] = (feat[(size_t)r * QW_MLP_IN + i] - cm.mean[i]) / cm.scale[i];
  float *d = (float *)ensure_scratch(sizeof(float) * (x.size() + rows) + 256);
  float *dy = d + x.size();
  CK(cudaMemcpyAsync(d, x.data(), x.size() * sizeof(float), cudaMemcpyHostToDevice, s));
  launch_mlp_forward(d_mlp, d, dy, rows, s);
  CK(cudaMemcpyAsync(out, dy, rows * sizeof(float), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  return out[0];
}

void costmodel_train(Engine *E, const float *feat, const float *tgt, uint64_t n, uint32_t epochs,
                     uint32_t batch, float lr, uint64_t seed, float *final_loss) {
  if (n == 0 || batch == 0) fail(QW_ERR_INVALID_ARG, "empty training set");
  CK(cudaSetDevice(E->device));
  cudaStream_t s = (cudaStream_t)E->stream;
  CostModel &cm = E->cm;
  // feature normalization and training ranges
  for (int i = 0; i < QW_MLP_IN; i++) {
    double mu = 0, sq = 0;
    float lo = 1e30f, hi = -1e30f;
    for (uint64_t r = 0; r < n; r++) {
      const float v = feat[r * QW_MLP_IN + i];
      mu += v; sq += (double)v * v;
      lo = std::min(lo, v); hi = std::max(hi, v);
    }
    mu /= n;
    const double var = std::max(0.0, sq / n - mu * mu);
    cm.mean[i] = (float)mu;
    cm.scale[i] = (float)(var > 1e-12 ? std::sqrt(var) : 1.0);
    cm.f_lo[i] = lo;
    cm.f_hi[i] = hi;
  }
  cm.y_lo = *std::min_element(tgt, tgt + n);
  cm.y_hi = *std::max_element(tgt, tgt + n);
  // init (He-uniform), bias of the output at the target mean
  std::mt19937_64 rng(seed);
  cm.params.assign(QW_MLP_PARAMS, 0.f);
  auto fill = [&](int off, int count, int fan_in) {
    const double a = std::sqrt(6.0 / fan_in);
    std::uniform_real_distribution<double> U(-a, a);
    for (int i = 0; i < count; i++) cm.params[off + i] = (float)U(rng);
  };
  fill(0, QW_MLP_IN * QW_MLP_HID, QW_MLP_IN);
  fill(QW_MLP_IN * QW_MLP_HID + QW_MLP_HID, QW_MLP_HID * QW_MLP_HID, QW_MLP_HID);
  fill(QW_MLP_IN * QW_MLP_HID + 2 * QW_MLP_HID + QW_MLP_HID * QW_MLP_HID, QW_MLP_HID, QW_MLP_HID);
  double ym = 0;
  for (uint64_t r = 0; r < n; r++) ym += tgt[r];
  cm.params[QW_MLP_PARAMS - 1] = (float)(ym / n);
  std::vector<float> xn(n * QW_MLP_IN);
  for (uint64_t r = 0; r < n; r++)
    for (int i = 0; i < QW_MLP_IN; i++) xn[r * QW_MLP_IN + i] = (feat[r * QW_MLP_IN + i] - cm.mean[i]) / cm.scale[i];
  DevArena ar;
  float *dX = ar.upload(xn, s);
  std::vector<float> tv(tgt, tgt + n);
  float *dT = ar.upload(tv, s);
  if (E->d_mlp) { cudaFree(E->d_mlp); E->d_mlp = nullptr; }
  CK(cudaMalloc(&E->d_mlp, QW_MLP_PARAMS * sizeof(float)));
  CK(cudaMemcpyAsync(E->d_mlp, cm.params.data(), QW_MLP_PARAMS * sizeof(float), cudaMemcpyHostToDevice, s));
  float *dG = (float *)ar.alloc(QW_MLP_PARAMS * sizeof(float));
  float *dM = (float *)ar.alloc(QW_MLP_PARAMS * sizeof(float));
  float *dV = (float *)ar.alloc(QW_MLP_PARAMS * sizeof(float));
  float *dL = (float *)ar.alloc(sizeof(float));
  float *dS = (float *)ar.alloc(mlp_scratch_floats(batch) * sizeof(float));
  float *dXb = (float *)ar.alloc((size_t)batch * QW_MLP_IN * sizeof(float));
  float *dTb = (float *)ar.alloc((size_t)batch * sizeof(float));
  CK(cudaMemsetAsync(dM, 0, QW_MLP_PARAMS * sizeof(float), s));
  CK(cudaMemsetAsync(dV, 0, QW_MLP_PARAMS * sizeof(float), s));
  std::vector<uint32_t> perm(n);
  for (uint64_t i = 0; i < n; i++) perm[i] = (uint32_t)i;
  std::vector<float> bx((size_t)batch * QW_MLP_IN), bt(batch);
  uint32_t step = 0;
  for (uint32_t ep = 0; ep < epochs; ep++) {
    std::shuffle(perm.begin(), perm.end(), rng);
    for (uint64_t b0 = 0; b0 < n; b0 += batch) {
      const uint32_t bs = (uint32_t)std::min<uint64_t>(batch, n - b0);
      for (uint32_t i = 0; i < bs; i++) {
        memcpy(&bx[(size_t)i * QW_MLP_IN], &xn[(size_t)perm[b0 + i] * QW_MLP_IN], QW_MLP_IN * sizeof(float));
        bt[i] = tgt[perm[b0 + i]];
      }
      CK(cudaMemcpyAsync(dXb, bx.data(), (size_t)bs * QW_MLP_IN * sizeof(float), cudaMemcpyHostToDevice, s));
      CK(cudaMemcpyAsync(dTb, bt.data(), (size_t)bs * sizeof(float), cudaMemcpyHostToDevice, s));
      launch_mlp_loss_grad(E->d_mlp, dXb, dTb, bs, dL, dG, dS, s);
      launch_mlp_adam(E->d_mlp, dG, dM, dV, QW_MLP_PARAMS, ++step, lr, 0.9f, 0.999f, 1e-8f, s);
      CK(cudaStreamSynchronize(s));  // bx/bt are reused by the next batch
    }
  }
  // final full-set loss
  float *dSall = (float *)ar.alloc(mlp_scratch_floats((uint32_t)n) * sizeof(float));
  launch_mlp_loss_grad(E->d_mlp, dX, dT, (uint32_t)n, dL, dG, dSall, s);
  float L = 0;
  CK(cudaMemcpyAsync(&L, dL, sizeof(float), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(cm.params.data(), E->d_mlp, QW_MLP_PARAMS * sizeof(float), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  ar.release();
  cm.trained = true;
  if (final_loss) *final_loss = L;
}

void costmodel_set(Engine *E, const float *params, const float *mean, const float *scale) {
  CK(cudaSetDevice(E->device));
  E->cm.params.assign(params, params + QW_MLP_PARAMS);
  memcpy(E->cm.mean, mean, sizeof(E->cm.mean));
  memcpy(E->cm.scale, scale, sizeof(E->cm.scale));
  for (int i = 0; i < QW_MLP_IN; i++) { E->cm.f_lo[i] = -1e30f; E->cm.f_hi[i] = 1e30f; }
  if (!E->d_mlp) CK(cudaMalloc(&E->d_mlp, QW_MLP_PARAMS * sizeof(float)));
  CK(cudaMemcpy(E->d_mlp, params, QW_MLP_PARAMS * sizeof(float), cudaMemcpyHostToDevice));
  E->cm.trained = true;
}

// timing probe: runs segments of the workload's statevector tasks on a
// scratch state and records (features, log2 ns)
void costmodel_probe(Engine *E, const Workload &W, float *feat, float *tgt, float *analytic, uint64_t cap,
                     uint64_t *n_rows) {
  CK(cudaSetDevice(E->device));
  cudaStream_t s = (cudaStream_t)E->stream;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  uint64_t rows = 0;
  std::mt19937_64 rng(777);
  std::vector<qw_gate> buf;
  for (const TaskData &T : W.tasks) {
    if (rows >= cap) break;
    if (T.mode == QW_MODE_TABLEAU || T.n_gates == 0) continue;
    const bool fp64 = T.mode == QW_MODE_SV_FP64;
    const uint32_t n_eff = std::max<uint32_t>(T.n, SV_G);
    // timings of the default FP32 arithmetic (compensated, as the
    // persistent suffix launch runs it)
    const int par = fp64 ? SV_AR_PLAIN : SV_AR_COMP;
    uint64_t n2 = 0;
    for (uint64_t i = 0; i < T.n_gates; i++) n2 += is_two_qubit_op(T.gate(i)->op) ? 1 : 0;
    TileConfig tc = E->tile_config(n_eff, fp64, par, gate_mix(n2, T.n_gates));
    const size_t S = sv_state_bytes(fp64, n_eff);
    void *st = E->ensure_scratch(S);
    CK(cudaMemsetAsync(st, 0, S, s));
    // segments: full list, and a prefix / suffix split at a random point
    const uint64_t c = 1 + rng() % std::max<uint64_t>(1, T.n_gates - 1);
    const std::pair<uint64_t, uint64_t> segs[3] = {{0, T.n_gates}, {0, c}, {c, T.n_gates}};
    for (auto sg : segs) {
      if (rows >= cap || sg.second <= sg.first) continue;
      T.copy_gates(sg.first, sg.second, buf);
      SvProgram pr = fuse_sv(buf.data(), buf.size(), n_eff, tc, fp64);
      SvTableBuilder tb(fp64);
      tb.add(pr);
      DevArena ar;
      SvTables Tt;
      Tt.passes = ar.upload(tb.passes, s);
      Tt.stages = ar.upload(tb.stages, s);
      Tt.ops = fp64 ? (const void *)ar.upload(tb.ops64, s) : (const void *)ar.upload(tb.ops32, s);
      Tt.ops_lo = fp64 ? nullptr : ar.upload(tb.ops32lo, s);
      Tt.ph = fp64 ? (const void *)ar.upload(tb.ph64, s) : (const void *)ar.upload(tb.ph, s);
      float best = 1e30f;
      for (int r = 0; r < 3; r++) {
        cudaEventRecord(e0, s);
        for (size_t p = 0; p < pr.passes.size(); p++)
          launch_sv_pass(fp64, Tt, (uint32_t)p, (uint32_t)pr.passes[p].q.size(), n_eff, st, st, s, par);
        cudaEventRecord(e1, s);
        CK(cudaEventSynchronize(e1));
        float ms;
        cudaEventElapsedTime(&ms, e0, e1);
        if (r) best = std::min(best, ms);
      }
      ar.release();
      features_for(T, sg.first, sg.second, 1, tc, 0.0, feat + rows * QW_MLP_IN);
      tgt[rows] = (float)std::log2(std::max(1.0, (double)best * 1e6));
      if (analytic) {
        // the planner's analytic cost: passes x measured time per pass
        const double per = tc.pass_ns > 0 ? tc.pass_ns : 2.0 * (double)S / E->hbm_gbs + E->launch_ns;
        const double ns = (double)pr.passes.size() * per;
        analytic[rows] = (float)std::log2(std::max(1.0, ns));
      }
      rows++;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  CK(cudaGetLastError());
  *n_rows = rows;
}

}  // namespace qw

// ---------------------------------------------------------------------------
// kernels on caller-owned device buffers
// ---------------------------------------------------------------------------
namespace qw {

// Host tables of one call, uploaded in one copy (each copy and allocation of
// a small call costs more than its kernels).
struct Blob {
  std::vector<char> bytes;
  template <typename T>
  size_t add(const std::vector<T> &v) { return add(v.data(), v.size() * sizeof(T)); }
  size_t add(const void *p, size_t n) {
    const size_t at = (bytes.size() + 255) & ~(size_t)255;
    bytes.resize(at + n);
    if (n && p) memcpy(bytes.data() + at, p, n);
    return at;
  }
};

// Stream-ordered workspace of one call from the engine's pool: freed on the
// same stream when the call's work is enqueued.
struct CallSpace {
  char *p = nullptr;
  cudaStream_t s;
  CallSpace(Engine *E, size_t bytes, cudaStream_t st) : s(st) {
    CK(cudaMallocFromPoolAsync((void **)&p, std::max<size_t>(16, bytes), (cudaMemPool_t)E->call_pool, s));
  }
  CallSpace(const CallSpace &) = delete;
  CallSpace &operator=(const CallSpace &) = delete;
  ~CallSpace() {
    if (p) cudaFreeAsync(p, s);
  }
};

qw_status sv_apply_dev(Engine *E, uint32_t mode, uint32_t n, void *state, const qw_gate *gates,
                       uint64_t n_gates, bool init, void *stream) {
  CK(cudaSetDevice(E->device));
  cudaStream_t s = (cudaStream_t)stream;
  const bool fp64 = mode == QW_MODE_SV_FP64;
  // FP32: compensated arithmetic with the remainder kept between passes, so
  // the state is rounded once, by the last pass (none where nothing rounds)
  int ar = fp64 ? SV_AR_PLAIN : SV_AR_REM;
  uint64_t n2 = 0;
  for (uint64_t i = 0; i < n_gates; i++) n2 += is_two_qubit_op(gates[i].op) ? 1 : 0;
  TileConfig tc = E->tile_config(n, fp64, SV_AR_COMP, gate_mix(n2, n_gates));
  tc.k_max = sv_permutes(gates, n_gates) ? sv_permute_tile(n, fp64, tc.k_max)
                                         : std::min<uint32_t>(tc.k_max, sv_max_tile(ar, fp64));
  SvProgram pr = fuse_sv(gates, n_gates, n, tc, fp64);
  if (ar == SV_AR_REM && sv_exact(pr)) ar = SV_AR_COMP;
  if (pr.passes.empty()) {
    if (!init) return QW_OK;
    HostPass hp;
    const uint32_t k = std::min(tc.k_max, n);
    for (uint32_t q = 0; q < k; q++) hp.q.push_back(q);
    hp.b = (n <= tc.k_max) ? n : std::min(tc.b, k - 2);
    pr.passes.push_back(hp);
  }
  SvTableBuilder tb(fp64);
  tb.add(pr);
  SvTables T;
  Blob bl;
  const size_t op = bl.add(tb.passes), os = bl.add(tb.stages), oo = fp64 ? bl.add(tb.ops64) : bl.add(tb.ops32);
  const size_t ol = bl.add(tb.ops32lo), oh = fp64 ? bl.add(tb.ph64) : bl.add(tb.ph);
  const size_t np = pr.passes.size();
  const size_t tab_bytes = (bl.bytes.size() + 255) & ~(size_t)255;
  const bool keep_rem = ar == SV_AR_REM && np > 1;
  CallSpace ws(E, tab_bytes + (keep_rem ? sv_state_bytes(false, n) : 0), s);
  CK(cudaMemcpyAsync(ws.p, bl.bytes.data(), bl.bytes.size(), cudaMemcpyHostToDevice, s));
  T.passes = (const SvPassDesc *)(ws.p + op);
  T.stages = (const SvStageDesc *)(ws.p + os);
  T.ops = ws.p + oo;
  T.ops_lo = (const float *)(ws.p + ol);
  T.ph = ws.p + oh;
  void *rem = keep_rem ? ws.p + tab_bytes : nullptr;
  for (size_t p = 0; p < np; p++)
    launch_sv_pass(fp64, T, (uint32_t)p, (uint32_t)pr.passes[p].q.size(), n,
                   (p == 0 && init) ? nullptr : state, state, s, ar, p > 0 ? rem : nullptr,
                   p + 1 < np ? rem : nullptr);
  CK(cudaGetLastError());
  return QW_OK;
}

qw_status sv_energy_dev(Engine *E, uint32_t mode, uint32_t n, const void *state, const qw_pauli_term *terms,
                        uint64_t n_terms, double *energy, double *norm2, void *stream) {
  CK(cudaSetDevice(E->device));
  cudaStream_t s = (cudaStream_t)stream;
  const bool fp64 = mode == QW_MODE_SV_FP64;
  const bool pair = en_pair(fp64, state);
  const EnLayout H = build_energy_layout(terms, n_terms, n, fp64, pair, en_rep_bits(n));
  Blob bl;
  const size_t oc = bl.add(H.classes), og = bl.add(H.groups), ot = bl.add(H.terms), oj = bl.add(nullptr, sizeof(EnJob));
  const size_t tab_bytes = (bl.bytes.size() + 255) & ~(size_t)255;
  CallSpace ws(E, tab_bytes + 2 * sizeof(double) * ((size_t)H.n_blocks + 1), s);
  double *dout = (double *)(ws.p + tab_bytes), *dpart = dout + 2;
  EnJob j{};
  j.state = state;
  j.out = dout;
  j.n = n;
  j.rep_bits = H.rep_bits;
  j.iter_bits = H.iter_bits;
  j.class_begin = 0;
  j.n_classes = (uint32_t)H.classes.size();
  j.block_begin = 0;
  j.n_blocks = H.n_blocks;
  memcpy(bl.bytes.data() + oj, &j, sizeof(j));
  CK(cudaMemcpyAsync(ws.p, bl.bytes.data(), bl.bytes.size(), cudaMemcpyHostToDevice, s));
  const EnTables tab{(const EnJob *)(ws.p + oj), (const EnClass *)(ws.p + oc), (const EnGroup *)(ws.p + og),
                     (const EnTerm *)(ws.p + ot), dpart};
  launch_energy(fp64, pair, tab, 1, H.n_blocks, H.rep_bits, s);
  double res[2];
  CK(cudaMemcpyAsync(res, dout, sizeof(res), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  *energy = res[0];
  if (norm2) *norm2 = res[1];
  return QW_OK;
}

qw_status sv_sample_dev(Engine *E, uint32_t mode, uint32_t n, const void *state, const double *u,
                        uint32_t shots, uint64_t *out, void *stream) {
  CK(cudaSetDevice(E->device));
  cudaStream_t s = (cudaStream_t)stream;
  if (shots == 0) return QW_OK;
  const bool fp64 = mode == QW_MODE_SV_FP64;
  SmpSource so{};
  so.state = state;
  so.n = n;
  so.n_blocks = (n >= (uint32_t)SMP_BLOCK_BITS) ? (1u << (n - SMP_BLOCK_BITS)) : 1u;
  so.block_begin = 0;
  // one workspace: results, the call's tables, block sums and offsets
  const size_t res_bytes = ((size_t)shots * sizeof(uint64_t) + 255) & ~(size_t)255;
  const size_t sh_bytes = (size_t)shots * sizeof(SmpShot);
  const size_t nb = so.n_blocks;
  const size_t o_src = res_bytes, o_sh = o_src + 256, o_sum = (o_sh + sh_bytes + 255) & ~(size_t)255;
  const size_t o_off = o_sum + nb * sizeof(double), o_last = o_off + (nb + 1) * sizeof(double);
  const size_t o_blast = o_last + sizeof(int64_t), total = o_blast + nb * sizeof(int32_t);
  CallSpace ws(E, total, s);
  std::vector<char> up(256 + sh_bytes);
  memcpy(up.data(), &so, sizeof(so));
  SmpShot *sh = (SmpShot *)(up.data() + 256);
  for (uint32_t k = 0; k < shots; k++) {
    SmpShot q{};
    q.u = u[k];
    q.out = (uint64_t *)ws.p + k;
    sh[k] = q;
  }
  CK(cudaMemcpyAsync(ws.p + o_src, up.data(), up.size(), cudaMemcpyHostToDevice, s));
  launch_sampling(fp64, (const SmpSource *)(ws.p + o_src), 1, so.n_blocks, (double *)(ws.p + o_sum),
                  (int32_t *)(ws.p + o_blast), (double *)(ws.p + o_off), (int64_t *)(ws.p + o_last),
                  (const SmpShot *)(ws.p + o_sh), shots, s);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(out, ws.p, (size_t)shots * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  return QW_OK;
}

}  // namespace qw
