// pdd_paths.cu -- dispatch of the path kernels by problem, and the per-node
// finalisation (eqs. F:Statistics_VR .. F:Rho, F:Pointwise_cost,
// F:VR_Pointwise_cost, F:nu).
#include <cuda_runtime.h>
#include <stdint.h>

#include "pdd_device.cuh"
#include "pdd_internal.h"
#include "pdd_launch.h"

namespace pdd {

// ---------------------------------------------------------------------------
// Finalisation: one thread per node turns the exact sums into FP64 moments.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void finalize_one(const unsigned long long* __restrict__ w,
                                             uint32_t i, double kappa, const StatPtrs& out) {
  const double inv1 = 1.0 / kFxScale, inv2 = inv1 * inv1;
  const double n = (double)w[14];
  const double s_phi = s128_to_double(w[0], w[1]) * inv1;
  const double s_phi2 = s128_to_double(w[2], w[3]) * inv2;
  const double s_psi = s128_to_double(w[4], w[5]) * inv1;
  const double s_psi2 = s128_to_double(w[6], w[7]) * inv2;
  const double s_pp = s128_to_double(w[8], w[9]) * inv2;
  const double s_k = u128_to_double(w[10], w[11]);
  const double m_phi = s_phi / n, m_psi = s_psi / n;
  // the exact sums' conversion to FP64 can leave a zero variance a rounding
  // below zero; clamp it (n = 1 stays NaN: 0 / 0)
  double v_phi = (s_phi2 - s_phi * m_phi) / (n - 1.0);
  double v_psi = (s_psi2 - s_psi * m_psi) / (n - 1.0);
  v_phi = v_phi < 0.0 ? 0.0 : v_phi;
  v_psi = v_psi < 0.0 ? 0.0 : v_psi;
  const double c_pp = (s_pp - s_phi * m_psi) / (n - 1.0);  // Cov[phi, phi + xi]
  const double c_px = c_pp - v_phi;                         // Cov[phi, xi]
  const double v_xi = v_psi + v_phi - 2.0 * c_pp;           // V[xi]
  if (out.mean_phi) out.mean_phi[i] = m_phi;
  if (out.var_phi) out.var_phi[i] = v_phi;
  if (out.mean_cv) out.mean_cv[i] = m_psi;
  if (out.var_cv) out.var_cv[i] = v_psi;
  if (out.cov_phi_xi) out.cov_phi_xi[i] = c_px;
  if (out.var_xi) out.var_xi[i] = v_xi;
  if (out.rho) out.rho[i] = c_px / sqrt(v_phi * v_xi);
  if (out.se_phi) out.se_phi[i] = sqrt(v_phi / n);
  if (out.se_cv) out.se_cv[i] = sqrt(v_psi / n);
  if (out.vr) out.vr[i] = v_psi / v_phi;
  if (out.pred_speedup) out.pred_speedup[i] = v_phi / (kappa * v_psi);
  if (out.mean_steps) out.mean_steps[i] = s_k / n;
  if (out.n_paths) out.n_paths[i] = w[14];
  if (out.n_truncated) out.n_truncated[i] = w[15];
}

__global__ void finalize_nodes(const unsigned long long* __restrict__ acc, uint32_t n_nodes,
                               double kappa, const __grid_constant__ StatPtrs out) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_nodes) return;
  finalize_one(acc + (size_t)i * kAccWords, i, kappa, out);
}

// One thread per pair of words of a record: seven 128-bit sums, and the two
// counts of the last pair.  Memory bound: copies x 128 B per record.
__global__ void merge_records(unsigned long long* __restrict__ acc, unsigned pairs, unsigned copies,
                              unsigned long long stride) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= pairs) return;
  ulonglong2* const p = (ulonglong2*)acc + t;
  ulonglong2 s = *p;
  const bool counts = t % (kAccWords / 2) == kAccWords / 2 - 1;
  for (unsigned c = 1; c < copies; ++c) {
    const ulonglong2 v = *(const ulonglong2*)((const unsigned long long*)p + c * stride);
    s.x += v.x;
    s.y += v.y + (!counts && s.x < v.x ? 1ull : 0ull);
  }
  *p = s;
}

// All levels of a launch in one kernel: thread t finalises record t of the
// contiguous record array, whose level is the last one with base <= t.
struct FinalizeLevels {
  uint32_t n_levels;
  uint32_t total;
  uint32_t base[kMaxSegments + 1];  // first record of each level; base[n_levels] = total
  double kappa[kMaxSegments];
  StatPtrs out[kMaxSegments];
};
static_assert(sizeof(FinalizeLevels) < 32000, "kernel parameter size");

__global__ void finalize_levels(const unsigned long long* __restrict__ acc,
                                const __grid_constant__ FinalizeLevels f) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= f.total) return;
  int lo = 0, hi = (int)f.n_levels - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (f.base[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  finalize_one(acc + (size_t)t * kAccWords, t - f.base[lo], f.kappa[lo], f.out[lo]);
}

// ---------------------------------------------------------------------------
// Dispatch by problem.
// ---------------------------------------------------------------------------
cudaError_t launch_paths(int kind, int precision, int cv, const PathArgs& args, int num_sms,
                         cudaStream_t st, int* blocks) {
  PathArgs a = args;
  if (precision == 1) {
    cudaError_t e = f64_tables(&a.f64);
    if (e != cudaSuccess) return e;
  }
  if (a.n_segs < 1 || a.n_segs > kMaxSegments) return cudaErrorInvalidValue;
  // the single-segment build follows the Euler Y rule only (see euler_step)
  const bool multi = a.n_segs > 1 || a.y_exp != 0;
  switch (kind) {
    case 0: return PathLaunch<Cfg0>::paths(precision, cv, multi, a, num_sms, st, blocks);
    case 1: return PathLaunch<Aniso>::paths(precision, cv, multi, a, num_sms, st, blocks);
    case 2: return PathLaunch<Cube3>::paths(precision, cv, multi, a, num_sms, st, blocks);
    case 4: return PathLaunch<PaperEx>::paths(precision, cv, multi, a, num_sms, st, blocks);
    default: return PathLaunch<Harmonic>::paths(precision, cv, multi, a, num_sms, st, blocks);
  }
}

cudaError_t occupancy_paths(int kind, int precision, int cv, bool multi, int threads, int* occ) {
  switch (kind) {
    case 0: return PathLaunch<Cfg0>::occupancy(precision, cv, multi, threads, occ);
    case 1: return PathLaunch<Aniso>::occupancy(precision, cv, multi, threads, occ);
    case 2: return PathLaunch<Cube3>::occupancy(precision, cv, multi, threads, occ);
    case 4: return PathLaunch<PaperEx>::occupancy(precision, cv, multi, threads, occ);
    default: return PathLaunch<Harmonic>::occupancy(precision, cv, multi, threads, occ);
  }
}

cudaError_t launch_coupled(int kind, int cv, const PathArgs& a, int num_sms, cudaStream_t st,
                           int* blocks) {
  switch (kind) {
    case 0: return PathLaunch<Cfg0>::coupled(cv, a, num_sms, st, blocks);
    case 1: return PathLaunch<Aniso>::coupled(cv, a, num_sms, st, blocks);
    case 2: return PathLaunch<Cube3>::coupled(cv, a, num_sms, st, blocks);
    case 3: return PathLaunch<Harmonic>::coupled(cv, a, num_sms, st, blocks);
    case 4: return PathLaunch<PaperEx>::coupled(cv, a, num_sms, st, blocks);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_finalize_levels(const unsigned long long* acc, int n_levels,
                                   const uint32_t* node_base, const uint32_t* n_nodes,
                                   const double* kappa, const StatPtrs* out, cudaStream_t st) {
  if (n_levels < 1 || n_levels > kMaxSegments) return cudaErrorInvalidValue;
  FinalizeLevels f{};
  uint32_t total = 0;
  int k = 0;
  for (int l = 0; l < n_levels; ++l) {
    if (n_nodes[l] == 0) continue;
    if (node_base[l] != total) return cudaErrorInvalidValue;  // records must be contiguous
    f.base[k] = total;
    f.kappa[k] = kappa[l];
    f.out[k] = out[l];
    total += n_nodes[l];
    ++k;
  }
  if (k == 0) return cudaSuccess;
  f.n_levels = (uint32_t)k;
  f.base[k] = total;
  f.total = total;
  const unsigned threads = 128;
  finalize_levels<<<(total + threads - 1) / threads, threads, 0, st>>>(acc, f);
  return cudaGetLastError();
}

cudaError_t launch_merge_records(unsigned long long* acc, unsigned n_records, unsigned copies,
                                 unsigned long long stride, cudaStream_t st) {
  const unsigned pairs = n_records * (kAccWords / 2), threads = 256;
  merge_records<<<(pairs + threads - 1) / threads, threads, 0, st>>>(acc, pairs, copies, stride);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const unsigned long long* acc, uint32_t n_nodes, double kappa,
                            const StatPtrs& out, cudaStream_t st) {
  const unsigned threads = 128;
  const unsigned blocks = (n_nodes + threads - 1) / threads;
  finalize_nodes<<<blocks, threads, 0, st>>>(acc, n_nodes, kappa, out);
  return cudaGetLastError();
}

}  // namespace pdd
