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

// All levels of a launch (or all requests that end with it) in one kernel:
// thread t finalises a record of the last level with base <= t.  Small levels
// are bound by the launch alone, whose cost grows with its parameters (an empty
// kernel and its wait, GB300: 8.6 us with 256 B, 10.4 with 16 KB), so the table
// has the least of three lengths that holds the levels.  The results may lie in
// page-locked host memory, which the threads then write themselves, with the
// launch's header: two copies less behind a call (4.2 us of 13.3).
template <int N>
struct FinalizeLevels {
  uint32_t n_levels;
  uint32_t total;
  const unsigned long long* header;  // kHeaderWords words copied to header_out
  unsigned long long* header_out;    // null: none
  uint32_t base[N + 1];              // first thread of each level; base[n_levels] = total
  double kappa[N];
  const unsigned long long* acc[N];
  StatPtrs out[N];
};
static_assert(sizeof(FinalizeLevels<kMaxSegments>) < 32000, "kernel parameter size");

template <int N>
__global__ void finalize_levels(const __grid_constant__ FinalizeLevels<N> f) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (uint32_t)kHeaderWords && f.header_out) f.header_out[t] = f.header[t];
  if (t >= f.total) return;
  int lo = 0, hi = (int)f.n_levels - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (f.base[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  const uint32_t i = t - f.base[lo];
  finalize_one(f.acc[lo] + (size_t)i * kAccWords, i, f.kappa[lo], f.out[lo]);
}

template <int N>
static cudaError_t launch_finalize_table(int n_levels, const unsigned long long* const* acc,
                                         const uint32_t* n_nodes, const double* kappa,
                                         const StatPtrs* out, const void* header, void* header_out,
                                         cudaStream_t st) {
  FinalizeLevels<N> f{};
  uint32_t total = 0;
  int k = 0;
  for (int l = 0; l < n_levels; ++l) {
    if (n_nodes[l] == 0) continue;
    f.base[k] = total;
    f.kappa[k] = kappa[l];
    f.acc[k] = acc[l];
    f.out[k] = out[l];
    total += n_nodes[l];
    ++k;
  }
  if (k == 0) return cudaErrorInvalidValue;  // the caller has a node to finalise
  f.n_levels = (uint32_t)k;
  f.base[k] = total;
  f.total = total;
  f.header = (const unsigned long long*)header;
  f.header_out = (unsigned long long*)header_out;
  const unsigned threads = 128;
  finalize_levels<N><<<(total + threads - 1) / threads, threads, 0, st>>>(f);
  return cudaGetLastError();
}

// Calls about to run (one, or the requests entering the server's batch): their
// records cleared and their coordinates fetched from page-locked host memory,
// blockIdx.y = the call.  In place of a memset and a copy in front of a path
// launch (GB300, whole calls on host arrays: 2,000 nodes x 20 paths 62.3 -> 59.6
// us, 256 x 100 52.9 -> 51.4, one node the same).
template <int N>
struct StageTable {
  StageRequest req[N];
};

template <int N>
__global__ void stage_requests(const __grid_constant__ StageTable<N> t) {
  const StageRequest r = t.req[blockIdx.y];
  const uint32_t step = gridDim.x * blockDim.x;
  for (size_t i = blockIdx.x * blockDim.x + threadIdx.x; i < r.n_records; i += step)
    r.records[i] = make_uint4(0, 0, 0, 0);
  for (size_t i = blockIdx.x * blockDim.x + threadIdx.x; i < r.n_coords; i += step)
    r.coords[i] = r.host_coords[i];
}

template <int N>
static cudaError_t launch_stage_table(const StageRequest* req, int n, cudaStream_t st) {
  StageTable<N> t;
  size_t most = 1;
  for (int i = 0; i < n; ++i) {
    t.req[i] = req[i];
    most = most > req[i].n_records ? most : req[i].n_records;
  }
  const size_t threads = 256, blocks = (most + threads - 1) / threads;
  stage_requests<N><<<dim3((unsigned)(blocks < 304 ? blocks : 304), (unsigned)n),
                      (unsigned)threads, 0, st>>>(t);
  return cudaGetLastError();
}

cudaError_t launch_stage_requests(const StageRequest* req, int n, cudaStream_t st) {
  if (n < 1 || n > kMaxSegments) return cudaErrorInvalidValue;
  return n == 1 ? launch_stage_table<1>(req, n, st) : launch_stage_table<kMaxSegments>(req, n, st);
}

// ---------------------------------------------------------------------------
// Dispatch by problem.
// ---------------------------------------------------------------------------
cudaError_t launch_paths(int kind, int precision, int cv, const PathArgs& args, int num_sms,
                         cudaStream_t st, LaunchInfo* info) {
  PathArgs a = args;
  if (precision == 1) {
    cudaError_t e = f64_tables(&a.f64);
    if (e != cudaSuccess) return e;
  }
  if (a.n_segs < 1 || a.n_segs > kMaxSegments) return cudaErrorInvalidValue;
  // the single-segment build follows the Euler Y rule only (see euler_step)
  const bool multi = a.n_segs > 1 || a.y_exp != 0;
  switch (kind) {
    case 0: return PathLaunch<Cfg0>::paths(precision, cv, multi, a, num_sms, st, info);
    case 1: return PathLaunch<Aniso>::paths(precision, cv, multi, a, num_sms, st, info);
    case 2: return PathLaunch<Cube3>::paths(precision, cv, multi, a, num_sms, st, info);
    case 4: return PathLaunch<PaperEx>::paths(precision, cv, multi, a, num_sms, st, info);
    default: return PathLaunch<Harmonic>::paths(precision, cv, multi, a, num_sms, st, info);
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
                           LaunchInfo* info) {
  switch (kind) {
    case 0: return PathLaunch<Cfg0>::coupled(cv, a, num_sms, st, info);
    case 1: return PathLaunch<Aniso>::coupled(cv, a, num_sms, st, info);
    case 2: return PathLaunch<Cube3>::coupled(cv, a, num_sms, st, info);
    case 3: return PathLaunch<Harmonic>::coupled(cv, a, num_sms, st, info);
    case 4: return PathLaunch<PaperEx>::coupled(cv, a, num_sms, st, info);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_finalize_levels(int n_levels, const unsigned long long* const* acc,
                                   const uint32_t* n_nodes, const double* kappa,
                                   const StatPtrs* out, const void* header, void* header_out,
                                   cudaStream_t st) {
  if (n_levels < 1 || n_levels > kMaxSegments) return cudaErrorInvalidValue;
  auto* const launch = n_levels == 1    ? launch_finalize_table<1>
                       : n_levels <= 16 ? launch_finalize_table<16>
                                        : launch_finalize_table<kMaxSegments>;
  return launch(n_levels, acc, n_nodes, kappa, out, header, header_out, st);
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
