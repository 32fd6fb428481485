// pdd_fit.cu -- fast fit of nodal constants (Bernal & Acebron, Sec. 5 H5 and
// Algorithm 3): all (node, h) pairs of an h-cloud run as levels of the
// persistent path kernel; the per-node fits are small regressions, a warp each.
//   first moments: E[eta_h] = E[eta_0] + B h^delta, normal noise and identity
//     link, i.e. ordinary least squares in x = h^delta;
//   variances: E[V[eta_h]] = V[eta_0] + B h^delta, gamma noise and identity
//     link, i.e. iteratively reweighted least squares with weights 1/mu^2.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "../../include/pdd.h"
#include "pdd_internal.h"

namespace pdd {
void set_error(const char* fmt, ...);
}

using namespace pdd;

namespace {

// The cloud's statistics (kF fields of n nodes per time step) and its abscissae
// are read by fit_nodes; kC coefficients per node come back.
constexpr int kF = 5;  // mean_phi, var_phi, mean_steps, cov(phi, xi), var_xi
enum { kEPhi, kBeta, kETau, kVPhi, kAlpha, kCov0, kVPsi, kC };
constexpr int kFits = 5;
constexpr int kStageDoubles = 6 * 1024;  // 48 KB of shared memory

// Sum over the warp, the same on every lane.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// y = a + b x by ordinary least squares; with `h`, of y h.
__device__ __forceinline__ void ols(const double* x, const double* y, size_t stride,
                                    const double* h, int m, double& a, double& b) {
  const int lane = (int)(threadIdx.x & 31u);
  auto at = [&](int j) { return h ? y[j * stride] * h[j] : y[j * stride]; };
  double mx = 0, my = 0;
  for (int j = lane; j < m; j += 32) {
    mx += x[j];
    my += at(j);
  }
  mx = warp_sum(mx) / (double)m;
  my = warp_sum(my) / (double)m;
  double sxy = 0, sxx = 0;
  for (int j = lane; j < m; j += 32) {
    const double dx = x[j] - mx;
    sxy += dx * (at(j) - my);
    sxx += dx * dx;
  }
  sxy = warp_sum(sxy);
  sxx = warp_sum(sxx);
  b = sxx > 0 ? sxy / sxx : 0.0;
  a = my - b * mx;
}

// mu = a + b x for gamma-distributed y (variance proportional to mu^2), identity
// link: weighted least squares with weights 1/mu^2 from the previous fit until
// the coefficients settle (Fisher scoring for this model), 200 times at most.
// Rounding often keeps them on a cycle of a few neighbouring values instead of
// one; the map is deterministic, so once a pair returns (Brent's test: against
// the pair kept at the last power of two) whole cycles are left out.
__device__ __forceinline__ void gamma_identity(const double* x, const double* y, size_t stride,
                                               int m, double& a, double& b) {
  ols(x, y, stride, nullptr, m, a, b);
  const int lane = (int)(threadIdx.x & 31u);
  double ymin = 1e300;
  for (int j = lane; j < m; j += 32) {
    const double v = fabs(y[j * stride]);
    ymin = v < ymin ? v : ymin;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double v = __shfl_xor_sync(0xffffffffu, ymin, o);
    ymin = v < ymin ? v : ymin;
  }
  const double low = ymin * 1e-6, floor_mu = low < 1e-300 ? 1e-300 : low;
  double a0 = a, b0 = b;  // the kept pair, `since` iterations ago
  int since = 0, keep = 1;
  for (int left = 200; left > 0; --left) {
    double sw = 0, swx = 0, swy = 0, swxx = 0, swxy = 0;
    for (int j = lane; j < m; j += 32) {
      const double xj = x[j], yj = y[j * stride], v = a + b * xj;
      const double mu = v < floor_mu ? floor_mu : v;
      const double w = 1.0 / (mu * mu), wx = w * xj;
      sw += w;
      swx += wx;
      swy += w * yj;
      swxx += wx * xj;
      swxy += wx * yj;
    }
    sw = warp_sum(sw);
    swx = warp_sum(swx);
    swy = warp_sum(swy);
    swxx = warp_sum(swxx);
    swxy = warp_sum(swxy);
    const double det = sw * swxx - swx * swx;
    if (!(det > 0)) break;
    const double nb = (sw * swxy - swx * swy) / det;
    const double na = (swy - nb * swx) / sw;
    const double change = fabs(na - a) + fabs(nb - b);
    a = na;
    b = nb;
    if (change <= 1e-14 * (fabs(na) + fabs(nb) + 1e-300)) break;
    ++since;
    if (a == a0 && b == b0) {
      left = 1 + (left - 1) % since;
      since = 0;  // fewer than a cycle remain: the pair does not return again
    } else if (since == keep) {
      a0 = a;
      b0 = b;
      keep *= 2;
      since = 0;
    }
  }
}

// Block = node, warp = one of its fits.  Bound by the chain of an iteration (a
// division per time step, five sums, two divisions) and the FP64 pipe.  Whole
// calls (GB300, 400 to 1,000 paths), against the same loops on a host core: 217
// nodes x 100 time steps 7.46 -> 2.63 ms, 24 x 100 1.45 -> 1.13, 3 x 100 0.46 ->
// 0.43, 24 x 20 0.48 both ways.
__global__ void __launch_bounds__(32 * kFits)
    fit_nodes(const double* __restrict__ stat, const double* __restrict__ hx, int m, size_t n,
              int staged, double* __restrict__ coef) {
  extern __shared__ double sm[];
  const size_t i = blockIdx.x;
  const int fit = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31u);
  constexpr int kField[kFits] = {0, 2, 1, 3, 4};
  const int f = kField[fit];
  const double* y = stat + (size_t)f * n + i;
  size_t stride = (size_t)kF * n;
  const double* x = hx + m;
  if (staged) {  // (a cloud too long for shared memory is read where it lies)
    double* const ys = sm + (size_t)fit * m;
    double* const xs = sm + (size_t)kFits * m;
    for (int j = lane; j < m; j += 32) ys[j] = y[j * stride];
    for (int j = (int)threadIdx.x; j < m; j += (int)blockDim.x) xs[j] = x[j];
    y = ys;
    x = xs;
    stride = 1;
    __syncthreads();
  }
  double a, b;
  if (f == 1 || f == 4) gamma_identity(x, y, stride, m, a, b);
  else ols(x, y, stride, f == 2 ? hx : nullptr, m, a, b);  // tau_h = k h
  if (lane == 0) {
    double* const c = coef + i * kC;
    if (fit == 0) { c[kEPhi] = a; c[kBeta] = b; }
    if (fit == 1) c[kETau] = a;
    if (fit == 2) { c[kVPhi] = a; c[kAlpha] = b; }
    if (fit == 3) c[kCov0] = a;
    if (fit == 4) c[kVPsi] = a;
  }
}

}  // namespace

extern "C" int pdd_fit_constants(pdd_problem* p, const pdd_fit_args* a, pdd_fit_out* out) {
  ProblemView pv;
  if (!p || !a || !out || !problem_view(p, &pv)) {
    set_error("pdd_fit_constants: NULL argument");
    return PDD_ERR_INVALID;
  }
  if (a->n_nodes < 1 || a->n_nodes >= ((int64_t)1 << 31) || a->n_h < 2 || a->n_h > 4096 ||
      !(a->h_min > 0) || !(a->h_max > a->h_min) || !std::isfinite(a->h_max) || a->n_paths < 2 ||
      !(a->delta > 0) || !(a->q > 0)) {
    set_error("pdd_fit_constants: bad arguments (need n_nodes >= 1, 2 <= n_h <= 4096, "
              "0 < h_min < h_max, n_paths >= 2, delta > 0, q > 0)");
    return PDD_ERR_INVALID;
  }
  for (int j = 0; j < pv.dim; ++j)
    if (!a->coords[j]) {
      set_error("pdd_fit_constants: coords[%d] is NULL", j);
      return PDD_ERR_INVALID;
    }
  const bool with_psi = a->grid_id != PDD_CV_NONE;
  const size_t n = (size_t)a->n_nodes, M = (size_t)a->n_h;
  // device: per (h, field, node) statistics, the nodes' coefficients, h and h^delta
  DeviceGuard guard(pv.device);  // restores the caller's device on return
  if (!guard.ok) {
    set_error("pdd_fit_constants: cannot select device %d", pv.device);
    return PDD_ERR_CUDA;
  }
  double* dstat = nullptr;
  const size_t n_stat = M * kF * n, n_back = n_stat + kC * n;
  cudaError_t e = cudaMalloc(&dstat, (n_back + 2 * M) * sizeof(double));
  if (e != cudaSuccess) {
    set_error("pdd_fit_constants: cudaMalloc: %s", cudaGetErrorString(e));
    return PDD_ERR_NOMEM;
  }
  std::vector<double> hs(2 * M);  // h, then h^delta
  for (size_t j = 0; j < M; ++j)
    hs[j] = a->h_max - (a->h_max - a->h_min) * (double)j / (double)(M - 1);
  int rc = PDD_OK;
  for (size_t j0 = 0; j0 < M && rc >= 0; j0 += PDD_MAX_LEVELS) {
    const size_t nl = std::min<size_t>(PDD_MAX_LEVELS, M - j0);
    std::vector<pdd_estimate_args> lv(nl);
    std::vector<pdd_node_stats> os(nl);
    for (size_t l = 0; l < nl; ++l) {
      const size_t j = j0 + l;
      pdd_estimate_args& x = lv[l];
      x = pdd_estimate_args{};
      x.n_nodes = a->n_nodes;
      for (int d = 0; d < 3; ++d) x.coords[d] = a->coords[d];
      x.coords_on_device = 1;
      x.grid_id = a->grid_id;
      x.n_paths = a->n_paths;
      x.dt = hs[j];
      x.kappa = 1.0;
      x.seed = a->seed;
      x.stream_tag = a->stream_tag_base + (uint32_t)j;
      pdd_node_stats& o = os[l];
      o = pdd_node_stats{};
      o.on_device = 1;
      double* base = dstat + j * kF * n;
      o.mean_phi = base;
      o.var_phi = base + n;
      o.mean_steps = base + 2 * n;
      o.cov_phi_xi = base + 3 * n;
      o.var_xi = base + 4 * n;
    }
    rc = pdd_estimate_levels(p, (int)nl, lv.data(), os.data(), 0);
  }
  std::vector<double> hstat(n_back);
  if (rc >= 0) {
    for (size_t j = 0; j < M; ++j) hs[M + j] = std::pow(hs[j], a->delta);
    double* const hx = dstat + n_back;
    const int staged = (kFits + 1) * M <= kStageDoubles;
    e = cudaMemcpyAsync(hx, hs.data(), 2 * M * sizeof(double), cudaMemcpyHostToDevice, pv.stream);
    if (e == cudaSuccess) {
      fit_nodes<<<(unsigned)n, 32 * (with_psi ? kFits : kFits - 2),
                  staged ? (kFits + 1) * M * sizeof(double) : 0, pv.stream>>>(
          dstat, hx, (int)M, n, staged, dstat + n_stat);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(hstat.data(), dstat, n_back * sizeof(double), cudaMemcpyDeviceToHost,
                          pv.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(pv.stream);
    if (e != cudaSuccess) {
      set_error("pdd_fit_constants: %s", cudaGetErrorString(e));
      rc = PDD_ERR_CUDA;
    }
    std::lock_guard<std::mutex> lk(*pv.mu);
    *pv.launches += 1;
  }
  cudaFree(dstat);
  if (rc < 0) return rc;
  auto stat = [&](size_t j, int f, size_t i) { return hstat[(j * kF + f) * n + i]; };
  for (size_t i = 0; i < n; ++i) {
    // A node whose paths all leave at k = 0 at some time step of the cloud
    // (mean exit index exactly 0, so phi is deterministic there: the node lies
    // inside the shrinkage layer c0 sqrt(h) of the boundary) is outside the
    // model E[eta_h] = E[eta_0] + B h^delta the fits assume: its constants are
    // NaN and the schedule leaves it out.
    bool degenerate = false;
    for (size_t j = 0; j < M; ++j) degenerate |= !(stat(j, 2, i) > 0.0);
    if (degenerate) {
      double* const outs[9] = {out->E_phi, out->beta, out->V_phi, out->alpha, out->E_tau,
                               out->K, out->cov_phi_psi, out->V_psi, out->rho_phi_psi};
      for (double* o : outs)
        if (o) o[i] = NAN;
    }
    const double* const c = hstat.data() + n_stat + i * kC;
    const double e_phi = c[kEPhi], beta = c[kBeta], v_phi = c[kVPhi], alpha = c[kAlpha],
                 e_tau = c[kETau], cov0 = with_psi ? c[kCov0] : NAN,  // E[psi phi]: E psi = 0
                 v_psi = with_psi ? c[kVPsi] : NAN;
    const double K = 4.0 * a->q * a->q * e_tau * std::pow(2.0 * std::fabs(beta), 1.0 / a->delta);
    if (!degenerate) {
      if (out->E_phi) out->E_phi[i] = e_phi;
      if (out->beta) out->beta[i] = beta;
      if (out->V_phi) out->V_phi[i] = v_phi;
      if (out->alpha) out->alpha[i] = alpha;
      if (out->E_tau) out->E_tau[i] = e_tau;
      if (out->K) out->K[i] = K;
      if (out->cov_phi_psi) out->cov_phi_psi[i] = cov0;
      if (out->V_psi) out->V_psi[i] = v_psi;
      if (out->rho_phi_psi) out->rho_phi_psi[i] = cov0 / std::sqrt(v_phi * v_psi);
    }
    if (out->cloud)
      for (size_t j = 0; j < M; ++j) {
        double* const c = out->cloud + (i * M + j) * 6;
        c[0] = hs[j];
        c[1] = stat(j, 0, i);
        c[2] = stat(j, 1, i);
        c[3] = stat(j, 2, i) * hs[j];
        c[4] = stat(j, 3, i);
        c[5] = stat(j, 4, i);
      }
  }
  return rc;
}

// ---------------------------------------------------------------------------
// Algorithm 4: scheduling of the tolerance sequence a_J > ... > a_1 > a_0.
// ---------------------------------------------------------------------------
namespace {

struct SchedData {
  const pdd_schedule_args* a;
  double p;  // 2 + 1/delta
};

// Nodes the schedule uses: finite fitted constants, V[phi] > 0 and beta != 0
// (a node Algorithm 3 could not fit has NaN constants and is left out).
bool usable(const pdd_schedule_args& s, int64_t i) {
  return std::isfinite(s.K[i]) && std::isfinite(s.beta[i]) && std::isfinite(s.alpha[i]) &&
         std::isfinite(s.V_phi[i]) && std::isfinite(s.V_psi[i]) &&
         std::isfinite(s.rho_phi_psi[i]) && s.V_phi[i] > 0.0 && s.beta[i] != 0.0;
}

// Predicted cost of the level with tolerance aj using the control variate of
// the coarser level with tolerance a (the minimised objective of Algorithm 4).
double sched_cost(const SchedData& d, double a, double aj) {
  const pdd_schedule_args& s = *d.a;
  double tot = 0.0;
  for (int64_t i = 0; i < s.n_nodes; ++i) {
    if (!usable(s, i)) continue;
    double r2 = 1.0 - s.V_psi[i] * a * a * (1.0 - s.rho_phi_psi[i] * s.rho_phi_psi[i]) /
                          (4.0 * s.V_phi[i]);
    if (r2 < 0.0) r2 = 0.0;
    const double r = std::sqrt(r2);
    const double vr = 1.0 - r2 + std::fabs(s.alpha[i] * r / s.beta[i]) * aj;
    tot += s.K[i] * s.V_phi[i] * (s.kappa * vr + std::pow(aj / a, d.p));
  }
  return tot;
}

}  // namespace

extern "C" int pdd_schedule(const pdd_schedule_args* s, double* a, double* speedup,
                            int max_levels, int* n_levels) {
  if (!s || !a || !n_levels || max_levels < 1 || s->n_nodes < 1 || !s->K || !s->beta ||
      !s->alpha || !s->V_phi || !s->V_psi || !s->rho_phi_psi || !(s->delta > 0) ||
      !(s->kappa > 0) || !(s->a0 > 0)) {
    set_error("pdd_schedule: bad arguments");
    return PDD_ERR_INVALID;
  }
  SchedData d{s, 2.0 + 1.0 / s->delta};
  double plain = 0.0, amax = 0.0;
  int64_t n_usable = 0;
  for (int64_t i = 0; i < s->n_nodes; ++i) {
    if (!usable(*s, i)) continue;
    ++n_usable;
    plain += s->K[i] * s->V_phi[i];
    const double c = s->V_psi[i] * (1.0 - s->rho_phi_psi[i] * s->rho_phi_psi[i]) /
                     (4.0 * s->V_phi[i]);
    if (c > 0) amax = std::max(amax, 1.0 / std::sqrt(c));
  }
  if (n_usable == 0) {
    set_error("pdd_schedule: no node has usable fitted constants");
    return PDD_ERR_INVALID;
  }
  const double min_s = s->min_speedup > 0 ? s->min_speedup : 1.5;
  a[0] = s->a0;
  int J = 0;
  double aj = s->a0;
  if (speedup)
    for (int k = 0; k <= max_levels; ++k) speedup[k] = NAN;  // steps not taken
  while (J < max_levels && aj < amax) {
    // log-spaced scan of (aj, amax], then golden-section refinement
    const int kScan = 2000;
    const double l0 = std::log(aj), l1 = std::log(amax);
    int best = 1;
    double bestv = 1e300;
    for (int k = 1; k <= kScan; ++k) {
      const double v = sched_cost(d, std::exp(l0 + (l1 - l0) * k / kScan), aj);
      if (v < bestv) {
        bestv = v;
        best = k;
      }
    }
    double lo = l0 + (l1 - l0) * (best - 1) / kScan, hi = l0 + (l1 - l0) * std::min(best + 1, kScan) / kScan;
    const double g = 0.5 * (std::sqrt(5.0) - 1.0);
    double x1 = hi - g * (hi - lo), x2 = lo + g * (hi - lo);
    double f1 = sched_cost(d, std::exp(x1), aj), f2 = sched_cost(d, std::exp(x2), aj);
    for (int it = 0; it < 200 && hi - lo > 1e-14; ++it) {
      if (f1 < f2) {
        hi = x2;
        x2 = x1;
        f2 = f1;
        x1 = hi - g * (hi - lo);
        f1 = sched_cost(d, std::exp(x1), aj);
      } else {
        lo = x1;
        x1 = x2;
        f1 = f2;
        x2 = lo + g * (hi - lo);
        f2 = sched_cost(d, std::exp(x2), aj);
      }
    }
    const double xbest = f1 < f2 ? x1 : x2;
    const double fbest = std::min(f1, f2);
    const double S = plain / std::min(fbest, bestv);
    const double anext = fbest <= bestv ? std::exp(xbest) : std::exp(l0 + (l1 - l0) * best / kScan);
    if (speedup) speedup[J] = S;
    if (S < min_s) break;
    a[++J] = anext;
    aj = anext;
  }
  *n_levels = J;
  return PDD_OK;
}

// ---------------------------------------------------------------------------
// Balanced simulation per node (Definition "Balanced MC simulation",
// eq. F:N_y_h) and the scheduling model's per-level prediction (Algorithm 4,
// eq. F:Sensitivity_formula), used to run the levels Algorithm 4 schedules
// (Algorithm 5: "for node x_i and a_j, determine h and N").
// ---------------------------------------------------------------------------
extern "C" int pdd_balanced_plan(int64_t n_nodes, double a, double q, double delta,
                                 const double* beta, const double* var, double h_min,
                                 double h_max, int64_t n_min, int64_t n_max, double* h,
                                 int64_t* n_paths) {
  if (n_nodes < 0 || !(a > 0) || !std::isfinite(a) || !(q > 0) || !(delta > 0) ||
      !(h_min > 0) || !(h_max >= h_min) || !std::isfinite(h_max) || n_min < 1 ||
      n_max < n_min || (n_nodes > 0 && (!beta || !var || !h || !n_paths))) {
    set_error("pdd_balanced_plan: bad arguments (need a, q, delta > 0, 0 < h_min <= h_max, "
              "1 <= n_min <= n_max, non-NULL arrays)");
    return PDD_ERR_INVALID;
  }
  for (int64_t i = 0; i < n_nodes; ++i) {
    // bias |beta| h^delta = a / 2 and statistical error q sqrt(V / N) = a / 2
    const double b = std::fabs(beta[i]);
    double hi = b > 0 ? std::pow(a / (2.0 * b), 1.0 / delta) : h_max;
    if (!(hi >= h_min)) hi = h_min;  // also catches NaN
    if (hi > h_max) hi = h_max;
    h[i] = hi;
    const double v = var[i] > 0 ? var[i] : 0.0;
    const double nn = std::ceil(4.0 * q * q * v / (a * a));
    int64_t ni = nn >= (double)n_max || !std::isfinite(nn) ? n_max : (int64_t)nn;
    if (ni < n_min) ni = n_min;
    n_paths[i] = ni;
  }
  return PDD_OK;
}

extern "C" int pdd_schedule_predict(const pdd_schedule_args* s, double a, double aj, double* rho2,
                                    double* cost) {
  if (!s || s->n_nodes < 1 || !s->K || !s->beta || !s->alpha || !s->V_phi || !s->V_psi ||
      !s->rho_phi_psi || !(s->delta > 0) || !(aj > 0) || !rho2 || !cost) {
    set_error("pdd_schedule_predict: bad arguments");
    return PDD_ERR_INVALID;
  }
  const double p = 2.0 + 1.0 / s->delta;
  const double scale = std::pow(aj, -p);
  for (int64_t i = 0; i < s->n_nodes; ++i) {
    const double base = s->K[i] * s->V_phi[i] * scale;  // plain cost at aj (eq. F:Pointwise_cost)
    if (!(a > 0)) {
      rho2[i] = 0.0;
      cost[i] = base;
      continue;
    }
    double r2 = 1.0 - s->V_psi[i] * a * a * (1.0 - s->rho_phi_psi[i] * s->rho_phi_psi[i]) /
                          (4.0 * s->V_phi[i]);
    if (r2 < 0.0) r2 = 0.0;
    const double r = std::sqrt(r2);
    const double loss = std::fabs(s->alpha[i] * r / s->beta[i]) * aj;
    rho2[i] = std::max(r2 - loss, 0.0);
    cost[i] = base * (1.0 - r2 + loss);
  }
  return PDD_OK;
}
