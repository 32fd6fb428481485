// pdd_f64.cu -- the tables of the FP64 paths' elementary functions (F64Tables).
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <memory>
#include <mutex>

#include "pdd_device.cuh"
#include "pdd_internal.h"

namespace pdd {

__device__ F64Tables g_f64;

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_mu;
std::atomic<const F64Tables*> g_tables[kMaxDevices];

// Every entry rounded once from extended precision.
void fill(F64Tables& t) {
  const long double pi = 3.14159265358979323846264338327950288L;
  const long double ln2 = 0.693147180559945309417232121458176568L;
  for (int i = 0; i < 4096; ++i) {
    const long double a = 2.0L * pi * i / 4096.0L;
    t.turn[i] = make_double2((double)cosl(a), (double)sinl(a));
  }
  for (int i = 0; i < 2048; ++i) {
    const long double a = 2.0L * pi * (i + 0.5L) / 8388608.0L, h = sinl(0.5L * a);
    t.fine[i] = make_double2((double)(-2.0L * h * h), (double)sinl(a));  // cos a - 1
  }
  for (int i = 0; i < 1024; ++i) {
    const double mid = (1.0 + (i + 0.5) / 1024.0) * (i < 512 ? 1.0 : 0.5);
    const double r = i == 0 || i == 1023 ? 1.0 : (double)(float)(1.0 / mid);
    t.ln[i] = make_double2(r, (double)(2.0L * logl((long double)r)));
  }
  for (int i = 0; i < 32; ++i) t.ln2[i] = (double)(2.0L * i * ln2);
  for (int i = 0; i <= 512; ++i) {
    const long double x = i / 256.0L, v[3] = {sinl(x), cosl(x), expl(x)};
    for (int k = 0; k < 3; ++k) {
      t.unit[i][k] = (double)v[k];
      t.unit[i][3 + k] = (double)(v[k] - t.unit[i][k]);
    }
  }
}

}  // namespace

cudaError_t f64_tables(const F64Tables** tables) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  *tables = g_tables[dev].load(std::memory_order_acquire);
  if (*tables != nullptr) return cudaSuccess;
  std::lock_guard<std::mutex> lk(g_mu);
  *tables = g_tables[dev].load(std::memory_order_acquire);
  if (*tables != nullptr) return cudaSuccess;
  void* p = nullptr;
  e = cudaGetSymbolAddress(&p, g_f64);
  if (e != cudaSuccess) return e;
  static const std::unique_ptr<const F64Tables> host = [] {
    auto t = std::make_unique<F64Tables>();
    fill(*t);
    return t;
  }();
  cudaStream_t st = nullptr;
  e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(p, host.get(), sizeof(F64Tables), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaStreamDestroy(st);
  if (e != cudaSuccess) return e;
  *tables = (const F64Tables*)p;
  g_tables[dev].store(*tables, std::memory_order_release);
  return cudaSuccess;
}

}  // namespace pdd
