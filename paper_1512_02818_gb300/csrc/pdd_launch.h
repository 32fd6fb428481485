// pdd_launch.h -- launchers of the path kernels of one problem.
#pragma once

#include <cuda_runtime.h>

#include "pdd_internal.h"

namespace pdd {

struct Cfg0;
struct Aniso;
struct Cube3;
struct Harmonic;
struct PaperEx;

// Defined in pdd_paths.cuh and instantiated once per problem (pdd_paths_*.cu).
template <class P>
struct PathLaunch {
  static cudaError_t paths(int precision, int cv, bool multi, const PathArgs& a, int num_sms,
                           cudaStream_t st, LaunchInfo* info);
  static cudaError_t occupancy(int precision, int cv, bool multi, int threads, int* occ);
  static cudaError_t coupled(int cv, const PathArgs& a, int num_sms, cudaStream_t st, LaunchInfo* info);
};

}  // namespace pdd
