// The path kernels of problem Cube3.
#include "pdd_paths.cuh"

template struct pdd::PathLaunch<pdd::Cube3>;
