// The path kernels of problem Aniso.
#include "pdd_paths.cuh"

template struct pdd::PathLaunch<pdd::Aniso>;
