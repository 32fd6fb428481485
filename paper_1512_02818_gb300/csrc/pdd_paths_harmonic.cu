// The path kernels of problem Harmonic.
#include "pdd_paths.cuh"

template struct pdd::PathLaunch<pdd::Harmonic>;
