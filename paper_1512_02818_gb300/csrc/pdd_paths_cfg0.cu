// The path kernels of problem Cfg0.
#include "pdd_paths.cuh"

template struct pdd::PathLaunch<pdd::Cfg0>;
