// The path kernels of problem PaperEx.
#include "pdd_paths.cuh"

template struct pdd::PathLaunch<pdd::PaperEx>;
