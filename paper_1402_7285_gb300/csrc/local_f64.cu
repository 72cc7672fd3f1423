// Instantiations of the local solver with Chebyshev sweeps for double vectors.
#include "local_engine.cuh"

namespace tbgf {

bool launch_local2_f64(LocalLaunch2 &L, int b) { return L.run<double>(b); }

} // namespace tbgf
