// Instantiations of the local solver with Chebyshev sweeps for df vectors.
#include "local_engine.cuh"

namespace tbgf {

bool launch_local2_df(LocalLaunch2 &L, int b) { return L.run<df>(b); }

} // namespace tbgf
