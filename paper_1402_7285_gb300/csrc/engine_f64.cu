// Instantiations of the persistent panel solver for double panel vectors.
#include "engine.cuh"

namespace tbgf {

bool launch_engine_f64(EngineLaunch &L, int b) { return L.run<double>(b); }

} // namespace tbgf
