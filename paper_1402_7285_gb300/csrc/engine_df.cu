// Instantiations of the persistent panel solver for df panel vectors.
#include "engine.cuh"

namespace tbgf {

bool launch_engine_df(EngineLaunch &L, int b) { return L.run<df>(b); }

} // namespace tbgf
