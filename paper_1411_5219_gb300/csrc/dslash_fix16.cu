// Instantiation of the sixteen-lane fixed-point FP64 hopping kernel.
#include "dslash_fix.cuh"

namespace qcd {

cudaError_t launch_dslash_fix_lanes(const DslashLaunch &a, cudaStream_t s) { return launch_dslash_fix16(a, s); }

}  // namespace qcd
