// Instantiation of the fixed-point FP64 hopping kernel, dagger = 0 (one
// translation unit per dagger value, so that they compile in parallel).
#include "dslash_fix.cuh"

namespace qcd {

cudaError_t launch_dslash_fix_d0(const DslashLaunch &a, cudaStream_t s) { return launch_dslash_fix_dag<0>(a, s); }

cudaError_t launch_dslash_fix_multi_d0(const DslashMulti &a, cudaStream_t s) { return launch_dslash_fix_multi<0>(a, s); }

}  // namespace qcd
