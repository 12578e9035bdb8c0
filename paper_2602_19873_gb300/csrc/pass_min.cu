// Instantiation of the neighborhood pass kernel for PASS_MIN, the distance to
// the nearest gather neighbor (a minimum reduction; pass_packed.cuh; tiles of
// fewer than 64 pairs: pass_impl.cuh).
#include "pass_impl.cuh"
#include "pass_packed.cuh"

namespace nlg {
cudaError_t launch_pass_min(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s)
{
    return a.packed ? launch_packed<PASS_MIN>(a, M, per, grid, threads, s)
                    : launch_k<PASS_MIN, false>(a, M, per, grid, threads, s);
}
}  // namespace nlg
