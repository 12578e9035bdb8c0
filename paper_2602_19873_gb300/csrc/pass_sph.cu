// Instantiation of the neighborhood pass kernel for PASS_SPH (pass_packed.cuh; tiles of
// fewer than 64 pairs and supports other than 2: pass_impl.cuh).
#include "pass_impl.cuh"
#include "pass_packed.cuh"

namespace nlg {
cudaError_t launch_pass_sph(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s)
{
    return a.packed ? launch_packed<PASS_SPH>(a, M, per, grid, threads, s)
                    : launch_k<PASS_SPH, true>(a, M, per, grid, threads, s);
}
}  // namespace nlg
