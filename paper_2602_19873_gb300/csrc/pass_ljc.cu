// Instantiation of the neighborhood pass kernel for PASS_LJC, Lennard-Jones
// plus Coulomb at an interaction cutoff inside the list radius (pass_packed.cuh; tiles of
// fewer than 64 pairs: pass_impl.cuh).
#include "pass_impl.cuh"
#include "pass_packed.cuh"

namespace nlg {
cudaError_t launch_pass_ljc(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s)
{
    return a.packed ? launch_packed<PASS_LJC>(a, M, per, grid, threads, s)
                    : launch_k<PASS_LJC, false>(a, M, per, grid, threads, s);
}
}  // namespace nlg
