// Resident steps of one storage precision (SF32): see resident_impl.cuh.
#include "resident_impl.cuh"

namespace cplbm {

cudaError_t launch_resident_f32(const ResidentArgs &a, bool batch, int grid, int threads,
                              size_t smem, cudaStream_t s)
{
    return launch_resident_t<SF32>(a, batch, grid, threads, smem, s);
}

}  // namespace cplbm
