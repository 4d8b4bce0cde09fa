// hop_f16.cu -- Wilson hop kernels with F16 storage (one translation unit per
// precision): the shared-memory staged kernel of hop_async.cuh, and, when the
// handle selects it, the tensor-core kernel of hop_mma.cuh for 8 or more
// right-hand sides; several right-hand sides with two-row links go to the
// kernel of hop_shared.cuh.
#include "hop_async.cuh"
#include "hop_mma.cuh"
#include "hop_shared.cuh"

namespace lq {
LQ_INDEX_FAULTS_READER(index_faults_f16)
cudaError_t launch_hop_f16(const HopArgs& a, bool r12, bool dag, int epi, int block, cudaStream_t st) {
    (void)block;
    if (hop_mma_applies(a, r12, epi)) return launch_hop_mma<LQ_F16>(a, dag, epi, st);
    if (r12 && hop_shared_applies<LQ_F16>(a)) return launch_hop_shared<LQ_F16, true>(a, dag, epi, st);
    return launch_hop_async<LQ_F16>(a, r12, dag, epi, st);
}
cudaError_t launch_hop_batch_f16(const HopArgs* args, const int* lat_off, int nlat, bool r12, bool dag, int epi,
                                 int grid, cudaStream_t st, int* occ) {
    return launch_hop_batch_prec<LQ_F16>(args, lat_off, nlat, r12, dag, epi, grid, st, occ);
}
}  // namespace lq
