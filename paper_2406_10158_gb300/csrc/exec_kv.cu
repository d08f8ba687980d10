// exec_kv.cu -- launchers of the key-value execute kernels (the workload
// policy is in kv_work.cuh).
#include "kv_work.cuh"

namespace gcc {
namespace {

template <int SC, int TPL = 0>
cudaError_t launch(uint32_t fb, const ExecArgs& a, int grid, int block, size_t smem, cudaStream_t s) {
    return fb == 16 ? launch_exec<SC, KvWork<16, TPL>>(a, grid, block, smem, s)
                    : launch_exec<SC, KvWork<8, TPL>>(a, grid, block, smem, s);
}
template <int SC>
cudaError_t launch_2pl(uint32_t fb, const ExecArgs& a, int grid, int block, size_t smem, cudaStream_t s) {
    return tpl_spread(a.n_meta) ? launch<SC, TPL_SPREAD>(fb, a, grid, block, smem, s)
                                : launch<SC>(fb, a, grid, block, smem, s);
}
template <int SC, int TPL = 0>
int occupancy(uint32_t fb, int block, size_t smem) {
    return fb == 16 ? exec_occupancy<SC, KvWork<16, TPL>>(block, smem)
                    : exec_occupancy<SC, KvWork<8, TPL>>(block, smem);
}
template <int SC>
int occupancy_2pl(uint32_t fb, uint64_t n_records, int block, size_t smem) {
    return tpl_spread(n_records) ? occupancy<SC, TPL_SPREAD>(fb, block, smem) : occupancy<SC>(fb, block, smem);
}

}  // namespace

cudaError_t launch_kv_exec(gcc_scheme scheme, uint32_t fb, const ExecArgs& a, int grid,
                           int block, size_t smem, cudaStream_t s) {
    switch (scheme) {
        case GCC_NO_WAIT_2PL: return launch_2pl<GCC_NO_WAIT_2PL>(fb, a, grid, block, smem, s);
        case GCC_2PL_WAIT_DIE: return launch_2pl<GCC_2PL_WAIT_DIE>(fb, a, grid, block, smem, s);
        case GCC_TO: return launch<GCC_TO>(fb, a, grid, block, smem, s);
        case GCC_OCC: return launch<GCC_OCC>(fb, a, grid, block, smem, s);
        case GCC_DET: return launch<GCC_DET>(fb, a, grid, block, smem, s);
        case GCC_TICTOC: return launch<GCC_TICTOC>(fb, a, grid, block, smem, s);
        case GCC_MVCC: return launch<GCC_MVCC>(fb, a, grid, block, smem, s);
    }
    return cudaErrorInvalidValue;
}

int kv_exec_occupancy(gcc_scheme scheme, uint32_t fb, uint64_t n_records, int block, size_t smem) {
    switch (scheme) {
        case GCC_NO_WAIT_2PL: return occupancy_2pl<GCC_NO_WAIT_2PL>(fb, n_records, block, smem);
        case GCC_2PL_WAIT_DIE: return occupancy_2pl<GCC_2PL_WAIT_DIE>(fb, n_records, block, smem);
        case GCC_TO: return occupancy<GCC_TO>(fb, block, smem);
        case GCC_OCC: return occupancy<GCC_OCC>(fb, block, smem);
        case GCC_DET: return occupancy<GCC_DET>(fb, block, smem);
        case GCC_TICTOC: return occupancy<GCC_TICTOC>(fb, block, smem);
        case GCC_MVCC: return occupancy<GCC_MVCC>(fb, block, smem);
    }
    return 0;
}

}  // namespace gcc
