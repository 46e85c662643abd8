// gbpf_multi64.cu -- the FP64 instantiations of gbpf_multi.cuh.
#include "gbpf_multi.cuh"

namespace gbpf {

int multi_clusters_f64(int C, size_t smem) { return multi_clusters_t<double>(C, smem); }

cudaError_t multi_run_f64(const MultiArgs &a, size_t smem, cudaStream_t s) {
    return multi_run_t<double>(a, smem, s);
}

cudaError_t multi_pack_f64(const MultiArgs *args, const int *order, int ngrid, unsigned *counter, size_t smem,
                           int groups, int C, cudaStream_t s) {
    return multi_pack_t<double>(args, order, ngrid, counter, smem, groups, C, s);
}

cudaError_t multi_lowrank_f64(const MultiArgs &a, int which, void *Z, size_t smem, cudaStream_t s) {
    return multi_lowrank_t<double>(a, which, Z, smem, s);
}

}  // namespace gbpf
