// The panel product on the split order (any number of subsystems; see dq_panel.cpp): the table of
// canonical pieces and the kernels of dq_panel.cuh with the mapped stores.
#include "dq_panel.cuh"

namespace dq {

// First canonical index of every piece of every panel (PanelPlan::piece).
__global__ void k_panel_pieces(PanelPlan P, DevSector S) {
    const uint64_t n = (uint64_t)P.npanels * P.npiece, step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += step) {
        const uint32_t s0 = P.panel_s0[i / P.npiece], q = (uint32_t)(i % P.npiece);
        const int nl = P.N - __popc(s0) - __popc(q);
        P.piece[i] = nl < 0 || nl > P.Llow ? 0  // no row of the panel has this pattern
                                           : d_rank(S, S.off, S.str, ((uint64_t)s0 << P.L1) | ((uint64_t)q << P.Llow) | P.lowfirst[nl]);
    }
}

int launch_panel_pieces(const dq_sector* s, const PanelPlan& P) {
    if (!s->has_device) return 0;
    k_panel_pieces<<<sm_count_cached() * 8, 256>>>(P, s->dev);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaStreamSynchronize(0));
}

template int run_panel_s<double, long long, 1, true>(const dq_sector*, const dq_terms*, const double*, double*, void*,
                                                     cudaStream_t);
template int run_panel_s<double, long long, 2, true>(const dq_sector*, const dq_terms*, const double*, double*, void*,
                                                     cudaStream_t);
template int run_panel_s<float, int, 1, true>(const dq_sector*, const dq_terms*, const float*, float*, void*, cudaStream_t);
template int run_panel_s<float, int, 2, true>(const dq_sector*, const dq_terms*, const float*, float*, void*, cudaStream_t);

}  // namespace dq
