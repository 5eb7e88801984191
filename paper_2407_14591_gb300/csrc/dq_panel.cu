// Launch of the panel product (dq_panel.cuh): the sector's own order here, the split order in
// dq_panel_split.cu.
#include "dq_panel.cuh"

namespace dq {

size_t panel_scratch_bytes(const dq_sector* s, int dtype) {
    size_t es = dtype == DQ_F64 ? 8 : 4;
    return 256 + ((size_t)(s->D + 8) * es + 255) / 256 * 256;
}

extern template int run_panel_s<double, long long, 1, true>(const dq_sector*, const dq_terms*, const double*, double*,
                                                            void*, cudaStream_t);
extern template int run_panel_s<double, long long, 2, true>(const dq_sector*, const dq_terms*, const double*, double*,
                                                            void*, cudaStream_t);
extern template int run_panel_s<float, int, 1, true>(const dq_sector*, const dq_terms*, const float*, float*, void*,
                                                     cudaStream_t);
extern template int run_panel_s<float, int, 2, true>(const dq_sector*, const dq_terms*, const float*, float*, void*,
                                                     cudaStream_t);

template <typename T, typename XT, int NA>
static int run_panel_n(const dq_sector* s, const dq_terms* t, const T* x, T* y, void* ws, cudaStream_t st) {
    return t->split ? run_panel_s<T, XT, NA, true>(s, t, x, y, ws, st) : run_panel_s<T, XT, NA, false>(s, t, x, y, ws, st);
}

int launch_panel_matvec_ws(const dq_sector* s, const dq_terms* t, const void* x, void* y, int dtype, void* ws,
                           void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int na = t->pp.nA;
    if (dtype == DQ_F64) {
        if (na <= 1 && !t->pp.fold) return run_panel_n<double, long long, 1>(s, t, (const double*)x, (double*)y, ws, st);
        return run_panel_n<double, long long, 2>(s, t, (const double*)x, (double*)y, ws, st);
    }
    if (na <= 1) return run_panel_n<float, int, 1>(s, t, (const float*)x, (float*)y, ws, st);
    return run_panel_n<float, int, 2>(s, t, (const float*)x, (float*)y, ws, st);
}

int launch_panel_matvec(const dq_sector* s, dq_terms* t, const void* x, void* y, int dtype, void* stream) {
    size_t need = panel_scratch_bytes(s, dtype);
    if (t->scratch_bytes < need) {
        if (t->scratch) cudaFree(t->scratch);
        t->scratch = nullptr;
        t->scratch_bytes = 0;
        cudaError_t e = cudaMalloc(&t->scratch, need);
        if (e != cudaSuccess) return (int)e;
        t->scratch_bytes = need;
    }
    return launch_panel_matvec_ws(s, t, x, y, dtype, t->scratch, stream);
}

}  // namespace dq
