// Resident step kernels of every shape for the storage types this translation
// unit is compiled for (included by resident_*.cu, so that they compile in
// parallel).
#include <cuda_runtime.h>

#include "resident.cuh"

namespace lbmfvm_fv {

using namespace lbmfvm_dev;

namespace {

template <class S, int I>
const void *kernel_of(ResForm f) {
    using G = typename ResConfig<S, I>::G;
    constexpr bool B = res_borders<S, G>();
    if constexpr (res_borders_apart<S, G>())
        if (!f.borders)
            return f.general ? reinterpret_cast<const void *>(resident_kernel<S, G, true, false>)
                             : reinterpret_cast<const void *>(resident_kernel<S, G, false, false>);
    return f.general ? reinterpret_cast<const void *>(resident_kernel<S, G, true, B>)
                     : reinterpret_cast<const void *>(resident_kernel<S, G, false, B>);
}

template <class S, int I>
cudaError_t prepare_i(ResForm form, int *blocks) {
    using G = typename ResConfig<S, I>::G;
    const void *k = kernel_of<S, I>(form);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k, G::BLOCK, G::SMEM);
    return e;
}

template <class S, int I>
cudaError_t launch_i(ResForm form, const ResArgs<S> &r, int tiles, cudaStream_t stream) {
    using G = typename ResConfig<S, I>::G;
    void *args[] = {const_cast<ResArgs<S> *>(&r)};
    return cudaLaunchCooperativeKernel(kernel_of<S, I>(form), dim3(tiles), dim3(G::BLOCK), args, G::SMEM, stream);
}

template <class S, int I>
ResShape shape_i() {
    using G = typename ResConfig<S, I>::G;
    return ResShape{G::TW, G::TH, G::MAIL_BYTES};
}

}  // namespace

#define LBMFVM_RES_SWITCH(i, CALL)   \
    switch (i) {                     \
        case 0: return CALL(0);      \
        case 1: return CALL(1);      \
        case 2: return CALL(2);      \
        case 3: return CALL(3);      \
        case 4: return CALL(4);      \
        case 5:                      \
            if constexpr (res_shapes<S>() > 5) return CALL(5); \
    }

template <class S>
ResShape resident_shape(int i) {
#define CALL(I) (shape_i<S, I>())
    LBMFVM_RES_SWITCH(i, CALL)
#undef CALL
    return ResShape{};
}
template <class S>
cudaError_t resident_prepare(int i, ResForm form, int *blocks) {
#define CALL(I) (prepare_i<S, I>(form, blocks))
    LBMFVM_RES_SWITCH(i, CALL)
#undef CALL
    return cudaErrorInvalidValue;
}
template <class S>
cudaError_t resident_launch(int i, ResForm form, const ResArgs<S> &r, int tiles, cudaStream_t stream) {
#define CALL(I) (launch_i<S, I>(form, r, tiles, stream))
    LBMFVM_RES_SWITCH(i, CALL)
#undef CALL
    return cudaErrorInvalidValue;
}

#define LBMFVM_RESIDENT_INSTANTIATE(S)                                       \
    template ResShape resident_shape<S>(int);                                \
    template cudaError_t resident_prepare<S>(int, ResForm, int *);              \
    template cudaError_t resident_launch<S>(int, ResForm, const ResArgs<S> &, int, cudaStream_t);

}  // namespace lbmfvm_fv
