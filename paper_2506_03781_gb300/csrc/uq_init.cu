// The initialization (uq_init.cuh) of every bit-width: q = 4 compiled here, the
// others in uq_init_q123.cu, side by side (one file takes two minutes).
#include "uq_init.cuh"

namespace uq {

extern template cudaError_t launch_init_q<1>(const Shape&, const void*, int, int, int, uq_params, uint8_t*, cudaStream_t);
extern template cudaError_t launch_init_q<2>(const Shape&, const void*, int, int, int, uq_params, uint8_t*, cudaStream_t);
extern template cudaError_t launch_init_q<3>(const Shape&, const void*, int, int, int, uq_params, uint8_t*, cudaStream_t);

cudaError_t launch_init(const Shape& sh, const void* W, int G, int T, int clip, uq_params p, uint8_t* codes,
                        cudaStream_t st) {
    switch (sh.q) {
        case 1: return launch_init_q<1>(sh, W, G, T, clip, p, codes, st);
        case 2: return launch_init_q<2>(sh, W, G, T, clip, p, codes, st);
        case 3: return launch_init_q<3>(sh, W, G, T, clip, p, codes, st);
        default: return launch_init_q<4>(sh, W, G, T, clip, p, codes, st);
    }
}

}  // namespace uq
