// FFT plans of the mesh sides 256, 288 (fft_kernels.cuh).
#include "fft_kernels.cuh"

namespace pmr {

const FFTOps* fft_plans_3(int N) {
    switch (N) {
        case 256: return Plan<Reg<16, 16>, Reg<16, 8>>::ops();
        case 288: return Plan<Reg<24, 12>, Reg<24, 6>>::ops();
        default: return nullptr;
    }
}

}  // namespace pmr
