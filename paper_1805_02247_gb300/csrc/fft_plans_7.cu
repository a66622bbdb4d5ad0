// FFT plans of the mesh sides 512 (fft_kernels.cuh).
#include "fft_kernels.cuh"

namespace pmr {

const FFTOps* fft_plans_7(int N) {
    switch (N) {
        case 512: return Plan<Reg<16, 32>, Reg<16, 16>>::ops();
        default: return nullptr;
    }
}

}  // namespace pmr
