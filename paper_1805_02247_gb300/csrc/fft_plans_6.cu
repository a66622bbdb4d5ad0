// FFT plans of the mesh sides 486 (fft_kernels.cuh).
#include "fft_kernels.cuh"

namespace pmr {

const FFTOps* fft_plans_6(int N) {
    switch (N) {
        case 486: return Plan<Reg<27, 18>, Reg<27, 9>>::ops();
        default: return nullptr;
    }
}

}  // namespace pmr
