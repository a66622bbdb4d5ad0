// FFT plans of the mesh sides 324, 384 (fft_kernels.cuh).
#include "fft_kernels.cuh"

namespace pmr {

const FFTOps* fft_plans_4(int N) {
    switch (N) {
        case 324: return Plan<Reg<18, 18>, Reg<18, 9>>::ops();
        case 384: return Plan<Reg<24, 16>, Reg<8, 24>>::ops();
        default: return nullptr;
    }
}

}  // namespace pmr
