// FFT plans of the mesh sides 432 (fft_kernels.cuh).
#include "fft_kernels.cuh"

namespace pmr {

const FFTOps* fft_plans_5(int N) {
    switch (N) {
        case 432: return Plan<Reg<36, 12, 8>,  // 16 columns: 154 us a pass against 130
                               Reg<18, 12>>::ops();
        default: return nullptr;
    }
}

}  // namespace pmr
