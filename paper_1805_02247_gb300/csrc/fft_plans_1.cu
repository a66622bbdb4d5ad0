// FFT plans of the mesh sides 72, 96, 108, 128, 144 (fft_kernels.cuh).
#include "fft_kernels.cuh"

namespace pmr {

const FFTOps* fft_plans_1(int N) {
    switch (N) {
        case 72: return Plan<Reg<12, 6>, Reg<6, 6>>::ops();
        case 96: return Plan<Reg<12, 8>, Reg<12, 4>>::ops();
        case 108: return Plan<Reg<18, 6>, Reg<9, 6>>::ops();
        case 128: return Plan<Reg<16, 8>, Reg<8, 8>>::ops();
        case 144: return Plan<Reg<12, 12>, Reg<12, 6>>::ops();
        default: return nullptr;
    }
}

}  // namespace pmr
