// fft_gen2.cu -- two-step register transforms (fft_gen.cuh) of the lengths 100, 108, 120, 135.
#include "fft_gen.cuh"

namespace claire {

bool gen_pass2(int n, const GenPass &a, cudaStream_t st) {
    switch (n) {
        case 100: gen_launch<100>(a, st); return true;
        case 108: gen_launch<108>(a, st); return true;
        case 120: gen_launch<120>(a, st); return true;
        case 135: gen_launch<135>(a, st); return true;
        default: return false;
    }
}

}  // namespace claire
