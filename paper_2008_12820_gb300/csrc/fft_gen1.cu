// fft_gen1.cu -- two-step register transforms (fft_gen.cuh) of the lengths 60, 72, 75, 80, 90.
#include "fft_gen.cuh"

namespace claire {

bool gen_pass1(int n, const GenPass &a, cudaStream_t st) {
    switch (n) {
        case 60: gen_launch<60>(a, st); return true;
        case 72: gen_launch<72>(a, st); return true;
        case 75: gen_launch<75>(a, st); return true;
        case 80: gen_launch<80>(a, st); return true;
        case 90: gen_launch<90>(a, st); return true;
        default: return false;
    }
}

}  // namespace claire
