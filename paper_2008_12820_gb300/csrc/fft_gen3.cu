// fft_gen3.cu -- two-step register transforms (fft_gen.cuh) of the lengths 144, 150, 180, 200.
#include "fft_gen.cuh"

namespace claire {

bool gen_pass3(int n, const GenPass &a, cudaStream_t st) {
    switch (n) {
        case 144: gen_launch<144>(a, st); return true;
        case 150: gen_launch<150>(a, st); return true;
        case 180: gen_launch<180>(a, st); return true;
        case 200: gen_launch<200>(a, st); return true;
        default: return false;
    }
}

}  // namespace claire
