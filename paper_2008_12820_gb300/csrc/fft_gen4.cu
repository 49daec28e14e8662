// fft_gen4.cu -- two-step register transforms (fft_gen.cuh) of the lengths 216, 225, 240.
#include "fft_gen.cuh"

namespace claire {

bool gen_pass4(int n, const GenPass &a, cudaStream_t st) {
    switch (n) {
        case 216: gen_launch<216>(a, st); return true;
        case 225: gen_launch<225>(a, st); return true;
        case 240: gen_launch<240>(a, st); return true;
        default: return false;
    }
}

}  // namespace claire
