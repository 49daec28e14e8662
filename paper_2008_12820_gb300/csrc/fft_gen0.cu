// fft_gen0.cu -- two-step register transforms (fft_gen.cuh) of the lengths 36, 40, 45, 48, 50, 54.
#include "fft_gen.cuh"

namespace claire {

bool gen_pass0(int n, const GenPass &a, cudaStream_t st) {
    switch (n) {
        case 36: gen_launch<36>(a, st); return true;
        case 40: gen_launch<40>(a, st); return true;
        case 45: gen_launch<45>(a, st); return true;
        case 48: gen_launch<48>(a, st); return true;
        case 50: gen_launch<50>(a, st); return true;
        case 54: gen_launch<54>(a, st); return true;
        default: return false;
    }
}

}  // namespace claire
