// fft_gen.cuh -- two-step register transforms for 22 lengths that are not 16 G
// (fft_reg.cuh): 36, 40, 45, 48, 50, 54, 60, 72, 75, 80, 90, 100, 108, 120, 135,
// 144, 150, 180, 200, 216, 225 and 240.  The list (fft_gen*.cu) ends there because
// these were instantiated and measured; 81, 125, 162, 243, 250, the lengths below
// 32 and those above 256 take the staged plans.
//
// The radices of the runtime plan (4s, then 2, 3s, 5s) are split into two
// groups with products G1 and G2, as equal as their order allows: step 1 takes
// the first group on the elements j + G2 r of a line in registers (outputs
// G1 j + r), step 2, after one exchange through shared memory, the second group
// on k + G1 m (outputs k + G1 m in natural order).  Butterflies, twiddles and
// order of operations are those of the staged runtime plan, which these passes
// replace at these lengths; its stages of radix at most
// 5 took a shared-memory round trip, a barrier and run-time index divisions
// each.  Three components, before and after: 240^3 x3 forward 181 -> 91 us, x2
// 161 -> 67, x1 with multiplier 358 -> 127, x3 inverse 239 -> 109, derivatives
// 311 -> 110 (gradient and divergence, mean); 120x135x150 40 -> 30, 35 -> 16,
// 77 -> 28, 44 -> 38, 77 -> 45.
//
// Shared-memory layout: element e at row (e / G1) (G1 | 1) + e % G1.
#pragma once

#include "fft_reg.cuh"

namespace claire {
namespace {

// radices of the runtime plan
__host__ __device__ constexpr int gen_radix(int n, int s) {
    int st = 0;
    while (n % 4 == 0) { if (st == s) return 4; n /= 4; ++st; }
    while (n % 2 == 0) { if (st == s) return 2; n /= 2; ++st; }
    while (n % 3 == 0) { if (st == s) return 3; n /= 3; ++st; }
    while (n % 5 == 0) { if (st == s) return 5; n /= 5; ++st; }
    return 0;
}
__host__ __device__ constexpr int gen_stages(int n) {
    int s = 0;
    while (gen_radix(n, s)) ++s;
    return s;
}
__host__ __device__ constexpr int gen_prod(int n, int s0, int s1) {
    int p = 1;
    for (int s = s0; s < s1; ++s) p *= gen_radix(n, s);
    return p;
}
// stages of step 1: the split with the smallest larger group
__host__ __device__ constexpr int gen_split(int n) {
    int best = 1, bw = n;
    for (int s = 1; s < gen_stages(n); ++s) {
        const int a = gen_prod(n, 0, s), b = n / a, w = a > b ? a : b;
        if (w < bw) { bw = w; best = s; }
    }
    return best;
}
// twiddles of the stages [s0, s1): stage s has (R - 1) * (product before it)
__host__ __device__ constexpr int gen_wsize(int n, int s0, int s1) {
    int w = 0;
    for (int s = s0; s < s1; ++s) w += (gen_radix(n, s) - 1) * gen_prod(n, 0, s);
    return w;
}

template <int N>
struct GenPlan {
    static constexpr int NS = gen_stages(N), SP = gen_split(N);
    static constexpr int G1 = gen_prod(N, 0, SP), G2 = N / G1;
    static constexpr int ST = G1 | 1, ROWS = ST * G2;
    static constexpr int GM = G1 > G2 ? G1 : G2;  // threads per line
    static constexpr int W = gen_wsize(N, 0, NS);
    static constexpr int TL = GM <= 16 ? 16 : 8;  // lines per block
    static constexpr int T = GM * TL;
    static constexpr int MINB = GM <= 16 ? 768 / T : 512 / T;  // 80 or 128 registers
    __host__ __device__ static constexpr int row(int e) { return e / G1 * ST + e % G1; }
};

// twiddle tables of all stages, stage by stage: entry (r - 1) * P + k' with
// P the product of the radices before the stage and k' = 0 .. P - 1
template <int N, int T>
__device__ __forceinline__ void gen_twiddles(float2 *w, const float2 *__restrict__ tw) {
    using P = GenPlan<N>;
    for (int i = threadIdx.x; i < P::W; i += T) {
        int q = i, t = 0;
#pragma unroll
        for (int s = 0; s < P::NS; ++s) {
            const int before = gen_prod(N, 0, s), R = gen_radix(N, s), size = (R - 1) * before;
            if (q >= 0 && q < size) t = (q / before + 1) * (q % before) * (N / (before * R));
            q -= size;
        }
        w[i] = __ldg(tw + t);
    }
}

// stages [S0, S1) of the plan on a[0 .. G): a[q * done + d] with `done` the
// product of this group's earlier radices; k: index below the group's first
// product (0 in step 1); natural digit order out
template <int N, int SGN, int S0, int S1, int S = S0>
__device__ __forceinline__ void gen_group(float2 *a, int k, const float2 *w, float s) {
    if constexpr (S < S1) {
        constexpr int R = gen_radix(N, S), G = gen_prod(N, S0, S1), NS0 = gen_prod(N, 0, S0);
        constexpr int done = gen_prod(N, S0, S), Q = G / done, QR = Q / R, WO = gen_wsize(N, 0, S);
        float2 b[G];
#pragma unroll
        for (int q = 0; q < QR; ++q)
#pragma unroll
            for (int dd = 0; dd < done; ++dd) {
                float2 c[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    c[r] = a[(q + r * QR) * done + dd];
                    if (r > 0 && (NS0 > 1 || dd > 0))
                        c[r] = reg_twmul<SGN>(c[r], w[WO + (r - 1) * NS0 * done + k + NS0 * dd], s);
                }
                dft<R>(c, s);
#pragma unroll
                for (int r = 0; r < R; ++r) b[q * done * R + dd + r * done] = c[r];
            }
#pragma unroll
        for (int i = 0; i < G; ++i) a[i] = b[i];
        gen_group<N, SGN, S0, S1, S + 1>(a, k, w, s);
    }
}
template <int N, int SGN>
__device__ __forceinline__ void gen_step1(float2 *a, const float2 *w, float s = (float)SGN) {
    gen_group<N, SGN, 0, GenPlan<N>::SP>(a, 0, w, s);
}
template <int N, int SGN>
__device__ __forceinline__ void gen_step2(float2 *a, int k, const float2 *w, float s = (float)SGN) {
    gen_group<N, SGN, GenPlan<N>::SP, GenPlan<N>::NS>(a, k, w, s);
}

// forward step 2, f(e, z) on every element, inverse step 1, between exchanges
// (as reg_middle); j: this thread's index within its line, GM per line
template <int N, typename AT, typename F>
__device__ __forceinline__ void gen_middle(float2 *sm, const float2 *w, int j, const AT &at, const F &f) {
    using P = GenPlan<N>;
    if (j < P::G1) {
        float2 b[P::G2];
#pragma unroll
        for (int m = 0; m < P::G2; ++m) b[m] = sm[at(j + P::G1 * m)];
        gen_step2<N, -1>(b, j, w);
#pragma unroll
        for (int m = 0; m < P::G2; ++m) sm[at(j + P::G1 * m)] = f(j + P::G1 * m, b[m]);
    }
    __syncthreads();
    float2 a[P::G1];
    if (j < P::G2) {
#pragma unroll
        for (int r = 0; r < P::G1; ++r) a[r] = sm[at(j + P::G2 * r)];
        gen_step1<N, 1>(a, w);
    }
    __syncthreads();
    if (j < P::G2) {
#pragma unroll
        for (int r = 0; r < P::G1; ++r) sm[at(P::G1 * j + r)] = a[r];
    }
    __syncthreads();
}

// ------------------------------------------------------- the 3D passes -----
template <int N>
__global__ void __launch_bounds__(GenPlan<N>::T, GenPlan<N>::MINB)
kg_c2c(float2 *__restrict__ data, const float2 *__restrict__ tw, RegLines q, float s, float scale) {
    using P = GenPlan<N>;
    constexpr int TL = P::TL;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    gen_twiddles<N, P::T>(w, tw);
    __syncthreads();
    const int l = threadIdx.x % TL, j = threadIdx.x / TL;
    long long off;
    int col;
    const bool ok = reg_line(q, blockIdx.x * TL + l, off, col);
    float2 *base = data + off + col;
    if (j < P::G2) {
        float2 a[P::G1];
#pragma unroll
        for (int r = 0; r < P::G1; ++r) a[r] = ok ? base[(j + P::G2 * r) * q.estride] : make_float2(0.f, 0.f);
        if (scale != 1.f) {
#pragma unroll
            for (int r = 0; r < P::G1; ++r) a[r] = make_float2(__fmul_rn(a[r].x, scale), __fmul_rn(a[r].y, scale));
        }
        gen_step1<N, 0>(a, w, s);
#pragma unroll
        for (int r = 0; r < P::G1; ++r) sm[(P::ST * j + r) * TL + l] = a[r];
    }
    __syncthreads();
    if (j < P::G1) {
        float2 a[P::G2];
#pragma unroll
        for (int m = 0; m < P::G2; ++m) a[m] = sm[(j + P::ST * m) * TL + l];
        gen_step2<N, 0>(a, j, w, s);
        if (ok) {
#pragma unroll
            for (int m = 0; m < P::G2; ++m) base[(j + P::G1 * m) * q.estride] = a[m];
        }
    }
}

template <int N>
__global__ void __launch_bounds__(GenPlan<N>::T, GenPlan<N>::MINB)
kg_r2c(const float *__restrict__ in, float2 *__restrict__ out, const float2 *__restrict__ tw, long long nlines,
       int p3) {
    using P = GenPlan<N>;
    constexpr int TL = P::TL, H = N / 2 + 1;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    gen_twiddles<N, P::T>(w, tw);
    __syncthreads();
    const long long line0 = 2 * (long long)blockIdx.x * TL;
    for (int i = threadIdx.x; i < P::G2 * TL; i += P::T) {
        const int j = i % P::G2, l = i / P::G2;
        const long long la = line0 + 2 * l;
        const float *pa = in + la * N + j;
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
        float2 a[P::G1];
#pragma unroll
        for (int r = 0; r < P::G1; ++r)
            a[r] = make_float2(ok0 ? __ldg(pa + P::G2 * r) : 0.f, ok1 ? __ldg(pa + N + P::G2 * r) : 0.f);
        gen_step1<N, -1>(a, w);
#pragma unroll
        for (int r = 0; r < P::G1; ++r) sm[l * P::ROWS + P::ST * j + r] = a[r];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < P::G1 * TL; i += P::T) {
        const int k = i % P::G1, l = i / P::G1;
        float2 a[P::G2];
#pragma unroll
        for (int m = 0; m < P::G2; ++m) a[m] = sm[l * P::ROWS + k + P::ST * m];
        gen_step2<N, -1>(a, k, w);
#pragma unroll
        for (int m = 0; m < P::G2; ++m) sm[l * P::ROWS + k + P::ST * m] = a[m];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < H * TL; i += P::T) {
        const int l = i / H, k = i - l * H;
        const long long la = line0 + 2 * l;
        const float2 z = sm[l * P::ROWS + P::row(k)], zn = sm[l * P::ROWS + P::row(k == 0 ? 0 : N - k)];
        const float2 fa = make_float2(0.5f * (z.x + zn.x), 0.5f * (z.y - zn.y));
        const float2 fb = make_float2(0.5f * (z.y + zn.y), -0.5f * (z.x - zn.x));
        if (la < nlines) out[la * p3 + k] = fa;
        if (la + 1 < nlines) out[(la + 1) * p3 + k] = fb;
    }
}

// real lines 2l and 2l + 1 from step 2 of an inverse transform in sm.  Step 2
// leaves runs of G1 consecutive elements to neighbouring threads; where an
// addend is read as well, short runs go back through shared memory and out in
// whole rows (x3 inverse passes of a 120x135x150 matvec and preconditioner,
// G1 = 6: 62 -> 38 us on average; plain stores gain nothing from it:
// derivatives there 44.5 -> 48).
template <int N, bool ADD, typename TO>
__device__ __forceinline__ void gen_store_x3(float2 *sm, const float2 *w, TO *out, const float *add, long long line0,
                                             long long nlines) {
    using P = GenPlan<N>;
    constexpr bool ROWS_OUT = ADD && P::G1 < 12;
    for (int i = threadIdx.x; i < P::G1 * P::TL; i += P::T) {
        const int k = i % P::G1, l = i / P::G1;
        const long long la = line0 + 2 * l;
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
        float2 a[P::G2];
#pragma unroll
        for (int m = 0; m < P::G2; ++m) a[m] = sm[l * P::ROWS + k + P::ST * m];
        gen_step2<N, 1>(a, k, w);
        if (ROWS_OUT) {
#pragma unroll
            for (int m = 0; m < P::G2; ++m) sm[l * P::ROWS + k + P::ST * m] = a[m];
        } else {
#pragma unroll
            for (int m = 0; m < P::G2; ++m) {
                const long long o = la * N + k + P::G1 * m;
                if (ok0) str(out + o, ADD ? a[m].x + add[o] : a[m].x);
                if (ok1) str(out + o + N, ADD ? a[m].y + add[o + N] : a[m].y);
            }
        }
    }
    if (ROWS_OUT) {
        __syncthreads();
#pragma unroll 4
        for (int i = threadIdx.x; i < N * P::TL; i += P::T) {
            const int l = i / N, e = i - l * N;
            const long long la = line0 + 2 * l, o = la * N + e;
            const float2 z = sm[l * P::ROWS + P::row(e)];
            if (la < nlines) str(out + o, ADD ? z.x + add[o] : z.x);
            if (la + 1 < nlines) str(out + o + N, ADD ? z.y + add[o + N] : z.y);
        }
    }
}

template <int N, bool ADD>
__global__ void __launch_bounds__(GenPlan<N>::T, GenPlan<N>::MINB)
kg_c2r(const float2 *__restrict__ in, float *out, const float *add, const float2 *__restrict__ tw, long long nlines,
       int p3) {
    using P = GenPlan<N>;
    constexpr int TL = P::TL;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    gen_twiddles<N, P::T>(w, tw);
    __syncthreads();
    const long long line0 = 2 * (long long)blockIdx.x * TL;
    for (int i = threadIdx.x; i < P::G2 * TL; i += P::T) {
        const int j = i % P::G2, l = i / P::G2;
        const long long la = line0 + 2 * l;
        const float2 *pa = in + la * p3;
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
        const float2 zero = make_float2(0.f, 0.f);
        float2 a[P::G1];
#pragma unroll
        for (int r = 0; r < P::G1; ++r) {
            const int e = j + P::G2 * r;
            const bool lo = 2 * e <= N;
            const int k = lo ? e : N - e;
            float2 fa = ok0 ? __ldg(pa + k) : zero, fb = ok1 ? __ldg(pa + p3 + k) : zero;
            if (e == 0 || 2 * e == N) {
                fa.y = 0.f;
                fb.y = 0.f;
            }
            a[r] = lo ? make_float2(fa.x - fb.y, fa.y + fb.x) : make_float2(fa.x + fb.y, -fa.y + fb.x);
        }
        gen_step1<N, 1>(a, w);
#pragma unroll
        for (int r = 0; r < P::G1; ++r) sm[l * P::ROWS + P::ST * j + r] = a[r];
    }
    __syncthreads();
    gen_store_x3<N, ADD>(sm, w, out, add, line0, nlines);
}

// x1 forward, multiplier, x1 inverse of three components, in place; the
// components go through the steps one after another, the multiplier runs where
// a thread holds fewer elements of each (step 2 or the inverse step 1)
template <int N>
struct GenMul {
    static constexpr int TL = 8, T = GenPlan<N>::GM * TL;
    static constexpr size_t smem = (size_t)(3 * GenPlan<N>::ROWS * TL + GenPlan<N>::W) * sizeof(float2);
};
template <int N, int OP>
__global__ void __launch_bounds__(GenMul<N>::T, 512 / GenMul<N>::T)
kg_mul(float2 *__restrict__ data, const float2 *__restrict__ tw, RegLines q, int n2, int n3, SpecParams sp) {
    using P = GenPlan<N>;
    constexpr int TL = GenMul<N>::TL, T = GenMul<N>::T, CS = P::ROWS * TL;
    extern __shared__ float2 sm[];
    float2 *w = sm + 3 * CS;
    gen_twiddles<N, T>(w, tw);
    __syncthreads();
    const int l = threadIdx.x % TL, j = threadIdx.x / TL;
    long long off;
    int col;
    const int line = blockIdx.x * TL + l, i2 = line / q.ncol;
    const bool ok = reg_line(q, line, off, col);
    float2 *base = data + off + col;
    if (j < P::G2) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 a[P::G1];
#pragma unroll
            for (int r = 0; r < P::G1; ++r)
                a[r] = ok ? base[c * q.cstride + (j + P::G2 * r) * q.estride] : make_float2(0.f, 0.f);
            gen_step1<N, -1>(a, w);
#pragma unroll
            for (int r = 0; r < P::G1; ++r) sm[c * CS + (P::ST * j + r) * TL + l] = a[r];
        }
    }
    __syncthreads();
    const float k2 = wavenumber(i2, n2), k2d = wavenumber_d1(i2, n2);
    const float k3 = (float)col, k3d = ((n3 & 1) == 0 && 2 * col == n3) ? 0.f : k3;
    auto mul = [&](int e, float2 &x, float2 &y, float2 &z) {
        const float k1 = wavenumber(e, N), k1d = wavenumber_d1(e, N);
        mul_point<OP>(x, y, z, k1, k1d, k2, k2d, k3, k3d, sp);
    };
    if (j < P::G1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 b[P::G2];
#pragma unroll
            for (int m = 0; m < P::G2; ++m) b[m] = sm[c * CS + (j + P::ST * m) * TL + l];
            gen_step2<N, -1>(b, j, w);
#pragma unroll
            for (int m = 0; m < P::G2; ++m) sm[c * CS + (j + P::ST * m) * TL + l] = b[m];
        }
        // this thread's own elements, component by component in shared memory
#pragma unroll
        for (int m = 0; m < P::G2; ++m) {
            float2 *z = sm + (j + P::ST * m) * TL + l;
            mul(j + P::G1 * m, z[0], z[CS], z[2 * CS]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float2 a[P::G1];
        if (j < P::G2) {
#pragma unroll
            for (int r = 0; r < P::G1; ++r) a[r] = sm[c * CS + P::row(j + P::G2 * r) * TL + l];
            gen_step1<N, 1>(a, w);
        }
        __syncthreads();
        if (j < P::G2) {
#pragma unroll
            for (int r = 0; r < P::G1; ++r) sm[c * CS + (P::ST * j + r) * TL + l] = a[r];
        }
    }
    __syncthreads();
    if (j < P::G1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 b[P::G2];
#pragma unroll
            for (int m = 0; m < P::G2; ++m) b[m] = sm[c * CS + (j + P::ST * m) * TL + l];
            gen_step2<N, 1>(b, j, w);
            if (ok) {
#pragma unroll
                for (int m = 0; m < P::G2; ++m) base[c * q.cstride + (j + P::G1 * m) * q.estride] = b[m];
            }
        }
    }
}

// ---------------------------------------------------- axis derivatives -----
template <int N>
__device__ __forceinline__ float2 gen_deriv(int e, float2 z, float sc) {
    const float k = wavenumber_d1(e, N) * sc;
    return make_float2(__fmul_rn(-k, z.y), __fmul_rn(k, z.x));
}

template <int N, bool ADD, typename TO>
__global__ void __launch_bounds__(GenPlan<N>::T, GenPlan<N>::MINB)
kg_deriv_x3(const float *__restrict__ in, TO *out, const float *add, const float2 *__restrict__ tw,
            long long nlines) {
    using P = GenPlan<N>;
    constexpr int TL = P::TL;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    gen_twiddles<N, P::T>(w, tw);
    __syncthreads();
    const float sc = 1.f / (float)N;
    const long long line0 = 2 * (long long)blockIdx.x * TL;
    const int j = threadIdx.x % P::GM, l = threadIdx.x / P::GM;
    if (j < P::G2) {
        const long long la = line0 + 2 * l;
        const float *pa = in + la * N + j;
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
        float2 a[P::G1];
#pragma unroll
        for (int r = 0; r < P::G1; ++r)
            a[r] = make_float2(ok0 ? __ldg(pa + P::G2 * r) : 0.f, ok1 ? __ldg(pa + N + P::G2 * r) : 0.f);
        gen_step1<N, -1>(a, w);
#pragma unroll
        for (int r = 0; r < P::G1; ++r) sm[l * P::ROWS + P::ST * j + r] = a[r];
    }
    __syncthreads();
    gen_middle<N>(sm, w, j, [l](int e) { return l * P::ROWS + P::row(e); },
                  [sc](int e, float2 z) { return gen_deriv<N>(e, z, sc); });
    gen_store_x3<N, ADD>(sm, w, out, add, line0, nlines);
}

template <int N, bool ADD, typename TO>
__global__ void __launch_bounds__(GenPlan<N>::T, GenPlan<N>::MINB)
kg_deriv_strided(const float *__restrict__ in, TO *out, const float *add, const float2 *__restrict__ tw, RegLines q,
                 int n3, int vec) {
    using P = GenPlan<N>;
    constexpr int TL = P::TL;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    gen_twiddles<N, P::T>(w, tw);
    __syncthreads();
    const float sc = 1.f / (float)N;
    const int l = threadIdx.x % TL, j = threadIdx.x / TL;
    long long off;
    int col;
    const bool ok0 = reg_line(q, blockIdx.x * TL + l, off, col), ok1 = ok0 && 2 * col + 1 < n3;
    off += 2 * col;
    if (j < P::G2) {
        float2 a[P::G1];
#pragma unroll
        for (int r = 0; r < P::G1; ++r) a[r] = ld_pair(in + off + (j + P::G2 * r) * q.estride, ok0, ok1, vec);
        gen_step1<N, -1>(a, w);
#pragma unroll
        for (int r = 0; r < P::G1; ++r) sm[(P::ST * j + r) * TL + l] = a[r];
    }
    __syncthreads();
    gen_middle<N>(sm, w, j, [l](int e) { return P::row(e) * TL + l; },
                  [sc](int e, float2 z) { return gen_deriv<N>(e, z, sc); });
    if (j < P::G1) {
        float2 a[P::G2];
#pragma unroll
        for (int m = 0; m < P::G2; ++m) a[m] = sm[(j + P::ST * m) * TL + l];
        gen_step2<N, 1>(a, j, w);
#pragma unroll
        for (int m = 0; m < P::G2; ++m) {
            const long long o = off + (j + P::G1 * m) * q.estride;
            if (ADD) a[m] = cadd(a[m], ld_pair(add + o, ok0, ok1, vec));
            st_pair(out + o, a[m], ok0, ok1, vec);
        }
    }
}

// ------------------------------------------------------------- launching ---
template <int N>
void gen_launch(const GenPass &a, cudaStream_t st) {
    using P = GenPlan<N>;
    const unsigned lines = (unsigned)((a.q.nlines + P::TL - 1) / P::TL);
    const unsigned pairs = (unsigned)((a.nlines + 2 * P::TL - 1) / (2 * P::TL));
    switch (a.kind) {
        case GenPass::C2C: kg_c2c<N><<<lines, P::T, 0, st>>>(a.spec, a.tw, a.q, a.s, a.scale); break;
        case GenPass::R2C: kg_r2c<N><<<pairs, P::T, 0, st>>>(a.in, a.spec, a.tw, a.nlines, a.p3); break;
        case GenPass::C2R:
            if (a.add) kg_c2r<N, true><<<pairs, P::T, 0, st>>>(a.spec, a.out, a.add, a.tw, a.nlines, a.p3);
            else kg_c2r<N, false><<<pairs, P::T, 0, st>>>(a.spec, a.out, a.add, a.tw, a.nlines, a.p3);
            break;
        case GenPass::MUL_A:
        case GenPass::MUL_AINV: {
            const unsigned blocks = (unsigned)((a.q.nlines + GenMul<N>::TL - 1) / GenMul<N>::TL);
            if (a.kind == GenPass::MUL_A) {
                set_smem<kg_mul<N, OP_A>>(GenMul<N>::smem);
                kg_mul<N, OP_A><<<blocks, GenMul<N>::T, GenMul<N>::smem, st>>>(a.spec, a.tw, a.q, a.n2, a.n3, a.sp);
            } else {
                set_smem<kg_mul<N, OP_AINV>>(GenMul<N>::smem);
                kg_mul<N, OP_AINV><<<blocks, GenMul<N>::T, GenMul<N>::smem, st>>>(a.spec, a.tw, a.q, a.n2, a.n3, a.sp);
            }
            break;
        }
        case GenPass::DERIV_X3:
            if (a.out_h) kg_deriv_x3<N, false><<<pairs, P::T, 0, st>>>(a.in, a.out_h, a.add, a.tw, a.nlines);
            else if (a.add) kg_deriv_x3<N, true><<<pairs, P::T, 0, st>>>(a.in, a.out, a.add, a.tw, a.nlines);
            else kg_deriv_x3<N, false><<<pairs, P::T, 0, st>>>(a.in, a.out, a.add, a.tw, a.nlines);
            break;
        case GenPass::DERIV_STRIDED:
            if (a.out_h)
                kg_deriv_strided<N, false><<<lines, P::T, 0, st>>>(a.in, a.out_h, a.add, a.tw, a.q, a.n3, a.vec);
            else if (a.add)
                kg_deriv_strided<N, true><<<lines, P::T, 0, st>>>(a.in, a.out, a.add, a.tw, a.q, a.n3, a.vec);
            else kg_deriv_strided<N, false><<<lines, P::T, 0, st>>>(a.in, a.out, a.add, a.tw, a.q, a.n3, a.vec);
            break;
    }
}

}  // namespace
}  // namespace claire
