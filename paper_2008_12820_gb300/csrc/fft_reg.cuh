// fft_reg.cuh -- register-resident line transforms for the lengths N = 16 G
// with G in {2, 4, 6, 8, 10, 12, 16}.
//
// A transform of such a length is two register steps with one exchange
// through shared memory between them, instead of one shared-memory round trip
// (and two barriers) per radix stage:
//   step 1: a thread holds the 16 elements j + G r of a line (read straight
//           from global memory) and takes their radix-16 DFT: outputs 16 j + r;
//   step 2: a thread holds the G elements k + 16 m, applies the remaining
//           stages (one radix G, or two radices with product G) in registers:
//           outputs k + 16 m, in natural order.
// Where G divides 16, the elements k + 16 m of the 16 / G butterflies
// k = j, j + G, ... are the elements j + G r that step 1 of the inverse
// transform needs: forward step 2, a pointwise multiplier and inverse step 1
// then run back to back in registers.  Butterflies, twiddles and the order of
// operations are those of the staged plans (radix_at).  When these passes came in,
// gradients, divergences, beta A and its inverse, matvecs and transported images
// were compared with the staged plans' and equal bit for bit on every grid tried;
// the x1 transforms without a multiplier (two-level preconditioner) may fuse other
// products: results 3e-8 to 1e-6 apart, both 4e-7 from 64 bits.
//
// Shared-memory layout: element e of a line lies at row e + e / 16.  With the
// lines innermost (strided passes) row stride TL, with the elements innermost
// (x3 passes) line stride 17 G: both steps then touch consecutive 8-byte
// words per 16 lanes, free of bank conflicts.
#pragma once

#include "fft_core.cuh"

namespace claire {
namespace {

// lengths that take the register-resident transforms
__host__ __device__ constexpr bool fft_reg(int n) {
    return n == 32 || n == 64 || n == 96 || n == 128 || n == 160 || n == 192 || n == 256;
}
__host__ __device__ constexpr bool reg_pow2(int n) { return (n & (n - 1)) == 0; }

template <int N>
struct RegPlan {
    static constexpr int G = N / 16;
    static constexpr bool P2 = reg_pow2(N);
    static constexpr int R1 = radix_at(N, 1);                      // first radix of step 2
    static constexpr int R2 = radix_at(N, 2) ? radix_at(N, 2) : 1;  // second, 1 if there is none
    static constexpr int ROWS = 17 * G;
    // twiddles of step 2, lanes k innermost: first radix, then second
    static constexpr int WA = 16 * (R1 - 1), WB = R2 > 1 ? 16 * R1 * (R2 - 1) : 0, W = WA + WB;
    // threads per line: step 1 has G items a line, step 2 sixteen
    static constexpr int TPL = P2 ? G : 16;
    static_assert(radix_at(N, 0) == 16 && R1 * R2 == G && num_stages(N) <= 3, "N = 16 G in at most three stages");
};

// the step-2 twiddles of a block, from the table tw[t] = exp(-2 pi i t / N)
template <int N, int T>
__device__ __forceinline__ void reg_twiddles(float2 *w, const float2 *__restrict__ tw) {
    using P = RegPlan<N>;
    for (int i = threadIdx.x; i < P::W; i += T) {
        int t;
        if (i < P::WA) {
            t = (i / 16 + 1) * (i % 16) * P::R2;
        } else {
            const int q = i - P::WA;
            t = (q / (16 * P::R1) + 1) * (q % (16 * P::R1));
        }
        w[i] = __ldg(tw + t);
    }
}

// Twiddle product of step 2; w = exp(-2 pi i t / N), conjugated for s = +1.
// The fused products are spelled out so that every pass rounds alike: S = -1
// and S = 0 (either direction, s = +-1 at run time) fuse a.x w, S = +1 fuses
// a.x w.x and a.y w.x.
template <int S>
__device__ __forceinline__ float2 reg_twmul(float2 a, float2 w, float s) {
    if constexpr (S > 0)
        return make_float2(__fmaf_rn(a.x, w.x, __fmul_rn(a.y, w.y)), __fmaf_rn(a.y, w.x, -__fmul_rn(a.x, w.y)));
    if constexpr (S == 0) w.y *= -s;
    return make_float2(__fmaf_rn(a.x, w.x, -__fmul_rn(a.y, w.y)), __fmaf_rn(a.x, w.y, __fmul_rn(a.y, w.x)));
}

// step 2 on the G elements k + 16 m, in place; w: reg_twiddles
template <int N, int S>
__device__ __forceinline__ void reg_step2(float2 *a, int k, const float2 *w, float s = (float)S) {
    using P = RegPlan<N>;
    if constexpr (P::R2 == 1) {
#pragma unroll
        for (int r = 1; r < P::R1; ++r) a[r] = reg_twmul<S>(a[r], w[(r - 1) * 16 + k], s);
        if constexpr (P::R1 == 8 && S == 0) dft8<false>(a, s);
        else dft<P::R1>(a, s);
    } else {
        float2 b[P::G];
#pragma unroll
        for (int r2 = 0; r2 < P::R2; ++r2) {
            float2 c[P::R1];
#pragma unroll
            for (int r = 0; r < P::R1; ++r) {
                c[r] = a[r2 + r * P::R2];
                if (r > 0) c[r] = reg_twmul<S>(c[r], w[(r - 1) * 16 + k], s);
            }
            dft<P::R1>(c, s);
#pragma unroll
            for (int r = 0; r < P::R1; ++r) b[r2 * P::R1 + r] = c[r];
        }
#pragma unroll
        for (int r1 = 0; r1 < P::R1; ++r1) {
            float2 c[P::R2];
#pragma unroll
            for (int r = 0; r < P::R2; ++r) {
                c[r] = b[r1 + r * P::R1];
                if (r > 0) c[r] = reg_twmul<S>(c[r], w[P::WA + (r - 1) * 16 * P::R1 + k + 16 * r1], s);
            }
            dft<P::R2>(c, s);
#pragma unroll
            for (int r = 0; r < P::R2; ++r) a[r1 + r * P::R1] = c[r];
        }
    }
}

// lines per block: 256 threads at N = 256 and 192, 128 below (more blocks on
// small grids), 64 at N = 32
template <int N>
struct RegTile {
    static constexpr int TL = N >= 128 ? 16 : (N == 96 ? 8 : 32);
    static constexpr int T = RegPlan<N>::TPL * TL;
};

// position of a block's line: offset of its plane and column within the row
__device__ __forceinline__ bool reg_line(const RegLines &q, int line, long long &off, int &col) {
    const int plane = line / q.ncol;
    col = line - plane * q.ncol;
    const int c = plane / q.nplane;
    off = c * q.cstride + (plane - c * q.nplane) * q.pstride;
    return line < q.nlines && col < q.nval;
}

// d/dx multiplier i k / n on element e (no contraction into a following add:
// the product is rounded as if it were stored)
template <int N>
__device__ __forceinline__ float2 reg_deriv(int e, float2 z, float sc) {
    const float k = wavenumber_d1(e, N) * sc;
    return make_float2(__fmul_rn(-k, z.y), __fmul_rn(k, z.x));
}

// forward step 2, pointwise multiplier f(e, z), inverse step 1, between two
// exchanges in `sm`; at(e) gives the word of element e of this thread's line.
// On entry the step-1 outputs lie in sm behind a barrier; on exit the inverse
// step-1 outputs do.  j: the thread's step-1 index, kk: its step-2 index
// (lines of composite G only; there every thread of a line has a kk).
template <int N, typename AT, typename F>
__device__ __forceinline__ void reg_middle(float2 *sm, const float2 *w, int j, const AT &at, const F &f) {
    using P = RegPlan<N>;
    float2 a[16];
    if constexpr (P::P2) {
        constexpr int I = 16 / P::G;
#pragma unroll
        for (int i = 0; i < I; ++i) {
            float2 b[P::G];
#pragma unroll
            for (int m = 0; m < P::G; ++m) b[m] = sm[at(j + P::G * i + 16 * m)];
            reg_step2<N, -1>(b, j + P::G * i, w);
#pragma unroll
            for (int m = 0; m < P::G; ++m) a[i + I * m] = f(j + P::G * i + 16 * m, b[m]);
        }
    } else {
        float2 b[P::G];
#pragma unroll
        for (int m = 0; m < P::G; ++m) b[m] = sm[at(j + 16 * m)];
        reg_step2<N, -1>(b, j, w);
#pragma unroll
        for (int m = 0; m < P::G; ++m) sm[at(j + 16 * m)] = f(j + 16 * m, b[m]);
        __syncthreads();
        if (j < P::G) {
#pragma unroll
            for (int r = 0; r < 16; ++r) a[r] = sm[at(j + P::G * r)];
        }
    }
    const bool act = P::P2 || j < P::G;
    if (act) dft<16>(a, 1.f);
    __syncthreads();  // the line's words are read; they may be overwritten
    if (act) {
#pragma unroll
        for (int r = 0; r < 16; ++r) sm[at(16 * j + r)] = a[r];
    }
    __syncthreads();
}

// The x1 pass's pointwise step at wavenumber (k1, k2, k3) for the three
// components a, b, c of one spectral point (kd = the wavenumber with an even
// axis's Nyquist index set to 0, used in the divergence penalty):
//   OP_A     beta |k|^2 I + gamma kd kd^T
//   OP_AINV  its inverse by Sherman-Morrison (identity at k = 0)
//   OP_X1INV scale only; OP_X1FWD nothing
// each times scale (the 1/N of the inverse transform).
template <int OP>
__device__ __forceinline__ void mul_point(float2 &pa, float2 &pb, float2 &pc, float k1, float k1d, float k2,
                                          float k2d, float k3, float k3d, const SpecParams &sp) {
    if (OP == OP_X1FWD) {
    } else if (OP == OP_X1INV) {
        pa = make_float2(pa.x * sp.scale, pa.y * sp.scale);
        pb = make_float2(pb.x * sp.scale, pb.y * sp.scale);
        pc = make_float2(pc.x * sp.scale, pc.y * sp.scale);
    } else {
        const float2 a = pa, b = pb, c = pc;
        const float kk = k1 * k1 + k2 * k2 + k3 * k3;
        const float kd2 = k1d * k1d + k2d * k2d + k3d * k3d;
        // fused products spelled out: every pass rounds alike
        const float2 kv = make_float2(__fmaf_rn(k3d, c.x, __fmaf_rn(k1d, a.x, __fmul_rn(k2d, b.x))),
                                      __fmaf_rn(k3d, c.y, __fmaf_rn(k1d, a.y, __fmul_rn(k2d, b.y))));
        float diag, coup;
        if (OP == OP_A) {
            diag = sp.beta * kk;
            coup = sp.gamma;
        } else {
            if (kk == 0.f) {
                diag = 1.f;
                coup = 0.f;
            } else {
                const float bk = sp.beta * kk;
                diag = 1.f / bk;
                coup = -sp.gamma * diag / (bk + sp.gamma * kd2);
            }
        }
        const float s = sp.scale;
        auto row = [&](float kd, const float2 &v) {
            const float ck = __fmul_rn(coup, kd);
            return make_float2(__fmul_rn(__fmaf_rn(diag, v.x, __fmul_rn(ck, kv.x)), s),
                               __fmul_rn(__fmaf_rn(diag, v.y, __fmul_rn(ck, kv.y)), s));
        };
        pa = row(k1d, a);
        pb = row(k2d, b);
        pc = row(k3d, c);
    }
}

// pair of adjacent columns i3, i3 + 1 (ok1: the second is inside the row)
__device__ __forceinline__ float2 ld_pair(const float *p, bool ok0, bool ok1, bool vec) {
    if (vec) return ok0 ? *reinterpret_cast<const float2 *>(p) : make_float2(0.f, 0.f);
    return make_float2(ok0 ? p[0] : 0.f, ok1 ? p[1] : 0.f);
}
__device__ __forceinline__ void st_pair(float *p, float2 v, bool ok0, bool ok1, bool vec) {
    if (vec) {
        if (ok0) *reinterpret_cast<float2 *>(p) = v;
    } else {
        if (ok0) p[0] = v.x;
        if (ok1) p[1] = v.y;
    }
}
__device__ __forceinline__ void st_pair(__half *p, float2 v, bool ok0, bool ok1, bool vec) {
    if (vec) {
        if (ok0) *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(v.x, v.y);
    } else {
        if (ok0) p[0] = __float2half_rn(v.x);
        if (ok1) p[1] = __float2half_rn(v.y);
    }
}

}  // namespace
}  // namespace claire
