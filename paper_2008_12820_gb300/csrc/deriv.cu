// deriv.cu -- eighth-order central finite differences for first derivatives
// (paper Section 4.2), the paper's GPU alternative to spectral differentiation:
//   df/dx_d (x) ~ (1/h_d) sum_{j=1..4} c_j (f(x + j e_d) - f(x - j e_d)),
//   c = (4/5, -1/5, 4/105, -1/280), periodic.
// A block covers 32 consecutive x3 points of 8 x2 rows and walks a few planes
// along x1: a thread keeps its nine x1 neighbours in registers (one new load per
// voxel) and the offsets of its x2 and x3 neighbours, wrapped once; those 16
// come through L1.  One thread per voxel, which wrapped and multiplied out 24
// addresses, was bound by that: gradient at 192^3 84 -> 57 us, divergence
// 82 -> 68 us (17 us at the copy rate; the latency of the remaining loads binds).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "claire_internal.cuh"

namespace claire {

namespace {

constexpr int DX = 32, DY = 8;

__device__ __forceinline__ int wrapn(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// outputs are FP32, or FP16 in the FP16-storage form (FP32 arithmetic)
__device__ __forceinline__ float ldd(const float *p) { return __ldg(p); }
__device__ __forceinline__ void std_(float *p, float v) { *p = v; }
__device__ __forceinline__ void std_(__half *p, float v) { *p = __float2half_rn(v); }


// the difference sum of a line: p(k), k = -4 .. 4
template <typename P>
__device__ __forceinline__ float fd8(const P &at, float ih) {
    const float c1 = 4.f / 5.f, c2 = -1.f / 5.f, c3 = 4.f / 105.f, c4 = -1.f / 280.f;
    float r = c4 * (at(4) - at(-4));
    r = fmaf(c3, at(3) - at(-3), r);
    r = fmaf(c2, at(2) - at(-2), r);
    r = fmaf(c1, at(1) - at(-1), r);
    return r * ih;
}

// walks the planes of a block's column of f1 along x1, calling body(o, at) with
// the voxel's offset and its x1 neighbours; at2, at3 offsets are the caller's
template <typename B>
__device__ __forceinline__ void march_x1(const float *__restrict__ f1, const Dims &d, int march, long long s1,
                                         long long o2, const B &body) {
    const int first = blockIdx.z * march, last = min(first + march, d.n1);
    float w[9];  // x1 neighbours i1 - 4 .. i1 + 4 (n1 >= 4: one period off at most)
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = ldd(f1 + wrapn(first + k - 4, d.n1) * s1 + o2);
    for (int i1 = first;;) {
        body(i1 * s1 + o2, [&](int k) { return w[k + 4]; });
        if (++i1 >= last) break;
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = w[k + 1];
        w[8] = ldd(f1 + wrapn(i1 + 4, d.n1) * s1 + o2);
    }
}

// the same for the one plane blockIdx.z
template <typename B>
__device__ __forceinline__ void one_x1(const float *__restrict__ f1, const Dims &d, long long s1, long long o2,
                                       const B &body) {
    const int i1 = blockIdx.z;
    body(i1 * s1 + o2, [&](int k) { return ldd(f1 + wrapn(i1 + k, d.n1) * s1 + o2); });
}

// offsets of the eight neighbours along an axis of length n and stride s
__device__ __forceinline__ void offsets8(int i, int n, int s, int *o) {
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
        o[3 + k] = (wrapn(i + k, n) - i) * s;
        o[4 - k] = (wrapn(i - k, n) - i) * s;
    }
}
__device__ __forceinline__ int slot8(int k) { return k > 0 ? 3 + k : 4 + k; }

template <typename TO, bool MANY>
__global__ void __launch_bounds__(DX * DY) k_grad_fd8(const float *__restrict__ f, TO *__restrict__ g,
                                                      Dims d, int march, float ih1, float ih2, float ih3) {
    const int i3 = blockIdx.x * DX + threadIdx.x, i2 = blockIdx.y * DY + threadIdx.y;
    if (i3 >= d.n3 || i2 >= d.n2) return;
    int o2[8], o3[8];
    offsets8(i2, d.n2, d.n3, o2);
    offsets8(i3, d.n3, 1, o3);
    const long long s1 = (long long)d.n2 * d.n3, col = (long long)i2 * d.n3 + i3;
    auto body = [&](long long o, const auto &at1) {
        std_(g + o, fd8(at1, ih1));
        std_(g + d.N + o, fd8([&](int k) { return ldd(f + o + o2[slot8(k)]); }, ih2));
        std_(g + 2 * d.N + o, fd8([&](int k) { return ldd(f + o + o3[slot8(k)]); }, ih3));
    };
    if (MANY) march_x1(f, d, march, s1, col, body);
    else one_x1(f, d, s1, col, body);
}

template <bool MANY>
__global__ void __launch_bounds__(DX * DY) k_div_fd8(const float *__restrict__ v, float *__restrict__ out,
                                                     Dims d, int march, float ih1, float ih2, float ih3) {
    const int i3 = blockIdx.x * DX + threadIdx.x, i2 = blockIdx.y * DY + threadIdx.y;
    if (i3 >= d.n3 || i2 >= d.n2) return;
    int o2[8], o3[8];
    offsets8(i2, d.n2, d.n3, o2);
    offsets8(i3, d.n3, 1, o3);
    const float *v2 = v + d.N, *v3 = v + 2 * d.N;
    const long long s1 = (long long)d.n2 * d.n3, col = (long long)i2 * d.n3 + i3;
    auto body = [&](long long o, const auto &at1) {
        out[o] = fd8(at1, ih1) + fd8([&](int k) { return ldd(v2 + o + o2[slot8(k)]); }, ih2) +
                 fd8([&](int k) { return ldd(v3 + o + o3[slot8(k)]); }, ih3);
    };
    if (MANY) march_x1(v, d, march, s1, col, body);
    else one_x1(v, d, s1, col, body);
}

// planes per block: 16, or 8 or 4 where that leaves less than eight blocks per
// SM, and one where 4 does (75x90x50: marching took 13-17 us, one plane 12)
inline int march_of(const Dims &d) {
    const long long cols = (long long)((d.n3 + DX - 1) / DX) * ((d.n2 + DY - 1) / DY);
    for (int m = 16; m >= 4; m /= 2)
        if (cols * ((d.n1 + m - 1) / m) >= 8 * 152) return m;
    return 1;
}
inline dim3 grid_d(const Dims &d, int march) {
    return dim3((d.n3 + DX - 1) / DX, (d.n2 + DY - 1) / DY, (d.n1 + march - 1) / march);
}

}  // namespace

namespace {
template <typename TO>
void grad_fd8(const Dims &d, const float *f, TO *g, cudaStream_t st) {
    const double tp = 6.283185307179586476925286766559;
    const float i1 = (float)(d.n1 / tp), i2 = (float)(d.n2 / tp), i3 = (float)(d.n3 / tp);
    const int m = march_of(d);
    if (m > 1) k_grad_fd8<TO, true><<<grid_d(d, m), dim3(DX, DY), 0, st>>>(f, g, d, m, i1, i2, i3);
    else k_grad_fd8<TO, false><<<grid_d(d, m), dim3(DX, DY), 0, st>>>(f, g, d, m, i1, i2, i3);
}
}  // namespace

void launch_grad_fd8(const Dims &d, const float *f, float *g, cudaStream_t st, Profiler *prof) {
    ProfScope ps(prof, CLAIRE_K_FD, st, 16.0 * d.N);
    grad_fd8(d, f, g, st);
}

void launch_grad_fd8(const Dims &d, const float *f, __half *g, cudaStream_t st, Profiler *prof) {
    ProfScope ps(prof, CLAIRE_K_FD, st, 10.0 * d.N);
    grad_fd8(d, f, g, st);
}

void launch_div_fd8(const Dims &d, const float *v, float *out, cudaStream_t st, Profiler *prof) {
    const double tp = 6.283185307179586476925286766559;
    ProfScope ps(prof, CLAIRE_K_FD, st, 16.0 * d.N);
    const float i1 = (float)(d.n1 / tp), i2 = (float)(d.n2 / tp), i3 = (float)(d.n3 / tp);
    const int m = march_of(d);
    if (m > 1) k_div_fd8<true><<<grid_d(d, m), dim3(DX, DY), 0, st>>>(v, out, d, m, i1, i2, i3);
    else k_div_fd8<false><<<grid_d(d, m), dim3(DX, DY), 0, st>>>(v, out, d, m, i1, i2, i3);
}

}  // namespace claire
