// fft.cu -- shared-memory pencil 3D FFT with fused spectral multipliers
// (paper Section 3, "Discretization": the vector Laplacian, the divergence
// penalty and their inverse are diagonal in Fourier space; first derivatives
// are spectral as well).
//
// A spectral operator out = F^-1[ M(k) F in ] runs as five pencil passes, each
// reading and writing HBM once:
//   1. x3 forward, real -> half spectrum.  Two real lines are packed into one
//      complex line, transformed, and separated by Hermitian symmetry.
//   2. x2 forward, complex, in place.
//   3. x1 forward, multiplier M(k) for all components at once (the divergence
//      penalty couples them), x1 inverse; in place.
//   4. x2 inverse, in place.
//   5. x3 inverse, half spectrum -> real, two lines per complex transform,
//      with an optional addend in the epilogue.
// Lengths 32, 64, 96, 128, 160, 192 and 256 (fft_reg.cuh) and 22 others from 36 to
// 240 (listed in fft_gen.cuh) run in registers around one exchange
// through shared memory.  At the remaining lengths a pass stages a tile of whole
// lines in shared memory and runs a mixed-radix Stockham FFT there.  Either way:
// natural-order output, no bit reversal, twiddles from a table computed in
// double on the host.
// Strided passes (x2, x1) load tiles of TK consecutive k3 columns so that
// every row access is a contiguous 8*TK-byte segment.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "claire_internal.cuh"
#include "fft_reg.cuh"

namespace claire {

namespace {
// ---------------------------------------------------------------- pass 1 ---
// x3 forward real -> half spectrum.  Block: L complex lines = 2L real lines.
template <int N, int L, typename TI = float>
__global__ void __launch_bounds__(kThreads)
k_r2c_x3(const TI *__restrict__ in, float2 *__restrict__ out, long long nlines, FftPlan p,
         int h3, int p3) {
    extern __shared__ float2 sm[];
    const int n = Fft<N>::size(p), ls = L + 1;
    float2 *A = sm, *B = sm + n * ls;
    const long long line0 = (long long)blockIdx.x * 2 * L;
    // real lines 2l and 2l+1 become the real and imaginary part of line l
        for (int t = threadIdx.x; t < L * n; t += blockDim.x) {
        const int l = t / n, e = t - l * n;
        const long long la = line0 + 2 * l;
        const float re = la < nlines ? ldr(in + la * n + e) : 0.f;
        const float im = la + 1 < nlines ? ldr(in + (la + 1) * n + e) : 0.f;
        A[e * ls + l] = make_float2(re, im);
    }
    __syncthreads();
    float2 *Rz = Fft<N>::template run<L>(A, B, p, ls, -1.f);
    if (N > 0) h3 = N / 2 + 1;
    for (int t = threadIdx.x; t < L * h3; t += blockDim.x) {
        const int l = t / h3, k = t - l * h3;
        const float2 z = Rz[k * ls + l];
        const float2 zn = Rz[((k == 0) ? 0 : (n - k)) * ls + l];
        // A_k = (Z_k + conj Z_{n-k})/2,  B_k = -i (Z_k - conj Z_{n-k})/2
        const float2 a = make_float2(0.5f * (z.x + zn.x), 0.5f * (z.y - zn.y));
        const float2 b = make_float2(0.5f * (z.y + zn.y), -0.5f * (z.x - zn.x));
        const long long la = line0 + 2 * l;
        if (la < nlines) out[la * p3 + k] = a;
        if (la + 1 < nlines) out[(la + 1) * p3 + k] = b;
    }
}

// Pass 1 with persistent blocks: the 2L real lines of the next tile (one
// contiguous chunk) are fetched by 16-byte cp.async into a staging buffer
// while the current tile is transformed, then transposed into the transform
// layout.  FP32 input, n a multiple of 4, 16-byte aligned (the launcher
// checks; otherwise the one-tile-per-block form above runs).
template <int N, int L>
__global__ void __launch_bounds__(kThreads, fft_in_place(N) ? 3 : 1)
k_r2c_x3_p(const float *__restrict__ in, float2 *__restrict__ out, long long nlines, FftPlan p, int h3, int p3,
           int nitems) {
    extern __shared__ float2 sm[];
    constexpr bool IP = fft_in_place(N);  // in-place transform: no scratch tile
    const int n = Fft<N>::size(p), ls = L + 1;
    float2 *A = sm, *B = sm + n * ls;
    float *S = reinterpret_cast<float *>(sm + (IP ? 1 : 2) * n * ls);
    auto load = [&](int item) {
        const long long line0 = (long long)item * 2 * L;
        const float *base = in + line0 * n;
        const int nch = (2 * L * n) / 4;
        for (int t = threadIdx.x; t < nch; t += blockDim.x) {
            const long long line = line0 + (4 * t) / n;
            const int bytes = line < nlines ? 16 : 0;
            cp_async16z(S + 4 * t, base + (bytes ? 4 * t : 0), bytes);
        }
        cp_async_commit_all();
    };
    const int i0 = blockIdx.x, stride = gridDim.x;
    if (i0 >= nitems) return;
    load(i0);
    if (N > 0) h3 = N / 2 + 1;
    for (int item = i0; item < nitems; item += stride) {
        cp_async_wait_n<0>();
        __syncthreads();
        // real lines 2l and 2l+1 become the real and imaginary part of line l
        for (int t = threadIdx.x; t < L * n; t += blockDim.x) {
            const int l = t / n, e = t - l * n;
            A[e * ls + l] = make_float2(S[(2 * l) * n + e], S[(2 * l + 1) * n + e]);
        }
        __syncthreads();
        if (item + stride < nitems) load(item + stride);
        float2 *Rz = A;
        if constexpr (IP) fft_ip<N, L, kThreads, L + 1>(A, p.tw, -1.f);
        else Rz = Fft<N>::template run<L>(A, B, p, ls, -1.f);
        const long long line0 = (long long)item * 2 * L;
        for (int t = threadIdx.x; t < L * h3; t += blockDim.x) {
            const int l = t / h3, k = t - l * h3;
            const float2 z = Rz[k * ls + l];
            const float2 zn = Rz[((k == 0) ? 0 : (n - k)) * ls + l];
            const float2 a = make_float2(0.5f * (z.x + zn.x), 0.5f * (z.y - zn.y));
            const float2 b = make_float2(0.5f * (z.y + zn.y), -0.5f * (z.x - zn.x));
            const long long la = line0 + 2 * l;
            if (la < nlines) out[la * p3 + k] = a;
            if (la + 1 < nlines) out[(la + 1) * p3 + k] = b;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- pass 2 ---
// x2 complex transform in place.  Persistent blocks walk the tiles (TK k3
// columns of one (c, i1) plane) and double-buffer them: cp.async fetches the
// next tile while the current one is transformed (measured at 256^3: the x2
// passes of a solve 3.09 -> 2.44 ms against one tile per block).
template <int N, int TK>
__global__ void __launch_bounds__(kThreads)
k_c2c_x2(float2 *__restrict__ data, FftPlan p, int h3, int p3, float s, int ntk, int nitems) {
    extern __shared__ float2 sm[];
    const int n = Fft<N>::size(p);
    float2 *A0 = sm, *A1 = sm + n * TK, *B = sm + 2 * n * TK;
    auto load = [&](int item, float2 *dst) {
        const int plane = item / ntk, k0 = (item - plane * ntk) * TK;
        const float2 *base = data + (long long)plane * n * p3 + k0;
        for (int t = threadIdx.x; t < n * (TK / 2); t += blockDim.x) {
            const int e = t / (TK / 2), ch = t - e * (TK / 2);
            const int col = k0 + 2 * ch;
            const int bytes = col + 2 <= h3 ? 16 : (col < h3 ? 8 : 0);
            const float2 *src = base + (long long)e * p3 + (bytes ? 2 * ch : 0);
            cp_async16z(dst + e * TK + 2 * ch, src, bytes);
        }
        cp_async_commit_all();
    };
    const int i0 = blockIdx.x, stride = gridDim.x;
    if (i0 >= nitems) return;
    load(i0, A0);
    bool cur0 = true;
    for (int item = i0; item < nitems; item += stride) {
        float2 *Acur = cur0 ? A0 : A1, *Anext = cur0 ? A1 : A0;
        if (item + stride < nitems) {
            load(item + stride, Anext);
            cp_async_wait_n<1>();
        } else {
            cp_async_wait_n<0>();
        }
        __syncthreads();
        float2 *R = Fft<N>::template run<TK>(Acur, B, p, TK, s);
        const int plane = item / ntk, k0 = (item - plane * ntk) * TK;
        float2 *base = data + (long long)plane * n * p3 + k0;
        for (int t = threadIdx.x; t < n * TK; t += blockDim.x) {
            const int e = t / TK, l = t - e * TK;
            if (k0 + l < h3) base[(long long)e * p3 + l] = R[e * TK + l];
        }
        __syncthreads();
        cur0 = !cur0;
    }
}

// Pass 2 for lengths with an in-place compile-time plan (stage_ip): the
// transform needs no scratch tile, so a block holds only the current and the
// next tile (three blocks per SM at n2 = 256), and stores two columns
// (16 bytes) at a time.
template <int N, int TK, int MT, int MINB>
__global__ void __launch_bounds__(MT, MINB)
k_c2c_x2_ip(float2 *__restrict__ data, FftPlan p, int h3, int p3, float s, int ntk, int nitems) {
    extern __shared__ float2 sm[];
    constexpr int CH = TK / 2;  // 16-byte chunks per row
    float2 *cur = sm, *nxt = sm + N * TK;
    const float2 *__restrict__ tw = p.tw;
    auto load = [&](int item, float2 *dst) {
        const int plane = item / ntk, k0 = (item - plane * ntk) * TK;
        const float2 *base = data + (long long)plane * N * p3 + k0;
        for (int t = threadIdx.x; t < N * CH; t += MT) {
            const int e = t / CH, ch = t - e * CH;
            const int col = k0 + 2 * ch;
            const int bytes = col + 2 <= h3 ? 16 : (col < h3 ? 8 : 0);
            cp_async16z(dst + e * TK + 2 * ch, base + (long long)e * p3 + (bytes ? 2 * ch : 0), bytes);
        }
        cp_async_commit_all();
    };
    const int i0 = blockIdx.x, stride = gridDim.x;
    if (i0 >= nitems) return;
    load(i0, cur);
    for (int item = i0; item < nitems; item += stride) {
        if (item + stride < nitems) {
            load(item + stride, nxt);
            cp_async_wait_n<1>();
        } else {
            cp_async_wait_n<0>();
        }
        __syncthreads();
        fft_ip<N, TK, MT>(cur, tw, s);
        const int plane = item / ntk, k0 = (item - plane * ntk) * TK;
        float2 *base = data + (long long)plane * N * p3 + k0;
        for (int t = threadIdx.x; t < N * CH; t += MT) {
            const int e = t / CH, ch = t - e * CH;
            const int col = k0 + 2 * ch;
            // one 16-byte shared load per two columns (two 8-byte loads at a
            // 16-byte lane stride would conflict in pairs of banks)
            const float4 q = *reinterpret_cast<const float4 *>(cur + e * TK + 2 * ch);
            float2 *g = base + (long long)e * p3 + 2 * ch;
            if (col + 2 <= h3) *reinterpret_cast<float4 *>(g) = q;
            else if (col < h3) *g = make_float2(q.x, q.y);
        }
        __syncthreads();
        float2 *t = cur;
        cur = nxt;
        nxt = t;
    }
}

// ---------------------------------------------------------------- pass 3 ---
// x1 forward, multiplier, x1 inverse, in place; all three components at once
// (the divergence penalty couples them).  Persistent blocks walk the items
// (TK k3 columns at one k2 index); the three component tiles of the next item
// are fetched by 16-byte cp.async (zero-filled past h3) while the current
// item is transformed, multiplied and transformed back.  Seven tiles of n1*TK:
// three current, three next, one scratch.
template <int N, int TK, int OP>
__global__ void __launch_bounds__(kThreads)
k_mul_x1(float2 *__restrict__ data, FftPlan p1, int n2, int n3, int h3, int p3, long long cstride, SpecParams sp,
           int ntk, int nitems) {
    constexpr bool FWD = OP != OP_X1INV, INV = OP != OP_X1FWD;
    extern __shared__ float2 sm[];
    const int n1 = Fft<N>::size(p1);
    const int tile = n1 * TK;
    float2 *cur[3] = {sm, sm + tile, sm + 2 * tile};
    float2 *scratch = sm + 3 * tile;
    float2 *nxt[3] = {sm + 4 * tile, sm + 5 * tile, sm + 6 * tile};
    const long long rowstride = (long long)n2 * p3;  // between consecutive i1
    constexpr int CH = TK / 2;                        // 16-byte chunks per row
    auto load = [&](int item, float2 *const *dst) {
        const int i2 = item / ntk, k0 = (item - i2 * ntk) * TK;
        const float2 *base = data + (long long)i2 * p3 + k0;
        for (int t = threadIdx.x; t < 3 * n1 * CH; t += blockDim.x) {
            const int c = t / (n1 * CH), r = t - c * n1 * CH;
            const int e = r / CH, ch = r - e * CH;
            const int col = k0 + 2 * ch;
            const int bytes = col + 2 <= h3 ? 16 : (col < h3 ? 8 : 0);
            cp_async16z(dst[c] + e * TK + 2 * ch, base + c * cstride + e * rowstride + (bytes ? 2 * ch : 0), bytes);
        }
        cp_async_commit_all();
    };
    const int i0 = blockIdx.x, stride = gridDim.x;
    if (i0 >= nitems) return;
    load(i0, cur);
    for (int item = i0; item < nitems; item += stride) {
        if (item + stride < nitems) {
            load(item + stride, nxt);
            cp_async_wait_n<1>();
        } else {
            cp_async_wait_n<0>();
        }
        __syncthreads();
        if (FWD) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float2 *r = Fft<N>::template run<TK>(cur[c], scratch, p1, TK, -1.f);
                if (r != cur[c]) { scratch = cur[c]; cur[c] = r; }
            }
        }
        const int i2 = item / ntk, k0 = (item - i2 * ntk) * TK;
        // multiplier at (k1, k2, k3)
        const float k2 = wavenumber(i2, n2), k2d = wavenumber_d1(i2, n2);
        for (int t = threadIdx.x; t < tile; t += blockDim.x) {
            const int e = t / TK, l = t - e * TK;
            const int i3 = k0 + l;
            const float k1 = wavenumber(e, n1), k1d = wavenumber_d1(e, n1);
            const float k3 = (float)i3, k3d = ((n3 & 1) == 0 && 2 * i3 == n3) ? 0.f : k3;
            const int id = e * TK + l;
            mul_point<OP>(cur[0][id], cur[1][id], cur[2][id], k1, k1d, k2, k2d, k3, k3d, sp);
        }
        __syncthreads();
        if (INV) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float2 *r = Fft<N>::template run<TK>(cur[c], scratch, p1, TK, +1.f);
                if (r != cur[c]) { scratch = cur[c]; cur[c] = r; }
            }
        }
        float2 *base = data + (long long)i2 * p3 + k0;
        for (int c = 0; c < 3; ++c) {
            for (int t = threadIdx.x; t < tile; t += blockDim.x) {
                const int e = t / TK, l = t - e * TK;
                if (k0 + l < h3) base[c * cstride + e * rowstride + l] = cur[c][e * TK + l];
            }
        }
        __syncthreads();
        // the next item's tiles become the current ones; the current tiles
        // (and the scratch the transforms left) are free again
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 *t = cur[c];
            cur[c] = nxt[c];
            nxt[c] = t;
        }
    }
}

// The same pass for lengths with a compile-time plan.  The three component
// tiles of an item are interleaved line by line -- 3 TK lines of n1 elements,
// buf[e * 3TK + c * TK + l] -- and transformed together, in place, by MT
// threads (stage_ip): one barrier pair per radix stage serves all three
// components, every thread holds a butterfly in every stage (at n1 = 256,
// TK = 8: 16 x 24 = 384 radix-16 butterflies for 384 threads), and no
// scratch tile is needed.  Six tiles of n1*TK: current and next item.
template <int N, int TK, int OP, int MT, int MINB>
__global__ void __launch_bounds__(MT, MINB)
k_mul_x1_ip(float2 *__restrict__ data, FftPlan p1, int n2, int n3, int h3, int p3, long long cstride,
            SpecParams sp, int ntk, int nitems) {
    constexpr bool FWD = OP != OP_X1INV, INV = OP != OP_X1FWD;
    constexpr int LL = 3 * TK, TILE = N * LL, CH = TK / 2;  // CH: 16-byte chunks per row and component
    extern __shared__ float2 sm[];
    float2 *cur = sm, *nxt = sm + TILE;
    const long long rowstride = (long long)n2 * p3;  // between consecutive i1
    const float2 *__restrict__ tw = p1.tw;
    auto load = [&](int item, float2 *dst) {
        const int i2 = item / ntk, k0 = (item - i2 * ntk) * TK;
        const float2 *base = data + (long long)i2 * p3 + k0;
        for (int t = threadIdx.x; t < 3 * N * CH; t += MT) {
            const int c = t / (N * CH), r = t - c * (N * CH);
            const int e = r / CH, ch = r - e * CH;
            const int col = k0 + 2 * ch;
            const int bytes = col + 2 <= h3 ? 16 : (col < h3 ? 8 : 0);
            cp_async16z(dst + e * LL + c * TK + 2 * ch, base + c * cstride + e * rowstride + (bytes ? 2 * ch : 0),
                        bytes);
        }
        cp_async_commit_all();
    };
    const int i0 = blockIdx.x, stride = gridDim.x;
    if (i0 >= nitems) return;
    load(i0, cur);
    for (int item = i0; item < nitems; item += stride) {
        if (item + stride < nitems) {
            load(item + stride, nxt);
            cp_async_wait_n<1>();
        } else {
            cp_async_wait_n<0>();
        }
        __syncthreads();
        if (FWD) fft_ip<N, LL, MT>(cur, tw, -1.f);
        const int i2 = item / ntk, k0 = (item - i2 * ntk) * TK;
        const float k2 = wavenumber(i2, n2), k2d = wavenumber_d1(i2, n2);
        for (int t = threadIdx.x; t < N * TK; t += MT) {
            const int e = t / TK, l = t - e * TK;
            const int i3 = k0 + l;
            const float k1 = wavenumber(e, N), k1d = wavenumber_d1(e, N);
            const float k3 = (float)i3, k3d = ((n3 & 1) == 0 && 2 * i3 == n3) ? 0.f : k3;
            float2 *q = cur + e * LL + l;
            mul_point<OP>(q[0], q[TK], q[2 * TK], k1, k1d, k2, k2d, k3, k3d, sp);
        }
        __syncthreads();
        if (INV) fft_ip<N, LL, MT>(cur, tw, +1.f);
        // back to global memory, two columns (16 bytes) per store
        float2 *base = data + (long long)i2 * p3 + k0;
        for (int t = threadIdx.x; t < 3 * N * CH; t += MT) {
            const int c = t / (N * CH), r = t - c * (N * CH);
            const int e = r / CH, ch = r - e * CH;
            const int col = k0 + 2 * ch;
            const float4 q = *reinterpret_cast<const float4 *>(cur + e * LL + c * TK + 2 * ch);
            float2 *g = base + c * cstride + e * rowstride + 2 * ch;
            if (col + 2 <= h3) *reinterpret_cast<float4 *>(g) = q;
            else if (col < h3) *g = make_float2(q.x, q.y);
        }
        __syncthreads();
        float2 *t = cur;
        cur = nxt;
        nxt = t;
    }
}

// ---------------------------------------------------------------- pass 5 ---
// x3 inverse half spectrum -> real, two real lines per complex transform.
template <int N, int L, int EPI, typename TO = float>
__global__ void __launch_bounds__(kThreads)
k_c2r_x3(const float2 *__restrict__ in, TO *__restrict__ out, const float *__restrict__ add,
         long long nlines, FftPlan p, int h3, int p3) {
    extern __shared__ float2 sm[];
    const int n = Fft<N>::size(p), ls = L + 1;
    float2 *A = sm, *B = sm + n * ls;
    const long long line0 = (long long)blockIdx.x * 2 * L;
    const bool even = (n & 1) == 0;
#pragma unroll
    for (int t = threadIdx.x; t < L * n; t += kThreads) {
        const int l = t / n, k = t - l * n;
        const long long la = line0 + 2 * l;
        const bool lo = k < h3;
        const int kk = lo ? k : n - k;
        float2 a = la < nlines ? in[la * p3 + kk] : make_float2(0.f, 0.f);
        float2 b = la + 1 < nlines ? in[(la + 1) * p3 + kk] : make_float2(0.f, 0.f);
        if (k == 0 || (even && 2 * k == n)) {
            a.y = 0.f;
            b.y = 0.f;
        }
        if (!lo) {
            a.y = -a.y;
            b.y = -b.y;
        }
        // Z = A + i B
        A[k * ls + l] = make_float2(a.x - b.y, a.y + b.x);
    }
    __syncthreads();
    float2 *R = Fft<N>::template run<L>(A, B, p, ls, +1.f);
    for (int t = threadIdx.x; t < L * n; t += blockDim.x) {
        const int l = t / n, e = t - l * n;
        const long long la = line0 + 2 * l;
        const float2 z = R[e * ls + l];
        if (la < nlines) {
            float val = z.x;
            if (EPI == EPI_ADD) val += add[la * n + e];
            str(out + la * n + e, val);
        }
        if (la + 1 < nlines) {
            float val = z.y;
            if (EPI == EPI_ADD) val += add[(la + 1) * n + e];
            str(out + (la + 1) * n + e, val);
        }
    }
}

// Pass 5 with persistent blocks: the 2L half-spectrum lines of the next tile
// (one contiguous chunk of 2L*p3 complex values) are fetched by 16-byte
// cp.async into a staging buffer while the current tile is transformed.
template <int N, int L, int EPI, typename TO = float>
__global__ void __launch_bounds__(kThreads, fft_in_place(N) ? 3 : 1)
k_c2r_x3_p(const float2 *__restrict__ in, TO *__restrict__ out, const float *__restrict__ add, long long nlines,
           FftPlan p, int h3, int p3, int nitems) {
    extern __shared__ float2 sm[];
    constexpr bool IP = fft_in_place(N);  // in-place transform: no scratch tile
    const int n = Fft<N>::size(p), ls = L + 1;
    float2 *A = sm, *B = sm + n * ls;
    float2 *S = sm + (IP ? 1 : 2) * n * ls;  // staging: 2L lines of p3 complex values
    const bool even = (n & 1) == 0;
    if (N > 0) h3 = N / 2 + 1;
    auto load = [&](int item) {
        const long long line0 = (long long)item * 2 * L;
        const float2 *base = in + line0 * p3;
        const int nch = L * p3;  // 2L * p3 complex values, two per chunk
        for (int t = threadIdx.x; t < nch; t += blockDim.x) {
            const long long line = line0 + (2 * t) / p3;
            const int bytes = line < nlines ? 16 : 0;
            cp_async16z(S + 2 * t, base + (bytes ? 2 * t : 0), bytes);
        }
        cp_async_commit_all();
    };
    const int i0 = blockIdx.x, stride = gridDim.x;
    if (i0 >= nitems) return;
    load(i0);
    for (int item = i0; item < nitems; item += stride) {
        cp_async_wait_n<0>();
        __syncthreads();
        // each stored coefficient k < h3 gives Z_k = A_k + i B_k and, by
        // Hermitian symmetry, Z_{n-k} = conj(A_k) + i conj(B_k): one read of
        // the staged lines for both
        for (int t = threadIdx.x; t < L * h3; t += blockDim.x) {
            const int l = t / h3, k = t - l * h3;
            float2 a = S[(2 * l) * p3 + k];
            float2 b = S[(2 * l + 1) * p3 + k];
            const bool self = k == 0 || (even && 2 * k == n);
            if (self) {
                a.y = 0.f;
                b.y = 0.f;
            }
            A[k * ls + l] = make_float2(a.x - b.y, a.y + b.x);
            if (!self) A[(n - k) * ls + l] = make_float2(a.x + b.y, -a.y + b.x);
        }
        __syncthreads();
        if (item + stride < nitems) load(item + stride);
        float2 *R = A;
        if constexpr (IP) fft_ip<N, L, kThreads, L + 1>(A, p.tw, +1.f);
        else R = Fft<N>::template run<L>(A, B, p, ls, +1.f);
        const long long line0 = (long long)item * 2 * L;
        for (int t = threadIdx.x; t < L * n; t += blockDim.x) {
            const int l = t / n, e = t - l * n;
            const long long la = line0 + 2 * l;
            const float2 z = R[e * ls + l];
            if (la < nlines) {
                float val = z.x;
                if (EPI == EPI_ADD) val += add[la * n + e];
                str(out + la * n + e, val);
            }
            if (la + 1 < nlines) {
                float val = z.y;
                if (EPI == EPI_ADD) val += add[(la + 1) * n + e];
                str(out + (la + 1) * n + e, val);
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------- register-resident passes ----
// The same five passes for the lengths N = 16 G (fft_reg.cuh): one tile per
// block, read from and written to global memory by the register steps
// themselves, so a pass has one exchange through shared memory per transform
// (x1 with the multiplier: two for both transforms where G divides 16) and
// three blocks per SM hide one another's loads.  The staged, double-buffered
// forms they replace at these lengths were bound by shared-memory round trips,
// barriers and issue.  Per pass over three components, before and after:
//   256^3 (59 us at the copy rate)  x3 forward 90 -> 66 us, x2 81 -> 70,
//         x1 with multiplier 145 -> 121, x3 inverse 117 -> 78 (mean of
//         calls without and with an addend, which is another 30 us of bytes)
//   192^3 (25 us)  50 -> 36, 61 -> 32, 93 -> 54, 64 -> 40
//   128^3 (7.5 us, and about 5 us of launch)  19 -> 15, 16.5 -> 12, 26 -> 19, 21 -> 13
// The x3 and x2 passes are within 0.84-0.88 of the copy rate at 256^3 inside a solve; the x1
// pass is bound by its registers (96 data values a thread, 12 warps per SM).

// x2 transform (S = 0: direction s) and the x1 transform without a multiplier
// (S = -1 forward, S = +1 inverse of the elements times `scale`), in place
template <int N, int S>
__global__ void __launch_bounds__(RegTile<N>::T, 768 / RegTile<N>::T)
kr_c2c(float2 *__restrict__ data, const float2 *__restrict__ tw, RegLines q, float s, float scale) {
    using P = RegPlan<N>;
    constexpr int TL = RegTile<N>::TL, T = RegTile<N>::T, G = P::G;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    reg_twiddles<N, T>(w, tw);
    const int l = threadIdx.x % TL, j = threadIdx.x / TL;
    long long off;
    int col;
    const bool ok = reg_line(q, blockIdx.x * TL + l, off, col);
    float2 *base = data + off + col;
    if (P::P2 || j < G) {
        float2 a[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) a[r] = ok ? base[(j + G * r) * q.estride] : make_float2(0.f, 0.f);
        if (S > 0) {
#pragma unroll
            for (int r = 0; r < 16; ++r) a[r] = make_float2(__fmul_rn(a[r].x, scale), __fmul_rn(a[r].y, scale));
        }
        dft<16>(a, S == 0 ? s : (float)S);
#pragma unroll
        for (int r = 0; r < 16; ++r) sm[(17 * j + r) * TL + l] = a[r];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16 / P::TPL; ++i) {
        const int k = j + P::TPL * i;
        float2 a[G];
#pragma unroll
        for (int m = 0; m < G; ++m) a[m] = sm[(k + 17 * m) * TL + l];
        reg_step2<N, S>(a, k, w, s);
        if (ok) {
#pragma unroll
            for (int m = 0; m < G; ++m) base[(k + 16 * m) * q.estride] = a[m];
        }
    }
}

// x3 forward, two real lines as one complex line; Z_{n-k} of the Hermitian
// split comes from the lane that holds it
template <int N>
__global__ void __launch_bounds__(RegTile<N>::T, 768 / RegTile<N>::T)
kr_r2c(const float *__restrict__ in, float2 *__restrict__ out, const float2 *__restrict__ tw, long long nlines,
       int p3) {
    using P = RegPlan<N>;
    constexpr int TL = RegTile<N>::TL, T = RegTile<N>::T, G = P::G;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    reg_twiddles<N, T>(w, tw);
    if (threadIdx.x < G * TL) {
        const int j = threadIdx.x % G, l = threadIdx.x / G;
        const long long la = 2 * ((long long)blockIdx.x * TL + l);
        const float *pa = in + la * N + j;
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
        float2 a[16];
#pragma unroll
        for (int r = 0; r < 16; ++r)
            a[r] = make_float2(ok0 ? __ldg(pa + G * r) : 0.f, ok1 ? __ldg(pa + N + G * r) : 0.f);
        dft<16>(a, -1.f);
#pragma unroll
        for (int r = 0; r < 16; ++r) sm[l * P::ROWS + 17 * j + r] = a[r];
    }
    __syncthreads();
    const int k = threadIdx.x % 16;
    const int src = ((threadIdx.x & 31) & 16) | ((16 - k) & 15);  // lane of index n - k
#pragma unroll
    for (int i = 0; i < 16 / P::TPL; ++i) {
        const int l = threadIdx.x / 16 + i * (T / 16);
        float2 a[G];
#pragma unroll
        for (int m = 0; m < G; ++m) a[m] = sm[l * P::ROWS + k + 17 * m];
        reg_step2<N, -1>(a, k, w);
        const long long la = 2 * ((long long)blockIdx.x * TL + l);
        float2 *oa = out + la * p3 + k;
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
#pragma unroll
        for (int m = 0; m <= G / 2; ++m) {
            // element k + 16 m (m = G / 2: only k = 0) and its mirror
            const float2 z = a[m];
            float2 zn;
            zn.x = __shfl_sync(0xffffffffu, a[G - 1 - m].x, src);
            zn.y = __shfl_sync(0xffffffffu, a[G - 1 - m].y, src);
            if (k == 0) zn = a[(G - m) % G];
            const float2 fa = make_float2(0.5f * (z.x + zn.x), 0.5f * (z.y - zn.y));
            const float2 fb = make_float2(0.5f * (z.y + zn.y), -0.5f * (z.x - zn.x));
            if (m < G / 2 || k == 0) {
                if (ok0) oa[16 * m] = fa;
                if (ok1) oa[p3 + 16 * m] = fb;
            }
        }
    }
}

// x3 inverse; every stored coefficient k gives Z_k = A_k + i B_k and its mirror
template <int N, int EPI>
__global__ void __launch_bounds__(RegTile<N>::T, 768 / RegTile<N>::T)
kr_c2r(const float2 *__restrict__ in, float *out, const float *add, const float2 *__restrict__ tw, long long nlines,
       int p3) {
    using P = RegPlan<N>;
    constexpr int TL = RegTile<N>::TL, T = RegTile<N>::T, G = P::G;
    __shared__ float2 w[P::W];
    __shared__ float2 sm[P::ROWS * TL];
    reg_twiddles<N, T>(w, tw);
    if (threadIdx.x < G * TL) {
        const int j = threadIdx.x % G, l = threadIdx.x / G;
        const long long la = 2 * ((long long)blockIdx.x * TL + l);
        const float2 *pa = in + la * p3;
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
        const float2 zero = make_float2(0.f, 0.f);
        float2 a[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int e = j + G * r;
            const bool lo = r < 8 || (r == 8 && j == 0);  // e <= N / 2
            const int k = lo ? e : N - e;
            float2 fa = ok0 ? __ldg(pa + k) : zero, fb = ok1 ? __ldg(pa + p3 + k) : zero;
            if ((r == 0 || r == 8) && j == 0) {
                fa.y = 0.f;
                fb.y = 0.f;
            }
            a[r] = lo ? make_float2(fa.x - fb.y, fa.y + fb.x) : make_float2(fa.x + fb.y, -fa.y + fb.x);
        }
        dft<16>(a, 1.f);
#pragma unroll
        for (int r = 0; r < 16; ++r) sm[l * P::ROWS + 17 * j + r] = a[r];
    }
    __syncthreads();
    const int k = threadIdx.x % 16;
#pragma unroll
    for (int i = 0; i < 16 / P::TPL; ++i) {
        const int l = threadIdx.x / 16 + i * (T / 16);
        const long long la = 2 * ((long long)blockIdx.x * TL + l);
        const bool ok0 = la < nlines, ok1 = la + 1 < nlines;
        float2 a[G], g[G];
#pragma unroll
        for (int m = 0; m < G; ++m) a[m] = sm[l * P::ROWS + k + 17 * m];
        if (EPI == EPI_ADD) {
#pragma unroll
            for (int m = 0; m < G; ++m)
                g[m] = make_float2(ok0 ? add[la * N + k + 16 * m] : 0.f, ok1 ? add[(la + 1) * N + k + 16 * m] : 0.f);
        }
        reg_step2<N, 1>(a, k, w);
#pragma unroll
        for (int m = 0; m < G; ++m) {
            if (ok0) out[la * N + k + 16 * m] = EPI == EPI_ADD ? a[m].x + g[m].x : a[m].x;
            if (ok1) out[(la + 1) * N + k + 16 * m] = EPI == EPI_ADD ? a[m].y + g[m].y : a[m].y;
        }
    }
}

// x1 forward, multiplier, x1 inverse, in place.  A thread holds the same
// elements of all three components, so the coupled multiplier needs no
// exchange of its own.
template <int N>
struct RegMul {
    static constexpr int TL = N == 32 ? 16 : 8;
    static constexpr int T = RegPlan<N>::TPL * TL;
    // resident threads per SM that the registers are cut for: 168 registers
    // (384) at 256 and the composite lengths, 255 (256) where the smaller
    // blocks spill more than the third block hides (x1 pass at 128^3 22.3 ->
    // 19.2 us, at 256^3 121 against 124)
    static constexpr int PER_SM = N == 256 || !RegPlan<N>::P2 ? 384 : 256;
    static constexpr size_t smem = (size_t)(3 * RegPlan<N>::ROWS * TL + RegPlan<N>::W) * sizeof(float2);
};
template <int N, int OP>
__global__ void __launch_bounds__(RegMul<N>::T, RegMul<N>::PER_SM / RegMul<N>::T)
kr_mul(float2 *__restrict__ data, const float2 *__restrict__ tw, RegLines q, int n2, int n3, SpecParams sp) {
    using P = RegPlan<N>;
    constexpr int TL = RegMul<N>::TL, T = RegMul<N>::T, G = P::G, CS = P::ROWS * TL;
    extern __shared__ float2 sm[];
    float2 *w = sm + 3 * CS;
    reg_twiddles<N, T>(w, tw);
    const int l = threadIdx.x % TL, j = threadIdx.x / TL;
    long long off;
    int col;
    const int line = blockIdx.x * TL + l, i2 = line / q.ncol;
    const bool ok = reg_line(q, line, off, col);
    float2 *base = data + off + col;
    const bool act = P::P2 || j < G;
    float2 a[3][16];
    if (act) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int r = 0; r < 16; ++r)
                a[c][r] = ok ? base[c * q.cstride + (j + G * r) * q.estride] : make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dft<16>(a[c], -1.f);
#pragma unroll
            for (int r = 0; r < 16; ++r) sm[c * CS + (17 * j + r) * TL + l] = a[c][r];
        }
    }
    __syncthreads();
    const float k2 = wavenumber(i2, n2), k2d = wavenumber_d1(i2, n2);
    const float k3 = (float)col, k3d = ((n3 & 1) == 0 && 2 * col == n3) ? 0.f : k3;
    auto mul = [&](int e, float2 &x, float2 &y, float2 &z) {
        const float k1 = wavenumber(e, N), k1d = wavenumber_d1(e, N);
        mul_point<OP>(x, y, z, k1, k1d, k2, k2d, k3, k3d, sp);
    };
    if constexpr (P::P2) {
        constexpr int I = 16 / G;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int i = 0; i < I; ++i) {
                float2 b[G];
#pragma unroll
                for (int m = 0; m < G; ++m) b[m] = sm[c * CS + (j + G * i + 17 * m) * TL + l];
                reg_step2<N, -1>(b, j + G * i, w);
#pragma unroll
                for (int m = 0; m < G; ++m) a[c][i + I * m] = b[m];
            }
#pragma unroll
        for (int r = 0; r < 16; ++r) mul(j + G * r, a[0][r], a[1][r], a[2][r]);
    } else {
        float2 b[3][G];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int m = 0; m < G; ++m) b[c][m] = sm[c * CS + (j + 17 * m) * TL + l];
            reg_step2<N, -1>(b[c], j, w);
        }
#pragma unroll
        for (int m = 0; m < G; ++m) mul(j + 16 * m, b[0][m], b[1][m], b[2][m]);
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int m = 0; m < G; ++m) sm[c * CS + (j + 17 * m) * TL + l] = b[c][m];
        __syncthreads();
        if (act) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    const int e = j + G * r;
                    a[c][r] = sm[c * CS + (e + e / 16) * TL + l];
                }
        }
    }
    if (act) {
#pragma unroll
        for (int c = 0; c < 3; ++c) dft<16>(a[c], 1.f);
    }
    __syncthreads();  // the forward results are read
    if (act) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int r = 0; r < 16; ++r) sm[c * CS + (17 * j + r) * TL + l] = a[c][r];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int i = 0; i < 16 / P::TPL; ++i) {
            const int k = j + P::TPL * i;
            float2 b[G];
#pragma unroll
            for (int m = 0; m < G; ++m) b[m] = sm[c * CS + (k + 17 * m) * TL + l];
            reg_step2<N, 1>(b, k, w);
            if (ok) {
#pragma unroll
                for (int m = 0; m < G; ++m) base[c * q.cstride + (k + 16 * m) * q.estride] = b[m];
            }
        }
}

// ------------------------------------------------ whole-plane passes -------
// x3 and x2 transforms of a square plane (n2 = n3 = N) in one launch, a plane
// per block, for planes that fit shared memory beside their exchange buffer.
// On grids this small a pass is a launch and one tile per block, so three
// launches instead of five count: (beta A)^-1 at 32^3 24.7 -> 16.5 us a call, at
// 64^3 24.9 -> 20.5, at 96^3 42.5 -> 32.2, at 128x96x96 49 -> 41.  At 128 a plane
// would leave one block per SM.  The steps are those of kr_r2c, kr_c2c and
// kr_c2r, bit for bit.
template <int N>
struct PlanePlan {
    using P = RegPlan<N>;
    static constexpr int H = N / 2 + 1, T = N <= 32 ? 128 : 256;
    static constexpr int PAIR = N / 2 * P::ROWS, COLS = P::ROWS * H;   // exchange: line pairs, columns
    static constexpr int X = PAIR > COLS ? PAIR : COLS, S = N * H;     // and the half spectrum of the plane
    static constexpr size_t smem = (size_t)(X + S + P::W) * sizeof(float2);
};
__host__ __device__ constexpr bool plane_fft(int n) { return n == 32 || n == 64 || n == 96; }

template <int N>
__global__ void __launch_bounds__(PlanePlan<N>::T, 512 / PlanePlan<N>::T)
kr_plane_fwd(const float *__restrict__ in, float2 *__restrict__ out, const float2 *__restrict__ tw, int p3, float s) {
    using P = RegPlan<N>;
    using Q = PlanePlan<N>;
    constexpr int G = P::G, H = Q::H, T = Q::T;
    extern __shared__ float2 sm[];
    float2 *x = sm, *sp = sm + Q::X, *w = sp + Q::S;
    reg_twiddles<N, T>(w, tw);
    const float *pl = in + (long long)blockIdx.x * N * N;
    for (int i = threadIdx.x; i < N / 2 * G; i += T) {
        const int j = i % G, l = i / G;
        const float *pa = pl + 2 * l * N + j;
        float2 a[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) a[r] = make_float2(__ldg(pa + G * r), __ldg(pa + N + G * r));
        dft<16>(a, -1.f);
#pragma unroll
        for (int r = 0; r < 16; ++r) x[l * P::ROWS + 17 * j + r] = a[r];
    }
    __syncthreads();
    // N / 2 line pairs of sixteen threads: whole warps (the shuffles)
    static_assert(N / 2 * 16 % T == 0, "every thread takes part in every round");
    for (int i = threadIdx.x; i < N / 2 * 16; i += T) {
        const int k = i % 16, l = i / 16, src = (threadIdx.x & 16) | ((16 - k) & 15);
        float2 a[G];
#pragma unroll
        for (int m = 0; m < G; ++m) a[m] = x[l * P::ROWS + k + 17 * m];
        reg_step2<N, -1>(a, k, w);
        float2 *oa = sp + 2 * l * H + k;
#pragma unroll
        for (int m = 0; m <= G / 2; ++m) {
            const float2 z = a[m];
            float2 zn;
            zn.x = __shfl_sync(0xffffffffu, a[G - 1 - m].x, src);
            zn.y = __shfl_sync(0xffffffffu, a[G - 1 - m].y, src);
            if (k == 0) zn = a[(G - m) % G];
            const float2 fa = make_float2(0.5f * (z.x + zn.x), 0.5f * (z.y - zn.y));
            const float2 fb = make_float2(0.5f * (z.y + zn.y), -0.5f * (z.x - zn.x));
            if (m < G / 2 || k == 0) {
                oa[16 * m] = fa;
                oa[H + 16 * m] = fb;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < H * G; i += T) {
        const int col = i % H, j = i / H;
        float2 a[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) a[r] = sp[(j + G * r) * H + col];
        dft<16>(a, s);
#pragma unroll
        for (int r = 0; r < 16; ++r) x[(17 * j + r) * H + col] = a[r];
    }
    __syncthreads();
    float2 *po = out + (long long)blockIdx.x * N * p3;
    for (int i = threadIdx.x; i < H * 16; i += T) {
        const int col = i % H, k = i / H;
        float2 a[G];
#pragma unroll
        for (int m = 0; m < G; ++m) a[m] = x[(k + 17 * m) * H + col];
        reg_step2<N, 0>(a, k, w, s);
#pragma unroll
        for (int m = 0; m < G; ++m) po[(k + 16 * m) * p3 + col] = a[m];
    }
}

template <int N, int EPI>
__global__ void __launch_bounds__(PlanePlan<N>::T, 512 / PlanePlan<N>::T)
kr_plane_inv(const float2 *__restrict__ in, float *out, const float *add, const float2 *__restrict__ tw, int p3,
             float s) {
    using P = RegPlan<N>;
    using Q = PlanePlan<N>;
    constexpr int G = P::G, H = Q::H, T = Q::T;
    extern __shared__ float2 sm[];
    float2 *x = sm, *sp = sm + Q::X, *w = sp + Q::S;
    reg_twiddles<N, T>(w, tw);
    const float2 *pi = in + (long long)blockIdx.x * N * p3;
    for (int i = threadIdx.x; i < H * G; i += T) {
        const int col = i % H, j = i / H;
        float2 a[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) a[r] = __ldg(pi + (j + G * r) * p3 + col);
        dft<16>(a, s);
#pragma unroll
        for (int r = 0; r < 16; ++r) x[(17 * j + r) * H + col] = a[r];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < H * 16; i += T) {
        const int col = i % H, k = i / H;
        float2 a[G];
#pragma unroll
        for (int m = 0; m < G; ++m) a[m] = x[(k + 17 * m) * H + col];
        reg_step2<N, 0>(a, k, w, s);
#pragma unroll
        for (int m = 0; m < G; ++m) sp[(k + 16 * m) * H + col] = a[m];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < N / 2 * G; i += T) {
        const int j = i % G, l = i / G;
        const float2 *pa = sp + 2 * l * H;
        float2 a[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int e = j + G * r;
            const bool lo = r < 8 || (r == 8 && j == 0);  // e <= N / 2
            const int k = lo ? e : N - e;
            float2 fa = pa[k], fb = pa[H + k];
            if ((r == 0 || r == 8) && j == 0) {
                fa.y = 0.f;
                fb.y = 0.f;
            }
            a[r] = lo ? make_float2(fa.x - fb.y, fa.y + fb.x) : make_float2(fa.x + fb.y, -fa.y + fb.x);
        }
        dft<16>(a, 1.f);
#pragma unroll
        for (int r = 0; r < 16; ++r) x[l * P::ROWS + 17 * j + r] = a[r];
    }
    __syncthreads();
    const long long o = (long long)blockIdx.x * N * N;
    for (int i = threadIdx.x; i < N / 2 * 16; i += T) {
        const int k = i % 16, l = i / 16;
        float2 a[G];
#pragma unroll
        for (int m = 0; m < G; ++m) a[m] = x[l * P::ROWS + k + 17 * m];
        reg_step2<N, 1>(a, k, w);
#pragma unroll
        for (int m = 0; m < G; ++m) {
            const long long q = o + 2 * l * N + k + 16 * m;
            out[q] = EPI == EPI_ADD ? a[m].x + add[q] : a[m].x;
            out[q + N] = EPI == EPI_ADD ? a[m].y + add[q + N] : a[m].y;
        }
    }
}

// -------------------------------------------------------------- launchers --
}  // namespace

int persistent_grid(long long nitems, size_t smem) {
    static int sms[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    if (!sms[dev]) {
        int c = 0;
        if (cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || c <= 0) c = 152;
        sms[dev] = c;
    }
    long long per_sm = (long long)(227 * 1024) / (long long)(smem + 1024);
    if (per_sm < 1) per_sm = 1;
    if (per_sm > 8) per_sm = 8;
    const long long g = per_sm * sms[dev];
    return (int)(nitems < g ? nitems : g);
}

namespace {

template <int N, int L, typename TI>
void r2c_l(const Dims &d, const FftPlan &p, const TI *in, float2 *out, long long nlines,
           cudaStream_t st) {
    if constexpr (std::is_same<TI, float>::value) {
        if (d.n3 % 4 == 0 && ((uintptr_t)in & 15) == 0) {
            const size_t smem = (fft_in_place(N) ? 1 : 2) * (size_t)d.n3 * (L + 1) * sizeof(float2) +
                                (size_t)2 * L * d.n3 * sizeof(float);
            const int nitems = (int)((nlines + 2 * L - 1) / (2 * L));
            set_smem<k_r2c_x3_p<N, L>>(smem);
            k_r2c_x3_p<N, L><<<persistent_grid(nitems, smem), kThreads, smem, st>>>(in, out, nlines, p, d.h3, d.p3,
                                                                                    nitems);
            return;
        }
    }
    const size_t smem = 2 * (size_t)d.n3 * (L + 1) * sizeof(float2);
    const long long blocks = (nlines + 2 * L - 1) / (2 * L);
    set_smem<k_r2c_x3<N, L, TI>>(smem);
    k_r2c_x3<N, L, TI><<<(unsigned)blocks, kThreads, smem, st>>>(in, out, nlines, p, d.h3, d.p3);
}

template <int N, typename TI>
void r2c_n(const Dims &d, const FftPlan &p, const TI *in, float2 *out, int ncomp,
           cudaStream_t st) {
    const long long nlines = (long long)ncomp * d.n1 * d.n2;
    if constexpr (fft_reg(N)) {
        constexpr int TL = RegTile<N>::TL;
        kr_r2c<N><<<(unsigned)((nlines + 2 * TL - 1) / (2 * TL)), RegTile<N>::T, 0, st>>>(in, out, p.tw, nlines, d.p3);
    } else if constexpr (N > 0) {
        r2c_l<N, lines_x3(N)>(d, p, in, out, nlines, st);
    } else {
        switch (lines_x3(d.n3)) {
            case 16: r2c_l<N, 16>(d, p, in, out, nlines, st); break;
            case 8: r2c_l<N, 8>(d, p, in, out, nlines, st); break;
            default: r2c_l<N, 4>(d, p, in, out, nlines, st); break;
        }
    }
}

template <typename TI>
void r2c_x3(const Dims &d, const FftPlan &p, const TI *in, float2 *out, int ncomp,
            cudaStream_t st) {
    switch (d.n3) {
#define CASE_N(NN) case NN: r2c_n<NN>(d, p, in, out, ncomp, st); return;
        CLAIRE_CT_SIZES(CASE_N)
#undef CASE_N
        default: break;
    }
    if constexpr (std::is_same<TI, float>::value) {
        GenPass a{GenPass::R2C};
        a.tw = p.tw;
        a.in = in;
        a.spec = out;
        a.nlines = (long long)ncomp * d.n1 * d.n2;
        a.p3 = d.p3;
        if (gen_pass(d.n3, a, st)) return;
    }
    r2c_n<0>(d, p, in, out, ncomp, st);
}

template <int N, int TK>
void c2c_t(const Dims &d, const FftPlan &p, float2 *data, int ncomp, float s, cudaStream_t st) {
    const size_t smem = 3 * (size_t)d.n2 * TK * sizeof(float2);
    const int ntk = (d.h3 + TK - 1) / TK, nitems = ntk * ncomp * d.n1;
    const int grid = persistent_grid(nitems, smem);
    set_smem<k_c2c_x2<N, TK>>(smem);
    k_c2c_x2<N, TK><<<grid, kThreads, smem, st>>>(data, p, d.h3, d.p3, s, ntk, nitems);
}

template <int N, int TK>
void c2c_ip(const Dims &d, const FftPlan &p, float2 *data, int ncomp, float s, cudaStream_t st) {
    constexpr int MT = 256;
    constexpr size_t smem = 2 * (size_t)N * TK * sizeof(float2);
    constexpr int MINB = smem <= 72 * 1024 ? 3 : 2;
    const int ntk = (d.h3 + TK - 1) / TK, nitems = ntk * ncomp * d.n1;
    set_smem<k_c2c_x2_ip<N, TK, MT, MINB>>(smem);
    k_c2c_x2_ip<N, TK, MT, MINB><<<persistent_grid(nitems, smem), MT, smem, st>>>(data, p, d.h3, d.p3, s, ntk,
                                                                                  nitems);
}

// register-resident transform of the lines of a spectrum along x2 or x1
template <int N, int S>
void c2c_reg(const FftPlan &p, float2 *data, const RegLines &q, float s, float scale, cudaStream_t st) {
    constexpr int TL = RegTile<N>::TL;
    kr_c2c<N, S><<<(q.nlines + TL - 1) / TL, RegTile<N>::T, 0, st>>>(data, p.tw, q, s, scale);
}
inline RegLines lines_x2(const Dims &d, int ncomp) {
    return RegLines{d.p3, (long long)d.n2 * d.p3, (long long)d.n1 * d.n2 * d.p3, d.n1, d.p3, d.h3, ncomp * d.n1 * d.p3};
}
inline RegLines lines_x1(const Dims &d, int ncomp) {
    return RegLines{(long long)d.n2 * d.p3, d.p3, (long long)d.n1 * d.n2 * d.p3, d.n2, d.p3, d.h3, ncomp * d.n2 * d.p3};
}

template <int N>
void c2c_n(const Dims &d, const FftPlan &p, float2 *data, int ncomp, float s, cudaStream_t st) {
    if constexpr (fft_reg(N)) {
        c2c_reg<N, 0>(p, data, lines_x2(d, ncomp), s, 1.f, st);
    } else if constexpr (fft_in_place(N)) {
        c2c_ip<N, tile_cols(N, 1)>(d, p, data, ncomp, s, st);
    } else if constexpr (N > 0) {
        c2c_t<N, tile_cols(N, 2)>(d, p, data, ncomp, s, st);
    } else {
        switch (tile_cols(d.n2, 2)) {
            case 16: c2c_t<N, 16>(d, p, data, ncomp, s, st); break;
            case 8: c2c_t<N, 8>(d, p, data, ncomp, s, st); break;
            default: c2c_t<N, 4>(d, p, data, ncomp, s, st); break;
        }
    }
}

void c2c_x2(const Dims &d, const FftPlan &p, float2 *data, int ncomp, float s, cudaStream_t st) {
    switch (d.n2) {
#define CASE_N(NN) case NN: c2c_n<NN>(d, p, data, ncomp, s, st); return;
        CLAIRE_CT_SIZES(CASE_N)
#undef CASE_N
        default: break;
    }
    GenPass a{GenPass::C2C};
    a.tw = p.tw;
    a.spec = data;
    a.q = lines_x2(d, ncomp);
    a.s = s;
    if (!gen_pass(d.n2, a, st)) c2c_n<0>(d, p, data, ncomp, s, st);
}

template <int N, int TK, int OP>
void mul_t(const Dims &d, const FftPlan &p, float2 *data, const SpecParams &sp, cudaStream_t st) {
    const size_t smem = (size_t)7 * d.n1 * TK * sizeof(float2);
    const long long cstride = (long long)d.n1 * d.n2 * d.p3;
    const int ntk = (d.h3 + TK - 1) / TK, nitems = ntk * d.n2;
    set_smem<k_mul_x1<N, TK, OP>>(smem);
    k_mul_x1<N, TK, OP><<<persistent_grid(nitems, smem), kThreads, smem, st>>>(data, p, d.n2, d.n3, d.h3, d.p3,
                                                                                cstride, sp, ntk, nitems);
}

// compile-time plans: the interleaved in-place form, 384 threads, six tiles
template <int N, int TK, int OP>
void mul_ip(const Dims &d, const FftPlan &p, float2 *data, const SpecParams &sp, cudaStream_t st) {
    constexpr int MT = 384;
    constexpr size_t smem = (size_t)6 * N * TK * sizeof(float2);
    constexpr int MINB = smem <= 112 * 1024 ? 2 : 1;
    const long long cstride = (long long)d.n1 * d.n2 * d.p3;
    const int ntk = (d.h3 + TK - 1) / TK, nitems = ntk * d.n2;
    set_smem<k_mul_x1_ip<N, TK, OP, MT, MINB>>(smem);
    k_mul_x1_ip<N, TK, OP, MT, MINB><<<persistent_grid(nitems, smem), MT, smem, st>>>(data, p, d.n2, d.n3, d.h3,
                                                                                       d.p3, cstride, sp, ntk, nitems);
}

template <int N, int OP>
void mul_n(const Dims &d, const FftPlan &p, float2 *data, const SpecParams &sp, cudaStream_t st) {
    constexpr int NB = 6;  // three component tiles for the current item, three for the next
    if constexpr (fft_reg(N) && OP == OP_X1FWD) {
        c2c_reg<N, -1>(p, data, lines_x1(d, 3), -1.f, 1.f, st);
    } else if constexpr (fft_reg(N) && OP == OP_X1INV) {
        c2c_reg<N, 1>(p, data, lines_x1(d, 3), 1.f, sp.scale, st);
    } else if constexpr (fft_reg(N)) {
        constexpr int TL = RegMul<N>::TL;
        const RegLines q = lines_x1(d, 1);
        set_smem<kr_mul<N, OP>>(RegMul<N>::smem);
        kr_mul<N, OP><<<(q.nlines + TL - 1) / TL, RegMul<N>::T, RegMul<N>::smem, st>>>(data, p.tw, q, d.n2, d.n3, sp);
    } else if constexpr (fft_in_place(N)) {
        // six tiles in all (no scratch): the column count of five data tiles and one more
        mul_ip<N, tile_cols(N, NB - 1), OP>(d, p, data, sp, st);
    } else if constexpr (N > 0) {
        mul_t<N, tile_cols(N, NB), OP>(d, p, data, sp, st);
    } else {
        switch (tile_cols(d.n1, NB)) {
            case 16: mul_t<N, 16, OP>(d, p, data, sp, st); break;
            case 8: mul_t<N, 8, OP>(d, p, data, sp, st); break;
            default: mul_t<N, 4, OP>(d, p, data, sp, st); break;
        }
    }
}

template <int OP>
void mul_x1_op(const Dims &d, const FftPlan &p, float2 *data, const SpecParams &sp,
               cudaStream_t st) {
    switch (d.n1) {
#define CASE_N(NN) case NN: mul_n<NN, OP>(d, p, data, sp, st); return;
        CLAIRE_CT_SIZES(CASE_N)
#undef CASE_N
        default: break;
    }
    const bool both = OP == OP_A || OP == OP_AINV;
    GenPass a{both ? (OP == OP_A ? GenPass::MUL_A : GenPass::MUL_AINV) : GenPass::C2C};
    a.tw = p.tw;
    a.spec = data;
    a.q = lines_x1(d, both ? 1 : 3);
    a.n2 = d.n2;
    a.n3 = d.n3;
    a.sp = sp;
    a.s = OP == OP_X1INV ? 1.f : -1.f;
    a.scale = OP == OP_X1INV ? sp.scale : 1.f;
    if (!gen_pass(d.n1, a, st)) mul_n<0, OP>(d, p, data, sp, st);
}

template <int N, int L, typename TO>
void c2r_l(const Dims &d, const FftPlan &p, const float2 *in, TO *out, const float *add,
           long long nlines, cudaStream_t st) {
    if (((uintptr_t)in & 15) == 0) {
        // the persistent form with the next tile staged by cp.async
        const size_t smem = (fft_in_place(N) ? 1 : 2) * (size_t)d.n3 * (L + 1) * sizeof(float2) +
                            (size_t)2 * L * d.p3 * sizeof(float2);
        const int nitems = (int)((nlines + 2 * L - 1) / (2 * L));
        const int grid = persistent_grid(nitems, smem);
        if (add) {
            set_smem<k_c2r_x3_p<N, L, EPI_ADD, TO>>(smem);
            k_c2r_x3_p<N, L, EPI_ADD, TO><<<grid, kThreads, smem, st>>>(in, out, add, nlines, p, d.h3, d.p3, nitems);
        } else {
            set_smem<k_c2r_x3_p<N, L, EPI_STORE, TO>>(smem);
            k_c2r_x3_p<N, L, EPI_STORE, TO><<<grid, kThreads, smem, st>>>(in, out, add, nlines, p, d.h3, d.p3,
                                                                          nitems);
        }
        return;
    }
    const size_t smem = 2 * (size_t)d.n3 * (L + 1) * sizeof(float2);
    const long long blocks = (nlines + 2 * L - 1) / (2 * L);
    if (add) {
        set_smem<k_c2r_x3<N, L, EPI_ADD, TO>>(smem);
        k_c2r_x3<N, L, EPI_ADD, TO><<<(unsigned)blocks, kThreads, smem, st>>>(in, out, add, nlines, p,
                                                                              d.h3, d.p3);
    } else {
        set_smem<k_c2r_x3<N, L, EPI_STORE, TO>>(smem);
        k_c2r_x3<N, L, EPI_STORE, TO><<<(unsigned)blocks, kThreads, smem, st>>>(in, out, add, nlines,
                                                                                p, d.h3, d.p3);
    }
}

template <int N, typename TO>
void c2r_n(const Dims &d, const FftPlan &p, const float2 *in, TO *out, const float *add,
           int ncomp, cudaStream_t st) {
    const long long nlines = (long long)ncomp * d.n1 * d.n2;
    if constexpr (fft_reg(N)) {
        constexpr int TL = RegTile<N>::TL, T = RegTile<N>::T;
        const unsigned grid = (unsigned)((nlines + 2 * TL - 1) / (2 * TL));
        if (add) kr_c2r<N, EPI_ADD><<<grid, T, 0, st>>>(in, out, add, p.tw, nlines, d.p3);
        else kr_c2r<N, EPI_STORE><<<grid, T, 0, st>>>(in, out, add, p.tw, nlines, d.p3);
    } else if constexpr (N > 0) {
        c2r_l<N, lines_x3(N)>(d, p, in, out, add, nlines, st);
    } else {
        switch (lines_x3(d.n3)) {
            case 16: c2r_l<N, 16>(d, p, in, out, add, nlines, st); break;
            case 8: c2r_l<N, 8>(d, p, in, out, add, nlines, st); break;
            default: c2r_l<N, 4>(d, p, in, out, add, nlines, st); break;
        }
    }
}

template <typename TO>
void c2r_x3(const Dims &d, const FftPlan &p, const float2 *in, TO *out, const float *add,
            int ncomp, cudaStream_t st) {
    switch (d.n3) {
#define CASE_N(NN) case NN: c2r_n<NN>(d, p, in, out, add, ncomp, st); return;
        CLAIRE_CT_SIZES(CASE_N)
#undef CASE_N
        default: break;
    }
    if constexpr (std::is_same<TO, float>::value) {
        GenPass a{GenPass::C2R};
        a.tw = p.tw;
        a.spec = const_cast<float2 *>(in);
        a.out = out;
        a.add = add;
        a.nlines = (long long)ncomp * d.n1 * d.n2;
        a.p3 = d.p3;
        if (gen_pass(d.n3, a, st)) return;
    }
    c2r_n<0>(d, p, in, out, add, ncomp, st);
}

// the x3 and x2 transforms of ncomp components in one launch, where planes are
// square and of a length with a whole-plane pass (false: nothing launched)
template <int N>
void plane_fwd(const Dims &d, const FftPlan &p, const float *in, float2 *out, int ncomp, cudaStream_t st) {
    set_smem<kr_plane_fwd<N>>(PlanePlan<N>::smem);
    kr_plane_fwd<N><<<ncomp * d.n1, PlanePlan<N>::T, PlanePlan<N>::smem, st>>>(in, out, p.tw, d.p3, -1.f);
}
template <int N>
void plane_inv(const Dims &d, const FftPlan &p, const float2 *in, float *out, const float *add, int ncomp,
               cudaStream_t st) {
    if (add) {
        set_smem<kr_plane_inv<N, EPI_ADD>>(PlanePlan<N>::smem);
        kr_plane_inv<N, EPI_ADD><<<ncomp * d.n1, PlanePlan<N>::T, PlanePlan<N>::smem, st>>>(in, out, add, p.tw, d.p3, 1.f);
    } else {
        set_smem<kr_plane_inv<N, EPI_STORE>>(PlanePlan<N>::smem);
        kr_plane_inv<N, EPI_STORE><<<ncomp * d.n1, PlanePlan<N>::T, PlanePlan<N>::smem, st>>>(in, out, add, p.tw, d.p3,
                                                                                            1.f);
    }
}

// forward transform along x3 and x2 (real to half spectrum), and back
void forward_32(const Dims &d, const FftPlan *ax, const float *in, float2 *spec, int ncomp, cudaStream_t st,
                Profiler *prof) {
    const double R = 4.0 * d.N, C = 8.0 * d.n1 * d.n2 * d.h3;
    if (d.n2 == d.n3 && plane_fft(d.n3)) {
        ProfScope ps(prof, CLAIRE_K_FFT_R2C, st, ncomp * (R + C));
        switch (d.n3) {
            case 32: plane_fwd<32>(d, ax[2], in, spec, ncomp, st); return;
            case 64: plane_fwd<64>(d, ax[2], in, spec, ncomp, st); return;
            default: plane_fwd<96>(d, ax[2], in, spec, ncomp, st); return;
        }
    }
    {
        ProfScope ps(prof, CLAIRE_K_FFT_R2C, st, ncomp * (R + C));
        r2c_x3(d, ax[2], in, spec, ncomp, st);
    }
    {
        ProfScope ps(prof, CLAIRE_K_FFT_C2C, st, ncomp * 2 * C);
        c2c_x2(d, ax[1], spec, ncomp, -1.f, st);
    }
}
void inverse_23(const Dims &d, const FftPlan *ax, float2 *spec, float *out, const float *add, int ncomp,
                cudaStream_t st, Profiler *prof) {
    const double R = 4.0 * d.N, C = 8.0 * d.n1 * d.n2 * d.h3;
    if (d.n2 == d.n3 && plane_fft(d.n3)) {
        ProfScope ps(prof, CLAIRE_K_FFT_C2R, st, ncomp * (R + C + (add ? R : 0.0)));
        switch (d.n3) {
            case 32: plane_inv<32>(d, ax[2], spec, out, add, ncomp, st); return;
            case 64: plane_inv<64>(d, ax[2], spec, out, add, ncomp, st); return;
            default: plane_inv<96>(d, ax[2], spec, out, add, ncomp, st); return;
        }
    }
    {
        ProfScope ps(prof, CLAIRE_K_FFT_C2C, st, ncomp * 2 * C);
        c2c_x2(d, ax[1], spec, ncomp, +1.f, st);
    }
    {
        ProfScope ps(prof, CLAIRE_K_FFT_C2R, st, ncomp * (R + C + (add ? R : 0.0)));
        c2r_x3(d, ax[2], spec, out, add, ncomp, st);
    }
}

// ------------------------------------------------------ grid resampling ---
__device__ __forceinline__ bool in_coarse_band(float k, int nc) { return 2.f * fabsf(k) < (float)nc; }
__device__ __forceinline__ int index_of(float k, int n) { return k < 0.f ? n + (int)k : (int)k; }

// thread per coarse (component, i1, i2, k3)
__global__ void k_spec_restrict(const float2 *__restrict__ sf, Dims df, float2 *__restrict__ sc,
                                Dims dc, float scale) {
    const long long per_c = (long long)dc.n1 * dc.n2 * dc.h3;
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= 3 * per_c) return;
    const int c = (int)(t / per_c);
    long long r = t - c * per_c;
    const int k3 = (int)(r % dc.h3);
    r /= dc.h3;
    const int i2 = (int)(r % dc.n2), i1 = (int)(r / dc.n2);
    const float k1 = wavenumber(i1, dc.n1), k2 = wavenumber(i2, dc.n2);
    float2 v = make_float2(0.f, 0.f);
    if (in_coarse_band(k1, dc.n1) && in_coarse_band(k2, dc.n2) && in_coarse_band((float)k3, dc.n3)) {
        const long long src = (((long long)c * df.n1 + index_of(k1, df.n1)) * df.n2 + index_of(k2, df.n2)) *
                              df.p3 + k3;
        const float2 f = sf[src];
        v = make_float2(f.x * scale, f.y * scale);
    }
    sc[(((long long)c * dc.n1 + i1) * dc.n2 + i2) * dc.p3 + k3] = v;
}

// thread per fine (i1, i2, k3), all three components (the inverse couples them)
__global__ void k_spec_twolevel(float2 *__restrict__ sf, Dims df, const float2 *__restrict__ sc,
                                Dims dc, float scale, float beta0, float gamma) {
    const long long per_c = (long long)df.n1 * df.n2 * df.h3;
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= per_c) return;
    long long r = t;
    const int k3i = (int)(r % df.h3);
    r /= df.h3;
    const int i2 = (int)(r % df.n2), i1 = (int)(r / df.n2);
    const long long cs = (long long)df.n1 * df.n2 * df.p3;
    const long long id = ((long long)i1 * df.n2 + i2) * df.p3 + k3i;
    const float k1 = wavenumber(i1, df.n1), k2 = wavenumber(i2, df.n2), k3 = (float)k3i;
    if (in_coarse_band(k1, dc.n1) && in_coarse_band(k2, dc.n2) && in_coarse_band(k3, dc.n3)) {
        const long long ccs = (long long)dc.n1 * dc.n2 * dc.p3;
        const long long src = ((long long)index_of(k1, dc.n1) * dc.n2 + index_of(k2, dc.n2)) * dc.p3 + k3i;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float2 f = sc[c * ccs + src];
            sf[c * cs + id] = make_float2(f.x * scale, f.y * scale);
        }
    } else {
        // (beta0 A)^{-1} by Sherman-Morrison (never k = 0 here)
        const float k1d = wavenumber_d1(i1, df.n1), k2d = wavenumber_d1(i2, df.n2);
        const float k3d = ((df.n3 & 1) == 0 && 2 * k3i == df.n3) ? 0.f : k3;
        const float kk = k1 * k1 + k2 * k2 + k3 * k3, kd2 = k1d * k1d + k2d * k2d + k3d * k3d;
        const float bk = beta0 * kk, diag = 1.f / bk, coup = -gamma * diag / (bk + gamma * kd2);
        const float2 a = sf[id], b = sf[cs + id], c = sf[2 * cs + id];
        const float2 kv = make_float2(k1d * a.x + k2d * b.x + k3d * c.x, k1d * a.y + k2d * b.y + k3d * c.y);
        sf[id] = make_float2(diag * a.x + coup * k1d * kv.x, diag * a.y + coup * k1d * kv.y);
        sf[cs + id] = make_float2(diag * b.x + coup * k2d * kv.x, diag * b.y + coup * k2d * kv.y);
        sf[2 * cs + id] = make_float2(diag * c.x + coup * k3d * kv.x, diag * c.y + coup * k3d * kv.y);
    }
}

}  // namespace

void spectral_apply(const Dims &d, const FftPlan *ax, SpecOp op, const SpecParams &sp,
                    const float *in, float *out, const float *add, float2 *spec, cudaStream_t st,
                    Profiler *prof) {
    // first derivatives go through the axis transforms (fft_axis.cu); the
    // 3D passes below serve the operators that couple wavenumbers, A and A^-1
    if (op == OP_GRAD) {
        spectral_grad_1d(d, ax, in, out, st, prof);
        return;
    }
    if (op == OP_DIV) {
        spectral_div_1d(d, ax, in, out, st, prof);
        return;
    }
    // algorithmic bytes: real fields 4 B/voxel, half spectra 8 B per stored mode
    forward_32(d, ax, in, spec, 3, st, prof);
    {
        ProfScope ps(prof, CLAIRE_K_FFT_MUL, st, 6 * 8.0 * d.n1 * d.n2 * d.h3);
        switch (op) {
            case OP_A: mul_x1_op<OP_A>(d, ax[0], spec, sp, st); break;
            case OP_AINV: mul_x1_op<OP_AINV>(d, ax[0], spec, sp, st); break;
            default: break;
        }
    }
    inverse_23(d, ax, spec, out, add, 3, st, prof);
}

}  // namespace claire

namespace claire {

void spectral_forward3(const Dims &d, const FftPlan *ax, const float *in, float2 *spec,
                       cudaStream_t st, Profiler *prof) {
    forward_32(d, ax, in, spec, 3, st, prof);
    ProfScope ps(prof, CLAIRE_K_FFT_MUL, st, 6 * 8.0 * d.n1 * d.n2 * d.h3);
    mul_x1_op<OP_X1FWD>(d, ax[0], spec, SpecParams{0.f, 0.f, 1.f}, st);
}

void spectral_inverse3(const Dims &d, const FftPlan *ax, float2 *spec, float *out, float scale,
                       cudaStream_t st, Profiler *prof) {
    {
        ProfScope ps(prof, CLAIRE_K_FFT_MUL, st, 6 * 8.0 * d.n1 * d.n2 * d.h3);
        mul_x1_op<OP_X1INV>(d, ax[0], spec, SpecParams{0.f, 0.f, scale}, st);
    }
    inverse_23(d, ax, spec, out, nullptr, 3, st, prof);
}

void launch_spec_restrict(const Dims &df, const float2 *specf, const Dims &dc, float2 *specc,
                          float scale, cudaStream_t st, Profiler *prof) {
    const long long n = 3LL * dc.n1 * dc.n2 * dc.h3;
    ProfScope ps(prof, CLAIRE_K_FFT_MUL, st, 16.0 * n);
    k_spec_restrict<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(specf, df, specc, dc, scale);
}

void launch_spec_twolevel(const Dims &df, float2 *specf, const Dims &dc, const float2 *specc,
                          float scale, float beta0, float gamma, cudaStream_t st, Profiler *prof) {
    const long long n = (long long)df.n1 * df.n2 * df.h3;
    ProfScope ps(prof, CLAIRE_K_FFT_MUL, st, 48.0 * n);
    k_spec_twolevel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(specf, df, specc, dc, scale, beta0,
                                                                 gamma);
}

}  // namespace claire
