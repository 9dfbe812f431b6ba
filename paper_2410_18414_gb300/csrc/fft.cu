// Shared-memory mixed-radix (4, 2, 3) Stockham FFT for the spectral field solve.
//
// The paper inverts the modified Helmholtz operator and takes every spatial
// derivative with the FFT on the periodic grid (sections 3.1 and 4).  Grids here
// are at most a few thousand points per side, so each CTA loads whole lines into
// shared memory, runs all radix passes there (ping-pong buffers, autosort
// Stockham ordering: no bit reversal) and writes the lines back once.
//
// Pass with radix R on lines of length n, Ns = product of the earlier radices:
//   for j in [0, n/R):  k = j mod Ns
//     a_r = src[j + r n/R] * w^(r k n/(Ns R)),  r = 0..R-1   (w = exp(sign 2 pi i / n))
//     b   = R-point DFT of a
//     dst[(j div Ns) Ns R + k + r Ns] = b_r
// which leaves the transform in natural order after the last pass.
#include "common.cuh"
#include "fixed.cuh"
#include "fft_device.cuh"
#include "gpic_internal.h"
#include "launch.cuh"

namespace gpic {

namespace {

constexpr int kThreads = 256;

// The largest magnitudes of at most four lines of m complex values as high words into top[8]
// (shared, zeroed; re, im of each line).
__device__ __forceinline__ void collect_max(const double2* res, int lines, int m, unsigned* top) {
    const int b = threadIdx.x & 3;
    unsigned re = 0, im = 0;
    for (int e = b < lines ? threadIdx.x >> 2 : m; e < m; e += blockDim.x >> 2) {
        const double2 v = res[b * m + e];
        re = max(re, (unsigned)__double2hiint(v.x) & 0x7fffffffu);
        im = max(im, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
    }
    for (int o = 16; o >= 4; o >>= 1) {
        re = max(re, __shfl_xor_sync(0xffffffffu, re, o));
        im = max(im, __shfl_xor_sync(0xffffffffu, im, o));
    }
    if ((threadIdx.x & 31) < lines) {
        atomicMax(top + 2 * b, re);
        atomicMax(top + 2 * b + 1, im);
    }
}

// A second set of arrays of the same launch (the CTAs of blockIdx.y = 1).
template <typename T>
struct FftSecond {
    const cplx_t<T>* in;
    cplx_t<T>* out;
    int nb;
    const longlong2* fix_in;
    longlong2* clear;
    int4* ffix;
    int* fexp;
};

// Transforms along y (contiguous): CTA = `rows` consecutive x-indices of all nb arrays.
template <typename T>
__global__ void __launch_bounds__(kThreads)
k_fft_y(const cplx_t<T>* __restrict__ in, cplx_t<T>* __restrict__ out, int nx, int ny, int nb,
        int rows, FftDesc d, const cplx_t<T>* __restrict__ tw, int sign, int interleave,
        const longlong2* __restrict__ fix_in, double unscale, longlong2* __restrict__ clear,
        int4* __restrict__ ffix, int* __restrict__ fexp, void* __restrict__ sums, int sums32, FftSecond<T> two) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* b0 = reinterpret_cast<C*>(smem_raw);
    if (blockIdx.y) {
        in = two.in;
        out = two.out;
        nb = two.nb;
        fix_in = two.fix_in;
        clear = two.clear;
        ffix = two.ffix;
        fexp = two.fexp;
    }
    const int lines = nb * rows;
    C* b1 = b0 + lines * ny;
    C* tws = b1 + lines * ny;  // twiddles, staged before the wait (they are constant)
    stage_twiddles(tw, tws, ny);
    __shared__ unsigned top[8];
    if (threadIdx.x < 8) top[threadIdx.x] = 0;
    const int i0 = blockIdx.x * rows;
    const size_t plane = (size_t)nx * ny;
    griddep_wait();  // the input is the previous kernel's output
    griddep_launch();
    if constexpr (sizeof(T) == 8) {
        if (sums) {  // nb values a node (FP64 or FP32), zeroed for the next sums; one row
            for (int e = threadIdx.x; e < lines * ny; e += blockDim.x) {
                const int jj = e / nb, b = e - jj * nb;
                const size_t src = (size_t)i0 * ny * nb + e;
                double2 v;
                if (sums32) {
                    float2* q = reinterpret_cast<float2*>(sums) + src;
                    v = make_double2(q->x, q->y);
                    *q = make_float2(0.f, 0.f);
                } else {
                    double2* q = reinterpret_cast<double2*>(sums) + src;
                    v = *q;
                    *q = make_double2(0.0, 0.0);
                }
                b0[b * ny + jj] = v;
            }
        }
    }
    for (int e = sums ? lines * ny : threadIdx.x; e < lines * ny; e += blockDim.x) {
        int l = e / ny, jj = e - l * ny;
        int b = l / rows, r = l - b * rows;
        const size_t src = b * plane + (size_t)(i0 + r) * ny + jj;
        if (fix_in) {  // fixed-point current sums, converted on load
            const longlong2 v = fix_in[src];
            if (clear) clear[src] = longlong2{0, 0};  // the other buffer, for the next deposit
            if constexpr (sizeof(T) == 4) {
                b0[e] = mk<C>((double)v.x * unscale, (double)v.y * unscale);
            } else {  // 128-bit sums: the high words follow the low ones
                const longlong2 hi = fix_in[plane + src];
                if (clear) clear[plane + src] = longlong2{0, 0};
                b0[e] = make_double2(fix128_value(hi.x, (unsigned long long)v.x, unscale),
                                     fix128_value(hi.y, (unsigned long long)v.y, unscale));
            }
        } else {
            b0[e] = in[src];
        }
    }
    __syncthreads();
    C* res = run_passes(b0, b1, d, lines, (const C*)tws, sign);
    if (interleave) {
        if constexpr (sizeof(T) == 8) {
            if (ffix) {  // one row, nb = 4 or 2: its fixed-point fields beside the FP64 ones
                collect_max(res, nb, ny, top);
                __syncthreads();
                if (threadIdx.x < 2 * nb) fexp[2 * nb * i0 + threadIdx.x] = row_exponent(top[threadIdx.x]);
                const int b = threadIdx.x & (nb - 1);
                const int er = row_exponent(top[2 * b]), ei = row_exponent(top[2 * b + 1]);
                for (int e = threadIdx.x; e < nb * ny; e += blockDim.x) {
                    const double2 v = res[b * ny + e / nb];
                    const int2 re = field_fix(v.x, er), im = field_fix(v.y, ei);
                    const size_t o = (size_t)i0 * ny * nb + e;
                    out[o] = v;
                    ffix[o] = make_int4(re.x, re.y, im.x, im.y);
                }
                return;
            }
        }
        for (int e = threadIdx.x; e < lines * ny; e += blockDim.x) {
            int b = e % nb, t = e / nb;
            int jj = t % ny, r = t / ny;
            out[((size_t)(i0 + r) * ny + jj) * nb + b] = res[(b * rows + r) * ny + jj];
        }
    } else {
        if constexpr (sizeof(T) == 8) {
            if (ffix) {  // nb = 1: the fixed-point values of the one or two rows as well
                collect_max(res, rows, ny, top);
                __syncthreads();
                if (threadIdx.x < 2 * rows) fexp[2 * i0 + threadIdx.x] = row_exponent(top[threadIdx.x]);
            }
        }
        for (int e = threadIdx.x; e < lines * ny; e += blockDim.x) {
            int l = e / ny, jj = e - l * ny;
            int b = l / rows, r = l - b * rows;
            const size_t o = b * plane + (size_t)(i0 + r) * ny + jj;
            out[o] = res[e];
            if constexpr (sizeof(T) == 8) {
                if (ffix) {
                    const int2 re = field_fix(res[e].x, row_exponent(top[2 * l]));
                    const int2 im = field_fix(res[e].y, row_exponent(top[2 * l + 1]));
                    ffix[o] = make_int4(re.x, re.y, im.x, im.y);
                }
            }
        }
    }
}

// Transforms along x (stride ny): CTA = `cols` consecutive y-indices of one array.
template <typename T>
__global__ void __launch_bounds__(kThreads)
k_fft_x(const cplx_t<T>* __restrict__ in, cplx_t<T>* __restrict__ out, int nx, int ny, int cols,
        FftDesc d, const cplx_t<T>* __restrict__ tw, int sign) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* b0 = reinterpret_cast<C*>(smem_raw);
    C* b1 = b0 + cols * nx;
    const int j0 = blockIdx.x * cols;
    const size_t off = (size_t)blockIdx.y * nx * ny;
    for (int t = threadIdx.x; t < nx * cols; t += blockDim.x) {
        int e = t / cols, c = t - e * cols;
        b0[c * nx + e] = in[off + (size_t)e * ny + j0 + c];
    }
    __syncthreads();
    C* res = run_passes(b0, b1, d, cols, tw, sign);
    for (int t = threadIdx.x; t < nx * cols; t += blockDim.x) {
        int e = t / cols, c = t - e * cols;
        out[off + (size_t)e * ny + j0 + c] = res[c * nx + e];
    }
}

template <typename T>
__global__ void k_twiddles(cplx_t<T>* tw, int n) {
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < n) {
        double s, c;
        sincospi(2.0 * (double)m / (double)n, &s, &c);
        tw[m] = mk<cplx_t<T>>(c, -s);
    }
}

constexpr size_t kSmemBudget = 96 * 1024;

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

template <typename T>
static cudaError_t fft_y_impl(const void* in, void* out, int nx, int ny, int nb, const FftDesc& d,
                              const void* tw, int sign, int interleave, const longlong2* fix_in,
                              double unscale, longlong2* clear, cudaStream_t s,
                              const FixFields* fix = nullptr, void* sums = nullptr,
                              bool sums32 = false, const FftSecond<T>* two = nullptr) {
    using C = cplx_t<T>;
    const size_t per_line = 2 * (size_t)ny * sizeof(C);
    const size_t tw_bytes = (size_t)ny * sizeof(C);
    // few lines per CTA: these transforms are latency-bound, so favour CTAs (one row of
    // all nb arrays each, or two rows when there is a single array)
    int rows = nb == 1 && nx % 2 == 0 ? 2 : 1;
    if ((size_t)rows * nb * per_line + tw_bytes > 200 * 1024) rows = 1;
    if ((size_t)rows * nb * per_line + tw_bytes > 200 * 1024) return cudaErrorInvalidValue;
    size_t smem = (size_t)rows * nb * per_line + tw_bytes;
    cudaError_t e = set_smem(k_fft_y<T>, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_fft_y<T>, dim3(nx / rows, two ? 2 : 1), dim3(kThreads), smem, s,
                      (const C*)in, (C*)out,
                      nx, ny, nb, rows, d, (const C*)tw, sign, interleave, fix_in, unscale, clear,
                      fix ? (int4*)fix->f : nullptr, fix ? fix->exp : nullptr, sums,
                      sums32 ? 1 : 0, two ? *two : FftSecond<T>{});
}

template <typename T>
cudaError_t launch_fft_y(const void* in, void* out, int nx, int ny, int nb, const FftDesc& d,
                         const void* tw, int sign, int interleave, cudaStream_t s,
                         const FixFields* fix) {
    if (fix && (sizeof(T) != 8 || !(nb == 4 ? interleave : nb == 1 && !interleave)))
        return cudaErrorInvalidValue;
    return fft_y_impl<T>(in, out, nx, ny, nb, d, tw, sign, interleave, nullptr, 0.0, nullptr, s,
                         fix);
}

cudaError_t launch_fft_y_from_sums(void* sums, bool f32, void* out, int nx, int ny,
                                   const FftDesc& d, const void* tw, cudaStream_t s) {
    return fft_y_impl<double>(nullptr, out, nx, ny, 4, d, tw, -1, 0, nullptr, 0.0, nullptr, s,
                              nullptr, sums, f32);
}

template <typename T>
cudaError_t launch_fft_y_from_fix(const longlong2* j, double unscale, void* out, int nx, int ny,
                                  const FftDesc& d, const void* tw, longlong2* clear,
                                  cudaStream_t s, const longlong2* j2, void* out2,
                                  longlong2* clear2) {
    const FftSecond<T> two{nullptr, (cplx_t<T>*)out2, 1, j2, clear2, nullptr, nullptr};
    return fft_y_impl<T>(nullptr, out, nx, ny, 1, d, tw, -1, 0, j, unscale, clear, s, nullptr,
                         nullptr, false, j2 ? &two : nullptr);
}

template <typename T>
cudaError_t launch_fft_y_fields(const void* f4, void* g, const void* f2, void* g2, int nx, int ny,
                                const FftDesc& d, const void* tw, const FixFields* fix,
                                const FixFields* fix2, cudaStream_t s) {
    if ((fix || fix2) && sizeof(T) != 8) return cudaErrorInvalidValue;
    const FftSecond<T> two{(const cplx_t<T>*)f2, (cplx_t<T>*)g2, 2, nullptr, nullptr,
                           fix2 ? (int4*)fix2->f : nullptr, fix2 ? fix2->exp : nullptr};
    return fft_y_impl<T>(f4, g, nx, ny, 4, d, tw, +1, 1, nullptr, 0.0, nullptr, s, fix, nullptr,
                         false, f2 ? &two : nullptr);
}

template <typename T>
cudaError_t launch_fft_x(const void* in, void* out, int nx, int ny, int nb, const FftDesc& d,
                         const void* tw, int sign, cudaStream_t s) {
    using C = cplx_t<T>;
    const size_t per_line = 2 * (size_t)nx * sizeof(C);
    int cols = 1;
    while (cols * 2 <= 16 && ny % (cols * 2) == 0 && (size_t)(cols * 2) * per_line <= kSmemBudget)
        cols *= 2;
    if ((size_t)cols * per_line > 200 * 1024) return cudaErrorInvalidValue;
    size_t smem = (size_t)cols * per_line;
    cudaError_t e = set_smem(k_fft_x<T>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(ny / cols, nb);
    k_fft_x<T><<<grid, kThreads, smem, s>>>((const C*)in, (C*)out, nx, ny, cols, d, (const C*)tw,
                                            sign);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_twiddles(void* tw, int n, cudaStream_t s) {
    k_twiddles<T><<<(n + 255) / 256, 256, 0, s>>>((cplx_t<T>*)tw, n);
    return cudaGetLastError();
}

template cudaError_t launch_fft_y<double>(const void*, void*, int, int, int, const FftDesc&,
                                          const void*, int, int, cudaStream_t, const FixFields*);
template cudaError_t launch_fft_y<float>(const void*, void*, int, int, int, const FftDesc&,
                                         const void*, int, int, cudaStream_t, const FixFields*);
template cudaError_t launch_fft_x<double>(const void*, void*, int, int, int, const FftDesc&,
                                          const void*, int, cudaStream_t);
template cudaError_t launch_fft_x<float>(const void*, void*, int, int, int, const FftDesc&,
                                         const void*, int, cudaStream_t);
template cudaError_t launch_fft_y_from_fix<double>(const longlong2*, double, void*, int, int,
                                                   const FftDesc&, const void*, longlong2*,
                                                   cudaStream_t, const longlong2*, void*,
                                                   longlong2*);
template cudaError_t launch_fft_y_fields<double>(const void*, void*, const void*, void*, int, int,
                                             const FftDesc&, const void*, const FixFields*,
                                             const FixFields*, cudaStream_t);
template cudaError_t launch_fft_y_from_fix<float>(const longlong2*, double, void*, int, int,
                                                   const FftDesc&, const void*, longlong2*,
                                                   cudaStream_t, const longlong2*, void*,
                                                   longlong2*);
template cudaError_t launch_fft_y_fields<float>(const void*, void*, const void*, void*, int, int,
                                             const FftDesc&, const void*, const FixFields*,
                                             const FixFields*, cudaStream_t);
template cudaError_t launch_twiddles<double>(void*, int, cudaStream_t);
template cudaError_t launch_twiddles<float>(void*, int, cudaStream_t);

}  // namespace gpic
