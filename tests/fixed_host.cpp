// Host build of the device arithmetic in fixed.cuh, for test_fixed_host.py: the CUDA functions it
// calls are given their meaning in plain C++, so the integer steps run on the CPU, under a
// sanitizer.  Reads binary values from standard input, writes int64 to standard output.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

using std::floor;
using std::max;
using std::min;

#define GPIC_HOST_OP(name, type, op) \
    static inline type name(type a, type b) { return a op b; }
GPIC_HOST_OP(__fmul_rn, float, *)
GPIC_HOST_OP(__dmul_rn, double, *)
GPIC_HOST_OP(__fadd_rn, float, +)
GPIC_HOST_OP(__dadd_rn, double, +)
GPIC_HOST_OP(__fsub_rn, float, -)
GPIC_HOST_OP(__dsub_rn, double, -)
GPIC_HOST_OP(__fdiv_rn, float, /)
GPIC_HOST_OP(__ddiv_rn, double, /)
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline float __fsqrt_rn(float a) { return std::sqrt(a); }
static inline double __dsqrt_rn(double a) { return std::sqrt(a); }
static inline double __longlong_as_double(long long v) {
    double d;
    std::memcpy(&d, &v, sizeof d);
    return d;
}
static inline double __hiloint2double(int hi, int lo) {
    return __longlong_as_double(
        (long long)(((unsigned long long)(unsigned)hi << 32) | (unsigned)lo));
}
static inline long long __double2ll_rn(double v) { return std::llrint(v); }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
static inline long long __mul64hi(long long a, long long b) {
    return (long long)(((__int128)a * b) >> 64);
}
static inline int __clzll(long long v) {
    return v ? __builtin_clzll((unsigned long long)v) : 64;
}

#include "fixed.cuh"

using namespace gpic;

namespace {

template <typename T>
std::vector<T> read_all() {
    std::vector<T> v;
    T x;
    while (std::fread(&x, sizeof x, 1, stdin) == 1) v.push_back(x);
    return v;
}

// shape P SH: fixed-point positions -> first node, the p+1 weights, the p+1 derivatives
template <int P>
void shape(int sh) {
    for (long long X : read_all<long long>()) {
        long long w[P + 1], d[P + 1], first = fix_weights<P>(X, sh, w);
        fix_dweights<P>(X, sh, d);
        std::fwrite(&first, sizeof first, 1, stdout);
        std::fwrite(w, sizeof w, 1, stdout);
        std::fwrite(d, sizeof d, 1, stdout);
    }
}

// deposit P SH: (v, X, Y) -> the (p+1)^2 contributions of v W_x W_y
template <int P>
void deposit(int sh) {
    const std::vector<long long> in = read_all<long long>();
    for (size_t k = 0; k + 2 < in.size(); k += 3) {
        long long wx[P + 1], wy[P + 1];
        fix_weights<P>(in[k + 1], sh, wx);
        fix_weights<P>(in[k + 2], sh, wy);
        for (int a = 0; a <= P; ++a)
            for (int b = 0; b <= P; ++b) {
                const long long x = deposit_value(deposit_row(in[k], wx[a]), deposit_col(wy[b]));
                std::fwrite(&x, sizeof x, 1, stdout);
            }
    }
}

// gather P SH: (nx, ny, n, the field [nx][ny], x and y of n particles in cells) -> per particle
// the value gathered as k_gather_push_fix does, then value, d/dx and d/dy by the separable sums
// of the reverse kernels (the bits of four doubles)
template <int P>
void gather(int sh) {
    constexpr int S1 = P + 1;
    const std::vector<double> in = read_all<double>();
    const int nx = (int)in[0], ny = (int)in[1], n = (int)in[2];
    const double *f = &in[3], *xs = f + (size_t)nx * ny, *ys = xs + n;
    std::vector<int2> F((size_t)nx * ny);
    std::vector<int> e(nx);
    for (int i = 0; i < nx; ++i) {
        unsigned top = 0;
        for (int j = 0; j < ny; ++j) {
            unsigned long long bits;
            std::memcpy(&bits, f + (size_t)i * ny + j, sizeof bits);
            top = max(top, (unsigned)(bits >> 32) & 0x7fffffffu);
        }
        e[i] = row_exponent(top);
        for (int j = 0; j < ny; ++j) F[(size_t)i * ny + j] = field_fix(f[(size_t)i * ny + j], e[i]);
    }
    const double scale = std::ldexp(1.0, sh);
    for (int p = 0; p < n; ++p) {
        const long long X = __double2ll_rn(xs[p] * scale), Y = __double2ll_rn(ys[p] * scale);
        long long wx[S1], wy[S1], dx[S1], dy[S1];
        const int ix = fix_weights<P>(X, sh, wx), iy = fix_weights<P>(Y, sh, wy);
        fix_dweights<P>(X, sh, dx);
        fix_dweights<P>(Y, sh, dy);
        int top = -900;
        for (int a = 0; a < S1; ++a) top = max(top, e[(ix + a + nx) % nx]);
        long long s0 = 0;
        LimbSum sum[3];
        for (int a = 0; a < S1; ++a) {
            const int gi = (ix + a + nx) % nx;
            LimbSum r0, rr, rs;
            for (int b = 0; b < S1; ++b) {
                const int2 v = F[(size_t)gi * ny + (iy + b + ny) % ny];
                r0.add(weight_limbs(mul62(wx[a], wy[b])), v.x, v.y);
                rr.add(weight_limbs(wy[b]), v.x, v.y);
                rs.add(weight_limbs(dy[b]), v.x, v.y);
            }
            const int d = top - e[gi];
            s0 += r0.shifted(d);
            const int2 r = limbs(rr.shifted(d));
            const int2 s = limbs(rs.shifted(d));
            sum[0].add(weight_limbs(wx[a]), r.x, r.y);
            sum[1].add(weight_limbs(dx[a]), r.x, r.y);
            sum[2].add(weight_limbs(wx[a]), s.x, s.y);
        }
        const double out[4] = {fix_value(s0, top), fix_value(sum[0].value(), top),
                               fix_value(sum[1].value(), top), fix_value(sum[2].value(), top)};
        std::fwrite(out, sizeof out, 1, stdout);
    }
}

template <typename F>
void by_degree(int p, F&& f) {
    if (p == 2) f(std::integral_constant<int, 2>());
    if (p == 3) f(std::integral_constant<int, 3>());
    if (p == 4) f(std::integral_constant<int, 4>());
}

}  // namespace

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    const std::string what = argv[1];
    const int p = std::atoi(argv[2]), sh = std::atoi(argv[3]);
    if (what == "shape") by_degree(p, [&](auto P) { shape<decltype(P)::value>(sh); });
    if (what == "gather") by_degree(p, [&](auto P) { gather<decltype(P)::value>(sh); });
    if (what == "deposit") by_degree(p, [&](auto P) { deposit<decltype(P)::value>(sh); });
    return 0;
}
