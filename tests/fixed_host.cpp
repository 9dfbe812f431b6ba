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
    if (what == "deposit") by_degree(p, [&](auto P) { deposit<decltype(P)::value>(sh); });
    return 0;
}
