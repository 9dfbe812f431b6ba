// Discrete adjoint of the step: the transpose of the Jacobian of one step of
// Algorithm 1 (section 4.2) with the BDF-k (section 3.2), CDF-2 (section 3.1) or DIRK
// (section 3.3) field solve, applied in reverse, for the gradient of an objective of the
// final state with respect to the initial velocities.
//
// Adjoint of a quantity z is written zb; the pairing is the plain sum over particles and
// grid nodes, and Re sum conj(zb) dz for a spectrum.  Reverse of step n -> n+1:
//
//   push + gather (k_adj_push_gather), per particle at x^{n+1}, from the fields the
//   forward push gathered (kept by the recording step):
//     u = P^{n+1} - q A_p, v^{n+1} = c^2 u / D, D = sqrt(c^2 |u|^2 + (m c^2)^2)
//     ub = (c^2/D) (vb - c^2 u (u . vb)/D^2);  Pb += ub;  A_p b = -q ub
//     P^{n+1} = P^n + q dt (-grad phi + (grad A) . v*):  (grad phi)b = -q dt Pb,
//       (d_l A_m)b = q dt Pb_l v*_m,  v*b_m = q dt sum_l Pb_l d_l A_m
//     v* = 2 v^n - v^{n-1}:  v^n b += 2 v*b,  v^{n-1} b = -v*b
//     the gather's transpose deposits the eight field adjoints with the same weights,
//     and x^{n+1} b gets sum_f gb_f grad(sum_node F_f W)
//   field solve (k_adj_modes / k_adj_columns), per mode, after forward transforms of the
//     deposited field adjoints: conj(i k) = -i k for the spectral gradients, then the
//     stepper's recurrences run backwards with their real per-mode multipliers (DIRK:
//     the transpose of the forward's per-mode 2 x 4 step matrix), ending in the
//     adjoint of the current spectrum, inverse-transformed to the mesh
//   deposit + move (k_adj_deposit_move), per particle:
//     J = q_p v^n W(x^{n+1}) / (dx dy):  v^n b += gather(Jb),
//       x^{n+1} b += v^n . grad gather(Jb)   (q_p/(dx dy) folded into Jb)
//     x^{n+1} = x^n + dt v^n:  x^n b = x^{n+1} b,  v^n b += dt x^{n+1} b
//   t = 0 (k_adj_init): P^0 = gamma m v^0 and the Taylor start v^{-1}(v^0, E^0).
//
// One thread per particle or per mode (the stencil passes share a particle among lanes, see
// k_adj_push_gather).  The particle kernels run in the storage type T of
// the forward they reverse: FP64 for the plain path, FP32 for the FP32 form (the adjoint
// of the step in exact arithmetic, evaluated along the FP32 form's trajectory; the
// fixed-point rounding of its current, piecewise constant, is differentiated as the
// identity).  The field adjoints they deposit are summed in FP64 (FP32 form: in FP32, the
// eight values of a node in two vector atomics), eight values a node side by side, and the
// reverse field solve is FP64 in both forms, as the forward's per-mode update is.  Shape weights come
// from Shape<P, T> (the forward's) and their derivatives from the closed forms below; in the
// fixed-point kernels (..._fix) from fix_weights and fix_dweights.
#include <algorithm>

#include "common.cuh"
#include "fft_device.cuh"
#include "fixed.cuh"
#include "gpic_internal.h"
#include "launch.cuh"

namespace gpic {

namespace {

constexpr int kThreads = 256;

inline int blocks_for(int64_t n) {
    int64_t b = (n + kThreads - 1) / kThreads;
    const int64_t cap = 152 * 16;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

// d w[a] / d xi for the weights of Shape<P, T>, from the same offset d.
template <int P, typename T> struct DShape;
template <typename T> struct DShape<2, T> {
    // w = ((1/2 - d)^2/2, 3/4 - d^2, (1/2 + d)^2/2)
    static __device__ __forceinline__ void dweights(T xi, T* dw) {
        const T d = xi - floor(xi + (T)0.5);
        dw[0] = d - (T)0.5;
        dw[1] = (T)-2 * d;
        dw[2] = d + (T)0.5;
    }
};
template <typename T> struct DShape<3, T> {
    // w = (e^3/6, 2/3 - d^2 + d^3/2, 2/3 - e^2 + e^3/2, d^3/6), e = 1 - d
    static __device__ __forceinline__ void dweights(T xi, T* dw) {
        const T d = xi - floor(xi), e = (T)1 - d;
        dw[0] = (T)-0.5 * e * e;
        dw[1] = d * ((T)1.5 * d - (T)2);
        dw[2] = e * ((T)2 - (T)1.5 * e);
        dw[3] = (T)0.5 * d * d;
    }
};
template <typename T> struct DShape<4, T> {
    // derivative of (55 + 20 t - 120 t^2 + 80 t^3 - 16 t^4)/96
    static __device__ __forceinline__ T dmid(T t) {
        return ((T)20 + t * ((T)-240 + t * ((T)240 - (T)64 * t))) * (T)(1.0 / 96.0);
    }
    // w = ((1-2d)^4/384, mid(1+d), (115 - 120 d^2 + 48 d^4)/192, mid(1-d), (1+2d)^4/384)
    static __device__ __forceinline__ void dweights(T xi, T* dw) {
        const T d = xi - floor(xi + (T)0.5);
        const T a = (T)1 - (T)2 * d, b = (T)1 + (T)2 * d;
        dw[0] = -a * a * a * (T)(1.0 / 48.0);
        dw[1] = dmid((T)1 + d);
        dw[2] = d * (d * d - (T)1.25);
        dw[3] = -dmid((T)1 - d);
        dw[4] = b * b * b * (T)(1.0 / 48.0);
    }
};

template <typename T>
__device__ __forceinline__ bool inside(T xi, int n) { return xi >= (T)0 && xi <= (T)n; }

constexpr int kAdjThreads = 128;

// The field adjoints of a warp's 32 particles, each left in shared memory by its lane (rec:
// the S2 products W_x W_y, then gb[8]; base: its first node): the warp's lanes become the
// doubles of ONE particle's stencil nodes (eight a node, side by side), so an atomic touches
// the p+1 rows of neighbouring nodes instead of 32 particles' nodes.
template <int P>
__device__ __forceinline__ void deposit_adjoints(const ParticleGeom& g, const double* rec,
                                                 int stride, const int* rbase,
                                                 double* __restrict__ Fb) {
    constexpr int S1 = P + 1, S2 = S1 * S1;
    constexpr int kWords = 8 * S2, kPasses = (kWords + 31) / 32;
    const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
#pragma unroll 2
    for (int k = 0; k < 32; ++k) {
        const int base = rbase[w0 + k];
        if (base < 0) continue;  // uniform for the warp
        const double* r = rec + (w0 + k) * stride;
        const double gb = r[S2 + (lane & 7)];
#pragma unroll
        for (int q = 0; q < kPasses; ++q) {
            const int word = lane + 32 * q;
            if (word >= kWords) break;
            const int node = word >> 3;
            const int a = node / S1, b = node - a * S1;
            int gi = (base >> 16) + a, gj = (base & 0xFFFF) + b;
            if (gi >= g.nx) gi -= g.nx;
            if (gj >= g.ny) gj -= g.ny;
            atomicAdd(Fb + 8 * ((size_t)gi * g.ny + gj) + (lane & 7), r[node] * gb);
        }
    }
}

// The adjoints of one particle's push: f[2..7] the gathered A, grad A; adds to Pb, sets gb,
// rotates the velocity adjoints.
template <typename T>
__device__ __forceinline__ void reverse_push(const PushParams& pp, const T* f, T px1, T py1, T vx,
                                             T vy, T vxo, T vyo, const AdjParticlesT<T>& ab,
                                             int64_t p, T* gb) {
    const T q = (T)pp.q, qdt = (T)(pp.q * pp.dt), c2 = (T)(pp.c * pp.c),
            mc2 = (T)(pp.m * pp.c * pp.c);
    // velocity: v = c^2 u / D
    const T ux = px1 - q * f[2], uy = py1 - q * f[3];
    const T D = sqrt(c2 * (ux * ux + uy * uy) + mc2 * mc2);
    const T id = (T)1 / D;
    const T vbx = ab.vx[p], vby = ab.vy[p];
    const T cd = c2 * id, udv = (ux * vbx + uy * vby) * cd * id;
    const T ubx = cd * (vbx - ux * udv), uby = cd * (vby - uy * udv);
    const T pbx = ab.px[p] + ubx, pby = ab.py[p] + uby;
    // momentum: P^{n+1} = P^n + q dt (-grad phi + (grad A) . v*)
    const T vsx = (T)2 * vx - vxo, vsy = (T)2 * vy - vyo;
    gb[0] = -qdt * pbx;
    gb[1] = -qdt * pby;
    gb[2] = -q * ubx;
    gb[3] = -q * uby;
    gb[4] = qdt * pbx * vsx;
    gb[5] = qdt * pby * vsx;
    gb[6] = qdt * pbx * vsy;
    gb[7] = qdt * pby * vsy;
    const T vsbx = qdt * (pbx * f[4] + pby * f[5]);
    const T vsby = qdt * (pbx * f[6] + pby * f[7]);
    ab.px[p] = pbx;
    ab.py[p] = pby;
    ab.vx[p] = ab.vxo[p] + (T)2 * vsbx;
    ab.vy[p] = ab.vyo[p] + (T)2 * vsby;
    ab.vxo[p] = -vsbx;
    ab.vyo[p] = -vsby;
}

// FP32: two lanes a particle read one node's fields side by side (16 lines a load instead of 32)
// and add its field adjoints side by side (an atomic's lanes cover 16 whole sectors).  The sums
// keep the order of one lane: s = sum_f gb_f F_f runs through the first lane's four fields, then
// the second's, which also carries the position gradient.  65,536 particles, 64 x 64, cubic, lean
// records: a lane per particle 34 us, now 25 us.  (Depositing particle by particle with a float4
// a lane, as deposit_adjoints does in FP64, was slower than either: the atomics then wait for
// the whole gather instead of running beside it.)
template <int P>
__global__ void __launch_bounds__(kAdjThreads)
k_adj_push_gather_pair(ParticleGeom g, PushParams pp, const float* __restrict__ x1,
                       const float* __restrict__ y1, const float* __restrict__ px1,
                       const float* __restrict__ py1, const float* __restrict__ vx,
                       const float* __restrict__ vy, const float* __restrict__ vxo,
                       const float* __restrict__ vyo, const double* __restrict__ gfa,
                       const float4* __restrict__ F, AdjParticlesT<float> ab,
                       float4* __restrict__ Fb, int64_t n, unsigned int* __restrict__ err) {
    constexpr int S1 = P + 1, kOut = 4 * S1, kStride = (kOut + 10) | 1;
    __shared__ float rec[kAdjThreads * kStride];  // W_x, W_y, dW_x, dW_y; f, then gb; xg, yg
    __shared__ int rbase[kAdjThreads];
    const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
    const float idx_ = (float)g.inv_dx, idy = (float)g.inv_dy;
    const int64_t p = blockIdx.x * (int64_t)kAdjThreads + threadIdx.x;
    float* mine = rec + threadIdx.x * kStride;
    int base = -1;
    griddep_wait();
    griddep_launch();
    if (p < n) {
        const float xi = rmul(x1[p], idx_), yj = rmul(y1[p], idy);
        if (!inside(xi, g.nx) || !inside(yj, g.ny)) {
            atomicOr(err, (unsigned)ERR_NONFINITE);
        } else {
            const int ix = Shape<P, float>::weights(xi, mine);
            const int iy = Shape<P, float>::weights(yj, mine + S1);
            DShape<P, float>::dweights(xi, mine + 2 * S1);
            DShape<P, float>::dweights(yj, mine + 3 * S1);
            base = (wrap_idx(ix, g.nx) << 16) | wrap_idx(iy, g.ny);
        }
    }
    rbase[threadIdx.x] = base;
    __syncwarp();
    const int q = lane & 1;
    if (!gfa) {  // the lean record: the forward's gather again, the same bits
#pragma unroll 1
        for (int t = 0; t < 2; ++t) {
            const int k = w0 + 16 * t + (lane >> 1), kb = rbase[k];
            if (kb < 0) continue;
            float* r = rec + k * kStride;
            float f[4] = {0, 0, 0, 0};
#pragma unroll
            for (int a = 0; a < S1; ++a) {
                int gi = (kb >> 16) + a;
                if (gi >= g.nx) gi -= g.nx;
                const float4* row = F + (size_t)gi * g.ny * 2 + q;
#pragma unroll
                for (int b = 0; b < S1; ++b) {
                    int gj = (kb & 0xFFFF) + b;
                    if (gj >= g.ny) gj -= g.ny;
                    const float4 v = __ldg(row + 2 * gj);
                    const float w = rmul(r[a], r[S1 + b]);
                    f[0] = rfma(w, v.x, f[0]);
                    f[1] = rfma(w, v.y, f[1]);
                    f[2] = rfma(w, v.z, f[2]);
                    f[3] = rfma(w, v.w, f[3]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) r[kOut + 4 * q + i] = f[i];
        }
        __syncwarp();
    }
    if (base >= 0) {
        float f[8], gb[8];
#pragma unroll
        for (int k = 2; k < 8; ++k) f[k] = gfa ? (float)gfa[(size_t)(k - 2) * n + p] : mine[kOut + k];
        reverse_push(pp, f, px1[p], py1[p], vx[p], vy[p], vxo[p], vyo[p], ab, p, gb);
#pragma unroll
        for (int k = 0; k < 8; ++k) mine[kOut + k] = gb[k];
    }
    __syncwarp();
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
        const int k = w0 + 16 * t + (lane >> 1), kb = rbase[k];
        float* r = rec + k * kStride;
        float gb[4] = {0, 0, 0, 0}, xg = 0.f, yg = 0.f;
        if (kb >= 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) gb[i] = r[kOut + 4 * q + i];
        }
#pragma unroll 1
        for (int a = 0; a < S1; ++a) {
            int gi = (max(kb, 0) >> 16) + a;
            if (gi >= g.nx) gi -= g.nx;
            const size_t row = (size_t)gi * g.ny;
            const float wxa = kb >= 0 ? r[a] : 0.f;
            float sx = 0.f, sy = 0.f;
#pragma unroll
            for (int b = 0; b < S1; ++b) {
                int gj = (max(kb, 0) & 0xFFFF) + b;
                if (gj >= g.ny) gj -= g.ny;
                const size_t o = 2 * (row + gj) + q;
                const float4 v = __ldg(F + o);
                float sn = 0.f;
                sn += gb[0] * v.x + gb[1] * v.y;
                sn += gb[2] * v.z + gb[3] * v.w;
                sn = __shfl_xor_sync(0xffffffffu, sn, 1);  // the second lane's start
                sn += gb[0] * v.x + gb[1] * v.y;
                sn += gb[2] * v.z + gb[3] * v.w;
                if (kb >= 0) {
                    const float wy = r[S1 + b], w = wxa * wy;
                    sx += wy * sn;
                    sy += r[3 * S1 + b] * sn;
                    atomicAdd(Fb + o, make_float4(w * gb[0], w * gb[1], w * gb[2], w * gb[3]));
                }
            }
            if (kb >= 0) {
                xg += r[2 * S1 + a] * sx;
                yg += wxa * sy;
            }
        }
        if (kb >= 0 && q) {
            r[kOut + 8] = xg;
            r[kOut + 9] = yg;
        }
    }
    __syncwarp();
    if (base >= 0) {
        ab.x[p] += idx_ * mine[kOut + 8];
        ab.y[p] += idy * mine[kOut + 9];
    }
}

// FP64 runs with few particles on the mesh (no fixed-point fields): a lane per particle.
template <int P>
__global__ void __launch_bounds__(kAdjThreads, 6)
k_adj_push_gather(ParticleGeom g, PushParams pp, const double* __restrict__ x1,
                  const double* __restrict__ y1, const double* __restrict__ px1,
                  const double* __restrict__ py1, const double* __restrict__ vx,
                  const double* __restrict__ vy, const double* __restrict__ vxo,
                  const double* __restrict__ vyo, const double* __restrict__ gfa,
                  const double2* __restrict__ F, AdjParticles ab, double* __restrict__ Fb,
                  int64_t n, unsigned int* __restrict__ err) {
    using T = double;
    using C = double2;
    const T idx_ = (T)g.inv_dx, idy = (T)g.inv_dy;
    const int64_t p = blockIdx.x * (int64_t)kAdjThreads + threadIdx.x;
    griddep_wait();
    griddep_launch();
    if (p < n) {
        const T xi = rmul(x1[p], idx_), yj = rmul(y1[p], idy);
        if (!inside(xi, g.nx) || !inside(yj, g.ny)) {
            atomicOr(err, (unsigned)ERR_NONFINITE);
        } else {
            T wx[P + 1], wy[P + 1], dwx[P + 1], dwy[P + 1];
            const int ix = Shape<P, T>::weights(xi, wx);
            const int iy = Shape<P, T>::weights(yj, wy);
            // the fields the forward push gathered at x^{n+1} (dphi/dx, dphi/dy, Ax, Ay,
            // dAx/dx, dAx/dy, dAy/dx, dAy/dy): from the record, or (gfa == NULL, the lean
            // record) gathered again from the step's fields F
            T f[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // f[0], f[1] (grad phi) are not needed here
            if (gfa) {
#pragma unroll
                for (int k = 2; k < 8; ++k) f[k] = (T)gfa[(size_t)(k - 2) * n + p];
            } else {
#pragma unroll 1
                for (int a = 0; a <= P; ++a) {
                    const C* row = F + (size_t)wrap_idx(ix + a, g.nx) * g.ny * 4;
#pragma unroll
                    for (int b = 0; b <= P; ++b) {
                        const C* node = row + (size_t)wrap_idx(iy + b, g.ny) * 4;
                        const T w = rmul(wx[a], wy[b]);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const C v = __ldg(node + k);
                            f[2 * k] = rfma(w, v.x, f[2 * k]);
                            f[2 * k + 1] = rfma(w, v.y, f[2 * k + 1]);
                        }
                    }
                }
            }
            T gb[8];
            reverse_push(pp, f, px1[p], py1[p], vx[p], vy[p], vxo[p], vyo[p], ab, p, gb);
            DShape<P, T>::dweights(xi, dwx);
            DShape<P, T>::dweights(yj, dwy);
            // one pass over the stencil: s = sum_f gb_f F_f at each node gives the position
            // gradient (separable: along y in the row, then across rows), and gb is deposited
            T xg = 0, yg = 0;
#pragma unroll 1
            for (int a = 0; a <= P; ++a) {
                const size_t row = (size_t)wrap_idx(ix + a, g.nx) * g.ny;
                const T wxa = wx[a];
                T sx = 0, sy = 0;
#pragma unroll
                for (int b = 0; b <= P; ++b) {
                    const size_t nd = row + wrap_idx(iy + b, g.ny);
                    const C* node = F + nd * 4;
                    T sn = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const C v = __ldg(node + k);
                        sn += gb[2 * k] * v.x + gb[2 * k + 1] * v.y;
                    }
                    sx += wy[b] * sn;
                    sy += dwy[b] * sn;
                    const T w = wxa * wy[b];
#pragma unroll
                    for (int k = 0; k < 8; ++k) atomicAdd(Fb + 8 * nd + k, w * gb[k]);
                }
                xg += dwx[a] * sx;
                yg += wxa * sy;
            }
            ab.x[p] += idx_ * xg;
            ab.y[p] += idy * yg;
        }
    }
}

// FP64 with the forward's fixed-point fields (k_gather_push_fix): the gathers the adjoint
// needs -- sum_node F_f d(W_x W_y) along x and along y for the position gradient
// sum_f gb_f grad F_f, and (lean record) A and grad A themselves -- are separable integer
// sums, four lanes a particle: along a row with W_y and dW_y, then across rows with W_x and
// dW_x.  The FP64 pipe is left with the push's adjoint and the products the atomics add
// (about 250 operations a particle instead of 600).  262,144 particles, 128 x 128, cubic: with
// FP64 gathers and a lane per particle 263 us, now 139 us.  Bound by the FP64 pipe (72%) and its
// latency: five CTAs an SM (96 registers, 32 bytes spilled) instead of four, 148 -> 137 us (with limbs of 29 bits); six
// are slower.  The lean form gains nothing at five (144.5 -> 146 us) and quartic shapes spill:
// they keep the four and three that their registers allow.
template <int P, bool kLean>
__global__ void __launch_bounds__(kAdjThreads, P > 3 ? 3 : P == 3 && kLean ? 4 : 5)
k_adj_push_gather_fix(ParticleGeom g, FixGeom fg, PushParams pp, const double* __restrict__ x1,
                      const double* __restrict__ y1, const double* __restrict__ px1,
                      const double* __restrict__ py1, const double* __restrict__ vx,
                      const double* __restrict__ vy, const double* __restrict__ vxo,
                      const double* __restrict__ vyo, const double* __restrict__ gfa,
                      const int4* __restrict__ F, const int* __restrict__ ex,
                      AdjParticles ab, double* __restrict__ Fb, int64_t n,
                      unsigned int* __restrict__ err) {
    constexpr int S1 = P + 1, S2 = S1 * S1, kOut = kLean ? 24 : 16;
    constexpr int kUse = 4 * S1 + kOut > S2 + 8 ? 4 * S1 + kOut : S2 + 8;
    constexpr int kStride = kUse | 1;
    __shared__ double rec[kAdjThreads * kStride];
    __shared__ int rbase[kAdjThreads];
    const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
    const int64_t p = blockIdx.x * (int64_t)kAdjThreads + threadIdx.x;
    double* mine = rec + threadIdx.x * kStride;
    long long X = 0, Y = 0;
    int base = -1;
    griddep_wait();
    griddep_launch();
    if (p < n) {
        X = __double2ll_rn(rmul(x1[p], fg.sx));
        Y = __double2ll_rn(rmul(y1[p], fg.sy));
        if (X < 0 || X > ((long long)g.nx << fg.sh) || Y < 0 || Y > ((long long)g.ny << fg.sh)) {
            atomicOr(err, (unsigned)ERR_NONFINITE);
        } else {
            int2* lim = reinterpret_cast<int2*>(mine);  // W_x, dW_x, W_y, dW_y
            long long w[S1];
            const int ix = fix_weights<P>(X, fg.sh, w);
#pragma unroll
            for (int a = 0; a < S1; ++a) lim[a] = weight_limbs(w[a]);
            const int iy = fix_weights<P>(Y, fg.sh, w);
#pragma unroll
            for (int a = 0; a < S1; ++a) lim[2 * S1 + a] = weight_limbs(w[a]);
            fix_dweights<P>(X, fg.sh, w);
#pragma unroll
            for (int a = 0; a < S1; ++a) lim[S1 + a] = weight_limbs(w[a]);
            fix_dweights<P>(Y, fg.sh, w);
#pragma unroll
            for (int a = 0; a < S1; ++a) lim[3 * S1 + a] = weight_limbs(w[a]);
            base = (wrap_idx(ix, g.nx) << 16) | wrap_idx(iy, g.ny);
        }
    }
    rbase[threadIdx.x] = base;
    __syncwarp();
#pragma unroll 1
    for (int t = 0; t < 4; ++t) {
        const int k = w0 + 8 * t + (lane >> 2), q = lane & 3;
        const int kb = rbase[k];
        if (kb < 0) continue;  // its quad of lanes alone; no warp-wide operation below
        const int2* lim = reinterpret_cast<const int2*>(rec + k * kStride);
        int row[S1], e0[S1], e1[S1], top0 = -900, top1 = -900;
#pragma unroll
        for (int a = 0; a < S1; ++a) {
            int gi = (kb >> 16) + a;
            if (gi >= g.nx) gi -= g.nx;
            row[a] = gi;
            const int2 u = __ldg(reinterpret_cast<const int2*>(ex) + 4 * gi + q);
            e0[a] = u.x;
            e1[a] = u.y;
            top0 = max(top0, e0[a]);
            top1 = max(top1, e1[a]);
        }
        LimbSum sx[2], sy[2], sw[2];
#pragma unroll
        for (int a = 0; a < S1; ++a) {
            const int4* F0 = F + (size_t)row[a] * g.ny * 4 + q;
            LimbSum rr[2], rs[2];  // along the row with W_y, dW_y
#pragma unroll
            for (int b = 0; b < S1; ++b) {
                int gj = (kb & 0xFFFF) + b;
                if (gj >= g.ny) gj -= g.ny;
                const int4 v = __ldg(F0 + 4 * gj);
                const int2 wy = lim[2 * S1 + b], dy = lim[3 * S1 + b];
                rr[0].add(wy, v.x, v.y);
                rr[1].add(wy, v.z, v.w);
                rs[0].add(dy, v.x, v.y);
                rs[1].add(dy, v.z, v.w);
            }
            const int2 wx = lim[a], dx = lim[S1 + a];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int d = c ? top1 - e1[a] : top0 - e0[a];
                const int2 r = limbs(rr[c].shifted(d));
                const int2 s = limbs(rs[c].shifted(d));
                sx[c].add(dx, r.x, r.y);
                sy[c].add(wx, s.x, s.y);
                if (kLean) sw[c].add(wx, r.x, r.y);
            }
        }
        double* out = rec + k * kStride + 4 * S1 + 2 * q;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int e = c ? top1 : top0;
            out[c] = fix_value(sx[c].value(), e);
            out[8 + c] = fix_value(sy[c].value(), e);
            if (kLean) out[16 + c] = fix_value(sw[c].value(), e);
        }
    }
    __syncwarp();
    if (base >= 0) {
        const double* got = mine + 4 * S1;
        double f[8];
#pragma unroll
        for (int k = 2; k < 8; ++k) f[k] = kLean ? got[16 + k] : gfa[(size_t)(k - 2) * n + p];
        double gb[8], xg = 0.0, yg = 0.0;
        reverse_push(pp, f, px1[p], py1[p], vx[p], vy[p], vxo[p], vyo[p], ab, p, gb);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            xg += gb[k] * got[k];
            yg += gb[k] * got[8 + k];
        }
        ab.x[p] += g.inv_dx * xg;
        ab.y[p] += g.inv_dy * yg;
        // the record now holds the products W_x W_y and gb
        // (w 2^-62 = w 2^(-2 - 60))
        long long w[S1];
        double wy[S1];
        fix_weights<P>(Y, fg.sh, w);
#pragma unroll
        for (int b = 0; b < S1; ++b) wy[b] = fix_value(w[b], -2);
        fix_weights<P>(X, fg.sh, w);
#pragma unroll
        for (int a = 0; a < S1; ++a) {
            const double wx = fix_value(w[a], -2);
#pragma unroll
            for (int b = 0; b < S1; ++b) mine[a * S1 + b] = wx * wy[b];
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) mine[S2 + k] = gb[k];
    }
    __syncwarp();
    deposit_adjoints<P>(g, rec, kStride, rbase, Fb);
}

template <typename T, int P>
__global__ void __launch_bounds__(kThreads)
k_adj_deposit_move(ParticleGeom g, const T* __restrict__ x1, const T* __restrict__ y1,
                   const T* __restrict__ vx, const T* __restrict__ vy,
                   const double2* __restrict__ Jb, AdjParticlesT<T> ab, int64_t n,
                   unsigned int* __restrict__ err) {
    const T idx_ = (T)g.inv_dx, idy = (T)g.inv_dy, dt = (T)g.dt;
    griddep_wait();
    griddep_launch();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const T xi = rmul(x1[p], idx_), yj = rmul(y1[p], idy);
        if (!inside(xi, g.nx) || !inside(yj, g.ny)) {
            atomicOr(err, (unsigned)ERR_NONFINITE);
            continue;
        }
        T wx[P + 1], wy[P + 1], dwx[P + 1], dwy[P + 1];
        const int ix = Shape<P, T>::weights(xi, wx);
        const int iy = Shape<P, T>::weights(yj, wy);
        DShape<P, T>::dweights(xi, dwx);
        DShape<P, T>::dweights(yj, dwy);
        // separable sums: row a first along y with wy and dwy, then across rows
        T sx = 0, sy = 0, dxx = 0, dxy = 0, dyx = 0, dyy = 0;
#pragma unroll
        for (int a = 0; a <= P; ++a) {
            const size_t row = (size_t)wrap_idx(ix + a, g.nx) * g.ny;
            T rx = 0, ry = 0, rdx = 0, rdy = 0;
#pragma unroll
            for (int b = 0; b <= P; ++b) {
                const double2 jd = __ldg(Jb + row + wrap_idx(iy + b, g.ny));
                const T jx = (T)jd.x, jy = (T)jd.y;
                rx += wy[b] * jx;
                ry += wy[b] * jy;
                rdx += dwy[b] * jx;
                rdy += dwy[b] * jy;
            }
            sx += wx[a] * rx;
            sy += wx[a] * ry;
            dxx += dwx[a] * rx;  // d/dxi of the gathered Jx adjoint
            dxy += dwx[a] * ry;  // d/dxi of the gathered Jy adjoint
            dyx += wx[a] * rdx;
            dyy += wx[a] * rdy;
        }
        const T vxp = vx[p], vyp = vy[p];
        const T xb = ab.x[p] + idx_ * (vxp * dxx + vyp * dxy);
        const T yb = ab.y[p] + idy * (vxp * dyx + vyp * dyy);
        ab.x[p] = xb;
        ab.y[p] = yb;
        ab.vx[p] = ab.vx[p] + sx + dt * xb;
        ab.vy[p] = ab.vy[p] + sy + dt * yb;
    }
}

// The same with the mesh adjoint current in fixed point (an int4 a node, two maxima a row):
// six separable integer sums, about 35 FP64 operations a particle left of 170.  Measured with
// FP64 sums 78 us, now 32 us (262,144 particles, cubic; four CTAs an SM of 128 registers, 34 us
// with three; quartic shapes would spill and keep two).
template <int P>
__global__ void __launch_bounds__(kAdjThreads, P > 3 ? 2 : 4)
k_adj_deposit_move_fix(ParticleGeom g, FixGeom fg, const double* __restrict__ x1,
                       const double* __restrict__ y1, const double* __restrict__ vx,
                       const double* __restrict__ vy, const int4* __restrict__ Jb,
                       const int* __restrict__ ex, AdjParticles ab, int64_t n,
                       unsigned int* __restrict__ err) {
    constexpr int S1 = P + 1;
    const int64_t p = blockIdx.x * (int64_t)kAdjThreads + threadIdx.x;
    griddep_wait();
    griddep_launch();
    if (p >= n) return;
    const long long X = __double2ll_rn(rmul(x1[p], fg.sx)), Y = __double2ll_rn(rmul(y1[p], fg.sy));
    if (X < 0 || X > ((long long)g.nx << fg.sh) || Y < 0 || Y > ((long long)g.ny << fg.sh)) {
        atomicOr(err, (unsigned)ERR_NONFINITE);
        return;
    }
    int2 wy[S1], dy[S1];
    long long wx[S1], dx[S1];
    const int iy = wrap_idx(fix_weights<P>(Y, fg.sh, wx), g.ny);
    fix_dweights<P>(Y, fg.sh, dx);
#pragma unroll
    for (int b = 0; b < S1; ++b) {
        wy[b] = weight_limbs(wx[b]);
        dy[b] = weight_limbs(dx[b]);
    }
    const int ix = wrap_idx(fix_weights<P>(X, fg.sh, wx), g.nx);
    fix_dweights<P>(X, fg.sh, dx);
    int e[2][S1], tops[2] = {-900, -900};
#pragma unroll
    for (int a = 0; a < S1; ++a) {
        int gi = ix + a;
        if (gi >= g.nx) gi -= g.nx;
        const int2 u = __ldg(reinterpret_cast<const int2*>(ex) + gi);
        e[0][a] = u.x;
        e[1][a] = u.y;
        tops[0] = max(tops[0], e[0][a]);
        tops[1] = max(tops[1], e[1][a]);
    }
    // per component: the value, d/dx and d/dy of the gathered current adjoint
    LimbSum sw[2], sx[2], sy[2];
#pragma unroll
    for (int a = 0; a < S1; ++a) {
        int gi = ix + a;
        if (gi >= g.nx) gi -= g.nx;
        const int4* row = Jb + (size_t)gi * g.ny;
        LimbSum rr[2], rs[2];
#pragma unroll
        for (int b = 0; b < S1; ++b) {
            int gj = iy + b;
            if (gj >= g.ny) gj -= g.ny;
            const int4 v = __ldg(row + gj);
            rr[0].add(wy[b], v.x, v.y);
            rr[1].add(wy[b], v.z, v.w);
            rs[0].add(dy[b], v.x, v.y);
            rs[1].add(dy[b], v.z, v.w);
        }
        const int2 wa = weight_limbs(wx[a]), da = weight_limbs(dx[a]);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int d = tops[c] - e[c][a];
            const int2 r = limbs(rr[c].shifted(d));
            const int2 s = limbs(rs[c].shifted(d));
            sw[c].add(wa, r.x, r.y);
            sx[c].add(da, r.x, r.y);
            sy[c].add(wa, s.x, s.y);
        }
    }
    double w[2], jx[2], jy[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        w[c] = fix_value(sw[c].value(), tops[c]);
        jx[c] = fix_value(sx[c].value(), tops[c]);
        jy[c] = fix_value(sy[c].value(), tops[c]);
    }
    const double vxp = vx[p], vyp = vy[p];
    const double xb = ab.x[p] + g.inv_dx * (vxp * jx[0] + vyp * jx[1]);
    const double yb = ab.y[p] + g.inv_dy * (vxp * jy[0] + vyp * jy[1]);
    ab.x[p] = xb;
    ab.y[p] = yb;
    ab.vx[p] = ab.vx[p] + w[0] + g.dt * xb;
    ab.vy[p] = ab.vy[p] + w[1] + g.dt * yb;
}

constexpr int kModeThreads = 256;

__device__ __forceinline__ zd zl(const double2* p) { return zd{p->x, p->y}; }
__device__ __forceinline__ void zs(double2* p, zd v) { *p = make_double2(v.re, v.im); }

// The eight field adjoints' spectra / (nx ny) of mode (kx, ky), from the packed pairs
// za[k] = F(f_2k + i f_2k+1)(k) and zb[k] = the same at -k, folded into the adjoints of
// the three potentials they are taken from: gradient fields i k_l u get -i k_l, the A
// fields themselves 1.  (The particles' phi is phi~ for CDF-2, the new level otherwise.)
__device__ __forceinline__ void gathered_adjoints(const ModeCommon& mc, double kx, double ky,
                                                  const zd* za, const zd* zb, zd& phi, zd& ax,
                                                  zd& ay) {
    zd a[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const zd c = zconj(zb[k]);
        const double h = 0.5 * mc.inv_n;
        a[2 * k] = h * (za[k] + c);
        const zd d = za[k] - c;  // 2i F(f_2k+1)
        a[2 * k + 1] = zd{h * d.im, -h * d.re};
    }
    phi = zi(-kx * a[0]) - zi(ky * a[1]);
    ax = a[2] - zi(kx * a[4]) - zi(ky * a[5]);
    ay = a[3] - zi(kx * a[6]) - zi(ky * a[7]);
}

// Reverse BDF-k field step of mode idx = i ny + j.  Updates the history adjoints of the
// mode and returns the packed adjoint current (Jx + i Jy) q_p/(dx dy).
__device__ __forceinline__ zd adj_mode(const ModeCommon& mc, const AdjModeParams& ap, int idx,
                                       double kx, double ky, const zd* za, const zd* zb) {
    zd phis, axs, ays;
    gathered_adjoints(mc, kx, ky, za, zb, phis, axs, ays);
    phis = zl(ap.phi[0] + idx) + phis;
    axs = zl(ap.ax[0] + idx) + axs;
    ays = zl(ap.ay[0] + idx) + ays;
    // u^{n+1} = (g S - sum_d C_d u^{n+1-d}) / (C_0 + g K)
    const double inv = mc.invd[idx];
    const int L = 2 * ap.k;
    for (int d = 1; d < L; ++d) {
        const double c = ap.C[d] * inv;
        zs(ap.phi[d] + idx, zl(ap.phi[d] + idx) - c * phis);
        zs(ap.ax[d] + idx, zl(ap.ax[d] + idx) - c * axs);
        zs(ap.ay[d] + idx, zl(ap.ay[d] + idx) - c * ays);
    }
    const double cl = ap.C[L] * inv;
    zs(ap.phi[0] + idx, -(cl * phis));
    zs(ap.ax[0] + idx, -(cl * axs));
    zs(ap.ay[0] + idx, -(cl * ays));
    // rho^{n+1} = -sum_j a_j rho^{n+1-j} - beta dt i k . J   (a_0 = 1); phi's source rho/eps0
    const zd rhos = zl(ap.rho[0] + idx) + (ap.g * inv / mc.eps0) * phis;
    for (int d = 1; d < ap.k; ++d) zs(ap.rho[d] + idx, zl(ap.rho[d] + idx) - ap.a[d] * rhos);
    zs(ap.rho[0] + idx, -(ap.a[ap.k] * rhos));
    // current: -beta dt i k_l (continuity) and g mu0 / (C_0 + g K) (A's source)
    const double ga = ap.g * mc.mu0 * inv;
    const zd jx = zi(ap.bdt * kx * rhos) + ga * axs;
    const zd jy = zi(ap.bdt * ky * rhos) + ga * ays;
    // packed (Jx + i Jy), times q_p/(dx dy): the adjoint of the raw deposit sums after
    // the unnormalised inverse transform
    return mc.jscale * (jx + zi(jy));
}

// Reverse CDF-2 field step of mode idx (section 3.1; form 0 implicit, 1 semi-implicit,
// 2 explicit).  cp holds the adjoints of the levels after the step by role (cur, prev);
// the adjoints of the levels before it are written into the other buffer of each pair
// (cur into prev, prev into cur), so the host swaps each pair after the launch, the
// mirror of the forward's swap.  The particles' phi~ = (phi^{n+3/2} + phi^{n+1/2})/2.
__device__ __forceinline__ zd adj_mode(const ModeCommon& mc, const CdfParams& cp, int idx,
                                       double kx, double ky, const zd* za, const zd* zb) {
    auto L = [&](void* p) { return zl(reinterpret_cast<const double2*>(p) + idx); };
    auto S = [&](void* p, zd v) { zs(reinterpret_cast<double2*>(p) + idx, v); };
    zd phic, axc, ayc;
    gathered_adjoints(mc, kx, ky, za, zb, phic, axc, ayc);
    const zd phin = L(cp.phi) + 0.5 * phic;   // phi^{n+3/2}
    zd phih = L(cp.phi_prev) + 0.5 * phic;    // phi^{n+1/2}
    zd rhon = L(cp.rho), rhoh = L(cp.rho_prev);
    const zd axn = L(cp.ax) + axc, ayn = L(cp.ay) + ayc;  // A^{n+1}
    zd axh = L(cp.ax_prev), ayh = L(cp.ay_prev);          // A^n
    zd jxn = L(cp.jx), jyn = L(cp.jy);                    // J^{n+1} (this step's)
    zd jxh = L(cp.jx_prev), jyh = L(cp.jy_prev);          // J^n
    zd rhop{0.0, 0.0}, jxp{0.0, 0.0}, jyp{0.0, 0.0};      // the oldest levels read
    const double dt = mc.dt, h2 = mc.c * mc.c * dt * dt;
    if (cp.form == 0) {
        // u^{n+1} = inv (2 u^n + th (S^{n+1} + S^{n-1})) - u^{n-1}, th = c^2 dt^2 / 2
        const double inv = mc.invd[idx], ts = inv * 0.5 * h2;
        phih = phih + (2.0 * inv) * phin;
        rhon = rhon + (ts / mc.eps0) * phin;
        rhop = (ts / mc.eps0) * phin;
        axh = axh + (2.0 * inv) * axn;
        ayh = ayh + (2.0 * inv) * ayn;
        jxn = jxn + (ts * mc.mu0) * axn;
        jyn = jyn + (ts * mc.mu0) * ayn;
        jxp = (ts * mc.mu0) * axn;
        jyp = (ts * mc.mu0) * ayn;
    } else {
        // semi: u^{n+1} = inv (2 u^n + c^2 dt^2 S^n) - u^{n-1};
        // explicit: u^{n+1} = (2 - c^2 dt^2 K) u^n - u^{n-1} + c^2 dt^2 S^n
        const double K = kx * kx + ky * ky;
        const double inv = cp.form == 1 ? mc.invd[idx] : 1.0;
        const double mu = cp.form == 1 ? 2.0 * inv : 2.0 - h2 * K, ss = inv * h2;
        phih = phih + mu * phin;
        rhoh = rhoh + (ss / mc.eps0) * phin;
        axh = axh + mu * axn;
        ayh = ayh + mu * ayn;
        jxh = jxh + (ss * mc.mu0) * axn;
        jyh = jyh + (ss * mc.mu0) * ayn;
    }
    // rho^{n+3/2} = rho^{n+1/2} - dt i k . J^{n+1}
    rhoh = rhoh + rhon;
    jxn = jxn + zi(dt * kx * rhon);
    jyn = jyn + zi(dt * ky * rhon);
    S(cp.phi_prev, phih);
    S(cp.phi, -phin);
    S(cp.rho_prev, rhoh);
    S(cp.rho, rhop);
    S(cp.ax_prev, axh);
    S(cp.ax, -axn);
    S(cp.ay_prev, ayh);
    S(cp.ay, -ayn);
    S(cp.jx_prev, jxh);
    S(cp.jx, jxp);
    S(cp.jy_prev, jyh);
    S(cp.jy, jyp);
    return mc.jscale * (jxn + zi(jyn));
}

// Reverse DIRK field step of mode idx (section 3.3): dp's state pointers hold the
// adjoints of the state after the step (phi, v_phi, A, v_A, rho, J^{n+1}), overwritten in
// place with those of the state before it (J^n in the J slots).
__device__ __forceinline__ zd adj_mode(const ModeCommon& mc, const DirkParams& dp, int idx,
                                       double kx, double ky, const zd* za, const zd* zb) {
    auto L = [&](void* p) { return zl(reinterpret_cast<const double2*>(p) + idx); };
    auto S = [&](void* p, zd v) { zs(reinterpret_cast<double2*>(p) + idx, v); };
    zd phic, axc, ayc;
    gathered_adjoints(mc, kx, ky, za, zb, phic, axc, ayc);
    // the forward's step matrix of this mode (mc.dirkm, built once from the stage
    // recurrence on unit inputs): the step is that linear map, so its transpose is exact
    double M[2][4];
    const double* Mf = mc.dirkm + (size_t)idx * 8;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        M[0][k] = __ldg(Mf + k);
        M[1][k] = __ldg(Mf + 4 + k);
    }
    const zd phiu = L(dp.phi) + phic, phiv = L(dp.vphi);
    const zd axu = L(dp.ax) + axc, axv = L(dp.vax);
    const zd ayu = L(dp.ay) + ayc, ayv = L(dp.vay);
    // transpose: input i gets M[0][i] u_bar' + M[1][i] v_bar'
    S(dp.phi, M[0][0] * phiu + M[1][0] * phiv);
    S(dp.vphi, M[0][1] * phiu + M[1][1] * phiv);
    S(dp.ax, M[0][0] * axu + M[1][0] * axv);
    S(dp.vax, M[0][1] * axu + M[1][1] * axv);
    S(dp.ay, M[0][0] * ayu + M[1][0] * ayv);
    S(dp.vay, M[0][1] * ayu + M[1][1] * ayv);
    // phi's sources rho^n/eps0 and rho^{n+1}/eps0; A's mu0 J^n and mu0 J^{n+1}
    const zd rhon = L(dp.rho) + (M[0][3] / mc.eps0) * phiu + (M[1][3] / mc.eps0) * phiv;
    // rho^{n+1} = rho^n - dt (r0 i k . J^n + r1 i k . J^{n+1})
    S(dp.rho, rhon + (M[0][2] / mc.eps0) * phiu + (M[1][2] / mc.eps0) * phiv);
    const double dt = mc.dt;
    const zd jxn = L(dp.jx) + mc.mu0 * (M[0][3] * axu + M[1][3] * axv) + zi(dt * dp.r1 * kx * rhon);
    const zd jyn = L(dp.jy) + mc.mu0 * (M[0][3] * ayu + M[1][3] * ayv) + zi(dt * dp.r1 * ky * rhon);
    S(dp.jx, mc.mu0 * (M[0][2] * axu + M[1][2] * axv) + zi(dt * dp.r0 * kx * rhon));
    S(dp.jy, mc.mu0 * (M[0][2] * ayu + M[1][2] * ayv) + zi(dt * dp.r0 * ky * rhon));
    return mc.jscale * (jxn + zi(jyn));
}

// One thread per mode over the transformed planes Zb (four planes of nx ny).
template <typename Params>
__global__ void __launch_bounds__(kModeThreads)
k_adj_modes(ModeCommon mc, Params ap, const double2* __restrict__ Zb, double2* __restrict__ Js) {
    const int ng = mc.nx * mc.ny;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= ng) return;
    const int i = idx / mc.ny, j = idx - i * mc.ny;
    const int ip = (i == 0) ? 0 : mc.nx - i;
    const int jp = (j == 0) ? 0 : mc.ny - j;
    const int idm = ip * mc.ny + jp;
    zd za[4], zb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        za[k] = zl(Zb + (size_t)k * ng + idx);
        zb[k] = zl(Zb + (size_t)k * ng + idm);
    }
    zs(Js + idx, adj_mode(mc, ap, idx, mc.kxt[i], mc.kyt[j], za, zb));
}

// Fused column pass of the reverse field step.  CTA j loads columns j and ny - j (mod ny)
// of the four row-transformed planes, transforms them along x in shared memory, updates
// the modes of column j and transforms column j of the adjoint current back along x;
// the caller finishes with the inverse transform along y.
template <typename Params>
__global__ void __launch_bounds__(kModeThreads)
k_adj_columns(ModeCommon mc, Params ap, const double2* __restrict__ Zb,
              double2* __restrict__ Js, FftDesc fd, const double2* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = mc.nx, ny = mc.ny;
    const size_t ng = (size_t)nx * ny;
    const int j = blockIdx.x;
    const int jp = (j == 0) ? 0 : ny - j;
    const int ncols = (jp == j) ? 1 : 2;
    double2* bufA = reinterpret_cast<double2*>(smem_raw);  // 8 lines of nx: line c*4 + k
    double2* bufB = bufA + 8 * nx;
    double2* tws = bufB + 8 * nx;
    stage_twiddles(tw, tws, nx);
    griddep_wait();
    griddep_launch();
    for (int t = threadIdx.x; t < 4 * ncols * nx; t += blockDim.x) {
        const int l = t / nx, i = t - l * nx;
        const int c = l >> 2, k = l & 3;
        bufA[t] = Zb[k * ng + (size_t)i * ny + (c ? jp : j)];
    }
    __syncthreads();
    double2* zc = run_passes(bufA, bufB, fd, 4 * ncols, (const double2*)tws, -1);
    double2* out = (zc == bufA) ? bufB : bufA;
    const double2* zp = zc + (size_t)(ncols - 1) * 4 * nx;
    const double ky = mc.kyt[j];
    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
        const int ip = (i == 0) ? 0 : nx - i;
        zd za[4], zb[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            za[k] = zl(zc + k * nx + i);
            zb[k] = zl(zp + k * nx + ip);
        }
        zs(out + i, adj_mode(mc, ap, i * ny + j, mc.kxt[i], ky, za, zb));
    }
    __syncthreads();
    double2* res = run_passes(out, zc, fd, 1, (const double2*)tws, +1);
    for (int i = threadIdx.x; i < nx; i += blockDim.x) Js[(size_t)i * ny + j] = res[i];
}

// Final-level seed of an objective sum bzb B_z: B_z = IDFT(i kx Ay - i ky Ax), so
// Ay b += -i kx DFT(bzb)/N and Ax b += i ky DFT(bzb)/N.
__global__ void __launch_bounds__(kModeThreads)
k_adj_seed(ModeCommon mc, const double2* __restrict__ zs_, double2* __restrict__ ax,
           double2* __restrict__ ay) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= mc.nx * mc.ny) return;
    const int i = idx / mc.ny, j = idx - i * mc.ny;
    const double kx = mc.kxt[i], ky = mc.kyt[j];
    const zd z = mc.inv_n * zl(zs_ + idx);
    zs(ay + idx, zl(ay + idx) - zi(kx * z));
    zs(ax + idx, zl(ax + idx) + zi(ky * z));
}

// (Ex + i Ey)/(nx ny) of E = -grad phi, for an inverse transform to the mesh E^0.
__global__ void __launch_bounds__(kModeThreads)
k_adj_e0(ModeCommon mc, const double2* __restrict__ phi, double2* __restrict__ out) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= mc.nx * mc.ny) return;
    const int i = idx / mc.ny, j = idx - i * mc.ny;
    const double kx = mc.kxt[i], ky = mc.kyt[j];
    const zd ph = zl(phi + idx);
    const zd ex = -zi(kx * ph), ey = -zi(ky * ph);
    zs(out + idx, mc.inv_n * (ex + zi(ey)));
}

// dst[k n + i] = src.p[k][i] (pack) or dst.p[k][i] = src[k n + i] (unpack), k = blockIdx.y.
template <typename T>
__global__ void k_pack8(Ptr8T<T> src, T* __restrict__ dst, int64_t n) {
    const T* s = src.p[blockIdx.y];
    T* d = dst + (size_t)blockIdx.y * n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        d[i] = s[i];
}
template <typename T>
__global__ void k_unpack8(const T* __restrict__ src, Ptr8T<T> dst, int64_t n) {
    const T* s = src + (size_t)blockIdx.y * n;
    T* d = const_cast<T*>(dst.p[blockIdx.y]);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        d[i] = s[i];
}

__global__ void k_real_to_cplx(const double* __restrict__ src, double2* __restrict__ dst,
                               int64_t n) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x)
        dst[p] = make_double2(src[p], 0.0);
}

// t = 0: P^0 = gamma m v^0 and v^{-1} = v^0 - kappa (E - v (v . E)/c^2), kappa =
// dt q/(gamma m), E = E^0 gathered at x^0.  Gradient with respect to v^0 (gv) and, with
// P^0 as the independent variable, with respect to P^0 (gp = (dv/dP)^T gv).
template <typename T, int P>
__global__ void __launch_bounds__(kThreads)
k_adj_init(ParticleGeom g, PushParams pp, const T* __restrict__ x0, const T* __restrict__ y0,
           const T* __restrict__ vx0, const T* __restrict__ vy0, const double2* __restrict__ E,
           AdjParticlesT<T> ab, double* __restrict__ gvx, double* __restrict__ gvy,
           double* __restrict__ gpx, double* __restrict__ gpy, int64_t n,
           unsigned int* __restrict__ err) {
    const T c2 = (T)(pp.c * pp.c), m = (T)pp.m;
    const T idx_ = (T)g.inv_dx, idy = (T)g.inv_dy;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const T xi = x0[p] * idx_, yj = y0[p] * idy;
        if (!inside(xi, g.nx) || !inside(yj, g.ny)) {
            atomicOr(err, (unsigned)ERR_NONFINITE);
            continue;
        }
        T wx[P + 1], wy[P + 1];
        const int ix = Shape<P, T>::weights(xi, wx);
        const int iy = Shape<P, T>::weights(yj, wy);
        T ex = 0, ey = 0;
#pragma unroll
        for (int a = 0; a <= P; ++a) {
            const size_t row = (size_t)wrap_idx(ix + a, g.nx) * g.ny;
#pragma unroll
            for (int b = 0; b <= P; ++b) {
                const double2 e = E[row + wrap_idx(iy + b, g.ny)];
                const T w = wx[a] * wy[b];
                ex += w * (T)e.x;
                ey += w * (T)e.y;
            }
        }
        const T vx = vx0[p], vy = vy0[p];
        const T gam = (T)1 / sqrt((T)1 - (vx * vx + vy * vy) / c2);
        // dP/dv = gamma m (I + gamma^2 v v^T / c^2)
        const T pbx = ab.px[p], pby = ab.py[p];
        const T pvb = vx * pbx + vy * pby;
        T gx = ab.vx[p] + gam * m * (pbx + gam * gam * vx * pvb / c2);
        T gy = ab.vy[p] + gam * m * (pby + gam * gam * vy * pvb / c2);
        // v^{-1}: transpose of I + kappa gamma^2 T v^T / c^2 + kappa (v E^T + (v.E) I)/c^2
        const T wxb = ab.vxo[p], wyb = ab.vyo[p];
        const T kap = (T)(pp.dt * pp.q) / (gam * m);
        const T vde = vx * ex + vy * ey;
        const T tx = ex - vx * vde / c2, ty = ey - vy * vde / c2;
        const T tw = tx * wxb + ty * wyb, vw = vx * wxb + vy * wyb;
        gx += wxb + kap * gam * gam * vx * tw / c2 + (kap / c2) * (ex * vw + vde * wxb);
        gy += wyb + kap * gam * gam * vy * tw / c2 + (kap / c2) * (ey * vw + vde * wyb);
        if (gvx) gvx[p] = (double)gx;
        if (gvy) gvy[p] = (double)gy;
        // dv/dP = (I - v v^T / c^2) / (gamma m)
        const T vg = vx * gx + vy * gy;
        if (gpx) gpx[p] = (double)((gx - vx * vg / c2) / (gam * m));
        if (gpy) gpy[p] = (double)((gy - vy * vg / c2) / (gam * m));
    }
}

inline int mode_blocks(const ModeCommon& mc) {
    return (mc.nx * mc.ny + kModeThreads - 1) / kModeThreads;
}

}  // namespace

#define GPIC_ADJ_DISPATCH(p, KERNEL, ...)                                                  \
    switch (p) {                                                                         \
        case 2: KERNEL<T, 2><<<blocks_for(n), kThreads, 0, s>>>(__VA_ARGS__); break;    \
        case 3: KERNEL<T, 3><<<blocks_for(n), kThreads, 0, s>>>(__VA_ARGS__); break;    \
        case 4: KERNEL<T, 4><<<blocks_for(n), kThreads, 0, s>>>(__VA_ARGS__); break;    \
        default: return cudaErrorInvalidValue;                                          \
    }

inline unsigned adj_blocks(int64_t n) { return (unsigned)((n + kAdjThreads - 1) / kAdjThreads); }

template <typename T>
cudaError_t launch_adj_push_gather(int p, const ParticleGeom& g, const PushParams& pp,
                                   const T* x1, const T* y1, const T* px1, const T* py1,
                                   const T* vx, const T* vy, const T* vxo, const T* vyo,
                                   const double* gf, bool lean, const void* F,
                                   const FixFields* fix, AdjParticlesT<T> ab, T* Fb, int64_t n,
                                   unsigned int* err, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const double* gfa = lean ? nullptr : gf + 4 * n;  // the gathered values of the record
    const dim3 grid(adj_blocks(n)), block(kAdjThreads);
    if constexpr (sizeof(T) == 8) {
        if (fix) {
#define GPIC_ADJ_FIX(PP, LEAN)                                                                 \
    launch_pdl(k_adj_push_gather_fix<PP, LEAN>, grid, block, 0, s, g, fix_geom(g), pp, x1, y1, \
               px1, py1, vx, vy, vxo, vyo, gfa, (const int4*)fix->f,                           \
               (const int*)fix->exp, ab, Fb, n, err)
            switch (2 * p + (lean ? 1 : 0)) {
                case 4: return GPIC_ADJ_FIX(2, false);
                case 5: return GPIC_ADJ_FIX(2, true);
                case 6: return GPIC_ADJ_FIX(3, false);
                case 7: return GPIC_ADJ_FIX(3, true);
                case 8: return GPIC_ADJ_FIX(4, false);
                case 9: return GPIC_ADJ_FIX(4, true);
                default: return cudaErrorInvalidValue;
            }
#undef GPIC_ADJ_FIX
        }
    }
#define GPIC_ADJ_PUSH(KERNEL, FIELDS, SUMS)                                                    \
    launch_pdl(KERNEL, grid, block, 0, s, g, pp, x1, y1, px1, py1, vx, vy, vxo, vyo, gfa,      \
               (const FIELDS*)F, ab, (SUMS*)Fb, n, err)
    if constexpr (sizeof(T) == 4) {
        switch (p) {
            case 2: return GPIC_ADJ_PUSH(k_adj_push_gather_pair<2>, float4, float4);
            case 3: return GPIC_ADJ_PUSH(k_adj_push_gather_pair<3>, float4, float4);
            case 4: return GPIC_ADJ_PUSH(k_adj_push_gather_pair<4>, float4, float4);
            default: return cudaErrorInvalidValue;
        }
    } else {
        switch (p) {
            case 2: return GPIC_ADJ_PUSH(k_adj_push_gather<2>, double2, double);
            case 3: return GPIC_ADJ_PUSH(k_adj_push_gather<3>, double2, double);
            case 4: return GPIC_ADJ_PUSH(k_adj_push_gather<4>, double2, double);
            default: return cudaErrorInvalidValue;
        }
    }
#undef GPIC_ADJ_PUSH
}

template <typename T>
cudaError_t launch_adj_deposit_move(int p, const ParticleGeom& g, const T* x1, const T* y1,
                                    const T* vx, const T* vy, const double2* Jb,
                                    const FixFields* fix, AdjParticlesT<T> ab, int64_t n,
                                    unsigned int* err, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        if (fix) {
#define GPIC_ADJ_MOVE(PP)                                                                       \
    launch_pdl(k_adj_deposit_move_fix<PP>, dim3(adj_blocks(n)), dim3(kAdjThreads), 0, s, g,     \
               fix_geom(g), x1, y1, vx, vy, (const int4*)fix->f, (const int*)fix->exp, ab, \
               n, err)
            switch (p) {
                case 2: return GPIC_ADJ_MOVE(2);
                case 3: return GPIC_ADJ_MOVE(3);
                case 4: return GPIC_ADJ_MOVE(4);
                default: return cudaErrorInvalidValue;
            }
#undef GPIC_ADJ_MOVE
        }
    }
#define GPIC_ADJ_MOVE(PP)                                                                    \
    launch_pdl(k_adj_deposit_move<T, PP>, dim3(blocks_for(n)), dim3(kThreads), 0, s, g, x1, y1, \
               vx, vy, Jb, ab, n, err)
    switch (p) {
        case 2: return GPIC_ADJ_MOVE(2);
        case 3: return GPIC_ADJ_MOVE(3);
        case 4: return GPIC_ADJ_MOVE(4);
        default: return cudaErrorInvalidValue;
    }
#undef GPIC_ADJ_MOVE
}

template <typename T>
cudaError_t launch_adj_init(int p, const ParticleGeom& g, const PushParams& pp, const T* x0,
                            const T* y0, const T* vx0, const T* vy0, const double2* E,
                            AdjParticlesT<T> ab, double* gvx, double* gvy, double* gpx,
                            double* gpy, int64_t n, unsigned int* err, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    GPIC_ADJ_DISPATCH(p, k_adj_init, g, pp, x0, y0, vx0, vy0, E, ab, gvx, gvy, gpx, gpy, n, err)
    return cudaGetLastError();
}

template <typename Params>
cudaError_t adj_modes(const ModeCommon& mc, const Params& ap, const double2* Zb, double2* Js,
                      cudaStream_t s) {
    k_adj_modes<Params><<<mode_blocks(mc), kModeThreads, 0, s>>>(mc, ap, Zb, Js);
    return cudaGetLastError();
}

cudaError_t launch_adj_modes(const ModeCommon& mc, int kind, const AdjModeParams& ap,
                             const CdfParams& cp, const DirkParams& dp, const double2* Zb,
                             double2* Js, cudaStream_t s) {
    if (kind == K_CDF2) return adj_modes(mc, cp, Zb, Js, s);
    if (kind == K_DIRK) return adj_modes(mc, dp, Zb, Js, s);
    return adj_modes(mc, ap, Zb, Js, s);
}

constexpr size_t kSms = 152, kSmemPerSm = 228 * 1024;

size_t adj_columns_smem(int nx) { return 17 * (size_t)nx * sizeof(double2); }

template <typename Params>
cudaError_t adj_columns(const ModeCommon& mc, const Params& ap, const double2* Zb, double2* Js,
                        const FftDesc& fd, const double2* tw, cudaStream_t s) {
    // Shared memory for as many CTAs an SM as spread over the SMs need, not more: started early,
    // beside the row transform before them, the CTAs (62 registers a thread with BDF, so four an
    // SM) crowded on the SMs that it leaves free and waited for each other's FP64 pipe.  A reversed
    // BDF-2 step of 262,144 particles on 128 x 128: FP32 form 129 -> 122 us, FP64 217 -> 210;
    // with events around the launch group 75 us of it were the field solve, now 44.
    const size_t per_sm = (mc.ny + kSms - 1) / kSms;
    const size_t sm = std::max(adj_columns_smem(mc.nx), kSmemPerSm / (per_sm + 1));
    cudaError_t e = cudaFuncSetAttribute(k_adj_columns<Params>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_adj_columns<Params>, dim3(mc.ny), dim3(kModeThreads), sm, s, mc, ap, Zb, Js,
                      fd, tw);
}

cudaError_t launch_adj_columns(const ModeCommon& mc, int kind, const AdjModeParams& ap,
                               const CdfParams& cp, const DirkParams& dp, const double2* Zb,
                               double2* Js, const FftDesc& fd, const double2* tw,
                               cudaStream_t s) {
    if (kind == K_CDF2) return adj_columns(mc, cp, Zb, Js, fd, tw, s);
    if (kind == K_DIRK) return adj_columns(mc, dp, Zb, Js, fd, tw, s);
    return adj_columns(mc, ap, Zb, Js, fd, tw, s);
}

cudaError_t launch_adj_seed(const ModeCommon& mc, const double2* zs_, double2* ax, double2* ay,
                            cudaStream_t s) {
    k_adj_seed<<<mode_blocks(mc), kModeThreads, 0, s>>>(mc, zs_, ax, ay);
    return cudaGetLastError();
}

cudaError_t launch_adj_e0(const ModeCommon& mc, const double2* phi, double2* out, cudaStream_t s) {
    k_adj_e0<<<mode_blocks(mc), kModeThreads, 0, s>>>(mc, phi, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pack8(Ptr8T<T> src, T* dst, int64_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const int bx = (int)std::min<int64_t>((n + kThreads - 1) / kThreads, 152 * 2);
    k_pack8<T><<<dim3(bx, 8), kThreads, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_unpack8(const T* src, Ptr8T<T> dst, int64_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const int bx = (int)std::min<int64_t>((n + kThreads - 1) / kThreads, 152 * 2);
    k_unpack8<T><<<dim3(bx, 8), kThreads, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_real_to_cplx(const double* src, double2* dst, int64_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_real_to_cplx<<<blocks_for(n), kThreads, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}

#define GPIC_ADJ_INST(T)                                                                    \
    template cudaError_t launch_adj_push_gather<T>(                                         \
        int, const ParticleGeom&, const PushParams&, const T*, const T*, const T*, const T*, \
        const T*, const T*, const T*, const T*, const double*, bool, const void*,            \
        const FixFields*, AdjParticlesT<T>, T*, int64_t, unsigned int*, cudaStream_t);      \
    template cudaError_t launch_adj_deposit_move<T>(int, const ParticleGeom&, const T*,     \
                                                    const T*, const T*, const T*,           \
                                                    const double2*, const FixFields*,       \
                                                    AdjParticlesT<T>, int64_t,              \
                                                    unsigned int*, cudaStream_t);           \
    template cudaError_t launch_adj_init<T>(int, const ParticleGeom&, const PushParams&,    \
                                            const T*, const T*, const T*, const T*,         \
                                            const double2*, AdjParticlesT<T>, double*,      \
                                            double*, double*, double*, int64_t,             \
                                            unsigned int*, cudaStream_t);                   \
    template cudaError_t launch_pack8<T>(Ptr8T<T>, T*, int64_t, cudaStream_t);              \
    template cudaError_t launch_unpack8<T>(const T*, Ptr8T<T>, int64_t, cudaStream_t);
GPIC_ADJ_INST(double)
GPIC_ADJ_INST(float)
#undef GPIC_ADJ_INST

}  // namespace gpic
