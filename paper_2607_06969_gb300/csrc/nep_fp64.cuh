// Shared by the FP64 kernels and the generic FP32 evaluation: the pair
// geometry, the basis, and the split of an atom's work over a group of lanes.
//
// The operators of Section 3.2 run in float64 as well as float32.  This path
// computes Eqs. 1-4 and 11-21 with every intermediate in double: positions
// (FP32 inputs) are promoted, the parameters are FP64, and pairs are kept by
// r < rc in double.  Hyper-parameters are runtime values, unrolled loops have
// compiled bounds (Dims64).  The same code in float is the generic FP32
// evaluation of shapes without compiled kernels.
//
// A group of G lanes takes an atom (32 up to kEvalLanes32 atoms, or
// kGenericLanes32 in float, then 8).
// Sums over the list run pair by pair in list order within a lane's share, the
// few sums that cross lanes in an xor butterfly, whose fixed tree leaves the
// same bits in every lane; for a given N, which fixes G, every result is
// deterministic.
#pragma once
#include <algorithm>
#include <type_traits>

#include <cuda_runtime.h>

#include "nep_device.cuh"
#include "nep_internal.h"

namespace nep {
namespace {

constexpr double kPi = 3.141592653589793;

// The evaluation below is written once for two argument types: F64Args (every
// intermediate in double) and F32Args (the generic FP32 evaluation, any
// hyper-parameters within the same bounds).  R is the argument type's scalar.
template <class A>
struct ScalarOf;
template <>
struct ScalarOf<F64Args> {
    using type = double;
};
template <>
struct ScalarOf<F32Args> {
    using type = float;
};
template <class A>
using ScalarT = typename ScalarOf<A>::type;

__device__ __forceinline__ void sincospi_r(double z, double* s, double* c) { sincospi(z, s, c); }
__device__ __forceinline__ void sincospi_r(float z, float* s, float* c) { sincospif(z, s, c); }
__device__ __forceinline__ double tanh_r(double x) { return tanh(x); }
__device__ __forceinline__ float tanh_r(float x) { return tanhf(x); }
__device__ __forceinline__ double sqrt_r(double x) { return sqrt(x); }
__device__ __forceinline__ float sqrt_r(float x) { return sqrtf(x); }
__device__ __forceinline__ double rint_r(double x) { return rint(x); }
__device__ __forceinline__ float rint_r(float x) { return rintf(x); }

// sum over the warp; every lane receives the same bits
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <class R>
struct FrameT {
    int i, ti, b;
    R L[3], x, y, z;
};
using Frame64 = FrameT<double>;
template <class A>
__device__ FrameT<ScalarT<A>> frame64(const A& a, int i) {
    FrameT<ScalarT<A>> fr;
    fr.i = i;
    fr.ti = a.type[i];
    fr.b = a.cfg[i];
    for (int c = 0; c < 3; ++c) fr.L[c] = a.box[3 * fr.b + c];
    fr.x = a.pos[i];
    fr.y = a.pos[a.N + i];
    fr.z = a.pos[2 * a.N + i];
    return fr;
}

// list slot s of atom fr.i: r_ij = (r_j - r_i) + s L in R, with the list's
// image or the minimum image; false when r >= rc_rad
template <class R>
struct PairT {
    int j, tj;
    R d[3], r, ir, u[3];
};
using Pair64 = PairT<double>;
template <class A, class R>
__device__ bool pair_at(const A& a, const FrameT<R>& fr, int s, PairT<R>& p) {
    const int N = a.N;
    p.j = a.nbr[(size_t)s * N + fr.i];
    const R ux = (R)a.pos[p.j] - fr.x, uy = (R)a.pos[N + p.j] - fr.y, uz = (R)a.pos[2 * N + p.j] - fr.z;
    R sx, sy, sz;
    if (a.shift) {
        int ix, iy, iz;
        unpack_shift(a.shift[(size_t)s * N + fr.i], ix, iy, iz);
        sx = (R)ix; sy = (R)iy; sz = (R)iz;
    } else {
        sx = -rint_r(ux / fr.L[0]);
        sy = -rint_r(uy / fr.L[1]);
        sz = -rint_r(uz / fr.L[2]);
    }
    // explicit FMAs: every kernel gets the same r for a pair, seen from either
    // atom (the scatter of the generic path relies on it)
    p.d[0] = fma_r(sx, fr.L[0], ux);
    p.d[1] = fma_r(sy, fr.L[1], uy);
    p.d[2] = fma_r(sz, fr.L[2], uz);
    p.r = sqrt_r(fma_r(p.d[2], p.d[2], fma_r(p.d[1], p.d[1], p.d[0] * p.d[0])));
    if (!(p.r < a.rc_rad)) return false;
    p.tj = a.type[p.j];
    p.ir = R(1.0) / p.r;
    for (int c = 0; c < 3; ++c) p.u[c] = p.d[c] * p.ir;
    return true;
}

// ------------------------------------------------------------ lane groups
// A group of G lanes per atom; the lanes take the list entries, then the
// harmonics m, the hidden units and the descriptors in turn, and hand results
// over in shared memory (sizes below in scalars).  In double the FP64 pipe
// bounds both kernels: a warp instruction occupies it for 16 cycles per SM
// whatever lanes are active, so the split is chosen for active lanes.  G = 8
// keeps nearly all of them busy (72 list entries, 24 harmonics, 30 hidden
// units); G = 32 gives a few hundred atoms four times the warps.
constexpr int kGroupTile = 32;   // hidden units at a time
// One warp per CTA: the FP64 pipe of an SM is the limit, and whole warps spread
// evenest over the SMs (2,593 atoms in CTAs of 4 warps: 163 CTAs on 152 SMs, the
// pipe 85% busy where there was work but 48% of the time).
constexpr int kF64Threads = 32;
template <int G>
struct Group64 {
    static constexpr int NG = kF64Threads / G, GS = G + 1;
    static constexpr int MPL = (kLM + G - 1) / G;              // harmonics per lane
    static constexpr int KW = G < kF64MaxK ? G : kF64MaxK;     // lanes that sum a basis function each
    static constexpr int KX = kF64MaxK / KW, PARTS = G / KW;
    int NAs, oG, oY, oT, oS, oF, oQ, oP, oJ, oSg, size;
    __host__ __device__ Group64(int T, int NA, int KR, int D) {
        NAs = NA | 1;
        oG = 0;                                // [G][NAs] g_n of a chunk's pairs
        oY = oG + G * NAs;                     // [24][GS] basis values, or harmonics, of them
        oQ = oY;                               // q, p, J and the hidden tile once the sums are done
        oP = oQ + D;
        oJ = oP + D;
        oSg = oJ + 5 * NA;
        const int endY = oY + kLM * GS, endQ = oSg + kGroupTile;
        oT = endY > endQ ? endY : endQ;        // [G] species of a chunk's pairs
        oS = oT + G;                           // [NA][24]
        oF = oS + NA * kLM;                    // [T][KR]
        size = oF + T * KR;
    }
};

// Bounds of a kernel's unrolled loops: n_ang <= NAX, k_rad and k_ang <= KX.
// EX: the model's values are the bounds (the compiled models' 6 or 8 by 8),
// so no operation is issued for an n or k past them; the FP64 pipe is busy for
// a predicated-off operation too.
template <int NAX_, int KX_, bool EX>
struct Dims64 {
    static constexpr int NAX = NAX_, KX = KX_;
    template <class A>
    static __device__ __forceinline__ int NA(const A& a) { return EX ? NAX : a.NA; }
    template <class A>
    static __device__ __forceinline__ int KA(const A& a) { return EX ? KX : a.KA; }
    template <class A>
    static __device__ __forceinline__ int KR(const A& a) { return EX ? KX : a.KR; }
};

__device__ __forceinline__ int warp_max_i(int v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ double cospi_r(double z) { return cospi(z); }
__device__ __forceinline__ float cospi_r(float z) { return cospif(z); }

// A cutoff, and x / rc.  In float the product with the rounded 1 / rc is off by
// the same fraction for every pair, up to 6e-8, which energies and virials add
// up instead of averaging out; one correction by the residual takes that away.
// Virial against 64 bits, 9,956 atoms: 11/7 functions and two species 1.5e-6
// without and 2.7e-7 with it, 5/3 functions 5.9e-7 and 6.7e-8 (134.1 / 134.9 us).
template <class R>
struct Cutoff {
    R rc, inv;
    __device__ explicit Cutoff(R c) : rc(c), inv(R(1.0) / c) {}
    __device__ __forceinline__ R over(R x) const {
        const R q = x * inv;
        if constexpr (std::is_same<R, float>::value) return fmaf(fmaf(-q, rc, x), inv, q);
        return q;
    }
};

// out(k, Q_k(r)) for k < K (Eqs. 12-15)
template <int KX, class R, class Out>
__device__ __forceinline__ void basis_values(R r, const Cutoff<R>& cut, int K, Out out) {
    const R z = cut.over(r), fc2 = R(0.25) * (R(1.0) + cospi_r(z)), t = z - R(1.0), x = R(2.0) * t * t - R(1.0);
    R Tm = R(1.0), Tk = x;
    out(0, R(2.0) * fc2);
    if (K > 1) out(1, (x + R(1.0)) * fc2);
#pragma unroll
    for (int k = 2; k < KX; ++k) {
        if (k >= K) break;
        const R Tn = R(2.0) * x * Tk - Tm;
        out(k, (Tn + R(1.0)) * fc2);
        Tm = Tk;
        Tk = Tn;
    }
}
// out(k, Q_k(r), dQ_k/dr) for k < K
template <int KX, class R, class Out>
__device__ __forceinline__ void basis_derivs(R r, const Cutoff<R>& cut, int K, Out out) {
    const R z = cut.over(r);
    R sp, cp;
    sincospi_r(z, &sp, &cp);
    const R fc2 = R(0.25) * (R(1.0) + cp), dfc2 = cut.over(R(-0.25 * kPi)) * sp;
    const R t = z - R(1.0), x = R(2.0) * t * t - R(1.0), a = cut.over(R(4.0) * t) * fc2;
    R Tm = R(1.0), Tk = x, dTm = R(0.0), dTk = R(1.0);
    out(0, R(2.0) * fc2, R(2.0) * dfc2);
    if (K > 1) out(1, (x + R(1.0)) * fc2, a + (x + R(1.0)) * dfc2);
#pragma unroll
    for (int k = 2; k < KX; ++k) {
        if (k >= K) break;
        const R Tn = R(2.0) * x * Tk - Tm;
        const R dTn = R(2.0) * (Tk + x * dTk) - dTm;
        out(k, (Tn + R(1.0)) * fc2, dTn * a + (Tn + R(1.0)) * dfc2);
        Tm = Tk; Tk = Tn; dTm = dTk; dTk = dTn;
    }
}

// Whether the angular force of a pair is computed by one of its atoms and
// handed to the other through the list's reverse slots (the generic path,
// whose workspace has the slots).  The FP64 path's workspace does not depend
// on the list's capacity: it computes both sides of a pair at both atoms.
template <class A>
constexpr bool kScatter = std::is_same<A, F32Args>::value;

// Up to this many atoms the kernels take 32 lanes per atom, else 8.  Packings in
// a graph, 32 / 8 lanes, evaluation and loss gradient:
//   38-30-1: 1,300 atoms 232 / 280 us, 516 / 652; 1,600 241 / 287, 562 / 664;
//     2,000 311 / 289, 779 / 672
//   52-64-1: 1,600 290 / 382, 757 / 900; 2,000 369 / 383, 952 / 908; 2,600
//     465 / 438, 1,139 / 1,052
//   11/7 radial/angular functions, 2 species: 1,300 370 / 430, 873 / 962; 1,600
//     433 / 333, 1,031 / 770
//   5/3 functions: 1,000 154 / 259, 388 / 572; 1,300 258 / 259, 593 / 574; 1,600
//     294 / 266, 714 / 582
// so the line lies in the middle of where the shapes cross, 1,300 to 2,000.
constexpr int kEvalLanes32 = 1500;
// the same for the generic path, whose pipe is not full at these sizes (32 / 8
// lanes, models of 11/7 and 5/3 radial/angular functions): 2,566 atoms 57.4 /
// 74.3 us, 60.1 / 70.2; 5,453 atoms 89.7 / 83.0, 89.1 / 74.7
constexpr int kGenericLanes32 = 4000;

// calls f with the loop bounds for the model's shape
template <class A, class F>
cudaError_t with_dims(const A& a, F f) {
    const int K = std::max(a.KR, a.KA);
    if constexpr (!kScatter<A>) {
        if (a.KR == 8 && a.KA == 8 && a.NA == 6) return f(Dims64<6, 8, true>{});
        if (a.KR == 8 && a.KA == 8 && a.NA == 8) return f(Dims64<8, 8, true>{});
    }
    if (a.NA <= 8 && K <= 8) return f(Dims64<8, 8, false>{});
    if constexpr (kScatter<A>)
        if (a.NA <= 8 && K <= 12) return f(Dims64<8, 12, false>{});
    return f(Dims64<16, 16, false>{});
}

}  // namespace
}  // namespace nep
