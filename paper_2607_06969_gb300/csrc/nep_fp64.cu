// FP64 evaluation of energies, forces and virial, the generic FP32 evaluation
// (the same kernels in float) and the FP64 loss.  Two passes over the list:
//   k64_atom  : the species-resolved radial basis sums F[t][k] and q_n
//               (Eq. 11), S_nlm and q_nl (Eqs. 16-17), q4_n, the network
//               (Eq. 2), E_i, the radial adjoint per neighbour species and
//               R_nlm = dE_i/dS_nlm
//   k64_force : F_i = sum_j [dE_i/dr_ij - dE_j/dr_ji] (Eq. 3) and the per-atom
//               virial (Eq. 4)
// then FP64 sums per 1,024-atom chunk and per configuration in a fixed order.
//
// Measured (38-30-1 model): FP64, 2,593 atoms 1,319 -> 382 us against one or
// more lanes per atom with runtime-indexed arrays and both sides of a pair
// evaluated apart; k64_force keeps the FP64 pipe, which bounds both kernels,
// busy 85% of the cycles.  Generic, 9,956 atoms of a two-species model 605 -> 136 us.
#include "nep_fp64.cuh"

namespace nep {
namespace {

__global__ void k_promote(const float* src, double* dst, int n) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < n) dst[x] = (double)src[x];
}

// Radial sums F and S_nlm of atom fr.i into the group's block; lane keeps
// S[n][x] of harmonic lane + x G.  NAX bounds n_ang.
template <int G, class DM, class A, class R>
__device__ void group64_sums(const A& a, const Group64<G>& o, R* gb, const FrameT<R>& fr, int nc, int lane,
                             R (&S)[DM::NAX][Group64<G>::MPL]) {
    constexpr int NAX = DM::NAX;
    constexpr int GS = Group64<G>::GS, MPL = Group64<G>::MPL, KW = Group64<G>::KW, KX = Group64<G>::KX;
    constexpr int PARTS = Group64<G>::PARTS;
    const int NA = DM::NA(a), KR = DM::KR(a), KA = DM::KA(a);
    const Cutoff<R> cutR((R)a.rc_rad), cutA((R)a.rc_ang);
    int* tj = reinterpret_cast<int*>(gb + o.oT);
    const int gbase = (threadIdx.x & 31) & ~(G - 1);
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u), below = (1u << lane) - 1u;
    const int kl = lane % KW, part = lane / KW;
    R F[KX][kMaxTypes];
#pragma unroll
    for (int x = 0; x < KX; ++x)
#pragma unroll
        for (int t = 0; t < kMaxTypes; ++t) F[x][t] = R(0.0);
#pragma unroll
    for (int n = 0; n < NAX; ++n)
#pragma unroll
        for (int x = 0; x < MPL; ++x) S[n][x] = R(0.0);
    const int cmax = warp_max_i(nc);
    for (int s0 = 0; s0 < cmax; s0 += G) {
        const int s = s0 + lane;
        PairT<R> p;
        const bool in = s < nc && pair_at(a, fr, s, p);
        const unsigned mi = (__ballot_sync(0xffffffffu, in) >> gbase) & gmask;
        const int ni = __popc(mi), ati = __popc(mi & below);
        if (in) {
            tj[ati] = p.tj;
            basis_values<DM::KX>(p.r, cutR, KR, [&](int k, R f) { gb[o.oY + k * GS + ati] = f; });
        }
        __syncwarp();
        for (int q = part; q < ni; q += PARTS) {
            const int t = tj[q];
#pragma unroll
            for (int x = 0; x < KX; ++x) {
                const int k = kl + x * KW;
                if (k >= KR) continue;
                const R f = gb[o.oY + k * GS + q];
#pragma unroll
                for (int u = 0; u < kMaxTypes; ++u)
                    if (t == u) F[x][u] += f;
            }
        }
        __syncwarp();
        const bool ang = in && p.r < (R)a.rc_ang;
        const unsigned any = __ballot_sync(0xffffffffu, ang);
        if (!any) continue;
        const unsigned ma = (any >> gbase) & gmask;
        const int na = __popc(ma), at = __popc(ma & below);
        if (ang) {
            R f[DM::KX];
            basis_values<DM::KX>(p.r, cutA, KA, [&](int k, R v) { f[k] = v; });
            const R* c = a.prm + a.L.off_cA + (size_t)(fr.ti * a.T + p.tj) * NA * KA;
#pragma unroll
            for (int n = 0; n < NAX; ++n) {
                if (n >= NA) break;
                R g = R(0.0);
#pragma unroll
                for (int k = 0; k < DM::KX; ++k)
                    if (k < KA) g += c[n * KA + k] * f[k];
                gb[o.oG + at * o.NAs + n] = g;
            }
            const Harm<R> ht = harm_of(p.u[0], p.u[1], p.u[2]);
#pragma unroll
            for (int m = 0; m < kLM; ++m) gb[o.oY + m * GS + at] = harm_value(m, ht);
        }
        __syncwarp();
        for (int q = 0; q < na; ++q) {
#pragma unroll
            for (int x = 0; x < MPL; ++x) {
                const int m = lane + x * G;
                if (m >= kLM) continue;
                const R Y = gb[o.oY + m * GS + q];
#pragma unroll
                for (int n = 0; n < NAX; ++n)
                    if (n < NA) S[n][x] += gb[o.oG + q * o.NAs + n] * Y;
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int x = 0; x < KX; ++x)
#pragma unroll
        for (int t = 0; t < kMaxTypes; ++t) {
            R v = F[x][t];
#pragma unroll
            for (int h = KW; h < G; h <<= 1) v += __shfl_xor_sync(0xffffffffu, v, h);
            if (part == 0 && kl + x * KW < KR && t < a.T) gb[o.oF + t * KR + kl + x * KW] = v;
        }
#pragma unroll
    for (int n = 0; n < NAX; ++n)
#pragma unroll
        for (int x = 0; x < MPL; ++x)
            if (n < NA && lane + x * G < kLM) gb[o.oS + n * kLM + lane + x * G] = S[n][x];
    __syncwarp();
}

// q and the 4-body gradients J, then E_i (returned in every lane) and
// p = dE/dq, in the group's block
template <int G, class A, class R>
__device__ R group64_network(const A& a, const Group64<G>& o, R* gb, int ti, int lane) {
    const int T = a.T, NR = a.NR, NA = a.NA, KR = a.KR, H = a.H, D = a.D;
    const R* cR = a.prm + a.L.off_cR + (size_t)ti * T * NR * KR;
    for (int n = lane; n < NR; n += G) {
        R v = R(0.0);
        for (int t = 0; t < T; ++t)
            for (int k = 0; k < KR; ++k) v += cR[(t * NR + n) * KR + k] * gb[o.oF + t * KR + k];
        gb[o.oQ + n] = v;
    }
    for (int x = lane; x < NA * 4; x += G) {
        const int n = x >> 2, l = x & 3, m0 = l * (l + 2);
        R v = R(0.0);
        for (int m = m0; m < m0 + 2 * l + 3; ++m) {
            const R s = gb[o.oS + n * kLM + m];
            v += (R)clm(m) * s * s;
        }
        gb[o.oQ + NR + x] = v;
    }
    if (a.H4)
        for (int n = lane; n < NA; n += G) gb[o.oQ + NR + NA * 4 + n] = fourbody<R>(gb + o.oS + n * kLM + 3, gb + o.oJ + 5 * n);
    for (int d = lane; d < D; d += G) gb[o.oP + d] = R(0.0);
    __syncwarp();
    const R* W0 = a.prm + (size_t)ti * a.L.mlp_stride;
    const R* b0 = W0 + (size_t)H * D;
    const R* w1 = b0 + H;
    R E = R(0.0);
    for (int h0 = 0; h0 < H; h0 += kGroupTile) {
        const int nh = min(kGroupTile, H - h0);
        for (int h = lane; h < nh; h += G) {
            const R* w = W0 + (size_t)(h0 + h) * D;
            R z0 = b0[h0 + h], z1 = R(0.0);
            int d = 0;
            for (; d + 1 < D; d += 2) {
                z0 += w[d] * gb[o.oQ + d];
                z1 += w[d + 1] * gb[o.oQ + d + 1];
            }
            if (d < D) z0 += w[d] * gb[o.oQ + d];
            const R th = tanh_r(z0 + z1), wh = w1[h0 + h];
            E += wh * th;
            gb[o.oSg + h] = wh * (R(1.0) - th * th);
        }
        __syncwarp();
        for (int d = lane; d < D; d += G) {
            const R* w = W0 + (size_t)h0 * D + d;
            R p0 = gb[o.oP + d], p1 = R(0.0);
            int h = 0;
            for (; h + 1 < nh; h += 2) {
                p0 += gb[o.oSg + h] * w[(size_t)h * D];
                p1 += gb[o.oSg + h + 1] * w[(size_t)(h + 1) * D];
            }
            if (h < nh) p0 += gb[o.oSg + h] * w[(size_t)h * D];
            gb[o.oP + d] = p0 + p1;
        }
        __syncwarp();
    }
#pragma unroll
    for (int h = G / 2; h > 0; h >>= 1) E += __shfl_xor_sync(0xffffffffu, E, h);
    return E + w1[H];
}

// g_n = sum_k c[n][k] Q_k and g'_n with Q'_k, c = cA[ti][tj]
template <class DM, class A, class R>
__device__ __forceinline__ void angular_g(const A& a, int ti, int tj, R r, const Cutoff<R>& cutA, int NA, int KA, R* g, R* gp) {
    R f[DM::KX], fp[DM::KX];
    basis_derivs<DM::KX>(r, cutA, KA, [&](int k, R v, R d) {
        f[k] = v;
        fp[k] = d;
    });
    const R* c = a.prm + a.L.off_cA + (size_t)(ti * a.T + tj) * NA * KA;
#pragma unroll
    for (int n = 0; n < DM::NAX; ++n) {
        g[n] = gp[n] = R(0.0);
        if (n >= NA) continue;
#pragma unroll
        for (int k = 0; k < DM::KX; ++k)
            if (k < KA) {
                g[n] += c[n * KA + k] * f[k];
                gp[n] += c[n * KA + k] * fp[k];
            }
    }
}

// the same for both orders of the pair: (g, g') from cA[ti][tj], (h, h') from cA[tj][ti]
template <class DM, class A, class R>
__device__ __forceinline__ void angular_g2(const A& a, int ti, int tj, R r, const Cutoff<R>& cutA, int NA, int KA, R* g, R* gp, R* h,
                                           R* hp) {
    R f[DM::KX], fp[DM::KX];
    basis_derivs<DM::KX>(r, cutA, KA, [&](int k, R v, R d) {
        f[k] = v;
        fp[k] = d;
    });
    const R* cij = a.prm + a.L.off_cA + (size_t)(ti * a.T + tj) * NA * KA;
    const R* cji = a.prm + a.L.off_cA + (size_t)(tj * a.T + ti) * NA * KA;
#pragma unroll
    for (int n = 0; n < DM::NAX; ++n) {
        g[n] = gp[n] = h[n] = hp[n] = R(0.0);
        if (n >= NA) continue;
#pragma unroll
        for (int k = 0; k < DM::KX; ++k)
            if (k < KA) {
                g[n] += cij[n * KA + k] * f[k];
                gp[n] += cij[n * KA + k] * fp[k];
                h[n] += cji[n * KA + k] * f[k];
                hp[n] += cji[n * KA + k] * fp[k];
            }
    }
}

// a group's sums of an atom's force and virial, acc = (F, W), to memory
template <int G, class A, class R>
__device__ __forceinline__ void group_store(const A& a, const R* acc, int i, int lane, bool valid) {
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        R v = acc[c];
#pragma unroll
        for (int h = G / 2; h > 0; h >>= 1) v += __shfl_xor_sync(0xffffffffu, v, h);
        if (valid && lane == c % G) {
            if (c < 3) a.force[(size_t)c * a.N + i] = v;
            else a.w[(size_t)(c - 3) * a.N + i] = v;
        }
    }
}

template <int G, class DM, class A>
__global__ void __launch_bounds__(kF64Threads) k64_atom(const A a) {
    constexpr int NAX = DM::NAX;
    using R = ScalarT<A>;
    extern __shared__ double smem64[];
    const Group64<G> o(a.T, a.NA, a.KR, a.D);
    const int lane = threadIdx.x % G, group = threadIdx.x / G;
    R* gb = reinterpret_cast<R*>(smem64) + group * o.size;
    const int ia = blockIdx.x * Group64<G>::NG + group, N = a.N;
    const bool valid = ia < N;
    const int i = valid ? ia : N - 1;
    const FrameT<R> fr = frame64(a, i);
    R S[NAX][Group64<G>::MPL];
    group64_sums<G, DM>(a, o, gb, fr, valid ? a.cnt[i] : 0, lane, S);
    const R E = group64_network<G>(a, o, gb, fr.ti, lane);
    const int T = a.T, NR = a.NR, NA = DM::NA(a), KR = DM::KR(a);
    if (valid && lane == 0) a.e[i] = E;
    // P[t][k] = sum_n p_n cR[ti][t][n][k], the radial adjoint of a neighbour of species t
    const R* cR = a.prm + a.L.off_cR + (size_t)fr.ti * T * NR * KR;
    for (int x = lane; x < T * KR; x += G) {
        R v = R(0.0);
        for (int n = 0; n < NR; ++n) v += gb[o.oP + n] * cR[((x / KR) * NR + n) * KR + x % KR];
        if (valid) a.p[(size_t)i * T * KR + x] = v;
    }
    // R_nlm = dE/dq_nl 2 C_lm S_nlm (+ dE/dq4_n dq4_n/dS_n2m)
#pragma unroll
    for (int x = 0; x < Group64<G>::MPL; ++x) {
        const int m = lane + x * G;
        if (m >= kLM) continue;
        const int l = lm_l(m);
        const R c2 = R(2.0) * (R)clm(m);
#pragma unroll
        for (int n = 0; n < NAX; ++n) {
            if (n >= NA) continue;
            R v = c2 * gb[o.oP + NR + n * 4 + l - 1] * S[n][x];
            if (a.H4 && l == 2) v += gb[o.oP + NR + NA * 4 + n] * gb[o.oJ + 5 * n + m - 3];
            if constexpr (kScatter<A>) gb[o.oS + n * kLM + m] = v;
            else if (valid) a.R[((size_t)i * NA + n) * kLM + m] = v;
        }
    }
    if constexpr (kScatter<A>) {
        // the owner's angular pair forces, and each pair's to its reverse slot
        __syncwarp();
        const R* Ri = gb + o.oS;
        const Cutoff<R> cutA((R)a.rc_ang);
        const int KA = DM::KA(a);
        R acc[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) acc[c] = R(0.0);
        const int na = valid ? a.cnt_ang[i] : 0;
        for (int s = lane; s < na; s += G) {
            PairT<R> p;
            if (!pair_at(a, fr, s, p) || !(p.r < (R)a.rc_ang)) continue;
            R g[NAX], gp[NAX];
            angular_g<DM>(a, fr.ti, p.tj, p.r, cutA, NA, KA, g, gp);
            const Harm<R> ht = harm_of(p.u[0], p.u[1], p.u[2]);
            HarmSums<R> hs(ht);
#pragma unroll
            for (int m = 0; m < kLM; ++m) {
                R am = R(0.0), bm = R(0.0);
#pragma unroll
                for (int n = 0; n < NAX; ++n)
                    if (n < NA) {
                        const R r = Ri[n * kLM + m];
                        am += r * g[n];
                        bm += r * gp[n];
                    }
                hs.add(m, ht, am, bm);
            }
            R f[3];
            hs.force(ht, p.ir, f[0], f[1], f[2]);
            a.fin[(size_t)a.rev[(size_t)s * N + i] * N + p.j] = make_float4(f[0], f[1], f[2], 0.0f);
            for (int c = 0; c < 3; ++c) {
                acc[c] += f[c];
                for (int d = 0; d < 3; ++d) acc[3 + 3 * c + d] -= f[c] * p.d[d];
            }
        }
        __syncwarp();
        group_store<G>(a, acc, i, lane, valid);
    }
}

// F_i and the per-atom virial.
//
// Generic path (kScatter): the radial pair forces of both directions from the
// projected adjoints, and the incoming angular forces of the reverse slots,
// are added to what k64_atom left; W_i = -sum_j f_ij (x) r_ij.
//
// FP64: dE_i/dr_ij and dE_j/dr_ji, both from both atoms' adjoints.  Seen from
// j the direction is -u, and the harmonics of degree l have parity (-1)^l, so
// j's coefficients join i's before the harmonics:
//   f_ij =          u sum_m b_m Y_m + (1/r) (1 - u u^T) sum_m a_m grad P_m
//   f_ji = - (-1)^l (the same with j's a, b).
// Each atom gets half of a pair's virial, -(f_ij - f_ji) (x) r_ij / 2, which
// sums to the same totals.  The angular pairs' slots are collected in the
// radial walk, so that the lanes of the angular one, which takes most of the
// time, are all busy.
constexpr int kF64Slots = 128;       // per atom; with more the list is walked again
template <int G, class DM, class A>
__global__ void __launch_bounds__(kF64Threads) k64_force(const A a) {
    using R = ScalarT<A>;
    constexpr int NAX = DM::NAX;
    extern __shared__ double smem64[];
    const int lane = threadIdx.x % G, group = threadIdx.x / G;
    const int T = a.T, NA = DM::NA(a), KR = DM::KR(a), N = a.N;
    constexpr int kSlotR = kScatter<A> ? 0 : kF64Slots * (int)sizeof(unsigned short) / (int)sizeof(R);
    const int own = kScatter<A> ? 0 : NA * kLM;
    R* Ri = reinterpret_cast<R*>(smem64) + group * (own + T * KR + kSlotR);
    R* Pi = Ri + own;
    unsigned short* slots = reinterpret_cast<unsigned short*>(Pi + T * KR);
    const int ia = blockIdx.x * Group64<G>::NG + group;
    const bool valid = ia < N;
    const int i = valid ? ia : N - 1;
    const FrameT<R> fr = frame64(a, i);
    if constexpr (!kScatter<A>)
        for (int x = lane; x < own; x += G) Ri[x] = a.R[(size_t)i * own + x];
    for (int x = lane; x < T * KR; x += G) Pi[x] = a.p[(size_t)i * T * KR + x];
    __syncwarp();
    const Cutoff<R> cutR((R)a.rc_rad);
    R acc[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = R(0.0);
    const int nc = valid ? a.cnt[i] : 0, cmax = warp_max_i(nc);
    const int gbase = (threadIdx.x & 31) & ~(G - 1);
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u), below = (1u << lane) - 1u;
    int na = 0;                          // generic: the list's angular prefix; FP64: pairs inside rc_ang so far
    if constexpr (kScatter<A>)
        if (valid) na = a.cnt_ang[i];
    for (int s0 = 0; s0 < cmax; s0 += G) {
        const int s = s0 + lane;
        PairT<R> p;
        const bool in = s < nc && pair_at(a, fr, s, p);
        bool ang = false;
        if (in) {
            ang = p.r < (R)a.rc_ang;
            const R* pi = Pi + p.tj * KR;
            const R* pj = a.p + ((size_t)p.j * T + fr.ti) * KR;
            R di = R(0.0), dj = R(0.0);
            basis_derivs<DM::KX>(p.r, cutR, KR, [&](int k, R, R fp) {
                di += pi[k] * fp;
                dj += pj[k] * fp;
            });
            const R all = di + dj, vir = kScatter<A> ? di : R(0.5) * all;
            for (int c = 0; c < 3; ++c) {
                acc[c] += all * p.u[c];
                for (int d = 0; d < 3; ++d) acc[3 + 3 * c + d] -= vir * p.u[c] * p.d[d];
            }
            if constexpr (kScatter<A>) {
                if (ang && s < na) {
                    const float4 g = a.fin[(size_t)s * N + i];
                    acc[0] -= g.x;
                    acc[1] -= g.y;
                    acc[2] -= g.z;
                }
            }
        }
        if constexpr (!kScatter<A>) {
            const unsigned m = (__ballot_sync(0xffffffffu, ang) >> gbase) & gmask;
            const int at = na + __popc(m & below);
            if (ang && at < kF64Slots) slots[at] = (unsigned short)s;
            na += __popc(m);
        }
    }
    __syncwarp();
    if constexpr (!kScatter<A>) {
        const Cutoff<R> cutA((R)a.rc_ang);
        const int KA = DM::KA(a);
        const bool kept = na <= kF64Slots && nc <= 65536;
        const int n2 = kept ? na : nc;
        for (int c2 = lane; c2 < n2; c2 += G) {
            PairT<R> p;
            if (!pair_at(a, fr, kept ? (int)slots[c2] : c2, p) || !(p.r < (R)a.rc_ang)) continue;
            R g[NAX], gp[NAX], h[NAX], hp[NAX];
            angular_g2<DM>(a, fr.ti, p.tj, p.r, cutA, NA, KA, g, gp, h, hp);
            const Harm<R> ht = harm_of(p.u[0], p.u[1], p.u[2]);
            const R* Rj = a.R + (size_t)p.j * NA * kLM;
            HarmSums<R> hs(ht);
#pragma unroll
            for (int m = 0; m < kLM; ++m) {
                // j's coefficients with the parity (-1)^l
                R am = R(0.0), bm = R(0.0);
#pragma unroll
                for (int n = 0; n < NAX; ++n)
                    if (n < NA) {
                        const R rj = Rj[n * kLM + m];
                        am += rj * h[n];
                        bm += rj * hp[n];
                    }
                if (lm_l(m) & 1) {
                    am = -am;
                    bm = -bm;
                }
#pragma unroll
                for (int n = 0; n < NAX; ++n)
                    if (n < NA) {
                        const R ri = Ri[n * kLM + m];
                        am += ri * g[n];
                        bm += ri * gp[n];
                    }
                hs.add(m, ht, am, bm);
            }
            R f[3];
            hs.force(ht, p.ir, f[0], f[1], f[2]);
            for (int c = 0; c < 3; ++c) {
                acc[c] += f[c];
                for (int d = 0; d < 3; ++d) acc[3 + 3 * c + d] -= R(0.5) * f[c] * p.d[d];
            }
        }
        __syncwarp();
    }
    if constexpr (kScatter<A>) {
        // on top of the owner's angular part
#pragma unroll
        for (int c = 0; c < 12; ++c)
            if (valid && lane == c % G) acc[c] += c < 3 ? a.force[(size_t)c * N + i] : a.w[(size_t)(c - 3) * N + i];
    }
    group_store<G>(a, acc, i, lane, valid);
}

__device__ int segment_of(const int* off, int B, int x) {
    int lo = 0, hi = B;   // off[lo] <= x < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// sum over a block: warp shuffles, then the warp sums in order
constexpr int kF64Red = 256;
__device__ double block_sum(double v, double* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    for (int q = 0; q < kF64Red / 32; ++q) s += red[q];
    return s;
}

// E and virial of every configuration: one CTA per chunk, a warp per
// component, FP64 sums in a fixed order; the CTA that finishes a
// configuration's last chunk adds the chunks' partials (as k_totals).  Atoms
// from n_owned on are left out (the owned prefix of a spatial decomposition).
template <class A>
__global__ void __launch_bounds__(320) k64_totals(const A a, double* e_tot, double* virial) {
    const int k = blockIdx.x, B = a.B, N = a.N, total = a.chunk_start[B];
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    auto put = [&](int b, double v) {
        if (lane) return;
        if (c == 0) {
            if (e_tot) e_tot[b] = v;
        } else if (virial) {
            virial[(size_t)b * 9 + c - 1] = v;
        }
    };
    if (k >= total) {                   // configurations without atoms
        for (int b = k - total; b < B; b += gridDim.x - total)
            if (a.chunk_start[b] == a.chunk_start[b + 1]) put(b, 0.0);
        return;
    }
    const int b = segment_of(a.chunk_start, B, k);
    const int k0 = a.chunk_start[b], nk = a.chunk_start[b + 1] - k0;
    const int a0 = a.atom_off[b] + (k - k0) * kChunk;
    const int a1 = min(min(a.atom_off[b + 1], a0 + kChunk), a.n_owned);
    const ScalarT<A>* src = c == 0 ? a.e : a.w + (size_t)(c - 1) * N;
    double v = 0.0;
#pragma unroll 4
    for (int i = a0 + lane; i < a1; i += 32) v += (double)src[i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (nk > 1) {
        if (lane == 0) {
            a.partial[(size_t)k * 10 + c] = v;
            __threadfence();
        }
        __shared__ int last;
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(a.ticket + b, 1) == nk - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (threadIdx.x == 0) a.ticket[b] = 0;
        v = 0.0;
        for (int q = lane; q < nk; q += 32) v += __ldcg(a.partial + (size_t)(k0 + q) * 10 + c);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    put(b, v);
}

// ------------------------------------------------------------ loss
// Per chunk: the force residual's squared sum and lam_i = dL/dF_i.
__global__ void __launch_bounds__(kF64Red) k64_loss_atoms(const F64Args a, const double* f_lbl, double wF,
                                                         double* lam, double* partial) {
    const int k = blockIdx.x, B = a.B, N = a.N;
    if (k >= a.chunk_start[B]) return;
    const int b = segment_of(a.chunk_start, B, k);
    const int a0 = a.atom_off[b] + (k - a.chunk_start[b]) * kChunk;
    const int a1 = min(a.atom_off[b + 1], a0 + kChunk);
    const double nb = (double)(a.atom_off[b + 1] - a.atom_off[b]);
    const double cf = 2.0 * wF / (3.0 * nb * (double)B);
    double acc = 0.0;
    for (int i = a0 + threadIdx.x; i < a1; i += kF64Red) {
        for (int c = 0; c < 3; ++c) {
            const double d = a.force[(size_t)c * N + i] - f_lbl[(size_t)c * N + i];
            lam[(size_t)c * N + i] = cf * d;
            acc += d * d;
        }
    }
    __shared__ double red[kF64Red / 32];
    const double v = block_sum(acc, red);
    if (threadIdx.x == 0) partial[k] = v;
}

// Per configuration: the loss terms and the energy and virial adjoints
// (modes as nep_param_grad); the batch loss in a fixed tree.
__global__ void __launch_bounds__(kF64Red) k64_loss_cfg(const F64Args a, const double* partial,
                                                       const double* e_tot, const double* vir,
                                                       const double* e_lbl, const double* v_lbl, double wE,
                                                       double wF, double wV, int mode, double* aE, double* mu,
                                                       double* loss) {
    const int B = a.B;
    double acc = 0.0;
    for (int b = threadIdx.x; b < B; b += kF64Red) {
        const double nb = (double)(a.atom_off[b + 1] - a.atom_off[b]);
        const double n = nb > 0.0 ? nb : 1.0;
        double sF = 0.0;
        for (int k = a.chunk_start[b]; k < a.chunk_start[b + 1]; ++k) sF += partial[k];
        const double dE = e_tot[b] - e_lbl[b];
        double sV = 0.0;
        for (int c = 0; c < 9; ++c) {
            const double dv = vir[9 * b + c] - v_lbl[9 * b + c];
            sV += dv * dv;
        }
        // mode 0: per-atom normalised energy and virial; mode 1: Eqs. 19-21
        const double nE = mode == 0 ? n * n : n, nV = mode == 0 ? 9.0 * n * n : 9.0 * n;
        const double Lb = wE * dE * dE / nE + wF * sF / (3.0 * n) + wV * sV / nV;
        aE[b] = 2.0 * wE * dE / nE / B;
        for (int c = 0; c < 9; ++c) mu[9 * b + c] = 2.0 * wV * (vir[9 * b + c] - v_lbl[9 * b + c]) / nV / B;
        if (nb > 0.0) acc += Lb;
    }
    __shared__ double red[kF64Red / 32];
    const double v = block_sum(acc, red);
    if (threadIdx.x == 0 && loss) *loss = v / B;
}

}  // namespace

cudaError_t launch_promote(const float* src, double* dst, int n, cudaStream_t st) {
    if (n > 0) k_promote<<<(n + 255) / 256, 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

namespace {
template <int G, class DM, class A>
cudaError_t launch_efv_g(const A& a, cudaStream_t st) {
    using R = ScalarT<A>;
    constexpr int NG = Group64<G>::NG;
    const int grid = (a.N + NG - 1) / NG;
    const size_t s1 = sizeof(R) * (size_t)NG * Group64<G>(a.T, a.NA, a.KR, a.D).size;
    const size_t s2 = sizeof(R) * (size_t)NG * a.T * a.KR +
                      (kScatter<A> ? 0 : NG * (sizeof(R) * a.NA * kLM + sizeof(unsigned short) * kF64Slots));
    cudaError_t e;
    if (s1 > 48 * 1024 &&
        (e = cudaFuncSetAttribute(k64_atom<G, DM, A>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)))
        return e;
    if (s2 > 48 * 1024 &&
        (e = cudaFuncSetAttribute(k64_force<G, DM, A>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)))
        return e;
    k64_atom<G, DM, A><<<grid, kF64Threads, s1, st>>>(a);
    k64_force<G, DM, A><<<grid, kF64Threads, s2, st>>>(a);
    return cudaGetLastError();
}
template <class A>
cudaError_t launch_efv_t(const A& a, int max_chunks, double* e_tot, double* virial, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    if (a.N > 0)
        e = with_dims(a, [&](auto dm) {
            using DM = decltype(dm);
            return a.N <= (kScatter<A> ? kGenericLanes32 : kEvalLanes32) ? launch_efv_g<32, DM>(a, st) : launch_efv_g<8, DM>(a, st);
        });
    if (e != cudaSuccess) return e;
    if (max_chunks > 0) k64_totals<A><<<max_chunks, 320, 0, st>>>(a, e_tot, virial);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_efv_fp64(const F64Args& a, int max_chunks, double* e_tot, double* virial,
                            cudaStream_t st) {
    return launch_efv_t(a, max_chunks, e_tot, virial, st);
}

cudaError_t launch_efv_generic(const F32Args& a, int max_chunks, double* e_tot, double* virial,
                               cudaStream_t st) {
    return launch_efv_t(a, max_chunks, e_tot, virial, st);
}

cudaError_t launch_loss_fp64(const F64Args& a, int max_chunks, const double* e_tot, const double* vir,
                             const double* e_lbl, const double* f_lbl, const double* v_lbl, const float* w,
                             int mode, double* lam, double* aE, double* mu, double* loss, cudaStream_t st) {
    // the per-chunk force sums reuse the evaluation's partials (consumed by then)
    if (max_chunks > 0) k64_loss_atoms<<<max_chunks, kF64Red, 0, st>>>(a, f_lbl, w[1], lam, a.partial);
    k64_loss_cfg<<<1, kF64Red, 0, st>>>(a, a.partial, e_tot, vir, e_lbl, v_lbl, w[0], w[1], w[2], mode, aE, mu,
                                        loss);
    return cudaGetLastError();
}

}  // namespace nep
