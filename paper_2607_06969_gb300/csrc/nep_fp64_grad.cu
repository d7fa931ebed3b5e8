// FP64 training gradient: the gradient of Phi = sum_b aE_b E_b + sum_i lam_i . F_i
// + sum_b mu_b : V_b at fixed adjoints (the loss gradient of Eqs. 18-21 when
// they are the loss adjoints).  With dr_ij = -(lam_j - lam_i) - mu r_ij,
// Phi = sum_i [aE E_i + p_i . dq_i], p = dE/dq, dq the tangent of q along dr.
//   k64_grad_atom : descriptors and network again, the tangent dq (radial
//                   DF[t][k] = sum_j Q'_k (rhat . dr), angular dS_nlm), the
//                   network's second-order terms (alpha, beta, gamma,
//                   rho = aE p + d(p . dq)/dq), P = dPhi/dS, R = dPhi/d(dS),
//                   and per angular pair X_n = sum_m P_nm Y_m + R_nm dY_m,
//                   Z_n = (rhat . dr) sum_m R_nm Y_m, summed into
//                   bins[t][n][k] = sum_{j of t} Q_k X_n + Q'_k Z_n; the
//                   per-atom factors of every parameter's gradient are staged
//   k64_grad_partial / k64_grad_final : per 1,024-atom chunk, each parameter
//                   summed over the chunk's atoms of its species; then the
//                   chunks in order
// Measured (38-30-1 model, 2,548 atoms): k64_grad_atom 1,659 -> 357 us,
// k64_grad_partial 5,787 -> 55 us.
#include "nep_fp64.cuh"

namespace nep {
namespace {

// ------------------------------------------------------------ gradient
// Staged per-atom factors, [field][N]: q, dq (D each), alpha, beta, gamma
// (H each), rho and p of the radial n (NR each), F and DF (T KR each), and
// bins (T NA KA).
struct GradFields {
    int q, dq, al, be, ga, rho, p, F, DF, bins, total;
};
__host__ __device__ GradFields grad_fields(const F64Args& a) {
    GradFields g;
    g.q = 0;
    g.dq = g.q + a.D;
    g.al = g.dq + a.D;
    g.be = g.al + a.H;
    g.ga = g.be + a.H;
    g.rho = g.ga + a.H;
    g.p = g.rho + a.NR;
    g.F = g.p + a.NR;
    g.DF = g.F + a.T * a.KR;
    g.bins = g.DF + a.T * a.KR;
    g.total = g.bins + a.T * a.NA * a.KA;
    return g;
}

// dr_ij = -(lam_j - lam_i) - mu r_ij
__device__ void tangent64(const F64Args& a, const double* li, const double* mu, const Pair64& p, double* dr) {
    const int N = a.N;
    for (int c = 0; c < 3; ++c)
        dr[c] = -(a.lam[(size_t)c * N + p.j] - li[c]) -
                (mu[3 * c] * p.d[0] + mu[3 * c + 1] * p.d[1] + mu[3 * c + 2] * p.d[2]);
}

// The per-atom backward, a group of G lanes per atom (as k64_atom).  One walk
// over the list gives the sums and their tangents together; the network's
// second-order terms follow, then P = dPhi/dS, R = dPhi/d(dS), and a walk over
// the angular pairs for X_n, Z_n, which the lanes (n, k) sum into the bins.
constexpr int kGrad64Threads = kF64Threads;
template <int G>
struct GradGroup64 {
    static constexpr int NG = kGrad64Threads / G, GS = G + 1;
    int NAs, oG, oB, oY, oQ, oDQ, oP, oRho, oJ, oDJ, oHb, oHc, oT, oS, oD, oF, oDF, size;
    __host__ __device__ GradGroup64(int T, int NA, int KR, int KA, int D) {
        NAs = NA | 1;
        oG = oB = 0;                               // [G][2 NAs] g, g' (rhat . dr) of a chunk's pairs, later the bins
        const int bins = T * NA * KA;
        oY = G * 2 * NAs > bins ? G * 2 * NAs : bins;
        int rows = 2 * kLM;                        // Y, dY; or Q, Q' (rhat . dr); or Q, Q', X, Z
        if (2 * KR > rows) rows = 2 * KR;
        if (2 * KA + 2 * NA > rows) rows = 2 * KA + 2 * NA;
        oQ = oY;                                   // the network's vectors between the walks
        oDQ = oQ + D;
        oP = oDQ + D;
        oRho = oP + D;
        oJ = oRho + D;
        oDJ = oJ + 5 * NA;
        oHb = oDJ + 5 * NA;
        oHc = oHb + kGroupTile;
        const int e1 = oY + rows * GS, e2 = oHc + kGroupTile;
        oT = e1 > e2 ? e1 : e2;
        oS = oT + G;
        oD = oS + NA * kLM;
        oF = oD + NA * kLM;
        oDF = oF + T * KR;
        size = oDF + T * KR;
    }
};

template <int G, class DM>
__global__ void __launch_bounds__(kGrad64Threads) k64_grad_atom(const F64Args a) {
    constexpr int NAX = DM::NAX;
    using L = Group64<G>;
    constexpr int GS = L::GS, MPL = L::MPL, KW = L::KW, KX = L::KX, PARTS = L::PARTS;
    extern __shared__ double smem64[];
    const int T = a.T, NR = a.NR, NA = DM::NA(a), KR = DM::KR(a), KA = DM::KA(a), H = a.H, D = a.D, N = a.N;
    const GradGroup64<G> o(T, NA, KR, KA, D);
    const int lane = threadIdx.x % G, group = threadIdx.x / G;
    double* gb = smem64 + group * o.size;
    int* tj = reinterpret_cast<int*>(gb + o.oT);
    const int gbase = (threadIdx.x & 31) & ~(G - 1);
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u), below = (1u << lane) - 1u;
    const int kl = lane % KW, part = lane / KW;
    const int ia = blockIdx.x * GradGroup64<G>::NG + group;
    const bool valid = ia < N;
    const int i = valid ? ia : N - 1;
    const GradFields gf = grad_fields(a);
    const Frame64 fr = frame64(a, i);
    const double li[3] = {a.lam[i], a.lam[N + i], a.lam[2 * N + i]};
    const double* mu = a.mu + 9 * fr.b;
    const double aE = a.aE[fr.b];
    const Cutoff<double> cutR(a.rc_rad), cutA(a.rc_ang);
    const int nc = valid ? a.cnt[i] : 0, cmax = warp_max_i(nc);

    // ---- F[t][k] = sum Q_k, DF[t][k] = sum Q'_k (rhat . dr); S_nlm and
    // dS_nlm = sum_j [g'_n (rhat . dr) Y_m + g_n dY_m], dY_m along the change of rhat
    double S[NAX][MPL], dS[NAX][MPL], F[KX][kMaxTypes], DF[KX][kMaxTypes];
#pragma unroll
    for (int n = 0; n < NAX; ++n)
#pragma unroll
        for (int x = 0; x < MPL; ++x) S[n][x] = dS[n][x] = 0.0;
#pragma unroll
    for (int x = 0; x < KX; ++x)
#pragma unroll
        for (int t = 0; t < kMaxTypes; ++t) F[x][t] = DF[x][t] = 0.0;
    int ang_end = 0;                               // end of the last chunk with an angular pair (of the warp)
    for (int s0 = 0; s0 < cmax; s0 += G) {
        const int s = s0 + lane;
        Pair64 p;
        const bool in = s < nc && pair_at(a, fr, s, p);
        double dr[3], udr = 0.0;
        const unsigned mi = (__ballot_sync(0xffffffffu, in) >> gbase) & gmask;
        const int ni = __popc(mi), ati = __popc(mi & below);
        if (in) {
            tangent64(a, li, mu, p, dr);
            udr = p.u[0] * dr[0] + p.u[1] * dr[1] + p.u[2] * dr[2];
            tj[ati] = p.tj;
            basis_derivs<DM::KX>(p.r, cutR, KR, [&](int k, double f, double fp) {
                gb[o.oY + k * GS + ati] = f;
                gb[o.oY + (KR + k) * GS + ati] = fp * udr;
            });
        }
        __syncwarp();
        for (int q = part; q < ni; q += PARTS) {
            const int t = tj[q];
#pragma unroll
            for (int x = 0; x < KX; ++x) {
                const int k = kl + x * KW;
                if (k >= KR) continue;
                const double f = gb[o.oY + k * GS + q], fd = gb[o.oY + (KR + k) * GS + q];
#pragma unroll
                for (int u = 0; u < kMaxTypes; ++u)
                    if (t == u) {
                        F[x][u] += f;
                        DF[x][u] += fd;
                    }
            }
        }
        __syncwarp();
        const bool ang = in && p.r < a.rc_ang;
        const unsigned any = __ballot_sync(0xffffffffu, ang);
        if (!any) continue;
        ang_end = s0 + G;
        const unsigned ma = (any >> gbase) & gmask;
        const int na = __popc(ma), at = __popc(ma & below);
        if (ang) {
            double f[DM::KX], fp[DM::KX];
            basis_derivs<DM::KX>(p.r, cutA, KA, [&](int k, double v, double d) {
                f[k] = v;
                fp[k] = d;
            });
            const double* c = a.prm + a.L.off_cA + (size_t)(fr.ti * T + p.tj) * NA * KA;
#pragma unroll
            for (int n = 0; n < NAX; ++n) {
                if (n >= NA) break;
                double g = 0.0, gp = 0.0;
#pragma unroll
                for (int k = 0; k < DM::KX; ++k)
                    if (k < KA) {
                        g += c[n * KA + k] * f[k];
                        gp += c[n * KA + k] * fp[k];
                    }
                gb[o.oG + at * 2 * o.NAs + n] = g;
                gb[o.oG + (at * 2 + 1) * o.NAs + n] = gp * udr;
            }
            const Harm<double> ht = harm_of(p.u[0], p.u[1], p.u[2]);
            const HarmD<double> hd = unit_tangent(ht, dr[0], dr[1], dr[2], udr, p.ir);
#pragma unroll
            for (int m = 0; m < kLM; ++m) {
                gb[o.oY + m * GS + at] = harm_value(m, ht);
                gb[o.oY + (kLM + m) * GS + at] = harm_dvalue(m, ht, hd);
            }
        }
        __syncwarp();
        for (int q = 0; q < na; ++q) {
#pragma unroll
            for (int x = 0; x < MPL; ++x) {
                const int m = lane + x * G;
                if (m >= kLM) continue;
                const double Y = gb[o.oY + m * GS + q], dY = gb[o.oY + (kLM + m) * GS + q];
#pragma unroll
                for (int n = 0; n < NAX; ++n)
                    if (n < NA) {
                        const double g = gb[o.oG + q * 2 * o.NAs + n];
                        S[n][x] += g * Y;
                        dS[n][x] += gb[o.oG + (q * 2 + 1) * o.NAs + n] * Y + g * dY;
                    }
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int x = 0; x < KX; ++x)
#pragma unroll
        for (int t = 0; t < kMaxTypes; ++t) {
            double v = F[x][t], w = DF[x][t];
#pragma unroll
            for (int h = KW; h < G; h <<= 1) {
                v += __shfl_xor_sync(0xffffffffu, v, h);
                w += __shfl_xor_sync(0xffffffffu, w, h);
            }
            if (part == 0 && kl + x * KW < KR && t < T) {
                gb[o.oF + t * KR + kl + x * KW] = v;
                gb[o.oDF + t * KR + kl + x * KW] = w;
            }
        }
#pragma unroll
    for (int n = 0; n < NAX; ++n)
#pragma unroll
        for (int x = 0; x < MPL; ++x)
            if (n < NA && lane + x * G < kLM) {
                gb[o.oS + n * kLM + lane + x * G] = S[n][x];
                gb[o.oD + n * kLM + lane + x * G] = dS[n][x];
            }
    __syncwarp();

    // ---- q, dq and the 4-body derivatives
    const double* cR = a.prm + a.L.off_cR + (size_t)fr.ti * T * NR * KR;
    for (int n = lane; n < NR; n += G) {
        double v = 0.0, w = 0.0;
        for (int t = 0; t < T; ++t)
            for (int k = 0; k < KR; ++k) {
                const double c = cR[(t * NR + n) * KR + k];
                v += c * gb[o.oF + t * KR + k];
                w += c * gb[o.oDF + t * KR + k];
            }
        gb[o.oQ + n] = v;
        gb[o.oDQ + n] = w;
    }
    for (int x = lane; x < NA * 4; x += G) {
        const int n = x >> 2, l = x & 3, m0 = l * (l + 2);
        double v = 0.0, w = 0.0;
        for (int m = m0; m < m0 + 2 * l + 3; ++m) {
            const double sv = gb[o.oS + n * kLM + m], c = (double)clm(m) * sv;
            v += c * sv;
            w += 2.0 * c * gb[o.oD + n * kLM + m];
        }
        gb[o.oQ + NR + x] = v;
        gb[o.oDQ + NR + x] = w;
    }
    if (a.H4)
        for (int n = lane; n < NA; n += G) {
            const double *s2 = gb + o.oS + n * kLM + 3, *d2 = gb + o.oD + n * kLM + 3;
            double *J = gb + o.oJ + 5 * n, w = 0.0;
            gb[o.oQ + NR + NA * 4 + n] = fourbody<double>(s2, nullptr);
            fourbody_jvp<double>(s2, d2, J, gb + o.oDJ + 5 * n);
            for (int m = 0; m < 5; ++m) w += J[m] * d2[m];
            gb[o.oDQ + NR + NA * 4 + n] = w;
        }
    for (int d = lane; d < D; d += G) gb[o.oP + d] = gb[o.oRho + d] = 0.0;
    __syncwarp();

    // ---- network and its second-order terms:
    // u = W0 dq, alpha = aE w1 s - 2 w1 u t s (coefficient of q in dW0, and
    // db0), beta = w1 s (coefficient of dq), gamma = aE t + s u (dw1);
    // p = W0^T (w1 s), rho = aE p + W0^T (-2 w1 u t s)
    const double* W0 = a.prm + (size_t)fr.ti * a.L.mlp_stride;
    const double* b0 = W0 + (size_t)H * D;
    const double* w1 = b0 + H;
    for (int h0 = 0; h0 < H; h0 += kGroupTile) {
        const int nh = min(kGroupTile, H - h0);
        for (int h = lane; h < nh; h += G) {
            const double* w = W0 + (size_t)(h0 + h) * D;
            double z = b0[h0 + h], u = 0.0;
            for (int d = 0; d < D; ++d) {
                z += w[d] * gb[o.oQ + d];
                u += w[d] * gb[o.oDQ + d];
            }
            const double t = tanh(z), sd = 1.0 - t * t, wh = w1[h0 + h];
            const double c2 = -2.0 * wh * u * t * sd;
            if (valid) {
                a.st[(size_t)(gf.al + h0 + h) * N + i] = aE * wh * sd + c2;
                a.st[(size_t)(gf.be + h0 + h) * N + i] = wh * sd;
                a.st[(size_t)(gf.ga + h0 + h) * N + i] = aE * t + sd * u;
            }
            gb[o.oHb + h] = wh * sd;
            gb[o.oHc + h] = c2;
        }
        __syncwarp();
        for (int d = lane; d < D; d += G) {
            const double* w = W0 + (size_t)h0 * D + d;
            double p = gb[o.oP + d], r = gb[o.oRho + d];
            for (int h = 0; h < nh; ++h) {
                const double v = w[(size_t)h * D];
                p += gb[o.oHb + h] * v;
                r += gb[o.oHc + h] * v;
            }
            gb[o.oP + d] = p;
            gb[o.oRho + d] = r;
        }
        __syncwarp();
    }
    for (int d = lane; d < D; d += G) gb[o.oRho + d] += aE * gb[o.oP + d];
    __syncwarp();
    if (valid) {
        for (int d = lane; d < D; d += G) {
            a.st[(size_t)(gf.q + d) * N + i] = gb[o.oQ + d];
            a.st[(size_t)(gf.dq + d) * N + i] = gb[o.oDQ + d];
        }
        for (int n = lane; n < NR; n += G) {
            a.st[(size_t)(gf.rho + n) * N + i] = gb[o.oRho + n];
            a.st[(size_t)(gf.p + n) * N + i] = gb[o.oP + n];
        }
        for (int x = lane; x < T * KR; x += G) {
            a.st[(size_t)(gf.F + x) * N + i] = gb[o.oF + x];
            a.st[(size_t)(gf.DF + x) * N + i] = gb[o.oDF + x];
        }
    }

    // ---- P over dS, R over S:
    // P_nm = 2 C_lm (rho_nl S_nm + p_nl dS_nm) (+ rho4 J_m + p4 dJ_m),
    // R_nm = 2 C_lm p_nl S_nm (+ p4 J_m)
#pragma unroll
    for (int x = 0; x < MPL; ++x) {
        const int m = lane + x * G;
        if (m >= kLM) continue;
        const int l = lm_l(m);
        const double c2 = 2.0 * (double)clm(m);
#pragma unroll
        for (int n = 0; n < NAX; ++n) {
            if (n >= NA) continue;
            const double pl = gb[o.oP + NR + n * 4 + l - 1], rl = gb[o.oRho + NR + n * 4 + l - 1];
            double Pv = c2 * (rl * S[n][x] + pl * dS[n][x]), Rv = c2 * pl * S[n][x];
            if (a.H4 && l == 2) {
                const double p4 = gb[o.oP + NR + NA * 4 + n], r4 = gb[o.oRho + NR + NA * 4 + n];
                const double J = gb[o.oJ + 5 * n + m - 3];
                Pv += r4 * J + p4 * gb[o.oDJ + 5 * n + m - 3];
                Rv += p4 * J;
            }
            gb[o.oD + n * kLM + m] = Pv;
            gb[o.oS + n * kLM + m] = Rv;
        }
    }
    __syncwarp();
    const int nb = T * NA * KA;
    for (int x = lane; x < nb; x += G) gb[o.oB + x] = 0.0;

    // ---- bins[t][n][k] = sum_{j of t} Q_k X_n + Q'_k Z_n over the angular pairs
    for (int s0 = 0; s0 < ang_end; s0 += G) {
        const int s = s0 + lane;
        Pair64 p;
        const bool ang = s < nc && pair_at(a, fr, s, p) && p.r < a.rc_ang;
        const unsigned ma = (__ballot_sync(0xffffffffu, ang) >> gbase) & gmask;
        const int na = __popc(ma), at = __popc(ma & below);
        if (ang) {
            double dr[3];
            tangent64(a, li, mu, p, dr);
            const double udr = p.u[0] * dr[0] + p.u[1] * dr[1] + p.u[2] * dr[2];
            tj[at] = p.tj;
            basis_derivs<DM::KX>(p.r, cutA, KA, [&](int k, double f, double fp) {
                gb[o.oY + k * GS + at] = f;
                gb[o.oY + (KA + k) * GS + at] = fp;
            });
            const Harm<double> ht = harm_of(p.u[0], p.u[1], p.u[2]);
            const HarmD<double> hd = unit_tangent(ht, dr[0], dr[1], dr[2], udr, p.ir);
            double X[NAX], Z[NAX];
#pragma unroll
            for (int n = 0; n < NAX; ++n) X[n] = Z[n] = 0.0;
#pragma unroll
            for (int m = 0; m < kLM; ++m) {
                const double Y = harm_value(m, ht), dY = harm_dvalue(m, ht, hd);
#pragma unroll
                for (int n = 0; n < NAX; ++n)
                    if (n < NA) {
                        const double R = gb[o.oS + n * kLM + m];
                        X[n] += gb[o.oD + n * kLM + m] * Y + R * dY;
                        Z[n] += R * Y;
                    }
            }
#pragma unroll
            for (int n = 0; n < NAX; ++n)
                if (n < NA) {
                    gb[o.oY + (2 * KA + n) * GS + at] = X[n];
                    gb[o.oY + (2 * KA + NA + n) * GS + at] = udr * Z[n];
                }
        }
        __syncwarp();
        for (int q = 0; q < na; ++q) {
            double* bin = gb + o.oB + tj[q] * NA * KA;
            for (int x = lane; x < NA * KA; x += G) {
                const int n = x / KA, k = x % KA;
                bin[x] += gb[o.oY + k * GS + q] * gb[o.oY + (2 * KA + n) * GS + q] +
                          gb[o.oY + (KA + k) * GS + q] * gb[o.oY + (2 * KA + NA + n) * GS + q];
            }
        }
        __syncwarp();
    }
    if (valid)
        for (int x = lane; x < nb; x += G) a.st[(size_t)(gf.bins + x) * N + i] = gb[o.oB + x];
}

// Each parameter's gradient over one 1,024-atom chunk: the sum, over the
// chunk's atoms of the parameter's species, of a1 b1 + a2 b2 (staged factors;
// b = 1 where absent; aE for b1).  A warp takes one item of up to eight
// parameters that share factors, its lanes the atoms of the species:
//   two-factor  (species, 2 rows x 4 columns): W0's alpha_h q_d + beta_h dq_d
//               and cR's rho_n F[t2][k] + p_n DF[t2][k]; 12 loads per atom
//               instead of 32 for the eight parameters
//   one-factor  (species, 4 rows): b0 (alpha_h), w1 (gamma_h), cA (bins)
//   b1          (species)
// The atoms are first ordered by species, so that no lane is spent on another
// species' atoms: GB300's FP64 pipe (about 1/64 of the FP32 rate) bounds the
// sums once the chip is full.  The grid splits the items as well as the chunks: with one CTA
// per chunk a batch of 2,548 atoms ran on 3 of 152 SMs and took 5.8 ms.
constexpr int kGradWarps = 8;
struct GradItems64 {
    int nW0, nB, nCR, nCA, total;   // W0, b0 + w1, cR and cA items
};
__host__ __device__ inline GradItems64 grad_items64(const F64Args& a) {
    GradItems64 g;
    g.nW0 = a.T * ((a.H + 1) / 2) * ((a.D + 3) / 4);
    g.nB = 2 * a.T * ((a.H + 3) / 4);
    g.nCR = a.T * a.T * ((a.NR + 1) / 2) * ((a.KR + 3) / 4);
    g.nCA = a.T * ((a.T * a.NA * a.KA + 3) / 4);
    g.total = g.nW0 + g.nCR + g.nB + g.nCA + a.T;
    return g;
}

__global__ void __launch_bounds__(32 * kGradWarps) k64_grad_partial(const F64Args a) {
    const int c = blockIdx.x, N = a.N, T = a.T, NR = a.NR, KR = a.KR, H = a.H, D = a.D;
    const ParamLayout& L = a.L;
    const GradFields gf = grad_fields(a);
    const GradItems64 gi = grad_items64(a);
    const int a0 = c * kChunk, na = min(N - a0, kChunk);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the chunk's atoms in species order (stable)
    __shared__ int order[kChunk];
    __shared__ int wcnt[kMaxTypes][kChunk / 32];
    __shared__ int first[kMaxTypes + 1];
    for (int r = warp; r < kChunk / 32; r += kGradWarps) {
        const int x = r * 32 + lane;
        const int sp = x < na ? a.type[a0 + x] : -1;
        for (int t = 0; t < T; ++t) {
            const unsigned m = __ballot_sync(0xffffffffu, sp == t);
            if (lane == 0) wcnt[t][r] = __popc(m);
        }
    }
    __syncthreads();
    if (warp == 0) {
        int base = 0;
        for (int t = 0; t < T; ++t) {
            const int v = wcnt[t][lane];
            int incl = v;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            wcnt[t][lane] = base + incl - v;
            if (lane == 0) first[t] = base;
            base += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) first[T] = base;
    }
    __syncthreads();
    for (int r = warp; r < kChunk / 32; r += kGradWarps) {
        const int x = r * 32 + lane;
        const int sp = x < na ? a.type[a0 + x] : -1;
        for (int t = 0; t < T; ++t) {
            const unsigned m = __ballot_sync(0xffffffffu, sp == t);
            if (sp == t) order[wcnt[t][r] + __popc(m & ((1u << lane) - 1u))] = a0 + x;
        }
    }
    __syncthreads();
    static_assert(kChunk / 32 == 32, "one lane per row of the chunk");
    double* out = a.gpart + (size_t)c * L.P;
    const double* st = a.st;
    for (int it = blockIdx.y * kGradWarps + warp; it < gi.total; it += gridDim.y * kGradWarps) {
        if (it < gi.nW0 + gi.nCR) {
            // rows r0, r0 + 1 of (A, B) times columns c0 .. c0 + 3 of (X, Y)
            int sp, r0, c0, nr, nc, fA, fB, fX, fY, pbase, pstride;
            if (it < gi.nW0) {
                const int DB = (D + 3) / 4, HB = (H + 1) / 2;
                c0 = 4 * (it % DB);
                r0 = 2 * ((it / DB) % HB);
                sp = it / (DB * HB);
                nr = H; nc = D;
                fA = gf.al; fB = gf.be; fX = gf.q; fY = gf.dq;
                pbase = sp * L.mlp_stride;
                pstride = D;
            } else {
                int x = it - gi.nW0;
                const int KB = (KR + 3) / 4, NB = (NR + 1) / 2;
                c0 = 4 * (x % KB);
                x /= KB;
                r0 = 2 * (x % NB);
                x /= NB;
                const int t2 = x % T;
                sp = x / T;
                nr = NR; nc = KR;
                fA = gf.rho; fB = gf.p; fX = gf.F + t2 * KR; fY = gf.DF + t2 * KR;
                pbase = L.off_cR + (sp * T + t2) * NR * KR;
                pstride = KR;
            }
            // a row or column past the end repeats the last one; its sum is dropped
            const double *pA[2], *pB[2], *pX[4], *pY[4];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                pA[r] = st + (size_t)(fA + min(r0 + r, nr - 1)) * N;
                pB[r] = st + (size_t)(fB + min(r0 + r, nr - 1)) * N;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                pX[k] = st + (size_t)(fX + min(c0 + k, nc - 1)) * N;
                pY[k] = st + (size_t)(fY + min(c0 + k, nc - 1)) * N;
            }
            double acc[2][4] = {};
            for (int x = first[sp] + lane; x < first[sp + 1]; x += 32) {
                const int i = order[x];
                double vA[2], vB[2], vX[4], vY[4];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    vA[r] = pA[r][i];
                    vB[r] = pB[r][i];
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    vX[k] = pX[k][i];
                    vY[k] = pY[k][i];
                }
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[r][k] += vA[r] * vX[k] + vB[r] * vY[k];
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const double v = warp_sum(acc[r][k]);
                    if (lane == 0 && r0 + r < nr && c0 + k < nc) out[pbase + (r0 + r) * pstride + c0 + k] = v;
                }
            continue;
        }
        int x = it - gi.nW0 - gi.nCR, sp, r0, nr, f, pbase;
        if (x < gi.nB) {
            const int HB = (H + 3) / 4, which = x / (T * HB), y = x % (T * HB);
            sp = y / HB;
            r0 = 4 * (y % HB);
            nr = H;
            f = which ? gf.ga : gf.al;
            pbase = sp * L.mlp_stride + H * D + which * H;
        } else if ((x -= gi.nB) < gi.nCA) {
            nr = T * a.NA * a.KA;
            const int BB = (nr + 3) / 4;
            sp = x / BB;
            r0 = 4 * (x % BB);
            f = gf.bins;
            pbase = L.off_cA + sp * nr;
        } else {
            sp = x - gi.nCA;
            double acc = 0.0;
            for (int y = first[sp] + lane; y < first[sp + 1]; y += 32) acc += a.aE[a.cfg[order[y]]];
            acc = warp_sum(acc);
            if (lane == 0) out[sp * L.mlp_stride + H * D + 2 * H] = acc;
            continue;
        }
        const double* pA[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) pA[r] = st + (size_t)(f + min(r0 + r, nr - 1)) * N;
        double acc[4] = {};
        for (int y = first[sp] + lane; y < first[sp + 1]; y += 32) {
            const int i = order[y];
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r] += pA[r][i];
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const double v = warp_sum(acc[r]);
            if (lane == 0 && r0 + r < nr) out[pbase + r0 + r] = v;
        }
    }
}

__global__ void k64_grad_final(const F64Args a, int nchunk) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.L.P) return;
    double acc = 0.0;
    for (int c = 0; c < nchunk; ++c) acc += a.gpart[(size_t)c * a.L.P + p];
    a.grad[p] = acc;
}

}  // namespace

int fp64_grad_fields(const F64Args& a) { return grad_fields(a).total; }

int fp64_grad_chunks(int N) { return (N + kChunk - 1) / kChunk; }

namespace {
template <int G, class DM>
cudaError_t launch_grad_atom(const F64Args& a, cudaStream_t st) {
    using M = GradGroup64<G>;
    const size_t smem = sizeof(double) * (size_t)M::NG * M(a.T, a.NA, a.KR, a.KA, a.D).size;
    cudaError_t e;
    if (smem > 48 * 1024 && (e = cudaFuncSetAttribute(k64_grad_atom<G, DM>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)))
        return e;
    k64_grad_atom<G, DM><<<(a.N + M::NG - 1) / M::NG, kGrad64Threads, smem, st>>>(a);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_grad_fp64(const F64Args& a, cudaStream_t st) {
    if (a.N > 0) {
        const cudaError_t e = with_dims(a, [&](auto dm) {
            using DM = decltype(dm);
            return a.N <= kEvalLanes32 ? launch_grad_atom<32, DM>(a, st) : launch_grad_atom<8, DM>(a, st);
        });
        if (e != cudaSuccess) return e;
        // about 1,024 CTAs, each with at least one item per warp
        const int nchunk = fp64_grad_chunks(a.N);
        const int most = (grad_items64(a).total + kGradWarps - 1) / kGradWarps;
        const int split = std::max(1, std::min(most, 1024 / nchunk));
        k64_grad_partial<<<dim3(nchunk, split), 32 * kGradWarps, 0, st>>>(a);
    }
    k64_grad_final<<<(a.L.P + 255) / 256, 256, 0, st>>>(a, fp64_grad_chunks(a.N));
    return cudaGetLastError();
}

}  // namespace nep
