// The per-atom training backward with a group of G lanes per atom (the
// counterpart of k_tangent in nep_train.cuh, see there for the formulas; the
// lanes' split is that of kg_atom).  kg_grad walks an atom's list once for the
// descriptors' sums and their tangents together (F, S and DF, dS), runs the
// network with its second-order terms, and walks the angular pairs once more
// for the coefficients X_n, Z_n and the angular c-gradient, which the lanes
// (n, k) sum from the pairs' X, Z, Q, Q' in shared memory.  It recomputes what
// it needs, so a vector-Jacobian product (nep_param_grad_adjoint) runs no
// forward evaluation, and the loss gradient's forward is the plain one,
// without the training variant's records.
#pragma once
#include "nep_group.cuh"

namespace nep {

#if defined(__CUDACC__)

constexpr int kGradBlocks = 3;   // resident CTAs per SM the registers are held to; 4 spill (20,405 atoms 283 / 305 us)

template <class C, int G>
struct GroupGradSmem {
    static constexpr int NA = C::NA, T = C::T, KR = C::KR, KA = C::KA, D = C::D;
    static constexpr int NG = kGroupThreads / G, GS = G + 1;
    static constexpr int NAp = round4(NA);
    // [G][2 NAp] g_n and g'_n (rhat . dr) of a chunk's pairs; then F and DF
    static constexpr int oG = 0;
    static constexpr int szG = round4(G * 2 * NAp > 2 * T * KR ? G * 2 * NAp : 2 * T * KR);
    static constexpr int oF = oG, oDF = oF + T * KR;
    // exchange buffer: Y_m, then dY_m; F partials, then DF's; the network's
    // vectors; then Q, Q', X, Z of a chunk's pairs
    static constexpr int oY = oG + szG;
    static constexpr int rows0 = kLM > T * KR ? kLM : T * KR;
    static constexpr int rows = rows0 > 2 * KA + 2 * NA ? rows0 : 2 * KA + 2 * NA;
    static constexpr int oQ = oY, oDQ = oQ + C::DW, oP = oDQ + C::DW, oRho = oP + C::DW;
    static constexpr int oJ = oRho + C::DW, oDJ = oJ + round4(5 * NA), oHb = oDJ + round4(5 * NA);
    static NEP_HD int oHc(int H) { return oHb + round4(H); }
    static NEP_HD int slots(int H) {
        const int a = round4(oY + rows * GS), b = oHc(H) + round4(H);
        return a > b ? a : b;
    }
    static NEP_HD int S(int H) { return slots(H) + kGroupSlots / 2; }   // [NA][24] S, then R = dPhi/d(dS)
    static NEP_HD int dS(int H) { return S(H) + NA * kLM; }             // [NA][24] dS, then P = dPhi/dS
    static NEP_HD int group_size(int H) { return dS(H) + NA * kLM; }
    static NEP_HD size_t bytes(int H) {
        return sizeof(float) * (size_t)(GroupSmem<C, G>::groups(H) + NG * group_size(H));
    }
};

// r_ij, d r_ij along the tangent and rhat . dr of list entry (j, shift) of atom i.
// r and 1/r come from one rsqrtf (dist_rinv), where k_tangent takes sqrtf and a
// rounded reciprocal: a difference of 2 ulp.  The gradient's error against 64 bits
// is level (20,405 atoms, three seeds: 3.5e-7, 1.5e-7, 2.3e-7 against 3.8e-7,
// 1.6e-7, 2.3e-7).
struct TangentPair {
    int j, tj;
    float dx, dy, dz, d2, r, ir, drx, dry, drz, udr;
};
__device__ __forceinline__ void tangent_pair(const EvalArgs& a, const AtomFrame& fr, float4 pj, float4 lj, int sh,
                                             float4 li, const float* mu, TangentPair& p) {
    p.tj = f2i(pj.w);
    pair_vector(fr.pi, pj, fr.Lx, fr.Ly, fr.Lz, fr.iLx, fr.iLy, fr.iLz, a.min_image, sh, p.dx, p.dy, p.dz);
    p.d2 = norm2(p.dx, p.dy, p.dz);
    dist_rinv(p.d2, p.r, p.ir);
    p.drx = -(lj.x - li.x) - (mu[0] * p.dx + mu[1] * p.dy + mu[2] * p.dz);
    p.dry = -(lj.y - li.y) - (mu[3] * p.dx + mu[4] * p.dy + mu[5] * p.dz);
    p.drz = -(lj.z - li.z) - (mu[6] * p.dx + mu[7] * p.dy + mu[8] * p.dz);
    p.udr = (p.dx * p.drx + p.dy * p.dry + p.dz * p.drz) * p.ir;
}

// sums over the group's lanes of the rows v[0..n) (one value per lane and
// row), through the exchange buffer; row o's sum goes to dst[o]
template <int G, int ROWS>
__device__ __forceinline__ void lanes_rows_sum(float* buf, const float* v, float* dst, int lane) {
    constexpr int GS = G + 1;
    __syncwarp();
#pragma unroll
    for (int o = 0; o < ROWS; ++o) buf[o * GS + lane] = v[o];
    __syncwarp();
    for (int o = lane; o < ROWS; o += G) {
        float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
        for (int l = 0; l < G; l += 2) {
            s0 += buf[o * GS + l];
            s1 += buf[o * GS + l + 1];
        }
        dst[o] = s0 + s1;
    }
}

template <class C, int G>
__global__ void __launch_bounds__(kGroupThreads, kGradBlocks) kg_grad(const TrainArgs t) {
    using M = GroupGradSmem<C, G>;
    using I = GroupSmem<C, G>;                       // the model image is kg_atom's
    constexpr int NR = C::NR, NA = C::NA, KR = C::KR, KA = C::KA, T = C::T, D = C::D;
    constexpr int MPL = (kLM + G - 1) / G, GS = M::GS, NAp = M::NAp;
    extern __shared__ float sm[];
    const EvalArgs& a = t.e;
    const int N = a.N, H = a.H;
    group_load_model<C, G>(sm, a.params, H);      // older than the kernel before this one
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x % G, group = threadIdx.x / G;
    float* gb = sm + I::groups(H) + group * M::group_size(H);
    float* gS = gb + M::S(H);
    float* gD = gb + M::dS(H);
    float* gHb = gb + M::oHb;
    float* gHc = gb + M::oHc(H);
    unsigned short* slots = reinterpret_cast<unsigned short*>(gb + M::slots(H));
    const int gbase = (threadIdx.x & 31) & ~(G - 1);
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u), below = (1u << lane) - 1u;
    const float rcR2 = a.rc_rad * a.rc_rad, rcA2 = a.rc_ang * a.rc_ang;
    const float irR = 1.0f / a.rc_rad, irA = 1.0f / a.rc_ang;
    bool first = true;
    const int ntiles = (N + M::NG - 1) / M::NG;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int ia = tile * M::NG + group;
        const bool valid = ia < N;
        const int i = valid ? ia : N - 1;
        const AtomFrame fr = atom_frame(a, i);
        const int ti = fr.ti;
        const int cnt = valid ? a.cnt[i] : 0, cnt_ang = valid ? a.cnt_ang[i] : 0;
        float4 li;
        float mu[9];
        adjoint_frame(t, i, li, mu);

        // ---- sums F, S and their tangents DF, dS over the list
        constexpr int NA2 = (NA + 1) / 2;
        float2 S[NA2][MPL], dS[NA2][MPL];            // rows n two by two (paired FMAs)
        auto row = [](const float2 (&v)[NA2][MPL], int n, int x) { return n % 2 ? v[n / 2][x].y : v[n / 2][x].x; };
        float fb[T * KR], df[T * KR];
#pragma unroll
        for (int n = 0; n < NA2; ++n)
#pragma unroll
            for (int x = 0; x < MPL; ++x) S[n][x] = dS[n][x] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int o = 0; o < T * KR; ++o) fb[o] = df[o] = 0.0f;
        const int cmax = warp_max(cnt), amax = warp_max(cnt_ang);
        int total = 0;
        int j1 = lane < cnt ? a.nbr[(size_t)lane * N + i] : i;
        int j2 = lane + G < cnt ? a.nbr[(size_t)(lane + G) * N + i] : i;
        float4 p1 = a.pos4[j1], l1 = t.lam4[j1];
        for (int s0 = 0; s0 < cmax; s0 += G) {
            const int s = s0 + lane;
            const bool act = s < cnt;
            const float4 pj = p1, lj = l1;
            const int sh = act && !a.min_image ? a.shift[(size_t)s * N + i] : 0;
            j1 = j2;
            p1 = a.pos4[j1];
            l1 = t.lam4[j1];
            j2 = s + 2 * G < cnt ? a.nbr[(size_t)(s + 2 * G) * N + i] : i;
            TangentPair p;
            tangent_pair(a, fr, pj, lj, sh, li, mu, p);
            if (act && p.d2 < rcR2) {
                float f[KR], fp[KR];
                basis_d<KR>(p.r, irR, f, fp);
#pragma unroll
                for (int u = 0; u < T; ++u) {
                    const float w = (p.tj == u) ? 1.0f : 0.0f, wd = (p.tj == u) ? p.udr : 0.0f;
#pragma unroll
                    for (int k = 0; k < KR; ++k) {
                        fb[u * KR + k] = fmaf(w, f[k], fb[u * KR + k]);
                        df[u * KR + k] = fmaf(wd, fp[k], df[u * KR + k]);
                    }
                }
            }
            if (s0 >= amax) continue;
            const bool ang = act && s < cnt_ang && p.d2 < rcA2;
            const unsigned m = (__ballot_sync(0xffffffffu, ang) >> gbase) & gmask;
            const int np = __popc(m), at = __popc(m & below);
            float dY[kLM];
            if (ang) {
                if (total + at < kGroupSlots) slots[total + at] = (unsigned short)s;
                float g[NA], gp[NA];
                {
                    float f[KA], fp[KA];
                    basis_d<KA>(p.r, irA, f, fp);
                    const float* c2 = sm + I::cA2() + (ti * T + p.tj) * C::SA;
                    contract_pairs<NA, KA>(c2, f, g);
                    contract_pairs<NA, KA>(c2, fp, gp);
                }
                float* gr = gb + M::oG + at * 2 * NAp;
#pragma unroll
                for (int n = 0; n < NAp; ++n) {
                    gr[n] = n < NA ? g[n] : 0.0f;
                    gr[NAp + n] = n < NA ? gp[n] * p.udr : 0.0f;
                }
                const Harm<float> ht = harm_of(p.dx * p.ir, p.dy * p.ir, p.dz * p.ir);
                const HarmD<float> hd = unit_tangent(ht, p.drx, p.dry, p.drz, p.udr, p.ir);
#pragma unroll
                for (int mm = 0; mm < kLM; ++mm) {
                    dY[mm] = harm_dvalue(mm, ht, hd);
                    gb[M::oY + mm * GS + at] = harm_value(mm, ht);
                }
            }
            // S += g Y, dS += g' (rhat . dr) Y, then dS += g dY
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (half) {
                    __syncwarp();
                    if (ang) {
#pragma unroll
                        for (int mm = 0; mm < kLM; ++mm) gb[M::oY + mm * GS + at] = dY[mm];
                    }
                }
                __syncwarp();
                for (int q = 0; q < np; ++q) {
                    float2 g[NAp / 2], A[NAp / 2];
#pragma unroll
                    for (int n = 0; n < NAp; n += 4) {
                        const float4 v = ld4(gb + M::oG + q * 2 * NAp + n);
                        g[n / 2] = make_float2(v.x, v.y);
                        g[n / 2 + 1] = make_float2(v.z, v.w);
                        if (!half) {
                            const float4 w = ld4(gb + M::oG + q * 2 * NAp + NAp + n);
                            A[n / 2] = make_float2(w.x, w.y);
                            A[n / 2 + 1] = make_float2(w.z, w.w);
                        }
                    }
#pragma unroll
                    for (int x = 0; x < MPL; ++x) {
                        if (lane + x * G >= kLM) continue;
                        const float Y = gb[M::oY + (lane + x * G) * GS + q];
                        const float2 Y2 = make_float2(Y, Y);
#pragma unroll
                        for (int n = 0; n < NA2; ++n) {
                            if (half) {
                                dS[n][x] = ffma2(g[n], Y2, dS[n][x]);
                            } else {
                                S[n][x] = ffma2(g[n], Y2, S[n][x]);
                                dS[n][x] = ffma2(A[n], Y2, dS[n][x]);
                            }
                        }
                    }
                }
            }
            total += np;
            __syncwarp();
        }
        lanes_rows_sum<G, T * KR>(gb + M::oY, fb, gb + M::oF, lane);
        lanes_rows_sum<G, T * KR>(gb + M::oY, df, gb + M::oDF, lane);
#pragma unroll
        for (int n = 0; n < NA; ++n)
#pragma unroll
            for (int x = 0; x < MPL; ++x)
                if (lane + x * G < kLM) {
                    gS[n * kLM + lane + x * G] = row(S, n, x);
                    gD[n * kLM + lane + x * G] = row(dS, n, x);
                }
        __syncwarp();
        if (first) {
            group_image_ready<C, G>(sm, H, 0);
            first = false;
        }

        // ---- q and dq
        for (int n = lane; n < NR; n += G) {
            float q = 0.0f, dq = 0.0f;
#pragma unroll
            for (int u = 0; u < T; ++u) {
                float c[KR], F[KR], DF[KR];
                load_row<KR>(sm + I::cR() + (ti * T + u) * C::SR + n * KR, c);
                load_row<KR>(gb + M::oF + u * KR, F);
                load_row<KR>(gb + M::oDF + u * KR, DF);
#pragma unroll
                for (int k = 0; k < KR; ++k) {
                    q = fmaf(c[k], F[k], q);
                    dq = fmaf(c[k], DF[k], dq);
                }
            }
            gb[M::oQ + n] = q;
            gb[M::oDQ + n] = dq;
        }
        for (int x = lane; x < NA * 4; x += G) {
            const int n = x >> 2, l = x & 3, m0 = l * (l + 2);
            float q = 0.0f, dq = 0.0f;
            for (int m = m0; m < m0 + 2 * l + 3; ++m) {
                const float s = gS[n * kLM + m], cs = sm[I::clmt() + m] * s;
                q = fmaf(cs, s, q);
                dq = fmaf(2.0f * cs, gD[n * kLM + m], dq);
            }
            gb[M::oQ + NR + x] = q;
            gb[M::oDQ + NR + x] = dq;
        }
        if (C::H4) {
            for (int n = lane; n < NA; n += G) {
                float s2[5], d2[5], J[5], dJ[5];
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    s2[m] = gS[n * kLM + 3 + m];
                    d2[m] = gD[n * kLM + 3 + m];
                }
                gb[M::oQ + NR + NA * 4 + n] = fourbody<float>(s2, nullptr);
                fourbody_jvp(s2, d2, J, dJ);
                float v = 0.0f;
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    v = fmaf(J[m], d2[m], v);
                    gb[M::oJ + 5 * n + m] = J[m];
                    gb[M::oDJ + 5 * n + m] = dJ[m];
                }
                gb[M::oDQ + NR + NA * 4 + n] = v;
            }
        }
        for (int d = D + lane; d < C::DW; d += G) gb[M::oQ + d] = gb[M::oDQ + d] = 0.0f;
        __syncwarp();
        if (valid) {
            for (int o = lane; o < T * KR; o += G) {
                a.fb_out[(size_t)o * N + i] = gb[M::oF + o];
                t.df[(size_t)o * N + i] = gb[M::oDF + o];
            }
            for (int d = lane; d < D; d += G) {
                a.q_out[(size_t)d * N + i] = gb[M::oQ + d];
                t.dq[(size_t)d * N + i] = gb[M::oDQ + d];
            }
        }

        // ---- network and its second-order terms
        const float aE = t.aE[a.cfg[i]];
        for (int h = lane; h < H; h += G) {
            const float* w = sm + I::W(H) + (ti * H + h) * I::WS;
            float z0 = sm[I::b0() + ti * H + h], z1 = 0.0f, u0 = 0.0f, u1 = 0.0f;
#pragma unroll
            for (int d = 0; d < D; d += 4) {
                const float4 q = ld4(gb + M::oQ + d), dq = ld4(gb + M::oDQ + d);
                z0 = fmaf(w[d], q.x, z0);
                u0 = fmaf(w[d], dq.x, u0);
                if (d + 1 < D) { z1 = fmaf(w[d + 1], q.y, z1); u1 = fmaf(w[d + 1], dq.y, u1); }
                if (d + 2 < D) { z0 = fmaf(w[d + 2], q.z, z0); u0 = fmaf(w[d + 2], dq.z, u0); }
                if (d + 3 < D) { z1 = fmaf(w[d + 3], q.w, z1); u1 = fmaf(w[d + 3], dq.w, u1); }
            }
            const float u = u0 + u1, th = tanh_f(z0 + z1), s = 1.0f - th * th;
            const float wh = sm[I::w1(H) + ti * H + h];
            const float c2 = -2.0f * wh * u * th * s;
            if (valid) {
                t.coef[(size_t)h * N + i] = fmaf(aE * wh, s, c2);
                t.coef[(size_t)(H + h) * N + i] = wh * s;
                t.coef[(size_t)(2 * H + h) * N + i] = fmaf(aE, th, s * u);
            }
            gHb[h] = wh * s;
            gHc[h] = c2;
        }
        __syncwarp();
        for (int d = lane; d < D; d += G) {
            const float* w = sm + I::W(H) + ti * H * I::WS + d;
            float p0 = 0.0f, p1 = 0.0f, r0 = 0.0f, r1 = 0.0f;
            int h = 0;
            for (; h + 1 < H; h += 2) {
                const float wa = w[h * I::WS], wb = w[(h + 1) * I::WS];
                p0 = fmaf(wa, gHb[h], p0);
                r0 = fmaf(wa, gHc[h], r0);
                p1 = fmaf(wb, gHb[h + 1], p1);
                r1 = fmaf(wb, gHc[h + 1], r1);
            }
            if (h < H) {
                p0 = fmaf(w[h * I::WS], gHb[h], p0);
                r0 = fmaf(w[h * I::WS], gHc[h], r0);
            }
            const float p = p0 + p1, rho = fmaf(aE, p, r0 + r1);
            gb[M::oP + d] = p;
            gb[M::oRho + d] = rho;
            if (valid) {
                a.p_out[(size_t)d * N + i] = p;
                t.rho[(size_t)d * N + i] = rho;
            }
        }
        __syncwarp();

        // ---- P = dPhi/dS over dS, R = dPhi/d(dS) over S: each lane its own m
#pragma unroll
        for (int x = 0; x < MPL; ++x) {
            const int m = lane + x * G;
            if (m >= kLM) continue;
            const int l = lm_l(m);
            const float c2 = 2.0f * sm[I::clmt() + m];
#pragma unroll
            for (int n = 0; n < NA; ++n) {
                const float pl = gb[M::oP + NR + n * 4 + l - 1], rl = gb[M::oRho + NR + n * 4 + l - 1];
                const float Sv = row(S, n, x);
                float P = c2 * fmaf(rl, Sv, pl * row(dS, n, x)), R = c2 * pl * Sv;
                if (C::H4 && l == 2) {
                    const float p4 = gb[M::oP + NR + NA * 4 + n], r4 = gb[M::oRho + NR + NA * 4 + n];
                    const float J = gb[M::oJ + 5 * n + m - 3];
                    P = fmaf(r4, J, fmaf(p4, gb[M::oDJ + 5 * n + m - 3], P));
                    R = fmaf(p4, J, R);
                }
                gD[n * kLM + m] = P;
                gS[n * kLM + m] = R;
            }
        }
        __syncwarp();
        // lane's (n, k) sums for each species of the neighbour
        constexpr int OPL = (NA * KA + G - 1) / G;
        float bins[T][OPL];
#pragma unroll
        for (int u = 0; u < T; ++u)
#pragma unroll
            for (int x = 0; x < OPL; ++x) bins[u][x] = 0.0f;

        // ---- X_n, Z_n of the angular pairs and the c-gradient bins
        const bool kept = total <= kGroupSlots && cnt_ang <= 65536;
        const int nc = kept ? total : cnt_ang;
        const int ncmax = warp_max(nc);
        for (int c0 = 0; c0 < ncmax; c0 += G) {
            const int c = c0 + lane;
            int s = -1;
            if (c < nc) s = kept ? (int)slots[c] : c;
            TangentPair p;
            p.tj = -1;
            bool in = s >= 0;
            if (in) {
                const int j = a.nbr[(size_t)s * N + i];
                tangent_pair(a, fr, a.pos4[j], t.lam4[j], a.min_image ? 0 : a.shift[(size_t)s * N + i], li, mu, p);
                in = p.d2 < rcA2;
            }
            if (in) {
                float f[KA], fp[KA];
                basis_d<KA>(p.r, irA, f, fp);
#pragma unroll
                for (int k = 0; k < KA; ++k) {
                    gb[M::oY + k * GS + lane] = f[k];
                    gb[M::oY + (KA + k) * GS + lane] = fp[k];
                }
                const Harm<float> ht = harm_of(p.dx * p.ir, p.dy * p.ir, p.dz * p.ir);
                const HarmD<float> hd = unit_tangent(ht, p.drx, p.dry, p.drz, p.udr, p.ir);
                float2 X[NA], Z[NA];
#pragma unroll
                for (int n = 0; n < NA; ++n) X[n] = Z[n] = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int m0 = 0; m0 < kLM; m0 += 4) {
                    float Y[4], dY[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        Y[u] = harm_value(m0 + u, ht);
                        dY[u] = harm_dvalue(m0 + u, ht, hd);
                    }
#pragma unroll
                    for (int n = 0; n < NA; ++n) {
                        const float4 P = ld4(gD + n * kLM + m0), R = ld4(gS + n * kLM + m0);
                        const float2 Y0 = make_float2(Y[0], Y[1]), Y1 = make_float2(Y[2], Y[3]);
                        const float2 R0 = make_float2(R.x, R.y), R1 = make_float2(R.z, R.w);
                        X[n] = ffma2(make_float2(P.x, P.y), Y0, X[n]);
                        X[n] = ffma2(R0, make_float2(dY[0], dY[1]), X[n]);
                        Z[n] = ffma2(R0, Y0, Z[n]);
                        X[n] = ffma2(make_float2(P.z, P.w), Y1, X[n]);
                        X[n] = ffma2(R1, make_float2(dY[2], dY[3]), X[n]);
                        Z[n] = ffma2(R1, Y1, Z[n]);
                    }
                    NEP_SCHED_BARRIER();
                }
#pragma unroll
                for (int n = 0; n < NA; ++n) {
                    gb[M::oY + (2 * KA + n) * GS + lane] = X[n].x + X[n].y;
                    gb[M::oY + (2 * KA + NA + n) * GS + lane] = p.udr * (Z[n].x + Z[n].y);
                }
            }
            const int tq = in ? p.tj : -1;
            __syncwarp();
            const int nq = min(G, ncmax - c0);
            for (int q = 0; q < nq; ++q) {
                const int u = __shfl_sync(0xffffffffu, tq, gbase + q);
                if (u < 0) continue;
#pragma unroll
                for (int x = 0; x < OPL; ++x) {
                    const int o = lane + x * G;
                    if (o >= NA * KA) continue;
                    const int n = o / KA, k = o % KA;
                    const float f = gb[M::oY + k * GS + q], fp = gb[M::oY + (KA + k) * GS + q];
                    const float X = gb[M::oY + (2 * KA + n) * GS + q], Z = gb[M::oY + (2 * KA + NA + n) * GS + q];
#pragma unroll
                    for (int v = 0; v < T; ++v)
                        if (u == v) bins[v][x] = fmaf(f, X, fmaf(fp, Z, bins[v][x]));
                }
            }
            __syncwarp();
        }
        if (valid) {
#pragma unroll
            for (int u = 0; u < T; ++u)
#pragma unroll
                for (int x = 0; x < OPL; ++x)
                    if (lane + x * G < NA * KA) t.bins[(size_t)(u * NA * KA + lane + x * G) * N + i] = bins[u][x];
        }
        __syncwarp();
    }
}

template <class C, int G>
int group_grad_per_sm(int H) {
    return std::max(1, std::min(kGradBlocks, kSmemPerSm / ((int)GroupGradSmem<C, G>::bytes(H) + 1024)));
}
template <class C, int G>
void launch_group_grad_g(const TrainArgs& t, cudaStream_t st) {
    constexpr int NG = kGroupThreads / G;
    launch_pdl(kg_grad<C, G>, persistent_grid((t.e.N + NG - 1) / NG, group_grad_per_sm<C, G>(t.e.H)), kGroupThreads,
               GroupGradSmem<C, G>::bytes(t.e.H), st, t);
}
#endif

}  // namespace nep
