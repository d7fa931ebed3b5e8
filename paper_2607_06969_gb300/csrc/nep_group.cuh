// Evaluation with a group of G lanes per atom, for systems too small to fill
// the GPU with one thread per atom (nep_eval.cuh).  With one thread per atom
// an evaluation of anything up to 10,000 atoms takes the time of one atom's
// serial walk over its ~70 list entries, three times over (25 + 40 + 31 us).
// Here the lanes of a group take
//   the list entries               for the radial sums and the pair forces,
//   the harmonics m                for S_nlm = sum_j g_n Y_m, with the pairs'
//                                  g_n and Y_m handed over in shared memory,
//   the hidden units h, the d      for the network and its adjoint,
// so every phase keeps most lanes busy and no sum crosses lanes but the final
// per-atom totals.  Two kernels make an evaluation:
//   kg_atom    radial sums, angular sums, network, angular pair forces
//              (k_radial + k_angular; the pair's reverse slot gets its force)
//   kg_finish  radial pair forces of both directions, incoming angular forces
// Sums run in a fixed order, so results repeat bitwise.
//
// Measured (one evaluation in a graph, rock salt, 38-30-1 model, the reductions
// included; three one-thread-per-atom kernels and two reductions -> the better
// of G = 8 and 32): 3,686 atoms 106 -> 34 us, 7,200 atoms 106 -> 48.  From about
// 10,000 atoms the radial sums by four lanes and the angular kernel take
// kg_atom's place, and kg_finish alone stays to 50,000 (nep_api.cu has the
// lines): 19,757 atoms 123 -> 77 us.  What bounds the group form: latency at a
// few hundred atoms; from about 10,000 atoms instruction issue (1,840 warp instructions per atom with G = 8, 2,900
// with G = 32) at 16 warps per SM.  G = 4 was slower than 8 at every size
// (its 32 atoms per CTA leave 3 CTAs per SM).
//
// In FP16/BF16 models q, W0 and g = w1 (1 - t^2) are rounded to the 16-bit
// type exactly where the tensor-core kernel rounds them and tanh is the same
// SFU instruction; products are exact in FP32 and accumulate there.
#pragma once
#include <cuda_pipeline.h>

#include "nep_eval.cuh"
#include "nep_mlp_tc.cuh"

namespace nep {

#if defined(__CUDACC__)

constexpr int kGroupThreads = 128;
constexpr int kGroupMinBlocks = 4;               // resident CTAs per SM the registers are held to (128 each)
constexpr size_t kMaxDynSmem = 227 * 1024;       // shared memory of one CTA / of an SM
constexpr int kSmemPerSm = 228 * 1024;
constexpr int kGroupSlots = 96;    // angular pairs whose list slots are kept; beyond, the prefix is walked again

// Shared memory of kg_atom, in floats: the model image, then one block per
// group.
template <class C, int G>
struct GroupSmem {
    static constexpr int NA = C::NA, T = C::T, D = C::D;
    static constexpr int NG = kGroupThreads / G;                 // groups per CTA
    static constexpr int WS = D % 2 ? D : D + 1;                 // odd row stride: lanes on consecutive rows
    static constexpr int NAp = round4(NA);
    static constexpr int FR = T * C::KR > kLM ? T * C::KR : kLM; // rows of the exchange buffer
    static constexpr int GS = G + 1;
    // offsets inside a group's block; F shares the place of the g_n, and the
    // network's vectors that of the exchange buffer, which the sums no longer
    // need by then (with 8 lanes per atom shared memory bounds the resident CTAs)
    static constexpr int oG = 0;                                 // [G][NAp] g_n of a chunk's pairs
    static constexpr int oF = 0;                                 // [T*KR]
    static constexpr int oY = G * NAp > T * C::KR ? G * NAp : round4(T * C::KR);
                                                                 // [FR][GS] Y_m of them, or F partials
    static constexpr int oQ = oY;                                // [DW]
    static constexpr int oP = oQ + C::DW;                        // [DW]
    static constexpr int oJ = oP + C::DW;                        // [NA][5]
    static constexpr int oSg = oJ + round4(NA * 5);              // [H]
    static constexpr int oSl = round4(oY + FR * GS);             // kGroupSlots shorts, if not past oSg + H
    static NEP_HD int slots(int H) { return oSg + round4(H) > oSl ? oSg + round4(H) : oSl; }
    static NEP_HD int S(int H) { return slots(H) + kGroupSlots / 2; }   // [NA][24] S, then dE/dS
    // image
    static NEP_HD int cA2() { return 0; }
    static NEP_HD int cR() { return T * T * C::SA; }
    static NEP_HD int clmt() { return cR() + T * T * C::SR; }
    static NEP_HD int b1() { return clmt() + kLM; }
    static NEP_HD int b0() { return b1() + 4; }
    static NEP_HD int w1(int H) { return b0() + round4(T * H); }
    static NEP_HD int W(int H) { return w1(H) + round4(T * H); }
    static NEP_HD int groups(int H) { return round4(W(H) + T * H * WS); }
    static NEP_HD int group_size(int H) { return S(H) + NA * kLM; }
    static NEP_HD size_t bytes(int H) { return sizeof(float) * (size_t)(groups(H) + NG * group_size(H)); }
};

__device__ __forceinline__ float round16(float x, int kind) {
    if (kind == 1) return __half2float(__float2half_rn(x));
    if (kind == 2) return __bfloat162float(__float2bfloat16_rn(x));
    return x;
}

// sum over the G lanes of a group (fixed butterfly, same bits in every lane)
template <int G>
__device__ __forceinline__ float lanes_sum(float v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int warp_max(int v) { return __reduce_max_sync(0xffffffffu, v); }

// The model image: rows of W0 at an odd stride, cA row-paired, cR as it is.
// The copies are asynchronous: the angular coefficients, which the list walk
// needs, are waited for here, the rest by group_image_ready after the first
// atom's sums.
template <class C, int G>
__device__ void group_load_model(float* sm, const float* prm, int H) {
    using M = GroupSmem<C, G>;
    constexpr int T = C::T, D = C::D;
    const ParamLayout L = param_layout(T, C::NR, C::NA, C::KR, C::KA, C::H4, H);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = kGroupThreads / 32;
    constexpr int nA = C::NA * C::KA, nR = C::NR * C::KR;
    for (int x = threadIdx.x; x < T * T * nA; x += kGroupThreads) {
        const int r = x % nA;
        __pipeline_memcpy_async(sm + M::cA2() + (x / nA) * C::SA + pair_index<C::KA>(r / C::KA, r % C::KA),
                                prm + L.off_cA + x, 4);
    }
    __pipeline_commit();
    for (int x = threadIdx.x; x < T * T * nR; x += kGroupThreads)
        __pipeline_memcpy_async(sm + M::cR() + (x / nR) * C::SR + x % nR, prm + L.off_cR + x, 4);
#pragma unroll 4
    for (int r = warp; r < T * H; r += nw) {
        const int t = r / H;
        const float* src = prm + t * L.mlp_stride + (r - t * H) * D;
        float* dst = sm + M::W(H) + r * M::WS;
#pragma unroll
        for (int d0 = 0; d0 < D; d0 += 32)
            if (d0 + lane < D) __pipeline_memcpy_async(dst + d0 + lane, src + d0 + lane, 4);
    }
    for (int t = 0; t < T; ++t) {
        const float* src = prm + t * L.mlp_stride + H * D;
        for (int h = threadIdx.x; h < H; h += kGroupThreads) {
            __pipeline_memcpy_async(sm + M::b0() + t * H + h, src + h, 4);
            __pipeline_memcpy_async(sm + M::w1(H) + t * H + h, src + H + h, 4);
        }
        if (threadIdx.x == 0) __pipeline_memcpy_async(sm + M::b1() + t, src + 2 * H, 4);
    }
    __pipeline_commit();
    if (C::NA % 2)
        for (int x = threadIdx.x; x < T * T * C::KA; x += kGroupThreads)
            sm[M::cA2() + (x / C::KA) * C::SA + pair_index<C::KA>(C::NA, x % C::KA)] = 0.0f;
    if (threadIdx.x < kLM) sm[M::clmt() + threadIdx.x] = clm(threadIdx.x);
    __pipeline_wait_prior(1);
    __syncthreads();
}

// waits for the whole image; W0 is then rounded to the operand type
template <class C, int G>
__device__ void group_image_ready(float* sm, int H, int kind) {
    using M = GroupSmem<C, G>;
    __pipeline_wait_prior(0);
    __syncthreads();
    if (!kind) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = warp; r < C::T * H; r += kGroupThreads / 32)
        for (int d = lane; d < C::D; d += 32) {
            float* w = sm + M::W(H) + r * M::WS + d;
            *w = round16(*w, kind);
        }
    __syncthreads();
}

// One list entry of an atom: neighbour, species, r_ij and its square
struct GroupPair {
    int j, tj;
    float dx, dy, dz, d2;
};
__device__ __forceinline__ GroupPair group_pair(const EvalArgs& a, const AtomFrame& fr, int i, int s) {
    GroupPair p;
    const size_t at = (size_t)s * a.N + i;
    p.j = a.nbr[at];
    const int sh = a.min_image ? 0 : a.shift[at];
    const float4 pj = a.pos4[p.j];
    p.tj = f2i(pj.w);
    pair_vector(fr.pi, pj, fr.Lx, fr.Ly, fr.Lz, fr.iLx, fr.iLy, fr.iLz, a.min_image, sh, p.dx, p.dy, p.dz);
    p.d2 = norm2(p.dx, p.dy, p.dz);
    return p;
}

// neighbour and image of list entry s, the atom itself past the end
__device__ __forceinline__ void list_entry(const EvalArgs& a, int i, int s, int cnt, bool images, int& j, int& sh) {
    const size_t at = (size_t)s * a.N + i;
    j = s < cnt ? a.nbr[at] : i;
    sh = images && s < cnt ? a.shift[at] : 0;
}

// Phases of one atom shared with the training kernels: radial sums F (shared
// memory) and S_nlm (lane m, m + G, ... keeps S[.][m]) over the list.
// Returns the number of angular pairs; their slots are in the group's list.
template <class C, int G>
__device__ int group_sums(const EvalArgs& a, const float* sm, float* gb, float* gS, unsigned short* slots,
                          const AtomFrame& fr, int i, int cnt, int cnt_ang, int lane,
                          float (&S)[C::NA][(kLM + G - 1) / G]) {
    using M = GroupSmem<C, G>;
    constexpr int NA = C::NA, KR = C::KR, KA = C::KA, T = C::T, MPL = (kLM + G - 1) / G;
    const float rcR2 = a.rc_rad * a.rc_rad, rcA2 = a.rc_ang * a.rc_ang;
    const float irR = 1.0f / a.rc_rad, irA = 1.0f / a.rc_ang;
    const int gbase = (threadIdx.x & 31) & ~(G - 1);
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u);
    float fb[T][KR];
#pragma unroll
    for (int t = 0; t < T; ++t)
#pragma unroll
        for (int k = 0; k < KR; ++k) fb[t][k] = 0.0f;
    constexpr int NA2 = (NA + 1) / 2;
    float2 S2[NA2][MPL];                 // rows n two by two (paired FMAs)
#pragma unroll
    for (int n = 0; n < NA2; ++n)
#pragma unroll
        for (int x = 0; x < MPL; ++x) S2[n][x] = make_float2(0.0f, 0.0f);
    const int cmax = warp_max(cnt), amax = warp_max(cnt_ang);
    int total = 0;
    // a chunk's entries are read one chunk ahead, the indices and images two
    const int N = a.N;
    const bool images = !a.min_image;
    int j1 = i, j2 = i, h1 = 0, h2 = 0;
    list_entry(a, i, lane, cnt, images, j1, h1);
    list_entry(a, i, lane + G, cnt, images, j2, h2);
    float4 p1 = a.pos4[j1];
    for (int s0 = 0; s0 < cmax; s0 += G) {
        const int s = s0 + lane;
        const bool act = s < cnt;
        const float4 pj = p1;
        const int sh = h1;
        j1 = j2;
        h1 = h2;
        p1 = a.pos4[j1];
        list_entry(a, i, s + 2 * G, cnt, images, j2, h2);
        GroupPair p;
        p.tj = f2i(pj.w);
        pair_vector(fr.pi, pj, fr.Lx, fr.Ly, fr.Lz, fr.iLx, fr.iLy, fr.iLz, a.min_image, sh, p.dx, p.dy, p.dz);
        p.d2 = act ? norm2(p.dx, p.dy, p.dz) : 1.0f;
        float r, ir;
        dist_rinv(p.d2, r, ir);
        if (act && p.d2 < rcR2) {
            float f[KR];
            basis<KR>(r, irR, f);
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const float w = (p.tj == t) ? 1.0f : 0.0f;
#pragma unroll
                for (int k = 0; k + 1 < KR; k += 2) {
                    const float2 v =
                        ffma2(make_float2(w, w), make_float2(f[k], f[k + 1]), make_float2(fb[t][k], fb[t][k + 1]));
                    fb[t][k] = v.x;
                    fb[t][k + 1] = v.y;
                }
                if (KR % 2) fb[t][KR - 1] = fmaf(w, f[KR - 1], fb[t][KR - 1]);
            }
        }
        if (s0 >= amax) continue;
        const bool ang = act && s < cnt_ang && p.d2 < rcA2;
        const unsigned m = (__ballot_sync(0xffffffffu, ang) >> gbase) & gmask;
        const int np = __popc(m);
        if (ang) {
            const int at = __popc(m & ((1u << lane) - 1u));
            if (total + at < kGroupSlots) slots[total + at] = (unsigned short)s;
            float f[KA], g[NA];
            basis<KA>(r, irA, f);
            contract_pairs<NA, KA>(sm + M::cA2() + (fr.ti * T + p.tj) * C::SA, f, g);
#pragma unroll
            for (int n = 0; n < M::NAp; ++n) gb[M::oG + at * M::NAp + n] = n < NA ? g[n] : 0.0f;
            const Harm<float> ht = harm_of(p.dx * ir, p.dy * ir, p.dz * ir);
#pragma unroll
            for (int mm = 0; mm < kLM; ++mm) gb[M::oY + mm * M::GS + at] = harm_value(mm, ht);
        }
        __syncwarp();
        for (int q = 0; q < np; ++q) {
            float2 g[M::NAp / 2];
#pragma unroll
            for (int n = 0; n < M::NAp; n += 4) {
                const float4 v = ld4(gb + M::oG + q * M::NAp + n);
                g[n / 2] = make_float2(v.x, v.y);
                g[n / 2 + 1] = make_float2(v.z, v.w);
            }
#pragma unroll
            for (int x = 0; x < MPL; ++x) {
                const int mm = lane + x * G;
                if (mm < kLM) {
                    const float Y = gb[M::oY + mm * M::GS + q];
#pragma unroll
                    for (int n = 0; n < NA2; ++n) S2[n][x] = ffma2(g[n], make_float2(Y, Y), S2[n][x]);
                }
            }
        }
        total += np;
        __syncwarp();
    }
    // F[t][k]: the lanes' partial sums, added in lane order
#pragma unroll
    for (int t = 0; t < T; ++t)
#pragma unroll
        for (int k = 0; k < KR; ++k) gb[M::oY + (t * KR + k) * M::GS + lane] = fb[t][k];
    __syncwarp();
    for (int o = lane; o < T * KR; o += G) {
        float v0 = 0.0f, v1 = 0.0f;
#pragma unroll
        for (int l = 0; l < G; l += 2) {
            v0 += gb[M::oY + o * M::GS + l];
            v1 += gb[M::oY + o * M::GS + l + 1];
        }
        gb[M::oF + o] = v0 + v1;
    }
#pragma unroll
    for (int n = 0; n < NA; ++n)
#pragma unroll
        for (int x = 0; x < MPL; ++x) {
            S[n][x] = n % 2 ? S2[n / 2][x].y : S2[n / 2][x].x;
            if (lane + x * G < kLM) gS[n * kLM + lane + x * G] = S[n][x];
        }
    __syncwarp();
    return total;
}

// q (rounded to the network's operand type), the 4-body gradients J, then
// E_i (returned in every lane) and p = dE/dq, all in the group's block
template <class C, int G>
__device__ float group_network(const float* sm, float* gb, const float* gS, int H, int ti, int lane, int kind) {
    using M = GroupSmem<C, G>;
    constexpr int NR = C::NR, NA = C::NA, KR = C::KR, T = C::T, D = C::D;
    for (int n = lane; n < NR; n += G) {
        float q = 0.0f;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            float c[KR], F[KR];
            load_row<KR>(sm + M::cR() + (ti * T + t) * C::SR + n * KR, c);
            load_row<KR>(gb + M::oF + t * KR, F);
#pragma unroll
            for (int k = 0; k < KR; ++k) q = fmaf(c[k], F[k], q);
        }
        gb[M::oQ + n] = round16(q, kind);
    }
    for (int x = lane; x < NA * 4; x += G) {
        const int n = x >> 2, l = x & 3;               // l + 1 is the degree; its harmonics start at (l+1)^2 - 1
        const int m0 = l * (l + 2);
        float q = 0.0f;
        for (int m = m0; m < m0 + 2 * l + 3; ++m) {
            const float s = gS[n * kLM + m];
            q = fmaf(sm[M::clmt() + m] * s, s, q);
        }
        gb[M::oQ + NR + x] = round16(q, kind);
    }
    if (C::H4) {
        for (int n = lane; n < NA; n += G) {
            float s2[5], J[5];
#pragma unroll
            for (int m = 0; m < 5; ++m) s2[m] = gS[n * kLM + 3 + m];
            gb[M::oQ + NR + NA * 4 + n] = round16(fourbody(s2, J), kind);
#pragma unroll
            for (int m = 0; m < 5; ++m) gb[M::oJ + n * 5 + m] = J[m];
        }
    }
    for (int d = D + lane; d < C::DW; d += G) gb[M::oQ + d] = 0.0f;
    __syncwarp();
    float E = 0.0f;
    for (int h = lane; h < H; h += G) {
        const float* w = sm + M::W(H) + (ti * H + h) * M::WS;
        float z0 = sm[M::b0() + ti * H + h], z1 = 0.0f, z2 = 0.0f, z3 = 0.0f;
#pragma unroll
        for (int d = 0; d < D; d += 4) {
            const float4 q = ld4(gb + M::oQ + d);
            z0 = fmaf(w[d], q.x, z0);
            if (d + 1 < D) z1 = fmaf(w[d + 1], q.y, z1);
            if (d + 2 < D) z2 = fmaf(w[d + 2], q.z, z2);
            if (d + 3 < D) z3 = fmaf(w[d + 3], q.w, z3);
        }
        const float z = (z0 + z1) + (z2 + z3);
        const float t = kind ? tanh_sfu(z) : tanh_f(z);
        const float wh = sm[M::w1(H) + ti * H + h];
        E = fmaf(wh, t, E);
        gb[M::oSg + h] = round16(wh * (1.0f - t * t), kind);
    }
    E = lanes_sum<G>(E) + sm[M::b1() + ti];
    __syncwarp();
    for (int d = lane; d < D; d += G) {
        const float* w = sm + M::W(H) + ti * H * M::WS + d;
        float p0 = 0.0f, p1 = 0.0f;
        int h = 0;
        for (; h + 3 < H; h += 4) {
            const float4 g = ld4(gb + M::oSg + h);
            p0 = fmaf(w[h * M::WS], g.x, p0);
            p1 = fmaf(w[(h + 1) * M::WS], g.y, p1);
            p0 = fmaf(w[(h + 2) * M::WS], g.z, p0);
            p1 = fmaf(w[(h + 3) * M::WS], g.w, p1);
        }
        for (; h < H; ++h) p0 = fmaf(w[h * M::WS], gb[M::oSg + h], p0);
        gb[M::oP + d] = p0 + p1;
    }
    __syncwarp();
    return E;
}

template <class C, int G>
__global__ void __launch_bounds__(kGroupThreads, kGroupMinBlocks) kg_atom(const EvalArgs a) {
    using M = GroupSmem<C, G>;
    constexpr int NR = C::NR, NA = C::NA, KR = C::KR, KA = C::KA, T = C::T, MPL = (kLM + G - 1) / G;
    extern __shared__ float sm[];
    const int N = a.N, H = a.H, kind = a.q16_kind;
    group_load_model<C, G>(sm, a.params, H);      // older than the kernel before this one
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x % G, group = threadIdx.x / G;
    float* gb = sm + M::groups(H) + group * M::group_size(H);
    float* gS = gb + M::S(H);
    unsigned short* slots = reinterpret_cast<unsigned short*>(gb + M::slots(H));
    bool first = true;
    const float rcA2 = a.rc_ang * a.rc_ang, irA = 1.0f / a.rc_ang;
    const int ntiles = (N + M::NG - 1) / M::NG;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int ia = tile * M::NG + group;
        const bool valid = ia < N;
        const int i = valid ? ia : N - 1;
        const AtomFrame fr = atom_frame(a, i);
        const int ti = fr.ti;
        const int cnt = valid ? a.cnt[i] : 0, cnt_ang = valid ? a.cnt_ang[i] : 0;
        float S[NA][MPL];
        const int total = group_sums<C, G>(a, sm, gb, gS, slots, fr, i, cnt, cnt_ang, lane, S);
        if (first) {
            group_image_ready<C, G>(sm, H, kind);
            first = false;
        }
        const float E = group_network<C, G>(sm, gb, gS, H, ti, lane, kind);
        if (valid) {
            if (lane == 0) a.e_atom[i] = E;
            // projected radial adjoint Pr[i][t][k] = sum_n p_n cR[ti][t][n][k]
            for (int o = lane; o < T * KR; o += G) {
                const float* c = sm + M::cR() + (ti * T + o / KR) * C::SR + o % KR;
                float v = 0.0f;
#pragma unroll
                for (int n = 0; n < NR; ++n) v = fmaf(gb[M::oP + n], c[n * KR], v);
                a.Pr[(size_t)i * T * KR + o] = v;
            }
        }
        // dE/dS in place of S: each lane its own m
#pragma unroll
        for (int x = 0; x < MPL; ++x) {
            const int m = lane + x * G;
            if (m < kLM) {
                const int l = lm_l(m);
                const float c2 = 2.0f * sm[M::clmt() + m];
#pragma unroll
                for (int n = 0; n < NA; ++n) {
                    float v = c2 * gb[M::oP + NR + n * 4 + l - 1] * S[n][x];
                    if (C::H4 && l == 2) v = fmaf(gb[M::oP + NR + NA * 4 + n], gb[M::oJ + n * 5 + m - 3], v);
                    gS[n * kLM + m] = v;
                }
            }
        }
        __syncwarp();
        // angular pair forces, the owner's sums and the scatter to the reverse slot
        const bool kept = total <= kGroupSlots && cnt_ang <= 65536;
        const int nc = kept ? total : cnt_ang;
        float acc[12];                                   // F, W
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = 0.0f;
        for (int c = lane; c < nc; c += G) {
            const int s = kept ? (int)slots[c] : c;
            const GroupPair p = group_pair(a, fr, i, s);
            if (!(p.d2 < rcA2)) continue;
            const int addr = a.rev[(size_t)s * N + i] * N + p.j;
            float r, ir;
            dist_rinv(p.d2, r, ir);
            float g[NA], gp[NA];
            {
                float f[KA], fp[KA];
                basis_d<KA>(r, irA, f, fp);
                const float* c2 = sm + M::cA2() + (ti * T + p.tj) * C::SA;
                contract_pairs<NA, KA>(c2, f, g);
                contract_pairs<NA, KA>(c2, fp, gp);
            }
            const Harm<float> ht = harm_of(p.dx * ir, p.dy * ir, p.dz * ir);
            HarmSums<float> hs(ht);
#pragma unroll
            for (int m0 = 0; m0 < kLM; m0 += 4) {
                float2 am[2] = {}, bm[2] = {};
#pragma unroll
                for (int n = 0; n < NA; ++n) {
                    const float4 s4 = ld4(gS + n * kLM + m0);
                    const float2 g2 = make_float2(g[n], g[n]), q2 = make_float2(gp[n], gp[n]);
                    const float2 s0 = make_float2(s4.x, s4.y), s1 = make_float2(s4.z, s4.w);
                    am[0] = ffma2(s0, g2, am[0]);
                    am[1] = ffma2(s1, g2, am[1]);
                    bm[0] = ffma2(s0, q2, bm[0]);
                    bm[1] = ffma2(s1, q2, bm[1]);
                }
                hs.add(m0, ht, am[0].x, bm[0].x);
                hs.add(m0 + 1, ht, am[0].y, bm[0].y);
                hs.add(m0 + 2, ht, am[1].x, bm[1].x);
                hs.add(m0 + 3, ht, am[1].y, bm[1].y);
                NEP_SCHED_BARRIER();
            }
            float fx, fy, fz;
            hs.force(ht, ir, fx, fy, fz);
            a.fin[addr] = make_float4(fx, fy, fz, 0.0f);
            acc[0] += fx; acc[1] += fy; acc[2] += fz;
            acc[3] -= fx * p.dx; acc[4] -= fx * p.dy; acc[5] -= fx * p.dz;
            acc[6] -= fy * p.dx; acc[7] -= fy * p.dy; acc[8] -= fy * p.dz;
            acc[9] -= fz * p.dx; acc[10] -= fz * p.dy; acc[11] -= fz * p.dz;
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            acc[k] = lanes_sum<G>(acc[k]);
            if (valid && lane == k % G) {
                if (k < 3) a.fpart[(size_t)k * N + i] = acc[k];
                else a.wat[(size_t)(k - 3) * N + i] = acc[k];
            }
        }
    }
}

// F_i and the per-atom virial: radial pair forces of both directions from the
// projected adjoints of both atoms, the owner's angular part, and the incoming
// angular slots (those whose pair lies inside rc_ang); in MD also the closing
// half kick, which saves small systems its launch.  Bound by the latency of a
// lane's entries: images are read with their indices, two entries ahead (48
// replicas, ten FP16 MD steps 2,019 -> 1,965 us with k_radial_split's).  Rows
// and slots also fetched an entry ahead measured slower (12,442 atoms 56.7 ->
// 64.4 us an evaluation: more registers).
template <class C, int G>
__global__ void __launch_bounds__(kGroupThreads) kg_finish(const EvalArgs a, const FinishArgs fa) {
    constexpr int KR = C::KR, T = C::T, NG = kGroupThreads / G;
    __shared__ __align__(16) float Pi[NG][round4(T * KR)];
    const int N = a.N, lane = threadIdx.x % G, group = threadIdx.x / G;
    const int ia = blockIdx.x * NG + group;
    const bool valid = ia < N;
    const int i = valid ? ia : N - 1;
    const AtomFrame fr = atom_frame(a, i);
    const int cnt = valid ? a.cnt[i] : 0, cnt_ang = a.cnt_ang[i];
    const float rcR2 = a.rc_rad * a.rc_rad, rcA2 = a.rc_ang * a.rc_ang, irR = 1.0f / a.rc_rad;
    float acc[9];                                        // F, then xx yy zz xy xz yz
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[k] = 0.0f;
    // positions are read one entry ahead, the indices and images two
    const bool images = !a.min_image;
    int j0 = i, j1 = i, h0 = 0, h1 = 0;
    list_entry(a, i, lane, cnt, images, j0, h0);
    list_entry(a, i, lane + G, cnt, images, j1, h1);
    float4 p0 = a.pos4[j0];
    pdl_wait();                              // the list and the positions are older than kg_atom
    pdl_trigger();
    const float* Pr = after_wait(a.Pr);
    for (int o = lane; o < T * KR; o += G) Pi[group][o] = Pr[(size_t)i * T * KR + o];
    __syncwarp();
    for (int s = lane; s < cnt; s += G) {
        GroupPair p;
        p.j = j0;
        const float4 pj = p0;
        const int sh = h0;
        j0 = j1;
        h0 = h1;
        p0 = a.pos4[j0];
        list_entry(a, i, s + 2 * G, cnt, images, j1, h1);
        p.tj = f2i(pj.w);
        pair_vector(fr.pi, pj, fr.Lx, fr.Ly, fr.Lz, fr.iLx, fr.iLy, fr.iLz, a.min_image, sh, p.dx, p.dy, p.dz);
        p.d2 = norm2(p.dx, p.dy, p.dz);
        if (!(p.d2 < rcR2)) continue;
        float Pj[KR];
        const float* row = Pr + ((size_t)p.j * T + fr.ti) * KR;
        if (KR % 8 == 0) {
#pragma unroll
            for (int k = 0; k < KR; k += 8) load8(row + k, Pj + k);
        } else {
#pragma unroll
            for (int k = 0; k < KR; ++k) Pj[k] = row[k];
        }
        float4 g = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (s < cnt_ang && p.d2 < rcA2) g = a.fin[(size_t)s * N + i];
        float r, ir;
        dist_rinv(p.d2, r, ir);
        float f[KR], fp[KR], pi[KR];
        basis_d<KR>(r, irR, f, fp);
        load_row<KR>(&Pi[group][p.tj * KR], pi);
        float dEi = 0.0f, dEj = 0.0f;
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            dEi = fmaf(pi[k], fp[k], dEi);
            dEj = fmaf(Pj[k], fp[k], dEj);
        }
        const float tot = (dEi + dEj) * ir, w = dEi * ir;
        acc[0] = fmaf(tot, p.dx, acc[0] - g.x);
        acc[1] = fmaf(tot, p.dy, acc[1] - g.y);
        acc[2] = fmaf(tot, p.dz, acc[2] - g.z);
        const float wx = w * p.dx, wy = w * p.dy, wz = w * p.dz;
        acc[3] = fmaf(wx, p.dx, acc[3]);
        acc[4] = fmaf(wy, p.dy, acc[4]);
        acc[5] = fmaf(wz, p.dz, acc[5]);
        acc[6] = fmaf(wx, p.dy, acc[6]);
        acc[7] = fmaf(wx, p.dz, acc[7]);
        acc[8] = fmaf(wy, p.dz, acc[8]);
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[k] = lanes_sum<G>(acc[k]);
    if (!valid) return;
    if (lane == 0) {
        float im = fa.inv_mass[0];
#pragma unroll
        for (int t = 1; t < kMaxTypes; ++t) im = fr.ti == t ? fa.inv_mass[t] : im;
        const float s = fa.half_dt * im;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t at = (size_t)c * N + i;
            const float F = a.fpart[at] + acc[c];
            fa.force[at] = F;
            if (fa.vel) fa.vel[at] = fmaf(s, F, fa.vel[at]);
        }
        if (fa.e_out) fa.e_out[i] = a.e_atom[i];
    }
    const float Wsym[9] = {acc[3], acc[6], acc[7], acc[6], acc[4], acc[8], acc[7], acc[8], acc[5]};
#pragma unroll
    for (int c = 0; c < 9; ++c)
        if (lane == c % G) a.wat[(size_t)c * N + i] -= Wsym[c];
}

// whether a model of H hidden units fits kg_atom's shared memory
template <class C>
bool group_fits_t(int H) { return GroupSmem<C, 32>::bytes(H) <= kMaxDynSmem && GroupSmem<C, 8>::bytes(H) <= kMaxDynSmem; }

// The grid of kg_atom follows from the registers and the shared memory of H
// hidden units, so it is computed for each launch's own model.
template <class C, int G>
int group_per_sm(int H) {
    const int smem_blk = (int)GroupSmem<C, G>::bytes(H) + 1024;
    return std::max(1, std::min(kGroupMinBlocks, kSmemPerSm / smem_blk));
}
template <class C, int G>
cudaError_t group_init_g() {
    return cudaFuncSetAttribute(kg_atom<C, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynSmem);
}

template <class C, int G>
cudaError_t launch_group_g(const EvalArgs& a, cudaStream_t st) {
    constexpr int NG = kGroupThreads / G;
    return launch_pdl(kg_atom<C, G>, persistent_grid((a.N + NG - 1) / NG, group_per_sm<C, G>(a.H)), kGroupThreads,
                      GroupSmem<C, G>::bytes(a.H), st, a);
}
template <class C, int G>
void launch_group_finish_g(const EvalArgs& a, const FinishArgs& f, cudaStream_t st) {
    constexpr int NG = kGroupThreads / G;
    launch_pdl(kg_finish<C, G>, (a.N + NG - 1) / NG, kGroupThreads, 0, st, a, f);
}

template <class C>
cudaError_t group_init_t(int H) {
    (void)H;
    cudaError_t e;
    sm_count();
    if ((e = group_init_g<C, 32>())) return e;
    return group_init_g<C, 8>();
}
template <class C>
cudaError_t launch_group_t(const EvalArgs& a, cudaStream_t st, int G) {
    return G == 32 ? launch_group_g<C, 32>(a, st) : launch_group_g<C, 8>(a, st);
}
template <class C>
cudaError_t launch_group_finish_t(const EvalArgs& a, const FinishArgs& f, int max_chunks, cudaStream_t st, int G) {
    if (G == 32) launch_group_finish_g<C, 32>(a, f, st);
    else if (G == 16) launch_group_finish_g<C, 16>(a, f, st);
    else launch_group_finish_g<C, 8>(a, f, st);
    return launch_totals(a, f, max_chunks, st);
}
#endif

}  // namespace nep
