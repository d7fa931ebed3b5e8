// Model-independent kernels of libnep: input packing, the cell-list
// neighbour build, the deterministic force gather with FP64 reductions, and
// the velocity-Verlet updates.
#include <algorithm>

#include <cuda_runtime.h>

#include "nep_device.cuh"
#include "nep_internal.h"

namespace nep {

namespace {

__device__ __forceinline__ void set_flag(int* status, int k) {
    if (status) atomicOr(status + k, 1);
}

// binary search: largest b with off[b] <= x, for off[0..B]
__device__ __forceinline__ int find_segment(const int* off, int B, int x) {
    int lo = 0, hi = B;   // invariant off[lo] <= x < off[hi]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (off[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// ------------------------------------------------------------------ packing
// Exclusive scan of the configurations' chunk counts by one CTA (any multiple
// of 32 threads up to 1,024), and the reduction tickets cleared.
__device__ void chunk_plan_block(const int* atom_off, int B, int* chunk_start, int* ticket) {
    if (B <= 32) {                       // one warp, no block-wide waits
        const int b = threadIdx.x;
        if (b >= 32) return;
        int x = b < B ? (atom_off[b + 1] - atom_off[b] + kChunk - 1) / kChunk : 0;
        const int v = x;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (b >= o) x += y;
        }
        if (b < B) {
            chunk_start[b] = x - v;
            if (ticket) ticket[b] = 0;
        }
        if (b == 31) chunk_start[B] = x;
        return;
    }
    __shared__ int carry;
    __shared__ int warp_sums[32];
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < B; base += blockDim.x) {
        const int b = base + threadIdx.x;
        int v = 0;
        if (b < B) {
            const int n = atom_off[b + 1] - atom_off[b];
            v = (n + kChunk - 1) / kChunk;
            if (ticket) ticket[b] = 0;
        }
        // block inclusive scan
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sums[w] = x;
        __syncthreads();
        if (w == 0) {
            int s = (lane < (int)(blockDim.x >> 5)) ? warp_sums[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            warp_sums[lane] = s;
        }
        __syncthreads();
        const int incl = x + (w > 0 ? warp_sums[w - 1] : 0);
        if (b < B) chunk_start[b] = carry + incl - v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry += incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) chunk_start[B] = carry;
}

__global__ void __launch_bounds__(1024) k_chunk_plan(const int* __restrict__ atom_off, int B, int* chunk_start,
                                                     int* ticket) {
    chunk_plan_block(atom_off, B, chunk_start, ticket);
}

__device__ __forceinline__ void pack_atom(float x, float y, float z, int t, const int* atom_off, int B, int T, int i,
                                          float4* pos4, int* cfg, int* status) {
    if (t < 0 || t >= T) {
        set_flag(status, 3);
        t = 0;
    }
    if (!(isfinite(x) && isfinite(y) && isfinite(z))) set_flag(status, 3);
    pos4[i] = make_float4(x, y, z, __int_as_float(t));
    cfg[i] = find_segment(atom_off, B, i);
}

// positions, species and configuration of each atom in the kernels' layout;
// with chunk_start, one more block plans the reduction chunks meanwhile
__global__ void __launch_bounds__(256) k_pack(const float* pos, const int* type,
                                              const int* atom_off, int N, int B, int T, float4* pos4,
                                              int* cfg, int* status, int* chunk_start, int* ticket) {
    pdl_wait();
    pdl_trigger();
    if (chunk_start && blockIdx.x == gridDim.x - 1) {
        chunk_plan_block(atom_off, B, chunk_start, ticket);
        return;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) pack_atom(pos[i], pos[N + i], pos[2 * (size_t)N + i], type[i], atom_off, B, T, i, pos4, cfg, status);
}

constexpr int kRedThreads = 256;

// (hi, lo) += x without rounding loss: Knuth's two-sum, in FP32.  The pair
// carries about 48 significant bits, so the per-thread and per-warp stages
// below are as exact as FP64 while running on the FP32 pipes (GB300 issues
// FP64 at a small fraction of the FP32 rate).
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x) {
    const float s = __fadd_rn(hi, x);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
    hi = s;
    lo = __fadd_rn(lo, err);
}

// E and virial of every configuration, one CTA per reduction chunk (atoms of
// one configuration) and one warp per component (E and the nine of V): each
// lane sums a fixed subset of the chunk's atoms in two-sum pairs, a fixed warp
// tree joins them, and the CTA that finishes a configuration's last chunk sums
// the chunks' FP64 partials in a fixed order (lanes take chunks l, l + 32, ...;
// a fixed tree).  Which CTA does that varies, what it computes does not.
// With a warp per component no sum crosses warps; the former two kernels (all
// ten components in every thread, then one CTA per configuration) took 4.4 +
// 5.8 us at 194 atoms and 21.9 + 8.8 us at 900,000.
constexpr int kTotalsThreads = 320;
__global__ void __launch_bounds__(kTotalsThreads) k_totals(const EvalArgs a, FinishArgs f) {
    const int k = blockIdx.x;
    const int B = a.B, N = a.N;
    const int total = f.chunk_start[B];
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    if (k >= total) {
        pdl_wait();
        pdl_trigger();
        // the blocks past the last chunk (at least one per empty configuration)
        // write the zeros of configurations without atoms
        for (int b = k - total; b < B; b += gridDim.x - total)
            if (f.chunk_start[b] == f.chunk_start[b + 1] && lane == 0) {
                if (c == 0) {
                    if (f.e_tot) f.e_tot[b] = 0.0;
                } else if (f.virial) {
                    f.virial[(size_t)b * 9 + c - 1] = 0.0;
                }
            }
        return;
    }
    const int b = find_segment(f.chunk_start, B, k);
    const int k0 = f.chunk_start[b], nk = f.chunk_start[b + 1] - k0;
    const int a0 = f.atom_off[b] + (k - k0) * kChunk;
    const int a1 = min(min(f.atom_off[b + 1], a0 + kChunk), f.n_owned);
    pdl_wait();                          // the plan is older than the kernel before this one (launch_totals)
    pdl_trigger();
    const float* src = c == 0 ? a.e_atom : a.wat + (size_t)(c - 1) * N;
    float h = 0.0f, l = 0.0f;
    constexpr int kAhead = 16;           // loads in flight per lane
    for (int i0 = a0 + lane; i0 < a1; i0 += 32 * kAhead) {
        float x[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) x[u] = i0 + 32 * u < a1 ? src[i0 + 32 * u] : 0.0f;
#pragma unroll
        for (int u = 0; u < kAhead; ++u) two_sum_add(h, l, x[u]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_down_sync(0xffffffffu, h, o);
        const float ol = __shfl_down_sync(0xffffffffu, l, o);
        two_sum_add(h, l, oh);
        l = __fadd_rn(l, ol);
    }
    double v = (double)h + (double)l;
    if (nk > 1) {
        if (lane == 0) {
            f.partial[(size_t)k * 10 + c] = v;
            __threadfence();
        }
        __shared__ int last;
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(f.ticket + b, 1) == nk - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (threadIdx.x == 0) f.ticket[b] = 0;   // ready for another reduction over the same plan
        v = 0.0;
        for (int q = lane; q < nk; q += 32) v += __ldcg(f.partial + (size_t)(k0 + q) * 10 + c);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    if (lane == 0) {
        if (c == 0) {
            if (f.e_tot) f.e_tot[b] = v;
        } else if (f.virial) {
            f.virial[(size_t)b * 9 + c - 1] = v;
        }
    }
}

// ------------------------------------------------------- neighbour build
// Cells per edge: floor(L / ((rc + 1e-3) / kCellDiv)) (at least 1), reduced
// while the cell count of a configuration exceeds 2 N_b + 27.  The stencil
// half-width is the number of cells needed to reach rc + 1e-3 (kCellDiv for
// large boxes).  Cells of a third of the cutoff offer (7/3)^3 = 12.7
// cutoff-sized cells' worth of candidates before the per-row cut below
// (half the cutoff: 15.6; the whole cutoff: 27); measured at 900k atoms, the
// rebuild takes 1.31 ms with thirds and 1.54 ms with halves.  An atom in cell
// c sees cells c + d, d in [-half, half], with image shift floor((c + d) /
// nc): every (j, image) within the cutoff is visited exactly once.
constexpr float kCellMargin = 1e-3f;
// margin (A) on the list cutoff when cells beyond it are skipped
#ifndef NEP_PRUNE_MARGIN
#define NEP_PRUNE_MARGIN 0.01f
#endif
constexpr float kPruneMargin = NEP_PRUNE_MARGIN;
constexpr int kCellDiv = 3;
// per-atom row starts of the angular prefix, for the reverse-slot search:
// stencils of up to kMaxRows (x, y) rows, angular capacity below 256; one
// atom's starts take kRowStride bytes of the workspace
constexpr int kMaxRows = (2 * kCellDiv + 1) * (2 * kCellDiv + 1);
static_assert(kMaxRows < kRowStride, "row starts must fit one atom's stride");

// plan of one configuration; base holds its cell count until the prefix is taken.
// The build kernel is chosen by the host's copy of the boxes.  A box on the
// device so much thinner that the cutoff reaches over more than max_images of
// it (0: any number) is invalid input: its stencil has no rows (-1 of them;
// k_build_warp alone sets a limit).
__device__ CellPlan cell_plan_of(const float* box, const int* atom_off, int b, float rc, int max_images, int* status) {
    const int nb = atom_off[b + 1] - atom_off[b];
    float L[3] = {box[3 * b], box[3 * b + 1], box[3 * b + 2]};
    int nc[3];
    for (int d = 0; d < 3; ++d) {
        if (!(L[d] > 0.0f) || !isfinite(L[d])) {
            set_flag(status, 3);
            L[d] = 1.0f;
        }
        const float r = floorf(L[d] / ((rc + kCellMargin) / (float)kCellDiv));
        nc[d] = r < 1.0f ? 1 : (r > 1024.0f ? 1024 : (int)r);
    }
    // The edge with the most cells loses one until the count fits.  That passes
    // through min(nc, t) for every t that is still too many, so where there are
    // many steps those down to the least such t are taken at once: one by one
    // they took some 240 us for 5,000 atoms in a box of 2,500 A.
    const long long cap = 2LL * nb + 27;
    auto cells = [&](int t) { return (long long)min(nc[0], t) * min(nc[1], t) * min(nc[2], t); };
    int t = max(nc[0], max(nc[1], nc[2])) - 8;
    if (t > 1 && cells(t) > cap) {
        int fits = 1;                               // cells(fits) <= cap < cells(t)
        while (t - fits > 1) {
            const int mid = (fits + t) >> 1;
            if (cells(mid) > cap) t = mid; else fits = mid;
        }
        for (int d = 0; d < 3; ++d) nc[d] = min(nc[d], t);
    }
    while ((long long)nc[0] * nc[1] * nc[2] > cap) {
        const bool y = nc[1] > nc[0], z = nc[2] > max(nc[0], nc[1]);
        nc[2] -= z;
        nc[1] -= y && !z;
        nc[0] -= !y && !z;
    }
    CellPlan p;
    for (int d = 0; d < 3; ++d) {
        p.nc[d] = nc[d];
        const float cs = L[d] / (float)nc[d];
        p.half[d] = (int)ceilf((rc + kCellMargin) / cs);
        if (p.half[d] < 1) p.half[d] = 1;
    }
    if (max_images && (p.half[0] > max_images * p.nc[0] || p.half[1] > max_images * p.nc[1] ||
                       p.half[2] > max_images * p.nc[2])) {
        set_flag(status, 3);
        p.half[0] = -1;
        p.half[1] = p.half[2] = 0;
    }
    p.base = nc[0] * nc[1] * nc[2];
    p.pad = 0;
    return p;
}

__global__ void k_cell_plan(const float* __restrict__ box, const int* __restrict__ atom_off, int B,
                            float rc, int max_images, CellPlan* plan, int* status) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) plan[b] = cell_plan_of(box, atom_off, b, rc, max_images, status);
}

__global__ void k_plan_scan(CellPlan* plan, int B) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int acc = 0;
    for (int b = 0; b < B; ++b) {
        const int c = plan[b].base;
        plan[b].base = acc;
        acc += c;
    }
}

__device__ __forceinline__ void cell_coords(const CellPlan& p, float x, float y, float z,
                                            const float* L, int* c) {
    const float v[3] = {x, y, z};
    for (int d = 0; d < 3; ++d) {
        int ci = (int)(v[d] * ((float)p.nc[d] / L[d]));
        ci = ci < 0 ? 0 : (ci >= p.nc[d] ? p.nc[d] - 1 : ci);
        c[d] = ci;
    }
}

__global__ void k_bin(const float* __restrict__ pos, const int* __restrict__ cfg,
                      const float* __restrict__ box, const CellPlan* __restrict__ plan, int N,
                      int* cell_of, int* rank, int* cell_cnt, int* status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int b = cfg[i];
    const CellPlan p = plan[b];
    const float L[3] = {box[3 * b], box[3 * b + 1], box[3 * b + 2]};
    const float x = pos[i], y = pos[N + i], z = pos[2 * N + i];
    if (!(x >= 0.0f && x < L[0] && y >= 0.0f && y < L[1] && z >= 0.0f && z < L[2]))
        set_flag(status, 3);
    int c[3];
    cell_coords(p, x, y, z, L, c);
    const int id = p.base + (c[0] * p.nc[1] + c[1]) * p.nc[2] + c[2];
    cell_of[i] = id;
    rank[i] = atomicAdd(cell_cnt + id, 1);
}

// exclusive scan in tiles of 2048 (1024 threads x 2)
constexpr int kScanTile = 2048;

__device__ int block_excl_scan_1024(int v, int* warp_sums, int* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = warp_sums[lane];
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        warp_sums[lane] = s;
    }
    __syncthreads();
    const int incl = x + (w > 0 ? warp_sums[w - 1] : 0);
    *total = warp_sums[31];
    __syncthreads();
    return incl - v;
}

__global__ void __launch_bounds__(1024) k_scan_tiles(const int* __restrict__ in, int n,
                                                     int* __restrict__ out, int* tile_sum) {
    __shared__ int ws[32];
    const int base = blockIdx.x * kScanTile;
    const int i0 = base + 2 * threadIdx.x;
    const int v0 = i0 < n ? in[i0] : 0;
    const int v1 = i0 + 1 < n ? in[i0 + 1] : 0;
    int total;
    const int ex = block_excl_scan_1024(v0 + v1, ws, &total);
    if (i0 < n) out[i0] = ex;
    if (i0 + 1 < n) out[i0 + 1] = ex + v0;
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_scan_sums(int* tile_sum, int ntiles, int* grand) {
    __shared__ int ws[32];
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < ntiles; base += 1024) {
        const int t = base + threadIdx.x;
        const int v = t < ntiles ? tile_sum[t] : 0;
        int total;
        const int ex = block_excl_scan_1024(v, ws, &total);
        if (t < ntiles) tile_sum[t] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *grand = carry;
}

__global__ void k_scan_add(int* out, int n, const int* tile_sum) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += tile_sum[i / kScanTile];
}

__global__ void k_fill(const int* __restrict__ cell_of, const int* __restrict__ rank,
                       const int* __restrict__ cell_start, int N, int* cell_atoms) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    cell_atoms[cell_start[cell_of[i]] + rank[i]] = i;
}

// order each cell's atoms by index so that lists do not depend on the order
// in which atomics handed out ranks, then write the positions in that order
// (x, y, z, atom index as bits): the list build reads a row's candidates as
// one contiguous range, with no dependent index load
__global__ void k_sort_cells(const int* __restrict__ cell_start, int ncell, int* cell_atoms,
                             const float4* __restrict__ pos4, float4* __restrict__ cell_pos) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    const int s0 = cell_start[c], s1 = cell_start[c + 1];
    for (int a = s0 + 1; a < s1; ++a) {
        const int v = cell_atoms[a];
        int b = a - 1;
        while (b >= s0 && cell_atoms[b] > v) {
            cell_atoms[b + 1] = cell_atoms[b];
            --b;
        }
        cell_atoms[b + 1] = v;
    }
    for (int a = s0; a < s1; ++a) {
        const int j = cell_atoms[a];
        const float4 q = pos4[j];
        cell_pos[a] = make_float4(q.x, q.y, q.z, i2f(j));
    }
}

__device__ __forceinline__ int floor_div(int a, int b) {
    int q = a / b;
    if ((a % b != 0) && ((a < 0) != (b < 0))) --q;
    return q;
}

// The whole binning of a small system in one CTA: status cleared, atoms packed
// (as k_pack), the configurations' cell plans and their prefix, atoms counted
// into cells in shared memory, the cells' scan, and the positions in cell
// order, atoms of a cell by index.  One launch in place of twelve of about 2
// us each: at 58 atoms those were half of the list build's time.  The line
// is what 32 KB of shared memory hold; near it the CTA alone is little faster
// on the device (the whole build replayed from a graph, twelve launches / one:
// 7,200 atoms 54.1 / 49.7 us, 7,653 atoms in 48 configurations 58.7 / 56.5), but
// called in sequence the twelve wait for the host: a list and an evaluation of
// 48 configurations with 5,800 atoms 139 / 121 us, ten steps with a rebuild at
// 7,200 atoms 586 / 566.  Bound by the latency of its phases: all atoms are
// loaded before the first is used, and configurations' offsets, boxes and
// plans are read from shared memory (7,200 atoms 19.8 -> 14.4 us).
constexpr int kCellsSmallN = 8192, kCellsSmallB = 256;
constexpr int kCellsSmallStatic = (int)(sizeof(int) * kCellsSmallN + (sizeof(CellPlan) + 3 * sizeof(float)) * kCellsSmallB +
                                        sizeof(int) * (kCellsSmallB + 1 + 32)) + 64;   // and padding
__global__ void __launch_bounds__(1024) k_cells_small(
    const float* pos, const int* type, const int* atom_off,
    const float* box, int N, int B, int T, float rc, int max_images, float4* pos4, int* cfg, int* status,
    CellPlan* plan, int* cell_of, int* cell_start, float4* cell_pos) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ int cnt[];                    // [cells], then the cells' ends
    __shared__ int in_cell[kCellsSmallN];           // atoms in cell order, any order within a cell
    __shared__ CellPlan plan_s[kCellsSmallB];
    __shared__ float box_s[3 * kCellsSmallB];
    __shared__ int off_s[kCellsSmallB + 1], ws[32];
    const int tid = threadIdx.x;
    constexpr int kPer = kCellsSmallN / 1024;
    int id[kPer];
    float4 q[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {                // every load in flight before the first is used
        const int i = tid + u * 1024;
        if (i < N) q[u] = make_float4(pos[i], pos[N + i], pos[2 * N + i], __int_as_float(type[i]));
    }
    if (tid < 4) status[tid] = 0;
    if (tid <= B) off_s[tid] = atom_off[tid];
    if (tid < 3 * B) box_s[tid] = box[tid];
    __syncthreads();
    CellPlan p;
    p.base = 0;
    if (tid < B) p = cell_plan_of(box_s, off_s, tid, rc, max_images, status);
    int ncell;
    const int base = block_excl_scan_1024(p.base, ws, &ncell);
    if (tid < B) {
        p.base = base;
        plan[tid] = plan_s[tid] = p;
    }
    for (int c = tid; c < ncell; c += 1024) cnt[c] = 0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = tid + u * 1024;
        id[u] = -1;
        if (i >= N) continue;
        int t = __float_as_int(q[u].w);
        if (t < 0 || t >= T) {
            set_flag(status, 3);
            q[u].w = __int_as_float(0);
        }
        const int b = find_segment(off_s, B, i);
        const float L[3] = {box_s[3 * b], box_s[3 * b + 1], box_s[3 * b + 2]};
        const float x = q[u].x, y = q[u].y, z = q[u].z;
        if (!(x >= 0.0f && x < L[0] && y >= 0.0f && y < L[1] && z >= 0.0f && z < L[2]))
            set_flag(status, 3);                    // NaN and infinities fail the test too
        pos4[i] = q[u];
        cfg[i] = b;
        const CellPlan& pb = plan_s[b];
        int c[3];
        cell_coords(pb, x, y, z, L, c);
        id[u] = pb.base + (c[0] * pb.nc[1] + c[1]) * pb.nc[2] + c[2];
        cell_of[i] = id[u];
        atomicAdd(cnt + id[u], 1);
    }
    __syncthreads();
    // exclusive scan of the counts, each thread a contiguous run of cells, an
    // odd number so that the runs of a warp's threads start on distinct banks
    const int per = ((ncell + 1023) / 1024) | 1, c0 = min(tid * per, ncell), c1 = min(c0 + per, ncell);
    int sum = 0;
    for (int c = c0; c < c1; ++c) sum += cnt[c];
    int total;
    int run = block_excl_scan_1024(sum, ws, &total);
    for (int c = c0; c < c1; ++c) {
        const int v = cnt[c];
        cnt[c] = run;
        run += v;
    }
    __syncthreads();
    for (int c = tid; c < ncell; c += 1024) cell_start[c] = cnt[c];
    if (tid == 0) cell_start[ncell] = N;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; ++u)
        if (id[u] >= 0) in_cell[atomicAdd(cnt + id[u], 1)] = tid + u * 1024;
    __syncthreads();
    // cnt[c] is now the end of cell c
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        if (id[u] < 0) continue;
        const int i = tid + u * 1024, s0 = id[u] > 0 ? cnt[id[u] - 1] : 0, s1 = cnt[id[u]];
        int rank = 0;
        for (int s = s0; s < s1; ++s) rank += in_cell[s] < i ? 1 : 0;
        cell_pos[s0 + rank] = make_float4(q[u].x, q[u].y, q[u].z, __int_as_float(i));
    }
}

// floor(a / n) and the remainder, 0 <= r < n; near: -n <= a < 2 n
__device__ __forceinline__ int wrap_cell(int a, int n, bool near, int& r) {
    const int q = near ? (a < 0 ? -1 : (a >= n ? 1 : 0)) : floor_div(a, n);
    r = a - q * n;
    return q;
}
// a / n for 0 <= a < 2^21: the quotient's distance from an integer is at least
// 0.5 / n, the rounding error below a / n * 2^-22
__device__ __forceinline__ int small_div(int a, int n) { return (int)(((float)a + 0.5f) * (1.0f / (float)n)); }

// One pass over the stencil.  The list is written in three groups:
// [d < rc_ang + skin] (the angular prefix) | [d < rc_rad] | [rc_rad <= d <
// rc_rad + skin].  Angular candidates fill it from slot 0 up, radial ones
// inside rc_rad from slot cap-1 down, the shell beyond rc_rad goes to a
// scratch buffer; at the end the downward block is reversed and moved behind
// the prefix and the shell appended, all in visit order.  With the pairs
// inside the cutoff first, a warp's late iterations are mostly outside the
// cutoff for all of its lanes and skip the pair work together.
//
// The stencil is visited row by row: for each (ox, oy) the cells oz =
// -half..half are consecutive cell ids (one range of the cell-ordered
// positions, which carry the atom index) except where they wrap around the
// box, which splits the row in two ranges with different z images.  The
// visit order is that of the cell triple loop.  For the reverse-slot search
// the kernel also records, per atom, where each row's angular entries start
// (row_start) and, per angular slot, its row.
//
// Bound by instruction issue with a third of the lanes active (rows of
// different lengths).  Wrapping by compares instead of divisions, row starts
// written 16 at a time, a shell of 4-byte entries where the list has no shifts
// and 8 CTAs per SM (64 registers; 10 spill: 1,174 -> 1,283 us): the list build
// of 900,000 atoms 1,274 -> 1,142 us, k_rev's part without the neighbour's
// count included.
__global__ void __launch_bounds__(128, 8) k_build(const float4* __restrict__ pos4,
                                               const int* __restrict__ cfg,
                                               const float* __restrict__ box,
                                               const CellPlan* __restrict__ plan,
                                               const int* __restrict__ cell_of,
                                               const int* __restrict__ cell_start,
                                               const float4* __restrict__ cell_pos, int N,
                                               float rc2_rad, float rc2_ang, float rc2_phys,
                                               int2* __restrict__ shell, unsigned char* __restrict__ row_start,
                                               unsigned char* __restrict__ slot_row, nep_nlist nl) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int b = cfg[i];
    const CellPlan p = plan[b];
    const float L[3] = {box[3 * b], box[3 * b + 1], box[3 * b + 2]};
    const float4 pi = pos4[i];
    const int c = cell_of[i] - p.base;
    const int cxy = c / p.nc[2], cz = c - cxy * p.nc[2];
    const int cx = cxy / p.nc[1], cy = cxy - cx * p.nc[1];
    const bool nearx = p.half[0] <= p.nc[0], neary = p.half[1] <= p.nc[1], nearz = p.half[2] <= p.nc[2];
    int n_ang = 0, n_in = 0, n_out = 0, w_ang = 0;
    const int cap = nl.cap, cap_ang = nl.cap_ang;
    const int rows = (2 * p.half[0] + 1) * (2 * p.half[1] + 1);
    const bool track = rows <= kMaxRows && cap_ang < 256;
    unsigned char* rs = row_start + (size_t)i * kRowStride;
    // Cells that cannot hold a candidate are skipped: for each stencil row
    // the z range shrinks to the cells that meet the sphere of the list
    // cutoff (plus a margin far above the rounding of the binning) around
    // atom i, given the row's distance from i in x and y.  Skipping only
    // cells whose every point is beyond the cutoff leaves the list, its
    // order and the row starts unchanged.
    const float cs[3] = {L[0] / (float)p.nc[0], L[1] / (float)p.nc[1], L[2] / (float)p.nc[2]};
    const float ics = 1.0f / cs[2];
    const float rl = sqrtf(rc2_rad) + kPruneMargin;
    const float rl2 = rl * rl;
    // the row starts go out 16 at a time: byte stores at a stride of an atom's
    // 64 bytes touch 32 sectors each
    uint4 starts = make_uint4(0u, 0u, 0u, 0u);
    auto row_starts = [&](int row, int n) {
        starts.w |= (unsigned)min(n, 255) << (8 * (row & 3));
        if ((row & 3) != 3) return;
        if ((row & 15) == 15) *reinterpret_cast<uint4*>(rs + row - 15) = starts;
        starts = make_uint4(starts.y, starts.z, starts.w, 0u);
    };
    int row = 0;
    for (int ox = -p.half[0]; ox <= p.half[0]; ++ox) {
        int wx, wy;
        const int ux = cx + ox, sx = wrap_cell(ux, p.nc[0], nearx, wx);
        const float gx = fmaxf(fmaxf((float)ux * cs[0] - pi.x, pi.x - (float)(ux + 1) * cs[0]), 0.0f);
        for (int oy = -p.half[1]; oy <= p.half[1]; ++oy, ++row) {
            const int uy = cy + oy, sy = wrap_cell(uy, p.nc[1], neary, wy);
            if (track) row_starts(row, n_ang);
            const float fx = mul_rn((float)sx, L[0]);
            const float fy = mul_rn((float)sy, L[1]);
            const int rowcell = p.base + (wx * p.nc[1] + wy) * p.nc[2];
            const float gy = fmaxf(fmaxf((float)uy * cs[1] - pi.y, pi.y - (float)(uy + 1) * cs[1]), 0.0f);
            const float rem = rl2 - gx * gx - gy * gy;
            // z range [cz - half, cz + half] cut to the cells that meet the
            // sphere, in pieces of one z image each
            int lo = cz - p.half[2];
            int hi = cz + p.half[2];
            if (rem <= 0.0f) {
                hi = lo - 1;
            } else {
                const float hz = rem * rsqrtf(rem);
                lo = max(lo, (int)floorf((pi.z - hz) * ics));
                hi = min(hi, (int)floorf((pi.z + hz) * ics));
            }
            while (lo <= hi) {
                int wz0;
                const int sz = wrap_cell(lo, p.nc[2], nearz, wz0), wz1 = min(wz0 + hi - lo, p.nc[2] - 1);
                lo += wz1 - wz0 + 1;
                const float fz = mul_rn((float)sz, L[2]);
                const bool zero_img = (sx == 0 && sy == 0 && sz == 0);
                const int sh = pack_shift(sx, sy, sz);
                const int q0 = cell_start[rowcell + wz0], q1 = cell_start[rowcell + wz1 + 1];
                // candidates one ahead
                float4 c_nx = q0 < q1 ? cell_pos[q0] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                for (int q = q0; q < q1; ++q) {
                    const float4 pj = c_nx;
                    if (q + 1 < q1) c_nx = cell_pos[q + 1];
                    const int j = f2i(pj.w);
                    if (j == i && zero_img) continue;
                    const float dx = add_rn(sub_rn(pj.x, pi.x), fx);
                    const float dy = add_rn(sub_rn(pj.y, pi.y), fy);
                    const float dz = add_rn(sub_rn(pj.z, pi.z), fz);
                    const float d2 = dist2(dx, dy, dz);
                    if (!(d2 < rc2_rad)) continue;
                    // the angular and the inside entries share one store
                    // path (slots from the bottom and from the top)
                    const bool ang = d2 < rc2_ang;
                    if (ang || d2 < rc2_phys) {
                        int slot;
                        if (ang) {
                            slot = n_ang < cap_ang && n_ang + n_in < cap ? n_ang : -1;
                            ++n_ang;
                            if (slot >= 0) w_ang = n_ang;
                        } else {
                            slot = n_ang + n_in < cap ? cap - 1 - n_in : -1;
                            ++n_in;
                        }
                        if (slot >= 0) {
                            const size_t at = (size_t)slot * N + i;
                            nl.nbr[at] = j;
                            if (nl.shift) nl.shift[at] = sh;
                            if (ang && track) slot_row[at] = (unsigned char)row;
                        }
                    } else {
                        if (n_out < cap) {
                            const size_t at = (size_t)n_out * N + i;
                            if (nl.shift) shell[at] = make_int2(j, sh);
                            else reinterpret_cast<int*>(shell)[at] = j;
                        }
                        ++n_out;
                    }
                }
            }
        }
    }
    if (track) {
        row_starts(rows, n_ang);
        for (int r = rows + 1; r & 15; ++r) row_starts(r, 0);
    }
    const int n_rest = n_in + n_out;
    const int n_total = n_ang + n_rest;
    const bool over = n_total > cap || n_ang > cap_ang;
    if (over) {
        set_flag(nl.status, 0);
        atomicMax(nl.status + 1, n_total);
        atomicMax(nl.status + 2, n_ang);
        // only the contiguous angular prefix that was written is kept
        nl.cnt[i] = w_ang;
        nl.cnt_ang[i] = w_ang;
        if (track)
            for (int r = 0; r <= rows; ++r) rs[r] = (unsigned char)min((int)rs[r], w_ang);
        return;
    }
    // the inside block sits reversed at [cap - n_in, cap).  Where it does not
    // overlap its target behind the prefix it is copied there in reverse
    // order; otherwise it is reversed in place, then copied down (ascending
    // copy, target never above source).  Then the shell is appended.
    const int base = cap - n_in;
    if (base >= n_ang + n_in) {
        for (int k = 0; k < n_in; ++k) {
            const size_t from = (size_t)(cap - 1 - k) * N + i, to = (size_t)(n_ang + k) * N + i;
            nl.nbr[to] = nl.nbr[from];
            if (nl.shift) nl.shift[to] = nl.shift[from];
        }
    } else {
        for (int k = 0; k < n_in / 2; ++k) {
            const size_t x = (size_t)(base + k) * N + i, y = (size_t)(cap - 1 - k) * N + i;
            const int t = nl.nbr[x];
            nl.nbr[x] = nl.nbr[y];
            nl.nbr[y] = t;
            if (nl.shift) {
                const int u = nl.shift[x];
                nl.shift[x] = nl.shift[y];
                nl.shift[y] = u;
            }
        }
        if (base != n_ang) {
            for (int k = 0; k < n_in; ++k) {
                const size_t from = (size_t)(base + k) * N + i, to = (size_t)(n_ang + k) * N + i;
                nl.nbr[to] = nl.nbr[from];
                if (nl.shift) nl.shift[to] = nl.shift[from];
            }
        }
    }
    for (int k = 0; k < n_out; ++k) {
        const size_t from = (size_t)k * N + i, to = (size_t)(n_ang + n_in + k) * N + i;
        if (nl.shift) {
            const int2 e = shell[from];
            nl.nbr[to] = e.x;
            nl.shift[to] = e.y;
        } else {
            nl.nbr[to] = reinterpret_cast<const int*>(shell)[from];
        }
    }
    nl.cnt[i] = n_total;
    nl.cnt_ang[i] = n_ang;
}

// The same list from a warp per atom, for systems too small to hide one
// thread's serial walk (82 to 124 us up to 10,000 atoms).  The stencil rows'
// candidate ranges go to shared memory in visit order, empty ones dropped;
// lanes then take consecutive candidates, and a bit per range start tells each
// its range (popcount).  The first pass over the candidates counts the three
// groups and keeps the hits in shared memory, the second writes every hit to
// its final slot, so the list is that of k_build entry for entry.  A range
// holds cells of one z image; a row has at most 2 half_z / nc_z + 2.
// Bound by instruction issue from a few thousand atoms on: divisions by the
// cell counts, a bisection for every candidate's range and a second walk over
// the candidates in the writing pass were two thirds of its 2,835 warp
// instructions per atom.  Without them the whole list build takes, before /
// after: 194 atoms 25.1 / 17.4 us, 7,200 49.7 / 39.5, 46,522 220 / 163.
constexpr int kBuildWarps = 4;
constexpr int kBuildSegs = 128;      // candidate ranges held at once
constexpr int kBuildRows = 64;       // stencil rows per round, two per lane
constexpr int kBuildHits = 192;      // hits kept for the second pass; beyond, it walks the candidates again
constexpr int kBuildWarpN = 70000;   // largest system: the whole list build, thread / warp per atom:
                                     // 57,600 atoms 191 / 174 us, 66,679 202 / 184, 76,666 207 / 208,
                                     // 112,500 244 / 288
// With few entries per atom a thread's walk is short and the warp's rows and
// scans are what counts, so the line falls with the mean list length that the
// boxes' volumes give (uniform gases, thread / warp per atom):
//   entries  28: 60,000 atoms 177 / 154 us, 69,000 180 / 169
//            14: 46,000 129 / 119, 60,000 133 / 140
//           9.3: 46,000 119 / 117, 50,000 120 / 121, 69,000 126 / 150
//           4.7: 30,000 95 / 89, 36,000 95 / 97, 69,000 110 / 145
//           2.3: 20,000 79 / 75, 25,000 79 / 81, 60,000 92 / 129
//           0.5: 14,000 68 / 64, 16,000 67 / 68, 30,000 70 / 85
//          0.05: 10,000 62 / 60, 12,000 61 / 62, 30,000 65 / 83
inline int build_warp_most(double entries) {
    return (int)std::min({12000.0 + 5000.0 * entries, 29000.0 + 1650.0 * entries, (double)kBuildWarpN});
}
static_assert(kBuildWarpN < 1 << 30, "a kept hit's kind shares a word with its atom");
constexpr int kBuildImages = 62;     // stencil half-width in boxes, at most, by the plan: 2 * 62 + 2 ranges per row
static_assert(2 * kBuildImages + 2 <= kBuildSegs, "one row's ranges must fit");
constexpr float kBuildMinEdge = 16.0f;   // shortest box edge: the list cutoff over this (17 boxes each way, 35 ranges per row)

__global__ void __launch_bounds__(32 * kBuildWarps, 8) k_build_warp(
    const float4* pos4, const int* cfg, const float* box,
    const CellPlan* plan, const int* cell_of, const int* cell_start,
    const float4* cell_pos, int N, float rc2_rad, float rc2_ang, float rc2_phys,
    unsigned char* __restrict__ row_start, unsigned char* __restrict__ slot_row, nep_nlist nl) {
    pdl_wait();
    pdl_trigger();
    __shared__ int2 s_seg[kBuildWarps][kBuildSegs];   // first atom less the candidates before; image | row << 24
    __shared__ int s_cum[kBuildWarps][kBuildSegs];    // candidates before the range
    __shared__ int2 s_hit[kBuildWarps][kBuildHits];   // atom | kind << 30; image | row << 24
    __shared__ unsigned s_mask[kBuildWarps][32];      // range starts among 1,024 candidates
    __shared__ int s_rowcnt[kBuildWarps][kMaxRows + 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * kBuildWarps + w;
    if (i >= N) return;
    int2 *seg = s_seg[w], *hit = s_hit[w];
    int *cum = s_cum[w], *rowcnt = s_rowcnt[w];
    unsigned* mask = s_mask[w];
    const int b = cfg[i];
    const CellPlan p = plan[b];
    const float L[3] = {box[3 * b], box[3 * b + 1], box[3 * b + 2]};
    const float4 pi = pos4[i];
    const int c = cell_of[i] - p.base;
    const int cxy = small_div(c, p.nc[2]), cz = c - cxy * p.nc[2];
    const int cx = small_div(cxy, p.nc[1]), cy = cxy - cx * p.nc[1];
    const int wy_rows = 2 * p.half[1] + 1, rows = (2 * p.half[0] + 1) * wy_rows;
    const bool nearx = p.half[0] <= p.nc[0], neary = p.half[1] <= p.nc[1], nearz = p.half[2] <= p.nc[2];
    const bool track = rows <= kMaxRows && nl.cap_ang < 256;
    if (track)
        for (int r = lane; r <= rows; r += 32) rowcnt[r] = 0;
    const float cs[3] = {L[0] / (float)p.nc[0], L[1] / (float)p.nc[1], L[2] / (float)p.nc[2]};
    const float rl = sqrtf(rc2_rad) + kPruneMargin;
    const float rl2 = rl * rl;
    const int maxseg = 2 * p.half[2] / p.nc[2] + 2;
    const int per_round = max(1, min(kBuildRows, kBuildSegs / maxseg));
    const unsigned below = (1u << lane) - 1u, upto = below | (1u << lane);
    int nseg = 0, ncand = 0;
    // the ranges of rows row0 .. row0 + per_round - 1
    auto ranges = [&](int row0) {
        // this lane's rows row0 + 2 lane, + 1: z cells lo..hi of each
        int lo[2], hi[2], rc[2], tag[2], mine = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int row = row0 + 2 * lane + u;
            lo[u] = 0;
            hi[u] = -1;
            rc[u] = tag[u] = 0;
            if (2 * lane + u >= per_round || row >= rows) continue;
            const int rx = small_div(row, wy_rows), ox = rx - p.half[0], oy = row - rx * wy_rows - p.half[1];
            int wx, wy;
            const int ux = cx + ox, sx = wrap_cell(ux, p.nc[0], nearx, wx);
            const float gx = fmaxf(fmaxf((float)ux * cs[0] - pi.x, pi.x - (float)(ux + 1) * cs[0]), 0.0f);
            const int uy = cy + oy, sy = wrap_cell(uy, p.nc[1], neary, wy);
            const float gy = fmaxf(fmaxf((float)uy * cs[1] - pi.y, pi.y - (float)(uy + 1) * cs[1]), 0.0f);
            const float rem = rl2 - gx * gx - gy * gy;
            if (rem <= 0.0f) continue;
            const float hz = sqrtf(rem);
            lo[u] = max(cz - p.half[2], (int)floorf((pi.z - hz) / cs[2]));
            hi[u] = min(cz + p.half[2], (int)floorf((pi.z + hz) / cs[2]));
            rc[u] = p.base + (wx * p.nc[1] + wy) * p.nc[2];
            tag[u] = pack_shift(sx, sy, 0) | (int)((unsigned)row << 24);
            int r;
            if (lo[u] <= hi[u])
                mine += wrap_cell(hi[u], p.nc[2], nearz, r) - wrap_cell(lo[u], p.nc[2], nearz, r) + 1;
        }
        int at = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += y;
        }
        const int all = __shfl_sync(0xffffffffu, at, 31);
        at -= mine;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            while (lo[u] <= hi[u]) {
                int z0;
                const int sz = wrap_cell(lo[u], p.nc[2], nearz, z0);
                const int z1 = min(z0 + hi[u] - lo[u], p.nc[2] - 1);
                lo[u] += z1 - z0 + 1;
                const int q0 = cell_start[rc[u] + z0];
                seg[at] = make_int2(q0, tag[u] | (sz & 0xff) << 16);
                cum[at] = cell_start[rc[u] + z1 + 1] - q0;
                ++at;
            }
        }
        __syncwarp();
        // drop the empty ranges; the candidates before each
        nseg = ncand = 0;
        for (int s0 = 0; s0 < all; s0 += 32) {
            const int v = s0 + lane < all ? cum[s0 + lane] : 0;
            const int2 sg = seg[min(s0 + lane, all - 1)];
            int x = v;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            const unsigned some = __ballot_sync(0xffffffffu, v > 0);
            __syncwarp();
            if (v > 0) {
                const int k = nseg + __popc(some & below), before = ncand + x - v;
                cum[k] = before;
                seg[k] = make_int2(sg.x - before, sg.y);
            }
            nseg += __popc(some);
            ncand += __shfl_sync(0xffffffffu, x, 31);
            __syncwarp();
        }
    };
    int n_ang = 0, n_in = 0, n_out = 0, nhit = 0;
    int ra = 0, ri = 0, ro = 0;               // entries of each group written so far
    bool over = false;
    // kind 1 angular, 2 inside, 3 shell, 0 none
    auto write = [&](int kind, int j, int tag) {
        const unsigned ma = __ballot_sync(0xffffffffu, kind == 1);
        const unsigned mi = __ballot_sync(0xffffffffu, kind == 2);
        const unsigned mo = __ballot_sync(0xffffffffu, kind == 3);
        if (kind) {
            const int slot = kind == 1   ? ra + __popc(ma & below)
                             : kind == 2 ? n_ang + ri + __popc(mi & below)
                                         : n_ang + n_in + ro + __popc(mo & below);
            // an overflowing list keeps the part of its angular prefix that fits
            if (!over || (kind == 1 && slot < min(nl.cap, nl.cap_ang))) {
                const size_t to = (size_t)slot * N + i;
                nl.nbr[to] = j;
                if (nl.shift) nl.shift[to] = tag & 0xffffff;
                if (kind == 1 && track) slot_row[to] = (unsigned char)((unsigned)tag >> 24);
            }
        }
        ra += __popc(ma);
        ri += __popc(mi);
        ro += __popc(mo);
    };
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1 && nhit <= kBuildHits) {
            for (int t0 = 0; t0 < nhit; t0 += 32) {
                const int2 h = hit[min(t0 + lane, nhit - 1)];
                write(t0 + lane < nhit ? (int)((unsigned)h.x >> 30) : 0, h.x & 0x3fffffff, h.y);
            }
            break;
        }
        for (int row0 = 0; row0 < rows; row0 += per_round) {
            if (pass == 0 || rows > per_round) ranges(row0);      // one round keeps its ranges
            int started = 0;                  // ranges that start before the chunk
            for (int t0 = 0; t0 < ncand; t0 += 32) {
                if ((t0 & 1023) == 0) {
                    __syncwarp();
                    mask[lane] = 0u;
                    __syncwarp();
                    for (int s = lane; s < nseg; s += 32) {
                        const unsigned d = (unsigned)(cum[s] - t0);
                        if (d < 1024u) atomicOr(mask + (d >> 5), 1u << (d & 31));
                    }
                    __syncwarp();
                }
                const unsigned m = mask[(t0 >> 5) & 31];
                const int t = min(t0 + lane, ncand - 1);
                const int2 sg = seg[started + __popc(m & upto) - 1];
                started += __popc(m);
                const float4 pj = cell_pos[sg.x + t];
                const int j = f2i(pj.w);
                int sx, sy, sz;
                unpack_shift(sg.y, sx, sy, sz);
                const float dx = add_rn(sub_rn(pj.x, pi.x), mul_rn((float)sx, L[0]));
                const float dy = add_rn(sub_rn(pj.y, pi.y), mul_rn((float)sy, L[1]));
                const float dz = add_rn(sub_rn(pj.z, pi.z), mul_rn((float)sz, L[2]));
                const float d2 = dist2(dx, dy, dz);
                int kind = 0;
                if (t0 + lane < ncand && d2 < rc2_rad && !(j == i && (sg.y & 0xffffff) == 0))
                    kind = d2 < rc2_ang ? 1 : (d2 < rc2_phys ? 2 : 3);
                if (pass == 0) {
                    const unsigned any = __ballot_sync(0xffffffffu, kind != 0);
                    if (kind) {
                        const int k = nhit + __popc(any & below);
                        if (k < kBuildHits) hit[k] = make_int2(j | (int)((unsigned)kind << 30), sg.y);
                        if (track && kind == 1) atomicAdd(rowcnt + (int)((unsigned)sg.y >> 24), 1);
                    }
                    nhit += __popc(any);
                    n_ang += kind == 1;
                    n_in += kind == 2;
                } else {
                    write(kind, j, sg.y);
                }
            }
            __syncwarp();
        }
        if (pass == 0) {
            n_ang = __reduce_add_sync(0xffffffffu, n_ang);
            n_in = __reduce_add_sync(0xffffffffu, n_in);
            n_out = nhit - n_ang - n_in;
            over = nhit > nl.cap || n_ang > nl.cap_ang;
        }
    }
    __syncwarp();
    const int kept = over ? min(n_ang, min(nl.cap, nl.cap_ang)) : n_ang;
    if (track) {
        // where each row's angular entries start, within the kept prefix
        unsigned char* rs = row_start + (size_t)i * kRowStride;
        int before = 0;
        for (int r0 = 0; r0 <= rows; r0 += 32) {
            const int r = r0 + lane, v = r < rows ? rowcnt[r] : 0;
            int x = v;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (r <= rows) rs[r] = (unsigned char)min(before + x - v, kept);
            before += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    if (lane == 0) {
        const int total = n_ang + n_in + n_out;
        if (over) {
            set_flag(nl.status, 0);
            atomicMax(nl.status + 1, total);
            atomicMax(nl.status + 2, n_ang);
        }
        nl.cnt[i] = over ? kept : total;
        nl.cnt_ang[i] = kept;
    }
}

// rev[s][i] = slot of i (with the opposite image) in the angular prefix of
// j = nbr[s][i].  j visits i in the mirrored stencil row, rows - 1 - row,
// so only that row's stretch of j's prefix is searched; stencils too large
// for the row table fall back to scanning j's whole prefix.
__device__ __forceinline__ void rev_slot(int N, int i, int s, int rows, bool track,
                                         const unsigned char* row_start, const unsigned char* slot_row,
                                         const nep_nlist& nl) {
    const int j = nl.nbr[(size_t)s * N + i];
    int want = 0;
    if (nl.shift) {
        int a, b, c;
        unpack_shift(nl.shift[(size_t)s * N + i], a, b, c);
        want = pack_shift(-a, -b, -c);
    }
    int t0 = 0, t1;
    if (track) {
        const int mr = rows - 1 - (int)slot_row[(size_t)s * N + i];
        const unsigned char* rj = row_start + (size_t)j * kRowStride;
        t0 = rj[mr];
        t1 = rj[mr + 1];
    } else {
        t1 = nl.cnt_ang[j];
    }
    int found = -1;
    for (int t = t0; t < t1; ++t) {
        if (nl.nbr[(size_t)t * N + j] == i && (!nl.shift || nl.shift[(size_t)t * N + j] == want)) {
            found = t;
            break;
        }
    }
    if (found < 0) {
        set_flag(nl.status, 0);
        found = 0;
    }
    nl.rev[(size_t)s * N + i] = found;
}

// G = 1: one thread per atom; G = 32: a warp per atom, a lane per slot.  The
// warps lose the coalescing of the slot-major list, but up to kRevWarpN atoms
// the shorter walk is worth more (the list build of 57,600 atoms 214 -> 203
// us, of 112,500 atoms 259 -> 262).  With few entries per atom most lanes have
// none (gases, thread / warp per atom: 4.7 entries, 50,000 atoms 106 / 104 us,
// 69,000 107 / 110; 2.3, 40,000 88 / 87, 46,000 89 / 90, 69,000 91 / 95; 0.5,
// 36,000 75 / 74, 40,000 71 / 75, 69,000 74 / 83).
constexpr int kRevWarpN = 80000, kRevWarpSparseN = 42000;
constexpr double kRevSparse = 4.0;
template <int G>
__global__ void __launch_bounds__(128) k_rev(int N, const int* cfg, const CellPlan* plan,
                                             const unsigned char* row_start,
                                             const unsigned char* slot_row, nep_nlist nl) {
    pdl_wait();
    pdl_trigger();
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) / G;
    if (i >= N) return;
    const int na = nl.cnt_ang[i];
    const CellPlan p = plan[cfg[i]];
    const int rows = (2 * p.half[0] + 1) * (2 * p.half[1] + 1);
    const bool track = rows <= kMaxRows && nl.cap_ang < 256;
    for (int s = threadIdx.x % G; s < na; s += G) rev_slot(N, i, s, rows, track, row_start, slot_row, nl);
}

// ------------------------------------------------------------ optimiser
// one Adam step per parameter; c1 = lr / (1 - beta1^t), c2 = 1 / sqrt(1 - beta2^t)
__global__ void k_adam(float* __restrict__ p, const float* g, float* __restrict__ m,
                       float* __restrict__ v, int n, float beta1, float beta2, float eps, float c1, float c2) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float gk = g[k];
    const float mk = beta1 * m[k] + (1.0f - beta1) * gk;
    const float vk = beta2 * v[k] + (1.0f - beta2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    p[k] -= c1 * mk / (sqrtf(vk) * c2 + eps);
}

// ------------------------------------------------------------ FP32 peak
// eight independent FMA chains per thread; a and b come from memory so that
// nothing folds, the sums are stored so that nothing is dropped
constexpr int kFmaIters = 4096;
__global__ void __launch_bounds__(256) k_fma_peak(const float* __restrict__ ab, float* __restrict__ out) {
    const float a = ab[0], b = ab[1];
    float x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = (float)(threadIdx.x + k) * 1e-3f;
    for (int it = 0; it < kFmaIters; ++it) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = fmaf(x[k], a, b);
    }
    float sum = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += x[k];
    out[blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

// ------------------------------------------------------------ integrator
struct InvMass {
    float v[kMaxTypes];
};

// every load before the first store; x: the new position (if pos is given)
__device__ __forceinline__ void kick_atom(float* vel, const float* force, int type, const InvMass& im, int N, int i,
                                          float half_dt, float* pos, float dt, float (&x)[3]) {
    const float s = half_dt * im.v[type & (kMaxTypes - 1)];
    float v[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const size_t at = (size_t)d * N + i;
        v[d] = vel[at] + s * force[at];
        x[d] = pos ? pos[at] : 0.0f;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const size_t at = (size_t)d * N + i;
        vel[at] = v[d];
        x[d] += dt * v[d];
        if (pos) pos[at] = x[d];
    }
}
__global__ void k_kick(float* __restrict__ vel, const float* force,
                       const int* type, InvMass im, int N, float half_dt,
                       float* __restrict__ pos, float dt) {
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float x[3];
    if (i < N) kick_atom(vel, force, type[i], im, N, i, half_dt, pos, dt, x);
}
// the opening half kick and the drift, then the atom packed at its new
// position (as k_pack, whose launch and pass over the positions this saves)
__global__ void __launch_bounds__(256) k_kick_pack(float* __restrict__ vel, const float* force,
                                                   const int* type, InvMass im, int N, float half_dt,
                                                   float* __restrict__ pos, float dt,
                                                   const int* atom_off, int B, int T, float4* pos4,
                                                   int* cfg, int* status, int* chunk_start, int* ticket) {
    pdl_wait();
    pdl_trigger();
    if (chunk_start && blockIdx.x == gridDim.x - 1) {
        chunk_plan_block(atom_off, B, chunk_start, ticket);
        return;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int t = type[i];
    float x[3];
    kick_atom(vel, force, t, im, N, i, half_dt, pos, dt, x);
    pack_atom(x[0], x[1], x[2], t, atom_off, B, T, i, pos4, cfg, status);
}

// x wrapped into [0, L)
__device__ __forceinline__ float wrap_coord(float x, float L) {
    x = x - L * floorf(x / L);
    if (x >= L) x -= L;
    if (x < 0.0f) x += L;
    if (!(x < L)) x = 0.0f;
    return x;
}
// each atom's configuration is found from the CSR offsets
__global__ void k_wrap_seg(float* pos, const int* atom_off, int B, const float* box,
                           int N) {
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int b = find_segment(atom_off, B, i);
    for (int d = 0; d < 3; ++d) pos[(size_t)d * N + i] = wrap_coord(pos[(size_t)d * N + i], box[3 * b + d]);
}

// ------------------------------------------------------------- loss adjoints
// sum over the block in a fixed order (thread 0): warp shuffles, then the
// warp sums in order, with one block-wide wait
__device__ __forceinline__ double block_sum_fixed(double v) {
    __shared__ double red[kRedThreads / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kRedThreads / 32; ++w) s += red[w];
    return s;
}

// Force residuals per chunk: lam_i = 2 wF (F_i - F_lbl,i) / (3 N_b B) and the
// FP64 partial sum of |dF|^2 (Eq. 20).
__global__ void __launch_bounds__(kRedThreads) k_loss_atoms(
    int N, int B, const int* atom_off, const int* chunk_start,
    const float* force, const float* f_lbl, float wF, float4* __restrict__ lam4,
    double* partial) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x;
    const int total = chunk_start[B];
    if (k >= total) return;
    const int b = find_segment(chunk_start, B, k);
    const int a0 = atom_off[b] + (k - chunk_start[b]) * kChunk;
    const int a1 = min(atom_off[b + 1], a0 + kChunk);
    const int nb = atom_off[b + 1] - atom_off[b];
    const float cf = 2.0f * wF / (3.0f * (float)nb * (float)B);
    double acc = 0.0;
    for (int i = a0 + threadIdx.x; i < a1; i += kRedThreads) {
        const float dx = force[i] - f_lbl[i];
        const float dy = force[N + i] - f_lbl[N + i];
        const float dz = force[2 * N + i] - f_lbl[2 * N + i];
        lam4[i] = make_float4(cf * dx, cf * dy, cf * dz, 0.0f);
        acc += (double)dx * dx + (double)dy * dy + (double)dz * dz;
    }
    acc = block_sum_fixed(acc);
    if (threadIdx.x == 0) partial[k] = acc;
}

// Per-configuration loss terms and energy/virial adjoints (Eqs. 18-21), and
// the batch loss summed in a fixed tree (one CTA).
__global__ void __launch_bounds__(kRedThreads) k_loss_cfg(
    int B, const int* atom_off, const int* chunk_start,
    const double* partial, const double* e_tot,
    const double* vir, const double* e_lbl,
    const double* v_lbl, float wE, float wF, float wV, int mode, float* aE, float* mu,
    double* loss) {
    pdl_wait();
    pdl_trigger();
    // FP64 division is slow on this GPU: each configuration divides once,
    // by its atom count, and the rest are products
    const double iB = 1.0 / (double)B;
    double acc = 0.0;
    for (int b = threadIdx.x; b < B; b += kRedThreads) {
        const double nb = (double)(atom_off[b + 1] - atom_off[b]);
        const double n = nb > 0.0 ? nb : 1.0;
        const double in = 1.0 / n;
        double sF = 0.0;
        for (int k = chunk_start[b]; k < chunk_start[b + 1]; ++k) sF += partial[k];
        const double dE = e_tot[b] - e_lbl[b];
        double sV = 0.0;
        for (int c = 0; c < 9; ++c) {
            const double dv = vir[9 * b + c] - v_lbl[9 * b + c];
            sV += dv * dv;
        }
        constexpr double third = 1.0 / 3.0, ninth = 1.0 / 9.0;
        double Lb;
        if (mode == 0) {
            const double e = dE * in;
            Lb = wE * e * e + wF * sF * (third * in) + wV * sV * (ninth * in * in);
            aE[b] = (float)(2.0 * wE * dE * (in * in) * iB);
            const double fv = 2.0 * wV * (ninth * in * in) * iB;
            for (int c = 0; c < 9; ++c) mu[9 * b + c] = (float)(fv * (vir[9 * b + c] - v_lbl[9 * b + c]));
        } else {
            Lb = wE * dE * dE * in + wF * sF * (third * in) + wV * sV * (ninth * in);
            aE[b] = (float)(2.0 * wE * dE * in * iB);
            const double fv = 2.0 * wV * (ninth * in) * iB;
            for (int c = 0; c < 9; ++c) mu[9 * b + c] = (float)(fv * (vir[9 * b + c] - v_lbl[9 * b + c]));
        }
        if (nb > 0.0) acc += Lb;
    }
    acc = block_sum_fixed(acc);
    if (threadIdx.x == 0 && loss) *loss = acc * iB;
}

// External adjoints (vector-Jacobian product) into the kernels' layout.
__global__ void k_pack_adjoint(int N, int B, const float* lam,
                               const double* a_e, const double* mu_in,
                               float4* lam4, float* aE, float* mu) {
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) lam4[i] = make_float4(lam[i], lam[N + i], lam[2 * N + i], 0.0f);
    if (i < B) {
        aE[i] = (float)a_e[i];
        for (int c = 0; c < 9; ++c) mu[9 * i + c] = (float)mu_in[9 * i + c];
    }
}

inline int blocks(int n, int t) { return (n + t - 1) / t; }

}  // namespace

// ------------------------------------------------------------ launchers
cudaError_t launch_pack(const float* pos, const int* type, const int* atom_off, int N, int B,
                        int T, float4* pos4, int* cfg, int* status, cudaStream_t st) {
    if (N > 0)
        launch_pdl(k_pack, blocks(N, 256), 256, 0, st, pos, type, atom_off, N, B, T, pos4, cfg, status, nullptr, nullptr);
    return cudaGetLastError();
}

// The plan rides in the packing launch, which saves one, unless its scan by one
// block of 256 threads outlasts the packing.  Evaluation of configurations of
// three atoms in a graph, fused / apart: 512 44.8 / 48.2 us, 2,040 93.9 / 97.0,
// 3,000 113.3 / 116.4, 4,000 129.8 / 128.7, 8,000 179.8 / 172.9; the line keeps
// some distance from where the forms are equal, since single atoms or none
// leave less packing beside the same scan.
constexpr int kPlanFusedB = 2048;
cudaError_t launch_pack_plan(const float* pos, const int* type, const int* atom_off, int N, int B, int T,
                             float4* pos4, int* cfg, int* status, int* chunk_start, int* ticket, cudaStream_t st) {
    const bool fused = B <= kPlanFusedB;
    if (fused) {
        launch_pdl(k_pack, blocks(N, 256) + 1, 256, 0, st, pos, type, atom_off, N, B, T, pos4, cfg, status, chunk_start,
                                                   ticket);
    } else {
        if (N > 0)
            launch_pdl(k_pack, blocks(N, 256), 256, 0, st, pos, type, atom_off, N, B, T, pos4, cfg, status, nullptr,
                                                   nullptr);
        k_chunk_plan<<<1, 1024, 0, st>>>(atom_off, B, chunk_start, ticket);
    }
    return cudaGetLastError();
}

// k_totals reads the chunk plan ahead of its wait, which needs a kernel between
// the plan's writer and itself.  Without atoms there is none: it follows the
// packing launch, which lets its successor start before the plan is written, so
// there it is an ordinary launch.
cudaError_t launch_totals(const EvalArgs& a, const FinishArgs& f, int max_chunks, cudaStream_t st) {
    if (max_chunks <= 0) return cudaGetLastError();
    if (a.N > 0)
        launch_pdl(k_totals, max_chunks, kTotalsThreads, 0, st, a, f);
    else
        k_totals<<<max_chunks, kTotalsThreads, 0, st>>>(a, f);
    return cudaGetLastError();
}

size_t nbr_cell_capacity(int N, int B) { return 2 * (size_t)N + 27 * (size_t)B; }

cudaError_t launch_neighbors(const float* pos, const int* type, int T, float4* pos4, const int* atom_off,
                             const float* box, int* cfg, int N, int B, float rc_list, float rc_list_ang,
                             float rc_phys, float min_edge, double density, nep_nlist* nl, const NbrWork& w,
                             cudaStream_t st) {
    cudaError_t e;
    const int cmax = w.cmax;
    const double entries = density * 4.18879 * rc_list * rc_list * rc_list;   // 4 pi / 3
    const bool warp_build = N <= build_warp_most(entries) && min_edge * kBuildMinEdge >= rc_list;
    const int max_images = warp_build ? kBuildImages : 0;
    if (N > 0 && N <= kCellsSmallN && B <= kCellsSmallB) {
        const int smem = (int)sizeof(int) * (cmax + 1);
        // with the static arrays past 48 KB (138 KB at most), which needs the attribute
        if (smem + kCellsSmallStatic > 48 * 1024 &&
            (e = cudaFuncSetAttribute(k_cells_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(int) * (2 * kCellsSmallN + 27 * kCellsSmallB + 1))))
            return e;
        launch_pdl(k_cells_small, 1, 1024, smem, st, pos, type, atom_off, box, N, B, T, rc_list, max_images,
                                             pos4, cfg, nl->status, w.plan, w.cell_of, w.cell_start, w.cell_pos);
    } else {
        if ((e = cudaMemsetAsync(nl->status, 0, 4 * sizeof(int), st))) return e;
        if (N == 0) return cudaSuccess;
        if ((e = launch_pack(pos, type, atom_off, N, B, T, pos4, cfg, nl->status, st))) return e;
        k_cell_plan<<<blocks(B, 128), 128, 0, st>>>(box, atom_off, B, rc_list, max_images, w.plan, nl->status);
        k_plan_scan<<<1, 32, 0, st>>>(w.plan, B);
        if ((e = cudaMemsetAsync(w.cell_cnt, 0, sizeof(int) * (size_t)(cmax + 1), st)) != cudaSuccess) return e;
        k_bin<<<blocks(N, 256), 256, 0, st>>>(pos, cfg, box, w.plan, N, w.cell_of, w.rank, w.cell_cnt, nl->status);
        const int n = cmax + 1;
        const int ntiles = blocks(n, kScanTile);
        k_scan_tiles<<<ntiles, 1024, 0, st>>>(w.cell_cnt, n, w.cell_start, w.scan_tmp);
        k_scan_sums<<<1, 1024, 0, st>>>(w.scan_tmp, ntiles, w.scan_tmp + ntiles);
        k_scan_add<<<blocks(n, 256), 256, 0, st>>>(w.cell_start, n, w.scan_tmp);
        k_fill<<<blocks(N, 256), 256, 0, st>>>(w.cell_of, w.rank, w.cell_start, N, w.cell_atoms);
        k_sort_cells<<<blocks(cmax, 128), 128, 0, st>>>(w.cell_start, cmax, w.cell_atoms, pos4, w.cell_pos);
    }
    const float rr = rc_list * rc_list, ra = rc_list_ang * rc_list_ang, rp = rc_phys * rc_phys;
    if (warp_build)
        launch_pdl(k_build_warp, blocks(N, kBuildWarps), 32 * kBuildWarps, 0, st, pos4, cfg, box, w.plan, w.cell_of,
                                                                          w.cell_start, w.cell_pos, N, rr, ra, rp,
                                                                          w.row_start, w.slot_row, *nl);
    else
        k_build<<<blocks(N, 128), 128, 0, st>>>(pos4, cfg, box, w.plan, w.cell_of, w.cell_start,
                                                w.cell_pos, N, rr, ra, rp, w.shell, w.row_start, w.slot_row, *nl);
    if (N <= (entries < kRevSparse ? kRevWarpSparseN : kRevWarpN))
        launch_pdl(k_rev<32>, blocks(N, 4), 128, 0, st, N, cfg, w.plan, w.row_start, w.slot_row, *nl);
    else
        k_rev<1><<<blocks(N, 128), 128, 0, st>>>(N, cfg, w.plan, w.row_start, w.slot_row, *nl);
    return cudaGetLastError();
}

cudaError_t launch_adam(float* p, const float* g, float* m, float* v, int n, float beta1, float beta2,
                        float eps, float c1, float c2, cudaStream_t st) {
    if (n > 0) launch_pdl(k_adam, blocks(n, 256), 256, 0, st, p, g, m, v, n, beta1, beta2, eps, c1, c2);
    return cudaGetLastError();
}

cudaError_t fp32_peak(cudaStream_t st, double* tflops) {
    int dev = 0, nsm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev))) return e;
    const int blocks_n = nsm * 8, threads = 256;
    float* buf = nullptr;
    if ((e = cudaMalloc(&buf, sizeof(float) * ((size_t)blocks_n * threads + 2)))) return e;
    const float ab[2] = {0.999f, 1e-3f};
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    float ms = 0.0f, best = 1e30f;
    if (!(e = cudaMemcpyAsync(buf, ab, sizeof ab, cudaMemcpyHostToDevice, st)) && !(e = cudaEventCreate(&e0)) &&
        !(e = cudaEventCreate(&e1))) {
        for (int r = 0; r < 4 && !e; ++r) {
            cudaEventRecord(e0, st);
            k_fma_peak<<<blocks_n, threads, 0, st>>>(buf, buf + 2);
            cudaEventRecord(e1, st);
            if (!(e = cudaEventSynchronize(e1)) && !(e = cudaEventElapsedTime(&ms, e0, e1)) && r > 0 && ms < best)
                best = ms;
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(buf);
    if (e) return e;
    *tflops = 2.0 * 8.0 * kFmaIters * (double)blocks_n * threads / (best * 1e-3) / 1e12;
    return cudaGetLastError();
}

cudaError_t launch_kick(float* vel, const float* force, const int* type, const float* inv_mass,
                        int N, float half_dt, float* pos, float dt, cudaStream_t st) {
    InvMass im;
    for (int t = 0; t < kMaxTypes; ++t) im.v[t] = inv_mass[t];
    if (N > 0) launch_pdl(k_kick, blocks(N, 256), 256, 0, st, vel, force, type, im, N, half_dt, pos, dt);
    return cudaGetLastError();
}

cudaError_t launch_kick_pack(float* vel, const float* force, const int* type, const float* inv_mass, int N, int B,
                             int T, float half_dt, float* pos, float dt, const int* atom_off, float4* pos4, int* cfg,
                             int* status, int* chunk_start, int* ticket, cudaStream_t st) {
    InvMass im;
    for (int t = 0; t < kMaxTypes; ++t) im.v[t] = inv_mass[t];
    const bool fused = B <= kPlanFusedB;
    if (N > 0 || fused)
        launch_pdl(k_kick_pack, blocks(N, 256) + (fused ? 1 : 0), 256, 0, st, vel, force, type, im, N, half_dt, pos, dt,
                                                                      atom_off, B, T, pos4, cfg, status,
                                                                      fused ? chunk_start : nullptr, ticket);
    if (!fused) k_chunk_plan<<<1, 1024, 0, st>>>(atom_off, B, chunk_start, ticket);
    return cudaGetLastError();
}

cudaError_t launch_loss(int N, int B, const int* atom_off, const int* chunk_start, int max_chunks,
                        const float* force, const float* f_lbl, const double* e_tot,
                        const double* vir, const double* e_lbl, const double* v_lbl,
                        const float* w, int mode, float4* lam4, float* aE, float* mu,
                        double* partial, double* loss, cudaStream_t st) {
    if (max_chunks > 0)
        launch_pdl(k_loss_atoms, max_chunks, kRedThreads, 0, st, N, B, atom_off, chunk_start, force, f_lbl, w[1],
                                                         lam4, partial);
    launch_pdl(k_loss_cfg, 1, kRedThreads, 0, st, B, atom_off, chunk_start, partial, e_tot, vir, e_lbl, v_lbl,
                                          w[0], w[1], w[2], mode, aE, mu, loss);
    return cudaGetLastError();
}

cudaError_t launch_pack_adjoint(int N, int B, const float* lam, const double* a_e, const double* mu_in,
                                float4* lam4, float* aE, float* mu, cudaStream_t st) {
    const int n = N > B ? N : B;
    if (n > 0) launch_pdl(k_pack_adjoint, blocks(n, 256), 256, 0, st, N, B, lam, a_e, mu_in, lam4, aE, mu);
    return cudaGetLastError();
}

cudaError_t launch_wrap_segments(float* pos, const int* atom_off, int B, const float* box, int N, cudaStream_t st) {
    if (N > 0) launch_pdl(k_wrap_seg, blocks(N, 256), 256, 0, st, pos, atom_off, B, box, N);
    return cudaGetLastError();
}

}  // namespace nep
