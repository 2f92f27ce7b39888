// All-pairs Cauchy sums z_i = sum_{j != i} w_j / (eta_i - eta_j)  (Sec. 2.5,
// Eqs. fmm-1, fmm-E) and the pointwise operators built on them (Secs. 3.3,
// 3.4, 4.3, 4.4).
//
// In every precision one kernel takes each unordered pair once (`_sym`): a block
// has a pair of node blocks, rows in registers, the columns' sums passed round the
// lanes, and 1/d serves both directions.  It writes partial sums to a
// [node block][rhs][N] buffer; a second kernel adds them in a fixed order
// (deterministic) in FP64 and applies the operator's epilogue (small FP64 sums do
// this themselves).
//
// The ordered kernels serve a source-chunk override and the calls for which the
// others' partial sums have no room: blocks along x own a tile of targets held in
// registers (T per thread); blocks along y a contiguous chunk of source tiles, which
// they stream through shared memory, with a [chunk][rhs][N] buffer.
//
// Per ordered pair: FP64 9 FP64-pipe instructions on 1/d
//   2 DADD (d = eta_i - eta_j), DMUL + DFMA (|d|^2), 3 DFMA to refine the
//   hardware reciprocal seed, 2 DMUL (Re, Im of 1/d)
// (two when it is formed on the FP32 pipe) and 4 DFMA on w / d; FP32 10 FP32-pipe
// instructions and one MUFU reciprocal; double-float about 97 and one MUFU.
#include <algorithm>
#include <cmath>

#include "gnk_internal.h"
#include "epilogue.cuh"
#include "pairmath.cuh"

namespace gnk {
namespace {

// Far-away position for padded sources of a ragged last tile: |d|^2 stays
// finite and the zero weight contributes exactly 0.
constexpr double kFar64 = 1e150;
constexpr float kFar32 = 1e18f;

// ------------------------------------------------------------------ FP64
struct Pair64Args {
    const double2* et;
    int N;
    const double2* w0;
    const double2* w1;
    const double* x0;
    const double* x1;
    const double2* s;
    double2* partial;
    int tiles_src;
    int tiles_per_chunk;
    const int* done;
};

template <int R, int MODE>
__global__ void __launch_bounds__(kThreads64) pairsum64_kernel(Pair64Args a) {
    constexpr int S = kSrcTile64, T = kTargets64, NT = kThreads64;
    __shared__ double2 s_pos[S];
    __shared__ double2 s_w[R][S];
    if (a.done != nullptr && *a.done) return;
    const int N = a.N;
    const int tgt0 = blockIdx.x * (NT * T);

    double px[T], py[T], ax[T][R], ay[T][R];
    int idx[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        idx[t] = tgt0 + t * NT + threadIdx.x;
        const double2 p = a.et[min(idx[t], N - 1)];
        px[t] = p.x;
        py[t] = p.y;
#pragma unroll
        for (int r = 0; r < R; ++r) ax[t][r] = ay[t][r] = 0.0;
    }

    const int tb = blockIdx.y * a.tiles_per_chunk;
    const int te = min(tb + a.tiles_per_chunk, a.tiles_src);
    for (int tile = tb; tile < te; ++tile) {
        const int j0 = tile * S;
        __syncthreads();
        for (int k = threadIdx.x; k < S; k += NT) {
            const int j = j0 + k;
            if (j < N) {
                s_pos[k] = a.et[j];
                if (MODE == W_COMPLEX) {
                    s_w[0][k] = a.w0[j];
                    if (R > 1) s_w[R - 1][k] = a.w1[j];
                } else {
                    const double2 sc = a.s[j];
                    const double x0 = a.x0[j];
                    s_w[0][k] = make_double2(sc.x * x0, sc.y * x0);
                    if (R > 1) {
                        const double x1 = a.x1[j];
                        s_w[R - 1][k] = make_double2(sc.x * x1, sc.y * x1);
                    }
                }
            } else {
                s_pos[k] = make_double2(kFar64, kFar64);
#pragma unroll
                for (int r = 0; r < R; ++r) s_w[r][k] = make_double2(0.0, 0.0);
            }
        }
        __syncthreads();
        const bool diag = (j0 < tgt0 + NT * T) && (tgt0 < j0 + S);
        if (!diag) {
#pragma unroll 2
            for (int k = 0; k < S; ++k) {
                const double2 sp = s_pos[k];
#pragma unroll
                for (int t = 0; t < T; ++t) {
                    const double dx = px[t] - sp.x, dy = py[t] - sp.y;
                    const double inv = recip_f64(fma(dx, dx, dy * dy));
                    const double ar = dx * inv, ai = dy * inv;  // 1/d = ar - i ai
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const double2 w = s_w[r][k];
                        ax[t][r] = fma(w.x, ar, ax[t][r]);
                        ax[t][r] = fma(w.y, ai, ax[t][r]);
                        ay[t][r] = fma(w.y, ar, ay[t][r]);
                        ay[t][r] = fma(-w.x, ai, ay[t][r]);
                    }
                }
            }
        } else {
            for (int k = 0; k < S; ++k) {
                const double2 sp = s_pos[k];
                const int j = j0 + k;
#pragma unroll
                for (int t = 0; t < T; ++t) {
                    const double dx = px[t] - sp.x, dy = py[t] - sp.y;
                    double inv = recip_f64(fma(dx, dx, dy * dy));
                    inv = (j == idx[t]) ? 0.0 : inv;  // the i = j term is excluded (Eq. fmm-E)
                    const double ar = dx * inv, ai = dy * inv;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const double2 w = s_w[r][k];
                        ax[t][r] = fma(w.x, ar, ax[t][r]);
                        ax[t][r] = fma(w.y, ai, ax[t][r]);
                        ay[t][r] = fma(w.y, ar, ay[t][r]);
                        ay[t][r] = fma(-w.x, ai, ay[t][r]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {
        if (idx[t] < N) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                a.partial[((size_t)blockIdx.y * R + r) * N + idx[t]] = make_double2(ax[t][r], ay[t][r]);
        }
    }
}

// ------------------------------------------------------------------ FP64, pairs taken once
// 1/(eta_j - eta_i) = -1/(eta_i - eta_j): a pair's difference and 1/d serve both
// directions.  The FP64 pipe (2 lanes per SM) bounds the sum; 1/d is formed on the
// FP32 pipe beside it (inv_conj_f64), so per unordered pair the kernel spends
//   2 + 8 R (both parts of z) or 2 + 4 (one part, R = 1)
// FP64 instructions instead of 2 (9 + 4 R).  A block takes one pair (I, J) of node blocks of SB =
// 32 W G nodes (W >= 2).  A warp holds 32 targets (one per lane) and meets 32 sources in
// 32 steps: in step k lane l takes source (l + k) mod 32, whose sum travels
// with it, handed to the next lane by a shuffle (issue slots are free: an
// FP64 instruction holds the pipe for 16 cycles).  Row sums stay in registers,
// column sums in shared memory between the warps' turns (warp w takes the
// 32 sources of slice (w + s) mod W in turn s: no two warps share a slice, and
// the order is fixed).  Block (I, J) writes I's sums to slot J and J's to slot
// I, so every node gets nt partial sums, added by the reduction in slot order.
// Measured: (D - diag(D1) + Lhat) x at N = 16,000, real A: 6.15 ms by ordered
// pairs, 3.00 with 9 + 4 FP64 instructions per unordered pair, 1.46 now.
struct Pair64SymArgs {
    const double2* et;
    int N;
    const double2* w0;
    const double2* w1;
    const double* x0;
    const double* x1;
    const double2* s;
    double2* partial;  // [slot][rhs][N]
    int nt;            // node blocks
    int G;             // sub-tiles of 32 W nodes per node block
    int* count;        // [nt] contributions per node block (32-node blocks; zero between products)
    const int* done;
};

template <int R, int MODE>
__device__ __forceinline__ void load_node64(const Pair64SymArgs& a, int j, double2& pos, double2 (&w)[R]) {
    if (j < a.N) {
        pos = a.et[j];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (MODE == W_COMPLEX) {
                w[r] = (r == 0) ? a.w0[j] : a.w1[j];
            } else {
                const double2 sc = a.s[j];
                const double x = (r == 0) ? a.x0[j] : a.x1[j];
                w[r] = make_double2(sc.x * x, sc.y * x);
            }
        }
    } else {
        pos = make_double2(kFar64, kFar64);
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = make_double2(0.0, 0.0);
    }
}

// acc += sign * (the wanted parts of w (ar - i ai)); COMP 0: both, 1: Im, 2: Re
template <int COMP, bool NEG>
__device__ __forceinline__ void add_term64(double* acc, double2 w, double ar, double ai) {
    const double wx = NEG ? -w.x : w.x, wy = NEG ? -w.y : w.y;
    if (COMP != 1) {
        acc[0] = fma(wx, ar, acc[0]);
        acc[0] = fma(wy, ai, acc[0]);
    }
    if (COMP != 2) {
        double& im = acc[COMP == 0 ? 1 : 0];
        im = fma(wy, ar, im);
        im = fma(-wx, ai, im);
    }
}

// Pair t of node blocks: (I, I + o mod nt) for the full offsets o, the half
// offset of an even nt, then the diagonal (half the work: last).
__device__ __forceinline__ void sym_blocks(int nt, int t, int& I, int& J) {
    const int off = nt * (nt - 1) / 2;
    if (t < off) {
        const int o = t / nt + 1;
        I = t - (o - 1) * nt;
        J = I + o;
        if (J >= nt) J -= nt;
    } else {
        I = J = t - off;
    }
}

template <int R, int MODE, int COMP, int W>
__global__ void __launch_bounds__(32 * W) pairsum64_sym_kernel(Pair64SymArgs a) {
    constexpr int NC = COMP == 0 ? 2 : 1;  // parts of z kept
    constexpr int NT = 32 * W;
    extern __shared__ __align__(16) double s_dyn64[];
    double2* s_pos = reinterpret_cast<double2*>(s_dyn64);  // [NT]
    double2* s_w = s_pos + NT;                             // [R][NT]
    double* s_col = reinterpret_cast<double*>(s_w + R * NT);  // [R][NC][SB]
    if (a.done != nullptr && *a.done) return;
    const int SB = NT * a.G;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int I, J;
    sym_blocks(a.nt, blockIdx.x, I, J);
    const bool diag = I == J;
    for (int e = threadIdx.x; e < R * NC * SB; e += NT) s_col[e] = 0.0;
    for (int gi = 0; gi < a.G; ++gi) {
        const int i = I * SB + gi * NT + threadIdx.x;
        if (I * SB + gi * NT >= a.N) break;
        double2 p, w[R];
        load_node64<R, MODE>(a, i, p, w);
        double acc[R][NC];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[r][c] = 0.0;
        for (int gj = diag ? gi : 0; gj < a.G; ++gj) {
            const int j0 = J * SB + gj * NT;
            if (j0 >= a.N) break;
            __syncthreads();  // the previous sub-tile is done with s_pos, s_w
            {
                double2 pj, wj[R];
                load_node64<R, MODE>(a, j0 + threadIdx.x, pj, wj);
                s_pos[threadIdx.x] = pj;
#pragma unroll
                for (int r = 0; r < R; ++r) s_w[r * NT + threadIdx.x] = wj[r];
            }
            const bool self = diag && gj == gi;
            const int turns = self ? W / 2 + 1 : W;  // a sub-tile with itself: each slice pair once
            for (int s = 0; s < turns; ++s) {
                __syncthreads();
                const int c = (wid + s) & (W - 1);  // W is a power of two
                if (self && s == 0) {  // the slice with itself: every ordered pair by its own row
#pragma unroll 4
                    for (int k = 0; k < 32; ++k) {
                        const int q = c * 32 + k;
                        const double2 sp = s_pos[q];
                        const double dx = p.x - sp.x, dy = p.y - sp.y;
                        double ar, ai;
                        inv_conj_f64(dx, dy, ar, ai);
                        if (k == lane) ar = ai = 0.0;  // the i = j term is excluded (Eq. fmm-E)
#pragma unroll
                        for (int r = 0; r < R; ++r) add_term64<COMP, false>(acc[r], s_w[r * NT + q], ar, ai);
                    }
                    continue;
                }
                if (self && s == W / 2 && wid >= W / 2) continue;  // the other warp of the slice pair has it
                double col[R][NC];
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int q = 0; q < NC; ++q) col[r][q] = s_col[(r * NC + q) * SB + gj * NT + c * 32 + lane];
#pragma unroll 4
                for (int k = 0; k < 32; ++k) {
                    const int q = c * 32 + ((lane + k) & 31);
                    const double2 sp = s_pos[q];
                    const double dx = p.x - sp.x, dy = p.y - sp.y;
                    double ar, ai;  // 1/d = ar - i ai
                    inv_conj_f64(dx, dy, ar, ai);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        add_term64<COMP, false>(acc[r], s_w[r * NT + q], ar, ai);
                        add_term64<COMP, true>(col[r], w[r], ar, ai);  // 1/(eta_j - eta_i) = -1/d
#pragma unroll
                        for (int u = 0; u < NC; ++u) col[r][u] = __shfl_sync(0xffffffffu, col[r][u], (lane + 1) & 31);
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int u = 0; u < NC; ++u) s_col[(r * NC + u) * SB + gj * NT + c * 32 + lane] = col[r][u];
            }
        }
        if (diag) {  // with the column sums of the same nodes
            __syncthreads();
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < NC; ++u) s_col[(r * NC + u) * SB + gi * NT + threadIdx.x] += acc[r][u];
        } else if (i < a.N) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                a.partial[((size_t)J * R + r) * a.N + i] = make_double2(COMP == 1 ? 0.0 : acc[r][0],
                                                                        COMP == 2 ? 0.0 : acc[r][NC - 1]);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < SB; e += NT) {
        const int j = J * SB + e;
        if (j >= a.N) break;
#pragma unroll
        for (int r = 0; r < R; ++r)
            a.partial[((size_t)I * R + r) * a.N + j] = make_double2(COMP == 1 ? 0.0 : s_col[(r * NC) * SB + e],
                                                                    COMP == 2 ? 0.0 : s_col[(r * NC + NC - 1) * SB + e]);
    }
}

// The same for blocks of 32 nodes, the 32 steps of a pair of blocks shared by
// kSymSplit warps (warp v takes the steps from 32 v / kSymSplit on), whose row
// and column sums are added in warp order.  At N = 768 an SM has two such
// pairs: with one warp each the FP64 pipe waits for the 64-cycle latency of
// dependent instructions (a product through the C ABI 30 us), with four it is
// busy (20 us; the kernel 8.4 us, 0.96 of the pipe's rate; the ordered kernel
// on 18 SMs took 82 to 125 us).  FAST: 1/d on the FP32 pipe; with few blocks per
// SM its longer chain is what counts (12.3 us at N = 768), so it is taken from
// kSymFastBlocks blocks per SM on.
constexpr int kSymSplit = 4;
constexpr int kSymFastBlocks = 6;

template <bool FAST>
__device__ __forceinline__ void pair_inv64(double dx, double dy, double& ar, double& ai) {
    if (FAST) {
        inv_conj_f64(dx, dy, ar, ai);
    } else {
        const double inv = recip_f64(fma(dx, dx, dy * dy));
        ar = dx * inv;
        ai = dy * inv;
    }
}

// The block that brings the last partial sums of a node block (an atomic count
// per node block; nothing waits) adds them in slot order and applies the
// operator's epilogue: one launch and about 2 us less per product than a
// reduction of its own, which was half as long as the sums at N = 768.
template <int R, int MODE, int COMP, bool FAST>
__global__ void __launch_bounds__(32 * kSymSplit) pairsum64_sym32_kernel(Pair64SymArgs a, ReduceArgs ra) {
    constexpr int NC = COMP == 0 ? 2 : 1, KS = 32 / kSymSplit;
    __shared__ double2 s_pos[32], s_w[R][32];
    __shared__ double s_row[kSymSplit][R * NC][32], s_col[kSymSplit][R * NC][32];
    __shared__ double2 s_sums[kSymSplit][R][32];
    if (a.done != nullptr && *a.done) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int I, J;
    sym_blocks(a.nt, blockIdx.x, I, J);
    const int i = I * 32 + lane, j = J * 32 + lane;
    double2 p, w[R];
    load_node64<R, MODE>(a, i, p, w);
    if (wid == 0) {
        double2 pj = p, wj[R];
#pragma unroll
        for (int r = 0; r < R; ++r) wj[r] = w[r];
        if (I != J) load_node64<R, MODE>(a, j, pj, wj);
        s_pos[lane] = pj;
#pragma unroll
        for (int r = 0; r < R; ++r) s_w[r][lane] = wj[r];
    }
    __syncthreads();
    double acc[R][NC], col[R][NC];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int u = 0; u < NC; ++u) acc[r][u] = col[r][u] = 0.0;
    const int k0 = wid * KS;
    if (I == J) {  // every ordered pair by its own row
#pragma unroll
        for (int k = k0; k < k0 + KS; ++k) {
            const double2 sp = s_pos[k];
            const double dx = p.x - sp.x, dy = p.y - sp.y;
            double ar, ai;
            pair_inv64<FAST>(dx, dy, ar, ai);
            if (k == lane) ar = ai = 0.0;  // the i = j term is excluded (Eq. fmm-E)
#pragma unroll
            for (int r = 0; r < R; ++r) add_term64<COMP, false>(acc[r], s_w[r][k], ar, ai);
        }
    } else {
#pragma unroll
        for (int k = k0; k < k0 + KS; ++k) {
            const int q = (lane + k) & 31;
            const double2 sp = s_pos[q];
            const double dx = p.x - sp.x, dy = p.y - sp.y;
            double ar, ai;
            pair_inv64<FAST>(dx, dy, ar, ai);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                add_term64<COMP, false>(acc[r], s_w[r][q], ar, ai);
                add_term64<COMP, true>(col[r], w[r], ar, ai);
#pragma unroll
                for (int u = 0; u < NC; ++u) col[r][u] = __shfl_sync(0xffffffffu, col[r][u], (lane + 1) & 31);
            }
        }
    }
    const int held = (lane + k0 + KS) & 31;  // the source whose sum this lane holds now
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            s_row[wid][r * NC + u][lane] = acc[r][u];
            s_col[wid][r * NC + u][held] = col[r][u];
        }
    __syncthreads();
    // warp 0: row sums to slot J; warp 1: column sums to slot I
    const int mine = wid == 0 ? i : j;
    if (wid <= (I != J ? 1 : 0) && mine < a.N) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            double v[NC];
#pragma unroll
            for (int u = 0; u < NC; ++u) {
                const double(*src)[R * NC][32] = wid == 0 ? s_row : s_col;
                v[u] = src[0][r * NC + u][lane];
#pragma unroll
                for (int q = 1; q < kSymSplit; ++q) v[u] += src[q][r * NC + u][lane];
            }
            a.partial[((size_t)(wid == 0 ? J : I) * R + r) * a.N + mine] =
                make_double2(COMP == 1 ? 0.0 : v[0], COMP == 2 ? 0.0 : v[NC - 1]);
        }
    }
    __shared__ int s_last;
    __threadfence();  // the sums before the counts
    __syncthreads();
    if (threadIdx.x == 0) {
        int last = atomicAdd(&a.count[I], 1) == a.nt - 1 ? 1 : 0;
        if (I != J && atomicAdd(&a.count[J], 1) == a.nt - 1) last |= 2;
        if (last & 1) a.count[I] = 0;  // every block has counted: ready for the next product
        if (last & 2) a.count[J] = 0;
        if (last) __threadfence();
        s_last = last;
    }
    __syncthreads();
    const int last = s_last;
    for (int which = 0; which < 2; ++which) {  // the same in every thread
        if (!(last >> which & 1)) continue;
        const int node = (which == 0 ? I : J) * 32 + lane;
        double2(*s_sum)[R][32] = s_sums;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            double sx = 0.0, sy = 0.0;
            if (node < a.N) {
#pragma unroll 8
                for (int q = wid; q < a.nt; q += kSymSplit) {
                    const double2 v = __ldcg(a.partial + ((size_t)q * R + r) * a.N + node);
                    sx += v.x;
                    sy += v.y;
                }
            }
            s_sum[wid][r][lane] = make_double2(sx, sy);
        }
        __syncthreads();
        if (wid == 0 && node < a.N) {
            double2 z[kMaxRHS] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int q = 0; q < kSymSplit; ++q) {
                    z[r].x += s_sum[q][r][lane].x;
                    z[r].y += s_sum[q][r][lane].y;
                }
            epilogue_apply(ra, node, z[0], z[1]);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ FP32
// Source positions are stored relative to one reference node per source tile
// (off32), and each target forms its own offset to that reference from its
// hi/lo split, so that the difference eta_i - eta_j of two nearby nodes keeps
// its leading bits instead of being lost to the magnitude of eta.
struct Pair32Args {
    const float4* et32;
    const float4* ref32;
    const float2* off32;
    int N;
    const double2* w0;
    const double2* w1;
    const double* x0;
    const double* x1;
    const float2* s32;
    float2* partial;
    int tiles_src;
    int tiles_per_chunk;
    const int* done;
};

template <int R, int MODE>
__global__ void __launch_bounds__(kThreads32) pairsum32_kernel(Pair32Args a) {
    constexpr int S = kSrcTile32, T = kTargets32, NT = kThreads32;
    static_assert(S == NT, "one source per thread per tile load");
    __shared__ float4 s_src[S];          // (off.x, off.y, w0.x, w0.y)
    __shared__ float2 s_w1[R > 1 ? S : 1];
    if (a.done != nullptr && *a.done) return;
    const int N = a.N;
    const int tgt0 = blockIdx.x * (NT * T);

    float4 th[T];
    float ox[T], oy[T], ax[T][R], ay[T][R];
    int idx[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        idx[t] = tgt0 + t * NT + threadIdx.x;
        th[t] = a.et32[min(idx[t], N - 1)];
#pragma unroll
        for (int r = 0; r < R; ++r) ax[t][r] = ay[t][r] = 0.0f;
    }

    const int tb = blockIdx.y * a.tiles_per_chunk;
    const int te = min(tb + a.tiles_per_chunk, a.tiles_src);
    for (int tile = tb; tile < te; ++tile) {
        const int j0 = tile * S;
        const float4 ref = a.ref32[tile];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            ox[t] = (th[t].x - ref.x) + (th[t].z - ref.z);
            oy[t] = (th[t].y - ref.y) + (th[t].w - ref.w);
        }
        __syncthreads();
        {
            const int k = threadIdx.x;
            const int j = j0 + k;
            float4 v;
            float2 w1 = make_float2(0.f, 0.f);
            if (j < N) {
                const float2 off = a.off32[j];
                float2 w0;
                if (MODE == W_COMPLEX) {
                    const double2 w = a.w0[j];
                    w0 = make_float2((float)w.x, (float)w.y);
                    if (R > 1) {
                        const double2 u = a.w1[j];
                        w1 = make_float2((float)u.x, (float)u.y);
                    }
                } else {
                    const float2 sc = a.s32[j];
                    const float x0 = (float)a.x0[j];
                    w0 = make_float2(sc.x * x0, sc.y * x0);
                    if (R > 1) {
                        const float x1 = (float)a.x1[j];
                        w1 = make_float2(sc.x * x1, sc.y * x1);
                    }
                }
                v = make_float4(off.x, off.y, w0.x, w0.y);
            } else {
                v = make_float4(kFar32, kFar32, 0.f, 0.f);
            }
            s_src[k] = v;
            if (R > 1) s_w1[k] = w1;
        }
        __syncthreads();
        const bool diag = (j0 < tgt0 + NT * T) && (tgt0 < j0 + S);
        if (!diag) {
#pragma unroll 4
            for (int k = 0; k < S; ++k) {
                const float4 sv = s_src[k];
                float2 u;
                if (R > 1) u = s_w1[k];
#pragma unroll
                for (int t = 0; t < T; ++t) {
                    const float dx = ox[t] - sv.x, dy = oy[t] - sv.y;
                    const float inv = recip_f32(fmaf(dx, dx, dy * dy));
                    const float ar = dx * inv, ai = dy * inv;
                    ax[t][0] = fmaf(sv.z, ar, ax[t][0]);
                    ax[t][0] = fmaf(sv.w, ai, ax[t][0]);
                    ay[t][0] = fmaf(sv.w, ar, ay[t][0]);
                    ay[t][0] = fmaf(-sv.z, ai, ay[t][0]);
                    if (R > 1) {
                        ax[t][R - 1] = fmaf(u.x, ar, ax[t][R - 1]);
                        ax[t][R - 1] = fmaf(u.y, ai, ax[t][R - 1]);
                        ay[t][R - 1] = fmaf(u.y, ar, ay[t][R - 1]);
                        ay[t][R - 1] = fmaf(-u.x, ai, ay[t][R - 1]);
                    }
                }
            }
        } else {
            for (int k = 0; k < S; ++k) {
                const float4 sv = s_src[k];
                float2 u;
                if (R > 1) u = s_w1[k];
                const int j = j0 + k;
#pragma unroll
                for (int t = 0; t < T; ++t) {
                    const float dx = ox[t] - sv.x, dy = oy[t] - sv.y;
                    float inv = recip_f32(fmaf(dx, dx, dy * dy));
                    inv = (j == idx[t]) ? 0.0f : inv;
                    const float ar = dx * inv, ai = dy * inv;
                    ax[t][0] = fmaf(sv.z, ar, ax[t][0]);
                    ax[t][0] = fmaf(sv.w, ai, ax[t][0]);
                    ay[t][0] = fmaf(sv.w, ar, ay[t][0]);
                    ay[t][0] = fmaf(-sv.z, ai, ay[t][0]);
                    if (R > 1) {
                        ax[t][R - 1] = fmaf(u.x, ar, ax[t][R - 1]);
                        ax[t][R - 1] = fmaf(u.y, ai, ax[t][R - 1]);
                        ay[t][R - 1] = fmaf(u.y, ar, ay[t][R - 1]);
                        ay[t][R - 1] = fmaf(-u.x, ai, ay[t][R - 1]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {
        if (idx[t] < N) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                a.partial[((size_t)blockIdx.y * R + r) * N + idx[t]] = make_float2(ax[t][r], ay[t][r]);
        }
    }
}

// Packed FP32 variant: each thread owns 2 x kPairs32 targets, two per float2
// (x and y lanes); sources are stored duplicated so that one packed
// instruction serves both lanes.
constexpr int kPairs32 = kTargets32 / 2;

// z += w / d = w conj(d) / |d|^2 for both lanes, inv = 1/|d|^2 (0 for i = j)
template <int R, int COMP>
__device__ __forceinline__ void accumulate32(const float4 (*s_w)[kSrcTile32], int k, float2 dx, float2 dy,
                                             float2 inv, float2* ax, float2* ay) {
    if (COMP == 0) {
        const float2 ar = mul2(dx, inv), ai = mul2(dy, inv);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 w = s_w[r][k];
            const float2 wx = make_float2(w.x, w.y), wy = make_float2(w.z, w.w);
            ax[r] = fma2(wx, ar, fma2(wy, ai, ax[r]));
            ay[r] = fma2(wy, ar, fma2(neg2(wx), ai, ay[r]));
        }
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 w = s_w[r][k];
            const float2 wx = make_float2(w.x, w.y), wy = make_float2(w.z, w.w);
            if (COMP == 1)  // Im(w conj d) = wy dx - wx dy
                ay[r] = fma2(fma2(neg2(wx), dy, mul2(wy, dx)), inv, ay[r]);
            else            // Re(w conj d) = wx dx + wy dy
                ax[r] = fma2(fma2(wy, dy, mul2(wx, dx)), inv, ax[r]);
        }
    }
}

// COMP = 1 (2): only Im z (Re z) is formed, 3 instead of 4 + 2 FP32 operations
// per pair and right-hand side; the other part of the partial sum is written as 0.
template <int R, int MODE, int COMP>
__global__ void __launch_bounds__(kThreads32) pairsum32x2_kernel(Pair32Args a) {
    constexpr int S = kSrcTile32, NT = kThreads32, P = kPairs32;
    static_assert(S == NT, "one source per thread per tile load");
    __shared__ float4 s_o[S];          // (ox, ox, oy, oy)
    __shared__ float4 s_w[R][S];       // (wx, wx, wy, wy)
    if (a.done != nullptr && *a.done) return;
    const int N = a.N;
    const int tgt0 = blockIdx.x * (NT * kTargets32);
    float4 th[2 * P];
    int idx[2 * P];
    float2 ax[P][R], ay[P][R];
#pragma unroll
    for (int t = 0; t < 2 * P; ++t) {
        idx[t] = tgt0 + t * NT + threadIdx.x;
        th[t] = a.et32[min(idx[t], N - 1)];
    }
#pragma unroll
    for (int u = 0; u < P; ++u)
#pragma unroll
        for (int r = 0; r < R; ++r) ax[u][r] = ay[u][r] = f2(0.f);
    const int tb = blockIdx.y * a.tiles_per_chunk;
    const int te = min(tb + a.tiles_per_chunk, a.tiles_src);
    for (int tile = tb; tile < te; ++tile) {
        const int j0 = tile * S;
        const float4 ref = a.ref32[tile];
        float2 ox[P], oy[P];
#pragma unroll
        for (int u = 0; u < P; ++u) {
            const float4 ta = th[2 * u], tb2 = th[2 * u + 1];
            ox[u] = make_float2((ta.x - ref.x) + (ta.z - ref.z), (tb2.x - ref.x) + (tb2.z - ref.z));
            oy[u] = make_float2((ta.y - ref.y) + (ta.w - ref.w), (tb2.y - ref.y) + (tb2.w - ref.w));
        }
        __syncthreads();
        {
            const int k = threadIdx.x;
            const int j = j0 + k;
            if (j < N) {
                const float2 off = a.off32[j];
                s_o[k] = make_float4(off.x, off.x, off.y, off.y);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float2 w;
                    if (MODE == W_COMPLEX) {
                        const double2 wd = (r == 0) ? a.w0[j] : a.w1[j];
                        w = make_float2((float)wd.x, (float)wd.y);
                    } else {
                        const float2 sc = a.s32[j];
                        const float xv = (float)((r == 0) ? a.x0[j] : a.x1[j]);
                        w = make_float2(sc.x * xv, sc.y * xv);
                    }
                    s_w[r][k] = make_float4(w.x, w.x, w.y, w.y);
                }
            } else {
                s_o[k] = make_float4(kFar32, kFar32, kFar32, kFar32);
#pragma unroll
                for (int r = 0; r < R; ++r) s_w[r][k] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        __syncthreads();
        const bool diag = (j0 < tgt0 + NT * kTargets32) && (tgt0 < j0 + S);
        if (!diag) {
#pragma unroll 4
            for (int k = 0; k < S; ++k) {
                const float4 so = s_o[k];
                const float2 sx = make_float2(so.x, so.y), sy = make_float2(so.z, so.w);
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    const float2 dx = sub2(ox[u], sx), dy = sub2(oy[u], sy);
                    const float2 r2 = fma2(dy, dy, mul2(dx, dx));
                    const float2 inv = make_float2(recip_f32(r2.x), recip_f32(r2.y));
                    accumulate32<R, COMP>(s_w, k, dx, dy, inv, ax[u], ay[u]);
                }
            }
        } else {
            for (int k = 0; k < S; ++k) {
                const float4 so = s_o[k];
                const float2 sx = make_float2(so.x, so.y), sy = make_float2(so.z, so.w);
                const int j = j0 + k;
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    const float2 dx = sub2(ox[u], sx), dy = sub2(oy[u], sy);
                    const float2 r2 = fma2(dy, dy, mul2(dx, dx));
                    float i0 = recip_f32(r2.x), i1 = recip_f32(r2.y);
                    i0 = (j == idx[2 * u]) ? 0.f : i0;
                    i1 = (j == idx[2 * u + 1]) ? 0.f : i1;
                    const float2 inv = make_float2(i0, i1);
                    accumulate32<R, COMP>(s_w, k, dx, dy, inv, ax[u], ay[u]);
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < P; ++u) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (idx[2 * u] < N)
                a.partial[((size_t)blockIdx.y * R + r) * N + idx[2 * u]] = make_float2(ax[u][r].x, ay[u][r].x);
            if (idx[2 * u + 1] < N)
                a.partial[((size_t)blockIdx.y * R + r) * N + idx[2 * u + 1]] = make_float2(ax[u][r].y, ay[u][r].y);
        }
    }
}

// Each unordered pair once: one reciprocal (the ordered kernel's bound) serves
// both directions.  As the double-float kernel below: a block takes a pair (I, J) of
// blocks of kSrcTile32 nodes; a warp has 128 rows, four per thread in two packs, so
// that the shared-memory reads and the shuffles of a step serve four pairs.  I - N
// with real A (a whole product): N = 2,048 23 us against 26 with the ordered kernel,
// 8,192 29.5 against 42, 16,384 72 against 103, 65,536 915 against 1,079.
constexpr int kSym32Warps = kSrcTile32 / 128;

template <int R, int MODE, int COMP>
__global__ void __launch_bounds__(32 * kSym32Warps) pairsum32_sym_kernel(Pair32Args a, int nt) {
    constexpr int S = kSrcTile32, NT = 32 * kSym32Warps, NS = S / 32, P = 2;
    constexpr int NC = COMP == 0 ? 2 : 1;  // parts of z kept: both, Im (COMP 1) or Re (COMP 2)
    static_assert(2 * P * NT == S, "four rows per thread");
    __shared__ float4 s_src[S];         // (x, y, wx, wy) of the first right-hand side
    __shared__ float2 s_w1[R > 1 ? S : 1];
    __shared__ float2 s_col[R][NC][S];  // column sums, one per lane of the packs
    if (a.done != nullptr && *a.done) return;
    const int N = a.N, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int I, J;
    sym_blocks(nt, blockIdx.x, I, J);
    const float4 ref = a.ref32[J];
    auto weight = [&](int r, int j) -> float2 {
        if (MODE == W_COMPLEX) {
            const double2 wd = (r == 0) ? a.w0[j] : a.w1[j];
            return make_float2((float)wd.x, (float)wd.y);
        }
        const float2 sc = a.s32[j];
        const float x = (float)((r == 0) ? a.x0[j] : a.x1[j]);
        return make_float2(sc.x * x, sc.y * x);
    };
    // rows; those past the end lie far on the other side than the columns past the
    // end, with weight 0
    const int ib = I * S + wid * 128 + lane;
    float2 ox[P], oy[P], wx[P][R], wy[P][R], acc[P][R][NC];
#pragma unroll
    for (int u = 0; u < P; ++u) {
        float px[2], py[2];
        float2 w[2][R];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int i = ib + 64 * u + 32 * v;
            px[v] = py[v] = -kFar32;
            if (i < N) {
                const float4 t = a.et32[i];
                px[v] = (t.x - ref.x) + (t.z - ref.z);
                py[v] = (t.y - ref.y) + (t.w - ref.w);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) w[v][r] = i < N ? weight(r, i) : f2(0.f);
        }
        ox[u] = make_float2(px[0], px[1]);
        oy[u] = make_float2(py[0], py[1]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            wx[u][r] = make_float2(w[0][r].x, w[1][r].x);
            wy[u][r] = make_float2(w[0][r].y, w[1][r].y);
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[u][r][c] = f2(0.f);
        }
    }
    for (int k = threadIdx.x; k < S; k += NT) {
        const int j = J * S + k;
        const float2 o = j < N ? a.off32[j] : f2(kFar32);
        const float2 w = j < N ? weight(0, j) : f2(0.f);
        s_src[k] = make_float4(o.x, o.y, w.x, w.y);
        if (R > 1) s_w1[k] = j < N ? weight(R - 1, j) : f2(0.f);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) s_col[r][c][k] = f2(0.f);
    }
    // z += w / d = w conj(d) / |d|^2
    auto add = [&](float2* z, float2 vx, float2 vy, float2 dx, float2 dy, float2 inv) {
        if (COMP == 0) {
            const float2 ar = mul2(dx, inv), ai = mul2(dy, inv);
            z[0] = fma2(vx, ar, fma2(vy, ai, z[0]));
            z[NC - 1] = fma2(vy, ar, fma2(neg2(vx), ai, z[NC - 1]));
        } else if (COMP == 1) {
            z[0] = fma2(fma2(neg2(vx), dy, mul2(vy, dx)), inv, z[0]);
        } else {
            z[0] = fma2(fma2(vy, dy, mul2(vx, dx)), inv, z[0]);
        }
    };
    if (I == J) {  // every ordered pair by its own row
        __syncthreads();
#pragma unroll 2
        for (int q = 0; q < S; ++q) {
            const float4 sv = s_src[q];
#pragma unroll
            for (int u = 0; u < P; ++u) {
                const float2 dx = sub2(ox[u], f2(sv.x)), dy = sub2(oy[u], f2(sv.y));
                const float2 r2 = fma2(dy, dy, mul2(dx, dx));
                float2 inv = make_float2(recip_f32(r2.x), recip_f32(r2.y));
                inv.x = (J * S + q == ib + 64 * u) ? 0.f : inv.x;  // the i = j term is excluded (Eq. fmm-E)
                inv.y = (J * S + q == ib + 64 * u + 32) ? 0.f : inv.y;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float2 v = r == 0 ? make_float2(sv.z, sv.w) : s_w1[R > 1 ? q : 0];
                    add(acc[u][r], f2(v.x), f2(v.y), dx, dy, inv);
                }
            }
        }
    } else {
        for (int s = 0; s < NS; ++s) {
            __syncthreads();  // the slices' sums are back in shared memory
            const int c0 = ((NS / kSym32Warps * wid + s) & (NS - 1)) * 32;
            float2 col[R][NC];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < NC; ++c) col[r][c] = s_col[r][c][c0 + lane];
#pragma unroll 4
            for (int k = 0; k < 32; ++k) {
                const int q = c0 + ((lane + k) & 31);
                const float4 sv = s_src[q];
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    const float2 dx = sub2(ox[u], f2(sv.x)), dy = sub2(oy[u], f2(sv.y));
                    const float2 r2 = fma2(dy, dy, mul2(dx, dx));
                    const float2 inv = make_float2(recip_f32(r2.x), recip_f32(r2.y));
                    const float2 ninv = neg2(inv);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float2 v = r == 0 ? make_float2(sv.z, sv.w) : s_w1[R > 1 ? q : 0];
                        add(acc[u][r], f2(v.x), f2(v.y), dx, dy, inv);
                        add(col[r], wx[u][r], wy[u][r], dx, dy, ninv);  // 1/(eta_j - eta_i) = -1/d
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        col[r][c].x = __shfl_sync(0xffffffffu, col[r][c].x, (lane + 1) & 31);
                        col[r][c].y = __shfl_sync(0xffffffffu, col[r][c].y, (lane + 1) & 31);
                    }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < NC; ++c) s_col[r][c][c0 + lane] = col[r][c];
        }
        __syncthreads();
        for (int k = threadIdx.x; k < S; k += NT) {  // column sums to slot I
            const int j = J * S + k;
            if (j >= N) break;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float2 re = s_col[r][0][k], im = s_col[r][NC - 1][k];
                a.partial[((size_t)I * R + r) * N + j] =
                    make_float2(COMP == 1 ? 0.f : re.x + re.y, COMP == 2 ? 0.f : im.x + im.y);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < P; ++u)  // row sums to slot J
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 re = acc[u][r][0], im = acc[u][r][NC - 1];
            const int i = ib + 64 * u;
            if (i < N)
                a.partial[((size_t)J * R + r) * N + i] = make_float2(COMP == 1 ? 0.f : re.x, COMP == 2 ? 0.f : im.x);
            if (i + 32 < N)
                a.partial[((size_t)J * R + r) * N + i + 32] =
                    make_float2(COMP == 1 ? 0.f : re.y, COMP == 2 ? 0.f : im.y);
        }
}

// ------------------------------------------------------------------ double-float (df32)
// (arithmetic helpers in pairmath.cuh)
struct PairDFArgs {
    const double2* et;
    const double2* ref64;
    const float4* offdf;   // per node: (dx.h, dy.h, dx.l, dy.l) of eta_j - ref(tile(j))
    int N;
    const double2* w0;
    const double2* w1;
    const double* x0;
    const double* x1;
    const double2* s;
    float4* partial;       // [chunk][rhs][N]: (re.h, re.l, im.h, im.l)
    int tiles_src;
    int tiles_per_chunk;
    const int* done;
};

template <int R, int MODE>
__global__ void __launch_bounds__(kThreadsDF) pairsumdf_kernel(PairDFArgs a) {
    constexpr int S = kSrcTile32, T = kTargetsDF, NT = kThreadsDF;
    static_assert(S == NT, "one source per thread per tile load");
    __shared__ float4 s_off[S];
    __shared__ float4 s_w[R][S];  // (wx.h, wx.l, wy.h, wy.l)
    if (a.done != nullptr && *a.done) return;
    const int N = a.N;
    const int tgt0 = blockIdx.x * (NT * T);

    double2 p[T];
    df acc_re[T][R], acc_im[T][R];
    int idx[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        idx[t] = tgt0 + t * NT + threadIdx.x;
        p[t] = a.et[min(idx[t], N - 1)];
#pragma unroll
        for (int r = 0; r < R; ++r) acc_re[t][r] = acc_im[t][r] = df{0.f, 0.f};
    }

    const int tb = blockIdx.y * a.tiles_per_chunk;
    const int te = min(tb + a.tiles_per_chunk, a.tiles_src);
    for (int tile = tb; tile < te; ++tile) {
        const int j0 = tile * S;
        const double2 ref = a.ref64[tile];
        df ox[T], oy[T];
#pragma unroll
        for (int t = 0; t < T; ++t) {  // target offsets, once per tile, in FP64
            ox[t] = df_split(p[t].x - ref.x);
            oy[t] = df_split(p[t].y - ref.y);
        }
        __syncthreads();
        {
            const int k = threadIdx.x;
            const int j = j0 + k;
            if (j < N) {
                s_off[k] = a.offdf[j];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    double2 w;
                    if (MODE == W_COMPLEX) {
                        w = (r == 0) ? a.w0[j] : a.w1[j];
                    } else {
                        const double2 sc = a.s[j];
                        const double x = (r == 0) ? a.x0[j] : a.x1[j];
                        w = make_double2(sc.x * x, sc.y * x);
                    }
                    const df wx = df_split(w.x), wy = df_split(w.y);
                    s_w[r][k] = make_float4(wx.h, wx.l, wy.h, wy.l);
                }
            } else {
                s_off[k] = make_float4(kFar32, kFar32, 0.f, 0.f);
#pragma unroll
                for (int r = 0; r < R; ++r) s_w[r][k] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        __syncthreads();
        const bool diag = (j0 < tgt0 + NT * T) && (tgt0 < j0 + S);
#pragma unroll 2
        for (int k = 0; k < S; ++k) {
            const float4 so = s_off[k];
            const int j = j0 + k;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const df dx = df_sub(ox[t].h, ox[t].l, so.x, so.z);
                const df dy = df_sub(oy[t].h, oy[t].l, so.y, so.w);
                // |d|^2 = dx.h^2 + dy.h^2 + 2 dx.h dx.l + 2 dy.h dy.l  (lo^2 terms below 2^-48)
                const float px = __fmul_rn(dx.h, dx.h);
                float ex = fmaf(dx.h, dx.h, -px);
                ex = fmaf(dx.h, dx.l + dx.l, ex);
                const float py = __fmul_rn(dy.h, dy.h);
                float ey = fmaf(dy.h, dy.h, -py);
                ey = fmaf(dy.h, dy.l + dy.l, ey);
                float rh, re;
                two_sum(px, py, rh, re);
                const float rl = __fadd_rn(__fadd_rn(ex, ey), re);
                // 1/|d|^2: one Newton step from the 2^-23 seed gives ~2^-46
                float y = recip_f32(rh);
                if (diag && j == idx[t]) y = 0.0f;  // the i = j term is excluded (Eq. fmm-E)
                float e = fmaf(-rh, y, 1.0f);
                e = fmaf(-rl, y, e);
                const df inv = df{y, __fmul_rn(y, e)};
                const df ar = df_mul(dx, inv);  // 1/d = ar - i ai
                const df ai = df_mul(dy, inv);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4 w = s_w[r][k];
                    const df wx{w.x, w.y}, wy{w.z, w.w};
                    // z += w (ar - i ai): re += wx ar + wy ai, im += wy ar - wx ai
                    df_acc(acc_re[t][r], df_mul(wx, ar));
                    df_acc(acc_re[t][r], df_mul(wy, ai));
                    df_acc(acc_im[t][r], df_mul(wy, ar));
                    const df q = df_mul(wx, ai);
                    df_acc(acc_im[t][r], df{-q.h, -q.l});
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {
        if (idx[t] < N) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                a.partial[((size_t)blockIdx.y * R + r) * N + idx[t]] =
                    make_float4(acc_re[t][r].h, acc_re[t][r].l, acc_im[t][r].h, acc_im[t][r].l);
        }
    }
}

// Packed variant: each thread owns two targets held in the x and y lanes of
// float2 registers; every double-float operation of a pair is one packed
// instruction for both targets.  Source values are stored duplicated (v, v)
// in shared memory so that they broadcast to both lanes.
template <int R, int MODE, int COMP>
__global__ void __launch_bounds__(kThreadsDF) pairsumdf2_kernel(PairDFArgs a) {
    constexpr int S = kSrcTile32, NT = kThreadsDF;
    static_assert(S == NT, "one source per thread per tile load");
    static_assert(kTargetsDF == 2, "two targets per thread, one per lane");
    __shared__ float4 s_off[2][S];       // (xh, xh, yh, yh), (xl, xl, yl, yl)
    __shared__ float4 s_w[R][2][S];      // (wxh, wxh, wxl, wxl), (wyh, wyh, wyl, wyl)
    if (a.done != nullptr && *a.done) return;
    const int N = a.N;
    const int tgt0 = blockIdx.x * (NT * 2);
    const int i0 = tgt0 + threadIdx.x, i1 = tgt0 + NT + threadIdx.x;
    const double2 p0 = a.et[min(i0, N - 1)], p1 = a.et[min(i1, N - 1)];
    df2 are[R], aim[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        are[r] = df2{f2(0.f), f2(0.f)};
        aim[r] = df2{f2(0.f), f2(0.f)};
    }
    const int tb = blockIdx.y * a.tiles_per_chunk;
    const int te = min(tb + a.tiles_per_chunk, a.tiles_src);
    for (int tile = tb; tile < te; ++tile) {
        const int j0 = tile * S;
        const double2 ref = a.ref64[tile];
        const df ox0 = df_split(p0.x - ref.x), ox1 = df_split(p1.x - ref.x);
        const df oy0 = df_split(p0.y - ref.y), oy1 = df_split(p1.y - ref.y);
        const float2 oxh = make_float2(ox0.h, ox1.h), oxl = make_float2(ox0.l, ox1.l);
        const float2 oyh = make_float2(oy0.h, oy1.h), oyl = make_float2(oy0.l, oy1.l);
        __syncthreads();
        {
            const int k = threadIdx.x;
            const int j = j0 + k;
            if (j < N) {
                const float4 o = a.offdf[j];
                s_off[0][k] = make_float4(o.x, o.x, o.y, o.y);
                s_off[1][k] = make_float4(o.z, o.z, o.w, o.w);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    double2 w;
                    if (MODE == W_COMPLEX) {
                        w = (r == 0) ? a.w0[j] : a.w1[j];
                    } else {
                        const double2 sc = a.s[j];
                        const double x = (r == 0) ? a.x0[j] : a.x1[j];
                        w = make_double2(sc.x * x, sc.y * x);
                    }
                    const df wx = df_split(w.x), wy = df_split(w.y);
                    s_w[r][0][k] = make_float4(wx.h, wx.h, wx.l, wx.l);
                    s_w[r][1][k] = make_float4(wy.h, wy.h, wy.l, wy.l);
                }
            } else {
                s_off[0][k] = make_float4(kFar32, kFar32, kFar32, kFar32);
                s_off[1][k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    s_w[r][0][k] = make_float4(0.f, 0.f, 0.f, 0.f);
                    s_w[r][1][k] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
        }
        __syncthreads();
        const bool diag = (j0 < tgt0 + NT * 2) && (tgt0 < j0 + S);
#pragma unroll 2
        for (int k = 0; k < S; ++k) {
            const float4 oa = s_off[0][k], ob = s_off[1][k];
            const df2 dx = df2_sub(oxh, oxl, make_float2(oa.x, oa.y), make_float2(ob.x, ob.y));
            const df2 dy = df2_sub(oyh, oyl, make_float2(oa.z, oa.w), make_float2(ob.z, ob.w));
            const float2 px = mul2(dx.h, dx.h);
            float2 ex = fma2(dx.h, dx.h, neg2(px));
            ex = fma2(dx.h, add2(dx.l, dx.l), ex);
            const float2 py = mul2(dy.h, dy.h);
            float2 ey = fma2(dy.h, dy.h, neg2(py));
            ey = fma2(dy.h, add2(dy.l, dy.l), ey);
            float2 rh, re;
            two_sum2(px, py, rh, re);
            const float2 rl = add2(add2(ex, ey), re);
            float y0 = recip_f32(rh.x), y1 = recip_f32(rh.y);
            if (diag) {  // the i = j term is excluded (Eq. fmm-E)
                y0 = (j0 + k == i0) ? 0.f : y0;
                y1 = (j0 + k == i1) ? 0.f : y1;
            }
            const float2 y = make_float2(y0, y1);
            float2 e = fma2(neg2(rh), y, f2(1.0f));
            e = fma2(neg2(rl), y, e);
            const df2 inv{y, mul2(y, e)};
            const df2 ar = df2_mul(dx, inv);  // 1/d = ar - i ai
            const df2 ai = df2_mul(dy, inv);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 wa = s_w[r][0][k], wb = s_w[r][1][k];
                const df2 wx{make_float2(wa.x, wa.y), make_float2(wa.z, wa.w)};
                const df2 wy{make_float2(wb.x, wb.y), make_float2(wb.z, wb.w)};
                if (COMP != 1) {
                    df2_acc(are[r], df2_mul(wx, ar));
                    df2_acc(are[r], df2_mul(wy, ai));
                }
                if (COMP != 2) {
                    df2_acc(aim[r], df2_mul(wy, ar));
                    df2_dec(aim[r], df2_mul(wx, ai));
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (i0 < N)
            a.partial[((size_t)blockIdx.y * R + r) * N + i0] =
                make_float4(are[r].h.x, are[r].l.x, aim[r].h.x, aim[r].l.x);
        if (i1 < N)
            a.partial[((size_t)blockIdx.y * R + r) * N + i1] =
                make_float4(are[r].h.y, are[r].l.y, aim[r].h.y, aim[r].l.y);
    }
}

// Each unordered pair once: 1/d (49 of the FP32 instructions) serves both
// directions.  A block takes a pair (I, J) of blocks of kSrcTile32 nodes, its four
// warps 64 rows each (two per thread, one per lane of the packed registers); at turn
// s warp v has the 32 columns of slice 2 v + s mod 8, whose sums travel round its
// lanes with the sources and wait in shared memory for the next warp.  At N = 16,384
// with real A a product takes 447 us (FP32 pipe 323; ordered 694), 644 with complex A
// (ordered 900); below 4,096 the 256 steps of one block, about 48 us.  The
// diagonal blocks (1/nt of the pairs) sum every ordered pair by its own row.
constexpr int kSymDFWarps = kSrcTile32 / 64;

template <int R, int MODE, int COMP>
__global__ void __launch_bounds__(32 * kSymDFWarps) pairsumdf_sym_kernel(PairDFArgs a, int nt) {
    constexpr int S = kSrcTile32, NT = 32 * kSymDFWarps, NS = S / 32;
    constexpr int NC = COMP == 0 ? 2 : 1;  // parts of z kept: both, Im (COMP 1) or Re (COMP 2)
    static_assert(2 * NT == S, "two rows per thread");
    __shared__ float4 s_off[2][S];      // (xh, xh, yh, yh), (xl, xl, yl, yl)
    __shared__ float4 s_w[R][2][S];     // (wxh, wxh, wxl, wxl), (wyh, wyh, wyl, wyl)
    __shared__ float4 s_col[R][NC][S];  // (h.x, h.y, l.x, l.y): column sums, one per row lane
    if (a.done != nullptr && *a.done) return;
    const int N = a.N, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int I, J;
    sym_blocks(nt, blockIdx.x, I, J);
    const double2 ref = a.ref64[J];
    auto weight = [&](int r, int j) -> double2 {
        if (MODE == W_COMPLEX) return (r == 0) ? a.w0[j] : a.w1[j];
        const double2 sc = a.s[j];
        const double x = (r == 0) ? a.x0[j] : a.x1[j];
        return make_double2(sc.x * x, sc.y * x);
    };
    // rows: positions against the column block's reference, in FP64 once; rows past
    // the end lie far on the other side than the columns past the end, with weight 0
    const int i0 = I * S + wid * 64 + lane, i1 = i0 + 32;
    df ox[2], oy[2];
    df2 wx[R], wy[R];
    {
        df px[R][2], py[R][2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = u == 0 ? i0 : i1;
            if (i < N) {
                const double2 p = a.et[i];
                ox[u] = df_split(p.x - ref.x);
                oy[u] = df_split(p.y - ref.y);
            } else {
                ox[u] = oy[u] = df{-kFar32, 0.f};
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const double2 w = i < N ? weight(r, i) : make_double2(0.0, 0.0);
                px[r][u] = df_split(w.x);
                py[r][u] = df_split(w.y);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            wx[r] = df2{make_float2(px[r][0].h, px[r][1].h), make_float2(px[r][0].l, px[r][1].l)};
            wy[r] = df2{make_float2(py[r][0].h, py[r][1].h), make_float2(py[r][0].l, py[r][1].l)};
        }
    }
    const float2 oxh = make_float2(ox[0].h, ox[1].h), oxl = make_float2(ox[0].l, ox[1].l);
    const float2 oyh = make_float2(oy[0].h, oy[1].h), oyl = make_float2(oy[0].l, oy[1].l);
    for (int k = threadIdx.x; k < S; k += NT) {
        const int j = J * S + k;
        const float4 o = j < N ? a.offdf[j] : make_float4(kFar32, kFar32, 0.f, 0.f);
        s_off[0][k] = make_float4(o.x, o.x, o.y, o.y);
        s_off[1][k] = make_float4(o.z, o.z, o.w, o.w);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double2 w = j < N ? weight(r, j) : make_double2(0.0, 0.0);
            const df vx = df_split(w.x), vy = df_split(w.y);
            s_w[r][0][k] = make_float4(vx.h, vx.h, vx.l, vx.l);
            s_w[r][1][k] = make_float4(vy.h, vy.h, vy.l, vy.l);
#pragma unroll
            for (int c = 0; c < NC; ++c) s_col[r][c][k] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    df2 acc[R][NC];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[r][c] = df2{f2(0.f), f2(0.f)};
    // 1/d = ar - i ai of the two rows and column q; `self`: i = j may occur (then 0, Eq. fmm-E)
    auto inverse = [&](int q, bool self, df2& ar, df2& ai) {
        const float4 oa = s_off[0][q], ob = s_off[1][q];
        const df2 dx = df2_sub(oxh, oxl, make_float2(oa.x, oa.y), make_float2(ob.x, ob.y));
        const df2 dy = df2_sub(oyh, oyl, make_float2(oa.z, oa.w), make_float2(ob.z, ob.w));
        const float2 px = mul2(dx.h, dx.h);
        float2 ex = fma2(dx.h, dx.h, neg2(px));
        ex = fma2(dx.h, add2(dx.l, dx.l), ex);
        const float2 py = mul2(dy.h, dy.h);
        float2 ey = fma2(dy.h, dy.h, neg2(py));
        ey = fma2(dy.h, add2(dy.l, dy.l), ey);
        float2 rh, re;
        two_sum2(px, py, rh, re);
        const float2 rl = add2(add2(ex, ey), re);
        float y0 = recip_f32(rh.x), y1 = recip_f32(rh.y);
        if (self) {
            y0 = (J * S + q == i0) ? 0.f : y0;
            y1 = (J * S + q == i1) ? 0.f : y1;
        }
        const float2 y = make_float2(y0, y1);
        float2 e = fma2(neg2(rh), y, f2(1.0f));
        e = fma2(neg2(rl), y, e);
        const df2 inv{y, mul2(y, e)};
        ar = df2_mul(dx, inv);
        ai = df2_mul(dy, inv);
    };
    auto row_terms = [&](int q, const df2& ar, const df2& ai) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 wa = s_w[r][0][q], wb = s_w[r][1][q];
            const df2 vx{make_float2(wa.x, wa.y), make_float2(wa.z, wa.w)};
            const df2 vy{make_float2(wb.x, wb.y), make_float2(wb.z, wb.w)};
            if (COMP != 1) {
                df2_acc(acc[r][0], df2_mul(vx, ar));
                df2_acc(acc[r][0], df2_mul(vy, ai));
            }
            if (COMP != 2) {
                df2_acc(acc[r][NC - 1], df2_mul(vy, ar));
                df2_dec(acc[r][NC - 1], df2_mul(vx, ai));
            }
        }
    };
    if (I == J) {
        __syncthreads();
#pragma unroll 2
        for (int q = 0; q < S; ++q) {
            df2 ar, ai;
            inverse(q, true, ar, ai);
            row_terms(q, ar, ai);
        }
    } else {
        for (int s = 0; s < NS; ++s) {
            __syncthreads();  // the slices' sums are back in shared memory
            const int c0 = ((2 * wid + s) & (NS - 1)) * 32;
            df2 col[R][NC];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float4 v = s_col[r][c][c0 + lane];
                    col[r][c] = df2{make_float2(v.x, v.y), make_float2(v.z, v.w)};
                }
#pragma unroll 2
            for (int k = 0; k < 32; ++k) {
                const int q = c0 + ((lane + k) & 31);
                df2 ar, ai;
                inverse(q, false, ar, ai);
                row_terms(q, ar, ai);
#pragma unroll
                for (int r = 0; r < R; ++r) {  // the other direction: 1/(eta_j - eta_i) = -1/d
                    if (COMP != 1) {
                        df2_dec(col[r][0], df2_mul(wx[r], ar));
                        df2_dec(col[r][0], df2_mul(wy[r], ai));
                    }
                    if (COMP != 2) {
                        df2_dec(col[r][NC - 1], df2_mul(wy[r], ar));
                        df2_acc(col[r][NC - 1], df2_mul(wx[r], ai));
                    }
                    const int next = (lane + 1) & 31;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        df2& v = col[r][c];
                        v.h.x = __shfl_sync(0xffffffffu, v.h.x, next);
                        v.h.y = __shfl_sync(0xffffffffu, v.h.y, next);
                        v.l.x = __shfl_sync(0xffffffffu, v.l.x, next);
                        v.l.y = __shfl_sync(0xffffffffu, v.l.y, next);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const df2 v = col[r][c];
                    s_col[r][c][c0 + lane] = make_float4(v.h.x, v.h.y, v.l.x, v.l.y);
                }
        }
        __syncthreads();
        for (int k = threadIdx.x; k < S; k += NT) {  // column sums to slot I
            const int j = J * S + k;
            if (j >= N) break;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                df v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float4 t = s_col[r][c][k];
                    float h, e;
                    two_sum(t.x, t.y, h, e);
                    v[c] = df{h, e + (t.z + t.w)};
                }
                a.partial[((size_t)I * R + r) * N + j] =
                    make_float4(COMP == 1 ? 0.f : v[0].h, COMP == 1 ? 0.f : v[0].l, COMP == 2 ? 0.f : v[NC - 1].h,
                                COMP == 2 ? 0.f : v[NC - 1].l);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)  // row sums to slot J
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = u == 0 ? i0 : i1;
            if (i >= N) continue;
            const df2 re = acc[r][0], im = acc[r][NC - 1];
            const float reh = u ? re.h.y : re.h.x, rel = u ? re.l.y : re.l.x;
            const float imh = u ? im.h.y : im.h.x, iml = u ? im.l.y : im.l.x;
            a.partial[((size_t)J * R + r) * N + i] = make_float4(COMP == 1 ? 0.f : reh, COMP == 1 ? 0.f : rel,
                                                                 COMP == 2 ? 0.f : imh, COMP == 2 ? 0.f : iml);
        }
}

// ------------------------------------------------------------------ reduce + epilogue
// Adds the partial sums of 32 nodes per block and applies the operator's
// epilogue: warp g takes the chunks g, g + 8, ... (coalesced over the nodes,
// all loads independent), then the eight sums are added in order by warp 0.
// Latency bounds it (one thread per node read its chunks one after the other).
constexpr int kReduceGroups = 8;

__global__ void __launch_bounds__(32 * kReduceGroups) reduce_epilogue_kernel(ReduceArgs a) {
    const PairJob& j = a.job;
    __shared__ double2 s_sum[kMaxRHS][kReduceGroups][32];
    if (j.done != nullptr && *j.done) return;
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    const int N = a.N;
    for (int r = 0; r < a.R; ++r) {
        double sx = 0.0, sy = 0.0;
        if (i < N) {
            if (a.ptype == 1) {
#pragma unroll 4
                for (int ch = g; ch < a.chunks; ch += kReduceGroups) {
                    const float2 p = a.p32[((size_t)ch * a.R + r) * N + i];
                    sx += (double)p.x;
                    sy += (double)p.y;
                }
            } else if (a.ptype == 2) {
#pragma unroll 4
                for (int ch = g; ch < a.chunks; ch += kReduceGroups) {
                    const float4 p = a.pdf[((size_t)ch * a.R + r) * N + i];
                    sx += (double)p.x + (double)p.y;
                    sy += (double)p.z + (double)p.w;
                }
            } else {
#pragma unroll 8
                for (int ch = g; ch < a.chunks; ch += kReduceGroups) {
                    const double2 p = a.p64[((size_t)ch * a.R + r) * N + i];
                    sx += p.x;
                    sy += p.y;
                }
            }
        }
        s_sum[r][g][lane] = make_double2(sx, sy);
    }
    __syncthreads();
    if (g != 0 || i >= N) return;
    double2 z[kMaxRHS] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    const int ng = min(kReduceGroups, a.chunks);
    for (int r = 0; r < a.R; ++r)
        for (int q = 0; q < ng; ++q) {
            z[r].x += s_sum[r][q][lane].x;
            z[r].y += s_sum[r][q][lane].y;
        }
    epilogue_apply(a, i, z[0], z[1]);
}

cudaError_t launch_reduce(const Boundary& b, const PairJob& job, int chunks, int ptype,
                          cudaStream_t st, const void* partial = nullptr) {
    ReduceArgs ra = reduce_args(b, job, chunks, ptype);
    if (partial) {
        ra.pdf = static_cast<const float4*>(partial);
        ra.p64 = static_cast<const double2*>(partial);
        ra.p32 = static_cast<const float2*>(partial);
    }
    const ProfToken tok = prof_begin(st, PK_REDUCE);
    reduce_epilogue_kernel<<<(b.N + 31) / 32, 32 * kReduceGroups, 0, st>>>(ra);
    const cudaError_t e = cudaGetLastError();
    // bytes: the partials read plus about four N-vectors of operands and output
    prof_end(tok, PK_REDUCE,
             (double)chunks * job.R * b.N * (ptype == 1 ? 8.0 : 16.0) + 4.0 * 8.0 * b.N, st);
    return e;
}

}  // namespace

// Chunking of the source range: choose the number of source tiles per chunk
// that maximises the fraction of useful block-slots over the launch's waves,
// so the grid covers all SMs even when few target tiles exist.
PairPlan make_plan(int N, int sms, int blocks_per_sm, int targets_per_block, int src_tile) {
    PairPlan p;
    p.tiles_tgt = (N + targets_per_block - 1) / targets_per_block;
    p.tiles_src = (N + src_tile - 1) / src_tile;
    const long slots = std::max(1L, (long)sms * blocks_per_sm);
    double best = -1.0;
    int best_tpc = p.tiles_src;
    const int max_chunks = 64;
    for (int tpc = p.tiles_src; tpc >= 1; --tpc) {
        const int chunks = (p.tiles_src + tpc - 1) / tpc;
        if (chunks > max_chunks) break;
        const long blocks = (long)p.tiles_tgt * chunks;
        const long waves = (blocks + slots - 1) / slots;
        const double eff = (double)p.tiles_tgt * p.tiles_src / ((double)waves * slots * tpc);
        if (eff > best * 1.02) {  // prefer fewer chunks unless clearly better
            best = eff;
            best_tpc = tpc;
        }
    }
    p.tiles_per_chunk = best_tpc;
    p.chunks = (p.tiles_src + best_tpc - 1) / best_tpc;
    return p;
}

// Node blocks of the FP64 kernel that takes each pair once: SB = 32 W G nodes,
// the size whose estimated time (FP64 pipe work of the busiest SM, then the
// partial sums written and read at about 4 TB/s) is least, at most kSymMaxBlocks
// of them (they give 8,256 pairs of blocks, 54 per SM, and 2 KB of partial
// sums per node and right-hand side); none (W = 0) beyond 524,288 nodes.  Small
// domains take 32-node blocks of one warp (N = 768: 300 blocks instead of the
// 18 of the ordered kernel).
constexpr int kSymMaxBlocks = kSymCounts;
constexpr size_t kSymArenaBytes = (size_t)4 << 20;  // N <= 2,048

SymPlan make_sym_plan(int N, int sms) {
    static const int kShape[][2] = {{1, 1}, {2, 1}, {4, 1}, {8, 1}, {8, 2}, {8, 4}, {8, 8}, {8, 16}};
    SymPlan best;
    double best_t = 0.0;
    for (const auto& sh : kShape) {
        const long long SB = 32LL * sh[0] * sh[1], nt = (N + SB - 1) / SB;
        if (nt > kSymMaxBlocks) continue;
        if (best.W == 1) break;  // 32-node blocks wherever they are enough: their kernel splits the steps
        const double blocks = 0.5 * nt * (nt - 1) + 0.5 * nt;  // the diagonal's blocks are half
        const double rounds = std::ceil(blocks / std::max(1, sms));
        const double t = rounds * (double)SB * SB * 10.0 / 4.1e9 + (double)nt * N * 32.0 / 4e12;
        if (best.W == 0 || t < best_t) {
            best_t = t;
            best.W = sh[0];
            best.G = sh[1];
            best.nt = (int)nt;
        }
    }
    return best;
}

int pair_workspace_bytes(const Boundary& b, size_t* bytes) {
    const size_t b64 = (size_t)b.plan64.chunks * kMaxRHS * b.N * sizeof(double2);
    const size_t b32 = (size_t)b.plan32.chunks * kMaxRHS * b.N * sizeof(float2);
    const size_t bdf = (size_t)b.plandf.chunks * kMaxRHS * b.N * sizeof(float4);
    *bytes = std::max(std::max(b64, b32), bdf);
    // the sums of the FP64 kernel that takes each pair once, where they are small
    // (sym_workspace has larger ones from the pool for the one product)
    const size_t bs = (size_t)b.sym64.nt * kMaxRHS * b.N * sizeof(double2);
    if (b.sym64.W > 0 && bs <= kSymArenaBytes) *bytes = std::max(*bytes, bs);
    return GNK_OK;
}

// Partial-sum workspace of `need` bytes: the handle's own, or one from the pool
// that is kept (and grown) with the handle.
static int partial_workspace(const Boundary& b, size_t need, void** partial, cudaStream_t st) {
    *partial = b.partial;
    if (need <= b.partial_bytes) return GNK_OK;
    if (need > b.partial_x_bytes) {
        if (b.partial_x) pool_free(b.partial_x, st);
        b.partial_x = nullptr;
        b.partial_x_bytes = 0;
        if (pool_alloc(&b.partial_x, need, st) != cudaSuccess) {
            cudaGetLastError();
            set_error("pair-sum workspace of %zu bytes: allocation failed", need);
            return GNK_ENOMEM;
        }
        b.partial_x_bytes = need;
    }
    *partial = b.partial_x;
    return GNK_OK;
}

// The plan of one launch: the handle's plan, or, under a source-chunk override
// (gnk_options.tile_chunks), that many chunks (at most one per source tile)
// with a partial-sum workspace large enough for them.
static int launch_plan(const Boundary& b, const PairPlan& base, size_t elem_bytes, PairPlan* p,
                       void** partial, cudaStream_t st) {
    *p = base;
    *partial = b.partial;
    if (b.tile_chunks <= 0) return GNK_OK;
    const int want = std::min(b.tile_chunks, p->tiles_src);
    p->tiles_per_chunk = (p->tiles_src + want - 1) / want;
    p->chunks = (p->tiles_src + p->tiles_per_chunk - 1) / p->tiles_per_chunk;
    return partial_workspace(b, (size_t)p->chunks * kMaxRHS * b.N * elem_bytes, partial, st);
}

// The workspace of the kernels that take each pair once: the handle's own where it
// is large enough, else a block of the pool for the length of the product, given back
// in the order of the stream (the sums are nt x N, up to 1 GB a right-hand side: a
// program that keeps many handles must not keep one for each).  None where the
// ordered kernel, which needs far less, is to serve the call: no memory for it, or a
// capturing stream and more than the handle's own holds.
struct SymSpace {
    void* p = nullptr;
    cudaStream_t st = nullptr;
    bool lent = false;
    SymSpace() = default;
    SymSpace(const SymSpace&) = delete;
    ~SymSpace() {
        if (lent) pool_free(p, st);
    }
};

static int sym_workspace(const Boundary& b, size_t need, SymSpace* s, cudaStream_t st) {
    if (need <= b.partial_bytes) {
        s->p = b.partial;
        return GNK_OK;
    }
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    GNK_TRY_CUDA(cudaStreamIsCapturing(st, &cs));
    if (cs != cudaStreamCaptureStatusNone) return GNK_OK;
    s->st = st;
    s->lent = pool_alloc(&s->p, need, st) == cudaSuccess;
    if (!s->lent) {
        cudaGetLastError();
        s->p = nullptr;
    }
    return GNK_OK;
}

template <int R, int MODE, int COMP, int W>
static cudaError_t launch_sym64(const Pair64SymArgs& a, cudaStream_t st) {
    constexpr int NT = 32 * W;
    const int SB = NT * a.G;
    const size_t smem = (size_t)NT * (1 + R) * sizeof(double2) + (size_t)R * (COMP == 0 ? 2 : 1) * SB * sizeof(double);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(pairsum64_sym_kernel<R, MODE, COMP, W>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    pairsum64_sym_kernel<R, MODE, COMP, W><<<a.nt * (a.nt + 1) / 2, NT, smem, st>>>(a);
    return cudaGetLastError();
}

template <int R, int MODE, int COMP>
static cudaError_t launch_sym64_w(int W, int sms, const Pair64SymArgs& a, const ReduceArgs& ra, cudaStream_t st) {
    switch (W) {
        case 1:
            if (a.nt * (a.nt + 1) / 2 >= kSymFastBlocks * sms)
                pairsum64_sym32_kernel<R, MODE, COMP, true><<<a.nt * (a.nt + 1) / 2, 32 * kSymSplit, 0, st>>>(a, ra);
            else
                pairsum64_sym32_kernel<R, MODE, COMP, false><<<a.nt * (a.nt + 1) / 2, 32 * kSymSplit, 0, st>>>(a, ra);
            return cudaGetLastError();
        case 2: return launch_sym64<R, MODE, COMP, 2>(a, st);
        case 4: return launch_sym64<R, MODE, COMP, 4>(a, st);
        default: return launch_sym64<R, MODE, COMP, 8>(a, st);
    }
}

// Whether the result of a job lies over one of its inputs.  The 32-node kernel writes
// results while other blocks still read the inputs, so such a product goes through the
// handle's scratch (the other kernels write their results in a launch of its own).
static bool in_place(const PairJob& job, int N) {
    const bool z = job.epi == EPI_Z;
    const char* out = z ? reinterpret_cast<const char*>(job.out_c) : reinterpret_cast<const char*>(job.out);
    const size_t nout = (size_t)N * (z ? job.R * sizeof(double2) : sizeof(double));
    for (int r = 0; r < job.R; ++r) {
        const char* in = job.mode == W_COMPLEX ? reinterpret_cast<const char*>(job.w[r])
                                               : reinterpret_cast<const char*>(job.x[r]);
        const size_t nin = (size_t)N * (job.mode == W_COMPLEX ? sizeof(double2) : sizeof(double));
        if (in < out + nout && out < in + nin) return true;
    }
    return false;
}

// The FP64 sum with each pair taken once.  *ran = false where the ordered kernel
// serves the call: a source-chunk override, more than 524,288 nodes, no memory for
// the partial sums, or a capturing stream (sym_workspace).
static int run_pairsum64_sym(const Boundary& b, const PairJob& job, cudaStream_t st, bool* ran) {
    *ran = false;
    const SymPlan& p = b.sym64;
    if (p.W == 0 || b.tile_chunks > 0) return GNK_OK;
    if (p.W == 1 && in_place(job, b.N)) {
        PairJob via = job;
        const bool z = job.epi == EPI_Z;
        if (z)
            via.out_c = b.zbuf;
        else
            via.out = reinterpret_cast<double*>(b.zbuf);
        GNK_TRY(run_pairsum64_sym(b, via, st, ran));
        if (*ran)
            GNK_TRY_CUDA(cudaMemcpyAsync(z ? (void*)job.out_c : (void*)job.out, b.zbuf,
                                         (size_t)b.N * (z ? job.R * sizeof(double2) : sizeof(double)),
                                         cudaMemcpyDeviceToDevice, st));
        return GNK_OK;
    }
    SymSpace space;
    GNK_TRY(sym_workspace(b, (size_t)p.nt * job.R * b.N * sizeof(double2), &space, st));
    if (!space.p) return GNK_OK;
    Pair64SymArgs a;
    a.et = b.et;
    a.N = b.N;
    a.w0 = job.w[0];
    a.w1 = job.w[1];
    a.x0 = job.x[0];
    a.x1 = job.x[1];
    a.s = job.s;
    a.partial = static_cast<double2*>(space.p);
    a.nt = p.nt;
    a.G = p.G;
    a.count = b.sym_count;
    a.done = job.done;
    ReduceArgs ra = reduce_args(b, job, p.nt, 0);
    const ProfToken tok = prof_begin(st);
    cudaError_t e;
    if (job.R == 1 && job.mode == W_SCALED && job.comp == 1)
        e = launch_sym64_w<1, W_SCALED, 1>(p.W, b.sms, a, ra, st);
    else if (job.R == 1 && job.mode == W_SCALED && job.comp == 2)
        e = launch_sym64_w<1, W_SCALED, 2>(p.W, b.sms, a, ra, st);
    else if (job.R == 1 && job.mode == W_SCALED)
        e = launch_sym64_w<1, W_SCALED, 0>(p.W, b.sms, a, ra, st);
    else if (job.R == 1)
        e = launch_sym64_w<1, W_COMPLEX, 0>(p.W, b.sms, a, ra, st);
    else if (job.mode == W_SCALED)
        e = launch_sym64_w<2, W_SCALED, 0>(p.W, b.sms, a, ra, st);
    else
        e = launch_sym64_w<2, W_COMPLEX, 0>(p.W, b.sms, a, ra, st);
    GNK_TRY_CUDA(e);
    // FP64 pipe per unordered pair: 2 (d; few blocks: 9) and per right-hand side
    // and direction 4 (one part of z: 2)
    const bool fast = p.W > 1 || p.nt * (p.nt + 1) / 2 >= kSymFastBlocks * b.sms;
    const double per_pair = (fast ? 2.0 : 9.0) + ((job.comp && job.R == 1) ? 4.0 : 8.0 * job.R);
    prof_end(tok, PK_PAIR64, (double)job.R * b.N * (b.N - 1.0), st, 0.5 * per_pair * b.N * (b.N - 1.0));
    if (p.W > 1) GNK_TRY_CUDA(launch_reduce(b, job, p.nt, 0, st, space.p));  // else done by the kernel
    count_launches(p.W > 1 ? 2 : 1);
    *ran = true;
    return GNK_OK;
}

int run_pairsum64(const Boundary& b, const PairJob& job, cudaStream_t st) {
    bool ran = false;
    GNK_TRY(run_pairsum64_sym(b, job, st, &ran));
    if (ran) return GNK_OK;
    PairPlan p;
    void* partial = nullptr;
    GNK_TRY(launch_plan(b, b.plan64, sizeof(double2), &p, &partial, st));
    Pair64Args a;
    a.et = b.et;
    a.N = b.N;
    a.w0 = job.w[0];
    a.w1 = job.w[1];
    a.x0 = job.x[0];
    a.x1 = job.x[1];
    a.s = job.s;
    a.partial = static_cast<double2*>(partial);
    a.tiles_src = p.tiles_src;
    a.tiles_per_chunk = p.tiles_per_chunk;
    a.done = job.done;
    dim3 grid(p.tiles_tgt, p.chunks);
    const ProfToken tok = prof_begin(st);
    if (job.R == 1 && job.mode == W_SCALED)
        pairsum64_kernel<1, W_SCALED><<<grid, kThreads64, 0, st>>>(a);
    else if (job.R == 1)
        pairsum64_kernel<1, W_COMPLEX><<<grid, kThreads64, 0, st>>>(a);
    else if (job.mode == W_SCALED)
        pairsum64_kernel<2, W_SCALED><<<grid, kThreads64, 0, st>>>(a);
    else
        pairsum64_kernel<2, W_COMPLEX><<<grid, kThreads64, 0, st>>>(a);
    GNK_TRY_CUDA(cudaGetLastError());
    // FP64 pipe per pair: 9 shared (d, |d|^2, reciprocal, 1/d) + 4 per right-hand side
    prof_end(tok, PK_PAIR64, (double)job.R * b.N * (b.N - 1.0), st,
             (9.0 + 4.0 * job.R) * b.N * (b.N - 1.0));
    GNK_TRY_CUDA(launch_reduce(b, job, p.chunks, 0, st, partial));
    count_launches(2);
    return GNK_OK;
}

constexpr int kSymMaxTiles = 256;  // N <= 65,536: 268 MB of double-float sums a right-hand side

// The FP32 sum with each pair taken once; *ran as for the double-float sum.
static int run_pairsum32_sym(const Boundary& b, const PairJob& job, cudaStream_t st, bool* ran) {
    *ran = false;
    const int nt = (b.N + kSrcTile32 - 1) / kSrcTile32, pairs = nt * (nt + 1) / 2;
    if (b.tile_chunks > 0 || b.f32_scalar || nt > kSymMaxTiles) return GNK_OK;
    if (job.mode == W_SCALED && job.s != b.q && job.s != b.A) return GNK_OK;  // refused by the caller
    SymSpace space;
    GNK_TRY(sym_workspace(b, (size_t)nt * job.R * b.N * sizeof(float2), &space, st));
    if (!space.p) return GNK_OK;
    Pair32Args a;
    a.et32 = b.et32;
    a.ref32 = b.ref32;
    a.off32 = b.off32;
    a.N = b.N;
    a.w0 = job.w[0];
    a.w1 = job.w[1];
    a.x0 = job.x[0];
    a.x1 = job.x[1];
    a.s32 = (job.s == b.q) ? b.q32 : b.A32;
    a.partial = static_cast<float2*>(space.p);
    a.tiles_src = nt;
    a.tiles_per_chunk = 1;
    a.done = job.done;
    const ProfToken tok = prof_begin(st);
    constexpr int NT = 32 * kSym32Warps;
    if (job.R == 1 && job.mode == W_SCALED && job.comp == 1)
        pairsum32_sym_kernel<1, W_SCALED, 1><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.R == 1 && job.mode == W_SCALED && job.comp == 2)
        pairsum32_sym_kernel<1, W_SCALED, 2><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.R == 1 && job.mode == W_SCALED)
        pairsum32_sym_kernel<1, W_SCALED, 0><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.R == 1)
        pairsum32_sym_kernel<1, W_COMPLEX, 0><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.mode == W_SCALED)
        pairsum32_sym_kernel<2, W_SCALED, 0><<<pairs, NT, 0, st>>>(a, nt);
    else
        pairsum32_sym_kernel<2, W_COMPLEX, 0><<<pairs, NT, 0, st>>>(a, nt);
    GNK_TRY_CUDA(cudaGetLastError());
    // FP32 pipe per unordered pair: 4 (|d|^2), then per direction 2 and 4 per
    // right-hand side (one part of z: 3)
    const double per_pair = 4.0 + ((job.comp && job.R == 1) ? 6.0 : 4.0 + 8.0 * job.R);
    prof_end(tok, PK_PAIR32, (double)job.R * b.N * (b.N - 1.0), st, 0.5 * per_pair * b.N * (b.N - 1.0));
    GNK_TRY_CUDA(launch_reduce(b, job, nt, 1, st, space.p));
    count_launches(2);
    *ran = true;
    return GNK_OK;
}

int run_pairsum32(const Boundary& b, const PairJob& job, cudaStream_t st) {
    bool ran = false;
    GNK_TRY(run_pairsum32_sym(b, job, st, &ran));
    if (ran) return GNK_OK;
    PairPlan p;
    void* partial = nullptr;
    GNK_TRY(launch_plan(b, b.plan32, sizeof(float2), &p, &partial, st));
    Pair32Args a;
    a.et32 = b.et32;
    a.ref32 = b.ref32;
    a.off32 = b.off32;
    a.N = b.N;
    a.w0 = job.w[0];
    a.w1 = job.w[1];
    a.x0 = job.x[0];
    a.x1 = job.x[1];
    a.s32 = (job.s == b.q) ? b.q32 : b.A32;
    a.partial = static_cast<float2*>(partial);
    a.tiles_src = p.tiles_src;
    a.tiles_per_chunk = p.tiles_per_chunk;
    a.done = job.done;
    if (job.mode == W_SCALED && job.s != b.q && job.s != b.A) {
        set_error("FP32 pair sum: the scale must be q or A of the handle");
        return GNK_EINVAL;
    }
    dim3 grid(p.tiles_tgt, p.chunks);
    const ProfToken tok = prof_begin(st);
    const int comp = b.f32_scalar ? 0 : job.comp;
    if (!b.f32_scalar) {
        if (job.R == 1 && job.mode == W_SCALED && comp == 1)
            pairsum32x2_kernel<1, W_SCALED, 1><<<grid, kThreads32, 0, st>>>(a);
        else if (job.R == 1 && job.mode == W_SCALED && comp == 2)
            pairsum32x2_kernel<1, W_SCALED, 2><<<grid, kThreads32, 0, st>>>(a);
        else if (job.R == 1 && job.mode == W_SCALED)
            pairsum32x2_kernel<1, W_SCALED, 0><<<grid, kThreads32, 0, st>>>(a);
        else if (job.R == 1)
            pairsum32x2_kernel<1, W_COMPLEX, 0><<<grid, kThreads32, 0, st>>>(a);
        else if (job.mode == W_SCALED)
            pairsum32x2_kernel<2, W_SCALED, 0><<<grid, kThreads32, 0, st>>>(a);
        else
            pairsum32x2_kernel<2, W_COMPLEX, 0><<<grid, kThreads32, 0, st>>>(a);
    } else if (job.R == 1 && job.mode == W_SCALED)
        pairsum32_kernel<1, W_SCALED><<<grid, kThreads32, 0, st>>>(a);
    else if (job.R == 1)
        pairsum32_kernel<1, W_COMPLEX><<<grid, kThreads32, 0, st>>>(a);
    else if (job.mode == W_SCALED)
        pairsum32_kernel<2, W_SCALED><<<grid, kThreads32, 0, st>>>(a);
    else
        pairsum32_kernel<2, W_COMPLEX><<<grid, kThreads32, 0, st>>>(a);
    GNK_TRY_CUDA(cudaGetLastError());
    // FP32 pipe per pair (plus one MUFU reciprocal): 6 shared + 4 per right-hand
    // side; one part of z only: 4 shared + 3 per right-hand side
    const double per_pair = (comp && job.R == 1) ? 4.0 + 3.0 : 6.0 + 4.0 * job.R;
    prof_end(tok, PK_PAIR32, (double)job.R * b.N * (b.N - 1.0), st, per_pair * b.N * (b.N - 1.0));
    GNK_TRY_CUDA(launch_reduce(b, job, p.chunks, 1, st, partial));
    count_launches(2);
    return GNK_OK;
}

// The double-float sum with each pair taken once; not faster at any size with the
// ordered kernel (I - N, real A: N = 512 to 4,096 48-50 against 54-56 us, the time of
// one block's 256 steps; 6,144 78 against 101; 16,384 447 against 694; 32,768 1,671
// against 2,348).  *ran = false where that one serves the call all the same: a
// source-chunk override, the scalar variant, partial sums (nt x N) past kSymMaxTiles
// node blocks, no memory for them, or a capturing stream (sym_workspace).

static int run_pairsumdf_sym(const Boundary& b, const PairJob& job, cudaStream_t st, bool* ran) {
    *ran = false;
    const int nt = (b.N + kSrcTile32 - 1) / kSrcTile32, pairs = nt * (nt + 1) / 2;
    if (b.tile_chunks > 0 || b.df_scalar || nt > kSymMaxTiles) return GNK_OK;
    SymSpace space;
    GNK_TRY(sym_workspace(b, (size_t)nt * job.R * b.N * sizeof(float4), &space, st));
    if (!space.p) return GNK_OK;
    PairDFArgs a;
    a.et = b.et;
    a.ref64 = b.ref64;
    a.offdf = b.offdf;
    a.N = b.N;
    a.w0 = job.w[0];
    a.w1 = job.w[1];
    a.x0 = job.x[0];
    a.x1 = job.x[1];
    a.s = job.s;
    a.partial = static_cast<float4*>(space.p);
    a.tiles_src = nt;
    a.tiles_per_chunk = 1;
    a.done = job.done;
    const ProfToken tok = prof_begin(st);
    constexpr int NT = 32 * kSymDFWarps;
    if (job.R == 1 && job.mode == W_SCALED && job.comp == 1)
        pairsumdf_sym_kernel<1, W_SCALED, 1><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.R == 1 && job.mode == W_SCALED && job.comp == 2)
        pairsumdf_sym_kernel<1, W_SCALED, 2><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.R == 1 && job.mode == W_SCALED)
        pairsumdf_sym_kernel<1, W_SCALED, 0><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.R == 1)
        pairsumdf_sym_kernel<1, W_COMPLEX, 0><<<pairs, NT, 0, st>>>(a, nt);
    else if (job.mode == W_SCALED)
        pairsumdf_sym_kernel<2, W_SCALED, 0><<<pairs, NT, 0, st>>>(a, nt);
    else
        pairsumdf_sym_kernel<2, W_COMPLEX, 0><<<pairs, NT, 0, st>>>(a, nt);
    GNK_TRY_CUDA(cudaGetLastError());
    // FP32 pipe per unordered pair: 49 (1/d) and per right-hand side and direction
    // 48 (one part of z: 24)
    const double per_pair = 49.0 + ((job.comp && job.R == 1) ? 48.0 : 96.0 * job.R);
    prof_end(tok, PK_PAIRDF, (double)job.R * b.N * (b.N - 1.0), st, 0.5 * per_pair * b.N * (b.N - 1.0));
    GNK_TRY_CUDA(launch_reduce(b, job, nt, 2, st, space.p));
    count_launches(2);
    *ran = true;
    return GNK_OK;
}

int run_pairsumdf(const Boundary& b, const PairJob& job, cudaStream_t st) {
    bool ran = false;
    GNK_TRY(run_pairsumdf_sym(b, job, st, &ran));
    if (ran) return GNK_OK;
    PairPlan p;
    void* partial = nullptr;
    GNK_TRY(launch_plan(b, b.plandf, sizeof(float4), &p, &partial, st));
    PairDFArgs a;
    a.et = b.et;
    a.ref64 = b.ref64;
    a.offdf = b.offdf;
    a.N = b.N;
    a.w0 = job.w[0];
    a.w1 = job.w[1];
    a.x0 = job.x[0];
    a.x1 = job.x[1];
    a.s = job.s;
    a.partial = static_cast<float4*>(partial);
    a.tiles_src = p.tiles_src;
    a.tiles_per_chunk = p.tiles_per_chunk;
    a.done = job.done;
    dim3 grid(p.tiles_tgt, p.chunks);
    const ProfToken tok = prof_begin(st);
    const int comp = b.df_scalar ? 0 : job.comp;
    if (!b.df_scalar) {
        if (job.R == 1 && job.mode == W_SCALED && comp == 1)
            pairsumdf2_kernel<1, W_SCALED, 1><<<grid, kThreadsDF, 0, st>>>(a);
        else if (job.R == 1 && job.mode == W_SCALED && comp == 2)
            pairsumdf2_kernel<1, W_SCALED, 2><<<grid, kThreadsDF, 0, st>>>(a);
        else if (job.R == 1 && job.mode == W_SCALED)
            pairsumdf2_kernel<1, W_SCALED, 0><<<grid, kThreadsDF, 0, st>>>(a);
        else if (job.R == 1)
            pairsumdf2_kernel<1, W_COMPLEX, 0><<<grid, kThreadsDF, 0, st>>>(a);
        else if (job.mode == W_SCALED)
            pairsumdf2_kernel<2, W_SCALED, 0><<<grid, kThreadsDF, 0, st>>>(a);
        else
            pairsumdf2_kernel<2, W_COMPLEX, 0><<<grid, kThreadsDF, 0, st>>>(a);
    } else if (job.R == 1 && job.mode == W_SCALED)
        pairsumdf_kernel<1, W_SCALED><<<grid, kThreadsDF, 0, st>>>(a);
    else if (job.R == 1)
        pairsumdf_kernel<1, W_COMPLEX><<<grid, kThreadsDF, 0, st>>>(a);
    else if (job.mode == W_SCALED)
        pairsumdf_kernel<2, W_SCALED><<<grid, kThreadsDF, 0, st>>>(a);
    else
        pairsumdf_kernel<2, W_COMPLEX><<<grid, kThreadsDF, 0, st>>>(a);
    GNK_TRY_CUDA(cudaGetLastError());
    // FP32 pipe per pair: 49 shared (d, |d|^2, reciprocal, 1/d) + 48 per right-hand
    // side (two products and two compensated sums per part of z)
    const double per_pair = (comp && job.R == 1) ? 49.0 + 24.0 : 49.0 + 48.0 * job.R;
    prof_end(tok, PK_PAIRDF, (double)job.R * b.N * (b.N - 1.0), st, per_pair * b.N * (b.N - 1.0));
    GNK_TRY_CUDA(launch_reduce(b, job, p.chunks, 2, st, partial));
    count_launches(2);
    return GNK_OK;
}

int pair_blocks_per_sm(int precision) {
    int nb = 1;
    cudaError_t e;
    if (precision == GNK_PREC_FP32)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pairsum32_kernel<2, W_SCALED>, kThreads32, 0);
    else if (precision == GNK_PREC_DF32)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pairsumdf_kernel<2, W_SCALED>, kThreadsDF, 0);
    else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pairsum64_kernel<2, W_SCALED>, kThreads64, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return nb < 1 ? 1 : nb;
}

// The part of z = E(q x) an epilogue reads: f_B reads Im(A z) and f_C reads
// Re(A z), which with Im A = 0 are A Im z and A Re z.
int pair_component_needed(const Boundary& b, const PairJob& job) {
    if (!b.A_real || job.R != 1 || job.mode != W_SCALED || job.s != b.q) return 0;
    if (job.epi == EPI_IMINUSN || job.epi == EPI_RESID) return 1;
    if (job.epi == EPI_M) return 2;
    return 0;
}

int run_pairsum(const Boundary& b, const PairJob& job, int precision, cudaStream_t st) {
    if (precision == GNK_PREC_FMM) return run_fmm(b, job, st);
    GNK_TRY(run_job_sides(b, job, st));
    PairJob j = job;
    j.comp = pair_component_needed(b, job);
    if (precision == GNK_PREC_FP32) return run_pairsum32(b, j, st);
    if (precision == GNK_PREC_DF32) return run_pairsumdf(b, j, st);
    return run_pairsum64(b, j, st);
}

}  // namespace gnk
