// Fast multipole evaluation of the Cauchy sum z_i = sum_{j != i} w_j / (eta_i - eta_j)
// (Sec. 2.5, Eqs. fmm-1, fmm-E: the paper forms E w with the FMM of zfmm2dpart,
// O((m+1)n) operations).  Uniform-depth quadtree over the bounding square of the
// nodes (levels 2 or 3..L, empty boxes pruned), expansions of order P scaled by the box
// width r (Greengard & Rokhlin's complex-analytic 2-D FMM):
//   multipole  phi(z) = sum_k a_k r^k / (z - c)^(k+1),  a_k = sum_j w_j ((s_j - c)/r)^k
//   local      phi(z) = sum_l b_l ((z - c)/r)^l
//   M2M  a0_m = sum_{k<=m} C(m,k) ((c1-c0)/r0)^(m-k) 2^-k a1_k
//   M2L  b_l  = (1/r) sum_k (-1)^(k+1) C(k+l,l) delta^-(k+l+1) a_k,  delta = (c1-c0)/r
//   L2L  b1_m = sum_{l>=m} C(l,m) ((c1-c0)/r0)^(l-m) 2^-m b0_l
// The near field (a leaf and its eight neighbours) is summed directly with the
// i = j term excluded.  The truncation error is below 0.43^P of
// sum_j |w_j / (eta_i - eta_j)| (about 2e-12 at P = 32 including round-off;
// checked against direct sums in the tests).
//
// One product is five to seven launches on two or three streams.  The far field:
// the upward pass (P2M, then the M2M chain carried by the warp that completes
// each box's last child, no launch per level), M2L for every box, L2L for four
// leaves per warp down their ancestor paths.  The near field runs beside it; where
// its geometry and factors are fixed (weights q x; in a solve also A x) it is
// streamed from an operator cache by bulk asynchronous copies, else the weights are
// gathered into tree order first and every pair is formed.  L2P adds the two after
// they join and applies the operator's epilogue.  M2M and L2L are fixed real Pascal
// matrices between exact Gaussian-integer scalings, M2L a fixed real Pascal
// matrix between two complex scalings per offset: no P x P table per relative
// position.  The fixed matrices multiply on the tensor cores (digits exact in
// FP16), everything else runs in complex double-float on the FP32 pipe (GB300's
// FP64 pipe is 1/64 of it).  A handle built for differentiation (GNK_BUILD_DIFF)
// keeps one fixed sequence of operations, the double-float translations.
//
// The tree is built once per handle (the geometry is fixed for all products),
// on the device when its lookup grids fit (fmm_tree.cu), else on the host:
// Morton keys of 16-bit box coordinates, a sort of (key, node) pairs, leaf
// level L = the deepest level whose non-empty boxes hold enough
// nodes on average, interaction and neighbour lists.  Every sum on the device
// runs in a fixed order, so results are reproducible.
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <complex>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <vector>

#include "fmm_internal.h"
#include "tma.cuh"
#include "epilogue.cuh"
#include "gnk_internal.h"
#include "pairmath.cuh"

namespace gnk {

namespace {

struct FmmArgs {
    int N, R, P;
    const int* perm;
    const double2* ps;
    const float4* p3;
    const float2* p3b;
    const int* leaf_start;
    const int* leaf_box;
    const double2* center;
    const double* width;
    const int* child_start;
    const int* child_count;
    const int* parent;
    const int* quad;
    const int* il_start;
    const int* il_src;
    const int* il_off;
    const int* nl_start;
    const int* nl_leaf;
    const float2* m2lH;   // C(k+l, l), [k][l] double-float
    const float4* m2lS;   // per offset code: (-1)^(k+1) delta^-(k+1), then delta^-l
    const float2* bUp;    // C(l, m) at [l][m] (0 for l < m): the L2L Pascal sums
    const float4* m2lT;   // per offset code: (-1)^(k+1) (2/delta)^k / delta, then (2/delta)^l
    const uint4* m2lA;    // digits of C(k+l, l) 2^-(k+l) as mma fragments,
    const uint4* upA;     // of C(m, k) 2^-m (M2M)
    const uint4* dnA;     // and of C(l, m) 2^-l (L2L)
    const unsigned* path; // [nleaf][depth]: box | quadrant << 30 of each leaf and its ancestors
    int depth;            // levels of the tree: L - l0 + 1
    int nleaf;
    float4* mult;
    float4* loc;
    float4* ws;
    int nbox;
    // weights
    int mode;
    const double2* w0;
    const double2* w1;
    const double* x0;
    const double* x1;
    const double2* s;
    double2* out;  // [R][N] in node order
    const int* done;
    const int2* items;  // near-field work items: (leaf, first target of a chunk of 32)
    int nitems;
    double2* zn;        // [R][N] near-field sums in sorted order
    double2* zf;        // [R][N] near-field sums of w/d^2 in sorted order (EF products)
    double2* outF;      // [R][N] F sums in node order (EF products)
    const int* node_box;  // leaf box of each node in sorted order
    int* ucnt;            // per box: children counted in the upward pass
    const long long* inv_off;  // inverse cache: first entry of each item,
    float4* inv_r;        // and 1/d = ar - i ai of every near pair (two sources an entry)
    float4* inv_i;
    int use_inv;          // the direct near field (R = 1) reads it
    int nsplit;           // shares of the near field, [share][R][N] in zn
    int gathered;         // ws holds the weights in sorted order (products with a direct near field)
    int near_scaled;      // zn holds the near field times the operator's factor (cached)
    const float4* tn;     // [N] offset t of every node from its leaf centre in leaf widths (double-float complex)
    int diff;             // a handle built for differentiation
    int* fault;           // set by a bounded wait that gave up
};

// The weight of right-hand side r at node j, double-float complex.
__device__ __forceinline__ float4 fmm_weight(const FmmArgs& a, int r, int j) {
    double2 w;
    if (a.mode == W_COMPLEX) {
        w = (r == 0) ? a.w0[j] : a.w1[j];
    } else {
        const double2 sc = a.s[j];
        const double x = (r == 0) ? a.x0[j] : a.x1[j];
        w = make_double2(sc.x * x, sc.y * x);
    }
    const df wx = df_split_fast(w.x), wy = df_split_fast(w.y);
    return make_float4(wx.h, wx.l, wy.h, wy.l);
}

// The weights in sorted order, for the products whose near field is summed
// directly (every leaf's sources are read by its neighbours); with a cached near
// field P2M is their only reader and forms them itself.
__global__ void fmm_gather_kernel(FmmArgs a) {
    if (a.done != nullptr && *a.done) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.N) return;
    const int j = a.perm[i];
    for (int r = 0; r < a.R; ++r) a.ws[(size_t)r * a.N + i] = fmm_weight(a, r, j);
}

// ---- complex double-float arithmetic for the far field (FP32 pipe).  The
// expansions and the M2L scalings are stored as float4 (re.h, re.l, im.h,
// im.l); sums keep their rounding errors in the low words (about 2^-46 relative
// per operation), far below the truncation error of the order-32 expansions.
struct cdf {
    df re, im;
};

__device__ __forceinline__ cdf cdf_of(float4 v) { return cdf{df{v.x, v.y}, df{v.z, v.w}}; }
__device__ __forceinline__ float4 cdf_pack(cdf c) { return make_float4(c.re.h, c.re.l, c.im.h, c.im.l); }
__device__ __forceinline__ cdf cdf_zero() { return cdf{df{0.f, 0.f}, df{0.f, 0.f}}; }
__device__ __forceinline__ cdf cdf_split(double2 v) { return cdf{df_split(v.x), df_split(v.y)}; }
__device__ __forceinline__ df df_neg(df a) { return df{-a.h, -a.l}; }

// a + b, renormalised
__device__ __forceinline__ df df_add(df a, df b) {
    float s, e;
    two_sum(a.h, b.h, s, e);
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    df r;
    fast_two_sum(s, e, r.h, r.l);
    return r;
}

__device__ __forceinline__ cdf cdf_mul(cdf a, cdf b) {
    return cdf{df_add(df_mul(a.re, b.re), df_neg(df_mul(a.im, b.im))),
               df_add(df_mul(a.re, b.im), df_mul(a.im, b.re))};
}

// acc += a b
__device__ __forceinline__ void cdf_mac(cdf& acc, cdf a, cdf b) {
    df_acc(acc.re, df_mul(a.re, b.re));
    df_acc(acc.re, df_neg(df_mul(a.im, b.im)));
    df_acc(acc.im, df_mul(a.re, b.im));
    df_acc(acc.im, df_mul(a.im, b.re));
}

__device__ __forceinline__ cdf cdf_add(cdf a, cdf b) { return cdf{df_add(a.re, b.re), df_add(a.im, b.im)}; }

__device__ __forceinline__ df2 df2_neg(df2 a) { return df2{neg2(a.h), neg2(a.l)}; }

// a + b (renormalised), two lanes
__device__ __forceinline__ df2 df2_add(df2 a, df2 b) {
    float2 s, e;
    two_sum2(a.h, b.h, s, e);
    e = add2(e, add2(a.l, b.l));
    df2 r;
    r.h = add2(s, e);
    r.l = sub2(e, sub2(r.h, s));
    return r;
}

// Translation kernels use kFmmTW warps per target box.
constexpr int kFmmTW = 4;
constexpr int kFmmMaxDepth = 24;  // ancestors of a leaf, the leaf included

// ---- M2M and L2L between exact scalings.  With delta =
// (c1 - c0)/r0 = g/4 for a child in quadrant q, g = (2 qa - 1) + i (2 qb - 1):
//   M2M  a0_m = delta^m sum_{k<=m} C(m,k) [(2 delta)^-k a1_k]
//   L2L  b1_m = (2 delta)^-m sum_{l>=m} C(l,m) [delta^l b0_l]
// and (2 delta)^-1 = conj(g).  The scale factors g^e 4^-e and conj(g)^e are
// Gaussian integers times powers of two, so multiplying by them is exact up
// to one rounding in each part.  The L2L Pascal sum is a product with the
// fixed real triangular matrix C(l,m) (a double-float table of 8 KB that stays
// in L1; C(l,m) < 2^29, exact), lane m accumulating its 32 terms (zero beyond
// the triangle) in two independent compensated sums: one transform has the
// latency of a 32-term dot product instead of 31 dependent passes.  The M2M
// sum takes the passes (binom_lower).
constexpr int kFmmUT = 32 * kFmmTW;  // threads of the upward and downward kernels

// angle of g in units of pi/4 for the quadrant q = 2 qa + qb
__device__ __forceinline__ int gauss_angle(int q) { return (q == 3) ? 1 : (q == 1) ? 3 : (q == 0) ? 5 : 7; }

// x g^e 2^s for g = sqrt(2) e^{i pi ang / 4} (ang odd): g^e = 2^floor(e/2) (c + i d), c, d in {0, +-1}
__device__ __forceinline__ cdf cdf_mul_gpow(cdf x, int ang, int e, int s) {
    const int a8 = (ang * e) & 7;
    const float m = ldexpf(1.f, (e >> 1) + s);
    const float gr = (a8 == 0 || a8 == 1 || a8 == 7) ? m : ((a8 >= 3 && a8 <= 5) ? -m : 0.f);
    const float gi = (a8 >= 1 && a8 <= 3) ? m : ((a8 >= 5) ? -m : 0.f);
    const df p{__fmul_rn(x.re.h, gr), __fmul_rn(x.re.l, gr)}, q{__fmul_rn(-x.im.h, gi), __fmul_rn(-x.im.l, gi)};
    const df u{__fmul_rn(x.im.h, gr), __fmul_rn(x.im.l, gr)}, v{__fmul_rn(x.re.h, gi), __fmul_rn(x.re.l, gi)};
    return cdf{df_add(p, q), df_add(u, v)};
}

__device__ __forceinline__ cdf cdf_shfl_up1(cdf v) {
    return cdf{df{__shfl_up_sync(0xffffffffu, v.re.h, 1), __shfl_up_sync(0xffffffffu, v.re.l, 1)},
               df{__shfl_up_sync(0xffffffffu, v.im.h, 1), __shfl_up_sync(0xffffffffu, v.im.l, 1)}};
}

// lane m: sum_{k<=m} C(m,k) v_k by P - 1 passes (pass i adds the left
// neighbour's pre-pass value on lanes m >= i).  The upward pass keeps this
// form: there the Pascal-table sum below measured slower (more loads while
// the P2M of other leaves competes for the SM).
__device__ __forceinline__ cdf binom_lower(cdf v, int lane) {
#pragma unroll 1
    for (int i = 1; i < kFmmP; ++i) {
        const cdf u = cdf_shfl_up1(v);
        if (lane >= i) v = cdf_add(v, u);
    }
    return v;
}

// lane m: sum_k T[k][m] v_k for a real double-float table T (P x P, [k][m])
// and the complex vector v staged by the warp in sv[0 .. P)
__device__ __forceinline__ cdf pascal_sum(const float2* __restrict__ T, const float4* sv, int lane) {
    df yr{0.f, 0.f}, yi{0.f, 0.f}, zr{0.f, 0.f}, zi{0.f, 0.f};
#pragma unroll 4
    for (int k = 0; k < kFmmP; k += 2) {
        const float2 h0 = __ldg(T + k * kFmmP + lane), h1 = __ldg(T + (k + 1) * kFmmP + lane);
        const float4 x0 = sv[k], x1 = sv[k + 1];
        df_acc(yr, df_mul(df{h0.x, h0.y}, df{x0.x, x0.y}));
        df_acc(yi, df_mul(df{h0.x, h0.y}, df{x0.z, x0.w}));
        df_acc(zr, df_mul(df{h1.x, h1.y}, df{x1.x, x1.y}));
        df_acc(zi, df_mul(df{h1.x, h1.y}, df{x1.z, x1.w}));
    }
    return cdf{df_add(yr, zr), df_add(yi, zi)};
}

// one warp: lane m of a1 (the child's multipole) -> lane m of its contribution
// to the parent's multipole
__device__ __forceinline__ cdf m2m_binom(cdf a1, int q, int lane) {
    const int ang = gauss_angle(q);
    const cdf c = cdf_mul_gpow(a1, 8 - ang, lane, 0);  // (2 delta)^-k a1_k
    return cdf_mul_gpow(binom_lower(c, lane), ang, lane, -2 * lane);  // delta^m S_m
}

__device__ __forceinline__ cdf l2l_pascal(cdf b0, int q, int lane, const float2* bUp, float4* sv) {
    const int ang = gauss_angle(q);
    const cdf e = cdf_mul_gpow(b0, ang, lane, -2 * lane);  // delta^l b0_l
    __syncwarp();
    sv[lane] = cdf_pack(e);
    __syncwarp();
    return cdf_mul_gpow(pascal_sum(bUp, sv, lane), 8 - ang, lane, 0);  // (2 delta)^-m T_m
}

__device__ __forceinline__ cdf reduce_warps(cdf acc, float4 (*s)[32], int wid, int lane) {
    s[wid][lane] = cdf_pack(acc);
    __syncthreads();
    cdf t = cdf_of(s[0][lane]);
    if (wid == 0)
        for (int w = 1; w < kFmmTW; ++w) t = cdf_add(t, cdf_of(s[w][lane]));
    __syncthreads();
    return t;  // valid in warp 0
}

__device__ __forceinline__ cdf cdf_sq(cdf a) { return cdf_mul(a, a); }

// M2L into one box, as a fixed real matrix between two diagonal scalings:
// with x_k = (-1)^(k+1) delta^-(k+1) a_k (delta the source-to-target centre
// offset in box widths),
//   b_l = (1/r) delta^-l sum_k C(k+l, l) x_k.
// The Pascal matrix C(k+l, l) (double-float, 8 KB) is the same for every
// pair and stays in L1; the scalings are 2 x 32 double-float complex values
// per offset code.  The terms are those of the matrix form, so the rounding
// error is of the same size.  Warp w takes the interaction-list entries w,
// w + kFmmTW, ...; the warps' sums are added in warp order; the 1/r factor is
// applied once at the end.  loc then holds the M2L part of the box's local
// expansion.
template <int R>
__device__ __forceinline__ void m2l_box(const FmmArgs& a, int box, int wid, int lane, float4 (*s_acc)[32],
                                        float4 (*s_x)[32]) {
    const int e0 = a.il_start[box], e1 = a.il_start[box + 1];
    const df sc = df_split(1.0 / a.width[box]);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        cdf acc = cdf_zero();
        for (int e = e0 + wid; e < e1; e += kFmmTW) {
            const float4* S = a.m2lS + (size_t)a.il_off[e] * 2 * kFmmP;
            const cdf x = cdf_mul(cdf_of(__ldcg(a.mult + ((size_t)r * a.nbox + a.il_src[e]) * kFmmP + lane)),
                                  cdf_of(__ldg(S + lane)));
            const cdf post = cdf_of(__ldg(S + kFmmP + lane));
            __syncwarp();
            s_x[wid][lane] = cdf_pack(x);
            __syncwarp();
            df yr{0.f, 0.f}, yi{0.f, 0.f}, zr{0.f, 0.f}, zi{0.f, 0.f};
#pragma unroll 4
            for (int k = 0; k < kFmmP; k += 2) {
                const float2 h0 = __ldg(a.m2lH + k * kFmmP + lane), h1 = __ldg(a.m2lH + (k + 1) * kFmmP + lane);
                const float4 x0 = s_x[wid][k], x1 = s_x[wid][k + 1];
                df_acc(yr, df_mul(df{h0.x, h0.y}, df{x0.x, x0.y}));
                df_acc(yi, df_mul(df{h0.x, h0.y}, df{x0.z, x0.w}));
                df_acc(zr, df_mul(df{h1.x, h1.y}, df{x1.x, x1.y}));
                df_acc(zi, df_mul(df{h1.x, h1.y}, df{x1.z, x1.w}));
            }
            acc = cdf_add(acc, cdf_mul(cdf{df_add(yr, zr), df_add(yi, zi)}, post));
        }
        acc = reduce_warps(acc, s_acc, wid, lane);
        if (wid == 0) a.loc[((size_t)r * a.nbox + box) * kFmmP + lane] = cdf_pack(cdf{df_mul(acc.re, sc), df_mul(acc.im, sc)});
    }
}

// Packed complex double-float: (re, im) in the lanes of a float2.
__device__ __forceinline__ df2 pc_of(float4 v) { return df2{make_float2(v.x, v.z), make_float2(v.y, v.w)}; }

__device__ __forceinline__ df2 pc_mul(df2 a, df2 b) {  // a b, renormalised
    const df2 ax{make_float2(a.h.y, a.h.x), make_float2(a.l.y, a.l.x)};
    const df2 p = df2_mul(a, df2{f2(b.h.x), f2(b.l.x)});
    const df2 q = df2_mul(ax, df2{make_float2(-b.h.y, b.h.y), make_float2(-b.l.y, b.l.y)});
    return df2_add(p, q);
}

// P2M of one leaf, a_k = sum_j w_j t_j^k: a warp takes chunks of 32 nodes (lane =
// node) and carries w t^k up four interleaved chains k = 8 c + m (c < 4) of
// eight products; every two steps the eight values of k in hand go through
// shared memory, where four lanes per k add eight nodes each.  The powers are
// formed anew for every product: 19 packed instructions a power, 2 us of the
// FP32 pipe at 65,536 nodes, where a table of them costs 512 bytes of memory
// traffic a node beside the near field's stream (the upward pass 41 us with the
// table at 65,536 nodes, 131 us at 524,288).  The warps' sums are added in warp order.
constexpr int kP2mStride = 36;  // float4 per row: conflict-free for the column reads below

template <int R>
__device__ __forceinline__ void p2m_leaf(const FmmArgs& a, int leaf, int box, int wid, int lane, float4* s_v,
                                         float4 (*s_acc)[32]) {
    const unsigned full = 0xffffffffu;
    const int j0 = a.leaf_start[leaf], j1 = a.leaf_start[leaf + 1];
    const int row = lane >> 2, grp = lane & 3;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        df2 acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = df2{f2(0.f), f2(0.f)};
        for (int base = j0 + 32 * wid; base < j1; base += 32 * kFmmTW) {
            const int j = base + lane;
            df2 t{f2(0.f), f2(0.f)}, v[4];
            v[0] = t;
            if (j < j1) {
                t = pc_of(__ldg(a.tn + j));
                v[0] = pc_of(a.gathered ? __ldcg(a.ws + (size_t)r * a.N + j) : fmm_weight(a, r, __ldg(a.perm + j)));
            }
            {
                const df2 t2 = pc_mul(t, t), t4 = pc_mul(t2, t2), t8 = pc_mul(t4, t4), t16 = pc_mul(t8, t8);
                v[1] = pc_mul(v[0], t8);
                v[2] = pc_mul(v[0], t16);
                v[3] = pc_mul(v[1], t16);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {  // m = 2 q, 2 q + 1
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        s_v[(2 * c + u) * kP2mStride + lane] = make_float4(v[c].h.x, v[c].h.y, v[c].l.x, v[c].l.y);
                        if (q < 3 || u < 1) v[c] = pc_mul(v[c], t);
                    }
                __syncwarp();
                df2 s{f2(0.f), f2(0.f)};
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 x = s_v[row * kP2mStride + i * 4 + grp];
                    df2_acc(s, df2{make_float2(x.x, x.y), make_float2(x.z, x.w)});
                }
                acc[q] = df2_add(acc[q], s);
                __syncwarp();
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {  // the four lanes of a k
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                df2 x;
                x.h = make_float2(__shfl_xor_sync(full, acc[q].h.x, o), __shfl_xor_sync(full, acc[q].h.y, o));
                x.l = make_float2(__shfl_xor_sync(full, acc[q].l.x, o), __shfl_xor_sync(full, acc[q].l.y, o));
                acc[q] = df2_add(acc[q], x);
            }
            if (grp == 0)
                s_acc[wid][8 * (row >> 1) + 2 * q + (row & 1)] =
                    make_float4(acc[q].h.x, acc[q].l.x, acc[q].h.y, acc[q].l.y);
        }
        __syncthreads();
        if (wid == 0) {
            cdf m = cdf_of(s_acc[0][lane]);
            for (int w = 1; w < kFmmTW; ++w) m = cdf_add(m, cdf_of(s_acc[w][lane]));
            a.mult[((size_t)r * a.nbox + box) * kFmmP + lane] = cdf_pack(m);
        }
        __syncthreads();
    }
}

// P2M of one leaf for the handles built for differentiation, one fixed sequence of
// operations: t^k by repeated products, and warp w's sum over the nodes j0 + w,
// j0 + w + kFmmTW, ... in this order.  Lane u forms the powers of node u of a batch of
// kPowBatch in shared memory, then lane k sums w_j t_j^k over the batch.  (A table of
// the powers, 512 bytes a node, gives the same bits and the same time to 0.4 %, 11.92
// against 11.97 ms for a gradient at N = 40,960; without it no allocation decides which
// form runs.)
constexpr int kPowBatch = 16;

template <int R>
__device__ __forceinline__ void p2m_leaf_diff(const FmmArgs& a, int leaf, int box, int wid, int lane,
                                              float4 (*s_pow)[kPowBatch + 1], float4 (*s_w)[kPowBatch],
                                              float4 (*s_acc)[32]) {
    cdf acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = cdf_zero();
    const int j0 = a.leaf_start[leaf], j1 = a.leaf_start[leaf + 1];
    for (int j = j0 + wid; j < j1; j += kFmmTW * kPowBatch) {
        const int cnt = min(kPowBatch, (j1 - j + kFmmTW - 1) / kFmmTW);
        __syncwarp();  // the last batch has been read
        if (lane < cnt) {
            const int jj = j + lane * kFmmTW;
#pragma unroll
            for (int r = 0; r < R; ++r) s_w[r][lane] = __ldcg(a.ws + (size_t)r * a.N + jj);
            const cdf t = cdf_of(__ldg(a.tn + jj));
            cdf v = cdf{df{1.f, 0.f}, df{0.f, 0.f}};
            for (int k = 0; k < kFmmP; ++k) {
                s_pow[k][lane] = cdf_pack(v);
                v = cdf_mul(v, t);
            }
        }
        __syncwarp();
#pragma unroll 4
        for (int u = 0; u < cnt; ++u) {
            const cdf pw = cdf_of(s_pow[lane][u]);
#pragma unroll
            for (int r = 0; r < R; ++r) cdf_mac(acc[r], cdf_of(s_w[r][u]), pw);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const cdf sm = reduce_warps(acc[r], s_acc, wid, lane);
        if (wid == 0) a.mult[((size_t)r * a.nbox + box) * kFmmP + lane] = cdf_pack(sm);
    }
}

// Upward pass of the handles built for differentiation, one block per leaf: P2M,
// then the multipoles move up the tree without a launch per level: the block that
// completes the last child of a box (an atomic count per box; nothing waits)
// forms that box's M2M from its children (warp w takes child w) and goes on
// to the parent.
template <int R>
__global__ void __launch_bounds__(kFmmUT) fmm_up_kernel(FmmArgs a) {
    __shared__ float4 s_pow[kFmmTW][kFmmP][kPowBatch + 1];
    __shared__ float4 s_w[kFmmTW][R][kPowBatch];
    __shared__ float4 s_acc[kFmmTW][32];
    __shared__ int s_last;
    if (a.done != nullptr && *a.done) return;
    const int leaf = blockIdx.x, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int box = a.leaf_box[leaf];
    p2m_leaf_diff<R>(a, leaf, box, wid, lane, s_pow[wid], s_w[wid], s_acc);
    for (;;) {
        if (wid == 0) __threadfence();  // the box's multipole (warp 0's stores) before the count
        __syncthreads();
        const int par = a.parent[box];
        if (par < 0) break;  // the topmost level
        if (threadIdx.x == 0) {
            const int last = atomicAdd(&a.ucnt[par], 1) == a.child_count[par] - 1;
            if (last) {
                a.ucnt[par] = 0;  // every child has counted: ready for the next product
                __threadfence();
            }
            s_last = last;
        }
        __syncthreads();
        if (!s_last) break;
        box = par;
        const int c0 = a.child_start[box], nc = a.child_count[box];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            cdf acc = cdf_zero();
            if (wid < nc) {
                const int ch = c0 + wid;
                acc = m2m_binom(cdf_of(__ldcg(a.mult + ((size_t)r * a.nbox + ch) * kFmmP + lane)), a.quad[ch],
                                lane);
            }
            acc = reduce_warps(acc, s_acc, wid, lane);
            if (wid == 0) a.mult[((size_t)r * a.nbox + box) * kFmmP + lane] = cdf_pack(acc);
        }
    }
}

// M2L for every box of levels 2 .. L (block = box)
template <int R>
__global__ void __launch_bounds__(kFmmUT) fmm_m2l_kernel(FmmArgs a) {
    __shared__ float4 s_acc[kFmmTW][32];
    __shared__ float4 s_x[kFmmTW][32];
    if (a.done != nullptr && *a.done) return;
    m2l_box<R>(a, blockIdx.x, threadIdx.x >> 5, threadIdx.x & 31, s_acc, s_x);
}

// L2L, one warp per leaf: the leaf's local expansion is formed from the M2L
// parts of its ancestors, level 2 first, each shifted to the next level by
// the Pascal-matrix L2L (the same operations, in the same order, as a
// level-by-level downward pass; boxes above the leaf are shifted once per
// leaf below them, which costs no waiting), and stored over the leaf's M2L part.
template <int R>
__global__ void __launch_bounds__(32) fmm_l2l_kernel(FmmArgs a) {
    __shared__ int s_path[kFmmMaxDepth];
    __shared__ int s_depth;
    __shared__ float4 s_sv[32];
    if (a.done != nullptr && *a.done) return;
    const int leaf = blockIdx.x, lane = threadIdx.x;
    const int box = a.leaf_box[leaf];
    if (lane == 0) {
        int d = 0;
        for (int bx = box; bx >= 0 && d < kFmmMaxDepth; bx = a.parent[bx]) s_path[d++] = bx;
        s_depth = d;
    }
    __syncwarp();
    const int D = s_depth;  // s_path[D - 1] is on level 2, s_path[0] is the leaf
    if (D < 2) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        cdf v = cdf_of(a.loc[((size_t)r * a.nbox + s_path[D - 1]) * kFmmP + lane]);
        for (int d = D - 2; d >= 0; --d) {
            const int bx = s_path[d];
            v = cdf_add(cdf_of(a.loc[((size_t)r * a.nbox + bx) * kFmmP + lane]),
                        l2l_pascal(v, a.quad[bx], lane, a.bUp, s_sv));
        }
        a.loc[((size_t)r * a.nbox + box) * kFmmP + lane] = cdf_pack(v);
    }
}

constexpr int kFmmWarps = kFmmNT / 32;

// Near field: one block per chunk of up to 32 targets of a leaf (lane = target).
// The sources of the (at most nine) neighbour leaves, taken as one list in
// neighbour order, are split into kFmmWarps equal ranges, one per warp, which
// the warp sums in tiles of 32; the warps' partial sums are added in warp
// order and stored in sorted node order (zn).  The near field runs in
// double-float on the FP32 pipe (GB300's FP64 pipe is 1/64 of it), two
// sources at a time in the two halves of packed float2 instructions (one
// issue for both): d from the exact three-float node coordinates, |d|^2 with
// Dekker products, one Newton step on the reciprocal, compensated
// accumulation into an even-source and an odd-source sum, added at the end.
// EF: also the sums of w_j / (eta_i - eta_j)^2 (to zf), for the gradient.

// d = p - q for two sources (one per half) from exact three-float splits: the
// TwoSums keep every rounding error, so close nodes get d to about 2^-47 |d|.
__device__ __forceinline__ df2 diff3_2(float2 p1, float2 p2, float2 p3, float2 q1, float2 q2, float2 q3) {
    float2 s1, e1, s2, e2, h, l;
    two_diff2(p1, q1, s1, e1);
    two_diff2(p2, q2, s2, e2);
    const float2 s3 = sub2(p3, q3);
    two_sum2(s1, s2, h, l);
    l = add2(l, add2(add2(e1, e2), s3));
    df2 r;
    r.h = add2(h, l);
    r.l = sub2(l, sub2(r.h, h));
    return r;
}

// ---- M2L on the tensor cores.  With x_k = (-1)^(k+1) (2/delta)^k / delta a_k
//   b_l = (1/r) (2/delta)^l sum_k C'(k, l) x_k,   C'(k, l) = C(k+l, l) 2^-(k+l) <= 1:
// for all pairs of boxes one fixed real 32 x 32 matrix times a real matrix whose
// columns are the pairs' real and imaginary parts.  Both sides are split into
// kTcD signed digits of 10 bits (C' once, x per pair below a power of two above
// its largest entry), exact in FP16; the products of digits i and j with
// i + j <= kTcD accumulate in FP32 by i + j, and every such sum is an integer
// below 2^24 (for C' the row sums of its digits bound it), so the tensor cores
// add them without rounding.  What is dropped is below 2^-49 of the largest
// entry times the row sum (<= 2); the double-float form rounds at 2^-46 per term.
// Four pairs make the eight columns of an m16n8k16 tile (lane g = lane / 4 forms
// the B fragment of column g: pair g / 2, part g mod 2; lane t = lane mod 4
// receives both parts of pair t), 76 mma per tile of four pairs.  The legacy
// mma.sync is enough: the tensor work is 2 us of a product, the splits, the
// scalings and the sums around it bound the kernel, and a tcgen05 tile of 128
// rows would be three quarters padding.  An M2L pair takes about 150 instructions
// of a warp; the double-float form 960.  Beside the near field it takes 15.6 us at
// 65,536 nodes (19,700 pairs) and 78 us at 524,288 (135,500); before 35 and 165 us.
// A warp takes tiles of four entries of the box's interaction list; the warps'
// sums are added in warp order.
constexpr int kTcD = 5;
// warps per box: two where there are boxes enough to fill the SMs (beside the near
// field 1, 2 and 4 are within 1.5 % at 1,700 boxes and more), eight in small trees,
// where the topmost boxes' 60 entries would be a chain of tiles
constexpr int kTcManyBoxes = 1024;

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint4 a, unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// round to nearest integer, |v| < 2^22, two lanes
__device__ __forceinline__ float2 rint2(float2 v) {
    const float2 M = f2(12582912.f);  // 1.5 2^23
    return sub2(add2(v, M), M);
}

__device__ __forceinline__ unsigned half2_bits(float2 v) {
    const __half2 h = __floats2half2_rn(v.x, v.y);
    return *reinterpret_cast<const unsigned*>(&h);
}

// y = T x for the eight columns of a tile.  In: x of column g (pair g / 2, part
// g mod 2) at k = 2t + 8q and the next, two k per float2.  Out: rows l = g + 8 i of
// pair t, (re, im) per float2.  T: the fixed matrix's digits as A fragments.
__device__ __forceinline__ void tc_transform(const uint4* __restrict__ T, const df2 (&x)[4], int lane, df2 (&y)[4]) {
    const unsigned full = 0xffffffffu;
    const int t = lane & 3;
    float mx = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) mx = fmaxf(mx, fmaxf(fabsf(x[q].h.x), fabsf(x[q].h.y)));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(full, mx, o));  // lanes of the pair
    const int ex = max((int)(__float_as_uint(mx) >> 23), 8);  // mx < 2^(ex - 126)
    // digits of 2^(135 - ex) x (below 512), as B fragments: k tiles 0 (q = 0, 1) and 1 (q = 2, 3)
    unsigned B[kTcD][4];
    const float2 up = f2(__uint_as_float((unsigned)(262 - ex) << 23)), K = f2(1024.f);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 h = mul2(x[q].h, up), l = mul2(mul2(x[q].l, up), f2(1048576.f));
        float2 d = rint2(h);
        B[0][q] = half2_bits(d);
        float2 v = mul2(sub2(h, d), K);
        d = rint2(v);
        B[1][q] = half2_bits(d);
        v = mul2(sub2(v, d), K);
        d = rint2(add2(v, l));
        B[2][q] = half2_bits(d);
        v = mul2(add2(sub2(v, d), l), K);  // exact: d is the nearest integer to v + l
        d = rint2(v);
        B[3][q] = half2_bits(d);
        v = mul2(sub2(v, d), K);
        B[4][q] = half2_bits(rint2(v));
    }
    float c[kTcD + 1][2][4];
#pragma unroll
    for (int s = 0; s <= kTcD; ++s)
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int u = 0; u < 4; ++u) c[s][m][u] = 0.f;
#pragma unroll
    for (int i = 0; i < kTcD; ++i) {
        uint4 H[2][2];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int kt = 0; kt < 2; ++kt) H[m][kt] = __ldg(T + ((i * 2 + m) * 2 + kt) * 32 + lane);
#pragma unroll
        for (int j = 0; j < kTcD; ++j) {
            if (i + j > kTcD) continue;
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int kt = 0; kt < 2; ++kt) mma_f16(c[i + j][m], H[m][kt], B[j][2 * kt], B[j][2 * kt + 1]);
        }
    }
    // pair t: y = 2^(ex - 126) sum_s c_s 2^(-18 - 10 s)
    const int ext = __shfl_sync(full, ex, 8 * t);
    const float2 dn = f2(__uint_as_float((unsigned)ext << 23));  // 2^(ex - 127), and 2 in w
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 v[kTcD + 1];
        float w = 2.f / 262144.f;
#pragma unroll
        for (int s = 0; s <= kTcD; ++s) {
            v[s] = mul2(make_float2(c[s][i >> 1][2 * (i & 1)], c[s][i >> 1][2 * (i & 1) + 1]), f2(w));
            w *= 1.f / 1024.f;
        }
        float2 h, l0, l1;
        two_sum2(v[0], v[1], h, l0);
        two_sum2(h, v[2], h, l1);
        l0 = add2(add2(l0, l1), add2(v[3], add2(v[4], v[5])));
        y[i].h = add2(h, l0);
        y[i].l = mul2(sub2(l0, sub2(y[i].h, h)), dn);
        y[i].h = mul2(y[i].h, dn);
    }
}

// acc summed over the lanes t (the pairs of a tile) in a fixed order
__device__ __forceinline__ df2 tc_sum_pairs(df2 acc) {
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        df2 v;
        v.h = make_float2(__shfl_xor_sync(full, acc.h.x, o), __shfl_xor_sync(full, acc.h.y, o));
        v.l = make_float2(__shfl_xor_sync(full, acc.l.x, o), __shfl_xor_sync(full, acc.l.y, o));
        acc = df2_add(acc, v);
    }
    return acc;
}

// g^e 2^s for g = sqrt(2) e^{i pi ang / 4} (ang odd): a Gaussian integer times a power of two
__device__ __forceinline__ float2 gauss_pow(int ang, int e, int s) {
    const int a8 = (ang * e) & 7;
    const float m = __uint_as_float((unsigned)(127 + (e >> 1) + s) << 23);
    return make_float2((a8 == 0 || a8 == 1 || a8 == 7) ? m : ((a8 >= 3 && a8 <= 5) ? -m : 0.f),
                       (a8 >= 1 && a8 <= 3) ? m : ((a8 >= 5) ? -m : 0.f));
}

// One part (re, im) of v_k g_k for k and k + 1: v as loaded (re.h, re.l, im.h, im.l), g exact
__device__ __forceinline__ df2 tc_scale_in(float4 v0, float4 v1, float2 g0, float2 g1, int part) {
    const float2 gr = make_float2(g0.x, g1.x), gi = make_float2(g0.y, g1.y);
    const df2 re{make_float2(v0.x, v1.x), make_float2(v0.y, v1.y)}, im{make_float2(v0.z, v1.z), make_float2(v0.w, v1.w)};
    const df2 u = part ? im : re, w = part ? re : df2{neg2(im.h), neg2(im.l)};
    return df2_add(df2{mul2(u.h, gr), mul2(u.l, gr)}, df2{mul2(w.h, gi), mul2(w.l, gi)});
}

// y g for a complex y = (re, im) and an exact factor g
__device__ __forceinline__ df2 tc_scale_out(df2 y, float2 g) {
    const float2 gr = f2(g.x), gi = make_float2(-g.y, g.y);
    const float2 xh = make_float2(y.h.y, y.h.x), xl = make_float2(y.l.y, y.l.x);
    return df2_add(df2{mul2(y.h, gr), mul2(y.l, gr)}, df2{mul2(xh, gi), mul2(xl, gi)});
}

template <int R, int W>
__global__ void __launch_bounds__(32 * W) fmm_m2l_tc_kernel(FmmArgs a) {
    __shared__ float4 s_acc[W][32];
    if (a.done != nullptr && *a.done) return;
    const int box = blockIdx.x, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3, part = g & 1;
    const int e0 = a.il_start[box], e1 = a.il_start[box + 1];
    const df sc = df_split_fast(recip_f64(a.width[box]));
#pragma unroll
    for (int r = 0; r < R; ++r) {
        df2 acc[4];  // (re, im) of rows l = g + 8 i
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = df2{f2(0.f), f2(0.f)};
        // the list entries of a tile are loaded during the one before
        int base = e0 + 4 * wid, ob = 0, sb = 0, oc = 0;
        if (base < e1) {
            ob = __ldg(a.il_off + min(base + (g >> 1), e1 - 1));
            sb = __ldg(a.il_src + min(base + (g >> 1), e1 - 1));
            oc = __ldg(a.il_off + min(base + t, e1 - 1));
        }
        for (; base < e1; base += 4 * W) {
            const float4* S = a.m2lT + (size_t)ob * 2 * kFmmP;
            const float4* A = a.mult + ((size_t)r * a.nbox + sb) * kFmmP;
            const float4* Q = a.m2lT + ((size_t)oc * 2 + 1) * kFmmP;
            if (base + 4 * W < e1) {
                ob = __ldg(a.il_off + min(base + 4 * W + (g >> 1), e1 - 1));
                sb = __ldg(a.il_src + min(base + 4 * W + (g >> 1), e1 - 1));
                oc = __ldg(a.il_off + min(base + 4 * W + t, e1 - 1));
            }
            const bool live = base + (g >> 1) < e1;
            df2 x[4], y[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = 2 * t + 8 * q;
                const float4 a0 = __ldcg(A + k), a1 = __ldcg(A + k + 1), s0 = __ldg(S + k), s1 = __ldg(S + k + 1);
                const df2 ar{make_float2(a0.x, a1.x), make_float2(a0.y, a1.y)};
                const df2 ai{make_float2(a0.z, a1.z), make_float2(a0.w, a1.w)};
                const df2 sr{make_float2(s0.x, s1.x), make_float2(s0.y, s1.y)};
                const df2 si{make_float2(s0.z, s1.z), make_float2(s0.w, s1.w)};
                // re = sr ar - si ai, im = sr ai + si ar
                const df2 u = part ? ai : ar, v = part ? ar : df2{neg2(ai.h), neg2(ai.l)};
                df2 w = df2_mul(sr, u);
                df2_acc(w, df2_mul(si, v));
                x[q].h = add2(w.h, w.l);
                x[q].l = sub2(w.l, sub2(x[q].h, w.h));
                if (!live) x[q] = df2{f2(0.f), f2(0.f)};
            }
            tc_transform(a.m2lA, x, lane, y);
#pragma unroll
            for (int i = 0; i < 4; ++i) {  // (2/delta)^l y_l
                const float4 q4 = __ldg(Q + g + 8 * i);
                df2_acc(acc[i], df2_mul(y[i], df2{f2(q4.x), f2(q4.y)}));
                const df2 yx{make_float2(y[i].h.y, y[i].h.x), make_float2(y[i].l.y, y[i].l.x)};
                df2_acc(acc[i], df2_mul(yx, df2{make_float2(-q4.z, q4.z), make_float2(-q4.w, q4.w)}));
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc[i] = tc_sum_pairs(acc[i]);
            if (t == 0) s_acc[wid][g + 8 * i] = make_float4(acc[i].h.x, acc[i].l.x, acc[i].h.y, acc[i].l.y);
        }
        __syncthreads();
        if (wid == 0) {
            cdf b = cdf_of(s_acc[0][lane]);
            for (int w = 1; w < W; ++w) b = cdf_add(b, cdf_of(s_acc[w][lane]));
            a.loc[((size_t)r * a.nbox + box) * kFmmP + lane] = cdf_pack(cdf{df_mul(b.re, sc), df_mul(b.im, sc)});
        }
        if (R > 1) __syncthreads();
    }
}

// ---- The upward pass, one block per leaf: P2M, then warp 0 alone carries the
// multipoles up: the warp that completes the last child of a box (an atomic
// count per box; nothing waits) forms that box's M2M from its at most four
// children, one tile of tc_transform, and goes on to the parent.  With g the child's
// Gaussian integer (above) and C(m,k) 2^-m the fixed matrix,
//   a0_m = (g/2)^m sum_k C(m,k) 2^-m [conj(g)^k a1_k].
// Latency bounds it: per level a fence, an atomic, the children's multipoles and
// one transform.  The leaf's path (boxes, child ranges) is read while the P2M runs.
template <int R>
__global__ void __launch_bounds__(kFmmUT) fmm_up_tc_kernel(FmmArgs a) {
    __shared__ float4 s_v[kFmmTW][8 * kP2mStride];
    __shared__ float4 s_acc[kFmmTW][32];
    if (a.done != nullptr && *a.done) return;
    const unsigned full = 0xffffffffu;
    const int leaf = blockIdx.x, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // lane d of warp 0: the leaf's ancestor d levels up
    int pbox = 0, pc0 = 0, pnc = 0;
    if (wid == 0 && lane < a.depth) {
        pbox = (int)(a.path[(size_t)leaf * a.depth + lane] & 0x3fffffffu);
        pc0 = a.child_start[pbox];
        pnc = a.child_count[pbox];
    }
    p2m_leaf<R>(a, leaf, a.leaf_box[leaf], wid, lane, s_v[wid], s_acc);
    if (wid != 0) return;
    const int g = lane >> 2, t = lane & 3, part = g & 1;
    for (int d = 1; d < a.depth; ++d) {
        const int box = __shfl_sync(full, pbox, d), c0 = __shfl_sync(full, pc0, d), nc = __shfl_sync(full, pnc, d);
        __threadfence();  // the child's multipole before the count
        __syncwarp();
        int last = 0;
        if (lane == 0) {
            last = atomicAdd(&a.ucnt[box], 1) == nc - 1;
            if (last) {
                a.ucnt[box] = 0;  // every child has counted: ready for the next product
                __threadfence();
            }
        }
        if (!__shfl_sync(full, last, 0)) return;
        const int cb = c0 + min(g >> 1, nc - 1);
        const bool live = (g >> 1) < nc;
        const int angb = gauss_angle(__ldg(a.quad + cb)), angc = gauss_angle(__ldg(a.quad + c0 + min(t, nc - 1)));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4* A = a.mult + ((size_t)r * a.nbox + cb) * kFmmP;
            df2 x[4], y[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = 2 * t + 8 * q;
                x[q] = tc_scale_in(__ldcg(A + k), __ldcg(A + k + 1), gauss_pow(8 - angb, k, 0),
                                   gauss_pow(8 - angb, k + 1, 0), part);
                if (!live) x[q] = df2{f2(0.f), f2(0.f)};
            }
            tc_transform(a.upA, x, lane, y);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int m = g + 8 * i;
                const df2 v = tc_sum_pairs(tc_scale_out(y[i], gauss_pow(angc, m, -m)));
                if (t == 0)
                    a.mult[((size_t)r * a.nbox + box) * kFmmP + m] = make_float4(v.h.x, v.l.x, v.h.y, v.l.y);
            }
        }
    }
}

// ---- L2L, one warp per four leaves (the pairs of a tile): each leaf's local
// expansion is carried down from its topmost ancestor, one tc_transform per
// level, the M2L part of the next box added:
//   b1_m = conj(g)^m sum_l C(l,m) 2^-l [(g/2)^l b0_l].
// Between levels the result goes from the rows of the accumulators to the
// columns of the next operand through shared memory.  (One warp per leaf with a
// 32-term double-float sum per lane and level: 13 us at 65,536 nodes.)
template <int R>
__global__ void __launch_bounds__(32) fmm_l2l_tc_kernel(FmmArgs a) {
    __shared__ float4 s_v[4][33];
    if (a.done != nullptr && *a.done) return;
    const int lane = threadIdx.x, g = lane >> 2, t = lane & 3, part = g & 1, pb = g >> 1;
    const int D = a.depth;
    const int leafb = min(4 * (int)blockIdx.x + pb, a.nleaf - 1), leafc = min(4 * (int)blockIdx.x + t, a.nleaf - 1);
    const unsigned *pathb = a.path + (size_t)leafb * D, *pathc = a.path + (size_t)leafc * D;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float4* loc = a.loc + (size_t)r * a.nbox * kFmmP;
        df2 v[4];
        {
            const float4* b = loc + (size_t)(pathc[D - 1] & 0x3fffffffu) * kFmmP;
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = pc_of(b[g + 8 * i]);
        }
        for (int d = D - 2; d >= 0; --d) {
            const unsigned eb = __ldg(pathb + d), ec = __ldg(pathc + d);
            const int angb = gauss_angle((int)(eb >> 30)), angc = gauss_angle((int)(ec >> 30));
            const float4* b = loc + (size_t)(ec & 0x3fffffffu) * kFmmP;
            float4 nxt[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) nxt[i] = b[g + 8 * i];
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) s_v[t][g + 8 * i] = make_float4(v[i].h.x, v[i].l.x, v[i].h.y, v[i].l.y);
            __syncwarp();
            df2 x[4], y[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = 2 * t + 8 * q;
                x[q] = tc_scale_in(s_v[pb][k], s_v[pb][k + 1], gauss_pow(angb, k, -k), gauss_pow(angb, k + 1, -k - 1),
                                   part);
            }
            tc_transform(a.dnA, x, lane, y);
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = df2_add(pc_of(nxt[i]), tc_scale_out(y[i], gauss_pow(8 - angc, g + 8 * i, 0)));
        }
        if (4 * (int)blockIdx.x + t < a.nleaf) {
            float4* b = loc + (size_t)(pathc[0] & 0x3fffffffu) * kFmmP;
#pragma unroll
            for (int i = 0; i < 4; ++i) b[g + 8 * i] = make_float4(v[i].h.x, v[i].l.x, v[i].h.y, v[i].l.y);
        }
    }
}

// The path of every leaf: itself, then its ancestors up to the topmost level.
__global__ void fmm_path_kernel(FmmArgs a, unsigned* path) {
    const int leaf = blockIdx.x * blockDim.x + threadIdx.x;
    if (leaf >= a.nleaf) return;
    int box = a.leaf_box[leaf];
    for (int d = 0; d < a.depth; ++d) {
        path[(size_t)leaf * a.depth + d] = (unsigned)box | ((unsigned)a.quad[box] << 30);
        box = a.parent[box];
    }
}

// INV: 0 forms 1/d; 1 forms and stores it (no sums: the build of the inverse
// cache); 2 reads it (bit for bit the same sums as 0); 3 forms it, folded: an item
// with 16 targets or fewer (the last of a leaf) would leave half its lanes idle, so
// the lanes form groups of `width`, each with its share of the source pairs (a leaf
// of 68 nodes takes 2 + 1/8 instead of 3 turns of its sources; one Cauchy sum at
// N = 65,536 169 -> 164 us).  Handles built for differentiation keep 0.
template <int R, bool EF, int INV = 0>
__global__ void __launch_bounds__(kFmmNT) fmm_near_kernel(FmmArgs a) {
    constexpr int RS = EF ? 2 * R : R;
    // one tile of 32 sources per warp, component by component, so that a
    // float2 read at pair p gives sources 2p and 2p + 1
    __shared__ float s_c[kFmmWarps][6][32];        // x1, x2, x3, y1, y2, y3
    __shared__ float s_w[kFmmWarps][R][4][32];     // wx.h, wx.l, wy.h, wy.l
    __shared__ int s_j[kFmmWarps][32];             // sorted index of each source (-1: padding)
    __shared__ double2 s_z[kFmmWarps][RS][32];
    __shared__ int s_cum[kFmmMaxNbr + 1];          // prefix sums of the neighbour leaves' sizes
    __shared__ int s_beg[kFmmMaxNbr];              // first source of each neighbour leaf
    if (a.done != nullptr && *a.done) return;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int2 it = a.items[blockIdx.x];  // (leaf, first target)
    const int leaf = it.x;
    const int t1 = a.leaf_start[leaf + 1];
    const int tn = min(32, t1 - it.y);
    int width = 32;  // lanes per group: group lane / width takes the pairs lane / width + (32 / width) u
    if (INV == 3)
        while (width > 2 && (width >> 1) >= tn) width >>= 1;
    const int lt = INV == 3 ? lane & (width - 1) : lane;  // the lane's target
    const int p0 = INV == 3 ? lane / width : 0, pstep = INV == 3 ? 32 / width : 1;
    const int i = it.y + lt;
    const bool act = i < t1;
    const float4 pa = (INV != 2) ? a.p3[act ? i : it.y] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float2 pb = (INV != 2) ? a.p3b[act ? i : it.y] : make_float2(0.f, 0.f);
    const float2 tx1 = f2(pa.x), tx2 = f2(pa.y), tx3 = f2(pa.z), ty1 = f2(pa.w), ty2 = f2(pb.x), ty3 = f2(pb.y);
    df2 are[RS], aim[RS];
#pragma unroll
    for (int r = 0; r < RS; ++r) are[r] = aim[r] = df2{f2(0.f), f2(0.f)};
    const int n0 = a.nl_start[leaf], nn = min(a.nl_start[leaf + 1] - n0, kFmmMaxNbr);
    if (threadIdx.x == 0) {
        int c = 0;
        for (int e = 0; e < nn; ++e) {
            const int nl = a.nl_leaf[n0 + e];
            s_beg[e] = a.leaf_start[nl];
            s_cum[e] = c;
            c += a.leaf_start[nl + 1] - a.leaf_start[nl];
        }
        s_cum[nn] = c;
    }
    __syncthreads();
    const int total = s_cum[nn];
    const int q0 = (int)((long long)total * wid / kFmmWarps), q1 = (int)((long long)total * (wid + 1) / kFmmWarps);
    long long entry = 0;  // of this warp's pair in hand: the items' entries, warp after warp, pair-major
    if (INV == 1 || INV == 2) {
        entry = a.inv_off[blockIdx.x];
        for (int w = 0; w < wid; ++w)
            entry += (long long)tn * (((int)((long long)total * (w + 1) / kFmmWarps) -
                                       (int)((long long)total * w / kFmmWarps) + 1) >> 1);
        entry += min(lane, tn - 1);
    }
    for (int qs = q0; qs < q1; qs += 32) {
        __syncwarp();
        const int cnt = min(32, q1 - qs);
        {
            const int q = qs + min(lane, cnt - 1);  // lanes past the end copy the last source, weight 0
            int e = 0;
            while (e + 1 < nn && s_cum[e + 1] <= q) ++e;
            const int j = s_beg[e] + (q - s_cum[e]);
            const bool pad = lane >= cnt;
            if (INV != 2) {
                const float4 c4 = a.p3[j];
                const float2 c2 = a.p3b[j];
                s_c[wid][0][lane] = c4.x;
                s_c[wid][1][lane] = c4.y;
                s_c[wid][2][lane] = c4.z;
                s_c[wid][3][lane] = c4.w;
                s_c[wid][4][lane] = c2.x;
                s_c[wid][5][lane] = c2.y;
                s_j[wid][lane] = pad ? -1 : j;
            }
#pragma unroll
            for (int r = 0; r < (INV == 1 ? 0 : R); ++r) {
                const float4 w4 = pad ? make_float4(0.f, 0.f, 0.f, 0.f) : a.ws[(size_t)r * a.N + j];
                s_w[wid][r][0][lane] = w4.x;
                s_w[wid][r][1][lane] = w4.y;
                s_w[wid][r][2][lane] = w4.z;
                s_w[wid][r][3][lane] = w4.w;
            }
        }
        __syncwarp();
        const int npair = (cnt + 1) >> 1;
        float4 vr[4], vi[4];  // INV == 2: four pairs' entries in flight
#pragma unroll 4
        for (int pp = p0; pp < npair; pp += pstep) {
            if (INV == 2 && (pp & 3) == 0) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (pp + u < npair) {
                        vr[u] = __ldcs(a.inv_r + entry + (long long)u * tn);
                        vi[u] = __ldcs(a.inv_i + entry + (long long)u * tn);
                    }
                entry += 4LL * tn;
            }
            df2 ar, ai;  // 1/d = ar - i ai
            if (INV == 2) {
                ar = df2{make_float2(vr[pp & 3].x, vr[pp & 3].y), make_float2(vr[pp & 3].z, vr[pp & 3].w)};
                ai = df2{make_float2(vi[pp & 3].x, vi[pp & 3].y), make_float2(vi[pp & 3].z, vi[pp & 3].w)};
            } else {
                const float2 qx1 = reinterpret_cast<const float2*>(s_c[wid][0])[pp];
                const float2 qx2 = reinterpret_cast<const float2*>(s_c[wid][1])[pp];
                const float2 qx3 = reinterpret_cast<const float2*>(s_c[wid][2])[pp];
                const float2 qy1 = reinterpret_cast<const float2*>(s_c[wid][3])[pp];
                const float2 qy2 = reinterpret_cast<const float2*>(s_c[wid][4])[pp];
                const float2 qy3 = reinterpret_cast<const float2*>(s_c[wid][5])[pp];
                const int2 jj = reinterpret_cast<const int2*>(s_j[wid])[pp];
                const df2 dx = diff3_2(tx1, tx2, tx3, qx1, qx2, qx3);
                const df2 dy = diff3_2(ty1, ty2, ty3, qy1, qy2, qy3);
                const float2 px = mul2(dx.h, dx.h);
                float2 ex = fma2(dx.h, dx.h, neg2(px));
                ex = fma2(dx.h, add2(dx.l, dx.l), ex);
                const float2 py = mul2(dy.h, dy.h);
                float2 ey = fma2(dy.h, dy.h, neg2(py));
                ey = fma2(dy.h, add2(dy.l, dy.l), ey);
                float2 rh, re;
                two_sum2(px, py, rh, re);
                const float2 rl = add2(add2(ex, ey), re);
                float2 y = make_float2(recip_f32(rh.x), recip_f32(rh.y));
                // the i = j term is excluded (Eq. fmm-E); padding slots (j < 0) add nothing
                y.x = (jj.x == i || jj.x < 0) ? 0.f : y.x;
                y.y = (jj.y == i || jj.y < 0) ? 0.f : y.y;
                float2 ee = fma2(neg2(rh), y, f2(1.0f));
                ee = fma2(neg2(rl), y, ee);
                const df2 inv{y, mul2(y, ee)};
                ar = df2_mul(dx, inv);
                ai = df2_mul(dy, inv);
            }
            if (INV == 1) {
                if (act) {
                    a.inv_r[entry] = make_float4(ar.h.x, ar.h.y, ar.l.x, ar.l.y);
                    a.inv_i[entry] = make_float4(ai.h.x, ai.h.y, ai.l.x, ai.l.y);
                }
                entry += tn;
                continue;
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const df2 wx{reinterpret_cast<const float2*>(s_w[wid][r][0])[pp],
                             reinterpret_cast<const float2*>(s_w[wid][r][1])[pp]};
                const df2 wy{reinterpret_cast<const float2*>(s_w[wid][r][2])[pp],
                             reinterpret_cast<const float2*>(s_w[wid][r][3])[pp]};
                df2_acc(are[r], df2_mul(wx, ar));
                df2_acc(are[r], df2_mul(wy, ai));
                df2_acc(aim[r], df2_mul(wy, ar));
                df2_dec(aim[r], df2_mul(wx, ai));
            }
            if (EF) {  // 1/d^2 = (ar - i ai)^2 = gr - i gi
                const df2 a2 = df2_mul(ar, ar), b2 = df2_mul(ai, ai), ab = df2_mul(ar, ai);
                const df2 gr = df2_add(a2, df2_neg(b2));
                const df2 gi{add2(ab.h, ab.h), add2(ab.l, ab.l)};
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const df2 wx{reinterpret_cast<const float2*>(s_w[wid][r][0])[pp],
                                 reinterpret_cast<const float2*>(s_w[wid][r][1])[pp]};
                    const df2 wy{reinterpret_cast<const float2*>(s_w[wid][r][2])[pp],
                                 reinterpret_cast<const float2*>(s_w[wid][r][3])[pp]};
                    df2_acc(are[R + r], df2_mul(wx, gr));
                    df2_acc(are[R + r], df2_mul(wy, gi));
                    df2_acc(aim[R + r], df2_mul(wy, gr));
                    df2_dec(aim[R + r], df2_mul(wx, gi));
                }
            }
        }
    }
    if (INV == 1) return;
#pragma unroll
    for (int r = 0; r < RS; ++r) {  // even + odd sums, then to FP64
        const df sr = df_add(df{are[r].h.x, are[r].l.x}, df{are[r].h.y, are[r].l.y});
        const df si = df_add(df{aim[r].h.x, aim[r].l.x}, df{aim[r].h.y, aim[r].l.y});
        double2 v = make_double2((double)sr.h + (double)sr.l, (double)si.h + (double)si.l);
        if (INV == 3)
            for (int o = width; o < 32; o <<= 1) {  // the groups' sums
                v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
            }
        s_z[wid][r][lane] = v;
    }
    __syncthreads();
    if (wid == 0 && act && lane == lt) {
#pragma unroll
        for (int r = 0; r < RS; ++r) {
            double2 v = s_z[0][r][lane];
            for (int w = 1; w < kFmmWarps; ++w) {
                v.x += s_z[w][r][lane].x;
                v.y += s_z[w][r][lane].y;
            }
            if (r < R)
                a.zn[(size_t)r * a.N + i] = v;
            else
                a.zf[(size_t)(r - R) * a.N + i] = v;
        }
    }
}

// The offset t = (s - c)/r of every node from the centre of its leaf in leaf
// widths, double-float complex, in sorted order: formed once per tree, read by
// P2M and L2P (whose FP64 subtraction and product it replaces).
__global__ void fmm_tn_build_kernel(FmmArgs a, float4* __restrict__ tn) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.N) return;
    const int box = a.node_box[i];
    const double2 c = a.center[box];
    const double ir = 1.0 / a.width[box];
    const double2 p = a.ps[i];
    const cdf t = cdf_split(make_double2((p.x - c.x) * ir, (p.y - c.y) * ir));
    tn[i] = cdf_pack(t);
}

// ---- Near-field operator caches.  The geometry of a handle is fixed for all
// its products, so the near-field part of an operator, the matrix
//   f_i w_j / (eta_i - eta_j)   (i = j: 0)
// over each work item's targets i (a chunk of tn <= 32 nodes of a leaf) and
// sources j (the nodes of its neighbour leaves, in neighbour order), is
// formed once, in double-float from the exact three-float coordinates like
// the near-field kernel above, and each product then only reads it:
//   f_i z_i = sum_j x_j f_i w_j / (eta_i - eta_j).
// (w, f) = (q, A) for the products z = E(q x), whose operators read A z, and
// (A, q) for the solves with z = E(A x), whose operators read Im(q z).  With
// the target's factor inside, an operator that needs one part of f z reads one
// part of the cache, 8 bytes per pair, whether or not f is real.
// Layout per item, for source pairs p = (2p, 2p + 1) and targets (lanes):
//   re[off + p tn + lane] = (Re hi of 2p, of 2p+1, Re lo of 2p, of 2p+1)
// and im likewise, so a float4 load gives the packed double-float operand
// of the two sources.

// The shape of every work item: S sources, tn targets, the entries, and the
// run of sorted nodes that each of its neighbour leaves is.
__global__ void fmm_nq_shape_kernel(FmmArgs a, long long* cnt, int2* nq_item, int2* nq_run) {
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= a.nitems) return;
    const int2 item = a.items[it];
    const int leaf = item.x;
    const int tn = min(32, a.leaf_start[leaf + 1] - item.y);
    const int n0 = a.nl_start[leaf], nn = min(a.nl_start[leaf + 1] - n0, kFmmMaxNbr);
    int c = 0;
    for (int e = 0; e < kFmmMaxNbr; ++e) {
        int2 run = make_int2(0, INT_MAX);
        if (e < nn) {
            const int nl = a.nl_leaf[n0 + e];
            const int j0 = a.leaf_start[nl];
            run = make_int2(j0, c);
            c += a.leaf_start[nl + 1] - j0;
        }
        nq_run[(size_t)it * kFmmMaxNbr + e] = run;
    }
    nq_item[it] = make_int2(c, tn);
    cnt[it] = (long long)((c + 1) / 2) * tn;
}

// Entries of each item's inverse cache: per warp of the direct near-field kernel
// its share of the sources, two per entry, times the targets.
__global__ void fmm_inv_count_kernel(FmmArgs a, long long* cnt) {
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= a.nitems) return;
    const int2 item = a.items[it];
    const int leaf = item.x;
    const int tn = min(32, a.leaf_start[leaf + 1] - item.y);
    const int n0 = a.nl_start[leaf], nn = min(a.nl_start[leaf + 1] - n0, kFmmMaxNbr);
    int total = 0;
    for (int e = 0; e < nn; ++e) total += a.leaf_start[a.nl_leaf[n0 + e] + 1] - a.leaf_start[a.nl_leaf[n0 + e]];
    long long c = 0;
    for (int w = 0; w < kFmmWarps; ++w)
        c += ((int)((long long)total * (w + 1) / kFmmWarps) - (int)((long long)total * w / kFmmWarps) + 1) >> 1;
    cnt[it] = c * tn;
}

// The sorted node of source q of an item: lane e of the warp holds run e
// (first source, sources before it).  Every lane of the warp calls it.
__device__ __forceinline__ int nq_source(int2 run, int q) {
    const unsigned full = 0xffffffffu;
    int j = __shfl_sync(full, run.x, 0) + q;
#pragma unroll
    for (int e = 1; e < kFmmMaxNbr; ++e) {
        const int beg = __shfl_sync(full, run.x, e), cum = __shfl_sync(full, run.y, e);
        if (q >= cum) j = beg + (q - cum);
    }
    return j;
}

// off[i] = cnt[0] + ... + cnt[i - 1] for i <= n (one block of 1024 threads,
// each a contiguous range, a block scan of the range sums in between).
__global__ void __launch_bounds__(1024) fmm_nq_scan_kernel(const long long* __restrict__ cnt, int n,
                                                            long long* __restrict__ off) {
    __shared__ long long s[1024];
    const int t = threadIdx.x;
    const int per = (n + 1023) / 1024;
    const int b0 = min(n, t * per), b1 = min(n, b0 + per);
    long long sum = 0;
    for (int i = b0; i < b1; ++i) sum += cnt[i];
    s[t] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const long long v = (t >= o) ? s[t - o] : 0;
        __syncthreads();
        s[t] += v;
        __syncthreads();
    }
    long long run = (t == 0) ? 0 : s[t - 1];
    for (int i = b0; i < b1; ++i) {
        off[i] = run;
        run += cnt[i];
    }
    if (t == 1023) off[n] = s[1023];
}

// The entries f_i w_j / (eta_i - eta_j): one block per work item, warp w taking
// its share of the source pairs.  RE: the real parts too; FC: f is complex
// (else only its real part is used).
template <bool RE, bool FC>
__global__ void __launch_bounds__(kFmmNT) fmm_nq_build_kernel(FmmArgs a, const double2* __restrict__ wgt,
                                                              const double2* __restrict__ fac,
                                                              const long long* __restrict__ off,
                                                              const int2* __restrict__ nq_item,
                                                              const int2* __restrict__ nq_run,
                                                              float4* __restrict__ out_re,
                                                              float4* __restrict__ out_im) {
    __shared__ float s_c[kFmmWarps][6][32];   // x1, x2, x3, y1, y2, y3 of the tile's sources
    __shared__ float s_q[kFmmWarps][4][32];   // weight: re.h, re.l, im.h, im.l
    __shared__ int s_j[kFmmWarps][32];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int it = blockIdx.x;
    const int2 shape = nq_item[it];
    const int S = shape.x, tn = shape.y;
    const int2 run = (lane < kFmmMaxNbr) ? nq_run[(size_t)it * kFmmMaxNbr + lane] : make_int2(0, INT_MAX);
    const int i = a.items[it].y + min(lane, tn - 1);
    const float4 pa = a.p3[i];
    const float2 pb = a.p3b[i];
    const float2 tx1 = f2(pa.x), tx2 = f2(pa.y), tx3 = f2(pa.z), ty1 = f2(pa.w), ty2 = f2(pb.x), ty3 = f2(pb.y);
    const double2 fi = fac[a.perm[i]];
    const df fr = df_split(fi.x), fm = df_split(fi.y);
    const df2 fre{f2(fr.h), f2(fr.l)}, fim{f2(fm.h), f2(fm.l)};
    const int npair = (S + 1) >> 1;
    const int p0 = (int)((long long)npair * wid / kFmmWarps), p1 = (int)((long long)npair * (wid + 1) / kFmmWarps);
    const long long base = off[it];
    for (int ps = p0; ps < p1; ps += 16) {
        __syncwarp();
        const int np = min(16, p1 - ps);
        const int cnt = min(2 * np, S - 2 * ps);  // sources of this tile
        {
            const int j = nq_source(run, 2 * ps + min(lane, cnt - 1));
            const float4 c4 = a.p3[j];
            const float2 c2 = a.p3b[j];
            s_c[wid][0][lane] = c4.x;
            s_c[wid][1][lane] = c4.y;
            s_c[wid][2][lane] = c4.z;
            s_c[wid][3][lane] = c4.w;
            s_c[wid][4][lane] = c2.x;
            s_c[wid][5][lane] = c2.y;
            s_j[wid][lane] = (lane < cnt) ? j : -1;
            const double2 qj = wgt[a.perm[j]];
            const df qr = df_split(qj.x), qi = df_split(qj.y);
            s_q[wid][0][lane] = qr.h;
            s_q[wid][1][lane] = qr.l;
            s_q[wid][2][lane] = qi.h;
            s_q[wid][3][lane] = qi.l;
        }
        __syncwarp();
        for (int pp = 0; pp < np; ++pp) {
            const float2 qx1 = reinterpret_cast<const float2*>(s_c[wid][0])[pp];
            const float2 qx2 = reinterpret_cast<const float2*>(s_c[wid][1])[pp];
            const float2 qx3 = reinterpret_cast<const float2*>(s_c[wid][2])[pp];
            const float2 qy1 = reinterpret_cast<const float2*>(s_c[wid][3])[pp];
            const float2 qy2 = reinterpret_cast<const float2*>(s_c[wid][4])[pp];
            const float2 qy3 = reinterpret_cast<const float2*>(s_c[wid][5])[pp];
            const int2 jj = reinterpret_cast<const int2*>(s_j[wid])[pp];
            const df2 dx = diff3_2(tx1, tx2, tx3, qx1, qx2, qx3);
            const df2 dy = diff3_2(ty1, ty2, ty3, qy1, qy2, qy3);
            const float2 px = mul2(dx.h, dx.h);
            float2 ex = fma2(dx.h, dx.h, neg2(px));
            ex = fma2(dx.h, add2(dx.l, dx.l), ex);
            const float2 py = mul2(dy.h, dy.h);
            float2 ey = fma2(dy.h, dy.h, neg2(py));
            ey = fma2(dy.h, add2(dy.l, dy.l), ey);
            float2 rh, re;
            two_sum2(px, py, rh, re);
            const float2 rl = add2(add2(ex, ey), re);
            float2 y = make_float2(recip_f32(rh.x), recip_f32(rh.y));
            y.x = (jj.x == i || jj.x < 0) ? 0.f : y.x;  // i = j excluded (Eq. fmm-E); padding
            y.y = (jj.y == i || jj.y < 0) ? 0.f : y.y;
            float2 ee = fma2(neg2(rh), y, f2(1.0f));
            ee = fma2(neg2(rl), y, ee);
            const df2 inv{y, mul2(y, ee)};
            const df2 ar = df2_mul(dx, inv), ai = df2_mul(dy, inv);  // 1/d = ar - i ai
            const df2 qre{reinterpret_cast<const float2*>(s_q[wid][0])[pp], reinterpret_cast<const float2*>(s_q[wid][1])[pp]};
            const df2 qim{reinterpret_cast<const float2*>(s_q[wid][2])[pp], reinterpret_cast<const float2*>(s_q[wid][3])[pp]};
            // w (ar - i ai) = (wre ar + wim ai) + i (wim ar - wre ai)
            df2 Qr = df2_mul(qre, ar), Qi = df2_mul(qim, ar);
            df2_acc(Qr, df2_mul(qim, ai));
            df2_dec(Qi, df2_mul(qre, ai));
            // times the target's factor
            df2 Pi = df2_mul(fre, Qi), Pr = df2_mul(fre, Qr);
            if (FC) {
                df2_acc(Pi, df2_mul(fim, Qr));
                df2_dec(Pr, df2_mul(fim, Qi));
            }
            if (lane < tn) {
                const size_t o = (size_t)(base + (long long)(ps + pp) * tn + lane);
                if (RE) out_re[o] = make_float4(Pr.h.x, Pr.h.y, Pr.l.x, Pr.l.y);
                out_im[o] = make_float4(Pi.h.x, Pi.h.y, Pi.l.x, Pi.l.y);
            }
        }
    }
}

// A cached near field, streamed into shared memory by the Tensor Memory
// Accelerator: one block per work item (or, where the items do not fill the
// SMs, per item and share of its sources); a producer thread issues bulk copies
// of the item's cache entries (contiguous, pair-major) in chunks of kNbPairs
// source pairs through a ring of kNbStages buffers (full/empty mbarriers).  The 8
// consumer warps first gather the x of the item's sources (at most nine runs of
// sorted nodes) through the node order into shared memory, all loads independent,
// while the first copies are in flight (lists of x written by a launch of their
// own took 19 us per product at 65,536 nodes and 350 us at 524,288; a gather by
// the producer, chunk by chunk, made small items a chain of load latencies, 26 us
// for 2,560 nodes); then lane = target, warp w taking pairs w, w + 8, ... of
// each chunk.  Even and odd sources go to the two halves of packed float2 sums,
// added at the end, then the warps' sums in warp order.  COMP = 1: the imaginary
// part only (the real part written as 0).  `stream`: the entries are marked
// evict-first in L2 (a cache larger than L2 read once per product must not push
// out what is reused).  Every wait is bounded (kNbSpin polls); one that gives up
// sets a.fault, and the producer still waits (bounded) for its copies in flight
// before leaving.
constexpr int kNbPairs = 24;                 // source pairs per chunk, three per consumer warp
constexpr int kNbStages = 3;
constexpr int kNbThreads = kFmmNT + 32;      // 8 consumer warps and the producer warp
constexpr int kNbSpin = 1 << 22;
constexpr int kNbSegChunks = 20;             // chunks whose x is gathered at once
constexpr int kNbX = 2 * kNbPairs * kNbSegChunks;

template <int R, int COMP>
struct NbLayout {
    static constexpr int kParts = COMP == 0 ? 2 : 1;
    static constexpr int kQ = kNbPairs * 32;                  // float4 entries of one part (tn <= 32)
    static constexpr int kStage = kParts * kQ;                // float4 per stage
    static constexpr int kBytes = kNbStages * kStage * 16 + R * kNbX * 8;  // dynamic shared memory
};

template <int R, int COMP>
__global__ void __launch_bounds__(kNbThreads) fmm_near_bulk_kernel(FmmArgs a, const long long* __restrict__ off,
                                                                   const int2* __restrict__ nq_item,
                                                                   const int2* __restrict__ nq_run,
                                                                   const float4* __restrict__ nq_re,
                                                                   const float4* __restrict__ nq_im, int stream) {
    using L = NbLayout<R, COMP>;
    extern __shared__ __align__(16) float4 nb_buf[];
    float2* s_x = reinterpret_cast<float2*>(nb_buf + kNbStages * L::kStage);  // [R][kNbX]
    __shared__ __align__(8) unsigned long long full[kNbStages], empty[kNbStages];
    __shared__ double2 s_z[kFmmWarps][R][32];
    if (a.done != nullptr && *a.done) return;  // set before this launch: the same in every thread
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int it = blockIdx.x;
    const int2 d = __ldg(nq_item + it);  // (S, tn)
    const long long o0 = __ldg(off + it);
    const int S = d.x, tn = d.y;
    const int npair = (S + 1) >> 1;
    const int nch = (npair + kNbPairs - 1) / kNbPairs;
    const int cb = nch * (int)blockIdx.y / (int)gridDim.y, ce = nch * ((int)blockIdx.y + 1) / (int)gridDim.y;
    if (threadIdx.x == kFmmNT) {
        for (int k = 0; k < kNbStages; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], kFmmWarps);
        }
    }
    __syncthreads();
    if (wid == kFmmWarps) {  // the producer
        if (lane == 0) {
            int c = cb;
            for (; c < ce; ++c) {
                const int u = c - cb, st = u % kNbStages;
                if (u >= kNbStages && !mbar_wait(&empty[st], (unsigned)((u / kNbStages - 1) & 1), kNbSpin)) {
                    atomicExch(a.fault, 1);
                    break;
                }
                const int p0 = c * kNbPairs, np = min(kNbPairs, npair - p0);
                const unsigned qbytes = (unsigned)(np * tn) * 16u;
                float4* stage = nb_buf + (size_t)st * L::kStage;
                mbar_expect_tx(&full[st], L::kParts * qbytes);
                const float4* im = nq_im + o0 + (long long)p0 * tn;
                const float4* re = (COMP == 0) ? nq_re + o0 + (long long)p0 * tn : nullptr;
                if (stream) {
                    bulk_load_stream(stage, im, qbytes, &full[st]);
                    if (COMP == 0) bulk_load_stream(stage + L::kQ, re, qbytes, &full[st]);
                } else {
                    bulk_load(stage, im, qbytes, &full[st]);
                    if (COMP == 0) bulk_load(stage + L::kQ, re, qbytes, &full[st]);
                }
            }
            // the copies still in flight land before the warp leaves
            for (int k = max(cb, c - kNbStages); k < c; ++k)
                mbar_wait(&full[(k - cb) % kNbStages], (unsigned)(((k - cb) / kNbStages) & 1), kNbSpin);
        }
        return;
    }
    const int2 run = (lane < kFmmMaxNbr) ? __ldg(nq_run + (size_t)it * kFmmMaxNbr + lane) : make_int2(0, INT_MAX);
    df2 are[R], aim[R];
#pragma unroll
    for (int r = 0; r < R; ++r) are[r] = aim[r] = df2{f2(0.f), f2(0.f)};
    bool ok = true;
    for (int seg = cb; seg < ce; seg += kNbSegChunks) {
        const int se = min(ce, seg + kNbSegChunks);
        if (seg > cb) asm volatile("bar.sync 1, %0;" ::"r"(kFmmNT) : "memory");  // the last segment's x has been read
        const int q0 = 2 * kNbPairs * seg, q1 = 2 * kNbPairs * se;
        for (int base = q0 + 32 * wid; base < q1; base += kFmmNT) {
            const int q = base + lane;
            const int j = nq_source(run, min(q, S - 1));
            const int node = __ldg(a.perm + j);
#pragma unroll
            for (int r = 0; r < R; ++r) {  // 0 past the item's sources
                const df v = df_split_fast((q < S) ? ((r == 0) ? a.x0 : a.x1)[node] : 0.0);
                if (q < q1) s_x[r * kNbX + q - q0] = make_float2(v.h, v.l);
            }
        }
        asm volatile("bar.sync 1, %0;" ::"r"(kFmmNT) : "memory");
        for (int c = seg; ok && c < se; ++c) {
            const int u = c - cb, st = u % kNbStages;
            // one decision per warp: lanes that gave up alone would wait at the next barrier
            // for the others, and these for them
            if (!__all_sync(0xffffffffu, mbar_wait(&full[st], (unsigned)((u / kNbStages) & 1), kNbSpin))) {
                atomicExch(a.fault, 1);
                ok = false;
                break;
            }
            const float4* qi = nb_buf + (size_t)st * L::kStage;
            const float4* qr = qi + L::kQ;
            const float4* xv4 = reinterpret_cast<const float4*>(s_x) + (c - seg) * kNbPairs;
            const int np = min(kNbPairs, npair - c * kNbPairs);
            if (lane < tn) {
#pragma unroll
                for (int v = 0; v < kNbPairs / kFmmWarps; ++v) {
                    const int pp = wid + v * kFmmWarps;
                    if (pp >= np) break;
                    const float4 wi = qi[pp * tn + lane];
                    const df2 Qi{make_float2(wi.x, wi.y), make_float2(wi.z, wi.w)};
                    df2 Qr{f2(0.f), f2(0.f)};
                    if (COMP == 0) {
                        const float4 wr = qr[pp * tn + lane];
                        Qr = df2{make_float2(wr.x, wr.y), make_float2(wr.z, wr.w)};
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float4 x = xv4[r * (kNbX / 2) + pp];  // (hi, lo) of sources 2pp and 2pp + 1
                        const df2 xv{make_float2(x.x, x.z), make_float2(x.y, x.w)};
                        if (COMP == 0) df2_acc(are[r], df2_mul(xv, Qr));
                        df2_acc(aim[r], df2_mul(xv, Qi));
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[st]);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const df sr = df_add(df{are[r].h.x, are[r].l.x}, df{are[r].h.y, are[r].l.y});
        const df si = df_add(df{aim[r].h.x, aim[r].l.x}, df{aim[r].h.y, aim[r].l.y});
        s_z[wid][r][lane] = make_double2((double)sr.h + (double)sr.l, (double)si.h + (double)si.l);
    }
    asm volatile("bar.sync 1, %0;" ::"r"(kFmmNT) : "memory");  // the consumer warps only
    if (wid == 0 && lane < tn) {
        const int i = a.items[it].y + lane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            double2 v = s_z[0][r][lane];
            for (int w = 1; w < kFmmWarps; ++w) {
                v.x += s_z[w][r][lane].x;
                v.y += s_z[w][r][lane].y;
            }
            a.zn[((size_t)blockIdx.y * R + r) * a.N + i] = v;
        }
    }
}

// L2P by Horner's rule in double-float plus the near-field sum; one thread per
// node in sorted order (the nodes of a leaf are adjacent, so a warp reads the
// same coefficients).  Without the derivative the order-32 polynomial is four
// interleaved Horner chains of 8 coefficients joined by t^8 (a dependent chain
// of 13 steps instead of 31).  EPI: the operator epilogue of the product is applied at
// once (epilogue_apply: e.g. f_B(x) = 2x + diag(B1) x + (2/n) Im(A z)), so the
// sums z never go to memory; otherwise z is written in node order.  A cached
// near field (a.near_scaled) comes already multiplied by the epilogue's factor.
// EF: also F = -d/dz of the far field (Horner's rule carries the derivative)
// plus the near-field sums of w/d^2, written to outF.
template <int R, bool EF, bool EPI, int EK = EPI_Z>
__global__ void __launch_bounds__(256) fmm_l2p_kernel(FmmArgs a, ReduceArgs e) {
    if (a.done != nullptr && *a.done) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.N) return;
    const int box = a.node_box[i];
    double ir = 0.0;
    cdf t;
    if (EF || a.diff) {
        const double2 c = a.center[box];
        ir = recip_f64(a.width[box]);  // (GB300's FP64 division is a long dependent chain)
        const double2 p = a.ps[i];
        t = cdf{df_split_fast((p.x - c.x) * ir), df_split_fast((p.y - c.y) * ir)};
    } else {
        t = cdf_of(__ldg(a.tn + i));
    }
    const int node = a.perm[i];
    double zx[kMaxRHS] = {0.0, 0.0}, zy[kMaxRHS] = {0.0, 0.0};
    double2 near[kMaxRHS] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    cdf t8{};
    if (!EF) t8 = cdf_sq(cdf_sq(cdf_sq(t)));
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float4* b = a.loc + ((size_t)r * a.nbox + box) * kFmmP;
        cdf u, du = cdf_zero();
        if (EF) {  // Horner's rule, carrying the derivative
            u = cdf_of(b[kFmmP - 1]);
            for (int l = kFmmP - 2; l >= 0; --l) {
                du = cdf_add(cdf_mul(du, t), u);
                const cdf m = cdf_mul(u, t);
                const cdf bl = cdf_of(b[l]);
                u = cdf{df_add(m.re, bl.re), df_add(m.im, bl.im)};
            }
        } else {  // four interleaved Horner chains of 8 coefficients, joined by powers of t^8
            cdf h[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) h[q] = cdf_of(b[8 * q + 7]);
#pragma unroll
            for (int m = 6; m >= 0; --m)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const cdf mm = cdf_mul(h[q], t);
                    const cdf bl = cdf_of(b[8 * q + m]);
                    h[q] = cdf{df_add(mm.re, bl.re), df_add(mm.im, bl.im)};
                }
            u = h[3];
#pragma unroll
            for (int q = 2; q >= 0; --q) {
                const cdf mm = cdf_mul(u, t8);
                u = cdf{df_add(mm.re, h[q].re), df_add(mm.im, h[q].im)};
            }
        }
        double2 zn = a.zn[(size_t)r * a.N + i];
        for (int p = 1; p < a.nsplit; ++p) {  // the shares of a split near field
            const double2 v = a.zn[((size_t)p * R + r) * a.N + i];
            zn.x += v.x;
            zn.y += v.y;
        }
        zx[r] = (double)u.re.h + (double)u.re.l;
        zy[r] = (double)u.im.h + (double)u.im.l;
        if (EPI && a.near_scaled) {
            near[r] = zn;
        } else {
            zx[r] += zn.x;
            zy[r] += zn.y;
        }
        if (!EPI) a.out[(size_t)r * a.N + node] = make_double2(zx[r], zy[r]);
        if (EF) {
            const double2 zf = a.zf[(size_t)r * a.N + i];
            a.outF[(size_t)r * a.N + node] = make_double2(-ir * ((double)du.re.h + (double)du.re.l) + zf.x,
                                                          -ir * ((double)du.im.h + (double)du.im.l) + zf.y);
        }
    }
    if (EPI)
        epilogue_apply_as<true>(e, EK, node, make_double2(zx[0], zy[0]), make_double2(zx[1], zy[1]), near[0], near[1]);
}

// ---------------------------------------------------------------- host: tables
using cld = std::complex<long double>;

// a complex value as a double-float pair per part (hi = nearest float, lo = the rest)
float4 cdf_host(const cld& v) {
    const float rh = (float)v.real(), ih = (float)v.imag();
    return make_float4(rh, (float)(v.real() - (long double)rh), ih, (float)(v.imag() - (long double)ih));
}

// i^quarters v, or of its conjugate
float4 turned(float4 v, bool conj, int quarters) {
    if (conj) v = make_float4(v.x, v.y, -v.z, -v.w);
    switch (quarters & 3) {
        case 1: return make_float4(-v.z, -v.w, v.x, v.y);
        case 2: return make_float4(-v.x, -v.y, -v.z, -v.w);
        case 3: return make_float4(v.z, v.w, -v.x, -v.y);
        default: return v;
    }
}

// The M2L tables: the Pascal matrix C(k+l, l) as double-float pairs (P x P
// float2, in kFmmHSlots float4 slots), then per offset code (dx + 7) 15 + (dy + 7)
// the scalings (-1)^(k+1) delta^-(k+1) and delta^-l, delta = dx + i dy.
// After the L2L table: the scalings with their powers of two (m2lT) and the
// digits of C(k+l, l) 2^-(k+l), C(m, k) 2^-m and C(l, m) 2^-l as A fragments of
// m16n8k16 (m2lA).
// Binomial coefficients by Pascal's triangle and powers by repeated products
// in long double: no library power functions, whose long double forms are
// slow where long double is emulated in software.
constexpr int kFmmHSlots = kFmmP * kFmmP / 2;
constexpr int kFmmSSlots = kFmmOffs * kFmmOffs * 2 * kFmmP;
// then the L2L Pascal table C(l,m) at [l][m] (double-float, zero outside the
// triangle), kFmmHSlots float4 slots; kFmmSSlots of m2lT; then m2lA
constexpr int kFmmASlots = kTcD * 2 * 2 * 32;
constexpr int kFmmTOff = 2 * kFmmHSlots + kFmmSSlots, kFmmAOff = kFmmTOff + kFmmSSlots;

void translation_tables(std::vector<float4>* tab) {
    const int P = kFmmP, PP = 2 * kFmmP + 1;
    std::vector<long double> C((size_t)PP * PP, 0.0L);  // C[n][k], n < 2P + 1
    for (int n = 0; n < PP; ++n) {
        C[(size_t)n * PP] = 1.0L;
        for (int k = 1; k <= n; ++k) C[(size_t)n * PP + k] = C[(size_t)(n - 1) * PP + k - 1] + C[(size_t)(n - 1) * PP + k];
    }
    tab->assign(kFmmAOff + 3 * kFmmASlots, make_float4(0.f, 0.f, 0.f, 0.f));
    float* BU = reinterpret_cast<float*>(tab->data() + kFmmHSlots + kFmmSSlots);  // [l][m] = C(l, m)
    for (int r = 0; r < P; ++r)
        for (int c = 0; c < P; ++c) {
            const long double up = (r >= c) ? C[(size_t)r * PP + c] : 0.0L;  // C(l = r, m = c)
            BU[2 * (r * P + c)] = (float)up;
            BU[2 * (r * P + c) + 1] = (float)(up - (long double)(float)up);
        }
    float* H = reinterpret_cast<float*>(tab->data());  // [k][l] (hi, lo)
    for (int k = 0; k < P; ++k)
        for (int l = 0; l < P; ++l) {
            const long double v = C[(size_t)(k + l) * PP + l];
            const float hi = (float)v;
            H[2 * (k * P + l)] = hi;
            H[2 * (k * P + l) + 1] = (float)(v - (long double)hi);
        }
    // The powers for 0 <= dy <= dx; the other offsets are i^rot delta or its conjugate,
    // whose powers are these with parts exchanged and signs turned, the same bits.  (Long
    // double is software on AArch64: the tables took 2.0 ms of a process's first FMM call
    // with all 216 offsets formed one by one, 0.4 with these 33.)
    for (int dx = 2; dx <= kFmmOffMax; ++dx)
        for (int dy = 0; dy <= dx; ++dy) {
            const cld iz = 1.0L / cld((long double)dx, (long double)dy);
            float4 S[2 * kFmmP], T[2 * kFmmP];
            int ex[2 * kFmmP];       // the power of 1/delta in each entry
            long double two = 1.0L;  // 2^e
            cld pw(1.0L, 0.0L);  // delta^-e
            for (int e = 0; e <= P; ++e) {
                if (e < P) {  // delta^-l, l = e
                    S[P + e] = cdf_host(pw);
                    T[P + e] = cdf_host(pw * two);
                    ex[P + e] = e;
                }
                if (e >= 1) {  // k = e - 1: (-1)^(k+1) = (-1)^e
                    const cld v = (e % 2 == 1) ? -pw : pw;
                    S[e - 1] = cdf_host(v);
                    T[e - 1] = cdf_host(v * (0.5L * two));
                    ex[e - 1] = e;
                }
                pw *= iz;
                two *= 2.0L;
            }
            for (int image = 0; image < 8; ++image) {
                const int rot = image & 3, conj = image >> 2;
                int ix = dx, iy = conj ? -dy : dy;
                for (int r = 0; r < rot; ++r) {  // times i
                    const int t = ix;
                    ix = -iy;
                    iy = t;
                }
                const size_t o = (size_t)((ix + kFmmOffMax) * kFmmOffs + iy + kFmmOffMax) * 2 * P;
                for (int u = 0; u < 2 * P; ++u) {
                    tab->data()[kFmmHSlots + o + u] = turned(S[u], conj, -rot * ex[u]);
                    tab->data()[kFmmTOff + o + u] = turned(T[u], conj, -rot * ex[u]);
                }
            }
        }
    // digits of c 2^-sh (row, column): round(c 2^(49 - sh)) in balanced base 1024,
    // most significant first
    for (int w = 0; w < 3; ++w) {
        std::vector<int> dig((size_t)kTcD * P * P);
        for (int row = 0; row < P; ++row)
            for (int col = 0; col < P; ++col) {
                long double c;
                int sh;
                if (w == 0) {  // M2L: row l, column k
                    c = C[(size_t)(row + col) * PP + row];
                    sh = row + col;
                } else if (w == 1) {  // M2M: row m, column k
                    c = C[(size_t)row * PP + col];
                    sh = row;
                } else {  // L2L: row m, column l
                    c = C[(size_t)col * PP + row];
                    sh = col;
                }
                const unsigned __int128 u = (unsigned __int128)(unsigned long long)c << 50;
                long long v = (long long)(((u >> sh) + 1) >> 1);
                for (int i = kTcD - 1; i >= 0; --i) {
                    const int d = (i > 0) ? (int)((v + 512) & 1023) - 512 : (int)v;
                    dig[((size_t)i * P + row) * P + col] = d;
                    v = (v - d) / 1024;
                }
            }
        __half* F = reinterpret_cast<__half*>(tab->data() + kFmmAOff + (size_t)w * kFmmASlots);
        for (int i = 0; i < kTcD; ++i)
            for (int m = 0; m < 2; ++m)
                for (int kt = 0; kt < 2; ++kt)
                    for (int lane = 0; lane < 32; ++lane)
                        for (int u = 0; u < 8; ++u) {  // row g (+ 8 for odd registers), column 2t + (u & 1) (+ 8)
                            const int row = 16 * m + (lane >> 2) + 8 * ((u >> 1) & 1);
                            const int col = 16 * kt + 2 * (lane & 3) + (u & 1) + 8 * (u >> 2);
                            F[((((i * 2 + m) * 2 + kt) * 32) + lane) * 8 + u] =
                                __float2half((float)dig[((size_t)i * P + row) * P + col]);
                        }
    }
}

// Pinned host staging for the tree upload (grown on demand, kept for the process).
std::mutex g_stage_mutex;
void* g_stage = nullptr;
size_t g_stage_bytes = 0;

// The M2L tables depend only on P: formed once per process.
const std::vector<float4>& cached_tables() {
    static std::once_flag once;
    static std::vector<float4> tab;
    std::call_once(once, [] { translation_tables(&tab); });
    return tab;
}

// v = s[0] + s[1] + s[2] exactly (each float takes the next 24 bits of the
// double's 53; exact for |v| between 2^-80 and 2^120, which holds for
// boundary nodes in any sane unit)
void split3(double v, float* s) {
    s[0] = (float)v;
    const double r1 = v - (double)s[0];  // exact
    s[1] = (float)r1;
    s[2] = (float)(r1 - (double)s[1]);  // exact: at most 5 bits remain
}

uint32_t spread16(uint32_t v) {
    v &= 0xffffu;
    v = (v | (v << 8)) & 0x00ff00ffu;
    v = (v | (v << 4)) & 0x0f0f0f0fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

}  // namespace

// The streams and events of FMM handles, kept per device for reuse (at most
// kPoolKeep of each kind), so that a caller that builds and frees a handle
// every step creates none after the first.  A stream returns to the pool only
// after it has been synchronised.
constexpr size_t kPoolKeep = 64;

struct StreamPool {
    std::mutex mu;
    std::vector<std::vector<cudaStream_t>> hi, lo;  // per device: high-priority and normal streams
    std::vector<std::vector<cudaEvent_t>> ev;
};

static StreamPool& stream_pool() {
    static StreamPool* p = new StreamPool();  // never destroyed: the streams outlive static teardown
    return *p;
}

static int fmm_high_priority();

static cudaError_t take_stream(bool high, cudaStream_t* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    StreamPool& P = stream_pool();
    {
        std::lock_guard<std::mutex> lock(P.mu);
        std::vector<std::vector<cudaStream_t>>& v = high ? P.hi : P.lo;
        if ((int)v.size() > dev && !v[dev].empty()) {
            *out = v[dev].back();
            v[dev].pop_back();
            return cudaSuccess;
        }
    }
    return high ? cudaStreamCreateWithPriority(out, cudaStreamNonBlocking, fmm_high_priority())
                : cudaStreamCreateWithFlags(out, cudaStreamNonBlocking);
}

static cudaError_t take_event(cudaEvent_t* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    StreamPool& P = stream_pool();
    {
        std::lock_guard<std::mutex> lock(P.mu);
        if ((int)P.ev.size() > dev && !P.ev[dev].empty()) {
            *out = P.ev[dev].back();
            P.ev[dev].pop_back();
            return cudaSuccess;
        }
    }
    return cudaEventCreateWithFlags(out, cudaEventDisableTiming);
}

static void give_stream(bool high, cudaStream_t s, int dev) {
    if (!s) return;
    cudaStreamSynchronize(s);
    StreamPool& P = stream_pool();
    std::lock_guard<std::mutex> lock(P.mu);
    std::vector<std::vector<cudaStream_t>>& v = high ? P.hi : P.lo;
    if ((int)v.size() <= dev) v.resize(dev + 1);
    if (v[dev].size() < kPoolKeep)
        v[dev].push_back(s);
    else
        cudaStreamDestroy(s);
}

static void give_event(cudaEvent_t e, int dev) {
    if (!e) return;
    StreamPool& P = stream_pool();
    std::lock_guard<std::mutex> lock(P.mu);
    if ((int)P.ev.size() <= dev) P.ev.resize(dev + 1);
    if (P.ev[dev].size() < kPoolKeep)
        P.ev[dev].push_back(e);
    else
        cudaEventDestroy(e);
}

void release_fmm(Boundary& b) {
    if (b.fmm) {
        give_stream(true, b.fmm->aux, b.device);
        give_event(b.fmm->ev_fork, b.device);
        give_event(b.fmm->ev_join, b.device);
        give_event(b.fmm->ev_solve, b.device);
        give_stream(false, b.fmm->bst, b.device);
        give_stream(false, b.fmm->nst, b.device);
        give_event(b.fmm->ev_nq, b.device);

        if (b.fmm->arena || b.fmm->sync || b.fmm->nq_item || b.fmm->tn || b.fmm->path || b.fmm->fault) {  // once no stream uses them
            cudaDeviceSynchronize();
            cudaGetLastError();
            pool_free(b.fmm->arena, 0);
            pool_free(b.fmm->sync, 0);
            pool_free(b.fmm->nq_cnt, 0);
            pool_free(b.fmm->nq_off, 0);
            pool_free(b.fmm->nq_item, 0);
            pool_free(b.fmm->nq_run, 0);
            pool_free(b.fmm->nq_re, 0);
            pool_free(b.fmm->nq_im, 0);
            pool_free(b.fmm->nt_im, 0);
            pool_free(b.fmm->inv_off, 0);
            pool_free(b.fmm->inv_r, 0);
            pool_free(b.fmm->inv_i, 0);
            pool_free(b.fmm->fault, 0);
            pool_free(b.fmm->tn, 0);
            pool_free(b.fmm->path, 0);
        }
        delete b.fmm;
        b.fmm = nullptr;
    }
}

// Builds the tree of the handle's nodes (once) with workspace for R right-hand sides.
// The host-side tree builder (used when the tree is too deep for the device
// builder's lookup grids): fills t and its device arena.
static int fmm_tree_host(const Boundary& b, FmmTree* t, cudaStream_t st) {
    const int N = b.N;
    std::vector<double2> et(N);
    GNK_TRY_CUDA(cudaMemcpyAsync(et.data(), b.et, (size_t)N * sizeof(double2), cudaMemcpyDeviceToHost, st));
    GNK_TRY_CUDA(cudaStreamSynchronize(st));
    double xmin = et[0].x, xmax = et[0].x, ymin = et[0].y, ymax = et[0].y;
    for (const double2& p : et) {
        xmin = std::min(xmin, p.x);
        xmax = std::max(xmax, p.x);
        ymin = std::min(ymin, p.y);
        ymax = std::max(ymax, p.y);
    }
    const double W = std::max(std::max(xmax - xmin, ymax - ymin) * (1.0 + 1e-9), 1e-300);
    const double x0 = 0.5 * (xmin + xmax) - 0.5 * W, y0 = 0.5 * (ymin + ymax) - 0.5 * W;
    std::vector<uint32_t> key0(N), key1(N);
    std::vector<int> ord0(N), ord1(N);
    for (int i = 0; i < N; ++i) {
        const double fx = (et[i].x - x0) / W * 65536.0, fy = (et[i].y - y0) / W * 65536.0;
        const uint32_t ix = (uint32_t)std::min(65535.0, std::max(0.0, std::floor(fx)));
        const uint32_t iy = (uint32_t)std::min(65535.0, std::max(0.0, std::floor(fy)));
        key0[i] = (spread16(ix) << 1) | spread16(iy);
        ord0[i] = i;
    }
    // LSD radix sort, four stable passes of 8 bits: (key, node) in increasing order
    for (int pass = 0; pass < 4; ++pass) {
        const int sh = 8 * pass;
        int cnt[257] = {0};
        for (int i = 0; i < N; ++i) ++cnt[((key0[i] >> sh) & 0xffu) + 1];
        for (int d = 0; d < 256; ++d) cnt[d + 1] += cnt[d];
        for (int i = 0; i < N; ++i) {
            const int dst = cnt[(key0[i] >> sh) & 0xffu]++;
            key1[dst] = key0[i];
            ord1[dst] = ord0[i];
        }
        key0.swap(key1);
        ord0.swap(ord1);
    }
    auto key_at = [&](int i, int l) { return key0[i] >> (2 * (16 - l)); };
    // leaf level: deepest level whose non-empty boxes hold enough nodes on
    // average (fmm_level_wanted).  Neighbours in key order first differ at level 16 - msb(x)/2.
    std::vector<long long> first_diff(18, 0);
    for (int i = 1; i < N; ++i) {
        const uint32_t x = key0[i] ^ key0[i - 1];
        if (x == 0) continue;
        const int msb = 31 - __builtin_clz(x);
        ++first_diff[16 - msb / 2];  // distinct from this level down
    }
    int L = 2;
    long long distinct = 1;
    double prev = 0.0;  // nodes per box one level up
    for (int l = 1; l <= 16; ++l) {
        distinct += first_diff[l];
        const double mean = (double)N / (double)distinct, above = prev;
        prev = mean;
        if (l < 3) continue;
        if (!fmm_level_wanted(b, l, mean, above)) break;
        L = l;
    }
    t->L = L;
    const int l0 = fmm_top_level(b, L);
    t->l0 = l0;
    // boxes per level (level index l - l0), sorted by key
    const int nlev = L - l0 + 1;
    std::vector<std::vector<uint32_t>> keys(nlev);
    std::vector<int> leaf_start;
    for (int i = 0; i < N; ++i) {
        const uint32_t k = key_at(i, L);
        if (i == 0 || k != keys[L - l0].back()) {
            keys[L - l0].push_back(k);
            leaf_start.push_back(i);
        }
    }
    leaf_start.push_back(N);
    for (int l = L - 1; l >= l0; --l)
        for (uint32_t k : keys[l + 1 - l0]) {  // the boxes of level l + 1
            const uint32_t pk = k >> 2;
            if (keys[l - l0].empty() || keys[l - l0].back() != pk) keys[l - l0].push_back(pk);
        }
    t->lvl_off.resize(nlev);
    t->lvl_cnt.resize(nlev);
    int nbox = 0;
    for (int l = l0; l <= L; ++l) {
        t->lvl_off[l - l0] = nbox;
        t->lvl_cnt[l - l0] = (int)keys[l - l0].size();
        nbox += (int)keys[l - l0].size();
    }
    t->nbox = nbox;
    t->nleaf = (int)keys[L - l0].size();
    auto compact = [](uint32_t v) {  // inverse of spread16
        v &= 0x55555555u;
        v = (v | (v >> 1)) & 0x33333333u;
        v = (v | (v >> 2)) & 0x0f0f0f0fu;
        v = (v | (v >> 4)) & 0x00ff00ffu;
        v = (v | (v >> 8)) & 0x0000ffffu;
        return v;
    };
    auto decode = [&](uint32_t key, int* ix, int* iy) {
        *ix = (int)compact(key >> 1);
        *iy = (int)compact(key);
    };
    // box geometry, parents and children: children of a box are contiguous in
    // key order, so one pass over each level links it to the level above
    std::vector<int> bix(nbox), biy(nbox);
    for (int l = l0; l <= L; ++l)
        for (int q = 0; q < t->lvl_cnt[l - l0]; ++q) decode(keys[l - l0][q], &bix[t->lvl_off[l - l0] + q],
                                                           &biy[t->lvl_off[l - l0] + q]);
    std::vector<double2> center(nbox);
    std::vector<double> width(nbox);
    std::vector<int> child_start(nbox, -1), child_count(nbox, 0), parent(nbox, -1), quad(nbox, 0);
    for (int l = l0; l <= L; ++l) {
        const double r = W / (double)(1 << l);
        for (int q = 0; q < t->lvl_cnt[l - l0]; ++q) {
            const int g = t->lvl_off[l - l0] + q;
            center[g] = make_double2(x0 + (bix[g] + 0.5) * r, y0 + (biy[g] + 0.5) * r);
            width[g] = r;
            quad[g] = ((bix[g] & 1) << 1) | (biy[g] & 1);
        }
        if (l == l0) continue;
        int pq = -1;
        uint32_t last = 0;
        for (int q = 0; q < t->lvl_cnt[l - l0]; ++q) {
            const uint32_t pk = keys[l - l0][q] >> 2;
            if (pq < 0 || pk != last) {
                ++pq;
                last = pk;
            }
            const int g = t->lvl_off[l - l0] + q, pg = t->lvl_off[l - 1 - l0] + pq;
            parent[g] = pg;
            if (child_start[pg] < 0) child_start[pg] = g;
            ++child_count[pg];
        }
    }
    // neighbour lists (adjacent boxes of the same level, the box itself included)
    // and interaction lists, level by level from the children of the parent's
    // neighbours; the topmost level compares all pairs
    std::vector<int> nb_start(nbox + 1, 0), nb;
    std::vector<int> il_start(nbox + 1, 0), il_src, il_off;
    nb.reserve((size_t)nbox * 6);
    il_src.reserve((size_t)nbox * 16);
    il_off.reserve((size_t)nbox * 16);
    auto visit = [&](int g, int c) {
        const int dx = bix[c] - bix[g], dy = biy[c] - biy[g];
        if (std::abs(dx) <= 1 && std::abs(dy) <= 1) {
            nb.push_back(c);
        } else {
            il_src.push_back(c);
            il_off.push_back((dx + kFmmOffMax) * kFmmOffs + dy + kFmmOffMax);
        }
    };
    for (int l = l0; l <= L; ++l)
        for (int q = 0; q < t->lvl_cnt[l - l0]; ++q) {
            const int g = t->lvl_off[l - l0] + q;
            if (l == l0) {
                for (int c = t->lvl_off[0]; c < t->lvl_off[0] + t->lvl_cnt[0]; ++c) visit(g, c);
            } else {
                const int pg = parent[g];
                for (int e = nb_start[pg]; e < nb_start[pg + 1]; ++e) {
                    const int qn = nb[e];
                    for (int c = child_start[qn]; c < child_start[qn] + child_count[qn]; ++c) visit(g, c);
                }
            }
            nb_start[g + 1] = (int)nb.size();
            il_start[g + 1] = (int)il_src.size();
        }
    // neighbour leaves of each leaf (the leaf itself included)
    std::vector<int> nl_start(t->nleaf + 1, 0), nl_leaf, leaf_box(t->nleaf);
    long long near_pairs = 0;
    const int loff = t->lvl_off[L - l0];
    for (int q = 0; q < t->nleaf; ++q) {
        leaf_box[q] = loff + q;
        const long long cnt_t = leaf_start[q + 1] - leaf_start[q];
        for (int e = nb_start[loff + q]; e < nb_start[loff + q + 1]; ++e) {
            const int lq = nb[e] - loff;
            nl_leaf.push_back(lq);
            near_pairs += cnt_t * (leaf_start[lq + 1] - leaf_start[lq]);
        }
        nl_start[q + 1] = (int)nl_leaf.size();
    }
    t->near_pairs = near_pairs;
    // near-field work items: chunks of 32 targets of a leaf, largest leaves first
    std::vector<int2> items;
    for (int q = 0; q < t->nleaf; ++q)
        for (int i = leaf_start[q]; i < leaf_start[q + 1]; i += 32) items.push_back(make_int2(q, i));
    std::stable_sort(items.begin(), items.end(), [&](const int2& u, const int2& v) {
        return (nl_start[u.x + 1] - nl_start[u.x]) > (nl_start[v.x + 1] - nl_start[v.x]);
    });
    t->nitems = (int)items.size();
    t->m2l_pairs = (long long)il_src.size();
    long long m2m_pairs = 0;
    for (int g = 0; g < nbox; ++g) m2m_pairs += child_count[g];
    t->m2m_pairs = m2m_pairs;
    const std::vector<int>& perm = ord0;
    std::vector<double2> ps(N);
    for (int i = 0; i < N; ++i) ps[i] = et[perm[i]];

    // one device allocation for the tree and the expansions
    const size_t P = kFmmP;
    struct Part {
        void** p;
        size_t bytes;
    };
    const size_t nil = std::max<size_t>(il_src.size(), 1), nnl = std::max<size_t>(nl_leaf.size(), 1);
    Part parts[] = {
        {(void**)&t->perm, N * sizeof(int)},
        {(void**)&t->ps, N * sizeof(double2)},
        {(void**)&t->p3, N * sizeof(float4)},
        {(void**)&t->p3b, N * sizeof(float2)},
        {(void**)&t->leaf_start, (t->nleaf + 1) * sizeof(int)},
        {(void**)&t->leaf_box, t->nleaf * sizeof(int)},
        {(void**)&t->center, nbox * sizeof(double2)},
        {(void**)&t->width, nbox * sizeof(double)},
        {(void**)&t->child_start, nbox * sizeof(int)},
        {(void**)&t->child_count, nbox * sizeof(int)},
        {(void**)&t->parent, nbox * sizeof(int)},
        {(void**)&t->quad, nbox * sizeof(int)},
        {(void**)&t->il_start, (nbox + 1) * sizeof(int)},
        {(void**)&t->il_src, nil * sizeof(int)},
        {(void**)&t->il_off, nil * sizeof(int)},
        {(void**)&t->nl_start, (t->nleaf + 1) * sizeof(int)},
        {(void**)&t->nl_leaf, nnl * sizeof(int)},
        {(void**)&t->items, std::max<size_t>(items.size(), 1) * sizeof(int2)},
        {(void**)&t->node_box, N * sizeof(int)},
        {(void**)&t->mult, (size_t)t->R * nbox * P * sizeof(float4)},
        {(void**)&t->loc, (size_t)t->R * nbox * P * sizeof(float4)},
        {(void**)&t->ws, (size_t)t->R * N * sizeof(float4)},
        {(void**)&t->zn, (size_t)fmm_near_splits(b, t->nitems) * t->R * N * sizeof(double2)},
        {(void**)&t->zf, (size_t)t->R * N * sizeof(double2)},
    };
    size_t total = 0;
    for (const Part& p : parts) total += (p.bytes + 255) / 256 * 256;
    if (pool_alloc(&t->arena, total, st) != cudaSuccess) {
        cudaGetLastError();
        t->arena = nullptr;
        set_error("FMM tree: device allocation of %zu bytes failed", total);
        return GNK_ENOMEM;
    }
    char* cur = static_cast<char*>(t->arena);
    for (const Part& p : parts) {
        *p.p = cur;
        cur += (p.bytes + 255) / 256 * 256;
    }
    // everything but the expansions goes up in one copy, staged in a pinned
    // host buffer laid out like the device arena
    const size_t upload = (size_t)((char*)t->mult - (char*)t->arena);
    std::lock_guard<std::mutex> lock(g_stage_mutex);
    if (g_stage_bytes < upload) {
        if (g_stage) cudaFreeHost(g_stage);
        g_stage = nullptr;
        g_stage_bytes = 0;
        if (cudaHostAlloc(&g_stage, upload, cudaHostAllocDefault) != cudaSuccess) {
            cudaGetLastError();
            g_stage = nullptr;
            set_error("FMM tree: pinned staging allocation of %zu bytes failed", upload);
            return GNK_ENOMEM;
        }
        g_stage_bytes = upload;
    }
    char* hb = static_cast<char*>(g_stage);
    auto put = [&](const void* dst, const void* src, size_t bytes) {
        if (bytes) std::memcpy(hb + ((const char*)dst - (const char*)t->arena), src, bytes);
    };
    put(t->perm, perm.data(), N * sizeof(int));
    put(t->ps, ps.data(), N * sizeof(double2));
    float4* p3 = reinterpret_cast<float4*>(hb + ((char*)t->p3 - (char*)t->arena));
    float2* p3b = reinterpret_cast<float2*>(hb + ((char*)t->p3b - (char*)t->arena));
    for (int i = 0; i < N; ++i) {
        float sx[3], sy[3];
        split3(ps[i].x, sx);
        split3(ps[i].y, sy);
        p3[i] = make_float4(sx[0], sx[1], sx[2], sy[0]);
        p3b[i] = make_float2(sy[1], sy[2]);
    }
    put(t->leaf_start, leaf_start.data(), leaf_start.size() * sizeof(int));
    put(t->leaf_box, leaf_box.data(), leaf_box.size() * sizeof(int));
    put(t->center, center.data(), nbox * sizeof(double2));
    put(t->width, width.data(), nbox * sizeof(double));
    put(t->child_start, child_start.data(), nbox * sizeof(int));
    put(t->child_count, child_count.data(), nbox * sizeof(int));
    put(t->parent, parent.data(), nbox * sizeof(int));
    put(t->quad, quad.data(), nbox * sizeof(int));
    put(t->il_start, il_start.data(), il_start.size() * sizeof(int));
    put(t->il_src, il_src.data(), il_src.size() * sizeof(int));
    put(t->il_off, il_off.data(), il_off.size() * sizeof(int));
    put(t->nl_start, nl_start.data(), nl_start.size() * sizeof(int));
    put(t->nl_leaf, nl_leaf.data(), nl_leaf.size() * sizeof(int));
    put(t->items, items.data(), items.size() * sizeof(int2));
    int* nbx = reinterpret_cast<int*>(hb + ((char*)t->node_box - (char*)t->arena));
    for (int q = 0; q < t->nleaf; ++q)
        for (int i = leaf_start[q]; i < leaf_start[q + 1]; ++i) nbx[i] = leaf_box[q];
    // the staging buffer is reused by the next build: finish the copy first
    cudaError_t e = cudaMemcpyAsync(t->arena, hb, upload, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("FMM tree upload failed: %s", cudaGetErrorString(e));
        return GNK_ECUDA;
    }
    return GNK_OK;
}

int fmm_device_tables(FmmTree* t, cudaStream_t st) {
    static std::mutex mu;
    static std::vector<float4*> per_device;  // indexed by device, never freed
    int dev = 0;
    GNK_TRY_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if ((int)per_device.size() <= dev) per_device.resize(dev + 1, nullptr);
    if (!per_device[dev]) {
        const std::vector<float4>& c = cached_tables();
        float4* d = nullptr;
        if (cudaMalloc(&d, c.size() * sizeof(float4)) != cudaSuccess) {
            cudaGetLastError();
            set_error("FMM: device allocation of the M2L tables failed");
            return GNK_ENOMEM;
        }
        cudaError_t e = cudaMemcpyAsync(d, c.data(), c.size() * sizeof(float4), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            cudaGetLastError();
            cudaFree(d);
            set_error("FMM: upload of the M2L tables failed");
            return GNK_ECUDA;
        }
        per_device[dev] = d;
    }
    t->m2lH = reinterpret_cast<const float2*>(per_device[dev]);
    t->m2lS = per_device[dev] + kFmmHSlots;
    t->bUp = reinterpret_cast<const float2*>(per_device[dev] + kFmmHSlots + kFmmSSlots);
    t->m2lT = per_device[dev] + kFmmTOff;
    t->m2lA = reinterpret_cast<const uint4*>(per_device[dev] + kFmmAOff);
    return GNK_OK;
}

// The highest stream priority of the device (the far-field chain's stream).
static int fmm_high_priority() {
    int least = 0, greatest = 0;
    if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return greatest;
}

static void fmm_args(const Boundary& b, FmmArgs& a);

// Builds the tree of the handle's nodes (once) with workspace for kMaxRHS
// right-hand sides: on the device when the lookup grids fit, else on the host.
int ensure_fmm(const Boundary& bc, int R, cudaStream_t st) {
    Boundary& b = const_cast<Boundary&>(bc);
    (void)R;
    if (b.fmm) return GNK_OK;
    FmmTree* t = new (std::nothrow) FmmTree();
    if (!t) {
        set_error("host allocation failed");
        return GNK_ENOMEM;
    }
    t->R = kMaxRHS;
    int rc = fmm_tree_device(b, t, st);
    if (rc == kFmmUseHost) rc = fmm_tree_host(b, t, st);
    if (rc == GNK_OK) rc = fmm_device_tables(t, st);
    if (rc == GNK_OK) {  // the upward pass's child counts, all zero
        const size_t nsync = (size_t)t->nbox;
        if (pool_alloc(reinterpret_cast<void**>(&t->sync), nsync * sizeof(int), st) != cudaSuccess ||
            cudaMemsetAsync(t->sync, 0, nsync * sizeof(int), st) != cudaSuccess ||
            pool_alloc(reinterpret_cast<void**>(&t->fault), sizeof(int), st) != cudaSuccess ||
            cudaMemsetAsync(t->fault, 0, sizeof(int), st) != cudaSuccess) {
            cudaGetLastError();
            set_error("FMM: allocation of the pass counters failed");
            rc = GNK_ENOMEM;
        }
    }
    if (rc == GNK_OK && pool_alloc(reinterpret_cast<void**>(&t->tn), (size_t)b.N * sizeof(float4), st) != cudaSuccess) {
        cudaGetLastError();
        set_error("FMM: allocation of the node offsets failed");
        rc = GNK_ENOMEM;
    }
    if (rc == GNK_OK &&
        pool_alloc(reinterpret_cast<void**>(&t->path), (size_t)t->nleaf * (t->L - t->l0 + 1) * sizeof(unsigned), st) !=
            cudaSuccess) {
        cudaGetLastError();
        set_error("FMM: allocation of the leaves' paths failed");
        rc = GNK_ENOMEM;
    }
    if (rc == GNK_OK) {
        FmmArgs a;
        b.fmm = t;
        fmm_args(b, a);
        fmm_tn_build_kernel<<<(b.N + 255) / 256, 256, 0, st>>>(a, t->tn);
        fmm_path_kernel<<<(t->nleaf + 127) / 128, 128, 0, st>>>(a, t->path);
        count_launches(2);
        if (cudaGetLastError() != cudaSuccess) {
            set_error("FMM: launch of the node offsets failed");
            rc = GNK_ECUDA;
        }
    }
    cudaGetLastError();
    if (rc == GNK_OK &&
        (take_stream(true, &t->aux) != cudaSuccess || take_stream(false, &t->nst) != cudaSuccess || take_event(&t->ev_fork) != cudaSuccess ||
         take_event(&t->ev_join) != cudaSuccess || take_event(&t->ev_solve) != cudaSuccess)) {
        cudaGetLastError();
        set_error("FMM: stream or event creation failed");
        rc = GNK_ECUDA;
    }
    b.fmm = t;  // owned by the handle from here on (freed by release_fmm)
    if (rc != GNK_OK) release_fmm(b);
    return rc;
}

// FP32-pipe instructions of one FMM product, for the roofline.  Translations on the
// tensor cores, per lane and tile of four pairs: 400 for tc_transform (184 for the
// digits, 216 for the sums), and around it 344 for M2L, 416 for M2M (one tile per box
// with children), 328 for L2L (one per four leaves and level).  In double-float
// (handles built for differentiation), per lane and pair: M2L 32 (2 Dekker products
// and 2 compensated sums, 24) for the real Pascal matrix, the two complex scalings (38
// each) and the sum (22); 840 for an L2L transform (32 terms of the Pascal sum at 24
// each, two exact scalings at 30 and two double-float additions), 742 for an M2M (31
// passes of a double-float complex addition, 22 each, and the two scalings).  P2M: 35
// complex products a node (38 each) and 16 per order for the sums (a handle built
// for differentiation 38 per order for the powers and 48 for the sums); L2P: 58 R per
// node and order (a complex product and sum), twice that with the derivative.
// which = 0: M2L; 1: the upward pass (P2M and the M2M climb); 2: L2L; 3: L2P;
// 4: L2P with the derivative.  (The near field: fmm_near_instr.)
double fmm_instr(const Boundary& b, int R, int which) {
    const FmmTree* t = b.fmm;
    if (!t) return 0.0;
    const double P = kFmmP, levels = t->L - t->l0;
    switch (which) {
        case 0: return R * (double)t->m2l_pairs * (b.diff ? (24.0 * P + 98.0) * P : 744.0 * 32.0 / 4.0);
        case 1:
            if (b.diff) return R * 742.0 * P * (double)t->m2m_pairs + (double)b.N * (38.0 + 48.0 * R) * P;
            return R * (816.0 * 32.0 * (double)(t->nbox - t->nleaf) + (double)b.N * (38.0 * 35.0 + 16.0 * P));
        case 2:
            return R * levels * (b.diff ? 840.0 * P * (double)t->nleaf : 728.0 * 32.0 * (double)((t->nleaf + 3) / 4));
        default: return R * (double)b.N * P * 58.0 * (which == 4 ? 2.0 : 1.0);
    }
}

double fmm_near_instr(const Boundary& b, int R) {
    return b.fmm ? (49.0 + 48.0 * R) * (double)b.fmm->near_pairs : 0.0;
}

// The cached near field per pair and right-hand side: a double-float product
// (4) and a compensated accumulation (8) per part of z; bytes: the cached
// entries read (8 per part and pair).
double fmm_near_cached_instr(const Boundary& b, int R, int comp) {
    return b.fmm ? 12.0 * R * (comp == 1 ? 1.0 : 2.0) * (double)b.fmm->near_pairs : 0.0;
}

double fmm_near_cached_bytes(const Boundary& b, int R, int comp) {
    // 8 bytes per near pair and part of z read from the cache, x in (8 bytes per
    // node) and z out (16 bytes per node) per right-hand side
    return b.fmm ? 8.0 * (double)b.fmm->near_pairs * (comp == 1 ? 1.0 : 2.0) + 24.0 * R * b.N : 0.0;
}

const int* fmm_fault_word(const Boundary& b) {
    return b.fmm ? b.fmm->fault : nullptr;
}

// The near-field operator caches of a handle, each formed once: allocated here
// (state 2), formed by near_cache_build on the first product that reads it;
// state -1 when it would exceed kNqMaxBytes or its allocation fails (the
// products then compute the near field directly).  `adj`: the cache of the
// solves with weights A x (imaginary part only), else that of the products with
// weights q x.
constexpr double kNqMaxBytes = 16.0 * (1 << 30);

static int ensure_near_cache(const Boundary& b, bool adj, cudaStream_t st) {
    FmmTree* t = b.fmm;
    int& state = adj ? t->nt_state : t->nq_state;
    if (state != 0) return GNK_OK;
    state = -1;
    if (t->nitems <= 0) return GNK_OK;
    // sizes from bounds the tree already gives, so that nothing waits for the
    // device: sum_items ceil(S/2) tn <= (near pairs + N)/2 entries
    const size_t ni = (size_t)t->nitems;
    const long long slots = (t->near_pairs + b.N) / 2 + 1;
    const size_t bytes = (size_t)slots * sizeof(float4);
    if (2.0 * (double)bytes > kNqMaxBytes) return GNK_OK;
    if (t->near_shape == 0) {
        if (pool_alloc(reinterpret_cast<void**>(&t->nq_cnt), ni * sizeof(long long), st) != cudaSuccess ||
            pool_alloc(reinterpret_cast<void**>(&t->nq_off), (ni + 1) * sizeof(long long), st) != cudaSuccess ||
            pool_alloc(reinterpret_cast<void**>(&t->nq_item), ni * sizeof(int2), st) != cudaSuccess ||
            pool_alloc(reinterpret_cast<void**>(&t->nq_run), ni * kFmmMaxNbr * sizeof(int2), st) != cudaSuccess) {
            cudaGetLastError();
            pool_free(t->nq_cnt, st);
            pool_free(t->nq_off, st);
            pool_free(t->nq_item, st);
            pool_free(t->nq_run, st);
            t->nq_cnt = nullptr;
            t->nq_off = nullptr;
            t->nq_item = nullptr;
            t->nq_run = nullptr;
            return GNK_OK;
        }
        t->near_shape = 1;
        t->nq_slots = slots;
    }
    float4** part[2] = {adj ? &t->nt_im : &t->nq_im, adj ? nullptr : &t->nq_re};
    for (float4** p : part) {
        if (p && pool_alloc(reinterpret_cast<void**>(p), bytes, st) != cudaSuccess) {
            cudaGetLastError();
            *p = nullptr;
            if (p == part[1]) {
                pool_free(*part[0], st);
                *part[0] = nullptr;
            }
            return GNK_OK;
        }
    }
    state = 2;
    return GNK_OK;
}

// The launches that form a cache (the items' shapes once, then the entries), on
// `st` after the product has forked its far field, so that they overlap it.
static int near_cache_build(const Boundary& b, bool adj, cudaStream_t st) {
    FmmTree* t = b.fmm;
    int& state = adj ? t->nt_state : t->nq_state;
    if (state != 2) return GNK_OK;
    FmmArgs a;
    fmm_args(b, a);
    if (t->near_shape == 1) {
        fmm_nq_shape_kernel<<<(t->nitems + 255) / 256, 256, 0, st>>>(a, t->nq_cnt, t->nq_item, t->nq_run);
        fmm_nq_scan_kernel<<<1, 1024, 0, st>>>(t->nq_cnt, t->nitems, t->nq_off);
        GNK_TRY_CUDA(cudaGetLastError());
        count_launches(2);
        pool_free(t->nq_cnt, st);
        t->nq_cnt = nullptr;
        t->near_shape = 2;
    } else if (t->nq_wait) {  // the shapes are being formed on the stream of the other cache
        GNK_TRY_CUDA(cudaStreamWaitEvent(st, t->ev_nq, 0));
    }
    const ProfToken tok = prof_begin(st, PK_OTHER);
    if (adj)
        fmm_nq_build_kernel<false, true><<<t->nitems, kFmmNT, 0, st>>>(a, b.A, b.q, t->nq_off, t->nq_item,
                                                                       t->nq_run, nullptr, t->nt_im);
    else if (b.A_real)
        fmm_nq_build_kernel<true, false><<<t->nitems, kFmmNT, 0, st>>>(a, b.q, b.A, t->nq_off, t->nq_item,
                                                                       t->nq_run, t->nq_re, t->nq_im);
    else
        fmm_nq_build_kernel<true, true><<<t->nitems, kFmmNT, 0, st>>>(a, b.q, b.A, t->nq_off, t->nq_item,
                                                                      t->nq_run, t->nq_re, t->nq_im);
    GNK_TRY_CUDA(cudaGetLastError());
    prof_end(tok, PK_OTHER, 0.0, st);
    count_launches(1);
    state = 1;
    return GNK_OK;
}

// The inverse cache of a handle built for differentiation: 1/(eta_i - eta_j) of
// every near pair (16 bytes), for the products with weights A x of its solves,
// whose sums must stay bit for bit those of the direct near field.  Formed by the
// first of them; a product then reads it instead of spending 49 of 97
// instructions per pair on 1/d beside the far field on the same pipe: a forward
// and a transposed solve at N = 40,960 with the gradient's E, F passes 13.3 -> 11.9 ms.
static int ensure_inverse_cache(const Boundary& b, cudaStream_t st) {
    FmmTree* t = b.fmm;
    if (t->inv_state != 0) return GNK_OK;
    t->inv_state = -1;
    if (t->nitems <= 0) return GNK_OK;
    // each of an item's kFmmWarps shares rounds up to whole entries
    const long long slots = t->near_pairs / 2 + (long long)(kFmmWarps / 2) * b.N + 1;
    const size_t ni = (size_t)t->nitems, bytes = (size_t)slots * sizeof(float4);
    if (2.0 * (double)bytes > kNqMaxBytes) return GNK_OK;
    long long* cnt = nullptr;
    if (pool_alloc(reinterpret_cast<void**>(&cnt), ni * sizeof(long long), st) != cudaSuccess ||
        pool_alloc(reinterpret_cast<void**>(&t->inv_off), (ni + 1) * sizeof(long long), st) != cudaSuccess ||
        pool_alloc(reinterpret_cast<void**>(&t->inv_r), bytes, st) != cudaSuccess ||
        pool_alloc(reinterpret_cast<void**>(&t->inv_i), bytes, st) != cudaSuccess) {
        cudaGetLastError();
        pool_free(cnt, st);
        pool_free(t->inv_off, st);
        pool_free(t->inv_r, st);
        t->inv_off = nullptr;
        t->inv_r = t->inv_i = nullptr;
        return GNK_OK;
    }
    FmmArgs a;
    fmm_args(b, a);
    fmm_inv_count_kernel<<<(t->nitems + 255) / 256, 256, 0, st>>>(a, cnt);
    fmm_nq_scan_kernel<<<1, 1024, 0, st>>>(cnt, t->nitems, t->inv_off);
    fmm_near_kernel<1, false, 1><<<t->nitems, kFmmNT, 0, st>>>(a);
    GNK_TRY_CUDA(cudaGetLastError());
    count_launches(3);
    pool_free(cnt, st);
    t->inv_state = 1;
    return GNK_OK;
}

// L2P with the product's epilogue, one instantiation per epilogue kind (the
// kind known at compile time: only its case is compiled in).
template <int R, int EK>
static void l2p_epi_launch(const FmmArgs& a, const ReduceArgs& e, int nb, cudaStream_t st) {
    fmm_l2p_kernel<R, false, true, EK><<<nb, 256, 0, st>>>(a, e);
}

template <int R>
static int l2p_epi(const FmmArgs& a, const ReduceArgs& e, int nb, cudaStream_t st) {
    switch (e.job.epi) {
        case EPI_Z: l2p_epi_launch<R, EPI_Z>(a, e, nb, st); break;
        case EPI_IMINUSN: l2p_epi_launch<R, EPI_IMINUSN>(a, e, nb, st); break;
        case EPI_M: l2p_epi_launch<R, EPI_M>(a, e, nb, st); break;
        case EPI_ADJ: l2p_epi_launch<R, EPI_ADJ>(a, e, nb, st); break;
        case EPI_RESID: l2p_epi_launch<R, EPI_RESID>(a, e, nb, st); break;
        case EPI_RESID_ADJ: l2p_epi_launch<R, EPI_RESID_ADJ>(a, e, nb, st); break;
        case EPI_H: l2p_epi_launch<R, EPI_H>(a, e, nb, st); break;
        case EPI_EONE: l2p_epi_launch<R, EPI_EONE>(a, e, nb, st); break;
        case EPI_RHS_FB: l2p_epi_launch<R, EPI_RHS_FB>(a, e, nb, st); break;
        case EPI_RESID_FC: l2p_epi_launch<R, EPI_RESID_FC>(a, e, nb, st); break;
        case EPI_IMINUSN_T: l2p_epi_launch<R, EPI_IMINUSN_T>(a, e, nb, st); break;
        case EPI_RESID_T: l2p_epi_launch<R, EPI_RESID_T>(a, e, nb, st); break;
        case EPI_MT: l2p_epi_launch<R, EPI_MT>(a, e, nb, st); break;
        case EPI_EONE_RHS: l2p_epi_launch<R, EPI_EONE_RHS>(a, e, nb, st); break;
        default:
            set_error("FMM: unknown epilogue kind %d", e.job.epi);
            return GNK_EINVAL;
    }
    return GNK_OK;
}

// Bytes of cache per product up to which it is left to L2's own policy (a third
// of the 129 MB, beside the nodes and the expansions); a larger one is
// streamed past it.
constexpr double kNbKeepBytes = 48e6;

template <int R, int COMP>
static int launch_near_bulk(const Boundary& b, const FmmArgs& a, bool adj, cudaStream_t st) {
    using L = NbLayout<R, COMP>;
    static std::mutex mu;
    static std::vector<char> ready;  // per device: the shared-memory attribute is set
    int dev = 0;
    GNK_TRY_CUDA(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lock(mu);
        if ((int)ready.size() <= dev) ready.resize(dev + 1, 0);
        if (!ready[dev]) {
            GNK_TRY_CUDA(cudaFuncSetAttribute(fmm_near_bulk_kernel<R, COMP>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize, L::kBytes));
            ready[dev] = 1;
        }
    }
    const FmmTree* t = b.fmm;
    const int stream = 8.0 * L::kParts * (double)t->near_pairs > kNbKeepBytes;
    fmm_near_bulk_kernel<R, COMP><<<dim3(t->nitems, a.nsplit), kNbThreads, L::kBytes, st>>>(
        a, t->nq_off, t->nq_item, t->nq_run, t->nq_re, adj ? t->nt_im : t->nq_im, stream);
    GNK_TRY_CUDA(cudaGetLastError());
    return GNK_OK;
}

// Starts forming the near-field cache right after the tree, on a stream of its
// own, so that it overlaps whatever the caller enqueues before the first cached
// product (the right-hand side's circulant, the first product's far field); that product waits for it.  For callers
// whose products are z = E(q x) (the FBIE and the equation's solves).
int fmm_start_near_cache(const Boundary& bc, cudaStream_t st) {
    Boundary& b = const_cast<Boundary&>(bc);
    if (b.plain) return GNK_OK;
    GNK_TRY(ensure_fmm(b, kMaxRHS, st));
    FmmTree* t = b.fmm;
    GNK_TRY(ensure_near_cache(b, false, st));
    if (t->nq_state != 2) return GNK_OK;
    if (!t->bst) {
        if (take_stream(false, &t->bst) != cudaSuccess || take_event(&t->ev_nq) != cudaSuccess) {
            cudaGetLastError();
            return GNK_OK;  // formed by the first cached product instead
        }
    }
    // the cache's buffers were allocated in the order of `st`
    GNK_TRY_CUDA(cudaEventRecord(t->ev_nq, st));
    GNK_TRY_CUDA(cudaStreamWaitEvent(t->bst, t->ev_nq, 0));
    GNK_TRY(near_cache_build(b, false, t->bst));
    GNK_TRY_CUDA(cudaEventRecord(t->ev_nq, t->bst));
    t->nq_wait = 1;
    return GNK_OK;
}

// One FMM product on the argument block `a` (weights, outputs set by the caller):
// gather, the far-field chain on the high-priority stream, the near field on
// `st`, and L2P after they join.  EF: also the sums of w/d^2 (to a.outF).
static int fmm_product(const Boundary& b, FmmArgs& a, int R, bool EF, const ReduceArgs* epi, cudaStream_t st,
                       int* nlaunch, int cached = -1, bool adj = false) {
    const FmmTree* t = b.fmm;
    // Inside a solve (st is the handle's own high-priority stream) the far field,
    // the longer chain, stays on it with the steps around it, and the near field
    // forks to a stream of its own; a product on a caller's stream forks the far
    // field instead, whose kernels then have the higher priority as well.
    const bool inside = st == t->aux;
    cudaStream_t fs = t->aux, ns = inside ? t->nst : st;
    int launches = 0;
    if (a.gathered) {
        fmm_gather_kernel<<<(b.N + 255) / 256, 256, 0, st>>>(a);
        launches = 1;
    }
    GNK_TRY_CUDA(cudaEventRecord(t->ev_fork, st));
    GNK_TRY_CUDA(cudaStreamWaitEvent(inside ? ns : fs, t->ev_fork, 0));
    // the far field on its stream: the upward pass (P2M and the M2M climb in
    // one launch), M2L for every box, L2L per leaf.  (Running the finest
    // level's M2L on a third stream beside the climb measured slower: the two
    // compete for the same SMs.)
    const ProfToken toku = prof_begin(fs, PK_FMMUP);
    if (b.diff && R == 2)
        fmm_up_kernel<2><<<t->nleaf, kFmmUT, 0, fs>>>(a);
    else if (b.diff)
        fmm_up_kernel<1><<<t->nleaf, kFmmUT, 0, fs>>>(a);
    else if (R == 2)
        fmm_up_tc_kernel<2><<<t->nleaf, kFmmUT, 0, fs>>>(a);
    else
        fmm_up_tc_kernel<1><<<t->nleaf, kFmmUT, 0, fs>>>(a);
    GNK_TRY_CUDA(cudaGetLastError());
    prof_end(toku, PK_FMMUP, 0.0, fs, fmm_instr(b, R, 1));
    const ProfToken tokm = prof_begin(fs, PK_FMM);
    if (b.diff && R == 2)
        fmm_m2l_kernel<2><<<t->nbox, kFmmUT, 0, fs>>>(a);
    else if (b.diff)
        fmm_m2l_kernel<1><<<t->nbox, kFmmUT, 0, fs>>>(a);
    else if (t->nbox >= kTcManyBoxes && R == 2)
        fmm_m2l_tc_kernel<2, 2><<<t->nbox, 64, 0, fs>>>(a);
    else if (t->nbox >= kTcManyBoxes)
        fmm_m2l_tc_kernel<1, 2><<<t->nbox, 64, 0, fs>>>(a);
    else if (R == 2)
        fmm_m2l_tc_kernel<2, 8><<<t->nbox, 256, 0, fs>>>(a);
    else
        fmm_m2l_tc_kernel<1, 8><<<t->nbox, 256, 0, fs>>>(a);
    GNK_TRY_CUDA(cudaGetLastError());
    prof_end(tokm, PK_FMM, (double)R, fs, fmm_instr(b, R, 0));  // work: Cauchy sums (products)
    launches += 2;
    if (t->L > t->l0) {
        const ProfToken tokd = prof_begin(fs, PK_FMML2L);
        if (b.diff && R == 2)
            fmm_l2l_kernel<2><<<t->nleaf, 32, 0, fs>>>(a);
        else if (b.diff)
            fmm_l2l_kernel<1><<<t->nleaf, 32, 0, fs>>>(a);
        else if (R == 2)
            fmm_l2l_tc_kernel<2><<<(t->nleaf + 3) / 4, 32, 0, fs>>>(a);
        else
            fmm_l2l_tc_kernel<1><<<(t->nleaf + 3) / 4, 32, 0, fs>>>(a);
        GNK_TRY_CUDA(cudaGetLastError());
        prof_end(tokd, PK_FMML2L, 0.0, fs, fmm_instr(b, R, 2));
        ++launches;
    }
    // what only the epilogue reads, behind the far field (the circulant product is
    // 38 us of a few blocks; before the product it held up both fields)
    if (epi) GNK_TRY(run_job_sides(b, epi->job, fs));
    if (!inside) GNK_TRY_CUDA(cudaEventRecord(t->ev_join, fs));
    // near field on its stream (from an operator cache when `cached`
    // is 0 (both parts) or 1 (the imaginary part)); the first product that reads
    // a cache forms it here, beside its far field
    if (cached >= 0) {
        if (!adj && t->nq_wait) {  // formed on its own stream since the tree was built
            GNK_TRY_CUDA(cudaStreamWaitEvent(ns, t->ev_nq, 0));
            b.fmm->nq_wait = 0;
        } else {
            GNK_TRY(near_cache_build(b, adj, ns));
        }
    }
    const ProfToken tokn = prof_begin(ns, PK_FMMNEAR);
    if (cached >= 0) {
        if (R == 2 && cached == 1)
            GNK_TRY((launch_near_bulk<2, 1>(b, a, adj, ns)));
        else if (R == 2)
            GNK_TRY((launch_near_bulk<2, 0>(b, a, adj, ns)));
        else if (cached == 1)
            GNK_TRY((launch_near_bulk<1, 1>(b, a, adj, ns)));
        else
            GNK_TRY((launch_near_bulk<1, 0>(b, a, adj, ns)));
    } else if (R == 2 && EF)
        b.diff ? fmm_near_kernel<2, true><<<t->nitems, kFmmNT, 0, ns>>>(a)
               : fmm_near_kernel<2, true, 3><<<t->nitems, kFmmNT, 0, ns>>>(a);
    else if (R == 2)
        b.diff ? fmm_near_kernel<2, false><<<t->nitems, kFmmNT, 0, ns>>>(a)
               : fmm_near_kernel<2, false, 3><<<t->nitems, kFmmNT, 0, ns>>>(a);
    else if (a.use_inv)
        fmm_near_kernel<1, false, 2><<<t->nitems, kFmmNT, 0, ns>>>(a);
    else if (EF)
        b.diff ? fmm_near_kernel<1, true><<<t->nitems, kFmmNT, 0, ns>>>(a)
               : fmm_near_kernel<1, true, 3><<<t->nitems, kFmmNT, 0, ns>>>(a);
    else
        b.diff ? fmm_near_kernel<1, false><<<t->nitems, kFmmNT, 0, ns>>>(a)
               : fmm_near_kernel<1, false, 3><<<t->nitems, kFmmNT, 0, ns>>>(a);
    ++launches;
    GNK_TRY_CUDA(cudaGetLastError());
    prof_end(tokn, PK_FMMNEAR, (double)R * t->near_pairs, ns,
             cached >= 0 ? fmm_near_cached_instr(b, R, cached) : fmm_near_instr(b, R) * (EF ? 2.0 : 1.0),
             cached >= 0 ? fmm_near_cached_bytes(b, R, cached) : 0.0);
    if (inside) GNK_TRY_CUDA(cudaEventRecord(t->ev_join, ns));
    GNK_TRY_CUDA(cudaStreamWaitEvent(st, t->ev_join, 0));
    const ProfToken tokp = prof_begin(st, PK_FMML2P);
    const int nb = (b.N + 255) / 256;
    const ReduceArgs e = epi ? *epi : ReduceArgs{};
    if (R == 2 && EF)
        fmm_l2p_kernel<2, true, false><<<nb, 256, 0, st>>>(a, e);
    else if (R == 2 && epi)
        GNK_TRY(l2p_epi<2>(a, e, nb, st));
    else if (R == 2)
        fmm_l2p_kernel<2, false, false><<<nb, 256, 0, st>>>(a, e);
    else if (EF)
        fmm_l2p_kernel<1, true, false><<<nb, 256, 0, st>>>(a, e);
    else if (epi)
        GNK_TRY(l2p_epi<1>(a, e, nb, st));
    else
        fmm_l2p_kernel<1, false, false><<<nb, 256, 0, st>>>(a, e);
    ++launches;
    GNK_TRY_CUDA(cudaGetLastError());
    prof_end(tokp, PK_FMML2P, 0.0, st, fmm_instr(b, R, EF ? 4 : 3));
    *nlaunch = launches;
    return GNK_OK;
}

static void fmm_args(const Boundary& b, FmmArgs& a) {
    const FmmTree* t = b.fmm;
    a.N = b.N;
    a.P = kFmmP;
    a.perm = t->perm;
    a.ps = t->ps;
    a.p3 = t->p3;
    a.p3b = t->p3b;
    a.leaf_start = t->leaf_start;
    a.leaf_box = t->leaf_box;
    a.center = t->center;
    a.width = t->width;
    a.child_start = t->child_start;
    a.child_count = t->child_count;
    a.parent = t->parent;
    a.quad = t->quad;
    a.il_start = t->il_start;
    a.il_src = t->il_src;
    a.il_off = t->il_off;
    a.nl_start = t->nl_start;
    a.nl_leaf = t->nl_leaf;
    a.items = t->items;
    a.nitems = t->nitems;
    a.zn = t->zn;
    a.zf = t->zf;
    a.node_box = t->node_box;
    a.m2lH = t->m2lH;
    a.m2lS = t->m2lS;
    a.bUp = t->bUp;
    a.m2lT = t->m2lT;
    a.m2lA = t->m2lA;
    a.upA = t->m2lA + kFmmASlots;
    a.dnA = t->m2lA + 2 * kFmmASlots;
    a.path = t->path;
    a.depth = t->L - t->l0 + 1;
    a.nleaf = t->nleaf;
    a.ucnt = t->sync;
    a.inv_off = t->inv_off;
    a.inv_r = t->inv_r;
    a.inv_i = t->inv_i;
    a.use_inv = 0;
    a.gathered = 1;
    a.nsplit = 1;
    a.near_scaled = 0;
    a.tn = t->tn;
    a.diff = b.diff;
    a.mult = t->mult;
    a.loc = t->loc;
    a.ws = t->ws;
    a.nbox = t->nbox;
    a.outF = nullptr;
    a.done = nullptr;
    a.fault = t->fault;
}

// The stream on which a solve with FMM products runs: the far field's, so that
// the chain product - Arnoldi step - product has no hop between streams (two of
// about 4 us each per step).  The caller orders it with events (ev_solve).
int fmm_solve_stream(const Boundary& b, cudaStream_t st, cudaStream_t* own, cudaEvent_t* ev) {
    GNK_TRY(ensure_fmm(b, kMaxRHS, st));
    *own = b.fmm->aux;
    *ev = b.fmm->ev_solve;
    return GNK_OK;
}

int run_fmm(const Boundary& b, const PairJob& job, cudaStream_t st) {
    GNK_TRY(ensure_fmm(b, job.R, st));
    FmmArgs a;
    fmm_args(b, a);
    a.R = job.R;
    a.mode = job.mode;
    a.w0 = job.w[0];
    a.w1 = job.w[1];
    a.x0 = job.x[0];
    a.x1 = job.x[1];
    a.s = job.s;
    a.out = nullptr;
    a.done = job.done;
    int launches = 0;
    // Products with the handle's own weights q x read the near field from its
    // operator cache (formed by the first of them), one part of it where the
    // operator reads Im(A z) alone.  Those with weights A x whose operator reads
    // Im(q z) do so inside a solve (job.done), which forms the cache: it costs
    // two or three products and a solve has many.
    int cached = -1;
    const bool im_only = job.R == 1 && (job.epi == EPI_IMINUSN || job.epi == EPI_RESID);
    const bool im_adj = job.R == 1 && (job.epi == EPI_ADJ || job.epi == EPI_RESID_ADJ || job.epi == EPI_IMINUSN_T ||
                                       job.epi == EPI_RESID_T);
    const bool adj = job.s != b.q && job.s == b.A && im_adj && !b.diff;
    if (job.mode == W_SCALED && !b.plain && (job.s == b.q || adj)) {
        if (!adj || job.done != nullptr) GNK_TRY(ensure_near_cache(b, adj, st));
        if ((adj ? b.fmm->nt_state : b.fmm->nq_state) >= 1) {
            cached = (adj || im_only) ? 1 : 0;
            a.gathered = b.diff;  // its P2M reads the sorted weights
            a.near_scaled = 1;
            a.nsplit = fmm_near_splits(b, b.fmm->nitems);
        }
    }
    if (b.diff && im_adj && job.mode == W_SCALED && job.s == b.A && !b.plain) {
        if (job.done != nullptr) GNK_TRY(ensure_inverse_cache(b, st));
        if (b.fmm->inv_state == 1) {
            a.inv_off = b.fmm->inv_off;
            a.inv_r = b.fmm->inv_r;
            a.inv_i = b.fmm->inv_i;
            a.use_inv = 1;
        }
    }
    // The direct circulant (n not a power of two) fills the FP64 pipes: it comes before
    // the product.  Behind the far field its blocks got the SMs that the near field left
    // first, up to eight on one (M at 64 x 1,030 nodes: 437 us, 294 now).
    PairJob sides = job;
    if (job.Lsrc && !b.fft_pow2) {
        GNK_TRY(run_circulant(b, job.Lsrc, b.r3, st));
        sides.Lsrc = nullptr;
    }
    const ReduceArgs e = reduce_args(b, sides, 1, 0);  // the epilogue runs inside L2P
    GNK_TRY(fmm_product(b, a, job.R, false, &e, st, &launches, cached, adj));
    count_launches(launches);
    return GNK_OK;
}

// E w and F w (sums of w_j/(eta_i - eta_j) and of w_j/(eta_i - eta_j)^2, i != j)
// for one or two complex weight vectors (w1 may be null), into E and F
// (R x N complex each, node order), by one FMM pass.
int run_fmm_ef(const Boundary& b, const double2* w0, const double2* w1, double2* E, double2* F, cudaStream_t st) {
    const int R = w1 ? 2 : 1;
    GNK_TRY(ensure_fmm(b, R, st));
    FmmArgs a;
    fmm_args(b, a);
    a.R = R;
    a.mode = W_COMPLEX;
    a.w0 = w0;
    a.w1 = w1;
    a.x0 = a.x1 = nullptr;
    a.s = nullptr;
    a.out = E;
    a.outF = F;
    int launches = 0;
    GNK_TRY(fmm_product(b, a, R, true, nullptr, st, &launches));
    count_launches(launches);
    return GNK_OK;
}

}  // namespace gnk
