// FMM tree shared by the host- and device-side tree builders and the FMM
// product (fmm.cu, fmm_tree.cu).  Internal header.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "gnk_internal.h"

namespace gnk {

constexpr int kFmmP = 32;     // expansion order (one warp lane per coefficient)
// M2L offsets between boxes of the topmost level span the grid of level 3
constexpr int kFmmOffMax = 7;
constexpr int kFmmOffs = 2 * kFmmOffMax + 1;  // offset code (dx + 7) 15 + (dy + 7)
constexpr int kFmmNT = 256;   // threads of the near-field kernel: 8 warps
constexpr int kFmmMaxNbr = 9;  // a leaf and its eight neighbours

struct FmmTree {
    int L = 0, nbox = 0, nleaf = 0, R = 0;
    int l0 = 2;                 // the topmost level with expansions
    std::vector<int> lvl_off;   // first global box index of level l (index l - l0), size L - l0 + 1
    std::vector<int> lvl_cnt;
    long long near_pairs = 0, m2l_pairs = 0, m2m_pairs = 0;
    void* arena = nullptr;
    int* perm = nullptr;        // sorted position -> node
    double2* ps = nullptr;      // node positions in sorted order
    float4* p3 = nullptr;       // the same split exactly into three floats: (x1, x2, x3, y1)
    float2* p3b = nullptr;      // (y2, y3)
    int* leaf_start = nullptr;  // nleaf + 1
    int* leaf_box = nullptr;    // global box index of each leaf
    double2* center = nullptr;  // per box
    double* width = nullptr;    // per box
    int* child_start = nullptr; // per box: first child (global), level < L
    int* child_count = nullptr;
    int* parent = nullptr;      // per box, -1 on level l0
    int* quad = nullptr;        // quadrant of a box in its parent: 2 qa + qb
    int* il_start = nullptr;    // interaction lists (nbox + 1), sources, offset codes
    int* il_src = nullptr;
    int* il_off = nullptr;
    int* nl_start = nullptr;    // neighbour leaves of each leaf (nleaf + 1)
    int* nl_leaf = nullptr;
    int2* items = nullptr;      // (leaf, first target) of every chunk of 32 targets
    int nitems = 0;
    const float2* m2lH = nullptr;  // M2L: the Pascal matrix C(k+l, l) [k][l] as double-float,
    const float4* m2lS = nullptr;  // and per offset code the two complex scalings (per-device cache)
    const float2* bUp = nullptr;   // L2L Pascal table C(l,m) [l][m]
    const float4* m2lT = nullptr;  // the scalings with their powers of two, and the digits of
    const uint4* m2lA = nullptr;   // C(k+l, l) 2^-(k+l) as tensor-core fragments
    float4* mult = nullptr;     // [R][nbox][P]
    float4* loc = nullptr;      // [R][nbox][P]
    float4* ws = nullptr;       // [R][N] weights in sorted order, double-float complex
    double2* zn = nullptr;      // [R][N] near-field sums in sorted order
    double2* zf = nullptr;      // [R][N] near-field sums of w/d^2 (gradient products)
    int* node_box = nullptr;    // leaf box of each node in sorted order
    int* sync = nullptr;        // [nbox]: children counted by the upward pass (zero between products)
    // near-field operator caches (fixed geometry): per work item the entries of
    //   A_i q_j / (eta_i - eta_j)  for the products with weights q x (both parts),
    //   q_i A_j / (eta_i - eta_j)  for the solves with weights A x (imaginary part),
    // double-float, for source pairs x targets.  The items' shapes are shared.
    int near_shape = 0;           // 1: nq_off, nq_item, nq_run are allocated; 2: formed
    long long* nq_cnt = nullptr;  // [nitems] build temporary of the shapes
    long long* nq_off = nullptr;  // per work item: first entry (nitems + 1)
    int2* nq_item = nullptr;      // per work item: (S sources, tn targets)
    int2* nq_run = nullptr;       // [nitems][kFmmMaxNbr]: (first source, sources before) of each
                                  // neighbour leaf; (0, INT_MAX) past the last
    long long nq_slots = 0;       // float4 entries of each of the arrays below
    // state 0 not formed, 2 allocated (formed by the first cached product),
    // 1 formed, -1 not used (too large)
    int nq_state = 0, nt_state = 0;
    float4* nq_re = nullptr;
    float4* nq_im = nullptr;
    float4* nt_im = nullptr;
    // handles built for differentiation: 1/(eta_i - eta_j) of every near pair (state as above)
    int inv_state = 0;
    long long* inv_off = nullptr;  // nitems + 1
    float4* inv_r = nullptr;
    float4* inv_i = nullptr;
    int* fault = nullptr;       // set by a bounded wait of an FMM kernel that gave up
    unsigned* path = nullptr;   // [nleaf][L - l0 + 1]: box | quadrant << 30 of each leaf and its ancestors
    float4* tn = nullptr;       // [N] offset of each node from its leaf centre in leaf widths
    cudaStream_t aux = nullptr; // high-priority stream of the far field (the near field runs beside it)
    cudaStream_t nst = nullptr; // the near field's stream inside a solve (which runs on aux)
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_solve = nullptr;
    cudaStream_t bst = nullptr; // stream of the near cache's formation when it starts early
    cudaEvent_t ev_nq = nullptr;
    int nq_wait = 0;            // the next cached product waits for ev_nq
};

// Builds the tree on the device (Morton keys, stable radix sort, boxes per level,
// interaction and neighbour lists) into t, with its device arena.  Returns
// GNK_OK, an error code, or kFmmUseHost when the tree is too deep for the
// device lookup grids (then the host builder runs).
constexpr int kFmmUseHost = 1;
constexpr int kMaxGridLevel = 11;  // the deepest level of those grids

// The topmost level with expansions.  From level 3 on in trees of level 4 and more (all of whose boxes then
// interact where they are not adjacent, at most 60 each) the climb and the descent
// are one level shorter: about 8 us of latency per product against some 2,000
// more M2L pairs.  Handles built for differentiation keep level 2.
inline int fmm_top_level(const Boundary& b, int L) { return (b.diff || L < 4) ? 2 : 3; }
int fmm_tree_device(const Boundary& b, FmmTree* t, cudaStream_t st);

// Whether the tree goes down to level l, given the mean number of nodes in its
// non-empty boxes.  Level 3 (a first M2M and L2L) wants 64 nodes: at N = 2,560 the
// adjoint slit map takes 8.9 ms with leaves of 160 on level 2, 10.1 with 46 on level
// 3.  Deeper ones want 44: M2L pairs cost the tensor cores little, near pairs 8
// bytes each (N = 524,288: 129 nodes per leaf 60.1 ms, 62 nodes 40.9, 30 nodes
// 45.3; adjoint solve at N = 16,830: 128 nodes 2.20 ms, 55 nodes 2.11; N = 65,536:
// 68 nodes 3.48 ms, 33 nodes 3.57).  Handles built for differentiation keep 64.
// Where the boxes fill the plane a level has up to four times the nodes of the next:
// there the line is the geometric mean of the two (62): 400 close circles at N = 40,000,
// 156 nodes per leaf 8.58 ms, 39 nodes 5.66; 576 at 36,864, 144 nodes 11.19, 36 nodes 8.14.
// Levels beyond the device builder's grids want 64 too: the host builds such a tree
// (196 small circles far apart, N = 156,800: the FBIE with its tree 6.96 ms with the 47
// nodes of level 12, 2.66 with the 95 of level 11).
inline bool fmm_level_wanted(const Boundary& b, int l, double mean_nodes, double parent_nodes) {
    if (l < 4 || l > kMaxGridLevel || b.diff) return mean_nodes >= 64.0;
    return mean_nodes >= 44.0 || (mean_nodes >= 28.0 && mean_nodes * parent_nodes >= 62.0 * 62.0);
}

// Shares that each work item of a cached near field is split into: four blocks run
// on an SM at once, and fewer items than that leave SMs idle.  Handles built for
// differentiation keep whole items.  (More items never give more shares, so a
// lower bound of their number, one per leaf and per 32 nodes, sizes the sums.)
inline int fmm_near_splits(const Boundary& b, int nitems) {
    const int want = 4 * b.sms / (nitems > 0 ? nitems : 1);
    return b.diff ? 1 : (want < 1 ? 1 : (want > 4 ? 4 : want));
}

// Points t at the translation tables on the current device (formed and uploaded
// once per device and process): the M2L Pascal matrix C(k+l, l)
// [P][P] and, per offset code, the scalings
// (-1)^(k+1) delta^-(k+1) and delta^-l; the L2L Pascal matrix C(l, m).
int fmm_device_tables(FmmTree* t, cudaStream_t st);

}  // namespace gnk
