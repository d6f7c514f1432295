// Hierarchical T o H product: w_a = sum_{b >= a} s[b-a] h[a+b] v_b in O(n) (Fig. 1 step 4 without
// the FFTs).
//
// s and h are Gamma ratios, smooth away from index 0, so the entries of a block of rows and
// columns that keeps its own width away from the diagonal are a polynomial in each index up to
// a small remainder: interpolation in P Chebyshev points of the block (rounded to integers, so
// that only table entries are ever needed) converges like 5.83^-P.  The upper triangle is cut
// into such blocks by a tree:
//   leaves of 32 packed indices; boxes of 32, 128, 512 and 2048 (four children each);
//   near field: each leaf with itself and its right neighbour, entry by entry;
//   a box takes from the boxes of its own size that are not adjacent to it and whose parents
//   are equal or adjacent; a 2048-box from every box of its size that is not adjacent.
// moments   M_q(box) = sum_b L_q(b) v_b             (leaves; parents from children)
// exchange  E_p(box) = sum_{far boxes j} sum_q s[y_q - x_p] h[x_p + y_q] M_q(j)
// local     E(child) += E(parent) at the child's points; w_a = sum_p L_p(a) E_p(leaf) + near.
// L_q are the Lagrange polynomials of the box's points x_q.
//
// Parity kinds (T_jk = 0 for odd k - j) run as two channels of packed indices, k = 2a + e,
// with s_m = t_{2m} and h_l = h_{2l}, the odd channel's Hankel table being the even one's
// shifted by one (h_{2(a+b)+2e}).  The transpose is the same product on reversed indices
// (k' = N - 1 - k, N whole boxes of the largest size that exchanges anything), with the reversed
// Hankel table.
#pragma once

#include "tdh_internal.cuh"

namespace tdh {

constexpr int kHierLeaf = 32;      // packed indices per leaf
constexpr int kHierLevels = 4;     // boxes of 32, 128, 512, 2048 packed indices
constexpr int kHierTop = 2048;
constexpr int kHierTopLeaves = kHierTop / kHierLeaf;
constexpr int kHierSZero = 32;     // zeros stored before s[0]
constexpr int kHierHPad = 512;     // zeros stored after the last Hankel entry

// Interpolation points: 8 give the far field to about 2e-8 of the result in float32 (below its
// rounding), 16 to below 1e-14 in float64.
template <typename T>
struct HierP {
    static constexpr int P = sizeof(T) == 4 ? 8 : 16;
};

// The points of a box, per level: round((size - 1)/2 (1 - cos(pi (2i + 1) / (2P)))), kept distinct.
template <int P>
__host__ __device__ constexpr int hier_point(int level, int i) {
    static_assert(P == 8 || P == 16, "points per box");
    if constexpr (P == 8) {
        constexpr int x[kHierLevels][8] = {{0, 3, 7, 12, 19, 24, 28, 31},
                                           {1, 11, 28, 51, 76, 99, 116, 126},
                                           {5, 43, 114, 206, 305, 397, 468, 506},
                                           {20, 172, 455, 824, 1223, 1592, 1875, 2027}};
        return x[level][i];
    } else {
        constexpr int x[kHierLevels][16] = {
            {0, 1, 2, 4, 6, 8, 11, 14, 17, 20, 23, 25, 27, 29, 30, 31},
            {0, 3, 7, 14, 23, 34, 45, 57, 70, 82, 93, 104, 113, 120, 124, 127},
            {1, 11, 30, 58, 93, 135, 181, 230, 281, 330, 376, 418, 453, 481, 500, 510},
            {5, 44, 121, 232, 374, 541, 726, 923, 1124, 1321, 1506, 1673, 1815, 1926, 2003, 2042}};
        return x[level][i];
    }
}

__host__ __device__ constexpr int hier_size(int level) { return kHierLeaf << (2 * level); }

}  // namespace tdh
