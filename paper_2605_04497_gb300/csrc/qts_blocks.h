// Block tables: the FP32 first-order and adjoint passes evaluate a whole small
// subtree (up to 8 leaves) against the merged elements its leaves share.
//
// A block is a node r of the tree with part of the subtree below it, h <= 3
// levels of splits (h = 0: a leaf), and the D merged elements of the path to r that
// all its leaves share.  With C(t) the product of the shared elements' factors
// a_l(t) = z_l + t (o_l - z_l), and G(t) the sum over the block's leaves of val
// times the factors of the elements met from r down,
//     sum over the block's leaves of val prod a = C(t) G(t),
// so the shared elements need one prefix and suffix sweep per block, whose suffix
// starts at G(t) instead of 1, and the element on an edge below r with the leaf
// sum G_c under it adds (o - z) sum_m w_m C_v G_c to its feature, C_v being C times
// the factors between r and the edge.  Per leaf of a full h = 3 block this is an
// eighth of the shared elements' work and about one edge's, where a path of its
// own costs every element again.
//
// A feature that is split on again below an edge merges with it, so its element
// differs between the leaves.  r itself may repeat a feature of its path: that
// element leaves the shared ones and r's edges carry the merged weights and
// interval.  A lower node that repeats one is cut out: its place in the block is an
// empty leaf (val = 0), and it is (part of) a block of its own.  Which nodes
// become blocks, and of which height, minimises an estimate of the kernels'
// instructions over the whole tree (blk_cost).
//
// The subtree is always complete: heap-numbered nodes 1.. (children of n: 2n,
// 2n + 1), where the lowest level's ("pair") nodes have two leaves and the others
// ("inner") two nodes.  A leaf higher up stands at the end of neutral nodes (zL = 1,
// zR = 0 on the tile's zero row, so o - z = 0 on both sides).  The kernels need no
// branch on the shape.
//
// Records, 16 bytes each: header {val, 0, 0, 0} (h = 0 only), D elements {z, z,
// lo, hi}, their feature words (four to a record), then the inner nodes
//   {zL, zL, zR, zR}, {theta, lo, hi, word}
// and the pair nodes
//   {valL, valR, zL, zR}, {theta, lo, hi, word}, {vz, vz, 0, 0}
// with vz the sum of val z.  Weights that the sample-pair kernels multiply by are
// stored as pairs.  [lo, hi) is what the splits above leave of the feature's range
// (all of it but at r); word: the feature, kNanOk and kDefLeft.
//
// FP64 ensembles keep the FP64 weights beside the records, per block: val (h = 0),
// z of the D elements, zL and zR of the inner nodes, {valL, valR, zL, zR, vz} of the
// pair nodes.
//
// Adjoint sums of a block ("slots"): the z-gradients of its D elements, of every
// inner node's two edges, then per pair node Q and for each leaf K (dL/dval = z Q
// + K, dL/dz = val Q).  h = 0: the D z-gradients and the leaf value's gradient.
#pragma once

#include <stdint.h>

#include "qts_internal.h"

namespace qts {

#ifdef __CUDACC__
#define QTS_HD __host__ __device__
#else
#define QTS_HD
#endif

constexpr int kBlkMaxH = 3;
// Highest block of width D: the adjoint keeps about 88 registers of state of an
// h = 3 subtree (36 for h = 2) beside 12 per shared element.
QTS_HD constexpr int blk_max_h(int D) { return D <= 9 ? 3 : D <= 16 ? 2 : 1; }

QTS_HD constexpr int blk_inner(int h) { return h >= 2 ? (1 << (h - 1)) - 1 : 0; }
QTS_HD constexpr int blk_pairs(int h) { return h >= 1 ? 1 << (h - 1) : 0; }
// records before the subtree, and of a whole block
QTS_HD constexpr int blk_head(int D) { return 1 + D + (D + 3) / 4; }
QTS_HD constexpr int blk_stride(int D, int h) { return blk_head(D) + 2 * blk_inner(h) + 3 * blk_pairs(h); }
// record offset after the head, and slot offset after the elements, of node n
QTS_HD constexpr int blk_rec(int h, int n) {
    return n <= blk_inner(h) ? 2 * (n - 1) : 2 * blk_inner(h) + 3 * (n - 1 - blk_inner(h));
}
QTS_HD constexpr int blk_slot(int h, int n) { return blk_rec(h, n); }
QTS_HD constexpr int blk_slots(int h) { return h == 0 ? 1 : 2 * blk_inner(h) + 3 * blk_pairs(h); }

// FP64 values of a block, and the offset of node n's among them
QTS_HD constexpr int blk_doubles(int D, int h) { return 1 + D + 2 * blk_inner(h) + 5 * blk_pairs(h); }
QTS_HD constexpr int blk_dbl(int D, int h, int n) {
    return 1 + D + (n <= blk_inner(h) ? 2 * (n - 1) : 2 * blk_inner(h) + 5 * (n - 1 - blk_inner(h)));
}

// Relative cost of a block: about the instructions per warp of the forward pass
// (36 per shared element, 65 per inner and 36 per pair node, 25 for the rest).
inline double blk_cost(int D, int h) { return 25.0 + 36.0 * D + 65.0 * blk_inner(h) + 36.0 * blk_pairs(h); }

constexpr double kBlkUnit = 300.0;

}  // namespace qts
