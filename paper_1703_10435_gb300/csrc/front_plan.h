// Elimination schedule of a local problem: the order in which its nodes are eliminated, and
// for every step which nodes are in the front (the nodes that touch an eliminated one or are
// about to) and in which slot of the front matrix each of them sits.  The schedule depends on
// the refinement level, the degree and the dimension only, so a mesh holds one per level.
#pragma once

#include <cstdint>
#include <vector>

namespace mhm {

// One step: the node in slot `ps` is eliminated (kNoSlot: none, at the start) and the node
// `enter` (-1: none) comes into slot `zs`.  A node enters no later than the step that
// eliminates its first neighbour.  m: slots in use during the step.
struct FrontStep {
    int pivot = -1, enter = -1;
    int ps = 255, zs = 255;
    int m = 0;
};

constexpr int kNoSlot = 255;      // step tables keep slots in a byte
constexpr int kMaxSlots = 250;
constexpr int kPivotSlot = 254;   // coupling entry: with the node eliminated in this step
constexpr int kDiagSlot = 253;    // coupling entry: a part of the entering node's diagonal

// Steps that eliminate the nodes in `order`, each node entering as late as one entry per
// step allows; *slots gets the largest front (none if it exceeds kMaxSlots).  cliques: nb nodes
// each, which couple with one another (fine triangles or sub-tetrahedra; -1: no node).
std::vector<FrontStep> front_schedule(const std::vector<int>& cliques, int nb, const std::vector<int>& order,
                                      int* slots);

// Tables of the 2-D refined triangle (N segments per face, degree P) as the kernels read
// them, in one array.  Steps first, 4 int32 each: ps | zs << 8 | m << 16; lattice point x | y << 16 of the
// entering node; the number of its fine triangles that carry its mass, and bit 8 + a if it
// lies on local face a; lattice point of the pivot.  Then the couplings, per step ncp entries
// of 2 uint32: slot | e0 << 8 | e1 << 16 and t0 | t1 << 16: the value kappa[t0] Ke[e0] + kappa[t1] Ke[e1] (t1 = 0xffff: one term; Ke[36 down + 6 a + b]),
// unused entries with slot kNoSlot; the last three hold the diagonal's (up to six) terms.
struct FrontPlan {
    int steps = 0, slots = 0, ncp = 0;   // steps = 0: no plan (front too large)
    std::vector<uint32_t> tab;
};
FrontPlan front_plan_2d(int P, int N);

// Tables of the refined tetrahedron, the DOF of most sub-tetrahedra left out (pinned; in the
// interior the pin holds the constants 3 to 10 times closer than a corner of one sub-tetrahedron
// does); node v is DOF v, or v + 1 from the pinned one on.  dofs: the nb DOFs of every
// sub-tetrahedron, cls its class, xyz the DOFs' lattice coordinates (A, B, C).  ev: 4 int32
// per step: ps | zs << 8 | m << 16; the entering DOF (-1: none); first and number of its
// entries.  ent: slot | terms << 8 | first term << 16, the first 8 of a node the parts of its
// diagonal; the value of an entry is the sum of its terms kappa[t] S[s] (con: t | s << 16,
// s = (class nb + a) nb + b).  Of three orders the one with the least work for R loads.
// The fourth value of a step also holds the pivot's node << 16; first_pivot: the
// first step that has one.  For products with the matrix: val: first term | terms << 16 of
// every off-diagonal value (in the order of the entries), then of every node's diagonal;
// rc: the off-diagonal values' nodes v | u << 16; rp, col: per node its row, as
// neighbour | value << 16.
struct FrontPlan3 {
    int steps = 0, slots = 0, first_pivot = 0, off = 0, pin = 0;
    std::vector<int32_t> ev, rp;
    std::vector<uint32_t> ent, con, val, rc, col;
};
FrontPlan3 front_plan_3d(int n, int nb, const std::vector<int32_t>& dofs, const std::vector<int8_t>& cls,
                         const std::vector<int32_t>& xyz, int R);

}  // namespace mhm
