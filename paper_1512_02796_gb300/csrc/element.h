// Element plan of a mesh (internal): the geometry of its tets, laid out per
// tet, per edge and per node, so that every sum over elements becomes a
// gather in a fixed order.
//
// For a P1 tet with gradients g_a of the hat functions and volume |T|, the
// off-diagonal stiffness factors s_ab = |T| g_a . g_b / 4 (6 edges) and
// vm = |T| / 120 are all that the operators of this library need:
//   K:   a_ij = sum_T s_ij (sum of the tet's 4 kappa)              (stiffness)
//             + sum_T vm Sm_T + (sum_T vm) (mu_i + mu_j)           (mass, Sm_T = sum of 4 mu)
//             + the Robin term of the edge's boundary faces;
//   M_delta blocks:  a_ij = sum_T 4 s_ij c_T,  |grad u|^2 = -sum_ab s_ab (u_a - u_b)^2 / (30 vm);
// over the tets T around edge (i, j), and the rows of a stiffness sum to 0.
// The geometry does not change with the coefficients, and FP64 arithmetic is
// scarce on GB300 (2 multiply-adds per SM and cycle), so it is computed once
// per mesh and read back.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "qpat_internal.h"

namespace qpat {

// Tet-local vertex pairs of the 6 edges, in slot order.
__host__ __device__ constexpr int edge_a(int slot) { return slot < 3 ? 0 : slot < 5 ? 1 : 2; }
__host__ __device__ constexpr int edge_b(int slot) { return slot < 3 ? slot + 1 : slot < 5 ? slot - 1 : 3; }

struct ElementPlan {
    int64_t NE = 0;                    // edges (i < j, library ids), numbered by i, then by i's row order
    std::vector<int32_t> tet;          // 4 E library ids, tets sorted by their lowest node (vertex order kept)
    std::vector<int64_t> node_ptr;     // N + 1: tets of each node, ascending
    std::vector<int32_t> node_tet;
    std::vector<int32_t> ent_edge;     // per SELL position of the K pattern: edge (-1: diagonal or padding)
    std::vector<int32_t> ent_col;      //   and the entry's node (the row itself on padding)
    std::vector<int32_t> pent_edge;    // per SELL position of the prior's pattern: edge
    std::vector<int32_t> edge;         // 2 NE
    std::vector<int32_t> tet_edge;     // 6 E
    std::vector<int64_t> edge_ptr;     // NE + 1: tets around each edge, ascending
    std::vector<uint32_t> edge_tet;    //   8 tet + slot of the edge in that tet (E < 2^29)
    std::vector<uint8_t> in_prior;     // NE: the prior's pattern holds the edge
    // pairs (0, Robin sum): |F| / 24 over the edge's boundary faces, |F| / 12 over the node's
    std::vector<double> edge_vr;       // 2 NE
    std::vector<double> node_vr;       // 2 N
};

ElementPlan build_element_plan(const HostMesh& h);
// Checks every id the device gathers by; "" if all hold.
std::string check_element_plan(const HostMesh& h, const ElementPlan& p);

// Device view of the plan with the geometry computed from the coordinates.
struct ElemDev {
    int64_t E = 0, NE = 0;
    const int4* tet = nullptr;
    const int64_t* node_ptr = nullptr;
    const int* node_tet = nullptr;
    const int* ent_edge = nullptr;
    const int* ent_col = nullptr;
    const int* pent_edge = nullptr;
    const int2* edge = nullptr;
    const int* tet_edge = nullptr;
    const int64_t* edge_ptr = nullptr;
    const uint32_t* edge_tet = nullptr;
    const uint8_t* in_prior = nullptr;
    double* s = nullptr;        // 6 E
    double* vm = nullptr;       // E
    double2* edge_vr = nullptr;  // NE: (sum of vm around the edge, Robin sum)
    double2* node_vr = nullptr;  // N: (sum of vm around the node, Robin sum)
};

// Scratch of one sequence of element kernels: one double2 per tet and per edge.
struct ElemScratch {
    double2* tet = nullptr;
    double2* edge = nullptr;
};

// Fills s, vm, edge_vr, node_vr (edge_vr.y and node_vr.y already hold the Robin sums).
cudaError_t launch_element_geometry(const MeshDev& m, const ElemDev& el, cudaStream_t s);

}  // namespace qpat
