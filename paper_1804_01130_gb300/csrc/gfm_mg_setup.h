// Host-side multigrid hierarchy of a handle's mesh; plain C++, no CUDA.
#pragma once

#include <cstdint>
#include <vector>

namespace gfm {

constexpr int kMgMaxLevels = 24;   // levels of the hierarchy, the mesh included (kMgLevels)
constexpr int kMgCoarsest = 4;     // stop coarsening at this many nodes

// One coarse level.  Its nodes are aggregates of the next finer level's
// nodes (of cells, on the first coarse level); its faces collect the finer
// faces that join two aggregates.
struct MgLevelHost {
    int n = 0, n_pad = 0, n_slices = 0, n_slots = 0, max_width = 0, max_child = 0, F = 0;
    std::vector<int32_t> slice_ptr;  // [n_slices + 1] sliced-ELL table of the level's graph, as Sell
    std::vector<int32_t> col;        // [n_slots]
    std::vector<int32_t> face;       // [n_slots] face + 1, 0 on padding slots
    std::vector<int32_t> child_ptr;  // [n_slices + 1] sliced-ELL list of each node's children
    std::vector<int32_t> child;      // finer node, -1 on padding slots
    std::vector<double> scale;       // [F] geometric factor of the face's coefficient
    std::vector<int32_t> mem_ptr;    // [F + 1] finer faces of each face, ascending
    std::vector<int32_t> mem;        // (caller faces or slots on the first coarse level)
};

// Coarse levels of the mesh (caller owner/neighbour, area vectors Sf [3][F]
// and centres C [3][n], perm = caller -> internal cell; n_pad internal cells).
// With the mesh table's slot_face [n_slots] (HostTables::face) the first
// level's members are its faces' slots in their owners' rows, which lie near
// each other, instead of caller faces.
std::vector<MgLevelHost> build_mg_levels(int n, int n_pad, int F, const int32_t *owner, const int32_t *nb,
                                         const double *Sf, const double *C, const int32_t *perm,
                                         const int32_t *slot_face = nullptr, int n_slots = 0);

}  // namespace gfm
