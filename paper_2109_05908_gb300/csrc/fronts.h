// Substructuring plan of a sparse symmetric matrix (see fronts.cu).
#pragma once
#include <cstdint>
#include <vector>

namespace amdd {

// One part: m interior unknowns at plan positions [i0, i0 + m) and nb boundary
// unknowns bnd[b0 .. b0 + nb) (plan positions of later stages, ascending).
// The boundary lies within the parent's interior and boundary.
struct Front {
    int m = 0, nb = 0, stage = 0, parent = -1;
    int64_t i0 = 0, b0 = 0;
};

struct FrontPlan {
    int64_t n = 0;
    std::vector<int32_t> perm;       // unknown at each plan position
    std::vector<Front> fronts;       // in stage order
    std::vector<int> stage_part;     // fronts of stage s: [stage_part[s], stage_part[s + 1])
    std::vector<int64_t> stage_off;  // their unknowns: [stage_off[s], stage_off[s + 1])
    std::vector<int32_t> bnd;
    int stages() const { return (int)stage_part.size() - 1; }
};

// Plan of a graph (ptr, adj: symmetric adjacency without self loops) whose
// vertex v stands for the wt[v] unknowns base[v] .. base[v] + wt[v] - 1.
FrontPlan plan_fronts(const std::vector<int32_t>& ptr, const std::vector<int32_t>& adj,
                      const std::vector<int32_t>& wt, const std::vector<int32_t>& base, int leaf, int ratio);

}  // namespace amdd
