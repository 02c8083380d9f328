// Hierarchical pair sums (tree.cu): plan, workspace layout and launchers.
#pragma once

#include "vesis_internal.cuh"

namespace vesis {

// 64-cell tiles per axis and in all; a grid has 64 times as many 16-cell
// tile slots (slots past the grid's end stay empty).
struct TreeDims {
    int nx, ny, nz, n2;
};

// Parts of a column's gradient terms: its x planes (direct rows), and its z
// range (nodes of levels 0 and 1).
constexpr int kRowParts = 2, kZParts0 = 4, kZParts1 = 4;

// One list of work items: item i is chunk i - first[tile] of its tile.
struct TreeList {
    int tiles = 0, len = 0, max_items = 0;
    size_t o_first = 0, o_item = 0;      // first[tiles + 1], item -> tile
};

// Workspace of one system (byte offsets into one allocation).
struct TreePlan {
    TreeDims d{};
    TreeList list[6];       // far atoms of levels 0, 1, 2; column atoms of levels 0, 1, 2
    int sf = 1;             // chunks of the level-2 gradient terms
    size_t o_tab = 0, o_cnt = 0, o_off = 0, o_cur = 0, o_coff = 0, o_id = 0, o_tmp = 0,
           o_ord = 0, o_xyzq = 0, o_ab = 0, o_cxyz = 0, o_cfc = 0, o_part = 0, o_v[3] = {0, 0, 0}, bytes = 0;
};

// Whether a system's fields and its gradient take the hierarchical kernels (a
// rule on the sizes, the spacing and the LJ radii alone; the gradient's
// implies the fields').  sum_sigma3: sum of the cubes of the LJ radii.
bool tree_fields_pay(const GridDesc &g, int n, double h, double rmin, double max_sigma);
bool tree_force_pays(const GridDesc &g, int n, double h, double rmin, double max_sigma,
                     double sum_sigma3);
// force: with the gradient's partials.
TreePlan plan_tree(const GridDesc &g, int n, int nsm, bool force);
size_t tree_tab_bytes();
void tree_fill_tab(void *host);
// U and E on every cell at the packed atoms.
void launch_tree_fields(const GridDesc &g, const TreePlan &p, uint8_t *ws, const AtomsDev &a,
                        float rho, float cfa, float rmin2, float *U, float *Ex, float *Ey,
                        float *Ez, cudaStream_t st);
// out[n][3] = scale x the grid gradient sums of the packed atoms a; cg: the
// direct kernel's cell groups (plan_pair_force); the solvent cells are added
// to *nsolvent.
void launch_tree_force(const GridDesc &g, const TreePlan &p, uint8_t *ws, const AtomsDev &a,
                       int cg, const uint8_t *chi, const float *Ex, const float *Ey,
                       const float *Ez, float rmin2, double scale, double *out,
                       unsigned long long *nsolvent, cudaStream_t st);

}  // namespace vesis
