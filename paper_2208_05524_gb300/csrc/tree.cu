// Hierarchical pair sums of the VESIS hot path (sm_103a, FP32 CUDA cores):
// the fields U, E on the grid (Eq. Ur) and the grid-to-atom gradient (Eq.
// GradientG) of large solutes, in far fewer pair terms than cells x atoms.
//
// The grid is cut into cubic tiles of 16, 32 and 64 cells (levels 0, 1, 2).
// Two tiles of a level are near if they touch (index distance at most 1 per
// axis).  An atom and a cell meet
//   directly, pair by pair, if their 16-cell tiles are near,
//   at level l if their level-l tiles are not near but their parents are
//     (level 2: if their 64-cell tiles are not near).
// At level l the field of the atoms is smooth over the cell's tile (the
// nearest such atom is more than two tile half-widths from its face), so it
// is summed at the tile's Chebyshev nodes and interpolated to the cells by
// tensor-product Lagrange polynomials (a target-side interpolating
// treecode; the interpolation from a tile's nodes to its children's nodes
// chains the levels).  The gradient is the transpose: the solvent mask and
// the field of a tile's cells are first gathered into weights at its nodes
// (the same polynomials), and an atom sums the pair terms of the nodes.
// There, near means that the tiles' columns touch: an atom meets the whole
// z rows of the 3 x 3 tile columns around it directly, in the stages of 256
// cells the direct kernel takes them in.  Every pair of an atom and a cell
// is counted once, by exactly one of the four ways.
//
// Why columns.  A z row that passes close to an atom starts with large terms
// and runs on through hundreds of small ones, whose FP32 rounding is the
// same for neighbouring cells; that, on the rows within 8 A, makes up nearly
// all of the direct kernel's rounding error.  With near tiles in three
// dimensions those small terms went through the nodes and the gradient was
// nine times closer to 64 bits and 1.3 times faster to sum, but further from
// what the direct kernel gives than the rows allow: with the rows kept whole
// the two share their largest rounding.  The grid part of the gradient is 0.6
// to 3.3e-8 (relative 2-norm; 2e-7 on 2048 x 2048 x 4 cells) from the direct
// kernel's for the same field, and both are equally far from 64 bits (rms ratio
// 0.97-1.04 over 16 boxes).
//
// Accuracy: at 16 cells >= 1.2 sigma the interpolation error (rms over
// cells, relative to the sum of the terms' magnitudes) of 12 nodes per axis
// at level 0 is 1e-10 for E and 2e-8 (h = 0.4) to 3e-7 (h = 0.3) for the LJ
// sum, against 3e-8 and 6e-7 of the FP32 rounding of the direct sum; 10
// nodes give 3e-9 and 7e-7 to 2e-6, 8 nodes 6e-8 and 3e-5.  The atoms of
// levels 1 and 2 are twice and four times as far, where the LJ sum is a few
// per cent of U, and take 10 nodes.  Finer grids keep the direct kernels
// (tree_fields_pay).  A node's rounding error is shared by all the cells it
// is interpolated to, so node sums are blocked (128 atoms at a time).
//
// Work per atom.  Fields: 27 x 4096 direct cells, at most 189 x 1728 nodes of
// level 0 and 189 x 1000 of level 1 whatever the grid, and 1000 for each of the
// level-2 tiles not near its own (0.6e6 pair terms and 1/262 of the grid's
// cells; 0.8e6 at 384^3, 4.7e6 at 1024^3).  Gradient: rows of 48 x 48 cells and
// 27 columns of level-0 and level-1 tiles, 2304 + 2916 + 844 pair terms per
// cell of a row's length, and the level-2 tiles outside its 3 x 3 columns as
// above.  The direct kernels meet every cell.
#include <algorithm>
#include <cmath>
#include <vector>

#include "f32x2.cuh"
#include "tree.cuh"
#include "vesis_internal.cuh"

namespace vesis {

constexpr int TC = 16;                  // cells per axis of a level-0 tile
constexpr int kP0 = 12, kP1 = 10;       // nodes per axis: level 0, levels 1 and 2
constexpr int kMaxP = kP0;
__host__ __device__ constexpr int tp(int lev) { return lev == 0 ? kP0 : kP1; }
// values of a tile: four planes of nodes
__host__ __device__ constexpr int tn4(int lev) { return 4 * tp(lev) * tp(lev) * tp(lev); }

// Interpolation tables, FP32 from FP64 (one buffer per system):
//   cell[16][12]    level-0 node polynomials at the 16 cell centres
//   child[l][side][child node][parent node]: the polynomials of a level
//                   l + 1 tile at its level-l child's nodes
//   node[l]         nodes on (-1, 1)
struct TreeTab {
    float cell[TC][kP0];
    float child[2][2][kMaxP][kMaxP];
    float node[3][kMaxP];
};

size_t tree_tab_bytes() { return sizeof(TreeTab); }

void tree_fill_tab(void *host)
{
    TreeTab &t = *static_cast<TreeTab *>(host);
    auto node = [](int P, int k) { return std::cos(M_PI * (k + 0.5) / P); };
    auto basis = [&](int P, double x, float *out) {
        for (int j = 0; j < P; ++j) {
            double v = 1.0;
            for (int k = 0; k < P; ++k)
                if (k != j) v *= (x - node(P, k)) / (node(P, j) - node(P, k));
            out[j] = (float)v;
        }
    };
    for (int l = 0; l < 3; ++l)
        for (int k = 0; k < tp(l); ++k) t.node[l][k] = (float)node(tp(l), k);
    // a level-l tile of T cells spans its cell centres: half-width (T - 1) / 2
    for (int c = 0; c < TC; ++c)
        basis(kP0, (c - 0.5 * (TC - 1)) / (0.5 * (TC - 1)), t.cell[c]);
    for (int l = 0; l < 2; ++l) {
        const double hc = 0.5 * ((TC << l) - 1), hp = 0.5 * ((TC << (l + 1)) - 1);
        const double off = 0.5 * (TC << l);              // child centre from the parent's
        for (int s = 0; s < 2; ++s)
            for (int k = 0; k < tp(l); ++k)
                basis(tp(l + 1), ((s ? off : -off) + node(tp(l), k) * hc) / hp, t.child[l][s][k]);
    }
}

// Tile ids are hierarchical: level-2 tiles row by row (z fastest), 8
// children of each, 8 children of those; a level-l tile is id >> 3 l of its
// level-0 descendants, so the atoms of any tile are one range of the sorted
// order.
__host__ __device__ __forceinline__ int tree_id0(const TreeDims &d, int x, int y, int z)
{
    const int l2 = ((x >> 2) * d.ny + (y >> 2)) * d.nz + (z >> 2);
    const int l1 = ((x >> 1) & 1) * 4 + ((y >> 1) & 1) * 2 + ((z >> 1) & 1);
    const int l0 = (x & 1) * 4 + (y & 1) * 2 + (z & 1);
    return (l2 * 8 + l1) * 8 + l0;
}

// Id of tile (x, y, z) of level LEV, and back.
template <int LEV>
__device__ __forceinline__ int tree_id(const TreeDims &d, int x, int y, int z)
{
    return tree_id0(d, x << LEV, y << LEV, z << LEV) >> (3 * LEV);
}

template <int LEV>
__device__ __forceinline__ void tree_coords(const TreeDims &d, int id, int &x, int &y, int &z)
{
    constexpr int B = 2 - LEV;           // child bits above this level
    const int l2 = id >> (3 * B);
    z = l2 % d.nz;
    y = (l2 / d.nz) % d.ny;
    x = l2 / (d.nz * d.ny);
#pragma unroll
    for (int b = B - 1; b >= 0; --b) {
        const int o = (id >> (3 * b)) & 7;
        x = 2 * x + (o >> 2);
        y = 2 * y + ((o >> 1) & 1);
        z = 2 * z + (o & 1);
    }
}

// Tiles of level lev on an axis of n cells, and the place of tile (x, y, z)
// among the tiles that hold cells (node values are kept for those alone: an id
// also numbers the slots past the grid's end, up to three of four per axis).
__host__ __device__ __forceinline__ int axis_tiles(int n, int lev)
{
    return (n + (TC << lev) - 1) / (TC << lev);
}

template <int LEV>
__device__ __forceinline__ size_t tile_place(const GridDesc &g, int x, int y, int z)
{
    return ((size_t)x * axis_tiles(g.ny, LEV) + y) * axis_tiles(g.nz, LEV) + z;
}

// Cell index of an atom's coordinate on an axis of n cells, clamped into the
// grid.  One function with fixed roundings: every kernel that asks for an
// atom's tile has to get the tile it was sorted into.
__device__ __forceinline__ int atom_cell(float v, float rh, float half, int n)
{
    return min(max((int)floorf(__fmaf_rn(v, rh, half + 0.5f)), 0), n - 1);
}

// Atoms of a level-LEV tile: [first, last) of the sorted order.
template <int LEV>
__device__ __forceinline__ int2 tree_range(const int *off, int id)
{
    return make_int2(off[id << (3 * LEV)], off[(id + 1) << (3 * LEV)]);
}

TreeDims tree_dims(const GridDesc &g)
{
    TreeDims d;
    const int T2 = TC << 2;
    d.nx = (g.nx + T2 - 1) / T2;
    d.ny = (g.ny + T2 - 1) / T2;
    d.nz = (g.nz + T2 - 1) / T2;
    d.n2 = d.nx * d.ny * d.nz;
    return d;
}

// Work items.  A tile's list of far atoms is cut into items of at most `len`
// atoms, so that blocks are alike whatever the density; the kernels launch
// the bound tiles + (all entries) / len and the blocks past the last item
// leave at once.  Lists 0-2: the far atoms of the tiles of levels 0, 1, 2
// (fields).  Lists 3-5: the atoms of the 3 x 3 columns around the tile columns
// of levels 0, 1, 2 (gradient; long lists fill the warps also where a column
// holds few atoms).
TreePlan plan_tree(const GridDesc &g, int n, int nsm, bool force)
{
    TreePlan p;
    p.d = tree_dims(g);
    const long long waves = 16ll * nsm;
    for (int l = 0; l < 3; ++l) {
        const long long slots = (long long)p.d.n2 << (3 * (2 - l));
        const long long per_atom = l == 2 ? p.d.n2 : std::min<long long>(189, slots);
        // tiles that hold cells (slots past the grid's end have no items)
        const long long tiles =
            (long long)axis_tiles(g.nx, l) * axis_tiles(g.ny, l) * axis_tiles(g.nz, l);
        TreeList &f = p.list[l], &m = p.list[3 + l];
        f.tiles = (int)slots;
        f.len = (int)std::max<long long>(256, (n * per_atom + waves - 1) / waves);
        f.max_items = (int)(tiles + n * per_atom / f.len);
        m.tiles = (p.d.nx * p.d.ny) << (2 * (2 - l));
        m.len = l == 0 ? 64 : 128;           // the atoms of a warp
        m.max_items = (int)(m.tiles + 9ll * n / m.len);
    }
    const int ca = (n + 127) / 128;
    p.sf = std::max(1, std::min({p.d.n2, 64, (8 * nsm + ca - 1) / ca}));
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t slots = (size_t)p.d.n2 * 64, cols = (size_t)p.d.nx * p.d.ny * 16;
    p.o_tab = take(tree_tab_bytes());
    p.o_cnt = take((slots + 1) * sizeof(int));
    p.o_off = take((slots + 1) * sizeof(int));
    p.o_cur = take((slots + 1) * sizeof(int));
    p.o_coff = take((cols + 1) * sizeof(int));
    p.o_id = take((size_t)n * sizeof(int));
    p.o_tmp = take((size_t)n * sizeof(int));
    p.o_ord = take((size_t)n * sizeof(int));
    p.o_xyzq = take((size_t)n * sizeof(float4));
    p.o_ab = take((size_t)n * sizeof(float2));
    p.o_cxyz = take((size_t)n * sizeof(float4));
    p.o_cfc = take((size_t)n * sizeof(float4));
    for (TreeList &l : p.list) {
        l.o_first = take(((size_t)l.tiles + 1) * sizeof(int));
        l.o_item = take((size_t)l.max_items * sizeof(int));
    }
    for (int l = 0; l < 3; ++l)     // per item (fields) or per tile with cells (gradient)
        p.o_v[l] = take((size_t)p.list[l].max_items * tn4(l) * sizeof(float));
    if (force)                      // FP64 partials per atom
        p.o_part = take((size_t)(9 * (kRowParts + kZParts0 + kZParts1) + p.sf) * n * 3 *
                        sizeof(double));
    p.bytes = o;
    return p;
}

// Which systems take these kernels: a rule on sizes, spacing and radii for
// each of the two sums.  Fields, direct -> hierarchical in us:
//   N = 400, 171^3 (2.0e9 pairs)     860 ->  450
//   N = 1000, 128^3 (2.1e9)          910 ->  496
//   N = 3000, 150^3 (1.0e10)        4030 -> 1026
// and faster on every shape of box tried at 2e9 pairs and more (1.1 times on 1 x
// 1500 x 1500 cells, 4 to 7 times on long and flat boxes).
// Few atoms round little when summed directly: the rms error against 64 bits
// of the hierarchical fields over the direct ones' (solvent cells, h = 0.3 to
// 0.5, boxes of 2e9 pairs to 384^3, means of three solutes) is, for U and E,
// 0.7-0.9 and 0.9-1.0 at 256 atoms but 1.1-1.4 on the half of the cells far from
// the solute, still up to 1.07 there at 300 and 350, and from 400 atoms on at
// most 0.87 (1.0 far away).  So solutes of fewer than 400 keep the direct sums.
// Interpolation needs every far pair beyond the clamp and the LJ core
// resolved (16 h >= 1.2 sigma keeps its error below FP32's).
constexpr int kTreeAtoms = 400;

bool tree_fields_pay(const GridDesc &g, int n, double h, double rmin, double max_sigma)
{
    const double pairs = (double)g.nx * g.ny * g.nz * n;
    return n >= kTreeAtoms && pairs >= 2.0e9 && TC * h >= 1.2 * max_sigma && TC * h > rmin;
}

// The gradient depends on the shape as well: its near part is whole columns of
// the box, so a long z makes every block's work long, and a box a few columns
// wide has little else.  Both times are estimated (us; fitted to 80 boxes and
// solutes, within 15 % on globules):
//   direct        the pairs with the solvent fraction s of the cells, 1.5e6 a us;
//   hierarchical  440 + 52 per tile of a column (the chains of blocks that do
//                 not fill the chip) + 55 per 1e6 cells (gather and merge) + its
//                 pair terms (rows of the near columns x s, nodes of the others)
//                 at 1.6e6 a us;
//   s             exp(-sum sigma^3 / volume): a packed atom and its share of the
//                 surface take about sigma^3 (globules 0.63-0.99 against 0.50-0.99).
// Measured, direct -> hierarchical in us (s of the tight start):
//   N = 256, 200^3, s 0.98         1336 ->  1790     not taken (pairs)
//   N = 1000, 166^3, 0.77          2392 ->  1994     taken
//   N = 5000, 184^3, 0.69         14575 ->  4595     taken
//   N = 2000, 70 x 70 x 925, 0.74  4383 ->  8316     not taken
//   N = 2000, 925 x 70 x 70, 0.74  4687 ->  1501     taken
//   N = 700, 65 x 65 x 1400, 0.73  2404 ->  8702     not taken
//   N = 2000, 90 x 90 x 359, 0.67  2595 ->  3275     not taken
//   N = 6000, 115 x 115 x 465, 0.59 14481 -> 9997    taken
//   N = 1000, 17 x 600 x 600, 0.69 3028 ->  4056     not taken
//   N = 1000, 600 x 600 x 17, 0.69 3522 ->  1346     taken
// Taken where the estimate is a tenth shorter; never below 4e9 pairs.
bool tree_force_pays(const GridDesc &g, int n, double h, double rmin, double max_sigma,
                     double sum_sigma3)
{
    const double G = (double)g.nx * g.ny * g.nz, pairs = G * n;
    if (pairs < 4.0e9 || !tree_fields_pay(g, n, h, rmin, max_sigma)) return false;
    const double s = std::exp(-sum_sigma3 / (G * h * h * h));
    // tile columns an atom meets at a level: those of the parents' 3 x 3 (level
    // 2: all) but for its own 3 x 3
    auto columns = [&](int lev) {
        const int x = axis_tiles(g.nx, lev), y = axis_tiles(g.ny, lev), w = lev < 2 ? 6 : 1 << 30;
        return (double)std::min(x, w) * std::min(y, w) - std::min(x, 3) * std::min(y, 3);
    };
    double terms = s * std::min(g.nx, 3 * TC) * std::min(g.ny, 3 * TC) * g.nz;
    for (int lev = 0; lev < 3; ++lev)
        terms += columns(lev) * axis_tiles(g.nz, lev) * tp(lev) * tp(lev) * tp(lev);
    const double direct = s * pairs / 1.5e6;
    const double tree = 440.0 + 52.0 * axis_tiles(g.nz, 0) + 55e-6 * G + n * terms / 1.6e6;
    return direct > 1.1 * tree;
}

// ------------------------------------------------------------- sorting
// Atoms are sorted by level-0 tile, by index within a tile, so that every
// sum runs in an order the positions alone decide.  Atoms outside the box
// (a trial step that will be rejected) are clamped into its border tiles:
// they are farther from every tile the border tile is not near.
__global__ void k_tree_count(GridDesc g, TreeDims d, const float4 *__restrict__ xyzq, int n,
                             int *__restrict__ id, int *__restrict__ cnt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 A = xyzq[i];
    const float r = 1.f / g.h;
    const int x = atom_cell(A.x, r, g.cx, g.nx) / TC;
    const int y = atom_cell(A.y, r, g.cy, g.ny) / TC;
    const int z = atom_cell(A.z, r, g.cz, g.nz) / TC;
    const int t = tree_id0(d, x, y, z);
    id[i] = t;
    atomicAdd(cnt + t, 1);
}

__global__ void k_tree_scatter(const int *__restrict__ id, int n, int *__restrict__ cur,
                               int *__restrict__ tmp)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) tmp[atomicAdd(cur + id[i], 1)] = i;
}

// The atoms of a tile arrive in any order; each takes its rank by index.
// vec: the second array to place (LJ constants of the fields, force
// coefficients of the gradient); ord (may be NULL): the sorted atoms' numbers.
template <class T>
__global__ void k_tree_place(const int *__restrict__ tmp, const int *__restrict__ id,
                             const int *__restrict__ off, int n, const float4 *__restrict__ xyzq,
                             const T *__restrict__ vec, int *__restrict__ ord,
                             float4 *__restrict__ xs, T *__restrict__ vs)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int i = tmp[p], t = id[i];
    const int b = off[t], e = off[t + 1];
    int rank = 0;
    for (int q = b; q < e; ++q) rank += tmp[q] < i ? 1 : 0;
    const int o = b + rank;
    if (ord) ord[o] = i;
    xs[o] = xyzq[i];
    vs[o] = vec[i];
}

// Columns of tiles, numbered like the tiles: level-2 columns row by row, 4
// children of each, 4 children of those.
__host__ __device__ __forceinline__ int col_id0(const TreeDims &d, int x, int y)
{
    const int l2 = (x >> 2) * d.ny + (y >> 2);
    return (l2 * 4 + ((x >> 1) & 1) * 2 + ((y >> 1) & 1)) * 4 + (x & 1) * 2 + (y & 1);
}

template <int LEV>
__device__ __forceinline__ void col_coords(const TreeDims &d, int id, int &x, int &y)
{
    constexpr int B = 2 - LEV;
    const int l2 = id >> (2 * B);
    x = l2 / d.ny;
    y = l2 - x * d.ny;
#pragma unroll
    for (int b = B - 1; b >= 0; --b) {
        const int o = (id >> (2 * b)) & 3;
        x = 2 * x + (o >> 1);
        y = 2 * y + (o & 1);
    }
}

__global__ void k_col_count(GridDesc g, TreeDims d, const float4 *__restrict__ xyzq, int n,
                            int *__restrict__ id, int *__restrict__ cnt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 A = xyzq[i];
    const float r = 1.f / g.h;
    const int t = col_id0(d, atom_cell(A.x, r, g.cx, g.nx) / TC, atom_cell(A.y, r, g.cy, g.ny) / TC);
    id[i] = t;
    atomicAdd(cnt + t, 1);
}

// ------------------------------------------------------------ atom lists
// A block's atoms as a list of ranges of the sorted order with their prefix
// sums; entry e of the flattened list is found by bisection.
constexpr int kMaxSeg = 216;            // 27 parents' neighbours x 8 children

struct SegList {
    int first[kMaxSeg];
    int pre[kMaxSeg + 1];
    int nseg;                            // ranges of a level-2 list
};

// Prefix sums of the ranges seg[0 .. nseg) (counts in pre[0 .. nseg) on
// entry) by the whole block; returns the number of atoms.
__device__ __forceinline__ int seg_scan(SegList &L, int nseg)
{
    __syncthreads();
    if (threadIdx.x < 32) {
        int base = 0;
        for (int b = 0; b < nseg; b += 32) {
            const int k = b + threadIdx.x;
            const int v = k < nseg ? L.pre[k] : 0;
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if ((int)threadIdx.x >= o) incl += u;
            }
            if (k < nseg) L.pre[k] = base + incl - v;
            base += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (threadIdx.x == 0) L.pre[nseg] = base;
    }
    __syncthreads();
    return L.pre[nseg];
}

__device__ __forceinline__ int seg_find(const SegList &L, int nseg, int e)
{
    int lo = 0, hi = nseg;               // pre[lo] <= e < pre[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (L.pre[mid] <= e) lo = mid;
        else hi = mid;
    }
    return lo;
}

// The atoms of the 27 tiles around tile (x, y, z) of level LEV; segment s is
// the neighbour at offset (s / 9 - 1, s / 3 % 3 - 1, s % 3 - 1).
template <int LEV>
__device__ __forceinline__ int seg_near(SegList &L, const TreeDims &d, const int *off, int x,
                                        int y, int z)
{
    constexpr int M = 2 - LEV;
    __syncthreads();
    if (threadIdx.x < 27) {
        const int s = threadIdx.x;
        const int a = x + s / 9 - 1, b = y + (s / 3) % 3 - 1, c = z + s % 3 - 1;
        int2 r = make_int2(0, 0);
        if (a >= 0 && b >= 0 && c >= 0 && a < (d.nx << M) && b < (d.ny << M) && c < (d.nz << M))
            r = tree_range<LEV>(off, tree_id<LEV>(d, a, b, c));
        L.first[s] = r.x;
        L.pre[s] = r.y - r.x;
    }
    return seg_scan(L, 27);
}

// Atoms of the 27 tiles around tile (x, y, z) of level LEV.
template <int LEV>
__device__ int near_total(const TreeDims &d, const int *off, int x, int y, int z)
{
    constexpr int M = 2 - LEV;
    int n = 0;
#pragma unroll
    for (int s = 0; s < 27; ++s) {
        const int a = x + s / 9 - 1, b = y + (s / 3) % 3 - 1, c = z + s % 3 - 1;
        if (a >= 0 && b >= 0 && c >= 0 && a < (d.nx << M) && b < (d.ny << M) && c < (d.nz << M)) {
            const int2 r = tree_range<LEV>(off, tree_id<LEV>(d, a, b, c));
            n += r.y - r.x;
        }
    }
    return n;
}

struct PlanArgs {
    int *first[3], *item[3];
    int tiles[3], len[3];
};

// Items of every tile of level LEV: its far atoms are those near its parent
// and not near it (at level 2 all that are not near); a list has at least
// one item (the tile's values must be written).
template <int LEV>
__device__ void plan_tile(const GridDesc &g, const TreeDims &d, const int *off, int natoms,
                          const PlanArgs &P, int id)
{
    constexpr int T = TC << LEV;
    int x, y, z, far = 0;
    tree_coords<LEV>(d, id, x, y, z);
    if (x * T < g.nx && y * T < g.ny && z * T < g.nz) {
        int up = natoms;
        if constexpr (LEV < 2) up = near_total<LEV + 1>(d, off, x >> 1, y >> 1, z >> 1);
        const int n = up - near_total<LEV>(d, off, x, y, z);
        far = max(1, (n + P.len[LEV] - 1) / P.len[LEV]);
    }
    P.first[LEV][id] = far;
}

__global__ void __launch_bounds__(128) k_tree_plan(GridDesc g, TreeDims d,
                                                   const int *__restrict__ off, int natoms,
                                                   PlanArgs P)
{
    int t = blockIdx.x * 128 + threadIdx.x;
    if (t < d.n2 * 64) {
        plan_tile<0>(g, d, off, natoms, P, t);
        return;
    }
    t -= d.n2 * 64;
    if (t < d.n2 * 8) {
        plan_tile<1>(g, d, off, natoms, P, t);
        return;
    }
    t -= d.n2 * 8;
    if (t < d.n2) plan_tile<2>(g, d, off, natoms, P, t);
}

// Exclusive scan of value(0 .. n) into out, the total into out[n], by a block
// of 1024 threads; each(k, start, count) sees every entry.
template <class Value, class Each>
__device__ __forceinline__ void block_scan(Value value, int n, int *out, Each each)
{
    __shared__ int s_w[32];
    __shared__ int s_base;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    for (int b = 0; b < n; b += 4096) {
        int c[4], sum = 0;
        const int at = b + 4 * threadIdx.x;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            c[q] = at + q < n ? value(at + q) : 0;
            sum += c[q];
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) s_w[w] = incl;
        __syncthreads();
        if (w == 0) {
            int t = s_w[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += u;
            }
            s_w[lane] = t;
        }
        __syncthreads();
        int run = s_base + (w ? s_w[w - 1] : 0) + incl - sum;
        const int total = s_w[31];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (at + q < n) {
                out[at + q] = run;
                each(at + q, run, c[q]);
            }
            run += c[q];
        }
        __syncthreads();
        if (threadIdx.x == 0) s_base += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) out[n] = s_base;
}

// Exclusive scan of the tile counts (one block).
__global__ void __launch_bounds__(1024) k_tree_scan(const int *__restrict__ cnt, int slots,
                                                    int *__restrict__ off, int *__restrict__ cur)
{
    block_scan([&](int k) { return cnt[k]; }, slots, off,
               [&](int k, int start, int) { cur[k] = start; });
}

// Item numbers of one list per block, in place, and the items' tiles.
__global__ void __launch_bounds__(1024) k_tree_items(PlanArgs P)
{
    const int q = blockIdx.x;
    int *first = P.first[q], *item = P.item[q];
    block_scan([&](int k) { return first[k]; }, P.tiles[q], first,
               [&](int k, int start, int count) {
                   for (int e = 0; e < count; ++e) item[start + e] = k;
               });
}

// The same for the columns of level blockIdx.x: a column's list holds the
// atoms of the 3 x 3 columns around it.
template <int LEV>
__device__ __forceinline__ int col_id(const TreeDims &d, int x, int y)
{
    return col_id0(d, x << LEV, y << LEV) >> (2 * LEV);
}

template <int LEV>
__device__ __forceinline__ int2 col_range(const TreeDims &d, const int *coff, int x, int y)
{
    constexpr int M = 2 - LEV;
    if (x < 0 || y < 0 || x >= (d.nx << M) || y >= (d.ny << M)) return make_int2(0, 0);
    const int id = col_id<LEV>(d, x, y);
    return make_int2(coff[id << (2 * LEV)], coff[(id + 1) << (2 * LEV)]);
}

template <int LEV>
__device__ void col_items(const GridDesc &g, const TreeDims &d, const int *coff, const PlanArgs &P)
{
    constexpr int T = TC << LEV;
    int *item = P.item[LEV];
    const int len = P.len[LEV];
    block_scan(
        [&](int k) {
            int x, y, n = 0;
            col_coords<LEV>(d, k, x, y);
            if (x * T >= g.nx || y * T >= g.ny) return 0;
#pragma unroll
            for (int s = 0; s < 9; ++s) {
                const int2 r = col_range<LEV>(d, coff, x + s / 3 - 1, y + s % 3 - 1);
                n += r.y - r.x;
            }
            return (n + len - 1) / len;
        },
        P.tiles[LEV], P.first[LEV], [&](int k, int start, int count) {
            for (int e = 0; e < count; ++e) item[start + e] = k;
        });
}

__global__ void __launch_bounds__(1024) k_col_items(GridDesc g, TreeDims d,
                                                    const int *__restrict__ coff, PlanArgs P)
{
    if (blockIdx.x == 0) col_items<0>(g, d, coff, P);
    else if (blockIdx.x == 1) col_items<1>(g, d, coff, P);
    else col_items<2>(g, d, coff, P);
}

// The atoms met at level LEV by tile (x, y, z): those of its parent's
// neighbours' children that it is not near; at level 2 all atoms but the
// near tiles'.
template <int LEV>
__device__ __forceinline__ int seg_far(SegList &L, const TreeDims &d, const int *off, int natoms,
                                       int x, int y, int z, int &nseg)
{
    __syncthreads();
    if (LEV == 2) {
        if (threadIdx.x == 0) {          // the gaps between the rows of near tiles
            int at = 0, m = 0;
            for (int s = 0; s < 9; ++s) {
                const int a = x + s / 3 - 1, b = y + s % 3 - 1;
                if (a < 0 || b < 0 || a >= d.nx || b >= d.ny) continue;
                const int c0 = max(z - 1, 0), c1 = min(z + 1, d.nz - 1);
                const int lo = off[((a * d.ny + b) * d.nz + c0) * 64];
                const int hi = off[((a * d.ny + b) * d.nz + c1 + 1) * 64];
                L.first[m] = at;
                L.pre[m++] = lo - at;
                at = hi;
            }
            L.first[m] = at;
            L.pre[m++] = natoms - at;
            L.nseg = m;
        }
        __syncthreads();
        nseg = L.nseg;
        return seg_scan(L, nseg);
    }
    constexpr int M = 2 - LEV;
    const int px = x >> 1, py = y >> 1, pz = z >> 1;
    for (int s = threadIdx.x; s < kMaxSeg; s += blockDim.x) {
        const int q = s >> 3, o = s & 7;
        const int a = 2 * (px + q / 9 - 1) + (o >> 2), b = 2 * (py + (q / 3) % 3 - 1) + ((o >> 1) & 1),
                  c = 2 * (pz + q % 3 - 1) + (o & 1);
        int2 r = make_int2(0, 0);
        const bool in = a >= 0 && b >= 0 && c >= 0 && a < (d.nx << M) && b < (d.ny << M) &&
                        c < (d.nz << M);
        const bool close = abs(a - x) <= 1 && abs(b - y) <= 1 && abs(c - z) <= 1;
        if (in && !close) r = tree_range<LEV>(off, tree_id<LEV>(d, a, b, c));
        L.first[s] = r.x;
        L.pre[s] = r.y - r.x;
    }
    nseg = kMaxSeg;
    return seg_scan(L, kMaxSeg);
}

static PlanArgs plan_args(const TreePlan &p, uint8_t *ws, int base)
{
    PlanArgs P;
    for (int q = 0; q < 3; ++q) {
        const TreeList &l = p.list[base + q];
        P.first[q] = (int *)(ws + l.o_first);
        P.item[q] = (int *)(ws + l.o_item);
        P.tiles[q] = l.tiles;
        P.len[q] = l.len;
    }
    return P;
}

// Sorts the packed atoms by tile and lists the work items of the fields.
static void launch_tree_sort(const GridDesc &g, const TreePlan &p, uint8_t *ws, const AtomsDev &a,
                             cudaStream_t st)
{
    const int slots = p.d.n2 * 64;
    int *cnt = (int *)(ws + p.o_cnt), *off = (int *)(ws + p.o_off), *cur = (int *)(ws + p.o_cur);
    int *id = (int *)(ws + p.o_id), *tmp = (int *)(ws + p.o_tmp);
    const PlanArgs P = plan_args(p, ws, 0);
    cudaMemsetAsync(cnt, 0, (size_t)slots * sizeof(int), st);
    count_launch(6);
    const unsigned nb = (unsigned)((a.n + 127) / 128);
    k_tree_count<<<nb, 128, 0, st>>>(g, p.d, a.xyzq, a.n, id, cnt);
    k_tree_scan<<<1, 1024, 0, st>>>(cnt, slots, off, cur);
    k_tree_scatter<<<nb, 128, 0, st>>>(id, a.n, cur, tmp);
    k_tree_place<<<nb, 128, 0, st>>>(tmp, id, off, a.n, a.xyzq, a.ab, nullptr,
                                     (float4 *)(ws + p.o_xyzq), (float2 *)(ws + p.o_ab));
    k_tree_plan<<<(unsigned)((p.d.n2 * 73 + 127) / 128), 128, 0, st>>>(g, p.d, off, a.n, P);
    k_tree_items<<<3, 1024, 0, st>>>(P);
}

// Box-centred coordinate of node u of tile t on an axis, T cells per tile.
__device__ __forceinline__ float node_pos(int t, int T, float u, float half, float h)
{
    return ((float)(t * T) + 0.5f * (float)(T - 1) - half + u * (0.5f * (float)(T - 1))) * h;
}

// acc[k] += v row[k] for the N (a multiple of 4) entries of a 16-byte
// aligned row of weights in shared memory.
template <int N>
__device__ __forceinline__ void axpy_row(float (&acc)[N], const float *row, float v)
{
#pragma unroll
    for (int k = 0; k < N; k += 4) {
        const float4 w = *reinterpret_cast<const float4 *>(row + k);
        acc[k] = fmaf(w.x, v, acc[k]);
        acc[k + 1] = fmaf(w.y, v, acc[k + 1]);
        acc[k + 2] = fmaf(w.z, v, acc[k + 2]);
        acc[k + 3] = fmaf(w.w, v, acc[k + 3]);
    }
}

// One axis of a tensor-product transform: a thread's column of NIN values at
// stride S becomes NOUT values out[k] = sum_j M[j][k] in[j] (rows of M padded
// to kMaxP).
template <int NIN, int S>
__device__ __forceinline__ void column(float (&o)[kMaxP], const float *in, const float (*M)[kMaxP])
{
#pragma unroll
    for (int k = 0; k < kMaxP; ++k) o[k] = 0.f;
#pragma unroll 5
    for (int j = 0; j < NIN; ++j) axpy_row<kMaxP>(o, M[j], in[j * S]);
}

// --------------------------------------------------------------- fields
// Node values of a level's tiles: the pair sums of the atoms met at this
// level at the tile's P^3 nodes (one z-pencil of P nodes per thread) plus
// the parent's values interpolated to them.  Bound by the FP32 pipe like the
// direct kernel (11 packed operations per two nodes and 3 per pencil).  One
// block per item (at most `len` atoms of the tile's list); the reader adds a
// tile's items in order.  The sums of every 128 staged atoms are added to
// running sums kept in shared memory, which bounds the rounding of long
// lists (a node's error is common to all the cells around it).
constexpr int TN_TILE = 128;            // atoms staged per pass
__host__ __device__ constexpr int tn_threads(int lev) { return lev == 0 ? 160 : 128; }

template <int LEV>
__global__ void __launch_bounds__(tn_threads(LEV), LEV == 0 ? 4 : 5)
k_tree_nodes(GridDesc g, TreeDims d, const TreeTab *__restrict__ tab, const int *__restrict__ off,
             const int *__restrict__ first, const int *__restrict__ items, int ntiles, AtomsDev a,
             const float *__restrict__ Vp, const int *__restrict__ firstp, float *__restrict__ V)
{
    constexpr int T = TC << LEV, P = tp(LEV), P2 = P * P, P3 = P2 * P, TH = tn_threads(LEV);
    constexpr int H = P / 2;             // packed node pairs of a pencil
    __shared__ __align__(16) AtomPairs s_at[TN_TILE];
    __shared__ f2 s_sum[4 * H][TH];
    __shared__ SegList L;
    __shared__ __align__(16) float s_m[LEV < 2 ? 3 : 1][kP1][kMaxP];   // [axis][parent][child]
    const int item = blockIdx.x;
    if (item >= first[ntiles]) return;
    const int id = items[item], chunk = item - first[id], S = first[id + 1] - first[id];
    int x, y, z;
    tree_coords<LEV>(d, id, x, y, z);
    int nseg;
    const int total = seg_far<LEV>(L, d, off, a.n, x, y, z, nseg);
    const int e0 = (int)((long long)total * chunk / S), e1 = (int)((long long)total * (chunk + 1) / S);
    const int tid = threadIdx.x;
    const f2 zero = pk2(0.f, 0.f);
    f2 run[4][H];
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int p = 0; p < H; ++p) run[f][p] = zero;
    if constexpr (LEV < 2) if (chunk == 0) {
        // the parent's node values (its items added in order), interpolated
        // axis by axis through two buffers over the running sums' area
        constexpr int Q = kP1, Q2 = Q * Q, Q3 = Q2 * Q;
        float *s_a = reinterpret_cast<float *>(&s_sum[0][0]), *s_b = s_a + P2 * Q;
        for (int e = tid; e < 3 * Q * kMaxP; e += TH) {
            const int ax = e / (Q * kMaxP), r = e - ax * Q * kMaxP, j = r / kMaxP, k = r % kMaxP;
            const int side = ax == 0 ? (x & 1) : ax == 1 ? (y & 1) : (z & 1);
            s_m[ax][j][k] = k < P ? tab->child[LEV][side][k][j] : 0.f;
        }
        const int c0 = firstp[id >> 3], c1 = firstp[(id >> 3) + 1];
#pragma unroll 1
        for (int f = 0; f < 4; ++f) {
            for (int e = tid; e < Q3; e += TH) {
                float v = 0.f;
                for (int c = c0; c < c1; ++c) v += Vp[(size_t)c * 4 * Q3 + f * Q3 + e];
                s_a[e] = v;
            }
            __syncthreads();
            float o[kMaxP];
            if (tid < Q2) {
                column<Q, Q2>(o, s_a + tid, s_m[0]);
#pragma unroll
                for (int k = 0; k < P; ++k) s_b[k * Q2 + tid] = o[k];
            }
            __syncthreads();
            if (tid < P * Q) {
                const int k0 = tid / Q, c = tid - k0 * Q;
                column<Q, Q>(o, s_b + k0 * Q2 + c, s_m[1]);
#pragma unroll
                for (int k = 0; k < P; ++k) s_a[(k0 * P + k) * Q + c] = o[k];
            }
            __syncthreads();
            if (tid < P2) {
                column<Q, 1>(o, s_a + tid * Q, s_m[2]);
#pragma unroll
                for (int ff = 0; ff < 4; ++ff)       // (static register indices)
                    if (ff == f)
#pragma unroll
                        for (int p = 0; p < H; ++p) run[ff][p] = pk2(o[2 * p], o[2 * p + 1]);
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int p = 0; p < H; ++p) s_sum[f * H + p][tid] = run[f][p];
    const int t = min(tid, P2 - 1);
    const int ia = t / P, ib = t - ia * P;
    const float px = node_pos(x, T, tab->node[LEV][ia], g.cx, g.h);
    const float py = node_pos(y, T, tab->node[LEV][ib], g.cy, g.h);
    f2 pz[H];
#pragma unroll
    for (int p = 0; p < H; ++p)
        pz[p] = pk2(node_pos(z, T, tab->node[LEV][2 * p], g.cz, g.h),
                    node_pos(z, T, tab->node[LEV][2 * p + 1], g.cz, g.h));
    const f2 px2 = pk2(px, px), py2 = pk2(py, py);
    for (int base = e0; base < e1; base += TN_TILE) {
        const int cnt = min(TN_TILE, e1 - base);
        __syncthreads();
        for (int m = tid; m < cnt; m += TH) {
            const int e = base + m, s = seg_find(L, nseg, e);
            const int i = L.first[s] + (e - L.pre[s]);
            const float4 A = a.xyzq[i];
            const float2 B = a.ab[i];
            AtomPairs at;
            at.x = pk2(A.x, A.x);
            at.y = pk2(A.y, A.y);
            at.z = pk2(A.z, A.z);
            at.q = pk2(A.w, A.w);
            at.a = pk2(B.x, B.x);
            at.nb = pk2(-B.y, -B.y);
            s_at[m] = at;
        }
        __syncthreads();
        f2 acc[4][H];
#pragma unroll
        for (int f = 0; f < 4; ++f)
#pragma unroll
            for (int p = 0; p < H; ++p) acc[f][p] = zero;
#pragma unroll 1
        for (int m = 0; m < cnt; ++m)
            energy_atom<false, P>(s_at[m], px2, py2, pz, 0.f, acc[0], acc[1], acc[2], acc[3]);
#pragma unroll
        for (int f = 0; f < 4; ++f)
#pragma unroll
            for (int p = 0; p < H; ++p)
                s_sum[f * H + p][tid] = add2(s_sum[f * H + p][tid], acc[f][p]);
    }
    if (tid < P2) {
        float *W = V + (size_t)item * 4 * P3 + tid * P;
#pragma unroll
        for (int f = 0; f < 4; ++f)
#pragma unroll
            for (int p = 0; p < H; ++p) {
                float v0, v1;
                upk2(s_sum[f * H + p][tid], v0, v1);
                *reinterpret_cast<float2 *>(W + f * P3 + 2 * p) = make_float2(v0, v1);
            }
    }
}

// Cells of a level-0 tile: the tile's node values interpolated to them plus
// the direct pairs of the atoms in the 27 near tiles.  Four blocks per tile
// (4 x-planes of 16 x 16 cells each); a thread owns 8 cells of a z-pencil.
// The results leave through shared memory as whole rows of 16 cells, so
// that any alignment of the rows writes full sectors.
constexpr int TP = kP0, TP2 = TP * TP, TP3 = TP2 * TP, TN4 = 4 * TP3;   // level 0
constexpr int TL_THREADS = 128;
constexpr int TL_X = 4;                 // x-planes per block
constexpr int TL_TILE = 128;            // atoms staged per pass

__global__ void __launch_bounds__(TL_THREADS, 4)
k_tree_cells(GridDesc g, TreeDims d, const TreeTab *__restrict__ tab, const int *__restrict__ off,
             AtomsDev a, const float *__restrict__ V, const int *__restrict__ first, float rho,
             float cfa, float rmin2, float *__restrict__ U, float *__restrict__ Ex, float *__restrict__ Ey,
             float *__restrict__ Ez)
{
    // node values, then the y-interpolated planes; afterwards the staged atoms
    // and the outgoing rows
    __shared__ __align__(16) float s_buf[TN4];
    __shared__ __align__(16) float s_x[4 * TL_X * TP2];
    __shared__ __align__(16) float s_zc[TP][TC];       // [node][cell]
    __shared__ SegList L;
    const int id = blockIdx.x >> 2, part = blockIdx.x & 3;
    int x, y, z;
    tree_coords<0>(d, id, x, y, z);
    const int i0 = x * TC + part * TL_X, j0 = y * TC, k0 = z * TC;
    if (i0 >= g.nx || j0 >= g.ny || k0 >= g.nz) return;
    const int total = seg_near<0>(L, d, off, x, y, z);
    for (int e = threadIdx.x; e < TC * TP; e += TL_THREADS)
        s_zc[e % TP][e / TP] = (&tab->cell[0][0])[e];
    const int c0 = first[id], c1 = first[id + 1];
    const float *P = V + (size_t)c0 * TN4;
    for (int e = threadIdx.x; e < TN4 / 4; e += TL_THREADS) {
        float4 v = reinterpret_cast<const float4 *>(P)[e];
        for (int c = c0 + 1; c < c1; ++c) {
            const float4 u = reinterpret_cast<const float4 *>(V + (size_t)c * TN4)[e];
            v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
        }
        reinterpret_cast<float4 *>(s_buf)[e] = v;
    }
    __syncthreads();
    // x: [12][12][12] -> [4][12][12] per field
#pragma unroll 1
    for (int e = threadIdx.x; e < 4 * TP2; e += TL_THREADS) {
        const int f = e / TP2, r = e - f * TP2;
        float o[TL_X] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < TP; ++k)
            axpy_row<TL_X>(o, &s_zc[k][part * TL_X], s_buf[f * TP3 + k * TP2 + r]);
#pragma unroll
        for (int q = 0; q < TL_X; ++q) s_x[(f * TL_X + q) * TP2 + r] = o[q];
    }
    __syncthreads();
    // y: -> [4][16][12] per field, over the node values
    float *s_y = s_buf;
#pragma unroll 1
    for (int e = threadIdx.x; e < 4 * TL_X * TP; e += TL_THREADS) {
        const int fq = e / TP, c = e - fq * TP;
        float o[TC];
#pragma unroll
        for (int r = 0; r < TC; ++r) o[r] = 0.f;
#pragma unroll 3
        for (int k = 0; k < TP; ++k) axpy_row<TC>(o, s_zc[k], s_x[fq * TP2 + k * TP + c]);
#pragma unroll
        for (int r = 0; r < TC; ++r) s_y[(fq * TC + r) * TP + c] = o[r];
    }
    __syncthreads();
    // z: the thread's 8 cells
    const int q = threadIdx.x >> 5, r = (threadIdx.x & 31) >> 1, zh = threadIdx.x & 1;
    f2 acc[4][4];
    const f2 zero = pk2(0.f, 0.f);
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[f][p] = zero;
#pragma unroll 2
    for (int c = 0; c < TP; ++c) {
        const f2 *w = reinterpret_cast<const f2 *>(&s_zc[c][8 * zh]);
        const f2 w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const float v = s_y[((f * TL_X + q) * TC + r) * TP + c];
            const f2 v2 = pk2(v, v);
            acc[f][0] = fma2(w0, v2, acc[f][0]);
            acc[f][1] = fma2(w1, v2, acc[f][1]);
            acc[f][2] = fma2(w2, v2, acc[f][2]);
            acc[f][3] = fma2(w3, v2, acc[f][3]);
        }
    }
    // direct pairs
    const float px = cell_pos(i0 + q, g.cx, g.h), py = cell_pos(j0 + r, g.cy, g.h);
    f2 pz[4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
        pz[p] = pk2(cell_pos(k0 + 8 * zh + 2 * p, g.cz, g.h),
                    cell_pos(k0 + 8 * zh + 2 * p + 1, g.cz, g.h));
    const f2 px2 = pk2(px, px), py2 = pk2(py, py);
    AtomPairs *s_at = reinterpret_cast<AtomPairs *>(s_buf);
    static_assert(sizeof(AtomPairs) * TL_TILE <= sizeof(float) * TN4, "staged atoms fit");
    for (int base = 0; base < total; base += TL_TILE) {
        const int cnt = min(TL_TILE, total - base);
        __syncthreads();
        for (int m = threadIdx.x; m < cnt; m += TL_THREADS) {
            const int e = base + m, s = seg_find(L, 27, e);
            const int i = L.first[s] + (e - L.pre[s]);
            const float4 A = a.xyzq[i];
            const float2 B = a.ab[i];
            AtomPairs at;
            at.x = pk2(A.x, A.x);
            at.y = pk2(A.y, A.y);
            at.z = pk2(A.z, A.z);
            at.q = pk2(A.w, A.w);
            at.a = pk2(B.x, B.x);
            at.nb = pk2(-B.y, -B.y);
            s_at[m] = at;
        }
        __syncthreads();
#pragma unroll 2
        for (int m = 0; m < cnt; ++m)
            energy_atom<true, 8>(s_at[m], px2, py2, pz, rmin2, acc[0], acc[1], acc[2], acc[3]);
    }
    __syncthreads();
    // rows out: plane p of the four fields at s_out[p][x][y][z]
    float *s_out = s_buf;
    const int at = threadIdx.x * 8;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        float l[2], u[2], v[2], w[2];
        upk2(acc[0][p], l[0], l[1]);
        upk2(acc[1][p], u[0], u[1]);
        upk2(acc[2][p], v[0], v[1]);
        upk2(acc[3][p], w[0], w[1]);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const float e2 = fmaf(u[hh], u[hh], fmaf(v[hh], v[hh], w[hh] * w[hh]));
            l[hh] = fmaf(cfa, e2, rho * l[hh]);
        }
        *reinterpret_cast<float2 *>(s_out + at + 2 * p) = make_float2(l[0], l[1]);
        *reinterpret_cast<float2 *>(s_out + 1024 + at + 2 * p) = make_float2(u[0], u[1]);
        *reinterpret_cast<float2 *>(s_out + 2048 + at + 2 * p) = make_float2(v[0], v[1]);
        *reinterpret_cast<float2 *>(s_out + 3072 + at + 2 * p) = make_float2(w[0], w[1]);
    }
    __syncthreads();
    const long long nyz = (long long)g.ny * g.nz;
    const int zz = threadIdx.x & 15;
    if (k0 + zz < g.nz)
        for (int row = threadIdx.x >> 4; row < TL_X * TC; row += TL_THREADS / 16) {
            const int i = i0 + (row >> 4), j = j0 + (row & 15);
            if (i >= g.nx || j >= g.ny) continue;
            const long long o = (long long)i * nyz + (long long)j * g.nz + k0 + zz;
            const int e = row * 16 + zz;
            U[o] = s_out[e];
            Ex[o] = s_out[1024 + e];
            Ey[o] = s_out[2048 + e];
            Ez[o] = s_out[3072 + e];
        }
}

void launch_tree_fields(const GridDesc &g, const TreePlan &p, uint8_t *ws, const AtomsDev &atoms,
                        float rho, float cfa, float rmin2, float *U, float *Ex, float *Ey,
                        float *Ez, cudaStream_t st)
{
    launch_tree_sort(g, p, ws, atoms, st);
    AtomsDev a;
    a.n = atoms.n;
    a.xyzq = (const float4 *)(ws + p.o_xyzq);
    a.ab = (const float2 *)(ws + p.o_ab);
    a.fcoef = nullptr;
    const TreeTab *tab = (const TreeTab *)(ws + p.o_tab);
    const int *off = (const int *)(ws + p.o_off);
    float *V[3];
    const int *first[3], *item[3];
    for (int l = 0; l < 3; ++l) {
        V[l] = (float *)(ws + p.o_v[l]);
        first[l] = (const int *)(ws + p.list[l].o_first);
        item[l] = (const int *)(ws + p.list[l].o_item);
    }
    count_launch(4);
    k_tree_nodes<2><<<p.list[2].max_items, tn_threads(2), 0, st>>>(
        g, p.d, tab, off, first[2], item[2], p.list[2].tiles, a, nullptr, nullptr, V[2]);
    k_tree_nodes<1><<<p.list[1].max_items, tn_threads(1), 0, st>>>(
        g, p.d, tab, off, first[1], item[1], p.list[1].tiles, a, V[2], first[2], V[1]);
    k_tree_nodes<0><<<p.list[0].max_items, tn_threads(0), 0, st>>>(
        g, p.d, tab, off, first[0], item[0], p.list[0].tiles, a, V[1], first[1], V[0]);
    k_tree_cells<<<(unsigned)p.d.n2 * 256, TL_THREADS, 0, st>>>(g, p.d, tab, off, a, V[0], first[0],
                                                                rho, cfa, rmin2, U, Ex, Ey, Ez);
}

// ------------------------------------------------------------- gradient
// Node weights of a level-0 tile: M[k] = sum over its cells of the product
// polynomial of node k times (solvent mask, E masked) - the transpose of the
// interpolation in k_tree_cells.  Four x-planes at a time: z (a thread's 8
// cells and its partner's), y, then x into registers.  Streams chi and E
// once (13 bytes per cell).
__global__ void __launch_bounds__(128, 4)
k_tree_gather(GridDesc g, TreeDims d, const TreeTab *__restrict__ tab,
              const uint8_t *__restrict__ chi, const float *__restrict__ Ex,
              const float *__restrict__ Ey, const float *__restrict__ Ez, float *__restrict__ V,
              unsigned long long *__restrict__ nsolvent)
{
    __shared__ __align__(16) float s_cell[TC][TP];     // [cell][node]
    __shared__ float s_z[4 * TL_X * TC * TP];      // [f][x][y][c]
    __shared__ float s_y[4 * TL_X * TP2];          // [f][x][b][c]
    const int id = blockIdx.x;
    int x, y, z;
    tree_coords<0>(d, id, x, y, z);
    if (x * TC >= g.nx || y * TC >= g.ny || z * TC >= g.nz) return;
    for (int e = threadIdx.x; e < TC * TP; e += 128) (&s_cell[0][0])[e] = (&tab->cell[0][0])[e];
    const int q = threadIdx.x >> 5, r = (threadIdx.x & 31) >> 1, zh = threadIdx.x & 1;
    const long long nyz = (long long)g.ny * g.nz;
    const int j = y * TC + r, kb = z * TC + 8 * zh;
    constexpr int NC = (4 * TP2 + 127) / 128;      // (f, b, c) columns per thread
    float acc[NC][TP];
#pragma unroll
    for (int m = 0; m < NC; ++m)
#pragma unroll
        for (int k = 0; k < TP; ++k) acc[m][k] = 0.f;
    unsigned seen = 0;
    __syncthreads();
#pragma unroll 1
    for (int xg = 0; xg < TC; xg += TL_X) {
        if (x * TC + xg >= g.nx) break;
        const int i = x * TC + xg + q;
        float v[4][8];
        const bool row = i < g.nx && j < g.ny;
        const long long o = (long long)i * nyz + (long long)j * g.nz + kb;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const bool s = row && kb + e < g.nz && chi[o + e] == 0;
            v[0][e] = s ? 1.f : 0.f;
            v[1][e] = s ? Ex[o + e] : 0.f;
            v[2][e] = s ? Ey[o + e] : 0.f;
            v[3][e] = s ? Ez[o + e] : 0.f;
            seen += s ? 1u : 0u;
        }
#pragma unroll 2
        for (int c = 0; c < TP; ++c) {
            float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float w = s_cell[8 * zh + e][c];
#pragma unroll
                for (int f = 0; f < 4; ++f) t[f] = fmaf(w, v[f][e], t[f]);
            }
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                t[f] += __shfl_xor_sync(0xffffffffu, t[f], 1);
                if ((c & 1) == zh) s_z[((f * TL_X + q) * TC + r) * TP + c] = t[f];
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int e = threadIdx.x; e < 4 * TL_X * TP; e += 128) {
            const int fq = e / TP, c = e - fq * TP;
            float u[TP];
#pragma unroll
            for (int b = 0; b < TP; ++b) u[b] = 0.f;
#pragma unroll 4
            for (int yy = 0; yy < TC; ++yy)
                axpy_row<TP>(u, s_cell[yy], s_z[(fq * TC + yy) * TP + c]);
#pragma unroll
            for (int b = 0; b < TP; ++b) s_y[fq * TP2 + b * TP + c] = u[b];
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const int e = threadIdx.x + 128 * m;
            if (e < 4 * TP2) {
                const int f = e / TP2, bc = e - f * TP2;
#pragma unroll
                for (int qq = 0; qq < TL_X; ++qq)
                    axpy_row<TP>(acc[m], s_cell[xg + qq], s_y[(f * TL_X + qq) * TP2 + bc]);
            }
        }
    }
    float *W = V + tile_place<0>(g, x, y, z) * TN4;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const int e = threadIdx.x + 128 * m;
        if (e < 4 * TP2) {
            const int f = e / TP2, bc = e - f * TP2;
#pragma unroll
            for (int k = 0; k < TP; ++k) W[f * TP3 + k * TP2 + bc] = acc[m][k];
        }
    }
    if (nsolvent) {
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) seen += __shfl_down_sync(0xffffffffu, seen, s);
        if ((threadIdx.x & 31) == 0 && seen) atomicAdd(nsolvent, (unsigned long long)seen);
    }
}

// Node weights of a level-LEV tile from its eight children's, one plane
// (blockIdx.y) per block: each child's nodes go through the transposed
// polynomials axis by axis, and the last axis adds into registers.
template <int LEV>
__global__ void __launch_bounds__(160)
k_tree_merge(GridDesc g, TreeDims d, const TreeTab *__restrict__ tab,
             const float *__restrict__ Vc, float *__restrict__ V)
{
    constexpr int T = TC << LEV, C = tp(LEV - 1), C2 = C * C, C3 = C2 * C;    // child nodes
    constexpr int P = tp(LEV), P2 = P * P, P3 = P2 * P;
    __shared__ float s_a[C3], s_b[C2 * P];
    __shared__ __align__(16) float s_m[2][C][kMaxP];    // [side][child][parent]
    const int id = blockIdx.x, f = blockIdx.y, t = threadIdx.x;
    int x, y, z;
    tree_coords<LEV>(d, id, x, y, z);
    if (x * T >= g.nx || y * T >= g.ny || z * T >= g.nz) return;
    for (int e = t; e < 2 * C * kMaxP; e += 160)
        (&s_m[0][0][0])[e] = e % kMaxP < P
                                 ? tab->child[LEV - 1][e / (C * kMaxP)][(e / kMaxP) % C][e % kMaxP]
                                 : 0.f;
    constexpr int NV = (C3 + 159) / 160;
    float nx[NV];                        // the next child's values, in flight
    auto inside = [&](int o) {
        return (2 * x + (o >> 2)) * (T / 2) < g.nx && (2 * y + ((o >> 1) & 1)) * (T / 2) < g.ny &&
               (2 * z + (o & 1)) * (T / 2) < g.nz;
    };
    auto fetch = [&](int o) {
        const bool ok = o < 8 && inside(o);
        const float *p = Vc + tile_place<LEV - 1>(g, 2 * x + (o >> 2), 2 * y + ((o >> 1) & 1),
                                                  2 * z + (o & 1)) * 4 * C3 + (size_t)f * C3;
#pragma unroll
        for (int m = 0; m < NV; ++m) nx[m] = ok && t + 160 * m < C3 ? __ldg(p + t + 160 * m) : 0.f;
    };
    float acc[P];
#pragma unroll
    for (int k = 0; k < P; ++k) acc[k] = 0.f;
    fetch(0);
#pragma unroll 1
    for (int o = 0; o < 8; ++o) {
#pragma unroll
        for (int m = 0; m < NV; ++m)
            if (t + 160 * m < C3) s_a[t + 160 * m] = nx[m];
        __syncthreads();
        fetch(o + 1);
        if (!inside(o)) {
            __syncthreads();
            continue;
        }
        float v[kMaxP];
        if (t < C2) {                    // z: [C][C][C] -> [C][C][P]
            column<C, 1>(v, s_a + t * C, s_m[o & 1]);
#pragma unroll
            for (int k = 0; k < P; ++k) s_b[t * P + k] = v[k];
        }
        __syncthreads();
        if (t < C * P) {                 // y: -> [C][P][P]
            const int i = t / P, c = t - i * P;
            column<C, P>(v, s_b + i * C * P + c, s_m[(o >> 1) & 1]);
#pragma unroll
            for (int k = 0; k < P; ++k) s_a[(i * P + k) * P + c] = v[k];
        }
        __syncthreads();
        if (t < P2) {                    // x: -> [P][P][P]
            column<C, P2>(v, s_a + t, s_m[o >> 2]);
#pragma unroll
            for (int k = 0; k < P; ++k) acc[k] += v[k];
        }
        __syncthreads();
    }
    if (t < P2) {
        float *W = V + tile_place<LEV>(g, x, y, z) * 4 * P3 + (size_t)f * P3;
#pragma unroll
        for (int k = 0; k < P; ++k) W[k * P2 + t] = acc[k];
    }
}

// A warp's 64 PAIRS atoms of a list, two per lane and packed pair.
constexpr int TF_WARPS = 4;
constexpr int TF_THREADS = 32 * TF_WARPS;

struct ColAtoms {
    const float4 *xyzq, *fcoef;          // sorted by column
    int n;
};

// The atoms of the 3 x 3 columns around column (x, y) of level LEV; segment
// s is the column at offset (s / 3 - 1, s % 3 - 1).
template <int LEV>
__device__ __forceinline__ int seg_cols(SegList &L, const TreeDims &d, const int *coff, int x, int y)
{
    __syncthreads();
    if (threadIdx.x < 9) {
        const int s = threadIdx.x;
        const int2 r = col_range<LEV>(d, coff, x + s / 3 - 1, y + s % 3 - 1);
        L.first[s] = r.x;
        L.pre[s] = r.y - r.x;
    }
    return seg_scan(L, 9);
}

template <int PAIRS>
struct LaneAtoms {
    f2 x[PAIRS], y[PAIRS], z[PAIRS], c1[PAIRS], c2[PAIRS], kq[PAIRS];
    int idx[2 * PAIRS];                  // sorted index, or -1
    int seg[2 * PAIRS];
};

// Loads list entries base + lane + 32 u; idle lanes sit far away with zero
// coefficients.
template <int PAIRS>
__device__ __forceinline__ void load_atoms(LaneAtoms<PAIRS> &A, const SegList &L, int nseg,
                                           const ColAtoms &a, int base, int total)
{
    const int lane = threadIdx.x & 31;
    float v[2 * PAIRS][6];
#pragma unroll
    for (int u = 0; u < 2 * PAIRS; ++u) {
        const int e = base + lane + 32 * u;
        A.idx[u] = -1;
        A.seg[u] = 0;
        v[u][0] = v[u][1] = v[u][2] = 1.0e6f;
        v[u][3] = v[u][4] = v[u][5] = 0.f;
        if (e < total) {
            const int s = seg_find(L, nseg, e);
            const int i = L.first[s] + (e - L.pre[s]);
            const float4 X = a.xyzq[i], F = a.fcoef[i];
            A.idx[u] = i;
            A.seg[u] = s;
            v[u][0] = X.x; v[u][1] = X.y; v[u][2] = X.z;
            v[u][3] = F.x; v[u][4] = F.y; v[u][5] = F.z;
        }
    }
#pragma unroll
    for (int p = 0; p < PAIRS; ++p) {
        A.x[p] = pk2(v[2 * p][0], v[2 * p + 1][0]);
        A.y[p] = pk2(v[2 * p][1], v[2 * p + 1][1]);
        A.z[p] = pk2(v[2 * p][2], v[2 * p + 1][2]);
        A.c1[p] = pk2(v[2 * p][3], v[2 * p + 1][3]);
        A.c2[p] = pk2(v[2 * p][4], v[2 * p + 1][4]);
        A.kq[p] = pk2(v[2 * p][5], v[2 * p + 1][5]);
    }
}

// The warps' double-float sums, added over the warps in FP64 and written to
// partial slot(u) of atom u.
template <int PAIRS, class Slot>
__device__ __forceinline__ void store_parts(const LaneAtoms<PAIRS> &A, const f2 (&hi)[PAIRS][3],
                                            const f2 (&lo)[PAIRS][3], double *s_acc, int natoms,
                                            double *part, Slot slot)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PAIRS; ++p)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float h0, h1, l0, l1;
            upk2(hi[p][c], h0, h1);
            upk2(lo[p][c], l0, l1);
            s_acc[((w * 2 * PAIRS + 2 * p) * 3 + c) * 32 + lane] = (double)h0 + (double)l0;
            s_acc[((w * 2 * PAIRS + 2 * p + 1) * 3 + c) * 32 + lane] = (double)h1 + (double)l1;
        }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int u = 0; u < 2 * PAIRS; ++u) {
            if (A.idx[u] < 0) continue;
            double *o = part + ((size_t)slot(u) * natoms + A.idx[u]) * 3;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                double t = 0.0;
#pragma unroll
                for (int q = 0; q < TF_WARPS; ++q)
                    t += s_acc[((q * 2 * PAIRS + u) * 3 + c) * 32 + lane];
                o[c] = t;
            }
        }
    }
}

// Direct gradient pairs: an item is 64 atoms of the 3 x 3 columns around a
// level-0 column, met by the column's z rows; blockIdx.y takes 8 of the 16 x
// planes, a warp every fourth.  The 16 rows of a plane are one run of the
// linear index; a warp walks it in the direct kernel's stages (256
// cells from a multiple of 256), compacts a stage's solvent cells by ballot
// into its own shared area and sums them as that kernel does: pencil by
// pencil in one FP32 run per stage and cell group (cg groups of every cg-th
// cell), into double-float accumulators.  No barrier between warps.  FP32
// pipe: 18 packed operations per two pairs.
constexpr int kStage = 256;
constexpr int kPlanes = TC / kRowParts; // x planes per part

template <bool CLAMP, int PAIRS>
__device__ __forceinline__ void row_cells(const CellQuad *s_c, int first, int en, int cg,
                                          const LaneAtoms<PAIRS> &A, const f2 (&dx)[PAIRS],
                                          const f2 (&dy)[PAIRS], const f2 (&dxy2)[PAIRS],
                                          const f2 (&nk3)[PAIRS], float rmin2, f2 (&sc)[PAIRS],
                                          f2 (&fz)[PAIRS], f2 (&gx)[PAIRS], f2 (&gy)[PAIRS],
                                          f2 (&gz)[PAIRS])
{
#pragma unroll 4
    for (int e = first; e < en; e += cg) {
        const CellQuad c = s_c[e];
#pragma unroll
        for (int p = 0; p < PAIRS; ++p)
            grad_pair2<CLAMP>(c, dx[p], dy[p], dxy2[p], A.z[p], A.c1[p], A.c2[p], nk3[p], rmin2,
                              sc[p], fz[p], gx[p], gy[p], gz[p]);
    }
}

__global__ void __launch_bounds__(TF_THREADS, 4)
k_tree_force_rows(GridDesc g, TreeDims d, const int *__restrict__ coff,
                  const int *__restrict__ first, const int *__restrict__ items, int ncols,
                  const uint8_t *__restrict__ chi, const float *__restrict__ Ex,
                  const float *__restrict__ Ey, const float *__restrict__ Ez, ColAtoms a,
                  float rmin2, int cg, double *__restrict__ part)
{
    constexpr int PAIRS = 1;
    __shared__ __align__(16) CellQuad s_c[TF_WARPS][kStage];
    __shared__ double s_acc[TF_WARPS * 2 * PAIRS * 3 * 32];
    __shared__ SegList L;
    const int item = blockIdx.x;
    if (item >= first[ncols]) return;
    const int id = items[item];
    int X, Y;
    col_coords<0>(d, id, X, Y);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    LaneAtoms<PAIRS> A;
    const int total = seg_cols<0>(L, d, coff, X, Y);
    load_atoms(A, L, 9, a, 64 * PAIRS * (item - first[id]), total);
    const f2 zero = pk2(0.f, 0.f), m3 = pk2(-3.f, -3.f);
    f2 nk3[PAIRS], hi[PAIRS][3], lo[PAIRS][3];
    // box of the warp's atoms, for the clamp test of a stage
    float bl[3] = {1e30f, 1e30f, 1e30f}, bh[3] = {-1e30f, -1e30f, -1e30f};
#pragma unroll
    for (int p = 0; p < PAIRS; ++p) {
        nk3[p] = mul2(m3, A.kq[p]);
#pragma unroll
        for (int c = 0; c < 3; ++c) hi[p][c] = lo[p][c] = zero;
        float v[3][2];
        upk2(A.x[p], v[0][0], v[0][1]);
        upk2(A.y[p], v[1][0], v[1][1]);
        upk2(A.z[p], v[2][0], v[2][1]);
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (A.idx[2 * p + e] >= 0)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    bl[c] = fminf(bl[c], v[c][e]);
                    bh[c] = fmaxf(bh[c], v[c][e]);
                }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            bl[c] = fminf(bl[c], __shfl_xor_sync(0xffffffffu, bl[c], o));
            bh[c] = fmaxf(bh[c], __shfl_xor_sync(0xffffffffu, bh[c], o));
        }
    const int j0 = TC * Y, j1 = min(TC * (Y + 1), g.ny);
    const int ia = TC * X + kPlanes * blockIdx.y;
#pragma unroll 1
    for (int i = ia + w; i < min(ia + kPlanes, g.nx); i += TF_WARPS) {
        const long long lo0 = ((long long)i * g.ny + j0) * g.nz, hi0 = ((long long)i * g.ny + j1) * g.nz;
        const float xx = cell_pos(i, g.cx, g.h);
        const f2 x2 = pk2(xx, xx);
        const float gapx = fmaxf(fmaxf(bl[0] - xx, xx - bh[0]), 0.f);
#pragma unroll 1
        for (long long s = lo0 / kStage * kStage; s < hi0; s += kStage) {
            unsigned bal[kStage / 32];
            int n = 0;
            // pencil and z of the stage's first cell of the run
            const long long b0 = max(s, lo0);
            const int lim = (int)(min(s + kStage, hi0) - s);
            int j = j0 + (int)(b0 - lo0) / g.nz;
            int k = (int)(b0 - lo0) % g.nz;
            __syncwarp();                // the previous stage is no longer read
#pragma unroll
            for (int v = 0; v < kStage / 32; ++v) {
                const int at = 32 * v + lane;
                const long long o = s + at;
                const bool in = o >= lo0 && at < lim && chi[o] == 0;
                bal[v] = __ballot_sync(0xffffffffu, in);
                if (in) {
                    const int kk = (int)(o - lo0) % g.nz;
                    const float zz = cell_pos(kk, g.cz, g.h);
                    CellQuad c;
                    c.z = pk2(zz, zz);
                    const float e0 = Ex[o], e1 = Ey[o], e2 = Ez[o];
                    c.ex = pk2(e0, e0);
                    c.ey = pk2(e1, e1);
                    c.ez = pk2(e2, e2);
                    s_c[w][n + __popc(bal[v] & ((1u << lane) - 1u))] = c;
                }
                n += __popc(bal[v]);
            }
            __syncwarp();
            if (n == 0) continue;
            // cells of the first m slots of the stage
            auto rank = [&](int m) {
                int r = 0;
#pragma unroll
                for (int v = 0; v < kStage / 32; ++v) {
                    const int left = m - 32 * v;
                    const unsigned mask = left >= 32 ? 0xffffffffu : left > 0 ? (1u << left) - 1u : 0u;
                    r += __popc(bal[v] & mask);
                }
                return r;
            };
#pragma unroll 1
            for (int grp = 0; grp < cg; ++grp) {
                f2 fx[PAIRS], fy[PAIRS], fz[PAIRS], gx[PAIRS], gy[PAIRS], gz[PAIRS];
#pragma unroll
                for (int p = 0; p < PAIRS; ++p)
                    fx[p] = fy[p] = fz[p] = gx[p] = gy[p] = gz[p] = zero;
                int at = (int)(b0 - s), jj = j, kk = k, st = 0;
#pragma unroll 1
                while (at < lim) {       // the pencils of the stage
                    const int next = min(at + g.nz - kk, lim);
                    const int en = rank(next);
                    if (en > st) {
                        const float yy = cell_pos(jj, g.cy, g.h);
                        const float z0 = cell_pos(kk, g.cz, g.h),
                                    z1 = cell_pos(kk + next - at - 1, g.cz, g.h);
                        const float gy0 = fmaxf(fmaxf(bl[1] - yy, yy - bh[1]), 0.f);
                        const float gz0 = fmaxf(fmaxf(bl[2] - z1, z0 - bh[2]), 0.f);
                        const f2 y2 = pk2(yy, yy);
                        f2 dx[PAIRS], dy[PAIRS], dxy2[PAIRS], sc[PAIRS];
#pragma unroll
                        for (int p = 0; p < PAIRS; ++p) {
                            dx[p] = sub2(x2, A.x[p]);
                            dy[p] = sub2(y2, A.y[p]);
                            dxy2[p] = fma2(dx[p], dx[p], mul2(dy[p], dy[p]));
                            sc[p] = zero;
                        }
                        const int f = st + ((grp - st) & (cg - 1));
                        if (gapx * gapx + gy0 * gy0 + gz0 * gz0 > rmin2)
                            row_cells<false>(s_c[w], f, en, cg, A, dx, dy, dxy2, nk3, rmin2, sc,
                                             fz, gx, gy, gz);
                        else
                            row_cells<true>(s_c[w], f, en, cg, A, dx, dy, dxy2, nk3, rmin2, sc,
                                            fz, gx, gy, gz);
#pragma unroll
                        for (int p = 0; p < PAIRS; ++p) {
                            fx[p] = fma2(sc[p], dx[p], fx[p]);
                            fy[p] = fma2(sc[p], dy[p], fy[p]);
                        }
                    }
                    st = en;
                    at = next;
                    kk = 0;
                    ++jj;
                }
#pragma unroll
                for (int p = 0; p < PAIRS; ++p) {
                    two_sum_acc(hi[p][0], lo[p][0], fma2(A.kq[p], gx[p], fx[p]));
                    two_sum_acc(hi[p][1], lo[p][1], fma2(A.kq[p], gy[p], fy[p]));
                    two_sum_acc(hi[p][2], lo[p][2], fma2(A.kq[p], gz[p], fz[p]));
                }
            }
        }
    }
    // segment s: the atom's column at offset (s / 3 - 1, s % 3 - 1) from this
    // one, so this one at the opposite offset from the atom's
    store_parts(A, hi, lo, s_acc, a.n, part,
                [&](int u) { return 9 * (int)blockIdx.y + 8 - A.seg[u]; });
}

// One node against the lane's atoms: the gradient pair with the node's
// weights (m2 the solvent weight, c the field's), never clamped.
__device__ __forceinline__ void grad_node2(f2 zn, f2 m2, f2 ex, f2 ey, f2 ez, f2 dx, f2 dy,
                                           f2 dxy2, f2 az, f2 c1, f2 c2, f2 nk3, f2 &sc, f2 &fz,
                                           f2 &gx, f2 &gy, f2 &gz)
{
    const f2 dz = sub2(zn, az);
    const f2 r2 = fma2(dz, dz, dxy2);
    float ra, rb;
    upk2(r2, ra, rb);
    const f2 ri = pk2(rsqrt_ftz(ra), rsqrt_ftz(rb));
    const f2 ri2 = mul2(ri, ri);
    const f2 ri3 = mul2(ri2, ri);
    const f2 ri6 = mul2(ri3, ri3);
    const f2 ri5 = mul2(ri3, ri2);
    const f2 t1 = mul2(m2, fma2(c1, ri6, c2));
    const f2 dE = fma2(dx, ex, fma2(dy, ey, mul2(dz, ez)));
    const f2 cd = mul2(ri5, fma2(ri3, t1, mul2(nk3, dE)));
    sc = add2(sc, cd);
    fz = fma2(cd, dz, fz);
    gx = fma2(ri3, ex, gx);
    gy = fma2(ri3, ey, gy);
    gz = fma2(ri3, ez, gz);
}

struct NodePair {
    f2 m, ex, ey, ez;
};

// One tile's P^3 nodes against the lane's atoms: warp w takes every fourth
// pair of adjacent pencils (2 P nodes, contiguous in memory), staged in its
// own shared area as packed pairs.  Sums go into double-float accumulators
// every 8 pairs of pencils.
template <int P, int PAIRS>
__device__ __forceinline__ void tile_nodes(const float *__restrict__ V, const float *s_nx,
                                           const float *s_ny, const f2 *s_nz, NodePair *s_n,
                                           const LaneAtoms<PAIRS> &A, const f2 (&az)[PAIRS],
                                           const f2 (&c1)[PAIRS], const f2 (&c2)[PAIRS],
                                           const f2 (&kq)[PAIRS], f2 (&hi)[PAIRS][3],
                                           f2 (&lo)[PAIRS][3])
{
    constexpr int P3 = P * P * P;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const f2 zero = pk2(0.f, 0.f), m3 = pk2(-3.f, -3.f);
    f2 nk3[PAIRS], fx[PAIRS], fy[PAIRS], fz[PAIRS], gx[PAIRS], gy[PAIRS], gz[PAIRS];
#pragma unroll
    for (int p = 0; p < PAIRS; ++p) {
        nk3[p] = mul2(m3, kq[p]);
        fx[p] = fy[p] = fz[p] = gx[p] = gy[p] = gz[p] = zero;
    }
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    auto fetch = [&](int pp) {
        if (pp < P * P / 2 && lane < 2 * P)
#pragma unroll
            for (int f = 0; f < 4; ++f) v[f] = __ldg(V + f * P3 + pp * 2 * P + lane);
    };
    auto flush = [&]() {
#pragma unroll
        for (int p = 0; p < PAIRS; ++p) {
            two_sum_acc(hi[p][0], lo[p][0], fma2(kq[p], gx[p], fx[p]));
            two_sum_acc(hi[p][1], lo[p][1], fma2(kq[p], gy[p], fy[p]));
            two_sum_acc(hi[p][2], lo[p][2], fma2(kq[p], gz[p], fz[p]));
            fx[p] = fy[p] = fz[p] = gx[p] = gy[p] = gz[p] = zero;
        }
    };
    fetch(w);
    int it = 0;
#pragma unroll 1
    for (int pp = w; pp < P * P / 2; pp += TF_WARPS, ++it) {
        __syncwarp();
        if (lane < 2 * P) {
            NodePair n;
            n.m = pk2(v[0], v[0]);
            n.ex = pk2(v[1], v[1]);
            n.ey = pk2(v[2], v[2]);
            n.ez = pk2(v[3], v[3]);
            s_n[lane] = n;
        }
        __syncwarp();
        fetch(pp + TF_WARPS);
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
            const int pen = 2 * pp + hf;
            const float xx = s_nx[pen / P], yy = s_ny[pen % P];
            const f2 x2 = pk2(xx, xx), y2 = pk2(yy, yy);
            f2 dx[PAIRS], dy[PAIRS], dxy2[PAIRS], sc[PAIRS];
#pragma unroll
            for (int p = 0; p < PAIRS; ++p) {
                dx[p] = sub2(x2, A.x[p]);
                dy[p] = sub2(y2, A.y[p]);
                dxy2[p] = fma2(dx[p], dx[p], mul2(dy[p], dy[p]));
                sc[p] = zero;
            }
#pragma unroll (P == 12 ? 4 : 5)
            for (int c = 0; c < P; ++c) {
                const NodePair n = s_n[hf * P + c];
                const f2 zn = s_nz[c];
#pragma unroll
                for (int p = 0; p < PAIRS; ++p)
                    grad_node2(zn, n.m, n.ex, n.ey, n.ez, dx[p], dy[p], dxy2[p], az[p], c1[p],
                               c2[p], nk3[p], sc[p], fz[p], gx[p], gy[p], gz[p]);
            }
#pragma unroll
            for (int p = 0; p < PAIRS; ++p) {
                fx[p] = fma2(sc[p], dx[p], fx[p]);
                fy[p] = fma2(sc[p], dy[p], fy[p]);
            }
        }
        if ((it & 7) == 7) flush();
    }
    flush();
}

// Gradient terms met at level LEV < 2: an item is 128 atoms of the 3 x 3
// columns around a level LEV + 1 column (a group), met by the nodes of the
// tiles of the group's four level-LEV columns (blockIdx.y: which of ZP cuts
// of the z range, so that small solutes fill the chip); an atom whose own
// column touches a tile's gets that tile's terms at a lower level (or
// directly) and takes nothing here.  LEV = 2: block (x, chunk) takes the
// level-2 tiles chunk, chunk + gridDim.y, ... against 128 atoms.
template <int LEV>
__global__ void __launch_bounds__(TF_THREADS, 3)
k_tree_force_nodes(GridDesc g, TreeDims d, const TreeTab *__restrict__ tab,
                   const int *__restrict__ coff, const int *__restrict__ first,
                   const int *__restrict__ items, int ncols, const float *__restrict__ V,
                   ColAtoms a, double *__restrict__ part)
{
    constexpr int PAIRS = 2, P = tp(LEV), T = TC << LEV;
    constexpr int GL = LEV < 2 ? LEV + 1 : 2;      // level of the groups
    constexpr int ZP = LEV == 0 ? kZParts0 : kZParts1;
    __shared__ __align__(16) NodePair s_n[TF_WARPS][2 * P];
    __shared__ float s_nx[P], s_ny[P];
    __shared__ f2 s_nz[P];
    __shared__ double s_acc[TF_WARPS * 2 * PAIRS * 3 * 32];
    __shared__ SegList L;
    const int w = threadIdx.x >> 5;
    LaneAtoms<PAIRS> A;
    int X = 0, Y = 0;
    if (LEV < 2) {
        const int item = blockIdx.x;
        if (item >= first[ncols]) return;
        const int id = items[item];
        col_coords<GL>(d, id, X, Y);
        const int total = seg_cols<GL>(L, d, coff, X, Y);
        load_atoms(A, L, 9, a, 128 * (item - first[id]), total);
    } else {
        if (threadIdx.x == 0) {
            L.first[0] = 0;
            L.pre[0] = a.n;
        }
        const int total = seg_scan(L, 1);
        load_atoms(A, L, 1, a, 128 * blockIdx.x, total);
    }
    const f2 zero = pk2(0.f, 0.f);
    const float rh = 1.f / g.h;
    // the atoms' columns of this level
    int tx[2 * PAIRS], ty[2 * PAIRS];
#pragma unroll
    for (int p = 0; p < PAIRS; ++p) {
        float v[2][2];
        upk2(A.x[p], v[0][0], v[1][0]);
        upk2(A.y[p], v[0][1], v[1][1]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            tx[2 * p + e] = atom_cell(v[e][0], rh, g.cx, g.nx) / T;
            ty[2 * p + e] = atom_cell(v[e][1], rh, g.cy, g.ny) / T;
        }
    }
    f2 hi[PAIRS][3], lo[PAIRS][3];
#pragma unroll
    for (int p = 0; p < PAIRS; ++p)
#pragma unroll
        for (int c = 0; c < 3; ++c) hi[p][c] = lo[p][c] = zero;
    const int nzt = (g.nz + T - 1) / T;            // tiles of a column
    // LEV < 2: the group's four columns, tiles zb .. ze of each
    const int zb = nzt * (int)blockIdx.y / ZP, ze = nzt * ((int)blockIdx.y + 1) / ZP;
    const int nzp = LEV < 2 ? max(1, ze - zb) : 1;
    const int o0 = LEV < 2 ? 0 : blockIdx.y, step = LEV < 2 ? 1 : gridDim.y;
    const int o1 = LEV < 2 ? 4 * (ze - zb) : d.n2;
#pragma unroll 1
    for (int o = o0; o < o1; o += step) {
        int cx, cy, cz;
        if (LEV < 2) {
            const int ch = o / nzp;
            cx = 2 * X + (ch >> 1);
            cy = 2 * Y + (ch & 1);
            cz = zb + o - ch * nzp;
        } else {
            tree_coords<LEV>(d, o, cx, cy, cz);
        }
        if (cx * T >= g.nx || cy * T >= g.ny || cz * T >= g.nz) continue;
        // an atom near the column (or an idle slot) gets zero coefficients
        // and a far z, so that nothing divides by zero
        f2 az[PAIRS], c1[PAIRS], c2[PAIRS], kq[PAIRS];
        bool any = false;
#pragma unroll
        for (int p = 0; p < PAIRS; ++p) {
            float z0, z1, a0, a1, b0, b1, k0, k1;
            upk2(A.z[p], z0, z1);
            upk2(A.c1[p], a0, a1);
            upk2(A.c2[p], b0, b1);
            upk2(A.kq[p], k0, k1);
            const int u = 2 * p;
            const bool f0 = A.idx[u] >= 0 && (abs(tx[u] - cx) > 1 || abs(ty[u] - cy) > 1);
            const bool f1 =
                A.idx[u + 1] >= 0 && (abs(tx[u + 1] - cx) > 1 || abs(ty[u + 1] - cy) > 1);
            any |= f0 || f1;
            az[p] = pk2(f0 ? z0 : 1.0e6f, f1 ? z1 : 1.0e6f);
            c1[p] = pk2(f0 ? a0 : 0.f, f1 ? a1 : 0.f);
            c2[p] = pk2(f0 ? b0 : 0.f, f1 ? b1 : 0.f);
            kq[p] = pk2(f0 ? k0 : 0.f, f1 ? k1 : 0.f);
        }
        // every warp holds the same atoms, so this is uniform in the block
        if (!__any_sync(0xffffffffu, any)) continue;
        __syncthreads();                 // the previous tile's nodes are no longer read
        if (threadIdx.x < P) {
            const float u = tab->node[LEV][threadIdx.x];
            s_nx[threadIdx.x] = node_pos(cx, T, u, g.cx, g.h);
            s_ny[threadIdx.x] = node_pos(cy, T, u, g.cy, g.h);
            const float zz = node_pos(cz, T, u, g.cz, g.h);
            s_nz[threadIdx.x] = pk2(zz, zz);
        }
        __syncthreads();
        tile_nodes<P, PAIRS>(V + tile_place<LEV>(g, cx, cy, cz) * tn4(LEV), s_nx, s_ny, s_nz, s_n[w], A, az, c1, c2, kq, hi,
                      lo);
    }
    store_parts(A, hi, lo, s_acc, a.n, part, [&](int u) {
        return LEV < 2 ? 9 * (int)blockIdx.y + 8 - A.seg[u] : (int)blockIdx.y;
    });
}

// Gradient of the sorted atom i: its partials in slot order (those of columns
// outside the grid hold nothing), scaled.
__global__ void k_tree_force_reduce(GridDesc g, const float4 *__restrict__ xyzq,
                                    const int *__restrict__ ord, const double *__restrict__ part,
                                    int n, int sf, double scale, double *__restrict__ out)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * n) return;
    const int i = t / 3, c = t - 3 * i;
    const float4 A = xyzq[i];
    const float rh = 1.f / g.h;
    const int x = atom_cell(A.x, rh, g.cx, g.nx) / TC, y = atom_cell(A.y, rh, g.cy, g.ny) / TC;
    double s = 0.0;
    constexpr int kParts = kRowParts + kZParts0 + kZParts1;
#pragma unroll 1
    for (int m = 0; m < kParts; ++m) {
        const int l = m < kRowParts ? 0 : m < kRowParts + kZParts0 ? 1 : 2;   // level of the columns
        const int T = TC << l;
        double v[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int a = (x >> l) + q / 3 - 1, b = (y >> l) + q % 3 - 1;
            v[q] = a >= 0 && b >= 0 && a * T < g.nx && b * T < g.ny
                       ? part[((size_t)(9 * m + q) * n + i) * 3 + c]
                       : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 9; ++q) s += v[q];
    }
#pragma unroll 8
    for (int q = 0; q < sf; ++q) s += part[((size_t)(9 * kParts + q) * n + i) * 3 + c];
    out[3 * ord[i] + c] = s * scale;
}

void launch_tree_force(const GridDesc &g, const TreePlan &p, uint8_t *ws, const AtomsDev &a,
                       int cg, const uint8_t *chi, const float *Ex, const float *Ey,
                       const float *Ez, float rmin2, double scale, double *out,
                       unsigned long long *nsolvent, cudaStream_t st)
{
    const TreeTab *tab = (const TreeTab *)(ws + p.o_tab);
    float *V[3];
    for (int l = 0; l < 3; ++l) V[l] = (float *)(ws + p.o_v[l]);
    const int n = a.n, cols = p.d.nx * p.d.ny * 16;
    const unsigned n2 = (unsigned)p.d.n2, nb = (unsigned)((n + 127) / 128);
    // atoms by column
    int *cnt = (int *)(ws + p.o_cnt), *cur = (int *)(ws + p.o_cur), *coff = (int *)(ws + p.o_coff);
    int *id = (int *)(ws + p.o_id), *tmp = (int *)(ws + p.o_tmp), *ord = (int *)(ws + p.o_ord);
    ColAtoms ca;
    ca.n = n;
    ca.xyzq = (const float4 *)(ws + p.o_cxyz);
    ca.fcoef = (const float4 *)(ws + p.o_cfc);
    const PlanArgs P = plan_args(p, ws, 3);
    cudaMemsetAsync(cnt, 0, (size_t)cols * sizeof(int), st);
    count_launch(13);
    k_col_count<<<nb, 128, 0, st>>>(g, p.d, a.xyzq, n, id, cnt);
    k_tree_scan<<<1, 1024, 0, st>>>(cnt, cols, coff, cur);
    k_tree_scatter<<<nb, 128, 0, st>>>(id, n, cur, tmp);
    k_tree_place<<<nb, 128, 0, st>>>(tmp, id, coff, n, a.xyzq, a.fcoef, ord,
                                     (float4 *)(ws + p.o_cxyz), (float4 *)(ws + p.o_cfc));
    k_col_items<<<3, 1024, 0, st>>>(g, p.d, coff, P);
    // node weights
    k_tree_gather<<<n2 * 64, 128, 0, st>>>(g, p.d, tab, chi, Ex, Ey, Ez, V[0], nsolvent);
    k_tree_merge<1><<<dim3(n2 * 8, 4), 160, 0, st>>>(g, p.d, tab, V[0], V[1]);
    k_tree_merge<2><<<dim3(n2, 4), 160, 0, st>>>(g, p.d, tab, V[1], V[2]);
    // pair terms
    const TreeList *l = p.list + 3;
    double *part = (double *)(ws + p.o_part);
    const size_t block = (size_t)n * 3;
    k_tree_force_rows<<<dim3(l[0].max_items, kRowParts), TF_THREADS, 0, st>>>(
        g, p.d, coff, P.first[0], P.item[0], P.tiles[0], chi, Ex, Ey, Ez, ca, rmin2, cg, part);
    double *pn = part + 9 * kRowParts * block;
    k_tree_force_nodes<0><<<dim3(l[1].max_items, kZParts0), TF_THREADS, 0, st>>>(
        g, p.d, tab, coff, P.first[1], P.item[1], P.tiles[1], V[0], ca, pn);
    pn += 9 * kZParts0 * block;
    k_tree_force_nodes<1><<<dim3(l[2].max_items, kZParts1), TF_THREADS, 0, st>>>(
        g, p.d, tab, coff, P.first[2], P.item[2], P.tiles[2], V[1], ca, pn);
    pn += 9 * kZParts1 * block;
    k_tree_force_nodes<2><<<dim3(nb, (unsigned)p.sf), TF_THREADS, 0, st>>>(
        g, p.d, tab, coff, nullptr, nullptr, 0, V[2], ca, pn);
    k_tree_force_reduce<<<(unsigned)((3 * n + 127) / 128), 128, 0, st>>>(g, ca.xyzq, ord, part, n,
                                                                         p.sf, scale, out);
}

}  // namespace vesis
