// Persistent narrow-band flip sweep (Sec. 3.1, Step 2) for sm_103a.
//
// All flip rounds of one interface relaxation run in a single cooperative
// launch.  The grid is cut into 8^3 tiles; a round only visits tiles that
// hold a cell that may flip or lie near one that just flipped, which keeps
// the work on the band around the interface the paper restricts the flips
// to.
//
// Selection rule (the data-parallel form of the min-heap flipping): every
// candidate cell (a face neighbour has the other label) whose flip lowers
// the energy (dE < 0 in FP64, Eqs. dGj1/dGj2) gets the key float(dE); the
// grid is cut into bricks of edge B (4 when r >= 3, else 2) aligned at
// index 0, and a brick's leader is its cell with the most negative key, the
// smaller linear index among equal keys.  A leader flips when no other
// brick's leader within Chebyshev distance r comes first.  The heap's top
// always flips, flipped cells are more than r apart, the kernel couples
// none of them, and a round lowers the energy by exactly the sum of their
// dE.
//
// A leader is one 64-bit word, larger = first:
//   (magnitude bits of float(dE)) << 33 | (2^32 - 1 - index) << 1 | label,
// zero for a brick without one (PL, one word per brick).
//
// Round k:
//   decide (a team of two warps per tile holding a leader): the words of the
//     6^3 bricks around the tile arrive together, four per thread; the
//     non-zero ones go to shared memory, and each warp tests its half of the
//     tile's leaders against them.  A winner flips its label and adds its dE,
//     and posts itself to every tile within r of it: a 16-bit entry (cell
//     within its brick, old label) in the slot of its brick among the 6^3
//     bricks that tile can see, the slot's bit, and the tile's bit in its
//     owner's update bitmap.
//   grid barrier
//   update (a team per tile that received a winner, a warp per half of 4 x 8
//     rows of 8 cells, a row per thread): W of the tile's own cells gets +-q_a
//     q_b q_c from each posted winner whose window covers them (W stays the
//     exact convolution, and only the team visiting the tile writes its
//     cells), then the half's candidates, their dE and its leaders are
//     recomputed.  Tiles no winner reached keep their leaders.
//   grid barrier
// The sweep stops when no tile holds a leader or after max_rounds rounds.
// An opening pass computes every tile's leaders from the starting labels.
//
// A round is bound by latency: two grid barriers (1.2 us each alone) and, in each
// phase, the chain from a tile's loads to its stores, which teams sharing an
// SM stretch for one another through the instructions they issue.  A half
// tile per warp keeps a tile's two warps apart but for one barrier: the
// bricks, their leaders and the verdicts on them are a warp's own.  Measured
// with eight teams per block, one block per SM (us per round, before = one
// warp per tile, 32 per block; two atoms in 128^3, 112^3 small solute, 256^3
// protein, 384^3 complex): 12.5, 12.4, 14.3, 29.8 before; 7.4, 8.0, 11.0, 22.4
// now; teams of four warps 9.4, 9.4, 12.0, 26.4; four teams per block 7.4,
// 8.8, 12.5, 29.5; twelve (80 registers a thread, spilling) 9.5, 9.9, 11.5,
// 23.7; 76 blocks instead of 152 11.1 for the 112^3 solute; one cluster of 16
// blocks with its barriers in shared memory 16.4 there.
//
// Only tiles whose verdict can change are decided: a leader's verdict is a
// function of the leader words within r of it, all inside the 27 tiles
// around its own, so a tile none of whose 27 neighbours (itself included)
// changed a leader word in the last update keeps its last verdict - it
// lost (a winner changes its own tile's words) - and is skipped.  Every
// update that changes one of the tile's words stamps its 27 neighbours (a
// bit in the owner's stamp bitmap, read and cleared by the next decide);
// round 0 decides every tile.  The winners, and so the rounds and labels,
// are those of deciding every tile every round.  The stamps only pay where
// teams have several tiles: the updates write them while the half tiles
// holding a leader outnumber the grid's warps (a count all blocks read alike),
// and a block reads them only after such an update and when its own leader
// halves outnumber its warps (deciding an unstamped tile is harmless).
//
// The grid barrier spins with a bound; on timeout it raises an error flag
// and every block returns.
#include <vector>

#include "vesis_internal.cuh"

namespace vesis {

constexpr int TS = 8;             // tile edge
constexpr int TEAM = 64;          // threads of a team: two warps, a half tile each
constexpr int NTEAM = 8;          // teams of a block (named barriers 1 .. 8)
constexpr int SW_THREADS = TEAM * NTEAM;
constexpr int kLine = 32;         // words per 128-byte line of the control block
// control block: the count of leader half tiles, then the barrier's counter
constexpr int kCtlWords = 2 * kLine;
constexpr int kMaxBricksPerTile = 64;         // (8 / 2)^3 for bricks of edge 2
constexpr int kHaloRows = (TS + 2) * (TS + 2);
// Bricks per axis a tile can see: the tile's own (8 / B) and ceil(r / B) on
// each side; 6 for r <= 8 with B = 4 and for r <= 2 with B = 2.  Leaders
// within r of a tile, and the rivals of a tile's own leaders, all lie there.
constexpr int kNbh = 6;
constexpr int kNbh3 = kNbh * kNbh * kNbh;
constexpr int kSlots = (kNbh3 + TEAM - 1) / TEAM;     // of those, per thread
// Posting area of a tile: 216 16-bit slots and an 8-word slot bitmap.
constexpr int kPostBytes = 512;
constexpr int kPostMaskOff = 448;
// A block keeps one bit per own tile (holds a leader) in shared memory:
// up to 32768 own tiles, more than a grid of 2^31 cells gives any block.
constexpr int kOwnWords = 1024;
// 1-D weights padded with zeros: entry a + kQ0 holds q_a, |a| <= 15
constexpr int kQ0 = 16;
// a row of the full stencil in shared memory: offsets -15 .. 15, zeros past r
constexpr int kKtRow = 31;

__host__ __device__ constexpr int sweep_edge(int r) { return r >= 3 ? 4 : 2; }

struct SweepArgs {
    GridDesc g;
    KernelW kw;
    double cD;          // c_N: dE = c_N N - s h^3 U
    double h3;
    float cDf, h3f;     // the same in FP32
    int qc3;            // k0, the kernel's centre weight
    int ksum;           // S, the sum of all kernel weights
    const int *k3;      // full stencil (device) or NULL for the product kernel
    uint8_t *chi;
    uint32_t *W;
    const float *U;
    double *dE;
    unsigned long long *PL;   // leader word per brick
    uint8_t *PO;              // leader cell within its brick: di | dj << 2 | dk << 4
    unsigned *CB;             // labels, one bit per cell: word w of column (i, j)
                              // at (w nx + i) ny + j (a tile's halo words adjoin)
    int nzw;
    uint8_t *post;            // posting area per tile (kPostBytes)
    // bitmaps over the launch's tiles, block by block: bit j of block b is bit
    // j % 32 of word b * bwords + j / 32 (see set_tile_bit); two of each, for
    // even and odd rounds, so that a block clears one while the other is used
    unsigned *upd;            // tile received a winner this round
    unsigned *stamp;          // tile must be decided next round
    int bwords;
    unsigned mapw;            // words of one bitmap
    unsigned tile0;           // the system's first tile among the launch's (multi)
    unsigned nblk, nblk_inv;  // gridDim and ceil(2^32 / gridDim)
    int ntx, nty, ntz;
    unsigned nty_inv, ntz_inv;    // ceil(2^32 / .)
    int bs, bsh;        // brick edge and its log2
    int reach;          // ceil(r / B)
    int nbx, nby, nbz;  // bricks per axis
    int vec;            // a tile's rows of W and U are loaded as two vectors each (2), as the
                        // three that cover them (1: rows at odd offsets) or cell by cell (0)
    unsigned ncell;
    unsigned *nlead;    // half tiles holding a leader (kept current by the updates)
    unsigned *bar;      // monotonic arrival counter (own 128-byte line)
    int *err;
    unsigned long long *part_flips;   // [gridDim.x]
    double *part_dE;                  // [gridDim.x]
    unsigned long long *part_tiles;   // [2][gridDim.x]: tiles decided, tiles updated
    int *rounds_out;
    int *capped_out;
    int max_rounds;
    long long spin_limit;     // polls before a barrier wait gives up
    int stamps;               // decide stamps: -1 by the leader count, 0 never, 1 always
    RoundState *rs;           // this system's totals (multi-system sweep)
    double *tile_dE;          // per half tile: its winners' dE, summed over rounds (multi)
    unsigned *tile_nf;        // per half tile: its flips (multi)
};

// A team's shared memory.  Every area has two copies, taken in turn: between
// the one barrier of a tile and that of the next, a warp may still read the
// copy the other warp wrote before the first.
struct TeamMem {
    unsigned long long lw[2][kMaxBricksPerTile];  // decide: the tile's leader words
    unsigned lc[2][kMaxBricksPerTile];            //   and their cells, 5 bits per axis
    unsigned long long cw[2][2][kSlots * 32];     //   the non-zero words each warp saw
    unsigned cc[2][2][kSlots * 32];               //   and their cells
    int ncw[2][2];                                //   their number
    unsigned long long bmax[kMaxBricksPerTile];   // update: new leader per brick
    unsigned hr[2][kHaloRows];   //   label bits of the halo rows (bit 0: z = -1)
    unsigned win[2][2][kSlots * 32];   // winners each warp found: tile coords + 8
                                       //   (5 bits each) | label << 15
    int nw[2][2];                      //   their number
};

__device__ __forceinline__ unsigned ld_relaxed_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Where a block of the sweep stands at the barrier between phases.
struct Barrier {
    unsigned *bar;            // monotonic arrival counter
    unsigned target;          // thread 0: arrivals the next barrier waits for
    int *err;
    long long spin_limit;
};

// Barrier of all blocks: number e (1, 2, ...) completes when the counter
// reaches e * gridDim.x.  Arrival is one release reduction (it orders the
// block's earlier writes, which bar.sync has made visible to thread 0); the
// wait polls with acquire loads, back to back, and needs no closing acquire.
// (Alone on its SM a block loses nothing to the L1 lines they invalidate; in a
// batched relaxation other systems' kernels share the SM, and relaxed polls
// with a closing acquire or a 32 ns sleep between polls changed batches of 8
// and 24 systems on 1 to 16 slots by less than 1.5 %, the spread of their runs.)
// The poll is bounded (spin_limit polls; 0 gives up at the first
// poll that finds the barrier open) and watches the error flag every 256
// polls; a timeout raises the flag and the caller returns.  (Spreading the
// arrivals over 4 or 8 counters, polled by as many lanes, cost 0.1 us a
// barrier more than one.)
__device__ __forceinline__ bool all_blocks(Barrier &B, int *abort_flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        B.target += gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" :: "l"(B.bar), "r"(1u)
                     : "memory");
        long long spins = 0;
        while ((int)(ld_acquire_u32(B.bar) - B.target) < 0) {
            if (++spins > B.spin_limit ||
                ((spins & 255) == 0 && *(volatile int *)B.err)) {
                atomicExch(B.err, 1);
                *abort_flag = 1;
                break;
            }
        }
    }
    __syncthreads();
    return *abort_flag == 0;
}

// Barrier of one team (hardware barriers 1 .. NTEAM; 0 is the block's).
__device__ __forceinline__ void team_sync(int team)
{
    asm volatile("bar.sync %0, %1;" :: "r"(team + 1), "n"(TEAM) : "memory");
}

__device__ __forceinline__ void red_or(unsigned *p, unsigned v)
{
    asm volatile("red.relaxed.gpu.global.or.b32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void red_add(unsigned *p, unsigned v)
{
    asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// Tiles are dealt to the blocks in groups of gridDim consecutive ones, each
// group rotated by a hash of its number: tile t is number j = t / gridDim of
// block (t + turn(j)) % gridDim.  (Unrotated, the tiles of one z layer share a
// block whenever gridDim and the tiles per axis have a common factor.)
__device__ __forceinline__ unsigned turn_of(unsigned j, unsigned nblk)
{
    return __umulhi(j * 0x9E3779B1u, nblk);
}

// Sets the bit of the system's tile t in a bitmap over the launch's tiles.
// The quotient by gridDim is exact: at most 2^15 tiles per block and 256 blocks.
__device__ __forceinline__ void set_tile_bit(const SweepArgs &A, unsigned *map, unsigned t)
{
    const unsigned tg = A.tile0 + t;
    const unsigned j = A.nblk == 1u ? tg : __umulhi(tg, A.nblk_inv);
    unsigned b = tg - j * A.nblk + turn_of(j, A.nblk);
    if (b >= A.nblk) b -= A.nblk;
    red_or(map + (size_t)b * A.bwords + (j >> 5), 1u << (j & 31));
}

// Tile number j of this block (may lie past the last tile).
__device__ __forceinline__ long long own_tile_no(int j)
{
    int r = (int)blockIdx.x - (int)turn_of((unsigned)j, gridDim.x);
    if (r < 0) r += (int)gridDim.x;
    return (long long)j * gridDim.x + r;
}

// A tile's number and coordinates.
struct Tile {
    int t, i, j, k;
};

// (Quotients exact: t < 2^22 and at most 512 tiles per axis.)
__device__ __forceinline__ Tile make_tile(const SweepArgs &A, int t)
{
    const int q = A.ntz == 1 ? t : (int)__umulhi((unsigned)t, A.ntz_inv);
    const int i = A.nty == 1 ? q : (int)__umulhi((unsigned)q, A.nty_inv);
    return {t, i, q - i * A.nty, t - q * A.ntz};
}

// What a thread of a team does in every tile: its slots of the 6^3 bricks,
// as a | b << 4 | c << 8 (brick relative to the first) | n << 12, n - 1 the
// brick's number among the tile's own if it is one (n = 0: it is not); bit
// 31: no slot.
struct Lane {
    int u, w, lane;            // thread of the team, warp, lane
    unsigned slot[kSlots];
};

__device__ __forceinline__ Lane make_lane(int bpt, int reach)
{
    Lane L;
    L.u = threadIdx.x % TEAM;
    L.w = L.u >> 5;
    L.lane = L.u & 31;
#pragma unroll
    for (int m = 0; m < kSlots; ++m) {
        const int q = L.u + TEAM * m;
        const int a = q / (kNbh * kNbh), b = (q / kNbh) % kNbh, c = q % kNbh;
        const int x = a - reach, y = b - reach, z = c - reach;
        const bool own = x >= 0 && y >= 0 && z >= 0 && x < bpt && y < bpt && z < bpt;
        L.slot[m] = q < kNbh3 ? (unsigned)(a | b << 4 | c << 8 |
                                           (own ? (x * bpt + y) * bpt + z + 1 : 0) << 12)
                              : 0x80000000u;
    }
    return L;
}

// Labels, W, dE, leader words, postings and tile bits change under other
// teams and blocks between phases: every read of them goes to L2
// (ld.global.cg), never to a stale L1 line.

// Decide phase for one tile; each warp settles half of its leaders (bricks of
// edge 4: x half w, eight lanes per leader; of edge 2: leaders 32 w .. 32 w +
// 31, one per lane).  e_lane, n_lane: dE and count of the winners; turn: which
// copy of the shared areas the tile uses.
__device__ __forceinline__ void tile_decide(const SweepArgs &A, TeamMem &M, const Lane &L,
                                            int team, const Tile &tile, int &turn,
                                            unsigned *upd, double &e_lane, unsigned &n_lane)
{
    const GridDesc &g = A.g;
    const int r = A.kw.r, bsh = A.bsh, reach = A.reach;
    const int bpt = TS >> bsh;
    const int nbx0 = tile.i * bpt - reach, nby0 = tile.j * bpt - reach, nbz0 = tile.k * bpt - reach;
    unsigned long long v[kSlots];
    unsigned off[kSlots];
#pragma unroll
    for (int m = 0; m < kSlots; ++m) {
        const int bx = nbx0 + (int)(L.slot[m] & 15u), by = nby0 + (int)((L.slot[m] >> 4) & 15u),
                  bz = nbz0 + (int)((L.slot[m] >> 8) & 15u);
        v[m] = 0ull;
        off[m] = 0u;
        if ((int)L.slot[m] >= 0 && (unsigned)bx < (unsigned)A.nbx &&
            (unsigned)by < (unsigned)A.nby && (unsigned)bz < (unsigned)A.nbz) {
            const int q = (bx * A.nby + by) * A.nbz + bz;
            v[m] = __ldcg(A.PL + q);
            off[m] = __ldcg(A.PO + q);
        }
    }
    // the tile's own words and all non-zero ones to shared memory, with their
    // cells relative to the neighbourhood's first cell
    const unsigned below = (1u << L.lane) - 1u;
    int at = 0;
#pragma unroll
    for (int m = 0; m < kSlots; ++m) {
        const unsigned c = ((L.slot[m] & 15u) << bsh) + (off[m] & 3u) +
                           (((((L.slot[m] >> 4) & 15u) << bsh) + ((off[m] >> 2) & 3u)) << 5) +
                           (((((L.slot[m] >> 8) & 15u) << bsh) + ((off[m] >> 4) & 3u)) << 10);
        const int own = (int)((L.slot[m] >> 12) & 127u) - 1;
        if (own >= 0) {
            M.lw[turn][own] = v[m];
            M.lc[turn][own] = c;
        }
        const unsigned bm = __ballot_sync(0xffffffffu, v[m] != 0ull);
        if (v[m] != 0ull) {
            const int to = at + __popc(bm & below);
            M.cw[turn][L.w][to] = v[m];
            M.cc[turn][L.w][to] = c;
        }
        at += __popc(bm);
    }
    if (L.lane == 0) M.ncw[turn][L.w] = at;
    team_sync(team);
    // a leader of the tile loses to any better word within r
    const int n0 = M.ncw[turn][0], ncw = n0 + M.ncw[turn][1];
    const int per = bpt == 2 ? 4 : 32;                 // leaders of a warp
    const int mine = per * L.w + (L.lane & (per - 1)), step = 32 / per;
    const unsigned long long lead = M.lw[turn][mine];
    bool beat = false;
    if (lead != 0ull) {
        const unsigned lc = M.lc[turn][mine];
        const int lx = (int)(lc & 31u) - r, ly = (int)((lc >> 5) & 31u) - r,
                  lz = (int)((lc >> 10) & 31u) - r;
        const unsigned long long *cw = M.cw[turn][0];
        const unsigned *cc = M.cc[turn][0];
#pragma unroll 2
        for (int q = bpt == 2 ? L.lane >> 2 : 0; q < ncw; q += step) {
            const int k = q < n0 ? q : q - n0 + kSlots * 32;
            const unsigned long long o = cw[k];
            const unsigned c = cc[k];
            beat |= (o > lead) & ((unsigned)((int)(c & 31u) - lx) <= 2u * r) &
                    ((unsigned)((int)((c >> 5) & 31u) - ly) <= 2u * r) &
                    ((unsigned)((int)((c >> 10) & 31u) - lz) <= 2u * r);
        }
    }
    // winners among the warp's leaders: bit l is leader per * w + l
    unsigned wm = __ballot_sync(0xffffffffu, beat);
    if (bpt == 2) {
        wm |= wm >> 16;
        wm |= wm >> 8;
        wm |= wm >> 4;
    }
    wm = __ballot_sync(0xffffffffu, lead != 0ull) & ~wm & (bpt == 2 ? 15u : 0xffffffffu);
    const int my = turn;
    turn ^= 1;
    // they flip and fetch dE (added at the end) ...
    double dv = 0.0;
    if ((wm >> L.lane) & 1u) {
        const unsigned long long won = M.lw[my][per * L.w + L.lane];
        const unsigned lc = M.lc[my][per * L.w + L.lane];
        const int ci = (nbx0 << bsh) + (int)(lc & 31u), cj = (nby0 << bsh) + (int)((lc >> 5) & 31u),
                  ck = (nbz0 << bsh) + (int)((lc >> 10) & 31u);
        const unsigned p = ~(unsigned)(won >> 1);
        A.chi[p] = (uint8_t)(1u - (unsigned)(won & 1ull));
        asm volatile("red.relaxed.gpu.global.xor.b32 [%0], %1;"
                     :: "l"(A.CB + (((ck >> 5) * g.nx + ci) * g.ny + cj)),
                        "r"(1u << (ck & 31)) : "memory");
        dv = __ldcg(A.dE + p);
        n_lane += 1u;
    }
    // ... and post themselves to every tile within r, a lane per tile
    for (unsigned todo = wm; todo; todo &= todo - 1) {
        const int b = per * L.w + __ffs(todo) - 1;
        const unsigned long long won = M.lw[my][b];
        const unsigned lc = M.lc[my][b];
        const int ci = (nbx0 << bsh) + (int)(lc & 31u), cj = (nby0 << bsh) + (int)((lc >> 5) & 31u),
                  ck = (nbz0 << bsh) + (int)((lc >> 10) & 31u);
        const int ta = (max(ci - r, 0) / TS) + L.lane / 9, tb = (max(cj - r, 0) / TS) + (L.lane / 3) % 3,
                  tc = (max(ck - r, 0) / TS) + L.lane % 3;
        if (L.lane < 27 && ta <= min(ci + r, g.nx - 1) / TS && tb <= min(cj + r, g.ny - 1) / TS &&
            tc <= min(ck + r, g.nz - 1) / TS) {
            const unsigned entry = (unsigned)(ci & (A.bs - 1)) | ((unsigned)(cj & (A.bs - 1)) << 2) |
                                   ((unsigned)(ck & (A.bs - 1)) << 4) |
                                   ((unsigned)(won & 1ull) << 6);
            const int tt = (ta * A.nty + tb) * A.ntz + tc;
            // the winner's brick among the 6^3 bricks tile tt sees
            const int sx = (ci >> bsh) - ((ta * TS) >> bsh) + reach;
            const int sy = (cj >> bsh) - ((tb * TS) >> bsh) + reach;
            const int sz = (ck >> bsh) - ((tc * TS) >> bsh) + reach;
            const int slot = (sx * kNbh + sy) * kNbh + sz;
            uint8_t *pa = A.post + (size_t)tt * kPostBytes;
            reinterpret_cast<unsigned short *>(pa)[slot] = (unsigned short)entry;
            red_or(reinterpret_cast<unsigned *>(pa + kPostMaskOff) + (slot >> 5),
                   1u << (slot & 31));
            set_tile_bit(A, upd, (unsigned)tt);
        }
    }
    e_lane += dv;
}

// Update phase for one tile, the half with 0 <= x - 4 w < 4 by warp w (bricks
// never straddle the halves).  first: the opening pass (no winners; every tile
// computes its leaders).  stamp: the bitmap (or NULL) in which the 27 tiles
// around it (itself included) are marked for the next decide if a leader word
// of the half changes.
// Returns whether the warp's half holds a leader.
template <bool STENCIL>
__device__ __forceinline__ bool tile_update(const SweepArgs &A, TeamMem &M, const int *qw,
                                            const int *kt, const Lane &L, int team,
                                            const Tile &tile, bool first, unsigned *stamp, int &turn)
{
    const GridDesc &g = A.g;
    const int nyz = g.ny * g.nz;
    const int r = A.kw.r, bsh = A.bsh, reach = A.reach;
    const int bpt = TS >> bsh;
    const int ti = tile.i, tj = tile.j, tk = tile.k;
    const int i0 = ti * TS, j0 = tj * TS, k0 = tk * TS;
    const int u = L.u;

    // ---------------------------------------------------------- loads
    // All of a thread's loads are issued before the first use.  Its cells:
    // row (cx, cy).
    const int cx = u >> 3, cy = u & 7;
    const bool rowok = i0 + cx < g.nx && j0 + cy < g.ny;
    const int zc = rowok ? min(TS, g.nz - k0) : 0;        // cells inside the grid
    const unsigned o = (unsigned)(i0 + cx) * (unsigned)nyz + (unsigned)((j0 + cy) * g.nz + k0);
    unsigned Wr[TS];
    float Ur[TS];
#pragma unroll
    for (int z = 0; z < TS; ++z) {
        Wr[z] = 0u;
        Ur[z] = 0.f;
    }
    if (A.vec == 2) {
        if (zc) {
#pragma unroll
            for (int h = 0; h < TS; h += 4) {
                const uint4 wv = __ldcg(reinterpret_cast<const uint4 *>(A.W + o + h));
                const float4 uv = __ldg(reinterpret_cast<const float4 *>(A.U + o + h));
                Wr[h] = wv.x; Wr[h + 1] = wv.y; Wr[h + 2] = wv.z; Wr[h + 3] = wv.w;
                Ur[h] = uv.x; Ur[h + 1] = uv.y; Ur[h + 2] = uv.z; Ur[h + 3] = uv.w;
            }
        }
    } else if (A.vec == 1 && (o & ~3u) + 12u <= A.ncell) {
        if (zc) {
            unsigned wv[12], uv[12];
#pragma unroll
            for (int h = 0; h < 12; h += 4) {
                const uint4 a = __ldcg(reinterpret_cast<const uint4 *>(A.W + ((o & ~3u) + h)));
                const uint4 b = __ldg(reinterpret_cast<const uint4 *>(A.U + ((o & ~3u) + h)));
                wv[h] = a.x; wv[h + 1] = a.y; wv[h + 2] = a.z; wv[h + 3] = a.w;
                uv[h] = b.x; uv[h + 1] = b.y; uv[h + 2] = b.z; uv[h + 3] = b.w;
            }
#pragma unroll
            for (int z = 0; z < 11; ++z) {
                wv[z] = o & 1u ? wv[z + 1] : wv[z];
                uv[z] = o & 1u ? uv[z + 1] : uv[z];
            }
#pragma unroll
            for (int z = 0; z < TS; ++z) {
                Wr[z] = o & 2u ? wv[z + 2] : wv[z];
                Ur[z] = __uint_as_float(o & 2u ? uv[z + 2] : uv[z]);
            }
        }
    } else {
#pragma unroll
        for (int z = 0; z < TS; ++z)
            if (z < zc) {
                Wr[z] = __ldcg(A.W + o + z);
                Ur[z] = __ldg(A.U + o + z);
            }
    }
    // halo label rows from the bit copy: row h = hx * 10 + hy is the cell
    // column (i0 - 1 + hx, j0 - 1 + hy); bit z + 1 is cell k0 + z, z = -1..8.
    // Cells k0..k0 + 7 share word k0 / 32 (k0 is a multiple of 8); cell k0 - 1
    // or k0 + 8 sits in the word before or after when k0 % 32 is 0 or 24.
    // Bits past the end of a row are zero (solvent, as outside the box).
    unsigned hm[2], hn[2];     // the word, and the word before or after
    const int sh = k0 & 31;
    const int pl = g.nx * g.ny;                           // words per plane
    const int side = sh == 0 ? (k0 > 0 ? -pl : 0) : sh == 24 ? (k0 + TS < g.nz ? pl : 0) : 0;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const int q = u + TEAM * m, hx = q / 10;
        const int i = i0 - 1 + hx, j = j0 - 1 + q - 10 * hx;
        hm[m] = hn[m] = 0u;
        if (q < kHaloRows && i >= 0 && j >= 0 && i < g.nx && j < g.ny) {
            const unsigned *col = A.CB + ((k0 >> 5) * pl + i * g.ny + j);
            hm[m] = __ldcg(col);
            if (side) hn[m] = __ldcg(col + side);
        }
    }
    // posted winners: thread q < 54 holds slots 4 q .. 4 q + 3 and their bits
    uint8_t *pa = A.post + (size_t)tile.t * kPostBytes;
    unsigned *pmask = reinterpret_cast<unsigned *>(pa + kPostMaskOff);
    unsigned long long ps = 0ull;
    unsigned pm = 0u;
    if (!first && u < kNbh3 / 4) {
        ps = __ldcg(reinterpret_cast<const unsigned long long *>(pa) + u);
        pm = __ldcg(pmask + (u >> 3));
    }
    // the leader word of the lane's brick before this update
    const int per = bpt == 2 ? 4 : 32;                 // bricks of a warp
    const int brick = per * L.w + (L.lane & (per - 1));
    int bq = -1;
    {
        const int gx = ti * bpt + brick / (bpt * bpt), gy = tj * bpt + (brick / bpt) % bpt,
                  gz = tk * bpt + brick % bpt;
        if (L.lane < per && gx < A.nbx && gy < A.nby && gz < A.nbz)
            bq = (gx * A.nby + gy) * A.nbz + gz;
    }
    unsigned long long oldw = 0ull;
    if (stamp && bq >= 0) oldw = __ldcg(A.PL + bq);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const unsigned lo = sh == 0 ? hn[m] >> 31 : (hm[m] >> (sh - 1)) & 1u;
        const unsigned hi = sh == 24 ? hn[m] & 1u : (hm[m] >> (sh + 8)) & 1u;
        if (u + TEAM * m < kHaloRows)
            M.hr[turn][u + TEAM * m] = lo | (((hm[m] >> sh) & 0xffu) << 1) | (hi << 9);
    }
    if (!first) {
        const unsigned set = (pm >> ((4 * u) & 31)) & 15u;
        int at = 0;      // the order of the winners is free: W is an integer sum
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const bool have = (set >> m) & 1u;
            const unsigned bm = __ballot_sync(0xffffffffu, have);
            if (have) {
                const int slot = 4 * u + m;
                const unsigned e = (unsigned)(ps >> (16 * m)) & 0xffffu;
                const int sx = slot / (kNbh * kNbh), sy = (slot / kNbh) % kNbh, sz = slot % kNbh;
                // winner cell relative to the tile origin
                const int wx = (sx - reach) * A.bs + (int)(e & 3u);
                const int wy = (sy - reach) * A.bs + (int)((e >> 2) & 3u);
                const int wz = (sz - reach) * A.bs + (int)((e >> 4) & 3u);
                M.win[turn][L.w][at + __popc(bm & ((1u << L.lane) - 1u))] =
                    (unsigned)(wx + 8) | ((unsigned)(wy + 8) << 5) | ((unsigned)(wz + 8) << 10) |
                    (((e >> 6) & 1u) << 15);
            }
            at += __popc(bm);
        }
        if (L.lane == 0) M.nw[turn][L.w] = at;
    }
    team_sync(team);

    // ------------------------------------------------- W of the own cells
    if (!first) {
        // the bitmap is consumed: clear it for the next round's postings
        if (u < kNbh3 / 4 && (u & 7) == 0 && pm) pmask[u >> 3] = 0u;
        const int n0 = M.nw[turn][0], nw = n0 + M.nw[turn][1];
        const unsigned *win = M.win[turn][0];
        bool changed = false;
        for (int e = 0; e < nw; ++e) {
            const unsigned wv = win[e < n0 ? e : e - n0 + kSlots * 32];
            const int ax = cx + 8 - (int)(wv & 31u), ay = cy + 8 - (int)((wv >> 5) & 31u),
                      az = 8 - (int)((wv >> 10) & 31u);
            const int sgn = ((wv >> 15) & 1u) ? -1 : 1;   // solute -> solvent lowers W
            if (STENCIL) {      // full stencil: the row of weights at (ax, ay)
                if (abs(ax) > r || abs(ay) > r) continue;
                const int *wr = kt + ((ax + r) * (2 * r + 1) + (ay + r)) * kKtRow + (kKtRow >> 1) + az;
#pragma unroll
                for (int z = 0; z < TS; ++z) Wr[z] += (unsigned)(sgn * wr[z]);
                changed = true;
            } else {
                const int qxy = sgn * qw[ax + kQ0] * qw[ay + kQ0];
                if (qxy == 0) continue;
#pragma unroll
                for (int z = 0; z < TS; ++z) Wr[z] += (unsigned)(qxy * qw[az + z + kQ0]);
                changed = true;
            }
        }
        if (changed && zc) {
            if (A.vec == 2) {
#pragma unroll
                for (int h = 0; h < TS; h += 4)
                    *reinterpret_cast<uint4 *>(A.W + o + h) =
                        make_uint4(Wr[h], Wr[h + 1], Wr[h + 2], Wr[h + 3]);
            } else {
#pragma unroll
                for (int z = 0; z < TS; ++z)
                    if (z < zc) A.W[o + z] = Wr[z];
            }
        }
    }

    // ------------------------------------ candidates, dE, new leaders
    // dE = c [s (1 - 2w) - g0] - s h^3 U with s = 1 - 2 chi, w = W / S and
    // g0 = k0 / S (S the sum of the kernel's weights, k0 its centre weight):
    // the bracket is the integer N = s (S - 2W) - k0 over S, so
    // c * bracket = c_N N with c_N = c / S and one rounding.  FP32 estimates
    // come first and leave the FP64 unit (2 results a clock per SM) the cells
    // that may lead their brick: an estimate is off by at most 4 ulp of
    // |c_N N| + |h^3 U| (2.4e-7 of it), so with bounds of 1e-6 of that sum a
    // cell whose lower bound is positive does not lower the energy, and one
    // whose lower bound lies above another's upper bound comes after it, also
    // in the rounded keys.  What is not finite is settled in FP64.
    {
        const int h = (cx + 1) * 10 + cy + 1;
        const unsigned *hr = M.hr[turn];
        const unsigned c = hr[h];
        const unsigned d = (c ^ hr[h - 10]) | (c ^ hr[h + 10]) | (c ^ hr[h - 1]) |
                           (c ^ hr[h + 1]) | (c ^ (c << 1)) | (c ^ (c >> 1));
        const unsigned cm = (d >> 1) & ((1u << zc) - 1u);
        const unsigned lab = c >> 1;
        unsigned open = 0u;
        float lo[TS], best[2] = {INFINITY, INFINITY};
#pragma unroll
        for (int z = 0; z < TS; ++z) {
            const bool solute = (lab >> z) & 1u;
            const int base = A.ksum - 2 * (int)Wr[z];
            const float t1 = A.cDf * (float)((solute ? -base : base) - A.qc3), t2 = A.h3f * Ur[z];
            const float est = solute ? t1 + t2 : t1 - t2;
            const float err = 1e-6f * (fabsf(t1) + fabsf(t2)) + 1e-30f;
            lo[z] = est - err;
            if (((cm >> z) & 1u) && !(lo[z] > 0.f)) {
                open |= 1u << z;
                best[z >> 2] = fminf(best[z >> 2], est + err);
            }
        }
        // bricks of edge 4: 16 lanes, lane bits 0, 1, 3, 4
        if (bsh == 2) {
#pragma unroll
            for (int m = 1; m <= 16; m = m == 2 ? 8 : 2 * m) {
                best[0] = fminf(best[0], __shfl_xor_sync(0xffffffffu, best[0], m));
                best[1] = fminf(best[1], __shfl_xor_sync(0xffffffffu, best[1], m));
            }
#pragma unroll
            for (int z = 0; z < TS; ++z)
                if (lo[z] > best[z >> 2]) open &= ~(1u << z);
        }
        while (open) {
            const int z = __ffs(open) - 1;
            open &= open - 1;
            unsigned Wv = Wr[0];
            float Uv = Ur[0];
#pragma unroll
            for (int y = 1; y < TS; ++y)
                if (z == y) {
                    Wv = Wr[y];
                    Uv = Ur[y];
                }
            const bool solute = (lab >> z) & 1u;
            const int base = A.ksum - 2 * (int)Wv;
            const int N = (solute ? -base : base) - A.qc3;
            const double t1 = __dmul_rn(A.cD, (double)N);
            const double t2 = __dmul_rn(A.h3, (double)Uv);
            const double e = __dadd_rn(t1, solute ? t2 : -t2);
            if (e < 0.0) {
                const unsigned p = o + (unsigned)z;
                A.dE[p] = e;
                const unsigned key = __float_as_uint(__double2float_rn(e)) & 0x7fffffffu;
                const unsigned long long w = ((unsigned long long)key << 33) |
                                             ((unsigned long long)~p << 1) |
                                             (unsigned long long)solute;
                atomicMax(&M.bmax[((cx >> bsh) * bpt + (cy >> bsh)) * bpt + (z >> bsh)], w);
            }
        }
    }
    __syncwarp();
    turn ^= 1;
    bool any = false, changed = false;
    if (L.lane < per) {
        const unsigned long long w = M.bmax[brick];
        M.bmax[brick] = 0ull;
        if (bq >= 0) {
            changed = w != oldw;
            any = w != 0ull;
            A.PL[bq] = w;
            if (any) {
                // the leader's cell from its linear index, without a division: the
                // offset from the brick's first cell is di nyz + dj nz + dk
                const int gx = ti * bpt + brick / (bpt * bpt), gy = tj * bpt + (brick / bpt) % bpt,
                          gz = tk * bpt + brick % bpt;
                int d = (int)~(unsigned)(w >> 1) -
                        ((gx << bsh) * nyz + (gy << bsh) * g.nz + (gz << bsh));
                unsigned di = 0, dj = 0;
                for (int s = 1; s < A.bs; ++s)
                    if (d >= nyz) {
                        d -= nyz;
                        ++di;
                    }
                for (int s = 1; s < A.bs; ++s)
                    if (d >= g.nz) {
                        d -= g.nz;
                        ++dj;
                    }
                A.PO[bq] = (uint8_t)(di | (dj << 2) | ((unsigned)d << 4));
            }
        }
    }
    if (stamp && __any_sync(0xffffffffu, changed) && L.lane < 27) {
        const int a = ti + L.lane / 9 - 1, b = tj + (L.lane / 3) % 3 - 1, c = tk + L.lane % 3 - 1;
        if (a >= 0 && b >= 0 && c >= 0 && a < A.ntx && b < A.nty && c < A.ntz)
            set_tile_bit(A, stamp, (unsigned)((a * A.nty + b) * A.ntz + c));
    }
    return __any_sync(0xffffffffu, any);
}

struct SweepShared {
    unsigned own[2][kOwnWords];    // half w of own tile j holds a leader
    int qw[2 * kQ0];
    double e[2 * NTEAM];
    unsigned nf[2 * NTEAM];
    unsigned ncnt;
    int nown;                  // own half tiles holding a leader
    int abort_flag;
};

// Visits this team's share of the block's tiles whose bit is set in word(k),
// k < words (bit b of word k is own tile 32 k + b): of the set bits in order,
// team q takes numbers q, q + NTEAM, ...  Every warp holds 32 words, one per
// lane, with a running count, and finds its next bit by rank (twelve
// instructions a visit; walking all the bits cost every warp eight per bit).
// Returns the number of set bits.
template <class Word, class Visit>
__device__ __forceinline__ int each_tile(int words, int team, Word word, Visit visit)
{
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int n = 0, next = team;
    for (int base = 0; base < words; base += 32) {
        const unsigned mine = base + lane < words ? word(base + lane) : 0u;
        const int cnt = __popc(mine);
        int upto = cnt;           // set bits of this and the lower lanes' words
        const int held = min(words - base, 32);
        for (int s = 1; s < held; s <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, upto, s);
            if (lane >= s) upto += v;
        }
        const int total = __shfl_sync(0xffffffffu, upto, held - 1);
        for (; next - n < total; next += NTEAM) {
            const int want = next - n;
            // the word holding it, then the bit of that rank in the word
            const int l = __ffs(__ballot_sync(0xffffffffu, upto > want)) - 1;
            const unsigned m = __shfl_sync(0xffffffffu, mine, l);
            const int rank = want - __shfl_sync(0xffffffffu, upto - cnt, l);
            const int bit = __ffs(__ballot_sync(0xffffffffu, ((m >> lane) & 1u) != 0u &&
                                                                 __popc(m & below) == rank)) - 1;
            visit(32 * (base + l) + bit);
        }
        n += total;
    }
    return n;
}

// Clears a block's words of a bitmap.
__device__ __forceinline__ void clear_words(unsigned *map, int words)
{
    for (int k = threadIdx.x; k < words; k += SW_THREADS) map[k] = 0u;
}

// Mask of the own tiles 32 k .. 32 k + 31 that exist among ntiles.
__device__ __forceinline__ unsigned tile_mask(int k, int nown, long long ntiles)
{
    unsigned m = 0u;
    for (int b = 0; b < 32; ++b)
        if (32 * k + b < nown && own_tile_no(32 * k + b) < ntiles) m |= 1u << b;
    return m;
}

// Records whether half w of own tile j holds a leader, keeping the counts.
__device__ __forceinline__ void set_own(SweepShared &S, int w, int j, bool now, unsigned *nlead,
                                        unsigned *nlead_sys)
{
    const unsigned bit = 1u << (j & 31);
    unsigned *word = &S.own[w][j >> 5];
    if (now == ((*word & bit) != 0u)) return;
    if (now) atomicOr(word, bit);
    else atomicAnd(word, ~bit);
    atomicAdd(&S.nown, now ? 1 : -1);
    red_add(nlead, now ? 1u : 0xffffffffu);
    if (nlead_sys) red_add(nlead_sys, now ? 1u : 0xffffffffu);
}

// Shared set-up of a sweep block: weights, stencil, counters, team areas.
__device__ __forceinline__ void sweep_init(SweepShared &S, TeamMem *TM, int *kt,
                                           const KernelW &kw, const int *k3)
{
    if (kt) {
        const int w = 2 * kw.r + 1;
        for (int a = threadIdx.x; a < w * w * kKtRow; a += SW_THREADS) {
            const int row = a / kKtRow, z = a - row * kKtRow - (kKtRow >> 1);
            kt[a] = abs(z) <= kw.r ? k3[row * w + z + kw.r] : 0;
        }
    }
    for (int a = threadIdx.x; a < 2 * kQ0; a += SW_THREADS) {
        const int d = a - kQ0;
        S.qw[a] = abs(d) <= kw.r ? kw.q[d + kw.r] : 0;
    }
    for (int a = threadIdx.x; a < 2 * kOwnWords; a += SW_THREADS)
        S.own[a / kOwnWords][a % kOwnWords] = 0u;
    for (int a = threadIdx.x; a < NTEAM * kMaxBricksPerTile; a += SW_THREADS)
        TM[a / kMaxBricksPerTile].bmax[a % kMaxBricksPerTile] = 0ull;
    if (threadIdx.x == 0) {
        S.abort_flag = 0;
        S.ncnt = 1u;
        S.nown = 0;
    }
    __syncthreads();
}

template <bool STENCIL>
__global__ void __launch_bounds__(SW_THREADS, 1)
k_sweep(SweepArgs A)
{
    __shared__ SweepShared S;
    extern __shared__ __align__(16) unsigned char dyn[];
    TeamMem *TM = reinterpret_cast<TeamMem *>(dyn);
    // the full stencil, if any, follows the teams' areas
    int *kt = STENCIL ? reinterpret_cast<int *>(dyn + NTEAM * sizeof(TeamMem)) : nullptr;
    const int ntiles = A.ntx * A.nty * A.ntz;
    const int nown = (ntiles + (int)gridDim.x - 1) / (int)gridDim.x;    // or one fewer
    const int words = (nown + 31) / 32;
    const int team = threadIdx.x / TEAM;
    TeamMem &M = TM[team];
    const Lane L = make_lane(TS >> A.bsh, A.reach);
    unsigned *upd = A.upd + (size_t)blockIdx.x * A.bwords;
    unsigned *stamp = A.stamp + (size_t)blockIdx.x * A.bwords;
    sweep_init(S, TM, kt, A.kw, A.k3);
    Barrier B{A.bar, 0u, A.err, A.spin_limit};
    auto own_tile = [&](int j) { return make_tile(A, (int)own_tile_no(j)); };
    int turn = 0, uturn = 0;
    double e_lane = 0.0;
    unsigned n_lane = 0;
    unsigned long long t_dec = 0, t_upd = 0;   // tiles visited per phase
    int round = 0, capped = 0;
    bool marked = false;      // the last update stamped the tiles to decide
    // opening pass: leaders of the starting labels
    each_tile(words, team, [&](int k) { return tile_mask(k, nown, ntiles); }, [&](int j) {
        const bool now =
            tile_update<STENCIL>(A, M, S.qw, kt, L, team, own_tile(j), true, nullptr, uturn);
        if (L.lane == 0) set_own(S, L.w, j, now, A.nlead, nullptr);
    });
    bool ok = all_blocks(B, &S.abort_flag);
    for (int k = 0; ok; ++k) {
        const unsigned here = (k & 1) * A.mapw, last = A.mapw - here;
        if (k >= A.max_rounds) {     // cap reached: capped if leaders are left
            round = k;
            capped = -1;
            break;
        }
        // decide (the global leader count is read meanwhile; it only
        // changes in the update phases)
        unsigned nl = 1u;
        if (threadIdx.x == 0) nl = ld_relaxed_u32(A.nlead);
        const bool stamped = marked && (A.stamps > 0 || S.nown > 2 * NTEAM);
        t_dec += (unsigned long long)each_tile(
            words, team,
            [&](int w) {
                const unsigned own = S.own[0][w] | S.own[1][w];
                return stamped ? own & __ldcg(stamp + last + w) : own;
            },
            [&](int j) {
                tile_decide(A, M, L, team, own_tile(j), turn, A.upd + here, e_lane, n_lane);
            });
        clear_words(upd + last, words);
        if (threadIdx.x == 0) S.ncnt = nl;
        ok = all_blocks(B, &S.abort_flag);
        if (!ok) break;
        // (S.ncnt: the leader half tiles of this round, alike in every block)
        if (S.ncnt == 0u) {          // no leader was left: converged
            round = k;
            break;
        }
        if (marked) clear_words(stamp + last, words);
        marked = A.stamps > 0 || (A.stamps < 0 && S.ncnt > (unsigned)(2 * NTEAM * gridDim.x));
        unsigned *mark = marked ? A.stamp + here : nullptr;
        t_upd += (unsigned long long)each_tile(
            words, team, [&](int w) { return __ldcg(upd + here + w); }, [&](int j) {
                const bool now =
                    tile_update<STENCIL>(A, M, S.qw, kt, L, team, own_tile(j), false, mark, uturn);
                if (L.lane == 0) set_own(S, L.w, j, now, A.nlead, nullptr);
            });
        ok = all_blocks(B, &S.abort_flag);
    }
    if (!ok) return;
    // FP64 sums of the flipped cells' dE and their counts: the lanes of the
    // warps, then the warps in order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        e_lane += __shfl_down_sync(0xffffffffu, e_lane, o);
        n_lane += __shfl_down_sync(0xffffffffu, n_lane, o);
    }
    if (L.lane == 0) {
        S.e[threadIdx.x >> 5] = e_lane;
        S.nf[threadIdx.x >> 5] = n_lane;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double te = 0.0;
        unsigned long long tf = 0;
        for (int q = 0; q < 2 * NTEAM; ++q) {
            te += S.e[q];
            tf += S.nf[q];
        }
        A.part_flips[blockIdx.x] = tf;
        A.part_dE[blockIdx.x] = te;
        A.part_tiles[blockIdx.x] = t_dec;
        A.part_tiles[gridDim.x + blockIdx.x] = t_upd;
        if (blockIdx.x == 0) {
            *A.rounds_out = round;
            *A.capped_out = capped < 0 ? (ld_relaxed_u32(A.nlead) != 0u) : 0;
        }
    }
}

// Totals over the blocks, one warp: lane l adds blocks l, l + 32, ... in
// order, then a fixed tree (one thread adding 152 blocks took 26 us).
__global__ void __launch_bounds__(32)
k_sweep_final(const unsigned long long *part_flips, const double *part_dE,
              const unsigned long long *part_tiles, int nb, const int *rounds, const int *capped,
              RoundState *rs)
{
    unsigned long long f = 0, td = 0, tu = 0;
    double e = 0.0;
    for (int b = threadIdx.x; b < nb; b += 32) {
        f += part_flips[b];
        e += part_dE[b];
        td += part_tiles[b];
        tu += part_tiles[nb + b];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        f += __shfl_down_sync(0xffffffffu, f, o);
        e += __shfl_down_sync(0xffffffffu, e, o);
        td += __shfl_down_sync(0xffffffffu, td, o);
        tu += __shfl_down_sync(0xffffffffu, tu, o);
    }
    if (threadIdx.x) return;
    rs->tiles_decide = td;
    rs->tiles_update = tu;
    rs->done = 1;
    rs->round = *rounds;
    rs->capped = *capped;
    rs->round_flips = 0;
    rs->total_flips = f;
    rs->round_dE = 0.0;
    rs->total_dE = e;
}

int sweep_tiles(const GridDesc &g)
{
    return ((g.nx + TS - 1) / TS) * ((g.ny + TS - 1) / TS) * ((g.nz + TS - 1) / TS);
}

int sweep_brick_edge(int r) { return sweep_edge(r); }

long long sweep_bricks(const GridDesc &g, int r)
{
    const int b = sweep_brick_edge(r);
    return (long long)((g.nx + b - 1) / b) * ((g.ny + b - 1) / b) * ((g.nz + b - 1) / b);
}

static size_t pad256(size_t x) { return (x + 255) / 256 * 256; }

// Words per block of a bitmap over nt tiles, and bytes of the bitmap, for a
// grid of `blocks` blocks (at most kMaxSweepBlocks).
constexpr int kMaxSweepBlocks = 256;
static int bitmap_words(size_t nt, int blocks) { return (int)((nt + 32ull * blocks - 1) / (32ull * blocks)); }
static size_t bitmap_bytes_max(size_t nt) { return pad256((nt / 32 + 2 * kMaxSweepBlocks) * 4); }

// Sweep state: leader words, leader offsets, the per-tile posting areas, the
// update and stamp bitmaps and the label bits.
size_t sweep_state_bytes(const GridDesc &g, int r)
{
    const size_t nt = (size_t)sweep_tiles(g);
    const size_t nb = (size_t)sweep_bricks(g, r);
    const size_t nzw = ((size_t)g.nz + 31) / 32;
    return nb * 8 + pad256(nb) + nt * kPostBytes + 4 * bitmap_bytes_max(nt) +
           (size_t)g.nx * g.ny * nzw * 4;
}

// Label bits: word w of column (i, j) holds cells 32 w .. 32 w + 31 of the
// column (bit = cell - 32 w), zero past its end; the words are stored plane
// by plane, word (w, i, j) at (w nx + i) ny + j.
__global__ void k_pack_labels(const uint8_t *__restrict__ chi, int nz, long long nxy,
                              long long nwords, unsigned *__restrict__ CB)
{
    const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nwords) return;
    const long long wz = w / nxy, col = w - wz * nxy;
    const int k0 = (int)wz * 32;
    const uint8_t *src = chi + col * nz + k0;
    const int n = min(32, nz - k0);
    unsigned b = 0u;
    if (n == 32 && ((uintptr_t)src & 15u) == 0) {   // two 16-byte loads
        const uint4 v0 = *reinterpret_cast<const uint4 *>(src);
        const uint4 v1 = *reinterpret_cast<const uint4 *>(src + 16);
        const unsigned q[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
        for (int k = 0; k < 32; ++k)
            b |= (((q[k >> 2] >> (8 * (k & 3))) & 0xffu) != 0u ? 1u : 0u) << k;
    } else {
        for (int k = 0; k < n; ++k) b |= (src[k] != 0 ? 1u : 0u) << k;
    }
    CB[w] = b;
}

// teams' areas plus room for the largest full stencil (17^2 rows)
constexpr size_t kSweepSmem =
    NTEAM * sizeof(TeamMem) + sizeof(int) * (2 * kMaxR + 1) * (2 * kMaxR + 1) * kKtRow;

cudaError_t sweep_grid_size(int nsm, int r, int *blocks)
{
    (void)r;
    cudaError_t e = cudaSuccess;
    int per = 1;          // one block per SM: a barrier of few blocks
    for (int q = 0; q < 2; ++q) {
        void *fn = q ? (void *)k_sweep<true> : (void *)k_sweep<false>;
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSweepSmem);
        if (e != cudaSuccess) return e;
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, SW_THREADS, kSweepSmem);
        if (e != cudaSuccess) return e;
        per = n < per ? n : per;
    }
    *blocks = per * nsm < kMaxSweepBlocks ? per * nsm : kMaxSweepBlocks;
    return *blocks > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

int sweep_ctl_words() { return kCtlWords; }

// Arguments of one system's sweep, with its set-up enqueued on st: the
// posting bitmaps and control words cleared and the label bits packed (leader
// words are all rewritten by the opening pass).
static SweepArgs sweep_setup(const GridDesc &g, const KernelW &kw, const int *k3,
                             const FlipConst &fc, uint8_t *chi, uint32_t *W, const float *U,
                             double *dE, void *state, unsigned *ctl, int *err, int max_rounds,
                             int blocks, long long spin_limit, cudaStream_t st)
{
    SweepArgs A;
    A.g = g;
    A.kw = kw;
    A.cD = fc.cN;
    A.h3 = fc.h3;
    A.cDf = (float)fc.cN;
    A.h3f = (float)fc.h3;
    A.qc3 = fc.k0;
    A.ksum = fc.S;
    A.k3 = k3;
    A.chi = chi;
    A.W = W;
    A.U = U;
    A.dE = dE;
    A.ntx = (g.nx + TS - 1) / TS;
    A.nty = (g.ny + TS - 1) / TS;
    A.ntz = (g.nz + TS - 1) / TS;
    A.bs = sweep_brick_edge(kw.r);
    A.bsh = A.bs == 4 ? 2 : 1;
    A.reach = (kw.r + A.bs - 1) / A.bs;
    A.nbx = (g.nx + A.bs - 1) / A.bs;
    A.nby = (g.ny + A.bs - 1) / A.bs;
    A.nbz = (g.nz + A.bs - 1) / A.bs;
    A.vec = (uintptr_t)W % 16 || (uintptr_t)U % 16 ? 0 : g.nz % TS == 0 ? 2 : 1;
    A.ncell = (unsigned)g.nx * (unsigned)(g.ny * g.nz);
    const size_t nb = (size_t)A.nbx * A.nby * A.nbz;
    const size_t nt = (size_t)A.ntx * A.nty * A.ntz;
    uint8_t *base = static_cast<uint8_t *>(state);
    A.PL = reinterpret_cast<unsigned long long *>(base);
    A.PO = base + nb * 8;
    A.post = A.PO + pad256(nb);
    uint8_t *maps = A.post + nt * kPostBytes;
    A.upd = reinterpret_cast<unsigned *>(maps);
    A.stamp = reinterpret_cast<unsigned *>(maps + 2 * bitmap_bytes_max(nt));
    A.CB = reinterpret_cast<unsigned *>(maps + 4 * bitmap_bytes_max(nt));
    A.mapw = (unsigned)(bitmap_bytes_max(nt) / 4);
    A.bwords = bitmap_words(nt, blocks);
    A.tile0 = 0;
    A.nblk = (unsigned)blocks;
    auto inv = [](int d) { return (unsigned)(((1ull << 32) + d - 1) / d); };
    A.nblk_inv = inv(blocks);
    A.nty_inv = inv(A.nty);
    A.ntz_inv = inv(A.ntz);
    A.nzw = (g.nz + 31) / 32;
    A.nlead = ctl;
    A.bar = ctl + kLine;
    A.err = err;
    A.part_flips = nullptr;
    A.part_dE = nullptr;
    A.part_tiles = nullptr;
    A.rounds_out = nullptr;
    A.capped_out = nullptr;
    A.max_rounds = max_rounds;
    A.spin_limit = spin_limit;
    A.stamps = -1;
    A.rs = nullptr;
    A.tile_dE = nullptr;
    A.tile_nf = nullptr;
    // postings start empty (a slot is only read under its bitmap bit)
    cudaMemset2DAsync(A.post + kPostMaskOff, kPostBytes, 0, 32, nt, st);
    cudaMemsetAsync(maps, 0, 4 * bitmap_bytes_max(nt), st);
    cudaMemsetAsync(ctl, 0, sweep_ctl_words() * sizeof(unsigned), st);
    cudaMemsetAsync(err, 0, sizeof(int), st);
    {
        const long long nwords = (long long)g.nx * g.ny * A.nzw;
        count_launch();
        k_pack_labels<<<(unsigned)((nwords + 255) / 256), 256, 0, st>>>(
            chi, g.nz, (long long)g.nx * g.ny, nwords, A.CB);
    }
    return A;
}

cudaError_t launch_sweep(const GridDesc &g, const KernelW &kw, const int *k3,
                         const FlipConst &fc,
                         uint8_t *chi, uint32_t *W, const float *U,
                         double *dE, void *state, unsigned *ctl, int *err,
                         unsigned long long *part_flips, double *part_dE,
                         unsigned long long *part_tiles,
                         int *rounds, int *capped, int max_rounds, int blocks,
                         long long spin_limit, int stamps, RoundState *rs, cudaStream_t st)
{
    {
        const size_t nt = (size_t)sweep_tiles(g);
        if ((nt + blocks - 1) / blocks > (size_t)kOwnWords * 32) return cudaErrorInvalidValue;
    }
    SweepArgs A = sweep_setup(g, kw, k3, fc, chi, W, U, dE, state, ctl, err, max_rounds, blocks,
                              spin_limit, st);
    A.part_flips = part_flips;
    A.part_dE = part_dE;
    A.part_tiles = part_tiles;
    A.rounds_out = rounds;
    A.capped_out = capped;
    A.stamps = stamps;
    void *args[] = {&A};
    count_launch();
    void *fn = k3 ? (void *)k_sweep<true> : (void *)k_sweep<false>;
    const cudaError_t e =
        cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(SW_THREADS), args, kSweepSmem, st);
    if (e != cudaSuccess) return e;
    count_launch();
    k_sweep_final<<<1, 32, 0, st>>>(part_flips, part_dE, part_tiles, blocks, rounds, capped, rs);
    return cudaGetLastError();
}


// ------------------------------------------------- many systems at once
// The same rounds for up to kMaxSweepSys systems in one cooperative launch:
// the systems' tiles are numbered one after another and dealt round-robin
// over the blocks, each round's decide and update phases serve the tiles of
// every system, and one grid barrier closes each phase for all of them.
// Every system's leaders, postings, labels and W live in its own state
// exactly as in the single-system sweep, so each system goes through the
// same rounds as alone.  A system whose leaders are gone contributes no
// tiles; the launch ends when no system has any.  The FP64 sum of a tile's
// flipped dE is kept per half tile (its warp adds it, round after round) and
// summed over the system's half tiles in order at the end.

// dynamic shared memory offset of the systems' arguments (16-byte aligned)
constexpr size_t kSweepSysOff = (kSweepSmem + 15) / 16 * 16;

struct MultiArgs {
    const SweepArgs *sys;     // [nsys] (device)
    const long long *toff;    // [nsys + 1]: first global tile of each system
    int nsys;
    int ntiles;
    unsigned *nlead;          // half tiles holding a leader, all systems (own line)
    unsigned *bar;            // grid barrier arrivals (own line)
    int *err;
    int *rounds;              // [nsys]
    int *capped;              // [nsys]
    unsigned *upd, *stamp;    // bitmaps over all systems' tiles, two of each
    int bwords;
    unsigned mapw;
    int max_rounds;
    long long spin_limit;
    int stamps;               // as SweepArgs::stamps, for all systems
    KernelW kw;
    const int *k3;
};

__device__ __forceinline__ int sys_of(const long long *toff, int nsys, long long tg)
{
    int lo = 0, hi = nsys;    // toff[lo] <= tg < toff[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (toff[mid] <= tg) lo = mid;
        else hi = mid;
    }
    return lo;
}

template <bool STENCIL>
__global__ void __launch_bounds__(SW_THREADS, 1)
k_sweep_multi(MultiArgs P)
{
    __shared__ SweepShared S;
    __shared__ long long s_toff[kMaxSweepSys + 1];
    __shared__ int s_rounds[kMaxSweepSys];
    extern __shared__ __align__(16) unsigned char dyn[];
    TeamMem *TM = reinterpret_cast<TeamMem *>(dyn);
    int *kt = STENCIL ? reinterpret_cast<int *>(dyn + NTEAM * sizeof(TeamMem)) : nullptr;
    // after the teams' areas and the stencil: the systems' arguments
    SweepArgs *s_sys = reinterpret_cast<SweepArgs *>(dyn + kSweepSysOff);
    const int nsys = P.nsys;
    const int nown = (P.ntiles + (int)gridDim.x - 1) / (int)gridDim.x;      // or one fewer
    const int words = (nown + 31) / 32;
    const int team = threadIdx.x / TEAM;
    TeamMem &M = TM[team];
    {
        const int nwords = nsys * (int)(sizeof(SweepArgs) / 4);
        const unsigned *src = reinterpret_cast<const unsigned *>(P.sys);
        unsigned *dst = reinterpret_cast<unsigned *>(s_sys);
        for (int a = threadIdx.x; a < nwords; a += SW_THREADS) dst[a] = src[a];
    }
    for (int a = threadIdx.x; a <= nsys; a += SW_THREADS) s_toff[a] = P.toff[a];
    for (int a = threadIdx.x; a < nsys; a += SW_THREADS) s_rounds[a] = 0;
    sweep_init(S, TM, kt, P.kw, P.k3);
    unsigned *upd = P.upd + (size_t)blockIdx.x * P.bwords;
    unsigned *stamp = P.stamp + (size_t)blockIdx.x * P.bwords;
    const Lane L = make_lane(TS / sweep_edge(P.kw.r), (P.kw.r + sweep_edge(P.kw.r) - 1) / sweep_edge(P.kw.r));
    Barrier B{P.bar, 0u, P.err, P.spin_limit};
    // own tile j: its system, and its number there
    auto own_sys = [&](int j, int &t) {
        const long long tg = own_tile_no(j);
        const int q = sys_of(s_toff, nsys, tg);
        t = (int)(tg - s_toff[q]);
        return q;
    };
    int uturn = 0;
    auto update = [&](int j, bool first, unsigned *mark) {
        int t;
        const SweepArgs &A = s_sys[own_sys(j, t)];
        const bool now =
            tile_update<STENCIL>(A, M, S.qw, kt, L, team, make_tile(A, t), first, mark, uturn);
        if (L.lane == 0) set_own(S, L.w, j, now, P.nlead, A.nlead);
    };
    int capped = 0, turn = 0;
    bool marked = false;
    // opening pass: leaders of every system's starting labels
    each_tile(words, team, [&](int k) { return tile_mask(k, nown, P.ntiles); },
              [&](int j) { update(j, true, nullptr); });
    if (!all_blocks(B, &S.abort_flag)) return;
    for (int k = 0;; ++k) {
        const unsigned here = (k & 1) * P.mapw, last = P.mapw - here;
        if (k >= P.max_rounds) {
            capped = 1;
            break;
        }
        unsigned nl = 1u;
        if (threadIdx.x == 0) nl = ld_relaxed_u32(P.nlead);
        if (blockIdx.x == 0)         // rounds of each system that still had leaders
            for (int q = threadIdx.x; q < nsys; q += SW_THREADS)
                if (ld_relaxed_u32(s_sys[q].nlead) != 0u) s_rounds[q] = k + 1;
        const bool stamped = marked && (P.stamps > 0 || S.nown > 2 * NTEAM);
        each_tile(
            words, team,
            [&](int w) {
                const unsigned own = S.own[0][w] | S.own[1][w];
                return stamped ? own & __ldcg(stamp + last + w) : own;
            },
            [&](int j) {
                int t;
                const SweepArgs &A = s_sys[own_sys(j, t)];
                double e = 0.0;
                unsigned nf = 0;
                tile_decide(A, M, L, team, make_tile(A, t), turn, P.upd + here, e, nf);
                if (__any_sync(0xffffffffu, nf != 0u)) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        e += __shfl_down_sync(0xffffffffu, e, o);
                        nf += __shfl_down_sync(0xffffffffu, nf, o);
                    }
                    if (L.lane == 0) {
                        A.tile_dE[2 * t + L.w] += e;
                        A.tile_nf[2 * t + L.w] += nf;
                    }
                }
            });
        clear_words(upd + last, words);
        if (threadIdx.x == 0) S.ncnt = nl;
        if (!all_blocks(B, &S.abort_flag)) return;
        if (S.ncnt == 0u) break;
        if (marked) clear_words(stamp + last, words);
        marked = P.stamps > 0 || (P.stamps < 0 && S.ncnt > (unsigned)(2 * NTEAM * gridDim.x));
        unsigned *mark = marked ? P.stamp + here : nullptr;
        each_tile(words, team, [&](int w) { return __ldcg(upd + here + w); },
                  [&](int j) { update(j, false, mark); });
        if (!all_blocks(B, &S.abort_flag)) return;
    }
    if (blockIdx.x == 0) {
        __syncthreads();
        for (int q = threadIdx.x; q < nsys; q += SW_THREADS) {
            P.rounds[q] = s_rounds[q];
            P.capped[q] = capped && ld_relaxed_u32(s_sys[q].nlead) != 0u;
        }
    }
}

// Totals of system blockIdx.x: its tiles' flip counts and dE sums added in
// a fixed order (strided per thread, then a tree over the threads).
__global__ void __launch_bounds__(256) k_sweep_multi_final(const SweepArgs *sys,
                                                           const int *rounds, const int *capped)
{
    __shared__ double se[256];
    __shared__ unsigned long long sf[256];
    const SweepArgs &A = sys[blockIdx.x];
    const int nt = 2 * A.ntx * A.nty * A.ntz;
    double e = 0.0;
    unsigned long long f = 0;
    for (int t = threadIdx.x; t < nt; t += 256) {
        e += A.tile_dE[t];
        f += A.tile_nf[t];
    }
    se[threadIdx.x] = e;
    sf[threadIdx.x] = f;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            se[threadIdx.x] += se[threadIdx.x + w];
            sf[threadIdx.x] += sf[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        RoundState *rs = A.rs;
        rs->done = 1;
        rs->round = rounds[blockIdx.x];
        rs->capped = capped[blockIdx.x];
        rs->round_flips = 0;
        rs->total_flips = sf[0];
        rs->round_dE = 0.0;
        rs->total_dE = se[0];
        rs->tiles_decide = 0;
        rs->tiles_update = 0;
    }
}

static size_t pad256z(size_t x) { return (x + 255) / 256 * 256; }

size_t sweep_multi_scratch_bytes(int nsys, long long tiles)
{
    return pad256z((size_t)nsys * sizeof(SweepArgs)) + pad256z((size_t)(nsys + 1) * 8) +
           pad256z(kCtlWords * sizeof(unsigned)) + pad256z(sizeof(int)) +
           2 * pad256z((size_t)nsys * sizeof(int)) + 4 * bitmap_bytes_max((size_t)tiles);
}

cudaError_t launch_sweep_multi(int nsys, const SweepSys *sys, const KernelW &kw, const int *k3,
                               int max_rounds, int blocks, long long spin_limit, int stamps,
                               void *scratch, int *err_out, cudaStream_t st)
{
    if (nsys < 1 || nsys > kMaxSweepSys) return cudaErrorInvalidValue;
    std::vector<SweepArgs> As((size_t)nsys);
    std::vector<long long> toff((size_t)nsys + 1, 0);
    for (int q = 0; q < nsys; ++q) {
        const SweepSys &y = sys[q];
        const int nt = sweep_tiles(y.g);
        toff[q + 1] = toff[q] + nt;
        As[q] = sweep_setup(y.g, kw, k3, y.fc, y.chi, y.W, y.U, y.dE, y.state, y.ctl, y.err,
                            max_rounds, blocks, spin_limit, y.st);
        As[q].rs = y.rs;
        As[q].tile_dE = y.tile_dE;
        As[q].tile_nf = y.tile_nf;
        cudaMemsetAsync(y.tile_dE, 0, (size_t)2 * nt * sizeof(double), y.st);
        cudaMemsetAsync(y.tile_nf, 0, (size_t)2 * nt * sizeof(unsigned), y.st);
    }
    if (toff[nsys] > 0x7fffffffll ||
        (toff[nsys] + blocks - 1) / blocks > (long long)kOwnWords * 32)
        return cudaErrorInvalidValue;
    // the systems' set-up ran on their own streams: st waits for all of it
    for (int q = 0; q < nsys; ++q) {
        cudaEvent_t ev;
        cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e != cudaSuccess) return e;
        cudaEventRecord(ev, sys[q].st);
        cudaStreamWaitEvent(st, ev, 0);
        cudaEventDestroy(ev);
    }
    uint8_t *b = static_cast<uint8_t *>(scratch);
    SweepArgs *d_sys = reinterpret_cast<SweepArgs *>(b);
    b += pad256z((size_t)nsys * sizeof(SweepArgs));
    long long *d_toff = reinterpret_cast<long long *>(b);
    b += pad256z((size_t)(nsys + 1) * 8);
    unsigned *d_ctl = reinterpret_cast<unsigned *>(b);
    b += pad256z(kCtlWords * sizeof(unsigned));
    int *d_err = reinterpret_cast<int *>(b);
    b += pad256z(sizeof(int));
    int *d_rounds = reinterpret_cast<int *>(b);
    b += pad256z((size_t)nsys * sizeof(int));
    int *d_capped = reinterpret_cast<int *>(b);
    b += pad256z((size_t)nsys * sizeof(int));
    // the tiles of all systems share the launch's two bitmaps
    const size_t map_bytes = bitmap_bytes_max((size_t)toff[nsys]);
    unsigned *d_upd = reinterpret_cast<unsigned *>(b);
    unsigned *d_stamp = reinterpret_cast<unsigned *>(b + 2 * map_bytes);
    const int bwords = bitmap_words((size_t)toff[nsys], blocks);
    cudaMemsetAsync(d_upd, 0, 4 * map_bytes, st);
    for (int q = 0; q < nsys; ++q) {
        As[q].upd = d_upd;
        As[q].stamp = d_stamp;
        As[q].bwords = bwords;
        As[q].mapw = (unsigned)(map_bytes / 4);
        As[q].tile0 = (unsigned)toff[q];
    }
    cudaMemcpyAsync(d_sys, As.data(), (size_t)nsys * sizeof(SweepArgs), cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_toff, toff.data(), (size_t)(nsys + 1) * 8, cudaMemcpyHostToDevice, st);
    cudaMemsetAsync(d_ctl, 0, kCtlWords * sizeof(unsigned), st);
    cudaMemsetAsync(d_err, 0, sizeof(int), st);
    MultiArgs P;
    P.sys = d_sys;
    P.toff = d_toff;
    P.nsys = nsys;
    P.ntiles = (int)toff[nsys];
    P.nlead = d_ctl;
    P.bar = d_ctl + kLine;
    P.err = d_err;
    P.rounds = d_rounds;
    P.capped = d_capped;
    P.upd = d_upd;
    P.stamp = d_stamp;
    P.bwords = bwords;
    P.mapw = (unsigned)(map_bytes / 4);
    P.max_rounds = max_rounds;
    P.spin_limit = spin_limit;
    P.stamps = stamps;
    P.kw = kw;
    P.k3 = k3;
    const size_t smem = kSweepSysOff + (size_t)nsys * sizeof(SweepArgs);
    void *fn = k3 ? (void *)k_sweep_multi<true> : (void *)k_sweep_multi<false>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kSweepSysOff + kMaxSweepSys * sizeof(SweepArgs)));
    if (e != cudaSuccess) return e;
    void *args[] = {&P};
    count_launch();
    e = cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(SW_THREADS), args, smem, st);
    if (e != cudaSuccess) return e;
    count_launch();
    k_sweep_multi_final<<<nsys, 256, 0, st>>>(d_sys, d_rounds, d_capped);
    if (err_out) cudaMemcpyAsync(err_out, d_err, sizeof(int), cudaMemcpyDeviceToHost, st);
    return cudaGetLastError();
}

}  // namespace vesis
