// Argument blocks of the packing kernel and the neighbour-list build.
#pragma once

#include "batch.cuh"
#include "neighbors.cuh"
#include "sph_internal.cuh"

namespace sph {

struct PackArgs {
    int n;
    int mixed;
    const double *x, *y, *h, *m, *p, *u, *v;
    double lo[2], Ad[2];        // anchor origin and side (FP64)
    Anchor an;
    float4 *pk;                 // {xl, yl, h, gx | gy << 16}
    float *mf, *pf, *uf, *vf;
};

// The permutation gather of a rebuild (f[perm[i]] to falt[i]; the first
// fields of g are x, y, u, v, p, rho, m, h), with everything the sorted
// order gives at once: levels, anchor records and float mirrors, and the
// cell table's entries.
struct GatherPackRec {
    int n;
    int lshift;                 // 2 * mbits: level = skey >> lshift
    const uint32_t *perm;
    GatherList g;
    const uint64_t *skey;
    uint64_t *tkey;
    uint32_t *tstart, *tend;
    uint32_t tmask;
    float *tmaxh;               // per slot: the cell's largest h
    uint8_t *lev;
    PackArgs p;                 // outputs, anchor lattice (inputs unused)
};

struct ListArgs {
    int n;
    Grid g;
    Domain d;
    Anchor an;
    const double *x, *y, *h;
    const float4 *pk;
    const uint8_t *lev;
    const uint64_t *skey;       // sorted cell keys (cells are runs of equal keys)
    uint32_t *own;              // entries found by i itself
    uint32_t *rev;              // reverse-entry counters / cursors
    uint32_t *off;              // n + 1 offsets
    uint32_t *list;             // neighbour indices
    uint32_t cap;               // list capacity (entries)
    int *overflow;
    uint32_t *longq, *nlong;    // particles with long reverse segments
    uint32_t *stage;            // n x stage_w staging rows of own entries
    uint32_t stage_w;           // row width (entries)
    uint32_t *max_own;          // largest own-entry count of the build
    uint32_t *queue, *nqueue;   // particles whose own entries overflow a row
    uint32_t *qref;             // per queued particle: its chunk's reference
                                // particle | 2^31 when the chunk spans two
                                // cells (cell-tile walks)
    // skin >= 1: lists hold every pair with r_ij < skin * 3 max(h_i, h_j)
    // (a superset of N(i) for particles that move less than the skin
    // allows); 1: exactly N(i)
    float skin;
    // rows (merged-chunk walk only): the passes read own entries from the
    // staging rows, which are interleaved by 32 particles (entry k of i at
    // [i / 32][k][i % 32]: a warp's loads of its k-th entries are one line);
    // the lists hold reverse entries, and the own entries of the particles
    // whose rows overflowed, whose count own[i] is then (zero for the
    // others)
    bool rows;
    uint32_t *rlen;             // rows: entries of i's row | those on its own
                                // level << 16 (they come first)
    // walk: 1 per-particle team walk, 2 cell tiles with 4-lane teams, 3
    // cell tiles with a lane per particle, 4 the same with neighbouring
    // cells of a level merged into one chunk while they hold at most 32
    // particles, anything else: by set size
    int walk;
};

void launch_pack(cudaStream_t s, const PackArgs &a);
void launch_gather_pack(cudaStream_t s, const GatherPackRec &r, int *launches);
// over the work items of several instances (batched step): the gather with
// the levels and the table entries (256-thread items), and the packing;
// blocks: the persistent grid (resident blocks per SM from the function
// below times the SMs)
void launch_gather_batch(cudaStream_t s, const GatherPackRec *args, const BatchSpan &sp);
void launch_pack_batch(cudaStream_t s, const PackArgs *args, const BatchSpan &sp,
                       int blocks);
int pack_batch_blocks_per_sm();

// Batched builds of small sets (batched step): the per-particle team walk,
// the placement, the queue walk and the segment sorts over the work items
// of several instances (one item: one block of the instance's
// single-launch grid; the queue walk and the long-segment sort take
// fill_queue_blocks() and sort_long_blocks(n) items an instance, which
// change no result).
struct SortSegRec {
    int n;
    uint32_t *off;
    const uint32_t *own;
    uint32_t *list;
    uint32_t cap;
    uint32_t *longq, *nlong;
};
bool list_rows_for(const ListArgs &a);   // whether the size rule takes rows
int list_walk_kind(const ListArgs &a);   // 1 team walk, 2 / 3 cell tiles
int list_place_team(int n);              // lanes per particle of the placement
int fill_queue_blocks();
int sort_long_blocks(int n);
void launch_list_gather_batch(cudaStream_t s, int team, const ListArgs *args, const BatchSpan &sp);
void launch_list_place_batch(cudaStream_t s, int team, const ListArgs *args, const BatchSpan &sp);
void launch_list_fill_queue_batch(cudaStream_t s, const ListArgs *args, const BatchSpan &sp);
void launch_list_sort_rev_batch(cudaStream_t s, const SortSegRec *args, const BatchSpan &sp);
void launch_list_sort_long_batch(cudaStream_t s, const SortSegRec *args, const BatchSpan &sp);
void launch_anchor_pack(cudaStream_t s, int n, const double *x,
                        const double *y, const double *h, const double *lo,
                        const double *A, const Anchor &an, float4 *pk);
// The walk (own entries staged, reverse entries counted), then the
// offsets (off has n + 1 entries), then the fill;
// entries past a.cap are dropped and flag a.overflow, and the offsets end at
// a.cap (list_sort_rev_at).  Before the walk,
// rev[0..n) and the counters nqueue, max_own and nlong must be zero (the
// rebuild's reset and key kernels do that).
void launch_list_walk(cudaStream_t s, const ListArgs &a, int *launches);
void list_offsets(cudaStream_t s, const ListArgs &a, SortScratch &sc, int *launches);
// *total = entries in the rows (ListArgs::rlen)
void launch_row_total(cudaStream_t s, int n, const uint32_t *rlen, unsigned long long *total,
                      int *launches);
// queue: launch the second walk for rows that overflowed (false when the
// caller knows none did).
void build_lists_fill(cudaStream_t s, ListArgs a, bool mixed, bool queue,
                      int *launches);
// Each segment [off[i], off[i+1]) of list in ascending order (short ones in
// registers, long ones queued in longq / *nlong, which must be zero, for a
// warp sort); offsets past cap cut to it.
void sort_segments(cudaStream_t s, int n, uint32_t *off, uint32_t *list,
                   uint32_t cap, uint32_t *longq, uint32_t *nlong,
                   int *launches);

}  // namespace sph
