// Per-rebuild packing (levels, FP32 anchor coordinates, float mirrors) and
// the CSR neighbour lists N(i) (definition and search in neighbors.cuh).
//
// List build: one walk per particle stages its own entries and counts the
// reverse ones -> exclusive scan -> place (own entries copied, reverse
// entries written into the coarser neighbours' lists) -> sort the reverse
// segment of each list, so lists are deterministic: own entries in
// traversal order, then the finer-level entries in ascending index.
#include "debug_checks.cuh"
#include "lists.cuh"
#include "neighbors.cuh"
#include "team.cuh"

#include <algorithm>
#include <type_traits>

namespace sph {

// ------------------------------------------------------------------ pack --
__device__ __forceinline__ void pack_at(const PackArgs &a, int i, double x, double y,
                                        double h, double m, double p, double u, double v) {
    a.pk[i] = anchor_record(x, y, d2f(h), a.lo, a.Ad, a.an);
    if (!a.mixed) return;
    a.mf[i] = d2f(m);
    a.pf[i] = d2f(p);
    a.uf[i] = d2f(u);
    a.vf[i] = d2f(v);
}

__device__ __forceinline__ void pack_at(const PackArgs &a, int i) {
    if (a.mixed)
        pack_at(a, i, a.x[i], a.y[i], a.h[i], a.m[i], a.p[i], a.u[i], a.v[i]);
    else
        pack_at(a, i, a.x[i], a.y[i], a.h[i], 0.0, 0.0, 0.0, 0.0);
}

__global__ void k_pack(PackArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    pack_at(a, i);
}

// The same over the work items of several instances (batched step).
__global__ void __launch_bounds__(BATCH_THREADS)
    k_pack_batch(const PackArgs *__restrict__ args, BatchSpan sp) {
    for (int item = blockIdx.x; item < sp.total; item += gridDim.x) {
        const int q = sp.find(item);
        const PackArgs a = args[q];
        const int i = (item - __ldg(&sp.first[q])) * BATCH_THREADS + (int)threadIdx.x;
        if (i < a.n) pack_at(a, i);
    }
}

// ----------------------------------------------------------- gather, pack --
// One thread a sorted position: the state in the new order, its level,
// anchor record and mirrors from the registers it passes through, and, by
// the thread of a cell's first particle, the cell's table entry.  A cell is
// a run of equal keys: its end and largest h come from the warp's ballot and
// a segmented maximum; the one run that leaves the warp is followed by the
// whole warp.  Bound by memory (88 B read by permutation, 88 + 33 B
// written a particle in a mixed step); one kernel here instead of a gather
// and a second pass over seven of the fields took 1.38 -> 0.71 ms at 16.8M
// particles.
// PACK = false: without the records and mirrors.
template <bool PACK>
__device__ __forceinline__ void gather_pack_at(const GatherPackRec &r, int i) {
    const int n = r.n, lane = threadIdx.x & 31;
    const bool ok = i < n;
    uint64_t key = 0;
    uint32_t hb = 0;
    if (ok) {
        key = r.skey[i];
        uint32_t src = r.perm[i];
        if (!SPH_DCHECK(src < (uint32_t)n)) src = (uint32_t)i;
        double f[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) f[k] = __ldg(&r.g.src[k][src]);
        const int64_t id = __ldg(&r.g.isrc[0][src]);
#pragma unroll
        for (int k = 0; k < 8; ++k) r.g.dst[k][i] = f[k];
        r.g.idst[0][i] = id;
        for (int k = 8; k < r.g.nd; ++k) r.g.dst[k][i] = __ldg(&r.g.src[k][src]);
        r.lev[i] = (uint8_t)(key >> r.lshift);
        if (PACK) pack_at(r.p, i, f[0], f[1], f[7], f[6], f[4], f[2], f[3]);
        hb = __float_as_uint(d2f_up(f[7]));
    }
    // cell heads, the lane after each lane's run, the run's largest h
    uint64_t prev = __shfl_up_sync(0xffffffffu, key, 1);
    if (lane == 0 && ok && i > 0) prev = r.skey[i - 1];
    const bool head = ok && (i == 0 || prev != key);
    const unsigned hm = __ballot_sync(0xffffffffu, head);
    const unsigned bm = hm | ~__ballot_sync(0xffffffffu, ok);
    const unsigned above = bm & ~((2u << lane) - 1u);
    const int next = above ? __ffs(above) - 1 : 32;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_down_sync(0xffffffffu, hb, o);
        if (lane + o < next) hb = max(hb, t);
    }
    uint32_t ext = 0;
    if (hm != 0u && (bm >> 31) == ((hm >> 31) & 1u)) {
        // lane 31 holds a particle, in a cell that starts in this warp
        const uint64_t k31 = __shfl_sync(0xffffffffu, key, 31);
        uint32_t eh = 0;
        for (int b = i - lane + 32; b < n; b += 32) {
            const int j = b + lane;
            const bool same = j < n && r.skey[j] == k31;
            const unsigned m = __ballot_sync(0xffffffffu, same);
            const int cnt = m == 0xffffffffu ? 32 : __ffs(~m) - 1;
            uint32_t hj = 0;
            if (lane < cnt) {
                uint32_t sj = r.perm[j];
                if (!SPH_DCHECK(sj < (uint32_t)n)) sj = (uint32_t)j;
                hj = __float_as_uint(d2f_up(__ldg(&r.g.src[7][sj])));
            }
            eh = max(eh, __reduce_max_sync(0xffffffffu, hj));
            ext += (uint32_t)cnt;
            if (cnt < 32) break;
        }
        if (next == 32) hb = max(hb, eh);
    }
    if (!head) return;
    const uint32_t end = (uint32_t)(i - lane + next) + (next == 32 ? ext : 0u);
    uint32_t slot = hash_slot(key, r.tmask);
    // The table holds at most n keys in 2n slots, so a free slot exists and
    // the probe ends within tmask + 1 steps.
    for (uint32_t it = 0; it <= r.tmask; ++it) {
        const unsigned long long old = atomicCAS((unsigned long long *)&r.tkey[slot],
                                                 (unsigned long long)EMPTY_KEY,
                                                 (unsigned long long)key);
        if (old == EMPTY_KEY || old == key) {
            r.tstart[slot] = (uint32_t)i;
            r.tend[slot] = end;
            r.tmaxh[slot] = __uint_as_float(hb);
            return;
        }
        slot = (slot + 1) & r.tmask;
    }
}

__global__ void __launch_bounds__(256) k_gather_pack(GatherPackRec r) {
    gather_pack_at<true>(r, blockIdx.x * blockDim.x + threadIdx.x);
}

// The same over the work items of several instances (batched step).
__global__ void __launch_bounds__(256)
    k_gather_batch(const GatherPackRec *__restrict__ args, BatchSpan sp) {
    for (int it = blockIdx.x; it < sp.total; it += gridDim.x) {
        const BatchItem b = batch_item(sp, it);
        gather_pack_at<false>(args[b.q], b.vb * 256 + (int)threadIdx.x);
    }
}

// Anchor coordinates of a particle set (static sets: walls, background).
__global__ void k_anchor_pack(int n, const double *x, const double *y,
                              const double *h, double lo0, double lo1,
                              double A0, double A1, Anchor an, float4 *pk) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double lo[2] = {lo0, lo1}, A[2] = {A0, A1};
    pk[i] = anchor_record(x[i], y[i], d2f(h[i]), lo, A, an);
}

// ------------------------------------------------------------ list build --
// A staged entry carries this bit when its particle lies on a coarser level
// than the row's owner (the pair also needs a reverse entry).  Particle
// indices stay below 2^31: a context holds far fewer particles.
constexpr uint32_t STAGE_COARSE = 0x80000000u;

// Membership of candidate j for particle i: FP32 anchor filter with the
// FP64 predicate in its band (exact, for both precisions).
__device__ __forceinline__ bool member(const ListArgs &a, const float4 &pi,
                                       double xi, double yi, double hi,
                                       int j) {
    float dx, dy, r2;
    if (a.skin > 1.0f) {
        // skin lists: a superset is all that is needed, and the skin is far
        // wider than the FP32 error of the separation
        const float4 pj = __ldg(&a.pk[j]);
        anchor_sep(a.an, pi, pj, dx, dy);
        const float R = a.skin * 3.0f * fmaxf(pi.z, pj.z);
        return fmaf(dx, dx, dy * dy) < R * R;
    }
    return pred_mixed(a.d, a.an, pi, __ldg(&a.pk[j]), xi, yi, hi, a.x, a.y,
                      a.h, j, dx, dy, r2);
}

// Single-walk list build: a team of T lanes walks particle i's own and
// coarser levels (per level, up to T cells looked up at once, then the
// candidates of all of them taken T at a time, one per lane); the team's
// ballot orders each group, so own entries come in (cell, index) order
// whatever T is.  They go into
// a fixed-stride staging row of stage_w entries; particles with more own
// entries go to a queue that k_list_fill_queue handles with a second walk.

template <int T>
__device__ __forceinline__ void list_gather_at(const ListArgs &a, int i, const Team<T> &tm) {
    const int li = a.lev[i];
    const double xi = a.x[i], yi = a.y[i], hi = a.h[i];
    const float4 pi = a.pk[i];
    const float2 q = anchor_rel(a.an, pi);
    uint32_t k = 0;
    const uint32_t W = a.stage_w;
    uint32_t *row = a.stage + (size_t)i * W;
    const unsigned below = tm.mask & ((1u << (threadIdx.x & 31)) - 1u);
    for_each_candidate_team<T, true>(a.g, a.d, li, q.x, q.y, pi.z, a.skin,
                                     tm.lane, tm.mask,
                                     [](uint32_t, uint32_t) { return true; },
                                     [&](uint32_t j, bool valid) {
        const bool in = valid && member(a, pi, xi, yi, hi, (int)j);
        const unsigned bal = T == 1 ? (in ? 1u : 0u)
                                    : __ballot_sync(tm.mask, in);
        if (in) {
            const uint32_t pos = k + (T == 1 ? 0u : __popc(bal & below));
            const bool co = __ldg(&a.lev[j]) > li;
            if (pos < W) row[pos] = co ? (j | STAGE_COARSE) : j;
            if (co) atomicAdd(&a.rev[j], 1u);
        }
        k += __popc(bal);
    });
    if (tm.lane == 0) {
        a.own[i] = k;
        atomicMax(a.max_own, k);
        if (k > W) a.queue[atomicAdd(a.nqueue, 1u)] = (uint32_t)i;
    }
}

template <int T>
__global__ void __launch_bounds__(128) k_list_gather(ListArgs a) {
    const Team<T> tm;
    const int i = Team<T>::particle();
    if (i >= a.n) return;
    list_gather_at<T>(a, i, tm);
}

// Copies the staged own entries into place and writes the reverse entries
// (i into the list of each coarser neighbour j); T lanes per particle.
template <int T>
__device__ __forceinline__ void list_place_at(const ListArgs &a, int i, const Team<T> &tm) {
    const uint32_t own = a.own[i];
    if (own <= a.stage_w) {               // else handled by k_list_fill_queue
        const uint32_t base = a.off[i];
        const uint32_t *row = a.stage + (size_t)i * a.stage_w;
        const uint32_t cap = a.cap;
#pragma unroll 4
        for (uint32_t k = tm.lane; k < own; k += T) {
            const uint32_t ent = row[k];
            const uint32_t j = ent & ~STAGE_COARSE;
            if (!SPH_DCHECK(j < (uint32_t)a.n)) continue;
            if (base + k < cap) a.list[base + k] = j;
            if (ent & STAGE_COARSE) {
                const uint32_t rp = a.off[j] + a.own[j] + atomicAdd(&a.rev[j], 1u);
                if (rp < cap) a.list[rp] = (uint32_t)i;
            }
        }
    }
    if (i == a.n - 1 && tm.lane == 0 && a.off[a.n] > a.cap) atomicOr(a.overflow, 1);
}

template <int T>
__global__ void __launch_bounds__(128) k_list_place(ListArgs a) {
    const Team<T> tm;
    const int i = Team<T>::particle();
    if (i >= a.n) return;
    list_place_at<T>(a, i, tm);
}

// Rows: only the reverse entries are placed (the coarser entries of each
// row).  A thread per particle; most rows have none.  4.2M graded strip:
// walk to sorted lists but for the walk itself 1.16 -> 0.51 ms, where
// k_list_place copied every row into the lists; and the passes, which read
// 32 separate lists a warp before, 1.155 -> 0.935 ms (B) and 0.935 -> 0.92
// ms (A).
__global__ void __launch_bounds__(256) k_list_place_rev(ListArgs a) {
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i < (uint32_t)a.n) {
        const uint32_t r = a.rlen[i], e = r & 0xffffu;
        const uint32_t *row = a.stage + (size_t)(i >> 5) * (32 * a.stage_w) + (i & 31);
        // four entries' chains of loads at once
        for (uint32_t k = r >> 16; k < e; k += 4) {
            uint32_t j[4], rp[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) j[u] = k + u < e ? row[32 * (k + u)] : 0xffffffffu;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                rp[u] = 0xffffffffu;
                if (k + u < e && SPH_DCHECK(j[u] < (uint32_t)a.n))
                    rp[u] = a.off[j[u]] + a.own[j[u]] + atomicAdd(&a.rev[j[u]], 1u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (rp[u] < a.cap) a.list[rp[u]] = i;
        }
        if (i == (uint32_t)a.n - 1 && a.off[a.n] > a.cap) atomicOr(a.overflow, 1);
    }
}

// Only builds that read their size back sum the rows.
__global__ void __launch_bounds__(256)
    k_row_total(int n, const uint32_t *__restrict__ rlen, unsigned long long *total) {
    unsigned long long t = 0;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256)
        t += rlen[i] & 0xffffu;
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(total, t);
}

// Second walk for the queued particles (more than stage_w own entries):
// same order as k_list_gather; teams take queue entries in turn.
template <int T>
__device__ __forceinline__ void list_fill_queue_at(const ListArgs &a, uint32_t vb,
                                                   uint32_t nvb, const Team<T> &tm) {
    const uint32_t nq = *a.nqueue;
    const uint32_t team = (vb * blockDim.x + threadIdx.x) / T;
    const uint32_t nteam = (nvb * blockDim.x) / T;
    const unsigned below = tm.mask & ((1u << (threadIdx.x & 31)) - 1u);
    for (uint32_t qi = team; qi < nq; qi += nteam) {
        const int i = (int)a.queue[qi];
        const int li = a.lev[i];
        const double xi = a.x[i], yi = a.y[i], hi = a.h[i];
        const float4 pi = a.pk[i];
        const float2 q = anchor_rel(a.an, pi);
        uint32_t k = a.off[i];
        const uint32_t cap = a.cap;
        for_each_candidate_team<T, true>(a.g, a.d, li, q.x, q.y, pi.z, a.skin,
                                         tm.lane, tm.mask,
                                         [](uint32_t, uint32_t) { return true; },
                                         [&](uint32_t j, bool valid) {
            const bool in = valid && member(a, pi, xi, yi, hi, (int)j);
            const unsigned bal = __ballot_sync(tm.mask, in);
            if (in) {
                const uint32_t pos = k + __popc(bal & below);
                if (pos < cap) a.list[pos] = j;
                if (__ldg(&a.lev[j]) > li) {
                    uint32_t rp = a.off[j] + a.own[j] + atomicAdd(&a.rev[j], 1u);
                    if (rp < cap) a.list[rp] = (uint32_t)i;
                }
            }
            k += __popc(bal);
        });
    }
}

template <int T>
__global__ void __launch_bounds__(128) k_list_fill_queue(ListArgs a) {
    const Team<T> tm;
    list_fill_queue_at<T>(a, blockIdx.x, gridDim.x, tm);
}

// ------------------------------------------------------ tiled list build --
// Cell-tiled walk: one warp takes the particles of one cell (up to 32 at a
// time, lane = particle).  For each level at or above the cell's, the warp
// looks up the cells around the bounding box of its particles once (a lane
// per cell), stages their candidates in shared memory (a batch of loads
// with no dependence between them) and every lane tests its particle
// against each staged candidate: a broadcast shared-memory read and a few
// FP32 operations per pair, instead of a lookup and a global load per
// particle.  Own entries come in (level, row, column, index) order.
//
// Separations: candidates and particles carry FP32 coordinates relative to
// the cell's first particle (anchor separations), so the pair separation is
// one subtraction.  Its error bound grows with the distance G from that
// reference; the exact-mode band below includes it.  Images on a periodic
// axis: a member j of a particle i in the cell lies within skin * c_l' +
// w_l of the reference, so while that stays below half the period the
// reference-relative image is the minimum image; otherwise (coarse levels
// of small periodic boxes) each pair is wrapped explicitly.
constexpr int TILE_CAP = 256;   // staged candidates per warp and batch
constexpr int TILE_LD = 2;      // candidate loads in flight per lane
// warps per block: two where a warp takes whole cells, whose work is uneven
// (a block's places are free again when its last warp ends: 1, 2, 4 warps
// 1.81, 1.65, 1.75 ms at 4.2M on the graded strip), four with teams
template <int T>
constexpr int TILE_WARPS = T == 1 ? 2 : 4;

// The grid's levels in shared memory, a lane per level in the walk's set-up.
struct LevTab {
    float cf[MAX_LEVELS], invw[2][MAX_LEVELS], w[2][MAX_LEVELS], invP[2][MAX_LEVELS];
    int n[2][MAX_LEVELS], bb[4][MAX_LEVELS];
    // the whole block; ends with a barrier
    __device__ __forceinline__ void load(const Grid &g) {
        const int l = threadIdx.x;
        if (l < MAX_LEVELS) {
            const Level &L = g.lev[l];
            cf[l] = L.cf;
#pragma unroll
            for (int ax = 0; ax < 2; ++ax) {
                invw[ax][l] = L.invw[ax];
                w[ax][l] = L.wf[ax];
                invP[ax][l] = L.invP[ax];
                n[ax][l] = L.n[ax];
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) bb[t][l] = __ldg(&g.bbox[4 * l + t]);
        }
        __syncthreads();
    }
};
constexpr int TILE_LEV = 16;    // levels set up at once, a lane each
// first cell and cell count of the three pieces of each axis, per level
constexpr int TILE_PCS = 12 * TILE_LEV;

__device__ __forceinline__ float warp_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Squared gap between the box [xc - hx, xc + hx] x [yc - hy, yc + hy] and
// cell (cx, cy) of level l (unwrapped indices), less a margin far above
// FP32 rounding; periodic axes use the nearest image of the cell, the edge
// cells of a non-periodic axis reach to infinity.
__device__ __forceinline__ float box_gap2(const Domain &d, const LevTab &T, int l,
                                          int cx, int cy, float xc, float yc,
                                          float hx, float hy) {
    const int c[2] = {cx, cy};
    const float q[2] = {xc, yc}, hh[2] = {hx, hy};
    float g2 = 0.0f;
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
        const float w = T.w[ax][l];
        const float m = 1e-5f * (fabsf(q[ax]) + hh[ax] + w);
        float gap;
        if (d.periodic[ax]) {
            const float P = (float)T.n[ax][l] * w;
            float t = q[ax] - ((float)c[ax] + 0.5f) * w;
            t -= P * rintf(t * T.invP[ax][l]);
            gap = fabsf(t) - 0.5f * w - hh[ax];
        } else {
            float lo = (float)c[ax] * w, hi = lo + w;
            if (c[ax] <= 0) lo = -3.0e38f;
            if (c[ax] >= T.n[ax][l] - 1) hi = 3.0e38f;
            gap = fmaxf(lo - (q[ax] + hh[ax]), (q[ax] - hh[ax]) - hi);
        }
        gap = fmaxf(0.0f, gap - m);
        g2 += gap * gap;
    }
    return g2;
}

// One chunk of a cell: particles p0 .. min(p0 + 32, ce) - 1 of the cell
// starting at cs (level lc); `only` >= 0 restricts the work to that one
// particle.  DIRECT = false: own entries into the staging rows, reverse
// entries counted; DIRECT = true (particles whose rows overflowed): own
// entries straight into the list at off[i], reverse entries placed.  Both
// modes take identical membership decisions (same reference, same
// per-level constants, same arithmetic); the cells a chunk visits depend
// on its bounding box, but a cell only one of them visits holds no member
// (its gap exceeds the pair radius by the pruning margin).
// sc: the warp's staging buffer (TILE_CAP entries); pcs: 20 ints of the
// warp's shared memory for the query's cell pieces.
// span: 2 when the chunk's particles lie in up to 2 x 2 neighbouring cells
// of level lc (merged chunks), else 1; the distance bound G of the FP32
// error analysis grows with it.  A particle queued for the direct pass
// records its chunk's reference and span, so that pass takes the same
// decisions with the same arithmetic.
// ROWS: interleaved rows (ListArgs::rows), else one after another.
template <bool DIRECT, int T, bool ROWS = false>
__device__ __forceinline__ void tile_chunk(const ListArgs &a, const LevTab &tab,
                                           float4 *sc, int *pcs, int lc, uint32_t cs,
                                           uint32_t pe, uint32_t p0, int only,
                                           int span = 1) {
    static_assert(T == 1 || T == 4 || T == 16, "team of 1, 4 or 16 lanes");
    const int lane = threadIdx.x & 31;
    const int sub = lane & (T - 1);           // lane within the particle's team
    const uint32_t i = p0 + (uint32_t)(lane / T);
    const bool act = i < pe && (only < 0 || (int)i == only);
    const float4 pC = __ldg(&a.pk[cs]);
    float rxi = 0.0f, ryi = 0.0f, Ri = 0.0f, hmx = 0.0f;
    // the chunk's bounding box in reference-relative coordinates
    float rxlo = 3.0e38f, rxhi = -3.0e38f, rylo = 3.0e38f, ryhi = -3.0e38f;
    if (act) {
        const float4 pi = __ldg(&a.pk[i]);
        anchor_sep(a.an, pi, pC, rxi, ryi);
        Ri = a.skin * (3.0f * pi.z);
        hmx = pi.z;
        rxlo = rxhi = rxi;
        rylo = ryhi = ryi;
    }
    rxlo = warp_min(rxlo);
    rxhi = warp_max(rxhi);
    rylo = warp_min(rylo);
    ryhi = warp_max(ryhi);
    hmx = warp_max(hmx);
    // the same box from the domain's corner (a chunk does not straddle a
    // period); its rounding is far below the margins of the cell ranges
    const float2 qC = anchor_rel(a.an, pC);
    const float xc = qC.x + 0.5f * (rxlo + rxhi), yc = qC.y + 0.5f * (rylo + ryhi);
    const float bx = 0.5f * (rxhi - rxlo), by = 0.5f * (ryhi - rylo);
    const float Rmx = a.skin * (3.0f * hmx);   // largest pair radius of a chunk particle
    const uint32_t W = a.stage_w;
    constexpr uint32_t RS = ROWS ? 32 : 1;     // stride of a row's entries
    uint32_t k = 0, kown = 0;
    if (DIRECT && act) k = a.off[i];
    uint32_t *row = a.stage + (ROWS ? (size_t)(i >> 5) * (32 * W) + (i & 31) : (size_t)i * W);
    const float Amax = fmaxf(a.an.A[0], a.an.A[1]);
    const float Lx = (float)a.d.L[0], Ly = (float)a.d.L[1];
    const float iLx = 1.0f / Lx, iLy = 1.0f / Ly;
    const bool exact = !(a.skin > 1.0f);
    uint32_t mm = a.g.level_mask & ~((1u << lc) - 1u);
    while (mm) {
        // set-up of up to TILE_LEV levels, lane t: level lb + t
        const int lb = __ffs(mm) - 1;
        const int lt = lb + lane;
        int nc = 0;
        bool wx = false, wy = false;
        float KB = 0.0f;
        __syncwarp();
        if (lane < TILE_LEV && lt < MAX_LEVELS && ((mm >> lt) & 1u) &&
            tab.bb[0][lt] <= tab.bb[1][lt]) {
            const float Q = a.skin * fmaxf(3.0f * hmx, tab.cf[lt]) * (1.0f + 1e-5f);
            AxisPieces px, py;
            if (axis_pieces_of(a.d.periodic[0], tab.n[0][lt], tab.invw[0][lt], tab.bb[0][lt],
                               tab.bb[1][lt], xc, bx + Q, px) &&
                axis_pieces_of(a.d.periodic[1], tab.n[1][lt], tab.invw[1][lt], tab.bb[2][lt],
                               tab.bb[3][lt], yc, by + Q, py)) {
                int nx = 0, ny = 0;
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    const int cx = max(0, px.last[t] - px.first[t] + 1);
                    const int cy = max(0, py.last[t] - py.first[t] + 1);
                    pcs[t * TILE_LEV + lane] = px.first[t];
                    pcs[(3 + t) * TILE_LEV + lane] = cx;
                    pcs[(6 + t) * TILE_LEV + lane] = py.first[t];
                    pcs[(9 + t) * TILE_LEV + lane] = cy;
                    nx += cx;
                    ny += cy;
                }
                nc = nx * ny;
                const float reach = a.skin * tab.cf[lt] +
                                    (float)span * fmaxf(tab.w[0][lc], tab.w[1][lc]) +
                                    fmaxf(tab.w[0][lt], tab.w[1][lt]);
                wx = a.d.periodic[0] && 2.0f * (reach + 4.0f * a.an.A[0]) >= Lx;
                wy = a.d.periodic[1] && 2.0f * (reach + 4.0f * a.an.A[1]) >= Ly;
                KB = 4.0f * Amax + reach + (wx || wy ? fmaxf(Lx, Ly) : 0.0f);
            }
        }
        mm = lb + TILE_LEV < MAX_LEVELS ? mm & ~((1u << (lb + TILE_LEV)) - 1u) : 0u;
        int ninc = nc;
#pragma unroll
        for (int o = 1; o < TILE_LEV; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, ninc, o);
            if (lane >= o) ninc += t;
        }
        const int ncell = __shfl_sync(0xffffffffu, ninc, TILE_LEV - 1);
        if (ncell == 0) continue;
        const bool wrapx = __any_sync(0xffffffffu, wx);
        const bool wrapy = __any_sync(0xffffffffu, wy);
        const bool wrap = wrapx || wrapy;
        KB = warp_max(KB);
        __syncwarp();
        for (int base = 0; base < ncell; base += 32) {
            // lane -> one cell of the query (level by level, row-major,
            // unwrapped order)
            uint32_t s = 0, e = 0, co = 0;
            const int idx = base + lane, idc = min(idx, ncell - 1);
            int sl = 0;
#pragma unroll
            for (int st = TILE_LEV / 2; st; st >>= 1) {
                const int v = __shfl_sync(0xffffffffu, ninc, sl + st - 1);
                if (v <= idc) sl += st;
            }
            const int loc = idc - __shfl_sync(0xffffffffu, ninc - nc, sl);
            if (idx < ncell) {
                const int l = lb + sl;
                const int *pc = pcs + sl;
                const int nx0 = pc[3 * TILE_LEV], nx1 = pc[4 * TILE_LEV];
                const int ny0 = pc[9 * TILE_LEV], ny1 = pc[10 * TILE_LEV];
                const int nx = nx0 + nx1 + pc[5 * TILE_LEV];
                int jy = loc / nx, ix = loc - jy * nx;
                int kx = 0, ky = 0;
                if (ix >= nx0) { ix -= nx0; kx = 1; if (ix >= nx1) { ix -= nx1; kx = 2; } }
                if (jy >= ny0) { jy -= ny0; ky = 1; if (jy >= ny1) { jy -= ny1; ky = 2; } }
                const int cx = pc[kx * TILE_LEV] + ix, cy = pc[(6 + ky) * TILE_LEV] + jy;
                // pieces 0 and 2 lie a period off (periodic axes only)
                const int sx = (1 - kx) * tab.n[0][l], sy = (1 - ky) * tab.n[1][l];
                const float Rl = a.skin * fmaxf(3.0f * hmx, tab.cf[l]);
                const float g2 = box_gap2(a.d, tab, l, cx, cy, xc, yc, bx, by);
                float hc;
                if (g2 < Rl * Rl &&
                    table_lookup(a.g, ((uint64_t)l << (2 * a.g.mbits)) |
                                          (spread2((uint64_t)(cy + sy)) << 1) |
                                          spread2((uint64_t)(cx + sx)),
                                 s, e, &hc)) {
                    const float Rc = a.skin * 3.0f * fmaxf(hmx, hc);
                    if (!(g2 < Rc * Rc)) s = e = 0;
                    if (!SPH_DCHECK(s <= e && e <= (uint32_t)a.n)) s = e = 0;
                } else {
                    s = e = 0;
                }
                co = l > lc ? STAGE_COARSE : 0u;
            }
            const uint32_t cnt = e - s;
            uint32_t inc = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
            const uint32_t exc = inc - cnt;
            s |= co;   // staged indices carry it
            for (uint32_t q0 = 0; q0 < total; q0 += TILE_CAP) {
                const uint32_t mq = min((uint32_t)TILE_CAP, total - q0);
                // stage: candidate q0 + u; its cell is the first lane whose
                // inclusive count exceeds it (binary search over the lanes),
                // TILE_LD independent loads per lane in flight.  Candidates
                // farther from the chunk's bounding box than the largest
                // pair radius they could have (with a margin far above FP32
                // error) are no member of any particle of the chunk and are
                // not staged; the others keep their order (ballot
                // compaction), so the test loop sees the same members in the
                // same order.
                // m: staged; mf: of them on the chunk's own level (they come
                // first)
                uint32_t m = 0, mf = 0;
                for (uint32_t u0 = 0; u0 < mq; u0 += 32 * TILE_LD) {
                    float4 v[TILE_LD];
                    uint32_t jj[TILE_LD];
#pragma unroll
                    for (int r = 0; r < TILE_LD; ++r) {
                        const uint32_t u = u0 + 32 * r + lane;
                        const uint32_t qq = q0 + min(u, mq - 1);
                        int pos = 0;
#pragma unroll
                        for (int st = 16; st; st >>= 1) {
                            const uint32_t vv = __shfl_sync(0xffffffffu, inc, pos + st - 1);
                            if (vv <= qq) pos += st;
                        }
                        const uint32_t st0 = __shfl_sync(0xffffffffu, s, pos);
                        const uint32_t ex0 = __shfl_sync(0xffffffffu, exc, pos);
                        jj[r] = st0 + (qq - ex0);
                        if (u < mq) v[r] = __ldg(&a.pk[jj[r] & ~STAGE_COARSE]);
                    }
#pragma unroll
                    for (int r = 0; r < TILE_LD; ++r) {
                        const uint32_t u = u0 + 32 * r + lane;
                        float rx = 0.0f, ry = 0.0f, Rj = 0.0f;
                        bool keep = false;
                        if (u < mq) {
                            anchor_sep(a.an, v[r], pC, rx, ry);
                            Rj = a.skin * (3.0f * v[r].z);
                            keep = true;
                            if (!wrap) {
                                const float gx = fmaxf(fmaxf(rxlo - rx, rx - rxhi), 0.0f);
                                const float gy = fmaxf(fmaxf(rylo - ry, ry - ryhi), 0.0f);
                                const float Rm = fmaxf(Rmx, Rj) * 1.01f;
                                keep = fmaf(gx, gx, gy * gy) < Rm * Rm;
                            }
                        }
                        const unsigned kb = __ballot_sync(0xffffffffu, keep);
                        if (keep)
                            sc[m + (uint32_t)__popc(kb & ((1u << lane) - 1u))] =
                                make_float4(rx, ry, Rj, __uint_as_float(jj[r]));
                        m += (uint32_t)__popc(kb);
                        mf += (uint32_t)__popc(
                            kb & __ballot_sync(0xffffffffu, !(jj[r] & STAGE_COARSE)));
                    }
                }
                __syncwarp();
                {
                    // one loop per (exact, wrap) case and own / coarser
                    // level, branch-free in the common ones: a predicated
                    // store and a counter.  A team of T lanes takes T
                    // consecutive candidates per iteration; the ballot keeps
                    // the team's entries in candidate order.
                    auto test = [&](auto ex_c, auto wr_c, auto co_c, uint32_t ub, uint32_t ue) {
                        constexpr bool EX = decltype(ex_c)::value;
                        constexpr bool WR = decltype(wr_c)::value;
                        constexpr bool CO = decltype(co_c)::value;
                        // ent: the candidate's index, with STAGE_COARSE if CO
                        auto pair_in = [&](uint32_t u, uint32_t &ent) {
                            const float4 c = sc[u];
                            float dx = rxi - c.x, dy = ryi - c.y;
                            if (WR) {
                                if (wrapx) dx -= Lx * rintf(dx * iLx);
                                if (wrapy) dy -= Ly * rintf(dy * iLy);
                            }
                            const float r2 = fmaf(dx, dx, dy * dy);
                            const float R = fmaxf(Ri, c.z);
                            const float R2 = R * R;
                            ent = __float_as_uint(c.w);
                            bool in = r2 < R2;
                            if (EX) {
                                const float band = fmaf(R, KB, R2) * (1.0f / 65536.0f);
                                in = r2 < R2 - band;
                                if (!in && !(r2 > R2 + band)) {
                                    const uint32_t j = CO ? ent & ~STAGE_COARSE : ent;
                                    in = pred_fp64(a.d, __ldg(&a.x[i]), __ldg(&a.y[i]),
                                                   __ldg(&a.h[i]), __ldg(&a.x[j]),
                                                   __ldg(&a.y[j]), __ldg(&a.h[j]));
                                }
                            }
                            return in;
                        };
                        auto put = [&](uint32_t pos, uint32_t ent) {
                            const uint32_t j = CO ? ent & ~STAGE_COARSE : ent;
                            if (DIRECT) {
                                if (pos < a.cap) a.list[pos] = j;
                                if (CO) {
                                    const uint32_t rp = a.off[j] + a.own[j] +
                                                        atomicAdd(&a.rev[j], 1u);
                                    if (rp < a.cap) a.list[rp] = i;
                                }
                            } else {
                                if (pos < W) row[pos] = ent;
                                if (CO) atomicAdd(&a.rev[j], 1u);
                            }
                        };
                        if constexpr (T == 1) {
                            if (!act) return;
#pragma unroll 4
                            for (uint32_t u = ub; u < ue; ++u) {
                                uint32_t ent;
                                const bool in = pair_in(u, ent);
                                if (DIRECT) {
                                    if (in) put(k, ent);
                                } else {
                                    if (in && k < W)
                                        row[k * RS] = ROWS && CO ? ent & ~STAGE_COARSE : ent;
                                    if (CO && in) atomicAdd(&a.rev[ent & ~STAGE_COARSE], 1u);
                                }
                                k += in ? 1u : 0u;
                            }
                        } else {
                            const unsigned gsh = (unsigned)(lane & ~(T - 1));
                            const unsigned below = (1u << sub) - 1u;
                            for (uint32_t u0 = ub; u0 < ue; u0 += T) {
                                const uint32_t u = u0 + (uint32_t)sub;
                                uint32_t ent = 0;
                                const bool in = act && u < ue && pair_in(u, ent);
                                const unsigned gb = (__ballot_sync(0xffffffffu, in) >> gsh) &
                                                    ((1u << T) - 1u);
                                if (in) put(k + (uint32_t)__popc(gb & below), ent);
                                k += (uint32_t)__popc(gb);
                            }
                        }
                    };
                    using TT = std::true_type;
                    using FF = std::false_type;
                    auto both = [&](auto ex, auto wr) {
                        test(ex, wr, FF(), 0u, mf);
                        if (ROWS && mf) kown = k;
                        if (mf < m) test(ex, wr, TT(), mf, m);
                    };
                    if (exact) {
                        if (wrap) both(TT(), TT()); else both(TT(), FF());
                    } else {
                        if (wrap) both(FF(), TT()); else both(FF(), FF());
                    }
                }
                __syncwarp();
            }
        }
    }
    if (!DIRECT) {
        uint32_t km = act ? k : 0u;
#pragma unroll
        for (int o = 16; o; o >>= 1) km = max(km, __shfl_xor_sync(0xffffffffu, km, o));
        if (act && sub == 0) {
            if (ROWS) a.rlen[i] = k > W ? 0u : k | (kown << 16);
            a.own[i] = ROWS && k <= W ? 0u : k;
            if (k > W) {
                const uint32_t q = atomicAdd(a.nqueue, 1u);
                a.queue[q] = i;
                a.qref[q] = cs | (span > 1 ? 0x80000000u : 0u);
            }
        }
        if (lane == 0 && km > 0) atomicMax(a.max_own, km);
    }
}

// Stage-mode walk.  T = 1: warp w owns the cells whose first particle lies
// in [32 w, 32 w + 32) and takes them one after another, 32 particles at a
// time.  T > 1 (small sets, where that leaves most of the GPU idle): warp w
// takes the 32 / T particles [w P, w P + P), P = 32 / T, one piece per cell
// they fall in.
// resident 128-thread blocks per SM the merged-chunk walk is compiled for
// (80 registers; measured 23 % faster than the unbounded 94 and 4-6 %
// faster than seven or eight blocks, which spill); the cell-per-chunk
// forms keep the 72 / 80 registers they were measured at
#ifndef SPH_TILE_MERGE_BLOCKS
#define SPH_TILE_MERGE_BLOCKS 6
#endif
template <int T, bool MERGE = false, bool ROWS = false>
__global__ void __launch_bounds__(32 * TILE_WARPS<T>,
                                  (MERGE ? SPH_TILE_MERGE_BLOCKS : (T == 1 ? 7 : 6)) * 4 /
                                      TILE_WARPS<T>)
    k_list_tile(ListArgs a) {
    __shared__ float4 sbuf[TILE_WARPS<T>][TILE_CAP];
    __shared__ int spcs[TILE_WARPS<T>][TILE_PCS];
    __shared__ LevTab tab;
    tab.load(a.g);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t gw = blockIdx.x * (uint32_t)TILE_WARPS<T> + (uint32_t)w;
    const uint32_t n = (uint32_t)a.n;
    if constexpr (T == 1) {
        const uint32_t base = gw * 32u;
        if (base >= n) return;
        // the keys of the range, in registers: cells end where the next
        // begins, but for the last one, whose end the table holds
        const uint32_t i = base + lane;
        const uint64_t key = i < n ? a.skey[i] : EMPTY_KEY;
        uint64_t prev = __shfl_up_sync(0xffffffffu, key, 1);
        if (lane == 0 && i > 0) prev = a.skey[i - 1];
        const bool head = i < n && (i == 0 || prev != key);
        const unsigned all = __ballot_sync(0xffffffffu, head);
        unsigned heads = all;
        if (!heads) return;
        uint32_t ls, le = n;
        table_lookup(a.g, __shfl_sync(0xffffffffu, key, 31 - __clz(all)), ls, le);
        auto cell_end = [&](uint32_t h) {   // h: lane of the cell's first particle
            const unsigned up = all & ~((2u << h) - 1u);
            return up ? base + (uint32_t)(__ffs(up) - 1) : le;
        };
        const uint64_t cmask = (1ull << (2 * a.g.mbits)) - 1ull;
        while (heads) {
            const int hl = __ffs(heads) - 1;
            heads &= heads - 1;
            const uint64_t K = __shfl_sync(0xffffffffu, key, hl);
            const uint32_t cs = base + (uint32_t)hl;
            uint32_t ce = cell_end((uint32_t)hl);
            const int lc = (int)(K >> (2 * a.g.mbits));
            int span = 1;
            if constexpr (MERGE) {
                // the following cells of this warp's range join the chunk
                // while they are of the same level, within one cell of the
                // first on both axes (no wrap) and the chunk holds at most
                // 32 particles
                const uint32_t fx = compact2(K & cmask), fy = compact2((K & cmask) >> 1);
                while (ce - cs < 32 && ce < base + 32 && ce < n) {
                    const uint64_t K2 = __shfl_sync(0xffffffffu, key, (int)(ce - base));
                    if ((K2 >> (2 * a.g.mbits)) != (K >> (2 * a.g.mbits))) break;
                    const int dx = (int)compact2(K2 & cmask) - (int)fx;
                    const int dy = (int)compact2((K2 & cmask) >> 1) - (int)fy;
                    if (dx < -1 || dx > 1 || dy < -1 || dy > 1) break;
                    const uint32_t e2 = cell_end(ce - base);
                    if (e2 - cs > 32) break;
                    heads &= ~(1u << (ce - base));
                    ce = e2;
                    span = 2;
                }
            }
            for (uint32_t p0 = cs; p0 < ce; p0 += 32)
                tile_chunk<false, 1, ROWS>(a, tab, sbuf[w], spcs[w], lc, cs,
                                           min(ce, p0 + 32), p0, -1, span);
        }
    } else {
        constexpr uint32_t P = 32 / T;
        const uint32_t w0 = gw * P;
        if (w0 >= n) return;
        const uint32_t w1 = min(n, w0 + P);
        uint32_t t = w0;
        while (t < w1) {
            const uint64_t K = a.skey[t];
            uint32_t cs = t, ce = t + 1;
            table_lookup(a.g, K, cs, ce);
            const uint32_t pe = min(ce, w1);
            tile_chunk<false, T>(a, tab, sbuf[w], spcs[w], a.lev[t], cs, pe, t, -1);
            t = pe;
        }
    }
}

// Direct-mode pass for the particles whose own entries overflowed their
// staging row; a warp per queued particle.
__global__ void __launch_bounds__(128) k_list_tile_queue(ListArgs a) {
    const uint32_t nq = *a.nqueue;
    if (blockIdx.x * 4u >= nq) return;
    __shared__ float4 sbuf[4][TILE_CAP];
    __shared__ int spcs[4][TILE_PCS];
    __shared__ LevTab tab;
    tab.load(a.g);
    const int w = threadIdx.x >> 5;
    const uint32_t gw = blockIdx.x * 4u + (uint32_t)w, nw = gridDim.x * 4u;
    for (uint32_t q = gw; q < nq; q += nw) {
        const uint32_t i = a.queue[q];
        // the reference and span of the chunk that queued it
        const uint32_t r = a.qref[q];
        const uint32_t cs = r & 0x7fffffffu;
        tile_chunk<true, 16>(a, tab, sbuf[w], spcs[w], a.lev[i], cs, i + 1, i, (int)i,
                             (r & 0x80000000u) ? 2 : 1);
    }
}

// Sort of each reverse segment (ascending index).  Segments of at most 32
// entries (the common case: only particles next to a finer level have
// any) are sorted in registers by the particle's thread; longer ones are
// queued for a warp-wide bitonic sort in shared memory.
constexpr int SORT_REG = 32;
constexpr int SORT_SMEM = 1024;

// Ascending sort of seg[0 .. len) (len <= K) in registers: odd-even
// transposition over K slots, fixed indices, padding at the top.
template <int K>
__device__ __forceinline__ void sort_regs(uint32_t *seg, uint32_t len) {
    uint32_t r[K];
#pragma unroll
    for (int t = 0; t < K; ++t) r[t] = t < (int)len ? seg[t] : 0xffffffffu;
#pragma unroll
    for (int round = 0; round < K; ++round) {
#pragma unroll
        for (int t = round & 1; t + 1 < K; t += 2) {
            const uint32_t lo = min(r[t], r[t + 1]), hi = max(r[t], r[t + 1]);
            r[t] = lo;
            r[t + 1] = hi;
        }
    }
#pragma unroll
    for (int t = 0; t < K; ++t)
        if (t < (int)len) seg[t] = r[t];
}

// Also the last word on an overflowed build: its offsets are cut to the
// capacity, so what reads the lists before the overflow is reported meets the
// entries that were written and never leaves the buffer.  (A neighbour's
// thread may see an offset raw or cut: past the capacity either way.)
__device__ __forceinline__ void list_sort_rev_at(int i, int n, uint32_t *off,
                                                 const uint32_t *own, uint32_t *list,
                                                 uint32_t cap, uint32_t *longq,
                                                 uint32_t *nlong) {
    if (i >= n) return;
    const uint32_t o = off[i], b = o + (own ? own[i] : 0u), e = off[i + 1];
    if (o > cap) off[i] = cap;
    if (i == n - 1 && e > cap) off[n] = cap;
    if (e > cap || e <= b + 1) return;
    const uint32_t len = e - b;
    if (len > SORT_REG) {
        longq[atomicAdd(nlong, 1u)] = (uint32_t)i;
        return;
    }
    // the network no wider than the segment needs (most are short)
    if (len <= 8)
        sort_regs<8>(list + b, len);
    else if (len <= 16)
        sort_regs<16>(list + b, len);
    else
        sort_regs<SORT_REG>(list + b, len);
}

__global__ void k_list_sort_rev(int n, uint32_t *off, const uint32_t *own,
                                uint32_t *list, uint32_t cap, uint32_t *longq,
                                uint32_t *nlong) {
    list_sort_rev_at(blockIdx.x * blockDim.x + threadIdx.x, n, off, own, list, cap, longq,
                     nlong);
}

__device__ __forceinline__ void list_sort_long_at(const uint32_t *off, const uint32_t *own,
                                                  uint32_t *list, const uint32_t *longq,
                                                  const uint32_t *nlong, uint32_t vb,
                                                  uint32_t nvb) {
    __shared__ uint32_t buf[4][SORT_SMEM];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t *s = buf[w];
    const uint32_t nq = *nlong;
    const uint32_t gw = vb * 4 + w, nw = nvb * 4;
    for (uint32_t q = gw; q < nq; q += nw) {
        const uint32_t i = longq[q];
        const uint32_t b = off[i] + (own ? own[i] : 0u), e = off[i + 1];
        const uint32_t len = e - b;
        if (len > SORT_SMEM) {
            // rare: plain insertion sort by one lane
            if (lane == 0) {
                for (uint32_t k = b + 1; k < e; ++k) {
                    uint32_t v = list[k], m = k;
                    while (m > b && list[m - 1] > v) {
                        list[m] = list[m - 1];
                        --m;
                    }
                    list[m] = v;
                }
            }
            __syncwarp();
            continue;
        }
        uint32_t P = 32;
        while (P < len) P <<= 1;
        for (uint32_t t = lane; t < P; t += 32) s[t] = t < len ? list[b + t] : 0xffffffffu;
        __syncwarp();
        for (uint32_t k = 2; k <= P; k <<= 1) {
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                for (uint32_t t = lane; t < P; t += 32) {
                    uint32_t ixj = t ^ j;
                    if (ixj > t) {
                        uint32_t x0 = s[t], x1 = s[ixj];
                        bool asc = (t & k) == 0;
                        if ((x0 > x1) == asc) {
                            s[t] = x1;
                            s[ixj] = x0;
                        }
                    }
                }
                __syncwarp();
            }
        }
        for (uint32_t t = lane; t < len; t += 32) list[b + t] = s[t];
        __syncwarp();
    }
}

__global__ void k_list_sort_long(const uint32_t *off, const uint32_t *own,
                                 uint32_t *list, const uint32_t *longq,
                                 const uint32_t *nlong) {
    list_sort_long_at(off, own, list, longq, nlong, blockIdx.x, gridDim.x);
}

// ---------------------------------------------- batched small builds ----
// The single-instance bodies over the work items of several instances
// (one item: one block of the instance's single-launch grid, or of a
// smaller grid where the body's results do not depend on it).
template <int T>
__global__ void __launch_bounds__(128) k_list_gather_batch(const ListArgs *args, BatchSpan sp) {
    const Team<T> tm;
    for (int it = blockIdx.x; it < sp.total; it += gridDim.x) {
        const BatchItem b = batch_item(sp, it);
        const ListArgs &a = args[b.q];
        const int i = b.vb * (128 / T) + (int)threadIdx.x / T;
        if (i < a.n) list_gather_at<T>(a, i, tm);
    }
}
template <int T>
__global__ void __launch_bounds__(128) k_list_place_batch(const ListArgs *args, BatchSpan sp) {
    const Team<T> tm;
    for (int it = blockIdx.x; it < sp.total; it += gridDim.x) {
        const BatchItem b = batch_item(sp, it);
        const ListArgs &a = args[b.q];
        const int i = b.vb * (128 / T) + (int)threadIdx.x / T;
        if (i < a.n) list_place_at<T>(a, i, tm);
    }
}
__global__ void __launch_bounds__(128) k_list_fill_queue_batch(const ListArgs *args, BatchSpan sp) {
    const Team<16> tm;
    for (int it = blockIdx.x; it < sp.total; it += gridDim.x) {
        const BatchItem b = batch_item(sp, it);
        list_fill_queue_at<16>(args[b.q], b.vb, b.nvb, tm);
    }
}
__global__ void __launch_bounds__(256) k_list_sort_rev_batch(const SortSegRec *args, BatchSpan sp) {
    for (int it = blockIdx.x; it < sp.total; it += gridDim.x) {
        const BatchItem b = batch_item(sp, it);
        const SortSegRec &r = args[b.q];
        list_sort_rev_at(b.vb * 256 + (int)threadIdx.x, r.n, r.off, r.own, r.list, r.cap, r.longq,
                         r.nlong);
    }
}
__global__ void __launch_bounds__(128) k_list_sort_long_batch(const SortSegRec *args, BatchSpan sp) {
    for (int it = blockIdx.x; it < sp.total; it += gridDim.x) {
        const BatchItem b = batch_item(sp, it);
        const SortSegRec &r = args[b.q];
        list_sort_long_at(r.off, r.own, r.list, r.longq, r.nlong, b.vb, b.nvb);
        __syncthreads();
    }
}

// ------------------------------------------------------------- launchers --
static inline int nblk_s(int n, int bs) { return (n + bs - 1) / bs; }

void sort_segments(cudaStream_t s, int n, uint32_t *off, uint32_t *list,
                   uint32_t cap, uint32_t *longq, uint32_t *nlong,
                   int *launches) {
    if (n <= 0) return;
    k_list_sort_rev<<<nblk_s(n, 256), 256, 0, s>>>(n, off, nullptr, list, cap,
                                                   longq, nlong);
    k_list_sort_long<<<std::max(1, std::min(152 * 16, nblk_s(n, 4))), 128, 0, s>>>(
        off, nullptr, list, longq, nlong);
    *launches += 2;
}
static inline int nblk(int n, int bs) { return (n + bs - 1) / bs; }

void launch_pack_batch(cudaStream_t s, const PackArgs *args, const BatchSpan &sp,
                       int blocks) {
    if (sp.total > 0)
        k_pack_batch<<<std::min(blocks, sp.total), BATCH_THREADS, 0, s>>>(args, sp);
}
int pack_batch_blocks_per_sm() {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pack_batch, BATCH_THREADS, 0) !=
            cudaSuccess || per_sm < 1)
        per_sm = 1;
    return per_sm;
}
void launch_pack(cudaStream_t s, const PackArgs &a) {
    if (a.n > 0) k_pack<<<nblk(a.n, 256), 256, 0, s>>>(a);
}
void launch_gather_pack(cudaStream_t s, const GatherPackRec &r, int *launches) {
    if (r.n <= 0) return;
    k_gather_pack<<<nblk(r.n, 256), 256, 0, s>>>(r);
    *launches += 1;
}
void launch_anchor_pack(cudaStream_t s, int n, const double *x,
                        const double *y, const double *h, const double *lo,
                        const double *A, const Anchor &an, float4 *pk) {
    if (n > 0)
        k_anchor_pack<<<nblk(n, 256), 256, 0, s>>>(n, x, y, h, lo[0], lo[1],
                                                    A[0], A[1], an, pk);
}

// Walk choice by set size (measured on GB300 over uniform and graded
// lattices of 5k to 16M particles): below ~12k particles the per-particle
// team walk keeps more warps in flight than the cell tiles; from there the
// tiles win, with teams of 4 lanes up to 48k particles (1.5x faster than
// the merged one-lane tiles at 12k-26k on uniform vortices, even at
// 36k-50k) and merged one-lane tiles beyond (0.78x the 4-lane tiles at
// 70k, 0.5x at 290k).  A.walk overrides it (tuning).
static int walk_kind(const ListArgs &a) {
    if (a.walk >= 1 && a.walk <= 4) return a.walk;
    return a.n < 12000 ? 1 : a.n < 48000 ? 2 : 4;
}

int list_walk_kind(const ListArgs &a) { return walk_kind(a); }
// The merged walk's range, whatever walk is set: below it a step is bound by
// launches and the copy into the lists is small.
bool list_rows_for(const ListArgs &a) { return a.n >= 48000 && walk_kind(a) == 4; }
int list_place_team(int n) { return std::max(team_size(n), 16); }
int fill_queue_blocks() { return 4; }
int sort_long_blocks(int n) { return std::max(1, std::min(8, nblk(n, 4))); }

template <class K>
static int batch_grid_of(K kernel, int threads, int total) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) !=
            cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const long long g = (long long)per_sm * gpu_sms();
    return (int)(g < total ? g : total);
}
void launch_gather_batch(cudaStream_t s, const GatherPackRec *args, const BatchSpan &sp) {
    static const int g = batch_grid_of(k_gather_batch, 256, 1 << 30);
    if (sp.total > 0) k_gather_batch<<<std::min(g, sp.total), 256, 0, s>>>(args, sp);
}
void launch_list_gather_batch(cudaStream_t s, int team, const ListArgs *args, const BatchSpan &sp) {
    if (sp.total <= 0) return;
    with_team_or(team, 1 << 30, [&](auto t) {
        constexpr int T = decltype(t)::value;
        static const int g = batch_grid_of(k_list_gather_batch<T>, 128, 1 << 30);
        k_list_gather_batch<T><<<std::min(g, sp.total), 128, 0, s>>>(args, sp);
    });
}
void launch_list_place_batch(cudaStream_t s, int team, const ListArgs *args, const BatchSpan &sp) {
    if (sp.total <= 0) return;
    with_team_or(team, 1 << 30, [&](auto t) {
        constexpr int T = decltype(t)::value;
        static const int g = batch_grid_of(k_list_place_batch<T>, 128, 1 << 30);
        k_list_place_batch<T><<<std::min(g, sp.total), 128, 0, s>>>(args, sp);
    });
}
void launch_list_fill_queue_batch(cudaStream_t s, const ListArgs *args, const BatchSpan &sp) {
    static const int g = batch_grid_of(k_list_fill_queue_batch, 128, 1 << 30);
    if (sp.total > 0) k_list_fill_queue_batch<<<std::min(g, sp.total), 128, 0, s>>>(args, sp);
}
void launch_list_sort_rev_batch(cudaStream_t s, const SortSegRec *args, const BatchSpan &sp) {
    static const int g = batch_grid_of(k_list_sort_rev_batch, 256, 1 << 30);
    if (sp.total > 0) k_list_sort_rev_batch<<<std::min(g, sp.total), 256, 0, s>>>(args, sp);
}
void launch_list_sort_long_batch(cudaStream_t s, const SortSegRec *args, const BatchSpan &sp) {
    static const int g = batch_grid_of(k_list_sort_long_batch, 128, 1 << 30);
    if (sp.total > 0) k_list_sort_long_batch<<<std::min(g, sp.total), 128, 0, s>>>(args, sp);
}

void launch_list_walk(cudaStream_t s, const ListArgs &a, int *launches) {
    const int n = a.n;
    if (n <= 0) return;
    const int kind = walk_kind(a);
    if (kind == 3) {
        k_list_tile<1><<<nblk(n, 64), 64, 0, s>>>(a);
    } else if (kind == 4) {
        if (a.rows)
            k_list_tile<1, true, true><<<nblk(n, 64), 64, 0, s>>>(a);
        else
            k_list_tile<1, true><<<nblk(n, 64), 64, 0, s>>>(a);
    } else if (kind == 2) {
        k_list_tile<4><<<nblk(n, 32), 128, 0, s>>>(a);
    } else {
        with_team(n, [&](auto t) {
            constexpr int T = decltype(t)::value;
            k_list_gather<T><<<nblk(n * T, 128), 128, 0, s>>>(a);
        });
    }
    *launches += 1;
}

void list_offsets(cudaStream_t s, const ListArgs &a, SortScratch &sc, int *launches) {
    const int n = a.n;
    if (n <= 0) {
        cudaMemsetAsync(a.off, 0, sizeof(uint32_t), s);
        return;
    }
    scan_list_offsets(s, a.own, a.rev, a.off, n, sc, launches);
}

void launch_row_total(cudaStream_t s, int n, const uint32_t *rlen, unsigned long long *total,
                      int *launches) {
    cudaMemsetAsync(total, 0, sizeof(*total), s);
    if (n <= 0) return;
    k_row_total<<<std::min(152 * 8, nblk(n, 256)), 256, 0, s>>>(n, rlen, total);
    *launches += 1;
}

void build_lists_fill(cudaStream_t s, ListArgs a, bool mixed, bool queue,
                      int *launches) {
    (void)mixed;
    const int n = a.n;
    if (n <= 0) return;
    // at least 16 lanes per particle: a list's entries are then read from
    // the staging row and written to the list in 64-byte runs
    if (a.rows)
        k_list_place_rev<<<nblk(n, 256), 256, 0, s>>>(a);
    else
        with_team(n, [&](auto t) {
            constexpr int T = decltype(t)::value;
            k_list_place<T><<<nblk(n * T, 128), 128, 0, s>>>(a);
        }, 16);
    if (queue) {
        if (walk_kind(a) != 1)
            k_list_tile_queue<<<152 * 4, 128, 0, s>>>(a);
        else
            k_list_fill_queue<16><<<152 * 4, 128, 0, s>>>(a);
    }
    k_list_sort_rev<<<nblk(n, 256), 256, 0, s>>>(n, a.off, a.own, a.list, a.cap,
                                                  a.longq, a.nlong);
    // up to one warp per particle (4 per block): the long segments are
    // sorted in parallel whatever their number; idle warps exit at once
    k_list_sort_long<<<std::max(1, std::min(152 * 16, nblk(n, 4))), 128, 0, s>>>(
        a.off, a.own, a.list, a.longq, a.nlong);
    *launches += 4;
}

SPH_DEBUG_COUNTER(debug_failures_lists)

}  // namespace sph
