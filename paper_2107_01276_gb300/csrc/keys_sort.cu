// Cell keys, stable LSD radix sort, exclusive scan, permutation gather and
// the cell hash table: the neighbour-structure rebuild that the paper runs
// before every iteration (section 3.4, step iii: "update the nearest
// neighbor search").  All HBM-bound; no tensor cores.
#include <algorithm>

#include "batch.cuh"
#include "debug_checks.cuh"
#include "sph_internal.cuh"

namespace sph {

// ------------------------------------------------------------------ keys --
// Level l_i: smallest l >= 0 with c0 2^l >= t, t = (3 h_i) / c0 in FP64,
// capped at lmax.  Cell index floor((x - lo) / w_l) clamped to the level's
// cell count.  skey = l << (2 mbits) | morton(ix, iy), ix on even bits.
__device__ __forceinline__ int level_of(double h, double c0, int lmax) {
    double t = __ddiv_rn(__dmul_rn(3.0, h), c0);
    int l = 0;
    if (t > 1.0) {
        int e;
        double f = frexp(t, &e);
        l = (f == 0.5) ? e - 1 : e;
    }
    return l > lmax ? lmax : l;
}

__device__ __forceinline__ int cell_coord(double x, double lo, double w,
                                          int ncell) {
    double q = floor(__ddiv_rn(__dsub_rn(x, lo), w));
    int c;
    if (!(q >= 0.0))   // a NaN too, which converts to the least integer and
        c = 0;         // would stretch the level's box to it
    else if (q > (double)(ncell - 1))
        c = ncell - 1;
    else
        c = (int)q;
    return c;
}

// Fast forms of the two quotients above, for a GPU that issues an FP64
// instruction every 64 cycles a sub-partition: one conversion for the
// level, one FMA a coordinate.
// Level: t = 3 h / c0 in FP32 (relative error below 2^-21); away from a
// power of two by 2^-17 its exponent is that of the exact quotient.
// Cell: (x - lo) / w by one FMA onto 1.5 2^30, whose result holds the
// quotient in fixed point with 22 fractional bits, off by less than one
// unit of them (the rounding half, the reciprocal an eighth), so where the
// fraction is 4 or more units from an integer the integer part is the exact
// floor.  Everything closer than that (or out of
// these ranges) takes the correctly rounded division.
constexpr double CELL_MAGIC = 1610612736.0;   // 1.5 2^30

__device__ __forceinline__ int level_of_fast(double h, double c0, float k3,
                                             int lmax) {
    const float t = (float)h * k3;
    if (t > 1e-30f && t < 1e30f) {
        if (t < 1.0f - 1e-5f) return 0;
        const uint32_t b = __float_as_uint(t), m = b & 0x7fffffu;
        if (m > 64u && m < 0x7fffffu - 64u) {
            const int e = (int)(b >> 23) - 126;   // 2^(e-1) < t < 2^e
            return e > lmax ? lmax : e;
        }
    }
    return level_of(h, c0, lmax);
}

__device__ __forceinline__ int cell_coord_fast(double x, double lo, double w,
                                               double invw, int ncell) {
    const double y = __fma_rn(__dsub_rn(x, lo), invw, CELL_MAGIC);
    const uint32_t hi = (uint32_t)__double2hiint(y), lw = (uint32_t)__double2loint(y);
    const uint32_t fr = lw & 0x3fffffu;
    // 1.5 2^30 + [-2^28, 2^28)
    if (hi - 0x41d40000u >= 0x80000u || fr < 4u || fr > 0x3fffffu - 4u)
        return cell_coord(x, lo, w, ncell);
    const int c = (int)(((hi - 0x41d80000u) << 10) | (lw >> 22));
    return c < 0 ? 0 : c > ncell - 1 ? ncell - 1 : c;
}

__device__ __forceinline__ void keys_at(const KeysRec &r, int vb) {
    const int n = r.n;
    const KeysArgs &a = r.a;
    const double *__restrict__ x = r.x;
    const double *__restrict__ y = r.y;
    const double *__restrict__ h = r.h;
    uint64_t *__restrict__ skey = r.skey;
    uint32_t *__restrict__ perm = r.perm;
    uint32_t *level_mask = r.level_mask;
    int *bbox = r.bbox;
    uint32_t *__restrict__ zero = r.zero;
    uint32_t *__restrict__ zero2 = r.zero2;
    uint32_t *__restrict__ zero3 = r.zero3;
    __shared__ int sb[MAX_LEVELS * 4];
    __shared__ uint32_t smask;
    for (int t = threadIdx.x; t < MAX_LEVELS * 4; t += blockDim.x)
        sb[t] = (t & 1) ? -1 : 0x7fffffff;
    if (threadIdx.x == 0) smask = 0;
    __syncthreads();
    const int i = vb * blockDim.x + threadIdx.x;
    const bool ok = i < n;
    int l = MAX_LEVELS, ix = 0, iy = 0;
    if (ok) {
        l = level_of_fast(h[i], a.c0, a.k3, a.lmax);
        const Level &L = a.lev[l];
        ix = cell_coord_fast(x[i], a.dom.lo[0], L.w[0], a.invw[l][0], L.n[0]);
        iy = cell_coord_fast(y[i], a.dom.lo[1], L.w[1], a.invw[l][1], L.n[1]);
        uint64_t m = spread2((uint64_t)ix) | (spread2((uint64_t)iy) << 1);
        skey[i] = ((uint64_t)l << (2 * a.mbits)) | m;
        perm[i] = (uint32_t)i;
        if (zero) zero[i] = 0;
        if (zero2) zero2[i] = 0;
        if (zero3) zero3[i] = 0;
    }
    // level boxes: reduced over the lanes of each level first (most warps
    // hold one or two levels, and every thread's five shared atomics on the
    // same words had been most of this kernel)
    const unsigned peers = __match_any_sync(0xffffffffu, l);
    const int x0 = __reduce_min_sync(peers, ix), x1 = __reduce_max_sync(peers, ix);
    const int y0 = __reduce_min_sync(peers, iy), y1 = __reduce_max_sync(peers, iy);
    if (ok && (int)(threadIdx.x & 31) == __ffs(peers) - 1) {
        atomicOr(&smask, 1u << l);
        atomicMin(&sb[l * 4 + 0], x0);
        atomicMax(&sb[l * 4 + 1], x1);
        atomicMin(&sb[l * 4 + 2], y0);
        atomicMax(&sb[l * 4 + 3], y1);
    }
    __syncthreads();
    uint32_t msk = smask;
    for (int t = threadIdx.x; t < MAX_LEVELS * 4; t += blockDim.x) {
        int l = t >> 2;
        if (!(msk & (1u << l))) continue;
        if (t & 1)
            atomicMax(&bbox[t], sb[t]);
        else
            atomicMin(&bbox[t], sb[t]);
    }
    if (threadIdx.x == 0 && msk) atomicOr(level_mask, msk);
}

__global__ void k_keys(KeysRec r) { keys_at(r, blockIdx.x); }

void compute_levels(const Domain &dom, double c0, Level *lev) {
    for (int l = 0; l < MAX_LEVELS; ++l) {
        double c = ldexp(c0, l);
        lev[l].c = c;
        lev[l].cf = (float)c;
        for (int ax = 0; ax < 2; ++ax) {
            double Lx = dom.L[ax];
            long long nc;
            double w;
            if (dom.periodic[ax]) {
                nc = (long long)floor(Lx / c);
                if (nc < 1) nc = 1;
                w = Lx / (double)nc;
            } else {
                nc = (long long)ceil(Lx / c);
                if (nc < 1) nc = 1;
                w = c;
            }
            if (nc > (1ll << MAX_MORTON_BITS)) nc = 1ll << MAX_MORTON_BITS;
            lev[l].n[ax] = (int)nc;
            lev[l].w[ax] = w;
            lev[l].invw[ax] = (float)(1.0 / w);
            lev[l].wf[ax] = (float)w;
            lev[l].invP[ax] = (float)(1.0 / ((double)nc * w));
        }
    }
}

KeysRec make_keys_rec(int n, const Domain &dom, double c0, int lmax, int mbits,
                      const Level *lev, const double *x, const double *y,
                      const double *h, uint64_t *skey, uint32_t *perm,
                      uint32_t *level_mask, int *bbox, uint32_t *zero,
                      uint32_t *zero2, uint32_t *zero3) {
    KeysRec r;
    r.n = n;
    KeysArgs &a = r.a;
    a.dom = dom;
    a.c0 = c0;
    a.lmax = lmax;
    a.mbits = mbits;
    a.k3 = (float)(3.0 / c0);
    for (int l = 0; l < MAX_LEVELS; ++l) {
        a.lev[l] = lev[l];
        a.invw[l][0] = 1.0 / lev[l].w[0];
        a.invw[l][1] = 1.0 / lev[l].w[1];
    }
    r.x = x;
    r.y = y;
    r.h = h;
    r.skey = skey;
    r.perm = perm;
    r.level_mask = level_mask;
    r.bbox = bbox;
    r.zero = zero;
    r.zero2 = zero2;
    r.zero3 = zero3;
    return r;
}

void launch_keys(cudaStream_t s, int n, const Domain &dom, double c0,
                 int lmax, int mbits, const Level *lev, const double *x,
                 const double *y, const double *h, uint64_t *skey,
                 uint32_t *perm, uint32_t *level_mask, int *bbox,
                 uint32_t *zero, uint32_t *zero2, uint32_t *zero3) {
    if (n <= 0) return;
    const KeysRec r = make_keys_rec(n, dom, c0, lmax, mbits, lev, x, y, h, skey, perm,
                                    level_mask, bbox, zero, zero2, zero3);
    int bs = 256;
    k_keys<<<(n + bs - 1) / bs, bs, 0, s>>>(r);
}

// ------------------------------------------------------------ radix sort --
// 8-bit digits, 256 threads (8 warps) per tile of 8 * 32 * ITEMS keys.
// Warp w ranks its contiguous sub-tile step by step with __match_any_sync;
// the per-(warp, digit) running counts in shared memory make the rank
// stable.  Tile counts are scanned digit-major, so the scatter keeps the
// input order among equal digits across tiles as well.
constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;

template <bool SCATTER>
__global__ void __launch_bounds__(RS_THREADS)
    k_radix(int n, int shift, int ntiles, const uint64_t *__restrict__ kin,
            const uint32_t *__restrict__ vin, uint64_t *__restrict__ kout,
            uint32_t *__restrict__ vout, uint32_t *__restrict__ counts) {
    __shared__ uint32_t cnt[RS_WARPS][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int t = threadIdx.x; t < RS_WARPS * 256; t += RS_THREADS)
        (&cnt[0][0])[t] = 0;
    __syncthreads();
    const int tile = blockIdx.x;
    const long long base = (long long)tile * RS_TILE + (long long)w * 32 * RS_ITEMS;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t rank[RS_ITEMS];
    uint64_t key[RS_ITEMS];
    int dig[RS_ITEMS];
#pragma unroll
    for (int s = 0; s < RS_ITEMS; ++s) {
        long long e = base + s * 32 + lane;
        bool ok = e < n;
        uint64_t k = ok ? kin[e] : 0;
        int d = ok ? (int)((k >> shift) & 255u) : 256;
        key[s] = k;
        dig[s] = d;
        unsigned peers = __match_any_sync(0xffffffffu, d);
        int leader = __ffs(peers) - 1;
        uint32_t before = 0;
        if (ok) before = cnt[w][d];
        __syncwarp();
        if (ok && lane == leader) cnt[w][d] = before + __popc(peers);
        __syncwarp();
        rank[s] = before + __popc(peers & lt);
    }
    __syncthreads();
    if (!SCATTER) {
        int d = threadIdx.x;
        uint32_t tot = 0;
#pragma unroll
        for (int ww = 0; ww < RS_WARPS; ++ww) tot += cnt[ww][d];
        counts[(size_t)d * ntiles + tile] = tot;
        return;
    }
    {
        int d = threadIdx.x;
        uint32_t run = 0;
#pragma unroll
        for (int ww = 0; ww < RS_WARPS; ++ww) {
            uint32_t c = cnt[ww][d];
            cnt[ww][d] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < RS_ITEMS; ++s) {
        long long e = base + s * 32 + lane;
        if (e >= n) continue;
        int d = dig[s];
        uint32_t pos = counts[(size_t)d * ntiles + tile] + cnt[w][d] + rank[s];
        kout[pos] = key[s];
        vout[pos] = vin[e];
    }
}

// Small sets (n <= RSS_MAX): every pass in one block of 32 warps.  Warp w
// owns a contiguous run of the (current) order, its keys and their input
// positions in registers (up to IT a lane).  A pass ranks them 32 at a time
// with __match_any_sync against per-(warp, digit) counts, scans the counts
// digit-major (a warp takes 8 digits, a lane a warp's count), scatters keys
// and positions into shared memory and reloads them in the new order, so
// the sort is stable exactly like the tiled form.  A key travels whole where
// that is 32 bits, or 64 and n <= RSS_MAX / 2.  TWO: as one 32-bit word for
// any width up to RSS_MAX, the low one through the first four passes, then
// the high one, fetched from its place in the input, and the whole key at the
// end (64-bit keys leave room for half the items; wide sets of 8193 to 16384
// particles would go to the tiled sort's fifteen launches or more: 12000, 100
// -> 57 us a call.  Up to a thousand, whole keys save the two fetches, 1 us).
// Bound by the latency of its chain of passes: 5 us at 2.5k particles and 3
// digits, 9.5 us at 16k (the former form, with two rankings a pass and
// passes through global memory, took 10 and 29).
constexpr int RSS_THREADS = 1024;
constexpr int RSS_WARPS = RSS_THREADS / 32;
constexpr int RSS_MAX = 16384;

// dynamic shared memory: key words and 16-bit positions
static size_t radix_small_smem(int n, bool whole64) { return (size_t)n * (whole64 ? 10 : 6); }
static bool radix_small_whole64(int n, int passes) { return passes > 4 && n <= RSS_MAX / 2; }

template <typename K, int IT, bool TWO>
__device__ __forceinline__ void radix_small_body(int n, int passes, uint64_t *ka,
                                                 uint32_t *va, uint32_t (*cnt)[257],
                                                 uint32_t *dtot) {
    extern __shared__ uint64_t rss_buf[];          // n key words, then n positions
    K *sk = (K *)rss_buf;
    uint16_t *si = (uint16_t *)(sk + n);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int rows = (n + RSS_THREADS - 1) / RSS_THREADS;   // items a lane, <= IT
    const int wb = w * rows * 32 + lane;
    K key[IT];
    uint32_t ir[IT];                               // position | rank << 16
#pragma unroll
    for (int s = 0; s < IT; ++s) {
        const int e = wb + s * 32;
        key[s] = 0;
        ir[s] = 0;
        if (s < rows && e < n) {
            key[s] = (K)ka[e];
            ir[s] = (uint32_t)e;
        }
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * (TWO ? p & 3 : p);
        if (TWO && p == 4) {
#pragma unroll
            for (int s = 0; s < IT; ++s)
                if (s < rows && wb + s * 32 < n) key[s] = (K)(ka[ir[s]] >> 32);
        }
        for (int t = threadIdx.x; t < RSS_WARPS * 257; t += RSS_THREADS) (&cnt[0][0])[t] = 0;
        __syncthreads();
#pragma unroll
        for (int s = 0; s < IT; ++s) {
            if (s < rows) {
                const bool ok = wb + s * 32 < n;
                const int d = ok ? (int)((key[s] >> shift) & 255u) : 256;
                const unsigned peers = __match_any_sync(0xffffffffu, d);
                const uint32_t before = cnt[w][d];
                __syncwarp();
                if (lane == __ffs(peers) - 1) cnt[w][d] = before + __popc(peers);
                __syncwarp();
                ir[s] = (ir[s] & 0xffffu) | ((before + __popc(peers & lt)) << 16);
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 256 / RSS_WARPS; ++k) {
            const int d = w * (256 / RSS_WARPS) + k;
            const uint32_t c = cnt[lane][d];
            uint32_t x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            cnt[lane][d] = x - c;
            if (lane == 31) dtot[d] = x;
        }
        __syncthreads();
        if (w == 0) {                              // digit bases: exclusive scan of 256
            uint32_t v[8], sum = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                v[k] = dtot[lane * 8 + k];
                sum += v[k];
            }
            uint32_t x = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            x -= sum;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                dtot[lane * 8 + k] = x;
                x += v[k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < IT; ++s) {
            if (s < rows && wb + s * 32 < n) {
                const int d = (int)((key[s] >> shift) & 255u);
                const uint32_t pos = dtot[d] + cnt[w][d] + (ir[s] >> 16);
                sk[pos] = key[s];
                si[pos] = (uint16_t)ir[s];
            }
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < IT; ++s) {
            const int e = wb + s * 32;
            if (s < rows && e < n) {
                key[s] = sk[e];
                ir[s] = si[e];
            }
        }
    }
    // the keys and values of the final order, all read before any is replaced
    if (TWO && passes > 4) {   // (the low words wait in shared memory)
#pragma unroll
        for (int s = 0; s < IT; ++s)
            if (s < rows && wb + s * 32 < n) sk[wb + s * 32] = (uint32_t)ka[ir[s]];
        __syncthreads();
#pragma unroll
        for (int s = 0; s < IT; ++s)
            if (s < rows && wb + s * 32 < n)
                ka[wb + s * 32] = ((uint64_t)key[s] << 32) | sk[wb + s * 32];
    } else {
#pragma unroll
        for (int s = 0; s < IT; ++s)
            if (s < rows && wb + s * 32 < n) ka[wb + s * 32] = key[s];
    }
#pragma unroll
    for (int s = 0; s < IT; ++s)
        if (s < rows && wb + s * 32 < n) ir[s] = va[ir[s]];
    __syncthreads();
#pragma unroll
    for (int s = 0; s < IT; ++s)
        if (s < rows && wb + s * 32 < n) va[wb + s * 32] = ir[s];
}

__device__ __forceinline__ void radix_small_at(int n, int passes, uint64_t *ka, uint32_t *va) {
    __shared__ uint32_t cnt[RSS_WARPS][257];       // padded: a lane a row is conflict-free
    __shared__ uint32_t dtot[256];
    radix_small_body<uint32_t, RSS_MAX / RSS_THREADS, true>(n, passes, ka, va, cnt, dtot);
}

// Alone, the sort is compiled for the items a lane really has: the unrolled
// 16 of the largest sets are many times the instructions that a set of a
// thousand needs, and their fetching was most of its time.
template <typename K, int IT, bool TWO>
__global__ void __launch_bounds__(RSS_THREADS)
    k_radix_small(int n, int passes, uint64_t *ka, uint32_t *va) {
    __shared__ uint32_t cnt[RSS_WARPS][257];
    __shared__ uint32_t dtot[256];
    radix_small_body<K, IT, TWO>(n, passes, ka, va, cnt, dtot);
}
using RadixSmallFn = void (*)(int, int, uint64_t *, uint32_t *);
template <typename K, bool TWO>
static RadixSmallFn radix_small_fn_of(int n) {
    constexpr int MOST = sizeof(K) == 8 ? 8 : RSS_MAX / RSS_THREADS;
    return n <= RSS_THREADS ? k_radix_small<K, 1, TWO>
           : n <= 4 * RSS_THREADS ? k_radix_small<K, 4, TWO>
           : n <= 8 * RSS_THREADS ? k_radix_small<K, 8, TWO>
                                  : k_radix_small<K, MOST, TWO>;
}
static RadixSmallFn radix_small_fn(int n, int passes) {
    if (passes <= 4) return radix_small_fn_of<uint32_t, false>(n);
    if (radix_small_whole64(n, passes)) return radix_small_fn_of<uint64_t, false>(n);
    return k_radix_small<uint32_t, RSS_MAX / RSS_THREADS, true>;
}

// The dynamic shared-memory limit of k_radix_small, raised once per device.
static bool radix_small_ready() {
    static signed char ok[64];   // 0 unknown, 1 ready, -1 unavailable
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return false;
    }
    if (ok[dev] == 0) {
        signed char r = 1;
        for (int passes : {4, 8})
            for (int n : {RSS_THREADS, 4 * RSS_THREADS, 8 * RSS_THREADS, RSS_MAX})
                if (cudaFuncSetAttribute(radix_small_fn(n, passes),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)radix_small_smem(RSS_MAX, false)) != cudaSuccess)
                    r = -1;
        if (r < 0) cudaGetLastError();
        ok[dev] = r;
    }
    return ok[dev] == 1;
}

size_t radix_counts_elems(size_t n) {
    return 256 * ((n + RS_TILE - 1) / RS_TILE);
}

void radix_sort(cudaStream_t s, int n, int bits, uint64_t *key,
                uint32_t *val, SortScratch &sc, int *launches) {
    if (n <= 1 || bits <= 0) return;
    if (n <= RSS_MAX && radix_small_ready()) {
        const int passes = (bits + 7) / 8;
        radix_small_fn(n, passes)<<<1, RSS_THREADS,
                                    radix_small_smem(n, radix_small_whole64(n, passes)), s>>>(
            n, passes, key, val);
        *launches += 1;
        return;
    }
    int ntiles = (n + RS_TILE - 1) / RS_TILE;
    uint64_t *ka = key, *kb = sc.key_alt;
    uint32_t *va = val, *vb = sc.val_alt;
    int passes = (bits + 7) / 8;
    for (int p = 0; p < passes; ++p) {
        int shift = 8 * p;
        k_radix<false><<<ntiles, RS_THREADS, 0, s>>>(n, shift, ntiles, ka, va,
                                                     kb, vb, sc.counts);
        exclusive_scan(s, sc.counts, sc.counts, 256 * ntiles, nullptr, sc,
                       launches);
        k_radix<true><<<ntiles, RS_THREADS, 0, s>>>(n, shift, ntiles, ka, va,
                                                    kb, vb, sc.counts);
        *launches += 2;
        uint64_t *tk = ka; ka = kb; kb = tk;
        uint32_t *tv = va; va = vb; vb = tv;
    }
    if (ka != key) {
        cudaMemcpyAsync(key, ka, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(val, va, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, s);
    }
}

// ------------------------------------------------------------------ scan --
constexpr int SC_THREADS = 256;
constexpr int SC_ITEMS = 8;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;

__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v,
                                                    uint32_t *total) {
    __shared__ uint32_t ws[SC_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t t = lane < SC_THREADS / 32 ? ws[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < SC_THREADS / 32) ws[lane] = t;
    }
    __syncthreads();
    uint32_t pre = (w > 0 ? ws[w - 1] : 0) + x - v;
    if (total) *total = ws[SC_THREADS / 32 - 1];
    __syncthreads();
    return pre;
}

// rev (may be NULL): the values are in[i] + rev[i] for i < nrev; the down
// sweep zeroes rev.
__global__ void k_scan_reduce(const uint32_t *__restrict__ in,
                              const uint32_t *__restrict__ rev, int n,
                              uint32_t *__restrict__ sums) {
    long long b0 = (long long)blockIdx.x * SC_TILE;
    uint32_t acc = 0;
#pragma unroll
    for (int s = 0; s < SC_ITEMS; ++s) {
        long long e = b0 + s * SC_THREADS + threadIdx.x;
        if (e < n) acc += in[e] + (rev ? rev[e] : 0u);
    }
    uint32_t tot;
    block_excl_scan(acc, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// offs: exclusive sums of the tiles before each; total_dev (may be NULL)
// receives the sum of all values.
__global__ void k_scan_down(const uint32_t *in, uint32_t *rev, uint32_t *out, int n,
                            const uint32_t *__restrict__ offs,
                            uint32_t *total_dev) {
    long long b0 = (long long)blockIdx.x * SC_TILE +
                   (long long)threadIdx.x * SC_ITEMS;
    uint32_t v[SC_ITEMS];
    uint32_t acc = 0;
#pragma unroll
    for (int s = 0; s < SC_ITEMS; ++s) {
        long long e = b0 + s;
        v[s] = e < n ? in[e] + (rev ? rev[e] : 0u) : 0;
        acc += v[s];
    }
    uint32_t tot;
    uint32_t pre = block_excl_scan(acc, &tot);
    pre += offs[blockIdx.x];
#pragma unroll
    for (int s = 0; s < SC_ITEMS; ++s) {
        long long e = b0 + s;
        if (e < n) {
            out[e] = pre;
            if (rev) rev[e] = 0;
        }
        pre += v[s];
    }
    if (total_dev && blockIdx.x == gridDim.x - 1 && threadIdx.x == SC_THREADS - 1)
        *total_dev = pre;
}

size_t scan_scratch_elems(size_t n) {
    size_t tot = 0;
    while (n > (size_t)SC_TILE) {
        n = (n + SC_TILE - 1) / SC_TILE;
        tot += n;
    }
    return tot + 1;
}

// One-block scans (n <= 1024 * 32): warp w owns a contiguous run of up to
// 32 rows of 32 values, a lane one value a row, so every load and store is
// coalesced; in may equal out.  With `rev`, the values are in[i] + rev[i]
// and rev is zeroed (the neighbour-list totals), and out[n] receives the
// total.  (A thread owning 32 contiguous values, the former form, touched a
// cache line a lane with every load: 18 us for 32k values against 3.)
constexpr int SS_THREADS = 1024;
constexpr int SS_MAX = SS_THREADS * 32;

__device__ __forceinline__ void scan_small_at(const uint32_t *in, uint32_t *rev,
                                              uint32_t *out, int n,
                                              uint32_t *total_dev,
                                              int write_total_at_n) {
    __shared__ uint32_t ws[SS_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int rows = (n + SS_THREADS - 1) / SS_THREADS;   // <= 32
    const int b = w * rows * 32 + lane;
    uint32_t v[32];
    uint32_t sum = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        v[k] = 0;
        if (k < rows && b + k * 32 < n)
            v[k] = in[b + k * 32] + (rev ? rev[b + k * 32] : 0u);
    }
#pragma unroll
    for (int k = 0; k < 32; ++k) sum += v[k];
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) ws[w] = sum;
    __syncthreads();
    if (w == 0) {
        uint32_t t = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    uint32_t pre = w > 0 ? ws[w - 1] : 0u;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        if (k < rows) {
            uint32_t x = v[k];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            const int i = b + k * 32;
            if (i < n) {
                if (rev) rev[i] = 0;
                out[i] = pre + x - v[k];
            }
            pre += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    if (threadIdx.x == 0) {
        if (total_dev) *total_dev = ws[SS_THREADS / 32 - 1];
        if (write_total_at_n) out[n] = ws[SS_THREADS / 32 - 1];
    }
}

__global__ void __launch_bounds__(SS_THREADS)
    k_scan_small(const uint32_t *in, uint32_t *rev, uint32_t *out, int n,
                 uint32_t *total_dev, int write_total_at_n) {
    scan_small_at(in, rev, out, n, total_dev, write_total_at_n);
}

// Larger ones: tile sums, their scan (one block up to 67M values) and the
// tiles' own scans.
static void scan_rec(cudaStream_t s, const uint32_t *in, uint32_t *rev, uint32_t *out, int n,
                     uint32_t *total_dev, uint32_t *tmp, int *launches) {
    const int nb = (n + SC_TILE - 1) / SC_TILE;
    uint32_t *sums = tmp;
    k_scan_reduce<<<nb, SC_THREADS, 0, s>>>(in, rev, n, sums);
    *launches += 2;
    if (nb <= SS_MAX) {
        k_scan_small<<<1, SS_THREADS, 0, s>>>(sums, nullptr, sums, nb, nullptr, 0);
        *launches += 1;
    } else {
        scan_rec(s, sums, nullptr, sums, nb, nullptr, tmp + nb, launches);
    }
    k_scan_down<<<nb, SC_THREADS, 0, s>>>(in, rev, out, n, sums, total_dev);
}

void exclusive_scan(cudaStream_t s, const uint32_t *in, uint32_t *out, int n,
                    uint32_t *total_dev, SortScratch &sc, int *launches) {
    if (n <= 0) {
        if (total_dev) cudaMemsetAsync(total_dev, 0, sizeof(uint32_t), s);
        return;
    }
    if (n <= SS_MAX) {
        k_scan_small<<<1, SS_THREADS, 0, s>>>(in, nullptr, out, n, total_dev, 0);
        *launches += 1;
        return;
    }
    scan_rec(s, in, nullptr, out, n, total_dev, sc.scan_tmp, launches);
}

void scan_list_offsets(cudaStream_t s, const uint32_t *own, uint32_t *rev,
                       uint32_t *off, int n, SortScratch &sc, int *launches) {
    if (n <= SS_MAX) {
        k_scan_small<<<1, SS_THREADS, 0, s>>>(own, rev, off, n, nullptr, 1);
        *launches += 1;
        return;
    }
    scan_rec(s, own, rev, off, n, off + n, sc.scan_tmp, launches);
}

// ---------------------------------------------------------------- gather --
__global__ void k_gather(int n, const uint32_t *__restrict__ perm, GatherList g) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t src = perm[i];
    if (!SPH_DCHECK(src < (uint32_t)n)) return;
    for (int k = 0; k < g.nd; ++k) g.dst[k][i] = g.src[k][src];
    for (int k = 0; k < g.ni; ++k) g.idst[k][i] = g.isrc[k][src];
}

void gather_by_perm(cudaStream_t s, int n, const uint32_t *perm,
                    const GatherList &g, int *launches) {
    if (n <= 0) return;
    int bs = 256;
    k_gather<<<(n + bs - 1) / bs, bs, 0, s>>>(n, perm, g);
    *launches += 1;
}

// ------------------------------------------------------------ cell table --
__global__ void k_table_insert(int n, const uint64_t *__restrict__ skey,
                               uint64_t *tkey, uint32_t *tstart,
                               uint32_t tmask) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t k = skey[i];
    if (i > 0 && skey[i - 1] == k) return;
    uint32_t slot = hash_slot(k, tmask);
    // The table holds at most n keys in 2n slots, so a free slot exists and
    // the probe ends within tmask + 1 steps.
    for (uint32_t it = 0; it <= tmask; ++it) {
        unsigned long long prev = atomicCAS((unsigned long long *)&tkey[slot],
                                            (unsigned long long)EMPTY_KEY,
                                            (unsigned long long)k);
        if (prev == EMPTY_KEY || prev == k) {
            tstart[slot] = (uint32_t)i;
            return;
        }
        slot = (slot + 1) & tmask;
    }
}

__global__ void k_table_end(int n, const uint64_t *__restrict__ skey,
                            const uint64_t *__restrict__ tkey, uint32_t *tend,
                            uint32_t tmask, const double *h, float *tmaxh) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    table_mark_end(i, n, skey, tkey, tend, tmask, h, tmaxh);
}

// Reset before a rebuild: level bounding boxes and mask, every table key,
// and up to four counters.
__device__ __forceinline__ void rebuild_reset_at(const RebuildReset &r, uint32_t vb,
                                                 uint32_t nvb) {
    const uint32_t t0 = vb * blockDim.x + threadIdx.x;
    const uint32_t st = nvb * blockDim.x;
    if (t0 < MAX_LEVELS * 4) r.bbox[t0] = (t0 & 1) ? -1 : 0x7fffffff;
    if (t0 == 0) *r.level_mask = 0;
    if (t0 < 5 && r.zero[t0]) *r.zero[t0] = 0;
    for (uint32_t k = t0; k < r.tslots; k += st) r.tkey[k] = EMPTY_KEY;
}

__global__ void k_rebuild_reset(RebuildReset r) { rebuild_reset_at(r, blockIdx.x, gridDim.x); }

__global__ void k_occupancy(int n, const uint64_t *__restrict__ key,
                            int lshift, const int *__restrict__ bbox,
                            uint32_t *occ) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t k = key[i];
    const int l = (int)(k >> lshift);
    const uint64_t m = k & ((1ull << lshift) - 1ull);
    const int ix = (int)compact2(m), iy = (int)compact2(m >> 1);
    const int *bb = bbox + 4 * l;
    const int bx = occ_block(ix, bb[0], bb[1]), by = occ_block(iy, bb[2], bb[3]);
    atomicOr(&occ[(l * OCC_N + by) * (OCC_N / 32) + (bx >> 5)], 1u << (bx & 31));
}

void launch_occupancy(cudaStream_t s, int n, const uint64_t *key, int lshift,
                      const int *bbox, uint32_t *occ, int *launches) {
    cudaMemsetAsync(occ, 0, sizeof(uint32_t) * OCC_WORDS, s);
    if (n <= 0) return;
    k_occupancy<<<(n + 255) / 256, 256, 0, s>>>(n, key, lshift, bbox, occ);
    *launches += 1;
}

// Smallest value of v over each cell of a sorted set, stored at the cell's
// first particle (other entries are left as they are).
__global__ void k_cell_min(int n, const uint64_t *__restrict__ skey,
                           const double *__restrict__ v, double *cmin) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t k = skey[i];
    if (i > 0 && skey[i - 1] == k) return;
    double m = v[i];
    for (int j = i + 1; j < n && skey[j] == k; ++j) m = fmin(m, v[j]);
    cmin[i] = m;
}

void launch_cell_min(cudaStream_t s, int n, const uint64_t *skey,
                     const double *v, double *cmin, int *launches) {
    if (n <= 0) return;
    k_cell_min<<<(n + 255) / 256, 256, 0, s>>>(n, skey, v, cmin);
    *launches += 1;
}

int rebuild_reset_blocks(uint32_t tslots) {
    int nb = (int)std::min<uint32_t>((tslots + 255) / 256, 608u);
    return nb < 1 ? 1 : nb;
}
void launch_rebuild_reset(cudaStream_t s, const RebuildReset &r, int *launches) {
    k_rebuild_reset<<<rebuild_reset_blocks(r.tslots), 256, 0, s>>>(r);
    *launches += 1;
}

// ---------------------------------------------- batched small builds ----
// The same bodies over the work items of several instances (each item one
// block of the instance's single-launch grid); a block syncs before its
// next item, whose shared memory it reuses.
template <class Rec, class F>
__device__ __forceinline__ void batch_blocks(const Rec *args, const BatchSpan &sp, F &&f) {
    for (int it = blockIdx.x; it < sp.total; it += gridDim.x) {
        const BatchItem b = batch_item(sp, it);
        f(args[b.q], b.vb, b.nvb);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256)
    k_rebuild_reset_batch(const RebuildReset *args, BatchSpan sp) {
    batch_blocks(args, sp, [](const RebuildReset &r, int vb, int nvb) {
        rebuild_reset_at(r, vb, nvb);
    });
}
__global__ void __launch_bounds__(256) k_keys_batch(const KeysRec *args, BatchSpan sp) {
    batch_blocks(args, sp, [](const KeysRec &r, int vb, int) { keys_at(r, vb); });
}
__global__ void __launch_bounds__(RSS_THREADS)
    k_radix_small_batch(const RadixSmallRec *args, BatchSpan sp) {
    batch_blocks(args, sp, [](const RadixSmallRec &r, int, int) {
        radix_small_at(r.n, r.passes, r.ka, r.va);
    });
}
__global__ void __launch_bounds__(SS_THREADS)
    k_scan_small_batch(const ScanSmallRec *args, BatchSpan sp) {
    batch_blocks(args, sp, [](const ScanSmallRec &r, int, int) {
        scan_small_at(r.in, r.rev, r.out, r.n, r.total_dev, r.write_total_at_n);
    });
}

int radix_small_max() { return RSS_MAX; }
bool radix_small_available() { return radix_small_ready(); }
int scan_small_max() { return SS_MAX; }

template <class K>
static int resident(K kernel, int threads, size_t smem) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) !=
            cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return per_sm;
}
static int batch_grid(int per_sm, int total) {
    const long long g = (long long)per_sm * gpu_sms();
    return (int)(g < total ? g : total);
}
void launch_rebuild_reset_batch(cudaStream_t s, const RebuildReset *args, const BatchSpan &sp) {
    static const int r = resident(k_rebuild_reset_batch, 256, 0);
    if (sp.total > 0) k_rebuild_reset_batch<<<batch_grid(r, sp.total), 256, 0, s>>>(args, sp);
}
void launch_keys_batch(cudaStream_t s, const KeysRec *args, const BatchSpan &sp) {
    static const int r = resident(k_keys_batch, 256, 0);
    if (sp.total > 0) k_keys_batch<<<batch_grid(r, sp.total), 256, 0, s>>>(args, sp);
}
bool launch_radix_small_batch(cudaStream_t s, const RadixSmallRec *args, const BatchSpan &sp,
                              int max_n) {
    static const bool ok = cudaFuncSetAttribute(k_radix_small_batch,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)radix_small_smem(RSS_MAX, false)) == cudaSuccess;
    if (!ok || max_n > RSS_MAX) {
        cudaGetLastError();
        return false;
    }
    if (sp.total > 0)
        k_radix_small_batch<<<std::min(sp.total, gpu_sms()), RSS_THREADS, radix_small_smem(max_n, false),
                              s>>>(args, sp);
    return true;
}
void launch_scan_small_batch(cudaStream_t s, const ScanSmallRec *args, const BatchSpan &sp) {
    static const int r = resident(k_scan_small_batch, SS_THREADS, 0);
    if (sp.total > 0) k_scan_small_batch<<<batch_grid(r, sp.total), SS_THREADS, 0, s>>>(args, sp);
}


void build_cell_table(cudaStream_t s, int n, const uint64_t *skey,
                      uint64_t *tkey, uint32_t *tstart, uint32_t *tend,
                      uint32_t tmask, int *launches, const double *h,
                      float *tmaxh) {
    cudaMemsetAsync(tkey, 0xff, sizeof(uint64_t) * ((size_t)tmask + 1), s);
    if (n <= 0) return;
    int bs = 256;
    k_table_insert<<<(n + bs - 1) / bs, bs, 0, s>>>(n, skey, tkey, tstart, tmask);
    k_table_end<<<(n + bs - 1) / bs, bs, 0, s>>>(n, skey, tkey, tend, tmask, h,
                                                 tmaxh);
    *launches += 2;
}

SPH_DEBUG_COUNTER(debug_failures_keys_sort)

}  // namespace sph
