// build.cu -- octree build, bottom-up moments and i-groups.
//
// Octree (the Barnes-Hut tree of Sect. 3.2; its rules are this library's
// reading): a node is a (level l, key prefix) pair holding >= 1 particle; it
// is a leaf iff it holds <= n_leaf particles or l = 21; an internal node's
// children are its non-empty octants in digit order.  Node ids are BFS
// order: level-major, prefix ascending.  All levels are built at once from
// the sorted keys, one thread per position (see the particle-parallel build
// below).
//
// Moments: M and S = sum m x are accumulated in FP64 with explicitly
// rounded adds and multiplies (no FMA), leaves sequentially over their
// particles, internal nodes sequentially over their children in octant
// order; COM = S / M.  These fixed orders make the centres of mass, and
// thus the opening decisions of the walk, reproducible bit for bit.  The
// traceless quadrupole Q_ab = sum m (3 d_a d_b - |d|^2 delta_ab) about the
// COM (Sect. 2.1.2: FDPS ships superparticles up to the quadrupole) is summed over particles
// for leaves and combined from the children with the parallel-axis shift
// for internal nodes.
//
// i-groups (Barnes 1990; Sect. 5.5): the maximal nodes with <= n_grp
// particles, and leaves with more (possible only at level 21), in order of
// their first particle.
#include <algorithm>

#include "fdps_internal.cuh"

namespace fdps {
namespace {

constexpr int kB = 256;  // block size of the partitioned kernels

// Contiguous tile range [t0, t1) of block b when `ntile` tiles of kB items
// are split over gridDim.x blocks; the same split in every launch keeps the
// per-block partial sums consistent between the count and write kernels.
__device__ __forceinline__ void block_tiles(int64_t nitems, int64_t* t0, int64_t* t1) {
    int64_t ntile = (nitems + kB - 1) / kB;
    int64_t per = (ntile + gridDim.x - 1) / gridDim.x;
    *t0 = blockIdx.x * per;
    *t1 = *t0 + per < ntile ? *t0 + per : ntile;
}

__device__ __forceinline__ uint32_t block_sum(uint32_t v) {
    __shared__ uint32_t s[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    if (lane == 0) s[w] = v;
    __syncthreads();
    uint32_t r = 0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) r += s[k];
    __syncthreads();
    return r;  // valid in thread 0
}

__device__ __forceinline__ uint32_t block_excl(uint32_t v, uint32_t* total) {
    __shared__ uint32_t s_w[33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if (lane >= off) inc += t;
    }
    if (lane == 31) s_w[w] = inc;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    if (w == 0) {
        uint32_t t = lane < nw ? s_w[lane] : 0u;
        uint32_t ti = t;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            uint32_t u = __shfl_up_sync(0xFFFFFFFFu, ti, off);
            if (lane >= off) ti += u;
        }
        if (lane < nw) s_w[lane] = ti - t;
        if (lane == nw - 1) s_w[32] = ti;
    }
    __syncthreads();
    uint32_t res = s_w[w] + inc - v;
    *total = s_w[32];
    __syncthreads();
    return res;
}

// Exclusive scan of part[0..np) in one block; returns the total in *tot.
__device__ void scan_partials(uint32_t* part, int np, uint32_t* tot) {
    const int per = (np + blockDim.x - 1) / blockDim.x;
    const int b = threadIdx.x * per;
    uint32_t sum = 0;
    for (int k = 0; k < per; ++k)
        if (b + k < np) sum += part[b + k];
    uint32_t total;
    uint32_t off = block_excl(sum, &total);
    for (int k = 0; k < per; ++k)
        if (b + k < np) {
            uint32_t c = part[b + k];
            part[b + k] = off;
            off += c;
        }
    *tot = total;
}

__device__ __forceinline__ uint32_t meta_level(uint32_t m) { return m & 0xFFu; }
__device__ __forceinline__ uint32_t meta_nchild(uint32_t m) { return (m >> 8) & 0xFFu; }
__device__ __forceinline__ bool meta_leaf(uint32_t m) { return (m >> 16) & 1u; }

// Level 0: one root per system (node k = root of system k, owning
// positions off[k] .. off[k+1]; a single root over all n if off is null).
// The other levels' nodes come from the particle-parallel kernels below.
struct RootArgs {
    int n_roots;
    const int64_t* off;
    int64_t n;
    int n_leaf;
    uint32_t* nd_first;
    uint32_t* nd_count;
    uint32_t* nd_child;
    uint32_t* nd_meta;
    uint32_t* nd_parent;
    uint64_t* nd_qlo;
};

// (done by the blocks of the count pass, grid-strided)
__device__ __forceinline__ void write_roots(const RootArgs& R) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < R.n_roots;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t a = R.off ? R.off[k] : 0, b = R.off ? R.off[k + 1] : R.n;
        R.nd_first[k] = (uint32_t)a;
        R.nd_count[k] = (uint32_t)(b - a);
        R.nd_child[k] = 0xFFFFFFFFu;
        R.nd_meta[k] = (b - a <= R.n_leaf ? 1u : 0u) << 16;
        R.nd_parent[k] = 0xFFFFFFFFu;
        R.nd_qlo[k] = 0;
    }
}

// ------------------------------------------------ particle-parallel build
//
// All levels at once from the sorted keys.  D_j, the first level at which
// the keys of positions j-1 and j differ (0 where a system starts, 22 for
// equal keys), marks cell boundaries: the level-l cell holding position i
// runs from the last j <= i with D_j <= l to before the next j > i with
// D_j <= l (positions outside [0, n) count as D = 0).  Cells shrink with
// the level, so the leaf holding i is at LL_i, the first level whose cell
// holds <= n_leaf particles (21 if none), and every coarser cell holding i
// is an internal node.  Hence the nodes starting at i are levels
// max(D_i, 1) .. LL_i, and the nodes ending at j (holding j - 1, not j) are
// levels max(D_j, 1) .. LL_{j-1}.  Whether a cell holds <= n_leaf particles
// is decided within n_leaf <= 16 positions either side.  Node ids stay
// breadth-first (level-major, first particle ascending): id = start of the
// level + number of the level's nodes starting before i, from per-tile
// counts scanned per level and per-warp counts within the tile.

constexpr int kBT = 256;                    // threads per tile
constexpr int kBWarps = kBT / 32;
constexpr int kBRows = 8;                   // rows of 32 positions per warp
constexpr int kBTile = kBT * kBRows;        // positions per tile
// Sets of at most kBuildSmall positions take one row per warp and tiles of
// kBT: the rows of a warp follow one another (about 3 us each in the node
// pass), and a tile of 2048 leaves all but a few SMs idle.  Plummer 2001
// particles: count and node pass 14 + 25 us with 8 rows; the whole build
// of 2^14 particles 46 us with 8 rows and 23 with one.
static_assert(kBuildTileSmall == kBT && kBuildSmall % kBT == 0, "tile shape shared with the allocation");
constexpr int kHalo = kMaxLeaf;             // window either side of a row
static_assert(kBTile == kBuildTile && kBWarps == kBuildWarps, "tile shape shared with the allocation");
static_assert(kHalo == 16, "a row's window is 64 positions: 16 before, 32 own, 16 after");

__device__ __forceinline__ uint32_t first_diff_level(int64_t j, int64_t n, const uint64_t* __restrict__ keys,
                                                     const uint32_t* __restrict__ sys) {
    if (j <= 0 || j >= n) return 0u;
    if (sys && sys[j] != sys[j - 1]) return 0u;
    const uint64_t x = keys[j - 1] ^ keys[j];
    // keys have 63 bits: bit 62 is the top bit of the level-1 digit
    return x ? ((uint32_t)__clzll((long long)x) - 1u) / 3u + 1u : 22u;
}

// Does the cell holding window position c hold <= n_leaf particles, given
// the window's boundaries M (bit k: D of window position k <= the level)?
// A boundary missing on either side means more than 16 particles.
__device__ __forceinline__ bool cell_fits(unsigned long long M, int c, int n_leaf) {
    const unsigned long long back = M & ((2ull << c) - 1ull);
    const unsigned long long fwd = M >> (c + 1);
    if (!back || !fwd) return false;
    const int s = 63 - __clzll((long long)back);
    const int e = c + __ffsll((long long)fwd);
    return e - s <= n_leaf;
}

// Per tile: D and LL of every position (pk = D | LL << 8) and the number of
// nodes of each level starting in each warp's positions, per warp
// (wcount[(l - 1) * nw + warp]) and per tile (tcount[(l - 1) * ntiles +
// tile]).  A warp takes 32 consecutive positions at a time: 22 ballots give
// each level's boundaries in the 64-position window around them, and each
// lane bisects the levels for its LL.
template <int ROWS>
__global__ void __launch_bounds__(kBT) k_tree_count(int64_t n, int n_leaf, const uint64_t* __restrict__ keys,
                                                    const uint32_t* __restrict__ sys, uint32_t* __restrict__ pk,
                                                    uint32_t* __restrict__ wcount, uint32_t* __restrict__ tcount,
                                                    int64_t nw, int64_t ntiles, RootArgs R) {
    constexpr int kSpan = 32 * ROWS, kTile = kBT * ROWS;
    write_roots(R);  // level 0 (no other work of this pass depends on it)
    __shared__ uint8_t sD[kTile + 2 * kHalo];
    __shared__ unsigned long long s_m[kBWarps][kMaxLevel + 1];
    __shared__ uint32_t s_wc[kMaxLevel][kBWarps];
    const int64_t t0 = (int64_t)blockIdx.x * kTile;
    for (int q = threadIdx.x; q < kTile + 2 * kHalo; q += kBT)
        sD[q] = (uint8_t)first_diff_level(t0 - kHalo + q, n, keys, sys);
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = kHalo + lane;  // own window position
    uint32_t cnt[kMaxLevel];
#pragma unroll
    for (int l = 0; l < kMaxLevel; ++l) cnt[l] = 0u;
    for (int r = 0; r < ROWS; ++r) {
        const int rb = w * kSpan + r * 32;  // tile position of the row's first position
        const int64_t i = t0 + rb + lane;
        const uint32_t dA = sD[rb + lane];       // window 0..31
        const uint32_t dB = sD[rb + 32 + lane];  // window 32..63
        const uint32_t d = sD[rb + kHalo + lane];
#pragma unroll
        for (int l = 0; l <= kMaxLevel; ++l) {
            const uint32_t a = __ballot_sync(0xFFFFFFFFu, dA <= (uint32_t)l);
            const uint32_t b = __ballot_sync(0xFFFFFFFFu, dB <= (uint32_t)l);
            if (lane == 0) s_m[w][l] = (unsigned long long)a | ((unsigned long long)b << 32);
        }
        __syncwarp();
        int lo = 0, hi = kMaxLevel;  // first fitting level in [lo, hi], or 21
#pragma unroll
        for (int it = 0; it < 5; ++it) {
            const int mid = (lo + hi) >> 1;
            if (lo < hi) {
                if (cell_fits(s_m[w][mid], c, n_leaf))
                    hi = mid;
                else
                    lo = mid + 1;
            }
        }
        const uint32_t LL = (uint32_t)lo;
        __syncwarp();  // s_m is rewritten by the next row
        if (i < n) pk[i] = d | (LL << 8);
        const uint32_t l0 = max(d, 1u);
        const uint32_t mask = (i < n && l0 <= LL) ? ((2u << LL) - (1u << l0)) : 0u;
#pragma unroll
        for (int l = 1; l <= kMaxLevel; ++l) cnt[l - 1] += __popc(__ballot_sync(0xFFFFFFFFu, (mask >> l) & 1u));
    }
    uint32_t mine = 0u;
#pragma unroll
    for (int l = 0; l < kMaxLevel; ++l)
        if (lane == l) mine = cnt[l];
    if (lane < kMaxLevel) {
        wcount[(int64_t)lane * nw + (int64_t)blockIdx.x * kBWarps + w] = mine;
        s_wc[lane][w] = mine;
    }
    __syncthreads();
    if (threadIdx.x < kMaxLevel) {
        uint32_t t = 0u;
#pragma unroll
        for (int k = 0; k < kBWarps; ++k) t += s_wc[threadIdx.x][k];
        tcount[(int64_t)threadIdx.x * ntiles + blockIdx.x] = t;
    }
}

// Exclusive scan of one level's per-tile counts (block l - 1 takes level
// l); the level's total goes to ltot[l - 1].
__global__ void __launch_bounds__(1024) k_tree_scan(uint32_t* tcount, int64_t ntiles, uint32_t* ltot) {
    uint32_t tot;
    scan_partials(tcount + (int64_t)blockIdx.x * ntiles, (int)ntiles, &tot);
    if (threadIdx.x == 0) ltot[blockIdx.x] = tot;
}

__device__ __forceinline__ uint32_t compact3(uint64_t v) {
    v &= 0x1249249249249249ull;
    v = (v | (v >> 2)) & 0x10C30C30C30C30C3ull;
    v = (v | (v >> 4)) & 0x100F00F00F00F00Full;
    v = (v | (v >> 8)) & 0x001F0000FF0000FFull;
    v = (v | (v >> 16)) & 0x001F00000000FFFFull;
    v = (v | (v >> 32)) & 0x1FFFFFull;
    return (uint32_t)v;
}

// Writes every node of levels >= 1: first particle, level and leaf flag,
// parent, first child, grid origin, and (in nd_count, turned into the
// count by k_tree_finish) the position after its last particle.  The
// level-l node holding j - 1 is the last level-l node that starts before j,
// so a position's exclusive rank at each level names both the nodes it
// starts and those it ends.  The blocks cover positions 0 .. n (every open
// node ends at n).  Each block derives the level starts from the totals
// (levels from the first that does not fit in the node arrays on are left
// empty, with the overflow flag set); block 0 also publishes them.
template <int ROWS>
__global__ void __launch_bounds__(kBT) k_tree_nodes(
    int64_t n, int n_roots, int64_t cap_nodes, const uint64_t* __restrict__ keys,
    const uint32_t* __restrict__ sys, const uint32_t* __restrict__ pk, const uint32_t* __restrict__ wcount,
    const uint32_t* __restrict__ tcount, int64_t nw, int64_t ntiles, const uint32_t* __restrict__ ltot,
    DevState* st, uint32_t* __restrict__ nd_first, uint32_t* __restrict__ nd_end, uint32_t* __restrict__ nd_child,
    uint32_t* __restrict__ nd_meta, uint32_t* __restrict__ nd_parent, uint64_t* __restrict__ nd_qlo) {
    constexpr int kSpan = 32 * ROWS, kTile = kBT * ROWS;
    __shared__ int64_t s_lvl[kMaxLevel + 3];
    __shared__ uint32_t s_tot[kMaxLevel], s_pre[kMaxLevel];  // a level's nodes: all, and in earlier tiles
    __shared__ int s_cut;
    if (ROWS == 1) {  // few tiles: every block sums their counts itself (no scan pass)
        for (int l = threadIdx.x >> 5; l < kMaxLevel; l += kBWarps) {
            uint32_t tot = 0, pre = 0;
            for (int64_t k = threadIdx.x & 31; k < ntiles; k += 32) {
                const uint32_t v = tcount[(int64_t)l * ntiles + k];
                tot += v;
                pre += k < (int64_t)blockIdx.x ? v : 0u;
            }
            tot = __reduce_add_sync(0xFFFFFFFFu, tot);
            pre = __reduce_add_sync(0xFFFFFFFFu, pre);
            if ((threadIdx.x & 31) == 0) {
                s_tot[l] = tot;
                s_pre[l] = pre;
            }
        }
    } else if (threadIdx.x < kMaxLevel) {
        const int l = threadIdx.x;
        s_tot[l] = ltot[l];
        // a tile past the counted ones holds only position n: all of the
        // level's nodes come before
        s_pre[l] = (int64_t)blockIdx.x < ntiles ? tcount[(int64_t)l * ntiles + blockIdx.x] : ltot[l];
    }
    __syncthreads();
    __shared__ uint32_t s_wc[kMaxLevel][kBWarps];
    __shared__ uint32_t sP[1 + kTile];  // pk of positions t0 - 1 .. t0 + kTile - 1
    if (threadIdx.x == 0) {
        int64_t s = n_roots;
        // keys left unsorted by a sort that gave up: roots only, so that
        // every later stage stays within its buffers until the retry
        const bool stalled = st->overflow & kSortInvalid;
        int cut = stalled ? 1 : kMaxLevel + 1, top = 0;
        s_lvl[0] = 0;
        for (int l = 1; l <= kMaxLevel; ++l) {
            s_lvl[l] = s;
            if (cut > kMaxLevel && s + s_tot[l - 1] > cap_nodes) cut = l;
            if (cut > kMaxLevel) {
                s += s_tot[l - 1];
                if (s_tot[l - 1]) top = l;
            }
        }
        for (int l = cut; l <= kMaxLevel + 2; ++l) s_lvl[l] = s;
        s_cut = cut;
        if (blockIdx.x == 0) {
            for (int l = 0; l < kMaxLevel + 3; ++l) st->lvl_start[l] = (int32_t)s_lvl[l];
            st->n_nodes = (int32_t)s;
            st->max_level = top;
            if (cut <= kMaxLevel && !stalled) st->overflow |= kOvfNodes;
        }
    }
    const int64_t tile = blockIdx.x;
    const int64_t t0 = tile * kTile;
    // positions at or past n: D = 0, no nodes
    for (int q = threadIdx.x; q < 1 + kTile; q += kBT) {
        const int64_t j = t0 - 1 + q;
        sP[q] = (j >= 0 && j < n) ? pk[j] : 0u;
    }
    if (threadIdx.x < kMaxLevel * kBWarps) {
        const int l = threadIdx.x / kBWarps, k = threadIdx.x % kBWarps;
        s_wc[l][k] = tile < ntiles ? wcount[(int64_t)l * nw + tile * kBWarps + k] : 0u;
    }
    __syncthreads();
    const int cut = s_cut;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    // next id of each level for this warp: level start + nodes of earlier
    // tiles + nodes of earlier warps of this tile
    uint32_t nxt = 0u;
    if (lane >= 1 && lane <= kMaxLevel) {
        nxt = (uint32_t)s_lvl[lane] + s_pre[lane - 1];
        for (int k = 0; k < w; ++k) nxt += s_wc[lane - 1][k];
    }
    uint32_t run[kMaxLevel];
#pragma unroll
    for (int l = 1; l <= kMaxLevel; ++l) run[l - 1] = __shfl_sync(0xFFFFFFFFu, nxt, l);
    for (int r = 0; r < ROWS; ++r) {
        const int p = w * kSpan + r * 32 + lane;
        const int64_t j = t0 + p;
        const uint32_t v = sP[1 + p], u = sP[p];
        const uint32_t d = v & 0xFFu, LL = (v >> 8) & 0xFFu;
        const uint32_t lo = max(d, 1u), hi = LL;
        const bool any = j < n && lo <= hi;
        // levels of the nodes that end here
        uint32_t elo = 32u, ehi = 0u;
        if (j >= 1 && j <= n && d <= (uint32_t)kMaxLevel) {
            elo = max(d, 1u);
            ehi = (u >> 8) & 0xFFu;
        }
        uint64_t key = 0;
        uint32_t qx = 0, qy = 0, qz = 0, root = 0;
        if (any) {
            key = keys[j];
            qx = compact3(key >> 2);
            qy = compact3(key >> 1);
            qz = compact3(key);
            if (sys) root = sys[j];
        }
        uint32_t prev_id = 0u, prev_excl = 0u;
#pragma unroll
        for (int l = 1; l <= kMaxLevel; ++l) {
            const bool h = any && lo <= (uint32_t)l && (uint32_t)l <= hi;
            const uint32_t bm = __ballot_sync(0xFFFFFFFFu, h);
            const uint32_t excl = run[l - 1] + __popc(bm & lt);
            run[l - 1] += __popc(bm);
            if (l < cut) {
                if (elo <= (uint32_t)l && (uint32_t)l <= ehi) nd_end[excl - 1u] = (uint32_t)j;
                if (h) {
                    const uint32_t id = excl;
                    uint32_t parent;
                    if ((uint32_t)l > lo) {
                        parent = prev_id;
                        nd_child[prev_id] = id;  // first child of this position's previous node
                    } else if (l == 1) {
                        parent = root;
                        if (d == 0u) nd_child[root] = id;  // a system's first position
                    } else {
                        parent = prev_excl - 1u;  // last node of level l - 1 starting before j
                    }
                    const uint32_t cm = ~((1u << (kMaxLevel - l)) - 1u) & kQMax;
                    nd_first[id] = (uint32_t)j;
                    nd_child[id] = 0xFFFFFFFFu;
                    nd_meta[id] = (uint32_t)l | (((uint32_t)l == hi ? 1u : 0u) << 16);
                    nd_parent[id] = parent;
                    nd_qlo[id] = ((uint64_t)(qx & cm) << 42) | ((uint64_t)(qy & cm) << 21) | (uint64_t)(qz & cm);
                    prev_id = id;
                }
            }
            prev_excl = excl;
        }
    }
}

// Counts (end - first) and children counts: node c is the last child of
// its parent P iff the next node has another parent; it then stores c -
// first child of P + 1 in P's meta (one writer per parent).
__global__ void __launch_bounds__(256) k_tree_finish(const DevState* __restrict__ st, int n_roots,
                                                     const uint32_t* __restrict__ nd_first,
                                                     uint32_t* __restrict__ nd_count,
                                                     const uint32_t* __restrict__ nd_parent,
                                                     const uint32_t* __restrict__ nd_child,
                                                     uint32_t* __restrict__ nd_meta) {
    const int64_t nn = st->n_nodes;
    for (int64_t c = n_roots + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nn;
         c += (int64_t)gridDim.x * blockDim.x) {
        nd_count[c] -= nd_first[c];
        const uint32_t P = nd_parent[c];
        if (c + 1 == nn || nd_parent[c + 1] != P) nd_meta[P] |= ((uint32_t)c - nd_child[P] + 1u) << 8;
    }
}

// ------------------------------------------------------------ moments

__device__ __forceinline__ void split_hilo(double v, float* hi, float* lo) { split_f32(v, *hi, *lo); }

// S / M correctly rounded.  With one reciprocal y = RN(1/M) for a node's three
// quotients, Markstein's correction q0 = RN(S y), r = RN(S - M q0) and
// q = RN(q0 + r y), each step one fused multiply-add, gives RN(S / M)
// (Markstein 1990); the exponent guards keep every intermediate a normal
// number, elsewhere the division instruction sequence runs.
__device__ __forceinline__ bool exp_mid(double v) {
    const int e = (int)((__double_as_longlong(v) >> 52) & 0x7FF);
    return e >= 200 && e <= 1850;
}
__device__ __forceinline__ double quot(double S, double M, double y, bool ok) {
    if (!ok || !exp_mid(S)) return __ddiv_rn(S, M);  // zero, tiny or huge S: the division
    const double q0 = __dmul_rn(S, y);
    return __fma_rn(__fma_rn(-M, q0, S), y, q0);
}

struct MomArgs {
    const DevState* st;
    const SysBox* box;
    const uint32_t* sys;
    const double* px;
    const double* py;
    const double* pz;
    const double* pm;
    const double* pmx;  // m x, m y, m z per particle, each product rounded once
    const double* pmy;
    const double* pmz;
    const float4* pf_hi;
    const float4* pf_lo;
    const uint32_t* nd_first;
    const uint32_t* nd_count;
    const uint32_t* nd_child;
    const uint32_t* nd_meta;
    const uint64_t* nd_qlo;
    // written here and read back for the parent in a later launch (read
    // through L2 with __ldcg)
    double* nd_sx;
    double* nd_sy;
    double* nd_sz;
    dvec4* nd_com;
    double* nd_quad;
    float4* nd_f;
    WalkRec* nd_walk;
    float4* nd_fq0;
    float2* nd_fq1;
};

// Moments of node i, whose children (if any) are complete.  M and S = sum
// m x in FP64 with every operation rounded on its own: leaves sequentially
// over their particles (the products m x come rounded from the reorder,
// where every lane has a particle; a lane here sums one leaf of up to
// n_leaf particles, so its multiplications would idle the lanes of the
// warp's smaller leaves on the narrow FP64 pipe), internal nodes over their
// children in octant order.  Quadrupole: FP64 (Q64) for the FP64 pipeline; otherwise FP32 from
// positions relative to the node's COM formed from FP32 hi/lo pairs, and the
// parallel-axis shift for internal nodes.
// AHEAD: a node's children are all loaded before the first is summed (where
// latency counts and registers are free).  PART: everything, or only what
// follows from the sums M and S (kept in the node by k_moments_small).
enum MomPart { kMomAll, kMomFinish };
template <bool QUAD, bool Q64, bool AHEAD, MomPart PART = kMomAll>
__device__ __forceinline__ void node_moments(const MomArgs& A, int64_t i) {
    const uint32_t meta = A.nd_meta[i];
    const bool leaf = meta_leaf(meta);
    const uint32_t f = A.nd_first[i], cnt = A.nd_count[i];
    const uint32_t c0 = A.nd_child[i], nc = meta_nchild(meta);
    const SysBox& bx = A.box[A.sys ? A.sys[f] : 0];
    double M = 0.0, Sx = 0.0, Sy = 0.0, Sz = 0.0;
    if (PART == kMomFinish) {
        M = __ldcg(&A.nd_com[i].w);
        Sx = __ldcg(&A.nd_sx[i]);
        Sy = __ldcg(&A.nd_sy[i]);
        Sz = __ldcg(&A.nd_sz[i]);
    } else if (leaf) {
#pragma unroll 1
        for (uint32_t p = f; p < f + cnt; ++p) {
            M = __dadd_rn(M, A.pm[p]);
            Sx = __dadd_rn(Sx, A.pmx[p]);
            Sy = __dadd_rn(Sy, A.pmy[p]);
            Sz = __dadd_rn(Sz, A.pmz[p]);
        }
    } else if (AHEAD) {
        double m8[8], x8[8], y8[8], z8[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t c = k < (int)nc ? c0 + k : (uint32_t)i;  // past its children: the node itself
            m8[k] = __ldcg(&A.nd_com[c].w);
            x8[k] = __ldcg(&A.nd_sx[c]);
            y8[k] = __ldcg(&A.nd_sy[c]);
            z8[k] = __ldcg(&A.nd_sz[c]);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < (int)nc) {
                M = __dadd_rn(M, m8[k]);
                Sx = __dadd_rn(Sx, x8[k]);
                Sy = __dadd_rn(Sy, y8[k]);
                Sz = __dadd_rn(Sz, z8[k]);
            }
    } else {
        for (uint32_t c = c0; c < c0 + nc; ++c) {
            M = __dadd_rn(M, __ldcg(&A.nd_com[c].w));
            Sx = __dadd_rn(Sx, __ldcg(&A.nd_sx[c]));
            Sy = __dadd_rn(Sy, __ldcg(&A.nd_sy[c]));
            Sz = __dadd_rn(Sz, __ldcg(&A.nd_sz[c]));
        }
    }
    if (PART != kMomFinish) {
        A.nd_sx[i] = Sx;
        A.nd_sy[i] = Sy;
        A.nd_sz[i] = Sz;
    }
    double cx = 0.0, cy = 0.0, cz = 0.0;
    if (M > 0.0) {
        const bool ok = exp_mid(M);
        const double y = ok ? __ddiv_rn(1.0, M) : 0.0;
        cx = quot(Sx, M, y, ok);
        cy = quot(Sy, M, y, ok);
        cz = quot(Sz, M, y, ok);
    }
    A.nd_com[i] = make_dvec4(cx, cy, cz, M);
    float hx, hy, hz, lx, ly, lz;
    split_hilo(cx - bx.c0[0], &hx, &lx);
    split_hilo(cy - bx.c0[1], &hy, &ly);
    split_hilo(cz - bx.c0[2], &hz, &lz);
    A.nd_f[2 * i] = make_float4(hx, hy, hz, to_f32(M));
    A.nd_f[2 * i + 1] = make_float4(lx, ly, lz, 0.0f);
    const uint64_t qlo = A.nd_qlo[i];
    const uint32_t lev = meta_level(meta);
    WalkRec rec;
    rec.r = make_uint4((uint32_t)(qlo >> 42) | (lev << 21) | ((leaf ? 1u : 0u) << 26) | (nc << 27),
                       (uint32_t)(qlo >> 21) & kQMax, (uint32_t)qlo & kQMax, leaf ? cnt : c0);
    rec.c = make_float4(hx, hy, hz, 0.0f);
    A.nd_walk[i] = rec;
    if (!QUAD) return;
    if (Q64) {
        double q[6] = {0, 0, 0, 0, 0, 0};
        if (leaf) {
            for (uint32_t p = f; p < f + cnt; ++p) {
                const double m = A.pm[p];
                const double dx = A.px[p] - cx, dy = A.py[p] - cy, dz = A.pz[p] - cz;
                const double d2 = dx * dx + dy * dy + dz * dz;
                q[0] += m * (3.0 * dx * dx - d2);
                q[1] += m * (3.0 * dy * dy - d2);
                q[2] += m * (3.0 * dz * dz - d2);
                q[3] += m * (3.0 * dx * dy);
                q[4] += m * (3.0 * dx * dz);
                q[5] += m * (3.0 * dy * dz);
            }
        } else {
            for (uint32_t c = c0; c < c0 + nc; ++c) {
                const double ccx = __ldcg(&A.nd_com[c].x), ccy = __ldcg(&A.nd_com[c].y),
                             ccz = __ldcg(&A.nd_com[c].z), ccm = __ldcg(&A.nd_com[c].w);
                const double dx = ccx - cx, dy = ccy - cy, dz = ccz - cz;
                const double d2 = dx * dx + dy * dy + dz * dz;
                const double* qc = A.nd_quad + 6 * (int64_t)c;
                q[0] += __ldcg(qc + 0) + ccm * (3.0 * dx * dx - d2);
                q[1] += __ldcg(qc + 1) + ccm * (3.0 * dy * dy - d2);
                q[2] += __ldcg(qc + 2) + ccm * (3.0 * dz * dz - d2);
                q[3] += __ldcg(qc + 3) + ccm * (3.0 * dx * dy);
                q[4] += __ldcg(qc + 4) + ccm * (3.0 * dx * dz);
                q[5] += __ldcg(qc + 5) + ccm * (3.0 * dy * dz);
            }
        }
        double* qo = A.nd_quad + 6 * i;
#pragma unroll
        for (int k = 0; k < 6; ++k) qo[k] = q[k];
        A.nd_fq0[i] = make_float4((float)q[0], (float)q[1], (float)q[2], (float)q[3]);
        A.nd_fq1[i] = make_float2((float)q[4], (float)q[5]);
    } else {
        float q[6] = {0, 0, 0, 0, 0, 0};
        if (leaf) {
#pragma unroll 1
            for (uint32_t p = f; p < f + cnt; ++p) {
                const float4 ph = A.pf_hi[p], pl = A.pf_lo[p];
                const float m = ph.w;
                const float dx = (ph.x - hx) + (pl.x - lx), dy = (ph.y - hy) + (pl.y - ly),
                            dz = (ph.z - hz) + (pl.z - lz);
                const float d2 = dx * dx + dy * dy + dz * dz;
                q[0] += m * (3.0f * dx * dx - d2);
                q[1] += m * (3.0f * dy * dy - d2);
                q[2] += m * (3.0f * dz * dz - d2);
                q[3] += m * (3.0f * dx * dy);
                q[4] += m * (3.0f * dx * dz);
                q[5] += m * (3.0f * dy * dz);
            }
        } else {
            auto shift = [&](const float4 ch, const float4 cl, const float4 q0, const float2 q1) {
                const float dx = (ch.x - hx) + (cl.x - lx), dy = (ch.y - hy) + (cl.y - ly),
                            dz = (ch.z - hz) + (cl.z - lz);
                const float d2 = dx * dx + dy * dy + dz * dz;
                const float m = ch.w;
                q[0] += q0.x + m * (3.0f * dx * dx - d2);
                q[1] += q0.y + m * (3.0f * dy * dy - d2);
                q[2] += q0.z + m * (3.0f * dz * dz - d2);
                q[3] += q0.w + m * (3.0f * dx * dy);
                q[4] += q1.x + m * (3.0f * dx * dz);
                q[5] += q1.y + m * (3.0f * dy * dz);
            };
            if (AHEAD) {
                float4 ch[8], cl[8], q0[8];
                float2 q1[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint32_t c = k < (int)nc ? c0 + k : (uint32_t)i;
                    ch[k] = __ldcg(&A.nd_f[2 * c]);
                    cl[k] = __ldcg(&A.nd_f[2 * c + 1]);
                    q0[k] = __ldcg(&A.nd_fq0[c]);
                    q1[k] = __ldcg(&A.nd_fq1[c]);
                }
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (k < (int)nc) shift(ch[k], cl[k], q0[k], q1[k]);
            } else {
                for (uint32_t c = c0; c < c0 + nc; ++c)
                    shift(__ldcg(&A.nd_f[2 * c]), __ldcg(&A.nd_f[2 * c + 1]), __ldcg(&A.nd_fq0[c]),
                          __ldcg(&A.nd_fq1[c]));
            }
        }
        A.nd_fq0[i] = make_float4(q[0], q[1], q[2], q[3]);
        A.nd_fq1[i] = make_float2(q[4], q[5]);
    }
}

// Leaves of every level in one launch, then the internal nodes level by
// level from the deepest but one up in one more: a barrier between levels, so that
// each internal node finds its children complete.  With a launch per level
// (21, most of them for levels with few or no nodes) the internal nodes were
// all latency below about 10^6 particles.  Up to kMomSmall particles one
// cluster of CTAs takes all levels (a cluster barrier costs a fraction of a
// launch, and a level's few hundred nodes fill 8 SMs); beyond, a cooperative
// grid with a barrier in global memory, whose block 0 alone, with block
// barriers, finishes the levels near the roots once they and all above hold
// at most kTopNodes nodes.  Systems of an ensemble go through the same passes (one CTA
// per system before: 256 clusters of 256 to 65536 particles waited for the
// largest).  The sums of a node keep their order, so results do not depend
// on the split.  Moments of Plummer 2^14: 136 -> 39 us; of
// Plummer 2^20 with quadrupoles 246 -> 168 us; of the 256 clusters 1.18 ->
// 0.27 ms.
constexpr int kMomBlock = 256;
constexpr int kMomCl = 8;
// (65,536 Plummer / Hernquist particles, monopoles: 76 / 88 us by the cluster, 80 / 111 by
// the grid; 90,000: 92 / 108 and 80 / 107)
constexpr int64_t kMomSmall = int64_t(1) << 16;
// and up to about this many nodes (grid / cluster by nodes, n_leaf 1 or 8: 14,000
// 76 / 57 us, 24,319 117 / 111, 27,700 86 / 82, 35,600 113 / 147, 97,000 135 / 336).
// Leaves of up to n_leaf >= 8 make about 3.5 n / n_leaf nodes, single particles 1.5 n.
constexpr int64_t kMomSmallNodes = 28672;
constexpr int kTopNodes = 4 * kMomBlock;
constexpr int kMaxGridSpin = 1 << 20;

// The pass over the leaves is bound by the FP64 pipe, which a warp
// instruction takes whatever its active lanes: a block collects the leaves of
// kLeafTile nodes ordered by their particle counts (a counting sort; a leaf
// holds more than kMaxLeaf particles only at the deepest level), so that a
// warp's lanes sum leaves of like size.  With the internal nodes
// collected likewise: moments of 2^24 particles (quadrupoles) 1.00 -> 0.92 ms, of
// 3M clumpy particles (monopoles) 0.36 -> 0.24 ms.
// The pass takes every node without children: beside the leaves the last kept
// level's internal nodes of a cut tree (node arrays too small, or roots only
// after a sort that gave up), whose records the passes over the levels do not
// reach.  Such a node gets no mass and a record without children, so that
// whatever follows a record stays within the tree.
constexpr int kLeafTile = kMomBlock;
template <bool QUAD, bool Q64>
__global__ void __launch_bounds__(kMomBlock) k_moments_leaves(MomArgs A) {
    __shared__ uint32_t s_id[kLeafTile];
    __shared__ uint32_t s_bin[32], s_total;
    const int t = threadIdx.x;
    const int64_t nn = A.st->n_nodes;
    for (int64_t base = (int64_t)blockIdx.x * kLeafTile; base < nn; base += (int64_t)gridDim.x * kLeafTile) {
        const int64_t i = base + t;
        uint32_t bin = 0, rank = 0;  // bin 0: no leaf
        if (t < 32) s_bin[t] = 0;
        __syncthreads();
        if (i < nn && meta_nchild(A.nd_meta[i]) == 0u) {
            const uint32_t c = A.nd_count[i];
            bin = c <= (uint32_t)kMaxLeaf ? c : (uint32_t)kMaxLeaf + 1u;
            rank = atomicAdd(&s_bin[bin], 1u);
        }
        __syncthreads();
        if (t < 32) {
            const uint32_t v = s_bin[t];
            uint32_t inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (t >= o) inc += u;
            }
            s_bin[t] = inc - v;
            if (t == 31) s_total = inc;
        }
        __syncthreads();
        if (bin) s_id[s_bin[bin] + rank] = (uint32_t)i;
        __syncthreads();
        if (t < (int)s_total) node_moments<QUAD, Q64, false>(A, s_id[t]);
        __syncthreads();  // the bins are rewritten
    }
}

// (A monopole tree's levels pass on the sums alone: the division and the FP32
// copies, two thirds of a node's chain of FP64 operations, follow for all
// internal nodes at once.  Four lanes share a node, one for each of M, Sx, Sy
// and Sz: a level's few nodes are a chain of loads and FP64 additions whose
// length counts, not their number; and a lane reads its node of the next level
// and that node's children's ids before it waits for this level.  Moments of
// 2^14 Plummer particles 55 -> 39 us, of 2001 39 -> 27 (49 and 35 with one lane a
// node and nothing read ahead).  A quadrupole needs its children's centres.)
template <bool QUAD, bool Q64>
__global__ void __cluster_dims__(kMomCl, 1, 1) __launch_bounds__(kMomBlock) k_moments_small(MomArgs A) {
    __shared__ int32_t s_lvl[kMaxLevel + 3];
    if (threadIdx.x < kMaxLevel + 3) s_lvl[threadIdx.x] = A.st->lvl_start[threadIdx.x];
    const int top = A.st->max_level - 1;
    __syncthreads();
    const int t = blockIdx.x * kMomBlock + threadIdx.x;
    if (top < 0) return;  // (the whole cluster)
    // monopoles: four lanes a node, one for each of M, Sx, Sy, Sz
    constexpr int kLanes = QUAD ? 1 : 4, kNodes = kMomCl * kMomBlock / kLanes;
    const int comp = t % 4;
    double* const sum = comp == 0 ? &A.nd_com[0].w : comp == 1 ? A.nd_sx : comp == 2 ? A.nd_sy : A.nd_sz;
    const int64_t stride = comp == 0 ? 4 : 1;
    int next = s_lvl[top] + t / kLanes;
    uint32_t next_meta = next < s_lvl[top + 1] ? A.nd_meta[next] : 0u;
    uint32_t next_child = next < s_lvl[top + 1] ? A.nd_child[next] : 0u;
    for (int l = top; l >= 0; --l) {
        int i = next;
        uint32_t meta = next_meta, child = next_child;
        if (l > 0) {
            next = s_lvl[l - 1] + t / kLanes;
            next_meta = next < s_lvl[l] ? A.nd_meta[next] : 0u;
            next_child = next < s_lvl[l] ? A.nd_child[next] : 0u;
        }
        while (i < s_lvl[l + 1]) {
            if (meta_leaf(meta)) {
            } else if (QUAD) {
                node_moments<QUAD, Q64, true>(A, i);
            } else {
                const int nc = (int)meta_nchild(meta);
                double v[8], S = 0.0;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    v[k] = __ldcg(sum + (int64_t)(k < nc ? child + k : (uint32_t)i) * stride);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (k < nc) S = __dadd_rn(S, v[k]);
                sum[i * stride] = S;
            }
            i += kNodes;
            if (i >= s_lvl[l + 1]) break;
            meta = A.nd_meta[i];
            child = A.nd_child[i];
        }
        cluster_barrier();  // this level complete before its parents
    }
    if (!QUAD)
        for (int i = t; i < s_lvl[top + 1]; i += kMomCl * kMomBlock)
            if (!meta_leaf(A.nd_meta[i])) node_moments<QUAD, Q64, true, kMomFinish>(A, i);
}

// Barrier over the grid (all blocks resident: a cooperative launch); count
// starts at zero and target is a multiple of the grid size, one more for
// each barrier.  The wait is bounded: beyond it the error bit of a device
// wait is set and the block goes on (its sums are then invalid, every access
// stays within the node arrays).
__device__ __forceinline__ void grid_barrier(uint32_t* count, uint32_t target, uint32_t* overflow,
                                             int max_spin = kMaxGridSpin) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1u);
        int spin = 0;
        while (*(volatile uint32_t*)count < target)
            if (++spin > max_spin) {
                atomicOr(overflow, kSortStall);
                break;
            }
        __threadfence();
    }
    __syncthreads();
}

// (A quarter or less of a level's nodes are internal: each warp collects 32
// of them before it sums any, for the FP64 pipe's sake as above.)
template <bool QUAD, bool Q64>
__global__ void __launch_bounds__(kMomBlock, 2) k_moments_levels(MomArgs A, uint32_t* count, uint32_t* overflow) {
    __shared__ uint32_t s_id[kMomBlock / 32][64];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)kMomBlock + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * kMomBlock) >> 5;
    uint32_t target = 0;
    int l = A.st->max_level - 1;
    for (; l >= 0; --l) {
        const int64_t a = A.st->lvl_start[l], b = A.st->lvl_start[l + 1];
        if (b <= kTopNodes) break;
        uint32_t held = 0;
        for (int64_t base = a + warp * 32; base < b; base += nwarps * 32) {
            const int64_t i = base + lane;
            const bool in = i < b && !meta_leaf(A.nd_meta[i]);
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, in);
            if (in) s_id[w][held + __popc(m & ((1u << lane) - 1u))] = (uint32_t)i;
            held += __popc(m);
            __syncwarp();
            if (held >= 32) {
                node_moments<QUAD, Q64, true>(A, s_id[w][lane]);
                held -= 32;
                const uint32_t rest = s_id[w][32 + lane];
                __syncwarp();
                if (lane < held) s_id[w][lane] = rest;
                __syncwarp();
            }
        }
        if (lane < held) node_moments<QUAD, Q64, true>(A, s_id[w][lane]);
        target += gridDim.x;
        grid_barrier(count, target, overflow);
    }
    if (blockIdx.x != 0) return;
    for (; l >= 0; --l) {
        const int64_t a = A.st->lvl_start[l], b = A.st->lvl_start[l + 1];
        for (int64_t i = a + threadIdx.x; i < b; i += kMomBlock)
            if (!meta_leaf(A.nd_meta[i])) node_moments<QUAD, Q64, true>(A, i);
        __threadfence_block();
        __syncthreads();  // this level complete before its parents
    }
}

// A barrier of one block that waits for an arrival that never comes.
__global__ void k_barrier_selftest(uint32_t* count, uint32_t* flags, int max_spin) {
    grid_barrier(count, 2u, flags, max_spin);
}

template <bool QUAD, bool Q64>
int launch_moments(fdps_ctx* ctx, const MomArgs& A, int64_t n, int n_leaf, DevState* st) {
    k_moments_leaves<QUAD, Q64><<<ctx->sm_count * 8, kMomBlock, 0, ctx->stream>>>(A);
    FDPS_LAUNCH_CHECK(ctx);
    if (n <= kMomSmall && std::min(3 * n / 2, 7 * n / (2 * n_leaf)) <= kMomSmallNodes) {
        k_moments_small<QUAD, Q64><<<kMomCl, kMomBlock, 0, ctx->stream>>>(A);
        FDPS_LAUNCH_CHECK(ctx);
        return FDPS_OK;
    }
    int per_sm = 0;
    FDPS_CUDA_TRY(ctx,
                  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_moments_levels<QUAD, Q64>, kMomBlock, 0));
    // every block resident, and no more than two per SM to meet at a barrier
    const int grid = ctx->sm_count * std::max(1, std::min(2, per_sm));
    MomArgs args = A;
    uint32_t* count = &st->mom_counter;
    uint32_t* overflow = &st->overflow;
    void* kargs[] = {&args, &count, &overflow};
    FDPS_CUDA_TRY(ctx, cudaLaunchCooperativeKernel((const void*)k_moments_levels<QUAD, Q64>, dim3((unsigned)grid),
                                                   dim3(kMomBlock), kargs, 0, ctx->stream));
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

// ------------------------------------------------------------- groups

__global__ void __launch_bounds__(256) k_group_mark(const DevState* __restrict__ st, int n_grp,
                                                    int n_roots,
                                                    const uint32_t* __restrict__ nd_first,
                                                    const uint32_t* __restrict__ nd_count,
                                                    const uint32_t* __restrict__ nd_meta,
                                                    const uint32_t* __restrict__ nd_parent,
                                                    uint32_t* __restrict__ head) {
    const int64_t nn = st->n_nodes;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nn;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = nd_count[i];
        const bool cand = c <= (uint32_t)n_grp || meta_leaf(nd_meta[i]);
        if (cand && (i < n_roots || nd_count[nd_parent[i]] > (uint32_t)n_grp)) head[nd_first[i]] = (uint32_t)i;
    }
}

// Group heads per block; the last block to finish (counted in
// st->grp_done, zero on entry) scans the per-block counts into offsets and
// publishes the number of groups.
__global__ void __launch_bounds__(kB) k_group_count(int64_t n, const uint32_t* __restrict__ head,
                                                    uint32_t* __restrict__ part, DevState* st,
                                                    int64_t cap_groups) {
    __shared__ bool s_last;
    int64_t t0, t1;
    block_tiles(n, &t0, &t1);
    uint32_t c = 0;
    for (int64_t t = t0; t < t1; ++t) {
        const int64_t i = t * kB + threadIdx.x;
        if (i < n && head[i] != 0xFFFFFFFFu) ++c;
    }
    uint32_t tot = block_sum(c);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = tot;
        __threadfence();  // the count is visible before the block counts itself done
        s_last = atomicAdd(&st->grp_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int np = (int)gridDim.x;
    const int per = (np + kB - 1) / kB;
    const int b = threadIdx.x * per;
    uint32_t sum = 0;
    for (int k = 0; k < per; ++k)
        if (b + k < np) sum += __ldcg(&part[b + k]);
    uint32_t total;
    uint32_t off = block_excl(sum, &total);
    for (int k = 0; k < per; ++k)
        if (b + k < np) {
            const uint32_t v = __ldcg(&part[b + k]);
            part[b + k] = off;
            off += v;
        }
    if (threadIdx.x == 0) {
        if ((int64_t)total > cap_groups) st->overflow |= kOvfGroups;
        st->n_groups = (int32_t)((int64_t)total > cap_groups ? cap_groups : total);
    }
}

__global__ void __launch_bounds__(kB) k_group_write(int64_t n, int64_t cap_groups,
                                                    const uint32_t* __restrict__ head,
                                                    const uint32_t* __restrict__ part,
                                                    const uint32_t* __restrict__ nd_count,
                                                    uint32_t* __restrict__ g_node,
                                                    uint32_t* __restrict__ g_first,
                                                    uint32_t* __restrict__ g_count) {
    int64_t t0, t1;
    block_tiles(n, &t0, &t1);
    uint32_t running = part[blockIdx.x];
    for (int64_t t = t0; t < t1; ++t) {
        const int64_t i = t * kB + threadIdx.x;
        const uint32_t h = i < n ? head[i] : 0xFFFFFFFFu;
        const uint32_t flag = h != 0xFFFFFFFFu ? 1u : 0u;
        uint32_t tot;
        const uint32_t rank = block_excl(flag, &tot);
        if (flag) {
            const int64_t g = (int64_t)running + rank;
            if (g < cap_groups) {
                g_node[g] = h;
                g_first[g] = (uint32_t)i;
                g_count[g] = nd_count[h];
            }
        }
        running += tot;
    }
}

// The i-groups of at most kGroupSmall positions in one block: heads as bits
// of a word per thread in shared memory, their ranks from one scan (a clear,
// a mark, a count and a write pass over the positions before, 17 us of which
// little was work; all group passes of 2^14
// particles 25 -> 16 us, of 2001 25 -> 12 us).
constexpr int kGroupSmallBlock = 1024;
constexpr int64_t kGroupSmall = 32 * kGroupSmallBlock;
// (the passes over the positions against the block, by groups: 1106 27 / 16 us,
// 2659 27 / 25, 3522 27 / 25, 5871 29 / 31, 11956 31 / 51)
constexpr int64_t kGroupSmallGroups = 4096;
__global__ void __launch_bounds__(kGroupSmallBlock) k_group_small(DevState* st, int n_grp, int n_roots,
                                                                  int64_t cap_groups,
                                                                  const uint32_t* __restrict__ nd_first,
                                                                  const uint32_t* __restrict__ nd_count,
                                                                  const uint32_t* __restrict__ nd_meta,
                                                                  const uint32_t* __restrict__ nd_parent,
                                                                  uint32_t* head, uint32_t* __restrict__ g_node,
                                                                  uint32_t* __restrict__ g_first,
                                                                  uint32_t* __restrict__ g_count) {
    __shared__ uint32_t s_bits[kGroupSmallBlock];
    const int t = threadIdx.x;
    s_bits[t] = 0;
    __syncthreads();
    const int nn = st->n_nodes;
    for (int i = t; i < nn; i += kGroupSmallBlock) {
        const bool cand = nd_count[i] <= (uint32_t)n_grp || meta_leaf(nd_meta[i]);
        if (cand && (i < n_roots || nd_count[nd_parent[i]] > (uint32_t)n_grp)) {
            const uint32_t p = nd_first[i];
            head[p] = (uint32_t)i;
            atomicOr(&s_bits[p >> 5], 1u << (p & 31u));
        }
    }
    __syncthreads();
    uint32_t bits = s_bits[t], total;
    int64_t g = block_excl(__popc(bits), &total);
    for (; bits; bits &= bits - 1u, ++g) {
        const uint32_t p = 32u * t + __ffs(bits) - 1u;
        const uint32_t h = head[p];
        if (g < cap_groups) {
            g_node[g] = h;
            g_first[g] = p;
            g_count[g] = nd_count[h];
        }
    }
    if (t == 0) {
        if ((int64_t)total > cap_groups) st->overflow |= kOvfGroups;
        st->n_groups = (int32_t)((int64_t)total > cap_groups ? cap_groups : total);
    }
}

__device__ __forceinline__ unsigned long long ord64(double v) {
    unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double unord64(unsigned long long o) {
    unsigned long long u = (o >> 63) ? (o & 0x7FFFFFFFFFFFFFFFull) : ~o;
    return __longlong_as_double((long long)u);
}

// FP64 box of each group (min / max over its particles), its grid box (the
// quantised corners: quantisation is monotone, so these are the minimum and
// maximum grid coordinates of the particles), FP64 centre and the FP32
// copies the walk's filter and the force kernel use.  A warp takes a run of
// up to kGrpRun groups: the lanes reduce each group's particles together, then
// lane 3 j + a finishes axis a of group j (the FP64 pipe is narrow: a lane
// per axis takes it for a third of the warp instructions of a lane per
// group).  Runs are short where there are few groups, so that all warps have
// one: each group of a run costs its loads' latency and 60 shuffles in turn
// (with runs of 32 the pass took 115 us on the 27,500 groups of 2^20
// particles, most of the GPU idle; with short
// runs all group passes together went from 143 to 59 us, on the 1,002 groups
// of 2^14 particles from 51 to 25 us).
constexpr int kGrpRun = 10;  // 30 of a warp's lanes
__global__ void __launch_bounds__(256) k_group_data(
    const DevState* __restrict__ st, const SysBox* __restrict__ box, const uint32_t* __restrict__ sys,
    const uint32_t* __restrict__ g_first,
    const uint32_t* __restrict__ g_count, const double* __restrict__ px,
    const double* __restrict__ py, const double* __restrict__ pz, double* __restrict__ g_box,
    uint32_t* __restrict__ g_qbox, dvec4* __restrict__ g_c64, float4* __restrict__ g_ch,
    float4* __restrict__ g_cl, float4* __restrict__ g_blo, float4* __restrict__ g_bhi) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t ng = st->n_groups;
    const int64_t per = (ng + nwarps - 1) / nwarps;
    const int run = per < kGrpRun ? (int)per : kGrpRun;
    const int lj = lane / 3, la = lane - 3 * lj;
    for (int64_t base = warp * run; base < ng; base += nwarps * run) {
        unsigned long long mlo = 0, mhi = 0;
        const int nb = ng - base < run ? (int)(ng - base) : run;
        for (int j = 0; j < nb; ++j) {
            const uint32_t f = g_first[base + j], c = g_count[base + j];
            unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
            for (uint32_t p = f + lane; p < f + c; p += 32) {
                unsigned long long v[3] = {ord64(px[p]), ord64(py[p]), ord64(pz[p])};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    lo[a] = v[a] < lo[a] ? v[a] : lo[a];
                    hi[a] = v[a] > hi[a] ? v[a] : hi[a];
                }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    unsigned long long l2 = __shfl_xor_sync(0xFFFFFFFFu, lo[a], off);
                    unsigned long long h2 = __shfl_xor_sync(0xFFFFFFFFu, hi[a], off);
                    lo[a] = l2 < lo[a] ? l2 : lo[a];
                    hi[a] = h2 > hi[a] ? h2 : hi[a];
                }
            if (lj == j) {
                mlo = la == 0 ? lo[0] : la == 1 ? lo[1] : lo[2];
                mhi = la == 0 ? hi[0] : la == 1 ? hi[1] : hi[2];
            }
        }
        if (lj >= nb) continue;
        const int64_t g = base + lj;
        const SysBox& bx = box[sys ? sys[g_first[g]] : 0];
        const double bl = unord64(mlo), bh = unord64(mhi);
        g_box[6 * g + la] = bl;
        g_box[6 * g + 3 + la] = bh;
        g_qbox[6 * g + la] = quantise(bl, bx.lo[la], bx.s);
        g_qbox[6 * g + 3 + la] = quantise(bh, bx.lo[la], bx.s);
        const double cc = __dmul_rn(__dadd_rn(bl, bh), 0.5);
        float ch, cl;
        split_hilo(cc - bx.c0[la], &ch, &cl);
        reinterpret_cast<double*>(g_c64 + g)[la] = cc;
        reinterpret_cast<float*>(g_ch + g)[la] = ch;
        reinterpret_cast<float*>(g_cl + g)[la] = cl;
        reinterpret_cast<float*>(g_blo + g)[la] = __double2float_rd(bl - cc);
        reinterpret_cast<float*>(g_bhi + g)[la] = __double2float_ru(bh - cc);
        if (la == 0) {  // the vectors' unused fourth components
            g_c64[g].w = 0.0;
            g_ch[g].w = g_cl[g].w = g_blo[g].w = g_bhi[g].w = 0.0f;
        }
    }
}

}  // namespace

int build_tree(fdps_tree* t, fdps_psys* ps) {
    fdps_ctx* ctx = t->ctx;
    cudaStream_t s = ctx->stream;
    const int64_t n = ps->n;
    const bool small = n <= kBuildSmall;
    const int64_t tile = small ? kBT : kBTile;
    const int64_t ntiles = n > 0 ? (n + tile - 1) / tile : 1;
    const int64_t nw = ntiles * kBWarps;
    uint32_t* wcount = t->bt_count;                 // [21][nw] per warp
    uint32_t* tcount = wcount + kMaxLevel * nw;     // [21][ntiles] per tile, then scanned
    uint32_t* ltot = tcount + kMaxLevel * ntiles;   // [21]
    const RootArgs R{ps->n_sys, ps->d_off, n, t->p.n_leaf, t->nd_first, t->nd_count,
                     t->nd_child, t->nd_meta, t->nd_parent, t->nd_qlo};
    // per-position scratch: t->head, rewritten by the group selection
    (small ? k_tree_count<1> : k_tree_count<kBRows>)<<<(unsigned)ntiles, kBT, 0, s>>>(
        n, t->p.n_leaf, t->keys_sorted, ps->d_sys, t->head, wcount, tcount, nw, ntiles, R);
    FDPS_LAUNCH_CHECK(ctx);
    if (!small) {
        k_tree_scan<<<kMaxLevel, 1024, 0, s>>>(tcount, ntiles, ltot);
        FDPS_LAUNCH_CHECK(ctx);
    }
    const unsigned grid_nodes = (unsigned)(n / tile + 1);  // positions 0 .. n
    (small ? k_tree_nodes<1> : k_tree_nodes<kBRows>)<<<grid_nodes, kBT, 0, s>>>(
        n, ps->n_sys, t->cap_nodes, t->keys_sorted, ps->d_sys, t->head, wcount, tcount, nw, ntiles, ltot, t->st,
        t->nd_first, t->nd_count, t->nd_child, t->nd_meta, t->nd_parent, t->nd_qlo);
    FDPS_LAUNCH_CHECK(ctx);
    k_tree_finish<<<ctx->sm_count * 4, 256, 0, s>>>(t->st, ps->n_sys, t->nd_first, t->nd_count, t->nd_parent,
                                                    t->nd_child, t->nd_meta);
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

int selftest_barrier_timeout(fdps_ctx* ctx, uint32_t* flags_out) {
    uint32_t* w = nullptr;  // count, flags
    uint32_t h[2] = {0, 0};
    if (dev_alloc(ctx, &w, 2) != cudaSuccess) return set_error(ctx, FDPS_ENOMEM, "self-test allocation failed");
    cudaStream_t s = ctx->stream;
    cudaError_t e = cudaMemsetAsync(w, 0, sizeof(h), s);
    if (!e) {
        k_barrier_selftest<<<1, kMomBlock, 0, s>>>(w, w + 1, 1 << 12);
        ++ctx->launches;
        e = cudaGetLastError();
    }
    if (!e) e = cudaMemcpyAsync(h, w, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    cudaFree(w);
    if (e) return set_error(ctx, FDPS_ECUDA, "self-test failed: %s", cudaGetErrorString(e));
    *flags_out = h[1];
    return FDPS_OK;
}

int compute_moments(fdps_tree* t, fdps_psys* ps) {
    fdps_ctx* ctx = t->ctx;
    const int c = ps->cur;
    MomArgs A;
    A.st = t->st;
    A.box = t->sys_box;
    A.sys = ps->d_sys;
    A.px = ps->x[c];
    A.py = ps->y[c];
    A.pz = ps->z[c];
    A.pm = ps->m[c];
    A.pmx = t->pmx;
    A.pmy = t->pmy;
    A.pmz = t->pmz;
    A.pf_hi = t->pf_hi;
    A.pf_lo = t->pf_lo;
    A.nd_first = t->nd_first;
    A.nd_count = t->nd_count;
    A.nd_child = t->nd_child;
    A.nd_meta = t->nd_meta;
    A.nd_qlo = t->nd_qlo;
    A.nd_sx = t->nd_sx;
    A.nd_sy = t->nd_sy;
    A.nd_sz = t->nd_sz;
    A.nd_com = t->nd_com;
    A.nd_quad = t->nd_quad;
    A.nd_f = t->nd_f;
    A.nd_walk = t->nd_walk;
    A.nd_fq0 = t->nd_fq0;
    A.nd_fq1 = t->nd_fq1;
    if (t->p.moment != FDPS_QUADRUPOLE) return launch_moments<false, false>(ctx, A, ps->n, t->p.n_leaf, t->st);
    if (t->p.precision == FDPS_FP64) return launch_moments<true, true>(ctx, A, ps->n, t->p.n_leaf, t->st);
    return launch_moments<true, false>(ctx, A, ps->n, t->p.n_leaf, t->st);
}

int select_groups(fdps_tree* t, fdps_psys* ps) {
    fdps_ctx* ctx = t->ctx;
    cudaStream_t s = ctx->stream;
    const int64_t n = ps->n;
    const int c = ps->cur;
    const int G = t->box_blocks;
    if (n <= kGroupSmall && t->est_groups <= kGroupSmallGroups) {
        k_group_small<<<1, kGroupSmallBlock, 0, s>>>(t->st, t->p.n_grp, ps->n_sys, t->cap_groups, t->nd_first,
                                                     t->nd_count, t->nd_meta, t->nd_parent, t->head, t->g_node,
                                                     t->g_first, t->g_count);
        FDPS_LAUNCH_CHECK(ctx);
    } else {
        FDPS_CUDA_TRY(ctx, cudaMemsetAsync(t->head, 0xFF, sizeof(uint32_t) * (size_t)n, s));
        k_group_mark<<<ctx->sm_count * 8, 256, 0, s>>>(t->st, t->p.n_grp, ps->n_sys, t->nd_first, t->nd_count,
                                                       t->nd_meta, t->nd_parent, t->head);
        FDPS_LAUNCH_CHECK(ctx);
        k_group_count<<<G, kB, 0, s>>>(n, t->head, t->grp_scan, t->st, t->cap_groups);
        FDPS_LAUNCH_CHECK(ctx);
        k_group_write<<<G, kB, 0, s>>>(n, t->cap_groups, t->head, t->grp_scan, t->nd_count, t->g_node,
                                       t->g_first, t->g_count);
        FDPS_LAUNCH_CHECK(ctx);
    }
    k_group_data<<<ctx->sm_count * 8, 256, 0, s>>>(t->st, t->sys_box, ps->d_sys, t->g_first, t->g_count, ps->x[c],
                                                   ps->y[c], ps->z[c], t->g_box, t->g_qbox,
                                                   t->g_c64, t->g_ch, t->g_cl, t->g_blo, t->g_bhi);
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

}  // namespace fdps
