// short.cu -- the short-range mode: neighbour search over the same tree.
//
// FDPS treats an interaction as short-range when it has a cutoff and finds
// the neighbours by a tree traversal (Sect. 2.1.2, 3.2), for four kinds of
// cutoff: fixed, j-dependent, i-dependent and symmetric.  Particle j is a
// neighbour of i (i itself included) iff r^2 < c^2, with r^2 evaluated in
// FP64 as (dx*dx + dy*dy) + dz*dz, each operation rounded on its own, and
//   fixed: c = r_fixed;  i-dependent: c = h_i;  j-dependent: c = h_j;
//   symmetric: c = max(h_i, h_j).
// The workload on the neighbours is the SPH density with the Wendland C6
// kernel of the paper's SPH runs (Sect. 4.3): rho_i = sum_j m_j W(r, H),
// H = r_fixed, h_i or h_j, and for the symmetric cutoff the mean of
// W(r, h_i) and W(r, h_j).
//
// Per i-group, a warp walks the tree from the system's root and keeps every
// leaf that may hold a neighbour: a cell is opened iff the smallest distance
// between its grid cube and the group's grid box (an exact lower bound in
// grid units) is below the largest cutoff that can apply (r_fixed, the
// group's largest h, the cell's largest h, or both), with a relative margin
// so that no neighbour's leaf is ever dropped.  The pair pass then decides
// each candidate pair exactly: an FP32 evaluation on hi/lo parts with a
// bound on its error settles all but the pairs within the bound of the
// cutoff, which are decided by the FP64 operation sequence above.
#include <type_traits>

#include "fdps_internal.cuh"
#include "packed.cuh"

namespace fdps {
namespace {

constexpr int kSBlock = 128;
constexpr int kSW = kSBlock / 32;
constexpr int kSTile = 128;                 // candidate particles per shared tile (even)
constexpr unsigned long long kSChunk = 1ull << 16;
constexpr float kU = 5.9604645e-08f;      // 2^-24
// Wendland C6, 3D, support H: W = 1365 / (64 pi H^3) (1-q)^8 (1 + 8q + 25q^2 + 32q^3)
constexpr float kWc6 = 6.7889530f;        // 1365 / (64 pi)

__global__ void k_short_h(int64_t n, const uint32_t* __restrict__ id, const double* __restrict__ h_user,
                          double* __restrict__ h_sorted, uint32_t* flag) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const double h = h_user[id[p]];
        if (!(h > 0.0) || !(h < 1e300)) atomicOr(flag, 1u);
        h_sorted[p] = h;
    }
}

__global__ void k_hmax_leaves(int64_t nn, const uint32_t* __restrict__ meta, const uint32_t* __restrict__ first,
                              const uint32_t* __restrict__ count, const double* __restrict__ h,
                              double* __restrict__ hmax) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nn;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!((meta[i] >> 16) & 1u)) continue;
        double m = 0.0;
        for (uint32_t p = first[i]; p < first[i] + count[i]; ++p) m = h[p] > m ? h[p] : m;
        hmax[i] = m;
    }
}

__global__ void k_hmax_internal(int64_t a, int64_t b, const uint32_t* __restrict__ meta,
                                const uint32_t* __restrict__ child, double* __restrict__ hmax) {
    for (int64_t i = a + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < b;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t mt = meta[i];
        if ((mt >> 16) & 1u) continue;
        const uint32_t c0 = child[i], nc = (mt >> 8) & 0xFFu;
        double m = 0.0;
        for (uint32_t c = c0; c < c0 + nc; ++c) m = hmax[c] > m ? hmax[c] : m;
        hmax[i] = m;
    }
}

__global__ void k_group_hmax(int64_t ng, const uint32_t* __restrict__ first, const uint32_t* __restrict__ count,
                             const double* __restrict__ h, double* __restrict__ ghmax) {
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ng;
         g += (int64_t)gridDim.x * blockDim.x) {
        double m = 0.0;
        for (uint32_t p = first[g]; p < first[g] + count[g]; ++p) m = h[p] > m ? h[p] : m;
        ghmax[g] = m;
    }
}

struct ShortWalkArgs {
    DevState* st;
    const WalkRec* nd_walk;
    const double* nd_hmax;
    const uint32_t* g_qbox;
    const uint32_t* g_first;
    const double* g_hmax;
    const uint32_t* sys;
    const SysBox* box;
    unsigned long long* g_off;
    uint32_t* g_len;
    uint32_t* g_nepj;  // candidate particles per group
    uint32_t* pool;
    unsigned long long cap_pool;
    uint32_t* frontier;
    uint32_t cap_frontier;
    int mode;
    float r_fixed;
};

// cutoff bound for a cell (cell's largest h) and a group (group's largest h)
__device__ __forceinline__ float short_bound(int mode, float r_fixed, float hcell, float hgroup) {
    return mode == 0 ? r_fixed : mode == 1 ? hgroup : mode == 2 ? hcell : fmaxf(hcell, hgroup);
}

__global__ void __launch_bounds__(kSBlock) k_short_walk(ShortWalkArgs A) {
    DevState* st = A.st;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    uint32_t* fa = A.frontier + wid * 2 * (int64_t)A.cap_frontier;
    uint32_t* fb = fa + A.cap_frontier;
    const uint32_t F = A.cap_frontier;
    const uint32_t ngroups = (uint32_t)st->n_groups;
    unsigned long long cursor = 0, chunk_end = 0, acc_entries = 0, acc_cand = 0;
    bool ovf = false;
    for (;;) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(&st->walk_counter, 1u);
        g = __shfl_sync(0xFFFFFFFFu, g, 0);
        if (g >= ngroups) break;
        const uint32_t sysid = A.sys ? A.sys[A.g_first[g]] : 0u;
        // cutoffs are compared in units of the grid spacing (its square need
        // not be a normal FP32 number)
        const float idq = 1.0f / (float)(A.box[sysid].L * (1.0 / 2097152.0));
        const uint32_t* qb = A.g_qbox + 6 * (int64_t)g;
        const uint32_t qmin0 = qb[0], qmin1 = qb[1], qmin2 = qb[2];
        const uint32_t qmax0 = qb[3], qmax1 = qb[4], qmax2 = qb[5];
        const float hg = A.g_hmax ? (float)A.g_hmax[g] : 0.f;
        unsigned long long gstart = cursor;
        uint32_t cand_lane = 0;
        uint32_t fsize = 1;
        if (lane == 0) fa[0] = sysid;
        __syncwarp();
        while (fsize > 0) {
            uint32_t nsize = 0;
            // node records (and the cells' radii) one batch ahead, frontier
            // ids two batches ahead, so that no batch waits on a load that
            // depends on another load
            uint32_t node_nx = lane < fsize ? fa[lane] : 0u;
            uint32_t node_nx2 = lane + 32 < fsize ? fa[lane + 32] : 0u;
            uint4 rec_nx = make_uint4(0, 0, 0, 0);
            float hc_nx = 0.f;
            if (lane < fsize) {
                rec_nx = A.nd_walk[node_nx].r;
                if (A.mode >= 2) hc_nx = (float)A.nd_hmax[node_nx];
            }
            for (uint32_t base = 0; base < fsize; base += 32) {
                const uint32_t idx = base + lane;
                const bool act = idx < fsize;
                const uint32_t node = node_nx;
                const uint4 rec = rec_nx;
                const float hc = hc_nx;
                if (idx + 32 < fsize) {
                    node_nx = node_nx2;
                    rec_nx = A.nd_walk[node_nx].r;
                    if (A.mode >= 2) hc_nx = (float)A.nd_hmax[node_nx];
                }
                if (idx + 64 < fsize) node_nx2 = fa[idx + 64];
                bool emit = false;
                uint32_t nch = 0, child = 0;
                if (act) {
                    const int level = (int)((rec.x >> 21) & 31u);
                    const bool leaf = (rec.x >> 26) & 1u;
                    const uint32_t w = (1u << (kMaxLevel - level)) - 1u;
                    const uint32_t qx = rec.x & kQMax, qy = rec.y, qz = rec.z;
                    // gaps between [q, q + w + 1) and [qmin, qmax + 1) in grid units
                    const float gx = (float)max(0, max((int)qx - (int)(qmax0 + 1), (int)qmin0 - (int)(qx + w + 1)));
                    const float gy = (float)max(0, max((int)qy - (int)(qmax1 + 1), (int)qmin1 - (int)(qy + w + 1)));
                    const float gz = (float)max(0, max((int)qz - (int)(qmax2 + 1), (int)qmin2 - (int)(qz + w + 1)));
                    const float d2 = gx * gx + gy * gy + gz * gz;
                    const float R = short_bound(A.mode, A.r_fixed, hc, hg) * idq;
                    // margin: FP32 rounding of the bound and of the gaps (a NaN,
                    // where a radius or the spacing is 0 or infinite in FP32,
                    // keeps the cell: the pairs are decided one by one)
                    const bool near = !(d2 > R * R * (1.0f + 64.0f * kU));
                    if (near) {
                        if (leaf) {
                            emit = true;
                            cand_lane += rec.w;
                        } else {
                            nch = rec.x >> 27;
                            child = rec.w;
                        }
                    }
                }
                const uint32_t emask = __ballot_sync(0xFFFFFFFFu, emit);
                const uint32_t k = __popc(emask);
                if (k) {
                    if (cursor + k > chunk_end) {
                        const unsigned long long sofar = cursor - gstart;
                        const unsigned long long want = 2 * (sofar + k) > kSChunk ? 2 * (sofar + k) : kSChunk;
                        unsigned long long nb = 0;
                        if (lane == 0) nb = atomicAdd(&st->pool_cursor, want);
                        nb = __shfl_sync(0xFFFFFFFFu, nb, 0);
                        if (!ovf && nb + want > A.cap_pool) {
                            if (lane == 0) atomicOr(&st->overflow, kOvfPool);
                            ovf = true;
                        }
                        if (!ovf) {
                            for (unsigned long long j = lane; j < sofar; j += 32) A.pool[nb + j] = A.pool[gstart + j];
                            __syncwarp();
                            gstart = nb;
                            cursor = nb + sofar;
                            chunk_end = nb + want;
                        } else {
                            chunk_end = ~0ull;
                        }
                    }
                    if (emit && !ovf) A.pool[cursor + __popc(emask & lt)] = node | kLeafTag;
                    cursor += k;
                }
                if (__ballot_sync(0xFFFFFFFFu, nch > 0u)) {  // deep in the tree most batches open none
                    uint32_t inc = nch;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const uint32_t tv = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                        if (lane >= off) inc += tv;
                    }
                    const uint32_t tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
                    if (nsize + tot > F) {
                        if (lane == 0) atomicOr(&st->overflow, kOvfFrontier);
                        ovf = true;
                    } else {
                        // at most 8 stores off one address
                        uint32_t* f = fb + (nsize + inc - nch);
#pragma unroll
                        for (uint32_t c = 0; c < 8; ++c)
                            if (c < nch) f[c] = child + c;
                        nsize += tot;
                    }
                }
            }
            __syncwarp();
            uint32_t* tmp = fa;
            fa = fb;
            fb = tmp;
            fsize = nsize;
        }
        const uint32_t cand = __reduce_add_sync(0xFFFFFFFFu, cand_lane);
        const unsigned long long len = cursor - gstart;
        if (lane == 0) {
            A.g_off[g] = gstart;
            A.g_len[g] = (uint32_t)len;
            A.g_nepj[g] = cand;
        }
        acc_entries += len;
        acc_cand += cand;
    }
    if (lane == 0) {
        atomicAdd(&st->pool_needed, acc_entries);
        atomicAdd(&st->list_entries, acc_entries);
        atomicAdd(&st->n_epj, acc_cand);
    }
}

struct ShortPairArgs {
    DevState* st;
    const uint32_t* g_first;
    const uint32_t* g_count;
    const unsigned long long* g_off;
    const uint32_t* g_len;
    const uint32_t* pool;
    const uint32_t* nd_first;
    const uint32_t* nd_count;
    const float4* pf_hi;  // (x hi - c0, y, z, m)
    const float4* pf_lo;  // (x lo, y lo, z lo, eps^2)
    const double* x;      // FP64 positions in key order
    const double* y;
    const double* z;
    const float4* g_ch;   // group centre (hi - c0, lo) and box relative to it
    const float4* g_cl;
    const float4* g_blo;
    const float4* g_bhi;
    const uint32_t* g_nepj;  // candidates in the group's list
    const double* g_hmax;    // largest cutoff radius of a group (i-dependent and symmetric types)
    const double* h;      // cutoff radii in key order (null for the fixed type)
    const uint32_t* id;   // key order -> caller's row
    const uint32_t* sys;
    const SysBox* box;
    uint32_t* count;      // caller order
    double* rho;
    unsigned long long* info;  // neighbour pairs, candidate pairs, FP64 decisions
    double r_fixed;
};

// (1 - q)^8 (1 + 8 q + 25 q^2 + 32 q^3) of two candidates at q^2 = x = r2 / H^2
// (the Wendland C6 kernel without its normalisation).  nih2 = -1 / H^2.  The
// root is s = x y, y the reciprocal root, with one Newton correction
// s + (x - s^2) y / 2 (Heron's iteration), evaluated as -q from -x so that
// nothing needs a change of sign; x is kept from 0 by 1e-30 (q = 0 to every
// digit of the result).  CLAMP: x may be anything, and the result is 0 from
// q = 1 on; otherwise x is at most 2e4 (the result then stays finite, and is
// read for q <= 1 + 1e-5 only, where (1 - q)^8 vanishes from q = 1 on).
template <bool CLAMP>
__device__ __forceinline__ f2 wendland_q2(f2 r2, f2 nih2) {
    f2 nx = f2_fma(r2, nih2, f2_pk(-1e-30f, -1e-30f));
    float a, b;
    f2_up(nx, a, b);
    if (CLAMP) {
        a = fmaxf(a, -4.0f);
        b = fmaxf(b, -4.0f);
        nx = f2_pk(a, b);
    }
    const f2 y = f2_pk(rsqrt_normal(-a), rsqrt_normal(-b));
    const f2 ns = f2_mul(nx, y), hy = f2_mul(y, f2_pk(0.5f, 0.5f));
    const f2 nq = f2_fma(f2_fma(ns, ns, nx), hy, ns);
    f2 u = f2_add(f2_pk(1.0f, 1.0f), nq);
    if (CLAMP) {
        f2_up(u, a, b);
        u = f2_pk(fmaxf(a, 0.0f), fmaxf(b, 0.0f));
    }
    const f2 u2 = f2_mul(u, u), u4 = f2_mul(u2, u2), u8 = f2_mul(u4, u4);
    const f2 p = f2_fma(nq, f2_fma(nq, f2_fma(nq, f2_pk(-32.0f, -32.0f), f2_pk(25.0f, 25.0f)), f2_pk(-8.0f, -8.0f)),
                        f2_pk(1.0f, 1.0f));
    return f2_mul(u8, p);
}

// Two thresholds on r^2 that decide the pairs of a cutoff c: r^2 < lo is a
// neighbour, r^2 > hi is none, between them the FP64 sequence decides.  With
// a = max |d|, Ea = 8u a + Eabs the error of a difference and M = 8u (r^2 +
// c^2) + 6 a Ea + 3 Ea^2 the bound on the error of r^2 - c^2: M <= Mmax for
// r^2 <= c^2 (a <= r <= c), and for r^2 > c^2, with a <= r <= (r^2 + c^2) /
// (2c), M <= (56u + 192u^2 + beta) r^2 + (8u + beta) c^2 + 3 Eabs^2, beta =
// 3 Eabs / c (slack for the FP32 evaluation of both).  A cutoff within a few
// Eabs sends every pair to the FP64 sequence, and so does one whose square's
// roundings come near the spacing of subnormal numbers (1.4e-45 against M >= 64u
// c^2 = 4e-40 from 1e-17 on).
__device__ __forceinline__ float2 pair_thresholds(float c, float Eabs) {
    const float c2 = c * c, beta = 3.0001f * Eabs / c;
    if (!(beta < 0.25f) || c < 1e-17f) return make_float2(-INFINITY, INFINITY);
    const float tq = fmaf(8.0f * kU, c, Eabs);
    const float Mmax = 64.0f * kU * c2 + 6.0f * c * Eabs + 3.0f * tq * tq;
    return make_float2(c2 - (1.01f * Mmax + 4.0f * kU * c2),
                       (c2 * (1.0f + 8.0f * kU + beta) + 3.0f * Eabs * Eabs) * (1.0f + 16.0f * kU) /
                           (1.0f - (56.0f * kU + 192.0f * kU * kU + beta)));
}

// A warp's tile of candidates; pairs (2 k, 2 k + 1) are read as one packed
// register.  R: with the candidates' own radii (j-dependent types).
template <bool R>
struct PairTile {
    float xh[kSTile], yh[kSTile], zh[kSTile], xl[kSTile], yl[kSTile], zl[kSTile], m[kSTile];
    uint32_t p[kSTile];
    float nih2[R ? kSTile : 2];            // -1 / h_j^2
    float mw[R ? kSTile : 2];              // m_j times the kernel's normalisation for h_j
    float lo[R ? kSTile : 2], hi[R ? kSTile : 2], hj[R ? kSTile : 2];
};
__device__ __forceinline__ f2 ld2(const float* a, uint32_t k) { return reinterpret_cast<const f2*>(a)[k]; }

// One warp per group.  The candidates of the group's list are tested against
// the group's box (no nearer to any of its particles than to the box) and
// only those within the largest cutoff that can apply are staged: of 3.4
// candidates a neighbour (310 neighbours in a uniform cube, groups of 8)
// the walk's leaves give, about 2 remain.  Lanes: P i-slots x nsl slices
// of the tile, so that small groups keep the whole warp busy; a lane takes
// two candidates at a time in packed FP32 instructions.  Where the cutoff is
// the i-particle's own and the group's box is at most half of it (nearly
// always: the groups of a uniform cube are a quarter of it), the kernel's
// argument is bounded and needs no clamps.  MODE is the cutoff type (FDPS_CUTOFF_*), fixed at compile time so
// that the pair loop carries no selection between them.  Issue-bound (78 % of
// the slots, ALU 61 %): pair pass of 2^20 particles 3.19 ms with one candidate a
// turn and no box test, 2.18 with them, 1.97 with a candidate's leaf from
// ballots, 1.78 without the clamps and with tiles of 128 (96 before).  FP32
// coordinates relative to the group's centre instead of the hi/lo pairs took
// 1.64, but a separation was then off by up to 10u of the cutoff instead of a
// few u of itself, and the density errors grew by up to 1 %: not taken.
template <int MODE>
__global__ void __launch_bounds__(kSBlock, 8) k_short_pairs(ShortPairArgs A) {
    constexpr bool R = MODE >= 2;
    __shared__ __align__(16) PairTile<R> s_t[kSW];
    DevState* st = A.st;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    PairTile<R>& T = s_t[w];
    const uint32_t ngroups = (uint32_t)st->n_groups;
    unsigned long long n_pairs = 0, n_cand = 0, n_fb = 0;
    for (;;) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(&st->force_counter, 1u);
        g = __shfl_sync(0xFFFFFFFFu, g, 0);
        if (g >= ngroups) break;
        const uint32_t gf = A.g_first[g], ni = A.g_count[g];
        const unsigned long long off = A.g_off[g];
        const uint32_t len = A.g_len[g];
        const float L = (float)A.box[A.sys ? A.sys[gf] : 0u].L;
        const float Eabs = 1e-13f * L;  // error of the FP64 -> FP32 hi/lo parts
        const float4 gch = A.g_ch[g], gcl = A.g_cl[g], blo = A.g_blo[g], bhi = A.g_bhi[g];
        // the box as half-widths about its centre (as in the gravity walk)
        const float hx = fmaxf(-blo.x, bhi.x), hy = fmaxf(-blo.y, bhi.y), hz = fmaxf(-blo.z, bhi.z);
        const float hb = fmaxf(hx, fmaxf(hy, hz));
        // what a cutoff grows by so that the FP32 distance to the box never
        // drops a pair that the thresholds or the FP64 sequence look at: the
        // distance's error is below 4u (C + 2 hb) + 2 Eabs; squares are compared
        // from 1e-34 on, far above the subnormal numbers
        const float pad = 64.0f * kU * hb + 16.0f * Eabs;
        const float hg = MODE == 0 ? (float)A.r_fixed : MODE == 2 ? 0.0f : (float)A.g_hmax[g];
        const uint32_t P = ni <= 16u ? ni : 32u;
        const uint32_t nsl = 32u / P;
        const uint32_t ip = lane % P, sl = lane / P;
        for (uint32_t ib = 0; ib < ni; ib += P) {
            const uint32_t i = ib + ip;
            const bool act = sl < nsl && i < ni;
            const uint32_t pi = gf + (act ? i : 0u);
            const float4 ih = A.pf_hi[pi], il = A.pf_lo[pi];
            const double hi64 = MODE != 0 ? A.h[pi] : A.r_fixed;
            const float hif = (float)hi64, invHi = 1.0f / hif, invHi2 = fminf(invHi * invHi, 3e38f);
            // no staged candidate is further than 137 of the lane's cutoffs
            const bool bounded = !R && __all_sync(0xFFFFFFFFu, !act || (hb <= 0.5f * hif && hg <= 8.0f * hif && hif > 1e-17f && hif < 1e17f));
            const float2 ti = MODE == 2 ? make_float2(0.0f, 0.0f)
                                        : pair_thresholds(hif, Eabs);
            const f2 ixh = f2_pk(ih.x, ih.x), iyh = f2_pk(ih.y, ih.y), izh = f2_pk(ih.z, ih.z);
            const f2 ixl = f2_pk(il.x, il.x), iyl = f2_pk(il.y, il.y), izl = f2_pk(il.z, il.z);
            const f2 niH2 = f2_pk(-invHi2, -invHi2);
            uint32_t cnt = 0, fbk = 0;
            f2 sum = 0ull, sumj = 0ull;  // sums of m_j w(q) with H = h_i, and with H = h_j
            // the staged candidates 0 .. m - 1 on the warp's i-particles
            auto pairs = [&](auto clamp, uint32_t m) {
                constexpr bool CLAMP = decltype(clamp)::value;
                if ((m & 1u) && lane == 0) {  // an even number: a candidate far from everything, without mass
                    const float far = 16.0f * (hb + hg) + (R ? 16.0f * T.hj[m - 1] : 0.0f);
                    // (as a low part: a few cutoffs may be lost in a sum with the
                    // centre's coordinate)
                    T.xh[m] = gch.x;
                    T.yh[m] = gch.y;
                    T.zh[m] = gch.z;
                    T.xl[m] = far;
                    T.yl[m] = T.zl[m] = T.m[m] = 0.0f;
                    T.p[m] = 0xFFFFFFFFu;
                    if (R) {
                        T.nih2[m] = T.nih2[m - 1];
                        T.mw[m] = 0.0f;
                        T.lo[m] = T.lo[m - 1];
                        T.hi[m] = T.hi[m - 1];
                        T.hj[m] = T.hj[m - 1];
                    }
                }
                __syncwarp();
                if (act) {
#pragma unroll 1
                    for (uint32_t k = sl; k < (m + 1u) / 2u; k += nsl) {
                        const f2 dx = f2_add(f2_sub(ld2(T.xh, k), ixh), f2_sub(ld2(T.xl, k), ixl));
                        const f2 dy = f2_add(f2_sub(ld2(T.yh, k), iyh), f2_sub(ld2(T.yl, k), iyl));
                        const f2 dz = f2_add(f2_sub(ld2(T.zh, k), izh), f2_sub(ld2(T.zl, k), izl));
                        const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
                        float ra, rb;
                        f2_up(r2, ra, rb);
                        float la = ti.x, lb = ti.x, ua = ti.y, ub = ti.y;
                        if (R) {
                            f2_up(ld2(T.lo, k), la, lb);
                            f2_up(ld2(T.hi, k), ua, ub);
                        }
                        if (MODE == 3) {  // the larger radius of the pair
                            float ha, hc;
                            f2_up(ld2(T.hj, k), ha, hc);
                            la = hif >= ha ? ti.x : la;
                            ua = hif >= ha ? ti.y : ua;
                            lb = hif >= hc ? ti.x : lb;
                            ub = hif >= hc ? ti.y : ub;
                        }
                        bool na = ra < la, nb = rb < lb;
                        const bool fa = !na && !(ra > ua), fb = !nb && !(rb > ub);
                        if (fa || fb) {  // inside the bound: the exact FP64 sequence
                            for (int c = 0; c < 2; ++c) {
                                const uint32_t pj = T.p[2 * k + c];
                                if (!(c ? fb : fa) || pj == 0xFFFFFFFFu) continue;
                                ++fbk;
                                const double ex = __dsub_rn(A.x[pj], A.x[pi]);
                                const double ey = __dsub_rn(A.y[pj], A.y[pi]);
                                const double ez = __dsub_rn(A.z[pj], A.z[pi]);
                                const double e2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)),
                                                            __dmul_rn(ez, ez));
                                const double hj64 = MODE != 0 ? A.h[pj] : A.r_fixed;
                                const double cc = MODE == 0 ? A.r_fixed
                                                : MODE == 1 ? hi64
                                                : MODE == 2 ? hj64
                                                            : (hi64 > hj64 ? hi64 : hj64);
                                (c ? nb : na) = e2 < __dmul_rn(cc, cc);
                            }
                        }
                        // the kernel for every candidate, kept for the
                        // neighbours only: half of the staged candidates
                        // are, so a branch would be taken by some lane of
                        // nearly every turn anyway
                        cnt += (na ? 1u : 0u) + (nb ? 1u : 0u);
                        if (MODE != 2) {
                            float ma, mb;
                            f2_up(ld2(T.m, k), ma, mb);
                            sum = f2_fma(f2_pk(na ? ma : 0.0f, nb ? mb : 0.0f), wendland_q2<CLAMP>(r2, niH2), sum);
                        }
                        if (R) {
                            float ma, mb;
                            f2_up(ld2(T.mw, k), ma, mb);
                            sumj = f2_fma(f2_pk(na ? ma : 0.0f, nb ? mb : 0.0f),
                                          wendland_q2<true>(r2, ld2(T.nih2, k)), sumj);
                        }
                    }
                }
                __syncwarp();
            };
            auto run = [&](uint32_t m) {
                if constexpr (!R) {
                    if (bounded) return pairs(std::false_type{}, m);
                }
                pairs(std::true_type{}, m);
            };
            uint32_t staged = 0;
            for (uint32_t base = 0; base < len; base += 32) {
                // leaves of this step: particle counts and offsets
                const uint32_t u = base + lane;
                const uint32_t node = u < len ? (A.pool[off + u] & ~kLeafTag) : 0u;
                const uint32_t c = u < len ? A.nd_count[node] : 0u;
                uint32_t inc = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t tv = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                    if (lane >= o) inc += tv;
                }
                const uint32_t total = __shfl_sync(0xFFFFFFFFu, inc, 31);
                const uint32_t first = u < len ? A.nd_first[node] : 0u;
                const uint32_t start = inc - c;
                for (uint32_t c0 = 0; c0 < total; c0 += 32) {
                    const uint32_t item = c0 + lane;
                    // the leaf of each item (none is empty): the leaves that
                    // start before these 32 items, and among them as bits
                    const uint32_t before = __popc(__ballot_sync(0xFFFFFFFFu, c > 0u && start < c0));
                    const uint32_t bits = __reduce_or_sync(
                        0xFFFFFFFFu, c > 0u && start >= c0 && start < c0 + 32u ? 1u << (start - c0) : 0u);
                    const int src = (int)(before + __popc(bits & (lt | (1u << lane)))) - 1;
                    const uint32_t pj = __shfl_sync(0xFFFFFFFFu, first, src) +
                                        (item - __shfl_sync(0xFFFFFFFFu, start, src));
                    bool keep = false;
                    float4 h4 = make_float4(0.f, 0.f, 0.f, 0.f), l4 = h4;
                    float dx = 0.0f, dy = 0.0f, dz = 0.0f;
                    float hj = 0.0f;
                    if (item < total) {
                        h4 = A.pf_hi[pj];
                        l4 = A.pf_lo[pj];
                        if (R) hj = (float)A.h[pj];
                        dx = (h4.x - gch.x) + (l4.x - gcl.x);
                        dy = (h4.y - gch.y) + (l4.y - gcl.y);
                        dz = (h4.z - gch.z) + (l4.z - gcl.z);
                        const float tx = fmaxf(fabsf(dx) - hx, 0.0f), ty = fmaxf(fabsf(dy) - hy, 0.0f),
                                    tz = fmaxf(fabsf(dz) - hz, 0.0f);
                        const float C = fmaf(fmaxf(hg, hj), 1.0f + 256.0f * kU, pad);
                        keep = !(fmaf(tx, tx, fmaf(ty, ty, tz * tz)) > fmaxf(C * C, 1e-34f));
                    }
                    const uint32_t mask = __ballot_sync(0xFFFFFFFFu, keep);
                    if (keep) {
                        const uint32_t k = staged + __popc(mask & lt);
                        T.xh[k] = h4.x;
                        T.yh[k] = h4.y;
                        T.zh[k] = h4.z;
                        T.xl[k] = l4.x;
                        T.yl[k] = l4.y;
                        T.zl[k] = l4.z;
                        T.m[k] = h4.w;
                        T.p[k] = pj;
                        if (R) {
                            const float ihj = 1.0f / hj;
                            const float2 tj = pair_thresholds(hj, Eabs);
                            T.nih2[k] = -fminf(ihj * ihj, 3e38f);
                            T.mw[k] = h4.w * (kWc6 * ihj * ihj * ihj);
                            T.lo[k] = tj.x;
                            T.hi[k] = tj.y;
                            T.hj[k] = hj;
                        }
                    }
                    staged += __popc(mask);
                    if (staged > (uint32_t)kSTile - 33u) {  // room for the next 32 and the padding
                        run(staged);
                        staged = 0;
                    }
                }
            }
            if (staged) run(staged);
            // the lane's two halves and the slices' partial counts and sums,
            // into the first slice
            float sa, sb, ja, jb;
            f2_up(sum, sa, sb);
            f2_up(sumj, ja, jb);
            const float norm = kWc6 * invHi * invHi * invHi;
            const float rho = MODE == 2   ? ja + jb
                              : MODE == 3 ? 0.5f * fmaf(norm, sa + sb, ja + jb)
                                          : norm * (sa + sb);
            uint32_t cnt_all = cnt;
            float sum_all = rho;
            for (uint32_t q = 1; q < nsl; ++q) {
                const int src = (int)((ip + q * P) & 31u);
                cnt_all += __shfl_sync(0xFFFFFFFFu, cnt, src);
                sum_all += __shfl_sync(0xFFFFFFFFu, rho, src);
            }
            if (act && sl == 0) {
                const uint32_t row = A.id[pi];
                A.count[row] = cnt_all;
                A.rho[row] = (double)sum_all;
                n_cand += A.g_nepj[g];
            }
            n_pairs += act ? cnt : 0u;
            n_fb += act ? fbk : 0u;
        }
    }
    // per-warp totals
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n_pairs += __shfl_xor_sync(0xFFFFFFFFu, n_pairs, o);
        n_cand += __shfl_xor_sync(0xFFFFFFFFu, n_cand, o);
        n_fb += __shfl_xor_sync(0xFFFFFFFFu, n_fb, o);
    }
    if (lane == 0 && A.info) {
        atomicAdd(&A.info[0], n_pairs);
        atomicAdd(&A.info[1], n_cand);
        atomicAdd(&A.info[2], n_fb);
    }
}

}  // namespace

int short_prepare(fdps_tree* t, fdps_psys* ps, int mode, const double* h_user) {
    fdps_ctx* ctx = t->ctx;
    cudaStream_t s = ctx->stream;
    const int64_t n = ps->n;
    if (mode == 0) return FDPS_OK;  // the fixed cutoff needs no radii
    if (t->cap_sr_h < n) {
        dev_free(t->sr_h);
        t->cap_sr_h = 0;
        if (dev_alloc(ctx, &t->sr_h, n) != cudaSuccess) {
            cudaGetLastError();
            return set_error(ctx, FDPS_ENOMEM, "cutoff radii allocation failed");
        }
        t->cap_sr_h = n;
    }
    FDPS_CUDA_TRY(ctx, cudaMemsetAsync(ps->d_flag, 0, sizeof(uint32_t), s));
    k_short_h<<<grid_for(n, 256, 4 * ctx->sm_count), 256, 0, s>>>(n, ps->id[ps->cur], h_user, t->sr_h, ps->d_flag);
    FDPS_LAUNCH_CHECK(ctx);
    uint32_t bad = 0;
    FDPS_CUDA_TRY(ctx, cudaMemcpyAsync(&bad, ps->d_flag, sizeof(bad), cudaMemcpyDeviceToHost, s));
    FDPS_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    if (bad) return set_error(ctx, FDPS_EINVAL, "cutoff radii must be positive and finite");
    // (the state word was read after the tree stages)
    const int64_t nn = t->h_st.n_nodes, ng = t->h_st.n_groups;
    if (t->cap_nd_hmax < nn) {
        dev_free(t->nd_hmax);
        t->cap_nd_hmax = 0;
        if (dev_alloc(ctx, &t->nd_hmax, t->cap_nodes) != cudaSuccess) {
            cudaGetLastError();
            return set_error(ctx, FDPS_ENOMEM, "node radii allocation failed");
        }
        t->cap_nd_hmax = t->cap_nodes;
    }
    if (t->cap_g_hmax < ng) {
        dev_free(t->g_hmax);
        t->cap_g_hmax = 0;
        if (dev_alloc(ctx, &t->g_hmax, t->cap_groups) != cudaSuccess) {
            cudaGetLastError();
            return set_error(ctx, FDPS_ENOMEM, "group radii allocation failed");
        }
        t->cap_g_hmax = t->cap_groups;
    }
    if (mode >= 2) {  // the cells' largest radii bound the j-dependent cutoffs only
        k_hmax_leaves<<<grid_for(nn, 256, 4 * ctx->sm_count), 256, 0, s>>>(nn, t->nd_meta, t->nd_first,
                                                                          t->nd_count, t->sr_h, t->nd_hmax);
        FDPS_LAUNCH_CHECK(ctx);
        for (int l = t->h_st.max_level - 1; l >= 0; --l) {
            const int64_t a = t->h_st.lvl_start[l], b = t->h_st.lvl_start[l + 1];
            if (b <= a) continue;
            k_hmax_internal<<<grid_for(b - a, 256, 4 * ctx->sm_count), 256, 0, s>>>(a, b, t->nd_meta,
                                                                                   t->nd_child, t->nd_hmax);
            FDPS_LAUNCH_CHECK(ctx);
        }
    }
    k_group_hmax<<<grid_for(ng, 256, 4 * ctx->sm_count), 256, 0, s>>>(ng, t->g_first, t->g_count, t->sr_h,
                                                                      t->g_hmax);
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

int launch_short_walk(fdps_tree* t, fdps_psys* ps, int mode, double r_fixed, int blocks) {
    fdps_ctx* ctx = t->ctx;
    ShortWalkArgs A;
    A.st = t->st;
    A.nd_walk = t->nd_walk;
    A.nd_hmax = mode >= 2 ? t->nd_hmax : nullptr;
    A.g_qbox = t->g_qbox;
    A.g_first = t->g_first;
    A.g_hmax = (mode == 1 || mode == 3) ? t->g_hmax : nullptr;
    A.sys = ps->d_sys;
    A.box = t->sys_box;
    A.g_off = t->g_off;
    A.g_len = t->g_len;
    A.g_nepj = t->g_nepj;
    A.pool = t->pool;
    A.cap_pool = (unsigned long long)t->cap_pool;
    A.frontier = t->frontier;
    A.cap_frontier = (uint32_t)t->cap_frontier;
    A.mode = mode;
    A.r_fixed = (float)r_fixed;
    k_short_walk<<<blocks, kSBlock, 0, ctx->stream>>>(A);
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

int launch_short_pairs(fdps_tree* t, fdps_psys* ps, int mode, double r_fixed, uint32_t* count, double* rho,
                       unsigned long long* info3) {
    fdps_ctx* ctx = t->ctx;
    const int c = ps->cur;
    ShortPairArgs A;
    A.st = t->st;
    A.g_first = t->g_first;
    A.g_count = t->g_count;
    A.g_off = t->g_off;
    A.g_len = t->g_len;
    A.pool = t->pool;
    A.nd_first = t->nd_first;
    A.nd_count = t->nd_count;
    A.pf_hi = t->pf_hi;
    A.pf_lo = t->pf_lo;
    A.x = ps->x[c];
    A.y = ps->y[c];
    A.z = ps->z[c];
    A.g_ch = t->g_ch;
    A.g_cl = t->g_cl;
    A.g_blo = t->g_blo;
    A.g_bhi = t->g_bhi;
    A.g_nepj = t->g_nepj;
    A.g_hmax = (mode == 1 || mode == 3) ? t->g_hmax : nullptr;
    A.h = mode == 0 ? nullptr : t->sr_h;
    A.id = ps->id[c];
    A.sys = ps->d_sys;
    A.box = t->sys_box;
    A.count = count;
    A.rho = rho;
    A.info = info3;
    A.r_fixed = r_fixed;
    void (*kern)(ShortPairArgs) = mode == 0 ? k_short_pairs<0> : mode == 1 ? k_short_pairs<1>
                                : mode == 2 ? k_short_pairs<2> : k_short_pairs<3>;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSBlock, 0) != cudaSuccess || per_sm < 1)
        per_sm = 4;
    kern<<<per_sm * ctx->sm_count, kSBlock, 0, ctx->stream>>>(A);
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

}  // namespace fdps
