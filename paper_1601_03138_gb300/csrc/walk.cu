// walk.cu -- interaction lists: one warp walks the tree for one i-group (one
// block in systems of few groups).
//
// The Barnes-Hut traversal with a fixed opening angle (Sect. 3.2), done
// once per i-group as in the modified tree algorithm of Barnes (1990) that
// the paper's cost model uses (Sect. 5.5, T_icalc,const).  The paper does
// not state the criterion; this library opens a cell C for group G iff
//   (a) C's grid cube meets G's grid box (closed integer intervals of the
//       quantised coordinates), or
//   (b) ell_C^2 >= theta^2 d^2, ell_C = L 2^-level, d = distance from C's
//       centre of mass to G's FP64 bounding box,
// and evaluates (b) as FP64 with each operation rounded on its own, in a
// fixed order.  The same FP64 decision is reproduced here at FP32 cost: the
// test is first evaluated in FP32 on double-float (hi + lo) copies of the
// positions relative to the group centre, with a rigorous bound on the
// FP32 error; only tests that land inside that bound are re-evaluated with
// the exact FP64 operation sequence.
//
// Traversal is breadth-first per warp: 32 cells of the current frontier are
// tested at a time; opened internal cells push their children (contiguous
// ids) to the next frontier, opened leaves append one EPJ entry (node id
// with bit 31 set: all of the leaf's particles), unopened cells one SPJ
// entry.  A group's list is contiguous in a pool handed out in chunks of at
// least 2^16 entries, its SPJ entries first and its leaves after them (they
// collect at the chunk's end and move down once the group is done), so that
// the force kernel stages superparticles and leaf particles without sorting
// them apart; when a chunk fills, the group's partial list moves to a fresh
// chunk twice its length.  Overflow of the pool or of the frontier sets a flag; the
// host then grows the buffer and repeats the walk.
#include "fdps_internal.cuh"

namespace fdps {

struct WalkArgs {
    DevState* st;
    const WalkRec* nd_walk;
    const float4* nd_f;    // COM hi/lo pairs per node
    const dvec4* nd_com;
    const uint32_t* g_count;
    const uint32_t* g_first;
    const uint32_t* sys;  // system of each particle position (null: one system)
    const SysBox* box;    // root box of each system
    const uint32_t* g_qbox;
    const double* g_box;
    const float4* g_ch;
    const float4* g_cl;
    const float4* g_blo;
    const float4* g_bhi;
    unsigned long long* g_off;
    uint32_t* g_len;
    uint32_t* g_nspj;
    uint32_t* g_nepj;
    uint32_t* pool;
    unsigned long long cap_pool;
    uint32_t* frontier;
    uint32_t cap_frontier;
    double theta2;
    float theta2f;
};

namespace {

constexpr unsigned long long kChunk = 1ull << 16;
constexpr float kU32 = 5.9604645e-08f;  // 2^-24, unit roundoff of FP32

__device__ __forceinline__ unsigned long long shfl_u64(unsigned long long v, int src) {
    return __shfl_sync(0xFFFFFFFFu, v, src);
}

// Exact FP64 opening test (b): the reference sequence of operations.
__device__ __forceinline__ bool open_fp64(double L, int level, double theta2, const dvec4 com,
                                       const double* box) {
    const double ell = ldexp(L, -level);
    const double c[3] = {com.x, com.y, com.z};
    double d2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double below = __dsub_rn(box[a], c[a]);
        const double above = __dsub_rn(c[a], box[3 + a]);
        const double da = below > 0.0 ? below : (above > 0.0 ? above : 0.0);
        d2 = __dadd_rn(d2, __dmul_rn(da, da));
    }
    return __dmul_rn(ell, ell) >= __dmul_rn(theta2, d2);
}

// What a warp carries from one group's walk to the next: its pool chunk
// and its totals for the device state word.  Every field but the total is
// the same in all lanes; lane k holds total k (list entries, EPJ, SPJ, EPJ and
// SPJ interactions).
struct WalkState {
    uint32_t* cptr;            // start of the warp's pool chunk
    uint32_t coff, clen;       // cursor and length within it
    bool ovf;
    unsigned long long total;
    uint32_t max_front;
};

__device__ __forceinline__ WalkState walk_state_init() {
    WalkState S;
    S.cptr = nullptr;
    S.coff = S.clen = 0;
    S.ovf = false;
    S.total = 0;
    S.max_front = 0;
    return S;
}


// What the opening tests of one group read: its grid box, its centre and its
// box about it in FP32, its system's root box size.  The box is kept as
// half-widths h, the larger side of each axis; the two sides differ by the
// roundings of the centre and of the corners, and the largest difference
// (exact: the parts nearly cancel) joins the error of a coordinate.
struct GroupGeom {
    uint32_t g;
    uint32_t sysid;  // the group's system: its root node (node id = system index) and box
    double L;
    uint32_t qmin0, qmin1, qmin2, qmax0, qmax1, qmax2;
    float4 gch;
    float hx, hy, hz, asym;
};

__device__ __forceinline__ GroupGeom group_geom(const WalkArgs& A, uint32_t g) {
    GroupGeom G;
    G.g = g;
    G.sysid = A.sys ? A.sys[A.g_first[g]] : 0u;
    G.L = A.box[G.sysid].L;
    const uint32_t* qb = A.g_qbox + 6 * (int64_t)g;
    G.qmin0 = qb[0];
    G.qmin1 = qb[1];
    G.qmin2 = qb[2];
    G.qmax0 = qb[3];
    G.qmax1 = qb[4];
    G.qmax2 = qb[5];
    G.gch = A.g_ch[g];
    const float4 lo = A.g_blo[g], hi = A.g_bhi[g];
    G.hx = fmaxf(-lo.x, hi.x);
    G.hy = fmaxf(-lo.y, hi.y);
    G.hz = fmaxf(-lo.z, hi.z);
    G.asym = fmaxf(fmaxf(fabsf(lo.x + hi.x), fabsf(lo.y + hi.y)), fabsf(lo.z + hi.z));
    return G;
}

// The two thresholds on d^2 of the FP32 filter for cells of `level`: below
// the first the cell opens, above the second it does not.  e0: the absolute
// error of a coordinate of the cell's offset from the group.
constexpr float kE0Hi = 6.2e-8f;   // times L: centre of mass and group centre rounded to FP32 (u L / 2 each)
constexpr float kE0Pair = 1e-13f;  // times L: both as FP32 hi/lo pairs
__device__ __forceinline__ float2 level_thresholds(const WalkArgs& A, const GroupGeom& G, int level,
                                                   float e0rel) {
    const float Lf = __double2float_rn(G.L);
    // the FP32 filter's bound holds while the squares of cell sizes stay
    // normal FP32 numbers (with or without flushing of subnormals): outside
    // this range of root boxes every test takes the exact FP64 sequence
    const bool filt = Lf >= 0x1p-40f && Lf <= 0x1p60f;
    const float hb = fmaxf(fmaxf(G.hx, G.hy), G.hz);
    // Coefficients of the filter's error bound as a polynomial in M = max|d| +
    // hb (d the FP32 offset of a cell's centre of mass, hb the largest
    // |corner| of the group box): with E = 4uM + e0 the error of one
    // coordinate and S1 = t_x + t_y + t_z <= 3M, theta^2 (2 E S1 + 3 E^2) <=
    // theta^2 (25 u M^2 + 7 e0 M + 4 e0^2); 1 % on top covers the rounding of
    // the bound's own FP32 evaluation.
    const float e0 = fmaf(e0rel, Lf, G.asym);
    const float mc1 = 1.01f * A.theta2f * 25.0f * kU32, mc2 = 1.01f * A.theta2f * 7.0f * e0,
                mc3 = 1.01f * A.theta2f * 4.0f * e0 * e0;
    // The bound's largest value over the cells each side can decide, as two
    // thresholds on d^2 per level (lane = level): a cell with d^2 <= D0^2 =
    // ell^2 / theta^2 has M <= D0 + 2 hb (|d_a| <= t_a + hb), so the margin
    // is at most Mo and d^2 < (ell^2 - Mo) / theta^2 opens it; beyond D0,
    // with (s + 2 hb)^2 <= 2 s^2 + 8 hb^2 and s = |t| <= (d^2 + D0^2) / (2 D0),
    // the margin is linear in d^2 and d^2 above hi rejects it.  Slack covers
    // the thresholds' own FP32 evaluation; outside the filter's range of L
    // (and at theta = 0, where every cell opens) no threshold decides.
    float lo = -INFINITY, hi = INFINITY;
    if (!filt) {
    } else if (A.theta2f == 0.0f) {
        lo = INFINITY;
    } else {
        const float ell = __int_as_float(__float_as_int(Lf) - (level << 23));
        const float l2 = ell * ell;
        const float D0 = sqrtf(l2 / A.theta2f);
        const float Mb = D0 + 2.0f * hb;
        const float Mo = fmaf(16.0f * kU32, l2, fmaf(fmaf(mc1, Mb, mc2), Mb, mc3));
        lo = (l2 - Mo) / A.theta2f * (1.0f - 8.0f * kU32);
        const float coef = A.theta2f - (8.0f * kU32 * A.theta2f + 2.0f * mc1 + mc2 / (2.0f * D0));
        const float rhs = l2 * (1.0f + 8.0f * kU32) + 8.0f * mc1 * hb * hb + mc2 * (0.5f * D0 + 2.0f * hb) + mc3;
        if (coef > 0.0f) hi = rhs * (1.0f + 16.0f * kU32) / coef;
    }
    return make_float2(lo, hi);
}

// Per-level thresholds of one group: for offsets from rounded centres, and
// for offsets from hi/lo pairs.
struct Thresholds {
    float2 hi[kMaxLevel + 1], pair[kMaxLevel + 1];
};

__device__ __forceinline__ float box_dist2(float hx, float hy, float hz, float dx, float dy, float dz) {
    const float tx = fmaxf(fabsf(dx) - hx, 0.0f);
    const float ty = fmaxf(fabsf(dy) - hy, 0.0f);
    const float tz = fmaxf(fabsf(dz) - hz, 0.0f);
    return tx * tx + ty * ty + tz * tz;
}

// What the rounded centres leave undecided (1 test in 10^3 or less down to
// levels where the cells are 10^-4 of the root box): the pairs' thresholds,
// and between those the FP64 sequence.
__device__ __noinline__ bool cell_opens_close(const WalkArgs& A, uint32_t g, uint32_t node, int level, double L,
                                              const float2 th) {
    const float4 fh = A.nd_f[2 * node], fl = A.nd_f[2 * node + 1];
    const float4 ch = A.g_ch[g], cl = A.g_cl[g];
    const float4 lo = A.g_blo[g], hi = A.g_bhi[g];
    const float d2 = box_dist2(fmaxf(-lo.x, hi.x), fmaxf(-lo.y, hi.y), fmaxf(-lo.z, hi.z), (fh.x - ch.x) + (fl.x - cl.x), (fh.y - ch.y) + (fl.y - cl.y),
                               (fh.z - ch.z) + (fl.z - cl.z));
    if (d2 < th.x) return true;
    if (d2 > th.y) return false;
    atomicAdd(&A.st->fallbacks, 1ull);  // rare: counted where it happens
    return open_fp64(L, level, A.theta2, A.nd_com[node], A.g_box + 6 * (int64_t)g);
}

// The opening test of one cell, from its walk record: the grid boxes, then
// the FP32 filter on rounded centres (half of the loads of the hi/lo pairs,
// which took the walk's L1 to 61 % of its rate beside 70 % of the issue
// slots; with the box as half-widths and the children stored off
// one address: 2^24 particles 5.95 -> 4.43 ms, 256 clusters 2.64 -> 1.88, 2^20
// 0.63 -> 0.48).
__device__ __forceinline__ bool cell_opens(const WalkArgs& A, const GroupGeom& G, uint32_t node, const uint4 rec,
                                           const float4 c, const Thresholds& thr) {
    const int level = (int)((rec.x >> 21) & 31u);
    const uint32_t w = (1u << (kMaxLevel - level)) - 1u;
    const uint32_t qx = rec.x & kQMax, qy = rec.y, qz = rec.z;
    if (qx <= G.qmax0 && qx + w >= G.qmin0 && qy <= G.qmax1 && qy + w >= G.qmin1 && qz <= G.qmax2 &&
        qz + w >= G.qmin2)
        return true;
    const float d2 = box_dist2(G.hx, G.hy, G.hz, c.x - G.gch.x, c.y - G.gch.y, c.z - G.gch.z);
    const float2 th = thr.hi[level];
    if (d2 < th.x) return true;
    if (d2 > th.y) return false;
    return cell_opens_close(A, G.g, node, level, G.L, thr.pair[level]);
}

// The list of group g, walked by the calling warp (all 32 lanes), with its
// two frontier buffers fa and fb and the warp's per-level thresholds thr.
__device__ __forceinline__ void walk_group(const WalkArgs& A, uint32_t g, uint32_t* fa, uint32_t* fb,
                                           Thresholds& thr, WalkState& S) {
    DevState* st = A.st;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t F = A.cap_frontier;
    const GroupGeom G = group_geom(A, g);
    __syncwarp();  // the previous group's walk has read thr
    if (lane <= kMaxLevel) {
        thr.hi[lane] = level_thresholds(A, G, lane, kE0Hi);
        thr.pair[lane] = level_thresholds(A, G, lane, kE0Pair);
    }
    __syncwarp();

    if (S.ovf) S.coff = 0;  // counting only
    uint32_t goff = S.coff;  // where the list starts in the chunk
    uint32_t nleaf = 0, nepj_lane = 0;
    uint32_t fsize = 1;
    if (lane == 0) fa[0] = G.sysid;
    __syncwarp();
    while (fsize > 0) {
        uint32_t nsize = 0;
        S.max_front = fsize > S.max_front ? fsize : S.max_front;
        // the first batch's frontier entries and node records;
        // every batch then fetches the next one's before testing its own
        // (frontier ids two batches ahead, records one batch ahead, so
        // no batch waits on a load that depends on another load)
        uint32_t node_nx = lane < fsize ? fa[lane] : 0u;
        uint32_t node_nx2 = lane + 32 < fsize ? fa[lane + 32] : 0u;
        uint4 rec_nx = make_uint4(0, 0, 0, 0);
        float4 c_nx = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane < fsize) ld_walk(A.nd_walk + node_nx, rec_nx, c_nx);
        for (uint32_t base = 0; base < fsize; base += 32) {
            const uint32_t idx = base + lane;
            const bool act = idx < fsize;
            const uint32_t node = node_nx;
            const uint4 rec = rec_nx;
            const float4 c = c_nx;
            if (idx + 32 < fsize) {
                node_nx = node_nx2;
                ld_walk(A.nd_walk + node_nx, rec_nx, c_nx);
            }
            if (idx + 64 < fsize) node_nx2 = fa[idx + 64];
            int action = 0;  // 1 SPJ, 2 EPJ leaf, 3 open internal
            uint32_t nch = 0, child = 0;
            if (act) {
                const bool leaf = (rec.x >> 26) & 1u;
                const bool open = cell_opens(A, G, node, rec, c, thr);
                if (!open) {
                    action = 1;
                } else if (leaf) {
                    action = 2;
                    nepj_lane += rec.w;  // the leaf's particle count
                } else {
                    action = 3;
                    child = rec.w;
                    nch = rec.x >> 27;
                }
            }
            // ---- append SPJ entries upwards, EPJ entries downwards from the
            // chunk's end
            const uint32_t smask = __ballot_sync(0xFFFFFFFFu, action == 1);
            const uint32_t lmask = __ballot_sync(0xFFFFFFFFu, action == 2);
            if (smask | lmask) {
                const uint32_t ks = __popc(smask), kl = __popc(lmask);
                if (S.coff + nleaf + ks + kl > S.clen) {
                    // new chunk: at least kChunk entries and twice the
                    // group's list so far, so long lists move O(log) times
                    const uint32_t nsp = S.coff - goff;
                    const unsigned long long sofar = (unsigned long long)nsp + nleaf;
                    const unsigned long long want =
                        2 * (sofar + ks + kl) > kChunk ? 2 * (sofar + ks + kl) : kChunk;
                    unsigned long long nb = 0;
                    if (lane == 0) nb = atomicAdd(&st->pool_cursor, want);
                    nb = shfl_u64(nb, 0);
                    if (!S.ovf && (nb + want > A.cap_pool || want > 0xFFFFFFFFull)) {
                        if (lane == 0) atomicOr(&st->overflow, kOvfPool);
                        S.ovf = true;
                    }
                    if (!S.ovf) {
                        uint32_t* np = A.pool + nb;
#pragma unroll 1
                        for (uint32_t j = lane; j < nsp; j += 32) np[j] = S.cptr[goff + j];
                        const uint32_t* lsrc = S.cptr + (S.clen - nleaf);
                        uint32_t* ldst = np + (want - nleaf);
#pragma unroll 1
                        for (uint32_t j = lane; j < nleaf; j += 32) ldst[j] = lsrc[j];
                        __syncwarp();
                        S.cptr = np;
                        S.clen = (uint32_t)want;
                    } else {
                        S.clen = 0xFFFFFFFFu;  // count only from here on
                    }
                    goff = 0;
                    S.coff = nsp;
                }
                if ((action == 1 || action == 2) && !S.ovf) {
                    const bool spj = action == 1;
                    const uint32_t r = __popc((spj ? smask : lmask) & lt);
                    S.cptr[spj ? S.coff + r : S.clen - 1u - nleaf - r] = spj ? node : node | kLeafTag;
                }
                S.coff += ks;
                nleaf += kl;
            }
            // ---- push children of opened internal cells (deep in the
            // tree most batches open none)
            if (__ballot_sync(0xFFFFFFFFu, nch > 0u)) {
                uint32_t inc = nch;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    uint32_t tv = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                    if (lane >= off) inc += tv;
                }
                const uint32_t tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
                if (nsize + tot > F) {
                    if (lane == 0) atomicOr(&st->overflow, kOvfFrontier);
                    S.ovf = true;
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
    // the leaves behind the superparticles (towards lower addresses, 128 at a
    // time: a batch is read before it is written, so the ranges may overlap)
    const uint32_t nspj = S.coff - goff;
    if (!S.ovf && S.clen - nleaf > S.coff) {
        const uint32_t* src = S.cptr + (S.clen - nleaf);
        uint32_t* dst = S.cptr + S.coff;
#pragma unroll 1
        for (uint32_t j = lane; j < ((nleaf + 31u) & ~31u); j += 128) {
            uint32_t e[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) e[r] = j + 32 * r < nleaf ? src[j + 32 * r] : 0u;
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (j + 32 * r < nleaf) dst[j + 32 * r] = e[r];
            __syncwarp();
        }
    }
    S.coff += nleaf;
    const uint32_t nepj = __reduce_add_sync(0xFFFFFFFFu, nepj_lane);
    const uint32_t len = nspj + nleaf;
    if (lane == 0) {
        A.g_off[g] = (unsigned long long)(S.cptr + goff - A.pool);
        A.g_len[g] = len;
        A.g_nspj[g] = nspj;
        A.g_nepj[g] = nepj;
    }
    const unsigned long long ni = A.g_count[g];
    const unsigned long long mul = lane < 3 ? 1ull : ni;
    S.total += mul * (lane == 0 ? len : (lane & 1) ? nepj : nspj);
}

// The warp's totals into the device state word.
__device__ __forceinline__ void walk_flush(const WalkArgs& A, const WalkState& S) {
    DevState* st = A.st;
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        atomicAdd(&st->pool_needed, S.total);
        atomicMax(&st->max_frontier, S.max_front);
    }
    if (lane < 5)
        atomicAdd(lane == 0   ? &st->list_entries
                  : lane == 1 ? &st->n_epj
                  : lane == 2 ? &st->n_spj
                  : lane == 3 ? &st->int_epj
                              : &st->int_spj,
                  S.total);
}

constexpr int kWalkBlock = 128;

__global__ void __launch_bounds__(kWalkBlock, 8) k_walk(WalkArgs A) {
    DevState* st = A.st;
    if (st->overflow & kTreeInvalid) return;  // the host redoes the build
    const int lane = threadIdx.x & 31;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    uint32_t* fa = A.frontier + wid * 2 * (int64_t)A.cap_frontier;
    uint32_t* fb = fa + A.cap_frontier;
    const uint32_t ngroups = (uint32_t)st->n_groups;
    __shared__ Thresholds s_thr[kWalkBlock / 32];
    WalkState S = walk_state_init();
    for (;;) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(&st->walk_counter, 1u);
        g = __shfl_sync(0xFFFFFFFFu, g, 0);
        if (g >= ngroups) break;
        walk_group(A, g, fa, fb, s_thr[threadIdx.x >> 5], S);
    }
    walk_flush(A, S);
}

// The walk for systems of at most kWalkFew particles and about kWalkFewGroups
// groups: a block per group.  Their groups are too few to give every warp one (1,002 groups of a 2^14
// Plummer sphere on 4,864 warps), and a warp alone takes a group's batches of
// 32 cells one latency after the other; four warps take a level 128 cells at
// a time, with the frontier in shared memory (its rest, beyond kFewFrontier,
// in the block's part of the frontier buffers).  The same tests and the same
// list layout as walk_group.  Plummer 2^14, n_grp 64: walk 96 -> 69 us.  A warp per
// group against a block, by groups: 645 49 / 41 us, 1106 51 / 41, 1835 68 / 66, 2141
// 53 / 59, 3522 64 / 88, 11956 143 / 303.
constexpr int64_t kWalkFew = int64_t(1) << 15;
constexpr int64_t kWalkFewGroups = 2048;
constexpr uint32_t kFewFrontier = 1536;
constexpr int kWalkWarps = kWalkBlock / 32;

__global__ void __launch_bounds__(kWalkBlock, 8) k_walk_few(WalkArgs A) {
    __shared__ Thresholds s_thr;
    __shared__ uint32_t s_fr[2][kFewFrontier];
    __shared__ uint32_t s_cnt[2][3][kWalkWarps];  // a batch's superparticles, leaves and children, per warp
    __shared__ uint32_t s_red[kWalkWarps];
    __shared__ unsigned long long s_nb;
    __shared__ uint32_t s_g;
    DevState* st = A.st;
    if (st->overflow & kTreeInvalid) return;  // as in k_walk
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t ngroups = (uint32_t)st->n_groups;
    const uint32_t F = kWalkWarps * A.cap_frontier;  // of the block, beyond the shared part
    uint32_t* const gfr = A.frontier + blockIdx.x * 2 * (int64_t)F;
    auto entry = [&](int p, uint32_t k) -> uint32_t& {
        return k < kFewFrontier ? s_fr[p][k] : gfr[(int64_t)p * F + (k - kFewFrontier)];
    };
    WalkState S = walk_state_init();
    int q = 0;  // the batch's half of s_cnt
    for (;;) {
        if (t == 0) s_g = atomicAdd(&st->walk_counter, 1u);
        __syncthreads();
        const uint32_t g = s_g;
        if (g >= ngroups) break;
        const GroupGeom G = group_geom(A, g);
        if (t <= kMaxLevel) {
            s_thr.hi[t] = level_thresholds(A, G, t, kE0Hi);
            s_thr.pair[t] = level_thresholds(A, G, t, kE0Pair);
        }
        if (t == 0) s_fr[0][0] = G.sysid;
        if (S.ovf) S.coff = 0;  // counting only
        uint32_t goff = S.coff;
        uint32_t nleaf = 0, nepj_lane = 0, fsize = 1;
        int p = 0;
        __syncthreads();
        while (fsize > 0) {
            uint32_t nsize = 0;
            S.max_front = fsize > S.max_front ? fsize : S.max_front;
            for (uint32_t base = 0; base < fsize; base += kWalkBlock) {
                const uint32_t idx = base + t;
                uint32_t node = 0, nch = 0, child = 0;
                bool spj = false, epj = false;
                if (idx < fsize) {
                    node = entry(p, idx);
                    uint4 rec;
                    float4 c;
                    ld_walk(A.nd_walk + node, rec, c);
                    const bool leaf = (rec.x >> 26) & 1u;
                    if (!cell_opens(A, G, node, rec, c, s_thr)) {
                        spj = true;
                    } else if (leaf) {
                        epj = true;
                        nepj_lane += rec.w;
                    } else {
                        child = rec.w;
                        nch = rec.x >> 27;
                    }
                }
                const uint32_t smask = __ballot_sync(0xFFFFFFFFu, spj), lmask = __ballot_sync(0xFFFFFFFFu, epj);
                uint32_t inc = nch;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t tv = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                    if (lane >= off) inc += tv;
                }
                if (lane == 31) {
                    s_cnt[q][0][w] = __popc(smask);
                    s_cnt[q][1][w] = __popc(lmask);
                    s_cnt[q][2][w] = inc;
                }
                __syncthreads();
                uint32_t ks = 0, kl = 0, kc = 0, rs = __popc(smask & lt), rl = __popc(lmask & lt), rc = inc - nch;
#pragma unroll
                for (int k = 0; k < kWalkWarps; ++k) {
                    const uint32_t cs = s_cnt[q][0][k], cl = s_cnt[q][1][k], cc = s_cnt[q][2][k];
                    if (k < w) {
                        rs += cs;
                        rl += cl;
                        rc += cc;
                    }
                    ks += cs;
                    kl += cl;
                    kc += cc;
                }
                q ^= 1;
                if (ks + kl > 0 && S.coff + nleaf + ks + kl > S.clen) {
                    // new chunk, as in walk_group
                    const uint32_t nsp = S.coff - goff;
                    const unsigned long long sofar = (unsigned long long)nsp + nleaf;
                    const unsigned long long want =
                        2 * (sofar + ks + kl) > kChunk ? 2 * (sofar + ks + kl) : kChunk;
                    if (t == 0) s_nb = atomicAdd(&st->pool_cursor, want);
                    __syncthreads();
                    const unsigned long long nb = s_nb;
                    if (!S.ovf && (nb + want > A.cap_pool || want > 0xFFFFFFFFull)) {
                        if (t == 0) atomicOr(&st->overflow, kOvfPool);
                        S.ovf = true;
                    }
                    if (!S.ovf) {
                        uint32_t* np = A.pool + nb;
                        for (uint32_t j = t; j < nsp; j += kWalkBlock) np[j] = S.cptr[goff + j];
                        const uint32_t* lsrc = S.cptr + (S.clen - nleaf);
                        uint32_t* ldst = np + (want - nleaf);
                        for (uint32_t j = t; j < nleaf; j += kWalkBlock) ldst[j] = lsrc[j];
                        S.cptr = np;
                        S.clen = (uint32_t)want;
                    } else {
                        S.clen = 0xFFFFFFFFu;  // count only from here on
                    }
                    goff = 0;
                    S.coff = nsp;
                    __syncthreads();  // s_nb has been read, the copies are written
                }
                if (!S.ovf) {
                    if (spj) S.cptr[S.coff + rs] = node;
                    if (epj) S.cptr[S.clen - 1u - nleaf - rl] = node | kLeafTag;
                }
                S.coff += ks;
                nleaf += kl;
                if (nsize + kc > kFewFrontier + F) {
                    if (t == 0) atomicOr(&st->overflow, kOvfFrontier);
                    S.ovf = true;
                } else {
                    const uint32_t o = nsize + rc;
                    for (uint32_t c = 0; c < nch; ++c) entry(p ^ 1, o + c) = child + c;
                    nsize += kc;
                }
            }
            __syncthreads();  // the next level's frontier is written
            p ^= 1;
            fsize = nsize;
        }
        // the leaves behind the superparticles, a batch read before it is
        // written
        const uint32_t nspj = S.coff - goff;
        if (!S.ovf && S.clen - nleaf > S.coff) {
            const uint32_t* src = S.cptr + (S.clen - nleaf);
            uint32_t* dst = S.cptr + S.coff;
            for (uint32_t j = 0; j < nleaf; j += 4 * kWalkBlock) {
                uint32_t e[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t k = j + r * kWalkBlock + t;
                    e[r] = k < nleaf ? src[k] : 0u;
                }
                __syncthreads();
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t k = j + r * kWalkBlock + t;
                    if (k < nleaf) dst[k] = e[r];
                }
                __syncthreads();
            }
        }
        S.coff += nleaf;
        const uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, nepj_lane);
        if (lane == 0) s_red[w] = wsum;
        __syncthreads();
        uint32_t nepj = 0;
#pragma unroll
        for (int k = 0; k < kWalkWarps; ++k) nepj += s_red[k];
        const uint32_t len = nspj + nleaf;
        if (t == 0) {
            A.g_off[g] = (unsigned long long)(S.cptr + goff - A.pool);
            A.g_len[g] = len;
            A.g_nspj[g] = nspj;
            A.g_nepj[g] = nepj;
        }
        const unsigned long long ni = A.g_count[g];
        const unsigned long long mul = lane < 3 ? 1ull : ni;
        S.total += mul * (lane == 0 ? len : (lane & 1) ? nepj : nspj);
    }
    if (w == 0) walk_flush(A, S);
}

}  // namespace

int walk_blocks(fdps_ctx* ctx) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_walk, kWalkBlock, 0) != cudaSuccess ||
        per_sm < 1)
        per_sm = 4;
    return per_sm * ctx->sm_count;
}

int walk_warps_per_block() { return kWalkBlock / 32; }

unsigned long long walk_chunk() { return kChunk; }

WalkArgs walk_args(fdps_tree* t, const uint32_t* sys) {
    WalkArgs A;
    A.st = t->st;
    A.nd_walk = t->nd_walk;
    A.nd_f = t->nd_f;
    A.nd_com = t->nd_com;
    A.g_count = t->g_count;
    A.g_first = t->g_first;
    A.sys = sys;
    A.box = t->sys_box;
    A.g_qbox = t->g_qbox;
    A.g_box = t->g_box;
    A.g_ch = t->g_ch;
    A.g_cl = t->g_cl;
    A.g_blo = t->g_blo;
    A.g_bhi = t->g_bhi;
    A.g_off = t->g_off;
    A.g_len = t->g_len;
    A.g_nspj = t->g_nspj;
    A.g_nepj = t->g_nepj;
    A.pool = t->pool;
    A.cap_pool = (unsigned long long)t->cap_pool;
    A.frontier = t->frontier;
    A.cap_frontier = (uint32_t)t->cap_frontier;
    A.theta2 = t->p.theta * t->p.theta;
    A.theta2f = (float)A.theta2;
    return A;
}

int launch_walk(fdps_tree* t, const uint32_t* sys, int blocks) {
    fdps_ctx* ctx = t->ctx;
    const WalkArgs A = walk_args(t, sys);
    if (t->n <= kWalkFew && t->est_groups <= kWalkFewGroups)
        k_walk_few<<<blocks, kWalkBlock, 0, ctx->stream>>>(A);
    else
        k_walk<<<blocks, kWalkBlock, 0, ctx->stream>>>(A);
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

}  // namespace fdps
