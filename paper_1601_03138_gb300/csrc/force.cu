// force.cu -- particle-particle (EPJ) and particle-superparticle (SPJ)
// forces from the interaction lists: one CTA per i-group (FP32-relative) or
// one cluster of CTAs per i-group (FP64 variant).
//
// Per i-particle (Sect. 2.2, Eqs. ParticleParticleNbody and
// ParticleSuperparticleNbody, G = 1, softening eps_i of the receiving
// particle):
//   a_i   = sum_EPJ m_j (x_j - x_i) / (r^2 + eps_i^2)^{3/2} + sum_SPJ f'
//   phi_i = -sum_EPJ m_j / (r^2 + eps_i^2)^{1/2} - ... + m_i / eps_i
// the last term removing the i-particle's own entry (its force term is zero).
// A quadrupole superparticle (mass M, traceless Q, r = x_i - com,
// R^2 = r^2 + eps_i^2) contributes phi = -M/R - (r.Q.r) / (2 R^5) and
// a = -M r / R^3 + Q r / R^5 - (5/2) (r.Q.r) r / R^7.  The FP32 kernel
// evaluates the same expressions regrouped as a = R^-5 (Q r + R^2 h r) and
// phi = R^-1 (h + 2 w), with w = (r.Q.r) R^-4 and h = -M - (5/2) w: 32 FP32
// operations per interaction (3 differences, 3 for R^2, 3 powers of 1/R,
// 9 for Q r, 3 for r.Q.r, w, h, R^2 h, 6 for a, 2 for phi) and one MUFU
// reciprocal square root.
//
// FP32-relative kernel (one CTA per i-group): list entries are gathered
// into shared memory as FP32 coordinates relative to the group centre,
// formed from FP32 hi/lo pairs so that near pairs keep full FP32 precision.
// A thread's i-particles are paired: the pair loop evaluates one list entry
// against two i-particles with packed two-lane FP32 instructions plus two
// MUFU rsqrt (one i-particle per thread: plain FP32); each thread
// accumulates one chunk of the list in plain FP32 and adds the chunk's sum to
// its running total with Kahan compensation.  A chunk is up to 512
// superparticles, or 1024 particles of up to 512 leaves (before the lists held
// the two apart: 512 entries, with all particles of the leaves among them).
// Small groups split their list over several threads per i-particle
// ("slices"), added with exact two-sums at the end.  The FP64 kernel
// (a cluster of CTAs per group) evaluates the same terms on FP64 absolute
// coordinates with FP64 sums.
#include <algorithm>

#include "fdps_internal.cuh"
#include "packed.cuh"

namespace fdps {

struct ForceArgs {
    DevState* st;
    const uint32_t* g_first;
    const uint32_t* g_count;
    const unsigned long long* g_off;
    const uint32_t* g_len;
    const uint32_t* g_nspj;
    const float4* g_ch;
    const float4* g_cl;
    const uint32_t* pool;
    const uint32_t* nd_first;
    const uint32_t* nd_count;
    const float4* nd_f;
    const float4* nd_fq0;
    const float2* nd_fq1;
    const dvec4* nd_com;
    const double* nd_quad;
    const float4* pf_hi;
    const float4* pf_lo;
    const double* px;
    const double* py;
    const double* pz;
    const double* pm;
    const double* peps;
    double* ax;
    double* ay;
    double* az;
    double* pot;
};

namespace {

// ---------------------------------------------------------------- FP32
// One CTA of CB threads (64, 128 or 256: the "block shape" the autotuner
// picks, with the cap KMAX on i-particles per thread) per i-group.  Thread t
// owns K <= KMAX i-particles (i = t % P + k P, k < K) and the list slice
// j = t / P (mod nsl); (K, P, nsl) is chosen per group to keep the most
// lanes busy.  A list holds its superparticles first and its opened leaves
// after them: the superparticles are consumed in chunks of 256 or 512 (the
// tile depth, EPT per thread), then the leaves' particles in tiles of up to
// 1024, staged in shared memory; each thread folds its FP32 partial sums of a
// chunk or tile into Kahan-compensated running sums.  With the two kinds
// mixed in the list, every chunk needed a scan and four smaller tiles with
// two barriers each, about 70 barriers a group instead of 21: the pass over
// 190,000 monopole groups of 16 particles (256 clusters, n_grp 64) took 7.51
// ms and took 6.02 with 21, 2^20 Plummer particles with quadrupoles at n_grp 128
// 3.94 and 3.72, 2^24 at n_grp 256 73.2 and 72.0 (FMA pipe 74 % busy: bound by
// the FP32 pipe and its register-operand conflicts), for 4 % in the walk.

struct GroupPlan {
    int K, P, nsl;
};

template <int CB, int KMAX>
__device__ __forceinline__ GroupPlan plan_group(uint32_t ni) {
    // maximise ni * nsl / (CB * K) over K in {1, ..., 5} (up to KMAX);
    // larger K on ties
    GroupPlan best{1, 1, 1};
    float bu = -1.f;
    // an odd K is packed pairs plus one scalar lane: the scalar lane issues
    // as many instructions per list entry as a pair for half the work, so an
    // odd K must fill the CTA 10 % better to be taken (2^24 particles: 73.4 ms
    // with no handicap, 72.3 with 3 %, 72.0 with 6, 71.5 with 10, 71.6 with 15)
    constexpr float kOdd = 1.1f;
    const int Ks[5] = {5, 4, 3, 2, 1};
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const int K = Ks[c];
        if (K > KMAX) continue;
        const int P = (int)((ni + K - 1) / K);
        if (P > CB) continue;
        const int nsl = CB / P;
        const float u = (float)ni * nsl / (float)(CB * K) / ((K & 1) && K > 1 ? kOdd : 1.0f);
        if (u > bu + 1e-6f) {
            bu = u;
            best = GroupPlan{K, P, nsl};
        }
    }
    if (bu < 0.f) best = GroupPlan{KMAX, CB, 1};  // more than KMAX CB particles: rounds
    return best;
}

// Block-wide exclusive scans of two values at once (CB threads).
template <int CB>
__device__ __forceinline__ void block_scan2(uint32_t a, uint32_t b, uint32_t* ea, uint32_t* eb,
                                            uint32_t* ta, uint32_t* tb, uint32_t* s_w) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t ia = a, ib = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t va = __shfl_up_sync(0xFFFFFFFFu, ia, o);
        const uint32_t vb = __shfl_up_sync(0xFFFFFFFFu, ib, o);
        if (lane >= o) {
            ia += va;
            ib += vb;
        }
    }
    if (lane == 31) {
        s_w[w] = ia;
        s_w[CB / 32 + w] = ib;
    }
    __syncthreads();
    uint32_t oa = 0, ob = 0, sa = 0, sb = 0;
#pragma unroll
    for (int k = 0; k < CB / 32; ++k) {
        const uint32_t xa = s_w[k], xb = s_w[CB / 32 + k];
        if (k < w) {
            oa += xa;
            ob += xb;
        }
        sa += xa;
        sb += xb;
    }
    *ea = oa + ia - a;
    *eb = ob + ib - b;
    *ta = sa;
    *tb = sb;
}

// Block-wide exclusive scan (CB threads); s_w holds CB / 32 words.
template <int CB>
__device__ __forceinline__ uint32_t block_scan1(uint32_t a, uint32_t* total, uint32_t* s_w) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t ia = a;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, ia, o);
        if (lane >= o) ia += v;
    }
    if (lane == 31) s_w[w] = ia;
    __syncthreads();
    uint32_t o = 0, sum = 0;
#pragma unroll
    for (int k = 0; k < CB / 32; ++k) {
        const uint32_t x = s_w[k];
        if (k < w) o += x;
        sum += x;
    }
    *total = sum;
    return o + ia - a;
}

// EPT consecutive u32 slots of one thread written as one vector.
template <int EPT>
__device__ __forceinline__ void store_entries(uint32_t* dst, const uint32_t (&v)[EPT]) {
    if (EPT == 8) {
        reinterpret_cast<uint4*>(dst)[0] = make_uint4(v[0], v[1 % EPT], v[2 % EPT], v[3 % EPT]);
        reinterpret_cast<uint4*>(dst)[1] = make_uint4(v[4 % EPT], v[5 % EPT], v[6 % EPT], v[7 % EPT]);
    } else if (EPT == 4)
        *reinterpret_cast<uint4*>(dst) = make_uint4(v[0], v[1 % EPT], v[2 % EPT], v[3 % EPT]);
    else if (EPT == 2)
        *reinterpret_cast<uint2*>(dst) = make_uint2(v[0], v[1 % EPT]);
    else
        for (int r = 0; r < EPT; ++r) dst[r] = v[r];
}

// Largest e in [0, CE) with scan[e] <= item (binary lifting: CE a power of
// two).
template <int CE>
__device__ __forceinline__ int owner_chunk(const uint32_t* scan, uint32_t item) {
    static_assert(CE > 0 && (CE & (CE - 1)) == 0, "list chunks of a power-of-two length");
    int lo = 0;
#pragma unroll
    for (int step = CE / 2; step > 0; step >>= 1)
        if (scan[lo + step] <= item) lo += step;
    return lo;
}

// hi + lo += v with an exact FP32 two-sum (Knuth): hi takes the rounded
// sum, lo the rounding error.
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float v) {
    const float s = hi + v;
    const float bb = s - hi;
    lo += (hi - (s - bb)) + (v - bb);
    hi = s;
}

// Kahan running sums of one thread in shared memory: sum of (q, c) at
// s_k[((q * 4 + c) * 2) * CB + t], its compensation CB further on.
template <int CB>
__device__ __forceinline__ void kahan_smem_add(float* s_k, int q, int c, float v) {
    float* s = s_k + ((q * 4 + c) * 2) * CB + threadIdx.x;
    float* cp = s + CB;
    const float y = v - *cp;
    const float t = *s + y;
    *cp = (t - *s) - y;
    *s = t;
}

// (the packed operations flush subnormals, as the whole file is compiled to)
__device__ __forceinline__ f2 f2_rsqrt(f2 v) {
    float a, b;
    f2_up(v, a, b);
    return f2_pk(rsqrtf(a), rsqrtf(b));
}
// Shared memory of the FP32 kernels (one CTA per group at a time;
// coordinates relative to the group centre).  The buffer u holds a chunk of
// superparticles, float4 (x, y, z, -M), float4 (Qxx, Qyy, Qzz, Qxy), float2
// (Qxz, Qyz) in three arrays (the first only for monopoles), and after them
// a tile of leaf particles, float4 (x, y, z, m), with the first particles
// and the scanned counts of a batch of leaves behind it.  A thread's
// i-particles are paired (2h, 2h+1) in the two lanes of a packed register;
// each list entry is broadcast to both lanes.
constexpr int cmax(int a, int b) { return a > b ? a : b; }
constexpr int cmin(int a, int b) { return a < b ? a : b; }
template <bool QUAD, int EPT, int CB, int KMAX>
struct F32Shared {
    static constexpr int kCE = CB * EPT;  // superparticles per chunk
    static constexpr int kCL = CB * EPT;  // leaves per batch
    static constexpr int kCJ = cmin((QUAD ? 8 : 4) * CB, 1024);  // leaf particles per tile
    __align__(16) unsigned char u[cmax(kCE * (QUAD ? 40 : 16), kCJ * 16 + 2 * kCL * 4)];
    uint32_t w[2 * (CB / 32)];
    float k[KMAX * 8 * CB];  // Kahan sums and compensations
};
__device__ __forceinline__ f2 f2_bc(float v) { return f2_pk(v, v); }

template <bool QUAD, int K, int EPT, int CB, int KMAX, int WARPS>
__device__ __forceinline__ void force_round_f32(const ForceArgs& A, uint32_t gf, uint32_t ni,
                                                unsigned long long off, uint32_t nspj, uint32_t len, float4 gch,
                                                float4 gcl, int P, int nsl, uint32_t ib,
                                                F32Shared<QUAD, EPT, CB, KMAX>& sm) {
    using SM = F32Shared<QUAD, EPT, CB, KMAX>;
    constexpr int kCJ = SM::kCJ;
    float4* const s_s0 = reinterpret_cast<float4*>(sm.u);
    float4* const s_s1 = reinterpret_cast<float4*>(sm.u + (QUAD ? SM::kCE * 16 : 0));
    float2* const s_s2 = reinterpret_cast<float2*>(sm.u + (QUAD ? SM::kCE * 32 : 0));
    float4* const s_j = reinterpret_cast<float4*>(sm.u);
    uint32_t* const s_ef = reinterpret_cast<uint32_t*>(sm.u + kCJ * 16);
    uint32_t* const s_es = s_ef + SM::kCL;
    float* const s_k = sm.k;
    // list entries per loop turn, measured (cells 2 to 10, leaf particles 1 to
    // 4): quadrupoles at 2^24 particles 73.5 ms with 2 and 2, 72.0 with 5 and 3;
    // monopoles of 256 clusters 5.39 ms with 6 and 2 at six CTAs per SM, 5.15
    // with 3 and 2 (3 in the second loop costs registers: 20 % more)
    constexpr int kUnrollSpj = QUAD ? 5 : WARPS > 16 ? 3 : 6, kUnrollEpj = QUAD ? 3 : 2;
    constexpr int KP = K / 2;  // i-pairs; an odd K takes its last i-particle on the scalar path
    const int t = threadIdx.x;
    const int ip = t % P, sl = t / P;
    const bool on = sl < nsl;
    float xi[K], yi[K], zi[K], e2[K];
    bool iv[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        const uint32_t i = ib + (uint32_t)(ip + q * P);
        iv[q] = on && i < ni;
        xi[q] = yi[q] = zi[q] = 0.f;
        e2[q] = 1.f;
        if (iv[q]) {
            const float4 h = A.pf_hi[gf + i], l = A.pf_lo[gf + i];
            xi[q] = (h.x - gch.x) + (l.x - gcl.x);
            yi[q] = (h.y - gch.y) + (l.y - gcl.y);
            zi[q] = (h.z - gch.z) + (l.z - gcl.z);
            e2[q] = l.w;
        }
    }
    f2 xp[KP > 0 ? KP : 1], yp[KP > 0 ? KP : 1], zp[KP > 0 ? KP : 1], ep[KP > 0 ? KP : 1];
#pragma unroll
    for (int h = 0; h < KP; ++h) {
        xp[h] = f2_pk(xi[2 * h], xi[2 * h + 1]);
        yp[h] = f2_pk(yi[2 * h], yi[2 * h + 1]);
        zp[h] = f2_pk(zi[2 * h], zi[2 * h + 1]);
        ep[h] = f2_pk(e2[2 * h], e2[2 * h + 1]);
    }
    const f2 cm25 = f2_bc(-2.5f), c2 = f2_bc(2.0f);
    const int kbeg = on ? sl : 0x3FFFFFFF;
#pragma unroll
    for (int k = 0; k < 8 * K; ++k) s_k[k * CB + t] = 0.0f;

    float sax[K], say[K], saz[K], spp[K];  // scalar path (K = 1)
    f2 pax[KP > 0 ? KP : 1], pay[KP > 0 ? KP : 1], paz[KP > 0 ? KP : 1], pp[KP > 0 ? KP : 1];
    auto clear = [&]() {
#pragma unroll
        for (int q = 0; q < K; ++q) sax[q] = say[q] = saz[q] = spp[q] = 0.f;
#pragma unroll
        for (int h = 0; h < KP; ++h) pax[h] = pay[h] = paz[h] = pp[h] = 0ull;
    };
    // the FP32 sums of a chunk into the Kahan sums
    auto fold = [&]() {
        if (K & 1) {
            kahan_smem_add<CB>(s_k, K - 1, 0, sax[K - 1]);
            kahan_smem_add<CB>(s_k, K - 1, 1, say[K - 1]);
            kahan_smem_add<CB>(s_k, K - 1, 2, saz[K - 1]);
            kahan_smem_add<CB>(s_k, K - 1, 3, spp[K - 1]);
        }
#pragma unroll
        for (int h = 0; h < KP; ++h) {
            float lo, hi;
            f2_up(pax[h], lo, hi);
            kahan_smem_add<CB>(s_k, 2 * h, 0, lo);
            kahan_smem_add<CB>(s_k, 2 * h + 1, 0, hi);
            f2_up(pay[h], lo, hi);
            kahan_smem_add<CB>(s_k, 2 * h, 1, lo);
            kahan_smem_add<CB>(s_k, 2 * h + 1, 1, hi);
            f2_up(paz[h], lo, hi);
            kahan_smem_add<CB>(s_k, 2 * h, 2, lo);
            kahan_smem_add<CB>(s_k, 2 * h + 1, 2, hi);
            f2_up(pp[h], lo, hi);
            kahan_smem_add<CB>(s_k, 2 * h, 3, lo);
            kahan_smem_add<CB>(s_k, 2 * h + 1, 3, hi);
        }
    };
    // ---- the list's superparticles, in chunks
    for (uint32_t base = 0; base < nspj; base += SM::kCE) {
        const uint32_t ns = nspj - base < (uint32_t)SM::kCE ? nspj - base : (uint32_t)SM::kCE;
        uint32_t node[EPT];
#pragma unroll
        for (int r = 0; r < EPT; ++r) {
            const uint32_t k = (uint32_t)(r * CB + t);
            node[r] = k < ns ? A.pool[off + base + k] : 0u;
        }
#pragma unroll
        for (int r = 0; r < EPT; ++r) {
            const int k = r * CB + t;
            if (k >= (int)ns) continue;
            const float4 fh = A.nd_f[2 * node[r]], fl = A.nd_f[2 * node[r] + 1];
            s_s0[k] = make_float4((fh.x - gch.x) + (fl.x - gcl.x), (fh.y - gch.y) + (fl.y - gcl.y),
                                  (fh.z - gch.z) + (fl.z - gcl.z), -fh.w);
            if (QUAD) {
                s_s1[k] = A.nd_fq0[node[r]];
                s_s2[k] = A.nd_fq1[node[r]];
            }
        }
        __syncthreads();
        clear();
#pragma unroll kUnrollSpj
        for (int k = kbeg; k < (int)ns; k += nsl) {
            const float4 a = s_s0[k];
            float4 q0;
            float2 q1;
            if (QUAD) {
                q0 = s_s1[k];
                q1 = s_s2[k];
            }
            if (K & 1) {  // the odd i-particle (index K - 1) in scalar FP32
                const float rx = xi[K - 1] - a.x, ry = yi[K - 1] - a.y, rz = zi[K - 1] - a.z;
                const float R2 = fmaf(rx, rx, fmaf(ry, ry, fmaf(rz, rz, e2[K - 1])));
                const float Ri = rsqrtf(R2);
                const float Ri2 = Ri * Ri;
                if (QUAD) {
                    const float Ri4 = Ri2 * Ri2;
                    const float Ri5 = Ri4 * Ri;
                    const float Qrx = fmaf(q0.x, rx, fmaf(q0.w, ry, q1.x * rz));
                    const float Qry = fmaf(q0.w, rx, fmaf(q0.y, ry, q1.y * rz));
                    const float Qrz = fmaf(q1.x, rx, fmaf(q1.y, ry, q0.z * rz));
                    const float rQr = fmaf(rx, Qrx, fmaf(ry, Qry, rz * Qrz));
                    const float w = rQr * Ri4;                 // r.Q.r / R^4
                    const float hh = fmaf(-2.5f, w, a.w);      // -M - 5/2 w
                    const float hR2 = hh * R2;
                    sax[K - 1] = fmaf(Ri5, fmaf(hR2, rx, Qrx), sax[K - 1]);
                    say[K - 1] = fmaf(Ri5, fmaf(hR2, ry, Qry), say[K - 1]);
                    saz[K - 1] = fmaf(Ri5, fmaf(hR2, rz, Qrz), saz[K - 1]);
                    spp[K - 1] = fmaf(Ri, fmaf(2.0f, w, hh), spp[K - 1]);  // (-M - w/2) / R
                } else {
                    const float Ri3 = Ri * Ri2;
                    const float nMRi3 = a.w * Ri3;
                    sax[K - 1] = fmaf(nMRi3, rx, sax[K - 1]);
                    say[K - 1] = fmaf(nMRi3, ry, say[K - 1]);
                    saz[K - 1] = fmaf(nMRi3, rz, saz[K - 1]);
                    spp[K - 1] = fmaf(a.w, Ri, spp[K - 1]);
                }
            }
            if (KP > 0) {
                const f2 jx = f2_bc(a.x), jy = f2_bc(a.y), jz = f2_bc(a.z), nM = f2_bc(a.w);
                f2 qxx, qyy, qzz, qxy, qxz, qyz;
                if (QUAD) {
                    qxx = f2_bc(q0.x);
                    qyy = f2_bc(q0.y);
                    qzz = f2_bc(q0.z);
                    qxy = f2_bc(q0.w);
                    qxz = f2_bc(q1.x);
                    qyz = f2_bc(q1.y);
                }
#pragma unroll
                for (int h = 0; h < KP; ++h) {
                    const f2 rx = f2_sub<true>(xp[h], jx), ry = f2_sub<true>(yp[h], jy), rz = f2_sub<true>(zp[h], jz);
                    const f2 R2 = f2_fma<true>(rx, rx, f2_fma<true>(ry, ry, f2_fma<true>(rz, rz, ep[h])));
                    const f2 Ri = f2_rsqrt(R2);
                    const f2 Ri2 = f2_mul<true>(Ri, Ri);
                    if (QUAD) {
                        const f2 Ri4 = f2_mul<true>(Ri2, Ri2);
                        const f2 Ri5 = f2_mul<true>(Ri4, Ri);
                        const f2 Qrx = f2_fma<true>(qxx, rx, f2_fma<true>(qxy, ry, f2_mul<true>(qxz, rz)));
                        const f2 Qry = f2_fma<true>(qxy, rx, f2_fma<true>(qyy, ry, f2_mul<true>(qyz, rz)));
                        const f2 Qrz = f2_fma<true>(qxz, rx, f2_fma<true>(qyz, ry, f2_mul<true>(qzz, rz)));
                        const f2 rQr = f2_fma<true>(rx, Qrx, f2_fma<true>(ry, Qry, f2_mul<true>(rz, Qrz)));
                        const f2 w = f2_mul<true>(rQr, Ri4);         // r.Q.r / R^4
                        const f2 hh = f2_fma<true>(cm25, w, nM);     // -M - 5/2 w
                        const f2 hR2 = f2_mul<true>(hh, R2);
                        pax[h] = f2_fma<true>(Ri5, f2_fma<true>(hR2, rx, Qrx), pax[h]);
                        pay[h] = f2_fma<true>(Ri5, f2_fma<true>(hR2, ry, Qry), pay[h]);
                        paz[h] = f2_fma<true>(Ri5, f2_fma<true>(hR2, rz, Qrz), paz[h]);
                        pp[h] = f2_fma<true>(Ri, f2_fma<true>(c2, w, hh), pp[h]);  // (-M - w/2) / R
                    } else {
                        const f2 Ri3 = f2_mul<true>(Ri, Ri2);
                        const f2 nMRi3 = f2_mul<true>(nM, Ri3);  // -M/R^3
                        pax[h] = f2_fma<true>(nMRi3, rx, pax[h]);
                        pay[h] = f2_fma<true>(nMRi3, ry, pay[h]);
                        paz[h] = f2_fma<true>(nMRi3, rz, paz[h]);
                        pp[h] = f2_fma<true>(nM, Ri, pp[h]);
                    }
                }
            }
        }
        fold();
        __syncthreads();  // the chunk is rewritten next
    }
    // ---- the opened leaves: their particle ranges in batches, the
    // particles in shared tiles
    for (uint32_t base = nspj; base < len; base += SM::kCL) {
        // this thread's EPT consecutive leaves
        uint32_t lcnt[EPT], lfirst[EPT], esc[EPT], npart = 0;
#pragma unroll
        for (int r = 0; r < EPT; ++r) {
            const uint32_t u = base + (uint32_t)(t * EPT + r);
            lfirst[r] = u < len ? A.pool[off + u] & ~kLeafTag : 0xFFFFFFFFu;
        }
#pragma unroll
        for (int r = 0; r < EPT; ++r) {
            const bool leaf = lfirst[r] != 0xFFFFFFFFu;
            lcnt[r] = leaf ? A.nd_count[lfirst[r]] : 0u;
            lfirst[r] = leaf ? A.nd_first[lfirst[r]] : 0u;
            npart += lcnt[r];
        }
        uint32_t total;
        uint32_t es = block_scan1<CB>(npart, &total, sm.w);
#pragma unroll
        for (int r = 0; r < EPT; ++r) {
            esc[r] = es;
            es += lcnt[r];
        }
        // each thread's EPT consecutive slots in one vector store (no bank conflicts)
        store_entries<EPT>(s_ef + t * EPT, lfirst);
        store_entries<EPT>(s_es + t * EPT, esc);
        __syncthreads();
        for (uint32_t c0 = 0; c0 < total; c0 += kCJ) {
            const uint32_t m = total - c0 < (uint32_t)kCJ ? total - c0 : (uint32_t)kCJ;
            if (c0 > 0) __syncthreads();  // previous tile fully consumed
            for (uint32_t k = t; k < m; k += CB) {
                const uint32_t item = c0 + k;
                const int src = owner_chunk<SM::kCL>(s_es, item);
                const uint32_t p = s_ef[src] + (item - s_es[src]);
                const float4 h = A.pf_hi[p], l = A.pf_lo[p];
                s_j[k] = make_float4((h.x - gch.x) + (l.x - gcl.x), (h.y - gch.y) + (l.y - gcl.y),
                                     (h.z - gch.z) + (l.z - gcl.z), h.w);
            }
            __syncthreads();
            clear();
#pragma unroll kUnrollEpj
            for (int k = kbeg; k < (int)m; k += nsl) {
                const float4 j = s_j[k];
                if (K & 1) {
                    const float dx = j.x - xi[K - 1], dy = j.y - yi[K - 1], dz = j.z - zi[K - 1];
                    const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, e2[K - 1])));
                    const float ri = rsqrtf(r2);
                    const float mri = j.w * ri;
                    const float mri3 = mri * (ri * ri);
                    sax[K - 1] = fmaf(mri3, dx, sax[K - 1]);
                    say[K - 1] = fmaf(mri3, dy, say[K - 1]);
                    saz[K - 1] = fmaf(mri3, dz, saz[K - 1]);
                    spp[K - 1] -= mri;
                }
                if (KP > 0) {
                    const f2 jx = f2_bc(j.x), jy = f2_bc(j.y), jz = f2_bc(j.z), jm = f2_bc(j.w);
#pragma unroll
                    for (int h = 0; h < KP; ++h) {
                        const f2 dx = f2_sub<true>(jx, xp[h]), dy = f2_sub<true>(jy, yp[h]), dz = f2_sub<true>(jz, zp[h]);
                        const f2 r2 = f2_fma<true>(dx, dx, f2_fma<true>(dy, dy, f2_fma<true>(dz, dz, ep[h])));
                        const f2 ri = f2_rsqrt(r2);
                        const f2 mri = f2_mul<true>(jm, ri);
                        const f2 mri3 = f2_mul<true>(mri, f2_mul<true>(ri, ri));
                        pax[h] = f2_fma<true>(mri3, dx, pax[h]);
                        pay[h] = f2_fma<true>(mri3, dy, pay[h]);
                        paz[h] = f2_fma<true>(mri3, dz, paz[h]);
                        pp[h] = f2_sub<true>(pp[h], mri);
                    }
                }
            }
            fold();
        }
        __syncthreads();  // chunk buffers are rewritten next
    }
    // ---- combine slices and write back.  A slice's Kahan pair (s, c) is the
    // double-float s + (-c); the pairs of a row's slices are added with exact
    // two-sums in FP32 and each component turned into FP64 once (FP64 is a
    // narrow pipe on this part).  A thread adds one component of one row, and
    // where those are fewer than the threads, every parts-th slice of it, the
    // parts meeting by shuffles (a thread per row, four components and up to
    // 32 slices each, took a fifth of the time of groups of 16 particles; 256
    // clusters at n_grp 64: 6.02 -> 5.76 ms).  The potential's self term is removed with the
    // value the list's own entry contributed, m_i rsqrt(eps_i^2) in FP32, so
    // that the two cancel.
    const int rows = P * K;  // i-slots of this round: row r = ip + q P
    const int items = 4 * rows;
    int parts = 1;
    while (parts < 32 && 2 * parts <= nsl && 2 * parts * items <= CB) parts *= 2;
    __syncthreads();  // every thread's Kahan sums are final
    for (int it0 = 0; it0 < items; it0 += CB / parts) {  // one turn if parts > 1
        const int it = it0 + t / parts, pt = t & (parts - 1);
        const int c = it / rows, r = it - c * rows;
        const uint32_t i = ib + (uint32_t)r;
        const bool valid = it < items && i < ni;
        float hi = 0.0f, lo = 0.0f;
        if (valid) {
            const int q = r / P, ipr = r - q * P;
            const float* sk = s_k + ((q * 4 + c) * 2) * CB + ipr;  // of slice s2: sk[s2 P], its compensation CB on
            for (int s2 = pt; s2 < nsl; s2 += parts) {
                two_sum_acc(hi, lo, sk[s2 * P]);
                lo -= sk[s2 * P + CB];
            }
        }
        for (int o = parts >> 1; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xFFFFFFFFu, hi, o), l2 = __shfl_xor_sync(0xFFFFFFFFu, lo, o);
            two_sum_acc(hi, lo, h2);
            lo += l2;
        }
        if (valid && pt == 0) {
            const uint32_t p = gf + i;
            if (c == 3) two_sum_acc(hi, lo, A.pf_hi[p].w * rsqrtf(A.pf_lo[p].w));
            double* out = c == 0 ? A.ax : c == 1 ? A.ay : c == 2 ? A.az : A.pot;
            out[p] = (double)hi + (double)lo;
        }
    }
    __syncthreads();
}

// Forces on the particles of group g, with the whole CTA.
template <bool QUAD, int EPT, int CB, int KMAX, int WARPS>
__device__ __forceinline__ void force_group(const ForceArgs& A, uint32_t g, F32Shared<QUAD, EPT, CB, KMAX>& sm) {
    const uint32_t ni = A.g_count[g], gf = A.g_first[g];
    const unsigned long long off = A.g_off[g];
    const uint32_t len = A.g_len[g], nspj = A.g_nspj[g];
    const float4 gch = A.g_ch[g], gcl = A.g_cl[g];
    for (uint32_t ib = 0; ib < ni;) {
        const GroupPlan pl = plan_group<CB, KMAX>(ni - ib);
        if (pl.K == 1) {
            force_round_f32<QUAD, 1, EPT, CB, KMAX, WARPS>(A, gf, ni, off, nspj, len, gch, gcl, pl.P, pl.nsl, ib, sm);
        } else if (KMAX >= 5 && pl.K == 5) {
            if constexpr (KMAX >= 5)
                force_round_f32<QUAD, 5, EPT, CB, KMAX, WARPS>(A, gf, ni, off, nspj, len, gch, gcl, pl.P, pl.nsl, ib, sm);
        } else if (KMAX >= 4 && pl.K == 3) {
            if constexpr (KMAX >= 4)
                force_round_f32<QUAD, 3, EPT, CB, KMAX, WARPS>(A, gf, ni, off, nspj, len, gch, gcl, pl.P, pl.nsl, ib, sm);
        } else if (KMAX == 2 || pl.K == 2) {
            force_round_f32<QUAD, 2, EPT, CB, KMAX, WARPS>(A, gf, ni, off, nspj, len, gch, gcl, pl.P, pl.nsl, ib, sm);
        } else {
            if constexpr (KMAX >= 4)
                force_round_f32<QUAD, 4, EPT, CB, KMAX, WARPS>(A, gf, ni, off, nspj, len, gch, gcl, pl.P, pl.nsl, ib, sm);
        }
        ib += (uint32_t)(pl.P * pl.K);
    }
}

// WARPS per SM.  Quadrupoles: 16 (four 128-thread CTAs, 128 registers a
// thread; with five they spill).  Monopoles: 24 (six CTAs, 80 registers): a
// third of their time on small groups is the latency of staging, and more
// CTAs hide it (256 clusters, n_grp 64: 5.76 ms with four CTAs, 5.27 with five,
// 5.15 with six; 3M clumpy particles, n_grp 256: 2.50, 2.46 and 2.45); but 16
// where the groups are few for their size, so that the last ones' own time
// counts (24 / 16 warps: 16 steps of 2001 particles, n_grp 64, 2.52 / 2.41 ms;
// Plummer, n_grp 16 1117 groups 29 / 31 us; n_grp 64 1835 groups 88 / 84, 6754 283 /
// 291; n_grp 128 6936 groups 574 / 557; n_grp 512 6668 groups 2.72 / 2.56 ms; n_grp
// 1024 278 groups 1.25 / 0.99 ms).
constexpr int64_t kFewGroups = 8192;
static bool few_groups(const fdps_tree* t, const fdps_psys* ps) {
    const int64_t w = std::min<int64_t>(t->p.n_grp, ps->n / ps->n_sys);
    return ps->n <= 13 * w * w && t->est_groups <= kFewGroups;
}
template <bool QUAD, int EPT, int CB, int KMAX, int WARPS>
__global__ void __launch_bounds__(CB, 32 * WARPS / CB) k_force_f32(ForceArgs A) {
    __shared__ F32Shared<QUAD, EPT, CB, KMAX> sm;
    __shared__ uint32_t s_g;
    DevState* st = A.st;
    // lists cut short by a buffer overflow may point past the pool: no work
    // (a step replayed from a graph is redone by the host)
    if (st->overflow & kStepInvalid) return;
    const uint32_t ngroups = (uint32_t)st->n_groups;
    for (;;) {
        if (threadIdx.x == 0) s_g = atomicAdd(&st->force_counter, 1u);
        __syncthreads();
        const uint32_t g = s_g;
        if (g >= ngroups) break;
        force_group<QUAD, EPT, CB, KMAX, WARPS>(A, g, sm);
    }
}

// ---------------------------------------------------------------- FP64
// One cluster of CL = 8 CTAs (B = 128 threads each) per i-group, or one CTA of 64
// threads where groups hold few particles (compute_forces).  Bound by the
// FP64 pipe (two lanes per SM and clock: a warp instruction takes it for 16
// clocks whatever its active lanes), so the split is the one that costs the
// pipe least: thread t of a CTA owns K <= 4 i-particles (i = t % P + k P) and
// slice t / P of the CTA's list entries, (K, P, slices) minimising the warps
// times K per entry (plan_f64: 9 in 10 lanes busy on groups of 30 to 128
// particles, where one warp per group kept 6 in 10 busy).  The entries of a
// list go to the cluster's CTAs in turn (entry u to CTA u % CL), so every
// CTA has the same mix of cells and opened leaves, and a group of a few
// thousand entries takes a twelfth of the time one CTA would need: with one
// warp or CTA per group the last groups of a 10^5-particle system left most
// of the SMs idle.  Entries are staged in shared memory by chunk.  Slices
// and CTAs are summed in a fixed order, through distributed shared memory.
// Plummer N = 100,003, quadrupoles, n_grp 128: 56.4 -> 19.4 ms for the
// whole force calculation (one warp per group before).
// (CL CTAs per cluster of B threads; a CTA stages B list entries per chunk, one
// per thread, and B leaf particles per tile)
constexpr int kK64 = 4;  // most i-particles per thread

template <int B>
struct F64Shared {
    dvec4 spj[B];            // centre of mass and -M
    double q[B][6];          // quadrupole (xx yy zz xy xz yz)
    dvec4 j[B];
    uint32_t ef[B];
    uint32_t es[B];
    uint32_t w[2 * (B / 32)];
    double part[kK64 * 4][B];  // a thread's sums: row q * 4 + component
    double row[4][kK64 * B];   // the CTA's sums of its i-rows
    uint32_t g;
};

template <int CL>
__device__ __forceinline__ void group_barrier() {
    if (CL > 1)
        cluster_barrier();
    else
        __syncthreads();
}

// (K, P, slices) of ni i-particles: least FP64 pipe time K * warps / slices
// per list entry; more slices on ties.
template <int B>
__device__ __forceinline__ GroupPlan plan_f64(uint32_t ni) {
    GroupPlan best{kK64, B, 1};  // more than a CTA holds: rounds
    float bc = 3.0e38f;
#pragma unroll
    for (int K = 1; K <= kK64; ++K) {
        const int P = (int)((ni + K - 1) / K);
        if (P > B) continue;
        const int nsl = B / P;
        const float c = (float)(K * ((P * nsl + 31) / 32)) / (float)nsl;
        if (c < bc - 1e-6f) {
            bc = c;
            best = GroupPlan{K, P, nsl};
        }
    }
    return best;
}

// One round of i-particles (ib .. ib + P K - 1 of the group) with K per
// thread, over this CTA's share of the list; called by the whole cluster.
template <bool QUAD, int CL, int B, int K>
__device__ __forceinline__ void force_round_f64(const ForceArgs& A, uint32_t gf, uint32_t ni,
                                                unsigned long long off, uint32_t len, int P, int nsl,
                                                uint32_t ib, uint32_t rank, F64Shared<B>& sm) {
    const int t = threadIdx.x;
    const int ip = t % P, sl = t / P;
    const bool on = sl < nsl;
    double xi[K], yi[K], zi[K], e2[K], ax[K], ay[K], az[K], pp[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        const uint32_t i = ib + (uint32_t)(ip + q * P);
        const bool iv = on && i < ni;
        const uint32_t p = gf + (iv ? i : 0u);
        const double e = iv ? A.peps[p] : 1.0;
        xi[q] = A.px[p];
        yi[q] = A.py[p];
        zi[q] = A.pz[p];
        e2[q] = e * e;
        ax[q] = ay[q] = az[q] = pp[q] = 0.0;
    }
    const int kbeg = on ? sl : 0x3FFFFFFF;
    // entries rank, rank + CL, ... of the list are this CTA's
    const uint32_t mine = len > rank ? (len - rank + CL - 1) / CL : 0u;
    for (uint32_t base = 0; base < mine; base += B) {
        const uint32_t u = base + t;
        const uint32_t ent = u < mine ? A.pool[off + rank + (unsigned long long)u * CL] : 0xFFFFFFFFu;
        const bool leaf = ent != 0xFFFFFFFFu && (ent & kLeafTag);
        const bool spj = ent != 0xFFFFFFFFu && !(ent & kLeafTag);
        const uint32_t node = ent & ~kLeafTag;
        const uint32_t cnt = leaf ? A.nd_count[node] : 0u;
        uint32_t rs, es, ns, total;
        block_scan2<B>(spj ? 1u : 0u, cnt, &rs, &es, &ns, &total, sm.w);
        if (spj) {
            const dvec4 c = A.nd_com[node];
            sm.spj[rs] = make_dvec4(c.x, c.y, c.z, -c.w);
            if (QUAD)
#pragma unroll
                for (int k = 0; k < 6; ++k) sm.q[rs][k] = A.nd_quad[6 * (int64_t)node + k];
        }
        sm.ef[t] = leaf ? A.nd_first[node] : 0u;
        sm.es[t] = es;
        __syncthreads();
        for (int k = kbeg; k < (int)ns; k += nsl) {
            const dvec4 c = sm.spj[k];
            double qxx, qyy, qzz, qxy, qxz, qyz;
            if (QUAD) {
                qxx = sm.q[k][0];
                qyy = sm.q[k][1];
                qzz = sm.q[k][2];
                qxy = sm.q[k][3];
                qxz = sm.q[k][4];
                qyz = sm.q[k][5];
            }
#pragma unroll
            for (int q = 0; q < K; ++q) {
                const double rx = xi[q] - c.x, ry = yi[q] - c.y, rz = zi[q] - c.z;
                const double R2 = fma(rx, rx, fma(ry, ry, fma(rz, rz, e2[q])));
                const double Ri = rsqrt(R2);
                const double Ri2 = Ri * Ri;
                if (QUAD) {
                    // v = r / R^2 stands for r in the quadrupole, so that no power
                    // beyond R^-3 appears: like the monopole's m / R^3 the term
                    // holds from R = 1e-102 to 1e102 (regrouped around R^-5 as in
                    // the FP32 kernel, one operation less, it vanished from 1e65 on)
                    const double vx = rx * Ri2, vy = ry * Ri2, vz = rz * Ri2;
                    const double Qvx = fma(qxx, vx, fma(qxy, vy, qxz * vz));
                    const double Qvy = fma(qxy, vx, fma(qyy, vy, qyz * vz));
                    const double Qvz = fma(qxz, vx, fma(qyz, vy, qzz * vz));
                    const double rQv = fma(rx, Qvx, fma(ry, Qvy, rz * Qvz));
                    const double w = rQv * Ri2;
                    const double hh = fma(-2.5, w, c.w);
                    const double Ri3 = Ri2 * Ri;
                    ax[q] = fma(Ri3, fma(hh, rx, Qvx), ax[q]);
                    ay[q] = fma(Ri3, fma(hh, ry, Qvy), ay[q]);
                    az[q] = fma(Ri3, fma(hh, rz, Qvz), az[q]);
                    pp[q] = fma(Ri, fma(2.0, w, hh), pp[q]);
                } else {
                    const double nMRi = c.w * Ri;
                    const double nMRi3 = nMRi * Ri2;
                    ax[q] = fma(nMRi3, rx, ax[q]);
                    ay[q] = fma(nMRi3, ry, ay[q]);
                    az[q] = fma(nMRi3, rz, az[q]);
                    pp[q] += nMRi;
                }
            }
        }
        for (uint32_t c0 = 0; c0 < total; c0 += B) {
            const uint32_t m = total - c0 < (uint32_t)B ? total - c0 : (uint32_t)B;
            if (c0 > 0) __syncthreads();  // previous tile fully consumed
            for (uint32_t k = t; k < m; k += B) {
                const uint32_t item = c0 + k;
                const int src = owner_chunk<B>(sm.es, item);
                const uint32_t p = sm.ef[src] + (item - sm.es[src]);
                sm.j[k] = make_dvec4(A.px[p], A.py[p], A.pz[p], A.pm[p]);
            }
            __syncthreads();
            for (int k = kbeg; k < (int)m; k += nsl) {
                const dvec4 j = sm.j[k];
#pragma unroll
                for (int q = 0; q < K; ++q) {
                    const double dx = j.x - xi[q], dy = j.y - yi[q], dz = j.z - zi[q];
                    const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, e2[q])));
                    const double ri = rsqrt(r2);
                    const double mri = j.w * ri;
                    const double mri3 = mri * ri * ri;
                    ax[q] = fma(mri3, dx, ax[q]);
                    ay[q] = fma(mri3, dy, ay[q]);
                    az[q] = fma(mri3, dz, az[q]);
                    pp[q] -= mri;
                }
            }
        }
        __syncthreads();  // chunk buffers are rewritten next
    }
    // slices, then the cluster's CTAs, in order
#pragma unroll
    for (int q = 0; q < K; ++q) {
        sm.part[q * 4 + 0][t] = ax[q];
        sm.part[q * 4 + 1][t] = ay[q];
        sm.part[q * 4 + 2][t] = az[q];
        sm.part[q * 4 + 3][t] = pp[q];
    }
    __syncthreads();
    const int rows = P * K;
    for (int k = t; k < 4 * rows; k += B) {
        const int c = k / rows, r = k - c * rows;
        const int q = r / P, ipr = r - q * P;
        double v = 0.0;
        for (int s2 = 0; s2 < nsl; ++s2) v += sm.part[q * 4 + c][s2 * P + ipr];
        sm.row[c][r] = v;
    }
    group_barrier<CL>();  // every CTA's rows are written
    // each CTA finishes every CL-th value
    for (int k = t * CL + (int)rank; k < 4 * rows; k += B * CL) {
        const int r = k >> 2, c = k & 3;
        const uint32_t i = ib + (uint32_t)r;
        if (i >= ni) continue;
        double v = 0.0;
#pragma unroll
        for (int b = 0; b < CL; ++b) v += CL > 1 ? ld_peer_f64(peer_smem(&sm.row[c][r], (uint32_t)b)) : sm.row[c][r];
        const uint32_t p = gf + i;
        if (c == 0)
            A.ax[p] = v;
        else if (c == 1)
            A.ay[p] = v;
        else if (c == 2)
            A.az[p] = v;
        else
            A.pot[p] = v + A.pm[p] / A.peps[p];  // without the particle's own entry
    }
    group_barrier<CL>();  // the rows have been read: they may be rewritten
}

template <bool QUAD, int CL, int B>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(B, 512 / B) k_force_f64(ForceArgs A) {
    extern __shared__ __align__(32) unsigned char f64_smem[];
    F64Shared<B>& sm = *reinterpret_cast<F64Shared<B>*>(f64_smem);
    DevState* st = A.st;
    if (st->overflow & kStepInvalid) return;  // as in the FP32 kernel
    const uint32_t ngroups = (uint32_t)st->n_groups;
    const uint32_t rank = CL > 1 ? cluster_rank() : 0u;
    for (;;) {
        if (rank == 0 && threadIdx.x == 0) sm.g = atomicAdd(&st->force_counter, 1u);
        group_barrier<CL>();
        const uint32_t g = CL > 1 ? ld_peer_u32(peer_smem(&sm.g, 0)) : sm.g;
        group_barrier<CL>();  // read by all before it is rewritten or its CTA ends
        if (g >= ngroups) break;
        const uint32_t ni = A.g_count[g], gf = A.g_first[g];
        const unsigned long long off = A.g_off[g];
        const uint32_t len = A.g_len[g];
        for (uint32_t ib = 0; ib < ni;) {
            const GroupPlan pl = plan_f64<B>(ni - ib);
            if (pl.K == 1)
                force_round_f64<QUAD, CL, B, 1>(A, gf, ni, off, len, pl.P, pl.nsl, ib, rank, sm);
            else if (pl.K == 2)
                force_round_f64<QUAD, CL, B, 2>(A, gf, ni, off, len, pl.P, pl.nsl, ib, rank, sm);
            else if (pl.K == 3)
                force_round_f64<QUAD, CL, B, 3>(A, gf, ni, off, len, pl.P, pl.nsl, ib, rank, sm);
            else
                force_round_f64<QUAD, CL, B, 4>(A, gf, ni, off, len, pl.P, pl.nsl, ib, rank, sm);
            ib += (uint32_t)(pl.P * pl.K);
        }
    }
}

}  // namespace

// One resident wave of FP32 force CTAs of the given shape (chunk CE
// entries, CB threads, at most KMAX i-particles a thread).
template <bool QUAD, int CE, int CB, int KMAX, int WARPS = QUAD ? 16 : 24>
void launch_f32(const ForceArgs& A, fdps_ctx* ctx, cudaStream_t s) {
    constexpr int EPT = CE / CB;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_force_f32<QUAD, EPT, CB, KMAX, WARPS>, CB, 0) !=
            cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    k_force_f32<QUAD, EPT, CB, KMAX, WARPS><<<per_sm * ctx->sm_count, CB, 0, s>>>(A);
}

template <bool QUAD, int CE>
void launch_f32_shape(const ForceArgs& A, fdps_ctx* ctx, cudaStream_t s, int cb, int kmax, bool few) {
    if (cb == 64) {
        if (kmax == 2)
            launch_f32<QUAD, CE, 64, 2>(A, ctx, s);
        else if (kmax == 4)
            launch_f32<QUAD, CE, 64, 4>(A, ctx, s);
        else
            launch_f32<QUAD, CE, 64, 5>(A, ctx, s);
    } else if (cb == 256) {
        launch_f32<QUAD, CE, 256, 2>(A, ctx, s);  // 256 x 4 does not fit static shared memory
    } else {
        if (kmax == 2)
            launch_f32<QUAD, CE, 128, 2>(A, ctx, s);
        else if (kmax == 4)
            launch_f32<QUAD, CE, 128, 4>(A, ctx, s);
        else if (!QUAD && few)
            launch_f32<QUAD, CE, 128, 5, 16>(A, ctx, s);
        else
            launch_f32<QUAD, CE, 128, 5>(A, ctx, s);
    }
}

// One resident wave of clusters of CL FP64 force CTAs of B threads.
template <bool QUAD, int CL, int B>
int launch_f64(const ForceArgs& A, fdps_ctx* ctx, cudaStream_t s) {
    const int bytes = (int)sizeof(F64Shared<B>);
    FDPS_CUDA_TRY(ctx, cudaFuncSetAttribute(k_force_f64<QUAD, CL, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_force_f64<QUAD, CL, B>, B, bytes) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    const int clusters = per_sm * ctx->sm_count / CL;
    k_force_f64<QUAD, CL, B><<<(clusters > 0 ? clusters : 1) * CL, B, bytes, s>>>(A);
    return FDPS_OK;
}

ForceArgs force_args(fdps_tree* t, fdps_psys* ps) {
    const int c = ps->cur;
    ForceArgs A;
    A.st = t->st;
    A.g_first = t->g_first;
    A.g_count = t->g_count;
    A.g_off = t->g_off;
    A.g_len = t->g_len;
    A.g_nspj = t->g_nspj;
    A.g_ch = t->g_ch;
    A.g_cl = t->g_cl;
    A.pool = t->pool;
    A.nd_first = t->nd_first;
    A.nd_count = t->nd_count;
    A.nd_f = t->nd_f;
    A.nd_fq0 = t->nd_fq0;
    A.nd_fq1 = t->nd_fq1;
    A.nd_com = t->nd_com;
    A.nd_quad = t->nd_quad;
    A.pf_hi = t->pf_hi;
    A.pf_lo = t->pf_lo;
    A.px = ps->x[c];
    A.py = ps->y[c];
    A.pz = ps->z[c];
    A.pm = ps->m[c];
    A.peps = ps->eps[c];
    A.ax = ps->ax;
    A.ay = ps->ay;
    A.az = ps->az;
    A.pot = ps->pot;
    return A;
}

int compute_forces(fdps_tree* t, fdps_psys* ps, int spj_kind) {
    fdps_ctx* ctx = t->ctx;
    const ForceArgs A = force_args(t, ps);
    const bool quad = spj_kind == FDPS_GRAV_SPJ_QUAD;
    cudaStream_t s = ctx->stream;
    if (t->p.precision == FDPS_FP64) {
        // Groups of few particles (n_grp, or whole systems of an ensemble) take
        // one CTA of 64 threads each: a cluster's barriers and its sums over 8 x
        // 128 slices outlast their lists.  Up to 8 particles always; up to 16 and
        // 32 where there are enough groups to keep the SMs busy to the end.
        // Plummer, monopoles, cluster / CTA: n_grp 8: 0.080 / 0.074 ms at 1000
        // particles, 9.00 / 4.79 at 10^5; n_grp 16: 0.27 / 0.32 at 5000, 1.25 /
        // 1.00 at 20000; n_grp 32: 1.10 / 1.40 at 20000, 28.4 / 26.0 at 400000; n_grp
        // 64: 29.5 / 29.6.  (One warp per group, before both: 5.9 ms at 10^5 and
        // n_grp 8, 40.6 at 400000 and n_grp 64.)
        const int64_t w = std::min<int64_t>(t->p.n_grp, ps->n / ps->n_sys);
        const bool cta = w <= 8 || (w <= 16 && ps->n >= (1 << 14)) || (w <= 32 && ps->n >= (1 << 17));
        const int rc = cta    ? (quad ? launch_f64<true, 1, 64>(A, ctx, s) : launch_f64<false, 1, 64>(A, ctx, s))
                       : quad ? launch_f64<true, 8, 128>(A, ctx, s)
                              : launch_f64<false, 8, 128>(A, ctx, s);
        if (rc) return rc;
    } else {
        // tile depth: list entries staged per chunk (0 = default 512); block
        // shape: threads per CTA (0 = 128) and i-particles per thread (0 = 5)
        const bool shallow = t->p.tile_depth == 256;
        const int cb = t->p.block ? t->p.block : 128;
        const int kmax = t->p.i_per_thread ? t->p.i_per_thread : 5;
        const bool few = few_groups(t, ps);
        if (quad) {
            if (shallow)
                launch_f32_shape<true, 256>(A, ctx, s, cb, kmax, few);
            else
                launch_f32_shape<true, 512>(A, ctx, s, cb, kmax, few);
        } else {
            if (shallow)
                launch_f32_shape<false, 256>(A, ctx, s, cb, kmax, few);
            else
                launch_f32_shape<false, 512>(A, ctx, s, cb, kmax, few);
        }
    }
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

}  // namespace fdps
