/* fdps_user_force.cuh -- user interaction laws over the library's lists.
 *
 * FDPS lets its user write the interaction law: the force kernels passed
 * to calcForceAllAndWriteBack take an array of i-particles, an array of
 * j-particles (or superparticles) and the force accumulators (Sect. 2.2).
 * This header is the GPU form of that contract.  The library builds the
 * tree and the interaction lists (fdps_tree_build_lists, or any force
 * calculation) and describes them by a view (fdps_tree_get_view); the
 * template below, compiled into the user's own CUDA code, walks every
 * group's list, stages the list entries in shared memory and calls the
 * user's functors:
 *
 *   struct Force { ...; __device__ void clear(); };
 *   struct Law {
 *     __device__ void operator()(const fdps_user::Epi& i,
 *                                const fdps_user::Epj* j, int nj, Force& f) const;
 *     __device__ void operator()(const fdps_user::Epi& i,
 *                                const fdps_user::Spj* j, int nj, Force& f) const;
 *   };
 *   fdps_tree_view v;  fdps_tree_get_view(tree, ps, &v);
 *   fdps_user::calc_force(v, Law{}, Law{}, out, stream);
 *
 * Each thread owns one i-particle; it calls the functors with tiles of up
 * to 64 particles of opened leaves (EPJ) and up to 32 superparticles (SPJ),
 * which together make the i-particle's group's whole list, the superparticles
 * and the opened leaves each in list order, in turn: in which order calls
 * with cells and calls with particles follow one another, and how many
 * entries a call gets, is the library's choice and may change.  Arrays of Epj
 * and Spj are to be indexed as such (they are 16 and 48 bytes, 16-byte
 * aligned, the last 8 bytes of an Spj without meaning).
 * The particle itself is among its EPJ (zero separation): the law decides
 * what that term contributes.  Positions are FP32 relative to the group's
 * centre, formed from hi/lo parts as in the built-in kernel.  out[row] gets
 * the Force of the particle in row `row` of the caller's arrays (cleared,
 * then accumulated by the functors), for every particle.  The work is
 * queued on `stream`; calc_force returns the launch status.
 *
 * The device part of this header (the types and calc_force_body) also
 * compiles under NVRTC, where fdps_user_law_compile builds user laws given
 * as source text at run time.
 */
#pragma once

#ifndef __CUDACC_RTC__
#include <cstdint>
#include <cuda_runtime.h>
#endif

#include "fdps_gpu.h"

namespace fdps_user {

// i-particle: position relative to its group's centre, softening eps^2 and
// the caller's row of the particle
struct Epi {
    float x, y, z, eps2;
    uint32_t row;
};
// particle of an opened leaf, relative to the group centre
struct __align__(16) Epj {
    float x, y, z, m;
};
// superparticle: a cell's centre of mass relative to the group centre, its
// mass and traceless quadrupole about the centre of mass (zero for a
// monopole tree).  Both list types are aligned for 16-byte loads.
struct __align__(16) Spj {
    float x, y, z, m;
    float qxx, qyy, qzz, qxy, qxz, qyz;
};

namespace detail {

constexpr int kThreads = 32;  // threads of a block (one warp), and list entries per step
constexpr int kSlots = 8;     // blocks sharing a group's i-particles (grid y)
constexpr int kEpjCall = 64;  // most leaf particles per functor call

__device__ __forceinline__ float4 ld4(const float* p, uint64_t i) {
    return reinterpret_cast<const float4*>(p)[i];
}

// The walk of the view's groups by a grid (any x, any y) of blocks of
// kThreads: block (x, y) takes groups x, x + gridDim.x, ... and of each the
// i-particles kThreads y .. + kThreads - 1 (and on by kThreads gridDim.y),
// one per thread.  The block stages kThreads list entries at a time.  The law's own instructions bound it (issue slots 74 % busy), so
// what counts is that every SM has warps with i-particles until the end: one
// block per group and 32 i-particles, started by the hardware as others
// finish, where a fixed share of the groups for each warp of one resident
// wave, eight passes over the list for a group of 256, left most of the SMs
// idle behind the warps with the large groups.  One warp a block: with two or
// four, groups of 30 particles leave warps that only wait at the barriers.
// Gravity with quadrupoles, lists and law on one stream: 2^20 Hernquist
// particles, n_grp 256, 13.9 ms before, 7.8 with 32 threads, 8.2 with 64, 8.0 with
// 128; 500,000 Plummer particles with monopoles, n_grp 64: 5.6, 4.5, 6.5 and 5.0
// ms.  (Calls of several contexts that overlap had filled the idle SMs with one
// another's work: 8.4 ms a call before, 7.7 now.)
template <class Force, class FEpj, class FSpj>
__device__ __forceinline__ void calc_force_body(const fdps_tree_view& v, const FEpj& f_epj,
                                                const FSpj& f_spj, Force* out) {
    __shared__ Spj s_spj[kThreads];
    __shared__ Epj s_epj[kEpjCall];
    __shared__ uint32_t s_first[kThreads];
    __shared__ uint32_t s_start[kThreads];
    const int t = threadIdx.x;
    const uint32_t lt = (1u << t) - 1u;
    for (int64_t g = blockIdx.x; g < v.n_groups; g += gridDim.x) {
        const uint32_t gf = v.g_first[g], ni = v.g_count[g];
        const unsigned long long off = v.g_off[g];
        const uint32_t len = v.g_len[g];
        const float4 ch = ld4(v.g_ch, (uint64_t)g), cl = ld4(v.g_cl, (uint64_t)g);
        // steps of kThreads entries, the first nsp of them with superparticles
        // (a list holds its superparticles before its leaves): every lane
        // probes one of 32 steps until none is left between two of them
        const uint32_t steps = (len + kThreads - 1) / kThreads;
        uint32_t nsp = 0;
        for (uint32_t n = steps; n > 0;) {
            const uint32_t stride = (n + 31) / 32, at = t * stride;
            const bool sp = at < n && !(v.pool[off + (uint64_t)(nsp + at) * kThreads] & v.leaf_tag);
            const uint32_t c = __popc(__ballot_sync(0xFFFFFFFFu, sp));
            if (c == 0) break;
            const uint32_t past = (c - 1) * stride + 1, end = c * stride < n ? c * stride : n;
            nsp += past;
            n = end - past;
        }
        for (uint32_t ib = blockIdx.y * kThreads; ib < ni; ib += kThreads * gridDim.y) {
            const uint32_t i = ib + t;
            const bool act = i < ni;
            Epi epi{0.f, 0.f, 0.f, 1.f, 0u};
            if (act) {
                const float4 h = ld4(v.pf_hi, gf + i), l = ld4(v.pf_lo, gf + i);
                epi.x = (h.x - ch.x) + (l.x - cl.x);
                epi.y = (h.y - ch.y) + (l.y - cl.y);
                epi.z = (h.z - ch.z) + (l.z - cl.z);
                epi.eps2 = l.w;
                epi.row = v.id[gf + i];
            }
            Force f;
            f.clear();
            // steps with superparticles and steps with leaves in turn, in
            // proportion: a law's plain sums round with every entry, by more
            // the larger they are, and either kind last costs up to half as
            // much error again
            uint32_t ks = 0, kl = 0;
            while (ks + kl < steps) {
                const bool cells = kl == steps - nsp || (ks < nsp && (uint64_t)ks * (steps - nsp) <= (uint64_t)kl * nsp);
                const uint32_t u = (cells ? ks++ : nsp + kl++) * kThreads + t;
                const bool valid = u < len;
                const uint32_t e = valid ? v.pool[off + u] : 0u;
                const bool leaf = valid && (e & v.leaf_tag);
                const bool spj = valid && !leaf;
                const uint32_t node = e & ~v.leaf_tag;
                // ranks of the superparticles and of the leaves' particles
                // in this step
                const uint32_t smask = __ballot_sync(0xFFFFFFFFu, spj);
                const uint32_t cnt = leaf ? v.nd_count[node] : 0u;
                uint32_t inc = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                    if (t >= o) inc += x;
                }
                const uint32_t nspj = __popc(smask), total = __shfl_sync(0xFFFFFFFFu, inc, 31);
                __syncwarp();  // the previous step's tiles are consumed
                if (spj) {
                    const float4 fh = ld4(v.nd_f, 2ull * node), fl = ld4(v.nd_f, 2ull * node + 1);
                    Spj s;
                    s.x = (fh.x - ch.x) + (fl.x - cl.x);
                    s.y = (fh.y - ch.y) + (fl.y - cl.y);
                    s.z = (fh.z - ch.z) + (fl.z - cl.z);
                    s.m = fh.w;
                    s.qxx = s.qyy = s.qzz = s.qxy = s.qxz = s.qyz = 0.f;
                    if (v.quadrupole) {
                        const float4 q0 = ld4(v.nd_fq0, node);
                        const float2 q1 = reinterpret_cast<const float2*>(v.nd_fq1)[node];
                        s.qxx = q0.x;
                        s.qyy = q0.y;
                        s.qzz = q0.z;
                        s.qxy = q0.w;
                        s.qxz = q1.x;
                        s.qyz = q1.y;
                    }
                    s_spj[__popc(smask & lt)] = s;
                }
                s_first[t] = leaf ? v.nd_first[node] : 0u;
                s_start[t] = inc - cnt;
                __syncwarp();
                if (act && nspj > 0) f_spj(epi, &s_spj[0], (int)nspj, f);
                for (uint32_t c0 = 0; c0 < total; c0 += kEpjCall) {
                    const uint32_t m = total - c0 < (uint32_t)kEpjCall ? total - c0 : (uint32_t)kEpjCall;
                    if (c0 > 0) __syncwarp();
                    for (uint32_t k = t; k < m; k += kThreads) {
                        // the owning entry: the last one whose start <= item
                        // (entries with no particles share the next one's start)
                        const uint32_t item = c0 + k;
                        int src = 0;
#pragma unroll
                        for (int step = kThreads / 2; step > 0; step >>= 1)
                            if (s_start[src + step] <= item) src += step;
                        const uint32_t p = s_first[src] + (item - s_start[src]);
                        const float4 h = ld4(v.pf_hi, p), l = ld4(v.pf_lo, p);
                        s_epj[k] = Epj{(h.x - ch.x) + (l.x - cl.x), (h.y - ch.y) + (l.y - cl.y),
                                       (h.z - ch.z) + (l.z - cl.z), h.w};
                    }
                    __syncwarp();
                    if (act) f_epj(epi, &s_epj[0], (int)m, f);
                }
            }
            if (act) out[epi.row] = f;
            __syncwarp();  // the tiles are rewritten for the next i-particles
        }
    }
}

template <class Force, class FEpj, class FSpj>
__global__ void __launch_bounds__(kThreads)
    calc_force_kernel(fdps_tree_view v, FEpj f_epj, FSpj f_spj, Force* out) {
    calc_force_body<Force>(v, f_epj, f_spj, out);
}

}  // namespace detail

#ifndef __CUDACC_RTC__

// Launch the user laws over every group of the view (see the top of this
// file).  `out` is a device array of v.n Force values.
template <class Force, class FEpj, class FSpj>
cudaError_t calc_force(const fdps_tree_view& v, const FEpj& f_epj, const FSpj& f_spj, Force* out,
                       cudaStream_t stream) {
    if (v.n_groups <= 0) return cudaSuccess;
    const int64_t most = 0x7FFFFFFF;
    const dim3 grid((unsigned)(v.n_groups < most ? v.n_groups : most), detail::kSlots);
    detail::calc_force_kernel<Force, FEpj, FSpj><<<grid, detail::kThreads, 0, stream>>>(v, f_epj, f_spj, out);
    return cudaGetLastError();
}
#endif  // __CUDACC_RTC__

}  // namespace fdps_user
