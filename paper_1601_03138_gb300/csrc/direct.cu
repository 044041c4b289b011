// direct.cu -- direct summation for a sample of particles, the exact
// reference of the tree force (Eq. ParticleParticleNbody summed over every
// other particle of the same system, softening of the receiving particle).
//
// Used to measure the tree's force error on the GPU and to choose the
// opening angle for an error target.  Arithmetic: positions as FP32 hi/lo
// parts relative to a common origin, so that separations keep about 48
// bits; each pair in FP32 with MUFU rsqrt; per-tile FP32 sums added into
// Kahan-compensated totals, finished in FP64.  Particle i's own term is
// skipped.
#include <algorithm>

#include "fdps_internal.cuh"
#include "packed.cuh"

namespace fdps {
namespace {

constexpr int kDB = 128;  // threads per block
constexpr int kDT = 256;  // j-particles per shared tile

__global__ void __launch_bounds__(256) k_direct_prep(int64_t n, const double* __restrict__ x,
                                                     const double* __restrict__ y,
                                                     const double* __restrict__ z,
                                                     const double* __restrict__ m,
                                                     const double* __restrict__ eps, double ox,
                                                     double oy, double oz, float4* __restrict__ hi,
                                                     float4* __restrict__ lo) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double rx = x[i] - ox, ry = y[i] - oy, rz = z[i] - oz;
        float hx, hy, hz, lx, ly, lz;
        split_f32(rx, hx, lx);
        split_f32(ry, hy, ly);
        split_f32(rz, hz, lz);
        hi[i] = make_float4(hx, hy, hz, to_f32(m[i]));
        lo[i] = make_float4(lx, ly, lz, to_f32(eps[i] * eps[i]));
    }
}

__global__ void k_invert_id(int64_t n, const uint32_t* __restrict__ id, uint32_t* __restrict__ inv) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x)
        inv[id[p]] = (uint32_t)p;
}

struct Comp4 {
    float s[4], c[4];
    __device__ __forceinline__ void add(int k, float v) {
        const float y = v - c[k];
        const float t = s[k] + y;
        c[k] = (t - s[k]) - y;
        s[k] = t;
    }
};

// one pair: (dx, dy, dz) from i to j, adds m/r^3 d and -m/r
__device__ __forceinline__ void pair(const float4 ih, const float4 il, const float4 jh, const float4 jl,
                                     float e2, float& ax, float& ay, float& az, float& pp) {
    const float dx = (jh.x - ih.x) + (jl.x - il.x);
    const float dy = (jh.y - ih.y) + (jl.y - il.y);
    const float dz = (jh.z - ih.z) + (jl.z - il.z);
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, e2)));
    const float ri = rsqrtf(r2);
    const float mri = jh.w * ri;
    const float mri3 = mri * ri * ri;
    ax = fmaf(mri3, dx, ax);
    ay = fmaf(mri3, dy, ay);
    az = fmaf(mri3, dz, az);
    pp -= mri;
}

// One tile of m j-particles on the 2 KP i-particles of a thread.  SELF: an i-particle of the warp is in the
// tile (at rel), and its own term gets no mass.  NORMAL: every eps^2
// of the warp is a normal FP32 number, so every r^2 is.
template <int KP, bool SELF, bool NORMAL>
__device__ __forceinline__ void direct_tile(const float4* s_h, const float4* s_l, int m,
                                            const uint32_t* rel, const f2* hx, const f2* hy, const f2* hz,
                                            const f2* lx, const f2* ly, const f2* lz, const f2* e2, f2* ax, f2* ay,
                                            f2* az, f2* pp) {
#pragma unroll 2
    for (int k = 0; k < m; ++k) {
        const float4 jh = s_h[k], jl = s_l[k];
        const f2 jx = f2_pk(jh.x, jh.x), jy = f2_pk(jh.y, jh.y), jz = f2_pk(jh.z, jh.z);
        const f2 kx = f2_pk(jl.x, jl.x), ky = f2_pk(jl.y, jl.y), kz = f2_pk(jl.z, jl.z);
        const f2 jm = f2_pk(jh.w, jh.w);
#pragma unroll
        for (int q = 0; q < KP; ++q) {
            const f2 dx = f2_add(f2_sub(jx, hx[q]), f2_sub(kx, lx[q]));
            const f2 dy = f2_add(f2_sub(jy, hy[q]), f2_sub(ky, ly[q]));
            const f2 dz = f2_add(f2_sub(jz, hz[q]), f2_sub(kz, lz[q]));
            const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_fma(dz, dz, e2[q])));
            float ra, rb;
            f2_up(r2, ra, rb);
            const bool oa = SELF && (uint32_t)k == rel[2 * q], ob = SELF && (uint32_t)k == rel[2 * q + 1];
            // (the own term of a vanishing eps^2 has an infinite 1/r)
            const f2 ri = NORMAL ? f2_pk(rsqrt_normal(ra), rsqrt_normal(rb))
                                 : f2_pk(oa ? 0.0f : rsqrtf(ra), ob ? 0.0f : rsqrtf(rb));
            const f2 mj = SELF ? f2_pk(oa ? 0.0f : jh.w, ob ? 0.0f : jh.w) : jm;
            const f2 mri = f2_mul(mj, ri);
            const f2 mri3 = f2_mul(f2_mul(mri, ri), ri);
            ax[q] = f2_fma(mri3, dx, ax[q]);
            ay[q] = f2_fma(mri3, dy, ay[q]);
            az[q] = f2_fma(mri3, dz, az[q]);
            pp[q] = f2_sub(pp[q], mri);
        }
    }
}

// The j range in tiles of up to kDT: slices of jper particles, tps tiles each.
struct DirectTiles {
    int64_t n, jper;
    int tps, total;
    __device__ __forceinline__ int64_t first(int id) const { return (int64_t)(id / tps) * jper + (int64_t)(id % tps) * kDT; }
    __device__ __forceinline__ int count(int id) const {
        const int64_t slice = (int64_t)(id / tps + 1) * jper, end = slice < n ? slice : n, m = end - first(id);
        return m <= 0 ? 0 : m < kDT ? (int)m : kDT;
    }
};

// One system: a block takes P sampled rows per i-slot of a thread (thread t
// rows (blockIdx.x * 2 KP + q) P + t % P) and tiles blockIdx.y tper and on, 128 / P
// of them at a time (a warp works on one); j-particles are staged in shared
// memory, FP32 sums of a tile, in its order whatever the split, go into Kahan
// sums, partial sums of a block's warps into part[].  Bound by the FP32 pipe: 19
// operations a pair term, in packed instructions for two i-particles, with each
// staged j-particle read once for the thread's 2 KP; the own-term check runs
// only on the tiles that hold one of the warp's i-particles.  4096 rows of 2^20
// particles: 5.76 ms of kernel time with one i-particle a thread and scalar
// instructions; the whole call 6.25 -> 3.24 ms (3.16 against 3.06 ms with four
// CTAs of 128 registers an SM instead of three of 153).
template <int KP>
__global__ void __launch_bounds__(kDB, KP == 2 ? 3 : 5) k_direct_tiled(DirectTiles J, int tper, int64_t ns, int P,
                                                      const uint32_t* __restrict__ inv,
                                                      const int64_t* __restrict__ rows,
                                                      const float4* __restrict__ hi,
                                                      const float4* __restrict__ lo,
                                                      double* __restrict__ part) {
    constexpr int kTiles = KP == 2 ? 1 : 4;  // the most that are staged at a time
    __shared__ float4 s_h[kTiles * kDT], s_l[kTiles * kDT];
    constexpr int K = 2 * KP;
    const int t = threadIdx.x;
    const int ip = t % P, sl = t / P, nsl = kDB / P;
    uint32_t p[K];  // positions of the i-particles (n < 2^31), all ones for none
    f2 hx[KP], hy[KP], hz[KP], lx[KP], ly[KP], lz[KP], e2[KP];
    bool normal = true;
#pragma unroll
    for (int q = 0; q < KP; ++q) {
        float4 h[2], l[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int64_t s = ((int64_t)blockIdx.x * K + 2 * q + c) * P + ip;
            p[2 * q + c] = s < ns ? inv[rows[s]] : 0xFFFFFFFFu;
            h[c] = s < ns ? hi[p[2 * q + c]] : make_float4(0.f, 0.f, 0.f, 0.f);
            l[c] = s < ns ? lo[p[2 * q + c]] : make_float4(0.f, 0.f, 0.f, 1.f);
            normal = normal && l[c].w >= 1.1754944e-38f;
        }
        hx[q] = f2_pk(h[0].x, h[1].x);
        hy[q] = f2_pk(h[0].y, h[1].y);
        hz[q] = f2_pk(h[0].z, h[1].z);
        lx[q] = f2_pk(l[0].x, l[1].x);
        ly[q] = f2_pk(l[0].y, l[1].y);
        lz[q] = f2_pk(l[0].z, l[1].z);
        e2[q] = f2_pk(l[0].w, l[1].w);
    }
    normal = __all_sync(0xFFFFFFFFu, normal);
    const int t0 = blockIdx.y * tper, t1 = t0 + tper < J.total ? t0 + tper : J.total;
    Comp4 acc[K];
#pragma unroll
    for (int i = 0; i < K; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i].s[k] = acc[i].c[k] = 0.f;
    for (int tb = t0; tb < t1; tb += nsl) {
        __syncthreads();
        for (int q = 0; q < nsl && tb + q < t1; ++q) {
            const int64_t jt = J.first(tb + q);
            const int m = J.count(tb + q);
            for (int k = t; k < m; k += kDB) {
                s_h[q * kDT + k] = hi[jt + k];
                s_l[q * kDT + k] = lo[jt + k];
            }
        }
        __syncthreads();
        if (tb + sl >= t1) break;  // the block's last tiles, none for this warp
        const int64_t jt = J.first(tb + sl);
        const int m = J.count(tb + sl);
        const float4 *th = s_h + sl * kDT, *tl = s_l + sl * kDT;
        bool self = false;
        uint32_t rel[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            rel[i] = p[i] - (uint32_t)jt;
            self = self || rel[i] < (uint32_t)m;
        }
        self = __any_sync(0xFFFFFFFFu, self);
        f2 ax[KP], ay[KP], az[KP], pp[KP];
#pragma unroll
        for (int q = 0; q < KP; ++q) ax[q] = ay[q] = az[q] = pp[q] = 0ull;
        if (!normal)
            direct_tile<KP, true, false>(th, tl, m, rel, hx, hy, hz, lx, ly, lz, e2, ax, ay, az, pp);
        else if (self)
            direct_tile<KP, true, true>(th, tl, m, rel, hx, hy, hz, lx, ly, lz, e2, ax, ay, az, pp);
        else
            direct_tile<KP, false, true>(th, tl, m, rel, hx, hy, hz, lx, ly, lz, e2, ax, ay, az, pp);
#pragma unroll
        for (int q = 0; q < KP; ++q) {
            const f2 v[4] = {ax[q], ay[q], az[q], pp[q]};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float a, b;
                f2_up(v[k], a, b);
                acc[2 * q].add(k, a);
                acc[2 * q + 1].add(k, b);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const int64_t s = ((int64_t)blockIdx.x * K + i) * P + ip;
        if (s < ns)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                part[(((int64_t)blockIdx.y * nsl + sl) * ns + s) * 4 + k] =
                    (double)acc[i].s[k] - (double)acc[i].c[k];
    }
}

// Several systems: each sampled particle sums over its own system's range.
__global__ void __launch_bounds__(kDB) k_direct_systems(int64_t ns, const uint32_t* __restrict__ inv,
                                                        const int64_t* __restrict__ rows,
                                                        const uint32_t* __restrict__ sys,
                                                        const int64_t* __restrict__ off,
                                                        const float4* __restrict__ hi,
                                                        const float4* __restrict__ lo,
                                                        double* __restrict__ part) {
    const int64_t s = blockIdx.x * (int64_t)kDB + threadIdx.x;
    if (s >= ns) return;
    const int64_t p = inv[rows[s]];
    const float4 ih = hi[p], il = lo[p];
    const uint32_t k = sys[p];
    Comp4 acc;
#pragma unroll
    for (int c = 0; c < 4; ++c) acc.s[c] = acc.c[c] = 0.f;
    for (int64_t jt = off[k]; jt < off[k + 1]; jt += kDT) {
        const int64_t je = jt + kDT < off[k + 1] ? jt + kDT : off[k + 1];
        float ax = 0.f, ay = 0.f, az = 0.f, pp = 0.f;
        for (int64_t j = jt; j < je; ++j) {
            if (j == p) continue;
            pair(ih, il, hi[j], lo[j], il.w, ax, ay, az, pp);
        }
        acc.add(0, ax);
        acc.add(1, ay);
        acc.add(2, az);
        acc.add(3, pp);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) part[s * 4 + c] = (double)acc.s[c] - (double)acc.c[c];
}

// The slices' partial sums of each row: a warp per row, lanes over the
// slices, in a fixed order.
__global__ void __launch_bounds__(256) k_direct_final(int64_t ns, int js, const double* __restrict__ part,
                                                      double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; s < ns;
         s += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int y = lane; y < js; y += 32)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] += part[((int64_t)y * ns + s) * 4 + k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] += __shfl_down_sync(0xFFFFFFFFu, v[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < 4; ++k) out[s * 4 + k] = v[k];
    }
}

// Tree results (acceleration, potential) at the sampled rows.
__global__ void k_gather_rows(int64_t ns, const uint32_t* __restrict__ inv, const int64_t* __restrict__ rows,
                              const double* __restrict__ ax, const double* __restrict__ ay,
                              const double* __restrict__ az, const double* __restrict__ pot,
                              double* __restrict__ out) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = inv[rows[s]];
        out[s * 4 + 0] = ax[p];
        out[s * 4 + 1] = ay[p];
        out[s * 4 + 2] = az[p];
        out[s * 4 + 3] = pot[p];
    }
}

}  // namespace

// Scratch of a sample: inverse of the id map, FP32 hi/lo copies (direct
// sums only), partial sums.  All device memory, freed by the caller with
// free_sample_scratch.
struct SampleScratch {
    uint32_t* inv = nullptr;
    float4* hi = nullptr;
    float4* lo = nullptr;
    double* part = nullptr;
};

static void free_sample_scratch(SampleScratch& sc) {
    cudaFree(sc.inv);
    cudaFree(sc.hi);
    cudaFree(sc.lo);
    cudaFree(sc.part);
    sc = SampleScratch{};
}

static int invert_ids(fdps_psys* ps, SampleScratch& sc) {
    fdps_ctx* ctx = ps->ctx;
    if (!sc.inv && dev_alloc(ctx, &sc.inv, ps->n) != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, FDPS_ENOMEM, "sample scratch allocation failed");
    }
    k_invert_id<<<grid_for(ps->n, 256, 4 * ctx->sm_count), 256, 0, ctx->stream>>>(ps->n, ps->id[ps->cur], sc.inv);
    FDPS_LAUNCH_CHECK(ctx);
    return FDPS_OK;
}

int direct_sample_device(fdps_psys* ps, int64_t ns, const int64_t* d_rows, double* d_out4) {
    fdps_ctx* ctx = ps->ctx;
    cudaStream_t s = ctx->stream;
    const int64_t n = ps->n;
    const int c = ps->cur;
    SampleScratch sc;
    int rc = invert_ids(ps, sc);
    const bool one = ps->n_sys == 1;
    // j-particles: slices that give four blocks an SM with one i-particle a
    // thread, in tiles of kDT; the FP32 sums run over these tiles.
    const int64_t bx1 = (ns + kDB - 1) / kDB;
    const int64_t sl1 = std::max<int64_t>(1, std::min<int64_t>({(4 * (int64_t)ctx->sm_count + bx1 - 1) / bx1, 1024}));
    DirectTiles J;
    J.n = n;
    J.jper = (n + sl1 - 1) / sl1;
    J.tps = (int)((J.jper + kDT - 1) / kDT);
    J.total = (int)sl1 * J.tps;
    // i-particles: 4 per thread where the rows fill a block of 128 threads
    // with them, else 2; fewer rows than threads leave the other warps to
    // other tiles.  Blocks: one resident wave.
    const int K = ns > 2 * kDB ? 4 : 2;
    const int P = ns > kDB || K == 4 ? kDB : ns > 64 ? 64 : 32;
    const int nsl = kDB / P, per_sm = K == 4 ? 3 : 5;
    const int64_t bx = one ? (ns + (int64_t)K * P - 1) / ((int64_t)K * P) : bx1;
    int64_t by = one ? (int64_t)per_sm * ctx->sm_count / bx : 1;
    by = std::max<int64_t>(1, std::min<int64_t>({by, 1024, (J.total + nsl - 1) / nsl}));
    const int tper = (int)((J.total + by - 1) / by);
    const int js = one ? (int)by * nsl : 1;
    if (!rc && (dev_alloc(ctx, &sc.hi, n) != cudaSuccess || dev_alloc(ctx, &sc.lo, n) != cudaSuccess ||
                dev_alloc(ctx, &sc.part, 4 * ns * js) != cudaSuccess)) {
        cudaGetLastError();
        rc = set_error(ctx, FDPS_ENOMEM, "sample scratch allocation failed");
    }
    if (!rc) {
        // origin: the first particle's position (separations are what count)
        double o[3];
        if (cudaMemcpyAsync(&o[0], ps->x[c], 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(&o[1], ps->y[c], 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(&o[2], ps->z[c], 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            rc = set_error(ctx, FDPS_ECUDA, "reading the origin failed");
        if (!rc) {
            k_direct_prep<<<grid_for(n, 256, 4 * ctx->sm_count), 256, 0, s>>>(
                n, ps->x[c], ps->y[c], ps->z[c], ps->m[c], ps->eps[c], o[0], o[1], o[2], sc.hi, sc.lo);
            FDPS_LAUNCH_CHECK(ctx);
            if (one) {
                const dim3 grid((unsigned)bx, (unsigned)by);
                if (K == 4)
                    k_direct_tiled<2><<<grid, kDB, 0, s>>>(J, tper, ns, P, sc.inv, d_rows, sc.hi, sc.lo, sc.part);
                else
                    k_direct_tiled<1><<<grid, kDB, 0, s>>>(J, tper, ns, P, sc.inv, d_rows, sc.hi, sc.lo, sc.part);
            } else {
                k_direct_systems<<<(unsigned)bx, kDB, 0, s>>>(ns, sc.inv, d_rows, ps->d_sys, ps->d_off, sc.hi,
                                                              sc.lo, sc.part);
            }
            FDPS_LAUNCH_CHECK(ctx);
            k_direct_final<<<grid_for(32 * ns, 256, 4 * ctx->sm_count), 256, 0, s>>>(ns, js, sc.part, d_out4);
            FDPS_LAUNCH_CHECK(ctx);
            if (cudaStreamSynchronize(s) != cudaSuccess) rc = set_error(ctx, FDPS_ECUDA, "direct sum failed");
        }
    }
    free_sample_scratch(sc);
    return rc;
}

int gather_rows_device(fdps_psys* ps, int64_t ns, const int64_t* d_rows, double* d_out4) {
    fdps_ctx* ctx = ps->ctx;
    SampleScratch sc;
    int rc = invert_ids(ps, sc);
    if (!rc) {
        k_gather_rows<<<grid_for(ns, 256, 1024), 256, 0, ctx->stream>>>(ns, sc.inv, d_rows, ps->ax, ps->ay,
                                                                       ps->az, ps->pot, d_out4);
        FDPS_LAUNCH_CHECK(ctx);
        if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) rc = set_error(ctx, FDPS_ECUDA, "gather failed");
    }
    free_sample_scratch(sc);
    return rc;
}

}  // namespace fdps
