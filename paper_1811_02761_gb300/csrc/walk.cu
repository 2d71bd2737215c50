// walk.cu -- walk dispatch, the direct O(N^2) sum of Eq. 1, small helpers.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace nb {

template <int IPL, bool QUAD>
cudaError_t launch_walk_ipl(cudaStream_t s, const WalkArgs &a, const WalkShape &sh, int nsm);
#define NB_WALK_EXTERN(I, Q) \
    extern template cudaError_t launch_walk_ipl<I, Q>(cudaStream_t, const WalkArgs &, const WalkShape &, int);
NB_WALK_EXTERN(1, false) NB_WALK_EXTERN(2, false) NB_WALK_EXTERN(3, false) NB_WALK_EXTERN(4, false)
NB_WALK_EXTERN(1, true) NB_WALK_EXTERN(2, true) NB_WALK_EXTERN(3, true) NB_WALK_EXTERN(4, true)
#undef NB_WALK_EXTERN

template <int IPL, bool QUAD>
cudaError_t launch_coop_ipl(cudaStream_t s, const WalkArgs &a, const WalkShape &sh, int nsm);
#define NB_COOP_EXTERN(I, Q) \
    extern template cudaError_t launch_coop_ipl<I, Q>(cudaStream_t, const WalkArgs &, const WalkShape &, int);
NB_COOP_EXTERN(1, false) NB_COOP_EXTERN(2, false) NB_COOP_EXTERN(3, false) NB_COOP_EXTERN(4, false)
NB_COOP_EXTERN(1, true) NB_COOP_EXTERN(2, true) NB_COOP_EXTERN(3, true) NB_COOP_EXTERN(4, true)
#undef NB_COOP_EXTERN

template <int IPL, bool QUAD>
cudaError_t launch_ordered_ipl(cudaStream_t s, const WalkArgs &a, const WalkShape &sh, int nsm);
#define NB_ORDERED_EXTERN(I, Q) \
    extern template cudaError_t launch_ordered_ipl<I, Q>(cudaStream_t, const WalkArgs &, const WalkShape &, int);
NB_ORDERED_EXTERN(1, false) NB_ORDERED_EXTERN(2, false) NB_ORDERED_EXTERN(3, false) NB_ORDERED_EXTERN(4, false)
NB_ORDERED_EXTERN(1, true) NB_ORDERED_EXTERN(2, true) NB_ORDERED_EXTERN(3, true) NB_ORDERED_EXTERN(4, true)
#undef NB_ORDERED_EXTERN

template <int IPL, bool QUAD>
static cudaError_t launch_both(cudaStream_t s, const WalkArgs &a, const WalkShape &sh, int nsm) {
    if (sh.ordered) return launch_ordered_ipl<IPL, QUAD>(s, a, sh, nsm);
    if (!sh.coop_only) {
        const cudaError_t e = launch_walk_ipl<IPL, QUAD>(s, a, sh, nsm);
        if (e != cudaSuccess || a.longest <= a.quota) return e;  // nothing can be cut
    }
    return launch_coop_ipl<IPL, QUAD>(s, a, sh, nsm);
}

cudaError_t launch_walk(cudaStream_t s, const WalkArgs &a, const WalkShape &sh, int nsm) {
    switch (sh.ipl) {
        case 1: return sh.quad ? launch_both<1, true>(s, a, sh, nsm) : launch_both<1, false>(s, a, sh, nsm);
        case 2: return sh.quad ? launch_both<2, true>(s, a, sh, nsm) : launch_both<2, false>(s, a, sh, nsm);
        case 3: return sh.quad ? launch_both<3, true>(s, a, sh, nsm) : launch_both<3, false>(s, a, sh, nsm);
        case 4: return sh.quad ? launch_both<4, true>(s, a, sh, nsm) : launch_both<4, false>(s, a, sh, nsm);
        default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------- direct sum
// Bound by the FP32 pipe (12 lane operations per pair, 16 with the Newton
// step, 1 more with the potential).  A CTA holds kDQ targets per lane, the
// same ones in all its warps, and streams the sources through shared memory in
// tiles; each warp takes every kDW-th pair of a tile.  The pairs are laid out
// for the packed FP32 instructions, as in the walk.  A cluster of C CTAs shares
// the sources of one block of targets, so that few targets still fill the GPU
// and no last wave runs nearly empty; the partial sums meet in shared memory,
// over the warps and then over the CTAs, always in the same order.
// One target per thread, scalar, one CTA per 128 targets / this, in us (plain;
// compensated with potential): N = 500 30, 34 / 22, 24; 8000 188, 248 / 51, 67;
// 50021 1486, 1941 / 1049, 1488; 300000 40751, 54967 / 35566, 50566.  Two slots
// per lane and 24 warps per SM instead of three and 16: 1065, 1548 at 50021.
constexpr int kDQ = 3, kDW = 8, kDT = 32 * kDW;  // slots per lane, warps, threads
constexpr int kDTile = 2 * kDT;                  // sources per tile: a pair per thread
constexpr int kDTargets = 32 * kDQ;

__device__ __forceinline__ void neumaier(float &s, float &c, float x) {
    float t = s + x;
    if (fabsf(s) >= fabsf(x))
        c += (s - t) + x;
    else
        c += (x - t) + s;
    s = t;
}

// COMP: the reciprocal square root gets one Newton-Raphson step,
// y <- y (3 - r2 y^2) / 2, and each tile's partial sum is added to the total
// with Neumaier compensation.
template <bool PHI, bool COMP, bool SAFE>
__global__ void __launch_bounds__(kDT, 2) direct_kernel(int64_t n, int64_t chunk,
                                                        const float *__restrict__ x,
                                                        const float *__restrict__ y,
                                                        const float *__restrict__ z,
                                                        const float *__restrict__ m, float eps2,
                                                        float G, float *ax, float *ay, float *az,
                                                        float *phi) {
    __shared__ float4 tile[2 * kDT];  // pair k: (x, x', y, y'), (z, z', m, m')
    __shared__ float4 red[kDW][kDTargets];
    __shared__ float4 part[kDTargets];
    const cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int lane = (int)(threadIdx.x & 31), w = (int)(threadIdx.x >> 5);
    const int64_t i0 = (int64_t)(blockIdx.x / C) * kDTargets;
    float2 nx[kDQ], ny[kDQ], nz[kDQ];
    float s[kDQ][4], c[kDQ][4];
    float2 run[kDQ][4];
#pragma unroll
    for (int q = 0; q < kDQ; q++) {
        const int64_t i = min(i0 + 32 * q + lane, n - 1);
        const float px = -x[i], py = -y[i], pz = -z[i];
        nx[q] = make_float2(px, px);
        ny[q] = make_float2(py, py);
        nz[q] = make_float2(pz, pz);
#pragma unroll
        for (int a = 0; a < 4; a++) {
            s[q][a] = c[q][a] = 0.0f;
            run[q][a] = make_float2(0.0f, 0.0f);
        }
    }
    const float2 e2 = make_float2(eps2, eps2), neg1 = make_float2(-1.0f, -1.0f);
    const float2 half = make_float2(-0.5f, -0.5f), c15 = make_float2(1.5f, 1.5f);
    const int64_t j0 = rank * chunk, j1 = min(n, j0 + chunk);
    // this thread's pair of the tile at `base`; past the end a massless,
    // distant source
    float v[2][4];
    auto load = [&](int64_t base) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int64_t j = base + 2 * threadIdx.x + h;
            const bool ok = j < j1;
            v[h][0] = ok ? x[j] : 1e18f;
            v[h][1] = ok ? y[j] : 1e18f;
            v[h][2] = ok ? z[j] : 1e18f;
            v[h][3] = ok ? m[j] : 0.0f;
        }
    };
    if (j0 < j1) load(j0);
    for (int64_t base = j0; base < j1; base += kDTile) {
        __syncthreads();
        tile[2 * threadIdx.x] = make_float4(v[0][0], v[1][0], v[0][1], v[1][1]);
        tile[2 * threadIdx.x + 1] = make_float4(v[0][2], v[1][2], v[0][3], v[1][3]);
        __syncthreads();
        if (base + kDTile < j1) load(base + kDTile);  // in flight during the tile
        const int np = (int)(min((int64_t)kDTile, j1 - base) + 1) >> 1;
        const float4 *pe = tile + 2 * np;
        for (const float4 *pk = tile + 2 * w; pk < pe; pk += 2 * kDW) {
            const float4 A = pk[0], B = pk[1];
            const float2 px = make_float2(A.x, A.y), py = make_float2(A.z, A.w);
            const float2 pz = make_float2(B.x, B.y), pm = make_float2(B.z, B.w);
#pragma unroll
            for (int q = 0; q < kDQ; q++) {
                const float2 dx = __fadd2_rn(px, nx[q]);
                const float2 dy = __fadd2_rn(py, ny[q]);
                const float2 dz = __fadd2_rn(pz, nz[q]);
                float2 r2 = __ffma2_rn(dx, dx, e2);
                r2 = __ffma2_rn(dy, dy, r2);
                r2 = __ffma2_rn(dz, dz, r2);
                float2 ri = make_float2(rsqrt_fast(r2.x), rsqrt_fast(r2.y));
                if constexpr (COMP)
                    ri = __fmul2_rn(ri, __ffma2_rn(__fmul2_rn(__fmul2_rn(half, r2), ri), ri, c15));
                if constexpr (SAFE) {
                    ri.x = r2.x >= 1.17549435e-38f ? ri.x : 0.0f;
                    ri.y = r2.y >= 1.17549435e-38f ? ri.y : 0.0f;
                }
                const float2 mr = __fmul2_rn(pm, ri);
                const float2 w3 = __fmul2_rn(mr, __fmul2_rn(ri, ri));
                run[q][0] = __ffma2_rn(w3, dx, run[q][0]);
                run[q][1] = __ffma2_rn(w3, dy, run[q][1]);
                run[q][2] = __ffma2_rn(w3, dz, run[q][2]);
                if constexpr (PHI) run[q][3] = __ffma2_rn(mr, neg1, run[q][3]);
            }
        }
        if constexpr (COMP) {
#pragma unroll
            for (int q = 0; q < kDQ; q++)
#pragma unroll
                for (int a = 0; a < (PHI ? 4 : 3); a++) {
                    neumaier(s[q][a], c[q][a], run[q][a].x + run[q][a].y);
                    run[q][a] = make_float2(0.0f, 0.0f);
                }
        }
    }
#pragma unroll
    for (int q = 0; q < kDQ; q++) {
        float r[4];
#pragma unroll
        for (int a = 0; a < 4; a++) r[a] = COMP ? s[q][a] + c[q][a] : run[q][a].x + run[q][a].y;
        red[w][32 * q + lane] = make_float4(r[0], r[1], r[2], r[3]);
    }
    __syncthreads();
    // sums of k = 0 .. count - 1 in order
    auto add_up = [&](int count, float (&r)[4], auto value) {
        float k4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int a = 0; a < 4; a++) r[a] = 0.0f;
        for (int k = 0; k < count; k++) {
            const float4 u = value(k);
            const float us[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int a = 0; a < 4; a++) {
                if constexpr (COMP) neumaier(r[a], k4[a], us[a]);
                else r[a] += us[a];
            }
        }
#pragma unroll
        for (int a = 0; a < 4; a++) r[a] += k4[a];
    };
    const int t = (int)threadIdx.x;
    float r[4];
    if (t < kDTargets) {
        add_up(kDW, r, [&](int k) { return red[k][t]; });
        part[t] = make_float4(r[0], r[1], r[2], r[3]);
    }
    if (C > 1) cluster.sync();
    const int64_t i = i0 + t;
    if (rank == 0 && t < kDTargets && i < n) {
        if (C > 1) add_up(C, r, [&](int k) { return cluster.map_shared_rank(part, k)[t]; });
        ax[i] = G * r[0];
        ay[i] = G * r[1];
        az[i] = G * r[2];
        if (PHI) {
            float self = 0.0f;
            if (!SAFE) {
                float rs = rsqrt_fast(eps2);
                if (COMP) rs = rs * (1.5f - 0.5f * eps2 * rs * rs);
                self = m[i] * rs;  // the j = i term, excluded by Eq. 1
            }
            phi[i] = G * (r[3] + self);
        }
    }
    if (C > 1) cluster.sync();  // the other CTAs' sums stay until they have been read
}

cudaError_t launch_direct(cudaStream_t s, int64_t n, const float *x, const float *y,
                          const float *z, const float *m, float G, float eps, bool compensated,
                          float *ax, float *ay, float *az, float *phi) {
    const float eps2 = eps * eps;
    const bool safe = !(eps2 > 0.0f);
    // clusters of eight while the targets alone would be fewer than about 27
    // waves of CTAs (two per SM)
    const int64_t blocks = (n + kDTargets - 1) / kDTargets;
    const int C = blocks >= 8192 ? 1 : 8;
    const int64_t chunk = ((n + C - 1) / C + 15) / 16 * 16;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)C;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((unsigned)(blocks * C));
    lc.blockDim = dim3(kDT);
    lc.stream = s;
    lc.attrs = &attr;
    lc.numAttrs = 1;
    void (*k)(int64_t, int64_t, const float *, const float *, const float *, const float *, float,
              float, float *, float *, float *, float *);
    if (phi) {
        if (compensated) k = safe ? direct_kernel<true, true, true> : direct_kernel<true, true, false>;
        else k = safe ? direct_kernel<true, false, true> : direct_kernel<true, false, false>;
    } else {
        if (compensated) k = safe ? direct_kernel<false, true, true> : direct_kernel<false, true, false>;
        else k = safe ? direct_kernel<false, false, true> : direct_kernel<false, false, false>;
    }
    return cudaLaunchKernelEx(&lc, k, n, chunk, x, y, z, m, eps2, G, ax, ay, az, phi);
}

// ---------------------------------------------------------------- helpers
__global__ void acc_mag_kernel(int64_t n, const float4 *__restrict__ acc, float *__restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float4 a = acc[i];
        out[i] = sqrtf(a.x * a.x + a.y * a.y + a.z * a.z);
    }
}

void launch_acc_mag(cudaStream_t s, int64_t n, const float4 *acc_sorted, float *aold_sorted) {
    int blocks = (int)((n + 255) / 256);
    if (blocks > 65535 * 8) blocks = 65535 * 8;
    acc_mag_kernel<<<blocks, 256, 0, s>>>(n, acc_sorted, aold_sorted);
}

__global__ void gather_f32_kernel(int64_t n, const uint32_t *__restrict__ perm,
                                  const float *__restrict__ src, float *__restrict__ dst) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[perm[i]];
}

void launch_gather_f32(cudaStream_t s, int64_t n, const uint32_t *perm, const float *src,
                       float *dst) {
    int blocks = (int)((n + 255) / 256);
    if (blocks > 65535 * 8) blocks = 65535 * 8;
    gather_f32_kernel<<<blocks, 256, 0, s>>>(n, perm, src, dst);
}

}  // namespace nb
