// mlp.cu -- learned cost model that orders the persistent walk's queue.
//
// A small MLP (8 group features -> 32 -> 32 -> 1, ReLU) predicts log2 of the
// walk cost of each i-group (interaction-list entries it processes).  It is
// trained online on the costs the walk itself logs, with hand-written
// forward / backward / Adam kernels: BF16 weights in the forward and backward
// passes, FP32 accumulation, FP32 master weights and Adam moments.  The
// persistent walk then pops groups in descending predicted cost (longest
// first), which shortens the tail of the walk; accelerations do not depend on
// the order (each group's walk is independent of which warp runs it, when).
//
// Parameter layout (kMlpParams floats): W1[8][32], b1[32], W2[32][32],
// b2[32], W3[32], b3 -- W1[i][j] connects input i to hidden unit j.
//
// Features of a group (computed here from the walk's own data):
//   0 log2 count            1 log2 r_g              2 log2 min |a_old|
//   3 log2 |c_g - com_root| 4 level of the group's cell
//   5 log2 (count / cell volume of that level)      6 log2 mean |a_old|
//   7 log2 N of the group's system
// The model input is the standardised feature (x - mean) / std with the
// statistics frozen from the first training batch.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.cuh"

namespace nb {

constexpr int kIn = 8, kH = 32;
constexpr int oW1 = 0, oB1 = oW1 + kIn * kH, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH,
              oB3 = oW3 + kH;
static_assert(oB3 + 1 == kMlpParams, "parameter layout");

__device__ __forceinline__ float safe_log2(float x) { return __log2f(fmaxf(x, 1e-30f)); }

// ---------------------------------------------------------------- features
__global__ void mlp_features_kernel(Layout L, const DevState *__restrict__ ds,
                                    const int32_t *__restrict__ grp_first,
                                    const int32_t *__restrict__ grp_count,
                                    const float4 *__restrict__ grp_sphere,
                                    const int32_t *__restrict__ grp_sys,
                                    const float *__restrict__ aold, const uint64_t *__restrict__ keys,
                                    const float4 *__restrict__ nodeA,
                                    const int32_t *__restrict__ sys_root,
                                    const SysBox *__restrict__ box, const int64_t *__restrict__ off,
                                    float *__restrict__ feat) {
    const int ng = ds->ngroups;
    const unsigned lane = lane_id();
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const int mbits = 3 * L.levels;
    for (int g = warp; g < ng; g += nw) {
        const int first = grp_first[g], cnt = grp_count[g];
        float amin = INFINITY, asum = 0.0f;
        for (int k = lane; k < cnt; k += 32) {
            float a = aold[first + k];
            amin = fminf(amin, a);
            asum += a;
        }
        for (int o = 16; o; o >>= 1) {
            amin = fminf(amin, __shfl_xor_sync(NB_FULL, amin, o));
            asum += __shfl_xor_sync(NB_FULL, asum, o);
        }
        if (lane == 0) {
            const int s = grp_sys[g];
            const float4 sph = grp_sphere[g];
            const int root = sys_root[s];
            const float4 rc = root >= 0 ? nodeA[root] : make_float4(sph.x, sph.y, sph.z, 0.f);
            const float dx = sph.x - rc.x, dy = sph.y - rc.y, dz = sph.z - rc.z;
            // level of the smallest cell holding the whole group
            uint64_t x = keys[first] ^ keys[first + cnt - 1];
            x &= mbits >= 64 ? ~0ull : ((1ull << mbits) - 1ull);
            const int level = x == 0 ? L.levels : (mbits - 1 - (63 - __clzll((long long)x))) / 3;
            const float Lbox = box[s].L;
            const float nsys = (float)(off[s + 1] - off[s]);
            float *f = feat + (int64_t)g * kIn;
            f[0] = safe_log2((float)cnt);
            f[1] = safe_log2(sph.w);
            f[2] = safe_log2(amin);
            f[3] = safe_log2(sqrtf(dx * dx + dy * dy + dz * dz));
            f[4] = (float)level;
            f[5] = safe_log2((float)cnt) - 3.0f * (safe_log2(Lbox) - (float)level);
            f[6] = safe_log2(asum / (float)cnt);
            f[7] = safe_log2(nsys);
        }
    }
}

// ---------------------------------------------------------------- forward
struct alignas(16) MlpSmem {
    float w[kMlpParams + 3];
    float mu[kIn], isd[kIn];
};
static_assert(oB1 % 4 == 0 && oW2 % 4 == 0 && oB2 % 4 == 0 && oW3 % 4 == 0, "weights read four at a time");

// The BF16 weights: wb, or (w32) FP32 parameters rounded here.
__device__ __forceinline__ void load_weights(MlpSmem &S, const __nv_bfloat16 *wb, const float *w32,
                                             const float *norm) {
    for (int p = threadIdx.x; p < kMlpParams; p += blockDim.x)
        S.w[p] = __bfloat162float(w32 ? __float2bfloat16_rn(w32[p]) : wb[p]);
    if (threadIdx.x < kIn) {
        S.mu[threadIdx.x] = norm ? norm[threadIdx.x] : 0.0f;
        S.isd[threadIdx.x] = norm ? 1.0f / norm[kIn + threadIdx.x] : 1.0f;
    }
    __syncthreads();
}

// Four consecutive weights in one shared-memory broadcast: with one load per
// product the loads, not the products, bound the pass.
__device__ __forceinline__ float4 w4(const MlpSmem &S, int p) {
    return *reinterpret_cast<const float4 *>(&S.w[p]);
}

constexpr int kHS = kH + 4;  // stride of a thread's row: 16-byte aligned, eight rows in distinct banks

__device__ __forceinline__ void put_row(float *row, const float (&v)[kH]) {
#pragma unroll
    for (int j = 0; j < kH; j += 4)
        *reinterpret_cast<float4 *>(row + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
}

// a += x (weights p .. p + 31)
__device__ __forceinline__ void add_row(const MlpSmem &S, int p, float x, float (&a)[kH]) {
#pragma unroll
    for (int k = 0; k < kH; k += 4) {
        const float4 w = w4(S, p + k);
        a[k] = fmaf(x, w.x, a[k]);
        a[k + 1] = fmaf(x, w.y, a[k + 1]);
        a[k + 2] = fmaf(x, w.z, a[k + 2]);
        a[k + 3] = fmaf(x, w.w, a[k + 3]);
    }
}

// Forward pass of one sample: the 32 sums of a layer in registers, an input at
// a time from this thread's rows in shared memory (xrow: standardised inputs,
// h1row: first activations), every sum in the order of its inputs.  h2: the
// second activations.
__device__ __forceinline__ float mlp_fwd(const MlpSmem &S, const float *x, float *xrow, float *h1row,
                                         float (&h2)[kH]) {
    float a[kH];
#pragma unroll
    for (int j = 0; j < kH; j++) a[j] = S.w[oB1 + j];
#pragma unroll 2
    for (int i = 0; i < kIn; i++) {
        const float v = (x[i] - S.mu[i]) * S.isd[i];
        xrow[i] = v;
        add_row(S, oW1 + i * kH, v, a);
    }
#pragma unroll
    for (int j = 0; j < kH; j++) a[j] = fmaxf(a[j], 0.0f);
    put_row(h1row, a);
#pragma unroll
    for (int k = 0; k < kH; k++) a[k] = S.w[oB2 + k];
#pragma unroll 1
    for (int j = 0; j < kH; j += 2) {
        const float2 h = *reinterpret_cast<const float2 *>(h1row + j);
        add_row(S, oW2 + j * kH, h.x, a);
        add_row(S, oW2 + (j + 1) * kH, h.y, a);
    }
    float y = S.w[oB3];
#pragma unroll
    for (int k = 0; k < kH; k++) {
        h2[k] = fmaxf(a[k], 0.0f);
        y = fmaf(h2[k], S.w[oW3 + k], y);
    }
    return y;
}

// tnorm (nullable): target mean and standard deviation; the network output
// is de-standardised with them.
__global__ void __launch_bounds__(128) mlp_forward_kernel(const int32_t *__restrict__ pn,
                                                          const float *__restrict__ feat,
                                                          const __nv_bfloat16 *__restrict__ wb,
                                                          const float *__restrict__ norm,
                                                          const float *__restrict__ tnorm,
                                                          float *__restrict__ pred) {
    __shared__ MlpSmem S;
    __shared__ __align__(16) float h1[128][kHS];
    __shared__ float xr[128][kIn + 1];
    load_weights(S, wb, nullptr, norm);
    const float tm = tnorm ? tnorm[0] : 0.0f, ts = tnorm ? tnorm[1] : 1.0f;
    const int64_t n = *pn;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n;
         g += (int64_t)gridDim.x * blockDim.x) {
        float h2[kH];
        pred[g] = fmaf(mlp_fwd(S, feat + g * kIn, xr[threadIdx.x], h1[threadIdx.x], h2), ts, tm);
    }
}

// ---------------------------------------------------------------- backward
constexpr int kGB = kMlpGradBlock;  // samples (and threads) per block in the gradient kernel
struct alignas(16) GradSmem {
    MlpSmem m;
    float h1[kGB][kHS];
    float d1[kGB][kHS];
    float h2[kGB][kHS];
    float d2[kGB][kHS];
    float xn[kGB][kIn + 1];
    float dy[kGB];
    float loss[kGB];
};

// Mean-squared-error gradient of one minibatch: samples idx = base + s *
// stride (s = 0 .. count-1); each block handles kGB of them, a thread each for
// the forward and backward pass, and then the block's weight gradients as
// small matrix products over its samples, a tile of outputs per thread (4 x 4
// of dW2, from one broadcast of four of each side per sample).  Writes the
// block's partial gradient (kMlpParams floats) and partial loss -- reduced in a
// fixed order afterwards, so training is deterministic.  pred (nullable): the
// network's outputs too.  Bound by the FP32 pipe and the shared-memory
// broadcasts (3.7k products per sample).  n = 60013: 42 us with a load per
// product and one gradient at a time, and 11 us more for the predictions; 25 us
// for both so.
__global__ void __launch_bounds__(kGB) mlp_grad_kernel(const float *__restrict__ feat,
                                                       const float *__restrict__ target,
                                                       int64_t base, int64_t stride, int count,
                                                       float inv_count,
                                                       const __nv_bfloat16 *__restrict__ wb,
                                                       const float *__restrict__ w32,
                                                       const float *__restrict__ norm,
                                                       float *__restrict__ gpart,
                                                       float *__restrict__ lpart,
                                                       float *__restrict__ pred) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    GradSmem &S = *reinterpret_cast<GradSmem *>(mlp_smem);
    load_weights(S.m, wb, w32, norm);
    const int t = threadIdx.x;
    const int s = blockIdx.x * kGB + t;
    {
        float *h1row = S.h1[t], *d1row = S.d1[t];
        float h2[kH], dy = 0.0f, loss = 0.0f;
        const bool on = s < count;
        const int64_t g = base + (int64_t)(on ? s : 0) * stride;
        const float y = mlp_fwd(S.m, feat + g * kIn, S.xn[t], h1row, h2);
        if (!on) {  // past the end (the batch's first sample was read): all zero
#pragma unroll
            for (int k = 0; k < kH; k++) h2[k] = 0.0f;
            put_row(h1row, h2);
#pragma unroll
            for (int i = 0; i < kIn; i++) S.xn[t][i] = 0.0f;
        }
        put_row(S.h2[t], h2);
        if (on) {
            if (pred) pred[g] = y;
            const float e = y - target[g];
            dy = 2.0f * e * inv_count;
            loss = e * e * inv_count;
        }
        float d2[kH];
#pragma unroll
        for (int k = 0; k < kH; k++) d2[k] = h2[k] > 0.0f ? dy * S.m.w[oW3 + k] : 0.0f;
        put_row(S.d2[t], d2);
#pragma unroll 2
        for (int j = 0; j < kH; j++) {
            float a = 0.0f;
#pragma unroll
            for (int k = 0; k < kH; k += 4) {
                const float4 w = w4(S.m, oW2 + j * kH + k);
                a = fmaf(d2[k], w.x, a);
                a = fmaf(d2[k + 1], w.y, a);
                a = fmaf(d2[k + 2], w.z, a);
                a = fmaf(d2[k + 3], w.w, a);
            }
            d1row[j] = h1row[j] > 0.0f ? a : 0.0f;
        }
        S.dy[t] = dy;
        S.loss[t] = loss;
    }
    __syncthreads();
    float *gp = gpart + (int64_t)blockIdx.x * kMlpParams;
    // every parameter's gradient is a sum over the block's samples, in order
    static_assert(kGB == 64, "the tiles below");
    {  // W2[j][k] = sum h1_j d2_k: rows 4 (t / 8) .., columns 4 (t % 8) ..
        const int j0 = 4 * (t >> 3), k0 = 4 * (t & 7);
        float acc[4][4] = {};
        for (int q = 0; q < kGB; q++) {
            const float4 h = *reinterpret_cast<const float4 *>(&S.h1[q][j0]);
            const float4 d = *reinterpret_cast<const float4 *>(&S.d2[q][k0]);
            const float hv[4] = {h.x, h.y, h.z, h.w}, dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
            for (int u = 0; u < 4; u++)
#pragma unroll
                for (int v = 0; v < 4; v++) acc[u][v] = fmaf(hv[u], dv[v], acc[u][v]);
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
#pragma unroll
            for (int v = 0; v < 4; v++) gp[oW2 + (j0 + u) * kH + k0 + v] = acc[u][v];
    }
    {  // W1[i][j] = sum xn_i d1_j: row t / 8, columns 4 (t % 8) ..
        const int i = t >> 3, j0 = 4 * (t & 7);
        float acc[4] = {};
        for (int q = 0; q < kGB; q++) {
            const float x = S.xn[q][i];
            const float4 d = *reinterpret_cast<const float4 *>(&S.d1[q][j0]);
            acc[0] = fmaf(x, d.x, acc[0]);
            acc[1] = fmaf(x, d.y, acc[1]);
            acc[2] = fmaf(x, d.z, acc[2]);
            acc[3] = fmaf(x, d.w, acc[3]);
        }
#pragma unroll
        for (int v = 0; v < 4; v++) gp[oW1 + i * kH + j0 + v] = acc[v];
    }
    {  // b1, b2 (one each per thread of a warp), W3
        const int k = t & 31;
        float a = 0.0f, c = 0.0f;
        if (t < 32) {
            for (int q = 0; q < kGB; q++) {
                a += S.d1[q][k];
                c += S.d2[q][k];
            }
            gp[oB1 + k] = a;
            gp[oB2 + k] = c;
        } else {
            for (int q = 0; q < kGB; q++) {
                a = fmaf(S.h2[q][k], S.dy[q], a);
                c += k == 0 ? S.dy[q] : S.loss[q];
            }
            gp[oW3 + k] = a;
            if (k == 0) gp[oB3] = c;
            if (k == 1) lpart[blockIdx.x] = c;
        }
    }
}

// Fixed-order reduction of the block partials; then one Adam step (Kingma &
// Ba 2015) on the FP32 master weights and the BF16 working copy.  A block has
// 32 parameters in 32 slices of the partials (every 32nd each, summed in
// order, then the slices in order): with one thread per parameter the chain of
// loads took 17 us for 469 blocks, so it takes 5.5 us for 938.  The last block adds the losses.
constexpr int kRS = 32;
__global__ void __launch_bounds__(32 * kRS) mlp_reduce_adam_kernel(
    int nblocks, const float *__restrict__ gpart, const float *__restrict__ lpart,
    float *__restrict__ grad, float *__restrict__ loss, float *__restrict__ w,
    float *__restrict__ m1, float *__restrict__ m2, __nv_bfloat16 *__restrict__ wb, float lr,
    float b1, float b2, float epsa, float c1, float c2, int do_update) {
    __shared__ float sh[kRS][33];
    const int lane = (int)lane_id(), sl = (int)(threadIdx.x >> 5);
    const bool losses = blockIdx.x == gridDim.x - 1;
    const int p = blockIdx.x * 32 + lane;
    float g = 0.0f;
    if (losses) {
        if (lane == 0)
            for (int b = sl; b < nblocks; b += kRS) g += lpart[b];
    } else if (p < kMlpParams) {
#pragma unroll 8
        for (int b = sl; b < nblocks; b += kRS) g += gpart[(int64_t)b * kMlpParams + p];
    }
    sh[sl][lane] = g;
    __syncthreads();
    if (sl != 0) return;
    g = 0.0f;
#pragma unroll
    for (int k = 0; k < kRS; k++) g += sh[k][lane];
    if (losses) {
        if (lane == 0 && loss) *loss = g;
        return;
    }
    if (p >= kMlpParams) return;
    if (grad) grad[p] = g;
    if (!do_update) return;
    const float mm = b1 * m1[p] + (1.0f - b1) * g;
    const float vv = b2 * m2[p] + (1.0f - b2) * g * g;
    m1[p] = mm;
    m2[p] = vv;
    const float wn = w[p] - lr * (mm * c1) / (sqrtf(vv * c2) + epsa);
    w[p] = wn;
    wb[p] = __float2bfloat16_rn(wn);
}

__global__ void mlp_round_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wb) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < kMlpParams) wb[p] = __float2bfloat16_rn(w[p]);
}

// Mean and standard deviation of each feature and of the raw target over n
// samples (one block): norm = {mean[8], std[8], target mean, target std}.
__global__ void mlp_norm_kernel(const int32_t *__restrict__ pn, const float *__restrict__ feat,
                                const float *__restrict__ target, float *__restrict__ norm) {
    constexpr int C = kIn + 1;
    __shared__ double s1[256][C], s2[256][C];
    const int64_t n = *pn;
    double a[C] = {0}, b[C] = {0};
    for (int64_t g = threadIdx.x; g < n; g += blockDim.x)
        for (int i = 0; i < C; i++) {
            const double v = i < kIn ? feat[g * kIn + i] : target[g];
            a[i] += v;
            b[i] += v * v;
        }
    for (int i = 0; i < C; i++) {
        s1[threadIdx.x][i] = a[i];
        s2[threadIdx.x][i] = b[i];
    }
    __syncthreads();
    if (threadIdx.x < C) {
        double t1 = 0, t2 = 0;
        for (int q = 0; q < 256; q++) {
            t1 += s1[q][threadIdx.x];
            t2 += s2[q][threadIdx.x];
        }
        const double mean = n ? t1 / (double)n : 0.0;
        const double var = n ? t2 / (double)n - mean * mean : 1.0;
        const float sd = (float)sqrt(var > 1e-12 ? var : 1.0);
        if (threadIdx.x < kIn) {
            norm[threadIdx.x] = (float)mean;
            norm[kIn + threadIdx.x] = sd;
        } else {
            norm[2 * kIn] = (float)mean;
            norm[2 * kIn + 1] = sd;
        }
    }
}

// log2 of the logged cost of each group (list entries, at least 1), then
// standardised with the frozen target statistics once they exist.
__global__ void mlp_target_kernel(const int32_t *__restrict__ pn, const int32_t *__restrict__ cost,
                                  const float *__restrict__ tnorm, float *__restrict__ target) {
    const int n = *pn;
    const float tm = tnorm ? tnorm[0] : 0.0f, its = tnorm ? 1.0f / tnorm[1] : 1.0f;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x)
        target[g] = (__log2f((float)max(cost[g], 1)) - tm) * its;
}

// Queue keys: descending score -> ascending key; value = group id.  The score
// of a group is its predicted log2 cost plus log2 of the i-slots it occupies.
__global__ void order_keys_kernel(const int32_t *__restrict__ pn, const float *__restrict__ score,
                                  const int32_t *__restrict__ grp_count, uint64_t *__restrict__ key,
                                  uint32_t *__restrict__ val) {
    const int n = *pn;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const float slots = (float)((grp_count[g] + 31) >> 5);
        const float sc = score[g] + __log2f(slots);
        key[g] = (uint64_t)(~f2ord(sc));
        val[g] = (uint32_t)g;
    }
}

// Last-cost heuristic: score of a group = log2 of the cost its first particle's
// group had in the previous walk.
__global__ void lastcost_score_kernel(const int32_t *__restrict__ pn,
                                      const int32_t *__restrict__ grp_first,
                                      const float *__restrict__ pcost, float *__restrict__ score) {
    const int n = *pn;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x)
        score[g] = __log2f(fmaxf(pcost[grp_first[g]], 1.0f));
}

// Spread each group's logged cost to its particles (sorted order).
__global__ void spread_cost_kernel(const int32_t *__restrict__ pn,
                                   const int32_t *__restrict__ grp_first,
                                   const int32_t *__restrict__ grp_count,
                                   const int32_t *__restrict__ cost, float *__restrict__ pcost) {
    const int n = *pn;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const float c = (float)cost[g];
        for (int k = 0; k < grp_count[g]; k++) pcost[grp_first[g] + k] = c;
    }
}

// ---------------------------------------------------------------- launchers
void launch_mlp_features(cudaStream_t s, const Layout &L, const DevState *ds,
                         const int32_t *grp_first, const int32_t *grp_count,
                         const float4 *grp_sphere, const int32_t *grp_sys, const float *aold,
                         const uint64_t *keys, const float4 *nodeA, const int32_t *sys_root,
                         const SysBox *box, const int64_t *off, float *feat, int nsm) {
    mlp_features_kernel<<<nsm * 8, 256, 0, s>>>(L, ds, grp_first, grp_count, grp_sphere, grp_sys,
                                                aold, keys, nodeA, sys_root, box, off, feat);
}

void launch_mlp_forward(cudaStream_t s, const int32_t *pn, const float *feat,
                        const __nv_bfloat16 *wb, const float *norm, const float *tnorm,
                        float *pred, int nsm) {
    mlp_forward_kernel<<<nsm * 4, 128, 0, s>>>(pn, feat, wb, norm, tnorm, pred);
}

cudaError_t launch_mlp_train_step(cudaStream_t s, const float *feat, const float *target,
                                  int64_t base, int64_t stride, int count,
                                  const __nv_bfloat16 *wb, const float *w32, const float *norm,
                                  float *gpart, float *lpart, float *grad, float *loss, float *w,
                                  float *m1, float *m2, __nv_bfloat16 *wb_out, float lr, int t,
                                  bool update, float *pred) {
    // per call: the attribute belongs to the current device's context
    cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(GradSmem));
    if (e != cudaSuccess) return e;
    const int nb = (count + kGB - 1) / kGB;
    mlp_grad_kernel<<<nb, kGB, sizeof(GradSmem), s>>>(feat, target, base, stride, count,
                                                      1.0f / (float)count, wb, w32, norm, gpart,
                                                      lpart, pred);
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f / (1.0f - powf(b1, (float)t)), c2 = 1.0f / (1.0f - powf(b2, (float)t));
    mlp_reduce_adam_kernel<<<(kMlpParams + 31) / 32 + 1, 32 * kRS, 0, s>>>(
        nb, gpart, lpart, grad, loss, w, m1, m2, wb_out, lr, b1, b2, 1e-8f, c1, c2, update ? 1 : 0);
    return cudaGetLastError();
}

void launch_mlp_round(cudaStream_t s, const float *w, __nv_bfloat16 *wb) {
    mlp_round_kernel<<<(kMlpParams + 255) / 256, 256, 0, s>>>(w, wb);
}

void launch_mlp_norm(cudaStream_t s, const int32_t *pn, const float *feat, const float *target,
                     float *norm) {
    mlp_norm_kernel<<<1, 256, 0, s>>>(pn, feat, target, norm);
}

void launch_mlp_target(cudaStream_t s, const int32_t *pn, const int32_t *cost, const float *tnorm,
                       float *target, int nsm) {
    mlp_target_kernel<<<nsm * 4, 256, 0, s>>>(pn, cost, tnorm, target);
}

void launch_order_keys(cudaStream_t s, const int32_t *pn, const float *score,
                       const int32_t *grp_count, uint64_t *key, uint32_t *val, int nsm) {
    order_keys_kernel<<<nsm * 4, 256, 0, s>>>(pn, score, grp_count, key, val);
}

void launch_lastcost_score(cudaStream_t s, const int32_t *pn, const int32_t *grp_first,
                           const float *pcost, float *score, int nsm) {
    lastcost_score_kernel<<<nsm * 4, 256, 0, s>>>(pn, grp_first, pcost, score);
}

void launch_spread_cost(cudaStream_t s, const int32_t *pn, const int32_t *grp_first,
                        const int32_t *grp_count, const int32_t *cost, float *pcost, int nsm) {
    spread_cost_kernel<<<nsm * 8, 256, 0, s>>>(pn, grp_first, grp_count, cost, pcost);
}

}  // namespace nb
