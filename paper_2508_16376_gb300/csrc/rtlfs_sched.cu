// rtlfs_sched.cu -- the learned and heuristic schedulers: per-fault features, the load
// predictor (a 5-64-64-1 MLP with BF16 weights and FP32 accumulation on the CUDA cores),
// its training kernels, and the device-side ordering of the work queue.
//
// The paper balances load with a runtime monitor: a node whose share of the run time
// exceeds a threshold is split over the fault dimension (Sec. IV-C-2). Here the same
// decision -- which work is heavy and what runs first -- is taken before the faulty
// kernels start, from a prediction of each fault's propagation load (node evaluations
// summed over cycles, which the simulator records). The prediction only orders and
// assigns work; results never depend on it.
#include "rtlfs_internal.h"
#include "rtlfs_sched.h"

#include <cuda_bf16.h>

namespace rtlfs {

// ---- features ------------------------------------------------------------------------
// One warp per fault: static features come from per-net tables built at load time, the
// toggle rate of the site bit from the good trace (lanes read 32 consecutive cycles).
__global__ void features_kernel(const DevDesign *__restrict__ designs, DevFaults f,
                                const float *__restrict__ const *net_static, float *X,
                                float *heur, uint32_t t_limit) {
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t lane = threadIdx.x & 31u;
    if (warp >= f.F) return;
    const uint32_t fid = warp;
    const uint32_t di = f.design[fid];
    const DevDesign &D = designs[di];
    const uint32_t site = f.site[fid], bit = f.bit[fid];
    const uint64_t *col = D.gcol + (size_t)site * D.T;
    const uint32_t T = min(D.T, t_limit);   // cycles the toggle rate is measured over
    uint32_t toggles = 0;
    uint32_t prev_last = 0;   // bit at the last cycle of the previous 32-cycle block
    for (uint32_t t0 = 0; t0 < T; t0 += 32) {
        const uint32_t t = t0 + lane;
        const uint32_t b = t < T ? (uint32_t)((__ldg(col + t) >> bit) & 1ull) : 0u;
        const uint32_t bits = __ballot_sync(0xFFFFFFFFu, b);
        const uint32_t valid = (T - t0) >= 32 ? 0xFFFFFFFFu : ((1u << (T - t0)) - 1u);
        // toggles inside the block, plus across the block boundary
        const uint32_t shifted = (bits << 1) | (t0 ? prev_last : (bits & 1u));
        toggles += __popc((bits ^ shifted) & valid);
        const uint32_t last = 31 - __clz(valid);
        prev_last = (bits >> last) & 1u;
    }
    if (lane == 0) {
        const float *ns = net_static[di];   // [n_net][4]: cone, level, regdepth, width
        const float cone = ns[4 * (size_t)site + 0];
        const float tog = T > 1 ? (float)toggles / (float)(T - 1) : 0.f;
        float *x = X + (size_t)fid * MLP_IN;
        x[0] = cone;
        x[1] = ns[4 * (size_t)site + 1];
        x[2] = ns[4 * (size_t)site + 2];
        x[3] = ns[4 * (size_t)site + 3];
        x[4] = tog;
        // heuristic score: static cone size x toggle rate (both as fractions of their range)
        heur[fid] = cone * tog;
    }
}

// ---- MLP -------------------------------------------------------------------------------
// Parameter layout (MLP_PARAMS values): W1[5][64], b1[64], W2[64][64], b2[64], w3[64], b3.
// W1[i][j] connects input i to hidden unit j; W2[i][j] hidden-1 unit i to hidden-2 unit j.
__device__ __forceinline__ void load_params(const __nv_bfloat16 *__restrict__ wb, float *sw) {
    for (uint32_t i = threadIdx.x; i < MLP_PARAMS; i += blockDim.x) sw[i] = __bfloat162float(wb[i]);
}

// One thread per sample; weights (as FP32 copies of the BF16 values) in shared memory.
__global__ void mlp_forward_kernel(const __nv_bfloat16 *__restrict__ wb, const float *__restrict__ X,
                                   uint32_t n, float *y) {
    __shared__ __align__(16) float sw[MLP_PARAMS];
    load_params(wb, sw);
    __syncthreads();
    const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const float *W1 = sw, *b1 = sw + MLP_OFF_B1, *W2 = sw + MLP_OFF_W2, *b2 = sw + MLP_OFF_B2;
    const float *w3 = sw + MLP_OFF_W3;
    float x[MLP_IN];
#pragma unroll
    for (int i = 0; i < MLP_IN; ++i) x[i] = X[(size_t)s * MLP_IN + i];
    float h1[MLP_H];
#pragma unroll
    for (int j = 0; j < MLP_H; ++j) {
        float a = b1[j];
#pragma unroll
        for (int i = 0; i < MLP_IN; ++i) a = fmaf(x[i], W1[i * MLP_H + j], a);
        h1[j] = a > 0.f ? a : 0.f;
    }
    float out = sw[MLP_OFF_B3];
#pragma unroll 1
    for (int j = 0; j < MLP_H; j += 4) {   // four units per 16-byte read of W2, the same for all lanes
        float a[4] = {b2[j], b2[j + 1], b2[j + 2], b2[j + 3]};
#pragma unroll
        for (int i = 0; i < MLP_H; ++i) {
            const float4 w = *reinterpret_cast<const float4 *>(W2 + i * MLP_H + j);
            a[0] = fmaf(h1[i], w.x, a[0]);
            a[1] = fmaf(h1[i], w.y, a[1]);
            a[2] = fmaf(h1[i], w.z, a[2]);
            a[3] = fmaf(h1[i], w.w, a[3]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) out = fmaf(a[k] > 0.f ? a[k] : 0.f, w3[j + k], out);
    }
    y[s] = out;
}

// Forward + backward of the mean squared error over n samples. A CTA walks tiles of 16 * SPT samples;
// its three 64-wide products per tile (layer 2, its input gradient, the gradient of W2) are register
// tiled: thread (ty, tx) holds SPT consecutive samples x the four units tx + 16 k, or the 4 x 4 block
// of W2's gradient, whose rows it keeps in registers over all tiles, as the other gradients, and
// adds to grad once (FP32 atomics; squared errors into loss_sum). Activations lie by unit and then
// sample, padded by four: both kinds of read are 16-byte loads without bank conflicts.
// Bound by the FP32 multiply-adds (1.8 GFLOP of them at 65537 samples). One output per thread with
// two shared loads per multiply-add, and an atomic per parameter and tile of 64 samples and per
// sample's error, made a call with 65537 samples 440 us; it is 123 so, half of it the copies.
template <int SPT> struct GradVec { float v[SPT]; };
template <int SPT> __device__ __forceinline__ GradVec<SPT> ld_vec(const float *p) {
    GradVec<SPT> r;
    if constexpr (SPT == 2) {
        const float2 a = *reinterpret_cast<const float2 *>(p);
        r.v[0] = a.x; r.v[1] = a.y;
    } else {
#pragma unroll
        for (int k = 0; k < SPT; k += 4) {
            const float4 a = *reinterpret_cast<const float4 *>(p + k);
            r.v[k] = a.x; r.v[k + 1] = a.y; r.v[k + 2] = a.z; r.v[k + 3] = a.w;
        }
    }
    return r;
}
template <int SPT> __device__ __forceinline__ void st_vec(float *p, const GradVec<SPT> &r) {
    if constexpr (SPT == 2) {
        *reinterpret_cast<float2 *>(p) = make_float2(r.v[0], r.v[1]);
    } else {
#pragma unroll
        for (int k = 0; k < SPT; k += 4) *reinterpret_cast<float4 *>(p + k) = make_float4(r.v[k], r.v[k + 1], r.v[k + 2], r.v[k + 3]);
    }
}

constexpr int GRAD_W1 = 2 * MLP_H * MLP_H;   // shared floats: W2 by rows and by columns, then
constexpr int GRAD_B1 = GRAD_W1 + MLP_IN * MLP_H, GRAD_B2 = GRAD_B1 + MLP_H, GRAD_W3 = GRAD_B2 + MLP_H;
constexpr int GRAD_B3 = GRAD_W3 + MLP_H, GRAD_ACT = GRAD_B3 + 4;
template <int SPT> constexpr int grad_floats() { return GRAD_ACT + 2 * MLP_H * (16 * SPT + 4) + MLP_IN * 16 * SPT; }

template <int SPT>
__global__ void __launch_bounds__(256, 2)
mlp_grad_kernel(const __nv_bfloat16 *__restrict__ wb, const float *__restrict__ X,
                const float *__restrict__ tgt, uint32_t n, float *grad, float *loss_sum) {
    constexpr int H = MLP_H, S = 16 * SPT, LD = S + 4;
    static_assert(H == 64, "16 x 16 threads hold four units each");
    extern __shared__ __align__(16) float gsh[];
    float *const w2r = gsh, *const w2c = gsh + H * H;   // [i][4 tx + k] = W2[i][tx + 16 k]; [j][4 tx + k] = W2[tx + 16 k][j]
    float *const W1 = gsh + GRAD_W1, *const b1 = gsh + GRAD_B1, *const b2 = gsh + GRAD_B2, *const w3 = gsh + GRAD_W3;
    float *const h1 = gsh + GRAD_ACT, *const d2 = h1 + H * LD, *const xs = d2 + H * LD;   // [unit][LD], [input][S]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int k = tid; k < MLP_PARAMS; k += 256) {
        const float w = __bfloat162float(wb[k]);
        if (k >= MLP_OFF_W2 && k < MLP_OFF_B2) {
            const int i = (k - MLP_OFF_W2) / H, j = (k - MLP_OFF_W2) % H;
            w2r[i * H + (j & 15) * 4 + (j >> 4)] = w;
            w2c[j * H + (i & 15) * 4 + (i >> 4)] = w;
        } else if (k < MLP_OFF_W2) {
            W1[k] = w;   // W1, b1
        } else {
            b2[k - MLP_OFF_B2] = w;   // b2, w3, b3
        }
    }
    float g2[4][4] = {}, g1[MLP_IN][4] = {}, gb1[4] = {}, gb2[4] = {}, gw3[4] = {}, gb3 = 0.f, loss = 0.f;
    const uint32_t tiles = n / S + (n % S != 0);
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const uint32_t s0 = tile * S;
        __syncthreads();   // the last tile's reads, and the weights
        for (int k = tid; k < S * MLP_IN; k += 256) {
            const int s = k / MLP_IN;
            xs[(k % MLP_IN) * S + s] = s0 + s < n ? X[(size_t)s0 * MLP_IN + k] : 0.f;
        }
        __syncthreads();
        for (int k = tid; k < S * H; k += 256) {   // layer 1
            const int j = k / S, s = k % S;
            float a = b1[j];
#pragma unroll
            for (int i = 0; i < MLP_IN; ++i) a = fmaf(xs[i * S + s], W1[i * H + j], a);
            h1[j * LD + s] = a > 0.f ? a : 0.f;
        }
        float t[SPT];
#pragma unroll
        for (int p = 0; p < SPT; ++p) t[p] = s0 + ty * SPT + p < n ? tgt[s0 + ty * SPT + p] : 0.f;
        __syncthreads();
        float acc[SPT][4];
#pragma unroll
        for (int p = 0; p < SPT; ++p)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[p][k] = b2[tx + 16 * k];
#pragma unroll 4
        for (int i = 0; i < H; ++i) {   // layer 2
            const GradVec<SPT> a = ld_vec<SPT>(h1 + i * LD + ty * SPT);
            const GradVec<4> w = ld_vec<4>(w2r + i * H + tx * 4);
#pragma unroll
            for (int p = 0; p < SPT; ++p)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[p][k] = fmaf(a.v[p], w.v[k], acc[p][k]);
        }
        // output, error and dL/dy = 2 (y - t) / n; dL/d(pre-activation 2)
        float dy[SPT];
#pragma unroll
        for (int p = 0; p < SPT; ++p) {
            float out = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc[p][k] = acc[p][k] > 0.f ? acc[p][k] : 0.f;
                out = fmaf(acc[p][k], w3[tx + 16 * k], out);
            }
#pragma unroll
            for (int o = 8; o; o >>= 1) out += __shfl_xor_sync(0xFFFFFFFFu, out, o);
            const float e = s0 + ty * SPT + p < n ? out + gsh[GRAD_B3] - t[p] : 0.f;
            dy[p] = 2.f * e / (float)n;
            if (tx == 0) {
                loss = fmaf(e, e, loss);
                gb3 += dy[p];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            GradVec<SPT> d;
#pragma unroll
            for (int p = 0; p < SPT; ++p) {
                d.v[p] = acc[p][k] > 0.f ? w3[tx + 16 * k] * dy[p] : 0.f;
                gb2[k] += d.v[p];
                gw3[k] = fmaf(acc[p][k], dy[p], gw3[k]);
            }
            st_vec<SPT>(d2 + (tx + 16 * k) * LD + ty * SPT, d);
        }
        __syncthreads();
#pragma unroll
        for (int p = 0; p < SPT; ++p)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[p][k] = 0.f;
#pragma unroll 4
        for (int j = 0; j < H; ++j) {   // dL/d(activation 1)
            const GradVec<SPT> a = ld_vec<SPT>(d2 + j * LD + ty * SPT);
            const GradVec<4> w = ld_vec<4>(w2c + j * H + tx * 4);
#pragma unroll
            for (int p = 0; p < SPT; ++p)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[p][k] = fmaf(w.v[k], a.v[p], acc[p][k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const GradVec<SPT> a = ld_vec<SPT>(h1 + (tx + 16 * k) * LD + ty * SPT);
#pragma unroll
            for (int p = 0; p < SPT; ++p) {
                acc[p][k] = a.v[p] > 0.f ? acc[p][k] : 0.f;
                gb1[k] += acc[p][k];
            }
        }
#pragma unroll
        for (int i = 0; i < MLP_IN; ++i) {
            const GradVec<SPT> x = ld_vec<SPT>(xs + i * S + ty * SPT);
#pragma unroll
            for (int p = 0; p < SPT; ++p)
#pragma unroll
                for (int k = 0; k < 4; ++k) g1[i][k] = fmaf(x.v[p], acc[p][k], g1[i][k]);
        }
#pragma unroll 2
        for (int s = 0; s < S; s += 4) {   // W2, rows ty + 16 i
            GradVec<4> a[4], d[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                a[k] = ld_vec<4>(h1 + (ty + 16 * k) * LD + s);
                d[k] = ld_vec<4>(d2 + (tx + 16 * k) * LD + s);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int k = 0; k < 4; ++k) g2[i][k] = fmaf(a[i].v[q], d[k].v[q], g2[i][k]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) atomicAdd(grad + MLP_OFF_W2 + (ty + 16 * i) * H + tx + 16 * k, g2[i][k]);
    // the rest over the 16 rows of threads: a warp's two, then the eight warps
    constexpr int V = 4 * (MLP_IN + 3);
    float *const red = h1;   // [8][16][V]
    static_assert(8 * 16 * V <= 2 * H * LD, "the reduction lies over the activations");
    __syncthreads();
    float own[V];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int i = 0; i < MLP_IN; ++i) own[4 * i + k] = g1[i][k];
        own[4 * MLP_IN + k] = gb1[k];
        own[4 * MLP_IN + 4 + k] = gb2[k];
        own[4 * MLP_IN + 8 + k] = gw3[k];
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        own[v] += __shfl_xor_sync(0xFFFFFFFFu, own[v], 16);
        if (tid % 32 < 16) red[((tid >> 5) * V + v) * 16 + tx] = own[v];
    }
    loss += __shfl_xor_sync(0xFFFFFFFFu, loss, 16);
    gb3 += __shfl_xor_sync(0xFFFFFFFFu, gb3, 16);
    if (tid % 32 == 0) {
        gsh[2 * (tid >> 5)] = loss;   // over the weights, whose last reads lie before the barrier
        gsh[2 * (tid >> 5) + 1] = gb3;
    }
    __syncthreads();
    for (int k = tid; k < 16 * V; k += 256) {
        const int v = k >> 4, u = (k & 15) + 16 * (v & 3), what = v >> 2;   // unit; input, b1, b2, w3
        float a = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) a += red[w * V * 16 + k];
        const int at = what < MLP_IN ? what * H : what == MLP_IN ? MLP_OFF_B1 : what == MLP_IN + 1 ? MLP_OFF_B2 : MLP_OFF_W3;
        atomicAdd(grad + at + u, a);
    }
    if (tid < 2) {
        float a = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) a += gsh[2 * w + tid];
        atomicAdd(tid == 0 ? loss_sum : grad + MLP_OFF_B3, a);
    }
}

// Adam step on the FP32 master parameters; the BF16 copy (round to nearest even) is what
// the forward pass uses. Clears the gradient for the next step.
__global__ void mlp_adam_kernel(float *master, __nv_bfloat16 *wb, float *grad, float *m, float *v,
                                float lr, float beta1, float beta2, float eps, float bc1, float bc2) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= MLP_PARAMS) return;
    const float g = grad[i];
    const float mi = beta1 * m[i] + (1.f - beta1) * g;
    const float vi = beta2 * v[i] + (1.f - beta2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float p = master[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    master[i] = p;
    wb[i] = __float2bfloat16_rn(p);
    grad[i] = 0.f;
}

// ---- queue order -----------------------------------------------------------------------
// Counting sort of the faults by score, descending, into SORT_BUCKETS buckets over [lo, hi].
// With k > 0 score classes (a power of two up to 64) the buckets are k classes of
// SORT_BUCKETS / k sub-buckets each: fault i of n goes to its class's sub-bucket
// i * (SORT_BUCKETS / k) / n, so inside a class the queue keeps the fault-list order (by
// site), at the granularity of a sub-bucket. Every bucket index is below SORT_BUCKETS.
__device__ __forceinline__ uint32_t bucket_of(float s, float lo, float hi, uint32_t i, uint32_t n,
                                              uint32_t k) {
    float u = hi > lo ? (s - lo) / (hi - lo) : 0.f;
    u = fminf(fmaxf(u, 0.f), 1.f);
    if (k == 0) {
        const uint32_t b = (uint32_t)(u * (float)(SORT_BUCKETS - 1) + 0.5f);
        return (SORT_BUCKETS - 1) - b;    // descending score = ascending bucket
    }
    const uint32_t per = SORT_BUCKETS / k;
    const uint32_t c = min((uint32_t)(u * (float)k), k - 1u);
    const uint32_t sb = min((uint32_t)(((uint64_t)i * per) / max(n, 1u)), per - 1u);
    return (k - 1u - c) * per + sb;
}

__device__ __forceinline__ int map_key(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : (int)(0x80000000u - (uint32_t)i);
}

__global__ void minmax_init_kernel(float *mm) {
    reinterpret_cast<int *>(mm)[0] = map_key(3.0e38f);
    reinterpret_cast<int *>(mm)[1] = map_key(-3.0e38f);
}

__device__ __forceinline__ float unmap_key(int k) {
    return k >= 0 ? __int_as_float(k) : __int_as_float((int)(0x80000000u - (uint32_t)k));
}

__global__ void minmax_kernel(const float *score, uint32_t n, float *mm) {
    float lo = 3.0e38f, hi = -3.0e38f;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        lo = fminf(lo, score[i]);
        hi = fmaxf(hi, score[i]);
    }
    for (int o = 16; o; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xFFFFFFFFu, hi, o));
    }
    if ((threadIdx.x & 31u) == 0) {
        // order-preserving float -> int mapping so that integer atomics compare floats
        atomicMin(reinterpret_cast<int *>(mm) + 0, map_key(lo));
        atomicMax(reinterpret_cast<int *>(mm) + 1, map_key(hi));
    }
}

__global__ void histogram_kernel(const float *score, uint32_t n, const float *mm, uint32_t *hist,
                                 uint32_t k) {
    __shared__ uint32_t h[SORT_BUCKETS];
    for (uint32_t b = threadIdx.x; b < SORT_BUCKETS; b += blockDim.x) h[b] = 0;
    __syncthreads();
    const float lo = unmap_key(reinterpret_cast<const int *>(mm)[0]);
    const float hi = unmap_key(reinterpret_cast<const int *>(mm)[1]);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        atomicAdd(&h[bucket_of(score[i], lo, hi, i, n, k)], 1u);
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < SORT_BUCKETS; b += blockDim.x)
        if (h[b]) atomicAdd(&hist[b], h[b]);
}

// Single CTA: exclusive scan of the histogram into bucket cursors.
__global__ void scan_kernel(uint32_t *hist) {
    __shared__ uint32_t part[1024];
    const uint32_t tid = threadIdx.x;
    constexpr uint32_t PER = SORT_BUCKETS / 1024;
    uint32_t loc[PER], sum = 0;
    for (uint32_t k = 0; k < PER; ++k) { loc[k] = hist[tid * PER + k]; sum += loc[k]; }
    part[tid] = sum;
    __syncthreads();
    for (uint32_t off = 1; off < 1024; off <<= 1) {
        const uint32_t v = tid >= off ? part[tid - off] : 0u;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    uint32_t run = part[tid] - sum;
    for (uint32_t k = 0; k < PER; ++k) { hist[tid * PER + k] = run; run += loc[k]; }
}

// Scatter fault ids into their buckets (order inside a bucket is unspecified), then the
// first n_heavy go to the heavy kernel's initial list and the rest form the light queue.
__global__ void scatter_kernel(const float *score, uint32_t n, const float *mm, uint32_t *cursor,
                               uint32_t *order, uint32_t k) {
    const float lo = unmap_key(reinterpret_cast<const int *>(mm)[0]);
    const float hi = unmap_key(reinterpret_cast<const int *>(mm)[1]);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t p = atomicAdd(&cursor[bucket_of(score[i], lo, hi, i, n, k)], 1u);
        order[p] = i;
    }
}

__global__ void heavy_items_kernel(const uint32_t *order, uint32_t n_heavy, HeavyItem *items) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_heavy) return;
    HeavyItem h{};
    h.fault = order[i];
    items[i] = h;
}

// ---- launchers ------------------------------------------------------------------------

cudaError_t launch_features(const DevDesign *d_designs, DevFaults f, const float *const *net_static,
                            float *X, float *heur, cudaStream_t s, uint32_t t_limit) {
    if (!f.F) return cudaSuccess;
    const uint32_t threads = 256, warps_per = threads / 32;
    features_kernel<<<(f.F + warps_per - 1) / warps_per, threads, 0, s>>>(d_designs, f, net_static, X, heur,
                                                                          t_limit);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const void *wb, const float *X, uint32_t n, float *y, cudaStream_t s) {
    if (!n) return cudaSuccess;
    mlp_forward_kernel<<<(n + 127) / 128, 128, 0, s>>>((const __nv_bfloat16 *)wb, X, n, y);
    return cudaGetLastError();
}

cudaError_t launch_mlp_grad(const void *wb, const float *X, const float *t, uint32_t n, float *grad,
                            float *loss_sum, uint32_t n_sm, cudaStream_t s) {
    if (!n) return cudaSuccess;
    // Tiles of 128 samples when they fill the SMs (152: from 19456 samples), else of 32, for more CTAs; two per SM
    // (65537 samples, the call: 123 us; one CTA per SM 127-135, tiles of 64 126).
    const bool big = n >= n_sm * 128u;
    const uint32_t S = big ? 128 : 32, tiles = n / S + (n % S != 0), grid = tiles < 2 * n_sm ? tiles : 2 * n_sm;
    const size_t smem = (big ? grad_floats<8>() : grad_floats<2>()) * sizeof(float);
    const auto fn = big ? mlp_grad_kernel<8> : mlp_grad_kernel<2>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    fn<<<grid, 256, smem, s>>>((const __nv_bfloat16 *)wb, X, t, n, grad, loss_sum);
    return cudaGetLastError();
}

cudaError_t launch_mlp_adam(float *master, void *wb, float *grad, float *m, float *v, float lr,
                            float beta1, float beta2, float eps, int step, cudaStream_t s) {
    const float bc1 = 1.f - powf(beta1, (float)step), bc2 = 1.f - powf(beta2, (float)step);
    mlp_adam_kernel<<<(MLP_PARAMS + 255) / 256, 256, 0, s>>>(master, (__nv_bfloat16 *)wb, grad, m, v, lr,
                                                            beta1, beta2, eps, bc1, bc2);
    return cudaGetLastError();
}

cudaError_t launch_order(const float *score, uint32_t n, float *mm, uint32_t *hist, uint32_t *order,
                         uint32_t n_heavy, HeavyItem *items, cudaStream_t s, uint32_t classes) {
    if (!n) return cudaSuccess;
    if (classes > 64 || (classes & (classes - 1))) return cudaErrorInvalidValue;
    minmax_init_kernel<<<1, 1, 0, s>>>(mm);
    cudaError_t e = cudaMemsetAsync(hist, 0, SORT_BUCKETS * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    const uint32_t g = (n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024;
    minmax_kernel<<<g, 256, 0, s>>>(score, n, mm);
    histogram_kernel<<<g, 256, 0, s>>>(score, n, mm, hist, classes);
    scan_kernel<<<1, 1024, 0, s>>>(hist);
    scatter_kernel<<<g, 256, 0, s>>>(score, n, mm, hist, order, classes);
    if (n_heavy) heavy_items_kernel<<<(n_heavy + 255) / 256, 256, 0, s>>>(order, n_heavy, items);
    return cudaGetLastError();
}

}  // namespace rtlfs
