// Kernels of the learned warm start: a 3D convolutional encoder-decoder trained and run with BF16
// activations and weights, FP32 accumulation, FP32 master weights and gradients.  The forward and
// backward-data convolutions and the weight gradient run on tcgen05 (pfnn_umma.cu); this file holds the
// data-movement, head and optimiser kernels.
//
// Layout: activations N x D x H x W x C (channels last), bf16; a tensor may be a channel slice
// [off, off + C) of a wider buffer with ld channels per voxel (skip concatenation is free).
// Convolutions are 3x3x3 with zero padding 1 and stride 1; weights are [27][Cout][Cin] bf16 with
// tap t = (dz+1)*9 + (dy+1)*3 + (dx+1).
//
// Implicit GEMM (forward): D[v][co] = sum over (t, ci) of X[v + off(t)][ci] W[t][co][ci].
// Backward data is the same GEMM on dY with flipped taps and transposed weights [27][Cin][Cout]:
//   dX[v][ci] = sum over (t, co) of dY[v - off(t)][co] W[t][co][ci].
// Backward weight, per tap: dW[t][co][ci] = sum over v of dY[v][co] X[v + off(t)][ci] (pfnn_umma.cu).
#include "../../include/pfnn.h"
#include "pf_internal.cuh"

#include <cuda_bf16.h>
#include <cstdint>
#include <initializer_list>
#include <type_traits>

namespace {

// The data-movement kernels move whole 16-byte vectors: a thread owns V consecutive channels of a voxel
// (V = 8 bf16 or 4 fp32) when the channel count, the leading dimensions, the offsets and the pointers allow
// it, else single channels (V = 1).  They are bound by memory; with one channel per thread they were bound
// by the index divisions instead (64-bit, one set per 2 or 4 bytes).  IX is unsigned where the item count
// is below 2^31 (32-bit divisions), else unsigned long long.

// V consecutive bf16 <-> fp32 registers
template <int V>
__device__ __forceinline__ void load_bf(const __nv_bfloat16* __restrict__ p, float (&f)[V]) {
    if constexpr (V == 8) {
        const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            f[2 * q] = __uint_as_float(w[q] << 16);
            f[2 * q + 1] = __uint_as_float(w[q] & 0xFFFF0000u);
        }
    } else {
        f[0] = __bfloat162float(p[0]);
    }
}
template <int V>
__device__ __forceinline__ void store_bf(__nv_bfloat16* p, const float (&f)[V]) {
    if constexpr (V == 8) {
        uint4 u;
        uint32_t* w = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(f[2 * q], f[2 * q + 1]);
            w[q] = *reinterpret_cast<const uint32_t*>(&h2);
        }
        *reinterpret_cast<uint4*>(p) = u;
    } else {
        p[0] = __float2bfloat16_rn(f[0]);
    }
}
template <int V>
__device__ __forceinline__ void load_f(const float* p, float (&f)[V]) {
    if constexpr (V % 4 == 0) {
#pragma unroll
        for (int q = 0; q < V / 4; ++q) {
            const float4 u = reinterpret_cast<const float4*>(p)[q];
            f[4 * q] = u.x; f[4 * q + 1] = u.y; f[4 * q + 2] = u.z; f[4 * q + 3] = u.w;
        }
    } else {
        f[0] = p[0];
    }
}
template <int V>
__device__ __forceinline__ void store_f(float* p, const float (&f)[V]) {
    if constexpr (V % 4 == 0) {
#pragma unroll
        for (int q = 0; q < V / 4; ++q)
            reinterpret_cast<float4*>(p)[q] = make_float4(f[4 * q], f[4 * q + 1], f[4 * q + 2], f[4 * q + 3]);
    } else {
        p[0] = f[0];
    }
}

// item -> channel of its vector, coarse voxel cv (linear) and linear index of the first of its eight
// children; offsets of the others: + 1 along x, + W along y, + H W along z (D, H, W: the fine grid)
template <int V, typename IX>
__device__ __forceinline__ void coarse_item(IX q, int c, int D, int H, int W, int& ch, IX& cv, IX& fv) {
    const IX nc = (IX)(c / V);
    ch = (int)(q % nc) * V;
    cv = q / nc;
    const IX w2 = W / 2, h2 = H / 2, d2 = D / 2;
    const IX x = cv % w2;
    IX r = cv / w2;
    const IX y = r % h2;
    r /= h2;
    const IX z = r % d2, b = r / d2;
    fv = ((b * D + 2 * z) * H + 2 * y) * (IX)W + 2 * x;
}
// child o (z, y, x bits) of a coarse cell
__device__ __forceinline__ long long child(int o, int H, int W) {
    return ((long long)(o >> 2) * H + ((o >> 1) & 1)) * W + (o & 1);
}

// Sums of the block's threads that own the same channels: thread t owns V channels starting at V (t % nc),
// nc | 256.  One atomic per channel and block, consecutive channels by consecutive threads (a warp's atomics are then one
// request to L2 for 32 channels; with the V channels of a thread apart they were four or eight, and 128 channels on 32^3 voxels took
// 25 us where the sums take 8).  Up to 16 owners a warp first add up by shuffles, so that a thread adds 8 nc of 32 values at
// most (4 channels on 32^3 10.4 us, of which the one thread per channel that added 256 values took three).
template <int V>
__device__ __forceinline__ void block_channel_sums(float (&acc)[V], int nc, float* sh, float* out) {
    const int step = nc < 32 ? 32 : nc;  // threads of the block that hold a sum: the first nc of every `step`
    for (int o = 16; o >= nc; o >>= 1)
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
#pragma unroll
    for (int q = 0; q < V; ++q) sh[q * 256 + threadIdx.x] = acc[q];
    __syncthreads();
    for (int k = threadIdx.x; k < V * nc; k += 256) {
        const int j = k / V, q = k - j * V;
        float t = 0.f;
        for (int m = j; m < 256; m += step) t += sh[q * 256 + m];
        atomicAdd(out + k, t);
    }
}

// c / V divides 256: the grid's stride is a multiple of it, so a thread keeps its channels
template <int V>
__global__ void __launch_bounds__(256) k_bias_grad(const float* __restrict__ dz, int ld, int off, int c, long long nvox,
                                                   float* db) {
    __shared__ float sh[V * 256];
    const int nc = c / V, ch = (int)(threadIdx.x % nc) * V, per = 256 / nc;
    float acc[V];
#pragma unroll
    for (int q = 0; q < V; ++q) acc[q] = 0.f;
    for (long long v = blockIdx.x * (long long)per + threadIdx.x / nc; v < nvox; v += (long long)gridDim.x * per) {
        float f[V];
        load_f<V>(dz + v * ld + off + ch, f);
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q] += f[q];
    }
    block_channel_sums<V>(acc, nc, sh, db);
}

// any channel count: one block column per 32 channels x 8 voxel lanes
__global__ void k_bias_grad_any(const float* __restrict__ dz, int ld, int off, int c, long long nvox, float* db) {
    const int ch = blockIdx.y * 32 + (threadIdx.x & 31);
    float s = 0.f;
    if (ch < c)
        for (long long v = blockIdx.x * 8 + (threadIdx.x >> 5); v < nvox; v += (long long)gridDim.x * 8)
            s += dz[v * ld + off + ch];
    __shared__ float sh[256];
    sh[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x < 32 && ch < c) {
        float t = 0.f;
        for (int q = 0; q < 8; ++q) t += sh[q * 32 + threadIdx.x];
        atomicAdd(&db[ch], t);
    }
}

// dz = dy * (y > 0) cast to bf16 (ReLU backward), or plain cast when y is NULL
template <int V, typename IX>
__global__ void __launch_bounds__(256)
k_relu_bwd_cast(const float* __restrict__ dy, int lddy, int dyoff, const __nv_bfloat16* __restrict__ y, int ldy, int yoff,
                int c, long long n, float* __restrict__ dzf, __nv_bfloat16* __restrict__ dzb) {
    const IX nc = (IX)(c / V);
    for (IX q = blockIdx.x * (IX)256 + threadIdx.x; q < (IX)n; q += (IX)gridDim.x * 256) {
        const long long v = q / nc;
        const int ch = (int)(q % nc) * V;
        float g[V], m[V];
        load_f<V>(dy + v * lddy + dyoff + ch, g);
        if (y) {
            load_bf<V>(y + v * ldy + yoff + ch, m);
#pragma unroll
            for (int k = 0; k < V; ++k) g[k] = m[k] > 0.f ? g[k] : 0.f;
        }
        if (dzf) store_f<V>(dzf + v * c + ch, g);
        store_bf<V>(dzb + v * c + ch, g);
    }
}

// The two above in one pass, without the fp32 copy of dz: the masked gradient goes to bf16 and its fp32
// values into the bias sums (V = 8, c / 8 divides 256, so a thread keeps its channels).  Memory bound: reads
// 4 + 2 bytes and writes 2 per value, where the two passes read 4 + 2 + 4 and write 4 + 2.
__global__ void __launch_bounds__(256)
k_relu_bwd_bias(const float* __restrict__ dy, int lddy, int dyoff, const __nv_bfloat16* __restrict__ y, int ldy, int yoff,
                int c, long long nvox, __nv_bfloat16* __restrict__ dzb, float* db) {
    __shared__ float sh[8 * 256];
    const int nc = c / 8, ch = (int)(threadIdx.x % nc) * 8, per = 256 / nc;
    float acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.f;
    for (long long v = blockIdx.x * (long long)per + threadIdx.x / nc; v < nvox; v += (long long)gridDim.x * per) {
        float g[8], m[8];
        load_f<8>(dy + v * lddy + dyoff + ch, g);
        load_bf<8>(y + v * ldy + yoff + ch, m);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            g[q] = m[q] > 0.f ? g[q] : 0.f;
            acc[q] += g[q];
        }
        store_bf<8>(dzb + v * c + ch, g);
    }
    block_channel_sums<8>(acc, nc, sh, db);
}

// [27][Cout][Cin] -> [27][Cin][Cout]
__global__ void k_wtranspose(const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wt, int cout, int cin) {
    const long long n = 27LL * cout * cin;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const int ci = (int)(q % cin);
        const int co = (int)((q / cin) % cout);
        const int t = (int)(q / ((long long)cin * cout));
        wt[((long long)t * cin + ci) * cout + co] = w[q];
    }
}

// 2x2x2 average pooling of a channel slice (even sizes), and its adjoint: a thread owns V channels of one
// coarse cell and its eight children
template <int V, typename IX>
__global__ void __launch_bounds__(256)
k_avgpool(const __nv_bfloat16* __restrict__ x, int ldx, int xoff, __nv_bfloat16* __restrict__ y, int ldy, int yoff, int c,
          long long n, int D, int H, int W) {
    for (IX q = blockIdx.x * (IX)256 + threadIdx.x; q < (IX)n; q += (IX)gridDim.x * 256) {
        int ch;
        IX cv, fv;
        coarse_item<V, IX>(q, c, D, H, W, ch, cv, fv);
        float s[V];
#pragma unroll
        for (int k = 0; k < V; ++k) s[k] = 0.f;
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            float f[V];
            load_bf<V>(x + ((long long)fv + child(o, H, W)) * ldx + xoff + ch, f);
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] += f[k];
        }
#pragma unroll
        for (int k = 0; k < V; ++k) s[k] *= 0.125f;
        store_bf<V>(y + (long long)cv * ldy + yoff + ch, s);
    }
}

template <int V, typename IX>
__global__ void __launch_bounds__(256)
k_avgpool_bwd(const float* __restrict__ dy, int c, float* __restrict__ dx, int lddx, int dxoff, long long n, int D, int H,
              int W) {
    for (IX q = blockIdx.x * (IX)256 + threadIdx.x; q < (IX)n; q += (IX)gridDim.x * 256) {
        int ch;
        IX cv, fv;
        coarse_item<V, IX>(q, c, D, H, W, ch, cv, fv);
        float g[V];
        load_f<V>(dy + (long long)cv * c + ch, g);
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            float* p = dx + ((long long)fv + child(o, H, W)) * lddx + dxoff + ch;
            float f[V];
            load_f<V>(p, f);
#pragma unroll
            for (int k = 0; k < V; ++k) f[k] += 0.125f * g[k];
            store_f<V>(p, f);
        }
    }
}

// x2 nearest-neighbour upsampling of a channel slice (D, H, W of the output), and its adjoint (sum of the 8
// children; D, H, W of the fine gradient)
template <int V, typename IX>
__global__ void __launch_bounds__(256)
k_upsample(const __nv_bfloat16* __restrict__ x, int c, __nv_bfloat16* __restrict__ y, int ldy, int yoff, long long n, int D,
           int H, int W) {
    for (IX q = blockIdx.x * (IX)256 + threadIdx.x; q < (IX)n; q += (IX)gridDim.x * 256) {
        int ch;
        IX cv, fv;
        coarse_item<V, IX>(q, c, D, H, W, ch, cv, fv);
        const __nv_bfloat16* src = x + (long long)cv * c + ch;
        __nv_bfloat16* dst = y + (long long)fv * ldy + yoff + ch;
        if constexpr (V == 8) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(src));
#pragma unroll
            for (int o = 0; o < 8; ++o) *reinterpret_cast<uint4*>(dst + child(o, H, W) * ldy) = u;
        } else {
            const __nv_bfloat16 u = src[0];
#pragma unroll
            for (int o = 0; o < 8; ++o) dst[child(o, H, W) * ldy] = u;
        }
    }
}

template <int V, typename IX>
__global__ void __launch_bounds__(256)
k_upsample_bwd(const float* __restrict__ dy, int lddy, int dyoff, int c, float* __restrict__ dx, long long n, int D, int H,
               int W, int overwrite) {
    for (IX q = blockIdx.x * (IX)256 + threadIdx.x; q < (IX)n; q += (IX)gridDim.x * 256) {
        int ch;
        IX cv, fv;
        coarse_item<V, IX>(q, c, D, H, W, ch, cv, fv);
        float s[V], f[V];
#pragma unroll
        for (int k = 0; k < V; ++k) s[k] = 0.f;
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            load_f<V>(dy + ((long long)fv + child(o, H, W)) * lddy + dyoff + ch, f);
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] += f[k];
        }
        if (!overwrite) {
            load_f<V>(dx + (long long)cv * c + ch, f);
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] += f[k];
        }
        store_f<V>(dx + (long long)cv * c + ch, s);
    }
}

// 1x1x1 head: logit[v] = sum_c x[v][c] w[c] + b; loss = mean of BCE(sigmoid(logit), target);
// dlogit = (sigmoid - target) / nvox written for the backward pass.  NV: 16-byte vectors per voxel (0: any
// channel count, one by one).
// The cross-entropy is taken in binary64 from u = log(1 + exp(-|s|)): log p = -(u + max(-s, 0)),
// log(1 - p) = -(u + max(s, 0)), each clamped to the logarithms of [1e-7, 1 - 1e-7] (the clamp of the
// probability itself, since log is monotone).  One binary64 exp and one log1p per voxel: the binary64 pipe
// bounds this kernel with a target.
constexpr double LOG_LO = -16.11809565095832;     // log(1e-7)
constexpr double LOG_HI = -1.0000000494736474e-07;  // log(1 - 1e-7)

// LOSS = false: no target (inference), without the registers of the binary64 part (1 channel on 128^3 voxels 10.3 -> 7.9 us).
template <int NV, bool LOSS>
__global__ void __launch_bounds__(256)
k_head_fwd_loss(const __nv_bfloat16* __restrict__ x, int c, const float* __restrict__ w, const float* __restrict__ bp,
                const float* __restrict__ target, long long nvox, float* __restrict__ prob, float* __restrict__ dlogit,
                double* loss) {
    double l = 0.0;
    const float b = bp[0];
    for (long long v = blockIdx.x * 256LL + threadIdx.x; v < nvox; v += (long long)gridDim.x * 256) {
        float s = b;
        if constexpr (NV > 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                float f[8];
                load_bf<8>(x + v * (8 * NV) + 8 * k, f);
#pragma unroll
                for (int q = 0; q < 8; ++q) s += f[q] * w[8 * k + q];
            }
        } else {
            for (int ch = 0; ch < c; ++ch) s += __bfloat162float(x[v * c + ch]) * w[ch];
        }
        const float p = 1.f / (1.f + expf(-s));
        if (prob) prob[v] = p;
        if constexpr (LOSS) {
            const float tf = target[v];
            const double t = tf, sd = s;
            const double u = log1p(exp(-fabs(sd)));
            const double lp = fmin(fmax(-(u + fmax(-sd, 0.0)), LOG_LO), LOG_HI);
            const double lq = fmin(fmax(-(u + fmax(sd, 0.0)), LOG_LO), LOG_HI);
            l -= t * lp + (1.0 - t) * lq;
            if (dlogit) dlogit[v] = (p - tf) / (float)nvox;
        }
    }
    if (LOSS && loss) {
        __shared__ double sh[256];
        sh[threadIdx.x] = l;
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) atomicAdd(loss, sh[0] / (double)nvox);
    }
}

// head backward: dx[v][c] = dlogit[v] w[c]; dw[c] += sum_v dlogit[v] x[v][c]; db += sum_v dlogit[v].
// NV as above.  The sums go through warp shuffles and shared memory to one atomic per channel and block
// (with one per channel and thread the atomics on c + 1 addresses took nearly all of its time: 2.75 ms for
// 4 x 64^3 voxels of 16 channels).  The terms (sigmoid - target) / nvox largely cancel, so the warps' sums
// are added in binary64; with `acc64` ([c] and one for the bias, zeroed) the blocks' are too.
template <int NV>
__global__ void __launch_bounds__(256)
k_head_bwd(const __nv_bfloat16* __restrict__ x, int c, const float* __restrict__ w, const float* __restrict__ dlogit,
           long long nvox, float* __restrict__ dx, float* dw, float* db, double* acc64) {
    constexpr int CM = NV > 0 ? 8 * NV : 32;
    float acc[CM + 1];
#pragma unroll
    for (int ch = 0; ch <= CM; ++ch) acc[ch] = 0.f;
    for (long long v = blockIdx.x * 256LL + threadIdx.x; v < nvox; v += (long long)gridDim.x * 256) {
        const float gl = dlogit[v];
        acc[CM] += gl;
        if constexpr (NV > 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                float f[8], o[8];
                load_bf<8>(x + v * CM + 8 * k, f);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    o[q] = gl * w[8 * k + q];
                    acc[8 * k + q] += gl * f[q];
                }
                store_f<8>(dx + v * CM + 8 * k, o);
            }
        } else {
#pragma unroll
            for (int ch = 0; ch < CM; ++ch)
                if (ch < c) {
                    dx[v * c + ch] = gl * w[ch];
                    acc[ch] += gl * __bfloat162float(x[v * c + ch]);
                }
        }
    }
    __shared__ float sh[CM + 1][8];
#pragma unroll
    for (int ch = 0; ch <= CM; ++ch) {
        for (int o = 16; o > 0; o >>= 1) acc[ch] += __shfl_xor_sync(0xffffffffu, acc[ch], o);
        if ((threadIdx.x & 31) == 0) sh[ch][threadIdx.x >> 5] = acc[ch];
    }
    __syncthreads();
    if (threadIdx.x <= CM) {
        const int ch = threadIdx.x;
        double t = 0.0;
        for (int q = 0; q < 8; ++q) t += sh[ch][q];
        if (ch < CM && NV == 0 && ch >= c) return;
        if (acc64) atomicAdd(acc64 + (ch == CM ? c : ch), t);
        else atomicAdd(ch == CM ? db : dw + ch, (float)t);
    }
}

__global__ void k_head_sums(const double* __restrict__ acc64, int c, float* dw, float* db) {
    const int ch = threadIdx.x;
    if (ch < c) dw[ch] += (float)acc64[ch];
    else if (ch == c) db[0] += (float)acc64[ch];
}

// Adam with bias correction on FP32 master weights; writes the bf16 working copy.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ gr, float* __restrict__ m, float* __restrict__ v,
                       __nv_bfloat16* __restrict__ pb, long long n, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const float gq = gr[q];
        const float mq = b1 * m[q] + (1.f - b1) * gq;
        const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        const float pq = p[q] - lr * (mq * c1) / (sqrtf(vq * c2) + eps);
        p[q] = pq;
        if (pb) pb[q] = __float2bfloat16_rn(pq);
    }
}

// network input: channel 0 = glass field G, 1..nfeat = per-sample features, the rest 0 (16 channels, two
// 16-byte vectors per voxel when the output is aligned)
template <int V, typename IX>
__global__ void __launch_bounds__(256)
k_pack_input(const float* __restrict__ G, const float* __restrict__ feat, int nfeat, long long vps, long long nvox,
             __nv_bfloat16* __restrict__ out) {
    for (IX v = blockIdx.x * (IX)256 + threadIdx.x; v < (IX)nvox; v += (IX)gridDim.x * 256) {
        const long long smp = v / (IX)vps;
        float f[16];
        f[0] = G[v];
#pragma unroll
        for (int k = 0; k < 15; ++k) f[1 + k] = k < nfeat ? __ldg(feat + smp * nfeat + k) : 0.f;
#pragma unroll
        for (int k = 0; k < 16 / V; ++k) {
            float o[V];
#pragma unroll
            for (int q = 0; q < V; ++q) o[q] = f[V * k + q];
            store_bf<V>(out + (long long)v * 16 + V * k, o);
        }
    }
}

int grid_for(long long n) {
    long long b = (n + 255) / 256;
    if (b > 152LL * 32) b = 152LL * 32;
    return (int)(b < 1 ? 1 : b);
}

// 16-byte vectors of `v` elements: every count a multiple of v, every (non-null) pointer on 16 bytes
bool vec_ok(int v, std::initializer_list<int> counts, std::initializer_list<const void*> ptrs) {
    for (int a : counts)
        if (a % v) return false;
    for (const void* q : ptrs)
        if (reinterpret_cast<uintptr_t>(q) % 16) return false;
    return true;
}
bool narrow(long long n) { return n < (1LL << 31) - 152LL * 32 * 256; }  // the grid stride stays below 2^32

}  // namespace

using bf16 = __nv_bfloat16;

extern "C" {


// vector width VV (16-byte vectors) or 1, and the index type (items and fine voxels VOX), chosen at run time
#define LAUNCH_VI(VEC, VV, N, VOX, KERNEL, ...)                                                         \
    do {                                                                                                \
        const long long items_ = (N) / ((VEC) ? (VV) : 1);                                              \
        const int grid_ = grid_for(items_);                                                             \
        const bool n32_ = narrow(items_) && narrow(VOX);                                                \
        if (VEC) {                                                                                      \
            if (n32_) KERNEL<VV, unsigned><<<grid_, 256, 0, (cudaStream_t)stream>>>(__VA_ARGS__);       \
            else KERNEL<VV, unsigned long long><<<grid_, 256, 0, (cudaStream_t)stream>>>(__VA_ARGS__);  \
        } else {                                                                                        \
            if (n32_) KERNEL<1, unsigned><<<grid_, 256, 0, (cudaStream_t)stream>>>(__VA_ARGS__);        \
            else KERNEL<1, unsigned long long><<<grid_, 256, 0, (cudaStream_t)stream>>>(__VA_ARGS__);   \
        }                                                                                               \
        pfgb::count_launch();                                                                           \
    } while (0)

pf_status pfnn_bias_grad(const float* dz, int ld, int off, int c, long long nvox, float* db, void* stream) {
    if (!dz || !db || c < 1) return PF_E_INVALID;
    if (vec_ok(4, {ld, off, c}, {dz}) && c <= 1024 && 256 % (c / 4) == 0) {
        const int per = 256 / (c / 4);
        long long b = (nvox + 4LL * per - 1) / (4LL * per);
        if (b > 152 * 8) b = 152 * 8;
        k_bias_grad<4><<<(unsigned)(b < 1 ? 1 : b), 256, 0, (cudaStream_t)stream>>>(dz, ld, off, c, nvox, db);
    } else {
        k_bias_grad_any<<<dim3(152 * 4, (c + 31) / 32), 256, 0, (cudaStream_t)stream>>>(dz, ld, off, c, nvox, db);
    }
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_relu_bwd_cast(const float* dy, int lddy, int dyoff, const void* y, int ldy, int yoff, int c,
                             long long nvox, float* dz_f32, void* dz_bf16, void* stream) {
    if (!dy || !dz_bf16 || c < 1) return PF_E_INVALID;
    const bool vec = vec_ok(8, {lddy, dyoff, c}, {dy, dz_f32, dz_bf16}) && (!y || vec_ok(8, {ldy, yoff}, {y}));
    const long long n = nvox * c / (vec ? 8 : 1);
    LAUNCH_VI(vec, 8, nvox * c, nvox, k_relu_bwd_cast, dy, lddy, dyoff, (const bf16*)y, ldy, yoff, c, n, dz_f32, (bf16*)dz_bf16);
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_weight_transpose(const void* w, void* wt, int cout, int cin, void* stream) {
    if (!w || !wt) return PF_E_INVALID;
    k_wtranspose<<<grid_for(27LL * cout * cin), 256, 0, (cudaStream_t)stream>>>((const bf16*)w, (bf16*)wt, cout, cin);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_avgpool(const void* x, int ldx, int xoff, void* y, int ldy, int yoff, int c, int n, int d, int h, int wd,
                       void* stream) {
    if (!x || !y || d % 2 || h % 2 || wd % 2) return PF_E_INVALID;
    const bool vec = vec_ok(8, {ldx, xoff, ldy, yoff, c}, {x, y});
    const long long items = (long long)n * d * h * wd / 8 * c;
    LAUNCH_VI(vec, 8, items, (long long)n * d * h * wd, k_avgpool, (const bf16*)x, ldx, xoff, (bf16*)y, ldy, yoff, c, items / (vec ? 8 : 1), d, h, wd);
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_avgpool_bwd(const float* dy, int c, float* dx, int lddx, int dxoff, int n, int d, int h, int wd,
                           void* stream) {
    if (!dy || !dx || d % 2 || h % 2 || wd % 2) return PF_E_INVALID;
    const bool vec = vec_ok(4, {c, lddx, dxoff}, {dy, dx});
    const long long items = (long long)n * d * h * wd / 8 * c;
    LAUNCH_VI(vec, 4, items, (long long)n * d * h * wd, k_avgpool_bwd, dy, c, dx, lddx, dxoff, items / (vec ? 4 : 1), d, h, wd);
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_upsample(const void* x, int c, void* y, int ldy, int yoff, int n, int d, int h, int wd, void* stream) {
    if (!x || !y || d % 2 || h % 2 || wd % 2) return PF_E_INVALID;
    const bool vec = vec_ok(8, {c, ldy, yoff}, {x, y});
    const long long items = (long long)n * d * h * wd / 8 * c;
    LAUNCH_VI(vec, 8, items, (long long)n * d * h * wd, k_upsample, (const bf16*)x, c, (bf16*)y, ldy, yoff, items / (vec ? 8 : 1), d, h, wd);
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

static pf_status upsample_bwd(const float* dy, int lddy, int dyoff, int c, float* dx, int n, int d, int h, int wd,
                              int overwrite, void* stream) {
    if (!dy || !dx) return PF_E_INVALID;
    const bool vec = vec_ok(4, {lddy, dyoff, c}, {dy, dx});
    const long long items = (long long)n * d * h * wd * c;
    LAUNCH_VI(vec, 4, items, 8LL * n * d * h * wd, k_upsample_bwd, dy, lddy, dyoff, c, dx, items / (vec ? 4 : 1), 2 * d, 2 * h,
              2 * wd, overwrite);
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_upsample_bwd(const float* dy, int lddy, int dyoff, int c, float* dx, int n, int d, int h, int wd,
                            void* stream) {
    return upsample_bwd(dy, lddy, dyoff, c, dx, n, d, h, wd, 0, stream);
}

pf_status pfnn_head_forward(const void* x, int c, const float* w, const float* b, const float* target, long long nvox,
                            float* prob, float* dlogit, double* loss, void* stream) {
    if (!x || !w || !b || c < 1 || c > 32) return PF_E_INVALID;
    const int nv = vec_ok(8, {c}, {x}) ? c / 8 : 0;
    auto pick = [&](auto l) {
        constexpr bool L = decltype(l)::value;
        return nv == 0 ? k_head_fwd_loss<0, L> : nv == 1 ? k_head_fwd_loss<1, L> : nv == 2 ? k_head_fwd_loss<2, L>
               : nv == 3 ? k_head_fwd_loss<3, L> : k_head_fwd_loss<4, L>;
    };
    auto k = target ? pick(std::true_type{}) : pick(std::false_type{});
    k<<<grid_for(nvox), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, c, w, b, target, nvox, prob, dlogit, loss);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

static pf_status head_backward(const void* x, int c, const float* w, const float* dlogit, long long nvox, float* dx,
                               float* dw, float* db, double* acc64, void* stream) {
    if (!x || !w || !dlogit || !dx || !dw || !db || c < 1 || c > 32) return PF_E_INVALID;
    auto k = !vec_ok(8, {c}, {x, dx}) ? k_head_bwd<0> : c == 8 ? k_head_bwd<1> : c == 16 ? k_head_bwd<2>
             : c == 24 ? k_head_bwd<3> : k_head_bwd<4>;
    long long blocks = (nvox + 511) / 512;  // two voxels per thread at least, four blocks per SM at most
    if (blocks > 152 * 4) blocks = 152 * 4;
    k<<<(unsigned)(blocks < 1 ? 1 : blocks), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, c, w, dlogit, nvox, dx, dw, db,
                                                                            acc64);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_head_backward(const void* x, int c, const float* w, const float* dlogit, long long nvox, float* dx,
                             float* dw, float* db, void* stream) {
    return head_backward(x, c, w, dlogit, nvox, dx, dw, db, nullptr, stream);
}

pf_status pfnn_pack_input(const float* G, const float* feat, int nfeat, long long vox_per_sample, long long nvox,
                          void* out, void* stream) {
    if (!G || !out || nfeat < 0 || nfeat > 15 || (nfeat && !feat) || vox_per_sample < 1) return PF_E_INVALID;
    const bool vec = vec_ok(8, {}, {out});
    const int grid = grid_for(nvox);
    cudaStream_t s = (cudaStream_t)stream;
    const bool small = narrow(nvox) && vox_per_sample < (1LL << 31);
    auto k = vec ? (small ? k_pack_input<8, unsigned> : k_pack_input<8, unsigned long long>)
                 : (small ? k_pack_input<1, unsigned> : k_pack_input<1, unsigned long long>);
    k<<<grid, 256, 0, s>>>(G, feat, nfeat, vox_per_sample, nvox, (bf16*)out);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status pfnn_adam(float* p, const float* g, float* m, float* v, void* p_bf16, long long n, float lr, float b1,
                    float b2, float eps, int step, void* stream) {
    if (!p || !g || !m || !v || step < 1) return PF_E_INVALID;
    const float c1 = 1.f / (1.f - powf(b1, (float)step));
    const float c2 = 1.f / (1.f - powf(b2, (float)step));
    k_adam<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(p, g, m, v, (bf16*)p_bf16, n, lr, b1, b2, eps, c1, c2);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

}  // extern "C"

namespace pfgb {

pf_status nn_upsample_bwd_set(const float* dy, int lddy, int dyoff, int c, float* dx, int n, int d, int h, int wd,
                              void* stream) {
    return upsample_bwd(dy, lddy, dyoff, c, dx, n, d, h, wd, 1, stream);
}

pf_status nn_head_backward64(const void* x, int c, const float* w, const float* dlogit, long long nvox, float* dx,
                             float* dw, float* db, double* acc64, void* stream) {
    if (cudaMemsetAsync(acc64, 0, sizeof(double) * (c + 1), (cudaStream_t)stream) != cudaSuccess) return PF_E_CUDA;
    pf_status s = head_backward(x, c, w, dlogit, nvox, dx, dw, db, acc64, stream);
    if (s != PF_OK) return s;
    k_head_sums<<<1, 64, 0, (cudaStream_t)stream>>>(acc64, c, dw, db);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

pf_status nn_relu_bwd_bias(const float* dy, int lddy, int dyoff, const void* y, int ldy, int yoff, int c, long long nvox,
                           void* dz_bf16, float* db, void* stream) {
    if (!dy || !y || !dz_bf16 || !db || !vec_ok(8, {lddy, dyoff, ldy, yoff, c}, {dy, y, dz_bf16}) || c > 2048 ||
        256 % (c / 8))
        return PF_E_INVALID;
    // about four voxels per thread, at most eight blocks per SM
    const long long per = 4LL * 256 / (c / 8);
    long long b = (nvox + per - 1) / per;
    if (b > 152 * 8) b = 152 * 8;
    k_relu_bwd_bias<<<(unsigned)(b < 1 ? 1 : b), 256, 0, (cudaStream_t)stream>>>(dy, lddy, dyoff, (const bf16*)y, ldy, yoff,
                                                                                c, nvox, (bf16*)dz_bf16, db);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

}  // namespace pfgb
