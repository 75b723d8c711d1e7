// Network-level C ABI of the learned warm start: the 3D convolutional encoder-decoder (4 levels,
// 16/32/64/128 channels) assembled from the layer kernels of include/pfnn.h, with its parameters, FP32
// master weights, BF16 working copies, gradients, Adam moments and activation buffers owned by the
// library.  Forward, backward and the optimiser step are sequences of the library's own kernels on the
// network's stream; nothing runs on the host but the sequencing.
//
// Architecture (two 3x3x3 convolutions + ReLU per level, 2x2x2 average-pool down, x2 nearest up + 3x3x3
// convolution, skip concatenation through channel slices of shared buffers, 1x1x1 sigmoid head):
//   in(16) -> e1a(16) -> e1b(16)=cat1[0:16] -> pool -> e2a(32) -> e2b(32)=cat2[0:32] -> pool
//          -> e3a(64) -> e3b(64)=cat3[0:64] -> pool -> e4a(128) -> e4b(128)
//          -> up -> u3(64)=cat3[64:128] -> d3a(64) -> d3b(64) -> up -> u2(32)=cat2[32:64] -> d2a(32) -> d2b(32)
//          -> up -> u1(16)=cat1[16:32] -> d1a(16) -> d1b(16) -> head(1) -> sigmoid
#include "../../include/pfnn.h"
#include "pf_internal.cuh"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

namespace pfgb {
// pfnn_conv.cu: dx = (not +=) the sum of the eight children; ReLU backward to bf16 with db[c] += its sums
pf_status nn_upsample_bwd_set(const float* dy, int lddy, int dyoff, int c, float* dx, int n, int d, int h, int wd,
                              void* stream);
pf_status nn_relu_bwd_bias(const float* dy, int lddy, int dyoff, const void* y, int ldy, int yoff, int c, long long nvox,
                           void* dz_bf16, float* db, void* stream);
// pfnn_head_backward with the sums over blocks in binary64 (acc64: scratch of c + 1 values)
pf_status nn_head_backward64(const void* x, int c, const float* w, const float* dlogit, long long nvox, float* dx,
                             float* dw, float* db, double* acc64, void* stream);
// pfnn_umma.cu: pfnn_conv3d_wgrad of a compact dy and 16-byte aligned rows of x (no scratch needed)
pf_status nn_wgrad(const void* dy, int cout, const void* x, int ldx, int xoff, int cin, float* dw, int n, int d, int h,
                   int wd, void* stream);
}  // namespace pfgb

namespace {

enum Buf { IN0, E1A, CAT1, P1, E2A, CAT2, P2, E3A, CAT3, P3, E4A, E4B, UP3, D3A, D3B, UP2, D2A, D2B, UP1, D1A, D1B, NBUF };
// channels and level (side S >> level) of each buffer
const int kBufC[NBUF] = {16, 16, 32, 16, 32, 64, 32, 64, 128, 64, 128, 128, 128, 64, 64, 64, 32, 32, 32, 16, 16};
const int kBufL[NBUF] = {0, 0, 0, 1, 1, 1, 2, 2, 2, 3, 3, 3, 2, 2, 2, 1, 1, 1, 0, 0, 0};

// what happens before a convolution: 0 none, 1 pool (src buffer, level, channels, dst buffer), 2 upsample
struct Layer {
    const char* name;
    int src, soff, cin, dst, doff, cout, lev;
    int pre;          // 0 none, 1 pool, 2 upsample
    int pre_src, pre_c, pre_dst, pre_lev;
};
const Layer kLayers[] = {
    {"e1a", IN0, 0, 16, E1A, 0, 16, 0, 0, 0, 0, 0, 0},
    {"e1b", E1A, 0, 16, CAT1, 0, 16, 0, 0, 0, 0, 0, 0},
    {"e2a", P1, 0, 16, E2A, 0, 32, 1, 1, CAT1, 16, P1, 0},
    {"e2b", E2A, 0, 32, CAT2, 0, 32, 1, 0, 0, 0, 0, 0},
    {"e3a", P2, 0, 32, E3A, 0, 64, 2, 1, CAT2, 32, P2, 1},
    {"e3b", E3A, 0, 64, CAT3, 0, 64, 2, 0, 0, 0, 0, 0},
    {"e4a", P3, 0, 64, E4A, 0, 128, 3, 1, CAT3, 64, P3, 2},
    {"e4b", E4A, 0, 128, E4B, 0, 128, 3, 0, 0, 0, 0, 0},
    {"u3", UP3, 0, 128, CAT3, 64, 64, 2, 2, E4B, 128, UP3, 2},
    {"d3a", CAT3, 0, 128, D3A, 0, 64, 2, 0, 0, 0, 0, 0},
    {"d3b", D3A, 0, 64, D3B, 0, 64, 2, 0, 0, 0, 0, 0},
    {"u2", UP2, 0, 64, CAT2, 32, 32, 1, 2, D3B, 64, UP2, 1},
    {"d2a", CAT2, 0, 64, D2A, 0, 32, 1, 0, 0, 0, 0, 0},
    {"d2b", D2A, 0, 32, D2B, 0, 32, 1, 0, 0, 0, 0, 0},
    {"u1", UP1, 0, 32, CAT1, 16, 16, 0, 2, D2B, 32, UP1, 0},
    {"d1a", CAT1, 0, 32, D1A, 0, 16, 0, 0, 0, 0, 0, 0},
    {"d1b", D1A, 0, 16, D1B, 0, 16, 0, 0, 0, 0, 0, 0},
};
constexpr int NCONV = sizeof(kLayers) / sizeof(kLayers[0]);
constexpr int NPARAM = NCONV + 1;   // + the 1x1x1 head (16 weights, 1 bias)
constexpr int NFEAT = 2;            // supercooling and surface-tension features

struct Param {
    long long nw = 0, nb = 0;
    float *w = nullptr, *b = nullptr, *gw = nullptr, *gb = nullptr;
    void* wb = nullptr;   // bf16 working copy [27][cout][cin]
    void* wt = nullptr;   // bf16 transposed copy [27][cin][cout] (backward data)
};

// splitmix64 (Steele, Lea, Flood 2014) and Box-Muller: the He-normal initial weights
uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
double normal(uint64_t& s) {
    const double u1 = ((splitmix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    const double u2 = ((splitmix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
}

// All parameters lie in one arena (and their gradients, moments, bf16 copies in others with the same
// layout): segment 2q the weights, 2q + 1 the biases of parameter q, each starting on a multiple of SEG
// elements, so the optimiser step is one launch (one block per SEG elements; 36 launches of a few blocks
// each took 130 us) and the gradients are zeroed by one memset.
constexpr int SEG = 1024, NSEG = 2 * NPARAM;
struct Segments {
    int block0[NSEG + 1];         // first block of each segment
    int n[NSEG];                  // elements
    int cout[NSEG], cin[NSEG];    // convolution weights [27][cout][cin] (0: no bf16 copies)
};

// segment of this block (uniform)
__device__ __forceinline__ int segment_of(const Segments& S) {
    int s = 0;
    while ((int)blockIdx.x >= S.block0[s + 1]) ++s;
    return s;
}

// the bf16 working copy of one weight and its transposed copy [27][cin][cout] (backward data)
__device__ __forceinline__ void store_copies(const Segments& S, int s, long long base, int e, float p,
                                             __nv_bfloat16* wb, __nv_bfloat16* wt) {
    const __nv_bfloat16 b = __float2bfloat16_rn(p);
    const int ci = e % S.cin[s], r = e / S.cin[s], co = r % S.cout[s], t = r / S.cout[s];
    wb[base + e] = b;
    wt[base + ((long long)t * S.cin[s] + ci) * S.cout[s] + co] = b;
}

// Adam with bias correction on the FP32 master parameters (the arithmetic of pfnn_adam)
__global__ void __launch_bounds__(256)
k_adam_all(const __grid_constant__ Segments S, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
           float* __restrict__ v, __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt, float lr, float b1,
           float b2, float eps, float c1, float c2) {
    const int s = segment_of(S);
    const long long base = (long long)S.block0[s] * SEG;
    const int e0 = ((int)blockIdx.x - S.block0[s]) * SEG;
#pragma unroll
    for (int k = 0; k < SEG / 256; ++k) {
        const int e = e0 + k * 256 + threadIdx.x;
        if (e >= S.n[s]) break;
        const long long q = base + e;
        const float gq = g[q];
        const float mq = b1 * m[q] + (1.f - b1) * gq;
        const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        const float pq = p[q] - lr * (mq * c1) / (sqrtf(vq * c2) + eps);
        p[q] = pq;
        if (S.cin[s]) store_copies(S, s, base, e, pq, wb, wt);
    }
}

// the bf16 copies of every convolution weight (after the parameters were set)
__global__ void __launch_bounds__(256)
k_copies_all(const __grid_constant__ Segments S, const float* __restrict__ p, __nv_bfloat16* __restrict__ wb,
             __nv_bfloat16* __restrict__ wt) {
    const int s = segment_of(S);
    if (!S.cin[s]) return;
    const long long base = (long long)S.block0[s] * SEG;
    const int e0 = ((int)blockIdx.x - S.block0[s]) * SEG;
    for (int e = e0 + threadIdx.x; e < e0 + SEG && e < S.n[s]; e += 256) store_copies(S, s, base, e, p[base + e], wb, wt);
}

}  // namespace

struct pfnn_net {
    Param p[NPARAM];
    Segments seg{};
    float *pw = nullptr, *pg = nullptr, *pm = nullptr, *pv = nullptr;   // arenas: parameters, gradients, moments
    __nv_bfloat16 *pb = nullptr, *pt = nullptr;                         // bf16 copies, plain and transposed
    cudaStream_t stream = nullptr;
    int step = 0;
    int n = 0, S = 0;                      // batch and side of the allocated activation buffers
    void* act[NBUF] = {};                  // bf16 activations
    float* grad[NBUF] = {};                // fp32 gradients of the activations
    float *logit_grad = nullptr, *prob = nullptr;
    void* dz_b = nullptr;
    double* loss = nullptr;                // the loss, then the 17 sums of the head's backward pass
    bool have_target = false;
    std::vector<void*> allocs, act_allocs;
    std::string err;
};

namespace {

pf_status nfail(pfnn_net* net, pf_status s, const std::string& m) {
    if (net) net->err = m;
    return s;
}

void* nalloc(std::vector<void*>& v, size_t bytes) {
    void* q = nullptr;
    if (cudaMalloc(&q, bytes) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    v.push_back(q);
    return q;
}

void free_acts(pfnn_net* net) {
    for (void* q : net->act_allocs) cudaFree(q);
    net->act_allocs.clear();
    for (int b = 0; b < NBUF; ++b) {
        net->act[b] = nullptr;
        net->grad[b] = nullptr;
    }
    net->logit_grad = net->prob = nullptr;
    net->dz_b = nullptr;
    net->n = net->S = 0;
}

pf_status ensure_acts(pfnn_net* net, int n, int S) {
    if (net->n == n && net->S == S) return PF_OK;
    free_acts(net);
    for (int b = 0; b < NBUF; ++b) {
        const long long s = S >> kBufL[b];
        const long long cells = (long long)n * s * s * s * kBufC[b];
        net->act[b] = nalloc(net->act_allocs, 2 * cells);
        net->grad[b] = (float*)nalloc(net->act_allocs, 4 * cells);
        if (!net->act[b] || !net->grad[b]) return nfail(net, PF_E_OOM, "activation buffers");
        if (cudaMemsetAsync(net->act[b], 0, 2 * cells, net->stream) != cudaSuccess)
            return nfail(net, PF_E_CUDA, "activation buffers");
    }
    // the input's gradient is never formed: it reads as zero
    if (cudaMemsetAsync(net->grad[IN0], 0, 4LL * n * S * S * S * kBufC[IN0], net->stream) != cudaSuccess)
        return nfail(net, PF_E_CUDA, "gradient buffers");
    const long long nvox = (long long)n * S * S * S;
    long long dz = 0;  // largest layer output
    for (int q = 0; q < NCONV; ++q) {
        const long long sd = S >> kLayers[q].lev, b = n * sd * sd * sd * kLayers[q].cout;
        dz = b > dz ? b : dz;
    }
    net->dz_b = nalloc(net->act_allocs, 2 * dz);
    net->logit_grad = (float*)nalloc(net->act_allocs, 4 * nvox);
    net->prob = (float*)nalloc(net->act_allocs, 4 * nvox);
    if (!net->dz_b || !net->logit_grad || !net->prob)
        return nfail(net, PF_E_OOM, "work buffers");
    net->n = n;
    net->S = S;
    return PF_OK;
}

#define NN_CK(net, call, what)                                                 \
    do {                                                                       \
        pf_status s_ = (call);                                                 \
        if (s_ != PF_OK) return nfail((net), s_, std::string(what) + " failed"); \
    } while (0)

}  // namespace

extern "C" {

int pfnn_net_params(void) { return NPARAM; }

pf_status pfnn_net_param_shape(int q, int* cin, int* cout) {
    if (q < 0 || q >= NPARAM) return PF_E_INVALID;
    if (cin) *cin = q < NCONV ? kLayers[q].cin : 16;
    if (cout) *cout = q < NCONV ? kLayers[q].cout : 1;
    return PF_OK;
}

const char* pfnn_net_param_name(int q) { return q >= 0 && q < NCONV ? kLayers[q].name : (q == NCONV ? "head" : ""); }

const char* pfnn_net_last_error(const pfnn_net* net) { return net ? net->err.c_str() : ""; }

int pfnn_net_buffers(void) { return NBUF; }

// layer q's wiring: input buffer and channel offset, cin, output buffer and offset, cout, level, and what
// runs before it (0 none, 1 pool of pre_c channels of buffer pre_src into pre_dst, 2 upsample)
pf_status pfnn_net_layer(int q, int* wiring) {
    if (q < 0 || q >= NCONV || !wiring) return PF_E_INVALID;
    const Layer& L = kLayers[q];
    const int v[12] = {L.src, L.soff, L.cin, L.dst, L.doff, L.cout, L.lev, L.pre, L.pre_src, L.pre_c, L.pre_dst, L.pre_lev};
    for (int k = 0; k < 12; ++k) wiring[k] = v[k];
    return PF_OK;
}

// buffer b: channels per voxel and level (side >> level)
pf_status pfnn_net_buffer(int b, int* channels, int* level) {
    if (b < 0 || b >= NBUF) return PF_E_INVALID;
    if (channels) *channels = kBufC[b];
    if (level) *level = kBufL[b];
    return PF_OK;
}

// copy buffer b of the last forward / backward to host arrays (bf16 activations, fp32 gradients; either
// may be NULL) of n (side >> level)^3 channels values; synchronous
pf_status pfnn_net_read_buffer(pfnn_net* net, int b, void* act, float* grad) {
    if (!net || b < 0 || b >= NBUF) return PF_E_INVALID;
    if (!net->S) return nfail(net, PF_E_STATE, "no forward yet");
    const long long s = net->S >> kBufL[b];
    const long long cells = (long long)net->n * s * s * s * kBufC[b];
    if ((act && cudaMemcpyAsync(act, net->act[b], 2 * cells, cudaMemcpyDeviceToHost, net->stream) != cudaSuccess) ||
        (grad && cudaMemcpyAsync(grad, net->grad[b], 4 * cells, cudaMemcpyDeviceToHost, net->stream) != cudaSuccess) ||
        cudaStreamSynchronize(net->stream) != cudaSuccess)
        return nfail(net, PF_E_CUDA, "read_buffer");
    return PF_OK;
}

pf_status pfnn_net_destroy(pfnn_net* net) {
    if (!net) return PF_OK;
    if (net->stream) cudaStreamSynchronize(net->stream);
    free_acts(net);
    for (void* q : net->allocs) cudaFree(q);
    delete net;
    return PF_OK;
}

pf_status pfnn_net_create(unsigned long long seed, void* stream, pfnn_net** out) {
    if (!out) return PF_E_INVALID;
    *out = nullptr;
    pfnn_net* net = new pfnn_net();
    net->stream = (cudaStream_t)stream;
    uint64_t rs = seed;
    Segments& G = net->seg;
    for (int q = 0; q < NPARAM; ++q) {
        Param& P = net->p[q];
        const int cin = q < NCONV ? kLayers[q].cin : 16, cout = q < NCONV ? kLayers[q].cout : 1;
        P.nw = q < NCONV ? 27LL * cout * cin : 16;
        P.nb = cout;
        G.n[2 * q] = (int)P.nw;
        G.n[2 * q + 1] = (int)P.nb;
        G.cin[2 * q] = q < NCONV ? cin : 0;
        G.cout[2 * q] = q < NCONV ? cout : 0;
    }
    for (int k = 0; k < NSEG; ++k) G.block0[k + 1] = G.block0[k] + (G.n[k] + SEG - 1) / SEG;
    const size_t total = (size_t)G.block0[NSEG] * SEG;
    for (float** f : {&net->pw, &net->pg, &net->pm, &net->pv}) *f = (float*)nalloc(net->allocs, 4 * total);
    for (__nv_bfloat16** f : {&net->pb, &net->pt}) *f = (__nv_bfloat16*)nalloc(net->allocs, 2 * total);
    if (!net->pw || !net->pg || !net->pm || !net->pv || !net->pb || !net->pt) {
        pfnn_net_destroy(net);
        return PF_E_OOM;
    }
    // He-normal weights for the ReLU layers (std sqrt(2 / fan_in)), sqrt(1/16) for the head; zero biases
    std::vector<float> w(total, 0.f);
    for (int q = 0; q < NPARAM; ++q) {
        Param& P = net->p[q];
        const size_t ow = (size_t)G.block0[2 * q] * SEG, ob = (size_t)G.block0[2 * q + 1] * SEG;
        P.w = net->pw + ow; P.gw = net->pg + ow;
        P.b = net->pw + ob; P.gb = net->pg + ob;
        if (q < NCONV) { P.wb = net->pb + ow; P.wt = net->pt + ow; }
        const double sd = q < NCONV ? std::sqrt(2.0 / (27.0 * kLayers[q].cin)) : std::sqrt(1.0 / 16.0);
        for (long long k = 0; k < P.nw; ++k) w[ow + k] = (float)(normal(rs) * sd);
    }
    cudaError_t e = cudaMemcpy(net->pw, w.data(), 4 * total, cudaMemcpyHostToDevice);
    for (float* f : {net->pg, net->pm, net->pv})
        if (e == cudaSuccess) e = cudaMemset(f, 0, 4 * total);
    if (e == cudaSuccess) {
        k_copies_all<<<G.block0[NSEG], 256>>>(G, net->pw, net->pb, net->pt);
        pfgb::count_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        pfnn_net_destroy(net);
        return PF_E_CUDA;
    }
    net->loss = (double*)nalloc(net->allocs, 18 * sizeof(double));
    if (!net->loss) {
        pfnn_net_destroy(net);
        return PF_E_OOM;
    }
    *out = net;
    return PF_OK;
}

// parameter q's FP32 master weights and biases from / to host arrays (w: [27][cout][cin], head: [16])
pf_status pfnn_net_set_params(pfnn_net* net, int q, const float* w, const float* b) {
    if (!net || q < 0 || q >= NPARAM || !w || !b) return PF_E_INVALID;
    Param& P = net->p[q];
    if (cudaMemcpyAsync(P.w, w, 4 * P.nw, cudaMemcpyHostToDevice, net->stream) != cudaSuccess ||
        cudaMemcpyAsync(P.b, b, 4 * P.nb, cudaMemcpyHostToDevice, net->stream) != cudaSuccess)
        return nfail(net, PF_E_CUDA, "set_params");
    if (P.wb) {
        k_copies_all<<<net->seg.block0[NSEG], 256, 0, net->stream>>>(net->seg, net->pw, net->pb, net->pt);
        pfgb::count_launch();
    }
    if (cudaStreamSynchronize(net->stream) != cudaSuccess) return nfail(net, PF_E_CUDA, "set_params");
    return PF_OK;
}

pf_status pfnn_net_get_params(pfnn_net* net, int q, float* w, float* b) {
    if (!net || q < 0 || q >= NPARAM) return PF_E_INVALID;
    const Param& P = net->p[q];
    if ((w && cudaMemcpyAsync(w, P.w, 4 * P.nw, cudaMemcpyDeviceToHost, net->stream) != cudaSuccess) ||
        (b && cudaMemcpyAsync(b, P.b, 4 * P.nb, cudaMemcpyDeviceToHost, net->stream) != cudaSuccess) ||
        cudaStreamSynchronize(net->stream) != cudaSuccess)
        return nfail(net, PF_E_CUDA, "get_params");
    return PF_OK;
}

pf_status pfnn_net_get_grads(pfnn_net* net, int q, float* gw, float* gb) {
    if (!net || q < 0 || q >= NPARAM) return PF_E_INVALID;
    const Param& P = net->p[q];
    if ((gw && cudaMemcpyAsync(gw, P.gw, 4 * P.nw, cudaMemcpyDeviceToHost, net->stream) != cudaSuccess) ||
        (gb && cudaMemcpyAsync(gb, P.gb, 4 * P.nb, cudaMemcpyDeviceToHost, net->stream) != cudaSuccess) ||
        cudaStreamSynchronize(net->stream) != cudaSuccess)
        return nfail(net, PF_E_CUDA, "get_grads");
    return PF_OK;
}

pf_status pfnn_net_forward(pfnn_net* net, const float* G, const float* feat, int n, int side, const float* target,
                           float* prob) {
    if (!net || !G || !feat || n < 1 || side < 8 || side % 8) return PF_E_INVALID;
    pf_status st = ensure_acts(net, n, side);
    if (st != PF_OK) return st;
    cudaStream_t s = net->stream;
    const long long vps = (long long)side * side * side, nvox = (long long)n * vps;
    auto dims = [&](int lev, int* d) { const int sd = side >> lev; d[0] = n; d[1] = d[2] = d[3] = sd; };
    NN_CK(net, pfnn_pack_input(G, feat, NFEAT, vps, nvox, net->act[IN0], s), "pack");
    for (int q = 0; q < NCONV; ++q) {
        const Layer& L = kLayers[q];
        int d[4];
        if (L.pre == 1) {
            dims(L.pre_lev, d);
            NN_CK(net, pfnn_avgpool(net->act[L.pre_src], kBufC[L.pre_src], 0, net->act[L.pre_dst], kBufC[L.pre_dst], 0,
                                    L.pre_c, d[0], d[1], d[2], d[3], s), "pool");
        } else if (L.pre == 2) {
            dims(L.pre_lev, d);
            NN_CK(net, pfnn_upsample(net->act[L.pre_src], L.pre_c, net->act[L.pre_dst], kBufC[L.pre_dst], 0, d[0], d[1],
                                     d[2], d[3], s), "upsample");
        }
        dims(L.lev, d);
        const Param& P = net->p[q];
        NN_CK(net, pfnn_conv3d(net->act[L.src], kBufC[L.src], L.soff, P.wb, L.cin, L.cout, P.b, 1, 0, net->act[L.dst],
                               nullptr, kBufC[L.dst], L.doff, 0, d[0], d[1], d[2], d[3], s), L.name);
    }
    if (cudaMemsetAsync(net->loss, 0, sizeof(double), s) != cudaSuccess) return nfail(net, PF_E_CUDA, "loss");
    const Param& H = net->p[NCONV];
    net->have_target = target != nullptr;
    NN_CK(net, pfnn_head_forward(net->act[D1B], 16, H.w, H.b, target, nvox, prob ? prob : net->prob,
                                 target ? net->logit_grad : nullptr, target ? net->loss : nullptr, s), "head");
    return PF_OK;
}

pf_status pfnn_net_infer(pfnn_net* net, const float* G, const float* feat, int n, int side, float* prob) {
    if (!prob) return PF_E_INVALID;
    return pfnn_net_forward(net, G, feat, n, side, nullptr, prob);
}

pf_status pfnn_net_loss(pfnn_net* net, double* loss) {
    if (!net || !loss) return PF_E_INVALID;
    if (cudaMemcpyAsync(loss, net->loss, sizeof(double), cudaMemcpyDeviceToHost, net->stream) != cudaSuccess ||
        cudaStreamSynchronize(net->stream) != cudaSuccess)
        return nfail(net, PF_E_CUDA, "loss");
    return PF_OK;
}

pf_status pfnn_net_backward(pfnn_net* net) {
    if (!net) return PF_E_INVALID;
    if (!net->have_target || !net->S) return nfail(net, PF_E_STATE, "backward needs a forward with a target");
    cudaStream_t s = net->stream;
    const int n = net->n, side = net->S;
    auto dims = [&](int lev, int* d) { const int sd = side >> lev; d[0] = n; d[1] = d[2] = d[3] = sd; };
    if (cudaMemsetAsync(net->pg, 0, 4 * (size_t)net->seg.block0[NSEG] * SEG, s) != cudaSuccess)
        return nfail(net, PF_E_CUDA, "zero gradients");
    // Every activation gradient is first written whole (the head's adjoint, a data gradient over all channels
    // of the buffer, or an upsampling's adjoint) and only then added to (a pooling's adjoint into the encoder
    // half of a skip buffer, whose decoder layer comes later in the forward order), so none is zeroed.
    const long long nvox0 = (long long)n * side * side * side;
    const Param& H = net->p[NCONV];
    NN_CK(net, pfgb::nn_head_backward64(net->act[D1B], 16, H.w, net->logit_grad, nvox0, net->grad[D1B], H.gw, H.gb,
                                        net->loss + 1, s), "head backward");
    for (int q = NCONV - 1; q >= 0; --q) {
        const Layer& L = kLayers[q];
        Param& P = net->p[q];
        int d[4];
        dims(L.lev, d);
        const long long nvox = (long long)d[0] * d[1] * d[2] * d[3];
        const int ldy = kBufC[L.dst];
        // ReLU backward on this layer's output slice, then the three products of the convolution
        NN_CK(net, pfgb::nn_relu_bwd_bias(net->grad[L.dst], ldy, L.doff, net->act[L.dst], ldy, L.doff, L.cout, nvox,
                                          net->dz_b, P.gb, s), "relu backward");
        NN_CK(net, pfgb::nn_wgrad(net->dz_b, L.cout, net->act[L.src], kBufC[L.src], L.soff, L.cin, P.gw, d[0], d[1], d[2],
                                  d[3], s), "weight gradient");
        if (L.src != IN0) {
            NN_CK(net, pfnn_conv3d(net->dz_b, L.cout, 0, P.wt, L.cout, L.cin, nullptr, 0, 1, nullptr, net->grad[L.src],
                                   kBufC[L.src], L.soff, 0, d[0], d[1], d[2], d[3], s), "data gradient");
        }
        // adjoint of the data movement that produced this layer's input
        if (L.pre == 1) {
            int e[4];
            dims(L.pre_lev, e);
            NN_CK(net, pfnn_avgpool_bwd(net->grad[L.pre_dst], L.pre_c, net->grad[L.pre_src], kBufC[L.pre_src], 0, e[0],
                                        e[1], e[2], e[3], s), "pool backward");
        } else if (L.pre == 2) {
            int e[4];
            dims(L.pre_lev + 1, e);  // the coarse side
            NN_CK(net, pfgb::nn_upsample_bwd_set(net->grad[L.pre_dst], kBufC[L.pre_dst], 0, L.pre_c,
                                                 net->grad[L.pre_src], e[0], e[1], e[2], e[3], s), "upsample backward");
        }
    }
    return PF_OK;
}

pf_status pfnn_net_adam_step(pfnn_net* net, float lr, float b1, float b2, float eps) {
    if (!net || !(lr > 0.f)) return PF_E_INVALID;
    net->step += 1;
    const float c1 = 1.f / (1.f - powf(b1, (float)net->step));
    const float c2 = 1.f / (1.f - powf(b2, (float)net->step));
    k_adam_all<<<net->seg.block0[NSEG], 256, 0, net->stream>>>(net->seg, net->pw, net->pg, net->pm, net->pv, net->pb,
                                                               net->pt, lr, b1, b2, eps, c1, c2);
    pfgb::count_launch();
    if (cudaGetLastError() != cudaSuccess) return nfail(net, PF_E_CUDA, "adam failed");
    return PF_OK;
}

}  // extern "C"
