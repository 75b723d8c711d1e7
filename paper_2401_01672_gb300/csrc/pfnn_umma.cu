// 3x3x3 convolution (forward and backward-data) of the learned warm start as an implicit GEMM on
// the fifth-generation tensor cores of sm_103a: TMA brings the operand tiles into shared memory,
// tcgen05.mma accumulates in tensor memory (TMEM), tcgen05.ld reads the accumulator back for the
// epilogue.
//
// GEMM view (forward): D[v][co] = sum over taps t and input channels ci of X[v + off(t)][ci] W[t][co][ci]
//   M = 128 voxels of one brick (wb x hb x db cells of one sample), N = cout, K = 27 taps x cin.
// Backward data is the same GEMM on dY with flipped taps and the transposed weights [27][cin][cout].
//
// A operand: one TMA box of the channels-last activation tensor per (tap, channel block): the brick
// shifted by the tap offset, ck channels deep.  Cells outside the grid (the convolution's zero
// padding) are filled with zeros by the TMA unit itself.  The box lands in shared memory as 128 rows
// (voxels, x fastest) of ck bf16 channels, swizzled with the pattern whose span equals the row length
// (32, 64 or 128 bytes), which is the K-major layout the MMA descriptors name.
// B operand: the [cout][ck] weight slice of the same tap and channel block (K-major, same swizzle).
//
// Roles (4 warps): thread 0 issues the TMA loads into a ring of shared-memory stages, thread 32 issues
// the MMAs (one per 16 channels) and commits each stage back to the producer, warp 2 owns the TMEM
// allocation; all four warps then read the 128 x cout fp32 accumulator (warp w owns TMEM lanes
// 32w..32w+31 = voxels 32w..32w+31 of the brick) and apply bias, ReLU and the bf16 or fp32 store.
// Every wait on an mbarrier gives up after a bounded number of tries, records the failure in a device
// flag (read by pfnn_status) and lets the block finish: no wait can hang the GPU.
#include "../../include/pfnn.h"
#include "pf_internal.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

namespace {

using bf16 = __nv_bfloat16;

constexpr int UM = 128;     // MMA M: voxels per tile
constexpr int UTHR = 128;   // threads per block (4 warps)
constexpr long long WAIT_TRIES = 1LL << 24;

// Test-only setting of the failure-path test, consumed by the next pfnn_conv3d call: the producer
// withholds the TMA loads of one stage and every wait gives up after g_test_tries tries.
static int g_test_withhold = -1;
static long long g_test_tries = 0;

__device__ int g_umma_status = 0;  // 0 = ok; 1 = an mbarrier wait gave up

struct UmmaArgs {
    int cin, cout, ck, nkb;       // channels in/out, channels per k block, k blocks per tap
    int wb, hb, db;               // brick (wb * hb * db = 128)
    int D, H, W;                  // grid of one sample
    int tx, ty, tz;               // bricks per sample along x, y, z
    int flip, relu, accumulate;
    int stages;
    int withhold;                 // stage whose loads are withheld (test of the failure path), -1 = none
    long long tries;              // bound of every mbarrier wait
    unsigned a_bytes, stage_bytes;  // shared-memory footprint of the A tile and of one stage (1024-byte units)
    unsigned tx_bytes;              // bytes the two TMA loads of one stage deliver
    unsigned idesc;               // MMA instruction descriptor
    unsigned long long desc_hi;   // constant high bits of the shared-memory descriptors
    int tmem_cols;
    const float* bias;
    bf16* y;
    float* yf;
    int ldy, yoff;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Wait for the phase of the given parity to complete; false (and the device flag set) after WAIT_TRIES.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long tries) {
    for (long long it = 0; it < tries; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    atomicExch(&g_umma_status, 1);
    return false;
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, "
        "%6, %7}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
        "[%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}

// Shared-memory matrix descriptor: start address (bits 0-13, in 16-byte units) over the constant
// part (stride between 8-row groups, descriptor version, swizzle mode).
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, unsigned long long hi) {
    return hi | (uint64_t)((addr >> 4) & 0x3FFFu);
}

__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrive on the mbarrier once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// The .aligned instructions on TMEM need all 32 lanes together: the lanes meet first, whatever the caller did for some of
// them only (cells outside the grid, waits that ended after different numbers of tries).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

// sixteen output channels of one cell at element offset `at`: bf16, or fp32 (added to what is there when accumulating)
__device__ __forceinline__ void store_cell16(bf16* y, float* yf, long long at, int accumulate, const float (&o)[16]) {
    if (yf) {
        float4* dst = reinterpret_cast<float4*>(yf + at);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float4 w = make_float4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
            if (accumulate) {
                const float4 r = dst[q];
                w.x += r.x; w.y += r.y; w.z += r.z; w.w += r.w;
            }
            dst[q] = w;
        }
    } else {
        uint4 pk[2];
        uint32_t* u = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(o[2 * q], o[2 * q + 1]);
            u[q] = *reinterpret_cast<const uint32_t*>(&h2);
        }
        uint4* dst = reinterpret_cast<uint4*>(y + at);
        dst[0] = pk[0];
        dst[1] = pk[1];
    }
}

__global__ void __launch_bounds__(UTHR)
k_conv_umma(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const UmmaArgs p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // stage tiles start on 1024-byte boundaries of the shared window (the swizzle patterns repeat there)
    unsigned char* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int S = p.stages;
    unsigned char* ctl = sm + (size_t)S * p.stage_bytes;  // barriers and the TMEM address slot
    const uint32_t full0 = smem_u32(ctl);                  // full[s]  at full0  + 8 s
    const uint32_t empty0 = full0 + 8u * S;                // empty[s] at empty0 + 8 s
    const uint32_t accum = empty0 + 8u * S;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(ctl + 16 * S + 8);
    __shared__ int s_fail;  // the MMA issuer gave up a wait: the accumulator is incomplete

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // brick of this block
    long long b = blockIdx.x;
    const int bx = (int)(b % p.tx);
    b /= p.tx;
    const int by = (int)(b % p.ty);
    b /= p.ty;
    const int bz = (int)(b % p.tz);
    const int bn = (int)(b / p.tz);
    const int x0 = bx * p.wb, y0 = by * p.hb, z0 = bz * p.db;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + 8u * s, 1);
            mbar_init(empty0 + 8u * s, 1);
        }
        mbar_init(accum, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int KB = 27 * p.nkb;
    const uint32_t sm0 = smem_u32(sm);

    int issued = 0;  // TMA stages issued (thread 0)
    if (threadIdx.x == 0) {
        // ---- producer: one stage = the A box and the B slice of one (tap, channel block)
        for (int kb = 0; kb < KB; ++kb, ++issued) {
            const int s = kb % S;
            const uint32_t use = (uint32_t)(kb / S);
            if (kb >= S && !mbar_wait(empty0 + 8u * s, (use & 1u) ^ 1u, p.tries)) break;
            const uint32_t fb = full0 + 8u * s;
            mbar_expect_tx(fb, p.tx_bytes);
            if (kb == p.withhold) continue;  // test of the failure path: this stage never fills
            const int tap = kb / p.nkb, cb = kb - tap * p.nkb;
            int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
            if (p.flip) { dz = -dz; dy = -dy; dx = -dx; }
            const uint32_t a_dst = sm0 + (uint32_t)s * p.stage_bytes;
            tma_load_5d(a_dst, &tmA, fb, cb * p.ck, x0 + dx, y0 + dy, z0 + dz, bn);
            tma_load_2d(a_dst + p.a_bytes, &tmB, fb, cb * p.ck, tap * p.cout);
        }
    } else if (threadIdx.x == 32) {
        // ---- MMA issuer: ck / 16 MMAs (K = 16 each) per stage, accumulating into TMEM
        bool ok = true;
        for (int kb = 0; kb < KB && ok; ++kb) {
            const int s = kb % S;
            const uint32_t use = (uint32_t)(kb / S);
            ok = mbar_wait(full0 + 8u * s, use & 1u, p.tries);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a_addr = sm0 + (uint32_t)s * p.stage_bytes;
            const uint32_t b_addr = a_addr + p.a_bytes;
            for (int k = 0; k < p.ck / 16; ++k) {
                // K step k starts 32 bytes further along the (swizzled) rows
                umma_f16(tmem, sdesc(a_addr + 32u * k, p.desc_hi), sdesc(b_addr + 32u * k, p.desc_hi), p.idesc,
                         (kb > 0 || k > 0) ? 1u : 0u);
            }
            umma_commit(empty0 + 8u * s);
        }
        // the accumulator barrier completes once every MMA issued above has retired, also after a
        // failed wait: TMEM and the stages are not released while an MMA may still use them
        if (!ok) s_fail = 1;
        umma_commit(accum);
    }
    __syncwarp();
    __syncthreads();  // s_fail is visible to every thread

    // ---- epilogue: warp w reads TMEM lanes 32w..32w+31 (voxels of the brick), 16 columns at a time
    const bool ready = mbar_wait(accum, 0u, p.tries) && !s_fail;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int m = warp * 32 + lane;
    const int dx = m % p.wb, dy = (m / p.wb) % p.hb, dz = m / (p.wb * p.hb);
    const int x = x0 + dx, y = y0 + dy, z = z0 + dz;
    const bool inside = ready && x < p.W && y < p.H && z < p.D;
    const long long v = (((long long)bn * p.D + z) * p.H + y) * p.W + x;
    for (int c0 = 0; c0 < p.cout; c0 += 16) {
        float o[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, o);  // whole warp, always
        if (inside) {
            if (p.bias) {
#pragma unroll
                for (int q = 0; q < 16; ++q) o[q] += p.bias[c0 + q];
            }
            if (p.relu) {
#pragma unroll
                for (int q = 0; q < 16; ++q) o[q] = fmaxf(o[q], 0.f);
            }
            store_cell16(p.y, p.yf, v * p.ldy + p.yoff + c0, p.accumulate, o);
        }
    }

    // after a failed wait, the TMA loads still in flight must land before the block's shared memory
    // is released (bounded as well); on success the completed accumulation implies that they have
    if (threadIdx.x == 0 && !ready) {
        for (int kb = issued - S < 0 ? 0 : issued - S; kb < issued; ++kb)
            mbar_wait(full0 + 8u * (kb % S), (uint32_t)(kb / S) & 1u, p.tries);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------- layers whose weights fit: marching bricks
// For cin x cout up to 2048 the weights of all taps stay in shared memory and a brick's input is loaded once, with a
// one-cell halo, instead of 27 shifted boxes per 128 voxels (k_conv_umma: bound by that traffic from L2, 775 us for
// 64 -> 32 channels on 128^3 voxels).  A brick is 8 x 16 columns of dz planes; its tile planes (10 x 18 cells, dz + 2 of
// them) come one by one through a ring of shared-memory slots, each written by one TMA box (zeros outside the grid) as
// rows of the cin channels of a cell (32, 64 or 128 bytes), swizzled with the span of a row.  (One box of
// 16-byte rows per 8 channels, unswizzled, took twice as long to load as the MMAs to run.)
//   A window of a plane at lateral offset (dy, dx) is the A operand: 128 rows (8 x by 16 y) from cell (dx + 1, dy + 1); 8
// consecutive x cells are an 8-row group, the next y row is 10 rows further.  The swizzle is a function of the address and
// the planes start on 1024 bytes, the longest pattern's period, so a window may start at any row.
//   One window serves the three taps dz of its (dy, dx): tile plane z' feeds the output planes o = z' - 1 - dz.  The B
// operand stacks the three taps' weights along N ([dy, dx][8-channel chunk][dz, cout][8 channels], unswizzled; backward data
// copies tap 26 - t there), and the accumulators of the planes lie in TMEM at decreasing columns, so the column groups of
// one MMA (N = 3 cout; 1 or 2 cout at the ends of the brick) are the accumulators of planes z', z' - 1, z' - 2.  Every output
// adds its products tap by tap in the order dz, dy, dx, channels.  MIRROR: backward data with the planes from the top down
// and the windows reversed, so that the products are added in the order of the weights' taps (as k_conv_umma does)
// without a flipped copy; used with 64 channels on a side, the flipped copy with 16 and 32.
//   Persistent: the blocks walk the bricks with a stride of the grid.  Warp 0 loads planes ahead, warp 1 issues MMAs, warps
// 2-5 store the accumulators of one brick while the next brick's MMAs fill the other set, so loads, MMAs and stores
// overlap (the form with one brick per block ran them one after another where only one block fits an SM).
//   Shared-memory reads bound it: an MMA reads 4 KB of A and 32 bytes per column of B, 43 clocks for N = 48 at 128 bytes a
// clock against 24 of multiplications.  Before (one brick per block, or
// k_conv_umma) and now: 256^3 voxels 16 -> 16 channels 390 and 325 us, 32 -> 16 958 and 470; 128^3 32 -> 32 305 and 96 us,
// 64 -> 32 772 and 179 (1296 TFLOP/s); 64^3 32 -> 64 109 and 37 us.
struct MarchArgs {
    int cin, cout;                // channels in/out
    int dz;                       // output planes per brick
    int slots;                    // tile plane slots
    int D, H, W;                  // grid of one sample
    int tx, ty, tz;               // bricks per sample
    int flip, relu, accumulate;
    int withhold;                 // >= 0: this plane of every brick is not loaded (failure-path test)
    long long tries, items;
    unsigned plane_bytes, plane_tx;  // slot pitch (1024-byte multiple), bytes a plane's load delivers
    unsigned w_bytes;             // weights of all taps
    unsigned idesc;               // MMA instruction descriptor without N
    unsigned long long a_hi;      // constant part of the A descriptors
    int tmem_cols;
    const float* bias;
    const bf16* w;
    bf16* y;
    float* yf;
    int ldy, yoff;
};

constexpr int MR_THR = 192;    // warp 0: TMA, warp 1: MMA, warps 2-5: epilogue
constexpr int MR_SLOTS = 8;    // most plane slots

constexpr int HB_X = 8, HB_Y = 16;            // brick extent along x and y (one plane = 128 voxels)
constexpr int HT_X = HB_X + 2, HT_Y = HB_Y + 2;

// unswizzled K-major descriptor: start, stride along K (LBO) and along M/N (SBO), version 1
__host__ __device__ __forceinline__ uint64_t desc_plain(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ULL << 46);
}

// tcgen05.mma with the descriptors given as 32-bit words (the issue loop advances the low words only)
__device__ __forceinline__ void umma_f16_w(uint32_t tmem_d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                           uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}" ::"r"(tmem_d),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The issuing warps below run their loops with all 32 lanes, and only the MMA and commit instructions are predicated on one
// elected lane: addresses and descriptors are then the same for the warp, and the compiler keeps them in uniform
// registers, where tcgen05.mma takes them from.  (In a branch for one thread every MMA moved its operands there first: about 60
// clocks per MMA and 700 to 900 per tile plane: 64 -> 32 channels on 128^3 voxels 229 us, 128 -> 64 on 64^3 223 us; with
// uniform operands 188 and 124 us.)
__device__ __forceinline__ uint32_t elect_lane() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e;
}
__device__ __forceinline__ void umma_elected(uint32_t lane, uint32_t tmem_d, uint32_t alo, uint32_t ahi, uint32_t blo,
                                             uint32_t bhi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "setp.ne.b32 q, %7, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}" ::"r"(tmem_d),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate), "r"(lane)
        : "memory");
}
__device__ __forceinline__ void commit_elected(uint32_t lane, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar),
        "r"(lane)
        : "memory");
}
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, long long tries) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, tries));
}

// zero the accumulator columns [0, cols) of this warp's TMEM lane quadrant
__device__ __forceinline__ void tmem_zero(uint32_t taddr, int cols) {
    const uint32_t z = 0u;
    __syncwarp();  // as in tmem_ld16
    for (int c = 0; c < cols; c += 16)
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
            "%1, %1};" ::"r"(taddr + (uint32_t)c), "r"(z)
            : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Weights of all taps into shared memory as [dy, dx][chunk][dz, cout][8] (tap t = 9 (dz + 1) + l,
// l = 3 (dy + 1) + (dx + 1); flipped: the tap 26 - t), in rounds of 7 16-byte vectors per thread: each
// round loads all of its vectors (read-only path) before storing them, so the copy costs one round trip
// to L2 per 14 KB (one for 16 x 16 channels, four for 32 x 32).
__device__ __forceinline__ void march_weights(const bf16* __restrict__ w, unsigned char* dst, int cout, int nkc,
                                             int flip) {
    constexpr int CAP = 7;
    const int nvec = 27 * cout * nkc;
    const uint4* src = reinterpret_cast<const uint4*>(w);
    for (int base = 0; base < nvec; base += CAP * MR_THR) {
        uint4 v[CAP];
#pragma unroll
        for (int j = 0; j < CAP; ++j) {
            const int q = base + threadIdx.x + j * MR_THR;
            if (q < nvec) v[j] = __ldg(src + q);
        }
#pragma unroll
        for (int j = 0; j < CAP; ++j) {
            const int q = base + threadIdx.x + j * MR_THR;
            if (q < nvec) {
                const int kc = q % nkc;
                const int co = (q / nkc) % cout;
                int t = q / (nkc * cout);
                if (flip) t = 26 - t;
                const int dzi = t / 9, l = t % 9;
                *reinterpret_cast<uint4*>(dst + ((size_t)(l * nkc + kc) * 3 * cout + dzi * cout + co) * 16) = v[j];
            }
        }
    }
}

struct Brick {
    int x0, y0, z0, n, planes;  // planes: output planes inside the grid
};
__device__ __forceinline__ Brick brick_of(const MarchArgs& p, long long q) {
    Brick r;
    r.x0 = (int)(q % p.tx) * HB_X;
    q /= p.tx;
    r.y0 = (int)(q % p.ty) * HB_Y;
    q /= p.ty;
    r.z0 = (int)(q % p.tz) * p.dz;
    r.n = (int)(q / p.tz);
    r.planes = min(p.dz, p.D - r.z0);
    return r;
}

// The MMAs of one tile plane: a, b: low descriptor words (the start field, bits 0-13 in 16-byte units, is advanced by adding
// to them; the shared window lies below 256 KB, so it never carries out).  d: accumulator of the first column group; idesc
// with N.  The accumulators start from zeros that the storing warps write: starting them by MMAs that overwrite
// takes an MMA per column group first.
template <int CK, bool MIRROR>
__device__ __forceinline__ void march_issue(uint32_t lane, uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi,
                                            uint32_t idesc, int cout) {
    const uint32_t bk = 6u * (uint32_t)cout;  // two 8-channel chunks of 3 cout rows
    uint32_t bl = b;
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const int at = MIRROR ? 8 - l : l;
        const uint32_t win = a + (uint32_t)(((at / 3) * HT_X + at % 3) * (CK / 8));
#pragma unroll
        for (int k = 0; k < CK / 16; ++k, bl += bk)
            umma_elected(lane, d, win + 2u * k, a_hi, bl, b_hi, idesc, 1u);
    }
}

template <int CK, bool MIRROR>
__global__ void __launch_bounds__(MR_THR)
k_conv_march(const __grid_constant__ CUtensorMap tmX, const MarchArgs p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t tile0 = smem_u32(sm), w0 = tile0 + (uint32_t)p.slots * p.plane_bytes;
    // barriers: plane full, plane empty, accumulators full, empty, all MMAs retired
    __shared__ __align__(8) unsigned long long bars[2 * MR_SLOTS + 5];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_fail;
    const uint32_t pfull = smem_u32(bars), pempty = pfull + 8 * MR_SLOTS, afull = pempty + 8 * MR_SLOTS;
    const uint32_t aempty = afull + 16, retired = aempty + 16;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int q = 0; q < 2 * MR_SLOTS; ++q) mbar_init(pfull + 8u * q, 1);
        for (int q = 0; q < 2; ++q) {
            mbar_init(afull + 8u * q, 1);
            mbar_init(aempty + 8u * q, 4);
        }
        mbar_init(retired, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    march_weights(p.w, sm + (size_t)p.slots * p.plane_bytes, p.cout, CK / 8, p.flip);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    const uint32_t set_cols = (uint32_t)p.tmem_cols / 2u;

    uint32_t filled = 0, phase = 0, pending = 0;  // producer, per slot: filled before, phase of the next fill, load issued
    if (threadIdx.x == 0) {
        bool ok = true;
        int slot = 0;
        for (long long q = blockIdx.x; q < p.items && ok; q += gridDim.x) {
            const Brick br = brick_of(p, q);
            for (int z = 0; z < br.planes + 2; ++z) {
                const uint32_t bit = 1u << slot;
                if (filled & bit) ok = mbar_wait(pempty + 8u * slot, ((phase >> slot) & 1u) ^ 1u, p.tries);
                if (!ok || s_fail) { ok = false; break; }
                mbar_expect_tx(pfull + 8u * slot, p.plane_tx);
                if (z != p.withhold) {
                    tma_load_5d(tile0 + (uint32_t)slot * p.plane_bytes, &tmX, pfull + 8u * slot, 0, br.x0 - 1, br.y0 - 1,
                                br.z0 - 1 + (MIRROR ? br.planes + 1 - z : z), br.n);
                    pending |= bit;
                } else {
                    pending &= ~bit;
                }
                filled |= bit;
                phase ^= bit;
                slot = slot + 1 == p.slots ? 0 : slot + 1;
            }
        }
    } else if (warp == 1) {
        const uint32_t one = elect_lane();
        bool ok = true;
        uint32_t ph = 0;
        int slot = 0, k = 0;
        const uint64_t db = desc_plain(w0, 3u * (uint32_t)p.cout * 16u, 128u);
        const uint32_t blo = (uint32_t)db, bhi = (uint32_t)(db >> 32);
        for (long long q = blockIdx.x; q < p.items && ok; q += gridDim.x, ++k) {
            const Brick br = brick_of(p, q);
            const int set = k & 1;
            const uint32_t acc = tmem + (uint32_t)set * set_cols;
            ok = mbar_wait_warp(aempty + 8u * set, (uint32_t)(k >> 1) & 1u, p.tries);  // stored and zeroed
            for (int z = 0; z < br.planes + 2 && ok; ++z) {
                ok = mbar_wait_warp(pfull + 8u * slot, (ph >> slot) & 1u, p.tries);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // group g (tap dz = g - 1) feeds plane z - g, whose accumulator is at (planes - 1 - z + g) cout
                const int g0 = max(0, z - br.planes + 1), g1 = min(2, z);
                march_issue<CK, MIRROR>(one, acc + (uint32_t)((br.planes - 1 - z + g0) * p.cout),
                                (uint32_t)p.a_hi | (((tile0 + (uint32_t)slot * p.plane_bytes) >> 4) & 0x3FFFu),
                                (uint32_t)(p.a_hi >> 32), blo + (uint32_t)(g0 * p.cout), bhi,
                                p.idesc | ((uint32_t)(((g1 - g0 + 1) * p.cout) >> 3) << 17), p.cout);
                commit_elected(one, pempty + 8u * slot);
                ph ^= 1u << slot;
                slot = slot + 1 == p.slots ? 0 : slot + 1;
            }
            if (!ok) s_fail = 1;
            commit_elected(one, afull + 8u * set);  // also after a failed wait: the storing warps see s_fail and stop
        }
        commit_elected(one, retired);  // completes once every MMA issued above has
    } else if (warp >= 2) {
        const int m = (warp & 3) * 32 + lane;  // a warp reads the TMEM lanes of its quarter: x = m % 8, y = m / 8
        tmem_zero(tmem + ((uint32_t)((warp & 3) * 32) << 16), p.tmem_cols);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane < 2) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(aempty + 8u * lane) : "memory");
        int k = 0;
        for (long long q = blockIdx.x; q < p.items; q += gridDim.x, ++k) {
            const Brick br = brick_of(p, q);
            const int set = k & 1;
            const bool done = mbar_wait(afull + 8u * set, (uint32_t)(k >> 1) & 1u, p.tries);
            if (__any_sync(0xffffffffu, !done || s_fail)) {
                s_fail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int x = br.x0 + m % HB_X, y = br.y0 + m / HB_X;
            const bool inside = x < p.W && y < p.H;
            const uint32_t acc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)set * set_cols;
            for (int c0 = 0; c0 < p.cout; c0 += 16) {
                float bias[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) bias[e] = p.bias ? __ldg(p.bias + c0 + e) : 0.f;
                for (int zo = 0; zo < br.planes; ++zo) {
                    const int z = br.z0 + (MIRROR ? br.planes - 1 - zo : zo);
                    const long long v = (((long long)br.n * p.D + z) * p.H + y) * p.W + x;
                    float o[16];
                    tmem_ld16(acc + (uint32_t)((br.planes - 1 - zo) * p.cout + c0), o);
                    if (inside) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) o[e] += bias[e];
                        if (p.relu) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] = fmaxf(o[e], 0.f);
                        }
                        store_cell16(p.y, p.yf, v * p.ldy + p.yoff + c0, p.accumulate, o);
                    }
                }
            }
            tmem_zero(acc, br.planes * p.cout);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(aempty + 8u * set) : "memory");
        }
    }
    __syncwarp();
    __syncthreads();
    // every MMA has retired (TMEM and the operands are free) and, after a failed wait, every load in flight has landed before
    // the block's memory is released; both waits are bounded
    mbar_wait(retired, 0u, p.tries);
    if (threadIdx.x == 0 && s_fail) {
        for (int q = 0; q < p.slots; ++q)
            if ((pending >> q) & 1u) mbar_wait(pfull + 8u * q, ((phase >> q) & 1u) ^ 1u, p.tries);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------- wide layers: marching pairs of bricks, streamed weights
// For larger cin x cout the weights do not fit shared memory beside the input (442 KB for 128 -> 64 channels).  Windows,
// stacked taps dz and the order of the products are those of k_conv_march; the weights of (dy, dx, block of ck channels),
// 3 nc rows (nc = 16, 32 or 64 output channels), come through a ring of three stages for every tile
// plane, and two bricks side by side (16 x 16 columns, one tile of 18 x 18 cells) use each stage, so a stage feeds about 800
// clocks of MMAs.  A work item marches along z over zc planes; the tile planes come through a ring of (plane, channel
// block) slots, the accumulators of each brick lie in a ring of four planes (a window's column groups wrap around its end:
// two MMAs then), and four warps store a plane as soon as its last tap is done.
//   The weights' stream from L2 (30 bytes a clock and SM) and the shared-memory reads bound it; k_conv_umma reads 27 boxes of
// the input per 128 voxels instead (46 bytes a clock).  64^3 voxels: 128 -> 64 channels
// 204 and 115 us, 64 -> 64 120 and 69 us.
constexpr int WD_RING = 3;       // weight stages
constexpr int WD_SLOTS = 4;      // most tile slots
constexpr int WD_ACC = 4;        // accumulator planes per brick
constexpr int WT_X = 2 * HB_X + 2;
struct WideArgs {
    int nc;                       // output channels
    int ck, ncb;                  // channels per K block, K blocks
    int zc, slots;                // output planes per work item, tile slots
    int D, H, W, tx, ty, tz;
    int relu, accumulate;
    int withhold;                 // >= 0: the weight loads of this (l, K block) are withheld (failure-path test)
    long long tries, items;
    unsigned tile_bytes, tile_tx, ring_bytes, ring_tx;
    unsigned idesc;               // without N
    unsigned long long a_hi, b_hi;
    const float* bias;
    bf16* y;
    float* yf;
    int ldy, yoff;
};

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                            int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

struct WideItem {
    int x0, y0, z0, n, planes;
};
__device__ __forceinline__ WideItem wide_item(const WideArgs& p, long long q) {
    WideItem r;
    r.x0 = (int)(q % p.tx) * (2 * HB_X);
    q /= p.tx;
    r.y0 = (int)(q % p.ty) * HB_Y;
    q /= p.ty;
    r.z0 = (int)(q % p.tz) * p.zc;
    r.n = (int)(q / p.tz);
    r.planes = min(p.zc, p.D - r.z0);
    return r;
}

template <int CK, bool MIRROR>
__global__ void __launch_bounds__(MR_THR, 1)
k_conv_wide(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const WideArgs p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t sm0 = smem_u32(smem_raw) + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t ring0 = sm0 + (uint32_t)p.slots * p.tile_bytes;
    // barriers: tile full / empty, ring full / empty, accumulator full / empty, all MMAs retired
    __shared__ __align__(8) unsigned long long bars[2 * (WD_SLOTS + WD_RING + WD_ACC) + 1];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_fail;
    const uint32_t tfull = smem_u32(bars), tempty = tfull + 8 * WD_SLOTS, rfull = tempty + 8 * WD_SLOTS;
    const uint32_t rempty = rfull + 8 * WD_RING, afull = rempty + 8 * WD_RING, aempty = afull + 8 * WD_ACC;
    const uint32_t retired = aempty + 8 * WD_ACC;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int q = 0; q < 2 * (WD_SLOTS + WD_RING) + WD_ACC; ++q) mbar_init(tfull + 8u * q, 1);
        for (int q = 0; q < WD_ACC; ++q) mbar_init(aempty + 8u * q, 4);
        mbar_init(retired, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);

    // producer, per slot: filled before, phase of the next fill, load issued
    uint32_t tfilled = 0, tphase = 0, tpending = 0, rfilled = 0, rphase = 0, rpending = 0;
    if (threadIdx.x == 0) {
        bool ok = true;
        int ts = 0, rs = 0;
        auto tile = [&](const WideItem& it, int z, int cb) {
            const uint32_t bit = 1u << ts;
            if (tfilled & bit) ok = mbar_wait(tempty + 8u * ts, ((tphase >> ts) & 1u) ^ 1u, p.tries);
            if (!ok || s_fail) { ok = false; return; }
            mbar_expect_tx(tfull + 8u * ts, p.tile_tx);
            tma_load_5d(sm0 + (uint32_t)ts * p.tile_bytes, &tmA, tfull + 8u * ts, cb * p.ck, it.x0 - 1, it.y0 - 1,
                        it.z0 - 1 + (MIRROR ? it.planes + 1 - z : z), it.n);
            tfilled |= bit;
            tpending |= bit;
            tphase ^= bit;
            ts = ts + 1 == p.slots ? 0 : ts + 1;
        };
        const int ahead = min(p.slots - p.ncb, p.ncb);  // blocks of the next plane whose slots this plane does not use
        for (long long q = blockIdx.x; q < p.items && ok; q += gridDim.x) {
            const WideItem it = wide_item(p, q);
            for (int z = 0; z < it.planes + 2 && ok; ++z)
                for (int l = 0; l < 9 && ok; ++l) {
                    for (int cb = 0; cb < p.ncb && ok; ++cb) {
                        // this plane's tiles, but for those loaded ahead (below)
                        if (l == 0 && (z == 0 || cb >= ahead)) tile(it, z, cb);
                        if (!ok) break;
                        const uint32_t bit = 1u << rs;
                        if (rfilled & bit) ok = mbar_wait(rempty + 8u * rs, ((rphase >> rs) & 1u) ^ 1u, p.tries);
                        if (!ok || s_fail) { ok = false; break; }
                        mbar_expect_tx(rfull + 8u * rs, p.ring_tx);
                        if (l * p.ncb + cb != p.withhold) {
                            tma_load_4d(ring0 + (uint32_t)rs * p.ring_bytes, &tmB, rfull + 8u * rs, cb * p.ck, 0, l, 0);
                            rpending |= bit;
                        } else {
                            rpending &= ~bit;
                        }
                        rfilled |= bit;
                        rphase ^= bit;
                        rs = rs + 1 == WD_RING ? 0 : rs + 1;
                    }
                    if (l == 4 && z < it.planes + 1)
                        for (int cb = 0; cb < ahead && ok; ++cb) tile(it, z + 1, cb);
                }
        }
    } else if (warp == 1) {
        const uint32_t one = elect_lane();
        bool ok = true;
        uint32_t tph = 0, rph = 0;
        int ts = 0, rs = 0;      // first tile slot of the plane, ring stage
        int done = 0;            // output planes of the items before, modulo 4
        constexpr uint32_t ROW16 = CK / 8;  // 16-byte units of a tile or weight row
        const uint32_t a_hi = (uint32_t)(p.a_hi >> 32), b_hi = (uint32_t)(p.b_hi >> 32);
        uint32_t aph = 0;        // accumulator slots' phases waited for, one bit each
        for (long long q = blockIdx.x; q < p.items && ok; q += gridDim.x) {
            const int planes = wide_item(p, q).planes;
            for (int z = 0; z < planes + 2 && ok; ++z) {
                if (z < planes) {  // the new plane's accumulators are stored and zeroed
                    const int o = (done + z) & 3;
                    ok = mbar_wait_warp(aempty + 8u * o, (aph >> o) & 1u, p.tries);
                    aph ^= 1u << o;
                }
                // group g (tap dz = g - 1) feeds plane z - g; plane o (counted over the items) is column group 3 - o mod 4
                const int g0 = max(0, z - planes + 1), g1 = min(2, z), ng = g1 - g0 + 1;
                const int s0 = 3 - ((done + z - g0) & 3), n1 = min(ng, WD_ACC - s0), n2 = ng - n1;
                const uint32_t d1 = tmem + (uint32_t)(s0 * p.nc), b1 = (uint32_t)(g0 * p.nc) * ROW16;
                const uint32_t b2 = b1 + (uint32_t)(n1 * p.nc) * ROW16;
                const uint32_t id1 = p.idesc | ((uint32_t)((n1 * p.nc) >> 3) << 17);
                const uint32_t id2 = p.idesc | ((uint32_t)((n2 * p.nc) >> 3) << 17);
                for (int l = 0; l < 9 && ok; ++l) {
                    const int at = MIRROR ? 8 - l : l;
                    const uint32_t win = (uint32_t)((at / 3) * WT_X + at % 3) * ROW16;
                    int t = ts;
                    for (int cb = 0; cb < p.ncb; ++cb) {
                        if (l == 0) {
                            ok = mbar_wait_warp(tfull + 8u * t, (tph >> t) & 1u, p.tries);
                            if (!ok) break;
                            tph ^= 1u << t;
                        }
                        ok = mbar_wait_warp(rfull + 8u * rs, (rph >> rs) & 1u, p.tries);
                        if (!ok) break;
                        rph ^= 1u << rs;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t b = (uint32_t)p.b_hi | (((ring0 + (uint32_t)rs * p.ring_bytes) >> 4) & 0x3FFFu);
                        const uint32_t a = ((uint32_t)p.a_hi | (((sm0 + (uint32_t)t * p.tile_bytes) >> 4) & 0x3FFFu)) + win;
#pragma unroll
                        for (int k = 0; k < CK / 16; ++k) {
#pragma unroll
                            for (int j = 0; j < 2; ++j) {  // the two bricks: independent accumulators
                                const uint32_t ak = a + (uint32_t)(j * HB_X) * ROW16 + 2u * k;
                                umma_elected(one, d1 + 256u * j, ak, a_hi, b + b1 + 2u * k, b_hi, id1, 1u);
                                if (n2 > 0) umma_elected(one, tmem + 256u * j, ak, a_hi, b + b2 + 2u * k, b_hi, id2, 1u);
                            }
                        }
                        commit_elected(one, rempty + 8u * rs);
                        rs = rs + 1 == WD_RING ? 0 : rs + 1;
                        if (l == 8) commit_elected(one, tempty + 8u * t);
                        t = t + 1 == p.slots ? 0 : t + 1;
                    }
                }
                for (int cb = 0; cb < p.ncb; ++cb) ts = ts + 1 == p.slots ? 0 : ts + 1;
                if (!ok) s_fail = 1;
                // plane z - 2 is complete (after a failed wait: the storing warps see s_fail and stop)
                if (z >= 2 || !ok) commit_elected(one, afull + 8u * (uint32_t)((done + max(z - 2, 0)) & 3));
            }
            done = (done + planes) & 3;
        }
        commit_elected(one, retired);  // completes once every MMA issued above has
    } else if (warp >= 2) {
        const int m = (warp & 3) * 32 + lane;  // a warp reads the TMEM lanes of its quarter: x = m % 8, y = m / 8
        tmem_zero(tmem + ((uint32_t)((warp & 3) * 32) << 16), 512);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane < WD_ACC) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(aempty + 8u * lane) : "memory");
        long long o = 0;
        bool ok = true;
        for (long long q = blockIdx.x; q < p.items && ok; q += gridDim.x) {
            const WideItem it = wide_item(p, q);
            const int y = it.y0 + m / HB_X;
            for (int zo = 0; zo < it.planes; ++zo, ++o) {
                const uint32_t slot = (uint32_t)(o & 3);
                const bool done = mbar_wait(afull + 8u * slot, (uint32_t)(o >> 2) & 1u, p.tries);
                if (__any_sync(0xffffffffu, !done || s_fail)) {
                    s_fail = 1;
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int z = it.z0 + (MIRROR ? it.planes - 1 - zo : zo);
                for (int j = 0; j < 2; ++j) {
                    const int x = it.x0 + j * HB_X + m % HB_X;
                    const bool inside = x < p.W && y < p.H;
                    const long long v = (((long long)it.n * p.D + z) * p.H + y) * p.W + x;
                    const uint32_t acc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 256u * j + (3u - slot) * (uint32_t)p.nc;
                    for (int c = 0; c < p.nc; c += 16) {
                        float r[16];
                        tmem_ld16(acc + (uint32_t)c, r);
                        if (inside) {
                            if (p.bias) {
#pragma unroll
                                for (int e = 0; e < 16; ++e) r[e] += __ldg(p.bias + c + e);
                            }
                            if (p.relu) {
#pragma unroll
                                for (int e = 0; e < 16; ++e) r[e] = fmaxf(r[e], 0.f);
                            }
                            store_cell16(p.y, p.yf, v * p.ldy + p.yoff + c, p.accumulate, r);
                        }
                    }
                    tmem_zero(acc, p.nc);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(aempty + 8u * slot) : "memory");
            }
        }
    }
    __syncwarp();
    __syncthreads();
    // every MMA has retired (TMEM and the operands are free) and, after a failed wait, every load in flight has landed before
    // the block's memory is released; both waits are bounded
    mbar_wait(retired, 0u, p.tries);
    if (threadIdx.x == 0 && s_fail) {
        for (int q = 0; q < p.slots; ++q)
            if ((tpending >> q) & 1u) mbar_wait(tfull + 8u * q, ((tphase >> q) & 1u) ^ 1u, p.tries);
        for (int q = 0; q < WD_RING; ++q)
            if ((rpending >> q) & 1u) mbar_wait(rfull + 8u * q, ((rphase >> q) & 1u) ^ 1u, p.tries);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ---------------------------------------------------------------- weight gradient on tcgen05
// dW[t][co][ci] = sum over voxels v of dY[v][co] X[v + off(t)][ci] (zero padding): GEMMs whose reduction
// runs over voxels, with both operands taken as they lie in memory.  A channels-last tile in shared memory
// whose cells are 16-byte rows (8 channels of one voxel) is an MN-major operand without swizzle: eight
// consecutive x cells are one core matrix (8 channels x 8 voxels of the reduction), so neither tensor is
// transposed or packed first.  (Packing both channel-major, dY three times, and streaming one shifted box
// per tap took 1.6 + 0.8 ms of a training step on 4 x 64^3 voxels and was bound by the 27 reads of dY from
// L2.)
//   A block marches along z over a column of 8 x 16 cells.  Per plane it loads dY (8 x 16, no halo, laid out
//   [chunk of 8 channels][y][x]) and X (10 x 18 with the halo, [y][chunk][x]), each by one TMA box, zeros
//   outside the grid, and keeps three planes of X, so every value is loaded once (and its halo).
//   A (M) = X: core matrices along M are 160 bytes apart, which walks the chunks of a row of the tile and
//   then the next row, so for 16 or 32 channels the three taps dy = -1, 0, +1 lie along M by themselves
//   ("stacked": 6 of 8 or 12 of 16 core matrices used); 128 channels fill M = 128 with one tap.
//   B (N) = dY, N = cout.  K = 16 voxels: two rows of 8 cells, 8 MMAs per tap and plane.  The taps dx and
//   dz are other start addresses (16 bytes further, another plane).
//   Accumulators: cout TMEM columns per tap (per three taps when stacked); where the 27 taps need more than
//   512 columns they are divided over blocks by dz (rule in wgrad_plan).  Taps dz whose planes all lie outside the grid
//   for a block (one-plane grids: two of three) are left out.
// Shared-memory reads bound it for 16 and 32 channels (2.5 to 5 KB per MMA of N = 16 or 32).
struct WgArgs {
    int cin, cout;
    int cb, nchunk;               // input channels of a block (16, 32 or 128; the last one's may exceed cin), cb / 8
    int stacked, ndz;             // taps dy along M; taps dz accumulated by one block
    int D, H, W, tx, ty;          // the grid's axes as the kernel takes them (wgrad_axes)
    int tapx, tapy, tapz;         // a step's distance in the tap index along each
    int zc, nzc;                  // planes per block, blocks along z
    int slots;
    unsigned x_tx, dy_tx;         // bytes of the two boxes
    unsigned x_bytes, slot_bytes; // their places in a slot
    unsigned idesc;
    unsigned long long a_hi, b_hi;  // descriptors without the start address
    int m64;                      // MMA M = 64 (16 channels; else 128)
    int tmem_cols;
    long long tries;
    float* dw;
};

constexpr unsigned WX_ROW = 10 * 16;  // bytes of one X tile row of one chunk

__global__ void __launch_bounds__(UTHR)
k_wgrad_umma(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmY, const WgArgs p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int S = p.slots;
    __shared__ __align__(8) unsigned long long s_bar[2 * 8 + 1];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    const uint32_t full0 = smem_u32(s_bar), empty0 = full0 + 8u * 8u, accum = empty0 + 8u * 8u;
    const uint32_t sm0 = smem_u32(sm);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // brick column, z chunk and sample
    int b = blockIdx.x;
    const int x0 = (b % p.tx) * 8;
    b /= p.tx;
    const int y0 = (b % p.ty) * 16;
    b /= p.ty;
    const int z0 = (b % p.nzc) * p.zc, bn = b / p.nzc;
    const int nsteps = min(p.zc, p.D - z0);
    // tap group and channel block
    const int ngrp = 3 / p.ndz, cb = blockIdx.y / ngrp;
    const int dz0 = p.ndz == 3 ? 0 : blockIdx.y % ngrp;
    const int ndyu = p.stacked ? 1 : 3;
    // the X planes of tap dz that the block multiplies, z0 + dz - 1 .. z0 + nsteps + dz - 2, meet the grid
    auto used = [&](int dz) { return z0 + nsteps + dz - 2 >= 0 && z0 + dz - 1 < p.D; };
    if (p.ndz == 1 && !used(dz0)) return;
    const int nacc = p.ndz * ndyu * 3;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + 8u * s, 1);
            mbar_init(empty0 + 8u * s, 1);
        }
        mbar_init(accum, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    tmem_zero(tmem + ((uint32_t)(warp * 32) << 16), nacc * p.cout);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    // load l brings X plane z0 + l + xoff and dY plane z0 + l (when in range); step k multiplies dY plane
    // z0 + k with the X planes of loads k .. k + ndz - 1
    const int xoff = p.ndz == 3 ? -1 : dz0 - 1, lead = p.ndz - 1, nloads = nsteps + lead;
    int issued = 0;
    if (threadIdx.x == 0) {
        for (int l = 0; l < nloads; ++l, ++issued) {
            const int s = l % S;
            if (l >= S && !mbar_wait(empty0 + 8u * s, (uint32_t)(l / S - 1) & 1u, p.tries)) break;
            const int zx = z0 + l + xoff;
            const bool xin = zx >= 0 && zx < p.D, yin = l < nsteps;
            const uint32_t fb = full0 + 8u * s, dst = sm0 + (uint32_t)s * p.slot_bytes;
            mbar_expect_tx(fb, (xin ? p.x_tx : 0u) + (yin ? p.dy_tx : 0u));
            if (xin) tma_load_5d(dst, &tmX, fb, 0, x0 - 1, cb * p.nchunk, y0 - 1, bn * p.D + zx);
            if (yin) tma_load_5d(dst + p.x_bytes, &tmY, fb, 0, x0, y0, 0, bn * p.D + z0 + l);
        }
    } else if (threadIdx.x == 32) {
        bool ok = true;
        int seen = 0;  // loads known to have landed
        const uint32_t alo = (uint32_t)p.a_hi, ahi = (uint32_t)(p.a_hi >> 32);
        const uint32_t blo = (uint32_t)p.b_hi, bhi = (uint32_t)(p.b_hi >> 32);
        const uint32_t yrow = (uint32_t)p.nchunk * (WX_ROW / 16);  // one row of the X tile, 16-byte units
        for (int k = 0; k < nsteps && ok; ++k) {
            for (; seen <= k + lead && ok; ++seen) ok = mbar_wait(full0 + 8u * (seen % S), (uint32_t)(seen / S) & 1u, p.tries);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // descriptor low words: the start field (16-byte units) is advanced by adding to them
            const uint32_t yl = blo + ((sm0 + (uint32_t)(k % S) * p.slot_bytes + p.x_bytes) >> 4);
            for (int dz = 0; dz < p.ndz; ++dz) {
                const int zx = z0 + k + dz + xoff;
                if (zx < 0 || zx >= p.D) continue;  // the zero padding: nothing to add
                uint32_t xl = alo + ((sm0 + (uint32_t)((k + dz) % S) * p.slot_bytes) >> 4);
                uint32_t dt = tmem + (uint32_t)(dz * ndyu * 3) * p.cout;
                for (int dy = 0; dy < ndyu; ++dy, xl += yrow)
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx, dt += p.cout)
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            umma_f16_w(dt, xl + dx + 2 * j * yrow, ahi, yl + 16 * j, bhi, p.idesc, 1u);
            }
            umma_commit(empty0 + 8u * (k % S));
        }
        if (!ok) s_fail = 1;
        umma_commit(accum);
    }
    __syncwarp();
    __syncthreads();

    // ---- epilogue: row r of the accumulators (TMEM lane r; with M = 64 rows 16w .. 16w + 15 lie in the first
    // 16 lanes of warp w's quadrant) is channel r % 8 of core matrix r / 8
    const bool ready = mbar_wait(accum, 0u, p.tries) && !s_fail;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int r = p.m64 ? warp * 16 + lane : warp * 32 + lane;
    const int core = r >> 3;
    const int dys = p.stacked ? core / p.nchunk : 0;
    const int ci = cb * p.cb + (p.stacked ? core % p.nchunk : core) * 8 + (r & 7);
    const bool live = ready && !(p.m64 && lane >= 16) && dys < 3 && ci < p.cin;
    for (int acc = 0; acc < nacc; ++acc) {
        const int dx = acc % 3, q = acc / 3;
        const int dy = p.stacked ? dys : q % ndyu, dz = dz0 + q / ndyu;
        if (!used(dz)) continue;  // (the same for the whole block)
        float* dst = p.dw + ((long long)(dz * p.tapz + dy * p.tapy + dx * p.tapx) * p.cout) * p.cin + ci;
        for (int c0 = 0; c0 < p.cout; c0 += 16) {
            float o[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * p.cout + c0), o);  // whole warp, always
            if (live) {
#pragma unroll
                for (int k = 0; k < 16; ++k) atomicAdd(dst + (long long)(c0 + k) * p.cin, o[k]);
            }
        }
    }

    // after a failed wait, the loads still in flight land before the shared memory is released
    if (threadIdx.x == 0 && !ready) {
        for (int l = issued - S < 0 ? 0 : issued - S; l < issued; ++l)
            mbar_wait(full0 + 8u * (l % S), (uint32_t)(l / S) & 1u, p.tries);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
    }
}

// compact copy of a channel slice (operands whose rows do not start on 16 bytes)
__global__ void k_compact(const __nv_bfloat16* __restrict__ x, int ld, int off, int c, long long n,
                          __nv_bfloat16* __restrict__ out) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        out[q] = x[(q / c) * ld + off + q % c];
}

// ---------------------------------------------------------------- host side

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    });
    return fn;
}

// swizzle span = row length of a k block (ck bf16 = 32, 64 or 128 bytes)
CUtensorMapSwizzle tma_swizzle(int ck) {
    return ck == 16 ? CU_TENSOR_MAP_SWIZZLE_32B : (ck == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B);
}
// the matching layout code of the MMA shared-memory descriptor (bits 61-63)
unsigned long long umma_layout(int ck) { return ck == 16 ? 6ULL : (ck == 32 ? 4ULL : 2ULL); }

unsigned round1024(unsigned v) { return (v + 1023u) & ~1023u; }

// the marching kernel: weights of all taps in up to 108 KB, on grids at least one brick across
bool march_shape(int cin, int cout, int d, int h, int wd) {
    return (cin == 16 || cin == 32 || cin == 64) && (cout == 16 || cout == 32 || cout == 64) && cin * cout <= 2048 &&
           wd >= HB_X && h >= HB_Y && d >= 4;
}

pf_status conv_march(const void* x, int ldx, int xoff, const void* w, int cin, int cout, const float* bias, int relu,
                     int flip, void* y_bf16, float* y_f32, int ldy, int yoff, int accumulate, int n, int d, int h,
                     int wd, cudaStream_t stream, PFN_cuTensorMapEncodeTiled_v12000 enc) {
    MarchArgs a{};
    a.cin = cin;
    a.cout = cout;
    a.D = d;
    a.H = h;
    a.W = wd;
    a.relu = relu;
    a.accumulate = accumulate;
    a.tries = g_test_tries > 0 ? g_test_tries : WAIT_TRIES;
    const int withhold = g_test_withhold;
    g_test_withhold = -1;
    g_test_tries = 0;
    a.w_bytes = (unsigned)(27 * cout * cin * 2);
    a.tx = (wd + HB_X - 1) / HB_X;
    a.ty = (h + HB_Y - 1) / HB_Y;
    const unsigned row = (unsigned)cin * 2;
    a.plane_tx = (unsigned)(HT_X * HT_Y) * row;
    a.plane_bytes = round1024(a.plane_tx);
    // Blocks per SM and planes per brick: the fewest clocks.  Up to four blocks share the 512 TMEM columns (two accumulator
    // sets each) and the shared memory.  An MMA of m cout columns takes the longer of its multiplications and its reads from
    // shared memory; a block's issuing warp takes about 38 clocks per MMA and 550 per plane (fitted to 16, 32 and 64 input
    // channels), so several blocks keep the tensor core busy where a plane has few MMAs.  The ends of a brick (m = 1, 2) cost
    // nearly as much as its middle.
    long long best = -1;
    int occ = 1;
    for (int o = 1; o <= 4; ++o) {
        const unsigned room = 216u * 1024u / o - 2048u * (o > 1);
        const int slots = room > a.w_bytes ? (int)((room - a.w_bytes) / a.plane_bytes) : 0;
        if (slots < 3) continue;
        for (int dz = 1; dz <= d && 2 * dz * cout <= (o == 3 ? 128 : 512 / o); ++dz) {
            const long long tz = (d + dz - 1) / dz, items = (long long)a.tx * a.ty * tz * n;
            long long clocks = 0;
            for (int z = 0; z < dz + 2; ++z) {
                const int m = std::min(2, z) - std::max(0, z - dz + 1) + 1;
                clocks += std::max(m * cout / 2, 32 + m * cout / 4);
            }
            const long long mmas = 9 * (cin / 16), issue = (dz + 2) * (550 + 38 * mmas);
            const long long cost = ((items + 152 * o - 1) / (152 * o)) * std::max(o * clocks * mmas, issue) + 3000;
            if (best < 0 || cost < best) {
                best = cost;
                occ = o;
                a.dz = dz;
                a.tz = (int)tz;
                a.items = items;
                a.slots = slots < MR_SLOTS ? slots : MR_SLOTS;
            }
        }
    }
    if (best < 0) return PF_E_INVALID;
    a.withhold = withhold < 0 ? -1 : withhold % (a.dz + 2);
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(UM >> 4) << 24);
    // K-major, swizzled with the span of a row; stride between 8-row groups: one tile row of 10 cells
    a.a_hi = (1ULL << 16) | (1ULL << 46) | (umma_layout(cin) << 61) | ((unsigned long long)(HT_X * row >> 4) << 32);
    const int cols = 2 * a.dz * cout;
    a.tmem_cols = cols <= 32 ? 32 : (cols <= 64 ? 64 : (cols <= 128 ? 128 : (cols <= 256 ? 256 : 512)));
    a.bias = bias;
    a.w = (const bf16*)w;
    a.y = (bf16*)y_bf16;
    a.yf = y_f32;
    a.ldy = ldy;
    a.yoff = yoff;
    alignas(64) CUtensorMap mX;
    const cuuint64_t dims[5] = {(cuuint64_t)cin, (cuuint64_t)wd, (cuuint64_t)h, (cuuint64_t)d, (cuuint64_t)n};
    const cuuint64_t xr = (cuuint64_t)ldx * 2;
    const cuuint64_t strides[4] = {xr, xr * wd, xr * wd * h, xr * wd * h * d};
    const cuuint32_t box[5] = {(cuuint32_t)cin, (cuuint32_t)HT_X, (cuuint32_t)HT_Y, 1, 1};
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    if (enc(&mX, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)((const bf16*)x + xoff), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, tma_swizzle(cin), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return PF_E_INVALID;
    const size_t smem = 1024 + (size_t)a.slots * a.plane_bytes + a.w_bytes;
    const bool mirror = flip && (cin == 64 || cout == 64);
    a.flip = flip && !mirror;
    auto k = cin == 16 ? (mirror ? k_conv_march<16, true> : k_conv_march<16, false>)
             : cin == 32 ? (mirror ? k_conv_march<32, true> : k_conv_march<32, false>)
                         : (mirror ? k_conv_march<64, true> : k_conv_march<64, false>);
    static std::once_flag attr_once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(attr_once, [] {
        for (auto f : {k_conv_march<16, false>, k_conv_march<32, false>, k_conv_march<64, false>, k_conv_march<16, true>,
                       k_conv_march<32, true>, k_conv_march<64, true>}) {
            const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 218 * 1024);
            if (e != cudaSuccess) attr_err = e;
        }
    });
    if (attr_err != cudaSuccess || smem > 218u * 1024u) return PF_E_CUDA;
    k<<<(unsigned)std::min<long long>(a.items, 152LL * occ), MR_THR, smem, stream>>>(mX, a);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

// Brick of 128 cells of k_conv_umma: 32 x 4 x 1, 16 x 8 x 1 or 8 x 8 x 2 (x fastest), the widest that the grid fills.
struct UmmaBricks {
    int wb, hb, db;
    long long tx, ty, tz;
};
UmmaBricks umma_bricks(int d, int h, int wd) {
    UmmaBricks b;
    b.wb = wd >= 32 ? 32 : (wd >= 16 ? 16 : 8);
    b.hb = b.wb == 32 ? 4 : 8;
    b.db = UM / (b.wb * b.hb);
    b.tx = (wd + b.wb - 1) / b.wb;
    b.ty = (h + b.hb - 1) / b.hb;
    b.tz = (d + b.db - 1) / b.db;
    return b;
}

// The wide-layer kernel: more weights than fit shared memory, in blocks of 32 or 64 input channels, all output channels in
// one pass (of several 32- or 64-channel passes each reads the input again: 128 -> 128 channels on 64^3 276 us, k_conv_umma
// 205; of 16-channel ones 64 -> 80 284 and 109), bricks of which no more hang over the grid than of k_conv_umma's (by less than 1.4: at
// 1.6, 20 rows, 64 -> 64 157 and 136 us, at 1.33, 24 rows, 157 and 165), and enough 16 x 16 planes of them for the chip (a
// work item needs two more tile planes than it has output planes: one plane 103 and 91 us, two 71 and 91).  64 -> 64
// channels: 128 planes 23 and 19 us, 297 of 33^3 39 and 33, 360 of 40^3 34 and 48, 512 39 and 62, 1024 64 and 107.
bool wide_shape(int cin, int cout, int n, int d, int h, int wd) {
    if (cin % 32 || (cout != 16 && cout != 32 && cout != 64) || cin * cout <= 2048) return false;
    const UmmaBricks b = umma_bricks(d, h, wd);
    const long long planes = (long long)((wd + 15) / 16) * ((h + 15) / 16) * d * n;
    return cin / (cin % 64 == 0 ? 64 : 32) <= 3 && d >= 2 && wd > HB_X && h >= HB_Y && planes >= 500 &&
           256.0 * planes <= 1.4 * UM * (double)(b.tx * b.ty * b.tz * n);
}

pf_status conv_wide(const void* x, int ldx, int xoff, const void* w, int cin, int cout, const float* bias, int relu,
                    int flip, void* y_bf16, float* y_f32, int ldy, int yoff, int accumulate, int n, int d, int h, int wd,
                    cudaStream_t stream, PFN_cuTensorMapEncodeTiled_v12000 enc) {
    WideArgs a{};
    a.nc = cout;
    a.ck = cin % 64 == 0 ? 64 : 32;
    a.ncb = cin / a.ck;
    a.D = d;
    a.H = h;
    a.W = wd;
    a.relu = relu;
    a.accumulate = accumulate;
    a.tries = g_test_tries > 0 ? g_test_tries : WAIT_TRIES;
    a.withhold = g_test_withhold < 0 ? -1 : g_test_withhold % (9 * a.ncb);
    g_test_withhold = -1;
    g_test_tries = 0;
    a.tx = (wd + 2 * HB_X - 1) / (2 * HB_X);
    a.ty = (h + HB_Y - 1) / HB_Y;
    // output planes per work item: the fewest waves x clocks.  An MMA of m nc columns takes the longer of its
    // multiplications and its reads from shared memory; half of the windows of three groups wrap around the ring
    const auto mma = [&](int m) { return std::max(m * a.nc / 2, 32 + m * a.nc / 4); };
    const long long full = (mma(3) + mma(1) + mma(2)) / 2;
    // the tile planes of an item: one and two groups at each end, three between them (one plane: one group each time)
    const long long ends = 2LL * (mma(1) + mma(2)), single = 3LL * mma(1);
    long long best = -1;
    for (int zc = 1; zc <= d; ++zc) {
        const long long tz = (d + zc - 1) / zc, items = (long long)a.tx * a.ty * tz * n;
        const long long clocks = zc == 1 ? single : ends + (zc - 2) * full;
        const long long cost = ((items + 151) / 152) * clocks * 2 * 9 * (cin / 16) + 4000;
        if (best < 0 || cost < best) {
            best = cost;
            a.zc = zc;
            a.tz = (int)tz;
            a.items = items;
        }
    }
    const unsigned row = (unsigned)a.ck * 2;
    a.tile_tx = (unsigned)(WT_X * HT_Y) * row;
    a.tile_bytes = round1024(a.tile_tx);
    a.ring_tx = 3u * (unsigned)a.nc * row;
    a.ring_bytes = round1024(a.ring_tx);
    const int slots = (int)((215u * 1024u - WD_RING * a.ring_bytes) / a.tile_bytes);
    a.slots = slots < WD_SLOTS ? slots : WD_SLOTS;
    if (a.slots < a.ncb) return PF_E_INVALID;
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(UM >> 4) << 24);
    // K-major, swizzled with the span of a row; stride between 8-row groups: one tile row of 18 cells, 8 weight rows
    const unsigned long long base = (1ULL << 16) | (1ULL << 46) | (umma_layout(a.ck) << 61);
    a.a_hi = base | ((unsigned long long)(WT_X * row >> 4) << 32);
    a.b_hi = base | ((unsigned long long)(8 * row >> 4) << 32);
    a.bias = bias;
    a.y = (bf16*)y_bf16;
    a.yf = y_f32;
    a.ldy = ldy;
    a.yoff = yoff;
    alignas(64) CUtensorMap mA, mB;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    {
        const cuuint64_t dims[5] = {(cuuint64_t)cin, (cuuint64_t)wd, (cuuint64_t)h, (cuuint64_t)d, (cuuint64_t)n};
        const cuuint64_t r = (cuuint64_t)ldx * 2;
        const cuuint64_t strides[4] = {r, r * wd, r * wd * h, r * wd * h * d};
        const cuuint32_t box[5] = {(cuuint32_t)a.ck, (cuuint32_t)WT_X, (cuuint32_t)HT_Y, 1, 1};
        if (enc(&mA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)((const bf16*)x + xoff), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, tma_swizzle(a.ck), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PF_E_INVALID;
    }
    {
        // [dz][l][cout][cin]: one box is the three taps dz of a lateral offset
        const cuuint64_t r = (cuuint64_t)cin * 2;
        const cuuint64_t dims[4] = {(cuuint64_t)cin, (cuuint64_t)cout, 9, 3};
        const cuuint64_t strides[3] = {r, r * cout, r * cout * 9};
        const cuuint32_t box[4] = {(cuuint32_t)a.ck, (cuuint32_t)a.nc, 1, 3};
        if (enc(&mB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(w), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, tma_swizzle(a.ck), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PF_E_INVALID;
    }
    const size_t smem = 1024 + (size_t)a.slots * a.tile_bytes + (size_t)WD_RING * a.ring_bytes;
    static std::once_flag attr_once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(attr_once, [] {
        for (auto f : {k_conv_wide<32, false>, k_conv_wide<64, false>, k_conv_wide<32, true>, k_conv_wide<64, true>}) {
            const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 216 * 1024);
            if (e != cudaSuccess) attr_err = e;
        }
    });
    if (attr_err != cudaSuccess || smem > 216u * 1024u) return PF_E_CUDA;
    auto k = a.ck == 32 ? (flip ? k_conv_wide<32, true> : k_conv_wide<32, false>)
                        : (flip ? k_conv_wide<64, true> : k_conv_wide<64, false>);
    k<<<(unsigned)std::min<long long>(a.items, 152), MR_THR, smem, stream>>>(mA, mB, a);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

// Division of a weight gradient's taps and channels over blocks.  Blocks of 32 input channels with dy along M (12 of 16 core
// matrices used); a last block of 16 reads zeros beyond.  (64 channels unstacked fill M = 64, at half the rate, in nine blocks for
// 64 output channels: 64 -> 64 channels on 4 x 64^3 voxels 689 us, now 360; 192 -> 128 on 2 x 33^3 392 and 215; 128 -> 128 on
// 4 x 64^3 1352 and 1083; 48 -> 32 on 50^3 in blocks of 16 105 and 73.)  128 channels unstacked with up to 32 output channels, whose
// taps dy share a block (128 -> 32 on 4 x 64^3 468 us, stacked 640).  A block takes every dz (each X plane loaded once) while
// its accumulators fit 512 TMEM columns, else one dz (dY loaded three times).
void wgrad_plan(WgArgs& a) {
    a.stacked = !(a.cin % 128 == 0 && a.cout <= 32);
    a.cb = !a.stacked ? 128 : (a.cin == 16 ? 16 : 32);
    a.nchunk = a.cb / 8;
    a.m64 = a.cb == 16;
    const int per_dz = (a.stacked ? 3 : 9) * a.cout;
    a.ndz = 3 * per_dz <= 512 ? 3 : 1;
    const int cols = a.ndz * per_dz;
    a.tmem_cols = cols <= 64 ? 64 : (cols <= 128 ? 128 : (cols <= 256 ? 256 : 512));
}

// The grid's axes in the order of the kernel's x (tiles of 8 cells), y (16) and z (marched along).  Neither operand is read along
// rows (a cell's 8 channels are a 16-byte piece), so any order loads as fast, and grids a few cells wide fill tiles laid
// along their long axes: taken where it leaves less than three quarters of the tile planes (128 -> 128 channels on 2000 x 2 x 2
// voxels 94 us, 244 in their own order).  Samples follow one another along the grid's z, so with several of them only x and y change places.
struct WgAxis {
    int n, tap;
    long long stride;  // voxels
};
struct WgAxes {
    WgAxis a[3];
};
WgAxes wgrad_axes(int n, int d, int h, int wd) {
    const WgAxis X{wd, 1, 1}, Y{h, 3, wd}, Z{d, 9, (long long)wd * h};
    const auto planes = [](const WgAxes& q) {
        return (double)((q.a[0].n + 7) / 8) * ((q.a[1].n + 15) / 16) * (q.a[2].n + 2.0);
    };
    const WgAxes own{{X, Y, Z}};
    WgAxes best = own;
    for (const WgAxes& q : {WgAxes{{Y, X, Z}}, WgAxes{{X, Z, Y}}, WgAxes{{Z, X, Y}}, WgAxes{{Y, Z, X}}, WgAxes{{Z, Y, X}}}) {
        if (n > 1 && q.a[2].tap != 9) continue;
        if (planes(q) < planes(best)) best = q;
    }
    return planes(best) < 0.75 * planes(own) ? best : own;
}

pf_status wgrad(const void* dy, int lddy, int dyoff, int cout, const void* x, int ldx, int xoff, int cin, float* dw, int n,
                int d, int h, int wd, cudaStream_t st) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return PF_E_CUDA;
    WgArgs a{};
    a.cin = cin;
    a.cout = cout;
    const WgAxes axes = wgrad_axes(n, d, h, wd);
    const WgAxis &ax = axes.a[0], &ay = axes.a[1], &az = axes.a[2];
    a.W = ax.n;
    a.H = ay.n;
    a.D = az.n;
    a.tapx = ax.tap;
    a.tapy = ay.tap;
    a.tapz = az.tap;
    a.tries = WAIT_TRIES;
    a.dw = dw;
    wgrad_plan(a);
    a.tx = (a.W + 7) / 8;
    a.ty = (a.H + 15) / 16;
    a.x_tx = 18u * (unsigned)a.nchunk * WX_ROW;
    a.dy_tx = 16u * 8u * 2u * (unsigned)cout;
    a.x_bytes = (a.x_tx + 127u) & ~127u;
    a.slot_bytes = (a.x_bytes + a.dy_tx + 127u) & ~127u;
    // the unused core matrices of a stacked A operand reach one row past a plane: at least 4 KB follow the slots
    const unsigned slack = 4096;
    // (with up to 256 TMEM columns the slots of two blocks share the 228 KB of a multiprocessor)
    const int want = a.ndz == 3 ? 6 : 4;
    int slots = (int)(((a.ndz == 1 && a.tmem_cols <= 256 ? 108u : 200u) * 1024u - slack) / a.slot_bytes);
    a.slots = slots < want ? slots : want;
    const size_t smem = 1024 + (size_t)a.slots * a.slot_bytes + slack;
    // MN-major, no swizzle (bits 15, 16 of the instruction descriptor = 1): leading offset = stride between
    // 8-voxel groups of K, stride offset = stride between 8-channel groups of M or N
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((unsigned)(cout >> 3) << 17) |
              ((unsigned)((a.m64 ? 64 : 128) >> 4) << 24);
    a.a_hi = desc_plain(0, (unsigned)a.nchunk * WX_ROW, WX_ROW);
    a.b_hi = desc_plain(0, 128u, 16u * 128u);
    const int groups = (3 / a.ndz) * ((cin + a.cb - 1) / a.cb);
    // about one wave: resident blocks by shared memory (228 KB per SM) and TMEM columns (512)
    int occ = (int)(228u * 1024u / (smem + 2048));
    if (occ > 512 / a.tmem_cols) occ = 512 / a.tmem_cols;
    if (occ < 1) occ = 1;
    // z chunks: the fewest (waves + blocks a multiprocessor takes, which share its loads and atomics) x (planes + about four for
    // the prologue, the extra X planes and the epilogue)
    const long long columns = (long long)a.tx * a.ty * n * groups, cap = 152LL * occ;
    long long best = -1;
    for (int nz = 1; nz <= a.D; nz += 1 + nz / 64) {
        const int zc = (a.D + nz - 1) / nz, chunks = (a.D + zc - 1) / zc;
        const long long blocks = columns * chunks, cost = ((blocks + cap - 1) / cap + (blocks + 151) / 152) * (zc + 4);
        if (best < 0 || cost < best) {
            best = cost;
            a.zc = zc;
            a.nzc = chunks;
        }
    }
    alignas(64) CUtensorMap mX, mY;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    {
        const cuuint64_t row = (cuuint64_t)ldx * 2;
        const cuuint64_t dims[5] = {8, (cuuint64_t)a.W, (cuuint64_t)(cin / 8), (cuuint64_t)a.H, (cuuint64_t)n * a.D};
        const cuuint64_t strides[4] = {row * ax.stride, 16, row * ay.stride, row * az.stride};
        const cuuint32_t box[5] = {8, 10, (cuuint32_t)a.nchunk, 18, 1};
        if (enc(&mX, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)((const bf16*)x + xoff), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PF_E_INVALID;
    }
    {
        const cuuint64_t row = (cuuint64_t)lddy * 2;
        const cuuint64_t dims[5] = {8, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)(cout / 8), (cuuint64_t)n * a.D};
        const cuuint64_t strides[4] = {row * ax.stride, row * ay.stride, 16, row * az.stride};
        const cuuint32_t box[5] = {8, 8, 16, (cuuint32_t)(cout / 8), 1};
        if (enc(&mY, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)((const bf16*)dy + dyoff), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PF_E_INVALID;
    }
    static std::once_flag wg_once;
    static cudaError_t wg_err = cudaSuccess;
    std::call_once(wg_once, [] {
        wg_err = cudaFuncSetAttribute(k_wgrad_umma, cudaFuncAttributeMaxDynamicSharedMemorySize, 202 * 1024);
    });
    if (wg_err != cudaSuccess) return PF_E_CUDA;
    const long long bx = (long long)a.tx * a.ty * a.nzc * n;
    if (bx > 0x7FFFFFFFLL) return PF_E_RANGE;
    k_wgrad_umma<<<dim3((unsigned)bx, (unsigned)groups), UTHR, smem, st>>>(mX, mY, a);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

}  // namespace

extern "C" {

pf_status pfnn_conv3d(const void* x, int ldx, int xoff, const void* w, int cin, int cout, const float* bias, int relu,
                      int flip, void* y_bf16, float* y_f32, int ldy, int yoff, int accumulate, int n, int d, int h,
                      int wd, void* stream) {
    if (!x || !w || (!y_bf16 && !y_f32) || n < 1 || d < 1 || h < 1 || wd < 1) return PF_E_INVALID;
    if (cin < 16 || cin % 16 || cout < 16 || cout % 16 || cout > 256 || ldx % 8 || xoff % 8 || ldx < xoff + cin ||
        ldy % 8 || yoff % 8 || ldy < yoff + cout)
        return PF_E_INVALID;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(y_bf16) |
         reinterpret_cast<uintptr_t>(y_f32)) % 16)
        return PF_E_INVALID;
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return PF_E_CUDA;
    if (march_shape(cin, cout, d, h, wd))
        return conv_march(x, ldx, xoff, w, cin, cout, bias, relu, flip, y_bf16, y_f32, ldy, yoff, accumulate, n, d, h,
                         wd, (cudaStream_t)stream, enc);

    if (wide_shape(cin, cout, n, d, h, wd))
        return conv_wide(x, ldx, xoff, w, cin, cout, bias, relu, flip, y_bf16, y_f32, ldy, yoff, accumulate, n, d, h,
                         wd, (cudaStream_t)stream, enc);

    UmmaArgs a{};
    a.cin = cin;
    a.cout = cout;
    a.ck = cin % 64 == 0 ? 64 : (cin % 32 == 0 ? 32 : 16);
    a.nkb = cin / a.ck;
    const UmmaBricks bricks = umma_bricks(d, h, wd);
    a.wb = bricks.wb;
    a.hb = bricks.hb;
    a.db = bricks.db;
    a.D = d;
    a.H = h;
    a.W = wd;
    a.tx = (int)bricks.tx;
    a.ty = (int)bricks.ty;
    a.tz = (int)bricks.tz;
    a.flip = flip;
    a.relu = relu;
    a.withhold = g_test_withhold;
    a.tries = g_test_tries > 0 ? g_test_tries : WAIT_TRIES;
    g_test_withhold = -1;
    g_test_tries = 0;
    a.accumulate = accumulate;
    a.a_bytes = round1024((unsigned)(UM * a.ck * 2));
    a.stage_bytes = a.a_bytes + round1024((unsigned)(cout * a.ck * 2));
    a.tx_bytes = (unsigned)((UM + cout) * a.ck * 2);
    int stages = (int)(98304u / a.stage_bytes);
    a.stages = stages < 2 ? 2 : (stages > 8 ? 8 : stages);
    // instruction descriptor, kind::f16: D f32 (bits 4-5 = 1), A and B bf16 (bits 7-9, 10-12 = 1),
    // both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(cout >> 3) << 17) | ((unsigned)(UM >> 4) << 24);
    // descriptor: leading offset 16 B (unused for swizzled K-major), stride between 8-row groups = 8 rows x
    // row bytes, version 1 (bit 46), swizzle layout code at bits 61-63
    const unsigned long long sbo = (unsigned long long)(8 * a.ck * 2);
    a.desc_hi = (1ULL << 16) | ((sbo >> 4) << 32) | (1ULL << 46) | (umma_layout(a.ck) << 61);
    a.tmem_cols = cout <= 32 ? 32 : (cout <= 64 ? 64 : (cout <= 128 ? 128 : 256));
    a.bias = bias;
    a.y = (bf16*)y_bf16;
    a.yf = y_f32;
    a.ldy = ldy;
    a.yoff = yoff;

    alignas(64) CUtensorMap mA, mB;
    {
        const cuuint64_t dims[5] = {(cuuint64_t)cin, (cuuint64_t)wd, (cuuint64_t)h, (cuuint64_t)d, (cuuint64_t)n};
        const cuuint64_t row = (cuuint64_t)ldx * 2;
        const cuuint64_t strides[4] = {row, row * wd, row * wd * h, row * wd * h * d};
        const cuuint32_t box[5] = {(cuuint32_t)a.ck, (cuuint32_t)a.wb, (cuuint32_t)a.hb, (cuuint32_t)a.db, 1};
        const cuuint32_t es[5] = {1, 1, 1, 1, 1};
        if (enc(&mA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)((const bf16*)x + xoff), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, tma_swizzle(a.ck), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PF_E_INVALID;
    }
    {
        const cuuint64_t dims[2] = {(cuuint64_t)cin, (cuuint64_t)(27 * cout)};
        const cuuint64_t strides[1] = {(cuuint64_t)cin * 2};
        const cuuint32_t box[2] = {(cuuint32_t)a.ck, (cuuint32_t)cout};
        const cuuint32_t es[2] = {1, 1};
        if (enc(&mB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(w), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, tma_swizzle(a.ck), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PF_E_INVALID;
    }
    const size_t smem = (size_t)a.stages * a.stage_bytes + 1024 + 16 * a.stages + 16;
    static std::once_flag attr_once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(attr_once, [] {
        attr_err = cudaFuncSetAttribute(k_conv_umma, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024 + 2048);
    });
    if (attr_err != cudaSuccess) return PF_E_CUDA;
    const long long blocks = (long long)a.tx * a.ty * a.tz * n;
    if (blocks > 0x7FFFFFFFLL) return PF_E_RANGE;
    k_conv_umma<<<(unsigned)blocks, UTHR, smem, (cudaStream_t)stream>>>(mA, mB, a);
    pfgb::count_launch();
    return cudaGetLastError() == cudaSuccess ? PF_OK : PF_E_CUDA;
}

// (more than the compact copies of both operands that pfnn_conv3d_wgrad may need: 2 (cout + cin) bytes a voxel)
long long pfnn_conv3d_wgrad_work_bytes(int cout, int cin, int n, int d, int h, int wd) {
    if (cout < 1 || cin < 1 || n < 1 || d < 1 || h < 1 || wd < 1) return -1;
    const long long vp = (long long)n * (d + 2) * (h + 2) * ((wd + 2 + 7) / 8 * 8);
    return 2LL * (3LL * cout + cin) * ((vp + 63) / 64 * 64);
}

pf_status pfnn_conv3d_wgrad(const void* dy, int lddy, int dyoff, int cout, const void* x, int ldx, int xoff, int cin,
                            float* dw, int n, int d, int h, int wd, void* work, long long work_bytes, void* stream) {
    if (!dy || !x || !dw || !work || n < 1 || d < 1 || h < 1 || wd < 1) return PF_E_INVALID;
    if ((cout != 16 && cout != 32 && cout != 64 && cout != 128) || cin < 16 || cin % 16 || cin > 256 ||
        lddy < dyoff + cout || ldx < xoff + cin || dyoff < 0 || xoff < 0)
        return PF_E_INVALID;
    if (work_bytes < pfnn_conv3d_wgrad_work_bytes(cout, cin, n, d, h, wd) || reinterpret_cast<uintptr_t>(work) % 16)
        return PF_E_INVALID;
    cudaStream_t st = (cudaStream_t)stream;
    // TMA reads rows that start on 16 bytes; other slices are copied to the scratch first
    const long long nvox = (long long)n * d * h * wd;
    bf16* scratch = (bf16*)work;
    auto aligned = [&](const void*& q, int& ld, int& off, int c) {
        if (ld % 8 == 0 && off % 8 == 0 && reinterpret_cast<uintptr_t>(q) % 16 == 0) return;
        long long blocks = (nvox * c + 255) / 256;
        if (blocks > 152LL * 32) blocks = 152LL * 32;
        k_compact<<<(unsigned)blocks, 256, 0, st>>>((const bf16*)q, ld, off, c, nvox * c, scratch);
        pfgb::count_launch();
        q = scratch;
        ld = c;
        off = 0;
        scratch += nvox * c;  // c is a multiple of 16: the next copy starts on 32 bytes
    };
    aligned(dy, lddy, dyoff, cout);
    aligned(x, ldx, xoff, cin);
    return wgrad(dy, lddy, dyoff, cout, x, ldx, xoff, cin, dw, n, d, h, wd, st);
}

pf_status pfnn_status(int* failed) {
    if (!failed) return PF_E_INVALID;
    int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_umma_status, sizeof(int)) != cudaSuccess) return PF_E_CUDA;
    if (v && cudaMemcpyToSymbol(g_umma_status, &zero, sizeof(int)) != cudaSuccess) return PF_E_CUDA;
    *failed = v;
    return v ? PF_E_TIMEOUT : PF_OK;
}

pf_status pfnn_test_withhold_stage(int stage, long long tries) {
    if (stage < 0 || tries < 1 || tries > WAIT_TRIES) return PF_E_INVALID;
    g_test_withhold = stage;
    g_test_tries = tries;
    return PF_OK;
}

}  // extern "C"

namespace pfgb {

pf_status nn_wgrad(const void* dy, int cout, const void* x, int ldx, int xoff, int cin, float* dw, int n, int d, int h,
                   int wd, void* stream) {
    return wgrad(dy, cout, 0, cout, x, ldx, xoff, cin, dw, n, d, h, wd, (cudaStream_t)stream);
}

}  // namespace pfgb
