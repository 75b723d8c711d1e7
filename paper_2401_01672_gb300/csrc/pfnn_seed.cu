// Warm-start constraint from the micro-scale model: it has no nucleation term, so ice can only exist
// where it grew from the seed through the pore space (Sec. 2.4: constant supercooling, the phase field
// of every ice region is connected to the initial ice).  The network's prediction is kept only in the
// predicted-ice region that is connected to the seed (and within `halo` cells of it, which keeps the
// diffuse interface profile), and never below the seed's own phase field; everywhere else, and in the
// cells whose water indicator is zero (they never change, eq. water-indicator), the initial phase field
// is kept.
//
// The predicted-ice mask is first eroded by `erode` cells (so that throats narrower than about twice
// that are cut: behind them the prediction may hold ice the seed does not reach through the throat, a
// different equilibrium of the same equations), the connected region is found by flood fill through the
// eroded mask: reached = seed, then repeatedly reached |= mask & (a face neighbour is reached), in place
// (the flags only go from 0 to 1, so the order in which threads see each other's updates changes only how
// many sweeps it takes), until a sweep changes nothing; it is then grown back by `erode` cells inside the
// original mask and by `halo` cells without it.
#include "../../include/pfnn.h"
#include "pf_internal.cuh"

#include <cuda_runtime.h>

namespace {

constexpr int SF_THREADS = 256;
constexpr int SWEEPS_PER_CHECK = 16;

int sf_blocks(long long n) {
    long long b = (n + SF_THREADS - 1) / SF_THREADS;
    if (b > 152LL * 16) b = 152LL * 16;
    return (int)(b < 1 ? 1 : b);
}

// flags: bit 0 = may carry ice (eroded), bit 1 = reached, bit 2 = marked in the current growth sweep,
// bit 3 = predicted ice (predicted phi > 1/2 and a water indicator above zero), bit 4 = marked for erosion
__global__ void k_sf_init(const float* __restrict__ prob, const double* __restrict__ seed, const double* __restrict__ G,
                          double zeta, long long n, unsigned char* __restrict__ fl) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const bool water = 1.0 - zeta * G[q] > 0.0;
        const bool ice = prob[q] > 0.5f && water;
        fl[q] = (unsigned char)((ice ? 9 : 0) | (seed[q] > 0.5 ? 2 : 0));
    }
}

// one erosion sweep: a cell of the mask with a face neighbour outside it (inside the grid) leaves it
__global__ void k_sf_erode(unsigned char* fl, int n1, int n2, int n3) {
    const long long plane = (long long)n1 * n2, n = plane * n3;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        if (!(fl[q] & 1)) continue;
        const int i = (int)(q % n1), j = (int)((q / n1) % n2), k = (int)(q / plane);
        const bool edge = (i > 0 && !(fl[q - 1] & 1)) || (i < n1 - 1 && !(fl[q + 1] & 1)) ||
                          (j > 0 && !(fl[q - n1] & 1)) || (j < n2 - 1 && !(fl[q + n1] & 1)) ||
                          (k > 0 && !(fl[q - plane] & 1)) || (k < n3 - 1 && !(fl[q + plane] & 1));
        if (edge) fl[q] |= 16;
    }
}

__global__ void k_sf_erode_commit(unsigned char* fl, long long n) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        if (fl[q] & 16) fl[q] = (unsigned char)(fl[q] & ~17);
}

__device__ __forceinline__ bool any_reached(const unsigned char* fl, long long q, int i, int j, int k, int n1, int n2,
                                            int n3, long long plane) {
    return (i > 0 && (fl[q - 1] & 2)) || (i < n1 - 1 && (fl[q + 1] & 2)) || (j > 0 && (fl[q - n1] & 2)) ||
           (j < n2 - 1 && (fl[q + n1] & 2)) || (k > 0 && (fl[q - plane] & 2)) || (k < n3 - 1 && (fl[q + plane] & 2));
}

// one flood-fill sweep (grow = 0: only through cells that may carry ice), one dilation sweep inside the
// predicted ice (grow = 2) or one dilation sweep everywhere (grow = 1)
__global__ void k_sf_sweep(unsigned char* fl, int n1, int n2, int n3, int grow, int* changed) {
    const long long plane = (long long)n1 * n2, n = plane * n3;
    int local = 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const unsigned char f = ((volatile unsigned char*)fl)[q];
        if ((f & 2) || (grow == 0 && !(f & 1)) || (grow == 2 && !(f & 8))) continue;
        const int i = (int)(q % n1), j = (int)((q / n1) % n2), k = (int)(q / plane);
        if (any_reached(fl, q, i, j, k, n1, n2, n3, plane)) {
            ((volatile unsigned char*)fl)[q] = (unsigned char)(f | (grow ? 4 : 2));
            local = 1;
        }
    }
    if (local) atomicOr(changed, 1);
}

// dilation marks (bit 2) become reached (bit 1) between dilation sweeps, so each sweep grows one cell
__global__ void k_sf_commit(unsigned char* fl, long long n) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        if (fl[q] & 4) fl[q] = (unsigned char)((fl[q] & ~4) | 2);
}

__global__ void k_sf_apply(const float* __restrict__ prob, const double* __restrict__ seed, const double* __restrict__ G,
                           double zeta, long long n, const unsigned char* __restrict__ fl, double* __restrict__ out) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const bool water = 1.0 - zeta * G[q] > 0.0;
        const double p = fminf(fmaxf(prob[q], 0.f), 1.f);
        // the seed itself stays ice where the prediction has less
        out[q] = (water && (fl[q] & 2)) ? fmax(p, seed[q]) : seed[q];
    }
}

// ---- Bit form: one bit per cell, 32 cells of a row to a word, so a mask of 256^3 cells is 2 MB and stays in L2.
// The byte form above swept 16.8 MB of flags from global memory once per cell of path length (10.1 ms for a 256^3 packing);
// here a block brings a tile of words to its own fixed point in shared memory before the next sweep, a word is filled
// along x by one carry, and the water indicator is kept as a mask, so G is read once: 0.51 ms (0.68 with tiles of 16
// planes, two barriers around every pass and a visit to every tile in every sweep).
struct BitGrid {
    int n1, n2, n3, W;  // W words per row
    unsigned tail;      // cells of a row's last word
};

__device__ __forceinline__ unsigned valid_bits(const BitGrid& g, int wx) { return wx == g.W - 1 ? g.tail : 0xffffffffu; }

// Masks of predicted ice, reached (seed) and water; a warp takes a row, WPI words at a time, so that 3 WPI loads per lane
// are in flight and no cell index is divided (20 bytes a cell; 102 us at 256^3, 3.3 TB/s).
constexpr int WPI = 4;
__global__ void __launch_bounds__(SF_THREADS) k_sb_init(const float* __restrict__ prob, const double* __restrict__ seed,
                                                        const double* __restrict__ G, double zeta, const BitGrid g,
                                                        unsigned* __restrict__ ice, unsigned* __restrict__ reached,
                                                        unsigned* __restrict__ water) {
    const int lane = threadIdx.x & 31;
    const int rows = g.n2 * g.n3, step = gridDim.x * (SF_THREADS / 32);
    for (int row = blockIdx.x * (SF_THREADS / 32) + (threadIdx.x >> 5); row < rows; row += step)
    for (int wx = 0; wx < g.W; wx += WPI) {
        const long long w0 = (long long)row * g.W + wx;
        float p[WPI];
        double s[WPI], gl[WPI];
        bool in[WPI];
#pragma unroll
        for (int r = 0; r < WPI; ++r) {
            const int x = (wx + r) * 32 + lane;
            in[r] = x < g.n1;
            const long long q = (long long)row * g.n1 + x;
            p[r] = in[r] ? prob[q] : 0.f;
            s[r] = in[r] ? seed[q] : 0.0;
            gl[r] = in[r] ? G[q] : 0.0;
        }
#pragma unroll
        for (int r = 0; r < WPI; ++r) {
            const bool wat = in[r] && 1.0 - zeta * gl[r] > 0.0;
            const unsigned bw = __ballot_sync(0xffffffffu, wat);
            const unsigned bi = __ballot_sync(0xffffffffu, wat && p[r] > 0.5f);
            const unsigned br = __ballot_sync(0xffffffffu, in[r] && s[r] > 0.5);
            if (lane == 0 && wx + r < g.W) {
                ice[w0 + r] = bi;
                reached[w0 + r] = br;
                water[w0 + r] = bw;
            }
        }
    }
}

// The six face neighbours of every cell of word (wx, j, k), ORed; cells outside the grid count as `out` (0 or ~0).
// With ERODE the masks are ANDed instead (pass out = ~0).
template <bool ERODE>
__device__ __forceinline__ unsigned face_neighbours(const unsigned* __restrict__ m, const BitGrid& g, int wx, int j, int k,
                                                    long long w, unsigned own) {
    const long long pl = (long long)g.W * g.n2;
    const unsigned out = ERODE ? 0xffffffffu : 0u;
    const unsigned lw = wx > 0 ? m[w - 1] : out, rw = wx < g.W - 1 ? m[w + 1] : out;
    // the cell behind the row's last one is outside the grid
    const unsigned o = ERODE ? own | ~valid_bits(g, wx) : own;
    const unsigned l = (o << 1) | (lw >> 31), r = (o >> 1) | (rw << 31);
    const unsigned a = j > 0 ? m[w - g.W] : out, b = j < g.n2 - 1 ? m[w + g.W] : out;
    const unsigned c = k > 0 ? m[w - pl] : out, d = k < g.n3 - 1 ? m[w + pl] : out;
    return ERODE ? (l & r & a & b & c & d) : (l | r | a | b | c | d);
}

// one erosion or dilation step from `in` to `to` (erosion: a cell with a face neighbour outside the mask leaves it;
// dilation: face neighbours join, inside `within` if that is given)
template <bool ERODE>
__global__ void __launch_bounds__(SF_THREADS) k_sb_step(const unsigned* __restrict__ in, unsigned* __restrict__ to,
                                                        const unsigned* __restrict__ within, const BitGrid g) {
    const long long words = (long long)g.W * g.n2 * g.n3;
    for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < words; w += (long long)gridDim.x * blockDim.x) {
        const long long row = w / g.W;
        const int wx = (int)(w - row * g.W), j = (int)(row % g.n2), k = (int)(row / g.n2);
        const unsigned own = in[w], nb = face_neighbours<ERODE>(in, g, wx, j, k, w, own);
        if constexpr (ERODE) to[w] = own & nb;
        else to[w] = own | (nb & (within ? within[w] : valid_bits(g, wx)));
    }
}

// bits of `m` connected along the word to a bit of s (s within m): adding s to m carries from each seed through the ones
// above it, so the bits the sum cleared are the run from the lowest seed up; the other direction on the reversed word
__device__ __forceinline__ unsigned fill_up(unsigned m, unsigned s) { return s | (m & ~(m + s)); }
__device__ __forceinline__ unsigned fill_word(unsigned m, unsigned s) {
    const unsigned u = fill_up(m, s);
    return __brev(fill_up(__brev(m), __brev(u)));
}

// One flood-fill sweep: a block loads a tile of TW x TY x TZ words with a one-word halo and fills it until nothing changes
// (the halo stays as loaded; masks only gain bits, so a word a neighbour block is about to extend is caught by the next
// sweep).  Only tiles with a face neighbour that the sweep before changed can change (all in the first sweep): tiles note a
// change in stamp, as the number of the sweep modulo 251 plus one, so nothing has to be cleared between sweeps (a note 251
// sweeps old reads as new, which costs a visit).  Sweep r sets flag r & 3 when it changed something, reads that of the sweep before
// (nothing changed then: the fixed point is reached, exit) and clears the next one's.
constexpr int SB_TW = 2, SB_TY = 16, SB_TZ = 32, SB_THREADS = SB_TW * SB_TY * SB_TZ / 2;
__global__ void __launch_bounds__(SB_THREADS) k_sb_flood(const unsigned* __restrict__ mask, unsigned* reached,
                                                                  const BitGrid g, int* flags, unsigned char* stamp,
                                                                  long long sweep) {
    __shared__ unsigned t[SB_TZ + 2][SB_TY + 2][SB_TW + 2];
    const int r = (int)(sweep & 3);
    if (blockIdx.x == 0 && threadIdx.x == 0) flags[(r + 1) & 3] = 0;
    if (((volatile int*)flags)[(r + 3) & 3] == 0) return;  // uniform over the grid: written by earlier launches only
    const int nbx = (g.W + SB_TW - 1) / SB_TW, nby = (g.n2 + SB_TY - 1) / SB_TY;
    const int bx = blockIdx.x % nbx, by = (blockIdx.x / nbx) % nby, bz = blockIdx.x / (nbx * nby);
    if (sweep > 0) {
        const int nbz = (g.n3 + SB_TZ - 1) / SB_TZ;
        const unsigned char last = (unsigned char)((sweep - 1) % 251 + 1);
        auto changed = [&](int dx, int dy, int dz) {
            const int x = bx + dx, y = by + dy, z = bz + dz;
            return x >= 0 && x < nbx && y >= 0 && y < nby && z >= 0 && z < nbz &&
                   ((volatile unsigned char*)stamp)[((long long)z * nby + y) * nbx + x] == last;
        };
        // (a neighbour's note of this very sweep may hide that of the last one: the tile is then visited in the next)
        bool any = false;
        if (threadIdx.x < 6) {
            const int s = threadIdx.x & 1 ? 1 : -1, a = threadIdx.x >> 1;
            any = changed(a == 0 ? s : 0, a == 1 ? s : 0, a == 2 ? s : 0);
        }
        if (!__syncthreads_or(any)) return;
    }
    const int x0 = bx * SB_TW - 1, y0 = by * SB_TY - 1, z0 = bz * SB_TZ - 1;
    constexpr int CELLS = (SB_TZ + 2) * (SB_TY + 2) * (SB_TW + 2), HALF = SB_TZ / 2;
    for (int q = threadIdx.x; q < CELLS; q += SB_THREADS) {
        const int lx = q % (SB_TW + 2), ly = (q / (SB_TW + 2)) % (SB_TY + 2), lz = q / ((SB_TW + 2) * (SB_TY + 2));
        const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
        const bool in = x >= 0 && x < g.W && y >= 0 && y < g.n2 && z >= 0 && z < g.n3;
        t[lz][ly][lx] = in ? ((volatile unsigned*)reached)[((long long)z * g.n2 + y) * g.W + x] : 0u;
    }
    // a thread owns two words, HALF planes apart
    const int lx = threadIdx.x % SB_TW + 1, ly = (threadIdx.x / SB_TW) % SB_TY + 1, lz = threadIdx.x / (SB_TW * SB_TY) + 1;
    const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
    const bool in[2] = {x < g.W && y < g.n2 && z < g.n3, x < g.W && y < g.n2 && z + HALF < g.n3};
    const long long w[2] = {((long long)z * g.n2 + y) * g.W + x, ((long long)(z + HALF) * g.n2 + y) * g.W + x};
    const unsigned m[2] = {in[0] ? mask[w[0]] : 0u, in[1] ? mask[w[1]] : 0u};
    __syncthreads();
    const unsigned first[2] = {t[lz][ly][lx], t[lz + HALF][ly][lx]};
    unsigned own[2] = {first[0], first[1]};
    // Rounds of PASSES passes without a barrier: threads see each other's words in any order, but words only gain bits, so a
    // round in which no word of the block changed ends at the fixed point.  Every round but the last reaches at least one
    // more cell of the tile.
    constexpr int PASSES = 6;
    volatile unsigned(*v)[SB_TY + 2][SB_TW + 2] = t;
    for (int it = 0; it <= 64 * SB_THREADS; ++it) {
        int ch = 0;
#pragma unroll 1
        for (int q = 0; q < PASSES; ++q) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = lz + h * HALF;
                const unsigned nb = (own[h] << 1) | (own[h] >> 1) | (v[k][ly][lx - 1] >> 31) | (v[k][ly][lx + 1] << 31) |
                                    v[k][ly - 1][lx] | v[k][ly + 1][lx] | v[k - 1][ly][lx] | v[k + 1][ly][lx] | own[h];
                const unsigned f = own[h] | fill_word(m[h], nb & m[h]);
                if (f != own[h]) {
                    v[k][ly][lx] = own[h] = f;
                    ch = 1;
                }
            }
        }
        if (!__syncthreads_or(ch)) break;
    }
    for (int h = 0; h < 2; ++h)
        if (in[h] && own[h] != first[h]) {
            reached[w[h]] = own[h];
            flags[r] = 1;  // every writer stores the same value, also in the note
            stamp[blockIdx.x] = (unsigned char)(sweep % 251 + 1);
        }
}

__global__ void __launch_bounds__(SF_THREADS) k_sb_apply(const float* __restrict__ prob, const double* seed,
                                                         const unsigned* __restrict__ reached,
                                                         const unsigned* __restrict__ water, const BitGrid g, double* out) {
    const int lane = threadIdx.x & 31;
    const int rows = g.n2 * g.n3, step = gridDim.x * (SF_THREADS / 32);
    for (int row = blockIdx.x * (SF_THREADS / 32) + (threadIdx.x >> 5); row < rows; row += step)
    for (int wx = 0; wx < g.W; wx += WPI) {
        const long long w0 = (long long)row * g.W + wx;
        float p[WPI];
        double s[WPI];
        long long q[WPI];
        bool in[WPI], put[WPI];
#pragma unroll
        for (int r = 0; r < WPI; ++r) {
            const int x = (wx + r) * 32 + lane;
            in[r] = x < g.n1;
            put[r] = in[r] && ((reached[w0 + r] & water[w0 + r]) >> lane & 1u);
            q[r] = (long long)row * g.n1 + x;
            s[r] = in[r] ? seed[q[r]] : 0.0;
            p[r] = put[r] ? prob[q[r]] : 0.f;
        }
#pragma unroll
        for (int r = 0; r < WPI; ++r)
            // the seed itself stays ice where the prediction has less
            if (in[r]) out[q[r]] = put[r] ? fmax((double)fminf(fmaxf(p[r], 0.f), 1.f), s[r]) : s[r];
    }
}

}  // namespace

extern "C" pf_status pfnn_seed_connect(const float* prob, const double* phi_seed, const double* G, int n1, int n2,
                                       int n3, double zeta, int erode, int halo, unsigned char* work, double* phi_out,
                                       void* stream, long long* sweeps) {
    if (!prob || !phi_seed || !G || !work || !phi_out || n1 < 1 || n2 < 1 || n3 < 1 || halo < 0 || halo > 64 ||
        erode < 0 || erode > 64 || !(zeta >= 0.0))
        return PF_E_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    const long long n = (long long)n1 * n2 * n3;
    {
        // Bit form: masks of ice (eroded in place of the original), reached, a second buffer for the steps, water and, with
        // erosion, the original ice, and four flags.  The scratch (one byte a cell) holds them but for rows of up to 16
        // cells (up to 20 and 33 to 40 with erosion) and grids of a few cells, which take the byte form.
        BitGrid g{n1, n2, n3, (n1 + 31) / 32, n1 % 32 ? (1u << (n1 % 32)) - 1u : 0xffffffffu};
        const long long words = (long long)g.W * n2 * n3;
        const int masks = erode ? 5 : 4;
        const long long tiles = ((g.W + SB_TW - 1) / SB_TW) * (long long)((n2 + SB_TY - 1) / SB_TY) * ((n3 + SB_TZ - 1) / SB_TZ);
        if (4 * masks * words + 16 + tiles <= 16 * ((n + 15) / 16) + 4 && words < (1LL << 30)) {
            int* flags = reinterpret_cast<int*>(work);
            unsigned* ice = reinterpret_cast<unsigned*>(work + 16);
            unsigned *reached = ice + words, *spare = reached + words, *water = spare + words, *whole = water + words;
            unsigned char* stamp = work + 16 + 4 * masks * words;
            const int nbi = sf_blocks((long long)n2 * n3 * 32), nbw = sf_blocks(words);
            k_sb_init<<<nbi, SF_THREADS, 0, s>>>(prob, phi_seed, G, zeta, g, ice, reached, water);
            pfgb::count_launch();
            if (erode && cudaMemcpyAsync(whole, ice, 4 * words, cudaMemcpyDeviceToDevice, s) != cudaSuccess) return PF_E_CUDA;
            for (int r = 0; r < erode; ++r) {
                k_sb_step<true><<<nbw, SF_THREADS, 0, s>>>(ice, spare, nullptr, g);
                pfgb::count_launch();
                unsigned* q = ice;
                ice = spare;
                spare = q;
            }
            long long done = 0;
            // every sweep that changes something reaches at least one more cell: at most n sweeps
            if (cudaMemsetAsync(flags, 0xff, 4 * sizeof(int), s) != cudaSuccess ||
                cudaMemsetAsync(stamp, 0, tiles, s) != cudaSuccess)
                return PF_E_CUDA;
            for (;;) {
                for (int r = 0; r < SWEEPS_PER_CHECK; ++r)
                    k_sb_flood<<<(unsigned)tiles, SB_THREADS, 0, s>>>(ice, reached, g, flags, stamp, done + r);
                pfgb::count_launch(SWEEPS_PER_CHECK);
                done += SWEEPS_PER_CHECK;
                int h = 0;
                if (cudaMemcpyAsync(&h, flags + ((done - 1) & 3), sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                    cudaStreamSynchronize(s) != cudaSuccess)
                    return PF_E_CUDA;
                if (!h || done > n) break;
            }
            for (int r = 0; r < erode + halo; ++r) {
                k_sb_step<false><<<nbw, SF_THREADS, 0, s>>>(reached, spare, r < erode ? whole : nullptr, g);
                pfgb::count_launch();
                unsigned* q = reached;
                reached = spare;
                spare = q;
            }
            k_sb_apply<<<nbi, SF_THREADS, 0, s>>>(prob, phi_seed, reached, water, g, phi_out);
            pfgb::count_launch();
            if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) return PF_E_CUDA;
            if (sweeps) *sweeps = done;
            return PF_OK;
        }
    }
    unsigned char* fl = work;
    int* changed = reinterpret_cast<int*>(work + ((n + 15) / 16) * 16);
    const int nb = sf_blocks(n);
    k_sf_init<<<nb, SF_THREADS, 0, s>>>(prob, phi_seed, G, zeta, n, fl);
    pfgb::count_launch();
    for (int r = 0; r < erode; ++r) {
        k_sf_erode<<<nb, SF_THREADS, 0, s>>>(fl, n1, n2, n3);
        k_sf_erode_commit<<<nb, SF_THREADS, 0, s>>>(fl, n);
        pfgb::count_launch(2);
    }
    long long done_sweeps = 0;
    // every sweep that changes something reaches at least one more cell: at most n sweeps
    for (;;) {
        if (cudaMemsetAsync(changed, 0, sizeof(int), s) != cudaSuccess) return PF_E_CUDA;
        for (int r = 0; r < SWEEPS_PER_CHECK; ++r) {
            k_sf_sweep<<<nb, SF_THREADS, 0, s>>>(fl, n1, n2, n3, 0, changed);
            pfgb::count_launch();
        }
        done_sweeps += SWEEPS_PER_CHECK;
        int h = 0;
        if (cudaMemcpyAsync(&h, changed, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return PF_E_CUDA;
        if (!h || done_sweeps > n) break;
    }
    for (int r = 0; r < erode + halo; ++r) {
        k_sf_sweep<<<nb, SF_THREADS, 0, s>>>(fl, n1, n2, n3, r < erode ? 2 : 1, changed);
        k_sf_commit<<<nb, SF_THREADS, 0, s>>>(fl, n);
        pfgb::count_launch(2);
    }
    k_sf_apply<<<nb, SF_THREADS, 0, s>>>(prob, phi_seed, G, zeta, n, fl, phi_out);
    pfgb::count_launch();
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) return PF_E_CUDA;
    if (sweeps) *sweeps = done_sweeps;
    return PF_OK;
}
