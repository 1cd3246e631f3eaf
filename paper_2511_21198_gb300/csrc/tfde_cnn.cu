// Warm-start network of the CN solves: four 3x3x3 convolutions with zero
// padding and ReLU between them, mapping per grid point the 11 input channels
//   (u / s, dt F / s, c_1..c_9),   s = max |u^m|,  c = nine problem constants,
// to (u^{m+1} - u^m) / s.  Not part of the paper: a learned initial guess for
// its Krylov solves; the FP64 residual test decides what the solver returns.
//
// Layout.  Activations are BF16, 16 channels (zero padded), on a grid with one
// layer of zero guard points on every side:
//   slot s = ((z + 1) (n2 + 2) + (y + 1)) R + (x + 1),   R = n1 + 2,
// so that every 3x3x3 tap is a constant shift of the slot index (dz P + dy R
// + dx, P = (n2 + 2) R) and the zero padding is the guard data itself.  The
// two channel halves are separate planes [half][slot][8 channels]: a run of
// slots of one half is contiguous in memory, so it is staged by ONE bulk copy
// (an interleaved layout needs a tensor copy with 16-byte rows, whose row rate
// bounded the convolution), and it lands as K-major core matrices.
//
// Forward / input-gradient convolution (tcgen05 implicit GEMM): M = 128
// slots, N = 16 output channels, K = 16 input channels per tap, 27 MMAs per
// 128 slots.  A tile is NT x 128 consecutive slots; per dz one run of
// tile + 2 R + 2 slots holds all nine (dy, dx) shifts (three runs per tile),
// so a slot is staged 3 (1 + (2 R + 2) / tile) times instead of nine; lines
// too long for two such stages take nine runs of tile + 2 slots.  The taps are
// shifts of the staged rows by 16 bytes each.  Warp 0 issues the copies, warp
// 1 the MMAs into double-buffered TMEM accumulators, warps 2..9 run the
// epilogue (bias, ReLU or ReLU-gradient mask, BF16 store of interior slots, or
// the FP32 output channel on the plain grid).
// Bound: the chain of 27 MMAs on one accumulator, about 256 cycles from one to
// the next (the time per layer is the same with N = 32, with M = 64, or with
// the operands exchanged, and without the copies or the epilogue).  So what
// counts is how many accumulators an SM has in flight: a CTA's NT = 4 tiles
// take the taps in turn, and two CTAs share an SM, which their memory allows
// because the ring holds planes (one dz of a tile, four of them) instead of
// whole tiles.  Measured on GB300 at 128^3: 107 us per layer with one CTA and
// two whole tiles, 75 us with two CTAs (162 us with nine 16-byte-row tensor
// copies per 128 slots); the tcgen05 pipe is then 83 % active (96^3).  Nine MMAs
// per 128 slots with the three dx taps side by side (N = 48, added up from
// neighbouring rows in the epilogue) took 85 us.
//
// Weight gradients: per tap a 16 x 16 matrix summed over all slots, on
// mma.sync m16n8k16 (tcgen05's smallest M of 64 would leave three quarters of
// the rows empty); the same staged runs as the convolution serve all 27 taps.
// One optimiser step of eight 64^3 samples: 2.2 ms, against 25.7 ms with the
// nine-copy convolution, a CUDA-core weight gradient per tap and 256-slot
// chunk (477 us per layer, 160 us for the sum of its partials), a one-block
// max |u| (183 us) and a 16-block bias sum (41 us).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "tfde_pdl.cuh"
#include "tfde_pow2conv.cuh"
#include "tfde_sum3.cuh"
#include "tfde_internal.h"
#include "tfde_stats.h"
#include "tfde_tc.h"
#include "tfde_tc_ptx.cuh"

namespace tfde {
namespace cnn {

constexpr int CH = 16;             // padded channels
constexpr int NL = 4;              // layers
constexpr int NTAP = 27;
constexpr int WSZ = CH * CH * NTAP;  // weights per layer (FP32 master [co][ci][tap])
constexpr int PSZ = WSZ + CH;        // + bias
constexpr int TM = 128;            // slots per MMA
constexpr int MAX_NT = 4;          // MMA tiles per staged tile: 1, 2 or 4
constexpr int STAGES = 2;
constexpr int W_BYTES = NTAP * 2 * CH * 16;              // 13824: [tap][khalf][co][8 ci]
constexpr int PLANES = 4;          // convolution: input planes (one dz of a tile) in the ring
constexpr int NUM_BARS = 2 * PLANES + 5;
constexpr int EPI_WARPS = 8;
constexpr int NUM_THREADS = 32 * (2 + EPI_WARPS);
constexpr int MAX_SMEM = 232448;
constexpr int CONV_FIXED_SMEM = 128 + W_BYTES + NUM_BARS * 8 + 16;
constexpr int WG_ROWS = 9;         // weight gradient: one warp per (dz, dy) ...
constexpr int WG_HALVES = 2;       // ... and half of the input channels
constexpr int WG_WARPS = WG_ROWS * WG_HALVES;
constexpr int WG_CLOSE = 2;        // blocks of 128 slots that a warp sums in FP32
constexpr int WG_THREADS = 32 * (WG_WARPS + 1);   // + the copy warp
constexpr int WG_SMEM_FIXED = 128 + 2 * STAGES * 8 + 16;
constexpr int GSZ = NTAP * 256 + CH;              // one partial: [tap][co][ci], then the bias

// How a tile's input rows are staged: nseg runs of seglen slots per channel
// half (3 runs, one per dz, or 9, one per (dz, dy)); row r = (dz + 1) 3 +
// (dy + 1) of the taps starts rowoff[r] slots into a half.  A plane is a
// third of it: plane_bytes per half, its row (dy + 1) rowoff[dy + 1] slots in.
struct Staging {
    int nt, tile, nseg, seglen, half_bytes, plane_bytes;
    int rowoff[9];
};

struct ConvParams {
    const uint8_t* in;             // activations, half 0; half 1 is half_stride bytes on
    long long half_stride;
    Staging st;
    const __nv_bfloat16* wts;      // [27][2][16][8] BF16 (B operand layout)
    const float* bias;             // [16] or null
    int relu;                      // apply ReLU after the bias
    const uint8_t* mask;           // activations or null: multiply by (mask > 0)
    uint8_t* out_act;              // activations or null
    float* out_f32;                // plain grid, channel 0, or null
    int n1, n2, n3;
    unsigned R, NY;                // slots per line, lines per plane (n2 + 2)
    long long P, first;
    int ntiles;
    int* err;
};

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     tc::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(tc::smem_u32(bar))
                 : "memory");
}

// The runs of plane dz (0, 1, 2 for dz = -1, 0, 1) of the tile from slot s0,
// both halves half_bytes apart, into `dst`; the caller has announced their
// bytes on `bar`.
__device__ __forceinline__ void stage_plane(uint8_t* dst, int half_bytes, const uint8_t* in, long long half_stride,
                                            const Staging& st, long long s0, int dz, long long P, unsigned R,
                                            uint64_t* bar) {
    const uint32_t bytes = (uint32_t)st.seglen * 16u;
    const long long first = s0 + (dz - 1) * P - (long long)R - 1;
    for (int h = 0; h < 2; ++h)
        for (int i = 0; i < st.nseg / 3; ++i)
            bulk_load(dst + h * half_bytes + i * bytes, in + h * half_stride + (first + i * (long long)R) * 16, bytes,
                      bar);
}

template <int NT>
__global__ void __launch_bounds__(NUM_THREADS, 2) conv_kernel(const __grid_constant__ ConvParams p) {
    using namespace tfde::tc;
    constexpr uint32_t TMEM_COLS = 2 * NT * CH;   // 32, 64 or 128
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    const int pbytes = 2 * p.st.plane_bytes;   // both halves of a plane
    uint8_t* wsm = smem;
    uint64_t* bars = reinterpret_cast<uint64_t*>(wsm + W_BYTES);
    uint8_t* ring = wsm + W_BYTES + ((NUM_BARS * 8 + 16 + 15) & ~15);
    uint64_t* full = bars;
    uint64_t* empty = bars + PLANES;
    uint64_t* tfull = bars + 2 * PLANES;
    uint64_t* tempty = bars + 2 * PLANES + 2;
    uint64_t* mma_done = bars + 2 * PLANES + 4;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NUM_BARS);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // weights into shared memory (generic proxy), made visible to the tensor core
    {
        const uint4* src = reinterpret_cast<const uint4*>(p.wts);
        uint4* dst = reinterpret_cast<uint4*>(wsm);
        for (int i = threadIdx.x; i < W_BYTES / 16; i += NUM_THREADS) dst[i] = src[i];
        fence_proxy_async_smem();
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < PLANES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], EPI_WARPS);
        }
        mbar_init(mma_done, 1);
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // the weights above were packed before the previous kernel began; the
    // activations are its output
    pdl_begin();

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0, filled = 0, last_ph = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
                for (int dz = 0; dz < 3; ++dz) {
                    if (!mbar_wait(&empty[s], ph ^ 1u, p.err)) { ok = false; break; }
                    mbar_expect_tx(&full[s], 2u * (uint32_t)p.st.plane_bytes);
                    stage_plane(ring + s * pbytes, p.st.plane_bytes, p.in, p.half_stride, p.st,
                                p.first + (long long)t * p.st.tile, dz, p.P, p.R, &full[s]);
                    filled |= 1u << s;
                    if (ph) last_ph |= 1u << s; else last_ph &= ~(1u << s);
                    if (++s == PLANES) { s = 0; ph ^= 1u; }
                }
            }
            for (int i = 0; i < PLANES; ++i)
                if (filled & (1u << i)) mbar_wait(&full[i], (last_ph >> i) & 1u, p.err, false);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = instr_desc(TM, CH, 0);
            // non-swizzled K-major: LBO = K-adjacent core matrix (channel half), SBO = next 8 rows
            const uint64_t a0 = smem_desc(smem_u32(ring), p.st.plane_bytes, 128, 0);
            const uint64_t b0 = smem_desc(smem_u32(wsm), 256, 128, 0);
            int s = 0;
            uint32_t ph = 0;
            int it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x, ++it) {
                const int buf = it & 1;
                const uint32_t use = (uint32_t)(it >> 1);
                if (!mbar_wait(&tempty[buf], (use & 1u) ^ 1u, p.err)) { ok = false; break; }
                for (int dz = 0; dz < 3; ++dz) {
                    if (!mbar_wait(&full[s], ph, p.err)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t as = a0 + (uint64_t)((s * pbytes) >> 4);
#pragma unroll
                    for (int k = 0; k < 9; ++k) {   // tap = 9 dz + k, k = (dy+1)*3 + (dx+1)
                        const uint64_t bd = b0 + (uint64_t)(((dz * 9 + k) * 512) >> 4);
                        const uint64_t at = as + (uint64_t)(p.st.rowoff[k / 3] + k % 3);
#pragma unroll
                        for (int m = 0; m < NT; ++m)
                            umma_bf16(tmem_base + (uint32_t)((buf * NT + m) * CH), at + (uint64_t)(m * TM), bd, idesc,
                                      dz + k > 0 ? 1u : 0u);
                    }
                    umma_commit(&empty[s]);
                    if (++s == PLANES) { s = 0; ph ^= 1u; }
                }
                if (ok) umma_commit(&tfull[buf]);
            }
            umma_commit(mma_done);
            mbar_wait(mma_done, 0, p.err, false);
        }
    } else {
        const int q = warp & 3;             // TMEM lane quadrant
        const int sub = (warp - 2) >> 2;    // which half of the tile's MMA tiles
        int it = 0;
        for (int t = blockIdx.x; t < p.ntiles; t += gridDim.x, ++it) {
            const int buf = it & 1;
            const uint32_t use = (uint32_t)(it >> 1);
            int ok = 1;
            if (lane == 0) ok = mbar_wait(&tfull[buf], use & 1u, p.err) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            __syncwarp();
            tc_fence_after();
#pragma unroll 1
            for (int m = sub; m < NT; m += 2) {
                const unsigned s = (unsigned)(p.first + (long long)t * p.st.tile) + m * TM + 32 * q + lane;
                const unsigned line = s / p.R, x1 = s - line * p.R;
                const unsigned z1 = line / p.NY, y1 = line - z1 * p.NY;
                const bool interior = x1 >= 1 && x1 <= (unsigned)p.n1 && y1 >= 1 && y1 <= (unsigned)p.n2 && z1 >= 1 &&
                                      z1 <= (unsigned)p.n3;
                uint4 mk[2];
                if (p.mask && interior) {
                    mk[0] = __ldg(reinterpret_cast<const uint4*>(p.mask + (size_t)s * 16));
                    mk[1] = __ldg(reinterpret_cast<const uint4*>(p.mask + p.half_stride + (size_t)s * 16));
                }
                __syncwarp();
                uint32_t r[16];
                tmem_ld16(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)((buf * NT + m) * CH), r);
                if (!interior) continue;
                float v[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    float a = __uint_as_float(r[c]);
                    if (p.bias) a += __ldg(p.bias + c);
                    if (p.relu) a = fmaxf(a, 0.f);
                    v[c] = a;
                }
                if (p.mask) {
                    const __nv_bfloat16* mb = reinterpret_cast<const __nv_bfloat16*>(mk);
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        if (!(__bfloat162float(mb[c]) > 0.f)) v[c] = 0.f;
                }
                if (p.out_act) {
                    uint4 o[2];
                    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(o);
#pragma unroll
                    for (int c = 0; c < 8; ++c) h[c] = __floats2bfloat162_rn(v[2 * c], v[2 * c + 1]);
                    *reinterpret_cast<uint4*>(p.out_act + (size_t)s * 16) = o[0];
                    *reinterpret_cast<uint4*>(p.out_act + p.half_stride + (size_t)s * 16) = o[1];
                }
                if (p.out_f32) p.out_f32[((size_t)(z1 - 1) * p.n2 + (y1 - 1)) * p.n1 + (x1 - 1)] = v[0];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
}

// ------------------------------------------------------------ weight gradient
struct WgradParams {
    const uint8_t* dz;             // gradient w.r.t. the layer's output
    const uint8_t* in;             // the layer's input activations
    long long half_stride;
    Staging st;
    unsigned R;
    long long P, first;
    int ntiles;
    float* part;                   // [gridDim.x][3][GSZ]: the parts of the sums
    int* err;
};

__device__ __forceinline__ void ldsm_t4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_t2(uint32_t addr, uint32_t (&r)[2]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Partial sums over this CTA's tiles of dW[tap][co][ci] = sum_s dZ[s][co]
// X[s + shift(tap)][ci] and db[co] = sum_s dZ[s][co] (dZ is zero on guard
// slots).  A warp takes the three dx taps of one row (dz, dy) for eight of the 16
// input channels: per 16 slots one transposed load of dZ (A, co x slots), two of
// X (B, slots x ci) and three MMAs; the bias is one more MMA of a row 4 warp
// against a matrix of ones.  Sums: 16 slots in the tensor core, WG_CLOSE blocks of
// 128 slots in FP32, and those in three-part FP32 sums, so that the error does not
// grow with the grid.  Bound: the MMAs, one per 8.4 cycles and SM.  One optimiser
// step of eight 64^3 samples: 2.22 ms; 2.27 with warps that take all 16 channels of
// every other block and sums in FP32 pairs, 2.72 with those sums in FP64.
__global__ void __launch_bounds__(WG_THREADS, 1) wgrad_kernel(const __grid_constant__ WgradParams p) {
    using namespace tfde::tc;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + STAGES;
    uint8_t* stages = smem + ((2 * STAGES * 8 + 15) & ~15);
    const int dz_half = p.st.tile * 16;
    const int stage_bytes = 2 * p.st.half_bytes + 2 * dz_half;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], WG_WARPS);
        }
        mbar_fence_init();
    }
    __syncthreads();
    pdl_begin();
    if (warp == WG_WARPS) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0, filled = 0, last_ph = 0;
            for (int t = blockIdx.x; t < p.ntiles; t += gridDim.x) {
                if (!mbar_wait(&empty[s], ph ^ 1u, p.err)) break;
                const long long s0 = p.first + (long long)t * p.st.tile;
                uint8_t* st = stages + s * stage_bytes;
                mbar_expect_tx(&full[s], 2u * (p.st.nseg * p.st.seglen + p.st.tile) * 16u);
                for (int dz = 0; dz < 3; ++dz)
                    stage_plane(st + dz * p.st.plane_bytes, p.st.half_bytes, p.in, p.half_stride, p.st, s0, dz, p.P, p.R,
                                &full[s]);
                for (int h = 0; h < 2; ++h)
                    bulk_load(st + 2 * p.st.half_bytes + h * dz_half, p.dz + h * p.half_stride + s0 * 16, dz_half,
                              &full[s]);
                filled |= 1u << s;
                if (ph) last_ph |= 1u << s; else last_ph &= ~(1u << s);
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
            for (int i = 0; i < STAGES; ++i)
                if (filled & (1u << i)) mbar_wait(&full[i], (last_ph >> i) & 1u, p.err, false);
        }
        return;
    }
    const int row = warp % WG_ROWS, half = warp / WG_ROWS;
    const bool bias = row == 4 && half == 0;
    Sum3 acc[14];    // 12 of the weights, 2 of the bias (every column the same)
    float sum[14];   // of the last blocks
    int held = 0;
#pragma unroll
    for (int i = 0; i < 14; ++i) sum[i] = 0.f;
    auto close = [&]() {
#pragma unroll
        for (int i = 0; i < 14; ++i) {
            acc[i].add(sum[i]);
            sum[i] = 0.f;
        }
        held = 0;
    };
    // A: matrices (slots 0-7, co 0-7), (0-7, 8-15), (8-15, 0-7), (8-15, 8-15);
    // B: slots 0-7 and 8-15 of dx = -1 and 0 (one load), then of dx = 1
    const int lr = lane & 7, lm = lane >> 3;
    const uint32_t aoff = (uint32_t)(2 * p.st.half_bytes + (lm & 1) * dz_half + ((lm >> 1) * 8 + lr) * 16);
    const uint32_t boff = (uint32_t)(half * p.st.half_bytes + ((lane & 15) + (lane >> 4) + p.st.rowoff[row]) * 16);
    const uint32_t one2 = 0x3F803F80u;
    int s = 0;
    uint32_t ph = 0;
    for (int t = blockIdx.x; t < p.ntiles; t += gridDim.x) {
        int ok = 1;
        if (lane == 0) ok = mbar_wait(&full[s], ph, p.err) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        __syncwarp();
        const uint32_t base = smem_u32(stages + s * stage_bytes);
        for (int k0 = 0; k0 < p.st.tile; k0 += TM) {
#pragma unroll 2
            for (int k = k0; k < k0 + TM; k += 16) {
                uint32_t a[4], b[4], b1[2];
                ldsm_t4(base + aoff + (uint32_t)k * 16u, a);
                ldsm_t4(base + boff + (uint32_t)k * 16u, b);
                ldsm_t2(base + boff + (uint32_t)(k + 2) * 16u, b1);
                float c[3][4] = {};
                mma_16816(c[0], a, b[0], b[1]);
                mma_16816(c[1], a, b[2], b[3]);
                mma_16816(c[2], a, b1[0], b1[1]);
#pragma unroll
                for (int i = 0; i < 12; ++i) sum[i] += c[i >> 2][i & 3];
                if (bias) {
                    float o[4] = {};
                    mma_16816(o, a, one2, one2);
                    sum[12] += o[0];
                    sum[13] += o[2];
                }
            }
            if (++held == WG_CLOSE) close();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
        if (++s == STAGES) { s = 0; ph ^= 1u; }
    }
    close();
    // accumulator (co = lane / 4 (+ 8), ci = 2 (lane % 4) (+ 1) (+ 8)); the sums' three parts in planes
    float* out = p.part + (size_t)blockIdx.x * 3 * GSZ;
    auto put = [&](int at, const Sum3& v) {
        out[at] = v.hi;
        out[GSZ + at] = v.mid;
        out[2 * GSZ + at] = v.lo;
    };
#pragma unroll
    for (int i = 0; i < 12; ++i) {
        const int dx = i >> 2, j = i & 3;
        const int co = (lane >> 2) + 8 * (j >> 1), ci = 8 * half + 2 * (lane & 3) + (j & 1);
        put((row * 3 + dx) * 256 + co * 16 + ci, acc[i]);
    }
    if (bias && (lane & 3) == 0)
#pragma unroll
        for (int j = 0; j < 2; ++j) put(NTAP * 256 + (lane >> 2) + 8 * j, acc[12 + j]);
}

// grad[layer][W co][ci][tap] (and the bias) += the sum of the partials, all layers
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float* __restrict__ part, int nparts,
                                                           float* __restrict__ grad) {
    __shared__ Sum3 sh[8][33];
    const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int idx = blockIdx.x * 32 + c;   // (tap, co, ci) or the bias
    const float* src = part + (size_t)blockIdx.y * nparts * 3 * GSZ;
    Sum3 acc;
    if (idx < GSZ) {
#pragma unroll 8
        for (int i = g; i < nparts; i += 8) {
            const float* v = src + (size_t)i * 3 * GSZ + idx;
            Sum3 t;
            t.hi = v[0];
            t.mid = v[GSZ];
            t.lo = v[2 * GSZ];
            acc += t;
        }
    }
    sh[g][c] = acc;
    __syncthreads();
    if (g == 0 && idx < GSZ) {
        for (int i = 1; i < 8; ++i) acc += sh[i][c];
        float* gl = grad + (size_t)blockIdx.y * PSZ;
        const float v = (float)acc.value();
        if (idx < NTAP * 256) {
            const int tap = idx / 256, co = (idx / 16) % 16, ci = idx % 16;
            gl[(co * CH + ci) * NTAP + tap] += v;
        } else {
            gl[WSZ + idx - NTAP * 256] += v;
        }
    }
}

// ------------------------------------------------------------ CUDA-core kernels
struct Grid {
    int n1, n2;
    unsigned R;
    long long P, half_stride;   // slots per plane; bytes between the channel halves
};
__device__ __forceinline__ size_t slot_of(unsigned p, const Grid& g) {
    const unsigned r = p / (unsigned)g.n1, x = p - r * (unsigned)g.n1;
    const unsigned z = r / (unsigned)g.n2, y = r - z * (unsigned)g.n2;
    return (size_t)(z + 1) * g.P + (size_t)((y + 1) * g.R + x + 1);
}

// max |u| as the bit pattern of a non-negative double (whose order is the
// integers'), NaNs passed over; *out starts at 0.  Bound by the read of u.
__global__ void __launch_bounds__(256) maxabs_kernel(const double* __restrict__ u, long long N,
                                                     unsigned long long* __restrict__ out) {
    const unsigned long long inf = 0x7ff0000000000000ull;
    unsigned long long m = 0;
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < N; i += gridDim.x * 256LL) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(u[i]) & 0x7fffffffffffffffull;
        if (b <= inf && b > m) m = b;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
        m = v > m ? v : m;
    }
    __shared__ unsigned long long sh[8];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) m = sh[i] > m ? sh[i] : m;
        if (m) atomicMax(out, m);
    }
}
__device__ __forceinline__ double scale_of(const unsigned long long* bits) {
    const unsigned long long b = *bits;
    return b ? __longlong_as_double((long long)b) : 1.0;
}

// 1 / scale, divided once per block: an FP64 division is about ten operations
// at two lanes per clock and SM, and a thread has one point at 64^3.
__device__ __forceinline__ double block_inverse(const unsigned long long* scale) {
    __shared__ double inv;
    if (threadIdx.x == 0) inv = 1.0 / scale_of(scale);
    __syncthreads();
    return inv;
}

// Conversions by integer operations (the same values: round to nearest even,
// exact), off the FP64 pipe, which bounds the element-wise kernels below: input
// packing at 128^3 53 -> 41 us; with the divisions above, the loss and its
// gradient at 64^3 17.5 -> 10.8 us.
__device__ __forceinline__ float to_f32(double v) {
    return f64_pow2_to_f32((unsigned long long)__double_as_longlong(v), 0);
}
__device__ __forceinline__ double to_f64(float v) { return f32_pow2_to_f64(v, 0); }

struct Coef {
    float c[9];
};

// X0[slot] = (u/s, dtF/s, c_0..c_8, d1/s, d2/s, 0...) for every interior grid
// point; d1 = u - u1 and d2 = u - 2 u1 + u2 are the first and second
// differences of the time history (zero channels without it)
__global__ void __launch_bounds__(256) pack_input_kernel(const double* __restrict__ u, const double* __restrict__ u1,
                                                         const double* __restrict__ u2, const double* __restrict__ dtF,
                                                         const unsigned long long* __restrict__ scale, const Coef coef,
                                                         const Grid g, unsigned N, uint8_t* __restrict__ X) {
    const double inv = block_inverse(scale);
    for (unsigned p = blockIdx.x * 256u + threadIdx.x; p < N; p += gridDim.x * 256u) {
        float v[16];
        const double up = u[p];
        v[0] = to_f32(up * inv);
        v[1] = dtF ? to_f32(dtF[p] * inv) : 0.f;
#pragma unroll
        for (int c = 0; c < 9; ++c) v[2 + c] = coef.c[c];
        v[11] = u1 ? to_f32((up - u1[p]) * inv) : 0.f;
        v[12] = (u1 && u2) ? to_f32((up - 2.0 * u1[p] + u2[p]) * inv) : 0.f;
#pragma unroll
        for (int c = 13; c < 16; ++c) v[c] = 0.f;
        uint4 o[2];
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(o);
#pragma unroll
        for (int c = 0; c < 8; ++c) h[c] = __floats2bfloat162_rn(v[2 * c], v[2 * c + 1]);
        uint8_t* dst = X + slot_of(p, g) * 16;
        *reinterpret_cast<uint4*>(dst) = o[0];
        *reinterpret_cast<uint4*>(dst + g.half_stride) = o[1];
    }
}

// The base the network corrects: u, or the polynomial extrapolation in time
// of the history (2u - u1 with one level, 3u - 3u1 + u2 with two).
__device__ __forceinline__ double guess_base(const double* u, const double* u1, const double* u2, long long p) {
    if (!u1) return u[p];
    if (!u2) return 2.0 * u[p] - u1[p];
    return 3.0 * u[p] - 3.0 * u1[p] + u2[p];
}

// x0 = base + s * out
__global__ void guess_kernel(const double* __restrict__ u, const double* __restrict__ u1,
                             const double* __restrict__ u2, const float* __restrict__ out,
                             const unsigned long long* __restrict__ scale, long long N, double* __restrict__ x0) {
    const double s = scale_of(scale);
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < N; p += (long long)gridDim.x * blockDim.x)
        x0[p] = guess_base(u, u1, u2, p) + s * to_f64(out[p]);
}

// loss partials and the output gradient: d = out - (u_next - u)/s ;
// dZ[slot] = (2 d / N, 0, ..) on every interior slot (both halves, so that the
// buffer needs no clearing: its guard slots are never written)
__global__ void __launch_bounds__(256) loss_grad_kernel(const float* __restrict__ out, const double* __restrict__ u,
                                                        const double* __restrict__ u1, const double* __restrict__ u2,
                                                        const double* __restrict__ un,
                                                        const unsigned long long* __restrict__ scale, const Grid g,
                                                        unsigned N, double two_n, uint8_t* __restrict__ dZ,
                                                        double* __restrict__ part) {
    __shared__ double sh[256];
    const double inv = block_inverse(scale);
    double acc = 0.0;
    for (unsigned p = blockIdx.x * 256u + threadIdx.x; p < N; p += gridDim.x * 256u) {
        const double d = to_f64(out[p]) - (un[p] - guess_base(u, u1, u2, p)) * inv;
        acc += d * d;
        uint8_t* dst = dZ + slot_of(p, g) * 16;
        const unsigned z = __bfloat16_as_ushort(__float2bfloat16_rn(to_f32(d * two_n)));
        *reinterpret_cast<uint4*>(dst) = make_uint4(z, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(dst + g.half_stride) = make_uint4(0u, 0u, 0u, 0u);
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// Forward weights [27][2][16][8] (B operand: N = co, K = ci) and input-gradient
// weights (N = ci, K = co, taps mirrored) from the FP32 master [co][ci][27];
// blockIdx.y is the layer.
__global__ void pack_weights_kernel(const float* __restrict__ prm, __nv_bfloat16* __restrict__ wf,
                                    __nv_bfloat16* __restrict__ wb) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;   // (tap, h, n, k8)
    if (idx >= NTAP * 256) return;
    const float* Wm = prm + (size_t)blockIdx.y * PSZ;
    const size_t at = (size_t)blockIdx.y * NTAP * 256 + idx;
    const int tap = idx / 256, h = (idx / 128) % 2, n = (idx / 8) % 16, k8 = idx % 8;
    const int k = 8 * h + k8;
    wf[at] = __float2bfloat16_rn(Wm[(n * CH + k) * NTAP + tap]);                  // W[co = n][ci = k][tap]
    wb[at] = __float2bfloat16_rn(Wm[(k * CH + n) * NTAP + (NTAP - 1 - tap)]);     // W[co = k][ci = n][-tap]
}

// Adam on all parameters (grads averaged over `count` samples), grads zeroed.
__global__ void adam_kernel(float* __restrict__ prm, float* __restrict__ grad, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2,
                            float inv_count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = grad[i] * inv_count;
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    prm[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    grad[i] = 0.f;
}

}  // namespace cnn
}  // namespace tfde

struct tfde_cnn {
    int n[3] = {};
    long long N = 0, R = 0, P = 0, S_total = 0, first = 0, count = 0;
    long long half_stride = 0;  // bytes between the channel halves of an activation buffer
    tfde::cnn::Staging conv_st, wg_st;   // tiles of the convolution and of the weight gradient
    int conv_tiles = 0, wg_tiles = 0, wg_grid = 0;
    float* prm = nullptr;      // FP32 master parameters, NL * PSZ
    float* grad = nullptr;
    float* adam_m = nullptr;
    float* adam_v = nullptr;
    int adam_t = 0;
    int accumulated = 0;
    __nv_bfloat16* wf = nullptr;  // packed forward weights, NL * 27*256
    __nv_bfloat16* wb = nullptr;  // packed input-gradient weights
    uint8_t* act[tfde::cnn::NL] = {};  // layer inputs X0..X3 (padded slots, two half planes)
    uint8_t* dz = nullptr;     // gradient buffers (padded slots), two
    uint8_t* dz2 = nullptr;
    float* out = nullptr;      // network output, plain grid
    unsigned long long* scale = nullptr;   // max |u| (bits of a double; 0: no scaling)
    float* wpart = nullptr;    // weight-gradient partials [NL][wg_grid][3][GSZ]
    double* lpart = nullptr;   // loss partials, then the error flag
    double* lpart_host = nullptr;
    int* err = nullptr;        // the word after lpart's partials
    bool packed = false;
};

namespace tfde {
namespace cnn {
namespace {

#define CN_TRY(expr)                                                                       \
    do {                                                                                   \
        cudaError_t e__ = (expr);                                                          \
        if (e__ != cudaSuccess)                                                            \
            return set_error(TFDE_ECUDA, std::string(#expr) + ": " + cudaGetErrorString(e__)); \
    } while (0)

int grid1(long long n) {
    long long g = (n + 255) / 256;
    if (g > 152LL * 8) g = 152LL * 8;
    return (int)(g < 1 ? 1 : g);
}

constexpr int LPART = 1216;   // loss partials (blocks of grid1)

// Tiles of nt x 128 slots, nt as large as leaves every SM a tile and smem(st)
// in `limit`, with three runs per tile (one per dz) where a tile of 128 slots
// fits so, else nine of two blocks.
template <typename F>
Staging staging(long long count, long long R, int limit, F smem) {
    Staging st{};
    auto make = [&](int nt, int nseg) {
        st.nt = nt;
        st.tile = nt * TM;
        st.nseg = nseg;
        st.seglen = (int)(nseg == 3 ? st.tile + 2 * R + 2 : st.tile + 2);
        st.plane_bytes = nseg / 3 * st.seglen * 16;
        st.half_bytes = 3 * st.plane_bytes;
        return smem(st) <= limit;
    };
    int nt = MAX_NT;
    while (nt > 1 && count < (long long)nt * TM * tc::num_sms()) nt /= 2;
    while (nt > 1 && !make(nt, 3)) nt /= 2;
    if (R > (1 << 20) || !make(nt, 3)) make(2, 9);
    for (int r = 0; r < 9; ++r)
        st.rowoff[r] = st.nseg == 3 ? (r / 3) * st.seglen + (int)((r % 3) * R) : r * st.seglen;
    return st;
}

// Two CTAs per SM share its 228 KB (1 KB of it reserved per CTA).
constexpr int CONV_SMEM_LIMIT = 116736 - 1024;
int conv_smem(const Staging& st) { return CONV_FIXED_SMEM + 16 + PLANES * 2 * st.plane_bytes; }
int wg_smem(const Staging& st) { return WG_SMEM_FIXED + STAGES * (2 * st.half_bytes + 2 * st.tile * 16); }

int conv(tfde_cnn* C, const uint8_t* in, const __nv_bfloat16* w, const float* bias, int relu, const uint8_t* mask,
         uint8_t* out_act, float* out_f32, cudaStream_t s) {
    ConvParams p;
    std::memset(&p, 0, sizeof(p));
    p.in = in;
    p.half_stride = C->half_stride;
    p.st = C->conv_st;
    p.wts = w;
    p.bias = bias;
    p.relu = relu;
    p.mask = mask;
    p.out_act = out_act;
    p.out_f32 = out_f32;
    p.n1 = C->n[0];
    p.n2 = C->n[1];
    p.n3 = C->n[2];
    p.R = (unsigned)C->R;
    p.NY = (unsigned)(C->n[1] + 2);
    p.P = C->P;
    p.first = C->first;
    p.ntiles = C->conv_tiles;
    p.err = C->err;
    const int grid = std::min(C->conv_tiles, 2 * tc::num_sms());
    const int smem = conv_smem(p.st);
    void* tok = stats_tc_begin(s, TFDE_KIND_CONV);
    // launched early: a block's set-up (weights, barriers, TMEM) runs as soon as
    // one of the previous kernel's blocks leaves its SM (with the weight gradient's:
    // one optimiser step of eight 64^3 samples 2.56 -> 2.28 ms)
    auto* kernel = p.st.nt == 4 ? conv_kernel<4> : (p.st.nt == 2 ? conv_kernel<2> : conv_kernel<1>);
    const cudaError_t e = launch_pdl_smem(true, kernel, grid, NUM_THREADS, smem, s, p);
    // algorithmic: the input activations read once, the output written once
    stats_tc_end(tok, s, TFDE_KIND_CONV, 64.0 * (double)C->N, 2.0 * NTAP * CH * CH * (double)C->N);
    if (e != cudaSuccess) return set_error(TFDE_ECUDA, std::string("conv_kernel launch: ") + cudaGetErrorString(e));
    return TFDE_OK;
}

int wgrad(tfde_cnn* C, int layer, const uint8_t* dz, cudaStream_t s) {
    WgradParams p;
    std::memset(&p, 0, sizeof(p));
    p.dz = dz;
    p.in = C->act[layer];
    p.half_stride = C->half_stride;
    p.st = C->wg_st;
    p.R = (unsigned)C->R;
    p.P = C->P;
    p.first = C->first;
    p.ntiles = C->wg_tiles;
    p.part = C->wpart + (size_t)layer * C->wg_grid * 3 * GSZ;
    p.err = C->err;
    stats_count_launch();
    CN_TRY(launch_pdl_smem(true, wgrad_kernel, C->wg_grid, WG_THREADS, wg_smem(p.st), s, p));
    return TFDE_OK;
}

int ensure_packed(tfde_cnn* C, cudaStream_t s) {
    if (C->packed) return TFDE_OK;
    stats_count_launch();
    pack_weights_kernel<<<dim3(NTAP, NL), 256, 0, s>>>(C->prm, C->wf, C->wb);
    C->packed = true;
    return TFDE_OK;
}

Grid grid_of(const tfde_cnn* C) { return Grid{C->n[0], C->n[1], (unsigned)C->R, C->P, C->half_stride}; }

// forward pass of (u, dtF, coef) into C->out (plain grid, output channel 0)
int forward(tfde_cnn* C, const double* u, const double* u1, const double* u2, const double* dtF,
            const double coef[9], cudaStream_t s) {
    Coef hc;
    for (int i = 0; i < 9; ++i) hc.c[i] = (float)coef[i];
    int st = ensure_packed(C, s);
    if (st) return st;
    stats_count_launch(2);
    CN_TRY(cudaMemsetAsync(C->scale, 0, sizeof(*C->scale), s));
    maxabs_kernel<<<grid1(C->N), 256, 0, s>>>(u, C->N, C->scale);
    pack_input_kernel<<<grid1(C->N), 256, 0, s>>>(u, u1, u2, dtF, C->scale, hc, grid_of(C), (unsigned)C->N, C->act[0]);
    for (int l = 0; l < NL; ++l) {
        const bool last = l + 1 == NL;
        if ((st = conv(C, C->act[l], C->wf + (size_t)l * NTAP * 256, C->prm + (size_t)l * PSZ + WSZ, last ? 0 : 1,
                       nullptr, last ? nullptr : C->act[l + 1], last ? C->out : nullptr, s)))
            return st;
    }
    return TFDE_OK;
}

// Reads the loss partials and the error flag behind them.
int check(tfde_cnn* C, cudaStream_t s) {
    CN_TRY(cudaMemcpyAsync(C->lpart_host, C->lpart, (LPART + 1) * sizeof(double), cudaMemcpyDeviceToHost, s));
    CN_TRY(cudaStreamSynchronize(s));
    if (*reinterpret_cast<const int*>(C->lpart_host + LPART))
        return set_error(TFDE_ETIMEOUT, "warm-start kernel wait ran out (device error flag set)");
    return TFDE_OK;
}

}  // namespace

int cnn_destroy(tfde_cnn* C);

int cnn_create(const int n[3], tfde_cnn** out) {
    *out = nullptr;
    for (int a = 0; a < 3; ++a)
        if (n[a] < 1) return set_error(TFDE_EINVAL, "grid sizes must be >= 1");
    tfde_cnn* C = new tfde_cnn();
    for (int a = 0; a < 3; ++a) C->n[a] = n[a];
    C->N = (long long)n[0] * n[1] * n[2];
    C->R = n[0] + 2;
    C->P = (long long)(n[1] + 2) * C->R;
    C->S_total = (long long)(n[2] + 2) * C->P;
    C->first = C->P + C->R + 1;
    C->count = C->S_total - 2 * C->first;   // slots from the first to the last interior point
    if (C->S_total + MAX_NT * TM >= (1LL << 31)) return set_error(TFDE_ENOMEM, "grid too large for the network");
    // the convolution's and the weight gradient's tiles; a tile may run past
    // the last interior slot, so every buffer ends in MAX_NT * TM more slots
    C->conv_st = staging(C->count, C->R, CONV_SMEM_LIMIT, conv_smem);
    C->wg_st = staging(C->count, C->R, MAX_SMEM, wg_smem);
    C->conv_tiles = (int)((C->count + C->conv_st.tile - 1) / C->conv_st.tile);
    C->wg_tiles = (int)((C->count + C->wg_st.tile - 1) / C->wg_st.tile);
    C->wg_grid = std::min(C->wg_tiles, tc::num_sms());
    C->half_stride = (C->S_total + MAX_NT * TM) * 16;
    const size_t act_bytes = 2 * (size_t)C->half_stride;
    for (auto f : {conv_kernel<1>, conv_kernel<2>, conv_kernel<4>})
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM) != cudaSuccess) {
            delete C;
            return set_error(TFDE_ECUDA, "cudaFuncSetAttribute(conv_kernel) failed");
        }
    if (cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM) != cudaSuccess) {
        delete C;
        return set_error(TFDE_ECUDA, "cudaFuncSetAttribute(wgrad_kernel) failed");
    }
    bool ok = cudaMalloc((void**)&C->prm, NL * PSZ * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void**)&C->grad, NL * PSZ * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void**)&C->adam_m, NL * PSZ * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void**)&C->adam_v, NL * PSZ * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void**)&C->wf, NL * NTAP * 256 * sizeof(__nv_bfloat16)) == cudaSuccess &&
              cudaMalloc((void**)&C->wb, NL * NTAP * 256 * sizeof(__nv_bfloat16)) == cudaSuccess &&
              cudaMalloc((void**)&C->dz, act_bytes) == cudaSuccess &&
              cudaMalloc((void**)&C->dz2, act_bytes) == cudaSuccess &&
              cudaMalloc((void**)&C->out, C->N * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void**)&C->scale, sizeof(*C->scale)) == cudaSuccess &&
              cudaMalloc((void**)&C->wpart, (size_t)NL * C->wg_grid * 3 * GSZ * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void**)&C->lpart, (LPART + 1) * sizeof(double)) == cudaSuccess &&
              cudaMallocHost((void**)&C->lpart_host, (LPART + 1) * sizeof(double)) == cudaSuccess;
    for (int l = 0; l < NL && ok; ++l) ok = cudaMalloc((void**)&C->act[l], act_bytes) == cudaSuccess;
    if (!ok) {
        cnn_destroy(C);
        return set_error(TFDE_ENOMEM, "allocation of the warm-start network workspace failed");
    }
    C->err = reinterpret_cast<int*>(C->lpart + LPART);
    // guard slots must stay zero: every buffer on the padded grid starts zeroed
    bool z = cudaMemset(C->dz, 0, act_bytes) == cudaSuccess && cudaMemset(C->dz2, 0, act_bytes) == cudaSuccess &&
             cudaMemset(C->prm, 0, NL * PSZ * sizeof(float)) == cudaSuccess &&
             cudaMemset(C->grad, 0, NL * PSZ * sizeof(float)) == cudaSuccess &&
             cudaMemset(C->adam_m, 0, NL * PSZ * sizeof(float)) == cudaSuccess &&
             cudaMemset(C->adam_v, 0, NL * PSZ * sizeof(float)) == cudaSuccess &&
             cudaMemset(C->lpart, 0, (LPART + 1) * sizeof(double)) == cudaSuccess;
    for (int l = 0; l < NL && z; ++l) z = cudaMemset(C->act[l], 0, act_bytes) == cudaSuccess;
    if (!z) {
        cnn_destroy(C);
        return set_error(TFDE_ECUDA, "zeroing of the warm-start workspace failed");
    }
    *out = C;
    return TFDE_OK;
}

int cnn_destroy(tfde_cnn* C) {
    if (!C) return TFDE_OK;
    cudaDeviceSynchronize();
    cudaFree(C->prm);
    cudaFree(C->grad);
    cudaFree(C->adam_m);
    cudaFree(C->adam_v);
    cudaFree(C->wf);
    cudaFree(C->wb);
    for (auto* a : C->act) cudaFree(a);
    cudaFree(C->dz);
    cudaFree(C->dz2);
    cudaFree(C->out);
    cudaFree(C->scale);
    cudaFree(C->wpart);
    cudaFree(C->lpart);
    if (C->lpart_host) cudaFreeHost(C->lpart_host);
    delete C;
    return TFDE_OK;
}

int cnn_set_params(tfde_cnn* C, const float* host) {
    CN_TRY(cudaMemcpy(C->prm, host, NL * PSZ * sizeof(float), cudaMemcpyHostToDevice));
    CN_TRY(cudaMemset(C->grad, 0, NL * PSZ * sizeof(float)));
    CN_TRY(cudaMemset(C->adam_m, 0, NL * PSZ * sizeof(float)));
    CN_TRY(cudaMemset(C->adam_v, 0, NL * PSZ * sizeof(float)));
    C->adam_t = 0;
    C->accumulated = 0;
    C->packed = false;
    return TFDE_OK;
}

int cnn_get(const tfde_cnn* C, int what, float* host) {
    const float* src = what == 0 ? C->prm : C->grad;
    CN_TRY(cudaMemcpy(host, src, NL * PSZ * sizeof(float), cudaMemcpyDeviceToHost));
    return TFDE_OK;
}

int cnn_predict(tfde_cnn* C, const double* u, const double* u1, const double* u2, const double* dtF,
                const double coef[9], double* x0, cudaStream_t s) {
    int st = forward(C, u, u1, u2, dtF, coef, s);
    if (st) return st;
    stats_count_launch();
    guess_kernel<<<grid1(C->N), 256, 0, s>>>(u, u1, u2, C->out, C->scale, C->N, x0);
    return check(C, s);
}

int cnn_accumulate(tfde_cnn* C, const double* u, const double* u1, const double* u2, const double* dtF,
                   const double coef[9], const double* u_next, double* loss, cudaStream_t s) {
    int st = forward(C, u, u1, u2, dtF, coef, s);
    if (st) return st;
    const int nb = grid1(C->N);
    stats_count_launch(2);
    loss_grad_kernel<<<nb, 256, 0, s>>>(C->out, u, u1, u2, u_next, C->scale, grid_of(C), (unsigned)C->N,
                                         2.0 / (double)C->N, C->dz, C->lpart);
    uint8_t* g = C->dz;      // gradient w.r.t. the output of layer l (pre-activation for l < NL - 1 after masking)
    uint8_t* g2 = C->dz2;
    for (int l = NL - 1; l >= 0; --l) {
        if ((st = wgrad(C, l, g, s))) return st;
        if (l > 0) {
            // gradient w.r.t. the input of layer l, masked by the ReLU of layer l - 1
            if ((st = conv(C, g, C->wb + (size_t)l * NTAP * 256, nullptr, 0, C->act[l], g2, nullptr, s))) return st;
            std::swap(g, g2);
        }
    }
    wgrad_reduce_kernel<<<dim3((GSZ + 31) / 32, NL), 256, 0, s>>>(C->wpart, C->wg_grid, C->grad);
    CN_TRY(cudaGetLastError());
    C->accumulated++;
    if ((st = check(C, s))) return st;
    double acc = 0.0;
    for (int b = 0; b < nb; ++b) acc += C->lpart_host[b];
    if (loss) *loss = acc / (double)C->N;
    return TFDE_OK;
}

int cnn_adam(tfde_cnn* C, float lr, cudaStream_t s) {
    if (C->accumulated == 0) return TFDE_OK;
    C->adam_t++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)C->adam_t), c2 = 1.f - std::pow(b2, (float)C->adam_t);
    const int n = NL * PSZ;
    stats_count_launch();
    adam_kernel<<<(n + 255) / 256, 256, 0, s>>>(C->prm, C->grad, C->adam_m, C->adam_v, n, lr, b1, b2, 1e-8f, c1, c2,
                                                1.f / (float)C->accumulated);
    C->accumulated = 0;
    C->packed = false;
    return check(C, s);
}

}  // namespace cnn
}  // namespace tfde
