// Gram-Schmidt building blocks of the FP32 Krylov cycles, shared by the
// single-problem and the batched kernels: inner products of one vector with up
// to eight basis vectors per sweep, the update, and both in one sweep.
//
// Bound: the basis is read once per sweep (L2, or HBM for large batches), so
// the elements go four at a time and eight vectors' loads are in flight per
// thread.  The other cost is the block reduction: FP64 adds issue at two lanes
// per clock and SM, and a shuffle tree per result (40 warp-wide adds for eight)
// took longer than the sweep at 128^3 (31 us per launch against 7).  The eight
// results share one tree (9 warp-wide adds and 3 across the warps), and the
// compensated FP32 sums go through it as three FP32 values (tfde_sum3.cuh, more
// accurate than FP64): their conversions to FP64 alone were 6000 lane operations
// per block.  The partial sums over the blocks are added by the last block of the
// sweep, which spares a launch each.  Both together: projection sweep of 64 uneven
// problems 167 -> 84 us, at 128^3 14.6 -> 11.1 us.
#pragma once

#include <cuda_runtime.h>

#include "tfde_sum3.cuh"

namespace tfde {
namespace gs {

constexpr int kThreads = 256;
constexpr int kWidth = 8;   // basis vectors per sweep

__device__ __forceinline__ Sum3 shfl_xor(const Sum3 v, int off) {
    Sum3 o;
    o.hi = __shfl_xor_sync(0xffffffffu, v.hi, off);
    o.mid = __shfl_xor_sync(0xffffffffu, v.mid, off);
    o.lo = __shfl_xor_sync(0xffffffffu, v.lo, off);
    return o;
}
__device__ __forceinline__ double shfl_xor(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
__device__ __forceinline__ double value_of(const Sum3 v) { return v.value(); }
__device__ __forceinline__ double value_of(double v) { return v; }

// Kahan-compensated FP32 accumulation.
struct KSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
    __device__ __forceinline__ Sum3 sum3() const {
        Sum3 t;
        t.hi = s;
        t.mid = -c;
        return t;
    }
};
__device__ __forceinline__ void add4(KSum& k, const float4 a, const float4 b) {
    k.add(a.x * b.x);
    k.add(a.y * b.y);
    k.add(a.z * b.z);
    k.add(a.w * b.w);
}
__device__ __forceinline__ void axpy4(float4& w, float h, const float4 v) {
    w.x = fmaf(-h, v.x, w.x);
    w.y = fmaf(-h, v.y, w.y);
    w.z = fmaf(-h, v.z, w.z);
    w.w = fmaf(-h, v.w, w.w);
}

// Block sums of eight values (double or Sum3) per thread, result j < mc handed
// to f(j, sum) by one thread.  Each exchange over the lanes halves the values a lane carries,
// so the warp needs 4 + 2 + 1 + 1 + 1 adds; fixed order.  Every thread of the
// (kThreads-wide) block calls it.
template <typename T, typename F>
__device__ __forceinline__ void block_sums8(T (&v)[kWidth], int mc, F f) {
    static_assert(kThreads == 256 && kWidth == 8, "eight warps' sums of eight values");
    __shared__ T sh[kWidth][kThreads / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {
        const int off = 4 * w;   // lanes 16, 8, 4 apart
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const T send = up ? v[i] : v[i + w];
            T keep = up ? v[i + w] : v[i];
            keep += shfl_xor(send, off);
            v[i] = keep;
        }
    }
    v[0] += shfl_xor(v[0], 2);
    v[0] += shfl_xor(v[0], 1);
    __syncthreads();   // the previous call's reads of sh are done
    if ((lane & 3) == 0) sh[lane >> 2][warp] = v[0];   // lane bits 4..2 are the value's index
    __syncthreads();
    if (warp == 0) {   // four lanes per value, two warps' sums each
        T t = sh[lane >> 2][lane & 3];
        t += sh[lane >> 2][(lane & 3) + 4];
        t += shfl_xor(t, 2);
        t += shfl_xor(t, 1);
        if ((lane & 3) == 0 && lane >> 2 < mc) f(lane >> 2, value_of(t));
    }
}
template <typename F>
__device__ __forceinline__ void block_sums8(KSum (&k)[kWidth], int mc, F f) {
    Sum3 v[kWidth];
#pragma unroll
    for (int j = 0; j < kWidth; ++j) v[j] = k[j].sum3();
    block_sums8(v, mc, f);
}
// the same for one value per thread
template <typename F>
__device__ __forceinline__ void block_sum1(const KSum& k, F f) {
    __shared__ Sum3 sh[kThreads / 32];
    Sum3 v = k.sum3();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += shfl_xor(v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = sh[threadIdx.x & 7];
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) v += shfl_xor(v, off);
        if (threadIdx.x == 0) f(v.value());
    }
}

// True in the one of `count` blocks that comes here last, once every one's
// earlier writes are visible to it.  *ticket starts at 0 and is left at 0.
__device__ __forceinline__ bool last_block(unsigned* ticket, unsigned count) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(ticket, count - 1) == count - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}
// f(j, sum over b < nblk of part[j * stride + b]), j < m, a warp per result,
// fixed order (one block; part written by the same kernel's blocks)
template <typename F>
__device__ __forceinline__ void sum_partials(const double* part, int stride, int nblk, int m, F f) {
    for (int j = threadIdx.x >> 5; j < m; j += kThreads / 32) {
        double acc = 0.0;
#pragma unroll 8
        for (int b = threadIdx.x & 31; b < nblk; b += 32) acc += __ldcg(part + (long long)j * stride + b);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) f(j, acc);
    }
}

// The elements [lo, hi) of a block in groups of four (lo a multiple of 4, the
// vectors 16-byte aligned) and the rest singly: f4(i) for the group at element
// i, f1(i) for one element.  Unaligned vectors (vec false) go singly.
template <typename F4, typename F1>
__device__ __forceinline__ void sweep(long long lo, long long hi, bool vec, F4 f4, F1 f1) {
    long long done = lo;
    if (vec) {
        done = lo + (hi - lo) / 4 * 4;
        for (long long i = lo + 4 * threadIdx.x; i < done; i += 4 * kThreads) f4(i);
    }
    for (long long i = done + threadIdx.x; i < hi; i += kThreads) f1(i);
}

// Partial sums <V_{m0 + j}, w>, j < mc <= 8, over [lo, hi)
template <typename F>
__device__ __forceinline__ void dots(const float* __restrict__ V, long long ldv, int m0, int mc,
                                     const float* w, long long lo, long long hi, bool vec, F out) {
    KSum k[kWidth];
    const float* V0 = V + (long long)m0 * ldv;
    sweep(
        lo, hi, vec,
        [&](long long i) {
            const float4 wi = *reinterpret_cast<const float4*>(w + i);
            float4 v[kWidth];
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                if (j < mc) v[j] = __ldg(reinterpret_cast<const float4*>(V0 + j * ldv + i));
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                if (j < mc) add4(k[j], v[j], wi);
        },
        [&](long long i) {
            const float wi = w[i];
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                if (j < mc) k[j].add(__ldg(V0 + j * ldv + i) * wi);
        });
    block_sums8(k, mc, [&](int j, double sum) { out(m0 + j, sum); });
}

// w -= sum_{j < m} hs[j] V_j at the four elements from i
__device__ __forceinline__ void update4(float4& w, const float* __restrict__ V, long long ldv, const float* hs, int m,
                                        long long i) {
    int j = 0;
    for (; j + 4 <= m; j += 4) {
        float4 v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) v[t] = __ldg(reinterpret_cast<const float4*>(V + (long long)(j + t) * ldv + i));
#pragma unroll
        for (int t = 0; t < 4; ++t) axpy4(w, hs[j + t], v[t]);
    }
    for (; j < m; ++j) axpy4(w, hs[j], __ldg(reinterpret_cast<const float4*>(V + (long long)j * ldv + i)));
}
__device__ __forceinline__ float update1(float w, const float* __restrict__ V, long long ldv, const float* hs, int m,
                                         long long i) {
    for (int j = 0; j < m; ++j) w = fmaf(-hs[j], __ldg(V + (long long)j * ldv + i), w);
    return w;
}

// w -= sum_{j < m} hs[j] V_j and the partial sums <V_j, w> of the updated w.
// Up to eight vectors: one read of the basis; beyond, the first sweep updates
// and forms the first eight, and each further eight take a sweep.
template <typename F>
__device__ __forceinline__ void update_dots(const float* __restrict__ V, long long ldv, const float* hs, int m,
                                            float* w, long long lo, long long hi, bool vec, F out) {
    KSum k[kWidth];
    const int mc = m < kWidth ? m : kWidth;
    sweep(
        lo, hi, vec,
        [&](long long i) {
            float4 wi = *reinterpret_cast<const float4*>(w + i);
            float4 v[kWidth];
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                if (j < mc) v[j] = __ldg(reinterpret_cast<const float4*>(V + j * ldv + i));
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                if (j < mc) axpy4(wi, hs[j], v[j]);
            if (m > kWidth) update4(wi, V + kWidth * ldv, ldv, hs + kWidth, m - kWidth, i);
            *reinterpret_cast<float4*>(w + i) = wi;
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                if (j < mc) add4(k[j], v[j], wi);
        },
        [&](long long i) {
            const float wi = update1(w[i], V, ldv, hs, m, i);
            w[i] = wi;
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                if (j < mc) k[j].add(__ldg(V + j * ldv + i) * wi);
        });
    block_sums8(k, mc, out);
    // each thread reads the elements of w it wrote
    for (int m0 = kWidth; m0 < m; m0 += kWidth)
        dots(V, ldv, m0, m - m0 < kWidth ? m - m0 : kWidth, w, lo, hi, vec, out);
}

// w -= sum_{j < m} hs[j] V_j and the partial sum of the updated w^2 (m = 0:
// the sum alone)
template <typename F>
__device__ __forceinline__ void update_norm(const float* __restrict__ V, long long ldv, const float* hs, int m,
                                            float* w, long long lo, long long hi, bool vec, F out) {
    KSum k;
    sweep(
        lo, hi, vec,
        [&](long long i) {
            float4 wi = *reinterpret_cast<const float4*>(w + i);
            if (m > 0) {
                update4(wi, V, ldv, hs, m, i);
                *reinterpret_cast<float4*>(w + i) = wi;
            }
            add4(k, wi, wi);
        },
        [&](long long i) {
            float wi = w[i];
            if (m > 0) w[i] = wi = update1(wi, V, ldv, hs, m, i);
            k.add(wi * wi);
        });
    block_sum1(k, out);
}

}  // namespace gs
}  // namespace tfde
