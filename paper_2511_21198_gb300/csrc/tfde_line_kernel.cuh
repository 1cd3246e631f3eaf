// Dense per-axis passes on CUDA cores in the arithmetic of the FFT passes
// (FP64 or FP32): the three pass forms of tfde_fft.cu (Toeplitz product with
// its mass terms, DST-I, DST-I pair around the Lambda division) as a product
// of the axis matrix with a tile of lines staged in shared memory.
//
// Work.  An FFT pass costs 2 transforms of length L >= 2n - 1 per line (pair)
// and, in the DST's chirp form, two per line; the dense product n^2
// multiply-adds, halved where the matrix commutes with the reversal of the
// line: S_n (sin((n+1-j) k pi/(n+1)) = (-1)^(k+1) sin(j k pi/(n+1))) and a
// symmetric Toeplitz matrix (k+ = k-).  There the line is folded first,
// e_j = x_j + x_{n-1-j} and o_j = x_j - x_{n-1-j}, and two products of half
// the size follow (odd / even k for the DST; E + O and E - O for the two ends
// of a Toeplitz line).
#pragma once

#include <cuda_runtime.h>

namespace tfde {
namespace fft {

enum { LINE_TOEPLITZ = 0, LINE_DST = 1, LINE_DST2 = 2 };

// One axis matrix as the kernel reads it, [k][row] (rows contiguous, padded
// with zeros to a multiple of 16).  Unsplit (half = 0): K = n, rows 0..n-1.  Split: K =
// ceil(n / 2); rows are in blocks of 2 RH: RH rows of the product with the
// folded sums, then the RH rows of the same indices with the differences, so
// that a block of the grid holds both ends of its outputs.
struct LineMatrix {
    const void* m = nullptr;
    int K = 0, ld = 0, half = 0;   // half: RH
};

struct LinePass {
    const void* in0;
    const void* in1;
    void* out0;
    void* out1;
    LineMatrix m;
    int n1, n2, n3, axis, n;
    long long lines;
    double alpha, beta;
    const void* lam;              // [mass x | y | z | tau x | y | z] (double or float) or null
    double c0, c1, c2;            // eta_a (k+ + k-)
    int half_power;               // divide by Lambda^{1/2} instead of Lambda
    const int* skip;              // optional: no work when *skip != 0
};

constexpr int LINE_ROWS = 128;    // matrix rows per block of the grid

constexpr int LINE_STAGES = 4;    // matrix chunks in flight
template <typename R>
constexpr int line_chunk() { return 64 / (int)sizeof(R); }   // matrix columns per chunk

// CNT consecutive values from shared memory in the widest accesses
template <typename R, int CNT>
__device__ __forceinline__ void line_lds(const R* p, R (&v)[CNT]) {
    if constexpr (CNT * sizeof(R) % 16 == 0) {
        constexpr int Q = 16 / sizeof(R);
#pragma unroll
        for (int i = 0; i < CNT / Q; ++i) {
            const uint4 q = *(reinterpret_cast<const uint4*>(p) + i);
            const R* e = reinterpret_cast<const R*>(&q);
#pragma unroll
            for (int k = 0; k < Q; ++k) v[i * Q + k] = e[k];
        }
    } else if constexpr (CNT * sizeof(R) == 8 && CNT > 1) {
        const uint2 q = *reinterpret_cast<const uint2*>(p);
        const R* e = reinterpret_cast<const R*>(&q);
#pragma unroll
        for (int k = 0; k < CNT; ++k) v[k] = e[k];
    } else {
#pragma unroll
        for (int k = 0; k < CNT; ++k) v[k] = p[k];
    }
}
__device__ __forceinline__ void line_cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// one element: lines start at any multiple of the element size
template <typename R>
__device__ __forceinline__ void line_cp1(R* dst, const R* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"((int)sizeof(R))
                 : "memory");
}
__device__ __forceinline__ void line_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void line_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory"); }

// Shares the positions j < cnt of BN lines out over the block's warps:
// f(g, j0, step) takes line g's positions j0, j0 + step, ..  Along x a warp
// covers 8 positions of 4 lines (shared-memory words in different banks,
// whole 32-byte sectors in global memory), along y and z the line runs
// fastest.  The line, and with it every address's base, is fixed per call.
template <int BN, typename F>
__device__ __forceinline__ void line_walk(bool xax, F f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (xax) {
        constexpr int GB = BN / 4;
        const int nsub = nw >= GB ? nw / GB : 1, sub = nw >= GB ? warp / GB : 0;
        if (sub >= nsub) return;
        for (int g4 = nw >= GB ? warp % GB : warp; g4 < GB; g4 += nw >= GB ? GB : nw)
            f(4 * g4 + (lane >> 3), (lane & 7) + 8 * sub, 8 * nsub);
    } else if constexpr (BN >= 32) {
#pragma unroll
        for (int h = 0; h < BN / 32; ++h) f(lane + 32 * h, warp, nw);
    } else {
        constexpr int JW = 32 / BN;
        f(lane % BN, warp * JW + lane / BN, nw * JW);
    }
}

// Block (line tile, LINE_ROWS matrix rows): TL threads x LT lines by
// blockDim / TL threads x RT rows.  The lines (and the second operand's, for
// the epilogue) arrive element by element through cp.async, so that all of
// them are in flight at once; the matrix follows in chunks, LINE_STAGES of
// them in flight.  A split pass folds the lines in place: sums at the near
// end, differences at the far end.  FP32 sums each chunk apart before adding
// it, so that the error grows with the square root of K / 16 + 16, not of K.
// Bound at FP32: the instructions around the multiply-adds (addresses,
// staging, fold and store), hence one line per thread and constant strides in
// every phase; at FP64: the FP64 pipe.
template <typename R, int MODE, int TL, int LT, int RT>
__global__ void __launch_bounds__(256, LT >= 4 ? 2 : 3) line_pass_kernel(const __grid_constant__ LinePass p) {
    constexpr int BN = TL * LT, BNS = BN + 16 / sizeof(R);
    constexpr int KC = line_chunk<R>();
    constexpr int Q = 16 / sizeof(R);
    extern __shared__ __align__(16) unsigned char line_smem[];
    const int n = p.n, K = p.m.K, half = p.m.half, ld = p.m.ld;
    const int rows = blockDim.x / TL * RT;                   // matrix rows of this block
    const int row0 = blockIdx.y * LINE_ROWS;
    const int fo = half ? n / 2 : 0;
    const long long l0 = (long long)blockIdx.x * BN;
    const long long st = p.axis == 0 ? 1LL : (p.axis == 1 ? (long long)p.n1 : (long long)p.n1 * p.n2);
    const R* __restrict__ in0 = static_cast<const R*>(p.in0);
    const R* __restrict__ in1 = static_cast<const R*>(p.in1);
    R* __restrict__ out0 = static_cast<R*>(p.out0);
    R* __restrict__ out1 = static_cast<R*>(p.out1);
    const int live = (int)min((long long)BN, p.lines - l0);
    const bool xax = p.axis == 0;
    // shared memory: the lines X (overlaid by the results Y, apart in the DST
    // pair), the second operand's lines Z, the matrix chunks A
    R* const X = reinterpret_cast<R*>(line_smem);
    R* const Y = MODE == LINE_DST2 ? X + (size_t)n * BNS : X;
    R* const Z = MODE == LINE_DST2 ? Y + (size_t)rows * BNS : X + (size_t)max(n, rows) * BNS;
    R* const A = Z + (MODE == LINE_TOEPLITZ && in1 ? (size_t)n * BNS : 0);

    // matrix chunk c, one commit group (empty past the last): this thread's 16
    // bytes of columns k0 and k0 + KC / 2
    const int per = rows / Q, k0 = threadIdx.x / per, r0 = (threadIdx.x - k0 * per) * Q;
    const R* M = static_cast<const R*>(p.m.m) + row0 + (size_t)k0 * ld + r0;
    R* const Ad = A + k0 * rows + r0;
    const int chunks = (K + KC - 1) / KC;
    auto fetch = [&](int c) {
        R* dst = Ad + (c % LINE_STAGES) * KC * rows;
        const R* src = M + (size_t)(c * KC) * ld;
        if (c * KC + k0 < K) line_cp16(dst, src);
        if (c * KC + k0 + KC / 2 < K) line_cp16(dst + KC / 2 * rows, src + (size_t)(KC / 2) * ld);
        line_commit();
    };
    // line l0 + g starts at: x: (l0 + g) n1; y: i + q n1 n2 with l = q n1 + i; z: l0 + g
    unsigned i0 = 0;
    long long q0 = 0;
    if (!xax) {
        q0 = l0 < (1LL << 32) ? (long long)((unsigned)l0 / (unsigned)p.n1) : l0 / p.n1;
        i0 = (unsigned)(l0 - q0 * p.n1);
    }
    auto split_line = [&](int g, unsigned* i, long long* q) {
        *i = i0 + (unsigned)g;
        *q = q0;
        if (*i >= (unsigned)p.n1) {
            *q += *i / (unsigned)p.n1;
            *i %= (unsigned)p.n1;
        }
    };
    auto line_start = [&](int g) -> long long {
        if (xax) return (l0 + g) * (long long)p.n1;
        if (p.axis == 2) return l0 + g;
        unsigned i;
        long long q;
        split_line(g, &i, &q);
        return (long long)i + q * (long long)p.n1 * p.n2;
    };
    auto fetch_lines = [&](R* dst, const R* src) {
        line_walk<BN>(xax, [&](int g, int j, int step) {
            if (g >= live) return;
            const R* from = src + line_start(g) + j * st;
            R* to = dst + j * BNS + g;
#pragma unroll 4
            for (; j < n; j += step) {
                line_cp1(to, from);
                from += step * st;
                to += step * BNS;
            }
        });
    };
    // launched with programmatic stream serialisation: the first matrix chunks
    // are on their way before the previous kernel has ended; its results are
    // read only after the wait
    for (int c = 0; c < LINE_STAGES - 1; ++c) fetch(c);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // (a long matrix streams from L2 through the whole product: the next
    // launch's first chunks would only get in its way, 511^2: 13.0 against 12.7 ms)
    if (K <= 256) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (p.skip && *reinterpret_cast<const volatile int*>(p.skip)) {
        line_wait<0>();
        return;
    }
    fetch_lines(X, in0);
    line_commit();
    if (MODE == LINE_TOEPLITZ && in1) fetch_lines(Z, in1);
    line_commit();
    line_wait<1>();   // the lines; the second operand's are waited for below
    __syncthreads();

    if (MODE == LINE_TOEPLITZ && out1) {
        // this block's share of out1 = M in0
        const int ja = n * (int)blockIdx.y / (int)gridDim.y, jb = n * ((int)blockIdx.y + 1) / (int)gridDim.y;
        line_walk<BN>(xax, [&](int g, int j, int step) {
            if (g >= live) return;
            j += ja;
            R* to = out1 + line_start(g) + j * st;
            const R* x = X + j * BNS + g;
#pragma unroll 2
            for (; j < jb; j += step) {
                const R lo = j > 0 ? x[-BNS] : R(0), hi = j + 1 < n ? x[BNS] : R(0);
                *to = fma(R(0.75), x[0], R(0.125) * (lo + hi));
                to += step * st;
                x += step * BNS;
            }
        });
        if (half) __syncthreads();
    }
    if (half) {
        line_walk<BN>(false, [&](int g, int j, int step) {
            R* lo = X + j * BNS + g;
            R* hi = X + (n - 1 - j) * BNS + g;
#pragma unroll 2
            for (; j < fo; j += step) {
                const R a = *lo, b = *hi;
                *lo = a + b;
                *hi = a - b;
                lo += step * BNS;
                hi -= step * BNS;
            }
        });
    }

    const int tl = threadIdx.x % TL, ti = threadIdx.x / TL;
    auto product = [&]() {
        // the block's rows: half of the sums, then half of the differences
        // (which run down from the far end)
        const bool diff = half && ti * RT >= half;
        const R* x = X + (diff ? (size_t)(n - 1) * BNS : 0) + tl * LT;
        const int xs = diff ? -BNS : BNS;
        R acc[RT][LT];
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int l = 0; l < LT; ++l) acc[r][l] = R(0);
        for (int c = 0; c < chunks; ++c) {
            line_wait<LINE_STAGES - 2>();
            __syncthreads();   // chunk c and the folded lines visible; chunk c - 1's buffer free
            fetch(c + LINE_STAGES - 1);
            const R* am = A + (c % LINE_STAGES) * KC * rows + ti * RT;
            const int kc = min(KC, K - c * KC);
            R part[RT][LT];
            if constexpr (sizeof(R) == 4) {
#pragma unroll
                for (int r = 0; r < RT; ++r)
#pragma unroll
                    for (int l = 0; l < LT; ++l) part[r][l] = R(0);
            }
            auto step = [&](int k) {
                R a[RT], v[LT];
                line_lds<R, RT>(am, a);
                line_lds<R, LT>(x, v);
                am += rows;
                x += xs;
#pragma unroll
                for (int r = 0; r < RT; ++r)
#pragma unroll
                    for (int l = 0; l < LT; ++l) {
                        if constexpr (sizeof(R) == 4) part[r][l] = fma(a[r], v[l], part[r][l]);
                        else acc[r][l] = fma(a[r], v[l], acc[r][l]);
                    }
            };
            if (kc == KC) {
#pragma unroll
                for (int k = 0; k < KC; ++k) step(k);
            } else {
#pragma unroll 1
                for (int k = 0; k < kc; ++k) step(k);
            }
            if constexpr (sizeof(R) == 4) {
#pragma unroll
                for (int r = 0; r < RT; ++r)
#pragma unroll
                    for (int l = 0; l < LT; ++l) acc[r][l] += part[r][l];
            }
        }
        line_wait<0>();
        __syncthreads();   // every read of X and A done: Y may overlay X
        R* y = Y + (size_t)ti * RT * BNS + tl * LT;
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int l = 0; l < LT; ++l) y[r * BNS + l] = acc[r][l];
    };
    product();
    if (MODE == LINE_DST2)
        for (int c = 0; c < LINE_STAGES - 1; ++c) fetch(c);
    __syncthreads();

    // Lambda along line g: m_a(j) U + t_a(j) V from the two other axes' eigenvalues
    const R* mx = static_cast<const R*>(p.lam);
    const R* my = mx + p.n1;
    const R* mz = my + p.n2;
    const R* tx = mz + p.n3;
    const R* ty = tx + p.n1;
    const R* tz = ty + p.n2;
    const R* ma = p.axis == 2 ? mz : my;
    const R* ta = p.axis == 2 ? tz : ty;
    auto line_lambda = [&](int g, R* U, R* V) {
        const R c0 = (R)p.c0, c1 = (R)p.c1, c2 = (R)p.c2;
        unsigned i;
        long long q;
        split_line(g, &i, &q);
        const R* mo = p.axis == 2 ? my : mz;   // the third axis
        const R* to = p.axis == 2 ? ty : tz;
        *U = fma(mo[q], fma(c0, tx[i], mx[i]), (p.axis == 2 ? c1 : c2) * to[q] * mx[i]);
        *V = (p.axis == 2 ? c2 : c1) * mo[q] * mx[i];
    };
    auto lambda = [&](R U, R V, int j) -> R {
        const R lam = fma(ma[j], U, ta[j] * V);
        return p.half_power ? sqrt(lam) : lam;
    };
    // DST output index j in this block's Y (odd j: the differences' rows)
    auto dst_row = [&](int j) { return (j & 1) * half + (j >> 1); };
    if constexpr (MODE == LINE_DST2) {
        // t = S in0 / Lambda, folded as the second transform's input (the
        // block holds every row)
        line_walk<BN>(false, [&](int g, int j, int step) {
            if (g >= live) return;
            R U, V;
            line_lambda(g, &U, &V);
#pragma unroll 2
            for (; j < K; j += step) {
                const R a = Y[dst_row(j) * BNS + g] / lambda(U, V, j);
                if (j < fo) {
                    const R b = Y[dst_row(n - 1 - j) * BNS + g] / lambda(U, V, n - 1 - j);
                    X[j * BNS + g] = a + b;
                    X[(n - 1 - j) * BNS + g] = a - b;
                } else {
                    X[j * BNS + g] = a;
                }
            }
        });
        product();   // its first barrier covers the writes of X
        __syncthreads();
    }

    // ---- store: rows r of the block (split: the pair of outputs that the sum
    // and the difference of row r give)
    const int i0r = half ? row0 / 2 : row0;
    const int rE = half ? min(half, K - i0r) : min(rows, n - row0);
    const int rO = half ? max(0, min(half, fo - i0r)) : 0;
    auto combine = [&](R v, const R* z, int j) -> R {   // alpha v + beta M in1
        v *= (R)p.alpha;
        if (in1) {
            const R lo = j > 0 ? z[-BNS] : R(0), hi = j + 1 < n ? z[BNS] : R(0);
            v = fma((R)p.beta, fma(R(0.75), z[0], R(0.125) * (lo + hi)), v);
        }
        return v;
    };
    line_walk<BN>(xax, [&](int g, int r, int step) {
        if (g >= live) return;
        R* base = out0 + line_start(g);
        const R* y = Y + r * BNS + g;
        const R* z = Z + g;
        R U = R(0), V = R(0);
        if (MODE == LINE_DST && p.lam) line_lambda(g, &U, &V);
#pragma unroll 2
        for (; r < rE; r += step, y += step * BNS) {
            const R e = y[0];
            if (MODE == LINE_TOEPLITZ) {
                const int j = i0r + r;
                if (r < rO) {
                    const R o = y[half * BNS];
                    base[(n - 1 - j) * st] = combine(e - o, z + (n - 1 - j) * BNS, n - 1 - j);
                    base[j * st] = combine(e + o, z + j * BNS, j);
                } else {
                    base[j * st] = combine(e, z + j * BNS, j);
                }
            } else {
                const int j = 2 * (i0r + r);
                const bool lam = MODE == LINE_DST && p.lam;
                base[j * st] = lam ? e / lambda(U, V, j) : e;
                if (r < rO) {
                    const R o = y[half * BNS];
                    base[(j + 1) * st] = lam ? o / lambda(U, V, j + 1) : o;
                }
            }
        }
    });
}

// The kernel's form of a row-major n x n matrix: form 0 unsplit, 1 symmetric
// Toeplitz (sums and differences of the two ends), 2 DST-I (rows of odd and of
// even index).  One thread per entry of the padded array.
template <typename R>
__global__ void line_matrix_kernel(const double* __restrict__ src, int n, int form, LineMatrix lm) {
    R* m = const_cast<R*>(static_cast<const R*>(lm.m));
    const int fo = n / 2, ce = (n + 1) / 2;
    const long long total = (long long)lm.K * lm.ld;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(e / lm.ld), row = (int)(e - (long long)j * lm.ld);
        double v = 0.0;
        if (form == 0) {
            if (row < n) v = src[(size_t)row * n + j];
        } else {
            const int blk = row / (2 * lm.half), in = row - blk * 2 * lm.half;
            const bool odd = in >= lm.half;
            const int r = blk * lm.half + in - (odd ? lm.half : 0);
            if (r < (odd ? fo : ce) && (!odd || j < fo)) {
                if (form == 2) v = src[(size_t)(2 * r + (odd ? 1 : 0)) * n + j];
                else if (j >= fo) v = src[(size_t)r * n + j];
                else {
                    const double a = src[(size_t)r * n + j], b = src[(size_t)r * n + n - 1 - j];
                    v = 0.5 * (odd ? a - b : a + b);
                }
            }
        }
        m[e] = (R)v;
    }
}

}  // namespace fft
}  // namespace tfde
