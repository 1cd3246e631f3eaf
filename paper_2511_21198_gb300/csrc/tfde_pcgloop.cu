// Device-side loop of the preconditioned CG iterations (Sec. 3.1) whose
// operator and preconditioner run on the FFT / line passes: the all-FP64 PCG
// and the FP32 inner PCG of the ragged-grid refinement.  One CUDA graph, built
// once per problem: a WHILE node whose body is one iteration, with alpha, beta,
// the stop test and the iteration count on the device.  A host-driven iteration
// reads three scalars (FP64) or one (FP32) back, and the GPU idles for each
// read: at 16^3 that was half of the time (14.9 ms for 16 steps; 7.2 ms of
// kernels).
#include <cmath>

#include "tfde_fft.h"
#include "tfde_gs.cuh"
#include "tfde_internal.h"
#include "tfde_pcgloop.h"
#include "tfde_pdl.cuh"
#include "tfde_stats.h"

namespace tfde {

namespace {

constexpr int kT = gs::kThreads;
// device scalars of the loop; kX: the address of the iterate
enum { kRZ = 0, kAlpha, kBeta, kRR, kThr, kNum };
// control words: done (skips the rest of the body), iterations, their limit,
// what ended the loop early (PCGLOOP_*)
enum { cDone = 0, cIters, cMax, cBad, cNum };

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double sh[kT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kT / 32; ++w) t += sh[w];
    return t;
}
__device__ __forceinline__ double warp_partials(const double* part, int nblk) {
    double acc = 0.0;
#pragma unroll 8
    for (int b = threadIdx.x; b < nblk; b += 32) acc += part[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    return acc;   // in lane 0
}
template <typename R>
__device__ __forceinline__ void block_range(long long N, long long& lo, long long& hi) {
    const long long per = ((N + gridDim.x - 1) / gridDim.x + 3) / 4 * 4;
    lo = min((long long)blockIdx.x * per, N);
    hi = min(lo + per, N);
}

// partial sums <a, b>: FP64 products and sums, or compensated FP32 per thread
template <typename R>
__global__ void __launch_bounds__(kT) dot_kernel(long long N, const R* a, const R* b, double* __restrict__ part,
                                                 const int* ctl) {
    pdl_begin();
    if (ctl[cDone]) return;
    long long lo, hi;
    block_range<R>(N, lo, hi);
    double t;
    if constexpr (sizeof(R) == 8) {
        double acc = 0.0;
#pragma unroll 8
        for (long long i = lo + threadIdx.x; i < hi; i += kT) acc = fma(a[i], b[i], acc);
        t = block_sum(acc);
    } else {
        gs::KSum k;
        gs::sweep(
            lo, hi, true,
            [&](long long i) {
                gs::add4(k, *reinterpret_cast<const float4*>(a + i), *reinterpret_cast<const float4*>(b + i));
            },
            [&](long long i) { k.add(a[i] * b[i]); });
        t = block_sum(k.value());
    }
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// <r, z> of the start
__global__ void first_kernel(const double* part, int nblk, double* S) {
    pdl_begin();
    const double t = warp_partials(part, nblk);
    if (threadIdx.x == 0) S[kRZ] = t;
}

// <p, A p>: alpha, or the end of the loop before anything is updated
__global__ void alpha_kernel(const double* part, int nblk, double* S, int* ctl) {
    pdl_begin();
    const double pq = warp_partials(part, nblk);
    if (threadIdx.x) return;
    S[kAlpha] = S[kRZ] / pq;
    if (!isfinite(pq)) ctl[cBad] = PCGLOOP_NAN_PAP;
    else if (!(pq > 0.0)) ctl[cBad] = PCGLOOP_BREAKDOWN;
}

// x += alpha p; r -= alpha q; partial sums of r.r (FP64 products and sums)
template <typename R>
__global__ void __launch_bounds__(kT) update_kernel(long long N, const double* S, const R* __restrict__ p,
                                                    const R* __restrict__ q, R* const* xp, R* __restrict__ r,
                                                    double* __restrict__ part, const int* ctl) {
    pdl_begin();
    if (ctl[cBad]) return;
    R* __restrict__ x = *xp;
    const R alpha = (R)S[kAlpha];
    long long lo, hi;
    block_range<R>(N, lo, hi);
    double acc = 0.0;
    auto one = [&](R pi, R qi, R& xi, R& ri) {
        xi = fma(alpha, pi, xi);
        ri = fma(-alpha, qi, ri);
        acc = fma((double)ri, (double)ri, acc);
    };
    if constexpr (sizeof(R) == 8) {
#pragma unroll 4
        for (long long i = lo + threadIdx.x; i < hi; i += kT) {
            R xi = x[i], ri = r[i];
            one(p[i], q[i], xi, ri);
            x[i] = xi;
            r[i] = ri;
        }
    } else {
        gs::sweep(
            lo, hi, true,
            [&](long long i) {
                const float4 pv = *reinterpret_cast<const float4*>(p + i), qv = *reinterpret_cast<const float4*>(q + i);
                float4 xv = *reinterpret_cast<float4*>(x + i), rv = *reinterpret_cast<float4*>(r + i);
                one(pv.x, qv.x, xv.x, rv.x);
                one(pv.y, qv.y, xv.y, rv.y);
                one(pv.z, qv.z, xv.z, rv.z);
                one(pv.w, qv.w, xv.w, rv.w);
                *reinterpret_cast<float4*>(x + i) = xv;
                *reinterpret_cast<float4*>(r + i) = rv;
            },
            [&](long long i) {
                R xi = x[i], ri = r[i];
                one(p[i], q[i], xi, ri);
                x[i] = xi;
                r[i] = ri;
            });
    }
    const double t = block_sum(acc);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// the stop test and the loop condition
__global__ void stop_kernel(const double* part, int nblk, double* S, int* ctl, cudaGraphConditionalHandle h) {
    pdl_begin();
    const double rr = warp_partials(part, nblk);
    if (threadIdx.x) return;
    int done = 1;
    if (!ctl[cBad]) {
        const int k = ++ctl[cIters];
        S[kRR] = rr;
        if (!isfinite(rr)) ctl[cBad] = PCGLOOP_NAN_RR;
        else done = rr <= S[kThr] || k >= ctl[cMax];
    }
    ctl[cDone] = done;
    cudaGraphSetConditional(h, done ? 0u : 1u);
}

// <r, z>: beta
__global__ void beta_kernel(const double* part, int nblk, double* S, const int* ctl) {
    pdl_begin();
    if (ctl[cDone]) return;
    const double t = warp_partials(part, nblk);
    if (threadIdx.x) return;
    S[kBeta] = t / S[kRZ];
    S[kRZ] = t;
}

// p = z + beta p
template <typename R>
__global__ void __launch_bounds__(kT) direction_kernel(long long N, const double* S,
                                                       const R* __restrict__ z, R* __restrict__ p, const int* ctl) {
    pdl_begin();
    if (ctl[cDone]) return;
    const R beta = (R)S[kBeta];
    long long lo, hi;
    block_range<R>(N, lo, hi);
    if constexpr (sizeof(R) == 8) {
#pragma unroll 4
        for (long long i = lo + threadIdx.x; i < hi; i += kT) p[i] = fma(beta, p[i], z[i]);
    } else {
        gs::sweep(
            lo, hi, true,
            [&](long long i) {
                const float4 zv = *reinterpret_cast<const float4*>(z + i);
                float4 pv = *reinterpret_cast<float4*>(p + i);
                pv = make_float4(fmaf(beta, pv.x, zv.x), fmaf(beta, pv.y, zv.y), fmaf(beta, pv.z, zv.z),
                                 fmaf(beta, pv.w, zv.w));
                *reinterpret_cast<float4*>(p + i) = pv;
            },
            [&](long long i) { p[i] = fma(beta, p[i], z[i]); });
    }
}

__global__ void start_kernel(double* S, int* ctl, void** xp, double thr, int maxit, void* x) {
    S[kThr] = thr;
    ctl[cDone] = 0;
    ctl[cIters] = 0;
    ctl[cMax] = maxit;
    ctl[cBad] = 0;
    *xp = x;
}

struct Loop {
    double* S = nullptr;    // kNum scalars, then the iterate's address, then the control words
    double* host = nullptr; // pinned mirror
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    bool failed = false;
    void** xp() const { return reinterpret_cast<void**>(S + kNum); }
    int* ctl() const { return reinterpret_cast<int*>(S + kNum + 1); }
};
constexpr size_t kWords = kNum + 1 + (cNum + 1) / 2;
constexpr int kBodyLaunches = 7;   // besides the operator's and the preconditioner's

int grid_for(size_t N) {
    const long long g = ((long long)N + 4 * kT - 1) / (4 * kT);
    return (int)(g > 304 * 4 ? 304 * 4 : (g < 1 ? 1 : g));
}

void release(Loop* L) {
    if (L->exec) cudaGraphExecDestroy(L->exec);
    if (L->graph) cudaGraphDestroy(L->graph);
    cudaFree(L->S);
    if (L->host) cudaFreeHost(L->host);
    delete L;
}

// The problem's loop with both of its buffers, or null (no memory for them).
template <typename R>
Loop* loop_of(const tfde_problem* P) {
    void*& slot = P->pcg_loop[sizeof(R) == 8 ? 0 : 1];
    if (!slot) {
        Loop* L = new Loop();
        if (cudaMalloc((void**)&L->S, kWords * sizeof(double)) != cudaSuccess ||
            cudaMallocHost((void**)&L->host, kWords * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            release(L);
            return nullptr;
        }
        slot = L;
    }
    return static_cast<Loop*>(slot);
}

template <typename R>
int build(const tfde_problem* P, Loop* L, const PcgLoopVectors<R>& v, cudaStream_t s) {
    if (L->exec || L->failed) return TFDE_OK;
    const int nblk = dot_blocks(P->nblk);
    const bool early = nblk <= kPdlBlocks;
    // once outside the capture: the passes' launch attributes are set on first use
    int st = fft::apply_A<R>(P, TFDE_OP_A, v.p, v.q, v.t[0], v.t[1], v.t[2], v.t[3], s);
    if (!st) st = fft::apply_Pinv<R>(P, v.r, v.z, v.t[0], v.t[2], s);
    if (st) return st;
    cudaGraphConditionalHandle h{};
    cudaGraphNodeParams cp = {};
    cudaGraphNode_t node;
    bool ok = cudaGraphCreate(&L->graph, 0) == cudaSuccess;
    if (ok) ok = cudaGraphConditionalHandleCreate(&h, L->graph, 1, cudaGraphCondAssignDefault) == cudaSuccess;
    if (ok) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        ok = cudaGraphAddNode(&node, L->graph, nullptr, nullptr, 0, &cp) == cudaSuccess;
    }
    const cudaStream_t c = capture_stream();   // the caller's may be the legacy default stream
    if (ok)
        ok = cudaStreamBeginCaptureToGraph(c, cp.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                           cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
        stats_set_capturing(true);
        const long long N = (long long)P->N;
        double* part = P->red;
        double* S = L->S;
        int* ctl = L->ctl();
        st = fft::apply_A<R>(P, TFDE_OP_A, v.p, v.q, v.t[0], v.t[1], v.t[2], v.t[3], c);
        launch_pdl(early, dot_kernel<R>, nblk, kT, c, N, v.p, v.q, part, ctl);
        launch_pdl(early, alpha_kernel, 1, 32, c, part, nblk, S, ctl);
        launch_pdl(early, update_kernel<R>, nblk, kT, c, N, S, v.p, v.q, reinterpret_cast<R* const*>(L->xp()), v.r, part, ctl);
        launch_pdl(early, stop_kernel, 1, 32, c, part, nblk, S, ctl, h);
        if (!st) st = fft::apply_Pinv<R>(P, v.r, v.z, v.t[0], v.t[2], c, ctl + cDone);
        launch_pdl(early, dot_kernel<R>, nblk, kT, c, N, v.r, v.z, part, ctl);
        launch_pdl(early, beta_kernel, 1, 32, c, part, nblk, S, ctl);
        launch_pdl(early, direction_kernel<R>, grid_for(P->N), kT, c, N, S, v.z, v.p, ctl);
        stats_set_capturing(false);
        cudaGraph_t out = nullptr;
        const cudaError_t e = cudaStreamEndCapture(c, &out);
        ok = st == TFDE_OK && e == cudaSuccess;
    }
    if (ok) ok = cudaGraphInstantiate(&L->exec, L->graph, 0) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        if (L->graph) cudaGraphDestroy(L->graph);
        L->graph = nullptr;
        L->exec = nullptr;
        L->failed = true;   // the host-driven iterations stay in use
        set_error(TFDE_OK, "");
    }
    return TFDE_OK;
}

}  // namespace

template <typename R>
int pcg_loop_reserve(const tfde_problem* P) {
    return loop_of<R>(P) ? TFDE_OK : set_error(TFDE_ENOMEM, "allocation of the PCG loop's scalars failed");
}
template int pcg_loop_reserve<double>(const tfde_problem*);
template int pcg_loop_reserve<float>(const tfde_problem*);

template <typename R>
int pcg_loop(const tfde_problem* P, const PcgLoopVectors<R>& v, R* x, double thr, int maxit, PcgLoopResult* res,
             cudaStream_t s) {
    res->ran = false;
    if (!P->fft || !P->device_loop || stats_timing() || maxit < 1) return TFDE_OK;
    Loop* L = loop_of<R>(P);   // there since assembly, but for a mixed solve's FP64 fallback
    if (!L) return TFDE_OK;
    if (int st = build<R>(P, L, v, s)) return st;
    if (!L->exec) return TFDE_OK;
    const int nblk = dot_blocks(P->nblk);
    int* ctl = L->ctl();
    stats_count_launch(4);
    start_kernel<<<1, 1, 0, s>>>(L->S, ctl, L->xp(), thr, maxit, x);
    if (int st = fft::apply_Pinv<R>(P, v.r, v.p, v.t[0], v.t[2], s)) return st;   // p_0 = z_0 = P^{-1} r_0
    dot_kernel<R><<<nblk, kT, 0, s>>>((long long)P->N, v.r, v.p, P->red, ctl);
    first_kernel<<<1, 32, 0, s>>>(P->red, nblk, L->S);
    if (cudaGraphLaunch(L->exec, s) != cudaSuccess ||
        cudaMemcpyAsync(L->host, L->S, kWords * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return set_error(TFDE_ECUDA, std::string("PCG loop: ") + cudaGetErrorString(cudaGetLastError()));
    const int* hc = reinterpret_cast<const int*>(L->host + kNum + 1);
    res->ran = true;
    res->iters = hc[cIters];
    res->bad = hc[cBad];
    res->rr = L->host[kRR];
    stats_count_launch((unsigned)(res->iters > 0 ? res->iters : 1) *
                       (kBodyLaunches + (unsigned)fft::operator_launches(P) + (unsigned)fft::preconditioner_launches<R>(P)));
    return TFDE_OK;
}
template int pcg_loop<double>(const tfde_problem*, const PcgLoopVectors<double>&, double*, double, int, PcgLoopResult*,
                              cudaStream_t);
template int pcg_loop<float>(const tfde_problem*, const PcgLoopVectors<float>&, float*, double, int, PcgLoopResult*,
                             cudaStream_t);

void pcg_loop_free(tfde_problem* P) {
    for (void*& slot : P->pcg_loop) {
        if (slot) release(static_cast<Loop*>(slot));
        slot = nullptr;
    }
}

}  // namespace tfde
