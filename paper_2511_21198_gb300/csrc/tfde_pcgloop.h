// Device-side PCG loop on the FFT / line passes (tfde_pcgloop.cu).
#pragma once

#include "tfde_internal.h"

namespace tfde {

// The problem's own vectors: residual, preconditioned residual, direction,
// operator output and the passes' four intermediates.  The loop's graph keeps
// their addresses, so they are the same for every solve of a problem.
template <typename R>
struct PcgLoopVectors {
    R *r, *z, *p, *q, *t[4];
};
// what ended the loop before its stop test: <p, A p> not finite (nothing
// updated) or not positive (nothing updated), <r, r> not finite
enum { PCGLOOP_OK = 0, PCGLOOP_NAN_PAP = 1, PCGLOOP_BREAKDOWN = 2, PCGLOOP_NAN_RR = 3 };
struct PcgLoopResult {
    bool ran = false;   // false: switched off, no graph or no memory (the caller iterates from the host)
    int iters = 0, bad = PCGLOOP_OK;
    double rr = 0.0;    // <r, r> of the recursive residual
};

// Allocates the loop's scalars (assembly of a problem whose solves take it).
template <typename R>
int pcg_loop_reserve(const tfde_problem* P);
// PCG on A x = b from the residual in v.r (p = P^{-1} r first) until <r, r> <=
// thr or maxit iterations; x is updated in place.  One host read.
template <typename R>
int pcg_loop(const tfde_problem* P, const PcgLoopVectors<R>& v, R* x, double thr, int maxit, PcgLoopResult* res,
             cudaStream_t s);
void pcg_loop_free(tfde_problem* P);

}  // namespace tfde
