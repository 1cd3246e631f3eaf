// The buffers of the device-side loops: allocated with the problem, both or
// neither, and a solve that finds no memory for them iterates from the host.
// Prints one line per failed check; exit status 1 on any.
#include <cstdio>

#include "fake_cudart.h"
#include "tfde.h"
#include "tfde_internal.h"

namespace tfde {
int pcg64(const tfde_problem*, const double*, double*, double, int, tfde_info*, cudaStream_t, bool);
}

static int failures = 0;
static void check(bool ok, const char* what) {
    if (ok) return;
    std::printf("FAILED: %s\n", what);
    ++failures;
}

static tfde_params params(int n1, int n2, int n3, bool sym) {
    tfde_params p{};
    const int n[3] = {n1, n2, n3};
    for (int a = 0; a < 3; ++a) {
        p.n[a] = n[a];
        p.lo[a] = 0.0;
        p.hi[a] = 1.0;
        p.delta[a] = 0.5;
        p.kp[a] = 1.0;
        p.km[a] = sym ? 1.0 : 0.5;
    }
    p.dt = 0.1;
    return p;
}

int main() {
    static double b[4096], x[4096];
    for (int mixed = 0; mixed < 2; ++mixed)
        for (int sym = 0; sym < 2; ++sym) {
            const tfde_params p = params(15, 16, 17, sym);
            tfde_problem* P = nullptr;
            check(tfde_assemble(&p, mixed ? TFDE_MIXED : TFDE_FP64, nullptr, &P) == TFDE_OK, "assembly");
            // a solve allocates nothing; a mixed one up to its loops (sums of ones
            // do not converge, so it goes on to the FP64 fallback, which may)
            const int before = fake.device_allocs + fake.host_allocs, launched = fake.graph_launches;
            if (sym) tfde_pcg(P, b, x, 1e-9, 3, nullptr, nullptr);
            else tfde_pgmres(P, b, x, 20, 1e-9, 3, nullptr, nullptr);
            if (sym || mixed) check(fake.graph_launches > launched, "the solve runs as a graph");
            const int after = mixed ? fake.allocs_at_graph : fake.device_allocs + fake.host_allocs;
            check(after == before, "the first solve allocates nothing");
            tfde_destroy(P);
        }
    check(fake.live.empty(), "everything is freed");

    // assembly without memory for the pinned mirrors: the usual status, nothing kept
    const tfde_params p = params(16, 16, 16, true);
    tfde_problem* P = nullptr;
    fake.fail_host = 2;   // the first pinned block is the reductions'
    check(tfde_assemble(&p, TFDE_FP64, nullptr, &P) == TFDE_ENOMEM, "assembly reports the failed allocation");
    fake.fail_host = 0;
    check(fake.live.empty(), "a failed assembly keeps nothing");

    // the FP64 fallback of a tensor-core problem allocates its loop on first use
    check(tfde_assemble(&p, TFDE_MIXED, nullptr, &P) == TFDE_OK, "assembly");
    for (int device = 0; device < 2; ++device) {
        (device ? fake.fail_device : fake.fail_host) = 1;
        const int launched = fake.graph_launches;
        const int st = tfde::pcg64(P, b, x, 1e-9, 3, nullptr, nullptr, false);
        check(st == TFDE_ENOCONV, "without memory the host iterates");   // three iterations of ones
        check(fake.graph_launches == launched, "no graph without its buffers");
        fake.fail_device = fake.fail_host = 0;
    }
    const int launched = fake.graph_launches;
    tfde::pcg64(P, b, x, 1e-9, 3, nullptr, nullptr, false);
    check(fake.graph_launches > launched, "with memory again the loop runs");
    check(fake.null_copies == 0, "no copy to or from null");
    tfde_destroy(P);
    check(fake.live.empty(), "everything is freed");
    if (!failures) std::printf("ok\n");
    return failures != 0;
}
