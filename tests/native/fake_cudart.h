// Controls and counters of fake_cudart.cpp.
#pragma once
#include <cstddef>
#include <functional>
#include <set>

struct FakeCuda {
    int device_allocs = 0, host_allocs = 0;   // calls so far
    int fail_device = 0, fail_host = 0;       // fail the k-th call from now (0: none)
    int null_copies = 0, graph_launches = 0;
    std::set<void*> live;                     // allocations not freed
    int allocs_at_graph = 0;                  // allocations before the last graph launch
    std::function<void(void*, size_t)> on_copy;
};
extern FakeCuda fake;
