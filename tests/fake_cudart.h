// What a test sees of the stand-in CUDA runtime (fake_cudart.cpp).
#pragma once

#include <stddef.h>

#include <functional>
#include <string>
#include <vector>

namespace fake {

struct Launch {
    std::string name;      // mangled kernel name
    unsigned grid;         // blocks along x
    size_t smem;           // dynamic shared memory
    bool programmatic;     // may start before the kernel in front of it has ended
    bool cooperative;
    void** args;           // valid while the launch call runs
};

extern std::vector<Launch> launches;
// Called before a launch takes effect; anything but cudaSuccess is what the launch returns.
extern std::function<int(const Launch&)> on_launch;
extern size_t alloc_limit;      // larger device allocations fail
extern int refused_allocs;

}  // namespace fake
