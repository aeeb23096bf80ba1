// A CUDA runtime made of host memory: allocations can be made to fail, kernels are recorded instead of run.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <functional>
#include <map>
#include <string>

namespace fake {

extern std::map<void*, size_t> live;  // "device" memory
extern std::map<std::string, int> launched;
extern std::function<void(const std::string&, void**)> on_launch;  // kernel (mangled), arguments
extern std::function<void(void*, size_t)> on_copy;                 // after a copy
extern int64_t allocs, fail_from, fail_count;  // allocations number fail_from .. + fail_count - 1 fail
extern size_t used, peak, capacity;
extern bool no_streams;  // streams cannot be created
extern int graph_launches, graphs;

[[noreturn]] void die(const char* fmt, ...);
bool named(const std::string& mangled, const char* kernel);
int launches(const char* kernel);
void need(const char* what, const void* p, size_t bytes);  // a live allocation of at least `bytes` starts at p

}  // namespace fake
