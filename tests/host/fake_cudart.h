// The state of the stand-in for the CUDA runtime (fake_cudart.cpp): what a test sets and reads.
#pragma once

#include <cuda_runtime_api.h>

#include <functional>
#include <string>
#include <vector>

namespace fake {
struct Launch {
    int device;
    std::string kernel;          // mangled name
    dim3 grid, block;
    size_t smem;
};
extern int device;                                             // the current device
extern std::vector<Launch> launches;
extern std::function<bool(size_t)> alloc_fails;                // whether an allocation of so many bytes fails
extern std::function<int(const std::string&)> registers;       // compiled register count of a kernel
extern std::function<int(int)> sms;                            // SMs of a device
std::vector<std::string> kernel_names();                       // of every kernel of the library
bool launched(const std::string& part);                        // a kernel whose name holds `part`
}  // namespace fake
