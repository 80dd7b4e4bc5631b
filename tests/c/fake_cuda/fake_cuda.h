/* A stand-in for the CUDA runtime with any number of devices and no GPU: kernels
 * do nothing, device addresses are only handed out, and what a launch depends on
 * (the current device, the dynamic shared memory allowed there) is kept as the
 * runtime keeps it.  For tests of the library's host side. */
#pragma once
#include <string>
#include <vector>

namespace fake {

struct Launch {
  std::string name;  // mangled
  int device;
  size_t smem;
  bool overlap;  // may be set up while its predecessor runs
  bool refused;
};
extern std::vector<Launch> launches;
extern std::vector<size_t> allocations;   // bytes of every cudaMalloc
extern std::vector<std::string> refuse;   // launches of kernels with such names fail
bool launched(const char* part);          // a launch of such a kernel went through

}  // namespace fake
