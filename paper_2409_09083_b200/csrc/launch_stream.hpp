// Stream of a launch, and whether the launch may overlap the one before it on that stream (launch.cuh).
#pragma once

#include <driver_types.h>

namespace ftp {
struct LaunchStream { cudaStream_t st; bool overlap; };
}  // namespace ftp
