// Instance of the resident network kernel: FP32.
#define SMALL_RESIDENT_KERNEL
#include "net_resident.cuh"

namespace small {
namespace resident {

Kernel resident_kernel_fp32() { return net_resident_kernel<0>; }

}  // namespace resident
}  // namespace small
