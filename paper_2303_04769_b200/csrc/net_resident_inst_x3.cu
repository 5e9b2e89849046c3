// Instance of the resident network kernel: 3xTF32.
#define SMALL_RESIDENT_KERNEL
#include "net_resident.cuh"

namespace small {
namespace resident {

Kernel resident_kernel_x3() { return net_resident_kernel<2>; }

}  // namespace resident
}  // namespace small
