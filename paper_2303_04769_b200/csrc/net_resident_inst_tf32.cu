// Instance of the resident network kernel: TF32.
#define SMALL_RESIDENT_KERNEL
#include "net_resident.cuh"

namespace small {
namespace resident {

Kernel resident_kernel_tf32() { return net_resident_kernel<1>; }

}  // namespace resident
}  // namespace small
