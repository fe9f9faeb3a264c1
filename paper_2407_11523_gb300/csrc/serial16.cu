// Serial-schedule kernels with 16 lanes per shot (serial_kernel.cuh), in a
// translation unit of their own so that they compile in parallel with the others.
#include "serial_kernel.cuh"

namespace bpq {
namespace sk {
SerialKernelFn pick_serial16(int variant, bool split) { BPQ_SERIAL_SWITCH(false, 16, 1) }
}  // namespace sk
}  // namespace bpq
