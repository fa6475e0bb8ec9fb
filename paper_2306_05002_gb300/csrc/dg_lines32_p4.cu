// Explicit instantiation of the FP32-bulk line kernels of order p = 4.
#include "dg_lines32.cuh"

namespace dgpf {
KernelSet32 lines_fp32_p4(bool viscous, bool st) { return lines_fp32_p<4>(viscous, st); }
}  // namespace dgpf
