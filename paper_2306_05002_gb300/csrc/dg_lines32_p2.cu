// Explicit instantiation of the FP32-bulk line kernels of order p = 2.
#include "dg_lines32.cuh"

namespace dgpf {
KernelSet32 lines_fp32_p2(bool viscous, bool st) { return lines_fp32_p<2>(viscous, st); }
}  // namespace dgpf
