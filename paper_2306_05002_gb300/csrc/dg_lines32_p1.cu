// Explicit instantiation of the FP32-bulk line kernels of order p = 1.
#include "dg_lines32.cuh"

namespace dgpf {
KernelSet32 lines_fp32_p1(bool viscous, bool st) { return lines_fp32_p<1>(viscous, st); }
}  // namespace dgpf
