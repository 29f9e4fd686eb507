// FP64 instantiations of the per-atom kernels: the all-FP64 terms over the cells that the FP32
// kernels certify (see dsasa_atoms.cuh).
#include "dsasa_atoms.cuh"

namespace dsasa {
cudaError_t launch_atoms_f64(const AtomArgs& a, bool grad, cudaStream_t s) { return launch_atoms_t<double>(a, grad, s); }
}  // namespace dsasa
