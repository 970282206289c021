// CRT kernels for t values packed by triples of moduli (crt_kernel.cuh).
#include "crt_kernel.cuh"

namespace ozlu {

void launch_crt_packed(const CrtArgs& a, const CrtTab& tab, cudaStream_t s) { launch_crt_pack<true>(a, tab, s); }

}  // namespace ozlu
