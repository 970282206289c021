// CRT kernels for t values stored as bytes (crt_kernel.cuh).
#include "crt_kernel.cuh"

namespace ozlu {

void launch_crt_bytes(const CrtArgs& a, const CrtTab& tab, cudaStream_t s) { launch_crt_pack<false>(a, tab, s); }

}  // namespace ozlu
