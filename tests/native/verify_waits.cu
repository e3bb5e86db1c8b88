// The verification kernels as tests/test_gpu_verify_waits.py builds them: with a wait limit of a millisecond, beside a kernel that
// lets its successor start at once and then takes its time.
#include "../../paper_2510_19705_b200/csrc/sampling.cu"

__global__ void occupy_kernel(unsigned long long ns) {
  chain_next();
  const unsigned long long t0 = hsd::ptx::globaltimer_ns();
  for (int i = 0; i < (1 << 24) && hsd::ptx::globaltimer_ns() - t0 < ns; ++i) {}
}

extern "C" int occupy(unsigned long long ns, void *stream) {
  occupy_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(ns);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
