// Fitness from device-resident logits without any device allocation: one kernel that keeps the
// per-pair losses of a cell on chip. It is for callers that cannot call cudaMalloc at the time they
// need the fitness (a serving loop whose device memory another allocator has fully reserved, or a
// latency-critical path that cannot take the implicit synchronisation of cudaMalloc / cudaFree).
#include "engine.h"
#include "lipz.h"

extern "C" LIPZ_API int lipz_fitness_from_logits_noalloc(const float* logits, int32_t cells,
                                                         int32_t batch, float* fit_g,
                                                         float* fit_d, void* stream) {
  if (!logits || !fit_g || !fit_d) return LIPZ_ERR_INVALID;
  if (cells < 1 || cells > LIPZ_NOALLOC_MAX_CELLS || batch < 1) return LIPZ_ERR_INVALID;
  // clear an error left by an unrelated earlier call, so that the check after the launch
  // reports this launch only
  cudaGetLastError();
  lipz::launch_fitness(logits, cells, batch, nullptr, nullptr, fit_g, fit_d, nullptr,
                       static_cast<cudaStream_t>(stream));
  if (cudaGetLastError() != cudaSuccess) return LIPZ_ERR_CUDA;
  return LIPZ_OK;
}
