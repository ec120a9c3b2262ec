// atomo_decode_spectral_static: the spectral decode for callers that must not allocate and have no context.
//
// Some callers cannot afford a cudaMalloc at decode time: a training process whose framework allocator has already
// reserved the whole device (a raw cudaMalloc then fails or fragments the pool), a decode issued from a latency-critical
// section where cudaMalloc's device-wide synchronisation would stall every other stream, or a memory-capped job that is
// not allowed to grow.  The layers' descriptors travel as kernel arguments, so the call needs no device memory of its own,
// no copy and no state shared between calls.
#include "atomo_kernels.cuh"

using namespace atomo;

extern "C" int atomo_decode_spectral_static(int device, const void* payload, const int64_t* rows, const int64_t* cols,
                                            float* const* out, int32_t n_layers, void* stream) {
  constexpr int kMaxDevices = 64, kTileRows = 64, kTileCols = 1024;
  if (device < 0 || device >= kMaxDevices || !payload || !rows || !cols || !out || n_layers <= 0)
    return ATOMO_ERR_INVALID_ARG;
  if (n_layers > ATOMO_STATIC_MAX_LAYERS) return ATOMO_ERR_CAPACITY;
  int64_t n_tiles = 0;
  for (int l = 0; l < n_layers; ++l) {
    if (!out[l] || rows[l] <= 0 || cols[l] <= 0) return ATOMO_ERR_INVALID_ARG;
    n_tiles += ((rows[l] + kTileRows - 1) / kTileRows) * ((cols[l] + kTileCols - 1) / kTileCols);
    if (n_tiles > ATOMO_STATIC_MAX_TILES) return ATOMO_ERR_CAPACITY;
  }
  if (cudaSetDevice(device) != cudaSuccess) return ATOMO_ERR_CUDA;
  launch_sp_decode(static_cast<const uint8_t*>(payload), nullptr, 1, rows, cols, out, n_layers, (cudaStream_t)stream);
  return cudaGetLastError() == cudaSuccess ? ATOMO_OK : ATOMO_ERR_CUDA;
}
