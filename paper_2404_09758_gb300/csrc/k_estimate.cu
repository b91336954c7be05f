// Small kernels around the estimators: an asset's launch descriptor (batched calls) and the image
// error of tiles that no triangle can reach.
#include <cuda_runtime.h>

#define SGE_FILE_ID 3  // range-check sites of this file (checked build)
#include "sge_device.cuh"

namespace sge {

namespace {

__global__ void k_put_desc(const AssetDesc d, AssetDesc* dst) {
  const int4* src = reinterpret_cast<const int4*>(&d);
  int4* out = reinterpret_cast<int4*>(dst);
  for (int i = threadIdx.x; i < (int)(sizeof(AssetDesc) / 16); i += blockDim.x) out[i] = src[i];
}

// Loss of pixels in tiles no triangle can reach: the background on both sides.
__global__ void k_background_loss(SceneDev S, Workspace ws, ViewList vl, float* loss) {
  const int slot = blockIdx.y, tile = blockIdx.x;
  const int ntl = n_tiles(S);
  if (ws.tile_count[slot * ntl + tile] != 0) return;
  const int view = vl.id[slot];
  const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
  const int px = tx * TILE + threadIdx.x % TILE, py = ty * TILE + threadIdx.x / TILE;
  float v = 0.0f;
  if (px < S.W && py < S.H) {
    const float* tp = S.targets + (((long long)view * S.H + py) * S.W + px) * 3;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float d = S.bg[c] - tp[c];
      v += d * d;
    }
  }
  __shared__ float red[TILE_PX / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float sum = 0.0f;
    for (int i = 0; i < TILE_PX / 32; ++i) sum += red[i];
    if (sum != 0.0f) atomicAdd(loss + slot, sum);
  }
}

}  // namespace

cudaError_t launch_put_desc(const AssetDesc& d, AssetDesc* dst, cudaStream_t st) {
  k_put_desc<<<1, 64, 0, st>>>(d, dst);
  return cudaGetLastError();
}

cudaError_t launch_background_loss(const SceneDev& S, const Workspace& ws, const ViewList& vl, float* loss,
                                   cudaStream_t st) {
  k_background_loss<<<dim3(n_tiles(S), vl.n), TILE_PX, 0, st>>>(S, ws, vl, loss);
  return cudaGetLastError();
}

}  // namespace sge
