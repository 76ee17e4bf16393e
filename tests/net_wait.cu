// The network tile's waits when they run out: a CTA whose weight stream is empty
// runs the layers of a tile pair, so the first layer waits for a chunk that
// nobody copies and the others for their turns. Prints the error word, or FAIL.
#include <cstdio>
#include "mlp.cuh"

using namespace sft;

__global__ void __launch_bounds__(2 * kGroupThreads, 1) k_expire(const float* P, int32_t* err, int32_t* left) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const FwdSmem S = fwd_smem(sm);
  const LayerWeights<3> W{{nullptr, nullptr, nullptr}};
  const uint32_t taddr = fwd_setup<3>(S, P, W, 0);   // no tiles: no chunk is copied
  const TileLane t = tile_lane(S, taddr);
  uint32_t lphase = 0;
  for (int l = 0; l < 3; ++l) tile_mma<3>(S, t, W, 2 * l + t.grp, lphase, err, [] {});
  fwd_teardown(S, taddr, err);
  atomicAdd(left, 1);
}

int main() {
  float* P = nullptr;
  int32_t *d = nullptr, h[2] = {0, 0};
  bool ok = cudaMalloc(&P, sizeof(float) * kNParam) == cudaSuccess && cudaMalloc(&d, sizeof(h)) == cudaSuccess &&
            cudaMemset(P, 0, sizeof(float) * kNParam) == cudaSuccess && cudaMemset(d, 0, sizeof(h)) == cudaSuccess &&
            cudaFuncSetAttribute(k_expire, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemFwd) == cudaSuccess;
  if (ok) {
    k_expire<<<1, 2 * kGroupThreads, kSmemFwd>>>(P, d, d + 1);
    ok = cudaGetLastError() == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess &&
         cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) == cudaSuccess;
  }
  ok = ok && h[0] == DEV_BARRIER_TIMEOUT && h[1] == 2 * kGroupThreads;
  std::printf("%s err %d threads %d\n", ok ? "ok" : "FAIL", h[0], h[1]);
  return ok ? 0 : 1;
}
