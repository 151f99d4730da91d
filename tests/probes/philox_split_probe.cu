// Test probe: the merge kernels' Philox4x32-10, whose first two rounds are made once per group
// and once per expert, for any counter (g low, g high, expert, tag) and key.
#include "philox.cuh"

__global__ void probe(const uint4* ctr, const uint2* key, unsigned n, uint4* out) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  uint32_t rk[10][2];
  for (int r = 0; r < 10; ++r) {
    rk[r][0] = key[t].x + (uint32_t)r * 0x9E3779B9u;
    rk[r][1] = key[t].y + (uint32_t)r * 0xBB67AE85u;
  }
  const uint4 c = ctr[t];
  const mp::Philox4 w = mp::philox_finish(mp::philox_group(c.x, c.w, rk), mp::philox_expert(c.y, c.z, rk), rk);
  out[t] = make_uint4(w.w[0], w.w[1], w.w[2], w.w[3]);
}

extern "C" int philox_split_probe(const void* ctr, const void* key, unsigned n, void* out) {
  probe<<<(n + 127) / 128, 128>>>((const uint4*)ctr, (const uint2*)key, n, (uint4*)out);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : -1;
}
