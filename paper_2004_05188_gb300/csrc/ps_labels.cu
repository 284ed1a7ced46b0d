// Randomised type labels: the companion statistic the paper computes by
// default next to every spatial statistic, with the type labels shuffled by a
// pseudo-random generator (Suppl. "Importance of high quality random number
// generators") so that the result can be compared with a random arrangement.
//
// GPU form: no sort.  perm is a pseudo-random permutation of [0, n) that every
// thread evaluates on its own: a 4-round Feistel network on 2h bits
// (2^(2h) >= n) whose round function is the splitmix64 finaliser of
// (half-block + round key), round key r = finaliser(seed + (r + 1) * golden
// gamma), restricted to [0, n) by cycle walking.  type_out[i] = type_in[perm(i)].
#include "ps_internal.cuh"

namespace ps {

__host__ __device__ __forceinline__ uint64_t sm_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

struct FeistelKey {
  uint64_t k[4];
  uint32_t h;
};

__device__ __forceinline__ uint64_t feistel4(uint64_t x, const FeistelKey& key) {
  const uint64_t mask = (1ull << key.h) - 1ull;
  uint64_t L = x >> key.h, R = x & mask;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const uint64_t t = L ^ (sm_mix(R + key.k[r]) & mask);
    L = R;
    R = t;
  }
  return (L << key.h) | R;
}

__global__ void __launch_bounds__(256) k_shuffle_labels(const uint8_t* __restrict__ in, uint8_t* __restrict__ out,
                                                        uint32_t* __restrict__ perm, uint64_t n, FeistelKey key,
                                                        int* __restrict__ status) {
  griddep_wait();
  griddep_launch();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t domain = 1ull << (2 * key.h);
  // One step of the permutation per turn: a thread whose value is below n writes it and goes on to its
  // next ion, one whose value is not walks on along the cycle.  The lanes of a warp so never wait for
  // the longest walk among them (up to 3 of 4 values are walked on).
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, y = i, walked = 0;
  while (i < n) {
    y = feistel4(y, key);
    // the cycle through i returns below n within `domain` steps
    if (y >= n && ++walked > domain) {  // not reachable for a permutation; never read out of bounds
      if (status) atomicCAS(status, 0, (int)PS_ERR_INVALID_INPUT);
      y = i;
    }
    if (y < n) {
      out[i] = in[y];
      if (perm) perm[i] = (uint32_t)y;
      i += stride;
      y = i;
      walked = 0;
    }
  }
}

// The same permutation with the round functions in tables: a half-block has h bits, so a round maps
// 2^h values, and its 2^h results (16 bits each, four rounds) are computed once per CTA into shared
// memory, before the labels are waited for.  A step is then four table loads and a few 32-bit operations
// instead of eight 64-bit multiplications.  The label read at the end of a walk is stored a turn
// later, so that the next walk's steps run meanwhile.  Bound by the tables' bank conflicts and by latency.
// Per call, this form against the one above (us): 2e5 and 1e6 ions 15 / 15 (the launch), 3e6 21 / 59, 8e6 69 / 265,
// 1.6e7 82 / 153, 1e8 (128 KB tables) 1180 / 4367, 2e8 2684 / 3498.  Half-blocks of more than 14 bits (2.7e8 ions)
// have no room for their tables.
constexpr uint32_t kTableThreads = 1024, kTableBits = 14;  // 4 x 2^14 entries: 128 KB

__global__ void __launch_bounds__(kTableThreads) k_shuffle_labels_table(const uint8_t* __restrict__ in,
                                                                        uint8_t* __restrict__ out,
                                                                        uint32_t* __restrict__ perm, uint32_t n,
                                                                        FeistelKey key, int* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint16_t* T = reinterpret_cast<uint16_t*>(smem);  // [4][2^h]
  const uint32_t h = key.h, size = 1u << h, mask = size - 1u;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    for (uint32_t x = threadIdx.x; x < size; x += blockDim.x) T[(r << h) + x] = (uint16_t)(sm_mix(x + key.k[r]) & mask);
  __syncthreads();
  griddep_wait();
  griddep_launch();
  const uint32_t stride = gridDim.x * blockDim.x, domain = 1u << (2 * h);
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, y = i, walked = 0, last = 0;
  uint8_t label = 0;
  bool pending = false;  // label belongs to ion `last`
  while (i < n) {  // one step of the permutation per turn, as above
    uint32_t L = y >> h, R = y & mask;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t t = L ^ T[(r << h) + R];
      L = R;
      R = t;
    }
    y = (L << h) | R;
    if (y >= n && ++walked > domain) {  // not reachable for a permutation; never read out of bounds
      if (status) atomicCAS(status, 0, (int)PS_ERR_INVALID_INPUT);
      y = i;
    }
    if (y < n) {
      if (pending) out[last] = label;
      label = in[y];
      pending = true;
      last = i;
      if (perm) perm[i] = y;
      i += stride;
      y = i;
      walked = 0;
    }
  }
  if (pending) out[last] = label;
}

}  // namespace ps

using namespace ps;

extern "C" int ps_shuffle_labels(const uint8_t* type_in, uint8_t* type_out, int64_t n, uint64_t seed, uint32_t* d_perm,
                                 void* stream) {
  if (n < 0 || n > (int64_t)UINT32_MAX) return fail(PS_ERR_INVALID_ARG, "ps_shuffle_labels: n out of range");
  if (n > 0 && (!type_in || !type_out)) return fail(PS_ERR_INVALID_ARG, "ps_shuffle_labels: NULL array");
  if (n > 0 && type_in == type_out) return fail(PS_ERR_INVALID_ARG, "ps_shuffle_labels: in and out must differ");
  if (n == 0) return PS_OK;
  FeistelKey key;
  key.h = 1;
  while ((1ull << (2 * key.h)) < (uint64_t)n) ++key.h;
  for (int r = 0; r < 4; ++r) key.k[r] = sm_mix(seed + (uint64_t)(r + 1) * 0x9e3779b97f4a7c15ULL);
  int dev = 0, sms = 0;
  PS_CUDA(cudaGetDevice(&dev));
  PS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (key.h <= kTableBits) {
    const uint32_t smem = 8u << key.h, per_sm = key.h < kTableBits ? 2u : 1u;
    const uint64_t want = ((uint64_t)n + kTableThreads - 1) / kTableThreads;
    const int blocks = (int)(want < (uint64_t)sms * per_sm ? want : (uint64_t)sms * per_sm);
    if (smem > 48u << 10)  // (the largest size, whichever is needed: calls from several threads set the same)
      PS_CUDA(cudaFuncSetAttribute(k_shuffle_labels_table, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 << kTableBits));
    PS_LAUNCH(PS_KID_LABELS, s,
              PS_CUDA(launch_pdl(k_shuffle_labels_table, blocks, kTableThreads, smem, s, type_in, type_out, d_perm, (uint32_t)n,
                                 key, static_cast<int*>(nullptr))));
    PS_CUDA(cudaGetLastError());
    return PS_OK;
  }
  PS_LAUNCH(PS_KID_LABELS, s,
            PS_CUDA(launch_pdl(k_shuffle_labels, sms * 8, 256, 0, s, type_in, type_out, d_perm, (uint64_t)n, key,
                               static_cast<int*>(nullptr))));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}
