// The passes after the first of the volume-preserving step's radix selection
// (mbo_select.cuh; the first is fused with the keys, k_vp_delta).
#include <algorithm>

#include "mbo_select.cuh"

namespace mbo {

// Key digit d (1 .. 5), then index digits (d - 6) of an index of `bits` bits.
__global__ void __launch_bounds__(kSelThreads)
k_select_pass(const unsigned long long* __restrict__ keys, long long P, SelectState* ss, int d, int bits) {
  __shared__ unsigned int h[kSelBins];
  __shared__ unsigned int part[kSelThreads / 32];
  __shared__ int s_flag;
  if (ss->done) return;
  const unsigned long long hi = ss->hi, k = ss->k;
  const unsigned int lo = ss->lo;
  sel_clear(h);
  int sh, w;
  const bool on_key = d < kSelKeyPasses;
  if (on_key) key_digit(d, sh, w);
  else idx_digit(bits, d - kSelKeyPasses, sh, w);
  const unsigned int mask = (1u << w) - 1;
  const int up = sh + w;  // <= 53 for a key digit, <= 32 for an index digit
  const long long step = (long long)gridDim.x * kSelThreads;
#pragma unroll 4
  for (long long x = blockIdx.x * (long long)kSelThreads + threadIdx.x; x < P; x += step) {
    const unsigned long long key = keys[x];
    if (on_key) {
      if (key >> up == hi >> up) atomicAdd(&h[(unsigned)(key >> sh) & mask], 1u);
    } else if (key == hi && (unsigned long long)x >> up == (unsigned long long)lo >> up) {
      atomicAdd(&h[(unsigned)((unsigned)x >> sh) & mask], 1u);
    }
  }
  if (!sel_flush(h, ss, &s_flag)) return;
  int digit = 0;
  unsigned long long rest = 0;
  bool whole = false;
  if (!sel_pick(ss, k, part, digit, rest, whole)) return;
  if (on_key) {
    sel_record_key(ss, hi, d, digit, rest, whole);
  } else {
    ss->lo = lo | (unsigned)digit << sh | (whole ? (1u << sh) - 1 : 0u);
    ss->k = rest;
    ss->done = whole ? 1 : 0;
  }
}

cudaError_t launch_select(const unsigned long long* keys, long long P, SelectState* ss, int blocks,
                          cudaStream_t s) {
  int bits = 1;
  while (bits < 32 && (1ll << bits) < P) ++bits;
  const int passes = kSelKeyPasses + (bits + 10) / 11;
  for (int d = 1; d < passes; ++d) k_select_pass<<<blocks, kSelThreads, 0, s>>>(keys, P, ss, d, bits);
  return cudaGetLastError();
}

}  // namespace mbo
