// Radix selection of the n_plus smallest (key, index) pairs, for the
// volume-preserving step (Sec. 7: the n_plus points of largest dE take the
// SO(n) class; the key is dE complemented so that smaller keys are larger dE,
// and the grid index breaks ties, lower index first).  MSB-first passes over
// 11-bit digits: six of the 64-bit key, then as many of the index as its range
// has.  Each pass histograms its digit in shared memory among the points that
// match the prefix found so far, and the last block of the grid to finish picks
// the bucket that holds the remaining rank, with a scan over the buckets by all
// of its threads.  The passes end early: once every point of the picked bucket
// is wanted the threshold is known, and the kernels that follow return at once
// (a real-valued dE usually leaves one candidate after three or four passes;
// 1024^2 points: 170 us for twelve 8-bit passes, each with a one-thread pick
// kernel, -> 25 us).
#pragma once
#include "mbo_dev.cuh"

namespace mbo {

constexpr int kSelThreads = 256;
constexpr int kSelPer = kSelBins / kSelThreads;
constexpr int kSelKeyPasses = 6;  // 11-bit digits of a 64-bit key: 53, 42, 31, 20, 9 and the last 9 bits

// Low bit and width of key digit d.
__device__ __forceinline__ void key_digit(int d, int& shift, int& width) {
  shift = d < 5 ? 53 - 11 * d : 0;
  width = d < 5 ? 11 : 9;
}
// Low bit and width of index digit j of an index of `bits` bits.
__device__ __forceinline__ void idx_digit(int bits, int j, int& shift, int& width) {
  const int top = bits - 11 * j;
  width = top < 11 ? top : 11;
  shift = top - width;
}

__device__ __forceinline__ void sel_clear(unsigned int* h) {
#pragma unroll
  for (int i = 0; i < kSelPer; ++i) h[threadIdx.x + i * kSelThreads] = 0;
  __syncthreads();
}

// The block's histogram into the grid's; the last block returns true.
__device__ __forceinline__ bool sel_flush(const unsigned int* h, SelectState* ss, int* s_flag) {
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSelPer; ++i) {
    const int b = threadIdx.x + i * kSelThreads;
    if (h[b]) atomicAdd(&ss->hist[b], h[b]);
  }
  return last_to_arrive(&ss->count, gridDim.x, s_flag);
}

// Last block: the bucket that holds rank k (1-based), the rank inside it, and
// whether the whole bucket is wanted; the grid's histogram is cleared for the
// next pass.  The caller writes the digit (thread with `mine`).
__device__ __forceinline__ bool sel_pick(SelectState* ss, unsigned long long k, unsigned int* part,
                                         int& digit, unsigned long long& rest, bool& whole) {
  const int tid = threadIdx.x;
  unsigned int c[kSelPer], sum = 0;
#pragma unroll
  for (int i = 0; i < kSelPer; ++i) c[i] = __ldcg(&ss->hist[tid * kSelPer + i]);
#pragma unroll
  for (int i = 0; i < kSelPer; ++i) {
    sum += c[i];
    ss->hist[tid * kSelPer + i] = 0;
  }
  // exclusive prefix of the threads' sums (counts stay below 2^32 points)
  unsigned int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int v = __shfl_up_sync(0xffffffffu, inc, o);
    if ((tid & 31) >= o) inc += v;
  }
  __syncthreads();
  if ((tid & 31) == 31) part[tid >> 5] = inc;
  __syncthreads();
  unsigned long long cum = inc - sum;
  for (int w = 0; w < (tid >> 5); ++w) cum += part[w];
  bool mine = false;
  if (cum < k && k <= cum + sum) {
    mine = true;
#pragma unroll
    for (int i = 0; i < kSelPer; ++i) {
      if (k <= cum + c[i]) {
        digit = tid * kSelPer + i;
        rest = k - cum;
        whole = rest == c[i];
        break;
      }
      cum += c[i];
    }
  }
  if (tid == 0) ss->count = 0;
  return mine;
}

// Record key digit d in the state (by the thread that found it).
__device__ __forceinline__ void sel_record_key(SelectState* ss, unsigned long long hi, int d, int digit,
                                               unsigned long long rest, bool whole) {
  int sh, w;
  key_digit(d, sh, w);
  hi |= (unsigned long long)digit << sh;
  if (whole) hi |= (1ull << sh) - 1;  // the rest of the bucket: any lower bits, any index
  ss->hi = hi;
  ss->lo = whole ? ~0u : 0u;
  ss->k = rest;
  ss->done = whole ? 1 : 0;
}

}  // namespace mbo
