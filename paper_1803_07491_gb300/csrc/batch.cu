// Small jobs of a structure build and of the solvers' loops, several to a
// launch: what costs at a few hundred atoms is the number of launches and
// copies (2 to 3 us each), not their work.
#include "kernels.h"

namespace {

// Zeroes the pieces: one block per piece and 4,096 words.
__global__ void __launch_bounds__(256) k_zero(ZeroArgs z) {
  int b = blockIdx.x, q = 0;
  while (b >= z.blocks[q]) b -= z.blocks[q++];
  const long long lo = (long long)b * ZERO_WORDS;
  const long long hi = lo + ZERO_WORDS < z.words[q] ? lo + ZERO_WORDS : z.words[q];
  for (long long i = lo + threadIdx.x; i < hi; i += 256) z.p[q][i] = 0u;
}

// Copies the pieces to pinned host memory.  Three copies of a few bytes took
// 9 us, one launch 4 us.
__global__ void __launch_bounds__(256) k_collect(CollectArgs a) {
  for (int q = 0; q < a.n; q++)
    for (int i = threadIdx.x; i < a.words[q]; i += 256) a.dst[a.at[q] + i] = __ldcg(a.src[q] + i);
}

// Exclusive prefix sums of up to two arrays of at most SCAN_SMALL elements,
// one block each.
template <class Tin, class Tout>
__global__ void __launch_bounds__(1024) k_scan_small(const Tin* in0, Tout* out0, const Tin* in1, Tout* out1, int n) {
  __shared__ Tout part[32];
  const Tin* in = blockIdx.x == 0 ? in0 : in1;
  Tout* out = blockIdx.x == 0 ? out0 : out1;
  constexpr int PER = SCAN_SMALL / 1024;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int per = (n + 1023) / 1024;  // elements of a thread, at most PER
  Tout v[PER], sum = 0;
#pragma unroll
  for (int q = 0; q < PER; q++) {
    const int i = tid * per + q;
    v[q] = q < per && i < n ? (Tout)in[i] : Tout(0);
    sum += v[q];
  }
  Tout inc = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const Tout t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) part[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    Tout p = part[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const Tout t = __shfl_up_sync(0xffffffffu, p, o);
      if (lane >= o) p += t;
    }
    part[lane] = p;
  }
  __syncthreads();
  Tout run = inc - sum + (wid > 0 ? part[wid - 1] : Tout(0));
#pragma unroll
  for (int q = 0; q < PER; q++) {
    const int i = tid * per + q;
    if (q < per && i < n) out[i] = run;
    run += v[q];
  }
}

int ok() { return cudaGetLastError() == cudaSuccess ? 0 : -1; }

}  // namespace

int launch_zero(ZeroArgs z, cudaStream_t s) {
  int blocks = 0;
  for (int q = 0; q < z.n; q++) blocks += z.blocks[q] = (int)((z.words[q] + ZERO_WORDS - 1) / ZERO_WORDS);
  if (blocks == 0) return 0;
  k_zero<<<blocks, 256, 0, s>>>(z);
  return ok();
}

int launch_collect(const CollectArgs& a, cudaStream_t s) {
  k_collect<<<1, 256, 0, s>>>(a);
  return ok();
}

template <class Tin, class Tout>
int launch_scan_small(const Tin* in0, Tout* out0, const Tin* in1, Tout* out1, int n, cudaStream_t s) {
  if (n < 1) return 0;
  k_scan_small<Tin, Tout><<<in1 != nullptr ? 2 : 1, 1024, 0, s>>>(in0, out0, in1, out1, n);
  return ok();
}
template int launch_scan_small<int, int>(const int*, int*, const int*, int*, int, cudaStream_t);
template int launch_scan_small<int, long long>(const int*, long long*, const int*, long long*, int, cudaStream_t);
template int launch_scan_small<long long, long long>(const long long*, long long*, const long long*, long long*, int,
                                                     cudaStream_t);
