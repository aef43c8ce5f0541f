// The learned-terminator network 18 -> 128 -> 128 -> 10 (GELU): training
// (FP32 forward and reverse of a batch in one kernel, then the sum of its
// partial gradients, then Adam) and inference (bfloat16 weights, FP32 or FP64
// activations) as tiled GEMMs with fused bias / GELU / GELU-derivative
// epilogues (FP32 on the tensor pipe, FP64 as SIMT tiles), plus the bop_mlp
// object of the C ABI.
//
// The layers are small dense contractions (K = 18, 128, 10) applied to
// every orbital of a structure (hundreds of thousands of rows).  Every
// reduction (weight gradients over a batch, the loss, the bias gradients, the
// normalisation statistics) runs in a fixed order, so training is
// deterministic.
#include <cuda_bf16.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>

#include "../../include/bopgb.h"
#include "kernels.h"

namespace {

constexpr int NI = BOP_MLP_NIN, NH = BOP_MLP_NHID, NO = BOP_MLP_NOUT;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NI, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NO * NH, NPAR = OFF_B3 + NO;
static_assert(NPAR == BOP_MLP_NPARAM, "parameter layout");
constexpr int NORM_XM = 0, NORM_XS = NI, NORM_LO = 2 * NI, NORM_HI = 3 * NI, NORM_YM = 4 * NI,
              NORM_YS = 4 * NI + NO;
static_assert(NORM_YS + NO == BOP_MLP_NNORM, "normalisation layout");

constexpr int GBM = 64, GBN = 64, GBK = 16, GT = 256;
constexpr int RT = 256;

__device__ __forceinline__ float ncdf(float x) { return normcdff(x); }
__device__ __forceinline__ double ncdf(double x) { return normcdf(x); }
__device__ __forceinline__ float nexp(float x) { return expf(x); }
__device__ __forceinline__ double nexp(double x) { return exp(x); }

// GELU(z) = z Phi(z); GELU'(z) = Phi(z) + z phi(z)
template <class T>
__device__ __forceinline__ T gelu(T z) {
  return z * ncdf(z);
}
template <class T>
__device__ __forceinline__ T gelu_d(T z) {
  return ncdf(z) + z * nexp(T(-0.5) * z * z) * T(0.39894228040143267794);
}

enum { EPI_NONE = 0, EPI_BIAS = 1, EPI_BIAS_GELU = 2, EPI_DGELU = 3 };

struct GemmArgs {
  int M, N, K, lda, ldb, ldc;
  const void* A;
  const void* B;
  void* C;
  const float* bias;  // EPI_BIAS, EPI_BIAS_GELU: [N]
  void* Z;            // EPI_BIAS_GELU: pre-activation out [M][ldc]; EPI_DGELU: pre-activation in
};

// C[m][n] = sum_k A[m lda + k] opB(k,n), opB(k,n) = TB ? B[n ldb + k] : B[k ldb + n].
// Tiles of 64 x 64, 16-deep slabs in shared memory, 4 x 4 outputs per thread;
// ragged edges guarded.
template <class T, bool TB, int EPI>
__global__ void __launch_bounds__(GT) k_gemm(GemmArgs g) {
  __shared__ T As[GBK][GBM + 4];
  __shared__ T Bs[GBK][GBN + 4];
  const T* A = static_cast<const T*>(g.A);
  const __nv_bfloat16* B = static_cast<const __nv_bfloat16*>(g.B);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int m0 = blockIdx.x * GBM, n0 = blockIdx.y * GBN;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc[i][j] = T(0);
  for (int k0 = 0; k0 < g.K; k0 += GBK) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int e = tid + q * GT;
      const int ml = e / GBK, kl = e % GBK;
      const int m = m0 + ml, k = k0 + kl;
      T v = T(0);
      if (m < g.M && k < g.K) v = A[(size_t)m * g.lda + k];
      As[kl][ml] = v;
      int nl, kl2;
      if (TB) { kl2 = e % GBK; nl = e / GBK; } else { nl = e % GBN; kl2 = e / GBN; }
      const int n = n0 + nl, k2 = k0 + kl2;
      T w = T(0);
      if (n < g.N && k2 < g.K) w = (T)__bfloat162float(B[TB ? (size_t)n * g.ldb + k2 : (size_t)k2 * g.ldb + n]);
      Bs[kl2][nl] = w;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GBK; kk++) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; i++) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; j++) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] += a[i] * b[j];
    }
    __syncthreads();
  }
  T* C = static_cast<T*>(g.C);
  T* Z = static_cast<T*>(g.Z);
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int m = m0 + ty * 4 + i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int n = n0 + tx * 4 + j;
      if (n >= g.N) continue;
      const size_t o = (size_t)m * g.ldc + n;
      T v = acc[i][j];
      if (EPI == EPI_BIAS) {
        v += (T)g.bias[n];
      } else if (EPI == EPI_BIAS_GELU) {
        v += (T)g.bias[n];
        Z[o] = v;
        v = gelu(v);
      } else if (EPI == EPI_DGELU) {
        v *= gelu_d(Z[o]);
      }
      C[o] = v;
    }
  }
}

template <class T, bool TB, int EPI>
int gemm(int M, int N, int K, const void* A, int lda, const void* B, int ldb, void* C, int ldc, const float* bias,
         void* Z, cudaStream_t s) {
  if (M <= 0 || N <= 0) return 0;
  GemmArgs g{M, N, K, lda, ldb, ldc, A, B, C, bias, Z};
  dim3 grid((M + GBM - 1) / GBM, (N + GBN - 1) / GBN);
  k_gemm<T, TB, EPI><<<grid, GT, 0, s>>>(g);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------- inference on the tensor pipe
// The FP32-activation inference GEMMs with bfloat16 weights on the tensor
// cores (mma.sync m16n8k16, bfloat16 operands, FP32 accumulation).  Every
// activation is split into three bfloat16 parts, a = a1 + a2 + a3 (a1 the
// rounding of a, a2 of the remainder, a3 of what is left: 24 significant
// bits, the FP32 value to within its last bits); the weights are exactly
// bfloat16, every product of parts is exact in FP32, and the three products
// accumulate in FP32, so that the result is the FP32 product of the FP32
// activations with the bfloat16 weights up to the order of the sums.
//
// C[m][n] = sum_k A[m][k] W(k, n) (+ epilogue), A float [M][lda] (k < K),
// W(k, n) = TB ? B[n ldb + k] : B[k ldb + n] (bfloat16), n < N.  KP, NP: K
// and N padded to the MMA tile (16, 8).  Persistent blocks of four warps,
// each warp 16 rows of a 64-row tile; the weights are staged once per block
// as Ws[n][k] (k contiguous: the B fragment's pairs are one 32-bit load).
constexpr int TC_WARPS = 4, TC_ROWS = 16 * TC_WARPS;

__device__ __forceinline__ unsigned pack_bf16x2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (unsigned)__bfloat16_as_ushort(lo) | ((unsigned)__bfloat16_as_ushort(hi) << 16);
}

// a = p[0] + p[1] + p[2] in bfloat16 parts
__device__ __forceinline__ void split3(float a, __nv_bfloat16 p[3]) {
  p[0] = __float2bfloat16_rn(a);
  float r = a - __bfloat162float(p[0]);
  p[1] = __float2bfloat16_rn(r);
  r = r - __bfloat162float(p[1]);
  p[2] = __float2bfloat16_rn(r);
}

__device__ __forceinline__ void mma_bf16(float c[4], const unsigned a[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int KP, int NP, bool TB, int EPI>
__global__ void __launch_bounds__(32 * TC_WARPS) k_gemm_tc(GemmArgs g) {
  static_assert(KP % 16 == 0 && NP % 8 == 0, "tile padding");
  constexpr int WS = KP + 8;  // bfloat16 per weight row (conflict-free fragment loads)
  constexpr int AS = KP + 8;  // floats per staged activation row
  extern __shared__ __align__(16) unsigned char tc_raw[];
  __nv_bfloat16* Ws = reinterpret_cast<__nv_bfloat16*>(tc_raw);
  float* As = reinterpret_cast<float*>(tc_raw + (size_t)NP * WS * sizeof(__nv_bfloat16));
  const float* A = static_cast<const float*>(g.A);
  const __nv_bfloat16* B = static_cast<const __nv_bfloat16*>(g.B);
  float* C = static_cast<float*>(g.C);
  float* Z = static_cast<float*>(g.Z);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gq = lane >> 2, tq = lane & 3;
  for (int q = tid; q < NP * KP; q += 32 * TC_WARPS) {
    const int n = q / KP, k = q % KP;
    __nv_bfloat16 w = __float2bfloat16_rn(0.f);
    if (n < g.N && k < g.K) w = TB ? B[(size_t)n * g.ldb + k] : B[(size_t)k * g.ldb + n];
    Ws[n * WS + k] = w;
  }
  float* Aw = As + (size_t)warp * 16 * AS;
  for (int m0 = blockIdx.x * TC_ROWS; m0 < g.M; m0 += gridDim.x * TC_ROWS) {
    __syncthreads();  // the weights (first tile) and the previous tile's reads are done
    const int r0 = m0 + warp * 16;
    for (int q = lane; q < 16 * KP; q += 32) {
      const int r = q / KP, k = q % KP;
      const int m = r0 + r;
      Aw[r * AS + k] = (m < g.M && k < g.K) ? A[(size_t)m * g.lda + k] : 0.f;
    }
    __syncwarp();
    float acc[NP / 8][4];
#pragma unroll
    for (int t = 0; t < NP / 8; t++)
#pragma unroll
      for (int j = 0; j < 4; j++) acc[t][j] = 0.f;
#pragma unroll
    for (int kk = 0; kk < KP; kk += 16) {
      // A fragments of the three parts: rows gq, gq + 8; columns 2tq, 2tq + 1 (+8)
      unsigned af[3][4];
      const int rr[4] = {gq, gq + 8, gq, gq + 8};
      const int cc[4] = {kk + 2 * tq, kk + 2 * tq, kk + 2 * tq + 8, kk + 2 * tq + 8};
#pragma unroll
      for (int f = 0; f < 4; f++) {
        const float2 v = *reinterpret_cast<const float2*>(Aw + rr[f] * AS + cc[f]);
        __nv_bfloat16 p0[3], p1[3];
        split3(v.x, p0);
        split3(v.y, p1);
#pragma unroll
        for (int sp = 0; sp < 3; sp++) af[sp][f] = pack_bf16x2(p0[sp], p1[sp]);
      }
#pragma unroll
      for (int t = 0; t < NP / 8; t++) {
        const __nv_bfloat16* wr = Ws + (t * 8 + gq) * WS + kk + 2 * tq;
        const unsigned b0 = *reinterpret_cast<const unsigned*>(wr);
        const unsigned b1 = *reinterpret_cast<const unsigned*>(wr + 8);
#pragma unroll
        for (int sp = 2; sp >= 0; sp--) mma_bf16(acc[t], af[sp], b0, b1);
      }
    }
    // epilogue: acc[t] = rows gq, gq + 8; columns t*8 + 2tq, + 1
#pragma unroll
    for (int t = 0; t < NP / 8; t++)
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int m = r0 + gq + 8 * h;
        if (m >= g.M) continue;
#pragma unroll
        for (int j = 0; j < 2; j++) {
          const int n = t * 8 + 2 * tq + j;
          if (n >= g.N) continue;
          const size_t o = (size_t)m * g.ldc + n;
          float v = acc[t][2 * h + j];
          if (EPI == EPI_BIAS) {
            v += g.bias[n];
          } else if (EPI == EPI_BIAS_GELU) {
            v += g.bias[n];
            Z[o] = v;
            v = gelu(v);
          } else if (EPI == EPI_DGELU) {
            v *= gelu_d(Z[o]);
          }
          C[o] = v;
        }
      }
  }
}

template <int KP, int NP, bool TB, int EPI>
int gemm_tc(int M, int N, int K, const float* A, int lda, const __nv_bfloat16* B, int ldb, float* C, int ldc,
            const float* bias, float* Z, cudaStream_t s) {
  if (M <= 0 || N <= 0) return 0;
  if (K > KP || N > NP) return -1;
  GemmArgs g{M, N, K, lda, ldb, ldc, A, B, C, bias, Z};
  constexpr size_t smem = (size_t)NP * (KP + 8) * sizeof(__nv_bfloat16) + (size_t)TC_ROWS * (KP + 8) * sizeof(float);
  auto fn = k_gemm_tc<KP, NP, TB, EPI>;
  static int per_sm = 0, sms = 0;
  if (per_sm == 0) {
    if (smem > 48 * 1024) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * TC_WARPS, smem);
    if (per_sm < 1) per_sm = 1;
  }
  const int tiles = (M + TC_ROWS - 1) / TC_ROWS;
  const int grid = tiles < sms * per_sm ? tiles : sms * per_sm;
  fn<<<grid, 32 * TC_WARPS, smem, s>>>(g);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------- training kernels
// One batch, forward and reverse, in a single persistent kernel: a block
// holds the FP32 weights in shared memory, takes tiles of 32 rows of the
// batch through the three layers and back, and keeps the sums of its weight
// gradients in registers over its tiles; k_gradient adds the blocks' sums.
//
// Bound: the shared-memory reads and the FP32 pipe: 60k multiply-adds per
// row are 15k issue cycles per tile and SM quarter, of 25k instructions in
// all.  Layer by layer through global memory (64 x 64 tiles, the batch in
// splits of 512 rows) the same work was 14 launches of 3 to 40 us on 16 to
// 128 blocks.  A tile of 32 rows puts a batch of 4,096 on 128 blocks; the
// products read 16-byte weights and broadcast activations, 64 multiply-adds
// per 10 loads.  Measured with Adam: 215 -> 41 us at a batch of 4,096 (27 us
// of it here; about 21 us per tile beyond the first), 211 -> 39 us at 512.
// The 1 / den of the loss (den = 10 sum of the batch's masks, known only at
// the end) is applied by k_gradient: the reverse is linear in it.
constexpr int TR = 32;        // batch rows per tile
constexpr int TT = 256;       // threads
constexpr int HS = NH + 4;    // row stride of the 128-wide arrays (16-byte rows, no bank conflicts)
constexpr int XS = 24;        // inputs 0..8 at 0, 9..17 at 12, zeros between: 16-byte halves
constexpr int WS1 = XS + 4;   // row stride of W1 in the same order
constexpr int YS = 16;        // outputs 0..4 at 0, 5..9 at 8
constexpr int PSTRIDE = (NPAR + 3) & ~3;  // floats of one block's sums
static_assert(NI == 18 && NH == 128 && NO == 10 && TT == 256 && TR == 32, "thread mappings of k_train");
static_assert(OFF_W2 % 4 == 0 && OFF_W3 % 4 == 0 && NPAR % 2 == 0, "16-byte rows of the parameters");

__device__ __forceinline__ int xslot(int j) { return j < 9 ? j : j + 3; }
__device__ __forceinline__ int yslot(int o) { return o < 5 ? o : o + 3; }

struct TrainSmem {
  float W2[NH * HS], W1[NH * WS1], W3[NO * HS];
  float H1[TR * HS], G1[TR * HS];  // GELU and its derivative; G1 becomes dL/dZ1
  float H2[TR * HS], G2[TR * HS];  // G2 becomes dL/dZ2
  float xs[TR * XS], dy[TR * YS];
  float b1[NH], b2[NH], b3[NO];
  double red[2 * TT / 32];
};

template <int N>  // N bytes, both addresses multiples of N
__device__ __forceinline__ void copy_async(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if (N == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// acc[i][j] = sum_k A[i][k] W[32 j][k]: 8 rows of A (stride SA; the same for
// a warp), 2 rows of W (stride SW; lane by lane), k ascending.
template <int K, int SA, int SW>
__device__ __forceinline__ void rows_product(const float* A, const float* W, float acc[8][2]) {
#pragma unroll
  for (int i = 0; i < 8; i++) acc[i][0] = acc[i][1] = 0.f;
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    const float4 w0 = *reinterpret_cast<const float4*>(W + k);
    const float4 w1 = *reinterpret_cast<const float4*>(W + 32 * SW + k);
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const float4 a = *reinterpret_cast<const float4*>(A + i * SA + k);
      acc[i][0] = fmaf(a.w, w0.w, fmaf(a.z, w0.z, fmaf(a.y, w0.y, fmaf(a.x, w0.x, acc[i][0]))));
      acc[i][1] = fmaf(a.w, w1.w, fmaf(a.z, w1.z, fmaf(a.y, w1.y, fmaf(a.x, w1.x, acc[i][1]))));
    }
  }
}

__device__ __forceinline__ void gelu_both(float z, float& h, float& g) {
  const float c = ncdf(z);
  h = z * c;
  g = c + z * nexp(-0.5f * z * z) * 0.39894228040143267794f;
}

// parts[block][NPAR]: the block's sums of den dL/dparam;
// red[2 block], red[2 block + 1]: its sums of m (Y - T)^2 and of m.  A row
// index outside [0, M) is a masked row of zeros and flagged in bad[0].
__global__ void __launch_bounds__(TT, 1) k_train(int B, long long M, unsigned* bad, const int* __restrict__ idx,
                                                 const float* __restrict__ x, const float* __restrict__ t,
                                                 const float* __restrict__ mask, const float* __restrict__ norm,
                                                 const float* __restrict__ P, float* parts, double* red) {
  extern __shared__ __align__(16) unsigned char train_raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(train_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gr = tid >> 3, gl = tid & 7;                       // gather and layer 3: row, lane of the row
  const int r0 = 8 * (warp & 3), ch = 64 * (warp >> 2);        // layers: 8 rows, 64 columns per warp
  const int kt = 4 * (tid & 15), nt = 4 * (tid >> 4);          // dW2: rows nt + {0,64} + 0..3, columns kt likewise
  const int c1 = tid & 127, half = tid >> 7;                   // dW1, dW3, biases: column, half of the others

  // weights in flight first, then the rows of the first tile
  for (int q = tid; q < NH * NH / 4; q += TT)
    copy_async<16>(S.W2 + (q / (NH / 4)) * HS + 4 * (q % (NH / 4)), P + OFF_W2 + 4 * q);
  for (int q = tid; q < NO * NH / 4; q += TT)
    copy_async<16>(S.W3 + (q / (NH / 4)) * HS + 4 * (q % (NH / 4)), P + OFF_W3 + 4 * q);
  for (int q = tid; q < NH * NI; q += TT) copy_async<4>(S.W1 + (q / NI) * WS1 + xslot(q % NI), P + OFF_W1 + q);
  if (tid < NH) {
    copy_async<4>(S.b1 + tid, P + OFF_B1 + tid);
    copy_async<4>(S.b2 + tid, P + OFF_B2 + tid);
  }
  if (tid < NO) copy_async<4>(S.b3 + tid, P + OFF_B3 + tid);
  const int tiles = (B - 1) / TR + 1;
  float xm[3], xd[3], tm[2], td[2];
#pragma unroll
  for (int q = 0; q < 3; q++) {
    const int j = gl + 8 * q < NI ? gl + 8 * q : 0;
    xm[q] = norm[NORM_XM + j];
    xd[q] = norm[NORM_XS + j];
  }
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const int o = gl + 8 * q < NO ? gl + 8 * q : 0;
    tm[q] = norm[NORM_YM + o];
    td[q] = norm[NORM_YS + o];
  }
  // the row of a tile: inputs gl, gl + 8, gl + 16 (< 18), targets gl, gl + 8 (< 10)
  float xv[3], tv[2], mv;
  auto fetch = [&](int tile) {
    const unsigned b = (unsigned)tile * TR + gr;
    xv[0] = xv[1] = xv[2] = tv[0] = tv[1] = mv = 0.f;
    if (b >= (unsigned)B) return;
    const long long r = idx[b];
    if (r < 0 || r >= M) {
      if (gl == 0) atomicOr(bad, 1u);
#pragma unroll
      for (int q = 0; q < 3; q++) xv[q] = xm[q];  // standardised to zero
#pragma unroll
      for (int q = 0; q < 2; q++) tv[q] = tm[q];
      return;
    }
#pragma unroll
    for (int q = 0; q < 3; q++)
      if (gl + 8 * q < NI) xv[q] = x[r * NI + gl + 8 * q];
#pragma unroll
    for (int q = 0; q < 2; q++)
      if (gl + 8 * q < NO) tv[q] = t[r * NO + gl + 8 * q];
    mv = mask[r];
  };
  fetch(blockIdx.x);
  for (int q = tid; q < (NH + TR) * 6; q += TT) {  // the gaps of W1 and xs
    const int r = q / 6, g = q % 6, k = g < 3 ? 9 + g : 18 + g;
    (r < NH ? S.W1 + r * WS1 : S.xs + (r - NH) * XS)[k] = 0.f;
  }

  float dW2[8][8], dW1[9], dW3[5], db12 = 0.f, db3 = 0.f;
#pragma unroll
  for (int i = 0; i < 8; i++)
#pragma unroll
    for (int j = 0; j < 8; j++) dW2[i][j] = 0.f;
#pragma unroll
  for (int j = 0; j < 9; j++) dW1[j] = 0.f;
#pragma unroll
  for (int j = 0; j < 5; j++) dW3[j] = 0.f;
  double loss = 0.0, msum = 0.0;

  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const bool in = (unsigned)tile * TR + gr < (unsigned)B;
    const float tg[2] = {(tv[0] - tm[0]) / td[0], (tv[1] - tm[1]) / td[1]}, m = mv;
#pragma unroll
    for (int q = 0; q < 3; q++)
      if (gl + 8 * q < NI) S.xs[gr * XS + xslot(gl + 8 * q)] = in ? (xv[q] - xm[q]) / xd[q] : 0.f;
    copy_wait();
    __syncthreads();
    if (tile + (int)gridDim.x < tiles) fetch(tile + gridDim.x);  // in flight through this tile
    float acc[8][2];
    // layer 1
    rows_product<XS, XS, WS1>(S.xs + r0 * XS, S.W1 + (ch + lane) * WS1, acc);
#pragma unroll
    for (int j = 0; j < 2; j++) {
      const int n = ch + lane + 32 * j;
#pragma unroll
      for (int i = 0; i < 8; i++) gelu_both(acc[i][j] + S.b1[n], S.H1[(r0 + i) * HS + n], S.G1[(r0 + i) * HS + n]);
    }
    __syncthreads();
    // layer 2
    rows_product<NH, HS, HS>(S.H1 + r0 * HS, S.W2 + (ch + lane) * HS, acc);
#pragma unroll
    for (int j = 0; j < 2; j++) {
      const int n = ch + lane + 32 * j;
#pragma unroll
      for (int i = 0; i < 8; i++) gelu_both(acc[i][j] + S.b2[n], S.H2[(r0 + i) * HS + n], S.G2[(r0 + i) * HS + n]);
    }
    __syncthreads();
    // layer 3: eight lanes per row, 16 of its 128 products each
    {
      float y[NO];
#pragma unroll
      for (int o = 0; o < NO; o++) y[o] = 0.f;
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int k = 4 * gl + 32 * q;
        const float4 h = *reinterpret_cast<const float4*>(S.H2 + gr * HS + k);
#pragma unroll
        for (int o = 0; o < NO; o++) {
          const float4 w = *reinterpret_cast<const float4*>(S.W3 + o * HS + k);
          y[o] = fmaf(h.w, w.w, fmaf(h.z, w.z, fmaf(h.y, w.y, fmaf(h.x, w.x, y[o]))));
        }
      }
#pragma unroll
      for (int o = 0; o < NO; o++)
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) y[o] += __shfl_xor_sync(0xffffffffu, y[o], d);
#pragma unroll
      for (int o = 0; o < NO; o++)
        if ((o & 7) == gl) {
          const float r = in ? (y[o] + S.b3[o] - tg[o >> 3]) * m : 0.f;
          S.dy[gr * YS + yslot(o)] = 2.0f * r;
          loss += (double)r * r;
        }
      if (gl == 0) msum += m;
    }
    __syncthreads();
    // dW3 = dy^T H2, db3; dZ2 = (dy W3) gelu'(Z2)
#pragma unroll 4
    for (int r = 0; r < TR; r++) {
      const float h = S.H2[r * HS + c1];
      const float4 d = *reinterpret_cast<const float4*>(S.dy + r * YS + 8 * half);
      dW3[0] = fmaf(d.x, h, dW3[0]);
      dW3[1] = fmaf(d.y, h, dW3[1]);
      dW3[2] = fmaf(d.z, h, dW3[2]);
      dW3[3] = fmaf(d.w, h, dW3[3]);
      dW3[4] = fmaf(S.dy[r * YS + 8 * half + 4], h, dW3[4]);
    }
    if (tid < NO)
      for (int r = 0; r < TR; r++) db3 += S.dy[r * YS + yslot(tid)];
    {
      float w[NO][2];
#pragma unroll
      for (int o = 0; o < NO; o++)
#pragma unroll
        for (int j = 0; j < 2; j++) w[o][j] = S.W3[o * HS + ch + lane + 32 * j];
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float* d = S.dy + (r0 + i) * YS;
#pragma unroll
        for (int j = 0; j < 2; j++) {
          float v = 0.f;
#pragma unroll
          for (int o = 0; o < NO; o++) v = fmaf(d[o < 5 ? o : o + 3], w[o][j], v);
          S.G2[(r0 + i) * HS + ch + lane + 32 * j] *= v;
        }
      }
    }
    __syncthreads();
    // dZ1 = (dZ2 W2) gelu'(Z1)
#pragma unroll
    for (int i = 0; i < 8; i++) acc[i][0] = acc[i][1] = 0.f;
#pragma unroll 2
    for (int n = 0; n < NH; n += 4) {
      float2 w[4];
#pragma unroll
      for (int q = 0; q < 4; q++) w[q] = *reinterpret_cast<const float2*>(S.W2 + (n + q) * HS + ch + 2 * lane);
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float4 d = *reinterpret_cast<const float4*>(S.G2 + (r0 + i) * HS + n);
        acc[i][0] = fmaf(d.w, w[3].x, fmaf(d.z, w[2].x, fmaf(d.y, w[1].x, fmaf(d.x, w[0].x, acc[i][0]))));
        acc[i][1] = fmaf(d.w, w[3].y, fmaf(d.z, w[2].y, fmaf(d.y, w[1].y, fmaf(d.x, w[0].y, acc[i][1]))));
      }
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
      float2* g = reinterpret_cast<float2*>(S.G1 + (r0 + i) * HS + ch + 2 * lane);
      const float2 v = *g;
      *g = make_float2(v.x * acc[i][0], v.y * acc[i][1]);
    }
    // dW2 = dZ2^T H1
#pragma unroll 2
    for (int r = 0; r < TR; r++) {
      float d[8], h[8];
#pragma unroll
      for (int q = 0; q < 2; q++) {
        *reinterpret_cast<float4*>(d + 4 * q) = *reinterpret_cast<const float4*>(S.G2 + r * HS + nt + 64 * q);
        *reinterpret_cast<float4*>(h + 4 * q) = *reinterpret_cast<const float4*>(S.H1 + r * HS + kt + 64 * q);
      }
#pragma unroll
      for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 8; j++) dW2[i][j] = fmaf(d[i], h[j], dW2[i][j]);
    }
    if (half == 1)
      for (int r = 0; r < TR; r++) db12 += S.G2[r * HS + c1];
    __syncthreads();
    // dW1 = dZ1^T xs, db1
#pragma unroll 4
    for (int r = 0; r < TR; r++) {
      const float d = S.G1[r * HS + c1];
      const float* xr = S.xs + r * XS + 12 * half;
      const float4 x0 = *reinterpret_cast<const float4*>(xr);
      const float4 x1 = *reinterpret_cast<const float4*>(xr + 4);
      dW1[0] = fmaf(d, x0.x, dW1[0]);
      dW1[1] = fmaf(d, x0.y, dW1[1]);
      dW1[2] = fmaf(d, x0.z, dW1[2]);
      dW1[3] = fmaf(d, x0.w, dW1[3]);
      dW1[4] = fmaf(d, x1.x, dW1[4]);
      dW1[5] = fmaf(d, x1.y, dW1[5]);
      dW1[6] = fmaf(d, x1.z, dW1[6]);
      dW1[7] = fmaf(d, x1.w, dW1[7]);
      dW1[8] = fmaf(d, xr[8], dW1[8]);
      if (half == 0) db12 += d;
    }
    __syncthreads();  // xs and the activations are free for the next tile
  }

  float* out = parts + (size_t)blockIdx.x * PSTRIDE;
#pragma unroll
  for (int i = 0; i < 8; i++)
#pragma unroll
    for (int q = 0; q < 2; q++)
      *reinterpret_cast<float4*>(out + OFF_W2 + (nt + (i & 3) + 64 * (i >> 2)) * NH + kt + 64 * q) =
          make_float4(dW2[i][4 * q], dW2[i][4 * q + 1], dW2[i][4 * q + 2], dW2[i][4 * q + 3]);
#pragma unroll
  for (int j = 0; j < 9; j++) out[OFF_W1 + c1 * NI + 9 * half + j] = dW1[j];
#pragma unroll
  for (int j = 0; j < 5; j++) out[OFF_W3 + (5 * half + j) * NH + c1] = dW3[j];
  out[(half ? OFF_B2 : OFF_B1) + c1] = db12;
  if (tid < NO) out[OFF_B3 + tid] = db3;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    loss += __shfl_xor_sync(0xffffffffu, loss, o);
    msum += __shfl_xor_sync(0xffffffffu, msum, o);
  }
  if (lane == 0) {
    S.red[2 * warp] = loss;
    S.red[2 * warp + 1] = msum;
  }
  __syncthreads();
  if (tid < 2) {
    double q = 0.0;
    for (int w = 0; w < TT / 32; w++) q += S.red[2 * w + tid];
    red[2 * blockIdx.x + tid] = q;
  }
}

// grad = sum over the blocks of k_train / den, loss = sum m (Y - T)^2 / den,
// den = 10 max(1, sum of the masks); grad_out, loss_out may be NULL.  64
// parameters per block, its eight warps take the blocks' sums in turn
// (80 KB per block of k_train, read once from L2), fixed order.
__global__ void __launch_bounds__(TT) k_gradient(int nb, const float* __restrict__ parts,
                                                 const double* __restrict__ red, float* grad, float* grad_out,
                                                 float* loss_out) {
  __shared__ float2 sh[TT / 32][32];
  __shared__ double sd[2][TT / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i = blockIdx.x * 64 + 2 * lane;
  float2 v = make_float2(0.f, 0.f);
  if (i < NPAR) {
#pragma unroll 8
    for (int b = warp; b < nb; b += TT / 32) {
      const float2 p = *reinterpret_cast<const float2*>(parts + (size_t)b * PSTRIDE + i);
      v.x += p.x;
      v.y += p.y;
    }
  }
  double l = 0.0, m = 0.0;
  for (int b = tid; b < nb; b += TT) {
    l += red[2 * b];
    m += red[2 * b + 1];
  }
  for (int o = 16; o > 0; o >>= 1) {
    l += __shfl_xor_sync(0xffffffffu, l, o);
    m += __shfl_xor_sync(0xffffffffu, m, o);
  }
  sh[warp][lane] = v;
  if (lane == 0) {
    sd[0][warp] = l;
    sd[1][warp] = m;
  }
  __syncthreads();
  if (warp != 0) return;
  l = m = 0.0;
  for (int w = 0; w < TT / 32; w++) {
    l += sd[0][w];
    m += sd[1][w];
  }
  const float den = (float)(NO * (m > 1.0 ? m : 1.0));
  if (blockIdx.x == 0 && lane == 0 && loss_out) loss_out[0] = (float)(l / den);
  if (i >= NPAR) return;
  for (int w = 1; w < TT / 32; w++) {
    v.x += sh[w][lane].x;
    v.y += sh[w][lane].y;
  }
  v.x /= den;
  v.y /= den;
  grad[i] = v.x;
  grad[i + 1] = v.y;
  if (grad_out) {
    grad_out[i] = v.x;
    grad_out[i + 1] = v.y;
  }
}

// Adam (bias-corrected), then the bfloat16 copy used for inference.
__global__ void k_adam(int n, float* p, const float* __restrict__ g, float* m, float* v, float lr, float b1, float b2,
                       float eps, float c1, float c2, __nv_bfloat16* wbf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float mh = mi / c1, vh = vi / c2;
  const float pi = p[i] - lr * mh / (sqrtf(vh) + eps);
  p[i] = pi;
  wbf[i] = __float2bfloat16_rn(pi);
}

__global__ void k_to_bf16(int n, const float* __restrict__ p, __nv_bfloat16* wbf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) wbf[i] = __float2bfloat16_rn(p[i]);
}

// Normalisation statistics, one block per column (18 inputs, then 10
// targets) over the rows with mask > 0: mean, population standard deviation
// (floored at 1e-6), and for inputs the range widened by 5 % of its span.
__global__ void __launch_bounds__(RT) k_norm_stats(long long M, const float* __restrict__ x,
                                                   const float* __restrict__ t, const float* __restrict__ mask,
                                                   float* norm) {
  __shared__ double sa[RT / 32], sb[RT / 32], smn[RT / 32], smx[RT / 32];
  __shared__ double mean_s;
  const int c = blockIdx.x;
  const bool isx = c < NI;
  const int j = isx ? c : c - NI;
  const float* src = isx ? x : t;
  const int ld_ = isx ? NI : NO;
  double s = 0.0, w = 0.0, mn = 1e300, mx = -1e300;
  for (long long r = threadIdx.x; r < M; r += RT) {
    if (!(mask[r] > 0.f)) continue;
    const double v = src[r * ld_ + j];
    s += v;
    w += 1.0;
    mn = fmin(mn, v);
    mx = fmax(mx, v);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    w += __shfl_xor_sync(0xffffffffu, w, o);
    mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    sa[threadIdx.x >> 5] = s;
    sb[threadIdx.x >> 5] = w;
    smn[threadIdx.x >> 5] = mn;
    smx[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double S = 0.0, W = 0.0, MN = 1e300, MX = -1e300;
    for (int q = 0; q < RT / 32; q++) {
      S += sa[q];
      W += sb[q];
      MN = fmin(MN, smn[q]);
      MX = fmax(MX, smx[q]);
    }
    mean_s = W > 0.0 ? S / W : 0.0;
    sa[0] = W;
    smn[0] = MN;
    smx[0] = MX;
  }
  __syncthreads();
  const double mean = mean_s, W = sa[0], MN = smn[0], MX = smx[0];
  double q2 = 0.0;
  for (long long r = threadIdx.x; r < M; r += RT) {
    if (!(mask[r] > 0.f)) continue;
    const double d = src[r * ld_ + j] - mean;
    q2 += d * d;
  }
  for (int o = 16; o > 0; o >>= 1) q2 += __shfl_xor_sync(0xffffffffu, q2, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sb[threadIdx.x >> 5] = q2;
  __syncthreads();
  if (threadIdx.x == 0) {
    double Q = 0.0;
    for (int q = 0; q < RT / 32; q++) Q += sb[q];
    double sd = W > 0.0 ? sqrt(Q / W) : 1.0;
    if (sd < 1e-6) sd = 1e-6;
    if (isx) {
      const double span = MX - MN;
      norm[NORM_XM + j] = (float)mean;
      norm[NORM_XS + j] = (float)sd;
      norm[NORM_LO + j] = (float)(MN - 0.05 * span);
      norm[NORM_HI + j] = (float)(MX + 0.05 * span);
    } else {
      norm[NORM_YM + j] = (float)mean;
      norm[NORM_YS + j] = (float)sd;
    }
  }
}

// Standardise raw inputs / de-standardise outputs (prediction entry point).
__global__ void k_standardise(long long M, const float* __restrict__ x, const float* __restrict__ norm, float* xs) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M * NI) return;
  const int j = (int)(i % NI);
  xs[i] = (x[i] - norm[NORM_XM + j]) / norm[NORM_XS + j];
}
__global__ void k_destandardise(long long M, const float* __restrict__ ys, const float* __restrict__ norm,
                                float* y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M * NO) return;
  const int j = (int)(i % NO);
  y[i] = norm[NORM_YM + j] + norm[NORM_YS + j] * ys[i];
}

int grid1(long long n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

// ---------------------------------------------------------------- inference (energy path)
// ys = net(xs) for M rows; Z1, Z2 keep the pre-activations for the reverse.
int mlp_infer_forward(int fp64, int M, const void* xs, const float* params, const void* wbf, void* Z1, void* H1,
                      void* Z2, void* H2, void* ys, cudaStream_t s) {
  const __nv_bfloat16* w = static_cast<const __nv_bfloat16*>(wbf);
  int r = 0;
  if (fp64) {
    r |= gemm<double, true, EPI_BIAS_GELU>(M, NH, NI, xs, NI, w + OFF_W1, NI, H1, NH,
                                                                         params + OFF_B1, Z1, s);
    r |= gemm<double, true, EPI_BIAS_GELU>(M, NH, NH, H1, NH, w + OFF_W2, NH, H2, NH,
                                                                         params + OFF_B2, Z2, s);
    r |= gemm<double, true, EPI_BIAS>(M, NO, NH, H2, NH, w + OFF_W3, NH, ys, NO,
                                                                    params + OFF_B3, nullptr, s);
  } else {  // tensor pipe (three bfloat16 parts per FP32 activation)
    r |= gemm_tc<32, 128, true, EPI_BIAS_GELU>(M, NH, NI, (const float*)xs, NI, w + OFF_W1, NI, (float*)H1, NH,
                                               params + OFF_B1, (float*)Z1, s);
    r |= gemm_tc<128, 128, true, EPI_BIAS_GELU>(M, NH, NH, (const float*)H1, NH, w + OFF_W2, NH, (float*)H2, NH,
                                                params + OFF_B2, (float*)Z2, s);
    r |= gemm_tc<128, 16, true, EPI_BIAS>(M, NO, NH, (const float*)H2, NH, w + OFF_W3, NH, (float*)ys, NO,
                                          params + OFF_B3, nullptr, s);
  }
  return r;
}

// xbar = (d ys / d xs)^T ybar for M rows; dZ1, dZ2 are scratch [M][128].
int mlp_infer_backward(int fp64, int M, const void* ybar, const void* wbf, void* Z1, void* Z2, void* dZ1, void* dZ2,
                       void* xbar, cudaStream_t s) {
  const __nv_bfloat16* w = static_cast<const __nv_bfloat16*>(wbf);
  int r = 0;
  if (fp64) {
    r |= gemm<double, false, EPI_DGELU>(M, NH, NO, ybar, NO, w + OFF_W3, NH, dZ2, NH,
                                                                      nullptr, Z2, s);
    r |= gemm<double, false, EPI_DGELU>(M, NH, NH, dZ2, NH, w + OFF_W2, NH, dZ1, NH,
                                                                      nullptr, Z1, s);
    r |= gemm<double, false, EPI_NONE>(M, NI, NH, dZ1, NH, w + OFF_W1, NI, xbar, NI,
                                                                     nullptr, nullptr, s);
  } else {  // tensor pipe (three bfloat16 parts per FP32 cotangent)
    r |= gemm_tc<16, 128, false, EPI_DGELU>(M, NH, NO, (const float*)ybar, NO, w + OFF_W3, NH, (float*)dZ2, NH,
                                            nullptr, (float*)Z2, s);
    r |= gemm_tc<128, 128, false, EPI_DGELU>(M, NH, NH, (const float*)dZ2, NH, w + OFF_W2, NH, (float*)dZ1, NH,
                                             nullptr, (float*)Z1, s);
    r |= gemm_tc<128, 24, false, EPI_NONE>(M, NI, NH, (const float*)dZ1, NH, w + OFF_W1, NI, (float*)xbar, NI,
                                           nullptr, nullptr, s);
  }
  return r;
}

// ---------------------------------------------------------------- the bop_mlp object
struct MBuf {
  void* p = nullptr;
  size_t bytes = 0;
};

struct bop_mlp {
  MBuf params, grad, am, av, wbf, norm;
  MBuf xs, Z1, H1, Z2, H2, y, parts, red, bad;
  int adam_t = 0;
  int batch_cap = 0;
  char err[256];
};

namespace {

int mfail(bop_mlp* n, int code, const char* fmt, ...) {
  if (n) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(n->err, sizeof(n->err), fmt, ap);
    va_end(ap);
  }
  return code;
}

int mensure(bop_mlp* n, MBuf& b, size_t bytes) {
  if (bytes == 0) bytes = 16;
  if (b.bytes >= bytes) return BOP_OK;
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.bytes = 0;
  if (cudaMalloc(&b.p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return mfail(n, BOP_ERR_OOM, "cudaMalloc(%zu) failed", bytes);
  }
  b.bytes = bytes;
  return BOP_OK;
}

template <class T>
T* MP(MBuf& b) {
  return reinterpret_cast<T*>(b.p);
}

#define MCK(call)                                                                                        \
  do {                                                                                                   \
    cudaError_t e_ = (call);                                                                             \
    if (e_ != cudaSuccess) return mfail(net, BOP_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_));     \
  } while (0)

// Buffers of a prediction over B rows.
int size_batch(bop_mlp* net, int B) {
  if (B <= net->batch_cap) return BOP_OK;
  int r;
  const size_t b = (size_t)B;
  if ((r = mensure(net, net->xs, sizeof(float) * b * NI)) || (r = mensure(net, net->Z1, sizeof(float) * b * NH)) ||
      (r = mensure(net, net->H1, sizeof(float) * b * NH)) || (r = mensure(net, net->Z2, sizeof(float) * b * NH)) ||
      (r = mensure(net, net->H2, sizeof(float) * b * NH)) || (r = mensure(net, net->y, sizeof(float) * b * NO)))
    return r;
  net->batch_cap = B;
  return BOP_OK;
}

}  // namespace

const float* mlp_params_dev(const bop_mlp* net) { return static_cast<const float*>(net->params.p); }
const void* mlp_wbf_dev(const bop_mlp* net) { return net->wbf.p; }
const float* mlp_norm_dev(const bop_mlp* net) { return static_cast<const float*>(net->norm.p); }

extern "C" {

int bop_mlp_create(bop_mlp** out, const float* params_host) {
  if (!out || !params_host) return BOP_ERR_ARG;
  *out = nullptr;
  bop_mlp* net = new (std::nothrow) bop_mlp();
  if (!net) return BOP_ERR_OOM;
  net->err[0] = 0;
  int r;
  if ((r = mensure(net, net->params, sizeof(float) * NPAR)) || (r = mensure(net, net->grad, sizeof(float) * NPAR)) ||
      (r = mensure(net, net->am, sizeof(float) * NPAR)) || (r = mensure(net, net->av, sizeof(float) * NPAR)) ||
      (r = mensure(net, net->wbf, sizeof(__nv_bfloat16) * NPAR)) ||
      (r = mensure(net, net->norm, sizeof(float) * BOP_MLP_NNORM)) || (r = mensure(net, net->bad, 16))) {
    bop_mlp_destroy(net);
    return r;
  }
  float norm0[BOP_MLP_NNORM];
  for (int j = 0; j < BOP_MLP_NNORM; j++) norm0[j] = 0.f;
  for (int j = 0; j < NI; j++) {
    norm0[NORM_XS + j] = 1.f;
    norm0[NORM_LO + j] = -3.0e38f;
    norm0[NORM_HI + j] = 3.0e38f;
  }
  for (int j = 0; j < NO; j++) norm0[NORM_YS + j] = 1.f;
  if (cudaMemcpy(net->params.p, params_host, sizeof(float) * NPAR, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(net->norm.p, norm0, sizeof(norm0), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(net->am.p, 0, sizeof(float) * NPAR) != cudaSuccess ||
      cudaMemset(net->av.p, 0, sizeof(float) * NPAR) != cudaSuccess ||
      cudaMemset(net->bad.p, 0, 16) != cudaSuccess) {
    bop_mlp_destroy(net);
    return BOP_ERR_CUDA;
  }
  k_to_bf16<<<grid1(NPAR, 256), 256>>>(NPAR, MP<float>(net->params), MP<__nv_bfloat16>(net->wbf));
  if (cudaDeviceSynchronize() != cudaSuccess) {
    bop_mlp_destroy(net);
    return BOP_ERR_CUDA;
  }
  *out = net;
  return BOP_OK;
}

int bop_mlp_destroy(bop_mlp* net) {
  if (!net) return BOP_OK;
  for (MBuf* b : {&net->params, &net->grad, &net->am, &net->av, &net->wbf, &net->norm, &net->xs, &net->Z1,
                  &net->H1, &net->Z2, &net->H2, &net->y, &net->parts, &net->red, &net->bad})
    if (b->p) cudaFree(b->p);
  delete net;
  return BOP_OK;
}

const char* bop_mlp_last_error(const bop_mlp* net) { return net ? net->err : "net is NULL"; }

int bop_mlp_get(bop_mlp* net, float* params_host, float* norm_host) {
  if (!net) return BOP_ERR_ARG;
  if (params_host) MCK(cudaMemcpy(params_host, net->params.p, sizeof(float) * NPAR, cudaMemcpyDeviceToHost));
  if (norm_host) MCK(cudaMemcpy(norm_host, net->norm.p, sizeof(float) * BOP_MLP_NNORM, cudaMemcpyDeviceToHost));
  return BOP_OK;
}

int bop_mlp_set_norm(bop_mlp* net, const float* norm_host) {
  if (!net || !norm_host) return BOP_ERR_ARG;
  for (int j = 0; j < NI; j++)
    if (!(norm_host[NORM_XS + j] > 0.f)) return mfail(net, BOP_ERR_ARG, "input standard deviation %d not > 0", j);
  for (int j = 0; j < NO; j++)
    if (!(norm_host[NORM_YS + j] > 0.f)) return mfail(net, BOP_ERR_ARG, "target standard deviation %d not > 0", j);
  MCK(cudaMemcpy(net->norm.p, norm_host, sizeof(float) * BOP_MLP_NNORM, cudaMemcpyHostToDevice));
  return BOP_OK;
}

int bop_mlp_fit_norm(bop_mlp* net, long long M, const float* x, const float* t, const float* mask,
                     bop_stream stream) {
  if (!net || M < 1 || !x || !t || !mask) return mfail(net, BOP_ERR_ARG, "need M >= 1, x, t and mask");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  k_norm_stats<<<NI + NO, RT, 0, s>>>(M, x, t, mask, MP<float>(net->norm));
  MCK(cudaGetLastError());
  return BOP_OK;
}

int bop_mlp_gradient(bop_mlp* net, long long M, const float* x, const float* t, const float* mask, const int* idx,
                     int batch, float* grad_out, float* loss_out, bop_stream stream) {
  if (!net || M < 1 || !x || !t || !mask || !idx || batch < 1)
    return mfail(net, BOP_ERR_ARG, "need M >= 1, x, t, mask, idx and batch >= 1");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int dev = 0, sms = 0;
  MCK(cudaGetDevice(&dev));
  MCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  MCK(cudaFuncSetAttribute(k_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)));
  const int tiles = (batch - 1) / TR + 1;
  const int nb = tiles < sms ? tiles : sms;
  int r;
  if ((r = mensure(net, net->parts, sizeof(float) * (size_t)nb * PSTRIDE)) ||
      (r = mensure(net, net->red, sizeof(double) * 2 * nb)))
    return r;
  float* parts = MP<float>(net->parts);
  double* red = MP<double>(net->red);
  k_train<<<nb, TT, sizeof(TrainSmem), s>>>(batch, M, MP<unsigned>(net->bad), idx, x, t, mask, MP<float>(net->norm),
                                            MP<float>(net->params), parts, red);
  k_gradient<<<grid1(NPAR, 64), TT, 0, s>>>(nb, parts, red, MP<float>(net->grad), grad_out, loss_out);
  MCK(cudaGetLastError());
  return BOP_OK;
}

int bop_mlp_check(bop_mlp* net, bop_stream stream) {
  if (!net) return BOP_ERR_ARG;
  unsigned h = 0;
  MCK(cudaMemcpyAsync(&h, net->bad.p, sizeof(unsigned), cudaMemcpyDeviceToHost, reinterpret_cast<cudaStream_t>(stream)));
  MCK(cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream)));
  if (!h) return BOP_OK;
  MCK(cudaMemset(net->bad.p, 0, sizeof(unsigned)));
  return mfail(net, BOP_ERR_ARG, "a batch row index was outside [0, M)");
  return BOP_OK;
}

int bop_mlp_adam(bop_mlp* net, float lr, bop_stream stream) {
  if (!net || !(lr > 0.f)) return mfail(net, BOP_ERR_ARG, "need lr > 0");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  net->adam_t += 1;
  const double b1 = 0.9, b2 = 0.999;
  const float c1 = (float)(1.0 - std::pow(b1, net->adam_t)), c2 = (float)(1.0 - std::pow(b2, net->adam_t));
  k_adam<<<grid1(NPAR, 256), 256, 0, s>>>(NPAR, MP<float>(net->params), MP<float>(net->grad), MP<float>(net->am),
                                          MP<float>(net->av), lr, (float)b1, (float)b2, 1e-8f, c1, c2,
                                          MP<__nv_bfloat16>(net->wbf));
  MCK(cudaGetLastError());
  return BOP_OK;
}

int bop_mlp_train_step(bop_mlp* net, long long M, const float* x, const float* t, const float* mask, const int* idx,
                       int batch, float lr, float* loss_out, bop_stream stream) {
  int r = bop_mlp_gradient(net, M, x, t, mask, idx, batch, nullptr, loss_out, stream);
  if (r) return r;
  return bop_mlp_adam(net, lr, stream);
}

int bop_mlp_predict(bop_mlp* net, long long M, const float* x, float* y, bop_stream stream) {
  if (!net || M < 1 || !x || !y) return mfail(net, BOP_ERR_ARG, "need M >= 1, x and y");
  if (M > 0x7fffffffLL / NH) return mfail(net, BOP_ERR_ARG, "M too large");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int r = size_batch(net, (int)M);
  if (r) return r;
  k_standardise<<<grid1(M * NI, 256), 256, 0, s>>>(M, x, MP<float>(net->norm), MP<float>(net->xs));
  if (mlp_infer_forward(0, (int)M, net->xs.p, MP<float>(net->params), net->wbf.p, net->Z1.p, net->H1.p, net->Z2.p,
                        net->H2.p, net->y.p, s))
    return mfail(net, BOP_ERR_CUDA, "gemm launch failed");
  k_destandardise<<<grid1(M * NO, 256), 256, 0, s>>>(M, MP<float>(net->y), MP<float>(net->norm), y);
  MCK(cudaGetLastError());
  return BOP_OK;
}

}  // extern "C"
