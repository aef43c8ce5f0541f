// Moments mu_n(i alpha) = <i alpha|H^n|i alpha> (Eq. momDOS) by the
// iterated interference paths Psi_k = H Psi_{k-1} (Eq. xi_rec) over every
// atom's cluster, with the merge property (Eq. xi_merge):
//   mu_2k = <Psi_k|Psi_k>,   mu_2k-1 = <Psi_k-1|Psi_k>,
// and the reverse sweep of the same recursion, which gives dU/dH for every
// bond and dU/dE for every onsite level from the weights w_n = dU/dmu_n
// (the Theta-tilde / transfer-path sums of Eqs. theta-tilde, Xi).
//
// Forward: one CTA per (spin, atom).  Psi_{k-1} and Psi_k live in shared
// memory (ping-pong) or global scratch; the last level Psi_K is only stored for
// a reverse sweep.  FP32: a thread per cluster site and pass, which gathers
// the 5x5 blocks of its bonds (15 unique elements, 16-element records) from
// L2 (for sd blocks 21 unique elements in 24-element records).  FP64: a thread
// per row of a site's block.  Moments written as double.
//
// Reverse: over the stored Psi, one CTA per work item with Psi-bar of two
// levels at a time; where the store does not fit, Psi_0..Psi_K and the
// cotangents Psi-bar_1..Psi-bar_K are recomputed in the CTA's slot of global
// scratch and the bond cotangents summed over levels per cluster edge.
#include "kernels.h"

namespace {

constexpr int MOM_THREADS = 256;

// stored elements of one bond block (unique upper triangle + pad to 16 bytes)
template <int NO>
__host__ __device__ constexpr int hb_count() {
  return NO == 1 ? 1 : (NO == 5 ? 16 : 24);
}

template <typename T>
struct Blk;
// Block records are 32-byte multiples on 32-byte boundaries (16 or 24 FP32
// values, 16 FP64 values): they are read with 256-bit loads, half as many
// L1 accesses per block as 128-bit loads.
__device__ __forceinline__ void ld256(const float* p, float* v) {
  asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
      : "l"(p));
}
template <>
struct Blk<float> {
  template <int HB>
  __device__ static void load(const float* __restrict__ h, float u[HB]) {
    static_assert(HB % 8 == 0, "block records of 32-byte multiples");
#pragma unroll
    for (int q = 0; q < HB / 8; q++) ld256(h + 8 * q, u + 8 * q);
  }
};
template <>
struct Blk<double> {
  template <int HB>
  __device__ static void load(const double* __restrict__ h, double u[HB]) {
    const double2* p = reinterpret_cast<const double2*>(h);
#pragma unroll
    for (int q = 0; q < HB / 2; q++) {
      double2 v = __ldg(p + q);
      u[2 * q] = v.x; u[2 * q + 1] = v.y;
    }
  }
};

// unique element of (row, col) in the upper triangle of an NO x NO block
template <int NO>
__device__ __forceinline__ constexpr int UI(int b, int g) {
  return b <= g ? b * NO - (b * (b - 1)) / 2 + (g - b) : g * NO - (g * (g - 1)) / 2 + (b - g);
}

// Stride of one bond's cotangents: the unique block elements, padded to a
// multiple of four for FP32 (vector atomics), unpadded for FP64.
template <typename T, int NO>
__host__ __device__ constexpr int hbar_stride() {
  return (NO == 1 || sizeof(T) == 8) ? NO * (NO + 1) / 2 : (NO * (NO + 1) / 2 + 3) / 4 * 4;
}

// Adds dL/dB (G[b][g] = dL/dB_bg of one orientation of a symmetric block)
// to the bond's unique elements: u(b, g) collects G[b][g] + G[g][b].  FP32
// cotangents go out as float4 reductions (four per d block instead of 15
// scalar ones), FP64 as scalar FP64 atomics.
template <typename T, int NO>
__device__ __forceinline__ void add_bond_cotangent(T* __restrict__ hbp, const T G[NO][NO]) {
  if constexpr (NO == 1) {
    atomicAdd(hbp, G[0][0]);
  } else if constexpr (sizeof(T) == 4) {
    constexpr int HV = hbar_stride<T, NO>();
    float v[HV];
#pragma unroll
    for (int q = 0; q < HV; q++) v[q] = 0.f;
#pragma unroll
    for (int b = 0; b < NO; b++)
#pragma unroll
      for (int g = b; g < NO; g++) v[UI<NO>(b, g)] = G[b][g] + (b != g ? G[g][b] : 0.f);
    float4* dst = reinterpret_cast<float4*>(hbp);
#pragma unroll
    for (int q = 0; q < HV / 4; q++) atomicAdd(dst + q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
  } else {
#pragma unroll
    for (int b = 0; b < NO; b++)
#pragma unroll
      for (int g = b; g < NO; g++) atomicAdd(hbp + UI<NO>(b, g), G[b][g] + (b != g ? G[g][b] : T(0)));
  }
}

// acc[r][c] += B[r][g] * x[g][c] for the symmetric block B given by u[].
template <typename T, int NO, int NC>
__device__ __forceinline__ void block_apply(const T* __restrict__ hrec, const T* __restrict__ x,
                                            T acc[NO][NC]) {
  if constexpr (NO == 1) {
    T h = hrec[0];
#pragma unroll
    for (int c = 0; c < NC; c++) acc[0][c] += h * x[c];
  } else {
    T u[hb_count<NO>()];
    Blk<T>::template load<hb_count<NO>()>(hrec, u);
    T xs[NO][NC];
#pragma unroll
    for (int g = 0; g < NO; g++)
#pragma unroll
      for (int c = 0; c < NC; c++) xs[g][c] = x[g * NC + c];
#pragma unroll
    for (int r = 0; r < NO; r++)
#pragma unroll
      for (int g = 0; g < NO; g++) {
        T h = u[UI<NO>(r, g)];
#pragma unroll
        for (int c = 0; c < NC; c++) acc[r][c] += h * xs[g][c];
      }
  }
}

// next 16-byte boundary (the staged adjacency holds int2 / u64 records); the
// launchers reserve 16 bytes of slack for it
__device__ __forceinline__ unsigned char* align16(unsigned char* p) {
  return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(p) + 15) & ~(uintptr_t)15);
}

// Hint to bring the 128-byte lines of a stored row into L2 before it is read.
template <typename T, int PS>
__device__ __forceinline__ void prefetch_row_l2(const T* p) {
  constexpr int BYTES = PS * (int)sizeof(T);
#pragma unroll
  for (int o = 0; o < BYTES; o += 128)
    asm volatile("{\n\t.reg .u64 ga;\n\tcvta.to.global.u64 ga, %0;\n\tprefetch.global.L2 [ga];\n\t}" ::"l"(
        reinterpret_cast<const char*>(p) + o));
  asm volatile("{\n\t.reg .u64 ga;\n\tcvta.to.global.u64 ga, %0;\n\tprefetch.global.L2 [ga];\n\t}" ::"l"(
      reinterpret_cast<const char*>(p) + BYTES - 1));
}

// Asynchronous copies global -> shared (cp.async, no register round trip),
// so that all of a thread's staging copies of a work item are in flight at
// once; cp_async_wait_all() waits for the thread's own copies, a barrier
// then publishes them to the CTA.
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Extent of one atom's cluster in the cluster arrays: first site, number of
// sites, adjacency range.  Read in two steps (sites, then adjacency) one work
// item ahead, so that the next item's staging starts without waiting on
// dependent loads.
struct ItemExt {
  long long s0, abase, aend;
  int nsite;
};
__device__ __forceinline__ void ext_sites(const ClusterView& cv, int atom, ItemExt& x) {
  x.s0 = cv.site_off[atom];
  x.nsite = cv.level_end[(size_t)atom * (cv.K + 1) + cv.K];
}
__device__ __forceinline__ void ext_adj(const ClusterView& cv, ItemExt& x) {
  x.abase = cv.adj_off[x.s0];
  x.aend = cv.adj_off[x.s0 + x.nsite];
}

// The consecutive work items of a CTA of a persistent kernel.  The first CTAs
// take the remainder of the division, one item each: those are one to an SM,
// so that an SM's CTAs do not all have the longer run and every resident CTA has
// work (131,072 items: reverse sweep 20.0 -> 18.9 ms, 1,372 items on 304 CTAs:
// no change, the five items of a CTA are the longest chain either way).
__device__ __forceinline__ void item_range(int n_items, int* w0, int* w1) {
  const int b = blockIdx.x, base = n_items / gridDim.x, rest = n_items % gridDim.x;
  *w0 = b * base + min(b, rest);
  *w1 = *w0 + base + (b < rest ? 1 : 0);
}

// One work item's cluster data in shared memory: the adjacency entries of its
// first nrow sites, their adjacency offsets (from the item's first entry) and
// level counts, and the atoms of all its sites.
__device__ __forceinline__ void stage_item(const ClusterView& cv, const ItemExt& x, int nrow, int nadj, int2* s_adj,
                                           int* s_off, unsigned long long* s_lvc, int* s_atom, int tid, int nthr) {
  const long long s0 = x.s0, abase = x.abase;
  for (int q = tid; q < nadj; q += nthr) cp_async8(s_adj + q, cv.adj + abase + q);
  for (int q = tid; q < nrow; q += nthr) cp_async8(s_lvc + q, cv.lvcnt + s0 + q);
  for (int q = tid; q < x.nsite; q += nthr) cp_async4(s_atom + q, cv.site_atom + s0 + q);
  for (int q = tid; q <= nrow; q += nthr) s_off[q] = (int)(cv.adj_off[s0 + q] - abase);
  cp_async_wait_all();
}

// Its row orders, likewise (before stage_item, whose wait covers these copies).
__device__ __forceinline__ void stage_order(const ClusterView& cv, const ItemExt& x, bool pair, unsigned* s_ord,
                                            unsigned* s_top, int tid, int nthr) {
  for (int q = tid; q < x.nsite; q += nthr) {
    cp_async4(s_ord + q, cv.order + x.s0 + q);
    if (pair) cp_async4(s_top + q, cv.top + x.s0 + q);
  }
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// y[t] = E_t * x[t] (t < ncol) + sum_{adjacent s < ncol} B_ts x[s], t < nrow.
// One thread per site; returns nothing, the caller consumes acc.
template <typename T, int NO, int NC>
__device__ __forceinline__ void gather_row(const ClusterView& cv, const T* __restrict__ H, int HS,
                                           const T* __restrict__ E, const int* __restrict__ satom,
                                           const long long* __restrict__ aoff, int t, int ncol,
                                           const T* __restrict__ x, T acc[NO][NC]) {
#pragma unroll
  for (int r = 0; r < NO; r++)
#pragma unroll
    for (int c = 0; c < NC; c++) acc[r][c] = T(0);
  if (t < ncol) {
    const T* e = E + (size_t)satom[t] * NO;
#pragma unroll
    for (int r = 0; r < NO; r++) {
      T er = e[r];
#pragma unroll
      for (int c = 0; c < NC; c++) acc[r][c] = er * x[(t * NO + r) * NC + c];
    }
  }
  const long long q1 = aoff[t + 1];
  for (long long q = aoff[t]; q < q1; q++) {
    int2 en = cv.adj[q];
    if (en.x >= ncol) break;
    block_apply<T, NO, NC>(H + (size_t)en.y * HS, x + (size_t)en.x * NO * NC, acc);
  }
}

// ------------------------------------------------------------------ forward
// Shared-memory row of one site: NO x NC values padded to 16-byte multiples
// so that a row is read with vector loads.
template <typename T, int N>
struct Row {
  static constexpr int PS = (sizeof(T) == 4) ? ((N + 3) / 4) * 4 : ((N + 1) / 2) * 2;
};
template <typename T, int N, int PS>
__device__ __forceinline__ void load_row(const T* __restrict__ p, T x[N]) {
  if constexpr (N == 1) {
    x[0] = p[0];
  } else if constexpr (sizeof(T) == 4) {
    const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int v = 0; v < PS / 4; v++) {
      float4 w = q[v];
      if (4 * v + 0 < N) x[4 * v + 0] = w.x;
      if (4 * v + 1 < N) x[4 * v + 1] = w.y;
      if (4 * v + 2 < N) x[4 * v + 2] = w.z;
      if (4 * v + 3 < N) x[4 * v + 3] = w.w;
    }
  } else {
    const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
    for (int v = 0; v < PS / 2; v++) {
      double2 w = q[v];
      if (2 * v + 0 < N) x[2 * v + 0] = w.x;
      if (2 * v + 1 < N) x[2 * v + 1] = w.y;
    }
  }
}

template <typename T, int N, int PS>
__device__ __forceinline__ void store_row(T* __restrict__ p, const T x[N]) {
  if constexpr (N == 1) {
    p[0] = x[0];
  } else if constexpr (sizeof(T) == 4) {
    float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
    for (int v = 0; v < PS / 4; v++) {
      float4 w;
      w.x = 4 * v + 0 < N ? x[4 * v + 0] : 0.f;
      w.y = 4 * v + 1 < N ? x[4 * v + 1] : 0.f;
      w.z = 4 * v + 2 < N ? x[4 * v + 2] : 0.f;
      w.w = 4 * v + 3 < N ? x[4 * v + 3] : 0.f;
      q[v] = w;
    }
  } else {
    double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
    for (int v = 0; v < PS / 2; v++) {
      double2 w;
      w.x = 2 * v + 0 < N ? x[2 * v + 0] : 0.0;
      w.y = 2 * v + 1 < N ? x[2 * v + 1] : 0.0;
      q[v] = w;
    }
  }
}

template <typename T, int NO>
__device__ __forceinline__ void load_bond(const T* __restrict__ h, T u[hb_count<NO>()]) {
  if constexpr (NO == 1) {
    u[0] = __ldg(h);
  } else {
    Blk<T>::template load<hb_count<NO>()>(h, u);
  }
}

// acc += B x for one symmetric block (unique elements u) and a site row x
template <typename T, int NO, int NC>
__device__ __forceinline__ void block_fma(const T* u, const T* x, T acc[NO][NC]) {
  if constexpr (NO == 1) {
#pragma unroll
    for (int c = 0; c < NC; c++) acc[0][c] += u[0] * x[c];
  } else {
#pragma unroll
    for (int r = 0; r < NO; r++)
#pragma unroll
      for (int g = 0; g < NO; g++) {
        const T h = u[UI<NO>(r, g)];
#pragma unroll
        for (int c = 0; c < NC; c++) acc[r][c] += h * x[g * NC + c];
      }
  }
}

// acc += sum over cnt adjacency entries of B_ts x[s],
// with the blocks of the next two entries in flight while the current one is
// applied.
template <typename T, int NO, int NC, int PS>
__device__ __forceinline__ void gather_pf2(const int2* __restrict__ ent, int cnt, const T* __restrict__ H,
                                           int HS, const T* __restrict__ x, T acc[NO][NC]) {
  constexpr int HB = hb_count<NO>();
  constexpr int N = NO * NC;
  if (cnt <= 0) return;
  int2 e0 = ent[0];
  int2 e1 = cnt > 1 ? ent[1] : e0;
  T h0[HB], h1[HB];
  load_bond<T, NO>(H + (size_t)e0.y * HS, h0);
  if (cnt > 1) load_bond<T, NO>(H + (size_t)e1.y * HS, h1);
  for (int e = 0; e < cnt; e++) {
    const int s = e0.x;
    T hc[HB];
#pragma unroll
    for (int q = 0; q < HB; q++) hc[q] = h0[q];
    e0 = e1;
#pragma unroll
    for (int q = 0; q < HB; q++) h0[q] = h1[q];
    if (e + 2 < cnt) {
      e1 = ent[e + 2];
      load_bond<T, NO>(H + (size_t)e1.y * HS, h1);
    }
    T xs[N];
    load_row<T, N, PS>(x + (size_t)s * PS, xs);
    block_fma<T, NO, NC>(hc, xs, acc);
  }
}

// The same, one entry at a time: fewer registers by two blocks.
template <typename T, int NO, int NC, int PS>
__device__ __forceinline__ void gather_plain(const int2* __restrict__ ent, int cnt, const T* __restrict__ H, int HS,
                                             const T* __restrict__ x, T acc[NO][NC]) {
  constexpr int N = NO * NC;
  for (int e = 0; e < cnt; e++) {
    const int2 en = ent[e];
    T hb[hb_count<NO>()], xs[N];
    load_bond<T, NO>(H + (size_t)en.y * HS, hb);
    load_row<T, N, PS>(x + (size_t)en.x * PS, xs);
    block_fma<T, NO, NC>(hb, xs, acc);
  }
}

// Adds one bond record of cotangents per lane (v: NO x NO unique elements,
// padded) to the bonds' cotangent records; bond < 0: none.  All lanes of the
// warp call it.  FP32: four lanes add one record together, 16 bytes each, so
// that a reduction instruction touches 8 records instead of 32 (the four
// quarters are exchanged between the lanes by 12 shuffles; reductions of
// scattered records cost the L1 unit one cycle per line).
template <typename T, int NO>
__device__ __forceinline__ void add_bond_records(T* __restrict__ Hbar, int HSh, int bond, const T G[NO][NO], int lane) {
  if constexpr (NO == 1 || sizeof(T) == 8) {
    if (bond >= 0) add_bond_cotangent<T, NO>(Hbar + (size_t)bond * HSh, G);
  } else {
    constexpr int HV = hbar_stride<T, NO>();
    float v[HV];
#pragma unroll
    for (int q = 0; q < HV; q++) v[q] = 0.f;
#pragma unroll
    for (int b = 0; b < NO; b++)
#pragma unroll
      for (int g = b; g < NO; g++) v[UI<NO>(b, g)] = G[b][g] + (b != g ? G[g][b] : 0.f);
    const int q = lane & 3;
#pragma unroll
    for (int d = 0; d < 4; d++) {
      // quarter q ^ d of this lane's record goes to lane q ^ d, whose quarter q comes here
      const int o = q ^ d;
      float4 x;
      x.x = (o & 2) ? ((o & 1) ? v[12] : v[8]) : ((o & 1) ? v[4] : v[0]);
      x.y = (o & 2) ? ((o & 1) ? v[13] : v[9]) : ((o & 1) ? v[5] : v[1]);
      x.z = (o & 2) ? ((o & 1) ? v[14] : v[10]) : ((o & 1) ? v[6] : v[2]);
      x.w = (o & 2) ? ((o & 1) ? v[15] : v[11]) : ((o & 1) ? v[7] : v[3]);
      int bd = bond;
      if (d > 0) {
        x.x = __shfl_xor_sync(0xffffffffu, x.x, d);
        x.y = __shfl_xor_sync(0xffffffffu, x.y, d);
        x.z = __shfl_xor_sync(0xffffffffu, x.z, d);
        x.w = __shfl_xor_sync(0xffffffffu, x.w, d);
        bd = __shfl_xor_sync(0xffffffffu, bond, d);
      }
      if (bd >= 0) atomicAdd(reinterpret_cast<float4*>(Hbar + (size_t)bd * HSh) + q, x);
    }
    if (bond >= 0) {
      float4* dst = reinterpret_cast<float4*>(Hbar + (size_t)bond * HSh);
#pragma unroll
      for (int w = 4; w < HV / 4; w++)
        atomicAdd(dst + w, make_float4(v[4 * w], v[4 * w + 1], v[4 * w + 2], v[4 * w + 3]));
    }
  }
}

// The reverse sweep's gather of one row by one lane: acc += B_ts x[s] over
// the entries first, first + step, ... of the row (or those of the bits of
// mask), with the blocks of two entries in flight.  HBAR: also the bond
// cotangents dL/dB = x[s] pt^T of the forward pairs (s, t), summed over the
// columns (x = Psi-bar_k, pt = Psi_k-1(t)); with gather false (level 1) only
// those.  All lanes of a warp call it (rows of no entries: cnt 0).
template <typename T, int NO, int NC, int PS, bool HBAR>
__device__ __forceinline__ void gather_rev(const int2* __restrict__ ent, int first, int step, int cnt, unsigned mask,
                                           bool use_mask, const T* __restrict__ H, int HS, const T* __restrict__ x,
                                           T acc[NO][NC], bool gather, const T pt[NO * NC], T* __restrict__ Hbar,
                                           int HSh, int lane) {
  constexpr int HB = hb_count<NO>();
  constexpr int N = NO * NC;
  const int mine = use_mask ? __popc(mask) : (cnt > first ? (cnt - first + step - 1) / step : 0);
  const int rounds = HBAR ? __reduce_max_sync(0xffffffffu, mine) : mine;
  int e = first;
  auto next = [&]() -> int2 {  // the row's next entry
    int i = e;
    if (use_mask) {
      i = __ffs(mask) - 1;
      mask &= mask - 1;
    }
    e += step;
    return ent[i];
  };
  int2 e0 = make_int2(0, -1), e1 = make_int2(0, -1);
  T h0[HB], h1[HB];
  if (mine > 0) {
    e0 = next();
    if (gather) load_bond<T, NO>(H + (size_t)e0.y * HS, h0);
  }
  if (mine > 1) {
    e1 = next();
    if (gather) load_bond<T, NO>(H + (size_t)e1.y * HS, h1);
  }
  for (int it = 0; it < rounds; it++) {
    const bool on = it < mine;
    const int sidx = e0.x, bond = on ? e0.y : -1;
    T hc[HB];
#pragma unroll
    for (int q = 0; q < HB; q++) hc[q] = h0[q];
    e0 = e1;
#pragma unroll
    for (int q = 0; q < HB; q++) h0[q] = h1[q];
    if (it + 2 < mine) {
      e1 = next();
      if (gather) load_bond<T, NO>(H + (size_t)e1.y * HS, h1);
    }
    T G[NO][NO];
    if (on) {
      T xs[N];
      load_row<T, N, PS>(x + (size_t)sidx * PS, xs);
      if (gather) block_fma<T, NO, NC>(hc, xs, acc);
      if constexpr (HBAR) {
#pragma unroll
        for (int b = 0; b < NO; b++)
#pragma unroll
          for (int g = 0; g < NO; g++) {
            T a = T(0);
#pragma unroll
            for (int c = 0; c < NC; c++) a += xs[b * NC + c] * pt[g * NC + c];
            G[b][g] = a;
          }
      }
    } else if constexpr (HBAR) {
#pragma unroll
      for (int b = 0; b < NO; b++)
#pragma unroll
        for (int g = 0; g < NO; g++) G[b][g] = T(0);
    }
    if constexpr (HBAR) add_bond_records<T, NO>(Hbar, HSh, bond, G, lane);
  }
}

// Forward kernel, FP32 (FP64: k_moments64).  A persistent CTA takes a run of
// consecutive work items (spin, atom); neighbouring atoms share most of their
// clusters' blocks, which then come from L1.  For each item the atom's
// adjacency, per-site offsets, level counts and site atoms are staged in
// shared memory (one coalesced copy) when they fit, so that the edge loop only
// waits for the bond blocks, which are fetched one edge ahead.  Each thread
// computes all columns of one site (NO^3 multiply-adds per edge); Psi rows are
// padded to 16-byte multiples and kept in two exactly sized buffers (even and
// odd levels) in shared memory, or where those do not fit (GMEM: clusters of
// 11 and more moments) in the Psi store or the CTA's slot of global scratch,
// from where the L2 serves them: one item with all columns takes 1/5 of the
// block loads of five items that fit.
//
// One lane per site, in site order, and the sums in that order: the band edges
// are a maximum over levels, and moments rounded differently send a few
// orbitals of 100,000 to the other side of a tie, where the forces jump.
// (Rows ordered by length and the pair form of k_moments64 gained 5 % here: the
// pass is bound by the L1 data path, which idle lanes do not load.)
constexpr int F32_THREADS = 192;

struct FwdSmem {
  int cap_even, cap_odd, max_sites, max_adj;
  bool stage;
};

// Whether site t (atom j) of centre i is selected (pair_selected).
__device__ __forceinline__ bool site_selected(const ClusterView& cv, long long s0, int i, int j, int t) {
  if (i != j) return pair_selected(i, j, 0, 0, 0);
  const signed char* im = cv.site_img + 3 * (s0 + t);
  return pair_selected(i, j, im[0], im[1], im[2]);
}

template <int NO, bool GMEM>
__global__ void __launch_bounds__(F32_THREADS, 2)
k_moments(ClusterView cv, const float* __restrict__ H, int HS, const float* __restrict__ onsite, int n, int n_on,
          int n_mom, FwdSmem L, int n_items, double* __restrict__ mu, float* __restrict__ pstore,
          const long long* __restrict__ psi_off, long long psi_tot, bool sel_store,
          float* __restrict__ scratch, size_t slot_elems) {
  using T = float;
  constexpr int NT = F32_THREADS, NC = NO;
  constexpr int N = NO * NC;
  constexpr int PS = (N == 1) ? 1 : Row<T, N>::PS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf[2];
  buf[0] = GMEM ? scratch + (size_t)blockIdx.x * slot_elems : reinterpret_cast<T*>(smem_raw);
  buf[1] = buf[0] + (size_t)L.cap_even * PS;
  unsigned char* tail = align16(GMEM ? smem_raw : reinterpret_cast<unsigned char*>(buf[1] + (size_t)L.cap_odd * PS));
  int2* s_adj = reinterpret_cast<int2*>(tail);
  unsigned long long* s_lvc = reinterpret_cast<unsigned long long*>(s_adj + (L.stage ? L.max_adj : 0));
  int* s_off = reinterpret_cast<int*>(s_lvc + (L.stage ? L.max_sites : 0));
  int* s_atom = s_off + (L.stage ? L.max_sites + 1 : 0);
  // per-warp partial sums of the two moments of a level, in two buffers
  // (level parity): the reads of level k's partials need no barrier before
  // level k + 1 starts writing its own
  __shared__ T red[2][2 * NC][NT / 32];
  const int K = cv.K;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int w0, w1;
  item_range(n_items, &w0, &w1);
  ItemExt nx{};
  if (w0 < w1) {
    ext_sites(cv, w0 % n, nx);
    ext_adj(cv, nx);
  }
  for (int w = w0; w < w1; w++) {
    const int spin = w / n, atom = w % n;
    const ItemExt cur = nx;
    const long long s0 = cur.s0, abase = cur.abase;
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const int2* adj = cv.adj + abase;
    const unsigned long long* lvc = cv.lvcnt + s0;
    const int* satom = L.stage ? s_atom : cv.site_atom + s0;
    const T* E = onsite + (size_t)spin * n_on * NO;
    if (L.stage)
      stage_item(cv, cur, cur.nsite, (int)(cur.aend - abase), s_adj, s_off, s_lvc, s_atom, tid, NT);
    const bool more = w + 1 < w1;
    if (more) ext_sites(cv, (w + 1) % n, nx);
    // stored Psi: item rows start at ib, level k at row lo_k = sum_{j<k} |C_j|
    T* pitem = nullptr;
    if (pstore != nullptr) {
      pitem = pstore + ((size_t)spin * psi_tot + psi_off[atom]) * PS;
      for (int q = tid; q < PS; q += NT) pitem[q] = T(q < N && q / NC == q % NC ? 1 : 0);
    }
    for (int q = tid; q < PS; q += NT) buf[0][q] = T(q < N && q / NC == q % NC ? 1 : 0);
    long long lo_k = 0;
    __syncthreads();
    double* out = mu + (size_t)w * NO * n_mom;
    if (tid < NC) out[(size_t)tid * n_mom] = 1.0;
    for (int k = 1; k <= K; k++) {
      const bool in_store = GMEM && pstore != nullptr;
      const T* prev = in_store ? pitem + (size_t)lo_k * PS : buf[(k - 1) & 1];
      lo_k += lev[k - 1];
      const int ncol = lev[k - 1], nrow = lev[k];
      T* next = buf[k & 1];
      T d1[NC], d2[NC];
#pragma unroll
      for (int c = 0; c < NC; c++) d1[c] = d2[c] = T(0);
      for (int t = tid; t < nrow; t += NT) {
        T acc[NO][NC];
        const bool in_prev = t < ncol;
        const int atom_t = satom[t];
        if (in_prev) {
          T pt[N];
          load_row<T, N, PS>(prev + (size_t)t * PS, pt);
          const T* e = E + (size_t)atom_t * NO;
#pragma unroll
          for (int r_ = 0; r_ < NO; r_++) {
            const T er = e[r_];
#pragma unroll
            for (int c = 0; c < NC; c++) acc[r_][c] = er * pt[r_ * NC + c];
          }
        } else {
#pragma unroll
          for (int r_ = 0; r_ < NO; r_++)
#pragma unroll
            for (int c = 0; c < NC; c++) acc[r_][c] = T(0);
        }
        const unsigned long long lc = L.stage ? s_lvc[t] : lvc[t];
        const int cnt = (int)((lc >> (8 * (k - 1))) & 0xff);
        const int q0 = L.stage ? s_off[t] : (int)(cv.adj_off[s0 + t] - abase);
        gather_pf2<T, NO, NC, PS>(L.stage ? s_adj + q0 : adj + q0, cnt, H, HS, prev, acc);
        // row t of Psi_k-1 again (shared memory), rather than kept live over the gather
        if (in_prev) {
          T pt[N];
          load_row<T, N, PS>(prev + (size_t)t * PS, pt);
#pragma unroll
          for (int r_ = 0; r_ < NO; r_++)
#pragma unroll
            for (int c = 0; c < NC; c++) d1[c] += pt[r_ * NC + c] * acc[r_][c];
        }
#pragma unroll
        for (int r_ = 0; r_ < NO; r_++)
#pragma unroll
          for (int c = 0; c < NC; c++) d2[c] += acc[r_][c] * acc[r_][c];
        if (k < K && !in_store) store_row<T, N, PS>(next + (size_t)t * PS, &acc[0][0]);
        if (pitem != nullptr && (k < K || !sel_store || site_selected(cv, s0, atom, atom_t, t)))
          store_row<T, N, PS>(pitem + (size_t)(lo_k + t) * PS, &acc[0][0]);
      }
#pragma unroll
      for (int c = 0; c < NC; c++) {
        T a = warp_sum(d1[c]), b = warp_sum(d2[c]);
        if (lane == 0) {
          red[k & 1][c][wid] = a;
          red[k & 1][NC + c][wid] = b;
        }
      }
      // level k's rows and partials are complete; level k + 1 writes the
      // other Psi buffer (read last at level k - 1) and the other partials
      __syncthreads();
      if (tid < 2 * NC) {
        T acc = T(0);
        for (int q = 0; q < NT / 32; q++) acc += red[k & 1][tid][q];
        const int c = tid % NC;
        out[(size_t)c * n_mom + (tid < NC ? 2 * k - 1 : 2 * k)] = (double)acc;
      }
    }
    if (more) ext_adj(cv, nx);
  }
}

// ------------------------------------------------------------------ FP64: a lane per row of a site's block
// FP64 is bound by the DFMA pipe (a warp's instruction takes 64 cycles of an SM
// sub-partition, whatever its active lanes), so the work goes into warps that
// are full and equally long: NO lanes per site, lane r holding row r of its
// NO x NO block (32 / NO sites per warp, 25 multiply-adds per entry and lane at
// NO = 5), longest rows first.  The lanes of a site read the same Psi row
// (one shared-memory broadcast) and the NO elements of their row of the bond
// block.  With one lane per site (and two for long rows of small levels) the
// lanes were 82 % and the pipe 81 % busy, the SMs 88 %, at 9 moments.  The
// work items go round the CTAs, so that cheap ones (surfaces) spread over
// them.
constexpr int F64_THREADS = 256;      // forward
constexpr int F64_REV_THREADS = 128;  // reverse (twice the registers per lane)

// Row r of NO x NO blocks: acc[c] += sum over the entries of sum_g B[r][g]
// x[s][g][c], with the block rows of two entries in flight.  u: positions of
// B[r][g] in the bond record.
template <int NO, int PS>
__device__ __forceinline__ void gather64(const int2* __restrict__ ent, int cnt, const double* __restrict__ H, int HS,
                                         const double* __restrict__ x, const int u[NO], double acc[NO]) {
  if (cnt <= 0) return;
  int2 e0 = ent[0], e1 = e0;
  double b0[NO], b1[NO];
#pragma unroll
  for (int g = 0; g < NO; g++) b0[g] = __ldg(H + (size_t)e0.y * HS + u[g]);
  if (cnt > 1) {
    e1 = ent[1];
#pragma unroll
    for (int g = 0; g < NO; g++) b1[g] = __ldg(H + (size_t)e1.y * HS + u[g]);
  }
  for (int e = 0; e < cnt; e++) {
    const int s = e0.x;
    double b[NO];
#pragma unroll
    for (int g = 0; g < NO; g++) {
      b[g] = b0[g];
      b0[g] = b1[g];
    }
    e0 = e1;
    if (e + 2 < cnt) {
      e1 = ent[e + 2];
#pragma unroll
      for (int g = 0; g < NO; g++) b1[g] = __ldg(H + (size_t)e1.y * HS + u[g]);
    }
    double xs[NO * NO];
    load_row<double, NO * NO, PS>(x + (size_t)s * PS, xs);
#pragma unroll
    for (int g = 0; g < NO; g++)
#pragma unroll
      for (int c = 0; c < NO; c++) acc[c] += b[g] * xs[g * NO + c];
  }
}

// Forward.  pair: the last level computes the selected sites only
// (pair_selected).  H^K is symmetric, so the block Z = Psi_K(t, i) holds
// Psi_K(i, t)^T too: its column sums go to this item's last two moments; its
// row sums belong to those of the site's atom and are written out for
// k_pair_sums (68 % of a bcc cluster's products at 9 moments are in that
// level).  Every sum has an order of its own: the rows of a level go to the
// warps there and back in their order, and no atomics, so that moments repeat
// bit for bit.  GMEM as k_moments.
template <int NO, bool GMEM>
__global__ void __launch_bounds__(F64_THREADS, 2)
k_moments64(ClusterView cv, const double* __restrict__ H, int HS, const double* __restrict__ onsite, int n, int n_on,
            int n_mom, FwdSmem L, int n_items, double* __restrict__ mu, double* __restrict__ pstore,
            const long long* __restrict__ psi_off, long long psi_tot, bool pair, double2* __restrict__ rowsum,
            long long nsite, double* __restrict__ scratch, size_t slot_elems) {
  constexpr int NT = F64_THREADS, NC = NO;
  constexpr int N = NO * NC;
  constexpr int PS = (N == 1) ? 1 : Row<double, N>::PS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* buf[2];
  buf[0] = GMEM ? scratch + (size_t)blockIdx.x * slot_elems : reinterpret_cast<double*>(smem_raw);
  buf[1] = buf[0] + (size_t)L.cap_even * PS;
  unsigned char* tail = align16(GMEM ? smem_raw : reinterpret_cast<unsigned char*>(buf[1] + (size_t)L.cap_odd * PS));
  int2* s_adj = reinterpret_cast<int2*>(tail);
  unsigned long long* s_lvc = reinterpret_cast<unsigned long long*>(s_adj + (L.stage ? L.max_adj : 0));
  int* s_off = reinterpret_cast<int*>(s_lvc + (L.stage ? L.max_sites : 0));
  int* s_atom = s_off + (L.stage ? L.max_sites + 1 : 0);
  unsigned* s_ord = reinterpret_cast<unsigned*>(s_atom + (L.stage ? L.max_sites : 0));
  unsigned* s_top = s_ord + (L.stage ? L.max_sites : 0);
  // per-warp partial sums of the two moments of a level, in two buffers
  // (level parity), as k_moments
  __shared__ double red[2][2 * NC][NT / 32];
  const int K = cv.K;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  ItemExt nx{};
  if ((int)blockIdx.x < n_items) {
    ext_sites(cv, blockIdx.x % n, nx);
    ext_adj(cv, nx);
  }
  for (int w = blockIdx.x; w < n_items; w += gridDim.x) {
    const int spin = w / n, atom = w % n;
    const ItemExt cur = nx;
    const long long s0 = cur.s0, abase = cur.abase;
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const int2* adj = cv.adj + abase;
    const int* satom = L.stage ? s_atom : cv.site_atom + s0;
    const unsigned* order = L.stage ? s_ord : cv.order + s0;
    const unsigned* top = L.stage ? s_top : cv.top + s0;
    const double* E = onsite + (size_t)spin * n_on * NO;
    if (L.stage) {
      stage_order(cv, cur, pair, s_ord, s_top, tid, NT);
      stage_item(cv, cur, cur.nsite, (int)(cur.aend - abase), s_adj, s_off, s_lvc, s_atom, tid, NT);
    }
    const int ntop = pair ? cv.ntop[atom] & 0xffff : 0;
    const bool more = n_items - w > (int)gridDim.x;
    if (more) ext_sites(cv, (w + gridDim.x) % n, nx);
    // stored Psi: item rows start at psi_off, level k at row lo_k = sum_{j<k} |C_j|
    double* pitem = nullptr;
    if (pstore != nullptr) {
      pitem = pstore + ((size_t)spin * psi_tot + psi_off[atom]) * PS;
      for (int q = tid; q < PS; q += NT) pitem[q] = q < N && q / NC == q % NC ? 1.0 : 0.0;
    }
    for (int q = tid; q < PS; q += NT) buf[0][q] = q < N && q / NC == q % NC ? 1.0 : 0.0;
    long long lo_k = 0;
    __syncthreads();
    double* out = mu + (size_t)w * NO * n_mom;
    if (tid < NC) out[(size_t)tid * n_mom] = 1.0;
    for (int k = 1; k <= K; k++) {
      const bool in_store = GMEM && pstore != nullptr;
      const double* prev = in_store ? pitem + (size_t)lo_k * PS : buf[(k - 1) & 1];
      lo_k += lev[k - 1];
      const int ncol = lev[k - 1], inner = k >= 2 ? lev[k - 2] : 0;
      const int nrow = pair && k == K ? ntop : lev[k];
      double* next = buf[k & 1];
      double d[2 * NC];
#pragma unroll
      for (int c = 0; c < 2 * NC; c++) d[c] = 0.0;
      // two copies of the rows' code: the sums of the half level cost the other
      // levels registers (2,000 atoms at 17 moments: 22.2 -> 21.7 ms)
      auto rows = [&](auto last) {
        constexpr bool half = decltype(last)::value;
        constexpr int NW = NT / 32;
        for (int p = 0; 32 * p * NW < nrow * NO; p++) {
          const int first = 32 * (p * NW + ((p & 1) ? NW - 1 - wid : wid));
          // (the lanes of a site need not be in one warp: 32 / NO is no whole number)
          const int q = (first + lane) / NO, r = (first + lane) % NO;
          if (q >= nrow) continue;
          int u[NO];
#pragma unroll
          for (int g = 0; g < NO; g++) u[g] = UI<NO>(r, g);
          // rows up to level k-2 are full, shell k-1 has entries up to its own
          // level, shell k of the one below
          const int t = half ? (int)(top[q] & 0xffffu)
                             : (q < inner ? q : (q < ncol ? (int)(order[q] >> 16) : (int)(order[q] & 0xffffu)));
          const bool in_prev = t < ncol;
          const int atom_t = satom[t];
          const double* pt = prev + (size_t)t * PS + r * NC;
          double acc[NC];
          if (in_prev) {
            const double er = E[(size_t)atom_t * NO + r];
#pragma unroll
            for (int c = 0; c < NC; c++) acc[c] = er * pt[c];
          } else {
#pragma unroll
            for (int c = 0; c < NC; c++) acc[c] = 0.0;
          }
          const unsigned long long lc = L.stage ? s_lvc[t] : cv.lvcnt[s0 + t];
          const int cnt = (int)((lc >> (8 * (k - 1))) & 0xff);
          const int q0 = L.stage ? s_off[t] : (int)(cv.adj_off[s0 + t] - abase);
          gather64<NO, PS>(L.stage ? s_adj + q0 : adj + q0, cnt, H, HS, prev, u, acc);
          if (in_prev) {
#pragma unroll
            for (int c = 0; c < NC; c++) d[c] += pt[c] * acc[c];
          }
#pragma unroll
          for (int c = 0; c < NC; c++) d[NC + c] += acc[c] * acc[c];
          if constexpr (half) {  // the row's sums, for the site's atom
            double a1 = 0.0, a2 = 0.0;
            if (in_prev) {
#pragma unroll
              for (int c = 0; c < NC; c++) a1 += pt[c] * acc[c];
            }
#pragma unroll
            for (int c = 0; c < NC; c++) a2 += acc[c] * acc[c];
            rowsum[((size_t)spin * nsite + s0 + t) * NO + r] = make_double2(a1, a2);
          }
          if (k < K && !in_store) {
#pragma unroll
            for (int c = 0; c < NC; c++) next[(size_t)t * PS + r * NC + c] = acc[c];
          }
          if (pitem != nullptr) {
#pragma unroll
            for (int c = 0; c < NC; c++) pitem[(size_t)(lo_k + t) * PS + r * NC + c] = acc[c];
          }
        }
      };
      if (pair && k == K) rows(std::true_type{});
      else rows(std::false_type{});
      int which;
      const double sum = warp_sums<2 * NC>(d, lane, &which);
      if (which >= 0) red[k & 1][which][wid] = sum;
      // level k's rows and partials are complete; level k + 1 writes the
      // other Psi buffer (read last at level k - 1) and the other partials
      __syncthreads();
      if (tid < 2 * NC) {
        double a = 0.0;
        for (int q = 0; q < NT / 32; q++) a += red[k & 1][tid][q];
        const int c = tid % NC;
        out[(size_t)c * n_mom + (tid < NC ? 2 * k - 1 : 2 * k)] = a;
      }
    }
    if (more) ext_adj(cv, nx);
  }
}

// The rest of the last two moments in the pair form: of every site that is not
// selected, the row sums that its pair left in the cluster of the site's atom
// (k_pair_mirror).  One block per (spin, atom): a lane per value of a site's row
// sums and 32 / (2 NO) sites at a time, so that FP64 additions have all lanes;
// eight warps, since what bounds it is the latency of a place and its row sums
// (432 atoms with two spins, cold cache: 18 us with one warp, 13 with eight).
// It is launched while the sweep still runs and waits for it (3 us a pass).  A
// pass of theirs takes 614 us, 603 with FP64 atomics and sites drawn from a
// counter, whose moments did not repeat.
constexpr int PS_THREADS = 256;

template <int NO>
__global__ void __launch_bounds__(PS_THREADS) k_pair_sums(ClusterView cv, int n, int n_mom,
                                                          const unsigned* __restrict__ mirror,
                                                          const double2* __restrict__ rowsum, long long nsite,
                                                          double* __restrict__ mu) {
  constexpr int V = 2 * NO, SW = 32 / V, NW = PS_THREADS / 32;
  __shared__ double sh[NW][V];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int w = blockIdx.x, spin = w / n, atom = w % n, K = cv.K;
  const int cnt = cv.level_end[(size_t)atom * (K + 1) + K] - (cv.ntop[atom] & 0xffff);
  const unsigned* list = mirror + cv.site_off[atom];
  const double* rs = reinterpret_cast<const double*>(rowsum + (size_t)spin * nsite * NO) + lane % V;
  cudaGridDependencySynchronize();  // the sweep's row sums and moments
  double a = 0.0;
  if (lane < V * SW) {
#pragma unroll 8
    for (int q = wid * SW + lane / V; q < cnt; q += NW * SW) a += __ldg(rs + (size_t)__ldg(list + q) * V);
  }
  double sum = a;
#pragma unroll
  for (int p = 1; p < SW; p++) sum += __shfl_sync(0xffffffffu, a, lane + p * V);
  if (lane < V) sh[wid][lane] = sum;
  __syncthreads();
  if (tid < V) {
    double m = 0.0;
#pragma unroll
    for (int q = 0; q < NW; q++) m += sh[q][tid];
    mu[((size_t)w * NO + tid / 2) * n_mom + 2 * K - 1 + tid % 2] += m;
  }
}

// ------------------------------------------------------------------ reverse sweep over stored Psi
// With every Psi_k of every work item stored in global memory (rows of the
// forward kernel, level k at rows lo_k .. lo_k + |C_k|), the reverse sweep
//   Psi-bar_K     = 2 w_2K Psi_K + w_2K-1 Psi_K-1
//   Psi-bar_k-1   = H Psi-bar_k (rows < |C_k-1|, columns < |C_k|)
//                   + 2 w_2k-2 Psi_k-1 + w_2k-1 Psi_k + w_2k-3 Psi_k-2
// runs like the forward kernel: Psi-bar_k and Psi-bar_k-1 in two buffers (even
// / odd levels) in shared memory or (GMEM) in the CTA's slot of global
// scratch, the adjacency of the rows (C_K-1) staged.  The
// onsite cotangents dL/dE_t = sum_k Psi-bar_k[t] . Psi_k-1[t] are accumulated
// per site in shared memory and added once per item.  With HBAR the gather of
// level k also forms the bond cotangents of its pairs, Psi-bar_k(s)
// Psi_k-1(t)^T for the forward pair (s in C_k, t in C_k-1), and adds them to
// the bond's unique elements; at k = 1 only these products run.
//
// A level of fewer rows than threads gives each row 2 to 16 adjacent lanes
// that share its entries and add their sums by shuffles (65 rows of 14 entries
// at level 3 of a bcc cluster, 15 at level 2): the levels' longest chains fall
// from 14 entries to 7 and 2.
//
// pair: the last level in the pair form of the forward kernel.  Z =
// Psi_K(t, i) enters the moments of the centre i by its columns and those of
// the site's atom j by its rows, so that its cotangent is 2 (w_i + w_j) Z
// + (w_i + w_j)' Psi_K-1(t) with column weights w_i and row weights w_j; the
// gather of level K runs over the selected entries of every row
// (ClusterView::topmask), rows in the order of their number.
struct RevSmem {
  int cap_even, cap_odd, max_sites, max_adj, cap_eb;
  bool stage;
};

template <typename T, int NO>
__host__ __device__ constexpr size_t eb_elems(int cap_eb) {
  return ((size_t)cap_eb * NO * sizeof(T) + 15) / 16 * 16 / sizeof(T);
}

constexpr int REV_SEL_WORDS = 256;  // selected sites as bits (a cluster with a pair form has at most 8,192 sites)

template <int NO, bool HBAR, bool GMEM>
__global__ void __launch_bounds__(F32_THREADS, 2)
k_adj_rev(ClusterView cv, const float* __restrict__ H, int HS, const float* __restrict__ onsite, int n, int n_on,
          int n_mom, RevSmem L, int n_items, const float* __restrict__ pstore,
          const long long* __restrict__ psi_off, long long psi_tot, const double* __restrict__ wts,
          float* __restrict__ Hbar, int HSh, double* __restrict__ Ebar, double* __restrict__ siteval,
          long long sv_stride, bool pair, float* __restrict__ scratch, size_t slot_elems) {
  using T = float;
  constexpr int NT = F32_THREADS, NC = NO;
  constexpr int N = NO * NC;
  constexpr int PS = (N == 1) ? 1 : Row<T, N>::PS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf[2];
  buf[0] = GMEM ? scratch + (size_t)blockIdx.x * slot_elems : reinterpret_cast<T*>(smem_raw);
  buf[1] = buf[0] + (size_t)L.cap_even * PS;
  // [cap_eb][NO], padded to 16 bytes
  T* eb = GMEM ? reinterpret_cast<T*>(smem_raw) : buf[1] + (size_t)L.cap_odd * PS;
  unsigned char* tail = align16(reinterpret_cast<unsigned char*>(eb + eb_elems<T, NO>(L.cap_eb)));
  int2* s_adj = reinterpret_cast<int2*>(tail);
  unsigned long long* s_lvc = reinterpret_cast<unsigned long long*>(s_adj + (L.stage ? L.max_adj : 0));
  int* s_off = reinterpret_cast<int*>(s_lvc + (L.stage ? L.cap_eb : 0));
  int* s_atom = s_off + (L.stage ? L.cap_eb + 1 : 0);
  __shared__ T ws[NC][BOP_MAX_NMOM];
  __shared__ int s_lev[BOP_MAX_K + 1];
  __shared__ long long s_lo[BOP_MAX_K + 1];
  __shared__ unsigned s_sel[REV_SEL_WORDS];
  const int K = cv.K;
  const int tid = threadIdx.x, lane = tid & 31;
  int w0, w1;
  item_range(n_items, &w0, &w1);
  ItemExt nx{};
  if (w0 < w1) {
    ext_sites(cv, w0 % n, nx);
    ext_adj(cv, nx);
  }
  for (int w = w0; w < w1; w++) {
    const int spin = w / n, atom = w % n;
    const ItemExt cur = nx;
    const long long s0 = cur.s0, abase = cur.abase;
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const unsigned long long* lvc = L.stage ? s_lvc : cv.lvcnt + s0;
    const int* satom = L.stage ? s_atom : cv.site_atom + s0;
    const unsigned* top = cv.top + s0;
    const T* E = onsite + (size_t)spin * n_on * NO;
    const size_t ib = ((size_t)spin * psi_tot + psi_off[atom]) * PS;
    const T* P = pstore + ib;
    if (L.stage) {
      const int nr = lev[K - 1];
      stage_item(cv, cur, nr, (int)(cv.adj_off[s0 + nr] - abase), s_adj, s_off, s_lvc, s_atom, tid, NT);
    }
    const int2* adj = L.stage ? s_adj : cv.adj + abase;
    const bool more = w + 1 < w1;
    if (more) ext_sites(cv, (w + 1) % n, nx);
    if (tid <= K) s_lev[tid] = lev[tid];
    if (tid == 0) {
      long long o = 0;
      for (int k = 0; k <= K; k++) {
        s_lo[k] = o;
        o += lev[k];
      }
    }
    for (int q = tid; q < NC * n_mom; q += NT) {
      const int c = q / n_mom, m = q % n_mom;
      ws[c][m] = (T)wts[((size_t)w * NO + c) * n_mom + m];
    }
    if (pair)
      for (int q = tid; q < REV_SEL_WORDS; q += NT) s_sel[q] = 0;
    __syncthreads();
    const int neb = s_lev[K - 1];
    for (int q = tid; q < neb * NO; q += NT) eb[q] = T(0);
    // Psi-bar_K
    T* xK = buf[K & 1];
    if (pair) {
      // rows that are not selected enter with zero
      const T zero[N] = {};
      for (int t = tid; t < neb; t += NT) store_row<T, N, PS>(xK + (size_t)t * PS, zero);
      __syncthreads();
    }
    const int nK = pair ? cv.ntop[atom] & 0xffff : s_lev[K];
    for (int q = tid; q < nK; q += NT) {
      const int t = pair ? (int)(top[q] & 0xffffu) : q;
      // weights of the site's atom (rows), in the pair form
      T wj2[NO], wj1[NO];
#pragma unroll
      for (int r = 0; r < NO; r++) wj2[r] = wj1[r] = T(0);
      if (pair) {
        if (t < neb) atomicOr(&s_sel[t >> 5], 1u << (t & 31));
        if (t != 0) {
          const double* wj = wts + ((size_t)spin * n + satom[t]) * NO * n_mom + 2 * K - 1;
#pragma unroll
          for (int r = 0; r < NO; r++) {
            wj1[r] = (T)wj[r * n_mom];
            wj2[r] = (T)wj[r * n_mom + 1];
          }
        }
      }
      T pk[N], row[N];
      load_row<T, N, PS>(P + (size_t)(s_lo[K] + t) * PS, pk);
#pragma unroll
      for (int v = 0; v < N; v++) row[v] = T(2) * (ws[v % NC][2 * K] + wj2[v / NC]) * pk[v];
      if (t < neb) {
        T pk1[N];
        load_row<T, N, PS>(P + (size_t)(s_lo[K - 1] + t) * PS, pk1);
#pragma unroll
        for (int v = 0; v < N; v++) row[v] += (ws[v % NC][2 * K - 1] + wj1[v / NC]) * pk1[v];
      }
      store_row<T, N, PS>(xK + (size_t)t * PS, row);
    }
    __syncthreads();
    for (int k = K; k >= 1; k--) {
      const bool half = pair && k == K;
      const T* xb = buf[k & 1];
      T* yb = buf[(k - 1) & 1];
      const int nrow = s_lev[k - 1];
      int psh = 0;  // lanes per row, as a shift
      if (!half)
        while (psh < 4 && (nrow << (psh + 1)) <= NT) psh++;
      const int part = tid & ((1 << psh) - 1);
      for (int r0 = 0; r0 < nrow; r0 += NT >> psh) {
        if (r0 + ((tid & ~31) >> psh) >= nrow) continue;  // whole warps
        const int rr = r0 + (tid >> psh);
        const bool live = rr < nrow;
        const int t = !live ? 0 : (half ? (int)(top[rr] >> 16) : rr);
        const T* r1 = P + (size_t)(s_lo[k - 1] + t) * PS;
        if (live && part == 0) {
          // the stored rows this site needs, towards L2 while the gather runs
          prefetch_row_l2<T, PS>(r1);
          if (k >= 2) {
            prefetch_row_l2<T, PS>(P + (size_t)(s_lo[k] + t) * PS);
            if (t < s_lev[k - 2]) prefetch_row_l2<T, PS>(P + (size_t)(s_lo[k - 2] + t) * PS);
          }
        }
        T acc[NO][NC];
#pragma unroll
        for (int r = 0; r < NO; r++)
#pragma unroll
          for (int c = 0; c < NC; c++) acc[r][c] = T(0);
        if (k >= 2 && live && part == 0) {
          T xt[N];
          load_row<T, N, PS>(xb + (size_t)t * PS, xt);
          const T* e = E + (size_t)satom[t] * NO;
#pragma unroll
          for (int r = 0; r < NO; r++) {
            const T er = e[r];
#pragma unroll
            for (int c = 0; c < NC; c++) acc[r][c] = er * xt[r * NC + c];
          }
        }
        if (k >= 2 || HBAR) {
          const int q0 = L.stage ? s_off[t] : (int)(cv.adj_off[s0 + t] - abase);
          int cnt = 0;
          if (live) {
            if (k < K) cnt = (int)((lvc[t] >> (8 * k)) & 0xff);
            else cnt = L.stage ? s_off[t + 1] - q0 : (int)(cv.adj_off[s0 + t + 1] - abase) - q0;
          }
          const unsigned mask = half && live ? cv.topmask[s0 + t] : 0u;
          T pt[N];
          if constexpr (HBAR) {
            if (live) {
              load_row<T, N, PS>(r1, pt);
            } else {
#pragma unroll
              for (int v = 0; v < N; v++) pt[v] = T(0);
            }
          }
          gather_rev<T, NO, NC, PS, HBAR>(adj + q0, part, 1 << psh, cnt, mask, half, H, HS, xb, acc, k >= 2, pt, Hbar,
                                          HSh, lane);
          for (int o = 1; o < (1 << psh); o <<= 1) {
#pragma unroll
            for (int r = 0; r < NO; r++)
#pragma unroll
              for (int c = 0; c < NC; c++) acc[r][c] += __shfl_xor_sync(0xffffffffu, acc[r][c], o);
          }
        }
        if (!live || part != 0) continue;
        // onsite cotangent of level k: Psi-bar_k[t] . Psi_k-1[t] (rows read after the gather)
        T p1[N];
        {
          T xt[N];
          load_row<T, N, PS>(xb + (size_t)t * PS, xt);
          load_row<T, N, PS>(r1, p1);
#pragma unroll
          for (int r = 0; r < NO; r++) {
            T a = T(0);
#pragma unroll
            for (int c = 0; c < NC; c++) a += xt[r * NC + c] * p1[r * NC + c];
            eb[t * NO + r] += a;
          }
        }
        if (k >= 2) {
          T row[N];
#pragma unroll
          for (int v = 0; v < N; v++) row[v] = acc[v / NC][v % NC] + T(2) * ws[v % NC][2 * k - 2] * p1[v];
          if (!half || (s_sel[t >> 5] >> (t & 31) & 1u)) {
            T pk[N], wj[NO];
            load_row<T, N, PS>(P + (size_t)(s_lo[k] + t) * PS, pk);
#pragma unroll
            for (int r = 0; r < NO; r++)
              wj[r] = half && t != 0 ? (T)wts[(((size_t)spin * n + satom[t]) * NO + r) * n_mom + 2 * K - 1] : T(0);
#pragma unroll
            for (int v = 0; v < N; v++) row[v] += (ws[v % NC][2 * k - 1] + wj[v / NC]) * pk[v];
          }
          if (t < s_lev[k - 2]) {
            T p2[N];
            load_row<T, N, PS>(P + (size_t)(s_lo[k - 2] + t) * PS, p2);
#pragma unroll
            for (int v = 0; v < N; v++) row[v] += ws[v % NC][2 * k - 3] * p2[v];
          }
          store_row<T, N, PS>(yb + (size_t)t * PS, row);
        }
      }
      __syncthreads();
    }
    if (Ebar != nullptr) {
      for (int q = tid; q < neb * NO; q += NT) {
        const int t = q / NO, r = q % NO;
        atomicAdd(Ebar + ((size_t)spin * n_on + satom[t]) * NO + r, (double)eb[q]);
      }
    }
    if (siteval != nullptr) {  // per-site sums over the orbitals (one row of the SCF Jacobian)
      for (int t = tid; t < neb; t += NT) {
        double a = 0.0;
#pragma unroll
        for (int r = 0; r < NO; r++) a += (double)eb[t * NO + r];
        atomicAdd(siteval + (size_t)spin * sv_stride + s0 + t, a);
      }
    }
    if (more) ext_adj(cv, nx);
    __syncthreads();
  }
}

// FP64 (see k_moments64): lane r of a site holds row r of its block.  HBAR: for
// the bond cotangents dL/dB = x[s] pt^T (x = Psi-bar_k, pt = Psi_k-1(t)) lane r
// forms column r from its row of pt and the whole x[s], rows taken in the order
// r, r + 1, .. (mod NO): what its unique elements (r, r), (r, r + 1), (r, r + 2)
// still lack then sits in the same place of another lane of the site, and two
// shuffles replace a sum over lanes.
//
// The entries first, first + step, ... of the row, or those of the bits of
// mask.  All lanes of a warp call it (rows of no entries: cnt 0); rounds run
// together with HBAR.  u[j], o[j]: positions of B[r][(r + j) % NO] in the bond
// record and of row (r + j) % NO in a Psi row.
template <int NO, int PS, bool HBAR>
__device__ __forceinline__ void gather_rev64(const int2* __restrict__ ent, int first, int step, int cnt, unsigned mask,
                                             bool use_mask, const double* __restrict__ H, int HS,
                                             const double* __restrict__ x, const int u[NO], const int o[NO],
                                             double acc[NO], bool gather, const double pt[NO],
                                             double* __restrict__ Hbar, int HSh, int lane, int r) {
  const int mine = use_mask ? __popc(mask) : (cnt > first ? (cnt - first + step - 1) / step : 0);
  const int rounds = HBAR ? __reduce_max_sync(0xffffffffu, mine) : mine;
  int e = first;
  auto next = [&]() -> int2 {  // the row's next entry
    int i = e;
    if (use_mask) {
      i = __ffs(mask) - 1;
      mask &= mask - 1;
    }
    e += step;
    return ent[i];
  };
  int2 e0 = make_int2(0, -1), e1 = make_int2(0, -1);
  double b0[NO], b1[NO];
#pragma unroll
  for (int j = 0; j < NO; j++) b0[j] = b1[j] = 0.0;
  auto load = [&](int bond, double b[NO]) {
#pragma unroll
    for (int j = 0; j < NO; j++) b[j] = __ldg(H + (size_t)bond * HS + u[j]);
  };
  if (mine > 0) {
    e0 = next();
    if (gather) load(e0.y, b0);
  }
  if (mine > 1) {
    e1 = next();
    if (gather) load(e1.y, b1);
  }
  for (int it = 0; it < rounds; it++) {
    const bool on = it < mine;
    const int s = e0.x, bond = on ? e0.y : -1;
    double b[NO];
#pragma unroll
    for (int j = 0; j < NO; j++) {
      b[j] = b0[j];
      b0[j] = b1[j];
    }
    e0 = e1;
    if (it + 2 < mine) {
      e1 = next();
      if (gather) load(e1.y, b1);
    }
    if constexpr (!HBAR) {
      double xs[NO * NO];
      load_row<double, NO * NO, PS>(x + (size_t)s * PS, xs);
      // (u is not rotated without HBAR)
#pragma unroll
      for (int g = 0; g < NO; g++)
#pragma unroll
        for (int c = 0; c < NO; c++) acc[c] += b[g] * xs[g * NO + c];
    } else {
      double G[NO];  // G[j] = dL/dB[(r + j) % NO][r]
#pragma unroll
      for (int j = 0; j < NO; j++) G[j] = 0.0;
      if (on) {
        const double* xr = x + (size_t)s * PS;
#pragma unroll
        for (int j = 0; j < NO; j++)
#pragma unroll
          for (int c = 0; c < NO; c++) {
            const double v = xr[o[j] + c];
            acc[c] += b[j] * v;
            G[j] += v * pt[c];
          }
      }
      double* hb = Hbar + (size_t)(bond < 0 ? 0 : bond) * HSh;
      if (bond >= 0) atomicAdd(hb + u[0], G[0]);
#pragma unroll
      for (int j = 1; j <= NO / 2; j++) {
        // lane (r + j) % NO of the site holds dL/dB[r][(r + j) % NO] as its G[NO - j]
        const double other = __shfl_sync(0xffffffffu, G[NO - j], lane + (r + j < NO ? j : j - NO));
        if (bond >= 0 && (2 * j < NO || r < j)) atomicAdd(hb + u[j], G[j] + other);
      }
    }
  }
}

template <int NO, bool HBAR, bool GMEM>
__global__ void __launch_bounds__(F64_REV_THREADS, 3)
k_adj_rev64(ClusterView cv, const double* __restrict__ H, int HS, const double* __restrict__ onsite, int n, int n_on,
            int n_mom, RevSmem L, int n_items, const double* __restrict__ pstore,
            const long long* __restrict__ psi_off, long long psi_tot, const double* __restrict__ wts,
            double* __restrict__ Hbar, int HSh, double* __restrict__ Ebar, double* __restrict__ siteval,
            long long sv_stride, bool pair, double* __restrict__ scratch, size_t slot_elems) {
  constexpr int NT = F64_REV_THREADS, NC = NO, RPW = 32 / NO;
  constexpr int N = NO * NC;
  constexpr int PS = (N == 1) ? 1 : Row<double, N>::PS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* buf[2];
  buf[0] = GMEM ? scratch + (size_t)blockIdx.x * slot_elems : reinterpret_cast<double*>(smem_raw);
  buf[1] = buf[0] + (size_t)L.cap_even * PS;
  // [cap_eb][NO], padded to 16 bytes
  double* eb = GMEM ? reinterpret_cast<double*>(smem_raw) : buf[1] + (size_t)L.cap_odd * PS;
  unsigned char* tail = align16(reinterpret_cast<unsigned char*>(eb + eb_elems<double, NO>(L.cap_eb)));
  int2* s_adj = reinterpret_cast<int2*>(tail);
  unsigned long long* s_lvc = reinterpret_cast<unsigned long long*>(s_adj + (L.stage ? L.max_adj : 0));
  int* s_off = reinterpret_cast<int*>(s_lvc + (L.stage ? L.cap_eb : 0));
  int* s_atom = s_off + (L.stage ? L.cap_eb + 1 : 0);
  __shared__ double ws[NC][BOP_MAX_NMOM];
  __shared__ int s_lev[BOP_MAX_K + 1], s_next[BOP_MAX_K + 1];
  __shared__ long long s_lo[BOP_MAX_K + 1];
  __shared__ unsigned s_sel[REV_SEL_WORDS];
  const int K = cv.K;
  const int tid = threadIdx.x, lane = tid & 31;
  const int grp = lane / NO, r = lane % NO;
  int u[NO], o[NO];
#pragma unroll
  for (int j = 0; j < NO; j++) {
    const int g = HBAR ? (r + j) % NO : j;
    u[j] = UI<NO>(r, g);
    o[j] = g * NC;
  }
  ItemExt nx{};
  if ((int)blockIdx.x < n_items) {
    ext_sites(cv, blockIdx.x % n, nx);
    ext_adj(cv, nx);
  }
  for (int w = blockIdx.x; w < n_items; w += gridDim.x) {
    const int spin = w / n, atom = w % n;
    const ItemExt cur = nx;
    const long long s0 = cur.s0, abase = cur.abase;
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const unsigned long long* lvc = L.stage ? s_lvc : cv.lvcnt + s0;
    const int* satom = L.stage ? s_atom : cv.site_atom + s0;
    const unsigned* top = cv.top + s0;
    const double* E = onsite + (size_t)spin * n_on * NO;
    const double* P = pstore + ((size_t)spin * psi_tot + psi_off[atom]) * PS;
    if (L.stage) {
      const int nr = lev[K - 1];
      stage_item(cv, cur, nr, (int)(cv.adj_off[s0 + nr] - abase), s_adj, s_off, s_lvc, s_atom, tid, NT);
    }
    const int2* adj = L.stage ? s_adj : cv.adj + abase;
    const bool more = n_items - w > (int)gridDim.x;
    if (more) ext_sites(cv, (w + gridDim.x) % n, nx);
    if (tid <= K) {
      s_lev[tid] = lev[tid];
      s_next[tid] = 0;
    }
    if (tid == 0) {
      long long lo = 0;
      for (int k = 0; k <= K; k++) {
        s_lo[k] = lo;
        lo += lev[k];
      }
    }
    for (int q = tid; q < NC * n_mom; q += NT) {
      const int c = q / n_mom, m = q % n_mom;
      ws[c][m] = wts[((size_t)w * NO + c) * n_mom + m];
    }
    if (pair)
      for (int q = tid; q < REV_SEL_WORDS; q += NT) s_sel[q] = 0;
    __syncthreads();
    const int neb = s_lev[K - 1];
    for (int q = tid; q < neb * NO; q += NT) eb[q] = 0.0;
    // Psi-bar_K
    double* xK = buf[K & 1];
    if (pair) {  // rows that are not selected enter with zero
      for (int q = tid; q < neb * PS; q += NT) xK[q] = 0.0;
      __syncthreads();
    }
    const int nK = pair ? cv.ntop[atom] & 0xffff : s_lev[K];
    for (int q = tid; q < nK * NO; q += NT) {
      const int i = q / NO, b = q % NO;
      const int t = pair ? (int)(top[i] & 0xffffu) : i;
      // weights of the site's atom (rows), in the pair form
      double wj2 = 0.0, wj1 = 0.0;
      if (pair) {
        if (b == 0 && t < neb) atomicOr(&s_sel[t >> 5], 1u << (t & 31));
        if (t != 0) {
          const double* wj = wts + (((size_t)spin * n + satom[t]) * NO + b) * n_mom + 2 * K - 1;
          wj1 = wj[0];
          wj2 = wj[1];
        }
      }
      const double* pk = P + (size_t)(s_lo[K] + t) * PS + b * NC;
      double* row = xK + (size_t)t * PS + b * NC;
      const double* p1 = P + (size_t)(s_lo[K - 1] + t) * PS + b * NC;
#pragma unroll
      for (int c = 0; c < NC; c++) {
        double v = 2.0 * (ws[c][2 * K] + wj2) * pk[c];
        if (t < neb) v += (ws[c][2 * K - 1] + wj1) * p1[c];
        row[c] = v;
      }
    }
    __syncthreads();
    for (int k = K; k >= 1; k--) {
      const bool half = pair && k == K;
      const double* xb = buf[k & 1];
      double* yb = buf[(k - 1) & 1];
      const int nrow = s_lev[k - 1];
      // lanes of few rows: P parts of a row's entries each on its own lanes,
      // where that shortens the rounds of the CTA's warps.  A row is priced at 16
      // entries, whatever its length (14 in bcc, 18 in fcc, fewer at a surface):
      // sweeps of 2,000 bcc / 1,372 fcc atoms at 9 moments and 686 bcc at 13 take
      // 2.89 / 3.33 / 5.56 ms so, 2.89 / 3.32 / 6.03 priced at 14, 2.89 / 3.24 /
      // 5.42 at 18, 3.59 / 3.33 / 5.95 at 64
      int parts = 1, rows = RPW;  // rows of a warp
      if (!half) {
        int best = 1 << 30;
#pragma unroll
        for (int p = 1; p <= (RPW < 8 ? RPW : 8); p++) {
          const int rp = RPW / p, len = (nrow + rp * (NT / 32) - 1) / (rp * (NT / 32)) * (16 / p + 1);
          if (len < best) {
            best = len;
            parts = p;
            rows = rp;
          }
        }
      }
      const int part = grp % parts, sub = grp / parts;
      while (true) {
        int first = 0;
        if (lane == 0) first = atomicAdd(&s_next[k], rows);
        first = __shfl_sync(0xffffffffu, first, 0);
        if (first >= nrow) break;
        const int rr = first + sub;
        const bool live = sub < rows && rr < nrow;
        const int t = !live ? 0 : (half ? (int)(top[rr] >> 16) : rr);
        const double* r1 = P + (size_t)(s_lo[k - 1] + t) * PS + r * NC;
        double pt[NC], acc[NC];
#pragma unroll
        for (int c = 0; c < NC; c++) {
          pt[c] = live ? r1[c] : 0.0;
          acc[c] = 0.0;
        }
        const bool own = live && part == 0;
        const double* xt = xb + (size_t)t * PS + r * NC;
        if (own) {
          if (r == 0 && k >= 2) {  // the stored rows this site needs, towards L2 while the gather runs
            prefetch_row_l2<double, PS>(P + (size_t)(s_lo[k] + t) * PS);
            if (t < s_lev[k - 2]) prefetch_row_l2<double, PS>(P + (size_t)(s_lo[k - 2] + t) * PS);
          }
          if (k >= 2) {
            const double er = E[(size_t)satom[t] * NO + r];
#pragma unroll
            for (int c = 0; c < NC; c++) acc[c] = er * xt[c];
          }
        }
        if (k >= 2 || HBAR) {
          const int q0 = L.stage ? s_off[t] : (int)(cv.adj_off[s0 + t] - abase);
          int cnt = 0;
          if (live) {
            if (k < K) cnt = (int)((lvc[t] >> (8 * k)) & 0xff);
            else cnt = L.stage ? s_off[t + 1] - q0 : (int)(cv.adj_off[s0 + t + 1] - abase) - q0;
          }
          const unsigned mask = half && live ? cv.topmask[s0 + t] : 0u;
          gather_rev64<NO, PS, HBAR>(adj + q0, part, parts, cnt, mask, half, H, HS, xb, u, o, acc, k >= 2, pt, Hbar,
                                     HSh, lane, r);
          __syncwarp();
          for (int p = 1; p < parts; p++)
#pragma unroll
            for (int c = 0; c < NC; c++) {
              const double v = __shfl_sync(0xffffffffu, acc[c], lane + p * NO);
              if (part == 0) acc[c] += v;
            }
        }
        if (!own) continue;
        // onsite cotangent of level k: Psi-bar_k[t] . Psi_k-1[t]
        double a = 0.0;
#pragma unroll
        for (int c = 0; c < NC; c++) a += xt[c] * pt[c];
        eb[t * NO + r] += a;
        if (k >= 2) {
          const bool has_k = !half || (s_sel[t >> 5] >> (t & 31) & 1u), has_2 = t < s_lev[k - 2];
          const double wj = half && t != 0 ? wts[(((size_t)spin * n + satom[t]) * NO + r) * n_mom + 2 * K - 1] : 0.0;
          const double* pk = P + (size_t)(s_lo[k] + t) * PS + r * NC;
          const double* p2 = P + (size_t)(s_lo[k - 2] + t) * PS + r * NC;
#pragma unroll
          for (int c = 0; c < NC; c++) {
            double v = acc[c] + 2.0 * ws[c][2 * k - 2] * pt[c];
            if (has_k) v += (ws[c][2 * k - 1] + wj) * pk[c];
            if (has_2) v += ws[c][2 * k - 3] * p2[c];
            yb[(size_t)t * PS + r * NC + c] = v;
          }
        }
      }
      __syncthreads();
    }
    if (Ebar != nullptr) {
      for (int q = tid; q < neb * NO; q += NT) {
        const int t = q / NO, b = q % NO;
        atomicAdd(Ebar + ((size_t)spin * n_on + satom[t]) * NO + b, eb[q]);
      }
    }
    if (siteval != nullptr) {  // per-site sums over the orbitals (one row of the SCF Jacobian)
      for (int t = tid; t < neb; t += NT) {
        double a = 0.0;
#pragma unroll
        for (int b = 0; b < NO; b++) a += eb[t * NO + b];
        atomicAdd(siteval + (size_t)spin * sv_stride + s0 + t, a);
      }
    }
    if (more) ext_adj(cv, nx);
    __syncthreads();
  }
}

// ------------------------------------------------------------------ adjoint (recompute)
__device__ __forceinline__ int site_level(const int* lev, int K, int t) {
  int k = 0;
  while (k < K && t >= lev[k]) k++;
  return k;
}

template <typename T, int NO>
__global__ void __launch_bounds__(MOM_THREADS)
k_moments_adj(ClusterView cv, const T* __restrict__ H, int HS, const T* __restrict__ onsite, int n, int n_on, int n_mom,
              int nwork, const double* __restrict__ wts, T* __restrict__ scratch, size_t slot_elems,
              T* __restrict__ Hbar, int HSh, double* __restrict__ Ebar) {
  constexpr int NC = NO;
  __shared__ T ws[NC][BOP_MAX_NMOM];
  __shared__ int s_lev[BOP_MAX_K + 1];
  __shared__ long long s_off[BOP_MAX_K + 2];
  const int K = cv.K;
  const int tid = threadIdx.x;
  T* psi = scratch + (size_t)blockIdx.x * slot_elems;
  for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
    const int spin = w / n, atom = w % n;
    const long long s0 = cv.site_off[atom];
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const int* satom = cv.site_atom + s0;
    const long long* aoff = cv.adj_off + s0;
    const T* E = onsite + (size_t)spin * n_on * NO;
    if (tid <= K) s_lev[tid] = lev[tid];
    if (tid == 0) {  // Psi_k at s_off[k], Psi-bar_k at s_off[K+1] + (s_off[k] - s_off[1])
      long long o = 0;
      for (int k = 0; k <= K; k++) {
        s_off[k] = o;
        o += (long long)lev[k] * NO * NC;
      }
      s_off[K + 1] = o;
    }
    for (int q = tid; q < NC * n_mom; q += blockDim.x) {
      int c = q / n_mom, m = q % n_mom;
      ws[c][m] = (T)wts[((size_t)w * NO + c) * n_mom + m];
    }
    __syncthreads();
    T* P = psi;
    T* Pb = psi + s_off[K + 1] - s_off[1];  // Pb + s_off[k] is Psi-bar_k (k >= 1)
    // forward: all levels
    for (int q = tid; q < NO * NC; q += blockDim.x) P[q] = T(q / NC == q % NC ? 1 : 0);
    __syncthreads();
    for (int k = 1; k <= K; k++) {
      const T* x = P + s_off[k - 1];
      T* y = P + s_off[k];
      for (int t = tid; t < s_lev[k]; t += blockDim.x) {
        T acc[NO][NC];
        gather_row<T, NO, NC>(cv, H, HS, E, satom, aoff, t, s_lev[k - 1], x, acc);
#pragma unroll
        for (int r = 0; r < NO; r++)
#pragma unroll
          for (int c = 0; c < NC; c++) y[(t * NO + r) * NC + c] = acc[r][c];
      }
      __syncthreads();
    }
    // Psi-bar_K = 2 w_2K Psi_K + w_2K-1 Psi_K-1
    {
      const T* PK = P + s_off[K];
      const T* PK1 = P + s_off[K - 1];
      T* B = Pb + s_off[K];
      for (int q = tid; q < s_lev[K] * NO * NC; q += blockDim.x) {
        int t = q / (NO * NC), c = q % NC;
        T v = T(2) * ws[c][2 * K] * PK[q];
        if (t < s_lev[K - 1]) v += ws[c][2 * K - 1] * PK1[q];
        B[q] = v;
      }
    }
    __syncthreads();
    // Psi-bar_{k-1} = H^T Psi-bar_k (rows < |C_k-1|, cols < |C_k|) + dot-product terms
    for (int k = K; k >= 2; k--) {
      const T* xb = Pb + s_off[k];
      T* yb = Pb + s_off[k - 1];
      const T* Pk = P + s_off[k];
      const T* Pk1 = P + s_off[k - 1];
      const T* Pk2 = P + s_off[k - 2];
      for (int t = tid; t < s_lev[k - 1]; t += blockDim.x) {
        T acc[NO][NC];
        gather_row<T, NO, NC>(cv, H, HS, E, satom, aoff, t, s_lev[k], xb, acc);
#pragma unroll
        for (int r = 0; r < NO; r++)
#pragma unroll
          for (int c = 0; c < NC; c++) {
            int q = (t * NO + r) * NC + c;
            T v = acc[r][c] + T(2) * ws[c][2 * k - 2] * Pk1[q] + ws[c][2 * k - 1] * Pk[q];
            if (t < s_lev[k - 2]) v += ws[c][2 * k - 3] * Pk2[q];
            yb[q] = v;
          }
      }
      __syncthreads();
    }
    // bond and onsite cotangents: dU/dH_ts = sum_k Psi-bar_k[t] Psi_k-1[s]^T
    for (int t = tid; t < s_lev[K]; t += blockDim.x) {
      const int lt = site_level(s_lev, K, t);
      const long long q1 = Hbar != nullptr ? aoff[t + 1] : aoff[t];  // no bond cotangents wanted
      for (long long q = aoff[t]; q < q1; q++) {
        int2 en = cv.adj[q];
        const int s = en.x;
        if (s >= s_lev[K - 1]) break;
        const int ls = site_level(s_lev, K, s);
        const int kmin = lt > ls + 1 ? lt : ls + 1;
        T G[NO][NO];
#pragma unroll
        for (int b = 0; b < NO; b++)
#pragma unroll
          for (int g = 0; g < NO; g++) G[b][g] = T(0);
        for (int k = kmin; k <= K; k++) {
          const T* pb = Pb + s_off[k] + (size_t)t * NO * NC;
          const T* ps = P + s_off[k - 1] + (size_t)s * NO * NC;
#pragma unroll
          for (int b = 0; b < NO; b++)
#pragma unroll
            for (int g = 0; g < NO; g++) {
              T a = T(0);
#pragma unroll
              for (int c = 0; c < NC; c++) a += pb[b * NC + c] * ps[g * NC + c];
              G[b][g] += a;
            }
        }
        add_bond_cotangent<T, NO>(Hbar + (size_t)en.y * HSh, G);
      }
      if (Ebar != nullptr) {
        double eb[NO];
#pragma unroll
        for (int b = 0; b < NO; b++) eb[b] = 0.0;
        for (int k = lt + 1; k <= K; k++) {
          const T* pb = Pb + s_off[k] + (size_t)t * NO * NC;
          const T* pt = P + s_off[k - 1] + (size_t)t * NO * NC;
#pragma unroll
          for (int b = 0; b < NO; b++) {
            T a = T(0);
#pragma unroll
            for (int c = 0; c < NC; c++) a += pb[b * NC + c] * pt[b * NC + c];
            eb[b] += (double)a;
          }
        }
        if (lt + 1 <= K) {
          double* ep = Ebar + ((size_t)spin * n_on + satom[t]) * NO;
#pragma unroll
          for (int b = 0; b < NO; b++) atomicAdd(ep + b, eb[b]);
        }
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ non-collinear spin moments
// Non-collinear magnetism (section "Magnetism", Eqs. onsite_CM and
// onsite-noncollinear).  Work item (atom i, orbital alpha); its two
// starting states are the local spin states of atom i, chi_up antiparallel
// to the moment direction s_i (eigenvalue -1 of s_i.sigma, the lower level)
// and chi_dn parallel, complex 2-spinors in the spin basis along z.  A site
// row holds NO x 8 reals, column c = nu * 4 + sp * 2 + ri (starting spinor
// nu, spin component sp, real / imaginary part).  The hopping H_e x 1 acts
// on the orbital index (block_apply with 8 columns); the onsite matrix
// Ebar + h.sigma, Ebar = (E_up + E_dn)/2, h = (E_dn - E_up)/2 s_j, mixes
// the four reals of each spinor.  In this real form every operator is
// symmetric, so the reverse sweep gathers with the same rows.
//   forward (wts == NULL): local channel moments mu_nu,n = <chi_nu|H^n|chi_nu>
//   into mu[nu] and Tr(sigma M_n) of the global 2x2 moments M_n into vmom;
//   reverse (wts != NULL): cotangents of L = sum w_nu,n mu_nu,n for every
//   bond block (Hbar, in the product type: float4 reductions in FP32) and
//   every onsite matrix
//   (obar = dL/d(Ebar, h_x, h_y, h_z)).
// Psi_0..Psi_K (and Psi-bar_1..Psi-bar_K) of the item live in the CTA's
// slot of global scratch, as in k_moments_adj.
constexpr int NCS = 8;

// chi_up = (-(x - i y), 1 + z) r, chi_dn = (1 + z, x + i y) r for z >= 0,
// chi_up = (1 - z, -(x + i y)) r, chi_dn = (x - i y, 1 - z) r otherwise
// (r normalises; the second form avoids the zero of 1 + z at s = -z).
__device__ __forceinline__ void start_spinors(const double* s, double* out) {
  const double x = s[0], y = s[1], z = s[2];
  if (z >= 0.0) {
    const double r = 1.0 / sqrt(2.0 * (1.0 + z));
    out[0] = -x * r; out[1] = y * r; out[2] = (1.0 + z) * r; out[3] = 0.0;
    out[4] = (1.0 + z) * r; out[5] = 0.0; out[6] = x * r; out[7] = y * r;
  } else {
    const double r = 1.0 / sqrt(2.0 * (1.0 - z));
    out[0] = (1.0 - z) * r; out[1] = 0.0; out[2] = -x * r; out[3] = -y * r;
    out[4] = x * r; out[5] = -y * r; out[6] = (1.0 - z) * r; out[7] = 0.0;
  }
}

// y = (Ebar + h.sigma) x for both spinors of one orbital row
template <typename T>
__device__ __forceinline__ void spin_onsite(T eb, T hx, T hy, T hz, const T* __restrict__ x, T* y) {
#pragma unroll
  for (int nu = 0; nu < 2; nu++) {
    const T ur = x[4 * nu], ui = x[4 * nu + 1], dr = x[4 * nu + 2], di = x[4 * nu + 3];
    y[4 * nu] = (eb + hz) * ur + hx * dr + hy * di;
    y[4 * nu + 1] = (eb + hz) * ui + hx * di - hy * dr;
    y[4 * nu + 2] = (eb - hz) * dr + hx * ur - hy * ui;
    y[4 * nu + 3] = (eb - hz) * di + hx * ui + hy * ur;
  }
}

// acc = (H x)[t] over columns s < ncol (onsite term when t < ncol)
template <typename T, int NO>
__device__ __forceinline__ void gather_row_nc(const ClusterView& cv, const T* __restrict__ H, int HS,
                                              const T* __restrict__ E, const double* __restrict__ sdir, int n,
                                              const int* __restrict__ satom, const long long* __restrict__ aoff,
                                              int t, int ncol, const T* __restrict__ x, T acc[NO][NCS]) {
#pragma unroll
  for (int r = 0; r < NO; r++)
#pragma unroll
    for (int c = 0; c < NCS; c++) acc[r][c] = T(0);
  if (t < ncol) {
    const int j = satom[t];
    const T sx = (T)sdir[3 * (size_t)j], sy = (T)sdir[3 * (size_t)j + 1], sz = (T)sdir[3 * (size_t)j + 2];
#pragma unroll
    for (int r = 0; r < NO; r++) {
      const T eu = E[(size_t)j * NO + r], ed = E[((size_t)n + j) * NO + r];
      const T f = T(0.5) * (ed - eu);
      spin_onsite<T>(T(0.5) * (eu + ed), f * sx, f * sy, f * sz, x + ((size_t)t * NO + r) * NCS, acc[r]);
    }
  }
  const long long q1 = aoff[t + 1];
  for (long long q = aoff[t]; q < q1; q++) {
    const int2 en = cv.adj[q];
    if (en.x >= ncol) break;
    block_apply<T, NO, NCS>(H + (size_t)en.y * HS, x + (size_t)en.x * NO * NCS, acc);
  }
}

// Tr(sigma M) of M = C L C^dagger, C = (chi_up chi_dn), L = [[Luu, Lud],
// [conj(Lud), Ldd]] the moments between the local states.
__device__ __forceinline__ void pauli_from_local(const double* chi, double Luu, double Ldd, double Lr, double Li,
                                                 double v[3]) {
  // C_a,nu = chi[nu * 4 + a * 2] + i chi[nu * 4 + a * 2 + 1]
  double M00 = 0.0, M11 = 0.0, M01r = 0.0, M01i = 0.0;
  const double L[2][2][2] = {{{Luu, 0.0}, {Lr, Li}}, {{Lr, -Li}, {Ldd, 0.0}}};  // [nu][nu'][re/im]
#pragma unroll
  for (int nu = 0; nu < 2; nu++)
#pragma unroll
    for (int mu_ = 0; mu_ < 2; mu_++) {
      const double lr = L[nu][mu_][0], li = L[nu][mu_][1];
      // M_ab += C_a,nu L_nu,mu conj(C_b,mu)
      const double c0r = chi[nu * 4], c0i = chi[nu * 4 + 1], c1r = chi[nu * 4 + 2], c1i = chi[nu * 4 + 3];
      const double d0r = chi[mu_ * 4], d0i = chi[mu_ * 4 + 1], d1r = chi[mu_ * 4 + 2], d1i = chi[mu_ * 4 + 3];
      // x = C_a,nu L
      const double x0r = c0r * lr - c0i * li, x0i = c0r * li + c0i * lr;
      const double x1r = c1r * lr - c1i * li, x1i = c1r * li + c1i * lr;
      M00 += x0r * d0r + x0i * d0i;
      M11 += x1r * d1r + x1i * d1i;
      M01r += x0r * d1r + x0i * d1i;
      M01i += x0i * d1r - x0r * d1i;
    }
  v[0] = 2.0 * M01r;
  v[1] = -2.0 * M01i;
  v[2] = M00 - M11;
}

template <typename T, int NO>
__global__ void __launch_bounds__(MOM_THREADS)
k_nc(ClusterView cv, const T* __restrict__ H, int HS, const T* __restrict__ onsite, const double* __restrict__ sdir,
     int n, int n_mom, int nwork, T* __restrict__ scratch, size_t slot_elems, double* __restrict__ mu,
     double* __restrict__ vmom, const double* __restrict__ wts, T* __restrict__ Hbar, int HSh,
     double* __restrict__ obar) {
  constexpr int RW = NO * NCS;
  __shared__ T ws[2][BOP_MAX_NMOM];
  __shared__ int s_lev[BOP_MAX_K + 1];
  __shared__ long long s_off[BOP_MAX_K + 2];
  __shared__ T red[8][MOM_THREADS / 32];
  __shared__ double chi[NCS];
  const bool rev = wts != nullptr;
  const int K = cv.K;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  T* psi = scratch + (size_t)blockIdx.x * slot_elems;
  for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
    const int atom = w / NO, al = w % NO;
    const long long s0 = cv.site_off[atom];
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const int* satom = cv.site_atom + s0;
    const long long* aoff = cv.adj_off + s0;
    if (tid <= K) s_lev[tid] = lev[tid];
    if (tid == 0) {  // Psi_k at s_off[k], Psi-bar_k at s_off[K+1] + (s_off[k] - s_off[1])
      long long o = 0;
      for (int k = 0; k <= K; k++) {
        s_off[k] = o;
        o += (long long)lev[k] * RW;
      }
      s_off[K + 1] = o;
      start_spinors(sdir + 3 * (size_t)atom, chi);
    }
    if (rev)
      for (int q = tid; q < 2 * n_mom; q += blockDim.x) {
        const int nu = q / n_mom, m = q % n_mom;
        ws[nu][m] = (T)wts[(((size_t)nu * n + atom) * NO + al) * n_mom + m];
      }
    __syncthreads();
    T* P = psi;
    T* Pb = psi + s_off[K + 1] - s_off[1];
    for (int q = tid; q < RW; q += blockDim.x) P[q] = (q / NCS == al) ? (T)chi[q % NCS] : T(0);
    if (!rev && tid < 2) {
      mu[(((size_t)tid * n + atom) * NO + al) * n_mom] = 1.0;
      vmom[(((size_t)atom * NO + al) * n_mom) * 3 + tid] = 0.0;
      if (tid == 0) vmom[(((size_t)atom * NO + al) * n_mom) * 3 + 2] = 0.0;
    }
    __syncthreads();
    for (int k = 1; k <= K; k++) {
      const T* x = P + s_off[k - 1];
      T* y = P + s_off[k];
      T d[8];
#pragma unroll
      for (int v = 0; v < 8; v++) d[v] = T(0);
      for (int t = tid; t < s_lev[k]; t += blockDim.x) {
        T acc[NO][NCS];
        gather_row_nc<T, NO>(cv, H, HS, onsite, sdir, n, satom, aoff, t, s_lev[k - 1], x, acc);
#pragma unroll
        for (int r = 0; r < NO; r++)
#pragma unroll
          for (int c = 0; c < NCS; c++) y[((size_t)t * NO + r) * NCS + c] = acc[r][c];
        if (!rev) {
          // <Psi^nu|Psi^nu'>: up-up, dn-dn, and Re / Im of up-dn
#pragma unroll
          for (int r = 0; r < NO; r++) {
            const T* a = acc[r];
            d[4] += a[0] * a[0] + a[1] * a[1] + a[2] * a[2] + a[3] * a[3];
            d[5] += a[4] * a[4] + a[5] * a[5] + a[6] * a[6] + a[7] * a[7];
            d[6] += a[0] * a[4] + a[1] * a[5] + a[2] * a[6] + a[3] * a[7];
            d[7] += a[0] * a[5] - a[1] * a[4] + a[2] * a[7] - a[3] * a[6];
            if (t < s_lev[k - 1]) {
              const T* p = x + ((size_t)t * NO + r) * NCS;
              d[0] += p[0] * a[0] + p[1] * a[1] + p[2] * a[2] + p[3] * a[3];
              d[1] += p[4] * a[4] + p[5] * a[5] + p[6] * a[6] + p[7] * a[7];
              d[2] += p[0] * a[4] + p[1] * a[5] + p[2] * a[6] + p[3] * a[7];
              d[3] += p[0] * a[5] - p[1] * a[4] + p[2] * a[7] - p[3] * a[6];
            }
          }
        }
      }
      if (!rev) {
#pragma unroll
        for (int v = 0; v < 8; v++) {
          const T r_ = warp_sum(d[v]);
          if (lane == 0) red[v][wid] = r_;
        }
        __syncthreads();
        if (tid < 2) {  // moment 2k-1 (tid 0) and 2k (tid 1)
          double L[4];
          for (int v = 0; v < 4; v++) {
            T a = T(0);
            for (int q = 0; q < MOM_THREADS / 32; q++) a += red[4 * tid + v][q];
            L[v] = (double)a;
          }
          const int m = 2 * k - 1 + tid;
          mu[((size_t)atom * NO + al) * n_mom + m] = L[0];
          mu[(((size_t)n + atom) * NO + al) * n_mom + m] = L[1];
          double v3[3];
          pauli_from_local(chi, L[0], L[1], L[2], L[3], v3);
          for (int xx = 0; xx < 3; xx++) vmom[(((size_t)atom * NO + al) * n_mom + m) * 3 + xx] = v3[xx];
        }
      }
      __syncthreads();
    }
    if (rev) {
      // Psi-bar_K = 2 w_2K Psi_K + w_2K-1 Psi_K-1 (weights of each spinor's columns)
      {
        const T* PK = P + s_off[K];
        const T* PK1 = P + s_off[K - 1];
        T* B = Pb + s_off[K];
        for (int q = tid; q < s_lev[K] * RW; q += blockDim.x) {
          const int t = q / RW, nu = (q % NCS) >> 2;
          T v = T(2) * ws[nu][2 * K] * PK[q];
          if (t < s_lev[K - 1]) v += ws[nu][2 * K - 1] * PK1[q];
          B[q] = v;
        }
      }
      __syncthreads();
      for (int k = K; k >= 2; k--) {
        const T* xb = Pb + s_off[k];
        T* yb = Pb + s_off[k - 1];
        const T* Pk = P + s_off[k];
        const T* Pk1 = P + s_off[k - 1];
        const T* Pk2 = P + s_off[k - 2];
        for (int t = tid; t < s_lev[k - 1]; t += blockDim.x) {
          T acc[NO][NCS];
          gather_row_nc<T, NO>(cv, H, HS, onsite, sdir, n, satom, aoff, t, s_lev[k], xb, acc);
#pragma unroll
          for (int r = 0; r < NO; r++)
#pragma unroll
            for (int c = 0; c < NCS; c++) {
              const size_t q = ((size_t)t * NO + r) * NCS + c;
              const int nu = c >> 2;
              T v = acc[r][c] + T(2) * ws[nu][2 * k - 2] * Pk1[q] + ws[nu][2 * k - 1] * Pk[q];
              if (t < s_lev[k - 2]) v += ws[nu][2 * k - 3] * Pk2[q];
              yb[q] = v;
            }
        }
        __syncthreads();
      }
      for (int t = tid; t < s_lev[K]; t += blockDim.x) {
        const int lt = site_level(s_lev, K, t);
        for (long long q = aoff[t]; q < aoff[t + 1]; q++) {
          const int2 en = cv.adj[q];
          const int sidx = en.x;
          if (sidx >= s_lev[K - 1]) break;
          const int ls = site_level(s_lev, K, sidx);
          const int kmin = lt > ls + 1 ? lt : ls + 1;
          T G[NO][NO];
#pragma unroll
          for (int b = 0; b < NO; b++)
#pragma unroll
            for (int g = 0; g < NO; g++) G[b][g] = T(0);
          for (int k = kmin; k <= K; k++) {
            const T* pb = Pb + s_off[k] + (size_t)t * RW;
            const T* ps = P + s_off[k - 1] + (size_t)sidx * RW;
#pragma unroll
            for (int b = 0; b < NO; b++)
#pragma unroll
              for (int g = 0; g < NO; g++) {
                T a = T(0);
#pragma unroll
                for (int c = 0; c < NCS; c++) a += pb[b * NCS + c] * ps[g * NCS + c];
                G[b][g] += a;
              }
          }
          add_bond_cotangent<T, NO>(Hbar + (size_t)en.y * HSh, G);
        }
        if (lt + 1 <= K) {
          // dL/d(Ebar, h) of the onsite matrix of (atom of t, b): the
          // derivatives of Ebar + h.sigma in the real form
          double* op = obar + (size_t)satom[t] * NO * 4;
#pragma unroll
          for (int b = 0; b < NO; b++) {
            T o0 = T(0), ox = T(0), oy = T(0), oz = T(0);
            for (int k = lt + 1; k <= K; k++) {
              const T* pb = Pb + s_off[k] + (size_t)t * RW + b * NCS;
              const T* pt = P + s_off[k - 1] + (size_t)t * RW + b * NCS;
#pragma unroll
              for (int nu = 0; nu < 2; nu++) {
                const T bur = pb[4 * nu], bui = pb[4 * nu + 1], bdr = pb[4 * nu + 2], bdi = pb[4 * nu + 3];
                const T pur = pt[4 * nu], pui = pt[4 * nu + 1], pdr = pt[4 * nu + 2], pdi = pt[4 * nu + 3];
                o0 += bur * pur + bui * pui + bdr * pdr + bdi * pdi;
                ox += bur * pdr + bui * pdi + bdr * pur + bdi * pui;
                oy += bur * pdi - bui * pdr - bdr * pui + bdi * pur;
                oz += bur * pur + bui * pui - bdr * pdr - bdi * pdi;
              }
            }
            atomicAdd(op + 4 * b, (double)o0);
            atomicAdd(op + 4 * b + 1, (double)ox);
            atomicAdd(op + 4 * b + 2, (double)oy);
            atomicAdd(op + 4 * b + 3, (double)oz);
          }
        }
      }
    }
    __syncthreads();
  }
}

// The same over stored Psi, as k_moments and k_adj_rev: work items (atom,
// alpha), the NO items of an atom consecutive in one CTA, which stages the
// atom's cluster once; Psi (Psi-bar) of two levels in shared memory, FP64 rows
// in the order of their length (FP32 ones in site order over 256 threads, for
// sums in a fixed order as in k_moments).  One site row holds NO x 8 reals, so
// that a block feeds 8 NO^2 multiply-adds.
//
// Forward in FP32 the resident warps hide the loads: blocks of two entries in
// flight cost registers (sd blocks spilled at the 128 of two CTAs, s blocks
// kept two CTAs where four fit).  Moments of 2,000 atoms at 9 moments, two
// entries in flight -> one at a time, s with four CTAs: s 0.155 -> 0.116, d
// 1.59 -> 1.47, sd 2.79 -> 2.34 ms.  In FP64, with half the threads, two in
// flight stay ahead for d and sd (432 atoms: 4.63 against 4.82 ms).
template <typename T, int NO>
struct NcFwd {
  static constexpr int THREADS = sizeof(T) == 4 ? 256 : 128;
  static constexpr int CTAS = NO == 1 ? 4 : 2;
};

template <typename T, int NO>
__global__ void __launch_bounds__(NcFwd<T, NO>::THREADS, NcFwd<T, NO>::CTAS)
k_nc_fwd(ClusterView cv, const T* __restrict__ H, int HS, const T* __restrict__ onsite,
         const double* __restrict__ sdir, int n, int n_mom, FwdSmem L, int n_items,
         double* __restrict__ mu, double* __restrict__ vmom, T* __restrict__ pstore,
         const long long* __restrict__ psi_off, long long psi_tot) {
  constexpr int NT = NcFwd<T, NO>::THREADS;
  constexpr bool ORDERED = sizeof(T) == 8;
  constexpr int PS = NO * NCS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf[2];
  buf[0] = reinterpret_cast<T*>(smem_raw);
  buf[1] = buf[0] + (size_t)L.cap_even * PS;
  int2* s_adj = reinterpret_cast<int2*>(align16(reinterpret_cast<unsigned char*>(buf[1] + (size_t)L.cap_odd * PS)));
  unsigned long long* s_lvc = reinterpret_cast<unsigned long long*>(s_adj + (L.stage ? L.max_adj : 0));
  int* s_off = reinterpret_cast<int*>(s_lvc + (L.stage ? L.max_sites : 0));
  int* s_atom = s_off + (L.stage ? L.max_sites + 1 : 0);
  unsigned* s_ord = reinterpret_cast<unsigned*>(s_atom + (L.stage ? L.max_sites : 0));
  __shared__ T red[2][8][NT / 32];
  __shared__ double chi[NCS];
  const int K = cv.K;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int w0, w1;
  item_range(n_items, &w0, &w1);
  int held = -1;  // the atom whose cluster is staged
  for (int w = w0; w < w1; w++) {
    const int atom = w / NO, al = w % NO;
    ItemExt cur;
    ext_sites(cv, atom, cur);
    ext_adj(cv, cur);
    const long long s0 = cur.s0, abase = cur.abase;
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const unsigned long long* lvc = L.stage ? s_lvc : cv.lvcnt + s0;
    const int* satom = L.stage ? s_atom : cv.site_atom + s0;
    const unsigned* order = L.stage ? s_ord : cv.order + s0;
    const int2* adj = L.stage ? s_adj : cv.adj + abase;
    if (atom != held) {
      if (L.stage) {
        if (ORDERED) stage_order(cv, cur, false, s_ord, nullptr, tid, NT);
        stage_item(cv, cur, cur.nsite, (int)(cur.aend - abase), s_adj, s_off, s_lvc, s_atom, tid, NT);
      }
      if (tid == 0) start_spinors(sdir + 3 * (size_t)atom, chi);
      held = atom;
      __syncthreads();
    }
    T* pitem = pstore != nullptr ? pstore + ((size_t)al * psi_tot + psi_off[atom]) * PS : nullptr;
    for (int q = tid; q < PS; q += NT) {
      const T v = (q / NCS == al) ? (T)chi[q % NCS] : T(0);
      buf[0][q] = v;
      if (pitem != nullptr) pitem[q] = v;
    }
    if (tid < 2) {
      mu[(((size_t)tid * n + atom) * NO + al) * n_mom] = 1.0;
      vmom[(((size_t)atom * NO + al) * n_mom) * 3 + tid] = 0.0;
      if (tid == 0) vmom[(((size_t)atom * NO + al) * n_mom) * 3 + 2] = 0.0;
    }
    __syncthreads();
    long long lo_k = 0;
    for (int k = 1; k <= K; k++) {
      lo_k += lev[k - 1];
      const int nrow = lev[k], ncol = lev[k - 1], inner = k >= 2 ? lev[k - 2] : 0;
      const T* prev = buf[(k - 1) & 1];
      T* next = buf[k & 1];
      T d[8];
#pragma unroll
      for (int v = 0; v < 8; v++) d[v] = T(0);
      for (int p = 0; p * NT < nrow; p++) {
        const int r = p * NT + (ORDERED && (p & 1) ? NT - 1 - tid : tid);
        if (r >= nrow) continue;
        const int t = !ORDERED || r < inner ? r : (r < ncol ? (int)(order[r] >> 16) : (int)(order[r] & 0xffffu));
        const bool in_prev = t < ncol;
        T acc[NO][NCS];
        if (in_prev) {
          const int j = satom[t];
          const T sx = (T)sdir[3 * (size_t)j], sy = (T)sdir[3 * (size_t)j + 1], sz = (T)sdir[3 * (size_t)j + 2];
          T pt[PS];
          load_row<T, PS, PS>(prev + (size_t)t * PS, pt);
#pragma unroll
          for (int b = 0; b < NO; b++) {
            const T eu = onsite[(size_t)j * NO + b], ed = onsite[((size_t)n + j) * NO + b];
            const T f = T(0.5) * (ed - eu);
            spin_onsite<T>(T(0.5) * (eu + ed), f * sx, f * sy, f * sz, pt + b * NCS, acc[b]);
          }
        } else {
#pragma unroll
          for (int b = 0; b < NO; b++)
#pragma unroll
            for (int c = 0; c < NCS; c++) acc[b][c] = T(0);
        }
        const int cnt = (int)((lvc[t] >> (8 * (k - 1))) & 0xff);
        const int q0 = L.stage ? s_off[t] : (int)(cv.adj_off[s0 + t] - abase);
        if constexpr (sizeof(T) == 4) gather_plain<T, NO, NCS, PS>(adj + q0, cnt, H, HS, prev, acc);
        else gather_pf2<T, NO, NCS, PS>(adj + q0, cnt, H, HS, prev, acc);
        T pt[PS];
        if (in_prev) {
          load_row<T, PS, PS>(prev + (size_t)t * PS, pt);
        } else {
#pragma unroll
          for (int v = 0; v < PS; v++) pt[v] = T(0);
        }
        // <Psi^nu|Psi^nu'>: up-up, dn-dn, and Re / Im of up-dn
#pragma unroll
        for (int b = 0; b < NO; b++) {
          const T* a = acc[b];
          const T* q = pt + b * NCS;
          d[4] += a[0] * a[0] + a[1] * a[1] + a[2] * a[2] + a[3] * a[3];
          d[5] += a[4] * a[4] + a[5] * a[5] + a[6] * a[6] + a[7] * a[7];
          d[6] += a[0] * a[4] + a[1] * a[5] + a[2] * a[6] + a[3] * a[7];
          d[7] += a[0] * a[5] - a[1] * a[4] + a[2] * a[7] - a[3] * a[6];
          d[0] += q[0] * a[0] + q[1] * a[1] + q[2] * a[2] + q[3] * a[3];
          d[1] += q[4] * a[4] + q[5] * a[5] + q[6] * a[6] + q[7] * a[7];
          d[2] += q[0] * a[4] + q[1] * a[5] + q[2] * a[6] + q[3] * a[7];
          d[3] += q[0] * a[5] - q[1] * a[4] + q[2] * a[7] - q[3] * a[6];
        }
        if (k < K) store_row<T, PS, PS>(next + (size_t)t * PS, &acc[0][0]);
        if (pitem != nullptr) store_row<T, PS, PS>(pitem + (size_t)(lo_k + t) * PS, &acc[0][0]);
      }
#pragma unroll
      for (int v = 0; v < 8; v++) {
        const T r_ = warp_sum(d[v]);
        if (lane == 0) red[k & 1][v][wid] = r_;
      }
      __syncthreads();
      if (tid < 2) {  // moment 2k-1 (tid 0) and 2k (tid 1)
        double Lm[4];
        for (int v = 0; v < 4; v++) {
          T a = T(0);
          for (int q = 0; q < NT / 32; q++) a += red[k & 1][4 * tid + v][q];
          Lm[v] = (double)a;
        }
        const int m = 2 * k - 1 + tid;
        mu[((size_t)atom * NO + al) * n_mom + m] = Lm[0];
        mu[(((size_t)n + atom) * NO + al) * n_mom + m] = Lm[1];
        double v3[3];
        pauli_from_local(chi, Lm[0], Lm[1], Lm[2], Lm[3], v3);
        for (int xx = 0; xx < 3; xx++) vmom[(((size_t)atom * NO + al) * n_mom + m) * 3 + xx] = v3[xx];
      }
    }
    __syncthreads();  // chi and the partials are read before the next item writes them
  }
}

// Reverse sweep over the stored spinor Psi (k_nc_fwd), with the bond
// cotangents and the onsite-matrix cotangents, the latter summed over the
// levels of an item in shared memory.  2,000 atoms, FP32: 10.2 ms with Psi
// recomputed in global scratch (k_nc) -> 2.7 ms.  128 threads: a row's Psi-bar, Psi_k-1,
// sums and blocks take more registers than 168.
template <typename T, int NO>
__global__ void __launch_bounds__(128, 2)
k_nc_rev(ClusterView cv, const T* __restrict__ H, int HS, const T* __restrict__ onsite,
         const double* __restrict__ sdir, int n, int n_mom, RevSmem L, int n_items,
         const T* __restrict__ pstore, const long long* __restrict__ psi_off, long long psi_tot,
         const double* __restrict__ wts, T* __restrict__ Hbar0, int HSh, size_t second, double* __restrict__ obar) {
  constexpr int NT = 128;
  constexpr int PS = NO * NCS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf[2];
  buf[0] = reinterpret_cast<T*>(smem_raw);
  buf[1] = buf[0] + (size_t)L.cap_even * PS;
  T* eb = buf[1] + (size_t)L.cap_odd * PS;  // [cap_eb][NO][4]
  int2* s_adj = reinterpret_cast<int2*>(align16(reinterpret_cast<unsigned char*>(eb + (size_t)L.cap_eb * NO * 4)));
  unsigned long long* s_lvc = reinterpret_cast<unsigned long long*>(s_adj + (L.stage ? L.max_adj : 0));
  int* s_off = reinterpret_cast<int*>(s_lvc + (L.stage ? L.cap_eb : 0));
  int* s_atom = s_off + (L.stage ? L.cap_eb + 1 : 0);
  __shared__ T ws[2][BOP_MAX_NMOM];
  const int K = cv.K;
  const int tid = threadIdx.x, lane = tid & 31;
  int w0, w1;
  item_range(n_items, &w0, &w1);
  int held = -1;
  for (int w = w0; w < w1; w++) {
    const int atom = w / NO, al = w % NO;
    ItemExt cur;
    ext_sites(cv, atom, cur);
    cur.abase = cv.adj_off[cur.s0];
    const long long s0 = cur.s0, abase = cur.abase;
    const int* lev = cv.level_end + (size_t)atom * (K + 1);
    const unsigned long long* lvc = L.stage ? s_lvc : cv.lvcnt + s0;
    const int* satom = L.stage ? s_atom : cv.site_atom + s0;
    const int2* adj = L.stage ? s_adj : cv.adj + abase;
    const int neb = lev[K - 1];
    if (L.stage && atom != held)
      stage_item(cv, cur, neb, (int)(cv.adj_off[s0 + neb] - abase), s_adj, s_off, s_lvc, s_atom, tid, NT);
    held = atom;
    for (int q = tid; q < neb * NO * 4; q += NT) eb[q] = T(0);
    const T* P = pstore + ((size_t)al * psi_tot + psi_off[atom]) * PS;
    T* Hbar = (atom & 1) ? Hbar0 + second : Hbar0;  // NcArgs::second
    for (int q = tid; q < 2 * n_mom; q += NT) {
      const int nu = q / n_mom, m = q % n_mom;
      ws[nu][m] = (T)wts[(((size_t)nu * n + atom) * NO + al) * n_mom + m];
    }
    long long lo = 0;  // first stored row of level k
    for (int k = 0; k < K; k++) lo += lev[k];
    __syncthreads();
    // Psi-bar_K
    for (int t = tid; t < lev[K]; t += NT) {
      T pk[PS];
      load_row<T, PS, PS>(P + (size_t)(lo + t) * PS, pk);
#pragma unroll
      for (int v = 0; v < PS; v++) pk[v] *= T(2) * ws[(v % NCS) >> 2][2 * K];
      if (t < neb) {
        T p1[PS];
        load_row<T, PS, PS>(P + (size_t)(lo - neb + t) * PS, p1);
#pragma unroll
        for (int v = 0; v < PS; v++) pk[v] += ws[(v % NCS) >> 2][2 * K - 1] * p1[v];
      }
      store_row<T, PS, PS>(buf[K & 1] + (size_t)t * PS, pk);
    }
    __syncthreads();
    for (int k = K; k >= 1; k--) {
      const T* xb = buf[k & 1];
      T* yb = buf[(k - 1) & 1];
      const int nrow = lev[k - 1], nrow2 = k >= 2 ? lev[k - 2] : 0;
      const long long lo1 = lo - nrow, lo2 = lo1 - nrow2;  // first rows of levels k-1, k-2
      // lanes per row, as a shift: level 1 only forms bond cotangents; the sums
      // of the others stay in entry order (the torques are small differences of
      // the onsite cotangents: split sums moved them by 1.5e-5)
      const int psh = k == 1 ? 4 : 0;
      const int part = tid & ((1 << psh) - 1);
      for (int r0 = 0; r0 < nrow; r0 += NT >> psh) {
        if (r0 + ((tid & ~31) >> psh) >= nrow) continue;  // whole warps
        const int rr = r0 + (tid >> psh);
        const bool live = rr < nrow;
        const int t = live ? rr : 0;
        T acc[NO][NCS];
#pragma unroll
        for (int b = 0; b < NO; b++)
#pragma unroll
          for (int c = 0; c < NCS; c++) acc[b][c] = T(0);
        const int j = satom[t];
        const T sx = (T)sdir[3 * (size_t)j], sy = (T)sdir[3 * (size_t)j + 1], sz = (T)sdir[3 * (size_t)j + 2];
        T pt[PS];
        if (live) {
          load_row<T, PS, PS>(P + (size_t)(lo1 + t) * PS, pt);
        } else {
#pragma unroll
          for (int v = 0; v < PS; v++) pt[v] = T(0);
        }
        if (live && part == 0) {
          // d/d(Ebar, h) of the onsite matrix of (atom of t, b), and the onsite term
          T xt[PS];
          load_row<T, PS, PS>(xb + (size_t)t * PS, xt);
#pragma unroll
          for (int b = 0; b < NO; b++) {
            T o0 = T(0), ox = T(0), oy = T(0), oz = T(0);
#pragma unroll
            for (int nu = 0; nu < 2; nu++) {
              const T* B = xt + b * NCS + 4 * nu;
              const T* Q = pt + b * NCS + 4 * nu;
              o0 += B[0] * Q[0] + B[1] * Q[1] + B[2] * Q[2] + B[3] * Q[3];
              ox += B[0] * Q[2] + B[1] * Q[3] + B[2] * Q[0] + B[3] * Q[1];
              oy += B[0] * Q[3] - B[1] * Q[2] - B[2] * Q[1] + B[3] * Q[0];
              oz += B[0] * Q[0] + B[1] * Q[1] - B[2] * Q[2] - B[3] * Q[3];
            }
            T* o = eb + ((size_t)t * NO + b) * 4;
            o[0] += o0;
            o[1] += ox;
            o[2] += oy;
            o[3] += oz;
            if (k >= 2) {
              const T eu = onsite[(size_t)j * NO + b], ed = onsite[((size_t)n + j) * NO + b];
              const T f = T(0.5) * (ed - eu);
              spin_onsite<T>(T(0.5) * (eu + ed), f * sx, f * sy, f * sz, xt + b * NCS, acc[b]);
            }
          }
        }
        const int q0 = L.stage ? s_off[t] : (int)(cv.adj_off[s0 + t] - abase);
        int cnt = 0;
        if (live) {
          if (k < K) cnt = (int)((lvc[t] >> (8 * k)) & 0xff);
          else cnt = L.stage ? s_off[t + 1] - q0 : (int)(cv.adj_off[s0 + t + 1] - abase) - q0;
        }
        gather_rev<T, NO, NCS, PS, true>(adj + q0, part, 1 << psh, cnt, 0u, false, H, HS, xb, acc, k >= 2, pt, Hbar,
                                         HSh, lane);
        if (!live || part != 0 || k < 2) continue;
        T* row = &acc[0][0];
#pragma unroll
        for (int v = 0; v < PS; v++) row[v] += T(2) * ws[(v % NCS) >> 2][2 * k - 2] * pt[v];
        T p[PS];
        load_row<T, PS, PS>(P + (size_t)(lo + t) * PS, p);
#pragma unroll
        for (int v = 0; v < PS; v++) row[v] += ws[(v % NCS) >> 2][2 * k - 1] * p[v];
        if (t < nrow2) {
          load_row<T, PS, PS>(P + (size_t)(lo2 + t) * PS, p);
#pragma unroll
          for (int v = 0; v < PS; v++) row[v] += ws[(v % NCS) >> 2][2 * k - 3] * p[v];
        }
        store_row<T, PS, PS>(yb + (size_t)t * PS, row);
      }
      lo = lo1;
      __syncthreads();
    }
    for (int q = tid; q < neb * NO * 4; q += NT) {
      const int t = q / (NO * 4);
      atomicAdd(obar + (size_t)satom[t] * NO * 4 + q % (NO * 4), (double)eb[q]);
    }
    __syncthreads();
  }
}

// Torques of Eq. torque, one thread per atom: dU/ds_i = sum_alpha
// [ (E_dn - E_up)/2 dU/dh_i alpha + sum_n (w_dn - w_up)/2 Tr(sigma M_n) ],
// t_i = dU/ds_i x s_i.
__global__ void k_torques(int n, int norb, int n_mom, const double* __restrict__ onsite,
                          const double* __restrict__ sdir, const double* __restrict__ w,
                          const double* __restrict__ vmom, const double* __restrict__ obar, double* __restrict__ t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double g[3] = {0.0, 0.0, 0.0};
  for (int a = 0; a < norb; a++) {
    const size_t o = (size_t)i * norb + a;
    const double half_delta = 0.5 * (onsite[(size_t)n * norb + o] - onsite[o]);
    for (int x = 0; x < 3; x++) g[x] += half_delta * obar[o * 4 + 1 + x];
    for (int m = 0; m < n_mom; m++) {
      const double c = 0.5 * (w[((size_t)n * norb + o) * n_mom + m] - w[o * n_mom + m]);
      for (int x = 0; x < 3; x++) g[x] += c * vmom[(o * n_mom + m) * 3 + x];
    }
  }
  const double sx = sdir[3 * (size_t)i], sy = sdir[3 * (size_t)i + 1], sz = sdir[3 * (size_t)i + 2];
  t[3 * (size_t)i] = g[1] * sz - g[2] * sy;
  t[3 * (size_t)i + 1] = g[2] * sx - g[0] * sz;
  t[3 * (size_t)i + 2] = g[0] * sy - g[1] * sx;
}

// CTAs of a persistent kernel, at most `most`; 0: not one fits an SM.
template <class F>
int persistent_grid(F fn, int threads, size_t smem, int n_items, int most) {
  int per_sm = 0, sms = 0, dev = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess || per_sm < 1) return 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int slots = sms * per_sm;
  if (slots > most) slots = most;
  return n_items < slots ? n_items : slots;
}

// Spinor sweeps with two levels in shared memory: -2 where they do not fit.
template <typename T, int NO>
int run_nc_fwd(const NcArgs& a, cudaStream_t s) {
  constexpr int NT = NcFwd<T, NO>::THREADS;
  FwdSmem L{a.cap_even, a.cap_odd, a.max_sites, a.max_adj, true};
  const size_t psi = (size_t)(a.cap_even + a.cap_odd) * NO * NCS * sizeof(T);
  size_t smem = psi + (size_t)a.max_adj * 8 + (size_t)a.max_sites * (sizeof(T) == 8 ? 16 : 12) +
                (size_t)(a.max_sites + 1) * 4 + 16;
  if (smem > 110 * 1024) {
    L.stage = false;
    smem = psi;
  }
  if (smem > SMEM_MAX) return -2;
  auto fn = k_nc_fwd<T, NO>;
  if (!allow_smem(fn)) return -1;
  const int n_items = a.n * NO;
  const int grid = persistent_grid(fn, NT, smem, n_items, n_items);
  if (grid < 1) return -1;
  fn<<<grid, NT, smem, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.sdir, a.n, a.n_mom, L, n_items, a.mu,
                            a.vmom, (T*)a.pstore, a.psi_off, a.psi_tot);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <typename T, int NO>
int run_nc_rev(const NcArgs& a, cudaStream_t s) {
  if (a.pstore == nullptr) return -1;
  RevSmem L{a.rev_even, a.rev_odd, a.max_sites, a.rev_adj, a.cap_eb, true};
  const size_t psi = ((size_t)(a.rev_even + a.rev_odd) * NO * NCS + (size_t)a.cap_eb * NO * 4) * sizeof(T) + 16;
  size_t smem = psi + (size_t)a.rev_adj * 8 + (size_t)a.cap_eb * 8 + (size_t)(a.cap_eb + 1) * 4 +
                (size_t)a.max_sites * 4;
  // stage the adjacency where that costs no resident CTA
  if (smem > (psi > 110 * 1024 ? 225 : 110) * 1024) {
    L.stage = false;
    smem = psi;
  }
  if (smem > SMEM_MAX) return -2;
  auto fn = k_nc_rev<T, NO>;
  if (!allow_smem(fn)) return -1;
  const int n_items = a.n * NO;
  const int grid = persistent_grid(fn, 128, smem, n_items, n_items);
  if (grid < 1) return -1;
  fn<<<grid, 128, smem, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.sdir, a.n, a.n_mom, L, n_items,
                             (const T*)a.pstore, a.psi_off, a.psi_tot, a.w, (T*)a.Hbar, a.HSh, a.second,
                             a.obar);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <typename T, int NO>
int run_nc(const NcArgs& a, cudaStream_t s) {
  const int nwork = a.n * NO;
  if (nwork == 0) return 0;
  if (a.scratch == nullptr) return a.w == nullptr ? run_nc_fwd<T, NO>(a, s) : run_nc_rev<T, NO>(a, s);
  const int grid = nwork < a.slots ? nwork : a.slots;
  k_nc<T, NO><<<grid, MOM_THREADS, 0, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.sdir, a.n, a.n_mom,
                                           nwork, (T*)a.scratch, a.slot_elems, a.mu, a.vmom, a.w, (T*)a.Hbar, a.HSh,
                                           a.obar);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace

// Most CTAs of a sweep: with Psi of two levels in global memory each CTA has a
// slot of the scratch, also where Psi_1 .. Psi_K are in the store (Psi_0 is
// written to the slot).
extern "C" int launch_max_ctas(int gmem, size_t scratch_bytes, size_t slot_bytes, int n_items) {
  if (!gmem) return n_items;
  const size_t slots = scratch_bytes / slot_bytes;
  return slots < (size_t)n_items ? (int)slots : n_items;
}

namespace {

template <typename T, int NO, bool GMEM>
int run_forward(const MomentsArgs& a, cudaStream_t s) {
  constexpr int N = NO * NO;
  constexpr int PS = (N == 1) ? 1 : Row<T, N>::PS;
  constexpr bool F64 = sizeof(T) == 8;
  constexpr int NT = F64 ? F64_THREADS : F32_THREADS;
  FwdSmem L{a.cap_even, a.cap_odd, a.max_sites, a.max_adj, true};
  const size_t psi = GMEM ? 0 : (size_t)(a.cap_even + a.cap_odd) * PS * sizeof(T);
  size_t stage = (size_t)a.max_adj * 8 + (size_t)a.max_sites * 8 + (size_t)(a.max_sites + 1) * 4 +
                 (size_t)a.max_sites * (sizeof(T) == 8 ? 12 : 4) + 16;
  size_t smem = psi + stage;
  // stage the adjacency only while two CTAs still fit on an SM
  if (smem > 110 * 1024) {
    L.stage = false;
    smem = psi;
  }
  auto fn = [] {
    if constexpr (F64) return k_moments64<NO, GMEM>;
    else return k_moments<NO, GMEM>;
  }();
  if (!allow_smem(fn)) return -1;
  const int n_items = a.n * a.n_spin;
  const size_t slot = (size_t)(a.cap_even + a.cap_odd) * PS;
  const int most = launch_max_ctas(GMEM, a.scratch_bytes, slot * sizeof(T), n_items);
  if (most < 1) return n_items == 0 ? 0 : -1;
  const int grid = persistent_grid(fn, NT, smem, n_items, most);
  if (grid < 1) return -1;
  if constexpr (F64) {
    fn<<<grid, NT, smem, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.n, a.n_on, a.n_mom, L, n_items, a.mu,
                              (T*)a.pstore, a.psi_off, a.psi_tot, a.pair, a.rowsum, a.nsite, (T*)a.scratch, slot);
    if (a.pair) {
      cudaLaunchAttribute early{};
      early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
      early.val.programmaticStreamSerializationAllowed = 1;
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = n_items;
      cfg.blockDim = PS_THREADS;
      cfg.stream = s;
      cfg.attrs = &early;
      cfg.numAttrs = 1;
      if (cudaLaunchKernelEx(&cfg, k_pair_sums<NO>, a.cv, a.n, a.n_mom, a.mirror, (const double2*)a.rowsum, a.nsite,
                             a.mu) != cudaSuccess)
        return -1;
    }
  } else
    fn<<<grid, NT, smem, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.n, a.n_on, a.n_mom, L, n_items, a.mu,
                              (T*)a.pstore, a.psi_off, a.psi_tot, a.pair, (T*)a.scratch, slot);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <typename T, int NO>
int run_adjoint(const AdjointArgs& a, cudaStream_t s) {
  const int nwork = a.n * a.n_spin;
  const int grid = nwork < a.slots ? nwork : a.slots;
  k_moments_adj<T, NO><<<grid, MOM_THREADS, 0, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.n, a.n_on,
                                                       a.n_mom, nwork, a.w, (T*)a.scratch, a.slot_elems,
                                                       (T*)a.Hbar, a.HSh, a.Ebar);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <typename T, int NO, bool HBAR, bool GMEM>
int run_reverse(const AdjointArgs& a, cudaStream_t s) {
  constexpr int N = NO * NO;
  constexpr int PS = (N == 1) ? 1 : Row<T, N>::PS;
  constexpr bool F64 = sizeof(T) == 8;
  constexpr int NT = F64 ? F64_REV_THREADS : F32_THREADS;
  RevSmem L{a.cap_even, a.cap_odd, a.max_sites, a.max_adj, a.cap_eb, true};
  const size_t slot = (size_t)(a.cap_even + a.cap_odd) * PS;
  const size_t psi = (GMEM ? 0 : slot * sizeof(T)) + eb_elems<T, NO>(a.cap_eb) * sizeof(T);
  const size_t stage = (size_t)a.max_adj * 8 + (size_t)a.cap_eb * 8 + (size_t)(a.cap_eb + 1) * 4 +
                       (size_t)a.max_sites * 4 + 16;
  auto fn = [] {
    if constexpr (F64) return k_adj_rev64<NO, HBAR, GMEM>;
    else return k_adj_rev<NO, HBAR, GMEM>;
  }();
  size_t smem = psi + stage;
  int per_sm = 0, per_sm_unstaged = 0;
  if (psi > SMEM_MAX) return -2;
  if (!allow_smem(fn)) return -1;
  if (smem <= SMEM_MAX) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, NT, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_unstaged, fn, NT, psi);
  if (per_sm < per_sm_unstaged) {  // staging the adjacency would cost a resident CTA
    L.stage = false;
    smem = psi;
  }
  const int n_items = a.n * a.n_spin;
  const int most = launch_max_ctas(GMEM, a.scratch_bytes, slot * sizeof(T), n_items);
  if (most < 1) return n_items == 0 ? 0 : -1;
  const int grid = persistent_grid(fn, NT, smem, n_items, most);
  if (grid < 1) return -1;
  if constexpr (F64)
    fn<<<grid, NT, smem, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.n, a.n_on, a.n_mom, L, n_items,
                              (const T*)a.pstore, a.psi_off, a.psi_tot, a.w, (T*)a.Hbar, a.HSh, a.Ebar, a.siteval,
                              a.sv_stride, a.pair, (T*)a.scratch, slot);
  else
    fn<<<grid, NT, smem, s>>>(a.cv, (const T*)a.H, a.HS, (const T*)a.onsite, a.n, a.n_on, a.n_mom, L, n_items,
                              (const T*)a.pstore, a.psi_off, a.psi_tot, a.w, (T*)a.Hbar, a.HSh, a.Ebar, a.siteval,
                              a.sv_stride, a.pair, (T*)a.scratch, slot);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <typename T, int NO>
int run_reverse_mode(const AdjointArgs& a, cudaStream_t s) {
  if (a.gmem) return a.Hbar ? run_reverse<T, NO, true, true>(a, s) : run_reverse<T, NO, false, true>(a, s);
  return a.Hbar ? run_reverse<T, NO, true, false>(a, s) : run_reverse<T, NO, false, false>(a, s);
}

template <typename T, int NO>
int run_forward_mode(const MomentsArgs& a, cudaStream_t s) {
  return a.gmem ? run_forward<T, NO, true>(a, s) : run_forward<T, NO, false>(a, s);
}

}  // namespace

// Psi rows (Psi-bar rows) of two levels of one work item.
size_t moments_slot_bytes(int norb, int cap_sum, int fp64) {
  const size_t N = (size_t)norb * norb;
  const size_t ps = N == 1 ? 1 : (fp64 ? (N + 1) / 2 * 2 : (N + 3) / 4 * 4);
  return (size_t)cap_sum * ps * (fp64 ? 8 : 4);
}

// Two levels of an item in shared memory (two CTAs per SM) or in global
// scratch.
bool moments_in_gmem(int norb, int cap_sum, int fp64) {
  return moments_slot_bytes(norb, cap_sum, fp64) > 104 * 1024;
}

int launch_moments(const MomentsArgs& a, int fp64, cudaStream_t s) {
  if (a.norb == 1) return fp64 ? run_forward_mode<double, 1>(a, s) : run_forward_mode<float, 1>(a, s);
  if (a.norb == 6) return fp64 ? run_forward_mode<double, 6>(a, s) : run_forward_mode<float, 6>(a, s);
  return fp64 ? run_forward_mode<double, 5>(a, s) : run_forward_mode<float, 5>(a, s);
}

int bond_cotangent_stride(int norb, int fp64) {
  if (norb == 1) return 1;
  if (norb == 5) return fp64 ? hbar_stride<double, 5>() : hbar_stride<float, 5>();
  return fp64 ? hbar_stride<double, 6>() : hbar_stride<float, 6>();
}

int launch_moments_adjoint(const AdjointArgs& a, int fp64, cudaStream_t s) {
  if (a.pstore != nullptr) {  // reverse sweep over stored Psi
    if (a.norb == 1) return fp64 ? run_reverse_mode<double, 1>(a, s) : run_reverse_mode<float, 1>(a, s);
    if (a.norb == 6) return fp64 ? run_reverse_mode<double, 6>(a, s) : run_reverse_mode<float, 6>(a, s);
    return fp64 ? run_reverse_mode<double, 5>(a, s) : run_reverse_mode<float, 5>(a, s);
  }
  if (a.norb == 1) return fp64 ? run_adjoint<double, 1>(a, s) : run_adjoint<float, 1>(a, s);
  if (a.norb == 6) return fp64 ? run_adjoint<double, 6>(a, s) : run_adjoint<float, 6>(a, s);
  return fp64 ? run_adjoint<double, 5>(a, s) : run_adjoint<float, 5>(a, s);
}

bool nc_fwd_in_shared(const NcArgs& a, int fp64) {
  return (size_t)(a.cap_even + a.cap_odd) * a.norb * NCS * (fp64 ? 8 : 4) <= SMEM_MAX;
}

bool nc_rev_in_shared(const NcArgs& a, int fp64) {
  const size_t rows = (size_t)(a.rev_even + a.rev_odd) * a.norb * NCS + (size_t)a.cap_eb * a.norb * 4;
  return rows * (fp64 ? 8 : 4) + 16 <= SMEM_MAX;
}

int launch_nc(const NcArgs& a, int fp64, cudaStream_t s) {
  if (a.norb == 1) return fp64 ? run_nc<double, 1>(a, s) : run_nc<float, 1>(a, s);
  if (a.norb == 6) return fp64 ? run_nc<double, 6>(a, s) : run_nc<float, 6>(a, s);
  return fp64 ? run_nc<double, 5>(a, s) : run_nc<float, 5>(a, s);
}

int launch_torques(int n, int norb, int n_mom, const double* onsite, const double* sdir, const double* w,
                   const double* vmom, const double* obar, double* t, cudaStream_t s) {
  if (n == 0) return 0;
  k_torques<<<(n + 127) / 128, 128, 0, s>>>(n, norb, n_mom, onsite, sdir, w, vmom, obar, t);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
