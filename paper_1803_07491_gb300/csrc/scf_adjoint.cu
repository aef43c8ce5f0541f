// Vector kernels of the SCF-response solve (bop_forces with an SCF): the
// multipliers y of J^T y = dE/du, with u the SCF unknowns (one onsite shift
// per atom, and for Stoner one moment per atom) and J the derivative of the
// SCF conditions at fixed E_F.  Products J^T v come from a reverse sweep of
// the moments (moments.cu) with weights c_{i,nu} dN/dmu; these kernels form
// those weights, project onsite-level cotangents onto u, and carry out the
// Gram-Schmidt and combination steps of GMRES.  Every reduction has a fixed
// order.
#include <cooperative_groups.h>

#include "kernels.h"

namespace {

constexpr int VT = 256;

// c_{i,nu} = s v[i] (+ sigma_nu v[n + i] for Stoner, sigma = +1 up, -1 down)
__global__ void k_scale_weights(int n, int norb, int S, int n_mom, double s, int stoner,
                                const double* __restrict__ v, double sign, const double* __restrict__ wN,
                                const double* __restrict__ wU, double* __restrict__ w) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long tot = (long long)S * n * norb * n_mom;
  if (q >= tot) return;
  const long long o = q / n_mom;                // orbital (spin-major)
  const int atom = (int)((o / norb) % n);
  const int spin = (int)(o / ((long long)norb * n));
  double c = s * v[atom];
  if (stoner) c += (spin == 0 ? 1.0 : -1.0) * v[n + atom];
  w[q] = (wU ? wU[q] : 0.0) + sign * c * wN[q];
}

__global__ void k_project(int n, int norb, int S, double I, const double* __restrict__ Eb,
                          const double* __restrict__ dUE, const double* __restrict__ m, double mcoef,
                          const double* __restrict__ v_m, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double gd = 0.0, gm = 0.0;
  for (int sp = 0; sp < S; sp++) {
    double a = 0.0;
    for (int al = 0; al < norb; al++) {
      const size_t o = ((size_t)sp * n + i) * norb + al;
      a += Eb[o] + (dUE ? dUE[o] : 0.0);
    }
    gd += a;
    gm += (sp == 0 ? -0.5 : 0.5) * I * a;
  }
  out[i] = gd;
  if (S == 2) {
    if (m) gm += mcoef * m[i];
    if (v_m) gm -= v_m[i];
    out[n + i] = gm;
  }
}

__global__ void k_precond_diag(int n, int norb, int S, double s, double floor_, const double* __restrict__ dos,
                               double* __restrict__ P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double d = 0.0;
  for (int sp = 0; sp < S; sp++)
    for (int al = 0; al < norb; al++) d += dos[((size_t)sp * n + i) * norb + al];
  d *= s;
  P[i] = -1.0 / (d > floor_ ? d : floor_);
  if (S == 2) P[n + i] = -1.0;
}

// out[k] = V[k] . w, one block per vector: strided partial sums, a fixed
// shuffle tree and a fixed cross-warp order.
__global__ void __launch_bounds__(VT) k_dots(int nu, const double* __restrict__ V, const double* __restrict__ w,
                                             double* __restrict__ out) {
  __shared__ double sh[VT / 32];
  const int k = blockIdx.x;
  const double* vk = V + (size_t)k * nu;
  double a = 0.0;
  for (int i = threadIdx.x; i < nu; i += VT) a += vk[i] * w[i];
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < VT / 32; q++) t += sh[q];
    out[k] = t;
  }
}

__global__ void k_axpy_multi(int nu, int nvec, const double* __restrict__ V, const double* __restrict__ coef,
                             double* __restrict__ w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nu) return;
  double a = w[i];
  for (int k = 0; k < nvec; k++) a -= coef[k] * V[(size_t)k * nu + i];
  w[i] = a;
}

__global__ void k_lincomb(int nu, int nvec, const double* __restrict__ V, const double* __restrict__ coef,
                          const double* __restrict__ P, double scale, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nu) return;
  double a = 0.0;
  for (int k = 0; k < nvec; k++) a += coef[k] * V[(size_t)k * nu + i];
  out[i] = scale * a * (P ? P[i] : 1.0);
}

__global__ void k_scale_vec(int nu, const double* __restrict__ x, const double* __restrict__ P, double a,
                            double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nu) return;
  out[i] = a * x[i] * (P ? P[i] : 1.0);
}

// Variational SCF: q_i and the E_F multiplier of U_B (see kernels.h).  Block
// partial sums in red[2 b], red[2 b + 1]; the last block adds them in block
// order (deterministic for a given grid).
__global__ void __launch_bounds__(VT) k_var_lambda(int n, int norb, double s, double J, double n0,
                                                   const double* __restrict__ N, const double* __restrict__ dos,
                                                   const double* __restrict__ onsite,
                                                   const FermiState* __restrict__ st, double* __restrict__ q,
                                                   double* __restrict__ lam, double* red, unsigned* counter) {
  __shared__ double sh[2][VT / 32];
  __shared__ bool last;
  const double ef = st->ef;
  double a = 0.0, b = 0.0;
  for (int i = blockIdx.x * VT + threadIdx.x; i < n; i += gridDim.x * VT) {
    double Ni = 0.0, Di = 0.0;
    for (int al = 0; al < norb; al++) {
      Ni += N[(size_t)i * norb + al];
      Di += dos[(size_t)i * norb + al];
    }
    const double qi = s * Ni - n0;
    Di *= s;
    q[i] = qi;
    a += Di * (ef - onsite[(size_t)i * norb] + J * qi);
    b += Di;
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sh[0][threadIdx.x >> 5] = a;
    sh[1][threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double ta = 0.0, tb = 0.0;
    for (int w = 0; w < VT / 32; w++) {
      ta += sh[0][w];
      tb += sh[1][w];
    }
    red[2 * blockIdx.x] = ta;
    red[2 * blockIdx.x + 1] = tb;
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x != 0) return;
  double ta = 0.0, tb = 0.0;
  for (int k = 0; k < (int)gridDim.x; k++) {
    ta += __ldcg(red + 2 * k);
    tb += __ldcg(red + 2 * k + 1);
  }
  lam[0] = tb > 0.0 ? ta / tb : 0.0;
  *counter = 0;
}

// u /= sqrt(*nsq) when *nsq > 0 (the norm stays on the device)
__global__ void k_scale_by_inv_norm(int nu, double* __restrict__ u, const double* __restrict__ nsq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const double q = *nsq;
  if (i >= nu || !(q > 0.0)) return;
  u[i] = u[i] * (1.0 / sqrt(q));
}

// Transpose of the Jacobian rows: for every atom j the entries (i, site)
// with site_atom[site] = j among the first |C_K-1| sites of i's cluster.
// Count, then fill (rows in arbitrary order within an atom).
__global__ void k_jt_count(int n, int K, const long long* __restrict__ site_off, const int* __restrict__ level_end,
                           const int* __restrict__ site_atom, int* __restrict__ cnt) {
  const int i = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  const long long s0 = site_off[i];
  const int neb = level_end[(size_t)i * (K + 1) + K - 1];
  for (int t = lane; t < neb; t += 32) atomicAdd(cnt + site_atom[s0 + t], 1);
}

__global__ void k_jt_fill(int n, int K, const long long* __restrict__ site_off, const int* __restrict__ level_end,
                          const int* __restrict__ site_atom, const long long* __restrict__ ptr,
                          int* __restrict__ fill, long long* __restrict__ idx, int* __restrict__ row) {
  const int i = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  const long long s0 = site_off[i];
  const int neb = level_end[(size_t)i * (K + 1) + K - 1];
  for (int t = lane; t < neb; t += 32) {
    const int j = site_atom[s0 + t];
    const long long q = ptr[j] + atomicAdd(fill + j, 1);
    idx[q] = s0 + t;
    row[q] = i;
  }
}

// One warp per (spin, atom j): Eb[spin][j] = sum over j's entries of
// c_{i,spin} val[spin][site], c = s v[i] (+ sigma_spin v[n + i] for Stoner).
__global__ void k_jt_gather(int n, int S, const long long* __restrict__ ptr, const long long* __restrict__ idx,
                            const int* __restrict__ row, const double* __restrict__ val, long long stride,
                            const double* __restrict__ v, double s, int stoner, double* __restrict__ Eb) {
  const int wg = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (wg >= S * n) return;
  const int spin = wg / n, j = wg % n;
  const double sg = spin == 0 ? 1.0 : -1.0;
  const double* vs = val + (size_t)spin * stride;
  double a = 0.0;
  for (long long q = ptr[j] + lane; q < ptr[j + 1]; q += 32) {
    const int i = row[q];
    double c = s * v[i];
    if (stoner) c += sg * v[n + i];
    a += c * vs[idx[q]];
  }
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) Eb[(size_t)spin * n + j] = a;
}

// The whole response solve over the stored rows of J in one cooperative
// launch: restarted GMRES, right-preconditioned with the diagonal P, classical
// Gram-Schmidt twice.  As separate kernels a step was 9 launches of 3 to 8 us
// and a read-back of its Hessenberg column for a few us of work.
//
// Bound: the latency of the three grid synchronisations of a step and of the
// loads between them.  Every block owns a contiguous slice of the atoms: it
// gathers u = J^T x for its slice (one warp per atom, both spins), keeps its
// slice of every basis vector to itself, and adds partial dot products of
// the slice to a table [block][vector] that each block sums for itself in
// block order after the synchronisation.  The newest vector is the only one
// that other blocks read: its owner writes P u before the norm is known, and
// the gather multiplies its sums by 1 / |u|.  The Givens rotations and the
// stopping rule run in every block on the same numbers.  Measured per step at
// 2,000 atoms: 52 us of kernels and a read-back of about 15 us -> 27 us.
constexpr int GT = 512;

// sum over the blocks of part[b][k], by one warp; the same in all lanes
__device__ __forceinline__ double block_sums(const double* part, int nb, int ld, int k, int lane) {
  double a = 0.0;
  for (int b = lane; b < nb; b += 32) a += __ldcg(part + (size_t)b * ld + k);
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

__global__ void __launch_bounds__(GT, 1) k_gmres(GmresArgs g) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  constexpr int LD = GM_KRYLOV + 1;
  __shared__ double Hh[GM_KRYLOV + 1][GM_KRYLOV], cs[GM_KRYLOV], sn[GM_KRYLOV], gv[GM_KRYLOV + 1];
  __shared__ double h1[GM_KRYLOV + 1], h2[GM_KRYLOV + 1], red[GT / 32], ctl[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = gridDim.x;
  const int n = g.n, nu = g.nu, comp = nu / n;
  const int a0 = (int)((long long)n * blockIdx.x / nb), na = (int)((long long)n * (blockIdx.x + 1) / nb) - a0;
  const int own = na * comp;  // owned elements: e -> (e / na) n + a0 + e % na
  auto at = [&](int e) { return e < na ? a0 + e : n + a0 + e - na; };
  double* part1 = g.part + (size_t)blockIdx.x * LD;
  double* part2 = g.part + (size_t)(nb + blockIdx.x) * LD;
  double* partn = g.part + (size_t)2 * nb * LD;

  // out (own slice) = scale J^T x for x complete in memory
  auto product = [&](const double* x, double scale, double* out) {
    for (int q = warp; q < na; q += GT / 32) {
      const int j = a0 + q;
      const long long p0 = g.ptr[j], p1 = g.ptr[j + 1];
      double a = 0.0, b = 0.0;
#pragma unroll 4
      for (long long p = p0 + lane; p < p1; p += 32) {
        const int i = g.row[p];
        const long long t = g.idx[p];
        const double c = g.s * __ldcg(x + i);
        if (comp == 1) {
          a += c * g.val[t];
        } else {
          const double m = __ldcg(x + n + i);
          a += (c + m) * g.val[t];
          b += (c - m) * g.val[g.stride + t];
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        if (comp == 2) b += __shfl_xor_sync(0xffffffffu, b, o);
      }
      if (lane == 0) {
        out[j] = scale * (a + b);
        if (comp == 2) out[n + j] = scale * (0.5 * g.I * (b - a) - __ldcg(x + n + j));
      }
    }
    __syncthreads();
  };
  // table[block][k] = own part of V_k . w for k < nvec
  auto dots = [&](int nvec, const double* w, double* table) {
    for (int k = warp; k < nvec; k += GT / 32) {
      const double* v = g.V + (size_t)k * nu;
      double a = 0.0;
      for (int e = lane; e < own; e += 32) a += v[at(e)] * w[at(e)];
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) table[k] = a;
    }
  };
  // w -= sum_k h_k V_k on the own slice, h summed from the blocks' table
  auto subtract = [&](int nvec, const double* table, double* h, double* w) {
    for (int k = warp; k < nvec; k += GT / 32) {
      const double a = block_sums(table, nb, LD, k, lane);
      if (lane == 0) h[k] = a;
    }
    __syncthreads();
    for (int e = tid; e < own; e += GT) {
      double a = w[at(e)];
#pragma unroll 4
      for (int k = 0; k < nvec; k++) a -= h[k] * g.V[(size_t)k * nu + at(e)];
      w[at(e)] = a;
    }
    __syncthreads();
  };
  // partn[block] = own part of w . w; px (if not NULL) = P w
  auto norm_part = [&](const double* w, double* px) {
    double a = 0.0;
    for (int e = tid; e < own; e += GT) {
      const double v = w[at(e)];
      a += v * v;
      if (px) px[at(e)] = v * g.P[at(e)];
    }
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int q = 0; q < GT / 32; q++) t += red[q];
      partn[blockIdx.x] = t;
    }
  };
  auto norm2 = [&]() {  // after the grid synchronisation; the same in all threads
    if (warp == 0) {
      const double a = block_sums(partn, nb, 1, 0, lane);
      if (lane == 0) ctl[0] = a;
    }
    __syncthreads();
    return ctl[0];
  };

  for (int e = tid; e < own; e += GT) g.y[at(e)] = 0.0;
  // r = rhs in the first cycle
  for (int e = tid; e < own; e += GT) g.V[at(e)] = g.rhs[at(e)];
  __syncthreads();
  norm_part(g.V, g.x);
  grid.sync();
  const double bnorm = sqrt(norm2());
  double beta = bnorm, rel = 0.0;
  int iters = 0;
  bool conv = bnorm == 0.0;
  for (int cyc = 0; cyc < GM_CYCLES && !conv && iters < g.max_it; cyc++) {
    if (cyc > 0) {  // r = rhs - J^T y into V_0
      for (int e = tid; e < own; e += GT) g.xy[at(e)] = g.y[at(e)];
      grid.sync();
      product(g.xy, 1.0, g.V);
      for (int e = tid; e < own; e += GT) g.V[at(e)] = g.rhs[at(e)] - g.V[at(e)];
      __syncthreads();
      norm_part(g.V, g.x);
      grid.sync();
      beta = sqrt(norm2());
    }
    if (beta <= g.rtol * bnorm) {
      conv = true;
      rel = beta / bnorm;
      break;
    }
    double inv = 1.0 / beta;
    for (int e = tid; e < own; e += GT) g.V[at(e)] *= inv;
    for (int q = tid; q <= GM_KRYLOV; q += GT) gv[q] = q == 0 ? beta : 0.0;
    __syncthreads();
    int k = 0;
    for (int j = 0; j < GM_KRYLOV; j++) {
      double* u = g.V + (size_t)(j + 1) * nu;
      product(g.x, inv, u);
      dots(j + 1, u, part1);
      grid.sync();
      subtract(j + 1, g.part, h1, u);
      dots(j + 1, u, part2);
      grid.sync();
      subtract(j + 1, g.part + (size_t)nb * LD, h2, u);
      norm_part(u, g.x);
      grid.sync();
      const double hn = sqrt(norm2());
      inv = 1.0 / hn;
      if (hn > 0.0)
        for (int e = tid; e < own; e += GT) u[at(e)] *= inv;
      if (tid == 0) {  // Givens rotations on the new Hessenberg column
        double t = h1[0] + h2[0];
        for (int q = 0; q < j; q++) {
          const double b = h1[q + 1] + h2[q + 1];
          Hh[q][j] = cs[q] * t + sn[q] * b;
          t = -sn[q] * t + cs[q] * b;
        }
        const double rr = hypot(t, hn);
        const double c = rr > 0.0 ? t / rr : 1.0, z = rr > 0.0 ? hn / rr : 0.0;
        cs[j] = c;
        sn[j] = z;
        Hh[j][j] = rr;
        gv[j + 1] = -z * gv[j];
        gv[j] = c * gv[j];
        ctl[1] = fabs(gv[j + 1]) / bnorm;
      }
      __syncthreads();
      k = j + 1;
      iters++;
      rel = ctl[1];
      if (rel <= g.rtol || hn == 0.0 || iters >= g.max_it) break;
    }
    // z = H^-1 gv (upper triangular) in gv, y += P sum z_q V_q
    if (warp == 0) {
      for (int q = k - 1; q >= 0; q--) {
        const double z = gv[q] / Hh[q][q];
        for (int r = lane; r < q; r += 32) gv[r] -= Hh[r][q] * z;
        __syncwarp();
        if (lane == 0) gv[q] = z;
        __syncwarp();
      }
    }
    __syncthreads();
    for (int e = tid; e < own; e += GT) {
      double a = 0.0;
      for (int q = 0; q < k; q++) a += gv[q] * g.V[(size_t)q * nu + at(e)];
      g.y[at(e)] += a * g.P[at(e)];
    }
    __syncthreads();
    conv = rel <= g.rtol;
  }
  if (blockIdx.x == 0 && tid == 0) {
    g.out[0] = iters;
    g.out[1] = rel;
    g.out[2] = conv ? 1.0 : 0.0;
  }
}

unsigned grid(long long n) { return (unsigned)((n + VT - 1) / VT); }
int ok() { return cudaGetLastError() == cudaSuccess ? 0 : -1; }

}  // namespace

int launch_scale_weights(int n, int norb, int S, int n_mom, double s, int stoner, const double* v, double sign,
                         const double* wN, const double* wU, double* w_out, cudaStream_t st) {
  const long long tot = (long long)S * n * norb * n_mom;
  k_scale_weights<<<grid(tot), VT, 0, st>>>(n, norb, S, n_mom, s, stoner, v, sign, wN, wU, w_out);
  return ok();
}

int launch_project(int n, int norb, int S, double I, const double* Eb, const double* dUE, const double* m,
                   double mcoef, const double* v_m, double* out, cudaStream_t st) {
  k_project<<<grid(n), VT, 0, st>>>(n, norb, S, I, Eb, dUE, m, mcoef, v_m, out);
  return ok();
}

int launch_precond_diag(int n, int norb, int S, double s, double floor_, const double* dos, double* P,
                        cudaStream_t st) {
  k_precond_diag<<<grid(n), VT, 0, st>>>(n, norb, S, s, floor_, dos, P);
  return ok();
}

int launch_dots(int nu, int nvec, const double* V, const double* w, double* out, cudaStream_t st) {
  if (nvec <= 0) return 0;
  k_dots<<<nvec, VT, 0, st>>>(nu, V, w, out);
  return ok();
}

int launch_axpy_multi(int nu, int nvec, const double* V, const double* coef, double* w, cudaStream_t st) {
  if (nvec <= 0) return 0;
  k_axpy_multi<<<grid(nu), VT, 0, st>>>(nu, nvec, V, coef, w);
  return ok();
}

int launch_lincomb(int nu, int nvec, const double* V, const double* coef, const double* P, double scale,
                   double* out, cudaStream_t st) {
  k_lincomb<<<grid(nu), VT, 0, st>>>(nu, nvec, V, coef, P, scale, out);
  return ok();
}

int launch_scale_vec(int nu, const double* x, const double* P, double a, double* out, cudaStream_t st) {
  k_scale_vec<<<grid(nu), VT, 0, st>>>(nu, x, P, a, out);
  return ok();
}

int launch_var_lambda(int n, int norb, double s, double J, double n0, const double* N, const double* dos,
                      const double* onsite, const FermiState* st, double* q, double* lam, double* red,
                      unsigned* counter, cudaStream_t stream) {
  unsigned g = grid(n);
  if (g < 1) g = 1;
  if (g > 1024) g = 1024;
  k_var_lambda<<<g, VT, 0, stream>>>(n, norb, s, J, n0, N, dos, onsite, st, q, lam, red, counter);
  return ok();
}

int launch_scale_by_inv_norm(int nu, double* u, const double* nsq, cudaStream_t stream) {
  k_scale_by_inv_norm<<<grid(nu), VT, 0, stream>>>(nu, u, nsq);
  return ok();
}

int launch_jt_build(int n, int K, const long long* site_off, const int* level_end, const int* site_atom,
                    int* cnt, int stage, const long long* ptr, long long* idx, int* row, cudaStream_t stream) {
  const long long threads = (long long)n * 32;
  if (stage == 0) k_jt_count<<<grid(threads), VT, 0, stream>>>(n, K, site_off, level_end, site_atom, cnt);
  else k_jt_fill<<<grid(threads), VT, 0, stream>>>(n, K, site_off, level_end, site_atom, ptr, cnt, idx, row);
  return ok();
}

int launch_jt_gather(int n, int S, const long long* ptr, const long long* idx, const int* row, const double* val,
                     long long stride, const double* v, double s, int stoner, double* Eb, cudaStream_t stream) {
  const long long threads = (long long)S * n * 32;
  k_jt_gather<<<grid(threads), VT, 0, stream>>>(n, S, ptr, idx, row, val, stride, v, s, stoner, Eb);
  return ok();
}

int launch_gmres(const GmresArgs& g, cudaStream_t stream) {
  int dev = 0, sms = 0, coop = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (!coop || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gmres, GT, 0) != cudaSuccess || per_sm < 1)
    return -2;
  // 8 atoms per block until every SM has a block: fewer blocks leave warps of
  // the gather unused, more lengthen the sums over the blocks
  int nb = (g.n + 7) / 8;
  if (nb > sms) nb = sms;
  if (nb > GMRES_BLOCKS) nb = GMRES_BLOCKS;
  GmresArgs a = g;
  void* args[] = {&a};
  const cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_gmres), nb, GT, args, 0, stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorCooperativeLaunchTooLarge ? -2 : -1;
  }
  return 0;
}
