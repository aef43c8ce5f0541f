// Hop levels of (atom, image) sites around every atom: the support of the
// self-returning paths of Eq. momDOS (C_0 = {i}, C_k = C_{k-1} plus all
// neighbours of C_{k-1}, inside the path radius when one is set:
// "Performance", item (iii)), with the adjacency between cluster sites that
// the moments kernels walk.
//
// Canonical order (reproducible bit for bit): level, then atom, then image
// (sx, sy, sz).  Each site's adjacency lists every neighbour inside the
// cluster as {local index, bond}, ascending local index.
//
// Two builders with the same results: the general one, one CTA per atom
// (grid-stride), a hash table of site keys in per-CTA global scratch, the new
// sites of a level sorted in shared memory; and the grid builder below it.
#include "kernels.h"

namespace {

constexpr unsigned long long EMPTY = ~0ull;
constexpr int CL_THREADS = 256;

__device__ __forceinline__ unsigned long long site_key(int atom, int sx, int sy, int sz) {
  return ((unsigned long long)(unsigned)atom << 24) | ((unsigned long long)(sx + 128) << 16) |
         ((unsigned long long)(sy + 128) << 8) | (unsigned long long)(sz + 128);
}
__device__ __forceinline__ int key_atom(unsigned long long k) { return (int)(k >> 24); }
__device__ __forceinline__ int key_img(unsigned long long k, int c) {
  return (int)((k >> (16 - 8 * c)) & 0xff) - 128;
}
__device__ __forceinline__ unsigned hash_slot(unsigned long long k, int mask) {
  unsigned long long x = k * 0x9E3779B97F4A7C15ull;
  return (unsigned)(x >> 32) & (unsigned)mask;
}

// Find key; returns slot or -1.  Bounded by the table size.
__device__ int h_find(const unsigned long long* __restrict__ hk, int hcap, unsigned long long key) {
  unsigned s = hash_slot(key, hcap - 1);
  for (int probe = 0; probe < hcap; probe++) {
    unsigned long long c = hk[s];
    if (c == key) return (int)s;
    if (c == EMPTY) return -1;
    s = (s + 1) & (hcap - 1);
  }
  return -1;
}

// Insert key if absent.  Returns 1 if this call inserted it, 0 if present,
// -1 if the table is full.
__device__ int h_insert(unsigned long long* hk, int hcap, unsigned long long key) {
  unsigned s = hash_slot(key, hcap - 1);
  for (int probe = 0; probe < hcap; probe++) {
    unsigned long long c = hk[s];
    if (c == key) return 0;
    if (c == EMPTY) {
      unsigned long long prev = atomicCAS(&hk[s], EMPTY, key);
      if (prev == EMPTY) return 1;
      if (prev == key) return 0;
    }
    s = (s + 1) & (hcap - 1);
  }
  return -1;
}

__device__ void block_sort_u64(unsigned long long* a, int cnt) {
  int P = 1;
  while (P < cnt) P <<= 1;
  for (int i = cnt + threadIdx.x; i < P; i += blockDim.x) a[i] = EMPTY;
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        int ixj = i ^ j;
        if (ixj > i) {
          bool up = (i & k) == 0;
          unsigned long long x = a[i], y = a[ixj];
          if ((x > y) == up) {
            a[i] = y;
            a[ixj] = x;
          }
        }
      }
      __syncthreads();
    }
}

// Exclusive scan of v[0..cnt) in place (chunks of blockDim), returns total.
__device__ int block_exclusive_scan(int* v, int cnt, int* warp_tmp) {
  int carry = 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int base = 0; base < cnt; base += blockDim.x) {
    int i = base + threadIdx.x;
    int x = i < cnt ? v[i] : 0;
    int incl = x;
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tmp[wid] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
      int acc = 0;
      for (int q = 0; q < nw; q++) {
        int t = warp_tmp[q];
        warp_tmp[q] = acc;
        acc += t;
      }
      warp_tmp[nw] = acc;
    }
    __syncthreads();
    if (i < cnt) v[i] = carry + warp_tmp[wid] + incl - x;
    carry += warp_tmp[nw];
    __syncthreads();
  }
  return carry;
}

template <int PASS, bool CUT>
__global__ void __launch_bounds__(CL_THREADS)
k_cluster(int n, int K, const long long* __restrict__ row_ptr, const int* __restrict__ col,
          const signed char* __restrict__ img, const int* __restrict__ bond_of_edge, PathCut pc, ClusterScratch sc,
          ClusterOut out, unsigned* __restrict__ status) {
  extern __shared__ unsigned long long newkeys[];  // [newcap], a power of two
  __shared__ int s_count, s_fail;
  __shared__ int s_lev[BOP_MAX_K + 1];
  __shared__ int warp_tmp[CL_THREADS / 32 + 1];
  unsigned long long* hk = sc.hkeys + (size_t)blockIdx.x * sc.hcap;
  int* hv = sc.hvals + (size_t)blockIdx.x * sc.hcap;
  unsigned long long* sk = sc.skeys + (size_t)blockIdx.x * sc.maxs;
  int* ss = sc.sslot + (size_t)blockIdx.x * sc.maxs;
  int* scnt = sc.scount + (size_t)blockIdx.x * sc.maxs;

  for (int atom = blockIdx.x; atom < n; atom += gridDim.x) {
    if (threadIdx.x == 0) {
      unsigned long long k0 = site_key(atom, 0, 0, 0);
      h_insert(hk, sc.hcap, k0);
      int sl = h_find(hk, sc.hcap, k0);
      s_fail = 0;
      if (sl < 0) {
        s_fail = 1;
        raise_error(status, BOP_DEV_ERR_CLUSTER);
        sl = 0;
      }
      hv[sl] = 0;
      sk[0] = k0;
      ss[0] = sl;
      s_lev[0] = 1;
    }
    __syncthreads();
    int nsite = 1;
    for (int k = 1; k <= K; k++) {
      if (threadIdx.x == 0) s_count = 0;
      __syncthreads();
      int f0 = k >= 2 ? s_lev[k - 2] : 0, f1 = s_lev[k - 1];
      for (int t = f0 + threadIdx.x; t < f1; t += blockDim.x) {
        unsigned long long kt = sk[t];
        int a = key_atom(kt);
        int ix = key_img(kt, 0), iy = key_img(kt, 1), iz = key_img(kt, 2);
        for (long long e = row_ptr[a]; e < row_ptr[a + 1]; e++) {
          int sx = ix + img[3 * e], sy = iy + img[3 * e + 1], sz = iz + img[3 * e + 2];
          if (sx < -127 || sx > 127 || sy < -127 || sy > 127 || sz < -127 || sz > 127) {
            s_fail = 1;
            raise_error(status, BOP_DEV_ERR_IMAGE);
            continue;
          }
          if (CUT) {  // path-radius cut: only sites closer than r_path to the atom
            double d[3];
            bond_vector(pc.pos + 3 * (size_t)atom, pc.pos + 3 * (size_t)col[e], pc.cell, sx, sy, sz, d);
            if (!(norm2_rn(d) < pc.r2)) continue;
          }
          unsigned long long key = site_key(col[e], sx, sy, sz);
          int r = h_insert(hk, sc.hcap, key);
          if (r == 1) {
            int q = atomicAdd(&s_count, 1);
            if (q < sc.newcap) newkeys[q] = key;
          } else if (r < 0) {
            s_fail = 1;
            raise_error(status, BOP_DEV_ERR_CLUSTER);
          }
        }
      }
      __syncthreads();
      int cnt = s_count;
      if (cnt > sc.newcap || nsite + cnt > sc.maxs) {
        if (threadIdx.x == 0) {
          s_fail = 1;
          raise_error(status, BOP_DEV_ERR_CLUSTER);
        }
        __syncthreads();
        cnt = 0;
      }
      if (s_fail) break;
      block_sort_u64(newkeys, cnt);
      for (int q = threadIdx.x; q < cnt; q += blockDim.x) {
        unsigned long long key = newkeys[q];
        int sl = h_find(hk, sc.hcap, key);
        if (sl < 0) {  // cannot happen for a key this level inserted; never index with it
          raise_error(status, BOP_DEV_ERR_CLUSTER);
          sl = 0;
        }
        hv[sl] = nsite + q;
        sk[nsite + q] = key;
        ss[nsite + q] = sl;
      }
      nsite += cnt;
      if (threadIdx.x == 0) s_lev[k] = nsite;
      __syncthreads();
    }
    __syncthreads();
    const bool ok = !s_fail;
    if (ok) {
      // adjacency: every neighbour inside the cluster (counts first)
      for (int t = threadIdx.x; t < nsite; t += blockDim.x) {
        unsigned long long kt = sk[t];
        int a = key_atom(kt);
        int ix = key_img(kt, 0), iy = key_img(kt, 1), iz = key_img(kt, 2);
        int c = 0;
        for (long long e = row_ptr[a]; e < row_ptr[a + 1]; e++) {
          int sx = ix + img[3 * e], sy = iy + img[3 * e + 1], sz = iz + img[3 * e + 2];
          if (sx < -127 || sx > 127 || sy < -127 || sy > 127 || sz < -127 || sz > 127) continue;
          if (h_find(hk, sc.hcap, site_key(col[e], sx, sy, sz)) >= 0) c++;
        }
        scnt[t] = c < BOP_MAX_DEG ? c : BOP_MAX_DEG;
      }
      __syncthreads();
      if (PASS == 0) {
        int tot = block_exclusive_scan(scnt, nsite, warp_tmp);
        if (threadIdx.x == 0) {
          out.atom_nsite[atom] = nsite;
          out.atom_nadj[atom] = tot;
          atomicMax(&out.max_level[K + 1], tot);  // largest adjacency
        }
        for (int k = threadIdx.x; k <= K; k += blockDim.x) {
          out.level_end[(size_t)atom * (K + 1) + k] = s_lev[k];
          atomicMax(&out.max_level[k], s_lev[k]);
        }
      } else {
        block_exclusive_scan(scnt, nsite, warp_tmp);
        long long s0 = out.site_off[atom], a0 = out.adj_base[atom];
        unsigned long long prod = 0;
        for (int t = threadIdx.x; t < nsite; t += blockDim.x) {
          unsigned long long kt = sk[t];
          out.site_atom[s0 + t] = key_atom(kt);
          out.site_img[3 * (s0 + t)] = (signed char)key_img(kt, 0);
          out.site_img[3 * (s0 + t) + 1] = (signed char)key_img(kt, 1);
          out.site_img[3 * (s0 + t) + 2] = (signed char)key_img(kt, 2);
          out.adj_off[s0 + t] = a0 + scnt[t];
          // recompute and write the sorted entries
          int a = key_atom(kt);
          int ix = key_img(kt, 0), iy = key_img(kt, 1), iz = key_img(kt, 2);
          int2 ent[BOP_MAX_DEG];
          int c = 0;
          for (long long e = row_ptr[a]; e < row_ptr[a + 1]; e++) {
            int sx = ix + img[3 * e], sy = iy + img[3 * e + 1], sz = iz + img[3 * e + 2];
            if (sx < -127 || sx > 127 || sy < -127 || sy > 127 || sz < -127 || sz > 127) continue;
            int sl = h_find(hk, sc.hcap, site_key(col[e], sx, sy, sz));
            if (sl < 0) continue;
            if (c < BOP_MAX_DEG) ent[c] = make_int2(hv[sl], bond_of_edge[e]);
            c++;
          }
          if (c > BOP_MAX_DEG) c = BOP_MAX_DEG;
          for (int x = 1; x < c; x++) {
            int2 v = ent[x];
            int y = x - 1;
            while (y >= 0 && ent[y].x > v.x) {
              ent[y + 1] = ent[y];
              y--;
            }
            ent[y + 1] = v;
          }
          long long o = a0 + scnt[t];
          for (int x = 0; x < c; x++) out.adj[o + x] = ent[x];
          // byte k: entries whose site lies in C_k (the gather of level k+1)
          unsigned long long lc = 0;
          for (int k = 0; k < K; k++) {
            unsigned cnt = 0;
            while ((int)cnt < c && ent[cnt].x < s_lev[k]) cnt++;
            lc |= (unsigned long long)cnt << (8 * k);
          }
          out.lvcnt[s0 + t] = lc;
          if (out.order != nullptr) out.order[s0 + t] = (unsigned)t | ((unsigned)t << 16);
          // forward levels k = max(lt, ls+1) .. K use the pair (t, s)
          int lt = 0;
          while (lt < K && t >= s_lev[lt]) lt++;
          for (int x = 0; x < c; x++) {
            int ls = 0;
            while (ls < K && ent[x].x >= s_lev[ls]) ls++;
            int k0 = lt > ls + 1 ? lt : ls + 1;
            if (k0 <= K) prod += (unsigned long long)(K - k0 + 1);
          }
        }
        if (prod) atomicAdd(out.n_products, prod);
      }
    } else if (PASS == 0 && threadIdx.x == 0) {
      out.atom_nsite[atom] = 0;
      out.atom_nadj[atom] = 0;
    }
    __syncthreads();
    // clear the hash table: every inserted key became a site (or the atom failed)
    for (int t = threadIdx.x; t < nsite; t += blockDim.x) {
      hk[ss[t]] = EMPTY;
    }
    if (!ok) {  // a failed atom may have left keys that never became sites
      for (int q = threadIdx.x; q < sc.hcap; q += blockDim.x) hk[q] = EMPTY;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- grid builder
// The same clusters (same canonical order, same adjacency and level counts)
// through a table in shared memory instead of a hash table.  Every site has
// an address: its linked cell relative to the cluster's atom, unwrapped over
// the periodic images, times the slots of a cell, plus its atom's slot in
// that cell.  The address of a neighbour is the site's address plus an offset
// that depends on the directed edge alone (k_pack_edges), so that looking a
// site up is one shared-memory load, with no key, hash or probe.
//
// Table size: sites lie within R_K cells of the atom along each axis,
// neighbours that are looked up within R_{K+1} (grid_plan).  A period of
// R_K + R_{K+1} + 1 cells keeps the address of every looked-up cell apart
// from that of every other cell a site can lie in, and only the addresses of
// sites need storage.
//
// Order without sorting the adjacency: a neighbour row is sorted by (atom,
// image), as the sites of one level are, and the neighbours of a site of
// level l lie in levels l-1, l, l+1.  An entry's place in its row is its rank
// among the entries of its own level (a ballot) after the entries of the
// levels below.  Rows take 16 or 32 lanes, one per edge, so that the loads of
// a row and its writes are contiguous.
//
// G threads per atom.  Pass 0 runs the breadth-first search (new sites are
// claimed in the table with an atomicOr, sorted per level), counts the
// adjacency and keeps the site records; pass 1 fills the table from them and
// writes sites, adjacency and level counts.
//
// What bounds it: issue slots (57 and 63 % used in the two passes), after the
// table's 14 to 76 KB per cluster has limited the CTAs on an SM, hence several
// warps per cluster.  The hash-table builder it replaces (one warp per atom,
// 64-bit keys) took 27.9 k and 34.4 k warp instructions per atom in the two
// passes, this one 16.5 k and 24.5 k (2,000 bcc atoms at 9 moments, with the
// pair form's outputs): 131,072 atoms at 9 moments 19.8 -> 6.7 ms, 2,000 atoms
// at 17 moments (one CTA per atom, hash table in global memory before) 10.6 ->
// 1.3 ms.
constexpr unsigned short GRID_CLAIM = 0x8000;  // pass 0: claimed, index not yet assigned; else index + 1
constexpr int ORDER_KEYS = (BOP_MAX_K + 1) * 33;  // (shell, entries) of a row

// site record: atom (24 bits), image bytes + 128 (24 bits), table address (16 bits)
__device__ __forceinline__ unsigned long long grid_rec(int atom, unsigned img, int addr) {
  return ((unsigned long long)(unsigned)atom << 40) | ((unsigned long long)img << 16) | (unsigned)addr;
}
__device__ __forceinline__ int rec_atom(unsigned long long r) { return (int)(r >> 40); }
__device__ __forceinline__ int rec_addr(unsigned long long r) { return (int)(r & 0xffff); }
__device__ __forceinline__ int rec_img(unsigned long long r, int c) { return (int)((r >> (16 + 8 * c)) & 0xff) - 128; }
// Image bytes of a packed edge or record: component 0 in the high byte, so
// that records order as (atom, sx, sy, sz).
__device__ __forceinline__ int epk_img(int y, int c) { return (int)(((unsigned)y >> (16 - 8 * c)) & 0xffu) - 128; }

// Image of a neighbour: the site's plus the edge's, per component, as bytes
// + 128; false if a component leaves [-127, 127].
__device__ __forceinline__ bool image_sum(unsigned long long rec, int epk, unsigned* img) {
  const unsigned ti = (unsigned)(rec >> 16), ei = (unsigned)epk;
  const unsigned x = ((ti >> 16) & 255u) + ((ei >> 16) & 255u) - 128u, y = ((ti >> 8) & 255u) + ((ei >> 8) & 255u) - 128u,
                 z = (ti & 255u) + (ei & 255u) - 128u;
  *img = (x << 16) | (y << 8) | z;
  return x - 1u < 255u && y - 1u < 255u && z - 1u < 255u;
}

template <int G>
__device__ __forceinline__ void group_sync() {
  if constexpr (G == 32) __syncwarp();
  else __syncthreads();
}

// One compare-exchange step with the key of index idx ^ j, in the merge of
// blocks of k.
__device__ __forceinline__ unsigned cmp_exchange(unsigned x, unsigned y, int idx, int j, int k) {
  return ((idx & j) == 0) == ((idx & k) == 0) ? min(x, y) : max(x, y);
}
// Strides 32 .. 1 of the merge of blocks of k over 64 keys of one warp: lane
// holds keys i0 (x0) and i0 + 32 (x1).
__device__ __forceinline__ void merge64(unsigned& x0, unsigned& x1, int i0, int k) {
  if (k >= 64) {
    const unsigned lo = min(x0, x1), hi = max(x0, x1);
    const bool up = (i0 & k) == 0;
    x0 = up ? lo : hi;
    x1 = up ? hi : lo;
  }
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    if (j >= k) continue;
    const unsigned y0 = __shfl_xor_sync(0xffffffffu, x0, j), y1 = __shfl_xor_sync(0xffffffffu, x1, j);
    x0 = cmp_exchange(x0, y0, i0, j, k);
    x1 = cmp_exchange(x1, y1, i0 + 32, j, k);
  }
}
// Ascending bitonic sort of a[0..cnt) by the group.  Every warp holds 64
// keys in registers and exchanges them by shuffles; only strides of 64 and
// more go through shared memory (three block barriers for 256 keys).  The
// keys were written before a group barrier.
template <int G>
__device__ __forceinline__ void group_sort(unsigned* a, int cnt, int tid) {
  int P = 64;
  while (P < cnt) P <<= 1;
  if (P <= 2 * G) {
    const int i0 = (tid >> 5) * 64 + (tid & 31), i1 = i0 + 32;
    const bool active = i0 < P;  // whole warps
    unsigned x0 = ~0u, x1 = ~0u;
    if (active) {
      if (i0 < cnt) x0 = a[i0];
      if (i1 < cnt) x1 = a[i1];
#pragma unroll
      for (int k = 2; k <= 64; k <<= 1) merge64(x0, x1, i0, k);
    }
    for (int k = 128; k <= P; k <<= 1) {
      for (int j = k >> 1; j >= 64; j >>= 1) {
        group_sync<G>();
        if (active) {
          a[i0] = x0;
          a[i1] = x1;
        }
        group_sync<G>();
        if (active) {
          x0 = cmp_exchange(x0, a[i0 ^ j], i0, j, k);
          x1 = cmp_exchange(x1, a[i1 ^ j], i1, j, k);
        }
      }
      if (active) merge64(x0, x1, i0, k);
    }
    group_sync<G>();
    if (active) {
      if (i0 < cnt) a[i0] = x0;
      if (i1 < cnt) a[i1] = x1;
    }
    group_sync<G>();
    return;
  }
  for (int i = cnt + tid; i < P; i += G) a[i] = ~0u;
  group_sync<G>();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int p = tid; p < P / 2; p += G) {
        const int i = ((p & ~(j - 1)) << 1) | (p & (j - 1)), l = i | j;
        const unsigned lo = min(a[i], a[l]), hi = max(a[i], a[l]);
        const bool up = (i & k) == 0;
        a[i] = up ? lo : hi;
        a[l] = up ? hi : lo;
      }
      group_sync<G>();
    }
}

// Stable order of the sites [0, cnt) by ascending key(t) < nkeys, by one warp:
// put(rank, t).  off: nkeys counters.  Sites of equal key keep their order, so
// that the result does not depend on timing.
template <class Key, class Put>
__device__ __forceinline__ void warp_order(int cnt, int nkeys, int* off, int lane, Key key, Put put) {
  for (int q = lane; q < nkeys; q += 32) off[q] = 0;
  __syncwarp();
  for (int t = lane; t < cnt; t += 32) atomicAdd(&off[key(t)], 1);
  __syncwarp();
  int run = 0;
  for (int q0 = 0; q0 < nkeys; q0 += 32) {
    const int q = q0 + lane, c = q < nkeys ? off[q] : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (q < nkeys) off[q] = run + incl - c;
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  for (int t0 = 0; t0 < cnt; t0 += 32) {
    const int t = t0 + lane;
    const int k = t < cnt ? key(t) : nkeys;
    const unsigned same = __match_any_sync(0xffffffffu, k);
    const int rank = __popc(same & ((1u << lane) - 1u));
    const int base = t < cnt ? off[k] : 0;
    __syncwarp();
    if (t < cnt) {
      if (rank == 0) off[k] = base + __popc(same);
      put(base + rank, t);
    }
    __syncwarp();
  }
}

// Keys of the atom alone: how far entry q of the sorted keys lies from its
// place among the images of its atom, which stand side by side.
__device__ __forceinline__ int image_rank(const unsigned* keys, const unsigned long long* nb, int q, int cnt,
                                          unsigned mask) {
  const unsigned long long r = nb[keys[q] & mask];
  int d = 0;
  for (int p = q - 1; p >= 0; p--) {
    const unsigned long long o = nb[keys[p] & mask];
    if (rec_atom(o) != rec_atom(r)) break;
    d -= o > r ? 1 : 0;
  }
  for (int p = q + 1; p < cnt; p++) {
    const unsigned long long o = nb[keys[p] & mask];
    if (rec_atom(o) != rec_atom(r)) break;
    d += o < r ? 1 : 0;
  }
  return d;
}

// What a row step needs of its site, in shared memory (written one thread per
// site, read by the row's lanes): the first edge, and the address and degree.
__device__ __forceinline__ int2 site_row(int2 row, int addr) { return make_int2(row.x, addr | (row.y << 16)); }

// Bytes of the table; in pass 1 at least those of the orders that follow it
// in its place.
__host__ __device__ __forceinline__ size_t grid_front(int pass, const GridArgs& a) {
  const size_t tab = (size_t)(a.tsize * 2 + 15) / 16 * 16;
  const size_t ord = (8 * (size_t)((a.sites + 1) & ~1) + 3 * ORDER_KEYS * sizeof(int) + 15) / 16 * 16;
  return pass == 0 || tab > ord ? tab : ord;
}

template <int PASS, bool CUT, int G>
__global__ void __launch_bounds__(G) k_cluster_grid(GridArgs A, PathCut pc, ClusterOut out) {
  extern __shared__ __align__(16) unsigned char grid_raw[];
  __shared__ int s_lev[BOP_MAX_K + 1];
  __shared__ int s_cnt, s_fail;
  __shared__ int s_warp[G / 32 + 1];
  unsigned short* tab = reinterpret_cast<unsigned short*>(grid_raw);
  const int tab16 = (A.tsize * 2 + 15) / 16;  // 16-byte words
  unsigned char* tail = grid_raw + grid_front(PASS, A);
  // pass 0: the new records of a level, their sort keys, site records, site rows
  unsigned long long* nb = reinterpret_cast<unsigned long long*>(tail);
  unsigned* keys = reinterpret_cast<unsigned*>(nb + A.newcap);
  unsigned long long* sk = reinterpret_cast<unsigned long long*>(keys + A.newcap);
  int2* srow = reinterpret_cast<int2*>(sk + A.maxs);
  // pass 1: per site {site row, first site of its level | first site of the
  // next level, row offset}, then entries per class
  int4* sinf = reinterpret_cast<int4*>(tail);
  // after the rows, in the table's place: the orders, and the counters of their sorts
  unsigned short* ord = reinterpret_cast<unsigned short*>(grid_raw);  // [4][sites]
  int* ocnt = reinterpret_cast<int*>(grid_raw + (size_t)8 * ((A.sites + 1) & ~1));  // [3][ORDER_KEYS]
  const int tid = threadIdx.x, lane = tid & 31;
  const int K = A.K;
  const int sub = tid >> A.lpr_shift, j = tid & ((1 << A.lpr_shift) - 1);  // row of the step, edge of the row
  const int rps = G >> A.lpr_shift;                                        // rows per step
  const unsigned hm = A.lpr_shift == 5 ? 0xffffffffu : (lane < 16 ? 0xffffu : 0xffff0000u);  // the row's lanes
  const unsigned below = hm & ((1u << lane) - 1u);
  constexpr int U = 2;  // row steps in flight
  unsigned long long prod = 0;
  for (int atom = blockIdx.x; atom < A.n; atom += gridDim.x) {
    for (int q = tid; q < tab16; q += G) reinterpret_cast<uint4*>(tab)[q] = make_uint4(0, 0, 0, 0);
    unsigned long long* gk = A.recs + (size_t)atom * A.maxs;
    unsigned char* gc = A.counts + (size_t)atom * A.maxs;
    if (tid == 0) s_fail = s_cnt = 0;
    if (PASS == 0) {
      group_sync<G>();
      if (tid == 0) {
        const int a0 = A.origin + A.slot[atom];
        tab[a0] = 1;
        const unsigned long long r = grid_rec(atom, 0x808080u, a0);
        sk[0] = gk[0] = r;
        srow[0] = site_row(A.rows[atom], a0);
        s_lev[0] = 1;
      }
      group_sync<G>();
      int nsite = 1, f0 = 0;
      int tot = 0;  // adjacency entries
      for (int k = 1; k <= K; k++) {
        const int f1 = nsite;
        for (int t0 = f0; t0 < f1; t0 += U * rps) {
          int2 sr[U];
          int ad[U];
#pragma unroll
          for (int u = 0; u < U; u++) {
            const int t = t0 + u * rps + sub;
            sr[u] = t < f1 ? srow[t] : make_int2(0, 0);
          }
#pragma unroll
          for (int u = 0; u < U; u++)
            ad[u] = j < (sr[u].y >> 16) ? (sr[u].y & 0xffff) + __ldg(&A.eoff[sr[u].x + j].x) : -1;
#pragma unroll
          for (int u = 0; u < U; u++) {
            // not yet a site of the cluster
            bool win = ad[u] != -1 && ((unsigned)ad[u] >= (unsigned)A.tsize || tab[ad[u]] == 0);
            const int t = t0 + u * rps + sub, e = sr[u].x + j;
            if (CUT && win) {  // path-radius cut: only sites closer than r_path to the atom
              const int2 pe = __ldg(A.epack + e);
              unsigned img;
              if (!image_sum(sk[t], pe.y, &img)) {
                s_fail = 1;
                raise_error(A.status, BOP_DEV_ERR_IMAGE);
                win = false;
              } else {
                double d[3];
                bond_vector(pc.pos + 3 * (size_t)atom, pc.pos + 3 * (size_t)pe.x, pc.cell, (int)(img >> 16) - 128,
                            (int)((img >> 8) & 255u) - 128, (int)(img & 255u) - 128, d);
                win = norm2_rn(d) < pc.r2;
              }
            }
            if (win && (unsigned)ad[u] >= (unsigned)A.tsize) {  // outside the planned table: the general builder
              s_fail = 1;
              win = false;
            }
            if (win) {
              const int sh = (ad[u] & 1) * 16;
              const unsigned old = atomicOr(reinterpret_cast<unsigned*>(tab) + (ad[u] >> 1), (unsigned)GRID_CLAIM << sh);
              if (((old >> sh) & 0xffffu) == 0) {
                const int q = atomicAdd(&s_cnt, 1);
                if (q < A.newcap) nb[q] = ((unsigned long long)(unsigned)e << 32) | (unsigned)t;
              }
            }
          }
        }
        group_sync<G>();
        const int cnt = s_cnt;
        const bool bad = s_fail != 0 || cnt > A.newcap || cnt > A.maxs - nsite;
        group_sync<G>();
        if (bad) {
          if (tid == 0) s_fail = 1;
          break;
        }
        // the claimed (site, edge) pairs become records; canonical order inside the level
        for (int q = tid; q < cnt; q += G) {
          const unsigned long long c = nb[q];
          const unsigned long long rt = sk[(unsigned)c];
          const int e = (int)(c >> 32);
          const int2 pe = __ldg(A.epack + e);
          unsigned img;
          if (!image_sum(rt, pe.y, &img)) {
            s_fail = 1;
            raise_error(A.status, BOP_DEV_ERR_IMAGE);
            img = 0x808080u;  // an image beyond a byte would reach the record's atom
          }
          nb[q] = grid_rec(pe.x, img, rec_addr(rt) + __ldg(&A.eoff[e].x));
          const unsigned code = (((img >> 16) - 128u + A.mx) * (2u * A.my + 1u) + ((img >> 8) & 255u) - 128u + A.my) *
                                    (2u * A.mz + 1u) + (img & 255u) - 128u + A.mz;
          keys[q] = (A.ncode > 0 ? (unsigned)pe.x * A.ncode + code : (unsigned)pe.x) << A.qbits | (unsigned)q;
        }
        group_sync<G>();
        group_sort<G>(keys, cnt, tid);
        for (int q = tid; q < cnt; q += G) {
          const unsigned long long r = nb[keys[q] & ((1u << A.qbits) - 1u)];
          const int t = nsite + q + (A.ncode > 0 ? 0 : image_rank(keys, nb, q, cnt, (1u << A.qbits) - 1u));
          const int2 row = __ldg(A.rows + rec_atom(r));
          sk[t] = gk[t] = r;
          srow[t] = site_row(row, rec_addr(r));
          tab[rec_addr(r)] = (unsigned short)(t + 1);
          // without a path cut every neighbour of a site within K-1 hops is in the cluster
          if (!CUT && k < K) {
            gc[t] = (unsigned char)row.y;
            tot += row.y;
          }
        }
        f0 = f1;
        nsite += cnt;
        if (tid == 0) {
          s_lev[k] = nsite;
          s_cnt = 0;
        }
        group_sync<G>();
      }
      group_sync<G>();
      if (s_fail) {
        if (tid == 0) {
          atomicOr(A.fail, 1);
          out.atom_nsite[atom] = 0;
          out.atom_nadj[atom] = 0;
        }
        group_sync<G>();
        continue;
      }
      // adjacency counts of the other sites
      if (!CUT && tid == 0) {
        gc[0] = (unsigned char)(srow[0].y >> 16);
        tot += srow[0].y >> 16;
      }
      for (int t0 = CUT ? 0 : f0; t0 < nsite; t0 += U * rps) {
        int2 sr[U];
        int ad[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int t = t0 + u * rps + sub;
          sr[u] = t < nsite ? srow[t] : make_int2(0, 0);
        }
#pragma unroll
        for (int u = 0; u < U; u++)
          ad[u] = j < (sr[u].y >> 16) ? (sr[u].y & 0xffff) + __ldg(&A.eoff[sr[u].x + j].x) : -1;
#pragma unroll
        for (int u = 0; u < U; u++) {
          const bool hit = (unsigned)ad[u] < (unsigned)A.tsize && tab[ad[u]] != 0;
          const int c = __popc(__ballot_sync(0xffffffffu, hit) & hm);
          const int t = t0 + u * rps + sub;
          if (j == 0 && t < nsite) {
            gc[t] = (unsigned char)c;
            tot += c;
          }
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      if (G > 32) {
        if (lane == 0) s_warp[tid >> 5] = tot;
        group_sync<G>();
        tot = 0;
        for (int w = 0; w < G / 32; w++) tot += s_warp[w];
      }
      if (tid == 0) {
        out.atom_nsite[atom] = nsite;
        out.atom_nadj[atom] = tot;
        if (tot > *(volatile int*)&out.max_level[K + 1]) atomicMax(&out.max_level[K + 1], tot);
      }
      for (int k = tid; k <= K; k += G) {
        out.level_end[(size_t)atom * (K + 1) + k] = s_lev[k];
        if (s_lev[k] > *(volatile int*)&out.max_level[k]) atomicMax(&out.max_level[k], s_lev[k]);
      }
      group_sync<G>();
    } else {
      for (int k = tid; k <= K; k += G) s_lev[k] = out.level_end[(size_t)atom * (K + 1) + k];
      const long long s0 = out.site_off[atom], a0 = out.adj_base[atom];
      group_sync<G>();
      const int nsite = s_lev[K];
      // sites, and the row offsets (exclusive sum of the counts of pass 0)
      int run = 0;
      for (int tb = 0; tb < nsite; tb += G) {
        const int t = tb + tid;
        int c = 0, lo = 0, hi = 0;
        int2 sr = make_int2(0, 0);
        if (t < nsite) {
          const unsigned long long r = gk[t];
          c = gc[t];
          sr = site_row(__ldg(A.rows + rec_atom(r)), rec_addr(r));
          const bool sel = pair_selected(atom, rec_atom(r), rec_img(r, 2), rec_img(r, 1), rec_img(r, 0));
          tab[rec_addr(r)] = (unsigned short)((t + 1) | (sel ? GRID_CLAIM : 0));
          out.site_atom[s0 + t] = rec_atom(r);
          signed char* si = out.site_img + 3 * (s0 + t);
          si[0] = (signed char)rec_img(r, 2);
          si[1] = (signed char)rec_img(r, 1);
          si[2] = (signed char)rec_img(r, 0);
          // first site of t's own level, of the one after
          int lt = 0;
          while (t >= s_lev[lt]) lt++;
          lo = lt > 0 ? s_lev[lt - 1] : 0;
          hi = s_lev[lt];
        }
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += v;
        }
        int base = run;
        if (G > 32) {
          if (lane == 31) s_warp[tid >> 5] = incl;
          group_sync<G>();
          int tot = 0;
          for (int w = 0; w < G / 32; w++) {
            if (w == (tid >> 5)) base = run + tot;
            tot += s_warp[w];
          }
          run += tot;
          group_sync<G>();
        } else {
          run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (t < nsite) {
          sinf[t] = make_int4(sr.x, sr.y, lo | (hi << 16), base + incl - c);
          out.adj_off[s0 + t] = a0 + base + incl - c;
        }
      }
      group_sync<G>();
      int2* adj = out.adj + a0;
      for (int t0 = 0; t0 < nsite; t0 += U * rps) {
        int4 si[U];
        int2 eo[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int t = t0 + u * rps + sub;
          si[u] = t < nsite ? sinf[t] : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < U; u++) eo[u] = j < (si[u].y >> 16) ? __ldg(A.eoff + si[u].x + j) : make_int2(-65536, 0);
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int ad = (si[u].y & 0xffff) + eo[u].x;
          const int w = (unsigned)ad < (unsigned)A.tsize ? (int)tab[ad] : 0;
          const int v = w & (GRID_CLAIM - 1);  // site + 1, or not in the cluster; the other bit: selected
          const int lo = si[u].z & 0xffff, hi = (unsigned)si[u].z >> 16;
          // the entries of the levels l-1, l, l+1, each in row order
          const unsigned ball = __ballot_sync(0xffffffffu, v != 0) & hm;
          const unsigned b1 = __ballot_sync(0xffffffffu, v > lo) & hm;  // levels >= l
          const unsigned b2 = __ballot_sync(0xffffffffu, v > hi) & hm;  // level l + 1
          const unsigned b0 = ball & ~b1;
          const int n0 = __popc(b0), n01 = n0 + __popc(b1 & ~b2);
          const unsigned mine = v > hi ? b2 : (v > lo ? (b1 & ~b2) : b0);
          const int first = v > hi ? n01 : (v > lo ? n0 : 0);
          const int pos = first + __popc(mine & below);
          if (v) adj[si[u].w + pos] = make_int2(v - 1, eo[u].y);
          const unsigned selm = __reduce_or_sync(hm, v != 0 && w >= GRID_CLAIM ? 1u << pos : 0u);
          // the row's counts replace its offset, the selected entries its first edge
          const int t = t0 + u * rps + sub;
          if (j == 0 && t < nsite) {
            sinf[t].x = (int)selm;
            sinf[t].w = n0 | (n01 << 8) | (__popc(ball) << 16);
          }
        }
      }
      group_sync<G>();
      for (int t = tid; t < nsite; t += G) {
        const int w = sinf[t].w, n0 = w & 255, n01 = (w >> 8) & 255, n012 = (w >> 16) & 255;
        int lt = 0;
        while (t >= s_lev[lt]) lt++;
        sinf[t].y = lt;
        // byte k: entries of level <= k, k < K
        unsigned long long lc = 0;
        for (int k = lt > 0 ? lt - 1 : 0; k < K; k++)
          lc |= (unsigned long long)(k < lt ? n0 : (k == lt ? n01 : n012)) << (8 * k);
        out.lvcnt[s0 + t] = lc;
        if (out.top != nullptr) out.topmask[s0 + t] = (unsigned)sinf[t].x;
        // forward levels k = max(lt, ls + 1) .. K use the pair (t, s)
        prod += (unsigned long long)(n0 * (K - lt + 1) + (n01 - n0) * (K - lt) + (n012 - n01) * (K > lt ? K - lt - 1 : 0));
      }
      group_sync<G>();
      // the orders (one warp each)
      const int S2 = A.sites;
      for (int w = tid >> 5; w < 3; w += G / 32) {
        int* off = ocnt + w * ORDER_KEYS;
        if (w < 2 && out.order == nullptr) continue;
        if (w < 2) {  // by shell, then descending entries of the level below / up to its own
          const int sh = 8 * w;
          warp_order(nsite, (K + 1) * 33, off, lane,
                     [&](int t) { return sinf[t].y * 33 + 32 - ((sinf[t].w >> sh) & 255); },
                     [&](int q, int t) { ord[w * S2 + q] = (unsigned short)t; });
        } else if (out.top != nullptr) {  // C_K-1 by descending selected entries
          warp_order(s_lev[K - 1], 33, off, lane, [&](int t) { return 32 - __popc((unsigned)sinf[t].x); },
                     [&](int q, int t) { ord[3 * S2 + q] = (unsigned short)t; });
        }
      }
      group_sync<G>();
      if (out.order != nullptr)
        for (int q = tid; q < nsite; q += G) out.order[s0 + q] = (unsigned)ord[q] | ((unsigned)ord[S2 + q] << 16);
      if (out.top != nullptr) {
        if (tid < 32) {  // the selected sites in the order of the last level's rows
          int run = 0, in = 0;
          const int l2 = K >= 2 ? s_lev[K - 2] : 0, l1 = s_lev[K - 1];
          for (int q0 = 0; q0 < nsite; q0 += 32) {
            const int q = q0 + lane;
            const int t = q >= nsite ? 0 : (out.order == nullptr || q < l2 ? q : (q < l1 ? ord[S2 + q] : ord[q]));
            bool sel = false;
            if (q < nsite) {
              const unsigned long long r = gk[t];
              sel = pair_selected(atom, rec_atom(r), rec_img(r, 2), rec_img(r, 1), rec_img(r, 0));
            }
            const unsigned bal = __ballot_sync(0xffffffffu, sel);
            if (sel) ord[2 * S2 + run + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)t;
            run += __popc(bal);
            in += __popc(__ballot_sync(0xffffffffu, sel && q < l1));
          }
          if (lane == 0) {
            s_cnt = run;
            out.ntop[atom] = run | (in << 16);
          }
        }
        group_sync<G>();
        const int nt = s_cnt, nr = s_lev[K - 1];
        for (int q = tid; q < nsite; q += G)
          out.top[s0 + q] = (q < nt ? (unsigned)ord[2 * S2 + q] : 0u) | ((q < nr ? (unsigned)ord[3 * S2 + q] : 0u) << 16);
      }
      group_sync<G>();
    }
  }
  if (PASS == 1) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) prod += __shfl_xor_sync(0xffffffffu, prod, o);
    if (lane == 0 && prod) atomicAdd(out.n_products, prod);
  }
}

}  // namespace

int launch_cluster(int pass, int n, int K, const long long* row_ptr, const int* col, const signed char* img,
                   const int* bond_of_edge, PathCut pc, ClusterScratch sc, ClusterOut out, int grid,
                   unsigned* status, cudaStream_t s) {
  size_t smem = (size_t)sc.newcap * sizeof(unsigned long long);  // newcap is a power of two
  // the path cut is a separate instantiation: its distance arithmetic costs
  // registers that the uncut BFS does not need
  const bool cut = pc.r2 > 0.0;
  auto fn = pass == 0 ? (cut ? k_cluster<0, true> : k_cluster<0, false>)
                      : (cut ? k_cluster<1, true> : k_cluster<1, false>);
  if (!allow_smem(fn)) return -1;
  fn<<<grid, CL_THREADS, smem, s>>>(n, K, row_ptr, col, img, bond_of_edge, pc, sc, out, status);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// What the grid builder needs of every directed edge i -> (j, image), one
// warp per atom: {col, image bytes + 128}, {address offset, bond}, and each
// atom's {first edge, degree}.
__global__ void k_pack_edges(int n, GridPlan p, Geometry g, const long long* __restrict__ row_ptr,
                             const int* __restrict__ col, const signed char* __restrict__ img,
                             const int* __restrict__ bond_of_edge, const int* __restrict__ cell_of,
                             const int* __restrict__ slot, int2* __restrict__ epack, int2* __restrict__ eoff,
                             int2* __restrict__ rows) {
  const int lane = threadIdx.x & 31;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= n) return;
  const long long e0 = row_ptr[i], e1 = row_ptr[i + 1];
  if (lane == 0) rows[i] = make_int2((int)e0, (int)(e1 - e0));
  const int ci = cell_of[i], si = slot[i];
  const int cx = ci / (g.nc[1] * g.nc[2]), cy = (ci / g.nc[2]) % g.nc[1], cz = ci % g.nc[2];
  for (long long e = e0 + lane; e < e1; e += 32) {
    const int jj = col[e], sx = img[3 * e], sy = img[3 * e + 1], sz = img[3 * e + 2];
    const int cj = cell_of[jj];
    const int dx = cj / (g.nc[1] * g.nc[2]) + sx * g.nc[0] - cx;
    const int dy = (cj / g.nc[2]) % g.nc[1] + sy * g.nc[1] - cy;
    const int dz = cj % g.nc[2] + sz * g.nc[2] - cz;
    epack[e] = make_int2(jj, (int)(((unsigned)(sx + 128) << 16) | ((unsigned)(sy + 128) << 8) | (unsigned)(sz + 128)));
    eoff[e] = make_int2(((dx * p.py + dy) * p.pz + dz) * p.slots + slot[jj] - si, bond_of_edge[e]);
  }
}

int launch_pack_edges(int n, const GridPlan& p, const Geometry& g, const long long* row_ptr, const int* col,
                      const signed char* img, const int* bond_of_edge, const int* cell_of, const int* slot,
                      int2* epack, int2* eoff, int2* rows, cudaStream_t s) {
  if (n <= 0) return 0;
  k_pack_edges<<<(n + 7) / 8, 256, 0, s>>>(n, p, g, row_ptr, col, img, bond_of_edge, cell_of, slot, epack, eoff, rows);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Structure maxima the grid builder is planned with: out[0] the largest
// degree, out[1] the most atoms of a linked cell, out[2..4] the largest bond
// component along each axis in units of linked cells, rounded up to
// 1/GRID_UNIT.  out starts at zero.
__global__ void k_grid_maxima(int n, const long long* __restrict__ row_ptr, int ncell,
                              const int* __restrict__ cell_start, long long nb, const double* __restrict__ bond_d,
                              Geometry g, int* __restrict__ out) {
  const long long q0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  int m[5] = {0, 0, 0, 0, 0};
  for (long long i = q0; i < n; i += step) m[0] = max(m[0], (int)(row_ptr[i + 1] - row_ptr[i]));
  for (long long i = q0; i < ncell; i += step) m[1] = max(m[1], cell_start[i + 1] - cell_start[i]);
  for (long long b = q0; b < nb; b += step) {
    const double x = bond_d[3 * b], y = bond_d[3 * b + 1], z = bond_d[3 * b + 2];
#pragma unroll
    for (int a = 0; a < 3; a++)
      m[2 + a] = max(m[2 + a], (int)(fabs(x * g.inv[a] + y * g.inv[3 + a] + z * g.inv[6 + a]) * g.nc[a] * GRID_UNIT) + 1);
  }
#pragma unroll
  for (int v = 0; v < 5; v++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m[v] = max(m[v], __shfl_xor_sync(0xffffffffu, m[v], o));
    if ((threadIdx.x & 31) == 0 && m[v] > 0) atomicMax(out + v, m[v]);
  }
}

void launch_grid_maxima(int n, const long long* row_ptr, int ncell, const int* cell_start, long long nb,
                        const double* bond_d, const Geometry& g, int* out, cudaStream_t s) {
  const long long work = nb > n ? nb : n;
  const int grid = (int)((work + 255) / 256 < 304 ? (work + 255) / 256 : 304);
  if (n > 0) k_grid_maxima<<<grid, 256, 0, s>>>(n, row_ptr, ncell, cell_start, nb, bond_d, g, out);
}

// Cells within k hops of an atom along one axis: at most the displacement in
// cells, plus one for the two atoms' places inside their cells (the slack
// covers atoms up to 1e-9 of the cell outside it, and the rounding of maxima).
static int hop_reach(int k, int unit_max) { return (int)((double)k * unit_max / GRID_UNIT + 1e-5) + 1; }

bool grid_plan(const Geometry& g, int K, const int* maxima, GridPlan* p) {
  int r[3], per[3];
  for (int a = 0; a < 3; a++) {
    r[a] = hop_reach(K, maxima[2 + a]);
    per[a] = r[a] + hop_reach(K + 1, maxima[2 + a]) + 1;
  }
  const long long half = ((long long)r[0] * per[1] + r[1]) * per[2] + r[2];
  p->py = per[1];
  p->pz = per[2];
  p->slots = maxima[1] > 0 ? maxima[1] : 1;
  const long long size = (2 * half + 1) * p->slots;
  if (size > 65535) return false;  // 16-bit addresses
  p->origin = (int)half * p->slots;
  // images of sites lie within m of the home cell
  int* m[3] = {&p->mx, &p->my, &p->mz};
  for (int a = 0; a < 3; a++) *m[a] = g.pbc[a] ? (r[a] + g.nc[a] - 1) / g.nc[a] : 0;
  p->tsize = (int)size;
  return true;
}

// Codes per atom in the 32-bit sort keys of a level (newcap entries) of a
// structure of n atoms with ncode images each: ncode where they fit, 0 (keys of
// the atom alone, its images put in order after the sort) up to 2^24 atoms at
// 256 entries, -1 beyond.  With 27 images the codes end at 621,378 atoms.
extern "C" int cluster_key_codes(int n, int ncode, int newcap) {
  int qbits = 0;
  while ((1 << qbits) < newcap) qbits++;
  const unsigned long long limit = 1ull << (32 - qbits);
  if ((unsigned long long)n * (unsigned)ncode < limit) return ncode;
  return (unsigned long long)n <= limit ? 0 : -1;
}

template <int PASS, bool CUT, int G>
static int run_grid(const GridArgs& a, const PathCut& pc, const ClusterOut& out, int sms, cudaStream_t s) {
  auto fn = k_cluster_grid<PASS, CUT, G>;
  const size_t smem = grid_front(PASS, a) + 
                      (PASS == 0 ? 16 * (size_t)a.maxs + 12 * (size_t)a.newcap : 16 * (size_t)a.sites);
  if (smem > SMEM_MAX) return -2;
  if (!allow_smem(fn)) return -1;
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, G, smem) != cudaSuccess) return -1;
  if (per < 1) return -2;
  const int grid = a.n < sms * per ? a.n : sms * per;
  fn<<<grid, G, smem, s>>>(a, pc, out);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <int G>
static int run_grid_pass(int pass, const GridArgs& a, const PathCut& pc, const ClusterOut& out, int sms, cudaStream_t s) {
  const bool cut = pc.r2 > 0.0;
  if (pass == 0) return cut ? run_grid<0, true, G>(a, pc, out, sms, s) : run_grid<0, false, G>(a, pc, out, sms, s);
  return cut ? run_grid<1, true, G>(a, pc, out, sms, s) : run_grid<1, false, G>(a, pc, out, sms, s);
}

int launch_cluster_grid(int pass, const GridArgs& a, const PathCut& pc, const ClusterOut& out, cudaStream_t s) {
  if (a.n == 0) return 0;
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // Threads per cluster, both passes with 128 / 256 / 512: eight rows a step for
  // many clusters (131,072 bcc atoms at 9 moments 6.70 / 7.04 / 9.15 ms, 2,000
  // atoms 0.123 / 0.126 / 0.159), twice the threads where a row takes 32 lanes,
  // and 512 where the clusters do not fill the SMs (250 atoms 0.059 / 0.047 /
  // 0.042 ms) or outgrow the first tier (2,000 atoms at 17 moments 3.18 / 1.93 /
  // 1.33 ms, 16,000 at 13 moments 4.54 / 3.01 / 2.91; 1,372 fcc atoms at 9
  // moments, the exception, 0.241 / 0.177 / 0.189).
  if (a.maxs <= 512 && a.n > 4 * sms)
    return a.lpr_shift == 4 ? run_grid_pass<128>(pass, a, pc, out, sms, s) : run_grid_pass<256>(pass, a, pc, out, sms, s);
  return run_grid_pass<512>(pass, a, pc, out, sms, s);
}

// The pair form's way back, one block per atom j: a site (i, s) of its cluster
// that is not selected is the selected site (j, -s) of i's cluster, in the same
// shell.  mirror + site_off[j]: the places of those among the sites of all
// clusters (a binary search of the shell's canonical order), in the order of
// j's sites.
constexpr int MIR_THREADS = 512;

__global__ void __launch_bounds__(MIR_THREADS) k_pair_mirror(int K, const long long* __restrict__ site_off,
                                                             const int* __restrict__ level_end,
                                                             const int* __restrict__ site_atom,
                                                             const signed char* __restrict__ site_img,
                                                             unsigned* __restrict__ mirror,
                                                             unsigned* __restrict__ status) {
  __shared__ int s_lev[BOP_MAX_K + 1], s_cnt[MIR_THREADS / 32];
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const long long s0 = site_off[j];
  if (tid <= K) s_lev[tid] = level_end[(size_t)j * (K + 1) + tid];
  __syncthreads();
  const int nsite = s_lev[K];
  int done = 0;  // entries of the rounds before
  for (int u0 = 0; u0 < nsite; u0 += MIR_THREADS) {
    const int u = u0 + tid;
    int i = j, sx = 0, sy = 0, sz = 0;  // (the centre is selected)
    if (u < nsite) {
      const signed char* im = site_img + 3 * (s0 + u);
      i = site_atom[s0 + u];
      sx = im[0];
      sy = im[1];
      sz = im[2];
    }
    const bool mine = !pair_selected(j, i, sx, sy, sz);
    const unsigned bal = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) s_cnt[wid] = __popc(bal);
    __syncthreads();
    int at = done + __popc(bal & ((1u << lane) - 1u));
    for (int w = 0; w < MIR_THREADS / 32; w++) {
      if (w < wid) at += s_cnt[w];
      done += s_cnt[w];
    }
    __syncthreads();
    if (!mine) continue;  // (barriers above only)
    int l = 1;
    while (u >= s_lev[l]) l++;
    const int* li = level_end + (size_t)i * (K + 1);
    const long long b = site_off[i];
    int lo = li[l - 1], hi = li[l];
    const int end = hi;
    auto order = [&](int m) {  // site m of i's cluster against (j, -s)
      const int a = site_atom[b + m];
      if (a != j) return a < j ? -1 : 1;
      const signed char* q = site_img + 3 * (b + m);
      if (q[0] != -sx) return q[0] < -sx ? -1 : 1;
      if (q[1] != -sy) return q[1] < -sy ? -1 : 1;
      return q[2] != -sz ? (q[2] < -sz ? -1 : 1) : 0;
    };
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (order(mid) < 0) lo = mid + 1;
      else hi = mid;
    }
    if (lo >= end || order(lo) != 0) {  // cannot happen: hops are symmetric
      raise_error(status, BOP_DEV_ERR_CLUSTER);
      lo = 0;
    }
    mirror[s0 + at] = (unsigned)(b + lo);
  }
}

int launch_pair_mirror(int n, int K, const long long* site_off, const int* level_end, const int* site_atom,
                       const signed char* site_img, unsigned* mirror, unsigned* status, cudaStream_t s) {
  if (n <= 0) return 0;
  k_pair_mirror<<<n, MIR_THREADS, 0, s>>>(K, site_off, level_end, site_atom, site_img, mirror, status);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Rows of one stored Psi sweep per atom: sum_{k=0..K} |C_k|.
__global__ void k_level_sums(int n, int K, const int* __restrict__ level_end, long long* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  long long a = 0;
  for (int k = 0; k <= K; k++) a += level_end[(size_t)i * (K + 1) + k];
  out[i] = a;
}

void launch_level_sums(int n, int K, const int* level_end, long long* out, cudaStream_t s) {
  k_level_sums<<<(n + 255) / 256, 256, 0, s>>>(n, K, level_end, out);
}
