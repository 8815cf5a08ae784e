// Galerkin coarse operators A_{l+1} = P^T A_l P (eq. (R), eq. (Ac)) on the
// device, with P = P_s (x) I_d and the rows of dead fine dofs masked.
//
// Pattern: the structural block product of P_s^T pattern(A_l) P_s plus the
// diagonal (pairs (I, J) generated per fine vertex, each fine vertex's coarse
// columns made unique locally first, then radix sorted and made unique).
// Values: one CTA per coarse row I forms the row S = P_I^T M A_l over the fine
// columns j it reaches (fine rows i ascending), then every block of its row
// as sum_j S_j M w_jJ (j ascending) -- a fixed order, so the result is
// deterministic.  Coarse dofs whose masked column of P is empty are dead and
// get identity rows.
#include "common.cuh"

namespace vasmg {

// Coarse columns a fine row i reaches: the union over the blocks k of A_l's
// row i of the columns of P's row j_k.  Up to GAL_UNION of them are collected,
// sorted and made unique in thread-local storage, so that each (I, J) pair is
// emitted once per fine row; a row with a longer candidate list emits its
// list as it is (the global sort and unique below remove the repeats either
// way, so the pattern is the same).
constexpr int GAL_UNION = 128;

__device__ __forceinline__ int gal_row_union(const int32_t* __restrict__ arp, const int32_t* __restrict__ aci,
                                             const int32_t* __restrict__ prp, const int32_t* __restrict__ pci,
                                             i64 i, int32_t* cols) {
  int n = 0;
  for (int32_t k = arp[i]; k < arp[i + 1]; ++k) {
    const int32_t j = aci[k];
    for (int32_t b = prp[j]; b < prp[j + 1]; ++b) {
      if (n == GAL_UNION) return -1;
      // insertion into the sorted prefix, skipping a repeat
      const int32_t J = pci[b];
      int p = n;
      while (p > 0 && cols[p - 1] > J) --p;
      if (p > 0 && cols[p - 1] == J) continue;
      for (int q = n; q > p; --q) cols[q] = cols[q - 1];
      cols[p] = J;
      ++n;
    }
  }
  return n;
}

__global__ void gal_count_kernel(const int32_t* __restrict__ arp, const int32_t* __restrict__ aci,
                                 const int32_t* __restrict__ prp, const int32_t* __restrict__ pci, i64 nf,
                                 long long* __restrict__ cnt) {
  int32_t cols[GAL_UNION];
  for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < nf; i += (i64)gridDim.x * blockDim.x) {
    long long s = gal_row_union(arp, aci, prp, pci, i, cols);
    if (s < 0) {
      s = 0;
      for (int32_t k = arp[i]; k < arp[i + 1]; ++k) {
        const int32_t j = aci[k];
        s += prp[j + 1] - prp[j];
      }
    }
    cnt[i] = s * (long long)(prp[i + 1] - prp[i]);
  }
}

__global__ void gal_pairs_kernel(const int32_t* __restrict__ arp, const int32_t* __restrict__ aci,
                                 const int32_t* __restrict__ prp, const int32_t* __restrict__ pci, i64 nf,
                                 const long long* __restrict__ off, u64* __restrict__ keys) {
  int32_t cols[GAL_UNION];
  for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < nf; i += (i64)gridDim.x * blockDim.x) {
    long long o = off[i];
    const int nu = gal_row_union(arp, aci, prp, pci, i, cols);
    for (int32_t a = prp[i]; a < prp[i + 1]; ++a) {
      const u64 I = (uint32_t)pci[a];
      if (nu >= 0) {
        for (int q = 0; q < nu; ++q) keys[o++] = (I << 32) | (uint32_t)cols[q];
      } else {
        for (int32_t k = arp[i]; k < arp[i + 1]; ++k) {
          const int32_t j = aci[k];
          for (int32_t b = prp[j]; b < prp[j + 1]; ++b) keys[o++] = (I << 32) | (uint32_t)pci[b];
        }
      }
    }
  }
}

__global__ void diag_pairs_kernel(i64 nc, u64* __restrict__ keys) {
  for (i64 I = (i64)blockIdx.x * blockDim.x + threadIdx.x; I < nc; I += (i64)gridDim.x * blockDim.x)
    keys[I] = ((u64)I << 32) | (u64)I;
}

__global__ void transpose_keys_kernel(const int32_t* __restrict__ prp, const int32_t* __restrict__ pci, i64 nf,
                                      u64* __restrict__ keys, int32_t* __restrict__ vals) {
  for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < nf; i += (i64)gridDim.x * blockDim.x)
    for (int32_t a = prp[i]; a < prp[i + 1]; ++a) {
      keys[a] = ((u64)(uint32_t)pci[a] << 32) | (u64)i;
      vals[a] = a;
    }
}

__global__ void low32_i_kernel(const u64* __restrict__ k, i64 n, int32_t* __restrict__ out) {
  for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (i64)gridDim.x * blockDim.x)
    out[i] = (int32_t)(k[i] & 0xffffffffull);
}

// The row S of a coarse row is kept in a hash table of fine columns in shared
// memory: slots, of which at most 3/4 may be taken.  A row that reaches more
// columns (with the default leaf thresholds, at most 470 in 3D; large thresholds
// and vertices with many neighbours go beyond) is left to gal_wide_kernel.
constexpr int ANY_WIDE_SLOTS = 64;  // levels with a flag of their own (a hierarchy has fewer)
template <int D>
constexpr int gal_slots() { return D == 2 ? 256 : 1024; }
template <int D>
constexpr int gal_threads() { return D == 2 ? 64 : 128; }
template <int D>
constexpr int gal_smem() { return gal_slots<D>() * (D * D * 8 + 4); }

__device__ __forceinline__ unsigned gal_hash(int32_t j, int slots) {
  return ((unsigned)j * 0x9E3779B1u) >> 16 & (unsigned)(slots - 1);
}

// The components of vertex j that are not dead, as bits.
template <int D>
__device__ __forceinline__ unsigned gal_alive(const uint8_t* __restrict__ fdead, i64 j) {
  unsigned f = 0;
#pragma unroll
  for (int s = 0; s < D; ++s) f |= fdead[j * D + s] ? 0u : 1u << s;
  return f;
}

// The coarse rows that the table could not hold (wide): a warp per block (I, J),
// which sums w_iI (M A_l M)_ij w_jJ over R's row J.  Groups of SUB lanes take one
// fine column j each at a time, and their lanes the fine rows i of j's pattern (7
// in 2D and 15 in 3D on a mesh; the pattern is symmetric); w_iI is looked up in
// P's row i, and block (i, j), where it counts, by bisection.  No two warps meet,
// and the sum's order is fixed: a lane's terms, then the xor tree.
// Bound by the latency of the look-ups, so as many warps as there are blocks take
// part.  vasmg_update_data, against a thread per block of the row that walked all
// the row's terms (and against the sum of every term into the row that preceded
// the table): 2D 200^2 with leaf threshold 64 3.34 -> 1.32 ms (2.0), 1000 29.8 ->
// 1.88 (13.0); 3D 33^3 with 64 30.7 -> 8.7 (26.9), 300 57.2 -> 7.9 (23.7); a disc
// around a vertex with 1100 neighbours 21.7 -> 10.0 (12.8).
template <int D>
__global__ void __launch_bounds__(256, 4) gal_wide_kernel(
    i64 nc, const uint8_t* __restrict__ wide, const int32_t* __restrict__ any_wide, const int32_t* __restrict__ rrp,
    const int32_t* __restrict__ rent, const u64* __restrict__ rkeys, const int32_t* __restrict__ prp,
    const int32_t* __restrict__ pci, const double* __restrict__ pw, const int32_t* __restrict__ arp,
    const int32_t* __restrict__ aci, const double* __restrict__ av, const uint8_t* __restrict__ fdead,
    const int32_t* __restrict__ crp, const int32_t* __restrict__ cci, const uint8_t* __restrict__ cdead,
    double* __restrict__ cv) {
  constexpr int DD = D * D, SUB = D == 2 ? 8 : 16, NG = 32 / SUB;
  __shared__ unsigned found[8];
  if (*any_wide == 0) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane / SUB, sub = lane % SUB;
  // the rows blockIdx.x, blockIdx.x + gridDim.x, ...: 256 rows' marks at once
  for (i64 base = 0; blockIdx.x + base * gridDim.x < nc; base += 256) {
    const i64 r = blockIdx.x + (base + threadIdx.x) * gridDim.x;
    const unsigned m = __ballot_sync(0xffffffffu, r < nc && wide[r] != 0);
    __syncthreads();
    if (lane == 0) found[warp] = m;
    __syncthreads();
    for (int w = 0; w < 8; ++w)
      for (unsigned left = found[w]; left; left &= left - 1) {
        const i64 I = blockIdx.x + (base + w * 32 + __ffs(left) - 1) * gridDim.x;
        for (int32_t e = crp[I] + warp + 8 * blockIdx.y; e < crp[I + 1]; e += 8 * gridDim.y) {
          const int32_t J = cci[e], t1 = rrp[J + 1];
          double acc[DD];
#pragma unroll
          for (int q = 0; q < DD; ++q) acc[q] = 0.0;
          for (int32_t t = rrp[J] + g; t < t1; t += NG) {
            const int32_t j = (int32_t)(rkeys[t] & 0xffffffffull);
            const double wJ = pw[rent[t]];
            const unsigned fj = gal_alive<D>(fdead, j);
            const int32_t k1 = arp[j + 1];
            for (int32_t k = arp[j] + sub; k < k1; k += SUB) {
              const i64 i = aci[k];
              int32_t b = prp[i];
              const int32_t b1 = prp[i + 1];
              while (b < b1 && pci[b] != (int32_t)I) ++b;
              if (b == b1) continue;
              const double wI = pw[b];
              const unsigned fi = gal_alive<D>(fdead, i);
              const int32_t end = arp[i + 1];
              int32_t lo = arp[i], hi = end;
              while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                if (aci[mid] < j) lo = mid + 1; else hi = mid;
              }
              if (lo == end || aci[lo] != j) continue;
#pragma unroll
              for (int q = 0; q < DD; ++q)
                if (((fi >> (q / D)) & 1u) && ((fj >> (q % D)) & 1u)) acc[q] = fma(wI * av[(i64)lo * DD + q], wJ, acc[q]);
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < DD; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
          if (lane == 0)
#pragma unroll
            for (int q = 0; q < DD; ++q)
              cv[(i64)e * DD + q] = J == (int32_t)I && q % (D + 1) == 0 && cdead[I * D + q / D] ? 1.0 : acc[q];
        }
      }
  }
}

// One CTA per coarse row I.  GB300 runs ~2 FP64 lane operations per clock and
// SM, so the work is arranged for few of them: S_j = sum_i w_iI A_ij over the
// row's fine rows i (a thread per block; the threads of one i add to different
// columns, a CTA barrier separates the i's), then one thread per block of the
// row gathers sum_j S_j w_jJ over the fine rows j of R's row J.  Summing every
// w_iI A_ij w_jJ into the row took 12 times the operations and a search of the
// row per term: 33^3, all levels, 19.0 ms per update.
template <int D>
__global__ void __launch_bounds__(gal_threads<D>()) gal_values_kernel(
    i64 nc, const int32_t* __restrict__ rrp, const int32_t* __restrict__ rent, const u64* __restrict__ rkeys,
    const int32_t* __restrict__ prp, const int32_t* __restrict__ pci, const double* __restrict__ pw,
    const int32_t* __restrict__ arp, const int32_t* __restrict__ aci, const double* __restrict__ av,
    const uint8_t* __restrict__ fdead, const int32_t* __restrict__ crp, const int32_t* __restrict__ cci,
    double* __restrict__ cv, uint8_t* __restrict__ cdead, uint8_t* __restrict__ wide, int32_t* __restrict__ any_wide) {
  constexpr int DD = D * D, SLOTS = gal_slots<D>(), T = gal_threads<D>(), EMPTY = -1;
  extern __shared__ __align__(16) unsigned char gal_mem[];
  double* S = reinterpret_cast<double*>(gal_mem);                       // [SLOTS][DD]
  int32_t* key = reinterpret_cast<int32_t*>(gal_mem + SLOTS * DD * 8);  // [SLOTS]
  __shared__ int taken;
  const int tid = threadIdx.x;
  for (i64 I = blockIdx.x; I < nc; I += gridDim.x) {
    __syncthreads();
    for (int q = tid; q < SLOTS; q += T) key[q] = EMPTY;
    if (tid == 0) taken = 0;
    __syncthreads();
    const int32_t t0 = rrp[I], t1 = rrp[I + 1], c0 = crp[I], c1 = crp[I + 1];
    unsigned alive = 0;
    bool full = false;
    // the fine row t, and the row of the next t in flight
    int32_t in = 0, kn0 = 0, kn1 = 0;
    double wn = 0.0;
    auto fetch_row = [&](int32_t t) {
      if (t >= t1) return;
      in = (int32_t)(rkeys[t] & 0xffffffffull);
      wn = pw[rent[t]];
      kn0 = arp[in];
      kn1 = arp[in + 1];
    };
    fetch_row(t0);
    for (int32_t t = t0; t < t1 && !full; ++t) {
      const i64 i = in;
      const double wI = wn;
      const int32_t k0 = kn0, k1 = kn1;
      fetch_row(t + 1);
      if (k1 - k0 > SLOTS - SLOTS / 4) {  // one fine row with more columns than the table takes
        full = true;
        break;
      }
      const unsigned fi = gal_alive<D>(fdead, i);
      alive |= fi;
      bool over = false;
      for (int32_t k = k0 + tid; k < k1; k += T) {
        const int32_t j = aci[k];
        double B[DD];
#pragma unroll
        for (int q = 0; q < DD; ++q) B[q] = ((fi >> (q / D)) & 1u) ? av[(i64)k * DD + q] : 0.0;
        unsigned s = gal_hash(j, SLOTS);
        bool fresh = false, found = false;
        for (int probe = 0; probe < SLOTS && !found; ++probe) {
          const int32_t old = atomicCAS(key + s, EMPTY, j);
          fresh = old == EMPTY;
          found = fresh || old == j;
          if (!found) s = (s + 1) & (SLOTS - 1);
        }
        if (fresh && atomicAdd(&taken, 1) >= SLOTS - SLOTS / 4) over = true;
        if (!found) {
          over = true;
          continue;
        }
        double* o = S + s * DD;
#pragma unroll
        for (int q = 0; q < DD; ++q) o[q] = fresh ? wI * B[q] : fma(wI, B[q], o[q]);
      }
      full = __syncthreads_or(over);
    }
    if (full) {
      unsigned mine = 0;
      for (int32_t t = t0 + tid; t < t1; t += T) mine |= gal_alive<D>(fdead, (i64)(rkeys[t] & 0xffffffffull));
#pragma unroll
      for (int r = 0; r < D; ++r) alive |= __syncthreads_or((mine >> r) & 1u) ? 1u << r : 0u;
    } else {
      for (int32_t e = c0 + tid; e < c1; e += T) {
        const int32_t J = cci[e];
        double acc[DD];
#pragma unroll
        for (int q = 0; q < DD; ++q) acc[q] = 0.0;
        const int32_t u0 = rrp[J], u1 = rrp[J + 1];
        for (int32_t u = u0; u < u1; u += 4) {
          int32_t j[4];
          double w[4];
          unsigned f[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            j[v] = u + v < u1 ? (int32_t)(rkeys[u + v] & 0xffffffffull) : EMPTY;
            w[v] = u + v < u1 ? pw[rent[u + v]] : 0.0;
          }
#pragma unroll
          for (int v = 0; v < 4; ++v) f[v] = j[v] >= 0 ? gal_alive<D>(fdead, j[v]) : 0u;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            if (f[v] == 0u) continue;
            unsigned s = gal_hash(j[v], SLOTS);
            while (key[s] != EMPTY && key[s] != j[v]) s = (s + 1) & (SLOTS - 1);
            if (key[s] == EMPTY) continue;  // the row does not reach column j
            const double* o = S + s * DD;
#pragma unroll
            for (int q = 0; q < DD; ++q)
              if ((f[v] >> (q % D)) & 1u) acc[q] = fma(o[q], w[v], acc[q]);
          }
        }
#pragma unroll
        for (int q = 0; q < DD; ++q) cv[(i64)e * DD + q] = acc[q];
      }
    }
    __syncthreads();
    if (tid == D) {
      wide[I] = full ? 1 : 0;
      if (full) *any_wide = 1;
    }
    // dead coarse dofs -> identity rows (their masked column of P is empty)
    if (tid < D) {
      int32_t lo = c0, hi = c1;
      while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (cci[mid] < (int32_t)I) lo = mid + 1; else hi = mid;
      }
      const bool al = (alive >> tid) & 1u;
      cdead[I * D + tid] = al ? 0 : 1;
      if (!al) cv[(i64)lo * DD + tid * D + tid] = 1.0;
    }
  }
}

void setup_galerkin(Ctx& c, int l) {
  cudaStream_t s = c.stream;
  const int d = c.dim;
  CanonLevel& f = c.C[l];
  CanonLevel& g = c.C[l + 1];
  // ---- symbolic
  DevBuf<long long> cnt;
  cnt.alloc(f.nv + 1, s);
  cnt.zero();
  gal_count_kernel<<<grid_for(f.nv, 256), 256, 0, s>>>(f.rp.get(), f.ci.get(), f.prp.get(), f.pci.get(), f.nv,
                                                        cnt.get());
  check_launch("gal_count");
  scan_exclusive_i64((const i64*)cnt.get(), (i64*)cnt.get(), f.nv + 1, s);
  const i64 m = fetch(cnt.get() + f.nv, s);
  DevBuf<u64> keys;
  keys.alloc(m + g.nv, s);
  gal_pairs_kernel<<<grid_for(f.nv, 128), 128, 0, s>>>(f.rp.get(), f.ci.get(), f.prp.get(), f.pci.get(), f.nv,
                                                        cnt.get(), keys.get());
  check_launch("gal_pairs");
  diag_pairs_kernel<<<grid_for(g.nv, 256), 256, 0, s>>>(g.nv, keys.get() + m);
  check_launch("diag_pairs");
  const int cb = bits_for((u64)g.nv);
  radix_sort(keys.get(), nullptr, m + g.nv, {{0, cb}, {32, 32 + cb}}, s);
  g.nnzb = unique_sorted(keys.get(), m + g.nv, s);
  VASMG_CHECK(g.nnzb < (i64)INT32_MAX, VASMG_ERR_UNSUPPORTED, "too many blocks for 32-bit indices");
  g.rp.alloc(g.nv + 1, s);
  g.ci.alloc(g.nnzb, s);
  rowptr_from_pairs(keys.get(), g.nnzb, g.nv, g.rp.get(), s);
  low32_i_kernel<<<grid_for(g.nnzb, 256), 256, 0, s>>>(keys.get(), g.nnzb, g.ci.get());
  check_launch("low32");
  keys.release();
  // ---- R = P^T as (coarse row, fine index) sorted pairs, kept on the fine level
  f.r_keys.alloc(f.pnnz, s);
  f.r_ent.alloc(f.pnnz, s);
  transpose_keys_kernel<<<grid_for(f.nv, 256), 256, 0, s>>>(f.prp.get(), f.pci.get(), f.nv, f.r_keys.get(),
                                                             f.r_ent.get());
  check_launch("transpose_keys");
  // the fine rows (low word) come in ascending order
  radix_sort(f.r_keys.get(), f.r_ent.get(), f.pnnz, {{32, 32 + cb}}, s);
  f.r_rp.alloc(g.nv + 1, s);
  rowptr_from_pairs(f.r_keys.get(), f.pnnz, g.nv, f.r_rp.get(), s);
  galerkin_values(c, l);
}

// ---- numeric: A_{l+1} = P^T A_l P on the pattern built above (eq. (Ac)),
// with dead-dof masks; also run again when A_l's values change.
void galerkin_values(Ctx& c, int l) {
  cudaStream_t s = c.stream;
  const int d = c.dim;
  CanonLevel& f = c.C[l];
  CanonLevel& g = c.C[l + 1];
  if (g.v.n != g.nnzb * d * d) g.v.alloc(g.nnzb * d * d, s);
  if (g.dead.n != g.nv * d) g.dead.alloc(g.nv * d, s);
  if (g.wide.n != g.nv) g.wide.alloc(g.nv, s);
  if (!c.any_wide.n) {
    c.any_wide.alloc(ANY_WIDE_SLOTS, s);
    c.any_wide.zero();
  }
  const int slot = std::min(l, ANY_WIDE_SLOTS - 1);
  int32_t* any = c.any_wide.get() + slot;
  auto launch = [&](auto kern, auto wide, int threads, int smem) {
    VASMG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    kern<<<grid_for(g.nv, 1), threads, smem, s>>>(g.nv, f.r_rp.get(), f.r_ent.get(), f.r_keys.get(), f.prp.get(),
                                                  f.pci.get(), f.pw.get(), f.rp.get(), f.ci.get(), f.v.get(),
                                                  f.dead.get(), g.rp.get(), g.ci.get(), g.v.get(), g.dead.get(),
                                                  g.wide.get(), any);
    check_launch("gal_values");
    // which levels have such rows is known once the setup is through (they follow
    // from the structure)
    if (!c.any_wide_host.empty() && c.any_wide_host[slot] == 0) return;
    wide<<<dim3(grid_for(g.nv, 1, 512), 8), 256, 0, s>>>(
        g.nv, g.wide.get(), any, f.r_rp.get(), f.r_ent.get(), f.r_keys.get(), f.prp.get(), f.pci.get(), f.pw.get(),
        f.rp.get(), f.ci.get(), f.v.get(), f.dead.get(), g.rp.get(), g.ci.get(), g.dead.get(), g.v.get());
    check_launch("gal_wide");
  };
  if (d == 2) launch(gal_values_kernel<2>, gal_wide_kernel<2>, gal_threads<2>(), gal_smem<2>());
  else launch(gal_values_kernel<3>, gal_wide_kernel<3>, gal_threads<3>(), gal_smem<3>());
}

}  // namespace vasmg
