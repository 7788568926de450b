// k_sym.cu -- Best Hit rows of the symmetric all-pairs form.
//
// The similarity J is symmetric (Eq. (5)), so S_ji is the transpose of S_ij
// and the all-against-all comparison needs each unordered genome pair walked
// once.  In the symmetric form (QuerySet::symbest) query a of genome i walks
// only the targets in genomes j > i and emits its forward Best Hits there
// (Eq. (8)); while it does so, every candidate b in such a genome j keeps the
// best ratio it reaches over the genes of G_i, with the gene that reaches it,
// and a list of exact ties.  That maximum over a column of S_ij gives the Best
// Hits of b in G_i (the reverse direction: Algorithm 3's column maximum).
//
// Row b of the result is then its Best Hits in the genomes before its own
// (the stored maxima and the ties that equal them, ascending) followed by its
// forward Best Hits in the genomes after its own -- ascending overall, since
// genes are numbered genome by genome.
//
// Listed pairs take the same form with a mask of target genomes, and a batch,
// whose segments are two genomes each, with one maximum a gene.
#include <algorithm>

#include "pd_internal.cuh"

namespace pdg {
namespace {

__device__ __forceinline__ void unpack(unsigned long long w, uint32_t* s, uint32_t* den, uint32_t* a) {
  *s = (uint32_t)(w >> 48);
  *den = (uint32_t)(w >> 31) & 0x1FFFFu;
  *a = (uint32_t)w & 0x7FFFFFFFu;
}

// Maxima a gene may have, and the one that gene a's genome keeps.
__device__ __forceinline__ uint32_t n_columns(const SymRows& R, uint32_t b) {
  return R.two_genomes ? 1u : R.gene_genome[b];
}
__device__ __forceinline__ size_t column_of(const SymRows& R, uint32_t a) {
  return R.two_genomes ? 0u : R.gene_genome[a];
}

// One thread per gene: stored maxima of the genomes before its own (the
// maxima are genome-major, so neighbouring threads read neighbouring words),
// and the length of its row (tiecnt null: no ties).
__global__ void __launch_bounds__(256) k_sym_count(SymRows R, const uint32_t* __restrict__ tiecnt,
                                                   uint32_t* __restrict__ stored, uint32_t* __restrict__ total) {
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < R.n_genes; b += gridDim.x * blockDim.x) {
    const uint32_t gb = n_columns(R, b);
    uint32_t n = 0;
    for (uint32_t g = 0; g < gb; ++g) n += R.symbest[(size_t)g * R.n_genes + b] != 0ull ? 1u : 0u;
    stored[b] = n;
    total[b] = n + (tiecnt ? tiecnt[b] : 0u) + R.fwd_len[b];
  }
}

// Is (b, a) new to the set?  Open addressing over `keys` (a power of two at
// least twice the ties, all-ones = empty), so a probe always ends.
__device__ __forceinline__ bool first_insert(unsigned long long* keys, unsigned long long mask,
                                             unsigned long long key) {
  unsigned long long h = (key * 0x9E3779B97F4A7C15ull) & mask;
  for (unsigned long long probe = 0; probe <= mask; ++probe) {
    const unsigned long long prev = atomicCAS(&keys[h], ~0ull, key);
    if (prev == ~0ull) return true;
    if (prev == key) return false;
    h = (h + 1) & mask;
  }
  return false;
}

// One thread per tie (b << 32 | a, s): valid when its ratio equals the final
// stored maximum of (b, genome of a), it is not the stored pair itself, and
// it is the first record of the pair (a query that a tier hands to the next
// after its Best Hit passes records its ties again).  Genes with valid ties are
// listed.
__global__ void k_sym_ties(SymRows R, uint32_t* __restrict__ tiecnt, uint8_t* __restrict__ tie_ok) {
  for (unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; t < R.n_ties;
       t += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long r = R.tie_rec[2 * t];
    const uint32_t b = (uint32_t)(r >> 32), a = (uint32_t)r, s = (uint32_t)R.tie_rec[2 * t + 1];
    const unsigned long long w = R.symbest[column_of(R, a) * R.n_genes + b];
    uint32_t ms, md, ma;
    unpack(w, &ms, &md, &ma);
    const bool ok = w != 0ull && ma != a && ratio_equal(s, R.La[a] + R.La[b] - s, ms, md) &&
                    first_insert(R.tie_set, R.tie_set_mask, r);
    tie_ok[t] = ok ? 1 : 0;
    if (ok && atomicAdd(&tiecnt[b], 1u) == 0u) R.tie_gene[atomicAdd(R.n_tie_genes, 1u)] = b;
  }
}

// One thread per gene: the stored maxima in genome order.
__global__ void __launch_bounds__(256)
    k_sym_write_rev(SymRows R, const unsigned long long* __restrict__ row_ptr, uint32_t* __restrict__ out_b,
                    uint32_t* __restrict__ out_s) {
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < R.n_genes; b += gridDim.x * blockDim.x) {
    const uint32_t gb = n_columns(R, b);
    unsigned long long at = row_ptr[b];
    for (uint32_t g = 0; g < gb; ++g) {
      const unsigned long long w = R.symbest[(size_t)g * R.n_genes + b];
      if (w == 0ull) continue;
      uint32_t s, den, a;
      unpack(w, &s, &den, &a);
      out_b[at] = a;
      out_s[at] = s;
      ++at;
    }
  }
}

// The same through shared memory, for datasets of at most kRevTileGenomes
// genomes: a block reads the maxima of 32 consecutive genes genome by genome
// (coalesced) into a tile, then one warp per gene writes its reverse part and,
// if asked to, its forward part (coalesced), leaving room for its ties between.  Genes
// are numbered genome by genome, so the tile's last gene has the largest genome
// of the 32.
constexpr uint32_t kRevTileGenomes = 372;  // 372 x 33 x 8 bytes < 96 KB of shared memory
// Up to this many genomes (16 KB of tile) a launch writes the forward parts too
// (50 genomes: 43 against 56 us); past it the tile leaves few blocks per SM to
// copy with, and they get a launch of their own (200: 0.83 against 1.07 ms).
constexpr uint32_t kRowTileGenomes = 62;
__global__ void __launch_bounds__(256)
    k_sym_write_tile(SymRows R, const uint32_t* __restrict__ tiecnt, const unsigned long long* __restrict__ row_ptr,
                     int forward, uint32_t* __restrict__ out_b, uint32_t* __restrict__ out_s) {
  extern __shared__ unsigned long long tile[];  // [genome][33]
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  for (uint32_t b0 = blockIdx.x * 32u; b0 < R.n_genes; b0 += gridDim.x * 32u) {
    const uint32_t nb = min(32u, R.n_genes - b0);
    const uint32_t gmax = n_columns(R, b0 + nb - 1);
    for (uint32_t g = warp; g < gmax; g += n_warps)
      tile[g * 33u + lane] = lane < nb ? R.symbest[(size_t)g * R.n_genes + b0 + lane] : 0ull;
    __syncthreads();
    for (uint32_t j = warp; j < nb; j += n_warps) {
      const uint32_t b = b0 + j, gb = n_columns(R, b);
      unsigned long long at = row_ptr[b];
      for (uint32_t g0 = 0; g0 < gb; g0 += 32) {
        const uint32_t g = g0 + lane;
        const unsigned long long w = g < gb ? tile[g * 33u + j] : 0ull;
        const uint32_t m = __ballot_sync(0xffffffffu, w != 0ull);
        if (w != 0ull) {
          uint32_t s, den, a;
          unpack(w, &s, &den, &a);
          const unsigned long long x = at + __popc(m & ((1u << lane) - 1u));
          out_b[x] = a;
          out_s[x] = s;
        }
        at += __popc(m);
      }
      if (!forward) continue;
      if (tiecnt) at += tiecnt[b];
      const unsigned long long fo = R.fwd_off[b];
      const uint32_t fl = R.fwd_len[b];
      for (uint32_t e = lane; e < fl; e += 32) {
        out_b[at + e] = R.fwd_b[fo + e];
        out_s[at + e] = R.fwd_s[fo + e];
      }
    }
    __syncthreads();
  }
}

// One warp per gene: the forward part, after the stored maxima and room for
// the gene's ties (tiecnt null: none).
__global__ void __launch_bounds__(256)
    k_sym_write(SymRows R, const uint32_t* __restrict__ stored, const uint32_t* __restrict__ tiecnt,
                const unsigned long long* __restrict__ row_ptr, uint32_t* __restrict__ out_b,
                uint32_t* __restrict__ out_s) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < R.n_genes; b += warps) {
    const unsigned long long base = row_ptr[b];
    const unsigned long long fwd = base + stored[b] + (tiecnt ? tiecnt[b] : 0u);
    const unsigned long long fo = R.fwd_off[b];
    const uint32_t fl = R.fwd_len[b];
    for (uint32_t e = lane; e < fl; e += 32) {
      out_b[fwd + e] = R.fwd_b[fo + e];
      out_s[fwd + e] = R.fwd_s[fo + e];
    }
  }
}

// Valid ties go after their gene's stored maxima.
__global__ void k_sym_put_ties(SymRows R, const uint8_t* __restrict__ tie_ok, const uint32_t* __restrict__ stored,
                               const unsigned long long* __restrict__ row_ptr, uint32_t* __restrict__ tie_fill,
                               uint32_t* __restrict__ out_b, uint32_t* __restrict__ out_s) {
  for (unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; t < R.n_ties;
       t += (unsigned long long)gridDim.x * blockDim.x) {
    if (!tie_ok[t]) continue;
    const unsigned long long r = R.tie_rec[2 * t];
    const uint32_t b = (uint32_t)(r >> 32), a = (uint32_t)r;
    const unsigned long long at = row_ptr[b] + stored[b] + atomicAdd(&tie_fill[b], 1u);
    out_b[at] = a;
    out_s[at] = (uint32_t)R.tie_rec[2 * t + 1];
  }
}

// One warp per gene with ties: its reverse part sorted by gene id.  The stored
// maxima are ascending already, so an entry's place is its index among them
// plus the ties below it, a tie's the stored below it (bisection) plus the ties
// below it.  The part is read before it is written, at most kTieLanes entries a
// lane; longer parts are left to k_sym_sort_long.
constexpr uint32_t kTieLanes = 16;
__global__ void __launch_bounds__(256)
    k_sym_sort_ties(SymRows R, const uint32_t* __restrict__ stored, const uint32_t* __restrict__ tiecnt,
                    const unsigned long long* __restrict__ row_ptr, uint32_t* __restrict__ out_b,
                    uint32_t* __restrict__ out_s) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t n_listed = *R.n_tie_genes;
  for (uint32_t x0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; x0 < n_listed; x0 += warps) {
    const uint32_t b = R.tie_gene[x0];
    const uint32_t ns = stored[b], nt = tiecnt[b], n = ns + nt;
    uint32_t* kb = out_b + row_ptr[b];
    uint32_t* ks = out_s + row_ptr[b];
    if (n <= 32u * kTieLanes) {
      uint32_t x[kTieLanes], y[kTieLanes], at[kTieLanes];
#pragma unroll
      for (uint32_t j = 0; j < kTieLanes; ++j) {
        const uint32_t i = j * 32u + lane;
        x[j] = y[j] = at[j] = 0;
        if (i < n) {
          x[j] = kb[i];
          y[j] = ks[i];
          uint32_t rank = i;  // a stored entry's index among the stored
          if (i >= ns) {
            uint32_t lo = 0, hi = ns;
            while (lo < hi) {
              const uint32_t mid = (lo + hi) >> 1;
              if (kb[mid] < x[j]) lo = mid + 1; else hi = mid;
            }
            rank = lo;
          }
          for (uint32_t t = 0; t < nt; ++t) rank += kb[ns + t] < x[j] ? 1u : 0u;
          at[j] = rank;
        }
      }
      __syncwarp();
#pragma unroll
      for (uint32_t j = 0; j < kTieLanes; ++j)
        if (j * 32u + lane < n) {
          kb[at[j]] = x[j];
          ks[at[j]] = y[j];
        }
    }
    __syncwarp();
  }
}

// One block per gene whose reverse part is longer than a warp takes: a bitonic
// network in the form whose exchanges all put the smaller entry at the lower
// place, so that the entries missing to a power of two need not exist.  In
// shared memory up to kLongShared entries, else in place (2000 genomes x 20
// genes, rows of 1000: 1.7 ms, where an insertion sort by one lane took 580).
constexpr uint32_t kLongShared = 4096;
__global__ void __launch_bounds__(256)
    k_sym_sort_long(SymRows R, const uint32_t* __restrict__ stored, const uint32_t* __restrict__ tiecnt,
                    const unsigned long long* __restrict__ row_ptr, uint32_t* __restrict__ out_b,
                    uint32_t* __restrict__ out_s) {
  __shared__ unsigned long long sh[kLongShared];
  __shared__ uint32_t longs;  // of the 32 genes, those with long rows
  const uint32_t n_listed = *R.n_tie_genes;
  auto network = [&](uint32_t n, auto exchange) {
    for (uint32_t size = 2; size / 2 < n; size <<= 1)
      for (uint32_t stride = size / 2; stride > 0; stride >>= 1) {
        for (uint32_t i = threadIdx.x;; i += blockDim.x) {
          const uint32_t lo = 2 * i - (i & (stride - 1));
          if (lo >= n) break;
          const uint32_t hi = stride == size / 2 ? lo ^ (size - 1) : lo + stride;
          if (hi < n) exchange(lo, hi);
        }
        __syncthreads();
      }
  };
  // few genes' rows are long: a block looks at 32 at a time
  for (uint32_t x0 = blockIdx.x * 32u; x0 < n_listed; x0 += gridDim.x * 32u) {
    if (threadIdx.x < 32u) {
      const uint32_t x = x0 + threadIdx.x, b = x < n_listed ? R.tie_gene[x] : 0u;
      const uint32_t m = __ballot_sync(0xffffffffu, x < n_listed && stored[b] + tiecnt[b] > 32u * kTieLanes);
      if (threadIdx.x == 0) longs = m;
    }
    __syncthreads();
    for (uint32_t left = longs; left; left &= left - 1u) {
      const uint32_t b = R.tie_gene[x0 + (uint32_t)__ffs((int)left) - 1u], n = stored[b] + tiecnt[b];
      uint32_t* kb = out_b + row_ptr[b];
      uint32_t* ks = out_s + row_ptr[b];
      if (n > kLongShared) {
        network(n, [&](uint32_t lo, uint32_t hi) {
          const uint32_t p = kb[lo], q = kb[hi];
          if (p > q) {
            const uint32_t s = ks[lo];
            kb[lo] = q;
            kb[hi] = p;
            ks[lo] = ks[hi];
            ks[hi] = s;
          }
        });
        continue;
      }
      for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) sh[i] = (unsigned long long)kb[i] << 32 | ks[i];
      __syncthreads();
      network(n, [&](uint32_t lo, uint32_t hi) {
        const unsigned long long p = sh[lo], q = sh[hi];
        if (p > q) {
          sh[lo] = q;
          sh[hi] = p;
        }
      });
      for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        kb[i] = (uint32_t)(sh[i] >> 32);
        ks[i] = (uint32_t)sh[i];
      }
      __syncthreads();
    }
    __syncthreads();
  }
}

// Bidirectional Best Hits of the symmetric form, one warp per forward row:
// a forward Best Hit a -> b (b in a later genome) is a BBH exactly when its
// ratio equals b's maximum over a's genome (Eq. (9): a is then among the Best
// Hits of b in G_i, ties included).  Pass 1 flags and counts, pass 2 writes
// at the row's scanned start, so pairs come out ascending.
__global__ void __launch_bounds__(256) k_sym_bbh_count(SymRows R, uint8_t* __restrict__ flag,
                                                       uint32_t* __restrict__ cnt) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t a = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; a < R.n_genes; a += warps) {
    const uint32_t La = R.La[a];
    const size_t col = column_of(R, a);
    const unsigned long long fo = R.fwd_off[a];
    const uint32_t fl = R.fwd_len[a];
    uint32_t n = 0;
    for (uint32_t e = lane; e < fl; e += 32) {
      const uint32_t b = R.fwd_b[fo + e], sv = R.fwd_s[fo + e];
      const unsigned long long w = R.symbest[col * R.n_genes + b];
      const bool f = ratio_equal(sv, La + R.La[b] - sv, (uint32_t)(w >> 48), (uint32_t)(w >> 31) & 0x1FFFFu);
      flag[fo + e] = f ? 1 : 0;
      n += f ? 1u : 0u;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0) cnt[a] = n;
  }
}

__global__ void __launch_bounds__(256) k_sym_bbh_write(SymRows R, const uint8_t* __restrict__ flag,
                                                       const uint32_t* __restrict__ start, int32_t* __restrict__ pa,
                                                       int32_t* __restrict__ pb) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t a = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; a < R.n_genes; a += warps) {
    const unsigned long long fo = R.fwd_off[a];
    const uint32_t fl = R.fwd_len[a];
    uint32_t pos = start[a];
    for (uint32_t e0 = 0; e0 < fl; e0 += 32) {
      const uint32_t e = e0 + lane;
      const bool f = e < fl && flag[fo + e];
      const uint32_t m = __ballot_sync(0xffffffffu, f);
      if (f) {
        const uint32_t at = pos + __popc(m & ((1u << lane) - 1u));
        pa[at] = (int32_t)a;
        pb[at] = (int32_t)R.fwd_b[fo + e];
      }
      pos += __popc(m);
    }
  }
}

unsigned grid_of(uint64_t items, unsigned per_block, unsigned cap) {
  uint64_t g = (items + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (unsigned)g;
}

}  // namespace

cudaError_t run_sym_count(Launcher* L, const SymRows& R, uint32_t* stored, uint32_t* tiecnt, uint8_t* tie_ok,
                          uint32_t* total, cudaStream_t s) {
  cudaError_t e;
  if (R.n_ties) {
    if ((e = launch_begin(L, "sym_ties")) != cudaSuccess) return e;
    k_sym_ties<<<grid_of(R.n_ties, 256, 152u * 16u), 256, 0, s>>>(R, tiecnt, tie_ok);
    if ((e = launch_end(L, "sym_ties")) != cudaSuccess) return e;
  }
  if ((e = launch_begin(L, "sym_count")) != cudaSuccess) return e;
  k_sym_count<<<grid_of((uint64_t)R.n_genes, 256, 152u * 16u), 256, 0, s>>>(R, R.n_ties ? tiecnt : nullptr, stored,
                                                                            total);
  return launch_end(L, "sym_count");
}

cudaError_t run_sym_write(Launcher* L, const SymRows& R, const uint32_t* stored, const uint32_t* tiecnt,
                          const uint8_t* tie_ok, const unsigned long long* row_ptr, uint32_t* tie_fill,
                          uint32_t* out_b, uint32_t* out_s, cudaStream_t s) {
  cudaError_t e;
  const uint32_t* ties = R.n_ties ? tiecnt : nullptr;
  const bool whole = R.n_genomes <= kRowTileGenomes;
  if ((e = launch_begin(L, "sym_write_rev")) != cudaSuccess) return e;
  if (R.n_genomes <= kRevTileGenomes) {
    const size_t smem = (size_t)R.n_genomes * 33u * sizeof(unsigned long long);
    // the largest, whatever this launch takes: the attribute is every thread's
    if ((e = cudaFuncSetAttribute(k_sym_write_tile, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(kRevTileGenomes * 33u * sizeof(unsigned long long)))) != cudaSuccess)
      return e;
    k_sym_write_tile<<<grid_of((uint64_t)R.n_genes, 32, 152u * 8u), 256, smem, s>>>(R, ties, row_ptr, whole, out_b,
                                                                                    out_s);
  } else {
    k_sym_write_rev<<<grid_of((uint64_t)R.n_genes, 256, 152u * 16u), 256, 0, s>>>(R, row_ptr, out_b, out_s);
  }
  if ((e = launch_end(L, "sym_write_rev")) != cudaSuccess) return e;
  if (!whole) {
    if ((e = launch_begin(L, "sym_write")) != cudaSuccess) return e;
    k_sym_write<<<grid_of((uint64_t)R.n_genes * 32, 256, 152u * 16u), 256, 0, s>>>(R, stored, ties, row_ptr, out_b,
                                                                                   out_s);
    if ((e = launch_end(L, "sym_write")) != cudaSuccess) return e;
  }
  if (R.n_ties == 0) return cudaSuccess;
  if ((e = launch_begin(L, "sym_put_ties")) != cudaSuccess) return e;
  k_sym_put_ties<<<grid_of(R.n_ties, 256, 152u * 16u), 256, 0, s>>>(R, tie_ok, stored, row_ptr, tie_fill, out_b,
                                                                      out_s);
  if ((e = launch_end(L, "sym_put_ties")) != cudaSuccess) return e;
  if ((e = launch_begin(L, "sym_sort_ties")) != cudaSuccess) return e;
  k_sym_sort_ties<<<grid_of(std::min<unsigned long long>(R.n_ties, R.n_genes) * 32, 256, 152u * 8u), 256, 0, s>>>(
      R, stored, tiecnt, row_ptr, out_b, out_s);
  if ((e = launch_end(L, "sym_sort_ties")) != cudaSuccess) return e;
  // a gene's reverse part holds a maximum for each other genome, and ties
  if (R.n_genomes + R.n_ties <= 32u * kTieLanes) return cudaSuccess;
  if ((e = launch_begin(L, "sym_sort_long")) != cudaSuccess) return e;
  k_sym_sort_long<<<grid_of(std::min<unsigned long long>(R.n_ties, R.n_genes), 32, 152u * 6u), 256, 0, s>>>(
      R, stored, tiecnt, row_ptr, out_b, out_s);
  return launch_end(L, "sym_sort_long");
}

cudaError_t run_sym_bbh_count(Launcher* L, const SymRows& R, uint8_t* flag, uint32_t* cnt, uint32_t* start,
                              void* scan_tmp, cudaStream_t s) {
  cudaError_t e = launch_begin(L, "sym_bbh_count");
  if (e != cudaSuccess) return e;
  k_sym_bbh_count<<<grid_of((uint64_t)R.n_genes * 32, 256, 152u * 16u), 256, 0, s>>>(R, flag, cnt);
  if ((e = launch_end(L, "sym_bbh_count")) != cudaSuccess) return e;
  return scan_u32(L, cnt, R.n_genes, start, scan_tmp, s);
}

cudaError_t run_sym_bbh_write(Launcher* L, const SymRows& R, const uint8_t* flag, const uint32_t* start, int32_t* pa,
                              int32_t* pb, cudaStream_t s) {
  cudaError_t e = launch_begin(L, "sym_bbh_write");
  if (e != cudaSuccess) return e;
  k_sym_bbh_write<<<grid_of((uint64_t)R.n_genes * 32, 256, 152u * 16u), 256, 0, s>>>(R, flag, start, pa, pb);
  return launch_end(L, "sym_bbh_write");
}

}  // namespace pdg
