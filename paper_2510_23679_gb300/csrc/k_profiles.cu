// k_profiles.cu -- k-mer profiles on the device: vectors of genes from outside
// a dataset, the dictionary they are looked up in, the query order and the
// export of the profiles.  (k_index.cu builds the profiles of a dataset.)
//
//   dictionary     one bit per possible code in 32-byte rank blocks (224 codes
//                  and the rank of the first): the dense id of a code is its
//                  rank among the codes present, found with one sector read.
//                  Marked from the index's sorted codes, so neighbouring
//                  threads mark neighbouring bits.
//   mv_build       per outside gene: ids of its windows (those the dictionary
//                  holds) counted in a shared-memory hash table, compacted into
//                  vector entries with their posting ranges (Eqs. (2)-(3)).
//   order          queries ordered by length bucket (at least 1024, 512, 256
//                  windows, then the rest: longest first, so the persistent
//                  sum-min launch ends on short queries) and within a bucket by
//                  a hash of the min-hash: genes that share their minimum hashed
//                  k-mer (likely homologs) run together and share posting
//                  lists in L2.
#include "pd_internal.cuh"

namespace pdg {
namespace {

constexpr int kMvThreads = 256;
constexpr int kMvLongThreads = 1024;
constexpr uint32_t kMvSmallCap = 2048;  // table slots of the shared-memory multiplicity-vector build
constexpr uint32_t kMvMidCap = 16384;   // ... of its 1024-thread variant (one block per SM)

// ------------------------------------------------------------ dictionary
__global__ void k_dict_mark(const uint32_t* __restrict__ code_lo, const uint8_t* __restrict__ code_hi, uint64_t n,
                            uint32_t* __restrict__ dict) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    unsigned long long blk;
    uint32_t w, bit;
    dict_locate(code_at(code_lo, code_hi, i), &blk, &w, &bit);
    atomicOr(&dict[blk * 8 + w], 1u << bit);
  }
}

// ------------------------------------------------------------ mv_build
// Multiplicity vector of outside gene g (Eqs. (2)-(3)): the dense ids of its
// windows are counted in an open-addressing table of 64-bit slots (id << 32 |
// count) of `cap` slots (a power of two, at least 1.5 x La), then the occupied
// slots are compacted into the gene's window range, in table order (nothing
// downstream depends on the order).  Windows whose k-mer the dictionary lacks
// are left out.  Called by every thread of the block.
__device__ __forceinline__ void mv_build_one(uint32_t g, unsigned long long* table, uint32_t cap,
                                             const uint8_t* __restrict__ lut, uint32_t* warp_tmp,
                                             const uint8_t* __restrict__ res, const int64_t* __restrict__ gene_ptr,
                                             const uint32_t* __restrict__ win_off, int k,
                                             const uint32_t* __restrict__ dict, const MvOut& M) {
  constexpr unsigned long long kFree = ~0ull;
  const uint32_t off = win_off[g];
  const uint32_t La = win_off[g + 1] - off;
  const uint8_t* s = res + gene_ptr[g];
  for (uint32_t h = threadIdx.x; h < cap; h += blockDim.x) table[h] = kFree;
  __syncthreads();
  for (uint32_t p = threadIdx.x; p < La; p += blockDim.x) {
    unsigned long long code = 0;
    for (int t = 0; t < k; ++t) {
      const uint32_t c = lut[s[p + t]];
      code = code * (unsigned long long)M.alpha + (c < (uint32_t)M.alpha ? c : 0u);
    }
    if (!dict_has(dict, code)) continue;
    const uint32_t id = dict_rank(dict, code);
    uint32_t h = mix32(id) & (cap - 1u);
    uint32_t probe = 0;
    for (; probe < cap; ++probe) {  // a free slot always exists: cap > La >= distinct ids
      const unsigned long long cur = *((volatile unsigned long long*)&table[h]);
      if (cur != kFree && (uint32_t)(cur >> 32) == id) {
        atomicAdd(&table[h], 1ull);
        break;
      }
      if (cur == kFree) {
        const unsigned long long prev = atomicCAS(&table[h], kFree, ((unsigned long long)id << 32) | 1ull);
        if (prev == kFree) break;
        if ((uint32_t)(prev >> 32) == id) {
          atomicAdd(&table[h], 1ull);
          break;
        }
      }
      h = (h + 1u) & (cap - 1u);
    }
    if (probe == cap) raise_error(M.err, PD_ERR_INTERNAL, g);  // unreachable by the bound above
  }
  __syncthreads();
  // compaction of the occupied slots (interleaved: slot = i * blockDim + tid)
  uint32_t mine = 0;
  for (uint32_t h = threadIdx.x; h < cap; h += blockDim.x) mine += table[h] != kFree ? 1u : 0u;
  uint32_t E;
  uint32_t pos = block_exclusive_scan(mine, warp_tmp, &E);
  for (uint32_t h = threadIdx.x; h < cap; h += blockDim.x) {
    const unsigned long long v = table[h];
    if (v == kFree) continue;
    const uint32_t id = (uint32_t)(v >> 32), first = M.post_ptr[id];
    M.mv[off + pos] = make_uint4(first, (uint32_t)v, M.post_ptr[id + 1] - first, 0u);
    ++pos;
  }
  if (threadIdx.x == 0) M.mv_n[g] = E;
  __syncthreads();
}

__host__ __device__ __forceinline__ uint32_t mv_table_cap(uint32_t La) {
  const uint32_t c = next_pow2(La + La / 2 + 1);
  return c < 64 ? 64 : c;
}

// Genes whose table fits `max_cap` slots of shared memory: all genes with a
// table of at most max_cap slots (list == nullptr), or the listed genes.
template <int kThreads>
__global__ void __launch_bounds__(kThreads)
    k_mv_build_smem(const uint8_t* __restrict__ res, const int64_t* __restrict__ gene_ptr,
                    const uint32_t* __restrict__ win_off, uint32_t n_genes, int k,
                    const uint32_t* __restrict__ dict, MvOut M,
                    uint32_t max_cap, const uint32_t* __restrict__ list, uint32_t n_list) {
  extern __shared__ unsigned long long table[];
  __shared__ uint8_t lut[256];
  __shared__ uint32_t warp_tmp[kThreads / 32 + 1];
  init_letter_table(lut, M.alpha);
  const uint32_t n = list ? n_list : n_genes;
  for (uint32_t x = blockIdx.x; x < n; x += gridDim.x) {
    const uint32_t g = list ? list[x] : x;
    const uint32_t cap = mv_table_cap(win_off[g + 1] - win_off[g]);
    if (cap > max_cap) continue;  // uniform over the block: built by a later launch
    mv_build_one(g, table, cap, lut, warp_tmp, res, gene_ptr, win_off, k, dict, M);
  }
}

// Genes too long for shared memory: tables in global scratch (one per gene).
__global__ void __launch_bounds__(kMvLongThreads)
    k_mv_build_long(const uint8_t* __restrict__ res, const int64_t* __restrict__ gene_ptr,
                    const uint32_t* __restrict__ win_off, int k, const uint32_t* __restrict__ dict, MvOut M,
                    const uint32_t* __restrict__ long_genes,
                    uint32_t n_long, unsigned long long* scratch, const unsigned long long* __restrict__ scratch_off) {
  __shared__ uint8_t lut[256];
  __shared__ uint32_t warp_tmp[kMvLongThreads / 32 + 1];
  init_letter_table(lut, M.alpha);
  for (uint32_t x = blockIdx.x; x < n_long; x += gridDim.x) {
    const uint32_t g = long_genes[x];
    mv_build_one(g, scratch + scratch_off[x], mv_table_cap(win_off[g + 1] - win_off[g]), lut, warp_tmp, res,
                 gene_ptr, win_off, k, dict, M);
  }
}

// ------------------------------------------------------------ query order
// Bucket of a gene: with length_buckets, two bits of length class above 14
// bits of the hashed min-hash (a min-hash itself lies near zero: hashed again
// it spreads over the buckets).
__device__ __forceinline__ uint32_t order_bucket(uint32_t minhash, uint32_t La, int length_buckets) {
  const uint32_t h = mix32(minhash);
  if (!length_buckets) return h >> 16;
  const uint32_t lb = La >= 1024u ? 0u : (La >= 512u ? 1u : (La >= 256u ? 2u : 3u));
  return (lb << 14) | (h >> 18);
}

// Also (cursor not null) the length of every gene's vector: what its cursor passed.
__global__ void k_order_count(const uint32_t* __restrict__ minhash, const uint32_t* __restrict__ La, uint32_t n_genes,
                              int length_buckets, const uint32_t* __restrict__ cursor,
                              const uint32_t* __restrict__ win_off, uint32_t* __restrict__ mv_n,
                              uint32_t* __restrict__ count) {
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n_genes; g += gridDim.x * blockDim.x) {
    atomicAdd(&count[order_bucket(minhash[g], La[g], length_buckets)], 1u);
    if (cursor) mv_n[g] = cursor[g] - win_off[g];
  }
}

__global__ void k_order_scatter(const uint32_t* __restrict__ minhash, const uint32_t* __restrict__ La,
                                uint32_t n_genes, int length_buckets, uint32_t* __restrict__ cursor,
                                uint32_t* __restrict__ order) {
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n_genes; g += gridDim.x * blockDim.x)
    order[atomicAdd(&cursor[order_bucket(minhash[g], La[g], length_buckets)], 1u)] = g;
}

// ------------------------------------------------------------ export
// Code of every dense id.
__global__ void k_export_codes(const uint32_t* __restrict__ code_lo, const uint8_t* __restrict__ code_hi, uint64_t n,
                               unsigned long long* __restrict__ codes) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    codes[i] = code_at(code_lo, code_hi, i);
}

// Export of the multiplicity vectors (inspection hook), transposed from the
// index: distinct k-mers per gene, then each gene's (code << 16 | count) keys
// in a power-of-two padded scratch region; one block sorts each region, then
// the keys are unpacked.
__global__ void k_export_mv_count(ProfilesView P, uint32_t* __restrict__ n) {
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < P.n_entries;
       e += (uint64_t)gridDim.x * blockDim.x)
    atomicAdd(&n[P.post[e] >> P.cnt_bits], 1u);
}

// A block takes kExportTile consecutive postings, however long their lists are (a
// thread a list: the call took 107 ms for 180 k genes at k = 1, now 2.3; 45 for 60 k
// at k = 2, now 7.2; at k = 6, of short lists, 12.4 and 12.2), and looks for each
// posting's id among those of its tile.
constexpr uint32_t kExportTile = 2048;

// Last id in [lo, hi) whose postings begin at or before e.
__device__ __forceinline__ uint64_t id_of_posting(const uint32_t* __restrict__ post_ptr, uint64_t lo, uint64_t hi,
                                                  uint64_t e) {
  while (hi - lo > 1) {
    const uint64_t mid = (lo + hi) >> 1;
    if (post_ptr[mid] <= e) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(256)
    k_export_mv_keys(ProfilesView P, const unsigned long long* __restrict__ pad_off, uint32_t* __restrict__ fill,
                     unsigned long long* __restrict__ pad) {
  __shared__ uint64_t id_lo, id_hi;
  const uint32_t mask = (1u << P.cnt_bits) - 1u;
  for (uint64_t e0 = (uint64_t)blockIdx.x * kExportTile; e0 < P.n_entries; e0 += (uint64_t)gridDim.x * kExportTile) {
    const uint64_t e1 = min(e0 + kExportTile, P.n_entries);
    if (threadIdx.x == 0) id_lo = id_of_posting(P.post_ptr, 0, P.n_distinct, e0);
    if (threadIdx.x == 32) id_hi = id_of_posting(P.post_ptr, 0, P.n_distinct, e1 - 1) + 1;
    __syncthreads();
    for (uint64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
      const uint64_t id = id_of_posting(P.post_ptr, id_lo, id_hi, e);
      const uint32_t p = P.post[e], g = p >> P.cnt_bits;
      uint32_t c = p & mask;
      if (c == P.cnt_cap) c = mv_count_of(P, g, P.post_ptr[id]);
      pad[pad_off[g] + atomicAdd(&fill[g], 1u)] = (code_at(P.code_lo, P.code_hi, id) << 16) | c;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(512) k_export_mv_sort(uint32_t n_genes, const unsigned long long* __restrict__ pad_off,
                                                        unsigned long long* pad) {
  for (uint32_t g = blockIdx.x; g < n_genes; g += gridDim.x) {
    const unsigned long long o = pad_off[g];
    const uint32_t n2 = (uint32_t)(pad_off[g + 1] - o);
    if (n2 > 1) block_bitonic_sort(pad + o, n2);
    __syncthreads();
  }
}

__global__ void k_export_mv(uint32_t n_genes, const unsigned long long* __restrict__ mv_ptr,
                            const unsigned long long* __restrict__ pad_off, const unsigned long long* __restrict__ pad,
                            unsigned long long* __restrict__ codes, uint32_t* __restrict__ counts) {
  for (uint32_t g = blockIdx.x; g < n_genes; g += gridDim.x) {
    const unsigned long long o = pad_off[g], dst = mv_ptr[g], n = mv_ptr[g + 1] - dst;
    for (uint32_t e = threadIdx.x; e < n; e += blockDim.x) {
      const unsigned long long v = pad[o + e];
      if (codes) codes[dst + e] = v >> 16;
      if (counts) counts[dst + e] = (uint32_t)(v & 0xFFFFu);
    }
  }
}

__global__ void k_export_index(ProfilesView P, int32_t* __restrict__ genes, uint32_t* __restrict__ counts) {
  const uint32_t mask = (1u << P.cnt_bits) - 1u;
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < P.n_entries;
       e += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t p = P.post[e];
    const uint32_t g = p >> P.cnt_bits;
    uint32_t c = p & mask;
    if (c == P.cnt_cap) {  // saturated: exact count from the gene's vector
      c = mv_count_of(P, g, P.post_ptr[id_of_posting(P.post_ptr, 0, P.n_distinct, e)]);
    }
    if (genes) genes[e] = (int32_t)g;
    if (counts) counts[e] = c;
  }
}

unsigned grid_for(uint64_t items, unsigned per_block, unsigned cap) {
  uint64_t b = (items + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

}  // namespace

#define PD_LAUNCH(L, name, ...)             \
  do {                                      \
    cudaError_t e_ = launch_begin(L, name); \
    if (e_ != cudaSuccess) return e_;       \
    __VA_ARGS__;                            \
    e_ = launch_end(L, name);               \
    if (e_ != cudaSuccess) return e_;       \
  } while (0)

cudaError_t run_dict_mark(Launcher* L, const uint32_t* code_lo, const uint8_t* code_hi, uint64_t n, uint32_t* dict,
                          cudaStream_t s) {
  PD_LAUNCH(L, "dict_mark", k_dict_mark<<<grid_for(n, 256, 152u * 16u), 256, 0, s>>>(code_lo, code_hi, n, dict));
  return cudaSuccess;
}

cudaError_t run_mv_build(Launcher* L, const uint8_t* res, const int64_t* gene_ptr, const uint32_t* win_off,
                         uint32_t n_genes, int k, const uint32_t* dict, const MvOut& M, const uint32_t* mid_genes, uint32_t n_mid, const uint32_t* long_genes,
                         uint32_t n_long, unsigned long long* long_scratch, const unsigned long long* long_scratch_off,
                         cudaStream_t s) {
  const size_t smem1 = (size_t)kMvSmallCap * 8, smem2 = (size_t)kMvMidCap * 8;
  cudaError_t ea = cudaFuncSetAttribute(k_mv_build_smem<kMvThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem1);
  if (ea != cudaSuccess) return ea;
  ea = cudaFuncSetAttribute(k_mv_build_smem<kMvLongThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2);
  if (ea != cudaSuccess) return ea;
  PD_LAUNCH(L, "mv_build",
            k_mv_build_smem<kMvThreads><<<grid_for(n_genes, 1, 152u * 64u), kMvThreads, smem1, s>>>(
                res, gene_ptr, win_off, n_genes, k, dict, M, kMvSmallCap, nullptr, 0u));
  if (n_mid) {
    PD_LAUNCH(L, "mv_build_mid",
              k_mv_build_smem<kMvLongThreads><<<grid_for(n_mid, 1, 152u), kMvLongThreads, smem2, s>>>(
                  res, gene_ptr, win_off, n_genes, k, dict, M, kMvMidCap, mid_genes, n_mid));
  }
  if (n_long) {
    PD_LAUNCH(L, "mv_build_long",
              k_mv_build_long<<<grid_for(n_long, 1, 152u), kMvLongThreads, 0, s>>>(
                  res, gene_ptr, win_off, k, dict, M, long_genes, n_long, long_scratch,
                  long_scratch_off));
  }
  return cudaSuccess;
}

uint32_t mv_build_table_cap(uint32_t La) { return mv_table_cap(La); }

cudaError_t run_order(Launcher* L, const uint32_t* minhash, const uint32_t* La, uint32_t n_genes, int length_buckets,
                      const uint32_t* cursor, const uint32_t* win_off, uint32_t* mv_n, uint32_t* count,
                      uint32_t* order, void* scan_tmp, cudaStream_t s) {
  PD_LAUNCH(L, "order_count", k_order_count<<<grid_for(n_genes, 256, 152u * 8u), 256, 0, s>>>(
                                  minhash, La, n_genes, length_buckets, cursor, win_off, mv_n, count));
  cudaError_t e = scan_u32(L, count, kOrderBuckets, count + kOrderBuckets, scan_tmp, s);  // n + 1 prefix entries
  if (e != cudaSuccess) return e;
  PD_LAUNCH(L, "order_scatter", k_order_scatter<<<grid_for(n_genes, 256, 152u * 8u), 256, 0, s>>>(
                                    minhash, La, n_genes, length_buckets, count + kOrderBuckets, order));
  return cudaSuccess;
}

cudaError_t run_export_codes(Launcher* L, const ProfilesView& P, unsigned long long* codes, cudaStream_t s) {
  PD_LAUNCH(L, "export_codes", k_export_codes<<<grid_for(P.n_distinct, 256, 152u * 16u), 256, 0, s>>>(
                                   P.code_lo, P.code_hi, P.n_distinct, codes));
  return cudaSuccess;
}

cudaError_t run_export_mv_count(Launcher* L, const ProfilesView& P, uint32_t* n, cudaStream_t s) {
  PD_LAUNCH(L, "export_mv_count", k_export_mv_count<<<grid_for(P.n_entries, 256, 152u * 16u), 256, 0, s>>>(P, n));
  return cudaSuccess;
}

cudaError_t run_export_mv(Launcher* L, const ProfilesView& P, const unsigned long long* mv_ptr,
                          const unsigned long long* pad_off, uint32_t* fill, unsigned long long* pad,
                          unsigned long long* codes, uint32_t* counts, cudaStream_t s) {
  const unsigned grid = grid_for(P.n_genes, 1, 152u * 16u);
  PD_LAUNCH(L, "export_mv_keys", k_export_mv_keys<<<grid_for(P.n_entries, kExportTile, 152u * 16u), 256, 0, s>>>(
                                     P, pad_off, fill, pad));
  PD_LAUNCH(L, "export_mv_sort", k_export_mv_sort<<<grid, 512, 0, s>>>(P.n_genes, pad_off, pad));
  PD_LAUNCH(L, "export_mv", k_export_mv<<<grid, 256, 0, s>>>(P.n_genes, mv_ptr, pad_off, pad, codes, counts));
  return cudaSuccess;
}

cudaError_t run_export_index(Launcher* L, const ProfilesView& P, int32_t* genes, uint32_t* counts, cudaStream_t s) {
  PD_LAUNCH(L, "export_index",
            k_export_index<<<grid_for(P.n_entries, 256, 152u * 16u), 256, 0, s>>>(P, genes, counts));
  return cudaSuccess;
}

}  // namespace pdg
