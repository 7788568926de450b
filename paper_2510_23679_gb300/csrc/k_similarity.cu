// k_similarity.cu -- sum-min of listed gene pairs: the similarity of Algorithm
// 2 ("Best Hit detection phase"), Eq. (5) numerator and denominator, for an
// explicit list of pairs.
//
// The all-against-all path finds the pairs that share a k-mer by walking the
// inverted index (k_summin.cu).  When the pairs are known beforehand -- the
// similarity of every BBH pair, a candidate list from elsewhere -- the two
// multiplicity vectors are joined:
//
//   1. the pairs are ordered by their first gene (counted, scanned,
//      scattered);
//   2. a warp takes up to 32 of them in that order (fewer where the list is
//      too short to give every warp of the chip 32).  It builds a hash table of
//      the first gene's vector in shared memory (k-mers are identified by the
//      start of their posting list), streams the second gene's vector past it,
//      adds the smaller count of every k-mer found, and rebuilds the table
//      where the first gene changes.  A vector longer than the table is joined
//      in parts, each of which reads the second vector again;
//   3. pairs whose first vector has more than kWarpEntries entries are left to a
//      block each, with a table 16 times as large.
//
// Against sorting every listed gene's vector (one block each, a bitonic
// network) and merging the sorted vectors, whole calls in ms (sorted and merged
// / 32 pairs a warp and no block form / this): 1 M pairs of 100 k genes of 300
// windows 9.2 / 2.4 / 1.8, 1000 pairs 0.27 / 0.40 / 0.11, 32 pairs 0.14 / 0.34 /
// 0.09; 400 pairs of genes of 8000 windows 0.6 / 43 / 0.12, 4000 of 30000 3.4 /
// 649 / 1.2, 100 k of 8000 10.8 / - / 6.1.  What remains of the longest is the
// second vectors, read from L2 and HBM.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "pd.h"
#include "pd_host.cuh"
#include "pd_internal.cuh"

using namespace pdh;

namespace {

// Most entries of a first vector that a warp joins: two parts of its table.  A
// third costs another pass over the second vector (1 M pairs of 100 k genes of
// 300 windows, whole call: 1.8 ms; with four parts 2.0, ten 2.4; 100 k pairs of
// genes of 5000: 2.6 and, with ten, 12.7).
constexpr uint32_t kWarpEntries = 818;

// Also sets *any_long if a first gene's vector is longer than a warp joins.
__global__ void k_pair_check(const uint32_t* __restrict__ a, const uint32_t* __restrict__ b, uint64_t n,
                             uint32_t n_genes, const uint32_t* __restrict__ mv_n, uint32_t* any_long,
                             pdg::DevErr* err) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    if (a[i] >= n_genes || b[i] >= n_genes)
      pdg::raise_error(err, PD_ERR_ARG, i);
    else if (mv_n[a[i]] > kWarpEntries)
      *any_long = 1u;
  }
}

__global__ void k_pair_count(const uint32_t* __restrict__ a, uint32_t n, uint32_t* __restrict__ count) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    atomicAdd(&count[a[i]], 1u);
}

__global__ void k_pair_order(const uint32_t* __restrict__ a, uint32_t n, uint32_t* __restrict__ cursor,
                             uint32_t* __restrict__ order) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    order[atomicAdd(&cursor[a[i]], 1u)] = i;
}

// Table of one warp: at least 2.5 slots per entry of a part, since most of the
// second gene's k-mers are not there and a search for one ends at a free slot
// (two thirds full, the longest of a warp's 32 searches took a dozen steps:
// 3.2 ms for 1 M pairs).
constexpr int kThreads = 128, kWarps = kThreads / 32, kBlocks = 9;  // resident blocks per SM (24 KB each)
constexpr uint32_t kSlots = 1024, kPart = 409;
static_assert(kPart * 5 / 2 <= kSlots, "2.5 slots per entry");
constexpr int kAhead = 4;  // the second gene's entries loaded ahead, per lane

// s and den of pair i = (ga, gb), whose joined counts sum to s.
__device__ __forceinline__ void put_pair(const pdg::ProfilesView& P, uint32_t i, uint32_t ga, uint32_t gb, uint32_t s,
                                         uint32_t* __restrict__ s_out, uint32_t* __restrict__ den_out) {
  const uint32_t La = P.La[ga], Lb = P.La[gb];
  if (ga == gb) s = La;  // the vectors leave out the gene's own k-mers
  if (s_out) s_out[i] = s;
  if (den_out) den_out[i] = La + Lb - s;
}

// per: pairs of a warp, at most 32.  longs (null: there are none): the pairs
// left out, whose number is counted in *n_longs.
__global__ void __launch_bounds__(kThreads)
    k_pair_similarity(pdg::ProfilesView P, const uint32_t* __restrict__ a, const uint32_t* __restrict__ b, uint32_t n,
                      uint32_t per, const uint32_t* __restrict__ order, uint32_t* __restrict__ s_out,
                      uint32_t* __restrict__ den_out, uint32_t* __restrict__ longs, uint32_t* n_longs,
                      const pdg::DevErr* err) {
  if (pdg::failed(err)) return;  // the scan of the places: the order is not whole
  __shared__ uint32_t keys[kWarps][kSlots];
  __shared__ uint16_t cnts[kWarps][kSlots];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t* key = keys[warp];
  uint16_t* cnt = cnts[warp];
  const uint32_t warps = gridDim.x * kWarps;
  const uint32_t n_chunks = (n + per - 1u) / per;
  for (uint32_t chunk = blockIdx.x * kWarps + warp; chunk < n_chunks; chunk += warps) {
    const uint32_t n_here = min(per, n - chunk * per);
    const uint32_t i = lane < n_here ? order[chunk * per + lane] : 0u;  // lane j holds pair j
    const uint32_t ga = lane < n_here ? a[i] : pdg::kEmpty, gb = lane < n_here ? b[i] : 0u;
    const uint32_t b0 = lane < n_here ? P.mv_off[gb] : 0u, bn = lane < n_here ? P.mv_n[gb] : 0u;
    uint32_t s = 0;
    bool left = false;
    for (uint32_t j0 = 0; j0 < n_here;) {
      const uint32_t g = __shfl_sync(0xffffffffu, ga, j0);
      const uint32_t run = __ballot_sync(0xffffffffu, ga == g);  // the pairs of this gene, j0 first
      const uint32_t j1 = j0 + (uint32_t)__popc(run);
      const uint32_t m0 = P.mv_off[g], na = P.mv_n[g];
      if (na > kWarpEntries) {
        if (ga == g) {
          longs[atomicAdd(n_longs, 1u)] = i;
          left = true;
        }
        j0 = j1;
        continue;
      }
      for (uint32_t part = 0; part < na; part += kPart) {
        const uint32_t np = min(kPart, na - part);
        const uint32_t bits = max(6u, 32u - (uint32_t)__clz(np * 5u / 2u - 1u)), shift = 32u - bits, mask = (1u << bits) - 1u;
        for (uint32_t h = lane; h <= mask; h += 32) key[h] = pdg::kEmpty;
        __syncwarp();
        for (uint32_t e = lane; e < np; e += 32) {
          const uint4 v = P.mv[m0 + part + e];
          uint32_t h = (v.x * 0x9E3779B1u) >> shift;
          while (atomicCAS(&key[h], pdg::kEmpty, v.x) != pdg::kEmpty) h = (h + 1u) & mask;  // a vector's k-mers differ
          cnt[h] = (uint16_t)v.y;
        }
        __syncwarp();
        for (uint32_t j = j0; j < j1; ++j) {
          const uint4* vb = P.mv + __shfl_sync(0xffffffffu, b0, j);
          const uint32_t nb = __shfl_sync(0xffffffffu, bn, j);
          uint32_t sum = 0;
          for (uint32_t e0 = lane; e0 < nb + lane; e0 += 32u * kAhead) {
            uint2 v[kAhead];  // list start, count
#pragma unroll
            for (int r = 0; r < kAhead; ++r) {
              const uint32_t e = e0 + 32u * r;
              v[r] = e < nb ? *reinterpret_cast<const uint2*>(vb + e) : make_uint2(pdg::kEmpty, 0u);
            }
#pragma unroll
            for (int r = 0; r < kAhead; ++r) {
              uint32_t h = (v[r].x * 0x9E3779B1u) >> shift, x = key[h];
              while (x != v[r].x && x != pdg::kEmpty) {  // the table has free slots
                h = (h + 1u) & mask;
                x = key[h];
              }
              if (x == v[r].x) sum += min((uint32_t)cnt[h], v[r].y);
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          if (lane == j) s += sum;
        }
        __syncwarp();
      }
      j0 = j1;
    }
    if (lane < n_here && !left) put_pair(P, i, ga, gb, s, s_out, den_out);
  }
}

// The pairs left out, one block each: the same join with a larger table.
constexpr int kLongThreads = 512;
constexpr uint32_t kLongSlots = 16384, kLongPart = 6553, kLongShift = 32 - 14;
constexpr size_t kLongBytes = (size_t)kLongSlots * 6;
static_assert(kLongPart * 5 / 2 <= kLongSlots && kLongSlots == 1u << (32 - kLongShift), "2.5 slots per entry");

__global__ void __launch_bounds__(kLongThreads, 2)
    k_pair_similarity_long(pdg::ProfilesView P, const uint32_t* __restrict__ a, const uint32_t* __restrict__ b,
                           const uint32_t* __restrict__ longs, const uint32_t* __restrict__ n_longs,
                           uint32_t* __restrict__ s_out, uint32_t* __restrict__ den_out) {
  extern __shared__ uint32_t key[];
  uint16_t* cnt = (uint16_t*)(key + kLongSlots);
  __shared__ uint32_t total;
  const uint32_t n = *n_longs, lane = threadIdx.x & 31u;
  for (uint32_t x = blockIdx.x; x < n; x += gridDim.x) {
    const uint32_t i = longs[x], ga = a[i], gb = b[i];
    const uint4 *va = P.mv + P.mv_off[ga], *vb = P.mv + P.mv_off[gb];
    const uint32_t na = P.mv_n[ga], nb = P.mv_n[gb];
    uint32_t sum = 0;
    if (threadIdx.x == 0) total = 0;
    for (uint32_t part = 0; part < na; part += kLongPart) {
      const uint32_t np = min(kLongPart, na - part);
      for (uint32_t h = threadIdx.x; h < kLongSlots; h += kLongThreads) key[h] = pdg::kEmpty;
      __syncthreads();
      for (uint32_t e = threadIdx.x; e < np; e += kLongThreads) {
        const uint4 v = va[part + e];
        uint32_t h = (v.x * 0x9E3779B1u) >> kLongShift;
        while (atomicCAS(&key[h], pdg::kEmpty, v.x) != pdg::kEmpty) h = (h + 1u) & (kLongSlots - 1u);
        cnt[h] = (uint16_t)v.y;
      }
      __syncthreads();
      for (uint32_t e = threadIdx.x; e < nb; e += kLongThreads) {
        const uint2 v = *reinterpret_cast<const uint2*>(vb + e);
        uint32_t h = (v.x * 0x9E3779B1u) >> kLongShift, y = key[h];
        while (y != v.x && y != pdg::kEmpty) {
          h = (h + 1u) & (kLongSlots - 1u);
          y = key[h];
        }
        if (y == v.x) sum += min((uint32_t)cnt[h], v.y);
      }
      __syncthreads();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0 && sum) atomicAdd(&total, sum);
    __syncthreads();
    if (threadIdx.x == 0) put_pair(P, i, ga, gb, total, s_out, den_out);
    __syncthreads();
  }
}

unsigned grid_of(uint64_t items, unsigned per_block, unsigned cap) {
  uint64_t g = (items + per_block - 1) / per_block;
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(g, cap));
}

// Pairs ordered and joined at a time (their places are 32-bit).
constexpr uint64_t kMaxPairs = 1ull << 30;

pd_status summin_list_impl(pd_ctx* c, const pd_profiles* P, const uint32_t* a, const uint32_t* b, uint64_t n,
                           uint32_t* s, uint32_t* den) {
  PhaseRange range_("pd: sum-min of listed pairs");
  pdg::Launcher* L = &c->L;
  const pdg::ProfilesView& v = P->view;
  const uint32_t G = v.n_genes;
  if (n == 0) return PD_OK;
  Buf d_a, d_b, tmp, longs, d_s, d_den;
  const uint32_t* pa = a;
  const uint32_t* pb = b;
  if (!is_device_ptr(a)) {
    ALLOC(d_a, sizeof(uint32_t) * n);
    CK(cudaMemcpyAsync(d_a.p, a, sizeof(uint32_t) * n, cudaMemcpyHostToDevice, c->stream));
    pa = d_a.as<uint32_t>();
  }
  if (!is_device_ptr(b)) {
    ALLOC(d_b, sizeof(uint32_t) * n);
    CK(cudaMemcpyAsync(d_b.p, b, sizeof(uint32_t) * n, cudaMemcpyHostToDevice, c->stream));
    pb = d_b.as<uint32_t>();
  }
  // zeroed: is any first vector long, how many such pairs, pairs of each gene
  const uint64_t most = std::min(n, kMaxPairs);
  Carve ct;
  const size_t o_words = ct.add(2 * sizeof(uint32_t)), o_count = ct.add(sizeof(uint32_t) * G), zeroed = ct.bytes,
               o_pos = ct.add(sizeof(uint32_t) * ((size_t)G + 1)), o_scan = ct.add(pdg::scan_temp_bytes(G + 1) + 64),
               o_order = ct.add(sizeof(uint32_t) * most);
  ALLOC(tmp, ct.bytes);
  uint32_t *words = piece<uint32_t>(tmp, o_words), *count = piece<uint32_t>(tmp, o_count),
           *pos = piece<uint32_t>(tmp, o_pos), *order = piece<uint32_t>(tmp, o_order);
  CK(cudaMemsetAsync(words, 0, zeroed, c->stream));
  CK(pdg::launch_begin(L, "pair_check"));
  k_pair_check<<<grid_of(n, 256, 152u * 16u), 256, 0, c->stream>>>(pa, pb, n, G, v.mv_n, words, c->d_err);
  CK(pdg::launch_end(L, "pair_check"));
  CK(cudaMemcpyAsync(c->h_build, words, sizeof(uint32_t), cudaMemcpyDeviceToHost, c->stream));
  pd_status st = check_dev_err(c);
  if (st != PD_OK) return fail(c, st, "pd_summin_list: a gene index is not below n_genes");
  const bool any_long = *(const uint32_t*)c->h_build != 0;
  if (any_long) {
    ALLOC(longs, sizeof(uint32_t) * most);
    CK(cudaFuncSetAttribute(k_pair_similarity_long, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLongBytes));
  }
  uint32_t* ps = s;
  uint32_t* pden = den;
  if (s && !is_device_ptr(s)) {
    ALLOC(d_s, sizeof(uint32_t) * n);
    ps = d_s.as<uint32_t>();
  }
  if (den && !is_device_ptr(den)) {
    ALLOC(d_den, sizeof(uint32_t) * n);
    pden = d_den.as<uint32_t>();
  }
  for (uint64_t p0 = 0; p0 < n; p0 += kMaxPairs) {
    const uint32_t m = (uint32_t)std::min(n - p0, kMaxPairs);
    // as many pairs a warp as give each resident warp some, sharing a first gene's table
    const uint32_t per = std::max(1u, std::min(32u, m / (152u * kBlocks * kWarps)));
    if (p0) CK(cudaMemsetAsync(words, 0, zeroed, c->stream));
    CK(pdg::launch_begin(L, "pair_count"));
    k_pair_count<<<grid_of(m, 256, 152u * 16u), 256, 0, c->stream>>>(pa + p0, m, count);
    CK(pdg::launch_end(L, "pair_count"));
    CK(pdg::scan_u32(L, count, G, pos, piece<void>(tmp, o_scan), c->stream));
    CK(pdg::launch_begin(L, "pair_order"));
    k_pair_order<<<grid_of(m, 256, 152u * 16u), 256, 0, c->stream>>>(pa + p0, m, pos, order);
    CK(pdg::launch_end(L, "pair_order"));
    uint32_t *s_part = ps ? ps + p0 : nullptr, *den_part = pden ? pden + p0 : nullptr;
    CK(pdg::launch_begin(L, "pair_similarity"));
    k_pair_similarity<<<grid_of(m, per * kWarps, 152u * 32u), kThreads, 0, c->stream>>>(
        v, pa + p0, pb + p0, m, per, order, s_part, den_part, longs.as<uint32_t>(), words + 1, c->d_err);
    CK(pdg::launch_end(L, "pair_similarity"));
    if (any_long) {
      CK(pdg::launch_begin(L, "pair_similarity_long"));
      k_pair_similarity_long<<<grid_of(m, 1, 152u * 2u), kLongThreads, kLongBytes, c->stream>>>(
          v, pa + p0, pb + p0, longs.as<uint32_t>(), words + 1, s_part, den_part);
      CK(pdg::launch_end(L, "pair_similarity_long"));
    }
  }
  if (ps != s) CK(cudaMemcpyAsync(s, ps, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost, c->stream));
  if (pden != den) CK(cudaMemcpyAsync(den, pden, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost, c->stream));
  return check_dev_err(c);  // synchronizes: the workspace ends here
}

}  // namespace

PD_API pd_status pd_summin_list(pd_ctx* c, const pd_profiles* P, const uint32_t* a, const uint32_t* b, uint64_t n,
                                uint32_t* s, uint32_t* den) {
  if (!c || !P || (n && (!a || !b))) return PD_ERR_ARG;
  try {
    CK(cudaSetDevice(c->device));
    return summin_list_impl(c, P, a, b, n, s, den);
  } catch (const std::bad_alloc&) {
    return fail(c, PD_ERR_OOM, "host allocation failed");
  } catch (...) {
    return fail(c, PD_ERR_INTERNAL, "exception in pd_summin_list");
  }
}
