// k_index.cu -- k-mer profiles and the inverted index by sorting
// ("Multiplicity vector building phase", Algorithm 1, Eqs. (1)-(3), and the
// index the sum-min kernel walks).
//
// Every k-mer window of every gene becomes one 64-bit record, its code above
// its gene (code << gene_bits | gene).  The records are produced in gene order
// and sorted by code with a stable radix sort, so equal (code, gene) records
// end up side by side (their number is the multiplicity, Eqs. (2)-(3)), a
// code's genes ascend, and the distinct codes, their dense ids, the posting
// lists and their bounds all come out of one more sequential pass.  No
// dictionary is looked up and no hash table is built: every pass streams.
//
//   check_letters  every residue is a letter of the alphabet.
//   code_hist      codes of all windows (Eq. (1), rolled along the gene):
//                  counts of every digit of every sort pass, and each gene's
//                  min-hash.
//   sort_windows   first sort pass, straight from the residues: a tile's codes
//                  are computed into shared memory and written out by digit.
//   sort_records   the later passes (least significant digit first).
//   dedupe         sorted records -> post (packed postings), post_ptr and
//                  the code of every id.
//   lists          every posting list of at least two genes -> one entry per
//                  posting, in its gene's vector.
//
// A k-mer of one gene only can never be shared, so the vectors the queries
// read hold the others (at 200 genomes x 4000 genes half of the distinct
// (k-mer, gene) pairs are such); the index keeps all of them, for the export
// calls and for queries from outside the dataset.
//
// Each sort pass reads and writes every record once: a tile's digit counts
// are combined with those of the tiles before it by decoupled look-back
// (Adinets and Merrill, "Onesweep", 2022).  A wait that runs out raises
// PD_ERR_INTERNAL and its tile writes nothing; the blocks and passes that start
// after it write nothing either, since what they would read was not written.
//
// Measured at 200 genomes x 4000 genes, k = 7 (266 M windows): 16.2 ms for the
// whole build against 23.4 ms for a dictionary of all codes (marked and looked
// up at random, 183 MB), hash tables per gene and a gather of every vector
// entry's list; 2.9 against 3.3 ms at 50 x 3000, k = 6.  Of the 16.2: windows
// counted 0.9, four sort passes 6.9 (each moves 4.2 GB in 1.6, 40% of the copy
// rate: bound by the latency of its phases at two blocks per SM), dedupe 2.2 (1.8
// without the counts of the vectors), list starts and codes copied 0.3, lists 5.4
// (an atomic and a 16-byte store at random for each of 130 M entries: bound by
// the rate of scattered requests to L2).
#include <algorithm>
#include <type_traits>

#include "pd_internal.cuh"

namespace pdg {
namespace {

typedef unsigned long long u64;

// ---------------------------------------------------------------- letters
// Flat form: the genes tile [0, n_res), so every byte is some gene's.
__global__ void __launch_bounds__(256)
    k_check_letters(const uint8_t* __restrict__ res, uint64_t n_res, int alpha, DevErr* err) {
  __shared__ uint8_t lut[256];
  init_letter_table(lut, alpha);
  const uint64_t head = min((uint64_t)((16 - ((uintptr_t)res & 15)) & 15), n_res);
  const uint64_t n_vec = (n_res - head) / 16;
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, n_thr = (uint64_t)gridDim.x * blockDim.x;
  const uint4* v = reinterpret_cast<const uint4*>(res + head);
  for (uint64_t i = tid; i < n_vec; i += n_thr) {
    const uint4 x = v[i];
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
    uint32_t worst = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int b = 0; b < 4; ++b) worst = max(worst, (uint32_t)lut[(w[j] >> (8 * b)) & 0xFFu]);
    if (worst >= (uint32_t)alpha) {
      for (int j = 0; j < 16; ++j)
        if (lut[res[head + 16 * i + j]] >= (uint32_t)alpha) raise_error(err, PD_ERR_ALPHABET, head + 16 * i + j);
    }
  }
  const uint64_t done = head + n_vec * 16, rest = head + (n_res - done);  // bytes outside the vectors
  for (uint64_t i = tid; i < rest; i += n_thr) {
    const uint64_t p = i < head ? i : done + (i - head);
    if (lut[res[p]] >= (uint32_t)alpha) raise_error(err, PD_ERR_ALPHABET, p);
  }
}

// Genes read in place of a larger input (gene_src): one warp per gene.
__global__ void __launch_bounds__(256)
    k_check_letters_genes(const uint8_t* __restrict__ res, const int64_t* __restrict__ gene_ptr,
                          const int64_t* __restrict__ gene_src, uint32_t n_genes, int alpha, DevErr* err) {
  __shared__ uint8_t lut[256];
  init_letter_table(lut, alpha);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < n_genes; g += warps) {
    const int64_t r0 = gene_src[g], len = gene_ptr[g + 1] - gene_ptr[g];
    for (int64_t p = lane; p < len; p += 32)
      if (lut[res[r0 + p]] >= (uint32_t)alpha) raise_error(err, PD_ERR_ALPHABET, (u64)(r0 + p));
  }
}

// ---------------------------------------------------------------- windows
// Window counts and genomes of the genes.  A gene whose offsets are malformed,
// or reach past the residues, is reported and gets no windows, so nothing after
// this kernel reads outside the residues.  The genome is the last that begins at
// or before the gene (genome offsets not checked yet only misplace it).
__global__ void k_gene_windows(const int64_t* __restrict__ gene_ptr, uint32_t n_genes, uint64_t n_res, int check_end,
                               int k, const int32_t* __restrict__ genome_ptr, uint32_t n_genomes,
                               uint32_t* __restrict__ La, uint16_t* __restrict__ gene_genome,
                               uint32_t* __restrict__ ginfo, uint32_t* __restrict__ minhash,
                               uint32_t* __restrict__ mv_n, DevErr* err) {
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n_genes; g += gridDim.x * blockDim.x) {
    const int64_t r0 = gene_ptr[g], r1 = gene_ptr[g + 1];
    const bool bad = r1 < r0 || r0 < 0 || (g == 0 && r0 != 0) ||
                     (check_end && ((uint64_t)r1 > n_res || (g + 1 == n_genes && (uint64_t)r1 != n_res)));
    uint64_t w = 0;
    if (bad) {
      raise_error(err, PD_ERR_ARG, g);
    } else {
      const int64_t len = r1 - r0;
      w = len >= k ? (uint64_t)(len - k + 1) : 0;
      if (w > PD_MAX_WINDOWS) {
        raise_error(err, PD_ERR_GENE_TOO_LONG, g);
        w = 0;
      }
    }
    uint32_t lo = 0, hi = n_genomes;
    while (hi - lo > 1u) {
      const uint32_t mid = (lo + hi) >> 1;
      if (genome_ptr[mid] <= (int32_t)g) lo = mid; else hi = mid;
    }
    La[g] = (uint32_t)w;
    gene_genome[g] = (uint16_t)lo;
    ginfo[g] = (uint32_t)w | (lo << 16);
    minhash[g] = kEmpty;
    mv_n[g] = 0;
  }
}

// Sort tiles: kItems consecutive windows (or records) per thread.  An odd
// number of 8-byte items per thread keeps the per-thread runs of the staged
// tile free of bank conflicts.
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 15;
constexpr uint32_t kTile = kThreads * kItems;
constexpr int kSortBlocks = 2;  // resident blocks per SM
constexpr int kMaxBins = kSortBins;  // digits of at most 9 bits

// Gene of the first window of every tile; tile_gene[n_tiles] = the last gene.
// Also the first free place of every gene's vector.
__global__ void k_tile_genes(const uint32_t* __restrict__ win_off, uint32_t n_genes, uint32_t n_tiles,
                             uint32_t* __restrict__ tile_gene, uint32_t* __restrict__ cursor) {
  if (blockIdx.x == 0 && threadIdx.x == 0) tile_gene[n_tiles] = n_genes - 1u;
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n_genes; g += gridDim.x * blockDim.x) {
    const uint64_t w0 = win_off[g], w1 = win_off[g + 1];
    cursor[g] = (uint32_t)w0;
    for (uint64_t t = (w0 + kTile - 1) / kTile; t * kTile < w1; ++t) tile_gene[t] = g;
  }
}

// Last gene g in [lo, hi) with win_off[g] <= w (it holds window w).
__device__ __forceinline__ uint32_t gene_of_window(const uint32_t* __restrict__ win_off, uint32_t lo, uint32_t hi,
                                                   uint32_t w) {
  while (hi - lo > 1u) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (win_off[mid] <= w) lo = mid; else hi = mid;
  }
  return lo;
}

// Calls emit(i, code, gene) for this thread's kItems consecutive windows of
// tile t, in order.  The code rolls along the gene: Eq. (1)'s value of the last
// k-1 letters, times alpha, plus the next letter; `recent` holds the digits of
// the window (5 bits each, 2 for nucleotides), whose oldest is taken off again.
// The thread's first gene is found among the tile's genes by bisection.
// Code: uint32_t when every code (with its segment's base) fits, else u64.
template <typename Code, typename Emit>
__device__ __forceinline__ void tile_windows(const WindowSource& S, const uint8_t* lut, uint32_t t, Emit emit) {
  const uint64_t w0 = (uint64_t)t * kTile + (uint64_t)threadIdx.x * kItems;
  if (w0 >= S.n_windows) return;
  const uint32_t g_hi = S.tile_gene[t + 1] + 1u;
  uint32_t g = gene_of_window(S.win_off, S.tile_gene[t], g_hi, (uint32_t)w0);
  const uint32_t bits = S.alpha == 4 ? 2u : 5u, drop = bits * (uint32_t)(S.k - 1);
  const u64 keep = (1ull << drop) - 1ull;
  const Code a = (Code)S.alpha;
  Code lead_w = 1;  // alpha^(k-1)
  for (int j = 1; j < S.k; ++j) lead_w *= a;
  uint32_t end = S.win_off[g + 1];
  const uint8_t* s = nullptr;  // next letter
  u64 recent = 0;
  Code code = 0, base = 0;
  bool fresh = true;
  const uint32_t n = (uint32_t)min((uint64_t)kItems, S.n_windows - w0);
#pragma unroll 1
  for (uint32_t i = 0; i < n; ++i) {
    const uint32_t w = (uint32_t)w0 + i;
    if (w == end) {
      g = gene_of_window(S.win_off, g, g_hi, w);
      end = S.win_off[g + 1];
      fresh = true;
    }
    if (fresh) {
      s = S.res + (S.gene_src ? S.gene_src[g] : S.gene_ptr[g]) + (w - S.win_off[g]);
      base = S.genome_code_base ? (Code)S.genome_code_base[S.gene_genome[g]] : (Code)0;
      code = 0;
      recent = 0;
      for (int j = 0; j + 1 < S.k; ++j) {
        const uint32_t c = lut[*s++];
        code = code * a + c;
        recent = (recent << bits) | c;
      }
      fresh = false;
    }
    const uint32_t c = lut[*s++];
    code = code * a + c;
    recent = (recent << bits) | c;
    emit(i, (code << S.code_shift) + base, g);
    code -= (Code)(uint32_t)(recent >> drop) * lead_w;
    recent &= keep;
  }
}

// Letter table with every other byte mapped to 0: an input holding one is
// refused (check_letters), and until then its codes must stay in range.
__device__ __forceinline__ void init_code_table(uint8_t* lut, int alpha) {
  init_letter_table(lut, alpha);
  for (int i = threadIdx.x; i < 256; i += blockDim.x)
    if (lut[i] >= (uint32_t)alpha) lut[i] = 0;
  __syncthreads();
}

// Digit counts of every pass (hist[pass * kMaxBins + digit]) over the windows
// of this slice, and the genes' min-hashes (minimum of a hash of the codes).
// Bound by the shared-memory atomics (one per window and pass).
template <typename Code, int kPasses>
__global__ void __launch_bounds__(kThreads)
    k_code_hist(WindowSource S, SortKey K, uint32_t n_tiles, uint32_t* __restrict__ hist,
                uint32_t* __restrict__ minhash) {
  __shared__ uint8_t lut[256];
  __shared__ uint32_t cnt[kPasses * kMaxBins];
  for (uint32_t d = threadIdx.x; d < kPasses * kMaxBins; d += kThreads) cnt[d] = 0;
  init_code_table(lut, S.alpha);
  const uint32_t dmask = (1u << K.width) - 1u;
  const bool all = K.n_slices == 1;
  for (uint32_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    uint32_t cur = kEmpty, low = kEmpty;
    tile_windows<Code>(S, lut, t, [&](uint32_t, Code code, uint32_t g) {
      if (minhash) {
        if (g != cur) {
          if (cur != kEmpty) atomicMin(&minhash[cur], low);
          cur = g;
          low = kEmpty;
        }
        low = min(low, mix32((uint32_t)code ^ (uint32_t)((u64)code >> 32)));
      }
      if (all || ((u64)code >> K.code_bits) == K.slice) {
#pragma unroll
        for (uint32_t p = 0; p < kPasses; ++p)
          atomicAdd(&cnt[p * kMaxBins + ((uint32_t)(code >> (K.skip + p * K.width)) & (p + 1 < kPasses ? dmask : K.last_mask))],
                    1u);
      }
    });
    if (minhash && cur != kEmpty) atomicMin(&minhash[cur], low);
  }
  __syncthreads();
  for (uint32_t d = threadIdx.x; d < kPasses * kMaxBins; d += kThreads)
    if (cnt[d]) atomicAdd(&hist[d], cnt[d]);
}

// ---------------------------------------------------------------- sort pass
template <int kBits>
struct PassShared {
  uint16_t wcnt[kWarps][1 << kBits];  // per warp: records of each digit, then its offset among the warps
  uint16_t tbase[1 << kBits];         // tile-local start of each digit
  u64 gbase[1 << kBits];              // output position of the tile's first record of each digit, less tbase
  uint32_t warp_tmp[kWarps + 1];
  uint32_t tile;
  int failed;
};

// Takes a tile, unless something failed before (false).  The first one also
// scans the digit counts into gbase (the digits' starts), so that the running
// sums over the tiles are output positions.
template <int kBits>
__device__ __forceinline__ bool begin_tile(PassShared<kBits>& sh, const uint32_t* __restrict__ hist, uint32_t* ticket,
                                           const DevErr* err) {
  for (uint32_t x = threadIdx.x; x < (kWarps << kBits) / 2; x += kThreads) ((uint32_t*)&sh.wcnt[0][0])[x] = 0;
  if (threadIdx.x == 0) {
    sh.failed = failed(err);
    if (!sh.failed) sh.tile = atomicAdd(ticket, 1u);
  }
  __syncthreads();
  if (sh.failed) return false;
  if (sh.tile == 0) {
    uint32_t carry = 0;
    for (uint32_t d0 = 0; d0 < (1u << kBits); d0 += kThreads) {
      const uint32_t d = d0 + threadIdx.x;
      uint32_t n;
      const uint32_t ex = block_exclusive_scan(d < (1u << kBits) ? hist[d] : 0u, sh.warp_tmp, &n);
      if (d < (1u << kBits)) sh.gbase[d] = carry + ex;
      carry += n;
    }
    __syncthreads();
  }
  return true;
}

// Stable counting step of one tile.  xr: the thread's records, striped within
// the warp's run of 32 * kItems (item r of lane l is position r * 32 + l).
// Ranks within the warp come from the lanes holding the same digit: each lane
// sets its bit in the digit's word of a table of the warp's (in the staging
// memory, not in use yet).  Finding them with one ballot per digit bit took
// four instructions a bit and kept the ALU the busiest pipe (266 M records, the
// whole run of 200 genomes x 4000 genes 46.0 ms against 44.7; 1.6 a pass now).
template <int kBits, typename T>
__device__ __forceinline__ void rank_and_write(u64 (&xr)[kItems], uint32_t valid_mask, uint32_t shift, T* status,
                                               u64* __restrict__ out, PassShared<kBits>& sh, u64* stage, DevErr* err) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  constexpr uint32_t bins = 1u << kBits, dmask = bins - 1u;
  constexpr int kOwn = (int)((bins + kThreads - 1) / kThreads);  // digits kOwn * t .. of thread t
  static_assert((size_t)kWarps * bins * 4 <= (size_t)kTile * 8, "the match table fits the staging memory");
  const uint32_t below = (1u << lane) - 1u;
  uint32_t* match = (uint32_t*)stage + warp * bins;
  for (uint32_t d = lane; d < bins; d += 32) match[d] = 0;
  __syncwarp();
  uint32_t rk[(kItems + 1) / 2];  // two 16-bit ranks each
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const bool valid = (valid_mask >> r) & 1u;
    const uint32_t d = (uint32_t)(xr[r] >> shift) & dmask;
    if (valid) atomicOr(&match[d], 1u << lane);
    __syncwarp();
    const uint32_t peers = *(volatile uint32_t*)&match[d], base = sh.wcnt[warp][d];
    const uint32_t before = (uint32_t)__popc(peers & below);
    __syncwarp();
    if (valid && before == 0) {
      sh.wcnt[warp][d] = (uint16_t)(base + (uint32_t)__popc(peers));
      match[d] = 0;
    }
    __syncwarp();
    if (r & 1) rk[r / 2] |= (base + before) << 16; else rk[r / 2] = base + before;
  }
  __syncthreads();
  // per digit: exclusive prefix over the warps and the tile's count
  uint32_t tot[kOwn], sum = 0;
#pragma unroll
  for (int j = 0; j < kOwn; ++j) {
    const uint32_t d = kOwn * threadIdx.x + (uint32_t)j;
    tot[j] = 0;
    if (d < bins) {
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = sh.wcnt[w][d];
        sh.wcnt[w][d] = (uint16_t)run;
        run += c;
      }
      tot[j] = run;
      // the first tile's sums are inclusive at once: the digit's start is known
      *(volatile T*)(status + (uint64_t)sh.tile * bins + d) =
          sh.tile == 0 ? Status<T>::kInclusive | (T)(sh.gbase[d] + run) : Status<T>::kAggregate | (T)run;
    }
    sum += tot[j];
  }
  uint32_t all;
  uint32_t tb = block_exclusive_scan(sum, sh.warp_tmp, &all);
#pragma unroll
  for (int j = 0; j < kOwn; ++j) {
    const uint32_t d = kOwn * threadIdx.x + (uint32_t)j;
    if (d < bins) sh.tbase[d] = (uint16_t)tb;
    tb += tot[j];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r)
    if ((valid_mask >> r) & 1u) {
      const uint32_t d = (uint32_t)(xr[r] >> shift) & dmask;
      stage[sh.tbase[d] + sh.wcnt[warp][d] + ((rk[r / 2] >> (16 * (r & 1))) & 0xFFFFu)] = xr[r];
    }
  // the tiles before this one
#pragma unroll
  for (int j = 0; j < kOwn; ++j) {
    const uint32_t d = kOwn * threadIdx.x + (uint32_t)j;
    if (d < bins) {
      T before = 0;
      if (sh.tile == 0) {
        before = (T)sh.gbase[d];
      } else {
        if (!look_back<T>(status + d, sh.tile, bins, &before, err)) {
          raise_error(err, PD_ERR_INTERNAL, sh.tile);
          sh.failed = 1;
        } else {
          volatile T* st = status + (uint64_t)sh.tile * bins + d;
          *st = Status<T>::kInclusive | (before + tot[j]);
        }
      }
      sh.gbase[d] = (u64)before - sh.tbase[d];
    }
  }
  __syncthreads();
  if (sh.failed) return;  // uniform: positions unknown
  for (uint32_t p = threadIdx.x; p < all; p += kThreads) {
    const u64 v = stage[p];
    out[sh.gbase[(uint32_t)(v >> shift) & dmask] + p] = v;
  }
}

template <int kBits, typename T, typename Code>
__global__ void __launch_bounds__(kThreads, kSortBlocks)
    k_sort_windows(WindowSource S, SortKey K, const uint32_t* __restrict__ hist, T* status, uint32_t* ticket,
                   u64* __restrict__ out, DevErr* err) {
  extern __shared__ u64 stage[];
  __shared__ PassShared<kBits> sh;
  __shared__ uint8_t lut[256];
  init_code_table(lut, S.alpha);
  if (!begin_tile<kBits>(sh, hist, ticket, err)) return;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t at = threadIdx.x * kItems;
  // the all-ones word is no record: the gene field never holds all ones
  for (int i = 0; i < kItems; ++i) stage[at + i] = ~0ull;
  const bool every = K.n_slices == 1;
  tile_windows<Code>(S, lut, sh.tile, [&](uint32_t i, Code code, uint32_t g) {
    if (every || ((u64)code >> K.code_bits) == K.slice)
      stage[at + i] = (((u64)code & ((1ull << K.code_bits) - 1ull)) << K.gene_bits) | g;
  });
  __syncthreads();
  u64 xr[kItems];
  uint32_t valid = 0;
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    xr[r] = stage[warp * 32u * kItems + r * 32u + lane];
    valid |= xr[r] != ~0ull ? 1u << r : 0u;
  }
  __syncthreads();
  rank_and_write<kBits, T>(xr, valid, K.gene_bits + K.skip, status, out, sh, stage, err);
}

template <int kBits, typename T>
__global__ void __launch_bounds__(kThreads, kSortBlocks)
    k_sort_records(const u64* __restrict__ in, uint64_t n, uint32_t shift, const uint32_t* __restrict__ hist,
                   T* status, uint32_t* ticket, u64* __restrict__ out, DevErr* err) {
  extern __shared__ u64 stage[];
  __shared__ PassShared<kBits> sh;
  if (!begin_tile<kBits>(sh, hist, ticket, err)) return;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint64_t t0 = (uint64_t)sh.tile * kTile + warp * 32u * kItems;
  u64 xr[kItems];
  uint32_t valid = 0;
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const uint64_t i = t0 + r * 32u + lane;
    xr[r] = i < n ? in[i] : 0ull;
    valid |= i < n ? 1u << r : 0u;
  }
  rank_and_write<kBits, T>(xr, valid, shift, status, out, sh, stage, err);
}

// ---------------------------------------------------------------- dedupe
// Tiles of sorted records, striped within each warp like the sort's.
constexpr int kDThreads = 512, kDWarps = kDThreads / 32, kDItems = 16;
constexpr uint32_t kDTile = kDThreads * kDItems;
// ... and of postings: those of half a tile of records (longer tiles wait less
// for one another, shorter ones leave room for more blocks of the lists pass).
constexpr int kLItems = 8;
constexpr uint32_t kLTile = kDThreads * kLItems, kHalves = kDTile / kLTile;
static_assert(kHalves == 2 && kDWarps % 2 == 0, "a list tile is half the warps of a dedupe tile");

// First record after i (in [lo, n)) whose key differs from `key`; records
// before lo are equal to it.  Runs are short, so the search gallops first.
__device__ __forceinline__ uint64_t run_end(const u64* __restrict__ rec, uint64_t lo, uint64_t n, u64 key) {
  uint64_t step = 1, hi = lo;
  while (hi < n && rec[hi] == key) {
    lo = hi + 1;
    hi = lo + step;
    step <<= 1;
  }
  hi = min(hi, n);
  while (lo < hi) {
    const uint64_t mid = (lo + hi) >> 1;
    if (rec[mid] == key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Sorted records of one slice -> postings, posting-list starts and codes.
// A posting is the first record of a run of equal ones, its count the length
// of the run.  tile_e / tile_id: postings and ids before each half tile (and,
// after the last, in all); totals[0], totals[1]: postings and ids so far, read and
// advanced by each slice.  kCount: also the vector entries of every gene (mv_n),
// one for each posting that the lists pass will keep (200 genomes x 4000 genes
// 2.2 against 1.8 ms).
template <bool kCount>
__global__ void __launch_bounds__(kDThreads, 2)
    k_dedupe(const u64* __restrict__ rec, uint64_t n, SortKey K, uint32_t n_tiles, uint32_t cnt_bits, uint32_t cnt_cap,
             u64* status_e, u64* status_id, uint32_t* ticket, u64* totals, uint32_t* __restrict__ post,
             uint32_t* __restrict__ post_ptr, uint32_t* __restrict__ code_lo, uint8_t* __restrict__ code_hi,
             uint32_t* __restrict__ tile_e, uint32_t* __restrict__ tile_id, uint32_t* mv_n, DevErr* err) {
  __shared__ uint32_t s_tile, s_we[kDWarps + 1], s_wi[kDWarps + 1];
  __shared__ u64 s_base[2];
  __shared__ int s_failed;
  // tile position of each posting's first record, with the top bit if it is an id's first
  constexpr uint32_t kIdHead = 0x80000000u, kPosition = kIdHead - 1u;
  __shared__ uint32_t head[kDTile + 1];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_failed = failed(err);
    if (!s_failed) s_tile = atomicAdd(ticket, 1u);
  }
  __syncthreads();
  if (s_failed) return;
  const uint32_t tile = s_tile;
  const uint64_t t0 = (uint64_t)tile * kDTile;
  const uint32_t p0 = warp * 32u * kDItems + lane;
  u64 xr[kDItems];
#pragma unroll
  for (int r = 0; r < kDItems; ++r) {
    const uint64_t i = t0 + p0 + r * 32u;
    xr[r] = i < n ? rec[i] : 0ull;
  }
  uint32_t he[kDItems], hi[kDItems];  // ballots: first records of postings, of ids
  uint32_t ne = 0, ni = 0;
  {
    const uint64_t w0 = t0 + warp * 32u * kDItems;
    u64 carry = (lane == 0 && w0 > 0 && w0 < n) ? rec[w0 - 1] : 0ull;  // lane 0: the record before
#pragma unroll
    for (int r = 0; r < kDItems; ++r) {
      const uint64_t i = t0 + p0 + r * 32u;
      u64 prev = __shfl_up_sync(0xffffffffu, xr[r], 1);
      if (lane == 0) prev = carry;
      he[r] = __ballot_sync(0xffffffffu, i < n && (i == 0 || xr[r] != prev));
      hi[r] = __ballot_sync(0xffffffffu, i < n && (i == 0 || (xr[r] >> K.gene_bits) != (prev >> K.gene_bits)));
      carry = __shfl_sync(0xffffffffu, xr[r], 31);
      ne += __popc(he[r]);
      ni += __popc(hi[r]);
    }
  }
  if (lane == 0) {
    s_we[warp] = ne;
    s_wi[warp] = ni;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t a = 0, b = 0;
    for (int w = 0; w < kDWarps; ++w) {
      const uint32_t x = s_we[w], y = s_wi[w];
      s_we[w] = a;
      s_wi[w] = b;
      a += x;
      b += y;
    }
    s_we[kDWarps] = a;
    s_wi[kDWarps] = b;
  }
  __syncthreads();
  if (warp < 2) {  // one column each: postings, ids
    using St = Status<u64>;
    volatile u64* st = warp == 0 ? status_e : status_id;
    const u64 mine = warp == 0 ? s_we[kDWarps] : s_wi[kDWarps];
    u64 before = totals[2 + warp];  // the slices before
    bool ok = true;
    if (tile != 0) {
      if (lane == 0) st[tile] = St::kAggregate | mine;
      ok = look_back_warp(st, tile, &before, err);
    }
    if (lane == 0) {
      if (ok) {
        st[tile] = St::kInclusive | (before + mine);
      } else {
        raise_error(err, PD_ERR_INTERNAL, tile);
        s_failed = 1;
      }
      s_base[warp] = before;
    }
  }
  // tile positions of the postings
  uint32_t le = s_we[warp];
#pragma unroll
  for (int r = 0; r < kDItems; ++r) {
    if ((he[r] >> lane) & 1u)
      head[le + __popc(he[r] & ((1u << lane) - 1u))] =
          (p0 + r * 32u) | (kCount && ((hi[r] >> lane) & 1u) ? kIdHead : 0u);
    le += __popc(he[r]);
  }
  if (threadIdx.x == 0) {
    const uint32_t n_e = s_we[kDWarps];
    const uint64_t t1 = min(n, t0 + kDTile);
    uint64_t end = t1;  // the tile's last posting may go on in the next tile
    if (n_e && t1 < n && rec[t1] == rec[t1 - 1]) end = run_end(rec, t1, n, rec[t1 - 1]);
    const bool id_ends = kCount && n_e && (end == n || (rec[end] >> K.gene_bits) != (rec[end - 1] >> K.gene_bits));
    head[n_e] = (uint32_t)min(end - t0, (uint64_t)kPosition) | (id_ends ? kIdHead : 0u);
  }
  __syncthreads();
  if (s_failed) return;
  const uint32_t e0 = (uint32_t)s_base[0], id0 = (uint32_t)s_base[1];
  if (threadIdx.x == 0) {
    for (uint32_t half = 0; half < kHalves; ++half) {
      tile_e[kHalves * tile + half] = e0 + s_we[half * (kDWarps / 2)];
      tile_id[kHalves * tile + half] = id0 + s_wi[half * (kDWarps / 2)];
    }
    if (tile + 1u == n_tiles) {
      const uint32_t e1 = e0 + s_we[kDWarps], id1 = id0 + s_wi[kDWarps];
      tile_e[kHalves * n_tiles] = e1;
      tile_id[kHalves * n_tiles] = id1;
      post_ptr[id1] = e1;
      totals[0] = e1;
      totals[1] = id1;
    }
  }
  const uint32_t gmask = (1u << K.gene_bits) - 1u;
  le = s_we[warp];
  uint32_t li = s_wi[warp];
#pragma unroll
  for (int r = 0; r < kDItems; ++r) {
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t e = le + __popc(he[r] & below);
    if ((he[r] >> lane) & 1u) {
      const uint32_t h = head[e], next = head[e + 1], c = (next & kPosition) - (h & kPosition);
      post[e0 + e] = (((uint32_t)xr[r] & gmask) << cnt_bits) | min(c, cnt_cap);
      if (kCount && (!(h & next & kIdHead) || c >= cnt_cap)) atomicAdd(&mv_n[(uint32_t)xr[r] & gmask], 1u);
    }
    if ((hi[r] >> lane) & 1u) {
      const uint32_t id = id0 + li + __popc(hi[r] & below);
      const u64 code = (K.slice << K.code_bits) | (xr[r] >> K.gene_bits);
      post_ptr[id] = e0 + e;
      code_lo[id] = (uint32_t)code;
      if (code_hi) code_hi[id] = (uint8_t)(code >> 32);
    }
    le += __popc(he[r]);
    li += __popc(hi[r]);
  }
}

// ---------------------------------------------------------------- lists
// For every posting of a list of at least two genes (or whose count does not
// fit its field: the vector then holds the exact one) the vector entry of its
// gene,
//   x = list start, y = count, z = list length | (another posting of the
//   gene's genome) << 31, w = offset in the list of the first posting past the
//   gene's genome,
// goes to the next free place of the gene's vector (cursor).  Tiles are halves
// of the dedupe's; blocks are persistent, so that the table that gives a gene's
// genome is built once per block: a gene's genome lies between those of the
// table's entries around it.  Runs of one genome are marked in a bit mask of the
// tile, whose next set bit gives w.  Also the longest list and the sum of
// squared lengths.
constexpr uint32_t kGenomeTable = 2048;
static_assert((kLTile + 2) * 4 + 3 * kLTile / 8 + kLTile * 2 + (kGenomeTable + 2) * 2 + PD_MAX_GENOMES * 4 <= 48 * 1024,
              "the lists pass fits the shared memory that every launch may use");

__device__ __forceinline__ uint32_t lower_bound_gene(const uint32_t* __restrict__ post, uint32_t lo, uint32_t hi,
                                                     uint32_t cnt_bits, uint32_t gene) {
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if ((post[mid] >> cnt_bits) < gene) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Records equal to `key`, whose first is in [lo, hi) (the posting's tile).
__device__ __forceinline__ uint32_t exact_count(const u64* __restrict__ rec, uint64_t lo, uint64_t hi, uint64_t n,
                                                u64 key) {
  while (lo < hi) {
    const uint64_t mid = (lo + hi) >> 1;
    if (rec[mid] < key) lo = mid + 1; else hi = mid;
  }
  return (uint32_t)(run_end(rec, lo, n, key) - lo);
}

__global__ void __launch_bounds__(kDThreads, 3)
    k_lists(const uint32_t* __restrict__ tile_e, const uint32_t* __restrict__ tile_id, uint32_t n_tiles,
            const u64* __restrict__ rec, uint64_t n_rec, SortKey K, const uint32_t* __restrict__ code_lo,
            const uint8_t* __restrict__ code_hi, const uint32_t* __restrict__ post,
            const uint32_t* __restrict__ post_ptr, uint32_t cnt_bits, uint32_t cnt_cap,
            const int32_t* __restrict__ genome_ptr, uint32_t n_genomes, uint32_t n_genes, uint32_t table_bits,
            uint32_t* cursor, uint4* __restrict__ mv, uint32_t* max_list, u64* join, const DevErr* err) {
  if (failed(err)) return;  // the same in every thread: nothing is reported from here
  __shared__ uint32_t start[kLTile + 2];
  __shared__ uint32_t is_head[kLTile / 32], run_head[kLTile / 32];
  __shared__ uint16_t genome[kLTile];
  __shared__ uint32_t before[kLTile / 32];  // list heads before each word
  __shared__ uint16_t table[kGenomeTable + 1];
  extern __shared__ int32_t gend[];  // first gene past each genome
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  for (uint32_t i = threadIdx.x; i < n_genomes; i += kDThreads) gend[i] = genome_ptr[i + 1];
  __syncthreads();
  // genome of a gene, known to lie in [lo, hi]: the first whose end is past it
  auto find = [&](uint32_t g, uint32_t lo, uint32_t hi) {
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if ((uint32_t)gend[mid] <= g) lo = mid + 1; else hi = mid;
    }
    return lo;
  };
  const uint32_t n_table = ((n_genes - 1u) >> table_bits) + 1u;
  for (uint32_t x = threadIdx.x; x <= n_table; x += kDThreads)
    table[x] = (uint16_t)find(min(x << table_bits, n_genes - 1u), 0u, n_genomes - 1u);
  auto genome_of = [&](uint32_t g) { return find(g, table[g >> table_bits], table[(g >> table_bits) + 1u]); };
  uint32_t longest = 0;
  u64 squares = 0;
  for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const uint32_t e0 = tile_e[tile], e1 = tile_e[tile + 1];
    const uint32_t id0 = tile_id[tile], id1 = tile_id[tile + 1];
    const uint32_t n = e1 - e0, n_heads = id1 - id0;
    __syncthreads();  // the table is built; the last tile's shared arrays are done with
    for (uint32_t i = threadIdx.x; i < kLTile / 32; i += kDThreads) is_head[i] = 0;
    __syncthreads();
    // start[l]: list l of the tile; list 0 is the one begun before it (if any)
    for (uint32_t l = threadIdx.x; l < n_heads + 2u; l += kDThreads) {
      const uint32_t p = l == 0 && id0 == 0 ? 0u : post_ptr[id0 + l - 1u];
      start[l] = p;
      if (l >= 1u && l <= n_heads) {
        atomicOr(&is_head[(p - e0) >> 5], 1u << ((p - e0) & 31u));
        const u64 len = post_ptr[id0 + l] - p;
        longest = max(longest, (uint32_t)len);
        squares += len * len;
      }
    }
    uint32_t pv[kLItems];
#pragma unroll
    for (int r = 0; r < kLItems; ++r) {
      const uint32_t i = (uint32_t)r * kDThreads + threadIdx.x;
      pv[r] = i < n ? post[e0 + i] : 0u;
    }
    __syncthreads();
    if (warp == 0) {
      uint32_t carry = 0;
      for (uint32_t w0 = 0; w0 < kLTile / 32; w0 += 32) {
        const uint32_t c = __popc(is_head[w0 + lane]);
        const uint32_t inc = warp_inclusive_scan(c);
        before[w0 + lane] = carry + inc - c;
        carry += __shfl_sync(0xffffffffu, inc, 31);
      }
    }
    __syncthreads();
    auto list_of = [&](uint32_t i) {
      return before[i >> 5] + __popc(is_head[i >> 5] & (0xFFFFFFFFu >> (31u - (i & 31u))));
    };
    // genomes of the postings of lists of two and more
    uint32_t kept = 0;
#pragma unroll
    for (int r = 0; r < kLItems; ++r) {
      const uint32_t i = (uint32_t)r * kDThreads + threadIdx.x;
      if (i < n) {
        const uint32_t l = list_of(i);
        if (start[l + 1] - start[l] >= 2u || (pv[r] & ((1u << cnt_bits) - 1u)) >= cnt_cap) {
          kept |= 1u << r;
          genome[i] = (uint16_t)genome_of(pv[r] >> cnt_bits);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kLItems; ++r) {
      const uint32_t i = (uint32_t)r * kDThreads + threadIdx.x;
      bool f = false;
      if (i < n) {
        const bool h = (is_head[i >> 5] >> (i & 31u)) & 1u;
        f = h || !((kept >> r) & 1u);
        if (!f) f = genome[i] != (i ? genome[i - 1] : (uint16_t)genome_of(post[e0 - 1] >> cnt_bits));
      }
      const uint32_t m = __ballot_sync(0xffffffffu, f);
      if (lane == 0) run_head[(r * kDThreads + warp * 32u) >> 5] = m;
    }
    __syncthreads();
    uint32_t at[kLItems];  // all places first: the atomics are in flight together
#pragma unroll
    for (int r = 0; r < kLItems; ++r)
      if ((kept >> r) & 1u) at[r] = atomicAdd(&cursor[pv[r] >> cnt_bits], 1u);
#pragma unroll
    for (int r = 0; r < kLItems; ++r) {
      if (!((kept >> r) & 1u)) continue;
      const uint32_t i = (uint32_t)r * kDThreads + threadIdx.x, l = list_of(i);
      const uint32_t s = start[l], t = start[l + 1];
      // next run after i, and whether i's own run has another posting
      uint32_t w = i >> 5, m = run_head[w] & ~(0xFFFFFFFFu >> (31u - (i & 31u)));
      while (m == 0 && ++w < (n + 31u) / 32u) m = run_head[w];
      uint32_t next;  // posting index
      if (m)
        next = e0 + w * 32u + (uint32_t)__ffs((int)m) - 1u;
      else
        next = t <= e1 ? t : lower_bound_gene(post, e1, t, cnt_bits, (uint32_t)gend[genome[i]]);
      const bool begins = (run_head[i >> 5] >> (i & 31u)) & 1u;
      const bool more = !begins || next > e0 + i + 1u;
      uint32_t c = pv[r] & ((1u << cnt_bits) - 1u);
      if (c >= cnt_cap) {
        const u64 code = code_at(code_lo, code_hi, id0 + l - 1u) & ((1ull << K.code_bits) - 1ull);
        const uint64_t t0 = (uint64_t)tile * kLTile;
        c = exact_count(rec, t0 + i, min(n_rec, t0 + kLTile), n_rec, (code << K.gene_bits) | (pv[r] >> cnt_bits));
      }
      mv[at[r]] = make_uint4(s, c, (t - s) | (more ? 0x80000000u : 0u), next - s);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    longest = max(longest, __shfl_xor_sync(0xffffffffu, longest, o));
    squares += __shfl_xor_sync(0xffffffffu, squares, o);
  }
  if (lane == 0 && longest) {
    atomicMax(max_list, longest);
    atomicAdd(join, squares);
  }
}

// Arrays moved to where they stay, 16 bytes at a time (all are padded to that).
__global__ void __launch_bounds__(256)
    k_pack(PackList L) {
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (uint64_t)gridDim.x * blockDim.x;
  for (int a = 0; a < L.n; ++a)
    for (uint64_t i = tid; i < (L.bytes[a] + 15) / 16; i += step) ((uint4*)L.to[a])[i] = ((const uint4*)L.from[a])[i];
}

unsigned grid_for(uint64_t items, unsigned per_block, unsigned cap) {
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((items + per_block - 1) / per_block, cap));
}

#define PD_LAUNCH(L, name, ...)             \
  do {                                      \
    cudaError_t e_ = launch_begin(L, name); \
    if (e_ != cudaSuccess) return e_;       \
    __VA_ARGS__;                            \
    e_ = launch_end(L, name);               \
    if (e_ != cudaSuccess) return e_;       \
  } while (0)

// Digit bits of pass p: at least 5 (the bits past the key's are zero).
uint32_t pass_bits(const SortKey& K, uint32_t p) {
  return std::max<uint32_t>(5u, p + 1 < K.passes ? K.width : K.code_bits - K.skip - (K.passes - 1) * K.width);
}

// Calls f with the digit bits as a compile-time constant.
template <typename F>
cudaError_t with_bits(uint32_t bits, F f) {
  switch (bits) {
    case 5: return f(std::integral_constant<int, 5>());
    case 6: return f(std::integral_constant<int, 6>());
    case 7: return f(std::integral_constant<int, 7>());
    case 8: return f(std::integral_constant<int, 8>());
    default: return f(std::integral_constant<int, 9>());
  }
}

template <typename T>
cudaError_t sort_passes(Launcher* L, const WindowSource& S, const SortKey& K, uint64_t n, uint8_t* scratch,
                        const SortScratch& X, u64* a, u64* b, u64** sorted, DevErr* err, cudaStream_t s) {
  const size_t smem = (size_t)kTile * sizeof(u64);
  uint32_t* ticket = (uint32_t*)(scratch + X.tickets);
  u64 *src = a, *dst = a;
  for (uint32_t p = 0; p < K.passes; ++p) {
    const uint32_t shift = K.gene_bits + K.skip + p * K.width;
    T* status = (T*)(scratch + X.pass[p]);
    const uint32_t* hist = (const uint32_t*)(scratch + X.hist) + p * kMaxBins;
    const cudaError_t e = with_bits(pass_bits(K, p), [&](auto w) -> cudaError_t {
      constexpr int kBits = decltype(w)::value;
      cudaError_t e1;
      if (p == 0) {
        // 32-bit codes for all but the longest k-mers and the largest segmented inputs
        auto kernel = K.total_bits <= 32 ? k_sort_windows<kBits, T, uint32_t> : k_sort_windows<kBits, T, u64>;
        if ((e1 = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
          return e1;
        PD_LAUNCH(L, "sort_windows", kernel<<<sort_tiles(S.n_windows), kThreads, smem, s>>>(S, K, hist, status,
                                                                                            ticket + p, dst, err));
      } else {
        if ((e1 = cudaFuncSetAttribute(k_sort_records<kBits, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem)) != cudaSuccess)
          return e1;
        PD_LAUNCH(L, "sort_records", k_sort_records<kBits, T><<<sort_tiles(n), kThreads, smem, s>>>(
                                         src, n, shift, hist, status, ticket + p, dst, err));
      }
      return cudaSuccess;
    });
    if (e != cudaSuccess) return e;
    src = dst;
    dst = dst == a ? b : a;
  }
  *sorted = src;
  return cudaSuccess;
}

}  // namespace

SortKey sort_key(uint64_t n_codes, uint32_t gene_bits, uint32_t skip) {
  SortKey K{};
  uint32_t bits = 1;
  while (bits < 63 && ((n_codes - 1) >> bits) != 0) ++bits;
  K.gene_bits = gene_bits;
  // codes that do not fit the record next to the gene are sorted in slices of
  // equal high bits, one after the other
  const uint32_t most = 64u - gene_bits;
  K.total_bits = bits;
  K.code_bits = std::min(bits, most);
  K.n_slices = bits > most ? 1u << (bits - most) : 1u;
  K.skip = skip;
  const uint32_t sorted = K.code_bits - skip;
  K.passes = (sorted + 8) / 9;
  K.width = (sorted + K.passes - 1) / K.passes;
  K.last_mask = (1u << (sorted - (K.passes - 1) * K.width)) - 1u;
  return K;
}

uint32_t sort_tiles(uint64_t n) { return (uint32_t)((n + kTile - 1) / kTile); }
static uint32_t dedupe_tiles(uint64_t n) { return (uint32_t)((n + kDTile - 1) / kDTile); }
uint32_t list_tiles(uint64_t n) { return kHalves * dedupe_tiles(n); }
// Zeroed scratch of one slice: tickets, digit counts, look-back statuses.
SortScratch sort_scratch(const SortKey& K, uint64_t n) {
  SortScratch x{};
  const uint64_t nt = sort_tiles(n), nd = dedupe_tiles(n);
  x.wide = n >= (1ull << 30);
  x.tickets = 0;
  x.hist = 64;
  size_t at = x.hist + kMaxSortPasses * kMaxBins * sizeof(uint32_t);
  x.dedupe = at;
  at += 2 * nd * sizeof(u64);
  for (uint32_t p = 0; p < K.passes; ++p) {
    x.pass[p] = at;
    at += (nt << pass_bits(K, p)) * (x.wide ? sizeof(u64) : sizeof(uint32_t));
  }
  x.bytes = at;
  return x;
}

cudaError_t run_gene_windows(Launcher* L, const int64_t* gene_ptr, uint32_t n_genes, uint64_t n_res, int check_end,
                             int k, const int32_t* genome_ptr, uint32_t n_genomes, uint32_t* La, uint16_t* gene_genome,
                             uint32_t* ginfo, uint32_t* minhash, uint32_t* mv_n, DevErr* err, cudaStream_t s) {
  PD_LAUNCH(L, "gene_windows", k_gene_windows<<<grid_for(n_genes, 256, 152u * 8u), 256, 0, s>>>(
                                   gene_ptr, n_genes, n_res, check_end, k, genome_ptr, n_genomes, La, gene_genome,
                                   ginfo, minhash, mv_n, err));
  return cudaSuccess;
}

cudaError_t run_check_letters(Launcher* L, const uint8_t* res, uint64_t n_res, const int64_t* gene_ptr,
                              const int64_t* gene_src, uint32_t n_genes, int alpha, DevErr* err, cudaStream_t s) {
  if (gene_src)
    PD_LAUNCH(L, "check_letters", k_check_letters_genes<<<grid_for((uint64_t)n_genes * 32, 256, 152u * 8u), 256, 0, s>>>(
                                      res, gene_ptr, gene_src, n_genes, alpha, err));
  else if (n_res)
    PD_LAUNCH(L, "check_letters",
              k_check_letters<<<grid_for(n_res, 4096, 152u * 8u), 256, 0, s>>>(res, n_res, alpha, err));
  return cudaSuccess;
}

cudaError_t run_tile_genes(Launcher* L, const uint32_t* win_off, uint32_t n_genes, uint64_t n_windows,
                           uint32_t* tile_gene, uint32_t* cursor, cudaStream_t s) {
  PD_LAUNCH(L, "tile_genes", k_tile_genes<<<grid_for(n_genes, 256, 152u * 8u), 256, 0, s>>>(
                                 win_off, n_genes, sort_tiles(n_windows), tile_gene, cursor));
  return cudaSuccess;
}

namespace {
template <typename Code>
void launch_code_hist(const WindowSource& S, const SortKey& K, uint32_t n_tiles, uint32_t* hist, uint32_t* minhash,
                      cudaStream_t s) {
  const unsigned grid = grid_for(n_tiles, 1, 152u * 4u);
  switch (K.passes) {
    case 1: k_code_hist<Code, 1><<<grid, kThreads, 0, s>>>(S, K, n_tiles, hist, minhash); break;
    case 2: k_code_hist<Code, 2><<<grid, kThreads, 0, s>>>(S, K, n_tiles, hist, minhash); break;
    case 3: k_code_hist<Code, 3><<<grid, kThreads, 0, s>>>(S, K, n_tiles, hist, minhash); break;
    default: k_code_hist<Code, 4><<<grid, kThreads, 0, s>>>(S, K, n_tiles, hist, minhash); break;
  }
}
}  // namespace

cudaError_t run_code_hist(Launcher* L, const WindowSource& S, const SortKey& K, uint8_t* scratch,
                          const SortScratch& X, uint32_t* minhash, cudaStream_t s) {
  const uint32_t n_tiles = sort_tiles(S.n_windows);
  uint32_t* hist = (uint32_t*)(scratch + X.hist);
  PD_LAUNCH(L, "code_hist", (K.total_bits <= 32 ? launch_code_hist<uint32_t>(S, K, n_tiles, hist, minhash, s)
                                                : launch_code_hist<u64>(S, K, n_tiles, hist, minhash, s)));
  return cudaSuccess;
}

cudaError_t run_sort(Launcher* L, const WindowSource& S, const SortKey& K, uint64_t n, uint8_t* scratch,
                     const SortScratch& X, u64* a, u64* b, u64** sorted, DevErr* err, cudaStream_t s) {
  return X.wide ? sort_passes<u64>(L, S, K, n, scratch, X, a, b, sorted, err, s)
                : sort_passes<uint32_t>(L, S, K, n, scratch, X, a, b, sorted, err, s);
}

cudaError_t run_dedupe(Launcher* L, const u64* rec, uint64_t n, const SortKey& K, uint8_t* scratch,
                       const SortScratch& X, uint32_t cnt_bits, uint32_t cnt_cap, u64* totals, uint32_t* post,
                       uint32_t* post_ptr, uint32_t* code_lo, uint8_t* code_hi, uint32_t* tile_e, uint32_t* tile_id,
                       uint32_t* mv_n, DevErr* err, cudaStream_t s) {
  const uint32_t nt = dedupe_tiles(n);
  u64* status = (u64*)(scratch + X.dedupe);
  // totals[2..3]: the postings and ids of the slices before
  if (K.slice) {
    cudaError_t e = cudaMemcpyAsync(totals + 2, totals, 2 * sizeof(u64), cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
  }
  auto kernel = mv_n ? k_dedupe<true> : k_dedupe<false>;
  PD_LAUNCH(L, "dedupe",
            kernel<<<nt, kDThreads, 0, s>>>(rec, n, K, nt, cnt_bits, cnt_cap, status, status + nt,
                                              (uint32_t*)(scratch + X.tickets) + kMaxSortPasses, totals, post, post_ptr,
                                              code_lo, code_hi, tile_e, tile_id, mv_n, err));
  return cudaSuccess;
}

cudaError_t run_pack(Launcher* L, const PackList& list, cudaStream_t s) {
  uint64_t most = 0;
  for (int a = 0; a < list.n; ++a) most = std::max(most, list.bytes[a]);
  PD_LAUNCH(L, "pack", k_pack<<<grid_for(most, 4096, 152u * 8u), 256, 0, s>>>(list));
  return cudaSuccess;
}

cudaError_t run_lists(Launcher* L, const u64* rec, uint64_t n, const SortKey& K, const uint32_t* tile_e,
                      const uint32_t* tile_id, const uint32_t* post, const uint32_t* post_ptr, const uint32_t* code_lo,
                      const uint8_t* code_hi, uint32_t cnt_bits, uint32_t cnt_cap, const int32_t* genome_ptr,
                      uint32_t n_genomes, uint32_t n_genes, uint32_t* cursor, uint4* mv, uint32_t* max_list, u64* join,
                      const DevErr* err, cudaStream_t s) {
  const uint32_t nt = list_tiles(n);
  uint32_t table_bits = 0;
  while (((n_genes - 1) >> table_bits) >= kGenomeTable) ++table_bits;
  const size_t smem = sizeof(int32_t) * n_genomes;  // at most 16 KB: beside the static arrays no attribute is needed
  PD_LAUNCH(L, "lists", k_lists<<<std::min(nt, 152u * 3u), kDThreads, smem, s>>>(
                            tile_e, tile_id, nt, rec, n, K, code_lo, code_hi, post, post_ptr, cnt_bits, cnt_cap,
                            genome_ptr, n_genomes, n_genes, table_bits, cursor, mv, max_list, join, err));
  return cudaSuccess;
}

}  // namespace pdg
