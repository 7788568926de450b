// k_summin.cu -- sum-min by inverted-index scatter, fused with Best Hit
// selection ("Best Hit detection phase", Algorithm 2, Eqs. (5) and (8)).
//
// One thread block owns one query gene a at a time:
//   1. stage a chunk of a's multiplicity vector in shared memory: for each
//      k-mer its multiplicity and posting range (stored with the vector, so
//      this read is coalesced; in the pair forms the range is narrowed by
//      binary search to the target genome, in the symmetric all-pairs form to
//      the genomes after a's own), and a block prefix sum of the range
//      lengths: the chunk's postings form one flat index space;
//   2. walk the postings, one of two ways chosen per launch: the merge-path
//      walk (thread t takes the flat range [t*P, (t+1)*P), finds its first
//      k-mer by one binary search and advances sequentially, four postings
//      loaded before any is used) or the warp-cooperative walk (each warp
//      reads 32 consecutive flat positions per round, the k-mer of each lane
//      found from the staged list starts by a warp OR-reduction); each
//      posting (b, mult_b) adds min(mult_a, mult_b) to b's accumulator in
//      shared memory: an open-addressing hash, or direct slots when the
//      query's targets are one gene range that fits the table.  After all
//      chunks acc[b] = s(a, b), the Eq. (5) numerator, exactly;
//   3. Best Hits: per target genome the maximum ratio s / (La + Lb - s) is
//      kept as an (s, den) pair updated by compare-and-swap under a 64-bit
//      cross-multiplication order; every accumulator whose ratio equals its
//      genome's maximum (again by cross-multiplication) is a Best Hit (Eq. (8),
//      ties kept).  The second pass also clears the slots it reads, so the
//      table is clean for the next query.  Each hit is written at its rank
//      among the query's hits (ascending gene): rows come out sorted without a
//      sorting network.
// In the symmetric all-pairs form each candidate b also keeps, in global
// memory, its best ratio over a's genome (the column maximum of Algorithm 3,
// with exact ties listed), from which k_sym.cu assembles the reverse rows.
// Served queries (new genomes against a resident set) may limit the targets
// to genes below a bound, and may also keep each target's best ratio over the
// query's genome in global memory (the reverse-direction maximum needed for
// the mutual check of Eq. (9)).
// The similarity matrix S_ij is never materialised: only pairs sharing a
// k-mer are touched.  Where queries are many, one warp each takes those that
// meet few targets (the warp tier below); blocks take the others.  A query
// whose insertions probe too far (a nearly full table), or whose Best Hit list
// does not fit, is deferred to the next tier: 4096 slots in shared memory (256
// threads) -> 16384 slots in shared memory (1024 threads, one block per SM) ->
// a global-memory table sized for every possible target.  Results are exact
// and independent of the tier.
#include <algorithm>

#include "pd_internal.cuh"

namespace pdg {
namespace {

struct Scalars {
  uint32_t n_out;
  uint32_t overflow;
  uint32_t base_lo, base_hi;
  uint32_t warp_tmp[33];
};


// Probes allowed before a query counts as overflowing its table.  Long chains
// mean a nearly full table; the query then moves to a larger tier, so the
// bound never changes a result, only where it is computed.
constexpr uint32_t kMaxProbe = 64;
// Two table layouts share the code below.
//   packed (tier 1): one word per slot, (b << cnt_bits) | s.  A posting is
//     packed the same way, so the walk keys the table with the posting's own
//     high bits ("bkey") and never unpacks the gene id.  Valid while s stays
//     below the all-ones count, which holds for every query with
//     La < 2^cnt_bits - 1 (s <= La); other queries go to tier 2.  The gene
//     field never holds all ones (that id is reserved), so the empty word
//     0xFFFFFFFF matches no key.
//   split (tiers 2 and 3): keys[] = b, vals[] = s.
// Slots are found by multiplicative hashing (top bits of key * odd constant)
// and linear probing.
template <bool kPacked, bool kFilter = false>
struct Acc {
  uint32_t* keys;  // packed: slot words
  uint32_t* vals;  // split only
  // filtered only: the sums of mult_a and of mult_b over the shared k-mers (Eq.
  // (7) numerators, a -> b and b -> a); packed: both in vpa, mult_b's above
  // 16 bits (each is at most its gene's windows, below 2^16)
  uint32_t* vpa;
  uint32_t* vpb;
  uint32_t cnt_bits;
  uint32_t hash_shift;  // 32 - log2(cap)
  // Target genes [dense_lo, dense_lo + cap) of a query whose targets fit the
  // table: slot = gene - dense_lo (direct, the first probe always lands);
  // kEmpty: hashed slots.
  uint32_t dense_lo;

  __device__ __forceinline__ void bump(uint32_t h, uint32_t m, uint32_t ca, uint32_t cb) const {
    atomicAdd(&vals[h], m);
    if (kFilter) {
      atomicAdd(&vpa[h], ca);
      atomicAdd(&vpb[h], cb);
    }
  }

  __device__ __forceinline__ uint32_t home(uint32_t key) const {
    if (dense_lo != kEmpty) return (kPacked ? key >> cnt_bits : key) - dense_lo;
    return (key * 0x9E3779B1u) >> hash_shift;
  }

  // key: bkey (packed) or b (split).  Returns false after kMaxProbe probes.
  // ca, cb (the two multiplicities) feed the directional sums of filtered queries.
  __device__ __forceinline__ bool add(uint32_t mask, uint32_t key, uint32_t m, uint32_t ca = 0,
                                      uint32_t cb = 0) const {
    uint32_t h = home(key);
    const uint32_t hi = ~((1u << cnt_bits) - 1u);
    for (uint32_t probe = 0; probe < kMaxProbe; ++probe) {
      const uint32_t k = *((volatile uint32_t*)&keys[h]);
      if (kPacked) {
        if ((k & hi) == key) {
          atomicAdd(&keys[h], m);
          if (kFilter) atomicAdd(&vpa[h], ca | cb << 16);
          return true;
        }
        if (k == kEmpty) {
          const uint32_t prev = atomicCAS(&keys[h], kEmpty, key | m);
          if (prev == kEmpty || (prev & hi) == key) {
            if (prev != kEmpty) atomicAdd(&keys[h], m);
            if (kFilter) atomicAdd(&vpa[h], ca | cb << 16);
            return true;
          }
        }
      } else {
        if (k == key) {
          bump(h, m, ca, cb);
          return true;
        }
        if (k == kEmpty) {
          const uint32_t prev = atomicCAS(&keys[h], kEmpty, key);
          if (prev == kEmpty || prev == key) {
            bump(h, m, ca, cb);
            return true;
          }
        }
      }
      h = (h + 1) & mask;
    }
    return false;
  }
  __device__ __forceinline__ bool occupied(uint32_t h) const { return keys[h] != kEmpty; }
  __device__ __forceinline__ void get(uint32_t h, uint32_t* b, uint32_t* s) const {
    const uint32_t k = keys[h];
    if (kPacked) {
      *b = k >> cnt_bits;
      *s = k & ((1u << cnt_bits) - 1u);
    } else {
      *b = k;
      *s = vals[h];
    }
  }
  __device__ __forceinline__ void sums(uint32_t h, uint32_t* pa, uint32_t* pb) const {
    *pa = kPacked ? vpa[h] & 0xFFFFu : vpa[h];
    *pb = kPacked ? vpa[h] >> 16 : vpb[h];
  }
  __device__ __forceinline__ void clear(uint32_t h) const {
    keys[h] = kEmpty;
    if (!kPacked) vals[h] = 0;
    if (kFilter) {
      vpa[h] = 0;
      if (!kPacked) vpb[h] = 0;
    }
  }
};

// Eqs. (6) and (7) as candidate masks: lengths |g| = La + k - 1 (a candidate
// shares a k-mer, so La >= 1 on both sides), directional sums against La.
__device__ __forceinline__ bool filter_pass(const QuerySet& Q, uint32_t k, uint32_t La_a, uint32_t La_b, uint32_t pa,
                                            uint32_t pb) {
  if (Q.theta_num) {
    const unsigned long long la = La_a + k - 1u, lb = La_b + k - 1u;
    if (la * Q.theta_den < (unsigned long long)Q.theta_num * lb) return false;
    if (lb * Q.theta_den < (unsigned long long)Q.theta_num * la) return false;
  }
  if (Q.tau_num) {
    if ((unsigned long long)pa * Q.tau_den < (unsigned long long)Q.tau_num * La_a) return false;
    if ((unsigned long long)pb * Q.tau_den < (unsigned long long)Q.tau_num * La_b) return false;
  }
  return true;
}

__device__ __forceinline__ uint32_t lower_bound_post(const uint32_t* __restrict__ post, uint32_t lo, uint32_t hi,
                                                     unsigned long long key) {
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if ((unsigned long long)post[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Max of (s, den) pairs by cross-multiplication, packed as s << 32 | den.
__device__ __forceinline__ void best_update(unsigned long long* slot, uint32_t s, uint32_t den) {
  unsigned long long old = *((volatile unsigned long long*)slot);
  const unsigned long long mine = ((unsigned long long)s << 32) | den;
  while (true) {
    const uint32_t os = (uint32_t)(old >> 32), od = (uint32_t)old;
    if (os != 0 && !ratio_greater(s, den, os, od)) return;
    const unsigned long long prev = atomicCAS(slot, old, mine);
    if (prev == old) return;
    old = prev;
  }
}

// Reverse-direction maximum of the symmetric form: the best (s, den) of
// target b over the query genome, with the query gene a that reaches it,
// packed s << 48 | den << 31 | a (s < 2^16, den < 2^17, a < 2^31); a pair
// that equals the stored maximum is listed as a tie (b << 32 | a, s).  Ties of
// a maximum later beaten stay in the list and are dropped when the rows are
// assembled.
// `old`: the stored word, read by the caller.
__device__ __forceinline__ void sym_update(const QuerySet& Q, unsigned long long* slot, unsigned long long old,
                                           uint32_t b, uint32_t a, uint32_t s, uint32_t den) {
  const unsigned long long mine =
      ((unsigned long long)s << 48) | ((unsigned long long)den << 31) | (unsigned long long)a;
  while (true) {
    if (old != 0ull) {
      const uint32_t os = (uint32_t)(old >> 48), od = (uint32_t)(old >> 31) & 0x1FFFFu;
      if (ratio_greater(os, od, s, den)) return;
      if (ratio_equal(os, od, s, den)) {
        const unsigned long long t = atomicAdd(Q.tie_count, 1ull);
        if (t < Q.tie_cap) {
          Q.tie_rec[2 * t] = ((unsigned long long)b << 32) | a;
          Q.tie_rec[2 * t + 1] = s;
        }
        return;
      }
    }
    const unsigned long long prev = atomicCAS(slot, old, mine);
    if (prev == old) return;
    old = prev;
  }
}

// Length field of a vector entry's z (the top bit marks lists holding another
// gene of the same genome).
constexpr uint32_t kListLength = 0x7FFFFFFFu;

// A query gene, its output row and its targets.
struct Query {
  uint32_t a, row;
  uint32_t own0, own1;  // all-pairs forms: genes that are no targets (its own genome)
  uint32_t tend;        // ... and those from here on
  uint32_t t0, t1;      // other forms: the target genes
  uint32_t col, self;   // column of the reverse maxima; a gene that is no target
  const uint32_t* mask; // target genomes (null: every other)
};

__device__ __forceinline__ bool wanted(const Query& q, uint32_t genome) {
  return !q.mask || ((q.mask[genome >> 5] >> (genome & 31u)) & 1u);
}

// Forms of a query set that a kernel may be compiled for: any of them, the
// symmetric all-pairs form, the plain one, one target range per query (no
// queries from outside the dataset but in the first).  The tiers that most
// queries pass know theirs: the others' branches cost them registers and
// instruction-cache misses (symmetric form, one kernel for all forms against
// its own: 50 genomes x 3000 genes 3.27 against 3.08 ms, 200 x 4000 24.4
// against 24.0, 23 x 1700 0.34 against 0.30).
enum Form { kAnyForm, kSymmetricForm, kAllPairsForm, kRangeForm };
template <int kForm>
__device__ __forceinline__ bool all_pairs(const QuerySet& Q) {
  return kForm == kAnyForm ? Q.all_pairs != 0 : kForm != kRangeForm;
}
template <int kForm>
__device__ __forceinline__ bool symmetric(const QuerySet& Q) {
  return kForm == kAnyForm ? Q.symbest != nullptr : kForm == kSymmetricForm;
}

// False if there is nothing to do for the query: another shard's, or a gene that is a target only.
template <int kForm>
__device__ __forceinline__ bool load_query(uint32_t qi, const ProfilesView& P, const QuerySet& Q, Query* q) {
  q->own0 = q->own1 = q->t0 = q->t1 = q->col = 0;
  q->tend = q->self = kEmpty;
  q->mask = nullptr;
  if (all_pairs<kForm>(Q)) {
    const uint32_t a = Q.order ? Q.order[qi] : Q.q0 + qi;
    if (Q.n_shards && a % Q.n_shards != Q.shard) return false;
    q->a = q->row = a;
    if (kForm == kAnyForm && Q.q_genome) {  // external query: no own genome among the targets
      const uint32_t x = Q.q_genome[a];
      q->own0 = q->own1 = kEmpty;
      if (Q.tgt_end) q->tend = Q.tgt_end[x];
      q->col = x;
    } else {
      const uint32_t gg = P.gene_genome[a];
      if (Q.two_genomes && (gg & 1u)) return false;  // no genome after its own: a target only
      q->own0 = (uint32_t)P.genome_ptr[gg];
      q->own1 = (uint32_t)P.genome_ptr[gg + 1];
      if (Q.two_genomes) q->tend = (uint32_t)P.genome_ptr[gg + 2];
      if (kForm == kAnyForm && Q.tgt_end) q->tend = Q.tgt_end[gg];
      if (Q.tgt_mask) q->mask = Q.tgt_mask + (size_t)gg * Q.mask_words;
      q->col = Q.two_genomes ? 0u : gg - Q.col_genome0;
    }
    return true;
  }
  q->row = qi;
  if (Q.q_gene) {
    q->a = Q.q_gene[qi];
    q->t0 = Q.q_t0[qi];
    q->t1 = Q.q_t1[qi];
  } else if (!all_pairs<kForm>(Q) && Q.paralog) {
    q->a = q->self = Q.q0 + qi;
    const uint32_t gg = P.gene_genome[q->a];
    q->t0 = (uint32_t)P.genome_ptr[gg];
    q->t1 = (uint32_t)P.genome_ptr[gg + 1];
  } else if (qi < Q.nA) {
    q->a = Q.qa0 + qi;
    q->t0 = Q.ta0;
    q->t1 = Q.ta1;
  } else {
    q->a = Q.qb0 + (qi - Q.nA);
    q->t0 = Q.tb0;
    q->t1 = Q.tb1;
  }
  return true;
}

// The part [lo, lo + len) of a vector entry's posting list that holds the
// query's targets.
template <int kForm>
__device__ __forceinline__ void narrow_list(const ProfilesView& P, const QuerySet& Q, const Query& q, const uint4& v,
                                            uint32_t* lo, uint32_t* len) {
  *lo = v.x;
  *len = v.z & kListLength;
  if (symmetric<kForm>(Q)) {  // the genomes after the query's own
    *lo += v.w;
    *len -= v.w;
  } else if (!all_pairs<kForm>(Q) && Q.paralog) {
    // its own genome: the entry says whether another gene of it is there, and where it ends
    const uint32_t end = v.x + v.w;
    if (v.z == *len) {
      *len = 0;
    } else {
      *lo = lower_bound_post(P.post, v.x, end, (unsigned long long)q.t0 << P.cnt_bits);
      *len = end - *lo;
    }
  } else if (!all_pairs<kForm>(Q)) {
    const uint32_t end = v.x + *len;
    *lo = lower_bound_post(P.post, v.x, end, (unsigned long long)q.t0 << P.cnt_bits);
    // few postings of a list lie in the range: its end is looked for from its
    // start, in steps that double (3000 + 6000 queries of a pair of 50 genomes
    // 0.174 ms, with a second bisection 0.195)
    const unsigned long long past = (unsigned long long)q.t1 << P.cnt_bits;
    uint32_t from = *lo, step = 1;
    while (from + step <= end && P.post[from + step - 1] < past) {
      from += step;
      step <<= 1;
    }
    *len = lower_bound_post(P.post, from, min(end, from + step - 1), past) - *lo;
  }
}

template <int kThreads>
struct Chunk {
  static constexpr uint32_t kSize = 2 * kThreads;  // query k-mers staged per round
  static constexpr uint32_t kItems = 2;
  // c_post (4 B), c_off (4 B, one more), c_cnt (2 B), c_ent (2 B) per k-mer
  static constexpr size_t kBytes =
      (((size_t)kSize * 4 + (size_t)(kSize + 1) * 4 + (size_t)kSize * 2 + (size_t)kSize * 2) + 15) & ~(size_t)15;
};

// Rounds of 32 postings a warp has in flight before accumulating them (the
// warp-cooperative walk), and the average posting-list length, weighted by
// use (a dataset's join over its vector entries), from which tier 1 takes
// that walk rather than the merge-path walk: a warp round then reads few
// lists, while for short lists each thread's run of postings stays within the
// sectors it has already loaded.
constexpr uint32_t kRounds = 4;
constexpr uint32_t kWarpWalkMinAvg = 16;
// ... and the smallest index (4-byte postings) for which the warp walk is
// taken: below a few L2 sizes the merge-path walk's runs of postings keep
// hitting the sectors they have already brought in.
constexpr uint64_t kWarpWalkMinIndexBytes = 512ull << 20;
// The warp tier pays when there are queries for several per resident warp (3648
// of them; whole calls, ms, blocks alone / warp tier too: 8 genomes x 1000 genes
// 0.28 / 0.36, 8 x 1500 0.27 / 0.26, 10 x 1600 0.31 / 0.28, 20 x 1000 0.41 / 0.32;
// of batched jobs, where half of the genes are queries, sum-min alone, 8000 genes
// 0.12 / 0.15, 16000 0.16 / 0.15), and for queries that meet few targets: those of one target range (paralogs of 180k genes 1.0 against 1.8
// ms), of short lists (39k queries of 23 genomes 0.33 against 0.50), and in
// the symmetric form those of few postings.  Where lists are long a query's
// vector length and the genes after its genome tell how many postings it will
// walk, and the ones of more than kWMaxPostings leave the warp tier at once,
// with a table that would have overflowed or a walk that a block does faster:
// both tiers' time, ms, warp tier for no / the short / every query:
//   50 genomes x 3000 genes 3.08 / 2.82 / 3.25, 30 x 2000 0.89 / 0.68 / -,
//   100 x 4000 7.70 / 7.23 / -, 200 x 4000 - / 24.2 / 24.8
// (1500 postings instead: 2.98 at 50 x 3000, 25.2 at 200 x 4000; 4000: 3.03
// and 24.4).  Queries of one target range are judged by the range's share of
// the dataset and leave at kWMaxRangePostings, since where lists are long most
// of their postings are another gene's (whole calls, ms, no limit / 2500 / 1250:
// three pairs of 3 genomes x 30000 genes, k = 5, 20.4 / 18.2 / 16.6; paralogs of
// 4 x 6000, k = 4, 9.9 / 6.6 / 6.6, of 20 x 9000, k = 5, 5.4 / 5.4 / 4.7).
// Without the symmetric form
// whole lists are walked and the warp tier takes short lists or, of an index
// far larger than L2, long ones; queries from outside the dataset stay with
// the blocks (16k queries of a served tick 0.25 ms more).
constexpr uint32_t kWarpTierMinQueries = 16384, kWarpTierMaxAvg = 8;
constexpr float kWMaxPostings = 2500.f, kWMaxRangePostings = 1250.f;
// Average list length from which two lanes rather than one share a list in the
// warp tier of the symmetric form (100 x 4000 7.23 against 7.94 ms, 50 x 3000,
// with lists of 12, 2.91 against 2.82; 60 x 3000, of 14, 3.57 against 3.48).
constexpr uint32_t kWPairMinAvg = 15;
// Target genomes from which a query's Best Hits are ranked through per-genome
// positions rather than pairwise.
constexpr uint32_t kRankByGenomeMin = 64;

// Memory of one call: table, the list of occupied slots (filled after the
// walk) and the hit list.
template <typename TIdx>
struct Table {
  uint32_t* keys;
  uint32_t* vals;          // split layout only
  uint32_t* vpa;           // filtered queries only
  uint32_t* vpb;
  TIdx* used;              // capacity used_cap
  unsigned long long* out; // capacity out_cap
  uint32_t cap;            // power of two, a multiple of the block size
  uint32_t out_cap;
  uint32_t used_cap;       // at most cap; a query with more occupied slots moves to the next tier
};

template <int kThreads, bool kEmitAll, bool kPacked, bool kFilter, typename TIdx, bool kWarpWalk, int kForm>
__device__ __forceinline__ void process_query(uint32_t qi, const ProfilesView& P, const QuerySet& Q,
                                              const HitsOut& O, const TierIO& T, DevErr* err,
                                              const Table<TIdx>& tb, uint32_t* c_post, uint32_t* c_off,
                                              uint16_t* c_cnt, unsigned long long* best, Scalars* sh) {
  constexpr uint32_t kChunk = Chunk<kThreads>::kSize, kItems = Chunk<kThreads>::kItems;
  Acc<kPacked, kFilter> acc{tb.keys, tb.vals, tb.vpa, tb.vpb, P.cnt_bits, 32u - (31u - (uint32_t)__clz(tb.cap)), kEmpty};
  uint16_t* c_ent = c_cnt + Chunk<kThreads>::kSize;  // chunk entry of each staged k-mer
  unsigned long long* out = tb.out;
  const uint32_t mask = tb.cap - 1u;
  Query q;
  if (!load_query<kForm>(qi, P, Q, &q)) return;  // not a query (uniform over the block)
  const uint32_t a = q.a, row = q.row, own0 = q.own0, own1 = q.own1, tend = q.tend, col = q.col, self = q.self;
  // one target range that fits the table: direct slots instead of hashing
  if (!all_pairs<kForm>(Q) && q.t1 > q.t0 && q.t1 - q.t0 <= tb.cap) acc.dense_lo = q.t0;
  // the query's own vector (its dataset's, or the external query arrays)
  const bool ext = kForm == kAnyForm && P.q_win_off != nullptr;
  const uint4* __restrict__ q_mv = ext ? P.q_mv : P.mv;
  const uint32_t m0 = (ext ? P.q_win_off : P.mv_off)[a], E = (ext ? P.q_mv_n : P.mv_n)[a];
  const uint32_t La_a = (ext ? P.q_La : P.La)[a];
  const uint32_t cnt_mask = (1u << P.cnt_bits) - 1u;
  const uint32_t tid = threadIdx.x;
  if (tid == 0) {
    sh->n_out = 0;
    // a packed slot holds s <= La_a: queries beyond the field go to tier 2
    sh->overflow = (kPacked && La_a >= cnt_mask) ? 1u : 0u;
  }
  __syncthreads();
  auto narrow = [&](const uint4& v, uint32_t& lo, uint32_t& len) { narrow_list<kForm>(P, Q, q, v, &lo, &len); };
  // the symmetric form walks targets only
  auto is_target = [&](uint32_t b) {
    if (kForm == kSymmetricForm) return true;
    if (kForm == kRangeForm) return b != self;
    return !((all_pairs<kForm>(Q) && ((b >= own0 && b < own1) || b >= tend)) || b == self);
  };
  unsigned long long walked = 0;
  const uint32_t lane = tid & 31u, warp = tid >> 5;
  constexpr uint32_t kWarps = kThreads / 32;
  for (uint32_t c0 = 0; c0 < E && !sh->overflow; c0 += kChunk) {
    const uint32_t n_in = min(kChunk, E - c0);
    // Each posting (b, mult_b) adds min(mult_a, mult_b) to b's accumulator.
    // Own-genome postings are accumulated too and dropped when the Best Hits
    // are chosen (a few slots per query), which keeps the walks free of
    // per-posting range tests.  `e` is the query's chunk entry of the k-mer.
    // False: the table is full, and the query leaves this tier.  A thread that
    // meets this ends its walk: every further gene that is not in the table would
    // cost it kMaxProbe probes more (tier 1, ms: 10 genomes x 2000 genes at k =
    // 4, where no query fits, 2.5 against 19.9; 400 x 150, k = 5, 23 against 50;
    // 200 x 4000, k = 7, where few overflow, the whole run 42.6 against 43.0).
    // Filtered queries walk on: the test costs theirs 1.5%.
    auto accumulate = [&](uint32_t p, uint32_t ca, uint32_t e) -> bool {
      uint32_t cb = p & cnt_mask;
      if (cb == P.cnt_cap && (kFilter || ca > cb)) cb = mv_count_of(P, p >> P.cnt_bits, q_mv[m0 + c0 + e].x);
      const uint32_t key = kPacked ? (p & ~cnt_mask) : (p >> P.cnt_bits);
      if (acc.add(mask, key, min(ca, cb), ca, cb)) return true;
      sh->overflow = 1;
      return false;
    };
    bool fits = true;
    if constexpr (kWarpWalk) {
      // ---- stage the chunk: posting ranges and their prefix sum.  Empty
      // ranges (the restricted forms narrow lists to a target genome) are
      // dropped, so the staged list starts strictly increase, as the walk's
      // k-mer lookup needs.
      uint32_t lo_loc[kItems], len_loc[kItems], cnt_loc[kItems];
      uint32_t my_sum = 0, my_n = 0;
#pragma unroll
      for (uint32_t r = 0; r < kItems; ++r) {
        const uint32_t e = tid * kItems + r;
        uint32_t lo = 0, len = 0;
        cnt_loc[r] = 0;
        if (e < n_in) {
          const uint4 v = q_mv[m0 + c0 + e];
          cnt_loc[r] = v.y;
          narrow(v, lo, len);
        }
        lo_loc[r] = lo;
        len_loc[r] = len;
        my_sum += len;
        my_n += len ? 1u : 0u;
      }
      uint32_t J_c, n_c;
      uint32_t run = block_exclusive_scan(my_sum, sh->warp_tmp, &J_c);
      uint32_t slot = block_exclusive_scan(my_n, sh->warp_tmp, &n_c);
#pragma unroll
      for (uint32_t r = 0; r < kItems; ++r) {
        const uint32_t e = tid * kItems + r;
        if (len_loc[r]) {
          c_post[slot] = lo_loc[r];
          c_cnt[slot] = (uint16_t)cnt_loc[r];
          c_ent[slot] = (uint16_t)e;
          c_off[slot] = run;
          ++slot;
        }
        run += len_loc[r];
      }
      if (tid == 0) c_off[n_c] = J_c;
      __syncthreads();
      walked += J_c;
      // ---- warp-cooperative walk.  Warp w takes the flat postings [x0, x1)
      // and reads them 32 consecutive positions per round, lane l position
      // xr + l, so a round reads one or a few lists contiguously.  The k-mer
      // of each lane's position comes from the starts of the next 32 staged
      // k-mers (one per lane): bit d of `starts` marks a k-mer starting d
      // positions after the round's first, and a lane's k-mer is the round's
      // first k-mer plus the number of starts at or before it.
      const uint32_t per_w = ((J_c + kWarps - 1) / kWarps + 31u) & ~31u;
      const uint32_t x0 = min(J_c, warp * per_w), x1 = min(J_c, x0 + per_w);
      if (x0 < x1) {
        uint32_t e_lo = 0, hi = n_c;  // the k-mer holding x0: last e with c_off[e] <= x0
        while (hi - e_lo > 1) {
          const uint32_t mid = (e_lo + hi) >> 1;
          if (c_off[mid] <= x0) e_lo = mid; else hi = mid;
        }
        for (uint32_t xb = x0; xb < x1; xb += 32u * kRounds) {
          uint32_t pv[kRounds], cav[kRounds], ev[kRounds];
#pragma unroll
          for (uint32_t u = 0; u < kRounds; ++u) {
            const uint32_t xr = xb + 32u * u, x = xr + lane;
            const uint32_t j = e_lo + 1u + lane;
            const uint32_t d = (j <= n_c && xr < x1) ? c_off[j] - xr : 0xFFFFFFFFu;
            const uint32_t starts = __reduce_or_sync(0xFFFFFFFFu, d < 32u ? (1u << d) : 0u);
            const uint32_t e = e_lo + __popc(starts & (0xFFFFFFFFu >> (31u - lane)));
            e_lo += __popc(starts) + (__ballot_sync(0xFFFFFFFFu, d == 32u) ? 1u : 0u);
            pv[u] = kEmpty;
            cav[u] = 0;
            ev[u] = 0;
            if (x < x1) {
              pv[u] = P.post[c_post[e] + (x - c_off[e])];
              cav[u] = c_cnt[e];
              ev[u] = c_ent[e];
            }
          }
#pragma unroll
          for (uint32_t u = 0; u < kRounds; ++u)
            if (fits && xb + 32u * u + lane < x1) fits = accumulate(pv[u], cav[u], ev[u]);
        }
      }
    } else {
      // ---- stage the chunk: posting ranges and their prefix sum
      uint32_t len_loc[kItems];
      uint32_t my_sum = 0;
#pragma unroll
      for (uint32_t r = 0; r < kItems; ++r) {
        const uint32_t e = tid * kItems + r;
        uint32_t len = 0;
        if (e < n_in) {
          const uint4 v = q_mv[m0 + c0 + e];
          uint32_t lo;
          narrow(v, lo, len);
          c_post[e] = lo;
          c_cnt[e] = (uint16_t)v.y;
        }
        len_loc[r] = len;
        my_sum += len;
      }
      uint32_t J_c;
      uint32_t run = block_exclusive_scan(my_sum, sh->warp_tmp, &J_c);
#pragma unroll
      for (uint32_t r = 0; r < kItems; ++r) {
        const uint32_t e = tid * kItems + r;
        if (e < n_in) c_off[e] = run;
        run += len_loc[r];
      }
      if (tid == 0) c_off[n_in] = J_c;
      __syncthreads();
      walked += J_c;
      // ---- merge-path walk: thread t takes the flat range [t*per,
      // (t+1)*per), finds its first k-mer by one binary search and then
      // advances sequentially, loading four postings before using any (a
      // thread's next postings mostly share the sector of its last one).
      const uint32_t per = (J_c + kThreads - 1) / kThreads;
      uint32_t x = min(J_c, tid * per);
      const uint32_t x_end = min(J_c, x + per);
      if (x < x_end) {
        uint32_t lo = 0, hi = n_in;
        while (hi - lo > 1) {
          const uint32_t mid = (lo + hi) >> 1;
          if (c_off[mid] <= x) lo = mid; else hi = mid;
        }
        uint32_t e = lo, e_end = c_off[lo + 1], base = c_post[lo] - c_off[lo], ca = c_cnt[lo];
        while (x < x_end) {
          uint32_t pv[4], cav[4], ev[4];
          uint32_t nb = 0;
#pragma unroll
          for (uint32_t j = 0; j < 4; ++j) {
            if (x < x_end) {
              while (x >= e_end) {
                ++e;
                e_end = c_off[e + 1];
                base = c_post[e] - c_off[e];
                ca = c_cnt[e];
              }
              pv[j] = P.post[base + x];
              cav[j] = ca;
              ev[j] = e;
              ++x;
              nb = j + 1;
            }
          }
#pragma unroll
          for (uint32_t j = 0; j < 4; ++j)
            if ((kFilter || fits) && j < nb) fits = accumulate(pv[j], cav[j], ev[j]);
          if (!kFilter && !fits) break;
        }
      }
    }
    __syncthreads();
  }

  bool overflow = sh->overflow != 0;
  const uint32_t n_best = all_pairs<kForm>(Q) ? P.n_genomes : 1u;
  // With few target genomes a row has few hits and ranking them pairwise is
  // cheaper than a block scan over the genomes.
  const bool by_genome = !kEmitAll && n_best >= kRankByGenomeMin;
  // Best Hits of each target genome, then (exclusive scan) the first output
  // position of each genome's hits: rows come out ordered by gene because
  // genes are numbered genome by genome
  uint32_t* hcnt = (uint32_t*)(best + n_best);
  // Slots are visited interleaved (slot = i * kThreads + tid: conflict-free).
  const uint32_t slots = tb.cap / kThreads;
  uint32_t n_occ = 0, pos = 0;
  if (!overflow) {
    // ---- count the occupied slots (block prefix sum over per-thread counts);
    // more than the list holds: the query moves to the next tier
    uint32_t n_mine = 0;
    for (uint32_t i = 0; i < slots; ++i) n_mine += acc.occupied(i * kThreads + tid) ? 1u : 0u;
    pos = block_exclusive_scan(n_mine, sh->warp_tmp, &n_occ);
    overflow = n_occ > tb.used_cap;  // uniform over the block
  }
  if (!overflow) {
    // ---- list them
    for (uint32_t i = 0; i < slots; ++i) {
      const uint32_t h = i * kThreads + tid;
      if (acc.occupied(h)) tb.used[pos++] = (TIdx)h;
    }
    __syncthreads();
    if (kEmitAll) {
      for (uint32_t u = tid; u < n_occ; u += kThreads) {
        const uint32_t h = tb.used[u];
        uint32_t b, s;
        acc.get(h, &b, &s);
        const uint32_t slot = atomicAdd(&sh->n_out, 1u);
        if (slot < tb.out_cap) out[slot] = ((unsigned long long)b << 32) | s;
        acc.clear(h);
      }
    } else {
      // ---- per target genome: the maximum ratio, then every entry at it
      for (uint32_t j = tid; j < n_best; j += kThreads) {
        best[j] = 0ull;
        if (by_genome) hcnt[j] = 0u;
      }
      __syncthreads();
      for (uint32_t u = tid; u < n_occ; u += kThreads) {
        uint32_t b, s;
        acc.get(tb.used[u], &b, &s);
        if (!is_target(b)) continue;
        const uint32_t gi = P.ginfo[b];
        if (!wanted(q, gi >> 16)) continue;
        if (kFilter) {
          uint32_t pa, pb;
          acc.sums(tb.used[u], &pa, &pb);
          if (!filter_pass(Q, P.k, La_a, gi & 0xFFFFu, pa, pb)) continue;
        }
        const uint32_t den = La_a + (gi & 0xFFFFu) - s;
        best_update(&best[all_pairs<kForm>(Q) ? (gi >> 16) : 0u], s, den);
        if (kForm == kAnyForm && Q.colbest) best_update(&Q.colbest[(size_t)b * Q.col_stride + col], s, den);
        if (symmetric<kForm>(Q)) {
          unsigned long long* slot = &Q.symbest[(size_t)col * P.n_genes + b];
          sym_update(Q, slot, *(volatile unsigned long long*)slot, b, a, s, den);
        }
      }
      __syncthreads();
      for (uint32_t u = tid; u < n_occ; u += kThreads) {
        const uint32_t h = tb.used[u];
        uint32_t b, s;
        acc.get(h, &b, &s);
        const uint32_t gi = P.ginfo[b];
        const unsigned long long bv = best[all_pairs<kForm>(Q) ? (gi >> 16) : 0u];
        uint32_t pa = 0, pb = 0;
        if (kFilter) acc.sums(h, &pa, &pb);
        if (is_target(b) && wanted(q, gi >> 16) &&
            (!kFilter || filter_pass(Q, P.k, La_a, gi & 0xFFFFu, pa, pb)) &&
            ratio_equal(s, La_a + (gi & 0xFFFFu) - s, (uint32_t)(bv >> 32), (uint32_t)bv)) {
          // s <= La <= 65535 and the genome < 65536: (b, genome, s) in one word
          const uint32_t g = all_pairs<kForm>(Q) ? (gi >> 16) : 0u;
          const uint32_t slot = atomicAdd(&sh->n_out, 1u);
          if (slot < tb.out_cap) out[slot] = ((unsigned long long)b << 32) | (g << 16) | s;
          if (by_genome) atomicAdd(&hcnt[g], 1u);
        }
        acc.clear(h);
      }
    }
  } else {
    // the walk stopped early, or the occupied slots do not fit the list: clear every slot
    for (uint32_t i = 0; i < slots; ++i) acc.clear(i * kThreads + tid);
  }
  __syncthreads();
  const uint32_t n_out = sh->n_out;
  if (overflow || n_out > tb.out_cap) {
    if (tid == 0) {
      if (T.def_list) {
        T.def_list[atomicAdd(T.def_count, 1u)] = qi;
      } else {
        raise_error(err, PD_ERR_INTERNAL, qi);  // the last tier holds every target
      }
      O.row_off[row] = 0;
      O.row_len[row] = 0;
    }
    __syncthreads();
    return;
  }
  if (by_genome) {
    // ---- first output position of each target genome's hits (exclusive
    // scan of the per-genome counts; each thread scans a run of genomes)
    const uint32_t per = (n_best + kThreads - 1) / kThreads;
    const uint32_t j0 = min(n_best, tid * per), j1 = min(n_best, j0 + per);
    uint32_t mine = 0;
    for (uint32_t j = j0; j < j1; ++j) mine += hcnt[j];
    uint32_t total;
    uint32_t run = block_exclusive_scan(mine, sh->warp_tmp, &total);
    for (uint32_t j = j0; j < j1; ++j) {
      const uint32_t c = hcnt[j];
      hcnt[j] = run;
      run += c;
    }
    if (tid == 0) hcnt[n_best] = total;
    __syncthreads();
  }
  // ---- append: each hit goes to its rank among the query's hits
  if (tid == 0) {
    const unsigned long long base = atomicAdd(O.cursor, (unsigned long long)n_out);
    sh->base_lo = (uint32_t)base;
    sh->base_hi = (uint32_t)(base >> 32);
    O.row_off[row] = base;
    O.row_len[row] = n_out;
    atomicAdd(O.walked, walked);
  }
  __syncthreads();
  const unsigned long long base = ((unsigned long long)sh->base_hi << 32) | sh->base_lo;
  if (base + n_out <= O.out_cap) {
    for (uint32_t t = tid; t < n_out; t += kThreads) {
      const unsigned long long v = out[t];
      const uint32_t b = (uint32_t)(v >> 32);
      uint32_t rank = 0, sv;
      if (!by_genome) {
        // rank = hits with a smaller gene id (the genome field sits below the
        // gene id, so comparing whole words orders by gene)
        for (uint32_t u = 0; u < n_out; ++u) rank += (out[u] < v) ? 1u : 0u;
        sv = kEmitAll ? (uint32_t)v : ((uint32_t)v & 0xFFFFu);
      } else {
        // the genome's first position, plus the tied hits of the same genome
        // with a smaller gene id (genomes with one Best Hit skip the loop)
        const uint32_t g = ((uint32_t)v >> 16) & 0xFFFFu;
        rank = hcnt[g];
        if (hcnt[g + 1] - rank > 1u)
          for (uint32_t u = 0; u < n_out; ++u) {
            const unsigned long long w = out[u];
            rank += ((((uint32_t)w >> 16) & 0xFFFFu) == g && (uint32_t)(w >> 32) < b) ? 1u : 0u;
          }
        sv = (uint32_t)v & 0xFFFFu;
      }
      O.out_b[base + rank] = b;
      O.out_s[base + rank] = sv;
    }
  }
  __syncthreads();
}

// ---- warp tier: one warp per query
// Most queries meet a few hundred targets, so a whole block spends more on its
// block-wide scans, table scans and barriers than on the postings.  Here one
// warp owns a query and a small table, and nothing waits for another warp:
//   * entries of the query's vector are staged 32 at a time in a ring;
//     groups of kGroup lanes take lists in turn, four postings a lane (one
//     16-byte load) at a step, a step's loads in flight while the postings of
//     the step before are accumulated;
//   * a posting looks at the two slots of its home bucket and adds to the one
//     that holds its gene; the others (first postings of a gene, the few whose
//     bucket is full) are put aside, and handled 32 together: probing, claiming
//     a slot and listing it;
//   * the Best Hit passes run over the listed slots only: the maxima of each
//     target genome, then the hits at the maximum counted per genome, whose
//     running sum is each genome's first position in the row.
// A query that lists more than kWUsed slots, or whose vector is longer than
// kWEntries, goes to the next tier.
constexpr uint32_t kWSlots = 1024, kWUsed = 832, kWEntries = 2048, kWPend = 160, kWRing = 64;
constexpr uint32_t kWBatch = 2;
constexpr int kWThreads = 128, kWWarps = kWThreads / 32;
// Target genomes up to which the warp tier runs (10 bytes each per warp).
constexpr uint32_t kWMaxGenomes = 512;
constexpr uint16_t kWHit = 0x8000u;  // mark of a listed slot that is a Best Hit
static_assert(kWSlots <= 0x8000u, "slot and mark share 16 bits");
static_assert(kWEntries <= 0x10000u && kWUsed < 0x10000u, "16-bit entries and counts");
__host__ __device__ constexpr size_t warp_tier_bytes(uint32_t n_best) {
  return ((size_t)kWSlots * 4 + kWRing * 12 + (size_t)n_best * 8 + (size_t)kWPend * 4 + 8 + (size_t)kWUsed * 2 +
          ((size_t)n_best + 1) * 2 + 15) & ~(size_t)15;
}

template <int kGroup, int kForm>
__global__ void __launch_bounds__(kWThreads, 6)
    k_summin_warp(ProfilesView P, QuerySet Q, HitsOut O, TierIO T, uint32_t* ticket, uint32_t n_best,
                  float avg_list) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  unsigned char* mine = smem + (size_t)warp * warp_tier_bytes(n_best);
  uint32_t* tab = (uint32_t*)mine;
  unsigned long long* best = (unsigned long long*)(tab + kWSlots);
  uint2* ring = (uint2*)(best + n_best);            // first and past-the-end posting
  uint32_t* ring_ce = (uint32_t*)(ring + kWRing);   // count | entry << 16
  uint32_t* n_pend = ring_ce + kWRing;
  uint32_t* pend = n_pend + 2;
  uint16_t* used = (uint16_t*)(pend + kWPend);
  uint16_t* hcnt = used + kWUsed;
  for (uint32_t h = lane; h < kWSlots; h += 32) tab[h] = kEmpty;
  if (lane == 0) *n_pend = 0;
  __syncwarp();
  constexpr uint32_t kAll = 0xFFFFFFFFu;
  const uint32_t cmask = (1u << P.cnt_bits) - 1u, hi = ~cmask, cap = P.cnt_cap;
  const uint32_t below = (1u << lane) - 1u;
  static_assert(kGroup == 1 || kGroup == 2, "lanes that share a list");
  constexpr uint32_t kFirst = kGroup == 1 ? 0xFFFFFFFFu : 0x55555555u;  // a lane of each group
  const uint32_t groups_below = kFirst & ((1u << (lane / kGroup * kGroup)) - 1u), part = (lane % kGroup) * 4u;
  const uint4* __restrict__ q_mv = P.mv;
  const uint32_t* __restrict__ post = P.post;
  static_assert(kWSlots == 2u << 9, "512 buckets of two slots");
  auto home = [](uint32_t key) { return ((key * 0x9E3779B1u) >> 22) & ~1u; };
  unsigned long long walked = 0;  // postings of the queries kept (another tier counts the others')
  for (;;) {
    uint32_t qi = 0;
    if (lane == 0) qi = atomicAdd(ticket, 1u);
    qi = __shfl_sync(kAll, qi, 0);
    if (qi >= Q.n_queries) break;
    Query q;
    if (!load_query<kForm>(qi, P, Q, &q)) continue;
    const uint32_t m0 = P.mv_off[q.a], E = P.mv_n[q.a];
    const uint32_t La_a = P.La[q.a];
    // a packed slot holds s <= La_a
    bool overflow = E > kWEntries || La_a >= cmask;
    // too many postings to be expected: of each list (avg_list; 0: not looked at)
    // the share of its genes that the query walks -- of the dataset's, or in a
    // batch, where a list holds the genes of one job, of the job's
    if (kForm != kAllPairsForm && avg_list > 0.f) {
      uint32_t walk = q.t1 - q.t0, of = P.n_genes;
      if (kForm == kSymmetricForm) {
        walk = (Q.two_genomes ? q.tend : P.n_genes) - q.own1;
        if (Q.two_genomes) of = q.tend - q.own0;
      }
      const float most = kForm == kRangeForm ? kWMaxRangePostings : kWMaxPostings;
      if ((float)E * avg_list * (float)walk > most * (float)of) overflow = true;
    }
    uint32_t n_used = 0, n_walked = 0;
    // Adds the postings put aside (words gene | min of the counts) in [from, to).
    auto flush = [&](uint32_t from, uint32_t to) {
      uint32_t claimed = kEmpty;
      bool lost = false;
      if (from + lane < to) {
        const uint32_t w = pend[from + lane], key = w & hi;
        uint32_t h = home(key), probe = 0;
        for (; probe < kMaxProbe; ++probe) {
          uint32_t k = *((volatile uint32_t*)&tab[h]);
          if (k == kEmpty) {
            k = atomicCAS(&tab[h], kEmpty, w);
            if (k == kEmpty) {
              claimed = h;
              break;
            }
          }
          if ((k & hi) == key) {
            atomicAdd(&tab[h], w & cmask);
            break;
          }
          h = (h + 1u) & (kWSlots - 1u);
        }
        lost = probe == kMaxProbe;
      }
      const uint32_t c = __ballot_sync(kAll, claimed != kEmpty);
      const uint32_t at = n_used + (uint32_t)__popc(c & below);
      if (claimed != kEmpty && at < kWUsed) used[at] = (uint16_t)claimed;
      n_used += (uint32_t)__popc(c);
      if (__any_sync(kAll, lost) || n_used > kWUsed) overflow = true;
      if (lane == 0) *n_pend = from;
      __syncwarp();
    };
    // ---- walk.  Ring: entries [taken, staged) wait; c0: the next ones of the vector.
    uint32_t staged = 0, taken = 0, c0 = 0;
    uint32_t at = 0, first = 0, end = 0, ce = 0;  // the group's list: next posting (a multiple of 4), bounds, count
    uint4 nv = make_uint4(0, 0, 0, 0);
    if (!overflow && lane < E) nv = q_mv[m0 + lane];
    auto stage = [&]() {  // 32 entries more, without those that have no targets
      uint32_t lo = 0, len = 0;
      if (c0 + lane < E) narrow_list<kForm>(P, Q, q, nv, &lo, &len);
      const uint32_t some = __ballot_sync(kAll, len != 0u);
      if (len) {
        const uint32_t x = (staged + (uint32_t)__popc(some & below)) & (kWRing - 1u);
        ring[x] = make_uint2(lo, lo + len);
        ring_ce[x] = nv.y | (c0 + lane) << 16;
      }
      staged += (uint32_t)__popc(some);
      n_walked += len;
      c0 += 32u;
      if (c0 + lane < E) nv = q_mv[m0 + c0 + lane];
      __syncwarp();
    };
    // Next step's postings (kEmpty where the lane has none) and their list's count.
    auto next = [&](uint4& p, uint32_t& c) {
      const uint32_t want = __ballot_sync(kAll, at >= end) & kFirst;
      if (at >= end) {
        const uint32_t x = taken + (uint32_t)__popc(want & groups_below);
        if (x < staged) {
          const uint2 t = ring[x & (kWRing - 1u)];
          ce = ring_ce[x & (kWRing - 1u)];
          first = t.x;
          end = t.y;
          at = t.x & ~3u;
        } else {
          at = end = 0;
        }
      }
      taken = min(staged, taken + (uint32_t)__popc(want));
      const uint32_t i = at + part;
      p = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
      if (i < end) {
        p = *reinterpret_cast<const uint4*>(post + i);
        if (i < first || i + 4u > end) {
          if (i < first) p.x = kEmpty;
          if (i + 1u < first || i + 1u >= end) p.y = kEmpty;
          if (i + 2u < first || i + 2u >= end) p.z = kEmpty;
          if (i + 3u >= end) p.w = kEmpty;
        }
      }
      c = ce;
      at += 4u * kGroup;
    };
    auto add = [&](const uint4& p, uint32_t c) {
      uint32_t w[4] = {p.x, p.y, p.z, p.w};
      const uint32_t ca = c & 0xFFFFu;
      unsigned long long k[4];
      uint32_t h[4], m[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h[j] = home(w[j] & hi);
        k[j] = *reinterpret_cast<volatile unsigned long long*>(&tab[h[j]]);
        m[j] = min(ca, w[j] & cmask);
      }
      // Counts that do not fit a posting.  No query that is kept has one (La_a <
      // cmask), but without the branch the compiler orders the loop in another
      // way: paralogs of 60 x 3000 genes 1.23 -> 1.15 ms, but 50 x 3000 6.04 -> 6.52
      // for the whole run, 23 x 1700 1.66 -> 1.73, 32 batched jobs 9.49 -> 9.77.
      if (ca > cap) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (w[j] != kEmpty && (w[j] & cmask) == cap)
            m[j] = min(ca, mv_count_of(P, w[j] >> P.cnt_bits, q_mv[m0 + (c >> 16)].x));
      }
      uint32_t miss = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t key = w[j] & hi;
        const bool f0 = (((uint32_t)k[j] ^ key) & hi) == 0u, f1 = (((uint32_t)(k[j] >> 32) ^ key) & hi) == 0u;
        if (w[j] != kEmpty) {
          if (f0 || f1) atomicAdd(&tab[h[j] + (f0 ? 0u : 1u)], m[j]);
          else miss |= 1u << j;
        }
      }
      if (miss) {
        uint32_t x = atomicAdd(n_pend, (uint32_t)__popc(miss));
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((miss >> j) & 1u) pend[x++] = (w[j] & hi) | m[j];
      }
      __syncwarp();
      for (uint32_t n = *(volatile uint32_t*)n_pend; n >= 32u; n -= 32u) flush(n - 32u, n);
    };
    if (!overflow && E) {
      stage();
      while (staged == 0 && c0 < E) stage();
      uint4 p, pn;
      uint32_t c, cn;
      next(p, c);
      while (!overflow) {
        while (staged - taken <= 32u && c0 < E) stage();
        const bool more = taken < staged || __any_sync(kAll, at < end);
        if (more) next(pn, cn);
        add(p, c);
        if (!more) break;
        p = pn;
        c = cn;
      }
      __syncwarp();
      const uint32_t n = *(volatile uint32_t*)n_pend;
      __syncwarp();
      if (n) flush(0, n);
    }
    if (overflow) {
      for (uint32_t h = lane; h < kWSlots; h += 32) tab[h] = kEmpty;
      if (lane == 0) {
        *n_pend = 0;
        T.def_list[atomicAdd(T.def_count, 1u)] = qi;
        O.row_off[q.row] = 0;
        O.row_len[q.row] = 0;
      }
      __syncwarp();
      continue;
    }
    walked += n_walked;
    // ---- per target genome: the maximum ratio, then the entries at it
    for (uint32_t j = lane; j <= n_best; j += 32) {
      if (j < n_best) best[j] = 0ull;
      hcnt[j] = 0u;
    }
    __syncwarp();
    auto is_target = [&](uint32_t b) {
      return kForm == kSymmetricForm || (kForm == kRangeForm ? b != q.self : b < q.own0 || b >= q.own1);
    };
    // kWBatch candidates a lane at a time, their gene words (and reverse
    // maxima) in flight together
    for (uint32_t u0 = lane; u0 < n_used; u0 += 32u * kWBatch) {
      uint32_t k[kWBatch], gi[kWBatch];
      unsigned long long old[kWBatch];
      bool live[kWBatch];
#pragma unroll
      for (uint32_t j = 0; j < kWBatch; ++j) {
        const uint32_t u = u0 + 32u * j;
        k[j] = u < n_used ? tab[used[u]] : 0u;
        live[j] = u < n_used && is_target(k[j] >> P.cnt_bits);
        gi[j] = live[j] ? P.ginfo[k[j] >> P.cnt_bits] : 0u;
      }
#pragma unroll
      for (uint32_t j = 0; j < kWBatch; ++j) {
        live[j] = live[j] && (kForm == kRangeForm || wanted(q, gi[j] >> 16));
        old[j] = 0ull;
        if (kForm == kSymmetricForm && live[j])
          old[j] = *(volatile unsigned long long*)&Q.symbest[(size_t)q.col * P.n_genes + (k[j] >> P.cnt_bits)];
      }
#pragma unroll
      for (uint32_t j = 0; j < kWBatch; ++j) {
        if (!live[j]) continue;
        const uint32_t b = k[j] >> P.cnt_bits, s = k[j] & cmask, den = La_a + (gi[j] & 0xFFFFu) - s;
        if (kForm == kSymmetricForm) sym_update(Q, &Q.symbest[(size_t)q.col * P.n_genes + b], old[j], b, q.a, s, den);
        best_update(&best[kForm != kRangeForm ? (gi[j] >> 16) : 0u], s, den);
      }
    }
    __syncwarp();
    for (uint32_t u0 = lane; u0 < n_used; u0 += 32u * kWBatch) {
      uint32_t h[kWBatch], k[kWBatch], gi[kWBatch];
      bool live[kWBatch];
#pragma unroll
      for (uint32_t j = 0; j < kWBatch; ++j) {
        const uint32_t u = u0 + 32u * j;
        h[j] = u < n_used ? used[u] : 0u;
        k[j] = tab[h[j]];
        live[j] = u < n_used && is_target(k[j] >> P.cnt_bits);
        gi[j] = live[j] ? P.ginfo[k[j] >> P.cnt_bits] : 0u;
      }
#pragma unroll
      for (uint32_t j = 0; j < kWBatch; ++j) {
        if (!live[j]) continue;
        const uint32_t s = k[j] & cmask, g = kForm != kRangeForm ? (gi[j] >> 16) : 0u;
        const unsigned long long bv = best[g];
        if ((kForm == kRangeForm || wanted(q, gi[j] >> 16)) &&
            ratio_equal(s, La_a + (gi[j] & 0xFFFFu) - s, (uint32_t)(bv >> 32), (uint32_t)bv)) {
          // 16-bit counts, two to a word
          atomicAdd((uint32_t*)((uintptr_t)&hcnt[g] & ~(uintptr_t)3), ((uintptr_t)&hcnt[g] & 2u) ? 0x10000u : 1u);
          used[u0 + 32u * j] = (uint16_t)(h[j] | kWHit);
        }
      }
    }
    __syncwarp();
    // ---- first position of each genome's hits in the row
    uint32_t n_out = 0;
    for (uint32_t j0 = 0; j0 <= n_best; j0 += 32) {
      const uint32_t c = j0 + lane < n_best ? hcnt[j0 + lane] : 0u;
      const uint32_t inc = warp_inclusive_scan(c);
      if (j0 + lane <= n_best) hcnt[j0 + lane] = (uint16_t)(n_out + inc - c);
      n_out += __shfl_sync(kAll, inc, 31);
    }
    unsigned long long base = 0;
    if (lane == 0) {
      base = atomicAdd(O.cursor, (unsigned long long)n_out);
      O.row_off[q.row] = base;
      O.row_len[q.row] = n_out;
    }
    base = __shfl_sync(kAll, base, 0);
    __syncwarp();
    const bool fits = base + n_out <= O.out_cap;
    for (uint32_t u = lane; u < n_used; u += 32) {
      const uint32_t w = used[u];
      if (!(w & kWHit) || !fits) continue;
      const uint32_t k = tab[w & (kWSlots - 1u)], b = k >> P.cnt_bits;
      const uint32_t g = kForm != kRangeForm ? (P.ginfo[b] >> 16) : 0u;
      uint32_t rank = hcnt[g];
      if (hcnt[g + 1] - rank > 1u)  // tied hits of one genome: by gene
        for (uint32_t x = 0; x < n_used; ++x) {
          if (!(used[x] & kWHit)) continue;
          const uint32_t y = tab[used[x] & (kWSlots - 1u)] >> P.cnt_bits;
          rank += y < b && (kForm == kRangeForm || (P.ginfo[y] >> 16) == g) ? 1u : 0u;
        }
      O.out_b[base + rank] = b;
      O.out_s[base + rank] = k & cmask;
    }
    __syncwarp();
    for (uint32_t u = lane; u < n_used; u += 32) tab[used[u] & (kWSlots - 1u)] = kEmpty;
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) walked += __shfl_xor_sync(kAll, walked, o);
  if (lane == 0 && walked) atomicAdd(O.walked, walked);
}

// ---- shared-memory tiers: [table][chunk | (used list, hits)][best]
template <int kThreads, uint32_t kCap, uint32_t kOutCap, bool kPacked, bool kFilter = false,
          uint32_t kUsedCap = kCap>
struct SmemTier {
  static_assert(kCap % kThreads == 0, "table must split evenly over the block");
  static_assert(kCap <= 65536, "slot indices are 16-bit");
  static_assert(kUsedCap <= kCap && kUsedCap % 8 == 0, "occupied-slot list");
  static constexpr size_t kTable = (size_t)kCap * (kPacked ? (kFilter ? 8 : 4) : (kFilter ? 16 : 8));
  static constexpr size_t kUsed = (size_t)kUsedCap * 2;
  static constexpr size_t kAfterWalk = kUsed + (size_t)kOutCap * 8;
  static constexpr size_t kUnion = Chunk<kThreads>::kBytes > kAfterWalk ? Chunk<kThreads>::kBytes : kAfterWalk;
  // per target genome: best ratio (8 B) and hit count / first position (4 B), one more position
  static constexpr size_t bytes(uint32_t n_best) { return kTable + kUnion + (size_t)(n_best ? n_best : 1) * 12 + 4; }
};

template <int kThreads, int kMinBlocks, uint32_t kCap, uint32_t kOutCap, bool kPacked, bool kEmitAll,
          bool kFilter = false, uint32_t kUsedCap = kCap, bool kWarpWalk = false, int kForm = kAnyForm>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_summin_smem(ProfilesView P, QuerySet Q, HitsOut O,
                                                                      TierIO T, DevErr* err) {
  using S = SmemTier<kThreads, kCap, kOutCap, kPacked, kFilter, kUsedCap>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Scalars sh;
  Table<uint16_t> tb;
  tb.keys = (uint32_t*)smem;
  tb.vals = kPacked ? nullptr : tb.keys + kCap;
  tb.vpa = kFilter ? (kPacked ? tb.keys : tb.vals) + kCap : nullptr;
  tb.vpb = kFilter && !kPacked ? tb.vpa + kCap : nullptr;
  tb.cap = kCap;
  tb.out_cap = kOutCap;
  tb.used_cap = kUsedCap;
  unsigned char* uni = smem + S::kTable;
  tb.used = (uint16_t*)uni;
  tb.out = (unsigned long long*)(uni + S::kUsed);
  uint32_t* c_post = (uint32_t*)uni;
  uint32_t* c_off = c_post + Chunk<kThreads>::kSize;
  uint16_t* c_cnt = (uint16_t*)(c_off + Chunk<kThreads>::kSize + 1);
  unsigned long long* best = (unsigned long long*)(uni + S::kUnion);
  for (uint32_t h = threadIdx.x; h < kCap; h += kThreads) {
    tb.keys[h] = kEmpty;
    if (!kPacked) tb.vals[h] = 0;
    if (kFilter) {
      tb.vpa[h] = 0;
      if (!kPacked) tb.vpb[h] = 0;
    }
  }
  __syncthreads();
  const uint32_t n = T.in_list ? *T.in_count : Q.n_queries;
  for (uint32_t x = blockIdx.x; x < n; x += gridDim.x)
    process_query<kThreads, kEmitAll, kPacked, kFilter, uint16_t, kWarpWalk, kForm>(T.in_list ? T.in_list[x] : x, P, Q, O, T, err, tb, c_post,
                                                         c_off, c_cnt, best, &sh);
}

// ---- global-memory tier: table, used list and hit list of each block in scratch
template <bool kEmitAll, bool kFilter = false>
__global__ void __launch_bounds__(256) k_summin_global(ProfilesView P, QuerySet Q, HitsOut O, TierIO T,
                                                       BigScratch B, DevErr* err) {
  constexpr int kThreads = 256;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Scalars sh;
  Table<uint32_t> tb;
  tb.keys = B.keys + (size_t)blockIdx.x * B.cap;
  tb.vals = B.vals + (size_t)blockIdx.x * B.cap;
  tb.vpa = kFilter ? B.vpa + (size_t)blockIdx.x * B.cap : nullptr;
  tb.vpb = kFilter ? B.vpb + (size_t)blockIdx.x * B.cap : nullptr;
  tb.used = B.used + (size_t)blockIdx.x * B.cap;
  tb.out = B.out + (size_t)blockIdx.x * B.out_cap;
  tb.cap = B.cap;
  tb.out_cap = B.out_cap;
  tb.used_cap = B.cap;
  uint32_t* c_post = (uint32_t*)smem;
  uint32_t* c_off = c_post + Chunk<kThreads>::kSize;
  uint16_t* c_cnt = (uint16_t*)(c_off + Chunk<kThreads>::kSize + 1);
  unsigned long long* best = (unsigned long long*)(smem + Chunk<kThreads>::kBytes);
  for (uint32_t h = threadIdx.x; h < B.cap; h += kThreads) {
    tb.keys[h] = kEmpty;
    tb.vals[h] = 0;
    if (kFilter) {
      tb.vpa[h] = 0;
      tb.vpb[h] = 0;
    }
  }
  __syncthreads();
  const uint32_t n = *T.in_count;
  for (uint32_t x = blockIdx.x; x < n; x += gridDim.x)
    process_query<kThreads, kEmitAll, false, kFilter, uint32_t, false, kAnyForm>(T.in_list[x], P, Q, O, T, err, tb, c_post, c_off, c_cnt, best,
                                                       &sh);
}

// Tier 1 (packed 4096-slot table, several blocks per SM) and tier 2 (split
// 16384-slot table, one 1024-thread block per SM) geometries.
constexpr int kT1Threads = 256, kT1MinBlocks = 6;
// Three tier-1 layouts, chosen per launch.  The compact one keeps six blocks
// within the 164 KB shared-memory carveout of an SM, which leaves 92 KB of
// the SM's 256 KB as L1 for the posting loads of the walk (with 4 KB more per
// block the carveout steps up to 196 KB and L1 shrinks to 60 KB): at most 3072
// listed occupied slots and 448 hits per query, a query beyond either moving
// to tier 2.  Past kT1CompactGenomes target genomes the per-genome maxima (12
// bytes each) no longer leave room for that; the middle layout lists at most
// 2048 occupied slots and 384 hits and stays within 164 KB up to
// kT1MidGenomes genomes.  Past that the full layout (4096 slots listed, 512
// hits) takes the blocks that fit 164 KB, five at first: as many as fit the SM
// would leave 28 KB of L1, which the walk's loads overrun (300 genomes x 600
// genes 19.9 against 10.5 ms, 500 x 400 22.6 against 11.5).
constexpr uint32_t kT1Cap = 4096, kT1OutEmit = 3072;
constexpr uint32_t kT1Out = 448, kT1Used = 3072;          // compact layout
constexpr uint32_t kT1OutFull = 512, kT1UsedFull = 4096;  // full layout
constexpr uint32_t kT1FullCarveout = 164;
constexpr uint32_t kT1UsedMid = 2048, kT1OutMid = 384;    // middle layout
constexpr int kT2Threads = 1024;
constexpr uint32_t kT2Cap = 16384, kT2Out = 2048, kT2OutEmit = 4096;
using T1 = SmemTier<kT1Threads, kT1Cap, kT1Out, true, false, kT1Used>;
using T1F = SmemTier<kT1Threads, kT1Cap, kT1OutFull, true, false, kT1UsedFull>;
using T1M = SmemTier<kT1Threads, kT1Cap, kT1OutMid, true, false, kT1UsedMid>;
using T1E = SmemTier<kT1Threads, kT1Cap, kT1OutEmit, true, false, kT1Used>;
// genomes up to which six compact blocks (with their static scalars and the
// 1 KB the runtime reserves per block) fit a 164 KB carveout
constexpr uint32_t kT1CompactGenomes =
    (uint32_t)((164u * 1024u / kT1MinBlocks - 1024u - sizeof(Scalars) - T1::kTable - T1::kUnion - 4u) / 12u);
static_assert(kT1CompactGenomes >= 50, "compact tier-1 layout holds tens of genomes");
// ... and six middle-layout blocks (a shorter occupied-slot list)
constexpr uint32_t kT1MidGenomes =
    (uint32_t)((164u * 1024u / kT1MinBlocks - 1024u - sizeof(Scalars) - T1M::kTable - T1M::kUnion - 4u) / 12u);
static_assert(kT1MidGenomes >= 200, "middle tier-1 layout holds hundreds of genomes");
using T2 = SmemTier<kT2Threads, kT2Cap, kT2Out, false>;
using T2E = SmemTier<kT2Threads, kT2Cap, kT2OutEmit, false>;
static_assert(T1F::bytes(PD_MAX_GENOMES) <= 227 * 1024, "tier 1 shared memory");
static_assert(T2::bytes(PD_MAX_GENOMES) <= 227 * 1024, "tier 2 shared memory");
static_assert(T2E::bytes(1) <= 227 * 1024, "tier 2 (emit-all, one target genome) shared memory");
// Filtered queries (Eqs. (6)-(7)): packed 4096-slot table, the two directional
// sums in one more word a slot; what does not fit goes to a split table of as
// many slots, then straight to the global tier.  Four blocks in a 196 KB
// carveout, which leaves 60 KB of L1 for the walk: 60 k queries of 30 genomes
// 1.02 ms, five blocks with 28 KB of L1 1.13, three with 92 KB 1.22 (a split
// table's two blocks, walking from both sides, 2.1 against 1.7 of the packed).
constexpr int kF1MinBlocks = 4;
constexpr uint32_t kF1Carveout = 196;
constexpr uint32_t kF1Cap = 4096, kF1Used = 2560, kF1Out = 448;
using TF1 = SmemTier<256, kF1Cap, kF1Out, true, true, kF1Used>;
static_assert(TF1::bytes(PD_MAX_GENOMES) <= 227 * 1024, "filtered tier shared memory");
constexpr int kFThreads = 256, kFMinBlocks = 2;
constexpr uint32_t kFCap = 4096, kFOut = 512;
using TF = SmemTier<kFThreads, kFCap, kFOut, false, true>;
static_assert(TF::bytes(PD_MAX_GENOMES) <= 227 * 1024, "filtered tier shared memory");

// Tier: the kernel's SmemTier; n_best: target genomes of the launch, at most
// kMaxBest.  A function's attributes are shared by every context and host
// thread, so the limit set is always the kernel's largest: another thread's
// launch between the two calls then finds room for its own size.  carveout (KB,
// 0: what the resident blocks take): shared memory of an SM to stay within,
// the rest being L1.
template <typename Tier, uint32_t kMaxBest = PD_MAX_GENOMES, typename K>
cudaError_t launch_smem(K kernel, Launcher* L, const char* name, int threads, uint32_t n_best, uint32_t max_grid,
                        const ProfilesView& P, const QuerySet& Q, const HitsOut& O, const TierIO& T, DevErr* err,
                        cudaStream_t s, uint32_t carveout = 0) {
  const size_t smem = Tier::bytes(n_best);
  cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tier::bytes(kMaxBest));
  if (e != cudaSuccess) return e;
  if (carveout && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            (int)(carveout * 100 / 228))) != cudaSuccess)
    return e;
  int per_sm = 1, dev = 0, n_sm = 152;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  if (carveout) per_sm = std::min<int>(per_sm, (int)(carveout * 1024u / (smem + 1024u + sizeof(Scalars))));
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t grid = std::max<uint32_t>(1, std::min<uint32_t>(max_grid, (uint32_t)n_sm * std::max(per_sm, 1)));
  if ((e = launch_begin(L, name)) != cudaSuccess) return e;
  kernel<<<grid, threads, smem, s>>>(P, Q, O, T, err);
  return launch_end(L, name);
}

// Tier 1 in the layout for n_best target genomes.
template <bool kWarpWalk, int kForm>
cudaError_t launch_t1(Launcher* L, uint32_t n_best, const ProfilesView& P, const QuerySet& Q, const HitsOut& O,
                      const TierIO& T, DevErr* err, cudaStream_t s) {
  constexpr int t = kT1Threads, b = kT1MinBlocks;
  if (n_best <= kT1CompactGenomes)
    return launch_smem<T1, kT1CompactGenomes>(k_summin_smem<t, b, kT1Cap, kT1Out, true, false, false, kT1Used, kWarpWalk, kForm>, L, "summin_bh",
                       t, n_best, Q.n_queries, P, Q, O, T, err, s);
  if (n_best <= kT1MidGenomes)
    return launch_smem<T1M, kT1MidGenomes>(k_summin_smem<t, b, kT1Cap, kT1OutMid, true, false, false, kT1UsedMid, kWarpWalk, kForm>, L,
                       "summin_bh", t, n_best, Q.n_queries, P, Q, O, T, err, s);
  return launch_smem<T1F>(k_summin_smem<t, b, kT1Cap, kT1OutFull, true, false, false, kT1UsedFull, kWarpWalk, kForm>, L,
                     "summin_bh", t, n_best, Q.n_queries, P, Q, O, T, err, s, kT1FullCarveout);
}

}  // namespace

cudaError_t run_summin_tiers(Launcher* L, const ProfilesView& P, const QuerySet& Q, const HitsOut& O, DevErr* err,
                             bool emit_all, cudaStream_t s) {
  if (Q.n_queries == 0) return cudaSuccess;
  const uint32_t n_best = Q.all_pairs ? P.n_genomes : 1u;
  if (Q.filter) {
    if (emit_all) return cudaErrorInvalidValue;
    TierIO tf1{nullptr, nullptr, O.def0, O.n_def0}, tf{O.def0, O.n_def0, O.def2, O.n_def2};
    const cudaError_t e1 =
        Q.symbest ? launch_smem<TF1>(k_summin_smem<256, kF1MinBlocks, kF1Cap, kF1Out, true, false, true, kF1Used, false,
                                              kSymmetricForm>,
                                L, "summin_bh_f1", 256, n_best, Q.n_queries, P, Q, O, tf1, err, s, kF1Carveout)
                  : launch_smem<TF1>(k_summin_smem<256, kF1MinBlocks, kF1Cap, kF1Out, true, false, true, kF1Used>, L,
                                "summin_bh_f1", 256, n_best, Q.n_queries, P, Q, O, tf1, err, s, kF1Carveout);
    if (e1 != cudaSuccess) return e1;
    return launch_smem<TF>(k_summin_smem<kFThreads, kFMinBlocks, kFCap, kFOut, false, false, true>, L, "summin_bh_f",
                       kFThreads, n_best, Q.n_queries, P, Q, O, tf, err, s);
  }
  TierIO t1{nullptr, nullptr, O.def1, O.n_def1};
  TierIO t2{O.def1, O.n_def1, O.def2, O.n_def2};
  cudaError_t e;
  // Where one warp per query pays (see kWarpTier*); tier 1 takes what it defers.
  const bool long_lists = P.n_join >= (uint64_t)kWarpWalkMinAvg * P.n_entries &&
                          P.n_entries * 4ull >= kWarpWalkMinIndexBytes;
  const bool short_lists = P.n_join < (uint64_t)kWarpTierMaxAvg * P.n_entries;
  if (!emit_all && !P.q_win_off && !Q.colbest && !Q.tgt_end && Q.walk == PD_WALK_AUTO && n_best <= kWMaxGenomes &&
      Q.n_queries >= kWarpTierMinQueries && (long_lists || short_lists || !Q.all_pairs || Q.symbest)) {
    const bool two = Q.symbest ? P.n_join >= (uint64_t)kWPairMinAvg * P.n_entries : long_lists;
    auto kernel = Q.symbest     ? (two ? k_summin_warp<2, kSymmetricForm> : k_summin_warp<1, kSymmetricForm>)
                  : Q.all_pairs ? (two ? k_summin_warp<2, kAllPairsForm> : k_summin_warp<1, kAllPairsForm>)
                                : (two ? k_summin_warp<2, kRangeForm> : k_summin_warp<1, kRangeForm>);
    const float avg_list = short_lists ? 0.f : (float)P.n_join / (float)P.n_entries;
    const size_t smem = kWWarps * warp_tier_bytes(n_best);
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(kWWarps * warp_tier_bytes(kWMaxGenomes)))) != cudaSuccess)
      return e;
    int per_sm = 1, dev = 0, n_sm = 152;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kWThreads, smem);
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const uint32_t grid = std::max<uint32_t>(1, std::min<uint32_t>((Q.n_queries + kWWarps - 1) / kWWarps,
                                                                   (uint32_t)n_sm * std::max(per_sm, 1)));
    TierIO t0{nullptr, nullptr, O.def0, O.n_def0};
    if ((e = launch_begin(L, "summin_warp")) != cudaSuccess) return e;
    kernel<<<grid, kWThreads, smem, s>>>(P, Q, O, t0, O.ticket, n_best, avg_list);
    if ((e = launch_end(L, "summin_warp")) != cudaSuccess) return e;
    t1.in_list = O.def0;
    t1.in_count = O.n_def0;
  }
  // tier 1: several resident blocks per SM, each looping over queries
  if (emit_all)
    e = launch_smem<T1E, 1>(k_summin_smem<kT1Threads, kT1MinBlocks, kT1Cap, kT1OutEmit, true, true, false, kT1Used>, L, "summin_pairs",
                    kT1Threads, n_best, Q.n_queries, P, Q, O, t1, err, s);
  else {
    // merge-path walk, or the warp-cooperative one for long lists
    const bool merge = Q.walk == PD_WALK_MERGE ||
                       (Q.walk != PD_WALK_WARP && (P.n_join < (uint64_t)kWarpWalkMinAvg * P.n_entries ||
                                                   P.n_entries * 4ull < kWarpWalkMinIndexBytes));
    const bool range = !Q.all_pairs && !P.q_win_off;
    auto launch = Q.symbest ? (merge ? launch_t1<false, kSymmetricForm> : launch_t1<true, kSymmetricForm>)
                  : range   ? (merge ? launch_t1<false, kRangeForm> : launch_t1<true, kRangeForm>)
                            : (merge ? launch_t1<false, kAnyForm> : launch_t1<true, kAnyForm>);
    e = launch(L, n_best, P, Q, O, t1, err, s);
  }
  if (e != cudaSuccess) return e;
  // tier 2: one 1024-thread block per SM over the deferred queries (exits at once if none)
  if (emit_all)
    e = launch_smem<T2E, 1>(k_summin_smem<kT2Threads, 1, kT2Cap, kT2OutEmit, false, true>, L, "summin_pairs_t2", kT2Threads,
                    n_best, Q.n_queries, P, Q, O, t2, err, s);
  else
    e = launch_smem<T2>(k_summin_smem<kT2Threads, 1, kT2Cap, kT2Out, false, false>, L, "summin_bh_t2", kT2Threads,
                    n_best, Q.n_queries, P, Q, O, t2, err, s);
  return e;
}

size_t summin_global_smem_bytes(uint32_t n_genomes) {
  return Chunk<256>::kBytes + (size_t)(n_genomes ? n_genomes : 1) * 12 + 4;
}

cudaError_t run_summin_global(Launcher* L, const ProfilesView& P, const QuerySet& Q, const HitsOut& O,
                              const BigScratch& B, uint32_t n_ctas, DevErr* err, bool emit_all, cudaStream_t s) {
  const size_t smem = summin_global_smem_bytes(Q.all_pairs ? P.n_genomes : 1u);
  const int most = (int)summin_global_smem_bytes(PD_MAX_GENOMES);
  TierIO t3{O.def2, O.n_def2, nullptr, nullptr};
  const char* name = Q.filter ? "summin_bh_f_t3" : (emit_all ? "summin_pairs_t3" : "summin_bh_t3");
  cudaError_t e;
  if (Q.filter) {
    if (emit_all || !B.vpa || !B.vpb) return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(k_summin_global<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
    if ((e = launch_begin(L, name)) != cudaSuccess) return e;
    k_summin_global<false, true><<<n_ctas, 256, smem, s>>>(P, Q, O, t3, B, err);
    return launch_end(L, name);
  }
  if (emit_all)
    e = cudaFuncSetAttribute(k_summin_global<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  else
    e = cudaFuncSetAttribute(k_summin_global<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e != cudaSuccess) return e;
  if ((e = launch_begin(L, name)) != cudaSuccess) return e;
  if (emit_all)
    k_summin_global<true><<<n_ctas, 256, smem, s>>>(P, Q, O, t3, B, err);
  else
    k_summin_global<false><<<n_ctas, 256, smem, s>>>(P, Q, O, t3, B, err);
  return launch_end(L, name);
}

}  // namespace pdg
