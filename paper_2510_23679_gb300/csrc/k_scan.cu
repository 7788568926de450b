// k_scan.cu -- device-wide exclusive prefix sums in one launch.
//
// Used for window offsets, rank bases of the k-mer dictionary blocks, query
// order buckets, and Best Hit / BBH row offsets.  A tile of kTile elements is
// one block; tiles get the sum of those before them by decoupled look-back (see
// pd_internal.cuh), so a scan is one launch and one memset of its status words
// (nothing but the launch for a single tile) where reduce, spine and down-sweep
// were three.  Loads are striped over each warp's run (coalesced); sums are
// 64-bit.
#include "pd_internal.cuh"

namespace pdg {
namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kItems = 16;
constexpr uint64_t kTile = (uint64_t)kThreads * kItems;

__device__ __forceinline__ unsigned long long warp_incl_u64(unsigned long long v) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= (uint32_t)o) v += y;
  }
  return v;
}

// Set bits of dictionary block i (its words 1..7; word 0 receives the scan).
struct DictIn {
  const uint32_t* d;
  __device__ __forceinline__ unsigned long long operator()(uint64_t i) const {
    const uint32_t* b = d + i * 8;
    uint32_t n = 0;
#pragma unroll
    for (int w = 1; w < 8; ++w) n += (uint32_t)__popc(b[w]);
    return n;
  }
};
struct U32In {
  const uint32_t* a;
  __device__ __forceinline__ unsigned long long operator()(uint64_t i) const { return a[i]; }
};

// out[i * stride] = sum of in(0..i-1); out[n * stride] = the total if
// write_last; *total_dst = the total if not null.  In and out may be the same
// array (a tile's inputs are read before its outputs are written).
template <typename In, typename Out, typename Total>
__global__ void __launch_bounds__(kThreads)
    k_scan(In in, uint64_t n, Out* out, int write_last, Total* total_dst, uint32_t stride,
           unsigned long long* status, uint32_t* ticket, DevErr* err) {
  using S = Status<unsigned long long>;
  __shared__ unsigned long long wsum[kWarps + 1], s_before;
  __shared__ uint32_t s_tile;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_tile = gridDim.x > 1 ? atomicAdd(ticket, 1u) : 0u;
  __syncthreads();
  const uint32_t tile = s_tile;
  const uint64_t base = (uint64_t)tile * kTile + (uint64_t)warp * (32 * kItems) + lane;
  unsigned long long v[kItems], run = 0;
#pragma unroll
  for (int r = 0; r < kItems; ++r) v[r] = base + r * 32 < n ? in(base + r * 32) : 0ull;
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const unsigned long long inc = warp_incl_u64(v[r]);
    const unsigned long long sum = __shfl_sync(0xffffffffu, inc, 31);
    v[r] = run + inc - v[r];
    run += sum;
  }
  if (lane == 31) wsum[warp] = run;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long w = lane < kWarps ? wsum[lane] : 0ull;
    const unsigned long long inc = warp_incl_u64(w);
    const unsigned long long all = __shfl_sync(0xffffffffu, inc, 31);
    unsigned long long before = 0;
    if (gridDim.x > 1) {
      volatile unsigned long long* st = status;
      if (tile == 0) {
        if (lane == 0) st[0] = S::kInclusive | all;
      } else {
        if (lane == 0) st[tile] = S::kAggregate | all;
        // reported; the offsets from here on, and the total, are then too small
        if (!look_back_warp(st, tile, &before, err)) {
          if (lane == 0) raise_error(err, PD_ERR_INTERNAL, tile);
          before = 0;
        }
        if (lane == 0) st[tile] = S::kInclusive | (before + all);
      }
    }
    __syncwarp();
    if (lane < kWarps) wsum[lane] = inc - w;
    if (lane == 0) {
      s_before = before;
      if (tile == gridDim.x - 1) {
        if (write_last) out[n * stride] = (Out)(before + all);
        if (total_dst) *total_dst = (Total)(before + all);
      }
    }
  }
  __syncthreads();
  const unsigned long long off = s_before + wsum[warp];
#pragma unroll
  for (int r = 0; r < kItems; ++r)
    if (base + r * 32 < n) out[(base + r * 32) * stride] = (Out)(off + v[r]);
}

template <typename In, typename Out, typename Total = Out>
cudaError_t scan_impl(Launcher* L, In in, uint64_t n, Out* out, int write_last, Total* total_dst, void* temp,
                      cudaStream_t s, uint32_t stride = 1) {
  uint64_t nb = (n + kTile - 1) / kTile;
  if (nb == 0) nb = 1;
  unsigned long long* status = (unsigned long long*)temp;
  cudaError_t e;
  if (nb > 1 && (e = cudaMemsetAsync(temp, 0, (nb + 1) * sizeof(unsigned long long), s)) != cudaSuccess) return e;
  if ((e = launch_begin(L, "scan")) != cudaSuccess) return e;
  k_scan<In, Out, Total><<<(unsigned)nb, kThreads, 0, s>>>(in, n, out, write_last, total_dst, stride, status,
                                                          (uint32_t*)(status + nb), launch_err(L));
  return launch_end(L, "scan");
}

}  // namespace

size_t scan_temp_bytes(uint64_t n) {
  uint64_t nb = (n + kTile - 1) / kTile;
  if (nb == 0) nb = 1;
  return (size_t)(nb + 1) * sizeof(unsigned long long);
}

cudaError_t scan_dict_blocks(Launcher* L, uint32_t* dict, uint64_t n_blocks, uint32_t* total, void* temp,
                             cudaStream_t s) {
  // in() reads words 1..7 of a block, out writes its word 0: no overlap
  return scan_impl<DictIn, uint32_t, uint32_t>(L, DictIn{dict}, n_blocks, dict, 0, total, temp, s, 8u);
}

cudaError_t scan_u32(Launcher* L, const uint32_t* in, uint64_t n, uint32_t* out_excl_np1, void* temp,
                     cudaStream_t s) {
  return scan_impl<U32In, uint32_t, uint32_t>(L, U32In{in}, n, out_excl_np1, 1, nullptr, temp, s);
}

cudaError_t scan_u32_to_u64(Launcher* L, const uint32_t* in, uint64_t n, unsigned long long* out_excl_np1,
                            void* temp, cudaStream_t s) {
  return scan_impl<U32In, unsigned long long, unsigned long long>(L, U32In{in}, n, out_excl_np1, 1, nullptr, temp, s);
}

cudaError_t scan_u32_total(Launcher* L, const uint32_t* in, uint64_t n, uint32_t* out_excl_np1,
                           unsigned long long* total, void* temp, cudaStream_t s) {
  return scan_impl<U32In, uint32_t, unsigned long long>(L, U32In{in}, n, out_excl_np1, 1, total, temp, s);
}

}  // namespace pdg
