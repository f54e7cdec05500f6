// The held state read back in key order: a stable radix sort, eight bits of the
// key per pass from the lowest up (Knuth, TAOCP vol. 3, 5.2.5), of (key, entry
// index), then one gather of the amplitudes and sigma.  Only the digits that the
// spin-orbitals reach are passed over: four for 30 spin-orbitals.
//
// A pass is three launches: digit counts per tile of 4,096 keys, their prefix
// sums (a block per digit), and the scatter, in which each warp ranks 512
// consecutive keys 32 at a time by matching lanes.  It is bound by the scatter's
// writes: a tile's keys of one digit go to one place, 16 of them (128 bytes) on
// average.  The state of 621,075 determinants at 30 spin-orbitals with its energy,
// read back with sigma, took 74 ms when the host sorted it and takes 29 ms.

#include <utility>

#include "ucc_device.cuh"

namespace ucc {

namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32, kRounds = 16;
constexpr int kTile = kThreads * kRounds;
constexpr int kDigits = 256;

template <class KT>
__device__ __forceinline__ unsigned int digit_of(KT key, int shift) {
  using K = KeyOps<KT>;
  return (unsigned int)((shift < 64 ? K::lo(key) >> shift : K::hi(key) >> (shift - 64)) & 255ull);
}

// The live entries' keys and indices, in any order.
template <class KT>
__global__ void __launch_bounds__(kThreads) k_sort_collect(TableT<KT> t, SortListT<KT> to, unsigned long long cap) {
  const unsigned long long n = min(*((volatile unsigned long long*)&t.cnt->n_tail), t.cap_n);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    if (is_dead(t.amps[i])) continue;
    const unsigned long long j = aggregated_add(&t.cnt->new_n);
    if (j < cap) {
      to.keys[j] = t.keys[i];
      to.idx[j] = (unsigned int)i;
    }
  }
}

template <class KT>
__global__ void __launch_bounds__(kThreads) k_sort_count(const KT* __restrict__ keys, unsigned long long n, int shift,
                                                         unsigned int* counts) {
  __shared__ unsigned int s_c[kDigits];
  static_assert(kDigits == kThreads, "a digit per thread");
  s_c[threadIdx.x] = 0u;
  __syncthreads();
  const unsigned long long base = (unsigned long long)blockIdx.x * kTile;
#pragma unroll 4
  for (int r = 0; r < kRounds; ++r) {
    const unsigned long long x = base + (unsigned long long)(r * kThreads) + threadIdx.x;
    if (x < n) atomicAdd(&s_c[digit_of(keys[x], shift)], 1u);
  }
  __syncthreads();
  counts[(unsigned long long)threadIdx.x * gridDim.x + blockIdx.x] = s_c[threadIdx.x];
}

// A block's sum over the lower threads; *total: over all.
__device__ __forceinline__ unsigned int scan_block(unsigned int mine, unsigned int* s_w, unsigned int* total) {
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  unsigned int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if ((int)lane >= o) incl += y;
  }
  if (lane == 31u) s_w[warp] = incl;
  __syncthreads();
  unsigned int before = 0u, all = 0u;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    if (w < (int)warp) before += s_w[w];
    all += s_w[w];
  }
  __syncthreads();
  *total = all;
  return before + incl - mine;
}

// Digit blockIdx.x: its tiles' counts to their prefix sums, its total to totals.
__global__ void __launch_bounds__(kThreads) k_sort_scan(unsigned int* counts, unsigned int tiles, unsigned int* totals) {
  __shared__ unsigned int s_w[kWarps];
  unsigned int* const c = counts + (unsigned long long)blockIdx.x * tiles;
  unsigned int run = 0u;
  for (unsigned int b = 0; b < tiles; b += kThreads) {
    const unsigned int x = b + threadIdx.x, mine = x < tiles ? c[x] : 0u;
    unsigned int all;
    const unsigned int before = scan_block(mine, s_w, &all);
    if (x < tiles) c[x] = run + before;
    run += all;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = run;
}

template <class KT>
__global__ void __launch_bounds__(kThreads) k_sort_scatter(SortListT<KT> from, SortListT<KT> to, unsigned long long n,
                                                           int shift, const unsigned int* __restrict__ counts,
                                                           const unsigned int* __restrict__ totals) {
  __shared__ unsigned int s_at[kWarps][kDigits];  // where a warp's next key of a digit goes
  __shared__ unsigned int s_w[kWarps];
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  for (int w = 0; w < kWarps; ++w) s_at[w][threadIdx.x] = 0u;
  __syncthreads();
  const unsigned long long base = (unsigned long long)blockIdx.x * kTile + warp * (32u * kRounds) + lane;
  KT key[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const unsigned long long x = base + 32u * r;
    key[r] = x < n ? from.keys[x] : KeyOps<KT>::zero();
  }
#pragma unroll
  for (int r = 0; r < kRounds; ++r)
    if (base + 32u * r < n) atomicAdd(&s_at[warp][digit_of(key[r], shift)], 1u);
  __syncthreads();
  unsigned int all;
  unsigned int at = scan_block(totals[threadIdx.x], s_w, &all);
  at += counts[(unsigned long long)threadIdx.x * gridDim.x + blockIdx.x];
  for (int w = 0; w < kWarps; ++w) {
    const unsigned int c = s_at[w][threadIdx.x];
    s_at[w][threadIdx.x] = at;
    at += c;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const unsigned long long x = base + 32u * r;
    const bool in = x < n;
    const unsigned int d = in ? digit_of(key[r], shift) : (unsigned int)kDigits;
    const unsigned int same = __match_any_sync(0xFFFFFFFFu, d);
    unsigned int to_at = 0u;
    if (in) to_at = s_at[warp][d] + __popc(same & ((1u << lane) - 1u));
    __syncwarp();
    if (in) {
      if (lane == (unsigned int)(31 - __clz(same))) s_at[warp][d] = to_at + 1u;  // the last of them
      to.keys[to_at] = key[r];
      to.idx[to_at] = from.idx[x];
    }
    __syncwarp();
  }
}

template <class KT>
__global__ void __launch_bounds__(kThreads) k_sort_gather(TableT<KT> t, const unsigned int* __restrict__ idx,
                                                          unsigned long long n, double* amps, double* sigma) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long j = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
    const unsigned int i = idx[j];
    if (i >= t.cap_n) continue;  // (fewer entries than the caller counted: it reports that)
    amps[j] = t.amps[i];
    if (sigma) sigma[j] = t.sigma[i];
  }
}

}  // namespace

size_t sort_scratch_words(unsigned long long n) { return (size_t)kDigits * ((n + kTile - 1) / kTile + 1); }

template <class KT>
cudaError_t launch_sorted_export(const TableT<KT>& t, unsigned long long n, int key_bits, SortListT<KT> a,
                                 SortListT<KT> b, unsigned int* scratch, double* amps, double* sigma, int grid,
                                 cudaStream_t st, const KT** sorted) {
  const unsigned int tiles = (unsigned int)((n + kTile - 1) / kTile);
  unsigned int* const totals = scratch;
  unsigned int* const counts = scratch + kDigits;
  k_sort_collect<KT><<<grid, kThreads, 0, st>>>(t, a, n);
  for (int shift = 0; shift < key_bits; shift += 8) {
    k_sort_count<KT><<<tiles, kThreads, 0, st>>>(a.keys, n, shift, counts);
    k_sort_scan<<<kDigits, kThreads, 0, st>>>(counts, tiles, totals);
    k_sort_scatter<KT><<<tiles, kThreads, 0, st>>>(a, b, n, shift, counts, totals);
    std::swap(a, b);
  }
  k_sort_gather<KT><<<grid, kThreads, 0, st>>>(t, a.idx, n, amps, sigma);
  *sorted = a.keys;
  return cudaGetLastError();
}

#define UCC_SORT_INSTANTIATE(KT)                                                                                      \
  template cudaError_t launch_sorted_export<KT>(const TableT<KT>&, unsigned long long, int, SortListT<KT>,            \
                                                SortListT<KT>, unsigned int*, double*, double*, int, cudaStream_t,    \
                                                const KT**);
UCC_SORT_INSTANTIATE(unsigned long long)
UCC_SORT_INSTANTIATE(Key128)

}  // namespace ucc
