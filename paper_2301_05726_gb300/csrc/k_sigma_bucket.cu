// Energy by buckets of shared cores: sigma_I = sum_{J in S} <I|H|J> c_J over
// the stored set S with work proportional to the connected pairs inside S.
//
// Two determinants I != J of S are connected by a double excitation exactly
// when they share the (n_e - 2)-electron core K2 = I minus two electrons =
// J minus two other electrons, and then K2 = I & J is unique; by a single
// excitation exactly when they share the (n_e - 1)-electron core K1 = I & J.
// So every stored I emits one record per removed set (n_e singles and
// n_e (n_e - 1) / 2 doubles, with c_I and its entry index); the records are
// hashed on the core into partitions that fit one block's shared memory, and
// within a partition the records of one core form a group whose pairs are
// exactly the connections (Slater-Condon rules; for doubles only the pairs
// whose removed sets are disjoint: the others are singles, counted in their
// K1 group, or the determinant itself).  The diagonal is added per entry.
// E = <psi|H|psi> / <psi|psi> (Results section) follows from sigma.
//
// Layout: records are 32 bytes (one DRAM sector, one 256-bit store) for
// either key width in HBM, written partition by partition in rounds whose
// records fit a fixed buffer, the cores of the double excitations in one range
// of partitions and those of the singles in another (their elements cost very
// different work).  A block takes a partition: it counts its records into bins
// on further bits of the core's hash (a core's records share a bin), places them
// into shared memory in bin order, and gives each record a thread that walks the
// record's bin.
//
// With a record's sign s_x taken against its core, |I> = s_x a+_p a+_q |K>, an
// element is <I|H|J> = s_x s_w <pq||rs>: c_w enters shared memory as s_w c_w,
// the sum leaves as s_x times it, and a pair costs one load and one FP64
// multiply-add: of (pr|qs) from g, whose index separates into (row of x) + (column
// of w), or for equal spins of (pr|qs) - (ps|qr) from a table.  Neighbouring threads
// walk the same bin, so they read the same w.  A single's element is h_pr plus one
// table entry per electron of the core, taken once for both of its records
// (launch_fock_tables lays the tables out, once per problem).
//
// What bounds it: the FP64 pipe (80 % busy at 30 spin-orbitals) where groups are
// large, the placement of the records where they are small.  Before,
// the ordered pairs of the bins were split evenly over the threads, each element
// from its four indices, its sign from four masks, a single's from two integrals
// per electron while the other lanes waited, and a partition above 3,072 records
// was walked quadratically in global memory.  k_sb_pairs then and now: 9.2e6
// determinants at 40 spin-orbitals (5.7e9 connected pairs) 536 and 77 ms, 8.6e6 at
// 64 (1.2e9 pairs in small groups) 197 and 55 ms, 621,075 at 30 (6.8e8) 38.3 and
// 5.5 ms, 245,025 at 24 (1.7e8) 12.8 and 1.6 ms.

#include <algorithm>

#include "ucc_steps.cuh"

namespace ucc {

namespace {

// Removed spin-orbitals of a record: p | q << 8, q = kSingle for a single.
constexpr unsigned int kSingle = 0xFFu;
// The pairs kernel's block: records in shared memory, counting-sort bins and
// threads.  A partition is a handful of phases with a barrier each, so several
// small blocks an SM hide each other's barriers (4 of 256 threads against 2 of
// 512 with twice the records: 77 against 88 ms at 40 spin-orbitals,
// 55 against 65 at 64); a core has at most 1,024 records
// in one word (32 by 32 orbitals with one electron each), more in two.
template <class KT>
struct SbBlock {
  static constexpr int kCap = sizeof(KT) == 8 ? 1024 : 2048;
  static constexpr int kBinBits = sizeof(KT) == 8 ? 9 : 10;
  static constexpr int kBins = 1 << kBinBits;  // a multiple of kThreads
  static constexpr int kThreads = kCap / 4;
  static constexpr int kPerSM = 1024 / kThreads;
};

template <class KT>
__device__ __forceinline__ unsigned long long core_hash(KT K) {
  return KeyOps<KT>::slot_hash(K);
}

// The top log2p bits of a core's hash; the cores of singles have their own
// partitions, after the 2^log2d of the doubles.
__device__ __forceinline__ unsigned long long top_bits(unsigned long long h, int log2p) {
  return log2p == 0 ? 0ull : (h >> (64 - log2p));
}
template <class KT>
__device__ __forceinline__ unsigned long long partition_of(KT core, unsigned int removed, SbParts pt) {
  const unsigned long long h = core_hash(core);
  return (removed >> 8) == kSingle ? (1ull << pt.log2d) + top_bits(h, pt.log2s) : top_bits(h, pt.log2d);
}

template <class KT>
__device__ __forceinline__ int bin_of(KT core, int log2p) {
  return (int)((core_hash(core) >> (64 - log2p - SbBlock<KT>::kBinBits)) &
               (unsigned long long)(SbBlock<KT>::kBins - 1));
}

// f(p) for every set bit p of k, ascending.
template <class F>
__device__ __forceinline__ void for_each_bit(unsigned long long k, int offset, F f) {
  for (unsigned long long x = k; x != 0ull; x &= x - 1ull) f(__ffsll((long long)x) - 1 + offset);
}
template <class F>
__device__ __forceinline__ void for_each_bit(Key128 k, int, F f) {
  for_each_bit(k.lo, 0, f);
  for_each_bit(k.hi, 64, f);
}

// f(core, removed) for the n_e single and n_e (n_e - 1) / 2 double cores of I.
template <class KT, class F>
__device__ __forceinline__ void for_each_core(KT I, F f) {
  using K = KeyOps<KT>;
  for_each_bit(I, 0, [&](int p) {
    const KT Ip = I ^ K::bit(p);
    f(Ip, (unsigned int)p | (kSingle << 8));
    // q > p: the bits of I above p
    for_each_bit(I & ~K::below(p + 1), 0, [&](int q) { f(Ip ^ K::bit(q), (unsigned int)p | ((unsigned int)q << 8)); });
  });
}

// Records per core partition.
template <class KT>
__global__ void __launch_bounds__(256) k_sb_count(TableT<KT> t, unsigned int* __restrict__ cnt, SbParts pt) {
  const unsigned long long n = min(*((volatile unsigned long long*)&t.cnt->n_tail), t.cap_n);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    if (is_dead(t.amps[i])) continue;
    for_each_core(t.keys[i],
                  [&](KT core, unsigned int removed) { atomicAdd(&cnt[partition_of(core, removed, pt)], 1u); });
  }
}

// Exclusive prefix sum of n counts into off[0..n] in two launches: the sums of
// tiles of kScanTile counts, kept behind the result (at off + n + 1), then each
// tile by a block that adds up the sums before it.  (One block walking all of
// them took 2.6 ms for 1.4e6 partitions; 26 us.)
constexpr int kScanThreads = 512;
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;
static_assert(kScanTile == kSbScanTile, "tile sums behind the offsets");

__device__ __forceinline__ unsigned long long scan_block_sum(unsigned long long v, unsigned long long* s_v) {
  v = warp_sum_u64(v);
  if ((threadIdx.x & 31u) == 0u) s_v[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long t = 0ull;
#pragma unroll
  for (int x = 0; x < kScanThreads / 32; ++x) t += s_v[x];
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(kScanThreads) k_sb_tile_sums(const unsigned int* __restrict__ cnt,
                                                               unsigned long long* __restrict__ off,
                                                               unsigned long long n) {
  __shared__ unsigned long long s_v[kScanThreads / 32];
  const unsigned long long lo = (unsigned long long)blockIdx.x * kScanTile;
  unsigned long long sum = 0ull;
#pragma unroll
  for (int u = 0; u < kScanPer; ++u) {
    const unsigned long long x = lo + (unsigned long long)(u * kScanThreads) + threadIdx.x;
    if (x < n) sum += cnt[x];
  }
  sum = scan_block_sum(sum, s_v);
  if (threadIdx.x == 0) off[n + 1ull + blockIdx.x] = sum;
}

__global__ void __launch_bounds__(kScanThreads) k_sb_scan(const unsigned int* __restrict__ cnt,
                                                          unsigned long long* __restrict__ off,
                                                          unsigned long long n) {
  __shared__ unsigned long long s_v[kScanThreads / 32];
  const unsigned long long* const tiles = off + n + 1ull;
  unsigned long long before = 0ull;
  for (unsigned int x = threadIdx.x; x < blockIdx.x; x += kScanThreads) before += tiles[x];
  before = scan_block_sum(before, s_v);
  // a thread takes kScanPer consecutive counts; a warp prefix, then the warps'
  const unsigned long long lo = (unsigned long long)blockIdx.x * kScanTile + (unsigned long long)(threadIdx.x * kScanPer);
  unsigned int c[kScanPer];
  unsigned long long sum = 0ull;
#pragma unroll
  for (int u = 0; u < kScanPer; ++u) {
    c[u] = lo + u < n ? cnt[lo + u] : 0u;
    sum += c[u];
  }
  unsigned long long incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if ((int)(threadIdx.x & 31u) >= d) incl += y;
  }
  if ((threadIdx.x & 31u) == 31u) s_v[threadIdx.x >> 5] = incl;
  __syncthreads();
  unsigned long long run = before + incl - sum;
#pragma unroll
  for (int x = 0; x < kScanThreads / 32; ++x)
    if ((unsigned int)x < (threadIdx.x >> 5)) run += s_v[x];
#pragma unroll
  for (int u = 0; u < kScanPer; ++u) {
    if (lo + u < n) off[lo + u] = run;
    run += c[u];
    if (lo + u + 1ull == n) off[n] = run;
  }
}

// A record as one 256-bit store (a whole 32-byte sector: no partial-sector
// write for the memory to merge).
__device__ __forceinline__ void store_words(void* at, unsigned long long a, unsigned long long b, unsigned long long c,
                                            unsigned long long d) {
  asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(at), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}
__device__ __forceinline__ void store_record(SigRecT<unsigned long long>* at, unsigned long long K, double c,
                                             unsigned int i, unsigned int pq) {
  store_words(at, K, (unsigned long long)__double_as_longlong(c), (unsigned long long)i | ((unsigned long long)pq << 32),
              0ull);
}
__device__ __forceinline__ void store_record(SigRecT<Key128>* at, Key128 K, double c, unsigned int i,
                                             unsigned int pq) {
  store_words(at, K.lo, K.hi, (unsigned long long)__double_as_longlong(c),
              (unsigned long long)i | ((unsigned long long)pq << 32));
}

// Where the first record of each partition of [p0, p1) goes: next[p] = off[p] - base.
__global__ void __launch_bounds__(256) k_sb_starts(const unsigned long long* __restrict__ off,
                                                   unsigned int* __restrict__ next, unsigned long long p0,
                                                   unsigned long long p1, unsigned long long base) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long p = p0 + (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; p < p1; p += stride)
    next[p] = (unsigned int)(off[p] - base);
}

// The records of partitions [p0, p1), at rec[next[p]++].  A record is two random
// accesses, the counter and the store, which bound this kernel; counters that
// start at zero cost two more, the partition's bounds (the energy of 8.6e6
// determinants at 64 spin-orbitals, 1.2e9 records: 102.8 ms with them, 97.1 so).
template <class KT>
__global__ void __launch_bounds__(256) k_sb_scatter(TableT<KT> t, unsigned int* __restrict__ next,
                                                    SigRecT<KT>* __restrict__ rec, SbParts pt, unsigned long long p0,
                                                    unsigned long long p1, unsigned int records) {
  const unsigned long long n = min(*((volatile unsigned long long*)&t.cnt->n_tail), t.cap_n);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const double c = t.amps[i];
    if (is_dead(c)) continue;
    for_each_core(t.keys[i], [&](KT core, unsigned int removed) {
      const unsigned long long p = partition_of(core, removed, pt);
      if (p < p0 || p >= p1) return;
      const unsigned int at = atomicAdd(&next[p], 1u);
      if (at >= records) {  // more records than counted: never written past
        raise_error(t.cnt, ERR_CAPACITY);
        return;
      }
      store_record(rec + at, core, c, (unsigned int)i, removed);
    });
  }
}

// A record's removed spin-orbitals as the pair walk wants them.  Doubles: the
// spatial orbitals a, b (a of the alpha one for opposite spins, else the lower),
// the column of its pair (a n^2 + b of g for opposite spins, the pair's number in
// the antisymmetrised table for equal ones), whether the spins are equal, and the
// parity of |I> = s a+_p a+_q |K>; 6 + 6 + 18 + 1 + 1 bits.  Singles: p, and the
// parity of |I> = s a+_p |K>.
constexpr unsigned int kColMask = (1u << 18) - 1u;
__device__ __forceinline__ unsigned int pair_number(unsigned int a, unsigned int b) { return b * (b - 1u) / 2u + a; }
template <class KT, bool SINGLE>
__device__ __forceinline__ unsigned int pair_meta(KT K, unsigned int pq, int n) {
  using Ko = KeyOps<KT>;
  const int p = (int)(pq & 0xFFu), q = (int)(pq >> 8);
  if (SINGLE) return (unsigned int)p | ((unsigned int)(Ko::popc(K & Ko::below(p)) & 1) << 31);
  const bool equal = ((p ^ q) & 1) == 0, turn = !equal && (p & 1) != 0;  // p beta, q alpha: two operators swap
  const unsigned int a = (unsigned int)(turn ? q : p) >> 1, b = (unsigned int)(turn ? p : q) >> 1;
  const unsigned int parity = (unsigned int)(Ko::popc(K & (Ko::below(p) ^ Ko::below(q))) + (turn ? 1 : 0)) & 1u;
  const unsigned int col = equal ? pair_number(a, b) : a * (unsigned int)(n * n) + b;
  return col | (a << 18) | (b << 24) | ((unsigned int)equal << 30) | (parity << 31);
}

// What the walk of a record's bin needs of the record itself.
struct PairRow {
  const double* v;    // doubles: its row, <pq||rs> = v[column of rs]
  unsigned int m, s;  // its meta word, and that with a and b swapped
};
__device__ __forceinline__ PairRow pair_row(const Integrals& in, unsigned int m) {
  PairRow r;
  const unsigned int a = (m >> 18) & 63u, b = (m >> 24) & 63u, n = (unsigned int)in.n;
  r.v = (m >> 30 & 1u) ? in.anti + (size_t)(m & kColMask) * (n * (n - 1u) / 2u)
                       : in.g + (size_t)(a * n * n * n + b * n);
  r.m = m;
  r.s = (b << 18) | (a << 24);
  return r;
}

// Whether records with meta words r.m and w of one core remove disjoint pairs.
__device__ __forceinline__ bool pair_disjoint(const PairRow& r, unsigned int w) {
  const unsigned int t = r.m ^ w;
  bool ok = (t & (63u << 18)) != 0u && (t & (63u << 24)) != 0u;
  if (w >> 30 & 1u) {
    const unsigned int u = r.s ^ w;
    ok = ok && (u & (63u << 18)) != 0u && (u & (63u << 24)) != 0u;
  }
  return ok;
}

// <pq||rs> of disjoint pairs: (pr|qs), less (ps|qr) for equal spins.
__device__ __forceinline__ double pair_integral(const PairRow& r, unsigned int w) {
  return __ldg(r.v + (w & kColMask));
}

// v + the table entries of the set bits k of the core's word: same[k >> 1]
// where k has the spin of p (word offset even, so its parity is the bit's), else
// other[k >> 1].  Four loads in flight.
__device__ __forceinline__ double add_fock(double v, unsigned long long bits, int offset, int p,
                                           const double* __restrict__ same, const double* __restrict__ other) {
  while (bits) {
    double x[4];
    int m = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[u] = 0.0;
      if (bits) {
        const int k = __ffsll((long long)bits) - 1 + offset;
        bits &= bits - 1ull;
        x[u] = __ldg(((k ^ p) & 1 ? other : same) + (k >> 1));
        ++m;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < m) v += x[u];
  }
  return v;
}

// h_rp + sum_{k in K} <rk||pk> of a single p -> r.
template <class KT>
__device__ __forceinline__ double single_integral(const Integrals& in, KT K, int p, int r) {
  double v = h_so(in, r, p);
  const int row = ((r >> 1) * in.n + (p >> 1)) * in.n;
  v = add_fock(v, KeyOps<KT>::lo(K), 0, p, in.fsame + row, in.fother + row);
  if (KeyOps<KT>::kWords == 2) v = add_fock(v, KeyOps<KT>::hi(K), 64, p, in.fsame + row, in.fother + row);
  return v;
}

// <I|H|J> s_x s_w for the records (K, mx) and (K, mw) of one core, in *h; false when
// they are no excitation of the group's kind.
template <class KT, bool SINGLE>
__device__ __forceinline__ bool pair_element(const Integrals& in, KT K, const PairRow& r, unsigned int mx,
                                             unsigned int mw, double* h) {
  if (SINGLE) {
    if (((mx ^ mw) & 0xFFu) == 0u) return false;
    *h = single_integral(in, K, (int)(mx & 0xFFu), (int)(mw & 0xFFu));
    return true;
  }
  if (!pair_disjoint(r, mw)) return false;
  *h = pair_integral(r, mw);
  return true;
}

// A bin too large for shared memory: every record of it walks the whole
// partition in global memory (quadratic, for cores of more than kCap records).
template <class KT, bool SINGLE>
__device__ unsigned int pairs_in_global(const TableT<KT>& t, const Integrals& in, const SigRecT<KT>* rec,
                                        unsigned long long m, int log2p, int bin) {
  unsigned int pairs = 0;
  for (unsigned long long x = threadIdx.x; x < m; x += blockDim.x) {
    const SigRecT<KT> a = rec[x];
    if (bin_of(a.K, log2p) != bin) continue;
    const unsigned int mx = pair_meta<KT, SINGLE>(a.K, a.pq, in.n);
    PairRow row{};
    if (!SINGLE) row = pair_row(in, mx);
    double acc = 0.0;
    for (unsigned long long z = 0; z < m; ++z) {
      const KT Kz = rec[z].K;
      if (z == x || !(Kz == a.K)) continue;
      const unsigned int mz = pair_meta<KT, SINGLE>(Kz, rec[z].pq, in.n);
      double h;
      if (pair_element<KT, SINGLE>(in, Kz, row, mx, mz, &h)) {
        acc = fma(h, neg_if(rec[z].c, (int)(mz >> 31)), acc);
        ++pairs;
      }
    }
    if (nonzero(acc)) atomicAdd(&t.sigma[a.i], neg_if(acc, (int)(mx >> 31)));
  }
  return pairs;
}

template <class KT, bool SINGLE>
constexpr size_t sb_smem_bytes() {
  using B = SbBlock<KT>;
  return (size_t)B::kCap * (sizeof(KT) + (SINGLE ? 2 : 1) * sizeof(double) + 2 * sizeof(unsigned int)) +
         (size_t)(2 * B::kBins + 4) * sizeof(unsigned int);
}

// Exclusive scan of the bins' counts into start (kSbBins + 1 entries, the total
// last); cnt is overwritten with the same (the placement cursors).  Every thread
// of the block calls this.
template <int kSbBins, int kSbThreads>
__device__ __forceinline__ void scan_bins(unsigned int* cnt, unsigned int* start, unsigned int* s_w) {
  constexpr int kPer = kSbBins / kSbThreads;
  constexpr int kWarps = kSbThreads / 32;
  const unsigned int tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
  unsigned int n[kPer], sum = 0u;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    n[u] = cnt[tid * kPer + u];
    sum += n[u];
  }
  unsigned int incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= (unsigned int)d) incl += y;
  }
  if (lane == 31u) s_w[wid] = incl;
  __syncthreads();
  // every warp scans the warp totals itself
  const unsigned int c = lane < (unsigned int)kWarps ? s_w[lane] : 0u;
  unsigned int wi = c;
#pragma unroll
  for (int d = 1; d < kWarps; d <<= 1) {
    const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, wi, d);
    if (lane >= (unsigned int)d) wi += y;
  }
  unsigned int run = __shfl_sync(0xFFFFFFFFu, wi - c, wid) + incl - sum;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    start[tid * kPer + u] = run;
    cnt[tid * kPer + u] = run;
    run += n[u];
  }
  if (tid == kSbThreads - 1u) start[kSbBins] = run;
  __syncthreads();
}

// One block per partition q of [q0, q1) (grid-stride; offsets at off[first + q]).
// Partitions above kCap records are taken bin range by bin range.
template <class KT, bool SINGLE>
__global__ void __launch_bounds__(SbBlock<KT>::kThreads, SbBlock<KT>::kPerSM)
    k_sb_pairs(TableT<KT> t, Integrals in, const SigRecT<KT>* __restrict__ rec,
               const unsigned long long* __restrict__ off, int log2p, unsigned long long first,
               unsigned long long q0, unsigned long long q1, unsigned long long base) {
  extern __shared__ __align__(16) unsigned char sb_smem[];
  constexpr int kSbCap = SbBlock<KT>::kCap, kSbBins = SbBlock<KT>::kBins, kSbThreads = SbBlock<KT>::kThreads;
  KT* sK = reinterpret_cast<KT*>(sb_smem);
  double* sc = reinterpret_cast<double*>(sK + kSbCap);                // s_w c_w
  double* so = sc + kSbCap;                                           // singles: s_x sigma_x
  unsigned int* si = reinterpret_cast<unsigned int*>(so + (SINGLE ? kSbCap : 0));
  unsigned int* sm = si + kSbCap;                                     // pair_meta
  unsigned int* cnt = sm + kSbCap;                                    // counts, then placement cursors
  unsigned int* start = cnt + kSbBins;                                // kSbBins + 1: records before each bin
  __shared__ unsigned int s_w[kSbThreads / 32];
  const unsigned int tid = threadIdx.x;
  unsigned long long pairs = 0;
  for (unsigned long long q = q0 + blockIdx.x; q < q1; q += gridDim.x) {
    const unsigned long long lo = off[first + q] - base, m = off[first + q + 1] - off[first + q];
    if (m == 0) continue;
    const SigRecT<KT>* const r = rec + lo;
    for (int b = (int)tid; b < kSbBins; b += kSbThreads) cnt[b] = 0u;
    __syncthreads();
    for (unsigned long long x = tid; x < m; x += kSbThreads) atomicAdd(&cnt[bin_of(r[x].K, log2p)], 1u);
    __syncthreads();
    scan_bins<kSbBins, kSbThreads>(cnt, start, s_w);
    for (int b0 = 0; b0 < kSbBins;) {  // block-uniform
      // the bins [b0, b1) that fit: all of them for an ordinary partition
      const unsigned int s0 = start[b0];
      int b1 = kSbBins;
      if (start[kSbBins] - s0 > (unsigned int)kSbCap) {
        int lo_b = b0, hi_b = kSbBins;  // the last b1 with start[b1] - s0 <= kSbCap
        while (hi_b - lo_b > 1) {
          const int mid = (lo_b + hi_b) >> 1;
          if (start[mid] - s0 <= (unsigned int)kSbCap)
            lo_b = mid;
          else
            hi_b = mid;
        }
        b1 = lo_b;
      }
      if (b1 == b0) {
        pairs += pairs_in_global<KT, SINGLE>(t, in, r, m, log2p, b0);
        ++b0;
        continue;
      }
      for (unsigned long long x = tid; x < m; x += kSbThreads) {
        const SigRecT<KT> a = r[x];
        const int b = bin_of(a.K, log2p);
        if (b < b0 || b >= b1) continue;
        const unsigned int at = atomicAdd(&cnt[b], 1u) - s0;
        const unsigned int meta = pair_meta<KT, SINGLE>(a.K, a.pq, in.n);
        sK[at] = a.K;
        sc[at] = neg_if(a.c, (int)(meta >> 31));
        si[at] = a.i;
        sm[at] = meta;
        if (SINGLE) so[at] = 0.0;
      }
      __syncthreads();
      const unsigned int count = start[b1] - s0;
      for (unsigned int x = tid; x < count; x += kSbThreads) {
        const KT K = sK[x];
        const int b = bin_of(K, log2p);
        const unsigned int w0 = start[b] - s0, w1 = start[b + 1] - s0;
        if (w1 - w0 < 2u) continue;
        const unsigned int mx = sm[x];
        PairRow row{};
        if (!SINGLE) row = pair_row(in, mx);
        double acc = 0.0;
        unsigned int found = 0u;
        if (SINGLE) {
          // An element is dear and serves both records: x takes the half of its
          // bin that follows it around the circle (every thread of a bin as many),
          // and sends the other record its share.
          const unsigned int len = w1 - w0, half = len / 2u;
          const double cx = sc[x];
          unsigned int w = x;
          for (unsigned int d = 1u; d <= half; ++d) {
            w = w + 1u < w1 ? w + 1u : w0;
            if (d == half && (len & 1u) == 0u && x - w0 >= half) break;  // an even circle's last step, once
            double h;
            if (sK[w] == K && pair_element<KT, SINGLE>(in, K, row, mx, sm[w], &h)) {
              acc = fma(h, sc[w], acc);
              atomicAdd(&so[w], h * cx);
              found += 2u;
            }
          }
          atomicAdd(&so[x], acc);
        } else {
          // two records at a time: their integrals travel together
          for (unsigned int w = w0; w < w1; w += 2u) {
            const unsigned int z = w + 1u < w1 ? w + 1u : w;
            const unsigned int ma = sm[w], mb = sm[z];
            const bool oa = sK[w] == K && pair_disjoint(row, ma);
            const bool ob = z != w && sK[z] == K && pair_disjoint(row, mb);
            double va = 0.0, vb = 0.0;
            if (oa) va = pair_integral(row, ma);
            if (ob) vb = pair_integral(row, mb);
            if (oa) acc = fma(va, sc[w], acc);
            if (ob) acc = fma(vb, sc[z], acc);
            found += (oa ? 1u : 0u) + (ob ? 1u : 0u);
          }
        }
        pairs += found;
        if (!SINGLE && nonzero(acc)) atomicAdd(&t.sigma[si[x]], neg_if(acc, (int)(mx >> 31)));
      }
      __syncthreads();  // shared arrays are refilled
      if (SINGLE) {
        for (unsigned int x = tid; x < count; x += kSbThreads)
          if (nonzero(so[x])) atomicAdd(&t.sigma[si[x]], neg_if(so[x], (int)(sm[x] >> 31)));
        __syncthreads();
      }
      b0 = b1;
    }
    __syncthreads();  // every thread has left the bin ranges' loop (start is rewritten)
  }
  pairs = warp_sum_u64(pairs);
  if ((tid & 31u) == 0 && pairs) atomicAdd(&t.cnt->sig_hits, pairs);
}

// Tables of the singles' elements and of the diagonal, n^3 each: entry
// (p n + r) n + k of fsame is (pr|kk) - (pk|kr), of fother (pr|kk).  And of the
// doubles of equal spins: entry (pair of a < b, pair of r < s) of anti is
// (ar|bs) - (as|br).
__global__ void __launch_bounds__(256) k_fock_tables(Integrals in, double* fsame, double* fother, double* anti) {
  const int n = in.n, total = n * n * n, n4 = total * n;
  for (int x = (int)(blockIdx.x * blockDim.x + threadIdx.x); x < n4; x += (int)(gridDim.x * blockDim.x)) {
    const unsigned int s = x % n, r = x / n % n, b = x / (n * n) % n, a = x / total;
    if (a < b && r < s)
      anti[(size_t)pair_number(a, b) * (size_t)(n * (n - 1) / 2) + pair_number(r, s)] =
          __dsub_rn(chem(in, a, r, b, s), chem(in, a, s, b, r));
  }
  for (int x = (int)(blockIdx.x * blockDim.x + threadIdx.x); x < total; x += (int)(gridDim.x * blockDim.x)) {
    const int k = x % n, r = x / n % n, p = x / (n * n);
    const double j = chem(in, p, r, k, k);
    fother[x] = j;
    fsame[x] = __dsub_rn(j, chem(in, p, k, k, r));
  }
}

// sigma_I += <I|H|I> c_I on every live entry, then E's numerator
// sum c_I sigma_I and <psi|psi> (block partials, summed in a fixed order by
// the last block).
template <class KT>
__global__ void __launch_bounds__(256) k_sb_finish(TableT<KT> t, Integrals in) {
  using Ko = KeyOps<KT>;
  const unsigned long long n = min(*((volatile unsigned long long*)&t.cnt->n_tail), t.cap_n);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  double acc_e = 0.0, acc_n = 0.0;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const double c = t.amps[i];
    if (is_dead(c)) continue;
    const KT I = t.keys[i];
    double d = 0.0;
    for_each_bit(I, 0, [&](int p) {
      // <pq||pq> = (pp|qq) - (pq|qp) [equal spins]
      const int row = ((p >> 1) * in.n + (p >> 1)) * in.n;
      d += h_so(in, p, p);
      for_each_bit(I & ~Ko::below(p + 1), 0,
                   [&](int q) { d += __ldg(((p ^ q) & 1 ? in.fother : in.fsame) + row + (q >> 1)); });
    });
    const double s = t.sigma[i] + d * c;
    t.sigma[i] = s;
    acc_e += c * s;
    acc_n += c * c;
  }
  const double be = block_sum(acc_e);
  const double bn = block_sum(acc_n);
  if (threadIdx.x == 0) {
    t.partials[2 * blockIdx.x] = be;
    t.partials[2 * blockIdx.x + 1] = bn;
  }
  if (last_block_arrive(t.cnt)) {
    double se = 0.0, sn = 0.0;
    for (unsigned int b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
      se += ld_cg(&t.partials[2 * b]);
      sn += ld_cg(&t.partials[2 * b + 1]);
    }
    se = block_sum(se);
    sn = block_sum(sn);
    if (threadIdx.x == 0) {
      t.cnt->e_num = se;
      t.cnt->norm2 = sn;
      t.cnt->done = 0u;
    }
  }
}

}  // namespace

size_t sb_record_bytes(int key_words) { return key_words == 2 ? sizeof(SigRecT<Key128>) : sizeof(SigRecT<unsigned long long>); }

template <class KT>
cudaError_t launch_sb_count(const TableT<KT>& t, unsigned int* cnt, SbParts pt, int grid, cudaStream_t st) {
  k_sb_count<KT><<<grid, 256, 0, st>>>(t, cnt, pt);
  return cudaGetLastError();
}

cudaError_t launch_sb_scan(const unsigned int* cnt, unsigned long long* off, unsigned long long n, cudaStream_t st) {
  const unsigned int tiles = (unsigned int)((n + kScanTile - 1) / kScanTile);
  k_sb_tile_sums<<<tiles, kScanThreads, 0, st>>>(cnt, off, n);
  k_sb_scan<<<tiles, kScanThreads, 0, st>>>(cnt, off, n);
  return cudaGetLastError();
}

cudaError_t launch_fock_tables(const Integrals& in, double* fsame, double* fother, double* anti, cudaStream_t st) {
  const int total = in.n * in.n * in.n * in.n;
  k_fock_tables<<<std::min(1024, (total + 255) / 256), 256, 0, st>>>(in, fsame, fother, anti);
  return cudaGetLastError();
}

template <class KT>
cudaError_t launch_sb_scatter(const TableT<KT>& t, const unsigned long long* off, unsigned int* next,
                              SigRecT<KT>* rec, SbParts pt, unsigned long long p0, unsigned long long p1,
                              unsigned long long base, unsigned int records, int grid, cudaStream_t st) {
  const int blocks = (int)std::min<unsigned long long>((unsigned long long)grid, (p1 - p0 + 255) / 256);
  k_sb_starts<<<blocks, 256, 0, st>>>(off, next, p0, p1, base);
  k_sb_scatter<KT><<<grid, 256, 0, st>>>(t, next, rec, pt, p0, p1, records);
  return cudaGetLastError();
}

// The pairs kernel's dynamic shared memory is above the default 48 KB limit:
// raised (for the current device) before every launch and occupancy query.
template <class KT, bool SINGLE>
cudaError_t sb_allow_smem() {
  return cudaFuncSetAttribute(k_sb_pairs<KT, SINGLE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sb_smem_bytes<KT, SINGLE>());
}

template <class KT>
cudaError_t launch_sb_pairs(const TableT<KT>& t, const Integrals& in, const SigRecT<KT>* rec,
                            const unsigned long long* off, SbParts pt, unsigned long long p0, unsigned long long p1,
                            unsigned long long base, int grid, cudaStream_t st) {
  const unsigned long long nd = 1ull << pt.log2d;
  cudaError_t e;
  if (p0 < std::min(p1, nd)) {
    const unsigned long long q1 = std::min(p1, nd);
    if ((e = sb_allow_smem<KT, false>()) != cudaSuccess) return e;
    k_sb_pairs<KT, false>
        <<<(int)std::min<unsigned long long>((unsigned long long)grid, q1 - p0), SbBlock<KT>::kThreads,
           sb_smem_bytes<KT, false>(), st>>>(t, in, rec, off, pt.log2d, 0ull, p0, q1, base);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (p1 > nd) {
    const unsigned long long q0 = std::max(p0, nd) - nd, q1 = p1 - nd;
    if ((e = sb_allow_smem<KT, true>()) != cudaSuccess) return e;
    k_sb_pairs<KT, true>
        <<<(int)std::min<unsigned long long>((unsigned long long)grid, q1 - q0), SbBlock<KT>::kThreads,
           sb_smem_bytes<KT, true>(), st>>>(t, in, rec, off, pt.log2s, nd, q0, q1, base);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <class KT>
cudaError_t launch_sb_finish(const TableT<KT>& t, const Integrals& in, int grid, cudaStream_t st) {
  k_sb_finish<KT><<<grid, 256, 0, st>>>(t, in);
  return cudaGetLastError();
}

int sb_blocks_per_sm(int key_words) {
  int nb = 0;
  cudaError_t e;
  if (key_words == 2) {
    e = sb_allow_smem<Key128, false>();
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_sb_pairs<Key128, false>, SbBlock<Key128>::kThreads,
                                                        sb_smem_bytes<Key128, false>());
  } else {
    e = sb_allow_smem<unsigned long long, false>();
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_sb_pairs<unsigned long long, false>,
                                                        SbBlock<unsigned long long>::kThreads,
                                                        sb_smem_bytes<unsigned long long, false>());
  }
  return e == cudaSuccess ? nb : 0;
}

int sb_partition_target(int key_words) {
  return (key_words == 2 ? SbBlock<Key128>::kCap : SbBlock<unsigned long long>::kCap) / 2;
}

#define UCC_SB_INSTANTIATE(KT)                                                                                      \
  template cudaError_t launch_sb_count<KT>(const TableT<KT>&, unsigned int*, SbParts, int, cudaStream_t);         \
  template cudaError_t launch_sb_scatter<KT>(const TableT<KT>&, const unsigned long long*, unsigned int*,         \
                                             SigRecT<KT>*, SbParts, unsigned long long, unsigned long long,        \
                                             unsigned long long, unsigned int, int, cudaStream_t);                 \
  template cudaError_t launch_sb_pairs<KT>(const TableT<KT>&, const Integrals&, const SigRecT<KT>*,               \
                                           const unsigned long long*, SbParts, unsigned long long,                 \
                                           unsigned long long, unsigned long long, int, cudaStream_t);             \
  template cudaError_t launch_sb_finish<KT>(const TableT<KT>&, const Integrals&, int, cudaStream_t);
UCC_SB_INSTANTIATE(unsigned long long)
UCC_SB_INSTANTIATE(Key128)

}  // namespace ucc
