// Resident passes: a run of factor steps of one wavefunction inside one
// thread-block cluster, with the whole table in the cluster's distributed
// shared memory.
//
// A table of a few thousand determinants (the paper's production cut keeps
// 5,000 to 8,000) leaves almost nothing to do per factor: a launch per factor
// and a dozen launches per cut are all latency.  Here one launch runs every
// factor.  Determinants are owned by the CTA that the top bits of their key's
// hash name; the owner keeps them in entry arrays (key, amplitude, birth
// factor, adjoint) and in a local hash of 4-byte slots, both in its shared
// memory.  A factor step:
//
//   A  every CTA scans its own keys into a queue of linked entries, then takes
//      the queue a thread per entry: one 16-byte read of the partner's bucket
//      in its owner's memory (most partners are absent), the rotation, and a
//      push of a created partner to the end of its owner's arrays;
//   -- cluster barrier --
//   B  every CTA hashes what was pushed to it (local work) while one warp
//      reads all CTAs' counts, from which every CTA takes the same decision:
//      cut, compact, stop, or go on;
//   -- cluster barrier --
//
// so a step costs two barriers and a few shared-memory round trips.  The cut
// is a histogram of |c| (4,096 bins over the exponents that amplitudes have),
// combined slice by slice over the cluster, and a pairwise rank of the few
// entries of the threshold's bin; compaction and rehashing are local to each
// CTA.  The reverse sweep has the same two phases: the sweep of factor k and
// the push of factor k - 1's tape records, then their hashing.
//
// What bounds it: latency.  A factor of the 64-spin-orbital, 10-electron
// problem with the production cut (about 6,000 keys scanned, 2,400 pairs, a cut
// after three factors of four) takes 8.5 us forward, and 5.8 us reverse with
// its 2,400 tape records, where a launch per factor and a launch chain per cut
// took 74 and 51 us: its gradient (5,270 factors) went from 672 to 100 ms, with
// two-word keys (72 spin-orbitals) from 725 to 111 ms; 12 spin-orbitals, 92
// factors: from 2.47 to 0.77 ms; 24 uneven jobs in one batch, a cluster per job
// in place of grid-wide steps: from 664 to 40 ms.
//
// The arithmetic, the eps rule, the cut's order and the pair ownership are
// those of the launch-per-factor kernels (rotate_member and its kin are
// shared), so states agree bit for bit.
//
// A CTA's share is a binomial draw of the table's entries, so its arrays are
// sized with a margin; a push past the end leaves the owner's count above its
// capacity, every CTA sees that at the same barrier, and the launch ends
// without having touched the table in global memory (forward) or with the
// pushes of that step taken back (reverse).  The host then runs the same
// factors with the launch-per-factor kernels.

#include <algorithm>
#include <cmath>

#include "ucc_steps.cuh"

namespace ucc {

namespace {

constexpr int kT = 512;  // threads per CTA
constexpr int kW = kT / 32;
constexpr int kBinBits = 12;
constexpr int kBins = 1 << kBinBits;
constexpr int kCand = 512;  // candidates of a cut ranked pairwise
constexpr int kOffRing = 256;
constexpr int kMaxLogC = 4;

// Byte offsets of a CTA's shared arrays, host and device.
struct ResLayout {
  unsigned int keys, amps, lam, born, slots, queue, hist, comb, cmag, ckey, red, bytes;
};

__host__ __device__ inline unsigned int up16(unsigned int x) { return (x + 15u) & ~15u; }

template <class KT>
__host__ __device__ inline ResLayout res_layout(const ResGeom& g, bool reverse) {
  ResLayout o{};
  unsigned int at = 0;
  auto take = [&](unsigned int bytes) {
    const unsigned int r = at;
    at = up16(at + bytes);
    return r;
  };
  o.keys = take((unsigned int)(g.L * sizeof(KT)));
  o.amps = take((unsigned int)g.L * 8u);
  o.born = take((unsigned int)g.L * 4u);
  o.slots = take(16u << g.logB);
  o.queue = take((unsigned int)g.L * 2u);
  if (reverse) {
    o.lam = take((unsigned int)g.L * 8u);
    o.red = take(2u * kT * 8u);
  } else {
    o.hist = take(kBins * 4u);
    o.comb = take((kBins * 4u) >> g.logC);
    o.cmag = take(kCand * 8u);
    o.ckey = take((unsigned int)(kCand * sizeof(KT)));
    o.red = take(kT * 8u);
  }
  o.bytes = at;
  return o;
}

// One CTA's view: local pointers (the same offsets hold in every CTA of the
// cluster) and the cluster's shape.
template <class KT>
struct ResView {
  KT* keys;
  double* amps;
  double* lam;
  unsigned int* born;
  unsigned int* slots;
  unsigned short* queue;
  unsigned int L, bmask;
  int logC, logB;
  unsigned int rank;

  // p in CTA r's shared memory
  template <class T>
  __device__ __forceinline__ T* at(T* p, unsigned int r) const {
    return cg::this_cluster().map_shared_rank(p, r);
  }
  __device__ __forceinline__ void sync() const {
    if (logC == 0)
      __syncthreads();
    else
      cg::this_cluster().sync();
  }
};

template <class KT>
__device__ __forceinline__ ResView<KT> res_view(unsigned char* smem, const ResLayout& o, const ResGeom& g,
                                                bool reverse) {
  ResView<KT> v;
  v.keys = reinterpret_cast<KT*>(smem + o.keys);
  v.amps = reinterpret_cast<double*>(smem + o.amps);
  v.lam = reverse ? reinterpret_cast<double*>(smem + o.lam) : nullptr;
  v.born = reinterpret_cast<unsigned int*>(smem + o.born);
  v.slots = reinterpret_cast<unsigned int*>(smem + o.slots);
  v.queue = reinterpret_cast<unsigned short*>(smem + o.queue);
  v.L = (unsigned int)g.L;
  v.logC = g.logC;
  v.logB = g.logB;
  v.bmask = (1u << g.logB) - 1u;
  v.rank = g.logC ? cg::this_cluster().block_rank() : 0u;
  return v;
}

// Where a key lives: owner CTA, home bucket of four slots, 16-bit tag.  The
// slot hash is folded and multiplied once more: its bits spread determinant
// keys over CTAs and buckets like random draws, which the sizing counts on.
struct Place {
  unsigned int owner, bucket, tag;
};

template <class KT>
__device__ __forceinline__ Place place_of(const ResView<KT>& v, KT key) {
  unsigned long long h = KeyOps<KT>::slot_hash(key);
  h ^= h >> 29;
  h *= kFilterMul;
  const unsigned int hi = (unsigned int)(h >> 32);
  Place p;
  p.owner = v.logC ? hi >> (32 - v.logC) : 0u;
  p.bucket = (hi << v.logC) >> (32 - v.logB);
  p.tag = ((unsigned int)h >> 8) & 0xFFFFu;
  return p;
}

struct ResHit {
  int state;  // Found
  unsigned int owner, idx;
  double amp;
};

// Look key up in its owner's hash.  Slots hold tag << 16 | index + 1, are
// claimed in order inside a bucket and never freed until the hash is rebuilt,
// so a bucket with an empty slot ends the search.
template <class KT>
__device__ __forceinline__ ResHit res_find(const ResView<KT>& v, KT key, unsigned int stamp) {
  ResHit r;
  r.state = ABSENT;
  r.idx = 0u;
  r.amp = 0.0;
  const Place p = place_of(v, key);
  r.owner = p.owner;
  const uint4* const slots = reinterpret_cast<const uint4*>(v.at(v.slots, p.owner));
  unsigned int b = p.bucket;
  for (unsigned int step = 0; step <= v.bmask; ++step) {
    const uint4 q = slots[b];
    const unsigned int w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (w[j] == 0u) return r;
      if ((w[j] >> 16) == p.tag) {
        const unsigned int i = (w[j] & 0xFFFFu) - 1u;
        if (*v.at(v.keys + i, p.owner) == key) {
          const double a = *v.at(v.amps + i, p.owner);
          r.idx = i;
          if (!is_dead(a)) {
            r.state = ALIVE;
            r.amp = a;
          } else {
            r.state = dead_stamp(a) == stamp ? DEAD_NOW : DEAD_OLD;
          }
          return r;
        }
      }
    }
    b = (b + 1u) & v.bmask;
  }
  return r;
}

// Hash entry i of this CTA.  A key that is there already belongs to a dropped
// entry (its slot then points to the new one); a live one is an error.
template <class KT>
__device__ __forceinline__ void res_link(const ResView<KT>& v, unsigned int i, Counters* c, int site) {
  const KT key = v.keys[i];
  const Place p = place_of(v, key);
  const unsigned int word = (p.tag << 16) | (i + 1u);
  unsigned int b = p.bucket;
  for (unsigned int step = 0; step <= v.bmask; ++step) {
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      unsigned int* const s = v.slots + 4u * b + (unsigned int)j;
      unsigned int w = *((volatile unsigned int*)s);
      if (w == 0u) {
        w = atomicCAS(s, 0u, word);
        if (w == 0u) return;
      }
      if ((w >> 16) == p.tag) {
        const unsigned int o = (w & 0xFFFFu) - 1u;
        if (v.keys[o] == key) {
          if (!is_dead(v.amps[o])) raise_consistency(c, site, KeyOps<KT>::lo(key));
          *((volatile unsigned int*)s) = word;
          return;
        }
      }
    }
    b = (b + 1u) & v.bmask;
  }
  raise_error(c, ERR_PROBE_BOUND);
}

// Rebuild this CTA's hash over its first n entries.  Every thread calls this.
template <class KT>
__device__ __forceinline__ void res_rehash(const ResView<KT>& v, unsigned int n, Counters* c) {
  uint4* const s = reinterpret_cast<uint4*>(v.slots);
  for (unsigned int x = threadIdx.x; x <= v.bmask; x += kT) s[x] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (unsigned int i = threadIdx.x; i < n; i += kT) res_link(v, i, c, SITE_REHASH_DUP);
  __syncthreads();
}

// Compact this CTA's first n entries in place: live entries that keep(a, key)
// accepts move down in order, drop(i, key, a, born, rank) is called for the
// live ones it rejects, rank counting them.  Returns the number kept.  Every
// thread calls this; the hash is stale afterwards.
template <class KT, class Keep, class Drop>
__device__ __forceinline__ unsigned int res_compact(const ResView<KT>& v, unsigned int n, Keep keep, Drop drop) {
  __shared__ unsigned int s_k[kW], s_d[kW];
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned int below_me = (1u << lane) - 1u;
  unsigned int kept = 0, dropped = 0;
  for (unsigned int base = 0; base < n; base += kT) {  // block-uniform
    const unsigned int i = base + threadIdx.x;
    const double a = i < n ? v.amps[i] : dead_value(0u);
    const bool live = !is_dead(a);
    KT key = KeyOps<KT>::zero();
    unsigned int born = 0u;
    double lam = 0.0;
    if (live) {
      key = v.keys[i];
      born = v.born[i];
      if (v.lam) lam = v.lam[i];
    }
    const bool kp = live && keep(a, key);
    const unsigned int mk = __ballot_sync(0xFFFFFFFFu, kp), md = __ballot_sync(0xFFFFFFFFu, live && !kp);
    if (lane == 0) {
      s_k[warp] = __popc(mk);
      s_d[warp] = __popc(md);
    }
    __syncthreads();  // ... and every thread has read its entry
    unsigned int pk = 0, pd = 0, tk = 0, td = 0;
#pragma unroll
    for (int x = 0; x < kW; ++x) {
      const unsigned int ck = s_k[x], cd = s_d[x];
      if ((unsigned int)x < warp) {
        pk += ck;
        pd += cd;
      }
      tk += ck;
      td += cd;
    }
    if (kp) {
      const unsigned int to = kept + pk + __popc(mk & below_me);
      v.keys[to] = key;
      v.amps[to] = a;
      v.born[to] = born;
      if (v.lam) v.lam[to] = lam;
    } else if (live) {
      drop(key, a, born, dropped + pd + __popc(md & below_me));
    }
    kept += tk;
    dropped += td;
    __syncthreads();
  }
  return kept;
}

// The block's entries [0, n) that are linked by f, into the queue (entry
// index, top bit for the excited member).  Every thread calls this; the queue
// and its length *qn are complete after the next __syncthreads.
template <class KT>
__device__ __forceinline__ void res_scan(const ResView<KT>& v, const FactorT<KT>& f, unsigned int n,
                                         unsigned int* qn) {
  const unsigned int lane = threadIdx.x & 31u;
  const unsigned int below_me = (1u << lane) - 1u;
  const KT m = f.occ | f.vir;
  for (unsigned int base = threadIdx.x - lane; base < n; base += kT) {  // warp-uniform
    const unsigned int i = base + lane;
    bool act = false, ex = false;
    if (i < n) {
      const KT tX = v.keys[i] & m;
      ex = tX == f.occ;
      act = (ex || tX == f.vir) && !is_dead(v.amps[i]);
    }
    const unsigned int mk = __ballot_sync(0xFFFFFFFFu, act);
    if (mk == 0u) continue;
    unsigned int at = 0u;
    if (lane == 0) at = atomicAdd(qn, __popc(mk));
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (act) v.queue[at + __popc(mk & below_me)] = (unsigned short)(i | (ex ? 0x8000u : 0u));
  }
}

// Counts of all CTAs, read by one warp after a barrier.
struct ResTotals {
  unsigned int tail, dead, most;
};

// Sum of kT doubles in shared memory by one warp (valid in every lane): each
// lane adds kW values, then a shuffle sum.  FP64 adds are scarce on this GPU:
// a warp sum in every warp would cost four times as many.
__device__ __forceinline__ double warp_sum_shared(const double* red, unsigned int count) {
  double s = 0.0;
  for (unsigned int x = threadIdx.x & 31u; x < count; x += 32u) s += red[x];
  return warp_sum(s);
}

template <class KT>
__device__ __forceinline__ unsigned long long mag_of(double a) {
  return (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull;
}

// First histogram digit of a magnitude: exponents 2^-63 .. 2^0 and six bits of
// the mantissa, clamped at both ends (monotone in |c|; amplitudes of a
// normalised state have no larger exponent).
__device__ __forceinline__ int coarse_digit(unsigned long long u) {
  const int e = (int)(u >> 52) - (1023 - 63);
  if (e < 0) return 0;
  if (e > 63) return kBins - 1;
  return (e << 6) | (int)((u >> 46) & 63ull);
}

// Copy the live entries of the table in global memory that this CTA owns into
// its arrays and hash them; *tail counts them (above L: they did not fit).
// Every thread of the cluster calls this.
template <class KT>
__device__ __forceinline__ void res_load(const ResView<KT>& v, const TableT<KT>& t, unsigned int* tail) {
  const unsigned int n = (unsigned int)min(*((volatile unsigned long long*)&t.cnt->n_tail), t.cap_n);
  for (unsigned int i = threadIdx.x; i < n; i += kT) {
    const double a = t.amps[i];
    if (is_dead(a)) continue;
    const KT key = t.keys[i];
    if (place_of(v, key).owner != v.rank) continue;
    const unsigned int j = atomicAdd(tail, 1u);
    if (j >= v.L) continue;
    v.keys[j] = key;
    v.amps[j] = a;
    v.born[j] = t.born[i];
    if (v.lam) v.lam[j] = t.lam[i];
  }
  __syncthreads();
}

// Write this CTA's n entries (compacted: all live) to the table in global
// memory, in the range it reserves there.  Every thread calls this.
template <class KT>
__device__ __forceinline__ void res_store(const ResView<KT>& v, const TableT<KT>& t, unsigned int n) {
  __shared__ unsigned long long s_base;
  if (threadIdx.x == 0) s_base = atomicAdd(&t.cnt->new_n, (unsigned long long)n);
  __syncthreads();
  const unsigned long long base = s_base;
  for (unsigned int i = threadIdx.x; i < n; i += kT) {
    if (base + i >= t.cap_n) {
      raise_error(t.cnt, ERR_CAPACITY);
      continue;
    }
    t.keys[base + i] = v.keys[i];
    t.amps[base + i] = v.amps[i];
    t.born[base + i] = v.born[i];
    if (v.lam) t.lam[base + i] = v.lam[i];
  }
}

// The table in global memory now holds what res_store wrote (one thread).
__device__ __forceinline__ void res_finish(Counters* c) {
  const unsigned long long n = ld_cg(&c->new_n);
  c->n_tail = n;
  c->n_scan = n;
  c->n_dead = 0ull;
  c->new_n = 0ull;
  c->stop_k = -1;
}

// Whether a table of `live` entries can take another step: at most twice as
// many entries (or `bound`, the size of the sector), whose largest share of a
// CTA is taken as the mean plus an eighth and six standard deviations.
__device__ __forceinline__ bool res_room(unsigned int live, unsigned int dead, unsigned long long bound,
                                         unsigned int L, int logC) {
  const unsigned long long most = min(2ull * live, bound) + dead;
  const float mean = (float)most / (float)(1 << logC);
  return logC == 0 ? most <= L : mean * 1.125f + 6.0f * sqrtf(mean) + 8.0f <= (float)L;
}

// The threshold of the cut over the cluster: the N_CUT-th live entry by (|c|
// descending, key ascending), as (*T, *Kt) in every thread.  n: this CTA's
// entries; live: the cluster's live ones.  Passes narrow the threshold's bin
// until it holds at most kCand entries (the first pass nearly always does),
// which CTA 0 collects and every CTA ranks.
template <class KT>
__device__ void res_threshold(const ResView<KT>& v, unsigned int n, unsigned int live, unsigned long long n_cut,
                              unsigned int* hist, unsigned int* comb, unsigned long long* cmag, KT* ckey,
                              unsigned int* ncand, Counters* cnt, unsigned long long* T, KT* Kt) {
  using K = KeyOps<KT>;
  __shared__ unsigned int s_slice, s_from, s_cum, s_bin, s_rest, s_cnt;
  __shared__ unsigned int s_w[kW];
  __shared__ unsigned long long s_T;
  __shared__ __align__(16) KT s_Kt;
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned int C = 1u << v.logC, nb = (unsigned int)kBins >> v.logC;
  unsigned int target = (unsigned int)n_cut, count = live;
  int coarse = -1;
  unsigned long long pu = 0, mu = 0, phi = 0, mhi = 0, plo = 0, mlo = 0;  // digits fixed so far and their masks
  auto inside = [&](unsigned long long u, KT key) {
    return (coarse < 0 || coarse_digit(u) == coarse) && (u & mu) == pu && (K::hi(key) & mhi) == phi &&
           (K::lo(key) & mlo) == plo;
  };
  if (threadIdx.x == 0) {
    s_slice = 0u;
    s_T = 0ull;
    if (v.rank == 0u) *ncand = 0u;
  }
  __syncthreads();
  // pass 0: the coarse digit; 1 to 6: |c| from the top; then the key's high word (if any), then its low one
  for (int pass = 0; pass <= 6 + 6 * K::kWords && (pass == 0 || count > (unsigned int)kCand); ++pass) {
    const int d = pass == 0 ? 0 : (pass - 1) % 6;
    const int word = pass <= 6 ? 0 : (K::kWords == 2 && pass <= 12 ? 2 : 1);  // 0 |c|, 1 low word, 2 high word
    const int shift = max(0, 64 - kBinBits * (d + 1));
    const int width = min(kBinBits, 64 - kBinBits * d);
    for (unsigned int i = threadIdx.x; i < n; i += kT) {
      const double a = v.amps[i];
      if (is_dead(a)) continue;
      const unsigned long long u = mag_of<KT>(a);
      const KT key = v.keys[i];
      if (!inside(u, key)) continue;
      const unsigned long long x = word == 0 ? u : (word == 1 ? K::lo(key) : K::hi(key));
      const unsigned int b =
          pass == 0 ? (unsigned int)coarse_digit(u) : (unsigned int)((x >> shift) & ((1ull << width) - 1ull));
      atomicAdd(&hist[b], 1u);
    }
    v.sync();
    // this CTA's slice of the bins, summed over the cluster
    unsigned int sum = 0u;
    for (unsigned int b = threadIdx.x; b < nb; b += kT) {
      unsigned int s = 0u;
      for (unsigned int r = 0; r < C; ++r) s += *v.at(hist + v.rank * nb + b, r);
      comb[b] = s;
      sum += s;
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0 && sum) atomicAdd(&s_slice, sum);
    v.sync();
    if (threadIdx.x == 0) {  // what a histogram short of the target (an inconsistent count) would leave
      s_bin = s_cnt = 0u;
      s_rest = 1u;
    }
    for (unsigned int b = threadIdx.x; b < (unsigned int)kBins; b += kT) hist[b] = 0u;
    // the slice that holds the target: |c| from the largest bin down, keys from the smallest up
    const bool down = word == 0;
    if (warp == 0) {
      if (lane == 0) s_from = s_cum = 0u;
      __syncwarp();
      const unsigned int r = down ? C - 1u - lane : lane;
      const unsigned int mine = lane < C ? *v.at(&s_slice, r) : 0u;
      unsigned int incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += y;
      }
      if (incl - mine < target && target <= incl) {
        s_from = r;
        s_cum = incl - mine;
      }
    }
    __syncthreads();
    const unsigned int from = s_from, want = target - s_cum;
    const unsigned int per = (nb + kT - 1u) / kT;
    unsigned int c[kBins / kT];
    unsigned int mine = 0u;
#pragma unroll
    for (unsigned int j = 0; j < (unsigned int)(kBins / kT); ++j) {
      const unsigned int o = threadIdx.x * per + j;
      c[j] = j < per && o < nb ? *v.at(comb + (down ? nb - 1u - o : o), from) : 0u;
      mine += c[j];
    }
    unsigned int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if ((int)lane >= o) incl += y;
    }
    if (lane == 31u) s_w[warp] = incl;
    __syncthreads();
    unsigned int before = incl - mine;
#pragma unroll
    for (int x = 0; x < kW; ++x)
      if ((unsigned int)x < warp) before += s_w[x];
    if (before < want && want <= before + mine) {
      unsigned int cum = before;
#pragma unroll
      for (unsigned int j = 0; j < (unsigned int)(kBins / kT); ++j) {
        if (cum < want && want <= cum + c[j]) {
          const unsigned int o = threadIdx.x * per + j;
          s_bin = from * nb + (down ? nb - 1u - o : o);
          s_rest = want - cum;
          s_cnt = c[j];
        }
        cum += c[j];
      }
    }
    __syncthreads();
    const unsigned long long bin = s_bin;
    target = s_rest;
    count = s_cnt;
    const unsigned long long dm = ((1ull << width) - 1ull) << shift;
    if (pass == 0) {
      coarse = (int)bin;
    } else if (word == 0) {
      pu |= bin << shift;
      mu |= dm;
    } else if (word == 1) {
      plo |= bin << shift;
      mlo |= dm;
    } else {
      phi |= bin << shift;
      mhi |= dm;
    }
    v.sync();  // every CTA has read this pass's slices
    if (threadIdx.x == 0) s_slice = 0u;
    __syncthreads();
  }
  // collect the bin's entries in CTA 0
  for (unsigned int i = threadIdx.x; i < n; i += kT) {
    const double a = v.amps[i];
    if (is_dead(a)) continue;
    const unsigned long long u = mag_of<KT>(a);
    const KT key = v.keys[i];
    if (!inside(u, key)) continue;
    const unsigned int q = atomicAdd(v.at(ncand, 0u), 1u);
    if (q < (unsigned int)kCand) {
      *v.at(cmag + q, 0u) = u;
      *v.at(ckey + q, 0u) = key;
    }
  }
  v.sync();
  const unsigned int nc = min(count, (unsigned int)kCand);
  if (v.rank != 0u) {
    for (unsigned int x = threadIdx.x; x < nc; x += kT) {
      cmag[x] = *v.at(cmag + x, 0u);
      ckey[x] = *v.at(ckey + x, 0u);
    }
    __syncthreads();
  }
  for (unsigned int x = threadIdx.x; x < nc; x += kT) {
    const unsigned long long u = cmag[x];
    const KT key = ckey[x];
    unsigned int before = 0u;
    for (unsigned int y = 0; y < nc; ++y)
      before += (cmag[y] > u || (cmag[y] == u && key_less(ckey[y], key))) ? 1u : 0u;
    if (before + 1u == target) {
      s_T = u;
      s_Kt = key;
    }
  }
  __syncthreads();
  if (nc == 0u && threadIdx.x == 0) raise_consistency(cnt, SITE_CUT_COUNT, live);
  *T = s_T;
  *Kt = s_Kt;
}

// ---------------------------------------------------------------------------
// Forward: factors [k0, k1) with the eps rule and the cut.
// ---------------------------------------------------------------------------
template <class KT, bool RECORD>
__global__ void __launch_bounds__(kT, 1) k_res_forward(ResJob<KT> one, const ResJob<KT>* __restrict__ many,
                                                       ResGeom g) {
  using K = KeyOps<KT>;
  extern __shared__ __align__(16) unsigned char res_smem[];
  constexpr int kFW = sizeof(FactorT<KT>) / 8;
  __shared__ __align__(16) unsigned long long s_f[2][kFW];
  __shared__ unsigned int s_tail, s_dead, s_qn, s_ncand, s_drop;
  __shared__ ResTotals s_tot;
  __shared__ unsigned long long s_tape, s_tape_now, s_tbase;  // s_tape: CTA 0's counts for the cluster
  __shared__ double s_dS[2];
  const ResLayout lo = res_layout<KT>(g, false);
  const ResJob<KT> job = many ? many[blockIdx.x >> g.logC] : one;
  const ResView<KT> v = res_view<KT>(res_smem, lo, g, false);
  unsigned int* const hist = reinterpret_cast<unsigned int*>(res_smem + lo.hist);
  unsigned int* const comb = reinterpret_cast<unsigned int*>(res_smem + lo.comb);
  unsigned long long* const cmag = reinterpret_cast<unsigned long long*>(res_smem + lo.cmag);
  KT* const ckey = reinterpret_cast<KT*>(res_smem + lo.ckey);
  double* const red = reinterpret_cast<double*>(res_smem + lo.red);
  Counters* const cnt = job.t.cnt;
  const unsigned int tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const unsigned int C = 1u << v.logC;
  const bool ent = job.t.entropy != nullptr;

  if (tid == 0) {
    s_tail = s_dead = s_qn = s_ncand = 0u;
    s_tape = *((volatile unsigned long long*)&cnt->tape_n);
    s_dS[0] = s_dS[1] = 0.0;
  }
  for (unsigned int b = tid; b < (unsigned int)kBins; b += kT) hist[b] = 0u;
  if (tid < (unsigned int)kFW)
    s_f[job.k0 & 1][tid] = reinterpret_cast<const unsigned long long*>(job.factors + job.k0)[tid];
  __syncthreads();
  res_load(v, job.t, &s_tail);
  res_rehash(v, min(s_tail, v.L), cnt);
  v.sync();

  // Decide before the first step as after every other: the same room rule.
  auto totals = [&]() {
    if (warp == 0) {
      const unsigned int tl = lane < C ? *((volatile unsigned int*)v.at(&s_tail, lane)) : 0u;
      const unsigned int dd = lane < C ? *((volatile unsigned int*)v.at(&s_dead, lane)) : 0u;
      const unsigned int st = __reduce_add_sync(0xFFFFFFFFu, tl), sd = __reduce_add_sync(0xFFFFFFFFu, dd);
      const unsigned int mt = __reduce_max_sync(0xFFFFFFFFu, tl);
      if (lane == 0) {
        s_tot.tail = st;
        s_tot.dead = sd;
        s_tot.most = mt;
        if (RECORD) s_tape_now = *((volatile unsigned long long*)v.at(&s_tape, 0u));
      }
    }
  };
  totals();
  __syncthreads();
  int status = RES_DONE, k = job.k0;
  unsigned long long tape_n = RECORD ? s_tape_now : 0ull;
  {
    const unsigned int live = s_tot.tail;
    if (s_tot.most > v.L || !res_room(live, 0u, job.bound, v.L, v.logC))
      status = RES_FULL;
    else if (RECORD && tape_n + 3ull * live + 64ull > job.tape.cap)
      status = RES_TAPE;
  }
  unsigned int n_scan = min(s_tail, v.L);
  unsigned int rot = 0, cre = 0, dnew = 0, dold = 0, rebuilds = 0, peak = s_tot.tail;
  unsigned long long scanned = 0, cut_total = 0;
  double entropy = cnt->entropy;
  bool stored_any = false;  // at least one factor applied
  v.sync();

  while (status == RES_DONE && k < job.k1) {
    const FactorT<KT> f = *reinterpret_cast<const FactorT<KT>*>(s_f[k & 1]);
    unsigned long long fw = 0ull;
    if (tid < (unsigned int)kFW && k + 1 < job.k1)
      fw = reinterpret_cast<const unsigned long long*>(job.factors + k + 1)[tid];
    const unsigned int stamp = (unsigned int)(k + 1);
    // Phase A
    res_scan(v, f, n_scan, &s_qn);
    __syncthreads();
    const unsigned int qn = s_qn;
    double dS = 0.0;
    for (unsigned int q = tid; q < qn; q += kT) {
      const unsigned int w = v.queue[q];
      const unsigned int i = w & 0x7FFFu;
      const bool ex = (w & 0x8000u) != 0u;
      const KT X = v.keys[i];
      const double cX = v.amps[i];
      const KT Y = X ^ (f.occ | f.vir);
      const ResHit r = res_find(v, Y, stamp);
      const bool partner_live = r.state == ALIVE;
      if (!ex && (partner_live || r.state == DEAD_NOW)) continue;  // E's thread owns the pair
      if (ex && r.state == DEAD_NOW) {
        raise_consistency(cnt, SITE_PAIR_OWNER);
        continue;
      }
      double nX, nY;
      rotate_member(f, X, cX, ex, partner_live, r.amp, nX, nY);
      ++rot;
      const bool xd = below_eps(nX, job.eps), yd = below_eps(nY, job.eps);
      if (ent)
        dS += entropy_term(xd ? 0.0 : nX) + entropy_term(yd ? 0.0 : nY) - entropy_term(cX) -
              (partner_live ? entropy_term(r.amp) : 0.0);
      auto record = [&](KT key, double val, unsigned int born) {
        const unsigned long long at = atomicAdd(v.at(&s_tape, 0u), 1ull);
        if (at < job.tape.cap) {
          TapeRecT<KT>& rec = tape_at(job.tape, at);
          rec.key = key;
          rec.val = val;
          rec.born = born;
        } else {
          raise_error(cnt, ERR_TAPE_FULL);
        }
      };
      if (xd) {
        if (RECORD) record(X, nX, v.born[i]);
        v.amps[i] = dead_value(stamp);
        atomicAdd(&s_dead, 1u);
        ++dold;
      } else {
        v.amps[i] = nX;
      }
      if (partner_live) {
        if (yd) {
          if (RECORD) record(Y, nY, *v.at(v.born + r.idx, r.owner));
          *v.at(v.amps + r.idx, r.owner) = dead_value(stamp);
          atomicAdd(v.at(&s_dead, r.owner), 1u);
          ++dold;
        } else {
          *v.at(v.amps + r.idx, r.owner) = nY;
        }
      } else if (yd) {
        ++dnew;
      } else {
        // created (or revived: phase B points the slot at the new entry)
        const unsigned int j = atomicAdd(v.at(&s_tail, r.owner), 1u);
        if (j < v.L) {
          *v.at(v.keys + j, r.owner) = Y;
          *v.at(v.amps + j, r.owner) = nY;
          if (RECORD) *v.at(v.born + j, r.owner) = (unsigned int)k;
        }
        ++cre;
      }
    }
    if (ent) red[tid] = dS;
    v.sync();
    // Phase B
    totals();
    if (ent && warp == 1) {
      const double s = warp_sum_shared(red, kT);
      if (lane == 0) s_dS[k & 1] = s;
    }
    if (ent && v.rank == 0u && k > job.k0 && warp == 2) {
      // the entropy of the factor before, whose changes every CTA has left
      double s = lane < C ? *v.at(&s_dS[(k - 1) & 1], lane) : 0.0;
      s = warp_sum(s);
      entropy += s;
      if (lane == 0) job.t.entropy[k - 1] = entropy;
    }
    const unsigned int tail = min(*((volatile unsigned int*)&s_tail), v.L);
    for (unsigned int i = n_scan + tid; i < tail; i += kT) res_link(v, i, cnt, SITE_CREATE_DUP);
    if (tid < (unsigned int)kFW) s_f[(k + 1) & 1][tid] = fw;
    if (tid == 0) {
      s_qn = 0u;
      scanned += n_scan;
    }
    __syncthreads();
    const ResTotals tot = s_tot;
    if (RECORD) tape_n = s_tape_now;
    if (tot.most > v.L) {
      status = RES_ABORT;  // every CTA sees the same counts
      break;
    }
    n_scan = tail;
    peak = max(peak, tot.tail);
    unsigned int live = tot.tail - tot.dead, dead = tot.dead;
    stored_any = true;
    if (job.n_max > 0ull && (unsigned long long)live > job.n_max) {
      unsigned long long T;
      KT Kt;
      res_threshold(v, n_scan, live, job.n_cut, hist, comb, cmag, ckey, &s_ncand, cnt, &T, &Kt);
      auto keep = [&](double a, KT key) {
        const unsigned long long u = mag_of<KT>(a);
        return u > T || (u == T && !key_less(Kt, key));
      };
      unsigned long long tbase = 0ull;
      if (RECORD) {
        // this CTA's share of the tape: one reservation
        if (tid == 0) s_drop = 0u;
        __syncthreads();
        unsigned int nd = 0u;
        for (unsigned int i = tid; i < n_scan; i += kT) {
          const double a = v.amps[i];
          nd += !is_dead(a) && !keep(a, v.keys[i]);
        }
        nd = __reduce_add_sync(0xFFFFFFFFu, nd);
        if (lane == 0 && nd) atomicAdd(&s_drop, nd);
        __syncthreads();
        if (tid == 0) s_tbase = atomicAdd(v.at(&s_tape, 0u), (unsigned long long)s_drop);
        __syncthreads();
        tbase = s_tbase;
      }
      double dC = 0.0;
      const unsigned int kept =
          res_compact(v, n_scan, keep, [&](KT key, double a, unsigned int born, unsigned int rank) {
            if (ent) dC -= entropy_term(a);
            if (RECORD) {
              const unsigned long long at = tbase + rank;
              if (at < job.tape.cap) {
                TapeRecT<KT>& rec = tape_at(job.tape, at);
                rec.key = key;
                rec.val = a;
                rec.born = born;
              } else {
                raise_error(cnt, ERR_TAPE_FULL);
              }
            }
          });
      if (ent) {
        red[tid] = dC;
        __syncthreads();
        if (warp == 1) {
          const double s = warp_sum_shared(red, kT);
          if (lane == 0) s_dS[k & 1] += s;
        }
      }
      if (tid == 0) {
        s_tail = kept;
        s_dead = 0u;
      }
      n_scan = kept;
      res_rehash(v, kept, cnt);
      if (RECORD) tape_n += (unsigned long long)live - job.n_cut;
      cut_total += (unsigned long long)live - job.n_cut;
      live = (unsigned int)job.n_cut;
      dead = 0u;
      ++rebuilds;
    } else if (dead > 64u * C ? 4u * dead > tot.tail : (dead > 0u && 2u * tot.most > v.L)) {
      v.sync();  // every CTA has read the counts
      const unsigned int kept =
          res_compact(v, n_scan, [](double, KT) { return true; }, [](KT, double, unsigned int, unsigned int) {});
      if (tid == 0) {
        s_tail = kept;
        s_dead = 0u;
      }
      n_scan = kept;
      res_rehash(v, kept, cnt);
      dead = 0u;
      ++rebuilds;
    }
    if (RECORD && v.rank == 0u && tid == 0) job.tape.off[k + 1] = tape_n;
    if (!res_room(live, dead, job.bound, v.L, v.logC))
      status = RES_FULL;
    else if (RECORD && tape_n + 3ull * live + 64ull > job.tape.cap)
      status = RES_TAPE;
    ++k;
    v.sync();
  }
  // RES_FULL / RES_TAPE after the last factor are no stops.
  if (k == job.k1 && status != RES_ABORT) status = RES_DONE;
  const bool store = status != RES_ABORT && stored_any;
  v.sync();
  if (store) {
    if (ent && v.rank == 0u && warp == 2) {
      double s = lane < C ? *v.at(&s_dS[(k - 1) & 1], lane) : 0.0;
      s = warp_sum(s);
      entropy += s;
      if (lane == 0) {
        job.t.entropy[k - 1] = entropy;
        cnt->entropy = entropy;
      }
    }
    const unsigned int kept =
        res_compact(v, n_scan, [](double, KT) { return true; }, [](KT, double, unsigned int, unsigned int) {});
    res_store(v, job.t, kept);
    const unsigned long long sr = warp_sum_u64(rot), sc = warp_sum_u64(cre), sn = warp_sum_u64(dnew),
                             so = warp_sum_u64(dold);
    if (lane == 0) {
      if (sr) atomicAdd(&cnt->rotations, sr);
      if (sc) atomicAdd(&cnt->created, sc);
      if (sn) atomicAdd(&cnt->dropped_new, sn);
      if (so) atomicAdd(&cnt->dropped_old, so);
    }
    if (tid == 0) atomicAdd(&cnt->scanned, scanned);
  }
  v.sync();  // every CTA's share is stored and counted
  if (v.rank == 0u && tid == 0) {
    if (store) res_finish(cnt);
    cnt->res_status = status;
    cnt->res_k = store ? k : job.k0;
    cnt->res_cut = store ? cut_total : 0ull;
    cnt->res_rebuilds = store ? rebuilds : 0u;
    cnt->res_peak = peak;
    if (store && RECORD) cnt->tape_n = tape_n;
  }
}

// ---------------------------------------------------------------------------
// Reverse: factors k1 - 1 .. k0 of a table that holds psi_{k1} and mu_{k1}.
// ---------------------------------------------------------------------------
template <class KT>
__global__ void __launch_bounds__(kT, 1) k_res_reverse(ResJob<KT> one, const ResJob<KT>* __restrict__ many,
                                                       ResGeom g) {
  extern __shared__ __align__(16) unsigned char res_smem[];
  constexpr int kFW = sizeof(FactorT<KT>) / 8;
  __shared__ __align__(16) unsigned long long s_f[2][kFW];
  __shared__ unsigned int s_tail, s_dead, s_qn;
  __shared__ ResTotals s_tot;
  __shared__ unsigned long long s_off[kOffRing + 1];
  __shared__ double s_g[2];
  __shared__ unsigned int s_gn[2];  // entries of red in use, by the factor's parity
  const ResLayout lo = res_layout<KT>(g, true);
  const ResJob<KT> job = many ? many[blockIdx.x >> g.logC] : one;
  const ResView<KT> v = res_view<KT>(res_smem, lo, g, true);
  double* const red = reinterpret_cast<double*>(res_smem + lo.red);
  Counters* const cnt = job.t.cnt;
  const unsigned int tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const unsigned int C = 1u << v.logC;

  if (tid == 0) {
    s_tail = s_dead = s_qn = 0u;
    s_g[0] = s_g[1] = 0.0;
    s_gn[0] = s_gn[1] = 0u;
  }
  __syncthreads();
  res_load(v, job.t, &s_tail);
  res_rehash(v, min(s_tail, v.L), cnt);
  v.sync();
  auto totals = [&]() {
    if (warp == 0) {
      const unsigned int tl = lane < C ? *((volatile unsigned int*)v.at(&s_tail, lane)) : 0u;
      const unsigned int dd = lane < C ? *((volatile unsigned int*)v.at(&s_dead, lane)) : 0u;
      const unsigned int st = __reduce_add_sync(0xFFFFFFFFu, tl), sd = __reduce_add_sync(0xFFFFFFFFu, dd);
      const unsigned int mt = __reduce_max_sync(0xFFFFFFFFu, tl);
      if (lane == 0) {
        s_tot.tail = st;
        s_tot.dead = sd;
        s_tot.most = mt;
      }
    }
  };
  totals();
  __syncthreads();
  const bool fits = s_tot.most <= v.L;  // the same in every CTA
  unsigned int n_scan = min(s_tail, v.L);
  unsigned int pairs = 0, compactions = 0;
  unsigned long long scanned = 0;
  int k = job.k1;  // factors from k on are undone
  int status = fits ? RES_DONE : RES_ABORT;
  int off_lo = job.k1 + 1;  // s_off covers [off_lo, off_lo + kOffRing]
  v.sync();

  auto off_at = [&](int x) { return s_off[x - off_lo]; };
  const unsigned int gid = v.rank * kT + tid, gstep = C * kT;
  // the first record of this thread for the factor about to be re-inserted
  bool have = false;
  TapeRecT<KT> pre;
  while (fits) {
    // Iteration k: sweep factor k (none in the first one, where k == k1), and
    // push the records of factor k - 1.
    const bool sweep = k < job.k1, push = k - 1 >= job.k0;
    if (push && k - 2 < off_lo) {  // block-uniform: refill the tape offsets, down to k - kOffRing
      __syncthreads();
      off_lo = max(job.k0, k - kOffRing);
      for (int x = (int)tid; x <= k - off_lo; x += kT) s_off[x] = min(job.tape.off[off_lo + x], job.tape.cap);
      __syncthreads();
      if (!sweep) {
        const unsigned long long x = off_at(k - 1) + gid;
        have = x < off_at(k);
        if (have) pre = tape_at(job.tape, x);
      }
    }
    unsigned long long fw = 0ull;
    if (push && tid < (unsigned int)kFW)
      fw = reinterpret_cast<const unsigned long long*>(job.factors + k - 1)[tid];
    const unsigned long long r0 = push ? off_at(k - 1) : 0ull, r1 = push ? off_at(k) : 0ull;
    if (push) {
      auto send = [&](const TapeRecT<KT>& rec) {
        const unsigned int o = place_of(v, rec.key).owner;
        const unsigned int j = atomicAdd(v.at(&s_tail, o), 1u);
        if (j < v.L) {
          *v.at(v.keys + j, o) = rec.key;
          *v.at(v.amps + j, o) = rec.val;
          *v.at(v.born + j, o) = rec.born;
          *v.at(v.lam + j, o) = 0.0;
        }
      };
      if (have) send(pre);
      for (unsigned long long x = r0 + gid + gstep; x < r1; x += gstep) send(tape_at(job.tape, x));
      // the next iteration's record travels while this one sweeps
      have = false;
      if (k - 2 >= job.k0 && k - 2 >= off_lo) {
        const unsigned long long x = off_at(k - 2) + gid;
        have = x < r0;
        if (have) pre = tape_at(job.tape, x);
      }
    }
    unsigned int used = 0u;
    if (sweep) {
      const FactorT<KT> f = *reinterpret_cast<const FactorT<KT>*>(s_f[k & 1]);
      const unsigned int stamp = 0x80000000u | (unsigned int)k;
      res_scan(v, f, n_scan, &s_qn);
      __syncthreads();
      const unsigned int qn = s_qn;
      double acc = 0.0;
      for (unsigned int q = tid; q < qn; q += kT) {
        const unsigned int w = v.queue[q];
        const unsigned int i = w & 0x7FFFu;
        const bool ex = (w & 0x8000u) != 0u;
        const KT X = v.keys[i];
        const double cX = v.amps[i];
        const KT Y = X ^ (f.occ | f.vir);
        const ResHit r = res_find(v, Y, stamp);
        const bool partner_live = r.state == ALIVE;
        if (!ex && (partner_live || r.state == DEAD_NOW)) continue;  // E's thread owns the pair
        const KT E = ex ? X : Y;
        const int parity = (KeyOps<KT>::popc(E & f.pmask) + f.pconst) & 1;
        const double ss = neg_if(f.s, parity);
        ++pairs;
        if (partner_live) {
          double e0, d0, lE, lD;
          unrotate_pair(f, ss, parity, cX, r.amp, v.lam[i], *v.at(v.lam + r.idx, r.owner), e0, d0, lE, lD, acc);
          if (v.born[i] == (unsigned int)k) {
            v.amps[i] = dead_value(stamp);
            atomicAdd(&s_dead, 1u);
          } else {
            v.amps[i] = e0;
            v.lam[i] = lE;
          }
          if (*v.at(v.born + r.idx, r.owner) == (unsigned int)k) {
            *v.at(v.amps + r.idx, r.owner) = dead_value(stamp);
            atomicAdd(v.at(&s_dead, r.owner), 1u);
          } else {
            *v.at(v.amps + r.idx, r.owner) = d0;
            *v.at(v.lam + r.idx, r.owner) = lD;
          }
        } else {
          double x0, l0;
          unrotate_lone(f, ss, parity, cX, v.lam[i], x0, l0, acc);
          v.amps[i] = x0;
          v.lam[i] = l0;
        }
      }
      used = min(qn, (unsigned int)kT);
      if (tid < used) red[(k & 1) * kT + tid] = acc;
      if (tid == 0) {
        s_gn[k & 1] = used;
        scanned += n_scan;
      }
    }
    v.sync();
    // Phase B
    if (warp == 1 && sweep) {
      const double s = warp_sum_shared(red + (k & 1) * kT, s_gn[k & 1]);
      if (lane == 0) s_g[k & 1] = s;
    }
    if (warp == 2 && v.rank == 0u && k + 1 < job.k1) {
      // dE/dtheta of the factor before, whose sums every CTA has left
      double s = lane < C ? *v.at(&s_g[(k + 1) & 1], lane) : 0.0;
      s = warp_sum(s);
      if (lane == 0) job.grad[k + 1] = 2.0 * s;
    }
    if (tid < (unsigned int)kFW && push) s_f[(k - 1) & 1][tid] = fw;
    if (tid == 0) s_qn = 0u;
    // Counts, hashing and compaction where records came (or, now and then,
    // where the sweep alone may have dropped entries).
    if (push && (r1 > r0 || (k & 7) == 0)) {
      totals();
      const unsigned int tail = min(*((volatile unsigned int*)&s_tail), v.L);
      __syncthreads();
      const ResTotals tot = s_tot;
      if (tot.most > v.L) {
        status = RES_FULL;  // the pushes do not count: factor k - 1 is the host's
        break;
      }
      if (tot.dead > 64u * C ? 3u * tot.dead > tot.tail : (tot.dead > 0u && 2u * tot.most > v.L)) {
        v.sync();  // every CTA has read the counts
        // (pushed entries may repeat the key of a dropped one: the dropped leave)
        const unsigned int kept =
            res_compact(v, tail, [](double, KT) { return true; }, [](KT, double, unsigned int, unsigned int) {});
        if (tid == 0) {
          s_tail = kept;
          s_dead = 0u;
        }
        n_scan = kept;
        res_rehash(v, kept, cnt);
        ++compactions;
      } else {
        for (unsigned int i = n_scan + tid; i < tail; i += kT) res_link(v, i, cnt, SITE_BULK_ALIVE);
        n_scan = tail;
      }
      v.sync();
    } else {
      __syncthreads();
    }
    if (!push) break;
    --k;
  }
  // grad[k] of the last factor swept, once every CTA's sum is there.
  v.sync();
  if (fits && k < job.k1 && v.rank == 0u && warp == 2) {
    double s = lane < C ? *v.at(&s_g[k & 1], lane) : 0.0;
    s = warp_sum(s);
    if (lane == 0) job.grad[k] = 2.0 * s;
  }
  if (fits) {
    const unsigned int kept =
        res_compact(v, n_scan, [](double, KT) { return true; }, [](KT, double, unsigned int, unsigned int) {});
    res_store(v, job.t, kept);
    const unsigned long long sp = warp_sum_u64(pairs);
    if (lane == 0 && sp) atomicAdd(&cnt->rev_pairs, sp);
    if (tid == 0) atomicAdd(&cnt->rev_scanned, scanned);
  }
  v.sync();  // every CTA's share is stored and counted
  if (v.rank == 0u && tid == 0) {
    if (fits) res_finish(cnt);
    cnt->res_status = status;
    cnt->res_k = k;
    cnt->res_rebuilds = fits ? compactions : 0u;
  }
}

// Launch configuration of a resident kernel; attr must outlive cfg.
template <class Kernel, class KT>
cudaError_t res_config(Kernel kernel, const KT&, int n_jobs, const ResGeom& g, bool reverse, cudaStream_t st,
                       cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  const unsigned int smem = res_layout<KT>(g, reverse).bytes;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (g.logC > 3) {  // a cluster of 16 is above the portable size
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cfg->gridDim = dim3((unsigned int)n_jobs << g.logC);
  cfg->blockDim = dim3(kT);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = 1u << g.logC;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  return cudaSuccess;
}

template <class Kernel, class KT>
cudaError_t res_launch(Kernel kernel, const ResJob<KT>& one, const ResJob<KT>* many, int n_jobs, const ResGeom& g,
                       bool reverse, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const cudaError_t e = res_config(kernel, KT{}, n_jobs, g, reverse, st, &cfg, attr);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, kernel, one, many, g);
}

// Entries a CTA holds at most: what fits 227 KB in either kernel.
constexpr int kMostOne = 4096, kMostTwo = 3584;

double largest_share(unsigned long long bound, int logC) {
  const double mean = (double)bound / (double)(1 << logC);
  return logC == 0 ? (double)bound : mean * 1.125 + 6.0 * std::sqrt(mean) + 8.0;
}

template <class KT>
int max_cluster() {
  for (int logC = kMaxLogC; logC >= 0; --logC) {
    ResGeom g{};
    g.logC = logC;
    g.L = sizeof(KT) == 16 ? kMostTwo : kMostOne;
    g.logB = 11;
    int n[2] = {0, 0};
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    if (res_config(k_res_forward<KT, true>, KT{}, 1, g, false, nullptr, &cfg, attr) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n[0], k_res_forward<KT, true>, &cfg) == cudaSuccess &&
        res_config(k_res_reverse<KT>, KT{}, 1, g, true, nullptr, &cfg, attr) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n[1], k_res_reverse<KT>, &cfg) == cudaSuccess && n[0] > 0 && n[1] > 0)
      return logC;
    cudaGetLastError();
  }
  return -1;
}

}  // namespace

int res_max_logC(int key_words) {
  static const int one = max_cluster<unsigned long long>(), two = max_cluster<Key128>();
  return key_words == 2 ? two : one;
}

ResGeom res_geometry(unsigned long long bound, int key_words, int max_logC) {
  const double most = key_words == 2 ? kMostTwo : kMostOne;
  // room for the largest share, and a quarter more for dropped entries
  auto want = [&](int logC) { return 1.25 * largest_share(bound, logC) + 64.0; };
  ResGeom g{};
  g.logC = bound <= 512 ? 0 : bound <= 2048 ? 2 : bound <= 6144 ? 3 : kMaxLogC;
  g.logC = std::min(g.logC, max_logC);
  while (g.logC < max_logC && want(g.logC) > most) ++g.logC;
  g.L = std::max(256, (int)std::min(most, want(g.logC)) / 16 * 16);
  g.logB = 0;  // buckets of four slots, at most half full
  while ((4 << g.logB) < 2 * g.L) ++g.logB;
  return g;
}

bool res_fits(unsigned long long bound, int key_words, int max_logC) {
  return max_logC >= 0 && largest_share(bound, max_logC) <= (key_words == 2 ? kMostTwo : kMostOne);
}

bool res_room_host(unsigned long long bound, const ResGeom& g) {
  return largest_share(bound, g.logC) <= (double)g.L;
}

template <class KT>
cudaError_t launch_res_forward(const ResJob<KT>& one, const ResJob<KT>* many, int n_jobs, const ResGeom& g,
                               int record, cudaStream_t st) {
  return record ? res_launch(k_res_forward<KT, true>, one, many, n_jobs, g, false, st)
                : res_launch(k_res_forward<KT, false>, one, many, n_jobs, g, false, st);
}

template <class KT>
cudaError_t launch_res_reverse(const ResJob<KT>& one, const ResJob<KT>* many, int n_jobs, const ResGeom& g,
                               cudaStream_t st) {
  return res_launch(k_res_reverse<KT>, one, many, n_jobs, g, true, st);
}

#define UCC_RES_INSTANTIATE(KT)                                                                                  \
  template cudaError_t launch_res_forward<KT>(const ResJob<KT>&, const ResJob<KT>*, int, const ResGeom&, int,    \
                                              cudaStream_t);                                                     \
  template cudaError_t launch_res_reverse<KT>(const ResJob<KT>&, const ResJob<KT>*, int, const ResGeom&,         \
                                              cudaStream_t);
UCC_RES_INSTANTIATE(unsigned long long)
UCC_RES_INSTANTIATE(Key128)

}  // namespace ucc
