// Resident passes: a run of factor steps of one wavefunction inside one launch,
// with the whole table in the shared memory of the CTAs that run it: a
// thread-block cluster for tables of up to some 25,000 determinants, every SM
// of the GPU for tables of up to some 700,000.
//
// A table of that size leaves little to do per factor: with a launch or two per
// factor and a dozen per cut, what runs is mostly launch and memory latency.
// Here determinants are owned by the CTA that a hash of their key names.  The
// owner keeps them in entry arrays (key, amplitude, birth factor, adjoint) and a
// local hash of 4-byte slots, and nobody else ever reads or writes them: CTAs
// only send each other messages.  A factor step:
//
//   A  every CTA scans its own keys for linked entries and sends each one's
//      amplitude to the owner of its partner's key;
//   -- barrier: it also sums what every CTA must know --
//   B  every CTA looks up its messages' keys: a stored key makes a pair, whose
//      owner now has both amplitudes and rotates its member; an absent one is
//      the partner that the factor creates.  Linked entries that no message
//      named are alone and are scaled.
//
// A pair's two members send to each other, so each side rotates its own member
// by the same formulas; the only traffic is one message per linked entry and
// the only wait one barrier (inboxes alternate between two buffers).  When the
// step might leave more than N_MAX determinants (the barrier's sums say so) a
// second barrier counts them, with the entries binned around the last cut's
// threshold, and a cut follows: the few entries of the threshold's bin are ranked
// pairwise (a first cut takes a histogram of |c|, 4,096 bins over the exponents that
// amplitudes have).  Dropping, compacting and rehashing are each CTA's own business.  The reverse sweep has the same two
// phases; factor k - 1's tape records travel with factor k's messages.
//
// Inside a cluster messages are remote shared-memory stores and the barrier is
// the cluster's; across the GPU the inboxes lie in L2 and the barrier is one
// 64-bit word whose arrivals carry the sums (a cooperative launch, every wait
// bounded: one that runs out ends the launch, and the host runs the same factors
// with a launch each).
//
// What bounds it: latency, of the barrier (0.8 us in a cluster of sixteen, 2 us
// across the GPU), of a message (0.5 and 1 us) and of the block's own phases.
// Times before (a launch per factor) and with it: a factor of the 64-spin-
// orbital, 10-electron problem at N_MAX 8,000 (6,000 keys scanned, 2,400 pairs, a
// cut after every other factor) 74 and 7.6 us forward, 51 and 7.9 us reverse, the
// gradient's 5,270 factors 655 and 82 ms (72 spin-orbitals, two-word keys: 709 and
// 93); N_MAX 160,000, a factor and its cuts 78 and 11.7 us; 245,025 determinants
// at 24 spin-orbitals, a factor 23.6 and 5.8 us forward, 18 and 7.2 reverse;
// 621,075 at 30, 23.8 and 7.4 us; 24 uneven jobs in one batch, a cluster each,
// 664 and 36 ms; 12 spin-orbitals (225 determinants, one CTA), 2.50 and 0.85 ms.
//
// The arithmetic, the eps rule, the cut's order and the counts are those of the
// launch-per-factor kernels, so states agree bit for bit.
//
// A CTA's share is a binomial draw of the table, so its arrays are sized with a
// margin.  A share or an inbox that outgrows them is flagged at the next
// barrier and the launch ends without having touched the table in global
// memory; the host then runs the same factors with a launch each.  Before a
// step that might outgrow them the launch writes its table back and stops.

#include <algorithm>
#include <cmath>
#include <mutex>

#include "ucc_steps.cuh"

namespace ucc {

namespace {

constexpr int kT = 512;  // threads per CTA
constexpr int kW = kT / 32;
constexpr int kBinBits = 12;
constexpr int kBins = 1 << kBinBits;
constexpr int kCand = 512;     // candidates of a cut ranked pairwise
constexpr int kWinBins = 512;  // bins of the window around the last cut's threshold
constexpr int kWinShift = 44;  // ... of 2^44 in |c|'s bits, 256 an octave
constexpr int kOffRing = 256;  // tape offsets held at a time
constexpr int kMaxC = 16;      // CTAs of a cluster
constexpr int kMaxG = 240;     // CTAs of a grid (arrivals are counted in 8 bits)

// What a barrier sums over the CTAs, in one 64-bit word: arrivals (8 bits),
// CTAs that must abort (8), CTAs that see the tape running low (8), linked
// entries (20), live entries (20).
__device__ __forceinline__ unsigned long long pack_word(bool abort, bool low, unsigned int linked, unsigned int live) {
  return 1ull | ((unsigned long long)abort << 8) | ((unsigned long long)low << 16) |
         ((unsigned long long)linked << 24) | ((unsigned long long)live << 44);
}
__device__ __forceinline__ bool word_abort(unsigned long long w) { return ((w >> 8) & 0xFFull) != 0ull; }
__device__ __forceinline__ bool word_low(unsigned long long w) { return ((w >> 16) & 0xFFull) != 0ull; }
__device__ __forceinline__ unsigned int word_linked(unsigned long long w) { return (unsigned int)(w >> 24) & 0xFFFFFu; }
__device__ __forceinline__ unsigned int word_live(unsigned long long w) { return (unsigned int)(w >> 44); }

__host__ __device__ inline unsigned int up16(unsigned int x) { return (x + 15u) & ~15u; }

// Byte offsets of a CTA's shared arrays, host and device.
struct ResLayout {
  unsigned int keys, amps, lam, born, slots, queue, done, hist, comb, cmag, ckey, win, ent, stage, inkey, ina, inb, bytes;
};

template <class KT>
__host__ __device__ inline ResLayout res_layout(const ResGeom& g, bool reverse) {
  ResLayout o{};
  unsigned int at = 0;
  auto take = [&](unsigned int bytes) {
    const unsigned int r = at;
    at = up16(at + bytes);
    return r;
  };
  const unsigned int L = (unsigned int)g.L, in = g.grid ? 0u : 2u * (unsigned int)g.Lin;
  o.keys = take(L * (unsigned int)sizeof(KT));
  o.amps = take(L * 8u);
  o.born = take(L * 4u);
  o.slots = take(16u << g.logB);
  o.queue = take(L * 2u);
  o.done = take((L + 31u) / 32u * 4u);
  o.inkey = take(in * (unsigned int)sizeof(KT));
  o.ina = take(in * 8u);
  if (reverse) {
    o.lam = take(L * 8u);
    o.inb = take(in * 8u);
    o.stage = take(kT * (unsigned int)sizeof(TapeRecT<KT>));
  } else {
    o.hist = take(g.grid ? kBins * 4u : 2u * kT * 4u);
    o.comb = take(g.grid ? 0u : (kBins * 4u) / (unsigned int)g.ctas);
    o.win = take(g.grid ? 0u : (unsigned int)g.ctas * kWinBins * 2u);
    o.cmag = take(kCand * 8u);
    o.ckey = take((unsigned int)(kCand * sizeof(KT)));
    o.ent = take(g.entropy ? L * 8u : 0u);
  }
  o.bytes = at;
  return o;
}

// A message: a key its receiver owns, an amplitude, and (reverse) the
// sender's adjoint or a tape record's birth factor.
template <class KT>
struct Msg {
  KT key;
  double a;
  unsigned long long b;
};

// Shared words of the message layer.
struct NetShared {
  unsigned long long words[2][kMaxC];  // cluster: every CTA's barrier word
  unsigned int count[2][2];            // cluster: messages received [buffer][kind]
  unsigned long long word;             // grid: the completed barrier word
};

// Messages and barriers inside a cluster: inboxes in the receivers' shared
// memory.  Kind 0 fills an inbox from its start, kind 1 from its end.
template <class KT>
struct ClusterNet {
  static constexpr bool kGrid = false;
  NetShared* s;
  KT* inkey;
  double* ina;
  unsigned long long* inb;
  unsigned int C, rank, Lin, epoch;

  template <class T>
  __device__ __forceinline__ T* at(T* p, unsigned int r) const {
    return cg::this_cluster().map_shared_rank(p, r);
  }
  template <bool B>
  __device__ __forceinline__ void push(int buf, int kind, unsigned int owner, KT key, double a, unsigned long long b) {
    const unsigned int j = atomicAdd(at(&s->count[buf][kind], owner), 1u);
    if (j >= Lin) return;  // the receiver's count says so
    const unsigned int x = (unsigned int)buf * Lin + (kind ? Lin - 1u - j : j);
    *at(inkey + x, owner) = key;
    *at(ina + x, owner) = a;
    if (B) *at(inb + x, owner) = b;
  }
  // A barrier in two halves: work that needs neither side's data fits between
  // them.  wait returns the sum of every CTA's word; messages sent before
  // arrive are there after it.
  __device__ __forceinline__ void arrive(unsigned long long word, Counters*) {
    if (threadIdx.x < C) *at(&s->words[epoch & 1u][rank], threadIdx.x) = word;
    if (C > 1u)
      asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    else
      __syncthreads();
  }
  __device__ __forceinline__ unsigned long long wait(Counters*) {
    const unsigned int e = epoch & 1u;
    ++epoch;
    if (C > 1u) asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    unsigned long long sum = 0ull;
#pragma unroll
    for (int r = 0; r < kMaxC; ++r)
      if ((unsigned int)r < C) sum += s->words[e][r];
    return sum;
  }
  __device__ __forceinline__ unsigned int received(int buf, int kind) const {
    return *((volatile unsigned int*)&s->count[buf][kind]);
  }
  template <bool B>
  __device__ __forceinline__ Msg<KT> get(int buf, int kind, unsigned int j) const {
    const unsigned int x = (unsigned int)buf * Lin + (kind ? Lin - 1u - j : j);
    Msg<KT> m;
    m.key = inkey[x];
    m.a = ina[x];
    m.b = B ? inb[x] : 0ull;
    return m;
  }
  __device__ __forceinline__ void clear(int buf) { s->count[buf][0] = s->count[buf][1] = 0u; }
  __device__ __forceinline__ void leave() {
    if (C > 1u) cg::this_cluster().sync();  // no CTA ends while another may still reach into its memory
  }
};

__device__ __forceinline__ unsigned long long ns_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned long long ld_key(const unsigned long long* p) { return __ldcg(p); }
__device__ __forceinline__ Key128 ld_key(const Key128* p) {
  const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(p));
  return {v.x, v.y};
}

// Both halves of a barrier at once.
template <class Net>
__device__ __forceinline__ unsigned long long net_sync(Net& net, unsigned long long word, Counters* c) {
  net.arrive(word, c);
  return net.wait(c);
}

// Messages and barriers across the GPU: inboxes in global memory (L2).
template <class KT>
struct GridNet {
  static constexpr bool kGrid = true;
  NetShared* s;
  ResControl* ctl;
  KT* inkey;
  double* ina;
  unsigned long long* inb;
  unsigned int C, rank, Lin, epoch;
  unsigned long long wait_ns;

  __device__ __forceinline__ unsigned int* counter(int buf, int kind, unsigned int owner) const {
    return &ctl->count[buf][kind][owner][0];
  }
  template <bool B>
  __device__ __forceinline__ void push(int buf, int kind, unsigned int owner, KT key, double a, unsigned long long b) {
    const unsigned int j = atomicAdd(counter(buf, kind, owner), 1u);
    if (j >= Lin) return;
    const size_t x = ((size_t)buf * C + owner) * Lin + (kind ? Lin - 1u - j : j);
    inkey[x] = key;
    ina[x] = a;
    if (B) inb[x] = b;
  }
  // One 64-bit word per barrier, in a ring of four: arrivals add their words
  // and the sum is complete when it counts all of them.  The word two barriers
  // ahead is cleared by CTA 0 once everybody is past its last use.
  __device__ __forceinline__ void arrive(unsigned long long word, Counters*) {
    __syncthreads();
    if (threadIdx.x == 0) {
      if (rank == 0u) *((volatile unsigned long long*)&ctl->words[(epoch + 2u) & 3u][0]) = 0ull;
      __threadfence();
      atomicAdd(&ctl->words[epoch & 3u][0], word);
    }
  }
  __device__ __forceinline__ unsigned long long wait(Counters* cnt) {
    if (threadIdx.x == 0) {
      unsigned long long* const w = &ctl->words[epoch & 3u][0];
      unsigned long long v = *((volatile unsigned long long*)w);
      if ((v & 0xFFull) != (unsigned long long)C) {
        const unsigned long long t0 = ns_now();
        unsigned int spins = 0u;
        for (;;) {
          v = *((volatile unsigned long long*)w);
          if ((v & 0xFFull) == (unsigned long long)C) break;
          if ((++spins & 255u) == 0u && ns_now() - t0 > wait_ns) {
            raise_error(cnt, ERR_TIMEOUT);
            v = pack_word(true, false, 0u, 0u);
            break;
          }
        }
      }
      __threadfence();
      s->word = v;
    }
    __syncthreads();
    ++epoch;
    return s->word;  // rewritten only after the next barrier's first __syncthreads
  }
  __device__ __forceinline__ unsigned int received(int buf, int kind) const {
    return *((volatile unsigned int*)counter(buf, kind, rank));
  }
  template <bool B>
  __device__ __forceinline__ Msg<KT> get(int buf, int kind, unsigned int j) const {
    const size_t x = ((size_t)buf * C + rank) * Lin + (kind ? Lin - 1u - j : j);
    Msg<KT> m;
    m.key = ld_key(inkey + x);
    m.a = ld_cg(ina + x);
    m.b = B ? ld_cg(inb + x) : 0ull;
    return m;
  }
  __device__ __forceinline__ void clear(int buf) {
    *((volatile unsigned int*)counter(buf, 0, rank)) = 0u;
    *((volatile unsigned int*)counter(buf, 1, rank)) = 0u;
  }
  __device__ __forceinline__ void leave() {}
};

// One CTA's table.
template <class KT>
struct ResView {
  KT* keys;
  double* amps;
  double* lam;
  double* ent;  // the entries' terms of the entropy (null: not recorded)
  unsigned int* born;
  unsigned int* slots;
  unsigned short* queue;
  unsigned int* done;  // a bit per entry: named by a message of this step
  unsigned int L, bmask;
  int logB;
  unsigned int C;
};

template <class KT>
__device__ __forceinline__ ResView<KT> res_view(unsigned char* smem, const ResLayout& o, const ResGeom& g,
                                                bool reverse) {
  ResView<KT> v;
  v.keys = reinterpret_cast<KT*>(smem + o.keys);
  v.amps = reinterpret_cast<double*>(smem + o.amps);
  v.lam = reverse ? reinterpret_cast<double*>(smem + o.lam) : nullptr;
  v.ent = !reverse && g.entropy ? reinterpret_cast<double*>(smem + o.ent) : nullptr;
  v.born = reinterpret_cast<unsigned int*>(smem + o.born);
  v.slots = reinterpret_cast<unsigned int*>(smem + o.slots);
  v.queue = reinterpret_cast<unsigned short*>(smem + o.queue);
  v.done = reinterpret_cast<unsigned int*>(smem + o.done);
  // (shared addresses: keeps the accesses off the generic path)
  __builtin_assume(__isShared(v.keys));
  __builtin_assume(__isShared(v.amps));
  __builtin_assume(__isShared(v.born));
  __builtin_assume(__isShared(v.slots));
  __builtin_assume(__isShared(v.queue));
  __builtin_assume(__isShared(v.done));
  v.L = (unsigned int)g.L;
  v.logB = g.logB;
  v.bmask = (1u << g.logB) - 1u;
  v.C = (unsigned int)g.ctas;
  return v;
}

template <class KT>
__device__ __forceinline__ ClusterNet<KT> make_net(ClusterNet<KT>*, unsigned char* smem, const ResLayout& o,
                                                   const ResGeom& g, const ResNet<KT>&, NetShared* s) {
  ClusterNet<KT> n;
  n.s = s;
  n.inkey = reinterpret_cast<KT*>(smem + o.inkey);
  n.ina = reinterpret_cast<double*>(smem + o.ina);
  n.inb = reinterpret_cast<unsigned long long*>(smem + o.inb);
  n.C = (unsigned int)g.ctas;
  n.rank = g.ctas > 1 ? cg::this_cluster().block_rank() : 0u;
  n.Lin = (unsigned int)g.Lin;
  n.epoch = 0u;
  return n;
}
template <class KT>
__device__ __forceinline__ GridNet<KT> make_net(GridNet<KT>*, unsigned char*, const ResLayout&, const ResGeom& g,
                                                const ResNet<KT>& r, NetShared* s) {
  GridNet<KT> n;
  n.s = s;
  n.ctl = r.ctl;
  n.inkey = r.key;
  n.ina = r.a;
  n.inb = r.b;
  n.C = (unsigned int)g.ctas;
  n.rank = blockIdx.x;
  n.Lin = (unsigned int)g.Lin;
  n.epoch = 0u;
  n.wait_ns = r.wait_ns;
  return n;
}

// Where a key lives: owner CTA, home bucket of four slots, 16-bit tag.  The
// slot hash is folded and multiplied once more: its bits spread determinant
// keys over CTAs and buckets like random draws, which the sizing counts on.
__device__ __forceinline__ unsigned long long place_hash(unsigned long long slot_hash) {
  unsigned long long h = slot_hash;
  h ^= h >> 29;
  h *= kFilterMul;
  return h ^ (h >> 32);
}
template <class KT>
__device__ __forceinline__ unsigned int owner_of(const ResView<KT>& v, KT key) {
  return __umulhi((unsigned int)(place_hash(KeyOps<KT>::slot_hash(key)) >> 32), v.C);
}
template <class KT>
__device__ __forceinline__ void home_of(const ResView<KT>& v, KT key, unsigned int& bucket, unsigned int& tag) {
  const unsigned int lo = (unsigned int)place_hash(KeyOps<KT>::slot_hash(key));
  bucket = lo >> (32 - v.logB);
  tag = (lo << v.logB) >> 16;
}

// The entry of this CTA holding key, or -1.  Slots hold tag << 16 | index + 1,
// are claimed in order inside a bucket and never freed until the hash is
// rebuilt, so a bucket with an empty slot ends the search.
template <class KT>
__device__ __forceinline__ int res_find(const ResView<KT>& v, KT key) {
  unsigned int b, tag;
  home_of(v, key, b, tag);
  for (unsigned int step = 0; step <= v.bmask; ++step) {
    const uint4 q = *reinterpret_cast<const uint4*>(v.slots + 4u * b);
    const unsigned int w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (w[j] == 0u) return -1;
      if ((w[j] >> 16) == tag && v.keys[(w[j] & 0xFFFFu) - 1u] == key) return (int)((w[j] & 0xFFFFu) - 1u);
    }
    b = (b + 1u) & v.bmask;
  }
  return -1;
}

// Hash entry i of this CTA, whose key is not there.
template <class KT>
__device__ __forceinline__ void res_insert(const ResView<KT>& v, KT key, unsigned int i, Counters* c) {
  unsigned int b, tag;
  home_of(v, key, b, tag);
  const unsigned int word = (tag << 16) | (i + 1u);
  for (unsigned int step = 0; step <= v.bmask; ++step) {
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      unsigned int* const s = v.slots + 4u * b + (unsigned int)j;
      if (*((volatile unsigned int*)s) == 0u && atomicCAS(s, 0u, word) == 0u) return;
    }
    b = (b + 1u) & v.bmask;
  }
  raise_error(c, ERR_PROBE_BOUND);
}

// Append (key, a, born[, zero adjoint]); false when the arrays are full.  The
// lanes that append together share one reservation.  The entry is hashed after
// the block's next barrier: searches of this phase never meet a slot whose
// entry is still being written.
template <class KT>
__device__ __forceinline__ bool res_append(const ResView<KT>& v, KT key, double a, unsigned int born,
                                           unsigned int* tail, double ent = 0.0) {
  cg::coalesced_group g = cg::coalesced_threads();
  unsigned int i = 0u;
  if (g.thread_rank() == 0) i = atomicAdd(tail, (unsigned int)g.size());
  i = g.shfl(i, 0) + (unsigned int)g.thread_rank();
  if (i >= v.L) return false;
  v.keys[i] = key;
  v.amps[i] = a;
  v.born[i] = born;
  if (v.lam) v.lam[i] = 0.0;
  if (v.ent) v.ent[i] = ent;
  return true;
}

// Rebuild this CTA's hash over its first n entries.  Every thread calls this.
template <class KT>
__device__ __forceinline__ void res_rehash(const ResView<KT>& v, unsigned int n, Counters* c) {
  uint4* const s = reinterpret_cast<uint4*>(v.slots);
  for (unsigned int x = threadIdx.x; x <= v.bmask; x += kT) s[x] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (unsigned int i = threadIdx.x; i < n; i += kT) res_insert(v, v.keys[i], i, c);
  __syncthreads();
}

// Compact this CTA's first n entries in place: live entries that keep(a, key)
// accepts move down in order, drop(key, a, born, rank) is called for the live
// ones it rejects, rank counting them.  Returns the number kept.  Every thread
// calls this; the hash is stale afterwards.
template <class KT, class Keep, class Drop>
__device__ __forceinline__ unsigned int res_compact(const ResView<KT>& v, unsigned int n, Keep keep, Drop drop) {
  __shared__ unsigned int s_kd[2][kW];  // kept | dropped << 16 of a round's warps, alternating
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned int below_me = (1u << lane) - 1u;
  unsigned int kept = 0, dropped = 0, round = 0;
  for (unsigned int base = 0; base < n; base += kT, ++round) {  // block-uniform
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
      if (v.ent) lam = v.ent[i];  // (never both)
    }
    const bool kp = live && keep(a, key);
    const unsigned int mk = __ballot_sync(0xFFFFFFFFu, kp), md = __ballot_sync(0xFFFFFFFFu, live && !kp);
    if (lane == 0) s_kd[round & 1u][warp] = __popc(mk) | (__popc(md) << 16);
    __syncthreads();  // ... and every thread has read its entry
    const unsigned int c = lane < (unsigned int)kW ? s_kd[round & 1u][lane] : 0u;
    unsigned int incl = c;
#pragma unroll
    for (int o = 1; o < kW; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if ((int)lane >= o) incl += y;
    }
    const unsigned int total = __shfl_sync(0xFFFFFFFFu, incl, kW - 1);
    const unsigned int mine = __shfl_sync(0xFFFFFFFFu, incl - c, warp);
    const unsigned int pk = mine & 0xFFFFu, pd = mine >> 16, tk = total & 0xFFFFu, td = total >> 16;
    if (kp) {
      const unsigned int to = kept + pk + __popc(mk & below_me);
      v.keys[to] = key;
      v.amps[to] = a;
      v.born[to] = born;
      if (v.lam) v.lam[to] = lam;
      if (v.ent) v.ent[to] = lam;
    } else if (live) {
      drop(key, a, born, dropped + pd + __popc(md & below_me));
    }
    kept += tk;
    dropped += td;
  }
  __syncthreads();
  return kept;
}

template <class KT>
__device__ __forceinline__ unsigned int res_squeeze(const ResView<KT>& v, unsigned int n) {
  return res_compact(v, n, [](double, KT) { return true; }, [](KT, double, unsigned int, unsigned int) {});
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
    if (lane == 0) v.done[base >> 5] = 0u;  // no message of this step yet
    if (mk == 0u) continue;
    unsigned int at = 0u;
    if (lane == 0) at = atomicAdd(qn, __popc(mk));
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (act) v.queue[at + __popc(mk & below_me)] = (unsigned short)(i | (ex ? 0x8000u : 0u));
  }
}

// *to += the warp's sum of x.  Called between the halves of a barrier, where
// the chain of FP64 adds (slow on this GPU) costs nothing; warps without a
// contribution skip it.
__device__ __forceinline__ void add_sum(double* to, double x) {
  if (!__any_sync(0xFFFFFFFFu, nonzero(x))) return;
  x = warp_sum(x);
  if ((threadIdx.x & 31u) == 0u) atomicAdd(to, x);
}

__device__ __forceinline__ unsigned long long mag_of(double a) {
  return (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull;
}

// First histogram digit of a magnitude: exponents 2^-31 .. 2^0 and seven bits
// of the mantissa, clamped at both ends (monotone in |c|; amplitudes of a
// normalised state have no larger exponent, and the threshold of a cut rarely
// lies below: the passes that follow find it there too).
__device__ __forceinline__ int coarse_digit(unsigned long long u) {
  const int e = (int)(u >> 52) - (1023 - 31);
  if (e < 0) return 0;
  if (e > 31) return kBins - 1;
  return (e << 7) | (int)((u >> 45) & 127ull);
}

// This CTA's share of the table in global memory, appended and hashed; false
// when it did not fit.  Every thread of every CTA calls this.
template <class KT, class Net>
__device__ __forceinline__ bool res_load(const ResView<KT>& v, Net& net, const TableT<KT>& t, unsigned int* tail) {
  const unsigned int n = (unsigned int)min(*((volatile unsigned long long*)&t.cnt->n_tail), t.cap_n);
  auto take = [&](KT key, unsigned int i) {
    const unsigned int j = atomicAdd(tail, 1u);
    if (j >= v.L) return;
    v.keys[j] = key;
    v.amps[j] = t.amps[i];
    v.born[j] = t.born[i];
    if (v.lam) v.lam[j] = t.lam[i];
    if (v.ent) v.ent[j] = entropy_term(v.amps[j]);
  };
  bool ok = true;
  if constexpr (Net::kGrid) {
    // a slice each, its keys and indices sent to their owners
    for (unsigned int i = net.rank * kT + threadIdx.x; i < n; i += net.C * kT) {
      if (is_dead(t.amps[i])) continue;
      const KT key = t.keys[i];
      net.template push<false>(0, 0, owner_of(v, key), key, __longlong_as_double((long long)i), 0ull);
    }
    ok = !word_abort(net_sync(net, pack_word(false, false, 0u, 0u), t.cnt));
    const unsigned int got = net.received(0, 0);
    if (ok)
      for (unsigned int x = threadIdx.x; x < min(got, net.Lin); x += kT) {
        const Msg<KT> m = net.template get<false>(0, 0, x);
        take(m.key, (unsigned int)__double_as_longlong(m.a));
      }
    __syncthreads();
    if (threadIdx.x == 0) net.clear(0);
    ok = ok && got <= net.Lin;
  } else {
    // small tables: every CTA reads all keys and keeps its own
    for (unsigned int i = threadIdx.x; i < n; i += kT) {
      if (is_dead(t.amps[i])) continue;
      const KT key = t.keys[i];
      if (owner_of(v, key) == net.rank) take(key, i);
    }
  }
  __syncthreads();
  res_rehash(v, min(*((volatile unsigned int*)tail), v.L), t.cnt);
  return ok && *((volatile unsigned int*)tail) <= v.L;
}

// Write this CTA's n entries (compacted: all live) to the table in global
// memory, in the range it reserves there.  Every thread calls this.
template <class KT>
__device__ __forceinline__ void res_store(const ResView<KT>& v, const TableT<KT>& t, unsigned int n) {
  __shared__ unsigned long long s_base;
  if (threadIdx.x == 0) {
    atomicAdd(&t.cnt->res_stored, 1u);
    s_base = atomicAdd(&t.cnt->res_n, (unsigned long long)n);
  }
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

// The largest share of a CTA of `most` entries spread over C CTAs: the mean, a
// little for the hash, and six standard deviations.
__host__ __device__ inline float largest_share(float most, int C) {
  const float mean = most / (float)C;
  return C == 1 ? most : mean * 1.03f + 6.0f * sqrtf(mean) + 8.0f;
}

// Whether a CTA's dropped entries should leave: they are a third of its
// entries, or an eighth where more than half of its room is taken.  Its room is a
// quarter above the largest share of live ones, so what may still come fits -- except
// where its shared memory holds less than that quarter (from some 600,000 one-word
// entries on the GPU): with the last ninth of the room taken they leave from 3 % on,
// so that a step may add a ninth.  (An exact test in the step itself, on the messages
// received, costs the energy at 24 spin-orbitals 0.4 % and, with two-word keys, the
// gradient at 72 3 %.  A cluster's room is never short: the second rule in its kernels,
// and below a look at the last barrier, whose waits cannot run out there, took the
// forward pass at N_MAX 8,000 from 40.3 to 40.6 ms.)
template <class Net>
__device__ __forceinline__ bool res_crowded(unsigned int n, unsigned int dead, unsigned int L) {
  if constexpr (Net::kGrid) {
    if (dead == 0u) return false;
    if (2u * n > L) return (9u * n > 8u * L ? 32u : 8u) * dead > n;
    return dead > 64u && 3u * dead > n;
  }
  return dead > 64u ? 3u * dead > n || (2u * n > L && 8u * dead > n) : dead > 0u && 2u * n > L && 8u * dead > n;
}

// Exclusive block prefix of one count per thread; *total in every thread.
__device__ __forceinline__ unsigned int block_scan(unsigned int mine, unsigned int* s_w) {
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  unsigned int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if ((int)lane >= o) incl += y;
  }
  __syncthreads();
  if (lane == 31u) s_w[warp] = incl;
  __syncthreads();
  unsigned int before = incl - mine;
#pragma unroll
  for (int x = 0; x < kW; ++x)
    if ((unsigned int)x < warp) before += s_w[x];
  return before;
}

// Shared arrays of a cut.
template <class KT>
struct CutShared {
  unsigned int *hist, *comb;
  uint4* win;  // cluster: every CTA's window, 16 bits a bin
  unsigned long long* cmag;
  KT* ckey;
};

// A cut's threshold lies near the last one's: before the barrier that counts
// the live entries, every CTA bins those within an octave of the last threshold
// (512 bins from `lo` up) and counts the ones above, and sends the counts along.
// When the cut is due, every CTA then knows the threshold's bin without another
// barrier; the full histogram takes one across the GPU and two in a cluster.  The
// gradient of the 64-spin-orbital, 10-electron problem at N_MAX 8,000 went from 90
// to 82 ms with it, its energy at N_MAX 160,000 from 73 to 64, two-word keys at 8,000
// from 102 to 93.  The first cut, and one whose threshold left the window or whose
// bin is too full, take the full histogram.
struct Window {
  bool known;                  // lo is set
  unsigned long long lo;
  int buf;                     // grid: the buffer of the next count
};
struct WindowShared {
  unsigned int above, aboves[kMaxC], found, bin, rest, cnt;
  unsigned int ncand;  // cluster, CTA 0's: the candidates collected
  unsigned int w[kW];
};

template <class KT, class Net>
__device__ __forceinline__ void window_count(const ResView<KT>& v, Net& net, unsigned int n, const Window& win,
                                             const CutShared<KT>& cs, WindowShared& ws) {
  const unsigned int tid = threadIdx.x;
  unsigned int above = 0u;
  for (unsigned int i = tid; i < n; i += kT) {
    const double a = v.amps[i];
    if (is_dead(a)) continue;
    const unsigned long long u = mag_of(a);
    if (u < win.lo) continue;
    const unsigned long long b = (u - win.lo) >> kWinShift;
    if (b < (unsigned long long)kWinBins)
      atomicAdd(&cs.hist[b], 1u);
    else
      ++above;
  }
  above = __reduce_add_sync(0xFFFFFFFFu, above);
  if ((tid & 31u) == 0u && above) atomicAdd(&ws.above, above);
  __syncthreads();
  static_assert(kWinBins == kT, "a bin per thread");
  if constexpr (Net::kGrid) {
    if (cs.hist[tid]) atomicAdd(&net.ctl->win[win.buf][tid], cs.hist[tid]);
    if (tid == 0 && ws.above) atomicAdd(&net.ctl->win[win.buf][kWinBins], ws.above);
  } else {
    constexpr unsigned int kPieces = kWinBins / 8;
    for (unsigned int x = tid; x < net.C * kPieces; x += kT) {
      const unsigned int to = x / kPieces, p = x % kPieces;
      const unsigned int* h = cs.hist + 8u * p;
      *net.at(cs.win + net.rank * kPieces + p, to) =
          make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
    }
    if (tid < net.C) *net.at(&ws.aboves[net.rank], tid) = ws.above;
  }
}

// After that barrier: the bin of the n_cut-th entry (ws.found, bin, rest, cnt);
// always called after window_count, also when no cut is due (it clears).
template <class KT, class Net>
__device__ __forceinline__ void window_pick(Net& net, Window& win, unsigned int n_cut, bool due,
                                            const CutShared<KT>& cs, WindowShared& ws) {
  const unsigned int tid = threadIdx.x, b = (unsigned int)kWinBins - 1u - tid;  // largest first
  cs.hist[tid] = 0u;
  if (tid == 0) {
    ws.above = 0u;
    ws.found = 0u;
  }
  if constexpr (Net::kGrid) {
    // the other buffer's readers are all past this barrier
    for (unsigned int x = net.rank * kT + tid; x <= (unsigned int)kWinBins; x += net.C * kT)
      net.ctl->win[win.buf ^ 1][x] = 0u;
  }
  if (due) {
    unsigned int mine = 0u, above = 0u;
    if constexpr (Net::kGrid) {
      mine = __ldcg(&net.ctl->win[win.buf][b]);
      above = __ldcg(&net.ctl->win[win.buf][kWinBins]);
    } else {
      const unsigned short* const h = reinterpret_cast<const unsigned short*>(cs.win);
#pragma unroll
      for (int r = 0; r < kMaxC; ++r)
        if ((unsigned int)r < net.C) {
          mine += h[(unsigned int)(r * kWinBins) + b];
          above += ws.aboves[r];
        }
    }
    const unsigned int before = above + block_scan(mine, ws.w);
    if (before < n_cut && n_cut <= before + mine) {
      ws.found = mine <= (unsigned int)kCand ? 1u : 0u;
      ws.bin = b;
      ws.rest = n_cut - before;
      ws.cnt = mine;
    }
  }
  win.buf ^= 1;
  __syncthreads();
}

// The threshold of the cut over all CTAs: the N_CUT-th live entry by (|c|
// descending, key ascending), as (*T, *Kt) in every thread.  n: this CTA's
// entries; live: all CTAs' live ones.  Without a bin from the window, passes
// narrow the threshold's bin until it holds at most kCand entries (the first
// pass nearly always does).  The bin's entries are collected and ranked by every
// CTA.  False: a barrier timed out.
template <class KT, class Net>
__device__ __forceinline__ bool res_threshold(const ResView<KT>& v, Net& net, unsigned int n, unsigned int live,
                                              unsigned long long n_cut, const CutShared<KT>& cs, const Window& win,
                                              WindowShared& ws, Counters* cnt, unsigned long long* T, KT* Kt) {
  using K = KeyOps<KT>;
  __shared__ unsigned int s_slice, s_slices[kMaxC], s_from, s_cum, s_bin, s_rest, s_cnt, s_list;
  __shared__ unsigned int s_w[kW];
  __shared__ unsigned long long s_T;
  __shared__ __align__(16) unsigned long long s_Kt[2];
  constexpr unsigned int kPer = kBins / kT;
  const unsigned int tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const unsigned long long word = pack_word(false, false, 0u, 0u);
  const unsigned int bins = Net::kGrid ? (unsigned int)kBins : (unsigned int)kBins / net.C;  // of a slice
  const bool windowed = win.known && ws.found != 0u;
  unsigned int target = windowed ? ws.rest : (unsigned int)n_cut, count = windowed ? ws.cnt : live;
  const unsigned long long wlo = windowed ? win.lo : 0ull, wbin = windowed ? ws.bin : 0ull;
  int coarse = -1;
  unsigned long long pu = 0, mu = 0, phi = 0, mhi = 0, plo = 0, mlo = 0;  // digits fixed so far and their masks
  auto inside = [&](unsigned long long u, KT key) {
    if (windowed) return u >= wlo && ((u - wlo) >> kWinShift) == wbin;
    return (coarse < 0 || coarse_digit(u) == coarse) && (u & mu) == pu && (K::hi(key) & mhi) == phi &&
           (K::lo(key) & mlo) == plo;
  };
  if (tid == 0) {
    s_slice = 0u;
    s_list = 0u;
  }
  // pass 0: the coarse digit; 1 to 6: |c| from the top; then the key's high word (if any), then its low one
  for (int pass = windowed ? 99 : 0; pass <= 6 + 6 * K::kWords && (pass == 0 || count > (unsigned int)kCand); ++pass) {
    const int d = pass == 0 ? 0 : (pass - 1) % 6;
    const int which = pass <= 6 ? 0 : (K::kWords == 2 && pass <= 12 ? 2 : 1);  // 0 |c|, 1 low word, 2 high word
    const int shift = max(0, 64 - kBinBits * (d + 1));
    const int width = min(kBinBits, 64 - kBinBits * d);
    const bool down = which == 0;  // |c| from the largest bin down, keys from the smallest up
    for (unsigned int i = tid; i < n; i += kT) {
      const double a = v.amps[i];
      if (is_dead(a)) continue;
      const unsigned long long u = mag_of(a);
      const KT key = v.keys[i];
      if (!inside(u, key)) continue;
      const unsigned long long x = which == 0 ? u : (which == 1 ? K::lo(key) : K::hi(key));
      const unsigned int b =
          pass == 0 ? (unsigned int)coarse_digit(u) : (unsigned int)((x >> shift) & ((1ull << width) - 1ull));
      if constexpr (Net::kGrid)
        atomicAdd(&cs.hist[b], 1u);
      else
        atomicAdd(net.at(cs.comb + (b & (bins - 1u)), b / bins), 1u);
    }
    unsigned int c[kPer];
    unsigned int want = target, base = 0u, nb = (unsigned int)kBins, per = kPer;
    if constexpr (Net::kGrid) {
      // this CTA's bins into the GPU's histogram, then all of it read by everyone
      __syncthreads();
      for (unsigned int b = tid; b < (unsigned int)kBins; b += kT) {
        const unsigned int h = cs.hist[b];
        cs.hist[b] = 0u;
        if (h) atomicAdd(&net.ctl->hist[b], h);
      }
      if (word_abort(net_sync(net, word, cnt))) return false;
#pragma unroll
      for (unsigned int j = 0; j < kPer; ++j) {
        const unsigned int o = tid * kPer + j;
        c[j] = __ldcg(&net.ctl->hist[down ? (unsigned int)kBins - 1u - o : o]);
      }
    } else {
      // every CTA holds a slice of the bins; then the target's slice is read by everyone
      const unsigned int C = net.C;
      nb = bins;
      per = (nb + kT - 1u) / kT;
      net_sync(net, word, cnt);
      unsigned int sum = 0u;
      for (unsigned int b = tid; b < nb; b += kT) sum += cs.comb[b];
      sum = __reduce_add_sync(0xFFFFFFFFu, sum);
      if (lane == 0 && sum) atomicAdd(&s_slice, sum);
      __syncthreads();
      if (tid < C) *net.at(&s_slices[net.rank], tid) = s_slice;
      net_sync(net, word, cnt);
      if (warp == 0) {
        if (lane == 0) s_from = s_cum = s_slice = 0u;
        __syncwarp();
        const unsigned int r = down ? C - 1u - lane : lane;
        const unsigned int mine = lane < C ? s_slices[r] : 0u;
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
      const unsigned int from = s_from;
      want = target - s_cum;
      base = from * nb;
#pragma unroll
      for (unsigned int j = 0; j < kPer; ++j) {
        const unsigned int o = tid * per + j;
        c[j] = j < per && o < nb ? *net.at(cs.comb + (down ? nb - 1u - o : o), from) : 0u;
      }
    }
    unsigned int mine = 0u;
#pragma unroll
    for (unsigned int j = 0; j < kPer; ++j) mine += c[j];
    if (tid == 0) {  // what a histogram short of the target (an inconsistent count) would leave
      s_bin = s_cnt = 0u;
      s_rest = 1u;
    }
    const unsigned int before = block_scan(mine, s_w);
    if (before < want && want <= before + mine) {
      unsigned int cum = before;
#pragma unroll
      for (unsigned int j = 0; j < kPer; ++j) {
        if (cum < want && want <= cum + c[j]) {
          const unsigned int o = tid * per + j;
          s_bin = base + (down ? nb - 1u - o : o);
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
    } else if (which == 0) {
      pu |= bin << shift;
      mu |= dm;
    } else if (which == 1) {
      plo |= bin << shift;
      mlo |= dm;
    } else {
      phi |= bin << shift;
      mhi |= dm;
    }
    if (count > (unsigned int)kCand) {  // another pass: the histogram is cleared between two barriers
      if (word_abort(net_sync(net, word, cnt))) return false;
      if constexpr (Net::kGrid) {
        for (unsigned int b = net.rank * kT + tid; b < (unsigned int)kBins; b += net.C * kT) net.ctl->hist[b] = 0u;
      } else {
        for (unsigned int b = tid; b < bins; b += kT) cs.comb[b] = 0u;
      }
      if (word_abort(net_sync(net, word, cnt))) return false;
    }
    __syncthreads();
  }
  // every CTA's entries of the bin, to all
  const unsigned int nc = min(count, (unsigned int)kCand);
  for (unsigned int i = tid; i < n; i += kT) {
    const double a = v.amps[i];
    if (is_dead(a)) continue;
    const unsigned long long u = mag_of(a);
    const KT key = v.keys[i];
    if (!inside(u, key)) continue;
    if constexpr (Net::kGrid) {
      const unsigned int q = atomicAdd(&net.ctl->ncand, 1u);
      if (q < (unsigned int)kCand) {
        net.ctl->cand_mag[q] = u;
        net.ctl->cand_key[2 * q] = K::lo(key);
        net.ctl->cand_key[2 * q + 1] = K::hi(key);
      }
    } else {
      const unsigned int q = atomicAdd(net.at(&ws.ncand, 0u), 1u);
      if (q < (unsigned int)kCand)
        for (unsigned int r = 0; r < net.C; ++r) {
          *net.at(cs.cmag + q, r) = u;
          *net.at(cs.ckey + q, r) = key;
        }
    }
  }
  if (word_abort(net_sync(net, word, cnt))) return false;
  if constexpr (Net::kGrid) {
    for (unsigned int x = tid; x < nc; x += kT) {
      cs.cmag[x] = ld_cg(&net.ctl->cand_mag[x]);
      cs.ckey[x] = K::from_words(ld_cg(&net.ctl->cand_key[2 * x]), ld_cg(&net.ctl->cand_key[2 * x + 1]));
    }
    // the histogram and the list are next used after other barriers
    if (!windowed)
      for (unsigned int b = net.rank * kT + tid; b < (unsigned int)kBins; b += net.C * kT) net.ctl->hist[b] = 0u;
    if (net.rank == 0u && tid == 0) net.ctl->ncand = 0u;
    __syncthreads();
  } else {
    // (next used after other barriers)
    if (tid == 0) ws.ncand = 0u;
    if (!windowed)
      for (unsigned int b = tid; b < bins; b += kT) cs.comb[b] = 0u;
  }
  // One thread per candidate.  Candidates of an unclamped bin share the bits
  // above 2^45 (of the window's, above 2^44 from lo on): nine bits at a time (the
  // block's own histogram) narrow them to a few, which are ranked pairwise;
  // ranking all of them so would cost more than the rest of the cut.
  static_assert(kCand == kT && 2 * kT <= kBins, "a candidate per thread");
  bool in = tid < nc;
  unsigned int left = nc;
  const bool narrow = windowed || (coarse > 0 && coarse < kBins - 1);
  for (int sh = windowed ? kWinShift - 9 : 36; sh > -9 && left > 24u && narrow; sh -= 9) {
    // (the last digit of the window's may repeat bits that are settled)
    const unsigned int o = in ? 511u - ((unsigned int)((cs.cmag[tid] - wlo) >> max(sh, 0)) & 511u) : 0u;  // largest first
    if (in) atomicAdd(&cs.hist[o], 1u);
    __syncthreads();
    const unsigned int mine = cs.hist[tid];
    const unsigned int before = block_scan(mine, s_w);  // (every count is read: it synchronises)
    cs.hist[tid] = 0u;
    if (before < target && target <= before + mine) {
      s_bin = tid;
      s_rest = target - before;
      s_cnt = mine;
    }
    __syncthreads();
    in = in && o == s_bin;
    target = s_rest;
    left = s_cnt;
    __syncthreads();
  }
  if (in) cs.hist[kT + atomicAdd(&s_list, 1u)] = tid;
  __syncthreads();
  if (in) {
    const unsigned long long u = cs.cmag[tid];
    const KT key = cs.ckey[tid];
    unsigned int before = 0u;
    for (unsigned int y = 0; y < left; ++y) {
      const unsigned int j = cs.hist[kT + y];
      before += (cs.cmag[j] > u || (cs.cmag[j] == u && key_less(cs.ckey[j], key))) ? 1u : 0u;
    }
    if (before + 1u == target) {
      s_T = u;
      s_Kt[0] = K::lo(key);
      s_Kt[1] = K::hi(key);
    }
  }
  __syncthreads();
  cs.hist[kT + tid] = 0u;  // all zero again
  if (nc == 0u && tid == 0) raise_consistency(cnt, SITE_CUT_COUNT, live);
  *T = s_T;
  *Kt = K::from_words(s_Kt[0], s_Kt[1]);
  return true;
}

// The end of a launch, by CTA 0 once every CTA has stored its entries: they
// become the table, and the per-factor counts of tape records (off, or null)
// and changes of the entropy (ent, or null) of factors [k0, k1) become running
// sums.  Chunks per thread, then a prefix over the threads; scratch: 16 kT
// bytes of shared memory that nothing else uses any more.
__device__ __forceinline__ void res_finish(Counters* c, unsigned long long* off, double* ent, int k0, int k1,
                                           unsigned char* scratch) {
  unsigned long long* const s_n = reinterpret_cast<unsigned long long*>(scratch);
  double* const s_d = reinterpret_cast<double*>(scratch) + kT;
  const int n = k1 - k0, tid = (int)threadIdx.x;
  const int per = (n + kT - 1) / kT, lo = k0 + min(n, tid * per), hi = k0 + min(n, (tid + 1) * per);
  if (off || ent) {
    unsigned long long sn = 0ull;
    double sd = 0.0;
    for (int k = lo; k < hi; ++k) {
      if (off) sn += __ldcg(&off[k + 1]);
      if (ent) sd += __ldcg(&ent[k]);
    }
    s_n[tid] = sn;
    s_d[tid] = sd;
    __syncthreads();
    for (int o = 1; o * per < n; o <<= 1) {  // inclusive prefix (Hillis-Steele) over the threads with a chunk
      const unsigned long long a = tid >= o ? s_n[tid - o] : 0ull;
      const double b = ent && tid >= o ? s_d[tid - o] : 0.0;
      __syncthreads();
      s_n[tid] += a;
      if (ent) s_d[tid] += b;
      __syncthreads();
    }
    sn = (off ? __ldcg(&off[k0]) : 0ull) + (tid ? s_n[tid - 1] : 0ull);
    const double e0 = ent ? c->entropy : 0.0;
    sd = e0 + (tid ? s_d[tid - 1] : 0.0);
    __syncthreads();
    if (ent && tid == 0) c->entropy = e0 + s_d[(n - 1) / per];
    for (int k = lo; k < hi; ++k) {
      if (off) {
        sn += __ldcg(&off[k + 1]);
        off[k + 1] = sn;
      }
      if (ent) {
        sd += __ldcg(&ent[k]);
        ent[k] = sd;
      }
    }
  }
  if (tid == 0) {
    const unsigned long long m = ld_cg(&c->res_n);
    c->n_tail = m;
    c->n_scan = m;
    c->n_dead = 0ull;
    c->res_n = 0ull;
    c->res_stored = 0u;
    c->stop_k = -1;
  }
}

// ---------------------------------------------------------------------------
// Forward: factors [k0, k1) with the eps rule and the cut.
// ---------------------------------------------------------------------------
template <class KT, bool RECORD, class Net>
__global__ void __launch_bounds__(kT, 1) k_res_forward(ResJob<KT> one, const ResJob<KT>* __restrict__ many,
                                                       ResGeom g, ResNet<KT> rnet) {
  extern __shared__ __align__(16) unsigned char res_smem[];
  constexpr int kFW = sizeof(FactorT<KT>) / 8;
  __shared__ __align__(16) unsigned long long s_f[4][kFW];  // a ring: factors travel two steps ahead
  __shared__ unsigned int s_tail, s_dead, s_qn, s_drop;
  __shared__ int s_full, s_low;
  __shared__ unsigned long long s_tbase;
  __shared__ NetShared s_net;
  if (Net::kGrid && blockIdx.x != 0u && blockIdx.x + 1u == rnet.skip_block) return;
  const ResLayout lo = res_layout<KT>(g, false);
  const ResJob<KT> job = many ? many[blockIdx.x / (unsigned int)g.ctas] : one;
  const ResView<KT> v = res_view<KT>(res_smem, lo, g, false);
  CutShared<KT> cs;
  cs.hist = reinterpret_cast<unsigned int*>(res_smem + lo.hist);
  cs.comb = reinterpret_cast<unsigned int*>(res_smem + lo.comb);
  cs.win = reinterpret_cast<uint4*>(res_smem + lo.win);
  cs.cmag = reinterpret_cast<unsigned long long*>(res_smem + lo.cmag);
  cs.ckey = reinterpret_cast<KT*>(res_smem + lo.ckey);
  __shared__ WindowShared s_win;
  Window win{false, 0ull, 0};
  Counters* const cnt = job.t.cnt;
  const unsigned int tid = threadIdx.x, lane = tid & 31u;
  const bool ent = v.ent != nullptr && job.t.entropy != nullptr;
  double dS_due = 0.0;  // this thread's share of the last factor's change of the entropy

  if (tid == 0) {
    s_tail = s_dead = s_qn = 0u;
    s_full = s_low = 0;
    s_win.above = s_win.found = s_win.ncand = 0u;
    s_net.count[0][0] = s_net.count[0][1] = s_net.count[1][0] = s_net.count[1][1] = 0u;
  }
  for (unsigned int b = tid; b < (g.grid ? (unsigned int)kBins : 2u * kT); b += kT) cs.hist[b] = 0u;
  if (!g.grid)
    for (unsigned int b = tid; b < (unsigned int)kBins / (unsigned int)g.ctas; b += kT) cs.comb[b] = 0u;
  auto factor_word = [&](int k) -> unsigned long long {
    return tid < (unsigned int)kFW && k < job.k1 ? reinterpret_cast<const unsigned long long*>(job.factors + k)[tid]
                                                 : 0ull;
  };
  // What the factors' counts are added to (the first addition comes barriers later).
  if ((g.grid ? blockIdx.x : blockIdx.x % (unsigned int)g.ctas) == 0u)
    for (int x = job.k0 + (int)tid; x < job.k1; x += kT) {
      if (RECORD) job.tape.off[x + 1] = 0ull;
      if (ent) job.t.entropy[x] = 0.0;
    }
  if (tid < (unsigned int)kFW) {
    s_f[job.k0 & 3][tid] = factor_word(job.k0);
    s_f[(job.k0 + 1) & 3][tid] = factor_word(job.k0 + 1);
  }
  unsigned long long fw = factor_word(job.k0 + 2);
  Net net = make_net(static_cast<Net*>(nullptr), res_smem, lo, g, rnet, &s_net);
  __syncthreads();
  net.leave();  // (a cluster's CTAs are all set up before the first message)
  const bool loaded = res_load(v, net, job.t, &s_tail);
  if (tid == 0 && !loaded) s_full = 1;

  int status = RES_DONE, k = job.k0;
  unsigned int n_scan = min(s_tail, v.L);
  unsigned int rot = 0, cre = 0, dnew = 0, dold = 0, rebuilds = 0, peak = 0;
  unsigned long long scanned = 0, cut_total = 0;
  // records that one step (and the stop after it) may need
  const unsigned long long slack = 6ull * job.most;

  // A dropped live entry's tape record.
  auto record = [&](KT key, double val, unsigned int born) {
    const unsigned long long at = aggregated_add(&cnt->tape_n);
    if (at + slack >= job.tape.cap) s_low = 1;
    if (at < job.tape.cap) {
      TapeRecT<KT>& rec = tape_at(job.tape, at);
      rec.key = key;
      rec.val = val;
      rec.born = born;
    } else {
      raise_error(cnt, ERR_TAPE_FULL);
    }
    atomicAdd(&s_drop, 1u);
  };

  // What entry at's new amplitude changes in the entropy; its old term is kept, so
  // a rotation takes one logarithm (with the old term taken anew, the 315 factors of
  // 3,136 determinants at 16 spin-orbitals: 2.2 ms, so 1.8).
  auto new_term = [&](int at, double c, bool out) {
    const double was = v.ent[at], now = out ? 0.0 : entropy_term(c);
    v.ent[at] = now;
    return now - was;
  };

  while (k < job.k1) {
    const FactorT<KT> f = *reinterpret_cast<const FactorT<KT>*>(s_f[k & 3]);
    const KT m = f.occ | f.vir;
    const unsigned int stamp = (unsigned int)(k + 1);
    const int buf = (k - job.k0 + 1) & 1;  // (loading used buffer 0)
    // Phase A: every linked entry's amplitude to the owner of its partner.
    res_scan(v, f, n_scan, &s_qn);
    if (tid == 0) s_drop = 0u;
    __syncthreads();
    const unsigned int qn = s_qn;
    for (unsigned int q = tid; q < qn; q += kT) {
      const unsigned int i = v.queue[q] & 0x7FFFu;
      const KT Y = v.keys[i] ^ m;
      net.template push<false>(buf, 0, owner_of(v, Y), Y, v.amps[i], 0ull);
    }
    net.arrive(pack_word(s_full != 0, s_low != 0, qn, min(s_tail, v.L) - s_dead), cnt);
    if (ent && k > job.k0) add_sum(&job.t.entropy[k - 1], dS_due);  // changes; summed up at the end
    dS_due = 0.0;
    const unsigned long long w = net.wait(cnt);
    if (word_abort(w)) {
      status = RES_ABORT;
      break;
    }
    const unsigned int live = word_live(w), linked = word_linked(w);
    if (RECORD && word_low(w)) {
      status = RES_TAPE;  // before this factor
      break;
    }
    const unsigned long long most = min((unsigned long long)(live + linked), job.bound);
    if (!(largest_share((float)most, (int)v.C) <= (float)v.L) || most >= (1ull << 20)) {
      status = RES_FULL;
      break;
    }
    peak = max(peak, live);
    if (tid == 0) s_qn = 0u;  // (every thread has its length)
    // Phase B: the messages' keys.  The first one is on its way while the count is.
    double dS = 0.0;
    Msg<KT> msg = net.template get<false>(buf, 0, min(tid, net.Lin - 1u));
    const unsigned int got = net.received(buf, 0);
    if (got > net.Lin) s_full = 1;
    for (unsigned int x = tid; x < min(got, net.Lin); x += kT) {
      if (x != tid) msg = net.template get<false>(buf, 0, x);
      const KT Z = msg.key;
      const bool zE = (Z & m) == f.occ;  // Z is the excited member
      const KT E = zE ? Z : Z ^ m;
      const double ss = neg_if(f.s, (KeyOps<KT>::popc(E & f.pmask) + f.pconst) & 1);  // s * sin(theta), exact
      const int at = res_find(v, Z);
      const double cZ = at >= 0 ? v.amps[at] : dead_value(0u);
      // c_E' = cos c_E - s sin c_D ;  c_D' = cos c_D + s sin c_E  (no contraction)
      const double pb = neg_if(__dmul_rn(ss, msg.a), zE ? 1 : 0);
      if (!is_dead(cZ)) {
        const double nZ = __dadd_rn(__dmul_rn(f.c, cZ), pb);
        atomicOr(&v.done[at >> 5], 1u << (at & 31));
        rot += zE;
        const bool out = below_eps(nZ, job.eps);
        if (ent) dS += new_term(at, nZ, out);
        if (out) {
          if (RECORD) record(Z, nZ, v.born[at]);
          v.amps[at] = dead_value(stamp);
          atomicAdd(&s_dead, 1u);
          ++dold;
        } else {
          v.amps[at] = nZ;
        }
      } else {
        // the partner that the factor creates: its own amplitude was +0.0
        const double nZ = nonzero(pb) ? pb : __dadd_rn(__dmul_rn(f.c, 0.0), pb);
        if (below_eps(nZ, job.eps)) {
          ++dnew;
          continue;
        }
        double eZ = 0.0;
        if (ent) dS += eZ = entropy_term(nZ);
        ++cre;
        if (at >= 0) {  // a dropped entry comes back
          if (ent) v.ent[at] = eZ;
          v.amps[at] = nZ;
          v.born[at] = (unsigned int)k;
          atomicSub(&s_dead, 1u);
        } else if (!res_append(v, Z, nZ, (unsigned int)k, &s_tail, eZ)) {
          s_full = 1;
        }
      }
    }
    __syncthreads();
    // Linked entries that no message named are alone.
    for (unsigned int q = tid; q < qn; q += kT) {
      const unsigned int e = v.queue[q], i = e & 0x7FFFu;
      if ((v.done[i >> 5] >> (i & 31u)) & 1u) continue;
      const bool ex = (e & 0x8000u) != 0u;
      const double cX = v.amps[i];
      double nX = __dmul_rn(f.c, cX);
      if (!nonzero(nX)) {  // the sign of a zero, as the full formula gives it
        const KT X = v.keys[i];
        const double ss = neg_if(f.s, (KeyOps<KT>::popc((ex ? X : X ^ m) & f.pmask) + f.pconst) & 1);
        nX = __dadd_rn(nX, neg_if(__dmul_rn(ss, 0.0), ex ? 1 : 0));
      }
      ++rot;
      const bool out = below_eps(nX, job.eps);
      if (ent) dS += new_term((int)i, nX, out);
      if (out) {
        if (RECORD) record(v.keys[i], nX, v.born[i]);
        v.amps[i] = dead_value(stamp);
        atomicAdd(&s_dead, 1u);
        ++dold;
      } else {
        v.amps[i] = nX;
      }
    }
    dS_due = dS;
    if (tid < (unsigned int)kFW) s_f[(k + 2) & 3][tid] = fw;
    fw = factor_word(k + 3);
    __syncthreads();
    if (tid == 0) {
      net.clear(buf);
      scanned += n_scan;
      if (RECORD && s_drop) atomicAdd(&job.tape.off[k + 1], (unsigned long long)s_drop);  // summed up at the end
    }
    unsigned int linked_to = n_scan;  // entries [linked_to, n_scan) are not hashed yet
    n_scan = min(s_tail, v.L);
    // More than N_MAX live entries are possible only if this many were linked.
    if (job.n_max > 0ull && most > job.n_max) {
      const bool counted = win.known;
      if (counted) window_count(v, net, n_scan, win, cs, s_win);
      const unsigned long long w2 = net_sync(net, pack_word(s_full != 0, false, 0u, n_scan - s_dead), cnt);
      if (word_abort(w2)) {
        status = RES_ABORT;
        break;
      }
      const unsigned int now = word_live(w2);
      if (counted) window_pick(net, win, (unsigned int)job.n_cut, (unsigned long long)now > job.n_max, cs, s_win);
      if ((unsigned long long)now > job.n_max) {
        unsigned long long T;
        KT Kt;
        if (!res_threshold(v, net, n_scan, now, job.n_cut, cs, win, s_win, cnt, &T, &Kt)) {
          status = RES_ABORT;
          break;
        }
        win.known = T >= (1ull << 53);
        win.lo = win.known ? T - (1ull << 52) : 0ull;  // an octave below, to one above
        auto keep = [&](double a, KT key) {
          const unsigned long long u = mag_of(a);
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
          if (tid == 0) {
            s_tbase = atomicAdd(&cnt->tape_n, (unsigned long long)s_drop);
            if (s_tbase + s_drop + slack >= job.tape.cap) s_low = 1;
            if (s_drop) atomicAdd(&job.tape.off[k + 1], (unsigned long long)s_drop);
          }
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
        dS_due += dC;
        if (tid == 0) {
          s_tail = kept;
          s_dead = 0u;
        }
        n_scan = linked_to = kept;
        res_rehash(v, kept, cnt);
        cut_total += (unsigned long long)now - job.n_cut;
        ++rebuilds;
      }
    }
    const unsigned int dead = s_dead;  // (block-uniform: written only in phase B)
    if (res_crowded<Net>(n_scan, dead, v.L)) {
      const unsigned int kept = res_squeeze(v, n_scan);
      if (tid == 0) {
        s_tail = kept;
        s_dead = 0u;
      }
      n_scan = linked_to = kept;
      res_rehash(v, kept, cnt);
      ++rebuilds;
    }
    for (unsigned int i = linked_to + tid; i < n_scan; i += kT) res_insert(v, v.keys[i], i, cnt);
    ++k;
  }
  // What happened in the last step is flagged here (nothing else is in flight).
  if (status != RES_ABORT && word_abort(net_sync(net, pack_word(s_full != 0, false, 0u, 0u), cnt))) status = RES_ABORT;
  bool store = status != RES_ABORT && k > job.k0;
  if (store) {
    if (ent && k > job.k0) add_sum(&job.t.entropy[k - 1], dS_due);
    const unsigned int kept = res_squeeze(v, n_scan);
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
    // every CTA's entries and counts are there, or a CTA gave up and never will be
    if (word_abort(net_sync(net, pack_word(false, false, 0u, 0u), cnt)) && Net::kGrid) {
      store = false;
      status = RES_ABORT;
    } else if (net.rank == 0u)
      res_finish(cnt, RECORD ? job.tape.off : nullptr, job.t.entropy, job.k0, k, res_smem);
  }
  if (net.rank == 0u && tid == 0) {
    cnt->res_status = status;
    cnt->res_k = store ? k : job.k0;
    cnt->res_cut = store ? cut_total : 0ull;
    cnt->res_rebuilds = store ? rebuilds : 0u;
    cnt->res_peak = peak;
  }
  net.leave();
}

// ---------------------------------------------------------------------------
// Reverse: factors k1 - 1 .. k0 of a table that holds psi_{k1} and mu_{k1}.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned int s = (unsigned int)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}

template <class KT, class Net>
__global__ void __launch_bounds__(kT, 1) k_res_reverse(ResJob<KT> one, const ResJob<KT>* __restrict__ many,
                                                       ResGeom g, ResNet<KT> rnet) {
  extern __shared__ __align__(16) unsigned char res_smem[];
  constexpr int kFW = sizeof(FactorT<KT>) / 8;
  __shared__ __align__(16) unsigned long long s_f[4][kFW];
  __shared__ unsigned int s_tail, s_dead, s_qn;
  __shared__ int s_full;
  __shared__ unsigned long long s_off[kOffRing + 1];
  __shared__ NetShared s_net;
  if (Net::kGrid && blockIdx.x != 0u && blockIdx.x + 1u == rnet.skip_block) return;
  const ResLayout lo = res_layout<KT>(g, true);
  const ResJob<KT> job = many ? many[blockIdx.x / (unsigned int)g.ctas] : one;
  const ResView<KT> v = res_view<KT>(res_smem, lo, g, true);
  // one record per thread on its way in
  TapeRecT<KT>* const stage = reinterpret_cast<TapeRecT<KT>*>(res_smem + lo.stage) + threadIdx.x;
  Counters* const cnt = job.t.cnt;
  const unsigned int tid = threadIdx.x, lane = tid & 31u;
  double acc = 0.0;  // this thread's share of the last factor's gradient entry / 2

  if (tid == 0) {
    s_tail = s_dead = s_qn = 0u;
    s_full = 0;
    s_net.count[0][0] = s_net.count[0][1] = s_net.count[1][0] = s_net.count[1][1] = 0u;
  }
  auto factor_word = [&](int k) -> unsigned long long {
    return tid < (unsigned int)kFW && k >= job.k0 ? reinterpret_cast<const unsigned long long*>(job.factors + k)[tid]
                                                  : 0ull;
  };
  // (the first addition to a gradient entry comes barriers later)
  if ((g.grid ? blockIdx.x : blockIdx.x % (unsigned int)g.ctas) == 0u)
    for (int x = job.k0 + (int)tid; x < job.k1; x += kT) job.grad[x] = 0.0;
  if (tid < (unsigned int)kFW) {
    s_f[(job.k1 - 1) & 3][tid] = factor_word(job.k1 - 1);
    s_f[(job.k1 - 2) & 3][tid] = factor_word(job.k1 - 2);
  }
  unsigned long long fw = factor_word(job.k1 - 3);
  Net net = make_net(static_cast<Net*>(nullptr), res_smem, lo, g, rnet, &s_net);
  __syncthreads();
  net.leave();  // (a cluster's CTAs are all set up before the first message)
  const bool loaded = res_load(v, net, job.t, &s_tail);
  if (tid == 0 && !loaded) s_full = 1;
  unsigned int n_scan = min(s_tail, v.L);
  unsigned int pairs = 0, compactions = 0;
  unsigned long long scanned = 0;
  int status = RES_DONE;
  int off_lo = job.k1 + 1;  // s_off covers [off_lo, off_lo + kOffRing]
  auto off_at = [&](int x) { return s_off[x - off_lo]; };
  const unsigned int gid = net.rank * kT + tid, gstep = net.C * kT;
  bool have = false;  // a record of the factor to be re-inserted next is in this thread's stage
  auto fetch = [&](int kk) {
    const unsigned long long x = off_at(kk) + gid;
    have = x < off_at(kk + 1);
    if (have) {
      const unsigned char* src = reinterpret_cast<const unsigned char*>(&tape_at(job.tape, x));
#pragma unroll
      for (unsigned int b = 0; b < sizeof(TapeRecT<KT>); b += 8u) cp_async8(reinterpret_cast<unsigned char*>(stage) + b, src + b);
    }
  };
  // Iteration k sweeps factor k (none in the first one, where k == k1) and
  // re-inserts the records of factor k - 1 after it.
  for (int k = job.k1;; --k) {
    const bool sweep = k < job.k1, push = k - 1 >= job.k0;
    const int buf = (job.k1 - k + 1) & 1;  // (loading used buffer 0)
    if (push && k - 2 < off_lo && off_lo > job.k0) {  // block-uniform: tape offsets down to k - kOffRing
      __syncthreads();
      off_lo = max(job.k0, k - kOffRing);
      for (int x = (int)tid; x <= k - off_lo; x += kT) s_off[x] = min(job.tape.off[off_lo + x], job.tape.cap);
      __syncthreads();
      if (!sweep) fetch(k - 1);
    }
    // Phase A
    if (push) {
      auto send = [&](const TapeRecT<KT>& rec) {
        net.template push<true>(buf, 1, owner_of(v, rec.key), rec.key, rec.val, (unsigned long long)rec.born);
      };
      if (have) {
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        send(*stage);
      }
      const unsigned long long r1 = off_at(k);
      for (unsigned long long x = off_at(k - 1) + gid + gstep; x < r1; x += gstep) send(tape_at(job.tape, x));
      have = false;
      if (k - 2 >= job.k0) fetch(k - 2);  // travels while this iteration sweeps
    }
    const FactorT<KT> f = *reinterpret_cast<const FactorT<KT>*>(s_f[k & 3]);  // (k == k1: not used)
    const KT m = f.occ | f.vir;
    unsigned int qn = 0u;
    if (sweep) {
      res_scan(v, f, n_scan, &s_qn);
      __syncthreads();
      qn = s_qn;
      for (unsigned int q = tid; q < qn; q += kT) {
        const unsigned int i = v.queue[q] & 0x7FFFu;
        const KT Y = v.keys[i] ^ m;
        net.template push<true>(buf, 0, owner_of(v, Y), Y, v.amps[i],
                                (unsigned long long)__double_as_longlong(v.lam[i]));
      }
    }
    net.arrive(pack_word(s_full != 0, false, 0u, 0u), cnt);
    if (k + 1 < job.k1) add_sum(&job.grad[k + 1], 2.0 * acc);
    if (word_abort(net.wait(cnt))) {
      status = RES_ABORT;
      break;
    }
    // Phase B: the first message of either kind is on its way while the counts are.
    if (tid == 0) s_qn = 0u;  // (every thread has its length)
    Msg<KT> msg = net.template get<true>(buf, 0, min(tid, net.Lin - 1u));
    Msg<KT> rec = net.template get<true>(buf, 1, min(tid, net.Lin - 1u));
    unsigned int got = net.received(buf, 0), recs = net.received(buf, 1);
    if (got + recs > net.Lin) {
      // The two kinds have overwritten each other: none is read (what a place holds
      // may be of either kind), and the next barrier ends the launch.
      s_full = 1;
      got = recs = 0u;
    }
    acc = 0.0;
    if (sweep) {
      const unsigned int stamp = 0x80000000u | (unsigned int)k;
      for (unsigned int x = tid; x < got; x += kT) {
        if (x != tid) msg = net.template get<true>(buf, 0, x);
        const KT Z = msg.key;
        const int at = res_find(v, Z);
        if (at < 0) continue;
        const double cZ = v.amps[at];
        if (is_dead(cZ)) continue;
        const bool zE = (Z & m) == f.occ;
        const int parity = (KeyOps<KT>::popc((zE ? Z : Z ^ m) & f.pmask) + f.pconst) & 1;
        const double ss = neg_if(f.s, parity);
        const double muZ = v.lam[at], muX = __longlong_as_double((long long)msg.b);
        atomicOr(&v.done[at >> 5], 1u << (at & 31));
        // (e, d) = U^T (e', d') and the same for the adjoint; each side its member.
        // s (lam_D psi_E - lam_E psi_D) is the same before and after the
        // rotation (a cross product), so E's side adds it from the old values.
        if (zE) {
          acc = fma(neg_if(muX, parity), cZ, acc);
          acc = fma(neg_if(muZ, parity ^ 1), msg.a, acc);
          ++pairs;
        }
        if (v.born[at] == (unsigned int)k) {
          v.amps[at] = dead_value(stamp);
          atomicAdd(&s_dead, 1u);
        } else {
          const double sx = neg_if(ss, zE ? 0 : 1);
          v.amps[at] = fma(f.c, cZ, sx * msg.a);
          v.lam[at] = fma(f.c, muZ, sx * muX);
        }
      }
      __syncthreads();
      // Linked entries that no message named are alone.
      for (unsigned int q = tid; q < qn; q += kT) {
        const unsigned int e = v.queue[q], i = e & 0x7FFFu;
        if ((v.done[i >> 5] >> (i & 31u)) & 1u) continue;
        const KT X = v.keys[i];
        const int parity = (KeyOps<KT>::popc(((e & 0x8000u) ? X : X ^ m) & f.pmask) + f.pconst) & 1;
        double x0, l0;
        unrotate_lone(f, neg_if(f.s, parity), parity, v.amps[i], v.lam[i], x0, l0, acc);
        v.amps[i] = x0;
        v.lam[i] = l0;
        ++pairs;
      }
    }
    // The records of factor k - 1: a key that is still stored was dropped.
    for (unsigned int x = tid; x < recs; x += kT) {
      if (x != tid) rec = net.template get<true>(buf, 1, x);
      const int at = res_find(v, rec.key);
      if (at >= 0) {
        if (!is_dead(v.amps[at])) raise_consistency(cnt, SITE_BULK_ALIVE, KeyOps<KT>::lo(rec.key));
        v.amps[at] = rec.a;
        v.lam[at] = 0.0;
        v.born[at] = (unsigned int)rec.b;
        atomicSub(&s_dead, 1u);
      } else if (!res_append(v, rec.key, rec.a, (unsigned int)rec.b, &s_tail)) {
        s_full = 1;
      }
    }
    if (tid < (unsigned int)kFW && sweep) s_f[(k - 2) & 3][tid] = fw;
    if (sweep) fw = factor_word(k - 3);
    __syncthreads();
    if (tid == 0) {
      net.clear(buf);
      if (sweep) scanned += n_scan;
    }
    unsigned int linked_to = n_scan;  // entries [linked_to, n_scan) are not hashed yet
    n_scan = min(s_tail, v.L);
    const unsigned int dead = s_dead;
    if (res_crowded<Net>(n_scan, dead, v.L)) {
      const unsigned int kept = res_squeeze(v, n_scan);
      if (tid == 0) {
        s_tail = kept;
        s_dead = 0u;
      }
      n_scan = linked_to = kept;
      res_rehash(v, kept, cnt);
      ++compactions;
    }
    for (unsigned int i = linked_to + tid; i < n_scan; i += kT) res_insert(v, v.keys[i], i, cnt);
    if (!push) break;
  }
  if (status != RES_ABORT && word_abort(net_sync(net, pack_word(s_full != 0, false, 0u, 0u), cnt))) status = RES_ABORT;
  if (status != RES_ABORT) {
    add_sum(&job.grad[job.k0], 2.0 * acc);
    const unsigned int kept = res_squeeze(v, n_scan);
    res_store(v, job.t, kept);
    const unsigned long long sp = warp_sum_u64(pairs);
    if (lane == 0 && sp) atomicAdd(&cnt->rev_pairs, sp);
    if (tid == 0) atomicAdd(&cnt->rev_scanned, scanned);
    // (as in the forward pass)
    if (word_abort(net_sync(net, pack_word(false, false, 0u, 0u), cnt)) && Net::kGrid)
      status = RES_ABORT;
    else if (net.rank == 0u)
      res_finish(cnt, nullptr, nullptr, job.k0, job.k0, res_smem);
  }
  if (net.rank == 0u && tid == 0) {
    cnt->res_status = status;
    cnt->res_k = status == RES_DONE ? job.k0 : job.k1;
    cnt->res_rebuilds = status == RES_DONE ? compactions : 0u;
  }
  net.leave();
}

// Entries a CTA holds at most: what fits its shared memory in either kernel
// (inside a cluster the inboxes lie there too).
constexpr int kMostCluster[3] = {0, 2048, 1792}, kMostGrid[3] = {0, 5632, 4352};

ResGeom shape(int ctas, bool grid, double L, bool entropy, int key_words) {
  ResGeom g{};
  g.ctas = ctas;
  g.grid = grid ? 1 : 0;
  const int most = grid ? kMostGrid[key_words] : kMostCluster[key_words];
  // (the sector of an uncut problem can be any size: clamped before it is an int)
  g.L = std::max(256, std::min(most, ((int)std::min(L, (double)most) + 31) / 32 * 32));
  g.Lin = g.L;
  g.entropy = entropy ? 1 : 0;
  g.logB = 4;  // buckets of four slots, at most three quarters full
  while (3 * (4 << g.logB) < 4 * g.L) ++g.logB;
  return g;
}

// The most dynamic shared memory that a launch of a kernel takes, over its shapes.
template <class KT>
unsigned int most_bytes(bool grid, bool reverse) {
  constexpr int kw = sizeof(KT) / 8;
  unsigned int most = 0;
  for (int ctas = 1; ctas <= (grid ? 1 : kMaxC); ctas *= 2)
    most = std::max(most, res_layout<KT>(shape(ctas, grid, grid ? kMostGrid[kw] : kMostCluster[kw], true, kw), reverse).bytes);
  return most;
}

// Launch configuration of a resident kernel; attr must outlive cfg.
template <class Kernel, class KT>
cudaError_t res_config(Kernel kernel, const KT&, int n_jobs, const ResGeom& g, bool reverse, cudaStream_t st,
                       cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  // The limit belongs to the function, not to the launch: it is the same for every
  // launch, whatever another host thread launches in between.
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)most_bytes<KT>(g.grid != 0, reverse));
  if (e != cudaSuccess) return e;
  if (!g.grid && g.ctas > 8) {  // a cluster of 16 is above the portable size
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cfg->gridDim = dim3((unsigned int)(n_jobs * g.ctas));
  cfg->blockDim = dim3(kT);
  cfg->dynamicSmemBytes = res_layout<KT>(g, reverse).bytes;
  cfg->stream = st;
  if (g.grid) {
    attr->id = cudaLaunchAttributeCooperative;
    attr->val.cooperative = 1;
  } else {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned int)g.ctas;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
  }
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  return cudaSuccess;
}

template <class Kernel, class KT>
cudaError_t res_launch(Kernel kernel, const ResJob<KT>& one, const ResJob<KT>* many, int n_jobs, const ResGeom& g,
                       const ResNet<KT>& net, bool reverse, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cudaError_t e = res_config(kernel, KT{}, n_jobs, g, reverse, st, &cfg, attr);
  if (e != cudaSuccess) return e;
  if (g.grid) {
    e = cudaMemsetAsync(net.ctl, 0, sizeof(ResControl), st);
    if (e != cudaSuccess) return e;
  }
  return cudaLaunchKernelEx(&cfg, kernel, one, many, g, net);
}

template <class KT>
ResLimits find_limits() {
  constexpr int kw = sizeof(KT) / 8;
  ResLimits r{};
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  for (int ctas = kMaxC; ctas >= 1 && r.cluster == 0; ctas /= 2) {
    const ResGeom g = shape(ctas, false, kMostCluster[kw], true, kw);
    int n[2] = {0, 0};
    if (res_config(k_res_forward<KT, true, ClusterNet<KT>>, KT{}, 1, g, false, nullptr, &cfg, attr) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n[0], k_res_forward<KT, true, ClusterNet<KT>>, &cfg) == cudaSuccess &&
        res_config(k_res_reverse<KT, ClusterNet<KT>>, KT{}, 1, g, true, nullptr, &cfg, attr) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n[1], k_res_reverse<KT, ClusterNet<KT>>, &cfg) == cudaSuccess && n[0] > 0 &&
        n[1] > 0)
      r.cluster = ctas;
    cudaGetLastError();
  }
  int dev = 0, sms = 0, coop = 0, a = 0, b = 0;
  const ResGeom g = shape(1, true, kMostGrid[kw], true, kw);
  if (cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
      res_config(k_res_forward<KT, true, GridNet<KT>>, KT{}, 1, g, false, nullptr, &cfg, attr) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_res_forward<KT, true, GridNet<KT>>, kT,
                                                    res_layout<KT>(g, false).bytes) == cudaSuccess &&
      res_config(k_res_reverse<KT, GridNet<KT>>, KT{}, 1, g, true, nullptr, &cfg, attr) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_res_reverse<KT, GridNet<KT>>, kT,
                                                    res_layout<KT>(g, true).bytes) == cudaSuccess &&
      a > 0 && b > 0)
    r.grid = std::min(sms, kMaxG);
  cudaGetLastError();
  return r;
}

}  // namespace

ResLimits res_limits(int key_words) {
  // kept per device: SM counts and cluster sizes may differ between them
  constexpr int kDevices = 64;
  static std::mutex mutex;
  static ResLimits found[2][kDevices];
  static bool have[2][kDevices];
  const int w = key_words == 2 ? 1 : 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return ResLimits{};
  std::lock_guard<std::mutex> lock(mutex);
  if (!have[w][dev]) {
    found[w][dev] = w ? find_limits<Key128>() : find_limits<unsigned long long>();
    have[w][dev] = true;
  }
  return found[w][dev];
}

bool res_room(unsigned long long entries, const ResGeom& g) {
  return entries < (1ull << 20) && largest_share((float)entries, g.ctas) <= (float)g.L;
}

bool res_cluster_shape(unsigned long long most, int key_words, int max_ctas, bool entropy, ResGeom* g) {
  if (max_ctas < 1) return false;
  // A recorded entropy takes a logarithm per rotation, some eighty FP64
  // instructions of 16 cycles a warp: its SMs are worth more than its barriers cost
  // (a factor at 100, 1,225 and 3,136 determinants: 5.5, 4.9 and 4.9 us with the
  // clusters of the other runs, 4.8, 4.7 and 4.7 with sixteen; the whole GPU: 6.0,
  // 5.7, 5.8).  Without entropies the other size matters too, a batch's jobs in
  // flight: 24 gradients over 3,136 determinants take 4.9, 7.0 and 10.6 ms with 4, 8
  // and 16 CTAs each, while one by itself gains little from more (us per factor,
  // forward and reverse: 225 determinants 3.0 and 3.4 with 1, 3.1 and 3.2 with 4, 3.0
  // and 2.9 with 8; 441: 3.1 and 3.6, 3.1 and 3.5, 3.0 and 3.2; 1,568: 3.4 and 4.4, 3.3
  // and 3.8, 3.1 and 3.5; 4,900: 3.7 and 4.6 with 4, 3.3 and 4.0 with 8, 3.3 and 3.9
  // with 16; 7,056: 3.3 and 4.0 with 8, 3.4 and 4.0 with 16; 10,584: 3.6 and 4.2, 3.3
  // and 3.8).
  int ctas = entropy ? kMaxC : most <= 512 ? 1 : most <= 2048 ? 4 : most <= 6144 ? 8 : 16;
  ctas = std::min(ctas, max_ctas);
  for (; ctas <= max_ctas; ctas *= 2) {
    // a quarter more than the largest share, for dropped entries and inboxes
    const double want = 1.25 * (double)largest_share((float)most, ctas) + 32.0;
    if (want <= (double)kMostCluster[key_words]) {
      *g = shape(ctas, false, want, entropy, key_words);
      return true;
    }
  }
  return false;
}

bool res_grid_shape(unsigned long long most, int key_words, int ctas, bool entropy, ResGeom* g) {
  if (ctas < 1) return false;
  *g = shape(ctas, true, 1.25 * (double)largest_share((float)most, ctas) + 32.0, entropy, key_words);
  return true;
}

template <class KT>
cudaError_t launch_res_forward(const ResJob<KT>& one, const ResJob<KT>* many, int n_jobs, const ResGeom& g,
                               const ResNet<KT>& net, int record, cudaStream_t st) {
  cudaError_t e;
  if (g.grid)
    e = record ? res_launch(k_res_forward<KT, true, GridNet<KT>>, one, many, n_jobs, g, net, false, st)
               : res_launch(k_res_forward<KT, false, GridNet<KT>>, one, many, n_jobs, g, net, false, st);
  else
    e = record ? res_launch(k_res_forward<KT, true, ClusterNet<KT>>, one, many, n_jobs, g, net, false, st)
               : res_launch(k_res_forward<KT, false, ClusterNet<KT>>, one, many, n_jobs, g, net, false, st);
  return e;
}

template <class KT>
cudaError_t launch_res_reverse(const ResJob<KT>& one, const ResJob<KT>* many, int n_jobs, const ResGeom& g,
                               const ResNet<KT>& net, cudaStream_t st) {
  return g.grid ? res_launch(k_res_reverse<KT, GridNet<KT>>, one, many, n_jobs, g, net, true, st)
                : res_launch(k_res_reverse<KT, ClusterNet<KT>>, one, many, n_jobs, g, net, true, st);
}

#define UCC_RES_INSTANTIATE(KT)                                                                                 \
  template cudaError_t launch_res_forward<KT>(const ResJob<KT>&, const ResJob<KT>*, int, const ResGeom&,        \
                                              const ResNet<KT>&, int, cudaStream_t);                            \
  template cudaError_t launch_res_reverse<KT>(const ResJob<KT>&, const ResJob<KT>*, int, const ResGeom&,        \
                                              const ResNet<KT>&, cudaStream_t);
UCC_RES_INSTANTIATE(unsigned long long)
UCC_RES_INSTANTIATE(Key128)

}  // namespace ucc
