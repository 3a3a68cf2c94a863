// One global switch round (Def. 2 of arXiv 2111.03005) of every chain of a
// pool, on one GB300, laid out as streaming passes so that no step needs a
// random DRAM access per switch.
//
//   k_clear          zero the per-round counters
//   k_permute        read the list in last-round slot order (applying the
//                    last round's legal switches on the fly), compute each
//                    position's Philox key and append (key bits, position,
//                    edge) to its bucket; the buckets' write frontiers stay
//                    in L2, so DRAM sees whole lines
//   k_scan_perm      bucket slot offsets
//   k_sortpair       per bucket: exact sort by (key, position) in shared
//                    memory; write the list back in this round's slot order;
//                    for each pair of slots (edge switch sigma_k, Def. 1)
//                    apply tau, the loop and shared-node rules and laziness,
//                    and append Algorithm 1's four tuples (e1, k, ERASE),
//                    (e2, k, ERASE), (e3, k, INSERT), (e4, k, INSERT) to
//                    the hash partitions of their edge ids
//   k_boundary       the same for pairs whose slots lie in two buckets
//   k_sources        the sources (ERASE tuples) of all switches, from the
//                    list in slot order, but only those whose edge id some
//                    target of the round may equal (target filter)
//   k_overflow_*     group the (rare) tuples that found their partition full
//   k_group          per partition: group by edge id in a shared-memory
//                    table and decide every target of wave 1 (Algorithm 1's
//                    first round): certainly present, free, or dependent on
//                    an undecided switch; edge ids with a dependency get an
//                    entry {p, q} for the later waves
//   k_wave1          per switch: legal, illegal or pending
//   k_wave_register  waves that more than kSoloPending pending switches enter,
//   k_wave_decide    on the whole GPU, one pair of kernels per wave
//   k_tail           all other waves, on one CTA
//
// The waves are Jacobi steps: a switch decided in wave w only uses decisions
// of waves < w (status words carry their wave), so the result and the wave
// count do not depend on thread timing.  The list after the round is the one
// the sequential loop of Def. 2 produces.
#include <algorithm>

#include "device_util.cuh"
#include "es_set.cuh"
#include "gesmc_internal.cuh"

namespace gesmc {
namespace {

// Permutation key K(i) of round `round` (purpose 0).
__device__ __forceinline__ unsigned long long perm_key(unsigned long long seed, unsigned long long round,
                                                       uint32_t i) {
  return word_of(philox(i >> 2, round, 0, 0, seed, 0), i & 3);
}

__device__ __forceinline__ uint32_t bucket_of(unsigned long long key, uint32_t B) {
  return B ? (uint32_t)(key >> (64 - B)) : 0u;
}

// The 32 key bits after the bucket bits.
__device__ __forceinline__ uint32_t mid_of(unsigned long long key, uint32_t B) {
  return (uint32_t)((key << B) >> 32);
}

// ---------------------------------------------------------------- edges
__device__ __forceinline__ uint32_t partition_of(unsigned long long h, uint32_t P) {
  return P ? (uint32_t)(h >> (64 - P)) : 0u;
}

// Edge switch (i, j, g = [i < j]) of a global switch (Def. 2): tau with the
// direction bit the permutation gives.
__device__ __forceinline__ uint32_t tau(uint32_t i, uint32_t j, unsigned long long e1, unsigned long long e2,
                                        unsigned long long &e3, unsigned long long &e4) {
  return tau_g(i < j ? 1u : 0u, e1, e2, e3, e4);
}


// ---------------------------------------------------------------- chains
// Round number of a chain in the current pool round, and whether status[]
// holds decisions of the chain's last round that still have to be applied.
__device__ __forceinline__ unsigned long long chain_round(const ChainDesc &ch, unsigned long long pool_round) {
  return ch.start_round + (pool_round - ch.join);
}
__device__ __forceinline__ bool chain_apply(const ChainDesc &ch, unsigned long long pool_round) {
  return pool_round > ch.added;
}

// Laziness word of switch k (the chain's own index): Philox, purpose 1.
__device__ __forceinline__ unsigned long long lazy_word(const ChainDesc &ch, unsigned long long round, uint32_t k) {
  return word_of(philox(k >> 2, round, 1, 0, ch.seed, 0), k & 3);
}

// Laziness (Def. 2, P_L).  Per-switch form: switch k is skipped iff its word
// is below the chain's threshold.  Exact l: the round runs its first ell
// switches only, ell = the number of words that pass (counted beforehand).
__device__ __forceinline__ bool is_lazy(const ChainDesc &ch, unsigned long long round, uint32_t k, uint32_t ell) {
  if (ch.lazy_threshold == 0) return false;
  if (ch.exact_ell) return k >= ell;
  return lazy_word(ch, round, k) < ch.lazy_threshold;
}

// The values of slots 2k, 2k+1 of a chain at the start of this round: the
// chain's last-round switch k rewired them if it was legal.
__device__ __forceinline__ void apply_last(const RoundArgs &a, const ChainDesc &ch, bool apply, uint32_t k,
                                           uint32_t i, uint32_t j, unsigned long long &e1, unsigned long long &e2) {
  if (apply && k < ch.L && (__ldcs(&a.status[ch.switch_base + k]) & 3u) == kLegal) {
    unsigned long long e3, e4;
    tau(i, j, e1, e2, e3, e4);
    e1 = e3;
    e2 = e4;
  }
}

// ---------------------------------------------------------------- build
// Append tuples to their hash partitions: partition ids and cursor atomics
// first (independent, in flight together), then the 16-byte stores.  A
// tuple in its partition is {id lo, id hi, value, low 32 bits of the id's
// hash} (the grouping kernel probes its table with those bits); one that
// finds its partition full goes to the overflow list with its partition id
// in place of the hash bits.
// The target filter's bit of an edge id with hash h.
__device__ __forceinline__ uint32_t filter_bit(const RoundArgs &a, unsigned long long h) {
  return (uint32_t)(h >> 24) & a.tfilter_mask;
}

template <int N>
__device__ __forceinline__ void emit_tuples(const RoundArgs &a, const ChainDesc &ch,
                                            const unsigned long long (&key)[N], const unsigned long long (&hash)[N],
                                            const uint32_t (&val)[N]) {
  uint32_t part[N], hlo[N], idx[N];
#pragma unroll
  for (int t = 0; t < N; ++t) {
    const unsigned long long h = hash[t];
    part[t] = partition_of(h, ch.P);
    hlo[t] = (uint32_t)h;
    idx[t] = key[t] != kEmptyKey ? atomicAdd(&a.tcount[ch.tcount_base + part[t] * ch.tstride], 1u) : 0u;
  }
#pragma unroll
  for (int t = 0; t < N; ++t) {
    if (key[t] == kEmptyKey) continue;
    if (idx[t] < ch.capt) {
      a.ptup[ch.tuple_base + (size_t)part[t] * ch.capt + idx[t]] =
          make_uint4((uint32_t)key[t], (uint32_t)(key[t] >> 32), val[t], hlo[t]);
    } else {
      const uint32_t o = atomicAdd(&a.ctl->ovf_count, 1u);
      if (o < a.ovf_cap)
        a.otup[o] = make_uint4((uint32_t)key[t], (uint32_t)(key[t] >> 32), val[t], ch.part_base + part[t]);
      else
        atomicOr(&a.ctl->err, kErrRecord);
    }
  }
}

// Switches k[t] (the chain's own indices; t < N, those with valid[t]) =
// (i, j, g) with sources e1, e2: record each reject code, mark the targets
// in the target filter and emit Algorithm 1's tuples (e3, k, INSERT),
// (e4, k, INSERT), with k made pool-wide; all N switches' atomics are in
// flight together.  Their ERASE tuples (e1, k), (e2, k) follow from
// k_sources when the filter says a target may need them.  A switch rejected
// outright has no targets.
template <int N>
__device__ __forceinline__ void build_switches(const RoundArgs &a, const ChainDesc &ch, unsigned long long round,
                                               uint32_t ell, const bool (&valid)[N], const uint32_t (&k)[N],
                                               const uint32_t (&i)[N], const unsigned long long (&e1)[N],
                                               const uint32_t (&j)[N], const unsigned long long (&e2)[N]) {
  unsigned long long key[2 * N], hash[2 * N];
  uint32_t val[2 * N];
#pragma unroll
  for (int t = 0; t < N; ++t) {
    unsigned long long e3 = kEmptyKey, e4 = kEmptyKey;
    const uint32_t kg = ch.switch_base + k[t];
    if (valid[t]) {
      const uint32_t code = is_lazy(ch, round, k[t], ell) ? kCodeLazy : tau(i[t], j[t], e1[t], e2[t], e3, e4);
      a.word[kg] = code;
      if (code) e3 = e4 = kEmptyKey;
    }
    key[2 * t] = e3;
    key[2 * t + 1] = e4;
    val[2 * t] = kg;
    val[2 * t + 1] = kg | kTupleWhich;
  }
#pragma unroll
  for (int t = 0; t < 2 * N; ++t) {
    hash[t] = mix64(key[t]);
    if (key[t] != kEmptyKey) {
      const uint32_t fb = filter_bit(a, hash[t]);
      atomicOr(&a.tfilter[fb >> 5], 1u << (fb & 31));
    }
  }
  emit_tuples<2 * N>(a, ch, key, hash, val);
}

// ---------------------------------------------------------------- decide
constexpr int kOk = 0, kWait = 1, kBad = 2;

__device__ __forceinline__ bool decided_before(uint32_t st, uint32_t wave) {
  const uint32_t w = st >> 2;
  return w != 0 && w < wave;
}

// Algorithm 1's test of one target edge of switch k in wave `wave` >= 2,
// from its dependency entry (p, q): kBad if the edge exists when k runs,
// kOk if it certainly does not, kWait if that depends on an undecided switch.
// The test, given the entry and the statuses of the eraser p and of the
// smallest inserter q (looked at only where they come before k).
__device__ __forceinline__ int judge_target(uint32_t k, uint32_t p, uint32_t q, uint32_t sp, uint32_t sq,
                                            uint32_t wave) {
  int res = kOk;
  if (p != kPNone) {             // the edge is in E at the start of the round
    if (p >= k) return kBad;     // erased later than k, or never
    if (decided_before(sp, wave)) {
      if ((sp & 3u) == kIllegal) return kBad;  // its eraser failed: still there
    } else {
      res = kWait;
    }
  }
  if (q != k) {
    // an earlier switch may insert it first
    if (q < k && decided_before(sq, wave) && (sq & 3u) == kLegal) return kBad;
    res = kWait;                 // q undecided, illegal but not yet replaced, or being replaced
  }
  return res;
}

__device__ __forceinline__ int check_target(const RoundArgs &a, uint32_t k, uint32_t d, uint32_t wave) {
  if (d == kTrivial) return kOk;
  const uint2 pq = __ldcg(&a.dep[d]);
  return judge_target(k, pq.x, pq.y, pq.x < k ? __ldcg(&a.status[pq.x]) : 0u,
                      pq.y < k ? __ldcg(&a.status[pq.y]) : 0u, wave);
}

// The dependency entries of switch k's targets, given its word (sw holds an
// entry only where the word says so: most switches have none, and their sw is
// not written at all).
__device__ __forceinline__ uint2 entries_of(uint32_t word, uint2 s) {
  if (!(word & kFlagEntry3)) s.x = kTrivial;
  if (!(word & kFlagEntry4)) s.y = kTrivial;
  return s;
}
__device__ __forceinline__ uint2 switch_entries(const RoundArgs &a, uint32_t k) {
  return entries_of(__ldcg(&a.word[k]), __ldcg(&a.sw[k]));
}

struct Tally {
  uint32_t accepted = 0, rej_loop = 0, rej_exists = 0, lazy = 0;
};

// An illegal switch no longer counts as an inserter: where it was the
// smallest one, clear the field; the waiting inserters re-register.
__device__ __forceinline__ void drop_inserter(const RoundArgs &a, uint32_t k, uint2 s) {
  if (s.x != kTrivial && __ldcg(&a.dep[s.x].y) == k) atomicCAS(&a.dep[s.x].y, k, kQNone);
  if (s.y != kTrivial && __ldcg(&a.dep[s.y].y) == k) atomicCAS(&a.dep[s.y].y, k, kQNone);
}

__device__ __forceinline__ void flush_tally(const RoundArgs &a, Tally t) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    t.accepted += __shfl_down_sync(0xffffffffu, t.accepted, off);
    t.rej_loop += __shfl_down_sync(0xffffffffu, t.rej_loop, off);
    t.rej_exists += __shfl_down_sync(0xffffffffu, t.rej_exists, off);
    t.lazy += __shfl_down_sync(0xffffffffu, t.lazy, off);
  }
  if ((threadIdx.x & 31) == 0) {
    if (t.accepted) atomicAdd(&a.st->accepted, (unsigned long long)t.accepted);
    if (t.rej_loop) atomicAdd(&a.st->rej_loop, (unsigned long long)t.rej_loop);
    if (t.rej_exists) atomicAdd(&a.st->rej_exists, (unsigned long long)t.rej_exists);
    if (t.lazy) atomicAdd(&a.st->lazy, (unsigned long long)t.lazy);
  }
}

// Per-chain count of accepted switches: each thread keeps a running count
// for the chain it last saw and hands it on when the chain changes; at the
// end, lanes of a warp holding the same chain add once (all lanes call).
struct ChainCount {
  uint32_t chain = kNoChain, n = 0;
};

__device__ __forceinline__ void count_accepted(const RoundArgs &a, ChainCount &cc, uint32_t chain) {
  if (chain != cc.chain) {
    if (cc.n) atomicAdd(&a.chain_accepted[cc.chain], (unsigned long long)cc.n);
    cc.chain = chain;
    cc.n = 0;
  }
  ++cc.n;
}

__device__ __forceinline__ void flush_count(const RoundArgs &a, const ChainCount &cc) {
  const unsigned same = __match_any_sync(0xffffffffu, cc.n ? cc.chain : kNoChain);
  unsigned long long n = cc.n;
  // sum n over the lanes of this group, result at its first lane
  const int lane = threadIdx.x & 31;
  unsigned long long total = 0;
  for (unsigned rest = same; rest; rest &= rest - 1) total += __shfl_sync(same, n, __ffs(rest) - 1);
  if (cc.n && (__ffs(same) - 1) == lane) atomicAdd(&a.chain_accepted[cc.chain], total);
}

// Warp-aggregated append of k to a list (all lanes of the warp must call).
__device__ __forceinline__ void append_if(bool take, uint32_t k, uint32_t *list, uint32_t *count) {
  const unsigned mask = __ballot_sync(0xffffffffu, take);
  if (!mask) return;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(mask) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(count, (uint32_t)__popc(mask));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (take) list[base + __popc(mask & ((1u << lane) - 1u))] = k;
}

// ---------------------------------------------------------------- kernels

__device__ __forceinline__ void clear_arrays(const RoundArgs &a) {
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  for (uint32_t b = tid; b < a.bucket_hw; b += nth) a.pcount[b] = 0;
  for (uint32_t p = tid; p < a.part_hw; p += nth) a.ocount[p] = 0;
  for (uint32_t p = tid; p < a.tcount_hw; p += nth) a.tcount[p] = 0;
  for (uint32_t c = tid; c < a.chain_hw; c += nth) a.chain_ell[c] = 0;
  if (a.any_work) {  // the target filter: at least 2^12 bits
    uint4 *const f = reinterpret_cast<uint4 *>(a.tfilter);
    for (uint32_t w = tid; w <= (a.tfilter_mask >> 7); w += nth) f[w] = make_uint4(0, 0, 0, 0);
  }
}

// One thread.
__device__ __forceinline__ void clear_counters(Counters *ctl) {
  ctl->pending[0] = 0;
  ctl->pending[1] = 0;
  ctl->boundary = 0;
  ctl->waves = 0;
  ctl->dep_count = 0;
  ctl->ovf_count = 0;
  ctl->cur = 0;
  ctl->wave_next = 2;
  ctl->wave_blocks = 0;
  ctl->wide = 0;
}

// The kernels of a round follow one another by programmatic dependent launch:
// each lets the next one start as soon as its own CTAs are all on the GPU
// (dep_launch) and reads and writes nothing that changes during a round before
// the one before it has ended (dep_wait).  A kernel waits for the one before
// it even where it does nothing else, so that "the one before has ended"
// means all of them.  Chain descriptors and owner maps do not change while
// rounds run.  A round of G(1000, 0.01) took 69 us replayed from a plain graph,
// 61 us so, and 53 us with the scatter on more SMs and the statistics closed by
// several warps (18 kernels: what is left is their own chains of L2 accesses).
__global__ void k_clear(RoundArgs a) {
  dep_launch();
  dep_wait();
  clear_arrays(a);
  if (blockIdx.x == 0 && threadIdx.x == 0) clear_counters(a.ctl);
}

__device__ __forceinline__ void store_record(const RoundArgs &a, uint32_t b, uint32_t idx, uint32_t keybits,
                                             uint32_t pos, unsigned long long e) {
  if (idx < (1u << a.bucket_log2))
    a.prec[((size_t)b << a.bucket_log2) + idx] = make_uint4(keybits, pos, (uint32_t)e, (uint32_t)(e >> 32));
  else
    atomicOr(&a.ctl->err, kErrBucket);
}

// The positions of the chain with few buckets (a pool of one chain with at
// most kAggBuckets buckets), each CTA taking `tile` (at most kThreads * kPairs)
// consecutive pairs of slots: the CTA counts its records per bucket in shared memory (a
// record's rank among the CTA's records of its bucket comes with it), takes
// each bucket's range with one cursor atomic, then stores its records, which
// stay in registers meanwhile.  With few buckets every cursor takes thousands
// of same-address atomics per round, which serialise in L2; here it takes one
// per CTA.  The order of records inside a bucket does not matter: the sort
// orders them by key and position.  Bound by the generator (a Philox block per
// position, about 400 instructions): with the keys computed again for the
// second pass it took 38 us for 9.5e5 positions and, on two CTAs of 2048 pairs, 19 us
// for 5,000; now 22 us (in full waves of equal CTAs), and 5.4 us on ten CTAs of
// 256 pairs.
template <int kThreads, int kPairs>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads) k_permute_agg(RoundArgs a, uint32_t tile) {
  __shared__ uint32_t sc[kAggBuckets];  // per bucket: the CTA's count, then its base
  dep_launch();
  const ChainDesc ch = a.chains[a.agg_chain];
  const uint32_t tid = threadIdx.x, nb = 1u << ch.B, npair = (ch.m + 1) >> 1;
  for (uint32_t b = tid; b < nb; b += kThreads) sc[b] = 0;
  dep_wait();
  const unsigned long long R = a.ctl->pool_round;
  const unsigned long long round = chain_round(ch, R);
  const bool apply = chain_apply(ch, R);
  const uint32_t x0 = blockIdx.x * tile + tid, x1 = min(blockIdx.x * tile + tile, npair);
  __syncthreads();
  uint32_t pos[2 * kPairs], mid[2 * kPairs], br[2 * kPairs];  // br: bucket, and the rank in the high half
  unsigned long long e[2 * kPairs];
#pragma unroll
  for (int j = 0; j < kPairs; ++j) {
    const uint32_t x = x0 + j * kThreads;
    br[2 * j] = br[2 * j + 1] = kNoChain;
    if (x >= x1) continue;
    const uint32_t gx = (ch.slot_base >> 1) + x;  // pair index in the pool's slots
    const bool two = 2 * x + 1 < ch.m;
    if (two) {
      const uint2 ij = __ldcs(reinterpret_cast<const uint2 *>(a.cpos) + gx);
      const ulonglong2 ee = __ldcs(reinterpret_cast<const ulonglong2 *>(a.cedge) + gx);
      e[2 * j] = ee.x;
      e[2 * j + 1] = ee.y;
      apply_last(a, ch, apply, x, ij.x, ij.y, e[2 * j], e[2 * j + 1]);
      pos[2 * j] = ij.x;
      pos[2 * j + 1] = ij.y;
    } else {  // odd m: the chain's last slot has no partner
      pos[2 * j] = a.cpos[2 * gx];
      e[2 * j] = a.cedge[2 * gx];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 1 && !two) continue;
      const unsigned long long K = perm_key(ch.seed, round, pos[2 * j + h]);
      const uint32_t b = bucket_of(K, ch.B);
      mid[2 * j + h] = mid_of(K, ch.B);
      br[2 * j + h] = b | (atomicAdd(&sc[b], 1u) << 16);
    }
  }
  __syncthreads();
  for (uint32_t b = tid; b < nb; b += kThreads) {
    const uint32_t n = sc[b];
    if (n) sc[b] = atomicAdd(&a.pcount[ch.bucket_base + b], n);
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 2 * kPairs; ++j)
    if (br[j] != kNoChain) {
      const uint32_t b = br[j] & 0xFFFFu;
      store_record(a, ch.bucket_base + b, sc[b] + (br[j] >> 16), mid[j], pos[j], e[j]);
    }
}

// Exact l (Def. 2 as printed): per chain in that mode, the number of its
// switches whose laziness word passes (>= threshold); the round then runs
// the chain's first l switches.  Each CTA takes a contiguous range of
// switches and each thread keeps a running count for its current chain.
__device__ __forceinline__ void lazy_count_body(const RoundArgs &a) {
  const unsigned long long R = a.ctl->pool_round;
  const uint32_t per = (a.switch_hw + gridDim.x - 1) / gridDim.x;
  const uint32_t chunk = (per + blockDim.x - 1) / blockDim.x * blockDim.x;
  const uint32_t beg = min(blockIdx.x * chunk, a.switch_hw), end = min(beg + chunk, a.switch_hw);
  uint32_t cur = kNoChain, n = 0;
  for (uint32_t k = beg + threadIdx.x; k < end; k += blockDim.x) {
    const uint32_t c = a.owner_switch[k];
    if (c == kNoChain) continue;
    const ChainDesc ch = a.chains[c];
    if (!ch.exact_ell || ch.lazy_threshold == 0) continue;
    if (c != cur) {
      if (n) atomicAdd(&a.chain_ell[cur], n);
      cur = c;
      n = 0;
    }
    n += lazy_word(ch, chain_round(ch, R), k - ch.switch_base) >= ch.lazy_threshold ? 1u : 0u;
  }
  if (n) atomicAdd(&a.chain_ell[cur], n);
}

__global__ void k_lazy_count(RoundArgs a) {
  dep_launch();
  dep_wait();
  lazy_count_body(a);
}

// Append every position, with its current edge, to its chain's bucket.
// Five CTAs of 256 per SM (48 registers, no spills): 3.16 ms per round on
// G(2^24) against 3.20 with six (40 registers and a few spilled) and 3.29
// with eight (32).  The round launches one pair per thread (short-lived
// CTAs): that measured 3.13 ms against 3.46 ms for a grid-stride loop over
// 8 CTAs per SM and 4.05 ms over one resident wave; the loop form serves the
// one-launch round.
__device__ __forceinline__ void permute_pair(const RoundArgs &a, uint32_t x, unsigned long long R) {
  const uint32_t s0 = 2 * x;
  const uint32_t c = a.owner_slot[s0];
  if (c == kNoChain) return;
  const ChainDesc ch = a.chains[c];
  const unsigned long long round = chain_round(ch, R);
  const uint32_t ls = s0 - ch.slot_base;
  if (ls + 1 < ch.m) {
    const uint2 ij = __ldcs(reinterpret_cast<const uint2 *>(a.cpos) + x);
    const ulonglong2 ee = __ldcs(reinterpret_cast<const ulonglong2 *>(a.cedge) + x);
    unsigned long long e1 = ee.x, e2 = ee.y;
    apply_last(a, ch, chain_apply(ch, R), ls >> 1, ij.x, ij.y, e1, e2);
    // both keys and both atomics before the two stores
    const unsigned long long K1 = perm_key(ch.seed, round, ij.x);
    const unsigned long long K2 = perm_key(ch.seed, round, ij.y);
    const uint32_t b1 = ch.bucket_base + bucket_of(K1, ch.B), b2 = ch.bucket_base + bucket_of(K2, ch.B);
    const uint32_t x1 = atomicAdd(&a.pcount[b1], 1u);
    const uint32_t x2 = atomicAdd(&a.pcount[b2], 1u);
    store_record(a, b1, x1, mid_of(K1, ch.B), ij.x, e1);
    store_record(a, b2, x2, mid_of(K2, ch.B), ij.y, e2);
  } else {  // odd m: the chain's last slot has no partner
    const uint32_t pos = a.cpos[s0];
    const unsigned long long K = perm_key(ch.seed, round, pos);
    const uint32_t b = ch.bucket_base + bucket_of(K, ch.B);
    store_record(a, b, atomicAdd(&a.pcount[b], 1u), mid_of(K, ch.B), pos, a.cedge[s0]);
  }
}

__device__ __forceinline__ void permute_body(const RoundArgs &a) {
  const unsigned long long R = a.ctl->pool_round;
  const uint32_t npair = (a.slot_hw + 1) >> 1;
  const uint32_t nth = gridDim.x * blockDim.x;
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < npair; x += nth) permute_pair(a, x, R);
}

// The CTA's place in a flat pass: CTA b takes range (b * stride) mod ctas.
__device__ __forceinline__ uint32_t scrambled_cta(uint32_t stride) {
  return (uint32_t)(((unsigned long long)blockIdx.x * stride) % gridDim.x);
}

// One pair of slots per thread, CTAs in scrambled order.
__global__ void __launch_bounds__(256, 5) k_permute(RoundArgs a) {
  dep_launch();
  const uint32_t x = scrambled_cta(a.permute_stride) * blockDim.x + threadIdx.x;
  dep_wait();
  if (x < (a.slot_hw + 1) >> 1) permute_pair(a, x, a.ctl->pool_round);
}

// Exclusive scan of n counters (n + 1 offsets) by one CTA of 1024 threads,
// in place if off == count; counts above `clamp` are clamped (their
// overflow was already reported).
__device__ __forceinline__ void cta_scan_1024(const uint32_t *count, uint32_t *off, uint32_t *copy, uint32_t n,
                                              uint32_t clamp) {
  __shared__ uint32_t part[1024];
  const uint32_t tid = threadIdx.x;
  const uint32_t per = (n + 1023) / 1024;
  const uint32_t beg = min(tid * per, n), end = min(beg + per, n);
  uint32_t sum = 0;
  for (uint32_t b = beg; b < end; ++b) sum += min(count[b], clamp);
  part[tid] = sum;
  __syncthreads();
  for (uint32_t d = 1; d < 1024; d <<= 1) {
    const uint32_t v = tid >= d ? part[tid - d] : 0;
    __syncthreads();
    part[tid] += v;
    __syncthreads();
  }
  uint32_t run = part[tid] - sum;
  for (uint32_t b = beg; b < end; ++b) {
    const uint32_t c = min(count[b], clamp);  // read before writing: count may be off itself
    off[b] = run;
    if (copy) copy[b] = run;
    run += c;
  }
  if (tid == 1023) off[n] = part[1023];
}

// Bucket slot offsets in two steps: each CTA scans a block of 1024 bucket
// counts (clamped to the capacity; an overflow was reported) and records the
// block's sum; one CTA then scans the block sums.  A bucket's offset is
// pblk[b / 1024] + poff[b].
__global__ void __launch_bounds__(1024) k_scan_perm(RoundArgs a) {
  __shared__ uint32_t warp_tot[32];
  dep_launch();
  dep_wait();
  const uint32_t b = blockIdx.x * 1024 + threadIdx.x;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t v = b < a.bucket_hw ? min(a.pcount[b], 1u << a.bucket_log2) : 0u;
  uint32_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= (uint32_t)d) incl += u;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t t = warp_tot[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= (uint32_t)d) t += u;
    }
    warp_tot[lane] = t;
  }
  __syncthreads();
  if (b < a.bucket_hw) a.poff[b] = incl - v + (warp ? warp_tot[warp - 1] : 0u);
  if (threadIdx.x == 1023) a.pblk[blockIdx.x] = warp_tot[31];
}

__global__ void __launch_bounds__(1024) k_scan_blocks(RoundArgs a) {
  dep_launch();
  dep_wait();
  const uint32_t nblk = (a.bucket_hw + 1023) / 1024;
  cta_scan_1024(a.pblk, a.pblk, nullptr, nblk, 0xFFFFFFFFu);
}

__device__ __forceinline__ uint32_t bucket_offset(const RoundArgs &a, uint32_t b) {
  return a.pblk[b >> 10] + a.poff[b];
}

// Overflow tuples (those that found their partition full), grouped by
// partition with exact counts.  Every kernel does nothing when there is no
// overflow, which is the normal case for a single chain.  The partition
// offsets are scanned like the bucket offsets: blocks of 1024 partitions on
// many CTAs (local offsets, and the cursors the scatter starts from), then
// the block sums on one CTA; partition p's list starts at
// oblk[p / 1024] + ooff[p].
__device__ __forceinline__ void overflow_count_body(const RoundArgs &a) {
  const uint32_t n = min(a.ctl->ovf_count, a.ovf_cap);
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
    atomicAdd(&a.ocount[a.otup[t].w], 1u);
}

__global__ void k_overflow_count(RoundArgs a) {
  dep_launch();
  dep_wait();
  overflow_count_body(a);
}

__global__ void __launch_bounds__(1024) k_overflow_scan_blocks(RoundArgs a) {
  dep_launch();
  dep_wait();
  if (a.ctl->ovf_count == 0) return;
  __shared__ uint32_t warp_tot[32];
  const uint32_t p = blockIdx.x * 1024 + threadIdx.x;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t v = p < a.part_hw ? a.ocount[p] : 0u;
  uint32_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= (uint32_t)d) incl += u;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t t = warp_tot[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= (uint32_t)d) t += u;
    }
    warp_tot[lane] = t;
  }
  __syncthreads();
  if (p < a.part_hw) {
    const uint32_t local = incl - v + (warp ? warp_tot[warp - 1] : 0u);
    a.ooff[p] = local;
    a.ocursor[p] = local;
  }
  if (threadIdx.x == 1023) a.oblk[blockIdx.x] = warp_tot[31];
}

__global__ void __launch_bounds__(1024) k_overflow_scan_top(RoundArgs a) {
  dep_launch();
  dep_wait();
  if (a.ctl->ovf_count == 0) return;
  const uint32_t nblk = (a.part_hw + 1023) / 1024;
  cta_scan_1024(a.oblk, a.oblk, nullptr, nblk, 0xFFFFFFFFu);  // oblk[nblk] = all overflow tuples
}

// Start of partition p's overflow list (p <= part_hw; part_hw gives the end).
__device__ __forceinline__ uint32_t overflow_offset(const RoundArgs &a, uint32_t p) {
  return p < a.part_hw ? a.oblk[p >> 10] + a.ooff[p] : a.oblk[(a.part_hw + 1023) >> 10];
}

__device__ __forceinline__ void overflow_scatter_body(const RoundArgs &a) {
  const uint32_t n = min(a.ctl->ovf_count, a.ovf_cap);
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const uint4 r = a.otup[t];
    const uint32_t dst = a.oblk[r.w >> 10] + atomicAdd(&a.ocursor[r.w], 1u);
    if (dst < n) a.stup[dst] = make_uint4(r.x, r.y, r.z, (uint32_t)mix64(((unsigned long long)r.y << 32) | r.x));
  }
}

__global__ void k_overflow_scatter(RoundArgs a) {
  dep_launch();
  dep_wait();
  overflow_scatter_body(a);
}

// In-place exclusive scan of 2^kLog2 counters by a CTA of kThreads.
template <int kThreads, int kLog2>
__device__ __forceinline__ void cta_exclusive_scan(uint32_t *h, uint32_t *warp_tot) {
  constexpr int n = 1 << kLog2;
  constexpr int per = n / kThreads;
  constexpr int nwarps = kThreads / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t loc[per];
  uint32_t sum = 0;
  if constexpr (per % 4 == 0) {  // (word by word, a warp's lanes would share few banks)
#pragma unroll
    for (int r = 0; r < per; r += 4) {
      const uint4 v = reinterpret_cast<const uint4 *>(h)[(tid * per + r) / 4];
      loc[r] = v.x;
      loc[r + 1] = v.y;
      loc[r + 2] = v.z;
      loc[r + 3] = v.w;
      sum += v.x + v.y + v.z + v.w;
    }
  } else {
#pragma unroll
    for (int r = 0; r < per; ++r) {
      loc[r] = h[tid * per + r];
      sum += loc[r];
    }
  }
  uint32_t incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t t = lane < nwarps ? warp_tot[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= d) t += v;
    }
    if (lane < nwarps) warp_tot[lane] = t;
  }
  __syncthreads();
  uint32_t run = incl - sum + (warp ? warp_tot[warp - 1] : 0);
#pragma unroll
  for (int r = 0; r < per; ++r) {
    const uint32_t c = loc[r];
    loc[r] = run;
    run += c;
  }
  if constexpr (per % 4 == 0) {
#pragma unroll
    for (int r = 0; r < per; r += 4)
      reinterpret_cast<uint4 *>(h)[(tid * per + r) / 4] = make_uint4(loc[r], loc[r + 1], loc[r + 2], loc[r + 3]);
  } else {
#pragma unroll
    for (int r = 0; r < per; ++r) h[tid * per + r] = loc[r];
  }
}

// Sum of v over the CTA's kThreads threads, returned to every thread
// (warp_tot: kThreads / 32 words of scratch).  Every thread calls it.
template <int kThreads>
__device__ __forceinline__ uint32_t cta_sum(uint32_t v, uint32_t *warp_tot) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) warp_tot[threadIdx.x >> 5] = v;
  __syncthreads();
  uint32_t total = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) total += warp_tot[w];
  __syncthreads();
  return total;
}

__device__ __forceinline__ bool full_key_less(unsigned long long seed, unsigned long long round, uint32_t i,
                                              uint32_t j) {
  const unsigned long long ki = perm_key(seed, round, i), kj = perm_key(seed, round, j);
  return ki < kj || (ki == kj && i < j);
}

// The shared memory of one bucket's sort: the bucket's records as copied,
// the record at each slot, the sub-bucket histogram, per-warp sums, and the
// mbarrier the bulk copy completes on.
struct SortSmem {
  uint4 *srec;       // {32 key bits, position, edge lo, edge hi}, room for a bucket
  uint16_t *sidx;    // record at each slot of the bucket
  uint32_t *hist;    // one counter per sub-bucket (as many as the bucket has room for records)
  uint32_t *warp_tot;
  unsigned long long *bar;
  // the one-launch round's straddling pairs (second bucket, first slot) of the
  // buckets sorted so far
  uint2 *meet = nullptr;
  uint32_t *meets = nullptr;
};

// Shared memory of a sort of buckets with room for 2^log2 records (the
// sub-bucket histogram has as many counters).
constexpr size_t sort_smem_bytes(uint32_t log2) {
  return (sizeof(uint4) + sizeof(uint16_t) + sizeof(uint32_t)) * (size_t(1) << log2) + sizeof(uint32_t) * 32 + 16;
}

// Bucket b, by one CTA of kThreads threads.  The bucket's records come into
// shared memory in one bulk copy (the TMA engine, cp.async.bulk, completing
// on the mbarrier's phase `parity`); an exact sort of record indices by
// (key, position) follows: a counting sort on the top key bits, insertion
// sort inside the sub-buckets, and a full-key fix for runs of equal 32-bit
// key parts.  Then the list is written back in this round's slot order and
// the switches of all pairs of consecutive slots inside the bucket are
// built.  Returns false (with kErrCopy set) if the copy did not land in time;
// the caller must stop then.  Every thread of the CTA calls it; `parity`
// tracks the barrier's phase across the buckets a CTA sorts.  A pair that
// straddles two buckets is listed for k_boundary, or (kMeet, the one-launch
// round, where that stage would cost a grid barrier) for meet_pairs.
template <int kThreads, int kLog2, bool kMeet = false>
__device__ __forceinline__ bool sort_bucket(const RoundArgs &a, uint32_t b, const SortSmem &sm, uint32_t &parity,
                                            bool local_offsets = false) {
  constexpr uint32_t kCap = 1u << kLog2;
  constexpr int kSubBits = kLog2;  // sub-buckets: about two per record
  uint4 *const srec = sm.srec;
  uint16_t *const sidx = sm.sidx;
  uint32_t *const hist = sm.hist;
  const int tid = threadIdx.x;
  constexpr int nsub = 1 << kSubBits;
  const uint32_t c = a.owner_bucket[b];
  if (c == kNoChain) return true;
  const uint32_t cnt = min(a.pcount[b], kCap);
  if (tid == 0 && cnt) {
    // the one-launch round: the records were appended by this launch's threads,
    // and the CTA's bucket before this one was read where the copy goes
    if constexpr (kMeet) proxy_fence();
    mbar_arrive_expect(sm.bar, cnt * (uint32_t)sizeof(uint4));
    bulk_copy_g2s(srec, a.prec + ((size_t)b << kLog2), cnt * (uint32_t)sizeof(uint4), sm.bar);
  }
  for (int s2 = tid; s2 < nsub; s2 += kThreads) hist[s2] = 0;
  const unsigned long long R = a.ctl->pool_round;
  const ChainDesc ch = a.chains[c];
  const unsigned long long round = chain_round(ch, R);
  const uint32_t ell = ch.exact_ell ? a.chain_ell[c] : 0u;
  // chain-local slot offset: from the scanned offsets, or summed here over
  // the chain's earlier buckets (a small chain in the one-launch round)
  uint32_t loff;
  if (local_offsets) {
    uint32_t sum = 0;
    for (uint32_t j = ch.bucket_base + tid; j < b; j += kThreads) sum += min(a.pcount[j], kCap);
    loff = cta_sum<kThreads>(sum, sm.warp_tot);
  } else {
    loff = bucket_offset(a, b) - bucket_offset(a, ch.bucket_base);
  }
  const uint32_t goff = ch.slot_base + loff;
  __syncthreads();  // the histogram is cleared
  const bool landed = cnt == 0 || mbar_wait(sm.bar, parity, kCopyWaitPolls);
  if (__syncthreads_or(!landed)) {
    // the copy did not complete in time: report it, give it a last bounded
    // wait (shared memory must not be released under a copy in flight), stop
    if (tid == 0) atomicOr(&a.ctl->err, kErrCopy);
    if (cnt) mbar_wait(sm.bar, parity, kCopyWaitPolls);
    return false;
  }
  if (cnt) parity ^= 1u;  // the barrier's next phase serves the CTA's next copy
  for (uint32_t t = tid; t < cnt; t += kThreads) atomicAdd(&hist[srec[t].x >> (32 - kSubBits)], 1u);
  __syncthreads();
  cta_exclusive_scan<kThreads, kSubBits>(hist, sm.warp_tot);
  __syncthreads();
  for (uint32_t t = tid; t < cnt; t += kThreads) sidx[atomicAdd(&hist[srec[t].x >> (32 - kSubBits)], 1u)] = t;
  __syncthreads();
  // hist[s] is now the end of sub-bucket s; sort each (a handful of items)
  // by (32 key bits, position)
  for (int s2 = tid; s2 < nsub; s2 += kThreads) {
    const uint32_t beg = s2 ? hist[s2 - 1] : 0, end = hist[s2];
    for (uint32_t x = beg + 1; x < end; ++x) {
      const uint16_t li = sidx[x];
      const unsigned long long val = ((unsigned long long)srec[li].x << 32) | srec[li].y;
      uint32_t y = x;
      for (; y > beg; --y) {
        const uint2 kp = *reinterpret_cast<const uint2 *>(&srec[sidx[y - 1]]);
        if ((((unsigned long long)kp.x << 32) | kp.y) <= val) break;
        sidx[y] = sidx[y - 1];
      }
      sidx[y] = li;
    }
  }
  __syncthreads();
  // equal 32-bit key parts: order those runs by the full key
  for (uint32_t t = tid; t + 1 < cnt; t += kThreads) {
    const uint32_t mt = srec[sidx[t]].x;
    if (srec[sidx[t + 1]].x == mt && (t == 0 || srec[sidx[t - 1]].x != mt)) {
      uint32_t e = t + 2;
      while (e < cnt && srec[sidx[e]].x == mt) ++e;
      for (uint32_t x = t + 1; x < e; ++x) {
        const uint16_t li = sidx[x];
        const uint32_t pos = srec[li].y;
        uint32_t y = x;
        while (y > t && full_key_less(ch.seed, round, pos, srec[sidx[y - 1]].y)) {
          sidx[y] = sidx[y - 1];
          --y;
        }
        sidx[y] = li;
      }
    }
  }
  __syncthreads();
  // slots of the bucket hold pi in order: write the list in slot order, a
  // pair of slots (a switch) per thread, and build the switch; a pair's first
  // slot is even in the pool (chains start on even slots), so both slots go
  // out in one 8-byte and one 16-byte store
  const uint32_t t0 = loff & 1u;
  const uint32_t npairs = cnt > t0 ? (cnt - t0) >> 1 : 0;
  for (uint32_t p = tid; p < npairs; p += kThreads) {
    const uint32_t t = t0 + 2 * p;
    const uint4 r1 = srec[sidx[t]], r2 = srec[sidx[t + 1]];
    const bool valid[1] = {true};
    const uint32_t k[1] = {(loff + t) >> 1}, i[1] = {r1.y}, j[1] = {r2.y};
    const unsigned long long e1[1] = {((unsigned long long)r1.w << 32) | r1.z};
    const unsigned long long e2[1] = {((unsigned long long)r2.w << 32) | r2.z};
    *reinterpret_cast<uint2 *>(&a.cpos[goff + t]) = make_uint2(r1.y, r2.y);
    *reinterpret_cast<ulonglong2 *>(&a.cedge[goff + t]) = make_ulonglong2(e1[0], e2[0]);
    build_switches<1>(a, ch, round, ell, valid, k, i, e1, j, e2);
  }
  // the slots in no pair of this bucket: the first (its pair started in the
  // bucket before) and the last (its pair ends in the next bucket, or m is odd)
  if (tid < 2 && cnt > 0) {
    const uint32_t t = tid == 0 ? 0u : cnt - 1;
    const bool alone = tid == 0 ? t0 == 1 : ((cnt - t0) & 1u) && cnt - 1 >= t0 && !(t0 == 1 && cnt == 1);
    if (alone) {
      const uint4 r = srec[sidx[t]];
      a.cpos[goff + t] = r.y;
      a.cedge[goff + t] = ((unsigned long long)r.w << 32) | r.z;
      if (kMeet && (tid == 0 || loff + cnt < ch.m)) {
        // the bucket with the pair's second slot (there is one unless a bucket
        // overflowed, which was reported), and the pair's first slot
        const uint32_t end = ch.bucket_base + (1u << ch.B);
        uint32_t second = b;
        if (tid == 1) do { ++second; } while (second < end && a.pcount[second] == 0);
        if (second < end) sm.meet[atomicAdd(sm.meets, 1u)] = make_uint2(second, tid == 0 ? goff - 1 : goff + t);
      }
    }
  }
  if (!kMeet && tid == 0 && t0 == 1 && cnt > 0) {
    // this bucket's first slot is the second of a pair started in an
    // earlier bucket: k_boundary builds that switch from the list
    const uint32_t idx = atomicAdd(&a.ctl->boundary, 1u);
    a.bnd[idx] = goff - 1;  // the pair's first slot
  }
  __syncthreads();  // the CTA's shared memory may take the next bucket's copy
  return true;
}

// The straddling pairs a CTA of the one-launch round has a slot of: the later
// of a pair's two CTAs to get here, which the count bnd[second bucket] tells,
// builds it, both slots being written then.  Every thread of the CTA calls it.
constexpr uint32_t kMeets = 256;
__device__ __forceinline__ void meet_pairs(const RoundArgs &a, const SortSmem &sm) {
  __syncthreads();
  const uint32_t n = *sm.meets;
  for (uint32_t x = threadIdx.x; x < n; x += blockDim.x) {
    const uint32_t second = sm.meet[x].x, g = sm.meet[x].y;
    __threadfence();
    if (atomicAdd(&a.bnd[second], 1u) == 0) continue;
    __threadfence();
    const uint32_t c = a.owner_bucket[second];
    const ChainDesc ch = a.chains[c];
    const bool valid[1] = {true};
    const uint32_t k[1] = {(g - ch.slot_base) >> 1}, i[1] = {__ldcg(&a.cpos[g])}, j[1] = {__ldcg(&a.cpos[g + 1])};
    const unsigned long long e1[1] = {__ldcg(&a.cedge[g])}, e2[1] = {__ldcg(&a.cedge[g + 1])};
    build_switches<1>(a, ch, chain_round(ch, a.ctl->pool_round), ch.exact_ell ? a.chain_ell[c] : 0u, valid, k, i, e1,
                      j, e2);
  }
  __syncthreads();
  if (threadIdx.x == 0) *sm.meets = 0;
  __syncthreads();
}

// One CTA per bucket (the round's launch over all buckets): buckets with
// room for 2^kLog2 records, CTAs of 2^(kLog2 - 3) threads, kMin of them
// per SM.  Seven CTAs of 128 threads (70 registers) sorted G(2^24)'s
// buckets in 3.85 ms per round, against 3.98 with six (80 registers), 4.02-
// 4.07 with eight (63) and 5.37 with nine (56).  The larger buckets run four
// CTAs of 256 threads (63 registers; three at 80 took 4.90 against 4.51 ms on
// the 4096-chain ensemble).
template <int kLog2, int kMin>
__global__ void __launch_bounds__(1 << (kLog2 - 3), kMin) k_sortpair(RoundArgs a) {
  constexpr int kThreads = 1 << (kLog2 - 3);
  __shared__ __align__(128) uint4 srec[1 << kLog2];
  __shared__ uint16_t sidx[1 << kLog2];
  __shared__ __align__(16) uint32_t hist[1 << kLog2];
  __shared__ uint32_t warp_tot[kThreads / 32];
  __shared__ __align__(8) unsigned long long bar;
  dep_launch();
  if (threadIdx.x == 0) mbar_init(&bar, 1);
  __syncthreads();
  dep_wait();
  const SortSmem sm{srec, sidx, hist, warp_tot, &bar};
  uint32_t parity = 0;
  if (sort_bucket<kThreads, kLog2>(a, blockIdx.x, sm, parity) && threadIdx.x == 0) mbar_inval(&bar);
}

__device__ __forceinline__ void boundary_body(const RoundArgs &a) {
  const uint32_t n = a.ctl->boundary;
  const unsigned long long R = a.ctl->pool_round;
  for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
    const uint32_t g = a.bnd[idx];  // first slot of the pair
    const uint32_t c = g < a.slot_hw ? a.owner_slot[g] : kNoChain;
    if (c == kNoChain) {  // cannot happen unless a bucket overflowed (reported)
      atomicOr(&a.ctl->err, kErrRecord);
      continue;
    }
    const ChainDesc ch = a.chains[c];
    const uint32_t k = (g - ch.slot_base) >> 1;
    if (k >= ch.L) {
      atomicOr(&a.ctl->err, kErrRecord);
      continue;
    }
    // both slots were written by the sort kernel (the list in this round's slot order)
    const bool valid[1] = {true};
    const uint32_t kk[1] = {k}, i[1] = {a.cpos[g]}, j[1] = {a.cpos[g + 1]};
    const unsigned long long e1[1] = {a.cedge[g]}, e2[1] = {a.cedge[g + 1]};
    build_switches<1>(a, ch, chain_round(ch, R), ch.exact_ell ? a.chain_ell[c] : 0u, valid, kk, i, e1, j, e2);
  }
}

__global__ void k_boundary(RoundArgs a) {
  dep_launch();
  dep_wait();
  boundary_body(a);
}

// The chain of a thread's current pair, kept while its consecutive pairs
// stay in it: pairs [lo, hi) are chain c's.  The only chain of a pool needs no
// owner map (G(2^24): k_sources 1.54 -> 1.48 ms, k_wave1 0.27 -> 0.17 with its
// counts summed per CTA; k_permute got slower by 3% and keeps the map).
struct PairChain {
  uint32_t c = kNoChain, lo = 1, hi = 0;
};

// Make pc the chain of pair x; false if no chain owns it.
__device__ __forceinline__ bool pair_chain(const RoundArgs &a, uint32_t x, PairChain &pc) {
  if (x >= pc.lo && x < pc.hi) return true;
  if (a.solo_chain != kNoChain) {
    pc.c = a.solo_chain;
    pc.lo = a.chains[pc.c].slot_base >> 1;
    pc.hi = pc.lo + ((a.chains[pc.c].m + 1) >> 1);
    return x >= pc.lo && x < pc.hi;
  }
  pc.c = a.owner_slot[2 * x];
  if (pc.c == kNoChain) {
    pc.lo = 1;
    pc.hi = 0;
    return false;
  }
  pc.lo = a.chains[pc.c].slot_base >> 1;
  pc.hi = pc.lo + ((a.chains[pc.c].m + 1) >> 1);
  return true;
}

// One pair of slots: its two sources, the ERASE value they carry, and
// where their tuples go (each key's partition cursor and storage, from its
// chain).  A key that needs no tuple becomes kEmptyKey.
struct SourcePair {
  unsigned long long key[2], hash[2];
  uint32_t val, cursor[2], capt, part[2];
  size_t base[2];
};

__device__ __forceinline__ void load_source_pair(const RoundArgs &a, uint32_t x, bool owned, uint32_t c,
                                                 ulonglong2 ee, SourcePair &sp) {
  sp.key[0] = ee.x;
  sp.key[1] = ee.y;
  sp.val = kTupleSource | kKeepK;
  if (!owned) {
    sp.key[0] = sp.key[1] = kEmptyKey;
    return;
  }
  const ChainDesc &ch = a.chains[c];
  const uint32_t ls = 2 * x - ch.slot_base;
  if (ls + 1 < ch.m) {
    const uint32_t kg = ch.switch_base + (ls >> 1);
    if ((__ldcs(&a.word[kg]) & kCodeMask) == 0) sp.val = kTupleSource | kg;
  } else {
    sp.key[1] = kEmptyKey;  // odd m: the unpaired last slot
  }
  sp.capt = ch.capt;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    sp.hash[t] = mix64(sp.key[t]);
    const uint32_t p = partition_of(sp.hash[t], ch.P);
    sp.cursor[t] = ch.tcount_base + p * ch.tstride;
    sp.base[t] = ch.tuple_base + (size_t)p * ch.capt;
    sp.part[t] = ch.part_base + p;
  }
}

// The sources of every switch (Algorithm 1's ERASE tuples) from the list in
// this round's slot order, two pairs per thread (x and x + 256): all loads
// first (list entries, reject words, filter words), then the cursor atomics
// of all four keys, then their stores.  Only an edge id that is some
// switch's target needs a tuple (the grouping only asks whether targets
// exist and who erases them), so a source whose filter bit is clear is
// dropped; a set bit can be a collision, which only adds a tuple nobody
// needs.  The unpaired last slot of an odd list is a source no switch
// erases, and so are the sources of a switch rejected outright.
__device__ __forceinline__ void source_pairs(const RoundArgs &a, uint32_t x, uint32_t y, uint32_t end) {
  PairChain pc;
  const ulonglong2 ex = __ldcs(reinterpret_cast<const ulonglong2 *>(a.cedge) + x);
  ulonglong2 ey = make_ulonglong2(kEmptyKey, kEmptyKey);
  if (y < end) ey = __ldcs(reinterpret_cast<const ulonglong2 *>(a.cedge) + y);
  SourcePair sp[2];
  const bool ox = pair_chain(a, x, pc);
  load_source_pair(a, x, ox, pc.c, ex, sp[0]);
  const bool oy = y < end && pair_chain(a, y, pc);
  load_source_pair(a, y, oy, pc.c, ey, sp[1]);
  uint32_t w[2][2];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int t = 0; t < 2; ++t)
      w[q][t] = sp[q].key[t] == kEmptyKey ? 0u : __ldcg(&a.tfilter[filter_bit(a, sp[q].hash[t]) >> 5]);
  uint32_t idx[2][2];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (!((w[q][t] >> (filter_bit(a, sp[q].hash[t]) & 31)) & 1u)) sp[q].key[t] = kEmptyKey;
      idx[q][t] = sp[q].key[t] != kEmptyKey ? atomicAdd(&a.tcount[sp[q].cursor[t]], 1u) : 0u;
    }
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const unsigned long long k = sp[q].key[t];
      if (k == kEmptyKey) continue;
      if (idx[q][t] < sp[q].capt) {
        a.ptup[sp[q].base[t] + idx[q][t]] = make_uint4((uint32_t)k, (uint32_t)(k >> 32), sp[q].val,
                                                       (uint32_t)sp[q].hash[t]);
      } else {
        const uint32_t o = atomicAdd(&a.ctl->ovf_count, 1u);
        if (o < a.ovf_cap)
          a.otup[o] = make_uint4((uint32_t)k, (uint32_t)(k >> 32), sp[q].val, sp[q].part[t]);
        else
          atomicOr(&a.ctl->err, kErrRecord);
      }
    }
}

// One launch of short-lived CTAs, two pairs per thread (measured faster than
// a grid-stride loop over a resident grid).
__global__ void __launch_bounds__(256, 4) k_sources(RoundArgs a) {
  dep_launch();
  const uint32_t end = a.slot_hw >> 1;
  dep_wait();
  const uint32_t x = scrambled_cta(a.sources_stride) * 2 * blockDim.x + threadIdx.x;
  if (x < end) source_pairs(a, x, x + blockDim.x, end);
}

// Grouping of one tuple partition by edge id (Algorithm 1's table T for the
// partition's edge ids).  Most targets are proposed by no other switch and
// equal no edge of the graph: two bitmaps over 15 bits of the ids' hashes tell
// them.  Every target sets its bit of `seen`; a bit met twice, or met by a
// source, is also set in `marked`; a target whose bit is not marked is free.
// The other targets, and the sources that met a target's bit, go into a
// shared-memory table of S slots: slot[s] = {key lo, key hi, p, q} with p the
// eraser (from the source tuple) and q the smallest inserter, and aux[s] = 1
// once a second inserter arrives.  Then wave 1 for each of these targets:
// present when k runs (p >= k), dependent on an undecided switch (p < k, or an
// earlier inserter q < k), or free.  Edge ids with a dependency get an entry
// {p, q} for the later waves, whose index replaces aux[s].  Slots are probed
// from the low bits of the id's hash, which the tuple carries; the bitmaps use
// other bits of it.
struct GroupSmem {
  uint4 *slot;
  uint32_t *aux;
  uint32_t *seen, *marked;
};

constexpr uint32_t kGroupBitsLog2 = 15, kGroupWords = 1u << (kGroupBitsLog2 - 5);

__device__ __forceinline__ GroupSmem group_smem(uint32_t S) {
  extern __shared__ uint4 group_dyn[];
  GroupSmem g;
  g.slot = group_dyn;
  g.aux = reinterpret_cast<uint32_t *>(group_dyn + S);
  g.seen = g.aux + S;
  g.marked = g.seen + kGroupWords;
  return g;
}

__device__ __forceinline__ unsigned long long *slot_key(const GroupSmem &g, uint32_t s) {
  return reinterpret_cast<unsigned long long *>(&g.slot[s]);
}

__device__ __forceinline__ void group_reset_slot(const GroupSmem &g, uint32_t s) {
  g.slot[s] = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, kPNone, kQNone);
  g.aux[s] = 0;
}

constexpr uint32_t kClaimed = 0x80000000u;  // slot result: this thread took the slot

// Insert one tuple; returns its slot (| kClaimed if this thread took the
// empty slot), or S if the table is full.
__device__ __forceinline__ uint32_t group_insert(const GroupSmem &g, uint32_t S, unsigned long long key, uint32_t h,
                                                 uint32_t v) {
  uint32_t s = h & (S - 1), n = 0, claimed = 0;
  for (; n < S; ++n) {
    const unsigned long long cur = *slot_key(g, s);
    if (cur == key) break;
    if (cur == kEmptyKey) {
      const unsigned long long prev = atomicCAS(slot_key(g, s), kEmptyKey, key);
      if (prev == kEmptyKey) {
        claimed = kClaimed;
        break;
      }
      if (prev == key) break;
    }
    s = (s + 1) & (S - 1);
  }
  if (n == S) return S;
  if (v & kTupleSource) {
    const uint32_t kk = v & kTupleK;
    g.slot[s].z = kk == kKeepK ? kPKeep : kk;  // one source per edge id (Obs. 2)
  } else if (atomicMin(&g.slot[s].w, v & kTupleK) != kQNone) {
    g.aux[s] = 1;  // a second inserter
  }
  return s | claimed;
}

// One dependency entry per edge id that some target depends on: an id
// inserted more than once, or inserted while in E at the round start.
// aux[s] is replaced by the entry index (kTrivial if none).
__device__ __forceinline__ void group_alloc(const RoundArgs &a, const GroupSmem &g, uint32_t s) {
  const uint32_t p = g.slot[s].z, q = g.slot[s].w;
  const bool need = q != kQNone && (g.aux[s] != 0 || p != kPNone);
  uint32_t idx = kTrivial;
  if (need) {
    idx = atomicAdd(&a.ctl->dep_count, 1u);
    if (idx < a.dep_cap) {
      a.dep[idx] = make_uint2(p, q);
    } else {
      idx = kTrivial;
      atomicOr(&a.ctl->err, kErrRecord);
    }
  }
  g.aux[s] = idx;
}

// Wave 1 for target tuple v in slot s.
__device__ __forceinline__ void group_decide(const RoundArgs &a, const GroupSmem &g, uint32_t s, uint32_t v) {
  const uint32_t k = v & kTupleK;
  const uint32_t p = g.slot[s].z, q = g.slot[s].w, d = g.aux[s];
  uint32_t flags = 0;
  if (p != kPNone && p >= k) flags = kFlagBad;                // present when k runs
  else if (p != kPNone || q != k) flags = kFlagDep;           // erased or inserted earlier, maybe
  if (d != kTrivial) {
    flags |= v & kTupleWhich ? kFlagEntry4 : kFlagEntry3;
    if (v & kTupleWhich) a.sw[k].y = d;
    else a.sw[k].x = d;
  }
  if (flags) atomicOr(&a.word[k], flags);
}

// Persistent CTAs over the partitions.  Fast path: a thread keeps the hash
// and the value of its R tuples (a quarter more in a partition of more than
// R T, if the table has room for so many ids) in registers, reads the ids of those that go into the table again, and
// clears the slots it claimed.  R T is the mean a partition may reach by its
// layout with every source in it, as in a graph so large that the filter lets
// nearly all through; half of those have more (G(2^27), 1.07e9 edges: 362 ms a
// round with them on the sub-pass path, 138 so).  Partitions with more tuples
// than that, or more distinct marked ids than slots, take the sub-pass path, all tuples into the table: the ids whose hash
// bits 16.. select them, split further until each sub-pass fits.
//
// What bounds it: the barriers and shared-memory latency of one partition
// after another, about a third of it the wait for its tuples.  With every tuple
// in a table of 64-bit keys, 1024-thread CTAs took 2.31 ms per round of G(2^24)
// and 0.169 of 256 mixed chains; so, 512-thread CTAs, three per SM, take 1.47
// and 0.123 (256 threads: 1.35, but the round 0.15 ms longer; 128: 2.84).
// Bring the own tuples of partition `part` (if it exists and is owned) into
// L2 with one bulk prefetch (the TMA engine), so that the CTA finds them
// there when it gets to that partition.
__device__ __forceinline__ void prefetch_partition(const RoundArgs &a, uint32_t part) {
  if (part >= a.part_hw) return;
  const uint32_t c = a.owner_part[part];
  if (c == kNoChain) return;
  const ChainDesc &cd = a.chains[c];
  const uint32_t n = min(a.tcount[cd.tcount_base + (part - cd.part_base) * cd.tstride], cd.capt);
  if (n) bulk_prefetch_l2(a.ptup + cd.tuple_base + (size_t)(part - cd.part_base) * cd.capt, n * (uint32_t)sizeof(uint4));
}

// A partition's tuples, R to a thread.  Returns true, with *overflow set and
// the slots claimed here cleared again, if the table was too small for them.
template <int T, int R>
__device__ __forceinline__ bool group_fast(const RoundArgs &a, const GroupSmem &g, uint32_t S, const uint4 *prim,
                                           uint32_t nprim, uint32_t obeg, uint32_t ntup, uint32_t *overflow) {
  const int tid = threadIdx.x;
  uint32_t h[R], v[R], todo = 0;  // todo: this thread's tuples that go into the table
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const uint32_t t = tid + j * T;
    v[j] = kTupleSource;
    if (t < ntup) {
      const uint2 zw = __ldcs(reinterpret_cast<const uint2 *>(t < nprim ? &prim[t] : &a.stup[obeg + (t - nprim)]) + 1);
      v[j] = zw.x;
      h[j] = zw.y;
      if (!(zw.x & kTupleSource)) {
        const uint32_t bit = h[j] >> (32 - kGroupBitsLog2), m = 1u << (bit & 31);
        if (atomicOr(&g.seen[bit >> 5], m) & m) atomicOr(&g.marked[bit >> 5], m);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < R; ++j)
    if (tid + j * T < ntup && (v[j] & kTupleSource)) {
      const uint32_t bit = h[j] >> (32 - kGroupBitsLog2), m = 1u << (bit & 31);
      if (g.seen[bit >> 5] & m) {
        atomicOr(&g.marked[bit >> 5], m);
        todo |= 1u << j;
      }
    }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < R; ++j)
    if (!(v[j] & kTupleSource)) {
      const uint32_t bit = h[j] >> (32 - kGroupBitsLog2);
      if ((g.marked[bit >> 5] >> (bit & 31)) & 1u) todo |= 1u << j;
    }
  // h of a tuple that goes into the table becomes its slot
#pragma unroll
  for (int j = 0; j < R; ++j)
    if ((todo >> j) & 1u) {
      const uint32_t t = tid + j * T;
      const uint2 id = *reinterpret_cast<const uint2 *>(t < nprim ? &prim[t] : &a.stup[obeg + (t - nprim)]);
      h[j] = group_insert(g, S, ((unsigned long long)id.y << 32) | id.x, h[j], v[j]);
      if (h[j] == S) {
        *overflow = 1;
        todo &= ~(1u << j);
      }
    }
  __syncthreads();
  const bool full = *overflow != 0;
  for (uint32_t w = tid; w < 2 * kGroupWords / 4; w += T)  // both bitmaps
    reinterpret_cast<uint4 *>(g.seen)[w] = make_uint4(0, 0, 0, 0);
  if (!full) {
#pragma unroll
    for (int j = 0; j < R; ++j)
      if (((todo >> j) & 1u) && (h[j] & kClaimed)) group_alloc(a, g, h[j] & ~kClaimed);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < R; ++j)
      if (((todo >> j) & 1u) && !(v[j] & kTupleSource)) group_decide(a, g, h[j] & ~kClaimed, v[j]);
  }
  __syncthreads();
  // (the next partition's first table access comes two barriers later)
#pragma unroll
  for (int j = 0; j < R; ++j)
    if (((todo >> j) & 1u) && (h[j] & kClaimed)) group_reset_slot(g, h[j] & ~kClaimed);
  return full;
}

template <int T, int R>
__device__ __forceinline__ void group_body(const RoundArgs &a) {
  const uint32_t S = 1u << a.group_log2;
  const GroupSmem g = group_smem(S);
  __shared__ uint32_t stk_sub[64], stk_n[64];
  __shared__ int stk_top;
  __shared__ uint32_t overflow;
  const int tid = threadIdx.x;
  for (uint32_t s = tid; s < S; s += T) group_reset_slot(g, s);
  for (uint32_t w = tid; w < 2 * kGroupWords; w += T) g.seen[w] = 0;
  if (tid == 0) overflow = 0;
  dep_wait();  // (does nothing in the one-launch round)
  const bool ovf = a.ctl->ovf_count != 0;
  __syncthreads();
  for (uint32_t part = blockIdx.x; part < a.part_hw; part += gridDim.x) {
    const uint32_t c = a.owner_part[part];
    if (c == kNoChain) continue;
    if (tid == 0) prefetch_partition(a, part + gridDim.x);
    const uint32_t pbase = a.chains[c].part_base, tbase = a.chains[c].tuple_base, capt = a.chains[c].capt;
    // the partition's tuples: its own region, then its overflow tuples
    const uint4 *prim = a.ptup + tbase + (size_t)(part - pbase) * capt;
    const ChainDesc &cd = a.chains[c];
    const uint32_t nprim = min(a.tcount[cd.tcount_base + (part - pbase) * cd.tstride], capt);
    const uint32_t obeg = ovf ? overflow_offset(a, part) : 0, oend = ovf ? overflow_offset(a, part + 1) : 0;
    const uint32_t ntup = nprim + (oend - obeg);
    constexpr int kWide = R + R / 4;
    if (ntup <= (uint32_t)((S >= R * T ? kWide : R) * T)) {
      const bool full = ntup <= (uint32_t)(R * T)
                            ? group_fast<T, R>(a, g, S, prim, nprim, obeg, ntup, &overflow)
                            : group_fast<T, kWide>(a, g, S, prim, nprim, obeg, ntup, &overflow);
      if (!full) continue;
      if (tid == 0) overflow = 0;
      __syncthreads();
    }
    // sub-pass path
    if (tid == 0) {
      atomicAdd(&a.st->subpass_partitions, 1ull);
      stk_top = 1;
      stk_sub[0] = 0;
      stk_n[0] = 1;
    }
    __syncthreads();
    while (stk_top > 0) {
      const uint32_t sub = stk_sub[stk_top - 1], ns = stk_n[stk_top - 1];
      __syncthreads();
      if (tid == 0) {
        --stk_top;
        overflow = 0;
      }
      for (uint32_t s = tid; s < S; s += T) group_reset_slot(g, s);
      __syncthreads();
      for (uint32_t t = tid; t < ntup; t += T) {
        const uint4 r = t < nprim ? prim[t] : a.stup[obeg + (t - nprim)];
        if (ns > 1 && ((r.w >> 16) & (ns - 1)) != sub) continue;
        if (group_insert(g, S, ((unsigned long long)r.y << 32) | r.x, r.w, r.z) == S) overflow = 1;
      }
      __syncthreads();
      if (overflow) {
        if (tid == 0) {
          if (ns >= (1u << 16) || stk_top + 2 > 64) {
            atomicOr(&a.ctl->err, kErrGroup);
          } else {
            stk_sub[stk_top] = sub + ns;
            stk_n[stk_top] = 2 * ns;
            stk_sub[stk_top + 1] = sub;
            stk_n[stk_top + 1] = 2 * ns;
            stk_top += 2;
          }
        }
        __syncthreads();
        continue;
      }
      for (uint32_t s = tid; s < S; s += T)
        if (*slot_key(g, s) != kEmptyKey) group_alloc(a, g, s);
      __syncthreads();
      for (uint32_t t = tid; t < ntup; t += T) {
        const uint4 r = t < nprim ? prim[t] : a.stup[obeg + (t - nprim)];
        if (r.z & kTupleSource) continue;
        if (ns > 1 && ((r.w >> 16) & (ns - 1)) != sub) continue;
        const unsigned long long key = ((unsigned long long)r.y << 32) | r.x;
        uint32_t s = r.w & (S - 1);
        for (uint32_t n = 0; n < S && *slot_key(g, s) != key; ++n) s = (s + 1) & (S - 1);
        group_decide(a, g, s, r.z);
      }
      __syncthreads();
    }
    // leave the table empty for the next partition
    for (uint32_t s = tid; s < S; s += T) group_reset_slot(g, s);
    if (tid == 0) overflow = 0;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kGroupThreads, kGroupMin) k_group(RoundArgs a) {
  dep_launch();
  group_body<kGroupThreads, 2048 / kGroupThreads>(a);
}

// Each CTA takes a contiguous range of switches, so that a thread's running
// per-chain count changes chain only at chain boundaries.  The counts leave the
// CTA once: by the warp, their atomics on a handful of words took 15 of the 20
// us of a power law of 1e6 edges.
__device__ __forceinline__ void wave1_body(const RoundArgs &a) {
  Tally t;
  ChainCount cc;
  const uint32_t per = (a.switch_hw + gridDim.x - 1) / gridDim.x;
  const uint32_t chunk = (per + blockDim.x - 1) / blockDim.x * blockDim.x;
  uint32_t beg = min(blockIdx.x * chunk, a.switch_hw), end = min(beg + chunk, a.switch_hw);
  if (a.solo_chain != kNoChain) {  // its switches only
    const uint32_t lo = a.chains[a.solo_chain].switch_base, hi = lo + a.chains[a.solo_chain].L;
    beg = max(beg, lo);
    end = min(end, hi);
  }
  for (uint32_t base = beg; base < end; base += blockDim.x) {
    const uint32_t k = base + threadIdx.x;
    bool wait = false;
    uint32_t c = kNoChain;
    if (k < end) c = a.solo_chain != kNoChain ? a.solo_chain : a.owner_switch[k];
    if (c != kNoChain) {
      const uint32_t w = __ldcs(&a.word[k]);
      const uint32_t code = w & kCodeMask;
      uint32_t state = kLegal;
      if (code) {
        state = kIllegal;
        if (code == kCodeLazy) ++t.lazy;
        else if (code == kCodeLoop) ++t.rej_loop;
        else ++t.rej_exists;
      } else if (w & kFlagBad) {
        state = kIllegal;
        ++t.rej_exists;
        drop_inserter(a, k, entries_of(w, a.sw[k]));
      } else if (w & kFlagDep) {
        state = kUndecided;
        wait = true;
      } else {
        ++t.accepted;
        count_accepted(a, cc, c);
      }
      a.status[k] = state == kUndecided ? 0u : ((1u << 2) | state);
    }
    append_if(wait, k, a.list0, &a.ctl->pending[0]);
  }
  __shared__ uint32_t sums[5], chain0;
  if (threadIdx.x < 5) sums[threadIdx.x] = 0;
  if (threadIdx.x == 5) chain0 = kNoChain;
  __syncthreads();
  const uint32_t counts[4] = {t.accepted, t.rej_loop, t.rej_exists, t.lazy};
  const bool lead = (threadIdx.x & 31) == 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t n = __reduce_add_sync(0xffffffffu, counts[i]);
    if (lead && n) atomicAdd(&sums[i], n);
  }
  const uint32_t first = __reduce_min_sync(0xffffffffu, cc.n ? cc.chain : kNoChain);
  if (lead && first != kNoChain) atomicMin(&chain0, first);
  __syncthreads();
  // the CTA's first chain, usually its only one, in one sum; other chains by the warp
  const bool own = cc.n && cc.chain == chain0;
  const uint32_t n0 = __reduce_add_sync(0xffffffffu, own ? cc.n : 0u);
  if (lead && n0) atomicAdd(&sums[4], n0);
  if (own) cc.n = 0;
  if (__any_sync(0xffffffffu, cc.n != 0)) flush_count(a, cc);
  __syncthreads();
  if (threadIdx.x < 4 && sums[threadIdx.x]) {
    unsigned long long *const to = threadIdx.x == 0   ? &a.st->accepted
                                   : threadIdx.x == 1 ? &a.st->rej_loop
                                   : threadIdx.x == 2 ? &a.st->rej_exists
                                                      : &a.st->lazy;
    atomicAdd(to, (unsigned long long)sums[threadIdx.x]);
  }
  if (threadIdx.x == 4 && sums[4]) atomicAdd(&a.chain_accepted[chain0], (unsigned long long)sums[4]);
}

__global__ void k_wave1(RoundArgs a) {
  dep_launch();
  dep_wait();
  wave1_body(a);
}

__device__ __forceinline__ uint32_t wave_cap(const RoundArgs &a) {
  return a.max_waves ? a.max_waves : kDefaultWaveCap;
}

// Waves from `wave` on over the n <= kSoloPending undecided switches of `in`,
// by one CTA of T threads (every thread calls it).  A switch stays with its
// thread, with its dependency entries and their erasers, until it is decided,
// so that a wave is a registration, two dependent accesses to L2 (the smallest
// inserters, then their statuses) and a decision: about 1.8 us, where the same
// from a list in memory took 5.7 us and a pair of whole-GPU kernels 6.  Returns
// the number after the last wave.
constexpr uint32_t kSoloPending = 2048;

template <int T>
__device__ __forceinline__ uint32_t solo_waves(const RoundArgs &a, const uint32_t *in, uint32_t n, uint32_t wave) {
  constexpr int R = (int)kSoloPending / T;
  const uint32_t tid = threadIdx.x;
  Tally t;
  ChainCount cc;
  uint32_t k[R], live = 0, prev_n = n + 1;
  uint2 d[R], p[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (tid + r * T >= n) continue;
    live |= 1u << r;
    k[r] = __ldcg(&in[tid + r * T]);
    d[r] = switch_entries(a, k[r]);
    p[r].x = d[r].x != kTrivial ? __ldcg(&a.dep[d[r].x].x) : kPNone;
    p[r].y = d[r].y != kTrivial ? __ldcg(&a.dep[d[r].y].x) : kPNone;
  }
  while (n != 0) {
    if (wave > wave_cap(a)) {
      if (tid == 0) atomicOr(&a.ctl->err, kErrWaveCap);
      break;
    }
    if (n >= prev_n) {  // no switch was decided in the last wave: impossible
      if (tid == 0) atomicOr(&a.ctl->err, kErrNoProgress);
      break;
    }
    prev_n = n;
    if (tid == 0 && wave < kWaveHist) a.st->last_pending[wave] = n;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!((live >> r) & 1u)) continue;
      if (d[r].x != kTrivial) atomicMin(&a.dep[d[r].x].y, k[r]);
      if (d[r].y != kTrivial) atomicMin(&a.dep[d[r].y].y, k[r]);
    }
    __syncthreads();
    uint32_t left = live;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!((live >> r) & 1u)) continue;
      // the inserters and the erasers' statuses first, then the inserters'
      const bool x = d[r].x != kTrivial, y = d[r].y != kTrivial;
      const uint32_t qx = x ? __ldcg(&a.dep[d[r].x].y) : k[r], qy = y ? __ldcg(&a.dep[d[r].y].y) : k[r];
      const uint32_t ex = p[r].x < k[r] ? __ldcg(&a.status[p[r].x]) : 0u;
      const uint32_t ey = p[r].y < k[r] ? __ldcg(&a.status[p[r].y]) : 0u;
      const uint32_t ix = qx < k[r] ? __ldcg(&a.status[qx]) : 0u, iy = qy < k[r] ? __ldcg(&a.status[qy]) : 0u;
      const int r3 = x ? judge_target(k[r], p[r].x, qx, ex, ix, wave) : kOk;
      const int r4 = y ? judge_target(k[r], p[r].y, qy, ey, iy, wave) : kOk;
      if (r3 == kBad || r4 == kBad) {
        a.status[k[r]] = (wave << 2) | kIllegal;
        if (x && qx == k[r]) atomicCAS(&a.dep[d[r].x].y, k[r], kQNone);  // no longer an inserter
        if (y && qy == k[r]) atomicCAS(&a.dep[d[r].y].y, k[r], kQNone);
        ++t.rej_exists;
        left &= ~(1u << r);
      } else if (r3 == kOk && r4 == kOk) {
        a.status[k[r]] = (wave << 2) | kLegal;
        ++t.accepted;
        count_accepted(a, cc, a.owner_switch[k[r]]);
        left &= ~(1u << r);
      }
    }
    live = left;
    n = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) n += __syncthreads_count((live >> r) & 1u);
    ++wave;
  }
  flush_tally(a, t);
  flush_count(a, cc);
  return wave;
}

// One wave after the first, on the whole GPU.  Registration: every
// undecided switch becomes an inserter of its targets again (the q fields
// of illegal minima were cleared); also empties the list of the next wave.
// Nothing to do once few switches are undecided (k_tail takes those), or past
// the wave cap (k_tail reports that).
__global__ void k_wave_register(RoundArgs a) {
  dep_launch();
  dep_wait();
  const uint32_t cur = a.ctl->cur, wave = a.ctl->wave_next;
  const uint32_t n = a.ctl->pending[cur];
  if (n <= kSoloPending || wave > wave_cap(a)) return;
  const uint32_t *in = cur ? a.list1 : a.list0;
  for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
    const uint32_t k = in[idx];
    const uint2 s = switch_entries(a, k);
    if (s.x != kTrivial) atomicMin(&a.dep[s.x].y, k);
    if (s.y != kTrivial) atomicMin(&a.dep[s.y].y, k);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.ctl->pending[cur ^ 1] = 0;
    if (wave < kWaveHist) a.st->last_pending[wave] = n;
  }
}

// Decision of the same wave: legal, illegal (dropping it as an inserter),
// or undecided again (appended to the next wave's list).  The last CTA to
// finish moves the wave number on and switches lists.
__global__ void k_wave_decide(RoundArgs a) {
  __shared__ bool last;
  dep_launch();
  dep_wait();
  const uint32_t cur = a.ctl->cur, wave = a.ctl->wave_next;
  const uint32_t n = a.ctl->pending[cur];
  const uint32_t active = min(gridDim.x, (n + blockDim.x - 1) / blockDim.x);  // CTAs with a switch
  if (n <= kSoloPending || blockIdx.x >= active || wave > wave_cap(a)) return;
  Tally t;
  ChainCount cc;
  const uint32_t *in = cur ? a.list1 : a.list0;
  uint32_t *out = cur ? a.list0 : a.list1;
  for (uint32_t base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
    const uint32_t idx = base + threadIdx.x;
    bool wait = false;
    uint32_t k = 0;
    if (idx < n) {
      k = in[idx];
      const uint2 s = switch_entries(a, k);
      const int r3 = check_target(a, k, s.x, wave);
      const int r4 = check_target(a, k, s.y, wave);
      if (r3 == kBad || r4 == kBad) {
        a.status[k] = (wave << 2) | kIllegal;
        drop_inserter(a, k, s);
        ++t.rej_exists;
      } else if (r3 == kWait || r4 == kWait) {
        wait = true;
      } else {
        a.status[k] = (wave << 2) | kLegal;
        ++t.accepted;
        count_accepted(a, cc, a.owner_switch[k]);
      }
    }
    append_if(wait, k, out, &a.ctl->pending[cur ^ 1]);
  }
  flush_tally(a, t);
  flush_count(a, cc);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&a.ctl->wave_blocks, 1u) == active - 1;
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    a.ctl->wave_blocks = 0;
    a.ctl->cur = cur ^ 1;
    a.ctl->wave_next = wave + 1;
    a.ctl->wide += 1;
  }
}

// End of a pool round: wave telemetry, statistics, and the pool's round
// counter.  Called by every thread of a CTA of 256 or more: each word is one
// warp's, so that their loads are in flight together (by one thread, one after
// another, they took k_tail 5 of its 7.5 us).
__device__ __forceinline__ void close_round(const RoundArgs &a, uint32_t wave) {
  const uint32_t waves = a.any_work ? wave - 1 : 0, tid = threadIdx.x;
  for (uint32_t w = wave + tid; w < kWaveHist; w += blockDim.x) a.st->last_pending[w] = 0;
  if (tid & 31u) return;
  switch (tid >> 5) {
    case 0:
      a.ctl->pool_round += 1;
      break;
    case 1:
      a.ctl->waves = waves;
      a.st->last_pending[1] = a.switch_hw;
      break;
    case 2:
      if (a.any_work) a.st->waves_total += waves;
      break;
    case 3:
      if (a.any_work && waves > a.st->waves_max) a.st->waves_max = waves;
      break;
    case 4:
      if (a.any_work) a.st->wave_hist[waves < kWaveHist ? waves : kWaveHist - 1] += 1;
      break;
    case 5:
      a.st->overflow_tuples += a.ctl->ovf_count;
      break;
    default:
      break;
  }
}

// The remaining waves, on one CTA: from a list as the pairs of wave kernels do
// while many switches are undecided (waves that the pool's rounds have not
// needed before), then solo_waves.  The kernel also closes the pool round (the
// round counter every chain derives its own round number from).
__global__ void __launch_bounds__(1024) k_tail(RoundArgs a) {
  __shared__ uint32_t s_n;
  dep_launch();
  dep_wait();
  Tally t;
  ChainCount cc;
  uint32_t cur = a.ctl->cur, wave = a.ctl->wave_next, prev_n = a.switch_hw + 1;
  volatile uint32_t *pend = a.ctl->pending;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_n = pend[cur];
    __syncthreads();
    const uint32_t n = s_n;
    if (n <= kSoloPending) {
      if (n) wave = solo_waves<1024>(a, cur ? a.list1 : a.list0, n, wave);
      break;
    }
    if (wave > wave_cap(a)) {
      if (threadIdx.x == 0) atomicOr(&a.ctl->err, kErrWaveCap);
      break;
    }
    if (n >= prev_n) {  // no switch was decided in the last wave: impossible
      if (threadIdx.x == 0) atomicOr(&a.ctl->err, kErrNoProgress);
      break;
    }
    prev_n = n;
    const uint32_t *in = cur ? a.list1 : a.list0;
    uint32_t *out = cur ? a.list0 : a.list1;
    for (uint32_t idx = threadIdx.x; idx < n; idx += blockDim.x) {
      const uint32_t k = in[idx];
      const uint2 s = switch_entries(a, k);
      if (s.x != kTrivial) atomicMin(&a.dep[s.x].y, k);
      if (s.y != kTrivial) atomicMin(&a.dep[s.y].y, k);
    }
    if (threadIdx.x == 0) {
      pend[cur ^ 1] = 0;
      if (wave < kWaveHist) a.st->last_pending[wave] = n;
    }
    __syncthreads();
    for (uint32_t base = 0; base < n; base += blockDim.x) {
      const uint32_t idx = base + threadIdx.x;
      bool wait = false;
      uint32_t k = 0;
      if (idx < n) {
        k = in[idx];
        const uint2 s = switch_entries(a, k);
        const int r3 = check_target(a, k, s.x, wave);
        const int r4 = check_target(a, k, s.y, wave);
        if (r3 == kBad || r4 == kBad) {
          a.status[k] = (wave << 2) | kIllegal;
          drop_inserter(a, k, s);
          ++t.rej_exists;
        } else if (r3 == kWait || r4 == kWait) {
          wait = true;
        } else {
          a.status[k] = (wave << 2) | kLegal;
          ++t.accepted;
          count_accepted(a, cc, a.owner_switch[k]);
        }
      }
      append_if(wait, k, out, (uint32_t *)&pend[cur ^ 1]);
    }
    cur ^= 1;
    ++wave;
    if (threadIdx.x == 0) a.ctl->wide += 1;
  }
  if (prev_n <= a.switch_hw) {  // some waves ran here
    flush_tally(a, t);
    flush_count(a, cc);
  }
  close_round(a, wave);
}

// ---------------------------------------------------------------- one-launch round

// Grid-wide barrier of a cooperative launch (every CTA resident).  Arrivals
// are counted on one monotonic counter: the CTA's thread 0 adds one with
// release-acquire semantics and polls (acquire) until every CTA has arrived
// at this barrier, i.e. the count has reached `target`, which every thread
// advances by the CTA count per barrier.  With the CTA barriers on both
// sides, every write before the barrier is visible after it.  The wait is
// bounded (kGridWaitPolls, each an access to L2): a CTA that gives up sets kErrGridSync and
// returns false, and its caller leaves the kernel; the other CTAs see the
// error bit while they wait and leave too.
__device__ __forceinline__ bool grid_sync(Counters *ctl, unsigned long long &target) {
  __shared__ uint32_t ok;
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long v;
    asm volatile("atom.add.acq_rel.gpu.u64 %0, [%1], 1;" : "=l"(v) : "l"(&ctl->gbar_arrived) : "memory");
    ++v;
    uint32_t it = 0;
    while (v < target && it < kGridWaitPolls) {
      if (*(volatile uint32_t *)&ctl->err & kErrGridSync) break;
      asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(&ctl->gbar_arrived) : "memory");
      ++it;
    }
    ok = v >= target;
    if (!ok) atomicOr(&ctl->err, kErrGridSync);
  }
  __syncthreads();
  return ok != 0;
}

// Exclusive scan of n counters (each clamped to `clamp`) by the calling CTA:
// off[b] (and copy[b], if given) receives the sum of the counters before b.
// Returns the total.  Every thread of the CTA calls it.
__device__ __forceinline__ uint32_t cta_scan_full(const uint32_t *count, uint32_t *off, uint32_t *copy, uint32_t n,
                                                  uint32_t clamp) {
  __shared__ uint32_t wsum[32];
  __shared__ uint32_t total;
  const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t per = (n + nt - 1) / nt;
  const uint32_t beg = min(tid * per, n), end = min(beg + per, n);
  uint32_t sum = 0;
  for (uint32_t b = beg; b < end; ++b) sum += min(count[b], clamp);
  uint32_t incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= (uint32_t)d) incl += v;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t t = lane < nt / 32 ? wsum[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= (uint32_t)d) t += v;
    }
    if (lane < nt / 32) wsum[lane] = t;
    if (lane == 31) total = t;
  }
  __syncthreads();
  uint32_t run = incl - sum + (warp ? wsum[warp - 1] : 0);
  for (uint32_t b = beg; b < end; ++b) {
    const uint32_t c = min(count[b], clamp);
    off[b] = run;
    if (copy) copy[b] = run;
    run += c;
  }
  const uint32_t tot = total;
  __syncthreads();
  return tot;
}

// The whole round of a pool in one cooperative launch of kFusedThreads-thread
// CTAs: the same stages as the multi-kernel round, in the same order, each
// spread over the launch's CTAs, with a grid barrier where the multi-kernel
// round has a kernel boundary.  The offset scans run on CTA 0 (the pools this
// launch is for have few buckets and partitions), and the waves after the
// first repeat register / decide until no switch is undecided, on CTA 0 alone
// once they are few.  The shared memory holds the sort's arrays and, later, the
// grouping table.  What bounds it: a grid barrier is about 1.5 us, a stage of a
// small chain a few dependent accesses to L2.  The arrays a round counts in
// are cleared by the round before (ctl->clean; the first round of a call
// clears its own), the straddling pairs are built in the sort and the last
// waves take no grid barriers: five barriers a round for a chain of 10,000
// edges where there were 13 to 17 (53 -> 44 us a round on 32 CTAs).
__global__ void __launch_bounds__(kFusedThreads, 1) k_round_fused(RoundArgs a) {
  extern __shared__ __align__(128) uint4 fused_dyn[];
  const uint32_t tid = threadIdx.x;
  const uint32_t gtid = blockIdx.x * blockDim.x + tid, nth = gridDim.x * blockDim.x;
  Counters *const ctl = a.ctl;
  // an earlier round of this call gave up at a barrier, which may have left
  // the barrier's counter behind: run nothing (every CTA reads the same
  // value, since no CTA can set the bit before all have passed the first
  // barrier below)
  if (*(volatile uint32_t *)&ctl->err & kErrGridSync) return;
  // the barrier count this launch starts from: earlier launches (all of this
  // CTA count) left it at a multiple of the CTA count, and fewer than that
  // many arrivals of this launch can precede this read
  __shared__ unsigned long long start_count;
  if (tid == 0) {
    const unsigned long long v = *(volatile unsigned long long *)&ctl->gbar_arrived;
    start_count = v / gridDim.x * gridDim.x;
  }
  __syncthreads();
  unsigned long long target = start_count;
  if (!*(volatile uint32_t *)&ctl->clean) {
    clear_arrays(a);
    for (uint32_t b = gtid; b < a.bucket_hw; b += nth) a.bnd[b] = 0;
    if (gtid == 0) clear_counters(ctl);
    if (!grid_sync(ctl, target)) return;
  }
  uint32_t wave = 2;
  if (a.any_work) {
    if (a.any_exact) {
      lazy_count_body(a);
      if (!grid_sync(ctl, target)) return;
    }
    permute_body(a);
    proxy_fence();  // the buckets' records are copied by the TMA engine
    if (!grid_sync(ctl, target)) return;
    if (!a.fused_local_offsets) {
      if (blockIdx.x == 0) {  // bucket offsets: full offsets in poff, zero block offsets
        cta_scan_full(a.pcount, a.poff, nullptr, a.bucket_hw, 1u << a.bucket_log2);
        for (uint32_t j = tid; j <= (a.bucket_hw + 1023) / 1024; j += blockDim.x) a.pblk[j] = 0;
      }
      if (!grid_sync(ctl, target)) return;
    }
    {
      // laid out for the pool's bucket room (the region has room for the largest)
      unsigned char *base = reinterpret_cast<unsigned char *>(fused_dyn);
      const size_t room = size_t(1) << a.bucket_log2;
      SortSmem sm;
      sm.srec = reinterpret_cast<uint4 *>(base);
      sm.hist = reinterpret_cast<uint32_t *>(base + sizeof(uint4) * room);
      sm.sidx = reinterpret_cast<uint16_t *>(sm.hist + room);
      sm.warp_tot = reinterpret_cast<uint32_t *>(sm.sidx + room);
      sm.bar = reinterpret_cast<unsigned long long *>(sm.warp_tot + 32);
      __shared__ uint2 meet[kMeets];
      __shared__ uint32_t meets;
      sm.meet = meet;
      sm.meets = &meets;
      if (tid == 0) {
        mbar_init(sm.bar, 1);
        meets = 0;
      }
      __syncthreads();
      uint32_t parity = 0;
      const bool local = a.fused_local_offsets != 0;
      for (uint32_t b = blockIdx.x; b < a.bucket_hw; b += gridDim.x) {
        if (!(a.bucket_log2 == kBucketLog2Small
                  ? sort_bucket<kFusedThreads, kBucketLog2Small, true>(a, b, sm, parity, local)
                  : sort_bucket<kFusedThreads, kBucketLog2Large, true>(a, b, sm, parity, local)))
          return;
        if (meets > kMeets - 2) meet_pairs(a, sm);  // (the same for every thread: read after a barrier)
      }
      meet_pairs(a, sm);
      if (tid == 0) mbar_inval(sm.bar);  // the grouping table takes these bytes next
    }
    if (!grid_sync(ctl, target)) return;
    const uint32_t npair = a.slot_hw >> 1;
    for (uint32_t base = blockIdx.x * 2 * blockDim.x; base < npair; base += 2 * nth) {
      const uint32_t x = base + tid;
      if (x < npair) source_pairs(a, x, x + blockDim.x, npair);
    }
    if (!grid_sync(ctl, target)) return;
    if (*(volatile uint32_t *)&ctl->ovf_count) {
      overflow_count_body(a);
      if (!grid_sync(ctl, target)) return;
      if (blockIdx.x == 0) {  // overflow offsets: full offsets in ooff, zero block offsets, the total last
        const uint32_t tot = cta_scan_full(a.ocount, a.ooff, a.ocursor, a.part_hw, 0xFFFFFFFFu);
        const uint32_t nblk = (a.part_hw + 1023) >> 10;
        for (uint32_t j = tid; j < nblk; j += blockDim.x) a.oblk[j] = 0;
        if (tid == 0) a.oblk[nblk] = tot;
      }
      if (!grid_sync(ctl, target)) return;
      overflow_scatter_body(a);
      if (!grid_sync(ctl, target)) return;
    }
    group_body<kFusedThreads, 2048 / kFusedThreads>(a);
    if (!grid_sync(ctl, target)) return;
    wave1_body(a);
    // what the stages so far counted in is not needed any more
    clear_arrays(a);
    for (uint32_t b = gtid; b < a.bucket_hw; b += nth) a.bnd[b] = 0;
    if (!grid_sync(ctl, target)) return;
    // waves 2, 3, ...: undecided switches re-register as inserters, then
    // decide; from kSoloPending undecided switches on by CTA 0 alone
    Tally t;
    ChainCount cc;
    uint32_t cur = 0, prev_n = a.switch_hw + 1;
    volatile uint32_t *pend = ctl->pending;
    for (;;) {
      const uint32_t n = pend[cur];  // the same for every thread: read after a barrier
      if (n <= kSoloPending) {
        if (n && blockIdx.x == 0) wave = solo_waves<kFusedThreads>(a, cur ? a.list1 : a.list0, n, wave);
        break;
      }
      if (wave > wave_cap(a)) {
        if (gtid == 0) atomicOr(&ctl->err, kErrWaveCap);
        break;
      }
      if (n >= prev_n) {  // no switch was decided in the last wave: impossible
        if (gtid == 0) atomicOr(&ctl->err, kErrNoProgress);
        break;
      }
      prev_n = n;
      const uint32_t *in = cur ? a.list1 : a.list0;
      uint32_t *out = cur ? a.list0 : a.list1;
      for (uint32_t idx = gtid; idx < n; idx += nth) {
        const uint32_t k = __ldcg(&in[idx]);
        const uint2 sv = switch_entries(a, k);
        if (sv.x != kTrivial) atomicMin(&a.dep[sv.x].y, k);
        if (sv.y != kTrivial) atomicMin(&a.dep[sv.y].y, k);
      }
      if (gtid == 0) {
        pend[cur ^ 1] = 0;
        if (wave < kWaveHist) a.st->last_pending[wave] = n;
      }
      if (!grid_sync(ctl, target)) return;
      for (uint32_t base = blockIdx.x * blockDim.x; base < n; base += nth) {
        const uint32_t idx = base + tid;
        bool wait = false;
        uint32_t k = 0;
        if (idx < n) {
          k = __ldcg(&in[idx]);
          const uint2 sv = switch_entries(a, k);
          const int r3 = check_target(a, k, sv.x, wave);
          const int r4 = check_target(a, k, sv.y, wave);
          if (r3 == kBad || r4 == kBad) {
            a.status[k] = (wave << 2) | kIllegal;
            drop_inserter(a, k, sv);
            ++t.rej_exists;
          } else if (r3 == kWait || r4 == kWait) {
            wait = true;
          } else {
            a.status[k] = (wave << 2) | kLegal;
            ++t.accepted;
            count_accepted(a, cc, a.owner_switch[k]);
          }
        }
        append_if(wait, k, out, (uint32_t *)&pend[cur ^ 1]);
      }
      if (!grid_sync(ctl, target)) return;
      cur ^= 1;
      ++wave;
    }
    flush_tally(a, t);
    flush_count(a, cc);
  }
  if (blockIdx.x == 0) {
    __syncthreads();  // CTA 0's threads have read the counters
    close_round(a, wave);
    __syncthreads();
    if (tid == 0) {
      const uint32_t waves = ctl->waves;
      clear_counters(ctl);
      ctl->waves = waves;  // (the host reads it)
      ctl->clean = a.any_work;
    }
  }
}

// ---------------------------------------------------------------- state in / out

__global__ void k_load_chain(RoundArgs a, ChainDesc ch, const unsigned long long *E) {
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < ch.m; s += gridDim.x * blockDim.x) {
    a.cpos[ch.slot_base + s] = s;
    a.cedge[ch.slot_base + s] = E[s];
  }
}

// A chain's list by position, with its last round's legal switches applied
// (status; null if there is nothing to apply).  The host says so: with the round
// counter read first, every access would wait for it (11.3 us a call for a
// small chain, with launch and synchronisation; 10.9 so).
__global__ void k_store_chain(const uint2 *cpos, const ulonglong2 *cedge, const uint32_t *status, uint32_t m,
                              unsigned long long *E) {
  const uint32_t npair = (m + 1) >> 1, L = m >> 1;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < npair; k += gridDim.x * blockDim.x) {
    if (k < L) {
      const uint32_t st = status ? __ldcs(&status[k]) : 0u;
      const uint2 ij = __ldcs(&cpos[k]);
      const ulonglong2 ee = __ldcs(&cedge[k]);
      unsigned long long e1 = ee.x, e2 = ee.y;
      if ((st & 3u) == kLegal) tau(ij.x, ij.y, ee.x, ee.y, e1, e2);
      E[ij.x] = e1;
      E[ij.y] = e2;
    } else {  // odd m: the last slot has no partner
      E[reinterpret_cast<const uint32_t *>(cpos)[2 * k]] = reinterpret_cast<const unsigned long long *>(cedge)[2 * k];
    }
  }
}

// A large list by position in two passes (a list that outgrows L2 written
// directly is one 32-byte sector read, changed and written per edge: 5.7 ms for
// 1.34e8 edges, 0.42 for 1.7e7; now 3.5 and 0.32 ms; at 8.4e6 edges the direct
// pass takes 0.07 against 0.19).  Positions are binned by their top bits, 2^bin_log2 of them a
// bin (at most kStoreBins bins): a bin's records, {position, 0, edge lo, edge
// hi}, fill exactly its range of `rec` (every position occurs once), each CTA
// taking a run of every bin with one cursor atomic; the second pass writes the
// records of one bin after another, whose part of the list stays in L2 until
// its lines are full.  Bound by the scattered stores of the first pass (2.6 of
// 3.5 ms, one 16-byte store an edge), not by memory (36 bytes an edge read, 24
// written).
constexpr int kStoreThreads = 512, kStorePairs = 4;
constexpr uint32_t kStoreBins = 1024;
constexpr uint32_t kStoreStride = 16;           // words between the bins' cursors (packed, they contend for L2 lines)
constexpr uint32_t kStoreMinEdges = 1u << 24;  // 128 MB of list, as much as L2 holds

__global__ void __launch_bounds__(kStoreThreads, 3) k_store_bin(RoundArgs a, ChainDesc ch, uint32_t bin_log2, uint4 *rec,
                                                             uint32_t *cursor) {
  __shared__ uint32_t cnt[kStoreBins];
  const bool apply = chain_apply(ch, a.ctl->pool_round);
  const uint32_t tid = threadIdx.x, npair = (ch.m + 1) >> 1;
  const uint32_t k0 = blockIdx.x * (kStoreThreads * kStorePairs) + tid;
  for (uint32_t b = tid; b < kStoreBins; b += kStoreThreads) cnt[b] = 0;
  __syncthreads();
  uint32_t pos[2 * kStorePairs], rank[2 * kStorePairs];
  unsigned long long e[2 * kStorePairs];
#pragma unroll
  for (int u = 0; u < kStorePairs; ++u) {
    const uint32_t k = k0 + u * kStoreThreads;
    pos[2 * u] = pos[2 * u + 1] = kNoChain;
    if (k >= npair) continue;
    const uint32_t s0 = ch.slot_base + 2 * k;  // (even)
    if (2 * k + 1 < ch.m) {
      const uint2 ij = __ldcs(reinterpret_cast<const uint2 *>(a.cpos + s0));
      const ulonglong2 ee = __ldcs(reinterpret_cast<const ulonglong2 *>(a.cedge + s0));
      e[2 * u] = ee.x;
      e[2 * u + 1] = ee.y;
      apply_last(a, ch, apply, k, ij.x, ij.y, e[2 * u], e[2 * u + 1]);
      pos[2 * u] = ij.x;
      pos[2 * u + 1] = ij.y;
    } else {
      pos[2 * u] = a.cpos[s0];
      e[2 * u] = a.cedge[s0];
    }
  }
#pragma unroll
  for (int u = 0; u < 2 * kStorePairs; ++u)
    if (pos[u] != kNoChain) rank[u] = atomicAdd(&cnt[pos[u] >> bin_log2], 1u);
  __syncthreads();
  for (uint32_t b = tid; b < kStoreBins; b += kStoreThreads) {
    const uint32_t n = cnt[b];
    if (n) cnt[b] = (b << bin_log2) + atomicAdd(&cursor[b * kStoreStride], n);
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 2 * kStorePairs; ++u)
    if (pos[u] != kNoChain) {
      const uint32_t at = cnt[pos[u] >> bin_log2] + rank[u];
      if (at < ch.m) rec[at] = make_uint4(pos[u], 0u, (uint32_t)e[u], (uint32_t)(e[u] >> 32));
    }
}

__global__ void __launch_bounds__(256) k_store_out(const uint4 *rec, uint32_t m, unsigned long long *E) {
  const uint32_t t0 = blockIdx.x * 1024 + threadIdx.x;
  uint4 r[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (t0 + u * 256 < m) r[u] = __ldcs(&rec[t0 + u * 256]);
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (t0 + u * 256 < m && r[u].x < m) E[r[u].x] = ((unsigned long long)r[u].w << 32) | r[u].z;
}

// ParES: the lists of the chains with a job, by position, with the last
// round's legal switches applied, and their edge sets; and back into their slots
// (slot s holds position s, nothing pending).  An edge goes into the set on the
// way to the list, whose entry then has its slot at once: with a pass of its own
// that read and wrote the list again, a call of one switch took 1126 us on 1.6e7
// edges and 58 us on 9,000, now 1085 and 54.
__global__ void k_es_store(RoundArgs a, const EsJob *jobs, const uint32_t *job_of, uint32_t *err) {
  const unsigned long long R = a.ctl->pool_round;
  const uint32_t npair = (a.slot_hw + 1) >> 1;
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < npair; x += gridDim.x * blockDim.x) {
    const uint32_t s0 = 2 * x;
    const uint32_t c = a.owner_slot[s0];
    if (c == kNoChain || job_of[c] == kNoChain) continue;
    const ChainDesc ch = a.chains[c];
    const EsJob &jb = jobs[job_of[c]];
    uint4 *const E = jb.E;
    unsigned long long *const H = jb.H;
    const uint32_t mask = (uint32_t)((1ull << jb.hlog2) - 1);
    auto put = [=](uint32_t pos, unsigned long long e) {
      uint32_t at = 0, tomb;
      if (H && (at = hset_insert(H, mask, e, hash32(e) & mask, &tomb)) == kNil) {
        atomicOr(err, kErrTableFull);
        at = 0;
      }
      E[pos] = make_uint4((uint32_t)e, (uint32_t)(e >> 32), at, 0u);
    };
    const uint32_t ls = s0 - ch.slot_base;
    if (ls + 1 < ch.m) {
      const uint32_t i = a.cpos[s0], j = a.cpos[s0 + 1];
      unsigned long long e1 = a.cedge[s0], e2 = a.cedge[s0 + 1];
      apply_last(a, ch, chain_apply(ch, R), ls >> 1, i, j, e1, e2);
      put(i, e1);
      put(j, e2);
    } else {
      put(a.cpos[s0], a.cedge[s0]);
    }
  }
}

__global__ void k_es_load(RoundArgs a, const EsJob *jobs, const uint32_t *job_of) {
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < a.slot_hw; s += gridDim.x * blockDim.x) {
    const uint32_t c = a.owner_slot[s];
    if (c == kNoChain || job_of[c] == kNoChain) continue;
    const ChainDesc ch = a.chains[c];
    const uint32_t ls = s - ch.slot_base;
    a.cpos[s] = ls;
    a.cedge[s] = *reinterpret_cast<const unsigned long long *>(&jobs[job_of[c]].E[ls]);
    if ((ls & 1u) == 0 && (ls >> 1) < ch.L) a.status[ch.switch_base + (ls >> 1)] = 0;  // nothing pending
  }
}

__global__ void k_fill_ranges(FillRanges r, uint32_t v) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < r.n[j]; i += gridDim.x * blockDim.x) r.p[j][i] = v;
}

// ---------------------------------------------------------------- create-time checks

__global__ void k_fill_u64(unsigned long long *p, unsigned long long n, unsigned long long v) {
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x)
    p[i] = v;
}

__global__ void k_duplicates(const unsigned long long *E, uint32_t m, unsigned long long *set, unsigned long long cap,
                             uint32_t *flags) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const unsigned long long key = E[i];
    unsigned long long s = __umul64hi(mix64(key), cap);
    bool placed = false;
    for (unsigned long long n = 0; n < cap && !placed; ++n) {
      const unsigned long long prev = atomicCAS(&set[s], kEmptyKey, key);
      if (prev == kEmptyKey) placed = true;
      else if (prev == key) {
        atomicOr(flags, kFlagMulti);
        placed = true;
      } else if (++s == cap) {
        s = 0;
      }
    }
    if (!placed) atomicOr(flags, kFlagTableFull);
  }
}

// Degree fingerprint term of one endpoint: the list's fingerprint is the sum
// (mod 2^64) over its edges of both endpoints' terms, a function of the
// multiset of endpoints, i.e. of the degree sequence, which a switch keeps.
__device__ __forceinline__ unsigned long long endpoint_term(uint32_t v) {
  return mix64(0x9E3779B97F4A7C15ull + v);
}

// The caller's list made canonical in place: flags for a loop or an id out of
// range, the largest id, and the degree fingerprint.
__global__ void k_canonicalise(unsigned long long *E, uint32_t m, unsigned long long n_bound, uint32_t *flags,
                               uint32_t *max_id, unsigned long long *fp) {
  uint32_t f = 0, mx = 0;
  unsigned long long sum = 0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const unsigned long long e = E[i];
    const uint32_t x = (uint32_t)(e >> 32), y = (uint32_t)e;
    if (x == y) f |= kFlagLoop;
    if (n_bound && (x >= n_bound || y >= n_bound)) f |= kFlagRange;
    mx = max(mx, max(x, y));
    sum += endpoint_term(x) + endpoint_term(y);
    E[i] = pack_edge(x, y);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, off);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) {
    if (sum) atomicAdd(fp, sum);
    if (mx) atomicMax(max_id, mx);
  }
  if (f) atomicOr(flags, f);
}

// Debug check of a position-order list: every entry canonical and
// loop-free (u < v) and in range (v < n, if n), and its degree fingerprint.
__global__ void k_list_check(const unsigned long long *E, uint32_t m, unsigned long long n, uint32_t *flags,
                             unsigned long long *fp) {
  uint32_t f = 0;
  unsigned long long sum = 0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const unsigned long long e = E[i];
    const uint32_t u = (uint32_t)(e >> 32), v = (uint32_t)e;
    if (!(u < v)) f |= kFlagLoop;
    if (n && v >= n) f |= kFlagRange;
    sum += endpoint_term(u) + endpoint_term(v);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, off);
  if ((threadIdx.x & 31) == 0 && sum) atomicAdd(fp, sum);
  if (f) atomicOr(flags, f);
}

inline int grid_for(unsigned long long work, int threads, int num_sms, int per_sm) {
  unsigned long long g = (work + threads - 1) / threads;
  const unsigned long long lim = (unsigned long long)num_sms * per_sm;
  if (g > lim) g = lim;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

size_t group_smem_bytes(uint32_t group_log2) { return ((size_t)kGroupSlotBytes << group_log2) + 8 * kGroupWords; }

cudaError_t prepare_kernels(uint32_t group_log2, int num_sms, LaunchShapes *shapes) {
  // opt in to the largest table any pool may use, so that pools with
  // different table sizes never lower each other's limit
  cudaError_t e = cudaFuncSetAttribute(k_group, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)group_smem_bytes(kMaxGroupLog2));
  if (e != cudaSuccess) return e;
  auto resident = [num_sms](const void *fn, int threads, size_t smem, uint32_t *grid) {
    int per_sm = 0;
    const cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    *grid = (uint32_t)(num_sms * (per_sm > 0 ? per_sm : 1));
    return r;
  };
  e = resident((const void *)k_group, kGroupThreads, group_smem_bytes(group_log2), &shapes->group);
  return e;
}



size_t fused_smem_bytes(uint32_t group_log2) {
  return std::max(sort_smem_bytes(kBucketLog2Large), group_smem_bytes(group_log2));
}

cudaError_t prepare_fused(uint32_t group_log2, int num_sms, uint32_t *max_ctas) {
  cudaError_t e = cudaFuncSetAttribute(k_round_fused, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)fused_smem_bytes(kMaxGroupLog2));
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_round_fused, kFusedThreads,
                                                    fused_smem_bytes(group_log2));
  *max_ctas = (uint32_t)(num_sms * (per_sm > 0 ? per_sm : 0));
  return e;
}

cudaError_t launch_round_fused(const RoundArgs &a, cudaStream_t s, uint32_t ctas) {
  RoundArgs arg = a;
  void *params[] = {&arg};
  return cudaLaunchCooperativeKernel((const void *)k_round_fused, dim3(ctas), dim3(kFusedThreads), params,
                                     fused_smem_bytes(a.group_log2), s);
}

cudaError_t launch_round(const RoundArgs &a, cudaStream_t s, int num_sms, cudaEvent_t *ev, bool after_round,
                         uint32_t *launches) {
  // ev (optional) receives kNumStages + 1 stage boundaries; stages that do
  // not run (no chain with two edges) still get both events (zero duration)
  auto mark = [&](int stage) {
    if (ev) cudaEventRecord(ev[stage], s);
  };
  uint32_t n = 0;
  const bool work = a.any_work != 0;
  // programmatic dependent launch, but for the first kernel unless the one
  // before it is a round's too (what came before may not wait as they do), and
  // not between the events of stage timing
  cudaError_t bad = cudaSuccess;
  auto go = [&](auto fn, uint32_t ctas, uint32_t threads, size_t smem = 0, auto... more) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = !ev && (n > 0 || after_round) ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, a, more...);
    if (e != cudaSuccess && bad == cudaSuccess) bad = e;
    ++n;
  };
  mark(kStageClear);
  const uint32_t clear = max(max(max(a.bucket_hw, a.part_hw), a.tcount_hw), work ? a.tfilter_mask >> 7 : 0u);
  go(k_clear, grid_for(clear, 256, num_sms, 4), 256);
  if (work && a.any_exact) go(k_lazy_count, grid_for(a.switch_hw, 256, num_sms, 8), 256);
  mark(kStagePermute);
  if (work && a.agg_chain != kNoChain) {
    if (a.agg_pairs <= (uint32_t)num_sms * 512) {  // few pairs: spread over the SMs
      go(k_permute_agg<256, 1>, (a.agg_pairs + 255) / 256, 256, 0, 256u);
    } else {  // more records per cursor atomic; one CTA per SM at a time, so full waves of equal CTAs
      const uint32_t wave = (uint32_t)num_sms * 2048, ctas = (a.agg_pairs + wave - 1) / wave * num_sms;
      const uint32_t tile = (a.agg_pairs + ctas - 1) / ctas;
      go(k_permute_agg<1024, 2>, (a.agg_pairs + tile - 1) / tile, 1024, 0, tile);
    }
  } else if (work) {
    go(k_permute, a.permute_ctas, 256);
  }
  mark(kStageScanPerm);
  if (work) {
    go(k_scan_perm, a.bucket_hw ? (a.bucket_hw + 1023) / 1024 : 1, 1024);
    go(k_scan_blocks, 1, 1024);
  }
  mark(kStageSortPair);
  if (work) {
    if (a.bucket_log2 == kBucketLog2Small)
      go(k_sortpair<kBucketLog2Small, 7>, a.bucket_hw, 1 << (kBucketLog2Small - 3));
    else
      go(k_sortpair<kBucketLog2Large, 4>, a.bucket_hw, 1 << (kBucketLog2Large - 3));
  }
  mark(kStageBoundary);
  if (work) go(k_boundary, grid_for(a.bucket_hw, 256, num_sms, 2), 256);
  mark(kStageSources);
  if (work) go(k_sources, a.sources_ctas, 256);
  mark(kStageOverflow);
  if (work) {
    const int g = grid_for(a.ovf_cap, 256, num_sms, 2);
    go(k_overflow_count, g, 256);
    go(k_overflow_scan_blocks, (a.part_hw + 1023) / 1024 ? (a.part_hw + 1023) / 1024 : 1, 1024);
    go(k_overflow_scan_top, 1, 1024);
    go(k_overflow_scatter, g, 256);
  }
  mark(kStageGroup);
  if (work) {
    const uint32_t ctas = a.group_grid ? a.group_grid : (uint32_t)num_sms;
    go(k_group, ctas < a.part_hw ? ctas : a.part_hw, kGroupThreads, group_smem_bytes(a.group_log2));
  }
  mark(kStageWave1);
  if (work) go(k_wave1, grid_for(a.switch_hw, 256, num_sms, 16), 256);
  mark(kStageWaves);
  if (work) {
    for (uint32_t w = 0; w < a.wave_kernels && w < kMaxWaveKernels; ++w) {
      go(k_wave_register, num_sms * 4, 256);
      go(k_wave_decide, num_sms * 4, 256);
    }
  }
  mark(kStageTail);
  go(k_tail, 1, 1024);
  mark(kNumStages);
  if (launches) *launches += n;
  const cudaError_t last = cudaGetLastError();
  return bad != cudaSuccess ? bad : last;
}

cudaError_t launch_load_chain(const RoundArgs &a, const ChainDesc &ch, const unsigned long long *E, cudaStream_t s,
                              int num_sms) {
  if (ch.m == 0) return cudaSuccess;
  k_load_chain<<<grid_for(ch.m, 256, num_sms, 8), 256, 0, s>>>(a, ch, E);
  return cudaGetLastError();
}

cudaError_t launch_store_chain(const RoundArgs &a, const ChainDesc &ch, uint64_t pool_round, unsigned long long *E,
                               cudaStream_t s, int num_sms) {
  if (ch.m == 0) return cudaSuccess;
  if (ch.m < kStoreMinEdges) {
    // (slot ranges start on even slots)
    k_store_chain<<<grid_for((ch.m + 1) / 2, 256, num_sms, 8), 256, 0, s>>>(
        reinterpret_cast<const uint2 *>(a.cpos + ch.slot_base),
        reinterpret_cast<const ulonglong2 *>(a.cedge + ch.slot_base),
        pool_round > ch.added ? a.status + ch.switch_base : nullptr, ch.m, E);
    return cudaGetLastError();
  }
  // between rounds the permutation records and the bucket counts are free (at
  // least 32 bytes and far more than kStoreBins counts for so many edges)
  uint32_t bin_log2 = 17;
  while (((ch.m - 1) >> bin_log2) >= kStoreBins) ++bin_log2;
  const cudaError_t e = cudaMemsetAsync(a.pcount, 0, 4 * kStoreBins * kStoreStride, s);
  if (e != cudaSuccess) return e;
  const uint32_t per = kStoreThreads * kStorePairs, npair = (ch.m + 1) / 2;
  k_store_bin<<<(npair + per - 1) / per, kStoreThreads, 0, s>>>(a, ch, bin_log2, a.prec, a.pcount);
  k_store_out<<<(ch.m + 1023) / 1024, 256, 0, s>>>(a.prec, ch.m, E);
  return cudaGetLastError();
}

cudaError_t launch_es_store(const RoundArgs &a, const EsJob *jobs, const uint32_t *job_of, uint32_t *err,
                            cudaStream_t s, int num_sms) {
  if (a.slot_hw == 0) return cudaSuccess;
  k_es_store<<<grid_for((a.slot_hw + 1) / 2, 256, num_sms, 8), 256, 0, s>>>(a, jobs, job_of, err);
  return cudaGetLastError();
}

cudaError_t launch_es_load(const RoundArgs &a, const EsJob *jobs, const uint32_t *job_of, cudaStream_t s,
                           int num_sms) {
  if (a.slot_hw == 0) return cudaSuccess;
  k_es_load<<<grid_for(a.slot_hw, 256, num_sms, 8), 256, 0, s>>>(a, jobs, job_of);
  return cudaGetLastError();
}

cudaError_t launch_fill_ranges(const FillRanges &r, uint32_t v, cudaStream_t s, int num_sms) {
  const uint32_t most = std::max(std::max(r.n[0], r.n[1]), std::max(r.n[2], r.n[3]));
  if (most == 0) return cudaSuccess;
  k_fill_ranges<<<grid_for(most, 256, num_sms, 8), 256, 0, s>>>(r, v);
  return cudaGetLastError();
}

cudaError_t launch_canonicalise(unsigned long long *E, uint32_t m, unsigned long long n_bound, uint32_t *flags,
                                uint32_t *max_id, unsigned long long *fp, cudaStream_t s, int num_sms) {
  k_canonicalise<<<grid_for(m, 256, num_sms, 8), 256, 0, s>>>(E, m, n_bound, flags, max_id, fp);
  return cudaGetLastError();
}

cudaError_t launch_list_check(const unsigned long long *E, uint32_t m, unsigned long long n, uint32_t *flags,
                              unsigned long long *fp, cudaStream_t s, int num_sms) {
  if (m == 0) return cudaSuccess;
  k_list_check<<<grid_for(m, 256, num_sms, 8), 256, 0, s>>>(E, m, n, flags, fp);
  return cudaGetLastError();
}

cudaError_t launch_duplicate_check(const unsigned long long *E, uint32_t m, unsigned long long *set,
                                   unsigned long long cap, uint32_t *flags, cudaStream_t s, int num_sms) {
  k_fill_u64<<<grid_for(cap, 256, num_sms, 8), 256, 0, s>>>(set, cap, kEmptyKey);
  k_duplicates<<<grid_for(m, 256, num_sms, 8), 256, 0, s>>>(E, m, set, cap, flags);
  return cudaGetLastError();
}

}  // namespace gesmc
