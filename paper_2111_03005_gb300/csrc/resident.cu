// Resident rounds: global switches (Def. 2, performed as Algorithm 1's
// decide / delay waves) of small chains, one CTA per chain, the chain's list
// in shared memory from the first round of a call to the last.
//
// The paper notes that small graphs are the weak case of a parallel global
// switch (too little work per round to pay for its synchronisation) and that
// dedicated base cases would help.  On the GPU a round of the general path
// is a dozen dependent stages spread over the device; for a chain of about
// 10^4 edges their barriers or launches cost more than the work.  Here one
// CTA holds the whole chain: E as one 32-bit word per edge (two 16-bit node
// ids), the permutation, the switch statuses and a hash table of target
// edge ids, all in shared memory, so a round's stages are separated by
// __syncthreads only and nothing goes to global memory between rounds.
//
// Per round (round number r of the chain):
//   1. keys K(i) = Philox4x64-10((i >> 2, r, 0, 0); (seed, 0))[i & 3], the
//      same keys as the general path; a counting sort of the positions into
//      m to 2m buckets by the keys' top bits, then each position's rank in
//      its bucket in (K, i) order: the argsort pi.
//   2. switch k = (pi(2k), pi(2k+1), [pi(2k) < pi(2k+1)]): the outright
//      rejects (laziness, a loop, a shared node) are ILLEGAL before the first
//      wave.  The targets of every other switch set their bits in a hashed
//      bitmap; a bit set twice (two targets, perhaps the same id), or the bit
//      of some edge of E (a source, perhaps the same id), is marked.  A
//      target whose bit is unmarked is in E for no switch and proposed by no
//      other switch: it is free.  A switch whose two targets are free is
//      LEGAL in the first wave and takes no further part.
//   3. the others, the candidates (few: the bitmap has 16 to 32 bits a
//      target), enter their marked targets into a table (linear probing) and
//      register there as inserters (the entry keeps the smallest inserter q);
//      the edges of E that hit a target's
//      bit record the eraser p of their entry, the switch whose slot holds
//      them (the unpaired slot of an odd m erases nothing: the edge stays, p =
//      "never").
//   4. Jacobi waves over the candidates: an undecided switch k decides from
//      the statuses of earlier waves only (a status word carries its wave):
//      ILLEGAL if a target is still there when k runs (erased by a later
//      switch or never, or its eraser failed, or an earlier inserter
//      succeeded), UNDECIDED if that depends on a switch not yet decided, else
//      LEGAL.  Where a switch turned illegal in the last wave, the smallest
//      inserters of the ids with two inserters or more are recomputed from the
//      switches that are not illegal (an id with one inserter is looked at by
//      that one only).
//   5. the legal switches write their targets to their two positions.
// After the last round of the launch the list goes back to the chain's slots
// in position order with nothing pending, as the general path would leave
// it after store and reload.
#include "device_util.cuh"
#include "gesmc_internal.cuh"
#include "resident.cuh"

namespace gesmc {
namespace {

constexpr uint32_t kEmpty32 = 0xFFFFFFFFu;  // no edge packs to this (low id < high id)
constexpr uint32_t kP16None = 0xFFFFu;      // the id is not in E at the round's start
constexpr uint32_t kP16Keep = 0xFFFEu;      // in E, erased by no switch
constexpr uint32_t kQ16None = 0xFFFFu;      // no inserter that is not illegal
constexpr uint32_t kFree = 0xFFFFu;         // no table slot: the target is free

struct ResidentJob {
  const uint32_t *jobs;
  uint32_t rounds;
  uint32_t *round_waves;
  uint32_t *last_pending;
  uint32_t final;
  uint32_t wave_cap;
  // permutations sorted beforehand (null: each CTA sorts its own): round t
  // of job j at pbuf + (t * njobs + j) * pstride, its l (exact laziness) at
  // ebuf[t * njobs + j]; job_base = index of jobs[0] among all jobs
  uint16_t *pbuf;
  uint32_t *ebuf;
  uint32_t pstride, njobs, job_base;
  uint32_t first;  // the first class's launch
};

// Byte offsets of a chain's pieces of shared memory (all grow with m).
struct ResLayout {
  uint32_t scat, perm, status, region, multi, nb_log2, slog2, bytes;
  uint32_t bits_log2;   // the target bitmaps have 2^bits_log2 bits each
  uint32_t lists;       // candidate and source lists (bytes from `region`)
  uint32_t list_slog2;  // largest table (log2 slots) that leaves the lists alone
};

__host__ __device__ inline uint32_t ceil_log2(uint32_t x) {
  uint32_t b = 0;
  while ((1u << b) < x) ++b;
  return b;
}

__host__ __device__ inline uint32_t align16(uint32_t x) { return (x + 15u) & ~15u; }

__host__ __device__ inline ResLayout res_layout(uint32_t m) {
  ResLayout l;
  const uint32_t lg = ceil_log2(m), lb = lg < 6 ? 6u : lg;
  l.nb_log2 = lb;                              // one key per bucket or fewer, at least 64 buckets
  l.slog2 = lg + 1 < 6 ? 6 : (lg + 1 > 14 ? 14 : lg + 1);  // >= 2m slots, at most 2^14 (m targets at most)
  l.scat = align16(4 * m);                     // E: u32 per position
  l.perm = l.scat + align16(2 * m);            // positions by bucket (u16 per slot), later the
                                               // targets' table slots (u32 per switch)
  l.status = l.perm + align16(2 * m);          // pi: u16 per slot
  l.region = l.status + align16(2 * (m / 2));  // status: u16 per switch
  // in the same bytes, one after another: the sort's keys (u32 per position)
  // and bucket counts; the two bitmaps (2^(lb + 4) bits each) and, behind
  // them, the lists (u16 per switch and per slot, below 2^(lb + 2) bytes);
  // the table (u32 key + u32 {p, q} per slot), over the bitmaps only while it
  // has at most 2^(lb - 1) slots, else over the lists too
  l.bits_log2 = lb + 4;
  l.lists = 2u << (l.bits_log2 - 3);
  l.list_slog2 = lb - 1;
  const uint32_t sort_bytes = align16(4 * m) + 4 * (1u << l.nb_log2);
  const uint32_t table_bytes = 8 * (1u << l.slog2);
  const uint32_t list_bytes = l.lists + align16(2 * (m / 2)) + align16(2 * m);
  uint32_t region = sort_bytes > table_bytes ? sort_bytes : table_bytes;
  if (list_bytes > region) region = list_bytes;
  l.multi = l.region + region;
  l.bytes = l.multi + align16((1u << l.slog2) / 8);  // one bit per table slot: two inserters or more
  return l;
}

// Home bit of an id in the target bitmaps.
__device__ __forceinline__ uint32_t bit_of(uint32_t e, uint32_t bits_log2) {
  return (e * 0x9E3779B1u) >> (32 - bits_log2);
}

__device__ __forceinline__ bool bit_set(const uint32_t *map, uint32_t b) { return (map[b >> 5] >> (b & 31)) & 1u; }

__device__ __forceinline__ uint32_t home_slot(uint32_t e, uint32_t slog2) { return (e * 0x9E3779B1u) >> (32 - slog2); }

// Slot of id e in the table (linear probing from its home slot), which e
// takes if it is not there yet; 2^slog2 if the table is full.
__device__ __forceinline__ uint32_t tab_insert(uint32_t *tkey, uint32_t slog2, uint32_t e) {
  const uint32_t mask = (1u << slog2) - 1;
  uint32_t s = home_slot(e, slog2);
  for (uint32_t n = 0; n <= mask; ++n) {
    const uint32_t old = atomicCAS(&tkey[s], kEmpty32, e);
    if (old == kEmpty32 || old == e) return s;
    s = (s + 1) & mask;
  }
  return mask + 1;
}

// Slot of id e, or 2^slog2 if absent (no insertions run meanwhile).
__device__ __forceinline__ uint32_t tab_find(const uint32_t *tkey, uint32_t slog2, uint32_t e) {
  const uint32_t mask = (1u << slog2) - 1;
  uint32_t s = home_slot(e, slog2);
  for (uint32_t n = 0; n <= mask; ++n) {
    const uint32_t cur = tkey[s];
    if (cur == e) return s;
    if (cur == kEmpty32) break;
    s = (s + 1) & mask;
  }
  return mask + 1;
}

// q of an entry (low 16 bits of {p, q}) lowered to k if k is smaller: one
// atomicMin of the whole word, since p (the high half) does not change while
// inserters register (all p are "none" at the first registration, and fixed
// by step 3 before any re-registration).
__device__ __forceinline__ uint32_t tab_qmin(uint32_t *tpq, uint32_t s, uint32_t k) {
  return atomicMin(&tpq[s], (tpq[s] & 0xFFFF0000u) | k);
}

__device__ __forceinline__ bool is_multi(const uint32_t *multi, uint32_t s) { return (multi[s >> 5] >> (s & 31)) & 1u; }

__device__ __forceinline__ bool decided_before(uint32_t st, uint32_t wave) {
  return (st & 3u) != kUndecided && (st >> 2) < wave;
}

// Sum over the threads before this one of `sum` (warp_sums: T / 32 words);
// has one barrier inside.
template <int T>
__device__ __forceinline__ uint32_t block_sum_before(uint32_t sum, uint32_t *warp_sums) {
  const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
  uint32_t x = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
    if ((int)lane >= off) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  // every warp adds up the warps before it
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < wid ? warp_sums[lane] : 0u);
  return before + x - sum;
}

// Exclusive scan of V 16-byte vectors of counters per thread, in place.
template <int T, int V>
__device__ __forceinline__ void vector_scan(uint32_t *v, uint32_t *warp_sums) {
  uint4 *const p = reinterpret_cast<uint4 *>(v) + threadIdx.x * V;
  uint4 c[V];
  uint32_t sum = 0;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    c[i] = p[i];
    sum += c[i].x + c[i].y + c[i].z + c[i].w;
  }
  uint32_t run = block_sum_before<T>(sum, warp_sums);
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const uint32_t x = run, y = x + c[i].x, z = y + c[i].y, w = z + c[i].z;
    p[i] = make_uint4(x, y, z, w);
    run = w + c[i].w;
  }
}

// Exclusive scan of v[0 .. n) in place (v on 16 bytes); ends with a barrier.
// Counts of 4 T to 16 T, those of the larger chains of each class, are read as
// 16-byte vectors: word by word, a thread's consecutive words put the lanes of
// a warp on 2 to 8 banks only.
template <int T>
__device__ void block_exclusive_scan(uint32_t *v, uint32_t n, uint32_t *warp_sums) {
  if (n == 4 * T) {
    vector_scan<T, 1>(v, warp_sums);
  } else if (n == 8 * T) {
    vector_scan<T, 2>(v, warp_sums);
  } else if (n == 16 * T) {
    vector_scan<T, 4>(v, warp_sums);
  } else {
    const uint32_t per = (n + T - 1) / T;
    const uint32_t lo = min(threadIdx.x * per, n), hi = min(lo + per, n);
    uint32_t sum = 0;
    for (uint32_t i = lo; i < hi; ++i) sum += v[i];
    uint32_t run = block_sum_before<T>(sum, warp_sums);
    for (uint32_t i = lo; i < hi; ++i) {
      const uint32_t c = v[i];
      v[i] = run;
      run += c;
    }
  }
  __syncthreads();
}

__device__ __forceinline__ uint32_t warp_sum(uint32_t x) { return __reduce_add_sync(0xffffffffu, x); }

// The most switches and the most Philox blocks (of four keys) a thread of a
// CTA of T threads takes: classes of at most 10240 (T = 1024), 4096, 2048 and
// 1024 edges.
template <int T>
struct ResPer {
  static constexpr uint32_t kMax = T == 1024 ? kResidentMaxEdges : T == 512 ? 4096 : T == 256 ? 2048 : 1024;
  static constexpr uint32_t kSwitches = (kMax / 2 + T - 1) / T;
  static constexpr uint32_t kBlocks = (kMax / 4 + T - 1) / T;
  static constexpr uint32_t kPermVec = (kMax / 8 + T - 1) / T;  // 16-byte pieces of a permutation
};

// Ranks again with full 64-bit keys (ties: the smaller position), for a
// round in which two keys of a bucket have the same 32 bits after the bucket
// bits: slots of the buckets as sort_round left them.
template <int T>
__device__ __noinline__ void rank_full(unsigned long long seed, unsigned long long round, uint32_t m, uint32_t nb_log2,
                                       const uint32_t *cnt, const uint16_t *spos, uint16_t *perm) {
  const uint32_t nb = 1u << nb_log2;
  for (uint32_t y = threadIdx.x; y < m; y += T) {
    const uint32_t x = spos[y];
    const unsigned long long kx = word_of(philox(x >> 2, round, 0, 0, seed, 0), x & 3);
    const uint32_t b = (uint32_t)(kx >> (64 - nb_log2)), lo = cnt[b], hi = b + 1 < nb ? cnt[b + 1] : m;
    uint32_t r = 0;
    for (uint32_t z = lo; z < hi; ++z) {
      const uint32_t v = spos[z];
      const unsigned long long kv = word_of(philox(v >> 2, round, 0, 0, seed, 0), v & 3);
      r += (kv < kx || (kv == kx && v < x)) ? 1u : 0u;
    }
    perm[lo + r] = (uint16_t)x;
  }
}

// pi of round `round` of chain ch into perm (shared memory): keys K(i) =
// Philox4x64-10((i >> 2, round, 0, 0); (seed, 0))[i & 3], counted per bucket
// (the top nb_log2 bits; the count gives the key's place among its bucket's
// arrivals), a scan, the next 32 key bits scattered by bucket, then each
// position's rank among its bucket's keys.  Where two keys of a bucket have
// the same 32 bits (once in about 10^6 rounds) the round's ranks are taken
// again with the full keys.  A key stays in its thread's registers from the
// count to the rank.  Returns l (exact laziness; L otherwise).  Every thread
// of the CTA calls it; it ends with a barrier.
template <int T>
__device__ __forceinline__ uint32_t sort_round(const ChainDesc &ch, unsigned long long round, uint32_t m, uint32_t L,
                                               uint32_t nb_log2, uint32_t *skey, uint32_t *cnt, uint16_t *spos,
                                               uint16_t *perm, uint32_t *s_warp, uint32_t *s_ell) {
  constexpr uint32_t KB = ResPer<T>::kBlocks;
  const uint32_t tid = threadIdx.x, nb = 1u << nb_log2;
  const bool exact = ch.exact_ell && ch.lazy_threshold;
  for (uint32_t b = tid; b < nb / 4; b += T) reinterpret_cast<uint4 *>(cnt)[b] = make_uint4(0, 0, 0, 0);
  if (tid == 0) *s_ell = 0;
  __syncthreads();
  if (exact) {
    uint32_t n = 0;
    const uint32_t nl = (L + 3) / 4;
    for (uint32_t q = tid; q < nl; q += T) {
      const U64x4 w0 = philox(q, round, 1, 0, ch.seed, 0);
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u) n += (4 * q + u < L && w0.w[u] >= ch.lazy_threshold) ? 1u : 0u;
    }
    n = warp_sum(n);
    if ((tid & 31u) == 0 && n) atomicAdd(s_ell, n);
  }
  uint32_t key[4 * KB], bk[4 * KB];  // bk: bucket, and the place among its arrivals in the high half
#pragma unroll
  for (uint32_t u = 0; u < KB; ++u) {
    const uint32_t q = tid + u * T;
    if (4 * q >= m) continue;
    const U64x4 w = philox(q, round, 0, 0, ch.seed, 0);
#pragma unroll
    for (uint32_t v = 0; v < 4; ++v) {
      const uint32_t hi = (uint32_t)(w.w[v] >> 32), b = hi >> (32 - nb_log2);
      key[4 * u + v] = __funnelshift_l((uint32_t)w.w[v], hi, nb_log2);
      bk[4 * u + v] = 4 * q + v < m ? b | (atomicAdd(&cnt[b], 1u) << 16) : 0u;
    }
  }
  __syncthreads();
  const uint32_t ell = exact ? *s_ell : L;
  block_exclusive_scan<T>(cnt, nb, s_warp);
#pragma unroll
  for (uint32_t u = 0; u < 4 * KB; ++u) {
    const uint32_t x = 4 * (tid + (u / 4) * T) + u % 4;
    if (x < m) {
      const uint32_t y = cnt[bk[u] & 0xFFFFu] + (bk[u] >> 16);
      skey[y] = key[u];
      spos[y] = (uint16_t)x;
    }
  }
  __syncthreads();
  bool tie = false;
#pragma unroll
  for (uint32_t u = 0; u < 4 * KB; ++u) {
    const uint32_t x = 4 * (tid + (u / 4) * T) + u % 4;
    if (x < m) {
      const uint32_t b = bk[u] & 0xFFFFu, lo = cnt[b], hi = b + 1 < nb ? cnt[b + 1] : m, own = lo + (bk[u] >> 16);
      uint32_t r = 0;
      for (uint32_t z = lo; z < hi; ++z) {
        const uint32_t kz = skey[z];
        r += kz < key[u] ? 1u : 0u;
        tie |= kz == key[u] && z != own;
      }
      perm[lo + r] = (uint16_t)x;
    }
  }
  if (__syncthreads_or(tie)) {
    rank_full<T>(ch.seed, round, m, nb_log2, cnt, spos, perm);
    __syncthreads();
  }
  return ell;
}

// The same as a call of its own, for the CTA of 1024 threads: inlined, the twelve
// keys of a thread and what the round keeps besides left it 324 bytes of
// spills, which go to L2 (shared memory takes nearly all of L1); so, the kernel
// has 252 and the call 116.  20 rounds of 200 chains of 8,011 edges: 1299 -> 1275
// us, of 9,641 (dense) 2320 -> 2114.  The smaller CTAs, eight keys a thread and
// 264 bytes of spills, are 3 to 4% slower so.
template <int T>
__device__ __noinline__ uint32_t sort_apart(const ChainDesc &ch, unsigned long long round, uint32_t m, uint32_t L,
                                            uint32_t nb_log2, uint32_t *skey, uint32_t *cnt, uint16_t *spos,
                                            uint16_t *perm, uint32_t *s_warp, uint32_t *s_ell) {
  return sort_round<T>(ch, round, m, L, nb_log2, skey, cnt, spos, perm, s_warp, s_ell);
}
template <int T>
constexpr bool kSortApart = T == 1024;

// The rounds of one chain on one CTA.  What bounds it: issued instructions
// (about 44 thousand warp instructions a round of 5,000 edges, two a cycle)
// and, between them, the chains of dependent shared-memory operations of each
// step; nothing goes to memory.  A table of all targets and a failing search
// of it for every edge of E took 18 us a round of G(1000, 0.01) with its
// permutations sorted beforehand; the bitmaps leave about a seventh of the
// switches to the table, 10.5 us.  50 rounds of 1024 chains of 100 to 9,600
// edges: 7.2 ms before, 3.8 ms now (sort, bitmaps, classes beside each other).
// kPre: the permutations were sorted beforehand (job.pbuf).
template <int T, bool kPre>
__global__ void __launch_bounds__(T, 1024 / T) k_round_resident(RoundArgs a, ResidentJob job) {
  extern __shared__ __align__(16) unsigned char res_dyn[];
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_ell;
  __shared__ uint32_t s_wave[3];  // per wave (mod 3): undecided, and decided in the high half
  __shared__ uint32_t s_cand, s_hit;  // candidates, edges of E on a target's bit
  const uint32_t tid = threadIdx.x;
  const uint32_t c = job.jobs[blockIdx.x];
  const ChainDesc &ch = a.chains[c];
  const uint32_t m = ch.m, L = ch.L;
  // after the permutations' launch, the first class's kernel waits for it before
  // the rounds and only then lets the next class start, so that no class
  // starts before them
  const bool after_perms = kPre && job.first;
  if (!after_perms) dep_launch();
  if (m < 2 || m > kResidentMaxEdges) {  // the host sends only chains that qualify
    dep_wait();
    return;
  }
  const ResLayout lay = res_layout(m);
  uint32_t *const E = reinterpret_cast<uint32_t *>(res_dyn);
  uint16_t *const scat = reinterpret_cast<uint16_t *>(res_dyn + lay.scat);   // positions by bucket
  uint32_t *const tslot = reinterpret_cast<uint32_t *>(res_dyn + lay.scat);  // later: the targets' slots
  uint16_t *const perm = reinterpret_cast<uint16_t *>(res_dyn + lay.perm);   // pi
  uint16_t *const status = reinterpret_cast<uint16_t *>(res_dyn + lay.status);
  uint32_t *const skey = reinterpret_cast<uint32_t *>(res_dyn + lay.region);
  uint32_t *const cnt = reinterpret_cast<uint32_t *>(res_dyn + lay.region + align16(4 * m));
  const uint32_t nb_log2 = lay.nb_log2, bits_log2 = lay.bits_log2, words = 1u << (bits_log2 - 5);
  uint32_t *const seen = reinterpret_cast<uint32_t *>(res_dyn + lay.region);  // bits of the round's targets
  uint32_t *const marked = seen + words;                                      // bits that need a closer look
  uint16_t *const cand = reinterpret_cast<uint16_t *>(res_dyn + lay.region + lay.lists);
  uint16_t *const hits = reinterpret_cast<uint16_t *>(res_dyn + lay.region + lay.lists + align16(2 * L));
  uint32_t *const tkey = reinterpret_cast<uint32_t *>(res_dyn + lay.region);
  uint32_t *const multi = reinterpret_cast<uint32_t *>(res_dyn + lay.multi);
  const unsigned long long R0 = *(volatile unsigned long long *)&a.ctl->pool_round;

  // the list by position, with the last round's decision of each pair of
  // slots applied (Def. 1's rewiring of a legal switch)
  bool bad = false;
  const bool apply = R0 > ch.added;
  for (uint32_t s = tid; s < m; s += T) {
    const uint32_t pos = a.cpos[ch.slot_base + s];
    unsigned long long e = a.cedge[ch.slot_base + s];
    const uint32_t k = s >> 1;
    if (apply && k < L && (a.status[ch.switch_base + k] & 3u) == kLegal) {
      const uint32_t s0 = ch.slot_base + 2 * k;
      unsigned long long e3, e4;
      tau_g(a.cpos[s0] < a.cpos[s0 + 1] ? 1u : 0u, a.cedge[s0], a.cedge[s0 + 1], e3, e4);
      e = (s & 1u) ? e4 : e3;
    }
    const uint32_t lo = (uint32_t)(e >> 32), hi = (uint32_t)e;
    if (pos >= m || lo >= hi || hi >= kResidentMaxNodes) {
      bad = true;
      continue;
    }
    E[pos] = (lo << 16) | hi;
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) atomicOr(&a.ctl->err, kErrRecord);
    dep_wait();
    return;
  }

  uint32_t acc = 0, rloop = 0, rexist = 0, rlazy = 0;  // this thread's tallies
  const bool exact = ch.exact_ell && ch.lazy_threshold;
  uint32_t err = 0;
  if (after_perms) {
    dep_wait();
    dep_launch();
  }
  bool dense = false;  // (the same in all threads) the bitmaps are left out
  constexpr uint32_t KS = ResPer<T>::kSwitches, KP = ResPer<T>::kPermVec;
  // a permutation sorted beforehand is loaded a round ahead, into registers
  const uint32_t nvec = (m + 7) / 8;
  const size_t prow = (size_t)job.njobs * job.pstride;
  const uint16_t *psrc = kPre ? job.pbuf + (size_t)(job.job_base + blockIdx.x) * job.pstride : nullptr;
  uint4 pvec[KP];
  if constexpr (kPre) {
#pragma unroll
    for (uint32_t u = 0; u < KP; ++u)
      if (tid + u * T < nvec) pvec[u] = __ldcg(reinterpret_cast<const uint4 *>(psrc) + tid + u * T);
  }
  for (uint32_t t = 0; t < job.rounds && !err; ++t) {
    const unsigned long long round = ch.start_round + (R0 + t - ch.join);
    // 1. pi of this round (sorted here, or beforehand on other SMs) and l
    uint32_t ell;
    if constexpr (kPre) {
#pragma unroll
      for (uint32_t u = 0; u < KP; ++u)
        if (tid + u * T < nvec) reinterpret_cast<uint4 *>(perm)[tid + u * T] = pvec[u];
      psrc += prow;
      if (t + 1 < job.rounds) {
#pragma unroll
        for (uint32_t u = 0; u < KP; ++u)
          if (tid + u * T < nvec) pvec[u] = __ldcg(reinterpret_cast<const uint4 *>(psrc) + tid + u * T);
      }
      ell = exact ? __ldcg(&job.ebuf[(size_t)t * job.njobs + job.job_base + blockIdx.x]) : L;
    } else {
      ell = kSortApart<T> ? sort_apart<T>(ch, round, m, L, nb_log2, skey, cnt, scat, perm, s_warp, &s_ell)
                          : sort_round<T>(ch, round, m, L, nb_log2, skey, cnt, scat, perm, s_warp, &s_ell);
    }

    // 2. switches: outright rejects, the others' targets into the bitmap
    // (the sort's keys are dead)
    if (!dense)
      for (uint32_t w = tid; w < words / 2; w += T) reinterpret_cast<uint4 *>(seen)[w] = make_uint4(0, 0, 0, 0);
    if (tid == 0) s_cand = s_hit = 0;
    __syncthreads();
    uint32_t lazies = 0;  // the thread's switches that laziness skips
    if (ch.lazy_threshold) {
#pragma unroll 1
      for (uint32_t u = 0; u < KS && tid + u * T < L; ++u) {
        const uint32_t k = tid + u * T;
        const bool lazy =
            exact ? k >= ell : word_of(philox(k >> 2, round, 1, 0, ch.seed, 0), k & 3) < ch.lazy_threshold;
        lazies |= lazy ? 1u << u : 0u;
      }
    }
    // a thread keeps its switches' positions and sources for the round
    uint32_t ij[KS], e1[KS], e2[KS], live = 0;
#pragma unroll
    for (uint32_t u = 0; u < KS; ++u) {
      const uint32_t k = tid + u * T;
      if (k >= L) continue;
      ij[u] = reinterpret_cast<const uint32_t *>(perm)[k];
      const uint32_t i = ij[u] & 0xFFFFu, j = ij[u] >> 16;
      e1[u] = E[i];
      e2[u] = E[j];
      uint32_t e3 = 0, e4 = 0;
      const uint32_t code = (lazies >> u) & 1u ? kCodeLazy : tau16(i < j ? 1u : 0u, e1[u], e2[u], e3, e4);
      if (code) {
        status[k] = (uint16_t)kIllegal;  // known before the first wave (wave field 0)
        if (code == kCodeLazy) ++rlazy;
        else if (code == kCodeLoop) ++rloop;
        else ++rexist;
        continue;
      }
      live |= 1u << u;
      if (dense) {
        status[k] = (uint16_t)kUndecided;
        continue;
      }
      const uint32_t b3 = bit_of(e3, bits_log2), b4 = bit_of(e4, bits_log2);
      if ((atomicOr(&seen[b3 >> 5], 1u << (b3 & 31)) >> (b3 & 31)) & 1u) atomicOr(&marked[b3 >> 5], 1u << (b3 & 31));
      if ((atomicOr(&seen[b4 >> 5], 1u << (b4 & 31)) >> (b4 & 31)) & 1u) atomicOr(&marked[b4 >> 5], 1u << (b4 & 31));
    }
    __syncthreads();
    uint32_t ncand = L, nhit = 0;
    if (!dense) {
      // edges of E on a target's bit (few; one counter atomic for a thread's)
      uint32_t mine = 0;
#pragma unroll
      for (uint32_t u = 0; u < KS; ++u) {
        if (tid + u * T >= L) continue;
        const uint32_t b1 = bit_of(e1[u], bits_log2), b2 = bit_of(e2[u], bits_log2);
        mine |= bit_set(seen, b1) ? 1u << (2 * u) : 0u;
        mine |= bit_set(seen, b2) ? 2u << (2 * u) : 0u;
      }
      if (mine) {
        uint32_t at = atomicAdd(&s_hit, (uint32_t)__popc(mine));
#pragma unroll
        for (uint32_t u = 0; u < KS; ++u) {
          const uint32_t k = tid + u * T, b1 = bit_of(e1[u], bits_log2), b2 = bit_of(e2[u], bits_log2);
          if ((mine >> (2 * u)) & 1u) {
            atomicOr(&marked[b1 >> 5], 1u << (b1 & 31));
            hits[at++] = (uint16_t)(2 * k);
          }
          if ((mine >> (2 * u)) & 2u) {
            atomicOr(&marked[b2 >> 5], 1u << (b2 & 31));
            hits[at++] = (uint16_t)(2 * k + 1);
          }
        }
      }
      if ((m & 1u) && tid == T - 1) {  // the unpaired slot
        const uint32_t b = bit_of(E[perm[m - 1]], bits_log2);
        if (bit_set(seen, b)) {
          atomicOr(&marked[b >> 5], 1u << (b & 31));
          hits[atomicAdd(&s_hit, 1u)] = (uint16_t)(m - 1);
        }
      }
      __syncthreads();
      // free targets: legal in the first wave; the others are candidates, with
      // which of their targets are marked in tslot
      mine = 0;
#pragma unroll
      for (uint32_t u = 0; u < KS; ++u) {
        if (!((live >> u) & 1u)) continue;
        const uint32_t k = tid + u * T;
        uint32_t e3, e4;
        tau16((ij[u] & 0xFFFFu) < (ij[u] >> 16) ? 1u : 0u, e1[u], e2[u], e3, e4);
        const uint32_t f = (bit_set(marked, bit_of(e3, bits_log2)) ? 1u : 0u) |
                           (bit_set(marked, bit_of(e4, bits_log2)) ? 2u : 0u);
        status[k] = (uint16_t)(f ? kUndecided : (1u << 2) | kLegal);
        tslot[k] = f;
        mine |= f ? 1u << u : 0u;
      }
      if (mine) {
        uint32_t at = atomicAdd(&s_cand, (uint32_t)__popc(mine));
#pragma unroll
        for (uint32_t u = 0; u < KS; ++u)
          if ((mine >> u) & 1u) cand[at++] = (uint16_t)(tid + u * T);
      }
      __syncthreads();
      ncand = s_cand;
      nhit = s_hit;
    }

    // 3. the candidates' marked targets into the table, over the bitmaps; a
    // table that does not fit there takes the lists' bytes too, and every
    // thread then goes through its own switches (and every edge of E is looked
    // up).  Where most switches are candidates (a dense graph: most targets are
    // edges), the call's next rounds enter all of them at once: the bitmaps are
    // a sixth of such a round (20 rounds of K_140 less a hundredth, 9,641 edges:
    // 929 us with them, 779 without; a quarter of free switches pays for them).
    uint32_t wave = 1;
    if (ncand) {
      uint32_t slog2 = 5;  // room for twice the marked targets (at most two a candidate)
      while (slog2 < lay.slog2 && (1u << slog2) < 4 * ncand) ++slog2;
      const bool listed = !dense && slog2 <= lay.list_slog2;
      if (!listed) slog2 = lay.slog2;
      const uint32_t S = 1u << slog2, ntake = listed ? ncand : L;
      uint32_t *const tpq = tkey + S;
      for (uint32_t s = tid; s < S / 2; s += T) reinterpret_cast<uint4 *>(tkey)[s] = make_uint4(~0u, ~0u, ~0u, ~0u);
      for (uint32_t w = tid; w < S / 32; w += T) multi[w] = 0;
      if (tid < 3) s_wave[tid] = 0;
      __syncthreads();
      // every candidate enters its marked targets, registers there as an
      // inserter (smallest q per id) and keeps their slots
      bool full = false;
      auto enter = [&](uint32_t k, uint32_t f, uint32_t i, uint32_t j, uint32_t x1, uint32_t x2) {
        uint32_t e3, e4, s3 = kFree, s4 = kFree;
        tau16(i < j ? 1u : 0u, x1, x2, e3, e4);
        if (f & 1u) s3 = tab_insert(tkey, slog2, e3);
        if (f & 2u) s4 = tab_insert(tkey, slog2, e4);
        if (s3 == S || s4 == S) {
          full = true;
          s3 = s4 = kFree;
        }
        // a slot whose q was already set has a second inserter
        if (s3 != kFree && (tab_qmin(tpq, s3, k) & 0xFFFFu) != kQ16None) atomicOr(&multi[s3 >> 5], 1u << (s3 & 31));
        if (s4 != kFree && (tab_qmin(tpq, s4, k) & 0xFFFFu) != kQ16None) atomicOr(&multi[s4 >> 5], 1u << (s4 & 31));
        tslot[k] = s3 | (s4 << 16);
      };
      if (listed) {
        for (uint32_t c = tid; c < ncand; c += T) {
          const uint32_t k = cand[c], pij = reinterpret_cast<const uint32_t *>(perm)[k], i = pij & 0xFFFFu, j = pij >> 16;
          enter(k, tslot[k], i, j, E[i], E[j]);
        }
      } else if constexpr (!kPre) {  // (the sort leaves no registers to unroll this)
#pragma unroll 1
        for (uint32_t k = tid; k < L; k += T) {
          const uint32_t f = status[k] != kUndecided ? 0u : dense ? 3u : tslot[k];
          const uint32_t pij = reinterpret_cast<const uint32_t *>(perm)[k], i = pij & 0xFFFFu, j = pij >> 16;
          if (f) enter(k, f, i, j, E[i], E[j]);
          else tslot[k] = kFree | (kFree << 16);
        }
      } else {
#pragma unroll
        for (uint32_t u = 0; u < KS; ++u) {
          const uint32_t k = tid + u * T;
          if (k >= L) continue;
          const uint32_t f = !((live >> u) & 1u) ? 0u : dense ? 3u : tslot[k];
          if (f) enter(k, f, ij[u] & 0xFFFFu, ij[u] >> 16, e1[u], e2[u]);
          else tslot[k] = kFree | (kFree << 16);
        }
      }
      if (__syncthreads_or(full)) {
        err = kErrTableFull;
        break;
      }
      // erasers of the edges that are targets
      auto erase = [&](uint32_t e, uint32_t p) {
        const uint32_t slot = tab_find(tkey, slog2, e);
        if (slot < S) atomicAnd(&tpq[slot], (p << 16) | 0xFFFFu);
      };
      if (listed || !kPre) {
        for (uint32_t x = tid; x < (listed ? nhit : m); x += T) {
          const uint32_t s = listed ? hits[x] : x;
          erase(E[perm[s]], (s >> 1) < L ? (s >> 1) : kP16Keep);
        }
      } else {
#pragma unroll
        for (uint32_t u = 0; u < KS; ++u) {
          const uint32_t k = tid + u * T;
          if (k >= L) continue;
          erase(e1[u], k);
          erase(e2[u], k);
        }
        if ((m & 1u) && tid == T - 1) erase(E[perm[m - 1]], kP16Keep);
      }
      __syncthreads();

      // 4. waves
      uint32_t entering = L;
      bool requeue = false;
      for (;;) {
        if (job.final && t + 1 == job.rounds && tid == 0 && wave >= 2 && wave < kWaveHist)
          atomicAdd(&job.last_pending[wave], entering);
        if (tid == 0) s_wave[(wave + 1) % 3] = 0;  // read two waves ago, written next wave
        if (requeue) {
          // q of every id with two inserters or more goes back to "none", and
          // the inserters that are not illegal register again; an id with one
          // inserter keeps it as q, since only that inserter looks at the id's q
          // (the switches known to fail before the first wave never registered)
          for (uint32_t c = tid; c < ntake; c += T) {
            const uint32_t k = listed ? cand[c] : c;
            if (status[k] == (uint16_t)kIllegal) continue;
            const uint32_t ts = tslot[k], s3 = ts & 0xFFFFu, s4 = ts >> 16;
            if (s3 != kFree && is_multi(multi, s3)) atomicOr(&tpq[s3], 0xFFFFu);
            if (s4 != kFree && is_multi(multi, s4)) atomicOr(&tpq[s4], 0xFFFFu);
          }
          __syncthreads();
          for (uint32_t c = tid; c < ntake; c += T) {
            const uint32_t k = listed ? cand[c] : c;
            if ((status[k] & 3u) == kIllegal) continue;
            const uint32_t ts = tslot[k], s3 = ts & 0xFFFFu, s4 = ts >> 16;
            if (s3 != kFree && is_multi(multi, s3)) tab_qmin(tpq, s3, k);
            if (s4 != kFree && is_multi(multi, s4)) tab_qmin(tpq, s4, k);
          }
          __syncthreads();
        }
        uint32_t und = 0, dec = 0;
        bool ill = false;  // an id with two inserters or more lost one
        for (uint32_t c = tid; c < ntake; c += T) {
          const uint32_t k = listed ? cand[c] : c;
          if (status[k] != kUndecided) continue;
          const uint32_t ts = tslot[k];
          bool illegal = false, wait = false, many = false;
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const uint32_t sl = x ? ts >> 16 : ts & 0xFFFFu;
            if (sl == kFree) continue;
            many |= is_multi(multi, sl);
            const uint32_t pq = tpq[sl];
            const uint32_t p = pq >> 16, q = pq & 0xFFFFu;
            if (p != kP16None) {      // the target is in E when the round starts
              if (p > k) {
                illegal = true;       // erased after k, or never
              } else {
                const uint32_t sp = status[p];
                if (!decided_before(sp, wave)) wait = true;
                else if ((sp & 3u) == kIllegal) illegal = true;  // its eraser failed
              }
            }
            if (q != kQ16None && q < k) {  // an earlier switch may insert it first
              const uint32_t sq = status[q];
              if (!decided_before(sq, wave)) wait = true;
              else if ((sq & 3u) == kLegal) illegal = true;
            }
          }
          if (!illegal && wait) {
            ++und;
            continue;
          }
          status[k] = (uint16_t)((wave << 2) | (illegal ? kIllegal : kLegal));
          ++dec;
          ill |= illegal && many;
        }
        // both counts in one word (at most 5120 switches)
        const uint32_t both = warp_sum(und | (dec << 16));
        if ((tid & 31u) == 0 && both) atomicAdd(&s_wave[wave % 3], both);
        const bool I = __syncthreads_or(ill);
        const uint32_t U = s_wave[wave % 3] & 0xFFFFu, D = s_wave[wave % 3] >> 16;
        if (U == 0) break;
        // impossible for a valid round: the smallest undecided switch decides
        // (in the first wave it may be one that is no candidate)
        if (D == 0 && (wave > 1 || ncand == L)) {
          err = kErrNoProgress;
          break;
        }
        if (wave >= job.wave_cap) {
          err = kErrWaveCap;
          break;
        }
        ++wave;
        entering = U;
        requeue = I;
      }
      if (err) break;
      dense = 4 * ncand > 3 * L;
    }
    if (tid == 0) atomicMax(&job.round_waves[t], wave);

    // 5. legal switches rewrite their positions
#pragma unroll
    for (uint32_t u = 0; u < KS; ++u) {
      if (!((live >> u) & 1u)) continue;
      const uint32_t k = tid + u * T;
      if ((status[k] & 3u) == kLegal) {
        const uint32_t i = ij[u] & 0xFFFFu, j = ij[u] >> 16;
        uint32_t e3, e4;
        tau16(i < j ? 1u : 0u, e1[u], e2[u], e3, e4);
        E[i] = e3;
        E[j] = e4;
        ++acc;
      } else {
        ++rexist;               // illegal by a wave: a target was in E when it ran
      }
    }
    __syncthreads();
  }
  if (err) {
    if (tid == 0) atomicOr(&a.ctl->err, err);
    dep_wait();
    return;
  }
  // the list back to the chain's slots, by position, nothing pending
  for (uint32_t x = tid; x < m; x += T) {
    const uint32_t e = E[x];
    a.cpos[ch.slot_base + x] = x;
    a.cedge[ch.slot_base + x] = ((unsigned long long)(e >> 16) << 32) | (e & 0xFFFFu);
  }
  for (uint32_t k = tid; k < L; k += T) a.status[ch.switch_base + k] = 0u;
  acc = warp_sum(acc);
  rloop = warp_sum(rloop);
  rexist = warp_sum(rexist);
  rlazy = warp_sum(rlazy);
  if ((tid & 31u) == 0) {
    if (acc) {
      atomicAdd(&a.st->accepted, (unsigned long long)acc);
      atomicAdd(&a.chain_accepted[c], (unsigned long long)acc);
    }
    if (rloop) atomicAdd(&a.st->rej_loop, (unsigned long long)rloop);
    if (rexist) atomicAdd(&a.st->rej_exists, (unsigned long long)rexist);
    if (rlazy) atomicAdd(&a.st->lazy, (unsigned long long)rlazy);
  }
  dep_wait();
}

// The permutations of all rounds of a launch, one CTA per (chain, round),
// ahead of the resident kernel, for pools of few chains: the keys and the
// sort depend only on the chain's seed, round number and m, never on its
// list, so other SMs sort them while the chain's own CTA would otherwise
// sit in the sort phases of each round.
template <int T>
__global__ void __launch_bounds__(T, 1024 / T) k_resident_perm(RoundArgs a, ResidentJob job) {
  extern __shared__ __align__(16) unsigned char res_dyn[];
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_ell;
  dep_launch();
  if (blockIdx.x == 0 && blockIdx.y == 0 && job.first)  // (the host zeroes them where no permutations come first)
    for (uint32_t w = threadIdx.x; w < job.rounds + kWaveHist; w += T) job.last_pending[w] = 0;
  const ChainDesc ch = a.chains[job.jobs[blockIdx.x]];
  const uint32_t m = ch.m;
  if (m < 2 || m > kResidentMaxEdges) {
    dep_wait();
    return;
  }
  const ResLayout lay = res_layout(m);
  uint16_t *const perm = reinterpret_cast<uint16_t *>(res_dyn);
  uint16_t *const spos = reinterpret_cast<uint16_t *>(res_dyn + align16(2 * m));
  uint32_t *const skey = reinterpret_cast<uint32_t *>(res_dyn + 2 * align16(2 * m));
  uint32_t *const cnt = reinterpret_cast<uint32_t *>(res_dyn + 2 * align16(2 * m) + align16(4 * m));
  const unsigned long long R0 = *(volatile unsigned long long *)&a.ctl->pool_round;
  const uint32_t t = blockIdx.y;
  const size_t jg = (size_t)t * job.njobs + job.job_base + blockIdx.x;
  const uint32_t ell = sort_round<T>(ch, ch.start_round + (R0 + t - ch.join), m, ch.L, lay.nb_log2, skey, cnt, spos,
                                     perm, s_warp, &s_ell);
  // out in 16-byte pieces (rows start on 16 bytes; the last piece's tail is
  // inside the row and never read)
  uint4 *const row = reinterpret_cast<uint4 *>(job.pbuf + jg * job.pstride);
  for (uint32_t v = threadIdx.x; v < (m + 7) / 8; v += T) row[v] = reinterpret_cast<const uint4 *>(perm)[v];
  if (threadIdx.x == 0) job.ebuf[jg] = ell;
  dep_wait();
}

__host__ __device__ inline uint32_t perm_smem_bytes(uint32_t m) {
  const ResLayout l = res_layout(m < 2 ? 2 : m);
  return 2 * align16(2 * m) + align16(4 * m) + 4 * (1u << l.nb_log2);
}

// The launch's rounds into the statistics (each round's wave count is the
// largest over its chains, as in the general path) and the pool round on.
__global__ void k_resident_fold(RoundArgs a, ResidentJob job) {
  dep_wait();
  __shared__ unsigned long long hist[kWaveHist];
  __shared__ unsigned long long total, most;
  const uint32_t tid = threadIdx.x;
  for (uint32_t i = tid; i < kWaveHist; i += blockDim.x) hist[i] = 0;
  if (tid == 0) total = most = 0;
  __syncthreads();
  for (uint32_t t = tid; t < job.rounds; t += blockDim.x) {
    const uint32_t w = job.round_waves[t];
    atomicAdd(&hist[w < kWaveHist ? w : kWaveHist - 1], 1ull);
    atomicAdd(&total, (unsigned long long)w);
    atomicMax(&most, (unsigned long long)w);
  }
  __syncthreads();
  if (a.any_work) {
    for (uint32_t i = tid; i < kWaveHist; i += blockDim.x)
      if (hist[i]) a.st->wave_hist[i] += hist[i];
  }
  if (tid == 0) {
    if (a.any_work) {
      a.st->waves_total += total;
      if (most > a.st->waves_max) a.st->waves_max = most;
    }
    if (job.final) {
      a.ctl->waves = (a.any_work && job.rounds) ? job.round_waves[job.rounds - 1] : 0u;
      a.st->last_pending[1] = a.switch_hw;
      for (uint32_t w = 2; w < kWaveHist; ++w) a.st->last_pending[w] = job.last_pending[w];
    }
    a.ctl->pool_round += job.rounds;
  }
}

// The most edges a chain of each class has (CTAs of 1024, 512, 256 and 128
// threads).
constexpr uint32_t kClassMaxEdges[kResidentClasses] = {kResidentMaxEdges, 4096, 2048, 1024};

// One class's kernel.  `beside`: it need not wait to start for the launch
// before it, another class's, and does as soon as that one's CTAs are all on the
// GPU (programmatic dependent launch).  Every kernel launched so waits for the one
// before it just before it ends, so what follows the last class follows all.
// 50 rounds of 1024 chains of 100 to 9,600 edges: 6.2 ms with one class after
// another, 4.4 ms beside each other (the largest class has one CTA an SM and
// about as many chains as there are SMs; the other classes fill up behind it).
template <class... Args>
cudaError_t launch_beside(void (*fn)(Args...), dim3 grid, uint32_t threads, uint32_t smem, cudaStream_t s, bool beside,
                          Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = beside ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

template <int T>
cudaError_t launch_class(const RoundArgs &a, const ResidentJob &j, uint32_t n, uint32_t max_m, bool perms, bool beside,
                         cudaStream_t s) {
  if (perms) return launch_beside(k_resident_perm<T>, dim3(n, j.rounds), T, perm_smem_bytes(max_m), s, beside, a, j);
  const uint32_t smem = res_layout(max_m < 2 ? 2 : max_m).bytes;
  if (j.pbuf) return launch_beside(k_round_resident<T, true>, dim3(n), T, smem, s, beside, a, j);
  return launch_beside(k_round_resident<T, false>, dim3(n), T, smem, s, beside, a, j);
}

}  // namespace

uint32_t resident_class(uint32_t m) {
  uint32_t c = 0;
  while (c + 1 < kResidentClasses && m <= kClassMaxEdges[c + 1]) ++c;
  return c;
}

size_t resident_smem_bytes(uint32_t m) { return res_layout(m).bytes; }

template <int T>
cudaError_t prepare_class(uint32_t max_m) {
  cudaError_t e = cudaFuncSetAttribute(k_round_resident<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)resident_smem_bytes(max_m));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_round_resident<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)resident_smem_bytes(max_m));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_resident_perm<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)perm_smem_bytes(max_m));
  return e;
}

cudaError_t prepare_resident() {
  cudaError_t e = prepare_class<1024>(kClassMaxEdges[0]);
  if (e == cudaSuccess) e = prepare_class<512>(kClassMaxEdges[1]);
  if (e == cudaSuccess) e = prepare_class<256>(kClassMaxEdges[2]);
  if (e == cudaSuccess) e = prepare_class<128>(kClassMaxEdges[3]);
  return e;
}

cudaError_t launch_round_resident(const RoundArgs &a, const uint32_t *jobs, const uint32_t (&count)[kResidentClasses],
                                  const uint32_t (&max_m)[kResidentClasses], uint32_t rounds, uint32_t *round_waves,
                                  uint32_t *last_pending, bool final, uint16_t *pbuf, uint32_t *ebuf, uint32_t pstride,
                                  cudaStream_t s, uint32_t *launches) {
  ResidentJob j;
  j.rounds = rounds;
  j.pbuf = pbuf;
  j.ebuf = ebuf;
  j.pstride = pstride;
  j.njobs = 0;
  for (uint32_t c = 0; c < kResidentClasses; ++c) j.njobs += count[c];
  j.round_waves = round_waves;
  j.last_pending = last_pending;
  j.final = final ? 1u : 0u;
  // status words hold the wave in 14 bits; a round needs at most L + 1 <= 5121 waves
  const uint32_t cap = a.max_waves ? a.max_waves : kDefaultWaveCap;
  j.wave_cap = cap < 16383u ? cap : 16383u;
  for (int perms = pbuf ? 1 : 0; perms >= 0; --perms) {
    uint32_t off = 0;
    for (uint32_t c = 0; c < kResidentClasses; ++c) {
      if (!count[c]) continue;
      j.jobs = jobs + off;
      j.job_base = off;
      const bool beside = off > 0 || (pbuf && !perms);
      j.first = off == 0 ? 1u : 0u;
      off += count[c];
      cudaError_t e = cudaSuccess;
      switch (c) {
        case 0: e = launch_class<1024>(a, j, count[c], max_m[c], perms, beside, s); break;
        case 1: e = launch_class<512>(a, j, count[c], max_m[c], perms, beside, s); break;
        case 2: e = launch_class<256>(a, j, count[c], max_m[c], perms, beside, s); break;
        default: e = launch_class<128>(a, j, count[c], max_m[c], perms, beside, s); break;
      }
      if (e != cudaSuccess) return e;
      ++*launches;
    }
  }
  j.jobs = jobs;
  ++*launches;
  return launch_beside(k_resident_fold, dim3(1), 256, 0, s, j.njobs > 0, a, j);
}

}  // namespace gesmc
