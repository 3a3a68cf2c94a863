// ParES (Algorithm 2 of arXiv 2111.03005): exact parallel ES-MC on one GB300.
//
// ES-MC runs independent edge switches sigma_k = (i, j, g) one after
// another (Def. 1's chain).  Algorithm 2 cuts the sequence into supersteps:
// maximal runs of consecutive switches of which no two share a source
// position.  Where a cut falls depends on the sampled positions only, never
// on the graph, so the switches of a whole batch are sampled beforehand on
// the whole GPU (k_es_sample), each with the distance to the last switch
// before it that has a source position in common with it: the superstep that
// starts at switch s ends before the first switch s + x whose distance is at
// most x.  A superstep has no source dependencies, so ParallelSuperstep
// (Algorithm 1) performs it with the sequential outcome: each target edge
// exists when its switch runs iff it was in E at the superstep's start and its
// eraser (the switch whose source it is) is not an earlier legal switch, or an
// earlier legal switch inserts it.
//
// Supersteps of ES-MC hold about sqrt(m) switches (the birthday bound), so
// one CTA (for the largest chains a cluster of eight) runs all supersteps of
// one chain, a switch per thread.  The list E
// (position order) and the edge set H (open addressing over canonical ids,
// tombstones on erase) live in HBM (small chains have both in shared memory,
// with a bit per pair of nodes for H where that fits); a list entry also holds
// its edge's slot in H, so that erasing it takes no search, and the search for
// a target ends at the slot where it would be inserted.  Most supersteps have no dependency at
// all: the targets go into a shared-memory table of fingerprints, and if no
// fingerprint is met twice, by two targets or by a source, a switch is legal
// iff none of its targets is in H.  Else the superstep's erasers and
// inserters go into shared-memory tables and Algorithm 1's waves run,
// separated by __syncthreads.  Many chains run as many CTAs of one launch.  A
// superstep is also cut at the window size (32 to 1024 switches, by the
// chain's size) and at the end of a batch; any cut into consecutive runs
// without source dependencies gives the sequential result.  When tombstones
// pile up, the set is rebuilt from the list between supersteps: in place by
// the CTA for the smaller windows, on the whole GPU between launches for the
// largest.
#include "device_util.cuh"
#include "es_set.cuh"
#include "gesmc_internal.cuh"

namespace gesmc {
namespace {

constexpr unsigned long long kNoKey = 0;  // {0, 0}: not an edge, empty or tombstone
constexpr uint8_t kEsUndecided = 0, kEsLegal = 1, kEsIllegal = 2;
// Window sizes by chain size (supersteps hold about 0.63 sqrt(m) switches:
// 450 at 2^19, 160 at 2^16, 57 at 2^13): chains of at least 2^19 edges run
// windows of 1024 switches, chains of at least 2^16 windows of 256 on CTAs of
// 256 threads (six per SM), chains of at least 2^13 windows of 128, smaller
// ones windows of 32 on one warp each (up to 32 per SM), whose barriers cost
// next to nothing; of these, a chain whose bit matrix or table fits in shared
// memory keeps its list and set there.
constexpr uint32_t kEsBigChain = 1u << 19;
constexpr uint32_t kEsMidChain = 1u << 16;
constexpr uint32_t kEsSmallChain = 1u << 13;

// ---------------------------------------------------------------- the list and the edge set H
// Loads of a chain's list and set by its CTA.  kL1: through the SM's L1, for
// the small windows, whose chains' lists and sets fit there (one CTA writes
// them while the kernel runs, and its barriers order its own accesses); else
// from L2.
template <bool kL1>
__device__ __forceinline__ unsigned long long set_load(const unsigned long long *p) {
  unsigned long long v;
  if constexpr (kL1) asm volatile("ld.global.ca.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  else asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
template <bool kL1>
__device__ __forceinline__ uint4 list_load(const uint4 *p) {
  uint4 v;
  if constexpr (kL1)
    asm volatile("ld.global.ca.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  else
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// One warp inserts its lanes' keys (those of `legal` lanes, none of them in
// the set) at once: every lane stores each of its keys in a free slot and
// looks whose store stayed there, and the others search on.  p3, p4: where
// the searches ended, f3, f4: whether that slot is known to be free; p3, p4, t3,
// t4 receive the slots taken and whether they held tombstones.  All in the
// SM's L1, where a compare-and-swap goes to L2 and back (512 chains of 65 to
// 118,000 edges, 2^14 switches each: 10.3 ms with it, 8.9 ms without).  All lanes call it.
__device__ __forceinline__ unsigned long long warp_load(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.cta.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void warp_store(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.cta.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// The first free slot from p on; false if the table is full.
__device__ __forceinline__ bool warp_find_free(const unsigned long long *H, uint32_t mask, uint32_t &p, uint32_t &t) {
  for (uint32_t n = 0; n <= mask; ++n) {
    const unsigned long long v = warp_load(&H[p]);
    if (v == kEmptyKey || v == kTombKey) {
      t = v == kTombKey;
      return true;
    }
    p = (p + 1) & mask;
  }
  return false;
}
__device__ __forceinline__ void warp_insert(unsigned long long *H, uint32_t mask, bool legal, unsigned long long e3,
                                            unsigned long long e4, uint32_t &p3, uint32_t &p4, bool f3, bool f4,
                                            uint32_t &t3, uint32_t &t4, uint32_t *err) {
  bool o3 = legal, o4 = legal;
  __syncwarp();  // the erasures
  for (int round = 0;; ++round) {
    bool full = false;
    if (o3 && !f3) full |= !(o3 = warp_find_free(H, mask, p3, t3));
    if (o4 && !f4) full |= !(o4 = warp_find_free(H, mask, p4, t4));
    if (full) atomicOr(err, kErrTableFull);
    __syncwarp();
    if (o3) warp_store(&H[p3], e3);
    if (o4) warp_store(&H[p4], e4);
    __syncwarp();
    if (o3) o3 = warp_load(&H[p3]) != e3;
    if (o4) o4 = warp_load(&H[p4]) != e4;
    if (!__any_sync(0xffffffffu, o3 || o4)) break;
    if (round > 64) {  // a slot in dispute goes to one of the 64 keys each time: only in a full table
      if (o3 || o4) atomicOr(err, kErrTableFull);
      break;
    }
    f3 = f4 = false;
  }
}

// The list by position: {edge lo, edge hi, its slot in H, 0}.
__device__ __forceinline__ unsigned long long rec_edge(const uint4 &r) {
  return ((unsigned long long)r.y << 32) | r.x;
}
__device__ __forceinline__ uint4 make_rec(unsigned long long e, uint32_t slot) {
  return make_uint4((uint32_t)e, (uint32_t)(e >> 32), slot, 0u);
}

// ---------------------------------------------------------------- shared memory
// Per CTA, for windows of B switches (one per thread): the fingerprints of
// the superstep's targets (always empty between supersteps), and, for the
// supersteps that have a dependency, tables of S = 4B slots: the erasers'
// and inserters' keys (u64), the erasers' switches, the inserters' list heads
// and links, and every switch's state.  Everything else a switch needs (its
// positions, edges, hashes, outcome) stays in its thread's registers.
template <int B>
struct EsShape {
  static constexpr int kSlots = 4 * B;
  static constexpr int kPrintLog2 = B == 1024 ? 13 : B == 256 ? 11 : B == 128 ? 10 : B == 32 ? 8 : -1;
  static constexpr int kPrints = 1 << (kPrintLog2 > 0 ? kPrintLog2 : 0);
  static constexpr size_t kBytes = 16ull * kSlots + 4ull * (2 * kSlots + 2 * B) + 4ull * kPrints + B;
  static_assert(kPrintLog2 > 0, "window of 32, 128, 256 or 1024 switches");
};

template <int B>
struct EsSmem {
  unsigned long long *skey, *ikey;  // key tables
  uint32_t *sval, *ihead, *tnext, *print;
  uint8_t *st;
};

template <int B>
__device__ __forceinline__ EsSmem<B> es_smem() {
  extern __shared__ unsigned long long es_dyn[];
  constexpr int S = EsShape<B>::kSlots;
  EsSmem<B> m;
  m.skey = es_dyn;
  m.ikey = es_dyn + S;
  uint32_t *q = reinterpret_cast<uint32_t *>(es_dyn + 2 * S);
  m.sval = q;
  m.ihead = q + S;
  m.tnext = q + 2 * S;
  m.print = q + 2 * S + 2 * B;
  m.st = reinterpret_cast<uint8_t *>(m.print + EsShape<B>::kPrints);
  return m;
}

// Sources of the superstep's switches (key -> switch) and its targets (key
// -> list of (switch, which) entries through next[]); h = hash32(key).
template <int S>
__device__ __forceinline__ uint32_t table_slot(unsigned long long *keys, unsigned long long key, uint32_t h,
                                               bool claim) {
  uint32_t s = h & (S - 1);
  for (int n = 0; n < S; ++n) {
    const unsigned long long cur = keys[s];
    if (cur == key) return s;
    if (cur == kEmptyKey) {
      if (!claim) return kNil;
      const unsigned long long prev = atomicCAS(&keys[s], kEmptyKey, key);
      if (prev == kEmptyKey || prev == key) return s;
    }
    s = (s + 1) & (S - 1);
  }
  return kNil;
}

// The CTA's barrier and vote (one warp: the warp's).
template <int B>
__device__ __forceinline__ void window_sync() {
  if constexpr (B == 32) __syncwarp();
  else __syncthreads();
}
template <int B>
__device__ __forceinline__ bool window_any(bool x) {
  if constexpr (B == 32) {
    __syncwarp();
    return __any_sync(0xffffffffu, x);
  } else {
    return __syncthreads_or(x);
  }
}

// ---------------------------------------------------------------- kernels
// H <- empty, for every job (blockIdx.y = job).
__global__ void k_es_clear(EsJob *jobs, uint32_t job_off, bool only_stopped) {
  const EsJob &jb = jobs[job_off + blockIdx.y];
  if (!jb.H || (only_stopped && jb.stopped != 1)) return;  // no list, no set; or a set that needs no rebuild
  const unsigned long long cap = 1ull << jb.hlog2;
  const unsigned long long nth = (unsigned long long)gridDim.x * blockDim.x;
  unsigned long long *const H = jb.H;
  for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s < cap; s += nth)
    H[s] = kEmptyKey;
  if (blockIdx.x == 0 && threadIdx.x == 0) jobs[job_off + blockIdx.y].tombs = 0;
}

// H <- the entries of E, each entry's slot into the list, for the stopped jobs.
__global__ void k_es_fill(const EsJob *jobs, uint32_t job_off, uint32_t *err) {
  const EsJob jb = jobs[job_off + blockIdx.y];
  if (!jb.H || jb.stopped != 1) return;
  const uint32_t mask = (uint32_t)((1ull << jb.hlog2) - 1);
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < jb.m; s += gridDim.x * blockDim.x) {
    const unsigned long long e = rec_edge(jb.E[s]);
    uint32_t tomb;
    const uint32_t at = hset_insert(jb.H, mask, e, hash32(e) & mask, &tomb);
    if (at == kNil) atomicOr(err, kErrTableFull);
    else jb.E[s] = make_rec(e, at);
  }
}

// The switches off .. off + n - 1 of every job's call: positions and
// direction, and for each the distance to the last switch before it, in this
// batch and within a window, that shares a position with it (0xFFFF: none).
// One CTA of C threads per C switches and job: it samples them and the W - 1
// before them and chains the positions in a shared-memory hash table; a
// position is in the table once for every switch that has it.
template <int W, int C>
__global__ void __launch_bounds__(C) k_es_sample(EsJob *jobs, uint32_t job_off, unsigned long long off, uint32_t n,
                                                 uint2 *samples, uint16_t *dists) {
  constexpr int kEntries = 2 * (C + W - 1);
  constexpr int kLog2 = kEntries <= 512 ? 9 : kEntries <= 1024 ? 10 : kEntries <= 2048 ? 11 : 12;
  static_assert(kEntries <= 4096, "table size");
  __shared__ uint32_t pos[kEntries];
  __shared__ uint16_t next[kEntries];
  __shared__ __align__(4) uint16_t head[1 << kLog2];
  EsJob &jb = jobs[job_off + blockIdx.y];
  const uint32_t x = threadIdx.x, beg = blockIdx.x * C;
  if (blockIdx.x == 0 && x == 0) {  // the batch starts
    jb.done = 0;
    jb.stopped = 0;
  }
  const unsigned long long k0 = jb.k0 + off, seed = jb.seed, m = jb.m;
  uint2 *const samp = samples + (size_t)jb.row * n;
  uint16_t *const dist = dists + (size_t)jb.row * n;
  for (uint32_t b = x; b < (1u << kLog2); b += C) head[b] = 0xFFFFu;
  __syncthreads();
  const uint32_t first = beg < W - 1 ? 0u : beg - (W - 1), end = min(beg + C, n);
  for (uint32_t k = first + x; k < end; k += C) {
    const U64x4 w = philox(k0 + k, 0, 2, 0, seed, 0);
    const uint32_t i = (uint32_t)__umul64hi(w.w[0], m), jj = (uint32_t)__umul64hi(w.w[1], m - 1);
    const uint32_t j = jj + (jj >= i ? 1u : 0u);
    if (k >= beg) samp[k] = make_uint2(i, j | ((uint32_t)(w.w[2] >> 63) << 31));
    const uint32_t t = 2 * (k - first);
    pos[t] = i;
    pos[t + 1] = j;
  }
  __syncthreads();
  const uint32_t ne = 2 * (end - first);
  for (uint32_t t = x; t < ne; t += C) {
    // (16-bit exchange as a loop over the 32-bit word that holds the head)
    const uint32_t b = (pos[t] * 0x9E3779B1u) >> (32 - kLog2);
    uint32_t *const word = reinterpret_cast<uint32_t *>(head) + (b >> 1);
    const uint32_t sh = (b & 1u) * 16;
    uint32_t cur = *word, old;
    do {
      old = cur;
      cur = atomicCAS(word, old, (old & ~(0xFFFFu << sh)) | (t << sh));
    } while (cur != old);
    next[t] = (uint16_t)(old >> sh);
  }
  __syncthreads();
  const uint32_t k = beg + x;
  if (k < end) {
    const uint32_t own = k - first;
    uint32_t last = 0;  // 1 + the last earlier switch with one of the two positions
    for (int h = 0; h < 2; ++h) {
      const uint32_t p = pos[2 * own + h];
      for (uint32_t t = head[(p * 0x9E3779B1u) >> (32 - kLog2)]; t != 0xFFFFu; t = next[t]) {
        const uint32_t v = t >> 1;
        if (v < own && pos[t] == p) last = max(last, v + 1);
      }
    }
    const uint32_t d = last ? own + 1 - last : 0xFFFFu;
    dist[k] = (uint16_t)(d < (uint32_t)W ? d : 0xFFFFu);
  }
}

// One CTA per job: the n switches of the batch from the job's last one
// (done) on, in windows of B switches (thread x holds switch x of the window).
// A CTA of the largest variant does not rebuild its chain's edge set itself
// (one SM reinserting millions of ids): it stops after the superstep that
// passes the tombstone limit (an eighth of the slots: rebuilds are cheap on
// the whole GPU, and fewer tombstones keep the probe chains short), records
// how far it got (done, stopped = 1, *nstop counted), and the host rebuilds
// the set on the whole GPU and launches the variant again; a job that is done
// with the batch does nothing then.  The smaller variants rebuild in place at
// a quarter.
//
// What bounds it: one chain's supersteps follow one another, each a chain of
// dependent accesses (list entries, set slots, insertion) between a few
// barriers; a window of 1024 switches is also bound by the 32-byte sectors
// that one SM moves to and from L2 (about 11 a switch, and one every two
// cycles or so at random addresses).  With sampling and first-touch tables in
// every window, key tables for every superstep and separate searches to find,
// erase and insert, 2^19 switches of a chain of 1e6 edges took 21.4 ms, then 7.2
// (26 -> 8.9 us a superstep; on a cluster 5.1, see below); 512 chains of 65 to
// 118,000 edges with 2^14 switches each 22.0 ms, then 8.9 (most were single warps:
// 2270 -> 430 instructions a superstep), now 5.4: the chains of few nodes or edges
// have left this kernel for shared memory, see below.
template <int B, bool kStopToRebuild>
__device__ __forceinline__ void es_run_body(EsJob *jobs, uint32_t job_off, uint32_t nsw, const uint2 *samples,
                                            const uint16_t *dists, StatsDev *stats, unsigned long long *chain_acc,
                                            uint32_t *err, uint32_t *nstop) {
  constexpr int S = EsShape<B>::kSlots, PL = EsShape<B>::kPrintLog2;
  constexpr bool kL1 = B <= 128;
  constexpr uint32_t kPrintMask = EsShape<B>::kPrints - 1;
  EsJob &job = jobs[job_off + blockIdx.x];
  const EsSmem<B> sm = es_smem<B>();
  __shared__ uint32_t s_cut[2], s_tombs;
  const uint32_t x = threadIdx.x;
  const uint32_t m = job.m;
  uint32_t acc = 0, rej_loop = 0, rej_exists = 0;
  uint4 *const E = job.E;
  unsigned long long *const H = job.H;
  const uint2 *const samp = samples + (size_t)job.row * nsw;
  const uint16_t *const dist = dists + (size_t)job.row * nsw;
  const uint32_t mask = (uint32_t)((1ull << job.hlog2) - 1);
  uint32_t s = job.done;
  if (kStopToRebuild && !job.alone) return;
  if (s >= nsw) {
    if (kStopToRebuild && x == 0) job.stopped = 0;
    return;
  }
  bool stop = false;
  if (x == 0) {
    s_tombs = job.tombs;
    s_cut[0] = s_cut[1] = B;
  }
  for (uint32_t t = x; t <= kPrintMask; t += B) sm.print[t] = 0;
  window_sync<B>();
  // the first window's switch, and where its superstep ends
  uint2 cur = make_uint2(0, 0);
  uint32_t d = 0xFFFFu;
  if (s + x < nsw) {
    cur = __ldcs(&samp[s + x]);
    d = __ldcs(&dist[s + x]);
  }
  uint32_t par = 0;
  if constexpr (B > 32) {
    if (d <= x) atomicMin(&s_cut[0], x);
    __syncthreads();
  }
  while (s < nsw) {
    uint32_t n = min((uint32_t)B, nsw - s);
    if constexpr (B == 32) {
      const unsigned hit = __ballot_sync(0xffffffffu, d <= x);
      if (hit) n = min(n, (uint32_t)__ffs(hit) - 1);
    } else {
      n = min(n, s_cut[par]);
    }
    const uint32_t i = cur.x, j = cur.y & 0x7FFFFFFFu, g = cur.y >> 31;
    // sources, targets and the outright rules
    uint4 r1 = make_uint4(0, 0, 0, 0), r2 = r1;
    if (x < n) {
      r1 = list_load<kL1>(&E[i]);
      r2 = list_load<kL1>(&E[j]);
    }
    // the next window's switch, ahead of its use
    d = 0xFFFFu;
    if (s + n + x < nsw) {
      cur = __ldcs(&samp[s + n + x]);
      d = __ldcs(&dist[s + n + x]);
    }
    if (B > 32 && x == 0) s_cut[par ^ 1] = B;  // last read a superstep ago
    const unsigned long long e1 = rec_edge(r1), e2 = rec_edge(r2);
    unsigned long long e3 = 0, e4 = 0;
    uint32_t code = 1;
    if (x < n) {
      code = tau_g(g, e1, e2, e3, e4);
      if (code == kCodeLoop) ++rej_loop;
      else if (code) ++rej_exists;  // shared node: the targets re-create the sources
    }
    // presence of the targets (the loads in flight while the fingerprints go
    // in); a target's fingerprint is the high half of its hash
    const bool live = code == 0;
    bool dep = false;
    uint32_t pres = 0, h3 = 0, h4 = 0, at3 = kNil, at4 = kNil, own3 = 0, own4 = 0;
    unsigned long long was3 = kNoKey, was4 = kNoKey;  // what at3 and at4 held (kNoKey: no free slot was met)
    if (live) {
      const unsigned long long m3 = mix64(e3), m4 = mix64(e4);
      h3 = (uint32_t)m3;
      h4 = (uint32_t)m4;
      uint32_t s3 = h3 & mask, s4 = h4 & mask;
      unsigned long long c3 = set_load<kL1>(&H[s3]), c4 = set_load<kL1>(&H[s4]);
      const uint32_t f3 = (uint32_t)(m3 >> 32) | 1u, f4 = (uint32_t)(m4 >> 32) | 1u;
      own3 = f3 >> (32 - PL);
      for (;;) {
        const uint32_t old = atomicCAS(&sm.print[own3], 0u, f3);
        if (old == 0) break;
        if (old == f3) {
          dep = true;
          own3 = kNil;
          break;
        }
        own3 = (own3 + 1) & kPrintMask;
      }
      own4 = f4 >> (32 - PL);
      for (;;) {
        const uint32_t old = atomicCAS(&sm.print[own4], 0u, f4);
        if (old == 0) break;
        if (old == f4) {
          dep = true;
          own4 = kNil;
          break;
        }
        own4 = (own4 + 1) & kPrintMask;
      }
      // both searches advance together; each ends at its key (present) or at
      // an empty slot; at3, at4: the first slot that could take the key
      uint32_t done = 0;
      for (uint32_t q = 0; q <= mask; ++q) {
        if (!(done & 1u)) {
          if (c3 == e3) {
            pres |= 1u;
            done |= 1u;
          } else {
            if ((c3 == kEmptyKey || c3 == kTombKey) && at3 == kNil) {
              at3 = s3;
              was3 = c3;
            }
            if (c3 == kEmptyKey) done |= 1u;
            else s3 = (s3 + 1) & mask;
          }
        }
        if (!(done & 2u)) {
          if (c4 == e4) {
            pres |= 2u;
            done |= 2u;
          } else {
            if ((c4 == kEmptyKey || c4 == kTombKey) && at4 == kNil) {
              at4 = s4;
              was4 = c4;
            }
            if (c4 == kEmptyKey) done |= 2u;
            else s4 = (s4 + 1) & mask;
          }
        }
        if (done == 3u) break;
        if (!(done & 1u)) c3 = set_load<kL1>(&H[s3]);
        if (!(done & 2u)) c4 = set_load<kL1>(&H[s4]);
      }
      if (at3 == kNil) at3 = s3;  // present, or the table is full: insertion searches on from here
      if (at4 == kNil) at4 = s4;
    }
    window_sync<B>();
    if constexpr (B > 32) {  // where the next superstep ends, published by a barrier below
      if (d <= x) atomicMin(&s_cut[par ^ 1], x);
    }
    // a source that is some target of the superstep
    if (live) {
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const uint32_t f = (uint32_t)(mix64(w ? e2 : e1) >> 32) | 1u;
        uint32_t t = f >> (32 - PL);
        for (;;) {
          const uint32_t v = sm.print[t];
          if (v == 0) break;
          if (v == f) {
            dep = true;
            break;
          }
          t = (t + 1) & kPrintMask;
        }
      }
    }
    const bool some = window_any<B>(dep);
    if (live) {  // the fingerprints have been read
      if (own3 != kNil) sm.print[own3] = 0;
      if (own4 != kNil) sm.print[own4] = 0;
    }
    uint8_t dec = !live ? kEsIllegal : pres ? kEsIllegal : kEsLegal;
    if (some) {
      // erasers and inserters of the superstep, and the waves of Algorithm 1
      const uint32_t h1 = hash32(e1), h2 = hash32(e2);
      for (uint32_t t = x; t < (uint32_t)S; t += B) {
        sm.skey[t] = kEmptyKey;
        sm.ikey[t] = kEmptyKey;
        sm.ihead[t] = kNil;
      }
      if (x < n) sm.st[x] = live ? kEsUndecided : kEsIllegal;
      window_sync<B>();
      if (live) {
        uint32_t t = table_slot<S>(sm.skey, e1, h1, true);
        if (t != kNil) sm.sval[t] = x;
        t = table_slot<S>(sm.skey, e2, h2, true);
        if (t != kNil) sm.sval[t] = x;
        t = table_slot<S>(sm.ikey, e3, h3, true);
        if (t != kNil) sm.tnext[2 * x] = atomicExch(&sm.ihead[t], 2 * x);
        else atomicOr(err, kErrTableFull);
        t = table_slot<S>(sm.ikey, e4, h4, true);
        if (t != kNil) sm.tnext[2 * x + 1] = atomicExch(&sm.ihead[t], 2 * x + 1);
        else atomicOr(err, kErrTableFull);
      }
      window_sync<B>();
      // a switch decided in wave w only uses decisions of earlier waves
      dec = live ? kEsUndecided : kEsIllegal;
      for (uint32_t wave = 1;; ++wave) {
        if (dec == kEsUndecided) {
          bool bad = false, wait = false;
          for (uint32_t w = 0; w < 2 && !bad; ++w) {
            const unsigned long long e = w ? e4 : e3;
            const uint32_t h = w ? h4 : h3;
            if ((pres >> w) & 1u) {  // in E at the start: present unless an earlier legal switch erased it
              const uint32_t t = table_slot<S>(sm.skey, e, h, false);
              const uint32_t p = t == kNil ? kNil : sm.sval[t];
              if (p == kNil || p >= x || sm.st[p] == kEsIllegal) bad = true;
              else if (sm.st[p] == kEsUndecided) wait = true;
            }
            if (bad) break;
            const uint32_t t = table_slot<S>(sm.ikey, e, h, false);
            for (uint32_t q = t == kNil ? kNil : sm.ihead[t]; q != kNil; q = sm.tnext[q]) {
              const uint32_t k = q >> 1;  // an earlier switch that inserts e
              if (k >= x) continue;
              if (sm.st[k] == kEsLegal) {
                bad = true;
                break;
              }
              if (sm.st[k] == kEsUndecided) wait = true;
            }
          }
          dec = bad ? kEsIllegal : (wait ? kEsUndecided : kEsLegal);
        }
        window_sync<B>();  // every read of this wave's states is done
        if (x < n) sm.st[x] = dec;
        if (!window_any<B>(dec == kEsUndecided)) break;
        if (wave > (uint32_t)B) {  // every wave decides the smallest undecided switch: cannot happen
          if (x == 0) atomicOr(err, kErrNoProgress);
          return;
        }
      }
    }
    // apply: erase the sources where they are, insert the targets where their
    // searches ended, rewire.  In no particular order: an insertion only takes
    // empty slots and tombstones, and an erasure only its own edge's slot.
    uint32_t tombs = 0;
    const bool legal = dec == kEsLegal;
    if (legal) {
      H[r1.z] = kTombKey;
      H[r2.z] = kTombKey;
    }
    uint32_t t3 = was3 == kTombKey, t4 = was4 == kTombKey, p3 = at3, p4 = at4;
    if constexpr (B == 32) {
      warp_insert(H, mask, legal, e3, e4, p3, p4, was3 != kNoKey, was4 != kNoKey, t3, t4, err);
    } else if (legal) {
      const unsigned long long g3 = atomicCAS(&H[at3], was3, e3), g4 = atomicCAS(&H[at4], was4, e4);
      if (g3 != was3) p3 = hset_insert(H, mask, e3, at3, &t3);  // taken meanwhile, or no free slot was met
      if (g4 != was4) p4 = hset_insert(H, mask, e4, at4, &t4);
      if (p3 == kNil || p4 == kNil) atomicOr(err, kErrTableFull);
    }
    if (legal) {
      E[i] = make_rec(e3, p3 & mask);  // (no slot, a full table, was reported: stay in bounds)
      E[j] = make_rec(e4, p4 & mask);
      tombs = 2u - t3 - t4;
      ++acc;
    } else if (live) {
      ++rej_exists;
    }
    tombs = __reduce_add_sync(0xffffffffu, tombs);
    if ((x & 31u) == 0 && tombs) {
      if constexpr (B == 32) s_tombs += tombs;
      else atomicAdd(&s_tombs, tombs);
    }
    window_sync<B>();
    s += n;
    par ^= 1u;
    if constexpr (kStopToRebuild) {
      if (s_tombs > (mask >> 3)) {  // a rebuild on the whole GPU is cheap: keep the probe chains short
        stop = s < nsw;             // the same in every thread; the batch's end needs no rebuild yet
        if (stop) break;
      }
    } else {
      if (s_tombs > (mask >> 2)) {  // rebuild the set from the list on this CTA
        window_sync<B>();           // every thread has read the count
        for (uint32_t t = x; t <= mask; t += B) H[t] = kEmptyKey;
        window_sync<B>();
        for (uint32_t t = x; t < m; t += B) {
          const unsigned long long e = rec_edge(list_load<kL1>(&E[t]));
          uint32_t tomb;
          const uint32_t at = hset_insert(H, mask, e, hash32(e) & mask, &tomb);
          if (at == kNil) atomicOr(err, kErrTableFull);
          else E[t] = make_rec(e, at);
        }
        if (x == 0) s_tombs = 0;
        window_sync<B>();
      }
    }
  }
  if (x == 0) {  // progress of the job (the host launches it again while stopped)
    job.tombs = s_tombs;
    job.done = s;
    if constexpr (kStopToRebuild) {
      job.stopped = stop ? 1u : 0u;
      if (stop) atomicAdd(nstop, 1u);
    }
  }
  // counts of this job
  const unsigned a32 = __reduce_add_sync(0xffffffffu, acc);
  const unsigned l32 = __reduce_add_sync(0xffffffffu, rej_loop);
  const unsigned r32 = __reduce_add_sync(0xffffffffu, rej_exists);
  if ((x & 31) == 0) {
    if (a32) {
      atomicAdd(&stats->accepted, (unsigned long long)a32);
      atomicAdd(&chain_acc[job.chain], (unsigned long long)a32);
    }
    if (l32) atomicAdd(&stats->rej_loop, (unsigned long long)l32);
    if (r32) atomicAdd(&stats->rej_exists, (unsigned long long)r32);
  }
}

// ---------------------------------------------------------------- small chains
// Chains of few edges or nodes, one warp each with the list and the set in
// shared memory (16-bit node ids: a word per edge).
// Their supersteps hold a handful of switches (five in a chain of 65 edges), so
// a pool's time is that of its smallest chains' dependent accesses: with list
// and set in L1 and L2 a superstep took 2.6 us, with the bits 0.35 (a chain of
// 1,000 edges: 6.0 and 0.6; with a hash table in shared memory 2.8: its loops
// are what takes the instructions).  As on the cluster
// below, a superstep ends before a switch that depends on an earlier one (the
// same target, found where both insert it, or a present target that an earlier
// switch erases, found by its slot), so it needs no tables and waves.
// Chains whose pairs of nodes fit as bits have the set as a bit matrix (no search,
// no tombstones), others of at most kEsSmallestEdges edges as a hash table.  The
// bit matrices run in three launches, by the shared memory they need (nine,
// three and one CTA an SM).
constexpr uint32_t kEsSmallestEdges = 2048;
constexpr uint32_t kEsBitMax = 220 << 10, kEsBitBytes[3] = {24 << 10, 72 << 10, kEsBitMax};
// Bytes of the bits of all pairs below n nodes and of a list of m edges.
__host__ __device__ inline unsigned long long bits_bytes(uint32_t m, unsigned long long n) {
  return 4 * ((n * (n - 1) / 2 + 31) / 32 + m);
}
constexpr uint32_t kEmpty32 = 0xFFFFFFFFu, kTomb32 = 0xFFFFFFFEu;  // no edges (not canonical)

__host__ __device__ inline uint32_t small_log2(uint32_t m) {  // at least four slots per edge
  uint32_t h = 10;
  while ((1u << h) < 4 * m) ++h;
  return h;
}

// Samples of a warp's chain, 32 a register: the window at s from the first two by
// shuffles, the third on its way (loaded where they are used, they would cost
// an access to L2 or memory a superstep).
struct SampleRing {
  uint2 c[3];
  uint32_t d[3], base;
  __device__ __forceinline__ void load(int v, uint32_t from, uint32_t nsw, const uint2 *samp, const uint16_t *dist) {
    c[v] = make_uint2(0, 0);
    d[v] = 0xFFFFu;
    const uint32_t k = from + threadIdx.x;
    if (k < nsw) {
      c[v] = __ldg(&samp[k]);
      d[v] = __ldg(&dist[k]);
    }
  }
  __device__ __forceinline__ void start(uint32_t nsw, const uint2 *samp, const uint16_t *dist) {
    base = 0;
#pragma unroll
    for (int v = 0; v < 3; ++v) load(v, 32 * v, nsw, samp, dist);
  }
  // The lane's switch of the window at s (at most 32 past the last one) and its distance.
  __device__ __forceinline__ uint2 window(uint32_t s, uint32_t nsw, const uint2 *samp, const uint16_t *dist,
                                          uint32_t &dd) {
    if (s - base >= 32) {
      c[0] = c[1];
      d[0] = d[1];
      c[1] = c[2];
      d[1] = d[2];
      base += 32;
      load(2, base + 64, nsw, samp, dist);
    }
    const uint32_t at = s - base + threadIdx.x;
    const uint32_t x0 = __shfl_sync(0xffffffffu, c[0].x, at), y0 = __shfl_sync(0xffffffffu, c[0].y, at);
    const uint32_t x1 = __shfl_sync(0xffffffffu, c[1].x, at), y1 = __shfl_sync(0xffffffffu, c[1].y, at);
    const uint32_t e0 = __shfl_sync(0xffffffffu, d[0], at), e1 = __shfl_sync(0xffffffffu, d[1], at);
    dd = at < 32 ? e0 : e1;
    return at < 32 ? make_uint2(x0, y0) : make_uint2(x1, y1);
  }
};

// The list of a small chain into shared memory (a word per edge), and back.
__device__ __forceinline__ void load_small(uint32_t *E, const uint4 *list, uint32_t m) {
#pragma unroll 8
  for (uint32_t t = threadIdx.x; t < m; t += 32) {
    const uint2 r = *reinterpret_cast<const uint2 *>(&list[t]);
    E[t] = (r.y << 16) | (r.x & 0xFFFFu);
  }
}
__device__ __forceinline__ void store_small(uint4 *list, const uint32_t *E, uint32_t m) {
  for (uint32_t t = threadIdx.x; t < m; t += 32) list[t] = make_uint4(E[t] & 0xFFFFu, E[t] >> 16, 0u, 0u);
}

// A warp's counts of its chain's switches.
__device__ __forceinline__ void count_small(const EsJob &job, uint32_t acc, uint32_t rej_loop, uint32_t rej_exists,
                                            StatsDev *stats, unsigned long long *chain_acc) {
  const unsigned a32 = __reduce_add_sync(0xffffffffu, acc);
  const unsigned l32 = __reduce_add_sync(0xffffffffu, rej_loop);
  const unsigned r32 = __reduce_add_sync(0xffffffffu, rej_exists);
  if (threadIdx.x == 0) {
    if (a32) {
      atomicAdd(&stats->accepted, (unsigned long long)a32);
      atomicAdd(&chain_acc[job.chain], (unsigned long long)a32);
    }
    if (l32) atomicAdd(&stats->rej_loop, (unsigned long long)l32);
    if (r32) atomicAdd(&stats->rej_exists, (unsigned long long)r32);
  }
}

// The set as a bit matrix: the bit of {u, v}, u < v, at v (v - 1) / 2 + u.
__global__ void __launch_bounds__(32) k_es_run_bits(EsJob *jobs, uint32_t job_off, uint32_t nsw, const uint2 *samples,
                                                    const uint16_t *dists, StatsDev *stats,
                                                    unsigned long long *chain_acc, uint32_t *err) {
  extern __shared__ uint32_t small_dyn[];
  dep_launch();
  const EsJob &job = jobs[job_off + blockIdx.x];
  const uint32_t x = threadIdx.x, m = job.m;
  if (m >= 2 && bits_bytes(m, job.n) <= kEsBitMax) {  // the host sends only chains that qualify
    const uint32_t words = (job.n * (job.n - 1) / 2 + 31) / 32;
    uint32_t *const M = small_dyn, *const E = M + words;
    const uint2 *const samp = samples + (size_t)job.row * nsw;
    const uint16_t *const dist = dists + (size_t)job.row * nsw;
    SampleRing ring;
    ring.start(nsw, samp, dist);
    load_small(E, job.E, m);
    for (uint32_t t = x; t < words; t += 32) M[t] = 0;
    __syncwarp();
    auto pair = [](uint32_t e) {  // (0 for the 0 of a lane without a switch)
      const uint32_t v = e & 0xFFFFu;
      return v * (v - 1) / 2 + (e >> 16);
    };
    for (uint32_t t = x; t < m; t += 32) {
      const uint32_t b = pair(E[t]);
      atomicOr(&M[b >> 5], 1u << (b & 31u));
    }
    __syncwarp();
    uint32_t acc = 0, rej_loop = 0, rej_exists = 0;
    for (uint32_t s = 0; s < nsw;) {
      uint32_t d;
      const uint2 cur = ring.window(s, nsw, samp, dist, d);
      uint32_t n = min(32u, nsw - s);
      const unsigned hit = __ballot_sync(0xffffffffu, d <= x);
      if (hit) n = min(n, (uint32_t)__ffs(hit) - 1);
      const uint32_t i = cur.x, j = cur.y & 0x7FFFFFFFu, g = cur.y >> 31;
      uint32_t e1 = 0, e2 = 0, e3 = 0, e4 = 0, code = kCodeLazy;
      if (x < n) {
        e1 = E[i];
        e2 = E[j];
        code = tau16(g, e1, e2, e3, e4);
      }
      const bool live = code == 0;
      const uint32_t i3 = pair(e3), i4 = pair(e4), w3 = i3 >> 5, w4 = i4 >> 5;
      const uint32_t b3 = 1u << (i3 & 31u), b4 = 1u << (i4 & 31u);
      bool p3 = false, p4 = false;  // present
      if (live) {
        p3 = (M[w3] & b3) != 0;
        p4 = (M[w4] & b4) != 0;
      }
      // the superstep ends before the first switch with a present target that
      // an earlier one erases
      uint32_t end = n;
      for (unsigned who = __ballot_sync(0xffffffffu, p3 || p4); who; who &= who - 1) {
        const int w = __ffs(who) - 1;
        const uint32_t k3 = __shfl_sync(0xffffffffu, p3 ? e3 : 0u, w), k4 = __shfl_sync(0xffffffffu, p4 ? e4 : 0u, w);
        const bool erases = live && (int)x < w && (e1 == k3 || e2 == k3 || e1 == k4 || e2 == k4);
        if (__any_sync(0xffffffffu, erases)) {
          end = min(end, (uint32_t)w);
          break;
        }
      }
      const bool clear = live && !p3 && !p4 && x < end;
      __syncwarp();
      bool o3 = false, o4 = false;  // this lane set the bit
      if (clear) {
        o3 = !(atomicOr(&M[w3], b3) & b3);
        o4 = !(atomicOr(&M[w4], b4) & b4);
      }
      // a bit that another lane has set: the superstep ends before this switch
      const unsigned two = __ballot_sync(0xffffffffu, clear && !(o3 && o4));
      if (two) {
        end = min(end, max(1u, (uint32_t)__ffs(two) - 1));
        if (clear && x >= end) {  // what it set is taken back
          if (o3) atomicAnd(&M[w3], ~b3);
          if (o4) atomicAnd(&M[w4], ~b4);
        }
        __syncwarp();
        if (clear && x == 0) {  // (the first switch always runs: another's bit may have been its own)
          atomicOr(&M[w3], b3);
          atomicOr(&M[w4], b4);
        }
      }
      if (x < end) {
        if (clear) {
          const uint32_t i1 = pair(e1), i2 = pair(e2);
          atomicAnd(&M[i1 >> 5], ~(1u << (i1 & 31u)));
          atomicAnd(&M[i2 >> 5], ~(1u << (i2 & 31u)));
          E[i] = e3;
          E[j] = e4;
          ++acc;
        } else if (code == kCodeLoop) {
          ++rej_loop;
        } else {
          ++rej_exists;
        }
      }
      s += end;
      __syncwarp();
    }
    store_small(job.E, E, m);
    count_small(job, acc, rej_loop, rej_exists, stats, chain_acc);
  }
  dep_wait();
}

// Insert a key from slot s on, which held `was` when its search ended; as
// insert_once.
__device__ __forceinline__ uint32_t insert_small(uint32_t *H, uint32_t mask, uint32_t key, uint32_t s, uint32_t was,
                                                 uint32_t *tomb, bool first, bool *twice, bool *full) {
  for (uint32_t n = 0; n <= mask; ++n) {
    if (was >= kTomb32) {
      const uint32_t got = atomicCAS(&H[s], was, key);
      if (got == was) {
        *tomb = was == kTomb32 ? 1u : 0u;
        return s;
      }
      was = got;
      continue;
    }
    if (was == key) {
      *twice = true;
      if (!first) return kNil;
    }
    s = (s + 1) & mask;
    was = H[s];
  }
  *full = true;
  return kNil;
}

__global__ void __launch_bounds__(32) k_es_run_small(EsJob *jobs, uint32_t job_off, uint32_t nsw, const uint2 *samples,
                                                     const uint16_t *dists, StatsDev *stats,
                                                     unsigned long long *chain_acc, uint32_t *err) {
  extern __shared__ uint32_t small_dyn[];
  dep_launch();
  EsJob &job = jobs[job_off + blockIdx.x];
  const uint32_t x = threadIdx.x, m = job.m, hlog2 = small_log2(m), mask = (1u << hlog2) - 1;
  if (m < 2 || m > kEsSmallestEdges) {  // the host sends only chains that qualify
    dep_wait();
    return;
  }
  uint32_t *const H = small_dyn, *const E = H + mask + 1;
  uint16_t *const slot = reinterpret_cast<uint16_t *>(E + m);  // of the edge at each position
  uint4 *const list = job.E;
  const uint2 *const samp = samples + (size_t)job.row * nsw;
  const uint16_t *const dist = dists + (size_t)job.row * nsw;
  SampleRing ring;
  ring.start(nsw, samp, dist);
  bool full = false;
  load_small(E, list, m);
  auto build = [&] {
    for (uint32_t t = x; t <= mask / 4; t += 32) reinterpret_cast<uint4 *>(H)[t] = make_uint4(~0u, ~0u, ~0u, ~0u);
    __syncwarp();
    for (uint32_t t = x; t < m; t += 32) {
      uint32_t tomb;
      bool twice = false;
      const uint32_t s = (E[t] * 0x9E3779B1u) >> (32 - hlog2);
      slot[t] = (uint16_t)insert_small(H, mask, E[t], s, H[s], &tomb, false, &twice, &full);
    }
    __syncwarp();
  };
  build();
  uint32_t acc = 0, rej_loop = 0, rej_exists = 0, tombs = 0;
  for (uint32_t s = 0; s < nsw;) {
    uint32_t d;
    const uint2 cur = ring.window(s, nsw, samp, dist, d);
    uint32_t n = min(32u, nsw - s);
    const unsigned hit = __ballot_sync(0xffffffffu, d <= x);
    if (hit) n = min(n, (uint32_t)__ffs(hit) - 1);
    const uint32_t i = cur.x, j = cur.y & 0x7FFFFFFFu, g = cur.y >> 31;
    uint32_t e3 = 0, e4 = 0, s1 = kNil, s2 = kNil, code = kCodeLazy;
    if (x < n) {
      const uint32_t e1 = E[i], e2 = E[j];
      s1 = slot[i] & mask;  // (a full table, which would have been reported: stay in bounds)
      s2 = slot[j] & mask;
      code = tau16(g, e1, e2, e3, e4);
    }
    const bool live = code == 0;
    // present targets' slots, and where the others can go
    uint32_t q3 = kNil, q4 = kNil, a3 = kNil, a4 = kNil, was3 = 0, was4 = 0;
    if (live) {
      uint32_t t = (e3 * 0x9E3779B1u) >> (32 - hlog2);
      for (uint32_t v = 0; v <= mask; ++v, t = (t + 1) & mask) {
        const uint32_t c = H[t];
        if (c == e3) {
          q3 = t;
          break;
        }
        if (c >= kTomb32 && a3 == kNil) {
          a3 = t;
          was3 = c;
        }
        if (c == kEmpty32) break;
      }
      t = (e4 * 0x9E3779B1u) >> (32 - hlog2);
      for (uint32_t v = 0; v <= mask; ++v, t = (t + 1) & mask) {
        const uint32_t c = H[t];
        if (c == e4) {
          q4 = t;
          break;
        }
        if (c >= kTomb32 && a4 == kNil) {
          a4 = t;
          was4 = c;
        }
        if (c == kEmpty32) break;
      }
    }
    // the superstep ends before the first switch with a present target that an
    // earlier one erases
    uint32_t end = n;
    for (unsigned who = __ballot_sync(0xffffffffu, q3 != kNil || q4 != kNil); who; who &= who - 1) {
      const int w = __ffs(who) - 1;
      const uint32_t t3 = __shfl_sync(0xffffffffu, q3, w), t4 = __shfl_sync(0xffffffffu, q4, w);
      const bool erases = live && (int)x < w && ((s1 == t3 || s2 == t3) || (s1 == t4 || s2 == t4));
      if (__any_sync(0xffffffffu, erases)) {
        end = min(end, (uint32_t)w);
        break;  // (the first such switch)
      }
    }
    const bool clear = live && q3 == kNil && q4 == kNil && x < end;
    uint32_t p3 = kNil, p4 = kNil, t3 = 0, t4 = 0;
    bool twice = false;
    __syncwarp();
    if (clear) {
      p3 = insert_small(H, mask, e3, a3, was3, &t3, x == 0, &twice, &full);
      p4 = insert_small(H, mask, e4, a4, was4, &t4, x == 0, &twice, &full);
    }
    const unsigned two = __ballot_sync(0xffffffffu, twice);
    if (two) end = min(end, max(1u, (uint32_t)__ffs(two) - 1));
    uint32_t dead = 0;
    if (clear && x < end) {
      H[s1] = kTomb32;
      H[s2] = kTomb32;
      E[i] = e3;
      E[j] = e4;
      slot[i] = (uint16_t)p3;
      slot[j] = (uint16_t)p4;
      dead = 2u - t3 - t4;
      ++acc;
    } else if (clear) {  // past the end: its insertions become tombstones
      if (p3 != kNil) {
        H[p3] = kTomb32;
        dead += 1u - t3;
      }
      if (p4 != kNil) {
        H[p4] = kTomb32;
        dead += 1u - t4;
      }
    }
    if (x < end && !clear) {
      if (code == kCodeLoop) ++rej_loop;
      else ++rej_exists;
    }
    s += end;
    tombs += __reduce_add_sync(0xffffffffu, dead);
    __syncwarp();
    if (tombs > (mask >> 3)) {
      build();
      tombs = 0;
    }
  }
  store_small(list, E, m);
  if (__any_sync(0xffffffffu, full) && x == 0) atomicOr(err, kErrTableFull);
  count_small(job, acc, rej_loop, rej_exists, stats, chain_acc);
  dep_wait();
}

// ---------------------------------------------------------------- large chains
// One chain on a cluster of kClusterCtas CTAs, for chains of at least
// kEsBigChain edges (windows of 1024 switches, thread x of CTA r holding switch
// r * T + x): one SM moves about one 32-byte sector to or from L2 every two
// cycles, and a window's switches need some 9,000, so that one CTA took 8.9 us
// a superstep (7.2 ms for 2^19 switches of a chain of 1.05e6 edges); so, 6.2 us
// (5.1 ms).  What is left is one superstep's chain of dependent accesses to L2
// (sources, set, insertion, the stores' way there) and three cluster barriers.
//
// The CTAs exchange almost nothing: every CTA finds the cut by itself, and the
// list and the set are in L2.  A superstep is
//   1. gather the sources, search the set for the targets; a present target is
//      an event, told to every CTA (its id and its switch);
//   2. insert the targets of the switches with none present, each where its
//      search ended.  Two switches with the same target meet in the same slot;
//      the later to get there ends the superstep before its own switch.  A
//      switch whose source is a later switch's present target ends it before
//      that one.  (A target's eraser that comes after the switch is no matter:
//      the edge is there when the switch runs.)
//   3. the switches before that end are independent of one another: those with
//      a present target are illegal, the others legal; they rewire and erase,
//      and the ones past the end take their insertions back as tombstones.
// Any cut into runs without a shared position gives the sequential result; the
// first switch always runs.
constexpr int kClusterCtas = 8;
constexpr uint32_t kEvents = 128;  // present targets of a superstep that are told apart
// Present targets a superstep on average (a graph with large hubs) from which
// on the chain is left to one CTA and its waves: the events cost every switch a
// comparison, and past kEvents of them end the superstep (a power law of 1.7e6
// edges with exponent 2.2, 1e5 switches: 3.7 ms here, 1.7 there).
constexpr uint32_t kBusyEvents = 16;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The same where only the threads with `told` have written anything that the
// other CTAs read next: the others need no fence (a release by every thread
// waits for all its stores and atomics on L2).
__device__ __forceinline__ void cluster_sync_told(bool told) {
  if (told) asm volatile("fence.acq_rel.cluster;" ::: "memory");
  asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The address in CTA `rank`'s shared memory of what is at `p` in this CTA's.
__device__ __forceinline__ uint32_t peer_addr(const void *p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t peer_add(uint32_t *p, uint32_t rank, uint32_t v) {
  uint32_t old;
  asm volatile("atom.relaxed.cluster.shared::cluster.add.u32 %0, [%1], %2;"
               : "=r"(old)
               : "r"(peer_addr(p, rank)), "r"(v)
               : "memory");
  return old;
}
// min / max / add into the same word of every CTA of the cluster.
__device__ __forceinline__ void all_min(uint32_t *p, uint32_t v) {
#pragma unroll 1
  for (uint32_t r = 0; r < kClusterCtas; ++r)
    asm volatile("red.relaxed.cluster.shared::cluster.min.u32 [%0], %1;" ::"r"(peer_addr(p, r)), "r"(v) : "memory");
}
__device__ __forceinline__ void all_max(uint32_t *p, uint32_t v) {
#pragma unroll 1
  for (uint32_t r = 0; r < kClusterCtas; ++r)
    asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" ::"r"(peer_addr(p, r)), "r"(v) : "memory");
}
__device__ __forceinline__ void all_add(uint32_t *p, uint32_t v) {
#pragma unroll 1
  for (uint32_t r = 0; r < kClusterCtas; ++r)
    asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(peer_addr(p, r)), "r"(v) : "memory");
}
__device__ __forceinline__ void all_store(unsigned long long *p, unsigned long long v) {
#pragma unroll 1
  for (uint32_t r = 0; r < kClusterCtas; ++r)
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(peer_addr(p, r)), "l"(v) : "memory");
}

// Search for a key from slot s on: whether it is in the set, else the first
// slot that could take it and what that held.
struct SetSearch {
  uint32_t s, at;
  unsigned long long was;
  bool present, done;
};
// One aligned group of four slots, a sector of L2 (the sets have 2^h >= 4 slots
// and start on 256 bytes).
struct Four {
  unsigned long long v[4];
};
__device__ __forceinline__ Four load_four(const unsigned long long *p) {
  Four f;
  asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(f.v[0]), "=l"(f.v[1]) : "l"(p) : "memory");
  asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(f.v[2]), "=l"(f.v[3]) : "l"(p + 2) : "memory");
  return f;
}
// The search over the group that holds slot q.s, from there on.
__device__ __forceinline__ void search_step(SetSearch &q, unsigned long long key, const Four &f, uint32_t mask) {
  const uint32_t from = q.s & 3u;
#pragma unroll
  for (uint32_t v = 0; v < 4; ++v) {
    if (v < from || q.done) continue;
    const unsigned long long cur = f.v[v];
    if (cur == key) {
      q.present = q.done = true;
      continue;
    }
    if ((cur == kEmptyKey || cur == kTombKey) && q.at == kNil) {
      q.at = (q.s & ~3u) + v;
      q.was = cur;
    }
    if (cur == kEmptyKey) q.done = true;
  }
  q.s = ((q.s & ~3u) + 4) & mask;
}

// Insert a key from slot s on, where a search ended; stops at the key itself,
// which another switch of the superstep has put there (*twice), or, for the
// superstep's first switch, takes the next free slot (the other switch will
// take its own back).  Returns the slot, or kNil if the table is full or the key
// was there.
__device__ __forceinline__ uint32_t insert_once(unsigned long long *H, uint32_t mask, unsigned long long key, uint32_t s,
                                                unsigned long long was, uint32_t *tomb, bool first, bool *twice, bool *full) {
  for (uint32_t n = 0; n <= mask; ++n) {
    if (was == kEmptyKey || was == kTombKey) {
      const unsigned long long got = atomicCAS(&H[s], was, key);
      if (got == was) {
        *tomb = was == kTombKey ? 1u : 0u;
        return s;
      }
      was = got;  // taken meanwhile: look at what is there now
      continue;
    }
    if (was == key) {
      *twice = true;
      if (!first) return kNil;
    }
    s = (s + 1) & mask;
    was = __ldcg(&H[s]);
  }
  *full = true;
  return kNil;
}

template <int T>
__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(T)
    k_es_run_cluster(EsJob *jobs, uint32_t job_off, uint32_t nsw, const uint2 *samples, const uint16_t *dists, StatsDev *stats,
                 unsigned long long *chain_acc, uint32_t *err, uint32_t *nstop) {
  constexpr uint32_t B = T * kClusterCtas;  // the window
  constexpr int kDist = kClusterCtas;       // distances a thread looks at for the cut
  // per parity of the superstep: events (told so far, in CTA 0: asked for), the
  // end they force, this CTA's tombstones; and the cuts of three supersteps, the
  // running one's, the next one's, and the one after that's, which is set up
  __shared__ uint32_t s_events[2], s_asked[2], s_end[2], s_mine[2], s_cut[3], s_tombs;
  __shared__ unsigned long long s_key[2][kEvents], s_who[2][kEvents];
  EsJob &job = jobs[job_off + blockIdx.x / kClusterCtas];
  const uint32_t rank = cluster_rank(), tid = threadIdx.x, x = rank * T + tid;
  uint4 *const E = job.E;
  unsigned long long *const H = job.H;
  const uint2 *const samp = samples + (size_t)job.row * nsw;
  const uint16_t *const dist = dists + (size_t)job.row * nsw;
  const uint32_t mask = (uint32_t)((1ull << job.hlog2) - 1), limit = mask >> 3;
  uint32_t s = job.done, acc = 0, rej_loop = 0, rej_exists = 0, tomb_total = 0;
  if (job.alone || s >= nsw) {  // (the same in every CTA of the cluster)
    if (x == 0 && !job.alone) job.stopped = 0;
    return;
  }
  if (tid < 2) {
    s_events[tid] = s_asked[tid] = s_mine[tid] = 0;
    s_end[tid] = B;
  }
  if (tid < 3) s_cut[tid] = B;
  if (tid == 0) s_tombs = job.tombs;
  uint2 cur;
  uint32_t d[kDist];
  // the window from s on: the thread's own switch, and its share of the
  // distances (the same in every CTA: the cut needs all of them)
  auto load_window = [&](uint32_t from) {
    cur = from + x < nsw ? __ldg(&samp[from + x]) : make_uint2(0, 0);
#pragma unroll
    for (int v = 0; v < kDist; ++v) {
      const uint32_t k = from + tid + v * T;
      d[v] = k < nsw ? __ldg(&dist[k]) : 0xFFFFu;
    }
  };
  auto find_cut = [&](uint32_t *cut) {
    uint32_t c = B;
#pragma unroll
    for (int v = kDist - 1; v >= 0; --v)
      if (d[v] <= tid + v * T) c = tid + v * T;
    c = __reduce_min_sync(0xffffffffu, c);
    if ((tid & 31u) == 0 && c < B) atomicMin(cut, c);
  };
  load_window(s);
  __syncthreads();
  find_cut(&s_cut[0]);
  cluster_sync();  // (every CTA's shared memory is set up)
  uint32_t stop = 0, steps = 0, met = 0;
  uint32_t cut = 0, next_cut = 1, last_cut = 2;
  for (uint32_t par = 0;; par ^= 1u) {
    const uint32_t n = min(min(B, nsw - s), s_cut[cut]);
    const uint32_t i = cur.x, j = cur.y & 0x7FFFFFFFu, g = cur.y >> 31;
    uint4 r1 = make_uint4(0, 0, 0, 0), r2 = r1;
    if (x < n) {
      r1 = __ldcg(&E[i]);
      r2 = __ldcg(&E[j]);
    }
    load_window(s + n);
    const unsigned long long e1 = rec_edge(r1), e2 = rec_edge(r2);
    unsigned long long e3 = 0, e4 = 0;
    const uint32_t code = x < n ? tau_g(g, e1, e2, e3, e4) : kCodeLazy;
    SetSearch q3 = {0, kNil, kNoKey, false, true}, q4 = q3;
    bool told = false;
    if (code == 0) {
      q3.s = hash32(e3) & mask;
      q4.s = hash32(e4) & mask;
      q3.done = q4.done = false;
      for (uint32_t v = 0; v <= mask && !(q3.done && q4.done); ++v) {
        Four c3, c4;
        if (!q3.done) c3 = load_four(&H[q3.s & ~3u]);
        if (!q4.done) c4 = load_four(&H[q4.s & ~3u]);
        if (!q3.done) search_step(q3, e3, c3, mask);
        if (!q4.done) search_step(q4, e4, c4, mask);
      }
      // present targets: told to every CTA; without room for them the
      // superstep ends before this switch
      for (int w = 0; w < 2; ++w) {
        if (!(w ? q4.present : q3.present)) continue;
        told = true;
        const uint32_t at = peer_add(&s_asked[par], 0, 1u);
        if (at < kEvents) {
          all_store(&s_key[par][at], w ? e4 : e3);
          all_store(&s_who[par][at], x);
          all_max(&s_events[par], at + 1);
        } else {
          all_min(&s_end[par], x ? x : 1u);
        }
      }
    }
    cluster_sync_told(told);
    // erasers of present targets, and the insertions
    told = false;
    const bool live = code == 0, clear = live && !q3.present && !q4.present;
    const uint32_t events = s_events[par];
    if (live) {
      for (uint32_t v = 0; v < events; ++v) {
        const uint32_t who = (uint32_t)s_who[par][v];
        const unsigned long long key = s_key[par][v];
        if (x < who && (key == e1 || key == e2)) {
          all_min(&s_end[par], who);
          told = true;
        }
      }
    }
    uint32_t p3 = kNil, p4 = kNil, t3 = 0, t4 = 0;
    if (clear) {
      bool twice = false, full = false;
      p3 = insert_once(H, mask, e3, q3.at, q3.was, &t3, x == 0, &twice, &full);
      p4 = insert_once(H, mask, e4, q4.at, q4.was, &t4, x == 0, &twice, &full);
      if (twice) all_min(&s_end[par], x ? x : 1u);
      told |= twice;
      if (full) atomicOr(err, kErrTableFull);
    }
    cluster_sync_told(told);
    const uint32_t end = min(n, s_end[par]);
    uint32_t tombs = 0;
    if (clear && x < end) {
      H[r1.z] = kTombKey;
      H[r2.z] = kTombKey;
      E[i] = make_rec(e3, p3 & mask);  // (no slot, a full table, was reported: stay in bounds)
      E[j] = make_rec(e4, p4 & mask);
      tombs = 2u - t3 - t4;
      ++acc;
    } else if (clear) {  // past the end: its insertions become tombstones
      if (p3 != kNil) {
        H[p3] = kTombKey;
        tombs += 1u - t3;
      }
      if (p4 != kNil) {
        H[p4] = kTombKey;
        tombs += 1u - t4;
      }
    }
    if (x < end && !clear) {
      if (code == kCodeLoop) ++rej_loop;
      else ++rej_exists;  // a shared node (the targets re-create the sources) or a present target
    }
    if (end < n) load_window(s + end);
    find_cut(&s_cut[next_cut]);
    tombs = __reduce_add_sync(0xffffffffu, tombs);
    if ((tid & 31u) == 0 && tombs) {
      tomb_total += tombs;
      atomicAdd(&s_mine[par], tombs);
    }
    if (tid == 0) {
      // the superstep before this one's tombstones to every CTA, and its words
      // for the next one (here, since the barriers above order nothing but what
      // was told)
      const uint32_t mine = s_mine[par ^ 1];
      if (mine) all_add(&s_tombs, mine);
      s_mine[par ^ 1] = s_events[par ^ 1] = s_asked[par ^ 1] = 0;
      s_end[par ^ 1] = B;
      s_cut[last_cut] = B;
    }
    const uint32_t freed = cut;
    cut = next_cut;
    next_cut = last_cut;
    last_cut = freed;
    s += end;
    ++steps;
    met += events;
    cluster_sync();
    if (s >= nsw) break;
    if (s_tombs > limit) {  // a rebuild on the whole GPU is cheap: keep the probe chains short
      stop = 1;             // (the same in every CTA)
      break;
    }
    if (steps >= 4 && met > kBusyEvents * steps) {
      stop = 2;
      break;
    }
  }
  if (tomb_total) atomicAdd(&job.tombs, tomb_total);
  if (x == 0) {  // progress of the job (the host launches it again while stopped)
    job.done = s;
    job.stopped = stop;
    if (stop == 2) job.alone = 1;
    if (stop) atomicAdd(nstop, 1u);
  }
  // counts of this job
  const unsigned a32 = __reduce_add_sync(0xffffffffu, acc);
  const unsigned l32 = __reduce_add_sync(0xffffffffu, rej_loop);
  const unsigned r32 = __reduce_add_sync(0xffffffffu, rej_exists);
  if ((tid & 31) == 0) {
    if (a32) {
      atomicAdd(&stats->accepted, (unsigned long long)a32);
      atomicAdd(&chain_acc[job.chain], (unsigned long long)a32);
    }
    if (l32) atomicAdd(&stats->rej_loop, (unsigned long long)l32);
    if (r32) atomicAdd(&stats->rej_exists, (unsigned long long)r32);
  }
}

// Windows of 32, 128 and 256 switches (the set rebuilt in place).
template <int B, int MIN_BLOCKS>
__global__ void __launch_bounds__(B, MIN_BLOCKS) k_es_run(EsJob *jobs, uint32_t job_off, uint32_t nsw,
                                                          const uint2 *samples, const uint16_t *dists,
                                                          StatsDev *stats, unsigned long long *chain_acc,
                                                          uint32_t *err) {
  dep_launch();
  es_run_body<B, false>(jobs, job_off, nsw, samples, dists, stats, chain_acc, err, nullptr);
  dep_wait();
}

// Windows of 1024 switches on one CTA (chains of at least 2^19 edges that the
// cluster left: the set rebuilt on the whole GPU between launches).
__global__ void __launch_bounds__(1024, 1) k_es_run_big(EsJob *jobs, uint32_t job_off, uint32_t nsw,
                                                        const uint2 *samples, const uint16_t *dists, StatsDev *stats,
                                                        unsigned long long *chain_acc, uint32_t *err,
                                                        uint32_t *nstop) {
  es_run_body<1024, true>(jobs, job_off, nsw, samples, dists, stats, chain_acc, err, nstop);
}

}  // namespace

uint32_t es_group(uint32_t m, uint64_t n) {
  if (m >= kEsBigChain) return 0;
  if (m >= kEsMidChain) return 1;
  if (m >= kEsSmallChain) return 2;
  for (uint32_t v = 0; v < 3; ++v)
    if (n <= 65536 && bits_bytes(m, n) <= kEsBitBytes[v]) return 7 - v;
  return m <= kEsSmallestEdges && n <= 65536 ? 4 : 3;
}

uint32_t es_smem_bytes(uint32_t m, uint32_t n) {
  const uint32_t g = es_group(m, n);
  if (g < 4) return 0;
  return g == 4 ? (4u << small_log2(m)) + 4 * m + 2 * m + 2 : (uint32_t)bits_bytes(m, n);
}

cudaError_t prepare_es_kernels() {
  cudaError_t f = cudaFuncSetAttribute(k_es_run_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)es_smem_bytes(kEsSmallestEdges, 65536));
  if (f == cudaSuccess)
    f = cudaFuncSetAttribute(k_es_run_bits, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kEsBitBytes[2]);
  if (f != cudaSuccess) return f;
  cudaError_t e = cudaFuncSetAttribute(k_es_run_big, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)EsShape<1024>::kBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_es_run<256, 6>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)EsShape<256>::kBytes);
}

cudaError_t launch_es_set(EsJob *jobs, uint32_t njobs, uint32_t *err, cudaStream_t s, int num_sms, bool rebuild,
                          uint64_t *launches) {
  for (uint32_t off = 0; off < njobs; off += 65535u) {
    const uint32_t nj = njobs - off < 65535u ? njobs - off : 65535u;
    const uint32_t gx = (uint32_t)((num_sms * 8 + nj - 1) / nj);
    const dim3 grid(gx < 1 ? 1 : gx, nj);
    k_es_clear<<<grid, 256, 0, s>>>(jobs, off, rebuild);
    if (rebuild) k_es_fill<<<grid, 256, 0, s>>>(jobs, off, err);
    *launches += rebuild ? 2 : 1;
  }
  return cudaGetLastError();
}

cudaError_t launch_es_sample(EsJob *jobs, const uint32_t (&group)[kEsGroups], unsigned long long off, uint32_t n,
                             uint2 *samples, uint16_t *dists, cudaStream_t s, uint32_t *launches) {
  uint32_t beg = 0;
  for (int w = 0; w < (int)kEsGroups; ++w) {
    for (uint32_t o = beg; o < beg + group[w]; o += 65535u, ++*launches) {
      const uint32_t nj = beg + group[w] - o < 65535u ? beg + group[w] - o : 65535u;
      if (w == 0) k_es_sample<1024, 1024><<<dim3((n + 1023) / 1024, nj), 1024, 0, s>>>(jobs, o, off, n, samples, dists);
      else if (w == 1) k_es_sample<256, 512><<<dim3((n + 511) / 512, nj), 512, 0, s>>>(jobs, o, off, n, samples, dists);
      else if (w == 2) k_es_sample<128, 256><<<dim3((n + 255) / 256, nj), 256, 0, s>>>(jobs, o, off, n, samples, dists);
      else k_es_sample<32, 128><<<dim3((n + 127) / 128, nj), 128, 0, s>>>(jobs, o, off, n, samples, dists);
    }
    beg += group[w];
  }
  return cudaGetLastError();
}

cudaError_t launch_es_run(EsJob *jobs, const uint32_t (&group)[kEsGroups], const uint32_t (&smem_of)[kEsGroups], uint32_t nsw, const uint2 *samples,
                          const uint16_t *dists, StatsDev *stats, unsigned long long *chain_acc, uint32_t *err,
                          uint32_t *nstop, bool alone, cudaStream_t s, cudaStream_t s2, cudaEvent_t fork,
                          cudaEvent_t join, uint32_t *launches) {
  // group[w] jobs with windows of 1024, 256, 128 and 32 switches, then the
  // small chains in shared memory, in that order; all but the two largest
  // groups run on s2 (after s, and joined back into s) when there is one,
  // beside the others
  uint32_t beg[kEsGroups + 1] = {};
  for (uint32_t w = 0; w < kEsGroups; ++w) beg[w + 1] = beg[w] + group[w];
  uint32_t n = 0;
  const bool side = s2 && fork && join && beg[2] > 0 && beg[kEsGroups] > beg[2];
  cudaStream_t ss = side ? s2 : s;
  if (side && (cudaEventRecord(fork, s) != cudaSuccess || cudaStreamWaitEvent(s2, fork, 0) != cudaSuccess))
    return cudaGetLastError();
  // The groups of the side stream need not wait for one another: each starts
  // when the CTAs of the one before are all on the GPU (programmatic dependent
  // launch), and every one of these kernels waits for the one before it just
  // before it ends, so that the last one's end is the end of all.
  uint32_t beside = 0;
  auto go = [&](auto fn, uint32_t ctas, uint32_t threads, size_t smem, uint32_t off) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ss;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = beside++ ? 1 : 0;
    cudaLaunchKernelEx(&cfg, fn, jobs, off, nsw, samples, dists, stats, chain_acc, err);
  };
  auto run = [&](int w, cudaStream_t st) {
    for (uint32_t off = beg[w]; off < beg[w + 1]; off += 65535u, ++n) {
      const uint32_t nj = beg[w + 1] - off < 65535u ? beg[w + 1] - off : 65535u, smem = smem_of[w];
      if (w == 0) {
        k_es_run_cluster<1024 / kClusterCtas><<<nj * kClusterCtas, 1024 / kClusterCtas, 0, st>>>(
            jobs, off, nsw, samples, dists, stats, chain_acc, err, nstop);
        if (alone) {
          k_es_run_big<<<nj, 1024, EsShape<1024>::kBytes, st>>>(jobs, off, nsw, samples, dists, stats, chain_acc, err,
                                                                nstop);
          ++n;
        }
      } else if (w == 1) {
        k_es_run<256, 6><<<nj, 256, EsShape<256>::kBytes, st>>>(jobs, off, nsw, samples, dists, stats, chain_acc, err);
      } else if (w == 2) {
        go(k_es_run<128, 12>, nj, 128, EsShape<128>::kBytes, off);
      } else if (w == 3) {
        go(k_es_run<32, 32>, nj, 32, EsShape<32>::kBytes, off);
      } else if (w == 4) {
        go(k_es_run_small, nj, 32, smem, off);
      } else {
        go(k_es_run_bits, nj, 32, smem, off);
      }
    }
  };
  // the groups that take longest first
  for (const int w : {3, 2, 4, 7, 6, 5}) run(w, ss);
  run(0, s);
  run(1, s);
  if (side && (cudaEventRecord(join, s2) != cudaSuccess || cudaStreamWaitEvent(s, join, 0) != cudaSuccess))
    return cudaGetLastError();
  if (launches) *launches = n;
  return cudaGetLastError();
}

}  // namespace gesmc
