// Minimum spanning forest by Boruvka's algorithm (Sec. 3.3) as an outlined
// multi-kernel Pipe (Sec. 4.3, 4.4):
//
//   Pipe {                                    // until no component has a cross edge
//     Invoke find_min(in -> out, retry)       // Atomic(component_lock) { keep the lighter edge }
//       [Invoke find_min(retry -> retry')]*   // Retry items re-run (Retry Backoff mapping)
//     Invoke link(components)                 // record the edges, hook the components
//     Iterate jump(all vertices)              // pointer jumping, Until !Any(changed)
//   }
//
// Edge order: the key (w, min(u,v), max(u,v)) is a strict order on distinct
// undirected edges, so every component has one lightest cross edge and the
// forest is unique. A component's lightest edge is a multi-word record (weight,
// both endpoints, CSR index, the other component), which no single atomic can
// update: the find_min kernel updates it inside an Atomic section on the
// component's lock, in one of three forms:
//   IRGL_LOCK_BLOCKING  divergence-safe atomicCAS retry loop (the lock attempt
//                       and the critical section share one branch), bounded
//   IRGL_LOCK_TICKET    ticket lock (take a ticket, wait for it to be served),
//                       bounded
//   IRGL_LOCK_RETRY     one atomicCAS attempt (Atomic ... Else); a vertex that
//                       misses the lock is pushed to the retry worklist and
//                       find_min is invoked again on that list, with contiguous
//                       blocks of items per thread (Retry Backoff), until it is
//                       empty.
// Before taking a lock a thread lowers the component's (w, min(u,v)) prefix with
// one 64-bit atomicMin; only a thread that lowered (or tied) it enters the Atomic
// section, and there only the owner of the current prefix writes, so of k threads
// that meet at a component about ln k lock instead of every one that saw no record
// yet.
//
// What bounds it: the live vertices' adjacency and the parent of each neighbour
// once per iteration, and a 32-byte record per component, one sector for prefix,
// lock and fields (six arrays before). The lists (vertices, components, retries,
// edges) are staged in shared memory and appended by one atomic per few hundred
// items: one atomic per component on single counters was a third of the time
// (2048^2 mesh, retry locks: link of the first iteration 2.03 ms of 6.4; 2.0 ms in
// all with these, blocking and ticket locks 14.7 and 13.0 -> 1.97 and 1.93 ms; then 1.65
// ms with the first iteration apart, where every vertex is its own component: no
// component reads, no contention for a record).
//
// Outlined (IRGL_PERSISTENT): the three kernels run back to back in one
// cooperative launch, separated by the grid barrier; the CTA size is chosen by
// the T_control rule over the kernels' block-size sets. IRGL_PER_LAUNCH: one
// launch per kernel invocation, with the host reading the counters in between.
#include <algorithm>
#include <chrono>
#include <cstring>

#include "irgl.h"
#include "irgl_internal.h"
#include "irgl_launch.h"

namespace irgl {

constexpr uint32_t kMsfMaxIters = 64;  // Boruvka halves the components with cross edges: 32 suffice

// Per-invocation counters, a ring of three: invocation j counts into slot j % 3
// and CTA 0 clears slot (j + 1) % 3 at its start (every CTA read that slot
// after the barrier that ended invocation j - 2, before arriving at the one
// that ended j - 1).
struct __align__(16) MsfSlot {
  uint32_t out;      // vertices pushed to the out-worklist (found a cross edge)
  uint32_t retry;    // vertices pushed to the retry worklist
  uint32_t comp;     // components whose record got its first edge this iteration
  uint32_t changed;  // pointer-jumping updates
};

struct MsfStatus {
  unsigned long long weight;  // total forest weight
  uint32_t edges;             // forest edges written
  uint32_t retries;           // retry pushes over the whole run
  uint32_t iterations;        // Boruvka iterations (Pipe repetitions)
  uint32_t invocations;       // kernel invocations inside the Pipe
  uint32_t locks;             // lock acquisitions
  uint32_t pad0[25];
  MsfSlot slot[3];
  uint32_t pad1[20];
};
static_assert(sizeof(MsfStatus) % 128 == 0, "status layout");

constexpr unsigned long long kNoRecord = ~0ull;

// A component's lightest cross edge, one 32-byte sector. wl is lowered by
// atomicMin before the lock is taken; tag is the prefix that hi, e and other
// belong to (written inside the Atomic section).
struct __align__(32) MsfRec {
  unsigned long long wl;   // (w << 32) | min(u,v) of the lightest edge found (~0: none yet)
  unsigned long long tag;  // prefix of the edge described below
  uint32_t hi;             // its larger endpoint
  uint32_t e;              // its CSR index
  uint32_t other;          // the component at its other end
  uint32_t lock;           // 0/1 (BLOCKING, RETRY) or now-serving (TICKET)
};
static_assert(sizeof(MsfRec) == 32, "one sector");

struct MsfParams {
  const uint32_t* __restrict__ row_ptr;
  const uint32_t* __restrict__ col;
  const int32_t* __restrict__ w;
  uint32_t n;
  uint32_t* comp;    // component (root vertex) of each vertex
  struct MsfRec* rec;  // per component
  uint32_t* ticket;    // per component: next ticket (TICKET)
  uint32_t* items[2];  // in/out worklists of vertices (capacity n each)
  uint32_t* retry[2];  // retry worklists (capacity n each)
  uint32_t* comps;     // components with a record this iteration (capacity n)
  uint32_t* out_edges;
  uint32_t out_cap;
  uint32_t lock_mode;
  DevStatus* st;
  MsfStatus* ms;
  unsigned long long timeout_ns;       // grid barrier waits
  unsigned long long lock_timeout_ns;  // lock waits and one find_min's retries: half the barrier's, so a
                                       // stuck lock is reported as such before the barrier gives up
  uint32_t held_lock;  // test hook: this component's lock starts held and is never released (kInf: none)
};

// Lexicographic order on (w, lo, hi).
__device__ __forceinline__ bool key_less(uint32_t w1, uint32_t l1, uint32_t h1, uint32_t w2, uint32_t l2, uint32_t h2) {
  if (w1 != w2) return w1 < w2;
  if (l1 != l2) return l1 < l2;
  return h1 < h2;
}

struct MinEdge {
  uint32_t w, lo, hi, e, other;
};

__device__ __forceinline__ MinEdge no_edge() { return MinEdge{kInf, kInf, kInf, 0u, 0u}; }

// Lightest cross-component edge among u's edges [beg, end), lanes taking
// every stride-th edge from beg + rank, four columns, then their components and
// weights in flight. FIRST: the first iteration, every vertex its own component.
template <bool FIRST>
__device__ __forceinline__ void scan_edges(const MsfParams& p, uint32_t u, uint32_t cu, uint32_t beg, uint32_t end,
                                           uint32_t rank, uint32_t stride, MinEdge& best) {
  for (unsigned long long e0 = static_cast<unsigned long long>(beg) + rank; e0 < end; e0 += 4ull * stride) {
    uint32_t v[4], cv[4], wt[4];
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) v[k] = e0 + k * stride < end ? __ldg(p.col + e0 + k * stride) : u;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      cv[k] = FIRST ? v[k] : v[k] != u ? __ldcg(p.comp + v[k]) : cu;
      wt[k] = e0 + k * stride < end ? static_cast<uint32_t>(__ldg(p.w + e0 + k * stride)) : kInf;
    }
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      if (cv[k] == cu) continue;
      const uint32_t lo = min(u, v[k]), hi = max(u, v[k]);
      if (key_less(wt[k], lo, hi, best.w, best.lo, best.hi))
        best = MinEdge{wt[k], lo, hi, static_cast<uint32_t>(e0) + k * stride, cv[k]};
    }
  }
}

__device__ __forceinline__ MinEdge warp_min_edge(MinEdge b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    MinEdge x;
    x.w = __shfl_xor_sync(kFull, b.w, o);
    x.lo = __shfl_xor_sync(kFull, b.lo, o);
    x.hi = __shfl_xor_sync(kFull, b.hi, o);
    x.e = __shfl_xor_sync(kFull, b.e, o);
    x.other = __shfl_xor_sync(kFull, b.other, o);
    if (key_less(x.w, x.lo, x.hi, b.w, b.lo, b.hi)) b = x;
  }
  return b;
}

// Three lists staged in the CTA's shared stage (L: vertices or edges, components,
// retries). Each thread pushes at most one item per list and tile; the stage is
// flushed at CTA-uniform points once a list might not hold another tile, with one
// atomic on the list's counter and coalesced stores.
template <int CTA>
struct MsfLists {
  static constexpr uint32_t kCap = (Smem<CTA>::kStage / 3) & ~31u;
  static_assert(kCap >= 2 * CTA, "room for the tile that follows the flush test");
  uint32_t n[3];
  uint32_t at[3];
};

template <int CTA>
__device__ __forceinline__ void stage_item(Smem<CTA>& sm, MsfLists<CTA>& ls, uint32_t L, bool pred, uint32_t item) {
  const unsigned m = __ballot_sync(kFull, pred);
  if (m == 0) return;
  const uint32_t lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  uint32_t pos = 0;
  if (lane == static_cast<uint32_t>(leader)) pos = atomicAdd(&ls.n[L], static_cast<uint32_t>(__popc(m)));
  pos = __shfl_sync(kFull, pos, leader) + __popc(m & lanemask_lt());
  if (pred) sm.stage[L * MsfLists<CTA>::kCap + pos] = item;
}

// Append the staged items: list L to dst[L][base[L] + ...] (capacity cap[L]), counted in *ctr[L].
struct MsfDest {
  uint32_t* dst[3];
  uint32_t* ctr[3];
  uint32_t base[3];
  uint32_t cap[3];
};
template <int CTA>
__device__ __forceinline__ void flush_lists(Smem<CTA>& sm, MsfLists<CTA>& ls, const MsfDest& d, uint32_t above,
                                            uint32_t* err) {
  constexpr uint32_t C = MsfLists<CTA>::kCap;
  if (!__syncthreads_or(ls.n[0] > above || ls.n[1] > above || ls.n[2] > above)) return;
  if (threadIdx.x < 3 && ls.n[threadIdx.x] != 0) {
    const uint32_t L = threadIdx.x;
    uint32_t* const ctr = L == 0 ? d.ctr[0] : L == 1 ? d.ctr[1] : d.ctr[2];
    ls.at[L] = (L == 0 ? d.base[0] : L == 1 ? d.base[1] : d.base[2]) + atomicAdd(ctr, ls.n[L]);
  }
  __syncthreads();
#pragma unroll
  for (uint32_t L = 0; L < 3; ++L) {
    const uint32_t k = ls.n[L], at = ls.at[L];
    for (uint32_t i = threadIdx.x; i < k; i += CTA) {
      if (at + i < d.cap[L]) __stcg(d.dst[L] + at + i, sm.stage[L * C + i]);
      else set_err(err, DERR_WL_OVERFLOW);
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) ls.n[threadIdx.x] = 0;
  __syncthreads();
}

__device__ __forceinline__ unsigned long long wl_of(const MinEdge& k) {
  return (static_cast<unsigned long long>(k.w) << 32) | k.lo;
}

// The critical section of the Atomic: the owner of the component's current
// prefix describes its edge; of equal prefixes the smaller larger end stays.
__device__ __forceinline__ void record_update(MsfRec* r, const MinEdge& k) {
  const unsigned long long wl = wl_of(k);
  const ulonglong2 cur = __ldcg(reinterpret_cast<const ulonglong2*>(r));  // wl, tag
  if (cur.x != wl || (cur.y == wl && k.hi >= __ldcg(&r->hi))) return;
  __stcg(&r->tag, wl);
  __stcg(reinterpret_cast<uint2*>(&r->hi), make_uint2(k.hi, k.e));
  __stcg(&r->other, k.other);
}

__device__ __forceinline__ unsigned long long msf_now() { return globaltimer_ns(); }

// Atomic(lock[c]) { record_update } in the configured form. Returns false when
// the lock was missed in RETRY mode (the caller retries the vertex). first: this
// edge is the component's first of the iteration; locks counts acquisitions.
__device__ __forceinline__ bool atomic_update(const MsfParams& p, uint32_t c, const MinEdge& k, bool& first,
                                              uint32_t& locks) {
  MsfRec* const r = p.rec + c;
  const unsigned long long wl = wl_of(k);
  if (wl > __ldcg(&r->wl)) return true;
  const unsigned long long before = atomicMin(&r->wl, wl);
  if (before < wl) return true;
  first = before == kNoRecord;
  if (p.lock_mode == IRGL_LOCK_TICKET) {
    const uint32_t t = atomicAdd(p.ticket + c, 1u);
    const unsigned long long t0 = msf_now();
    for (uint32_t spins = 1;; ++spins) {
      uint32_t serving;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(serving) : "l"(&r->lock) : "memory");
      if (serving == t) break;
      if ((spins & 63u) == 0 && (msf_now() - t0 > p.lock_timeout_ns || __ldcg(&p.st->err) == DERR_LOCK_TIMEOUT)) {
        set_err(&p.st->err, DERR_LOCK_TIMEOUT);
        return true;
      }
    }
    record_update(r, k);
    ++locks;
    asm volatile("st.release.gpu.global.u32 [%0], %1;" : : "l"(&r->lock), "r"(t + 1u) : "memory");
    return true;
  }
  const bool blocking = p.lock_mode == IRGL_LOCK_BLOCKING;
  const unsigned long long t0 = blocking ? msf_now() : 0ull;
  for (uint32_t spins = 1;; ++spins) {
    // the attempt and the critical section in one branch: no thread waits on
    // a lock held by a lane of its own warp that cannot be scheduled
    uint32_t old;
    asm volatile("atom.acquire.gpu.global.cas.b32 %0, [%1], 0, 1;" : "=r"(old) : "l"(&r->lock) : "memory");
    if (old == 0u) {
      record_update(r, k);
      ++locks;
      asm volatile("st.release.gpu.global.u32 [%0], 0;" : : "l"(&r->lock) : "memory");
      return true;
    }
    if (!blocking) return false;  // Atomic ... Else: Retry
    if ((spins & 63u) == 0 && (msf_now() - t0 > p.lock_timeout_ns || __ldcg(&p.st->err) == DERR_LOCK_TIMEOUT)) {
      set_err(&p.st->err, DERR_LOCK_TIMEOUT);
      return true;
    }
    __nanosleep(min(32u << min(spins, 5u), 1024u));  // exponential backoff: waiters leave the line to the holder
  }
}

// Lanes of a warp whose vertices share a component send only the lightest of
// their edges to the Atomic section (the others cannot change the record).
// Returns true when that lane missed the lock in RETRY mode.
__device__ __forceinline__ bool aggregate_update(const MsfParams& p, bool found, uint32_t cu, const MinEdge& best,
                                                 bool& first, uint32_t& locks) {
  const unsigned active = __ballot_sync(kFull, found);
  if (!found) return false;
  const unsigned peers = __match_any_sync(active, cu);
  const uint32_t mw = __reduce_min_sync(peers, best.w);
  const uint32_t ml = __reduce_min_sync(peers, best.w == mw ? best.lo : kInf);
  const uint32_t mh = __reduce_min_sync(peers, best.w == mw && best.lo == ml ? best.hi : kInf);
  if (best.w != mw || best.lo != ml || best.hi != mh) return false;
  return !atomic_update(p, cu, best, first, locks);
}

// The Atomic section of a component of one vertex, in the first iteration: no other
// thread touches its record, so the lock (free unless the test hook holds it) need not
// be taken and the record is two plain stores.
__device__ __forceinline__ bool first_update(const MsfParams& p, uint32_t u, const MinEdge& k, bool& first, uint32_t& locks) {
  if (u == p.held_lock) return atomic_update(p, u, k, first, locks);
  MsfRec* const r = p.rec + u;
  __stcg(reinterpret_cast<ulonglong2*>(r), make_ulonglong2(wl_of(k), wl_of(k)));
  __stcg(reinterpret_cast<uint4*>(&r->hi), make_uint4(k.hi, k.e, k.other, 0u));
  first = true;
  return true;
}

// find_min over a worklist: `in` (nullptr = vertices 0..in_n-1, in the first iteration). Default
// mapping: a warp takes 32 consecutive items; lists of 32 edges or more are
// scanned by the whole warp. Retry mapping (Retry Backoff): thread t takes the
// contiguous block [t * B, (t + 1) * B) and scans each list alone. Trip counts
// are CTA-uniform (the lists are flushed by the whole CTA).
template <int CTA, bool FIRST>
__device__ void msf_find_min(const MsfParams& p, Smem<CTA>& sm, MsfLists<CTA>& ls, const uint32_t* in, uint32_t in_n,
                             bool backoff, uint32_t* out, uint32_t out_base, uint32_t* retry_out, MsfSlot* slot,
                             uint32_t comp_base) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t gtid = blockIdx.x * CTA + threadIdx.x, nthreads = gridDim.x * CTA;
  constexpr uint32_t kFlush = MsfLists<CTA>::kCap - CTA;
  const MsfDest d{{out, p.comps, retry_out}, {&slot->out, &slot->comp, &slot->retry}, {out_base, comp_base, 0u}, {p.n, p.n, p.n}};
  uint32_t locks = 0;
  const uint32_t trips = backoff ? (in_n + nthreads - 1) / nthreads
                                 : static_cast<uint32_t>((static_cast<unsigned long long>(in_n) + nthreads - 1u -
                                                          min(in_n, blockIdx.x * CTA)) / nthreads);
  for (uint32_t t = 0; t < trips; ++t) {
    const unsigned long long idx = backoff ? static_cast<unsigned long long>(gtid) * trips + t
                                           : static_cast<unsigned long long>(t) * nthreads + gtid;
    const bool valid = idx < in_n;
    uint32_t u = 0, cu = 0, beg = 0, end = 0;
    if (valid) {
      u = FIRST ? static_cast<uint32_t>(idx) : __ldcg(in + idx);
      cu = FIRST ? u : __ldcg(p.comp + u);
      beg = __ldg(p.row_ptr + u);
      end = __ldg(p.row_ptr + u + 1);
    }
    MinEdge best = no_edge();
    const bool big = !backoff && valid && end - beg >= 32u;
    if (valid && !big) scan_edges<FIRST>(p, u, cu, beg, end, 0, 1, best);
    for (unsigned m = __ballot_sync(kFull, big); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      MinEdge wb = no_edge();
      scan_edges<FIRST>(p, __shfl_sync(kFull, u, l), __shfl_sync(kFull, cu, l), __shfl_sync(kFull, beg, l),
                 __shfl_sync(kFull, end, l), lane, 32, wb);
      wb = warp_min_edge(wb);
      if (lane == static_cast<uint32_t>(l)) best = wb;
    }
    const bool found = best.w != kInf;
    bool first = false;
    bool missed;
    if (FIRST) missed = found && !first_update(p, u, best, first, locks);
    else missed = aggregate_update(p, found, cu, best, first, locks);
    __syncwarp();
    stage_item<CTA>(sm, ls, 0, found && !missed, u);
    stage_item<CTA>(sm, ls, 1, first, cu);
    stage_item<CTA>(sm, ls, 2, missed, u);
    flush_lists<CTA>(sm, ls, d, kFlush, &p.st->err);
  }
  flush_lists<CTA>(sm, ls, d, 0u, &p.st->err);
  locks = __reduce_add_sync(kFull, locks);
  if (lane == 0 && locks) atomicAdd(&p.ms->locks, locks);
}

// link over the components with a record: record the edge (once per mutual
// pair: by the smaller component) and hook the component to the other one
// (a mutual pair's smaller component stays the root), then clear the record.
// The forest's edges go through the stage, its weight is summed per warp.
template <int CTA>
__device__ void msf_link(const MsfParams& p, Smem<CTA>& sm, MsfLists<CTA>& ls, uint32_t comp_n) {
  const uint32_t gtid = blockIdx.x * CTA + threadIdx.x, nthreads = gridDim.x * CTA;
  constexpr uint32_t kFlush = MsfLists<CTA>::kCap - CTA;
  const MsfDest d{{p.out_edges, nullptr, nullptr}, {&p.ms->edges, nullptr, nullptr}, {0u, 0u, 0u}, {p.out_cap, 0u, 0u}};
  unsigned long long weight = 0;
  const uint32_t trips = static_cast<uint32_t>((static_cast<unsigned long long>(comp_n) + nthreads - 1u -
                                                min(comp_n, blockIdx.x * CTA)) / nthreads);
  for (uint32_t t = 0; t < trips; ++t) {
    const unsigned long long i = static_cast<unsigned long long>(t) * nthreads + gtid;
    bool take = false;
    uint32_t edge = 0;
    if (i < comp_n) {
      const uint32_t c = __ldcg(p.comps + i);
      MsfRec* const r = p.rec + c;
      const uint4 f = __ldcg(reinterpret_cast<const uint4*>(&r->hi));  // hi, e, other, lock
      const uint32_t w = static_cast<uint32_t>(__ldcg(&r->wl) >> 32);
      const uint32_t c2 = f.z;
      const bool mutual = __ldcg(&p.rec[c2].other) == c;
      take = !mutual || c < c2;
      edge = f.y;
      if (take) weight += w;
      if (!mutual || c > c2) __stcg(p.comp + c, c2);
      __stcg(reinterpret_cast<ulonglong2*>(r), make_ulonglong2(kNoRecord, kNoRecord));
    }
    stage_item<CTA>(sm, ls, 0, take, edge);
    flush_lists<CTA>(sm, ls, d, kFlush, &p.st->err);
  }
  flush_lists<CTA>(sm, ls, d, 0u, &p.st->err);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) weight += __shfl_xor_sync(kFull, weight, o);
  if ((threadIdx.x & 31) == 0 && weight) atomicAdd(&p.ms->weight, weight);
}

// One pointer-jumping pass over every vertex: each follows its pointers to the
// root, kJumpSteps at most, four vertices in flight per thread. Returns how many
// stopped short of a root (the pass is repeated while any did): a hooked tree is
// rarely deeper, so one pass does what took four or five of one step each, and a
// long chain still shrinks by more than kJumpSteps a pass.
constexpr uint32_t kJumpSteps = 64;
__device__ uint32_t msf_jump(const MsfParams& p, uint32_t gtid, uint32_t nthreads) {
  constexpr uint32_t U = 4;
  uint32_t open = 0;
  for (unsigned long long i = gtid; i < p.n; i += static_cast<unsigned long long>(U) * nthreads) {
    uint32_t c[U], x[U];
#pragma unroll
    for (uint32_t k = 0; k < U; ++k) {
      const unsigned long long v = i + static_cast<unsigned long long>(k) * nthreads;
      c[k] = v < p.n ? __ldcg(p.comp + v) : 0u;
    }
#pragma unroll
    for (uint32_t k = 0; k < U; ++k) x[k] = __ldcg(p.comp + c[k]);
#pragma unroll
    for (uint32_t k = 0; k < U; ++k) {
      const unsigned long long v = i + static_cast<unsigned long long>(k) * nthreads;
      if (v >= p.n || x[k] == c[k]) continue;
      uint32_t r = x[k], y = __ldcg(p.comp + r);
      for (uint32_t s = 2; y != r && s < kJumpSteps; ++s) {
        r = y;
        y = __ldcg(p.comp + r);
      }
      open += y != r ? 1u : 0u;
      __stcg(p.comp + v, r);
    }
  }
  return open;
}

__device__ void msf_init(const MsfParams& p, uint32_t gtid, uint32_t nthreads) {
  for (unsigned long long i = gtid; i < p.n; i += nthreads) {
    const uint32_t v = static_cast<uint32_t>(i);
    __stcg(p.comp + v, v);
    // a held lock: 1 for the CAS forms, a now-serving value no ticket reaches
    const uint32_t lock = v == p.held_lock ? (p.ticket ? kInf : 1u) : 0u;
    __stcg(reinterpret_cast<ulonglong2*>(p.rec + v), make_ulonglong2(kNoRecord, kNoRecord));
    __stcg(reinterpret_cast<uint4*>(&p.rec[v].hi), make_uint4(0u, 0u, 0u, lock));
    if (p.ticket) __stcg(p.ticket + v, 0u);
  }
}

template <int CTA>
__device__ __forceinline__ uint32_t cta_sum_u32(Smem<CTA>& sm, uint32_t x) {
  unsigned long long s = cta_sum_u64<CTA>(sm, x);
  return static_cast<uint32_t>(s);
}

// The outlined Pipe: every kernel invocation of every iteration in one
// cooperative launch.
template <int CTA>
__global__ void __launch_bounds__(CTA, MinBlocks<CTA>::value) k_msf(MsfParams p) {
  __shared__ Smem<CTA> sm;
  __shared__ MsfLists<CTA> ls;
  if (threadIdx.x < 3) ls.n[threadIdx.x] = 0;
  init_smem<CTA>(sm);
  DevStatus* st = p.st;
  MsfStatus* ms = p.ms;
  const uint32_t gtid = blockIdx.x * CTA + threadIdx.x, nthreads = gridDim.x * CTA;
  const uint32_t ep0 = __ldcg(&st->epoch);
  uint32_t gen = 0, inv = 0;
  bool ok = true;

  auto begin_invocation = [&]() {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      MsfSlot* s = &ms->slot[(inv + 1) % 3];
      s->out = s->retry = s->comp = s->changed = 0;
    }
    sm.round_pushes = 0;
  };
  auto end_invocation = [&]() -> MsfSlot {
    ok = grid_barrier<CTA>(sm, st, gen, p.timeout_ns);
    MsfSlot r{0, 0, 0, 0};
    if (ok && sm.pub_err == DERR_NONE) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(&ms->slot[inv % 3]));
      r = MsfSlot{v.x, v.y, v.z, v.w};
    } else {
      ok = false;
    }
    ++inv;
    return r;
  };

  begin_invocation();
  msf_init(p, gtid, nthreads);
  end_invocation();

  uint32_t cur = 0, in_n = p.n, iters = 0, retries = 0;
  const uint32_t* in = nullptr;  // iteration 0: every vertex
  while (ok) {
    if (iters >= kMsfMaxIters) {
      if (blockIdx.x == 0 && threadIdx.x == 0) set_err(&st->err, DERR_MSF_ITERS);
      break;
    }
    ++iters;
    uint32_t* out = p.items[cur ^ 1u];
    // find_min, then its retries
    uint32_t out_total = 0, comp_total = 0, rb = 0;
    const uint32_t* fin = in;
    uint32_t fin_n = in_n;
    bool backoff = false;
    const unsigned long long t_retry0 = msf_now();
    for (;;) {
      begin_invocation();
      if (fin == nullptr)
        msf_find_min<CTA, true>(p, sm, ls, fin, fin_n, false, out, out_total, p.retry[rb], &ms->slot[inv % 3], comp_total);
      else
        msf_find_min<CTA, false>(p, sm, ls, fin, fin_n, backoff, out, out_total, p.retry[rb], &ms->slot[inv % 3], comp_total);
      const MsfSlot s = end_invocation();
      if (!ok) break;
      out_total += s.out;
      comp_total += s.comp;
      retries += s.retry;
      if (s.retry == 0) break;
      // the retries of one find_min end within the lock time limit (every CTA
      // reads the same clock values closely enough; the flag makes it uniform)
      if (threadIdx.x == 0 && msf_now() - t_retry0 > p.lock_timeout_ns) set_err(&st->err, DERR_LOCK_TIMEOUT);
      fin = p.retry[rb];
      fin_n = min(s.retry, p.n);
      rb ^= 1u;
      backoff = true;
    }
    if (!ok || out_total == 0) break;  // no component has a cross edge: the forest is complete
    begin_invocation();
    msf_link<CTA>(p, sm, ls, min(comp_total, p.n));
    end_invocation();
    for (uint32_t pass = 0; ok; ++pass) {
      begin_invocation();
      sm.round_pushes = 0;
      const uint32_t changed = cta_sum_u32<CTA>(sm, msf_jump(p, gtid, nthreads));
      if (threadIdx.x == 0 && changed) atomicAdd(&ms->slot[inv % 3].changed, changed);
      const MsfSlot s = end_invocation();
      if (s.changed == 0) break;
    }
    in = out;
    in_n = min(out_total, p.n);
    cur ^= 1u;
  }
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ms->iterations = iters;
    ms->invocations = inv;
    ms->retries = retries;
  }
  persistent_exit<CTA>(sm, st, ok, inv, 0u, ep0, 0ull, nullptr, 0);
}

// Per-launch form: one kernel per invocation; the host clears the slot it
// counts into and reads it afterwards.
enum : uint32_t { MSF_INIT = 0, MSF_FIND = 1, MSF_FIND_RETRY = 2, MSF_LINK = 3, MSF_JUMP = 4 };

struct MsfStep {
  uint32_t phase;
  const uint32_t* in;
  uint32_t in_n;
  uint32_t* out;
  uint32_t out_base;
  uint32_t* retry_out;
  uint32_t comp_base;
  uint32_t comp_n;
  uint32_t slot;
};

template <int CTA>
__global__ void __launch_bounds__(CTA, MinBlocks<CTA>::value) k_msf_step(MsfParams p, MsfStep s) {
  __shared__ Smem<CTA> sm;
  __shared__ MsfLists<CTA> ls;
  if (threadIdx.x < 3) ls.n[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t gtid = blockIdx.x * CTA + threadIdx.x, nthreads = gridDim.x * CTA;
  MsfSlot* slot = &p.ms->slot[s.slot];
  switch (s.phase) {
    case MSF_INIT: msf_init(p, gtid, nthreads); break;
    case MSF_FIND:
    case MSF_FIND_RETRY:
      if (s.in == nullptr)
        msf_find_min<CTA, true>(p, sm, ls, s.in, s.in_n, false, s.out, s.out_base, s.retry_out, slot, s.comp_base);
      else
        msf_find_min<CTA, false>(p, sm, ls, s.in, s.in_n, s.phase == MSF_FIND_RETRY, s.out, s.out_base, s.retry_out, slot,
                                 s.comp_base);
      break;
    case MSF_LINK: msf_link<CTA>(p, sm, ls, s.comp_n); break;
    case MSF_JUMP: {
      const uint32_t c = msf_jump(p, gtid, nthreads);
      if (c) atomicAdd(&slot->changed, c);
      break;
    }
  }
}

// Block-size sets of the Pipe's kernels (bit b = CTA 128 << b). Each is a
// FixedBlock template (CTA is a template parameter: launch bounds and the
// shared-memory layout of the barrier depend on it) compiled for the four sizes.
constexpr uint32_t kMsfFindMask = 0xFu, kMsfLinkMask = 0xFu, kMsfJumpMask = 0xFu;

template <int CTA>
cudaError_t msf_occupancy(bool outlined, int* nb) {
  return outlined ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, k_msf<CTA>, CTA, 0)
                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, k_msf_step<CTA>, CTA, 0);
}

cudaError_t msf_occupancy_cta(uint32_t cta, bool outlined, int* nb) {
  switch (cta) {
    case 128: return msf_occupancy<128>(outlined, nb);
    case 256: return msf_occupancy<256>(outlined, nb);
    case 512: return msf_occupancy<512>(outlined, nb);
    case 1024: return msf_occupancy<1024>(outlined, nb);
  }
  return cudaErrorInvalidValue;
}

template <int CTA>
cudaError_t msf_launch_outlined(uint32_t grid, const MsfParams& p, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(CTA);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_msf<CTA>, p);
}

cudaError_t msf_launch_outlined_cta(uint32_t cta, uint32_t grid, const MsfParams& p, cudaStream_t s) {
  switch (cta) {
    case 128: return msf_launch_outlined<128>(grid, p, s);
    case 256: return msf_launch_outlined<256>(grid, p, s);
    case 512: return msf_launch_outlined<512>(grid, p, s);
    case 1024: return msf_launch_outlined<1024>(grid, p, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t msf_launch_step_cta(uint32_t cta, uint32_t grid, const MsfParams& p, const MsfStep& st, cudaStream_t s) {
  switch (cta) {
    case 128: k_msf_step<128><<<grid, 128, 0, s>>>(p, st); break;
    case 256: k_msf_step<256><<<grid, 256, 0, s>>>(p, st); break;
    case 512: k_msf_step<512><<<grid, 512, 0, s>>>(p, st); break;
    case 1024: k_msf_step<1024><<<grid, 1024, 0, s>>>(p, st); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace irgl

using namespace irgl;

extern "C" {

irgl_status irgl_msf(irgl_ctx* ctx, irgl_graph* g, irgl_mode mode, irgl_lock lock, uint32_t* out_edges,
                     uint32_t cap, int out_on_host, const irgl_tuning* tin, irgl_msf_stats* stats) {
  if (!ctx || !g || !out_edges) return fail(IRGL_ERR_INVALID_ARG, "NULL argument");
  if (!g->w) return fail(IRGL_ERR_INVALID_ARG, "the minimum spanning forest needs edge weights");
  if (!(g->flags & IRGL_SYMMETRIC))
    return fail(IRGL_ERR_NOT_SYMMETRIC, "the minimum spanning forest needs a graph loaded with IRGL_SYMMETRIC");
  if (mode != IRGL_PERSISTENT && mode != IRGL_PER_LAUNCH) return fail(IRGL_ERR_INVALID_ARG, "unknown mode");
  if (lock != IRGL_LOCK_BLOCKING && lock != IRGL_LOCK_TICKET && lock != IRGL_LOCK_RETRY)
    return fail(IRGL_ERR_INVALID_ARG, "unknown lock form %d", static_cast<int>(lock));
  const uint32_t n = g->n;
  const uint32_t need = n > 0 ? n - 1 : 0;
  if (cap < need) return fail(IRGL_ERR_INVALID_ARG, "out_edges holds %u edges, a forest may need %u", cap, need);
  irgl_tuning t;
  irgl_status s = resolve_tuning(tin, &t);
  if (s != IRGL_OK) return s;
  if (stats) std::memset(stats, 0, sizeof(*stats));
  if (n == 0) return IRGL_OK;
  DeviceGuard guard(ctx->device);

  // T_control over find_min, link and jump (Sec. 4.4)
  const uint32_t masks[3] = {kMsfFindMask, kMsfLinkMask, kMsfJumpMask};
  uint32_t cta = 0;
  s = control_cta(masks, 3, t.cta_size, &cta);
  if (s != IRGL_OK) return s;

  // workspace: the status block, then 16 arrays of N words (N a multiple of
  // 64, so every array starts on a 256-byte boundary; the records take eight)
  const uint64_t n_round = (static_cast<uint64_t>(n) + 63u) & ~63ull;
  if (n_round > 0xFFFFFFC0ull) return fail(IRGL_ERR_INVALID_ARG, "n = %u is too large for the forest workspace", n);
  if (ctx->msf_n < n_round || !ctx->msf_buf) {
    cudaStreamSynchronize(ctx->stream);
    cudaFree(ctx->msf_buf);
    ctx->msf_buf = nullptr;
    ctx->msf_n = 0;
    const size_t words = static_cast<size_t>(n_round) * 16 + sizeof(MsfStatus) / 4;
    cudaError_t e = cudaMalloc(&ctx->msf_buf, words * sizeof(uint32_t));
    if (e != cudaSuccess) return cuda_fail(e, "minimum spanning forest workspace");
    ctx->msf_n = static_cast<uint32_t>(n_round);
  }
  if (!ctx->msf_host) {
    cudaError_t e = cudaMallocHost(&ctx->msf_host, sizeof(MsfStatus));
    if (e != cudaSuccess) return cuda_fail(e, "status staging");
  }
  uint32_t* b = ctx->msf_buf;
  const size_t N = ctx->msf_n;
  MsfParams p;
  std::memset(&p, 0, sizeof(p));
  p.row_ptr = g->row_ptr;
  p.col = g->col;
  p.w = g->w;
  p.n = n;
  MsfStatus* ms = reinterpret_cast<MsfStatus*>(b);  // 128-byte multiple at the start
  uint32_t* a = b + sizeof(MsfStatus) / 4;
  p.rec = reinterpret_cast<MsfRec*>(a);  // eight arrays' worth
  p.comp = a + 8 * N;
  p.ticket = lock == IRGL_LOCK_TICKET ? a + 9 * N : nullptr;
  p.items[0] = a + 10 * N;
  p.items[1] = a + 11 * N;
  p.retry[0] = a + 12 * N;
  p.retry[1] = a + 13 * N;
  p.comps = a + 14 * N;
  uint32_t* dev_out = out_on_host ? a + 15 * N : out_edges;
  p.out_edges = dev_out;
  p.out_cap = out_on_host ? n : cap;
  p.lock_mode = static_cast<uint32_t>(lock);
  p.st = ctx->st;
  p.ms = ms;
  p.timeout_ns = ctx->dbg_timeout_us ? ctx->dbg_timeout_us * 1000ull : 2000000000ull;
  p.lock_timeout_ns = p.timeout_ns / 2;
  p.held_lock = ctx->dbg_held_lock < n ? ctx->dbg_held_lock : kInf;
  cudaError_t e = cudaMemsetAsync(ms, 0, sizeof(MsfStatus), ctx->stream);
  if (e != cudaSuccess) return cuda_fail(e, "status clear");

  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  cudaEventCreate(&ev0);
  cudaEventCreate(&ev1);
  cudaEventRecord(ev0, ctx->stream);
  irgl_msf_stats local;
  std::memset(&local, 0, sizeof(local));
  local.cta_size = cta;
  uint32_t launches = 0, invocations = 0, iters = 0, retries = 0;

  int nb = 0;
  e = msf_occupancy_cta(cta, mode == IRGL_PERSISTENT, &nb);
  if (e != cudaSuccess || nb <= 0) {
    cudaEventDestroy(ev0);
    cudaEventDestroy(ev1);
    return e != cudaSuccess ? cuda_fail(e, "occupancy") : fail(IRGL_ERR_CUDA, "MSF kernel cannot be made resident");
  }
  if (t.blocks_per_sm && static_cast<int>(t.blocks_per_sm) < nb) nb = static_cast<int>(t.blocks_per_sm);
  uint32_t grid = static_cast<uint32_t>(nb) * static_cast<uint32_t>(ctx->sm_count);
  if (t.max_blocks && t.max_blocks < grid) grid = t.max_blocks;
  grid = std::max<uint32_t>(1, std::min<uint32_t>(grid, kMaxGrid));
  local.grid = grid;

  if (mode == IRGL_PERSISTENT) {
    e = msf_launch_outlined_cta(cta, grid, p, ctx->stream);
    if (e != cudaSuccess) {
      cudaEventDestroy(ev0);
      cudaEventDestroy(ev1);
      return cuda_fail(e, "MSF launch");
    }
    launches = 1;
  } else {
    // the host drives the Pipe: one launch per invocation, counters read in between
    MsfStep st;
    std::memset(&st, 0, sizeof(st));
    auto step = [&](MsfStep& x) -> irgl_status {
      x.slot = 0;
      cudaError_t er = cudaMemsetAsync(&ms->slot[0], 0, sizeof(MsfSlot), ctx->stream);
      if (er == cudaSuccess) er = msf_launch_step_cta(cta, grid, p, x, ctx->stream);
      if (er == cudaSuccess)
        er = cudaMemcpyAsync(ctx->msf_host, ms, sizeof(MsfStatus), cudaMemcpyDeviceToHost, ctx->stream);
      if (er == cudaSuccess) er = cudaStreamSynchronize(ctx->stream);
      if (er != cudaSuccess) return cuda_fail(er, "MSF step");
      ++launches;
      ++invocations;
      return read_status(ctx, nullptr);
    };
    st.phase = MSF_INIT;
    s = step(st);
    uint32_t cur = 0, in_n = n;
    const uint32_t* in = nullptr;
    while (s == IRGL_OK) {
      if (iters >= kMsfMaxIters) {
        s = fail(IRGL_ERR_CUDA, "Boruvka did not converge within %u iterations", kMsfMaxIters);
        break;
      }
      ++iters;
      uint32_t* out = p.items[cur ^ 1u];
      uint32_t out_total = 0, comp_total = 0, rb = 0;
      const uint32_t* fin = in;
      uint32_t fin_n = in_n;
      bool backoff = false;
      const auto t_retry0 = std::chrono::steady_clock::now();
      for (;;) {
        st.phase = backoff ? MSF_FIND_RETRY : MSF_FIND;
        st.in = fin;
        st.in_n = fin_n;
        st.out = out;
        st.out_base = out_total;
        st.retry_out = p.retry[rb];
        st.comp_base = comp_total;
        s = step(st);
        if (s != IRGL_OK) break;
        const MsfSlot r = static_cast<MsfStatus*>(ctx->msf_host)->slot[0];
        out_total += r.out;
        comp_total += r.comp;
        retries += r.retry;
        if (r.retry == 0) break;
        if (std::chrono::steady_clock::now() - t_retry0 > std::chrono::nanoseconds(p.lock_timeout_ns)) {
          s = fail(IRGL_ERR_LOCK_TIMEOUT, "retries of a component lock exceeded the time limit");
          break;
        }
        fin = p.retry[rb];
        fin_n = std::min(r.retry, n);
        rb ^= 1u;
        backoff = true;
      }
      if (s != IRGL_OK || out_total == 0) break;
      st.phase = MSF_LINK;
      st.comp_n = std::min(comp_total, n);
      s = step(st);
      while (s == IRGL_OK) {
        st.phase = MSF_JUMP;
        s = step(st);
        if (s != IRGL_OK || static_cast<MsfStatus*>(ctx->msf_host)->slot[0].changed == 0) break;
      }
      in = out;
      in_n = std::min(out_total, n);
      cur ^= 1u;
    }
    if (s != IRGL_OK) {
      cudaEventDestroy(ev0);
      cudaEventDestroy(ev1);
      if (stats) *stats = local;
      return s;
    }
  }
  cudaEventRecord(ev1, ctx->stream);
  e = cudaMemcpyAsync(ctx->msf_host, ms, sizeof(MsfStatus), cudaMemcpyDeviceToHost, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) {
    cudaEventDestroy(ev0);
    cudaEventDestroy(ev1);
    return cuda_fail(e, "MSF status readback");
  }
  float ms_elapsed = 0.f;
  cudaEventElapsedTime(&ms_elapsed, ev0, ev1);
  cudaEventDestroy(ev0);
  cudaEventDestroy(ev1);
  s = read_status(ctx, nullptr);
  if (s != IRGL_OK) {
    if (stats) *stats = local;
    return s;
  }
  const MsfStatus& h = *static_cast<MsfStatus*>(ctx->msf_host);
  local.edges = h.edges;
  local.weight = h.weight;
  local.locks = h.locks;
  if (mode == IRGL_PERSISTENT) {
    local.iterations = h.iterations;
    local.invocations = h.invocations;
    local.retries = h.retries;
  } else {
    local.iterations = iters;
    local.invocations = invocations;
    local.retries = retries;
  }
  local.launches = launches;
  local.device_ms = ms_elapsed;
  if (h.edges > need) {
    if (stats) *stats = local;
    return fail(IRGL_ERR_CUDA, "forest has %u edges, more than n - 1 = %u", h.edges, need);
  }
  if (out_on_host && h.edges) {
    e = cudaMemcpyAsync(out_edges, dev_out, sizeof(uint32_t) * h.edges, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_fail(e, "forest copy");
  }
  if (stats) *stats = local;
  return IRGL_OK;
}

}  // extern "C"
