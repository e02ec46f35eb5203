// Iteration-outlined Iterate for graphs that fit in one CTA's shared memory.
//
// The Sec. 3.4 outlining puts every round of an Iterate into one launch and
// separates the rounds by SyncRunningThreads; on a graph of a few thousand
// vertices the rounds are then a chain of dependent global-memory round trips
// (pop, row offsets, column, value, atomic, push) plus a grid barrier, each
// round a few microseconds although it touches a few hundred bytes. When the
// whole graph, its values and both worklists fit in the 227 KB of shared
// memory one CTA may use, a single CTA of 1024 threads copies the CSR in once
// and runs every round there: the grid barrier becomes __syncthreads, every
// access is a shared-memory one, and the values are written back at the end.
// Same operator, worklist discipline (pops from `in`, pushes to `out`, swapped
// each round) and fixed point as the grid-wide kernels; only the schedule of
// the pops differs, which the unique fixed point does not see.
//
// What bounds it: the round's chain of dependent shared-memory reads and atomics
// (about 30 and 100 cycles each) and its barrier; with over a thousand items also the
// one SM's instruction issue. So a round has one barrier (three list counters in turn),
// and a frontier of up to 256 items gives every item four lanes, dealt across the warps.
// Above that a lane walks a list of its own, in worklist order where no list of the graph
// is long (neighbours in memory stay neighbours in the banks), and lists of more than
// eight edges are dealt to the warp's lanes by a scan. Before -> now, each a call and the
// wait for it: 64 x 64 grid BFS 179 -> 107 us (narrow rounds below included), its min-label
// CC 373 -> 332; R-MAT of 2^10 vertices SSSP 95 -> 56; CC of a path of 3000 vertices 4.2 ->
// 4.0 ms. With every list dealt by the scan, CC took 633 us and 11.2 ms; with the items
// of R-MAT rounds in worklist order SSSP took 65 us.
//
// Shared-memory layout (32-bit words): row_ptr[n + 1], col[m], w[m] (SSSP),
// value[n], stamp[n] (SSSP and CC: the round that last pushed the vertex, so
// each vertex is pushed at most once per round), wl[2][n].
#include <algorithm>

#include "irgl_launch.h"

namespace irgl {

namespace {

constexpr int kSmemCta = 1024;
constexpr uint32_t kSmemWarps = kSmemCta / 32;
constexpr uint32_t kSmemLane = 8;               // a lane walks lists of at most this many edges itself
constexpr uint32_t kSmemFour = kSmemCta / 4;  // frontiers of at most this many items give each four lanes
// Narrow rounds: a frontier of at most 64 items is one pass of eight warps, which cross a
// barrier of their own faster than 32 warps cross the CTA's; the others wait at the next
// CTA barrier until a frontier outgrows them (64 x 64 grid BFS 104 -> 87 us a call without
// the wait, SSSP on a 20 x 24 mesh 51 -> 42; 256 threads for the whole run instead slow
// down wider frontiers: SSSP on a 50 x 60 mesh 89 -> 110).
constexpr uint32_t kNarrowWarps = 8;
constexpr uint32_t kNarrow = kNarrowWarps * 8;

// Barrier of the first kNarrowWarps warps with the or of `p`.
__device__ __forceinline__ int narrow_sync_or(int p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred a, b;\n\tsetp.ne.s32 a, %1, 0;\n\tbarrier.cta.red.or.pred b, 1, %2, a;\n\tselp.s32 %0, 1, 0, b;\n\t}"
      : "=r"(r) : "r"(p), "n"(kNarrowWarps * 32) : "memory");
  return r;
}
constexpr uint32_t kInitMark = 0xFFFFFFFEu;  // stamp of the round-0 items (CC)

// Warp-aggregated push: one shared atomic per warp that pushes anything.
__device__ __forceinline__ void smem_push(uint32_t* out, uint32_t* out_n, uint32_t cap, bool p, uint32_t v, uint32_t* err) {
  const unsigned m = __ballot_sync(kFull, p);
  if (m == 0) return;
  const int ld = __ffs(m) - 1;
  uint32_t pos = 0;
  if ((threadIdx.x & 31) == static_cast<uint32_t>(ld)) pos = atomicAdd(out_n, static_cast<uint32_t>(__popc(m)));
  pos = __shfl_sync(kFull, pos, ld) + __popc(m & lanemask_lt());
  if (p) {
    if (pos < cap) out[pos] = v;
    else atomicCAS(err, DERR_NONE, DERR_WL_OVERFLOW);
  }
}

// Relax edge k of a popped vertex whose operator value is `val` (BFS: the level
// to assign; SSSP: its distance; CC: its label): true when v is to be pushed.
template <uint32_t OP>
__device__ __forceinline__ bool smem_relax(const uint32_t* w, uint32_t* val_arr, uint32_t* stamp, uint32_t k, uint32_t v,
                                           uint32_t val, uint32_t r) {
  if (OP == OP_BFS) return val_arr[v] == kInf && atomicCAS(val_arr + v, kInf, val) == kInf;
  const uint32_t nd = OP == OP_SSSP ? val + w[k] : val;
  return nd < val_arr[v] && nd < atomicMin(val_arr + v, nd) && atomicExch(stamp + v, r) != r;
}

// A short list [b, e) walked by one lane.
template <uint32_t OP>
__device__ __forceinline__ void smem_walk(const uint32_t* col, const uint32_t* w, uint32_t* val_arr, uint32_t* stamp,
                                          uint32_t b, uint32_t e, uint32_t val, uint32_t r, uint32_t* out, uint32_t* out_n,
                                          uint32_t cap, uint32_t* err) {
  for (uint32_t k = b; k < e; ++k) {
    const uint32_t v = col[k];
    if (!smem_relax<OP>(w, val_arr, stamp, k, v, val, r)) continue;
    const uint32_t pos = atomicAdd(out_n, 1u);  // one instruction for the lanes that are here together
    if (pos < cap) out[pos] = v;
    else atomicCAS(err, DERR_NONE, DERR_WL_OVERFLOW);
  }
}

// A round over at most 8 * warps items by `warps` warps: four lanes per item, items
// dealt across the warps, so a short list is one step of one warp without a search
// for an edge's owner. Returns the edges of the lists this lane leads.
template <uint32_t OP>
__device__ __forceinline__ uint32_t smem_four(const uint32_t* in, uint32_t in_n, uint32_t warps, const uint32_t* rp,
                                              const uint32_t* col, const uint32_t* w, uint32_t* val, uint32_t* stamp,
                                              uint32_t r, uint32_t* out, uint32_t* out_n, uint32_t n, uint32_t* err) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & 3;
  if (warp >= in_n) return 0u;
  const uint32_t i = (lane >> 2) * warps + warp;
  uint32_t b = 0, e = 0, x = 0;
  if (i < in_n) {
    const uint32_t u = in[i];
    b = rp[u];
    e = rp[u + 1];
    x = OP == OP_BFS ? r + 1u : val[u];
  }
  const bool lng = e - b > 32u;
  const uint32_t trips = __reduce_max_sync(kFull, lng ? 0u : (e - b + 3u) >> 2);
  for (uint32_t t = 0; t < trips; ++t) {
    const uint32_t k = b + 4u * t + sub;
    const bool mine = !lng && k < e;
    const uint32_t v = mine ? col[k] : 0u;
    smem_push(out, out_n, n, mine && smem_relax<OP>(w, val, stamp, k, v, x, r), v, err);
  }
  for (unsigned mk = __ballot_sync(kFull, lng && sub == 0); mk; mk &= mk - 1) {
    const int ld = __ffs(mk) - 1;
    const uint32_t lb = __shfl_sync(kFull, b, ld), le = __shfl_sync(kFull, e, ld);
    const uint32_t lx = __shfl_sync(kFull, x, ld);
    for (uint32_t k0 = lb; k0 < le; k0 += 32) {
      const uint32_t k = k0 + lane;
      const uint32_t v = k < le ? col[k] : 0u;
      smem_push(out, out_n, n, k < le && smem_relax<OP>(w, val, stamp, k, v, lx, r), v, err);
    }
  }
  return sub == 0 ? e - b : 0u;
}

template <uint32_t OP>
__global__ void __launch_bounds__(kSmemCta, 1) k_smem_iterate(KParams p) {
  extern __shared__ __align__(16) uint32_t sh[];
  __shared__ uint32_t s_n[3];  // worklist sizes by round mod 3
  __shared__ uint32_t s_err;
  __shared__ uint32_t s_round, s_done;  // where the narrow rounds ended
  __shared__ unsigned long long s_edges;
  const unsigned long long t_start = p.trace ? globaltimer_ns() : 0ull;
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const uint32_t n = p.n;
  const uint32_t m = __ldg(p.row_ptr + n);
  uint32_t* rp = sh;
  uint32_t* col = rp + n + 1;
  uint32_t* w = col + m;
  uint32_t* val = w + (OP == OP_SSSP ? m : 0u);
  uint32_t* stamp = val + n;
  uint32_t* wl0 = stamp + (OP == OP_BFS ? 0u : n);
  uint32_t* wl1 = wl0 + n;
  if (tid == 0) {
    s_n[0] = s_n[1] = s_n[2] = 0;
    s_err = DERR_NONE;
    s_edges = 0;
  }
  // the graph, once (plain loads; the CSR arrays are read-only here)
  for (uint32_t i = tid; i <= n; i += kSmemCta) rp[i] = __ldg(p.row_ptr + i);
  for (uint32_t i = tid; i < m; i += kSmemCta) col[i] = __ldg(p.col + i);
  if (OP == OP_SSSP)
    for (uint32_t i = tid; i < m; i += kSmemCta) w[i] = static_cast<uint32_t>(__ldg(p.w + i));
  // Iterate initial values: BFS/SSSP INF (sources 0 below), CC label v
  for (uint32_t v = tid; v < n; v += kSmemCta) {
    val[v] = OP == OP_CC ? v : kInf;
    if (OP != OP_BFS) stamp[v] = kInf;
  }
  __syncthreads();
  // round-0 worklist: the caller's initial items (CC without them: every vertex)
  const uint32_t init_n = p.isrc_n ? p.isrc_n : p.init_count ? min(__ldcg(p.init_count), p.init_cap) : n;
  for (uint32_t base = 0; base < init_n; base += kSmemCta) {
    const uint32_t i = base + tid;
    bool push = false;
    uint32_t s = 0;
    if (i < init_n) {
      if (p.isrc_n) {
#pragma unroll
        for (uint32_t k = 0; k < kInlineSrc; ++k) s = i == k ? p.isrc[k] : s;
      } else {
        s = p.init_items ? __ldcg(p.init_items + i) : i;
      }
      // a repeated source or item is pushed once (CC: a mark no round id reaches, rounds stay below n)
      if (s >= n) atomicCAS(&s_err, DERR_NONE, DERR_BAD_ITEM);
      else push = OP == OP_CC ? atomicExch(stamp + s, kInitMark) != kInitMark : atomicExch(val + s, 0u) != 0u;
    }
    smem_push(wl0, &s_n[0], n, push, s, &s_err);
  }
  bool any_long = false;
  for (uint32_t v = tid; v < n; v += kSmemCta) any_long |= rp[v + 1] - rp[v] > kSmemLane;
  const bool longs = __syncthreads_or(any_long) != 0;
  trace_prologue(p.trace, p.trace_cap, t_start, s_n[0]);
  const uint32_t warp = tid >> 5;
  uint32_t edges = 0, rounds = 0, last_out = 0;
  bool done = false;
  for (uint32_t r = 0; !done; ++r) {
    const uint32_t in_n = min(s_n[r % 3], n);  // a worklist holds at most n items
    if (in_n <= kNarrow) {
      // narrow rounds, until the frontier outgrows them or the run ends; every thread
      // has read the sizes of the rounds before when they start to reuse the counters
      __syncthreads();
      if (warp < kNarrowWarps) {
        for (uint32_t now = in_n;; ++r) {
          uint32_t* const out_n = &s_n[(r + 1) % 3];
          if (tid == 0) s_n[(r + 2) % 3] = 0;
          edges += smem_four<OP>((r & 1) ? wl1 : wl0, now, kNarrowWarps, rp, col, w, val, stamp, r, (r & 1) ? wl0 : wl1,
                                 out_n, n, &s_err);
          const int bad = narrow_sync_or(*reinterpret_cast<volatile uint32_t*>(&s_err) != DERR_NONE);
          last_out = min(*reinterpret_cast<volatile uint32_t*>(out_n), n);
          rounds = r + 1;
          trace_round(p.trace, p.trace_cap, rounds, now, last_out);
          done = last_out == 0 || bad;
          if (!done && rounds >= p.max_rounds) {
            if (tid == 0) atomicCAS(&s_err, DERR_NONE, DERR_MAX_ROUNDS);
            done = true;
          }
          if (done || last_out > kNarrow) break;
          now = last_out;
        }
        if (tid == 0) {
          s_round = r;
          s_done = done;
        }
      }
      __syncthreads();
      r = s_round;  // the last round that ran
      done = s_done != 0;
      continue;
    }
    uint32_t* in = (r & 1) ? wl1 : wl0;
    uint32_t* out = (r & 1) ? wl0 : wl1;
    uint32_t* out_n = &s_n[(r + 1) % 3];
    // the counter of round r + 1's pushes: last read at the start of round r - 1, before its barrier
    if (tid == 0) s_n[(r + 2) % 3] = 0;
    if (in_n <= kSmemFour) {
      edges += smem_four<OP>(in, in_n, kSmemWarps, rp, col, w, val, stamp, r, out, out_n, n, &s_err);
    } else if (!longs) {
      // every list is short: items in worklist order, one per lane, which walks its list
      for (uint32_t i = tid; i < in_n; i += kSmemCta) {
        const uint32_t u = in[i], b = rp[u], e = rp[u + 1];
        smem_walk<OP>(col, w, val, stamp, b, e, OP == OP_BFS ? r + 1u : val[u], r, out, out_n, n, &s_err);
        edges += e - b;
      }
    } else {
      // lists of at most kSmemLane edges by the lane that holds the item; the longer
      // ones of the warp (items dealt across the warps, or in worklist order when there
      // is more than one per thread) have their edges dealt out to its lanes, two per
      // lane and step, owners by a shuffle search
      for (uint32_t base = 0; base < in_n; base += kSmemCta) {
        const uint32_t i = base + (in_n > kSmemCta ? tid : lane * kSmemWarps + ((warp + lane) & (kSmemWarps - 1u)));
        uint32_t b = 0, d = 0, x = 0;
        if (i < in_n) {
          const uint32_t u = in[i];
          b = rp[u];
          d = rp[u + 1] - b;
          x = OP == OP_BFS ? r + 1u : val[u];
        }
        edges += d;
        const unsigned lng = __ballot_sync(kFull, d > kSmemLane);
        if (d <= kSmemLane) {
          smem_walk<OP>(col, w, val, stamp, b, b + d, x, r, out, out_n, n, &s_err);
          d = 0;
        }
        __syncwarp();
        if (lng == 0) continue;
        const uint32_t incl = warp_incl_scan(d), excl = incl - d;
        const uint32_t total = __shfl_sync(kFull, incl, 31);
        for (uint32_t s = 0; s < total; s += 64) {
          uint32_t k[2], v[2], xx[2];
          bool mine[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint32_t ed = s + 32u * j + lane;
            mine[j] = ed < total;
            const uint32_t own = warp_find<uint32_t>(excl, mine[j] ? ed : total - 1u, 32);
            k[j] = __shfl_sync(kFull, b - excl, own) + ed;
            xx[j] = __shfl_sync(kFull, x, own);
            v[j] = mine[j] ? col[k[j]] : 0u;
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const bool push = mine[j] && smem_relax<OP>(w, val, stamp, k[j], v[j], xx[j], r);
            smem_push(out, out_n, n, push, v[j], &s_err);
          }
        }
      }
    }
    // the round's pushes are in; the only barrier of a round, and the error flag with it
    // (read after it, a thread already in the next round could split the CTA's decision)
    const int bad = __syncthreads_or(*reinterpret_cast<volatile uint32_t*>(&s_err) != DERR_NONE);
    last_out = min(*out_n, n);
    rounds = r + 1;
    trace_round(p.trace, p.trace_cap, rounds, in_n, last_out);
    done = last_out == 0 || bad;
    if (!done && rounds >= p.max_rounds) {
      if (tid == 0) atomicCAS(&s_err, DERR_NONE, DERR_MAX_ROUNDS);
      done = true;
    }
  }
  for (uint32_t v = tid; v < n; v += kSmemCta) __stcg(p.state + v, val[v]);
  // summed per warp: a 64-bit shared atomic by each of the 1024 threads took 13 us
  edges = __reduce_add_sync(kFull, edges);
  if (lane == 0) atomicAdd(&s_edges, static_cast<unsigned long long>(edges));
  __syncthreads();
  trace_end(p.trace, p.trace_cap, rounds);
  if (tid == 0) {
    DevStatus* st = p.st;
    atomicAdd(&st->edges, s_edges);
    st->rounds = rounds;
    st->last_out = last_out;
    if (s_err != DERR_NONE) atomicCAS(&st->err, DERR_NONE, s_err);
    if (p.rec != nullptr) write_rec(st, p.rec, p.rec_seq, rounds, last_out, __ldcg(&st->epoch));
  }
}

template <uint32_t OP>
cudaError_t launch_op(const KParams& p, size_t bytes, cudaStream_t s) {
  // the opt-in size is set per launch: cheap, and correct on any device current
  cudaError_t e = cudaFuncSetAttribute(k_smem_iterate<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(bytes));
  if (e != cudaSuccess) return e;
  k_smem_iterate<OP><<<1, kSmemCta, bytes, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

size_t smem_iterate_bytes(uint32_t op, uint32_t n, uint64_t m) {
  const uint64_t words = (n + 1ull) + m + (op == OP_SSSP ? m : 0ull) + n + (op == OP_BFS ? 0ull : n) + 2ull * n;
  return static_cast<size_t>(4ull * words);
}

bool smem_iterate_fits(uint32_t op, uint32_t n, uint64_t m, size_t limit) {
  if (op != OP_BFS && op != OP_SSSP && op != OP_CC) return false;
  if (n == 0 || m >= 0xFFFFFFFFull) return false;
  return smem_iterate_bytes(op, n, m) <= limit;
}

cudaError_t launch_smem_iterate(uint32_t op, const KParams& p, uint64_t m, cudaStream_t s) {
  const size_t bytes = smem_iterate_bytes(op, p.n, m);
  switch (op) {
    case OP_BFS: return launch_op<OP_BFS>(p, bytes, s);
    case OP_SSSP: return launch_op<OP_SSSP>(p, bytes, s);
    case OP_CC: return launch_op<OP_CC>(p, bytes, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace irgl
