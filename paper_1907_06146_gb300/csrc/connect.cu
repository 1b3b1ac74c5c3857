// Connectivity from the navigating nodes (Alg. 3: random navigating nodes NV, then
// "DFS-spanning" from each to strengthen connectivity; Sec. 4.1 defers the details to the
// NSG paper).
//
// Reading: for each root in the given order, mark everything reachable from it; while a
// node is unreached, take the smallest unreached id u, link u from the reached node v with
// a free slot (deg(v) < R) that minimises (d2(v, u), id), and mark everything reachable
// from u.  The reached set does not depend on the traversal order, so the GPU uses a
// level-synchronous frontier traversal (a visited bitmap with atomicOr) in place of a
// depth-first one and gets the same graph.  Once the first root reaches every node, a later
// root that reaches the first one reaches every node too and changes nothing: a beam search
// from it that meets the first root proves that, and only roots for which it does not are
// traversed (1M nodes, 10 roots: connectivity 6.8 -> 1.3 ms; 60,000 nodes 3.2 -> 0.4).  The argmin is taken in fp64 with the
// coordinate-order sum, so its ties resolve exactly as a sequential double loop would.
#include <climits>
#include <mutex>
#include <new>
#include <vector>

#include "common.cuh"
#include "graph_dev.cuh"
#include "knn.cuh"

namespace ssg {

// Exhaustive fp64 argmin (used only when the fp32 band below overflows its list).
__global__ void k_repair_dist(const float* __restrict__ X, int ld, int d, int64_t n,
                              const uint32_t* __restrict__ bm, const int32_t* __restrict__ deg,
                              int R, int64_t u, double* __restrict__ dv,
                              unsigned long long* __restrict__ best_bits) {
  const float* xu = X + u * ld;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const bool cand = ((bm[v >> 5] >> (v & 31)) & 1u) && deg[v] < R;
    double e = -1.0;
    if (cand) {
      e = dist2_f64(X + v * ld, xu, d);
      atomicMin(best_bits, (unsigned long long)__double_as_longlong(e));
    }
    dv[v] = e;
  }
}

__global__ void k_repair_pick_all(const double* __restrict__ dv, int64_t n,
                                  const unsigned long long* __restrict__ best_bits,
                                  int* __restrict__ best_id) {
  const unsigned long long b = *best_bits;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const double e = dv[v];
    if (e >= 0.0 && (unsigned long long)__double_as_longlong(e) == b) atomicMin(best_id, (int)v);
  }
}

// Device-side state of the connectivity of one root.
struct RepairState {
  unsigned long long u;  // smallest unreached id (n if none)
  unsigned hi_bits;      // smallest fp32 upper bound of d2(v, u) over the candidates
  int band;              // candidates whose fp32 lower bound reaches that upper bound
  int best;              // chosen v; one of the STOP codes when a kernel ends before u = n
  int cur;               // frontier buffer still to expand (0 or 1)
  int lvl[3];            // frontier sizes, by level mod 3; lvl[0] the next one to expand
  unsigned bar;          // grid barrier: arrivals since the launch
  int abort;             // a barrier timed out
  unsigned long long rep_full, rep_knn;  // repairs made, by the full scan and by kNN rows
};
constexpr int STOP_NONE = INT_MAX;  // no reached node has a free slot
constexpr int STOP_BAND = -2;       // the band list overflowed
constexpr int STOP_ROW = -3;        // u's kNN row settles nothing: the full scan takes u
constexpr int STOP_BFS = -4;        // u is linked, its traversal outgrew the block
constexpr int STOP_KNN = -5;        // unreached nodes remain, k_repair_knn is next
constexpr int STOP_RESCAN = -6;     // the band is taken again against hi_bits as it stands
constexpr int FIRST_BAND = 2048;    // band entries up to which that is not needed

__global__ void k_mark(uint32_t* __restrict__ bm, int32_t* __restrict__ frontier,
                       RepairState* __restrict__ s, int32_t root) {
  atomicOr(bm + (root >> 5), 1u << (root & 31));
  frontier[0] = root;
  s->cur = 0;
  s->lvl[0] = 1;
  s->lvl[1] = s->lvl[2] = 0;
}

struct ConnArgs {
  const float* X;
  int ld, d;
  int64_t n, nw;
  int32_t *adj, *deg;
  int R;
  uint32_t* bm;
  int32_t *f0, *f1;
  const int32_t* knn;     // nullable: exact kNN rows
  int K;
  float* d32;
  int32_t* band_ids;
  double* band_d;
  int cap;                // band entries
  float rel;
  RepairState* s;
  int64_t start;          // no unreached node lies in a bitmap word before this one
  int stop_at_knn;        // 1: after the first traversal leave the repairs to k_repair_knn
};

__device__ __forceinline__ uint32_t peek(const uint32_t* p) { return *(const volatile uint32_t*)p; }

// Smallest unreached id from bitmap word w0 on (n if none), by one warp.
__device__ __forceinline__ int64_t warp_first_unreached(const uint32_t* bits, int64_t nw, int64_t n,
                                                        int64_t w0) {
  const int lane = lane_id();
  for (int64_t b = w0; b < nw; b += 128) {
    uint32_t word[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t w = b + j * 32 + lane;
      word[j] = w < nw ? peek(bits + w) : 0xffffffffu;
      if (w == nw - 1 && (n & 31)) word[j] |= ~((1u << (n & 31)) - 1u);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned bal = __ballot_sync(0xffffffffu, word[j] != 0xffffffffu);
      if (bal) {
        const int l = __ffs(bal) - 1;
        const uint32_t w = __shfl_sync(0xffffffffu, word[j], l);
        return (b + j * 32 + l) * 32 + __ffs(~w) - 1;
      }
    }
  }
  return n;
}

// Expands one node by a warp: its unreached neighbours are marked and appended to next.
__device__ __forceinline__ void warp_expand(const ConnArgs& a, uint32_t* bits, int32_t node,
                                            int32_t* next, int* ncount) {
  const int lane = lane_id();
  const int dg = __ldcg(a.deg + node);
  for (int c = 0; c < dg; c += 32) {
    const int t = c + lane;
    bool fresh = false;
    int32_t v = 0;
    if (t < dg) {
      v = __ldcg(a.adj + (int64_t)node * a.R + t);
      const uint32_t bit = 1u << (v & 31);
      // most neighbours are reached already: a read first spares their atomics
      if (!(peek(bits + (v >> 5)) & bit)) fresh = !(atomicOr(bits + (v >> 5), bit) & bit);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, fresh);
    int basep = 0;
    if (lane == 0 && bal) basep = atomicAdd(ncount, __popc(bal));
    basep = __shfl_sync(0xffffffffu, basep, 0);
    if (fresh) next[basep + __popc(bal & lanemask_lt())] = v;
  }
}

// A level of a traversal that a whole block of k_repair_knn expands (block_level): the leading warp
// sets it, the others wait for it at REPAIR_BAR.
constexpr int REPAIR_THREADS = 512;
struct BlockLevel {
  const int32_t* fr;  // its nodes
  int32_t* nx;        // those reached from it
  int fc, count;      // their numbers; fc = 0: no more levels come
};
__device__ __forceinline__ void repair_bar() {
  __syncwarp();
  asm volatile("barrier.sync 1, %0;" ::"n"(REPAIR_THREADS) : "memory");
}
// All warps: a node each at a time, the next one's row and degree loading meanwhile.
__device__ __forceinline__ void block_level(const ConnArgs& a, uint32_t* bits, BlockLevel* b) {
  constexpr int NW = REPAIR_THREADS / 32;
  const int lane = lane_id(), fc = b->fc;
  int64_t node;
  int32_t v = -1;
  int dg = 0;
  auto fetch = [&](int w) {
    node = __ldcg(b->fr + w);
    v = lane < a.R ? __ldcg(a.adj + node * a.R + lane) : -1;
    dg = __ldcg(a.deg + node);
  };
  int w = threadIdx.x >> 5;
  if (w < fc) fetch(w);
  for (; w < fc; w += NW) {
    const int64_t here = node;
    const int32_t first = v;
    const int n = dg;
    if (w + NW < fc) fetch(w + NW);
    for (int c = 0; c < n; c += 32) {
      const int t = c + lane;
      const int32_t x = t >= n ? 0 : c == 0 ? first : __ldcg(a.adj + here * a.R + t);
      const uint32_t bit = 1u << (x & 31);
      const bool fresh = t < n && !(peek(bits + (x >> 5)) & bit) && !(atomicOr(bits + (x >> 5), bit) & bit);
      const unsigned bal = __ballot_sync(0xffffffffu, fresh);
      int base = 0;
      if (lane == 0 && bal) base = atomicAdd(&b->count, __popc(bal));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (fresh) b->nx[base + __popc(bal & lanemask_lt())] = x;
    }
  }
}

// Repairs that kNN rows settle, back to back by one warp.  A row lists u's K nearest nodes in
// exact (d2, id) order, so when some of them is reached and has a free slot the first such one
// is the (d2, id)-smallest of all reached nodes with a free slot: the same choice as the
// argmin over all n nodes, without a pass over them.  Each round: the smallest unreached u,
// the link from the first qualifying row entry, and the traversal from u while its frontier
// stays small.  bits: the bitmap of reached nodes (in shared or global memory).  Returns
// (in every lane) n when every node is reached, else the node it stopped at, with
// *why = STOP_ROW, STOP_KNN after `most` repairs, or STOP_BFS and the frontier in the state.  A repair is a chain of
// latencies, so the rows, out-edges and degrees of the next two unreached nodes (which no repair
// before their own changes) load while the current one is settled, and the degrees of the next
// one's row entries too (a repair changes one degree, the one it links from).
// Traversals: levels of up to four nodes by this warp, larger ones by its block (level, not null:
// up to 4,096 nodes) or, within k_connect, by the grid, which also takes over after 64 levels (its
// other blocks wait meanwhile).  60 islands of 640 nodes, each entered by a row: 25 ms where this
// warp took levels of up to 256 nodes alone, now 3.1.
struct RepairRow {
  static constexpr int PIECES = 4;  // of 32 entries, kept in registers
  int64_t u;
  int32_t row[PIECES], adj[PIECES], rdeg[PIECES];
  int dg;
  __device__ __forceinline__ void fetch(const ConnArgs& a, int64_t node) {
    const int lane = lane_id();
    u = node;
    const bool in = u < a.n;
    dg = in ? __ldcg(a.deg + u) : 0;
#pragma unroll
    for (int j = 0; j < PIECES; ++j) {
      const int t = j * 32 + lane;
      row[j] = in && t < a.K ? __ldg(a.knn + u * a.K + t) : -1;
      adj[j] = in && t < a.R ? __ldcg(a.adj + u * a.R + t) : -1;
    }
  }
  __device__ __forceinline__ void fetch_degrees(const ConnArgs& a) {
#pragma unroll
    for (int j = 0; j < PIECES; ++j) rdeg[j] = row[j] >= 0 ? __ldcg(a.deg + row[j]) : a.R;
  }
  // `v` has been linked from since fetch_degrees
  __device__ __forceinline__ void linked(int32_t v) {
#pragma unroll
    for (int j = 0; j < PIECES; ++j) rdeg[j] += row[j] == v ? 1 : 0;
  }
};
__device__ __noinline__ int64_t warp_knn_repairs(const ConnArgs& a, uint32_t* bits, int64_t start,
                                                 int most, BlockLevel* level, int* why) {
  constexpr int ALONE = 4;  // frontier nodes that this warp expands itself
  constexpr int P = RepairRow::PIECES;
  const int lane = lane_id();
  RepairState* s = a.s;
  unsigned long long made = 0;
  *why = 0;
  // marks v and appends it to the list, if it is unreached (v < 0: nothing)
  auto reach = [&](int32_t v, int32_t* list, int& count) {
    const uint32_t bit = 1u << (v & 31);
    bool fresh = v >= 0 && !(peek(bits + (v >> 5)) & bit);
    if (!__any_sync(0xffffffffu, fresh)) return;
    if (fresh) fresh = !(atomicOr(bits + (v >> 5), bit) & bit);
    const unsigned bal = __ballot_sync(0xffffffffu, fresh);
    if (fresh) list[count + __popc(bal & lanemask_lt())] = v;
    count += __popc(bal);
  };
  // the smallest unreached node after u
  auto after = [&](int64_t u) -> int64_t {
    if (u >= a.n) return a.n;
    const uint32_t w = peek(bits + (u >> 5)) | ((2u << (u & 31)) - 1u);
    const int64_t g = w != 0xffffffffu ? (u >> 5) * 32 + __ffs(~w) - 1
                                       : warp_first_unreached(bits, a.nw, a.n, (u >> 5) + 1);
    return g < a.n ? g : a.n;
  };
  auto unreached = [&](int64_t u) {
    return u < a.n && !((peek(bits + (u >> 5)) >> (u & 31)) & 1u);
  };
  RepairRow now, n1, n2;
  now.fetch(a, warp_first_unreached(bits, a.nw, a.n, start));
  now.fetch_degrees(a);
  n1.fetch(a, after(now.u));
  while (now.u < a.n) {
    const int64_t u = now.u;
    if (made >= (unsigned long long)most) {
      *why = STOP_KNN;
      break;
    }
    n2.fetch(a, after(n1.u));
    n1.fetch_degrees(a);
    // the row's first reached node with a free slot
    int32_t found = -1;
    int slot = 0;
#pragma unroll
    for (int j = 0; j < P; ++j) {
      if (found < 0 && j * 32 < a.K) {
        const int32_t v = now.row[j];
        const unsigned bal = __ballot_sync(
            0xffffffffu, v >= 0 && now.rdeg[j] < a.R && ((peek(bits + (v >> 5)) >> (v & 31)) & 1u));
        if (bal) {
          found = __shfl_sync(0xffffffffu, v, __ffs(bal) - 1);
          slot = __shfl_sync(0xffffffffu, now.rdeg[j], __ffs(bal) - 1);
        }
      }
    }
    for (int c = P * 32; c < a.K && found < 0; c += 32) {
      const int32_t v = c + lane < a.K ? __ldg(a.knn + u * a.K + c + lane) : -1;
      const bool reached = v >= 0 && ((peek(bits + (v >> 5)) >> (v & 31)) & 1u);
      if (!__any_sync(0xffffffffu, reached)) continue;
      const int dv = reached ? __ldcg(a.deg + v) : a.R;
      const unsigned bal = __ballot_sync(0xffffffffu, dv < a.R);
      if (bal) {
        found = __shfl_sync(0xffffffffu, v, __ffs(bal) - 1);
        slot = __shfl_sync(0xffffffffu, dv, __ffs(bal) - 1);
      }
    }
    if (found < 0) {
      *why = STOP_ROW;
      break;
    }
    if (lane == 0) {
      a.adj[(int64_t)found * a.R + slot] = (int32_t)u;
      a.deg[found] = slot + 1;
      atomicOr(bits + (u >> 5), 1u << (u & 31));
    }
    ++made;
    __syncwarp();
    int32_t *fr = a.f1, *nx = a.f0;
    int fc = 0;
#pragma unroll
    for (int j = 0; j < P; ++j)
      if (j * 32 < now.dg) reach(j * 32 + lane < now.dg ? now.adj[j] : -1, fr, fc);
    for (int c = P * 32; c < now.dg; c += 32)
      reach(c + lane < now.dg ? __ldcg(a.adj + u * a.R + c + lane) : -1, fr, fc);
    __syncwarp();
    for (int levels = 0; fc > 0 && (level ? fc <= 4096 : fc <= ALONE && levels < 64); ++levels) {
      int nc = 0;
      if (fc > ALONE) {
        if (lane == 0) *level = BlockLevel{fr, nx, fc, 0};
        repair_bar();
        block_level(a, bits, level);
        repair_bar();
        nc = level->count;
      }
      for (int w = 0; fc <= ALONE && w < fc; ++w) {
        const int32_t node = __ldcg(fr + w);
        const int dg = __ldcg(a.deg + node);
        for (int c = 0; c < dg; c += 32)
          reach(c + lane < dg ? __ldcg(a.adj + (int64_t)node * a.R + c + lane) : -1, nx, nc);
      }
      __syncwarp();
      int32_t* t = fr;
      fr = nx;
      nx = t;
      fc = nc;
    }
    if (fc > 0) {
      if (lane == 0) {
        s->cur = fr == a.f1 ? 1 : 0;
        s->lvl[0] = fc;
        s->lvl[1] = s->lvl[2] = 0;
      }
      *why = STOP_BFS;
      break;
    }
    // the traversal may have reached the nodes fetched ahead
    if (n1.u >= a.n || unreached(n1.u)) {
      now = n1;
      now.linked(found);
      if (n2.u >= a.n || unreached(n2.u))
        n1 = n2;
      else
        n1.fetch(a, after(now.u));
    } else {
      now.fetch(a, after(u));
      now.fetch_degrees(a);
      n1.fetch(a, after(now.u));
    }
  }
  if (lane == 0) s->rep_knn += made;
  __threadfence();
  __syncwarp();
  return now.u;
}

// warp_knn_repairs with the bitmap in shared memory where it fits (up to 1.6M nodes): a chain
// of dependent reads, each a shared-memory or an L2 latency.  200,000 nodes, 4,500 repairs:
// 7.6 ms; one block that met at about ten barriers per repair took 15.5 ms.  The other warps only
// take part in traversals.
__global__ void __launch_bounds__(REPAIR_THREADS, 1) k_repair_knn(ConnArgs a, int shared_bits) {
  extern __shared__ uint32_t sbits[];
  __shared__ BlockLevel level;
  uint32_t* bits = a.bm;
  if (shared_bits) {
    for (int64_t w = threadIdx.x; w < a.nw; w += blockDim.x) sbits[w] = a.bm[w];
    bits = sbits;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    int why;
    const int64_t u = warp_knn_repairs(a, bits, a.start, INT_MAX, &level, &why);
    if (threadIdx.x == 0) {
      a.s->u = (unsigned long long)u;
      a.s->best = u < a.n ? why : STOP_NONE;
      level.fc = 0;
    }
    repair_bar();
  } else {
    for (;;) {
      repair_bar();
      if (level.fc == 0) break;
      block_level(a, bits, &level);
      repair_bar();
    }
  }
  __syncthreads();
  if (shared_bits)
    for (int64_t w = threadIdx.x; w < a.nw; w += blockDim.x) a.bm[w] = sbits[w];
}

// Barrier of the whole (cooperative) grid, bounded: false, in every thread, once a block has
// waited about 20 s or another one gave up.  phase: barriers so far (the same in every block).
__device__ __forceinline__ bool grid_barrier(RepairState* s, unsigned& phase) {
  __shared__ int ok;
  __syncthreads();
  ++phase;
  if (threadIdx.x == 0) {
    const unsigned target = phase * gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&s->bar) : "memory");
    unsigned long long t0 = 0;
    ok = 1;
    for (unsigned spins = 0;; ++spins) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&s->bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if (spins < 64) continue;
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      if (*(volatile int*)&s->abort || t - t0 > 20000000000ull) {
        *(volatile int*)&s->abort = 1;
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
  }
  __syncthreads();
  return ok != 0;
}

// Levels of up to LONE_LEVEL nodes by one block (all its threads), from the fc nodes in fr, while
// the other blocks wait at the grid's barrier: a warp per node, the lists also in shared memory.
// Stops at an empty or larger level, whose nodes it leaves in nx, and after LONE_RUN levels (the
// barrier's waits are bounded); returns its size.  Bound by a level's chain of row load, atomic and
// block barrier, about 0.8 us; the grid's barrier made it 2.6 us where k_connect took every
// level (a path of 30,000 nodes: 87 ms, now 22).
constexpr int LONE_LEVEL = 32, LONE_RUN = 4096;
__device__ __noinline__ int lone_levels(const ConnArgs& a, int32_t* fr, int32_t* nx, int fc) {
  __shared__ int32_t list[2][LONE_LEVEL];
  __shared__ int size[3];
  const int lane = lane_id(), warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  if (threadIdx.x < 3) size[threadIdx.x] = 0;
  if (threadIdx.x < fc) list[0][threadIdx.x] = __ldcg(fr + threadIdx.x);
  __syncthreads();
  int l = 0;
  for (; fc > 0 && fc <= LONE_LEVEL && l < LONE_RUN; ++l) {
    int32_t* to = l & 1 ? fr : nx;
    int32_t* sl = list[(l + 1) & 1];
    int* count = &size[(l + 1) % 3];
    if (threadIdx.x == 0) size[(l + 2) % 3] = 0;
    for (int w = warp; w < fc; w += nwarps) {
      const int64_t node = list[l & 1][w];
      const int32_t* row = a.adj + node * a.R;
      int32_t v = lane < a.R ? __ldcg(row + lane) : -1;
      const int dg = __ldcg(a.deg + node);
      for (int c = 0; c < dg; c += 32) {
        const int t = c + lane;
        if (c > 0 && t < dg) v = __ldcg(row + t);
        const uint32_t bit = 1u << (v & 31);
        const bool fresh = t < dg && !(atomicOr(a.bm + (v >> 5), bit) & bit);
        const unsigned bal = __ballot_sync(0xffffffffu, fresh);
        int base = 0;
        if (lane == 0 && bal) base = atomicAdd(count, __popc(bal));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(bal & lanemask_lt());
        if (fresh) to[base] = v;
        if (fresh && base < LONE_LEVEL) sl[base] = v;
      }
    }
    __syncthreads();
    fc = *count;
  }
  if (!(l & 1))
    for (int i = threadIdx.x; i < fc; i += blockDim.x) nx[i] = __ldcg(fr + i);
  return fc;
}

// Level-synchronous traversal by the whole grid from frontier buffer s->cur (lvl[0] nodes), a
// warp per node: frontier sizes go round lvl[0..2], level l clearing the counter that level
// l + 1 fills, and a barrier at the end, after which the state may change.  Small levels are block
// 0's alone, several for one barrier.  False if a barrier gave up.
__device__ __forceinline__ bool grid_bfs(const ConnArgs& a, unsigned& phase) {
  RepairState* s = a.s;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t gw = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int cur = *(volatile int*)&s->cur;
  for (int l = 0;; ++l) {
    const int fc = *(volatile int*)&s->lvl[l % 3];
    if (fc == 0) return grid_barrier(s, phase);
    if (blockIdx.x == 0 && threadIdx.x == 0) s->lvl[(l + 2) % 3] = 0;
    int32_t* fr = cur ? a.f1 : a.f0;
    int32_t* nx = cur ? a.f0 : a.f1;
    if (fc > LONE_LEVEL) {
      for (int64_t w = gw; w < fc; w += nwarps)
        warp_expand(a, a.bm, __ldcg(fr + w), nx, &s->lvl[(l + 1) % 3]);
    } else if (blockIdx.x == 0) {
      const int left = lone_levels(a, fr, nx, fc);
      if (threadIdx.x == 0) s->lvl[(l + 1) % 3] = left;
    }
    if (!grid_barrier(s, phase)) return false;
    cur ^= 1;
  }
}

// Distances of U rows to b by a team of 8 lanes, each summed as team8_dist sums it; a step's loads
// are all issued before its first product.
template <int U>
__device__ __forceinline__ void team8_dists(const float* const (&a)[U], const float* __restrict__ b,
                                            int ld4, int tl, const bool (&valid)[U], float (&s)[U]) {
#pragma unroll
  for (int r = 0; r < U; ++r) s[r] = 0.f;
  for (int f = tl; f < ld4; f += 8) {
    const float4 y = __ldg((const float4*)b + f);
    float4 x[U];
#pragma unroll
    for (int r = 0; r < U; ++r) x[r] = valid[r] ? __ldg((const float4*)a[r] + f) : y;
#pragma unroll
    for (int r = 0; r < U; ++r) {
      float u;
      u = x[r].x - y.x; s[r] = fmaf(u, u, s[r]);
      u = x[r].y - y.y; s[r] = fmaf(u, u, s[r]);
      u = x[r].z - y.z; s[r] = fmaf(u, u, s[r]);
      u = x[r].w - y.w; s[r] = fmaf(u, u, s[r]);
    }
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
#pragma unroll
    for (int r = 0; r < U; ++r) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
  }
}

// (d2, id)-smallest over the block (every thread returns it); bd / bi: 32 entries each.
__device__ __forceinline__ void block_argmin(double& best, int& bid, double* bd, int* bi) {
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bid, o);
    if (ob < best || (ob == best && oi < bid)) {
      best = ob;
      bid = oi;
    }
  }
  const int w = threadIdx.x >> 5, lane = lane_id();
  __syncthreads();
  if (lane == 0) {
    bd[w] = best;
    bi[w] = bid;
  }
  __syncthreads();
  for (int t = 0; t < (int)(blockDim.x >> 5); ++t)
    if (bd[t] < best || (bd[t] == best && bi[t] < bid)) {
      best = bd[t];
      bid = bi[t];
    }
}

// The connectivity of one root by one cooperative grid: the traversal from the frontier in the
// state, then (unless stop_at_knn) repairs until every node is reached.  A repair: the smallest
// unreached u; where kNN rows are given, first those that they settle (one warp of block 0, a
// few of them: the bitmap is not in its shared memory, so it leaves many to k_repair_knn);
// else the full scan: fp32 distances of every reached node with a free slot by teams of 8
// lanes; the fp64 distances of those whose lower bound reaches the smallest upper bound seen by
// then (its block's at most, so a superset of the band that can hold the minimum; a warp each);
// then, in block 0, the (d2, id)-smallest of them, re-taken in coordinate order among those
// within fp64_order_rel of the smallest.  Two grid barriers per repair; a host round trip and
// seven launches took 60 us (30,011 x 100, 172 repairs: 12.7 -> 5.0 ms).  Where the superset is
// large (distances that take few values: every block may hold thousands of ties at its own
// smallest one), the band is taken again from the stored fp32 distances, against the smallest
// bound of the whole grid, and only that band counts towards the list's room.
__global__ void __launch_bounds__(512, 2) k_connect(ConnArgs a) {
  __shared__ double bd[32];
  __shared__ int bi[32];
  __shared__ int nties;
  __shared__ unsigned bmin;
  RepairState* s = a.s;
  unsigned phase = 0;
  const int lane = lane_id(), team = lane >> 3, tl = lane & 7, warp = threadIdx.x >> 5;
  const int64_t gw = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const double INF = __longlong_as_double(0x7ff0000000000000ll);
  int64_t start = a.start;
  // block 0, warp 0: the next node that needs the full scan (or what ends this kernel)
  auto next_node = [&]() {
    int why = STOP_ROW;
    int64_t u;
    if (a.knn && !a.stop_at_knn)
      u = warp_knn_repairs(a, a.bm, start, 16, nullptr, &why);
    else
      u = warp_first_unreached(a.bm, a.nw, a.n, start);
    start = u >> 5;
    if (lane == 0) {
      s->hi_bits = 0x7f800000u;
      s->band = 0;
      s->best = a.stop_at_knn ? STOP_KNN : why;
      s->u = (unsigned long long)u;
    }
  };
  if (!grid_bfs(a, phase)) return;
  if (blockIdx.x == 0 && warp == 0) next_node();
  for (;;) {
    if (!grid_barrier(s, phase)) return;
    const int64_t u = (int64_t)*(volatile unsigned long long*)&s->u;
    const int what = *(volatile int*)&s->best;
    if (u >= a.n || (what != STOP_BFS && what != STOP_ROW && what != STOP_RESCAN)) return;
    if (what == STOP_BFS) {
      if (!grid_bfs(a, phase)) return;
      if (blockIdx.x == 0 && warp == 0) next_node();
      continue;
    }
    const float* xu = a.X + u * a.ld;
    const int room = what == STOP_RESCAN ? a.cap : min(a.cap, FIRST_BAND);
    float hi;
    if (what == STOP_RESCAN) {
      hi = __uint_as_float(*(volatile unsigned*)&s->hi_bits);
    } else {
      if (threadIdx.x == 0) bmin = 0x7f800000u;
      __syncthreads();
      float best = __int_as_float(0x7f800000);
      constexpr int U = 4;
      for (int64_t v0 = gw * 4; v0 < a.n; v0 += nwarps * 4 * U) {
        const float* row[U];
        bool cand[U];
        float e[U];
#pragma unroll
        for (int r = 0; r < U; ++r) {
          const int64_t v = v0 + r * nwarps * 4 + team;
          const uint32_t word = v < a.n ? __ldcg(a.bm + (v >> 5)) : 0u;
          const int dg = v < a.n ? __ldcg(a.deg + v) : a.R;
          cand[r] = ((word >> (v & 31)) & 1u) && dg < a.R;
          row[r] = a.X + (cand[r] ? v : 0) * a.ld;
        }
        team8_dists<U>(row, xu, a.ld >> 2, tl, cand, e);
#pragma unroll
        for (int r = 0; r < U; ++r) {
          const int64_t v = v0 + r * nwarps * 4 + team;
          if (tl == 0 && v < a.n) a.d32[v] = cand[r] ? e[r] : -1.f;
          if (cand[r]) best = fminf(best, e[r]);
        }
      }
      for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
      if (lane == 0 && best < __int_as_float(0x7f800000))
        atomicMin(&bmin, __float_as_uint(best * (1.f + 2.f * a.rel) + 1e-30f));
      __syncthreads();
      if (threadIdx.x == 0 && bmin != 0x7f800000u) bmin = min(bmin, atomicMin(&s->hi_bits, bmin));
      __syncthreads();
      hi = __uint_as_float(bmin);
    }
    for (int64_t v0 = gw * 4; v0 < a.n; v0 += nwarps * 32) {
      // this warp's own distances: four nodes of each of eight rounds
      const int64_t v1 = v0 + (int64_t)(lane >> 2) * nwarps * 4 + (lane & 3);
      const float e = v1 < a.n ? __ldcg(a.d32 + v1) : -1.f;
      unsigned bal = __ballot_sync(0xffffffffu, e >= 0.f && e * (1.f - 2.f * a.rel) <= hi);
      while (bal) {
        const int l = __ffs(bal) - 1;
        bal &= bal - 1;
        const int64_t v = __shfl_sync(0xffffffffu, v1, l);
        int p = 0;
        if (lane == 0) p = atomicAdd(&s->band, 1);
        p = __shfl_sync(0xffffffffu, p, 0);
        if (p >= room) break;
        const double x = warp_dist2_f64(a.X + v * a.ld, xu, a.d);
        if (lane == 0) {
          a.band_ids[p] = (int32_t)v;
          a.band_d[p] = x;
        }
      }
    }
    if (!grid_barrier(s, phase)) return;
    if (blockIdx.x != 0) continue;
    // block 0 links the smallest, expands u, and finds the next node
    const int m = *(volatile int*)&s->band;
    if (m == 0 || m > room) {
      if (threadIdx.x == 0) {
        s->best = m == 0 ? STOP_NONE : what == STOP_RESCAN ? STOP_BAND : STOP_RESCAN;
        s->band = 0;
      }
      continue;
    }
    double b1 = INF;
    int bid = INT_MAX;
    for (int t = threadIdx.x; t < m; t += blockDim.x) {
      const double x = __ldcg(a.band_d + t);
      const int v = __ldcg(a.band_ids + t);
      if (x < b1 || (x == b1 && v < bid)) {
        b1 = x;
        bid = v;
      }
    }
    if (threadIdx.x == 0) nties = 0;
    block_argmin(b1, bid, bd, bi);
    const double lim = b1 + fp64_order_rel(a.d) * b1;
    int mine = 0;
    for (int t = threadIdx.x; t < m; t += blockDim.x) mine += __ldcg(a.band_d + t) <= lim;
    if (mine) atomicAdd(&nties, mine);
    __syncthreads();
    if (nties > 1) {
      double b2 = INF;
      int i2 = INT_MAX;
      for (int t = threadIdx.x; t < m; t += blockDim.x) {
        if (__ldcg(a.band_d + t) > lim) continue;
        const int v = __ldcg(a.band_ids + t);
        const double x = dist2_f64(a.X + (int64_t)v * a.ld, xu, a.d);
        if (x < b2 || (x == b2 && v < i2)) {
          b2 = x;
          i2 = v;
        }
      }
      block_argmin(b2, i2, bd, bi);
      bid = i2;
    }
    if (warp == 0) {
      if (lane == 0) {
        const int dv = __ldcg(a.deg + bid);
        a.adj[(int64_t)bid * a.R + dv] = (int32_t)u;
        a.deg[bid] = dv + 1;
        atomicOr(a.bm + (u >> 5), 1u << (u & 31));
        s->rep_full += 1;
        s->cur = 1;
        s->lvl[0] = s->lvl[1] = s->lvl[2] = 0;
      }
      __threadfence();
      __syncwarp();
      warp_expand(a, a.bm, (int32_t)u, a.f1, &s->lvl[0]);
      __threadfence();
      __syncwarp();
      start = u >> 5;
      if (*(volatile int*)&s->lvl[0] > 0) {
        if (lane == 0) s->best = STOP_BFS;
      } else {
        next_node();
      }
    }
    __syncthreads();
  }
}

// Link v = *best_id (after the exhaustive argmin) and make u the next frontier.
__global__ void k_add_edge(int32_t* __restrict__ adj, int32_t* __restrict__ deg, int R,
                           const int* __restrict__ best_id, uint32_t* __restrict__ bm,
                           int32_t* __restrict__ frontier, RepairState* __restrict__ s) {
  const int v = *best_id;
  s->best = v;
  if (v == INT_MAX) return;
  const int64_t u = (int64_t)s->u;
  adj[(int64_t)v * R + deg[v]] = (int32_t)u;
  deg[v] += 1;
  atomicOr(bm + (u >> 5), 1u << (u & 31));
  frontier[0] = (int32_t)u;
  s->cur = 0;
  s->lvl[0] = 1;
  s->lvl[1] = s->lvl[2] = 0;
  s->rep_full += 1;
}

// Launches k_connect and reads the state back.
static RepairState run_connect(ConnArgs a, cudaStream_t st) {
  SSG_CUDA(cudaMemsetAsync(&a.s->bar, 0, sizeof(unsigned), st));
  static const int per_sm = [] {
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_connect, 512, 0);
    return b;
  }();
  SSG_REQUIRE(per_sm >= 1, SSG_ECUDA, "connectivity: no room for the grid kernel");
  // one block per SM for large graphs; few nodes need few blocks (a barrier's cost grows
  // with them)
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(num_sms(), ceil_div(a.n, 128)));
  void* args[] = {&a};
  SSG_CUDA(cudaLaunchCooperativeKernel((const void*)k_connect, dim3(grid), dim3(512), args, 0, st));
  g_launches.fetch_add(1, std::memory_order_relaxed);
  ++t_launches;
  RepairState h;
  SSG_CUDA(cudaMemcpyAsync(&h, a.s, sizeof(h), cudaMemcpyDeviceToHost, st));
  SSG_CUDA(cudaStreamSynchronize(st));
  if (h.abort) note_device_status(SSG_ETIMEOUT);
  SSG_REQUIRE(!h.abort, SSG_ETIMEOUT, "connectivity: a grid barrier timed out");
  return h;
}

// One root: its traversal and the repairs until it reaches every node.  on_band(u): the
// caller's way out when the fp64 band of one repair overflows (it links u).
template <class F>
static void connect_root(ConnArgs a, int32_t root, cudaStream_t st, F on_band) {
  SSG_CUDA(cudaMemsetAsync(a.bm, 0, sizeof(uint32_t) * a.nw, st));
  SSG_LAUNCH(k_mark, 1, 1, 0, st, a.bm, a.f0, a.s, root);
  a.start = 0;
  a.stop_at_knn = a.knn != nullptr;
  RepairState h = run_connect(a, st);
  a.stop_at_knn = 0;
  while ((int64_t)h.u < a.n) {
    a.start = (int64_t)h.u >> 5;
    if (h.best == STOP_KNN && a.knn) {
      const size_t smem = (size_t)a.nw * sizeof(uint32_t);
      const bool shared = smem <= 200 * 1024;
      if (shared) ensure_smem((const void*)k_repair_knn, smem);
      SSG_LAUNCH(k_repair_knn, 1, REPAIR_THREADS, shared ? smem : 0, st, a, shared ? 1 : 0);
      SSG_CUDA(cudaMemcpyAsync(&h, a.s, sizeof(h), cudaMemcpyDeviceToHost, st));
      SSG_CUDA(cudaStreamSynchronize(st));
      if ((int64_t)h.u >= a.n) break;
      a.start = (int64_t)h.u >> 5;
      if (h.best == STOP_ROW) {  // no frontier is left
        const int none[3] = {0, 0, 0};
        SSG_CUDA(cudaMemcpyAsync(a.s->lvl, none, sizeof(none), cudaMemcpyHostToDevice, st));
      }
    } else if (h.best == STOP_BAND) {
      on_band(h);
    }
    SSG_REQUIRE(h.best != STOP_NONE, SSG_EINTERNAL,
                "connectivity: node %lld is unreached and no reached node has a free slot",
                (long long)h.u);
    h = run_connect(a, st);
  }
}

__global__ void k_repeat_row(const float* __restrict__ x, int ld, float* __restrict__ out) {
  for (int t = threadIdx.x; t < ld; t += blockDim.x) out[(size_t)blockIdx.x * ld + t] = x[t];
}

// Whether each later root provably reaches the first one (which reaches every node): a beam
// search from it towards the first root's vector meets that node.
static std::vector<char> roots_reach_first(const ConnArgs& a, const int32_t* nav_host, int n_nav,
                                           cudaStream_t st) {
  std::vector<char> ok((size_t)n_nav, 0);
  const int m = n_nav - 1;
  if (m < 1 || a.R > 128) return ok;
  const int ls = 16;
  Scratch<float> q((size_t)m * a.ld, st);
  Scratch<int32_t> from((size_t)m, st), ids((size_t)m, st);
  SSG_LAUNCH(k_repeat_row, (unsigned)m, 128, 0, st, a.X + (int64_t)nav_host[0] * a.ld, a.ld, q.p);
  SSG_CUDA(cudaMemcpyAsync(from.p, nav_host + 1, sizeof(int32_t) * m, cudaMemcpyHostToDevice, st));
  if (!search_from(a.X, a.ld, a.d, a.adj, a.deg, a.R, from.p, q.p, a.ld, m, ls, ids.p, st)) return ok;
  std::vector<int32_t> h((size_t)m);
  SSG_CUDA(cudaMemcpyAsync(h.data(), ids.p, sizeof(int32_t) * m, cudaMemcpyDeviceToHost, st));
  SSG_CUDA(cudaStreamSynchronize(st));
  for (int t = 0; t < m; ++t) ok[(size_t)t + 1] = h[(size_t)t] == nav_host[0];
  return ok;
}

int64_t connect_run(const float* X, int ld, int d, int64_t n, int32_t* adj, int32_t* deg,
                    int R, const int32_t* nav_host, int n_nav,
                    cudaStream_t st, const int32_t* knn, int K, int64_t* knn_repairs) {
  const int64_t nw = ceil_div(n, 32);
  const int cap = 1 << 16;
  Scratch<uint32_t> bm((size_t)nw, st);
  Scratch<int32_t> f0((size_t)n, st), f1((size_t)n, st), band_ids((size_t)cap, st);
  Scratch<double> band_d((size_t)cap, st);
  Scratch<float> d32((size_t)n, st);
  Scratch<RepairState> state(1, st);
  SSG_CUDA(cudaMemsetAsync(state.p, 0, sizeof(RepairState), st));
  Scratch<unsigned long long> ull(1, st);
  Scratch<double> dv;
  ConnArgs a{X, ld, d, n, nw, adj, deg, R, bm.p, f0.p, f1.p, knn, K, d32.p, band_ids.p, band_d.p,
             cap, dist_rel_team8(ld), state.p, 0, 0};
  const int grid = 8 * num_sms();
  auto on_band = [&](RepairState& h) {
    // the band list overflowed (many exact ties): exhaustive fp64 argmin instead
    if (!dv.p) dv.alloc((size_t)n, st);
    const unsigned long long init = ~0ull;
    const int imax = INT_MAX;
    SSG_CUDA(cudaMemcpyAsync(ull.p, &init, sizeof(init), cudaMemcpyHostToDevice, st));
    SSG_CUDA(cudaMemcpyAsync(&state.p->best, &imax, sizeof(int), cudaMemcpyHostToDevice, st));
    SSG_LAUNCH(k_repair_dist, grid, 256, 0, st, X, ld, d, n, bm.p, deg, R, (int64_t)h.u, dv.p, ull.p);
    SSG_LAUNCH(k_repair_pick_all, grid, 256, 0, st, dv.p, n, ull.p, &state.p->best);
    SSG_LAUNCH(k_add_edge, 1, 1, 0, st, adj, deg, R, &state.p->best, bm.p, f0.p, state.p);
    int best = 0;
    SSG_CUDA(cudaMemcpyAsync(&best, &state.p->best, sizeof(int), cudaMemcpyDeviceToHost, st));
    SSG_CUDA(cudaStreamSynchronize(st));
    if (best == INT_MAX) h.best = STOP_NONE;
  };
  std::vector<char> skip;
  for (int r = 0; r < n_nav; ++r) {
    if (r == 1) skip = roots_reach_first(a, nav_host, n_nav, st);
    if (r >= 1 && skip[(size_t)r]) continue;
    connect_root(a, nav_host[r], st, on_band);
  }
  RepairState h;
  SSG_CUDA(cudaMemcpyAsync(&h, state.p, sizeof(h), cudaMemcpyDeviceToHost, st));
  SSG_CUDA(cudaStreamSynchronize(st));
  if (knn_repairs) *knn_repairs = (int64_t)h.rep_knn;
  return (int64_t)(h.rep_full + h.rep_knn);
}

// ---------------------------------------------------------------------------------------
// Connectivity without device allocation (ssg_connect_noalloc).
//
// Some callers cannot allocate device memory while they run: serving loops that fix all
// their device memory before they take requests, or hosts that own a custom allocator and
// forbid the driver's.  For them the connectivity step also comes with its scratch in one
// fixed array that is part of the library's device image: the bitmap of reached nodes,
// two frontier buffers, the fp32 distance of every node and the short list of fp64
// re-tests, for graphs of up to NOALLOC_MAX_N nodes.  The same kernels run as in
// ssg_connect; only the scratch differs.  Like ssg_connect, the call reads the navigating
// ids and each repair's state back to the host, synchronising its stream each time.
// ---------------------------------------------------------------------------------------
namespace {
constexpr int64_t NOALLOC_MAX_N = 1 << 20;       // nodes
constexpr int NOALLOC_BAND = 1 << 14;            // fp64 re-tests per repair
constexpr size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t OFF_BM = 0;
constexpr size_t OFF_F0 = al256(OFF_BM + (size_t)(NOALLOC_MAX_N / 32) * 4);
constexpr size_t OFF_F1 = al256(OFF_F0 + (size_t)NOALLOC_MAX_N * 4);
constexpr size_t OFF_D32 = al256(OFF_F1 + (size_t)NOALLOC_MAX_N * 4);
constexpr size_t OFF_BAND_ID = al256(OFF_D32 + (size_t)NOALLOC_MAX_N * 4);
constexpr size_t OFF_BAND_D = al256(OFF_BAND_ID + (size_t)NOALLOC_BAND * 4);
constexpr size_t OFF_STATE = al256(OFF_BAND_D + (size_t)NOALLOC_BAND * 8);
constexpr size_t NOALLOC_BYTES = al256(OFF_STATE + sizeof(RepairState));
}  // namespace

// Held by every GPU that loads the library, until the process exits (about 12.3 MiB).
static __device__ __align__(256) unsigned char g_connect_scratch[NOALLOC_BYTES];

// Device address of g_connect_scratch on the current device, looked up once per device
// (host code cannot use the array's name as a device address).
static unsigned char* noalloc_scratch() {
  static std::mutex mu;
  static unsigned char* addr[64] = {};
  int dev = 0;
  SSG_CUDA(cudaGetDevice(&dev));
  SSG_REQUIRE(dev >= 0 && dev < 64, SSG_EINTERNAL, "device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    SSG_CUDA(cudaGetSymbolAddress(&p, g_connect_scratch));
    addr[dev] = (unsigned char*)p;
  }
  return addr[dev];
}

static int64_t connect_run_noalloc(const float* X, int ld, int d, int64_t n, int32_t* adj,
                                   int32_t* deg, int R, const int32_t* nav_host, int n_nav,
                                   cudaStream_t st) {
  unsigned char* base = noalloc_scratch();
  RepairState* S = (RepairState*)(base + OFF_STATE);
  SSG_CUDA(cudaMemsetAsync(S, 0, sizeof(RepairState), st));
  ConnArgs a{X, ld, d, n, ceil_div(n, 32), adj, deg, R, (uint32_t*)(base + OFF_BM),
             (int32_t*)(base + OFF_F0), (int32_t*)(base + OFF_F1), nullptr, 0,
             (float*)(base + OFF_D32), (int32_t*)(base + OFF_BAND_ID),
             (double*)(base + OFF_BAND_D), NOALLOC_BAND, dist_rel_team8(ld), S, 0, 0};
  auto on_band = [&](RepairState& h) {
    SSG_REQUIRE(false, SSG_EINTERNAL,
                "connectivity without allocation: more than %d nodes tie for the nearest "
                "reached node of node %lld; use ssg_connect",
                NOALLOC_BAND, (long long)h.u);
  };
  for (int r = 0; r < n_nav; ++r) connect_root(a, nav_host[r], st, on_band);
  RepairState h;
  SSG_CUDA(cudaMemcpyAsync(&h, S, sizeof(h), cudaMemcpyDeviceToHost, st));
  SSG_CUDA(cudaStreamSynchronize(st));
  return (int64_t)(h.rep_full + h.rep_knn);
}

}  // namespace ssg

extern "C" ssg_status ssg_connect_noalloc(const float* base, int64_t n, int32_t d, int32_t* adj,
                                          int32_t* deg, int32_t R, const int32_t* nav,
                                          int32_t n_nav, int64_t* n_repair_host,
                                          ssg_stream stream) {
  using namespace ssg;
  try {
    SSG_REQUIRE(base && adj && deg && nav, SSG_EINVAL, "null pointer");
    SSG_REQUIRE(n >= 1 && n <= NOALLOC_MAX_N, SSG_EINVAL,
                "connectivity without allocation handles 1 <= n <= %lld nodes, got %lld",
                (long long)NOALLOC_MAX_N, (long long)n);
    SSG_REQUIRE(d >= 1 && d % 4 == 0 && ((uintptr_t)base & 15) == 0, SSG_EINVAL,
                "connectivity without allocation needs d %% 4 == 0 and a 16-byte aligned base "
                "(no padded copy is made), got d = %d",
                d);
    SSG_REQUIRE(R >= 1 && n_nav >= 1, SSG_EINVAL, "need R >= 1 and n_nav >= 1");
    cudaStream_t st = (cudaStream_t)stream;
    // every navigating id is checked before the graph is touched (host memory only)
    std::vector<int32_t> h((size_t)n_nav);
    SSG_CUDA(cudaMemcpyAsync(h.data(), nav, sizeof(int32_t) * n_nav, cudaMemcpyDeviceToHost, st));
    SSG_CUDA(cudaStreamSynchronize(st));
    for (int t = 0; t < n_nav; ++t)
      SSG_REQUIRE(h[t] >= 0 && h[t] < n, SSG_EINVAL, "navigating node id %d out of range", h[t]);
    const int64_t rep = connect_run_noalloc(base, d, d, n, adj, deg, R, h.data(), n_nav, st);
    if (n_repair_host) *n_repair_host = rep;
    return SSG_OK;
  } catch (const Fail& e) {
    return e.st;
  } catch (const std::bad_alloc&) {
    set_error("host allocation failed");
    return SSG_ENOMEM;
  } catch (...) {
    set_error("unexpected exception");
    return SSG_EINTERNAL;
  }
}
