// kNN graph selection on the 5th-generation tensor cores (tcgen05, sm_103a): every row's KS
// nearest columns by the distance of bf16 operands.  Exact for integer data that bf16 holds
// exactly (|x| <= 256, and the bounds of DataInfo::exact); on other data the caller certifies
// the result (knn_cert.cu).
//
// The GEMM is augmented so that the accumulator already holds what the threshold test
// needs: A = [x | 1 1 1 1 0..], B = [y | -p1 -p2 -p3 -p4 0..] with p1 + .. + p4 = |y|^2 / 2
// (bf16 parts of an integer or half-integer below 2^23), so acc = x.y - |y|^2 / 2 and
// d2 = |x|^2 - 2 acc.  On exact data every product and partial sum is a multiple of 1/2 below
// 2^23 in magnitude (2 d max|x|^2 <= 2^24 for non-negative data, 4 d max|x|^2 <= 2^24
// otherwise), so the accumulation is exact in fp32 whatever its order, and so is d2.
//
// k_knn_pair: persistent clusters of two CTAs (one CTA per SM), 10 warps each.  A work item is
// a block of 512 query rows, 256 per CTA, and one of `nseg` interleaved shares of the column
// tiles it visits (256 columns, 128 rows of B in each CTA).
//   warp 0      TMA producer: the CTA's query rows (A; resident for rows of up to 128 values,
//               else streamed with B in 64-value chunks) and its half of the column tiles,
//               bf16 with 128-byte swizzle, plus the 16-element augmentation rows with 32-byte
//               swizzle.  All of them complete on the leader CTA's barriers;
//   warp 1      allocates 512 TMEM columns; the leader's issues tcgen05.mma of the pair: M =
//               256 (128 rows of each CTA), N = 128 (streamed: 256), into four accumulators of
//               128 columns: two column halves for each of the two 128-row halves of a CTA's
//               rows, so the epilogue drains some while the MMAs fill others;
//   warps 2..9  epilogue, one thread per query row (TMEM lane): tcgen05.ld 64 columns at a
//               time, their largest accumulator against the row's threshold (a tree of
//               three-input maxes), and only where some lane passes, the passing (id,
//               accumulator) pairs go straight from registers to the row's buffer in global
//               scratch; a warp cuts a full buffer back to its KS largest with a bisection.
// k_knn_finish then takes each row's KS largest from the buffers of its shares, sorts them by
// (distance, original id) and writes the K neighbours, with many rows per SM in flight.
//
// Why this shape.  A pair reads half of B per CTA for an MMA of four times the work of one
// CTA's 128 x 128, and each column tile is read from L2 once for 512 rows instead of 256 (773
// GB of DRAM reads for a graph of 1M x 128 before).  The epilogue holds an accumulator for two
// TMEM loads of 64 columns, about 900 cycles with the handoff, against the 2,300 the four take
// to fill at d = 128 (two accumulators of 256 columns, held for four loads, were the bound:
// 1M x 128, K = 200, 249 -> 223 ms).  Appending from registers needs no stash in shared memory
// (its scan cost about 250 cycles per chunk).  Few row blocks (10,000 queries, a sample of 256
// rows) used to leave most SMs idle: their columns are shared out over `nseg` items per block,
// and the shares exchange thresholds through global memory.  What bounds it now: the epilogue
// of the tiles in which rows still append (a warp's chunk with appends takes 500-1,800 cycles,
// a cut of a row's buffer 3,000-5,000), then the MMAs.
// Measured, whole kNN stage, against the kernel of one CTA and 128 x 128 MMAs: 1M x 128,
// K = 200, 341 -> 223 ms; 10,000 queries over 1M rows, K = 100, 15.0 -> 6.0 ms.
//
// Columns are visited in 256-wide tiles, in id order or (large self-joins) nearest cluster
// first; ties at the threshold are admitted and settled by original id at the end.
// Every wait on an mbarrier is bounded (about 2 s); a wait that runs out sets an error
// word, tells the other roles to stop, and the CTA releases its TMEM and exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <type_traits>

#include "common.cuh"
#include "knn.cuh"
#include "knn_select.cuh"
#include "tc_common.cuh"

namespace ssg {
namespace {

using namespace tc;

constexpr int BM = 512;               // query rows per work item (256 per CTA of the pair)
constexpr int CM = 256;               // query rows per CTA: two halves of 128 TMEM lanes
constexpr int BN = 256;               // base columns per tile (UMMA_N), 128 rows of B per CTA
constexpr int API_TILE = 128;         // tile limits are given in 128-point tiles
constexpr uint32_t IDESC = idesc_bf16_pair(BN), IDESC_HALF = idesc_bf16_pair(BN / 2);
constexpr int NBUF = 4;               // TMEM accumulators of 128 columns: two per half of the rows
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 64 + EPI_WARPS * 32;
constexpr int TMEM_COLS = 512;        // NBUF x 128 fp32 columns
constexpr int MAX_STAGES = 6;
constexpr int MAX_D_RESIDENT = 128;   // rows of up to this many values stay resident
constexpr int MAX_D_STREAM = 4096;    // longer ones, up to this, are streamed
constexpr int AUG = 16;               // augmentation K-step (bf16 elements)
constexpr int AUG_BYTES = AUG * 2;    // one augmentation row: 32 bytes
constexpr float LOWEST = -3.402823466e38f;  // the threshold that every finite value meets
constexpr uint32_t A_CHUNK = CM * 128;        // 64 values of the CTA's query rows: 32 KB
constexpr uint32_t B_CHUNK = (BN / 2) * 128;  // 64 values of its half of a tile: 16 KB
constexpr uint32_t A_AUG = 128 * AUG_BYTES;   // one half's rows (all halves' rows are alike)
constexpr uint32_t B_AUG = (BN / 2) * AUG_BYTES;

struct TcArgs {
  int64_t na;           // query rows
  int64_t nb;           // base rows: stored column positions >= nb are padding
  int64_t rb0, nrb;     // row blocks of this launch: rb0 .. rb0 + nrb - 1
  int64_t tstride;      // length of each cluster's tile list
  int64_t nwalk;        // tiles each block of rows visits (all, or fewer for Alg. 4)
  int nseg;             // shares of a block's tiles
  int kchunks;          // row width / 64
  int dp_chunks, d;     // chunks of one part of a row (bf16 pairs: three parts), its values
  int stages;
  int KS;
  uint2* rowbuf;        // [rows of this launch][nseg][C] (id, accumulator bits)
  int* cnt;             // [rows of this launch][nseg]
  uint32_t* ts_g;       // nullable, per query row: order bits of a lower bound of its KS-th
                        // largest accumulator (read first; with shares, raised by all)
  int* err;
  const int32_t* perm;        // stored position -> original id (null: the identity)
  const int32_t* tile_order;  // tile lists, tstride entries apart (null: in order)
  const int32_t* rb_cluster;  // list of each block of BM stored query rows (null: its own)
  // limited walks: block rb0 + i has the i-th list, of walk_len[i] entries tile << 8 | mask, bit
  // 4 r + 2 h + c: rows 128 h .. of CTA r visit the tile's columns 128 c ..
  const int32_t* walk_len;
};

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Largest of eight values.
__device__ __forceinline__ float max8(const uint32_t* v) {
  const float a = fmax3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
  const float b = fmax3(__uint_as_float(v[3]), __uint_as_float(v[4]), __uint_as_float(v[5]));
  return fmax3(a, b, fmaxf(__uint_as_float(v[6]), __uint_as_float(v[7])));
}

// The order keys of one row's values (ascending: larger accumulators first; absent ones
// 0xFFFFFFFF) are spread over the warp, E per lane.  Finds hi such that between KS and `good`
// keys are at most hi (more only where ties at the KS-th force it) by a search over the bits,
// three pivots a step; lo .. hi: the present keys' range, n: their number, at least KS.
// Returns the number of keys at most hi.
template <int E>
__device__ __forceinline__ int search_keys(const uint32_t (&k)[E], int KS, int good, uint32_t lo,
                                           uint32_t& hi, int n) {
  while (lo < hi) {
    const uint32_t q = (hi - lo) >> 2;
    const uint32_t m1 = lo + q, m2 = lo + ((hi - lo) >> 1), m3 = m2 + q;
    uint32_t c12[4] = {0u, 0u, 0u, 0u}, c3[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int e = 0; e < E; ++e) {
      c12[e & 3] += (k[e] <= m1 ? 1u : 0u) + (k[e] <= m2 ? 0x10000u : 0u);
      c3[e & 3] += k[e] <= m3 ? 1u : 0u;
    }
    const uint32_t a12 = __reduce_add_sync(0xffffffffu, (c12[0] + c12[1]) + (c12[2] + c12[3]));
    const int a3 = (int)__reduce_add_sync(0xffffffffu, (c3[0] + c3[1]) + (c3[2] + c3[3]));
    const int a1 = (int)(a12 & 0xffffu), a2 = (int)(a12 >> 16);
    if (a1 >= KS) {
      hi = m1;
      n = a1;
    } else if (a2 >= KS) {
      lo = m1 + 1;
      hi = m2;
      n = a2;
    } else if (a3 >= KS) {
      lo = m2 + 1;
      hi = m3;
      n = a3;
    } else {
      lo = m3 + 1;
      continue;
    }
    if (n <= good) break;
  }
  return n;
}

// Of the keys equal to hi, the largest original id such that `want` of them have an id up to
// it; id(e): the original id of key e.
template <int E, class Id>
__device__ __forceinline__ uint32_t tie_bound(const uint32_t (&k)[E], uint32_t hi, int KS, Id id) {
  int below = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) below += k[e] < hi ? 1 : 0;
  const int want = KS - __reduce_add_sync(0xffffffffu, below);
  uint32_t l2 = 0u, h2 = 0x7FFFFFFFu;
  while (l2 < h2) {
    const uint32_t mid = l2 + ((h2 - l2) >> 1);
    int c = 0;
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (k[e] == hi) c += id(e) <= mid ? 1 : 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if (c >= want)
      h2 = mid;
    else
      l2 = mid + 1;
  }
  return h2;
}

// Cuts the buffers of the warp's rows named by `need` (lane l's has mycnt of lane l, more than
// KS, (id, accumulator) pairs) back to the entries at or above a threshold with between KS and
// `good` of them; if ties at the KS-th largest would keep more than `cap`, exactly KS stay, the
// ties with the smallest original ids.  Returns (new count, threshold bits) of this lane's
// row: at least KS entries are not below the threshold.  Out of line: it runs rarely, and one
// copy keeps the scan small in the instruction cache.
template <int C>
__device__ __noinline__ uint2 cut_rows(uint2* __restrict__ wbuf, uint32_t lstride, unsigned need,
                                       int mycnt, int KS, int good, int cap,
                                       const int32_t* __restrict__ perm) {
  constexpr int E = C / 32;
  const int lane = lane_id();
  const unsigned lt = lanemask_lt();
  uint2 mine = make_uint2((uint32_t)mycnt, 0u);
  while (need) {
    const int l = __ffs(need) - 1;
    need &= need - 1;
    const int cnt = __shfl_sync(0xffffffffu, mycnt, l);
    uint2* buf = wbuf + (size_t)l * lstride;
    uint2 v[E];
#pragma unroll
    for (int e = 0; e < E; ++e)
      v[e] = ((e << 5) | lane) < cnt ? buf[(e << 5) | lane] : make_uint2(0u, 0u);
    uint32_t k[E];
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const bool in = ((e << 5) | lane) < cnt;
      k[e] = in ? ~float_order_bits(__uint_as_float(v[e].y)) : 0xFFFFFFFFu;
      lo = min(lo, k[e]);
      hi = max(hi, in ? k[e] : 0u);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    const int n = search_keys<E>(k, KS, good, lo, hi, cnt);
    auto orig = [&](int e) { return perm ? (uint32_t)perm[v[e].x] : v[e].x; };
    uint32_t idmax = 0xFFFFFFFFu;  // of the entries equal to hi, those with an id up to this stay
    if (n > cap) idmax = tie_bound<E>(k, hi, KS, orig);
    unsigned b[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      bool in = k[e] <= hi;
      if (idmax != 0xFFFFFFFFu && in && k[e] == hi) in = orig(e) <= idmax;
      b[e] = __ballot_sync(0xffffffffu, in);
    }
    int base = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if ((b[e] >> lane) & 1u) buf[base + __popc(b[e] & lt)] = v[e];
      base += __popc(b[e]);
    }
    if (lane == l) mine = make_uint2((uint32_t)base, __float_as_uint(order_bits_float(~hi)));
  }
  __syncwarp();
  return mine;
}

// LIMITED: a walk over part of the tiles, with masked list entries (TcArgs::walk_len).  A kernel of
// its own: the mask's test in the one for full walks cost 258 -> 270 ms for a build of 1M x 128.
template <int C, bool STREAM, bool LIMITED>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
k_knn_pair(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
           const __grid_constant__ CUtensorMap tmAaug, const __grid_constant__ CUtensorMap tmBaug,
           TcArgs p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int S = p.stages;
  // a stage: the tile's B rows, whole (resident A), or one chunk of A and of B; then the
  // tile's augmentation rows (streamed: with the last chunk)
  const int cps = STREAM ? 1 : p.kchunks;            // chunks per stage
  const int spt = STREAM ? p.kchunks : 1;            // stages per tile
  const uint32_t b_off = STREAM ? A_CHUNK : 0;
  const uint32_t g_off = b_off + (uint32_t)cps * B_CHUNK;
  const uint32_t stage_bytes = g_off + B_AUG;
  const uint32_t a_bytes = STREAM ? 0u : (uint32_t)p.kchunks * A_CHUNK;
  unsigned char* sA = sm;
  unsigned char* sG = sA + a_bytes;                  // A's augmentation rows
  unsigned char* sS = sG + A_AUG;
  uint64_t* bars = (uint64_t*)(sS + (size_t)S * stage_bytes);
  uint64_t* a_full = bars;                           // leader's
  uint64_t* a_empty = bars + 1;                      // both
  uint64_t* s_full = bars + 2;                       // leader's
  uint64_t* s_empty = s_full + MAX_STAGES;           // both
  uint64_t* t_full = s_empty + MAX_STAGES;           // both, per accumulator (2 half + column half)
  uint64_t* t_empty = t_full + NBUF;                 // leader's, per accumulator
  uint32_t* tmem_slot = (uint32_t*)(t_empty + NBUF);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t rank = cluster_rank();
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(a_full), 1);
    mbar_init(smem_u32(a_empty), STREAM ? 1 : 2);   // once both halves are done with the rows
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(s_full + s), 1);
      mbar_init(smem_u32(s_empty + s), 2);            // both halves
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(smem_u32(t_full + b), 1);
      mbar_init(smem_u32(t_empty + b), EPI_WARPS);   // four warps of each CTA
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int nseg = p.nseg;
  const int64_t nitems = p.nrb * nseg;
  const int64_t ncl = gridDim.x >> 1, cl = blockIdx.x >> 1;
  // item i: row block rb0 + i / nseg, tiles i % nseg, i % nseg + nseg, ...
  auto tiles_of = [&](int64_t rb) -> const int32_t* {
    if (LIMITED) return p.tile_order + (rb - p.rb0) * p.tstride;
    return p.tile_order
               ? p.tile_order + (p.rb_cluster ? (int64_t)p.rb_cluster[rb] : rb) * p.tstride
               : nullptr;
  };
  auto walk_of = [&](int64_t rb) -> int64_t {
    if (LIMITED) return (int64_t)p.walk_len[rb - p.rb0];
    // a full walk has no lengths; with p.nwalk alone the compiler lays this kernel out slower (145
    // registers for 143; kNN stage of 1M x 128 224.7 ms, so 223.6; of 60,000 x 128 4.09 and 4.05)
    return p.walk_len ? (int64_t)p.walk_len[rb] : p.nwalk;
  };
  constexpr int MASK_BITS = LIMITED ? 8 : 0;  // of a list entry

  if (warp == 0) {
    // ---------------- TMA producer (of each CTA) ----------------
    if (lane == 0) {
      int s = 0;         // next stage
      uint32_t ph = 0;   // and the parity of its use
      uint32_t aph = 1;
      bool ok = true;
      const uint32_t a_bar = map_to_rank(smem_u32(a_full), 0);
      bool first = true;
      for (int64_t it = cl; it < nitems && ok; it += ncl) {
        const int64_t rb = p.rb0 + it / nseg;
        const int seg = (int)(it % nseg);
        const int row0 = (int)(rb * BM + rank * CM);
        if (!STREAM || first) {
          // the query rows (resident), and once the augmentation rows
          ok = mbar_wait(smem_u32(a_empty), aph, abort_flag);
          if (!ok) break;
          aph ^= 1;
          if (rank == 0)
            mbar_expect_tx(smem_u32(a_full), 2 * (a_bytes + (first ? A_AUG : 0u)));
          if (!STREAM)
            for (int kc = 0; kc < p.kchunks; ++kc)
              tma_load_2d_pair(smem_u32(sA + (size_t)kc * A_CHUNK), &tmA, a_bar, kc * 64, row0);
          if (first) tma_load_2d_pair(smem_u32(sG), &tmAaug, a_bar, 0, 0);
          first = false;
        }
        const int32_t* tl = tiles_of(rb);
        const int64_t nwalk = walk_of(rb);
        int64_t tn = tl ? tl[seg] : seg;  // tile index, read one tile ahead
        for (int64_t i = seg; i < nwalk && ok; i += nseg) {
          const int j0 = (int)((tn >> MASK_BITS) * BN + rank * (BN / 2));
          if (i + nseg < nwalk) tn = tl ? tl[i + nseg] : i + nseg;
          for (int kc = 0; kc < spt; ++kc) {
            ok = mbar_wait(smem_u32(s_empty + s), ph ^ 1, abort_flag);
            if (!ok) break;
            const bool last = kc == spt - 1;
            const uint32_t bar = map_to_rank(smem_u32(s_full + s), 0);
            if (rank == 0) mbar_expect_tx(smem_u32(s_full + s), 2 * (g_off + (last ? B_AUG : 0u)));
            unsigned char* dst = sS + (size_t)s * stage_bytes;
            if (STREAM) tma_load_2d_pair(smem_u32(dst), &tmA, bar, kc * 64, row0);
            for (int c = 0; c < cps; ++c)
              tma_load_2d_pair(smem_u32(dst + b_off + (size_t)c * B_CHUNK), &tmB, bar,
                               (STREAM ? kc : c) * 64, j0);
            if (last) tma_load_2d_pair(smem_u32(dst + g_off), &tmBaug, bar, 0, j0);
            if (++s == S) {
              s = 0;
              ph ^= 1;
            }
          }
        }
      }
      // every commit on this CTA's barriers has arrived before the CTA can end
      for (int k = 0; k < S && ok; ++k) {
        ok = mbar_wait(smem_u32(s_empty + s), ph ^ 1, abort_flag);
        if (++s == S) {
          s = 0;
          ph ^= 1;
        }
      }
      if (!STREAM && ok) ok = mbar_wait(smem_u32(a_empty), aph, abort_flag);
      if (!ok) {
        atomicOr(p.err, 1 << 1);
        *abort_flag = 1;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (the leader's) ----------------
    // The whole warp runs the loop and one lane issues, so that the descriptors stay in
    // uniform registers: issued from a single-lane branch each MMA cost about 200 cycles of
    // moves and 64-bit adds, more than the 128 the tensor cores need for it (1M x 128, MMAs
    // and copies alone: 205 -> 115 ms).
    // The two halves run ahead of each other by up to the pipeline's stages: whichever half's
    // accumulator is free gets its next stage, so that a half whose epilogue is held up by an
    // append or a cut does not hold up the other (200,000 x 128, K = 200: 24.2 -> 22.2 ms with
    // closer thresholds from the cuts).
    if (rank == 0) {
      struct Half {
        int64_t it, i;   // item and tile
        int64_t nwalk;   // tiles of the item's block
        int seg, sub, s; // share, step within the tile, pipeline slot
        uint32_t ph, aph, tph;
        bool fresh;      // the item's first step: its rows may not have landed
        int64_t done;    // steps issued
      };
      Half hf[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        hf[h].it = cl;
        hf[h].seg = (int)(cl % nseg);
        hf[h].i = hf[h].seg;
        hf[h].nwalk = walk_of(p.rb0 + cl / nseg);
        hf[h].sub = hf[h].s = 0;
        hf[h].ph = hf[h].aph = 0u;
        hf[h].tph = 1u;
        hf[h].fresh = true;
        hf[h].done = 0;
      }
      bool ok = true;
      const bool issue = elect_one();
      const uint64_t aug_a = sdesc_sw32(smem_u32(sG));
      const uint32_t st0 = smem_u32(sS);
      const uint64_t a_desc = sdesc_sw128(STREAM ? st0 : smem_u32(sA));
      const uint64_t b_desc = sdesc_sw128(st0 + b_off);
      const uint64_t g_desc = sdesc_sw32(st0 + g_off);
      // The next step of half h, if its barriers allow it.  Resident rows: a step is one column
      // half of a tile (all its K-steps, an N = 128 MMA each); streamed rows: one 64-value chunk
      // of both column halves (N = 256).
      const int nsub = STREAM ? spt : 2;
      auto advance = [&](Half& u, int h) -> bool {
        if (u.it >= nitems) return false;
        bool ready = mbar_test(smem_u32(s_full + u.s), u.ph);
        if (!STREAM) ready = ready && mbar_test_cluster(smem_u32(t_empty + 2 * h + u.sub), u.tph);
        if (STREAM && u.sub == 0)
          ready = ready && mbar_test_cluster(smem_u32(t_empty + 2 * h), u.tph) &&
                  mbar_test_cluster(smem_u32(t_empty + 2 * h + 1), u.tph);
        if (u.fresh) ready = ready && mbar_test(smem_u32(a_full), u.aph);
        if (!__all_sync(0xffffffffu, ready)) return false;
        tc_fence_after();
        // descriptors: the 14-bit start-address field (bytes / 16) plus an offset; shared
        // addresses stay below 256 KB, so the sum never carries out of the field
        const uint64_t so = (uint64_t)(((uint32_t)u.s * stage_bytes) >> 4);
        const bool last = u.sub == nsub - 1;
        const uint32_t d_tmem = tmem_base + (uint32_t)(h * BN + (STREAM ? 0 : u.sub * (BN / 2)));
        const uint64_t ad = a_desc + (STREAM ? so : 0ull) + (uint64_t)((h * 128 * 128) >> 4);
        // column half u.sub: B's rows 64 u.sub .. + 63 of each CTA
        const uint64_t bd = b_desc + so + (STREAM ? 0ull : (uint64_t)(u.sub * ((64 * 128) >> 4)));
        const uint64_t gd = g_desc + so + (STREAM ? 0ull : (uint64_t)(u.sub * ((64 * AUG_BYTES) >> 4)));
        const bool item_end = last && u.i + nseg >= u.nwalk;
        if (issue) {
#pragma unroll
          for (int c = 0; c < (STREAM ? 1 : MAX_D_RESIDENT / 64); ++c) {
            // K-steps of this chunk that hold values (the rest are zero padding)
            const int left = STREAM ? p.d - (u.sub % p.dp_chunks) * 64 : p.d - c * 64;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (kk * 16 < left)
                umma_bf16_pair(d_tmem, ad + (uint64_t)((c * A_CHUNK + kk * 32) >> 4),
                               bd + (uint64_t)((c * B_CHUNK + kk * 32) >> 4),
                               STREAM ? IDESC : IDESC_HALF,
                               STREAM ? (uint32_t)(u.sub | kk) : (uint32_t)(c | kk));
          }
          if (!STREAM || last) {
            umma_bf16_pair(d_tmem, aug_a, gd, STREAM ? IDESC : IDESC_HALF, 1u);
            umma_commit_pair(smem_u32(t_full + 2 * h + (STREAM ? 0 : u.sub)));
            if (STREAM) umma_commit_pair(smem_u32(t_full + 2 * h + 1));
          }
          if (STREAM || last) umma_commit_pair(smem_u32(s_empty + u.s));
          if (!STREAM && item_end) umma_commit_pair(smem_u32(a_empty));
        }
        __syncwarp();
        ++u.done;
        u.fresh = false;
        if (STREAM || last) {
          if (++u.s == S) {
            u.s = 0;
            u.ph ^= 1u;
          }
        }
        if (!last) {
          ++u.sub;
        } else {
          u.sub = 0;
          u.tph ^= 1u;
          u.i += nseg;
          if (item_end) {
            u.it += ncl;
            if (u.it < nitems) u.nwalk = walk_of(p.rb0 + u.it / nseg);
            u.seg = (int)(u.it % nseg);
            u.i = u.seg;
            if (!STREAM) {
              u.fresh = true;
              u.aph ^= 1u;
            }
          }
        }
        return true;
      };
      uint64_t idle_since = 0;
      while (hf[0].it < nitems || hf[1].it < nitems) {
        // the half that is behind goes first
        bool any;
        if (hf[1].done < hf[0].done)
          any = advance(hf[1], 1) || advance(hf[0], 0);
        else
          any = advance(hf[0], 0) || advance(hf[1], 1);
        if (any) {
          idle_since = 0;
        } else {
          const uint64_t now = global_ns();
          if (idle_since == 0) idle_since = now;
          ok = !*abort_flag && now - idle_since <= WAIT_NS;
          if (!__all_sync(0xffffffffu, ok)) {
            ok = false;
            break;
          }
        }
      }
      if (!ok && lane == 0) {
        atomicOr(p.err, 1 << 2);
        *abort_flag = 1;
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: one thread per query row ----------------
    const int ew = warp - 2;
    const int h = ew >> 2;          // which 128-row half
    const int q = warp & 3;         // TMEM lane quadrant this warp may access
    const int row_in_cta = h * 128 + q * 32 + lane;
    const uint32_t my_empty = map_to_rank(smem_u32(t_empty + 2 * h), 0);
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * BN);
    const float INF = __int_as_float(0x7f800000);
    // a row is cut once it holds more than trig entries (a chunk pair adds up to 64), back to
    // `good` at most: a threshold close to the KS-th largest costs a few more search steps per
    // cut and saves appends and cuts
    const int trig = min(C - 64, max(3 * p.KS, p.KS + 64));
    const int good = p.KS + (trig - p.KS) / 8;
    uint32_t tph = 0;
    bool ok = true;
    for (int64_t it = cl; it < nitems && ok; it += ncl) {
      const int64_t rbl = it / nseg;
      const int seg = (int)(it % nseg);
      const int64_t lrow = rbl * BM + rank * CM + row_in_cta;   // row of this launch
      const int64_t row = p.rb0 * BM + lrow;
      uint2* wbuf = p.rowbuf + ((lrow - lane) * nseg + seg) * C;  // lane 0's buffer
      const uint32_t lstride = (uint32_t)nseg * C;                // entries between lanes' buffers
      const uint32_t off0 = lane * lstride;
      uint32_t off = off0;                                        // next free entry, from wbuf
      // a column is admitted from this accumulator on; padding rows admit nothing
      float ts = row < p.na ? LOWEST : INF;
      if (p.ts_g && row < p.na) ts = order_bits_float(__ldcg(p.ts_g + row));
      const int32_t* tl = tiles_of(p.rb0 + rbl);
      const int64_t nwalk = walk_of(p.rb0 + rbl);
      int64_t tn = tl ? tl[seg] : seg;
      // the row's new count and threshold
      auto settle = [&](uint2 r) {
        off = off0 + r.x;
        float t2 = __uint_as_float(r.y);
        if (nseg > 1) {
          const uint32_t b = float_order_bits(t2);
          t2 = order_bits_float(max(b, atomicMax(p.ts_g + row, b)));
        }
        ts = fmaxf(ts, t2);
      };
      for (int64_t i = seg; i < nwalk; i += nseg) {
        const int32_t j0 = (int32_t)((tn >> MASK_BITS) * BN);
        // columns that these rows do not visit (bit c: the half c)
        const uint32_t skip = LIMITED ? ~((uint32_t)tn >> (4 * rank + 2 * h)) & 3u : 0u;
        if (i + nseg < nwalk) tn = tl ? tl[i + nseg] : i + nseg;
        // with shares: the other shares' thresholds, read while the tile is computed
        uint32_t other = 0u;
        if (nseg > 1 && row < p.na) other = __ldcg(p.ts_g + row);
        // the tile's two column halves, an accumulator each, in 64-column chunks: chunk c & 1 of
        // half c >> 1
        uint32_t v[2][32];
#pragma unroll 1
        for (int c = 0; c < BN / 64; ++c) {
          if (!(c & 1)) {
            ok = mbar_wait(smem_u32(t_full + 2 * h + (c >> 1)), tph, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (c == 0 && nseg > 1 && row < p.na) ts = fmaxf(ts, order_bits_float(other));
          }
          tmem_ld32(taddr + (uint32_t)c * 64, v[0]);
          tmem_ld32(taddr + (uint32_t)c * 64 + 32, v[1]);
          tmem_wait_ld(v[0]);
          tmem_dep(v[1]);
          if (c & 1) {
            // every lane's loads are complete (tmem_wait_ld) and fenced before the warp's barrier,
            // behind which lane 0 arrives for all of them.  A second fence behind the barrier could
            // only order lane 0's own loads once more (1M x 128 223.6 ms, without it 222.1).
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(my_empty + (c >> 1) * (uint32_t)sizeof(uint64_t));
          }
          if (LIMITED && ((skip >> (STREAM ? c >> 1 : c & 1)) & 1u)) continue;
          // resident rows: a column half is 64 columns of each CTA's 128
          const int32_t jc = j0 + (STREAM ? c * 64 : (c >> 1) * 64 + (c & 1) * (BN / 2));
          if (jc + 64 > p.nb) {  // the last tile's padding columns are never admitted
#pragma unroll
            for (int e = 0; e < 64; ++e)
              if (jc + e >= p.nb) v[e >> 5][e & 31] = 0x7fffffffu;  // NaN: no comparison holds
          }
          float m8[8];
#pragma unroll
          for (int g = 0; g < 8; ++g) m8[g] = max8(&v[g >> 2][(g & 3) * 8]);
          const float m = fmax3(fmax3(m8[0], m8[1], m8[2]), fmax3(m8[3], m8[4], m8[5]),
                                fmaxf(m8[6], m8[7]));
          if (!__any_sync(0xffffffffu, m >= ts)) continue;
          uint32_t pm = 0u;  // this lane's groups of eight columns with one to append
#pragma unroll
          for (int g = 0; g < 8; ++g) pm |= m8[g] >= ts ? 1u << g : 0u;
          if (__reduce_max_sync(0xffffffffu, (unsigned)__popc(pm)) <= 3u) {
            // Few per lane (the usual case once the threshold has settled): each lane takes its
            // own groups one by one, their values picked by selects on the group's bits.  Walking
            // every group that some lane passes (below) costs a vote, a branch and eight
            // dependent appends for each.
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              uint32_t pq = (pm >> (4 * hh)) & 15u;
              while (__any_sync(0xffffffffu, pq != 0u)) {
                const int g = pq ? __ffs(pq) - 1 : 0;
                const bool g1 = g & 2, g0 = g & 1;
                const float lim = pq != 0u ? ts : __int_as_float(0x7fffffff);  // NaN: through
                const int32_t jg = jc + hh * 32 + g * 8;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                  const uint32_t a = g1 ? v[hh][16 + e] : v[hh][e];
                  const uint32_t b = g1 ? v[hh][24 + e] : v[hh][8 + e];
                  const uint32_t x = g0 ? b : a;
                  if (__uint_as_float(x) >= lim) {
                    wbuf[off] = make_uint2((uint32_t)(jg + e), x);
                    ++off;
                  }
                }
                pq &= pq - 1u;
              }
            }
          } else {
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              if (__any_sync(0xffffffffu, m8[g] >= ts)) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                  const uint32_t a = v[g >> 2][(g & 3) * 8 + e];
                  if (__uint_as_float(a) >= ts) {
                    wbuf[off] = make_uint2((uint32_t)(jc + g * 8 + e), a);
                    ++off;
                  }
                }
              }
            }
          }
          // buffers that the next 64 columns could overflow drop to the entries at or above
          // their KS-th largest accumulator
          __syncwarp();
          const unsigned need = __ballot_sync(0xffffffffu, off - off0 > (uint32_t)trig);
          if (need) {
            const uint2 r = cut_rows<C>(wbuf, lstride, need, (int)(off - off0), p.KS, good, trig, p.perm);
            if ((need >> lane) & 1u) settle(r);
          }
        }
        if (!ok) break;
        tph ^= 1;
      }
      if (!ok) break;
      p.cnt[lrow * nseg + seg] = (int)(off - off0);
    }
    if (!ok && lane == 0) {
      atomicOr(p.err, 1 << 3);
      *abort_flag = 1;
    }
  }
  __syncwarp();
  if (*abort_flag) {
    // a role gave up: let the copies already in flight land before the CTA can go
    const uint64_t t0 = global_ns();
    while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
  cluster_sync();
}

// ---------------------------------------------------------------------------------------
// The end of each row: its KS largest accumulators among the buffers of its shares, sorted by
// (distance, original id).  One warp per row.
// ---------------------------------------------------------------------------------------
struct FinArgs {
  const int* err;             // a walk that gave up leaves no counts to read
  const uint2* rowbuf;
  const int* cnt;
  int nseg, C, KS, K, self;
  int64_t row0, rows;         // query rows row0 .. row0 + rows - 1 of this launch
  const float* a_norm;        // |x|^2 of the stored query rows
  const int32_t* perm;
  const int32_t* qid;         // nullable: query row r is base row qid[r] (the self column);
                              // outputs then go to row r
  const float* tau_in;        // nullable: the admission bound a row started from
  int32_t* out_id;
  float* out_d2;
  float* out_thresh;          // nullable: per output row, the KS-th smallest distance kept (or,
                              // with fewer kept, the final admission bound)
  uint32_t* ts_out;           // nullable: only the order bits of the KS-th largest accumulator
  int sorted;                 // 0: the K neighbours in any order (for a caller that reorders them)
  int slots;                  // keys per warp: a power of two, at least KS
  int tcap;                   // entries of all shares at most
};

// Sorts n <= 32 E keys and writes the row: the first K after dropping the row itself.
template <int E>
__device__ __noinline__ void sort_out(const FinArgs& p, const uint64_t* keys, int n, int64_t row) {
  const int lane = lane_id();
  const float INF = __int_as_float(0x7f800000);
  uint64_t v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = e * 32 + lane < n ? keys[e * 32 + lane] : KEY_NONE;
  warp_sort_regs<E * 32>(v);
  const int c2 = n < p.KS ? n : p.KS;
  const int64_t ro = p.qid ? row : (p.perm ? (int64_t)p.perm[row] : row);
  const int32_t sid = p.qid ? p.qid[row] : (int32_t)ro;
  int selfpos = c2;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int t = e * 32 + lane;
    if (p.self) {
      const unsigned m = __ballot_sync(0xffffffffu, t < c2 && key_id(v[e]) == sid);
      if (m && selfpos == c2) selfpos = e * 32 + __ffs(m) - 1;
    }
    if (p.out_thresh && t == p.KS - 1 && t < c2) p.out_thresh[ro] = key_dist(v[e]);
  }
  if (p.out_thresh && c2 < p.KS && lane == 0) p.out_thresh[ro] = p.tau_in ? p.tau_in[row] : INF;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int t = e * 32 + lane;
    const int o = t < selfpos ? t : t - 1;
    if (t < c2 && t != selfpos && o < p.K) {
      p.out_id[ro * p.K + o] = key_id(v[e]);
      p.out_d2[ro * p.K + o] = key_dist(v[e]);
    }
  }
  const int got = selfpos < c2 ? c2 - 1 : c2;
  for (int t = got + lane; t < p.K; t += 32) {
    p.out_id[ro * p.K + t] = -1;
    p.out_d2[ro * p.K + t] = INF;
  }
}

// The same without the sort: the n <= KS keys that stay, in any order, less the row itself (or,
// where it is not among KS of them, the last in order).
__device__ __forceinline__ void raw_out(const FinArgs& p, const uint64_t* keys, int n, int64_t row) {
  const int lane = lane_id();
  const float INF = __int_as_float(0x7f800000);
  const int64_t ro = p.qid ? row : (p.perm ? (int64_t)p.perm[row] : row);
  const int32_t sid = p.qid ? p.qid[row] : (int32_t)ro;
  uint64_t last = 0ull;
  int drop = n;
  for (int e = 0; e < n; e += 32) {
    const uint64_t k = e + lane < n ? keys[e + lane] : 0ull;
    last = k > last ? k : last;
    if (p.self && drop == n) {
      const unsigned m = __ballot_sync(0xffffffffu, e + lane < n && key_id(k) == sid);
      if (m) drop = e + __ffs(m) - 1;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t k = __shfl_xor_sync(0xffffffffu, last, o);
    last = k > last ? k : last;
  }
  if (p.out_thresh && lane == 0)
    p.out_thresh[ro] = n >= p.KS ? key_dist(last) : (p.tau_in ? p.tau_in[row] : INF);
  if (p.self && drop == n && n >= p.KS) {
    for (int e = 0; e < n; e += 32) {
      const unsigned m = __ballot_sync(0xffffffffu, e + lane < n && keys[e + lane] == last);
      if (m) {
        drop = e + __ffs(m) - 1;
        break;
      }
    }
  }
  const int got = drop < n ? n - 1 : n;
  for (int t = lane; t < p.K; t += 32) {
    const uint64_t k = t < got ? keys[t < drop ? t : t + 1] : KEY_NONE;
    p.out_id[ro * p.K + t] = k == KEY_NONE ? -1 : key_id(k);
    p.out_d2[ro * p.K + t] = k == KEY_NONE ? INF : key_dist(k);
  }
}

__global__ void __launch_bounds__(128) k_knn_finish(FinArgs p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = lane_id();
  uint64_t* keys = (uint64_t*)(smem_raw + (size_t)warp * ((size_t)p.slots * 8 + (size_t)p.tcap * 4));
  uint32_t* ob = (uint32_t*)(keys + p.slots);
  const int64_t r = (int64_t)blockIdx.x * 4 + warp;
  if (r >= p.rows || (*p.err >> 1) != 0) return;
  const int64_t row = p.row0 + r;
  const uint2* rb = p.rowbuf + (size_t)r * p.nseg * p.C;
  const int* cn = p.cnt + r * p.nseg;
  int T = 0;
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
  for (int s = 0; s < p.nseg; ++s) {
    const int c = cn[s];
#pragma unroll 4
    for (int t = lane; t < c; t += 32) {
      const uint32_t k = ~float_order_bits(__uint_as_float(__ldcg(&rb[(size_t)s * p.C + t].y)));
      ob[T + t] = k;
      lo = min(lo, k);
      hi = max(hi, k);
    }
    T += c;
  }
  __syncwarp();
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  const int good = p.ts_out || !p.sorted ? p.KS : p.slots;
  int n = T;  // entries <= hi
  if (T > good) {
    while (lo < hi) {
      const uint32_t mid = lo + ((hi - lo) >> 1);
      int c = 0;
      for (int t = lane; t < T; t += 32) c += ob[t] <= mid ? 1 : 0;
      c = __reduce_add_sync(0xffffffffu, c);
      if (c >= p.KS) {
        hi = mid;
        n = c;
        if (c <= good) break;
      } else {
        lo = mid + 1;
      }
    }
  }
  if (p.ts_out) {
    // (a loop that stopped at exactly KS may leave hi above the KS-th largest's bits: still a
    // bound that KS entries meet)
    if (lane == 0)
      p.ts_out[row] = T >= p.KS ? ~hi : float_order_bits(LOWEST);
    return;
  }
  uint32_t idmax = 0xFFFFFFFFu;
  if (n > good) {
    // more ties at the KS-th distance than that: those with the smallest original ids stay
    int below = 0;
    for (int t = lane; t < T; t += 32) below += ob[t] < hi ? 1 : 0;
    const int need = p.KS - __reduce_add_sync(0xffffffffu, below);
    uint32_t l2 = 0u, h2 = 0x7FFFFFFFu;
    while (l2 < h2) {
      const uint32_t mid = l2 + ((h2 - l2) >> 1);
      int c = 0, base = 0;
      for (int s = 0; s < p.nseg; ++s) {
        for (int t = lane; t < cn[s]; t += 32)
          if (ob[base + t] == hi) {
            const uint32_t id = rb[(size_t)s * p.C + t].x;
            c += (p.perm ? (uint32_t)p.perm[id] : id) <= mid ? 1 : 0;
          }
        base += cn[s];
      }
      c = __reduce_add_sync(0xffffffffu, c);
      if (c >= need)
        h2 = mid;
      else
        l2 = mid + 1;
    }
    idmax = h2;
  }
  const float nx = p.a_norm[row];
  int kept = 0, base = 0;
  for (int s = 0; s < p.nseg; ++s) {
    const int c = cn[s];
    for (int t0 = 0; t0 < c; t0 += 32) {
      const int t = t0 + lane;
      bool keep = t < c && ob[base + t] <= hi;
      uint64_t key = 0ull;
      if (keep) {
        const uint2 v = __ldcg(&rb[(size_t)s * p.C + t]);
        const int32_t id = p.perm ? p.perm[v.x] : (int32_t)v.x;
        if (ob[base + t] == hi && (uint32_t)id > idmax) keep = false;
        key = make_key(fmaf(-2.f, __uint_as_float(v.y), nx), id);
      }
      const unsigned b = __ballot_sync(0xffffffffu, keep);
      if (keep) keys[kept + __popc(b & lanemask_lt())] = key;
      kept += __popc(b);
    }
    base += c;
  }
  __syncwarp();
  if (!p.sorted)
    raw_out(p, keys, kept, row);
  else if (kept <= 32)
    sort_out<1>(p, keys, kept, row);
  else if (kept <= 64)
    sort_out<2>(p, keys, kept, row);
  else if (kept <= 128)
    sort_out<4>(p, keys, kept, row);
  else if (kept <= 256)
    sort_out<8>(p, keys, kept, row);
  else if (kept <= 512)
    sort_out<16>(p, keys, kept, row);
  else
    sort_out<32>(p, keys, kept, row);
}

// Initial thresholds of the walk: from the caller's admission bounds (every column whose
// distance is at most tau is admitted), or none.
__global__ void k_ts_init(const float* __restrict__ tau, const float* __restrict__ a_norm, int64_t n,
                          uint32_t* __restrict__ ts) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float INF = __int_as_float(0x7f800000);
  const float t = tau ? tau[i] : INF;
  // d2 = fmaf(-2, acc, |x|^2) <= tau as the kernel forms it: one value below the rounded half
  // difference covers the rounding of both
  float v = LOWEST;
  if (t < INF) {
    v = 0.5f * (a_norm[i] - t);
    v -= (fabsf(a_norm[i]) + fabsf(t)) * 1.1920929e-07f;
  }
  ts[i] = float_order_bits(v);
}

// bf16 copy with rows padded to dp; with perm, stored row r holds row perm[r] (and its norm);
// with mu, the rows are centred first (x - mu rounded to fp32, then to bf16).
// Rows of width dp (pairs = 0) or of three parts of width dp (pairs = 1: [hi | lo | hi],
// pairs = 2: [lo | hi | hi], hi = bf16(v), lo = bf16(v - hi), v the centred value), so
// that the accumulator takes the small products hi.lo and lo.hi before hi.hi.
// Blocks of (2^txl, 256 / 2^txl) threads, eight values (two float4 loads, one 16-byte store)
// per thread and step.  Bound by memory: 1M x 128 gathered through perm 0.12 ms (6.3 TB/s
// read and written); one value per thread with a 64-bit division each took 0.51 ms.
__global__ void __launch_bounds__(256) k_to_bf16(
    const float* __restrict__ X, int64_t n, int d, int ld, __nv_bfloat16* __restrict__ Y, int dp,
    const int32_t* __restrict__ perm, const float* __restrict__ norm_in,
    float* __restrict__ norm_out, const float* __restrict__ mu, int pairs, int txl) {
  const int w8 = (pairs ? 3 * dp : dp) >> 3, dp8 = dp >> 3;
  const int tx = threadIdx.x & ((1 << txl) - 1);
  const int rows = 256 >> txl;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int64_t r = (int64_t)blockIdx.x * rows + (threadIdx.x >> txl); r < n;
       r += (int64_t)gridDim.x * rows) {
    const int64_t src = perm ? (int64_t)perm[r] : r;
    if (norm_out && tx == 0) norm_out[r] = norm_in[src];
    const float* x = X + src * ld;
    for (int c8 = tx; c8 < w8; c8 += 1 << txl) {
      const int part = c8 / dp8, c = (c8 - part * dp8) << 3;
      // rows are zero from d to ld, so a float4 that starts below d never leaves the row
      float4 a = c < d ? __ldg((const float4*)(x + c)) : zero;
      float4 b = c + 4 < d ? __ldg((const float4*)(x + c + 4)) : zero;
      float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
      const bool low = (pairs == 1 && part == 1) || (pairs == 2 && part == 0);
      __align__(16) __nv_bfloat16 o[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (mu && c + k < d) v[k] = __fsub_rn(v[k], __ldg(mu + c + k));
        const __nv_bfloat16 hi = __float2bfloat16_rn(v[k]);
        o[k] = low ? __float2bfloat16_rn(__fsub_rn(v[k], __bfloat162float(hi))) : hi;
      }
      *((uint4*)Y + r * w8 + c8) = *(const uint4*)o;
    }
  }
}

// Augmentation rows of the base: -|y|^2 / 2 as four bf16 parts (each the bf16 rounding of
// what the previous ones leave), then zeros (two 16-byte stores: 1M rows in 8 us, 94 us with
// sixteen 2-byte ones).  err is set if a row's
// parts do not add up to the value exactly.
__global__ void k_aug_rows(const float* __restrict__ norm, int64_t n, __nv_bfloat16* __restrict__ aug,
                           int* __restrict__ err, int approx) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    float rest = -0.5f * norm[r];
    __align__(16) __nv_bfloat16 o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) o[k] = __float2bfloat16_rn(0.f);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o[k] = __float2bfloat16_rn(rest);
      rest -= __bfloat162float(o[k]);
    }
    if (rest != 0.f && !approx) atomicOr(err, 1);
    static_assert(AUG == 16, "two 16-byte stores per augmentation row");
    uint4* dst = (uint4*)(aug + r * AUG);
    dst[0] = *(const uint4*)o;
    dst[1] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// Augmentation rows of the queries: four ones, then zeros (128 identical rows).
__global__ void k_aug_ones(__nv_bfloat16* __restrict__ aug) {
  for (int i = threadIdx.x; i < 128 * AUG; i += blockDim.x)
    aug[i] = __float2bfloat16_rn((i % AUG) < 4 ? 1.f : 0.f);
}

constexpr size_t SMEM_MAX = 225 * 1024;

// Shared memory of the kernel: resident A (kchunks 64-value chunks) or streamed (kchunks = 0).
size_t tc_smem_bytes(int kchunks, int stages) {
  const size_t stage = kchunks ? (size_t)kchunks * B_CHUNK + B_AUG : (size_t)A_CHUNK + B_CHUNK + B_AUG;
  return 1024 + (size_t)kchunks * A_CHUNK + A_AUG + (size_t)stages * stage +
         sizeof(uint64_t) * (2 + 2 * MAX_STAGES + 2 * NBUF) + 16;
}

struct TcMaps {
  CUtensorMap a, b, a_aug, b_aug;
};

template <int C, bool STREAM, bool LIMITED>
void launch_tc(const TcMaps& m, TcArgs& a, size_t smem, cudaStream_t st) {
  ensure_smem((const void*)k_knn_pair<C, STREAM, LIMITED>, smem);
  const int64_t pairs = std::min<int64_t>(a.nrb * a.nseg, num_sms() / 2);
  SSG_LAUNCH((k_knn_pair<C, STREAM, LIMITED>), (unsigned)(2 * pairs), THREADS, smem, st, m.a, m.b, m.a_aug,
             m.b_aug, a);
}

// Shares of each block's tiles.  A share more per block fills clusters that would idle, in the
// last wave or when there are few blocks; each share has its own climb to the threshold, about
// as long as `climb` tiles.  The shares' buffers of C entries are merged by one warp in
// shared memory, which bounds their number.
int pick_shares(int64_t nrb, int64_t nwalk, int C, int KS, int64_t clusters) {
  const int64_t smax = std::max<int64_t>(1, std::min<int64_t>({nwalk, (int64_t)(4096 / C), 16}));
  const double climb = 8.0 + KS / 4.0;
  int best = 1;
  double best_cost = 0.0;
  for (int64_t s = 1; s <= smax; ++s) {
    const double cost = (double)ceil_div(nrb * s, clusters) * ((double)ceil_div(nwalk, s) + climb);
    if (s == 1 || cost < best_cost) {
      best = (int)s;
      best_cost = cost;
    }
  }
  return best;
}

}  // namespace

bool knn_tc_available(int d) {
  static const int avail = [] {
    int dev = 0, major = 0, minor = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) == cudaSuccess)
      return (major == 10 && minor == 3 && encode_fn() != nullptr) ? 1 : 0;
    return 0;
  }();
  return avail == 1 && d >= 1 && d <= MAX_D_STREAM;
}

int knn_tc_max_k(int d, bool limited) {
  // a row buffer holds 1,024 entries: KS = K + 1 and room for a chunk of new ones (a limited
  // walk: for KS new ones)
  const int room = d <= MAX_D_RESIDENT ? 128 : 256;
  return limited ? (1024 - room) / 2 - 1 : 1024 - room - 1;
}

void rows_to_bf16(const float* X, int64_t n, int d, int ld, __nv_bfloat16* Y, int dp,
                  const int32_t* perm, const float* norm_in, float* norm_out, const float* mu,
                  int pairs, cudaStream_t st) {
  int txl = 3;  // threads per row: the largest power of two within the row's 16-byte pieces
  while (txl < 5 && (2 << txl) <= (pairs ? 3 : 1) * (dp >> 3)) ++txl;
  const int64_t want = ceil_div(n, (int64_t)(256 >> txl));
  SSG_LAUNCH(k_to_bf16, (unsigned)std::min<int64_t>(want, 16 * num_sms()), 256, 0, st, X, n, d, ld,
             Y, dp, perm, norm_in, norm_out, mu, pairs, txl);
}

void knn_exact_tc(const float* A, int64_t na, int lda, const float* a_norm, const float* B,
                  int64_t nb, int ldb, const float* b_norm, int d, int self, int K,
                  int32_t* out_id, float* out_d2, cudaStream_t st, StageTimer* gemm_timer,
                  int max_tiles, bool approx, const TcExtra& ex) {
  const int dp = (d + 63) & ~63;
  const int dpe = ex.pairs ? 3 * dp : dp;  // row width the tensor cores see
  const int kchunks = dpe / 64;
  SSG_REQUIRE(dpe <= MAX_D_STREAM, SSG_EINVAL,
              "tensor-core kNN: d = %d is too large for the shared-memory pipeline", d);
  // rows too long to stay resident stream through the pipeline with the tiles
  const bool stream = dpe > MAX_D_RESIDENT || ex.stream_rows;
  int stages = MAX_STAGES;
  while (stages > 2 && tc_smem_bytes(stream ? 0 : kchunks, stages) > SMEM_MAX) --stages;
  const size_t smem = tc_smem_bytes(stream ? 0 : kchunks, stages);
  const int KS = self ? K + 1 : K;
  // Near-first column order for large self-joins with a deep top-K (where the streaming
  // threshold otherwise falls slowly and many candidates are appended).
  KnnOrder ord;
  Scratch<float> norm_p;
  // same: the query rows are the base rows (a self-join); with ex.qid the query rows are a
  // gathered subset of the base and only the self column is excluded
  const bool same = self && !ex.qid;
  // A limited walk's lists set what each row is compared with: max_tiles 128-point tiles for each
  // block of 256 rows, or (rows longer than 128 values) as many points in 256-point tiles for each
  // block of 128.  A work item walks the tiles of all its blocks' lists, and each block's rows
  // take only those of their own.
  const int list_rows = max_tiles == 0 ? BM : stream ? 128 : 256;
  const int list_tile = max_tiles == 0 || stream ? BN : API_TILE;
  SSG_REQUIRE(max_tiles == 0 || (same && knn_order_fits(na, list_tile)), SSG_EINVAL,
              "a tile limit needs a self-join whose cluster order fits");
  // (not for streamed rows: their tiles are long enough that the appends a slowly falling
  // threshold costs matter less than L2 reuse, which needs every cluster to walk the columns in
  // the same order: 200,000 x 960 with bf16 pairs, 270 -> 227 ms, the near-first walks kept
  // DRAM 78% busy at a 34% L2 hit rate)
  const bool ordered =
      max_tiles > 0 || (!stream && same && na >= (1 << 16) && K >= 16 && knn_order_fits(na, BN));
  if (ordered) {
    const float* on = ex.order_norm ? ex.order_norm : a_norm;
    knn_cluster_order(A, lda, d, na, list_rows, list_tile, st, ord,
                      ceil_div((int64_t)max_tiles * API_TILE, list_tile), on);
    norm_p.alloc((size_t)na, st);
  }
  const int32_t* perm = ordered ? (const int32_t*)ord.perm.p : nullptr;
  Scratch<__nv_bfloat16> ab((size_t)na * dpe, st);
  Scratch<__nv_bfloat16> bb;
  rows_to_bf16(A, na, d, lda, ab.p, dp, perm, a_norm, ordered ? norm_p.p : nullptr, ex.mu,
               ex.pairs ? 1 : 0, st);
  if (ordered) a_norm = b_norm = norm_p.p;
  const __nv_bfloat16* bptr = ab.p;
  if (!same || ex.pairs) {
    // bf16 pairs: the base side has its own layout (in the self-join's stored order)
    bb.alloc((size_t)nb * dpe, st);
    rows_to_bf16(B, nb, d, ldb, bb.p, dp, same ? perm : nullptr, nullptr, nullptr, ex.mu,
                 ex.pairs ? 2 : 0, st);
    bptr = bb.p;
  }
  Scratch<__nv_bfloat16> aug_b((size_t)nb * AUG, st), aug_a((size_t)128 * AUG, st);
  Scratch<int> err(1, st);
  SSG_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
  SSG_LAUNCH(k_aug_rows, (unsigned)std::min<int64_t>(ceil_div(nb, 256), 8 * num_sms()), 256, 0, st,
             b_norm, nb, aug_b.p, err.p, approx ? 1 : 0);
  SSG_LAUNCH(k_aug_ones, 1, 256, 0, st, aug_a.p);
  TcMaps maps;
  maps.a = make_map(ab.p, na, dpe, 64, CM, CU_TENSOR_MAP_SWIZZLE_128B);
  maps.b = make_map(bptr, nb, dpe, 64, BN / 2, CU_TENSOR_MAP_SWIZZLE_128B);
  maps.a_aug = make_map(aug_a.p, 128, AUG, AUG, 128, CU_TENSOR_MAP_SWIZZLE_32B);
  maps.b_aug = make_map(aug_b.p, nb, AUG, AUG, BN / 2, CU_TENSOR_MAP_SWIZZLE_32B);
  // A row buffer holds C entries and is cut back once 64 columns could overflow it.  A limited
  // walk spends most of its tiles while the threshold is still falling, so it gets room for
  // about KS more entries between cuts.
  const int room = dpe <= MAX_D_RESIDENT ? 128 : 256;
  const int need = max_tiles > 0 ? 2 * KS + room : KS + room;
  SSG_REQUIRE(need <= 1024, SSG_EINVAL, "tensor-core kNN: K = %d is too large for %d-value rows", K,
              dpe);
  const int C = need <= 256 ? 256 : (need <= 512 ? 512 : 1024);
  const int64_t ntiles = ceil_div(nb, BN), nrb = ceil_div(na, BM);
  TcArgs a{};
  a.na = na;
  a.nb = nb;
  a.nwalk = ntiles;
  a.tstride = max_tiles > 0 ? std::min<int64_t>(BM / list_rows * ord.tstride, ntiles)
                            : (ordered ? ord.tstride : ntiles);
  a.nseg = max_tiles > 0 ? 1 : pick_shares(nrb, a.nwalk, C, KS, num_sms() / 2);
  a.kchunks = kchunks;
  a.dp_chunks = dp / 64;
  a.d = d;
  a.stages = stages;
  a.KS = KS;
  a.err = err.p;
  if (ordered) {
    a.perm = ord.perm.p;
    a.tile_order = ord.tile_order.p;
    a.rb_cluster = ord.rb_cluster.p;
  }
  // Near-first full walks may be preceded by one over each block's prepass_tiles nearest tiles
  // that only records each row's KS-th largest accumulator there, from which the full walk
  // starts.
  const int64_t pre_tiles = ceil_div((int64_t)ex.prepass_tiles * API_TILE, BN);
  const bool prepass = ordered && max_tiles == 0 && pre_tiles > 0 && ntiles > 2 * pre_tiles;
  // thresholds per query row: to start from, and for the shares to exchange
  Scratch<uint32_t> ts;
  if (ex.tau_in || a.nseg > 1 || prepass) {
    ts.alloc((size_t)na, st);
    SSG_LAUNCH(k_ts_init, (unsigned)ceil_div(na, 256), 256, 0, st, ex.tau_in, a_norm, na, ts.p);
    a.ts_g = ts.p;
  }
  // The row buffers of one launch take up to 2 GB, or an eighth of the memory that is left where
  // that is less; more rows go in several launches, whole rounds of the clusters each.
  const int64_t round = std::max<int64_t>(1, num_sms() / 2);
  int64_t rounds = ceil_div(nrb, round);
  if (rounds > 1) {
    const size_t round_bytes = (size_t)round * BM * a.nseg * C * sizeof(uint2);
    const size_t room = std::min<size_t>(2ull << 30, scratch_room() / 8);
    rounds = std::min(rounds, std::max<int64_t>(1, (int64_t)(room / round_bytes)));
  }
  int64_t per_launch = std::min<int64_t>(nrb, rounds * round);
  Scratch<uint2> rowbuf;
  while (!rowbuf.try_alloc((size_t)per_launch * BM * a.nseg * C, st)) {
    // where the device has less room: fewer rounds, then fewer shares, down to one round of rows
    // whose columns are not shared out (SMs / 2 x 512 rows x C entries: 160 MB at C = 512)
    if (rounds > 1)
      rounds = ceil_div(rounds, 2);
    else if (a.nseg > 1)
      a.nseg = (a.nseg + 1) / 2;
    else
      throw Fail{SSG_ENOMEM};
    per_launch = std::min<int64_t>(nrb, rounds * round);
  }
  Scratch<int> cnt((size_t)per_launch * BM * a.nseg, st);
  a.rowbuf = rowbuf.p;
  a.cnt = cnt.p;
  // a limited walk's lists of one launch's items
  Scratch<int32_t> item_tiles, item_len;
  if (max_tiles > 0) {
    item_tiles.alloc((size_t)(per_launch * a.tstride), st);
    item_len.alloc((size_t)per_launch, st);
    a.tile_order = item_tiles.p;
    a.rb_cluster = nullptr;
    a.walk_len = item_len.p;
  }
  FinArgs f{};
  f.err = err.p;
  f.rowbuf = rowbuf.p;
  f.cnt = cnt.p;
  f.C = C;
  f.KS = KS;
  f.K = K;
  f.self = self;
  f.sorted = !ex.any_order;
  f.a_norm = a_norm;
  f.perm = a.perm;
  f.qid = ex.qid;
  f.tau_in = ex.tau_in;
  f.out_id = out_id;
  f.out_d2 = out_d2;
  f.out_thresh = ex.out_thresh;
  f.slots = next_pow2(std::max(KS, 32));
  auto walk = [&](TcArgs args, FinArgs fin) {
    args.nseg = (int)std::min<int64_t>(args.nseg, args.nwalk);
    fin.nseg = args.nseg;
    fin.tcap = args.nseg * C;
    const size_t fsm = 4 * ((size_t)fin.slots * 8 + (size_t)fin.tcap * 4);
    ensure_smem((const void*)k_knn_finish, fsm);
    for (int64_t rb = 0; rb < nrb; rb += per_launch) {
      args.rb0 = rb;
      args.nrb = std::min<int64_t>(per_launch, nrb - rb);
      if (max_tiles > 0)
        knn_item_tiles(ord, na, list_rows, list_tile, rb, args.nrb, args.tstride, item_tiles.p,
                       item_len.p, st);
      auto launch = [&](auto size) {
        constexpr int S = decltype(size)::value;
        if (max_tiles > 0)
          stream ? launch_tc<S, true, true>(maps, args, smem, st)
                 : launch_tc<S, false, true>(maps, args, smem, st);
        else
          stream ? launch_tc<S, true, false>(maps, args, smem, st)
                 : launch_tc<S, false, false>(maps, args, smem, st);
      };
      if (C == 256)
        launch(std::integral_constant<int, 256>());
      else if (C == 512)
        launch(std::integral_constant<int, 512>());
      else
        launch(std::integral_constant<int, 1024>());
      fin.row0 = rb * BM;
      fin.rows = std::min<int64_t>(args.nrb * BM, na - fin.row0);
      SSG_LAUNCH(k_knn_finish, (unsigned)ceil_div(fin.rows, 4), 128, fsm, st, fin);
    }
  };
  if (gemm_timer) gemm_timer->start();
  if (prepass) {
    TcArgs a0 = a;
    a0.nwalk = pre_tiles;
    FinArgs f0 = f;
    f0.ts_out = ts.p;
    walk(a0, f0);
  }
  walk(a, f);
  if (gemm_timer) gemm_timer->stop();
  int h = 0;
  SSG_CUDA(cudaMemcpyAsync(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
  SSG_CUDA(cudaStreamSynchronize(st));
  if (h != 0) note_device_status(h == 1 ? SSG_EINTERNAL : SSG_ETIMEOUT);
  SSG_REQUIRE(h != 1, SSG_EINTERNAL, "tensor-core kNN: a squared norm is not split exactly");
  SSG_REQUIRE(h == 0, SSG_ETIMEOUT, "tensor-core kNN: a pipeline wait timed out (code %d)", h);
}

}  // namespace ssg
