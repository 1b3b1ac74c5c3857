// Search-on-Graph (Alg. 1) from the navigating node nearest the query (Sec. 4.1).
//
// One warp per query.  The candidate pool S (at most L_search entries, sorted by (d2, id),
// with a checked flag in each key's last bit) lives in shared memory; each round expands the
// first unchecked entry, gathers its adjacency row, computes the distances of the neighbours
// not seen before, and merges those below the pool's last key into it: a sort in registers, one
// binary search for each new key's place and duplicate test, and a move of the entries behind
// the first new one.
//
// Rows: float32, or -- for data that are integers 0..255 -- a byte copy of the same
// values.  A byte row of 128 dimensions is one 128-byte line instead of four; every lane
// converts its bytes to the same float values and sums them in the same order as the
// float path, so the distances and results are bit for bit those of the float rows.
//
// Visited set: a direct-mapped cache of ids in shared memory.  Alg. 1 never re-adds a
// visited node; here a node that fell out of the cache may be met again and its distance
// recomputed, but the result is the same: a node that is still in S has the same key and
// is dropped by the duplicate check of the merge, and a node that left S (or never
// entered it) did so because S was full and its key was above the L_search-th key, which
// never increases once S is full, so it is cut again.  Before S first fills nothing has
// left it.  The cache only saves distance computations.
#include <type_traits>

#include "common.cuh"
#include "graph_dev.cuh"
#include "knn.cuh"

namespace ssg {

// Four consecutive values of a row as floats: one float4 load, or one 32-bit load of four
// bytes (each byte b becomes the float 2^23 + b by placing it under the exponent bits of
// 2^23, then b exactly by subtracting 2^23).
__device__ __forceinline__ float4 row_raw(const float* x, int f) {
  return __ldg((const float4*)x + f);
}
__device__ __forceinline__ uint32_t row_raw(const uint8_t* x, int f) {
  return __ldg((const unsigned int*)x + f);
}
__device__ __forceinline__ float4 raw_f4(float4 v) { return v; }
__device__ __forceinline__ float byte_f(uint32_t w, uint32_t sel) {
  return __uint_as_float(__byte_perm(w, 0x4B000000u, sel)) - 8388608.f;
}
__device__ __forceinline__ float4 raw_f4(uint32_t w) {
  return make_float4(byte_f(w, 0x7440), byte_f(w, 0x7441), byte_f(w, 0x7442), byte_f(w, 0x7443));
}
template <typename T>
struct RawOf;
template <>
struct RawOf<float> {
  using type = float4;
  static __device__ __forceinline__ float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
};
template <>
struct RawOf<uint8_t> {
  using type = uint32_t;
  static __device__ __forceinline__ uint32_t zero() { return 0u; }
};

// Squared distances of the query to NR rows per team of four lanes (8 NR rows per warp): row r is
// X + ids[r] * ld (rows with valid[r] false give 0).  Lane tl of a team sums float4 groups 2 tl
// and 2 tl + 1 modulo 8, each modulus in one sequence; the eight sums of a row are then added
// pairwise.  (The order of teams of eight lanes with one modulus each, kept so that results
// stay the same to the bit; four lanes need two shuffles per row set instead of three.)
template <typename T, int NR>
__device__ __forceinline__ void team4_dist_q(const float* __restrict__ qs, const T* __restrict__ X,
                                             int ld, const int32_t (&ids)[NR],
                                             const bool (&valid)[NR], int tl, float (&out)[NR]) {
  using Raw = typename RawOf<T>::type;
  const float4* q4 = (const float4*)qs;
  const int ld4 = ld >> 2;
  float s[NR][2];
#pragma unroll
  for (int r = 0; r < NR; ++r) s[r][0] = s[r][1] = 0.f;
  for (int f0 = 2 * tl; f0 < ld4; f0 += 32) {
    Raw raw[NR][8];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const T* x = X + (int64_t)ids[r] * ld;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int f = f0 + 8 * (i >> 1) + (i & 1);
        raw[r][i] = (valid[r] && f < ld4) ? row_raw(x, f) : RawOf<T>::zero();
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int f = f0 + 8 * (i >> 1) + (i & 1);
      if (f < ld4) {
        const float4 q = q4[f];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const float4 v = raw_f4(raw[r][i]);
          float u;
          u = q.x - v.x; s[r][i & 1] = fmaf(u, u, s[r][i & 1]);
          u = q.y - v.y; s[r][i & 1] = fmaf(u, u, s[r][i & 1]);
          u = q.z - v.z; s[r][i & 1] = fmaf(u, u, s[r][i & 1]);
          u = q.w - v.w; s[r][i & 1] = fmaf(u, u, s[r][i & 1]);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    out[r] = valid[r] ? s[r][0] + s[r][1] : 0.f;
    out[r] += __shfl_xor_sync(0xffffffffu, out[r], 1);
    out[r] += __shfl_xor_sync(0xffffffffu, out[r], 2);
  }
}

// The same for float rows, by teams of eight lanes (4 NR rows per warp): a load instruction of
// the warp then takes whole 128-byte lines of four rows, where teams of four would take half
// lines of eight.  The eight sums of a row are added in the same pairs, each lane handing on half
// of its rows at every step: the distance of row team8_row<NR>(tl) is returned in lane tl.
template <int NR>
__device__ __forceinline__ int team8_row(int tl) {
  return NR == 4 ? 2 * (tl & 1) + ((tl >> 1) & 1) : tl & 1;
}
template <int NR>
__device__ __forceinline__ float team8_dist_q(const float* __restrict__ qs,
                                              const float* __restrict__ X, int ld,
                                              const int32_t (&ids)[NR], const bool (&valid)[NR],
                                              int tl) {
  static_assert(NR == 2 || NR == 4, "two or four rows per team");
  const float4* q4 = (const float4*)qs;
  const int ld4 = ld >> 2;
  float s[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) s[r] = 0.f;
  for (int f0 = tl; f0 < ld4; f0 += 32) {
    float4 raw[NR][4];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const float* x = X + (int64_t)ids[r] * ld;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int f = f0 + 8 * i;
        raw[r][i] = (valid[r] && f < ld4) ? row_raw(x, f) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int f = f0 + 8 * i;
      if (f < ld4) {
        const float4 q = q4[f];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const float4 v = raw[r][i];
          float u;
          u = q.x - v.x; s[r] = fmaf(u, u, s[r]);
          u = q.y - v.y; s[r] = fmaf(u, u, s[r]);
          u = q.z - v.z; s[r] = fmaf(u, u, s[r]);
          u = q.w - v.w; s[r] = fmaf(u, u, s[r]);
        }
      }
    }
  }
  const bool odd = tl & 1, two = tl & 2;
  float t;
  if constexpr (NR == 4) {
    const float a = odd ? s[0] : s[2], b = odd ? s[1] : s[3];
    float k0 = odd ? s[2] : s[0], k1 = odd ? s[3] : s[1];
    k0 += __shfl_xor_sync(0xffffffffu, a, 1);
    k1 += __shfl_xor_sync(0xffffffffu, b, 1);
    t = two ? k1 : k0;
    t += __shfl_xor_sync(0xffffffffu, two ? k0 : k1, 2);
  } else {
    t = odd ? s[1] : s[0];
    t += __shfl_xor_sync(0xffffffffu, odd ? s[0] : s[1], 1);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
  }
  t += __shfl_xor_sync(0xffffffffu, t, 4);
  return t;
}

// Integer queries (every value an integer 0..255) against byte rows: with the query's bytes
// packed four to a word (qw) and q2 = |q|^2, d2 = q2 + |x|^2 - 2 q.x from byte dot products
// (dp4a), all in exact integer arithmetic.  Every value and partial sum of the float path
// is an integer below 2^24 in that case, so the float path's sums are exact too and the two
// give the same distances.  Rows of a multiple of 16 bytes load in 16-byte pieces, others (WORDS) in
// words; either way a step's loads are all issued before the first product (words loaded and used one
// by one: 50,000 x 100, L_search 10, 10,000 queries 355 us, teams of eight with all loads first 256,
// now 214).
__device__ __forceinline__ int sum_dp4a(uint32_t q, uint32_t x, int s) {
  return s + (int)__dp4a(x, x, 0u) - 2 * (int)__dp4a(q, x, 0u);
}
template <int NR, bool WORDS>
__device__ __forceinline__ void team4_dist_qi(const uint32_t* __restrict__ qw,
                                              const uint8_t* __restrict__ X, int ld,
                                              const int32_t (&ids)[NR], const bool (&valid)[NR],
                                              int tl, int q2, float (&out)[NR]) {
  int s[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) s[r] = 0;
  if constexpr (!WORDS) {
    const int np = ld >> 4;
    for (int c0 = tl; c0 < np; c0 += 8) {
      uint4 raw[NR][2];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const uint4* x = (const uint4*)(X + (int64_t)ids[r] * ld);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int c = c0 + 4 * i;
          raw[r][i] = (valid[r] && c < np) ? __ldg(x + c) : make_uint4(0u, 0u, 0u, 0u);
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int c = c0 + 4 * i;
        if (c < np) {
          const uint4 q = ((const uint4*)qw)[c];
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            s[r] = sum_dp4a(q.x, raw[r][i].x, s[r]);
            s[r] = sum_dp4a(q.y, raw[r][i].y, s[r]);
            s[r] = sum_dp4a(q.z, raw[r][i].z, s[r]);
            s[r] = sum_dp4a(q.w, raw[r][i].w, s[r]);
          }
        }
      }
    }
  } else {
    const int nw = ld >> 2;
    for (int w0 = tl; w0 < nw; w0 += 32) {
      uint32_t raw[NR][8];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const uint8_t* x = X + (int64_t)ids[r] * ld;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int w = w0 + 4 * i;
          raw[r][i] = (valid[r] && w < nw) ? row_raw(x, w) : 0u;
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int w = w0 + 4 * i;
        if (w < nw) {
          const uint32_t q = qw[w];
#pragma unroll
          for (int r = 0; r < NR; ++r) s[r] = sum_dp4a(q, raw[r][i], s[r]);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    s[r] += __shfl_xor_sync(0xffffffffu, s[r], 1);
    s[r] += __shfl_xor_sync(0xffffffffu, s[r], 2);
    out[r] = (float)(q2 + s[r]);
  }
}

// Pool keys: (distance bits, id, checked flag) packed so that they sort by (distance, id).
__device__ __forceinline__ uint64_t pool_key(float d, int32_t id) {
  return ((uint64_t)float_order_bits(d) << 32) | ((uint32_t)id << 1);
}
__device__ __forceinline__ int32_t pool_id_of(uint64_t k) { return (int32_t)((uint32_t)k >> 1); }

// One compare-exchange step of a bitonic network over the warp (one key per lane).
__device__ __forceinline__ uint64_t exchange(uint64_t b, int j, bool take_min) {
  const uint64_t o = __shfl_xor_sync(0xffffffffu, b, j);
  return take_min == (o < b) ? o : b;
}
// Ascending sort of one key per lane within groups of N lanes (a power of two).
template <int N>
__device__ __forceinline__ uint64_t warp_bitonic(uint64_t b, int lane) {
#pragma unroll
  for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1)
      b = exchange(b, j, ((lane & j) == 0) == (k == N || (lane & k) == 0));
  }
  return b;
}

// number of entries of a[0, len) that are < x (a sorted ascending)
__device__ __forceinline__ int count_less(const uint64_t* a, int len, uint64_t x) {
  int lo = 0, hi = len;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a[mid] < x)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// The candidate pool S of one warp, sorted, in shared memory.
struct Pool {
  uint64_t* p;
  uint64_t worst;  // the Ls-th key, above every key with its node (KEY_NONE until S is full)
  int s, Ls;       // entries, and their largest number
  int lo;          // every entry before this one is checked

  __device__ __forceinline__ void init(uint64_t* buf, uint64_t first, int size) {
    p = buf;
    Ls = size;
    if (lane_id() == 0) p[0] = first;
    s = 1;
    lo = 0;
    worst = Ls == 1 ? first | 1ull : KEY_NONE;
    __syncwarp();
  }
  // The first unchecked entry's id (marked checked), or -1; second: the id of the one after it.
  __device__ __forceinline__ int32_t take(int32_t& second) {
    const int lane = lane_id();
    int32_t first = -1;
    second = -1;
    for (int c = lo & ~31; c < s; c += 32) {
      const uint32_t w = c + lane < s ? (uint32_t)p[c + lane] : 1u;
      unsigned bal = __ballot_sync(0xffffffffu, !(w & 1u));
      if (!bal) continue;
      const int l = __ffs(bal) - 1;
      if (first < 0) {
        first = (int32_t)(__shfl_sync(0xffffffffu, w, l) >> 1);
        if (lane == l) p[c + l] |= 1ull;
        lo = c + l + 1;
        bal &= bal - 1u;
      }
      if (bal) {
        second = (int32_t)(__shfl_sync(0xffffffffu, w, __ffs(bal) - 1) >> 1);
        break;
      }
    }
    __syncwarp();
    return first;
  }
  // Merges up to 32 keys (mine: one per lane, KEY_NONE for none; flags clear) into S: those
  // below the pool's last key, without the nodes it holds.  Most expansions late in a search
  // leave few of them, so the sort is as small as they allow, and only the entries behind the
  // first new one move.  tmp: room for 32 keys.
  __device__ __forceinline__ void merge(uint64_t mine, uint64_t* tmp) {
    const int lane = lane_id();
    const unsigned lt = lanemask_lt();
    unsigned bal = __ballot_sync(0xffffffffu, mine < worst);
    if (!bal) return;
    const int m = __popc(bal);
    uint64_t x = mine < worst ? mine : KEY_NONE;
    if (m <= 16) {
      __syncwarp();
      if (mine < worst) tmp[__popc(bal & lt)] = mine;
      __syncwarp();
      x = lane < m ? tmp[lane] : KEY_NONE;
      x = m <= 8 ? warp_bitonic<8>(x, lane) : warp_bitonic<16>(x, lane);
    } else {
      x = warp_bitonic<32>(x, lane);
    }
    int r = 0;
    bool keep = false;
    if (lane < m) {
      r = count_less(p, s, x);
      keep = r >= s || (p[r] ^ x) >= 2ull;
    }
    bal = __ballot_sync(0xffffffffu, keep);
    if (!bal) return;
    const int kept = __popc(bal), j = __popc(bal & lt);
    __syncwarp();
    if (keep) tmp[j] = x;
    const int r0 = __shfl_sync(0xffffffffu, r, __ffs(bal) - 1);
    __syncwarp();
    // entries move up, so the last 32 go first
    for (int c = (s - 1) & ~31; c + 31 >= r0 && c >= 0; c -= 32) {
      const int i = c + lane;
      const bool moves = i >= r0 && i < s;
      const uint64_t a = moves ? p[i] : 0ull;
      const int pos = moves ? i + count_less(tmp, kept, a) : Ls;
      __syncwarp();
      if (pos < Ls) p[pos] = a;
    }
    __syncwarp();
    if (keep && r + j < Ls) p[r + j] = x;
    s = s + kept < Ls ? s + kept : Ls;
    lo = r0 < lo ? r0 : lo;
    __syncwarp();
    if (s == Ls) worst = p[Ls - 1] | 1ull;
  }
};

struct SearchLayout {
  int Ls, RP, ld, log2h;  // Ls: the largest pool, even; RP: a multiple of 32, at least R
  int qb;                 // bytes for the query packed to bytes (float rows: none)
  __host__ __device__ size_t per_warp() const {
    return (size_t)Ls * 8 + (size_t)(RP + 32) * 8 + (size_t)ld * 4 + (size_t)qb + ((size_t)4 << log2h);
  }
};

// One warp per query.  Per expansion: the node's neighbours not in the visited cache (its row
// and degree load together, and the row of the next unchecked entry is fetched ahead, so that
// the next expansion often starts with it), their distances by teams of four lanes (byte
// rows) or eight (float rows) with all loads of 16 or 8 rows issued at once, and a merge of those below the pool's last key.  Bound by
// that chain of latencies and by its instructions, not by memory.  Against teams of eight lanes,
// a dependent degree and row load, and a sort of all new neighbours merged into a second copy
// of the pool: 10,000 queries over 1M x 128 byte rows, L_search 40, 0.74 -> 0.54 ms; one query
// 128 -> 90 us.  Byte rows take 24 warps per SM with 16 rows in flight (32 warps, 0.56 ms, spill;
// 32 rows 0.63).  Float rows take teams of eight: 50,000 x 128, L_search 40, 10,000 queries 883 ->
// 723 us, one query 172 -> 122 (teams of four: 796 and 181; 32 warps per SM with spills 738).  A
// pool in registers with an insertion per accepted neighbour was slower (0.93 ms): on the way to
// the query about half the neighbours are accepted.
// WORDS: byte rows of no multiple of 16 bytes, a kernel of their own: with both loads in one, rows of 128
// bytes took 1-2% longer (one query over 200,000 x 128 91.4 us, now 89.8; 10,000 over 1M 550 / 545).
template <typename T, int NR, int MIN_BLOCKS, bool WORDS>
__global__ void __launch_bounds__(256, MIN_BLOCKS)
    k_search(const T* __restrict__ X, int ld, int d, const int32_t* __restrict__ adj,
             const int32_t* __restrict__ deg, int R, const int32_t* __restrict__ nav, int n_nav,
             const float* __restrict__ Q, int ldq, int64_t nq, int k, int ls,
             const int32_t* __restrict__ qk, const int32_t* __restrict__ qls,
             const int32_t* __restrict__ from, int ldo, SearchLayout lay,
             int32_t* __restrict__ out_ids, float* __restrict__ out_d2,
             unsigned long long* __restrict__ work) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  constexpr bool BYTES = std::is_same<T, uint8_t>::value;
  constexpr int TEAMS = BYTES ? 8 : 4;  // a team takes NR rows at once
  constexpr int PIECES = 4;          // of 32 neighbours (R <= 128)
  const int wpb = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = lane_id();
  const int team = lane / (32 / TEAMS), tl = lane % (32 / TEAMS);
  unsigned char* base = sm_raw + (size_t)warp * lay.per_warp();
  uint64_t* pool = (uint64_t*)base;
  uint64_t* newk = pool + lay.Ls;                        // [RP] ids, then keys
  uint64_t* tmp = newk + lay.RP;                         // [32]
  float* qs = (float*)(tmp + 32);                        // [ld]
  uint32_t* qw = (uint32_t*)(qs + ld);                   // the query's bytes, if integer 0..255
  int32_t* cache = (int32_t*)((unsigned char*)qw + lay.qb);
  const int hcap = 1 << lay.log2h;

  for (int64_t qi = (int64_t)blockIdx.x * wpb + warp; qi < nq; qi += (int64_t)gridDim.x * wpb) {
    // per-query pool size and result count (a batch may mix them; the layout holds the
    // largest pool)
    const int Ls = qls ? qls[qi] : ls;
    const int kq = qk ? qk[qi] : k;
    const float* qg = Q + qi * ldq;
    for (int t = lane; t < ld; t += 32) qs[t] = t < d ? qg[t] : 0.f;
    for (int t = lane * 4; t < hcap; t += 128) *(int4*)(cache + t) = make_int4(-1, -1, -1, -1);
    __syncwarp();
    bool qint = false;
    int q2 = 0;
    if constexpr (BYTES) {
      bool ok = true;
      int sq = 0;
      for (int t = lane; t < ld; t += 32) {
        const float v = qs[t];
        ok = ok && v >= 0.f && v <= 255.f && v == rintf(v);
        const int iv = ok ? (int)v : 0;
        sq += iv * iv;
      }
      qint = __all_sync(0xffffffffu, ok);
      if (qint) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        q2 = sq;
        for (int w = lane; w < ld >> 2; w += 32)
          qw[w] = (uint32_t)qs[4 * w] | ((uint32_t)qs[4 * w + 1] << 8) |
                  ((uint32_t)qs[4 * w + 2] << 16) | ((uint32_t)qs[4 * w + 3] << 24);
        __syncwarp();
      }
    }

    // entry: the nearest navigating node by (d2, id), or the query's own start node
    uint64_t best = KEY_NONE;
    const int32_t* starts = from ? from + qi : nav;
    if constexpr (BYTES) {
      for (int s0 = 0; s0 < n_nav; s0 += 8) {
        const bool valid[1] = {s0 + team < n_nav};
        const int32_t id[1] = {valid[0] ? starts[s0 + team] : 0};
        float dd[1];
        team4_dist_q<T, 1>(qs, X, ld, id, valid, tl, dd);
        const uint64_t key = valid[0] ? pool_key(dd[0], id[0]) : KEY_NONE;
        best = key < best ? key : best;
      }
    } else {
      for (int s0 = 0; s0 < n_nav; s0 += TEAMS * NR) {
        int32_t ir[NR];
        bool vr[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int t = s0 + TEAMS * r + team;
          vr[r] = t < n_nav;
          ir[r] = vr[r] ? starts[t] : 0;
        }
        const float dd = team8_dist_q<NR>(qs, X, ld, ir, vr, tl);
        const int t = s0 + TEAMS * team8_row<NR>(tl) + team;
        const uint64_t key = t < n_nav ? pool_key(dd, starts[t]) : KEY_NONE;
        best = key < best ? key : best;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t other = __shfl_xor_sync(0xffffffffu, best, o);
      best = other < best ? other : best;
    }
    Pool S;
    S.init(pool, best, Ls);
    if (lane == 0) {
      const int32_t e = pool_id_of(best);
      cache[((uint32_t)e * 2654435761u) >> (32 - lay.log2h)] = e;
    }
    unsigned long long w_exp = 0, w_dist = (unsigned long long)n_nav, w_adj = 0;
    __syncwarp();

    // a node's row and degree (entries past the degree are dropped when it is expanded)
    int32_t row[PIECES];
    int dg = 0;
    auto fetch = [&](int32_t node) {
      dg = deg[node];
#pragma unroll
      for (int c = 0; c < PIECES; ++c)
        row[c] = c * 32 + lane < R ? adj[(int64_t)node * R + c * 32 + lane] : -1;
    };
    int32_t have = -1;  // the node whose row is in the registers
    for (;;) {
      int32_t ahead;
      const int32_t node = S.take(ahead);
      if (node < 0) break;
      if (node != have) fetch(node);
      int cnt = 0;
      const int dgn = dg;
#pragma unroll
      for (int c = 0; c < PIECES; ++c) {
        if (c * 32 < dgn) {
          bool fresh = false;
          const int32_t id = row[c];
          if (c * 32 + lane < dgn) {
            const uint32_t slot = ((uint32_t)id * 2654435761u) >> (32 - lay.log2h);
            if (cache[slot] != id) {
              cache[slot] = id;
              fresh = true;
            }
          }
          const unsigned bal = __ballot_sync(0xffffffffu, fresh);
          if (fresh) newk[cnt + __popc(bal & lanemask_lt())] = (uint64_t)(uint32_t)id;
          cnt += __popc(bal);
        }
      }
      have = ahead;
      if (ahead >= 0) fetch(ahead);
      ++w_exp;
      w_adj += (unsigned long long)dgn;
      w_dist += (unsigned long long)cnt;
      __syncwarp();
      for (int t0 = 0; t0 < cnt; t0 += TEAMS * NR) {
        int32_t ir[NR];
        bool vr[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int t = t0 + TEAMS * r + team;
          vr[r] = t < cnt;
          ir[r] = vr[r] ? (int32_t)(uint32_t)newk[t] : 0;
        }
        if constexpr (BYTES) {
          float dd[NR];
          if (qint)
            team4_dist_qi<NR, WORDS>(qw, X, ld, ir, vr, tl, q2, dd);
          else
            team4_dist_q<T, NR>(qs, X, ld, ir, vr, tl, dd);
          __syncwarp();
          if (tl == 0) {
#pragma unroll
            for (int r = 0; r < NR; ++r)
              if (vr[r]) newk[t0 + TEAMS * r + team] = pool_key(dd[r], ir[r]);
          }
        } else {
          const float dd = team8_dist_q<NR>(qs, X, ld, ir, vr, tl);
          const int t = t0 + TEAMS * team8_row<NR>(tl) + team;
          const int32_t id = t < cnt ? (int32_t)(uint32_t)newk[t] : 0;
          __syncwarp();
          if (tl < NR && t < cnt) newk[t] = pool_key(dd, id);
        }
      }
      __syncwarp();
      for (int c = 0; c < cnt; c += 32)
        S.merge(c + lane < cnt ? newk[c + lane] : KEY_NONE, tmp);
      __syncwarp();
    }
    for (int t = lane; t < ldo; t += 32) {
      const bool v = t < S.s && t < kq;
      out_ids[qi * ldo + t] = v ? pool_id_of(pool[t]) : -1;
      if (out_d2) out_d2[qi * ldo + t] = v ? key_dist(pool[t]) : __int_as_float(0x7f800000);
    }
    if (work && lane == 0) {
      atomicAdd(work, w_exp);
      atomicAdd(work + 1, w_dist);
      atomicAdd(work + 2, w_adj);
    }
    __syncwarp();
  }
}

// Four values (one 16-byte load, one 4-byte store) per thread and step; rows are zero from d
// to ld.  1M x 128: 0.09 ms, 0.26 ms with one value per thread.
__global__ void k_rows_u8(const float4* __restrict__ X, int64_t n4, uchar4* __restrict__ out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n4;
       e += (int64_t)gridDim.x * blockDim.x) {
    const float4 v = __ldg(X + e);
    out[e] = make_uchar4((uint8_t)__float2uint_rn(v.x), (uint8_t)__float2uint_rn(v.y),
                         (uint8_t)__float2uint_rn(v.z), (uint8_t)__float2uint_rn(v.w));
  }
}

void rows_to_u8(const float* X, int ld, int64_t n, uint8_t* out, cudaStream_t st) {
  const int64_t n4 = n * ld / 4;
  SSG_LAUNCH(k_rows_u8, (unsigned)std::min<int64_t>(ceil_div(n4, 256), 16 * num_sms()), 256, 0, st,
             (const float4*)X, n4, (uchar4*)out);
}

// A launch of k_search<T, NR, MIN_BLOCKS, WORDS>: warps per block, shared memory, blocks per SM.
struct SearchPlan {
  SearchLayout lay;
  int wpb, per_sm;
  size_t smem;
  int warps() const { return wpb * per_sm; }  // per SM
};

// ls: the pool size, or the largest one of qls.  Warps per block: eight, fewer where there are
// too few queries to give every SM a block of eight (a query alone on an SM runs without the
// others' instructions in its way).
template <typename T, int NR, int MIN_BLOCKS, bool WORDS = false>
static SearchPlan plan_rows(int ld, int R, int64_t nq, int ls, int log2h, bool work) {
  const void* kernel = (const void*)k_search<T, NR, MIN_BLOCKS, WORDS>;
  SearchPlan p;
  p.lay.Ls = (ls + 1) & ~1;
  p.lay.RP = (R + 31) & ~31;
  p.lay.ld = ld;
  p.lay.qb = std::is_same<T, uint8_t>::value ? (ld + 15) & ~15 : 0;
  p.lay.log2h = log2h;
  p.wpb = work ? 2 : 8;
  p.wpb = (int)std::min<int64_t>(p.wpb, std::max<int64_t>(1, ceil_div(nq, num_sms())));
  while (p.lay.per_warp() * p.wpb > 200 * 1024 && p.lay.log2h > 8) --p.lay.log2h;
  while (p.lay.per_warp() * p.wpb > 200 * 1024 && p.wpb > 1) p.wpb >>= 1;
  p.smem = p.lay.per_warp() * p.wpb;
  SSG_REQUIRE(p.smem <= 220 * 1024, SSG_EINVAL, "search: L_search and d too large for shared memory");
  ensure_smem(kernel, p.smem);
  p.per_sm = 0;
  SSG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p.per_sm, kernel, p.wpb * 32, p.smem));
  p.per_sm = std::max(1, p.per_sm);
  return p;
}

template <typename T, int NR, int MIN_BLOCKS, bool WORDS = false>
static void launch_rows(const SearchPlan& p, const T* X, int ld, int d, const int32_t* adj,
                        const int32_t* deg, int R, const int32_t* nav, int n_nav, const float* Q,
                        int ldq, int64_t nq, int k, int ls, const int32_t* qk, const int32_t* qls,
                        const int32_t* from, int ldo, int32_t* out_ids, float* out_d2,
                        unsigned long long* work, cudaStream_t st) {
  const int grid = (int)std::min<int64_t>(ceil_div(nq, p.wpb), (int64_t)p.per_sm * num_sms());
  SSG_LAUNCH((k_search<T, NR, MIN_BLOCKS, WORDS>), grid, p.wpb * 32, p.smem, st, X, ld, d, adj, deg, R, nav,
             n_nav, Q, ldq, nq, k, ls, qk, qls, from, ldo, p.lay, out_ids, out_d2, work);
}

static void launch_search(const uint8_t* X, int ld, int d, const int32_t* adj, const int32_t* deg,
                          int R, const int32_t* nav, int n_nav, const float* Q, int ldq, int64_t nq,
                          int k, int ls, const int32_t* qk, const int32_t* qls, const int32_t* from,
                          int ldo, int log2h, int32_t* out_ids, float* out_d2,
                          unsigned long long* work, cudaStream_t st) {
  const bool w = work != nullptr;
  if (ld & 15)
    launch_rows<uint8_t, 2, 3, true>(plan_rows<uint8_t, 2, 3, true>(ld, R, nq, ls, log2h, w), X, ld, d, adj,
                                     deg, R, nav, n_nav, Q, ldq, nq, k, ls, qk, qls, from, ldo, out_ids,
                                     out_d2, work, st);
  else
    launch_rows<uint8_t, 2, 3>(plan_rows<uint8_t, 2, 3>(ld, R, nq, ls, log2h, w), X, ld, d, adj, deg, R,
                               nav, n_nav, Q, ldq, nq, k, ls, qk, qls, from, ldo, out_ids, out_d2, work, st);
}
// Float rows: while every warp of the batch fits two blocks of eight per SM, 16 rows in flight
// per warp and 16 warps per SM; above, 8 rows and 24 warps.  50,000 x 128, us at L_search 40 and
// 200, 16 rows / 8 rows: 600 queries 217 / 245 and 923 / 1,001; 10,000 queries 709 / 723 and
// 3,834 / 3,080; 10,000 over 100,000 x 96: 588 / 462 and 2,446 / 1,832.  Between 24 and 32 queries
// per SM 32 warps of 64 registers take them all at once where shared memory lets them: 4,000
// queries, L_search 200, 50,000 x 61 and x 128 2,307 -> 1,848 and 2,111 -> 1,786, 100,000 x 96
// 1,035 -> 977.  Rows of more than 512 values that leave shared memory for no more than those 16
// warps anyway take 16 rows in flight at any batch size: 10,000 queries over 20,000 x 1,500, L_search
// 10, 1,223 -> 1,008 us, x 2,500, L_search 40, 6,239 -> 5,325 (shorter rows under large pools gain
// nothing: x 200, L_search 1,024, 23.6 / 24.1 ms).
static void launch_search(const float* X, int ld, int d, const int32_t* adj, const int32_t* deg,
                          int R, const int32_t* nav, int n_nav, const float* Q, int ldq, int64_t nq,
                          int k, int ls, const int32_t* qk, const int32_t* qls, const int32_t* from,
                          int ldo, int log2h, int32_t* out_ids, float* out_d2,
                          unsigned long long* work, cudaStream_t st) {
  const int64_t sms = num_sms();
  const bool w = work != nullptr;
  if (nq > 16 * sms) {
    const SearchPlan p3 = plan_rows<float, 2, 3>(ld, R, nq, ls, log2h, w);
    if (p3.warps() > 16 || ld <= 512) {
      if (nq > 24 * sms && nq <= 32 * sms) {
        const SearchPlan p4 = plan_rows<float, 2, 4>(ld, R, nq, ls, log2h, w);
        if (nq <= p4.warps() * sms) {
          launch_rows<float, 2, 4>(p4, X, ld, d, adj, deg, R, nav, n_nav, Q, ldq, nq, k, ls, qk, qls,
                                   from, ldo, out_ids, out_d2, work, st);
          return;
        }
      }
      launch_rows<float, 2, 3>(p3, X, ld, d, adj, deg, R, nav, n_nav, Q, ldq, nq, k, ls, qk, qls, from,
                               ldo, out_ids, out_d2, work, st);
      return;
    }
  }
  launch_rows<float, 4, 2>(plan_rows<float, 4, 2>(ld, R, nq, ls, log2h, w), X, ld, d, adj, deg, R, nav,
                           n_nav, Q, ldq, nq, k, ls, qk, qls, from, ldo, out_ids, out_d2, work, st);
}

// The sizes a call may have: those of which eight queries' (a counting call: two) pools, each twice
// and with a byte per entry, rows and smallest caches fit 220 KB.  The kernel needs less and takes
// fewer warps per block where they do not fit; the limit is the interface's.
static void require_sizes(int ls, int R, int ld, bool work) {
  const auto up16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
  const size_t per = up16((size_t)ls * 16 + up16((size_t)ls * 2) +
                          (size_t)std::max(32, next_pow2(R)) * 8 + (size_t)ld * 4 + 1024 + up16(ld));
  SSG_REQUIRE(per * (work ? 2 : 8) <= 220 * 1024, SSG_EINVAL,
              "search: L_search and d too large for shared memory");
}

// A 1,024-entry visited cache: its size only sets how often a distance is taken again, and a
// larger one costs warps per SM.
constexpr int CACHE_LOG2 = 10;

void search_run_mixed(const float* X, const uint8_t* X8, int ld, int d, const int32_t* adj,
                      const int32_t* deg, int R, const int32_t* nav, int n_nav, const float* Q,
                      int ldq, int64_t nq, const int32_t* qk, const int32_t* qls, int ls_max,
                      int ldo, int32_t* out_ids, float* out_d2, cudaStream_t st) {
  if (nq == 0) return;
  require_sizes(ls_max, R, ld, false);
  if (X8)
    launch_search(X8, ld, d, adj, deg, R, nav, n_nav, Q, ldq, nq, 0, ls_max, qk, qls, nullptr, ldo,
                  CACHE_LOG2, out_ids, out_d2, (unsigned long long*)nullptr, st);
  else
    launch_search(X, ld, d, adj, deg, R, nav, n_nav, Q, ldq, nq, 0, ls_max, qk, qls, nullptr, ldo,
                  CACHE_LOG2, out_ids, out_d2, (unsigned long long*)nullptr, st);
}

void search_run(const float* X, const uint8_t* X8, int ld, int d, int64_t n, const int32_t* adj,
                const int32_t* deg, int R, const int32_t* nav, int n_nav, const float* Q,
                int ldq, int64_t nq, int k, int Ls, int32_t* out_ids, float* out_d2,
                cudaStream_t st, unsigned long long* work) {
  (void)n;
  if (nq == 0) return;
  require_sizes(Ls, R, ld, work != nullptr);
  // a call that counts the work takes a 16,384-entry cache, so that its distance count is
  // Alg. 1's (each node once) and not inflated by recomputations after cache evictions
  const int log2h = work ? 14 : CACHE_LOG2;
  if (X8)
    launch_search(X8, ld, d, adj, deg, R, nav, n_nav, Q, ldq, nq, k, Ls, (const int32_t*)nullptr,
                  (const int32_t*)nullptr, nullptr, k, log2h, out_ids, out_d2, work, st);
  else
    launch_search(X, ld, d, adj, deg, R, nav, n_nav, Q, ldq, nq, k, Ls, (const int32_t*)nullptr,
                  (const int32_t*)nullptr, nullptr, k, log2h, out_ids, out_d2, work, st);
}

bool search_from(const float* X, int ld, int d, const int32_t* adj, const int32_t* deg, int R,
                 const int32_t* from, const float* Q, int ldq, int64_t nq, int Ls, int32_t* out_ids,
                 cudaStream_t st) {
  SearchLayout lay;
  lay.Ls = Ls + 1;
  lay.RP = (R + 31) & ~31;
  lay.ld = ld;
  lay.qb = 0;
  lay.log2h = 8;
  if (lay.per_warp() > 200 * 1024) return false;
  launch_search(X, ld, d, adj, deg, R, from, 1, Q, ldq, nq, 1, Ls, (const int32_t*)nullptr,
                (const int32_t*)nullptr, from, 1, CACHE_LOG2, out_ids, (float*)nullptr,
                (unsigned long long*)nullptr, st);
  return true;
}

}  // namespace ssg
