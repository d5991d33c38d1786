// Tiles of 64 rows: which rows of which sequence a thread block of a tile grid works on, the gates of
// one channel, and the cumulative decays within a tile with its cut into chunks.  Shared by the kernels
// that prepare gated operands tile by tile.
#pragma once

#include "ddts_common.cuh"
#include "ddts_tc_ptx.cuh"

namespace ddts {
namespace {

constexpr int kTile = 64;               // rows of a tile, and of a chunk unless decays are strong
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLg2Ln2 = -0.5287663729448977f;   // log2(ln 2)
constexpr float kRange2 = 60.f * kLog2e;          // largest decay range of a chunk, log2 units

// The tile of one (head, slot): packed sequences take slots floor(start / 64) + n ... , which are
// disjoint for consecutive sequences; a slot may belong to none.
struct TileRef {
  int n, t, nr;            // sequence, tile of the sequence, live rows (0: no such tile)
  int len;                 // rows of the sequence
  long long row0;          // first row of the tile
};
struct TileGeometry {
  const int32_t* cu;       // packed sequences, or nullptr
  int n_seq, T;
  int div;                 // dense: heads per sequence in the grid's first index
};

__device__ __forceinline__ void seq_range(const int32_t* cu, int n, int T, int& lo, int& hi) {
  lo = cu[n];
  hi = cu[n + 1];
  lo = lo < 0 ? 0 : (lo > T ? T : lo);
  hi = hi < lo ? lo : (hi > T ? T : hi);
}

// Block-wide: every one of the block's THREADS threads takes part.
template <int THREADS>
__device__ __forceinline__ TileRef find_tile(const TileGeometry& a, int head, int local) {
  TileRef r;
  if (!a.cu) {
    r.n = head / a.div;
    r.t = local;
    r.len = a.T;
    r.nr = min(kTile, a.T - r.t * kTile);
    r.row0 = (long long)head * a.T + (long long)r.t * kTile;
    return r;
  }
  // the last sequence whose first slot is not beyond this one
  r.n = last_that_holds<THREADS>(a.n_seq, [&](int n) {
    int lo, hi;
    seq_range(a.cu, n, a.T, lo, hi);
    return lo / kTile + n <= local;
  });
  __shared__ int s_found;      // (through shared memory the kernels spill fewer registers)
  if (threadIdx.x == 0) s_found = r.n;
  __syncthreads();
  r.n = *(volatile int*)&s_found;
  r.nr = 0;
  if (r.n < 0) return r;
  int lo, hi;
  seq_range(a.cu, r.n, a.T, lo, hi);
  r.t = local - (lo / kTile + r.n);
  r.len = hi - lo;
  r.row0 = (long long)head * a.T + lo + (long long)r.t * kTile;
  if (r.t >= 0) r.nr = min(kTile, r.len - r.t * kTile);      // (negative only for a bad cu_seqlens)
  return r;
}

__device__ __forceinline__ float2 unpack_bf16(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
// hi + lo = x to 16 bits of mantissa, both bf16; packed for two values.
__device__ __forceinline__ void split_bf16(float x, float y, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16(x, y);
  const float2 h = unpack_bf16(hi);
  lo = pack_bf16(x - h.x, y - h.y);
}

// Everything the gates need of one channel (Eq. "alpha_def"), hardware exponential / logarithm
// approximations (relative error about 2^-21, far inside the rounding of bf16 results) with the
// places where they would lose digits written out.
struct Gate {
  float g2;        // softplus(x) * log2(e)
  float e, r;      // e^-|x|, 1 / (1 + e)
  float tau;
  float la2, lh2;  // log2 alpha (not below -kRange2), log2 ahat
};
__device__ __forceinline__ Gate gate_of(float x, float y, int ingate) {
  Gate o;
  o.e = ex2f(-fabsf(x) * kLog2e);
  const float l1p2 = o.e < 9.765625e-4f ? o.e * fmaf(-0.72134752f, o.e, kLog2e) : lg2f(1.f + o.e);
  o.g2 = fmaf(fmaxf(x, 0.f), kLog2e, l1p2);
  o.tau = rcpf(1.f + ex2f(-y * kLog2e));
  o.la2 = fmaxf(-o.g2 * o.tau, -kRange2);
  if (ingate == RODIMUS_INGATE_POW_G) {
    const float lg = x < -8.f ? fmaf(-0.5f, o.e, x) * kLog2e : lg2f(o.g2) + kLg2Ln2;
    o.lh2 = o.tau * lg;
  } else {
    o.lh2 = -o.tau * fmaf(fmaxf(-x, 0.f), kLog2e, l1p2);
  }
  return o;
}

// Row r's chunk: the last set bit of the mask at or before r.
__device__ __forceinline__ int chunk_start(unsigned long long mask, int r) {
  return 63 - __clzll((long long)(mask & (~0ull >> (63 - r))));
}
// one past the chunk's last row
__device__ __forceinline__ int chunk_end(unsigned long long mask, int r, int nr) {
  const unsigned long long later = r == 63 ? 0ull : mask & (~0ull << (r + 1));
  return later ? __ffsll((long long)later) - 1 : nr;
}

// A sum of up to 64 decays (log2, none below -kRange2) without rounding: multiples of 2^-10, whose sums fit
// 24 bits, and the rest, whose sums stay below 2^-5.
struct ExactSum {
  float h, l;
};
struct __align__(16) ExactSum2 {
  ExactSum x, y;
};
__device__ __forceinline__ float sum1(float a, float b) { return a + b; }
__device__ __forceinline__ ExactSum sum1(ExactSum a, ExactSum b) {
  const float2 r = __fadd2_rn(make_float2(a.h, a.l), make_float2(b.h, b.l));
  return {r.x, r.y};
}
__device__ __forceinline__ float2 sum2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ ExactSum2 sum2(ExactSum2 a, ExactSum2 b) { return {sum1(a.x, b.x), sum1(a.y, b.y)}; }
__device__ __forceinline__ bool beyond_range(float s) { return s < -kRange2; }
__device__ __forceinline__ bool beyond_range(ExactSum s) { return s.h + s.l < -kRange2; }

// Cumulative decay (log2) since the chunk's start, in place, for ROWS rows of two of the CTA's CH
// channels; v holds the rows' own log2 decays on entry.  `part` is a [kTile / ROWS][CH] tile,
// `la` a [kTile][CH] one that is used only where a tile has several chunks; la_of(i) then gives row i's
// own decays again.  Returns the tile's chunk mask: the given one or, when MAKE_MASK, the one it
// determines (dyadic blocks whose decay exceeds the range in some channel are cut in the middle).
// V: two channels' decays as S each, float or ExactSum.
template <int ROWS, int CH, bool MAKE_MASK, typename V, typename S, typename LaOf>
__device__ __forceinline__ unsigned long long tile_scan(V (&v)[ROWS], int cp, int rg, int nr, S* la, S* part,
                                                        unsigned long long* s_mask, unsigned long long mask, LaOf la_of) {
  constexpr int kGroups = kTile / ROWS;
#pragma unroll
  for (int i = 1; i < ROWS; ++i) v[i] = sum2(v[i], v[i - 1]);
  *reinterpret_cast<V*>(part + rg * CH + 2 * cp) = v[ROWS - 1];
  __syncthreads();
  V pre = {}, all = {};                        // of the row groups before this one, of the tile
  bool mine = true;                            // this thread knows `all`
  if constexpr (sizeof(V) == 8) {
#pragma unroll
    for (int w = 0; w < kGroups; ++w) {
      if (w == rg) pre = all;
      all = sum2(all, *reinterpret_cast<const V*>(part + w * CH + 2 * cp));
    }
  } else {                                     // (exact sums are twice as long: no more are read than needed)
#pragma unroll
    for (int w = 0; w < kGroups - 1; ++w)
      if (w < rg) pre = sum2(pre, *reinterpret_cast<const V*>(part + w * CH + 2 * cp));
    all = sum2(pre, v[ROWS - 1]);
    mine = rg == kGroups - 1;
  }
  bool whole;
  if (MAKE_MASK) {
    whole = __syncthreads_or(mine && (beyond_range(all.x) || beyond_range(all.y))) == 0;
    mask = 1ull;
  } else {
    whole = mask == 1ull;
  }
  if (whole) {
#pragma unroll
    for (int i = 0; i < ROWS; ++i) v[i] = sum2(v[i], pre);
    return mask;
  }
  // ---- rare: several chunks in the tile
#pragma unroll 1
  for (int i = 0; i < ROWS; ++i) *reinterpret_cast<V*>(la + (rg * ROWS + i) * CH + 2 * cp) = la_of(i);
  if (MAKE_MASK) {
    if (threadIdx.x == 0) *s_mask = 1ull;
    __syncthreads();
    for (int d = threadIdx.x; d < CH; d += blockDim.x) {
      unsigned long long m = 0ull;
#pragma unroll 1
      for (int len = kTile; len >= 2; len >>= 1)
#pragma unroll 1
        for (int r0 = 0; r0 < nr; r0 += len) {
          S s = {};
          for (int r = r0; r < min(r0 + len, nr); ++r) s = sum1(s, la[r * CH + d]);
          if (beyond_range(s) && r0 + len / 2 < nr) m |= 1ull << (r0 + len / 2);
        }
      if (m) atomicOr(s_mask, m);
    }
    __syncthreads();
    mask = *s_mask;
  } else {
    __syncthreads();
  }
#pragma unroll 1
  for (int i = 0; i < ROWS; ++i) {
    const int r = rg * ROWS + i;
    V acc = {};
    if (r < nr) {
      for (int j = chunk_start(mask, r); j <= r; ++j) {
        acc.x = sum1(acc.x, la[j * CH + 2 * cp]);
        acc.y = sum1(acc.y, la[j * CH + 2 * cp + 1]);
      }
    }
#pragma unroll
    for (int u = 0; u < ROWS; ++u)
      if (u == i) v[u] = acc;
  }
  __syncthreads();                            // `la` is the caller's again, whatever the mask
  return mask;
}

}  // namespace
}  // namespace ddts
