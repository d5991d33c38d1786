// Backward pass of the chunked prefill for bf16 tokens on the 5th-generation tensor cores:
// gradients with respect to q, k, x, y, v and the initial state, given dL/do and dL/dS_T.
//
// Adjoint of the chunkwise form (appendix "Chunkwise Parallel Representation of the Rodimus
// Block"), chunk length 64, per chunk with b_r = sum_{j<=r in chunk} log alpha_j, D = e^{b_C}:
//   Qe_r = scale q_r e^{b_r}     Ki_i = ahat_i k_i e^{-b_i}
//   dA_ri = do_r . v_i,  A_ri = Qe_r . Ki_i                                    (i <= r)
//   forward sweep:  raw_q_r = S do_r + sum_{i<=r} dA_ri Ki_i       S <- D . (S + Ki^T V)
//   reverse sweep:  G' = D . G      raw_k_i = G' v_i + sum_{r>=i} dA_ri Qe_r
//                   dv_i = Ki_i G' + sum_{r>=i} A_ri do_r          G <- G' + Qe^T dO
//   dL/d(scale q_r) = e^{b_r} . raw_q_r          dL/d(ahat k)_i = e^{-b_i} . raw_k_i
// and the gates from suffix sums of u = q . dq and w = (ahat k) . d(ahat k): every pair (r,i)
// with i < t <= r appears once in the sum of u and never in that of w,
//   dL/dlog alpha_t = sum_{s>=t} (u_s - w_s) + sum_j dS_T[.,j] S_T[.,j].
//
// Three launches.
//   ddts_bwd_pre_kernel    a CTA per 64-row tile: gates, cumulative decays, Qe and Ki as pairs of
//                          bf16 (high and low part, 16 bits of mantissa together), chunk decays.
//                          Where a tile decays by more than e^-60 in some channel it is cut in
//                          halves until every chunk fits (down to single rows, which always fit
//                          because a step's decay is applied as at least e^-60).
//   ddts_bwd_sweep_tc_kernel  the three serial scans per (sequence, head) (raw_q; raw_k; dv), each
//                          optionally cut into time segments that hand their state on.  No gate
//                          arithmetic: every operand arrives by TMA in the form the tensor core
//                          reads, which leaves a sweep bound by its contractions.
//   ddts_bwd_post_kernel   a CTA per tile from the last to the first: scales raw_q, raw_k, suffix
//                          sums chained from tile to tile (fp64), dq, dk, dx, dy.
// What this replaces for bf16 - one launch of 16-row chunks on mma.sync with the gates computed in
// each of six CTAs per (sequence, head), bound by instruction issue - took 1.79 ms on the layer
// shape (B=4 H=16 T=2048); this takes 0.34 ms there (0.35 run for seconds): 52 us (4.1 TB/s; issue slots 70 % busy) + 170 us
// (shared memory, see the sweeps) + 120 us (3.3 TB/s; issue slots 50 %, special-function units 41 %, the
// rest latency: 18 warps on an SM on average, a third of their stalls waiting for loads).
#include <cuda.h>

#include <cstring>

#include "ddts_common.cuh"
#include "ddts_tc_ptx.cuh"
#include "ddts_tiles.cuh"

namespace ddts {
namespace {

constexpr int DK = 128, DV = 256;       // the widths these kernels are built for

struct BwdTcArgs {
  const __nv_bfloat16 *q, *k, *gx, *ty;
  const float *s0, *dsT;
  __nv_bfloat16 *dq, *dk, *dx, *dy, *dv;
  float* ds0;
  // The operands Qe, Ki live in the OUTPUT buffers until the last kernel writes the gradients there:
  // high and low parts, [rows][DK] bf16 each (Qe in d_q, d_k; Ki in d_gate_x, d_temp_y).
  uint32_t *qe_hi, *qe_lo, *ki_hi, *ki_lo;
  // scratch
  float* dtile;               // [slots][DK]: decay of the whole tile (tiles that are one chunk)
  unsigned long long* mask;   // [slots]: bit r = row r of the tile starts a chunk
  float *raw_q, *raw_k;       // [rows][DK]; within a tile [groups of 8 rows][DK][rows of the group]
  int32_t* tile_flag;         // [slots][4]: suffix sums of this tile and 32 channels are there
  int2* tile_order;           // packed: (sequence, tile) of every head's tiles as the last kernel takes them
  float *c, *c2;              // [n_seq * H][DK]: the constant of the suffix sums, in two halves
  float* seg_state;           // [n_seq * H * 3][32][256] of 16 bytes: state of a sweep cut in two, at the
                              // cut, as the 256 threads of the state group hold it
  int32_t* seg_flag;          // [n_seq * H * 3]: 8 when that state is there; then the ticket counter
  const int32_t *cu, *order;
  WorkspaceHeader* hdr;
  long long n_flags;          // entries of seg_flag with the counter
  int H, T, n_seq;
  int heads;                  // tile grids: (batch, head) pairs of a dense call, heads of a packed one
  int slots_per_head;
  float scale;
  int ingate;
  long long limit;
};
__device__ __forceinline__ TileGeometry geometry(const BwdTcArgs& a) { return {a.cu, a.n_seq, a.T, a.cu ? 1 : a.H}; }

__device__ __forceinline__ int32_t ld_acquire_s32(const int32_t* p) {
  int32_t v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_s32(int32_t* p, int32_t v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_release_add(int32_t* p, int32_t v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---------------------------------------------------------------------------------------------
// Gates and operands of one tile
// ---------------------------------------------------------------------------------------------
constexpr int kPreThreads = 512, kPreRows = kTile / (kPreThreads / 64);   // 8 rows x 2 channels a thread

// Packed sequences: the order in which the last kernel takes a head's tiles.  The tiles of a sequence are
// chained from its end, a hop being about 2 us; with the sequences one after another the chain runs through
// all of them, so the order is: the last tile of every sequence, then the last but one of all that have
// one, and so on (sequences longest first, so those are a prefix of the list).  Block-wide.
__device__ void order_tiles(const BwdTcArgs& a, int* s_nt, int* s_scan) {
  const int tid = threadIdx.x, N = a.n_seq;
  auto tiles_of = [&](int n) {
    int lo, hi;
    seq_range(a.cu, n, a.T, lo, hi);
    return (hi - lo + kTile - 1) / kTile;
  };
  if (N > kMaxSortedSeqs) {   // not sorted: sequence after sequence, from the last one's end
    for (int pos = tid; pos < a.slots_per_head; pos += kPreThreads) a.tile_order[pos] = make_int2(-1, 0);
    __syncthreads();
    for (int n = tid; n < N; n += kPreThreads) {
      int lo, hi;
      seq_range(a.cu, n, a.T, lo, hi);
      for (int t = 0, nt = tiles_of(n); t < nt; ++t)
        a.tile_order[a.slots_per_head - 1 - (lo / kTile + n + t)] = make_int2(n, t);
    }
    return;
  }
  for (int j = tid; j < N; j += kPreThreads) s_nt[j] = tiles_of(a.order[j]);
  __syncthreads();
  const int most = s_nt[0];
  int at = 0;                 // tiles before this batch of kPreThreads ranks
  for (int r0 = 0; r0 < most; r0 += kPreThreads) {
    int cnt = 0;              // sequences with more than r tiles
    const int r = r0 + tid;
    if (r < most) {
      int hi = N;
      while (cnt < hi) {
        const int mid = (cnt + hi) >> 1;
        if (s_nt[mid] > r) cnt = mid + 1;
        else hi = mid;
      }
    }
    s_scan[tid] = cnt;
    __syncthreads();
    for (int d = 1; d < kPreThreads; d <<= 1) {
      const int v = tid >= d ? s_scan[tid - d] : 0;
      __syncthreads();
      s_scan[tid] += v;
      __syncthreads();
    }
    // a warp per rank: its sequences, the first s_scan[i] - s_scan[i - 1] of the list, lie side by side
    for (int i = tid >> 5; i < min(kPreThreads, most - r0); i += kPreThreads / 32) {
      const int before = i > 0 ? s_scan[i - 1] : 0, n = s_scan[i] - before;
      for (int j = tid & 31; j < n; j += 32) a.tile_order[at + before + j] = make_int2(a.order[j], s_nt[j] - 1 - (r0 + i));
    }
    at += s_scan[kPreThreads - 1];
    __syncthreads();
  }
  for (int pos = at + tid; pos < a.slots_per_head; pos += kPreThreads) a.tile_order[pos] = make_int2(-1, 0);
}

__global__ void __launch_bounds__(kPreThreads, 2) ddts_bwd_pre_kernel(const BwdTcArgs a) {
  __shared__ __align__(16) float s_la[kTile * DK];
  __shared__ __align__(16) float s_part[(kTile / kPreRows) * DK];
  __shared__ unsigned long long s_mask;
  const int tid = threadIdx.x;
  if (blockIdx.x == 0 && tid == 0 && !a.cu) a.hdr->status = RODIMUS_OK;
  for (long long i = (long long)blockIdx.x * kPreThreads + tid; i < a.n_flags; i += (long long)gridDim.x * kPreThreads)
    a.seg_flag[i] = 0;
  if (a.cu && blockIdx.x == gridDim.x - 1) {   // one block more than there are slots
    wait_for_previous_kernel();
    // (ranges of a refused cu_seqlens may overlap: there is no bound on their tiles, and nobody reads the order)
    if (*(volatile int32_t*)&a.hdr->status == RODIMUS_ERR_SEQLENS) return;
    order_tiles(a, reinterpret_cast<int*>(s_la), reinterpret_cast<int*>(s_part));
    return;
  }
  const int head = (int)(blockIdx.x / (unsigned)a.slots_per_head), local = (int)(blockIdx.x % (unsigned)a.slots_per_head);
  const TileRef tr = find_tile<kPreThreads>(geometry(a), head, local);
  const long long slot = (long long)head * a.slots_per_head + local;
  if (tid < 4) a.tile_flag[slot * 4 + tid] = 0;
  if (tr.nr <= 0) return;
  const int cp = tid & 63, rg = tid >> 6;
  const int live = tr.nr - rg * kPreRows;                  // rows of this thread that exist
  const long long e0 = (tr.row0 + rg * kPreRows) * 64 + cp;
  const uint32_t* gx = reinterpret_cast<const uint32_t*>(a.gx) + e0;
  const uint32_t* ty = reinterpret_cast<const uint32_t*>(a.ty) + e0;
  const uint32_t* q = reinterpret_cast<const uint32_t*>(a.q) + e0;
  const uint32_t* k = reinterpret_cast<const uint32_t*>(a.k) + e0;
  uint32_t wx[kPreRows], wy[kPreRows], wq[kPreRows], wk[kPreRows];
#pragma unroll
  for (int i = 0; i < kPreRows; ++i) {
    wx[i] = wy[i] = wq[i] = wk[i] = 0u;
    if (i < live) {
      wx[i] = __ldg(gx + i * 64);
      wy[i] = __ldg(ty + i * 64);
      wq[i] = __ldg(q + i * 64);
      wk[i] = __ldg(k + i * 64);
    }
  }
  float2 b[kPreRows], lh2[kPreRows];
#pragma unroll
  for (int i = 0; i < kPreRows; ++i) {
    const float2 x = unpack_bf16(wx[i]), y = unpack_bf16(wy[i]);
    const Gate g0 = gate_of(x.x, y.x, a.ingate), g1 = gate_of(x.y, y.y, a.ingate);
    b[i] = i < live ? make_float2(g0.la2, g1.la2) : make_float2(0.f, 0.f);
    lh2[i] = make_float2(g0.lh2, g1.lh2);
  }
  auto la_of = [&](int i) {
    if (i >= live) return make_float2(0.f, 0.f);
    const float2 x = unpack_bf16(__ldg(gx + i * 64)), y = unpack_bf16(__ldg(ty + i * 64));
    return make_float2(gate_of(x.x, y.x, a.ingate).la2, gate_of(x.y, y.y, a.ingate).la2);
  };
  const unsigned long long mask = tile_scan<kPreRows, DK, true>(b, cp, rg, tr.nr, s_la, s_part, &s_mask, 0ull, la_of);
  if (tid == 0) a.mask[slot] = mask;
#pragma unroll
  for (int i = 0; i < kPreRows; ++i) {
    if (i < live) {
      const float2 qv = unpack_bf16(wq[i]), kv = unpack_bf16(wk[i]);
      const float ex = ex2f(b[i].x), ey = ex2f(b[i].y);
      uint32_t hi, lo;
      split_bf16(qv.x * a.scale * ex, qv.y * a.scale * ey, hi, lo);
      a.qe_hi[e0 + i * 64] = hi;
      a.qe_lo[e0 + i * 64] = lo;
      split_bf16(kv.x * ex2f(lh2[i].x - b[i].x), kv.y * ex2f(lh2[i].y - b[i].y), hi, lo);
      a.ki_hi[e0 + i * 64] = hi;
      a.ki_lo[e0 + i * 64] = lo;
      if (i + 1 == live || (i + 1 == kPreRows && rg * kPreRows + i + 1 == tr.nr))
        *reinterpret_cast<float2*>(a.dtile + slot * DK + 2 * cp) = make_float2(ex, ey);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// The sweeps
// ---------------------------------------------------------------------------------------------
// A persistent CTA per SM, 20 warps, takes pieces of sweeps one after another (see get_piece); barriers
// and chunk counters run on from piece to piece, so that the next piece's tiles are on their way while
// the last one ends.  The three sweeps share one skeleton:
// with operand tiles X, Y, P (64 rows of 512 bytes each) and a state of 256 tensor-memory columns,
//               X      Y      P        state                       results
//   raw_q       V      dO     Ki       S  [lane = key channel]     raw_q^T  [channel][row]
//   raw_k       dO     V      Qe       G' [lane = key channel]     raw_k^T  [channel][row]
//   dv          Qe     Ki     dO       G'^T, two blocks of 128     dv^T     [value column][row],
//                                      lanes (value columns)                 two blocks
// a chunk is
//   M0  T   = Y X^T                  [64 x 64]; then masked and split into bf16 pairs by warps
//   M1  O   = state Y32^T            A = the fp32 state in TENSOR MEMORY (tf32), B = Y as fp32
//   M2  state += P^T X               in place, fp32
//   M3  O  += P^T T^T
// Nothing of the state goes through shared memory; once per chunk it makes a trip through registers
// to be scaled by the chunk decay D (forward: after the update; reverse: before the use).
// Precision: V and dO are exact; Qe, Ki and T are bf16 pairs (products of two pairs drop low x low,
// 2^-16); the state is read as tf32 by M1 and kept in fp32.
// The issue order is M1 M0 M2 M3: the chain of the state is M1, M0, M2, then its trip, during which M3
// runs and Y of the next chunk, which has two buffers, is expanded.  (With M0 of the next chunk at the
// end, X in two buffers and Y in one, the layer shape took 361 us a call, so 354.)
// What bounds it: about 500 KiB go through shared memory per chunk (M0 64, M1 64, M2 96, M3 72, expanding
// Y 96, tiles in 96, T 16), 3900 cycles at 128 bytes a clock; a chunk takes 6000, a 32 KiB tile 3000 to
// 4000 cycles to arrive although it comes from L2 (prefetching it there changes nothing).
constexpr int kSlab = kTile * 128;                 // [64 rows][128 bytes], 128-byte swizzled
constexpr int kOpBytes = 4 * kSlab;                // X, Y (two buffers), P: 32 KiB each
constexpr int kOffX = 0, kOffY = kOpBytes, kOffP = 3 * kOpBytes, kOffY32 = 4 * kOpBytes;
constexpr int kOffT = kOffY32 + 2 * kOpBytes;      // T: high and low parts, 8 KiB each
constexpr int kOffOut = kOffY32 + kOpBytes;        // dv only (its Y32 is half as large): output tile
constexpr int kOffD = kOffT + 2 * kSlab;           // float [4][DK]: chunk decays, per chunk (c & 3)
constexpr int kOffBar = kOffD + 4 * DK * 4;
constexpr int kSwBars = 32;
constexpr int kOffCtl = kOffBar + kSwBars * 8;
constexpr int kSwSmemUsed = kOffCtl + 256;
constexpr int kSwSmem = kSwSmemUsed + 1024;        // slack for 1024-byte alignment
static_assert(kSwSmem <= 232448, "shared memory budget");
constexpr int kSwThreads = 640;
constexpr uint32_t kColS = 0, kColO = 256, kColT = 384, kSwTmemCols = 512;

enum { SB_DESC0 = 0,                       // [4] descriptor and decays of a chunk      (1 + bytes)
       SB_FX = 4, SB_FY0, SB_FY1, SB_FP,   // tiles landed                              (1 + bytes)
       SB_EX, SB_EP,                       // tile reusable: its contractions are done  (1)
       SB_EY0, SB_EY1,                     // Y reusable: M0 done, expanded             (1 + 8 warps)
       SB_TFULL, SB_TREADY,                // T computed (1), masked into shared memory (4 warps)
       SB_M1, SB_UFULL,                    // M1 / M2 complete                          (1)
       SB_SREADY,                          // state scaled, Y32 written                 (8 warps)
       SB_OFULL0, SB_OFULL1,               // results complete                          (1)
       SB_OFREE0, SB_OFREE1,               // results read                              (4 warps)
       SB_DRDY,                            // decays of a chunk of a cut tile computed           (4 warps)
       SB_OTFULL,                          // dv output tile written                    (4 warps)
       SB_OTFREE0, SB_OTFREE1,             // dv output tile read by its copies         (1); two barriers in turn:
                                           // the state group may ask for a tile while the one before is out
       SB_TICKET0, SB_TICKET1,             // a ticket is in its slot                   (1)
       SB_TKFREE0, SB_TKFREE1,             // every warp has read it                    (20 warps)
       SB_DRAIN, SB_COUNT };
static_assert(SB_COUNT <= kSwBars, "barrier count");

struct ChunkDesc {
  long long row;     // first row of the chunk
  int nr;            // rows
  int roff;          // first row within the tile
  int nr_tile;       // rows of the tile
  int flags;         // kLast, kWhole
};
constexpr int kLast = 1, kWhole = 2;   // last chunk of the piece; the tile is one chunk
struct SwCtl {
  uint32_t tmem_base;
  int pad;
  WaitCtl wait;
  int n_x, n_y, n_p, n_d;    // loads issued (for the clean exit)
  uint32_t ticket[2];        // of the next piece (packed calls)
  ChunkDesc desc[4];
};
static_assert(sizeof(SwCtl) <= 256, "control block");

__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D += A B, both operands in shared memory, bf16
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\n.reg .b64 da, db;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "mov.b64 da, {%1, %5};\nmov.b64 db, {%2, %5};\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(acc), "r"(kDescHi) : "memory");
}
// D += A B with A [128 lanes x 8 columns] fp32 in tensor memory read as tf32, B [N rows][8] K-major fp32.
__device__ __forceinline__ void umma_tf32_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc,
                                             uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\n.reg .b64 db;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "mov.b64 db, {%2, %5};\n"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], db, %3, p;\n}"
      ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(acc), "r"(kDescHi) : "memory");
}
__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

struct SweepMaps {
  CUtensorMap v, dout, qe_hi, qe_lo, ki_hi, ki_lo, dv, dv8, dv1;
};

// A piece of a sweep: its tiles i_lo .. i_hi-1, counted in the order of the sweep.
struct Piece {
  int kind, n, h;
  int i_lo, i_hi;
  bool wait, hand;   // the state comes from the piece before / goes to the piece after
};

// The k-th piece of CTA `cta` of `ctas`.  Sweeps are numbered from the longest kind to the shortest.
// Dense calls have sweeps of equal length: laid end to end, each CTA takes an equal share of the tiles,
// so a sweep may be cut in two (never in three: there are no more CTAs than sweeps).  A CTA takes the
// beginning of its last sweep first, so that the CTA after it has the state it needs, then its whole
// sweeps, then the end of the sweep that the CTA before it (lower index: running or done) has begun.
// Layer shape, 192 sweeps of 32 tiles on 148 SMs: 42 tiles each; as 576 CTAs of a third of a sweep, four
// rounds of set-up and state hand-over, the launch took 215 us.
// Packed calls: whole sweeps, drawn as tickets from the longest sequence to the shortest, the costlier
// kinds first; the first ticket is the CTA's index.  (Dealt back and forth instead, 7 sequences of 50 to
// 600 tokens, 16 heads: the CTAs end after 143 us, 100 on average; a raw_q or raw_k sweep takes 5 us a
// tile there, a dv sweep 3.)
template <bool VARLEN>
__device__ __forceinline__ bool get_piece(const BwdTcArgs& a, int cta, int ctas, int k, uint32_t ticket, Piece& p) {
  const int items = a.n_seq * a.H, sweeps = 3 * items, nt = VARLEN ? 0 : (a.T + kTile - 1) / kTile;
  p.wait = p.hand = false;
  int s;
  if (nt == 0) {
    const long long at = VARLEN ? (long long)ticket : (long long)k * ctas + cta;
    if (at >= sweeps) return false;
    const int of = 3 * a.H, rem = (int)(at % of);
    p.kind = rem / a.H;
    p.h = rem % a.H;
    p.n = (int)(at / of);
    p.i_lo = p.i_hi = 0;
    if (VARLEN) {
      p.n = a.order[p.n];
      int lo, hi;
      seq_range(a.cu, p.n, a.T, lo, hi);
      p.i_hi = (hi - lo + kTile - 1) / kTile;
    }
    return true;
  }
  const long long total = (long long)sweeps * nt, lo = total * cta / ctas, hi = total * (cta + 1) / ctas;
  const int s_lo = (int)(lo / nt), r_lo = (int)(lo % nt), s_hi = (int)(hi / nt), r_hi = (int)(hi % nt);
  const int first = s_lo + (r_lo > 0), n_head = r_hi > 0 ? 1 : 0;
  if (k < n_head) {                                   // beginning of the last sweep
    s = s_hi;
    p.i_lo = 0;
    p.i_hi = r_hi;
    p.hand = true;
  } else if (k - n_head < s_hi - first) {             // a whole one
    s = first + k - n_head;
    p.i_lo = 0;
    p.i_hi = nt;
  } else if (k - n_head == s_hi - first && r_lo > 0) {   // end of the first one
    s = s_lo;
    p.i_lo = r_lo;
    p.i_hi = nt;
    p.wait = true;
  } else {
    return false;
  }
  p.kind = 2 - s / items;
  p.n = s % items / a.H;
  p.h = s % items % a.H;
  return true;
}

// What a thread carries from piece to piece: the number of the next chunk, chunks of cut tiles and dv
// output tiles so far, and whether every wait has been satisfied.
struct Carry {
  int c, n_cut, n_ot;
  bool ok;
};

// KIND 0: raw_q (forward), 1: raw_k, 2: dv (both reverse)
template <int KIND, bool VARLEN>
__device__ __forceinline__ void sweep_piece(const BwdTcArgs& a, const SweepMaps& maps, const Piece& pc, const uint32_t base,
                                            uint8_t* gbase, const uint32_t tmem, Carry& k) {
  constexpr bool REV = KIND != 0, DVK = KIND == 2;
  auto bar = [&](int i) { return base + kOffBar + 8u * (uint32_t)i; };
  volatile SwCtl* ctl = reinterpret_cast<volatile SwCtl*>(gbase + kOffCtl);
  volatile WaitCtl* wc = &ctl->wait;
  float* sD = reinterpret_cast<float*>(gbase + kOffD);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q4 = warp & 3;
  WorkspaceHeader* hdr = a.hdr;
  const long long sh = (long long)pc.n * a.H + pc.h;

  long long row0;
  int len, slot_base;
  if (VARLEN) {
    int lo, hi;
    seq_range(a.cu, pc.n, a.T, lo, hi);
    row0 = (long long)pc.h * a.T + lo;
    len = hi - lo;
    slot_base = pc.h * a.slots_per_head + lo / kTile + pc.n;   // of masks and decays
  } else {
    row0 = sh * a.T;
    len = a.T;
    slot_base = (int)(sh * a.slots_per_head);
  }
  const int ntiles = (len + kTile - 1) / kTile;
  const int i_lo = pc.i_lo, i_hi = pc.i_hi;
  const bool any = i_hi > i_lo;
  const int first = k.c;               // number of the piece's first chunk
  // warp-uniform bounded wait (the tensor-memory accesses need whole warps)
  auto wait_all = [&](uint32_t b, uint32_t parity) -> bool {
    return __all_sync(0xffffffffu, mbar_wait(b, parity, wc, hdr)) != 0;
  };

  if (warp == 0) {
    // ===================================== producer ========================================
    if (any && elect_one() && k.ok) {
      // a tile of four 64-column slabs: one copy, or (high and low parts) two
      struct Src { const CUtensorMap *m0, *m1; };
      const Src v = {&maps.v, nullptr}, dout = {&maps.dout, nullptr};
      const Src qe = {&maps.qe_hi, &maps.qe_lo}, ki = {&maps.ki_hi, &maps.ki_lo};
      const Src mx = KIND == 0 ? v : (KIND == 1 ? dout : qe);
      const Src my = KIND == 0 ? dout : (KIND == 1 ? v : ki);
      const Src mp = KIND == 0 ? ki : (KIND == 1 ? qe : dout);
      // chunk iterator
      int i = i_lo, t = REV ? ntiles - 1 - i : i;
      unsigned long long mask = __ldcg(a.mask + slot_base + t), mask_next = 0ull;
      int nr_tile = min(kTile, len - t * kTile);
      auto peek = [&]() {
        if (i + 1 < i_hi) mask_next = __ldcg(a.mask + slot_base + (REV ? t - 1 : t + 1));
      };
      peek();
      int r = REV ? chunk_start(mask, nr_tile - 1) : 0;   // first row of the chunk within the tile
      bool more = true;
      auto load4 = [&](uint32_t dst, const Src& m, int row, uint32_t b) {
        mbar_expect_tx(b, kOpBytes);
        tma_load_3d(dst, m.m0, 0, row, 0, b);
        if (m.m1) tma_load_3d(dst + 2 * kSlab, m.m1, 0, row, 0, b);
      };
      auto row_of = [&](int c) { return (int)ctl->desc[c & 3].row; };
      // descriptor, decays and Y tile of chunk number c
      auto start_chunk = [&](int c) -> bool {
        if (!mbar_wait(bar(SB_EY0 + (c & 1)), ((c >> 1) & 1) ^ 1, wc, hdr)) return false;
        const int end = chunk_end(mask, r, nr_tile);
        volatile ChunkDesc* d = &ctl->desc[c & 3];
        const long long row = row0 + (long long)t * kTile + r;
        d->row = row;
        d->nr = end - r;
        d->roff = r;
        d->nr_tile = nr_tile;
        const bool whole = mask == 1ull;
        const float* decays = a.dtile + (long long)(slot_base + t) * DK;
        // step to the chunk after this one
        bool last = false;
        if (!REV ? end < nr_tile : r > 0) {
          r = REV ? chunk_start(mask, r - 1) : end;
        } else if (i + 1 < i_hi) {
          ++i;
          t = REV ? t - 1 : t + 1;
          mask = mask_next;
          nr_tile = min(kTile, len - t * kTile);
          peek();
          r = REV ? chunk_start(mask, nr_tile - 1) : 0;
        } else {
          last = true;
        }
        d->flags = (last ? kLast : 0) | (whole ? kWhole : 0);
        more = !last;
        const uint32_t db = bar(SB_DESC0 + (c & 3));
        if (whole) {
          mbar_expect_tx(db, DK * 4);
          bulk_load(base + kOffD + (c & 3) * DK * 4, decays, DK * 4, db);
        } else {
          mbar_arrive(db);   // the state group computes them
        }
        ctl->n_d = c + 1;
        load4(base + kOffY + (c & 1) * kOpBytes, my, (int)row, bar(SB_FY0 + (c & 1)));
        ctl->n_y = c + 1;
        return true;
      };
      // Tiles are asked for in the order in which their buffers come free: X(c) with M2(c-1), Y(c+1) with
      // M0 and the expansion of c-1, P(c) with M3(c-1).
      bool ok = start_chunk(first);
      for (int c = first; ok; ++c) {
        k.c = c + 1;
        if (!(ok = mbar_wait(bar(SB_EX), (c & 1) ^ 1, wc, hdr))) break;
        load4(base + kOffX, mx, row_of(c), bar(SB_FX));
        ctl->n_x = c + 1;
        const bool next = more;
        if (next && !(ok = start_chunk(c + 1))) break;
        if (!(ok = mbar_wait(bar(SB_EP), (c & 1) ^ 1, wc, hdr))) break;
        load4(base + kOffP, mp, row_of(c), bar(SB_FP));
        ctl->n_p = c + 1;
        if (!next) break;
      }
      k.ok = ok;
    }
    __syncwarp();
  } else if (warp == 1) {
    // ====================================== issuer =========================================
    // Every lane walks the chunks; what is issued sits in elect_one() blocks.  (That form matters:
    // with a branch on the lane number instead an instruction costs its thread 80 to 110 cycles, here
    // 32 to 48, which is what the tensor core needs for it.)  The loops are rolled: this code runs once
    // per chunk, and what does not stay in the instruction cache is fetched anew each time.
    if (any && k.ok) {
      constexpr uint32_t kI0 = make_idesc(64, 64, 0, 0), kI1 = idesc_tf32(128, 64);
      constexpr uint32_t kI2 = DVK ? make_idesc(128, 128, 1, 1) : make_idesc(128, 256, 1, 1);
      constexpr uint32_t kI3 = make_idesc(128, 64, 1, 0);
      const uint32_t dy0 = desc_lo_kmajor(base + kOffY), dx = desc_lo_kmajor(base + kOffX);
      const uint32_t dy32 = desc_lo_kmajor(base + kOffY32), dt = desc_lo_kmajor(base + kOffT);
      const uint32_t dxm = desc_lo_mnmajor(base + kOffX, kSlab), dp = desc_lo_mnmajor(base + kOffP, kSlab);
      constexpr uint32_t kS = kSlab >> 4;              // one slab, in descriptor units
      const uint32_t t_s = tmem + kColS, t_t = tmem + kColT;
      bool ok = true;
      for (int c = first; ok; ++c) {
        k.c = c + 1;
        const uint32_t ph = c & 1;
        if (!(ok = wait_all(bar(SB_DESC0 + (c & 3)), (c >> 2) & 1))) break;
        const bool last = (ctl->desc[c & 3].flags & kLast) != 0;
        if (!(ok = wait_all(bar(SB_SREADY), ph))) break;
        // the results' columns must have been read: two buffers in turn, or (dv, and a piece's first
        // chunk, which may follow a dv piece) one
        if (!DVK && c > first) {
          if (!(ok = wait_all(bar(SB_OFREE0 + (c & 1)), ((c >> 1) & 1) ^ 1))) break;
        } else if (c > 0) {
          if (!(ok = wait_all(bar(SB_OFREE0 + ((c - 1) & 1)), ((c - 1) >> 1) & 1))) break;
        }
        tc_fence_after();
        const uint32_t o = tmem + kColO + (DVK ? 0u : ph * 64u);
        // M1
        if (elect_one()) {
#pragma unroll 1
          for (uint32_t i = 0; i < 8; ++i) {           // 32 columns of the state (dv: four per block)
            const uint32_t od = o + (DVK ? (i >> 2) * 64u : 0u), b = dy32 + (DVK ? i & 3 : i) * kS;
#pragma unroll
            for (uint32_t kk = 0; kk < 4; ++kk)
              umma_tf32_ts(od, t_s + 32 * i + 8 * kk, b + 2 * kk, kI1, (DVK ? i & 3 : i) | kk);
          }
          umma_commit(bar(SB_M1));
        }
        __syncwarp();
        if (!(ok = wait_all(bar(SB_FX), ph))) break;
        tc_fence_after();
        // M0 (Y has landed: the state group has expanded it)
        const uint32_t dy = dy0 + ph * 4 * kS;
        if (elect_one()) {
#pragma unroll 1
          for (uint32_t i = 0; i < (DVK ? 6u : 4u); ++i) {
            // dv: slab pairs (high, high), (high, low), (low, high) of the 128 channels' two slabs
            const uint32_t ya = dy + (DVK ? (i & 1) + (i >= 4 ? 2u : 0u) : i) * kS;
            const uint32_t xa = dx + (DVK ? (i & 1) + ((i >> 1) == 1 ? 2u : 0u) : i) * kS;
#pragma unroll
            for (uint32_t kk = 0; kk < 4; ++kk) umma_ss(t_t, ya + 2 * kk, xa + 2 * kk, kI0, i | kk);
          }
          umma_commit(bar(SB_TFULL));
          umma_commit(bar(SB_EY0 + ph));
        }
        __syncwarp();
        if (!(ok = wait_all(bar(SB_FP), ph))) break;
        tc_fence_after();
        // M2
        if (elect_one()) {
#pragma unroll 1
          for (uint32_t i = 0; i < (DVK ? 4u : 2u); ++i) {
            const uint32_t d = t_s + (DVK ? (i >> 1) * 128u : 0u);
            const uint32_t pa = dp + (DVK ? i & 2 : 2 * i) * kS, xa = dxm + (DVK ? (i & 1) * 2 * kS : 0u);
#pragma unroll
            for (uint32_t kk = 0; kk < 4; ++kk) umma_ss(d, pa + 128 * kk, xa + 128 * kk, kI2, 1u);
          }
          umma_commit(bar(SB_UFULL));
          umma_commit(bar(SB_EX));
        }
        __syncwarp();
        if (!(ok = wait_all(bar(SB_TREADY), ph))) break;
        tc_fence_after();
        // M3: (P high, T high), (P high, T low), (P low, T high); dv: block by T high, low
        if (elect_one()) {
#pragma unroll 1
          for (uint32_t i = 0; i < (DVK ? 4u : 3u); ++i) {
            const uint32_t od = o + (DVK ? (i >> 1) * 64u : 0u);
            const uint32_t pa = dp + (DVK ? i & 2 : (i == 2 ? 2u : 0u)) * kS;
            const uint32_t ta = dt + (DVK ? i & 1 : (i == 1 ? 1u : 0u)) * kS;
#pragma unroll
            for (uint32_t kk = 0; kk < 4; ++kk) umma_ss(od, pa + 128 * kk, ta + 2 * kk, kI3, 1u);
          }
          // (the commit that somebody waits for, also after the last chunk, comes last: none arrives after the CTA's end)
          umma_commit(bar(SB_EP));
          umma_commit(bar(SB_OFULL0 + ph));
        }
        __syncwarp();
        if (last) break;
      }
      k.ok = ok;
    }
  } else if (warp >= 4 && warp < 8) {
    // ==================================== mask group =======================================
    // T [n][k]: kept where k <= n (forward) or k >= n (reverse), as bf16 pairs, K-major tiles.  The
    // M = 64 accumulator keeps this warp's rows 16 q4 .. 16 q4 + 15 in the first 16 lanes of its
    // tensor-memory quarter; the 16x256b load hands them out as 8x8-matrix fragments.
    const int mat_k = lane & 7, mat_h = (lane >> 3) & 1, mat_j = lane >> 4;
    const int rl = lane >> 2, c0 = 2 * (lane & 3);   // row and first column of the thread's pair in a fragment
    const bool keep0 = REV ? c0 >= rl : c0 <= rl, keep1 = REV ? c0 + 1 >= rl : c0 + 1 <= rl;
    const uint32_t diag = (keep0 ? 0x0000FFFFu : 0u) | (keep1 ? 0xFFFF0000u : 0u);
    const uint32_t t_lane = tmem + ((uint32_t)(q4 * 32) << 16);
    const uint32_t dst = base + kOffT + (q4 * 16 + mat_h * 8 + mat_k) * 128;
    bool ok = k.ok;
    for (int c = first; ok && any; ++c) {
      k.c = c + 1;
      if (!(ok = wait_all(bar(SB_TFULL), c & 1))) break;
      if (c > 0 && !(ok = wait_all(bar(SB_OFULL0 + ((c - 1) & 1)), ((c - 1) >> 1) & 1))) break;   // T's last reader
      if (!(ok = wait_all(bar(SB_DESC0 + (c & 3)), (c >> 2) & 1))) break;
      const bool last = (ctl->desc[c & 3].flags & kLast) != 0;
      tc_fence_after();
#pragma unroll
      for (int jp = 0; jp < 4; ++jp) {
        uint32_t hi[4] = {0u, 0u, 0u, 0u}, lo[4] = {0u, 0u, 0u, 0u};   // (rows lo, cols j0) (hi, j0) (lo, j1) (hi, j1)
        if (REV ? jp >= q4 : jp <= q4) {
          uint32_t r[8];
          tmem_ld_16x256b_x2(t_lane + kColT + 16 * jp, r);
          tmem_ld_wait();
#pragma unroll
          for (int m = 0; m < 4; ++m)
            split_bf16(__uint_as_float(r[2 * m]), __uint_as_float(r[2 * m + 1]), hi[m], lo[m]);
          if (jp == q4) {
            hi[0] &= diag; lo[0] &= diag;
            hi[3] &= diag; lo[3] &= diag;
            hi[REV ? 1 : 2] = 0u;
            lo[REV ? 1 : 2] = 0u;
          }
        }
        const uint32_t at = dst + (((uint32_t)(2 * jp + mat_j) ^ (uint32_t)mat_k) << 4);
        stmatrix_x4(at, hi[0], hi[1], hi[2], hi[3]);
        stmatrix_x4(at + kSlab, lo[0], lo[1], lo[2], lo[3]);
      }
      fence_proxy_async();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(SB_TREADY));
      if (last) break;
    }
    k.ok = ok;
  } else if (warp >= 8 && warp < 12) {
    // =================================== output group ======================================
    const uint32_t t_lane = tmem + ((uint32_t)(q4 * 32) << 16);
    bool ok = k.ok;
    for (int c = first; ok && any; ++c) {
      k.c = c + 1;
      if (!(ok = wait_all(bar(SB_DESC0 + (c & 3)), (c >> 2) & 1))) break;
      if (!(ok = wait_all(bar(SB_OFULL0 + (c & 1)), (c >> 1) & 1))) break;
      const volatile ChunkDesc* d = &ctl->desc[c & 3];
      const long long row = d->row;
      const int nr = d->nr, roff = d->roff, nr_tile = d->nr_tile, flags = d->flags;
      const bool last = (flags & kLast) != 0;
      tc_fence_after();
      if (!DVK) {
        // lane = key channel, column = row of the chunk: 32 contiguous bytes per thread and group
        // of 8 rows, 1 KiB per warp
        const int ch = q4 * 32 + lane;
        float* raw = (KIND == 0 ? a.raw_q : a.raw_k) + (row - roff) * DK;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t r[32];
          tmem_ld32(t_lane + kColO + (uint32_t)(c & 1) * 64u + 32 * hf, r);
          tmem_ld_wait();
          if (hf == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(SB_OFREE0 + (c & 1)));
          }
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const int r0 = 32 * hf + 8 * g;            // row of the chunk
            if (r0 + 8 <= nr && (flags & kWhole)) {
              float4* dst = reinterpret_cast<float4*>(raw + (r0 / 8 * DK + ch) * 8);
              __stcg(dst, make_float4(__uint_as_float(r[8 * g]), __uint_as_float(r[8 * g + 1]),
                                      __uint_as_float(r[8 * g + 2]), __uint_as_float(r[8 * g + 3])));
              __stcg(dst + 1, make_float4(__uint_as_float(r[8 * g + 4]), __uint_as_float(r[8 * g + 5]),
                                          __uint_as_float(r[8 * g + 6]), __uint_as_float(r[8 * g + 7])));
            } else {                                   // a ragged group, or a chunk of a cut tile
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                const int rr = roff + r0 + e, w = min(8, nr_tile - (rr & ~7));
                if (r0 + e < nr) raw[(rr & ~7) * DK + ch * w + (rr & 7)] = __uint_as_float(r[8 * g + e]);
              }
            }
          }
        }
      } else {
        // dv^T fragments [value column][row] are transposed by stmatrix.trans into four swizzled
        // 64-column slabs and leave by tensor copies
        const int mat_k = lane & 7, mat_h = (lane >> 3) & 1, mat_j = lane >> 4;
        if (k.n_ot > 0 && !(ok = wait_all(bar(SB_OTFREE0 + ((k.n_ot - 1) & 1)), ((k.n_ot - 1) >> 1) & 1))) break;
#pragma unroll
        for (int bl = 0; bl < 2; ++bl) {
          const uint32_t mat = base + kOffOut + (2 * bl + (q4 >> 1)) * kSlab + (mat_j * 8 + mat_k) * 128;
#pragma unroll 1
          for (int hv = 0; hv < 2; ++hv) {
            uint32_t r[32];
            tmem_ld_16x256b_x8(t_lane + ((uint32_t)(16 * hv) << 16) + kColO + 64 * bl, r);
            tmem_ld_wait();
            if (bl == 1 && hv == 1) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(bar(SB_OFREE0 + (c & 1)));
            }
            const uint32_t chunk = (uint32_t)(4 * (q4 & 1) + 2 * hv + mat_h);
            const uint32_t dst = mat + ((chunk ^ (uint32_t)mat_k) << 4);
#pragma unroll
            for (int jp = 0; jp < 4; ++jp) {
              const int j0 = 2 * jp, j1 = 2 * jp + 1;
              stmatrix_x4_trans(dst + jp * 16 * 128,
                                pack_bf16(__uint_as_float(r[4 * j0]), __uint_as_float(r[4 * j0 + 1])),
                                pack_bf16(__uint_as_float(r[4 * j0 + 2]), __uint_as_float(r[4 * j0 + 3])),
                                pack_bf16(__uint_as_float(r[4 * j1]), __uint_as_float(r[4 * j1 + 1])),
                                pack_bf16(__uint_as_float(r[4 * j1 + 2]), __uint_as_float(r[4 * j1 + 3])));
            }
          }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(SB_OTFULL));
        if (q4 == 0) {
          if (!(ok = wait_all(bar(SB_OTFULL), k.n_ot & 1))) break;
          if (nr == kTile) {
            if (lane < 4) tma_store_2d(&maps.dv, 64 * lane, (int)row, base + kOffOut + lane * kSlab);
          } else {   // boxes of 8 rows and of 1 row, so that no row of another chunk is touched
            const int n8 = nr >> 3, n1 = nr & 7;
            for (int e = lane; e < 4 * (n8 + n1); e += 32) {
              const int s = e & 3, v = e >> 2;
              if (v < n8)
                tma_store_2d(&maps.dv8, 64 * s, (int)row + 8 * v, base + kOffOut + s * kSlab + 8 * v * 128);
              else
                tma_store_2d(&maps.dv1, 64 * s, (int)row + 8 * n8 + (v - n8),
                             base + kOffOut + s * kSlab + (8 * n8 + (v - n8)) * 128);
            }
          }
          bulk_commit();
          bulk_wait_read<0>();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(SB_OTFREE0 + (k.n_ot & 1)));
        }
        ++k.n_ot;
      }
      if (last) break;
    }
    k.ok = ok;
  } else if (warp >= 12) {
    // ==================================== state group ======================================
    // 8 warps: tensor-memory quarter q4, columns 128 half .. 128 half + 127 of the state.
    const int half = (warp - 12) >> 2, rt = tid - 12 * 32;
    const uint32_t t_st = tmem + ((uint32_t)(q4 * 32) << 16) + kColS + 128 * half;
    const int ln = q4 * 32 + lane;
    // element (column c of this thread) of the state in the layout of s0, [DK][DV]
    auto elem = [&](int c) -> long long {
      return DVK ? (long long)c * DV + 128 * half + ln : (long long)ln * DV + 128 * half + c;
    };
    const float* init = KIND == 0 ? a.s0 : a.dsT;
    if (init) init += sh * (long long)DK * DV;
    bool ok = k.ok;
    if (ok && pc.wait) {
      // The piece before this one is the first one of a CTA with a lower index, and CTAs start in the
      // order of their index: it is running or done.  The wait is bounded all the same.
      const int32_t* flag = a.seg_flag + sh * 3 + KIND;
      if (lane == 0) {
        const long long t0 = clock64();
        while (ld_acquire_s32(flag) < 8) {
          if (wc->abort_flag) { ok = false; break; }
          if (clock64() - t0 >= a.limit) {
            ok = ld_acquire_s32(flag) >= 8;
            if (!ok) {
              wc->abort_flag = 1;
              atomicMax(&hdr->status, (int)RODIMUS_ERR_TIMEOUT);
            }
            break;
          }
          __nanosleep(200);
        }
      }
      ok = __all_sync(0xffffffffu, ok) != 0;
      init = a.seg_state + (sh * 3 + KIND) * (long long)DK * DV;
    }
    // (a state handed over is read and written 16 bytes per thread, 512 contiguous bytes per warp)
    auto handed = [&](const float* p, int piece, int e) { return p + ((8 * piece + e / 4) * 256 + rt) * 4; };
    auto expand = [&](int c) {
      const int r = rt & 63;
      const uint32_t src = base + kOffY + (c & 1) * kOpBytes + r * 128, dst = base + kOffY32 + r * 128, sw = (uint32_t)(r & 7);
      // (loads are issued ahead of the stores, four at a time)
      if (!DVK) {
#pragma unroll
        for (uint32_t hf = 0; hf < 2; ++hf) {
          uint4 w[4];
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u) {
            const uint32_t c16 = (uint32_t)(rt >> 6) + 4 * (4 * hf + u);     // 16-byte piece (8 values) of the row
            w[u] = lds128(src + (c16 >> 3) * kSlab + (((c16 & 7) ^ sw) << 4));
          }
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u) {
            const uint32_t c16 = (uint32_t)(rt >> 6) + 4 * (4 * hf + u);
            const uint32_t d = dst + (c16 >> 2) * kSlab, j = (c16 & 3) * 2;
            sts128(d + ((j ^ sw) << 4), w[u].x << 16, w[u].x & 0xffff0000u, w[u].y << 16, w[u].y & 0xffff0000u);
            sts128(d + (((j + 1) ^ sw) << 4), w[u].z << 16, w[u].z & 0xffff0000u, w[u].w << 16, w[u].w & 0xffff0000u);
          }
        }
      } else {
        uint4 wh[4], wl[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
          const uint32_t c16 = (uint32_t)(rt >> 6) + 4 * u;     // of the 128 channels
          const uint32_t s = src + (c16 >> 3) * kSlab + (((c16 & 7) ^ sw) << 4);
          wh[u] = lds128(s);
          wl[u] = lds128(s + 2 * kSlab);
        }
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
          const uint32_t c16 = (uint32_t)(rt >> 6) + 4 * u;
          const uint32_t h4[4] = {wh[u].x, wh[u].y, wh[u].z, wh[u].w}, l4[4] = {wl[u].x, wl[u].y, wl[u].z, wl[u].w};
          uint32_t f[8];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 hv = unpack_bf16(h4[e]), lv = unpack_bf16(l4[e]);
            f[2 * e] = __float_as_uint(tf32_rna(hv.x + lv.x));
            f[2 * e + 1] = __float_as_uint(tf32_rna(hv.y + lv.y));
          }
          const uint32_t d = dst + (c16 >> 2) * kSlab, j = (c16 & 3) * 2;
          sts128(d + ((j ^ sw) << 4), f[0], f[1], f[2], f[3]);
          sts128(d + (((j + 1) ^ sw) << 4), f[4], f[5], f[6], f[7]);
        }
      }
    };
    // r *= D, by lane or by column
    auto scale_by = [&](uint32_t (&r)[32], const float* dv, int piece) {
      if (!DVK) {
        const float d = dv[ln];
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * d);
      } else {
#pragma unroll
        for (int e4 = 0; e4 < 8; ++e4) {
          const float4 d = *reinterpret_cast<const float4*>(dv + 32 * piece + 4 * e4);
          r[4 * e4] = __float_as_uint(__uint_as_float(r[4 * e4]) * d.x);
          r[4 * e4 + 1] = __float_as_uint(__uint_as_float(r[4 * e4 + 1]) * d.y);
          r[4 * e4 + 2] = __float_as_uint(__uint_as_float(r[4 * e4 + 2]) * d.z);
          r[4 * e4 + 3] = __float_as_uint(__uint_as_float(r[4 * e4 + 3]) * d.w);
        }
      }
    };
    // (a caller's state is read through L1: 16 bytes a thread are half a sector, the other half is the next
    // load's.  Past L1 the packed shape of get_piece took 8 us more.)
    auto load_init = [&](uint32_t (&r)[32], int piece) {
      if (!init) {
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = 0u;
      } else if (DVK && !pc.wait) {
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__ldcg(init + elem(32 * piece + e)));
      } else {
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          const float4 v = pc.wait ? __ldcg(reinterpret_cast<const float4*>(handed(init, piece, e)))
                                   : __ldg(reinterpret_cast<const float4*>(init + elem(32 * piece + e)));
          r[e] = __float_as_uint(v.x);
          r[e + 1] = __float_as_uint(v.y);
          r[e + 2] = __float_as_uint(v.z);
          r[e + 3] = __float_as_uint(v.w);
        }
      }
    };
    int c = first;
    if (ok && !any) {   // nothing to sweep: the state is only passed on
#pragma unroll 1
      for (int piece = 0; piece < 4; ++piece) {
        uint32_t r[32];
        load_init(r, piece);
        tmem_st32(t_st + 32 * piece, r);
      }
      tmem_st_wait();
    }
    bool last = !any;
    // the dv output tile lies where the other kinds keep half of their expanded Y: its copies are done
    if (ok && !DVK && k.n_ot > 0) ok = wait_all(bar(SB_OTFREE0 + ((k.n_ot - 1) & 1)), ((k.n_ot - 1) >> 1) & 1);
    while (ok && !last) {
      if (!(ok = wait_all(bar(SB_FY0 + (c & 1)), (c >> 1) & 1))) break;
      if (c > 0 && !(ok = wait_all(bar(SB_M1), (c - 1) & 1))) break;    // Y32's last reader
      expand(c);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(SB_EY0 + (c & 1)));
      if (!(ok = wait_all(bar(SB_DESC0 + (c & 3)), (c >> 2) & 1))) break;
      const int nr = ctl->desc[c & 3].nr, flags = ctl->desc[c & 3].flags;
      last = (flags & kLast) != 0;
      if (!(flags & kWhole)) {
        // a chunk of a cut tile: its decays, from the same additions in the same order as its operands'
        if (rt < DK) {
          const long long e = ctl->desc[c & 3].row * DK + rt;
          float acc = 0.f;
          for (int r = 0; r < nr; ++r)
            acc += gate_of(__bfloat162float(a.gx[e + r * DK]), __bfloat162float(a.ty[e + r * DK]), a.ingate).la2;
          sD[(c & 3) * DK + rt] = ex2f(acc);
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(SB_DRDY));
        }
        if (!(ok = wait_all(bar(SB_DRDY), k.n_cut & 1))) break;
        ++k.n_cut;
      }
      const float* dvec = sD + ((REV ? c : c - 1) & 3) * DK;   // forward: of the chunk before
      if (c > first) {
        if (!(ok = wait_all(bar(SB_UFULL), (c - 1) & 1))) break;
        tc_fence_after();
      }
#pragma unroll 1
      for (int piece = 0; piece < 4; ++piece) {
        uint32_t r[32];
        if (c > first) {
          tmem_ld32(t_st + 32 * piece, r);
          tmem_ld_wait();
        } else {
          load_init(r, piece);
        }
        if (REV || c > first) scale_by(r, dvec, piece);
        tmem_st32(t_st + 32 * piece, r);
      }
      if (nr < kTile) {
        // a short chunk: the rows past it belong to other chunks, or to another sequence.  With those of P and X zero
        // they contribute nothing, whatever they hold (of P alone: a NaN or an infinity would not vanish).
        if (!(ok = wait_all(bar(SB_FP), c & 1) && wait_all(bar(SB_FX), c & 1))) break;
        const uint32_t at = base + ((rt >> 3) & 3) * kSlab + (rt & 7) * 16;   // (a warp's row: 8 x 16 bytes of 4 slabs)
#pragma unroll
        for (int u = 0; u < kTile / 8; ++u) {
          const int r = nr + (rt >> 5) + 8 * u;
          if (r < kTile) {
            sts128(at + kOffP + r * 128, 0u, 0u, 0u, 0u);
            sts128(at + kOffX + r * 128, 0u, 0u, 0u, 0u);
          }
        }
        fence_proxy_async();
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(SB_SREADY));
      ++c;
    }
    k.c = c;
    if (DVK) k.n_ot += c - first;
    // ---- after the last chunk
    if (ok && any) ok = wait_all(bar(SB_UFULL), (c - 1) & 1);
    if (ok) {
      tc_fence_after();
      const bool hand_on = pc.hand;
      float* dst = nullptr;
      if (hand_on) dst = a.seg_state + (sh * 3 + KIND) * (long long)DK * DV;
      else if (KIND == 1 && a.ds0) dst = a.ds0 + sh * (long long)DK * DV;
      const bool dot = KIND == 0 && !hand_on && a.dsT != nullptr;
      const float* dsT = dot ? a.dsT + sh * (long long)DK * DV : nullptr;
      if (dst || dot) {
        float acc = 0.f;
#pragma unroll 1
        for (int piece = 0; piece < 4; ++piece) {
          uint32_t r[32];
          tmem_ld32(t_st + 32 * piece, r);
          tmem_ld_wait();
          if (!REV && any) scale_by(r, sD + ((c - 1) & 3) * DK, piece);
          if (dst) {   // (of the dv sweep only the handed-over state is ever wanted)
#pragma unroll
            for (int e = 0; e < 32; e += 4)
              __stcg(reinterpret_cast<float4*>(const_cast<float*>(hand_on ? handed(dst, piece, e) : dst + elem(32 * piece + e))),
                     make_float4(__uint_as_float(r[e]), __uint_as_float(r[e + 1]), __uint_as_float(r[e + 2]),
                                 __uint_as_float(r[e + 3])));
          }
          if (dot) {
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const float4 v = __ldg(reinterpret_cast<const float4*>(dsT + elem(32 * piece + e)));
              acc = fmaf(__uint_as_float(r[e]), v.x, fmaf(__uint_as_float(r[e + 1]), v.y,
                    fmaf(__uint_as_float(r[e + 2]), v.z, fmaf(__uint_as_float(r[e + 3]), v.w, acc))));
            }
          }
        }
        if (dot) (half ? a.c2 : a.c)[sh * DK + ln] = acc;
        if (hand_on) {
          __threadfence();
          __syncwarp();
          if (lane == 0) red_release_add(a.seg_flag + sh * 3 + KIND, 1);
        }
      }
      tc_fence_before();
    }
    k.ok = ok;
  }
}

template <bool VARLEN>
__global__ void __launch_bounds__(kSwThreads, 1)
ddts_bwd_sweep_tc_kernel(const __grid_constant__ SweepMaps maps, const BwdTcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
  auto bar = [&](int i) { return base + kOffBar + 8u * (uint32_t)i; };
  volatile SwCtl* ctl = reinterpret_cast<volatile SwCtl*>(gbase + kOffCtl);
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    ctl->wait.abort_flag = 0;
    ctl->wait.limit = a.limit;
    ctl->n_x = ctl->n_y = ctl->n_p = ctl->n_d = 0;
    for (int i = 0; i < SB_COUNT; ++i) {
      int cnt = 1;
      if (i == SB_EY0 || i == SB_EY1) cnt = 9;
      if (i == SB_SREADY) cnt = 8;
      if (i == SB_TKFREE0 || i == SB_TKFREE1) cnt = kSwThreads / 32;
      if (i == SB_TREADY || i == SB_OFREE0 || i == SB_OFREE1 || i == SB_OTFULL || i == SB_DRDY) cnt = 4;
      mbar_init(bar(i), cnt);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(base + kOffCtl), "r"(kSwTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;

  wait_for_previous_kernel();   // the operands are there
  // (bad cu_seqlens have been reported: nothing to compute)
  if (!VARLEN || *(volatile int32_t*)&a.hdr->status != RODIMUS_ERR_SEQLENS) {
    Carry k = {0, 0, 0, true};
    Piece pc;
    for (int i = 0;; ++i) {
      uint32_t ticket = blockIdx.x;
      if (VARLEN && i > 0) {
        // The producer's warp draws the next ticket when it has asked for the last tile of a piece; two
        // slots, so that a slow warp can still read the one before.
        const int slot = i & 1;
        const uint32_t ph = (uint32_t)((i - 1) >> 1) & 1;   // slot 1 is first used for i = 1, slot 0 for i = 2
        if (warp == 0) {
          if (!__all_sync(0xffffffffu, mbar_wait(bar(SB_TKFREE0 + slot), ph ^ 1, &ctl->wait, a.hdr))) break;
          if (elect_one()) {
            ctl->ticket[slot] = gridDim.x + atomicAdd(reinterpret_cast<unsigned int*>(a.seg_flag + a.n_flags - 1), 1u);
            mbar_arrive(bar(SB_TICKET0 + slot));
          }
          __syncwarp();
        }
        if (!__all_sync(0xffffffffu, mbar_wait(bar(SB_TICKET0 + slot), ph, &ctl->wait, a.hdr))) break;
        ticket = ctl->ticket[slot];
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(bar(SB_TKFREE0 + slot));
      }
      if (!get_piece<VARLEN>(a, (int)blockIdx.x, (int)gridDim.x, i, ticket, pc)) break;
      if (pc.kind == 0) sweep_piece<0, VARLEN>(a, maps, pc, base, gbase, tmem, k);
      else if (pc.kind == 1) sweep_piece<1, VARLEN>(a, maps, pc, base, gbase, tmem, k);
      else sweep_piece<2, VARLEN>(a, maps, pc, base, gbase, tmem, k);
    }
  }

  // ------------------------------------------ teardown ------------------------------------------
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (ctl->wait.abort_flag != 0) {   // nothing may still be writing this CTA's shared or tensor memory
    if (tid == 0) {
      for (int back = 1; back <= 2; ++back)
        if (ctl->n_y >= back) mbar_drain(bar(SB_FY0 + ((ctl->n_y - back) & 1)), ((ctl->n_y - back) >> 1) & 1);
      if (ctl->n_x > 0) mbar_drain(bar(SB_FX), (ctl->n_x - 1) & 1);
      if (ctl->n_p > 0) mbar_drain(bar(SB_FP), (ctl->n_p - 1) & 1);
      for (int back = 1; back <= 4; ++back)
        if (ctl->n_d >= back) mbar_drain(bar(SB_DESC0 + ((ctl->n_d - back) & 3)), ((ctl->n_d - back) >> 2) & 1);
    }
    if (warp == 1 && elect_one()) {   // a commit follows the contractions of the thread that makes it
      umma_commit(bar(SB_DRAIN));
      mbar_drain(bar(SB_DRAIN), 0);
    }
  }
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSwTmemCols) : "memory");
}

// ---------------------------------------------------------------------------------------------
// dq, dk, dx, dy of one tile
// ---------------------------------------------------------------------------------------------
//   dg   = -tau dla + w tau u'/u        dtau = -g dla + w ln u         (u = g, or 1 - e^-g = sigmoid(x))
//   dx   = dg sigmoid(x)  =  w tau sigmoid(x) u'/u  -  dla tau sigmoid(x)
//   dy   = dtau tau (1 - tau)  =  (1 - tau) (dla log alpha + w log ahat)
// One CTA per (tile, 32 channels).  Tiles run from the end of the sequences to their start (see
// order_tiles): a CTA waits (bounded) for the suffix sums of the tile after it, whose CTA has a lower index.
constexpr int kPostThreads = 256, kPostCh = 32, kPostRows = 4;   // 4 rows x 2 channels a thread
static_assert(kPostThreads == kPostCh / 2 * (kTile / kPostRows), "one thread per 4 rows x 2 channels");

__global__ void __launch_bounds__(kPostThreads, 3) ddts_bwd_post_kernel(const BwdTcArgs a) {
  __shared__ __align__(16) float s_la[kTile * kPostCh];
  __shared__ __align__(16) float s_part[(kTile / kPostRows) * kPostCh];
  __shared__ __align__(16) double s_sum[(kTile / kPostRows) * kPostCh];
  __shared__ int s_late;
  wait_for_previous_kernel();
  if (a.cu && *(volatile int32_t*)&a.hdr->status == RODIMUS_ERR_SEQLENS) return;
  const int tid = threadIdx.x;
  const int quarter = (int)(blockIdx.x & 3u), hs = (int)(blockIdx.x >> 2);
  const int head = hs % a.heads, pos = hs / a.heads;
  TileRef tr;
  long long slot;
  if (a.cu) {
    const int2 e = __ldg(a.tile_order + pos);
    if (e.x < 0) return;
    int lo, hi;
    seq_range(a.cu, e.x, a.T, lo, hi);
    tr.n = e.x;
    tr.t = e.y;
    tr.len = hi - lo;
    tr.row0 = (long long)head * a.T + lo + (long long)e.y * kTile;
    slot = (long long)head * a.slots_per_head + lo / kTile + e.x + e.y;
  } else {
    tr.n = head / a.H;
    tr.t = a.slots_per_head - 1 - pos;
    tr.len = a.T;
    tr.row0 = (long long)head * a.T + (long long)tr.t * kTile;
    slot = (long long)head * a.slots_per_head + tr.t;
  }
  tr.nr = min(kTile, tr.len - tr.t * kTile);
  const int cp = tid & 15, rg = tid >> 4, ch = quarter * kPostCh + 2 * cp;
  const int live = tr.nr - rg * kPostRows;
  const long long e0 = (tr.row0 + rg * kPostRows) * 64 + ch / 2;
  const uint32_t* gx = reinterpret_cast<const uint32_t*>(a.gx) + e0;
  const uint32_t* ty = reinterpret_cast<const uint32_t*>(a.ty) + e0;
  const uint32_t* q = reinterpret_cast<const uint32_t*>(a.q) + e0;
  const uint32_t* k = reinterpret_cast<const uint32_t*>(a.k) + e0;
  uint32_t wx[kPostRows], wy[kPostRows], wq[kPostRows], wk[kPostRows];
#pragma unroll
  for (int i = 0; i < kPostRows; ++i) {
    wx[i] = wy[i] = wq[i] = wk[i] = 0u;
    if (i < live) {
      wx[i] = __ldg(gx + i * 64);
      wy[i] = __ldg(ty + i * 64);
      wq[i] = __ldg(q + i * 64);
      wk[i] = __ldg(k + i * 64);
    }
  }
  float rq[2][kPostRows], rk[2][kPostRows];
  {
    const int r0 = (rg * kPostRows) & ~7, w = min(8, tr.nr - r0);    // the group of 8 rows and its rows
    const long long o = (tr.row0 + r0) * DK + ch * w + (rg * kPostRows & 7);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (w == 8) {
        const float4 vq = __ldcs(reinterpret_cast<const float4*>(a.raw_q + o + 8 * e));
        const float4 vk = __ldcs(reinterpret_cast<const float4*>(a.raw_k + o + 8 * e));
        rq[e][0] = vq.x; rq[e][1] = vq.y; rq[e][2] = vq.z; rq[e][3] = vq.w;
        rk[e][0] = vk.x; rk[e][1] = vk.y; rk[e][2] = vk.z; rk[e][3] = vk.w;
      } else {
#pragma unroll
        for (int i = 0; i < kPostRows; ++i) {
          rq[e][i] = i < live ? __ldcs(a.raw_q + o + e * w + i) : 0.f;
          rk[e][i] = i < live ? __ldcs(a.raw_k + o + e * w + i) : 0.f;
        }
      }
    }
  }
  const unsigned long long mask = __ldg(a.mask + slot);
  // per element: la2 (then the cumulative b), and what dx, dy need once dla is known:
  // dx = w cx - dla cs,  dy = omt (dla la + w lh) ln 2
  float2 b[kPostRows], la2[kPostRows], lh2[kPostRows], cs[kPostRows], cx[kPostRows], omt[kPostRows];
#pragma unroll
  for (int i = 0; i < kPostRows; ++i) {
    const float2 x2 = unpack_bf16(wx[i]), y2 = unpack_bf16(wy[i]);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float x = e ? x2.y : x2.x, y = e ? y2.y : y2.x;
      const Gate g = gate_of(x, y, a.ingate);
      const float ey = ex2f(-fabsf(y) * kLog2e), ry = rcpf(1.f + ey), rx = rcpf(1.f + g.e);
      const float om = y >= 0.f ? ey * ry : ry, sx = x >= 0.f ? rx : g.e * rx;
      const float s = g.tau * sx;
      // tau sigmoid(x) u'/u: u = g gives sigmoid(x) / g, u = sigmoid(x) gives 1 - sigmoid(x)
      const float c = a.ingate == RODIMUS_INGATE_POW_G ? s * rcpf(g.g2) * kLog2e : g.tau * (x >= 0.f ? g.e * rx : rx);
      if (e) { la2[i].y = g.la2; lh2[i].y = g.lh2; cs[i].y = s; cx[i].y = c; omt[i].y = om * 0.6931471805599453f; }
      else { la2[i].x = g.la2; lh2[i].x = g.lh2; cs[i].x = s; cx[i].x = c; omt[i].x = om * 0.6931471805599453f; }
    }
    b[i] = i < live ? la2[i] : make_float2(0.f, 0.f);
  }
  tile_scan<kPostRows, kPostCh, false>(b, cp, rg, tr.nr, s_la, s_part, nullptr, mask,
                                       [&](int i) {
                                         float2 v = make_float2(0.f, 0.f);
#pragma unroll
                                         for (int u = 0; u < kPostRows; ++u)
                                           if (u == i && u < live) v = la2[u];
                                         return v;
                                       });
  uint32_t* dq = reinterpret_cast<uint32_t*>(a.dq) + e0;
  uint32_t* dk = reinterpret_cast<uint32_t*>(a.dk) + e0;
  float2 w[kPostRows], uw[kPostRows];
  double t0 = 0.0, t1 = 0.0;
#pragma unroll
  for (int i = 0; i < kPostRows; ++i) {
    const float2 qv = unpack_bf16(wq[i]), kv = unpack_bf16(wk[i]);
    const float gq0 = a.scale * rq[0][i] * ex2f(b[i].x), gq1 = a.scale * rq[1][i] * ex2f(b[i].y);
    const float gk0 = rk[0][i] * ex2f(lh2[i].x - b[i].x), gk1 = rk[1][i] * ex2f(lh2[i].y - b[i].y);
    w[i] = make_float2(kv.x * gk0, kv.y * gk1);
    uw[i] = make_float2(fmaf(qv.x, gq0, -w[i].x), fmaf(qv.y, gq1, -w[i].y));
    if (i < live) {
      dq[i * 64] = pack_bf16(gq0, gq1);
      dk[i * 64] = pack_bf16(gk0, gk1);
      t0 += (double)uw[i].x;
      t1 += (double)uw[i].y;
    }
  }
  *reinterpret_cast<double2*>(s_sum + rg * kPostCh + 2 * cp) = make_double2(t0, t1);
  const bool chained = (tr.t + 1) * kTile < tr.len;
  if (tid == 0) {
    s_late = 0;
    if (chained) {
      const int32_t* flag = a.tile_flag + (slot + 1) * 4 + quarter;
      const long long c0 = clock64();
      while (ld_acquire_s32(flag) == 0) {
        if (clock64() - c0 >= a.limit) {
          if (ld_acquire_s32(flag) != 0) break;
          s_late = 1;
          atomicMax(&a.hdr->status, (int)RODIMUS_ERR_TIMEOUT);
          break;
        }
        __nanosleep(32);
      }
    }
  }
  __syncthreads();
  if (s_late) return;
  // The suffix sums of a (tile, 32 channels) take the place of its own raw values of rows 0..7, which this
  // CTA alone reads: channels 0..15 in raw_q, 16..31 in raw_k (128 bytes each, also of a one-row tile).
  auto suffix_of = [&](int t) {
    const long long row = tr.row0 + (long long)(t - tr.t) * kTile;
    const int w0 = min(8, tr.len - t * kTile);
    return reinterpret_cast<double2*>((cp < 8 ? a.raw_q : a.raw_k) + row * DK + quarter * kPostCh * w0) + (cp & 7);
  };
  double acc0, acc1;
  if (chained) {
    const double2 v = __ldcg(suffix_of(tr.t + 1));
    acc0 = v.x;
    acc1 = v.y;
  } else {
    const long long e = (long long)(tr.n * a.H + (a.cu ? head : head % a.H)) * DK + ch;
    acc0 = a.dsT ? (double)(a.c[e] + a.c2[e]) : 0.0;
    acc1 = a.dsT ? (double)(a.c[e + 1] + a.c2[e + 1]) : 0.0;
  }
#pragma unroll 1
  for (int g = kTile / kPostRows - 1; g > rg; --g) {
    const double2 v = *reinterpret_cast<const double2*>(s_sum + g * kPostCh + 2 * cp);
    acc0 += v.x;
    acc1 += v.y;
  }
  if (rg == 0) {   // these threads end with the tile's suffix: half a warp, published before the outputs
    __stcg(suffix_of(tr.t), make_double2(acc0 + t0, acc1 + t1));
    __threadfence();
  }
  __syncwarp();
  if (tid == 0) st_release_s32(a.tile_flag + slot * 4 + quarter, 1);
  uint32_t* dx = reinterpret_cast<uint32_t*>(a.dx) + e0;
  uint32_t* dy = reinterpret_cast<uint32_t*>(a.dy) + e0;
#pragma unroll
  for (int i = kPostRows - 1; i >= 0; --i) {
    if (i >= live) continue;
    acc0 += (double)uw[i].x;
    acc1 += (double)uw[i].y;
    const float d0 = (float)acc0, d1 = (float)acc1;
    dx[i * 64] = pack_bf16(fmaf(w[i].x, cx[i].x, -d0 * cs[i].x), fmaf(w[i].y, cx[i].y, -d1 * cs[i].y));
    dy[i * 64] = pack_bf16(omt[i].x * fmaf(d0, la2[i].x, w[i].x * lh2[i].x), omt[i].y * fmaf(d1, la2[i].y, w[i].y * lh2[i].y));
  }
}

std::atomic<unsigned long long> g_sweep_smem_done[2];   // dense, packed

// Workspace beyond header and order: raw_q and raw_k (1 KiB per row), c, and an area that holds the
// states of sweeps cut in two (384 KiB per (sequence, head), dense calls of more than one tile) and the
// few words per tile; where those fit into the 384 KiB the size does not change.
struct Scratch {
  size_t raw_q, raw_k, c, c2, dtile, mask, tile_flag, tile_order, seg_flag, seg_state, bytes;
  long long slots;
  int slots_per_head, heads;
};

Scratch scratch_layout(const rodimus_ddts_bwd_params& p) {
  Scratch s;
  const size_t rows = (size_t)p.B * p.H * p.T;
  const bool varlen = p.cu_seqlens != nullptr;
  const size_t nseq = varlen ? (size_t)p.N : (size_t)p.B, items = nseq * p.H;
  s.heads = varlen ? p.H : p.B * p.H;
  s.slots_per_head = varlen ? p.T / kTile + p.N : (p.T + kTile - 1) / kTile;
  s.slots = (long long)s.heads * s.slots_per_head;
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  s.raw_q = 0;
  s.raw_k = rows * DK * 4;
  s.c = 2 * rows * DK * 4;
  const size_t area = up(s.c + items * DK * 4), states = items * 3 * (size_t)DK * DV * 4;
  s.seg_state = area;
  size_t at = area + (!varlen && p.T > kTile ? states : 0);
  auto take = [&](size_t bytes) {
    const size_t o = at;
    at += up(bytes);
    return o;
  };
  s.dtile = take((size_t)s.slots * DK * 4);
  s.mask = take((size_t)s.slots * 8);
  s.tile_flag = take((size_t)s.slots * 16);
  s.seg_flag = take((items * 3 + 1) * 4);
  s.c2 = take(items * DK * 4);
  s.tile_order = take(varlen ? (size_t)s.slots_per_head * 8 : 0);
  const size_t least = area + states + up(items * 6 * 4);
  s.bytes = at > least ? at : least;
  return s;
}

}  // namespace

size_t bwd_tc_scratch_bytes(const rodimus_ddts_bwd_params& p) { return scratch_layout(p).bytes; }

cudaError_t launch_bwd_tc(const rodimus_ddts_bwd_params& p, size_t scratch_offset, int* n_launches) {
  *n_launches = 0;
  const Scratch s = scratch_layout(p);
  char* ws = reinterpret_cast<char*>(p.workspace) + scratch_offset;
  BwdTcArgs a;
  a.q = (const __nv_bfloat16*)p.q; a.k = (const __nv_bfloat16*)p.k;
  a.gx = (const __nv_bfloat16*)p.gate_x; a.ty = (const __nv_bfloat16*)p.temp_y;
  a.s0 = p.s0; a.dsT = p.d_sT;
  a.dq = (__nv_bfloat16*)p.d_q; a.dk = (__nv_bfloat16*)p.d_k;
  a.dx = (__nv_bfloat16*)p.d_gate_x; a.dy = (__nv_bfloat16*)p.d_temp_y; a.dv = (__nv_bfloat16*)p.d_v;
  a.ds0 = p.d_s0;
  a.qe_hi = (uint32_t*)p.d_q; a.qe_lo = (uint32_t*)p.d_k;
  a.ki_hi = (uint32_t*)p.d_gate_x; a.ki_lo = (uint32_t*)p.d_temp_y;
  a.dtile = (float*)(ws + s.dtile);
  a.mask = (unsigned long long*)(ws + s.mask);
  a.raw_q = (float*)(ws + s.raw_q); a.raw_k = (float*)(ws + s.raw_k);
  a.tile_flag = (int32_t*)(ws + s.tile_flag);
  a.c = (float*)(ws + s.c);
  a.c2 = (float*)(ws + s.c2);
  a.tile_order = (int2*)(ws + s.tile_order);
  a.seg_state = (float*)(ws + s.seg_state);
  a.seg_flag = (int32_t*)(ws + s.seg_flag);
  a.cu = p.cu_seqlens;
  a.hdr = reinterpret_cast<WorkspaceHeader*>(p.workspace);
  a.order = reinterpret_cast<const int32_t*>(reinterpret_cast<char*>(p.workspace) + sizeof(WorkspaceHeader));
  a.H = p.H; a.T = p.T; a.n_seq = p.cu_seqlens ? p.N : p.B;
  a.heads = s.heads;
  a.slots_per_head = s.slots_per_head;
  a.scale = p.scale; a.ingate = p.ingate;
  a.limit = main_loop_wait_cycles();
  const long long items = (long long)a.n_seq * p.H;
  if (items == 0) return cudaSuccess;
  a.n_flags = items * 3 + 1;
  int dev = 0, sms = 0;
  cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(p.stream);

  if (items * 3 > 0x7fffffffLL || s.slots > 0x1fffffffLL) return cudaErrorInvalidValue;
  SweepMaps m;
  const uint64_t rows = (uint64_t)p.B * p.H * p.T;
  if (rows > 0) {
    if (!encode_bf16_slab_map(&m.v, p.v, rows, DV, 4) || !encode_bf16_slab_map(&m.dout, p.d_o, rows, DV, 4) ||
        !encode_bf16_slab_map(&m.qe_hi, a.qe_hi, rows, DK, 2) || !encode_bf16_slab_map(&m.qe_lo, a.qe_lo, rows, DK, 2) ||
        !encode_bf16_slab_map(&m.ki_hi, a.ki_hi, rows, DK, 2) || !encode_bf16_slab_map(&m.ki_lo, a.ki_lo, rows, DK, 2) ||
        !encode_bf16_map(&m.dv, p.d_v, rows, DV, kTile) || !encode_bf16_map(&m.dv8, p.d_v, rows, DV, 8) ||
        !encode_bf16_map(&m.dv1, p.d_v, rows, DV, 1))
      return cudaErrorInvalidValue;
  } else {
    memset(&m, 0, sizeof(m));   // never used: no tiles
    e = cudaMemsetAsync(a.seg_flag, 0, sizeof(int32_t) * (size_t)a.n_flags, st);
    if (e == cudaSuccess && !p.cu_seqlens) e = cudaMemsetAsync(a.hdr, 0, sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
  }
  auto* const sweep = p.cu_seqlens ? ddts_bwd_sweep_tc_kernel<true> : ddts_bwd_sweep_tc_kernel<false>;
  e = opt_in_shared_memory(sweep, kSwSmem, dev, g_sweep_smem_done[p.cu_seqlens != nullptr]);
  if (e != cudaSuccess) return e;
  if (rows > 0) {
    // (packed: beside the plan of the sequences, which only its last block reads)
    if (p.cu_seqlens) e = launch_overlapped(ddts_bwd_pre_kernel, (unsigned)s.slots + 1u, kPreThreads, 0, st, a);
    else ddts_bwd_pre_kernel<<<(unsigned)s.slots, kPreThreads, 0, st>>>(a);
    if (e != cudaSuccess) return e;
    ++*n_launches;
  }
  // (each of these is launched while the one before it ends, and waits for it before it reads anything of
  // its; allowed to start when that one STARTS, their CTAs took room from it: layer shape 352 -> 440 us,
  // with the launches overlapped only 347)
  // Dense: as many CTAs for each kind of sweep.  Every kind is then cut at the same places, and the two
  // reverse sweeps of a (sequence, head), which share Qe and dO, run side by side and find them in L2 (layer
  // shape, 148 -> 147 CTAs: 350 -> 339 us; before, the launch read 557 MB from DRAM, 268 of it once).
  const long long most = p.cu_seqlens ? sms : sms - sms % 3;
  e = launch_overlapped(sweep, (unsigned)(items * 3 < most ? items * 3 : most), kSwThreads, kSwSmem, st, m, a);
  if (e != cudaSuccess) return e;
  ++*n_launches;
  if (rows > 0) {
    e = launch_overlapped(ddts_bwd_post_kernel, (unsigned)(s.slots * 4), kPostThreads, 0, st, a);
    if (e != cudaSuccess) return e;
    ++*n_launches;
  }
  return cudaGetLastError();
}

}  // namespace ddts
