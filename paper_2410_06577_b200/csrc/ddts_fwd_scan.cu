// Chunked DDTS prefill in two launches, for calls whose gates serve several CTAs or whose items are
// too few to fill the device: operands first, then the scan (in two phases where it is split along time,
// see Segments).
//
// Chunk algebra (appendix "Chunkwise Parallel Representation of the Rodimus Block"; chunk length 64,
// log2 domain, decays anchored at the chunk start, b_r = sum_{j<=r} log2 alpha_j <= 0):
//   Qt_r = scale q_r 2^{b_r}      Kt_i = k_i ahat_i 2^{-b_i}      D = 2^{b_C}
//   P = mask(Qt Kt^T)             O = P V + Qt S_in               S_out = D . (S_in + Kt^T V)
// Everything that depends on the gates - Qt, Kt, D and also P - is the same for all value columns.
//
//   ddts_operands_kernel   a CTA per 64-row tile of every set of gates: Kt, Qt, P and D of the tile as
//                          ONE block of global memory, laid out as the tensor core reads it from
//                          shared memory (128-byte swizzle), so that a single bulk copy brings it in
//   ddts_scan_kernel       a CTA per (sequence, head, 128 value columns): no gate arithmetic, per
//                          chunk two bulk copies, a tensor copy of the v tile and three contractions
// In the layout with one set of gates for all heads the first kernel does 1/H of the work that every
// head's own gates would be, and its blocks are read from L2 by all H dv / 128 CTAs of a sequence.
// Figures (layer shape, B=4 H=16 T=2048 dv=256): one set of gates, dk = 64: 9.6 us + 36 us, the scan
// bound by the issue of its contractions (1670 cycles per chunk of 28 instructions, 1216 cycles of tensor
// work) with 11 TB/s out of L2; gates per head, dk = 128: operands 55 us (bound by no one unit: with a
// third fewer instructions as long), scan 36 us (218 MB, 6 TB/s).
//
// dk = 128: operands in bf16, the precision of the kernel with the gates inside.  dk = 64 (the paper's
// own key width): Kt as three bf16 parts (24 bits), Qt, P and the state's copy for the readout as two
// (16 bits), gates with accurate functions: fp32 accuracy in the state, 2^-16 before the rounding of o.
//
// Where a tile decays by more than e^-60 in some channel it is cut in halves until every chunk fits
// (down to single rows, which always fit because a step's decay is applied as at least e^-60): P
// then keeps pairs of the same chunk only, and the scan takes the tile once per chunk, with the other
// rows of Kt set to zero.
//
// The rows of v behind a sequence's end are zeros: against the zero rows of Kt alone a NaN or an infinity of the
// sequence or head that follows would not vanish.  Behind a head's end the tensor map sees to it, behind a packed
// sequence's warp 3 or the warps of the value gate.
#include <cuda.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>

#include "ddts_common.cuh"
#include "ddts_tc_ptx.cuh"
#include "ddts_tiles.cuh"

namespace ddts {
namespace {

constexpr int kSlab = kTile * 128;          // [64 rows][128 bytes], 128-byte swizzled

// The block of a tile: slabs of Kt and P, then of Qt, then D.
template <int DK>
struct Block {
  static constexpr bool kExact = DK == 64;
  static constexpr int kSlabs = DK / 64;                    // slabs of one part of Kt or Qt
  static constexpr int kKp = kExact ? 3 : 1, kQp = kExact ? 2 : 1;   // parts of Kt; of Qt and P
  static constexpr int kK = 0, kP = kKp * kSlabs * kSlab, kQ = kP + kQp * kSlab, kD = kQ + kQp * kSlabs * kSlab;
  static constexpr int kBytes = kD + 1024;                  // (blocks begin at multiples of 1 KiB)
};

struct ScanArgs {
  const __nv_bfloat16 *q, *k, *gx, *ty;
  const float *s0;
  float* sT;
  const float* feed_d;
  unsigned char* blocks;
  unsigned long long* masks;   // of every tile: bit r = its row r starts a chunk
  const int32_t *cu, *order;
  WorkspaceHeader* hdr;
  int H, T, dv, n_seq;
  int gate_heads;       // sets of gates per sequence: H, or 1 when all heads share one
  int slots_per_head;   // tiles of one (batch, set) of a dense call, of one set of a packed one
  int cols;             // slices of 128 value columns
  int has_beta;
  float scale;
  int ingate;
  long long limit;
  // Calls split along time (see Segments): how the tiles are cut, which of the two launches this is, the final
  // states of segments 0..G-1 (of 1..G-1 from a zero state) and the decays of segments 1..G-1.
  int seg_count, seg_tiles0, seg_tiles, phase;
  float *seg_state, *seg_decay;
};

// Decays and their sums.  dk = 64: exact sums, so that 2^b is as exact as the rows' own decays are.  (An fp32
// sum near -60 carries 2^-19 into every operand made of it: 1e-6 of the final state where gates decay fast,
// 2e-7 in the fp32 kernel, which forms differences before the exponential, 1e-7 here.  It costs 0.6 % of a
// call at the layer shape, 3.7 % with a set of gates per head; sums in fp64, as exact, 2.7 % at the layer shape.)
template <bool EXACT>
struct Decay {
  using One = float;
  using Two = float2;
};
template <>
struct Decay<true> {
  using One = ExactSum;
  using Two = ExactSum2;
};
// 2^b, and 2^(lh - b)
__device__ __forceinline__ float exp2_of(float b) { return ex2f(b); }
__device__ __forceinline__ float exp2_of(float lh, float b) { return ex2f(lh - b); }
__device__ __forceinline__ float scaled(float e, float rest) { return fmaf(e, rest * 0.69314718f, e); }   // e 2^rest, rest tiny
__device__ __forceinline__ float exp2_of(ExactSum b) {
  const float t = b.h + b.l;                                  // b = t + ((b.h - t) + b.l)
  return scaled(ex2f(t), (b.h - t) + b.l);
}
__device__ __forceinline__ float exp2_of(float lh, ExactSum b) {
  const float t = b.h + b.l, r = (b.h - t) + b.l;
  const float u = lh - t, z = u - lh, d = (lh - (u - z)) - (t + z);   // lh - t = u + d
  return scaled(ex2f(u), d - r);
}

template <bool EXACT>
__device__ __forceinline__ void gate_pair(float x, float y, int ingate, typename Decay<EXACT>::One& la2, float& lh2) {
  if constexpr (EXACT) {
    float la;
    gate_logs_f32(x, y, ingate, la, lh2);
    const float p = fmaxf(la * kLog2e, -kRange2);
    const float rest = p > -kRange2 ? fmaf(la, kLog2e, -p) + la * 1.925963e-8f : 0.f;   // log2 e to 48 bits
    constexpr float kRound = 12288.f;                         // 1.5 * 2^13: adding it rounds to 2^-10
    la2.h = (p + kRound) - kRound;
    la2.l = (p - la2.h) + rest;
    lh2 *= kLog2e;
  } else {
    const Gate g = gate_of(x, y, ingate);
    la2 = g.la2;
    lh2 = g.lh2;
  }
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------------------------
// Operands of one tile
// ---------------------------------------------------------------------------------------------
constexpr int kOpThreads = 512;
template <int DK>
constexpr int kOpRowsOf = DK / 16;          // 4 or 8 rows x 2 channels a thread
template <int DK>
constexpr int kOpSmem = Block<DK>::kBytes + (kTile / kOpRowsOf<DK>) * DK * (int)sizeof(typename Decay<Block<DK>::kExact>::One) + 1024;

template <int DK>
__global__ void __launch_bounds__(kOpThreads, 2) ddts_operands_kernel(const ScanArgs a) {
  using B = Block<DK>;
  using Sum = typename Decay<B::kExact>::One;
  using Sums = typename Decay<B::kExact>::Two;
  constexpr int kOpRows = kOpRowsOf<DK>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ unsigned long long s_mask;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
  Sum* s_part = reinterpret_cast<Sum*>(gbase + B::kBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (!a.cu && blockIdx.x == 0 && tid == 0) a.hdr->status = RODIMUS_OK;
  const int head = (int)(blockIdx.x / (unsigned)a.slots_per_head), local = (int)(blockIdx.x % (unsigned)a.slots_per_head);
  const TileRef tr = find_tile<kOpThreads>({a.cu, a.n_seq, a.T, a.cu ? 1 : a.gate_heads}, head, local);
  let_next_kernel_start();
  if (tr.nr <= 0) return;
  const int cp = tid & (DK / 2 - 1), rg = tid / (DK / 2);
  const int live = tr.nr - rg * kOpRows;
  const long long e0 = (tr.row0 + rg * kOpRows) * (DK / 2) + cp;
  const uint32_t* gx = reinterpret_cast<const uint32_t*>(a.gx) + e0;
  const uint32_t* ty = reinterpret_cast<const uint32_t*>(a.ty) + e0;
  const uint32_t* q = reinterpret_cast<const uint32_t*>(a.q) + e0;
  const uint32_t* k = reinterpret_cast<const uint32_t*>(a.k) + e0;
  uint32_t wx[kOpRows], wy[kOpRows], wq[kOpRows], wk[kOpRows];
#pragma unroll
  for (int i = 0; i < kOpRows; ++i) {
    wx[i] = wy[i] = wq[i] = wk[i] = 0u;       // rows past the end: q = k = 0
    if (i < live) {
      wx[i] = __ldg(gx + i * (DK / 2));
      wy[i] = __ldg(ty + i * (DK / 2));
      wq[i] = __ldg(q + i * (DK / 2));
      wk[i] = __ldg(k + i * (DK / 2));
    }
  }
  Sums b[kOpRows];
  float2 lh2[kOpRows];
#pragma unroll
  for (int i = 0; i < kOpRows; ++i) {
    const float2 x = unpack_bf16(wx[i]), y = unpack_bf16(wy[i]);
    gate_pair<B::kExact>(x.x, y.x, a.ingate, b[i].x, lh2[i].x);
    gate_pair<B::kExact>(x.y, y.y, a.ingate, b[i].y, lh2[i].y);
    if (i >= live) b[i] = {};
  }
  auto la_of = [&](int i) {
    Sums la = {};
    if (i >= live) return la;
    const float2 x = unpack_bf16(__ldg(gx + i * (DK / 2))), y = unpack_bf16(__ldg(ty + i * (DK / 2)));
    float lh;
    gate_pair<B::kExact>(x.x, y.x, a.ingate, la.x, lh);
    gate_pair<B::kExact>(x.y, y.y, a.ingate, la.y, lh);
    return la;
  };
  // (the scan's scratch lies where the operands go next)
  const unsigned long long mask = tile_scan<kOpRows, DK, true>(b, cp, rg, tr.nr, reinterpret_cast<Sum*>(gbase), s_part,
                                                               &s_mask, 0ull, la_of);
  {
    const uint32_t w = base + (cp >> 5) * kSlab + ((cp & 3) << 2), c16 = (uint32_t)(cp & 31) >> 2;
#pragma unroll
    for (int i = 0; i < kOpRows; ++i) {
      const int r = rg * kOpRows + i;
      const uint32_t at = w + r * 128 + ((c16 ^ (uint32_t)(r & 7)) << 4);
      const float2 qv = unpack_bf16(wq[i]), kv = unpack_bf16(wk[i]);
      const float ex = exp2_of(b[i].x), ey = exp2_of(b[i].y);
      float qx = qv.x * a.scale * ex, qy = qv.y * a.scale * ey;
#pragma unroll
      for (int p = 0; p < B::kQp; ++p) {
        const uint32_t h = pack_bf16(qx, qy);
        sts32(at + B::kQ + p * B::kSlabs * kSlab, h);
        const float2 f = unpack_bf16(h);
        qx -= f.x;
        qy -= f.y;
      }
      float kx = kv.x * exp2_of(lh2[i].x, b[i].x), ky = kv.y * exp2_of(lh2[i].y, b[i].y);
#pragma unroll
      for (int p = 0; p < B::kKp; ++p) {
        const uint32_t h = pack_bf16(kx, ky);
        sts32(at + B::kK + p * B::kSlabs * kSlab, h);
        const float2 f = unpack_bf16(h);
        kx -= f.x;
        ky -= f.y;
      }
      if (r + 1 == tr.nr) *reinterpret_cast<float2*>(gbase + B::kD + 8 * cp) = make_float2(ex, ey);
    }
    if (tid == 0) a.masks[(long long)head * a.slots_per_head + local] = mask;
  }
  __syncthreads();
  // P = mask(Qt Kt^T): 16 x 16 blocks, those right of the diagonal are zero
  {
#pragma unroll 1
    for (int blk = warp; blk < 16; blk += kOpThreads / 32) {
      const int wr = blk >> 2, wc = blk & 3;
      float acc[2][4] = {};
      if (wc <= wr) {
        const int ra = 16 * wr + (lane & 15), rb = 16 * wc + (lane & 7) + ((lane >> 4) << 3);
#pragma unroll
        for (int kk = 0; kk < DK / 16; ++kk) {
          const uint32_t ca = (uint32_t)(2 * kk + (lane >> 4)), cb = (uint32_t)(2 * kk + ((lane >> 3) & 1));
          const uint32_t aa = base + B::kQ + (ca >> 3) * kSlab + ra * 128 + (((ca & 7) ^ (uint32_t)(ra & 7)) << 4);
          const uint32_t ab = base + B::kK + (cb >> 3) * kSlab + rb * 128 + (((cb & 7) ^ (uint32_t)(rb & 7)) << 4);
          uint32_t fa[4], fb[4];
          ldmatrix_x4(aa, fa);
          ldmatrix_x4(ab, fb);
          mma_bf16_16816(acc[0], fa, fb[0], fb[1]);
          mma_bf16_16816(acc[1], fa, fb[2], fb[3]);
          if (B::kExact) {                    // high x low, low x high
            uint32_t la[4], lb[4];
            ldmatrix_x4(aa + kSlab, la);
            ldmatrix_x4(ab + kSlab, lb);
            mma_bf16_16816(acc[0], fa, lb[0], lb[1]);
            mma_bf16_16816(acc[1], fa, lb[2], lb[3]);
            mma_bf16_16816(acc[0], la, fb[0], fb[1]);
            mma_bf16_16816(acc[1], la, fb[2], fb[3]);
          }
        }
      }
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int r = 16 * wr + 8 * hf + (lane >> 2);
        const int lo = mask == 1ull ? 0 : chunk_start(mask, r);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const int i = 16 * wc + 8 * nt + 2 * (lane & 3);
          const float v0 = i <= r && i >= lo ? acc[nt][2 * hf] : 0.f;
          const float v1 = i + 1 <= r && i + 1 >= lo ? acc[nt][2 * hf + 1] : 0.f;
          const uint32_t at = base + B::kP + r * 128 + (((uint32_t)(2 * wc + nt) ^ (uint32_t)(r & 7)) << 4) + ((lane & 3) << 2);
          const uint32_t h = pack_bf16(v0, v1);
          sts32(at, h);
          if (B::kExact) {
            const float2 f = unpack_bf16(h);
            sts32(at + kSlab, pack_bf16(v0 - f.x, v1 - f.y));
          }
        }
      }
    }
  }
  fence_proxy_async();
  __syncthreads();
  if (tid == 0) {
    bulk_store(a.blocks + ((long long)head * a.slots_per_head + local) * B::kBytes, base, B::kBytes);
    bulk_commit();
    bulk_wait_read<0>();
  }
}

// ---------------------------------------------------------------------------------------------
// The scan
// ---------------------------------------------------------------------------------------------
// Everything is computed with the value column as the M extent (tensor-memory lane = value column):
//   dS^T = V^T Kt              [128 value columns x dk]    A = V^T, B = Kt (shared memory)
//   O^T  = V^T P^T + Sb Qt^T   [128 x 64 rows]             A = V^T / Sb (tensor memory), B = P, Qt
// The fp32 state lives in the REGISTERS of the state group: per chunk it takes dS of the chunk before
// out of tensor memory, S <- D . (S + dS), and writes the copy Sb that the readout contracts with.  So
// no contraction but the readout depends on the state's trip, and dS, O and Sb each have two buffers:
// the tensor core works on dS and P V of a chunk while the state that enters it is being formed.  (With
// the state accumulated in tensor memory instead, the chain update -> scaling -> update took 2270
// cycles per chunk of dk = 64.)
// What bounds it at dk = 128: shared memory.  About 160 KiB go through it per pass (57 in by TMA, 72 read
// by the contractions, 32 for the output tile), 1300 of the pass's 1500 cycles at 128 bytes a clock; the
// value gate and the feed-through add 96 KiB (2500 cycles a pass).  Twice as many state warps, or dS of
// the next pass issued before the readout of this one, change nothing or cost 2 to 4 %.
// Roles: warp 0 loads, 1 issues the contractions, 2 sends the output tiles (and fetches the feed-
// through's), 3 prepares chunks of cut tiles, 4-11 state group (tensor-memory quarter = warp % 4, half
// of the key channels each), 12-15 outputs, 16-19 (BLOCK) apply the value gate to the v tile.
// Two rings: A (Kt, P and the v tile, free once P V is done) and Q (Qt and D).
template <int DK, bool BLOCK>
struct Scan {
  using B = Block<DK>;
  static constexpr int kABytes = B::kQ, kQBytes = B::kBytes - B::kQ;
  static constexpr int kAStages = DK == 128 && !BLOCK ? 3 : 2, kQStages = 3;
  static constexpr int kOffV = kABytes, kOffBeta = kOffV + 2 * kSlab;
  static constexpr int kAStage = kOffBeta + (BLOCK ? 2 * kSlab : 0);
  static constexpr int kOffQ = kAStages * kAStage;
  static constexpr int kOffOt = kOffQ + kQStages * kQBytes;  // two output tiles of two slabs
  static constexpr int kOffDc = kOffOt + 4 * kSlab;          // float [8][DK]: decays of chunks of cut tiles
  static constexpr int kOffBar = kOffDc + 8 * DK * 4;
  static constexpr int kOffCtl = kOffBar + 48 * 8;
  static constexpr int kSmem = kOffCtl + 512 + 1024;         // + slack for 1024-byte alignment
  static constexpr int kThreads = BLOCK ? 640 : 512;
  // dk = 64: the high and middle parts of Kt lie one behind the other in shared memory and are taken as
  // one operand with N = 128 (64 cycles instead of 2 x 48, and half the instructions); dS is then a pair
  // of accumulators, added when it is read.  (P and Qt the same way would leave room for one O buffer
  // only: 2080 cycles per chunk instead of 1740.)
  static constexpr uint32_t kColS = 0, kDsCols = 128, kColO = 256, kColSb = 384, kSbCols = 64;
  static_assert(kSmem <= 232448, "shared memory budget");
};

enum { FB_AFULL0 = 0,                   // [3] Kt, P, v landed                          (1 + bytes)
       FB_AEMPTY0 = 3,                  // [3] their contractions are done              (1 + warp 3)
       FB_QFULL0 = 6,                   // [3] Qt, D landed                             (1 + bytes)
       FB_QEMPTY0 = 9,                  // [3] readout done, D read                     (outputs' warp 12 + 8 warps)
       FB_VREADY0 = 12,                 // [3] value gate applied                       (4 warps)
       FB_SREADY0 = 15, FB_SREADY1,     // state entering the chunk is in tensor memory, Qt landed (8 warps)
       FB_SFULL0, FB_SFULL1,            // dS complete                                  (1)
       FB_OFULL0, FB_OFULL1,            // outputs complete                             (1)
       FB_OFREE0, FB_OFREE1,            // outputs read from tensor memory              (4 warps)
       FB_OTFULL0, FB_OTFULL1,          // output tile written                          (4 warps)
       FB_OTFREE0, FB_OTFREE1,          // output tile's copies have read it            (1)
       FB_XFULL0, FB_XFULL1,            // feed-through tile landed in the output tile  (1 + bytes)
       FB_CUT0,                         // [8] a chunk of a cut tile is prepared        (1)
       FB_TAIL = FB_CUT0 + 8,           // the last tile's rows of v behind the end are zeros (1; tiles of one chunk)
       FB_DRAIN, FB_COUNT };
static_assert(FB_COUNT <= 48, "barrier count");

struct PassDesc {
  long long row;       // first row of the tile in v, o
  long long rowq;      // the same in q, k, x, y
  int lo, hi;          // rows of the chunk within the tile
  int flags;           // kLastPass, kCutTile, kTail
  int nr;              // rows of the tile
};
constexpr int kLastPass = 1, kCutTile = 2, kTail = 4;   // kTail: rows of another sequence follow
struct ScanCtl {
  uint32_t tmem_base;
  int pad;
  WaitCtl wait;
  int n_a, n_q, n_x;   // loads issued (for the clean exit)
  int pad2;
  PassDesc desc[8];    // pass & 7: the outputs may be a few passes behind the loads
  __align__(16) unsigned long long mask[16];   // of eight tiles, each beside a neighbour's
};
static_assert(sizeof(ScanCtl) <= 512 && offsetof(ScanCtl, mask) % 16 == 0, "control block");

struct ScanMaps {
  CUtensorMap v, beta, fx, o, o8, o1;
};

template <int DK, bool BLOCK, bool SPLIT>
__global__ void __launch_bounds__(Scan<DK, BLOCK>::kThreads, 1)
ddts_scan_kernel(const __grid_constant__ ScanMaps maps, const ScanArgs a) {
  using B = Block<DK>;
  using C = Scan<DK, BLOCK>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
  auto bar = [&](int i) { return base + C::kOffBar + 8u * (uint32_t)i; };
  volatile ScanCtl* ctl = reinterpret_cast<volatile ScanCtl*>(gbase + C::kOffCtl);
  volatile WaitCtl* wc = &ctl->wait;
  WorkspaceHeader* hdr = a.hdr;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q4 = warp & 3;

  // ---- the item
  unsigned item = blockIdx.x;
  int seg = 0;
  if constexpr (SPLIT) {
    const unsigned items = gridDim.x / (unsigned)a.seg_count;
    seg = (int)(item / items) + a.phase - 1;
    item %= items;
  }
  const bool only = SPLIT && a.phase == 1 && seg > 0;      // the final state and the decay, no outputs
  const int slice = (int)(item % (unsigned)a.cols);
  const int sh = (int)(item / (unsigned)a.cols), h = sh % a.H;
  int n = sh / a.H;
  const int hq = a.gate_heads == 1 ? 0 : h;
  long long row0, rowq0;
  int len, vrow0, vhead;       // (vhead, vrow0): first row as the maps of v and beta_hat count
  long long slot0;
  if (a.cu) {
    // (The plan ended before the operand kernel began.  A cu_seqlens that it has refused may leave blocks
    // unwritten: no tile of it is looked at.  Read here the verdict costs nothing; after the wait for the
    // operands it was 1.2 us of a small call, 24.6 us.)
    const bool refused = *(volatile int32_t*)&hdr->status == RODIMUS_ERR_SEQLENS;
    n = a.order[n];
    int lo, hi;
    seq_range(a.cu, n, a.T, lo, hi);
    len = refused ? 0 : hi - lo;
    row0 = (long long)h * a.T + lo;
    vhead = h;
    vrow0 = lo;
    rowq0 = (long long)hq * a.T + lo;
    slot0 = (long long)hq * a.slots_per_head + lo / kTile + n;
  } else {
    len = a.T;
    vhead = sh;
    vrow0 = 0;
    row0 = (long long)sh * a.T;
    rowq0 = ((long long)n * a.gate_heads + hq) * a.T;
    slot0 = ((long long)n * a.gate_heads + hq) * a.slots_per_head;
    if constexpr (SPLIT) {
      const int t0 = seg == 0 ? 0 : a.seg_tiles0 + (seg - 1) * a.seg_tiles;
      len = min(a.T, (a.seg_tiles0 + seg * a.seg_tiles) * kTile) - t0 * kTile;
      row0 += (long long)t0 * kTile;
      vrow0 = t0 * kTile;
      rowq0 += (long long)t0 * kTile;
      slot0 += t0;
    }
  }
  const int col0 = slice * 128;
  const int ntiles = (len + kTile - 1) / kTile;
  const long long state_off = ((long long)n * a.H + h) * DK * (long long)a.dv + col0;
  const long long states = (long long)a.n_seq * a.H * DK * a.dv, decays = (long long)a.n_seq * a.H * DK;
  const float* s0 = a.s0;
  float* sT = a.sT;
  if constexpr (SPLIT) {
    if (a.phase == 2) {
      s0 = a.seg_state + (seg - 1) * states;
      if (seg != a.seg_count) sT = nullptr;
    } else {
      if (only) s0 = nullptr;
      sT = a.seg_state + seg * states;
    }
  }

  if (tid == 0) {
    if (!a.cu && a.T == 0 && blockIdx.x == 0) hdr->status = RODIMUS_OK;   // (no operand kernel then)
    ctl->wait.abort_flag = 0;
    ctl->wait.limit = a.limit;
    ctl->n_a = ctl->n_q = ctl->n_x = 0;
    for (int i = 0; i < FB_COUNT; ++i) {
      int cnt = 1;
      if (i >= FB_QEMPTY0 && i < FB_QEMPTY0 + 3) cnt = 9;
      if (i >= FB_AEMPTY0 && i < FB_AEMPTY0 + 3) cnt = 2;
      if (i == FB_SREADY0 || i == FB_SREADY1) cnt = 8;
      if ((i >= FB_VREADY0 && i < FB_VREADY0 + 3) || i == FB_OFREE0 || i == FB_OFREE1 || i == FB_OTFULL0 || i == FB_OTFULL1)
        cnt = 4;
      mbar_init(bar(i), cnt);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(base + C::kOffCtl), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  wait_for_previous_kernel();   // the operands are there
  auto wait_all = [&](int b, uint32_t parity) -> bool {   // whole warps: tensor-memory accesses need them
    return __all_sync(0xffffffffu, mbar_wait(bar(b), parity, wc, hdr)) != 0;
  };

  if (warp == 0) {
    // ======================================= loads =========================================
    if (ntiles > 0 && elect_one()) {
      const unsigned char* blk = a.blocks + slot0 * B::kBytes;
      // Split calls: the chunk masks arrive seven tiles ahead, two to a copy of 16 bytes.  Fetched one tile ahead, a
      // mask kept this thread waiting for as long as L2 takes to answer, which was what a pass without readout took
      // (1570 cycles; 32 x 16384 tokens 429 -> 399 us).  A full pass takes as long anyway.
      const uint32_t masks = base + C::kOffCtl + (uint32_t)offsetof(ScanCtl, mask);
      auto ask_mask = [&](int t) {
        if (t < ntiles) copy_16_async(masks + 16 * (t & 7), a.masks + ((slot0 + t) & ~1ll));
        copies_commit();
      };
      unsigned long long next_mask = 0ull;
      if constexpr (SPLIT) {
        for (int t = 0; t < 7; ++t) ask_mask(t);
      } else {
        next_mask = __ldcg(a.masks + slot0);
      }
      uint32_t s = 0, ph = 1, qs = 0, qph = 1;
      int pass = 0;
      bool ok = true;
      for (int t = 0; ok && t < ntiles; ++t) {
        unsigned long long mask = next_mask;
        if constexpr (SPLIT) {
          ask_mask(t + 7);
          copies_wait<7>();
          mask = ctl->mask[2 * (t & 7) + (int)((slot0 + t) & 1)];
        } else if (t + 1 < ntiles) {
          next_mask = __ldcg(a.masks + slot0 + t + 1);
        }
        const int nr = min(kTile, len - t * kTile);
        for (int lo = 0; lo < nr; ++pass) {
          if (!(ok = mbar_wait(bar(FB_AEMPTY0 + s), ph, wc, hdr))) break;
          const int hi = chunk_end(mask, lo, nr);
          volatile PassDesc* d = &ctl->desc[pass & 7];
          const long long row = row0 + (long long)t * kTile;
          d->row = row;
          d->rowq = rowq0 + (long long)t * kTile;
          d->lo = lo;
          d->hi = hi;
          d->flags = (t + 1 == ntiles && hi == nr ? kLastPass : 0) | (mask != 1ull ? kCutTile : 0) | (a.cu && nr < kTile ? kTail : 0);
          d->nr = nr;
          const uint32_t st = base + s * C::kAStage, fb = bar(FB_AFULL0 + s);
          const bool beta = BLOCK && a.has_beta;
          const int a_bytes = only ? B::kP : C::kABytes;       // (Kt alone)
          mbar_expect_tx(fb, a_bytes + 2 * kSlab + (beta ? 2 * kSlab : 0));
          const int vrow = vrow0 + t * kTile;
          tma_load_4d(st + C::kOffV, &maps.v, 0, vrow, col0 >> 6, vhead, fb);
          if (beta) tma_load_4d(st + C::kOffBeta, &maps.beta, 0, vrow, col0 >> 6, vhead, fb);
          bulk_load(st, blk + (long long)t * B::kBytes, a_bytes, fb);
          ctl->n_a = pass + 1;
          if (lo == 0 && t + C::kAStages < ntiles) {   // asked into L2 before its stage is free
            tma_prefetch_4d(&maps.v, 0, vrow + C::kAStages * kTile, col0 >> 6, vhead);
            if (beta) tma_prefetch_4d(&maps.beta, 0, vrow + C::kAStages * kTile, col0 >> 6, vhead);
            if (BLOCK && a.feed_d && !only) tma_prefetch_3d(&maps.fx, 0, (int)row + C::kAStages * kTile, col0 >> 6);
          }
          if (++s == C::kAStages) { s = 0; ph ^= 1; }
          if (!(ok = mbar_wait(bar(FB_QEMPTY0 + qs), qph, wc, hdr))) break;
          const int q_skip = only ? B::kD - B::kQ : 0;         // (D alone)
          mbar_expect_tx(bar(FB_QFULL0 + qs), C::kQBytes - q_skip);
          bulk_load(base + C::kOffQ + qs * C::kQBytes + q_skip, blk + (long long)t * B::kBytes + B::kQ + q_skip, C::kQBytes - q_skip,
                    bar(FB_QFULL0 + qs));
          ctl->n_q = pass + 1;
          if (++qs == C::kQStages) { qs = 0; qph ^= 1; }
          lo = hi;
        }
      }
      if constexpr (SPLIT) copies_wait<0>();
    }
    __syncwarp();
  } else if (warp == 1) {
    // ==================================== contractions =====================================
    if (ntiles > 0 && elect_one()) {
      constexpr uint32_t kIs = make_idesc(128, 128, 1, 1);   // dS^T = V^T Kt
      constexpr uint32_t kIv = make_idesc(128, 64, 1, 0);   // O^T  = V^T P^T
      constexpr uint32_t kIq = make_idesc(128, 64, 0, 0);   // O^T += Sb Qt^T, A in tensor memory
      uint32_t s = 0, ph = 0, qs = 0;
      int n_cut = 0;
      for (int c = 0;; ++c) {
        if (!mbar_wait(bar(FB_AFULL0 + s), ph, wc, hdr)) break;
        if (BLOCK && a.has_beta && !mbar_wait(bar(FB_VREADY0 + s), ph, wc, hdr)) break;
        const int flags = ctl->desc[c & 7].flags;
        if (flags & kCutTile) {
          if (!mbar_wait(bar(FB_CUT0 + (n_cut & 7)), (n_cut >> 3) & 1, wc, hdr)) break;
          ++n_cut;
        } else if ((flags & kTail) && !(BLOCK && a.has_beta)) {
          if (!mbar_wait(bar(FB_TAIL), 0, wc, hdr)) break;
        }
        const uint32_t st = base + s * C::kAStage, sq = base + C::kOffQ + qs * C::kQBytes;
        const uint32_t dv = desc_lo_mnmajor(st + C::kOffV, kSlab);
        // (no readout in between: the state group has taken dS of two chunks before when it reports for the last)
        if (only && c > 0 && !mbar_wait(bar(FB_SREADY0 + ((c - 1) & 1)), ((c - 1) >> 1) & 1, wc, hdr)) break;
        tc_fence_after();
        // dS (buffer c & 1: the state group has taken dS of two chunks before, or the readout of the
        // chunk before could not have been issued)
        {
          const uint32_t d = tmem + C::kColS + (c & 1) * C::kDsCols;
          const uint32_t dk = desc_lo_mnmajor(st + B::kK, kSlab);       // 128 channels, or high and middle parts
          umma_bf16_lo<false>(d, dv, dk, kIs);
#pragma unroll
          for (int kk = 1; kk < 4; ++kk) umma_bf16_lo<true>(d, dv + 128 * kk, dk + 128 * kk, kIs);
          if (B::kExact) {
            const uint32_t dl = desc_lo_mnmajor(st + B::kK + 2 * kSlab, kSlab);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma_bf16_lo<true>(d + 64, dv + 128 * kk, dl + 128 * kk, make_idesc(128, 64, 1, 1));
          }
        }
        umma_commit(bar(FB_SFULL0 + (c & 1)));
        if (only) {
          if (flags & kLastPass) break;        // (nobody would wait for that commit: it could arrive after the CTA's end)
          umma_commit(bar(FB_AEMPTY0 + s));
          if (++s == C::kAStages) { s = 0; ph ^= 1; }
          continue;
        }
        if (!mbar_wait(bar(FB_OFREE0 + (c & 1)), ((c >> 1) & 1) ^ 1, wc, hdr)) break;
        tc_fence_after();
        const uint32_t o = tmem + C::kColO + (c & 1) * 64, sb = tmem + C::kColSb + (c & 1) * C::kSbCols;
#pragma unroll
        for (int p = 0; p < B::kQp; ++p) {
          const uint32_t dp = desc_lo_kmajor(st + B::kP + p * kSlab);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            if (p == 0 && kk == 0) umma_bf16_lo<false>(o, dv, dp, kIv);
            else umma_bf16_lo<true>(o, dv + 128 * kk, dp + 2 * kk, kIv);
          }
        }
        umma_commit(bar(FB_AEMPTY0 + s));
        if (!mbar_wait(bar(FB_SREADY0 + (c & 1)), (c >> 1) & 1, wc, hdr)) break;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < DK / 16; ++kk)
          umma_bf16_atmem<true>(o, sb + 8 * kk, desc_lo_kmajor(sq + (kk >> 2) * kSlab) + 2 * (kk & 3), kIq);
        if (B::kExact) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)                     // high part of the state x low part of Qt
            umma_bf16_atmem<true>(o, sb + 8 * kk, desc_lo_kmajor(sq + kSlab) + 2 * kk, kIq);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)                     // low x high
            umma_bf16_atmem<true>(o, sb + 32 + 8 * kk, desc_lo_kmajor(sq) + 2 * kk, kIq);
        }
        umma_commit(bar(FB_OFULL0 + (c & 1)));
        if (flags & kLastPass) break;
        if (++s == C::kAStages) { s = 0; ph ^= 1; }
        if (++qs == C::kQStages) qs = 0;
      }
    }
    __syncwarp();
  } else if (warp == 2 && !only) {
    // ================================= output tiles to global ==============================
    // Feed-through: the x' tile of a pass is fetched INTO its output tile, to be combined with the
    // accumulators in place; two passes ahead, as soon as the copies have read that tile (one pass ahead
    // a fetch and a store were on the way of every pass: 2.7 us a tile instead of 1.2).
    const bool feed = BLOCK && a.feed_d != nullptr;
    int xt = 0, xlo = 0;                               // tile and first row of the next chunk to fetch for
    auto mask_of = [&](int t) { return __ldcg(a.masks + slot0 + t); };
    unsigned long long xmask = feed && ntiles > 0 ? mask_of(0) : 0ull;
    auto fetch_x = [&](int c) {
      if (xt >= ntiles) return;
      if (elect_one()) {
        mbar_expect_tx(bar(FB_XFULL0 + (c & 1)), 2 * kSlab);
        tma_load_3d(base + C::kOffOt + (c & 1) * 2 * kSlab, &maps.fx, 0, (int)(row0 + (long long)xt * kTile), col0 >> 6,
                    bar(FB_XFULL0 + (c & 1)));
        ctl->n_x = c + 1;
      }
      __syncwarp();
      const int nr = min(kTile, len - xt * kTile);
      xlo = chunk_end(xmask, xlo, nr);
      if (xlo == nr) {
        xlo = 0;
        if (++xt < ntiles) xmask = mask_of(xt);
      }
    };
    if (feed) {
      fetch_x(0);
      fetch_x(1);
    }
    for (int c = 0; ntiles > 0; ++c) {
      const uint32_t pr = c & 1;
      const uint32_t ot = base + C::kOffOt + pr * 2 * kSlab;
      if (!wait_all(FB_OTFULL0 + pr, (c >> 1) & 1)) break;
      const volatile PassDesc* d = &ctl->desc[c & 7];
      const long long row = d->row;
      const int lo = d->lo, hi = d->hi;
      const bool last = (d->flags & kLastPass) != 0;
      if (lo == 0 && hi == kTile) {
        if (elect_one()) {
          tma_store_3d(&maps.o, 0, (int)row, col0 >> 6, ot);
          bulk_commit();
          bulk_wait_read<0>();
        }
      } else {
        // part of a tile: boxes of 8 rows and of 1 row, so that no other row is touched
        const int n8 = (hi - lo) >> 3, n1 = (hi - lo) & 7;    // at most 7 + 7 boxes per slab
        const int slab = lane & 1, v = lane >> 1;
        const int r = v < n8 ? lo + 8 * v : lo + 8 * n8 + (v - n8);
        if (v < n8) tma_store_2d(&maps.o8, col0 + 64 * slab, (int)row + r, ot + slab * kSlab + r * 128);
        else if (v < n8 + n1) tma_store_2d(&maps.o1, col0 + 64 * slab, (int)row + r, ot + slab * kSlab + r * 128);
        bulk_commit();
        bulk_wait_read<0>();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(FB_OTFREE0 + pr));
      if (last) break;
      if (feed) fetch_x(c + 2);
    }
  } else if (warp == 3) {
    // ======================= chunks of cut tiles, rows behind the end ======================
    // rows of other chunks contribute nothing to a chunk's update; the chunk's decays come from the
    // same additions as its operands'
    uint32_t s = 0, ph = 0;
    int n_cut = 0;
    for (int c = 0; ntiles > 0; ++c) {
      if (!wait_all(FB_AFULL0 + s, ph)) break;
      const volatile PassDesc* d = &ctl->desc[c & 7];
      const int lo = d->lo, hi = d->hi, flags = d->flags;
      if ((flags & kTail) && !(BLOCK && a.has_beta)) {
        const uint32_t v = base + s * C::kAStage + C::kOffV;
#pragma unroll 4
        for (int at = d->nr * 128 + lane * 16; at < kSlab; at += 512) {
          sts128(v + at, 0u, 0u, 0u, 0u);
          sts128(v + kSlab + at, 0u, 0u, 0u, 0u);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0 && !(flags & kCutTile)) mbar_arrive(bar(FB_TAIL));
      }
      if (flags & kCutTile) {
        const uint32_t k = base + s * C::kAStage + B::kK;
        for (int e = lane; e < B::kKp * B::kSlabs * kTile * 8; e += 32) {
          const int r = (e >> 3) & (kTile - 1);
          if (r < lo || r >= hi) sts128(k + e * 16, 0u, 0u, 0u, 0u);
        }
        fence_proxy_async();
        // (eight buffers: this one's last reader, the state's trip eight passes back, precedes the
        // contractions whose end let the tile of this pass in)
        float* dc = reinterpret_cast<float*>(gbase + C::kOffDc) + (n_cut & 7) * DK;
        for (int ch = lane; ch < DK; ch += 32) {
          const long long e = d->rowq * DK + ch;
          typename Decay<B::kExact>::One acc = {}, la;
          float lh;
          for (int r = lo; r < hi; ++r) {
            gate_pair<B::kExact>(__bfloat162float(a.gx[e + r * DK]), __bfloat162float(a.ty[e + r * DK]), a.ingate, la, lh);
            acc = sum1(acc, la);
          }
          dc[ch] = exp2_of(acc);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(FB_CUT0 + (n_cut & 7)));
        ++n_cut;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(FB_AEMPTY0 + s));
      if (flags & kLastPass) break;
      if (++s == C::kAStages) { s = 0; ph ^= 1; }
    }
  } else if (warp >= 4 && warp < 12) {
    // ======================================= state =========================================
    constexpr int kHalf = DK / 2;
    const int ch0 = ((warp - 4) >> 2) * kHalf;
    const uint32_t t_lane = tmem + ((uint32_t)(q4 * 32) << 16);
    // element (channel d, own value column) of the state: off + d * dv
    const long long off = state_off + q4 * 32 + lane + (long long)ch0 * a.dv;
    float2 S[kHalf / 2];
#pragma unroll
    for (int e = 0; e < kHalf / 2; ++e) {
      S[e] = make_float2(0.f, 0.f);
      if constexpr (SPLIT) {
        if (s0) S[e] = make_float2(__ldcg(s0 + off + (long long)(2 * e) * a.dv), __ldcg(s0 + off + (long long)(2 * e + 1) * a.dv));
      } else {
        if (a.s0) S[e] = make_float2(__ldg(a.s0 + off + (long long)(2 * e) * a.dv), __ldg(a.s0 + off + (long long)(2 * e + 1) * a.dv));
      }
    }
    uint32_t qs = 0, qph = 0;
    int n_cut = 0;
    bool ok = true;
    // S <- D . (S + dS) with dS and D of pass c
    auto advance = [&](int c, const float* D) {
      constexpr int kLd = BLOCK ? 16 : 32;              // (fewer registers a thread with 20 warps)
#pragma unroll
      for (int piece = 0; piece < kHalf / kLd; ++piece) {
        uint32_t r[kLd];
        const uint32_t ds = t_lane + C::kColS + (c & 1) * C::kDsCols + ch0 + kLd * piece;
        if constexpr (kLd == 16) tmem_ld16(ds, r);
        else tmem_ld32(ds, r);
        if constexpr (B::kExact) {
          uint32_t r2[32];
          tmem_ld32(ds + 64, r2);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(r2[e]));
        } else {
          tmem_ld_wait();
        }
#pragma unroll
        for (int e = 0; e < kLd / 4; ++e) {
          const float4 d = *reinterpret_cast<const float4*>(D + ch0 + kLd * piece + 4 * e);   // broadcast
          float2* x = S + kLd / 2 * piece + 2 * e;
          x[0] = __fmul2_rn(__fadd2_rn(x[0], make_float2(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]))), make_float2(d.x, d.y));
          x[1] = __fmul2_rn(__fadd2_rn(x[1], make_float2(__uint_as_float(r[4 * e + 2]), __uint_as_float(r[4 * e + 3]))), make_float2(d.z, d.w));
        }
      }
    };
    if (ntiles > 0) {
      for (int c = 0;; ++c) {
        // the state entering pass c, as bf16 parts (the readout of pass c - 2, the buffer's last reader,
        // precedes dS of pass c - 1 in the tensor pipe)
        const uint32_t t_sb = t_lane + C::kColSb + (c & 1) * C::kSbCols + ch0 / 2;
#pragma unroll
        for (int piece = 0; piece < kHalf / 32; ++piece) {
          if (only) break;
          uint32_t w[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) w[e] = pack_bf16(S[16 * piece + e].x, S[16 * piece + e].y);
          tmem_st16(t_sb + 16 * piece, w);
          if (B::kExact) {
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const float2 f = unpack_bf16(w[e]);
              w[e] = pack_bf16(S[16 * piece + e].x - f.x, S[16 * piece + e].y - f.y);
            }
            tmem_st16(t_sb + DK / 2 + 16 * piece, w);
          }
        }
        if (!(ok = wait_all(FB_QFULL0 + qs, qph))) break;   // (for the readout as well)
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(FB_SREADY0 + (c & 1)));
        const int flags = ctl->desc[c & 7].flags;
        const float* D = reinterpret_cast<const float*>(gbase + C::kOffQ + qs * C::kQBytes + (B::kD - B::kQ));
        if (flags & kCutTile) {
          if (!(ok = wait_all(FB_CUT0 + (n_cut & 7), (n_cut >> 3) & 1))) break;
          D = reinterpret_cast<const float*>(gbase + C::kOffDc) + (n_cut & 7) * DK;
          ++n_cut;
        }
        if ((flags & kLastPass) && !sT) break;
        if (!(ok = wait_all(FB_SFULL0 + (c & 1), (c >> 1) & 1))) break;
        tc_fence_after();
        advance(c, D);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(FB_QEMPTY0 + qs));
        if (flags & kLastPass) break;
        if (++qs == C::kQStages) { qs = 0; qph ^= 1; }
      }
    }
    if (ok && sT) {
#pragma unroll
      for (int e = 0; e < kHalf / 2; ++e) {
        sT[off + (long long)(2 * e) * a.dv] = S[e].x;
        sT[off + (long long)(2 * e + 1) * a.dv] = S[e].y;
      }
    }
  } else if (only && warp == 12) {
    // ============================== the segment's decay ====================================
    float prod[DK / 32];
#pragma unroll
    for (int i = 0; i < DK / 32; ++i) prod[i] = 1.f;
    uint32_t qs = 0, qph = 0;
    int n_cut = 0;
    for (int c = 0; ntiles > 0; ++c) {
      if (!wait_all(FB_QFULL0 + qs, qph)) break;
      const int flags = ctl->desc[c & 7].flags;
      const float* D = reinterpret_cast<const float*>(gbase + C::kOffQ + qs * C::kQBytes + (B::kD - B::kQ));
      if (flags & kCutTile) {
        if (!wait_all(FB_CUT0 + (n_cut & 7), (n_cut >> 3) & 1)) break;
        D = reinterpret_cast<const float*>(gbase + C::kOffDc) + (n_cut & 7) * DK;
        ++n_cut;
      }
#pragma unroll
      for (int i = 0; i < DK / 32; ++i) prod[i] *= D[lane + 32 * i];
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(FB_QEMPTY0 + qs));
      if (flags & kLastPass) break;
      if (++qs == C::kQStages) { qs = 0; qph ^= 1; }
    }
    if (slice == 0) {
      float* d = a.seg_decay + (seg - 1) * decays + ((long long)n * a.H + h) * DK + lane;
#pragma unroll
      for (int i = 0; i < DK / 32; ++i) d[32 * i] = prod[i] < FLT_MIN ? FLT_MIN : prod[i];
      // (no decay is zero: an infinite state stays infinite over any number of steps, and is no NaN behind a segment)
    }
  } else if (!only && warp >= 12 && warp < 16) {
    // ====================================== outputs ========================================
    // O^T has the value columns in the tensor-memory lanes.  The 16x256b load hands out 8x8 fragments
    // [value column][row]; stmatrix.trans writes them transposed into a tile of two swizzled 64-column
    // slabs, which leaves through a tensor copy.  Two tiles alternate.
    const int mat_k = lane & 7, mat_h = (lane >> 3) & 1, mat_j = lane >> 4;
    const uint32_t t_lane = tmem + ((uint32_t)(q4 * 32) << 16);
    const bool feed = BLOCK && a.feed_d != nullptr;
    uint32_t qs = 0;
    for (int c = 0; ntiles > 0; ++c) {
      const uint32_t pr = c & 1, ph = (c >> 1) & 1;
      if (!wait_all(FB_OFULL0 + pr, ph)) break;
      if (warp == 12 && lane == 0) mbar_arrive(bar(FB_QEMPTY0 + qs));
      if (++qs == C::kQStages) qs = 0;
      tc_fence_after();
      const bool last = (ctl->desc[c & 7].flags & kLastPass) != 0;
      if (feed) {   // (asked for once the tile was free)
        if (!wait_all(FB_XFULL0 + pr, ph)) break;
      } else {
        if (!wait_all(FB_OTFREE0 + pr, ph ^ 1)) break;
      }
      // this thread addresses output row 8 * (2 jp + mat_j) + mat_k of column block mat_h
      const uint32_t ot_mat = base + C::kOffOt + pr * 2 * kSlab + (q4 >> 1) * kSlab + (mat_j * 8 + mat_k) * 128;
#pragma unroll 1
      for (int hv = 0; hv < 2; ++hv) {                  // lanes 0..15 / 16..31 of the quarter
        uint32_t r[32];
        tmem_ld_16x256b_x8(t_lane + ((uint32_t)(16 * hv) << 16) + C::kColO + pr * 64, r);
        tmem_ld_wait();
        if (hv == 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(FB_OFREE0 + pr));
        }
        const uint32_t chunk = (uint32_t)(4 * (q4 & 1) + 2 * hv + mat_h);
        const uint32_t dst = ot_mat + ((chunk ^ (uint32_t)mat_k) << 4);
        if (feed) {
          const float* dh = a.feed_d + h * (long long)a.dv + col0 + q4 * 32 + 16 * hv + (lane >> 2);
          const float d_lo = __ldg(dh), d_hi = __ldg(dh + 8);
#pragma unroll
          for (int jp = 0; jp < 4; ++jp) {
            uint32_t xf[4];
            ldmatrix_x4_trans(dst + jp * 16 * 128, xf);
#pragma unroll
            for (int mi = 0; mi < 4; ++mi) {            // (lo, j0) (hi, j0) (lo, j1) (hi, j1)
              const int ri = 4 * (2 * jp + (mi >> 1)) + 2 * (mi & 1);
              const float dd = (mi & 1) ? d_hi : d_lo;
              const float2 xv = unpack_bf16(xf[mi]);
              r[ri] = __float_as_uint(fmaf(dd, xv.x, __uint_as_float(r[ri])));
              r[ri + 1] = __float_as_uint(fmaf(dd, xv.y, __uint_as_float(r[ri + 1])));
            }
          }
        }
#pragma unroll
        for (int jp = 0; jp < 4; ++jp) {                // output rows 16 jp .. 16 jp + 15
          const int j0 = 2 * jp, j1 = 2 * jp + 1;
          stmatrix_x4_trans(dst + jp * 16 * 128,
                            pack_bf16(__uint_as_float(r[4 * j0]), __uint_as_float(r[4 * j0 + 1])),
                            pack_bf16(__uint_as_float(r[4 * j0 + 2]), __uint_as_float(r[4 * j0 + 3])),
                            pack_bf16(__uint_as_float(r[4 * j1]), __uint_as_float(r[4 * j1 + 1])),
                            pack_bf16(__uint_as_float(r[4 * j1 + 2]), __uint_as_float(r[4 * j1 + 3])));
        }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(FB_OTFULL0 + pr));
      if (last) break;
    }
  } else if (BLOCK && warp >= 16) {
    // ===================================== value gate ======================================
    // v becomes beta_hat . v in place (the exact product of two bf16 rounded once)
    uint32_t s = 0, ph = 0;
    for (int c = 0; a.has_beta && ntiles > 0; ++c) {
      if (!wait_all(FB_AFULL0 + s, ph)) break;
      const int flags = ctl->desc[c & 7].flags;
      const bool last = (flags & kLastPass) != 0;
      const uint32_t st = base + s * C::kAStage + C::kOffV + (tid - 512) * 16;
#pragma unroll 4
      for (int u = 0; u < 2 * kSlab / (128 * 16); ++u) {
        const uint32_t at = st + u * 128 * 16;
        const uint4 v = lds128(at), g = lds128(at + (C::kOffBeta - C::kOffV));
        sts128(at, hmul2_bf16(v.x, g.x), hmul2_bf16(v.y, g.y), hmul2_bf16(v.z, g.z), hmul2_bf16(v.w, g.w));
      }
      if (flags & kTail) {                               // rows behind the end, each thread those of its pieces
        const int nr = ctl->desc[c & 7].nr;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (((tid - 512) >> 3) + 16 * u >= nr) {
            sts128(st + u * 128 * 16, 0u, 0u, 0u, 0u);
            sts128(st + kSlab + u * 128 * 16, 0u, 0u, 0u, 0u);
          }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(FB_VREADY0 + s));
      if (last) break;
      if (++s == C::kAStages) { s = 0; ph ^= 1; }
    }
  }

  // ------------------------------------------ teardown ------------------------------------------
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (ctl->wait.abort_flag) {   // nothing may still be writing this CTA's shared or tensor memory
    if (tid == 0) {
      for (int back = 1; back <= C::kAStages && back <= ctl->n_a; ++back) {
        const int f = ctl->n_a - back;
        mbar_drain(bar(FB_AFULL0 + f % C::kAStages), (f / C::kAStages) & 1);
      }
      for (int back = 1; back <= C::kQStages && back <= ctl->n_q; ++back) {
        const int f = ctl->n_q - back;
        mbar_drain(bar(FB_QFULL0 + f % C::kQStages), (f / C::kQStages) & 1);
      }
      for (int back = 1; back <= 2 && back <= ctl->n_x; ++back) {
        const int f = ctl->n_x - back;
        mbar_drain(bar(FB_XFULL0 + (f & 1)), (f >> 1) & 1);
      }
    }
    if (warp == 1 && elect_one()) {   // a commit follows the contractions of the thread that makes it
      umma_commit(bar(FB_DRAIN));
      mbar_drain(bar(FB_DRAIN), 0);
    }
  }
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// Between the two launches of a split call: S_start(1) is state 0, S_start(k+1) = D_k . S_start(k) + dS_k takes the
// place of dS_k.  A thread per four columns of a row; `rows` = sequences x heads x dk.
constexpr int kJoinThreads = 256;
__global__ void __launch_bounds__(kJoinThreads) ddts_join_kernel(float* state, const float* decay, int G, long long rows, int dv) {
  wait_for_previous_kernel();
  const long long i = (long long)blockIdx.x * kJoinThreads + threadIdx.x;
  if (i >= rows * (dv / 4)) return;
  const long long row = i / (dv / 4), states = rows * dv;
  float4* at = reinterpret_cast<float4*>(state) + i;
  float4 S = __ldcg(at);
  for (int k = 1; k < G; k += 5) {          // (loads of five segments at a time)
    float4 x[5];
    float d[5];
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      if (k + u >= G) continue;
      x[u] = __ldcg(at + (k + u) * (states / 4));
      d[u] = __ldcg(decay + (k + u - 1) * rows + row);
    }
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      if (k + u >= G) continue;
      S = make_float4(fmaf(d[u], S.x, x[u].x), fmaf(d[u], S.y, x[u].y), fmaf(d[u], S.z, x[u].z), fmaf(d[u], S.w, x[u].w));
      __stcg(at + (k + u) * (states / 4), S);
    }
  }
}

template <int DK>
size_t blocks_bytes(long long slots) { return (size_t)slots * Block<DK>::kBytes; }

// Few (sequence, head, 128 columns) and long sequences: split along time.  The state recurrence is linear,
// S_end = D_seg . S_start + dS_seg, with dS_seg the segment's final state from a zero start and D_seg the product of
// its decays.  A dense call is cut into a head segment 0 and G equal segments 1..G, and scanned in two launches with a small one between:
//   phase 1   segment 0 as it stands; segments 1..G-1 from a zero state, without readout: dS and D
//   join      S_start(k+1) = D_k . S_start(k) + dS_k
//   phase 2   segments 1..G, each from its S_start
// The operands are formed once.  A pass without readout takes kStateOnly of a full one, and the head segment is that
// much shorter, so that phase 1 ends everywhere at once.
struct Segments {
  int G = 0;                  // 0: not split
  int tiles0 = 0, tiles = 0;  // of the head segment, of each later one (the last may be shorter)
};
constexpr int kMaxSegments = 16, kMinSegmentTiles = 8;
constexpr double kStateOnly = 0.4;

// As many segments as there is room for on the SMs, where the passes saved (0.8 us each) are worth more than 17 us, 20
// with two segments: two more launches, with a start and an end each, cost about that (one set of gates: two segments,
// dk = 128, 32 heads x 2589 tokens, 14 us, 43.0 us whole, 47.6 split, dk = 64, 4 x 8 x 4096, 21 us, 80.8 and 75.8;
// four segments, 16 x 2048, 17.5 us, 41.3 and 33.4, dv = 128 with gates per head 32 x 2048, 63.8 and 61.8).  Both sides
// measured, whole or split by the pair kernel against here (sets of gates x tokens, us):
//   one set of gates   dk = 64, 4 heads x 32768 468 -> 98, 16 x 8192 126 -> 75; dk = 128, 16 x 16384 226 -> 111
//   gates per head     dv = 256 8 x 2048 39 -> 33, 16 x 2048 49 -> 46, 4 x 4000 60 -> 35, 8 x 4096 109 -> 46,
//                      8 x 8192 130 -> 74, 4 x 32768 153 -> 129, 16 x 8192 140 -> 126, 32 x 4096 129 -> 122;
//                      no gain where the operands do not stay in L2: 10 x 32768 273 -> 270, 16 x 32768 409 -> 411,
//                      32 x 16384 358 -> 399.  With both block terms 16 x 32768 613 -> 541, 32 x 8192 305 -> 278;
//                      dv = 512 8 x 32768 408 -> 301, 16 x 16384 358 -> 288; dv = 128 16 x 16384 335 -> 191, but
//                      64 x 4096, two segments of operands from DRAM, 177 -> 183.  Below 4096 tokens the other side
//                      is not split: 37 x 4000, two segments, 132 -> 134, with block terms 159 -> 170, 32 x 3900
//                      with one set of gates 60.5 -> 61.6.
// The fewest items gain the most (one call, the other form against here, us): 1 x 4096 102 -> 28.5, 1 x 32768 133 -> 73,
// 2 x 16384 128 -> 54, 4 x 4096 103 -> 33, 4 x 6000 140 -> 40, 7 x 9000 132 -> 71, with both block terms 1 x 32768 180 ->
// 107, 7 x 9000 182 -> 92, one set of gates 7 x 9000 129 -> 43; dk = 64, one slice of 128 columns, 1985 tokens 40 -> 31,
// 32768 453 -> 84, three slices 547 -> 135.  (Their errors against fp64 are those of the other form: dk = 64, gates of
// slow to fast decay, final state 2.7e-7 to 8.4e-8 in both; dk = 128 1.5e-3 to 1.8e-3 in both.)
// Blocks of 86 MB (4 x 32768, 32 x 4096) are read back from L2 (126 MB) for the most part, those of 172 MB and more (16 x
// 16384) from DRAM; the line lies between.
constexpr size_t kStaysInL2 = (size_t)136 << 20;

Segments plan_segments(const rodimus_ddts_fwd_params& p, int sms) {
  Segments s;
  if (p.cu_seqlens || p.cu_seqlens_host) return s;
  const long long items = (long long)p.B * p.H * (p.dv / 128), tiles = (p.T + kTile - 1) / kTile;
  if (items <= 0) return s;
  const int g = (int)std::min<long long>(std::min<long long>(sms / items, kMaxSegments), tiles / kMinSegmentTiles);
  if (g < 2 || 0.8 * tiles * (1.0 - (1.0 + kStateOnly) / (g + kStateOnly)) < (g == 2 ? 20.0 : 17.0)) return s;
  if (p.dk == 128 && !p.shared_gates && (size_t)(p.B * (long long)p.H * tiles) * Block<128>::kBytes > kStaysInL2) {
    if (p.dv == 256 && !p.beta_hat && !p.feed_d) return s;
    if (p.dv % 256 && g == 2) return s;
  }
  if (p.dk == 128 && p.dv % 256 == 0 && g == 2 && p.T < 4096) return s;
  const int each = (int)std::ceil(tiles / (g + kStateOnly));
  const long long first = tiles - (long long)g * each;
  s.tiles0 = first > 0 ? (int)first : 1;
  s.tiles = (int)((tiles - s.tiles0 + g - 1) / g);
  s.G = (int)((tiles - s.tiles0 + s.tiles - 1) / s.tiles);
  return s;
}

struct ScanPlan {
  long long slots;        // tiles, over all sets of gates
  int slots_per_head, gate_heads;
  Segments seg;
  size_t blocks, masks, seg_state, seg_decay, bytes;   // workspace: offsets of the blocks, masks, segments' states and decays; total
};

ScanPlan scan_plan(const rodimus_ddts_fwd_params& p, const Segments& seg) {
  ScanPlan s;
  const bool varlen = p.cu_seqlens || p.cu_seqlens_host;
  s.gate_heads = p.shared_gates ? 1 : p.H;
  s.slots_per_head = varlen ? p.T / kTile + p.N : (p.T + kTile - 1) / kTile;
  s.slots = (long long)s.slots_per_head * s.gate_heads * (varlen ? 1 : p.B);
  size_t order = (size_t)(varlen ? p.N : 0) * sizeof(int32_t);
  s.blocks = sizeof(WorkspaceHeader) + ((order + 1023) & ~(size_t)1023);
  s.bytes = s.blocks + (p.dk == 64 ? blocks_bytes<64>(s.slots) : blocks_bytes<128>(s.slots));
  s.masks = s.bytes;
  s.bytes += ((size_t)s.slots * sizeof(unsigned long long) + 255) & ~(size_t)255;
  s.seg = seg;
  s.seg_state = s.bytes;
  const size_t per = (size_t)p.B * p.H * p.dk * sizeof(float);
  s.seg_decay = s.seg_state + (size_t)s.seg.G * per * p.dv;
  if (s.seg.G > 0) s.bytes = s.seg_decay + (size_t)(s.seg.G - 1) * per;
  return s;
}

template <int DK, bool BLOCK>
cudaError_t launch_scan(const ScanMaps& m, ScanArgs& a, long long slots, long long items, int dev, cudaStream_t st, int* n_launches) {
  static std::atomic<unsigned long long> opted_ops{0}, opted{0}, opted_split{0};   // per instantiation
  using C = Scan<DK, BLOCK>;
  cudaError_t e = opt_in_shared_memory(ddts_operands_kernel<DK>, kOpSmem<DK>, dev, opted_ops);
  if (e == cudaSuccess) e = a.seg_count ? opt_in_shared_memory(ddts_scan_kernel<DK, BLOCK, true>, C::kSmem, dev, opted_split)
                                        : opt_in_shared_memory(ddts_scan_kernel<DK, BLOCK, false>, C::kSmem, dev, opted);
  if (e != cudaSuccess) return e;
  if (slots > 0) {
    ddts_operands_kernel<DK><<<(unsigned)slots, kOpThreads, kOpSmem<DK>, st>>>(a);
    ++*n_launches;
    // The scan may start while the operand kernel's last CTAs run: it sets up (barriers, tensor memory)
    // and waits for that kernel before it reads a block.
    if (a.seg_count) {
      const unsigned grid = (unsigned)(items * a.seg_count);
      const long long rows = (long long)a.n_seq * a.H * DK;
      a.phase = 1;
      e = launch_overlapped(ddts_scan_kernel<DK, BLOCK, true>, grid, C::kThreads, C::kSmem, st, m, a);
      if (e == cudaSuccess)
        e = launch_overlapped(ddts_join_kernel, (unsigned)((rows * (a.dv / 4) + kJoinThreads - 1) / kJoinThreads), kJoinThreads, 0, st,
                              a.seg_state, a.seg_decay, a.seg_count, rows, a.dv);
      a.phase = 2;
      if (e == cudaSuccess) e = launch_overlapped(ddts_scan_kernel<DK, BLOCK, true>, grid, C::kThreads, C::kSmem, st, m, a);
      *n_launches += 3;
    } else {
      e = launch_overlapped(ddts_scan_kernel<DK, BLOCK, false>, (unsigned)items, C::kThreads, C::kSmem, st, m, a);
      ++*n_launches;
    }
  } else {
    // No tokens: what is in front now is the plan of the sequences, whose order the scan reads before it
    // waits for anything.  So it starts when that has ended.
    ddts_scan_kernel<DK, BLOCK, false><<<(unsigned)items, C::kThreads, C::kSmem, st>>>(m, a);
    ++*n_launches;
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

namespace {
// One set of gates for all heads, against the pair kernel: microseconds of both for rows of `tiles` tiles in
// each of n_seq sequences, `slabs` of 256 value columns that share a set, on `sms` SMs.  A pair of SMs takes
// 3 us for the start and end of an item and 2.3 us a tile, two CTAs of the scan 5.2 and 1.1, and the operands
// of a tile, formed once for all slabs, 2.2 us of such a pair.  (Fitted to 99 shapes of 2 to 16 slabs, 16 to
// 2048 tokens and 8 to 4096 sequences; at none does the choice cost more than 4 %.  64 sequences of 1024
// tokens, 4 slabs: pair 158 us, scan 115; 4096 of 1 to 16 tokens: 1629 and 1905.)
bool scan_pays_with_shared_gates(long long n_seq, double tiles, double slabs, bool varlen, int sms) {
  const double rounds = 2.0 * (double)n_seq * slabs / sms;
  const double pair = 6.0 + 3.0 * rounds + 2.3 * tiles * (varlen ? rounds : std::ceil(rounds));
  const double scan = 5.2 * rounds + tiles * rounds * (1.1 + 2.2 / slabs);
  return scan < pair;
}
}  // namespace

namespace {
// What the kernels of this file can compute at all.
bool scan_supported(const rodimus_ddts_fwd_params& p) {
  if (p.dtype != RODIMUS_BF16 || p.value_decay || p.dv % 128) return false;
  const bool block = p.beta_hat || p.feed_d;
  return p.dk == 64 ? !block : p.dk == 128 && (p.dv % 256 == 0 || (!block && !p.shared_gates));
}
}  // namespace

// Which requests this file's kernels compute unsplit, given room for the tiles' blocks; bytes of that room
// (0: not this path).  All timings are one call, the other kernel against this path.
//   dk = 64            always (B=4 H=16 T=2048, one set of gates: fp32 CUDA-core kernel 3.9 ms, here
//                      47 us; 20000 sequences of 1 to 8 tokens 29 -> 12 ms); not with block terms, whose
//                      products the fp32 kernel does not round.
//   one set of gates   where the pair kernel would be the other choice (same precision), by the cost of both
//                      (above); layer shape 82 -> 40 us.
//   gates per head     the gates cost the same in both, here their operands travel through memory, and
//                      here they are formed by all SMs however few the heads are.
//       dv % 256 == 0  against the pair kernel.  Dense, up to one item of 256 columns for every two SMs: the
//                      scan starts and ends sooner, and with the block's terms it takes less a tile;
//                      without them less only up to a quarter as many items as SMs.  Items x rows, us:
//                      16 x 2048 72 -> 47, 37 x 2048 74 -> 73, 48 x 333 22.6 -> 20.5, 48 x 777 37 -> 39, 64 x
//                      64 11.8 -> 11.4, 64 x 192 15.8 -> 16.3, 64 x 2048 77 -> 103; with both block terms 64
//                      x 64 12.8 -> 12.4, 48 x 333 29.6 -> 24.6, 64 x 2048 127 -> 124, 74 x 777 63.6 ->
//                      64.2; with one 64 x 240 21.3 -> 19.2, 64 x 1000 60 -> 62.
//                      Packed, whose longest sequence keeps the other pairs waiting, three eighths as many
//                      as SMs, of four tiles or more on average (56 items of 64..1000 rows 45 -> 40 us, of
//                      1..4096 135 -> 123; 72 items 45 -> 49 and 138 -> 143).  Packed sequences of one
//                      length would change sides sooner: 56 items of 300 rows 24.6 either way, of 1500
//                      64 -> 80.
//       odd multiples  against the single-CTA kernel, from four tiles on; it forms the gates in every CTA and
//       of 128         takes the same time for one item and for one on every SM.  Dense: up to three sets of gates
//                      for four CTAs of its rounds (T=2048, dv=128: 100 items 141 -> 131 us, 148 144 ->
//                      181, 149 274 -> 201, 256 280 -> 307; dv=384, three slices a set, always: 64 sets x
//                      1000 150 -> 73).  Packed: one slice a set, up to seven items for eight SMs (128
//                      items of 64..1000 rows 72 -> 60, of 650 62 -> 69, 148 of 650 62 -> 78), more slices,
//                      up to one for every SM.
size_t fwd_scan_workspace_bytes(const rodimus_ddts_fwd_params& p) {
  if (!scan_supported(p)) return 0;
  const bool varlen = p.cu_seqlens || p.cu_seqlens_host;
  const bool block = p.beta_hat || p.feed_d, whole = p.dv % 256 == 0;
  const long long n_seq = varlen ? p.N : p.B, sets = n_seq * p.H, items = sets * (p.dv / 128);
  int dev = 0, sms = 0;
  if (current_device(&dev, &sms) != cudaSuccess) {
    cudaGetLastError();
    sms = 0;
  }
  if (p.dk == 128) {
    if (sms == 0 || items == 0) return 0;
    if (p.shared_gates) {
      const double tiles = varlen ? (double)p.T / ((double)n_seq * kTile) + 0.5 : (double)((p.T + kTile - 1) / kTile);
      if (!scan_pays_with_shared_gates(n_seq, tiles, p.H * (p.dv / 256.0), varlen, sms)) return 0;
    } else {
      if (whole && !varlen) {
        const double fill = (double)items / sms, tiles = (double)((p.T + kTile - 1) / kTile);
        const double more = !block ? 2.8 * fill - 1.47 : (p.beta_hat && p.feed_d ? 1.95 * fill - 1.65 : 2.2 * fill - 1.6);
        if (fill > 1.0 || tiles * more > (block ? 3.0 : 3.5)) return 0;   // us of a tile more; of a call less
      } else if (p.T / (varlen ? n_seq : 1) < 4 * kTile) {
        return 0;
      } else if (whole) {
        if (4 * items > 3 * sms) return 0;
      } else if (varlen) {
        if (block || (p.dv == 128 ? 8 * items > 7 * sms : items > sms)) return 0;
      } else if (block || 4 * sets > 3 * sms * ((items + sms - 1) / sms)) {
        return 0;
      }
    }
  }
  const ScanPlan s = scan_plan(p, Segments{});
  if (s.slots > 0x7fffffffLL || items > 0x7fffffffLL) return 0;
  return s.bytes;
}

size_t fwd_scan_split_workspace_bytes(const rodimus_ddts_fwd_params& p) {
  if (!scan_supported(p)) return 0;
  int dev = 0, sms = 0;
  if (current_device(&dev, &sms) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const Segments seg = plan_segments(p, sms);
  if (seg.G == 0) return 0;
  const ScanPlan s = scan_plan(p, seg);
  return s.slots > 0x7fffffffLL ? 0 : s.bytes;
}

cudaError_t launch_fwd_scan(const rodimus_ddts_fwd_params& p, int* n_launches) {
  *n_launches = 0;
  int dev = 0, sms = 0;
  cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  ScanPlan s = scan_plan(p, plan_segments(p, sms));
  if (p.workspace_bytes < s.bytes) s = scan_plan(p, Segments{});   // room for the blocks alone
  const long long n_seq = p.cu_seqlens ? p.N : p.B, items = n_seq * p.H * (p.dv / 128);
  if (items == 0) return cudaSuccess;
  char* ws = reinterpret_cast<char*>(p.workspace);
  ScanArgs a;
  a.q = (const __nv_bfloat16*)p.q; a.k = (const __nv_bfloat16*)p.k;
  a.gx = (const __nv_bfloat16*)p.gate_x; a.ty = (const __nv_bfloat16*)p.temp_y;
  a.s0 = p.s0; a.sT = p.sT; a.feed_d = p.feed_d;
  a.blocks = reinterpret_cast<unsigned char*>(ws + s.blocks);
  a.masks = reinterpret_cast<unsigned long long*>(ws + s.masks);
  a.cu = p.cu_seqlens;
  a.order = reinterpret_cast<const int32_t*>(ws + sizeof(WorkspaceHeader));
  a.hdr = reinterpret_cast<WorkspaceHeader*>(ws);
  a.H = p.H; a.T = p.T; a.dv = p.dv; a.n_seq = (int)n_seq;
  a.gate_heads = s.gate_heads;
  a.slots_per_head = s.slots_per_head;
  a.cols = p.dv / 128;
  a.has_beta = p.beta_hat != nullptr;
  a.scale = p.scale; a.ingate = p.ingate;
  a.limit = main_loop_wait_cycles();
  a.seg_count = s.seg.G; a.seg_tiles0 = s.seg.tiles0; a.seg_tiles = s.seg.tiles;
  a.phase = 0;
  a.seg_state = reinterpret_cast<float*>(ws + s.seg_state);
  a.seg_decay = reinterpret_cast<float*>(ws + s.seg_decay);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(p.stream);
  ScanMaps m;
  const uint64_t rows = (uint64_t)p.B * p.H * p.T, dv = (uint64_t)p.dv;
  if (rows > 0) {
    const uint64_t heads = (uint64_t)p.B * p.H, T = (uint64_t)p.T;
    if (!encode_bf16_heads_map(&m.v, p.v, heads, T, dv, kTile, 2) || !encode_bf16_slab_map(&m.o, p.o, rows, dv, 2) ||
        !encode_bf16_map(&m.o8, p.o, rows, dv, 8) || !encode_bf16_map(&m.o1, p.o, rows, dv, 1))
      return cudaErrorInvalidValue;
    m.beta = m.fx = m.v;
    if (p.beta_hat && !encode_bf16_heads_map(&m.beta, p.beta_hat, heads, T, dv, kTile, 2)) return cudaErrorInvalidValue;
    if (p.feed_x && !encode_bf16_slab_map(&m.fx, p.feed_x, rows, dv, 2)) return cudaErrorInvalidValue;
  } else {
    memset(&m, 0, sizeof(m));   // never used: no tiles
  }
  const long long slots = rows > 0 ? s.slots : 0;
  if (p.dk == 64) return launch_scan<64, false>(m, a, slots, items, dev, st, n_launches);
  if (p.beta_hat || p.feed_d) return launch_scan<128, true>(m, a, slots, items, dev, st, n_launches);
  return launch_scan<128, false>(m, a, slots, items, dev, st, n_launches);
}

}  // namespace ddts
