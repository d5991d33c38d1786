// Sliding-window shared-key attention on tcgen05 (bf16 tokens, head size 128):
//   s_ti = scale <q^h_t, k_i>,  t - W < i <= t      p_ti = softmax_i(s_ti)      o^h_t = sum_i p_ti v^h_i
// (Sec. "Shared-Key Attention for Lossless Head Compression": one key per token for all heads.)
//
// An item is (batch, head, 128 queries).  A CTA - 4 softmax warps, one warp that issues the contractions and one
// that issues the TMA loads - takes items one after another: near the end of one it asks the hardware's scheduler
// for a launch that has not begun and does that work itself (clusterlaunchcontrol), so that the loads and the first
// scores of the next item are on their way while the last rows of this one are divided and stored.  (A CTA per
// item: 65.2 us at the layer shape, 37.0 with a window of 128 over 8 x 16 x 1024; this way 60.2 and 28.9.  Asked
// for at the START of an item the next one is dealt out before anybody knows who will be done first: 16 heads x
// 5001 tokens, window 2048, 72.9 us, 68.7 now, 71.6 with a CTA per item.  Shares fixed beforehand, the two CTAs of
// an SM in one: 74.9.)  Query row = tensor-memory lane = softmax thread: a row's maximum and
// sum need no exchange (two threads per row, which exchanged both through shared memory: 78.7 us at
// the layer shape, one: 68.1).  Per key tile of 64 tokens:
//   S = Q K^T        tcgen05.mma, Q tile and K tile K-major in shared memory (TMA, 128-byte
//                    swizzle), accumulator [128 x 64] fp32 in tensor memory, TWO buffers: the
//                    scores of tile i+1 are computed while the softmax of tile i runs
//   softmax          each thread reads its row of S (tcgen05.ld), keeps a reference exponent and a
//                    sum in the log2 domain, rescales its row of O in tensor memory when the
//                    reference moved (lazily: only when a tile's maximum exceeds it by more than
//                    2^8), and writes the probabilities back over S as packed bf16 (tcgen05.st)
//   O += P V         tcgen05.mma, A = P from tensor memory, B = the V tile (token-major, i.e.
//                    N-major) from shared memory
// What bounds it: run for seconds, the power limit (1000 W at 1.67 GHz, layer shape 69 us); in a burst, the softmax
// of a tile, 1200 cycles in a warp of which 800 are the exponentials, two warps a scheduler: two CTAs on an SM take
// 775 cycles per key tile, in which the tensor cores are busy for 640 (S 384: from shared memory at N = 64 the
// operand reads, not the arithmetic, set the rate; O 256) and the special-function units for 512.  (A quarter or an
// eighth of the exponentials on the FMA units by a polynomial of degree 5: 60.4 -> 61.4, 61.1 us.  Two heads a CTA
// that share the key tiles, tiles of 128 keys, scores of one head while the softmax of the other runs, single
// score buffers: 70 us with one thread a row, 95 with two.)
// Calls of at most two items an SM have an instantiation without the exchange with the scheduler (see ALONE): with it
// calls of one or two key tiles were 3 to 9 % slower than without (2 x 16 heads x 129 tokens 6.7 us, 6.1; 1 x 4 x 1 5.0, 4.7).
// One warp issues every contraction and one every load, under elect_one(): with a test of the lane
// number instead an instruction cost its thread about a hundred cycles (layer shape 84.1 us, now 79.6).  (One thread
// that walks the tiles, in place of a warp of which one thread issues: 61.7 us, 60.2.)
// The first loads leave before the block has met, and O leaves through shared memory by tensor copies of 32 rows x
// 64 columns.  Tensor memory: 256 columns (S twice 64, O 128); shared memory 112 KiB (Q 32, two K tiles, two V
// tiles, 16 for O; a tile is requested two tiles ahead, as soon as the contraction that read its slot is complete):
// two CTAs per SM.  Only key tiles that touch the 128 queries' windows are visited.  Every wait is bounded; a wait
// that runs out ends the kernel cleanly (copies, requests and contractions in flight are waited for, tensor memory
// is freed) and raises RODIMUS_ERR_TIMEOUT in the status word.  No hardware barrier is used inside the
// loop (a role that gave up would leave the others at it).
#include "ddts_tc_ptx.cuh"

namespace ddts {
namespace {

constexpr int kD = 128, kBM = 128, kBN = 64;
constexpr int kSoftmaxWarps = 4, kIssuerWarp = 4, kProducerWarp = 5, kThreads = 32 * (kSoftmaxWarps + 2);
constexpr uint32_t kQSlabBytes = kBM * 128;           // [128 rows][64 columns] bf16
constexpr uint32_t kSlabBytes = kBN * 128;            // [64 rows][64 columns] bf16
constexpr uint32_t kTileBytes = 2 * kSlabBytes;       // 64 x 128 bf16
constexpr uint32_t kOutBytes = 32 * 128;              // a warp's 32 rows x 64 columns on their way out
constexpr uint32_t kOffQ = 0, kOffK = 2 * kQSlabBytes, kOffV = kOffK + 2 * kTileBytes, kOffOut = kOffV + 2 * kTileBytes;
constexpr uint32_t kOffCtl = kOffOut + kSoftmaxWarps * kOutBytes;
constexpr uint32_t kSmemBytes = kOffCtl + 256;
static_assert(2 * (kSmemBytes + 1024) <= 233472, "two CTAs per SM");
constexpr uint32_t kTmemCols = 256, kColS = 0, kColO = 128;
constexpr float kLog2e = 1.4426950408889634f;

enum { BAR_Q = 0, BAR_K0, BAR_K1, BAR_V0, BAR_V1, BAR_S0, BAR_S1, BAR_P0, BAR_P1, BAR_O0, BAR_O1,
       BAR_NEXT0, BAR_NEXT1,           // the next item is known                          (1 + bytes)
       BAR_TAKEN0, BAR_TAKEN1,         // every role has read it                          (6)
       BAR_DRAIN, kNumBars };

struct SwCtl {
  uint4 next[2];       // answers of the hardware's scheduler
  uint64_t bar[kNumBars];
  uint32_t tmem_base;
  int abort;
  long long limit;
  int n_q, n_k, n_v, n_next;   // loads, items asked for (for the clean exit)
};
static_assert(sizeof(SwCtl) <= 256, "control block");

// Two fp32 operations in one instruction (packed pairs in 64-bit registers) and the three-input
// maximum: the softmax loop is bound by instruction issue and by the special-function unit, and
// these halve the count of everything around the exponentials.
__device__ __forceinline__ uint64_t pair_f32(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpair_f32(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

struct SwTcArgs {
  __nv_bfloat16* o;
  int32_t* status;   // may be nullptr
  int B, H, T, window, n_qtiles;
  float scale;
  long long limit;
};

__device__ __noinline__ bool sw_wait_slow(uint32_t bar, uint32_t parity, volatile SwCtl* c, int32_t* status) {
  const long long limit = c->limit, t0 = clock64();
  while (true) {
    if (limit > 0) {
#pragma unroll 1
      for (int i = 0; i < 16; ++i)
        if (mbar_try_park(bar, parity)) return true;
    }
    if (c->abort) return mbar_try(bar, parity);
    if (clock64() - t0 >= limit) {
      if (mbar_try(bar, parity)) return true;
      c->abort = 1;
      if (status) atomicMax(status, (int)RODIMUS_ERR_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ bool sw_wait(uint32_t bar, uint32_t parity, volatile SwCtl* c, int32_t* status) {
  if (mbar_try(bar, parity)) return true;
  return sw_wait_slow(bar, parity, c, status);
}

// An item: (batch, head, 128 queries), numbered from the longest on.  Query tiles late in a sequence see the most
// keys, so the index runs over the query tiles from the last one down and, within one tile position, over all
// (batch, head).
struct SwItem {
  int m0, lo, n;   // queries m0..m0+127 see keys of n tiles from tile lo on
  int b, bh;
};
__device__ __forceinline__ SwItem sw_item(const SwTcArgs& a, int at) {
  SwItem it;
  const int n_bh = a.B * a.H;
  it.bh = at % n_bh;
  it.b = it.bh / a.H;
  it.m0 = (a.n_qtiles - 1 - at / n_bh) * kBM;
  it.lo = max(0, it.m0 - a.window + 1) / kBN;
  it.n = min(it.m0 + kBM - 1, a.T - 1) / kBN - it.lo + 1;
  return it;
}
// The grid has a CTA per item.  A running CTA takes the place of one that has not been launched yet: it asks the
// hardware's scheduler to cancel the next launch and gets its index.  The answer, 16 bytes, lands in shared memory.
__device__ __forceinline__ void ask_for_launch(uint32_t dst, uint32_t bar) {
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
               ::"r"(dst), "r"(bar) : "memory");
}
__device__ __forceinline__ int launch_taken(uint32_t src) {   // index of the launch, -1: there is none left
  uint32_t ok, x;
  asm volatile(
      "{\n.reg .pred p;\n.reg .b128 h;\n"
      "ld.shared.b128 h, [%2];\n"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n"
      "selp.b32 %0, 1, 0, p;\n"
      "mov.b32 %1, 0;\n"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, h;\n}"
      : "=r"(ok), "=r"(x) : "r"(src) : "memory");
  return ok ? (int)x : -1;
}

// ALONE: every launch finds room at once, so no CTA will find one to take over: it ends without asking.
template <bool ALONE>
__global__ void __launch_bounds__(kThreads, 2)
swska_fwd_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o,
                    const SwTcArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];   // (the swizzled tiles need the alignment)
  const uint32_t base = smem_u32(smem_raw);
  volatile SwCtl* ctl = reinterpret_cast<volatile SwCtl*>(smem_raw + kOffCtl);
  auto bar = [&](int i) { return base + kOffCtl + (uint32_t)offsetof(SwCtl, bar) + 8u * (uint32_t)i; };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int T = a.T, W = a.window;

  // Loads of tile g, counted over all items of the CTA; a copy is 64 (queries: 128) rows of one head, rows past its
  // end are zeros.
  auto fill = [&](const CUtensorMap* map, uint32_t dst, int row, int head, int which, uint32_t bytes) {
    mbar_expect_tx(bar(which), bytes);
    tma_load_4d(base + dst, map, 0, row, 0, head, bar(which));
  };
  auto fill_q = [&](const SwItem& it) { fill(&map_q, kOffQ, it.m0, it.bh, BAR_Q, 2 * kQSlabBytes); };
  auto fill_k = [&](const SwItem& it, int j, int g) {
    fill(&map_k, kOffK + (g & 1) * kTileBytes, (it.lo + j) * kBN, it.b, BAR_K0 + (g & 1), kTileBytes);
  };
  auto fill_v = [&](const SwItem& it, int j, int g) {
    fill(&map_v, kOffV + (g & 1) * kTileBytes, (it.lo + j) * kBN, it.bh, BAR_V0 + (g & 1), kTileBytes);
  };
  SwItem it = sw_item(a, (int)blockIdx.x);
  // The thread that sets the barriers up asks for the first tiles at once: their way is as long as the
  // allocation of tensor memory and the block's first meeting together.
  if (warp == kProducerWarp && elect_one()) {
    ctl->abort = 0;
    ctl->limit = a.limit;
    for (int i = 0; i < kNumBars; ++i)
      mbar_init(bar(i), i == BAR_P0 || i == BAR_P1 ? kSoftmaxWarps : i == BAR_TAKEN0 || i == BAR_TAKEN1 ? kSoftmaxWarps + 2 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    fill_k(it, 0, 0);
    fill_q(it);
    fill_v(it, 0, 0);
    if (it.n > 1) { fill_k(it, 1, 1); fill_v(it, 1, 1); }
    ctl->n_q = 1;
    ctl->n_k = ctl->n_v = min(2, it.n);
    ctl->n_next = 0;
  }
  __syncwarp();
  if (warp == kIssuerWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(base + kOffCtl + (uint32_t)offsetof(SwCtl, tmem_base)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;

  // Item k of this CTA, for the thread (one) or the whole warp that asks; false when there is none, or on a timeout.
  auto next_item = [&](int k, bool one, SwItem& it) -> bool {
    if (k == 0) return true;
    if (ALONE) return false;
    const int slot = k & 1;
    const uint32_t ph = (uint32_t)((k - 1) >> 1) & 1;       // slot 1 is first used for k = 1, slot 0 for k = 2
    const bool got = sw_wait(bar(BAR_NEXT0 + slot), ph, ctl, a.status);
    if (!(one ? got : __all_sync(0xffffffffu, got) != 0)) return false;
    const int at = launch_taken(base + kOffCtl + (uint32_t)offsetof(SwCtl, next) + 16 * slot);
    fence_proxy_async();
    if (!one) __syncwarp();
    if (one || lane == 0) mbar_arrive(bar(BAR_TAKEN0 + slot));
    if (at < 0) return false;
    it = sw_item(a, at);
    return true;
  };

  if (warp == kProducerWarp) {
    // =========================== producer warp: every TMA load ================================
    if (elect_one()) {
      auto wait = [&](int b, int g) { return sw_wait(bar(b + (g & 1)), (g >> 1) & 1, ctl, a.status); };   // of tile g
      bool ok = true;
      int g = 0;
      // a slot is refilled as soon as the contraction that read it is complete: K two tiles ahead of the scores
      // that will read it, V two tiles ahead of its O += P V; the next item's queries after this one's last scores
      for (int k = 0; ok && next_item(k, true, it); ++k) {
        // The item after this one is asked for four tiles before the end: early enough to be known in time, late
        // enough for the CTAs that end first to get it.
        const int slot = (k + 1) & 1;
        auto ask = [&]() {
          if (!(ok = sw_wait(bar(BAR_TAKEN0 + slot), (uint32_t)((k >> 1) & 1) ^ 1, ctl, a.status))) return;
          mbar_expect_tx(bar(BAR_NEXT0 + slot), 16);
          ask_for_launch(base + kOffCtl + (uint32_t)offsetof(SwCtl, next) + 16 * slot, bar(BAR_NEXT0 + slot));
          ctl->n_next = k + 1;
        };
        int j = 0;
        if (k == 0) j = g = min(2, it.n);
        if (!ALONE && it.n - 4 < j) ask();
        for (; ok && j < it.n; ++j, ++g) {
          if (!ALONE && j == it.n - 4) ask();
          if (!ok) break;
          if (g >= 2 && !(ok = wait(BAR_S0, g - 2))) break;
          fill_k(it, j, g);
          ctl->n_k = g + 1;
          if (j == 0) {
            if (!(ok = wait(BAR_S0, g - 1))) break;
            fill_q(it);
            ctl->n_q = k + 1;
          }
          if (g >= 2 && !(ok = wait(BAR_O0, g - 2))) break;
          fill_v(it, j, g);
          ctl->n_v = g + 1;
        }
      }
    }
    __syncwarp();
  } else if (warp == kIssuerWarp) {
    // =========================== issuing warp: every contraction ==============================
    // Every lane walks the tiles; what is issued sits in elect_one() blocks.
    {
      constexpr uint32_t kIdescS = make_idesc(kBM, kBN, 0, 0);   // S = Q K^T, both K-major
      constexpr uint32_t kIdescO = make_idesc(kBM, kD, 0, 1);    // O += P V: A in tensor memory, B N-major
      auto wait = [&](int b, int g) {      // of tile g
        return __all_sync(0xffffffffu, sw_wait(bar(b + (g & 1)), (g >> 1) & 1, ctl, a.status)) != 0;
      };
      const uint32_t dq0 = desc_lo_kmajor(base + kOffQ), dq1 = desc_lo_kmajor(base + kOffQ + kQSlabBytes);
      auto scores = [&](int g) -> bool {   // of tile g into buffer g & 1
        if (!wait(BAR_K0, g)) return false;
        tc_fence_after();
        const uint32_t ks = base + kOffK + (g & 1) * kTileBytes;
        const uint32_t dk0 = desc_lo_kmajor(ks), dk1 = desc_lo_kmajor(ks + kSlabBytes);
        const uint32_t d = tmem + kColS + (g & 1) * kBN;
        if (elect_one()) {
          umma_bf16_lo<false>(d, dq0, dk0, kIdescS);
#pragma unroll
          for (int kk = 1; kk < 4; ++kk) umma_bf16_lo<true>(d, dq0 + 2 * kk, dk0 + 2 * kk, kIdescS);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) umma_bf16_lo<true>(d, dq1 + 2 * kk, dk1 + 2 * kk, kIdescS);
          umma_commit(bar(BAR_S0 + (g & 1)));
        }
        __syncwarp();
        return true;
      };
      bool ok = true;
      int g = 0;
      for (int k = 0; ok && next_item(k, false, it); ++k) {
        if (!(ok = __all_sync(0xffffffffu, sw_wait(bar(BAR_Q), k & 1, ctl, a.status)) && scores(g))) break;
        for (int j = 0; j < it.n; ++j, ++g) {
          if (j + 1 < it.n && !(ok = scores(g + 1))) break;        // while this tile's softmax runs
          if (!(ok = wait(BAR_V0, g) && wait(BAR_P0, g))) break;   // probabilities in place
          tc_fence_after();
          const uint32_t dv = desc_lo_mnmajor(base + kOffV + (g & 1) * kTileBytes, kSlabBytes);
          const uint32_t pa = tmem + kColS + (g & 1) * kBN;
          if (elect_one()) {
            if (j == 0) umma_bf16_atmem<false>(tmem + kColO, pa, dv, kIdescO);
            else umma_bf16_atmem<true>(tmem + kColO, pa, dv, kIdescO);
#pragma unroll
            for (int kk = 1; kk < 4; ++kk) umma_bf16_atmem<true>(tmem + kColO, pa + 8 * kk, dv + 128 * kk, kIdescO);
            umma_commit(bar(BAR_O0 + (g & 1)));   // (two barriers, by tile parity: a waiter is never two phases behind)
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
  } else {
    // =========================== softmax warps =================================================
    // thread = query row = tensor-memory lane
    const uint32_t t_row = tmem + ((uint32_t)(warp * 32) << 16);
    const float sc = a.scale * kLog2e;        // > 0 (checked by the host)
    bool ok = true;
    int g = 0;
    auto wait = [&](int b, int g) -> bool {   // of tile g; whole warps: tensor-memory accesses need them
      return __all_sync(0xffffffffu, sw_wait(bar(b + (g & 1)), (g >> 1) & 1, ctl, a.status)) != 0;
    };
    auto publish = [&](int sb) {
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(BAR_P0 + sb));
    };
    for (int k = 0; ok && next_item(k, false, it); ++k) {
      const int row = it.m0 + tid;
      // Reference exponent of the row (log2 domain).  It follows the running maximum lazily: it
      // moves only when a tile's maximum exceeds it by more than 8, so probabilities stay below 2^8
      // and O, l are rescaled rarely; the final division by l makes the result independent of it.
      float m_ref = -INFINITY, l_run = 0.f;
      for (int j = 0; j < it.n; ++j, ++g) {
        const int sb = g & 1;
        const int n0 = (it.lo + j) * kBN;
        const uint32_t t_s = t_row + kColS + sb * kBN;
        if (!(ok = wait(BAR_S0, g))) break;
        tc_fence_after();
        // the visible keys of the row are e_lo .. e_hi (none when e_lo > e_hi)
        const int e_lo = max(0, row - W + 1 - n0), e_hi = min(kBN - 1, row - n0);
        if (__all_sync(0xffffffffu, e_lo > e_hi)) {
          // on the diagonal and at the window's far edge whole warps see no key of a tile: they
          // write zeros, without the arithmetic
          uint32_t z[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) z[e] = 0u;
          tmem_st32(t_s, z);
          publish(sb);
          continue;
        }
        // ---- the row of S: mask, maximum (four independent chains of three-input steps)
        float sv[kBN];
        {
          uint32_t r0[32], r1[32];
          tmem_ld32(t_s, r0);
          tmem_ld32(t_s + 32, r1);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            sv[e] = __uint_as_float(r0[e]);
            sv[32 + e] = __uint_as_float(r1[e]);
          }
        }
        if (!__all_sync(0xffffffffu, e_lo == 0 && e_hi == kBN - 1)) {
          const unsigned long long bits = e_lo > e_hi ? 0ull : ((~0ull >> (kBN - 1 - e_hi)) & (~0ull << e_lo));
          const uint32_t b0 = (uint32_t)bits, b1 = (uint32_t)(bits >> 32);
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            sv[e] = ((b0 >> e) & 1u) ? sv[e] : -INFINITY;
            sv[32 + e] = ((b1 >> e) & 1u) ? sv[32 + e] : -INFINITY;
          }
        }
        float m4[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float* s16 = sv + 16 * c;
          float m = max3(s16[0], s16[1], s16[2]);
#pragma unroll
          for (int e = 3; e < 15; e += 2) m = max3(m, s16[e], s16[e + 1]);
          m4[c] = fmaxf(m, s16[15]);
        }
        const float m_tile = fmaxf(max3(m4[0], m4[1], m4[2]), m4[3]) * sc;   // (-inf stays -inf: sc > 0)
        if (__any_sync(0xffffffffu, m_tile > m_ref + 8.f)) {     // rare but for the first tile
          float alpha = 1.f;
          if (m_tile > m_ref + 8.f) {
            alpha = ex2f(m_ref - m_tile);           // 0 when nothing had been seen
            m_ref = m_tile;
          }
          l_run *= alpha;
          if (j > 0) {                              // O += P V of the tile before is complete
            if (!(ok = wait(BAR_O0, g - 1))) break;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              uint32_t r[32];
              tmem_ld32(t_row + kColO + 32 * c, r);
              tmem_ld_wait();
#pragma unroll
              for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
              tmem_st32(t_row + kColO + 32 * c, r);
            }
          }
        }
        const float m_use = m_ref == -INFINITY ? 0.f : m_ref;
        uint64_t ps[4] = {0ull, 0ull, 0ull, 0ull};     // four pairs of partial sums: short dependent chains
        const uint64_t sc2 = pair_f32(sc, sc), nm2 = pair_f32(-m_use, -m_use);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            float x0, x1;
            unpair_f32(fma2(pair_f32(sv[32 * hf + e], sv[32 * hf + e + 1]), sc2, nm2), x0, x1);
            const float p0 = ex2f(x0), p1 = ex2f(x1);
            ps[(e >> 1) & 3] = add2(ps[(e >> 1) & 3], pair_f32(p0, p1));
            pk[e >> 1] = pack_bf16(p0, p1);
          }
          tmem_st16(t_s + 16 * hf, pk);                // over S, two keys per column
        }
        publish(sb);
        float s0, s1;
        unpair_f32(add2(add2(ps[0], ps[1]), add2(ps[2], ps[3])), s0, s1);
        l_run += s0 + s1;
      }
      if (!ok || !(ok = wait(BAR_O0, g - 1))) break;
      // ---- divide the row by its sum and store it: 32 rows x 64 columns at a time through the warp's own piece of
      // shared memory, which a tensor copy takes away (rows past the sequence's end are not written).  Without a next
      // item the queries' tile is free by now: both halves go through its slabs, and neither waits for the other; or,
      // of at most 64 rows, the threads store them at once (16 heads x 129 tokens 6.2 us, 6.0; of 104 rows 17.1, 17.5).
      tc_fence_after();
      const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        uint32_t r0[32], r1[32];
        tmem_ld32(t_row + kColO + 64 * hf, r0);
        tmem_ld32(t_row + kColO + 64 * hf + 32, r1);
        tmem_ld_wait();
        if (ALONE && T - it.m0 <= 64) {
          if (row < T) {
            uint4* to = reinterpret_cast<uint4*>(a.o + ((long long)it.bh * T + row) * kD + 64 * hf);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const uint32_t* r = c < 4 ? r0 + 8 * c : r1 + 8 * (c - 4);
              uint32_t w[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) w[u] = pack_bf16(__uint_as_float(r[2 * u]) * inv, __uint_as_float(r[2 * u + 1]) * inv);
              to[c] = make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
          continue;
        }
        const uint32_t out = base + (ALONE ? kOffQ + hf * kQSlabBytes : kOffOut) + warp * kOutBytes;
        if (!ALONE) {
          if (elect_one()) bulk_wait_read<0>();     // the copy before has read it
          __syncwarp();
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {               // 16-byte pieces of the row
          const uint32_t* r = c < 4 ? r0 + 8 * c : r1 + 8 * (c - 4);
          uint32_t w[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) w[u] = pack_bf16(__uint_as_float(r[2 * u]) * inv, __uint_as_float(r[2 * u + 1]) * inv);
          sts128(out + lane * 128 + ((uint32_t)(c ^ (lane & 7)) << 4), w[0], w[1], w[2], w[3]);
        }
        fence_proxy_async();
        __syncwarp();
        if (it.m0 + 32 * warp < T && elect_one()) {
          tma_store_4d(&map_o, 0, it.m0 + 32 * warp, hf, it.bh, out);
          bulk_commit();
        }
        __syncwarp();
      }
      tc_fence_before();       // (before this warp's next probabilities, which let the next item's O begin)
    }
    if (elect_one()) bulk_wait_read<0>();
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (ctl->abort) {   // clean exit: nothing may still be writing this CTA's shared or tensor memory
    if (tid == 0) {
      mbar_drain(bar(BAR_Q), (ctl->n_q - 1) & 1);
      if (ctl->n_next > 0) mbar_drain(bar(BAR_NEXT0 + (ctl->n_next & 1)), ((ctl->n_next - 1) >> 1) & 1);
      for (int f = max(0, ctl->n_k - 2); f < ctl->n_k; ++f) mbar_drain(bar(BAR_K0 + (f & 1)), (f >> 1) & 1);
      for (int f = max(0, ctl->n_v - 2); f < ctl->n_v; ++f) mbar_drain(bar(BAR_V0 + (f & 1)), (f >> 1) & 1);
    }
    if (warp == kIssuerWarp && elect_one()) {   // (a commit follows the contractions of the thread that makes it)
      umma_commit(bar(BAR_DRAIN));            // completes when every contraction issued so far has
      mbar_drain(bar(BAR_DRAIN), 0);
    }
  }
  __syncthreads();
  if (warp == kIssuerWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

struct SwMapCache {     // the four maps of the last call on this host thread
  const void *q = nullptr, *k = nullptr, *v = nullptr, *o = nullptr;
  int B = 0, H = 0, T = 0;
  CUtensorMap mq, mk, mv, mo;
};
thread_local SwMapCache t_sw_maps;
std::atomic<unsigned long long> g_sw_tc_smem_done[2];

}  // namespace

cudaError_t launch_swska_tc(const rodimus_swska_fwd_params& p, int* n_launches) {
  *n_launches = 0;
  const uint64_t bh = (uint64_t)p.B * p.H, T = (uint64_t)p.T;
  SwMapCache& c = t_sw_maps;
  if (c.q != p.q || c.k != p.k || c.v != p.v || c.o != p.o || c.B != p.B || c.H != p.H || c.T != p.T) {
    c.q = nullptr;
    if (!encode_bf16_heads_map(&c.mq, p.q, bh, T, kD, kBM, 2) || !encode_bf16_heads_map(&c.mk, p.k, (uint64_t)p.B, T, kD, kBN, 2) ||
        !encode_bf16_heads_map(&c.mv, p.v, bh, T, kD, kBN, 2) || !encode_bf16_heads_map(&c.mo, p.o, bh, T, kD, 32, 1))
      return cudaErrorInvalidValue;
    c.q = p.q; c.k = p.k; c.v = p.v; c.o = p.o; c.B = p.B; c.H = p.H; c.T = p.T;
  }
  int dev = 0, sms = 0;
  cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(p.stream);
  SwTcArgs a;
  a.o = reinterpret_cast<__nv_bfloat16*>(p.o);
  a.status = reinterpret_cast<int32_t*>(p.workspace);
  a.B = p.B; a.H = p.H; a.T = p.T; a.window = p.window; a.scale = p.scale;
  a.n_qtiles = (p.T + kBM - 1) / kBM;
  const long long n_items = (long long)a.n_qtiles * p.B * p.H;
  if (n_items > 0x7fffffffLL) return cudaErrorInvalidValue;
  const bool alone = n_items <= 2LL * sms;   // (two CTAs on an SM)
  auto* const kernel = alone ? swska_fwd_tc_kernel<true> : swska_fwd_tc_kernel<false>;
  e = opt_in_shared_memory(kernel, (int)kSmemBytes, dev, g_sw_tc_smem_done[alone]);
  if (e != cudaSuccess) return e;
  a.limit = main_loop_wait_cycles();
  if (a.status) {
    e = cudaMemsetAsync(a.status, 0, sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
  }
  kernel<<<(unsigned)n_items, kThreads, kSmemBytes, st>>>(c.mq, c.mk, c.mv, c.mo, a);
  *n_launches = 1;
  return cudaGetLastError();
}

}  // namespace ddts
