// Sliding-window shared-key attention on tcgen05 (bf16 tokens, head size 128):
//   s_ti = scale <q^h_t, k_i>,  t - W < i <= t      p_ti = softmax_i(s_ti)      o^h_t = sum_i p_ti v^h_i
// (Sec. "Shared-Key Attention for Lossless Head Compression": one key per token for all heads.)
//
// One CTA per (batch, head, 128 queries): 4 softmax warps, one warp that issues the contractions and
// one that issues the TMA loads.  Query row = tensor-memory lane = softmax thread: a row's maximum and
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
// What bounds it: two CTAs on an SM take 825 cycles per key tile, in which the tensor cores are busy
// for 640 (S 384: from shared memory at N = 64 the operand reads, not the arithmetic, set the rate;
// O 256) and the special-function units for 512.
// One warp issues every contraction and one every load, under elect_one(): with a test of the lane
// number instead an instruction cost its thread about a hundred cycles (layer shape 84.1 us, now 79.6).
// The first loads leave before the block has met, and a whole tile of O leaves through shared memory
// by tensor copies instead of 16-byte pieces 256 bytes apart: 3.3 us less at the layer shape
// (4 x 16 x 2048, window 1024: 64.5 us), 4 us of 41 with a window of 128.
// Tensor memory: 256 columns
// (S twice 64, O 128); shared memory 96 KiB (Q 32, two K tiles, two V tiles; a tile is requested
// two tiles ahead, as soon as the contraction that read its slot is complete): two CTAs per SM.  Only key tiles that
// touch the 128 queries' windows are visited.  Every wait is bounded; a wait that runs out ends
// the kernel cleanly (copies and contractions in flight are waited for, tensor memory is freed)
// and raises RODIMUS_ERR_TIMEOUT in the status word.  No hardware barrier is used inside the
// loop (a role that gave up would leave the others at it).
#include "ddts_tc_ptx.cuh"

namespace ddts {
namespace {

constexpr int kD = 128, kBM = 128, kBN = 64;
constexpr int kSoftmaxWarps = 4, kIssuerWarp = 4, kProducerWarp = 5, kThreads = 32 * (kSoftmaxWarps + 2);
constexpr uint32_t kQSlabBytes = kBM * 128;           // [128 rows][64 columns] bf16
constexpr uint32_t kSlabBytes = kBN * 128;            // [64 rows][64 columns] bf16
constexpr uint32_t kTileBytes = 2 * kSlabBytes;       // 64 x 128 bf16
constexpr uint32_t kOffQ = 0, kOffK = 2 * kQSlabBytes, kOffV = kOffK + 2 * kTileBytes;
constexpr uint32_t kOffCtl = kOffV + 2 * kTileBytes;
constexpr uint32_t kSmemBytes = kOffCtl + 256 + 1024;  // + slack for 1024-byte alignment
constexpr uint32_t kTmemCols = 256, kColS = 0, kColO = 128;
constexpr float kLog2e = 1.4426950408889634f;

enum { BAR_Q = 0, BAR_K0, BAR_K1, BAR_V0, BAR_V1, BAR_S0, BAR_S1, BAR_P0, BAR_P1, BAR_O0, BAR_O1,
       BAR_OUT, BAR_DRAIN, kNumBars };

struct SwCtl {
  uint64_t bar[kNumBars];
  uint32_t tmem_base;
  int abort;
  long long limit;
  int k_sent, v_sent, k_seen, v_seen;   // loads asked for / seen complete (for the clean exit)
};

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
  void* o;
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

__global__ void __launch_bounds__(kThreads, 2)
swska_fwd_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o,
                    const SwTcArgs a) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* gen = smem_raw + (base - smem_u32(smem_raw));
  volatile SwCtl* ctl = reinterpret_cast<volatile SwCtl*>(gen + kOffCtl);
  auto bar = [&](int i) { return base + kOffCtl + 8u * (uint32_t)i; };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // Query tiles late in the sequence see the most keys.  CTAs are handed out in the order of
  // their index, so the index runs over the query tiles from the last one down and, within one
  // tile position, over all (batch, head): every long tile of the call starts before any short
  // one, and the short ones fill the tail.
  const int T = a.T, W = a.window;
  const int n_bh = a.B * a.H;
  const int m0 = (a.n_qtiles - 1 - (int)(blockIdx.x / (unsigned)n_bh)) * kBM;
  const long long bh = blockIdx.x % (unsigned)n_bh;
  const int b = (int)(bh / a.H);
  const long long qrow0 = bh * T + m0;           // row of the [B*H*T, 128] views of q, o
  const int krow0 = b * T;                       // row of the [B*T, 128] view of k
  const int vrow0 = (int)(bh * T);               // row of the [B*H*T, 128] view of v
  const int first_key = max(0, m0 - W + 1);
  const int nt_lo = first_key / kBN, nt_hi = min(m0 + kBM - 1, T - 1) / kBN;
  const int n_tiles = nt_hi - nt_lo + 1;

  auto load = [&](const CUtensorMap* map, uint32_t dst, uint32_t slab, int row, int which, uint32_t bytes) {
    mbar_expect_tx(bar(which), bytes);
    tma_load_2d(base + dst, map, 0, row, bar(which));
    tma_load_2d(base + dst + slab, map, 64, row, bar(which));
  };
  auto fill_k = [&](int j) {
    load(&map_k, kOffK + (j & 1) * kTileBytes, kSlabBytes, krow0 + (nt_lo + j) * kBN, BAR_K0 + (j & 1), kTileBytes);
  };
  auto fill_v = [&](int j) {
    load(&map_v, kOffV + (j & 1) * kTileBytes, kSlabBytes, vrow0 + (nt_lo + j) * kBN, BAR_V0 + (j & 1), kTileBytes);
  };
  // The thread that sets the barriers up asks for the first tiles at once: their way is as long as the
  // allocation of tensor memory and the block's first meeting together.
  if (warp == kProducerWarp && elect_one()) {
    ctl->abort = 0;
    ctl->limit = a.limit;
    ctl->k_seen = ctl->v_seen = 0;
    for (int i = 0; i < kNumBars; ++i) {
      mbar_init(bar(i), i == BAR_P0 || i == BAR_P1 || i == BAR_OUT ? kSoftmaxWarps : 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    fill_k(0);
    load(&map_q, kOffQ, kQSlabBytes, (int)qrow0, BAR_Q, 2 * kQSlabBytes);
    fill_v(0);
    if (n_tiles > 1) { fill_k(1); fill_v(1); }
    ctl->k_sent = ctl->v_sent = min(2, n_tiles);
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

  if (warp == kProducerWarp) {
    // =========================== producer warp: every TMA load ================================
    if (elect_one()) {
      int k_sent = min(2, n_tiles), v_sent = k_sent;
      bool ok = true;
      // a slot is refilled as soon as the contraction that read it is complete: K two tiles ahead
      // of the scores that will read it, V two tiles ahead of its O += P V
      for (int it = 0; ok && it + 2 < n_tiles; ++it) {
        if (!(ok = sw_wait(bar(BAR_S0 + (it & 1)), (it >> 1) & 1, ctl, a.status))) break;
        fill_k(it + 2);
        ++k_sent;
        if (!(ok = sw_wait(bar(BAR_O0 + (it & 1)), (it >> 1) & 1, ctl, a.status))) break;
        fill_v(it + 2);
        ++v_sent;
      }
      ctl->k_sent = k_sent;
      ctl->v_sent = v_sent;
    }
    __syncwarp();
  } else if (warp == kIssuerWarp) {
    // =========================== issuing warp: every contraction ==============================
    // Every lane walks the tiles; what is issued sits in elect_one() blocks.
    {
      constexpr uint32_t kIdescS = make_idesc(kBM, kBN, 0, 0);   // S = Q K^T, both K-major
      constexpr uint32_t kIdescO = make_idesc(kBM, kD, 0, 1);    // O += P V: A in tensor memory, B N-major
      int k_seen = 0, v_seen = 0;
      auto wait = [&](int b, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, sw_wait(bar(b), parity, ctl, a.status)) != 0;
      };
      const uint32_t dq0 = desc_lo_kmajor(base + kOffQ), dq1 = desc_lo_kmajor(base + kOffQ + kQSlabBytes);
      auto issue_s = [&](int j) {   // scores of tile j into buffer j & 1
        const uint32_t ks = base + kOffK + (j & 1) * kTileBytes;
        const uint32_t dk0 = desc_lo_kmajor(ks), dk1 = desc_lo_kmajor(ks + kSlabBytes);
        const uint32_t d = tmem + kColS + (j & 1) * kBN;
        if (elect_one()) {
          umma_bf16_lo<false>(d, dq0, dk0, kIdescS);
#pragma unroll
          for (int kk = 1; kk < 4; ++kk) umma_bf16_lo<true>(d, dq0 + 2 * kk, dk0 + 2 * kk, kIdescS);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) umma_bf16_lo<true>(d, dq1 + 2 * kk, dk1 + 2 * kk, kIdescS);
          umma_commit(bar(BAR_S0 + (j & 1)));
        }
        __syncwarp();
      };
      bool ok = wait(BAR_Q, 0);
      if (ok) { ok = wait(BAR_K0, 0); k_seen += ok; }
      if (ok) { tc_fence_after(); issue_s(0); }
      for (int it = 0; ok && it < n_tiles; ++it) {
        const int sb = it & 1;
        const uint32_t ph = (it >> 1) & 1;
        if (it + 1 < n_tiles) {            // the next tile's scores, while this tile's softmax runs
          ok = wait(BAR_K0 + (sb ^ 1), ((it + 1) >> 1) & 1);
          k_seen += ok;
          if (!ok) break;
          tc_fence_after();
          issue_s(it + 1);
        }
        if (!(ok = wait(BAR_P0 + sb, ph))) break;   // probabilities in place
        ok = wait(BAR_V0 + sb, ph);
        v_seen += ok;
        if (!ok) break;
        tc_fence_after();
        const uint32_t dv = desc_lo_mnmajor(base + kOffV + sb * kTileBytes, kSlabBytes);
        const uint32_t pa = tmem + kColS + sb * kBN;
        if (elect_one()) {
          if (it == 0) umma_bf16_atmem<false>(tmem + kColO, pa, dv, kIdescO);
          else umma_bf16_atmem<true>(tmem + kColO, pa, dv, kIdescO);
#pragma unroll
          for (int kk = 1; kk < 4; ++kk) umma_bf16_atmem<true>(tmem + kColO, pa + 8 * kk, dv + 128 * kk, kIdescO);
          umma_commit(bar(BAR_O0 + sb));   // (two barriers, by tile parity: a waiter is never two phases behind)
        }
        __syncwarp();
      }
      if (lane == 0) {
        ctl->k_seen = k_seen;
        ctl->v_seen = v_seen;
      }
    }
    __syncwarp();
  } else {
    // =========================== softmax warps =================================================
    // thread = query row = tensor-memory lane
    const int row = m0 + tid;
    const uint32_t t_row = tmem + ((uint32_t)(warp * 32) << 16);
    const float sc = a.scale * kLog2e;        // > 0 (checked by the host)
    // Reference exponent of the row (log2 domain).  It follows the running maximum lazily: it
    // moves only when a tile's maximum exceeds it by more than 8, so probabilities stay below 2^8
    // and O, l are rescaled rarely; the final division by l makes the result independent of it.
    float m_ref = -INFINITY, l_run = 0.f;
    bool ok = true;
    auto wait = [&](int b, uint32_t parity) -> bool {   // whole warps: tensor-memory accesses need them
      return __all_sync(0xffffffffu, sw_wait(bar(b), parity, ctl, a.status)) != 0;
    };
    auto publish = [&](int sb) {
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(BAR_P0 + sb));
    };
    for (int it = 0; it < n_tiles; ++it) {
      const int sb = it & 1;
      const int n0 = (nt_lo + it) * kBN;
      const uint32_t t_s = t_row + kColS + sb * kBN;
      if (!(ok = wait(BAR_S0 + sb, (it >> 1) & 1))) break;
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
        if (it > 0) {                             // O += P V of the tile before is complete
          if (!(ok = wait(BAR_O0 + ((it - 1) & 1), ((it - 1) >> 1) & 1))) break;
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
    // ---- the last O += P V, then normalise and store the row
    if (ok) ok = wait(BAR_O0 + ((n_tiles - 1) & 1), ((n_tiles - 1) >> 1) & 1);
    if (ok) {
      tc_fence_after();
      const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
      // A whole tile goes through shared memory (where Q was: its last reader is done) and leaves by two
      // tensor copies; in the last tile of a sequence every thread stores its own row, 256 bytes apart
      // from its neighbour's, so that no row of the next head is touched.
      const bool whole = m0 + kBM <= T;
      const uint32_t orow_s = base + kOffQ + tid * 128;
      __nv_bfloat16* orow = (__nv_bfloat16*)a.o + (qrow0 + tid) * kD;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t r[32];
        tmem_ld32(t_row + kColO + 32 * c, r);
        tmem_ld_wait();
        if (row < T) {
#pragma unroll
          for (int e = 0; e < 32; e += 8) {
            const uint32_t c16 = (uint32_t)(4 * c + e / 8);        // 16-byte piece of the row
            uint4 w;
            w.x = pack_bf16(__uint_as_float(r[e]) * inv, __uint_as_float(r[e + 1]) * inv);
            w.y = pack_bf16(__uint_as_float(r[e + 2]) * inv, __uint_as_float(r[e + 3]) * inv);
            w.z = pack_bf16(__uint_as_float(r[e + 4]) * inv, __uint_as_float(r[e + 5]) * inv);
            w.w = pack_bf16(__uint_as_float(r[e + 6]) * inv, __uint_as_float(r[e + 7]) * inv);
            if (whole) sts128(orow_s + (c16 >> 3) * kQSlabBytes + (((c16 & 7) ^ (uint32_t)(tid & 7)) << 4), w.x, w.y, w.z, w.w);
            else *reinterpret_cast<uint4*>(orow + 32 * c + e) = w;
          }
        }
      }
      if (whole) {
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(BAR_OUT));
        if (warp == 0) {
          if (wait(BAR_OUT, 0) && elect_one()) {
            tma_store_2d(&map_o, 0, (int)qrow0, base + kOffQ);
            tma_store_2d(&map_o, 64, (int)qrow0, base + kOffQ + kQSlabBytes);
            bulk_commit();
            bulk_wait_read<0>();
          }
          __syncwarp();
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (ctl->abort) {   // clean exit: nothing may still be writing this CTA's shared or tensor memory
    if (tid == 0) {
      mbar_drain(bar(BAR_Q), 0);
      for (int j = ctl->k_seen; j < ctl->k_sent; ++j) mbar_drain(bar(BAR_K0 + (j & 1)), (j >> 1) & 1);
      for (int j = ctl->v_seen; j < ctl->v_sent; ++j) mbar_drain(bar(BAR_V0 + (j & 1)), (j >> 1) & 1);
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
  uint64_t rows_q = 0, rows_k = 0;
  CUtensorMap mq, mk, mv, mo;
};
thread_local SwMapCache t_sw_maps;
std::atomic<unsigned long long> g_sw_tc_smem_done{0};

}  // namespace

cudaError_t launch_swska_tc(const rodimus_swska_fwd_params& p, int* n_launches) {
  *n_launches = 0;
  const uint64_t rows_q = (uint64_t)p.B * p.H * p.T, rows_k = (uint64_t)p.B * p.T;
  SwMapCache& c = t_sw_maps;
  if (c.q != p.q || c.k != p.k || c.v != p.v || c.o != p.o || c.rows_q != rows_q || c.rows_k != rows_k) {
    if (!encode_bf16_map(&c.mq, p.q, rows_q, kD, kBM) || !encode_bf16_map(&c.mk, p.k, rows_k, kD, kBN) ||
        !encode_bf16_map(&c.mv, p.v, rows_q, kD, kBN) || !encode_bf16_map(&c.mo, p.o, rows_q, kD, kBM)) {
      c.q = nullptr;
      return cudaErrorInvalidValue;
    }
    c.q = p.q; c.k = p.k; c.v = p.v; c.o = p.o; c.rows_q = rows_q; c.rows_k = rows_k;
  }
  int dev = 0, sms = 0;
  cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  e = opt_in_shared_memory(swska_fwd_tc_kernel, (int)kSmemBytes, dev, g_sw_tc_smem_done);
  if (e != cudaSuccess) return e;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(p.stream);
  SwTcArgs a;
  a.o = p.o;
  a.status = reinterpret_cast<int32_t*>(p.workspace);
  a.B = p.B; a.H = p.H; a.T = p.T; a.window = p.window; a.scale = p.scale;
  a.n_qtiles = (p.T + kBM - 1) / kBM;
  const long long n_ctas = (long long)a.n_qtiles * p.B * p.H;
  if (n_ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
  a.limit = main_loop_wait_cycles();
  if (a.status) {
    e = cudaMemsetAsync(a.status, 0, sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((unsigned)n_ctas);
  swska_fwd_tc_kernel<<<grid, kThreads, kSmemBytes, st>>>(c.mq, c.mk, c.mv, c.mo, a);
  *n_launches = 1;
  return cudaGetLastError();
}

}  // namespace ddts
