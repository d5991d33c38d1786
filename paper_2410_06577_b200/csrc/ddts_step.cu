// One-token decode: S <- diag(alpha) S + (ahat . k)^T v in place, o = scale * q S
// (Eq. "rodimus_recurrent_form" applied once).  Pure HBM streaming: every fp32 state element
// is read once and written once with 16-byte accesses; nothing else is comparable in size.
//
// Work item = (sequence, head, tile of 4 LC state columns).  A CTA of W warps walks the dk rows of its
// tile, 32 / LC rows per warp-wide access; a lane owns four columns.  Rows are processed in batches of
// BATCH accesses per warp with all loads of a batch in flight at once; the first batch is issued before
// the gate math so that its latency hides the token loads and the transcendental work.
//   W = 4, LC = 32, BATCH = 16   128 columns, every access one 512-byte row segment: the shape for
//                                streaming many states (256 x 16 states 168 us, 0.98 of the copy rate)
//   W = 8, LC = 8,  BATCH = 8    32 columns, up to 256 rows in flight at once: calls too small to fill
//                                the device are latency, and this spreads them over 4 times the CTAs
//                                (device time of a step, 16 states: 4.4 us on wide tiles, 2.95 on narrow)
// Both sum q S over the rows in one order, so that a sequence's output does not depend on how many others are
// in the call: rows g, g + 4, g + 8, g + 12 of a block of 16 in turn; the blocks' results in turn; the four g
// in turn.  A thread of the wide tile meets its rows in that order, one of the narrow tile has a g of a block.
// (The wide tile's plain order in the narrow one took a trip of the state through shared memory, 0.2 us; the
// narrow one's former order in the wide one eight sums a thread, 5 to 20 % of calls of 50 to 1000 states.)
#include <type_traits>

#include "ddts_common.cuh"

namespace ddts {
namespace {

constexpr int kMaxDk = 256;

__device__ __forceinline__ float4 ld_stream(const float4* p) { return __ldcs(p); }
__device__ __forceinline__ void st_stream(float4* p, const float4& v) { __stcs(p, v); }

// VDECAY: the value-side decay beta_t of the general transition is given (the paper's ablation
// arm); a separate instantiation, so that the plain path carries none of it.
template <typename T, bool VDECAY, int W, int LC, int BATCH>
__global__ void __launch_bounds__(32 * W, W == 4 ? 4 : 2)
ddts_step_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ gx,
                 const T* __restrict__ ty, const T* __restrict__ v, T* __restrict__ o,
                 float* __restrict__ state, int n_seq_heads, int dk, int dv, float scale,
                 int ingate, const T* __restrict__ beta_hat, const float* __restrict__ feed_d,
                 const T* __restrict__ feed_x, int H, int shared, const T* __restrict__ vdecay) {
  constexpr int kThreads = 32 * W, kTileCols = 4 * LC, kSub = 32 / LC;
  static_assert(W * kSub == 4 || W * kSub == 32, "a wide or a narrow tile");
  constexpr bool kWide = W * kSub == 4;
  __shared__ float s_alpha[kMaxDk];
  __shared__ float s_w[kMaxDk];   // ahat * k
  __shared__ float s_q[kMaxDk];   // scale * q
  __shared__ float4 s_red[kWide ? 1 : kMaxDk / 16][4][LC];   // [block of rows][g]

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int cl = lane % LC;
  // row j of this thread's batch that begins at row `base`
  const int row0 = kWide ? warp : warp * 16 + lane / LC;
  auto row_of = [&](int base, int j) { return base + row0 + (kWide ? 4 * j : (j >> 2) * 128 + (j & 3) * 4); };
  const int tiles = (dv + kTileCols - 1) / kTileCols;
  const long long n_items = (long long)n_seq_heads * tiles;

  for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
    const long long nh = item / tiles;
    const int col = (int)(item % tiles) * kTileCols + cl * 4;
    const bool col_ok = col < dv;
    float* S = state + nh * (long long)dk * dv + col;

    // First batch of state rows: issued before anything else of this item.
    float4 buf[BATCH];
#pragma unroll
    for (int j = 0; j < BATCH; ++j) {
      const int r = row_of(0, j);
      if (col_ok && r < dk) buf[j] = ld_stream(reinterpret_cast<const float4*>(S + (long long)r * dv));
    }

    // Gates of this token (fp32 throughout).
    for (int d = tid; d < dk; d += kThreads) {
      const long long i = (shared ? nh / H : nh) * dk + d;   // shared: q,k,gx,ty are [Nseq,1,dk]
      float la, lh;
      gate_logs_f32(to_f32(gx[i]), to_f32(ty[i]), ingate, la, lh);
      s_alpha[d] = expf(la);
      s_w[d] = expf(lh) * to_f32(k[i]);
      s_q[d] = scale * to_f32(q[i]);
    }
    float4 vv = make_float4(0.f, 0.f, 0.f, 0.f);
    if (col_ok) {
      const T* vp = v + nh * dv + col;
      vv = make_float4(to_f32(vp[0]), to_f32(vp[1]), to_f32(vp[2]), to_f32(vp[3]));
      if (beta_hat) {   // value gate (Eq. "beta_def"): v enters the state as beta_hat * v
        const T* bp = beta_hat + nh * dv + col;
        vv.x *= to_f32(bp[0]); vv.y *= to_f32(bp[1]); vv.z *= to_f32(bp[2]); vv.w *= to_f32(bp[3]);
      }
    }
    float4 bd = make_float4(1.f, 1.f, 1.f, 1.f);
    if (VDECAY && col_ok) {
      const T* dp = vdecay + nh * dv + col;
      bd = make_float4(to_f32(dp[0]), to_f32(dp[1]), to_f32(dp[2]), to_f32(dp[3]));
    }
    __syncthreads();

    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), sum = acc;
    for (int base = 0; base < dk; base += W * kSub * BATCH) {
#pragma unroll
      for (int j = 0; j < BATCH; ++j) {
        const int r = row_of(base, j);
        if (col_ok && r < dk) {
          const float a = s_alpha[r], w = s_w[r], qq = s_q[r];
          float4 s = buf[j];
          if (VDECAY) {
            s.x = fmaf(a * bd.x, s.x, w * vv.x);
            s.y = fmaf(a * bd.y, s.y, w * vv.y);
            s.z = fmaf(a * bd.z, s.z, w * vv.z);
            s.w = fmaf(a * bd.w, s.w, w * vv.w);
          } else {
            s.x = fmaf(a, s.x, w * vv.x);
            s.y = fmaf(a, s.y, w * vv.y);
            s.z = fmaf(a, s.z, w * vv.z);
            s.w = fmaf(a, s.w, w * vv.w);
          }
          acc.x = fmaf(qq, s.x, acc.x);
          acc.y = fmaf(qq, s.y, acc.y);
          acc.z = fmaf(qq, s.z, acc.z);
          acc.w = fmaf(qq, s.w, acc.w);
          if ((j & 3) == 3) {                   // a block's result
            if (kWide) {
              sum.x += acc.x; sum.y += acc.y; sum.z += acc.z; sum.w += acc.w;
            } else {
              s_red[r >> 4][lane / LC][cl] = acc;
            }
            acc = make_float4(0.f, 0.f, 0.f, 0.f);
          }
          st_stream(reinterpret_cast<float4*>(S + (long long)r * dv), s);
        }
      }
      const int next = base + W * kSub * BATCH;
      if (next < dk) {
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
          const int r = row_of(next, j);
          if (col_ok && r < dk)
            buf[j] = ld_stream(reinterpret_cast<const float4*>(S + (long long)r * dv));
        }
      }
    }

    // o = the blocks' results, then the four g
    if (kWide) s_red[0][warp][lane] = sum;
    __syncthreads();
    if (warp == 0) {
      float4 t;
      if (kWide) {
        t = s_red[0][0][lane];
#pragma unroll
        for (int g = 1; g < 4; ++g) {
          const float4 u = s_red[0][g][lane];
          t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
        }
      } else {                                  // a g and four columns a lane
        t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int b = 0; b < dk / 16; ++b) {
          const float4 u = s_red[b][lane / LC][cl];
          t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
        }
        const float4 t0 = t;
#pragma unroll
        for (int g = 1; g < 4; ++g) {
          t.x += __shfl_down_sync(0xffffffffu, t0.x, g * LC);
          t.y += __shfl_down_sync(0xffffffffu, t0.y, g * LC);
          t.z += __shfl_down_sync(0xffffffffu, t0.z, g * LC);
          t.w += __shfl_down_sync(0xffffffffu, t0.w, g * LC);
        }
      }
      if (lane < LC && col_ok) {
        if (feed_d) {     // feed-through: o = scale q S + d . x'
          const float* dp = feed_d + (nh % H) * dv + col;
          const T* fp = feed_x + nh * dv + col;
          t.x = fmaf(dp[0], to_f32(fp[0]), t.x); t.y = fmaf(dp[1], to_f32(fp[1]), t.y);
          t.z = fmaf(dp[2], to_f32(fp[2]), t.z); t.w = fmaf(dp[3], to_f32(fp[3]), t.w);
        }
        T* op = o + nh * dv + col;
        op[0] = from_f32<T>(t.x);
        op[1] = from_f32<T>(t.y);
        op[2] = from_f32<T>(t.z);
        op[3] = from_f32<T>(t.w);
      }
    }
    __syncthreads();  // s_alpha / s_red are rewritten by the next item
  }
}

}  // namespace

cudaError_t launch_step(const rodimus_ddts_step_params& p, int* n_launches) {
  *n_launches = 0;
  const long long nh = (long long)p.Nseq * p.H;
  if (nh == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(p.stream);
  // One CTA per item: measured 6 % faster than a persistent grid of 8 CTAs per SM (the hardware
  // block scheduler balances the tail better than a fixed stride does).  The in-kernel loop only
  // matters beyond the grid-size limit.
  auto grid = [&](int cols) {
    const long long items = nh * ((p.dv + cols - 1) / cols);
    return (unsigned)(items < 0x7fffffffLL ? items : 0x7fffffffLL);
  };
  // The narrow tile while its CTAs are all resident at once, two per SM (16 states 5.3 us against 7.5,
  // 32 states 5.1 against 6.2; 64 states 8.2 against 6.2).
  const bool small = grid(32) <= 2u * (unsigned)sms;
  auto launch = [&](auto tag, auto decay) {
    using T = decltype(tag);
    constexpr bool VD = decltype(decay)::value;
    auto kernel = small ? ddts_step_kernel<T, VD, 8, 8, 8> : ddts_step_kernel<T, VD, 4, 32, 16>;
    kernel<<<grid(small ? 32 : 128), small ? 256 : 128, 0, st>>>(
        (const T*)p.q, (const T*)p.k, (const T*)p.gate_x, (const T*)p.temp_y, (const T*)p.v,
        (T*)p.o, p.state, (int)nh, p.dk, p.dv, p.scale, p.ingate, (const T*)p.beta_hat, p.feed_d,
        (const T*)p.feed_x, p.H, p.shared_gates, (const T*)p.value_decay);
  };
  if (p.dtype == RODIMUS_BF16) {
    if (p.value_decay) launch(__nv_bfloat16{}, std::true_type{});
    else launch(__nv_bfloat16{}, std::false_type{});
  } else {
    if (p.value_decay) launch(float{}, std::true_type{});
    else launch(float{}, std::false_type{});
  }
  *n_launches = 1;
  return cudaGetLastError();
}

}  // namespace ddts
