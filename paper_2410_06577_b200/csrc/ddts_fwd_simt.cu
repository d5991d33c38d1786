// Chunked prefill on the CUDA cores, all arithmetic in fp32 (the validation build, and the
// kernel for every shape the tensor-core kernel does not cover).
//
// Same algebra as the appendix "Chunkwise Parallel Representation of the Rodimus Block", with
// the state entering the chunk in the inter-chunk readout:
//   b_r   = sum_{j<=r in chunk} log alpha_j                      (per key channel)
//   P_ri  = sum_d q_rd k_id ahat_id exp(b_rd - b_id),  i <= r    (difference formed BEFORE exp)
//   O_r   = sum_{i<=r} P_ri v_i + (q_r . exp(b_r)) S_in
//   S_out = diag(exp(b_C)) S_in + sum_i (k_i . ahat_i . exp(b_C - b_i))^T v_i
// Every exponent is <= 0 apart from log ahat, so no input in the documented domain overflows,
// whatever the decay.
//
// Optional value-side decay beta_t (general transition of Sec. 3.1.1, the arm the paper ablates
// and drops): with c_r = sum_{j<=r in chunk} log beta_j per value column,
//   O_r   = sum_{i<=r} P_ri (v_i . exp(c_r - c_i)) + exp(c_r) . ((q_r . exp(b_r)) S_in)
//   S_out = (exp(b_C)^T exp(c_C)) . S_in + sum_i (k_i . ahat_i . exp(b_C - b_i))^T (v_i . exp(c_C - c_i))
//
// Two forms.  Where the states of all 16-row chunks stay in L2, the chunks are computed side by side:
// per chunk the operands, the scores and its own contribution to the state; an elementwise pass that
// turns contributions into the states entering the chunks, S <- D . S + dS; per chunk the outputs.
// Elsewhere (and where the caller's workspace has no room, and with the value-side decay) one CTA per
// (sequence, head, kTileV state columns) walks the sequence with its slice of the state in shared memory.
#include "ddts_common.cuh"

namespace ddts {
namespace {

constexpr int kC = 16;          // chunk length
constexpr int kTileV = 64;      // state columns per CTA
constexpr int kThreads = 256;
constexpr int kMaxDk = 256;

struct SimtArgs {
  const void *q, *k, *gx, *ty, *v;
  const void *beta_hat, *feed_x;   // optional: value gate [.., dv], feed-through input [.., dv]
  const void *vdecay;              // optional: value-side decay beta_t [.., dv], numbers in (0,1]
  const float* feed_d;             // optional: feed-through weight [H, dv]
  void* o;
  const float* s0;
  float* sT;
  const int32_t* cu;  // device cu_seqlens or nullptr
  WorkspaceHeader* hdr;
  int H, T, dk, dv, n_seq, tiles;
  float scale;
  int ingate;
  int shared;   // 1: q,k,gx,ty are [B,1,T,dk], one set per token for all heads
};

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) ddts_fwd_simt_kernel(const SimtArgs a) {
  extern __shared__ float smem[];
  const int dk = a.dk, dv = a.dv;
  const int ld = dk + 1;                       // padded row stride of the [kC, dk] arrays
  float* sS = smem;                            // [dk][kTileV]  state slice
  float* sQ = sS + dk * kTileV;                // [kC][ld]      q
  float* sW = sQ + kC * ld;                    // [kC][ld]      ahat * k
  float* sB = sW + kC * ld;                    // [kC][ld]      b (cumulative log decay)
  float* sV = sB + kC * ld;                    // [kC][kTileV]
  float* sP = sV + kC * kTileV;                // [kC][kC]
  float* sE = sP + kC * kC;                    // [dk]          b at the chunk end
  float* sC = sE + dk;                         // [kC][kTileV]  c (cumulative log beta), if given

  const int tid = threadIdx.x;
  const long long item = blockIdx.x;
  // dense calls have no planning kernel in front: the first CTA clears the device status
  if (!a.cu && item == 0 && tid == 0) a.hdr->status = RODIMUS_OK;
  const int tile = (int)(item % a.tiles);
  const long long sh = item / a.tiles;         // sequence * H + head
  const int h = (int)(sh % a.H);
  const long long n = sh / a.H;
  const int col0 = tile * kTileV;

  long long row0;
  int len;
  if (a.cu) {
    int lo = a.cu[n], hi = a.cu[n + 1];
    lo = lo < 0 ? 0 : (lo > a.T ? a.T : lo);
    hi = hi < lo ? lo : (hi > a.T ? a.T : hi);
    row0 = (long long)h * a.T + lo;
    len = hi - lo;
  } else {
    row0 = sh * a.T;
    len = a.T;
  }
  // rows of q,k,gx,ty: the head's own, or the sequence's single shared set
  const long long rq = a.shared ? row0 - ((long long)h + (a.cu ? 0 : n * (a.H - 1))) * a.T : row0;
  const T* q = (const T*)a.q + rq * dk;
  const T* k = (const T*)a.k + rq * dk;
  const T* gx = (const T*)a.gx + rq * dk;
  const T* ty = (const T*)a.ty + rq * dk;
  const T* v = (const T*)a.v + row0 * dv;
  T* o = (T*)a.o + row0 * dv;
  const T* bh = a.beta_hat ? (const T*)a.beta_hat + row0 * dv : nullptr;
  const T* fx = a.feed_d ? (const T*)a.feed_x + row0 * dv : nullptr;
  const float* fd = a.feed_d ? a.feed_d + (long long)h * dv : nullptr;
  const T* bd = a.vdecay ? (const T*)a.vdecay + row0 * dv : nullptr;
  const long long s_off = sh * (long long)dk * dv;

  for (int e = tid; e < dk * kTileV; e += kThreads) {
    const int d = e / kTileV, c = e % kTileV;
    sS[e] = (a.s0 && col0 + c < dv) ? a.s0[s_off + (long long)d * dv + col0 + c] : 0.f;
  }
  __syncthreads();

  for (int t0 = 0; t0 < len; t0 += kC) {
    const int nr = min(kC, len - t0);
    // (1) gates and in-chunk cumulative log decay: one thread per key channel
    for (int d = tid; d < dk; d += kThreads) {
      float b = 0.f;
      for (int r = 0; r < nr; ++r) {
        const long long i = (long long)(t0 + r) * dk + d;
        float la, lh;
        gate_logs_f32(to_f32(gx[i]), to_f32(ty[i]), a.ingate, la, lh);
        b += la;
        sB[r * ld + d] = b;
        sW[r * ld + d] = expf(lh) * to_f32(k[i]);
        sQ[r * ld + d] = to_f32(q[i]);
      }
      sE[d] = b;
    }
    for (int e = tid; e < kC * kTileV; e += kThreads) {
      const int r = e / kTileV, c = e % kTileV;
      float vv = 0.f;
      if (r < nr && col0 + c < dv) {
        const long long i = (long long)(t0 + r) * dv + col0 + c;
        vv = to_f32(v[i]);
        if (bh) vv *= to_f32(bh[i]);   // value gate (Eq. "beta_def")
      }
      sV[e] = vv;
    }
    if (bd) {   // cumulative log of the value-side decay: one thread per state column
      for (int c = tid; c < kTileV; c += kThreads) {
        float cum = 0.f;
        for (int r = 0; r < kC; ++r) {
          if (r < nr && col0 + c < dv)
            cum += logf(fmaxf(to_f32(bd[(long long)(t0 + r) * dv + col0 + c]), 1e-37f));
          sC[r * kTileV + c] = cum;
        }
      }
    }
    __syncthreads();
    // (2) intra-chunk scores, causal mask with the diagonal kept
    {
      const int r = tid / kC, i = tid % kC;
      float p = 0.f;
      if (i <= r && r < nr) {
        const float *qr = sQ + r * ld, *br = sB + r * ld, *wi = sW + i * ld, *bi = sB + i * ld;
        for (int d = 0; d < dk; ++d) p = fmaf(qr[d] * wi[d], expf(br[d] - bi[d]), p);
      }
      sP[tid] = p;
    }
    __syncthreads();
    // fold exp(b_r) into q for the inter-chunk readout (after the scores have used raw q)
    for (int e = tid; e < nr * dk; e += kThreads) {
      const int r = e / dk, d = e % dk;
      sQ[r * ld + d] *= expf(sB[r * ld + d]);
    }
    __syncthreads();
    // (3) output rows
    for (int e = tid; e < kC * kTileV; e += kThreads) {
      const int r = e / kTileV, c = e % kTileV;
      if (r < nr && col0 + c < dv) {
        float acc = 0.f;
        const float* qr = sQ + r * ld;
        if (bd) {
          const float cr = sC[r * kTileV + c];
          for (int d = 0; d < dk; ++d) acc = fmaf(qr[d], sS[d * kTileV + c], acc);
          acc *= expf(cr);
          for (int i = 0; i <= r; ++i)
            acc = fmaf(sP[r * kC + i], sV[i * kTileV + c] * expf(cr - sC[i * kTileV + c]), acc);
        } else {
          for (int i = 0; i <= r; ++i) acc = fmaf(sP[r * kC + i], sV[i * kTileV + c], acc);
          for (int d = 0; d < dk; ++d) acc = fmaf(qr[d], sS[d * kTileV + c], acc);
        }
        const long long i = (long long)(t0 + r) * dv + col0 + c;
        acc *= a.scale;
        if (fd) acc = fmaf(fd[col0 + c], to_f32(fx[i]), acc);   // feed-through d . x'
        o[i] = from_f32<T>(acc);
      }
    }
    __syncthreads();
    // (4) state update: fold exp(b_C - b_i) into ahat*k once, then contract over the chunk
    for (int e = tid; e < nr * dk; e += kThreads) {
      const int i = e / dk, d = e % dk;
      sW[i * ld + d] *= expf(sE[d] - sB[i * ld + d]);
    }
    if (bd) {   // v_i . exp(c_C - c_i), in place (the outputs are done with v)
      for (int e = tid; e < nr * kTileV; e += kThreads)
        sV[e] *= expf(sC[(kC - 1) * kTileV + e % kTileV] - sC[e]);
    }
    __syncthreads();
    for (int e = tid; e < dk * kTileV; e += kThreads) {
      const int d = e / kTileV, c = e % kTileV;
      float acc = expf(sE[d]) * sS[e];
      if (bd) acc *= expf(sC[(kC - 1) * kTileV + c]);
      for (int i = 0; i < nr; ++i) acc = fmaf(sW[i * ld + d], sV[i * kTileV + c], acc);
      sS[e] = acc;
    }
    __syncthreads();
  }

  if (a.sT) {
    for (int e = tid; e < dk * kTileV; e += kThreads) {
      const int d = e / kTileV, c = e % kTileV;
      if (col0 + c < dv) a.sT[s_off + (long long)d * dv + col0 + c] = sS[e];
    }
  }
}

size_t simt_smem_bytes(int dk) {
  const int ld = dk + 1;
  return sizeof(float) * ((size_t)dk * kTileV + 3 * (size_t)kC * ld + 2 * kC * kTileV + kC * kC + dk);
}

// ---------------------------------------------------------------------------------------------
// Chunks side by side
// ---------------------------------------------------------------------------------------------
struct ChunkArgs {
  SimtArgs s;
  float *states;          // [chunk slots of all heads][dk][dv]: dS of the chunk, then the state entering it
  float *qe, *scores, *decay;   // [slots][kC][dk], [slots][kC][kC], [slots][dk]
  int slots_per_head, heads;    // dense: (batch, head) pairs; packed: heads
  long long slots;
};

// A sequence's chunks have consecutive slots: packed sequence n of a head starts at floor(start / 16) + n.
struct ChunkRef {
  int n, h, t, nr, len;         // sequence, head, chunk of the sequence, live rows (0: no such chunk)
  long long row0, slot0;        // first row and first slot of the sequence
};
__device__ __forceinline__ void sequence_of(const ChunkArgs& a, int n, int h, ChunkRef& r) {
  r.n = n;
  r.h = h;
  if (a.s.cu) {
    int lo = a.s.cu[n], hi = a.s.cu[n + 1];
    lo = lo < 0 ? 0 : (lo > a.s.T ? a.s.T : lo);
    hi = hi < lo ? lo : (hi > a.s.T ? a.s.T : hi);
    r.len = hi - lo;
    r.row0 = (long long)h * a.s.T + lo;
    r.slot0 = (long long)h * a.slots_per_head + lo / kC + n;
  } else {
    r.len = a.s.T;
    r.row0 = ((long long)n * a.s.H + h) * a.s.T;
    r.slot0 = ((long long)n * a.s.H + h) * a.slots_per_head;
  }
}
// Block-wide: every one of the block's THREADS threads takes part.
template <int THREADS>
__device__ __forceinline__ ChunkRef chunk_of(const ChunkArgs& a, long long slot) {
  ChunkRef r;
  const int head = (int)(slot / a.slots_per_head), local = (int)(slot % a.slots_per_head);
  if (!a.s.cu) {
    sequence_of(a, head / a.s.H, head % a.s.H, r);
  } else {
    // the last sequence whose first slot is not beyond this one
    const int n = last_that_holds<THREADS>(a.s.n_seq, [&](int m) {
      ChunkRef c;
      sequence_of(a, m, 0, c);
      return c.slot0 <= local;
    });
    r.nr = 0;
    if (n < 0) return r;
    sequence_of(a, n, head, r);
  }
  r.t = (int)(slot - r.slot0);
  r.nr = r.t < 0 ? 0 : min(kC, r.len - r.t * kC);            // (negative only for a bad cu_seqlens)
  return r;
}

// Operands, scores and state contribution of one chunk.  Bound by the latency of its phases.
constexpr int kOpsThreads = 1024;
template <typename T>
__global__ void __launch_bounds__(kOpsThreads, 1) ddts_chunk_ops_kernel(const ChunkArgs a) {
  extern __shared__ float smem[];
  const int dk = a.s.dk, dv = a.s.dv, ld = dk + 1, tid = threadIdx.x;
  float* sQ = smem;                 // [kC][ld] q
  float* sW = sQ + kC * ld;         // [kC][ld] ahat k
  float* sB = sW + kC * ld;         // [kC][ld] log decay, then cumulative
  float* sV = sB + kC * ld;         // [kC][kTileV]
  if (!a.s.cu && blockIdx.x == 0 && tid == 0) a.s.hdr->status = RODIMUS_OK;
  const long long slot = blockIdx.x;
  let_next_kernel_start();
  const ChunkRef r = chunk_of<kOpsThreads>(a, slot);
  if (r.nr <= 0) return;
  const long long row = r.row0 + (long long)r.t * kC;
  // rows of q,k,gx,ty: the head's own, or the sequence's single shared set
  const long long rq = a.s.shared ? row - ((long long)r.h + (a.s.cu ? 0 : (long long)r.n * (a.s.H - 1))) * a.s.T : row;
  for (int e = tid; e < kC * dk; e += kOpsThreads) {
    const int rr = e / dk, d = e % dk;
    float la = 0.f, lh = 0.f, qv = 0.f, kv = 0.f;
    if (rr < r.nr) {
      const long long i = rq * dk + e;
      qv = to_f32(((const T*)a.s.q)[i]);
      kv = to_f32(((const T*)a.s.k)[i]);
      gate_logs_f32(to_f32(((const T*)a.s.gx)[i]), to_f32(((const T*)a.s.ty)[i]), a.s.ingate, la, lh);
    }
    sB[rr * ld + d] = la;
    sW[rr * ld + d] = expf(lh) * kv;
    sQ[rr * ld + d] = qv;
  }
  __syncthreads();
  for (int d = tid; d < dk; d += kOpsThreads) {
    float b = 0.f;
#pragma unroll
    for (int rr = 0; rr < kC; ++rr) {
      b += sB[rr * ld + d];
      sB[rr * ld + d] = b;
    }
    a.decay[slot * dk + d] = expf(b);
  }
  __syncthreads();
  // scores, the difference of the exponents formed before the exponential; four threads a pair
  constexpr int kPairs = kC * (kC + 1) / 2;
  if (tid < 4 * kPairs) {                                     // (whole warps: 544 threads)
    const int p = tid >> 2;
    int rr = 0, i = p;
    while (i > rr) i -= ++rr;
    float v = 0.f;
#pragma unroll 4
    for (int d = tid & 3; d < dk; d += 4)
      v = fmaf(sQ[rr * ld + d] * sW[i * ld + d], expf(sB[rr * ld + d] - sB[i * ld + d]), v);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if ((tid & 3) == 0) a.scores[slot * (kC * kC) + rr * kC + i] = v;
  }
  __syncthreads();
  for (int e = tid; e < kC * dk; e += kOpsThreads) {
    const int rr = e / dk, d = e % dk;
    const float b = sB[rr * ld + d];
    a.qe[slot * (kC * dk) + e] = sQ[rr * ld + d] * expf(b);
    sW[rr * ld + d] *= expf(sB[(kC - 1) * ld + d] - b);       // (rows past the end: decay 0, operand 0)
  }
  const T* v = (const T*)a.s.v + row * dv;
  const T* bh = a.s.beta_hat ? (const T*)a.s.beta_hat + row * dv : nullptr;
  float* ds = a.states + slot * (long long)dk * dv;
  const int c = tid & (kTileV - 1), dg = tid / kTileV, per = dk / (kOpsThreads / kTileV);
  for (int col0 = 0; col0 < dv; col0 += kTileV) {
    __syncthreads();
    for (int e = tid; e < kC * kTileV; e += kOpsThreads) {
      const int rr = e / kTileV, cc = col0 + e % kTileV;
      float vv = 0.f;
      if (rr < r.nr && cc < dv) {
        vv = to_f32(v[(long long)rr * dv + cc]);
        if (bh) vv *= to_f32(bh[(long long)rr * dv + cc]);
      }
      sV[e] = vv;
    }
    __syncthreads();
    if (col0 + c < dv) {
      float vr[kC];
#pragma unroll
      for (int rr = 0; rr < kC; ++rr) vr[rr] = sV[rr * kTileV + c];
      for (int j = 0; j < per; ++j) {
        const int d = dg * per + j;
        float acc = 0.f;
#pragma unroll
        for (int rr = 0; rr < kC; ++rr) acc = fmaf(sW[rr * ld + d], vr[rr], acc);
        ds[(long long)d * dv + col0 + c] = acc;
      }
    }
  }
}

// States entering the chunks and the final state; a thread per four state columns of a key channel.
__global__ void __launch_bounds__(128) ddts_chunk_states_kernel(const ChunkArgs a) {
  let_next_kernel_start();
  const int v4 = a.s.dv / 4;
  const long long per = (long long)a.s.dk * v4;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long sh = idx / per;
  if (sh >= (long long)a.s.n_seq * a.s.H) return;
  const int d = (int)(idx % per / v4), c = (int)(idx % v4) * 4;
  ChunkRef r;
  sequence_of(a, (int)(sh / a.s.H), (int)(sh % a.s.H), r);
  const long long size = (long long)a.s.dk * a.s.dv, e = (long long)d * a.s.dv + c;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (a.s.s0) s = *reinterpret_cast<const float4*>(a.s.s0 + sh * size + e);
  wait_for_previous_kernel();
  const int chunks = (r.len + kC - 1) / kC;
  float* st = a.states + r.slot0 * size + e;
  const float* dec = a.decay + r.slot0 * a.s.dk + d;
  constexpr int kAhead = 8;
  for (int c0 = 0; c0 < chunks; c0 += kAhead) {
    float4 ds[kAhead];
    float f[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      if (c0 + j < chunks) {
        ds[j] = *reinterpret_cast<const float4*>(st + (c0 + j) * size);
        f[j] = dec[(long long)(c0 + j) * a.s.dk];
      }
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      if (c0 + j < chunks) {
        *reinterpret_cast<float4*>(st + (c0 + j) * size) = s;
        s = make_float4(fmaf(f[j], s.x, ds[j].x), fmaf(f[j], s.y, ds[j].y), fmaf(f[j], s.z, ds[j].z), fmaf(f[j], s.w, ds[j].w));
      }
    }
  }
  if (a.s.sT) *reinterpret_cast<float4*>(a.s.sT + sh * size + e) = s;
}

// Outputs of one chunk and kTileV value columns: a thread per column and row.
constexpr int kOutThreads = kC * kTileV;
template <typename T>
__global__ void __launch_bounds__(kOutThreads) ddts_chunk_out_kernel(const ChunkArgs a) {
  extern __shared__ float smem[];
  const int dk = a.s.dk, dv = a.s.dv, tid = threadIdx.x;
  float* sS = smem;                    // [dk][kTileV]
  float* sQ = sS + dk * kTileV;        // [kC][dk]
  float* sV = sQ + kC * dk;            // [kC][kTileV]
  float* sP = sV + kC * kTileV;        // [kC][kC]
  const long long slot = blockIdx.x / (unsigned)a.s.tiles;
  const int col0 = (int)(blockIdx.x % (unsigned)a.s.tiles) * kTileV;
  const ChunkRef r = chunk_of<kOutThreads>(a, slot);
  if (r.nr <= 0) return;
  const long long row = r.row0 + (long long)r.t * kC;
  const int c = tid & (kTileV - 1), rr = tid / kTileV;
  const bool live = rr < r.nr && col0 + c < dv;
  const long long at = (row + rr) * dv + col0 + c;
  float vv = 0.f, fx = 0.f;
  if (live) {
    vv = to_f32(((const T*)a.s.v)[at]);
    if (a.s.beta_hat) vv *= to_f32(((const T*)a.s.beta_hat)[at]);
    if (a.s.feed_d) fx = a.s.feed_d[(long long)r.h * dv + col0 + c] * to_f32(((const T*)a.s.feed_x)[at]);
  }
  wait_for_previous_kernel();
  const float* S = a.states + slot * (long long)dk * dv + col0;
  for (int e = tid; e < dk * (kTileV / 4); e += kOutThreads) {
    const int d = e / (kTileV / 4), c4 = e % (kTileV / 4) * 4;
    if (col0 + c4 < dv) *reinterpret_cast<float4*>(sS + d * kTileV + c4) = *reinterpret_cast<const float4*>(S + (long long)d * dv + c4);
  }
  for (int e = tid; e < kC * dk; e += kOutThreads) sQ[e] = a.qe[slot * (kC * dk) + e];
  if (tid < kC * kC) sP[tid] = a.scores[slot * (kC * kC) + tid];
  sV[tid] = vv;
  __syncthreads();
  if (!live) return;
  float acc = 0.f, acc2 = 0.f;
  for (int i = 0; i <= rr; ++i) acc = fmaf(sP[rr * kC + i], sV[i * kTileV + c], acc);
#pragma unroll 8
  for (int d = 0; d < dk; d += 2) {
    acc = fmaf(sQ[rr * dk + d], sS[d * kTileV + c], acc);
    acc2 = fmaf(sQ[rr * dk + d + 1], sS[(d + 1) * kTileV + c], acc2);
  }
  ((T*)a.s.o)[at] = from_f32<T>(fmaf(acc + acc2, a.s.scale, fx));
}

struct ChunkPlan {
  long long slots;
  int slots_per_head, heads;
  size_t states, qe, scores, decay, bytes;   // workspace offsets, total
};
ChunkPlan chunk_plan(const rodimus_ddts_fwd_params& p) {
  ChunkPlan c;
  const bool varlen = p.cu_seqlens || p.cu_seqlens_host;
  c.heads = varlen ? p.H : p.B * p.H;
  c.slots_per_head = varlen ? p.T / kC + p.N : (p.T + kC - 1) / kC;
  c.slots = (long long)c.heads * c.slots_per_head;
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  c.states = sizeof(WorkspaceHeader) + up((size_t)(varlen ? p.N : 0) * sizeof(int32_t));
  c.qe = c.states + up((size_t)c.slots * p.dk * p.dv * 4);
  c.scores = c.qe + up((size_t)c.slots * kC * p.dk * 4);
  c.decay = c.scores + up((size_t)c.slots * kC * kC * 4);
  c.bytes = c.decay + up((size_t)c.slots * p.dk * 4);
  return c;
}

int chunk_ops_smem_bytes(int dk) { return (int)sizeof(float) * (3 * kC * (dk + 1) + kC * kTileV); }
int chunk_out_smem_bytes(int dk) { return (int)sizeof(float) * (dk * kTileV + kC * dk + kC * kTileV + kC * kC); }

// (The kernels are opted in to the shared memory of the widest keys, once: set to each call's own need, the
// limit could be lowered by another thread between this call's setting and its launch.)
template <typename T>
cudaError_t launch_chunks(const ChunkArgs& a, int dev, cudaStream_t st) {
  static std::atomic<unsigned long long> opted_ops{0}, opted_out{0};   // per instantiation
  const int smem_ops = chunk_ops_smem_bytes(a.s.dk), smem_out = chunk_out_smem_bytes(a.s.dk);
  cudaError_t e = opt_in_shared_memory(ddts_chunk_ops_kernel<T>, chunk_ops_smem_bytes(kMaxDk), dev, opted_ops);
  if (e == cudaSuccess) e = opt_in_shared_memory(ddts_chunk_out_kernel<T>, chunk_out_smem_bytes(kMaxDk), dev, opted_out);
  if (e != cudaSuccess) return e;
  const long long threads = (long long)a.s.n_seq * a.s.H * a.s.dk * (a.s.dv / 4);
  ddts_chunk_ops_kernel<T><<<(unsigned)a.slots, kOpsThreads, smem_ops, st>>>(a);
  e = launch_overlapped(ddts_chunk_states_kernel, (unsigned)((threads + 127) / 128), 128, 0, st, a);
  if (e == cudaSuccess)
    e = launch_overlapped(ddts_chunk_out_kernel<T>, (unsigned)(a.slots * a.s.tiles), kOutThreads, smem_out, st, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Workspace with which this kernel's chunks are computed side by side; 0: they are not.  The states of
// the chunks cross memory four times: up to 64 MiB of them, which stay in L2 (126 MB).
// B=1 H=1 T=256 dk=dv=64 fp32: one CTA walking the 16 chunks 318 us, side by side 16.4 us a call.
// The walk takes 4 to 45 us a chunk (dk = 16 to 256) whether it has sixteen rows or one, for several CTAs on
// an SM at once (one with dk > 128); this form pays for every chunk and column tile, so it is not taken where
// chunks are mostly empty and more than fill the device by themselves: 1024 items of 17 rows, dk = dv = 64,
// 121 us in the walk and 174 side by side, of 48 rows 364 and 304; 300 items of 33 rows 101 and 82; 148 of
// 17 31 and 31; 64 of 17, dk = dv = 256, 133 and 99.  And one block forms a chunk's whole contribution to the
// state, one column tile after another: with dk = 256, dv = 1024 in 110 us, so that needs three chunks to pay
// (17 rows 68 and 123 us, 33 113 and 124, 48 141 and 124), two where the walk's CTAs take several rounds (16
// items of 17 rows 133 and 160, of 32 190 and 172).
size_t fwd_simt_chunks_workspace_bytes(const rodimus_ddts_fwd_params& p) {
  if (p.value_decay || (long long)p.B * p.H * p.T == 0 || p.T <= kC) return 0;
  const bool varlen = p.cu_seqlens || p.cu_seqlens_host;
  if (varlen && p.N == 0) return 0;
  const ChunkPlan c = chunk_plan(p);
  const long long tiles = (p.dv + kTileV - 1) / kTileV;
  if (c.slots * tiles > 0x7fffffffLL) return 0;
  if (c.qe - c.states > (size_t)64 << 20) return 0;
  int dev = 0, sms = 0;
  if (current_device(&dev, &sms) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  // chunks of a head: of a packed call about half of a chunk a sequence is left over
  const double chunks = varlen ? (double)p.T / kC + 0.5 * p.N : (double)c.slots_per_head;
  const double rows = p.T / chunks, work = chunks * c.heads * tiles;
  if (rows < 12.0 && work > (rows < 10.0 ? 2.0 : 16.0) * (p.dk > 128 ? 4.0 : 1.0) * sms) return 0;
  const long long n_seq = varlen ? p.N : p.B;
  if (p.dk * p.dv > 65536 && p.T < (n_seq * p.H * tiles > sms ? 2 : 3) * kC * (varlen ? n_seq : 1)) return 0;
  return c.bytes;
}

cudaError_t launch_fwd_simt(const rodimus_ddts_fwd_params& p, int* n_launches) {
  *n_launches = 0;
  SimtArgs a;
  a.q = p.q; a.k = p.k; a.gx = p.gate_x; a.ty = p.temp_y; a.v = p.v; a.o = p.o;
  a.beta_hat = p.beta_hat; a.feed_x = p.feed_x; a.feed_d = p.feed_d; a.vdecay = p.value_decay;
  a.s0 = p.s0; a.sT = p.sT; a.cu = p.cu_seqlens;
  a.hdr = reinterpret_cast<WorkspaceHeader*>(p.workspace);
  a.H = p.H; a.T = p.T; a.dk = p.dk; a.dv = p.dv;
  a.n_seq = p.cu_seqlens ? p.N : p.B;
  a.tiles = (p.dv + kTileV - 1) / kTileV;
  a.scale = p.scale; a.ingate = p.ingate; a.shared = p.shared_gates;
  const long long items = (long long)a.n_seq * p.H * a.tiles;
  if (items == 0) return cudaSuccess;
  if (items > 0x7fffffffLL) return cudaErrorInvalidValue;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(p.stream);
  int dev = 0, sms = 0;
  cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  const size_t chunks = fwd_simt_chunks_workspace_bytes(p);
  if (chunks > 0 && p.workspace_bytes >= chunks) {
    const ChunkPlan c = chunk_plan(p);
    char* ws = reinterpret_cast<char*>(p.workspace);
    ChunkArgs ca;
    ca.s = a;
    ca.states = reinterpret_cast<float*>(ws + c.states);
    ca.qe = reinterpret_cast<float*>(ws + c.qe);
    ca.scores = reinterpret_cast<float*>(ws + c.scores);
    ca.decay = reinterpret_cast<float*>(ws + c.decay);
    ca.slots_per_head = c.slots_per_head;
    ca.heads = c.heads;
    ca.slots = c.slots;
    e = p.dtype == RODIMUS_BF16 ? launch_chunks<__nv_bfloat16>(ca, dev, st) : launch_chunks<float>(ca, dev, st);
    *n_launches = 3;
    return e;
  }
  const bool bf16 = p.dtype == RODIMUS_BF16;
  auto* const kernel = bf16 ? ddts_fwd_simt_kernel<__nv_bfloat16> : ddts_fwd_simt_kernel<float>;
  static std::atomic<unsigned long long> opted[2];
  e = opt_in_shared_memory(kernel, (int)simt_smem_bytes(kMaxDk), dev, opted[bf16]);
  if (e != cudaSuccess) return e;
  kernel<<<(unsigned)items, kThreads, simt_smem_bytes(p.dk), st>>>(a);
  *n_launches = 1;
  return cudaGetLastError();
}

}  // namespace ddts
