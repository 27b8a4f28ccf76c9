// KV append: store the new tokens, refresh the block statistics the Taylor score reads (Section 3.1,
// Eq. taylor-2nd: block key mean and diagonal population covariance) and advance the global linear-attention
// state S_bar += phi(k_t)^T v_t in fp32 (Section 3.2, Eq. rla-impl-1, "Numerical Stability").
//
// Appends of up to 32 tokens per sequence (the decode loop) run as ONE fused kernel, see append_fused_kernel.
// Longer appends of a bf16 cache with d = 128 run as one pass on the tensor cores (append_bulk.cu); all others as three
// kernels in stream order, all reading the OLD sequence lengths until the last one bumps them:
//   block  : one CTA per touched block: its keys (cached ones below the old length, new ones above) are staged in
//            shared memory once; from there the new tokens go to the cache (k_new, v_new -> cache), their
//            logsumexp of phi_scale * k to tok_lse, and the block's mean / variance records are recomputed (two
//            exact passes, so the result does not depend on how the tokens were split across append calls)
//   state  : rank-n update of S_bar on the FMA pipe, shares of the tokens side by side and then added
//   lengths: seq_lens += n_new
#include "spla_internal.h"

namespace spla {

constexpr int kStateRows = 16;     // rows of S_bar per CTA where there are few units
constexpr int kStateTokens = 32;   // tokens staged per inner step
constexpr int kStateShare = 256;   // tokens per share of a unit, at least (below, a share's fixed cost outweighs what it takes off)

__device__ __forceinline__ int tokens_to_add(const Params& p, const int* n_new, int max_new, int b, int L) {
  int n = n_new ? n_new[b] : max_new;
  n = max(0, min(n, max_new));
  if (L < 0 || L + n > p.max_context) return -1;   // would overflow (or a corrupt length): skip this sequence, the caller is told via status
  return n;
}

template <int BYTES>
__device__ __forceinline__ void copy_bytes(void* dst, const void* src) {
  if constexpr (BYTES == 16) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
  else if constexpr (BYTES == 8) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src);
  else *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(src);
}

// Mean and population variance of one selection window of one block (window w covers the block's tokens
// [w * win_s, w * win_s + win_C); without strided windows that is the whole block), two exact passes, by
// kStatThreads threads (groups of D threads take every TG-th token; the partial sums are combined in a fixed
// order, so every append path gives the same bits).  `key_at(t)` returns channel (tid % D) of the block's token t.
// A window that holds no token yet is left alone.
constexpr int kStatThreads = 256;
template <int D, bool WIN, typename KeyAt>
__device__ __forceinline__ void block_stats_core(const Params& p, int u, int blk, int w, int L_total, bool act,
                                                 float (*red_s)[D], float* mean_s, KeyAt key_at) {
  constexpr int TG = kStatThreads / D;
  const int tid = threadIdx.x;
  const int t0 = blk * p.B;
  const int t_lo = WIN ? w * p.win_s : 0;
  const int t_hi = act ? (WIN ? min(min(p.B, L_total - t0), t_lo + p.win_C) : min(p.B, L_total - t0)) : 0;   // tokens [t_lo, t_hi)
  const int cnt = max(0, t_hi - t_lo);
  act = act && cnt > 0;
  const int tg = tid / D, c = tid % D;
  float sum = 0.f;
#pragma unroll 8
  for (int t = t_lo + tg; t < t_hi; t += TG) sum += key_at(t);
  red_s[tg][c] = sum;
  __syncthreads();
  if (tg == 0) {
    float tot = 0.f;
#pragma unroll
    for (int g2 = 0; g2 < TG; ++g2) tot += red_s[g2][c];
    mean_s[c] = cnt > 0 ? tot / (float)cnt : 0.f;
  }
  __syncthreads();
  const float mean = mean_s[c];
  float ss = 0.f;
#pragma unroll 8
  for (int t = t_lo + tg; t < t_hi; t += TG) {
    const float dv = key_at(t) - mean;
    ss = fmaf(dv, dv, ss);
  }
  __syncthreads();
  red_s[tg][c] = ss;
  __syncthreads();
  if (tg == 0 && act) {
    float tot = 0.f;
#pragma unroll
    for (int g2 = 0; g2 < TG; ++g2) tot += red_s[g2][c];
    const size_t rec_off = (WIN ? ((size_t)u * p.max_blocks + blk) * p.NW + w : (size_t)u * p.max_blocks + blk) * 2 * D;
    if (p.flags & kStatsBf16) {                      // 16-bit records: rounded once, here
      __nv_bfloat16* rec = reinterpret_cast<__nv_bfloat16*>(p.stats) + rec_off;
      rec[c] = __float2bfloat16_rn(mean);
      rec[D + c] = __float2bfloat16_rn(tot / (float)cnt);
    } else {
      float* rec = p.stats + rec_off;
      rec[c] = mean;
      rec[D + c] = tot / (float)cnt;
    }
  }
}

// The same from global memory: token t of the block comes from the cache if its position is below `L_cached`,
// else from the new tokens `kn`.
template <typename T, int D, bool WIN>
__device__ __forceinline__ void block_stats_role(const Params& p, int u, int blk, int w, int L_cached, int L_total, const T* kn,
                                                 bool act, float (*red_s)[D], float* mean_s) {
  const int t0 = blk * p.B;
  const int c = threadIdx.x % D;
  const T* kc = reinterpret_cast<const T*>(p.k_cache) + ((size_t)u * p.max_blocks * p.B + t0) * D + c;
  // One address per token (cached or new) and one load from it: no branch around the loads, so that the
  // unrolled loop keeps several of them in flight.
  block_stats_core<D, WIN>(p, u, blk, w, L_total, act, red_s, mean_s, [&](int t) {
    const int pos = t0 + t;
    const T* src = pos < L_cached ? kc + (size_t)t * D : kn + (size_t)(pos - L_cached) * D + c;
    return to_float(*src);
  });
}

// Bulk append, one CTA per touched block (blockIdx.x-th block at or after the one the old length falls in).  The
// block's keys are staged once in shared memory, 16 bytes per thread and load, several loads in flight: cached
// keys below the old length, new keys above it; the new keys and values go on to the cache from the same
// registers.  Then, from shared memory: the per-token logsumexp of the new tokens (one warp per token) and the
// statistics records of all the block's windows.
constexpr int kBlockLoads = 4;                       // 16-byte loads of K (and of V) in flight per thread
template <typename T, int D>
__global__ void __launch_bounds__(kStatThreads) append_block_kernel(const Params p, const T* __restrict__ k_new,
                                                                    const T* __restrict__ v_new,
                                                                    const int* __restrict__ n_new, int max_new) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  __shared__ float red_s[kStatThreads / D][D];
  __shared__ float mean_s[D];
  constexpr int VEC = D / 32;
  pdl_wait();
  constexpr int CH = D * (int)sizeof(T) / 16;        // 16-byte chunks per token
  T* tile = reinterpret_cast<T*>(tile_raw);          // [B][D]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int u = blockIdx.y, b = u / p.Hkv;
  const int L = p.seq_lens[b];
  const int n = tokens_to_add(p, n_new, max_new, b, L);
  if (n < 0) {
    if (blockIdx.x == 0 && tid == 0) atomicExch(p.status, kStatusCapacity);
    return;
  }
  const int blk = L / p.B + blockIdx.x;
  const int t0 = blk * p.B;
  if (n == 0 || t0 >= L + n) return;                 // CTA-uniform
  const int cnt = min(p.B, L + n - t0);              // tokens the block holds after the append
  if ((p.flags & kDebugBounds) && (blk < 0 || blk >= p.max_blocks)) {   // checked build: the block must exist (CTA-uniform)
    if (tid == 0) atomicExch(p.status, kStatusBounds);
    return;
  }
  const int t_new = max(0, L - t0);                  // its first new token

  const size_t blk_tok0 = (size_t)u * p.max_blocks * p.B + t0;
  uint4* kc = reinterpret_cast<uint4*>(reinterpret_cast<T*>(p.k_cache) + blk_tok0 * D);
  uint4* vc = reinterpret_cast<uint4*>(reinterpret_cast<T*>(p.v_cache) + blk_tok0 * D);
  // new token i of the unit sits at chunk (t0 - L + t) * CH + ch of kn / vn
  const uint4* kn = reinterpret_cast<const uint4*>(k_new + (size_t)u * max_new * D) + (ptrdiff_t)(t0 - L) * CH;
  const uint4* vn = reinterpret_cast<const uint4*>(v_new + (size_t)u * max_new * D) + (ptrdiff_t)(t0 - L) * CH;
  uint4* tile4 = reinterpret_cast<uint4*>(tile_raw);
  const int total = cnt * CH, first_new = t_new * CH;
  for (int base = 0; base < total; base += kBlockLoads * kStatThreads) {
    uint4 kk[kBlockLoads], vv[kBlockLoads];
#pragma unroll
    for (int j = 0; j < kBlockLoads; ++j) {
      const int idx = base + j * kStatThreads + tid;
      if (idx < total) {
        if (idx >= first_new) { kk[j] = __ldcs(kn + idx); vv[j] = __ldcs(vn + idx); }
        else kk[j] = kc[idx];
      }
    }
#pragma unroll
    for (int j = 0; j < kBlockLoads; ++j) {
      const int idx = base + j * kStatThreads + tid;
      if (idx < total) {
        tile4[idx] = kk[j];
        if (idx >= first_new) { kc[idx] = kk[j]; vc[idx] = vv[j]; }
      }
    }
  }
  __syncthreads();

  // per-token logsumexp of phi_scale * k, the value the decode and the state update read
  for (int t = t_new + warp; t < cnt; t += kStatThreads / 32) {
    float k[VEC];
    load_vec<VEC>(tile + (size_t)t * D + lane * VEC, k);
    const float lse = token_lse<VEC>(k, p.phi_scale);
    if (lane == 0) p.tok_lse[blk_tok0 + t] = lse;
  }

  const int c = tid % D;
  for (int w = 0; w < p.NW; ++w) {
    block_stats_core<D, true>(p, u, blk, w, L + n, true, red_s, mean_s,
                              [&](int t) { return to_float(tile[(size_t)t * D + c]); });
    __syncthreads();                                 // the next window reuses the reduction buffers
  }
  // Only now: the small CTAs of the state kernel, started earlier, crowd onto the SMs that have room first (bf16, d = 64, 255 tokens
  // x 32 units: 57 us a call against 21; 600 tokens x 400 units 138 against 100).
  pdl_launch_dependents();
}

// S_bar += phi(K)^T V on the FMA pipe: ROWS rows of S_bar per CTA over one share of a unit's new tokens, staged kStateTokens at a
// time (the next ones are on their way to registers meanwhile); a thread owns RT x 8 outputs, so that a staged value feeds eight
// or RT products.  Every output adds its tokens in order; shares are added in share order by append_merge_state_kernel.
// Bound by issuing FMAs (two per instruction).  One CTA per 16 rows used to walk all tokens, one load per token in the chain:
// fp32, d = 64, 16384 tokens x 4 units 1860 -> 52 us a call, 255 tokens 37 -> 19; fp32, d = 128 3399 -> 109.
template <typename T, int D, int ROWS, int RT>
__global__ void __launch_bounds__(ROWS / RT * (D / 8)) append_state_kernel(const Params p, const T* __restrict__ k_new,
                                                                           const T* __restrict__ v_new,
                                                                           const int* __restrict__ n_new, int max_new) {
  constexpr int NT = ROWS / RT * (D / 8);
  constexpr int E = 16 / (int)sizeof(T);                    // elements per 16-byte piece
  constexpr int CHK = ROWS / E, CHV = D / E;                // pieces per token: of the CTA's channels of K, of V
  constexpr int NK = (kStateTokens * CHK + NT - 1) / NT, NV = (kStateTokens * CHV + NT - 1) / NT;
  __shared__ __align__(16) float phi_s[kStateTokens][ROWS];
  __shared__ __align__(16) float v_s[kStateTokens][D];
  pdl_wait();
  pdl_launch_dependents();
  const int u = blockIdx.y, b = u / p.Hkv, tid = threadIdx.x;
  const int L = p.seq_lens[b];
  const int n = max(0, tokens_to_add(p, n_new, max_new, b, L));
  const int S = gridDim.z, share = blockIdx.z;
  const int per = ((n + S - 1) / S + kStateTokens - 1) / kStateTokens * kStateTokens;
  const int t_lo = min(n, share * per), t_hi = min(n, t_lo + per);
  const int row0 = blockIdx.x * ROWS;
  if (S == 1 && n == 0) return;
  const float a2 = p.phi_scale * kLog2e;
  const float* lse = p.tok_lse + (size_t)u * p.max_blocks * p.B + L;
  const T* kn = k_new + (size_t)u * max_new * D + row0;
  const T* vn = v_new + (size_t)u * max_new * D;
  uint4 kr[NK], vr[NV];
  float lr[NK];
  auto fetch = [&](int t0) {
#pragma unroll
    for (int j = 0; j < NK; ++j) {
      const int x = j * NT + tid, t = x / CHK, c = x % CHK;
      const bool in = t < kStateTokens && t0 + t < t_hi;
      kr[j] = in ? __ldg(reinterpret_cast<const uint4*>(kn + (size_t)(t0 + t) * D) + c) : make_uint4(0u, 0u, 0u, 0u);
      lr[j] = in ? -__ldcg(lse + t0 + t) * kLog2e : -INFINITY;    // (phi of a token that is not there: 0)
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int x = j * NT + tid, t = x / CHV, c = x % CHV;
      const bool in = t < kStateTokens && t0 + t < t_hi;
      vr[j] = in ? __ldg(reinterpret_cast<const uint4*>(vn + (size_t)(t0 + t) * D) + c) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  auto floats = [](const uint4& r, float (&x)[E]) {
    if constexpr (E == 4) {
      x[0] = __uint_as_float(r.x); x[1] = __uint_as_float(r.y); x[2] = __uint_as_float(r.z); x[3] = __uint_as_float(r.w);
    } else {
      x[0] = bf16_lo(r.x); x[1] = bf16_hi(r.x); x[2] = bf16_lo(r.y); x[3] = bf16_hi(r.y);
      x[4] = bf16_lo(r.z); x[5] = bf16_hi(r.z); x[6] = bf16_lo(r.w); x[7] = bf16_hi(r.w);
    }
  };
  const int rg = tid / (D / 8) * RT, c4 = tid % (D / 8) * 4;  // the thread's rows; its columns c4 .. + 3 and D / 2 + c4 .. + 3
  float2 acc[RT][4];
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.f, 0.f);
  if (t_lo < t_hi) fetch(t_lo);
  for (int t0 = t_lo; t0 < t_hi; t0 += kStateTokens) {
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NK; ++j) {
      const int x = j * NT + tid, t = x / CHK, c = x % CHK;
      if (t < kStateTokens) {
        float k[E];
        floats(kr[j], k);
#pragma unroll
        for (int e = 0; e < E; ++e) k[e] = exp2f(fmaf(k[e], a2, lr[j]));
#pragma unroll
        for (int e = 0; e < E; e += 4) *reinterpret_cast<float4*>(&phi_s[t][c * E + e]) = make_float4(k[e], k[e + 1], k[e + 2], k[e + 3]);
      }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int x = j * NT + tid, t = x / CHV, c = x % CHV;
      if (t < kStateTokens) {
        float v[E];
        floats(vr[j], v);
#pragma unroll
        for (int e = 0; e < E; e += 4) *reinterpret_cast<float4*>(&v_s[t][c * E + e]) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
      }
    }
    __syncthreads();
    if (t0 + kStateTokens < t_hi) fetch(t0 + kStateTokens);
    const int nt = min(kStateTokens, t_hi - t0);
#pragma unroll 2
    for (int t = 0; t < nt; ++t) {
      float f[RT];
#pragma unroll
      for (int r = 0; r < RT; r += 2) {
        if constexpr (RT % 4 == 0) {
          if (r % 4 == 0) {
            const float4 x = *reinterpret_cast<const float4*>(&phi_s[t][rg + r]);
            f[r] = x.x; f[r + 1] = x.y; f[r + 2] = x.z; f[r + 3] = x.w;
          }
        } else {
          const float2 x = *reinterpret_cast<const float2*>(&phi_s[t][rg + r]);
          f[r] = x.x; f[r + 1] = x.y;
        }
      }
      const float4 v0 = *reinterpret_cast<const float4*>(&v_s[t][c4]), v1 = *reinterpret_cast<const float4*>(&v_s[t][D / 2 + c4]);
      const float2 v[4] = {make_float2(v0.x, v0.y), make_float2(v0.z, v0.w), make_float2(v1.x, v1.y), make_float2(v1.z, v1.w)};
#pragma unroll
      for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = __ffma2_rn(make_float2(f[r], f[r]), v[c], acc[r][c]);
    }
  }
  float* dst = (S > 1 ? p.state_part + ((size_t)u * S + share) * D * D : p.state + (size_t)u * D * D) + (size_t)(row0 + rg) * D + c4;
#pragma unroll
  for (int r = 0; r < RT; ++r) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4* d4 = reinterpret_cast<float4*>(dst + (size_t)r * D + h * (D / 2));
      float4 o = S > 1 ? make_float4(0.f, 0.f, 0.f, 0.f) : *d4;
      o.x += acc[r][2 * h].x; o.y += acc[r][2 * h].y; o.z += acc[r][2 * h + 1].x; o.w += acc[r][2 * h + 1].y;
      *d4 = o;
    }
  }
}

__global__ void append_lengths_kernel(const Params p, const int* __restrict__ n_new, int max_new) {
  pdl_wait();
  pdl_launch_dependents();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= p.batch) return;
  const int L = p.seq_lens[b];
  const int n = tokens_to_add(p, n_new, max_new, b, L);
  if (n > 0) p.seq_lens[b] = L + n;
}

// ---------------------------------------------------------------------------------------------------------
// Decode-step appends (a few tokens per sequence): everything above in ONE launch.  CTAs take one of three roles
// by blockIdx.x; no role needs another's output, because the new tokens are read from k_new / v_new directly
// (statistics of the open block: cached keys below the old length, new keys above it; state: the per-token
// log-sum-exp is recomputed from the new keys).  Every CTA reads the old lengths; the last CTA to have read them
// (atomic ticket at the start, nobody waits) advances them.
constexpr int kFusedThreads = 256;
constexpr int kFusedMaxNew = kAppendStepMax;

// ROWS: rows of S_bar per CTA of the state role.  Few rows spread a unit over many SMs where there are few units; with many
// units the launch is bound by the number of its CTAs, and each takes more (512 units: 28 -> 20 us with
// 32 rows and one statistics CTA per block that one token can touch; 64 and 128 rows 20 and 24 us).
template <typename T, int D, bool WIN, int ROWS>
__global__ void __launch_bounds__(kFusedThreads, 4) append_fused_kernel(const Params p, const T* __restrict__ k_new,
                                                                     const T* __restrict__ v_new,
                                                                     const int* __restrict__ n_new, int max_new, int n_copy,
                                                                     int n_stats) {
  constexpr int VEC = D / 32;
  constexpr int TG = kFusedThreads / D;            // thread groups of D threads
  __shared__ float red_s[TG][D];
  __shared__ float mean_s[D];
  __shared__ float phi_s[kFusedMaxNew][ROWS];
  __shared__ float lse_s[kFusedMaxNew];
  __shared__ int last_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int u = blockIdx.y, b = u / p.Hkv;
  int role = blockIdx.x;

  pdl_wait();                                      // the preceding decode still reads the cache and the lengths
  pdl_launch_dependents();
  const int L = p.seq_lens[b];
  const int n = tokens_to_add(p, n_new, max_new, b, L);
  const T* kn = k_new + (size_t)u * max_new * D;
  const T* vn = v_new + (size_t)u * max_new * D;
  const size_t unit_tok0 = (size_t)u * p.max_blocks * p.B;

  // ---- the lengths are advanced by whichever CTA is the last to have read them ----------------------------------
  // Every CTA works from the length it read above.  Once all CTAs of the launch hold theirs (the barrier below
  // consumes each thread's value, so no load of a length is still in flight), the last one to check in may store the
  // new lengths while the others are still busy: nothing in this launch reads them again, and the next kernel
  // starts after this grid has completed.  No fence and no wait at the end of the kernel.
  if (__syncthreads_or(L < 0)) return;               // (lengths are never negative)
  if (tid == 0) {
    const int t = atomicAdd(p.append_ticket, 1);
    last_s = (t == (int)(gridDim.x * gridDim.y) - 1);
    if (last_s) *p.append_ticket = 0;
  }
  __syncthreads();
  if (last_s) {
    for (int bb = tid; bb < p.batch; bb += kFusedThreads) {
      const int Lb = p.seq_lens[bb];
      const int nb = tokens_to_add(p, n_new, max_new, bb, Lb);
      if (nb > 0) p.seq_lens[bb] = Lb + nb;
    }
  }

  if (role < n_copy) {
    // ---- copy role: one warp per token; also the per-token log-sum-exp the decode reads ------------------
    if (n < 0 && role == 0 && tid == 0) atomicExch(p.status, kStatusCapacity);
    const int i = role * (kFusedThreads / 32) + warp;
    bool in_cache = true;
    if ((p.flags & kDebugBounds) && n > 0 && i < n && L + i >= p.max_blocks * p.B) {   // checked build
      if (lane == 0) atomicExch(p.status, kStatusBounds);
      in_cache = false;
    }
    if (n > 0 && i < n && in_cache) {
      const size_t pos = unit_tok0 + (size_t)(L + i);
      float k[VEC];
      load_vec<VEC>(kn + (size_t)i * D + lane * VEC, k);
      copy_bytes<VEC * sizeof(T)>(reinterpret_cast<T*>(p.k_cache) + pos * D + lane * VEC, kn + (size_t)i * D + lane * VEC);
      copy_bytes<VEC * sizeof(T)>(reinterpret_cast<T*>(p.v_cache) + pos * D + lane * VEC, vn + (size_t)i * D + lane * VEC);
      const float lse = token_lse<VEC>(k, p.phi_scale);
      if (lane == 0) p.tok_lse[pos] = lse;
    }
  } else if ((role -= n_copy) < n_stats) {
    // ---- statistics role: one touched block; cached keys below the old length, new keys above it -----------
    const int blk = L / p.B + (WIN ? role / p.NW : role);
    block_stats_role<T, D, WIN>(p, u, blk, WIN ? role % p.NW : 0, L, L + max(n, 0), kn, n > 0 && blk * p.B < L + n, red_s, mean_s);
  } else if (!(p.flags & 4u)) {
    // ---- state role: S_bar[row0 .. row0 + ROWS - 1][:] += sum_t phi(k_t)[row] v_t ------------------------------------
    role -= n_stats;
    const int row0 = role * ROWS;
    const int nn = max(n, 0);
    const float a2 = p.phi_scale * kLog2e;
    // The rows of S_bar this thread will update are requested first: the load comes from DRAM and would
    // otherwise sit at the end of the role's dependency chain.
    constexpr int RPT = ROWS / TG;                         // rows per thread
    const int tg = tid / D, j = tid % D;
    float* S = p.state + (size_t)u * D * D + (size_t)(row0 + tg * RPT) * D + j;
    float s_old[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) s_old[r] = nn > 0 ? __ldcs(S + (size_t)r * D) : 0.f;
    // log-sum-exp of every new token: 8 threads per token, D / 8 consecutive channels each, loaded up front
    {
      constexpr int CPT = D / 8;                                 // channels per thread
      const int t = tid >> 3, part = tid & 7;
      float x[CPT];
      if (t < nn) {
#pragma unroll
        for (int c4 = 0; c4 < CPT / 4; ++c4) {
          float y[4];
          load_vec<4>(kn + (size_t)t * D + part * CPT + c4 * 4, y);
#pragma unroll
          for (int v = 0; v < 4; ++v) x[c4 * 4 + v] = y[v] * a2;
        }
      } else {
#pragma unroll
        for (int v = 0; v < CPT; ++v) x[v] = -INFINITY;
      }
      float mx = -INFINITY, sm = 0.f;
#pragma unroll
      for (int v = 0; v < CPT; ++v) mx = fmaxf(mx, x[v]);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
      if (t < nn) {
#pragma unroll
        for (int v = 0; v < CPT; ++v) sm += exp2f(x[v] - mx);
      }
      sm += __shfl_xor_sync(0xffffffffu, sm, 1);
      sm += __shfl_xor_sync(0xffffffffu, sm, 2);
      sm += __shfl_xor_sync(0xffffffffu, sm, 4);
      if (t < nn && part == 0) lse_s[t] = mx + log2f(sm);        // base-2 domain
    }
    __syncthreads();
    for (int idx = tid; idx < nn * ROWS; idx += kFusedThreads) {
      const int t = idx / ROWS, r = idx % ROWS;
      phi_s[t][r] = exp2f(to_float(kn[(size_t)t * D + row0 + r]) * a2 - lse_s[t]);
    }
    __syncthreads();
    float acc[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) acc[r] = 0.f;
    for (int t = 0; t < nn; ++t) {
      const float v = to_float(vn[(size_t)t * D + j]);
#pragma unroll
      for (int r = 0; r < RPT; ++r) acc[r] = fmaf(phi_s[t][tg * RPT + r], v, acc[r]);
    }
    if (nn > 0) {
#pragma unroll
      for (int r = 0; r < RPT; ++r) S[(size_t)r * D] = s_old[r] + acc[r];
    }
  }

}

template <typename T, int D>
static cudaError_t launch_typed(const Params& p, const void* k_new, const void* v_new, const int* n_new, int max_new,
                                const AttendMaps* maps, const AttendMaps* fresh_maps, cudaStream_t stream) {
  const int U = p.batch * p.Hkv;
  const T* kn = reinterpret_cast<const T*>(k_new);
  const T* vn = reinterpret_cast<const T*>(v_new);
  if (max_new <= kFusedMaxNew) {
    const int n_copy = (max_new + kFusedThreads / 32 - 1) / (kFusedThreads / 32);
    const int n_stats = ((max_new + p.B - 2) / p.B + 1) * p.NW;   // one CTA per window of every block that can be touched
    const bool wide = (long long)U * (D / kStateRows) > 4LL * 148;   // more small state CTAs than run at once
    constexpr int kWideRows = 32;
    const int n_state = (p.flags & 4u) ? 0 : D / (wide ? kWideRows : kStateRows);
    // Same shared-memory carve-out as the decode kernels around it: a change of carve-out drains the SMs.
    auto kern = p.NW > 1 ? (wide ? append_fused_kernel<T, D, true, kWideRows> : append_fused_kernel<T, D, true, kStateRows>)
                         : (wide ? append_fused_kernel<T, D, false, kWideRows> : append_fused_kernel<T, D, false, kStateRows>);
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return launch_ex(kern, dim3(n_copy + n_stats + n_state, U), dim3(kFusedThreads), 0, stream, 0, true,
                     p, kn, vn, n_new, max_new, n_copy, n_stats);
  }
  // bf16 with d = 128: everything in one pass, the state on the tensor cores; the rest in three kernels.  Among those a few tokens
  // of many sequences of different lengths: the pass takes a CTA per unit and SM whatever a unit adds, 0.1 us per unit, the
  // kernels take less the less there is (1 to 33, 40 tokens, 512 units: 26, 28 us against 53; 1024 units 44, 47 against 96; 304 units
  // 21, 21 against 39; all at the longest, 512 units: 33, 35 against 55).  The line was drawn where an earlier state kernel fell
  // behind; with this one the kernels stay ahead further on, up to about 80 tokens and below 296 units too (1 to 48, 64, 80, 128
  // tokens, 512 units: 31, 33, 41, 57 us against 53, 53, 54, 58; 296 units 22, 23, 30, 41 against 30, 30, 30, 35).
  const bool few_of_many = n_new && U > 2 * 148 && max_new < 48;
  if (sizeof(T) == 2 && D == 128 && maps && maps->valid && fresh_maps && fresh_maps->valid && !few_of_many)
    return launch_append_bulk(p, *maps, *fresh_maps, n_new, max_new, stream);
  {
    const size_t tile_bytes = (size_t)p.B * D * sizeof(T);
    auto kern = append_block_kernel<T, D>;
    if (tile_bytes > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_bytes);
    const cudaError_t e = launch_ex(kern, dim3((max_new + p.B - 1) / p.B + 1, U), dim3(kStatThreads), tile_bytes, stream, 0, true, p, kn, vn, n_new, max_new);
    if (e != cudaSuccess) return e;
  }
  if (!(p.flags & 4u)) {
    const int most = append_max_shares(U), want = (max_new + kStateShare - 1) / kStateShare, S = want < most ? want : most;
    // All rows per CTA where units and shares fill the device (less is staged more than once), 16 rows where they do not.
    cudaError_t e;
    if ((long long)U * S >= 148)
      e = launch_ex(append_state_kernel<T, D, D, D / 16>, dim3(1, U, S), dim3(2 * D), 0, stream, 0, true, p, kn, vn, n_new, max_new);
    else
      e = launch_ex(append_state_kernel<T, D, kStateRows, 2>, dim3(D / kStateRows, U, S), dim3(D), 0, stream, 0, true, p, kn, vn, n_new, max_new);
    if (e == cudaSuccess && S > 1) e = launch_append_merge_state(p, S, stream);
    if (e != cudaSuccess) return e;
  }
  return launch_ex(append_lengths_kernel, dim3((p.batch + 127) / 128), dim3(128), 0, stream, 0, true, p, n_new, max_new);
}

cudaError_t launch_append(const Params& p, const void* k_new, const void* v_new, const int* n_new, int max_new,
                          const AttendMaps* maps, const AttendMaps* fresh_maps, cudaStream_t stream) {
  if (p.kv_bf16)
    return p.d == 128 ? launch_typed<__nv_bfloat16, 128>(p, k_new, v_new, n_new, max_new, maps, fresh_maps, stream)
                      : launch_typed<__nv_bfloat16, 64>(p, k_new, v_new, n_new, max_new, maps, fresh_maps, stream);
  return p.d == 128 ? launch_typed<float, 128>(p, k_new, v_new, n_new, max_new, maps, fresh_maps, stream)
                    : launch_typed<float, 64>(p, k_new, v_new, n_new, max_new, maps, fresh_maps, stream);
}

}  // namespace spla
