// Per-position pieces of the tensor-core prefill path that precede the scoring: the log mass of every position's own,
// growing block, and the recurrent state at the start of every range of SB tokens.
//
// Section 3.1 (Eq. taylor-2nd) and Section 3.2 (Eq. rla-impl-1) of the paper, for every prefix that ends inside the
// chunk.  Nothing here touches more than the chunk's own tokens (and the open block before it).
#include "prefill_chunk.h"
#include "umma.cuh"

namespace spla {

namespace {

constexpr int kOwnThreads = 256;
constexpr int kOwnGroup = 16;              // positions whose prefix statistics are in shared memory together
constexpr int kOwnRows = 4;                // (position, head) rows a warp works on side by side
// a / n, correctly rounded, from y = 1 / n correctly rounded: one step of refinement with exact remainder (Markstein 1990; the
// quotients here are far from the ends of the exponent range).  The plain division was a third of the kernel's instructions.
__device__ __forceinline__ float2 div_by_count(float2 a, float n, float y) {
  const float2 yy = make_float2(y, y), q = __fmul2_rn(a, yy);
  return __ffma2_rn(__ffma2_rn(q, make_float2(-n, -n), a), yy, q);
}
template <int VEC> struct QueryVec { using type = uint2; };      // a lane's VEC query elements
template <> struct QueryVec<2> { using type = uint32_t; };

// One CTA per (block the chunk touches, unit).  The statistics of ALL prefixes of the block that end inside the chunk, each by
// the two exact passes and in the summation order of the append kernels (256 / D running sums of every 256 / D-th token, added
// in order), so that a position's own record has the bits a token-by-token append would have left there: with 16-bit records
// a last-bit difference would round to the other neighbour, 2^-8 away.  The block's keys are staged in shared memory; thread
// (channel pair, slot) takes every kSlots-th position of a group of kOwnGroup: running sums give the means, then one walk
// over the older tokens serves all its positions.  After every group the eight warps form the dots of those prefixes with
// their positions' queries.
// Bound by instructions issued (three quarters of the issue slots): 8192 tokens x 8 units, G = 4, 60 us (a running mean with
// reciprocals, other bits, took 51); 512 tokens x 16 units 14 us, as that did.  Without the division by refinement, row / G by
// multiplication and the packed dots it was 87 and 18 us; three CTAs an SM (80 registers, a few spilled) are no faster than two.
template <int D>
__global__ void __launch_bounds__(kOwnThreads, 2) prefill_own_kernel(const Params p, const PrefillChunk pc,
                                                                  const __nv_bfloat16* __restrict__ q, float* __restrict__ out,
                                                                  int* __restrict__ sel_user) {
  constexpr int VEC = D / 32;
  constexpr int TG = kOwnThreads / D;                          // running sums of a prefix
  constexpr int kSlots = kOwnThreads / (D / 2);
  constexpr int NP = kOwnGroup / kSlots;                       // positions of a thread
  static_assert(kSlots % TG == 0 && kOwnGroup % TG == 0, "a position's newest token is of the same sum in every group");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float inv_s[128], ln_s[128];                      // 1 / n, correctly rounded; ln(n / B)
  float* mean_s = reinterpret_cast<float*>(smem_raw);          // [kOwnGroup][D]
  float* var_s = mean_s + kOwnGroup * D;                       // [kOwnGroup][D]
  uint32_t* key_s = reinterpret_cast<uint32_t*>(var_s + kOwnGroup * D);   // [B][D / 2] channel pairs
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const PrefillUnit r = prefill_unit_of(p, pc, blockIdx.y);
  const int G = p.G;
  if (r.first < 0 && blockIdx.x == 0) {                        // positions of a refused append: empty prefix, zero output
    for (int t = 0; t < min(pc.T, -r.first); ++t) {
      for (int x = tid; x < G * D; x += kOwnThreads) out[(((size_t)r.b * pc.T + t) * p.Hq + (size_t)r.h * G) * D + x] = 0.f;
      for (int x = tid; x < p.top_k; x += kOwnThreads) {
        pc.sel[((size_t)r.u * pc.T + t) * p.top_k + x] = -1;
        if (sel_user) sel_user[(((size_t)r.b * pc.T + t) * p.Hkv + r.h) * p.top_k + x] = -1;
      }
    }
  }
  const int blk = r.L0 / p.B + blockIdx.x;
  const int t0 = blk * p.B;
  if (t0 >= r.L_end) return;                                   // CTA-uniform
  if ((p.flags & kDebugBounds) && blk >= p.max_blocks) {       // checked build
    if (tid == 0) atomicExch(p.status, kStatusBounds);
    return;
  }
  const int cnt = min(p.B, r.L_end - t0);
  const uint4* kc = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.k_cache) + ((size_t)r.u * p.max_blocks * p.B + t0) * D);
  const bool round16 = (p.flags & kStatsBf16) != 0;
  // Queries of kOwnRows (position, head) rows of the group that starts at token g0, requested before they are needed:
  // fetched one row at a time where they are used, their latency was half of this kernel's time (33 -> 15 us for 144 CTAs).
  using QV = typename QueryVec<VEC>::type;
  QV qn[kOwnRows];
  const uint32_t g_inv = 65536u / G + 1u;
  auto of_row = [&](int row) { return (int)(row * g_inv >> 16); };   // row / G: exact for G <= 16 and rows below 4096
  const __nv_bfloat16* q_unit = q + ((size_t)r.b * pc.T * p.Hq + (size_t)r.h * G) * D + lane * VEC;
  const size_t q_step = (size_t)p.Hq * D;
  auto fetch = [&](int g0, int row0, int ng) {
#pragma unroll
    for (int i = 0; i < kOwnRows; ++i) {
      const int row = row0 + i, j = of_row(row), pos = t0 + g0 + j;
      const bool ok = row < ng * G && pos >= r.L0;
      qn[i] = ok ? __ldg(reinterpret_cast<const QV*>(q_unit + (size_t)(pos - r.first) * q_step + (row - j * G) * D)) : QV();
    }
  };
  const int g_begin = max(0, r.L0 - t0) / kOwnGroup * kOwnGroup;   // the first group with a position of the chunk
  fetch(g_begin, warp * kOwnRows, min(kOwnGroup, cnt - g_begin));
  {
    uint4* dst = reinterpret_cast<uint4*>(key_s);              // rows past the end: zeros, in no prefix
#pragma unroll 4
    for (int x = tid; x < p.B * (D / 8); x += kOwnThreads) dst[x] = x < cnt * (D / 8) ? kc[x] : make_uint4(0u, 0u, 0u, 0u);
  }
  if (tid < 128) {
    inv_s[tid] = __frcp_rn((float)(tid + 1));
    ln_s[tid] = logf((float)(tid + 1) / (float)p.B);
  }
  __syncthreads();
  const int cp = tid % (D / 2), slot = tid / (D / 2);
  const uint32_t* col = key_s + cp;
  auto key2 = [&](int t) { const uint32_t w = col[t * (D / 2)]; return make_float2(bf16_lo(w), bf16_hi(w)); };
  float2 run[TG];                                              // running sums over the tokens before the group
#pragma unroll
  for (int g = 0; g < TG; ++g) run[g] = make_float2(0.f, 0.f);
  for (int g0 = 0; g0 < cnt; g0 += kOwnGroup) {
    const int ng = min(kOwnGroup, cnt - g0);
    const bool wanted = g0 >= g_begin;
    float2 nm[NP];                                             // minus the mean of each of the thread's positions
#pragma unroll
    for (int b = 0; b < NP; ++b)                               // (blocks are whole groups: the reads stay inside the block)
#pragma unroll
      for (int j = 0; j < kSlots; ++j) {
        run[j % TG] = __fadd2_rn(run[j % TG], key2(g0 + b * kSlots + j));
        if (j == slot) {
          nm[b] = run[0];
#pragma unroll
          for (int g = 1; g < TG; ++g) nm[b] = __fadd2_rn(nm[b], run[g]);
        }
      }
    if (!wanted) continue;
    float2 ss[NP][TG];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const int j = g0 + i * kSlots + slot;
      const float2 mean = div_by_count(nm[i], (float)(j + 1), inv_s[j]);
      nm[i] = make_float2(-mean.x, -mean.y);
#pragma unroll
      for (int g = 0; g < TG; ++g) ss[i][g] = make_float2(0.f, 0.f);
    }
    auto add = [&](int i, int g, float2 x) {
      const float2 dv = __fadd2_rn(x, nm[i]);
      ss[i][g] = __ffma2_rn(dv, dv, ss[i][g]);
    };
#pragma unroll 2
    for (int t = 0; t < g0; t += TG) {                         // tokens of earlier groups: in every prefix of this one
#pragma unroll
      for (int g = 0; g < TG; ++g) {
        const float2 x = key2(t + g);
#pragma unroll
        for (int i = 0; i < NP; ++i) add(i, g, x);
      }
    }
#pragma unroll
    for (int b = 0; b < NP; ++b)                               // the group's own tokens: those up to the position
#pragma unroll
      for (int j = 0; j < kSlots; ++j) {
        const float2 x = key2(g0 + b * kSlots + j);
        if (j <= slot) add(b, j % TG, x);
#pragma unroll
        for (int i = b + 1; i < NP; ++i) add(i, j % TG, x);
      }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const int j = i * kSlots + slot;
      float2 tot = ss[i][0];
#pragma unroll
      for (int g = 1; g < TG; ++g) tot = __fadd2_rn(tot, ss[i][g]);
      float2 mm = make_float2(-nm[i].x, -nm[i].y), vv = div_by_count(tot, (float)(g0 + j + 1), inv_s[g0 + j]);
      if (round16) {
        const uint32_t m16 = pack_bf16(mm.x, mm.y), v16 = pack_bf16(vv.x, vv.y);
        mm = make_float2(bf16_lo(m16), bf16_hi(m16));
        vv = make_float2(bf16_lo(v16), bf16_hi(v16));
      }
      *reinterpret_cast<float2*>(mean_s + j * D + 2 * cp) = mm;
      *reinterpret_cast<float2*>(var_s + j * D + 2 * cp) = vv;
    }
    __syncthreads();
    for (int row0 = warp * kOwnRows; row0 < ng * G; row0 += kOwnRows * (kOwnThreads / 32)) {
      float vals[2 * kOwnRows];
#pragma unroll
      for (int i = 0; i < kOwnRows; ++i) {
        const int j = min(of_row(row0 + i), ng - 1);
        float x[VEC], mv[VEC], vv[VEC];
        load_vec<VEC>(reinterpret_cast<const __nv_bfloat16*>(&qn[i]), x);
        load_vec<VEC>(mean_s + j * D + lane * VEC, mv);
        load_vec<VEC>(var_s + j * D + lane * VEC, vv);
        float2 dm = make_float2(0.f, 0.f), dv = dm;
#pragma unroll
        for (int v = 0; v < VEC; v += 2) {
          const float2 qh = __fmul2_rn(make_float2(x[v], x[v + 1]), make_float2(p.sm_scale, p.sm_scale));
          dm = __ffma2_rn(qh, make_float2(mv[v], mv[v + 1]), dm);
          dv = __ffma2_rn(__fmul2_rn(qh, qh), make_float2(vv[v], vv[v + 1]), dv);
        }
        vals[i] = dm.x + dm.y;
        vals[kOwnRows + i] = dv.x + dv.y;
      }
      fetch(g0, row0 + kOwnRows * (kOwnThreads / 32), ng);       // the next rows of this group ...
      warp_reduce_multi<2 * kOwnRows>(vals, lane);               // value lane / 4: the mean dots, then the variance dots
      float dv = __shfl_xor_sync(0xffffffffu, vals[0], 16);
      if (p.flags & 2u) dv = 0.f;
      const int row = row0 + (lane >> 2), j = of_row(row), pos = t0 + g0 + j;
      if (lane < 16 && (lane & 3) == 0 && row < ng * G && pos >= r.L0)
        pc.ell_own[((size_t)r.u * pc.T + (pos - r.first)) * G + (row - j * G)] = ln_s[g0 + j] + vals[0] + __logf(fmaf(0.5f, dv, 1.f));
    }
    if (g0 + kOwnGroup < cnt) fetch(g0 + kOwnGroup, warp * kOwnRows, min(kOwnGroup, cnt - g0 - kOwnGroup));   // ... or the first of the next
    __syncthreads();
  }
}

// What the chunk's tokens of one SB range add to the recurrent state: phi(K)^T V, [d][d] per CTA, warp-level tensor-core
// products.  phi enters as three bf16 parts (24 significant bits), V exactly; the sums are fp32 over at most 128 tokens.
// Warp w takes the rows (features) 16 (w % (D / 16)) .. + 15 and its share of the columns.
template <int D>
__global__ void __launch_bounds__(256) prefill_local_state_kernel(const Params p, const PrefillChunk pc) {
  constexpr int PAD = 8;                                       // 16-byte row offset: ldmatrix without bank conflicts
  constexpr int LD = D + PAD;
  constexpr int MT = D / 16;                                   // row tiles
  constexpr int WPM = 8 / MT;                                  // warps per row tile
  constexpr int NT = D / 8 / WPM;                              // column tiles of a warp
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __nv_bfloat16* phi = reinterpret_cast<__nv_bfloat16*>(smem_raw);    // [3][64][LD]
  __nv_bfloat16* vs = phi + 3 * 64 * LD;                              // [64][LD]
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const PrefillUnit r = prefill_unit_of(p, pc, blockIdx.y);
  const int start = prefill_range_start(pc, r, blockIdx.x);
  const int lo = max(start, r.L0), hi = min(start + pc.SB, r.L_end);  // tokens of this range
  const size_t tok0 = (size_t)r.u * p.max_blocks * p.B;
  const uint4* kc = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.k_cache) + tok0 * D);
  const uint4* vc = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.v_cache) + tok0 * D);
  const float a2 = p.phi_scale * kLog2e;
  const int mt = warp % MT, wn = warp / MT;
  const int g = lane >> 2, t = lane & 3, mi = lane >> 3, r8 = lane & 7;
  float acc[NT][4];
#pragma unroll
  for (int n = 0; n < NT; ++n) { acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f; }
  constexpr int CH = D / 8;                                    // 16-byte chunks per token
  for (int s0 = start; s0 < hi; s0 += 64) {
    if (s0 > start) __syncthreads();
    for (int idx = tid; idx < 64 * CH; idx += 256) {
      const int row = idx / CH, ch = idx % CH, pos = s0 + row;
      uint4 kk = make_uint4(0u, 0u, 0u, 0u), vv = kk;
      float nl2 = -INFINITY;
      if (pos >= lo && pos < hi) {
        kk = kc[(size_t)pos * CH + ch];
        vv = vc[(size_t)pos * CH + ch];
        nl2 = -p.tok_lse[tok0 + pos] * kLog2e;
      }
      const uint32_t w[4] = {kk.x, kk.y, kk.z, kk.w};
      uint32_t h[4], m[4], l[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float f0 = ex2(fmaf(bf16_lo(w[e]), a2, nl2)), f1 = ex2(fmaf(bf16_hi(w[e]), a2, nl2));
        h[e] = pack_bf16(f0, f1);
        const float r0 = f0 - bf16_lo(h[e]), r1 = f1 - bf16_hi(h[e]);
        m[e] = pack_bf16(r0, r1);
        l[e] = pack_bf16(r0 - bf16_lo(m[e]), r1 - bf16_hi(m[e]));
      }
      *reinterpret_cast<uint4*>(phi + (size_t)row * LD + ch * 8) = make_uint4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<uint4*>(phi + (size_t)(64 + row) * LD + ch * 8) = make_uint4(m[0], m[1], m[2], m[3]);
      *reinterpret_cast<uint4*>(phi + (size_t)(128 + row) * LD + ch * 8) = make_uint4(l[0], l[1], l[2], l[3]);
      *reinterpret_cast<uint4*>(vs + (size_t)row * LD + ch * 8) = vv;
    }
    __syncthreads();
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {                           // 16 tokens per step
      uint32_t a[3][4];
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        // A[m][k] = phi[token k][feature m]: four transposed 8x8 matrices (m 0-7, k 0-7), (m 8-15, k 0-7), (m 0-7, k 8-15), ...
        const uint32_t addr = smem_u32(phi + (size_t)(part * 64 + ks * 16 + (mi >> 1) * 8 + r8) * LD + mt * 16 + (mi & 1) * 8);
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(a[part][0]), "=r"(a[part][1]), "=r"(a[part][2]), "=r"(a[part][3]) : "r"(addr));
      }
#pragma unroll
      for (int np = 0; np < NT / 2; ++np) {
        uint32_t b[4];
        const uint32_t addr = smem_u32(vs + (size_t)(ks * 16 + (mi & 1) * 8 + r8) * LD + (wn * NT + np * 2 + (mi >> 1)) * 8);
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(addr));
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          mma_bf16(acc[2 * np], a[part][0], a[part][1], a[part][2], a[part][3], b[0], b[1]);
          mma_bf16(acc[2 * np + 1], a[part][0], a[part][1], a[part][2], a[part][3], b[2], b[3]);
        }
      }
    }
  }
  float* dst = pc.snap + ((size_t)r.u * pc.n_sb + blockIdx.x) * D * D;
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    const int col = (wn * NT + n) * 8 + 2 * t;
    *reinterpret_cast<float2*>(dst + (size_t)(mt * 16 + g) * D + col) = make_float2(acc[n][0], acc[n][1]);
    *reinterpret_cast<float2*>(dst + (size_t)(mt * 16 + g + 8) * D + col) = make_float2(acc[n][2], acc[n][3]);
  }
}

// The ranges' contributions become, in place, the state before each range; the cache's state is advanced over the chunk.
// One thread per two entries, the next eight ranges requested before this eight are written.  Bound by the memory traffic
// (64 KB read and written per range and unit at d = 128): 129 ranges x 8 units (135 MB) 19 us = 7 TB/s, partly from L2;
// with four entries a thread and nothing ahead 74 us.
template <int D>
__global__ void __launch_bounds__(128) prefill_scan_state_kernel(const Params p, const PrefillChunk pc) {
  constexpr int N2 = D * D / 2, AHEAD = 8;
  pdl_wait();
  pdl_launch_dependents();
  const int idx = blockIdx.x * 128 + threadIdx.x;
  const int u = blockIdx.y;
  float2* st = reinterpret_cast<float2*>(p.state + (size_t)u * D * D) + idx;
  float2* x = reinterpret_cast<float2*>(pc.snap + (size_t)u * pc.n_sb * D * D) + idx;
  float2 s = *st;
  float2 nx[AHEAD];
  auto fetch = [&](int i0) {
#pragma unroll
    for (int j = 0; j < AHEAD; ++j)
      if (i0 + j < pc.n_sb) nx[j] = x[(size_t)(i0 + j) * N2];
  };
  fetch(0);
  for (int i0 = 0; i0 < pc.n_sb; i0 += AHEAD) {
    float2 a[AHEAD];
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) a[j] = nx[j];
    fetch(i0 + AHEAD);
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) {
      if (i0 + j < pc.n_sb) {
        x[(size_t)(i0 + j) * N2] = s;
        s.x += a[j].x; s.y += a[j].y;
      }
    }
  }
  *st = s;
}

template <int D>
cudaError_t own_d(const Params& p, const PrefillChunk& c, const void* q, float* out, int* sel_user, cudaStream_t s) {
  const size_t smem = (size_t)2 * kOwnGroup * D * 4 + (size_t)p.B * D * 2;
  auto kern = prefill_own_kernel<D>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // (not launched ahead of the append's end like the others: its CTAs would crowd onto the SMs that are free first; 512 tokens
  // on 32768 x 2: 293 us so, 306 us launched ahead)
  return launch_ex(kern, dim3((c.T + p.B - 2) / p.B + 1, p.batch * p.Hkv), dim3(kOwnThreads), smem, s, 0, false,
                   p, c, reinterpret_cast<const __nv_bfloat16*>(q), out, sel_user);
}

template <int D>
cudaError_t state_d(const Params& p, const PrefillChunk& c, cudaStream_t s) {
  const size_t smem = (size_t)4 * 64 * (D + 8) * 2;
  auto kern = prefill_local_state_kernel<D>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = launch_ex(kern, dim3(c.n_sb, p.batch * p.Hkv), dim3(256), smem, s, 0, true, p, c);
  if (e != cudaSuccess) return e;
  return launch_ex(prefill_scan_state_kernel<D>, dim3(D * D / 2 / 128, p.batch * p.Hkv), dim3(128), 0, s, 0, true, p, c);
}

}  // namespace

cudaError_t launch_prefill_own(const Params& p, const PrefillChunk& c, const void* q, float* out, int* sel_user, cudaStream_t s) {
  return p.d == 128 ? own_d<128>(p, c, q, out, sel_user, s) : own_d<64>(p, c, q, out, sel_user, s);
}
cudaError_t launch_prefill_state(const Params& p, const PrefillChunk& c, cudaStream_t s) {
  return p.d == 128 ? state_d<128>(p, c, s) : state_d<64>(p, c, s);
}

}  // namespace spla
