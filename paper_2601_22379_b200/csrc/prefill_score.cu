// Block scores and selection of every position of a prefill chunk (Section 3.1, Eq. taylor-2nd; Section 2.2, grouped
// BlockScore; Section 2.1, Select), as a contraction instead of one pass over the statistics per position.
//
// For the complete blocks the Taylor log masses of 128 query rows (P positions x G heads) and 32 records are two
// matrix products, q . mean and (q^2) . var, on the warp-level tensor cores.  Precision is that of fp32 products: q is
// bf16 already and its square has 16 significant bits, exactly two bf16 parts; an fp32 record element enters as three
// bf16 parts (24 bits), a 16-bit one as itself; scale factors are applied to the fp32 sums.  Eight products per record
// and row with fp32 records, three with 16-bit ones.
#include "prefill_chunk.h"

namespace spla {

namespace {

constexpr int kPsThreads = 256;
constexpr int kPsRec = 32;                 // records staged together

__device__ __forceinline__ void ldm_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

// One CTA: one tile of query rows, `rec_per_cta` consecutive records.  Warp w holds rows 16 w .. 16 w + 15 as the left
// operand in registers; the records' parts are staged in shared memory once per 32 records, the next 32 already on their
// way into registers.
template <int D, bool R16>
__global__ void __launch_bounds__(kPsThreads, 2) prefill_score_kernel(const Params p, const PrefillChunk pc,
                                                                      const __nv_bfloat16* __restrict__ q, int rec_per_cta) {
  constexpr int LD = D + 8;                                    // padded row: ldmatrix without bank conflicts
  constexpr int NP = R16 ? 1 : 3;                              // parts of a record element
  constexpr int KS = D / 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __nv_bfloat16* ms = reinterpret_cast<__nv_bfloat16*>(smem_raw);   // [NP][kPsRec][LD]
  __nv_bfloat16* vs = ms + NP * kPsRec * LD;                        // [NP][kPsRec][LD]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g8 = lane >> 2, t4 = lane & 3;
  const PrefillUnit r = prefill_unit_of(p, pc, blockIdx.z);
  const int G = p.G;
  const int sb = pc.s0 + blockIdx.y / pc.nt, tile = blockIdx.y % pc.nt;
  const int sb_start = prefill_range_start(pc, r, sb);
  const int pos0 = sb_start + tile * pc.P;                     // position of row 0 (may lie before the chunk)
  const int pos_hi = min(min(pos0 + pc.P, sb_start + pc.SB), r.L_end);   // one past the last position
  if (pos_hi <= max(pos0, r.L0)) return;
  const int n_rec = (pos_hi - 1) / p.B;                        // complete blocks of the last position
  const int rec0 = blockIdx.x * rec_per_cta, rec1 = min(n_rec, rec0 + rec_per_cta);
  if (rec0 >= rec1) return;
  if ((p.flags & kDebugBounds) && rec1 > p.max_blocks) {       // checked build
    if (tid == 0) atomicExch(p.status, kStatusBounds);
    return;
  }

  // the rows this thread holds: warp * 16 + g8 and + 8
  int pos_r[2];
  bool ok_r[2];
  uint32_t qa[KS][4];
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int row = warp * 16 + g8 + 8 * hf;
    pos_r[hf] = pos0 + row / G;
    ok_r[hf] = row < pc.P * G && pos_r[hf] >= r.L0 && pos_r[hf] < pos_hi;
    const size_t off = (((size_t)r.b * pc.T + (ok_r[hf] ? pos_r[hf] - r.first : 0)) * p.Hq + (size_t)r.h * G + row % G) * D;
    const uint32_t* qr = reinterpret_cast<const uint32_t*>(q + off);
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
      qa[kk][hf] = ok_r[hf] ? __ldg(qr + 8 * kk + t4) : 0u;
      qa[kk][2 + hf] = ok_r[hf] ? __ldg(qr + 8 * kk + 4 + t4) : 0u;
    }
  }

  // staging: thread t takes 16-byte pieces t, t + 256, ... of the 32 records
  constexpr int kPieces = kPsRec * 2 * D * (R16 ? 2 : 4) / 16 / kPsThreads;    // per thread: 8 (d = 128, fp32) .. 2
  constexpr int kPerRec = 2 * D * (R16 ? 2 : 4) / 16;                           // pieces of a record
  const uint4* recs = reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(p.stats) +
                                                     (size_t)r.u * p.max_blocks * 2 * D * (R16 ? 2 : 4));
  uint4 st[kPieces];
  auto fetch = [&](int base) {
#pragma unroll
    for (int j = 0; j < kPieces; ++j) {
      const int x = j * kPsThreads + tid;
      st[j] = base + x / kPerRec < rec1 ? __ldg(recs + (size_t)base * kPerRec + x) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  fetch(rec0);
  const float ln_full = logf((float)p.B);
  const float half_s2 = (p.flags & 2u) ? 0.f : 0.5f * p.sm_scale * p.sm_scale;
  for (int base = rec0; base < rec1; base += kPsRec) {
    __syncthreads();                                           // the previous records have been read
#pragma unroll
    for (int j = 0; j < kPieces; ++j) {
      const int x = j * kPsThreads + tid, rec = x / kPerRec, pc16 = x % kPerRec;
      const bool var = pc16 >= kPerRec / 2;
      __nv_bfloat16* dst = (var ? vs : ms) + (size_t)rec * LD;
      const int piece = var ? pc16 - kPerRec / 2 : pc16;
      if constexpr (R16) {
        *reinterpret_cast<uint4*>(dst + piece * 8) = st[j];
      } else {
        const float f0 = __uint_as_float(st[j].x), f1 = __uint_as_float(st[j].y), f2 = __uint_as_float(st[j].z), f3 = __uint_as_float(st[j].w);
        const uint32_t h0 = pack_bf16(f0, f1), h1 = pack_bf16(f2, f3);
        const float a0 = f0 - bf16_lo(h0), a1 = f1 - bf16_hi(h0), a2 = f2 - bf16_lo(h1), a3 = f3 - bf16_hi(h1);
        const uint32_t m0 = pack_bf16(a0, a1), m1 = pack_bf16(a2, a3);
        const uint32_t l0 = pack_bf16(a0 - bf16_lo(m0), a1 - bf16_hi(m0)), l1 = pack_bf16(a2 - bf16_lo(m1), a3 - bf16_hi(m1));
        *reinterpret_cast<uint2*>(dst + piece * 4) = make_uint2(h0, h1);
        *reinterpret_cast<uint2*>(dst + (size_t)kPsRec * LD + piece * 4) = make_uint2(m0, m1);
        *reinterpret_cast<uint2*>(dst + (size_t)2 * kPsRec * LD + piece * 4) = make_uint2(l0, l1);
      }
    }
    __syncthreads();
    if (base + kPsRec < rec1) fetch(base + kPsRec);
    float cm[4][4], cv[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int x = 0; x < 4; ++x) { cm[n][x] = 0.f; cv[n][x] = 0.f; }
    // ldmatrix: lane addresses row (lane & 7) of matrix lane / 8: matrices (rec 0-7, k 0-7), (rec 0-7, k 8-15), (rec 8-15, ...)
    const uint32_t lane_off = (uint32_t)(((((lane >> 4) & 1) * 8 + (lane & 7)) * LD + ((lane >> 3) & 1) * 8) * 2);
    const uint32_t ms0 = smem_u32(ms) + lane_off, vs0 = smem_u32(vs) + lane_off;
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
      uint32_t qh[4], ql[4];                                   // q^2 in two bf16 parts: exact
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float a = bf16_lo(qa[kk][x]), b = bf16_hi(qa[kk][x]);
        const float a2 = a * a, b2 = b * b;
        qh[x] = pack_bf16(a2, b2);
        ql[x] = pack_bf16(a2 - bf16_lo(qh[x]), b2 - bf16_hi(qh[x]));
      }
#pragma unroll
      for (int np = 0; np < 2; ++np) {
        const uint32_t off = (uint32_t)((np * 16 * LD + kk * 16) * 2);
#pragma unroll
        for (int part = 0; part < NP; ++part) {
          uint32_t m[4], v[4];
          ldm_x4(m, ms0 + off + (uint32_t)(part * kPsRec * LD * 2));
          ldm_x4(v, vs0 + off + (uint32_t)(part * kPsRec * LD * 2));
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            mma_bf16(cm[2 * np + e], qa[kk][0], qa[kk][1], qa[kk][2], qa[kk][3], m[2 * e], m[2 * e + 1]);
            mma_bf16(cv[2 * np + e], qh[0], qh[1], qh[2], qh[3], v[2 * e], v[2 * e + 1]);
            if (part < 2) mma_bf16(cv[2 * np + e], ql[0], ql[1], ql[2], ql[3], v[2 * e], v[2 * e + 1]);
          }
        }
      }
    }
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      if (!ok_r[hf]) continue;
      const int row = warp * 16 + g8 + 8 * hf;
      const size_t slot = ((size_t)r.u * pc.ns + (sb - pc.s0)) * pc.SB + (pos_r[hf] - sb_start);
      float* dst = pc.ell + (slot * G + row % G) * pc.stride + base + 2 * t4;
#pragma unroll
      for (int n = 0; n < 4; ++n)
        *reinterpret_cast<float2*>(dst + n * 8) =
            make_float2(ln_full + cm[n][2 * hf] * p.sm_scale + __logf(1.f + half_s2 * cv[n][2 * hf]),
                        ln_full + cm[n][2 * hf + 1] * p.sm_scale + __logf(1.f + half_s2 * cv[n][2 * hf + 1]));
    }
  }
}

// Selection of one position by W warps (W = 1: one warp per position, up to 32 NK blocks; W = 8: a CTA per position, up to
// 256 NK).  Each lane keeps the keys of its NK blocks in registers.  The k-th best key is found bit by bit from the top
// (counting the keys at or above a candidate, with a stop as soon as exactly k are), which needs no scratch and no sort;
// the list then comes out in ascending order by ballots.
template <int W, int NK>
__global__ void __launch_bounds__(256, 2) prefill_select_kernel(const Params p, const PrefillChunk pc, int* __restrict__ sel_user) {
  __shared__ float red_s[8][2];
  __shared__ int cnt_s[2][8];
  constexpr int L = W * 32;                                    // lanes of a position
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const PrefillUnit r = prefill_unit_of(p, pc, blockIdx.y);
  const int G = p.G;
  const int slot = blockIdx.x * (8 / W) + (W == 1 ? warp : 0);   // position within the launch's SB ranges
  const int sb_start = prefill_range_start(pc, r, pc.s0 + slot / pc.SB);
  const int pos = sb_start + slot % pc.SB;
  if (slot >= pc.ns * pc.SB || pos < r.L0 || pos >= r.L_end) return;   // uniform over the position's warps
  const int t = pos - r.first;
  const int own = pos / p.B, nblk = own + 1;
  const int k_eff = min(p.top_k, nblk);
  const int l = W == 1 ? lane : tid;
  auto reduce = [&](float v, bool is_max) -> float {
    v = is_max ? warp_max(v) : warp_sum(v);
    if constexpr (W > 1) {
      __syncthreads();
      if (lane == 0) red_s[warp][0] = v;
      __syncthreads();
      float x = red_s[0][0];
#pragma unroll
      for (int w = 1; w < W; ++w) x = is_max ? fmaxf(x, red_s[w][0]) : x + red_s[w][0];
      v = x;
    }
    return v;
  };
  int phase = 0;
  auto count = [&](int c) -> int {
    c = __reduce_add_sync(0xffffffffu, c);
    if constexpr (W > 1) {                                     // (two buffers in turn: one barrier per count)
      if (lane == 0) cnt_s[phase][warp] = c;
      __syncthreads();
      int x = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) x += cnt_s[phase][w];
      c = x;
      phase ^= 1;
    }
    return c;
  };

  // aggregated score of the lane's blocks: per head softmax over the position's blocks, summed over the group
  float sc[NK];
#pragma unroll
  for (int k = 0; k < NK; ++k) sc[k] = 0.f;
  const float* ell = pc.ell + (((size_t)r.u * pc.ns * pc.SB + slot) * G) * pc.stride;
  for (int g = 0; g < G; ++g) {
    const float e_own = pc.ell_own[((size_t)r.u * pc.T + t) * G + g];
    float e[NK], mx = -INFINITY;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const int i = k * L + l;
      e[k] = i < own ? ell[(size_t)g * pc.stride + i] : (i == own ? e_own : -INFINITY);
      mx = fmaxf(mx, e[k]);
    }
    mx = reduce(mx, true);
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < NK; ++k) { e[k] = __expf(e[k] - mx); sum += e[k]; }
    const float inv = 1.f / reduce(sum, false);
#pragma unroll
    for (int k = 0; k < NK; ++k) sc[k] = fmaf(e[k], inv, sc[k]);
  }
  // keys: 0 for blocks that do not exist, all ones for the forced ones, else the score's bits + 1 (positive floats order
  // like integers)
  uint32_t key[NK];
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    const int i = k * L + l;
    key[k] = i >= nblk ? 0u : (i < p.n_sink || i >= nblk - p.n_local) ? 0xffffffffu : __float_as_uint(sc[k]) + 1u;
  }
  uint32_t thr = 1u;
  int n_eq = k_eff;                                            // of the keys equal to thr, the first n_eq are taken
  if (k_eff < nblk) {
    thr = 0u;
    bool exact = false;
    for (int bit = 30; bit >= 0; --bit) {
      const uint32_t cand = thr | (1u << bit);
      int c = 0;
#pragma unroll
      for (int k = 0; k < NK; ++k) c += key[k] >= cand;
      c = count(c);
      if (c >= k_eff) {
        thr = cand;
        if (c == k_eff) { exact = true; break; }
      }
    }
    if (!exact) {
      int c = 0;
#pragma unroll
      for (int k = 0; k < NK; ++k) c += key[k] > thr;
      n_eq = k_eff - count(c);
    }
  }
  // ascending list: position = number of taken blocks with a smaller index (blocks are dealt to lanes in index order)
  int* sel_w = pc.sel + ((size_t)r.u * pc.T + t) * p.top_k;
  int* sel_o = sel_user ? sel_user + (((size_t)r.b * pc.T + t) * p.Hkv + r.h) * p.top_k : nullptr;
  int base = 0, eq_base = 0;
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    if (k * L >= nblk) break;                                  // uniform
    const bool eq = key[k] == thr;
    const uint32_t eq_mask = __ballot_sync(0xffffffffu, eq);
    int eq_before = eq_base + __popc(eq_mask & below), eq_all = __popc(eq_mask);
    if constexpr (W > 1) {
      if (lane == 0) cnt_s[phase][warp] = eq_all;
      __syncthreads();
      eq_all = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) { if (w < warp) eq_before += cnt_s[phase][w]; eq_all += cnt_s[phase][w]; }
      phase ^= 1;
    }
    const bool take = key[k] > thr || (eq && eq_before < n_eq);
    const uint32_t mask = __ballot_sync(0xffffffffu, take);
    int before = base + __popc(mask & below), all = __popc(mask);
    if constexpr (W > 1) {
      if (lane == 0) cnt_s[phase][warp] = all;
      __syncthreads();
      all = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) { if (w < warp) before += cnt_s[phase][w]; all += cnt_s[phase][w]; }
      phase ^= 1;
    }
    if (take) {
      const int i = k * L + l;
      sel_w[before] = i;
      if (sel_o) sel_o[before] = i;
    }
    base += all;
    eq_base += eq_all;
  }
  for (int s = k_eff + l; s < p.top_k; s += L) {
    sel_w[s] = -1;
    if (sel_o) sel_o[s] = -1;
  }
}

template <int D, bool R16>
cudaError_t score_d(const Params& p, const PrefillChunk& c, const void* q, int max_blocks_seen, int sm_count, cudaStream_t s) {
  const size_t smem = (size_t)2 * (R16 ? 1 : 3) * kPsRec * (D + 8) * 2;
  auto kern = prefill_score_kernel<D, R16>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // records per CTA: as many as leave about two waves of CTAs, at least 64 (the query rows are loaded once per CTA)
  const int U = p.batch * p.Hkv;
  const long long tiles = (long long)c.ns * c.nt * U;
  int rec = 64;
  while (rec < 1024 && tiles * ((max_blocks_seen + rec - 1) / rec) > 4LL * sm_count) rec *= 2;
  const int ny = (max_blocks_seen + rec - 1) / rec;
  kern<<<dim3(ny < 1 ? 1 : ny, c.ns * c.nt, U), kPsThreads, smem, s>>>(p, c, reinterpret_cast<const __nv_bfloat16*>(q), rec);
  ++g_launch_count;
  return cudaGetLastError();
}

template <int W, int NK>
cudaError_t select_w(const Params& p, const PrefillChunk& c, int* sel_user, cudaStream_t s) {
  const int slots = c.ns * c.SB;
  prefill_select_kernel<W, NK><<<dim3((slots + 8 / W - 1) / (8 / W), p.batch * p.Hkv), 256, 0, s>>>(p, c, sel_user);
  ++g_launch_count;
  return cudaGetLastError();
}

}  // namespace

// Log masses of the complete blocks, for the positions of SB ranges c.s0 .. c.s0 + c.ns - 1.  max_blocks_seen: blocks of the
// longest sequence after the chunk.
cudaError_t launch_prefill_score(const Params& p, const PrefillChunk& c, const void* q, int max_blocks_seen, int sm_count, cudaStream_t s) {
  if (p.flags & kStatsBf16)
    return p.d == 128 ? score_d<128, true>(p, c, q, max_blocks_seen, sm_count, s) : score_d<64, true>(p, c, q, max_blocks_seen, sm_count, s);
  return p.d == 128 ? score_d<128, false>(p, c, q, max_blocks_seen, sm_count, s) : score_d<64, false>(p, c, q, max_blocks_seen, sm_count, s);
}

// Selection for the same positions.  Up to 1024 blocks a warp holds a position's keys; above, a CTA does (513 blocks, 512 positions x 16
// units: 121 us by CTAs, whose barriers cost more than the wider registers of one warp, 55 us by warps).
cudaError_t launch_prefill_select(const Params& p, const PrefillChunk& c, int max_blocks_seen, int* sel_user, cudaStream_t s) {
  if (max_blocks_seen <= 32 * 2) return select_w<1, 2>(p, c, sel_user, s);
  if (max_blocks_seen <= 32 * 4) return select_w<1, 4>(p, c, sel_user, s);
  if (max_blocks_seen <= 32 * 8) return select_w<1, 8>(p, c, sel_user, s);
  if (max_blocks_seen <= 32 * 16) return select_w<1, 16>(p, c, sel_user, s);
  if (max_blocks_seen <= 32 * 32) return select_w<1, 32>(p, c, sel_user, s);
  if (max_blocks_seen <= 256 * 16) return select_w<8, 16>(p, c, sel_user, s);
  return select_w<8, 64>(p, c, sel_user, s);
}

}  // namespace spla
