// Attention of a prefill chunk on the 5th-generation tensor cores: exact softmax attention over every position's selected
// blocks (Section 2.2 of the paper, Eq. gqa-sparse), the residual linear branch (Section 3.2, Eq. rla-impl-1..3) and the
// RMSNorm merge (Section 3.3), one kernel.
//
// A CTA takes one tile of 128 query rows (P neighbouring positions x the G heads of one KV head) and walks the UNION of
// the blocks those positions selected, 64 tokens at a time; a row that did not select a block is masked out there.
// Neighbouring positions select much the same blocks, and a 128-row product costs what eight 16-row ones would; K and V
// come from L2 once per tile of positions instead of once per position.
//
// The linear branch is computed as a difference of sums over tokens rather than as o_bar - o_tilde: with S_base the state
// before the tile's SB range (its first token: base),
//     o_rla = phi(q) S_base - sum over selected tokens t < base  of (phi(q).phi(k_t)) v_t
//                           + sum over unselected tokens t >= base of (phi(q).phi(k_t)) v_t,
// which equals o_bar - o_tilde and leaves out what cancels between the two (the local blocks).
//
// Per 64-token tile and 128 rows, all with fp32 accumulators in tensor memory:
//     S  = Q K^T                     bf16, exact products
//     A  = phi(Q) phi(K)^T           fp16 head + remainder on both sides (scaled by 2^14): 22 significant bits, 3 products
//     O += P V,  R += C V            P and the signed coefficients C in two bf16 parts each (17 bits), from tensor memory
// The softmax keeps a stale row maximum and rescales O only when the maximum grows by more than 2^8, which is rare after
// the first tiles.  The tensor core truncates when it adds into an accumulator, so the residual, which later subtracts
// large parts of itself, is drained into fp32 registers every kFlush tiles (the drain hides behind the next tile's
// first products).
//
// 16 warps: TMA for K (warp 0) and for V (warp 2), the MMA issuer (warp 1); softmax (4 warps, one row per thread); linear
// coefficients, drain and epilogue (4 warps); phi(K) (4 warps).  Two-deep rings everywhere, released as early as each
// operand allows.  setmaxnreg moves registers to the linear warps, whose row of R takes 128.
//
// The tensor pipe needs about 2560 cycles per tile (8 products of 128 x 64 x 128; the four whose left operand comes from
// shared memory run at 3/4 of the rate).  What bounds the kernel above that is issuing: four roles with different code share
// each scheduler, so code size counts (with every loop unrolled 43 % of all stalls were instruction fetches, 9000 cycles per
// tile; with 16-token loop bodies 3600), and the MMA warp runs converged with one elected lane (a one-lane branch cost 75 to
// 110 cycles per MMA instead of 50 to 65).  A prompt of 8192 tokens (8 KV heads, G = 4, d = 128, 32 of up to 128 blocks of
// 64): 60.6 ms as one virtual unit per position on the general kernels, 2.87 ms with this kernel unrolled, 1.62 ms now, of
// which it takes 1.27 ms.
//
// Every wait is an mbarrier poll with an iteration limit; on expiry the CTA raises its abort flag, all roles leave their
// loops, tensor memory is released and the time-out status is latched.  No multicast anywhere.
#include <cuda_fp16.h>

#include "prefill_chunk.h"
#include "umma.cuh"

namespace spla {

namespace {

constexpr int kPaThreads = 512;
constexpr int kPaTile = 64;                        // tokens per tile
constexpr int kFlush = 4;                          // tiles accumulated into R before it is drained
constexpr int kPhiExp = 14;                        // phi is scaled by 2^14 (at most 2^14 then, well inside fp16)
constexpr uint32_t kPaTmemCols = 512;

template <int D>
struct PaSmem {
  static constexpr int H = D / 64;                               // arrays of 128-byte rows per operand
  static constexpr int kQ = 0;                                   // [H][128 rows][128 B]  q
  static constexpr int kQBytes = H * kPfRows * 128;
  static constexpr int kFh = kQ + kQBytes;                       // phi(q), head
  static constexpr int kFl = kFh + kQBytes;                      // phi(q), remainder
  static constexpr int kTileBytes = H * kPaTile * 128;
  static constexpr int kHalf = kPaTile * 128;                    // one array of a K or V tile
  static constexpr int kK = kFl + kQBytes;                       // [2] K tiles
  static constexpr int kV = kK + 2 * kTileBytes;                 // [2] V tiles
  static constexpr int kPhi = kV + 2 * kTileBytes;               // [2] phi(K) tiles: head, remainder (first: S_base in fp16 parts)
  static constexpr int kBitmap = kPhi + 4 * kTileBytes;          // [512] words: the union of the selected blocks
  static constexpr int kLse = kBitmap + kPfMaxBlocks / 8;        // float [2][64]
  static constexpr int kBars = kLse + 2 * kPaTile * 4;
  static constexpr int kMisc = kBars + 23 * 8;                   // tensor-memory base, abort flag, tile count
  static constexpr int kBytes = kMisc + 32;
  static_assert(kBytes <= 227 * 1024, "shared memory of the attend kernel");
  static_assert(2 * H * D * 128 <= 4 * kTileBytes, "S_base fits the phi(K) ring");
};

__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
  const __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float h2_lo(uint32_t x) { return __low2float(*reinterpret_cast<const __half2*>(&x)); }
__device__ __forceinline__ float h2_hi(uint32_t x) { return __high2float(*reinterpret_cast<const __half2*>(&x)); }
__device__ __forceinline__ uint64_t low_bits(int n) { return n >= 64 ? ~0ull : (n <= 0 ? 0ull : (1ull << n) - 1ull); }

// Walks the tiles of 64 tokens over the set bits of the bitmap.  Blocks of 64 tokens or more: one block, token offset
// `off` inside it; smaller ones: 64 / B consecutive set bits together (blk[s] < 0: none left).
struct TileWalk {
  const uint32_t* bm;
  int w, w_end, B;
  uint32_t word;
  int blk[4], off;
  __device__ __forceinline__ void start(const uint32_t* bitmap, int B_, int last_blk) {
    bm = bitmap;
    w = 0;
    w_end = (last_blk >> 5) + 1;
    B = B_;
    word = bm[0];
    off = B_;
    blk[0] = -1;
  }
  // Block number s of a tile of small blocks (of a short last tile: the first again).  A select, so that blk[] stays in registers.
  __device__ __forceinline__ int sub_block(int s) const {
    int r = blk[0];
#pragma unroll
    for (int x = 1; x < 4; ++x) r = s == x ? blk[x] : r;
    return r < 0 ? blk[0] : r;
  }
  __device__ __forceinline__ int next_bit() {
    while (word == 0u) {
      if (++w >= w_end) { w = w_end; return -1; }                 // (a tile of small blocks may run past the last one)
      word = bm[w];
    }
    const int i = w * 32 + __ffs(word) - 1;
    word &= word - 1u;
    return i;
  }
  __device__ __forceinline__ void next() {
    if (B >= kPaTile) {
      off += kPaTile;
      if (off >= B) { blk[0] = next_bit(); off = 0; }
    } else {
      off = 0;
#pragma unroll
      for (int s = 0; s < 4; ++s) blk[s] = s * B < kPaTile ? next_bit() : -1;
    }
  }
};

// A position's ascending selection list, followed along the walk; the entry after the current one is already loaded.
struct SelCursor {
  const int* list;
  int left, cur, nxt;
  __device__ __forceinline__ void start(const int* l, int top_k) {
    list = l;
    left = l ? top_k : 0;
    cur = left > 0 ? l[0] : -1;
    nxt = left > 1 ? l[1] : -1;
  }
  __device__ __forceinline__ bool at(int blk) const { return cur == blk; }
  __device__ __forceinline__ void pass() {
    cur = nxt;
    --left;
    ++list;
    nxt = left > 1 ? list[1] : -1;
  }
};

// The tokens of the current tile that row `pos` attends to (bit j: token j of the tile), and those after `base` it leaves
// out (the two halves of the linear branch).  Moves the cursor.
__device__ __forceinline__ void tile_masks(const TileWalk& tw, SelCursor& sc, int pos, int base, uint64_t& sel, uint64_t& neg, uint64_t& posv) {
  sel = neg = posv = 0ull;
  if (tw.B >= kPaTile) {
    const int tok0 = tw.blk[0] * tw.B + tw.off;
    const bool s = sc.at(tw.blk[0]);                             // (never for a row without a position: its list is empty)
    if (s && tw.off + kPaTile >= tw.B) sc.pass();
    if (tok0 + kPaTile <= base) {                                // (uniform: wholly before the tile's positions)
      sel = neg = s ? ~0ull : 0ull;
      return;
    }
    if (pos < 0) return;
    const uint64_t seen = low_bits(pos + 1 - tok0), old = low_bits(base - tok0);
    if (s) { sel = seen; neg = seen & old; } else { posv = seen & ~old; }
  } else {
    if (pos < 0) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (q * tw.B >= kPaTile || tw.blk[q] < 0) continue;
      const int tok0 = tw.blk[q] * tw.B;
      const bool s = sc.at(tw.blk[q]);
      if (s) sc.pass();
      const uint64_t seen = low_bits(min(tw.B, pos + 1 - tok0)), old = low_bits(min(tw.B, base - tok0));
      if (s) { sel |= seen << (q * tw.B); neg |= (seen & old) << (q * tw.B); } else { posv |= (seen & ~old) << (q * tw.B); }
    }
  }
}

// Whether the tile holds rows past the sequence's end (the open block; of a short last tile the repeated first block).
__device__ __forceinline__ bool tile_past(const TileWalk& tw, int L_end) {
  if (tw.B >= kPaTile) return tw.blk[0] * tw.B + tw.off + kPaTile > L_end;
  bool past = false;
#pragma unroll
  for (int s = 0; s < 4; ++s)
    if (s * tw.B < kPaTile) past |= ((tw.blk[s] < 0 ? tw.blk[0] : tw.blk[s]) + 1) * tw.B > L_end;
  return past;
}

// A product with a value that is not finite is not finite, even with a probability of 0; a position must not see that of a token
// it does not attend to (a later one, or one of a block it did not select), which shares its tile.  So such values leave the
// tile, and the positions that do attend to them are marked.  (With the residual they are in S_bar and reach every later
// position anyway.)  One maximum per pair of values finds them: 8192 tokens 1144 -> 1161 us without the residual (looking at
// every value by itself 1268).
__device__ __forceinline__ uint32_t not_finite2(uint32_t w) { return ((w & 0x7f807f80u) + 0x00800080u) & 0x80008000u; }   // bits 15, 31
template <int D>
__device__ __forceinline__ void take_out_not_finite(uint4* vp, int tok, int blk, int ch, const int* sel_unit, int first, int top_k, int pos0,
                                                    int pos_lo, int pos_hi, uint32_t* marks) {
  uint32_t w[4] = {vp->x, vp->y, vp->z, vp->w}, bits = 0u;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const uint32_t bad = not_finite2(w[e]);
    if (bad & 0x8000u) { bits |= 1u << (2 * e); w[e] &= 0xffff0000u; }
    if (bad & 0x80000000u) { bits |= 2u << (2 * e); w[e] &= 0x0000ffffu; }
  }
  *vp = make_uint4(w[0], w[1], w[2], w[3]);
#pragma unroll 1
  for (int pos = max(pos_lo, tok); pos < pos_hi; ++pos) {
    const int* list = sel_unit + (size_t)(pos - first) * top_k;
    bool has = false;
#pragma unroll 1
    for (int x = 0; x < top_k; ++x) has |= list[x] == blk;
    if (has) atomicOr(marks + (pos - pos0) * (D / 32) + ch / 4, bits << (ch % 4 * 8));
  }
}

template <int D, bool RLA>
__global__ void __launch_bounds__(kPaThreads, 1)
    prefill_attend_kernel(const Params p, const PrefillChunk pc, const __grid_constant__ CUtensorMap map_k,
                          const __grid_constant__ CUtensorMap map_v, const __nv_bfloat16* __restrict__ q,
                          const float* __restrict__ rms_weight, float* __restrict__ out) {
  using SM = PaSmem<D>;
  constexpr int H = SM::H, KS = D / 16;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::kBars);
  uint64_t *k_full = bars, *k_empty = bars + 2, *v_full = bars + 4, *v_empty = bars + 6, *phi_ready = bars + 8, *phi_empty = bars + 10,
           *s_full = bars + 12, *a_full = bars + 14, *p_ready = bars + 16, *c_ready = bars + 18, *r_full = bars + 20, *r_empty = bars + 21,
           *done = bars + 22;
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(smem + SM::kMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SM::kMisc + 4);
  int* n_set_s = reinterpret_cast<int*>(smem + SM::kMisc + 8);
  uint32_t* bitmap = reinterpret_cast<uint32_t*>(smem + SM::kBitmap);
  float* lse_s = reinterpret_cast<float*>(smem + SM::kLse);
  float* l_s = reinterpret_cast<float*>(smem + SM::kQ);           // (the queries are dead by then)
  uint32_t* marks = reinterpret_cast<uint32_t*>(smem + SM::kFh);  // without the residual: [position][D / 32] bits, see take_out_not_finite

  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wg = warp >> 2;
  const int G = p.G, B = p.B;
  const PrefillUnit r = prefill_unit_of(p, pc, pc.u0 + blockIdx.y);
  // the last positions of a chunk see most: their tiles start first
  const int tq = pc.q0 + pc.nq - 1 - (int)blockIdx.x, sb = tq / pc.nt, tile = tq % pc.nt;
  const int sb_start = prefill_range_start(pc, r, sb);
  const int pos0 = sb_start + tile * pc.P;
  const int pos_lo = max(pos0, r.L0), pos_hi = min(min(pos0 + pc.P, sb_start + pc.SB), r.L_end);
  if (pos_lo >= pos_hi) return;                                   // CTA-uniform
  const int base = max(sb_start, r.L0);
  const size_t unit_row0 = (size_t)r.u * p.max_blocks * B;

  // ---------------------------------------------------------------- prologue (all threads) ------------------------
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&k_full[s], 1);  mbar_init(&k_empty[s], 5);   // four transform warps and the MMA
      mbar_init(&v_full[s], 1);  mbar_init(&v_empty[s], 1);
      mbar_init(&phi_ready[s], 4);  mbar_init(&phi_empty[s], 1);
      mbar_init(&s_full[s], 1);  mbar_init(&a_full[s], 1);
      mbar_init(&p_ready[s], 4);  mbar_init(&c_ready[s], 4);
    }
    mbar_init(r_full, 1);
    mbar_init(r_empty, 4);
    mbar_init(done, 1);
    mbar_init_done();
    *abort_flag = 0;
    *n_set_s = 0;
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
  }
  if (warp == 1) tmem_alloc(tmem_base_s, kPaTmemCols);
  if constexpr (!RLA)
    for (int x = tid; x < kPfRows * (D / 32); x += kPaThreads) marks[x] = 0u;
  bitmap[tid] = 0u;                                               // kPfMaxBlocks / 32 == kPaThreads words
  static_assert(kPfMaxBlocks / 32 == kPaThreads, "one bitmap word per thread");
  float4 sv[D * D / 4 / kPaThreads];
  float smax = 0.f;
  if constexpr (RLA) {                                            // S_base: entry 4 (j * 512 + tid) .. + 3
    const float4* S = reinterpret_cast<const float4*>(pc.snap + ((size_t)r.u * pc.n_sb + sb) * D * D);
#pragma unroll
    for (int j = 0; j < D * D / 4 / kPaThreads; ++j) sv[j] = __ldg(S + j * kPaThreads + tid);
  }
  {                                                               // q and phi(q): four threads per row
    constexpr int NCH = D / 32;                                   // 16-byte pieces per thread
    const int row = tid >> 2, part = tid & 3;
    const int pos = pos0 + row / G;
    const bool ok = row < pc.P * G && pos >= pos_lo && pos < pos_hi;
    const uint4* qr = reinterpret_cast<const uint4*>(
        q + (((size_t)r.b * pc.T + (ok ? pos - r.first : 0)) * p.Hq + (size_t)r.h * G + row % G) * D) + part * NCH;
    uint4 raw[NCH];
#pragma unroll
    for (int j = 0; j < NCH; ++j) raw[j] = ok ? __ldg(qr + j) : make_uint4(0u, 0u, 0u, 0u);
    float f[NCH * 8], mx = -INFINITY, sum = 0.f;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      const uint32_t w[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) { f[j * 8 + 2 * e] = bf16_lo(w[e]); f[j * 8 + 2 * e + 1] = bf16_hi(w[e]); }
    }
    const float a2 = p.phi_scale * kLog2e;
#pragma unroll
    for (int x = 0; x < NCH * 8; ++x) mx = fmaxf(mx, f[x]);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
#pragma unroll
    for (int x = 0; x < NCH * 8; ++x) { f[x] = exp2f((f[x] - mx) * a2); sum += f[x]; }
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    const float inv = ok ? (float)(1 << kPhiExp) / sum : 0.f;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      uint32_t h[4], l[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float f0 = f[j * 8 + 2 * e] * inv, f1 = f[j * 8 + 2 * e + 1] * inv;
        h[e] = pack_h2(f0, f1);
        l[e] = pack_h2(f0 - h2_lo(h[e]), f1 - h2_hi(h[e]));
      }
      const int ch = part * NCH + j;                              // 16-byte piece of the row
      const int off = (ch >> 3) * (kPfRows * 128) + row * 128 + (((ch & 7) ^ (row & 7)) << 4);
      *reinterpret_cast<uint4*>(smem + SM::kQ + off) = raw[j];
      if constexpr (RLA) {
        *reinterpret_cast<uint4*>(smem + SM::kFh + off) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(smem + SM::kFl + off) = make_uint4(l[0], l[1], l[2], l[3]);
      }
    }
  }
  if constexpr (RLA) {
#pragma unroll
    for (int j = 0; j < D * D / 4 / kPaThreads; ++j)
      smax = fmaxf(smax, fmaxf(fmaxf(fabsf(sv[j].x), fabsf(sv[j].y)), fmaxf(fabsf(sv[j].z), fabsf(sv[j].w))));
    smax = warp_max(smax);
    if (lane == 0) lse_s[warp] = smax;
  }
  __syncthreads();                                                // bitmap cleared; the warps' maxima
  // union of the selections, and (residual) every block of the SB range up to the last own one
  const int own_hi = (pos_hi - 1) / B;
  {
    const int* sel = pc.sel + ((size_t)r.u * pc.T + (pos_lo - r.first)) * p.top_k;
    for (int x = tid; x < (pos_hi - pos_lo) * p.top_k; x += kPaThreads) {
      const int blk = sel[x];
      if (blk >= 0 && blk <= own_hi) atomicOr(&bitmap[blk >> 5], 1u << (blk & 31));
      else if (blk > own_hi) atomicExch(p.status, kStatusBounds);
    }
    if (RLA)
      for (int blk = sb_start / B + tid; blk <= own_hi; blk += kPaThreads) atomicOr(&bitmap[blk >> 5], 1u << (blk & 31));
  }
  int s_exp = 0;                                                  // S_base is scaled by 2^s_exp into fp16's range
  if constexpr (RLA) {
    float m = 0.f;
#pragma unroll
    for (int w = 0; w < kPaThreads / 32; ++w) m = fmaxf(m, lse_s[w]);
    if (m > 0.f) s_exp = min(60, max(-60, 13 - (int)(((__float_as_uint(m) >> 23) & 255u) - 127u)));
    const float sc = exp2f((float)s_exp);
#pragma unroll
    for (int j = 0; j < D * D / 4 / kPaThreads; ++j) {
      const int e = (j * kPaThreads + tid) * 4, row = e / D, col = e % D;
      const float f0 = sv[j].x * sc, f1 = sv[j].y * sc, f2 = sv[j].z * sc, f3 = sv[j].w * sc;
      const uint32_t h0 = pack_h2(f0, f1), h1 = pack_h2(f2, f3);
      const uint32_t l0 = pack_h2(f0 - h2_lo(h0), f1 - h2_hi(h0)), l1 = pack_h2(f2 - h2_lo(h1), f3 - h2_hi(h1));
      const int off = (col >> 6) * (D * 128) + row * 128 + ((((col & 63) >> 3) ^ (row & 7)) << 4) + (col & 7) * 2;
      *reinterpret_cast<uint2*>(smem + SM::kPhi + off) = make_uint2(h0, h1);
      *reinterpret_cast<uint2*>(smem + SM::kPhi + H * D * 128 + off) = make_uint2(l0, l1);
    }
  }
  proxy_fence();                                                  // operands written above -> visible to the tensor core
  tc_fence_before();
  __syncthreads();                                                // (bitmap complete)
  tc_fence_after();
  {
    const int c = __reduce_add_sync(0xffffffffu, __popc(bitmap[tid]));
    if (lane == 0 && c) atomicAdd(n_set_s, c);
  }
  __syncthreads();
  const uint32_t tmem = *tmem_base_s;
  const int n_set = *n_set_s;
  const int n_tiles = B >= kPaTile ? n_set * (B / kPaTile) : (n_set * B + kPaTile - 1) / kPaTile;
  const uint32_t tO = tmem, tR = tmem + D, tSA = tmem + 256;      // S, A of buffer b: tSA + 128 b, + 64
  const uint32_t sbase = smem_u32(smem);
  const int lim = p.wait_limit;

  if (wg == 0) {
    warpgroup_reg_dec<56>();
    if ((warp == 0 || warp == 2) && lane == 0) {
      // ------------------------------------------------------------ TMA: K and the tokens' log-sum-exp, or V -----------
      const bool is_k = warp == 0;
      const int nsub = B < kPaTile ? kPaTile / B : 1, rows = B < kPaTile ? B : kPaTile;
      uint64_t *full = is_k ? k_full : v_full, *empty = is_k ? k_empty : v_empty;
      const CUtensorMap* map = is_k ? &map_k : &map_v;
      TileWalk tw;
      tw.start(bitmap, B, own_hi);
      int issued = 0;
      for (int i = 0; i < n_tiles && !*abort_flag; ++i) {
        tw.next();
        const int b = i & 1;
        if (i >= 2 && !mbar_wait(&empty[b], ((i >> 1) - 1) & 1, lim)) { *abort_flag = 1; break; }
        mbar_expect_tx(&full[b], SM::kTileBytes + (is_k ? kPaTile * 4 : 0) + (uint32_t)p.dbg_tx_extra);
        const uint32_t dst = sbase + (is_k ? SM::kK : SM::kV) + b * SM::kTileBytes;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (s >= nsub) break;
          int blk = tw.blk[s] < 0 ? tw.blk[0] : tw.blk[s];         // (a short last tile: any valid rows, masked out)
          if ((p.flags & kDebugBounds) && blk >= p.max_blocks) { atomicExch(p.status, kStatusBounds); blk = 0; }   // checked build
          const size_t row = unit_row0 + (size_t)blk * B + tw.off;
#pragma unroll
          for (int hh = 0; hh < H; ++hh) tma_load_box(dst + hh * SM::kHalf + s * rows * 128, map, hh * 64, (int)row, &full[b]);
          if (is_k) bulk_g2s(lse_s + b * kPaTile + s * rows, p.tok_lse + row, (uint32_t)(rows * 4), &full[b]);
        }
        issued = i + 1;
      }
      // every copy has landed before the CTA leaves, whatever the other roles do
      for (int j = max(0, issued - 2); j < issued; ++j) mbar_wait(&full[j & 1], (j >> 1) & 1, lim);
    } else if (warp == 1) {
      // ------------------------------------------------------------ MMA issuer -------------------------------------
      constexpr uint32_t id_s = umma_idesc(true, false, false, kPfRows, kPaTile);
      constexpr uint32_t id_a = umma_idesc(false, false, false, kPfRows, kPaTile);
      constexpr uint32_t id_o = umma_idesc(true, false, true, kPfRows, D);
      constexpr uint32_t id_r0 = umma_idesc(false, false, true, kPfRows, D);
      const uint32_t one = elect_one();                           // (the whole warp runs this loop: see umma_ss_one)
      bool ok = true;
      // The loops are rolled as far as they can be (four products per trip): the roles of a CTA run on the same schedulers
      // and their code competes for the instruction cache.
      const uint32_t q0 = umma_desc_lo(sbase + SM::kQ, 16), fh0 = umma_desc_lo(sbase + SM::kFh, 16), fl0 = umma_desc_lo(sbase + SM::kFl, 16);
      constexpr uint32_t kQStep = kPfRows * 128 / 16, kKStep = SM::kHalf / 16;   // to the next 64 channels of q, of a K tile
      // D (+)= X Y^T over all channels: both K-major, 16 channels = 32 bytes per step, 64 per array of rows
      auto xyT = [&](uint32_t d, uint32_t x, uint32_t y, uint32_t idesc, uint32_t acc) {
#pragma unroll
        for (int hh = 0; hh < H; ++hh) umma_ss4_one<2, 2>(one, d, x + hh * kQStep, y + hh * kKStep, idesc, hh > 0 ? 1u : acc);
      };
      // D (+)= C V for the two parts of C, 16 tokens per step
      auto cv = [&](uint32_t d, uint32_t c, uint32_t v, uint32_t acc) {
#pragma unroll
        for (int part = 0; part < 2; ++part) umma_ts4_one<16, 2048 / 16>(one, d, c + part * 8, v, id_o, part > 0 ? 1u : acc);
      };
      auto first_products = [&](int i) {                          // S and A of tile i
        const int b = i & 1, par = (i >> 1) & 1;
        const uint32_t d = tSA + b * 128;
        if (!warp_waits(&k_full[b], par, lim)) { ok = false; return; }
        tc_fence_after();
        xyT(d, q0, umma_desc_lo(sbase + SM::kK + b * SM::kTileBytes, 16), id_s, 0u);
        umma_commit_one(one, &k_empty[b]);
        umma_commit_one(one, &s_full[b]);
        if constexpr (RLA) {
          if (!warp_waits(&phi_ready[b], par, lim)) { ok = false; return; }
          tc_fence_after();
          const uint32_t ph = umma_desc_lo(sbase + SM::kPhi + b * 2 * SM::kTileBytes, 16);
#pragma unroll 1
          for (int part = 0; part < 3; ++part)                    // head x head, remainder x head, head x remainder
            xyT(d + 64, part == 1 ? fl0 : fh0, part == 2 ? ph + SM::kTileBytes / 16 : ph, id_a, part > 0);
          umma_commit_one(one, &phi_empty[b]);
          umma_commit_one(one, &a_full[b]);
        }
      };
      if constexpr (RLA) {                                        // R = phi(q) S_base
#pragma unroll 1
        for (int part = 0; part < 3; ++part) {
          const uint32_t x = part == 1 ? fl0 : fh0, y = umma_desc_lo(sbase + SM::kPhi + (part == 2 ? H * D * 128 : 0), D * 128);
#pragma unroll 1
          for (int kk = 0; kk < KS; ++kk)
            umma_ss_one(one, tR, umma_desc_of(x + (kk >> 2) * kQStep + (kk & 3) * 2), umma_desc_of(y + kk * (2048 / 16)), id_r0, part > 0 || kk > 0);
        }
        umma_commit_one(one, &phi_empty[0]);
        umma_commit_one(one, &phi_empty[1]);
      }
#pragma unroll 1
      for (int i = -1; i < n_tiles && ok && !warp_aborted(abort_flag); ++i) {
        if (i + 1 < n_tiles) first_products(i + 1);
        if (!ok) break;
        if (i < 0) continue;
        const int b = i & 1, par = (i >> 1) & 1;
        if (!warp_waits(&p_ready[b], par, lim) || !warp_waits(&v_full[b], par, lim)) { ok = false; break; }
        if (!RLA && !warp_waits(&phi_ready[b], par, lim)) { ok = false; break; }   // (the values have been looked over)
        tc_fence_after();
        const uint32_t a = tSA + b * 128, v = umma_desc_lo(sbase + SM::kV + b * SM::kTileBytes, SM::kHalf);
        cv(tO, a, v, i > 0);
        if constexpr (RLA) {
          const bool fresh = i > 0 && i % kFlush == 0;            // R was drained: the sum starts over
          if (fresh && !warp_waits(r_empty, (i / kFlush - 1) & 1, lim)) { ok = false; break; }
          if (!warp_waits(&c_ready[b], par, lim)) { ok = false; break; }
          tc_fence_after();
          cv(tR, a + 64, v, !fresh);
        }
        umma_commit_one(one, &v_empty[b]);
        if (RLA && (i % kFlush == kFlush - 1 || i == n_tiles - 1)) umma_commit_one(one, r_full);
      }
      // This warp reaches the CTA-wide barrier before the merge only when all its products are complete: the merge reads O,
      // stages rows over the K and V tiles, and tensor memory is released after it, on expiry of a wait too.
      umma_commit_one(one, done);
      if (!warp_waits(done, 0, lim)) ok = false;
      if (!ok) *abort_flag = 1;
    }
  } else if (wg == 1) {
    // -------------------------------------------------------------- softmax: one row per thread ---------------------
    warpgroup_reg_inc<136>();
    const int row = tid - 128, pi = row / G;
    const int pos = (row < pc.P * G && pos0 + pi >= pos_lo && pos0 + pi < pos_hi) ? pos0 + pi : -1;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const float sc2 = p.sm_scale * kLog2e;
    TileWalk tw;
    tw.start(bitmap, B, own_hi);
    SelCursor cur;
    cur.start(pos >= 0 ? pc.sel + ((size_t)r.u * pc.T + (pos - r.first)) * p.top_k : nullptr, p.top_k);
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int i = 0; i < n_tiles && !warp_aborted(abort_flag); ++i) {
      tw.next();
      uint64_t sel, neg, posv;
      tile_masks(tw, cur, pos, base, sel, neg, posv);
      const int b = i & 1;
      const uint32_t src = tSA + b * 128 + lane_off;
      if (!warp_waits(&s_full[b], (i >> 1) & 1, lim)) { ok = false; break; }
      tc_fence_after();
      // Rows that attend to all of the tile or to none of it need no mask per token (a row that attends to none gets its
      // zeros from an infinite offset); tiles that reach past the sequence's end always take the masked form: what lies
      // there may be anything.
      const bool plain = __all_sync(0xffffffffu, sel == ~0ull || sel == 0ull) && !tile_past(tw, r.L_end);
      float mt = -INFINITY;
      {
        uint32_t s0[32], s1[32];
        tmem_ld32_async(src, s0);
        tmem_ld32_async(src + 32, s1);
        tmem_ld_wait32(s0);
        tmem_ld_wait32(s1);
        if (plain) {
          float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            mx0 = fmaxf(mx0, fmaxf(__uint_as_float(s0[j]), __uint_as_float(s0[j + 1])));
            mx1 = fmaxf(mx1, fmaxf(__uint_as_float(s1[j]), __uint_as_float(s1[j + 1])));
          }
          if (sel) mt = fmaxf(mx0, mx1) * sc2;                    // (sc2 > 0)
        } else {
          const uint32_t m0 = (uint32_t)sel, m1 = (uint32_t)(sel >> 32);
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (m0 & (1u << j)) mt = fmaxf(mt, __uint_as_float(s0[j]));
            if (m1 & (1u << j)) mt = fmaxf(mt, __uint_as_float(s1[j]));
          }
          mt *= sc2;
        }
      }
      // The first selected tile of a row sets its maximum (its row of O is zero so far); later ones only move it when it
      // would let a probability exceed 2^8.
      const bool grow = mt > m + 8.f && m > -INFINITY;
      if (m == -INFINITY) m = mt;
      if (__any_sync(0xffffffffu, grow)) {
        // every product with P so far must be done before O is touched
        if (!warp_waits(&v_empty[(i - 1) & 1], ((i - 1) >> 1) & 1, lim)) { ok = false; break; }
        tc_fence_after();
        const float m_new = grow ? mt : m;
        const float f = m > -INFINITY ? ex2(m - m_new) : 1.f;
        m = m_new;
        l *= f;
#pragma unroll 1
        for (int c = 0; c < D; c += 16) {
          uint32_t o[16];
          tmem_ld16_async(tO + lane_off + c, o);
          tmem_ld_wait16(o);
#pragma unroll
          for (int x = 0; x < 16; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * f);
          tmem_st16(tO + lane_off + c, o);
        }
      }
      const float nm = sel ? -m : -INFINITY;                      // (m is finite for a row that has selected anything)
      float2 sum = make_float2(0.f, 0.f);
      auto probs = [&](uint32_t (&s)[16], int c) {                // 16 tokens: scores -> head and remainder, in place
        if (!plain) {
          const uint32_t bits = (uint32_t)(sel >> (16 * c));
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (!(bits & (1u << j))) s[j] = 0xff800000u;
        }
        uint32_t pk[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[2 * j]), __uint_as_float(s[2 * j + 1])), make_float2(sc2, sc2), make_float2(nm, nm));
          const float2 pr = make_float2(ex2(x.x), ex2(x.y));
          sum = __fadd2_rn(sum, pr);
          pk[j] = pack_bf16(pr.x, pr.y);
          const float2 lo = __fadd2_rn(pr, make_float2(-bf16_lo(pk[j]), -bf16_hi(pk[j])));
          pk[8 + j] = pack_bf16(lo.x, lo.y);
        }
        tmem_st16(src + 16 * c, pk);
      };
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {                               // (rolled, like the other roles' loops: see the top)
        uint32_t cur16[16];
        tmem_ld16_async(src + 16 * c, cur16);
        tmem_ld_wait16(cur16);
        probs(cur16, c);
      }
      l += sum.x + sum.y;
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive1(&p_ready[b]);
    }
    if (!ok) *abort_flag = 1;
    l_s[row] = l;                                                 // (every S product has completed, or the CTA gives up)
  } else if (wg == 2) {
    // -------------------------------------------------------------- linear coefficients: one row per thread ---------
    warpgroup_reg_inc<232>();
    const int row = tid - 256, pi = row / G;
    const int pos = (row < pc.P * G && pos0 + pi >= pos_lo && pos0 + pi < pos_hi) ? pos0 + pi : -1;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    bool ok = true;
    float acc[RLA ? D : 1];
    if constexpr (RLA) {
      TileWalk tw;
      tw.start(bitmap, B, own_hi);
      SelCursor cur;
      cur.start(pos >= 0 ? pc.sel + ((size_t)r.u * pc.T + (pos - r.first)) * p.top_k : nullptr, p.top_k);
      const float cs = exp2f((float)(s_exp - kPhiExp));           // A carries 2^28, R shall carry 2^(14 + s_exp)
#pragma unroll
      for (int x = 0; x < D; ++x) acc[x] = 0.f;
#pragma unroll 1
      for (int i = 0; i <= n_tiles && !warp_aborted(abort_flag); ++i) {
        if (i == n_tiles || (i > 0 && i % kFlush == 0)) {         // a finished group of tiles, hidden behind the next one's first products
          if (!warp_waits(r_full, ((i - 1) / kFlush) & 1, lim)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < D; c += 32) {
            float v[32];
            tmem_ld32(tR + lane_off + c, v);
#pragma unroll
            for (int x = 0; x < 32; ++x) acc[c + x] += v[x];
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive1(r_empty);
          if (i == n_tiles) break;
        }
        tw.next();
        uint64_t sel, neg, posv;
        tile_masks(tw, cur, pos, base, sel, neg, posv);
        const int b = i & 1;
        const uint32_t src = tSA + b * 128 + 64 + lane_off;
        if (!warp_waits(&a_full[b], (i >> 1) & 1, lim)) { ok = false; break; }
        tc_fence_after();
        // signed coefficients: -A for selected tokens before the base, +A for unselected ones from it on, else 0 (never
        // 0 x A: a column past the sequence's end may hold anything)
        const bool plain = __all_sync(0xffffffffu, posv == 0ull && (neg == 0ull || neg == ~0ull)) && !tile_past(tw, r.L_end);
        const float mul = neg ? -cs : 0.f;
        auto coefs = [&](uint32_t (&x)[16], int c) {              // 16 tokens: A -> head and remainder, in place
          if (plain) {
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              const float2 y = __fmul2_rn(make_float2(__uint_as_float(x[j]), __uint_as_float(x[j + 1])), make_float2(mul, mul));
              x[j] = __float_as_uint(y.x);
              x[j + 1] = __float_as_uint(y.y);
            }
          } else {
            const uint32_t nb = (uint32_t)(neg >> (16 * c)), pb = (uint32_t)(posv >> (16 * c));
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float y = __uint_as_float(x[j]) * cs;
              x[j] = (nb & (1u << j)) ? __float_as_uint(-y) : (pb & (1u << j)) ? __float_as_uint(y) : 0u;
            }
          }
          uint32_t pk[16];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float2 c = make_float2(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1]));
            pk[j] = pack_bf16(c.x, c.y);
            const float2 lo = __fadd2_rn(c, make_float2(-bf16_lo(pk[j]), -bf16_hi(pk[j])));
            pk[8 + j] = pack_bf16(lo.x, lo.y);
          }
          tmem_st16(src + 16 * c, pk);
        };
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {                             // (rolled, like the other roles' loops: see the top)
          uint32_t cur16[16];
          tmem_ld16_async(src + 16 * c, cur16);
          tmem_ld_wait16(cur16);
          coefs(cur16, c);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive1(&c_ready[b]);
      }
    }
    if (!ok) *abort_flag = 1;
    __syncthreads();                                              // l of every row is there; every product is complete (see the issuer)
    tc_fence_after();
    if (!warp_aborted(abort_flag)) {
      // merge: out = O / l + gamma R rsqrt(mean R^2 + eps); rows staged in shared memory (16-byte pieces swizzled by row)
      const float inv_l = 1.f / l_s[row];
      const int nblk = pos / B + 1;
      const bool res = RLA && pos >= 0 && nblk > p.top_k;         // everything selected: the residual is exactly zero
      float rms = 0.f;
      if constexpr (RLA) {
        const float un = exp2f((float)(-kPhiExp - s_exp));
        float sq = 0.f;
#pragma unroll
        for (int x = 0; x < D; ++x) { acc[x] *= un; sq = fmaf(acc[x], acc[x], sq); }
        rms = res ? rsqrtf(sq / D + p.rms_eps) : 0.f;
      }
      const float4* gm = reinterpret_cast<const float4*>(rms_weight + ((size_t)r.h * G + row % G) * D);
      unsigned char* stage = smem + SM::kK + row * (D * 4);
#pragma unroll
      for (int c = 0; c < D; c += 32) {
        float o[32];
        tmem_ld32(tO + lane_off + c, o);
#pragma unroll
        for (int x = 0; x < 32; x += 4) {
          float4 v = make_float4(o[x] * inv_l, o[x + 1] * inv_l, o[x + 2] * inv_l, o[x + 3] * inv_l);
          if constexpr (RLA) {
            if (res) {
              const float4 g = __ldg(gm + (c + x) / 4);
              v.x = fmaf(g.x * rms, acc[c + x], v.x); v.y = fmaf(g.y * rms, acc[c + x + 1], v.y);
              v.z = fmaf(g.z * rms, acc[c + x + 2], v.z); v.w = fmaf(g.w * rms, acc[c + x + 3], v.w);
            }
          }
          *reinterpret_cast<float4*>(stage + ((((c + x) / 4) ^ (row & 7)) << 4)) = v;
        }
      }
      tc_fence_before();
    }
  } else {
    // -------------------------------------------------------------- phi(K), and zero value rows past the end ---------
    warpgroup_reg_dec<88>();
    const int tg = tid - 384;
    const float a2 = p.phi_scale * kLog2e;
    TileWalk tw;
    tw.start(bitmap, B, own_hi);
    bool ok = true;
    for (int i = 0; i < n_tiles && !warp_aborted(abort_flag); ++i) {
      tw.next();
      const int b = i & 1, par = (i >> 1) & 1;
      if (!warp_waits(&k_full[b], par, lim)) { ok = false; break; }
      if constexpr (RLA) {
        if (!warp_waits(&phi_empty[b], par, lim)) { ok = false; break; }
        // thread tg owns the 16-byte pieces tg, tg + 128, ...: rows tg / 8 + 16 j of every array; the swizzle moves pieces
        // only inside their row, and phi is elementwise given the token's log-sum-exp
        const unsigned char* kt = smem + SM::kK + b * SM::kTileBytes + tg * 16;
        unsigned char* ph = smem + SM::kPhi + b * 2 * SM::kTileBytes + tg * 16;
#pragma unroll 2
        for (int j = 0; j < SM::kTileBytes / 2048; ++j) {
          const float nl2 = fmaf(-lse_s[b * kPaTile + (tg >> 3) + 16 * (j & 3)], kLog2e, (float)kPhiExp);
          const uint4 raw = *reinterpret_cast<const uint4*>(kt + j * 2048);
          const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
          uint32_t h[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 x = __ffma2_rn(make_float2(bf16_lo(w[e]), bf16_hi(w[e])), make_float2(a2, a2), make_float2(nl2, nl2));
            const float2 f = make_float2(ex2(x.x), ex2(x.y));
            h[e] = pack_h2(f.x, f.y);
            const float2 d = __fadd2_rn(f, make_float2(-h2_lo(h[e]), -h2_hi(h[e])));
            lo[e] = pack_h2(d.x, d.y);
          }
          *reinterpret_cast<uint4*>(ph + j * 2048) = make_uint4(h[0], h[1], h[2], h[3]);
          *reinterpret_cast<uint4*>(ph + SM::kTileBytes + j * 2048) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      }
      // rows past the sequence's end hold whatever the cache memory holds; 0 x V must be 0
      const bool past = tile_past(tw, r.L_end);                   // uniform over the four warps
      bool look = past;
      if constexpr (!RLA) {                                       // the largest magnitude of the thread's pieces, NaN above all
        if (!warp_waits(&v_full[b], par, lim)) { ok = false; break; }
        const unsigned char* vt = smem + SM::kV + b * SM::kTileBytes + tg * 16;
        __nv_bfloat162 most = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll 4
        for (int j = 0; j < SM::kTileBytes / 2048; ++j) {
          const uint4 v = *reinterpret_cast<const uint4*>(vt + j * 2048);
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) most = __hmax2_nan(most, __habs2(*reinterpret_cast<const __nv_bfloat162*>(&w[e])));
        }
        look |= not_finite2(*reinterpret_cast<const uint32_t*>(&most)) != 0u;
      }
      if (look) {
        if (RLA && !warp_waits(&v_full[b], par, lim)) { ok = false; break; }
#pragma unroll 1
        for (int j = 0; j < SM::kTileBytes / 2048; ++j) {          // the thread's pieces: rows tg / 8 + 16 j of either array
          const int rw = (tg >> 3) + 16 * (j & 3), ch = ((tg & 7) ^ (rw & 7)) + 8 * (j >> 2);
          uint4* vp = reinterpret_cast<uint4*>(smem + SM::kV + b * SM::kTileBytes + tg * 16 + j * 2048);
          uint32_t bad = 0u;
          if constexpr (!RLA) {
            const uint4 v = *vp;
            bad = not_finite2(v.x) | not_finite2(v.y) | not_finite2(v.z) | not_finite2(v.w);
          }
          if (!past && !bad) continue;
          const int blk = B < kPaTile ? tw.sub_block(rw / B) : tw.blk[0];
          const int tok = blk * B + tw.off + (B < kPaTile ? rw % B : rw);
          if (tok >= r.L_end) *vp = make_uint4(0u, 0u, 0u, 0u);
          else if (bad) take_out_not_finite<D>(vp, tok, blk, ch, pc.sel + (size_t)r.u * pc.T * p.top_k, r.first, p.top_k, pos0, pos_lo, pos_hi, marks);
        }
      }
      proxy_fence();                                              // phi(K) and V writes -> tensor core; K reads before the next copy
      __syncwarp();
      if (lane == 0) { mbar_arrive1(&phi_ready[b]); mbar_arrive1(&k_empty[b]); }
    }
    if (!ok) *abort_flag = 1;
  }

  // ---------------------------------------------------------------- end: rows out, tensor memory back -----------------
  __syncwarp();
  if (wg != 2) __syncthreads();                                   // (pairs with the linear warps' barrier before the merge)
  __syncthreads();
  if (!*abort_flag) {
    constexpr int Q4 = D / 4;
    for (int x = tid; x < kPfRows * Q4; x += kPaThreads) {
      const int row = x / Q4, c4 = x % Q4, pi = row / G, pos = pos0 + pi;
      if (row >= pc.P * G || pos < pos_lo || pos >= pos_hi) continue;
      float4 v = *reinterpret_cast<const float4*>(smem + SM::kK + row * (D * 4) + ((c4 ^ (row & 7)) << 4));
      if constexpr (!RLA) {
        const uint32_t mk = marks[pi * (D / 32) + c4 / 8] >> (c4 % 8 * 4);
        const float nan = __uint_as_float(0x7fffffffu);
        if (mk & 1u) v.x = nan;
        if (mk & 2u) v.y = nan;
        if (mk & 4u) v.z = nan;
        if (mk & 8u) v.w = nan;
      }
      *reinterpret_cast<float4*>(out + (((size_t)r.b * pc.T + (pos - r.first)) * p.Hq + (size_t)r.h * G + row % G) * D + c4 * 4) = v;
    }
  } else if (tid == 0) {
    atomicExch(p.status, kStatusTimeout);
  }
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_free(tmem, kPaTmemCols);
  }
}

template <int D, bool RLA>
cudaError_t attend_d(const Params& p, const PrefillChunk& c, const AttendMaps& maps, const void* q, const float* w, float* out, cudaStream_t s) {
  auto kern = prefill_attend_kernel<D, RLA>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PaSmem<D>::kBytes);
  if (e != cudaSuccess) return e;
  // Launched ahead of the selection's end up to two waves of CTAs (288: 294 -> 290 us per chunk; 2064: 1553 -> 1569 us).
  const bool ahead = (long long)c.nq * c.nu <= 2 * 148;
  return launch_ex(kern, dim3(c.nq, c.nu), dim3(kPaThreads), PaSmem<D>::kBytes, s, 0, ahead,
                   p, c, *reinterpret_cast<const CUtensorMap*>(maps.k), *reinterpret_cast<const CUtensorMap*>(maps.v),
                   reinterpret_cast<const __nv_bfloat16*>(q), w, out);
}

}  // namespace

cudaError_t launch_prefill_attend(const Params& p, const PrefillChunk& c, const AttendMaps& maps, const void* q, const float* rms_weight,
                                  float* out, cudaStream_t s) {
  if (p.flags & 4u)
    return p.d == 128 ? attend_d<128, false>(p, c, maps, q, rms_weight, out, s) : attend_d<64, false>(p, c, maps, q, rms_weight, out, s);
  return p.d == 128 ? attend_d<128, true>(p, c, maps, q, rms_weight, out, s) : attend_d<64, true>(p, c, maps, q, rms_weight, out, s);
}

}  // namespace spla
