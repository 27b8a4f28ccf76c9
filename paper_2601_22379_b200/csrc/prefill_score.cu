// Block scores and selection of every position of a prefill chunk (Section 3.1, Eq. taylor-2nd; Section 2.2, grouped
// BlockScore; Section 2.1, Select), as a contraction instead of one pass over the statistics per position.
//
// For the complete blocks the Taylor log masses of 128 query rows (P positions x G heads) and 64 records are two matrix
// products, q . mean and (q^2) . var, on the 5th-generation tensor cores.  Precision is that of fp32 products: q is bf16
// already and its square has 16 significant bits, exactly two bf16 parts; an fp32 record element enters as three bf16 parts
// (24 bits), a 16-bit one as itself; scale factors are applied to the fp32 sums.  Eight products per record and row with
// fp32 records, three with 16-bit ones.  Log masses are kept relative to ln B, the count term of every complete block (the
// softmax over blocks does not see it): in front of 4.2 (B = 64) their own rounding was most of their error.  Against 64 bits,
// aggregated scores of 500 blocks, G = 4: 1.4e-7 with ln B in front, 1.0e-7 on the general kernels (which keep it), 0.9e-7 to 1.0e-7 now (G = 16: 1.0e-7 against 0.5e-7;
// what is left is the tensor core cutting off when it adds).
#include "prefill_chunk.h"
#include "umma.cuh"

namespace spla {

namespace {

constexpr int kPsThreads = 416;            // 4 warps: rows in, log masses out; 8: records; 1: products
constexpr int kPsLoaders = 256;
constexpr int kPsRec = 64;                 // records of a tile: the N of the products
constexpr uint32_t kPsTmemCols = 512;

template <int D, bool R16>
struct PsSmem {
  static constexpr int H = D / 64;                             // arrays of 128-byte rows per part
  static constexpr int NP = R16 ? 1 : 3;                       // parts of a record element
  static constexpr int kHalf = kPsRec * 128;
  static constexpr int kPart = H * kHalf;
  static constexpr int kStage = 2 * NP * kPart;                // means, variances: 96 KB (d = 128, fp32)
  static constexpr int kBars = 2 * kStage;
  static constexpr int kMisc = kBars + 10 * 8;                 // tensor-memory base, abort flag
  static constexpr int kBytes = kMisc + 16;
};

__device__ __forceinline__ void store8(float* dst, const float (&v)[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
               "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// One CTA: one tile of query rows, `rec_per_cta` consecutive records, 64 at a time.  The rows (q and the two parts of q^2)
// stay in tensor memory as the left operand; eight warps cut the records into their parts, two tiles in shared memory and a
// third on its way in registers; one warp issues the products into two pairs of accumulators; four warps turn finished sums
// into log masses, one row per thread, in whole 32-byte sectors.
//
// Bound by the tensor pipe: 64 products of 128 x 64 x 16 per tile, 45 cycles each (2900 per
// tile), and by a CTA's start where it has few tiles.  512 tokens on 32768 x 2 (16 units, 513 blocks, fp32): 132 us on the
// warp-level tensor cores (the same products, operands through ldmatrix), 52 us now; the 8192-token prompt: 145 us, 115 us.
//
// Every wait has an iteration limit; on expiry all roles leave, tensor memory is released and the time-out is latched.
template <int D, bool R16>
__global__ void __launch_bounds__(kPsThreads, 1) prefill_score_kernel(const Params p, const PrefillChunk pc,
                                                                      const __nv_bfloat16* __restrict__ q, int rec_per_cta) {
  using SM = PsSmem<D, R16>;
  constexpr int H = SM::H, NP = SM::NP;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::kBars);
  uint64_t *r_full = bars, *r_empty = bars + 2, *c_full = bars + 4, *c_empty = bars + 6, *q_ready = bars + 8, *done = bars + 9;
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(smem + SM::kMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SM::kMisc + 4);
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const PrefillUnit r = prefill_unit_of(p, pc, pc.u0 + blockIdx.z);
  const int G = p.G;
  const int sb = (pc.q0 + (int)blockIdx.y) / pc.nt, tile = (pc.q0 + (int)blockIdx.y) % pc.nt;
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
  const int n_tiles = (rec1 - rec0 + kPsRec - 1) / kPsRec;
  const int lim = p.wait_limit;
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&r_full[s], kPsLoaders / 32);  mbar_init(&r_empty[s], 1);
      mbar_init(&c_full[s], 1);  mbar_init(&c_empty[s], 4);
    }
    mbar_init(q_ready, 4);
    mbar_init(done, 1);
    mbar_init_done();
    *abort_flag = 0;
  }
  if (warp == 12) tmem_alloc(tmem_base_s, kPsTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  const uint32_t tQ = tmem + 256;                              // q, then q^2 head and remainder, D / 2 columns each
  bool ok = true;

  if (warp < 4) {
    // ---------------------------------------------------------------- rows in, log masses out: one row per thread ----
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
    const int row = tid, pos = pos0 + row / G;
    const bool live = row < pc.P * G && pos >= r.L0 && pos < pos_hi;
    {
      const uint4* qr = reinterpret_cast<const uint4*>(
          q + (((size_t)r.b * pc.T + (live ? pos - r.first : 0)) * p.Hq + (size_t)r.h * G + row % G) * D);
      uint4 raw[D / 8];
#pragma unroll
      for (int j = 0; j < D / 8; ++j) raw[j] = live ? __ldg(qr + j) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {                       // 32 channels = 16 columns
        uint32_t w[16], h[16], l[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint4 x = raw[c * 4 + j];
          w[4 * j] = x.x; w[4 * j + 1] = x.y; w[4 * j + 2] = x.z; w[4 * j + 3] = x.w;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {                         // q^2 in two bf16 parts: exact
          const float a = bf16_lo(w[j]), b = bf16_hi(w[j]), a2 = a * a, b2 = b * b;
          h[j] = pack_bf16(a2, b2);
          l[j] = pack_bf16(a2 - bf16_lo(h[j]), b2 - bf16_hi(h[j]));
        }
        tmem_st16(tQ + lane_off + c * 16, w);
        tmem_st16(tQ + lane_off + D / 2 + c * 16, h);
        tmem_st16(tQ + lane_off + D + c * 16, l);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive1(q_ready);
    }
    const size_t slot = ((size_t)blockIdx.z * pc.nq + blockIdx.y) * pc.P + (live ? pos - pos0 : 0);
    float* dst = pc.ell + (slot * G + row % G) * pc.stride + rec0;
    const float half_s2 = (p.flags & 2u) ? 0.f : 0.5f * p.sm_scale * p.sm_scale;
#pragma unroll 1
    for (int i = 0; i < n_tiles && !warp_aborted(abort_flag); ++i) {
      const int b = i & 1;
      if (!warp_waits(&c_full[b], (i >> 1) & 1, lim)) { ok = false; break; }
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < kPsRec && rec0 + i * kPsRec + c < rec1; c += 32) {   // (a row of ell has room for whole groups of 32)
        uint32_t m[32], v[32];
        tmem_ld32_async(tmem + b * 128 + lane_off + c, m);
        tmem_ld32_async(tmem + b * 128 + 64 + lane_off + c, v);
        tmem_ld_wait32(m);
        tmem_ld_wait32(v);
        if (live) {
#pragma unroll
          for (int x = 0; x < 32; x += 8) {
            float e[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
              e[j] = __uint_as_float(m[x + j]) * p.sm_scale + __logf(1.f + half_s2 * __uint_as_float(v[x + j]));
            store8(dst + i * kPsRec + c + x, e);
          }
        }
        __syncwarp();
      }
      tc_fence_before();
      if (lane == 0) mbar_arrive1(&c_empty[b]);
    }
  } else if (warp < 12) {
    // ---------------------------------------------------------------- records: 16-byte pieces, cut into bf16 parts ----
    constexpr int kPerRec = 2 * D * (R16 ? 2 : 4) / 16;        // pieces of a record
    constexpr int kStep = kPsLoaders / kPerRec;                // records between a thread's pieces
    constexpr int kPieces = kPsRec / kStep;                    // per thread and tile: 16 (d = 128, fp32) .. 4
    const int t = tid - 128, rec_t = t / kPerRec, pc16 = t % kPerRec;
    const bool var = pc16 >= kPerRec / 2;
    const int ch = (var ? pc16 - kPerRec / 2 : pc16) * (R16 ? 8 : 4);   // first channel of the thread's pieces
    const uint4* recs = reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(p.stats) +
                                                       (size_t)r.u * p.max_blocks * 2 * D * (R16 ? 2 : 4));
    uint4 st[kPieces];
    auto fetch = [&](int base) {
#pragma unroll
      for (int j = 0; j < kPieces; ++j) {
        const int rec = base + j * kStep + rec_t;
        st[j] = rec < rec1 ? __ldg(recs + (size_t)rec * kPerRec + pc16) : make_uint4(0u, 0u, 0u, 0u);
      }
    };
    fetch(rec0);
    unsigned char* dst0 = smem + (var ? NP * SM::kPart : 0) + (ch >> 6) * SM::kHalf + (ch & 4) * 2;
#pragma unroll 1
    for (int i = 0; i < n_tiles && !warp_aborted(abort_flag); ++i) {
      const int b = i & 1;
      if (i >= 2 && !warp_waits(&r_empty[b], ((i >> 1) - 1) & 1, lim)) { ok = false; break; }
      unsigned char* stage = dst0 + b * SM::kStage;
#pragma unroll
      for (int j = 0; j < kPieces; ++j) {
        const int rec = j * kStep + rec_t;
        unsigned char* dst = stage + rec * 128 + ((((ch & 63) >> 3) ^ (rec & 7)) << 4);
        if constexpr (R16) {
          *reinterpret_cast<uint4*>(dst) = st[j];
        } else {
          const float f0 = __uint_as_float(st[j].x), f1 = __uint_as_float(st[j].y), f2 = __uint_as_float(st[j].z), f3 = __uint_as_float(st[j].w);
          const uint32_t h0 = pack_bf16(f0, f1), h1 = pack_bf16(f2, f3);
          const float a0 = f0 - bf16_lo(h0), a1 = f1 - bf16_hi(h0), a2 = f2 - bf16_lo(h1), a3 = f3 - bf16_hi(h1);
          const uint32_t m0 = pack_bf16(a0, a1), m1 = pack_bf16(a2, a3);
          const uint32_t l0 = pack_bf16(a0 - bf16_lo(m0), a1 - bf16_hi(m0)), l1 = pack_bf16(a2 - bf16_lo(m1), a3 - bf16_hi(m1));
          *reinterpret_cast<uint2*>(dst) = make_uint2(h0, h1);
          *reinterpret_cast<uint2*>(dst + SM::kPart) = make_uint2(m0, m1);
          *reinterpret_cast<uint2*>(dst + 2 * SM::kPart) = make_uint2(l0, l1);
        }
      }
      proxy_fence();                                           // -> visible to the tensor core
      __syncwarp();
      if (lane == 0) mbar_arrive1(&r_full[b]);
      if (i + 1 < n_tiles) fetch(rec0 + (i + 1) * kPsRec);
    }
  } else {
    // ---------------------------------------------------------------- products (a converged warp, one lane issues) ----
    constexpr uint32_t idesc = umma_idesc(true, false, false, kPfRows, kPsRec);
    constexpr int kProducts = R16 ? 3 : 8;                     // q x NP parts, head of q^2 x NP, its remainder x the first one or two
    const uint32_t one = elect_one();
    const uint32_t lo0 = umma_desc_lo(smem_u32(smem), 16);
    ok = warp_waits(q_ready, 0, lim);
#pragma unroll 1
    for (int i = 0; i < n_tiles && ok && !warp_aborted(abort_flag); ++i) {
      const int b = i & 1;
      if (!warp_waits(&r_full[b], (i >> 1) & 1, lim) || (i >= 2 && !warp_waits(&c_empty[b], ((i >> 1) - 1) & 1, lim))) { ok = false; break; }
      tc_fence_after();
#pragma unroll 1
      for (int x = kProducts - 1; x >= 0; --x) {               // (small terms first)
        const uint32_t a = tQ + (x < NP ? 0 : x < 2 * NP ? D / 2 : D);
        const uint32_t part = x < 2 * NP ? x : x - NP;
        const uint32_t lo = lo0 + (uint32_t)(b * SM::kStage) / 16 + part * (SM::kPart / 16);
        const uint32_t acc = x != kProducts - 1 && x != NP - 1;
#pragma unroll
        for (int hh = 0; hh < H; ++hh)
          umma_ts4_one<8, 2>(one, tmem + b * 128 + (x < NP ? 0 : 64), a + hh * 32, lo + hh * (SM::kHalf / 16), idesc, hh > 0 ? 1u : acc);
      }
      umma_commit_one(one, &r_empty[b]);
      umma_commit_one(one, &c_full[b]);
    }
    umma_commit_one(one, done);
    if (!warp_waits(done, 0, lim)) ok = false;                 // nothing in flight when tensor memory is released
  }
  if (!ok) {
    *abort_flag = 1;
    if (lane == 0) atomicExch(p.status, kStatusTimeout);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 12) tmem_free(tmem, kPsTmemCols);
}

// Selection of one position by W warps (W = 1: one warp per position, up to 32 NK blocks; W = 8: a CTA per position, up to
// 256 NK).  Each lane keeps the keys of its NK blocks in registers.  The k-th best key is found bit by bit from the top
// (counting the keys at or above a candidate, with a stop as soon as exactly k are), which needs no scratch and no sort;
// the list then comes out in ascending order by ballots.  A warp with 16 or more keys per lane first bounds the k-th best key
// from below by that of the 64 best ones of half a lane each, and ranks the few keys that reach the bound instead (513
// blocks, 512 positions x 16 units: 55 -> 42 us, bound by instructions issued).
constexpr int kFew = 64;
template <int W, int NK>
__global__ void __launch_bounds__(256, 2) prefill_select_kernel(const Params p, const PrefillChunk pc, int* __restrict__ sel_user) {
  __shared__ float red_s[8][2];
  __shared__ int cnt_s[2][8];
  constexpr bool FEW = W == 1 && NK >= 16;
  __shared__ __align__(16) unsigned long long flat_s[FEW ? 8 : 1][kFew];   // keys that reach the bound, with their blocks
  __shared__ __align__(16) int pick_s[FEW ? 8 : 1][kFew];
  constexpr int L = W * 32;                                    // lanes of a position
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const PrefillUnit r = prefill_unit_of(p, pc, pc.u0 + blockIdx.y);
  const int G = p.G;
  const int slot = blockIdx.x * (8 / W) + (W == 1 ? warp : 0);   // position within the launch's row tiles
  const int tq = pc.q0 + slot / pc.P, in_range = tq % pc.nt * pc.P + slot % pc.P;
  const int pos = prefill_range_start(pc, r, tq / pc.nt) + in_range;
  if (slot >= pc.nq * pc.P || in_range >= pc.SB || pos < r.L0 || pos >= r.L_end) return;   // uniform over the position's warps
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

  // aggregated score of the lane's blocks: per head softmax over the position's blocks, summed over the group.  Up to 64 blocks, where
  // latency counts, the next head's log masses are on their way meanwhile, and only as many keys as the position has blocks (511
  // tokens x 4 units, G = 8: 82.3 -> 79.9 us a call; 77 tokens x 4 units 48.3 -> 47.5; with more keys it is instructions that count: the
  // 8192-token prompt, four keys, 1680 -> 1690).
  constexpr bool AHEAD = NK <= 2;
  float sc[NK];
#pragma unroll
  for (int k = 0; k < NK; ++k) sc[k] = 0.f;
  const float* ell = pc.ell + (((size_t)blockIdx.y * pc.nq * pc.P + slot) * G) * pc.stride;
  const float* own_row = pc.ell_own + ((size_t)r.u * pc.T + t) * G;
  float nxt[AHEAD ? NK : 1];
  auto ahead = [&](int g) {
#pragma unroll
    for (int k = 0; k < (AHEAD ? NK : 0); ++k) {
      if (k > 0 && k * L >= nblk) break;                       // (uniform)
      const int i = k * L + l;
      nxt[k] = i < nblk ? *(i < own ? ell + (size_t)g * pc.stride + i : own_row + g) : -INFINITY;
    }
  };
  if constexpr (AHEAD) ahead(0);
  for (int g = 0; g < G; ++g) {
    float e[NK], mx = -INFINITY;
    if constexpr (AHEAD) {
#pragma unroll
      for (int k = 0; k < NK; ++k) e[k] = nxt[k];
      if (g + 1 < G) ahead(g + 1);
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        if (k > 0 && k * L >= nblk) break;
        mx = fmaxf(mx, e[k]);
      }
    } else {
      const float e_own = own_row[g];
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        const int i = k * L + l;
        e[k] = i < own ? ell[(size_t)g * pc.stride + i] : (i == own ? e_own : -INFINITY);
        mx = fmaxf(mx, e[k]);
      }
    }
    mx = reduce(mx, true);
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      if (AHEAD && k > 0 && k * L >= nblk) break;
      e[k] = __expf(e[k] - mx);
      sum += e[k];
    }
    const float inv = 1.f / reduce(sum, false);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      if (AHEAD && k > 0 && k * L >= nblk) break;
      sc[k] = fmaf(e[k], inv, sc[k]);
    }
  }
  // keys: 0 for blocks that do not exist, all ones for the forced ones, else the score's bits + 1 (positive floats order
  // like integers)
  uint32_t key[NK];
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    const int i = k * L + l;
    key[k] = i >= nblk ? 0u : (i < p.n_sink || i >= nblk - p.n_local) ? 0xffffffffu : __float_as_uint(sc[k]) + 1u;
  }
  int* sel_w = pc.sel + ((size_t)r.u * pc.T + t) * p.top_k;
  int* sel_o = sel_user ? sel_user + (((size_t)r.b * pc.T + t) * p.Hkv + r.h) * p.top_k : nullptr;
  if constexpr (FEW) {
    if (k_eff < nblk) {
      uint32_t m0 = 0u, m1 = 0u;
#pragma unroll
      for (int k = 0; k < NK; k += 2) { m0 = max(m0, key[k]); m1 = max(m1, key[k + 1]); }
      uint32_t low = 0u;                                       // k_eff of the 64 maxima, of different blocks, are at least this
#pragma unroll 1
      for (int bit = 31; bit >= 0; --bit) {
        const uint32_t cand = low | (1u << bit);
        const int c = __popc(__ballot_sync(0xffffffffu, m0 >= cand)) + __popc(__ballot_sync(0xffffffffu, m1 >= cand));
        if (c >= k_eff) low = cand;
        if (c == k_eff) break;
      }
      int c = 0;
#pragma unroll
      for (int k = 0; k < NK; ++k) c += key[k] >= low;
      int dst = c;                                             // where the lane's keys start: the sum of the lanes before
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, dst, o);
        if (lane >= o) dst += x;
      }
      const int total = __shfl_sync(0xffffffffu, dst, 31);
      if (low > 0u && total <= kFew) {
        unsigned long long* flat = flat_s[warp];
        int* pick = pick_s[warp];
        flat[lane] = flat[32 + lane] = 0ull;
        __syncwarp();
        dst -= c;
#pragma unroll
        for (int k = 0; k < NK; ++k)
          if (key[k] >= low) flat[dst++] = ((unsigned long long)key[k] << 32) | (uint32_t)(0x7fffffff - (k * L + l));   // (ties: the smaller block first)
        __syncwarp();
        const unsigned long long a0 = flat[lane], a1 = flat[32 + lane];
        int r0 = 0, r1 = 0;
#pragma unroll 4
        for (int j = 0; j < total; j += 2) {
          const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(flat + j);
          r0 += (x.x > a0) + (x.y > a0);
          r1 += (x.x > a1) + (x.y > a1);
        }
        const bool take0 = lane < total && r0 < k_eff, take1 = 32 + lane < total && r1 < k_eff;
        const int i0 = 0x7fffffff - (int)(uint32_t)a0, i1 = 0x7fffffff - (int)(uint32_t)a1;
        pick[lane] = take0 ? i0 : 0x7fffffff;
        pick[32 + lane] = take1 ? i1 : 0x7fffffff;
        __syncwarp();
        int p0 = 0, p1 = 0;
#pragma unroll 4
        for (int j = 0; j < total; j += 4) {
          const int4 x = *reinterpret_cast<const int4*>(pick + j);
          p0 += (x.x < i0) + (x.y < i0) + (x.z < i0) + (x.w < i0);
          p1 += (x.x < i1) + (x.y < i1) + (x.z < i1) + (x.w < i1);
        }
        if (take0) { sel_w[p0] = i0; if (sel_o) sel_o[p0] = i0; }
        if (take1) { sel_w[p1] = i1; if (sel_o) sel_o[p1] = i1; }
        for (int s = k_eff + l; s < p.top_k; s += L) {
          sel_w[s] = -1;
          if (sel_o) sel_o[s] = -1;
        }
        return;
      }
    }
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
  constexpr size_t smem = PsSmem<D, R16>::kBytes;
  auto kern = prefill_score_kernel<D, R16>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // Tiles of records per CTA: what leaves the fewest tile times, a CTA's start counted as one (one CTA per SM).
  const int all = (max_blocks_seen + kPsRec - 1) / kPsRec;
  const long long row_tiles = (long long)c.nq * c.nu;
  int per = all;
  long long best = -1;
  for (int ny = 1; ny <= all; ++ny) {
    const int n = (all + ny - 1) / ny;
    const long long cost = (row_tiles * ((all + n - 1) / n) + sm_count - 1) / sm_count * (n + 1);
    if (best < 0 || cost < best) { best = cost; per = n; }
  }
  return launch_ex(kern, dim3((all + per - 1) / per, c.nq, c.nu), dim3(kPsThreads), smem, s, 0, true,
                   p, c, reinterpret_cast<const __nv_bfloat16*>(q), per * kPsRec);
}

template <int W, int NK>
cudaError_t select_w(const Params& p, const PrefillChunk& c, int* sel_user, cudaStream_t s) {
  const int slots = c.nq * c.P;
  return launch_ex(prefill_select_kernel<W, NK>, dim3((slots + 8 / W - 1) / (8 / W), c.nu), dim3(256), 0, s, 0, true, p, c, sel_user);
}

}  // namespace

// Log masses of the complete blocks, for the row tiles and units of one launch.  max_blocks_seen: blocks of the
// longest sequence after the chunk.
cudaError_t launch_prefill_score(const Params& p, const PrefillChunk& c, const void* q, int max_blocks_seen, int sm_count, cudaStream_t s) {
  if (p.flags & kStatsBf16)
    return p.d == 128 ? score_d<128, true>(p, c, q, max_blocks_seen, sm_count, s) : score_d<64, true>(p, c, q, max_blocks_seen, sm_count, s);
  return p.d == 128 ? score_d<128, false>(p, c, q, max_blocks_seen, sm_count, s) : score_d<64, false>(p, c, q, max_blocks_seen, sm_count, s);
}

// Selection for the same positions.  Up to 1024 blocks a warp holds a position's keys; above, a CTA does (513 blocks, 512 positions x 16
// units: 121 us by CTAs, whose barriers cost more than the wider registers of one warp, 42 us by warps).
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
