// Bulk append of a bf16 cache with d = 128 in one pass over the new tokens: K and V go into the cache, the per-token
// log-sum-exp, the block statistics (Section 3.1 of the paper, Eq. taylor-2nd) and the recurrent state
// S_bar += phi(K)^T V (Section 3.2, Eq. rla-impl-1; "Numerical Stability": kept in fp32) are formed from the same
// shared-memory tiles.
//
// The state update is a dense [d x n] . [n x d] contraction per (sequence, KV head) unit on tcgen05: M = 128 features of
// phi(k), N = 128 value channels, K = tokens, the 128 x 128 fp32 accumulator in tensor memory.  A token's d channels are
// contiguous, so both operands are MN-major, and a TMA box of 64 tokens x 64 channels with the 128-byte swizzle lands in
// the canonical layout the matrix descriptors name.
//
// One CTA takes a contiguous share of a unit's 64-token tiles (tiles are aligned in the sequence, so a tile holds whole
// blocks, or half of a 128-token one).  16 warps:
//   warp 0      TMA loads of the new K and V rows into a ring of four tiles;
//   warp 1      issues the products: phi as two or three bf16 parts against V, 8 or 12 MMAs per tile;
//   warp 2      TMA stores of whole tiles from the ring into the cache;
//   warps 4-11  two groups taking the tiles in turn: log-sum-exp and phi(k) = exp(phi_scale k - lse) of a row by the eight
//               lanes that hold it; on tiles that are not wholly new also the row-wise cache writes and the zeroing of what
//               is not new.  They also drain the accumulator into fp32 registers every tile or two: the tensor core does not
//               round to nearest when it adds (1e-4 relative after a chain of 4000 instructions);
//   warps 12-15 block statistics: two exact passes in the summation order of the other append kernels (same bits), one
//               channel pair and every second token per thread.
// The lengths are advanced by the last CTA to have read them (a ticket; nobody waits).  Shares of a unit are added to S_bar
// in share order by a second small kernel (reproducible); with one share per unit the CTA adds to S_bar itself.
//
// Bound by HBM: every token is read once and written once.  Before, one kernel copied (K staged once more for the
// statistics) and a second read everything again for the state.
// 131072 tokens x 32 units (4.3 GB in and out): copy and state kernels 1.44 ms, this one 0.84 ms a call = 5.1 TB/s, 0.79 of the
// measured copy rate; 50 to 700 tokens x 128 units on a history: 45 -> 32 us.  What keeps it from the copy rate: 16 warps in five roles issue from code that does not
// fit the SM's instruction cache (fewer rows or tokens per loop body cost more in latency than they gain there).
//
// Every wait is an mbarrier poll with an iteration limit; a role whose wait runs out raises the CTA's abort flag and leaves its
// loop, the others then run into their own limits; the copies and products in flight are waited for, tensor memory is
// released, the share counts as zero in S_bar and the time-out status is latched.  No multicast anywhere.
#include "spla_internal.h"
#include "umma.cuh"

namespace spla {

namespace {

constexpr int kAbD = 128;
constexpr int kAbTile = 64;                                  // tokens per tile
constexpr int kAbStages = 4;
constexpr int kAbRows = 2;                                   // rows a phi thread works on side by side
constexpr int kAbThreads = 512;
constexpr int kAbHalf = kAbTile * 128;                       // one TMA box: 64 tokens x 64 channels bf16
constexpr int kAbTileBytes = 2 * kAbHalf;                    // 16 KB: all 128 channels
constexpr int kAbMaxParts = 3;                               // bf16 parts of phi, at most
constexpr int kAbTwoParts = 256;                             // new tokens per sequence from which two parts are used
// Tiles accumulated in tensor memory before a drain: two; one where phi has all its bits, whose sums would otherwise show the
// cuts of the tensor core's adder (S_bar after 40 to 255 tokens, against 64 bits: 1.0e-7 to 1.4e-7 so, 3.4e-7 to 4.5e-7 after two
// tiles and the largest terms first, 2.6e-7 to 5.9e-7 from the fp32 kernels; 255 tokens x 512 units 90 -> 92 us).
template <int PARTS> constexpr int kAbGroupOf = PARTS == 3 ? 1 : 2;
constexpr int kAbTmemCols = 256;                             // two 128-column accumulators, used in turn
// shared memory: ring [stage][K, V], phi [2][part], reduction buffers of the statistics, barriers
constexpr int kAbPhi = kAbStages * 2 * kAbTileBytes;
constexpr int kAbRed = kAbPhi + 2 * kAbMaxParts * kAbTileBytes; // float [2 passes][2 parities][128]
constexpr int kAbBars = kAbRed + 2 * 2 * kAbD * 4;
constexpr int kAbNumBars = 2 * kAbStages + 9;
constexpr int kAbMisc = kAbBars + kAbNumBars * 8;            // tensor-memory base, abort flag
constexpr int kAbSmem = kAbMisc + 16;
static_assert(kAbSmem <= 227 * 1024, "shared memory of the bulk append");

constexpr uint32_t kAbIdesc = umma_idesc(true, true, true, kAbD, kAbD);   // A and B MN-major bf16, 128 x 128

// One TMA box from shared memory into the cache (its own bulk group is committed by the caller).
__device__ __forceinline__ void tma_store_box(const CUtensorMap* map, int x, int y, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(x), "r"(y), "r"(src) : "memory");
}

// PARTS: bf16 parts of phi.  Two (16 significant bits, rounded to nearest) for long appends, three (24 bits) for short ones.
template <int PARTS>
__global__ void __launch_bounds__(kAbThreads, 1)
    append_bulk_kernel(const Params p, const __grid_constant__ CUtensorMap map_kn, const __grid_constant__ CUtensorMap map_vn,
                       const __grid_constant__ CUtensorMap map_kc, const __grid_constant__ CUtensorMap map_vc,
                       const int* __restrict__ n_new, int max_new) {
  constexpr int D = kAbD, kAbGroup = kAbGroupOf<PARTS>;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kAbBars);   // TMA -> everybody
  uint64_t* empty = full + kAbStages;                             // everybody -> TMA
  uint64_t* phi_ready = empty + kAbStages;                        // [2] transform -> MMA
  uint64_t* phi_empty = phi_ready + 2;                            // [2] MMA -> transform
  uint64_t* acc_full = phi_empty + 2;                             // [2] MMA -> drain: a group's accumulator is complete
  uint64_t* acc_empty = acc_full + 2;                             // [2] drain -> MMA: it may be overwritten
  uint64_t* done = acc_empty + 2;                                 // every product issued has completed
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(smem + kAbMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kAbMisc + 4);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wg = warp >> 2;
  const int u = blockIdx.y, b = u / p.Hkv;
  const int share = blockIdx.x, S = gridDim.x;
  const bool rla = !(p.flags & 4u);

  if (tid == 0) {
    for (int s = 0; s < kAbStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], rla ? 10 : 9); }   // store 1, phi 4, statistics 4, MMA 1
    for (int s = 0; s < 2; ++s) {
      mbar_init(&phi_ready[s], 4); mbar_init(&phi_empty[s], 1); mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 8);
    }
    mbar_init(done, 1);
    mbar_init_done();
    *abort_flag = 0;
  }
  if (warp == 1 && rla) tmem_alloc(tmem_base_s, kAbTmemCols);
  pdl_wait();                                            // the preceding kernels still read the cache and the lengths
  const int L = p.seq_lens[b];
  int n = n_new ? n_new[b] : max_new;
  n = max(0, min(n, max_new));
  if (L < 0 || L + n > p.max_context) {                  // would overflow (or a corrupt length): this sequence is skipped
    n = 0;
    if (share == 0 && tid == 0) atomicExch(p.status, kStatusCapacity);
  }
  tc_fence_before();
  // Every CTA works from the length it read above; once all have theirs (this barrier consumes each thread's value), the
  // last one to check in stores the new lengths: nothing in this launch reads them again.
  __syncthreads_or(L == -1);
  tc_fence_after();
  auto check_in = [&]() {                                // one warp
    int t = 0;
    if (lane == 0) t = atomicAdd(p.append_ticket, 1);
    if (__shfl_sync(0xffffffffu, t, 0) != (int)(gridDim.x * gridDim.y) - 1) return;
    if (lane == 0) *p.append_ticket = 0;
    for (int bb = lane; bb < p.batch; bb += 32) {
      const int Lb = p.seq_lens[bb];
      int nb = n_new ? n_new[bb] : max_new;
      nb = max(0, min(nb, max_new));
      if (Lb >= 0 && Lb + nb <= p.max_context) p.seq_lens[bb] = Lb + nb;
    }
  };

  const int gran = p.B > kAbTile ? p.B / kAbTile : 1;    // tiles per block where a block is more than a tile
  const int g0 = L / (kAbTile * gran), g1 = n > 0 ? (L + n - 1) / (kAbTile * gran) + 1 : g0;
  const int per = (g1 - g0 + S - 1) / S;
  const int my_g0 = min(g1, g0 + share * per), my_g1 = min(g1, my_g0 + per);
  const int tile0 = my_g0 * gran;
  const int tile1 = min(my_g1 * gran, (L + n + kAbTile - 1) / kAbTile);
  const int n_tiles = max(0, tile1 - tile0);
  const size_t unit_tok0 = (size_t)u * p.max_blocks * p.B;
  auto whole = [&](int i) { const int t0 = (tile0 + i) * kAbTile; return t0 >= L && t0 + kAbTile <= L + n; };   // every row is new
  const uint32_t sbase = smem_u32(smem);
  const uint32_t tmem = rla ? *tmem_base_s : 0u;
  const int lim = p.wait_limit;

  if (n_tiles > 0) {
    if (wg == 0) {
      warpgroup_reg_dec<64>();
      if (warp == 0 && lane == 0) {
        // -------------------------------------------------------------- loads -----------------------------------------
        int issued = 0;
        for (int i = 0; i < n_tiles && !*abort_flag; ++i) {
          const int s = i % kAbStages;
          if (i >= kAbStages && !mbar_wait(&empty[s], ((i / kAbStages) - 1) & 1, lim)) { *abort_flag = 1; break; }
          const uint32_t base = sbase + s * 2 * kAbTileBytes;
          const int row = (int)((long long)u * max_new + ((tile0 + i) * kAbTile - L));   // (rows that are not new: of a neighbour, or zeros)
          mbar_expect_tx(&full[s], 2 * kAbTileBytes + (uint32_t)p.dbg_tx_extra);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            tma_load_box(base + h * kAbHalf, &map_kn, h * 64, row, &full[s]);
            tma_load_box(base + kAbTileBytes + h * kAbHalf, &map_vn, h * 64, row, &full[s]);
          }
          issued = i + 1;
        }
        // every copy has landed before the CTA leaves, whatever the other roles do
        for (int j = max(0, issued - kAbStages); j < issued; ++j) mbar_wait(&full[j % kAbStages], (j / kAbStages) & 1, lim);
      } else if (warp == 1 && rla) {
        // -------------------------------------------------------------- products (whole warp, one lane issues) ---------
        const uint32_t one = elect_one();
        bool ok = true;
#pragma unroll 1
        for (int i = 0; i < n_tiles && ok; ++i) {
          const int s = i % kAbStages, pb = i & 1;
          const int g = i / kAbGroup, ab = g & 1;
          const bool first = i % kAbGroup == 0, last = i % kAbGroup == kAbGroup - 1 || i == n_tiles - 1;
          if (first && g >= 2 && !warp_waits(&acc_empty[ab], ((g >> 1) - 1) & 1, lim)) { ok = false; break; }
          if (!warp_waits(&phi_ready[pb], (i >> 1) & 1, lim)) { ok = false; break; }   // (the tile itself arrived before that)
          tc_fence_after();
          const uint32_t a = umma_desc_lo(sbase + kAbPhi + pb * PARTS * kAbTileBytes, kAbHalf);
          const uint32_t v = umma_desc_lo(sbase + s * 2 * kAbTileBytes + kAbTileBytes, kAbHalf);
#pragma unroll
          for (int x = 0; x < PARTS; ++x) {           // 16 tokens (two swizzle atoms of 8 rows) per instruction
            const int part = PARTS == 3 ? PARTS - 1 - x : x;   // (small terms first)
            umma_ss4_one<2048 / 16, 2048 / 16>(one, tmem + ab * D, a + part * (kAbTileBytes / 16), v, kAbIdesc, !first || x > 0);
          }
          umma_commit_one(one, &phi_empty[pb]);
          umma_commit_one(one, &empty[s]);
          if (last) umma_commit_one(one, &acc_full[ab]);
        }
        umma_commit_one(one, done);                      // nothing in flight when tensor memory is released, on expiry of a wait too
        if (!warp_waits(done, 0, lim)) ok = false;
        if (!ok) *abort_flag = 1;
      } else if (warp == 2 && lane == 0) {
        // -------------------------------------------------------------- whole tiles into the cache --------------------
        bool ok = true;
        for (int i = 0; i < n_tiles && !*abort_flag; ++i) {
          const int s = i % kAbStages;
          if (!mbar_wait(&full[s], (i / kAbStages) & 1, lim)) { ok = false; break; }
          int row = (int)(unit_tok0 + (size_t)(tile0 + i) * kAbTile);
          bool store = whole(i);
          if ((p.flags & kDebugBounds) && store && (tile0 + i + 1) * kAbTile > p.max_blocks * p.B) {   // checked build
            atomicExch(p.status, kStatusBounds);
            store = false;
          }
          if (store) {
            const uint32_t base = sbase + s * 2 * kAbTileBytes;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              tma_store_box(&map_kc, h * 64, row, base + h * kAbHalf);
              tma_store_box(&map_vc, h * 64, row, base + kAbTileBytes + h * kAbHalf);
            }
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          if (i > 0) {                                   // the tile before has been read: its place may be refilled
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            mbar_arrive1(&empty[(i - 1) % kAbStages]);
          }
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        if (!ok) *abort_flag = 1;
      } else if (warp == 3) {
        check_in();
      }
    } else if (wg < 3) {
      // ---------------------------------------------------------------- log-sum-exp and phi(k); drain ------------------
      // Thread tg of a group owns the 16-byte pieces tg, tg + 128, ... of a tile (no bank conflicts): rows r0 + 16 k, one
      // piece of either half; the eight lanes of a row hold all its channels.  The swizzle moves pieces only inside their
      // 128-byte row: lane l holds channels 8 (l ^ row) .. + 7 (mod 64) of both halves.
      warpgroup_reg_inc<176>();
      const int wt = wg - 1, tg = (tid - 128) & 127;
      const int r0 = tg >> 3;
      const int ch = (tg & 7) ^ (r0 & 7);                // logical 16-byte piece (rows r0 + 16 k agree in row & 7)
      const float a2 = p.phi_scale * kLog2e;
      bool ok = true;
      const int q = warp & 3;                            // drain: rows 32 q + lane of the accumulator, columns 64 wt .. + 63
      const int n_groups = (n_tiles + kAbGroup - 1) / kAbGroup;
      int drained = 0;
      float acc[64];
#pragma unroll
      for (int x = 0; x < 64; ++x) acc[x] = 0.f;
#pragma unroll 1
      for (int i = wt; ; i += 2) {
        const bool more = i < n_tiles;
        if (more) {
          const int s = i % kAbStages;
          const int t0 = (tile0 + i) * kAbTile;
          const bool edge = !whole(i);
          if (!warp_waits(&full[s], (i / kAbStages) & 1, lim)) { ok = false; break; }
          if (rla && i >= 2 && !warp_waits(&phi_empty[wt], ((i >> 1) - 1) & 1, lim)) { ok = false; break; }
          unsigned char* kt = smem + s * 2 * kAbTileBytes + tg * 16;
          unsigned char* ph = smem + kAbPhi + wt * PARTS * kAbTileBytes + tg * 16;
#pragma unroll 1
          for (int kk = 0; kk < 4; kk += kAbRows, kt += kAbRows * 2048, ph += kAbRows * 2048) {
          // (rows side by side: every step is a chain of latencies; the loop is rolled because the roles' code competes for the
          // instruction cache: with all four rows unrolled its next level was 91 % busy)
          float mx[kAbRows], e[kAbRows][2][8], sum[kAbRows];
#pragma unroll
          for (int k = 0; k < kAbRows; ++k) {
            uint4 raw[2];
            __nv_bfloat162 m[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              raw[h] = *reinterpret_cast<const uint4*>(kt + k * 2048 + h * kAbHalf);
              const __nv_bfloat162* w = reinterpret_cast<const __nv_bfloat162*>(&raw[h]);
              m[h] = __hmax2(__hmax2(w[0], w[1]), __hmax2(w[2], w[3]));
              const uint32_t x[4] = {raw[h].x, raw[h].y, raw[h].z, raw[h].w};
#pragma unroll
              for (int y = 0; y < 4; ++y) { e[k][h][2 * y] = bf16_lo(x[y]); e[k][h][2 * y + 1] = bf16_hi(x[y]); }
            }
            m[0] = __hmax2(m[0], m[1]);
            mx[k] = fmaxf(__low2float(m[0]), __high2float(m[0]));
          }
#pragma unroll
          for (int o = 1; o < 8; o <<= 1)
#pragma unroll
            for (int k = 0; k < kAbRows; ++k) mx[k] = fmaxf(mx[k], __shfl_xor_sync(0xffffffffu, mx[k], o));
          {
            float2 sq[kAbRows];                                // sums of the two quads of a piece, over both halves
#pragma unroll
            for (int k = 0; k < kAbRows; ++k) {
              mx[k] = __fmul_rn(mx[k], a2);
              float2 quad[2];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int x = 0; x < 8; x += 2) {
                  const float2 a = __ffma2_rn(make_float2(e[k][h][x], e[k][h][x + 1]), make_float2(a2, a2), make_float2(-mx[k], -mx[k]));
                  e[k][h][x] = ex2(a.x);
                  e[k][h][x + 1] = ex2(a.y);
                }
                quad[h] = make_float2(e[k][h][0], e[k][h][4]);
#pragma unroll
                for (int x = 1; x < 4; ++x) quad[h] = __fadd2_rn(quad[h], make_float2(e[k][h][x], e[k][h][4 + x]));
              }
              // (the order in which the warp-per-token kernels sum: channels + 64, + 32, + 16, + 8, + 4)
              sq[k] = __fadd2_rn(quad[0], quad[1]);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
#pragma unroll
              for (int k = 0; k < kAbRows; ++k) {
                const float2 other = make_float2(__shfl_xor_sync(0xffffffffu, sq[k].x, o), __shfl_xor_sync(0xffffffffu, sq[k].y, o));
                sq[k] = __fadd2_rn(sq[k], other);
              }
#pragma unroll
            for (int k = 0; k < kAbRows; ++k) sum[k] = sq[k].x + sq[k].y;
          }
          {                                              // the first lanes of a row's eight write one row's log-sum-exp each
            const int k = tg & 7;
            float m = mx[0], sm = sum[0];
#pragma unroll
            for (int x = 1; x < kAbRows; ++x)
              if (k == x) { m = mx[x]; sm = sum[x]; }
            const int pos = t0 + r0 + 16 * (kk + k);
            if (k < kAbRows && pos >= L && pos < L + n) p.tok_lse[unit_tok0 + pos] = lse_from_base2(m, sm);
          }
          if (edge) {
#pragma unroll 1
            for (int k = 0; k < kAbRows; ++k) {
              const int pos = t0 + r0 + 16 * (kk + k);
              const bool valid = pos >= L && pos < L + n;
              const size_t off = (unit_tok0 + pos) * (D / 8) + ch;
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint4* kp = reinterpret_cast<uint4*>(kt + k * 2048 + h * kAbHalf);
                uint4* vp = reinterpret_cast<uint4*>(kt + kAbTileBytes + k * 2048 + h * kAbHalf);
                if (valid) {
                  reinterpret_cast<uint4*>(p.k_cache)[off + 8 * h] = *kp;
                  reinterpret_cast<uint4*>(p.v_cache)[off + 8 * h] = *vp;
                } else if (rla) {
                  *vp = make_uint4(0u, 0u, 0u, 0u);      // V of a row that is not a new token
                }
              }
              if (!valid) {                              // (what such a row holds may be anything)
#pragma unroll
                for (int x = 0; x < kAbRows; ++x) if (x == k) sum[x] = INFINITY;
              }
            }
          }
          if (rla) {
#pragma unroll
            for (int k = 0; k < kAbRows; ++k) {
              float inv;
              asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(sum[k]));
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t part[PARTS][4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                  float2 f = __fmul2_rn(make_float2(e[k][h][2 * x], e[k][h][2 * x + 1]), make_float2(inv, inv));
                  if (edge && inv == 0.f) f = make_float2(0.f, 0.f);
                  if constexpr (PARTS == 2) {
                    part[0][x] = pack_bf16(f.x, f.y);
                    f = __fadd2_rn(f, make_float2(-bf16_lo(part[0][x]), -bf16_hi(part[0][x])));
                    part[1][x] = pack_bf16(f.x, f.y);
                  } else {                               // 8 bits each, cut off: exact remainders
#pragma unroll
                    for (int pt = 0; pt < PARTS; ++pt) {
                      const uint32_t lo = __float_as_uint(f.x), hi = __float_as_uint(f.y);
                      part[pt][x] = __byte_perm(lo, hi, 0x7632);
                      if (pt + 1 < PARTS)
                        f = __fadd2_rn(f, make_float2(-__uint_as_float(lo & 0xffff0000u), -__uint_as_float(hi & 0xffff0000u)));
                    }
                  }
                }
#pragma unroll
                for (int pt = 0; pt < PARTS; ++pt)
                  *reinterpret_cast<uint4*>(ph + pt * kAbTileBytes + k * 2048 + h * kAbHalf) =
                      make_uint4(part[pt][0], part[pt][1], part[pt][2], part[pt][3]);
              }
            }
          }
          }
          proxy_fence();                                 // generic writes -> the tensor core's reads; reads -> the next copy
          __syncwarp();
          if (lane == 0) {
            if (rla) mbar_arrive1(&phi_ready[wt]);
            mbar_arrive1(&empty[s]);
          }
        }
        if (!rla) { if (more) continue; break; }
        // one accumulator group behind the issuer: by now those instructions have long completed
        const int upto = more ? i / kAbGroup : n_groups;
#pragma unroll 1
        for (; drained < upto && ok; ++drained) {
          if (!warp_waits(&acc_full[drained & 1], (drained >> 1) & 1, lim)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int cb = 0; cb < 2; ++cb) {
            float v[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((drained & 1) * D + wt * 64 + cb * 32), v);
#pragma unroll
            for (int x = 0; x < 32; ++x) acc[cb * 32 + x] += v[x];
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive1(&acc_empty[drained & 1]);
        }
        if (!more || !ok) break;
      }
      if (!ok) *abort_flag = 1;
      if (rla && ok && !warp_aborted(abort_flag)) {
        float* dst = (S > 1 ? p.state_part + ((size_t)u * S + share) * D * D : p.state + (size_t)u * D * D) + (size_t)(q * 32 + lane) * D + wt * 64;
        if (S == 1) {                                    // (all loads before the first use: one at a time they took 17000 cycles)
          float4 old[16];
#pragma unroll
          for (int x = 0; x < 16; ++x) old[x] = reinterpret_cast<const float4*>(dst)[x];
#pragma unroll
          for (int x = 0; x < 16; ++x) { acc[4 * x] += old[x].x; acc[4 * x + 1] += old[x].y; acc[4 * x + 2] += old[x].z; acc[4 * x + 3] += old[x].w; }
        }
#pragma unroll
        for (int x = 0; x < 64; x += 4) *reinterpret_cast<float4*>(dst + x) = make_float4(acc[x], acc[x + 1], acc[x + 2], acc[x + 3]);
      }
    } else {
      // ---------------------------------------------------------------- block statistics ------------------------------
      // Thread (parity, channel pair): every second token of a block (or window) in order, both parities' sums added in
      // order: what block_stats_core of the other append kernels computes, bit for bit.
      warpgroup_reg_dec<96>();
      const int st = tid - 384, par = st >> 6, cp = st & 63;
      float* red = reinterpret_cast<float*>(smem + kAbRed);            // [2][2][D]
      const uint32_t col = (uint32_t)((cp >> 5) * kAbHalf + (cp & 3) * 4);
      const int piece = (cp & 31) >> 2;
      const bool r16 = (p.flags & kStatsBf16) != 0;
      auto meet = [&]() { asm volatile("bar.sync 3, 128;" ::: "memory"); };
      bool ok = true;
#pragma unroll 1
      for (int i = 0; i < n_tiles; i += gran) {
        bool go = true;
        const int have = min(gran, n_tiles - i);
        for (int j = 0; j < have && go; ++j) go = warp_waits(&full[(i + j) % kAbStages], ((i + j) / kAbStages) & 1, lim);
        uint32_t stop;                                                 // one decision for the four warps: barrier counts must match
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.ne.u32 q, %1, 0;\n\t"
            "bar.red.or.pred p, 3, 128, q;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(stop) : "r"(go ? 0u : 1u) : "memory");
        if (stop) { ok = false; break; }
        const unsigned char* k0 = smem + (i % kAbStages) * 2 * kAbTileBytes;
        const unsigned char* k1 = smem + ((i + 1) % kAbStages) * 2 * kAbTileBytes;
        const int t0 = (tile0 + i) * kAbTile;                          // first token here
        const int t_end = min(t0 + have * kAbTile, L + n);
        const int blk0 = max(L, t0) / p.B;                             // first block that changes
        if (blk0 * p.B < L) {                                          // its older tokens come from the cache (once per unit)
          for (int x = st; x < (min(L, t_end) - blk0 * p.B) * (D / 8); x += 128) {
            const int pos = blk0 * p.B + x / (D / 8), c8 = x % (D / 8), rr = pos - t0;
            unsigned char* kd = const_cast<unsigned char*>(rr >= kAbTile ? k1 : k0);
            *reinterpret_cast<uint4*>(kd + (c8 >> 3) * kAbHalf + (rr & 63) * 128 + (((c8 & 7) ^ (rr & 7)) << 4)) =
                reinterpret_cast<const uint4*>(p.k_cache)[(unit_tok0 + pos) * (D / 8) + c8];
          }
          meet();
        }
        auto key2 = [&](int rr) -> float2 {                            // both channels of row rr of the tile (pair)
          const unsigned char* kd = rr >= kAbTile ? k1 : k0;
          const uint32_t w = *reinterpret_cast<const uint32_t*>(kd + col + (rr & 63) * 128 + ((piece ^ (rr & 7)) << 4));
          return make_float2(bf16_lo(w), bf16_hi(w));
        };
        if (p.B == kAbTile && p.NW == 1 && t_end - t0 == kAbTile && !(p.flags & kDebugBounds)) {
          // a whole block of 64, the common case: addresses are a pointer and four offsets (with the general loop below this
          // role took 4700 cycles per tile and bounded the kernel)
          const unsigned char* kb = k0 + col + par * 128;
          uint32_t off[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) off[j] = (uint32_t)(j * 256 + ((piece ^ (par + 2 * j)) << 4));
          float2 sum = make_float2(0.f, 0.f);
#pragma unroll 2
          for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t w = *reinterpret_cast<const uint32_t*>(kb + t * 1024 + off[j]);
              sum = __fadd2_rn(sum, make_float2(bf16_lo(w), bf16_hi(w)));
            }
          *reinterpret_cast<float2*>(red + par * D + 2 * cp) = sum;
          meet();
          const float2 s0 = *reinterpret_cast<const float2*>(red + 2 * cp), s1 = *reinterpret_cast<const float2*>(red + D + 2 * cp);
          const float2 mean = __fmul2_rn(__fadd2_rn(s0, s1), make_float2(1.f / kAbTile, 1.f / kAbTile));   // (a power of two: the same as dividing)
          float2 ss = make_float2(0.f, 0.f);
#pragma unroll 2
          for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t w = *reinterpret_cast<const uint32_t*>(kb + t * 1024 + off[j]);
              const float2 dv = __fadd2_rn(make_float2(bf16_lo(w), bf16_hi(w)), make_float2(-mean.x, -mean.y));
              ss = __ffma2_rn(dv, dv, ss);
            }
          *reinterpret_cast<float2*>(red + 2 * D + par * D + 2 * cp) = ss;
          meet();
          float2 val = mean;
          if (par == 1) {
            const float2 q0 = *reinterpret_cast<const float2*>(red + 2 * D + 2 * cp), q1 = *reinterpret_cast<const float2*>(red + 3 * D + 2 * cp);
            val = __fmul2_rn(__fadd2_rn(q0, q1), make_float2(1.f / kAbTile, 1.f / kAbTile));
          }
          const size_t rec = ((size_t)u * p.max_blocks + blk0) * 2 * D + par * D + 2 * cp;
          if (r16) *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(p.stats) + rec) = __floats2bfloat162_rn(val.x, val.y);
          else *reinterpret_cast<float2*>(p.stats + rec) = val;
        } else
        for (int blk = blk0; blk * p.B < t_end; ++blk) {
          if ((p.flags & kDebugBounds) && blk >= p.max_blocks) {       // checked build
            if (st == 0) atomicExch(p.status, kStatusBounds);
            break;
          }
          const int held = min(p.B, L + n - blk * p.B), first_row = blk * p.B - t0;
          for (int w = 0; w < p.NW; ++w) {
            const int lo = w * p.win_s, hi = min(held, lo + p.win_C), cnt = hi - lo;
            if (cnt <= 0) break;                                       // (a window that holds no token yet is left alone)
            float2 sum = make_float2(0.f, 0.f);
#pragma unroll 8
            for (int t = lo + par; t < hi; t += 2) sum = __fadd2_rn(sum, key2(first_row + t));
            *reinterpret_cast<float2*>(red + par * D + 2 * cp) = sum;
            meet();
            const float2 s0 = *reinterpret_cast<const float2*>(red + 2 * cp), s1 = *reinterpret_cast<const float2*>(red + D + 2 * cp);
            const float2 mean = make_float2((s0.x + s1.x) / (float)cnt, (s0.y + s1.y) / (float)cnt);
            float2 ss = make_float2(0.f, 0.f);
#pragma unroll 8
            for (int t = lo + par; t < hi; t += 2) {
              const float2 dv = __fadd2_rn(key2(first_row + t), make_float2(-mean.x, -mean.y));
              ss = __ffma2_rn(dv, dv, ss);
            }
            *reinterpret_cast<float2*>(red + 2 * D + par * D + 2 * cp) = ss;
            meet();
            float2 val = mean;                                         // parity 0 writes the mean, parity 1 the variance
            if (par == 1) {
              const float2 q0 = *reinterpret_cast<const float2*>(red + 2 * D + 2 * cp), q1 = *reinterpret_cast<const float2*>(red + 3 * D + 2 * cp);
              val = make_float2((q0.x + q1.x) / (float)cnt, (q0.y + q1.y) / (float)cnt);
            }
            const size_t rec = (((size_t)u * p.max_blocks + blk) * p.NW + w) * 2 * D + par * D + 2 * cp;
            if (r16) *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(p.stats) + rec) = __floats2bfloat162_rn(val.x, val.y);
            else *reinterpret_cast<float2*>(p.stats + rec) = val;
          }
        }
        proxy_fence();                                                 // reads and writes here -> the next copy into these places
        __syncwarp();
        if (lane == 0)
          for (int j = 0; j < have; ++j) mbar_arrive1(&empty[(i + j) % kAbStages]);
      }
      if (!ok) *abort_flag = 1;
    }
  }
  if (n_tiles == 0 && warp == 3) check_in();
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  if (warp == 1 && rla) {
    __syncwarp();
    tc_fence_after();
    tmem_free(tmem, kAbTmemCols);
  }
  if (tid == 0 && *abort_flag) atomicExch(p.status, kStatusTimeout);
  if ((n_tiles == 0 || *abort_flag) && rla && S > 1) {   // an empty share adds nothing, nor does one that gave up (no old sums)
    float4* part = reinterpret_cast<float4*>(p.state_part + ((size_t)u * S + share) * D * D);
    for (int idx = tid; idx < D * D / 4; idx += kAbThreads) part[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Shares of every unit onto S_bar, in share order.
constexpr int kAbMergeThreads = 256;
__global__ void __launch_bounds__(kAbMergeThreads) append_merge_state_kernel(const Params p, int S) {
  const int N4 = p.d * p.d / 4;
  pdl_wait();
  const int idx = blockIdx.x * kAbMergeThreads + threadIdx.x, u = blockIdx.y;
  const float4* part = reinterpret_cast<const float4*>(p.state_part) + (size_t)u * S * N4 + idx;
  float4* st = reinterpret_cast<float4*>(p.state) + (size_t)u * N4 + idx;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f), o = *st;
  for (int s0 = 0; s0 < S; s0 += 16) {
    float4 x[16];
#pragma unroll
    for (int s = 0; s < 16; ++s) x[s] = s0 + s < S ? __ldcg(part + (size_t)(s0 + s) * N4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s = 0; s < 16; ++s) { a.x += x[s].x; a.y += x[s].y; a.z += x[s].z; a.w += x[s].w; }
  }
  o.x += a.x; o.y += a.y; o.z += a.z; o.w += a.w;
  *st = o;
  pdl_launch_dependents();
}

}  // namespace

// Shares of a unit's tokens.  One CTA fits an SM, and per CTA the work is bounded by the roles' latencies, so what counts is
// that all 148 SMs have the same: either one wave, or, where that leaves many SMs idle (32 units: 4 x 32 = 128 CTAs) and
// the shares stay long (16 tiles), two (9 x 32 = 288 of 296 places; 131072 tokens x 32 units as first built: 0.95 -> 0.92 ms).  A fixed SM
// count, because the partial buffer is sized from the configuration alone, before any device is known.
constexpr int kAbMaxShares = 72;
static int shares_in_waves(int units, int waves) {
  const int s = 148 * waves / (units > 0 ? units : 1);
  return s < 1 ? 1 : (s > kAbMaxShares ? kAbMaxShares : s);
}
static int append_bulk_shares(int units, int tiles) {
  const int one = shares_in_waves(units, 1), two = shares_in_waves(units, 2);
  const bool fuller = 100 * two > 210 * one;             // at least 5 % more of the places in use
  const int s = fuller && tiles >= 16 * two ? two : one;
  return s < tiles ? s : tiles;
}

int append_max_shares(int units) { return shares_in_waves(units, 2); }

size_t append_bulk_part_bytes(int units, int d) {
  const int s = append_max_shares(units);
  return s > 1 ? (size_t)units * s * d * d * 4 : 0;
}

cudaError_t launch_append_merge_state(const Params& p, int S, cudaStream_t stream) {
  return launch_ex(append_merge_state_kernel, dim3(p.d * p.d / 4 / kAbMergeThreads, p.batch * p.Hkv), dim3(kAbMergeThreads), 0, stream, 0, true, p, S);
}

// cache: maps of the K / V cache, fresh: of k_new / v_new as [units * max_new][128]; boxes of 64 rows x 64 columns.
cudaError_t launch_append_bulk(const Params& p, const AttendMaps& cache, const AttendMaps& fresh, const int* n_new, int max_new,
                               cudaStream_t stream) {
  const int U = p.batch * p.Hkv;
  const int span = p.B > kAbTile ? p.B : kAbTile;
  const int most = (max_new + span - 2) / span + 1;      // tiles (blocks of 128 tokens) a sequence can touch
  const int S = append_bulk_shares(U, most);
  // the tensor-core state has 16 bits of phi from 256 tokens on; shorter appends keep the fp32 kernels' accuracy
  auto kern = max_new >= kAbTwoParts ? append_bulk_kernel<2> : append_bulk_kernel<3>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kAbSmem);
  if (e != cudaSuccess) return e;
  e = launch_ex(kern, dim3(S, U), dim3(kAbThreads), kAbSmem, stream, 0, true, p,
                *reinterpret_cast<const CUtensorMap*>(fresh.k), *reinterpret_cast<const CUtensorMap*>(fresh.v),
                *reinterpret_cast<const CUtensorMap*>(cache.k), *reinterpret_cast<const CUtensorMap*>(cache.v), n_new, max_new);
  if (e == cudaSuccess && S > 1 && !(p.flags & 4u)) e = launch_append_merge_state(p, S, stream);
  return e;
}

}  // namespace spla
