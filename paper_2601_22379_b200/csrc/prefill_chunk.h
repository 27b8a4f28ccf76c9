// Geometry and buffers of the tensor-core prefill path, shared by its kernels (not part of the public ABI).
#pragma once

#include "spla_internal.h"

namespace spla {

constexpr int kPfRows = 128;             // query rows (positions x heads of the group) of one tile: the M of the tensor-core products
constexpr int kPfMaxBlocks = 16384;      // blocks per sequence the path serves (the tile's bitmap of selected blocks is 2 KB)

// The positions of a chunk are cut at absolute multiples of SB tokens (64, or the block size where that is larger), so
// that a tile's base - the recurrent state before its SB range - is a block boundary; an SB range holds nt tiles of P
// positions each.  Which positions share a tile depends on nothing but their place in the sequence.
struct PrefillChunk {
  int T;                // positions per sequence
  int SB, P, nt;
  int n_sb;             // SB ranges of the chunk, at most; nt row tiles each
  int q0, nq;           // row tiles of this launch ...
  int u0, nu;           // ... and units
  int stride;           // floats per (position, head) row of ell
  float* ell;           // [nu][nq * P][G][stride]  log masses of the complete blocks less ln B, for the positions of this launch
  float* ell_own;       // [U][T][G]                log mass of every position's own, growing block, less ln B
  float* snap;          // [U][n_sb][d][d]          the recurrent state at the start of every SB range (the first: of the chunk)
  int* sel;             // [U][T][top_k]            selected blocks, ascending, padded with -1
};

// The chunk of one unit.  first: absolute position of chunk token 0 (negative only where the append was refused on the
// device: those positions see nothing).
struct PrefillUnit {
  int u, b, h, L_end, first, L0;
};
__device__ __forceinline__ PrefillUnit prefill_unit_of(const Params& p, const PrefillChunk& c, int u) {
  PrefillUnit r;
  r.u = u;
  r.b = u / p.Hkv;
  r.h = u % p.Hkv;
  r.L_end = cover_len(p, checked_len(p, r.b), (long long)c.stride * p.B);   // (what the host sized the launch for)
  r.first = r.L_end - c.T;
  r.L0 = max(0, r.first);
  return r;
}
__device__ __forceinline__ int prefill_range_start(const PrefillChunk& c, const PrefillUnit& r, int i) { return (r.L0 / c.SB + i) * c.SB; }

// SB ranges a chunk of T tokens can touch.
inline int prefill_ranges(int T, int SB) { return (T + SB - 2) / SB + 1; }
inline void prefill_tiling(int G, int B, int* SB, int* P, int* nt) {
  *SB = (B == 128 || G == 1) ? 128 : 64;
  const int cap = kPfRows / G;                    // positions that fit the rows of a tile
  *nt = (*SB + cap - 1) / cap;
  *P = (*SB + *nt - 1) / *nt;
}

// prefill_state.cu
cudaError_t launch_prefill_own(const Params& p, const PrefillChunk& c, const void* q, float* out, int* sel_user, cudaStream_t s);
cudaError_t launch_prefill_state(const Params& p, const PrefillChunk& c, cudaStream_t s);
// prefill_score.cu
cudaError_t launch_prefill_score(const Params& p, const PrefillChunk& c, const void* q, int max_blocks_seen, int sm_count, cudaStream_t s);
cudaError_t launch_prefill_select(const Params& p, const PrefillChunk& c, int max_blocks_seen, int* sel_user, cudaStream_t s);
// prefill_attend.cu
cudaError_t launch_prefill_attend(const Params& p, const PrefillChunk& c, const AttendMaps& maps, const void* q, const float* rms_weight,
                                  float* out, cudaStream_t s);

}  // namespace spla
