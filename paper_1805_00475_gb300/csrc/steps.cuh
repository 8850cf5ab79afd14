// The big steps of a contraction on the CUDA cores: grid-wide steps, steps with
// one small operand, split-K steps; and the extraction of the results.
#pragma once

#include "kernels.cuh"

namespace tnc_dev {

// The residue groups of a pass run side by side: blockIdx.y is the group, with
// its own primes, its own copy of the arena (arena_stride words further) and
// its own split-K partials.  (A formula with 2^24 products or fewer spends most of
// its time between launches; 20 residues in five passes took five times the
// launches.)
constexpr int kMaxGroups = 14;
struct Pass {
  ModGroup mg[kMaxGroups];
  uint64_t arena_stride, part_stride;  // words
};

template <int RG, typename W = uint32_t>
__global__ void __launch_bounds__(256) leaf_fill_kernel(const LeafDesc* __restrict__ leaves, int n_leaves,
                                                        const uint32_t* __restrict__ tables,
                                                        W* __restrict__ arena0, const __grid_constant__ Pass ps) {
  W* __restrict__ arena = arena0 + blockIdx.y * ps.arena_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  for (int l = blockIdx.x; l < n_leaves; l += gridDim.x) {
    const LeafDesc ld = leaves[l];
    const uint64_t n = 1ull << ld.rank;
    W* dst = arena + ld.off * RG;
    for (uint64_t idx = threadIdx.x; idx < n; idx += blockDim.x) {
      uint32_t v[RG];
#pragma unroll
      for (int r = 0; r < RG; r++) v[r] = leaf_value(ld.kind, ld.rank, (uint32_t)idx, tables, ld.table_off, mg.p[r]);
      store_entry<RG, W>(dst + idx * RG, v);
    }
  }
}

// All the small steps of one tree level in one launch: they are independent,
// so their output entries form one index space (step i owns [work_lo,
// work_lo + 2^c)); each thread finds its step by binary search.
template <int RG, typename W = uint32_t, bool N30 = false>
__global__ void __launch_bounds__(256) level_kernel(const StepDesc* __restrict__ steps, uint32_t n_steps,
                                                    uint32_t total, W* arena0, const __grid_constant__ Pass ps) {
  W* arena = arena0 + blockIdx.y * ps.arena_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < total; w += gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = n_steps - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (steps[mid].work_lo <= w) lo = mid;
      else hi = mid - 1;
    }
    const StepDesc& d = steps[lo];
    step_entry<RG, W, N30>(d, w - d.work_lo, arena + d.a_off * RG, arena + d.b_off * RG, arena + d.c_off * RG, mg);
  }
}

// A step launched over the whole GPU.  With S = 2^s threads in the grid, a
// thread visits o, o + S, o + 2S, ...: from one to the next the counter o >> s
// gains one, which clears its trailing ones and sets bit t, so each operand
// address changes by the precomputed delta[t] = w[t] - sum_{s <= j < t} w[j]
// (w[j] = operand weight of output bit j).  Any bit permutation costs the
// same two adds per entry.
struct GridStep {
  StepDesc d;
  uint64_t wA[32], wB[32];  // operand address weight of output bit j
  uint64_t dA[32], dB[32];  // address delta when the counter sets bit t
  uint16_t s;               // log2(the step's threads)
  uint16_t log_split;       // split-K: log2 of the K slices
  uint32_t block_lo;        // its first block in the launch
  uint32_t final_lo;        // split-K: its first block in the launch that adds the slices
  uint32_t part_off;        // split-K: its first partial (of RG residues)
};

// A launch serves up to all the steps of one kind in a tree level (of every
// plan of a group): their blocks lie side by side, and a block finds its step
// by binary search over the steps' first blocks.  (One launch per step cost
// 4 to 8 us each on steps of a few us; 48 plans of uneven 1-in-3 formulas had
// 136 + 98 pairs of them.)
template <uint32_t GridStep::*LO>
__device__ __forceinline__ const GridStep* step_of_block(const GridStep* steps, uint32_t n) {
  uint32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (steps[mid].*LO <= blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  return steps + lo;
}

template <int RG, typename W = uint32_t, bool N30 = false>
__global__ void __launch_bounds__(256) step_kernel(const GridStep* __restrict__ steps, uint32_t n_steps,
                                                   W* __restrict__ arena0, const __grid_constant__ Pass ps) {
  W* __restrict__ arena = arena0 + blockIdx.y * ps.arena_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  const GridStep* __restrict__ g = step_of_block<&GridStep::block_lo>(steps, n_steps);
  const uint32_t c = g->d.c, k = g->d.k, ka = g->d.ka, kb = g->d.kb, s = g->s;
  const uint64_t n = 1ull << c;
  const W* A0 = arena + g->d.a_off * RG;
  const W* B0 = arena + g->d.b_off * RG;
  W* C0 = arena + g->d.c_off * RG;
  uint64_t o = (uint64_t)(blockIdx.x - g->block_lo) * blockDim.x + threadIdx.x;
  if (o >= n) return;
  uint64_t ia = 0, ib = 0;
  for (uint32_t j = 0; j < c; j++)
    if ((o >> j) & 1ull) {
      ia += g->wA[j];
      ib += g->wB[j];
    }
  for (;;) {
    step_entry_at<RG, W, N30>(k, ka, kb, o, ia, ib, A0, B0, C0, mg);
    const uint64_t u = o >> s;
    o += 1ull << s;
    if (o >= n) break;
    const uint32_t t = s + (uint32_t)(__ffsll((long long)~u) - 1);
    ia += g->dA[t];
    ib += g->dB[t];
  }
}

// The bigger of these steps in register tiles: a thread computes 2^kTileA rows
// x 2^kTileB columns of outputs (the operands' highest free bits), so each
// operand entry it loads serves several products.  The other output bits are
// walked as in step_kernel, with the output's address by deltas too.  (Byte
// residues, 10 launches of a cubic VC formula with n = 180: 111 -> 78 us; u32
// residues, 2^20 outputs: 9.6 -> 7.4 us.  4 x 4 outputs: no faster on these, and the dense
// steps it would help run in shared-memory tiles.)
constexpr int kTileA = 1, kTileB = 1;
struct TileStep {
  uint64_t a_off, b_off, c_off;
  uint32_t wA[32], wB[32], wC[32];  // address weights of the bits walked
  uint32_t dA[32], dB[32], dC[32];  // address deltas when the counter sets bit t
  uint32_t tA[1 << kTileA], cA[1 << kTileA];  // operand and output offsets of the tile's rows
  uint32_t tB[1 << kTileB], cB[1 << kTileB];  // and columns
  uint32_t n_bits, block_lo;        // bits walked; first block in the launch
  uint8_t k, ka, kb, s;             // 2^s threads
  uint32_t pad;
};

template <int RG, typename W = uint32_t, bool N30 = false>
__global__ void __launch_bounds__(256) tile_kernel(const TileStep* __restrict__ steps, uint32_t n_steps,
                                                   W* __restrict__ arena0, const __grid_constant__ Pass ps) {
  W* __restrict__ arena = arena0 + blockIdx.y * ps.arena_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  uint32_t lo = 0, hi = n_steps - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (steps[mid].block_lo <= blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const TileStep* __restrict__ g = steps + lo;
  constexpr int NA = 1 << kTileA, NB = 1 << kTileB;
  using Acc = std::conditional_t<sizeof(W) == 1, uint32_t, uint64_t>;
  const uint32_t s = g->s, K = 1u << g->k;
  const uint64_t n = 1ull << g->n_bits;
  const uint64_t sa = (uint64_t)RG << g->ka, sb = (uint64_t)RG << g->kb;
  uint64_t t = (uint64_t)(blockIdx.x - g->block_lo) * blockDim.x + threadIdx.x;
  if (t >= n) return;
  uint32_t ia = 0, ib = 0, ic = 0;
  for (uint32_t j = 0; j < g->n_bits; j++)
    if ((t >> j) & 1ull) {
      ia += g->wA[j];
      ib += g->wB[j];
      ic += g->wC[j];
    }
  uint64_t oa[NA], ob[NB];
#pragma unroll
  for (int i = 0; i < NA; i++) oa[i] = (uint64_t)g->tA[i] * RG;
#pragma unroll
  for (int i = 0; i < NB; i++) ob[i] = (uint64_t)g->tB[i] * RG;
  for (;;) {
    const W* A = arena + (g->a_off + ia) * RG;
    const W* B = arena + (g->b_off + ib) * RG;
    Acc acc[NA][NB][RG];
#pragma unroll
    for (int i = 0; i < NA; i++)
#pragma unroll
      for (int j = 0; j < NB; j++)
#pragma unroll
        for (int r = 0; r < RG; r++) acc[i][j][r] = 0;
    auto product = [&] {
      uint32_t va[NA][RG], vb[NB][RG];
#pragma unroll
      for (int i = 0; i < NA; i++) load_entry<RG, W>(A + oa[i], va[i]);
#pragma unroll
      for (int j = 0; j < NB; j++) load_entry<RG, W>(B + ob[j], vb[j]);
      A += sa;
      B += sb;
#pragma unroll
      for (int i = 0; i < NA; i++)
#pragma unroll
        for (int j = 0; j < NB; j++)
#pragma unroll
          for (int r = 0; r < RG; r++) acc[i][j][r] += (Acc)va[i][r] * vb[j][r];
    };
    uint32_t q = 0;
#pragma unroll 1
    for (; q + 4 <= K; q += 4) {
#pragma unroll
      for (int u = 0; u < 4; u++) product();
      if (((q + 4) & mg.red_mask) == 0) {
#pragma unroll
        for (int i = 0; i < NA; i++)
#pragma unroll
          for (int j = 0; j < NB; j++)
#pragma unroll
            for (int r = 0; r < RG; r++) acc[i][j][r] = reduce_acc<N30>(acc[i][j][r], mg, r);
      }
    }
    for (; q < K; q++) product();  // K < 4
    W* C = arena + (g->c_off + ic) * RG;
#pragma unroll
    for (int i = 0; i < NA; i++)
#pragma unroll
      for (int j = 0; j < NB; j++) {
        uint32_t out[RG];
#pragma unroll
        for (int r = 0; r < RG; r++) out[r] = reduce_acc<N30>(acc[i][j][r], mg, r);
        store_entry<RG, W>(C + (uint64_t)(g->cA[i] + g->cB[j]) * RG, out);
      }
    const uint64_t u = t >> s;
    t += 1ull << s;
    if (t >= n) break;
    const uint32_t b = s + (uint32_t)(__ffsll((long long)~u) - 1);
    ia += g->dA[b];
    ib += g->dB[b];
    ic += g->dC[b];
  }
}

// The densest of these steps (u32 residues) in shared-memory tiles, as a
// modular matrix product: a CTA computes 2^LA rows x 2^LB columns, staging 16
// shared values of its rows and columns at a time (cp.async, three stages,
// running on across its tiles), a thread 2^RA x 2^RB of the outputs.  Without
// the staging every warp reads its operands from L2 (about 7 TB/s at 2^21
// outputs of 512 products, which is what bounds step_kernel there), and with
// 2^16 outputs a thread per output leaves most of each SM idle.  A tile's
// output bits other than the thread's own (the rows' RA highest, the columns'
// RB highest) go to lanes and warps by output weight, lightest first, so that a
// warp's stores are as close together as the step's bit map allows.
// Bound by the 64-bit multiply-adds: 2^21 outputs of 512 products, 4 residues,
// 1190 -> 724 us = 5.9e12 products/s, the rate of the bare primitive
// (tnc_probe_modmac 5.8e12); the 16 shared values of a stage fully unrolled (by 4:
// 908 us, by 8: 823) at two CTAs per SM.  2^24 outputs of 16 products: 474 ->
// 216 us; 2^16 outputs of 256 products, 2 residues of wide primes: 34 -> 17 us.
constexpr int kBlkK = 16, kBlkStages = 3;
// Shapes by the step's outputs: 64 x 32 (4 x 2 a thread) from 2^19 on, 32 x 32
// (2 x 2) from 2^17 on, 32 x 16 (2 x 1) at 2^16: at least 128 tiles.
template <int SHAPE>
struct Blk {
  static constexpr int LA = SHAPE == 0 ? 6 : 5, LB = SHAPE == 2 ? 4 : 5, RA = SHAPE == 0 ? 2 : 1, RB = SHAPE == 2 ? 0 : 1;
};
// A thread's operand entries of one shared value: its N rows (or columns) of the
// staged ones at s, `apart` entries from one to the next.  (A host function too:
// its bounds are checked there.)
template <int N, int RG>
__host__ __device__ __forceinline__ void load_rows(const uint32_t* s, uint32_t apart, uint32_t (&v)[N][RG]) {
#pragma unroll
  for (int i = 0; i < N; i++) {
    const uint32_t* e = s + i * apart * RG;
    if constexpr (RG == 4) {
      const uint4 t = *reinterpret_cast<const uint4*>(e);
      v[i][0] = t.x; v[i][1] = t.y; v[i][2] = t.z; v[i][3] = t.w;
    } else if constexpr (RG == 2) {
      const uint2 t = *reinterpret_cast<const uint2*>(e);
      v[i][0] = t.x; v[i][1] = t.y;
    } else {
      v[i][0] = *e;
    }
  }
}

struct BlockStep {
  uint64_t a_off, b_off, c_off;
  uint32_t wA[32], wB[32];  // output weight of row bit j / column bit j
  uint8_t bit[8];           // thread bit i: column bit j (0x80 | j) or row bit j
  uint32_t k, ka, kb, tile_lo;
};

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

template <int RG, int SHAPE, bool N30 = false>
__global__ void __launch_bounds__(256, 2) block_kernel(const BlockStep* __restrict__ steps, uint32_t n_steps,
                                                       uint32_t n_tiles, uint32_t* __restrict__ arena0,
                                                       const __grid_constant__ Pass ps) {
  uint32_t* __restrict__ arena = arena0 + blockIdx.y * ps.arena_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  constexpr int kBlkA = Blk<SHAPE>::LA, kBlkB = Blk<SHAPE>::LB, RA = Blk<SHAPE>::RA, RB = Blk<SHAPE>::RB;
  constexpr int TA = 1 << RA, TB = 1 << RB;
  constexpr uint32_t NA = 1u << kBlkA, NB = 1u << kBlkB, kStage = (NA + NB) * kBlkK * RG;  // words
  extern __shared__ __align__(16) uint32_t sm[];
  const uint32_t tid = threadIdx.x;
  auto step_of = [&](uint32_t tile) {
    uint32_t lo = 0, hi = n_steps - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (steps[mid].tile_lo <= tile) lo = mid;
      else hi = mid - 1;
    }
    return steps + lo;
  };
  // the loader runs kBlkStages - 1 chunks ahead of the products
  uint32_t l_tile = blockIdx.x, l_chunk = 0, l_n = 0, l_slot = 0;
  const uint32_t *l_a = nullptr, *l_b = nullptr;
  uint64_t l_sa = 0, l_sb = 0;
  auto load_next = [&] {
    if (l_tile < n_tiles) {
      if (l_chunk == 0) {
        const BlockStep* g = step_of(l_tile);
        const uint32_t t = l_tile - g->tile_lo, ta = t & ((1u << (g->ka - kBlkA)) - 1u), tb = t >> (g->ka - kBlkA);
        l_n = 1u << (g->k - 4);
        l_sa = (uint64_t)RG << g->ka;
        l_sb = (uint64_t)RG << g->kb;
        l_a = arena + (g->a_off + ((uint64_t)ta << kBlkA)) * RG;
        l_b = arena + (g->b_off + ((uint64_t)tb << kBlkB)) * RG;
      }
      uint32_t* dst = sm + l_slot * kStage;
#pragma unroll
      for (uint32_t i = 0; i < NA * kBlkK / 256; i++) {
        const uint32_t e = tid + 256 * i, q = e >> kBlkA, row = e & (NA - 1);
        cp_async<4 * RG>(dst + e * RG, l_a + q * l_sa + row * RG);
      }
#pragma unroll
      for (uint32_t i = 0; i < NB * kBlkK / 256; i++) {  // (at least one)
        const uint32_t e = tid + 256 * i, q = e >> kBlkB, col = e & (NB - 1);
        cp_async<4 * RG>(dst + (NA * kBlkK + e) * RG, l_b + q * l_sb + col * RG);
      }
      l_a += kBlkK * l_sa;
      l_b += kBlkK * l_sb;
      if (++l_slot == kBlkStages) l_slot = 0;
      if (++l_chunk == l_n) {
        l_chunk = 0;
        l_tile += gridDim.x;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int i = 0; i < kBlkStages - 1; i++) load_next();
  uint32_t slot = 0;
  const BlockStep* cur = nullptr;
  uint32_t row = 0, col = 0, off = 0;
  for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const BlockStep* g = step_of(tile);
    if (g != cur) {  // this thread's place in a tile of the step
      cur = g;
      row = col = off = 0;
#pragma unroll
      for (int i = 0; i < 8; i++)
        if ((tid >> i) & 1u) {
          const uint32_t b = g->bit[i];
          if (b & 0x80u) {
            col |= 1u << (b & 31u);
            off += g->wB[b & 31u];
          } else {
            row |= 1u << b;
            off += g->wA[b];
          }
        }
    }
    uint64_t acc[TA][TB][RG];
#pragma unroll
    for (int i = 0; i < TA; i++)
#pragma unroll
      for (int j = 0; j < TB; j++)
#pragma unroll
        for (int r = 0; r < RG; r++) acc[i][j][r] = 0;
    const uint32_t chunks = 1u << (g->k - 4);
    for (uint32_t c = 0; c < chunks; c++) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kBlkStages - 2) : "memory");
      __syncthreads();  // the chunk has landed for every thread, and the slot that is loaded next is free
      load_next();
      const uint32_t* sa = sm + slot * kStage + row * RG;
      const uint32_t* sb = sm + slot * kStage + (NA * kBlkK + col) * RG;
      if (++slot == kBlkStages) slot = 0;
#pragma unroll 16
      for (uint32_t q = 0; q < kBlkK; q++) {
        uint32_t va[TA][RG], vb[TB][RG];
        load_rows(sa + q * NA * RG, NA / TA, va);
        load_rows(sb + q * NB * RG, NB / TB, vb);
#pragma unroll
        for (int i = 0; i < TA; i++)
#pragma unroll
          for (int j = 0; j < TB; j++)
#pragma unroll
            for (int r = 0; r < RG; r++) acc[i][j][r] += (uint64_t)va[i][r] * vb[j][r];
        if (!N30 && ((q + 1) & mg.red_mask) == 0) {  // (16 products fit for the default primes)
#pragma unroll
          for (int i = 0; i < TA; i++)
#pragma unroll
            for (int j = 0; j < TB; j++)
#pragma unroll
              for (int r = 0; r < RG; r++) acc[i][j][r] = reduce64<N30>(acc[i][j][r], mg, r);
        }
      }
      if (N30) {
#pragma unroll
        for (int i = 0; i < TA; i++)
#pragma unroll
          for (int j = 0; j < TB; j++)
#pragma unroll
            for (int r = 0; r < RG; r++) acc[i][j][r] = reduce64<N30>(acc[i][j][r], mg, r);
      }
    }
    const uint32_t t = tile - g->tile_lo, ta = t & ((1u << (g->ka - kBlkA)) - 1u), tb = t >> (g->ka - kBlkA);
    uint32_t o = off;
    for (uint32_t j = kBlkA; j < g->ka; j++)
      if ((ta >> (j - kBlkA)) & 1u) o += g->wA[j];
    for (uint32_t j = kBlkB; j < g->kb; j++)
      if ((tb >> (j - kBlkB)) & 1u) o += g->wB[j];
    uint32_t* C = arena + g->c_off * RG;
#pragma unroll
    for (int i = 0; i < TA; i++)
#pragma unroll
      for (int j = 0; j < TB; j++) {
        uint32_t out[RG];
#pragma unroll
        for (int r = 0; r < RG; r++) out[r] = (uint32_t)acc[i][j][r];  // (reduced after every chunk)
        uint32_t e = o;
#pragma unroll
        for (int b = 0; b < RA; b++)
          if ((i >> b) & 1) e += g->wA[kBlkA - RA + b];
#pragma unroll
        for (int b = 0; b < RB; b++)
          if ((j >> b) & 1) e += g->wB[kBlkB - RB + b];
        store_entry<RG>(C + (uint64_t)e * RG, out);
      }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// A big step with one small operand (Sec. 2.1 with a skinny matrix): S has
// 2^fs <= 16 rows, the shared dimension 2^k <= 8, the large operand L 2^fl
// rows.  S's 2^(fs+k) entries are staged in shared memory; a thread takes a
// row l of L, loads its 2^k entries once (consecutive threads, consecutive
// rows: coalesced) and writes the 2^fs outputs C[oS(s) + oL(l)].  When S's
// free bits are C's lowest bits (contig) those outputs are contiguous and a
// thread writes them with vector stores (byte residues, 4 per entry).
struct OuterStep {
  uint64_t s_off, l_off, c_off;  // entry offsets of S, L, C in the arena
  uint64_t oS[16];               // output offset of S's row s
  uint64_t oL[32];               // output weight of L's free bit i
  uint32_t fs, fl, k, contig;
  uint32_t block_lo, blocks;     // its blocks in the launch
};

template <int RG, typename W = uint32_t, bool N30 = false>
__global__ void __launch_bounds__(256) outer_kernel(const OuterStep* __restrict__ steps, uint32_t n_steps,
                                                    W* __restrict__ arena0, const __grid_constant__ Pass ps) {
  W* __restrict__ arena = arena0 + blockIdx.y * ps.arena_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  __shared__ uint32_t sm[256 * RG];  // S entry (s, q) at (s + (q << fs)) * RG + r
  __shared__ OuterStep os;
  {
    uint32_t lo = 0, hi = n_steps - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (steps[mid].block_lo <= blockIdx.x) lo = mid;
      else hi = mid - 1;
    }
    static_assert(sizeof(OuterStep) % 8 == 0, "copied by 8-byte words");
    for (uint32_t i = threadIdx.x; i < sizeof(OuterStep) / 8; i += blockDim.x)
      reinterpret_cast<uint64_t*>(&os)[i] = reinterpret_cast<const uint64_t*>(steps + lo)[i];
  }
  __syncthreads();
  const uint32_t fs = os.fs, fl = os.fl, K = 1u << os.k, NS = 1u << fs;
  for (uint32_t i = threadIdx.x; i < (NS << os.k); i += blockDim.x) {
    uint32_t v[RG];
    load_entry<RG, W>(arena + (os.s_off + i) * RG, v);
#pragma unroll
    for (int r = 0; r < RG; r++) sm[i * RG + r] = v[r];
  }
  __syncthreads();
  using Acc = std::conditional_t<sizeof(W) == 1, uint32_t, uint64_t>;
  const W* L0 = arena + os.l_off * RG;
  W* C0 = arena + os.c_off * RG;
  const uint64_t nl = 1ull << fl;
  for (uint64_t l = (uint64_t)(blockIdx.x - os.block_lo) * blockDim.x + threadIdx.x; l < nl;
       l += (uint64_t)os.blocks * blockDim.x) {
    uint32_t lv[8][RG];
#pragma unroll
    for (uint32_t q = 0; q < 8; q++)
      if (q < K) load_entry<RG, W>(L0 + (l + ((uint64_t)q << fl)) * RG, lv[q]);
    uint64_t ol = 0;
    for (uint32_t i = 0; i < fl; i++)
      if ((l >> i) & 1ull) ol += os.oL[i];
    // output s of this row: sum over q of S(s, q) L(l, q), reduced
    auto entry = [&](uint32_t s, uint32_t (&out)[RG]) {
      Acc acc[RG];
#pragma unroll
      for (int r = 0; r < RG; r++) acc[r] = 0;
#pragma unroll
      for (uint32_t q = 0; q < 8; q++) {
        if (q < K) {
          const uint32_t* sv = sm + (s + (q << fs)) * RG;
#pragma unroll
          for (int r = 0; r < RG; r++) acc[r] += (Acc)sv[r] * lv[q][r];
          if (((q + 1) & mg.red_mask) == 0 && q + 1 < K) {
#pragma unroll
            for (int r = 0; r < RG; r++) acc[r] = reduce_acc<N30>(acc[r], mg, r);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < RG; r++) out[r] = reduce_acc<N30>(acc[r], mg, r);
    };
    bool done = false;
    if constexpr (sizeof(W) == 1 && RG == 4) {
      if (os.contig) {  // C entries ol .. ol + NS - 1, 4 bytes each; ol is a multiple of NS
        uint32_t* dst = reinterpret_cast<uint32_t*>(C0 + ol * RG);
        for (uint32_t s0 = 0; s0 < NS; s0 += 4) {
          uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
          for (uint32_t j = 0; j < 4; j++)
            if (s0 + j < NS) {
              uint32_t out[RG];
              entry(s0 + j, out);
              w[j] = out[0] | (out[1] << 8) | (out[2] << 16) | (out[3] << 24);
            }
          if (NS >= 4) *reinterpret_cast<uint4*>(dst + s0) = make_uint4(w[0], w[1], w[2], w[3]);
          else if (NS == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
          else dst[0] = w[0];
        }
        done = true;
      }
    }
    if (!done)
      for (uint32_t s = 0; s < NS; s++) {
        uint32_t out[RG];
        entry(s, out);
        store_entry<RG, W>(C0 + (os.oS[s] + ol) * RG, out);
      }
  }
}

// Split-K for steps with few output entries and a long shared dimension (a
// final dot product, a rank-19 tensor against a rank-19 tensor, ...): block
// (o, part) sums A*B over its slice of the 2^k shared values, the block's
// threads combine their residues with modular additions, and a second kernel
// adds the parts of each output.  part[o * n_split + j] holds RG residues.
template <int RG, typename W = uint32_t, bool N30 = false>
__global__ void __launch_bounds__(256) splitk_partial_kernel(const GridStep* __restrict__ steps, uint32_t n_steps,
                                                             const W* arena0, uint32_t* __restrict__ part0,
                                                             const __grid_constant__ Pass ps) {
  const W* arena = arena0 + blockIdx.y * ps.arena_stride;
  uint32_t* __restrict__ part = part0 + blockIdx.y * ps.part_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  __shared__ uint32_t red[256 * RG];
  const GridStep* __restrict__ g = step_of_block<&GridStep::block_lo>(steps, n_steps);
  const uint32_t log_split = g->log_split, blk = blockIdx.x - g->block_lo;
  const uint32_t n_split = 1u << log_split;
  const uint64_t o = blk >> log_split;
  const uint32_t j = blk & (n_split - 1);
  const uint32_t k = g->d.k, ka = g->d.ka, kb = g->d.kb, c = g->d.c;
  uint64_t ia = 0, ib = 0;
  for (uint32_t b = 0; b < c; b++)
    if ((o >> b) & 1ull) {
      ia += g->wA[b];
      ib += g->wB[b];
    }
  const W* A = arena + (g->d.a_off + ia) * RG;
  const W* B = arena + (g->d.b_off + ib) * RG;
  const uint64_t per = (1ull << k) >> log_split;
  // byte residues: products below 2^16, sums of 16 of them in 32 bits
  using Acc = std::conditional_t<sizeof(W) == 1, uint32_t, uint64_t>;
  Acc acc[RG];
#pragma unroll
  for (int r = 0; r < RG; r++) acc[r] = 0;
  uint32_t cnt = 0;
  bool dot = false;
  if constexpr (sizeof(W) == 1 && RG == 4) {
    // a dot product of contiguous byte-residue operands (no free bits): a
    // thread loads 4 entries of each operand (16 bytes), regroups the bytes
    // by residue (two rounds of byte permutes) and adds 4 products per
    // residue with one dp4a; 1024 products (below 2^26) between reductions
    if (ka == 0 && kb == 0 && (per & 1023u) == 0) {
      dot = true;
      for (uint64_t q = j * per + 4u * threadIdx.x; q < (j + 1) * per; q += 4u * blockDim.x) {
        const uint4 a4 = *reinterpret_cast<const uint4*>(A + q * 4);
        const uint4 b4 = *reinterpret_cast<const uint4*>(B + q * 4);
        const uint32_t ta0 = __byte_perm(a4.x, a4.y, 0x5140), ta1 = __byte_perm(a4.x, a4.y, 0x7362);
        const uint32_t ta2 = __byte_perm(a4.z, a4.w, 0x5140), ta3 = __byte_perm(a4.z, a4.w, 0x7362);
        const uint32_t tb0 = __byte_perm(b4.x, b4.y, 0x5140), tb1 = __byte_perm(b4.x, b4.y, 0x7362);
        const uint32_t tb2 = __byte_perm(b4.z, b4.w, 0x5140), tb3 = __byte_perm(b4.z, b4.w, 0x7362);
        acc[0] = __dp4a(__byte_perm(ta0, ta2, 0x5410), __byte_perm(tb0, tb2, 0x5410), acc[0]);
        acc[1] = __dp4a(__byte_perm(ta0, ta2, 0x7632), __byte_perm(tb0, tb2, 0x7632), acc[1]);
        acc[2] = __dp4a(__byte_perm(ta1, ta3, 0x5410), __byte_perm(tb1, tb3, 0x5410), acc[2]);
        acc[3] = __dp4a(__byte_perm(ta1, ta3, 0x7632), __byte_perm(tb1, tb3, 0x7632), acc[3]);
        if ((++cnt & 255u) == 0) {
#pragma unroll
          for (int r = 0; r < RG; r++) acc[r] = reduce_acc<N30>(acc[r], mg, r);
        }
      }
    }
  }
  if (!dot)
  for (uint64_t q = j * per + threadIdx.x; q < (j + 1) * per; q += blockDim.x) {
    uint32_t va[RG], vb[RG];
    load_entry<RG, W>(A + (q << ka) * RG, va);
    load_entry<RG, W>(B + (q << kb) * RG, vb);
#pragma unroll
    for (int r = 0; r < RG; r++) acc[r] += (Acc)va[r] * vb[r];
    if ((++cnt & mg.red_mask) == 0) {
#pragma unroll
      for (int r = 0; r < RG; r++) acc[r] = reduce_acc<N30>(acc[r], mg, r);
    }
  }
#pragma unroll
  for (int r = 0; r < RG; r++) red[threadIdx.x * RG + r] = reduce_acc<N30>(acc[r], mg, r);
  __syncthreads();
  for (uint32_t h = blockDim.x >> 1; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
#pragma unroll
      for (int r = 0; r < RG; r++) {
        uint32_t x = red[threadIdx.x * RG + r] + red[(threadIdx.x + h) * RG + r];
        if (x >= mg.p[r]) x -= mg.p[r];
        red[threadIdx.x * RG + r] = x;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x < RG) part[((uint64_t)g->part_off + blk) * RG + threadIdx.x] = red[threadIdx.x];
}

// One block per output entry: its threads add the parts, then combine.
template <int RG, typename W = uint32_t, bool N30 = false>
__global__ void __launch_bounds__(256) splitk_final_kernel(const GridStep* __restrict__ steps, uint32_t n_steps,
                                                           W* arena0, const uint32_t* __restrict__ part0,
                                                           const __grid_constant__ Pass ps) {
  W* arena = arena0 + blockIdx.y * ps.arena_stride;
  const ModGroup& mg = ps.mg[blockIdx.y];
  const uint32_t* __restrict__ part = part0 + blockIdx.y * ps.part_stride;
  __shared__ uint32_t red[256 * RG];
  const GridStep* __restrict__ g = step_of_block<&GridStep::final_lo>(steps, n_steps);
  const uint32_t log_split = g->log_split;
  const uint64_t o = blockIdx.x - g->final_lo;
  uint64_t s[RG];
#pragma unroll
  for (int r = 0; r < RG; r++) s[r] = 0;
  for (uint32_t j = threadIdx.x; j < (1u << log_split); j += blockDim.x) {
#pragma unroll
    for (int r = 0; r < RG; r++) s[r] += part[(g->part_off + (o << log_split) + j) * RG + r];  // < 2^31 each, < 2^20 of them
  }
#pragma unroll
  for (int r = 0; r < RG; r++) red[threadIdx.x * RG + r] = reduce64<N30>(s[r], mg, r);
  __syncthreads();
  for (uint32_t h = blockDim.x >> 1; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
#pragma unroll
      for (int r = 0; r < RG; r++) {
        uint32_t x = red[threadIdx.x * RG + r] + red[(threadIdx.x + h) * RG + r];
        if (x >= mg.p[r]) x -= mg.p[r];
        red[threadIdx.x * RG + r] = x;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x < RG) arena[(g->d.c_off + o) * RG + threadIdx.x] = (W)red[threadIdx.x];
}

struct RootMap {
  uint8_t perm[24];  // root bit j -> open variable index
  int n_open;
};

// Root tensors -> result residues [entry][R], entry index bit i = open var i,
// of up to kMaxRoots plans: plan w's entries are [res_lo, res_lo of the next).
struct Root {
  uint64_t root_off, res_lo;
  RootMap map;
};
constexpr int kMaxRoots = 64;
struct Roots {
  Root r[kMaxRoots];
  int n;
  uint64_t n_entries;  // of all of them, from r[0].res_lo
};

template <int RG, typename W = uint32_t>
__global__ void __launch_bounds__(256) extract_kernel(const W* __restrict__ arena0, uint64_t arena_stride,
                                                      const __grid_constant__ Roots rs, uint32_t* __restrict__ results,
                                                      int R, int col0) {
  const W* __restrict__ arena = arena0 + blockIdx.y * arena_stride;
  const int col = col0 + RG * (int)blockIdx.y;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rs.n_entries;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t e = rs.r[0].res_lo + i;
    int lo = 0, hi = rs.n - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (rs.r[mid].res_lo <= e) lo = mid;
      else hi = mid - 1;
    }
    const Root& rt = rs.r[lo];
    const uint32_t J = (uint32_t)(e - rt.res_lo);
    uint64_t a = 0;
    for (int j = 0; j < rt.map.n_open; j++) a |= (uint64_t)((J >> rt.map.perm[j]) & 1u) << j;
#pragma unroll
    for (int r = 0; r < RG; r++)
      if (col + r < R) results[e * R + col + r] = arena[(rt.root_off + a) * RG + r];  // (a group may be filled up)
  }
}

// The CRT of few entries, a warp each: Garner's digits one after the other, but
// every prime's running value v0 + v1 p0 + .. (mod p_i) and its next weight
// p0 .. p_k (mod p_i) kept by a lane of its own (two primes a lane).  One
// thread alone does R^2 / 2 dependent steps: 20 us for 20 residues; this way 2 R,
// and the limbs: 12 us.
__global__ void __launch_bounds__(128) crt_warp_kernel(const uint32_t* __restrict__ residues, uint64_t n_entries,
                                                       const __grid_constant__ CrtConsts cc,
                                                       uint32_t* __restrict__ limbs) {
  const uint64_t e = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (e >= n_entries) return;  // (whole warps)
  const uint32_t lane = threadIdx.x & 31u;
  const int R = cc.R;
  uint32_t r[2], p[2], acc[2] = {0, 0}, wt[2] = {1, 1};  // primes lane and lane + 32
  uint64_t mu[2];
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int i = (int)lane + 32 * h < R ? (int)lane + 32 * h : 0;
    p[h] = cc.p[i];
    mu[h] = cc.mu[i];
    r[h] = residues[e * R + i] % p[h];
  }
  uint32_t x[kCrtMaxLimbs];  // the value, most significant digit first (all lanes alike)
  uint32_t digit[2] = {0, 0};
  for (int k = 0; k < R; k++) {
    uint32_t v = 0;
#pragma unroll
    for (int h = 0; h < 2; h++)
      if ((k >> 5) == h) {
        const uint32_t diff = r[h] >= acc[h] ? r[h] - acc[h] : r[h] + (p[h] - acc[h]);
        v = mod_reduce((uint64_t)diff * cc.inv[k], p[h], mu[h]);  // (meant for lane k mod 32)
      }
    v = __shfl_sync(0xFFFFFFFFu, v, k & 31);
    if ((int)lane == (k & 31)) digit[k >> 5] = v;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      acc[h] = mod_reduce((uint64_t)v * wt[h] + acc[h], p[h], mu[h]);
      wt[h] = mod_reduce((uint64_t)wt[h] * cc.p[k], p[h], mu[h]);
    }
  }
  for (int l = 0; l < kCrtMaxLimbs; l++) x[l] = 0;
  for (int k = R - 1; k >= 0; k--) {
    uint64_t carry = __shfl_sync(0xFFFFFFFFu, digit[k >> 5], k & 31);
#pragma unroll
    for (int l = 0; l < kCrtMaxLimbs; l++) {
      if (l < cc.n_limbs) {
        const uint64_t t = (uint64_t)x[l] * cc.p[k] + carry;
        x[l] = (uint32_t)t;
        carry = t >> 32;
      }
    }
  }
#pragma unroll
  for (int l = 0; l < kCrtMaxLimbs; l++)
    if (l < cc.n_limbs && (int)lane == l) limbs[e * cc.n_limbs + l] = x[l];
}

}  // namespace tnc_dev
