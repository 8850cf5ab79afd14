// Device code of libtnc: modular arithmetic, leaf tensors, the fused
// permute-and-multiply step, the persistent batch kernel and the CRT.
#pragma once

#include <cstdint>
#include <type_traits>

#include "modarith.cuh"
#include "step_desc.h"

namespace tnc_dev {

// An entry holds the RG residues of its group side by side, one word W per
// residue: u32 words for primes below 2^31, bytes for the 8-bit primes of the
// TNC_PATH_TC_P8 arithmetic (four residues in one 32-bit word).
template <int RG, typename W = uint32_t>
__device__ __forceinline__ void load_entry(const W* src, uint32_t (&v)[RG]) {
  if constexpr (sizeof(W) == 1) {
    if constexpr (RG == 4) {
      const uint32_t t = *reinterpret_cast<const uint32_t*>(src);
      v[0] = t & 0xFFu; v[1] = (t >> 8) & 0xFFu; v[2] = (t >> 16) & 0xFFu; v[3] = t >> 24;
    } else if constexpr (RG == 2) {
      const uint32_t t = *reinterpret_cast<const uint16_t*>(src);
      v[0] = t & 0xFFu; v[1] = t >> 8;
    } else {
      v[0] = *src;
    }
  } else if constexpr (RG == 4) {
    const uint4 t = *reinterpret_cast<const uint4*>(src);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else if constexpr (RG == 2) {
    const uint2 t = *reinterpret_cast<const uint2*>(src);
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = *src;
  }
}

// (byte words: every residue is below 2^8)
template <int RG, typename W = uint32_t>
__device__ __forceinline__ void store_entry(W* dst, const uint32_t (&v)[RG]) {
  if constexpr (sizeof(W) == 1) {
    if constexpr (RG == 4) {
      *reinterpret_cast<uint32_t*>(dst) = v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24);
    } else if constexpr (RG == 2) {
      *reinterpret_cast<uint16_t*>(dst) = (uint16_t)(v[0] | (v[1] << 8));
    } else {
      dst[0] = (W)v[0];
    }
  } else if constexpr (RG == 4) {
    *reinterpret_cast<uint4*>(dst) = make_uint4(v[0], v[1], v[2], v[3]);
  } else if constexpr (RG == 2) {
    *reinterpret_cast<uint2*>(dst) = make_uint2(v[0], v[1]);
  } else {
    dst[0] = v[0];
  }
}

// Operand addresses of output entry o (descriptor in global or shared memory).
__device__ __forceinline__ void map_addr(const StepDesc& d, uint64_t o, uint64_t& ia, uint64_t& ib) {
  ia = 0;
  ib = 0;
  if (d.nra != TNC_BITMAP) {
    for (int i = 0; i < d.nra; i++) {
      const TncRun r = d.map.runs.ra[i];
      ia |= ((o >> r.src) & ((1ull << r.len) - 1ull)) << r.dst;
    }
    for (int i = 0; i < d.nrb; i++) {
      const TncRun r = d.map.runs.rb[i];
      ib |= ((o >> r.src) & ((1ull << r.len) - 1ull)) << r.dst;
    }
  } else {
    for (int j = 0; j < d.c; j++) {
      const uint32_t m = d.map.bit[j];
      const uint64_t bit = ((o >> j) & 1ull) << (m & 63u);
      if (m & 0x80u) ib |= bit;
      else ia |= bit;
    }
  }
}

// Leaf tensor entry (Sec. 2.1, Sec. 3.2): COPY (Eq. var; rank 0 is the sum
// over the variable's two values, 2), exactly-one (Eq. 1in3), OR (Eq. or),
// NAND, or an explicit table already permuted to the leaf's layout.
__device__ __forceinline__ uint32_t leaf_value(uint32_t kind, uint32_t rank, uint32_t idx,
                                               const uint32_t* tables, uint32_t toff, uint32_t p) {
  const uint32_t all = (uint32_t)((1ull << rank) - 1ull);
  switch (kind) {
    case 0: return __popc(idx) == 1 ? 1u : 0u;
    case 1: return idx != 0u ? 1u : 0u;
    case 2: return idx != all ? 1u : 0u;
    case 3: return tables[toff + idx] % p;
    default: return rank == 0 ? 2u : ((idx == 0u || idx == all) ? 1u : 0u);
  }
}

// Sum over the 2^k shared-bond values of A*B for every residue of the group
// (A, B point at the operands' first shared-bond entry; consecutive shared
// values are 2^ka and 2^kb entries apart).  A product of residues is below
// (p-1)^2, so red_mask+1 of them plus a reduced partial sum fit in 64 bits:
// reduce after every (red_mask+1)-th product and once at the end.
template <int RG, typename W = uint32_t, bool N30 = false>
__device__ __forceinline__ void step_sum(uint32_t k, uint32_t ka, uint32_t kb, const W* A, const W* B,
                                         const ModGroup& mg, uint32_t (&out)[RG]) {
  const uint64_t sa = (uint64_t)RG << ka, sb = (uint64_t)RG << kb;
  const uint32_t K = 1u << k;
  if constexpr (sizeof(W) == 1) {
    // byte residues (primes <= 251): a product is below 2^16, so red_mask + 1
    // <= 16 of them plus a reduced sum stay below 2^32 -- 32-bit multiply-adds
    uint32_t acc[RG];
#pragma unroll
    for (int r = 0; r < RG; r++) acc[r] = 0;
    uint32_t q = 0;
    for (; q + 4 <= K; q += 4) {
#pragma unroll
      for (int u = 0; u < 4; u++) {
        uint32_t va[RG], vb[RG];
        load_entry<RG, W>(A + (uint64_t)(q + u) * sa, va);
        load_entry<RG, W>(B + (uint64_t)(q + u) * sb, vb);
#pragma unroll
        for (int r = 0; r < RG; r++) acc[r] += va[r] * vb[r];
      }
      if (((q + 4) & mg.red_mask) == 0) {
#pragma unroll
        for (int r = 0; r < RG; r++) acc[r] = mod_reduce32(acc[r], mg.p[r], (uint32_t)(mg.mu[r] >> 32));
      }
    }
    for (; q < K; q++) {
      uint32_t va[RG], vb[RG];
      load_entry<RG, W>(A + (uint64_t)q * sa, va);
      load_entry<RG, W>(B + (uint64_t)q * sb, vb);
#pragma unroll
      for (int r = 0; r < RG; r++) acc[r] += va[r] * vb[r];
    }
#pragma unroll
    for (int r = 0; r < RG; r++) out[r] = mod_reduce32(acc[r], mg.p[r], (uint32_t)(mg.mu[r] >> 32));
    return;
  }
  uint64_t acc[RG];
#pragma unroll
  for (int r = 0; r < RG; r++) acc[r] = 0;
  uint32_t q = 0;
  for (; q + 4 <= K; q += 4) {
#pragma unroll
    for (int u = 0; u < 4; u++) {
      uint32_t va[RG], vb[RG];
      load_entry<RG, W>(A + (uint64_t)(q + u) * sa, va);
      load_entry<RG, W>(B + (uint64_t)(q + u) * sb, vb);
#pragma unroll
      for (int r = 0; r < RG; r++) acc[r] += (uint64_t)va[r] * vb[r];
    }
    if (((q + 4) & mg.red_mask) == 0) {
#pragma unroll
      for (int r = 0; r < RG; r++) acc[r] = reduce64<N30>(acc[r], mg, r);
    }
  }
  for (; q < K; q++) {  // K < 4 here: at most 3 products on a reduced sum
    uint32_t va[RG], vb[RG];
    load_entry<RG, W>(A + (uint64_t)q * sa, va);
    load_entry<RG, W>(B + (uint64_t)q * sb, vb);
#pragma unroll
    for (int r = 0; r < RG; r++) acc[r] += (uint64_t)va[r] * vb[r];
  }
#pragma unroll
  for (int r = 0; r < RG; r++) out[r] = reduce64<N30>(acc[r], mg, r);
}

// A partial sum reduced mod p_r: 64-bit sums by reduce64, 32-bit sums (byte
// residues) by a 32-bit Barrett step.
template <bool N30>
__device__ __forceinline__ uint32_t reduce_acc(uint64_t x, const ModGroup& mg, int r) {
  return reduce64<N30>(x, mg, r);
}
template <bool N30>
__device__ __forceinline__ uint32_t reduce_acc(uint32_t x, const ModGroup& mg, int r) {
  return mod_reduce32(x, mg.p[r], (uint32_t)(mg.mu[r] >> 32));
}

// One output entry of a pairwise step (Sec. 2.1: the permuted operands
// multiplied as matrices): entry o of C from the operand entries ia, ib.
template <int RG, typename W = uint32_t, bool N30 = false>
__device__ __forceinline__ void step_entry_at(uint32_t k, uint32_t ka, uint32_t kb, uint64_t o, uint64_t ia,
                                              uint64_t ib, const W* A0, const W* B0, W* C0, const ModGroup& mg) {
  uint32_t out[RG];
  step_sum<RG, W, N30>(k, ka, kb, A0 + ia * RG, B0 + ib * RG, mg, out);
  store_entry<RG, W>(C0 + o * RG, out);
}

template <int RG, typename W = uint32_t, bool N30 = false>
__device__ __forceinline__ void step_entry(const StepDesc& d, uint64_t o, const W* A0, const W* B0, W* C0,
                                           const ModGroup& mg) {
  uint64_t ia, ib;
  map_addr(d, o, ia, ib);
  step_entry_at<RG, W, N30>(d.k, d.ka, d.kb, o, ia, ib, A0, B0, C0, mg);
}

// Chinese remaindering by Garner's mixed radix:
//   v0 = r0,  v_i = (r_i - (v0 + v1 p0 + ... + v_{i-1} p0..p_{i-2})) * inv_i  mod p_i,
//   X = v0 + p0 (v1 + p1 (v2 + ...)),  0 <= X < p0 p1 ... p_{R-1}.
constexpr int kCrtMaxResidues = 64;
constexpr int kCrtMaxLimbs = 17;
struct CrtConsts {
  uint32_t p[kCrtMaxResidues];
  uint64_t mu[kCrtMaxResidues];
  uint32_t inv[kCrtMaxResidues];  // (p0 ... p_{i-1})^{-1} mod p_i
  int R;
  int n_limbs;                    // <= kCrtMaxLimbs
};

// Residues r[0..R) of one entry to its n_limbs limbs.
__device__ __forceinline__ void crt_entry(const uint32_t* r, const CrtConsts& cc, uint32_t* limbs) {
  uint32_t v[kCrtMaxResidues];
  for (int i = 0; i < cc.R; i++) {
    const uint32_t p = cc.p[i];
    const uint64_t mu = cc.mu[i];
    uint32_t ri = r[i] % p;
    if (i == 0) {
      v[0] = ri;
      continue;
    }
    uint32_t t = mod_reduce(v[i - 1], p, mu);
    for (int j = i - 2; j >= 0; j--) t = mod_reduce((uint64_t)t * cc.p[j] + v[j], p, mu);
    const uint32_t diff = ri >= t ? ri - t : ri + (p - t);
    v[i] = mod_reduce((uint64_t)diff * cc.inv[i], p, mu);
  }
  uint32_t x[kCrtMaxLimbs];
  for (int l = 0; l < kCrtMaxLimbs; l++) x[l] = 0;
  x[0] = v[cc.R - 1];
  for (int i = cc.R - 2; i >= 0; i--) {
    uint64_t carry = v[i];
    for (int l = 0; l < cc.n_limbs; l++) {
      const uint64_t t = (uint64_t)x[l] * cc.p[i] + carry;
      x[l] = (uint32_t)t;
      carry = t >> 32;
    }
  }
  for (int l = 0; l < cc.n_limbs; l++) limbs[l] = x[l];
}

__global__ void crt_kernel(const uint32_t* __restrict__ residues, uint64_t n_entries,
                           const __grid_constant__ CrtConsts cc, uint32_t* __restrict__ limbs) {
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n_entries;
       e += (uint64_t)gridDim.x * blockDim.x)
    crt_entry(residues + e * cc.R, cc, limbs + e * cc.n_limbs);
}

// ------------------------------------------------------- persistent batch

// Packed batch descriptors.  Everything one formula's contraction looks up is
// one contiguous, 16-byte aligned blob (steps, segments, packed items, bit-map
// runs, address deltas, level table), copied to shared memory in one coalesced
// pass when a CTA starts the formula.  Offsets are relative to the formula's
// own arena; a run is a u16: src | dst << 5 | len << 10.
struct BStep {
  uint32_t a_off, b_off, c_off;
  uint16_t run0;  // first run of A's map (blob-relative); B's map follows
  uint16_t dl0;   // first address delta (blob-relative, int2 units)
  uint8_t c, k, ka, kb;
  uint8_t nra, nrb, g, pad;  // g: log2 of the entry stride of a lane group (5 - sh)
};

// The unit of work of one warp.  An output entry whose sum runs over 2^k
// shared values may be split over 2^sh lanes (sh <= min(k, 5)): lane slice j
// sums the shared values j, j + 2^sh, ..., and the lanes of the entry add
// their residues with butterfly shuffles.  A segment is either a block of one
// step: step = step index, o0 = first entry, n = V entries per lane group: the
// 2^(5 - sh) lane groups take entries o0 + group + i 2^(5 - sh), i < V, the
// operand addresses advancing from one to the next by the step's precomputed
// deltas (the output counter o >> g gains one, clearing its trailing ones and
// setting bit t: each address changes by delta[t - g]); or, for steps whose
// entries need fewer than 32 lanes, the lanes of several such entries packed
// side by side: step = kPacked, o0 = first of n lane items, each item =
// step | entry << 16 | slice << 21 | sh << 26, the entries' lane groups
// aligned to their size; sh is then the largest split in the segment.
constexpr uint16_t kPacked = 0xFFFF;
struct Seg {
  uint32_t o0;
  uint16_t step;
  uint8_t n;   // whole-warp block: entries per lane group V; packed: active lanes
  uint8_t sh;  // log2 lanes per entry (packed: the largest)
};

// Sum of A*B over 2^KK shared values (KK <= 4) for residues whose products
// fit 16 to a 64-bit accumulator (the default primes below 2^30): fully
// unrolled, one reduction per residue at the end.  Operand entries of the
// batch arena are addressed by 32-bit entry indices.
template <int RG, bool N30, int KK>
__device__ __forceinline__ void step_sum_fixed(uint32_t ka, uint32_t kb, const uint32_t* A, const uint32_t* B,
                                               const ModGroup& mg, uint32_t (&out)[RG]) {
  uint64_t acc[RG];
#pragma unroll
  for (int r = 0; r < RG; r++) acc[r] = 0;
  const size_t sa = (size_t)RG << ka, sb = (size_t)RG << kb;
#pragma unroll
  for (uint32_t q = 0; q < (1u << KK); q++) {
    uint32_t va[RG], vb[RG];
    load_entry<RG>(A, va);
    load_entry<RG>(B, vb);
    A += sa;
    B += sb;
#pragma unroll
    for (int r = 0; r < RG; r++) acc[r] += (uint64_t)va[r] * vb[r];
  }
#pragma unroll
  for (int r = 0; r < RG; r++) out[r] = reduce64<N30>(acc[r], mg, r);
}

// step_sum for the batch kernel.  For the default primes (16 products fit a
// 64-bit accumulator between reductions): up to 4 products fully unrolled;
// longer sums in unrolled groups of 4 (one group's loads in flight at a
// time, which bounds the registers), reduced after every 16th product.
// Other primes: the general loop.
template <int RG, bool N30>
__device__ __forceinline__ void batch_sum(uint32_t k, uint32_t ka, uint32_t kb, const uint32_t* A, const uint32_t* B,
                                          const ModGroup& mg, uint32_t (&out)[RG]) {
  if (N30) {
    switch (k) {
      case 0: step_sum_fixed<RG, N30, 0>(ka, kb, A, B, mg, out); return;
      case 1: step_sum_fixed<RG, N30, 1>(ka, kb, A, B, mg, out); return;
      case 2: step_sum_fixed<RG, N30, 2>(ka, kb, A, B, mg, out); return;
      default: {
        uint64_t acc[RG];
#pragma unroll
        for (int r = 0; r < RG; r++) acc[r] = 0;
        const uint32_t K = 1u << k;
        const size_t sa = (size_t)RG << ka, sb = (size_t)RG << kb;
#pragma unroll 1
        for (uint32_t q = 0; q < K; q += 4) {
#pragma unroll
          for (uint32_t u = 0; u < 4; u++) {
            uint32_t va[RG], vb[RG];
            load_entry<RG>(A, va);
            load_entry<RG>(B, vb);
            A += sa;
            B += sb;
#pragma unroll
            for (int r = 0; r < RG; r++) acc[r] += (uint64_t)va[r] * vb[r];
          }
          if (((q + 4) & 15u) == 0 && q + 4 < K) {
#pragma unroll
            for (int r = 0; r < RG; r++) acc[r] = reduce64<N30>(acc[r], mg, r);
          }
        }
#pragma unroll
        for (int r = 0; r < RG; r++) out[r] = reduce64<N30>(acc[r], mg, r);
        return;
      }
    }
  }
  step_sum<RG, uint32_t, N30>(k, ka, kb, A, B, mg, out);
}

struct BLeaf {
  uint32_t off;
  uint32_t table_off;
  uint8_t kind, rank, pad0, pad1;
};

struct BForm {
  uint32_t blob;                     // first uint4 of the formula's blob
  uint32_t blob_n;                   // uint4 count
  uint32_t segs_at, items_at, runs_at, lvl_at;  // byte offsets of the blob sections (steps at 0)
  uint32_t nlev, leaf0, nleaf, res_off, n_out, perm_off;
  uint32_t n_open, root_off, arena, dl_at;  // arena: entries this formula needs; dl_at: deltas
};

constexpr uint32_t kSlotCounter = 32;  // a launch's slot counter lies this far behind its work counter

struct BatchArgs {
  const BForm* forms;
  const uint4* blobs;
  const BLeaf* leaves;
  const uint32_t* tables;
  const uint8_t* perms;
  const uint32_t* order;  // queue slot -> formula (largest first)
  uint32_t n_forms;
  uint32_t* queue;        // work counter, zeroed before the launch (with the slot counter)
  uint32_t* results;      // [entry][R]
  uint32_t* garena;       // global arenas, one slot per CTA, reused by every formula the CTA takes
  uint64_t slot_entries;  // entries of a slot (the largest formula's arena; cluster launches: the largest light one's)
  uint32_t blob_cap;      // bytes of dynamic shared memory reserved for a blob
  uint32_t smem_cap;      // entries of dynamic shared memory available for an arena
  int R;
  int col;                // first residue column of this group
  // cluster launches only
  uint32_t n_heavy;       // the first n_heavy formulas of `order` are contracted by whole clusters
  uint32_t* limbs;        // not NULL: this launch also runs the CRT (one formula, the last residue group)
};

// Every thread of the CTAs of a cluster, with the memory ordering of a
// __syncthreads over all of them (global memory included).
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_ctas() {
  uint32_t n;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return n;
}
__device__ __forceinline__ uint32_t cluster_cta() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ uint32_t map_runs(uint32_t o, const uint16_t* runs, int n) {
  uint32_t a = 0;
  for (int i = 0; i < n; i++) {
    const uint32_t r = runs[i];
    const uint32_t src = r & 31u, dst = (r >> 5) & 31u, len = r >> 10;
    a |= ((o >> src) & ((1u << len) - 1u)) << dst;
  }
  return a;
}

// Each CTA repeatedly takes the next formula from the queue and contracts it
// alone, tree level by tree level: all steps of a level are independent, so
// the level is a list of segments shared out over the CTA's warps, with one
// barrier per level.  Descriptors are read from shared memory; the tensors
// live in shared memory when the formula's arena fits, else in the CTA's own
// slot of global memory, reused by each formula the CTA takes, so that the
// live arenas (CTAs x slot) stay in L2 instead of every formula's arena being
// written back to DRAM.
//
// CLUSTER: the grid is made of clusters.  The batch's heaviest formulas (the
// first n_heavy) are contracted first, each by all CTAs of one cluster: the
// segments of a level are shared out over the warps of the cluster, the
// barrier between levels is the cluster's, the tensors live in the slot of the
// cluster (formula t goes to cluster t, then back and forth).  A
// formula that takes longer alone than the batch's average CTA would
// otherwise be what the launch ends with.  Then every CTA takes formulas from
// the queue as above, into the next free one of the slots for light formulas
// (no more of them than light formulas: a CTA that finds none is not needed).
// kBatchSolo: one formula; cluster g contracts it for residue group g (its
// primes in mg[g], its arena in slot g), a single group's cluster also runs the CRT.
enum BatchMode { kBatchCtas, kBatchClusters, kBatchSolo };
// (Beside BatchArgs, not in it: the plain kernel's registers depend on the
// layout of its parameters, 62 or, with spills, 48 for two residues.)
struct ClusterConsts {
  uint64_t heavy_entries;  // entries of a cluster's slot (the largest heavy formula's arena)
  uint64_t light_off;      // entries of all clusters' slots; behind them
  uint32_t light_slots;    // the slots for CTAs with a light formula
};
struct SoloConsts : ClusterConsts {
  CrtConsts crt;
  ModGroup mg[4];
};
template <int MODE>
using BatchConsts = std::conditional_t<MODE == kBatchSolo, SoloConsts, std::conditional_t<MODE == kBatchClusters, ClusterConsts, int>>;
template <int RG, bool N30 = false, int MODE = kBatchCtas>
__global__ void __launch_bounds__(256, MODE == kBatchCtas ? 0 : (MODE == kBatchSolo ? 1 : (RG == 4 && !N30 ? 3 : 4)))
    batch_kernel(BatchArgs a, ModGroup mg, const __grid_constant__ BatchConsts<MODE> sc) {
  constexpr bool CLUSTER = MODE != kBatchCtas;
  extern __shared__ uint4 smem_raw[];
  __shared__ uint32_t task;
  const int lane = threadIdx.x & 31;
  uint4* blob = smem_raw;
  uint32_t* sarena = reinterpret_cast<uint32_t*>(smem_raw + (a.blob_cap >> 4));
  if constexpr (MODE == kBatchSolo) {
    mg = sc.mg[blockIdx.x / cluster_ctas()];
    a.col += RG * (int)(blockIdx.x / cluster_ctas());
  }
  bool coop = CLUSTER;       // contracting the heavy formulas, cluster by cluster
  uint32_t round = 0, slot = 0;
  for (;;) {
    uint32_t t;
    if (CLUSTER && coop) {
      const uint32_t nc = gridDim.x / cluster_ctas(), c = blockIdx.x / cluster_ctas();
      t = MODE == kBatchSolo ? round : round * nc + ((round & 1u) ? nc - 1u - c : c);
      round++;
      if (t >= a.n_heavy) {
        if (a.n_heavy == a.n_forms) break;
        coop = false;
        if constexpr (MODE == kBatchClusters) {
          if (threadIdx.x == 0) task = atomicAdd(a.queue + kSlotCounter, 1u);
          __syncthreads();
          slot = task;
          __syncthreads();  // (the queue's next value goes to the same place)
          if (slot >= sc.light_slots) break;
        }
        continue;
      }
    } else {
      if (threadIdx.x == 0) task = atomicAdd(a.queue, 1u);
      __syncthreads();
      t = task;
      if (CLUSTER) t += a.n_heavy;
      if (t >= a.n_forms) break;
    }
    // the threads and warps that share this formula
    uint32_t tid = threadIdx.x, nthreads = blockDim.x;
    if (CLUSTER && coop) {
      tid += cluster_cta() * blockDim.x;
      nthreads *= cluster_ctas();
    }
    const uint32_t warp = tid >> 5, nwarps = nthreads >> 5;
    const BForm f = a.forms[a.order[t]];
    for (uint32_t i = threadIdx.x; i < f.blob_n; i += blockDim.x) blob[i] = a.blobs[f.blob + i];
    uint32_t* arena = a.garena;
    if constexpr (CLUSTER) {
      if (coop) arena += (uint64_t)(blockIdx.x / cluster_ctas()) * sc.heavy_entries * RG;
      else arena = f.arena <= a.smem_cap ? sarena : arena + (sc.light_off + slot * a.slot_entries) * RG;
    } else {
      arena = f.arena <= a.smem_cap ? sarena : arena + (uint64_t)blockIdx.x * a.slot_entries * RG;
    }
    auto barrier = [&] {
      if (CLUSTER && coop) cluster_barrier();
      else __syncthreads();
    };
    for (uint32_t l = tid; l < f.nleaf; l += nthreads) {
      const BLeaf ld = a.leaves[f.leaf0 + l];
      uint32_t* dst = arena + (uint64_t)ld.off * RG;
      const uint32_t n = 1u << ld.rank;
      for (uint32_t idx = 0; idx < n; idx++) {
        uint32_t v[RG];
#pragma unroll
        for (int r = 0; r < RG; r++) v[r] = leaf_value(ld.kind, ld.rank, idx, a.tables, ld.table_off, mg.p[r]);
        store_entry<RG>(dst + (uint64_t)idx * RG, v);
      }
    }
    barrier();
    const char* bb = reinterpret_cast<const char*>(blob);
    const BStep* steps = reinterpret_cast<const BStep*>(bb);
    const Seg* segs = reinterpret_cast<const Seg*>(bb + f.segs_at);
    const uint32_t* items = reinterpret_cast<const uint32_t*>(bb + f.items_at);
    const uint16_t* runs_all = reinterpret_cast<const uint16_t*>(bb + f.runs_at);
    const uint32_t* lvl = reinterpret_cast<const uint32_t*>(bb + f.lvl_at);
    const int2* deltas = reinterpret_cast<const int2*>(bb + f.dl_at);
    for (uint32_t l = 0; l < f.nlev; l++) {
      const uint32_t s1 = lvl[l + 1];
      for (uint32_t sg = lvl[l] + warp; sg < s1; sg += nwarps) {
        const Seg seg = segs[sg];
        if (seg.step != kPacked) {
          // a block of V entries per lane group of one step
          const BStep d = steps[seg.step];
          const uint32_t sh = seg.sh, g = d.g;
          uint32_t o = seg.o0 + (lane >> sh);
          const uint32_t slice = lane & ((1u << sh) - 1u);
          const uint16_t* runs = runs_all + d.run0;
          uint32_t ia = map_runs(o, runs, d.nra) + (slice << d.ka);
          uint32_t ib = map_runs(o, runs + d.nra, d.nrb) + (slice << d.kb);
          const uint32_t* A0 = arena + (uint64_t)d.a_off * RG;
          const uint32_t* B0 = arena + (uint64_t)d.b_off * RG;
          uint32_t* C0 = arena + (uint64_t)d.c_off * RG;
          const int2* dl = deltas + d.dl0;
          for (uint32_t v = 0; v < seg.n; v++) {
            uint32_t out[RG];
            batch_sum<RG, N30>(d.k - sh, d.ka + sh, d.kb + sh, A0 + ia * RG, B0 + ib * RG, mg, out);
            for (uint32_t m = 1; m < (1u << sh); m <<= 1) {
#pragma unroll
              for (int r = 0; r < RG; r++) {
                const uint32_t t = out[r] + __shfl_xor_sync(0xFFFFFFFFu, out[r], m);
                out[r] = t >= mg.p[r] ? t - mg.p[r] : t;
              }
            }
            if (slice == 0) store_entry<RG>(C0 + o * RG, out);
            if (v + 1 < seg.n) {
              const int2 dd = dl[__ffs(~(o >> g)) - 1];
              o += 1u << g;
              ia += (uint32_t)dd.x;
              ib += (uint32_t)dd.y;
            }
          }
          continue;
        }
        // packed lanes of small steps, one entry per lane
        const bool active = lane < seg.n;
        const uint32_t it = items[seg.o0 + (active ? lane : 0)];
        const uint32_t st = it & 0xFFFFu, o = (it >> 16) & 31u, slice = (it >> 21) & 31u, sh = it >> 26;
        const BStep d = steps[st];
        uint32_t out[RG];
        if (active) {
          const uint16_t* runs = runs_all + d.run0;
          const uint32_t ia = map_runs(o, runs, d.nra) + (slice << d.ka);
          const uint32_t ib = map_runs(o, runs + d.nra, d.nrb) + (slice << d.kb);
          batch_sum<RG, N30>(d.k - sh, d.ka + sh, d.kb + sh, arena + ((uint64_t)d.a_off + ia) * RG,
                             arena + ((uint64_t)d.b_off + ib) * RG, mg, out);
        } else {
#pragma unroll
          for (int r = 0; r < RG; r++) out[r] = 0;
        }
        // lanes of one entry add their partial sums (all lanes take part in
        // every shuffle; a lane keeps only its own group's partners)
        for (uint32_t m = 1; m < (1u << seg.sh); m <<= 1) {
#pragma unroll
          for (int r = 0; r < RG; r++) {
            const uint32_t v = __shfl_xor_sync(0xFFFFFFFFu, out[r], m);
            if (m < (1u << sh)) {
              const uint32_t t = out[r] + v;
              out[r] = t >= mg.p[r] ? t - mg.p[r] : t;
            }
          }
        }
        if (active && slice == 0) store_entry<RG>(arena + ((uint64_t)d.c_off + o) * RG, out);
      }
      barrier();
    }
    for (uint32_t J = tid; J < f.n_out; J += nthreads) {
      uint32_t ad = 0;
      for (uint32_t j = 0; j < f.n_open; j++) ad |= ((J >> a.perms[f.perm_off + j]) & 1u) << j;
#pragma unroll
      for (int r = 0; r < RG; r++)
        if (RG != 4 || a.col + r < a.R)  // (a group of four may be filled up)
          a.results[((uint64_t)f.res_off + J) * a.R + a.col + r] = arena[((uint64_t)f.root_off + ad) * RG + r];
    }
    barrier();
    if constexpr (MODE == kBatchSolo)
      if (a.limbs)
      for (uint32_t J = tid; J < f.n_out; J += nthreads)
        crt_entry(a.results + (uint64_t)J * a.R, sc.crt, a.limbs + (uint64_t)J * sc.crt.n_limbs);
  }
}

}  // namespace tnc_dev
