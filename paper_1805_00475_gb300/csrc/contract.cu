// C ABI, device half.  Contraction of one formula or of a group of formulas
// (tnc_contract, tnc_contract_many, tnc_contract_sliced) runs tree level by
// tree level: one level_kernel launch for the level's small steps of every
// plan of the group, one launch each for its big, one-small-operand and
// split-K steps, and the dense steps on the tensor-core paths (tc.cu,
// tc_p8.cu); then the component product and the CRT.  The allocation-free
// variant (tnc_contract_noalloc) runs the steps in order in a fixed array.
// The persistent batch (tnc_batch_*) contracts many small plans in one
// graph-captured launch of batch_kernel.
#include <type_traits>
#include <cuda.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "kernels.cuh"
#include "steps.cuh"
#include "tnc_internal.h"

using namespace tnc;
using tnc_dev::BatchArgs;
using tnc_dev::CrtConsts;
using tnc_dev::ModGroup;

namespace {

#define CUDA_TRY(call)                                                                      \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return set_error(TNC_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
  } while (0)

constexpr size_t kAlign = 256;

// An NVTX range for profilers (nvtx is header-only and costs nothing when no
// tool is attached): whole calls, tree levels, dense steps, batch launches.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// Dense-step timing of tnc_contract (off unless tnc_set_step_timing(1)).
thread_local bool g_time_dense = false;
thread_local double g_dense_ms = 0.0;
thread_local int g_dense_launches = 0;
thread_local double g_total_ms = 0.0;
thread_local tnc_launch_counts g_launches{};
thread_local tnc_kernel_launches g_kernels{};
thread_local std::vector<tnc_dense_step_time> g_dense_steps;  // timing mode: per dense launch
thread_local uint64_t g_h2d_bytes = 0, g_d2h_bytes = 0;  // host <-> device copies of the last contraction
size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
  return n;
}

uint32_t powmod(uint64_t a, uint64_t e, uint32_t p) {
  uint64_t r = 1;
  a %= p;
  while (e) {
    if (e & 1) r = r * a % p;
    a = a * a % p;
    e >>= 1;
  }
  return (uint32_t)r;
}

// Residues are processed in groups of 4, 2 or 1 primes (one pass each).
struct Groups {
  std::vector<int> rg, col;
};

// fill: three residues left over are a group of four with one that nobody asked for.
Groups split_groups(int R, bool fill) {
  Groups g;
  int c = 0;
  for (int s : {4, 2, 1})
    while (R - c >= s || (fill && s == 4 && R - c == 3)) {
      g.rg.push_back(s);
      g.col.push_back(c);
      c += s;
    }
  return g;
}

struct Arith {
  int R = 0;
  std::vector<uint32_t> primes;
  CrtConsts crt{};
  double log2_prod = 0;
  Groups groups;
  ModGroup group(int gi) const {
    uint32_t p[4];
    for (int r = 0; r < 4; r++) {  // (a filled-up group repeats its first prime)
      const int i = groups.col[gi] + r;
      p[r] = primes[r < groups.rg[gi] && i < R ? i : groups.col[gi]];
    }
    return tnc_dev::make_mod_group(p);
  }
};

int make_arith(const tnc_contract_opts* o, Arith& a) {
  if (!o) return set_error(TNC_ERR_INVALID, "contract opts NULL");
  if (o->path != TNC_PATH_INT64 && o->path != TNC_PATH_TC && o->path != TNC_PATH_TC_P8)
    return set_error(TNC_ERR_INVALID, "unknown arithmetic path");
  const bool p8 = o->path == TNC_PATH_TC_P8;
  const int max_r = p8 ? kP8MaxResidues : 16;
  if (o->n_residues < 1 || o->n_residues > max_r)
    return set_error(TNC_ERR_INVALID, p8 ? "n_residues must be in [1, 53]" : "n_residues must be in [1, 16]");
  a.R = o->n_residues;
  a.primes = p8 ? default_primes_p8(a.R) : default_primes(a.R);
  if (o->primes && !std::equal(a.primes.begin(), a.primes.end(), o->primes)) {  // (the default ones need no test)
    a.primes.assign(o->primes, o->primes + a.R);
    for (int i = 0; i < a.R; i++) {
      uint32_t p = a.primes[i];
      if (p8 ? (p < 3 || p > kP8PrimeMax || !is_prime_u32(p))
             : (p <= (1u << 29) || p >= (1u << 31) || !is_prime_u32(p)))
        return set_error(TNC_ERR_INVALID, p8 ? "primes must be primes in [3, 251]" : "primes must be primes in (2^29, 2^31)");
      for (int j = 0; j < i; j++)
        if (a.primes[j] == p) return set_error(TNC_ERR_INVALID, "primes must be distinct");
    }
  }
  a.crt = CrtConsts{};
  a.crt.R = a.R;
  a.log2_prod = 0;
  for (int i = 0; i < a.R; i++) {
    const uint32_t p = a.primes[i];
    a.crt.p[i] = p;
    a.crt.mu[i] = ~0ull / p;
    uint64_t prod = 1;
    for (int j = 0; j < i; j++) prod = prod * (a.primes[j] % p) % p;
    a.crt.inv[i] = i == 0 ? 1u : powmod(prod, p - 2, p);
    a.log2_prod += std::log2((double)p);
  }
  // limbs of the CRT value: enough for prod p < 2^(32 n_limbs)
  a.crt.n_limbs = p8 ? (int)std::floor(a.log2_prod / 32.0) + 1 : (31 * a.R + 31) / 32;
  a.groups = split_groups(a.R, false);
  return TNC_OK;
}

uint32_t result_flags(const tnc_plan_t* p, const Arith& a) {
  return p->net.log2_bound >= a.log2_prod - 1e-9 ? TNC_MAYBE_WRAPPED : 0u;
}

// The word type of a residue in a pass (u32, or a byte on the 8-bit-prime path).
template <typename T>
struct WordTag {
  using type = T;
};

template <typename F>
int dispatch_rg(int rg, F&& f) {
  switch (rg) {
    case 4: return f(std::integral_constant<int, 4>());
    case 2: return f(std::integral_constant<int, 2>());
    default: return f(std::integral_constant<int, 1>());
  }
}

// ---------------------------------------------------------------- single formula

// One pass over the steps: `groups` residue groups of rg residues each, side
// by side in one launch per kind of step, from residue `col` on (the last group
// of a filled-up pass has fewer).
struct PassShape {
  int rg, groups, col;
};

// Workspace of a group of plans contracted together (one plan: the
// single-formula layout).  Descriptors of all plans side by side; every plan's
// tensors in its own part of one arena (arena_base, in entries, a multiple of
// 64 so that every plan's entries start 16-byte aligned); scratch shared by
// the group's steps, which run one after another on one stream.
struct SeqLayout {
  size_t off_leaves, off_tables, off_steps, off_small, off_tc, off_err, off_part, off_results, off_limbs, off_p8,
      off_arena, total;
  int path;        // of the choice laid out
  uint64_t n_out;  // result entries of the whole group
  uint64_t part_bytes, p8_bytes;  // the sections' sizes
  std::vector<PassShape> passes;
  uint64_t arena_entries;  // of one residue group's arena
  size_t n_dense;
  std::vector<uint64_t> arena_base, res_base, leaf_base, table_base;
};

using tnc_dev::GridStep;

// Launch shape of a grid-wide step: S = threads * blocks = 2^s <= 2^c.
void grid_shape(int c, int* threads, int* blocks, int* s) {
  const int t = c >= 8 ? 8 : c;
  const int b = c >= 8 ? std::min(c - 8, 10) : 0;
  *threads = 1 << t;
  *blocks = 1 << b;
  *s = t + b;
}

// Split-K for steps with at most 2^12 outputs and at least 2^9 shared values:
// returns log2 of the number of K slices (0 = no split).  A block sums one
// slice of one output: slices keep at least 256 shared values (one per
// thread), the grid aims at 2^10 blocks (about 7 per SM; a final dot product
// of two rank-22 tensors then sums 16 values per thread instead of one) and
// keeps at least two slices; outputs x slices stays at most 2^13.  (Capping
// the values per thread at 64 with more slices measured 6 % slower on the
// 1-in-3 batch's heavy formulas and no faster on C4-sized ones.)
uint32_t splitk_log(const StepDesc& d) {
  if (d.c > 12 || d.k < 9) return 0;
  const uint32_t ls = d.c < 9 ? 10u - d.c : 1u;
  return std::min<uint32_t>(ls, d.k - 8u);
}

// Output bit j of a step comes from bit dst[j] of operand op[j] (0: A, 1: B).
struct BitMap {
  int op[64] = {0}, dst[64] = {0};
  explicit BitMap(const StepDesc& d) {
    if (d.nra != TNC_BITMAP) {
      for (int side = 0; side < 2; side++)
        for (int i = 0; i < (side ? d.nrb : d.nra); i++) {
          const TncRun& x = side ? d.map.runs.rb[i] : d.map.runs.ra[i];
          for (int q = 0; q < x.len; q++) {
            op[x.src + q] = side;
            dst[x.src + q] = x.dst + q;
          }
        }
    } else {
      for (int j = 0; j < d.c; j++) {
        op[j] = d.map.bit[j] >> 7;
        dst[j] = d.map.bit[j] & 63;
      }
    }
  }
};

// Grid-wide steps of u32 residues with at least 16 shared values run in
// shared-memory tiles (block_kernel); the tile shape, -1 if none.
int block_shape(const StepDesc& d) {
  const int shape = d.c >= 19 ? 0 : d.c >= 17 ? 1 : d.c >= 16 ? 2 : -1;
  const int la = std::max(d.ka, d.kb), lb = std::min(d.ka, d.kb);
  if (shape < 0 || d.k < 4) return -1;
  if (la >= (shape == 0 ? 6 : 5) && lb >= (shape == 2 ? 4 : 5)) return shape;
  return -1;
}

template <int SHAPE>
tnc_dev::BlockStep make_block_step(const StepDesc& d) {
  using B = tnc_dev::Blk<SHAPE>;
  tnc_dev::BlockStep g;
  std::memset(&g, 0, sizeof(g));
  // rows from the operand with more free bits (LA >= LB)
  const int rows = d.ka >= d.kb ? 0 : 1;
  g.a_off = rows ? d.b_off : d.a_off;
  g.b_off = rows ? d.a_off : d.b_off;
  g.c_off = d.c_off;
  g.k = d.k;
  g.ka = rows ? d.kb : d.ka;
  g.kb = rows ? d.ka : d.kb;
  const BitMap m(d);
  for (int j = 0; j < d.c; j++) (m.op[j] == rows ? g.wA : g.wB)[m.dst[j]] = 1u << j;
  int n = 0;
  for (int j = 0; j < d.c; j++) {  // ascending output weight
    const bool row = m.op[j] == rows;
    if (m.dst[j] < (row ? B::LA - B::RA : B::LB - B::RB)) g.bit[n++] = (uint8_t)(m.dst[j] | (row ? 0 : 0x80));
  }
  return g;
}
static_assert(sizeof(tnc_dev::BlockStep) <= sizeof(GridStep), "either fits the step's part of the workspace");

// Register tiles (tile_kernel) for grid-wide steps that leave enough threads.
constexpr int kTileMinC = 18, kTileMinCBytes = 16;
bool tile_eligible(const StepDesc& d, bool bytes) {
  return d.c >= (bytes ? kTileMinCBytes : kTileMinC) && d.ka >= tnc_dev::kTileA && d.kb >= tnc_dev::kTileB;
}

tnc_dev::TileStep make_tile_step(const StepDesc& d) {
  using tnc_dev::kTileA;
  using tnc_dev::kTileB;
  tnc_dev::TileStep t;
  std::memset(&t, 0, sizeof(t));
  t.a_off = d.a_off;
  t.b_off = d.b_off;
  t.c_off = d.c_off;
  t.k = d.k;
  t.ka = d.ka;
  t.kb = d.kb;
  const BitMap m(d);
  uint32_t out_a[kTileA] = {}, out_b[kTileB] = {};  // output bits of the operands' highest free bits
  for (int j = 0; j < d.c; j++) {
    const int top = m.op[j] ? m.dst[j] - (d.kb - kTileB) : m.dst[j] - (d.ka - kTileA);
    if (top >= 0) {
      (m.op[j] ? out_b : out_a)[top] = (uint32_t)j;
    } else {
      t.wA[t.n_bits] = m.op[j] ? 0u : 1u << m.dst[j];
      t.wB[t.n_bits] = m.op[j] ? 1u << m.dst[j] : 0u;
      t.wC[t.n_bits++] = 1u << j;
    }
  }
  for (uint32_t i = 0; i < (1u << kTileA); i++) {
    t.tA[i] = i << (d.ka - kTileA);
    for (int b = 0; b < kTileA; b++)
      if ((i >> b) & 1u) t.cA[i] += 1u << out_a[b];
  }
  for (uint32_t i = 0; i < (1u << kTileB); i++) {
    t.tB[i] = i << (d.kb - kTileB);
    for (int b = 0; b < kTileB; b++)
      if ((i >> b) & 1u) t.cB[i] += 1u << out_b[b];
  }
  int threads, blocks, sh;
  grid_shape((int)t.n_bits, &threads, &blocks, &sh);
  t.s = (uint8_t)sh;
  for (uint32_t b = (uint32_t)sh; b < t.n_bits; b++) {
    t.dA[b] = t.wA[b];
    t.dB[b] = t.wB[b];
    t.dC[b] = t.wC[b];
    for (uint32_t j = (uint32_t)sh; j < b; j++) {  // (modulo 2^32)
      t.dA[b] -= t.wA[j];
      t.dB[b] -= t.wB[j];
      t.dC[b] -= t.wC[j];
    }
  }
  return t;
}
static_assert(sizeof(tnc_dev::TileStep) <= sizeof(GridStep), "either fits the step's part of the workspace");

GridStep make_grid_step(const StepDesc& d) {
  GridStep g;
  std::memset(&g, 0, sizeof(g));
  g.d = d;
  const BitMap m(d);
  for (int j = 0; j < d.c; j++) {
    g.wA[j] = m.op[j] == 0 ? 1ull << m.dst[j] : 0ull;
    g.wB[j] = m.op[j] == 1 ? 1ull << m.dst[j] : 0ull;
  }
  int threads, blocks, sh;
  grid_shape(d.c, &threads, &blocks, &sh);
  g.s = (uint16_t)sh;
  g.log_split = (uint16_t)splitk_log(d);
  for (int t = sh; t < d.c; t++) {
    uint64_t sa = 0, sb = 0;
    for (int j = sh; j < t; j++) {
      sa += g.wA[j];
      sb += g.wB[j];
    }
    g.dA[t] = g.wA[t] - sa;
    g.dB[t] = g.wB[t] - sb;
  }
  return g;
}

// A big step with one small operand (at most 2^4 free rows, at most 2^3
// shared values) runs as outer_kernel: the small operand staged in shared
// memory, one row of the large operand per thread.
bool outer_eligible(const StepDesc& d) {
  return splitk_log(d) == 0 && d.c >= 16 && std::min(d.ka, d.kb) <= 4 && std::max(d.ka, d.kb) <= 32 && d.k <= 3;
}

tnc_dev::OuterStep make_outer_step(const StepDesc& d) {
  tnc_dev::OuterStep o;
  std::memset(&o, 0, sizeof(o));
  const int s_side = d.ka <= d.kb ? 0 : 1;  // the small operand: A, or B
  o.fs = s_side ? d.kb : d.ka;
  o.fl = s_side ? d.ka : d.kb;
  o.k = d.k;
  o.s_off = s_side ? d.b_off : d.a_off;
  o.l_off = s_side ? d.a_off : d.b_off;
  o.c_off = d.c_off;
  o.blocks = (uint32_t)std::min<uint64_t>(((1ull << o.fl) + 255) / 256, (uint64_t)sm_count() * 8);
  const BitMap m(d);
  uint64_t wS[4] = {0, 0, 0, 0};
  for (int j = 0; j < d.c; j++) {
    if (m.op[j] == s_side) wS[m.dst[j]] = 1ull << j;
    else o.oL[m.dst[j]] = 1ull << j;
  }
  for (uint32_t x = 0; x < (1u << o.fs); x++)
    for (uint32_t i = 0; i < o.fs; i++)
      if ((x >> i) & 1u) o.oS[x] += wS[i];
  o.contig = 1;
  for (uint32_t i = 0; i < o.fs; i++)
    if (wS[i] != (1ull << i)) o.contig = 0;
  return o;
}

// What one plan adds to a group's workspace: counts of descriptors, result
// entries and arena entries (summed over the group), and scratch bytes (the
// group's maximum).
struct Foot {
  size_t leaves = 0, tables = 0, nseq = 0, nlvl = 0, n_dense = 0;
  uint64_t n_out = 0, arena = 0;
  double cost = 0;  // multiply-adds and entries per residue
  // bytes per residue of the largest step: split-K partials; on the
  // tensor-core paths a dense step's planes, and its partials or small residues
  uint64_t split = 0, planes = 0, parts = 0;
  uint64_t kept = 0;  // (kept_split_bytes)
  std::vector<uint64_t> lvl_planes, lvl_parts;  // of all dense steps of a tree level
  void add(const Foot& f) {
    leaves += f.leaves;
    tables += f.tables;
    nseq += f.nseq;
    nlvl += f.nlvl;
    n_dense += f.n_dense;
    n_out += f.n_out;
    arena += f.arena;
    cost += f.cost;
    split = std::max(split, f.split);
    planes = std::max(planes, f.planes);
    parts = std::max(parts, f.parts);
    kept = std::max(kept, f.kept);
    lvl_planes.resize(std::max(lvl_planes.size(), f.lvl_planes.size()));
    lvl_parts.resize(std::max(lvl_parts.size(), f.lvl_parts.size()));
    for (size_t l = 0; l < f.lvl_planes.size(); l++) {
      lvl_planes[l] += f.lvl_planes[l];
      lvl_parts[l] += f.lvl_parts[l];
    }
  }
};

// Residue groups run side by side while their arenas together stay within
// kMergeArena: 16 to 20 residues of cubic VC formulas with 100 to 160 vertices
// on TNC_PATH_TC_P8 took 1.4 to 2.4 times as long in one pass per group. (512
// MiB, 2 GiB, 8 GiB: 48 1-in-3 formulas 5.98, 5.87, 5.49 ms; 4 slices of a
// formula with n = 160 1.82, 1.49, 1.48 ms; n = 180, 20 residues 11.0, 11.1,
// 10.5 ms.)
constexpr uint64_t kMergeArena = 8192ull << 20;

// The last group is filled up to four residues, instead of passes of two and of
// one, where the residues that nobody asked for cost less than the launches
// saved: a pass is 15 to 25 launches (50 to 100 us), a residue `cost`
// multiply-adds at about 5e12 per second on the CUDA cores, 5e14 on
// TNC_PATH_TC_P8 and a tenth of that on TNC_PATH_TC.
bool fill_up(int R, double cost, int path) {
  const int rest = R % 4, saved = rest == 3 ? (R > 4 ? 2 : 1) : (R > 4 ? 1 : 0);
  const double rate = path == TNC_PATH_TC_P8 ? 5e14 : path == TNC_PATH_TC ? 5e13 : 5e12;
  return rest && (4 - rest) * cost / rate < saved * 50e-6;
}

// The dense steps of a level are launched together as far as their planes and
// partials fit; up to these sizes the sections grow beyond the largest single
// step's for that (steps that need more fill the GPU by themselves).
constexpr uint64_t kGroupPlanes = 256ull << 20, kGroupParts = 64ull << 20;
// TNC_PATH_TC keeps all residues of a pass together where these allow it (its
// planes take 18 to 24 bytes per residue and operand entry, its small residues
// 9 to 12 per output entry: residue by residue the output's 16-byte entries
// would be written a quarter at a time).
constexpr uint64_t kTcPlanes = 2048ull << 20, kTcBytes = 1024ull << 20;

// Step i of a plan's level schedule as TNC_PATH_TC_P8 runs it: direct planes
// of its operands and output.
uint32_t p8_flags(const Lowered& lw, uint32_t i) {
  const int sa = lw.lvl_src_a[i], sb = lw.lvl_src_b[i];
  return (lw.p8_direct[i] ? kP8DirectOut : 0u) | (sa >= 0 && lw.p8_direct[sa] ? kP8DirectA : 0u) |
         (sb >= 0 && lw.p8_direct[sb] ? kP8DirectB : 0u);
}

// TNC_PATH_TC dense steps whose planes do not fit are summed in 2^chunks parts of
// their shared values, up to 2^kMaxChunkLog.
constexpr uint32_t kMaxChunkLog = 3;
StepDesc tc_part(const StepDesc& d, uint32_t chunks, uint64_t part) {
  StepDesc x = d;
  x.k = (uint8_t)(d.k - chunks);
  x.a_off += part << (x.k + d.ka);  // (shared values are the operands' highest bits)
  x.b_off += part << (x.k + d.kb);
  return x;
}
bool tc_chunks(const StepDesc& d, uint64_t planes, uint64_t bytes, uint32_t* chunks) {
  for (*chunks = 0; *chunks <= kMaxChunkLog; ++*chunks) {
    const StepDesc x = tc_part(d, *chunks, 0);
    if (!tc_eligible(x)) return false;
    if (tc_plane_bytes(x) <= planes && tc_byte_bytes(x) <= bytes) return true;
  }
  return false;
}

// Bytes that the CUDA-core layout sets aside for a dense step's K split and
// (per residue) descriptor.  No kernel uses them any more; they stay because
// tnc_contract_noalloc takes or refuses a plan by this layout's size.
uint64_t kept_split_bytes(const StepDesc& d) {
  const bool swap = !(d.ka >= 7 && d.kb >= 5);
  const uint32_t fa = swap ? d.kb : d.ka, fb = swap ? d.ka : d.kb;
  const uint64_t tiles = (1ull << (fa - 7)) << (fb - 5);
  uint32_t ls = 0;
  while ((tiles << ls) < 304 && d.k - ls > 7 && (1ull << (d.c + ls + 1)) <= (1ull << 24)) ls++;
  return ls ? 4ull << (d.c + ls) : 0;
}
constexpr size_t kKeptDenseBytes = 600;

Foot foot_of(const tnc_plan_t* p, int path) {
  Foot f;
  f.leaves = p->low.leaves.size();
  f.tables = p->low.leaf_tables.size();
  f.nseq = p->low.seq_steps.size();
  f.nlvl = p->low.lvl_steps.size();
  f.n_out = 1ull << p->net.open_vars.size();
  f.cost = p->cost.macs + p->cost.entries;
  const bool p8 = path == TNC_PATH_TC_P8, tc = path == TNC_PATH_TC;
  for (size_t l = 0; l + 1 < p->low.lvl_start.size(); l++) {
    uint64_t sum_planes = 0, sum_parts = 0;
    for (uint32_t i = p->low.lvl_start[l]; i < p->low.lvl_start[l + 1]; i++) {
      const StepDesc& d = p->low.lvl_steps[i];
      if (splitk_log(d) > 0)
        f.split = std::max<uint64_t>(f.split, (1ull << (d.c + splitk_log(d))) * sizeof(uint32_t));
      uint64_t planes = 0, parts = 0;
      if (p8 && p8_eligible(d)) {
        planes = p8_scratch_bytes(P8Step{d, p8_flags(p->low, i)}, 1);
        parts = p8_part_bytes(d, 1);
        f.n_dense++;
      } else if (!p8 && tc_eligible(d)) {
        f.n_dense++;
        if (tc) {
          planes = tc_plane_bytes(d);
          parts = tc_byte_bytes(d);
        } else {
          f.kept = std::max<uint64_t>(f.kept, kept_split_bytes(d));
        }
      }
      f.planes = std::max<uint64_t>(f.planes, planes);
      f.parts = std::max<uint64_t>(f.parts, parts);
      sum_planes += planes;
      sum_parts += parts;
    }
    f.lvl_planes.push_back(sum_planes);
    f.lvl_parts.push_back(sum_parts);
  }
  uint64_t arena = std::max(p->low.seq_arena_entries, p->low.lvl_arena_entries);
  if (p8) arena = std::max(arena, p->low.p8_arena_entries);
  f.arena = (arena + 63) / 64 * 64;
  return f;
}

// How a call may lay its workspace out, from the fastest to the smallest.
enum Fit {
  kWide,    // residue groups side by side as far as kMergeArena allows, scratch for the dense steps of a level together
  kNarrow,  // one residue group at a time
  kLeast,   // and scratch for one dense step at a time (TNC_PATH_TC: one residue of it)
  kSingle,  // and one residue at a time
  kSpare    // TNC_PATH_TC: one residue at a time, its scratch what the workspace leaves
};
struct Choice {
  int path;  // TNC_PATH_TC runs on the CUDA cores alone where too few of its planes fit
  Fit fit;
};
// A path's choices; the last is the least that works, no more than the path
// needed before tensor-core steps had planes (TNC_PATH_TC: TNC_PATH_INT64's).
const std::vector<Choice>& choices(int path) {
  static const std::vector<Choice> int64{{TNC_PATH_INT64, kWide}, {TNC_PATH_INT64, kNarrow}};
  static const std::vector<Choice> p8{{TNC_PATH_TC_P8, kWide}, {TNC_PATH_TC_P8, kNarrow}, {TNC_PATH_TC_P8, kLeast},
                                      {TNC_PATH_TC_P8, kSingle}};
  static const std::vector<Choice> tc{{TNC_PATH_TC, kWide}, {TNC_PATH_TC, kNarrow}, {TNC_PATH_TC, kLeast},
                                      {TNC_PATH_TC, kSingle}, {TNC_PATH_TC, kSpare}, {TNC_PATH_INT64, kNarrow}};
  return path == TNC_PATH_TC_P8 ? p8 : path == TNC_PATH_TC ? tc : int64;
}

// Offsets of the workspace sections for the group footprint f (of the choice's path).
SeqLayout layout_of(const Foot& f, int R, Choice ch) {
  SeqLayout s{};
  const int path = s.path = ch.path;
  const bool wide = ch.fit == kWide, together = ch.fit <= kNarrow, spare = ch.fit == kSpare;
  const bool p8 = path == TNC_PATH_TC_P8, tc = path == TNC_PATH_TC;
  const size_t word = p8 ? 1 : sizeof(uint32_t);  // bytes per residue
  // the passes
  int quads = R / 4, rest = R % 4;
  if (wide && fill_up(R, f.cost, path)) {
    quads++;
    rest = 0;
  }
  if (ch.fit >= kSingle) {
    quads = rest = 0;
    for (int r = 0; r < R; r++) s.passes.push_back(PassShape{1, 1, r});
  }
  int most = 1;
  if (wide && quads > 1) {
    most = (int)std::max<uint64_t>(1, std::min<uint64_t>(quads, kMergeArena / std::max<uint64_t>(1, f.arena * 4 * word)));
    const int n = (quads + most - 1) / most;
    most = (quads + n - 1) / n;  // evenly
  }
  for (int q = 0; q < quads; q += most) s.passes.push_back(PassShape{4, std::min(most, quads - q), 4 * q});
  if (rest & 2) s.passes.push_back(PassShape{2, 1, 4 * quads});
  if (rest & 1) s.passes.push_back(PassShape{1, 1, 4 * quads + (rest & 2)});
  const uint64_t res = (uint64_t)s.passes[0].rg * s.passes[0].groups;  // residues of the widest pass
  uint64_t kinds = 0;  // residues and groups of the different passes (their dense descriptors)
  uint64_t kind_groups = 0;
  for (size_t i = 0; i < s.passes.size(); i++) {
    if (i && s.passes[i].rg == s.passes[i - 1].rg && s.passes[i].groups == s.passes[i - 1].groups) continue;
    kinds += (uint64_t)s.passes[i].rg * s.passes[i].groups;
    kind_groups += s.passes[i].groups;
  }
  size_t o = 0;
  auto sect = [&](size_t& off, size_t bytes) {
    off = o;
    o = align_up(o + bytes);
  };
  sect(s.off_leaves, f.leaves * sizeof(LeafDesc));
  sect(s.off_tables, f.tables * sizeof(uint32_t));
  if ((p8 || tc) && f.n_dense && !spare) {
    // contract_group stages its descriptors without gaps: a step on the CUDA cores has
    // one, of at most sizeof(GridStep), a dense one only that of section off_tc
    sect(s.off_steps, (f.nlvl - f.n_dense) * sizeof(GridStep));
    sect(s.off_small, 2048);  // (each array at a multiple of 128 bytes)
  } else {
    sect(s.off_steps, std::max(f.nseq, f.nlvl) * sizeof(GridStep));
    sect(s.off_small, f.nlvl * sizeof(StepDesc));
  }
  // planes and partials: of the largest step (one residue of it on TNC_PATH_TC),
  // or of a level's steps together as far as the limits allow
  // (kSpare: none yet)
  uint64_t part = std::max(std::max(f.split, p8 ? f.parts : 0) * res, std::max(f.kept, tc && !spare ? f.parts : 0));
  uint64_t planes = p8 ? f.planes * res : spare ? 0 : f.planes;
  if (together) {
    for (uint64_t v : f.lvl_parts) part = std::max(part, std::min(v * res, tc ? kTcBytes : kGroupParts));
    for (uint64_t v : f.lvl_planes) planes = std::max(planes, std::min(v * res, tc ? kTcPlanes : kGroupPlanes));
  }
  s.part_bytes = part;
  s.p8_bytes = planes;
  sect(s.off_tc, p8   ? f.n_dense * kind_groups * p8_step_bytes()
                 : tc ? f.n_dense * (spare ? 1 << kMaxChunkLog : kinds) * tc_unit_bytes()
                      : f.n_dense * R * kKeptDenseBytes);
  sect(s.off_part, part);
  sect(s.off_err, 64);
  sect(s.off_results, f.n_out * R * sizeof(uint32_t));
  sect(s.off_limbs, f.n_out * ((31 * R + 31) / 32) * sizeof(uint32_t));
  sect(s.off_p8, planes);
  sect(s.off_arena, f.arena * res * word);
  s.total = o;
  s.n_out = f.n_out;
  s.n_dense = f.n_dense;
  s.arena_entries = f.arena;
  return s;
}

SeqLayout group_layout(const tnc_plan_t* const* plans, int n, int R, Choice ch) {
  Foot sum;
  std::vector<uint64_t> arena_base, res_base, leaf_base, table_base;
  for (int i = 0; i < n; i++) {
    const Foot f = foot_of(plans[i], ch.path);
    leaf_base.push_back(sum.leaves);
    table_base.push_back(sum.tables);
    res_base.push_back(sum.n_out);
    arena_base.push_back(sum.arena);
    sum.add(f);
  }
  SeqLayout s = layout_of(sum, R, ch);
  s.arena_base = std::move(arena_base);
  s.res_base = std::move(res_base);
  s.leaf_base = std::move(leaf_base);
  s.table_base = std::move(table_base);
  return s;
}

// kSpare: the dense steps' scratch is what `budget` leaves beside one residue's
// arena.  Of the sizes of the small residues' section those that a dense step
// needs are tried, the rest is for planes (of a part of the shared values where that is
// all that fits); the one is taken with which most of the multiply-adds run on the tensor
// cores, if that is at least half of them (else one residue at a time costs more
// than it gains).  In workspaces of TNC_PATH_INT64's least, on the CUDA cores
// alone -> this way: cubic VC, n = 180, 8 residues 104.5 -> 27.5 ms and 722 -> 517, 3
// residues 147.8 -> 65.6; n = 160, 3 residues 12.6 -> 8.3; n = 130, 3 residues 1.79 -> 1.90.
SeqLayout spare_layout(const tnc_plan_t* const* plans, int n, int R, size_t budget) {
  SeqLayout s = group_layout(plans, n, R, {TNC_PATH_TC, kSpare});
  std::vector<StepDesc> dense;
  double all = 0, most = 0;
  for (int i = 0; i < n; i++) {
    all += plans[i]->cost.macs;
    for (const StepDesc& d : plans[i]->low.lvl_steps)
      if (tc_eligible(d)) dense.push_back(d);
  }
  uint64_t left = budget > s.total ? (budget - s.total) / kAlign * kAlign : 0, part = 0;
  // (not below the least that needs no such choice: that stays the least)
  if (budget < group_layout(plans, n, R, choices(TNC_PATH_TC).back()).total) left = 0;
  for (const StepDesc& x : dense)
    for (uint32_t c = 0; c <= kMaxChunkLog && tc_eligible(tc_part(x, c, 0)); c++) {
      const uint64_t bytes = align_up(tc_byte_bytes(tc_part(x, c, 0)));
      if (bytes >= left) continue;
      double covered = 0;
      for (const StepDesc& d : dense) {
        uint32_t chunks;
        if (tc_chunks(d, left - bytes, bytes, &chunks)) covered += std::ldexp(1.0, d.ka + d.kb + d.k);
      }
      if (covered > most) {
        most = covered;
        part = bytes;
      }
    }
  if (most < 0.5 * all) {
    s.total = SIZE_MAX;
    return s;
  }
  // (the small residues in place of the section of the K splits, if larger)
  const uint64_t more = part > s.part_bytes ? part - align_up(s.part_bytes) : 0;
  s.part_bytes = std::max(s.part_bytes, part);
  s.p8_bytes = left - more;
  for (size_t* at : {&s.off_err, &s.off_results, &s.off_limbs, &s.off_p8}) *at += more;
  s.off_arena += left;
  s.total += left;
  return s;
}

// The first of the path's choices that fits `budget` bytes (the last one if none does).
SeqLayout fitting_layout(const tnc_plan_t* const* plans, int n, int R, int path, size_t budget) {
  SeqLayout s;
  for (const Choice& ch : choices(path)) {
    s = ch.fit == kSpare ? spare_layout(plans, n, R, budget) : group_layout(plans, n, R, ch);
    if (s.total <= budget) break;
  }
  return s;
}

// Consecutive groups of the plans, [begin, end) ranges: as many plans as fit
// `budget` bytes one residue group at a time, or one plan that fits in any way.
int plan_groups(const tnc_plan_t* const* plans, int n, int R, int path, size_t budget,
                std::vector<std::pair<int, int>>& out) {
  out.clear();
  int b = 0;
  Foot sum;
  for (int i = 0; i < n; i++) {
    Foot f = foot_of(plans[i], path);
    Foot t = sum;
    t.add(f);
    if (i > b && layout_of(t, R, {path, kNarrow}).total > budget) {
      out.push_back({b, i});
      b = i;
      t = f;
    }
    if (i == b && layout_of(f, R, {path, kNarrow}).total > budget) {
      const size_t least = fitting_layout(plans + i, 1, R, path, budget).total;
      if (least > budget)
        return set_error(TNC_ERR_BUFFER, "plan " + std::to_string(i) + " alone needs " + std::to_string(least) +
                                             " bytes of workspace");
    }
    sum = t;
  }
  if (b < n) out.push_back({b, n});
  return TNC_OK;
}

// What a call is given for a group of plans on a path: its first choice, unless
// scratch of very large steps makes that more than twice the least and more than
// kMostExtra above it.  (TNC_PATH_TC, cubic VC with 180 vertices, rank 29: 15 GiB of
// planes above 11 to 17; with 12 GiB as the limit 16 such formulas took 1041 ms
// instead of 930.)
constexpr uint64_t kMostExtra = 16ull << 30;
size_t group_bytes(const tnc_plan_t* const* plans, int n, int R, int path) {
  const size_t least = group_layout(plans, n, R, choices(path).back()).total;
  size_t bytes = least;
  for (const Choice& ch : choices(path)) {
    if (ch.fit == kSpare) continue;  // (has no size of its own)
    bytes = group_layout(plans, n, R, ch).total;
    if (bytes <= least + std::max<uint64_t>(least, kMostExtra)) break;
  }
  return bytes;
}
size_t plan_bytes(const tnc_plan_t* p, int R, int path) { return group_bytes(&p, 1, R, path); }

// One residue group at a time on the CUDA cores (tnc_contract_noalloc).
SeqLayout seq_layout(const tnc_plan_t* p, int R) { return group_layout(&p, 1, R, {TNC_PATH_INT64, kNarrow}); }

int fill_count(tnc_count* out, uint64_t n_out, const Arith& a, const uint32_t* res, const uint32_t* limbs,
               uint32_t flags) {
  out->n_out = (int32_t)n_out;
  out->n_limbs = a.crt.n_limbs;
  out->flags = flags;
  if (out->cap_out < (int32_t)n_out) return set_error(TNC_ERR_BUFFER, "count buffer holds fewer entries than 2^n_open");
  if (out->residues) std::memcpy(out->residues, res, n_out * a.R * sizeof(uint32_t));
  if (out->limbs) {
    if (out->cap_limbs < a.crt.n_limbs) return set_error(TNC_ERR_BUFFER, "need " + std::to_string(a.crt.n_limbs) + " limbs");
    for (uint64_t e = 0; e < n_out; e++) {
      std::memset(out->limbs + e * out->cap_limbs, 0, out->cap_limbs * sizeof(uint32_t));
      std::memcpy(out->limbs + e * out->cap_limbs, limbs + e * a.crt.n_limbs, a.crt.n_limbs * sizeof(uint32_t));
    }
  }
  return TNC_OK;
}

// ---------------------------------------------------- packed descriptors

using tnc_dev::BForm;
using tnc_dev::BLeaf;
using tnc_dev::BStep;
using tnc_dev::Seg;

// Launch configuration of clusters of `ctas` CTAs.
struct ClusterLaunch {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  ClusterLaunch(unsigned grid, unsigned threads, size_t smem, cudaStream_t st, unsigned ctas) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  ClusterLaunch(const ClusterLaunch&) = delete;
};

uint16_t pack_run(int src, int dst, int len) { return (uint16_t)(src | (dst << 5) | (len << 10)); }

// Appends `bytes` at a 16-byte boundary of the blob; returns the offset.
size_t blob_put(std::vector<char>& blob, const void* src, size_t bytes) {
  const size_t at = (blob.size() + 15) / 16 * 16;
  blob.resize(at + bytes);
  if (bytes) std::memcpy(blob.data() + at, src, bytes);
  return at;
}

// One formula's descriptor blob (the sections that batch_kernel copies to
// shared memory) and the fields of its BForm that do not depend on the batch,
// for `threads` threads sharing the formula.
int pack_form(const tnc_plan_t* p, uint32_t threads, std::vector<char>& blob, BForm& f) {
  if (p->tree.nodes.empty()) return set_error(TNC_ERR_INVALID, "batch formula with an empty network");
  if (p->cost.max_rank > 24 || !p->low.lvl_fits)
    return set_error(TNC_ERR_TOO_LARGE, "batch formulas must have plan rank <= 24");
  const Lowered& lw = p->low;
  if (lw.lvl_arena_entries >= (1ull << 32)) return set_error(TNC_ERR_TOO_LARGE, "formula arena above 2^32 entries");
  if (lw.lvl_steps.size() >= 65535) return set_error(TNC_ERR_TOO_LARGE, "more than 65534 steps in one formula");
  std::memset(&f, 0, sizeof(f));
  blob.clear();
  // per level: the share of one of the formula's `threads` lanes (at least
  // 16 products), and per step the lane split sh of its long shared sums: an
  // entry of a step is split over 2^sh lanes so that no lane sums much more
  // than that share
  const uint32_t nlev = lw.lvl_start.empty() ? 0 : (uint32_t)lw.lvl_start.size() - 1;
  std::vector<uint32_t> lvl_log_t(nlev, 4), step_sh(lw.lvl_steps.size(), 0);
  for (uint32_t l = 0; l < nlev; l++) {
    uint64_t work = 0;
    for (uint32_t si = lw.lvl_start[l]; si < lw.lvl_start[l + 1]; si++)
      work += 1ull << (lw.lvl_steps[si].c + lw.lvl_steps[si].k);
    uint32_t log_t = 4;
    while (log_t < 24 && (1ull << log_t) * threads < work) log_t++;
    lvl_log_t[l] = log_t;
    for (uint32_t si = lw.lvl_start[l]; si < lw.lvl_start[l + 1]; si++) {
      const StepDesc& d = lw.lvl_steps[si];
      uint32_t sh = 0;
      while (sh < 5 && sh < d.k && d.k - sh > log_t) sh++;
      step_sh[si] = sh;
    }
  }
  // steps, runs and address deltas.  A lane group of a whole-warp block
  // advances its entry by 2^g (g = 5 - sh): delta[t - g] = w[t] -
  // sum_{g <= j < t} w[j] for the operand weights w[j] of output bit j.
  std::vector<BStep> steps;
  std::vector<uint16_t> runs;
  std::vector<int32_t> dls;  // pairs (A, B)
  for (size_t si = 0; si < lw.lvl_steps.size(); si++) {
    const StepDesc& d = lw.lvl_steps[si];
    BStep bs;
    std::memset(&bs, 0, sizeof(bs));
    bs.a_off = (uint32_t)d.a_off;
    bs.b_off = (uint32_t)d.b_off;
    bs.c_off = (uint32_t)d.c_off;
    bs.c = d.c;
    bs.k = d.k;
    bs.ka = d.ka;
    bs.kb = d.kb;
    if (runs.size() >= 65535 || dls.size() / 2 >= 65535)
      return set_error(TNC_ERR_TOO_LARGE, "formula descriptors beyond 2^16 runs or deltas");
    bs.run0 = (uint16_t)runs.size();
    int64_t wA[32] = {0}, wB[32] = {0};
    if (d.nra != TNC_BITMAP) {
      for (int r = 0; r < d.nra; r++) {
        const TncRun& x = d.map.runs.ra[r];
        runs.push_back(pack_run(x.src, x.dst, x.len));
        for (int q = 0; q < x.len; q++) wA[x.src + q] = 1ll << (x.dst + q);
      }
      for (int r = 0; r < d.nrb; r++) {
        const TncRun& x = d.map.runs.rb[r];
        runs.push_back(pack_run(x.src, x.dst, x.len));
        for (int q = 0; q < x.len; q++) wB[x.src + q] = 1ll << (x.dst + q);
      }
      bs.nra = d.nra;
      bs.nrb = d.nrb;
    } else {
      for (int side = 0; side < 2; side++)
        for (int j = 0; j < d.c; j++)
          if ((d.map.bit[j] >> 7) == side) {
            runs.push_back(pack_run(j, d.map.bit[j] & 63, 1));
            (side ? bs.nrb : bs.nra)++;
            (side ? wB : wA)[j] = 1ll << (d.map.bit[j] & 63);
          }
    }
    const uint32_t g = 5 - step_sh[si];
    bs.g = (uint8_t)g;
    bs.dl0 = (uint16_t)(dls.size() / 2);
    for (uint32_t t = g; t < d.c; t++) {
      int64_t sa = 0, sb = 0;
      for (uint32_t j = g; j < t; j++) {
        sa += wA[j];
        sb += wB[j];
      }
      dls.push_back((int32_t)(wA[t] - sa));
      dls.push_back((int32_t)(wB[t] - sb));
    }
    steps.push_back(bs);
  }
  // segments per level: steps whose entries take 32+ lanes get whole-warp
  // blocks of V entries per lane group (V such that a lane's work is about
  // half the level's share, at most 4); the others share packed segments
  // lane by lane.  Segments are ordered by cost, longest first.
  std::vector<Seg> segs;
  std::vector<uint32_t> items, lvl{0};
  for (uint32_t l = 0; l < nlev; l++) {
    const uint32_t log_t = lvl_log_t[l];
    struct Group {
      uint32_t si, o, sh, cost;
    };
    std::vector<Group> small;
    std::vector<std::pair<uint32_t, Seg>> lsegs;  // (cost, segment)
    for (uint32_t si = lw.lvl_start[l]; si < lw.lvl_start[l + 1]; si++) {
      const StepDesc& d = lw.lvl_steps[si];
      const uint32_t sh = step_sh[si];
      const uint32_t cost = 1u << (d.k - sh);
      const uint32_t nout = 1u << d.c;
      if ((nout << sh) < 32) {
        for (uint32_t o = 0; o < nout; o++) small.push_back(Group{si, o, sh, cost});
        continue;
      }
      const uint32_t G = 32u >> sh;
      uint32_t V = 1;
      while (V < 4 && 2 * V * G <= nout && (2 * V) * cost <= (1u << (log_t - 1))) V *= 2;
      for (uint32_t o0 = 0; o0 < nout; o0 += G * V)
        lsegs.push_back({cost * V, Seg{o0, (uint16_t)si, (uint8_t)V, (uint8_t)sh}});
    }
    // widest groups first: each group then starts at a multiple of its size
    // and never crosses a 32-lane boundary
    std::stable_sort(small.begin(), small.end(), [](const Group& x, const Group& y) {
      return x.sh != y.sh ? x.sh > y.sh : x.cost > y.cost;
    });
    for (size_t g = 0; g < small.size();) {
      const uint32_t first = (uint32_t)items.size();
      uint32_t lanes = 0, cost = 0;
      const uint8_t sh0 = (uint8_t)small[g].sh;
      while (g < small.size() && lanes + (1u << small[g].sh) <= 32) {
        const Group& q = small[g];
        for (uint32_t j = 0; j < (1u << q.sh); j++) items.push_back(q.si | q.o << 16 | j << 21 | q.sh << 26);
        lanes += 1u << q.sh;
        cost = std::max(cost, q.cost);
        g++;
      }
      lsegs.push_back({cost, Seg{first, tnc_dev::kPacked, (uint8_t)lanes, sh0}});
    }
    std::stable_sort(lsegs.begin(), lsegs.end(),
                     [](const std::pair<uint32_t, Seg>& x, const std::pair<uint32_t, Seg>& y) {
                       return x.first > y.first;
                     });
    for (const auto& x : lsegs) segs.push_back(x.second);
    lvl.push_back((uint32_t)segs.size());
  }
  // the blob
  blob_put(blob, steps.data(), steps.size() * sizeof(BStep));
  f.segs_at = (uint32_t)blob_put(blob, segs.data(), segs.size() * sizeof(Seg));
  f.items_at = (uint32_t)blob_put(blob, items.data(), items.size() * sizeof(uint32_t));
  f.runs_at = (uint32_t)blob_put(blob, runs.data(), runs.size() * sizeof(uint16_t));
  f.dl_at = (uint32_t)blob_put(blob, dls.data(), dls.size() * sizeof(int32_t));
  f.lvl_at = (uint32_t)blob_put(blob, lvl.data(), lvl.size() * sizeof(uint32_t));
  blob.resize((blob.size() + 15) / 16 * 16);
  f.blob_n = (uint32_t)(blob.size() / 16);
  f.nlev = nlev;
  f.nleaf = (uint32_t)lw.leaves.size();
  f.n_open = (uint32_t)p->net.open_vars.size();
  f.n_out = 1u << f.n_open;
  f.root_off = (uint32_t)(lw.lvl_steps.empty() ? lw.lvl_leaf_off[p->tree.root] : lw.lvl_root_off);
  f.arena = (uint32_t)lw.lvl_arena_entries;
  return TNC_OK;
}

// The leaves of a formula, their weight tables starting at table0.
void pack_leaves(const Lowered& lw, uint32_t table0, std::vector<BLeaf>& leaves) {
  for (size_t l = 0; l < lw.leaves.size(); l++) {
    BLeaf bl;
    std::memset(&bl, 0, sizeof(bl));
    bl.off = (uint32_t)lw.lvl_leaf_off[l];
    bl.table_off = lw.leaves[l].table_off + table0;
    bl.kind = lw.leaves[l].kind;
    bl.rank = lw.leaves[l].rank;
    leaves.push_back(bl);
  }
}

// ---------------------------------------------------------------- one launch
//
// A small formula on TNC_PATH_INT64 runs as one launch per residue group: one
// cluster contracts it level by level (batch_kernel's heavy-formula form, leaf
// fill and result extraction included) and the last group's launch also runs
// the CRT; descriptors go up in one copy, results come down in one.  The
// launches of contract_group take 3 to 6 us per tree level whatever the
// level's work, and its copies of pageable memory about 10 us each.
// Up to kSoloMax multiply-adds and entries per residue (contract_group behind
// its launches uses all SMs; same box, both ways, 4 residues: 2^12.6 205 ->
// 134 us, 2^15.8 244 -> 135, 2^19.7 256 -> 158, 2^21.9 254 -> 262, 2^24.4
// 328 -> 522), on clusters of 16 CTAs from kSoloWide on (2^19.7: 158 us
// against 180 on 8; 2^15: no difference).
constexpr double kSoloMax = 4e6, kSoloWide = 3e4;
constexpr int kSoloSmem = 160 * 1024;  // most descriptor bytes

}  // namespace

namespace tnc {
struct SoloPack {
  bool ok = false;
  uint32_t ctas = 1;
  std::vector<char> bytes;  // forms, blob, leaves, tables, perms, order: copied to the workspace as they are
  size_t off_blob = 0, off_leaves = 0, off_tables = 0, off_perms = 0, off_order = 0;
  size_t blob_bytes = 0;
  int long_sums = 0;  // steps of the split-K shapes with their sums split over lanes
};
}  // namespace tnc

namespace {

void make_solo(const tnc_plan_t* p, SoloPack& s) {
  const double cost = p->cost.macs + p->cost.entries;
  if (p->tree.nodes.empty() || cost > kSoloMax || p->cost.max_rank > 24 || !p->low.lvl_fits) return;
  s.ctas = cost < kSoloWide ? 8 : 16;
  std::vector<char> blob;
  BForm f;
  if (pack_form(p, 256 * s.ctas, blob, f) != TNC_OK) {  // (descriptor limits: the general path takes it)
    clear_error();
    return;
  }
  std::vector<BLeaf> leaves;
  pack_leaves(p->low, 0, leaves);
  const uint32_t first = 0;
  s.blob_bytes = blob.size();
  blob_put(s.bytes, &f, sizeof(f));
  s.off_blob = blob_put(s.bytes, blob.data(), blob.size());
  s.off_leaves = blob_put(s.bytes, leaves.data(), leaves.size() * sizeof(BLeaf));
  s.off_tables = blob_put(s.bytes, p->low.leaf_tables.data(), p->low.leaf_tables.size() * sizeof(uint32_t));
  s.off_perms = blob_put(s.bytes, p->low.root_perm.data(), p->low.root_perm.size());
  s.off_order = blob_put(s.bytes, &first, sizeof(first));
  const BStep* steps = reinterpret_cast<const BStep*>(blob.data());
  for (size_t i = 0; i < p->low.lvl_steps.size(); i++) s.long_sums += splitk_log(p->low.lvl_steps[i]) > 0 && steps[i].g < 5;
  s.ok = blob.size() <= (size_t)kSoloSmem;
}

// The CRT of n entries: a warp each while that is at most four warps per
// scheduler of the GPU, else a thread each.
void launch_crt(const uint32_t* residues, uint64_t n, const CrtConsts& cc, uint32_t* limbs, cudaStream_t st) {
  if (n <= 2048)
    tnc_dev::crt_warp_kernel<<<(unsigned)((n + 3) / 4), 128, 0, st>>>(residues, n, cc, limbs);
  else
    tnc_dev::crt_kernel<<<(unsigned)std::min<uint64_t>((n + 127) / 128, 1024), 128, 0, st>>>(residues, n, cc, limbs);
  launched(n <= 2048 ? &tnc_kernel_launches::crt_warp : &tnc_kernel_launches::crt);
  g_launches.crt++;
}

// The kernel's limits for clusters of `ctas` CTAs with `smem` bytes of dynamic shared memory each.
template <typename K>
int cluster_limits(K kernel, uint32_t ctas, size_t smem) {
  if (smem > 48 * 1024 - 64) CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSoloSmem));
  if (ctas > 8) CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  return TNC_OK;
}

// Can a cluster of `ctas` CTAs of this kernel be resident?  Asked once per kernel,
// cluster size and device, for the most shared memory.
template <int RG, bool N30>
int solo_fits(uint32_t ctas, bool* fits) {
  static std::atomic<int> known[2][64];  // 0: not asked yet, 1: yes, -1: no
  const auto kernel = tnc_dev::batch_kernel<RG, N30, tnc_dev::kBatchSolo>;
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  std::atomic<int>* at = dev >= 0 && dev < 64 ? &known[ctas > 8][dev] : nullptr;
  int k = at ? at->load(std::memory_order_relaxed) : 0;
  if (!k) {
    if (int rc = cluster_limits(kernel, ctas, kSoloSmem)) return rc;
    const ClusterLaunch cl(ctas, 256, kSoloSmem, nullptr, ctas);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cl.cfg) != cudaSuccess) {
      cudaGetLastError();  // (a size that the device does not have)
      n = 0;
    }
    k = n > 0 ? 1 : -1;
    if (at) at->store(k, std::memory_order_relaxed);
  }
  *fits = k > 0;
  return TNC_OK;
}

// A pass of the one-launch contraction: its primes by residue group.
struct SoloPass {
  tnc_dev::SoloConsts sc{};
  bool near30 = true;
  SoloPass(const PassShape& shape, const Arith& a) {
    for (int g = 0; g < shape.groups; g++) {
      uint32_t gp[4];
      for (int r = 0; r < 4; r++) {
        const int i = shape.col + g * shape.rg + r;
        gp[r] = a.primes[r < shape.rg && i < a.R ? i : shape.col + g * shape.rg];
      }
      sc.mg[g] = tnc_dev::make_mod_group(gp);
      near30 = near30 && sc.mg[g].near30;
    }
  }
};

// CTAs of the clusters that contract the formula: as many as it was packed for, 8 where
// no such cluster can be resident (a partition of the GPU, other work on it),
// 0 where none of 8 can either: the formula then goes level by level.
int solo_ctas(const SoloPack& s, const SeqLayout& L, const std::vector<SoloPass>& passes, uint32_t* ctas) {
  *ctas = 0;
  for (uint32_t c = s.ctas; c >= 8; c -= 8) {  // (16, 8)
    bool all = !inject_hit(TNC_INJECT_CLUSTER);
    for (size_t i = 0; i < passes.size() && all; i++) {
      const int rc = dispatch_rg(L.passes[i].rg, [&](auto rgc) -> int {
        constexpr int RG = decltype(rgc)::value;
        return passes[i].near30 ? solo_fits<RG, true>(c, &all) : solo_fits<RG, false>(c, &all);
      });
      if (rc) return rc;
    }
    if (all) {
      *ctas = c;
      return TNC_OK;
    }
  }
  return TNC_OK;
}

// Enqueues the one-launch contraction (descriptors up, a launch per residue
// group); results and limbs are left in their workspace sections.
int solo_enqueue(const SoloPack& s, uint32_t ctas, std::vector<SoloPass>& passes, const SeqLayout& L, const Arith& a,
                 char* ws, cudaStream_t st) {
  CUDA_TRY(cudaMemcpyAsync(ws, s.bytes.data(), s.bytes.size(), cudaMemcpyHostToDevice, st));
  g_h2d_bytes += s.bytes.size();
  for (size_t i = 0; i < passes.size(); i++) {
    const PassShape& shape = L.passes[i];
    tnc_dev::SoloConsts& sc = passes[i].sc;
    tnc_dev::BatchArgs args{};
    args.forms = (const BForm*)ws;
    args.blobs = (const uint4*)(ws + s.off_blob);
    args.leaves = (const BLeaf*)(ws + s.off_leaves);
    args.tables = (const uint32_t*)(ws + s.off_tables);
    args.perms = (const uint8_t*)(ws + s.off_perms);
    args.order = (const uint32_t*)(ws + s.off_order);
    args.n_forms = args.n_heavy = 1;
    args.results = (uint32_t*)(ws + L.off_results);
    args.garena = (uint32_t*)(ws + L.off_arena);
    args.blob_cap = (uint32_t)s.blob_bytes;
    args.R = a.R;
    args.col = shape.col;
    const bool alone = L.passes.size() == 1 && shape.groups == 1;
    args.limbs = alone ? (uint32_t*)(ws + L.off_limbs) : nullptr;
    sc.heavy_entries = L.arena_entries;
    if (alone) sc.crt = a.crt;
    int rc = dispatch_rg(shape.rg, [&](auto rgc) -> int {
      constexpr int RG = decltype(rgc)::value;
      const auto k = passes[i].near30 ? tnc_dev::batch_kernel<RG, true, tnc_dev::kBatchSolo>
                                      : tnc_dev::batch_kernel<RG, false, tnc_dev::kBatchSolo>;
      if (int rc2 = cluster_limits(k, ctas, s.blob_bytes)) return rc2;
      const ClusterLaunch cl(ctas * (unsigned)shape.groups, 256, s.blob_bytes, st, ctas);
      CUDA_TRY(cudaLaunchKernelEx(&cl.cfg, k, args, sc.mg[0], sc));
      return TNC_OK;
    });
    if (rc) return rc;
    launched(&tnc_kernel_launches::one_launch);
    // the record of the work: the one launch does all of it
    g_launches.leaf_fill++;
    g_launches.level++;
    g_launches.extract++;
    g_launches.splitk += s.long_sums;
  }
  if (L.passes.size() == 1 && L.passes[0].groups == 1) g_launches.crt++;
  else launch_crt((const uint32_t*)(ws + L.off_results), L.n_out, a.crt, (uint32_t*)(ws + L.off_limbs), st);
  CUDA_TRY(cudaGetLastError());
  return TNC_OK;
}

}  // namespace

extern "C" size_t tnc_workspace_bytes(const tnc_plan_t* plan, int32_t n_residues) {
  if (!plan || n_residues < 1 || n_residues > 16) return 0;
  return std::max(plan_bytes(plan, n_residues, TNC_PATH_INT64), plan_bytes(plan, n_residues, TNC_PATH_TC));
}

extern "C" void tnc_set_step_timing(int32_t on) { g_time_dense = on != 0; }

extern "C" int tnc_last_dense_time(double* ms, int32_t* n_steps) {
  if (ms) *ms = g_dense_ms;
  if (n_steps) *n_steps = g_dense_launches;
  return TNC_OK;
}

extern "C" int tnc_last_dense_steps(tnc_dense_step_time* out, int32_t cap, int32_t* n) {
  if (n) *n = (int32_t)g_dense_steps.size();
  if (!out) return TNC_OK;
  if (cap < (int32_t)g_dense_steps.size())
    return set_error(TNC_ERR_BUFFER, "need " + std::to_string(g_dense_steps.size()) + " entries");
  std::copy(g_dense_steps.begin(), g_dense_steps.end(), out);
  return TNC_OK;
}

extern "C" int tnc_last_contract_time(double* device_ms) {
  if (device_ms) *device_ms = g_total_ms;
  return TNC_OK;
}

tnc_launch_counts& tnc::launch_counts() { return g_launches; }
void tnc::launched(int32_t tnc_kernel_launches::*kernel) {
  g_kernels.*kernel += 1;
  g_kernels.total += 1;
}

extern "C" int tnc_last_kernel_launches(tnc_kernel_launches* out) {
  if (!out) return set_error(TNC_ERR_INVALID, "NULL argument");
  *out = g_kernels;
  return TNC_OK;
}

extern "C" int tnc_last_launch_counts(tnc_launch_counts* out) {
  if (!out) return set_error(TNC_ERR_INVALID, "NULL argument");
  *out = g_launches;
  return TNC_OK;
}

extern "C" int tnc_last_io_bytes(uint64_t* h2d_bytes, uint64_t* d2h_bytes) {
  if (h2d_bytes) *h2d_bytes = g_h2d_bytes;
  if (d2h_bytes) *d2h_bytes = g_d2h_bytes;
  return TNC_OK;
}

extern "C" size_t tnc_workspace_bytes_opts(const tnc_plan_t* plan, const tnc_contract_opts* opts) {
  clear_error();
  Arith a;
  if (!plan || make_arith(opts, a)) return 0;
  return plan_bytes(plan, a.R, opts->path);
}

// Residues r of a sum of contractions: acc[e R + r] = (acc + sum_w src_w) mod
// p_r, src_w the w-th of n_src arrays of n residues (all below p < 2^31).
__global__ void residue_add_kernel(uint32_t* __restrict__ acc, const uint32_t* __restrict__ src, uint64_t n,
                                   uint32_t n_src, int R, const __grid_constant__ CrtConsts cc) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t s = acc[i];
    for (uint32_t w = 0; w < n_src; w++) s += src[w * n + i];
    acc[i] = (uint32_t)(s % cc.p[i % R]);
  }
}

// The contraction of a group of plans, their tree levels merged: level l of
// every plan of the group runs together (one launch for all their steps with
// fewer than 2^16 outputs, one launch each for big, split-K and dense steps).
// With sum_into == nullptr every plan's count is finished (CRT, copy to
// outs[i]); otherwise the residues [2^n_open][R] of every plan are added into
// the device buffer sum_into (the plans are the slices of one count) and
// nothing else is returned.
static int contract_group(const tnc_plan_t* const* plans, int n, const tnc_contract_opts* opts, void* dev_ws,
                          size_t ws_bytes, void* cuda_stream, tnc_count* outs, uint32_t* sum_into) {
  if (!plans || n <= 0 || (!outs && !sum_into)) return set_error(TNC_ERR_INVALID, "NULL argument");
  for (int i = 0; i < n; i++)
    if (!plans[i]) return set_error(TNC_ERR_INVALID, "NULL plan");
  Arith a;
  int rc = make_arith(opts, a);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // empty networks (the empty product, 1) are answered on the host
  std::vector<const tnc_plan_t*> work;
  std::vector<int> work_idx;
  for (int i = 0; i < n; i++) {
    if (!plans[i]->tree.nodes.empty()) {
      work.push_back(plans[i]);
      work_idx.push_back(i);
      continue;
    }
    std::vector<uint32_t> res(a.R, 1u), limbs(a.crt.n_limbs, 0u);
    limbs[0] = 1;
    if (sum_into) {
      if (!dev_ws || ws_bytes < (size_t)a.R * 4) return set_error(TNC_ERR_BUFFER, "workspace too small");
      CUDA_TRY(cudaMemcpyAsync(dev_ws, res.data(), a.R * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
      residue_add_kernel<<<1, 64, 0, st>>>(sum_into, (const uint32_t*)dev_ws, (uint64_t)a.R, 1, a.R, a.crt);
      launched(&tnc_kernel_launches::residue_add);
      CUDA_TRY(cudaGetLastError());
      CUDA_TRY(cudaStreamSynchronize(st));
    } else {
      rc = fill_count(&outs[i], 1, a, res.data(), limbs.data(), 0);
      if (rc) return rc;
    }
  }
  if (work.empty()) return TNC_OK;
  const int nw = (int)work.size();
  const SeqLayout L = fitting_layout(work.data(), nw, a.R, opts->path, ws_bytes);
  if (!dev_ws || ws_bytes < L.total) return set_error(TNC_ERR_BUFFER, "workspace smaller than tnc_workspace_bytes");
  if (((uintptr_t)dev_ws) % kAlign) return set_error(TNC_ERR_INVALID, "workspace must be 256-byte aligned");
  if (inject_hit(TNC_INJECT_LAUNCH)) return set_error(TNC_ERR_CUDA, "injected failure (TNC_INJECT_LAUNCH)");
  char* ws = (char*)dev_ws;
  if (nw == 1 && !sum_into && opts->path == TNC_PATH_INT64 && !g_time_dense) {
    std::call_once(work[0]->solo_once, [&] {
      auto s = std::make_shared<SoloPack>();
      make_solo(work[0], *s);
      work[0]->solo = std::move(s);
    });
    const SoloPack& s = *work[0]->solo;
    uint32_t ctas = 0;
    std::vector<SoloPass> passes;
    if (s.ok && s.bytes.size() <= L.off_results) {  // (the descriptor sections and scratch before the results)
      passes.reserve(L.passes.size());
      for (const PassShape& shape : L.passes) passes.emplace_back(shape, a);
      if ((rc = solo_ctas(s, L, passes, &ctas))) return rc;
    }
    if (ctas) {
      rc = solo_enqueue(s, ctas, passes, L, a, ws, st);
      if (rc) return rc;
      std::vector<uint32_t> h((L.off_limbs - L.off_results) / 4 + L.n_out * a.crt.n_limbs);
      CUDA_TRY(cudaMemcpyAsync(h.data(), ws + L.off_results, h.size() * 4, cudaMemcpyDeviceToHost, st));
      g_d2h_bytes += h.size() * 4;
      CUDA_TRY(cudaStreamSynchronize(st));
      if (inject_hit(TNC_INJECT_TIMEOUT)) return set_error(TNC_ERR_TIMEOUT, "a tensor-core step timed out waiting for its MMAs");
      return fill_count(&outs[work_idx[0]], L.n_out, a, h.data(), h.data() + (L.off_limbs - L.off_results) / 4,
                        result_flags(work[0], a));
    }
  }
  // Every plan runs level by level (the tree-level schedule of the lowering);
  // offsets are shifted to the plan's part of the group's arena, tables and
  // results.  All descriptors are staged in one buffer and copied at once.
  const bool p8 = L.path == TNC_PATH_TC_P8;
  const bool tc = L.path == TNC_PATH_TC || p8;
  const int sms = sm_count();
  std::vector<char> stage;
  auto put = [&](const void* src, size_t bytes) {  // 128-byte aligned; returns the offset
    const size_t at = (stage.size() + 127) / 128 * 128;
    stage.resize(at + bytes);
    if (bytes) std::memcpy(stage.data() + at, src, bytes);
    return at;
  };
  std::vector<LeafDesc> leaves;
  std::vector<uint32_t> tables;
  size_t n_lev = 0;
  for (int w = 0; w < nw; w++) {
    const Lowered& lw = work[w]->low;
    for (size_t i = 0; i < lw.leaves.size(); i++) {
      LeafDesc ld = lw.leaves[i];
      ld.off = (p8 ? lw.p8_leaf_off[i] : lw.lvl_leaf_off[i]) + L.arena_base[w];
      ld.table_off += (uint32_t)L.table_base[w];
      leaves.push_back(ld);
    }
    tables.insert(tables.end(), lw.leaf_tables.begin(), lw.leaf_tables.end());
    n_lev = std::max(n_lev, lw.lvl_start.empty() ? (size_t)0 : lw.lvl_start.size() - 1);
  }
  // the group's steps by level: small ones (one index space per level across
  // the plans), big, one-small-operand, split-K and dense ones: each kind one
  // launch per level (split-K and dense steps as many as their scratch holds)
  struct Range {
    uint32_t lo, n, blocks, finals;
  };
  struct Level {
    uint32_t small_lo = 0, small_n = 0, small_work = 0;
    Range grid{}, tile{}, block[3] = {}, outer{};
    std::vector<Range> split;
    std::vector<std::pair<uint32_t, uint32_t>> p8;   // ranges of p8 steps launched together
    std::vector<std::pair<StepDesc, uint32_t>> dense;  // TNC_PATH_TC dense steps, their parts (log2)
  };
  std::vector<Level> lev(n_lev);
  std::vector<GridStep> gsteps;
  std::vector<tnc_dev::OuterStep> outers;
  std::vector<tnc_dev::TileStep> tiles;
  std::vector<tnc_dev::BlockStep> blocked[3];  // by tile shape
  std::vector<StepDesc> small;
  std::vector<P8Step> p8steps;
  const int res_max = L.passes[0].rg * L.passes[0].groups;  // residues of the widest pass
  for (size_t l = 0; l < n_lev; l++) {
    Level& lv = lev[l];
    lv.small_lo = (uint32_t)small.size();
    uint64_t wk = 0;
    std::vector<GridStep> split;
    lv.grid.lo = (uint32_t)gsteps.size();
    lv.outer.lo = (uint32_t)outers.size();
    lv.tile.lo = (uint32_t)tiles.size();
    for (int q = 0; q < 3; q++) lv.block[q].lo = (uint32_t)blocked[q].size();
    uint64_t block_tiles[3] = {0, 0, 0};
    const uint32_t p8_lo = (uint32_t)p8steps.size();
    for (int w = 0; w < nw; w++) {
      const Lowered& lw = work[w]->low;
      if (l + 1 >= lw.lvl_start.size()) continue;
      const uint64_t base = L.arena_base[w];
      for (uint32_t i = lw.lvl_start[l]; i < lw.lvl_start[l + 1]; i++) {
        StepDesc d = p8 ? lw.p8_steps[i] : lw.lvl_steps[i];
        d.a_off += base;
        d.b_off += base;
        d.c_off += base;
        const uint32_t flags = p8 ? p8_flags(lw, i) : 0u;
        if (p8 && p8_eligible(d)) {
          p8steps.push_back(P8Step{d, flags});
        } else if (uint32_t chunks; tc && !p8 && tc_eligible(d) && tc_chunks(d, L.p8_bytes, L.part_bytes, &chunks)) {
          lv.dense.push_back({d, chunks});
        } else if (flags) {
          return set_error(TNC_ERR_INVALID, "internal: direct fp16 planes on a CUDA-core step");
        } else if (outer_eligible(d)) {
          outers.push_back(make_outer_step(d));
          outers.back().block_lo = lv.outer.blocks;
          lv.outer.blocks += outers.back().blocks;
        } else if (splitk_log(d) > 0) {
          split.push_back(make_grid_step(d));
        } else if (const int q = p8 ? -1 : block_shape(d); q >= 0) {
          blocked[q].push_back(q == 0 ? make_block_step<0>(d) : q == 1 ? make_block_step<1>(d) : make_block_step<2>(d));
          blocked[q].back().tile_lo = (uint32_t)block_tiles[q];
          block_tiles[q] += 1ull << (d.c - 11 + q);  // (2^11, 2^10 or 2^9 outputs a tile)
        } else if (tile_eligible(d, p8)) {
          tiles.push_back(make_tile_step(d));
          tiles.back().block_lo = lv.tile.blocks;
          lv.tile.blocks += 1u << (tiles.back().s - 8);  // 256 threads per block
        } else if (d.c >= 16) {
          gsteps.push_back(make_grid_step(d));
          gsteps.back().block_lo = lv.grid.blocks;
          lv.grid.blocks += 1u << (gsteps.back().s - 8);  // 256 threads per block (c >= 16)
        } else {
          d.work_lo = (uint32_t)wk;
          wk += 1u << d.c;
          small.push_back(d);
        }
      }
    }
    if (wk >= (1ull << 32)) return set_error(TNC_ERR_TOO_LARGE, "a merged level has more than 2^32 small outputs");
    lv.small_n = (uint32_t)small.size() - lv.small_lo;
    lv.small_work = (uint32_t)wk;
    lv.grid.n = (uint32_t)gsteps.size() - lv.grid.lo;
    lv.outer.n = (uint32_t)outers.size() - lv.outer.lo;
    lv.tile.n = (uint32_t)tiles.size() - lv.tile.lo;
    for (int q = 0; q < 3; q++) {
      if (block_tiles[q] >= (1ull << 31)) return set_error(TNC_ERR_TOO_LARGE, "a merged level has too many tiles");
      lv.block[q].n = (uint32_t)blocked[q].size() - lv.block[q].lo;
      lv.block[q].blocks = (uint32_t)block_tiles[q];
    }
    // split-K steps: as many per launch as the partials' section holds
    const uint64_t part_cap = L.part_bytes / ((uint64_t)res_max * sizeof(uint32_t));
    for (GridStep& g : split) {
      const uint32_t parts = 1u << (g.d.c + g.log_split);
      if (lv.split.empty() || (uint64_t)lv.split.back().blocks + parts > part_cap)
        lv.split.push_back(Range{(uint32_t)gsteps.size(), 0, 0, 0});
      Range& r = lv.split.back();
      g.block_lo = g.part_off = r.blocks;
      g.final_lo = r.finals;
      r.n++;
      r.blocks += parts;
      r.finals += 1u << g.d.c;
      gsteps.push_back(g);
    }
    // dense steps of the 8-bit-prime path: likewise (one at a time while they
    // are timed)
    uint64_t planes = 0, parts = 0;
    for (uint32_t i = p8_lo; i < (uint32_t)p8steps.size(); i++) {
      const uint64_t pl = p8_scratch_bytes(p8steps[i], res_max), pt = p8_part_bytes(p8steps[i].d, res_max);
      if (lv.p8.empty() || g_time_dense || planes + pl > L.p8_bytes || parts + pt > L.part_bytes ||
          (i - lv.p8.back().first + 1) * L.passes[0].groups > p8_max_steps()) {
        lv.p8.push_back({i, i});
        planes = parts = 0;
      }
      lv.p8.back().second = i + 1;
      planes += pl;
      parts += pt;
    }
  }
  const size_t at_leaves = put(leaves.data(), leaves.size() * sizeof(LeafDesc));
  const size_t at_tables = put(tables.data(), tables.size() * sizeof(uint32_t));
  const size_t at_small = put(small.data(), small.size() * sizeof(StepDesc));
  const size_t at_grid = put(gsteps.data(), gsteps.size() * sizeof(GridStep));
  const size_t at_outer = put(outers.data(), outers.size() * sizeof(tnc_dev::OuterStep));
  size_t at_block[3];
  for (int q = 0; q < 3; q++) at_block[q] = put(blocked[q].data(), blocked[q].size() * sizeof(tnc_dev::BlockStep));
  const size_t at_tile = put(tiles.data(), tiles.size() * sizeof(tnc_dev::TileStep));
  // dense descriptors, for each shape of a pass
  uint32_t* part = (uint32_t*)(ws + L.off_part);
  struct TcLaunch {
    TcBatch b;
    StepDesc first;
  };
  struct Dense {
    int rg, groups;
    std::vector<P8Batch> p8;
    std::vector<std::vector<TcLaunch>> tc;  // by level
    size_t at;
  };
  std::vector<Dense> dense;
  const size_t word = p8 ? 1 : sizeof(uint32_t);
  for (const PassShape& ps : L.passes) {
    if (!tc || (!dense.empty() && dense.back().rg == ps.rg && dense.back().groups == ps.groups)) continue;
    dense.push_back(Dense{ps.rg, ps.groups, {}, {}, 0});
    Dense& dn = dense.back();
    const uint32_t rg = (uint32_t)ps.rg;
    std::vector<char> host;
    const uint64_t group_bytes = L.arena_entries * rg * word;
    for (const Level& lv : lev) {
      for (const auto& r : lv.p8) {
        dn.p8.emplace_back();
        rc = p8_batch(p8steps.data() + r.first, (int)(r.second - r.first), rg, ps.groups, group_bytes,
                      (uint8_t*)(ws + L.off_arena), group_bytes, (uint8_t*)(ws + L.off_p8), (uint8_t*)part, host,
                      dn.p8.back());
        if (rc) return rc;
      }
      dn.tc.emplace_back();
      std::vector<TcUnit> units;  // steps with all residues of a group, or a residue of a step each
      uint64_t planes = 0, bytes = 0;
      uint32_t nr = 0;
      auto flush = [&]() -> int {
        if (units.empty()) return TNC_OK;
        dn.tc.back().push_back(TcLaunch{TcBatch{}, units[0].d});
        const int rc2 = tc_batch(units.data(), (int)units.size(), nr, rg, (uint32_t*)(ws + L.off_arena), group_bytes / 4,
                                 group_bytes, (uint8_t*)(ws + L.off_p8), (uint8_t*)part, host, dn.tc.back().back().b);
        units.clear();
        planes = bytes = 0;
        return rc2;
      };
      for (const auto& [d, chunks] : lv.dense) {
        if (chunks) {  // part after part, a residue at a time; each adds to the ones before
          for (uint32_t gr = 0; gr < (uint32_t)ps.groups * rg; gr++)
            for (uint32_t j = 0; j < 1u << chunks; j++) {
              if ((rc = flush())) return rc;
              nr = 1;
              units.push_back(TcUnit{tc_part(d, chunks, j), gr / rg, gr % rg, j > 0});
            }
          if ((rc = flush())) return rc;
          continue;
        }
        const uint64_t pl = tc_plane_bytes(d), by = tc_byte_bytes(d);
        const uint32_t m = rg * pl <= L.p8_bytes && rg * by <= L.part_bytes ? rg : 1u;
        for (uint32_t gr = 0; gr < (uint32_t)ps.groups * rg; gr += m) {
          if (m != nr || planes + m * pl > L.p8_bytes || bytes + m * by > L.part_bytes ||
              units.size() >= tc_max_units(m) || (g_time_dense && gr == 0))
            if ((rc = flush())) return rc;
          nr = m;
          units.push_back(TcUnit{d, gr / rg, gr % rg, false});
          planes += m * pl;
          bytes += m * by;
        }
      }
      if ((rc = flush())) return rc;
    }
    dn.at = put(host.data(), host.size());
  }
  if (stage.size() > L.off_part) return set_error(TNC_ERR_INVALID, "internal: descriptors beyond their section");
  CUDA_TRY(cudaMemcpyAsync(ws, stage.data(), stage.size(), cudaMemcpyHostToDevice, st));
  g_h2d_bytes += stage.size();
  uint32_t* d_err = (uint32_t*)(ws + L.off_err);
  if (tc) CUDA_TRY(cudaMemsetAsync(d_err, 0, 64, st));  // (the CUDA-core kernels wait for nothing)
  // dense-step events (tnc_set_step_timing), destroyed on every return
  std::vector<cudaEvent_t> dense_events;
  std::vector<tnc_dense_step_time> dense_info;  // shapes of the timed dense launches
  struct EventGuard {
    std::vector<cudaEvent_t>& v;
    ~EventGuard() {
      for (cudaEvent_t e : v) cudaEventDestroy(e);
    }
  } event_guard{dense_events};
  cudaEvent_t whole[2] = {nullptr, nullptr};  // the device work of the whole contraction (timing mode)
  if (g_time_dense) {
    CUDA_TRY(cudaEventCreate(&whole[0]));
    CUDA_TRY(cudaEventCreate(&whole[1]));
    dense_events.push_back(whole[0]);
    dense_events.push_back(whole[1]);
    CUDA_TRY(cudaEventRecord(whole[0], st));
  }
  const GridStep* d_steps = (const GridStep*)(ws + at_grid);
  const StepDesc* d_small = (const StepDesc*)(ws + at_small);
  const tnc_dev::TileStep* d_tile = (const tnc_dev::TileStep*)(ws + at_tile);
  const tnc_dev::OuterStep* d_outer = (const tnc_dev::OuterStep*)(ws + at_outer);
  uint32_t* results = (uint32_t*)(ws + L.off_results);
  std::vector<tnc_dev::Roots> roots;
  for (int w = 0; w < nw; w++) {
    if (w % tnc_dev::kMaxRoots == 0) roots.push_back(tnc_dev::Roots{});
    const Lowered& lw = work[w]->low;
    tnc_dev::Roots& rs = roots.back();
    tnc_dev::Root& rt = rs.r[rs.n++];
    rt.map.n_open = (int)work[w]->net.open_vars.size();
    for (int j = 0; j < rt.map.n_open; j++) rt.map.perm[j] = lw.root_perm[j];
    rt.root_off = L.arena_base[w] + (lw.lvl_steps.empty() ? (p8 ? lw.p8_leaf_off : lw.lvl_leaf_off)[work[w]->tree.root]
                                                          : (p8 ? lw.p8_root_off : lw.lvl_root_off));
    rt.res_lo = L.res_base[w];
    rs.n_entries += 1ull << rt.map.n_open;
  }
  for (const PassShape& shape : L.passes) {
    const unsigned ng = (unsigned)shape.groups;
    tnc_dev::Pass ps{};
    std::vector<uint32_t> primes;  // of the pass; a filled-up group repeats its first
    bool near30 = true;
    for (unsigned g = 0; g < ng; g++) {
      uint32_t gp[4];
      for (int r = 0; r < 4; r++) {
        const int i = shape.col + (int)g * shape.rg + r;
        gp[r] = a.primes[r < shape.rg && i < a.R ? i : shape.col + (int)g * shape.rg];
        if (r < shape.rg) primes.push_back(gp[r]);
      }
      ps.mg[g] = tnc_dev::make_mod_group(gp);
      near30 = near30 && ps.mg[g].near30;
    }
    ps.arena_stride = L.arena_entries * shape.rg;
    ps.part_stride = L.part_bytes / ((uint64_t)res_max * sizeof(uint32_t)) * shape.rg;
    const Dense* dn = nullptr;
    for (const Dense& x : dense)
      if (x.rg == shape.rg && x.groups == shape.groups) dn = &x;
    // one pass over its residue groups; the 8-bit-prime path stores a residue
    // per byte
    auto pass = [&](auto rgc, auto wtag, auto n30tag) -> int {
      constexpr int RG = decltype(rgc)::value;
      using W = typename decltype(wtag)::type;
      constexpr bool N30 = decltype(n30tag)::value;
      W* arena = reinterpret_cast<W*>(ws + L.off_arena);
      const int nl = (int)leaves.size();
      size_t next_p8 = 0;
      const std::vector<char> dense_consts =
          tc && !p8 ? tc_consts(primes.data(), (uint32_t)primes.size()) : std::vector<char>();
      tnc_dev::leaf_fill_kernel<RG, W><<<dim3(std::min(nl, sms * 8), ng), 64, 0, st>>>(
          (const LeafDesc*)(ws + at_leaves), nl, (const uint32_t*)(ws + at_tables), arena, ps);
      launched(&tnc_kernel_launches::leaf_fill);
      // (recorded per residue group, on TNC_PATH_TC per residue)
      g_launches.leaf_fill += tc && !p8 ? std::min((int)ng * RG, a.R - shape.col) : (int)ng;
      // a timed dense launch: events around it and its shape
      auto timed = [&](const StepDesc& d, uint32_t residues, auto&& launch) -> int {
        cudaEvent_t ev[2] = {nullptr, nullptr};
        if (g_time_dense) {
          CUDA_TRY(cudaEventCreate(&ev[0]));
          CUDA_TRY(cudaEventCreate(&ev[1]));
          dense_events.push_back(ev[0]);
          dense_events.push_back(ev[1]);
          CUDA_TRY(cudaEventRecord(ev[0], st));
        }
        if (int rc2 = launch()) return rc2;
        if (g_time_dense) {
          CUDA_TRY(cudaEventRecord(ev[1], st));
          tnc_dense_step_time info{};
          info.macs = std::ldexp(1.0, d.ka + d.kb + d.k);
          info.rows_log2 = d.ka;
          info.cols_log2 = d.kb;
          info.k_log2 = d.k;
          info.residues = (int32_t)residues;
          info.tile_n = (int32_t)p8_tile_width(d);
          info.log_split = (int32_t)p8_split_log(d);
          dense_info.push_back(info);
        }
        return TNC_OK;
      };
      for (const Level& lv : lev) {
        NvtxRange level_range("tnc level");
        if (lv.small_n) {
          const unsigned blocks = (unsigned)std::min<uint64_t>((lv.small_work + 255) / 256, (uint64_t)sms * 8);
          tnc_dev::level_kernel<RG, W, N30><<<dim3(blocks, ng), 256, 0, st>>>(d_small + lv.small_lo, lv.small_n,
                                                                             lv.small_work, arena, ps);
          g_launches.level++;
          launched(&tnc_kernel_launches::level);
        }
        if (lv.outer.n) {
          tnc_dev::outer_kernel<RG, W, N30><<<dim3(lv.outer.blocks, ng), 256, 0, st>>>(d_outer + lv.outer.lo, lv.outer.n,
                                                                                       arena, ps);
          g_launches.outer++;
          launched(&tnc_kernel_launches::outer);
        }
        if constexpr (sizeof(W) == 4) {
          auto blocks = [&](auto shape) -> int {
            constexpr int Q = decltype(shape)::value;
            const Range& r = lv.block[Q];
            if (!r.n) return TNC_OK;
            using B = tnc_dev::Blk<Q>;
            constexpr size_t smem =
                (size_t)tnc_dev::kBlkStages * ((1 << B::LA) + (1 << B::LB)) * tnc_dev::kBlkK * RG * sizeof(uint32_t);
            auto k = tnc_dev::block_kernel<RG, Q, N30>;
            if (smem > 48 * 1024) CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k<<<dim3(std::min(r.blocks, (2u * (unsigned)sms + ng - 1) / ng), ng), 256, smem, st>>>(
                (const tnc_dev::BlockStep*)(ws + at_block[Q]) + r.lo, r.n, r.blocks, arena, ps);
            g_launches.grid_step++;
            launched(Q == 0 ? &tnc_kernel_launches::block_64x32
                            : Q == 1 ? &tnc_kernel_launches::block_32x32 : &tnc_kernel_launches::block_32x16);
            return TNC_OK;
          };
          int rc2 = blocks(std::integral_constant<int, 0>());
          if (!rc2) rc2 = blocks(std::integral_constant<int, 1>());
          if (!rc2) rc2 = blocks(std::integral_constant<int, 2>());
          if (rc2) return rc2;
        }
        if (lv.tile.n) {
          tnc_dev::tile_kernel<RG, W, N30><<<dim3(lv.tile.blocks, ng), 256, 0, st>>>(d_tile + lv.tile.lo, lv.tile.n, arena,
                                                                                     ps);
          g_launches.grid_step++;
          launched(&tnc_kernel_launches::tile);
        }
        if (lv.grid.n) {
          tnc_dev::step_kernel<RG, W, N30><<<dim3(lv.grid.blocks, ng), 256, 0, st>>>(d_steps + lv.grid.lo, lv.grid.n, arena,
                                                                                     ps);
          g_launches.grid_step++;
          launched(&tnc_kernel_launches::step);
        }
        for (const Range& r : lv.split) {
          tnc_dev::splitk_partial_kernel<RG, W, N30><<<dim3(r.blocks, ng), 256, 0, st>>>(d_steps + r.lo, r.n, arena, part,
                                                                                         ps);
          tnc_dev::splitk_final_kernel<RG, W, N30><<<dim3(r.finals, ng), 256, 0, st>>>(d_steps + r.lo, r.n, arena, part, ps);
          g_launches.splitk++;
          launched(&tnc_kernel_launches::splitk_partial);
          launched(&tnc_kernel_launches::splitk_final);
        }
        if (tc && !p8)
          for (const TcLaunch& x : dn->tc[&lv - lev.data()]) {
            NvtxRange dense_range("tnc dense steps");
            if (int rc2 = timed(x.first, x.b.n_units * x.b.nr, [&] {
                  return tc_run(x.b, ws + dn->at, dense_consts, RG, d_err, sms, st);
                }))
              return rc2;
          }
        for (const auto& r : lv.p8) {
          NvtxRange dense_range("tnc dense steps");
          const P8Batch& b = dn->p8[next_p8++];
          if (int rc2 = timed(p8steps[r.first].d, RG * ng, [&] {
                return p8_run(b, ws + dn->at, primes.data(), (uint32_t)primes.size(), RG, d_err, sms, st);
              }))
            return rc2;
        }
      }
      for (const tnc_dev::Roots& rs : roots) {
        const unsigned blocks = (unsigned)std::min<uint64_t>((rs.n_entries + 255) / 256, 1024);
        tnc_dev::extract_kernel<RG, W><<<dim3(blocks, ng), 256, 0, st>>>(arena, ps.arena_stride, rs, results, a.R,
                                                                        shape.col);
        g_launches.extract++;
        launched(&tnc_kernel_launches::extract);
      }
      CUDA_TRY(cudaGetLastError());
      return TNC_OK;
    };
    rc = dispatch_rg(shape.rg, [&](auto rgc) -> int {
      if (p8) return pass(rgc, WordTag<uint8_t>(), std::false_type());
      return near30 ? pass(rgc, WordTag<uint32_t>(), std::true_type())
                       : pass(rgc, WordTag<uint32_t>(), std::false_type());
    });
    if (rc) return rc;
  }
  uint32_t h_err = 0;
  if (sum_into) {  // terms of a sum: add every plan's residues, check the device status
    const uint64_t m = (1ull << roots[0].r[0].map.n_open) * (uint64_t)a.R;  // (the same for every plan)
    residue_add_kernel<<<(unsigned)std::min<uint64_t>((m + 255) / 256, 1024), 256, 0, st>>>(sum_into, results, m,
                                                                                           (uint32_t)nw, a.R, a.crt);
    launched(&tnc_kernel_launches::residue_add);
    CUDA_TRY(cudaGetLastError());
    if (tc) {
      CUDA_TRY(cudaMemcpyAsync(&h_err, d_err, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
      g_d2h_bytes += sizeof(uint32_t);
    }
    CUDA_TRY(cudaStreamSynchronize(st));
    if (inject_hit(TNC_INJECT_TIMEOUT)) h_err = 1;
    if (h_err) return set_error(TNC_ERR_TIMEOUT, "a tensor-core step timed out waiting for its MMAs");
    return TNC_OK;
  }
  uint32_t* limbs = (uint32_t*)(ws + L.off_limbs);
  launch_crt(results, L.n_out, a.crt, limbs, st);
  CUDA_TRY(cudaGetLastError());
  if (g_time_dense) CUDA_TRY(cudaEventRecord(whole[1], st));
  // status, residues and limbs: consecutive sections, one copy
  std::vector<uint32_t> down((L.off_limbs - L.off_err) / 4 + L.n_out * a.crt.n_limbs);
  CUDA_TRY(cudaMemcpyAsync(down.data(), d_err, down.size() * 4, cudaMemcpyDeviceToHost, st));
  g_d2h_bytes += down.size() * 4;
  CUDA_TRY(cudaStreamSynchronize(st));
  const uint32_t *h_res = down.data() + (L.off_results - L.off_err) / 4,
                 *h_limbs = down.data() + (L.off_limbs - L.off_err) / 4;
  h_err = tc ? down[0] : 0u;
  if (inject_hit(TNC_INJECT_TIMEOUT)) h_err = 1;
  if (h_err) return set_error(TNC_ERR_TIMEOUT, "a tensor-core step timed out waiting for its MMAs");
  for (size_t e = 0; e + 1 < dense_events.size(); e += 2) {  // pair 0: the whole contraction
    float ms = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms, dense_events[e], dense_events[e + 1]));
    if (e == 0) {
      g_total_ms += ms;
      continue;
    }
    g_dense_ms += ms;
    g_dense_launches++;
    tnc_dense_step_time info = dense_info[e / 2 - 1];
    info.ms = ms;
    g_dense_steps.push_back(info);
  }
  for (int w = 0; w < nw; w++) {
    rc = fill_count(&outs[work_idx[w]], 1ull << work[w]->net.open_vars.size(), a, h_res + L.res_base[w] * a.R,
                    h_limbs + L.res_base[w] * a.crt.n_limbs, result_flags(work[w], a));
    if (rc) return rc;
  }
  return TNC_OK;
}

// Resets the per-call records (launch counts, copies, timing) of the calling
// thread.
static void reset_records() {
  g_launches = tnc_launch_counts{};
  g_kernels = tnc_kernel_launches{};
  g_h2d_bytes = g_d2h_bytes = 0;
  g_dense_ms = 0.0;
  g_dense_launches = 0;
  g_total_ms = 0.0;
  g_dense_steps.clear();
}

extern "C" int tnc_contract(const tnc_plan_t* plan, const tnc_contract_opts* opts, void* dev_ws, size_t ws_bytes,
                            void* cuda_stream, tnc_count* out) {
  clear_error();
  reset_records();
  NvtxRange range("tnc_contract");
  if (!plan || !out) return set_error(TNC_ERR_INVALID, "NULL argument");
  return contract_group(&plan, 1, opts, dev_ws, ws_bytes, cuda_stream, out, nullptr);
}

// Slices of one count: the sum of the plans' counts (each plan the network of
// the formula with some variables fixed), exact as residues, one CRT at the end.
static size_t sliced_head_bytes(uint64_t n_out, const Arith& a) {
  return align_up(n_out * a.R * sizeof(uint32_t)) + align_up(n_out * a.crt.n_limbs * sizeof(uint32_t));
}

extern "C" size_t tnc_workspace_bytes_sliced(const tnc_plan_t* const* plans, int32_t n, const tnc_contract_opts* opts) {
  clear_error();
  Arith a;
  if (!plans || n <= 0 || make_arith(opts, a)) return 0;
  size_t body = 256;
  for (int i = 0; i < n; i++) {
    if (!plans[i]) return 0;
    body = std::max(body, plan_bytes(plans[i], a.R, opts->path));
  }
  return sliced_head_bytes(1ull << plans[0]->net.open_vars.size(), a) + body;
}

extern "C" int tnc_contract_sliced(const tnc_plan_t* const* plans, int32_t n, const tnc_contract_opts* opts,
                                   void* dev_ws, size_t ws_bytes, void* cuda_stream, tnc_count* out) {
  clear_error();
  reset_records();
  NvtxRange range("tnc_contract_sliced");
  if (!plans || n <= 0 || !out || !opts) return set_error(TNC_ERR_INVALID, "NULL argument");
  Arith a;
  int rc = make_arith(opts, a);
  if (rc) return rc;
  const size_t n_open = plans[0] ? plans[0]->net.open_vars.size() : 0;
  double bound = 0;  // log2 of the sum of the slices' certified bounds
  for (int i = 0; i < n; i++) {
    if (!plans[i]) return set_error(TNC_ERR_INVALID, "NULL plan");
    if (plans[i]->net.open_vars.size() != n_open) return set_error(TNC_ERR_INVALID, "slices differ in open variables");
    const double b = plans[i]->net.log2_bound;
    bound = i == 0 ? b : std::max(bound, b) + std::log2(1.0 + std::exp2(-std::fabs(bound - b)));
  }
  const size_t head = sliced_head_bytes(1ull << n_open, a);
  if (!dev_ws || ws_bytes < head + 256)
    return set_error(TNC_ERR_BUFFER, "workspace smaller than tnc_workspace_bytes_sliced");
  // as many slices at a time as the workspace holds, their levels merged
  std::vector<std::pair<int, int>> grp;
  if ((rc = plan_groups(plans, n, a.R, opts->path, ws_bytes - head, grp))) return rc;
  if (((uintptr_t)dev_ws) % kAlign) return set_error(TNC_ERR_INVALID, "workspace must be 256-byte aligned");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const uint64_t n_out = 1ull << n_open;
  char* ws = (char*)dev_ws;
  uint32_t* acc = (uint32_t*)ws;
  uint32_t* limbs = (uint32_t*)(ws + align_up(n_out * a.R * sizeof(uint32_t)));
  CUDA_TRY(cudaMemsetAsync(acc, 0, n_out * a.R * sizeof(uint32_t), st));
  for (const auto& g : grp) {
    rc = contract_group(plans + g.first, g.second - g.first, opts, ws + head, ws_bytes - head, cuda_stream, nullptr,
                        acc);
    if (rc) return rc;
  }
  launch_crt(acc, n_out, a.crt, limbs, st);
  CUDA_TRY(cudaGetLastError());
  std::vector<uint32_t> down((limbs - acc) + n_out * a.crt.n_limbs);  // residues and limbs: one copy
  CUDA_TRY(cudaMemcpyAsync(down.data(), acc, down.size() * 4, cudaMemcpyDeviceToHost, st));
  g_d2h_bytes += down.size() * 4;
  CUDA_TRY(cudaStreamSynchronize(st));
  return fill_count(out, n_out, a, down.data(), down.data() + (limbs - acc), bound >= a.log2_prod - 1e-9 ? TNC_MAYBE_WRAPPED : 0u);
}

extern "C" size_t tnc_workspace_bytes_many(const tnc_plan_t* const* plans, int32_t n, const tnc_contract_opts* opts,
                                           int32_t group) {
  clear_error();
  Arith a;
  if (!plans || n <= 0 || group <= 0 || make_arith(opts, a)) return 0;
  size_t need = 256;
  for (int i = 0; i < n; i += group) {
    const int m = std::min<int>(group, n - i);
    for (int j = i; j < i + m; j++)
      if (!plans[j]) return 0;
    need = std::max(need, group_bytes(plans + i, m, a.R, opts->path));
  }
  return need;
}

extern "C" size_t tnc_workspace_bytes_below(const tnc_plan_t* const* plans, int32_t n, const tnc_contract_opts* opts,
                                            int32_t sliced, size_t below) {
  clear_error();
  Arith a;
  if (!plans || n <= 0 || make_arith(opts, a)) return 0;
  size_t least = 256;
  std::vector<size_t> need(choices(opts->path).size(), 256);  // of every choice, for the largest plan
  for (int i = 0; i < n; i++) {
    if (!plans[i]) return 0;
    size_t own = SIZE_MAX;
    for (size_t c = 0; c < need.size(); c++) {
      if (choices(opts->path)[c].fit == kSpare) {  // (has no size of its own)
        need[c] = 0;
        continue;
      }
      const size_t b = group_layout(plans + i, 1, a.R, choices(opts->path)[c]).total;
      need[c] = std::max(need[c], b);
      own = std::min(own, b);
    }
    least = std::max(least, own);
  }
  need.push_back(least);
  const size_t head = sliced ? sliced_head_bytes(1ull << plans[0]->net.open_vars.size(), a) : 0;
  size_t most = 0;
  for (size_t b : need)
    if (b && b + head < below) most = std::max(most, b + head);
  return most;
}

extern "C" int tnc_contract_many(const tnc_plan_t* const* plans, int32_t n, const tnc_contract_opts* opts,
                                 void* dev_ws, size_t ws_bytes, void* cuda_stream, tnc_count* outs) {
  clear_error();
  reset_records();
  NvtxRange range("tnc_contract_many");
  if (!plans || n <= 0 || !outs || !opts) return set_error(TNC_ERR_INVALID, "NULL argument");
  Arith a;
  int rc = make_arith(opts, a);
  if (rc) return rc;
  for (int i = 0; i < n; i++)
    if (!plans[i]) return set_error(TNC_ERR_INVALID, "NULL plan");
  std::vector<std::pair<int, int>> grp;
  rc = plan_groups(plans, n, a.R, opts->path, ws_bytes, grp);
  if (rc) return rc;
  for (const auto& g : grp) {
    rc = contract_group(plans + g.first, g.second - g.first, opts, dev_ws, ws_bytes, cuda_stream, outs + g.first,
                        nullptr);
    if (rc) return rc;
  }
  return TNC_OK;
}

// ======================================================================= batch

struct tnc_batch_s {
  std::vector<const tnc_plan_t*> plans;
  Arith a;
  // packed descriptors (host staging in pinned memory, same layout as the
  // workspace prefix starting at off_forms)
  char* staging = nullptr;
  size_t off_queue = 0, off_forms = 0, off_blobs = 0, off_leaves = 0, off_tables = 0, off_perms = 0, off_order = 0,
         off_results = 0, off_limbs = 0, off_arena = 0, total = 0;
  size_t desc_bytes = 0;
  uint32_t n_forms = 0;
  uint32_t n_heavy = 0;      // formulas contracted by whole clusters (the first of the order)
  uint64_t total_out = 0;
  std::vector<uint64_t> res_off;
  uint64_t max_arena = 0;    // entries (of the light formulas, where clusters take the heavy ones)
  uint64_t max_blob = 0;     // bytes of the largest descriptor blob
  uint64_t slot_entries = 0;  // global arena slot of one CTA (entries)
  uint32_t slots = 0;         // arena slots: CTAs any launch shape can have
  uint64_t heavy_entries = 0;  // the same of a cluster, for the heavy formulas
  uint32_t heavy_slots = 0, max_clusters = 0;
  // launch configuration (autotuned)
  int threads = 128;
  int cta_cap = 0;           // CTAs per SM cap (0: as many as fit)
  size_t smem_bytes = 0;     // dynamic shared memory for arenas (per CTA), beyond the blob
  std::vector<int> grid;     // per residue group
  // graph cache
  cudaGraphExec_t gexec = nullptr;
  void* g_ws = nullptr;
  cudaStream_t g_stream = nullptr;
  ~tnc_batch_s() {
    if (gexec) cudaGraphExecDestroy(gexec);
    if (staging) cudaFreeHost(staging);
  }
};

namespace {

constexpr size_t kSmemMax = 227 * 1024;

// Batch formulas contracted by whole clusters: those with more than
// kHeavyShare of the batch's work (multiply-adds and entries) per resident CTA
// (four per SM; per formula where there are fewer), and more than kHeavyLevel
// per tree level; none unless the largest exceeds kHeavyTop.  Measured on 2048
// cubic VC formulas with n = 60 (4 residues; three seeds): no clusters 498-709
// us, shares of 0.5 / 0.7 / 1 / 1.4 / 2: 430 / 365 / 328 / 370 / 520 us; on 700
// with n = 64: 850, 416, 331, 280 us for none / 0.7 / 1 / 1.4; on 777 uneven
// 1-in-3 formulas (2 residues): 1330-3130 us without, 226-545 us with.
// kHeavyLevel: a cluster's barrier per level costs about 0.7 us more than a
// CTA's.  Formulas alone, on a cluster against on one CTA (70 of them, 4
// residues): 0.7-0.9 of the speed below 4000 per level, 0.9-1.0 up to 5500,
// 1.0-1.2 up to 10000, 1.3-1.6 at 20000, 2-3 at 50000.
constexpr uint32_t kClusterCtas = 8;
constexpr double kHeavyShare = 1.2, kHeavyLevel = 5500.0, kHeavyTop = 131072.0;

// Three residues left over are filled up to four where the largest formula has at
// most kFillTop multiply-adds and entries: one launch takes less than one with
// two residues and one with one (3 residues, cubic VC and uneven 1-in-3 formulas,
// 5 to 1500 of them: 1.04-1.5 times the speed with the largest at 3.8e6 or less;
// with 1e7, where its cluster's products count, 0.82-0.97).  With 3 residues
// the arenas double: only up to kFillArena bytes of them.
constexpr double kFillTop = 5e6;
constexpr uint64_t kFillArena = 1ull << 30;

// CTAs of batch_kernel<RG, N30, MODE> per SM for (threads, dynamic shared memory),
// capped at `cap` (0: no cap).  The L1 / shared-memory split is then set to
// the smallest shared-memory share that holds those CTAs, so that the rest of
// the SM's 256 KiB serves as L1 for the formulas' global arenas.
template <int RG, bool N30, int MODE>
int occupancy(int threads, size_t smem, int cap, int* blocks, int* clusters) {
  auto k = tnc_dev::batch_kernel<RG, N30, MODE>;
  // the limit is a property of the kernel, shared by every batch in the
  // process: set it to the device's maximum, not to this batch's need (a batch
  // configured later with smaller descriptors would otherwise make an earlier
  // batch's launches fail)
  int optin = 0, dev0 = 0;
  cudaFuncAttributes fa{};
  CUDA_TRY(cudaGetDevice(&dev0));
  CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev0));
  CUDA_TRY(cudaFuncGetAttributes(&fa, k));
  const int dyn_max = optin - (int)fa.sharedSizeBytes;  // the opt-in limit covers static + dynamic
  if (smem > (size_t)std::max(dyn_max, 0))
    return set_error(TNC_ERR_TOO_LARGE, "batch kernel needs more shared memory than a CTA has");
  CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max));
  CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  int occ = 0;
  CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, smem));
  if (cap > 0) occ = std::min(occ, cap);
  int dev = 0, per_sm = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  CUDA_TRY(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  if (occ > 0 && per_sm > 0) {
    const size_t need = (size_t)occ * (smem + 1024 + 64);
    const int pct = (int)std::min<size_t>(100, (need * 100 + per_sm - 1) / per_sm);
    CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct));
    int occ2 = 0;
    CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, k, threads, smem));
    if (occ2 < occ) CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  }
  *blocks = occ;
  if (MODE != tnc_dev::kBatchCtas && occ > 0) {
    const ClusterLaunch cl(kClusterCtas * (unsigned)sm_count(), (unsigned)threads, smem, nullptr, kClusterCtas);
    CUDA_TRY(cudaOccupancyMaxActiveClusters(clusters, k, &cl.cfg));
  }
  return TNC_OK;
}

// Launch shape for (threads, smem, CTAs per SM cap) on every residue group.
int batch_configure(tnc_batch_t* b, int threads, size_t smem, int cap) {
  const int sms = sm_count();
  std::vector<int> grid;
  for (size_t gi = 0; gi < b->a.groups.rg.size(); gi++) {
    int occ = 0, clusters = 0;
    const bool n30 = b->a.group((int)gi).near30 != 0;
    int rc = dispatch_rg(b->a.groups.rg[gi], [&](auto rgc) -> int {
      constexpr int RG = decltype(rgc)::value;
      const size_t sm = b->max_blob + smem;
      if (b->n_heavy)
        return n30 ? occupancy<RG, true, tnc_dev::kBatchClusters>(threads, sm, cap, &occ, &clusters)
                   : occupancy<RG, false, tnc_dev::kBatchClusters>(threads, sm, cap, &occ, &clusters);
      return n30 ? occupancy<RG, true, tnc_dev::kBatchCtas>(threads, sm, cap, &occ, &clusters)
                 : occupancy<RG, false, tnc_dev::kBatchCtas>(threads, sm, cap, &occ, &clusters);
    });
    if (rc) return rc;
    if (occ <= 0) return set_error(TNC_ERR_TOO_LARGE, "batch kernel does not fit on an SM");
    if (b->n_heavy) {  // clusters resident at once, as many as there is work for
      const int n_light = (int)(b->n_forms - b->n_heavy), cs = (int)kClusterCtas;
      int nc = std::min(clusters, std::max(1, sms * occ / cs));
      nc = std::min(nc, (int)b->n_heavy + (n_light + cs - 1) / cs);  // (the light ones wait for no heavy one)
      nc = std::min(nc, (int)b->max_clusters);
      if (clusters <= 0 || nc <= 0) return set_error(TNC_ERR_TOO_LARGE, "no cluster of the batch kernel fits");
      grid.push_back(nc * cs);
      continue;
    }
    grid.push_back(std::max(1, std::min<int>(std::min<int>(sms * occ, (int)b->n_forms), (int)b->slots)));
  }
  b->threads = threads;
  b->smem_bytes = smem;
  b->cta_cap = cap;
  b->grid = grid;
  if (b->gexec) {
    cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
  }
  return TNC_OK;
}

// Can clusters be resident on the device at all, for every residue group's kernel and
// any launch shape (one CTA per SM)?  Otherwise every formula is a light one.
bool clusters_fit(tnc_batch_t* b) {
  if (inject_hit(TNC_INJECT_CLUSTER)) return false;
  for (size_t gi = 0; gi < b->a.groups.rg.size(); gi++) {
    int occ = 0, clusters = 0;
    const bool n30 = b->a.group((int)gi).near30 != 0;
    const int rc = dispatch_rg(b->a.groups.rg[gi], [&](auto rgc) -> int {
      constexpr int RG = decltype(rgc)::value;
      return n30 ? occupancy<RG, true, tnc_dev::kBatchClusters>(256, kSmemMax - 256, 0, &occ, &clusters)
                 : occupancy<RG, false, tnc_dev::kBatchClusters>(256, kSmemMax - 256, 0, &occ, &clusters);
    });
    if (rc || clusters <= 0) {
      clear_error();
      cudaGetLastError();
      return false;
    }
  }
  return true;
}

int batch_pack(tnc_batch_t* b) {
  const uint32_t n = b->n_forms;
  std::vector<BForm> forms(n);
  std::vector<char> blobs, blob;  // all formulas' blobs, each 16-byte aligned
  std::vector<BLeaf> leaves;
  std::vector<uint32_t> tables;
  std::vector<uint8_t> perms;
  b->res_off.assign(n, 0);
  uint64_t out = 0;
  uint64_t heavy_arena = 0;
  b->max_arena = 8;
  b->max_blob = 16;
  // largest formulas first (longest-processing-time order)
  std::vector<uint32_t> order(n);
  for (uint32_t i = 0; i < n; i++) order[i] = i;
  auto cost = [&](uint32_t i) { return b->plans[i]->cost.macs + b->plans[i]->cost.entries; };
  std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) { return cost(x) > cost(y); });
  double total = 0;
  for (uint32_t i = 0; i < n; i++) total += cost(i);
  // heavy formulas, contracted by whole clusters (batch_kernel)
  const uint32_t ctas = 4u * (uint32_t)sm_count();  // resident at once
  const double share = n <= ctas / kClusterCtas / 2 ? 0.0 : total / std::min(n, ctas);
  if (cost(order[0]) > kHeavyTop && clusters_fit(b)) {
    const auto light = std::stable_partition(order.begin(), order.end(), [&](uint32_t i) {
      return cost(i) > std::max(kHeavyShare * share, kHeavyLevel * (double)(b->plans[i]->low.lvl_start.size() - 1));
    });
    b->n_heavy = (uint32_t)(light - order.begin());
  }
  std::vector<uint32_t> threads(n, 256);
  for (uint32_t i = 0; i < b->n_heavy; i++) threads[order[i]] = 256 * kClusterCtas;
  for (uint32_t i = 0; i < n; i++) {
    const tnc_plan_t* p = b->plans[i];
    const Lowered& lw = p->low;
    BForm& f = forms[i];
    int rc = pack_form(p, threads[i], blob, f);
    if (threads[i] > 256 && (rc || blob.size() > kSmemMax - 256)) {
      // (a cluster's finer segments take up to a few KiB more of descriptors: with
      // one CTA's, which a cluster shares out just as well, the formula fits as a
      // light one does; 256: a CTA's static shared memory and more)
      clear_error();
      rc = pack_form(p, 256, blob, f);
    }
    if (rc) return rc;
    f.blob = (uint32_t)(blobs.size() / 16);
    blobs.insert(blobs.end(), blob.begin(), blob.end());
    b->max_blob = std::max<uint64_t>(b->max_blob, blob.size());
    f.leaf0 = (uint32_t)leaves.size();
    f.res_off = (uint32_t)out;
    f.perm_off = (uint32_t)perms.size();
    b->res_off[i] = out;
    out += f.n_out;
    pack_leaves(lw, (uint32_t)tables.size(), leaves);
    tables.insert(tables.end(), lw.leaf_tables.begin(), lw.leaf_tables.end());
    perms.insert(perms.end(), lw.root_perm.begin(), lw.root_perm.end());
    uint64_t& most = threads[i] > 256 ? heavy_arena : b->max_arena;
    most = std::max<uint64_t>(most, lw.lvl_arena_entries);
  }
  if (blobs.size() / 16 >= (1ull << 32)) return set_error(TNC_ERR_TOO_LARGE, "batch descriptors above 64 GiB");
  b->total_out = out;
  // global arena slots: one per CTA, at most 32 CTAs per SM in any launch
  // shape, of the largest (light) formula's arena; before them one of the
  // largest heavy formula's arena for each cluster that takes heavy formulas.
  // All slots together are no more than formulas, or than CTAs.
  const uint32_t max_ctas = (uint32_t)sm_count() * 32u;
  b->slot_entries = (b->max_arena + 7) / 8 * 8;
  b->heavy_entries = (heavy_arena + 7) / 8 * 8;
  b->max_clusters = max_ctas / kClusterCtas;
  b->heavy_slots = std::min(b->n_heavy, b->max_clusters);
  b->slots = std::min(n - b->n_heavy, max_ctas - b->heavy_slots);
  const uint64_t arena = (uint64_t)b->slots * b->slot_entries + (uint64_t)b->heavy_slots * b->heavy_entries;
  b->a.groups = split_groups(b->a.R, cost(order[0]) <= kFillTop && (b->a.R > 4 || arena * 16 <= kFillArena));
  const int rg_max = b->a.groups.rg.empty() ? 1 : b->a.groups.rg[0];
  // workspace layout
  size_t o = 0;
  auto sect = [&](size_t& off, size_t bytes) {
    off = o;
    o = align_up(o + bytes);
  };
  static_assert(tnc_dev::kSlotCounter >= 16, "at most 16 residue groups, a counter each");
  sect(b->off_queue, 64 * sizeof(uint32_t));
  sect(b->off_forms, forms.size() * sizeof(BForm));
  sect(b->off_blobs, blobs.size());
  sect(b->off_leaves, leaves.size() * sizeof(BLeaf));
  sect(b->off_tables, tables.size() * sizeof(uint32_t));
  sect(b->off_perms, perms.size());
  sect(b->off_order, order.size() * sizeof(uint32_t));
  b->desc_bytes = o - b->off_forms;
  sect(b->off_results, out * b->a.R * sizeof(uint32_t));
  sect(b->off_limbs, out * b->a.crt.n_limbs * sizeof(uint32_t));
  sect(b->off_arena, (size_t)arena * rg_max * sizeof(uint32_t));
  b->total = o;
  CUDA_TRY(cudaMallocHost((void**)&b->staging, std::max<size_t>(b->desc_bytes, 1)));
  std::memset(b->staging, 0, b->desc_bytes);
  char* s = b->staging - b->off_forms;
  auto put = [&](size_t off, const void* src, size_t bytes) {
    if (bytes) std::memcpy(s + off, src, bytes);
  };
  put(b->off_forms, forms.data(), forms.size() * sizeof(BForm));
  put(b->off_blobs, blobs.data(), blobs.size());
  put(b->off_leaves, leaves.data(), leaves.size() * sizeof(BLeaf));
  put(b->off_tables, tables.data(), tables.size() * sizeof(uint32_t));
  put(b->off_perms, perms.data(), perms.size());
  put(b->off_order, order.data(), order.size() * sizeof(uint32_t));
  // default launch shape (the autotuner's usual pick): 256 threads, arenas in
  // global memory, as many CTAs per SM as fit
  if (b->max_blob > kSmemMax) return set_error(TNC_ERR_TOO_LARGE, "a formula's descriptors exceed shared memory");
  return batch_configure(b, 256, 0, 0);
}

int batch_enqueue(tnc_batch_t* b, void* dev_ws, cudaStream_t st) {
  char* ws = (char*)dev_ws;
  CUDA_TRY(cudaMemsetAsync(ws + b->off_queue, 0, 64 * sizeof(uint32_t), st));
  for (size_t gi = 0; gi < b->a.groups.rg.size(); gi++) {
    const int rg = b->a.groups.rg[gi];
    BatchArgs args{};
    args.forms = (const BForm*)(ws + b->off_forms);
    args.blobs = (const uint4*)(ws + b->off_blobs);
    args.leaves = (const BLeaf*)(ws + b->off_leaves);
    args.tables = (const uint32_t*)(ws + b->off_tables);
    args.perms = (const uint8_t*)(ws + b->off_perms);
    args.order = (const uint32_t*)(ws + b->off_order);
    args.n_forms = b->n_forms;
    args.queue = (uint32_t*)(ws + b->off_queue) + gi;
    args.results = (uint32_t*)(ws + b->off_results);
    args.garena = (uint32_t*)(ws + b->off_arena);
    args.slot_entries = b->slot_entries;
    args.blob_cap = (uint32_t)b->max_blob;
    args.smem_cap = (uint32_t)(b->smem_bytes / (rg * sizeof(uint32_t)));
    args.R = b->a.R;
    args.col = b->a.groups.col[gi];
    args.n_heavy = b->n_heavy;
    const tnc_dev::ClusterConsts cc{b->heavy_entries, b->heavy_slots * b->heavy_entries, b->slots};
    const ModGroup mg = b->a.group((int)gi);
    const int grid = b->grid[gi];
    const size_t smem = b->max_blob + b->smem_bytes;
    const int threads = b->threads;
    int rc = dispatch_rg(rg, [&](auto rgc) -> int {
      constexpr int RG = decltype(rgc)::value;
      if (b->n_heavy) {
        const ClusterLaunch cl((unsigned)grid, (unsigned)threads, smem, st, kClusterCtas);
        CUDA_TRY(cudaLaunchKernelEx(
            &cl.cfg,
            mg.near30 ? tnc_dev::batch_kernel<RG, true, tnc_dev::kBatchClusters>
                      : tnc_dev::batch_kernel<RG, false, tnc_dev::kBatchClusters>,
            args, mg, cc));
        return TNC_OK;
      }
      if (mg.near30) tnc_dev::batch_kernel<RG, true><<<grid, threads, smem, st>>>(args, mg, 0);
      else tnc_dev::batch_kernel<RG, false><<<grid, threads, smem, st>>>(args, mg, 0);
      CUDA_TRY(cudaGetLastError());
      return TNC_OK;
    });
    if (rc) return rc;
  }
  tnc_dev::crt_kernel<<<(unsigned)std::max<uint64_t>(1, std::min<uint64_t>((b->total_out + 127) / 128, 4096)), 128, 0,
                        st>>>((const uint32_t*)(ws + b->off_results), b->total_out, b->a.crt,
                              (uint32_t*)(ws + b->off_limbs));
  CUDA_TRY(cudaGetLastError());
  return TNC_OK;
}

}  // namespace

extern "C" int tnc_batch_create(const tnc_plan_t* const* plans, int32_t n, const tnc_contract_opts* opts,
                                tnc_batch_t** out) {
  clear_error();
  if (!plans || n <= 0 || !out) return set_error(TNC_ERR_INVALID, "bad batch arguments");
  *out = nullptr;
  try {
    if (inject_hit(TNC_INJECT_NOMEM)) throw std::bad_alloc();
    auto* b = new tnc_batch_t();
    int rc = make_arith(opts, b->a);
    if (!rc && opts->path == TNC_PATH_TC_P8)
      rc = set_error(TNC_ERR_INVALID, "TNC_PATH_TC_P8 is a tnc_contract path; batches run TNC_PATH_INT64");
    if (!rc) {
      for (int i = 0; i < n; i++) {
        if (!plans[i]) rc = set_error(TNC_ERR_INVALID, "NULL plan in batch");
        b->plans.push_back(plans[i]);
      }
    }
    b->n_forms = (uint32_t)n;
    if (!rc) rc = batch_pack(b);
    if (rc) {
      delete b;
      return rc;
    }
    *out = b;
    return TNC_OK;
  } catch (const std::bad_alloc&) {
    return set_error(TNC_ERR_NOMEM, "out of host memory");
  }
}

extern "C" size_t tnc_batch_workspace_bytes(const tnc_batch_t* b) { return b ? b->total : 0; }

extern "C" int tnc_batch_info(const tnc_batch_t* b, size_t* h2d_bytes, size_t* d2h_bytes, uint64_t* n_entries,
                              int32_t* kernels_per_launch) {
  clear_error();
  if (!b) return set_error(TNC_ERR_INVALID, "batch is NULL");
  if (h2d_bytes) *h2d_bytes = b->desc_bytes;
  if (d2h_bytes) *d2h_bytes = b->total_out * (size_t)(b->a.R + b->a.crt.n_limbs) * sizeof(uint32_t);
  if (n_entries) *n_entries = b->total_out;
  if (kernels_per_launch) *kernels_per_launch = (int32_t)b->a.groups.rg.size() + 1;
  return TNC_OK;
}

extern "C" int tnc_batch_upload(tnc_batch_t* b, void* dev_ws, size_t ws_bytes, void* cuda_stream) {
  clear_error();
  if (!b || !dev_ws) return set_error(TNC_ERR_INVALID, "NULL argument");
  if (ws_bytes < b->total) return set_error(TNC_ERR_BUFFER, "workspace smaller than tnc_batch_workspace_bytes");
  if (((uintptr_t)dev_ws) % kAlign) return set_error(TNC_ERR_INVALID, "workspace must be 256-byte aligned");
  CUDA_TRY(cudaMemcpyAsync((char*)dev_ws + b->off_forms, b->staging, b->desc_bytes, cudaMemcpyHostToDevice,
                           (cudaStream_t)cuda_stream));
  return TNC_OK;
}

extern "C" int tnc_batch_launch(tnc_batch_t* b, void* dev_ws, void* cuda_stream) {
  clear_error();
  if (!b || !dev_ws) return set_error(TNC_ERR_INVALID, "NULL argument");
  if (inject_hit(TNC_INJECT_LAUNCH)) return set_error(TNC_ERR_CUDA, "injected failure (TNC_INJECT_LAUNCH)");
  NvtxRange range("tnc_batch_launch");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (st == nullptr) return batch_enqueue(b, dev_ws, st);  // legacy stream: cannot capture
  if (b->gexec && (b->g_ws != dev_ws || b->g_stream != st)) {
    cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
  }
  if (!b->gexec) {
    CUDA_TRY(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    int rc = batch_enqueue(b, dev_ws, st);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(st, &g);
    if (rc) {
      if (g) cudaGraphDestroy(g);
      return rc;
    }
    if (e != cudaSuccess) return set_error(TNC_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(e));
    e = cudaGraphInstantiate(&b->gexec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      b->gexec = nullptr;
      return set_error(TNC_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
    }
    b->g_ws = dev_ws;
    b->g_stream = st;
  }
  CUDA_TRY(cudaGraphLaunch(b->gexec, st));
  return TNC_OK;
}

extern "C" int tnc_batch_autotune(tnc_batch_t* b, void* dev_ws, void* cuda_stream, int32_t* threads_out,
                                  int32_t* smem_out, int32_t* ctas_out) {
  clear_error();
  if (!b || !dev_ws) return set_error(TNC_ERR_INVALID, "NULL argument");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int rg_max = b->a.groups.rg.empty() ? 1 : b->a.groups.rg[0];
  const size_t need = b->max_arena * rg_max * sizeof(uint32_t);
  std::vector<size_t> smems{0};
  for (size_t s : {16u << 10, 32u << 10, 48u << 10, 64u << 10, 96u << 10, 128u << 10, 192u << 10})
    if (s + b->max_blob <= kSmemMax) smems.push_back(std::min(s, need));
  std::sort(smems.begin(), smems.end());
  smems.erase(std::unique(smems.begin(), smems.end()), smems.end());
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  CUDA_TRY(cudaEventCreate(&e0));
  CUDA_TRY(cudaEventCreate(&e1));
  float best = 1e30f;
  int best_t = b->threads, best_c = b->cta_cap;
  size_t best_s = b->smem_bytes;
  int rc = TNC_OK;
  for (int threads : {64, 128, 256}) {
    for (size_t sm : smems) {
      int prev_grid = -1;
      for (int cap : {0, 2, 1}) {
        rc = batch_configure(b, threads, sm, cap);
        if (rc == TNC_ERR_TOO_LARGE) {
          rc = TNC_OK;
          break;
        }
        if (rc) break;
        if (b->grid[0] == prev_grid) continue;  // the cap changes nothing
        prev_grid = b->grid[0];
        float ms = 1e30f;
        for (int rep = 0; rep < 2 && !rc; rep++) {
          cudaEventRecord(e0, st);
          rc = batch_enqueue(b, dev_ws, st);
          cudaEventRecord(e1, st);
          if (!rc && cudaEventSynchronize(e1) != cudaSuccess) rc = set_error(TNC_ERR_CUDA, "autotune launch failed");
          float t = 0;
          if (!rc) cudaEventElapsedTime(&t, e0, e1);
          if (rep == 1) ms = t;
        }
        if (rc) break;
        if (ms < best) {
          best = ms;
          best_t = threads;
          best_s = sm;
          best_c = cap;
        }
      }
      if (rc) break;
    }
    if (rc) break;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  rc = batch_configure(b, best_t, best_s, best_c);
  if (threads_out) *threads_out = best_t;
  if (smem_out) *smem_out = (int32_t)best_s;
  if (ctas_out) *ctas_out = best_c;
  return rc;
}

extern "C" int tnc_batch_set_launch(tnc_batch_t* b, int32_t threads, int32_t smem_bytes, int32_t ctas_per_sm) {
  clear_error();
  if (!b) return set_error(TNC_ERR_INVALID, "NULL argument");
  if (threads != 64 && threads != 128 && threads != 256)
    return set_error(TNC_ERR_INVALID, "threads must be 64, 128 or 256");
  if (ctas_per_sm < 0) return set_error(TNC_ERR_INVALID, "ctas_per_sm must be >= 0");
  if (smem_bytes < 0 || (size_t)smem_bytes + b->max_blob > kSmemMax)
    return set_error(TNC_ERR_TOO_LARGE, "shared-memory arena too large");
  return batch_configure(b, threads, (size_t)smem_bytes, ctas_per_sm);
}

extern "C" int tnc_batch_get_launch(const tnc_batch_t* b, int32_t* threads, int32_t* smem_bytes,
                                    int32_t* ctas_per_sm) {
  clear_error();
  if (!b) return set_error(TNC_ERR_INVALID, "NULL argument");
  if (threads) *threads = b->threads;
  if (smem_bytes) *smem_bytes = (int32_t)b->smem_bytes;
  if (ctas_per_sm) *ctas_per_sm = b->cta_cap;
  return TNC_OK;
}

extern "C" int tnc_batch_download(tnc_batch_t* b, const void* dev_ws, void* cuda_stream, tnc_count* outs) {
  clear_error();
  if (!b || !dev_ws || !outs) return set_error(TNC_ERR_INVALID, "NULL argument");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  std::vector<uint32_t> res(b->total_out * b->a.R), limbs(b->total_out * b->a.crt.n_limbs);
  CUDA_TRY(cudaMemcpyAsync(res.data(), (const char*)dev_ws + b->off_results, res.size() * 4, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpyAsync(limbs.data(), (const char*)dev_ws + b->off_limbs, limbs.size() * 4, cudaMemcpyDeviceToHost,
                           st));
  CUDA_TRY(cudaStreamSynchronize(st));
  for (uint32_t i = 0; i < b->n_forms; i++) {
    const tnc_plan_t* p = b->plans[i];
    const uint64_t n_out = 1ull << p->net.open_vars.size();
    int rc = fill_count(&outs[i], n_out, b->a, res.data() + b->res_off[i] * b->a.R,
                        limbs.data() + b->res_off[i] * b->a.crt.n_limbs, result_flags(p, b->a));
    if (rc) return rc;
  }
  return TNC_OK;
}

extern "C" int tnc_batch_download_flat(tnc_batch_t* b, const void* dev_ws, void* cuda_stream, uint32_t* residues,
                                       uint32_t* limbs, uint32_t* flags) {
  clear_error();
  if (!b || !dev_ws) return set_error(TNC_ERR_INVALID, "NULL argument");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (residues)
    CUDA_TRY(cudaMemcpyAsync(residues, (const char*)dev_ws + b->off_results, b->total_out * b->a.R * sizeof(uint32_t),
                             cudaMemcpyDeviceToHost, st));
  if (limbs)
    CUDA_TRY(cudaMemcpyAsync(limbs, (const char*)dev_ws + b->off_limbs,
                             b->total_out * b->a.crt.n_limbs * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
  if (flags)
    for (uint32_t i = 0; i < b->n_forms; i++) flags[i] = result_flags(b->plans[i], b->a);
  CUDA_TRY(cudaStreamSynchronize(st));
  return TNC_OK;
}

extern "C" int tnc_batch_status(tnc_batch_t* b, const void* dev_ws, void* cuda_stream) {
  clear_error();
  if (!b || !dev_ws) return set_error(TNC_ERR_INVALID, "NULL argument");
  CUDA_TRY(cudaStreamSynchronize((cudaStream_t)cuda_stream));
  return TNC_OK;
}

extern "C" void tnc_free_batch(tnc_batch_t* b) { delete b; }

extern "C" int tnc_contract_batch(const tnc_plan_t* const* plans, int32_t n, const tnc_contract_opts* opts, void* dev_ws,
                                  size_t ws_bytes, void* cuda_stream, tnc_count* outs) {
  tnc_batch_t* b = nullptr;
  int rc = tnc_batch_create(plans, n, opts, &b);
  if (rc) return rc;
  rc = tnc_batch_upload(b, dev_ws, ws_bytes, cuda_stream);
  if (!rc) rc = batch_enqueue(b, dev_ws, (cudaStream_t)cuda_stream);
  if (!rc) rc = tnc_batch_download(b, dev_ws, cuda_stream, outs);
  tnc_free_batch(b);
  return rc;
}

// =============================================== allocation-free single formula
//
// For callers that must not allocate device memory (see tnc_contract_noalloc
// in tnc.h).  All device scratch -- leaf descriptors, weight tables, step
// descriptors, the tensor arena, residues and CRT limbs -- lives in one
// file-scope array that every GPU loading this library holds until exit.
// Nothing in the path needs it to start zeroed: the leaf fill writes every
// leaf entry, every step writes each output entry before any later step
// reads it, and the residue and limb regions are written in full.  Host-side
// work uses fixed-size stack buffers only.

static __device__ __align__(256) unsigned char g_noalloc_scratch[TNC_NOALLOC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_base[kMaxDevices] = {nullptr};
CUcontext g_noalloc_ctx[kMaxDevices] = {nullptr};

// The driver's current context, fetched through the runtime (no link-time
// dependency on the driver library); nullptr if unavailable.
CUcontext current_context() {
  using GetCtx = CUresult (*)(CUcontext*);
  static GetCtx fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<GetCtx>(p);
  }();
  CUcontext c = nullptr;
  if (!fn || fn(&c) != CUDA_SUCCESS) return nullptr;
  return c;
}

// Device address of the scratch array on the current device.  In host code
// `g_noalloc_scratch` names a host-side shadow, not device memory, so the
// address is looked up once per device, with that device current, and kept
// with the context it belongs to: after a device reset the runtime makes a
// new context (and loads the module again), and the address is looked up
// anew.  (Before the runtime has made a context current the context reads as
// nullptr; the next call then looks the address up once more.)
int noalloc_base(void** out) {
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return set_error(TNC_ERR_INVALID, "device ordinal out of range");
  const CUcontext ctx = current_context();
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_base[dev] || g_noalloc_ctx[dev] != ctx) {
    void* p = nullptr;
    CUDA_TRY(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    if (!p) return set_error(TNC_ERR_CUDA, "cudaGetSymbolAddress returned NULL");
    g_noalloc_base[dev] = p;
    g_noalloc_ctx[dev] = ctx;
  }
  *out = g_noalloc_base[dev];
  return TNC_OK;
}

}  // namespace

extern "C" int tnc_contract_noalloc(const tnc_plan_t* plan, const tnc_contract_opts* opts, void* cuda_stream,
                                    tnc_count* out) {
  clear_error();
  g_launches = tnc_launch_counts{};
  g_kernels = tnc_kernel_launches{};
  NvtxRange range("tnc_contract_noalloc");
  if (!plan || !opts || !out) return set_error(TNC_ERR_INVALID, "NULL argument");
  if (opts->path != TNC_PATH_INT64)
    return set_error(TNC_ERR_INVALID, "tnc_contract_noalloc supports TNC_PATH_INT64 only");
  const int R = opts->n_residues;
  if (R < 1 || R > 16) return set_error(TNC_ERR_INVALID, "n_residues must be in [1, 16]");
  // primes and CRT constants, on the stack
  uint32_t primes[16];
  if (opts->primes) {
    for (int i = 0; i < R; i++) {
      const uint32_t p = opts->primes[i];
      if (p <= (1u << 29) || p >= (1u << 31) || !is_prime_u32(p))
        return set_error(TNC_ERR_INVALID, "primes must be primes in (2^29, 2^31)");
      for (int j = 0; j < i; j++)
        if (primes[j] == p) return set_error(TNC_ERR_INVALID, "primes must be distinct");
      primes[i] = p;
    }
  } else {
    int n = 0;
    for (uint32_t x = kDefaultPrimeBound - 1; n < R; x -= 2)
      if (is_prime_u32(x)) primes[n++] = x;
  }
  CrtConsts cc{};
  cc.R = R;
  double log2_prod = 0;
  for (int i = 0; i < R; i++) {
    const uint32_t p = primes[i];
    cc.p[i] = p;
    cc.mu[i] = ~0ull / p;
    uint64_t prod = 1;
    for (int j = 0; j < i; j++) prod = prod * (primes[j] % p) % p;
    cc.inv[i] = i == 0 ? 1u : powmod(prod, p - 2, p);
    log2_prod += std::log2((double)p);
  }
  cc.n_limbs = (31 * R + 31) / 32;
  int n_groups = 0, grp_rg[16], grp_col[16];
  for (int c = 0, s = 4; s >= 1; s /= 2)
    while (R - c >= s) {
      grp_rg[n_groups] = s;
      grp_col[n_groups++] = c;
      c += s;
    }

  const SeqLayout L = seq_layout(plan, R);
  const uint64_t n_out = L.n_out;
  out->n_out = (int32_t)n_out;
  out->n_limbs = cc.n_limbs;
  out->flags = plan->net.log2_bound >= log2_prod - 1e-9 ? TNC_MAYBE_WRAPPED : 0u;
  if (out->cap_out < (int32_t)n_out) return set_error(TNC_ERR_BUFFER, "count buffer holds fewer entries than 2^n_open");
  if (out->limbs && out->cap_limbs < cc.n_limbs)
    return set_error(TNC_ERR_BUFFER, "need " + std::to_string(cc.n_limbs) + " limbs");
  if (plan->tree.nodes.empty()) {  // empty network: the empty product, 1
    out->flags = 0;
    if (out->residues)
      for (int r = 0; r < R; r++) out->residues[r] = 1u;
    if (out->limbs) {
      std::memset(out->limbs, 0, (size_t)out->cap_limbs * sizeof(uint32_t));
      out->limbs[0] = 1u;
    }
    return TNC_OK;
  }
  if (L.total > (size_t)TNC_NOALLOC_SCRATCH_BYTES)
    return set_error(TNC_ERR_TOO_LARGE, "plan needs " + std::to_string(L.total) +
                                            " bytes of scratch; tnc_contract_noalloc holds " +
                                            std::to_string((size_t)TNC_NOALLOC_SCRATCH_BYTES));
  if (inject_hit(TNC_INJECT_LAUNCH)) return set_error(TNC_ERR_CUDA, "injected failure (TNC_INJECT_LAUNCH)");
  void* base = nullptr;
  int rc = noalloc_base(&base);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  char* ws = (char*)base;

  // descriptors: through small stack buffers (pageable copies return once the
  // source has been staged, so the buffer can be refilled right away)
  {
    LeafDesc buf[64];
    const size_t nl = plan->low.leaves.size();
    for (size_t i0 = 0; i0 < nl; i0 += 64) {
      const size_t m = std::min<size_t>(64, nl - i0);
      for (size_t i = 0; i < m; i++) {
        buf[i] = plan->low.leaves[i0 + i];
        buf[i].off = plan->low.seq_leaf_off[i0 + i];
      }
      CUDA_TRY(cudaMemcpyAsync(ws + L.off_leaves + i0 * sizeof(LeafDesc), buf, m * sizeof(LeafDesc),
                               cudaMemcpyHostToDevice, st));
    }
  }
  if (!plan->low.leaf_tables.empty())
    CUDA_TRY(cudaMemcpyAsync(ws + L.off_tables, plan->low.leaf_tables.data(),
                             plan->low.leaf_tables.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
  {
    GridStep buf[8];
    const size_t ns = plan->low.seq_steps.size();
    for (size_t i0 = 0; i0 < ns; i0 += 8) {
      const size_t m = std::min<size_t>(8, ns - i0);
      for (size_t i = 0; i < m; i++) buf[i] = make_grid_step(plan->low.seq_steps[i0 + i]);  // (a launch each)
      CUDA_TRY(cudaMemcpyAsync(ws + L.off_steps + i0 * sizeof(GridStep), buf, m * sizeof(GridStep),
                               cudaMemcpyHostToDevice, st));
    }
  }
  const GridStep* d_steps = (const GridStep*)(ws + L.off_steps);
  uint32_t* arena = (uint32_t*)(ws + L.off_arena);
  uint32_t* results = (uint32_t*)(ws + L.off_results);
  uint32_t* limbs = (uint32_t*)(ws + L.off_limbs);
  uint32_t* part = (uint32_t*)(ws + L.off_part);
  tnc_dev::Roots roots{};
  roots.n = 1;
  roots.n_entries = n_out;
  roots.r[0].map.n_open = (int)plan->net.open_vars.size();
  for (int j = 0; j < roots.r[0].map.n_open; j++) roots.r[0].map.perm[j] = plan->low.root_perm[j];
  const int nl = (int)plan->low.leaves.size();
  const int sms = sm_count();
  roots.r[0].root_off = plan->low.seq_steps.empty() ? plan->low.seq_leaf_off[plan->tree.root] : plan->low.seq_root_off;
  for (int gi = 0; gi < n_groups; gi++) {
    uint32_t gp[4];
    for (int r = 0; r < 4; r++) gp[r] = r < grp_rg[gi] ? primes[grp_col[gi] + r] : primes[grp_col[gi]];
    tnc_dev::Pass ps{};
    ps.mg[0] = tnc_dev::make_mod_group(gp);
    rc = dispatch_rg(grp_rg[gi], [&](auto rgc) -> int {
      constexpr int RG = decltype(rgc)::value;
      tnc_dev::leaf_fill_kernel<RG><<<std::min(nl, sms * 8), 64, 0, st>>>(
          (const LeafDesc*)(ws + L.off_leaves), nl, (const uint32_t*)(ws + L.off_tables), arena, ps);
      g_launches.leaf_fill++;
      launched(&tnc_kernel_launches::leaf_fill);
      for (size_t i = 0; i < plan->low.seq_steps.size(); i++) {
        const StepDesc& d = plan->low.seq_steps[i];
        const uint32_t ls = splitk_log(d);
        if (ls > 0) {  // few outputs, long shared sum: K split over blocks, as in tnc_contract
          tnc_dev::splitk_partial_kernel<RG><<<(unsigned)(1ull << (d.c + ls)), 256, 0, st>>>(d_steps + i, 1, arena, part,
                                                                                           ps);
          tnc_dev::splitk_final_kernel<RG><<<(unsigned)(1ull << d.c), 256, 0, st>>>(d_steps + i, 1, arena, part, ps);
          g_launches.splitk++;
          launched(&tnc_kernel_launches::splitk_partial);
          launched(&tnc_kernel_launches::splitk_final);
          continue;
        }
        int threads, blocks, sh;
        grid_shape(d.c, &threads, &blocks, &sh);
        tnc_dev::step_kernel<RG><<<blocks, threads, 0, st>>>(d_steps + i, 1, arena, ps);
        g_launches.grid_step++;
        launched(&tnc_kernel_launches::step);
      }
      tnc_dev::extract_kernel<RG><<<(unsigned)std::min<uint64_t>((n_out + 255) / 256, 1024), 256, 0, st>>>(
          arena, 0, roots, results, R, grp_col[gi]);
      g_launches.extract++;
      launched(&tnc_kernel_launches::extract);
      CUDA_TRY(cudaGetLastError());
      return TNC_OK;
    });
    if (rc) return rc;
  }
  tnc_dev::crt_kernel<<<(unsigned)std::min<uint64_t>((n_out + 127) / 128, 1024), 128, 0, st>>>(results, n_out, cc,
                                                                                                limbs);
  g_launches.crt++;
  launched(&tnc_kernel_launches::crt);
  CUDA_TRY(cudaGetLastError());
  if (out->residues)
    CUDA_TRY(cudaMemcpyAsync(out->residues, results, n_out * R * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
  if (out->limbs) {
    std::memset(out->limbs, 0, n_out * (size_t)out->cap_limbs * sizeof(uint32_t));
    CUDA_TRY(cudaMemcpy2DAsync(out->limbs, (size_t)out->cap_limbs * sizeof(uint32_t), limbs,
                               (size_t)cc.n_limbs * sizeof(uint32_t), (size_t)cc.n_limbs * sizeof(uint32_t), n_out,
                               cudaMemcpyDeviceToHost, st));
  }
  CUDA_TRY(cudaStreamSynchronize(st));
  return TNC_OK;
}
