// Dense pairwise steps of TNC_PATH_TC on the 5th-generation tensor cores,
// exact modulo primes below 2^31.
//
// A step C[m,n] = sum_q A[m,q] B[n,q] mod p (A: M x K, B: N x K, u32 residues;
// the bit maps of the lowering make both operands plain column-major
// matrices) is an integer product S = A B^T with 0 <= S < 2^k (p-1)^2, taken
// mod p at the end.  S is computed modulo small primes q_1..q_n (the largest
// below 2^8) whose product exceeds it, each product with exact fp16 operands
// on the GEMM of the 8-bit-prime path (tc_p8.cu), and rebuilt modulo p by the
// Chinese remainder theorem.  That is 9 products up to k = 8 and 10 up to k = 15
// (12 for small steps, tc_small_primes); splitting the residues into 8-bit limbs (fp16 exact, but at most 64
// shared values to an exact fp32 sum) takes 16 products, and 7 accumulators
// folded into integers every 64 shared values.  The dense steps of a cubic VC
// formula with n = 160 (2^34.4 products per residue, 4 residues): 7.09 ms with
// limbs (operands staged by all threads, tensor pipe 15 % active), 3.58 ms
// this way: GEMMs 2.17 (1.37 PFLOP/s on the largest step, 2^13 x 2^10 x 2^11),
// packing 0.75 (2^24 entries 376 us: the integer multiply pipe is 92 % busy, 4.7
// TB/s of HBM), joining 0.66 (its loads' latency; 3.0 TB/s).
//
//   rns_pack_kernel   entries -> one fp16 plane per small prime (balanced)
//   p8_gemm_kernel    four, two or one small primes at a time -> bytes
//   rns_join_kernel   bytes (K-split partials added) -> residues mod p
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "modarith.cuh"
#include "tnc_internal.h"

namespace tnc_rns {

constexpr uint32_t kMaxSmall = 12;
__host__ __device__ constexpr uint32_t small_prime(uint32_t i) {
  constexpr uint32_t q[kMaxSmall] = {251, 241, 239, 233, 229, 227, 223, 211, 199, 197, 193, 191};
  return q[i];
}
// floor(2^39 / q): for x < 2^31, x m / 2^39 is at most x / q and within 2^-8 of it
__host__ __device__ constexpr uint32_t small_magic(uint32_t i) { return (uint32_t)((1ull << 39) / small_prime(i)); }

// The small primes of a step come in groups of 4, 2 and 1 (the residues per
// item of the GEMM): 9 = 4 + 4 + 1, 10 = 4 + 4 + 2, 11 = 4 + 4 + 2 + 1, 12 =
// 4 + 4 + 4.
__host__ __device__ constexpr uint32_t group_size(uint32_t n, uint32_t at) {
  return n - at >= 4 ? 4u : (n - at >= 2 ? 2u : 1u);
}

// The operands of one step for NR consecutive residues of the entries (a, b:
// the first one's word of entry 0, entries `stride` words apart; 2^f rows, 2^k
// shared values, shared index high).  Residue by residue, n planes of operand A
// then n of B: plane i of an operand at + i 2^(f+k), row-contiguous (the
// entries' own order, mn) or, for a column operand of fewer than 64 rows,
// K-contiguous.  Operand `scaled` (0: A, 1: B) carries the reconstruction's factors.
struct alignas(64) PackUnit {
  const uint32_t *a, *b;
  __half* y;
  uint32_t fa, fb, k, n;
  uint32_t mn_a, mn_b, scaled, tile_lo, tiles_a;  // tiles of 1024 entries; the first in the launch; of operand A
};

// The output of one step for those residues: residue by residue, the small
// residues of entry o, group after group, each [K slice][2^c][group size]
// bytes; the residues mod p go to out[o * stride ..].
struct alignas(64) JoinUnit {
  const uint8_t* bytes;
  uint32_t* out;
  uint32_t c, log_split, n, r0;  // r0: the first residue's place among the launch's primes
  uint32_t block_lo, add;        // add: to the residues there (of the shared values before)
};
constexpr uint32_t kTcPrimes = 16;

constexpr uint32_t kMaxUnits = 256;

__device__ __forceinline__ uint32_t find_last(const uint32_t* lo, uint32_t n, uint32_t x) {
  uint32_t a = 0, b = n - 1;
  while (a < b) {
    const uint32_t m = (a + b + 1) >> 1;
    if (lo[m] <= x) a = m;
    else b = m - 1;
  }
  return a;
}

// hi(a b) + c, 32-bit high product
__device__ __forceinline__ uint32_t mad_hi(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// x < 2^31 minus the multiple of q_i nearest to it: |r| <= (q + 1) / 2 (the
// rounded quotient is off by one only within 2^-8 of a half).
template <int I>
__device__ __forceinline__ uint32_t balanced(uint32_t x) {
  return x - (mad_hi(x, small_magic(I), 64u) >> 7) * small_prime(I);
}

// Factors of the reconstruction for n = 9 + i small primes of product Q: w =
// (Q / q_j)^-1 mod q_j.
struct PackConsts {
  uint32_t w[4][kMaxSmall];
};

// Planes of four entries' values x of one residue: the half with bits 0x6400 |
// b is 1024 + b, minus 1152 leaves b - 128 (exact).  With w, the small
// residues are multiplied by w[I].
template <int I>
__device__ __forceinline__ void put_planes(const uint32_t (&x)[4], uint32_t n, __half* y, uint64_t plane,
                                           const uint32_t* w) {
  if constexpr (I < (int)kMaxSmall) {
    if ((uint32_t)I < n) {
      uint32_t h[2], v[4];
#pragma unroll
      for (int j = 0; j < 4; j++) v[j] = balanced<I>(x[j]);
      if (w) {
        const uint32_t f = w[I];
#pragma unroll
        for (int j = 0; j < 4; j++) v[j] = balanced<I>(v[j] * f + 256u * small_prime(I));  // (|v f| < 2^15)
      }
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const uint32_t t = v[2 * j] + 0x64806480u + v[2 * j + 1] * 65536u;
        asm("add.rn.f16x2 %0, %1, %2;" : "=r"(h[j]) : "r"(t), "r"(0xE480E480u));
      }
      *reinterpret_cast<uint2*>(y + (uint64_t)I * plane) = make_uint2(h[0], h[1]);
      put_planes<I + 1>(x, n, y, plane, w);
    }
  }
}

template <int NR>
__device__ __forceinline__ void load_words(const uint32_t* p, uint32_t (&v)[NR]) {
  if constexpr (NR == 4) {
    const uint4 t = *reinterpret_cast<const uint4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else if constexpr (NR == 2) {
    const uint2 t = *reinterpret_cast<const uint2*>(p);
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = *p;
  }
}

// Four entries per thread, so that a plane's writes are 8 bytes per lane; per
// value and small prime a high product, a shift and a multiply-add, half an
// add and half a packed subtraction.  Writes 2 bytes per small prime and
// residue: 18 to 20 bytes where it reads 4 (HBM at 0.69 of the measured copy
// rate: the multiplies bound it).
template <int NR>
__global__ void __launch_bounds__(256) rns_pack_kernel(const PackUnit* __restrict__ units, uint32_t n_units,
                                                       uint32_t n_tiles, uint32_t stride,
                                                       const __grid_constant__ PackConsts pc) {
  __shared__ uint32_t lo[kMaxUnits];
  if (threadIdx.x < n_units) lo[threadIdx.x] = units[threadIdx.x].tile_lo;
  __syncthreads();
  for (uint32_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const PackUnit& u = units[find_last(lo, n_units, t)];
    uint32_t tile = t - u.tile_lo;
    const bool isA = tile < u.tiles_a;
    if (!isA) tile -= u.tiles_a;
    const uint32_t f = isA ? u.fa : u.fb, n = u.n;
    const uint32_t* X = isA ? u.a : u.b;
    const uint64_t plane = 1ull << (f + u.k), pair = (uint64_t)n * ((1ull << (u.fa + u.k)) + (1ull << (u.fb + u.k)));
    __half* Y = u.y + (isA ? 0ull : (uint64_t)n << (u.fa + u.k));
    const uint32_t* w = u.scaled == (isA ? 0u : 1u) ? pc.w[n - 9u] : nullptr;
    uint64_t e0, step, at;  // entries e0, e0 + step, ..; their place in a plane
    if (isA ? u.mn_a : u.mn_b) {
      e0 = at = (uint64_t)tile * 1024u + threadIdx.x * 4u;
      step = 1;
    } else {  // row r, shared values q .. q + 3; a warp takes 8 rows x 16 shared values: a row's 4 lanes write a
              // whole 32-byte sector (lanes along 32 rows: 552 us instead of 132 for 2^22 entries, 4 residues)
      const uint64_t i = (uint64_t)tile * 256u + threadIdx.x, hi = i >> 5;
      const uint64_t r = (hi & ((1u << (f - 3)) - 1u)) * 8u + (i & 7u), q = ((hi >> (f - 3)) * 4u + ((i >> 3) & 3u)) * 4u;
      e0 = (q << f) + r;
      step = 1ull << f;
      at = (r << u.k) + q;
    }
    uint32_t x[4][NR];
#pragma unroll
    for (int j = 0; j < 4; j++) load_words<NR>(X + (e0 + j * step) * stride, x[j]);
#pragma unroll
    for (int r = 0; r < NR; r++) {
      const uint32_t v[4] = {x[0][r], x[1][r], x[2][r], x[3][r]};
      put_planes<0>(v, n, Y + r * pair + at, plane, w);
    }
  }
}

// Constants of the reconstruction for n = 9 + i small primes of product Q and
// each of the pass's primes p, packed for dp4a, four small primes j a word:
// byte b of Q / q_j mod p in c[b]; neg = p - Q mod p.
struct JoinConsts {
  struct {
    uint32_t c[3][4], neg;
  } by_p[4][kTcPrimes];
  uint32_t p[kTcPrimes];
  uint64_t mu[kTcPrimes];
};

// round(2^15 / q_j), four a word (131 .. 172; 0 beyond n: those bytes are 0)
__host__ __device__ constexpr uint32_t inv_word(uint32_t g) {
  uint32_t v = 0;
  for (uint32_t j = 0; j < 4; j++) v |= ((65536u / small_prime(4 * g + j) + 1u) / 2u) << (8 * j);
  return v;
}

// With y_j = S (Q / q_j)^-1 mod q_j, the factor already in the operand's
// planes: S = sum_j y_j Q / q_j - t Q with t = floor(sum_j y_j / q_j).  S / Q <
// 3/4 and each y_j round(2^15 / q_j) is within 2^7 of 2^15 y_j / q_j, so t =
// floor(sum + 1/8) exactly.  The sums are dot products of bytes: five dp4a per
// four small primes (the coefficients by bytes).
template <int NR>
__global__ void __launch_bounds__(256) rns_join_kernel(const JoinUnit* __restrict__ units, uint32_t n_units,
                                                       uint32_t stride, const __grid_constant__ JoinConsts jc) {
  __shared__ uint32_t lo[kMaxUnits];
  if (threadIdx.x < n_units) lo[threadIdx.x] = units[threadIdx.x].block_lo;
  __syncthreads();
  const JoinUnit u = units[find_last(lo, n_units, blockIdx.x)];
  const uint64_t o = (uint64_t)(blockIdx.x - u.block_lo) * 256u + threadIdx.x;
  if (o >> u.c) return;
  const uint32_t n = u.n, n_split = 1u << u.log_split;
  uint32_t res[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) {
    const uint8_t* g = u.bytes + (((uint64_t)r * n) << (u.c + u.log_split));
    uint32_t y[3] = {0, 0, 0};
    if (n_split == 1) {
      y[0] = *reinterpret_cast<const uint32_t*>(g + 4 * o);
      y[1] = *reinterpret_cast<const uint32_t*>(g + (4ull << u.c) + 4 * o);
      const uint8_t* h = g + (8ull << u.c);
      if (n == 9) y[2] = h[o];
      else if (n == 12) y[2] = *reinterpret_cast<const uint32_t*>(h + 4 * o);
      else y[2] = *reinterpret_cast<const uint16_t*>(h + 2 * o);
      if (n == 11) y[2] |= (uint32_t)h[(2ull << u.c) + o] << 16;
    } else {  // add the K slices and reduce again
#pragma unroll
      for (int q4 = 0; q4 < 3; q4++) {
        uint32_t s[4] = {0, 0, 0, 0};
        const uint32_t m = q4 < 2 ? 4u : n - 8u;  // small primes of this word
        for (uint32_t k = 0; k < n_split; k++) {
          const uint64_t e = ((uint64_t)k << u.c) + o;
          uint32_t v;
          if (m == 4) {
            v = *reinterpret_cast<const uint32_t*>(g + 4 * e);
          } else {
            v = m == 1 ? (uint32_t)g[e] : (uint32_t)*reinterpret_cast<const uint16_t*>(g + 2 * e);
            if (m == 3) v |= (uint32_t)g[((2ull << u.c) << u.log_split) + e] << 16;
          }
          s[0] += v & 0xFFu;
          s[1] += (v >> 8) & 0xFFu;
          s[2] += (v >> 16) & 0xFFu;
          s[3] += v >> 24;
        }
        g += ((uint64_t)m << u.c) << u.log_split;
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const uint32_t q = small_prime(4 * q4 + j);
          uint32_t v = s[j] - (__umulhi(s[j], small_magic(4 * q4 + j)) >> 7) * q;
          if (v >= q) v -= q;
          y[q4] |= v << (8 * j);
        }
      }
    }
    const auto& cc = jc.by_p[n - 9u][u.r0 + r];
    uint32_t f = 1u << 12, b[4] = {0, 0, 0, 0};
#pragma unroll
    for (int q4 = 0; q4 < 3; q4++) {
      f = __dp4a(y[q4], inv_word(q4), f);
#pragma unroll
      for (int i = 0; i < 4; i++) b[i] = __dp4a(y[q4], cc.c[q4][i], b[i]);
    }
    const uint64_t acc = (uint64_t)(b[0] + (b[1] << 8)) + ((uint64_t)(b[2] + (b[3] << 8)) << 16) +
                         (uint64_t)(f >> 15) * cc.neg;
    res[r] = tnc_dev::mod_reduce(acc, jc.p[u.r0 + r], jc.mu[u.r0 + r]);
  }
  uint32_t* dst = u.out + o * stride;
  if (u.add) {
    uint32_t old[NR];
    load_words<NR>(dst, old);
#pragma unroll
    for (int r = 0; r < NR; r++) {  // (both below p < 2^31)
      const uint32_t s = res[r] + old[r], p = jc.p[u.r0 + r];
      res[r] = s >= p ? s - p : s;
    }
  }
  if constexpr (NR == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(res[0], res[1], res[2], res[3]);
  else if constexpr (NR == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(res[0], res[1]);
  else *dst = res[0];
}

}  // namespace tnc_rns

namespace tnc {

using tnc_rns::group_size;
using tnc_rns::kMaxSmall;
using tnc_rns::small_prime;

// Can this step run on the tensor cores (possibly with A and B exchanged)?
bool tc_eligible(const StepDesc& d) {
  const int fa = d.ka, fb = d.kb;
  return d.k >= 6 && ((fa >= 7 && fb >= 5) || (fb >= 7 && fa >= 5));
}

// S < 2^(62 + k) (2^(60 + k) for the default primes, which then need one prime
// less for two values of k in eight: not worth a second rule); Q >= 4/3 S.
// Small steps take all 12: three groups of four are one GEMM launch (6 to 8 us)
// where 9 to 11 are two or three, and up to 2^kFewMacs products the extra ones
// take less (2^25 products, one residue: launches of 15 + 10 us -> one of 15).
constexpr uint32_t kFewMacs = 27;
uint32_t tc_small_primes(const StepDesc& d) {
  if (d.ka + d.kb + d.k <= kFewMacs) return kMaxSmall;  // (k <= 15: Q is large enough)
  double bits = 0;
  for (uint32_t n = 0; n < kMaxSmall; n++) {
    bits += std::log2((double)small_prime(n));
    if (n >= 8 && bits >= 62.0 + d.k + 0.4151) return n + 1;
  }
  return 0;
}

uint64_t tc_plane_bytes(const StepDesc& d) {
  return 2ull * tc_small_primes(d) * ((1ull << (d.ka + d.k)) + (1ull << (d.kb + d.k)));
}

uint64_t tc_byte_bytes(const StepDesc& d) { return (uint64_t)tc_small_primes(d) << (d.c + p8_split_log(d)); }

size_t tc_unit_bytes() { return sizeof(tnc_rns::PackUnit) + sizeof(tnc_rns::JoinUnit) + 4 * p8_prob_bytes() + 256; }
uint32_t tc_max_units(uint32_t nr) { return tnc_rns::kMaxUnits / 3 / nr; }  // (up to three groups of four primes a residue)

int tc_batch(const TcUnit* units, int n, uint32_t nr, uint32_t rg, uint32_t* arena0, uint64_t arena_stride,
             uint64_t arena_bytes, uint8_t* planes, uint8_t* bytes, std::vector<char>& host, TcBatch& b) {
  using namespace tnc_rns;
  b = TcBatch{};
  b.nr = nr;
  if (n > (int)tc_max_units(nr)) return set_error(TNC_ERR_INVALID, "internal: too many dense steps in a launch");
  std::vector<PackUnit> packs;
  std::vector<JoinUnit> joins;
  P8Probs probs[3];  // residues per item 4, 2, 1
  uint64_t tiles = 0, blocks = 0;
  for (int i = 0; i < n; i++) {
    const StepDesc& d = units[i].d;
    const uint32_t nq = tc_small_primes(d), ls = p8_split_log(d);
    if (!nq) return set_error(TNC_ERR_TOO_LARGE, "dense step with too many shared values");
    uint32_t* const arena = arena0 + units[i].group * arena_stride;
    if (units[i].r + nr > rg || (nr != 1 && nr != rg) || (units[i].group + 1) * rg > kTcPrimes) return set_error(TNC_ERR_INVALID, "internal: residues outside their pass");
    {
      const uint64_t ea = 1ull << (d.ka + d.k), eb = 1ull << (d.kb + d.k), ec = 1ull << d.c, w = 4ull * rg;
      if ((d.a_off + ea) * w > arena_bytes || (d.b_off + eb) * w > arena_bytes || (d.c_off + ec) * w > arena_bytes)
        return set_error(TNC_ERR_INVALID, "internal: dense step range outside the arena");
    }
    PackUnit pk;
    std::memset(&pk, 0, sizeof(pk));
    pk.a = arena + d.a_off * rg + units[i].r;
    pk.b = arena + d.b_off * rg + units[i].r;
    pk.y = reinterpret_cast<__half*>(planes);
    pk.fa = d.ka;
    pk.fb = d.kb;
    pk.k = d.k;
    pk.n = nq;
    pk.mn_a = p8_operand_mn(d, 0);
    pk.mn_b = p8_operand_mn(d, 1);
    pk.scaled = d.ka <= d.kb ? 0u : 1u;  // (the smaller operand)
    pk.tile_lo = (uint32_t)tiles;
    pk.tiles_a = 1u << (d.ka + d.k - 10);  // (k >= 6, at least 32 rows: whole tiles of 1024 entries)
    tiles += pk.tiles_a + (1ull << (d.kb + d.k - 10));
    packs.push_back(pk);
    JoinUnit ju;
    std::memset(&ju, 0, sizeof(ju));
    ju.bytes = bytes;
    ju.out = arena + d.c_off * rg + units[i].r;
    ju.c = d.c;
    ju.log_split = ls;
    ju.n = nq;
    ju.r0 = units[i].group * rg + units[i].r;
    ju.block_lo = (uint32_t)blocks;
    ju.add = units[i].add;
    blocks += ((1ull << d.c) + 255) / 256;
    joins.push_back(ju);
    for (uint32_t r = 0; r < nr; r++) {
      __half *ya = reinterpret_cast<__half*>(planes), *yb = ya + ((uint64_t)nq << (d.ka + d.k));
      uint8_t* out = bytes;
      for (uint32_t at = 0; at < nq; at += group_size(nq, at)) {
        const uint32_t gs = group_size(nq, at);
        const int rc = p8_gemm_desc(d, gs, ya + ((uint64_t)at << (d.ka + d.k)), yb + ((uint64_t)at << (d.kb + d.k)), out,
                                    at, probs[gs == 4 ? 0 : (gs == 2 ? 1 : 2)]);
        if (rc) return rc;
        out += ((uint64_t)gs << d.c) << ls;
      }
      planes += tc_plane_bytes(d);
      bytes += tc_byte_bytes(d);
    }
    if (units[i].r == 0 && units[i].group == 0 && !units[i].add) {
      b.steps++;
      b.splits += ls > 0;
    }
  }
  if (std::max(tiles, blocks) >= (1ull << 31)) return set_error(TNC_ERR_TOO_LARGE, "dense steps of a level have too many tiles");
  auto put = [&](const void* src, size_t size) {
    const size_t at = size ? (host.size() + 127) / 128 * 128 : host.size();  // (the tensor maps' alignment)
    host.resize(at + size);
    if (size) std::memcpy(host.data() + at, src, size);
    return at;
  };
  b.n_units = (uint32_t)n;
  b.pack_tiles = (uint32_t)tiles;
  b.blocks = (uint32_t)blocks;
  b.pack_off = put(packs.data(), packs.size() * sizeof(PackUnit));
  b.join_off = put(joins.data(), joins.size() * sizeof(JoinUnit));
  for (int g = 0; g < 3; g++)
    for (int v = 0; v < 6; v++) {
      b.gemm[g][v].n = probs[g].n[v];
      b.gemm[g][v].items = (uint32_t)probs[g].items[v];
      b.gemm[g][v].off = put(probs[g].descs[v].data(), probs[g].descs[v].size());
    }
  return TNC_OK;
}

namespace {

uint32_t pow_mod(uint64_t a, uint32_t e, uint32_t p) {
  uint64_t r = 1;
  for (a %= p; e; e >>= 1) {
    if (e & 1) r = r * a % p;
    a = a * a % p;
  }
  return (uint32_t)r;
}

// Product of the first n small primes without the j-th (all of them: j = n), mod p.
uint32_t cofactor(uint32_t n, uint32_t j, uint32_t p) {
  uint64_t x = 1 % p;
  for (uint32_t i = 0; i < n; i++)
    if (i != j) x = x * small_prime(i) % p;
  return (uint32_t)x;
}

const tnc_rns::PackConsts& pack_consts() {
  static const tnc_rns::PackConsts pc = [] {
    tnc_rns::PackConsts c{};
    for (uint32_t n = 9; n <= kMaxSmall; n++)
      for (uint32_t j = 0; j < n; j++)
        c.w[n - 9][j] = pow_mod(cofactor(n, j, small_prime(j)), small_prime(j) - 2, small_prime(j));
    return c;
  }();
  return pc;
}

}  // namespace

std::vector<char> tc_consts(const uint32_t* primes, uint32_t n_primes) {
  tnc_rns::JoinConsts jc;
  std::memset(&jc, 0, sizeof(jc));
  for (uint32_t r = 0; r < std::min(n_primes, tnc_rns::kTcPrimes); r++) {
    jc.p[r] = primes[r];
    jc.mu[r] = ~0ull / primes[r];
    for (uint32_t n = 9; n <= kMaxSmall; n++) {
      for (uint32_t j = 0; j < n; j++) {
        const uint32_t c = cofactor(n, j, primes[r]);
        for (uint32_t i = 0; i < 4; i++) jc.by_p[n - 9][r].c[j / 4][i] |= ((c >> (8 * i)) & 0xFFu) << (8 * (j % 4));
      }
      jc.by_p[n - 9][r].neg = primes[r] - cofactor(n, n, primes[r]);
    }
  }
  const char* p = reinterpret_cast<const char*>(&jc);
  return std::vector<char>(p, p + sizeof(jc));
}

int tc_run(const TcBatch& b, const char* dev, const std::vector<char>& consts, uint32_t rg, uint32_t* dev_err, int sms,
           void* stream) {
  using namespace tnc_rns;
  cudaStream_t st = (cudaStream_t)stream;
  uint32_t small[kMaxSmall];
  for (uint32_t i = 0; i < kMaxSmall; i++) small[i] = small_prime(i);
  const unsigned pack_blocks = (unsigned)std::min<uint64_t>(b.pack_tiles, (uint64_t)sms * 16);
  const PackUnit* pu = reinterpret_cast<const PackUnit*>(dev + b.pack_off);
  if (b.nr == 4) rns_pack_kernel<4><<<pack_blocks, 256, 0, st>>>(pu, b.n_units, b.pack_tiles, rg, pack_consts());
  else if (b.nr == 2) rns_pack_kernel<2><<<pack_blocks, 256, 0, st>>>(pu, b.n_units, b.pack_tiles, rg, pack_consts());
  else rns_pack_kernel<1><<<pack_blocks, 256, 0, st>>>(pu, b.n_units, b.pack_tiles, rg, pack_consts());
  launched(&tnc_kernel_launches::rns_pack);
  for (int v = 6; v-- > 0;)
    for (int g = 0; g < 3; g++)
      if (b.gemm[g][v].n)
        if (int rc = p8_gemm_launch(4u >> g, v, dev + b.gemm[g][v].off, b.gemm[g][v].n, b.gemm[g][v].items, small,
                                    kMaxSmall, dev_err, sms, stream))
          return rc;
  JoinConsts jc;
  std::memcpy(&jc, consts.data(), sizeof(jc));
  const JoinUnit* ju = reinterpret_cast<const JoinUnit*>(dev + b.join_off);
  if (b.nr == 4) rns_join_kernel<4><<<b.blocks, 256, 0, st>>>(ju, b.n_units, rg, jc);
  else if (b.nr == 2) rns_join_kernel<2><<<b.blocks, 256, 0, st>>>(ju, b.n_units, rg, jc);
  else rns_join_kernel<1><<<b.blocks, 256, 0, st>>>(ju, b.n_units, rg, jc);
  launched(&tnc_kernel_launches::rns_join);
  launch_counts().tc_gemm += (int32_t)b.steps;
  launch_counts().tc_split += (int32_t)b.splits;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return set_error(TNC_ERR_CUDA, std::string("tc launch: ") + cudaGetErrorString(e));
  return TNC_OK;
}

}  // namespace tnc
