// FP64-accurate complex GEMM on the BF16 tensor cores (error-free splitting in
// the manner of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012), used for the FP64 filter (also
// grouped over many problems for the batched sequence), the Lanczos block
// product, the Rayleigh-Ritz products, the residual product A V and the
// CholeskyQR products.
//
// Same planar real form as the mixed filter: W = [Ar | Ai] [[Yr, Yi], [-Yi, Yr]].
// The diagonal of A is taken out of the digit planes and applied exactly in
// FP64 in the epilogue (A_ii B_ij): the row scales then follow the off-diagonal
// entries, which keeps their relative precision when A is diagonally dominant.
// Row i of the left operand is scaled by 2^-e_i and column j of the right one
// by 2^-f_j so every entry x has |x| < 1/2, then cut into S = 6 signed 8-bit
// digits, x = sum_s d_s 2^-8s + r with |r| <= 2^-49 and |d_s| <= 128 (the
// balanced base-256 digits of rint(x 2^48), in integer arithmetic); every digit
// is exact in BF16. The product keeps the 21 digit pairs
// (s, t) with s + t <= 7; pair (s, t) contributes at weight 2^-8(s+t).
// Digit products are < 2^14 and exact; the FP32 tensor-memory accumulator of
// one level L = s + t stays an exact integer over a chunk of 256 K values
// (at most (L-1) 2^22 <= 2^24 for L <= 5), so after every chunk the epilogue
// warps move levels 2-5 into exact int64 accumulators (shifted into one common
// scale, at most 2^54 in total; levels 2 and 3, which have one and two pairs,
// every fourth and second chunk) and levels 6-7, whose weights are at most
// 2^-32 of the leading level, into an FP32 accumulator (its rounding is then
// below 2^-56 of the leading level).
// The result is W = 2^(e_i + f_j) (acc 2^-40 + acc67 2^-48), accurate to a few
// units of 2^-48 relative to |A_i.| |Y_.j| per term: FP64-class.
// Extended variant (LMAX = 8): the five pairs of level 8 are kept too (26 pairs
// per K step instead of 21, levels 6-8 drained into a second int64 accumulator
// at weight 2^-64). The dropped pairs then weigh at most 2^-58 instead of 2^-50 of
// 2^(e_i + f_j) per term, so a product over K terms whose result cancels
// almost completely (a Gram of nearly orthonormal columns with entries near 1,
// the residual X - T U of a triangular solve) keeps an error near the digit
// rounding of its operands instead of sqrt(K) 2^-50 of the scales.
//
// Kernel structure (128 x 64 real output tile = 32 complex columns, 10 warps):
//   warp 0    TMA producer: 6 A digit tiles (128 x 32) and 6 B digit tiles
//             (64 x 32) per K block into a 3-stage ring (64B swizzle)
//   warp 1    TMEM allocator and MMA issuer: the 21 (26) digit pairs of a
//             16-wide K step as 13 (21) tcgen05.mma (M=128, N=64 or 128, K=16)
//             on 8 accumulators of 64 TMEM columns; after each 256-wide chunk it
//             hands the accumulators to the epilogue and waits until they are
//             drained
//   warps 2-9 epilogue: warp w owns TMEM lane quarter w % 4 and half of the
//             complex columns; int64/FP32 accumulators in registers; at the
//             end forms the FP64 result and applies the fused update.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdio>
#include <type_traits>
#include <vector>

#include "ozaki.cuh"

namespace chase {
namespace {

constexpr int OS = 6;                    // digits per operand
static_assert(OS == 6, "the epilogue keeps levels 2-5 exact and levels 6-7 in FP32");
constexpr int OS7 = 7;                   // digits of the fine product
constexpr int TM = 128, TN = 64, TK = 32, STAGES = 3;
constexpr int CHUNK_KB = 8;              // K blocks per exact chunk (256 values)
// a chunk's sum of level L is an integer of at most (L - 1) 2^22, so level 2 may
// run over four chunks and level 3 over two before it leaves 2^24
constexpr int kDrain2 = 4, kDrain3 = 2;
constexpr int A_TILE = TM * TK * 2;      // 8 KB per digit
constexpr int B_TILE = TN * TK * 2;      // 4 KB per digit
constexpr int STAGE_BYTES = OS * (A_TILE + B_TILE);  // 72 KB
// ring: three stages of six digits or two of seven
constexpr int stages(int ns) { return ns == OS ? STAGES : 2; }
constexpr int stage_bytes(int ns) { return ns * (A_TILE + B_TILE); }
static_assert(stages(OS7) * stage_bytes(OS7) <= STAGES * STAGE_BYTES, "one shared-memory size");
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr int NTHREADS = 320;
constexpr uint32_t TMEM_COLS = 512;
constexpr int KPAD = 128;                // K-half padding: 2 Np is a multiple of 256
constexpr int HC = TN / 4;               // complex columns per epilogue warp half (16)
constexpr int CT = TN / 2;               // complex columns per tile (32)
constexpr int kEpiThreads = 256;         // epilogue warps' threads
static_assert(2 * HC * kEpiThreads * 16 <= STAGES * STAGE_BYTES, "the sums fit the ring");
constexpr unsigned long long kWaitLimitNs = 4000000000ull;
constexpr unsigned kGroup = 8;           // row blocks per sweep of the column tiles

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err, int code) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  while (true) {
    if (mbar_try(bar, parity)) return true;
    if (globaltimer() - t0 > kWaitLimitNs) {
      atomicExch(err, code);
      return false;
    }
  }
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
// K-major operand, 64-byte swizzle: 8-row x 64-byte atoms, SBO = 512 B.
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}
// FP32 accumulate, BF16 A and B, both K-major, M = TM, N = n columns.
constexpr uint32_t idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(TM >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t id,
                                          uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}
// TMEM accumulators (TN columns each). Levels that get a neighbour's product
// in the same MMA lie side by side; a primed slot takes the one pair of its
// level that has no neighbour (added in the epilogue). An accumulator is only
// ever written by MMAs of one shape and one destination, which execute in issue
// order.
template <int LMAX> struct Slots;
template <> struct Slots<7> {
  static constexpr int L2 = 0, L3 = 1, L4 = 2, L5 = 3, L6 = 4, L7 = 5, L5b = 6, L7b = 7;
};
template <> struct Slots<8> {
  static constexpr int L2 = 0, L3 = 1, L4 = 2, L5 = 3, L6 = 4, L7 = 5, L8 = 6, L7b = 7;
};
// The digit pairs of one 16-wide K step. An MMA of N = 64 moves 6 KB of
// operands through shared memory in the 32 cycles its products take, more than
// the 128 bytes a cycle it has; one of N = 128 moves 8 KB in 64. So A digit s
// meets B digits t and t + 1 in one MMA wherever the two results are neighbours
// (the B digit tiles lie one after the other, their 64 rows are whole swizzle
// atoms). 36 filter steps with N = 9273 and up to 316 columns: 132 ms with 21
// MMAs of N = 64 and every level drained per chunk, 99 ms so.
// r2, r3, r: this step restarts levels 2, 3 and the others.
template <int LMAX, int NS>
__device__ __forceinline__ void digit_pairs(uint32_t tmem, uint32_t sa, uint32_t sb, bool r2,
                                            bool r3, bool r) {
  using S = Slots<LMAX>;
  auto one = [&](int slot, int s, int t, bool restart) {
    umma_bf16(tmem + (uint32_t)(slot * TN), sdesc_sw64(sa + (s - 1) * A_TILE),
              sdesc_sw64(sb + (t - 1) * B_TILE), idesc(TN), restart ? 0u : 1u);
  };
  auto two = [&](int slot, int s, int t, bool restart) {  // digits t, t + 1
    umma_bf16(tmem + (uint32_t)(slot * TN), sdesc_sw64(sa + (s - 1) * A_TILE),
              sdesc_sw64(sb + (t - 1) * B_TILE), idesc(2 * TN), restart ? 0u : 1u);
  };
  one(S::L2, 1, 1, r2);
  one(S::L3, 1, 2, r3);
  one(S::L3, 2, 1, false);
  if constexpr (LMAX == 7) {
#pragma unroll
    for (int s = 1; s <= 3; ++s) two(S::L4, s, 4 - s, r && s == 1);
    one(S::L5b, 4, 1, r);
  } else {
#pragma unroll
    for (int s = 1; s <= 3; ++s) one(S::L4, s, 4 - s, r && s == 1);
#pragma unroll
    for (int s = 1; s <= 4; ++s) one(S::L5, s, 5 - s, r && s == 1);
  }
#pragma unroll
  for (int s = 1; s <= 5; ++s) two(S::L6, s, 6 - s, r && s == 1);
  one(S::L7b, 6, 1, r);
  if constexpr (LMAX == 8) {
#pragma unroll
    for (int s = 8 - NS; s <= NS; ++s) one(S::L8, s, 8 - s, r && s == 8 - NS);
  }
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}
// 16 consecutive TMEM columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// acc += v 2^SH for an integer-valued v of at most 2^24
template <int SH>
__device__ __forceinline__ void add_level(long long& acc, float v) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(__float2int_rn(v)), "r"(1 << SH));
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// B^T row of complex column j: tiles of CT complex columns, TN rows each,
// real parts first.
__device__ __forceinline__ int64_t brow_re(int64_t j) { return (j / CT) * TN + (j % CT); }

struct Params {
  int64_t N, Np, j0, ncols;   // rows, padded K half, first active column, end column
  int64_t brows;              // rows of one B digit plane
  int64_t arows;              // rows of one A digit plane (= N)
  const int* escale_a;        // per row: exponent e_i
  const double2* diag;        // diagonal of A, applied exactly in FP64
  const double2* Bsrc;        // right operand in FP64 (absolute columns, ld ldbs)
  int64_t ldbs;
  const int* escale_b;        // per complex column: exponent f_j
  int mode;                   // EPI_STORE / EPI_FILTER / EPI_RESID
  double alpha, beta, gamma;  // filter
  const double2* X;           // filter/resid: B operand in FP64 (ld ldx)
  int64_t ldx;
  double2* Y;                 // store/filter destination (ld ldy)
  int64_t ldy;
  const double* theta;        // resid
  double* partial;            // resid: [32-row tile + col * ceil(N / 32)]
  int* err;
  const int* skip;            // seven digits: the product is not formed where this is set
  int nrow, ncol;             // tiles
  int split;                  // CTAs that share a tile's K range
};

// ------------------------------------------------- dependent launches
// The kernels of a product (column exponents, digits, MMAs) follow each other in the
// stream by the dozen and are short, so each may be launched while its predecessor
// still runs (programmatic stream serialization): its CTAs get onto free SMs, the
// product kernel sets up its barriers and tensor memory, and then every thread waits
// here until the predecessor has finished and its writes are visible. Every kernel
// of the chain waits before its first access, so finishing implies that all before
// it have finished too. 20 filter steps with 512 rows: 0.57 -> 0.49 ms.
__device__ __forceinline__ void wait_for_predecessor() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void let_successor_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ------------------------------------------------------- cluster helpers
// Cluster-wide barrier (release / acquire): every thread of every CTA arrives.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Rank in the cluster of part 0 of this CTA's tile.
__device__ __forceinline__ unsigned cluster_base(int split, unsigned part) {
  return split > 1 ? cluster_rank() - part : 0u;
}
// The same shared-memory variable in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t remote_smem(const void* p, unsigned rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ long long ld_cluster(uint32_t a, long long*) {
  long long v;
  asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float ld_cluster(uint32_t a, float*) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

// (acc 2^24 + low) 2^(e - 64), rounded to nearest even, in integer operations (the
// FP64 pipe's conversions and adds took most of a tile's epilogue).
__device__ __forceinline__ double fixed_to_double(long long acc, long long low, int e) {
  acc += low >> 24;
  unsigned lo = (unsigned)low & 0xffffffu;
  const bool neg = acc < 0;
  if (neg) {
    acc = lo ? ~acc : -acc;
    lo = lo ? (1u << 24) - lo : 0u;
  }
  const unsigned long long A = (unsigned long long)acc;
  const int n = __clzll((long long)A);
  unsigned long long W;
  unsigned rest = 0;
  int ex = e - 64;
  if (n >= 24) {
    W = (A << 24) | lo;
  } else {
    const int sh = 24 - n;
    W = (A << n) | (lo >> sh);
    rest = lo & ((1u << sh) - 1u);
    ex += sh;
  }
  if (W == 0) return 0.0;
  const int z = __clzll((long long)W);
  W <<= z;
  ex -= z;
  unsigned long long m = W >> 11;  // 53 bits
  const unsigned tail = (unsigned)W & 0x7ffu;
  if (tail > 0x400u || (tail == 0x400u && (rest != 0 || (m & 1)))) ++m;
  const int E = ex + 1086;
  if (E < 1 || E > 2045) {
    const double v = ldexp((double)m, ex + 11);
    return neg ? -v : v;
  }
  return __longlong_as_double((long long)((((unsigned long long)E << 52) + (m - (1ull << 52))) |
                                          ((unsigned long long)neg << 63)));
}
__device__ __forceinline__ long long low_fixed(long long v) { return v; }
__device__ __forceinline__ long long low_fixed(float v) { return __float2ll_rn(v * 65536.0f); }

// ---------------------------------------------------------------- kernel
// CTA `local` of a product: tile local / split (128 x 64 outputs), part local %
// split of its K blocks; the per-problem kernel and the grouped kernel (the filter
// steps of many problems in one launch) both run it. The CTAs of a tile are
// consecutive ranks of a cluster: each leaves its sums in its own shared memory
// and then adds up and finishes 1 / split of the tile's columns. clustered: the
// launch has clusters of more than one CTA, all of which meet at the two cluster
// barriers; CTAs past the last tile (padding of a group's problem) only do that.
template <int LMAX, int NS>
__device__ __forceinline__ void ozaki_tile(const CUtensorMap* tmA, const CUtensorMap* tmB,
                                           const Params& P, unsigned local, bool maps_in_global,
                                           bool clustered) {
  const unsigned part = local % (unsigned)P.split;
  if (local / (unsigned)P.split >= (unsigned)P.nrow * (unsigned)P.ncol) {
    cluster_sync();
    cluster_sync();
    return;
  }
  unsigned rb, ct;  // row block and column tile (grouped raster order)
  grouped_tile(local / (unsigned)P.split, (unsigned)P.nrow, (unsigned)P.ncol, kGroup, rb, ct);
  constexpr int kStages = stages(NS), kStage = stage_bytes(NS);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
  // [0,S) full, [S,2S) empty, [2S] accumulators full, [2S+1] accumulators empty
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 2);
  __shared__ int s_abort;

  // the epilogue's sums, in the ring once that is free: [2 HC][kEpiThreads]
  using Acc67 = typename std::conditional<LMAX == 8, long long, float>::type;
  long long* acc_s = reinterpret_cast<long long*>(smem);
  Acc67* low_s = reinterpret_cast<Acc67*>(acc_s + 2 * HC * kEpiThreads);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t m0 = (int64_t)rb * TM;
  const int64_t tile = P.j0 / CT + ct;            // absolute CT-column tile
  const int nkb_all = (int)((2 * P.Np) / TK);
  const int kb0 = (int)part * nkb_all / P.split;  // this CTA's K blocks, its chunks from there
  int nkb = ((int)part + 1) * nkb_all / P.split - kb0;
  int nchunks = (nkb + CHUNK_KB - 1) / CHUNK_KB;

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&bars[s]), 1);
      mbar_init(smem_u32(&bars[kStages + s]), 1);
    }
    mbar_init(smem_u32(&bars[2 * kStages]), 1);
    mbar_init(smem_u32(&bars[2 * kStages + 1]), 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  wait_for_predecessor();

  // a product that is not to be formed (the same in every CTA) has no K blocks
  bool go = true;
  if constexpr (NS == OS7) {
    go = *P.skip == 0;
    if (!go) nkb = nchunks = 0;
  }
  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------ TMA producer
      if (maps_in_global) {  // tensor maps read from global memory by the TMA unit
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(tmA)
                     : "memory");
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(tmB)
                     : "memory");
      }
      int issued = 0;
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % kStages;
        const uint32_t ph = (uint32_t)(kb / kStages) & 1u;
        if (!mbar_wait(smem_u32(&bars[kStages + s]), ph ^ 1u, P.err, 11)) {
          s_abort = 1;
          break;
        }
        if (*(volatile int*)&s_abort) break;
        const uint32_t full = smem_u32(&bars[s]);
        uint8_t* st = smem + s * kStage;
        mbar_expect_tx(full, kStage);
        const int kx = (kb0 + kb) * TK;
#pragma unroll
        for (int d = 0; d < NS; ++d) {
          // digit planes are stacked along rows: digit d of row r is row d * rows + r
          tma_load_2d(smem_u32(st + d * A_TILE), tmA, kx, (int)(d * P.arows + m0), full);
        }
#pragma unroll
        for (int d = 0; d < NS; ++d) {
          tma_load_2d(smem_u32(st + NS * A_TILE + d * B_TILE), tmB, kx,
                      (int)(d * P.brows + tile * TN), full);
        }
        ++issued;
      }
      for (int kb = issued > kStages ? issued - kStages : 0; kb < issued; ++kb)
        mbar_wait(smem_u32(&bars[kb % kStages]), (uint32_t)(kb / kStages) & 1u, P.err, 12);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------ MMA issuer
      int kb = 0;
      bool ok = true;
      for (int c = 0; c < nchunks && ok; ++c) {
        if (c > 0 && !mbar_wait(smem_u32(&bars[2 * kStages + 1]), (uint32_t)(c - 1) & 1u, P.err, 13)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int kc = 0; kc < CHUNK_KB && kb < nkb; ++kc, ++kb) {
          const int s = kb % kStages;
          const uint32_t ph = (uint32_t)(kb / kStages) & 1u;
          if (!mbar_wait(smem_u32(&bars[s]), ph, P.err, 14) || *(volatile int*)&s_abort) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st = smem_u32(smem + s * kStage);
#pragma unroll
          for (int kk = 0; kk < TK / 16; ++kk) {
            const uint32_t off = kk * 32;
            // levels restart often enough to stay exact integers: see kDrain2, kDrain3
            const bool r = kc == 0 && kk == 0;
            digit_pairs<LMAX, NS>(tmem, st + off, st + NS * A_TILE + off, r && c % kDrain2 == 0,
                              r && c % kDrain3 == 0, r);  // c = 0 restarts all
          }
          umma_commit(smem_u32(&bars[kStages + s]));
        }
        umma_commit(smem_u32(&bars[2 * kStages]));  // chunk c ready
      }
      if (!ok) {
        s_abort = 1;
        umma_commit(smem_u32(&bars[2 * kStages]));
      }
    }
  } else {
    // ------------------------------------------------------- epilogue warps
    const int q = warp & 3;                   // TMEM lane quarter
    const int h = (warp - 2) >> 2;            // complex column half: [h HC, h HC + HC)
    const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16);
    long long acc[2 * HC];                    // re[0..16), im[16..32): levels 2-5, weight 2^-40
    // levels 6-LMAX. In FP32 at weight 2^-48; in the extended variant in int64 at
    // weight 2^-64: its products are Grams whose diagonal adds squared digits
    // coherently (sum_k d_3(x_k)^2 grows like K), where FP32 sums over
    // K = 80000 lost about 2^-44 of the scale (orthogonality 2e-11 at
    // N = 40000 after CholeskyQR2); per chunk the values stay below 2^25.
    Acc67 acc67[2 * HC];
#pragma unroll
    for (int j = 0; j < 2 * HC; ++j) {
      acc[j] = 0;
      acc67[j] = Acc67(0);
    }
    for (int c = 0; c < nchunks; ++c) {
      const bool ok = mbar_wait(smem_u32(&bars[2 * kStages]), (uint32_t)c & 1u, P.err, 15);
      go = __all_sync(0xffffffffu, ok && !*(volatile int*)&s_abort);
      if (!go) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // levels 2..5 are exact integers of at most 2^24: int64 at weight 2^-40
      // (level L times 2^(8 (5 - L)), one wide multiply-add per value). Levels 6
      // and 7 (weights 2^-48, 2^-56, at most 2^-24 of the leading level) go to
      // FP32 registers per chunk. (Accumulating them in TMEM over the whole K
      // range instead lost accuracy at K = 80000: a Ritz-value floor near 1e-10
      // ||A||.) Loads are issued three slots at a time, one wait each.
      using S = Slots<LMAX>;
      const bool last = c == nchunks - 1;
      const bool d2 = last || c % kDrain2 == kDrain2 - 1, d3 = last || c % kDrain3 == kDrain3 - 1;
#pragma unroll
      for (int part = 0; part < 2; ++part) {  // real columns, then imaginary
        const uint32_t tp = tl + (uint32_t)(part * CT + h * HC);
        long long* ac = acc + part * HC;
        Acc67* af = acc67 + part * HC;
        float v[3][HC];
        tmem_ld16(tp + S::L4 * TN, v[0]);
        tmem_ld16(tp + S::L5 * TN, v[1]);
        if constexpr (LMAX == 7) tmem_ld16(tp + Slots<7>::L5b * TN, v[2]);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < HC; ++j) {
          add_level<8>(ac[j], v[0][j]);
          add_level<0>(ac[j], LMAX == 7 ? v[1][j] + v[2][j] : v[1][j]);
        }
        if constexpr (LMAX == 7) {
          tmem_ld16(tp + S::L6 * TN, v[0]);
          tmem_ld16(tp + S::L7 * TN, v[1]);
          tmem_ld16(tp + S::L7b * TN, v[2]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < HC; ++j) {
            af[j] += v[0][j];
            af[j] = fmaf(0x1p-8f, v[1][j] + v[2][j], af[j]);
          }
        } else {
          tmem_ld16(tp + S::L7 * TN, v[0]);
          tmem_ld16(tp + S::L7b * TN, v[1]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < HC; ++j) add_level<8>(af[j], v[0][j] + v[1][j]);
          tmem_ld16(tp + S::L6 * TN, v[0]);
          tmem_ld16(tp + Slots<8>::L8 * TN, v[1]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < HC; ++j) {
            add_level<16>(af[j], v[0][j]);
            add_level<0>(af[j], v[1][j]);
          }
        }
        if (d3) {
          tmem_ld16(tp + S::L3 * TN, v[0]);
          if (d2) tmem_ld16(tp + S::L2 * TN, v[1]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < HC; ++j) add_level<16>(ac[j], v[0][j]);
          if (d2) {
#pragma unroll
            for (int j = 0; j < HC; ++j) add_level<24>(ac[j], v[1][j]);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars[2 * kStages + 1]));
    }
    // the ring is free: every MMA of this CTA has been waited for above
    const int e = (warp - 2) * 32 + lane;
#pragma unroll
    for (int j = 0; j < 2 * HC; ++j) {
      acc_s[j * kEpiThreads + e] = acc[j];
      low_s[j * kEpiThreads + e] = acc67[j];
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncwarp();
  if (clustered) cluster_sync();
  if (warp >= 2 && go) {
    // ------------------------------------------------ FP64 result + update
    const int q = warp & 3, h = (warp - 2) >> 2;
    const int64_t row = m0 + q * 32 + lane;
    const int e = (warp - 2) * 32 + lane;
    const bool in_row = row < P.N;
    const int ea = in_row ? P.escale_a[row] : 0;
    const double2 dg = (in_row && P.diag) ? P.diag[row] : make_double2(0.0, 0.0);
    // A_ii B_ij - gamma X_ij as one product where X is the right operand (gamma
    // is the column's Ritz value in the residual)
    const bool same = P.diag && P.mode != EPI_STORE && P.X == P.Bsrc && P.ldx == P.ldbs;
    const double dgx = P.alpha * (dg.x - P.gamma), dgy = P.alpha * dg.y;
    const double ag = P.alpha * P.gamma;
    const unsigned base = cluster_base(P.split, part);
    const int64_t nt32 = (P.N + 31) / 32, t32 = (int64_t)rb * 4 + q;
    const int per = HC / P.split;
#pragma unroll 2
    for (int i = 0; i < per; ++i) {
      const int jj = (int)part * per + i;
      const int64_t col = tile * CT + h * HC + jj;
      const bool in = in_row && col >= P.j0 && col < P.ncols;
      double rsq = 0.0;
      double2 x = make_double2(0.0, 0.0), y0 = x, b = x;
      if (in) {
        if (P.mode != EPI_STORE && (same || P.mode == EPI_RESID || P.gamma != 0.0))
          x = P.X[row + col * P.ldx];
        if (P.diag && !same) b = P.Bsrc[row + col * P.ldbs];
        if (P.mode == EPI_FILTER && P.beta != 0.0) y0 = P.Y[row + col * P.ldy];
        long long hr = acc_s[jj * kEpiThreads + e], hi = acc_s[(HC + jj) * kEpiThreads + e];
        Acc67 lr = low_s[jj * kEpiThreads + e], li = low_s[(HC + jj) * kEpiThreads + e];
        if (P.split > 1) {
          hr = hi = 0;
          lr = li = Acc67(0);
          for (int p = 0; p < P.split; ++p) {
            const unsigned rk = base + (unsigned)p;
            hr += ld_cluster(remote_smem(acc_s + jj * kEpiThreads + e, rk), acc_s);
            hi += ld_cluster(remote_smem(acc_s + (HC + jj) * kEpiThreads + e, rk), acc_s);
            lr += ld_cluster(remote_smem(low_s + jj * kEpiThreads + e, rk), low_s);
            li += ld_cluster(remote_smem(low_s + (HC + jj) * kEpiThreads + e, rk), low_s);
          }
        }
        const int ex = ea + P.escale_b[col];
        double wr = fixed_to_double(hr, low_fixed(lr), ex);
        double wi = fixed_to_double(hi, low_fixed(li), ex);
        if (P.diag && !same) {
          wr = fma(dg.x, b.x, wr);
          wi = fma(dg.x, b.y, wi);
          if (dg.y != 0.0) {
            wr = fma(-dg.y, b.y, wr);
            wi = fma(dg.y, b.x, wi);
          }
        }
        double2* yp = P.Y + row + col * P.ldy;
        if (P.mode == EPI_STORE) {
          *yp = make_double2(wr, wi);
        } else if (P.mode == EPI_FILTER) {
          double vr = P.alpha * wr, vi = P.alpha * wi;
          if (same) {
            vr = fma(dgx, x.x, vr);
            vi = fma(dgx, x.y, vi);
            if (dgy != 0.0) {
              vr = fma(-dgy, x.y, vr);
              vi = fma(dgy, x.x, vi);
            }
          } else if (P.gamma != 0.0) {
            vr = fma(-ag, x.x, vr);
            vi = fma(-ag, x.y, vi);
          }
          if (P.beta != 0.0) {
            vr = fma(P.beta, y0.x, vr);
            vi = fma(P.beta, y0.y, vi);
          }
          *yp = make_double2(vr, vi);
        } else {
          const double th = P.theta[col];
          const double f = same ? dg.x - th : -th;
          double dx = fma(f, x.x, wr), dy = fma(f, x.y, wi);
          if (same && dg.y != 0.0) {
            dx = fma(-dg.y, x.y, dx);
            dy = fma(dg.y, x.x, dy);
          }
          rsq = fma(dx, dx, dy * dy);
        }
      }
      if (P.mode == EPI_RESID) {
        // per column: sum over this warp's 32 rows, one partial per 32-row tile
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) rsq += __shfl_xor_sync(0xffffffffu, rsq, off);
        if (lane == 0 && t32 < nt32 && col >= P.j0 && col < P.ncols) P.partial[t32 + col * nt32] = rsq;
      }
    }
  }
  if (clustered) cluster_sync();  // the others have read this CTA's sums
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

template <int LMAX, int NS>
__global__ void __launch_bounds__(NTHREADS, 1)
    ozaki_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      Params P) {
  let_successor_start();
  ozaki_tile<LMAX, NS>(&tmA, &tmB, P, blockIdx.x, false, P.split > 1);
}

// Many problems' filter steps in one launch: entry p of the table holds problem
// p's tensor maps, step parameters and first CTA index; CTA id finds its
// problem (binary search on the first indices) and runs that problem's tile
// id - first in the raster order of the per-problem launch, so each problem's
// result is that of its own launch.
struct OzGroupEntry {  // aligned as its tensor maps
  CUtensorMap a, b;
  Params P;
  int first, pad;
};

__global__ void __launch_bounds__(NTHREADS, 1)
    ozaki_filter_grouped_kernel(const OzGroupEntry* __restrict__ tab, int count, bool clustered) {
  const int id = (int)blockIdx.x;
  int lo = 0, hi = count - 1;
  while (lo < hi) {  // last entry with first <= id
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].first <= id) lo = mid;
    else hi = mid - 1;
  }
  const OzGroupEntry* e = tab + lo;
  const Params P = e->P;
  ozaki_tile<7, OS>(&e->a, &e->b, P, (unsigned)(id - e->first), true, clustered);
}

// ------------------------------------------------------------ digit prep
// |x| < 1/2: x = sum_s d_s 2^-8s + r with |r| <= 2^-49 and integer digits
// |d_s| <= 128 (exact in BF16). X = rint(x 2^48) (|X| <= 2^47) is written in
// balanced base 256, the low digits in [-128, 127] and the leading one in
// [-128, 128]; so sum_s d_s 2^-8s = X 2^-48 exactly.
//
// The FP64 pipe runs at 1/64 of the FP32 rate on this part and conversions at a
// half to a quarter of it, so everything below is integer work and FP32 adds:
// X is the significand shifted and rounded to even, all low digits come from
// the bytes of X + 0x8080808080 (the additions of 128 that balance each digit,
// with their carries, done at once), and a byte b becomes the float b - 128
// through the bit pattern of 2^23 + b. A BF16 digit is the upper half of that
// float. (With FP64 scaling and one conversion per digit and format, slicing a
// 20000-row matrix took 8.8 ms, 2.9 of the copy bandwidth's 6.8 TB/s.)
template <int BITS>
__device__ __forceinline__ long long fixed(double x, int e) {  // rint(x 2^(BITS - e))
  const long long b = __double_as_longlong(x);
  const int E = (int)(b >> 52) & 0x7ff;
  const long long m = (b & 0xfffffffffffffll) | (E ? 1ll << 52 : 0);
  const int sh = 1075 - BITS - (E ? E : 1) + e;
  if (E == 0x7ff || sh < 48 - BITS - 2)  // a zero whose row or column has a tiny scale, or no number
    return m == 0 ? 0 : __double2ll_rn(ldexp(x * ldexp(1.0, -e), BITS));
  if (sh > 53) return 0;
  if (sh < 1) return b < 0 ? -(m << -sh) : m << -sh;  // more bits than x has
  const long long X = (m + (1ll << (sh - 1)) - 1 + ((m >> sh) & 1)) >> sh;
  return b < 0 ? -X : X;
}
template <int NS>
struct Digits {
  float d[NS];  // leading digit first
};
template <int NS>
__device__ __forceinline__ Digits<NS> digits_of(double x, int e) {
  const unsigned long long X = (unsigned long long)fixed<8 * NS>(x, e) +
                               (NS == OS ? 0x8080808080ull : 0x808080808080ull);
  const unsigned lo = (unsigned)X, hi = (unsigned)(X >> 32);
  Digits<NS> r;
#pragma unroll
  for (int s = 0; s < NS - 1; ++s) {  // byte s of X: digit NS - 1 - s
    const unsigned f = __byte_perm(s < 4 ? lo : hi, 0x4b000000u, 0x7440u | (unsigned)(s & 3));
    r.d[NS - 1 - s] = __uint_as_float(f) - 8388736.0f;  // 2^23 + 128
  }
  r.d[0] = (float)((int)hi >> (8 * (NS - OS + 1)));
  return r;
}
// BF16 of two digits, the first one in the lower half. Digits of finite values
// have at most eight significant bits, so their lower halves are zero.
__device__ __forceinline__ unsigned pack_digits(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}
// max(|a.x|, |a.y|) and running maxima as bit patterns of non-negative doubles
// (monotone in unsigned order); NaN counts as 0, as in fmax
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & ~(1ull << 63);
  return b > 0x7ff0000000000000ull ? 0ull : b;
}
__device__ __forceinline__ unsigned long long max_bits(unsigned long long m, double2 a) {
  const unsigned long long x = abs_bits(a.x), y = abs_bits(a.y);
  m = x > m ? x : m;
  return y > m ? y : m;
}

__device__ __forceinline__ int scale_exp(double mx) {
  if (!(mx > 0.0)) return 0;
  int E;
  frexp(mx, &E);  // mx = f 2^E, f in [0.5, 1)
  return E + 1;   // mx 2^-(E+1) in [0.25, 0.5)
}

// the same from the bit pattern of a maximum
__device__ __forceinline__ int exp_of_bits(unsigned long long b) {
  const int f = (int)(b >> 52);
  if (f == 0 || f == 0x7ff) return scale_exp(__longlong_as_double((long long)b));
  return f - 1021;
}

// The seven-digit product X B moves a power of two 2^t_k from column k of X to row k of
// B before the digits are cut, so that their largest entries are of one size: the
// digits' error follows max_k |x_ik| max_k |b_kj|, and FP64's, which it must not exceed,
// sum_k |x_ik| |b_kj|. (Columns graded over 2, 8 and 16 decades on one side and their
// inverse on the other cost 6e-16, 3e-10 and 3e-2 of Abar.) No entry is touched: t_k
// only enters the exponents. A k whose column or row is zero is dropped, lest the other
// side set the scales.
constexpr int kDrop = 1 << 20;    // t_k of a dropped k: the exponents put its digits at zero
constexpr int kNoExp = -100000;   // exponent of zero
// E with 2^(E - 1) <= x < 2^E for x > 0 given by its bit pattern
__device__ __forceinline__ int bin_exp(unsigned long long b) {
  const int f = (int)(b >> 52);
  return f != 0 ? f - 1022 : b != 0 ? 64 - 1074 - __clzll((long long)b) : kNoExp;
}
__device__ __forceinline__ int bin_exp(double2 a) {
  const unsigned long long x = (unsigned long long)__double_as_longlong(a.x) & ~(1ull << 63);
  const unsigned long long y = (unsigned long long)__double_as_longlong(a.y) & ~(1ull << 63);
  return bin_exp(x > y ? x : y);  // 1025 for an infinity or NaN
}
// exponent to cut an entry of X (SIGN 1) or B (-1) with, in a row or column of scale e
template <int SIGN>
__device__ __forceinline__ int cut_exp(int e, int t) {
  return e + (t == kDrop ? kDrop : SIGN * t);
}
__device__ __forceinline__ int block_max(int m, int* red) {  // 256 threads
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) m = max(m, red[w]);
  return m;
}

// t_k (kexp), one CTA per k, and *bad = 1 where an entry is an infinity or NaN, which
// digits cannot carry. X (M x K) and B (K x n) are read once more for it: 7 us for M = n =
// 1500, K = 480.
__global__ void __launch_bounds__(256)
    balance_kernel(int64_t M, int64_t n, const double2* __restrict__ X, int64_t ldx,
                   const double2* __restrict__ B, int64_t ldb, int* __restrict__ kexp,
                   int* __restrict__ bad) {
  __shared__ int red[2][8];
  const int64_t k = blockIdx.x;
  int x = kNoExp, b = kNoExp;
  for (int64_t i = threadIdx.x; i < M; i += 256) x = max(x, bin_exp(X[i + k * ldx]));
  for (int64_t j = threadIdx.x; j < n; j += 256) b = max(b, bin_exp(B[k + j * ldb]));
  x = block_max(x, red[0]);
  b = block_max(b, red[1]);
  if (threadIdx.x != 0) return;
  kexp[k] = x == kNoExp || b == kNoExp ? kDrop : (x - b) >> 1;
  if (max(x, b) > 1024) *bad = 1;
}
// Scales of the rows of X (M x K): ea[i] = the largest exponent of X_ik 2^-t_k, plus one.
// ea starts far below every exponent. kRowK columns a CTA: K is a few hundred here, and
// a chain of 128 columns in 6 CTAs took 40 us for 1500 rows.
constexpr int kRowK = 16;
__global__ void row_scale_kernel(int64_t M, int64_t K, const double2* __restrict__ X, int64_t ldx,
                                 const int* __restrict__ kexp, int* __restrict__ ea) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const int64_t k0 = (int64_t)blockIdx.y * kRowK, k1 = min(K, k0 + kRowK);
  int m = kNoExp;
#pragma unroll 8
  for (int64_t k = k0; k < k1; ++k) {
    const int t = kexp[k];
    if (t != kDrop) m = max(m, bin_exp(X[i + k * ldx]) - t);
  }
  atomicMax(&ea[i], max(m + 1, kNoExp));
}

// Row maxima of A (column-major): amax[i] = max_k max(|Re A_ik|, |Im A_ik|),
// as the bit pattern of a non-negative double (monotone in unsigned order).
__global__ void rowmax_kernel(int64_t M, int64_t K, bool skip_diag, const double2* __restrict__ A,
                              int64_t lda, unsigned long long* __restrict__ amax) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const int64_t k0 = (int64_t)blockIdx.y * 256, k1 = min(K, k0 + 256);
  unsigned long long m = 0;
#pragma unroll 8
  for (int64_t k = k0; k < k1; ++k) {
    if (skip_diag && k == i) continue;  // the diagonal is applied separately, exactly
    m = max_bits(m, A[i + k * lda]);
  }
  atomicMax(&amax[i], m);
}

__global__ void diag_kernel(int64_t N, const double2* __restrict__ A, int64_t lda,
                            double2* __restrict__ d) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) d[i] = A[i + i * lda];
}

__global__ void exps_kernel(int64_t n, const unsigned long long* __restrict__ mx, int* __restrict__ e) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) e[i] = scale_exp(__longlong_as_double((long long)mx[i]));
}

// A (M x K, column-major) -> OS digit planes, each M rows x 2 Np (row-major
// [Ar | Ai]), stacked, and the rows' exponents from their maxima (of seven digits: ea
// holds them, kexp the columns' own); skip_diag leaves the diagonal out (square A). A warp
// writes a row of 64 entries, two per lane: 128 bytes of each of its 12 rows.
constexpr int SA_K = 64;
template <int NS>
__global__ void __launch_bounds__(256)
    slice_a_kernel(int64_t M, int64_t K, int64_t Np, bool skip_diag,
                   const double2* __restrict__ A, int64_t lda,
                   const unsigned long long* __restrict__ amax, const int* __restrict__ kexp,
                   int* __restrict__ ea, __nv_bfloat16* __restrict__ out) {
  __shared__ double2 tile[SA_K][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * SA_K;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
#pragma unroll
  for (int r = ty; r < SA_K; r += 8) {
    const int64_t i = i0 + tx, k = k0 + r;
    tile[r][tx] = (i < M && k < K && !(skip_diag && i == k)) ? A[i + k * lda]
                                                             : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const int64_t ld = 2 * Np;
  const size_t plane = (size_t)M * ld;
  const int64_t k = k0 + 2 * tx;  // k + 1 may be K: the padding's digits are zero
  if (k >= K) return;
  int t0 = 0, t1 = 0;
  if constexpr (NS == OS7) {
    t0 = kexp[k];
    t1 = k + 1 < K ? kexp[k + 1] : 0;
  }
  for (int r = ty; r < 32; r += 8) {
    const int64_t i = i0 + r;
    if (i >= M) continue;
    const double2 a0 = tile[2 * tx][r], a1 = tile[2 * tx + 1][r];
    int e0, e1;
    if constexpr (NS == OS7) {
      e0 = cut_exp<1>(ea[i], t0);
      e1 = cut_exp<1>(ea[i], t1);
    } else {
      e0 = e1 = exp_of_bits(amax[i]);
      if (k0 == 0 && tx == 0) ea[i] = e0;
    }
    const Digits<NS> r0 = digits_of<NS>(a0.x, e0), r1 = digits_of<NS>(a1.x, e1);
    const Digits<NS> c0 = digits_of<NS>(a0.y, e0), c1 = digits_of<NS>(a1.y, e1);
    __nv_bfloat16* o = out + i * ld + k;
#pragma unroll
    for (int d = 0; d < NS; ++d) {
      *reinterpret_cast<unsigned*>(o + d * plane) = pack_digits(r0.d[d], r1.d[d]);
      *reinterpret_cast<unsigned*>(o + d * plane + Np) = pack_digits(c0.d[d], c1.d[d]);
    }
  }
}

// X (M x K, column-major) <- the value its six digits represent when X is the
// left operand (row i scaled by 2^-e_i): sum_s d_s 2^(e_i - 8s).
__global__ void round_left_kernel(int64_t M, int64_t K, double2* __restrict__ X, int64_t ldx,
                                  const int* __restrict__ ea) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t k = blockIdx.y;
  if (i >= M || k >= K) return;
  const double2 x = X[i + k * ldx];
  const int e = ea[i];
  // exact: 48 bits below the scale
  X[i + k * ldx] = make_double2(ldexp((double)fixed<48>(x.x, e), e - 48),
                                ldexp((double)fixed<48>(x.y, e), e - 48));
}

// Left operand X^H for X (K x M, column-major): row i of X^H is conj(X[:, i]),
// contiguous, so no transpose is needed. Exponents per row come from colexp. Entries
// k, k + 1 (zero past K) of a row.
__device__ __forceinline__ void slice_ct_pair(int64_t K, int64_t Np, size_t plane, int64_t k,
                                              const double2* __restrict__ X, int e,
                                              __nv_bfloat16* __restrict__ row) {
  const double2 x0 = X[k];
  const double2 x1 = k + 1 < K ? X[k + 1] : make_double2(0.0, 0.0);
  const Digits<OS> r0 = digits_of<OS>(x0.x, e), r1 = digits_of<OS>(x1.x, e);
  const Digits<OS> c0 = digits_of<OS>(-x0.y, e), c1 = digits_of<OS>(-x1.y, e);
#pragma unroll
  for (int d = 0; d < OS; ++d) {
    *reinterpret_cast<unsigned*>(row + d * plane + k) = pack_digits(r0.d[d], r1.d[d]);
    *reinterpret_cast<unsigned*>(row + d * plane + Np + k) = pack_digits(c0.d[d], c1.d[d]);
  }
}
__global__ void slice_ct_kernel(int64_t M, int64_t K, int64_t Np, const double2* __restrict__ X,
                                int64_t ldx, const int* __restrict__ ea,
                                __nv_bfloat16* __restrict__ out) {
  const int64_t k = 2 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  const int64_t i = blockIdx.y;
  if (k >= K) return;
  slice_ct_pair(K, Np, (size_t)M * 2 * Np, k, X + i * ldx, ea[i], out + i * 2 * Np);
}

// Column maxima of Y (complex columns j0 .. j0 + gridDim.x): one CTA per column.
__device__ __forceinline__ unsigned long long block_max_bits(unsigned long long m,
                                                             unsigned long long* red) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, off);
    m = o > m ? o : m;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) m = red[w] > m ? red[w] : m;
  return m;
}
__device__ __forceinline__ unsigned long long column_max(int64_t N, const double2* __restrict__ Y,
                                                         unsigned long long* red) {
  unsigned long long m = 0;
#pragma unroll 4
  for (int64_t k = threadIdx.x; k < N; k += 256) m = max_bits(m, Y[k]);
  return block_max_bits(m, red);
}
// Scale of a column of the right operand: the exponent of its maximum, plus one; with
// seven digits of its entries times 2^t_k.
template <int NS>
__device__ __forceinline__ int column_scale(int64_t N, const double2* __restrict__ Y,
                                            const int* __restrict__ kexp,
                                            unsigned long long* red) {
  if constexpr (NS == OS) {
    return scale_exp(__longlong_as_double((long long)column_max(N, Y, red)));
  } else {
    int m = kNoExp;
#pragma unroll 4
    for (int64_t k = threadIdx.x; k < N; k += 256) {
      const int t = kexp[k];
      if (t != kDrop) m = max(m, bin_exp(Y[k]) + t);
    }
    return max(block_max(m, reinterpret_cast<int*>(red)) + 1, kNoExp);
  }
}
template <int NS>
__global__ void __launch_bounds__(256)
    colexp_kernel(int64_t N, int64_t j0, const double2* __restrict__ Y, int64_t ldy,
                  const int* __restrict__ kexp, int* __restrict__ eb) {
  __shared__ unsigned long long red[8];
  const int64_t j = j0 + blockIdx.x;
  let_successor_start();
  wait_for_predecessor();
  const int e = column_scale<NS>(N, Y + j * ldy, kexp, red);
  if (threadIdx.x == 0) eb[j] = e;
}

// Digits of entries k, k + 1 (zero past N) of one column of the right operand
// into its rows of B^T. Real row: [Yr | -Yi]; imaginary row: [Yi | Yr].
template <int NS>
__device__ __forceinline__ void slice_b_pair(int64_t N, int64_t Np, size_t plane, int64_t k,
                                             const double2* __restrict__ Y, int e,
                                             const int* __restrict__ kexp,
                                             __nv_bfloat16* __restrict__ re,
                                             __nv_bfloat16* __restrict__ im) {
  const double2 y0 = Y[k];
  const double2 y1 = k + 1 < N ? Y[k + 1] : make_double2(0.0, 0.0);
  int e0 = e, e1 = e;
  if constexpr (NS == OS7) {
    e0 = cut_exp<-1>(e, kexp[k]);
    if (k + 1 < N) e1 = cut_exp<-1>(e, kexp[k + 1]);
  }
  const Digits<NS> r0 = digits_of<NS>(y0.x, e0), r1 = digits_of<NS>(y1.x, e1);
  const Digits<NS> c0 = digits_of<NS>(y0.y, e0), c1 = digits_of<NS>(y1.y, e1);
#pragma unroll
  for (int d = 0; d < NS; ++d) {
    const unsigned r = pack_digits(r0.d[d], r1.d[d]), c = pack_digits(c0.d[d], c1.d[d]);
    *reinterpret_cast<unsigned*>(re + d * plane + k) = r;
    *reinterpret_cast<unsigned*>(re + d * plane + Np + k) = c ^ 0x80008000u;
    *reinterpret_cast<unsigned*>(im + d * plane + k) = c;
    *reinterpret_cast<unsigned*>(im + d * plane + Np + k) = r;
  }
}

// Y columns -> OS digit planes of B^T (rows: 32-column tiles of 64 rows), stacked
// with `brows` rows per plane; two entries per thread.
template <int NS>
__global__ void slice_b_kernel(int64_t N, int64_t Np, int64_t brows, int64_t j0,
                               const double2* __restrict__ Y, int64_t ldy, const int* __restrict__ eb,
                               const int* __restrict__ kexp, __nv_bfloat16* __restrict__ out) {
  const int64_t k = 2 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  const int64_t j = j0 + blockIdx.y;
  let_successor_start();
  wait_for_predecessor();
  if (k >= N) return;
  const int64_t ld = 2 * Np, br = brow_re(j);
  slice_b_pair<NS>(N, Np, (size_t)brows * ld, k, Y + j * ldy, eb[j], kexp, out + br * ld,
                   out + (br + CT) * ld);
}

// Maximum, exponent and digits of one column of the right operand by one CTA of 256
// threads (the second reading comes from the caches). A separate pass for the
// exponents costs a launch: 4.3 us against 2 + 2.3 us and the gap between them for 60
// columns of 512 rows. Longer columns, which one CTA reads too slowly (64 of 2048
// rows: 10.4 against 5.5 us), take the two passes.
constexpr int64_t kOnePass = 1024;
template <int NS>
__device__ __forceinline__ void slice_b_column(int64_t N, int64_t Np, int64_t brows, int64_t j,
                                               const double2* __restrict__ Y,
                                               const int* __restrict__ kexp,
                                               int* __restrict__ eb, __nv_bfloat16* __restrict__ out,
                                               unsigned long long* red) {
  const int ex = column_scale<NS>(N, Y, kexp, red);
  if (threadIdx.x == 0) eb[j] = ex;
  const int64_t ld = 2 * Np, br = brow_re(j);
  for (int64_t k = 2 * threadIdx.x; k < N; k += 512)
    slice_b_pair<NS>(N, Np, (size_t)brows * ld, k, Y, ex, kexp, out + br * ld,
                     out + (br + CT) * ld);
}
template <int NS>
__global__ void __launch_bounds__(256)
    slice_b_column_kernel(int64_t N, int64_t Np, int64_t brows, int64_t j0,
                          const double2* __restrict__ Y, int64_t ldy, const int* __restrict__ kexp,
                          int* __restrict__ eb, __nv_bfloat16* __restrict__ out) {
  __shared__ unsigned long long red[8];
  const int64_t j = j0 + blockIdx.x;
  let_successor_start();
  wait_for_predecessor();
  slice_b_column<NS>(N, Np, brows, j, Y + j * ldy, kexp, eb, out, red);
}
// The same for the left operand X^H: row i is the conjugate of X's column i.
__global__ void __launch_bounds__(256)
    slice_ct_column_kernel(int64_t M, int64_t K, int64_t Np, const double2* __restrict__ X,
                           int64_t ldx, int* __restrict__ el, __nv_bfloat16* __restrict__ out) {
  __shared__ unsigned long long red[8];
  const int64_t i = blockIdx.x;
  const double2* Xi = X + i * ldx;
  const int ex = scale_exp(__longlong_as_double((long long)column_max(K, Xi, red)));
  if (threadIdx.x == 0) el[i] = ex;
  const int64_t ld = 2 * Np;
  for (int64_t k = 2 * threadIdx.x; k < K; k += 512)
    slice_ct_pair(K, Np, (size_t)M * ld, k, Xi, ex, out + i * ld);
}

// The right-operand digits of many problems' filter steps in one launch: one
// CTA (256 threads) per active column of every problem. It forms the column's
// maximum with the reduction of colexp_kernel, then the column's digits as
// slice_b_kernel does, so each problem's planes are those of its own launches.
struct OzSliceEntry {
  const double2* B;          // right operand (absolute columns, ld ldb)
  int64_t ldb, N, Np, brows, j0;
  int* eb;                   // column exponents
  __nv_bfloat16* out;        // digit planes
  int first, pad;            // first CTA of this problem
};

__global__ void __launch_bounds__(256)
    slice_b_grouped_kernel(const OzSliceEntry* __restrict__ tab, int count) {
  __shared__ unsigned long long red[8];
  const int id = (int)blockIdx.x;
  int lo = 0, hi = count - 1;
  while (lo < hi) {  // last entry with first <= id
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].first <= id) lo = mid;
    else hi = mid - 1;
  }
  const OzSliceEntry& e = tab[lo];
  const int64_t N = e.N, j = e.j0 + (id - e.first);
  const double2* __restrict__ Y = e.B + j * e.ldb;
  slice_b_column<OS>(N, e.Np, e.brows, j, Y, nullptr, e.eb, e.out, red);
}

PFN_cuTensorMapEncodeTiled_v12000 lookup_encoder() {
  cudaDriverEntryPointQueryResult q;
  void* fn = nullptr;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                       &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    return nullptr;
  return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
}
// The driver's tensor-map encoder, looked up once (thread-safe static
// initialisation; contexts may be created from several host threads).
PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = lookup_encoder();
  return fn;
}
bool get_encoder() { return encoder() != nullptr; }
bool make_map(CUtensorMap* m, void* base, int64_t rows, int64_t Np, int box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)(2 * Np), (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)(2 * Np * 2)};
  const cuuint32_t box[2] = {(cuuint32_t)TK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  return encoder()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

struct Maps {
  CUtensorMap a, b;
};

// CTAs per tile. A tile costs its chunks plus about one chunk's time to start
// and, undivided, one and a half to finish; a wave of tiles takes as long as its
// slowest. Tiles that fill the chip several times over stay whole; a product of
// few tiles (the 8 of a 512 x 60 block, the 30 of a 316 x 316 Gram over 9273
// rows) is cut so that its parts fill one wave. A cut has to gain a tenth: parts
// read the right operand no less often and meet at two cluster barriers. Past five
// waves there is nothing to even out (a 1072 x 1072 Gram over 13379 rows, 306 tiles: 8
// parts a tile took 0.4 ms more than 2). It
// depends on the product alone, so a problem's result is the same in a group.
constexpr int kMaxSplit = 8;
int choose_split(int64_t tiles, int64_t Np) {
  const int64_t nkb = 2 * Np / TK, sms = num_sms();
  int best = 1;
  double best_cost = 1e300;
  for (int s = 1; s <= kMaxSplit && 4 * s <= nkb; s *= 2) {  // at least half a chunk each
    if (s > 1 && tiles * s > 5 * sms) break;
    const double cost = (double)cdiv(tiles * s, sms) *
                        ((double)cdiv(nkb, s) / CHUNK_KB + 1.0 + 1.5 / s);
    if (cost < 0.9 * best_cost) {
      best_cost = cost;
      best = s;
    }
  }
  return best;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_clusters(void (*kernel)(KArgs...), unsigned ctas, int cluster, bool early,
                            cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas, 1, 1);
  cfg.blockDim = dim3(NTHREADS, 1, 1);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = s;
  cudaLaunchAttribute at[2]{};
  if (cluster > 1) {
    cudaLaunchAttribute& c = at[cfg.numAttrs++];
    c.id = cudaLaunchAttributeClusterDimension;
    c.val.clusterDim.x = (unsigned)cluster;
    c.val.clusterDim.y = c.val.clusterDim.z = 1;
  }
  if (early) {
    cudaLaunchAttribute& e = at[cfg.numAttrs++];
    e.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    e.val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = at;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
enum Pairs { PAIRS_21, PAIRS_26, PAIRS_28 };
cudaError_t launch_product(cudaStream_t s, const CUtensorMap& a, const CUtensorMap& b,
                           const Params& P, Pairs pairs) {
  const unsigned ctas = (unsigned)P.nrow * (unsigned)P.ncol * (unsigned)P.split;
  auto* k = pairs == PAIRS_21   ? ozaki_gemm_kernel<7, OS>
            : pairs == PAIRS_26 ? ozaki_gemm_kernel<8, OS>
                                : ozaki_gemm_kernel<8, OS7>;
  return launch_clusters(k, ctas, P.split, true, s, a, b, P);
}
void set_tiles(Params& P) {
  P.nrow = (int)cdiv(P.N, TM);
  P.ncol = (int)((P.ncols - 1) / CT - P.j0 / CT + 1);
  P.split = choose_split((int64_t)P.nrow * P.ncol, P.Np);
}

// Launch parameters of A * B[:, j0:ncols_end] with epilogue ep (A's digits in w).
Params product_params(const OzakiWork& w, int64_t ncols_end, int64_t j0, const double2* B,
                      int64_t ldb, const Epilogue& ep) {
  Params P;
  P.N = w.N;
  P.Np = w.Np;
  P.brows = w.brows;
  P.arows = w.N;
  P.j0 = j0;
  P.ncols = ncols_end;
  P.escale_a = w.ea;
  P.escale_b = w.eb;
  P.diag = w.diag;
  P.Bsrc = B;
  P.ldbs = ldb;
  P.mode = ep.mode;
  P.alpha = ep.alpha;
  P.beta = ep.beta;
  P.gamma = ep.gamma;
  P.X = ep.X;
  P.ldx = ep.ldx;
  P.Y = ep.Y;
  P.ldy = ep.ldy;
  P.theta = ep.theta;
  P.partial = ep.partial;
  P.err = w.err;
  P.skip = w.bad;
  set_tiles(P);
  return P;
}

}  // namespace

int64_t ozaki_np(int64_t N) { return cdiv(N, KPAD) * KPAD; }

cudaError_t ozaki_alloc(OzakiWork& w, int64_t N, int64_t ne) {
  w.N = N;
  w.ne = ne;
  w.Np = ozaki_np(N);
  w.brows = cdiv(ne, CT) * TN;
  const size_t a_elems = (size_t)OS * N * 2 * w.Np;
  const size_t b_elems = (size_t)OS * w.brows * 2 * w.Np;
  if (!get_encoder()) return cudaErrorNotSupported;
  cudaError_t e;
  if ((e = cudaMalloc(&w.Ad, a_elems * 2)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.Bd, b_elems * 2)) != cudaSuccess) return e;
  if ((e = cudaMemset(w.Ad, 0, a_elems * 2)) != cudaSuccess) return e;
  if ((e = cudaMemset(w.Bd, 0, b_elems * 2)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.ea, N * sizeof(int))) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.eb, std::max(N, ne) * sizeof(int))) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.amax, N * sizeof(unsigned long long))) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.diag, N * sizeof(double2))) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.err, 2 * sizeof(int))) != cudaSuccess) return e;
  if ((e = cudaMemset(w.err, 0, 2 * sizeof(int))) != cudaSuccess) return e;
  w.bad = w.err + 1;
  // general left operands of the N x n^2 products: X^H (ne x N) or Q (N x ne)
  const int64_t npe = ozaki_np(ne);
  w.l_elems = (size_t)OS7 * std::max((size_t)ne * 2 * w.Np, (size_t)N * 2 * npe);
  if ((e = cudaMalloc(&w.Ld, w.l_elems * 2)) != cudaSuccess) return e;
  if ((e = cudaMemset(w.Ld, 0, w.l_elems * 2)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.el, std::max(N, ne) * sizeof(int))) != cudaSuccess) return e;
  Maps* maps = nullptr;
  if ((e = cudaMallocHost(&maps, sizeof(Maps))) != cudaSuccess) return e;
  w.maps = maps;
  // digit planes stacked along rows: OS * N rows (A), OS * brows rows (B)
  if (!make_map(&maps->a, w.Ad, (int64_t)OS * N, w.Np, TM) ||
      !make_map(&maps->b, w.Bd, (int64_t)OS * w.brows, w.Np, TN))
    return cudaErrorInvalidValue;
  for (auto k : {ozaki_gemm_kernel<7, OS>, ozaki_gemm_kernel<8, OS>, ozaki_gemm_kernel<8, OS7>})
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES)) !=
        cudaSuccess)
      return e;
  return cudaSuccess;
}

void ozaki_free(OzakiWork& w) {
  void* bufs[] = {w.Ad, w.Bd, w.ea, w.eb, w.amax, w.err, w.diag, w.Ld, w.el};
  for (void* b : bufs)
    if (b) cudaFree(b);
  if (w.maps) cudaFreeHost(w.maps);
  w = OzakiWork{};
}

cudaError_t ozaki_prepare_a(cudaStream_t s, const double2* A, int64_t lda, OzakiWork& w) {
  const int64_t N = w.N;
  cudaError_t e = cudaMemsetAsync(w.amax, 0, N * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  rowmax_kernel<<<dim3((unsigned)cdiv(N, 256), (unsigned)cdiv(N, 256), 1), 256, 0, s>>>(
      N, N, true, A, lda, w.amax);
  count_launch();
  diag_kernel<<<(unsigned)cdiv(N, 256), 256, 0, s>>>(N, A, lda, w.diag);
  count_launch();
  slice_a_kernel<OS><<<dim3((unsigned)cdiv(N, 32), (unsigned)cdiv(N, SA_K), 1), dim3(32, 8, 1), 0, s>>>(
      N, N, w.Np, true, A, lda, w.amax, nullptr, w.ea, static_cast<__nv_bfloat16*>(w.Ad));
  count_launch();
  w.A_ready = A;
  return cudaGetLastError();
}

namespace {
// Launch that may begin while its predecessor in the stream still runs; the kernel
// waits for it (wait_for_predecessor).
template <typename... KArgs, typename... Args>
cudaError_t launch_early(void (*kernel)(KArgs...), dim3 grid, int threads, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
// Digits of columns j0 .. j0 + n of B (K rows) into w.Bd (`brows` rows a plane). A
// product must not follow a refused launch: it would take the digits of another block.
template <int NS>
cudaError_t slice_right(cudaStream_t s, int64_t K, int64_t j0, int64_t n, const double2* B, int64_t ldb,
                        int64_t brows, const int* kexp, OzakiWork& w) {
  __nv_bfloat16* out = static_cast<__nv_bfloat16*>(w.Bd);
  const int64_t Kp = ozaki_np(K);
  if (K <= kOnePass)
    return launch_early(slice_b_column_kernel<NS>, dim3((unsigned)n, 1, 1), 256, s, K, Kp, brows,
                        j0, B, ldb, kexp, w.eb, out);
  const cudaError_t e =
      launch_early(colexp_kernel<NS>, dim3((unsigned)n, 1, 1), 256, s, K, j0, B, ldb, kexp, w.eb);
  if (e != cudaSuccess) return e;
  return launch_early(slice_b_kernel<NS>, dim3((unsigned)cdiv(K, 512), (unsigned)n, 1), 256, s, K,
                      Kp, brows, j0, B, ldb, (const int*)w.eb, kexp, out);
}

}  // namespace

cudaError_t ozaki_gemm(cudaStream_t s, int64_t ncols_end, int64_t j0, const double2* B,
                       int64_t ldb, const Epilogue& ep, OzakiWork& w) {
  const int64_t N = w.N;
  const int64_t n = ncols_end - j0;
  if (n <= 0) return cudaSuccess;
  const cudaError_t e = slice_right<OS>(s, N, j0, n, B, ldb, w.brows, nullptr, w);
  if (e != cudaSuccess) return e;
  const Maps* maps = static_cast<const Maps*>(w.maps);
  const Params P = product_params(w, ncols_end, j0, B, ldb, ep);
  return launch_product(s, maps->a, maps->b, P, PAIRS_21);
}

namespace {
// Digits of the left operand X (M x K) into w.Ld, row exponents into w.el.
template <int NS>
cudaError_t slice_left(cudaStream_t s, int64_t M, int64_t K, const double2* X, int64_t ldx,
                       const int* kexp, OzakiWork& w) {
  const unsigned rows = (unsigned)cdiv(M, 256);
  cudaError_t e;
  if constexpr (NS == OS7) {
    if ((e = cudaMemsetAsync(w.el, 0x80, M * sizeof(int), s)) != cudaSuccess) return e;
    row_scale_kernel<<<dim3(rows, (unsigned)cdiv(K, kRowK), 1), 256, 0, s>>>(M, K, X, ldx, kexp, w.el);
  } else {
    if ((e = cudaMemsetAsync(w.amax, 0, M * sizeof(unsigned long long), s)) != cudaSuccess) return e;
    rowmax_kernel<<<dim3(rows, (unsigned)cdiv(K, 256), 1), 256, 0, s>>>(M, K, false, X, ldx,
                                                                        w.amax);
  }
  count_launch();
  slice_a_kernel<NS><<<dim3((unsigned)cdiv(M, 32), (unsigned)cdiv(K, SA_K), 1), dim3(32, 8, 1), 0,
                       s>>>(M, K, ozaki_np(K), false, X, ldx, w.amax, kexp, w.el,
                            static_cast<__nv_bfloat16*>(w.Ld));
  count_launch();
  return cudaGetLastError();
}
// The K padding of the left planes must be zero (the right operand's padding then
// only has to be finite, which digits always are). The slicing writes k < K only,
// so the planes are cleared whenever their layout changes.
cudaError_t clear_left(cudaStream_t s, int64_t M, int64_t K, int ns, OzakiWork& w) {
  if (M == w.l_M && K == w.l_K && ns == w.l_ns) return cudaSuccess;
  w.l_M = M;
  w.l_K = K;
  w.l_ns = ns;
  return cudaMemsetAsync(w.Ld, 0, (size_t)ns * M * 2 * ozaki_np(K) * 2, s);
}
// Parameters of a product with the left planes in w.Ld (no diagonal split).
Params general_params(int64_t M, int64_t K, int64_t ncols, const double2* B, int64_t ldb,
                      int64_t brows, const Epilogue& ep, OzakiWork& w) {
  Params P;
  P.N = M;
  P.Np = ozaki_np(K);
  P.brows = brows;
  P.arows = M;
  P.j0 = 0;
  P.ncols = ncols;
  P.escale_a = w.el;
  P.escale_b = w.eb;
  P.diag = nullptr;
  P.Bsrc = B;
  P.ldbs = ldb;
  P.mode = ep.mode;
  P.alpha = ep.alpha;
  P.beta = ep.beta;
  P.gamma = ep.gamma;
  P.X = ep.X;
  P.ldx = ep.ldx;
  P.Y = ep.Y;
  P.ldy = ep.ldy;
  P.theta = ep.theta;
  P.partial = ep.partial;
  P.err = w.err;
  P.skip = w.bad;
  set_tiles(P);
  return P;
}
}  // namespace

cudaError_t ozaki_gemm_general(cudaStream_t s, int64_t M, int64_t K, const double2* X,
                               int64_t ldx, bool conj_trans, int64_t ncols, const double2* B,
                               int64_t ldb, const Epilogue& ep, OzakiWork& w, bool extended) {
  if (M <= 0 || ncols <= 0 || K <= 0) return cudaSuccess;
  const int64_t Kp = ozaki_np(K);
  if (Kp > w.Np || ncols > w.ne || (size_t)OS * M * 2 * Kp > w.l_elems)
    return cudaErrorInvalidValue;
  cudaError_t e = clear_left(s, M, K, OS, w);
  if (e != cudaSuccess) return e;
  if (conj_trans) {  // left = X^H, X is K x M
    __nv_bfloat16* L = static_cast<__nv_bfloat16*>(w.Ld);
    count_launch();
    if (K <= kOnePass) {
      slice_ct_column_kernel<<<(unsigned)M, 256, 0, s>>>(M, K, Kp, X, ldx, w.el, L);
    } else {
      colexp_kernel<OS><<<(unsigned)M, 256, 0, s>>>(K, 0, X, ldx, nullptr, w.el);
      slice_ct_kernel<<<dim3((unsigned)cdiv(K, 512), (unsigned)M, 1), 256, 0, s>>>(M, K, Kp, X, ldx,
                                                                                   w.el, L);
      count_launch();
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else if ((e = slice_left<OS>(s, M, K, X, ldx, nullptr, w)) != cudaSuccess) {  // left = X, M x K
    return e;
  }
  if ((e = slice_right<OS>(s, K, 0, ncols, B, ldb, w.brows, nullptr, w)) != cudaSuccess) return e;
  CUtensorMap ma, mb;
  if (!make_map(&ma, w.Ld, (int64_t)OS * M, Kp, TM) ||
      !make_map(&mb, w.Bd, (int64_t)OS * w.brows, Kp, TN))
    return cudaErrorInvalidValue;
  const Params P = general_params(M, K, ncols, B, ldb, w.brows, ep, w);
  return launch_product(s, ma, mb, P, extended ? PAIRS_26 : PAIRS_21);
}

int64_t ozaki_fine_inner(const OzakiWork& w, int64_t M) {
  const int64_t left = (int64_t)(w.l_elems / ((size_t)OS7 * M * 2)) / KPAD * KPAD;
  // one column tile of the right operand has to fit too
  const int64_t right = OS * w.brows * w.Np / (OS7 * TN) / KPAD * KPAD;
  return std::min(left, right);
}

cudaError_t ozaki_fine_begin(cudaStream_t s, int64_t M, int64_t K, const double2* X, int64_t ldx,
                             int64_t ncols, const double2* B, int64_t ldb, int* kexp,
                             OzakiWork& w) {
  const cudaError_t e = cudaMemsetAsync(w.bad, 0, sizeof(int), s);
  if (e != cudaSuccess || M <= 0 || ncols <= 0 || K <= 0) return e;
  balance_kernel<<<(unsigned)K, 256, 0, s>>>(M, ncols, X, ldx, B, ldb, kexp, w.bad);
  count_launch();
  return cudaGetLastError();
}

cudaError_t ozaki_fine_end(cudaStream_t s, const OzakiWork& w, bool* formed) {
  int bad = 0;
  const cudaError_t e = cudaMemcpyAsync(&bad, w.bad, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  *formed = false;
  const cudaError_t se = cudaStreamSynchronize(s);
  if (se == cudaSuccess) *formed = bad == 0;
  return se;
}

cudaError_t ozaki_gemm_fine(cudaStream_t s, int64_t M, int64_t K, const double2* X, int64_t ldx,
                            int64_t ncols, const double2* B, int64_t ldb, const int* kexp,
                            const Epilogue& ep, OzakiWork& w) {
  if (M <= 0 || ncols <= 0 || K <= 0) return cudaSuccess;
  const int64_t Kp = ozaki_np(K);
  if (M > w.N || Kp > ozaki_fine_inner(w, M)) return cudaErrorInvalidValue;
  cudaError_t e = clear_left(s, M, K, OS7, w);
  if (e != cudaSuccess || (e = slice_left<OS7>(s, M, K, X, ldx, kexp, w)) != cudaSuccess)
    return e;
  // as many columns at a time as the right operand's planes hold, in whole tiles, and
  // as a grid has rows
  const int64_t fit = OS * w.brows * w.Np / (OS7 * Kp) / TN * CT;
  const int64_t block = std::min({ncols, fit, std::max(w.N, w.ne), (int64_t)65535 / CT * CT});
  const int64_t brows = cdiv(block, CT) * TN;
  CUtensorMap ma, mb;
  if (!make_map(&ma, w.Ld, (int64_t)OS7 * M, Kp, TM) ||
      !make_map(&mb, w.Bd, (int64_t)OS7 * brows, Kp, TN))
    return cudaErrorInvalidValue;
  for (int64_t c0 = 0; c0 < ncols; c0 += block) {
    const int64_t nc = std::min(block, ncols - c0);
    if ((e = slice_right<OS7>(s, K, 0, nc, B + c0 * ldb, ldb, brows, kexp, w)) != cudaSuccess)
      return e;
    Epilogue ec = ep;
    if (ec.X) ec.X += c0 * ec.ldx;
    if (ec.Y) ec.Y += c0 * ec.ldy;
    const Params P = general_params(M, K, nc, B + c0 * ldb, ldb, brows, ec, w);
    if ((e = launch_product(s, ma, mb, P, PAIRS_28)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t ozaki_round_left(cudaStream_t s, int64_t M, int64_t K, double2* X, int64_t ldx,
                             OzakiWork& w) {
  if (M <= 0 || K <= 0) return cudaSuccess;
  if (M > w.N) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(w.amax, 0, M * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  rowmax_kernel<<<dim3((unsigned)cdiv(M, 256), (unsigned)cdiv(K, 256), 1), 256, 0, s>>>(
      M, K, false, X, ldx, w.amax);
  count_launch();
  exps_kernel<<<(unsigned)cdiv(M, 256), 256, 0, s>>>(M, w.amax, w.el);
  count_launch();
  round_left_kernel<<<dim3((unsigned)cdiv(M, 256), (unsigned)K, 1), 256, 0, s>>>(M, K, X, ldx,
                                                                                 w.el);
  count_launch();
  return cudaGetLastError();
}

namespace {
__global__ void exp_max_kernel(int64_t n, const int* __restrict__ e, int* __restrict__ out) {
  __shared__ int red[256];
  int m = -100000;
  for (int64_t i = threadIdx.x; i < n; i += 256) m = max(m, e[i]);
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = 128; w >= 1; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] = max(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}
}  // namespace

cudaError_t ozaki_left_exp_max(cudaStream_t s, int64_t M, OzakiWork& w, int* out) {
  if (M <= 0) return cudaSuccess;
  exp_max_kernel<<<1, 256, 0, s>>>(M, w.el, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t ozaki_group_reserve(OzakiGroupTable& t, size_t entries) {
  if (entries <= t.capacity) return cudaSuccess;
  ozaki_group_free(t);
  cudaError_t e;
  if ((e = cudaMalloc(&t.dev, entries * sizeof(OzGroupEntry))) != cudaSuccess) return e;
  if ((e = cudaMallocHost(&t.host, entries * sizeof(OzGroupEntry))) != cudaSuccess) return e;
  if ((e = cudaMalloc(&t.sdev, entries * sizeof(OzSliceEntry))) != cudaSuccess) return e;
  if ((e = cudaMallocHost(&t.shost, entries * sizeof(OzSliceEntry))) != cudaSuccess) return e;
  t.capacity = entries;
  return cudaSuccess;
}

void ozaki_group_free(OzakiGroupTable& t) {
  if (t.dev) cudaFree(t.dev);
  if (t.host) cudaFreeHost(t.host);
  if (t.sdev) cudaFree(t.sdev);
  if (t.shost) cudaFreeHost(t.shost);
  t = OzakiGroupTable{};
}

size_t ozaki_group_entries(int count, const OzakiGroupItem* items) {
  size_t n = 0;
  for (int k = 0; k < count; ++k)
    if (items[k].ncols > 0) n += (size_t)items[k].degs[items[k].ncols - 1];
  return n;
}

int ozaki_filter_grouped(cudaStream_t s, int count, const OzakiGroupItem* items,
                         OzakiGroupTable& t, int* launches) {
  static std::once_flag attr_once[kMaxDevices];
  once_per_device(attr_once, []() {
    cudaFuncSetAttribute(ozaki_filter_grouped_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         SMEM_BYTES);
  });
  int dmax_all = 0;
  for (int k = 0; k < count; ++k) {
    const OzakiGroupItem& it = items[k];
    if (it.ncols == 0) continue;
    if (!it.w || !it.w->maps || !it.w->A_ready || it.N != it.w->N || it.ncols > it.w->ne ||
        !it.V || !it.W || it.ldv < it.N || it.ldw < it.N)
      return CHASE_ERR_INVALID_ARG;
    dmax_all = std::max(dmax_all, (int)it.degs[it.ncols - 1]);
  }
  if (dmax_all == 0) return CHASE_OK;
  if (ozaki_group_entries(count, items) > t.capacity) return CHASE_ERR_INVALID_ARG;
  // step table: for step i the entries of the problems still filtering, with
  // their first CTA indices (gemm) and first column indices (digits)
  OzGroupEntry* host = static_cast<OzGroupEntry*>(t.host);
  OzSliceEntry* shost = static_cast<OzSliceEntry*>(t.shost);
  std::vector<size_t> off(dmax_all + 2, 0);
  std::vector<int> ctas(dmax_all + 1, 0), cols(dmax_all + 1, 0), cluster(dmax_all + 1, 1);
  size_t n = 0;
  for (int i = 1; i <= dmax_all; ++i) {
    off[i] = n;
    int first = 0, sfirst = 0;
    for (int k = 0; k < count; ++k) {
      const OzakiGroupItem& it = items[k];
      if (it.ncols == 0 || it.degs[it.ncols - 1] < i) continue;
      OzakiWork& w = *it.w;
      // the per-problem filter's step i (Eq. 1): Y_d = al[i] (A - c I) Y_s + be[i] Y_d
      const int64_t j0 = std::lower_bound(it.degs, it.degs + it.ncols, i) - it.degs;
      double2* buf[2] = {it.V, it.W};
      const int64_t ld[2] = {it.ldv, it.ldw};
      const int sp = (i - 1) & 1, d = i & 1;
      Epilogue ep{};
      ep.mode = EPI_FILTER;
      ep.alpha = it.al[i];
      ep.beta = (i == 1) ? 0.0 : it.be[i];
      ep.gamma = it.c;
      ep.X = buf[sp];
      ep.ldx = ld[sp];
      ep.Y = buf[d];
      ep.ldy = ld[d];
      OzSliceEntry& se = shost[n];
      se.B = buf[sp];
      se.ldb = ld[sp];
      se.N = it.N;
      se.Np = w.Np;
      se.brows = w.brows;
      se.j0 = j0;
      se.eb = w.eb;
      se.out = static_cast<__nv_bfloat16*>(w.Bd);
      se.first = sfirst;
      se.pad = 0;
      sfirst += (int)(it.ncols - j0);
      OzGroupEntry& e = host[n];
      const Maps* maps = static_cast<const Maps*>(w.maps);
      e.a = maps->a;
      e.b = maps->b;
      e.P = product_params(w, it.ncols, j0, buf[sp], ld[sp], ep);
      e.pad = 0;
      cluster[i] = std::max(cluster[i], e.P.split);
      ++n;
    }
    // a cluster holds CTAs of one problem: each starts on a cluster boundary
    for (size_t q = off[i]; q < n; ++q) {
      host[q].first = first;
      first += (int)cdiv((int64_t)host[q].P.nrow * host[q].P.ncol * host[q].P.split, cluster[i]) *
               cluster[i];
    }
    ctas[i] = first;
    cols[i] = sfirst;
  }
  off[dmax_all + 1] = n;
  if (cudaMemcpyAsync(t.dev, host, n * sizeof(OzGroupEntry), cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaMemcpyAsync(t.sdev, shost, n * sizeof(OzSliceEntry), cudaMemcpyHostToDevice, s) !=
          cudaSuccess)
    return CHASE_CUDA_FAIL();
  // the degree steps of all problems as one CUDA graph: per step one grouped
  // digit launch and one grouped product launch
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
    return CHASE_CUDA_FAIL();
  const OzGroupEntry* dev = static_cast<const OzGroupEntry*>(t.dev);
  const OzSliceEntry* sdev = static_cast<const OzSliceEntry*>(t.sdev);
  cudaError_t first = cudaSuccess;  // a graph without one of its steps is not launched
  for (int i = 1; i <= dmax_all && first == cudaSuccess; ++i) {
    const int cnt = (int)(off[i + 1] - off[i]);
    slice_b_grouped_kernel<<<(unsigned)cols[i], 256, 0, s>>>(sdev + off[i], cnt);
    count_launch();
    if ((first = cudaGetLastError()) == cudaSuccess)
      first = launch_clusters(ozaki_filter_grouped_kernel, (unsigned)ctas[i], cluster[i], false, s,
                              dev + off[i], cnt, cluster[i] > 1);
  }
  const cudaError_t ce = cudaStreamEndCapture(s, &graph);
  if (first != cudaSuccess || ce != cudaSuccess || !graph) {
    if (ce == cudaSuccess && graph) cudaGraphDestroy(graph);
    return CHASE_CUDA_FAIL();
  }
  const cudaError_t ie = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (ie != cudaSuccess) return CHASE_CUDA_FAIL();
  const cudaError_t le = cudaGraphLaunch(exec, s);
  const cudaError_t se = le == cudaSuccess ? cudaStreamSynchronize(s) : le;
  cudaGraphExecDestroy(exec);
  if (se != cudaSuccess) return CHASE_CUDA_FAIL();
  if (launches) *launches = 2 * dmax_all;
  int rc = CHASE_OK;
  for (int k = 0; k < count; ++k)
    if (items[k].ncols > 0) {
      const int r = ozaki_check(s, *items[k].w);
      if (rc == CHASE_OK) rc = r;
    }
  return rc;
}

int ozaki_check(cudaStream_t s, OzakiWork& w) {
  int herr = 0;
  if (cudaMemcpyAsync(&herr, w.err, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CHASE_CUDA_FAIL();
  if (herr != 0) {
    fprintf(stderr, "[chase] emulated-FP64 GEMM: pipeline wait expired (code %d)\n", herr);
    cudaMemsetAsync(w.err, 0, sizeof(int), s);
    return CHASE_CUDA_FAIL();
  }
  return CHASE_OK;
}

}  // namespace chase
