// Products with H on the BF16 tensor cores (tcgen05) in residue arithmetic:
//
//   C[:, j] = alpha * (H X[:, j] - shift * X[:, j]) + beta * C[:, j],  j in [j0, j1)
//
// Why.  GB300 runs FP64 at about 1 TFLOP/s and BF16 at about 1.7 PFLOP/s.  A
// product of integer matrices can be formed modulo a set of small coprime
// numbers, one plain BF16 GEMM per modulus, and put back together by the
// Chinese remainder theorem (the idea of Ozaki, Uchino and Imamura's "Ozaki
// scheme II", arXiv 2504.08009, there for INT8): n moduli of 9 bits cover a
// product of 9n bits, where cutting both operands into s digits takes
// s (s + 1) / 2 GEMMs for the same accuracy.
//
//  * Operands become integers: row r of H is scaled by 2^s_r so that its
//    2-norm is just below 2^L, column c of X by 2^s_c likewise, and rounded.
//    By Cauchy-Schwarz every entry of the product is below 2^(2L) < P / 2
//    with P the product of the moduli, so it is determined by its residues:
//    the integer product is exact whatever the entries are, and the only
//    error is the rounding of the operands, 2^-L of a row's or column's norm
//    (11 moduli: L = 48; 14 moduli: L = 60, below the rounding of an FP64
//    GEMM; 7 moduli: L = 30).
//  * Complex products take two real GEMMs per modulus instead of four: the
//    moduli are products of primes = 1 mod 4, so each has a j with j^2 = -1,
//    and (ar + j ai)(br + j bi), (ar - j ai)(br - j bi) mod p are re + j im
//    and re - j im of the product.  11 moduli execute 5.5 BF16 FLOPs per
//    algorithmic FLOP (a split of both operands into seven 7-bit digits: 28).
//  * Residues lie in [-255, 255] and are exact in BF16.  Their products sum
//    exactly in the FP32 accumulator while K h^2 <= 2^24 (h = (p + 1) / 2),
//    i.e. over a chunk of 256 to 448 K, after which the epilogue warps reduce
//    the accumulator modulo p into FP32 registers.  Two accumulators take
//    turns, so the tensor pipe never waits for that reduction.
//
// The result does not depend on tile shapes, K order or what else runs: it
// is an integer.
//
// Structure of the GEMM kernel (a CTA pair = 256 rows of H x BN columns):
// both CTAs' warp 0 load their half of the operands by TMA (64-wide K,
// 128-byte swizzle) into a ring of stages whose barriers live in the even
// CTA; its warp 1 issues tcgen05.mma.cta_group::2 (M = 256, N = BN), so each
// CTA reads only half of B from shared memory; warps 2-17 of each CTA reduce
// and store its 128 rows.  Persistent pairs walk the tiles of all residue
// planes.  Every wait is bounded.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <type_traits>

#include "common.cuh"
#include "context.hpp"

namespace chase {
namespace rns {

// Pairwise coprime, every prime factor = 1 mod 4, largest first.
constexpr int kModuli[kRnsMaxModuli] = {509, 505, 493, 481, 461, 457, 449,
                                        433, 421, 409, 401, 397, 389, 373};
constexpr int BM = 128;          // rows per CTA (256 per pair)
constexpr int BK = 64;           // K per stage: one 128-byte swizzle row
constexpr int kEpiWarps = 16;    // four per TMEM lane quarter
constexpr int kThreads = (2 + kEpiWarps) * 32;
constexpr int kLimbBits = 13;
constexpr int kNonFinite = 0x7fffffff;  // exponent of a row or column with an Inf or NaN
constexpr float kRound = 12582912.f;    // 1.5 * 2^23: adding it rounds to an integer

// ---------------------------------------------------------------------------
// PTX helpers for CTA pairs
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::
                   : "memory");
}
// True in one lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile(
      "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(e));
  return e != 0;
}
// Address, in the cluster's shared window, of the same variable in CTA `rank`.
__device__ __forceinline__ uint32_t map_to_rank(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
// The barriers of a pair order TMA writes, MMAs and TMEM reads, all of which
// complete before the arrival that announces them (complete_tx, commit,
// tcgen05.wait::ld); no generic-proxy data passes between the CTAs.  So CTA
// scope is enough: at cluster scope every wait and arrival drained the warp's
// memory pipe first, the largest stall of the GEMM (N = 4096, 788 columns, 22
// planes: 701 -> 669 us).
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n"
      " mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// A whole warp's wait, with one answer for all lanes: lanes that disagreed about
// a time-out would part and wait for one another in different places.
__device__ __forceinline__ bool wait_cluster_bounded(uint64_t* bar, uint32_t parity) {
  if (__all_sync(0xffffffffu, try_wait_cluster(bar, parity))) return true;
  const long long t0 = clock64();
  while (!__all_sync(0xffffffffu, try_wait_cluster(bar, parity))) {
    if (__any_sync(0xffffffffu, clock64() - t0 > kWaitBudgetCycles)) return false;
  }
  return true;
}
// TMA load into this CTA's shared memory, completion counted on a barrier of
// either CTA of the pair.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int x, int y,
                                              int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                          uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}
// Arrive on the barrier at this offset in both CTAs once every MMA issued so
// far has completed.
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
  asm volatile(
      "{\n .reg .b16 m;\n mov.b16 m, 3;\n"
      " tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], m;\n}\n" ::"r"(smem_u32(bar))
      : "memory");
}
// K-major operand, 128-byte swizzled rows: 8-row atoms of 1024 bytes.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;             // LBO (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;   // SBO: 8 rows x 128 B
  d |= (uint64_t)1 << 46;             // version
  d |= (uint64_t)2 << 61;             // SWIZZLE_128B
  return d;
}

// MN-major operand: 128-byte swizzled rows along M, one per K, in 8-row atoms
// of 1024 bytes; the next 64 of M come 8192 bytes on.
__device__ __forceinline__ uint64_t desc_sw128_mn(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(8192 >> 4) << 16;   // LBO: the next 64 of M
  d |= (uint64_t)(1024 >> 4) << 32;   // SBO: the next 8 of K
  d |= (uint64_t)1 << 46;             // version
  d |= (uint64_t)2 << 61;             // SWIZZLE_128B
  return d;
}

// 8 columns of this thread's row of an accumulator.  The load is asynchronous:
// its registers may not be read, and so not packed in pairs either, before
// tmem_wait_ld, through which they pass so that no use can be scheduled earlier.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&u)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]),
                 "=r"(u[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&u)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]),
                 "+r"(u[7])::"memory");
}
// Two FP32 operations in one instruction, each rounded as its scalar form.
__device__ __forceinline__ unsigned long long pack_b32x2(uint32_t lo, uint32_t hi) {
  return static_cast<unsigned long long>(lo) | static_cast<unsigned long long>(hi) << 32;
}
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi) {
  return pack_b32x2(__float_as_uint(lo), __float_as_uint(hi));
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b,
                                                        unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long add_f32x2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// ---------------------------------------------------------------------------
// The residue GEMM: G[plane] = A[plane] B[plane] mod p, entries in
// [-(p+1)/2, (p+1)/2] as int16
// ---------------------------------------------------------------------------
template <int BN_>
struct Cfg {
  static constexpr int BN = BN_;
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = (BN / 2) * BK * 2;
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int NSTAGE = 196608 / STAGE > 8 ? 8 : 196608 / STAGE;
  static constexpr int BUF = BN <= 32 ? 32 : BN <= 64 ? 64 : BN <= 128 ? 128 : 256;
  static constexpr int TMEM = 2 * BUF;  // two accumulators
  static constexpr int HC = BN / 4;     // columns per epilogue warp
  // more than half an SM's shared memory: one CTA per SM, so the pairs of
  // concurrent kernels never wait for one another's TMEM
  static constexpr int SMEM = 1024 + NSTAGE * STAGE + 256;
  static_assert(BN % 32 == 0 && BN >= 32 && BN <= 256, "tile columns");
  static_assert(SMEM > 116 * 1024 && SMEM <= 232448, "shared memory per CTA");
};

// Per modulus of the GEMM kernel: p, 1 / p and the stages of one exact chunk.
struct Modulus {
  float p, invp;
  int chunk;
};
struct GemmTab {
  Modulus m[kRnsMaxModuli];
};

// One output tile (256 rows x BN columns of one residue plane).
struct Tile {
  const CUtensorMap* mapA;
  const CUtensorMap* mapB;
  int row0, col0;      // first row, first column of the tile
  int planeA, planeB;  // plane of A and of B
  bool trans;          // the tile of A is a transposed one of its plane
  // whether the stage at k loads a transposed tile: with TRI, right of the
  // diagonal's 256 x 256 block
  template <bool TRI>
  __device__ __forceinline__ bool transposed(int k) const {
    return TRI ? k >= row0 + 2 * BM : trans;
  }
  int modulus;         // index of the plane's modulus
  int nst;             // stages (K / 64, rounded up)
  int M, ncols;        // rows, columns of the product
  int16_t* G;          // the plane's residues, column-major
  long long ldg;
};

// The pair's tiles: first, first + step, ... below last.
struct Walk {
  int first, last, step;
};
template <int BN, class TileFn>
__device__ __forceinline__ void gemm_body(TileFn& tile, const Walk w, const GemmTab& tab,
                                          int maps_in_global, int* __restrict__ err) {
  using C = Cfg<BN>;
  constexpr int NSTAGE = C::NSTAGE;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* sA = sm;
  unsigned char* sB = sm + NSTAGE * C::A_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + NSTAGE * C::STAGE);  // [NSTAGE] (even CTA)
  uint64_t* empty = full + NSTAGE;          // [NSTAGE] (each CTA)
  uint64_t* acc_full = empty + NSTAGE;      // [2] (each CTA)
  uint64_t* acc_empty = acc_full + 2;       // [2] (even CTA)
  uint64_t* done = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * kEpiWarps);
    }
    mbar_init(done, 1);
    fence_barrier_init();
  }
  __syncthreads();
  cluster_sync();  // both CTAs are running before the pair allocates TMEM
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(C::TMEM));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  cluster_sync();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // the set-up above overlaps the kernel before; its results are read below
  pdl_wait();

  // Warps 0 and 1 run their loops with all lanes, and one elected lane issues:
  // with only lane 0 in the loop the operands of every TMA and MMA went
  // through per-instruction transfers to uniform registers, and the tensor
  // pipe idled between the MMAs of a stage (same product: 669 -> 528 us).
  const bool leader = elect_one();
  if (warp == 0) {
    {  // ---------------- TMA producer (both CTAs)
      // Stage and parity are counted along: these loops have a few hundred
      // cycles per stage, and 64-bit divisions for them took 4 to 5 % of every
      // product.  A wait for the phase before a barrier's first returns at once.
      long long g = 0;  // stages issued by this CTA
      int st = 0;
      uint32_t ph = 1;
      bool ok = true;
      const CUtensorMap* last = nullptr;
      for (int t = w.first; t < w.last && ok; t += w.step) {
        Tile T;
        tile(t, T);
        if (T.mapA != last) {
          if (leader) {
            if (maps_in_global) {
              asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;\n" ::"l"(T.mapA)
                           : "memory");
              asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;\n" ::"l"(T.mapB)
                           : "memory");
            }
            prefetch_tmap(T.mapA);
            prefetch_tmap(T.mapB);
          }
          last = T.mapA;
        }
        const int ra = T.row0 + static_cast<int>(rank) * BM;
        const int cb = T.col0 + static_cast<int>(rank) * (BN / 2);
        for (int ks = 0; ks < T.nst; ++ks, ++g) {
          if (!wait_cluster_bounded(&empty[st], ph)) {
            if (leader) atomicOr(err, KERR_TIMEOUT_EMPTY);
            ok = false;
            break;
          }
          const uint32_t bar = map_to_rank(&full[st], 0);
          if (leader) {
            if (rank == 0) mbar_arrive_expect_tx(&full[st], 2 * C::STAGE);
            // two boxes of 64 x 64: 64 rows each, or 64 of M each when transposed
            const uint32_t a = smem_u32(sA + st * C::A_BYTES);
            const bool tr = T.template transposed<TileFn::kTri>(ks * BK);
            const int x = tr ? ra : ks * BK, y = tr ? ks * BK : ra;
            tma_load_pair(a, T.mapA, x, y, T.planeA, bar);
            tma_load_pair(a + C::A_BYTES / 2, T.mapA, tr ? x + 64 : x, tr ? y : y + 64, T.planeA,
                          bar);
            tma_load_pair(smem_u32(sB + st * C::B_BYTES), T.mapB, ks * BK, cb, T.planeB, bar);
          }
          if (++st == NSTAGE) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
      // no copy may be in flight when the pair ends (the even CTA's barriers
      // count the copies of both; the odd CTA waits at the cluster barrier)
      if (rank == 0)
        for (long long k = (g > NSTAGE ? g - NSTAGE : 0); k < g; ++k)
          if (!wait_cluster_bounded(&full[k % NSTAGE], static_cast<uint32_t>((k / NSTAGE) & 1)) &&
              leader)
            atomicOr(err, KERR_TIMEOUT_FULL);
    }
  } else if (warp == 1) {
    if (rank == 0) {  // ---------------- MMA issuer
      // kind::f16: FP32 D, BF16 A and B, K-major (bit 15: A MN-major), M = 256, N = BN
      constexpr uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) |
                                  ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);
      const uint64_t ak = desc_sw128(smem_u32(sA)), amn = desc_sw128_mn(smem_u32(sA));
      const uint64_t b0 = desc_sw128(smem_u32(sB));
      bool ok = true;
      int st = 0, buf = 0;               // stage, accumulator
      uint32_t ph = 0, acc_ph = 1;
      for (int t = w.first; t < w.last && ok; t += w.step) {
        Tile T;
        tile(t, T);
        const int cs = tab.m[T.modulus].chunk;
        for (int k0 = 0; k0 < T.nst && ok; k0 += cs) {  // a chunk per accumulator
          if (!wait_cluster_bounded(&acc_empty[buf], acc_ph)) {
            if (leader) atomicOr(err, KERR_TIMEOUT_FULL);
            ok = false;
            break;
          }
          const int k1 = min(k0 + cs, T.nst);
          const uint32_t d = tmem + static_cast<uint32_t>(buf) * C::BUF;
          for (int ks = k0; ks < k1; ++ks) {
            if (!wait_cluster_bounded(&full[st], ph)) {
              if (leader) atomicOr(err, KERR_TIMEOUT_FULL);
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const bool tr = T.template transposed<TileFn::kTri>(ks * BK);
            const uint32_t idesc = tr ? idesc0 | (1u << 15) : idesc0;
            const uint64_t da = (tr ? amn : ak) + static_cast<uint64_t>(st * (C::A_BYTES >> 4));
            const uint64_t db = b0 + static_cast<uint64_t>(st * (C::B_BYTES >> 4));
            const uint64_t step = (tr ? 16 * 128 : 32) >> 4;  // 16 of K
            if (leader) {
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                umma_pair(d, da + k * step, db + k * (32 >> 4), idesc,
                          (ks == k0 && k == 0) ? 0u : 1u);
              commit_pair(&empty[st]);
              if (ks == k1 - 1) commit_pair(&acc_full[buf]);
            }
            if (++st == NSTAGE) {
              st = 0;
              ph ^= 1u;
            }
          }
          buf ^= 1;
          if (buf == 0) acc_ph ^= 1u;
        }
      }
      // every MMA of this pair has completed when this fires
      if (leader) commit_pair(done);
      __syncwarp();
      if (!wait_cluster_bounded(done, 0) && leader) atomicOr(err, KERR_TIMEOUT_FULL);
    }
  } else {
    // ---------------- reduction (warps 2..17): lanes 32 (w % 4) .. +31 (one
    // row each), quarter hf of the columns
    const int q = warp & 3;
    const int hf = (warp - 2) >> 2;
    const int rit = static_cast<int>(rank) * BM + q * 32 + lane;  // row in the tile
    const uint32_t tbase = tmem + (static_cast<uint32_t>(q * 32) << 16) + hf * C::HC;
    const uint32_t bar_e0 = map_to_rank(&acc_empty[0], 0), bar_e1 = map_to_rank(&acc_empty[1], 0);
    unsigned c = 0;  // chunk: accumulator c & 1, its phase c >> 1
    bool ok = true;
    for (int t = w.first; t < w.last && ok; t += w.step) {
      Tile T;
      tile(t, T);
      const Modulus m = tab.m[T.modulus];
      // column pairs: packed FP32 arithmetic halves the instructions of what
      // bounded the kernel then (same product: 528 -> 442 us; four warps per
      // lane quarter instead of two, a load ahead: 426 us, 1.36 PFLOP/s)
      unsigned long long acc[C::HC / 2];
#pragma unroll
      for (int j = 0; j < C::HC / 2; ++j) acc[j] = 0ull;
      const unsigned long long invp2 = pack_f32x2(m.invp, m.invp), mp2 = pack_f32x2(-m.p, -m.p),
                               rnd2 = pack_f32x2(kRound, kRound),
                               mrnd2 = pack_f32x2(-kRound, -kRound);
      for (int left = T.nst; left > 0; left -= m.chunk, ++c) {
        if (!wait_cluster_bounded(&acc_full[c & 1], static_cast<uint32_t>((c >> 1) & 1))) {
          if (lane == 0) atomicOr(err, KERR_TIMEOUT_FULL);
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t tb = tbase + static_cast<uint32_t>(c & 1) * C::BUF;
        // the load of the next 8 columns is in flight while these are reduced
        uint32_t r[2][8];
        tmem_ld8(tb, r[0]);
#pragma unroll
        for (int j0 = 0; j0 < C::HC; j0 += 8) {
          tmem_wait_ld(r[(j0 / 8) & 1]);
          if (j0 + 8 < C::HC) tmem_ld8(tb + j0 + 8, r[(j0 / 8 + 1) & 1]);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // |v| <= 2^24, an integer; v - p rint(v / p), exact
            const unsigned long long v =
                pack_b32x2(r[(j0 / 8) & 1][2 * j], r[(j0 / 8) & 1][2 * j + 1]);
            const unsigned long long k = add_f32x2(fma_f32x2(v, invp2, rnd2), mrnd2);
            acc[j0 / 2 + j] = add_f32x2(acc[j0 / 2 + j], fma_f32x2(k, mp2, v));
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) arrive_cluster((c & 1) ? bar_e1 : bar_e0);
      }
      if (!ok) break;
      const int row = T.row0 + rit;
      if (row < T.M) {
        const int cb = T.col0 + hf * C::HC;
        int16_t* gp = T.G + static_cast<long long>(cb) * T.ldg + row;
#pragma unroll
        for (int j = 0; j < C::HC; ++j) {
          if (cb + j < T.ncols) {
            const float a = __uint_as_float(
                static_cast<uint32_t>(j % 2 ? acc[j / 2] >> 32 : acc[j / 2]));
            const float k = __fadd_rn(fmaf(a, m.invp, kRound), -kRound);
            const float x = fmaf(-k, m.p, a);
            // the low bits of x + 1.5 * 2^23 are x as a two's complement integer
            gp[j * T.ldg] = static_cast<int16_t>(__float_as_uint(__fadd_rn(x, kRound)) & 0xffffu);
          }
        }
      }
    }
  }
  // not earlier: blocks of the next kernel would gather, waiting, on the SMs
  // whose pairs end first, and run there alone
  pdl_next();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  cluster_sync();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(C::TMEM));
}

// Tiles of one product: the column tile runs fastest, so the pairs working at
// one time share rows of A and the B plane stays in L2; then row tiles, then
// planes.
template <bool TRI>
struct OneProduct {
  static constexpr bool kTri = TRI;
  const CUtensorMap* mapA;
  const CUtensorMap* mapB;
  int rtiles, ctiles, plane0, per_modulus, swap_a, sym, bn, nst, M, ncols;
  int16_t* G;
  long long ldg, gplane;
  __device__ __forceinline__ void operator()(int t, Tile& T) const {
    const int ct = t % ctiles, rest = t / ctiles;
    const int rt = rest % rtiles, pl = rest / rtiles;
    T.mapA = mapA;
    T.mapB = mapB;
    T.row0 = rt * 2 * BM;
    T.col0 = ct * bn;
    T.planeA = sym ? pl >> 1 : pl ^ swap_a;
    T.trans = sym && (pl & 1);
    T.planeB = plane0 + pl;
    T.modulus = T.planeB / per_modulus;
    T.nst = nst;
    T.M = M;
    T.ncols = ncols;
    T.G = G + T.planeB * gplane;
    T.ldg = ldg;
  }
};

// TRI is a template parameter: its test in every stage, where no stage needs it,
// made a warm split solve's filter at N = 4095 6 % slower.
template <int BN, bool TRI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    rns_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ GemmTab tab, int rtiles, int ctiles, int nplanes,
                    int plane0, int per_modulus, int swap_a, int sym, int nst, int M, int ncols,
                    int16_t* __restrict__ G,
                    long long ldg, long long gplane, int* __restrict__ err) {
  OneProduct<TRI> p{&tmA, &tmB, rtiles, ctiles, plane0, per_modulus, swap_a, sym, BN, nst, M, ncols,
               G, ldg, gplane};
  gemm_body<BN>(p, Walk{static_cast<int>(blockIdx.x >> 1), rtiles * ctiles * nplanes,
                        static_cast<int>(gridDim.x >> 1)},
                tab, 0, err);
}

// ---------------------------------------------------------------------------
// Residues of an operand.  x = round(v 2^s) is cut into 13-bit limbs centred
// on zero, x = sum_k l_k 2^(13 k); x mod p is sum_k l_k (2^(13 k) mod p)
// reduced once: every partial sum stays below 2^24, so FP32 holds it exactly,
// and FP32 runs 64 times wider than this GPU's FP64 pipe.
// ---------------------------------------------------------------------------
struct SliceMod {  // each constant twice, for packed arithmetic on two entries
  unsigned long long mp, invp;  // -p, 1 / p
  unsigned long long c[5];      // 2^(13 k) mod p, centred
  unsigned long long jc[5];     // j 2^(13 k) mod p, centred
};
struct SliceTab {
  SliceMod m[kRnsMaxModuli];
  float log2_norm;  // L: the scaled 2-norm stays below 2^L
};

// High word of |v|: exponent and 20 leading mantissa bits.
__device__ __forceinline__ uint32_t abs_hi(double v) {
  return static_cast<uint32_t>(__double2hiint(v)) & 0x7FFFFFFFu;
}
// |v| 2^-off as FP32, truncated, from its bits (no FP64 arithmetic: that pipe
// is 64 times narrower); 0 below FP32's normal range.
__device__ __forceinline__ float abs_f32(double v, int off) {
  const int h = static_cast<int>(abs_hi(v)) - (896 + off) * (1 << 20);
  const uint32_t f = (static_cast<uint32_t>(h) << 3) | (static_cast<uint32_t>(__double2loint(v)) >> 29);
  return h >= (1 << 20) ? __uint_as_float(h < (255 << 20) ? f : 0x7F7FFFFFu) : 0.f;
}
__device__ __forceinline__ uint32_t low_word(double v) {
  return static_cast<uint32_t>(__double2loint(v));
}
// The same of an FP32 value: the high word of |v| as a double.
__device__ __forceinline__ uint32_t abs_hi(float v) {
  const float a = fabsf(v);
  if (!(a < INFINITY)) return 0x7FF00000u;
  if (a == 0.f) return 0u;
  const bool small = a < 1.17549435e-38f;  // denormal: normalise, exactly
  const uint32_t u = __float_as_uint(small ? a * 16777216.f : a);
  return (u >> 3) + ((small ? 896u - 24u : 896u) << 20);
}
__device__ __forceinline__ float abs_f32(float v, int off) {
  return off == 0 ? fabsf(v) : scalbnf(fabsf(v), -off);
}
__device__ __forceinline__ uint32_t low_word(float) { return 0u; }

// round(v 2^s) (ties away from zero), |v 2^s| < 2^62
__device__ __forceinline__ long long scaled_int(double v, int s) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(v));
  const int eb = static_cast<int>((bits >> 52) & 0x7FF);
  unsigned long long m = bits & ((1ull << 52) - 1);
  int sh = s - 1074;  // v = m 2^sh after scaling
  if (eb != 0) {
    m |= 1ull << 52;
    sh = s + eb - 1075;
  }
  unsigned long long x;
  if (sh >= 0)
    x = m << sh;
  else
    x = sh > -64 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0ull;
  return (bits >> 63) ? -static_cast<long long>(x) : static_cast<long long>(x);
}

__device__ __forceinline__ long long scaled_int(float v, int s) {
  const uint32_t bits = __float_as_uint(v);
  const int eb = static_cast<int>((bits >> 23) & 0xFF);
  unsigned long long m = bits & ((1u << 23) - 1);
  int sh = s - 149;
  if (eb != 0) {
    m |= 1ull << 23;
    sh = s + eb - 150;
  }
  unsigned long long x;
  if (sh >= 0)
    x = m << sh;
  else
    x = sh > -64 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0ull;
  return (bits >> 31) ? -static_cast<long long>(x) : static_cast<long long>(x);
}

// Limbs 0 .. NL-2 in [-4096, 4095], the top one what is left.
template <int NL>
__device__ __forceinline__ void limbs(long long x, float* l) {
  constexpr long long kHalf = 1LL << (kLimbBits - 1);
  long long bias = 0;
#pragma unroll
  for (int k = 0; k < NL - 1; ++k) bias += kHalf << (kLimbBits * k);
  const long long y = x + bias;
#pragma unroll
  for (int k = 0; k < NL - 1; ++k) {
    const unsigned u = static_cast<unsigned>(y >> (kLimbBits * k)) & ((1u << kLimbBits) - 1);
    l[k] = __fadd_rn(__uint_as_float(0x4B000000u | u), -(8388608.f + 4096.f));
  }
  const int top = static_cast<int>(y >> (kLimbBits * (NL - 1)));
  l[NL - 1] = __fadd_rn(__uint_as_float(0x4B400000u + static_cast<unsigned>(top)), -kRound);
}

__device__ __forceinline__ unsigned long long reduce2(unsigned long long n, const SliceMod& m) {
  const unsigned long long k = add_f32x2(fma_f32x2(n, m.invp, pack_f32x2(kRound, kRound)),
                                         pack_f32x2(-kRound, -kRound));
  return fma_f32x2(k, m.mp, n);
}

// Two small integers as packed BF16 (exact: their FP32 bits end in zeros).
__device__ __forceinline__ uint32_t pack2(unsigned long long v) {
  return __byte_perm(static_cast<uint32_t>(v), static_cast<uint32_t>(v >> 32), 0x7632);
}

__device__ __forceinline__ double re_of(double2 v) { return v.x; }
__device__ __forceinline__ double im_of(double2 v) { return v.y; }
__device__ __forceinline__ double re_of(float2 v) { return v.x; }
__device__ __forceinline__ double im_of(float2 v) { return v.y; }
__device__ __forceinline__ double re_of(double v) { return v; }
__device__ __forceinline__ double im_of(double) { return 0.0; }
__device__ __forceinline__ double re_of(float v) { return v; }
__device__ __forceinline__ double im_of(float) { return 0.0; }

// The same in the operand's own type.
__device__ __forceinline__ double re_in(double2 v) { return v.x; }
__device__ __forceinline__ double im_in(double2 v) { return v.y; }
__device__ __forceinline__ float re_in(float2 v) { return v.x; }
__device__ __forceinline__ float im_in(float2 v) { return v.y; }
__device__ __forceinline__ double re_in(double v) { return v; }
__device__ __forceinline__ double im_in(double) { return 0.0; }
__device__ __forceinline__ float re_in(float v) { return v; }
__device__ __forceinline__ float im_in(float) { return 0.f; }

template <class E>
constexpr bool is_single = std::is_same<E, float2>::value || std::is_same<E, float>::value;
template <class E>
constexpr bool is_complex = std::is_same<E, double2>::value || std::is_same<E, float2>::value;

constexpr int kSliceThreads = 256;

// Sum of ss and maximum of mb over the block.
__device__ __forceinline__ void reduce_block(float& ss, uint32_t& mb, float* sf, uint32_t* su) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) {
    sf[warp] = ss;
    su[warp] = mb;
  }
  __syncthreads();
  ss = 0.f;
  mb = 0;
#pragma unroll
  for (int w = 0; w < kSliceThreads / 32; ++w) {
    ss += sf[w];
    mb = max(mb, su[w]);
  }
}

// The range of largest magnitudes whose FP32 squares neither overflow nor
// lose a part of the sum that matters: [2^-40, 2^40).
constexpr uint32_t kSafeLo = (1023 - 40) << 20, kSafeHi = (1023 + 40) << 20;

// Exponent s with ||v|| 2^s just below 2^L for n real entries with largest
// magnitude (high word) mb and ||v 2^-off||^2 = ss, as FP32 sums it:
// truncated entries and the summation take off less than the margin.
__device__ __forceinline__ int scale_exponent(float ss, uint32_t mb, int off, float n, float L) {
  if (mb >= 0x7FF00000u) return kNonFinite;
  const float margin = 2e-4f + 1e-9f * n;
  if (mb < (1u << 20))  // zero or denormal: all below 2^-1022
    return ss == 0.f && mb == 0 ? 0 : static_cast<int>(floorf(L - margin - 0.5f * log2f(n))) + 1022;
  return static_cast<int>(floorf(L - margin - 0.5f * log2f(ss))) - off;
}

// Residues in planes [m0, m1) of two neighbouring integers (xr + i xi).
// With BOTH the plane of re - j im follows that of re + j im.
template <int NM, int NL, bool CP, bool BOTH = CP>
__device__ __forceinline__ void store_residues(const long long (&xr)[2], const long long (&xi)[2],
                                               __nv_bfloat16* __restrict__ o, long long stride,
                                               const SliceTab& tab, int m0, int m1) {
  float lr[2][NL], li[2][NL];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    limbs<NL>(xr[h], lr[h]);
    if constexpr (CP) limbs<NL>(xi[h], li[h]);
  }
  unsigned long long pr[NL], pi[NL];
#pragma unroll
  for (int i = 0; i < NL; ++i) {
    pr[i] = pack_f32x2(lr[0][i], lr[1][i]);
    if constexpr (CP) pi[i] = pack_f32x2(li[0][i], li[1][i]);
  }
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    if (m < m0 || m >= m1) continue;
    const SliceMod& t = tab.m[m];
    unsigned long long nr = pr[0];
#pragma unroll
    for (int i = 1; i < NL; ++i) nr = fma_f32x2(pr[i], t.c[i], nr);
    if constexpr (CP) {
      unsigned long long ni = fma_f32x2(pi[0], t.jc[0], 0ull);
#pragma unroll
      for (int i = 1; i < NL; ++i) ni = fma_f32x2(pi[i], t.jc[i], ni);
      *reinterpret_cast<uint32_t*>(o) = pack2(reduce2(add_f32x2(nr, ni), t));
      if constexpr (BOTH)
        *reinterpret_cast<uint32_t*>(o + stride) =
            pack2(reduce2(fma_f32x2(ni, pack_f32x2(-1.f, -1.f), nr), t));
      o += BOTH ? 2 * stride : stride;
    } else {
      *reinterpret_cast<uint32_t*>(o) = pack2(reduce2(nr, t));
      o += stride;
    }
  }
}

// Exponent (scale_exponent) of a vector of n entries, the one at `skip` left
// out; *nonzero: whether any other is not zero.  Block-wide.
template <class E>
__device__ __forceinline__ int vector_exponent(const E* __restrict__ v, int n, int skip, float L,
                                               bool* nonzero) {
  constexpr bool CP = is_complex<E>;
  __shared__ float sf[kSliceThreads / 32];
  __shared__ uint32_t su[kSliceThreads / 32];
  float ss = 0.f;
  uint32_t mb = 0, any = 0;
  for (int k = threadIdx.x; k < n; k += kSliceThreads) {
    if (k == skip) continue;
    const E e = v[k];
    const float fa = abs_f32(re_in(e), 0);
    ss = fmaf(fa, fa, ss);
    mb = max(mb, abs_hi(re_in(e)));
    any |= low_word(re_in(e));
    if constexpr (CP) {
      const float fb = abs_f32(im_in(e), 0);
      ss = fmaf(fb, fb, ss);
      mb = max(mb, abs_hi(im_in(e)));
      any |= low_word(im_in(e));
    }
  }
  // a magnitude whose high word is zero is still not zero
  if (mb == 0 && any != 0) mb = 1;
  reduce_block(ss, mb, sf, su);
  int off = 0;
  if ((mb < kSafeLo || mb >= kSafeHi) && mb >= (1u << 20) && mb < 0x7FF00000u) {
    // once more with the largest magnitude scaled to about one
    off = static_cast<int>(mb >> 20) - 1023;
    ss = 0.f;
    for (int k = threadIdx.x; k < n; k += kSliceThreads) {
      if (k == skip) continue;
      const E e = v[k];
      const float fa = abs_f32(re_in(e), off), fb = CP ? abs_f32(im_in(e), off) : 0.f;
      ss = fmaf(fa, fa, fmaf(fb, fb, ss));
    }
    uint32_t same = mb;
    reduce_block(ss, same, sf, su);
  }
  *nonzero = mb != 0;
  return scale_exponent(ss, mb, off, (CP ? 2.f : 1.f) * n, L);
}

// One vector of n entries (a column of X, or column r of the Hermitian H as
// row r conjugated) to its residues in planes [m0, m1): element k of plane
// (m - m0) goes to out[plane * stride + k].  skip: index left out (set to
// zero), -1 for none.  Integer and packed FP32 arithmetic only, two entries at
// a time; the norm that sets the scale is summed in FP32 from truncated bits,
// with a margin for what that loses.
template <int NM, int NL, class E>
__device__ __forceinline__ void slice_vector(const E* __restrict__ v, int n, bool conj, int skip,
                                             __nv_bfloat16* __restrict__ out, long long stride,
                                             int* __restrict__ exponent, const SliceTab& tab, int m0,
                                             int m1) {
  constexpr bool CP = is_complex<E>;
  bool nonzero;
  const int s = vector_exponent(v, n, skip, tab.log2_norm, &nonzero);
  if (threadIdx.x == 0) *exponent = s;
  const bool zero = s == kNonFinite;
  for (int k = 2 * threadIdx.x; k < n; k += 2 * kSliceThreads) {
    long long xr[2] = {}, xi[2] = {};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (k + h < n && k + h != skip && !zero) {
        const E e = v[k + h];
        xr[h] = scaled_int(re_in(e), s);
        if constexpr (CP) {
          xi[h] = scaled_int(im_in(e), s);
          if (conj) xi[h] = -xi[h];
        }
      }
    }
    // rows are padded to 64 entries, so the second of a pair is inside
    store_residues<NM, NL, CP>(xr, xi, out + k, stride, tab, m0, m1);
  }
}

// Row r of the Hermitian (symmetric) H from its column r, without the
// diagonal (the epilogue applies it in FP64: it is often far larger than the
// other entries, whose bits a scale set by it would waste).
template <int NM, int NL, class E>
__global__ void __launch_bounds__(kSliceThreads)
    rns_slice_h_kernel(const E* __restrict__ H, long long ldh, int N,
                       const __grid_constant__ SliceTab tab, int m0, int m1,
                       __nv_bfloat16* __restrict__ A, long long Kp, int* __restrict__ Ex,
                       double* __restrict__ Dg) {
  const int r = blockIdx.x;
  const E* col = H + static_cast<long long>(r) * ldh;
  if (threadIdx.x == 0) Dg[r] = re_of(col[r]);
  slice_vector<NM, NL, E>(col, N, true, r, A + r * Kp, static_cast<long long>(N) * Kp, Ex + r, tab,
                          m0, m1);
}

// Exponent of every row of the Hermitian H (from its column, without the
// diagonal), and the least and the largest over the rows that are not zero.
template <class E>
__device__ __forceinline__ void row_exponent(const E* __restrict__ H, long long ldh, int N, int r,
                                             float L, int* __restrict__ Ex,
                                             int* __restrict__ minmax) {
  bool nonzero;
  const int s = vector_exponent(H + r * ldh, N, r, L, &nonzero);
  if (threadIdx.x == 0) {
    Ex[r] = s;
    if (nonzero) {
      atomicMin(&minmax[0], s);
      atomicMax(&minmax[1], s);
    }
  }
}
template <class E>
__global__ void __launch_bounds__(kSliceThreads)
    rns_row_exponent_kernel(const E* __restrict__ H, long long ldh, int N, float L,
                            int* __restrict__ Ex, int* __restrict__ minmax) {
  row_exponent(H, ldh, N, blockIdx.x, L, Ex, minmax);
}

// One 64 x 64 tile of the lower triangle of a Hermitian H, scaled by 2^s, to
// one residue plane per modulus.  Complex: re + j im at (r, k) and, its
// conjugate's, re - j im at (k, r); the second plane of the modulus is the
// transpose of the first.  Real: the lower triangle, with the 256 x 256 blocks
// on the diagonal whole; products load the rest transposed.  Only the lower
// triangle is read, so the plane is exactly that of a Hermitian matrix
// whatever rounding left in H.
constexpr int kSymTile = 64;
constexpr int kSymSmem = 2 * kSymTile * (kSymTile + 1) * 8;
template <int NM, int NL, class E>
__device__ __forceinline__ void slice_sym_tile(const E* __restrict__ H, long long ldh, int N, int idx,
                                               int s, const SliceTab& tab, int m0, int m1,
                                               __nv_bfloat16* __restrict__ A, long long Kp,
                                               int* __restrict__ Ex, double* __restrict__ Dg) {
  constexpr bool CP = is_complex<E>;
  extern __shared__ long long sym_smem[];
  auto re_t = reinterpret_cast<long long (*)[kSymTile + 1]>(sym_smem);
  auto im_t = re_t + kSymTile;
  int R = static_cast<int>((sqrtf(8.f * idx + 1.f) - 1.f) * 0.5f);
  while ((R + 1) * (R + 2) / 2 <= idx) ++R;
  while (R * (R + 1) / 2 > idx) --R;
  const int K = idx - R * (R + 1) / 2, r0 = R * kSymTile, k0 = K * kSymTile;
  const bool diag = R == K;
  for (int e = threadIdx.x; e < kSymTile * kSymTile; e += kSliceThreads) {
    const int r = e % kSymTile, k = e / kSymTile;
    if (diag && r < k) continue;
    long long xr = 0, xi = 0;
    if (r0 + r < N && k0 + k < N) {
      const E v = H[(k0 + k) * ldh + r0 + r];
      if (diag && r == k) {
        Dg[r0 + r] = re_of(v);
        Ex[r0 + r] = s;
      } else {
        xr = scaled_int(re_in(v), s);
        if constexpr (CP) xi = scaled_int(im_in(v), s);
      }
    }
    re_t[r][k] = xr;
    if constexpr (CP) im_t[r][k] = xi;
    if (diag && r > k) {
      re_t[k][r] = xr;
      if constexpr (CP) im_t[k][r] = -xi;
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long plane = N * Kp;
  for (int q = warp; q < kSymTile; q += kSliceThreads / 32) {
    if (r0 + q < N) {
      const long long xr[2] = {re_t[q][2 * lane], re_t[q][2 * lane + 1]};
      long long xi[2] = {};
      if constexpr (CP) {
        xi[0] = im_t[q][2 * lane];
        xi[1] = im_t[q][2 * lane + 1];
      }
      store_residues<NM, NL, CP, false>(xr, xi, A + (r0 + q) * Kp + k0 + 2 * lane, plane, tab, m0,
                                        m1);
    }
    constexpr int kBlock = 2 * BM / kSymTile;
    if ((CP ? !diag : !diag && R / kBlock == K / kBlock) && k0 + q < N) {
      const long long xr[2] = {re_t[2 * lane][q], re_t[2 * lane + 1][q]};
      long long xi[2] = {};
      if constexpr (CP) {
        xi[0] = -im_t[2 * lane][q];
        xi[1] = -im_t[2 * lane + 1][q];
      }
      store_residues<NM, NL, CP, false>(xr, xi, A + (k0 + q) * Kp + r0 + 2 * lane, plane, tab, m0,
                                        m1);
    }
  }
}
template <int NM, int NL, class E>
__global__ void __launch_bounds__(kSliceThreads)
    rns_slice_sym_kernel(const E* __restrict__ H, long long ldh, int N, int s,
                         const __grid_constant__ SliceTab tab, int m0, int m1,
                         __nv_bfloat16* __restrict__ A, long long Kp, int* __restrict__ Ex,
                         double* __restrict__ Dg) {
  slice_sym_tile<NM, NL, E>(H, ldh, N, blockIdx.x, s, tab, m0, m1, A, Kp, Ex, Dg);
}

// Columns [j0, j0 + gridDim.x) of X.
template <int NM, int NL, class E>
__global__ void __launch_bounds__(kSliceThreads)
    rns_slice_x_kernel(const E* __restrict__ X, long long ldx, int N, int j0,
                       const __grid_constant__ SliceTab tab, __nv_bfloat16* __restrict__ B,
                       long long Kp, long long plane, int* __restrict__ Fx) {
  pdl_next();
  pdl_wait();
  const int c = blockIdx.x;
  slice_vector<NM, NL, E>(X + static_cast<long long>(j0 + c) * ldx, N, false, -1, B + c * Kp, plane,
                          Fx + c, tab, 0, NM);
}

// Rows of a column-major X (M x K) as vectors: row r of plane q goes to
// out[q * plane + r * Kp]. A block takes RB rows; reads are coalesced along
// the rows, and an RB x 64 tile of scaled integers in shared memory turns them
// into stores along K.  Bound by the 2 bytes per plane and entry it writes
// when there are rows for all SMs; with fewer, blocks of 8 rows instead of 32
// (M = K = 197: 33 -> 15 us; M = 1000, K = 70: 16 -> 7 us).
template <int RB, int NM, int NL, class E>
__global__ void __launch_bounds__(kSliceThreads)
    rns_slice_rows_kernel(const E* __restrict__ X, long long ldx, int M, int K,
                          const __grid_constant__ SliceTab tab, __nv_bfloat16* __restrict__ out,
                          long long Kp, long long plane, int* __restrict__ Ex) {
  constexpr bool CP = is_complex<E>;
  constexpr int W = CP ? 2 : 1;
  constexpr int G = kSliceThreads / RB;  // threads per row
  __shared__ float sf[G][RB];
  __shared__ uint32_t su[G][RB];
  __shared__ long long tile[W][RB][65];
  pdl_next();
  pdl_wait();
  const int row = threadIdx.x % RB, grp = threadIdx.x / RB;
  const int r0 = blockIdx.x * RB;
  const bool in = r0 + row < M;
  const E* x = X + r0 + row;
  float ss = 0.f;
  uint32_t mb = 0, any = 0;
  if (in)
    for (int k = grp; k < K; k += G) {
      const E e = x[k * ldx];
      const float fa = abs_f32(re_in(e), 0), fb = CP ? abs_f32(im_in(e), 0) : 0.f;
      ss = fmaf(fa, fa, fmaf(fb, fb, ss));
      mb = max(mb, max(abs_hi(re_in(e)), abs_hi(im_in(e))));
      any |= low_word(re_in(e)) | low_word(im_in(e));
    }
  if (mb == 0 && any != 0) mb = 1;
  auto reduce_rows = [&]() {
    __syncthreads();
    sf[grp][row] = ss;
    su[grp][row] = mb;
    __syncthreads();
    ss = 0.f;
    mb = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      ss += sf[g][row];
      mb = max(mb, su[g][row]);
    }
  };
  reduce_rows();
  int off = 0;
  const bool again = (mb < kSafeLo || mb >= kSafeHi) && mb >= (1u << 20) && mb < 0x7FF00000u;
  if (__syncthreads_or(again)) {
    const float before = ss;
    if (again) off = static_cast<int>(mb >> 20) - 1023;
    ss = 0.f;
    if (in && again)
      for (int k = grp; k < K; k += G) {
        const E e = x[k * ldx];
        const float fa = abs_f32(re_in(e), off), fb = CP ? abs_f32(im_in(e), off) : 0.f;
        ss = fmaf(fa, fa, fmaf(fb, fb, ss));
      }
    reduce_rows();
    if (!again) ss = before;
  }
  const int s = scale_exponent(ss, mb, off, (CP ? 2.f : 1.f) * K, tab.log2_norm);
  if (grp == 0 && in) Ex[r0 + row] = s;
  const bool zero = s == kNonFinite;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k0 = 0; k0 < K; k0 += 64) {
    __syncthreads();
    for (int kk = grp; kk < 64; kk += G) {
      long long a = 0, b = 0;
      if (in && k0 + kk < K && !zero) {
        const E e = x[(k0 + kk) * ldx];
        a = scaled_int(re_in(e), s);
        if constexpr (CP) b = scaled_int(im_in(e), s);
      }
      tile[0][row][kk] = a;
      if constexpr (CP) tile[W - 1][row][kk] = b;
    }
    __syncthreads();
    for (int q = warp; q < RB && r0 + q < M; q += kSliceThreads / 32) {
      long long xr[2], xi[2] = {};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        xr[h] = tile[0][q][2 * lane + h];
        if constexpr (CP) xi[h] = tile[W - 1][q][2 * lane + h];
      }
      store_residues<NM, NL, CP>(xr, xi, out + (r0 + q) * Kp + k0 + 2 * lane, plane, tab, 0, NM);
    }
  }
}

// ---------------------------------------------------------------------------
// Reconstruction and the recurrence's epilogue.  With q_i = (P / p_i)^-1 mod
// p_i, X / P = frac(sum_i x_i q_i / p_i): each residue times a fixed-point
// fraction of 80 bits (64 + 16), summed modulo one in integer registers.
// For complex planes (u = re + j im, w = re - j im) the fractions of re and
// im fold the 1/2 and 1/(2 j) in, so neither needs a modular reduction.
// ---------------------------------------------------------------------------
struct CrtMod {
  unsigned long long re_hi, im_hi;  // leading 64 bits
  unsigned re_lo, im_lo;            // next 16
};
struct CrtTab {
  CrtMod m[kRnsMaxModuli];
  double P, P_lo;  // 2^-64 times the product of the moduli, as the sum of two doubles
};

// X / P 2^64
__device__ __forceinline__ long long crt_fraction(unsigned long long hi, int lo) {
  return static_cast<long long>(hi +
                                static_cast<unsigned long long>(static_cast<long long>(lo >> 16)));
}
__device__ __forceinline__ double crt_value(unsigned long long hi, int lo) {
  return static_cast<double>(crt_fraction(hi, lo));
}
// v 2^e for v 2^e below overflow; 0 for 0 and where it would be denormal
__device__ __forceinline__ double scale_pow2(double v, int e) {
  const int h = __double2hiint(v);
  return ((h >> 20) & 0x7FF) + e > 0 && (h & 0x7FF00000) != 0
             ? __hiloint2double(h + e * (1 << 20), __double2loint(v))
             : 0.0;
}

template <class E>
struct Out;
template <>
struct Out<double2> {
  using S = double;
};
template <>
struct Out<float2> {
  using S = float;
};
template <>
struct Out<double> {
  using S = double;
};
template <>
struct Out<float> {
  using S = float;
};

// Two rows (r, r + 1) per thread, columns blockIdx.y, + gridDim.y, ...
//
// The FP64 pipe bounds this kernel (two FMAs a cycle and SM), so it does as
// little as the recurrence allows: one conversion and, per real component,
// T (alpha P 2^e) + (alpha (H_rr - shift)) x + beta y, with powers of two
// applied to exponent bits and every test on integers (about 19 FP64
// instructions a component before, 4 now).  With the slicing likewise moved off
// that pipe, a product with N = 4096 and 788 columns (11 moduli) takes 115 us
// less outside its GEMM (205 us before).
//
// With the FP64 moduli (ACC) the constants that every product of a filter
// shares, alpha P and alpha (H_rr - shift), carry a second part, 2^-53 of the
// first: their rounding would be the same in every degree step and so add up
// over the recurrence, where the roundings of an FP64 GEMM average out.  Its
// terms are formed in FP32 from truncated operands (24 bits of a 2^-53 part),
// and in FP64 where they leave FP32's range (FP64 filter N = 4096: 4420 -> 4346
// us, N = 1000: 932 -> 909 us, the errors against 64 bits as before).

// What two rows of a product share over its columns.
struct CrtRows {
  float df[2], dfl[2];  // single precision: alpha (H_rr - shift) as two floats
  float dl32[2];        // dl in FP32
  int er[2];
  double dh[2], dl[2];  // plain: alpha (H_rr - shift), else H_rr - shift (as two doubles)
  bool diag[2];
  bool f32[2];          // single precision: df is in FP32's range
};
__device__ __forceinline__ void crt_constants(CrtRows& k, int r0, int M, const int* __restrict__ Ex,
                                              const double* __restrict__ Dg, const RnsScale& sc) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool in = r0 + h < M;
    k.er[h] = in ? Ex[r0 + h] : 0;
    const double a = in && Dg ? Dg[r0 + h] : 0.0, b = -sc.shift;
    double d = a + b;
    const double t = d - a;
    double l = (a - (d - t)) + (b - t);
    k.diag[h] = d != 0.0;
    if (sc.plain) {
      const double p = sc.alpha * d;
      l = fma(sc.alpha, d, -p) + sc.alpha * l;
      d = p;
    }
    k.dh[h] = d;
    k.dl[h] = l;
    k.df[h] = static_cast<float>(d);
    k.dfl[h] = static_cast<float>(d - k.df[h]);
    // beyond 2^100 the low part, or its product, may leave FP32's range; left out
    // there, the constant is the rounded one
    k.f32[h] = abs_hi(d) < ((1023u + 100u) << 20);
    k.dl32[h] = k.f32[h] ? static_cast<float>(l) : 0.f;
  }
}

// v as FP32, truncated, by its bits, for |v| < 2^100; 0 below FP32's range
__device__ __forceinline__ float truncate_f32(double v) {
  return copysignf(abs_f32(v, 0), __int_as_float(__double2hiint(v)));
}
// v as a double, by its bits; 0 for a denormal
__device__ __forceinline__ double extend_f64(float v) {
  const int u = __float_as_int(v), m = u & 0x7FFFFFFF;
  const int h = (u & static_cast<int>(0x80000000u)) | ((m >> 3) + (896 << 20));
  return m >= (1 << 23) ? __hiloint2double(h, m << 29) : 0.0;
}

// v 2^e for a normal float whose result is one too; 0 where it would not be
__device__ __forceinline__ float scale_pow2f(float v, int e) {
  const int u = __float_as_int(v), x = ((u >> 23) & 0xFF) + e;
  return x > 0 && (u & 0x7F800000) != 0 ? __int_as_float(u + e * (1 << 23)) : 0.f;
}

// Rows r0, r0 + 1 of column j0 + c of the product: written to C and returned.
template <int NM, class E>
__device__ __forceinline__ void crt_pair(const CrtRows& k, int r0, int c,
                                         const int16_t* __restrict__ G, long long ldg,
                                         long long gplane, const CrtTab& tab,
                                         const int* __restrict__ Fx, int M, int j0,
                                         const E* __restrict__ X, long long ldx,
                                         E* __restrict__ C, long long ldc, const RnsScale& sc,
                                         E (&out)[2]) {
  constexpr bool CP = is_complex<E>;
  constexpr int W = CP ? 2 : 1;
  constexpr bool ACC = NM == kRnsFp64;
  using S = typename Out<E>::S;
  const int16_t* g = G + static_cast<long long>(c) * ldg + r0;
  unsigned long long hi[2][W] = {};
  int lo[2][W] = {};
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    const CrtMod& t = tab.m[m];
    if constexpr (CP) {
      const uint32_t u = *reinterpret_cast<const uint32_t*>(g + (2 * m) * gplane);
      const uint32_t w = *reinterpret_cast<const uint32_t*>(g + (2 * m + 1) * gplane);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int a = static_cast<int16_t>(u >> (16 * h)), b = static_cast<int16_t>(w >> (16 * h));
        const int s = a + b, d = a - b;
        hi[h][0] += static_cast<unsigned long long>(static_cast<long long>(s)) * t.re_hi;
        hi[h][1] += static_cast<unsigned long long>(static_cast<long long>(d)) * t.im_hi;
        lo[h][0] += s * static_cast<int>(t.re_lo);
        lo[h][1] += d * static_cast<int>(t.im_lo);
      }
    } else {
      const uint32_t u = *reinterpret_cast<const uint32_t*>(g + m * gplane);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int a = static_cast<int16_t>(u >> (16 * h));
        hi[h][0] += static_cast<unsigned long long>(static_cast<long long>(a)) * t.re_hi;
        lo[h][0] += a * static_cast<int>(t.re_lo);
      }
    }
  }
  const int fc = Fx[c];
  const long long jc = j0 + c;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = r0 + h;
    if (r >= M) break;
    const bool bad = k.er[h] == kNonFinite || fc == kNonFinite;
    const int e = bad ? 0 : -(k.er[h] + fc);
    E* cp = C + jc * ldc + r;
    const E x = k.diag[h] ? X[jc * ldx + r] : E{};
    const E y = sc.has_beta ? *cp : E{};
    double v[2];
    if constexpr (is_single<E>) {
      // results are stored in FP32: each constant as two floats, so what the
      // steps share is not rounded to one, and one FP32 FMA per term
      const int x0 = ((__float_as_int(sc.apf) >> 23) & 0xFF) + e;
      if (sc.single && k.f32[h] && !bad && x0 >= 27 && x0 <= 190) {
        const float f = scale_pow2f(sc.apf, e), fl = scale_pow2f(sc.apf_lo, e);
        float q[2] = {};
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const float T = static_cast<float>(crt_fraction(hi[h][w], lo[h][w]));
          const float xw = w == 0 ? re_in(x) : im_in(x), yw = w == 0 ? re_in(y) : im_in(y);
          float a = T * fl;
          if (sc.has_beta) a = fmaf(sc.bf_lo, yw, a);
          if (k.diag[h]) a = fmaf(k.dfl[h], xw, a);
          if (sc.has_beta) a = fmaf(sc.bf, yw, a);
          if (k.diag[h]) a = fmaf(k.df[h], xw, a);
          q[w] = fmaf(T, f, a);
        }
        if constexpr (CP)
          out[h] = E{q[0], q[1]};
        else
          out[h] = q[0];
        *cp = out[h];
        continue;
      }
    }
    if (sc.plain && !bad && e >= -800 && e <= 800) {
      const double f = scale_pow2(sc.ap, e), fl = ACC ? scale_pow2(sc.ap_lo, e) : 0.0;
      if constexpr (ACC) {
        // the low parts of the constants, 2^-53 of the others, in FP32, where
        // their terms are in its range
        const int xf = (__double2hiint(f) >> 20) & 0x7FF;
        uint32_t big = abs_hi(re_in(x));
        if constexpr (CP) big = max(big, abs_hi(im_in(x)));
        if (xf >= 1023 - 85 && xf <= 1023 + 60 && big < ((1023u + 60u) << 20)) {
          const float fl32 = truncate_f32(scale_pow2(sc.ap_lo, e + 32));
#pragma unroll
          for (int w = 0; w < W; ++w) {
            const long long t = crt_fraction(hi[h][w], lo[h][w]);
            const double xw = w == 0 ? re_of(x) : im_of(x), yw = w == 0 ? re_of(y) : im_of(y);
            float a = static_cast<float>(static_cast<int>(t >> 32)) * fl32;
            if (k.diag[h]) a = fmaf(k.dl32[h], truncate_f32(xw), a);
            double q = extend_f64(a);
            if (sc.has_beta) q = fma(sc.beta, yw, q);
            if (k.diag[h]) q = fma(k.dh[h], xw, q);
            v[w] = fma(static_cast<double>(t), f, q);
          }
          if constexpr (CP)
            out[h] = E{static_cast<S>(v[0]), static_cast<S>(v[1])};
          else
            out[h] = static_cast<S>(v[0]);
          *cp = out[h];
          continue;
        }
      }
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const double T = crt_value(hi[h][w], lo[h][w]);
        const double xw = w == 0 ? re_of(x) : im_of(x), yw = w == 0 ? re_of(y) : im_of(y);
        double q = 0.0;
        if (sc.has_beta) q = sc.beta * yw;
        if constexpr (ACC) q = fma(T, fl, q);
        if (k.diag[h]) {
          if constexpr (ACC) q = fma(k.dl[h], xw, q);
          q = fma(k.dh[h], xw, q);
        }
        v[w] = fma(T, f, q);
      }
    } else {  // scales that alpha P 2^e may not reach, non-finite operands
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const double T = crt_value(hi[h][w], lo[h][w]);
        const double xw = w == 0 ? re_of(x) : im_of(x), yw = w == 0 ? re_of(y) : im_of(y);
        double q = bad ? __longlong_as_double(0x7FF8000000000000ll)
                       : ldexp(ACC ? fma(T, tab.P, T * tab.P_lo) : T * tab.P, e);
        if (!sc.plain) q *= sc.alpha;
        else if (!bad) q = ldexp(ACC ? fma(T, sc.ap, T * sc.ap_lo) : T * sc.ap, e);
        if (k.diag[h]) {
          if constexpr (ACC) q = fma(sc.plain ? k.dl[h] : sc.alpha * k.dl[h], xw, q);
          q = fma(sc.plain ? k.dh[h] : sc.alpha * k.dh[h], xw, q);
        }
        v[w] = sc.has_beta ? fma(sc.beta, yw, q) : q;
      }
    }
    if constexpr (CP)
      out[h] = E{static_cast<S>(v[0]), static_cast<S>(v[1])};
    else
      out[h] = static_cast<S>(v[0]);
    *cp = out[h];
  }
}

template <int NM, class E>
__device__ __forceinline__ void crt_rows(int r0, int c0, int c1, int cstep,
                                         const int16_t* __restrict__ G, long long ldg,
                                         long long gplane, const CrtTab& tab,
                                         const int* __restrict__ Ex, const int* __restrict__ Fx,
                                         const double* __restrict__ Dg, int M, int j0,
                                         const E* __restrict__ X, long long ldx,
                                         E* __restrict__ C, long long ldc, const RnsScale& sc) {
  CrtRows k;
  crt_constants(k, r0, M, Ex, Dg, sc);
  E out[2];
  for (int c = c0; c < c1; c += cstep)
    crt_pair<NM, E>(k, r0, c, G, ldg, gplane, tab, Fx, M, j0, X, ldx, C, ldc, sc, out);
}

template <int NM, class E>
__global__ void __launch_bounds__(128)
    rns_crt_kernel(const int16_t* __restrict__ G, long long ldg, long long gplane,
                   const __grid_constant__ CrtTab tab, const int* __restrict__ Ex,
                   const int* __restrict__ Fx, const double* __restrict__ Dg, int M, int ncols,
                   int j0, const E* __restrict__ X, long long ldx, E* __restrict__ C, long long ldc,
                   const __grid_constant__ RnsScale sc) {
  pdl_wait();
  const int r0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (r0 < M)
    crt_rows<NM, E>(r0, blockIdx.y, ncols, gridDim.y, G, ldg, gplane, tab, Ex, Fx, Dg, M, j0, X,
                    ldx, C, ldc, sc);
  pdl_next();  // late, for the reason the GEMM gives
}

// Reconstruction of one degree step and slicing for the next in one kernel, for
// blocks whose columns a cluster holds in registers (two rows a thread, at
// most 8 x 256 threads): the columns from `next0` on, just computed, go straight
// to their residues.  Their norm needs the whole column, so the cluster's
// blocks exchange partial sums through shared memory; the sums add up in rank
// order, the same in every block.  Saves a launch and two reads of the column
// (filter N = 1000: 1139 -> 1039 us; complex64 N = 2000: 1722 -> 1623; split N =
// 2048: 1889 -> 1833; real N = 2501: 2515 -> 2348).  What the rows share over
// the columns is formed anew by every cluster, on the FP64 pipe: with complex N
// = 4096 that costs more than it saves (4541 -> 4649).
constexpr int kStepRows = 4096;                     // largest N, real
constexpr int kStepRowsComplex = kStepRows / 2;
template <int NM, int NL, class E>
__global__ void __launch_bounds__(256)
    rns_step_kernel(const int16_t* __restrict__ G, long long ldg, long long gplane,
                    const __grid_constant__ CrtTab tab, const int* __restrict__ Ex,
                    const int* __restrict__ Fx, const double* __restrict__ Dg, int M, int ncols,
                    int j0, const E* __restrict__ X, long long ldx, E* __restrict__ C, long long ldc,
                    const __grid_constant__ RnsScale sc, const __grid_constant__ SliceTab stab,
                    int next0, __nv_bfloat16* __restrict__ B, long long Kp, long long plane,
                    int* __restrict__ Fnext) {
  constexpr bool CP = is_complex<E>;
  __shared__ float wf[8];
  __shared__ uint32_t wu[8];
  // partial sums by cluster rank: [column parity][first pass, rescaled pass]
  __shared__ float cf[2][2][8];
  __shared__ uint32_t cu[2][2][8];
  uint32_t size;
  asm volatile("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(size));
  const uint32_t rank = cluster_rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int r0 = 2 * (rank * blockDim.x + threadIdx.x);
  CrtRows k;
  crt_constants(k, r0, M, Ex, Dg, sc);  // H's own, not of the kernel before
  cluster_sync();  // every block runs before another writes to it
  pdl_wait();
  // sum of ss and maximum of mb over the cluster
  auto reduce_cluster = [&](float& ss, uint32_t& mb, int par, int pass) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ss += __shfl_xor_sync(0xffffffffu, ss, o);
      mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    }
    __syncthreads();
    if (lane == 0) {
      wf[warp] = ss;
      wu[warp] = mb;
    }
    __syncthreads();
    ss = 0.f;
    mb = 0;
    for (int w = 0; w < nwarps; ++w) {
      ss += wf[w];
      mb = max(mb, wu[w]);
    }
    if (size > 1) {
      if (threadIdx.x < size) {
        asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(
                         map_to_rank(&cf[par][pass][rank], threadIdx.x)),
                     "f"(ss)
                     : "memory");
        asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(
                         map_to_rank(&cu[par][pass][rank], threadIdx.x)),
                     "r"(mb)
                     : "memory");
      }
      __syncwarp();
      cluster_sync();
      ss = 0.f;
      for (uint32_t q = 0; q < size; ++q) {
        ss += cf[par][pass][q];
        mb = max(mb, cu[par][pass][q]);
      }
    }
  };
  int par = 0;
  for (int c = blockIdx.x / size; c < ncols; c += gridDim.x / size) {
    E v[2] = {};
    if (r0 < M)
      crt_pair<NM, E>(k, r0, c, G, ldg, gplane, tab, Fx, M, j0, X, ldx, C, ldc, sc, v);
    const int nc = j0 + c - next0;
    if (nc < 0) continue;
    float ss = 0.f;
    uint32_t mb = 0, any = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float fa = abs_f32(re_in(v[h]), 0), fb = CP ? abs_f32(im_in(v[h]), 0) : 0.f;
      ss = fmaf(fa, fa, fmaf(fb, fb, ss));
      mb = max(mb, max(abs_hi(re_in(v[h])), abs_hi(im_in(v[h]))));
      any |= low_word(re_in(v[h])) | low_word(im_in(v[h]));
    }
    if (mb == 0 && any != 0) mb = 1;
    reduce_cluster(ss, mb, par, 0);
    int off = 0;
    if ((mb < kSafeLo || mb >= kSafeHi) && mb >= (1u << 20) && mb < 0x7FF00000u) {
      off = static_cast<int>(mb >> 20) - 1023;
      ss = 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float fa = abs_f32(re_in(v[h]), off), fb = CP ? abs_f32(im_in(v[h]), off) : 0.f;
        ss = fmaf(fa, fa, fmaf(fb, fb, ss));
      }
      uint32_t same = mb;
      reduce_cluster(ss, same, par, 1);
    }
    par ^= 1;
    const int s = scale_exponent(ss, mb, off, (CP ? 2.f : 1.f) * M, stab.log2_norm);
    if (rank == 0 && threadIdx.x == 0) Fnext[nc] = s;
    if (r0 < M) {
      const bool zero = s == kNonFinite;
      long long xr[2] = {}, xi[2] = {};
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (!zero) {
          xr[h] = scaled_int(re_in(v[h]), s);
          if constexpr (CP) xi[h] = scaled_int(im_in(v[h]), s);
        }
      store_residues<NM, NL, CP>(xr, xi, B + nc * Kp + r0, plane, stab, 0, NM);
    }
  }
  pdl_next();
  cluster_sync();  // no block leaves while another may still write to it
}

// ---------------------------------------------------------------------------
// Many problems per launch (the batched filter): one degree step slices the
// active columns of every problem, multiplies, and puts the products together
// in three launches.  A launch's work is listed in the step's entries; blocks
// find theirs by binary search, the persistent GEMM pairs by walking on from
// their last tile.
// ---------------------------------------------------------------------------
// Last entry whose prefix (a member of the entries) is not above g.
template <class S>
__device__ __forceinline__ int find_entry(const S* s, int n, int S::*prefix, int g) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (s[mid].*prefix <= g) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(kSliceThreads)
    rns_grouped_row_exponent_kernel(const GroupedSliceH* __restrict__ probs, int P, float L,
                                    int* __restrict__ minmax) {
  const int p = find_entry(probs, P, &GroupedSliceH::row0, blockIdx.x);
  const GroupedSliceH& q = probs[p];
  row_exponent(q.H, q.ldh, q.n, blockIdx.x - q.row0, L, q.E, minmax + 2 * p);
}
template <int NM, int NL>
__global__ void __launch_bounds__(kSliceThreads)
    rns_grouped_slice_sym_kernel(const GroupedSliceH* __restrict__ probs, int P,
                                 const __grid_constant__ SliceTab tab) {
  const GroupedSliceH& q = probs[find_entry(probs, P, &GroupedSliceH::tile0, blockIdx.x)];
  slice_sym_tile<NM, NL, double2>(q.H, q.ldh, q.n, blockIdx.x - q.tile0, q.s, tab, 0, NM,
                                  static_cast<__nv_bfloat16*>(q.A), q.Kp, q.E, q.Dg);
}
template <int NM, int NL>
__global__ void __launch_bounds__(kSliceThreads)
    rns_grouped_slice_h_kernel(const GroupedSliceH* __restrict__ probs, int P,
                               const __grid_constant__ SliceTab tab) {
  const GroupedSliceH& q = probs[find_entry(probs, P, &GroupedSliceH::row0, blockIdx.x)];
  const int r = blockIdx.x - q.row0;
  const double2* col = q.H + static_cast<long long>(r) * q.ldh;
  if (threadIdx.x == 0) q.Dg[r] = col[r].x;
  slice_vector<NM, NL, double2>(col, q.n, true, r, static_cast<__nv_bfloat16*>(q.A) + r * q.Kp,
                                q.n * q.Kp, q.E + r, tab, 0, NM);
}

template <int NM, int NL>
__global__ void __launch_bounds__(kSliceThreads)
    rns_grouped_slice_x_kernel(const GroupedProblem* __restrict__ probs,
                               const GroupedStep* __restrict__ steps, int nact, int parity,
                               const __grid_constant__ SliceTab tab) {
  const GroupedStep& st = steps[find_entry(steps, nact, &GroupedStep::col0, blockIdx.x)];
  const GroupedProblem& q = probs[st.prob];
  const int c = blockIdx.x - st.col0;
  const double2* x = (parity ? q.buf1 : q.buf0) + (st.s + c) * (parity ? q.ld1 : q.ld0);
  slice_vector<NM, NL, double2>(x, q.n, false, -1, static_cast<__nv_bfloat16*>(q.Bsl) + c * q.Kp,
                                q.bcap * q.Kp, q.F + c, tab, 0, NM);
}

// Tiles of a step: per problem the column tile runs fastest, then row tiles,
// then planes.
struct GroupedTiles {
  static constexpr bool kTri = false;
  const GroupedProblem* probs;
  const GroupedStep* steps;
  int bn, nact, at;  // at: entry of the last tile
  __device__ __forceinline__ void operator()(int t, Tile& T) {
    // the first tile's entry by binary search, then a walk forward
    if (at < 0) at = find_entry(steps, nact, &GroupedStep::tile0, t);
    while (steps[at + 1].tile0 <= t) ++at;
    const GroupedStep& st = steps[at];
    const GroupedProblem& q = probs[st.prob];
    const int rtiles = (q.n + 2 * BM - 1) / (2 * BM), ctiles = (q.b - st.s + bn - 1) / bn;
    const int u = t - st.tile0;
    const int ct = u % ctiles, rest = u / ctiles;
    const int rt = rest % rtiles, pl = rest / rtiles;
    T.mapA = q.mapA;
    T.mapB = q.mapB0 + (bn / 32 - 1);  // one map per tile width
    T.row0 = rt * 2 * BM;
    T.col0 = ct * bn;
    T.planeA = q.sym ? pl >> 1 : pl;
    T.planeB = pl;
    T.trans = q.sym && (pl & 1);
    T.modulus = pl / 2;
    T.nst = (q.n + BK - 1) / BK;
    T.M = q.n;
    T.ncols = q.b - st.s;
    T.ldg = q.Kp;
    T.G = static_cast<int16_t*>(q.G) + static_cast<long long>(pl) * q.bcap * q.Kp;
  }
};

template <int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    rns_grouped_gemm_kernel(const GroupedProblem* __restrict__ probs,
                            const GroupedStep* __restrict__ steps, int nact, int ntiles, int in_row,
                            const __grid_constant__ GemmTab tab, int* __restrict__ err) {
  GroupedTiles g{probs, steps, BN, nact, -1};
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int per = (ntiles + npairs - 1) / npairs;
  const Walk w = in_row ? Walk{min(pair * per, ntiles), min((pair + 1) * per, ntiles), 1}
                        : Walk{pair, ntiles, npairs};
  gemm_body<BN>(g, w, tab, 1, err);
}

// Columns per block of the grouped reconstruction: a block of a small problem has
// few rows, and one column after the other only lengthens its chain.
__host__ __device__ constexpr int crt_cols(int n) { return n <= 256 ? 1 : 4; }

template <int NM>
__global__ void __launch_bounds__(128)
    rns_grouped_crt_kernel(const GroupedProblem* __restrict__ probs,
                           const GroupedStep* __restrict__ steps, int nact, int parity,
                           const __grid_constant__ CrtTab tab) {
  const GroupedStep& st = steps[find_entry(steps, nact, &GroupedStep::blk0, blockIdx.x)];
  const GroupedProblem& q = probs[st.prob];
  const int rchunks = (q.n + 255) / 256, u = blockIdx.x - st.blk0;
  const int cols = crt_cols(q.n);
  const int r0 = 2 * (u % rchunks * 128 + threadIdx.x), c0 = u / rchunks * cols;
  if (r0 >= q.n) return;
  crt_rows<NM, double2>(r0, c0, min(c0 + cols, q.b - st.s), 1, static_cast<int16_t*>(q.G), q.Kp,
                        static_cast<long long>(q.bcap) * q.Kp, tab, q.E, q.F, q.Dg, q.n, st.s,
                        parity ? q.buf1 : q.buf0, parity ? q.ld1 : q.ld0,
                        parity ? q.buf0 : q.buf1, parity ? q.ld0 : q.ld1, st.sc);
}

// ---------------------------------------------------------------------------
// Host: tables
// ---------------------------------------------------------------------------
namespace {
int mod_inverse(int a, int p) {  // p <= 512: trial
  a %= p;
  for (int x = 1; x < p; ++x)
    if (a * x % p == 1) return x;
  return 0;
}
int centred(int v, int p) {
  v %= p;
  if (v < 0) v += p;
  return v > p / 2 ? v - p : v;
}
int root_of_minus_one(int p) {
  for (int j = 2; j < p; ++j)
    if ((j * j + 1) % p == 0) return j;
  return 0;
}

struct Tables {
  GemmTab gemm;
  SliceTab slice;
  CrtTab crt;
};

Tables make_tables(int nm, bool cplx) {
  Tables t{};
  double log2P = 0.0;
  for (int i = 0; i < nm; ++i) log2P += std::log2(static_cast<double>(kModuli[i]));
  // both norms below 2^L with 2^(2L) < P / 2; the slack covers the rounding
  // of the entries (at most sqrt(2 K) / 2 against 2^L) and of log2
  t.slice.log2_norm = static_cast<float>(0.5 * (log2P - 1.0) - 1.0 / 256);
  // P = hi + lo: hi the rounded product, lo what is left, exactly (P < 2^126)
  unsigned __int128 whole = 1;
  for (int i = 0; i < nm; ++i) whole *= static_cast<unsigned>(kModuli[i]);
  const double hi = static_cast<double>(whole);
  const unsigned __int128 hi_int = static_cast<unsigned __int128>(hi);
  const double lo = whole >= hi_int ? static_cast<double>(whole - hi_int)
                                    : -static_cast<double>(hi_int - whole);
  t.crt.P = std::ldexp(hi, -64);
  t.crt.P_lo = std::ldexp(lo, -64);
  for (int i = 0; i < nm; ++i) {
    // the FP32 quotient of reduce() may round a remainder near p / 2 to the
    // other side: |residue| <= (p + 1) / 2
    const int p = kModuli[i], h = (p + 1) / 2;
    t.gemm.m[i].p = static_cast<float>(p);
    t.gemm.m[i].invp = 1.0f / static_cast<float>(p);
    t.gemm.m[i].chunk = (1 << 24) / (h * h) / BK;  // K h^2 <= 2^24
    SliceMod& s = t.slice.m[i];
    auto twice = [](float v) {
      uint32_t u;
      std::memcpy(&u, &v, 4);
      return static_cast<unsigned long long>(u) << 32 | u;
    };
    s.mp = twice(-t.gemm.m[i].p);
    s.invp = twice(t.gemm.m[i].invp);
    const int j = root_of_minus_one(p);
    int pw = 1;
    for (int k = 0; k < 5; ++k) {
      s.c[k] = twice(static_cast<float>(centred(pw, p)));
      s.jc[k] = twice(static_cast<float>(centred(pw * j, p)));
      pw = pw * (1 << kLimbBits) % p;
    }
    int rest = 1;  // P / p_i mod p_i
    for (int o = 0; o < nm; ++o)
      if (o != i) rest = rest * (kModuli[o] % p) % p;
    const int q = mod_inverse(rest, p);
    const int tr = cplx ? mod_inverse(2, p) * q % p : q;
    const int ti = cplx ? mod_inverse(2 * j, p) * q % p : 0;
    auto fraction = [p](int x, unsigned long long* hi, unsigned* lo) {
      // floor(x 2^80 / p), x < p
      unsigned __int128 n = static_cast<unsigned __int128>(x) << 80;
      n /= static_cast<unsigned>(p);
      *hi = static_cast<unsigned long long>(n >> 16);
      *lo = static_cast<unsigned>(n & 0xffff);
    };
    fraction(tr, &t.crt.m[i].re_hi, &t.crt.m[i].re_lo);
    fraction(ti, &t.crt.m[i].im_hi, &t.crt.m[i].im_lo);
  }
  return t;
}

const Tables& tables(int nm, bool cplx) {
  // thread-safe one-time initialisation per configuration
  static const Tables t7c = make_tables(7, true), t8c = make_tables(8, true),
                      t11c = make_tables(11, true), t12c = make_tables(12, true), t14c = make_tables(14, true),
                      t7r = make_tables(7, false), t8r = make_tables(8, false),
                      t11r = make_tables(11, false), t12r = make_tables(12, false), t14r = make_tables(14, false);
  if (cplx) return nm == 7 ? t7c : nm == 8 ? t8c : nm == 11 ? t11c : nm == 12 ? t12c : t14c;
  return nm == 7 ? t7r : nm == 8 ? t8r : nm == 11 ? t11r : nm == 12 ? t12r : t14r;
}

RnsScale crt_scale(const CrtTab& t, double alpha, double beta, double shift) {
  RnsScale s{};
  s.alpha = alpha;
  s.beta = beta;
  s.shift = shift;
  s.ap = alpha * t.P;
  s.ap_lo = std::fma(alpha, t.P, -s.ap) + alpha * t.P_lo;
  s.plain = std::fabs(alpha) >= std::ldexp(1.0, -100) && std::fabs(alpha) <= std::ldexp(1.0, 100);
  s.has_beta = beta != 0.0;
  s.apf = static_cast<float>(s.ap);
  s.apf_lo = static_cast<float>(s.ap - s.apf);
  s.bf = static_cast<float>(beta);
  s.bf_lo = static_cast<float>(beta - s.bf);
  s.single = s.plain && std::fabs(s.ap) >= std::ldexp(1.0, -100) &&
             std::fabs(s.ap) <= std::ldexp(1.0, 100) && std::fabs(beta) <= std::ldexp(1.0, 100);
  return s;
}

// CTA pairs that fit the device at one time.
template <int BN>
int pairs_on_device() {
  static const int v = [] {
    using C = Cfg<BN>;
    if (cudaFuncSetAttribute(rns_gemm_kernel<BN, false>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(rns_gemm_kernel<BN, true>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = C::SMEM;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, rns_gemm_kernel<BN, false>, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return 0;
    }
    return n;
  }();
  return v;
}

struct GemmArgs {
  const void* A;
  int64_t K, M, Kp, a_planes;  // A: a_planes of M x Kp
  const void* B;
  int64_t b_rows, b_planes;  // B: b_planes of b_rows x Kp (plane stride), ncols rows used
  int ncols, nplanes, plane0, per_modulus;
  int swap_a = 0;  // 1: A conjugated (the two planes of a modulus change places)
  int sym = 0;     // 1: A has one plane per modulus, the other is its transpose; 2: A's
                   // planes are symmetric and hold the lower triangle
  int16_t* G;
  int64_t ldg, gplane;
  const GemmTab* tab;
};

template <int BN>
int launch_gemm(Dev& d, const GemmArgs& a) {
  using C = Cfg<BN>;
  const int pairs = pairs_on_device<BN>();
  if (pairs < 1) {
    set_error("residue GEMM: no CTA pair fits this device");
    return CHASE_CUDA_ERROR;
  }
  CUtensorMap tmA, tmB;
  CHASE_TRY(make_tmap_bf16_3d(&tmA, a.A, a.K, a.M, a.a_planes, a.Kp * 2, a.Kp * 2 * a.M, BK, 64, 1));
  CHASE_TRY(make_tmap_bf16_3d(&tmB, a.B, a.K, a.ncols, a.b_planes, a.Kp * 2, a.Kp * 2 * a.b_rows,
                              BK, BN / 2, 1));
  const int rt = static_cast<int>((a.M + 2 * BM - 1) / (2 * BM));
  const int ct = (a.ncols + BN - 1) / BN;
  const int64_t tiles = static_cast<int64_t>(rt) * ct * a.nplanes;
  const unsigned grid = 2 * static_cast<unsigned>(std::min<int64_t>(tiles, pairs));
  const auto kernel = a.sym == 2 ? rns_gemm_kernel<BN, true> : rns_gemm_kernel<BN, false>;
  CHASE_CUDA(launch_pdl(kernel, dim3(grid), dim3(kThreads), C::SMEM, d.st, tmA, tmB,
                        *a.tab, rt, ct, a.nplanes, a.plane0, a.per_modulus, a.swap_a, a.sym == 1 ? 1 : 0,
                        static_cast<int>((a.K + BK - 1) / BK), static_cast<int>(a.M), a.ncols, a.G,
                        a.ldg, a.gplane, d.err));
  note_launch();
  return CHASE_OK;
}

// A 64-wide K step of a pair streams 256 + BN operand rows and multiplies BN
// columns; narrow tiles are bound by the streaming.
double stage_cost(int bn) { return std::max(1.0 * bn, 0.5 * (256 + bn)); }

// Columns per tile: the width whose busiest pair (of the 76 that the 152 SMs
// make) has the least to do.
int choose_bn(int64_t M, int ncols, int nplanes) {
  const int64_t rt = (M + 2 * BM - 1) / (2 * BM);
  int best = 32;
  double best_cost = 0.0;
  for (int bn = 32; bn <= 256; bn += 32) {
    const int64_t tiles = rt * ((ncols + bn - 1) / bn) * nplanes;
    const int64_t per = (tiles + 75) / 76;
    const double cost = static_cast<double>(per) * stage_cost(bn);
    if (best_cost == 0.0 || cost < 0.995 * best_cost) {
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

int run_gemm(Dev& d, const GemmArgs& a) {
  switch (choose_bn(a.M, a.ncols, a.nplanes)) {
    case 32: return launch_gemm<32>(d, a);
    case 64: return launch_gemm<64>(d, a);
    case 96: return launch_gemm<96>(d, a);
    case 128: return launch_gemm<128>(d, a);
    case 160: return launch_gemm<160>(d, a);
    case 192: return launch_gemm<192>(d, a);
    case 224: return launch_gemm<224>(d, a);
    default: return launch_gemm<256>(d, a);
  }
}

bool same_scale(int lo, int hi) {
  return lo <= hi && hi != kNonFinite && static_cast<long long>(hi) - lo <= 1;
}

// Limbs of an operand scaled to 2^L: 13 bits each, the top one up to 14.
constexpr int limbs_of(int nm) { return nm <= 8 ? 3 : nm <= 12 ? 4 : 5; }

int sym_tiles(int64_t n) {
  const int64_t t = (n + kSymTile - 1) / kSymTile;
  return static_cast<int>(t * (t + 1) / 2);
}
template <int NM, class E>
int slice_h(Dev& d, const RnsH& h, int m0, int m1) {
  const SliceTab& tab = tables(NM, is_complex<E>).slice;
  if (h.sym) {
    auto kernel = rns_slice_sym_kernel<NM, limbs_of(NM), E>;
    static const cudaError_t ready = cudaFuncSetAttribute(
        kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSymSmem);
    CHASE_CUDA(ready);
    kernel<<<sym_tiles(h.N), kSliceThreads, kSymSmem, d.st>>>(
        static_cast<const E*>(h.src), h.lds, static_cast<int>(h.N), h.exponent, tab, m0, m1,
        static_cast<__nv_bfloat16*>(h.A), h.Kp, h.E, h.Dg);
    note_launch();
    CHASE_CUDA(cudaGetLastError());
    return CHASE_OK;
  }
  rns_slice_h_kernel<NM, limbs_of(NM), E><<<static_cast<unsigned>(h.N), kSliceThreads, 0, d.st>>>(
      static_cast<const E*>(h.src), h.lds, static_cast<int>(h.N), tab, m0, m1,
      static_cast<__nv_bfloat16*>(h.A), h.Kp, h.E, h.Dg);
  note_launch();
  CHASE_CUDA(cudaGetLastError());
  return CHASE_OK;
}
// Whether all rows of H want the same scale, give or take one bit, and which.
template <class E>
int row_scales(Dev& d, const E* H, int64_t ldh, RnsH& h) {
  int* mm = nullptr;
  CHASE_TRY(d.alloc(&mm, 2));
  int host[2] = {kNonFinite, -kNonFinite};
  CHASE_CUDA(cudaMemcpyAsync(mm, host, sizeof(host), cudaMemcpyHostToDevice, d.st));
  rns_row_exponent_kernel<E><<<static_cast<unsigned>(h.N), kSliceThreads, 0, d.st>>>(
      H, ldh, static_cast<int>(h.N), tables(h.nmod, true).slice.log2_norm, h.E, mm);
  note_launch();
  CHASE_CUDA(cudaGetLastError());
  CHASE_CUDA(cudaMemcpyAsync(host, mm, sizeof(host), cudaMemcpyDeviceToHost, d.st));
  CHASE_TRY(d.sync_check("residues of H"));
  d.release(mm);
  h.sym = same_scale(host[0], host[1]);
  h.exponent = host[0];
  return CHASE_OK;
}
template <class E>
int slice_h_any(Dev& d, const RnsH& h, int m0, int m1) {
  if (h.nmod == 7) return slice_h<7, E>(d, h, m0, m1);
  if (h.nmod == 8) return slice_h<8, E>(d, h, m0, m1);
  if constexpr (!is_single<E>) {  // single precision takes the low sets
    if (h.nmod == 11) return slice_h<11, E>(d, h, m0, m1);
    if (h.nmod == 12) return slice_h<12, E>(d, h, m0, m1);
    if (h.nmod == kRnsFp64) return slice_h<kRnsFp64, E>(d, h, m0, m1);
  }
  set_error("residue planes: %d moduli", h.nmod);
  return CHASE_INVALID_ARG;
}
int slice_h_moduli(Dev& d, const RnsH& h, int m0, int m1) {
  switch (h.src_kind) {
    case 0: return slice_h_any<double2>(d, h, m0, m1);
    case 1: return slice_h_any<double>(d, h, m0, m1);
    case 2: return slice_h_any<float2>(d, h, m0, m1);
    default: return slice_h_any<float>(d, h, m0, m1);
  }
}

template <int NM, class E>
int product(Dev& d, const RnsH& h, RnsX& x, const E* X, int64_t ldx, int j0, int j1, E* C,
            int64_t ldc, double alpha, double beta, double shift, bool sliced, int next0) {
  constexpr bool CP = is_complex<E>;
  constexpr int PP = CP ? 2 : 1;  // planes per modulus
  const Tables& t = tables(NM, CP);
  const int N = static_cast<int>(h.N);
  if (NM * PP > x.planes || (CP ? 1 : 0) != h.cplx || x.Kp != h.Kp) {
    set_error("residue product: workspace of another kind");
    return CHASE_INVALID_ARG;
  }
  const int64_t bplane = static_cast<int64_t>(x.cap_cols) * x.Kp;
  const int64_t gplane = static_cast<int64_t>(x.cap_cols) * x.ldg;
  for (int c0 = j0; c0 < j1; c0 += x.cap_cols) {
    const int w = std::min(x.cap_cols, j1 - c0);
    int* F = x.F + (x.flip ? x.cap_cols : 0);
    if (!sliced) {
      CHASE_CUDA(launch_pdl(rns_slice_x_kernel<NM, limbs_of(NM), E>, dim3(w), dim3(kSliceThreads),
                            0, d.st, X, ldx, N, c0, t.slice, static_cast<__nv_bfloat16*>(x.B), x.Kp,
                            bplane, F));
      note_launch();
    }
    const double alg = (CP ? 8.0 : 2.0) * N * static_cast<double>(N) * w;
    KernelTimer kt(d.st, NM == kRnsFp64 ? CHASE_TIMED_FP64_PRODUCT : CHASE_TIMED_SPLIT_PRODUCT);
    int launched = 0;
    for (int m0 = 0; m0 < NM; m0 += h.resident) {
      const int m1 = std::min(NM, m0 + h.resident);
      if (h.resident < NM) CHASE_TRY(slice_h_moduli(d, h, m0, m1));
      GemmArgs a;
      a.A = h.A;
      a.K = N;
      a.M = N;
      a.Kp = h.Kp;
      a.a_planes = static_cast<int64_t>(h.resident) * (h.sym ? 1 : PP);
      a.sym = h.sym ? (CP ? 1 : 2) : 0;
      a.B = x.B;
      a.b_rows = x.cap_cols;
      a.b_planes = NM * PP;
      a.ncols = w;
      a.nplanes = (m1 - m0) * PP;
      a.plane0 = m0 * PP;
      a.per_modulus = PP;
      a.G = x.G;
      a.ldg = x.ldg;
      a.gplane = gplane;
      a.tab = &t.gemm;
      CHASE_TRY(run_gemm(d, a));
      ++launched;
    }
    // NM moduli x PP planes of 2 N^2 b BF16 FLOPs
    kt.end(launched, alg, alg * NM * PP * 2.0 / (CP ? 8.0 : 2.0));
    if (next0 >= 0) {
      // two rows a thread; as many blocks as keep the SMs busy, a cluster per column
      const int threads = N <= kStepRows / 2 ? 128 : 256;
      const unsigned size = static_cast<unsigned>((N + 2 * threads - 1) / (2 * threads));
      const unsigned clusters = std::min(static_cast<unsigned>(w), 152u * 8u / size);
      CHASE_CUDA(launch_pdl_cluster(rns_step_kernel<NM, limbs_of(NM), E>, size,
                                    dim3(size * clusters), dim3(threads), 0, d.st, x.G, x.ldg,
                                    gplane, t.crt, h.E, F, h.Dg, N, w, c0, X, ldx, C, ldc,
                                    crt_scale(t.crt, alpha, beta, shift), t.slice, next0,
                                    static_cast<__nv_bfloat16*>(x.B), x.Kp, bplane,
                                    x.F + (x.flip ? 0 : x.cap_cols)));
      note_launch();
      x.flip ^= 1;
      continue;
    }
    // about 16 blocks of 128 threads per SM
    const int gx = (N + 255) / 256;
    const dim3 grid(static_cast<unsigned>(gx),
                    static_cast<unsigned>(std::min(w, std::max(1, 16 * 152 / gx))));
    CHASE_CUDA(launch_pdl(rns_crt_kernel<NM, E>, grid, dim3(128), 0, d.st, x.G, x.ldg, gplane,
                          t.crt, h.E, F, h.Dg, N, w, c0, X, ldx, C, ldc,
                          crt_scale(t.crt, alpha, beta, shift)));
    note_launch();
  }
  return CHASE_OK;
}

template <class E>
int product_any(Dev& d, const RnsH& h, RnsX& x, const E* X, int64_t ldx, int j0, int j1, E* C,
                int64_t ldc, double alpha, double beta, double shift, bool sliced, int next0) {
  if (j1 <= j0) return CHASE_OK;
  if (h.nmod == 7) return product<7>(d, h, x, X, ldx, j0, j1, C, ldc, alpha, beta, shift, sliced,
                      next0);
  if (h.nmod == 8) return product<8>(d, h, x, X, ldx, j0, j1, C, ldc, alpha, beta, shift, sliced,
                      next0);
  if constexpr (!is_single<E>) {
    if (h.nmod == 11)
      return product<11>(d, h, x, X, ldx, j0, j1, C, ldc, alpha, beta, shift, sliced,
                      next0);
    if (h.nmod == 12)
      return product<12>(d, h, x, X, ldx, j0, j1, C, ldc, alpha, beta, shift, sliced,
                      next0);
    if (h.nmod == kRnsFp64)
      return product<kRnsFp64>(d, h, x, X, ldx, j0, j1, C, ldc, alpha, beta, shift, sliced,
                      next0);
  }
  set_error("residue product: %d moduli", h.nmod);
  return CHASE_INVALID_ARG;
}

template <class E>
int slice_columns(Dev& d, const E* X, int64_t ldx, RnsBlock& b) {
  CHASE_CUDA(launch_pdl(rns_slice_x_kernel<kRnsFp64, limbs_of(kRnsFp64), E>,
                        dim3(static_cast<unsigned>(b.n)), dim3(kSliceThreads), 0, d.st, X, ldx,
                        static_cast<int>(b.K), 0, tables(kRnsFp64, is_complex<E>).slice,
                        static_cast<__nv_bfloat16*>(b.P), b.Kp, b.n * b.Kp, b.E));
  note_launch();
  return CHASE_OK;
}
template <int RB, class E>
int slice_rows_by(Dev& d, const E* X, int64_t ldx, RnsBlock& b) {
  CHASE_CUDA(launch_pdl(rns_slice_rows_kernel<RB, kRnsFp64, limbs_of(kRnsFp64), E>,
                        dim3(static_cast<unsigned>((b.n + RB - 1) / RB)), dim3(kSliceThreads), 0,
                        d.st, X, ldx, static_cast<int>(b.n), static_cast<int>(b.K),
                        tables(kRnsFp64, is_complex<E>).slice, static_cast<__nv_bfloat16*>(b.P),
                        b.Kp, b.n * b.Kp, b.E));
  note_launch();
  return CHASE_OK;
}
template <class E>
int slice_rows(Dev& d, const E* X, int64_t ldx, RnsBlock& b) {
  return b.n < 32 * 152 ? slice_rows_by<8>(d, X, ldx, b) : slice_rows_by<32>(d, X, ldx, b);
}
template <class E>
int dense(Dev& d, const RnsBlock& a, bool conj_a, const RnsBlock& b, E* C, int64_t ldc,
          double alpha, double beta) {
  constexpr bool CP = is_complex<E>;
  constexpr int PP = CP ? 2 : 1;
  const Tables& t = tables(kRnsFp64, CP);
  const int64_t ldg = (a.n + 7) / 8 * 8, gplane = ldg * b.n;
  int16_t* G = nullptr;
  CHASE_TRY(d.alloc(&G, static_cast<size_t>(gplane) * kRnsFp64 * PP));
  GemmArgs g;
  g.A = a.P;
  g.K = a.K;
  g.M = a.n;
  g.Kp = a.Kp;
  g.a_planes = kRnsFp64 * PP;
  g.B = b.P;
  g.b_rows = b.n;
  g.b_planes = kRnsFp64 * PP;
  g.ncols = static_cast<int>(b.n);
  g.nplanes = kRnsFp64 * PP;
  g.plane0 = 0;
  g.per_modulus = PP;
  g.swap_a = CP && conj_a ? 1 : 0;
  g.G = G;
  g.ldg = ldg;
  g.gplane = gplane;
  g.tab = &t.gemm;
  CHASE_TRY(run_gemm(d, g));
  const int gx = static_cast<int>((a.n + 255) / 256);
  const dim3 grid(static_cast<unsigned>(gx),
                  static_cast<unsigned>(std::min<int64_t>(b.n, std::max(1, 16 * 152 / gx))));
  CHASE_CUDA(launch_pdl(rns_crt_kernel<kRnsFp64, E>, grid, dim3(128), 0, d.st, G, ldg, gplane,
                        t.crt, a.E, b.E, nullptr, static_cast<int>(a.n), static_cast<int>(b.n), 0,
                        nullptr, 0, C, ldc, crt_scale(t.crt, alpha, beta, 0.0)));
  note_launch();
  d.release(G);
  return CHASE_OK;
}

template <int BN>
int grouped_pairs() {
  static const int v = [] {
    using C = Cfg<BN>;
    if (cudaFuncSetAttribute(rns_grouped_gemm_kernel<BN>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return pairs_on_device<BN>();
  }();
  return v;
}
template <int BN>
int launch_grouped_gemm(Dev& d, const GroupedProblem* probs, const GroupedStep* steps, int nact,
                        int ntiles, bool in_row, const GemmTab& tab) {
  const int pairs = grouped_pairs<BN>();
  if (pairs < 1) {
    set_error("residue GEMM: no CTA pair fits this device");
    return CHASE_CUDA_ERROR;
  }
  rns_grouped_gemm_kernel<BN><<<2 * std::min(ntiles, pairs), kThreads, Cfg<BN>::SMEM, d.st>>>(
      probs, steps, nact, ntiles, in_row ? 1 : 0, tab, d.err);
  note_launch();
  CHASE_CUDA(cudaGetLastError());
  return CHASE_OK;
}

// One of the three moduli counts of the batched filter.
template <class F>
int with_moduli(int nmod, F&& f) {
  switch (nmod) {
    case 11: return f(std::integral_constant<int, 11>());
    case 12: return f(std::integral_constant<int, 12>());
    case kRnsFp64: return f(std::integral_constant<int, kRnsFp64>());
  }
  set_error("grouped residue product: %d moduli", nmod);
  return CHASE_INVALID_ARG;
}
}  // namespace
}  // namespace rns

namespace {
template <class T>
struct Kind;
template <>
struct Kind<chase_c64> {
  static constexpr int k = 0;
  using D = double2;
};
template <>
struct Kind<double> {
  static constexpr int k = 1;
  using D = double;
};
template <>
struct Kind<chase_c32> {
  static constexpr int k = 2;
  using D = float2;
};
template <>
struct Kind<float> {
  static constexpr int k = 3;
  using D = float;
};
}  // namespace

// The rounding of the operands, relative to a product, grows like sqrt(N); the
// splits into 7-bit digits that these stand for had errors independent of N, but
// with a bias that added up over a filter's steps.  Degree 20: 4.4e-12 at N =
// 20000 (digits 6.5e-12), 4.8e-12 at N = 30000 (7.9e-12), uniform spectrum
// 3.8e-12 at both (3.5e-12, 4.5e-12).  Degree 2, uniform, sums of K = 2 N: 4.3e-13
// at N = 8192 (5.0e-13), 5.9e-13 at 16384 (3.6e-13), 8.3e-13 at 30000 (4.7e-13).
// One modulus more, a sixteenth of the error, takes over where they would meet,
// and for few steps of long sums before that.
int rns_split_moduli(int64_t N, bool cplx, int least_degree) {
  return N > 32768 || ((cplx ? 2 : 1) * N > 16384 && least_degree < 8) ? 12 : 11;
}
int rns_low_moduli(int64_t N) { return N <= 8192 ? 7 : 8; }

// One plane per modulus instead of two (real: one triangle of it) halves what a
// product streams, once the planes outgrow about half of the L2; below, the pass over H that looks for a
// common scale costs more (filter N = 1000, 57 MB: 1150 us with two planes,
// 1170 with one; complex64 N = 2000, 115 MB: 1876 and 1722; split N = 2048, 185
// MB: 2167 and 1889; N = 4096, 940 MB: 5210 and 4541; real N = 2501, 179 MB:
// 2362 and 2232).
bool rns_sym_pays(int planes, double entries) { return 2.0 * planes * entries > 64e6; }

namespace rns {
namespace {
// From here on (bytes of planes) the driver is asked what is free, about 3 us,
// so that the planes leave `reserve`; below, only an allocation that fails makes
// fewer moduli resident.
constexpr size_t kLargePlanes = size_t(1) << 25;

template <class T>
int prepare_h(Dev& d, const T* H, int64_t N, int64_t ldh, int nmod, int most, size_t reserve,
              bool many, RnsH& out) {
  out.N = N;
  out.Kp = (N + BK - 1) / BK * BK;
  out.src_kind = Kind<T>::k;
  out.cplx = out.src_kind % 2 == 0 ? 1 : 0;
  out.nmod = nmod;
  out.src = H;
  out.lds = ldh;
  CHASE_TRY(d.alloc(&out.E, static_cast<size_t>(N)));
  CHASE_TRY(d.alloc(&out.Dg, static_cast<size_t>(N)));
  if (many && rns_sym_pays(out.cplx ? 2 * nmod : nmod, static_cast<double>(N) * out.Kp))
    CHASE_TRY(row_scales(d, reinterpret_cast<const typename Kind<T>::D*>(H), ldh, out));
  const size_t per = static_cast<size_t>(out.cplx && !out.sym ? 2 : 1) * N * out.Kp * 2;  // bytes per modulus
  // all moduli resident where the memory allows it; else fewer, sliced anew
  // for every product
  out.resident = std::min(nmod, std::max(most, 1));
  if (per * nmod > kLargePlanes || d.limit != std::numeric_limits<size_t>::max()) {
    size_t free_b = 0;
    CHASE_TRY(d.free_bytes(&free_b));
    while (out.resident > 1 && per * out.resident + reserve > free_b) out.resident /= 2;
    if (per * out.resident + reserve > free_b) {
      set_error("residue planes of H: %zu bytes a modulus do not fit the memory", per);
      return CHASE_OUT_OF_MEMORY;
    }
  }
  int st = CHASE_OUT_OF_MEMORY;
  for (; out.resident >= 1; out.resident /= 2) {
    st = d.alloc_bytes(&out.A, per * out.resident);
    if (st != CHASE_OUT_OF_MEMORY) break;
  }
  CHASE_TRY(st);
  return out.resident == nmod ? slice_h_moduli(d, out, 0, nmod) : CHASE_OK;
}
}  // namespace
}  // namespace rns

void rns_release(Dev& d, RnsH& h) {
  for (void* p : {h.A, static_cast<void*>(h.E), static_cast<void*>(h.Dg)})
    if (p) d.release(p);
  h = RnsH{};
}
void rns_release(Dev& d, RnsX& x) {
  for (void* p : {x.B, static_cast<void*>(x.G), static_cast<void*>(x.F)})
    if (p) d.release(p);
  x = RnsX{};
}

template <class T>
int rns_prepare_h(Dev& d, const T* H, int64_t N, int64_t ldh, int nmod, int most, size_t reserve,
                  bool many, RnsH& out) {
  const int st = rns::prepare_h(d, H, N, ldh, nmod, most, reserve, many, out);
  if (st == CHASE_OUT_OF_MEMORY) rns_release(d, out);
  return st;
}

int rns_alloc_x(Dev& d, int64_t N, int max_cols, int max_moduli, bool cplx, RnsX& out) {
  out.planes = max_moduli * (cplx ? 2 : 1);
  out.Kp = (N + rns::BK - 1) / rns::BK * rns::BK;
  out.ldg = out.Kp;
  // fewer columns at a time where the memory does not hold them all
  int st = CHASE_OUT_OF_MEMORY;
  for (out.cap_cols = std::max(max_cols, 1);; out.cap_cols = (out.cap_cols + 1) / 2) {
    const size_t bytes = static_cast<size_t>(out.planes) * out.cap_cols * out.Kp * 2;
    st = d.alloc_bytes(&out.B, bytes);
    if (st == CHASE_OK) {
      void* g = nullptr;
      st = d.alloc_bytes(&g, bytes);
      out.G = static_cast<int16_t*>(g);
      if (st != CHASE_OK) {
        d.release(out.B);
        out.B = nullptr;
      }
    }
    if (st != CHASE_OUT_OF_MEMORY || out.cap_cols == 1) break;
  }
  if (st == CHASE_OK) st = d.alloc(&out.F, 2 * static_cast<size_t>(out.cap_cols));
  if (st == CHASE_OUT_OF_MEMORY) rns_release(d, out);
  return st;
}

bool rns_chains(const RnsH& h, int b, const RnsX& x) {
  return h.N <= (h.cplx ? rns::kStepRowsComplex : rns::kStepRows) && b <= x.cap_cols;
}

template <class T>
int rns_product(Dev& d, const RnsH& h, RnsX& x, const T* X, int64_t ldx, int j0, int j1, T* C,
                int64_t ldc, double alpha, double beta, double shift, bool sliced, int next0) {
  using D = typename Kind<T>::D;
  return rns::product_any<D>(d, h, x, reinterpret_cast<const D*>(X), ldx, j0, j1,
                             reinterpret_cast<D*>(C), ldc, alpha, beta, shift, sliced, next0);
}

namespace {
template <class T>
int alloc_block(Dev& d, int64_t n, int64_t K, RnsBlock& out) {
  out.n = n;
  out.K = K;
  out.Kp = (K + rns::BK - 1) / rns::BK * rns::BK;
  const size_t planes = kRnsFp64 * (rns::is_complex<typename Kind<T>::D> ? 2 : 1);
  CHASE_TRY(d.alloc_bytes(&out.P, planes * n * out.Kp * 2));
  const int st = d.alloc(&out.E, static_cast<size_t>(n));
  if (st != CHASE_OK) rns_release(d, out);
  return st;
}
}  // namespace

template <class T>
int rns_columns(Dev& d, const T* X, int64_t ldx, int64_t K, int n, RnsBlock& out) {
  using D = typename Kind<T>::D;
  CHASE_TRY(alloc_block<T>(d, n, K, out));
  return rns::slice_columns<D>(d, reinterpret_cast<const D*>(X), ldx, out);
}

template <class T>
int rns_rows(Dev& d, const T* X, int64_t ldx, int64_t M, int K, RnsBlock& out) {
  using D = typename Kind<T>::D;
  CHASE_TRY(alloc_block<T>(d, M, K, out));
  return rns::slice_rows<D>(d, reinterpret_cast<const D*>(X), ldx, out);
}

void rns_release(Dev& d, RnsBlock& b) {
  if (b.P) d.release(b.P);
  if (b.E) d.release(b.E);
  b = RnsBlock{};
}

template <class T>
int rns_dense(Dev& d, const RnsBlock& a, bool conj_a, const RnsBlock& b, T* C, int64_t ldc,
              double alpha, double beta) {
  using D = typename Kind<T>::D;
  return rns::dense<D>(d, a, conj_a, b, reinterpret_cast<D*>(C), ldc, alpha, beta);
}

#define CHASE_INSTANTIATE_DENSE(T)                                                                 \
  template int rns_columns<T>(Dev&, const T*, int64_t, int64_t, int, RnsBlock&);                   \
  template int rns_rows<T>(Dev&, const T*, int64_t, int64_t, int, RnsBlock&);                      \
  template int rns_dense<T>(Dev&, const RnsBlock&, bool, const RnsBlock&, T*, int64_t, double,     \
                            double);
CHASE_INSTANTIATE_DENSE(chase_c64)
CHASE_INSTANTIATE_DENSE(double)
#undef CHASE_INSTANTIATE_DENSE

int64_t rns_k_padded(int64_t N) { return (N + rns::BK - 1) / rns::BK * rns::BK; }

RnsScale rns_scale(int nmod, double alpha, double beta, double shift) {
  return rns::crt_scale(rns::tables(nmod, true).crt, alpha, beta, shift);
}

int rns_grouped_row_exponents(Dev& d, int nmod, const GroupedSliceH* probs, int P, int total_rows,
                              int* minmax) {
  rns::rns_grouped_row_exponent_kernel<<<static_cast<unsigned>(total_rows), rns::kSliceThreads, 0,
                                         d.st>>>(
      probs, P, rns::tables(nmod, true).slice.log2_norm, minmax);
  note_launch();
  CHASE_CUDA(cudaGetLastError());
  return CHASE_OK;
}
bool rns_same_scale(int lo, int hi) { return rns::same_scale(lo, hi); }
int rns_sym_tiles(int64_t n) { return rns::sym_tiles(n); }

int rns_grouped_prepare_h(Dev& d, int nmod, const GroupedSliceH* probs, int P, int total_rows) {
  return rns::with_moduli(nmod, [&](auto nm) -> int {
    constexpr int NM = decltype(nm)::value;
    rns::rns_grouped_slice_h_kernel<NM, rns::limbs_of(NM)>
        <<<static_cast<unsigned>(total_rows), rns::kSliceThreads, 0, d.st>>>(
            probs, P, rns::tables(NM, true).slice);
    note_launch();
    CHASE_CUDA(cudaGetLastError());
    return CHASE_OK;
  });
}
int rns_grouped_prepare_sym(Dev& d, int nmod, const GroupedSliceH* probs, int P, int total_tiles) {
  return rns::with_moduli(nmod, [&](auto nm) -> int {
    constexpr int NM = decltype(nm)::value;
    auto kernel = rns::rns_grouped_slice_sym_kernel<NM, rns::limbs_of(NM)>;
    static const cudaError_t ready = cudaFuncSetAttribute(
        kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, rns::kSymSmem);
    CHASE_CUDA(ready);
    kernel<<<static_cast<unsigned>(total_tiles), rns::kSliceThreads, rns::kSymSmem, d.st>>>(
        probs, P, rns::tables(NM, true).slice);
    note_launch();
    CHASE_CUDA(cudaGetLastError());
    return CHASE_OK;
  });
}

int rns_grouped_maps(CUtensorMap* mapA, CUtensorMap* mapB, int nmod, int bn, bool sym, const void* A,
                     const void* B, int64_t n, int64_t b, int64_t bcap) {
  const int64_t Kp = rns_k_padded(n);
  CHASE_TRY(make_tmap_bf16_3d(mapA, A, n, n, sym ? nmod : 2 * nmod, Kp * 2, Kp * 2 * n, rns::BK, 64, 1));
  return make_tmap_bf16_3d(mapB, B, n, b, 2 * nmod, Kp * 2, Kp * 2 * bcap, rns::BK, bn / 2, 1);
}

int rns_grouped_tiles(int nmod, int bn, int n, int cols) {
  return (n + 2 * rns::BM - 1) / (2 * rns::BM) * ((cols + bn - 1) / bn) * 2 * nmod;
}
int rns_grouped_crt_blocks(int n, int cols) {
  return (n + 255) / 256 * ((cols + rns::crt_cols(n) - 1) / rns::crt_cols(n));
}
double rns_stage_cost(int bn) { return rns::stage_cost(bn); }

int rns_grouped_slice_x(Dev& d, int nmod, const GroupedProblem* probs, const GroupedStep* steps,
                        int nact, int ncols, int parity) {
  return rns::with_moduli(nmod, [&](auto nm) -> int {
    constexpr int NM = decltype(nm)::value;
    rns::rns_grouped_slice_x_kernel<NM, rns::limbs_of(NM)>
        <<<static_cast<unsigned>(ncols), rns::kSliceThreads, 0, d.st>>>(
            probs, steps, nact, parity, rns::tables(NM, true).slice);
    note_launch();
    CHASE_CUDA(cudaGetLastError());
    return CHASE_OK;
  });
}
int rns_grouped_gemm(Dev& d, int nmod, int bn, const GroupedProblem* probs,
                     const GroupedStep* steps, int nact, int ntiles, bool in_row) {
  const rns::GemmTab& tab = rns::tables(nmod, true).gemm;
  switch (bn) {
    case 32: return rns::launch_grouped_gemm<32>(d, probs, steps, nact, ntiles, in_row, tab);
    case 64: return rns::launch_grouped_gemm<64>(d, probs, steps, nact, ntiles, in_row, tab);
    case 96: return rns::launch_grouped_gemm<96>(d, probs, steps, nact, ntiles, in_row, tab);
    case 128: return rns::launch_grouped_gemm<128>(d, probs, steps, nact, ntiles, in_row, tab);
    case 160: return rns::launch_grouped_gemm<160>(d, probs, steps, nact, ntiles, in_row, tab);
    case 192: return rns::launch_grouped_gemm<192>(d, probs, steps, nact, ntiles, in_row, tab);
    case 224: return rns::launch_grouped_gemm<224>(d, probs, steps, nact, ntiles, in_row, tab);
    default: return rns::launch_grouped_gemm<256>(d, probs, steps, nact, ntiles, in_row, tab);
  }
}
int rns_grouped_ready() {
  return rns::grouped_pairs<32>() > 0 && rns::grouped_pairs<64>() > 0 &&
                 rns::grouped_pairs<96>() > 0 && rns::grouped_pairs<128>() > 0 &&
                 rns::grouped_pairs<160>() > 0 && rns::grouped_pairs<192>() > 0 &&
                 rns::grouped_pairs<224>() > 0 && rns::grouped_pairs<256>() > 0
             ? CHASE_OK
             : CHASE_CUDA_ERROR;
}
int rns_grouped_crt(Dev& d, int nmod, const GroupedProblem* probs, const GroupedStep* steps,
                    int nact, int nblocks, int parity) {
  return rns::with_moduli(nmod, [&](auto nm) -> int {
    constexpr int NM = decltype(nm)::value;
    rns::rns_grouped_crt_kernel<NM><<<static_cast<unsigned>(nblocks), 128, 0, d.st>>>(
        probs, steps, nact, parity, rns::tables(NM, true).crt);
    note_launch();
    CHASE_CUDA(cudaGetLastError());
    return CHASE_OK;
  });
}

#define CHASE_INSTANTIATE_RNS(T)                                                                 \
  template int rns_prepare_h<T>(Dev&, const T*, int64_t, int64_t, int, int, size_t, bool, RnsH&); \
  template int rns_product<T>(Dev&, const RnsH&, RnsX&, const T*, int64_t, int, int, T*, int64_t, \
                              double, double, double, bool, int);
CHASE_INSTANTIATE_RNS(chase_c64)
CHASE_INSTANTIATE_RNS(double)
CHASE_INSTANTIATE_RNS(chase_c32)
CHASE_INSTANTIATE_RNS(float)
#undef CHASE_INSTANTIATE_RNS

}  // namespace chase
