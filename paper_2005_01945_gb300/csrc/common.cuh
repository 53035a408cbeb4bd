// common.cuh -- shared definitions of the sm_103a TFHE kernels.
//
// Ring and gadget shape are compile-time: N = 1024, k = 1, l = 2,
// Bg = 2^10, key switch t = 8, base 4.  The LWE dimension n is a runtime
// value (n <= 511).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/tfhe_gb.h"

namespace tgb {

constexpr int kN = 1024;                 // TLWE ring degree
constexpr int kL = 2;                    // gadget levels
constexpr int kRows = 2 * kL;            // rows of a TGSW sample (k = 1)
constexpr int kBgBit = 10;               // log2 Bg
constexpr int kKsT = 8;                  // key-switch levels
constexpr int kKsBaseBit = 2;            // log2 key-switch base
constexpr int kKsDigits = (1 << kKsBaseBit) - 1;
constexpr int kLweStride = TFHE_LWE_STRIDE;
constexpr int kBigStride = TFHE_BIG_STRIDE;
constexpr int kMaxN = kLweStride - 1;
constexpr uint32_t kMu = 1u << 29;       // 1/8

// Word offset that turns signed gadget digits into unsigned bit fields:
// 1/2 Bg per level plus the rounding half of the last level.
constexpr uint32_t kDecompOffset = (1u << 31) + (1u << 21) + (1u << 11);

// Two NTT primes below 2^27 with 2048 | q - 1.  Their product P ~ 2^54
// exceeds twice the largest magnitude of an exact external-product
// coefficient, 4 * N * 2^9 * 2^31 = 2^52, so the centred CRT lift is the
// exact integer.  q < 2^27 keeps every lazy value below 32 q < 2^32 and the
// 4-term pointwise sum of products of values within 8q and within q / 2 below
// 16 q^2 < q 2^31.
constexpr uint32_t kQ0 = 134215681u;     // 0x07FFF801
constexpr uint32_t kQ1 = 134203393u;     // 0x07FFC801
static_assert(32ull * kQ0 < (1ull << 32) && 32ull * kQ1 < (1ull << 32), "lazy bound");
static_assert((kQ0 - 1) % 2048 == 0 && (kQ1 - 1) % 2048 == 0, "2N-th roots of unity");
static_assert((unsigned __int128)kQ0 * kQ1 > ((unsigned __int128)1 << 53), "centred CRT lift");

// Status word bits (device-side errors).
constexpr uint32_t kErrGather = 1u;
constexpr uint32_t kErrScatter = 2u;
constexpr uint32_t kErrTimeout = 4u;
constexpr uint32_t kErrOpcode = 8u;

#if defined(__CUDACC__)
// x * w mod q in [0, 2q) for any 32-bit x, with wp = floor(w 2^32 / q)
// (Shoup's precomputed-quotient multiplication).
__device__ __forceinline__ uint32_t mul_shoup(uint32_t x, uint32_t w, uint32_t wp, uint32_t q)
{
    return x * w - __umulhi(x, wp) * q;
}

// x in [0, 2m) -> [0, m): subtract m when x >= m (unsigned min trick).
__device__ __forceinline__ uint32_t csub(uint32_t x, uint32_t m)
{
    return min(x, x - m);
}

// Shared-memory matrix descriptor: K-major, no swizzle; lbo = byte distance
// of core matrices adjacent in K, sbo = of 8-row groups.
__device__ __forceinline__ uint64_t tb_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) |
           ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}

// 16 consecutive columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tb_ld16(uint32_t t, uint32_t (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
                 "%10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                   "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]),
                   "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(t));
}
#endif  // __CUDACC__

// Blind-rotation shape codes: one bootstrap on a CTA's 16 warps, and one
// bootstrap on a cluster of two CTAs (one prime each).  1 is the throughput
// shape (4 bootstraps per CTA); 2, 4, kBrStaged, kBrStagedCtl and kBrFive are
// accepted for options and tuning files that name them and run it too.
constexpr int kBrSplit = 8;
constexpr int kBrPair = 16;
constexpr int kBrStaged = 32;
constexpr int kBrStagedCtl = 33;
constexpr int kBrFive = 5;
// Accepted as another name of kBrSplit.
constexpr int kBrSplitStaged = 40;
// Accepted as another name of kBrPair.
constexpr int kBrPairStaged = 48;
// Key-switch launch code for the tiled kernel (shared-memory key stages);
// the codes 1 .. 32 are j-chunks of the direct kernel.
constexpr int kKsTiled = 64;
// ... and for the tensor-pipe kernel (one-hot digits times key limbs).
constexpr int kKsTensor = 65;
// Device bytes of the key-switching key's limbs: 3 fp16 limbs of 512 words.
constexpr size_t kKlBytes = (size_t)kN * kKsT * kKsDigits * kLweStride * 3 * 2;
// Device bytes of the tensor-pipe first pass's constant operands and the signed
// inverse twiddles.
constexpr int kTbDevBytes = 28672;

// Per-context device pointers and sizes shared by the kernels.
struct DevKeys {
    const uint4 *bk_ntt;   // [n][2 poly][2 prime][32 reg][32 lane] x uint4(4 rows)
    const uint4 *ksk;      // [N][t][base-1][kLweStride/4] words
    const uint4 *ksk_limb; // fp16 limbs of it for the tensor-pipe key switch (kKlBytes)
    const uint2 *twb;      // stage-B twiddles [2 prime][2 dir][32 reg][32 lane] (w, w')
    const uint4 *tb_op;    // tensor-pipe first pass: constant operands, inverse twiddles
    int n;
    int br_group;          // blind-rotation shape code, 0 = tuned or by batch size
    int ks_kernel;         // key-switch kernel: kKsTiled, j-chunks 1 .. 32 of the
                           // direct kernel, 0 = tuned or by batch size
    int ks_stall;          // test hook (TFHE_OPT_TEST_KS_STALL): the stage waits
                           // of the tiled and tensor key switch run out
    int br_stall;          // test hook (TFHE_OPT_TEST_BR_STALL): the wait for this
                           // product, step or gate (by shape; from 1) runs out
    // Autotuned launch shapes per level-width bucket (0 = not tuned): bucket b
    // covers widths up to kTuneEdge[b] (the last bucket is unbounded).
    int8_t tune_br[8];     // blind-rotation shape
    int8_t tune_ks[8];     // key-switch kernel: kKsTiled, or j-chunks 1 .. 32
    // Autotuned time (ms) of one full blind-rotation wave, 4 bootstraps per
    // SM, in [0]; 0 = not measured ([1] keeps the tuning file's line format).
    float wave_ms[2];
    // Autotuned time (ms) of a level at each bucket's widest width with the
    // bucket's chosen shape; 0 = not measured.
    float tune_ms[8];
};

constexpr long kTuneEdge[8] = {152, 304, 608, 1216, 2432, 4864, 9728, 1L << 40};

inline int tune_bucket(long count)
{
    int b = 0;
    while (b < 7 && count > kTuneEdge[b])
        ++b;
    return b;
}

}  // namespace tgb
