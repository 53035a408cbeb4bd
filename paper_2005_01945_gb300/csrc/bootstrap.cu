// bootstrap.cu -- blind rotation (n CMux external products), fused with the
// gate combine, mod switch, test-vector rotation and sample extraction.
//
// The method: TFHE gate bootstrapping as adopted by the paper (section II-A;
// bootstrapping and key switching are timed separately in Table
// "differentialtime").  For every gate the accumulator starts as
// (0, X^-bbar v), v = mu (1 + X + ... + X^(N-1)), and for i < n becomes
// acc + BK_i [x] (X^abar_i acc - acc), where [x] decomposes the two
// polynomials of the TLWE sample into l = 2 signed base-2^10 digit
// polynomials each and sums digit_r * BK_i[r] in Z[X]/(X^N + 1) mod 2^32.
//
// GB300 design (not the paper's: it used cuFFT in floating point):
//  * the products are exact: a negacyclic NTT modulo two primes below 2^27
//    and a centred CRT lift back to Z/2^32;
//  * 4 warps own one bootstrap; a CTA of 16 warps per SM runs four that
//    share constants and otherwise run independently, looping over gates
//    (persistent grid); the accumulators never leave shared memory.  For
//    levels of at most one bootstrap per SM one bootstrap takes the 16 warps
//    (k_blind_rotate_wide), or a cluster of two CTAs (one prime each);
//  * the first pass of the forward transforms, on digits of 10 bits, is an
//    exact fp16 matrix product on the tensor pipe (k_blind_rotate_tc);
//  * one 1024-point transform is one warp: 32 coefficients per lane,
//    a 32-point transform in registers, a twiddle, one shared-memory
//    transpose, and a second 32-point transform (four-step NTT);
//  * the bootstrapping key is pre-transformed, scaled by 2^32 N^-1 and
//    interleaved so that lane l reads its 4 rows for one register as one
//    16-byte load; the 33 MB key stays L2-resident across gates.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace tgb {

// Shared-memory slots of 33 x 32 words: a transpose written as
// slot[i * 33 + lane] and read as slot[lane * 33 + j] is conflict-free with
// register + immediate addresses (no per-element address arithmetic).
constexpr int kSlot = 33 * 32;

struct NttConst {
    uint32_t za[2][32][2];   // forward stage A: w64^brv5(k), Shoup companion
    uint32_t zd[2][32][2];   // forward stage D: cyclic size-32 twiddles
    uint32_t iza[2][32][2];  // inverse of stage A
    uint32_t izd[2][32][2];  // inverse of stage D
    // signed transforms, centred (w, round(2^32 w / q)): stage D twiddles, the
    // inverse's by position ln + j, and the last pass's w64^-r
    int32_t zs[2][32][2], izs[2][32][2], post[2][32][2];
    int32_t one[2];          // round(2^32 / q)
    uint32_t q_inv[2];       // q^-1 mod 2^32
    int32_t crt_c, crt_cp;   // q0^-1 mod q1, centred, and round(2^32 crt_c / q1)
    uint32_t bk_scale[2][2]; // 2^32 N^-1 mod q and companion
};

__constant__ NttConst c_ntt;

__host__ __device__ constexpr int brv5(int k)
{
    return ((k & 1) << 4) | ((k & 2) << 2) | (k & 4) | ((k & 8) >> 2) | ((k & 16) >> 4);
}

// The transforms take the prime as a runtime value (one of two) so that a
// single copy of each transform serves both primes; twiddles are read from
// the constant bank with an offset on the prime.
struct Prime {
    uint32_t q, q2, P;
    __device__ __forceinline__ explicit Prime(uint32_t p)
        : q(p ? kQ1 : kQ0), q2(2 * (p ? kQ1 : kQ0)), P(p) {}
    // K q for K in {1, 2, 4, 8, 16, 32} (32 q < 2^32 for both primes)
    __device__ __forceinline__ uint32_t kq(int K) const
    {
        return K == 1 ? q : K == 2 ? q2 : K == 4 ? q2 << 1 : K == 8 ? q2 << 2
             : K == 16 ? q2 << 3 : q2 << 4;
    }
};

// ---------------------------------------------------------------------
// Lazy reductions.  Values are kept in [0, b q) with a per-element bound b
// known at compile time; a reduction csub(x, K q) (valid for b <= 2K)
// leaves [0, K q).  LazyPlan walks the 80 butterflies of a 32-point pass
// in the same order as the code and places the fewest reductions that keep
// every sum below thr q (<= kLazyMax q < 2^32), and the final outputs below
// fin q:
// CT butterfly (u, v) -> (u + t, u - t + K' q), t = v (trivial twiddle) or
// Shoup(v) in [0, 2q), K' >= bound(t) the smallest power of two.  The reduction is applied to the larger operand until the sum fits.
// ---------------------------------------------------------------------
struct LazyStep {
    uint8_t ru[4], nru;     // csub multiples K applied to u, in order
    uint8_t rv[4], nrv;     // ... to v (t of a trivial CT butterfly)
    uint8_t off;            // K' of the difference
};
struct LazyPlan {
    LazyStep st[5][16];     // [level][butterfly g * ln + jj]
    uint8_t fin[32][4], nfin[32];
    int reductions;
    bool ok;
};

constexpr int kLazyMax = 32;   // every lazy value stays below 32 q < 2^32

__host__ __device__ constexpr int lazy_off(int b)
{
    return b <= 1 ? 1 : b <= 2 ? 2 : b <= 4 ? 4 : b <= 8 ? 8 : b <= 16 ? 16 : 32;
}

// One reduction step of a value with bound b: the smallest K in
// {1, 2, 4, 8, 16} with 2K >= b; returns the new bound (or b if none
// applies).
__host__ __device__ constexpr int lazy_step(int b, int &K)
{
    K = b <= 2 ? 1 : b <= 4 ? 2 : b <= 8 ? 4 : b <= 16 ? 8 : b <= 32 ? 16 : 0;
    if (K == 0 || K >= b)
        return b;
    return K > b - K ? K : b - K;
}

__host__ __device__ constexpr LazyPlan make_lazy_plan(bool trivial_first, int in_b, int thr, int fin)
{
    LazyPlan P{};
    P.ok = true;
    int b[32] = {};
    for (int i = 0; i < 32; ++i)
        b[i] = in_b;
    for (int it = 0; it < 5; ++it) {
        const int s = it;
        const int m = 1 << s, ln = 16 >> s;
        for (int g = 0; g < m; ++g) {
            const bool triv = trivial_first && g == 0;
            for (int jj = 0; jj < ln; ++jj) {
                const int j = 2 * g * ln + jj;
                LazyStep &L = P.st[s][g * ln + jj];
                int bu = b[j], bv = b[j + ln];
                for (int guard = 0; guard < 8; ++guard) {
                    const int bt = triv ? bv : 2;
                    if (bu + bt <= thr && bu + lazy_off(bt) <= kLazyMax)
                        break;
                    int K = 0;
                    if (triv && bt >= bu) {
                        const int nb = lazy_step(bv, K);
                        if (nb == bv || L.nrv == 4) { P.ok = false; break; }
                        L.rv[L.nrv++] = (uint8_t)K;
                        bv = nb;
                    } else {
                        const int nb = lazy_step(bu, K);
                        if (nb == bu || L.nru == 4) { P.ok = false; break; }
                        L.ru[L.nru++] = (uint8_t)K;
                        bu = nb;
                    }
                }
                const int bt = triv ? bv : 2;
                L.off = (uint8_t)lazy_off(bt);
                P.reductions += L.nru + L.nrv;
                b[j] = bu + bt;
                b[j + ln] = bu + L.off;
                if (b[j] > kLazyMax || b[j + ln] > kLazyMax)
                    P.ok = false;
            }
        }
    }
    for (int i = 0; i < 32; ++i) {
        while (b[i] > fin) {
            int K = 0;
            const int nb = lazy_step(b[i], K);
            if (nb == b[i] || P.nfin[i] == 4) { P.ok = false; break; }
            P.fin[i][P.nfin[i]++] = (uint8_t)K;
            b[i] = nb;
        }
        P.reductions += P.nfin[i];
    }
    return P;
}

// Stage A (negacyclic twiddles, inputs [0, 2q), outputs < 12q, no reduction
// needed) and stage D (cyclic, the first twiddle of every level is 1; inputs
// [0, 2q), outputs [0, 8q) for the pointwise products).  The thresholds are the
// ones that need the fewest reductions.
constexpr LazyPlan kPlanFwdA = make_lazy_plan(false, 2, 12, kLazyMax);
constexpr LazyPlan kPlanFwdD = make_lazy_plan(true, 2, 8, 8);
static_assert(kPlanFwdA.ok && kPlanFwdD.ok, "lazy plan");
static_assert(kPlanFwdA.reductions == 0 && kPlanFwdD.reductions == 33, "lazy plan size");

__device__ __forceinline__ uint32_t lazy_reduce_n(uint32_t x, const uint8_t (&ks)[4], int n,
                                                  const Prime &pr)
{
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < n)
            x = csub(x, pr.kq(ks[k]));
    return x;
}

// 32-point Cooley-Tukey pass in registers (CYC false: stage A, negacyclic
// twiddles; CYC true: stage D, cyclic twiddles), reductions by plan.
template <bool CYC>
__device__ __forceinline__ void ct32(uint32_t (&x)[32], const Prime &pr)
{
    constexpr LazyPlan PL = CYC ? kPlanFwdD : kPlanFwdA;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int m = 1 << s, ln = 16 >> s;
#pragma unroll
        for (int g = 0; g < m; ++g) {
            const uint32_t(*tb)[32][2] = CYC ? c_ntt.zd : c_ntt.za;
            const uint32_t w = tb[pr.P][m + g][0];
            const uint32_t wp = tb[pr.P][m + g][1];
#pragma unroll
            for (int jj = 0; jj < ln; ++jj) {
                const int j = 2 * g * ln + jj;
                const LazyStep &L = PL.st[s][g * ln + jj];
                const uint32_t u = lazy_reduce_n(x[j], L.ru, L.nru, pr);
                const uint32_t t = (CYC && g == 0) ? lazy_reduce_n(x[j + ln], L.rv, L.nrv, pr)
                                                   : mul_shoup(x[j + ln], w, wp, pr.q);
                x[j] = u + t;
                x[j + ln] = u - t + pr.kq(L.off);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 32; ++r)
        x[r] = lazy_reduce_n(x[r], PL.fin[r], PL.nfin[r], pr);
}

// ---------------------------------------------------------------------
// Signed passes (k_blind_rotate_tc).  With centred twiddles (|w| <= q / 2, w' =
// round(2^32 w / q)) a Shoup product of a signed x, |x| <= a q <= 16 q, lies in
// [-a / 64, 1 + a / 64] q.  A decimation-in-time butterfly then takes four
// instructions,
//     hi = mulhi(x, w');  s = (x w + u) - hi q;  d = 2 u - s,
// where an unsigned one takes five (a sum, and a difference with an offset),
// and bounds grow by one q a stage except along the twiddles 1, so that a
// forward pass needs 7 reductions instead of 33.  (The sum and difference of a
// product formed first: 608 gates 5.93 ms, so 5.56.)
// ---------------------------------------------------------------------
struct SignedPlan {
    bool ru[5][16], rv[5][16];   // reduce u / v of a butterfly first
    bool fin[32];                // reduce the output
    int reductions;
    bool ok;
};

// Intervals in units of q / 64: inputs [lo, hi], no sum beyond thr, outputs
// within +-out.  dit: distances 1 .. 16, twiddle 1 at j = 0; else distances
// 16 .. 1, twiddle 1 in group 0.
__host__ __device__ constexpr SignedPlan make_signed_plan(bool dit, int lo0, int hi0, int thr, int out)
{
    SignedPlan P{};
    P.ok = true;
    int lo[32] = {}, hi[32] = {};
    for (int i = 0; i < 32; ++i)
        lo[i] = lo0, hi[i] = hi0;
    for (int s = 0; s < 5; ++s) {
        const int ln = dit ? 1 << s : 16 >> s;
        for (int b = 0; b < 16; ++b) {
            const int g = b / ln, j = b % ln, iu = 2 * g * ln + j, iv = iu + ln;
            const bool triv = dit ? j == 0 : g == 0;
            for (int guard = 0; guard < 3; ++guard) {
                const int av = lo[iv] < -hi[iv] ? -lo[iv] : hi[iv], au = lo[iu] < -hi[iu] ? -lo[iu] : hi[iu];
                const int t = triv ? av : 64 + (av + 63) / 64;
                if (au + t <= thr)
                    break;
                const bool v = triv && av >= au;
                const int i = v ? iv : iu, a = ((v ? av : au) + 63) / 64;
                (v ? P.rv : P.ru)[s][b] = true;
                lo[i] = -a, hi[i] = 64 + a;
                ++P.reductions;
                P.ok = P.ok && guard < 2;
            }
            const int a = ((lo[iv] < -hi[iv] ? -lo[iv] : hi[iv]) + 63) / 64;
            const int tl = triv ? lo[iv] : -a, th = triv ? hi[iv] : 64 + a;
            const int ul = lo[iu], uh = hi[iu];
            lo[iu] = ul + tl, hi[iu] = uh + th;
            lo[iv] = ul - th, hi[iv] = uh - tl;
        }
    }
    for (int i = 0; i < 32; ++i) {
        P.fin[i] = lo[i] < -out || hi[i] > out;
        P.reductions += P.fin[i];
    }
    return P;
}

constexpr int kSignedMax = 15 * 64;   // 15 q < 2^31
// Forward second pass: inputs below q (1 + 4 / 32), outputs within 8q for the
// pointwise products.  Inverse passes: inputs from the pointwise step
// (-q, q), then from the twiddle; outputs into a Shoup product.
constexpr SignedPlan kSignedFwd = make_signed_plan(false, 0, 72, kSignedMax, 8 * 64);
constexpr SignedPlan kSignedInvD = make_signed_plan(true, -64, 64, kSignedMax, kSignedMax);
constexpr SignedPlan kSignedInvA = make_signed_plan(true, -16, 80, kSignedMax, kSignedMax);
static_assert(kSignedFwd.ok && kSignedInvD.ok && kSignedInvA.ok, "signed plan");
static_assert(kSignedFwd.reductions == 7 && kSignedInvD.reductions == 3 &&
              kSignedInvA.reductions == 3, "signed plan size");

__device__ __forceinline__ int32_t mul_signed(int32_t x, int32_t w, int32_t wp, int32_t q)
{
    return (int32_t)((uint32_t)x * (uint32_t)w - (uint32_t)__mulhi(x, wp) * (uint32_t)q);
}

__device__ __forceinline__ int32_t reduce_signed(int32_t x, const Prime &pr)
{
    return (int32_t)((uint32_t)x - (uint32_t)__mulhi(x, c_ntt.one[pr.P]) * pr.q);
}

// DIT false: ct32<true>; true: 32 times its inverse, input in ct32's output order.
template <bool DIT, bool LAST = false>
__device__ __forceinline__ void pass32_signed(int32_t (&x)[32], const Prime &pr)
{
    constexpr SignedPlan PL = !DIT ? kSignedFwd : LAST ? kSignedInvA : kSignedInvD;
    const int32_t(*tb)[2] = DIT ? c_ntt.izs[pr.P] : c_ntt.zs[pr.P];
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int ln = DIT ? 1 << s : 16 >> s;
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            const int g = b / ln, j = b % ln, iu = 2 * g * ln + j, iv = iu + ln;
            const bool triv = DIT ? j == 0 : g == 0;
            const int32_t u = PL.ru[s][b] ? reduce_signed(x[iu], pr) : x[iu];
            const int32_t v = PL.rv[s][b] ? reduce_signed(x[iv], pr) : x[iv];
            if (triv) {
                x[iu] = u + v;
                x[iv] = u - v;
            } else {
                const int k = DIT ? ln + j : (1 << s) + g;
                const int32_t hi = __mulhi(v, tb[k][1]);
                const uint32_t sum = ((uint32_t)v * (uint32_t)tb[k][0] + (uint32_t)u) -
                                     (uint32_t)hi * pr.q;
                x[iu] = (int32_t)sum;
                x[iv] = (int32_t)((uint32_t)u + (uint32_t)u - sum);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 32; ++r)
        if (PL.fin[r])
            x[r] = reduce_signed(x[r], pr);
}

// Forward negacyclic NTT of one polynomial held by one warp.
// In : lane l, register r holds coefficient l + 32 r, value in [0, 2q).
// Out: lane l, register r holds the evaluation at psi^(2 (l + 32 brv5(r)) + 1),
//      value in [0, 8q).  sbuf: kSlot words of this warp's shared memory.
__device__ __forceinline__ void fwd_ntt(uint32_t (&x)[32], uint32_t *sbuf, int lane,
                                        const uint2 *__restrict__ twb, const Prime &pr)
{
    ct32<false>(x, pr);
    const uint2 *tw = twb + (pr.P * 2 + 0) * 1024 + lane;
#pragma unroll
    for (int r = 0; r < 32; ++r) {   // any 32-bit input -> [0, 2q)
        const uint2 t = __ldg(tw + r * 32);
        x[r] = mul_shoup(x[r], t.x, t.y, pr.q);
    }
    uint32_t *wr = sbuf + lane, *rd = sbuf + lane * 33;
#pragma unroll
    for (int r = 0; r < 32; ++r)
        wr[brv5(r) * 33] = x[r];       // lane i1, k1 = brv5(r) -> slot[k1][i1]
    __syncwarp();
#pragma unroll
    for (int i1 = 0; i1 < 32; ++i1)
        x[i1] = rd[i1];                // lane k1 reads slot[k1][i1]
    __syncwarp();
    ct32<true>(x, pr);
}

// ---------------------------------------------------------------------
// Bootstrapping key -> NTT domain
// ---------------------------------------------------------------------

// One warp per (i, row, poly, prime).  bk: int32 [n][4][2][N] coefficient
// form.  Output element (i, p, q, reg, lane) is a uint4 over the 4 rows.
__global__ void __launch_bounds__(128) k_bk_to_ntt(const int32_t *__restrict__ bk, uint32_t *out,
                                                   int n, const uint2 *__restrict__ twb)
{
    __shared__ uint32_t sbuf[4][kSlot];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long task = (long)blockIdx.x * 4 + warp;  // ((i * 4 + r) * 2 + p) * 2 + q
    if (task >= (long)n * kRows * 2 * 2)
        return;
    const int qsel = task & 1, p = (task >> 1) & 1, r = (task >> 2) & 3;
    const long i = task >> 4;
    const int32_t *src = bk + ((i * kRows + r) * 2 + p) * kN;
    uint32_t x[32];
    const uint32_t q = qsel == 0 ? kQ0 : kQ1;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        int64_t v = src[lane + 32 * k];               // centred representative
        int64_t m = v % (int64_t)q;
        x[k] = (uint32_t)(m < 0 ? m + q : m);
    }
    fwd_ntt(x, sbuf[warp], lane, twb, Prime((uint32_t)qsel));
    const uint32_t sc = c_ntt.bk_scale[qsel][0], scp = c_ntt.bk_scale[qsel][1];
    // element index in uint32 words: ((((i*2+p)*2+q)*32 + reg)*32 + lane)*4 + r
    uint32_t *dst = out + ((((i * 2 + p) * 2 + qsel) * 32) * 32 + lane) * 4 + r;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        uint32_t v = x[k] % q;                         // [0, 8q) -> [0, q)
        v = csub(mul_shoup(v, sc, scp, q), q);        // * 2^32 N^-1, in [0, q)
        dst[k * 32 * 4] = v > q / 2 ? v - q : v;       // centred
    }
}

// ---------------------------------------------------------------------
// Blind rotation
// ---------------------------------------------------------------------

struct BrArgs {
    DevKeys keys;
    const int32_t *in_a, *in_b, *in_c;    // ciphertext bases (row stride kLweStride)
    const int32_t *idx_a, *idx_b, *idx_c; // optional gather rows (nullptr: row g)
    long rows_a, rows_b, rows_c;          // rows addressable through the bases
    const uint8_t *ops;              // gate opcodes (nullptr: bootstrap in_a as is)
    int32_t *big;                    // out: LWE_N samples [count][kBigStride]
    long first, count;               // gates first .. count - 1
    uint32_t mu;                     // test-vector amplitude
    uint32_t *status;
};

// Tries of a bounded wait, about 4 us each: about a second (a constant: with the
// limit as an argument the two-CTA shape took 1.7 % longer).
constexpr long kBkSpin = 1L << 18;

__device__ __forceinline__ uint32_t br_saddr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Bounded wait for phase `parity` of a barrier; false if it ran out.
__device__ __forceinline__ bool bk_wait(unsigned long long *bar, uint32_t parity)
{
    uint32_t ok;
    // the first try suspends for the hardware's own time, not a timer's
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(br_saddr(bar)), "r"(parity)
                 : "memory");
    if (ok)
        return true;
    for (long i = 0; i < kBkSpin; ++i) {
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(br_saddr(bar)), "r"(parity), "r"(1000u)
                     : "memory");
        if (ok)
            return true;
    }
    return false;
}

// Phase 4: CRT of (v0 mod q0, v1 mod q1), any representatives within 8q of each
// other (the signed inverse leaves [-q / 4, 5 q / 4], the others [0, 8q)), to
// the centred integer, mod 2^32.  Garner: the exact coefficient S satisfies
// |S| <= 4 N 2^9 2^31 = 2^52, so u = (S - v0) / q0 is an integer of magnitude
// at most 2^25 + 8, about q1 / 4, and u = (v1 - v0) q0^-1 mod q1.  The
// product's quotient by q1 is rounded to nearest: the approximate reciprocal
// is off by at most |v1 - v0| / 2^33 < 1/8, and 1/4 + 1/8 < 1/2, so u comes
// out centred and exact without a correction.  (With residues in [0, q), a
// floor quotient and a compare for the centring: 608 gates 5.94 ms, now 5.87.)
__device__ __forceinline__ uint32_t crt_lift(uint32_t v0, uint32_t v1, int32_t c, int32_t cp)
{
    const int32_t x = (int32_t)(v1 - v0);
    const int32_t k = (int32_t)(((int64_t)x * cp + 0x80000000ll) >> 32);
    const uint32_t u = (uint32_t)x * (uint32_t)c - (uint32_t)k * kQ1;
    return v0 + kQ0 * u;
}

// Linear part of gate `op`: c = mu + aa ca + ab cb + ac cc.  Returns false
// for an unknown opcode.
__device__ __forceinline__ bool gate_consts(int op, uint32_t &mu, uint32_t &aa, uint32_t &ab,
                                            uint32_t &ac)
{
    ac = 0u;
    switch (op) {
    case TFHE_NAND:  mu = kMu;           aa = ab = 0u - 1u; return true;
    case TFHE_AND:   mu = 0u - kMu;      aa = ab = 1u;      return true;
    case TFHE_OR:    mu = kMu;           aa = ab = 1u;      return true;
    case TFHE_XOR:   mu = 2u * kMu;      aa = ab = 2u;      return true;
    case TFHE_NOR:   mu = 0u - kMu;      aa = ab = 0u - 1u; return true;
    case TFHE_XNOR:  mu = 0u - 2u * kMu; aa = ab = 0u - 2u; return true;
    case TFHE_MAJ:   mu = 0u;            aa = ab = ac = 1u; return true;
    case TFHE_ANDNY: mu = 0u - kMu;      aa = 0u - 1u; ab = 1u; return true;
    case TFHE_ANDYN: mu = 0u - kMu;      aa = 1u; ab = 0u - 1u; return true;
    case TFHE_ORNY:  mu = kMu;           aa = 0u - 1u; ab = 1u; return true;
    case TFHE_ORYN:  mu = kMu;           aa = 1u; ab = 0u - 1u; return true;
    default:         mu = 0u;            aa = ab = 0u;      return false;
    }
}

// Gate combine + mod switch (the fused prologue) of gate slot g into
// abar[0..n] by the T threads of one bootstrap.  An empty slot (g >= count)
// or a bad one runs with abar = 0; a bad slot (opcode without its inputs,
// gather index out of range) is flagged in the status word and, when
// `writer`, its output row is zeroed.  Returns whether the slot is active.
template <int T>
__device__ __forceinline__ bool br_prologue(const BrArgs &A, long g, int tb, uint16_t *abar,
                                            bool writer)
{
    const int n = A.keys.n;
    bool active = g < A.count;
    long ra = 0, rb = 0, rc = -1;
    uint32_t mu_g = 0, aa = 1, ab = 0, ac = 0;
    if (active) {
        uint32_t err = 0;
        if (A.ops && !gate_consts(A.ops[g], mu_g, aa, ab, ac))
            err = kErrOpcode;
        ra = A.idx_a ? (long)A.idx_a[g] : g;
        rb = A.ops ? (A.idx_b ? (long)A.idx_b[g] : g) : 0;
        if (ac) {
            if (!A.in_c)
                err |= kErrOpcode;
            else
                rc = A.idx_c ? (long)A.idx_c[g] : g;
        }
        if (!(ra >= 0 && ra < A.rows_a && (!A.ops || (rb >= 0 && rb < A.rows_b)) &&
              (!ac || !A.in_c || (rc >= 0 && rc < A.rows_c))))
            err |= kErrGather;
        if (err) {
            if (writer) {
                if (tb == 0)
                    atomicOr(A.status, err);
                int32_t *bg = A.big + g * kBigStride;
                for (int k = tb; k <= kN; k += T)
                    bg[k] = 0;
            }
            active = false;
        }
    }
    if (active) {
        const int32_t *ca = A.in_a + ra * kLweStride;
        const int32_t *cb = A.ops ? A.in_b + rb * kLweStride : nullptr;
        const int32_t *cc = ac ? A.in_c + rc * kLweStride : nullptr;
        for (int i = tb; i <= n; i += T) {
            uint32_t c = (uint32_t)ca[i];
            if (A.ops) {
                c = aa * c + ab * (uint32_t)cb[i];
                if (ac)
                    c += ac * (uint32_t)cc[i];
            }
            if (i == n)
                c += mu_g;
            abar[i] = (uint16_t)(((c + (1u << 20)) >> 21) & (2 * kN - 1));
        }
    } else {
        for (int i = tb; i <= n; i += T)
            abar[i] = 0;
    }
    return active;
}

// acc = (0, X^(-bbar) v), v = mu (1 + X + ... + X^(N-1)).
template <int T>
__device__ __forceinline__ void br_acc_init(const BrArgs &A, uint32_t (*acc)[kN], int bbar, int tb)
{
    const int m = (2 * kN - bbar) & (2 * kN - 1);
    for (int k = tb; k < kN; k += T) {
        bool pos = k >= (m & (kN - 1));
        if (m >= kN)
            pos = !pos;
        acc[0][k] = 0u;
        acc[1][k] = pos ? A.mu : 0u - A.mu;
    }
}

// Sample extraction of coefficient 0: a'_0 = a_0, a'_j = -a_(N-j), b' = b_0.
template <int T>
__device__ __forceinline__ void br_extract(const BrArgs &A, long g, const uint32_t (*acc)[kN],
                                           int tb)
{
    int32_t *bg = A.big + g * kBigStride;
    for (int k = tb; k < kN; k += T)
        bg[k] = (int32_t)(k == 0 ? acc[0][0] : 0u - acc[0][kN - k]);
    if (tb == 0)
        bg[kN] = (int32_t)acc[1][0];
}

// ---------------------------------------------------------------------
// Blind rotation with the forward transforms' first pass on the tensor pipe
// ---------------------------------------------------------------------
//
// The first pass of every forward transform is 32 negacyclic 32-point
// transforms of digits, and digits are small (10 bits), so the pass is an
// exact matrix product on the tensor pipe: for digit row s (of 4) and
// column i1,
//     V_h[s, i1][k1] = sum_i2 d_s[i1 + 32 i2] * psi_h^(32 (2 k1 + 1) i2),
// i.e. a [128 x 32] fp16 matrix of digits (row 32 s + i1, exact: |d| <= 512)
// times a constant [32 x 96] fp16 matrix per prime: the centred powers in
// three balanced base-512 limbs (|limb| <= 256, exact in fp16).  Each fp32
// sum s_l is at most 512 sum |limb| < 2^22 (checked when the operand is
// built): an exact integer.  The accumulators start at 1.5 2^23 (one more
// K step, 2048 x 6144), so a sum's bits are 0x4B400000 + s_l.
//
// A lane then forms x = sum_l 512^l s_l - Q q + 2q, Q = round(sum / q) from
// two fp32 multiply-adds (off by less than 1.6, so x lies in (0, 4q)), and
// the twiddle as a Shoup product: 17 issue cycles per point (2 ffma, 3 imad
// or shift-adds at 2, 1 add, Shoup 8) against 35 of an 80-butterfly pass and
// its twiddle product.  The twiddles of both primes stay in TMEM beside the
// accumulators (128 words per lane, columns 384 on, read like them), so the
// pass takes nothing from the load/store pipe but its result's transpose.
constexpr int kTbCols = 96;                        // 32 outputs x 3 limbs of one prime
constexpr uint32_t kTbOpBytes = kTbCols * 32 * 2;  // constant operand of one prime, 6 KB
static_assert(2 * kTbOpBytes + 2 * 1024 * sizeof(int2) == kTbDevBytes, "operand buffer");
constexpr int kTbTw = 4 * kTbCols;                 // TMEM column of the twiddles
constexpr uint32_t kMagicBits = 0x4B400000u;

// Transposes in 36-word rows: 16-byte rows for vector accesses along the row
// (eight lanes cover all banks), consecutive words across.
constexpr int kRowV = 36;
constexpr int kSlotV = 32 * kRowV;

// Word of (register r, lane) in a vector-ordered row of kN words: four
// consecutive registers of a lane are one 16-byte access.
__host__ __device__ constexpr int vec_word(int r, int lane)
{
    return ((r >> 2) * 32 + lane) * 4 + (r & 3);
}

struct TbSmem {                 // one bootstrap
    uint32_t acc[2][kN];        // TLWE accumulator (a(X), b(X))
    uint32_t fwd[2][4][kSlotV]; // forward outputs [prime][digit row] (vec_word); scratch
    uint16_t abar[kLweStride];  // mod-switched mask and body
};

struct TbOps {                  // one CTA
    // constant operands, 8 x 8 fp16 core matrices [K group][column group]
    uint8_t b[2][kTbOpBytes];
    uint8_t b1[kTbCols * 16 * 2];   // the K step of the accumulators' start value
    uint8_t a1[128 * 16 * 2];
    unsigned long long bar[4];  // MMA completion of each bootstrap
    unsigned long long spare[4];    // test hook: completion of the product whose wait runs out
                                    // (two-CTA shape: of all, after a wait that ran out)
    uint32_t tmem;
    volatile int abort[4];      // a wait of the bootstrap ran out (two-CTA shape: in this
                                // step, from 1)
};

// Barrier of the 128 threads of bootstrap slot `bi`.
__device__ __forceinline__ void boot_sync(int bi)
{
    asm volatile("bar.sync %0, 128;" ::"r"(1 + bi) : "memory");
}

// Inverse transform up to the factor N, signed: lane k1, register k2 (bit-
// reversed), values in (-q, q), to lane i1, register i2, residues in
// [-q / 4, 5 q / 4].  The transpose is written by words and read as 16-byte
// vectors.  The last pass is the cyclic one and a product by w64^-r behind it:
// 49 + 31 products in four-instruction butterflies and alone, where the
// negacyclic pass has 80 in five-instruction ones.
__device__ __forceinline__ void inv_ntt_v(int32_t (&x)[32], uint32_t *sbuf, int lane, int lane_brv,
                                          const int2 *__restrict__ tw, const Prime &pr, int bi)
{
    pass32_signed<true>(x, pr);
    boot_sync(bi);   // the other warps have read the row that is the scratch
    uint32_t *wr = sbuf + lane_brv, *rd = sbuf + lane * kRowV;
    // products and stores alternate (all stores behind the products: 608 gates
    // 6.07 ms, so 5.56)
#pragma unroll
    for (int r = 0; r < 32; ++r) {     // lane k1, i1 = r -> slot[i1][brv5(k1)]
        const int2 t = __ldg(tw + r * 32);
        wr[r * kRowV] = (uint32_t)mul_signed(x[r], t.x, t.y, pr.q);
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 32; r += 4) {  // lane i1 reads slot[i1][r ..]
        const int4 v = *reinterpret_cast<const int4 *>(rd + r);
        x[r] = v.x;
        x[r + 1] = v.y;
        x[r + 2] = v.z;
        x[r + 3] = v.w;
    }
    __syncwarp();
    pass32_signed<true, true>(x, pr);
    x[0] = reduce_signed(x[0], pr);
#pragma unroll
    for (int r = 1; r < 32; ++r)
        x[r] = mul_signed(x[r], c_ntt.post[pr.P][r][0], c_ntt.post[pr.P][r][1], pr.q);
}

__device__ __forceinline__ void store_vec(uint32_t *row, const int32_t (&x)[32], int lane)
{
#pragma unroll
    for (int r = 0; r < 32; r += 4)
        *reinterpret_cast<int4 *>(row + vec_word(r, lane)) =
            make_int4(x[r], x[r + 1], x[r + 2], x[r + 3]);
}

// Key vectors of registers 4 g .. 4 g + 3.
__device__ __forceinline__ void key_ld4(uint4 (&k)[4], const uint4 *__restrict__ bkp, int g, int lane)
{
#pragma unroll
    for (int e = 0; e < 4; ++e)
        k[e] = __ldg(bkp + (4 * g + e) * 32 + lane);
}

// Phase 2 of registers 4 g .. 4 g + 3 on vector-ordered rows (values within
// 8q) into x[at ..], in (-q, q); their key vectors (centred) are k[at ..] (k[0 ..]
// of an array of four).  Montgomery: with |s| <= 4 8q q/2 < 2^31 q and m = s
// q^-1 mod 2^32 signed, (s - m q) 2^-32 is the difference of the high words.
template <int M, int KN, int W>
__device__ __forceinline__ void pointwise_4(int32_t (&x)[M], int at, const uint32_t (*f)[W], int g,
                                            const uint4 (&k)[KN], int lane, const Prime &pr)
{
    const uint32_t qn = c_ntt.q_inv[pr.P];
    const int o = vec_word(4 * g, lane);
    const int4 f0 = *reinterpret_cast<const int4 *>(f[0] + o);
    const int4 f1 = *reinterpret_cast<const int4 *>(f[1] + o);
    const int4 f2 = *reinterpret_cast<const int4 *>(f[2] + o);
    const int4 f3 = *reinterpret_cast<const int4 *>(f[3] + o);
    const int32_t a0[4] = {f0.x, f0.y, f0.z, f0.w}, a1[4] = {f1.x, f1.y, f1.z, f1.w};
    const int32_t a2[4] = {f2.x, f2.y, f2.z, f2.w}, a3[4] = {f3.x, f3.y, f3.z, f3.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint4 b = k[KN == 4 ? e : at + e];
        int64_t s = (int64_t)a0[e] * (int32_t)b.x;
        s += (int64_t)a1[e] * (int32_t)b.y;
        s += (int64_t)a2[e] * (int32_t)b.z;
        s += (int64_t)a3[e] * (int32_t)b.w;
        const int32_t m = (int32_t)((uint32_t)s * qn);
        x[at + e] = (int32_t)(s >> 32) - __mulhi(m, (int32_t)pr.q);
    }
}

// Phase 2 on vector-ordered rows; `k` holds the key vectors of group 0,
// loaded before the barrier that made the rows complete.  The key vectors
// of the next group are in flight while a group is multiplied.
__device__ __forceinline__ void pointwise_v(int32_t (&x)[32], const uint32_t (*f)[kSlotV],
                                            uint4 (&k)[4], const uint4 *__restrict__ bkp, int lane,
                                            const Prime &pr)
{
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        uint4 nk[4];
        if (g < 7)
            key_ld4(nk, bkp, g + 1, lane);
        pointwise_4(x, 4 * g, f, g, k, lane, pr);
        if (g < 7)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                k[e] = nk[e];
    }
}

// Phase 4 (crt_lift) of registers r0 .. r0 + NR - 1 on vector-ordered
// residue rows.
template <int NR>
__device__ __forceinline__ void crt_rows_v(uint32_t *acc, const uint32_t *x0, const uint32_t *x1,
                                           int r0, int lane)
{
    const int32_t c = c_ntt.crt_c, cp = c_ntt.crt_cp;
#pragma unroll
    for (int rr = 0; rr < NR; rr += 4) {
        const int o = vec_word(r0 + rr, lane);
        const uint4 v0 = *reinterpret_cast<const uint4 *>(x0 + o);
        const uint4 v1 = *reinterpret_cast<const uint4 *>(x1 + o);
        const uint32_t a0[4] = {v0.x, v0.y, v0.z, v0.w}, a1[4] = {v1.x, v1.y, v1.z, v1.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            acc[(r0 + rr + e) * 32 + lane] += crt_lift(a0[e], a1[e], c, cp);
    }
}


// kind::f16, fp16 A and B (K-major), fp32 accumulator, M = 128, N = 96.
constexpr uint32_t kTbIdesc = (1u << 4) | ((uint32_t)(kTbCols >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

__device__ __forceinline__ void tb_mma1(uint32_t d, uint64_t a, uint64_t b, uint32_t acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                 "l"(a), "l"(b), "r"(kTbIdesc), "r"(acc)
                 : "memory");
}

// One thread: V_h of one bootstrap into TMEM columns d .. d + 95, completion
// on `bar`.  The digit operand `a` holds 8 x 8 core matrices [K group 4][row
// group 16].
__device__ __forceinline__ void tb_mma(uint32_t d, uint32_t a, const TbOps &O, int prime,
                                       unsigned long long *bar)
{
    tb_mma1(d, tb_desc(br_saddr(O.a1), 2048, 128), tb_desc(br_saddr(O.b1), kTbCols * 16, 128), 0);
#pragma unroll
    for (int kk = 0; kk < 2; ++kk)
        tb_mma1(d, tb_desc(a + kk * 2 * 2048, 2048, 128),
                tb_desc(br_saddr(&O.b[prime][0]) + kk * 2 * (kTbCols * 16), kTbCols * 16, 128), 1);
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     br_saddr(bar))
                 : "memory");
}

// 8 consecutive columns of this warp's 32 TMEM lanes (16: tb_ld16).
__device__ __forceinline__ void tb_ld8(uint32_t t, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                   "=r"(v[6]), "=r"(v[7])
                 : "r"(t));
}

// Both digits of the words u0 and u1 (offset added) as fp16 pairs.
// 1024 + field is exact in fp16 (bits 0x6400 | field).
__device__ __forceinline__ void tb_digit2(uint32_t u0, uint32_t u1, uint32_t &d0, uint32_t &d1)
{
    const uint32_t hi = (__byte_perm(u0, u1, 0x7632) >> 6) & 0x03FF03FFu;   // bits 22..31
    const uint32_t lo = (__byte_perm(u0, u1, 0x6521) >> 4) & 0x03FF03FFu;   // bits 12..21
    const __half2 off = __half2half2(__ushort_as_half(0x6600));   // 1536 = 1024 + 512
    const uint32_t h1 = hi | 0x64006400u, l1 = lo | 0x64006400u;
    const __half2 x0 = __hsub2(*reinterpret_cast<const __half2 *>(&h1), off);
    const __half2 x1 = __hsub2(*reinterpret_cast<const __half2 *>(&l1), off);
    d0 = *reinterpret_cast<const uint32_t *>(&x0);
    d1 = *reinterpret_cast<const uint32_t *>(&x1);
}

// Both digits of the coefficients lane + 32 r, r = 16 half .. + 15, of
// polynomial c of X^a acc - acc, as fp16 into rows (2c + j) 32 + lane of the
// digit operand.
__device__ __forceinline__ void tb_digits(const uint32_t *ac, uint8_t *op, int c, int half, int a,
                                          int lane)
{
#pragma unroll
    for (int g = 0; g < 2; ++g) {   // K group: 8 consecutive r
        uint32_t d0[4], d1[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            uint32_t u[2];
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const int k = lane + 32 * (16 * half + 8 * g + 2 * e + o);
                const int idx = (k - a) & (2 * kN - 1);
                uint32_t v = ac[idx & (kN - 1)];
                v = idx >= kN ? 0u - v : v;
                u[o] = v - ac[k] + kDecompOffset;
            }
            tb_digit2(u[0], u[1], d0[e], d1[e]);
        }
        uint8_t *p = op + (2 * half + g) * 2048 + (64 * c + lane) * 16;
        *reinterpret_cast<uint4 *>(p) = make_uint4(d0[0], d0[1], d0[2], d0[3]);
        *reinterpret_cast<uint4 *>(p + 32 * 16) = make_uint4(d1[0], d1[1], d1[2], d1[3]);
    }
}

// (a0, a1) * b + c of packed fp32 bits, and the same from two words.
__device__ __forceinline__ uint64_t ffma2_of(uint32_t a0, uint32_t a1, float b, float c)
{
    uint64_t r;
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %3};\n\t"
        "mov.b64 c, {%4, %4};\n\tfma.rn.f32x2 %0, a, b, c;\n\t}"
        : "=l"(r)
        : "r"(a0), "r"(a1), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ void ffma2(uint32_t &a0, uint32_t &a1, float b, uint64_t c)
{
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %2};\n\t"
        "fma.rn.f32x2 a, a, b, %3;\n\tmov.b64 {%0, %1}, a;\n\t}"
        : "+r"(a0), "+r"(a1)
        : "f"(b), "l"(c));
}

// Second half of the first pass for one digit row: the warp's 32 TMEM lanes
// (lane i1) hold the sums of column k1 at t + 24 (k1 / 8) + 8 l + k1 % 8 and
// its twiddle (w, w') at tw + 2 k1; twiddled residues in [0, 2q) go to
// slot[i1][k1].
__device__ __forceinline__ void tb_combine(uint32_t t, uint32_t tw, uint32_t *slot, const Prime &pr,
                                           int k_lo = 0, int k_hi = 32)
{
    const float c1 = pr.P ? (float)(512.0 / kQ1) : (float)(512.0 / kQ0);
    const float c2 = pr.P ? (float)(262144.0 / kQ1) : (float)(262144.0 / kQ0);
    const float c0 = pr.P ? (float)(12582912.0 * (1.0 - 262656.0 / kQ1))
                          : (float)(12582912.0 * (1.0 - 262656.0 / kQ0));
    const uint32_t off = 2u * pr.q + kMagicBits * pr.q - kMagicBits * (1u + 512u + 262144u);
    const uint32_t nq = 0u - pr.q;
#pragma unroll 1
    for (int k0 = k_lo; k0 < k_hi; k0 += 8) {
        uint32_t s0[8], s1[8], s2[8], w[16];
        tb_ld8(t + 3 * k0, s0);
        tb_ld8(t + 3 * k0 + 8, s1);
        tb_ld8(t + 3 * k0 + 16, s2);
        tb_ld16(tw + 2 * k0, w);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int v = 0; v < 8; v += 4) {
            uint32_t o[4], f[4];   // f: the quotients' bits
#pragma unroll
            for (int k = 0; k < 4; k += 2) {
                const int e = v + k;
                f[k] = s2[e], f[k + 1] = s2[e + 1];
                ffma2(f[k], f[k + 1], c2, ffma2_of(s1[e], s1[e + 1], c1, c0));
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int e = v + k;
                const uint32_t y = (s1[e] << 9) + ((s2[e] << 18) + s0[e]);
                const uint32_t x = f[k] * nq + (y + off);
                o[k] = mul_shoup(x, w[2 * e], w[2 * e + 1], pr.q);
            }
            *reinterpret_cast<uint4 *>(slot + k0 + v) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

// Prologue of a 512-thread CTA: constant operands, barriers, all of TMEM, and
// the forward twiddles at TMEM column tw_col.
__device__ __forceinline__ void tb_setup(const BrArgs &A, TbOps &O, int tid, int tw_col)
{
    const int warp = tid >> 5, lane = tid & 31;
    for (int e = tid; e < (int)(2 * kTbOpBytes / 16); e += 512)
        reinterpret_cast<uint4 *>(&O.b[0][0])[e] = __ldg(A.keys.tb_op + e);
    // start value 2048 x 6144 = 1.5 2^23: K value 0 of every row and column
    for (int e = tid; e < (int)(sizeof(O.a1) / 16); e += 512)
        reinterpret_cast<uint4 *>(O.a1)[e] = make_uint4(e < 128 ? 0x6800u : 0u, 0u, 0u, 0u);
    for (int e = tid; e < (int)(sizeof(O.b1) / 16); e += 512)
        reinterpret_cast<uint4 *>(O.b1)[e] = make_uint4(e < kTbCols ? 0x6E00u : 0u, 0u, 0u, 0u);
    if (tid < 4) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(br_saddr(&O.bar[tid]))
                     : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(br_saddr(&O.spare[tid]))
                     : "memory");
        O.abort[tid] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         br_saddr(&O.tmem)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp < 4) {
        const uint32_t tl = O.tmem + ((uint32_t)(32 * warp) << 16);
        // forward twiddles of column i1 = lane: (w, w') of prime P, output k1
        // at column tw_col + 2 (32 P + k1)
        for (int c = 0; c < 64; c += 4) {
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int P = (c + e) >> 5, k1 = (c + e) & 31;
                const uint2 f = __ldg(A.keys.twb + ((P * 2) * 32 + brv5(k1)) * 32 + lane);
                v[2 * e] = f.x;
                v[2 * e + 1] = f.y;
            }
            asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, "
                         "%8};" ::"r"(tl + tw_col + 2 * c),
                         "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]),
                         "r"(v[6]), "r"(v[7])
                         : "memory");
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Frees TMEM; the last thing a CTA does.
__device__ __forceinline__ void tb_release(uint32_t tmem, int warp)
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                     : "memory");
    }
}

// Four bootstraps per CTA (one CTA per SM, 16 warps), 4 warps each, that
// share the constant operands and twiddles and otherwise run independently
// (barriers of 128 threads): one bootstrap's waits and memory phases are
// covered by the other three.  Gate slots run through all CTAs first, so a
// level of fewer than four bootstraps per SM spreads over the SMs.  Per CMux
// step of a bootstrap:
//   digits     warp wr: half of polynomial wr >> 1, both digits
//   products   one thread: V_0 (TMEM, 96 columns)
//   pass 1, 2  warp s (the TMEM lanes it can read): digit row s modulo q_0,
//              while V_1 runs once every warp has read V_0; then modulo q_1
//   pointwise, inverse, CRT as warp (p, h)
// Bound: the integer multiplies (IMAD 2, IMAD.HI and IMAD.WIDE 4 cycles of the
// one pipe that has them): 4.1K cycles of that pipe per warp and step, busy 80 %
// of the time.  608 bootstraps: 5.36 ms (113K/s); with the key switch 5.56 ms when
// that took 0.22, against 7.85 ms with both passes as unsigned butterflies.  The same first
// pass in CTAs whose bootstraps run in lockstep took 7.4-8.1 ms: every wait and
// table load stood alone.  The inverse's last pass on the tensor pipe too
// (three limbs of each residue, CRT from the sums): 6.4 ms; the products take
// 1.6K cycles of a bootstrap's step, its splitting and sums as many
// instructions as the butterflies.
__global__ void __launch_bounds__(512, 1) k_blind_rotate_tc(const BrArgs A)
{
    constexpr int T = 128;
    extern __shared__ uint4 smem_raw[];
    TbSmem *all = reinterpret_cast<TbSmem *>(smem_raw);
    TbOps &O = *reinterpret_cast<TbOps *>(all + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bi = warp / 4, wr = warp % 4, tb = tid % T;
    TbSmem &S = all[bi];
    const int lane_brv = brv5(lane);
    const int n = A.keys.n;
    const int p = wr >> 1, h = wr & 1;
    const Prime pr((uint32_t)h);

    tb_setup(A, O, tid, kTbTw);
    const uint32_t tmem = O.tmem;
    const uint32_t tl = tmem + ((uint32_t)(32 * wr) << 16);   // this warp's TMEM lanes
    const uint32_t acc_cols = tmem + (uint32_t)(bi * kTbCols);
    const uint32_t dig_op = br_saddr(&S.fwd[1][0][0]);
    const int2 *tw_inv = reinterpret_cast<const int2 *>(A.keys.tb_op + 2 * kTbOpBytes / 16) +
                         1024 * h + lane;
    uint32_t phase = 0;   // products waited for (the same in the bootstrap's threads)

    for (long g = A.first + blockIdx.x + (long)bi * gridDim.x; g < A.count && !O.abort[bi];
         g += 4L * gridDim.x) {
        const bool active = br_prologue<T>(A, g, tb, S.abar, true);
        boot_sync(bi);
        br_acc_init<T>(A, S.acc, S.abar[n], tb);
        boot_sync(bi);

        for (int i = 0; i < n; ++i) {
            const int a = S.abar[i];
            if (a == 0)
                continue;   // X^0 acc - acc = 0: nothing changes
            tb_digits(S.acc[p], reinterpret_cast<uint8_t *>(&S.fwd[1][0][0]), p, h, a, lane);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            boot_sync(bi);
            if (tb == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                tb_mma(acc_cols, dig_op, O, 0,
                       phase + 1 == (uint32_t)A.keys.br_stall ? &O.spare[bi] : &O.bar[bi]);
            }
            int32_t x[32];
            const uint4 *bki = A.keys.bk_ntt + (((long)i * 2 + p) * 2 + h) * 1024;
            // unrolled: with the prime known, twiddles are operands in the constant
            // bank and not loaded (608 gates 6.10 -> 5.74 ms)
#pragma unroll
            for (int ph = 0; ph < 2; ++ph) {
                const Prime pq((uint32_t)ph);
                uint32_t *sl = S.fwd[ph][wr];
                if (!bk_wait(&O.bar[bi], phase & 1)) {
                    O.abort[bi] = 1;
                    atomicOr(A.status, kErrTimeout);
                }
                ++phase;
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                tb_combine(tl + bi * kTbCols, tl + kTbTw + 64 * ph, sl + lane * kRowV, pq);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                if (ph == 0) {
                    // V_1 overwrites V_0 once the four warps have read it (where a
                    // wait for V_0 ran out, too: both are waited for at the end)
                    if (wr == 0) {
                        asm volatile("bar.sync %0, 128;" ::"r"(5 + bi) : "memory");
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        if (lane == 0)
                            tb_mma(acc_cols, dig_op, O, 1, &O.bar[bi]);
                    } else {
                        asm volatile("bar.arrive %0, 128;" ::"r"(5 + bi) : "memory");
                    }
                }
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 32; ++r)
                    x[r] = (int32_t)sl[r * kRowV + lane];   // lane k1 reads slot[i1][k1]
                __syncwarp();
                pass32_signed<false>(x, pq);
                store_vec(sl, x, lane);
            }
            uint4 kv[4];
            key_ld4(kv, bki, 0, lane);
            boot_sync(bi);
            pointwise_v(x, S.fwd[h], kv, bki, lane, pr);
            inv_ntt_v(x, S.fwd[0][wr], lane, lane_brv, tw_inv, pr, bi);
            store_vec(S.fwd[1][wr], x, lane);
            boot_sync(bi);
            crt_rows_v<16>(S.acc[p], S.fwd[1][p * 2 + 0], S.fwd[1][p * 2 + 1], 16 * h, lane);
            boot_sync(bi);
            if (O.abort[bi])
                break;
        }

        if (active && !O.abort[bi])
            br_extract<T>(A, g, S.acc, tb);
        boot_sync(bi);
    }
    // after a wait that ran out: the step's two products get a bounded time to
    // finish, in their order, before TMEM is freed (an even phase and an odd one; a
    // wait for a phase that is not the barrier's current one would end at once)
    if (O.abort[bi] && tb == 0) {
        (void)bk_wait(&O.bar[bi], phase & 1);
        (void)bk_wait(&O.bar[bi], (phase + 1) & 1);
    }
    tb_release(tmem, warp);
}

// ---------------------------------------------------------------------
// One bootstrap on the 16 warps of a CTA, for levels of at most one
// bootstrap per SM, whose time is the length of a CMux step.
// ---------------------------------------------------------------------
//
// The arithmetic of k_blind_rotate_tc with every phase spread over all 16
// warps (q, z) = (warp % 4, warp / 4); a 32-point pass is cut into register
// blocks that exchange through shared memory:
//   digits      polynomial q >> 1, 4 coefficients per lane
//   first pass  digit row q (the TMEM lanes it can read), prime z >> 1,
//               outputs 16 (z & 1) ..; both primes' products run at once
//   second pass the same row and prime, output half z & 1
//   pointwise, inverse passes   (p, h) = (q >> 1, q & 1), 8 registers; after
//               three stages the four warps of a (p, h) exchange and run the
//               last two on two quadruples
//   CRT         polynomial p, 4 coefficients per lane (kept in registers: the
//               same as the digits')
// The key of a step is loaded behind the fence of its digits (which would wait
// for it), the inverse's twiddles once.
// Bound: the integer multiplies (their pipe is busy 60 % of a step's 7.9K cycles)
// and the waits between nine barriers.  One gate 2.43 -> 2.05 ms, 152 gates
// 2.65 -> 2.09 ms against a shape of 8 warps whose first pass was butterflies.
struct WideSmem {
    uint32_t acc[2][kN];            // TLWE accumulator (a(X), b(X))
    uint8_t dig[128 * 32 * 2];      // digit operand
    uint32_t slot[2][4][kSlotV];    // transposes of the forward transforms
    uint32_t fwd[2][4][kN];         // forward outputs [prime][digit row] (vec_word)
    uint32_t ex[4][kN];             // exchange of the inverse passes [p * 2 + h]
    uint32_t tr[4][kSlotV];         // transposes of the inverse transforms
    uint32_t res[4][kN];            // residues [p * 2 + h][reg*32+lane]
    uint16_t abar[kLweStride];
};

template <int T>
__device__ __forceinline__ void warps_sync(int bar)
{
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(T) : "memory");
}

// Half K (registers 16 K .. 16 K + 15) of ct32<true>: the first stage reads
// all 32 inputs, the others stay inside the half.
template <int K>
__device__ __forceinline__ void ct32_cyc_half(uint32_t (&y)[32], const uint32_t *row, int stride,
                                              const Prime &pr)
{
    constexpr LazyPlan PL = kPlanFwdD;
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) {
        const LazyStep &L = PL.st[0][jj];
        const uint32_t u = lazy_reduce_n(row[jj * stride], L.ru, L.nru, pr);
        const uint32_t v = lazy_reduce_n(row[(jj + 16) * stride], L.rv, L.nrv, pr);
        y[16 * K + jj] = K == 0 ? u + v : u - v + pr.kq(L.off);
    }
#pragma unroll
    for (int s = 1; s < 5; ++s) {
        const int m = 1 << s, ln = 16 >> s;
#pragma unroll
        for (int g = K * m / 2; g < (K + 1) * m / 2; ++g) {
            const uint32_t w = c_ntt.zd[pr.P][m + g][0];
            const uint32_t wp = c_ntt.zd[pr.P][m + g][1];
#pragma unroll
            for (int jj = 0; jj < ln; ++jj) {
                const int j = 2 * g * ln + jj;
                const LazyStep &L = PL.st[s][g * ln + jj];
                const uint32_t u = lazy_reduce_n(y[j], L.ru, L.nru, pr);
                const uint32_t t = g == 0 ? lazy_reduce_n(y[j + ln], L.rv, L.nrv, pr)
                                          : mul_shoup(y[j + ln], w, wp, pr.q);
                y[j] = u + t;
                y[j + ln] = u - t + pr.kq(L.off);
            }
        }
    }
#pragma unroll
    for (int r = 16 * K; r < 16 * K + 16; ++r)
        y[r] = lazy_reduce_n(y[r], PL.fin[r], PL.nfin[r], pr);
}

// The first three stages of a 32-point Gentleman-Sande pass (the inverse of ct32,
// 32 times) on the register block 8 z .. 8 z + 7;
// inputs [0, 2q).  The bounds by position are 16, 8, 4, 4, 2, 2, 2, 2 (times
// q), the first two reduced to `fin` (a group whose twiddle is 1 takes its
// product too, so that the four warps run the same code).
template <bool CYC>
__device__ __forceinline__ void gs32_block(uint32_t (&x)[8], int z, const Prime &pr)
{
    const uint32_t(*tb)[2] = CYC ? c_ntt.izd[pr.P] : c_ntt.iza[pr.P];
#pragma unroll
    for (int s = 4; s >= 2; --s) {
        const int m = 1 << s, ln = 16 >> s;
#pragma unroll
        for (int gl = 0; gl < m / 4; ++gl) {
            const uint32_t w = tb[m + z * (m / 4) + gl][0], wp = tb[m + z * (m / 4) + gl][1];
#pragma unroll
            for (int jj = 0; jj < ln; ++jj) {
                const int j = 2 * gl * ln + jj;
                const uint32_t u = x[j], v = x[j + ln];
                x[j] = u + v;
                x[j + ln] = mul_shoup(u - v + pr.kq(2 * ln), w, wp, pr.q);
            }
        }
    }
    x[0] = csub(x[0], pr.kq(8));
    if (!CYC) {
        x[0] = csub(x[0], pr.kq(4));
        x[1] = csub(x[1], pr.kq(4));
    }
}

// The last two stages of that pass on registers jj, jj + 8, jj + 16, jj + 24.
// CYC: inputs below 8q, results below 32q (into a Shoup product); else inputs
// below 4q, results below 8q.
template <bool CYC>
__device__ __forceinline__ void gs32_last(uint32_t &a0, uint32_t &a1, uint32_t &a2, uint32_t &a3,
                                          const Prime &pr)
{
    const uint32_t(*tb)[2] = CYC ? c_ntt.izd[pr.P] : c_ntt.iza[pr.P];
    constexpr int B = CYC ? 8 : 4;
    const uint32_t t0 = a0 + a1, t2 = a2 + a3;
    uint32_t t1 = a0 - a1 + pr.kq(B);
    if (!CYC)
        t1 = mul_shoup(t1, tb[2][0], tb[2][1], pr.q);
    const uint32_t t3 = mul_shoup(a2 - a3 + pr.kq(B), tb[3][0], tb[3][1], pr.q);
    a0 = t0 + t2;
    a1 = t1 + t3;
    a2 = t0 - t2 + pr.kq(2 * B);
    a3 = t1 - t3 + pr.kq(2);
    if (!CYC) {
        a0 = csub(a0, pr.kq(8));
        a2 = mul_shoup(a2, tb[1][0], tb[1][1], pr.q);
        a3 = mul_shoup(a3, tb[1][0], tb[1][1], pr.q);
    }
}

// One 32-point inverse pass of a (p, h): x holds registers 8 z + e, on
// return registers 2 z + (e & 1) + 8 (e >> 1).
template <bool CYC>
__device__ __forceinline__ void gs32_four(uint32_t (&x)[8], uint32_t *ex, int z, int lane, int bar,
                                          const Prime &pr)
{
    gs32_block<CYC>(x, z, pr);
#pragma unroll
    for (int e = 0; e < 8; ++e)
        ex[(8 * z + e) * 32 + lane] = x[e];
    warps_sync<128>(bar);
#pragma unroll
    for (int e = 0; e < 8; ++e)
        x[e] = ex[(2 * z + (e & 1) + 8 * (e >> 1)) * 32 + lane];
    gs32_last<CYC>(x[0], x[2], x[4], x[6], pr);
    gs32_last<CYC>(x[1], x[3], x[5], x[7], pr);
}

// Both digits of the thread's four coefficients lane + 32 (c_lo + e) of one
// polynomial, 8 bytes each at o (level 1) and 32 rows on (level 2).
__device__ __forceinline__ void wide_digits(const uint32_t *ac, const uint32_t (&own)[4], uint8_t *o,
                                            int c_lo, int a, int lane)
{
    uint32_t u[4], d0[2], d1[2];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int idx = (lane + 32 * (c_lo + e) - a) & (2 * kN - 1);
        uint32_t v = ac[idx & (kN - 1)];
        v = idx >= kN ? 0u - v : v;
        u[e] = v - own[e] + kDecompOffset;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
        tb_digit2(u[2 * e], u[2 * e + 1], d0[e], d1[e]);
    *reinterpret_cast<uint2 *>(o) = make_uint2(d0[0], d0[1]);
    *reinterpret_cast<uint2 *>(o + 32 * 16) = make_uint2(d1[0], d1[1]);
}

// Inverse transform by four warps (block z of each), see gs32_four.
__device__ __forceinline__ void wide_inverse(uint32_t (&x)[8], uint32_t *ex, uint32_t *tr,
                                             const uint2 (&tw)[8], int z, int lane, int lane_brv,
                                             int bar, const Prime &pr)
{
    gs32_four<true>(x, ex, z, lane, bar, pr);
    uint32_t *wr = tr + lane_brv;
#pragma unroll
    for (int e = 0; e < 8; ++e)   // lane k1, i1 -> row i1
        wr[(2 * z + (e & 1) + 8 * (e >> 1)) * kRowV] = mul_shoup(x[e], tw[e].x, tw[e].y, pr.q);
    warps_sync<128>(bar);
    const uint32_t *rd = tr + lane * kRowV + 8 * z;
    const uint4 v0 = *reinterpret_cast<const uint4 *>(rd);
    const uint4 v1 = *reinterpret_cast<const uint4 *>(rd + 4);
    x[0] = v0.x, x[1] = v0.y, x[2] = v0.z, x[3] = v0.w;
    x[4] = v1.x, x[5] = v1.y, x[6] = v1.z, x[7] = v1.w;
    gs32_four<false>(x, ex, z, lane, bar, pr);
}

__device__ __forceinline__ void wide_crt(uint32_t *ac, uint32_t (&own)[4], const uint32_t *x0,
                                         const uint32_t *x1, int c_lo, int lane)
{
    const int32_t cc = c_ntt.crt_c, cp = c_ntt.crt_cp;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = (c_lo + e) * 32 + lane;
        own[e] += crt_lift(x0[k], x1[k], cc, cp);
        ac[k] = own[e];
    }
}

__global__ void __launch_bounds__(512, 1) k_blind_rotate_wide(const BrArgs A)
{
    extern __shared__ uint4 smem_raw[];
    WideSmem &S = *reinterpret_cast<WideSmem *>(smem_raw);
    TbOps &O = *reinterpret_cast<TbOps *>(&S + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, z = warp >> 2, p = q >> 1, h = q & 1, hz = z & 1;
    const int lane_brv = brv5(lane);
    const int n = A.keys.n;
    const Prime pr((uint32_t)h), pf((uint32_t)(z >> 1));
    tb_setup(A, O, tid, 2 * kTbCols);
    const uint32_t tmem = O.tmem;
    const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
    const int c_lo = 8 * z + 4 * h;   // this thread's coefficients lane + 32 (c_lo + e)
    uint2 tw[8];
#pragma unroll
    for (int e = 0; e < 8; ++e)
        tw[e] = __ldg(A.keys.twb + ((h * 2 + 1) * 32 + 2 * z + (e & 1) + 8 * (e >> 1)) * 32 + lane);
    uint32_t phase = 0;   // executed CMux steps
    const uint32_t stall = (uint32_t)A.keys.br_stall;   // test hook: V_1 of this step (from 1)

    for (long g = A.first + blockIdx.x; g < A.count && !O.abort[0]; g += gridDim.x) {
        const bool active = br_prologue<512>(A, g, tid, S.abar, true);
        __syncthreads();
        br_acc_init<512>(A, S.acc, S.abar[n], tid);
        __syncthreads();
        uint32_t own[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            own[e] = S.acc[p][(c_lo + e) * 32 + lane];

        for (int i = 0; i < n; ++i) {
            const int a = S.abar[i];
            if (a == 0)
                continue;   // X^0 acc - acc = 0: nothing changes
            wide_digits(S.acc[p], own, S.dig + z * 2048 + (64 * p + lane) * 16 + 8 * h, c_lo, a,
                        lane);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                tb_mma(tmem, br_saddr(S.dig), O, 0, &O.bar[0]);
                tb_mma(tmem + kTbCols, br_saddr(S.dig), O, 1,
                       phase + 1 == stall ? &O.spare[1] : &O.bar[1]);
            }
            uint4 kv[8];
            const uint4 *bki = A.keys.bk_ntt + (((long)i * 2 + p) * 2 + h) * 1024 + 8 * z * 32 + lane;
#pragma unroll
            for (int e = 0; e < 8; ++e)
                kv[e] = __ldg(bki + e * 32);
            if (!bk_wait(&O.bar[pf.P], phase & 1)) {
                O.abort[0] = 1;
                atomicOr(A.status, kErrTimeout);
            }
            ++phase;
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t *sl = S.slot[pf.P][q];
            tb_combine(tl + kTbCols * pf.P, tl + 2 * kTbCols + 64 * pf.P, sl + lane * kRowV, pf,
                       16 * hz, 16 * hz + 16);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            warps_sync<64>(1 + 2 * q + (z >> 1));
            {
                uint32_t y[32];
                uint32_t *out = S.fwd[pf.P][q];
                if (hz == 0) {
                    ct32_cyc_half<0>(y, sl + lane, kRowV, pf);
#pragma unroll
                    for (int r = 0; r < 16; r += 4)
                        *reinterpret_cast<uint4 *>(out + vec_word(r, lane)) =
                            make_uint4(y[r], y[r + 1], y[r + 2], y[r + 3]);
                } else {
                    ct32_cyc_half<1>(y, sl + lane, kRowV, pf);
#pragma unroll
                    for (int r = 16; r < 32; r += 4)
                        *reinterpret_cast<uint4 *>(out + vec_word(r, lane)) =
                            make_uint4(y[r], y[r + 1], y[r + 2], y[r + 3]);
                }
            }
            __syncthreads();
            int32_t y[8];
            uint32_t x[8];
            pointwise_4(y, 0, S.fwd[h], 2 * z, kv, lane, pr);
            pointwise_4(y, 4, S.fwd[h], 2 * z + 1, kv, lane, pr);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                x[e] = (uint32_t)y[e] + pr.q;
            wide_inverse(x, S.ex[q], S.tr[q], tw, z, lane, lane_brv, 9 + q, pr);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                S.res[q][(2 * z + (e & 1) + 8 * (e >> 1)) * 32 + lane] = x[e];
            warps_sync<256>(13 + p);
            wide_crt(S.acc[p], own, S.res[2 * p], S.res[2 * p + 1], c_lo, lane);
            warps_sync<256>(13 + p);
            if (O.abort[0])
                break;
        }

        __syncthreads();
        if (active && !O.abort[0])
            br_extract<512>(A, g, S.acc, tid);
        __syncthreads();
    }
    // after a wait that ran out: products still in flight get a bounded time
    // to finish before TMEM is freed
    if (O.abort[0] && tid == 0) {
        (void)bk_wait(&O.bar[0], (phase - 1) & 1);
        if (phase == stall)
            (void)bk_wait(&O.spare[1], 0);
        else
            (void)bk_wait(&O.bar[1], (phase - 1) & 1);
    }
    tb_release(tmem, warp);
}

// ---------------------------------------------------------------------
// One bootstrap on a cluster of two CTAs (two SMs): CTA h works modulo
// prime h for the whole CMux and the two exchange their inverse-transform
// residues through distributed shared memory for the CRT.  For levels of at
// most one bootstrap per two SMs, whose time is the length of a CMux step.
// ---------------------------------------------------------------------
//
// As k_blind_rotate_wide, with the phases of one prime spread over a CTA's 16
// warps (q, z):
//   digits, CRT   as there (both CTAs hold and update the whole accumulator)
//   first pass    digit row q, outputs 8 z ..
//   second pass   digit row q, registers 8 z ..
//   pointwise, inverse passes   warps z < 2: polynomial z, 8 registers
// Residues go to both CTAs by asynchronous stores that count on the receiver's
// barrier, so that no cluster barrier (and its memory fences) stands in a
// step.  Their buffers alternate by executed CMux: one is rewritten two steps
// after it was read, and the sender of the later step has waited for what the
// reader sent in the step between.  Control flow is the same in both CTAs (same
// gate, same abar), so each step's stores are sent by both.
// A CTA whose wait runs out executes one more step, without waiting, and ends; its
// partner's next wait for residues then runs out, and it ends the same way.  Both
// meet before they end, and each gives what is still on its way into it a bounded
// time (pair_drain).  (The flag tested at other places of the step: one gate 1.64 to
// 1.67 ms, so 1.61.)
// Bound: the chain of a step (6.3K cycles, the multiply pipe busy half of them,
// seven barriers and two waits).  One gate 1.61 ms against 2.06 ms on one CTA;
// the shape it replaces (8 warps per CTA, butterflies in the first pass, key
// staged by bulk copies) took 2.53 ms.
struct PairSmem {
    uint32_t acc[2][kN];            // TLWE accumulator (the same in both CTAs)
    uint8_t dig[128 * 32 * 2];      // digit operand
    uint32_t slot[4][kSlotV];       // transposes of the forward transforms
    uint32_t fwd[4][kN];            // forward outputs [digit row] (vec_word)
    uint32_t ex[2][kN];             // exchange of the inverse passes [p]
    uint32_t tr[2][kSlotV];         // transposes of the inverse transforms
    uint32_t res[2][2][2][kN];      // residues [buffer][prime][p] (pair_word)
    unsigned long long got[2];      // residues of both CTAs have arrived [buffer]
    uint16_t abar[kLweStride];
};
constexpr uint32_t kPairBytes = 2 * 2 * kN * sizeof(uint32_t);   // residues of one step

// Word of register r = 2 q + o + 8 b of a lane in a residue row: registers of
// the producer's (q, b >> 1) are 16 bytes, the reader's r, r + 1 8 bytes.
__host__ __device__ constexpr int pair_word(int r, int lane)
{
    return ((((r >> 4) * 4 + ((r >> 1) & 3)) * 32 + lane) * 4) + ((r >> 3) & 1) * 2 + (r & 1);
}

// Four words to shared memory of a CTA of the cluster (an address of the
// shared::cluster window); their arrival counts on that CTA's barrier `bar`.
__device__ __forceinline__ void pair_send(uint32_t to, uint32_t a, uint32_t b, uint32_t c, uint32_t d,
                                          uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], "
                 "{%1, %2, %3, %4}, [%5];" ::"r"(to),
                 "r"(a), "r"(b), "r"(c), "r"(d), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ uint32_t pair_addr(const void *p, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(br_saddr(p)), "r"(rank));
    return r;
}

// Registers 8 z .. 8 z + 7 of ct32<true> (groups whose twiddle is 1 take their
// product too, so that the four warps run the same code): inputs [0, 2q),
// each stage adds at most 2q, outputs reduced from 12q to [0, 8q).
__device__ __forceinline__ void ct32_cyc_block(uint32_t (&y)[8], const uint32_t *row, int stride,
                                               int z, const Prime &pr)
{
    const uint32_t(*tb)[2] = c_ntt.zd[pr.P];
    const int k = z >> 1;
    const uint32_t m0 = k ? ~0u : 0u, m1 = (z & 1) ? ~0u : 0u;
    const uint32_t o0 = k ? pr.q2 + 1u : 0u, o1 = (z & 1) ? pr.q2 + 1u : 0u;
    const uint32_t w1 = tb[2 + k][0], wp1 = tb[2 + k][1];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        // stage 0: u + v, or u - v + 2q; then stage 1 the same way
        const uint32_t u = row[e * stride] + (row[(16 + e) * stride] ^ m0) + o0;
        const uint32_t v = row[(8 + e) * stride] + (row[(24 + e) * stride] ^ m0) + o0;
        y[e] = u + (mul_shoup(v, w1, wp1, pr.q) ^ m1) + o1;
    }
#pragma unroll
    for (int s = 2; s < 5; ++s) {
        const int m = 1 << s, ln = 16 >> s;
#pragma unroll
        for (int gl = 0; gl < m / 4; ++gl) {
            const uint32_t w = tb[m + z * (m / 4) + gl][0], wp = tb[m + z * (m / 4) + gl][1];
#pragma unroll
            for (int jj = 0; jj < ln; ++jj) {
                const int j = 2 * gl * ln + jj;
                const uint32_t u = y[j], t = mul_shoup(y[j + ln], w, wp, pr.q);
                y[j] = u + t;
                y[j + ln] = u - t + pr.q2;
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e)
        y[e] = csub(y[e], pr.kq(8));
}

// After a wait that ran out, one thread, behind the cluster's last barrier (both
// CTAs have issued all they will): products and residues still on their way get a
// bounded time before TMEM and shared memory are freed.  `steps` were executed
// here; the partner's wait for the residues of the next one runs out, and it sends
// its own of that one and of one more.
__device__ __forceinline__ void pair_drain(PairSmem &S, TbOps &O, uint32_t steps)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     br_saddr(&O.spare[0]))
                 : "memory");
    (void)bk_wait(&O.spare[0], 0);
    for (uint32_t s = steps < 2 ? 0 : steps - 2; s < steps + 2; ++s) {
        unsigned long long *bar = &S.got[s & 1];
        if (s >= steps)   // the step has not posted its bytes: the partner's half
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(br_saddr(bar)),
                         "r"(kPairBytes / 2)
                         : "memory");
        if (!bk_wait(bar, (s >> 1) & 1))
            return;   // the partner has sent nothing further
    }
}

__global__ void __launch_bounds__(512, 1) k_blind_rotate_pair(const BrArgs A)
{
    extern __shared__ uint4 smem_raw[];
    PairSmem &S = *reinterpret_cast<PairSmem *>(smem_raw);
    TbOps &O = *reinterpret_cast<TbOps *>(&S + 1);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, z = warp >> 2, p = q >> 1;
    const int lane_brv = brv5(lane);
    const int n = A.keys.n;
    const Prime pr((uint32_t)rank);
    const long nclusters = gridDim.x / 2, cid = blockIdx.x / 2;
    tb_setup(A, O, tid, 2 * kTbCols);
    const uint32_t tmem = O.tmem;
    const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
    const int c_lo = 8 * z + 4 * (q & 1);   // this thread's coefficients lane + 32 (c_lo + e)
    // inverse roles of the warps z < 2: polynomial z, registers 8 q ..
    uint2 tw[8];
#pragma unroll
    for (int e = 0; e < 8; ++e)
        tw[e] = __ldg(A.keys.twb + ((rank * 2 + 1) * 32 + 2 * q + (e & 1) + 8 * (e >> 1)) * 32 + lane);
    const uint32_t res_at[2] = {pair_addr(S.res, rank), pair_addr(S.res, rank ^ 1)};
    const uint32_t got_at[2] = {pair_addr(S.got, rank), pair_addr(S.got, rank ^ 1)};
    uint32_t phase = 0;   // executed CMux steps
    if (tid < 2) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(br_saddr(&S.got[tid])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cl.sync();   // the partner's shared memory and barriers are there

    for (long g = A.first + cid; g < A.count && !O.abort[0]; g += nclusters) {
        const bool active = br_prologue<512>(A, g, tid, S.abar, rank == 0);
        if (tid == 0 && rank == 1 && g + 1 == A.keys.br_stall && !(phase & 1)) {
            // test hook: two products complete a phase from here on (phases restart
            // at 0), so the wait for the next one runs out
            asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(br_saddr(&O.bar[0])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;" ::"r"(br_saddr(&O.bar[0])) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();
        br_acc_init<512>(A, S.acc, S.abar[n], tid);
        __syncthreads();
        uint32_t own[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            own[e] = S.acc[p][(c_lo + e) * 32 + lane];

        for (int i = 0; i < n; ++i) {
            const int a = S.abar[i];
            const uint32_t left = (uint32_t)O.abort[0] - 1u;
            if (a == 0)
                continue;   // X^0 acc - acc = 0: nothing changes
            // a wait ran out in the step before the last one: every thread finds
            // that here, where one of the last step may not be seen by all
            if (left < phase - 1u)
                break;
            const uint32_t use = phase++;
            const int par = use & 1;
            wide_digits(S.acc[p], own, S.dig + z * 2048 + (64 * p + lane) * 16 + 8 * (q & 1), c_lo,
                        a, lane);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                tb_mma(tmem, br_saddr(S.dig), O, rank, &O.bar[0]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                                 br_saddr(&S.got[par])),
                             "r"(kPairBytes)
                             : "memory");
            }
            uint4 kv[8];
            if (z < 2) {
                const uint4 *bki = A.keys.bk_ntt + (((long)i * 2 + z) * 2 + rank) * 1024 +
                                   8 * q * 32 + lane;
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    kv[e] = __ldg(bki + e * 32);
            }
            if (!O.abort[0] && !bk_wait(&O.bar[0], use & 1)) {
                O.abort[0] = (int)phase;   // wait no more; the status word has it
                atomicOr(A.status, kErrTimeout);
            }
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t *sl = S.slot[q];
            tb_combine(tl, tl + 2 * kTbCols + 64 * rank, sl + lane * kRowV, pr, 8 * z, 8 * z + 8);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            warps_sync<128>(1 + q);
            uint32_t x[8];
            ct32_cyc_block(x, sl + lane, kRowV, z, pr);
            uint32_t *out = S.fwd[q] + vec_word(8 * z, lane);
            *reinterpret_cast<uint4 *>(out) = make_uint4(x[0], x[1], x[2], x[3]);
            *reinterpret_cast<uint4 *>(out + vec_word(4, 0)) = make_uint4(x[4], x[5], x[6], x[7]);
            __syncthreads();
            if (z < 2) {
                int32_t y[8];
                pointwise_4(y, 0, S.fwd, 2 * q, kv, lane, pr);
                pointwise_4(y, 4, S.fwd, 2 * q + 1, kv, lane, pr);
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    x[e] = (uint32_t)y[e] + pr.q;
                wide_inverse(x, S.ex[z], S.tr[z], tw, q, lane, lane_brv, 9 + z, pr);
                const uint32_t at = (((par * 2 + rank) * 2 + z) * kN + pair_word(2 * q, lane)) * 4;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    pair_send(res_at[c] + at, x[0], x[1], x[2], x[3], got_at[c] + 8 * par);
                    pair_send(res_at[c] + at + 4 * pair_word(16, 0), x[4], x[5], x[6], x[7],
                              got_at[c] + 8 * par);
                }
            }
            if (!O.abort[0] && !bk_wait(&S.got[par], (use >> 1) & 1)) {
                O.abort[0] = (int)phase;
                atomicOr(A.status, kErrTimeout);
            }
            {
                const int32_t cc = c_ntt.crt_c, cp = c_ntt.crt_cp;
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                    const int w = pair_word(c_lo + e, lane);
                    const uint2 v0 = *reinterpret_cast<const uint2 *>(&S.res[par][0][p][w]);
                    const uint2 v1 = *reinterpret_cast<const uint2 *>(&S.res[par][1][p][w]);
                    own[e] += crt_lift(v0.x, v1.x, cc, cp);
                    own[e + 1] += crt_lift(v0.y, v1.y, cc, cp);
                    S.acc[p][(c_lo + e) * 32 + lane] = own[e];
                    S.acc[p][(c_lo + e + 1) * 32 + lane] = own[e + 1];
                }
            }
            warps_sync<256>(13 + p);
        }
        __syncthreads();
        if (active && rank == 0 && !O.abort[0])
            br_extract<512>(A, g, S.acc, tid);
        __syncthreads();
    }
    cl.sync();   // neither CTA ends while the other may write to it
    if (O.abort[0] && tid == 0)
        pair_drain(S, O, phase);
    tb_release(tmem, warp);
}

// ---------------------------------------------------------------------
// Host side: constants and launchers
// ---------------------------------------------------------------------

static uint64_t mulmod(uint64_t a, uint64_t b, uint64_t m) { return (a * b) % m; }

static uint64_t powmod(uint64_t b, uint64_t e, uint64_t m)
{
    uint64_t r = 1;
    b %= m;
    while (e) {
        if (e & 1)
            r = mulmod(r, b, m);
        b = mulmod(b, b, m);
        e >>= 1;
    }
    return r;
}

static uint32_t shoup_of(uint32_t w, uint32_t q) { return (uint32_t)(((uint64_t)w << 32) / q); }

// A primitive 2N-th root of unity: psi^N = -1.
static uint32_t find_psi(uint32_t q)
{
    for (uint64_t x = 2; x < 100000; ++x) {
        uint64_t psi = powmod(x, (q - 1) / (2 * kN), q);
        if (powmod(psi, kN, q) == q - 1)
            return (uint32_t)psi;
    }
    return 0;
}

static int bitrev(int k, int bits)
{
    int r = 0;
    for (int b = 0; b < bits; ++b)
        if (k & (1 << b))
            r |= 1 << (bits - 1 - b);
    return r;
}

// Centred representative of v mod q.
static int64_t centred(int64_t v, int64_t q)
{
    v %= q;
    if (v < 0)
        v += q;
    return v > q / 2 ? v - q : v;
}

static int32_t signed_shoup_of(int32_t w, uint32_t q)
{
    return (int32_t)std::llround((double)w * 0x1p32 / (double)q);
}

// Constant operand of the tensor-pipe first pass, op[prime] in its
// shared-memory order.  Returns false if a bound the kernel relies on does
// not hold.
static bool build_tb_operand(uint16_t *op)
{
    const uint32_t qs[2] = {kQ0, kQ1};
    for (int P = 0; P < 2; ++P) {
        const int64_t q = qs[P];
        const uint64_t psi = find_psi(qs[P]);
        double smax[32][3] = {};   // largest |sum| of column (k1, limb)
        for (int k1 = 0; k1 < 32; ++k1)
            for (int i2 = 0; i2 < 32; ++i2) {
                int64_t v = centred((int64_t)powmod(psi, 32ull * (2 * k1 + 1) * i2, q), q);
                for (int l = 0; l < 3; ++l) {
                    const int64_t d = l < 2 ? ((v + (256 + (1 << 30))) & 511) - 256 : v;
                    v = (v - d) / 512;
                    if (d < -256 || d > 256)
                        return false;
                    smax[k1][l] += 512.0 * (double)(d < 0 ? -d : d);
                    // column 24 (k1 / 8) + 8 l + k1 % 8, core matrices [i2 / 8][column / 8]
                    const int col = (k1 / 8) * 24 + 8 * l + k1 % 8;
                    const __half hv = __float2half((float)d);
                    uint16_t bits;
                    std::memcpy(&bits, &hv, 2);
                    op[P * (kTbOpBytes / 2) +
                       (((i2 / 8) * (kTbCols / 8) + col / 8) * 8 + col % 8) * 8 + i2 % 8] = bits;
                }
            }
        for (int k1 = 0; k1 < 32; ++k1)
            for (int l = 0; l < 3; ++l)
                if (smax[k1][l] >= 0x1p22)
                    return false;
    }
    return true;
}

// Builds the NTT constants into c_ntt (current device) and the stage-B
// twiddle table into twb_dev ([2][2][32][32] uint2), and the constant operand
// of the tensor-pipe first pass (kTbOpBytes per prime) and the signed inverse
// twiddles ([2][32][32] int2) into tb_op_dev.
cudaError_t upload_ntt_constants(uint2 *twb_dev, uint4 *tb_op_dev, cudaStream_t stream)
{
    NttConst C;
    std::memset(&C, 0, sizeof(C));
    std::vector<uint2> twb(2 * 2 * 32 * 32);
    std::vector<uint16_t> op(kTbDevBytes / 2);
    int2 *tws = reinterpret_cast<int2 *>(op.data() + kTbOpBytes);   // signed inverse twiddles
    const uint32_t qs[2] = {kQ0, kQ1};
    for (int P = 0; P < 2; ++P) {
        const uint32_t q = qs[P];
        const uint64_t psi = find_psi(q), ipsi = powmod(psi, q - 2, q);
        const uint64_t w64 = powmod(psi, 32, q), w32 = powmod(psi, 64, q);
        const uint64_t iw64 = powmod(w64, q - 2, q), iw32 = powmod(w32, q - 2, q);
        for (int k = 0; k < 32; ++k) {
            uint32_t a = (uint32_t)powmod(w64, brv5(k), q), ia = (uint32_t)powmod(iw64, brv5(k), q);
            C.za[P][k][0] = a;
            C.za[P][k][1] = shoup_of(a, q);
            C.iza[P][k][0] = ia;
            C.iza[P][k][1] = shoup_of(ia, q);
        }
        for (int m = 1; m <= 16; m <<= 1) {
            int lg = 0;
            while ((1 << lg) < m)
                ++lg;
            for (int g = 0; g < m; ++g) {
                const int e = bitrev(g, lg) * (16 / m);
                uint32_t d = (uint32_t)powmod(w32, e, q), id = (uint32_t)powmod(iw32, e, q);
                C.zd[P][m + g][0] = d;
                C.zd[P][m + g][1] = shoup_of(d, q);
                C.izd[P][m + g][0] = id;
                C.izd[P][m + g][1] = shoup_of(id, q);
            }
        }
        const auto put = [q](int32_t (&d)[2], uint64_t w) {
            d[0] = (int32_t)centred((int64_t)w, q);
            d[1] = signed_shoup_of(d[0], q);
        };
        for (int k = 1; k < 32; ++k) {
            put(C.zs[P][k], C.zd[P][k][0]);
            int ln = 16;
            while (ln > k)
                ln >>= 1;
            put(C.izs[P][k], powmod(iw32, (uint64_t)(k - ln) * (16 / ln), q));
            put(C.post[P][k], powmod(iw64, k, q));
        }
        C.one[P] = signed_shoup_of(1, q);
        for (int r = 0; r < 32; ++r)
            for (int l = 0; l < 32; ++l) {
                // forward: lane i1 = l, register r carries k1 = brv5(r)
                uint32_t f = (uint32_t)powmod(psi, (uint64_t)(2 * brv5(r) + 1) * l, q);
                // inverse: lane k1 = l, register i1 = r
                uint32_t iv = (uint32_t)powmod(ipsi, (uint64_t)(2 * l + 1) * r, q);
                twb[((P * 2 + 0) * 32 + r) * 32 + l] = make_uint2(f, shoup_of(f, q));
                twb[((P * 2 + 1) * 32 + r) * 32 + l] = make_uint2(iv, shoup_of(iv, q));
                const int32_t ivc = (int32_t)centred(iv, q);
                tws[(P * 32 + r) * 32 + l] = make_int2(ivc, signed_shoup_of(ivc, q));
            }
        // q^-1 mod 2^32 by Newton iteration
        uint32_t inv = q;
        for (int it = 0; it < 5; ++it)
            inv *= 2u - q * inv;
        C.q_inv[P] = inv;
        const uint64_t ninv = powmod(kN, q - 2, q);
        const uint32_t sc = (uint32_t)mulmod((((uint64_t)1 << 32) % q), ninv, q);
        C.bk_scale[P][0] = sc;
        C.bk_scale[P][1] = shoup_of(sc, q);
    }
    C.crt_c = (int32_t)centred((int64_t)powmod(kQ0, kQ1 - 2, kQ1), kQ1);
    C.crt_cp = (int32_t)std::llround((double)C.crt_c * 0x1p32 / (double)kQ1);
    cudaError_t e = cudaMemcpyToSymbolAsync(c_ntt, &C, sizeof(C), 0, cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess)
        return e;
    e = cudaMemcpyAsync(twb_dev, twb.data(), twb.size() * sizeof(uint2), cudaMemcpyHostToDevice,
                        stream);
    if (e != cudaSuccess)
        return e;
    if (!build_tb_operand(op.data()))
        return cudaErrorInvalidValue;
    e = cudaMemcpyAsync(tb_op_dev, op.data(), kTbDevBytes, cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess)
        return e;
    return cudaStreamSynchronize(stream);
}

cudaError_t launch_bk_to_ntt(const int32_t *bk_dev, uint32_t *bk_ntt, int n, const uint2 *twb,
                             cudaStream_t stream)
{
    const long tasks = (long)n * kRows * 2 * 2;
    k_bk_to_ntt<<<(unsigned)((tasks + 3) / 4), 128, 0, stream>>>(bk_dev, bk_ntt, n, twb);
    return cudaGetLastError();
}

// Shape of a launch: the forced or tuned code, else by batch size.
static bool br_shape_ok(int v)
{
    return v == 1 || v == 2 || v == 4 || v == kBrSplit || v == kBrPair || v == kBrStaged ||
           v == kBrStagedCtl || v == kBrSplitStaged || v == kBrFive || v == kBrPairStaged;
}

static int br_group(long count, int num_sms, int forced, const int8_t *tuned)
{
    if (br_shape_ok(forced))
        return forced;
    // at most one bootstrap per SM: 2.03 ms on 16 warps (152 gates) against
    // 2.75 ms for the throughput shape; 301 gates: 4.06 against 3.50 ms
    const int t = tuned[tune_bucket(count)];
    const int shape = br_shape_ok(t) ? t : count > num_sms ? 1 : kBrSplit;
    // at most one per two SMs: 1.60 ms on two CTAs (76 gates) against 2.03 ms on
    // one (a tuned choice stands for its bucket's widest level)
    return shape == kBrSplit && 2 * count <= num_sms ? kBrPair : shape;
}

static cudaError_t launch_tc(const BrArgs &A, unsigned blocks, int dev, cudaStream_t stream)
{
    constexpr int smem = 4 * (int)sizeof(TbSmem) + (int)sizeof(TbOps);
    static int prepared[64] = {0};
    if (dev >= 0 && dev < 64 && !prepared[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_blind_rotate_tc,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess)
            return e;
        prepared[dev] = 1;
    }
    BrArgs B = A;
    if (B.keys.br_stall)   // test hook: of the step's two products the first
        B.keys.br_stall = 2 * B.keys.br_stall - 1;
    k_blind_rotate_tc<<<blocks, 512, smem, stream>>>(B);
    return cudaGetLastError();
}

static cudaError_t launch_wide(const BrArgs &A, long sms, int dev, cudaStream_t stream)
{
    const long count = A.count - A.first;
    const unsigned blocks = (unsigned)(count < sms ? count : sms);
    constexpr int smem = (int)sizeof(WideSmem) + (int)sizeof(TbOps);
    static int prepared[64] = {0};
    if (dev >= 0 && dev < 64 && !prepared[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_blind_rotate_wide,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess)
            return e;
        prepared[dev] = 1;
    }
    k_blind_rotate_wide<<<blocks, 512, smem, stream>>>(A);
    return cudaGetLastError();
}

// One CTA per SM: `pairs` clusters at a time.
static cudaError_t launch_pair(const BrArgs &A, long pairs, int dev, cudaStream_t stream)
{
    constexpr int smem = (int)sizeof(PairSmem) + (int)sizeof(TbOps);
    static int prepared[64] = {0};
    if (dev >= 0 && dev < 64 && !prepared[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_blind_rotate_pair,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess)
            return e;
        prepared[dev] = 1;
    }
    cudaLaunchConfig_t cfg = {};
    const long count = A.count - A.first;
    cfg.gridDim = dim3((unsigned)(2 * (count < pairs ? count : pairs)));
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_blind_rotate_pair, A);
}

static cudaError_t launch_shape(const BrArgs &A, int shape, long nsm, int dev, cudaStream_t stream)
{
    const long count = A.count - A.first;
    if (shape == kBrPair || shape == kBrPairStaged)
        return launch_pair(A, nsm >= 2 ? nsm / 2 : 1, dev, stream);
    if (shape == kBrSplit || shape == kBrSplitStaged)
        return launch_wide(A, nsm, dev, stream);
    // the throughput shape (the other codes are accepted for saved tuning
    // files and options)
    return launch_tc(A, (unsigned)(count < nsm ? count : nsm), dev, stream);
}

// Gates at the end of a level that leave at most one bootstrap per SM for its
// last wave of the throughput shape: they run on the shapes of narrow levels
// instead, behind it (a wave of one per SM takes 2.6 - 2.75 ms there, 1.6 - 2.0
// ms on those; two per SM, 3.5 ms, would take two rounds).
static long br_tail(long count, long nsm, int forced, int shape)
{
    const long tail = count % (4 * nsm);
    return forced == 0 && shape == 1 && count > 4 * nsm && tail <= nsm ? tail : 0;
}

cudaError_t launch_blind_rotate(const DevKeys &keys, const uint8_t *ops, const int32_t *in_a,
                                const int32_t *idx_a, long rows_a, const int32_t *in_b,
                                const int32_t *idx_b, long rows_b, int32_t *big, long count,
                                uint32_t mu, uint32_t *status, cudaStream_t stream,
                                const int32_t *in_c, const int32_t *idx_c, long rows_c)
{
    if (count <= 0)
        return cudaSuccess;
    BrArgs A;
    A.keys = keys;
    A.in_a = in_a;
    A.in_b = in_b;
    A.in_c = in_c;
    A.idx_a = idx_a;
    A.idx_b = idx_b;
    A.idx_c = idx_c;
    A.rows_a = rows_a;
    A.rows_b = rows_b;
    A.rows_c = rows_c;
    A.ops = ops;
    A.big = big;
    A.mu = mu;
    A.status = status;
    int dev = 0;
    cudaGetDevice(&dev);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long nsm = sms > 0 ? sms : 1;
    const int shape = br_group(count, (int)nsm, keys.br_group, keys.tune_br);
    const long tail = br_tail(count, nsm, keys.br_group, shape);
    A.first = 0;
    A.count = count - tail;
    cudaError_t e = launch_shape(A, shape, nsm, dev, stream);
    if (tail && e == cudaSuccess) {
        A.first = count - tail;
        A.count = count;
        e = launch_shape(A, 2 * tail <= nsm ? kBrPair : kBrSplit, nsm, dev, stream);
    }
    return e;
}

int blind_rotate_kernels(long count, int num_sms, const DevKeys &keys)
{
    if (count <= 0)
        return 0;
    const long nsm = num_sms > 0 ? num_sms : 1;
    const int shape = br_group(count, (int)nsm, keys.br_group, keys.tune_br);
    return br_tail(count, nsm, keys.br_group, shape) ? 2 : 1;
}

}  // namespace tgb
