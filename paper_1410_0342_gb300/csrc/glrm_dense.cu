// Dense, fully observed form of the alternating proximal-gradient sweep
// (Algorithm 2 of Udell et al., "Generalized Low Rank Models", with Omega =
// every (i, j)) on the fifth-generation tensor cores.
//
// Naming: in a half-step the "own" factor F is the one being updated (X in
// the X-step, Y in the Y-step) and the "other" factor W is held fixed.  Each
// half-step is five launches:
//   pack   W split into BF16 parts x = hi + mid + lo (+ at most 2^-26 |x|) in
//          the tensor core's swizzled K-major shared-memory layouts: with K = k
//          (B operand of GEMM1) and, per 64-row chunk, with K = the chunk rows
//          (B operand of GEMM2);
//   grad   per 128 own rows and a range of 64-wide chunks of the other
//          dimension: U = F W^T (GEMM1), L(U, A) and its derivative R against
//          the A tile (staged by tensor TMA; a NaN cell is a missing entry and
//          contributes nothing), R split in three into tensor memory, G += R W
//          (GEMM2);
//   prox   f+ = prox(f - alpha g) per row / column (shared with the sparse form);
//   loss   the candidate's losses (GEMM1 and L only);
//   decide accept when the objective did not increase (shared with the
//          sparse form).
// Both GEMMs sum the six BF16 products of the splits whose order is at least
// 2^-18 (hi.hi, hi.mid, mid.hi, mid.mid, hi.lo, lo.hi) in FP32 in tensor
// memory; the dropped terms (mid.lo, lo.mid, lo.lo) and the split remainders
// are about 2^-25 of sum |f_c w_c|, below FP32's own rounding of a k-term
// dot product, so losses, the accept / reject test and the gradients see FP32
// quality values.
//
// Pipeline of one CTA (one lane each of three producer warps issues the
// GEMM1 MMAs, the copies and the GEMM2 MMAs; 16 warps run the per-entry
// work): GEMM1 runs up to two chunks ahead into a double-buffered
// accumulator, so the tensor core computes U of chunk q + 1 while the warps
// evaluate the losses of chunk q; R is double-buffered in tensor memory, so
// the warps write R of chunk q while GEMM2 of chunk q - 1 still reads the
// other buffer; W's GEMM1 and GEMM2 parts are triple-buffered, the A tiles two
// to four times.
#include <cuda.h>

#include <string.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <functional>
#include <queue>
#include <vector>

#include "glrm_tc.cuh"

namespace glrm {

constexpr int kDnNT = 64;        // chunk of the other dimension (UMMA N of GEMM1, K of GEMM2)
constexpr int kDnRows = 128;     // own rows per CTA (UMMA M)
constexpr int kDnWarps = 16;     // evaluating warp w: TMEM lanes 32 (w % 4) .. + 31, chunk columns 16 (w / 4) .. + 15
constexpr int kDnThreads = (kDnWarps + 3) * 32;  // + the GEMM1 warp, the copy warp, the GEMM2 warp
// TMEM columns: U at [0, 64) and [64, 128), two buffers of R (hi, mid, lo; 32
// columns each) at [128, 224) and [224, 320), G from 320 (two accumulators of
// up to 48 columns or one of 64), the own rows (hi, mid, lo; KP / 2 columns
// each) from 416
constexpr int kDnTmem = 512;
constexpr int kDnColR = 128, kDnColG = 320, kDnColOwn = 416;
constexpr int kDnMaxStages = 4;

// Column loss with its parameters in FP32 (kind as int bits, Huber
// threshold, ordinal level count, unused).
using LossF = float4;

struct DenseArgs {
    int64_t nown, nother;
    int k;
    const float *F;           // own factor, nown x k
    const __nv_bfloat16 *pk;  // other factor, K-major over k: parts hi, mid, lo (each pack_part)
    const __nv_bfloat16 *pt;  // other factor per chunk, K-major over the chunk rows: parts hi, mid, lo
    int64_t pack_part;        // elements per part
    const LossF *lossf;       // n column losses; w: the kind of the column's 16-column group, else -1
    const float *wcol;        // WGT kernels: n per-column loss weights (the scaled losses of Section 4.3)
    const DnItem *items;      // one per CTA
    const int32_t *blocks;    // Y-step: per tile its four 32-column blocks (-1: none)
    const int32_t *segchunk;  // own index -> first partial slot
    int nA;
    float *part_grad;     // slots x k
    double *part_loss;    // slots
    int *err;
};

// Dynamic shared memory of one CTA: the A stages first (1024-byte aligned for
// the swizzled boxes; 1024 bytes of slack align the base), then three stages
// of W's three GEMM1 parts, three stages of W's three GEMM2 parts and one loss
// table per A stage (every operand buffer on a 1024-byte boundary).
template <bool XSTEP, bool GRAD, int KP>
struct DnSmem {
    static constexpr size_t pk = (size_t)kDnNT * KP * 2;
    static constexpr size_t pt = GRAD ? (size_t)KP * kDnNT * 2 : 0;
    static constexpr size_t ls = XSTEP ? (size_t)kDnNT * sizeof(LossF) : 0;
    static constexpr size_t a = (size_t)kDnNT * kDnRows * 4;  // 32 KB A tile
    static constexpr size_t fixed = 9 * pk + 9 * pt + kDnMaxStages * ls;
    static size_t bytes(int nA) { return 1024 + fixed + (size_t)nA * a; }
};

__device__ __forceinline__ uint32_t bf2_bits(__nv_bfloat162 v)
{
    return *reinterpret_cast<uint32_t *>(&v);
}

// 2-D tiled TMA load of one box into shared memory, completion on the mbarrier.
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// x = hi + mid + lo in BF16 (each remainder exact in FP32).
__device__ __forceinline__ void split3(float v, __nv_bfloat16 &hi, __nv_bfloat16 &mid, __nv_bfloat16 &lo)
{
    hi = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(hi);
    mid = __float2bfloat16_rn(r1);
    lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
}

// One MMA with A read from tensor memory: D[taddr] (+)= A[a_taddr] B^T.
__device__ __forceinline__ void umma_bf16_ta(uint32_t taddr, uint32_t a_taddr, uint64_t bdesc, uint32_t idesc,
                                             bool accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(taddr),
        "r"(a_taddr), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}

// Eight 32-bit columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ unsigned long long fadd2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ unsigned long long fmul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ unsigned long long dup2(float v) { return pk2(v, v); }

// floor / ceil of two values in [0, 2^22]: the sum with 2^23 rounded down / up
// is exact to an integer.
__device__ __forceinline__ unsigned long long floor2(unsigned long long a)
{
    unsigned long long d;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(dup2(8388608.f)));
    return fadd2(d, dup2(-8388608.f));
}

__device__ __forceinline__ unsigned long long ceil2(unsigned long long a)
{
    unsigned long long d;
    asm("add.rp.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(dup2(8388608.f)));
    return fadd2(d, dup2(-8388608.f));
}

// Whether a kind's derivative is a whole number of magnitude at most 256 for
// every entry (hinge 0, +-1; l1 0, +-1; ordinal hinge up to levels - 1): such
// a derivative is a BF16 value, its mid and lo parts are 0.
__device__ __forceinline__ bool whole_deriv(int kind, float lev)
{
    return kind == kLossHinge || kind == kLossL1 || (kind == kLossOrdinal && lev <= 257.f);
}

// The logistic entries of a mixed block, with the scalar functions the X-step
// of mixed columns uses; a loop over copies in local memory, so that this rare
// path takes no registers from the others.
__device__ __forceinline__ void dn_block_loop(const float (&u)[16], const float (&a)[16], float (&rr)[16], float &lsum)
{
    float uu[16], aa[16];
#pragma unroll
    for (int w = 0; w < 16; ++w) {
        uu[w] = u[w];
        aa[w] = a[w];
    }
#pragma unroll 1
    for (int w = 0; w < 16; ++w) {
        const bool v = aa[w] == aa[w];
        float L;
        const float d = loss_deriv_k<kLossLogistic, float>(uu[w], aa[w], 0.f, 0.f, L);
        lsum += v ? L : 0.f;
        uu[w] = v ? d : 0.f;
    }
#pragma unroll
    for (int w = 0; w < 16; ++w) rr[w] = uu[w];
}

// The losses and derivatives of the scalar functions the sparse paths use,
// for kinds without a packed form.
template <int KIND, bool MISS>
__device__ __forceinline__ void dn_block_plain(const float (&u)[16], const float (&a)[16], float prm, float lev,
                                               float (&rr)[16], float &lsum)
{
#pragma unroll
    for (int w = 0; w < 16; ++w) {
        const bool v = !MISS || a[w] == a[w];
        float L;
        const float d = loss_deriv_k<KIND, float>(u[w], a[w], prm, lev, L);
        lsum += v ? L : 0.f;
        rr[w] = v ? d : 0.f;
    }
}

// Losses and derivatives of 16 entries that all lie inside the table and
// share one loss kind with parameters prm (Huber threshold) and lev (ordinal
// level count).  MISS: a NaN value marks a missing entry, which contributes
// nothing whatever its product.  The passes are bound by the instructions of
// this block (44 per cell in the gradient and 29 in the loss passes with the
// scalar branches of loss_deriv_k, the issue slots 40% and the FMA pipe 13%
// busy), so every kind is written without branches, two entries at a time in
// packed FP32 where the operation exists in that form:
//   Huber    c = clamp(x, -d, d) is the derivative, c (x - c / 2) the loss
//   hinge    a NaN value fails z > 0 and loses against 0 in max(z, 0): the
//            missing cells need no test
//   logistic e = exp(-|z|) = 2^i exp(r), i the nearest whole number to
//            -|z| log2 e and r the remainder (ln 2 in two parts), exp(r) =
//            1 + r + r^2 E(r); log1p(e) = e + e^2 Q(e); E and Q by minimax fits
//            whose coefficients are rounded to FP32 one after the other
//            (relative errors of exp 3.1e-9 on |r| <= ln 2 / 2, of log1p 5.2e-9 on
//            [0, 1]); the quotient by 1 + e from an approximate reciprocal and one
//            correction by its own remainder.  Cells of |z| <= 8 against 64 bits, in
//            units of 2^-24, root mean square / largest: derivative 0.72 / 2.8, loss
//            0.56 / 2.1; CUDA's functions (the scalar form) 0.80 / 3.5 and 0.62 /
//            2.6; ex2.approx, 4% faster (50,000 x 2,000, k = 32, three passes: 670
//            against 698 us), 0.99 / 4.8 and 0.82 / 3.4
//   ordinal  with uc = clamp(u, 1, d): p = (ceil(uc) - a)_+ levels above a and
//            n = (floor(uc) - a)_- below it are active, never both, so the
//            derivative is q = p + n and the loss q (u - a - q / 2) + |q| / 2
template <int KIND, bool MISS>
__device__ __forceinline__ void dn_block(const float (&u)[16], const float (&a)[16], float prm, float lev,
                                         float (&rr)[16], float &lsum)
{
    const unsigned long long m1 = dup2(-1.f), mh = dup2(-0.5f);
    unsigned long long acc = 0ull;
    // u - a of entries w, w + 1; 0 where the value is missing
    auto resid = [&](int w) {
        const unsigned long long x = ffma2(pk2(a[w], a[w + 1]), m1, pk2(u[w], u[w + 1]));
        if constexpr (!MISS) {
            return x;
        } else {
            float x0, x1;
            upk2(x, x0, x1);
            return pk2(a[w] == a[w] ? x0 : 0.f, a[w + 1] == a[w + 1] ? x1 : 0.f);
        }
    };
    if constexpr (KIND == kLossQuad) {
#pragma unroll
        for (int w = 0; w < 16; w += 2) {
            const unsigned long long r = resid(w);
            acc = ffma2(r, r, acc);
            upk2(fadd2(r, r), rr[w], rr[w + 1]);
        }
    } else if constexpr (KIND == kLossHuber) {
#pragma unroll
        for (int w = 0; w < 16; w += 2) {
            const unsigned long long x = resid(w);
            float x0, x1;
            upk2(x, x0, x1);
            rr[w] = fmaxf(fminf(x0, prm), -prm);
            rr[w + 1] = fmaxf(fminf(x1, prm), -prm);
            const unsigned long long c = pk2(rr[w], rr[w + 1]);
            acc = ffma2(c, ffma2(c, mh, x), acc);
        }
    } else if constexpr (KIND == kLossHinge) {
        const unsigned long long one = dup2(1.f);
#pragma unroll
        for (int w = 0; w < 16; w += 2) {
            const unsigned long long na = fmul2(pk2(a[w], a[w + 1]), m1);
            float n0, n1, z0, z1;
            upk2(na, n0, n1);
            upk2(ffma2(na, pk2(u[w], u[w + 1]), one), z0, z1);
            rr[w] = z0 > 0.f ? n0 : 0.f;
            rr[w + 1] = z1 > 0.f ? n1 : 0.f;
            acc = fadd2(acc, pk2(fmaxf(z0, 0.f), fmaxf(z1, 0.f)));
        }
    } else if constexpr (KIND == kLossLogistic) {
        constexpr float kE[5] = {0.49999994f, 0.16666521f, 0.041668262f, 0.0083686709f, 0.0013820895f};
        constexpr float kQ[9] = {-0.49999934f, 0.33330551f, -0.24958938f, 0.19696993f, -0.15359527f,
                                 0.10686939f, -0.057722557f, 0.020233344f, -0.0033244395f};
        const unsigned long long one = dup2(1.f), magic = dup2(12582912.f), mmagic = dup2(-12582912.f);
#pragma unroll
        for (int w = 0; w < 16; w += 2) {
            const unsigned long long av = pk2(a[w], a[w + 1]);
            float x0, x1, y0, y1, p0, p1;  // -z, -|z| (exp is 0 in FP32 from -88 on), max(z, 0); a NaN stays one
            upk2(fmul2(av, pk2(u[w], u[w + 1])), x0, x1);
            asm("max.NaN.f32 %0, %1, %2;" : "=f"(y0) : "f"(-fabsf(x0)), "f"(-88.f));
            asm("max.NaN.f32 %0, %1, %2;" : "=f"(y1) : "f"(-fabsf(x1)), "f"(-88.f));
            asm("max.NaN.f32 %0, %1, %2;" : "=f"(p0) : "f"(-x0), "f"(0.f));
            asm("max.NaN.f32 %0, %1, %2;" : "=f"(p1) : "f"(-x1), "f"(0.f));
            const unsigned long long y = pk2(y0, y1);
            const unsigned long long t = ffma2(y, dup2(1.44269504f), magic);  // its low bits: i
            const unsigned long long i = fadd2(t, mmagic);
            unsigned long long r = ffma2(i, dup2(-0.693147182f), y);  // ln 2 = 0.693147182 - 1.90465430e-9
            r = ffma2(i, dup2(1.90465430e-9f), r);
            unsigned long long e = dup2(kE[4]);
#pragma unroll
            for (int c = 3; c >= 0; --c) e = ffma2(e, r, dup2(kE[c]));
            e = ffma2(ffma2(e, r, one), r, one);
            float t0, t1;
            upk2(t, t0, t1);
            e = fmul2(e, pk2(__uint_as_float((__float_as_uint(t0) << 23) + 0x3f800000u),
                             __uint_as_float((__float_as_uint(t1) << 23) + 0x3f800000u)));
            unsigned long long Q = dup2(kQ[8]);
#pragma unroll
            for (int c = 7; c >= 0; --c) Q = ffma2(Q, e, dup2(kQ[c]));
            float L0, L1, e0, e1, v0, v1, r0, r1, d0, d1;
            upk2(ffma2(e, ffma2(Q, e, one), pk2(p0, p1)), L0, L1);
            const unsigned long long v = fadd2(e, one);
            upk2(v, v0, v1);
            upk2(e, e0, e1);
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(-v0));
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(-v1));
            // -sigma(z) = -num / v
            const unsigned long long rc = pk2(r0, r1), num = pk2(x0 <= 0.f ? 1.f : e0, x1 <= 0.f ? 1.f : e1);
            const unsigned long long q = fmul2(num, rc);
            upk2(fmul2(av, ffma2(ffma2(q, v, num), rc, q)), d0, d1);
            const bool ok0 = !MISS || a[w] == a[w], ok1 = !MISS || a[w + 1] == a[w + 1];
            rr[w] = ok0 ? d0 : 0.f;
            rr[w + 1] = ok1 ? d1 : 0.f;
            acc = fadd2(acc, pk2(ok0 ? L0 : 0.f, ok1 ? L1 : 0.f));
        }
    } else if constexpr (KIND == kLossOrdinal) {
#pragma unroll
        for (int w = 0; w < 16; w += 2) {
            const unsigned long long uc =
                pk2(fminf(fmaxf(u[w], 1.f), lev), fminf(fmaxf(u[w + 1], 1.f), lev));
            const unsigned long long av = pk2(a[w], a[w + 1]);
            float p0, p1, n0, n1;
            upk2(ffma2(av, m1, ceil2(uc)), p0, p1);
            upk2(ffma2(av, m1, floor2(uc)), n0, n1);
            const unsigned long long p = pk2(fmaxf(p0, 0.f), fmaxf(p1, 0.f));  // 0 for a NaN value
            const unsigned long long n = pk2(fminf(n0, 0.f), fminf(n1, 0.f));
            const unsigned long long q = fadd2(p, n);
            acc = ffma2(q, ffma2(q, mh, resid(w)), acc);
            acc = ffma2(p, dup2(0.5f), acc);
            acc = ffma2(n, mh, acc);
            upk2(q, rr[w], rr[w + 1]);
        }
    } else {
        dn_block_plain<KIND, MISS>(u, a, prm, lev, rr, lsum);
    }
    float l0, l1;
    upk2(acc, l0, l1);
    lsum += l0 + l1;
}

template <bool MISS>
__device__ __forceinline__ void dn_block_kind(int kind, const float (&u)[16], const float (&a)[16], float prm,
                                              float lev, float (&rr)[16], float &lsum)
{
    switch (kind) {
    case kLossQuad: dn_block<kLossQuad, MISS>(u, a, prm, lev, rr, lsum); break;
    case kLossHuber: dn_block<kLossHuber, MISS>(u, a, prm, lev, rr, lsum); break;
    case kLossHinge: dn_block<kLossHinge, MISS>(u, a, prm, lev, rr, lsum); break;
    case kLossLogistic: dn_block<kLossLogistic, MISS>(u, a, prm, lev, rr, lsum); break;
    case kLossOrdinal: dn_block<kLossOrdinal, MISS>(u, a, prm, lev, rr, lsum); break;
    case kLossL1: dn_block<kLossL1, MISS>(u, a, prm, lev, rr, lsum); break;
    default: dn_block<kLossQuantile, MISS>(u, a, prm, lev, rr, lsum); break;
    }
}

// The X-step with any mix of kinds: the entries are 16 columns (losses in lf;
// the branches are uniform over the warp); entries outside the table (bit
// clear in `valid`) and missing entries (NaN) give 0.
__device__ __forceinline__ void dn_block_any(const float (&u)[16], const float (&a)[16], const LossF *lf,
                                             uint32_t valid, float (&rr)[16], float &lsum)
{
#pragma unroll
    for (int w = 0; w < 16; ++w) {
        const LossF sp = lf[w];
        float L;
        const float d = loss_deriv_kind<float>(__float_as_int(sp.x), u[w], a[w], sp.y, sp.z, L);
        const bool v = ((valid >> w) & 1u) && a[w] == a[w];
        lsum += v ? L : 0.f;
        rr[w] = v ? d : 0.f;
    }
}

// The X-step with per-column loss weights: 16 entries of 16 columns, each
// loss and derivative times its column's weight (wt: the weights of these
// columns; read only for entries inside the table).
__device__ __forceinline__ void dn_block_w(const float (&u)[16], const float (&a)[16], const LossF *lf,
                                           const float *__restrict__ wt, uint32_t valid, float (&rr)[16],
                                           float &lsum)
{
#pragma unroll
    for (int w = 0; w < 16; ++w) {
        const LossF sp = lf[w];
        float L;
        const float d = loss_deriv_kind<float>(__float_as_int(sp.x), u[w], a[w], sp.y, sp.z, L);
        const bool v = ((valid >> w) & 1u) && a[w] == a[w];
        const float c = v ? __ldg(wt + w) : 0.f;
        lsum += v ? c * L : 0.f;
        rr[w] = v ? c * d : 0.f;
    }
}

// One pass over a (128 own rows) x (range of chunks) block.  GRAD: partial
// gradient rows and partial losses; otherwise partial losses only.
// A tiles: X-step, two boxes of 32 columns x 128 own rows with the 128-byte
// swizzle (16-byte unit u of row r at u ^ (r % 8): conflict-free row reads);
// Y-step, one box of 128 own columns x 64 rows, unswizzled.
// Warps 0 .. 15 evaluate the entries; one lane each of warp 16 issues GEMM1,
// of warp 17 the copies, of warp 18 GEMM2 (two warps: beside four evaluating
// warps on its scheduler an issuing warp spends 70 to 170 cycles per MMA, and
// both GEMMs of a chunk from one warp took longer than its evaluation).
// A warp's chunk is a chain of latencies (tensor memory load, shared-memory
// load, barrier polls) and only four warps share a scheduler, so the loads of
// chunk c + 1 are started in the middle of chunk c, as soon as its losses are
// formed (the registers of U and A are free then), and land behind the split
// and the stores of R.
// barU[c % 4]: every warp holds U of chunk c in registers; the GEMM1 warp
// issues GEMM1 of c + 2 into that accumulator, the copy warp W's part of c + 3
// into the stage GEMM1 of c has read.  barE[c % 4]: the entries of chunk c are
// done (A stage read, R written); the GEMM2 warp issues GEMM2 of c, the copy
// warp refills the A stage.  barG1[c % 2] completes when GEMM1 of chunk c is
// done, the copy warp has seen A of c land (with two A stages the tile is
// requested too late for that: the evaluating warps poll barA themselves) and
// the GEMM2 warp has seen GEMM2 of c - 3 end, so that an evaluating warp polls
// one barrier per chunk (a poll that succeeds at once takes 100 to 400 cycles
// beside busy warps): waited for in the middle of chunk c - 1, it also frees
// the R buffer that chunk c - 1 writes.
// No waiter falls two phases behind barG1 or four behind the others: all
// arrivals of barG1 for chunk c + 2 follow barU or barE of c.  A warp reads U of
// chunk c + 4 only after GEMM1 of c + 4, which is issued after the GEMM1
// warp's wait for barU of c + 2 and needs W's part of c + 4, issued by the
// copy warp after its waits for barE of c and barU of c + 1; barG1 of c + 4
// has the GEMM2 warp's arrival, made after its waits for barE of c + 2 and
// barG2 of c + 1; GEMM2 of c + 3 needs W's part of c + 3, issued after the copy
// warp's wait for barG2 of c - 1 and of c.
// B16 (gradient passes of the BF16 form): GEMM2 takes the single product of
// R's and W's BF16 high parts (FP32 accumulation) and only R's high part is
// written to tensor memory; GEMM1, the losses, derivatives and objectives
// keep the six-product FP32 quality.
template <bool XSTEP, bool GRAD, int KP, bool MISS, bool B16 = false, bool WGT = false>
__global__ void __launch_bounds__(kDnThreads, 1)
dense_pass_kernel(const DenseArgs p, const __grid_constant__ CUtensorMap amap)
{
    using SM = DnSmem<XSTEP, GRAD, KP>;
    extern __shared__ __align__(1024) unsigned char dsm_dense[];
    __shared__ uint64_t barA[kDnMaxStages], barP[3], barT[3], barG1[2], barG2[4], barU[4], barE[4];
    __shared__ __align__(16) uint8_t whole_s[4][kDnWarps];  // per chunk (mod 4) and warp: R has no lower parts
    __shared__ uint32_t tslot;
    __shared__ double red[4][kDnRows];
    unsigned char *base = dsm_dense + ((1024 - (smem_u32(dsm_dense) & 1023)) & 1023);
    unsigned char *ast = base;                                   // A stage s at ast + s * a
    unsigned char *fx = base + (size_t)p.nA * SM::a;             // fixed buffers
    unsigned char *pkst = fx;                                    // pk stage s at pkst + s * 3 pk
    unsigned char *ptst = pkst + 9 * SM::pk;                     // pt stage s at ptst + s * 3 pt
    unsigned char *lsst = ptst + 9 * SM::pt;                     // loss table of A stage s at lsst + s * ls

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quarter = warp & 3, grp = (warp >> 2) & 3;
    const int orow = quarter * 32 + lane;
    const DnItem item = p.items[blockIdx.x];
    const int64_t o0 = (int64_t)item.tile * kDnRows;
    const int64_t qb = item.q0;
    const int nq = item.nq;
    const int nA = p.nA;
    // GEMM2's width in coordinates, and whether its hi . hi products have an
    // accumulator of their own.  An MMA rounds the running sum it adds to, so
    // with all six products in one accumulator the five small ones of every
    // chunk cost as much rounding as the large one: 24 roundings a chunk instead
    // of 4 (error of Yt after a sweep of the 100,000 x 1,000 mixed table,
    // k = 20: 1.02e-6 against 9.7e-8; time 688 against 691 us).  Ranks over 48 leave no
    // columns for a second one.
    const int gw = KP <= 32 ? KP : (p.k <= 48 ? 48 : 64);
    const bool two = !B16 && gw <= 48;
    const bool producer = warp >= kDnWarps;  // kDnWarps: GEMM1, kDnWarps + 1: copies, kDnWarps + 2: GEMM2
    // this thread's own row (X-step) or column (Y-step: quarter q of the tile
    // is the 32-column block blocks[4 tile + q]), and its partial slot
    int64_t own = o0 + orow;
    if (!XSTEP) {
        const int32_t b = producer ? -1 : p.blocks[4 * (int64_t)item.tile + quarter];
        own = b < 0 ? p.nown : 32 * (int64_t)b + lane;
    }
    const bool own_ok = !producer && own < p.nown;
    const int64_t slot = own_ok ? (int64_t)p.segchunk[own] + item.part : 0;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const int tb = grp * 16;  // this warp's columns of a chunk

    // warps 0 .. 3: the own rows, one per thread, on their way while the
    // barriers and tensor memory are set up
    float fv[KP];
    if (grp == 0 && !producer) {
        const float *f = p.F + own * p.k;
        if (p.k % 4 == 0 && reinterpret_cast<uintptr_t>(p.F) % 16 == 0) {
#pragma unroll
            for (int c = 0; c < KP; c += 4) {
                const float4 v = (own_ok && c < p.k) ? *reinterpret_cast<const float4 *>(f + c)
                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                fv[c] = v.x;
                fv[c + 1] = v.y;
                fv[c + 2] = v.z;
                fv[c + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int c = 0; c < KP; ++c) fv[c] = (own_ok && c < p.k) ? f[c] : 0.f;
        }
    }
    if (warp == kDnWarps) tmem_alloc(&tslot, kDnTmem);
    if (warp == kDnWarps + 1 && lane == 0) {
        for (int s = 0; s < kDnMaxStages; ++s) mbar_init(&barA[s], 1);
        for (int s = 0; s < 3; ++s) mbar_init(&barP[s], 1);
        for (int s = 0; s < 3; ++s) mbar_init(&barT[s], 1);
        for (int s = 0; s < 2; ++s) mbar_init(&barG1[s], 1 + (nA > 2) + (GRAD ? 1 : 0));
        for (int s = 0; s < 4; ++s) mbar_init(&barG2[s], 1);
        for (int s = 0; s < 4; ++s) mbar_init(&barU[s], kDnWarps);
        for (int s = 0; s < 4; ++s) mbar_init(&barE[s], kDnWarps);
    }
    // Y-step: this thread's column loss, and whether the warp shares one kind
    LossF myspec = make_float4(__int_as_float(kLossQuad), 0.f, 0.f, 0.f);
    if (!XSTEP && own_ok) myspec = p.lossf[own];
    // Y-step with column weights: this thread's column's weight
    const float wown = (!XSTEP && WGT && own_ok) ? p.wcol[own] : 1.f;
    // (a block past the table's last column: lane 0 is inside, the lanes outside
    // take its kind and parameters)
    int wkind = -1;
    unsigned wkinds = 0;  // the kinds present
    bool wwhole = false;
    if constexpr (!XSTEP) {
        const int k0 = __shfl_sync(0xffffffffu, __float_as_int(myspec.x), 0);
        const float y0 = __shfl_sync(0xffffffffu, myspec.y, 0), z0 = __shfl_sync(0xffffffffu, myspec.z, 0);
        if (!own_ok) myspec = make_float4(__int_as_float(k0), y0, z0, 0.f);
        wkind = __all_sync(0xffffffffu, __float_as_int(myspec.x) == k0) ? k0 : -1;
        wkinds = __reduce_or_sync(0xffffffffu, 1u << __float_as_int(myspec.x));
        wwhole = __all_sync(0xffffffffu, whole_deriv(__float_as_int(myspec.x), myspec.z));
    }

    bool ok = true;
    float lacc = 0.f, lcomp = 0.f;
    // producer bookkeeping (lane 0 of the producer warps)
    int p_issued = 0, a_issued = 0, t_issued = 0, g1_issued = 0, g2_issued = 0;
    auto issue_pack = [&](int64_t q) {  // GEMM1's W parts, stage q % 3
        const int s = (int)((q - qb) % 3);
        unsigned char *st = pkst + s * 3 * SM::pk;
        const int64_t t0 = q * kDnNT;
        mbar_expect_tx(&barP[s], (unsigned)(3 * SM::pk));
#pragma unroll
        for (int w = 0; w < 3; ++w)
            bulk_g2s(st + w * SM::pk, p.pk + w * p.pack_part + t0 * KP, (unsigned)SM::pk, &barP[s]);
        ++p_issued;
    };
    auto issue_pt = [&](int64_t q) {  // GEMM2's W parts, stage q % 3
        const int s = (int)((q - qb) % 3);
        unsigned char *st = ptst + s * 3 * SM::pt;
        mbar_expect_tx(&barT[s], (unsigned)(3 * SM::pt));
#pragma unroll
        for (int w = 0; w < 3; ++w)
            bulk_g2s(st + w * SM::pt, p.pt + w * p.pack_part + q * KP * kDnNT, (unsigned)SM::pt, &barT[s]);
        ++t_issued;
    };
    // Y-step: the tile's 32-column blocks (box q of a stage holds block q)
    int32_t blk[4] = {-1, -1, -1, -1};
    unsigned nblk = 0;
    if (!XSTEP && warp == kDnWarps + 1) {
        for (int qd = 0; qd < 4; ++qd) {
            blk[qd] = p.blocks[4 * (int64_t)item.tile + qd];
            nblk += blk[qd] >= 0 ? 1u : 0u;
        }
    }
    // the A tile (out-of-range elements read as 0) and, X-step, the chunk's
    // column losses, stage q % nA
    auto issue_a = [&](int64_t q) {
        const int s = (int)((q - qb) % nA);
        unsigned char *dst = ast + s * SM::a;
        const int t0 = (int)(q * kDnNT);
        if constexpr (XSTEP) {
            const int nv = (int)(p.nother - t0 < kDnNT ? p.nother - t0 : kDnNT);
            mbar_expect_tx(&barA[s], (unsigned)(SM::a + nv * sizeof(LossF)));
            tma_load_2d(dst, &amap, t0, (int)o0, &barA[s]);
            tma_load_2d(dst + SM::a / 2, &amap, t0 + 32, (int)o0, &barA[s]);
            bulk_g2s(lsst + s * SM::ls, p.lossf + t0, (unsigned)(nv * sizeof(LossF)), &barA[s]);
        } else {
            mbar_expect_tx(&barA[s], nblk * (unsigned)(SM::a / 4));
            for (int qd = 0; qd < 4; ++qd)
                if (blk[qd] >= 0) tma_load_2d(dst + qd * (SM::a / 4), &amap, 32 * blk[qd], t0, &barA[s]);
        }
        ++a_issued;
    };
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = tslot;
    // the first copies start while the own rows are written to tensor memory
    if (warp == kDnWarps + 1 && elect_one()) {
        for (int s = 0; s < 3 && s < nq; ++s) issue_pack(qb + s);
        for (int s = 0; s < nA && s < nq; ++s) issue_a(qb + s);
        if (GRAD)
            for (int s = 0; s < 2 && s < nq; ++s) issue_pt(qb + s);
    }
    // own rows split in three into tensor memory (GEMM1's A operand, two BF16
    // values per column along k)
    if (grp == 0 && !producer) {
#pragma unroll
        for (int c0 = 0; c0 < KP; c0 += 16) {
            uint32_t hv[8], mv[8], lv[8];
#pragma unroll
            for (int w = 0; w < 16; w += 2) {
                __nv_bfloat16 h0, m0, l0, h1, m1, l1;
                split3(fv[c0 + w], h0, m0, l0);
                split3(fv[c0 + w + 1], h1, m1, l1);
                hv[w / 2] = bf2_bits(__halves2bfloat162(h0, h1));
                mv[w / 2] = bf2_bits(__halves2bfloat162(m0, m1));
                lv[w / 2] = bf2_bits(__halves2bfloat162(l0, l1));
            }
            tmem_st8(taddr + lane_base + (uint32_t)(kDnColOwn + c0 / 2), hv);
            tmem_st8(taddr + lane_base + (uint32_t)(kDnColOwn + KP / 2 + c0 / 2), mv);
            tmem_st8(taddr + lane_base + (uint32_t)(kDnColOwn + KP + c0 / 2), lv);
        }
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (producer) {
        const bool lead = elect_one();  // the lane that issues
        // (own or R part, W part) of the six products, smallest first; hi . hi last
        constexpr int pa[6] = {1, 0, 2, 0, 1, 0};
        constexpr int pb[6] = {1, 2, 0, 1, 0, 0};
        if (warp == kDnWarps && lead) {
            // GEMM1 warp
            for (int c = 0; ok && c < nq; ++c) {
                const int s = c % 3, b = c & 1;
                // U of chunk c - 2 is in registers, W's parts of chunk c are in
                if (c > 1) ok = mbar_wait_bounded(&barU[(c - 2) & 3], (unsigned)((c - 2) >> 2) & 1u);
                ok = ok && mbar_wait_bounded(&barP[s], (unsigned)(c / 3) & 1u);
                if (!ok) break;
                tc_fence_after();
                constexpr uint32_t idesc = umma_idesc_bf16(kDnRows, kDnNT);
                constexpr uint32_t RB = 2 * KP;  // bytes per W row; a K step of 16 is 32 bytes, 8 own columns
                const uint64_t d0 = umma_desc_sw(pkst + s * 3 * SM::pk, RB);
#pragma unroll
                for (int pr = 0; pr < 6; ++pr)
#pragma unroll
                    for (int ks = 0; ks < KP / 16; ++ks)
                        umma_bf16_ta(taddr + (uint32_t)(b * kDnNT),
                                     taddr + (uint32_t)(kDnColOwn + pa[pr] * (KP / 2) + ks * 8),
                                     d0 + ((pb[pr] * SM::pk + ks * 32) >> 4), idesc, pr > 0 || ks > 0);
                umma_commit(&barG1[b]);
                ++g1_issued;
            }
        } else if (GRAD && warp == kDnWarps + 2 && lead) {
            // GEMM2 warp: G += R W, R from tensor memory (a K = 16 step of R is 8 columns)
            mbar_arrive(&barG1[0]);
            if (nq > 1) mbar_arrive(&barG1[1]);
            for (int c = 0; ok && c < nq; ++c) {
                const int s = c % 3;
                ok = mbar_wait_bounded(&barT[s], (unsigned)(c / 3) & 1u);
                ok = ok && mbar_wait_bounded(&barE[c & 3], (unsigned)(c >> 2) & 1u);  // R of chunk c is written
                // GEMM2 of c - 1 is done: chunk c + 1 may write its R buffer once
                // the warps have seen barG1 of c + 2
                if (c > 0) ok = ok && mbar_wait_bounded(&barG2[(c - 1) & 3], (unsigned)((c - 1) >> 2) & 1u);
                if (!ok) break;
                if (c + 2 < nq) mbar_arrive(&barG1[c & 1]);
                tc_fence_after();
                const uint64_t d0 = umma_desc_sw(ptst + s * 3 * SM::pt, 2 * kDnNT);
                const uint32_t r0 = taddr + (uint32_t)(kDnColR + (c & 1) * 96);
                // the four warps of each 16 chunk columns say whether R has
                // lower parts there: MMAs over zeros are left out (half of
                // them on a table of Boolean and ordinal columns)
                uint32_t wh[4];
                *reinterpret_cast<uint4 *>(wh) = *reinterpret_cast<const uint4 *>(whole_s[c & 3]);
                const uint32_t idesc = umma_idesc_bf16(kDnRows, gw);
                constexpr int P0 = B16 ? 5 : 0;  // the BF16 form: hi . hi only
#pragma unroll
                for (int pr = P0; pr < 6; ++pr)
#pragma unroll
                    for (int ks = 0; ks < kDnNT / 16; ++ks) {
                        // an accumulator's first MMA of chunk 0 sets it
                        const bool first = ks == 0 && (pr == P0 || (pr == 5 && two));
                        if ((pr == P0 && ks == 0) || pa[pr] == 0 || wh[ks] != 0x01010101u)
                            umma_bf16_ta(taddr + kDnColG + (two && pr < 5 ? gw : 0), r0 + pa[pr] * 32 + ks * 8,
                                         d0 + ((pb[pr] * SM::pt + ks * 32) >> 4), idesc, c > 0 || !first);
                    }
                umma_commit(&barG2[c & 3]);
                ++g2_issued;
            }
        } else if (warp == kDnWarps + 1 && lead) {
            for (int c = 0; ok && nA > 2 && c < 2 && c < nq; ++c) {
                ok = mbar_wait_bounded(&barA[c], 0);
                if (ok) mbar_arrive(&barG1[c]);
            }
            for (int it = 0; ok && it < nq; ++it) {
                const int64_t q = qb + it;
                // U of chunk it is read, so GEMM1 of it has read its W stage
                ok = mbar_wait_bounded(&barU[it & 3], (unsigned)(it >> 2) & 1u);
                if (!ok) break;
                if (it + 3 < nq) issue_pack(q + 3);
                if (nA > 2 && it + 2 < nq) {  // barG1's arrival for the A tile of it + 2
                    ok = mbar_wait_bounded(&barA[(it + 2) % nA], (unsigned)((it + 2) / nA) & 1u);
                    if (!ok) break;
                    mbar_arrive(&barG1[it & 1]);
                }
                // the entries of chunk it are done: its A stage is free
                ok = mbar_wait_bounded(&barE[it & 3], (unsigned)(it >> 2) & 1u);
                if (!ok) break;
                if (it + nA < nq) issue_a(q + nA);
                if (GRAD && it + 2 < nq) {
                    // GEMM2 of it - 1 leaves the stage of it + 2
                    if (it > 0) ok = mbar_wait_bounded(&barG2[(it - 1) & 3], (unsigned)((it - 1) >> 2) & 1u);
                    if (ok) issue_pt(q + 2);
                }
            }
        }
    } else {
        int sA = 0;  // ring position of the A stage, a counter (a chunk is few hundred instructions: no division)
        const bool own_all = __all_sync(0xffffffffu, own_ok), own_any = __any_sync(0xffffffffu, own_ok);
        int64_t left = p.nother - qb * kDnNT - tb;  // entries of the other dimension from this warp's first on
        float u[16], a[16];
        uint32_t ur[16];
        // this warp's cells of the A stage sA
        auto load_a = [&]() {
            const unsigned char *as = ast + sA * SM::a;
            if constexpr (XSTEP) {
                // box tb / 32, row orow: 16-byte units (tb % 32) / 4 .. + 3, swizzled
                const unsigned char *row = as + (tb >> 5) * (SM::a / 2) + orow * 128;
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const float4 v =
                        *reinterpret_cast<const float4 *>(row + ((((tb & 31) >> 2) + w) ^ (orow & 7)) * 16);
                    a[4 * w] = v.x;
                    a[4 * w + 1] = v.y;
                    a[4 * w + 2] = v.z;
                    a[4 * w + 3] = v.w;
                }
            } else {
                // box `quarter`: 64 chunk rows x 32 columns
                const float *af = reinterpret_cast<const float *>(as) + quarter * (kDnNT * 32);
#pragma unroll
                for (int w = 0; w < 16; ++w) a[w] = af[(tb + w) * 32 + lane];
            }
        };
        // wait for U and A of chunk c (stage sA) and start loading both; whole
        // warp, false when the wait ran out
        auto start_loads = [&](int c) -> bool {
            bool w = mbar_wait_bounded(&barG1[c & 1], (unsigned)(c >> 1) & 1u);
            if (nA == 2) w = w && mbar_wait_bounded(&barA[sA], (unsigned)(c >> 1) & 1u);
            tc_fence_after();
            w = __all_sync(0xffffffffu, w);  // tcgen05.ld / st are warp-collective
            if (w) {
                tmem_ld16_start(taddr + lane_base + (uint32_t)((c & 1) * kDnNT + tb), ur);
                load_a();
            }
            return w;
        };
        ok = start_loads(0);
        for (int it = 0; ok && it < nq; ++it, left -= kDnNT) {
            tmem_ld16_wait(ur, u);
            // U of this chunk is in registers: its accumulator may take GEMM1 of it + 2
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&barU[it & 3]);
            float lsum = 0.f;
            float rr[16];
            bool whole = false;  // every derivative is a whole number BF16 holds
            {
                const bool full = own_all && left >= 16;
                const uint32_t valid =
                    !own_ok ? 0u : (left >= 16 ? 0xffffu : (left <= 0 ? 0u : (1u << left) - 1u));
                const LossF *lf = reinterpret_cast<const LossF *>(lsst + sA * SM::ls) + tb;
                // the kind (and parameters) the 16 entries share, -1 if they do not:
                // X-step, kept in the w of each column's loss; Y-step, the warp's columns
                int kind = wkind;
                float prm = myspec.y, lev = myspec.z;
                if constexpr (XSTEP) {
                    const LossF l0 = lf[0];
                    kind = left > 0 ? __float_as_int(l0.w) : -1;
                    prm = l0.y;
                    lev = l0.z;
                }
                if (XSTEP && WGT) {
                    if constexpr (XSTEP && WGT)
                        dn_block_w(u, a, lf, p.wcol + (qb + it) * kDnNT + tb, valid, rr, lsum);
                } else if (!own_any || left <= 0) {  // nothing of this warp lies inside the table
#pragma unroll
                    for (int w = 0; w < 16; ++w) rr[w] = 0.f;
                    whole = true;
                } else if (XSTEP && kind < 0) {
                    dn_block_any(u, a, lf, valid, rr, lsum);
                } else {
                    whole = !WGT && (XSTEP ? whole_deriv(kind, lev) : wwhole);
                    if (!full) {  // cells outside the table count as missing
#pragma unroll
                        for (int w = 0; w < 16; ++w)
                            if (!((valid >> w) & 1u)) a[w] = __int_as_float(0x7fffffff);
                    }
                    if (!MISS && full && kind >= 0) {
                        dn_block_kind<false>(kind, u, a, prm, lev, rr, lsum);
                    } else if (XSTEP || kind >= 0) {
                        dn_block_kind<true>(kind, u, a, prm, lev, rr, lsum);
                    } else {
                        // Y-step, a 32-column block that mixes kinds: kind by
                        // kind, the lanes of that kind
                        for (unsigned todo = wkinds; todo; todo &= todo - 1u) {
                            const int kd = __ffs((int)todo) - 1;
                            if (kd == __float_as_int(myspec.x)) {
                                if (kd == kLossLogistic) dn_block_loop(u, a, rr, lsum);
                                else dn_block_kind<true>(kd, u, a, prm, lev, rr, lsum);
                            }
                            __syncwarp();
                        }
                    }
                }
                if constexpr (!XSTEP && WGT) {  // the column's weight on its 16 entries
                    lsum *= wown;
#pragma unroll
                    for (int w = 0; w < 16; ++w) rr[w] *= wown;
                }
            }
            // the next chunk's loads start here
            if (++sA == nA) sA = 0;
            if (it + 1 < nq) ok = start_loads(it + 1);
            else if (GRAD && nq > 2) {  // (no later U to wait for)
                ok = mbar_wait_bounded(&barG2[(nq - 3) & 3], (unsigned)((nq - 3) >> 2) & 1u);
                tc_fence_after();
                ok = __all_sync(0xffffffffu, ok);
            }
            if (!ok) break;
            // compensated FP32 running sum of the chunk sums
            {
                const float y = lsum - lcomp;
                const float t = lacc + y;
                lcomp = (t - lacc) - y;
                lacc = t;
            }
            if constexpr (GRAD) {
                uint32_t hi[8], mi[8], lo[8];
                const unsigned long long m1 = pk2(-1.f, -1.f);
                if (B16 || whole) {  // (whole: warp-uniform) the high parts are all of R
#pragma unroll
                    for (int w = 0; w < 16; w += 2) {
                        hi[w / 2] = bf2_bits(__floats2bfloat162_rn(rr[w], rr[w + 1]));
                        mi[w / 2] = lo[w / 2] = 0u;
                    }
                } else {
#pragma unroll
                    for (int w = 0; w < 16; w += 2) {
                        // r = hi + mid + lo, each remainder exact in FP32
                        const __nv_bfloat162 h2 = __floats2bfloat162_rn(rr[w], rr[w + 1]);
                        const float2 hf = __bfloat1622float2(h2);
                        const unsigned long long r1 = ffma2(pk2(hf.x, hf.y), m1, pk2(rr[w], rr[w + 1]));
                        float a0, a1;
                        upk2(r1, a0, a1);
                        const __nv_bfloat162 m2 = __floats2bfloat162_rn(a0, a1);
                        const float2 mf = __bfloat1622float2(m2);
                        float b0, b1;
                        upk2(ffma2(pk2(mf.x, mf.y), m1, r1), b0, b1);
                        hi[w / 2] = bf2_bits(h2);
                        mi[w / 2] = bf2_bits(m2);
                        lo[w / 2] = bf2_bits(__floats2bfloat162_rn(b0, b1));
                    }
                }
                const uint32_t rcol = kDnColR + (uint32_t)((it & 1) * 96 + tb / 2);
                tmem_st8(taddr + lane_base + rcol, hi);
                if constexpr (!B16) {
                    tmem_st8(taddr + lane_base + rcol + 32, mi);
                    tmem_st8(taddr + lane_base + rcol + 64, lo);
                }
                tmem_wait_st();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (GRAD) whole_s[it & 3][4 * grp + quarter] = whole ? 1 : 0;
                mbar_arrive(&barE[it & 3]);
            }
        }
        if (GRAD && ok) {
            ok = mbar_wait_bounded(&barG2[(nq - 1) & 3], (unsigned)((nq - 1) >> 2) & 1u);
            tc_fence_after();
            ok = __all_sync(0xffffffffu, ok);
        }
    }
    const bool fail = __syncthreads_or(!ok) != 0;
    if (!fail && !producer) {
        red[grp][orow] = (double)lacc - (double)lcomp;
        if (GRAD && grp == 0) {
            float *g = p.part_grad + slot * p.k;
#pragma unroll
            for (int bb = 0; bb < KP / 16; ++bb) {
                if (16 * bb >= gw) break;
                float v[16];
                if (two) {
                    uint32_t hi[16], lo[16];
                    float low[16];
                    tmem_ld16_start(taddr + lane_base + (uint32_t)(kDnColG + 16 * bb), hi);
                    tmem_ld16_start(taddr + lane_base + (uint32_t)(kDnColG + gw + 16 * bb), lo);
                    tmem_ld16_wait(hi, v);
                    tmem_ld16_wait(lo, low);
#pragma unroll
                    for (int w = 0; w < 16; ++w) v[w] += low[w];
                } else {
                    tmem_ld16(taddr + lane_base + (uint32_t)(kDnColG + 16 * bb), v);
                }
                if (own_ok) {
#pragma unroll
                    for (int w = 0; w < 16; ++w)
                        if (16 * bb + w < p.k) g[16 * bb + w] = v[w];
                }
            }
        }
    }
    __syncthreads();
    if (!fail && !producer && grp == 0 && own_ok)
        p.part_loss[slot] = red[0][orow] + red[1][orow] + red[2][orow] + red[3][orow];
    if (fail && producer && elect_one()) {  // each producer warp drains what it issued (the same lane as above)
        atomicOr(p.err, 1);
        // wait (bounded) for the last copy into each stage and the last MMA
        // batches: every earlier one completed before a later one was issued
        for (int c = p_issued - 3 > 0 ? p_issued - 3 : 0; c < p_issued; ++c)
            mbar_wait_bounded(&barP[c % 3], (unsigned)(c / 3) & 1u);
        for (int c = a_issued - nA > 0 ? a_issued - nA : 0; c < a_issued; ++c)
            mbar_wait_bounded(&barA[c % nA], (unsigned)(c / nA) & 1u);
        for (int c = t_issued - 3 > 0 ? t_issued - 3 : 0; c < t_issued; ++c)
            mbar_wait_bounded(&barT[c % 3], (unsigned)(c / 3) & 1u);
        for (int c = g1_issued - 2 > 0 ? g1_issued - 2 : 0; c < g1_issued; ++c)
            mbar_wait_bounded(&barG1[c & 1], (unsigned)(c >> 1) & 1u);
        for (int c = g2_issued - 2 > 0 ? g2_issued - 2 : 0; c < g2_issued; ++c)
            mbar_wait_bounded(&barG2[c & 3], (unsigned)(c >> 2) & 1u);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kDnWarps) {
        tc_fence_after();
        tmem_dealloc(taddr, kDnTmem);
    }
}

// The other factor W (rows x k, FP32) split x = hi + mid + lo into both packed
// layouts, swizzled K-major (sw_off): over k (row r, coordinate c of part w at
// byte w part 2 + sw_off(r, c, 2 KP)), all three parts; and, per chunk of
// kDnNT rows, over the chunk rows (chunk q, element (c, t) of part w at byte
// w part 2 + q KP kDnNT 2 + sw_off(c, t, 2 kDnNT)), all three parts.  Rows
// from `rows` to rows_pad and coordinates from k to KP are zero.
template <int KP>
__global__ void __launch_bounds__(256) dense_pack_kernel(const float *__restrict__ W, int64_t rows, int k,
                                                         int64_t part, __nv_bfloat16 *__restrict__ pk,
                                                         __nv_bfloat16 *__restrict__ pt)
{
    // one CTA per chunk of kDnNT rows, staged in shared memory; every store
    // is a 16-byte unit of eight BF16 values
    __shared__ float tile[kDnNT][KP + 1];
    const int64_t q = blockIdx.x, r0 = q * kDnNT;
    for (int i = threadIdx.x; i < kDnNT * KP; i += blockDim.x) {
        const int r = i / KP, c = i - r * KP;
        tile[r][c] = (r0 + r < rows && c < k) ? W[(r0 + r) * k + c] : 0.f;
    }
    __syncthreads();
    auto pack8 = [](const float (&v)[8], uint4 &h, uint4 &m, uint4 &l) {
        uint32_t hv[4], mv[4], lv[4];
#pragma unroll
        for (int w = 0; w < 8; w += 2) {
            __nv_bfloat16 h0, m0, l0, h1, m1, l1;
            split3(v[w], h0, m0, l0);
            split3(v[w + 1], h1, m1, l1);
            hv[w / 2] = bf2_bits(__halves2bfloat162(h0, h1));
            mv[w / 2] = bf2_bits(__halves2bfloat162(m0, m1));
            lv[w / 2] = bf2_bits(__halves2bfloat162(l0, l1));
        }
        h = make_uint4(hv[0], hv[1], hv[2], hv[3]);
        m = make_uint4(mv[0], mv[1], mv[2], mv[3]);
        l = make_uint4(lv[0], lv[1], lv[2], lv[3]);
    };
    for (int i = threadIdx.x; i < kDnNT * (KP / 8); i += blockDim.x) {
        // K-major over k: row r, coordinates 8 g .. 8 g + 7
        const int r = i / (KP / 8), g = i - r * (KP / 8);
        float v[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) v[w] = tile[r][8 * g + w];
        uint4 h, m, l;
        pack8(v, h, m, l);
        const int64_t o = r0 * KP + sw_off((uint32_t)r, (uint32_t)(8 * g), 2 * KP) / 2;
        *reinterpret_cast<uint4 *>(pk + o) = h;
        *reinterpret_cast<uint4 *>(pk + part + o) = m;
        *reinterpret_cast<uint4 *>(pk + 2 * part + o) = l;
        // K-major over the chunk rows: coordinate c (= i / 8 here), rows 8 t .. 8 t + 7
        const int c = i / (kDnNT / 8), tg = i - c * (kDnNT / 8);
#pragma unroll
        for (int w = 0; w < 8; ++w) v[w] = tile[8 * tg + w][c];
        pack8(v, h, m, l);
        const int64_t ot = q * KP * kDnNT + sw_off((uint32_t)c, (uint32_t)(8 * tg), 2 * kDnNT) / 2;
        *reinterpret_cast<uint4 *>(pt + ot) = h;
        *reinterpret_cast<uint4 *>(pt + part + ot) = m;
        *reinterpret_cast<uint4 *>(pt + 2 * part + ot) = l;
    }
}

// Values outside a column loss's domain (flag 64) or not finite (flag 8).
static __global__ void dense_validate_kernel(const float *__restrict__ A, int64_t lda, int64_t m, int64_t n,
                                             const LossSpec *__restrict__ loss, int *__restrict__ flag)
{
    int f = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m * n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / n, j = i - r * n;
        const float a = A[r * lda + j];
        if (!isfinite(a)) {
            f |= 8;
            continue;
        }
        const LossSpec s = loss[j];
        if ((s.kind == kLossHinge || s.kind == kLossLogistic) && a != 1.f && a != -1.f) f |= 64;
        if (s.kind == kLossOrdinal && (a != floorf(a) || a < 1.f || a > (float)s.levels)) f |= 64;
    }
    if (f) atomicOr(flag, f);
}

// Omega's values (CSR) into a dense table that holds NaN everywhere else:
// one warp per row writes the row's NaN fill, then its entries.
// Rows 0 .. m - 1 of rowptr (which may point into the middle of a pointer
// array: entry indices are absolute) into rows of A; a column index outside
// [0, n) is skipped, so rows whose checks are still running may be scattered.
static __global__ void dense_scatter_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                                            const float *__restrict__ val, int64_t m, int64_t n, int64_t lda,
                                            float *__restrict__ A)
{
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= m) return;
    float *row = A + i * lda;
    for (int64_t c = threadIdx.x & 31; c < lda; c += 32) row[c] = __int_as_float(0x7fffffff);
    __syncwarp();
    for (int e = rowptr[i] + (threadIdx.x & 31); e < rowptr[i + 1]; e += 32) {
        const int32_t j = colidx[e];
        if (j >= 0 && j < n) row[j] = val[e];
    }
}

static __global__ void dense_alpha_kernel(float *__restrict__ alpha, int64_t nseg, float value)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nseg) alpha[s] = value;
}

// Segment s (row s % 128 of own tile s / 128) -> its first partial slot;
// tb holds per tile {first slot, parts}; sc[nseg] = total slots.
static __global__ void dense_segchunk_kernel(int32_t *__restrict__ sc, int64_t nseg, const int64_t *__restrict__ tb,
                                             int64_t total)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nseg) {
        const int64_t t = s / kDnRows;
        sc[s] = (int32_t)(tb[2 * t] + (s - t * kDnRows) * tb[2 * t + 1]);
    } else if (s == nseg) {
        sc[s] = (int32_t)total;
    }
}

namespace {

int dense_width(int k)
{
    for (int K : {16, 32, 64})
        if (k <= K) return K;
    return 0;
}

template <bool XSTEP, bool GRAD, int KP, bool MISS, bool B16, bool WGT>
cudaError_t launch_dense_kp(glrm_s *h, const DenseArgs &a, int nA, unsigned items)
{
    const size_t smem = DnSmem<XSTEP, GRAD, KP>::bytes(nA);
    cudaError_t e = cudaFuncSetAttribute(dense_pass_kernel<XSTEP, GRAD, KP, MISS, B16, WGT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const CUtensorMap *map = reinterpret_cast<const CUtensorMap *>(XSTEP ? h->dn.tmap_x : h->dn.tmap_y);
    dense_pass_kernel<XSTEP, GRAD, KP, MISS, B16, WGT><<<items, kDnThreads, smem, h->stream>>>(a, *map);
    h->launches += 1;
    return cudaGetLastError();
}

// A stages that fit next to the fixed buffers and the kernel's static shared
// memory (at most kDnMaxStages; fewer than 2 is refused by the caller).
template <bool XSTEP, bool GRAD, int KP, bool MISS, bool B16, bool WGT>
int stages_kp(int optin)
{
    using SM = DnSmem<XSTEP, GRAD, KP>;
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, dense_pass_kernel<XSTEP, GRAD, KP, MISS, B16, WGT>) != cudaSuccess) return 0;
    if ((size_t)optin < fa.sharedSizeBytes) return 0;
    const size_t room = (size_t)optin - fa.sharedSizeBytes;
    if (room < SM::bytes(0)) return 0;
    const int n = (int)((room - SM::bytes(0)) / SM::a);
    return n < kDnMaxStages ? n : kDnMaxStages;
}

template <bool XSTEP, bool GRAD>
cudaError_t launch_dense(glrm_s *h, const float *F, float *part_grad, double *part_loss)
{
    const Dense &d = h->dn;
    DenseArgs a;
    a.nown = XSTEP ? h->m : h->n;
    a.nother = XSTEP ? h->n : h->m;
    a.k = h->k;
    a.F = F;
    a.pk = d.pk;
    a.pt = d.pt;
    a.pack_part = d.pack_part;
    a.lossf = d.lossf;
    a.wcol = (const float *)h->lscale;
    a.items = XSTEP ? d.items_x : d.items_y;
    a.blocks = XSTEP ? nullptr : d.blocks_y;
    a.segchunk = XSTEP ? d.segchunk_x : d.segchunk_y;
    a.part_grad = part_grad;
    a.part_loss = part_loss;
    a.err = h->s.err;
    const unsigned tiles = (unsigned)(XSTEP ? d.nitems_x : d.nitems_y);
    int optin = 0;
    cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device);
    if (e != cudaSuccess) return e;
    // the BF16 form's gradient passes take the single-product GEMM2
    const bool b16 = GRAD && h->prec == GLRM_BF16;
#define GLRM_DENSE_GO(KK, MS, B, WG)                                               \
    {                                                                              \
        a.nA = stages_kp<XSTEP, GRAD, KK, MS, B, WG>(optin);                       \
        if (a.nA < 2) return cudaErrorInvalidConfiguration;                        \
        return launch_dense_kp<XSTEP, GRAD, KK, MS, B, WG>(h, a, a.nA, tiles);     \
    }
    // weighted losses (FP32 models only) take the variant that also tests for
    // missing cells, whatever the table: the test never fires on a full one
#define GLRM_DENSE_CASE(KK)                                                        \
    if (d.KP == KK) {                                                              \
        if (a.wcol) GLRM_DENSE_GO(KK, true, false, true)                           \
        if constexpr (GRAD) {                                                      \
            if (b16) {                                                             \
                if (d.missing) GLRM_DENSE_GO(KK, true, true, false)                \
                GLRM_DENSE_GO(KK, false, true, false)                              \
            }                                                                      \
        }                                                                          \
        if (d.missing) GLRM_DENSE_GO(KK, true, false, false)                       \
        GLRM_DENSE_GO(KK, false, false, false)                                     \
    }
    GLRM_DENSE_CASE(16)
    GLRM_DENSE_CASE(32)
    GLRM_DENSE_CASE(64)
#undef GLRM_DENSE_CASE
#undef GLRM_DENSE_GO
    return cudaErrorInvalidValue;
}

cudaError_t dense_pack(glrm_s *h, const float *W, int64_t rows)
{
    const Dense &d = h->dn;
    const int64_t rows_pad = (rows + kDnRows - 1) / kDnRows * kDnRows;
    tmark(h, "dense_pack");
    const unsigned nchunks = (unsigned)(rows_pad / kDnNT);
    if (d.KP == 16)
        dense_pack_kernel<16><<<nchunks, 256, 0, h->stream>>>(W, rows, h->k, d.pack_part, d.pk, d.pt);
    else if (d.KP == 32)
        dense_pack_kernel<32><<<nchunks, 256, 0, h->stream>>>(W, rows, h->k, d.pack_part, d.pk, d.pt);
    else
        dense_pack_kernel<64><<<nchunks, 256, 0, h->stream>>>(W, rows, h->k, d.pack_part, d.pk, d.pt);
    h->launches += 1;
    return cudaGetLastError();
}

// Relative cost of evaluating one entry of a 16- or 32-wide group of columns
// (instructions of the loss blocks, the split of R and the per-entry load and
// sum work): a group whose columns share one kind takes that kind's block; a
// group that mixes kinds takes the per-entry switch and pays for every kind
// present (its lanes diverge).
double group_cost(const std::vector<LossSpec> &loss, int64_t j0, int width)
{
    auto extra = [](int kind) -> double {
        switch (kind) {
        case kLossQuad: return 6;
        case kLossHuber: return 9;
        case kLossHinge: return 4;
        case kLossLogistic: return 24;
        case kLossL1: return 8;
        case kLossQuantile: return 10;
        default: return 12;
        }
    };
    const int64_t n = (int64_t)loss.size(), j1 = std::min<int64_t>(n, j0 + width);
    bool uniform = true;
    unsigned seen = 0;
    for (int64_t j = j0; j < j1; ++j) {
        if (loss[j].kind != loss[j0].kind) uniform = false;
        seen |= 1u << loss[j].kind;
    }
    if (j0 >= j1) return 6;
    if (uniform) return 6 + extra(loss[j0].kind);
    double c = 16;
    for (int kd = 0; kd < kLossKinds; ++kd)
        if (seen >> kd & 1u) c += 2 * extra(kd);
    return c;
}

// Work items of one pass: own tile t (rows t * 128 ..) takes parts_t items,
// each a contiguous range of the other dimension's 64-wide chunks.  Entry
// costs vary with the column losses: along the chunks in the X-step (the
// columns are the other dimension), between the tiles in the Y-step.
//
// Plan: parts sized so items carry about equal cost, about four items per SM
// (no fewer than tiles, none empty), launched in the order of the middle of
// their chunk range (items reading the same chunks of the other factor run
// close together).  One CTA is resident per SM, and a finished CTA's SM takes
// the next item in launch order, so the pass ends when the last SM does:
// the per-item cost target and the number of items split in two (halves
// launched after the rest, to fill the last wave) are chosen by simulating
// that schedule, with each item paying a fixed pipeline fill and drain of
// about 1.3 average chunks on top of its entries.
struct PlanRange {
    int64_t tile, q0, q1;
    bool tail;  // a half of a split item: launched after the others
};

// End of a list schedule of the items on `slots` SMs, or the first end found
// at or beyond `limit`.  A binary heap of the times at which the SMs are free.
double list_schedule_end(const std::vector<double> &t, int slots, double limit)
{
    std::vector<double> h(slots + 1, 0.0);
    h[slots] = HUGE_VAL;
    double end = 0;
    for (double c : t) {
        const double f = h[0] + c;
        end = std::max(end, f);
        if (end >= limit) return end;
        int i = 0;  // the SM's new time sinks from the root
        for (int u = 1; u < slots; u = 2 * i + 1) {
            u += h[u + 1] < h[u];
            if (h[u] >= f) break;
            h[i] = h[u];
            i = u;
        }
        h[i] = f;
    }
    return end;
}

ItemPlan plan_items(int64_t nown, int64_t nother, int sms, const std::vector<double> &tile_cost,
                    const std::vector<double> &chunk_cost)
{
    const int64_t tiles = (nown + kDnRows - 1) / kDnRows;
    const int64_t nch = std::max<int64_t>(1, (nother + kDnNT - 1) / kDnNT);
    std::vector<double> pre(nch + 1, 0.0);
    for (int64_t q = 0; q < nch; ++q) pre[q + 1] = pre[q] + chunk_cost[q];
    double total = 0;
    for (int64_t t = 0; t < tiles; ++t) total += tile_cost[t] * pre[nch];
    const double fill = 1.3 * total / (double)(tiles * nch);
    auto mid = [](const PlanRange &r) { return r.q0 + r.q1; };
    auto order = [&](std::vector<PlanRange>::iterator a, std::vector<PlanRange>::iterator b) {
        std::stable_sort(a, b, [&](const PlanRange &u, const PlanRange &v) { return mid(u) < mid(v); });
    };
    // the tile's chunks in np ranges of about equal cost, at least one chunk each
    auto build = [&](double per_item) {
        std::vector<PlanRange> v;
        for (int64_t t = 0; t < tiles; ++t) {
            int64_t np = (int64_t)std::llround(tile_cost[t] * pre[nch] / per_item);
            np = std::max<int64_t>(1, std::min<int64_t>(np, nch));
            int64_t q = 0;
            for (int64_t i = 0; i < np; ++i) {
                int64_t e = nch;
                if (i + 1 < np) {
                    const double goal = pre[nch] * (double)(i + 1) / (double)np;
                    e = std::lower_bound(pre.begin(), pre.end(), goal) - pre.begin();
                    e = std::max<int64_t>(e, q + 1);
                    e = std::min<int64_t>(e, nch - (np - 1 - i));
                }
                v.push_back({t, q, e, false});
                q = e;
            }
        }
        order(v.begin(), v.end());
        return v;
    };
    // the last `s` items of the launch order split in two at the middle of their
    // cost (those of one chunk stay whole), the halves after all others
    std::vector<PlanRange> w;
    auto split = [&](const std::vector<PlanRange> &v, int64_t s) {
        w.assign(v.begin(), v.end() - s);
        for (auto r = v.end() - s; r != v.end(); ++r)
            if (r->q1 - r->q0 < 2) w.push_back(*r);
        const int64_t whole = (int64_t)w.size();
        for (auto r = v.end() - s; r != v.end(); ++r) {
            if (r->q1 - r->q0 < 2) continue;
            const double goal = 0.5 * (pre[r->q0] + pre[r->q1]);
            int64_t e = std::lower_bound(pre.begin() + r->q0, pre.begin() + r->q1, goal) - pre.begin();
            e = std::max<int64_t>(r->q0 + 1, std::min<int64_t>(e, r->q1 - 1));
            w.push_back({r->tile, r->q0, e, true});
            w.push_back({r->tile, e, r->q1, true});
        }
        order(w.begin() + whole, w.end());
    };
    std::vector<double> t;
    auto finish_time = [&](const std::vector<PlanRange> &v, double limit) {
        t.resize(v.size());
        double sum = 0;
        for (size_t i = 0; i < v.size(); ++i)
            sum += t[i] = tile_cost[v[i].tile] * (pre[v[i].q1] - pre[v[i].q0]) + fill;
        return sum >= limit * sms ? sum / sms : list_schedule_end(t, sms, limit);
    };
    const double per0 = total / (double)std::max<int64_t>(tiles, 4LL * sms);
    std::vector<PlanRange> best = build(per0);
    if ((int64_t)best.size() <= 64LL * sms) {  // beyond that the last wave is a small share
        double best_end = finish_time(best, HUGE_VAL);
        std::vector<PlanRange> last;
        for (int f = 0; f <= 10; ++f) {
            const std::vector<PlanRange> v = build(per0 * (1.0 + 0.03 * f));
            const int64_t n = (int64_t)v.size();
            if (std::equal(v.begin(), v.end(), last.begin(), last.end(), [](const PlanRange &a, const PlanRange &b) {
                    return a.tile == b.tile && a.q0 == b.q0 && a.q1 == b.q1;
                }))
                continue;  // tiles of one part each, say, are those of every target
            last = v;
            for (int g = 0; g <= 24; ++g) {
                split(v, n * g / 24);
                const double limit = best_end * (1.0 - 1e-9), end = finish_time(w, limit);
                if (end < limit) {
                    best_end = end;
                    best = w;
                }
            }
        }
    }
    // parts per tile in chunk order, slots, items in launch order
    ItemPlan pl;
    pl.tiles.assign(2 * tiles, 0);
    std::vector<std::vector<size_t>> by_tile(tiles);
    for (size_t i = 0; i < best.size(); ++i) by_tile[best[i].tile].push_back(i);
    pl.items.resize(best.size());
    for (int64_t t = 0; t < tiles; ++t) {
        std::vector<size_t> &ix = by_tile[t];
        std::sort(ix.begin(), ix.end(), [&](size_t a, size_t b) { return best[a].q0 < best[b].q0; });
        const int64_t rows = std::min<int64_t>(kDnRows, nown - t * kDnRows);
        pl.tiles[2 * t] = pl.slots;
        pl.tiles[2 * t + 1] = (int64_t)ix.size();
        for (size_t p = 0; p < ix.size(); ++p) {
            const PlanRange &r = best[ix[p]];
            DnItem it{};
            it.tile = (int32_t)t;
            it.part = (int32_t)p;
            it.parts = (int32_t)ix.size();
            it.q0 = (int32_t)r.q0;
            it.nq = (int32_t)(r.q1 - r.q0);
            it.base = pl.slots;
            pl.items[ix[p]] = it;
        }
        pl.slots += rows * (int64_t)ix.size();
    }
    return pl;
}

}  // namespace

bool dense_supported(int k) { return dense_width(k) != 0; }

void dense_free(glrm_s *h)
{
    Dense &d = h->dn;
    for (void *p : {(void *)d.A, (void *)d.pk, (void *)d.pt, (void *)d.lossf, (void *)d.segchunk_x,
                    (void *)d.segchunk_y, (void *)d.items_x, (void *)d.items_y, (void *)d.blocks_y})
        if (p) cudaFreeAsync(p, h->stream);
    d = Dense();
}

namespace {

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Tensor maps of A (FP32, dims n x m, row pitch lda): X-step boxes of 32
// columns x 128 rows with the 128-byte swizzle, Y-step boxes of 32 columns x
// 64 rows.  Out-of-range elements load as zero.
cudaError_t encode_maps(glrm_s *h)
{
    static EncodeTiled encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q;
        void *fn = nullptr;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<EncodeTiled>(fn);
    }
    Dense &d = h->dn;
    const cuuint64_t dims[2] = {(cuuint64_t)h->n, (cuuint64_t)h->m};
    const cuuint64_t strides[1] = {(cuuint64_t)d.lda * sizeof(float)};
    const cuuint32_t estr[2] = {1, 1};
    const cuuint32_t box_x[2] = {32, (cuuint32_t)kDnRows};
    const cuuint32_t box_y[2] = {32, (cuuint32_t)kDnNT};
    CUresult r = encode(reinterpret_cast<CUtensorMap *>(d.tmap_x), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, d.A, dims,
                        strides, box_x, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    r = encode(reinterpret_cast<CUtensorMap *>(d.tmap_y), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, d.A, dims, strides,
               box_y, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

// Packs, work items and the segment -> partial-slot tables the shared prox
// and decide kernels read (segment s owns slots segchunk[s] .. segchunk[s + 1]).
cudaError_t dense_prepare(glrm_s *h)
{
    Dense &d = h->dn;
    d.KP = dense_width(h->k);
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e != cudaSuccess) return e;
    const int64_t rows_pad = (std::max(h->m, h->n) + kDnRows - 1) / kDnRows * kDnRows;
    d.pack_part = rows_pad * d.KP;
    if ((e = dalloc(h, &d.pk, 3 * (size_t)d.pack_part * sizeof(__nv_bfloat16))) != cudaSuccess) return e;
    if ((e = dalloc(h, &d.pt, 3 * (size_t)d.pack_part * sizeof(__nv_bfloat16))) != cudaSuccess) return e;
    if ((e = encode_maps(h)) != cudaSuccess) return e;
    // column losses in FP32, each with the kind its 16-column group shares
    // (-1: mixed)
    std::vector<float4> lf(h->n);
    for (int64_t j = 0; j < h->n; ++j) {
        const LossSpec &L = h->loss_host[j];
        int32_t kb = L.kind;
        float kf;
        memcpy(&kf, &kb, sizeof kf);
        lf[j] = make_float4(kf, (float)L.param, (float)L.levels, 0.f);
    }
    const int64_t ngroups = (h->n + kDnNT - 1) / kDnNT * (kDnNT / 16);
    std::vector<int32_t> gk(ngroups, kLossQuad);
    for (int64_t g = 0; g * 16 < h->n; ++g) {
        const LossSpec &L0 = h->loss_host[g * 16];
        int32_t kd = L0.kind;
        for (int64_t j = g * 16; j < std::min<int64_t>(h->n, g * 16 + 16); ++j) {
            const LossSpec &L = h->loss_host[j];
            if (L.kind != L0.kind || (float)L.param != (float)L0.param || L.levels != L0.levels) kd = -1;
        }
        gk[g] = kd;
    }
    for (int64_t j = 0; j < h->n; ++j) {
        const int32_t kd = gk[j / 16];
        memcpy(&lf[j].w, &kd, sizeof kd);
    }
    if ((e = dalloc(h, &d.lossf, (size_t)h->n * sizeof(float4))) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(d.lossf, lf.data(), lf.size() * sizeof(float4), cudaMemcpyHostToDevice,
                             h->stream)) != cudaSuccess)
        return e;

    // X-step: chunks are 64 columns (four 16-column groups), tiles alike;
    // Y-step: tiles are 128 columns (four 32-column warps), chunks alike
    const int64_t tiles_x = (h->m + kDnRows - 1) / kDnRows, tiles_y = (h->n + kDnRows - 1) / kDnRows;
    const int64_t nch_x = std::max<int64_t>(1, (h->n + kDnNT - 1) / kDnNT);
    const int64_t nch_y = std::max<int64_t>(1, (h->m + kDnNT - 1) / kDnNT);
    DensePlan &pl = h->dnplan;  // depends only on m, n, the losses and the device: made once per handle
    if (!pl.ready) {
        std::vector<double> cx(nch_x, 0.0), cy(tiles_y, 0.0);
        for (int64_t q = 0; q < nch_x; ++q)
            for (int g = 0; g < kDnNT / 16; ++g) cx[q] += 16 * group_cost(h->loss_host, q * kDnNT + 16 * g, 16);
        // Y-step tiles: the 32-column blocks in order of cost (then loss kind),
        // four to a tile.  A tile advances at the pace of its slowest block: a
        // block's four warps (warp indices equal mod 4) share one SM
        // sub-partition, and the four blocks move through the chunks in step;
        // tiles of like blocks leave no sub-partition waiting on another.
        const int64_t nb = (h->n + 31) / 32;
        std::vector<double> bc(nb);
        std::vector<int64_t> order(nb);
        for (int64_t b = 0; b < nb; ++b) {
            bc[b] = group_cost(h->loss_host, 32 * b, 32);
            order[b] = b;
        }
        std::stable_sort(order.begin(), order.end(), [&](int64_t u, int64_t v) {
            return bc[u] != bc[v] ? bc[u] < bc[v] : h->loss_host[32 * u].kind < h->loss_host[32 * v].kind;
        });
        pl.blocks_y.assign(4 * tiles_y, -1);
        std::vector<int64_t> tile_of(nb);
        for (int64_t i = 0; i < nb; ++i) {
            pl.blocks_y[i] = (int32_t)order[i];
            tile_of[order[i]] = i / 4;
            cy[i / 4] = std::max(cy[i / 4], kDnRows * bc[order[i]]);
        }
        pl.x = plan_items(h->m, h->n, sms, std::vector<double>(tiles_x, 1.0), cx);
        pl.y = plan_items(h->n, h->m, sms, cy, std::vector<double>(nch_y, 1.0));
        // Y slots in column order: column j owns parts-of-its-tile slots
        pl.seg_y.resize(h->n + 1);
        int64_t run = 0;
        for (int64_t j = 0; j < h->n; ++j) {
            pl.seg_y[j] = (int32_t)std::min<int64_t>(run, INT32_MAX);
            run += pl.y.tiles[2 * tile_of[j / 32] + 1];
        }
        pl.seg_y[h->n] = (int32_t)std::min<int64_t>(run, INT32_MAX);
        pl.y.slots = run;
        pl.ready = true;
    }
    const ItemPlan &px = pl.x, &py = pl.y;
    if (px.slots > INT32_MAX || py.slots > INT32_MAX) return cudaErrorInvalidValue;
    d.nitems_x = (int64_t)px.items.size();
    d.nitems_y = (int64_t)py.items.size();
    d.slots_x = px.slots;
    d.slots_y = py.slots;
    d.slots = std::max(px.slots, py.slots);
    int64_t *tb = nullptr;
    if ((e = dalloc(h, &d.items_x, px.items.size() * sizeof(DnItem))) != cudaSuccess) return e;
    if ((e = dalloc(h, &d.items_y, py.items.size() * sizeof(DnItem))) != cudaSuccess) return e;
    if ((e = dalloc(h, &d.blocks_y, pl.blocks_y.size() * sizeof(int32_t))) != cudaSuccess) return e;
    if ((e = dalloc(h, &d.segchunk_x, (size_t)(h->m + 1) * sizeof(int32_t))) != cudaSuccess) return e;
    if ((e = dalloc(h, &d.segchunk_y, (size_t)(h->n + 1) * sizeof(int32_t))) != cudaSuccess) return e;
    if ((e = dalloc(h, &tb, px.tiles.size() * sizeof(int64_t))) != cudaSuccess) return e;
    const std::pair<const void *, void *> copies[5] = {{px.items.data(), d.items_x},
                                                       {py.items.data(), d.items_y},
                                                       {pl.blocks_y.data(), d.blocks_y},
                                                       {pl.seg_y.data(), d.segchunk_y},
                                                       {px.tiles.data(), tb}};
    const size_t sizes[5] = {px.items.size() * sizeof(DnItem), py.items.size() * sizeof(DnItem),
                             pl.blocks_y.size() * sizeof(int32_t), pl.seg_y.size() * sizeof(int32_t),
                             px.tiles.size() * sizeof(int64_t)};
    for (int c = 0; c < 5; ++c)
        if ((e = cudaMemcpyAsync(copies[c].second, copies[c].first, sizes[c], cudaMemcpyHostToDevice, h->stream)) !=
            cudaSuccess)
            return e;
    dense_segchunk_kernel<<<(unsigned)((h->m + 256) / 256), 256, 0, h->stream>>>(d.segchunk_x, h->m, tb, px.slots);
    e = cudaGetLastError();
    dfree(tb, h->stream);
    return e;
}

cudaError_t launch_dense_scatter(glrm_s *h, float *A, int64_t lda, cudaStream_t st, int64_t r0, int64_t r1)
{
    if (r1 < 0) r1 = h->m;
    if (r1 <= r0) return cudaSuccess;
    dense_scatter_kernel<<<(unsigned)((r1 - r0 + 7) / 8), 256, 0, st>>>(
        h->csr.ptr + r0, h->csr.idx, (const float *)h->csr.val, r1 - r0, h->n, lda, A + r0 * lda);
    h->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_dense_validate(const float *A, int64_t lda, int64_t m, int64_t n, const LossSpec *loss,
                                  int *flag, cudaStream_t st)
{
    const int64_t total = m * n;
    const unsigned nb = (unsigned)std::min<int64_t>(4096, std::max<int64_t>(1, (total + 255) / 256));
    dense_validate_kernel<<<nb, 256, 0, st>>>(A, lda, m, n, loss, flag);
    return cudaGetLastError();
}

// alpha = 1 / max(n_i, 1): every row has n observed entries, every column m.
cudaError_t dense_reset_steps(glrm_s *h)
{
    dense_alpha_kernel<<<(unsigned)((h->m + 255) / 256), 256, 0, h->stream>>>(
        (float *)h->alpha_x, h->m, 1.f / (float)std::max<int64_t>(h->n, 1));
    dense_alpha_kernel<<<(unsigned)((h->n + 255) / 256), 256, 0, h->stream>>>(
        (float *)h->alpha_y, h->n, 1.f / (float)std::max<int64_t>(h->m, 1));
    h->launches += 2;
    return cudaGetLastError();
}

cudaError_t dense_half_step(glrm_s *h, bool xstep)
{
    const int64_t nseg = xstep ? h->m : h->n;
    const int32_t *segchunk = xstep ? h->dn.segchunk_x : h->dn.segchunk_y;
    float *F = (float *)(xstep ? h->X : h->Yt);
    const float *W = (const float *)(xstep ? h->Yt : h->X);
    float *alpha = (float *)(xstep ? h->alpha_x : h->alpha_y);
    const int rk = reg_code(h, xstep);
    const float rw = (float)(xstep ? h->rx_w : h->ry_w);
    Scratch &s = h->s;
    cudaStream_t st = h->stream;
    cudaError_t e = dense_pack(h, W, xstep ? h->n : h->m);
    if (e != cudaSuccess) return e;
    tmark(h, xstep ? "dense_grad_x" : "dense_grad_y");
    e = xstep ? launch_dense<true, true>(h, F, (float *)s.part_grad, s.part_loss)
              : launch_dense<false, true>(h, F, (float *)s.part_grad, s.part_loss);
    if (e != cudaSuccess) return e;
    tmark(h, xstep ? "prox_x" : "prox_y");
    e = launch_prox<float>(nseg, segchunk, (const float *)s.part_grad, s.part_loss, F, alpha, h->k, rk, rw,
                           (float *)s.cand, s.f_old, s.r_old, s.r_new, st, xstep ? h->dn.slots_x : h->dn.slots_y);
    if (e != cudaSuccess) return e;
    tmark(h, xstep ? "dense_loss_x" : "dense_loss_y");
    e = xstep ? launch_dense<true, false>(h, (const float *)s.cand, nullptr, s.part_loss2)
              : launch_dense<false, false>(h, (const float *)s.cand, nullptr, s.part_loss2);
    if (e != cudaSuccess) return e;
    tmark(h, xstep ? "decide_x" : "decide_y");
    e = launch_decide<float>(nseg, segchunk, s.part_loss2, s.f_old, s.r_old, s.r_new, (const float *)s.cand, F,
                             alpha, h->k, xstep ? s.kept_obj_x : s.kept_obj_y, xstep ? s.kept_reg_x : s.kept_reg_y,
                             xstep ? s.acc_x : s.acc_y, st);
    tmark(h, nullptr);
    h->launches += 2;
    return e;
}

cudaError_t dense_objective_at(glrm_s *h, const float *X, const float *Yt, double *out)
{
    Scratch &s = h->s;
    cudaError_t e = dense_pack(h, Yt, h->n);
    if (e != cudaSuccess) return e;
    tmark(h, "dense_objective");
    if ((e = launch_dense<true, false>(h, X, nullptr, s.part_loss)) != cudaSuccess) return e;
    tmark(h, "reduce");
    reduce_kernel<float><<<reduce_blocks(h->dn.slots_x + (h->m + h->n) * h->k), 256, 0, h->stream>>>(
        s.part_loss, h->dn.slots_x, nullptr, 0, X, h->m, reg_code(h, true), (float)h->rx_w, Yt, h->n,
        reg_code(h, false), (float)h->ry_w, h->k, nullptr, 0, nullptr, 0, s.red_part, s.red_cnt, s.ticket, out,
        nullptr);
    tmark(h, nullptr);
    h->launches += 1;
    return cudaGetLastError();
}

cudaError_t dense_grad_at(glrm_s *h, const float *X, const float *Yt, float *GX, float *GYt, bool reg,
                          const double *scale)
{
    Scratch &s = h->s;
    cudaError_t e = dense_pack(h, Yt, h->n);
    if (e != cudaSuccess) return e;
    tmark(h, "dense_grad_x");
    if ((e = launch_dense<true, true>(h, X, (float *)s.part_grad, s.part_loss)) != cudaSuccess) return e;
    tmark(h, "grad_seg_x");
    if ((e = launch_seg_grad<float>(h->m, h->dn.segchunk_x, (const float *)s.part_grad, X, h->k, reg_code(h, true),
                                    (float)h->rx_w, reg, scale, GX, h->stream, h->dn.slots_x)) != cudaSuccess)
        return e;
    if ((e = dense_pack(h, X, h->m)) != cudaSuccess) return e;
    tmark(h, "dense_grad_y");
    if ((e = launch_dense<false, true>(h, Yt, (float *)s.part_grad, s.part_loss)) != cudaSuccess) return e;
    tmark(h, "grad_seg_y");
    e = launch_seg_grad<float>(h->n, h->dn.segchunk_y, (const float *)s.part_grad, Yt, h->k, reg_code(h, false),
                               (float)h->ry_w, reg, scale, GYt, h->stream, h->dn.slots_y);
    tmark(h, nullptr);
    h->launches += 2;
    return e;
}

}  // namespace glrm
