// Gradient pass of the BF16 form for large ranks (48 < k <= 64, k a multiple
// of 8) with the gathered rows staged in shared memory by cp.async.
//
// Four lanes share an entry, as in the passes of glrm_engine.cuh, and hold its
// coordinates interleaved by 16-byte units.  Every lane copies exactly the
// units it will read, to a place of its own in shared memory (unit h of block
// t at ((t H + h) 32 + lane) 16 bytes): no bank conflicts, and no lane waits
// for another's copies, only for its own (cp.async groups).  The copies need
// no registers, so a warp streams its chunk's entries through a ring of kRing
// blocks of eight, where the register version keeps one gather in flight and
// waits on its latency.  200,000 x 20,000 completion table, k = 64: 1.35 -> 0.93
// ms (X-step) and 1.05 -> 0.81 ms (Y-step).  The same ring with FP32 rows
// (twice the bytes) was slower than the registers: 6.0 against 5.0 ms for the
// 2e8-entry Y-step gradient pass, 6.3 against 3.2 ms for the loss pass, which
// already fills the L1 pipe.
#include "glrm_engine.cuh"
#include "glrm_tiled.cuh"

namespace glrm {

constexpr int kRing = 8;       // blocks of eight entries in flight per warp
constexpr int kPassWarps = 4;  // warps per CTA of the streaming pass

template <int K>
struct StLane {
    static constexpr int S = K / 4;    // coordinates per lane
    static constexpr int VW = 8;       // values per 16-byte unit
    static constexpr int H = S / VW;   // units per lane
    static_assert(S % VW == 0, "whole units");
    __device__ static __forceinline__ int coord(int s, int gl) { return VW * ((s / VW) * 4 + gl) + s % VW; }
};

__device__ __forceinline__ void cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A row's coordinates of lane gl, FP32 from global memory (0 beyond k).
template <int K>
__device__ __forceinline__ void st_own(float (&v)[K / 4], const float *__restrict__ row, int gl, int k)
{
#pragma unroll
    for (int s = 0; s < K / 4; ++s) {
        const int c = StLane<K>::coord(s, gl);
        v[s] = c < k ? __ldg(row + c) : 0.f;
    }
}

// Request a row's units of lane gl into its place; units beyond k are zeroed.
template <int K>
__device__ __forceinline__ void st_request(unsigned char *place, const __nv_bfloat16 *__restrict__ W, int64_t j, int gl,
                                           int k)
{
    using LN = StLane<K>;
#pragma unroll
    for (int h = 0; h < LN::H; ++h) {
        const int c = LN::VW * (4 * h + gl);
        if (c < k) cp16(place + h * 512, W + j * k + c);
        else *reinterpret_cast<uint4 *>(place + h * 512) = make_uint4(0, 0, 0, 0);
    }
}

template <int K>
__device__ __forceinline__ void st_read(float (&w)[K / 4], const unsigned char *place)
{
#pragma unroll
    for (int h = 0; h < StLane<K>::H; ++h) {
        const uint4 v = *reinterpret_cast<const uint4 *>(place + h * 512);
        const uint32_t t[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            w[8 * h + 2 * q] = __uint_as_float(t[q] << 16);
            w[8 * h + 2 * q + 1] = __uint_as_float(t[q] & 0xffff0000u);
        }
    }
}

// Dot product over an entry's four lanes (every lane gets the sum).
template <int S>
__device__ __forceinline__ float st_dot(const float (&f)[S], const float (&w)[S])
{
    unsigned long long a = 0ull;
#pragma unroll
    for (int s = 0; s < S; s += 2) a = ffma2(pk2(f[s], f[s + 1]), pk2(w[s], w[s + 1]), a);
    float lo, hi;
    upk2(a, lo, hi);
    float u = lo + hi;
    u += shfl_xor(u, 1);
    u += shfl_xor(u, 2);
    return u;
}

template <int S>
__device__ __forceinline__ void st_axpy(float (&g)[S], float d, const float (&w)[S])
{
    const unsigned long long dd = pk2(d, d);
#pragma unroll
    for (int s = 0; s < S; s += 2)
        upk2(ffma2(dd, pk2(w[s], w[s + 1]), pk2(g[s], g[s + 1])), g[s], g[s + 1]);
}

// Partial gradient and loss at F of a warp's chunk; `sel` / `want` as in
// pass_kernel.  uniform: every column has loss[0].
template <int K, bool XSTEP>
__global__ void __launch_bounds__(kPassWarps * 32)
staged_pass_kernel(int64_t nchunks, const int4 *__restrict__ chunks, const int32_t *__restrict__ order,
                   const int32_t *__restrict__ idx, const float *__restrict__ val, const float *__restrict__ F,
                   const __nv_bfloat16 *__restrict__ W, int k, const LossSpecF *__restrict__ loss, bool uniform,
                   float *__restrict__ part_grad, double *__restrict__ part_loss, const int32_t *__restrict__ sel,
                   int want)
{
    using LN = StLane<K>;
    constexpr int S = LN::S, H = LN::H;
    extern __shared__ __align__(16) unsigned char st_raw[];
    __shared__ float ash[kPassWarps][kRing][32];
    __shared__ int jsh[XSTEP ? kPassWarps : 1][XSTEP ? kRing : 1][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, gl = lane & 3, grp = lane >> 2;
    const int64_t lin = (int64_t)blockIdx.x * kPassWarps + wid;
    if (lin >= nchunks) return;
    const int64_t c = order ? (int64_t)__ldg(order + lin) : lin;
    const int4 ch = chunks[c];
    if (sel && ((__ldg(sel + ch.x) != 0) != (want != 0))) return;  // another launch takes this segment
    unsigned char *ring = st_raw + (size_t)wid * kRing * H * 512 + lane * 16;
    float f[S], g[S];
    st_own<K>(f, F + (int64_t)ch.x * k, gl, k);
#pragma unroll
    for (int s = 0; s < S; ++s) g[s] = 0.f;
    LossSpecF sp = loss[XSTEP ? 0 : ch.x];
    const int len = ch.z - ch.y, nb = (len + 7) / 8;
    // indices and values come 32 entries at a time, one batch ahead
    int ji = 0, jn = 0;
    float ai = 0.f, an = 0.f;
    auto batch = [&](int q, int &j, float &a) {
        const int e = ch.y + 32 * q + lane;
        if (e < ch.z) {
            j = __ldg(idx + e);
            a = __ldg(val + e);
        }
    };
    batch(0, ji, ai);
    batch(1, jn, an);
    auto issue = [&](int t) {
        const int src = (t & 3) * 8 + grp;
        const int j = __shfl_sync(0xffffffffu, ji, src);
        const float a = __shfl_sync(0xffffffffu, ai, src);
        const int r = t & (kRing - 1);
        if (8 * t + grp < len) st_request<K>(ring + r * H * 512, W, j, gl, k);
        ash[wid][r][lane] = a;
        if constexpr (XSTEP) jsh[wid][r][lane] = j;
        if ((t & 3) == 3) {
            ji = jn;
            ai = an;
            batch(t / 4 + 2, jn, an);
        }
    };
    for (int t = 0; t < kRing - 1; ++t) {
        if (t < nb) issue(t);
        cp_commit();
    }
    float l0 = 0.f;
    for (int t = 0; t < nb; ++t) {
        if (t + kRing - 1 < nb) issue(t + kRing - 1);
        cp_commit();
        cp_wait<kRing - 1>();
        const int r = t & (kRing - 1);
        const bool in = 8 * t + grp < len;
        float w[S];
        st_read<K>(w, ring + r * H * 512);
        const float u = st_dot<S>(f, w);
        if (in) {
            const float a = ash[wid][r][lane];
            if constexpr (XSTEP) {
                if (!uniform) sp = loss[jsh[wid][r][lane]];
            }
            float L;
            const float d = loss_deriv<float>(sp, u, a, L);
            if (gl == 0) l0 += L;
            st_axpy<S>(g, d, w);
        }
    }
    cp_wait<0>();
#pragma unroll
    for (int s = 0; s < S; ++s) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) g[s] += shfl_xor(g[s], o);
    }
    if (grp == 0) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int cc = LN::coord(s, gl);
            if (cc < k) part_grad[c * k + cc] = g[s];
        }
    }
    const double s0 = warp_sum((double)l0);
    if (lane == 0) part_loss[c] = s0;
}

// 48 < k <= 64, whole 16-byte units of BF16 and an aligned copy.
bool staged_bf16_ok(int k, const void *W)
{
    return k > 48 && k <= 64 && k % 8 == 0 && reinterpret_cast<uintptr_t>(W) % 16 == 0;
}

template <bool XSTEP>
static cudaError_t go_pass(glrm_s *h, const Orient &o, const float *F, const __nv_bfloat16 *W, float *pg, double *pl,
                           const int32_t *sel, int want)
{
    if (o.nchunks == 0) return cudaSuccess;
    auto kern = staged_pass_kernel<64, XSTEP>;
    constexpr size_t smem = (size_t)kPassWarps * kRing * StLane<64>::H * 512;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<blocks_for(o.nchunks, kPassWarps), kPassWarps * 32, smem, h->stream>>>(
        o.nchunks, o.chunks, o.order, o.idx, (const float *)o.val, F, W, h->k, h->loss_f, h->loss_uniform, pg, pl, sel,
        want);
    return cudaGetLastError();
}

cudaError_t staged_pass_bf16(glrm_s *h, bool xstep, const float *F, const __nv_bfloat16 *W, float *pg, double *pl,
                             const int32_t *sel, int want)
{
    return xstep ? go_pass<true>(h, h->csr, F, W, pg, pl, sel, want) : go_pass<false>(h, h->csc, F, W, pg, pl, sel, want);
}

}  // namespace glrm
