// Alternating minimisation for quadratic loss with gamma ||.||^2 on both
// factors (Algorithm 1 of Udell et al., with the row and column problems of
// Section 2.4 solved exactly, the Gram matrices restricted to each row's or
// column's observed entries as in Section 2.5).  A half-step solves, for
// every segment s (row in the X-step, column in the Y-step),
//     (sum_{e in s} w_e w_e^T + gamma I) f_s = sum_{e in s} a_e w_e.
// Launch 1 (per chunk): partial Gram lower triangle and right-hand side in
// the element type.  Launch 2 (per segment): sum of the partials in a fixed
// order, then the solve: FP64 models (and prox-prox) an FP64 Cholesky
// factorisation and two triangular solves in shared memory, one warp per
// segment; FP32 models the refined solve of glrm_spd.cuh, K lanes per segment,
// with the FP64 factorisation for the systems it does not settle.
#pragma once

#include "glrm_engine.cuh"
#include "glrm_spd.cuh"

namespace glrm {

constexpr int kAlsWarps = 4;

template <int K>
struct Tri {
    static constexpr int N = K * (K + 1) / 2;  // lower-triangle entries
    static constexpr int P = N + K;            // + right-hand side
};

// Row r and column c (c <= r) of lower-triangle entry p (row-major order).
__device__ __forceinline__ void tri_rc(int p, int &r, int &c)
{
    r = (int)((sqrtf(8.f * (float)p + 1.f) - 1.f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= p) ++r;
    while (r * (r + 1) / 2 > p) --r;
    c = p - r * (r + 1) / 2;
}

// One warp per chunk.  Rows of the other factor come in batches of kRows
// through two shared-memory buffers filled by cp.async (16-byte pieces when
// the rows allow it: eight lanes fetch one 128-byte row, where a lane per row
// touched 32 lines with every load); the 32 / K lane groups take the batch's
// entries in turn, each accumulating its whole K x K tile in registers
// (GramTile), and are summed at the end.  On the 100,000 x 20,000 completion
// table (k = 32, 2e7 entries) 4.5 -> 0.94 (rows) and 4.7 -> 1.02 ms (columns).
// Bound by the shared-memory reads of the tiles' operands (that pipe is 79 / 67%
// busy, the FP32 multiply-adds of the full square, 1,024 per entry, 40 / 37%).
template <class T, int K>
__global__ void __launch_bounds__(kAlsWarps * 32)
als_gram_kernel(int64_t nchunks, const int4 *__restrict__ chunks, const int32_t *__restrict__ idx,
                const T *__restrict__ val, const T *__restrict__ W, int k, bool vec, T *__restrict__ part)
{
    using TR = Tri<K>;
    using GT = GramTile<T, K>;
    constexpr int kRows = sizeof(T) == 4 ? 32 : 16;   // entries per batch
    constexpr int GR = 32 / K;                        // lane groups
    constexpr int PPR = K * (int)sizeof(T) / 16;      // 16-byte pieces per row
    __shared__ __align__(16) T wsh[kAlsWarps][2][kRows][K];
    __shared__ T ash[kAlsWarps][2][kRows];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t c = (int64_t)blockIdx.x * kAlsWarps + wid;
    if (c >= nchunks) return;
    const int4 ch = chunks[c];
    // coordinates from k to K are zero and stay so
    for (int q = lane; q < 2 * kRows * K; q += 32) (&wsh[wid][0][0][0])[q] = T(0);
    __syncwarp();
    GT g;
    g.init(lane % K);
    int j = 0;
    T a = T(0);
    auto fetch = [&](int base) {  // index and value of entry base + lane
        if (lane < kRows && base + lane < ch.z) {
            j = __ldg(idx + base + lane);
            a = __ldg(val + base + lane);
        }
    };
    auto issue = [&](int buf, int base) {  // the fetched batch's rows into a buffer
        const int cnt = min(kRows, ch.z - base);
        if (vec) {
#pragma unroll
            for (int q = 0; q < kRows * PPR / 32; ++q) {
                const int row = (q * 32 + lane) / PPR, piece = (q * 32 + lane) % PPR;
                const int jr = __shfl_sync(0xffffffffu, j, row);
                if (row < cnt && piece * (16 / (int)sizeof(T)) < k)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                     smem_u32(&wsh[wid][buf][row][piece * (16 / (int)sizeof(T))])),
                                 "l"(W + (int64_t)jr * k + piece * (16 / (int)sizeof(T)))
                                 : "memory");
            }
        } else {
            for (int e = 0; e < cnt; ++e) {
                const int jr = __shfl_sync(0xffffffffu, j, e);
                if (lane < k)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(&wsh[wid][buf][e][lane])),
                                 "l"(W + (int64_t)jr * k + lane), "n"((int)sizeof(T))
                                 : "memory");
            }
        }
        if (lane < kRows) ash[wid][buf][lane] = a;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(ch.y);
    issue(0, ch.y);
    fetch(ch.y + kRows);
    int buf = 0;
    for (int base = ch.y; base < ch.z; base += kRows, buf ^= 1) {
        if (base + kRows < ch.z) {
            issue(buf ^ 1, base + kRows);
            fetch(base + 2 * kRows);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        const int cnt = min(kRows, ch.z - base);
#pragma unroll 2
        for (int t = lane / K; t < cnt; t += GR) g.add(wsh[wid][buf][t], ash[wid][buf][t]);
        __syncwarp();
    }
#pragma unroll
    for (int o = K; o < 32; o <<= 1) {
#pragma unroll
        for (int i = 0; i < GT::TR; ++i) {
            g.b[i] += shfl_xor(g.b[i], o);
#pragma unroll
            for (int q = 0; q < GT::TC; ++q) g.acc[i][q] += shfl_xor(g.acc[i][q], o);
        }
    }
    if (lane >= K) return;
    T *out = part + c * TR::P;
#pragma unroll
    for (int i = 0; i < GT::TR; ++i) {
        const int r = g.r0 + i;
#pragma unroll
        for (int q = 0; q < GT::TC; ++q)
            if (g.c0 + q <= r) out[r * (r + 1) / 2 + g.c0 + q] = g.acc[i][q];
        if (g.c0 == 0) out[TR::N + r] = g.b[i];
    }
}

template <class T, int K>
__global__ void __launch_bounds__(kAlsWarps * 32)
als_solve_kernel(int64_t nseg, const int32_t *__restrict__ segchunk, const T *__restrict__ part,
                 int k, double gamma, T *__restrict__ F, int *__restrict__ err)
{
    using TR = Tri<K>;
    __shared__ double G[kAlsWarps][K][K + 1];
    __shared__ double b[kAlsWarps][K];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t s = (int64_t)blockIdx.x * kAlsWarps + wid;
    if (s >= nseg) return;
    const int cb = segchunk[s], ce = segchunk[s + 1];
    for (int p = lane; p < TR::N; p += 32) {
        int r, c;
        tri_rc(p, r, c);
        double v = 0.0;
        for (int q = cb; q < ce; ++q) v += (double)part[(int64_t)q * TR::P + p];
        if (r == c) v += gamma;
        G[wid][r][c] = v;
    }
    if (lane < K) {
        double v = 0.0;
        for (int q = cb; q < ce; ++q) v += (double)part[(int64_t)q * TR::P + TR::N + lane];
        b[wid][lane] = v;
    }
    __syncwarp();
    // unused rows / columns beyond k become identity rows of a K x K system
    for (int c = k + lane; c < K; c += 32) {
        for (int q = 0; q < c; ++q) G[wid][c][q] = 0.0;
        G[wid][c][c] = 1.0;
        b[wid][c] = 0.0;
    }
    __syncwarp();
    // a failed factorisation keeps the segment's factor and raises the flag
    if (!warp_cholesky_solve<K, K + 1>(G[wid], b[wid])) {
        if (lane == 0) atomicOr(err, kErrPivot);
        return;
    }
    if (lane < k) F[s * k + lane] = (T)b[wid][lane];
}

// FP32 models: K lanes per segment (32 / K segments per warp), the refined
// solve of glrm_spd.cuh.  The warps walk the segments with a grid stride, so
// the (row, column) of a lane's triangle entries are worked out once.  With
// the FP64 factorisation for every system the FP64 pipe was 85% busy; on the
// 100,000 systems of the k = 32 completion table 4.83 -> 1.10 ms.
template <int K>
__global__ void __launch_bounds__(kAlsWarps * 32)
als_solve_refined_kernel(int64_t nseg, const int32_t *__restrict__ segchunk, const float *__restrict__ part, int k,
                         double gamma, float *__restrict__ F, int *__restrict__ err)
{
    using TR = Tri<K>;
    constexpr int GR = 32 / K, NQ = (TR::N + K - 1) / K;
    extern __shared__ __align__(16) unsigned char spd_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, grp = lane / K, lr = lane % K;
    SpdSmem<K> &S = reinterpret_cast<SpdSmem<K> *>(spd_raw)[wid * GR + grp];
    int rc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        int r, c;
        tri_rc(lr + K * q < TR::N ? lr + K * q : 0, r, c);
        rc[q] = r << 8 | c;
    }
    const int64_t step = (int64_t)gridDim.x * kAlsWarps * GR;
    for (int64_t s0 = ((int64_t)blockIdx.x * kAlsWarps + wid) * GR; s0 < nseg; s0 += step) {
        const int64_t s = s0 + grp;
        const bool live = s < nseg;
        const int cb = live ? segchunk[s] : 0, ce = live ? segchunk[s + 1] : 0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int p = lr + K * q;
            if (p < TR::N) {
                const int r = rc[q] >> 8, c = rc[q] & 0xff;
                double v = 0.0;
                float f = 0.f;
                if (ce - cb == 1) {
                    f = part[(int64_t)cb * TR::P + p];
                    v = (double)f;
                } else {
                    for (int t = cb; t < ce; ++t) {
                        const float w = part[(int64_t)t * TR::P + p];
                        v += (double)w;
                        f += w;
                    }
                }
                if (r == c) {  // unused rows / columns beyond k: an identity
                    v = r < k ? v + gamma : 1.0;
                    f = r < k ? f + (float)gamma : 1.f;
                }
                S.G[r * K + c] = S.G[c * K + r] = v;
                S.L[r * (K + 1) + c] = S.L[c * (K + 1) + r] = f;
            }
        }
        double b = 0.0;
        if (lr < k)
            for (int t = cb; t < ce; ++t) b += (double)part[(int64_t)t * TR::P + TR::N + lr];
        S.b[lr] = b;
        __syncwarp();
        double x;
        bool ok = spd_solve_refined<K>(S, x);
        if (__any_sync(0xffffffffu, live && !ok)) {
            // the systems not settled, one after the other: FP64 Cholesky (a
            // failed one keeps the segment's factor and raises the flag)
            for (int g = 0; g < GR; ++g) {
                if (!(__shfl_sync(0xffffffffu, live && !ok ? 1 : 0, g * K))) continue;
                SpdSmem<K> &Q = reinterpret_cast<SpdSmem<K> *>(spd_raw)[wid * GR + g];
                const bool solved =
                    warp_cholesky_solve<K, K>(reinterpret_cast<double(*)[K]>(Q.G), Q.b);
                if (grp == g) {
                    x = Q.b[lr];
                    ok = solved;
                    if (!solved && lr == 0) atomicOr(err, kErrPivot);
                }
                __syncwarp();
            }
        }
        if (live && ok && lr < k) F[s * k + lr] = (float)x;
        __syncwarp();
    }
}

// Prox-prox update for quadratic loss (Section 7.2, "Prox-prox method"; the
// cached factorisation of Section 7.3), one warp per segment: with the
// segment's Gram matrix G and right-hand side b (the ALS partials), factor
// M = 2 alpha G + I once in FP64, then `inner` times
//     f <- prox_{alpha r}(M^{-1} (2 alpha b + f)),
// prox_{alpha f}(f) = argmin alpha sum_e (f . w_e - a_e)^2 + ||f' - f||^2 / 2
// being M^{-1}(2 alpha b + f).  A failed factorisation keeps the factor and
// raises the status flag.
template <class T, int K>
__global__ void __launch_bounds__(kAlsWarps * 32)
proxprox_solve_kernel(int64_t nseg, const int32_t *__restrict__ segchunk, const T *__restrict__ part,
                      int k, double alpha, int inner, int rkind, double rw, T *__restrict__ F,
                      int *__restrict__ err)
{
    using TR = Tri<K>;
    __shared__ double G[kAlsWarps][K][K + 1];
    __shared__ double b[kAlsWarps][K];
    __shared__ double x[kAlsWarps][K];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t s = (int64_t)blockIdx.x * kAlsWarps + wid;
    if (s >= nseg) return;
    const int cb = segchunk[s], ce = segchunk[s + 1];
    for (int p = lane; p < TR::N; p += 32) {
        int r, c;
        tri_rc(p, r, c);
        double v = 0.0;
        for (int q = cb; q < ce; ++q) v += (double)part[(int64_t)q * TR::P + p];
        G[wid][r][c] = 2.0 * alpha * v + (r == c ? 1.0 : 0.0);
    }
    if (lane < K) {
        double v = 0.0;
        for (int q = cb; q < ce; ++q) v += (double)part[(int64_t)q * TR::P + TR::N + lane];
        b[wid][lane] = 2.0 * alpha * v;
    }
    __syncwarp();
    // unused rows / columns beyond k become identity rows of a K x K system
    for (int c = k + lane; c < K; c += 32) {
        for (int q = 0; q < c; ++q) G[wid][c][q] = 0.0;
        G[wid][c][c] = 1.0;
        b[wid][c] = 0.0;
    }
    __syncwarp();
    if (!warp_cholesky_factor<K, K + 1>(G[wid])) {
        if (lane == 0) atomicOr(err, kErrPivot);
        return;
    }
    double f = lane < k ? (double)F[s * k + lane] : 0.0;
    for (int it = 0; it < inner; ++it) {
        if (lane < K) x[wid][lane] = b[wid][lane] + f;
        __syncwarp();
        warp_cholesky_subst<K, K + 1>(G[wid], x[wid]);
        if (lane < K) f = lane < k ? prox1<double>(reg_kind_at(rkind, lane, k), rw, alpha, x[wid][lane]) : 0.0;
        __syncwarp();
    }
    if (lane < k) F[s * k + lane] = (T)f;
}

// Whether a factor's rows can be copied in 16-byte pieces.
template <class T>
bool gram_vec(const T *W, int k)
{
    return k * sizeof(T) % 16 == 0 && reinterpret_cast<uintptr_t>(W) % 16 == 0;
}

template <class T, int K>
cudaError_t launch_als_half(glrm_s *h, bool xstep, double gamma)
{
    const Orient &o = xstep ? h->csr : h->csc;
    T *F = (T *)(xstep ? h->X : h->Yt);
    const T *W = (const T *)(xstep ? h->Yt : h->X);
    const size_t need = (size_t)std::max<int64_t>(1, std::max(h->csr.nchunks, h->csc.nchunks)) *
                        Tri<K>::P * sizeof(T);
    if (h->s.als_bytes < need) {
        dfree(h->s.als_part, h->stream);
        h->s.als_part = nullptr;
        h->s.als_bytes = 0;
        cudaError_t e = dalloc(h, &h->s.als_part, need);
        if (e != cudaSuccess) return e;
        h->s.als_bytes = need;
    }
    T *part = (T *)h->s.als_part;
    h->launches += 1 + (o.nchunks ? 1 : 0);
    tmark(h, xstep ? "als_gram_x" : "als_gram_y");
    if (o.nchunks)
        als_gram_kernel<T, K><<<blocks_for(o.nchunks, kAlsWarps), kAlsWarps * 32, 0, h->stream>>>(
            o.nchunks, o.chunks, o.idx, (const T *)o.val, W, h->k, gram_vec<T>(W, h->k), part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    tmark(h, xstep ? "als_solve_x" : "als_solve_y");
    if constexpr (sizeof(T) == 4) {
        constexpr size_t smem = sizeof(SpdSmem<K>) * (32 / K) * kAlsWarps;
        int sms = 0, per = 0;
        if ((e = cudaFuncSetAttribute(als_solve_refined_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem)) != cudaSuccess)
            return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, als_solve_refined_kernel<K>, kAlsWarps * 32,
                                                               smem)) != cudaSuccess)
            return e;
        const int64_t want = blocks_for(o.nseg, kAlsWarps * (32 / K));
        als_solve_refined_kernel<K>
            <<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * std::max(per, 1))),
               kAlsWarps * 32, smem, h->stream>>>(o.nseg, o.segchunk, part, h->k, gamma, F, h->s.err);
    } else {
        als_solve_kernel<T, K><<<blocks_for(o.nseg, kAlsWarps), kAlsWarps * 32, 0, h->stream>>>(
            o.nseg, o.segchunk, part, h->k, gamma, F, h->s.err);
    }
    tmark(h, nullptr);
    return cudaGetLastError();
}

template <class T, int K>
cudaError_t launch_proxprox_half(glrm_s *h, bool xstep, double alpha, int inner)
{
    // the Gram partials of the ALS half-step (no solve), then the prox-prox solves
    const Orient &o = xstep ? h->csr : h->csc;
    T *F = (T *)(xstep ? h->X : h->Yt);
    const T *W = (const T *)(xstep ? h->Yt : h->X);
    const size_t need = (size_t)std::max<int64_t>(1, std::max(h->csr.nchunks, h->csc.nchunks)) *
                        Tri<K>::P * sizeof(T);
    if (h->s.als_bytes < need) {
        dfree(h->s.als_part, h->stream);
        h->s.als_part = nullptr;
        h->s.als_bytes = 0;
        cudaError_t e = dalloc(h, &h->s.als_part, need);
        if (e != cudaSuccess) return e;
        h->s.als_bytes = need;
    }
    T *part = (T *)h->s.als_part;
    h->launches += 1 + (o.nchunks ? 1 : 0);
    tmark(h, xstep ? "als_gram_x" : "als_gram_y");
    if (o.nchunks)
        als_gram_kernel<T, K><<<blocks_for(o.nchunks, kAlsWarps), kAlsWarps * 32, 0, h->stream>>>(
            o.nchunks, o.chunks, o.idx, (const T *)o.val, W, h->k, gram_vec<T>(W, h->k), part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    tmark(h, xstep ? "proxprox_x" : "proxprox_y");
    proxprox_solve_kernel<T, K><<<blocks_for(o.nseg, kAlsWarps), kAlsWarps * 32, 0, h->stream>>>(
        o.nseg, o.segchunk, part, h->k, alpha, inner, reg_code(h, xstep),
        xstep ? h->rx_w : h->ry_w, F, h->s.err);
    tmark(h, nullptr);
    return cudaGetLastError();
}

template <class T>
cudaError_t Engine<T>::proxprox_half(glrm_s *h, bool xstep, double alpha, int inner)
{
    const int k = h->k;
    if (k <= 4) return launch_proxprox_half<T, 4>(h, xstep, alpha, inner);
    if (k <= 8) return launch_proxprox_half<T, 8>(h, xstep, alpha, inner);
    if (k <= 16) return launch_proxprox_half<T, 16>(h, xstep, alpha, inner);
    if (k <= 32) return launch_proxprox_half<T, 32>(h, xstep, alpha, inner);
    return cudaErrorInvalidValue;
}

template <class T>
cudaError_t Engine<T>::als_half(glrm_s *h, bool xstep, double gamma)
{
    const int k = h->k;
    if (k <= 4) return launch_als_half<T, 4>(h, xstep, gamma);
    if (k <= 8) return launch_als_half<T, 8>(h, xstep, gamma);
    if (k <= 16) return launch_als_half<T, 16>(h, xstep, gamma);
    if (k <= 32) return launch_als_half<T, 32>(h, xstep, gamma);
    return cudaErrorInvalidValue;
}

}  // namespace glrm
