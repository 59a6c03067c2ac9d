// Gram matrices and small symmetric positive definite solves of the
// alternating minimisation (Section 2.4 of Udell et al., "Generalized Low Rank
// Models": every row / column problem is a k x k linear system), shared by the
// single-model ALS and prox-prox half-steps (glrm_als.cuh) and the batched
// form (glrm_batch.cu).  A group of K lanes owns one system (32 / K systems
// per warp side by side).
#pragma once

#include "glrm_tiled.cuh"

namespace glrm {

// A lane's share of sum_e w_e w_e^T and sum_e a_e w_e: rows r0 .. r0 + TR - 1,
// columns c0 .. c0 + TC - 1 of the full K x K matrix (TR TC = K, so the K
// lanes of a group tile it) in registers.  Reading a triangle's entries one by
// one from shared memory takes two loads per multiply-add (the shared-memory
// pipe was 98% busy); a tile takes TR + TC values for TR TC multiply-adds.
template <class T, int K>
struct GramTile {
    static constexpr int TC = K == 32 ? 8 : 4, TR = K / TC;
    T acc[TR][TC], b[TR];
    int r0, c0;

    __device__ __forceinline__ void init(int lr)
    {
        r0 = lr / (K / TC) * TR;
        c0 = lr % (K / TC) * TC;
#pragma unroll
        for (int i = 0; i < TR; ++i) {
            b[i] = T(0);
#pragma unroll
            for (int j = 0; j < TC; ++j) acc[i][j] = T(0);
        }
    }
    // One entry: its row of the other factor (K values, 16-byte aligned) and its value.
    __device__ __forceinline__ void add(const T *row, T a)
    {
        T wr[TR], wc[TC];
#pragma unroll
        for (int i = 0; i < TR; ++i) wr[i] = row[r0 + i];
#pragma unroll
        for (int j = 0; j < TC; ++j) wc[j] = row[c0 + j];
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                const unsigned long long w2 = pk2(wr[i], wr[i]);
#pragma unroll
                for (int j = 0; j < TC; j += 2)
                    upk2(ffma2(w2, pk2(wc[j], wc[j + 1]), pk2(acc[i][j], acc[i][j + 1])), acc[i][j], acc[i][j + 1]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = fma(wr[i], wc[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < TR; ++i) b[i] = fma(a, wr[i], b[i]);
    }
};

// Largest value over the lanes of a K-lane group (K a power of two, groups
// aligned), on every lane of it.
template <int K, class T>
__device__ __forceinline__ T group_max(T v)
{
#pragma unroll
    for (int o = K / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Shared memory of one group's solve.
template <int K>
struct SpdSmem {
    double G[K * K];        // the matrix, both triangles
    double b[K];            // the right-hand side
    double x[K];
    float L[K * (K + 1)];   // the matrix in FP32, then its factor
    float col[2][K];        // the current column of the factorisation
};

// Solve G x = b for the K x K system of every lane group at once (lane lr
// owns row lr and receives x_lr): an FP32 L D L^T factorisation as the
// preconditioner of an iterative refinement whose residual b - G x is formed
// in FP64, until the correction is below 2^-30 of the solution (the error is
// then that correction times the refinement's contraction, about 1e-12 or
// less; the results are stored in FP32).  Two rounds are usual for systems of
// condition number up to 1e4: 2 K FP64 multiply-adds per lane, against the
// K^2 / 6 + 12 K of an FP64 Cholesky factorisation with its pivots' reciprocal
// roots on one lane, on a pipe of 1/64 of the FP32 rate.  Returns, to every
// lane of the group, false where a pivot was not positive and finite or the
// corrections did not shrink below the bound in kSpdRounds rounds: the caller
// then factorises that system in FP64.
constexpr int kSpdRounds = 6;

template <int K>
__device__ bool spd_solve_refined(SpdSmem<K> &S, double &x)
{
    const int lr = (threadIdx.x & 31) % K;
    float a[K];
#pragma unroll
    for (int j = 0; j < K; ++j) a[j] = S.L[lr * (K + 1) + j];
    bool ok = true;
    float dinv = 0.f;
#pragma unroll
    for (int c = 0; c < K; ++c) {
        float *col = S.col[c & 1];
        col[lr] = a[c];
        __syncwarp();
        const float d = col[c];
        ok = ok && d > 0.f && d < 3.0e38f;
        const float r = __frcp_rn(d);
        const float l = a[c] * r;
#pragma unroll
        for (int j = c + 1; j < K; ++j) a[j] = fmaf(-l, col[j], a[j]);  // (lanes up to c hold nothing that is read again)
        if (lr > c) a[c] = l;
        if (lr == c) dinv = r;
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < K; ++c) S.L[lr * (K + 1) + c] = a[c];
    __syncwarp();
    auto apply = [&](float v) {  // (L D L^T)^-1 v
#pragma unroll
        for (int c = 0; c < K - 1; ++c) {
            const float vc = __shfl_sync(0xffffffffu, v, c, K);
            if (lr > c) v = fmaf(-a[c], vc, v);
        }
        v *= dinv;
#pragma unroll
        for (int c = K - 1; c > 0; --c) {
            const float vc = __shfl_sync(0xffffffffu, v, c, K);
            if (lr < c) v = fmaf(-S.L[c * (K + 1) + lr], vc, v);
        }
        return v;
    };
    x = (double)apply((float)S.b[lr]);
    bool done = false;
    for (int it = 0; it < kSpdRounds; ++it) {
        S.x[lr] = x;
        __syncwarp();
        double r0 = S.b[lr], r1 = 0.0;
#pragma unroll
        for (int c = 0; c < K; c += 2) {
            r0 = fma(-S.G[c * K + lr], S.x[c], r0);
            r1 = fma(-S.G[(c + 1) * K + lr], S.x[c + 1], r1);
        }
        __syncwarp();
        const float dx = apply((float)(r0 + r1));
        const float dm = group_max<K>(fabsf(dx)), xm = group_max<K>(fabsf((float)x));
        if (!done) x += (double)dx;
        done = done || dm <= 0x1p-30f * xm;  // false for NaN
        if (__all_sync(0xffffffffu, done || !ok)) break;
    }
    return ok && done;  // the same on every lane of the group: both follow from its shared values
}

}  // namespace glrm
