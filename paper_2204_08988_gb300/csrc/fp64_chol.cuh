// fp64_chol.cuh -- FP64 building blocks of the parameter and split/merge steps: staging a
// (sub-)cluster's statistics block in shared memory and a right-looking Cholesky (LDL)
// factorisation written for GB300's FP64 pipe (about two operations per clock per SM,
// 64-cycle dependent latency): the only serial work per pivot is one reciprocal, and the
// block meets one barrier per panel of four pivots.
#pragma once
#include "dpmm_internal.cuh"

namespace dpmm {

// out[e] = statistics entry e of slot (k, h) of the table S (E entries per sub-cluster);
// h = -1 sums the two sub-clusters (the cluster).  Every thread of the block calls it.
__device__ inline void stage_slot(const double* S, int E, int k, int h, double* out) {
    const double* s0 = S + (size_t)(2 * k + (h < 0 ? 0 : h)) * E;
    const double* s1 = S + (size_t)(2 * k + 1) * E;
    const int nt = blockDim.x;
    for (int e0 = threadIdx.x; e0 < E; e0 += 4 * nt) {  // four entries' loads in flight per thread
        double a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = e0 + u * nt;
            a[u] = e < E ? s0[e] : 0.0;
            b[u] = e < E && h < 0 ? s1[e] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (e0 + u * nt < E) out[e0 + u * nt] = h < 0 ? a[u] + b[u] : a[u];
    }
}

// Row i0 and column l0 (l0 <= i0) of entry e of a lower triangle enumerated row by row.
__device__ inline void tri_index(int e, int& i0, int& l0) {
    int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    if ((i + 1) * (i + 2) / 2 <= e) ++i;
    if (i * (i + 1) / 2 > e) --i;
    i0 = i;
    l0 = e - i * (i + 1) / 2;
}

__device__ inline float rsqrt_t(float x) { return rsqrtf(x); }
__device__ inline double rsqrt_t(double x) { return rsqrt(x); }

// 1 / v of a positive v in [2^-1000, 2^1000): the FP32 reciprocal of the mantissa, refined by one
// third-order (Householder) step r (1 + e + e^2), e = 1 - v r, so that three dependent FP64
// operations remain (a dependent one takes 64 cycles).  The division is kept out of line: beside
// this, inlined, it was executed for every pivot and its result dropped.
__device__ inline bool recip_range(double v) {  // false for NaN and what is not positive too
    return (unsigned)(__double2hiint(v) - (23 << 20)) < (unsigned)(2000 << 20);
}
__device__ inline double recip_fast(double v) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int e = (hi >> 20) - 1023;
    const float m = __int_as_float(0x3f800000 | (hi & 0xfffff) << 3 | (int)((unsigned)lo >> 29));
    const int rb = __float_as_int(__fdividef(1.f, m));  // in [1/2, 1]
    const double r = __hiloint2double((rb >> 3) + ((1023 - 127 - e) << 20), rb << 29);
    const double err = fma(-v, r, 1.0);
    return fma(r, fma(err, err, err), r);
}
static __device__ __noinline__ double recip_any(double v) { return 1.0 / v; }

// In-place factorisation of the symmetric matrix whose lower triangle is in A (d x d,
// row-major with row stride ld, shared memory; an odd ld keeps the column reads free of
// bank conflicts), in working type T.  Pivot j is v_j = the (j, j) entry of the Schur
// complement; the update is A_il -= (A_ij / v_j) A_lj for j < l <= i, so column j keeps its
// unscaled values.  On return piv[j] = v_j: Psi = U U^T with U_jj = sqrt(v_j),
// U_ij = A_ij / sqrt(v_j) (i > j), and log|Psi| = sum_j log v_j.
//
// Blocked by panels of four pivots with one panel of lookahead, one barrier a panel: warp 0
// applies the previous panel to the next four columns and factorises them while the other
// warps apply it to the rest of the lower triangle.  The four pivots are a serial chain of
// latencies (reciprocal, scaling, update) in registers, lane = row; the panel's 4 x 4 block passes by
// shuffle (in every lane redundantly it costs 16 FP64 instructions a panel, at 19 cycles of the pipe).  Every entry receives
// the same fused multiply-adds in the same order as in the unblocked algorithm.  At d = 32 in
// FP64 33,800 cycles, in FP32 8,000 (52,000 and 24,300 with the panel's columns in shared memory, a barrier on either
// side of the panel and rsqrt of every pivot in the chain).
// A pivot v_j that is not positive, or NaN, or in FP32 not above rel * dg[j], sets *fail
// (shared memory) and/or the device error word *derr (DPMM_ENUMERIC) and is replaced by
// the smallest normal value of T.  cols, cols2: 4 d values of T each (shared memory), scratch.
// Called by threads 0 .. nt - 1 (at least two warps); sync() is their barrier.
template <typename T, typename Sync>
__device__ inline void chol_ldl_blk(T* A, int d, int ld, T* piv, T* cols, T* cols2, const T* dg, T rel, int* fail,
                                    int* derr, int nt, Sync sync) {
    const int tid = threadIdx.x;
    for (int j0 = 0; j0 < d; j0 += 4) {
        const int pw = min(4, d - j0);
        T* cb = j0 & 4 ? cols2 : cols;        // this panel's scaled columns
        const T* pb = j0 & 4 ? cols : cols2;  // the previous panel's
        if (tid < 32) {
            if (j0 > 0) {
                for (int i = j0 + tid; i < d; i += 32) {
                    T c[4], a[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) c[q] = pb[q * d + i];
#pragma unroll
                    for (int l = 0; l < 4; ++l)
                        if (l < pw && i >= j0 + l) a[l] = A[i * ld + j0 + l];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int l = 0; l < 4; ++l)
                            if (l < pw && i >= j0 + l) a[l] = fma(-c[q], A[(j0 + l) * ld + j0 - 4 + q], a[l]);
#pragma unroll
                    for (int l = 0; l < 4; ++l)
                        if (l < pw && i >= j0 + l) A[i * ld + j0 + l] = a[l];
                }
                __syncwarp();
            }
            // the panel's first 32 rows with the pivots: lane = row; what the lanes need of the 4 x 4
            // block comes by shuffle (D_lq = A_l,j0+q)
            const int i0 = j0 + tid;
            T a[4], D[4][4], inv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) a[q] = i0 < d && tid >= q && q < pw ? A[i0 * ld + j0 + q] : T(0);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (q >= pw) break;
                T v = __shfl_sync(0xffffffffu, a[q], q);
#pragma unroll
                for (int l = q + 1; l < 4; ++l) D[l][q] = __shfl_sync(0xffffffffu, a[q], l);
                if constexpr (sizeof(T) == 8) {
                    if (recip_range(v)) {
                        inv[q] = recip_fast(v);
                    } else {
                        if (!(v > 0.0)) {
                            if (tid == 0 && fail) *fail = 1;
                            if (tid == 0 && derr) atomicExch(derr, (int)DPMM_ENUMERIC);
                            v = 2.2250738585072014e-308;
                        }
                        inv[q] = recip_any(v);
                    }
                } else {
                    if (!(v > (rel > T(0) ? rel * dg[j0 + q] : T(0)))) {
                        if (tid == 0 && fail) *fail = 1;
                        if (tid == 0 && derr) atomicExch(derr, (int)DPMM_ENUMERIC);
                        v = 1.17549435e-38f;
                    }
                    const T r = rsqrt_t(v);
                    inv[q] = r * r;
                }
                if (tid == 0) piv[j0 + q] = v;
                const T c = a[q] * inv[q];
#pragma unroll
                for (int l = q + 1; l < 4; ++l) a[l] = fma(-c, D[l][q], a[l]);  // kept where l <= row
                if (i0 < d && tid > q) cb[q * d + i0] = c;
            }
#pragma unroll
            for (int q = 1; q < 4; ++q)
                if (q < pw && i0 < d && tid >= q) A[i0 * ld + j0 + q] = a[q];
            for (int i = i0 + 32; i < d; i += 32) {  // the rows below
                T b[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q < pw) b[q] = A[i * ld + j0 + q];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q >= pw) break;
                    const T c = b[q] * inv[q];
                    cb[q * d + i] = c;
#pragma unroll
                    for (int l = q + 1; l < 4; ++l)
                        if (l < pw) b[l] = fma(-c, D[l][q], b[l]);
                }
#pragma unroll
                for (int q = 1; q < 4; ++q)
                    if (q < pw) A[i * ld + j0 + q] = b[q];
            }
        } else if (j0 > 0) {  // entries (i, l), l beyond this panel
            const int m = d - j0 - pw, n = m * (m + 1) / 2, st = nt - 32;
            for (int e0 = tid - 32; e0 < n; e0 += 4 * st) {  // four chains of updates at a time
                int ii[4], ll[4];
                T a[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    tri_index(min(e0 + u * st, n - 1), ii[u], ll[u]);
                    ii[u] += j0 + pw;
                    ll[u] += j0 + pw;
                    a[u] = A[ii[u] * ld + ll[u]];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (e0 + u * st < n) a[u] = fma(-pb[q * d + ii[u]], A[ll[u] * ld + j0 - 4 + q], a[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e0 + u * st < n) A[ii[u] * ld + ll[u]] = a[u];
            }
        }
        sync();
    }
}

}  // namespace dpmm
